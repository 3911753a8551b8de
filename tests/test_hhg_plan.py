"""Launch geometry of the HHG spectra (csrc/hhg_plan.h, compiled here with g++): within the grid
limits, covering every sample once, for all step counts that a propagation accepts; and, on the
GPU, one current that is longer than a grid has blocks along time."""
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2502_05635_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "hhg_plan.h"
int main() {
    int t, b, f;
    while (std::scanf("%d %d %d", &t, &b, &f) == 3) {
        const tdagw::HhgPlan p = tdagw::hhg_plan(t, b, f);
        std::printf("%d %d %d %d %d %d\n", p.tb, p.clen, p.cpb, p.gx, p.gy, p.nz);
    }
}
"""


def test_geometry_stays_within_the_grid(tmp_path):
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = tmp_path / "plan"
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(tmp_path / "main.cpp"), "-o", str(exe)], check=True)
    edge = 65535 * 256
    cases = [(t, b, f)
             for t in (0, 1, 31, 255, 256, 2000, edge - 2, edge - 1, edge, edge + 1, 1 << 25, 1 << 26, 2 ** 31 - 1)
             for b in (1, 3, 4, 8, 60, 65535) for f in (1, 33, 64, 512, 100000)]
    out = subprocess.run([str(exe)], input="\n".join("%d %d %d" % c for c in cases), text=True, check=True,
                         capture_output=True).stdout.split("\n")
    for (t, b, f), line in zip(cases, out):
        tb, clen, cpb, gx, gy, nz = map(int, line.split())
        assert gx * 128 >= f and gy * tb >= b and gx < 2 ** 31 and 1 <= gy <= 65535, (t, b, f)
        assert 1 <= nz <= 65535 and 1 <= clen <= 256, (t, b, f)
        assert (nz - 1) * cpb * clen < t + 1 <= nz * cpb * clen, (t, b, f)
        assert nz == 1 or nz * f * b * 16 <= 64 << 20, (t, b, f)


@pytest.mark.gpu
def test_run_longer_than_a_grid_of_chunks():
    """65535 chunks of 256 samples and a remainder, one frequency.  omega dt = 0.5 and omega n dt
    are exact, so the reference's phases are exact.  Bound: rounding of at most 4 (256 + cpb + nz)
    terms in sequence (phasor recurrence within a chunk, sums over chunks and blocks) relative to
    sum |J|, that is 3e-11, and twice that, times sum |J| / |F| = 2 for a resonant cosine, on the
    square."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2502_05635_gb300 as tg
    T = 65535 * 256 + 300
    ph = 0.5 * np.arange(T + 1)
    J = np.cos(ph)
    got = tg.tdagw_hhg_spectrum(J[:, None], [T], 0.25, np.array([2.0]))
    ref = 0.25 * (np.dot(J, J) ** 2 + np.dot(J, np.sin(ph)) ** 2)
    np.testing.assert_allclose(got[0, 0], ref, rtol=1.2e-10)
