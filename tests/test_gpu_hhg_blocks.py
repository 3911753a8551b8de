"""HHG spectra at the edges of the kernel's blocks: trajectory groups of 1, 4 and 8 with
remainders, runs around a chunk's length, one frequency and one past a block, uneven lengths
with NaN after the end, against numpy in FP64 (relative 1e-10: sums of at most 1500 terms of
unit size in 2^-53 arithmetic, phases re-seeded per chunk)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2502_05635_gb300 as tg  # noqa: E402


@pytest.mark.parametrize("B,T,nfreq", [(1, 0, 1), (1, 31, 129), (3, 255, 33), (4, 256, 128), (7, 257, 5), (8, 1, 130),
                                       (9, 1500, 40), (17, 513, 257)])
def test_blocks(B, T, nfreq):
    rng = np.random.default_rng(B + T)
    steps = rng.integers(0, T + 1, B)
    steps[B // 2] = T
    obs = rng.standard_normal((T + 1, B, 3))
    for b in range(B):
        obs[steps[b] + 1:, b] = np.nan
    w = np.linspace(0.05, 2.0, nfreq)
    got = tg.tdagw_hhg_spectrum(obs, steps, 0.2, w, component=1)
    for b in range(B):
        t = 0.2 * np.arange(steps[b] + 1)
        F = np.exp(-1j * w[:, None] * t) @ obs[:steps[b] + 1, b, 1]
        ref = np.abs(w * F * 0.2) ** 2
        np.testing.assert_allclose(got[:, b], ref, rtol=1e-10, atol=1e-12 * max(ref.max(), 1e-300))
