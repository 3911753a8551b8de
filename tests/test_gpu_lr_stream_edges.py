"""The streaming single-trajectory low-rank kernel, for factors too large to stay on the chip,
around the edges of its V pass by row subsets (ranks up to 512: 2, 3 and 10 subsets, odd ranks,
threads beyond the last subset) and of its L2 prefetch (factors above two and above four times
L2, ragged shares of k-points): against the FP64 oracle, the stage-wise kernels and itself in
two parts.  Tolerances: those of the on-chip kernel's tests, for the same arithmetic."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2502_05635_gb300 as tg  # noqa: E402
import workloads as wl  # noqa: E402
from oracle import lowrank as olr  # noqa: E402
from test_gpu_resident import _run  # noqa: E402


@pytest.mark.parametrize("L,nc,rank", [(36, 2, 101), (24, 2, 300), (25, 2, 340), (23, 2, 511), (24, 2, 512),
                                       (24, 2, 513), (36, 2, 830), (48, 2, 900)])
def test_streamed_lowrank(L, nc, rank):
    p = wl.small_model(L, nc)
    U, S, V, d = wl.random_factors(p.N, rank, seed=rank + L)
    _run(p, tg.LOWRANK, lambda m: (lambda v: olr.apply_lowrank(d, U, S, V, v)),
         lambda c: tg.tdagw_set_factors(c.h, U, S, V, d), T=12)
