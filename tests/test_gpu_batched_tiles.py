"""FP32 batched products at the edges of their register tiles and of the work split, vs the
FP64 oracle: ranks on both sides of every tile height, row counts per CTA from one k-point to
several tiles, trajectory counts around the 32-column tile, active counts that change the split
from step to step.

Tolerance: 1e-5 relative L2 of the observables per trajectory, the bound of every FP32 path
(inputs rounded to 2^-24, sums of at most a few thousand FP32 terms: about 1e-7 to 1e-6)."""
import numpy as np
import pytest

import workloads as wl
from oracle import kernel as ok
from oracle import lowrank as olr
from oracle import model as om
from oracle import propagate as op

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2502_05635_gb300 as tg  # noqa: E402


def _check(mode, apply, mdl, ctx, B, flags=0):
    pulses = wl.early_pulses(B)
    steps = [3 + (7 * b) % 9 for b in range(B)]
    got = ctx.propagate_batch(pulses, steps, 0.2, mode, tg.FLAG_RESET | flags)
    for b in sorted({0, 1, B // 2, B - 1}):
        s = op.half_step_samples(pulses[b], 0.2, steps[b])
        ref, _ = op.rk4(mdl, apply, s, 0.2, steps[b], direction=(pulses[b].dir_x, pulses[b].dir_y))
        assert op.rel_l2(got[:steps[b] + 1, b], ref) < 1e-5, (b, steps[b])
        assert np.all(np.isnan(got[steps[b] + 1:, b]))


@pytest.mark.parametrize("L,nc,rank,B", [(9, 1, 1, 2), (9, 1, 64, 33), (9, 1, 65, 31), (9, 1, 129, 65),
                                         (13, 1, 257, 32), (13, 1, 300, 97), (20, 1, 63, 260), (5, 2, 128, 40),
                                         (14, 2, 40, 7)])
def test_lowrank_tile_edges(L, nc, rank, B):
    p = wl.small_model(L, nc)
    mdl = om.Model(p)
    U, S, V, d = wl.random_factors(p.N, rank, seed=rank)
    ctx = tg.Context(p, tg.C64, stream=torch.cuda.current_stream().cuda_stream)
    tg.tdagw_set_factors(ctx.h, U, S, V, d)
    _check(tg.LOWRANK, lambda v: olr.apply_lowrank(d, U, S, V, v), mdl, ctx, B)


@pytest.mark.parametrize("L,nc,B", [(3, 1, 2), (9, 1, 33), (5, 2, 70), (13, 1, 150)])
def test_dense_tile_edges(L, nc, B):
    p = wl.small_model(L, nc)
    mdl = om.Model(p)
    K = ok.dense_kernel(mdl)
    ctx = tg.Context(p, tg.C64, stream=torch.cuda.current_stream().cuda_stream)
    _check(tg.FULL, lambda v: K @ v, mdl, ctx, B)
