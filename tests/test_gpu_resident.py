"""The single-trajectory kernel that keeps K, or U and V, in shared memory: against the FP64
oracle and the stage-wise kernels, at the smallest and largest models that it takes and just
outside, odd and tiny ranks, ragged shares of k-points, both band counts, with and without
compensation, and continued runs.

Tolerance: 1e-5 relative L2 of the observables against the oracle, the bound of every FP32
path, and 2e-6 against the stage-wise kernels (the same FP32 arithmetic in another order)."""
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

PULSE = wl.Pulse(E0=5e-3, omega=0.12, t0=3.0, sigma=1.2, dir_x=0.6, dir_y=0.8)


def _run(p, mode, apply, install=None, T=24):
    mdl = om.Model(p)
    ref, _ = op.rk4(mdl, apply(mdl), op.half_step_samples(PULSE, 0.2, T), 0.2, T, direction=(0.6, 0.8))
    ctx = tg.Context(p, tg.C64, stream=torch.cuda.current_stream().cuda_stream)
    if install:
        install(ctx)
    got = ctx.propagate(PULSE, T, 0.2, mode)
    assert op.rel_l2(got, ref) < 1e-5
    sw = ctx.propagate(PULSE, T, 0.2, mode, tg.FLAG_RESET | tg.FLAG_STAGEWISE)
    assert op.rel_l2(got, sw) < 2e-6
    plain = ctx.propagate(PULSE, T, 0.2, mode, tg.FLAG_RESET | tg.FLAG_NO_KAHAN)
    assert op.rel_l2(plain, ref) < 1e-5
    # a run in two parts repeats the whole run bit for bit (the streaming kernel, for factors
    # too large to stay resident, sums the observables of the cut's first row elsewhere)
    a = ctx.propagate(PULSE, 9, 0.2, mode)
    b = ctx.propagate(PULSE, T - 9, 0.2, mode, flags=0)
    np.testing.assert_array_equal(a, got[:10])
    np.testing.assert_array_equal(b[1:], got[10:])
    np.testing.assert_allclose(b[0], got[9], rtol=1e-10, atol=1e-15)


@pytest.mark.parametrize("L,nc", [(8, 1), (9, 1), (5, 2), (12, 1), (13, 1), (7, 2), (21, 1), (22, 1), (11, 2), (23, 1)])
def test_dense(L, nc):
    _run(wl.small_model(L, nc), tg.FULL, lambda m: (lambda K: (lambda v: K @ v))(ok.dense_kernel(m)))


@pytest.mark.parametrize("L,nc,rank", [(2, 1, 1), (3, 2, 2), (9, 1, 7), (12, 1, 29), (23, 1, 235), (24, 1, 256),
                                       (24, 1, 400), (11, 2, 129), (13, 2, 64), (5, 1, 100), (30, 1, 511),
                                       (12, 1, 300), (12, 1, 340), (24, 1, 70), (3, 1, 36), (16, 2, 33)])
def test_lowrank(L, nc, rank):
    p = wl.small_model(L, nc)
    U, S, V, d = wl.random_factors(p.N, rank, seed=rank + L)
    _run(p, tg.LOWRANK, lambda m: (lambda v: olr.apply_lowrank(d, U, S, V, v)),
         lambda c: tg.tdagw_set_factors(c.h, U, S, V, d))


def test_dense_completes_with_the_timeout_hook():
    ctx = tg.Context(wl.small_model(12, 1), tg.C64, stream=torch.cuda.current_stream().cuda_stream)
    got = ctx.propagate(PULSE, 6, 0.2, tg.FULL, tg.FLAG_RESET | tg.FLAG_TEST_TIMEOUT)
    np.testing.assert_array_equal(got, ctx.propagate(PULSE, 6, 0.2, tg.FULL, tg.FLAG_RESET | tg.FLAG_STAGEWISE))
