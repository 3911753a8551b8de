"""On-chip low-rank runs with many columns over many CTAs, against the oracle and the stage-wise
kernels, and the forms of a single-trajectory call that a model's size no longer reaches by itself: runs
replayed from a captured graph against the same launches made directly (32 steps per replay, a
tail of direct steps), continued runs on the stage-wise kernels, and the bounded waits of the
streaming low-rank kernel beside those of the on-chip one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2502_05635_gb300 as tg  # noqa: E402
import workloads as wl  # noqa: E402
from oracle import lowrank as olr  # noqa: E402
from oracle import propagate as op  # noqa: E402
from test_gpu_resident import _run  # noqa: E402

PULSE = wl.Pulse(E0=5e-3, omega=0.12, t0=3.0, sigma=1.2, dir_x=0.6, dir_y=0.8)


def _ctx(L, nc, mode, rank=0, dtype=tg.C64, kblocks=0):
    p = wl.small_model(L, nc)
    P, Nk = p.Nb ** 2, L * L
    c = tg.Context(p, dtype, stream=torch.cuda.current_stream().cuda_stream)
    if mode == tg.LOWRANK:
        U, S, V, d = wl.random_factors(p.N, rank, seed=rank)
        tg.tdagw_set_kdiag_blocks(c.h, kblocks)
        tg.tdagw_set_factors(c.h, U, S, V, np.zeros((Nk, P, P), complex) if kblocks else d)
    elif mode == tg.CHANNEL:
        rng = np.random.default_rng(rank)
        U = (rng.standard_normal((P, P, Nk, rank)) + 1j * rng.standard_normal((P, P, Nk, rank))) / np.sqrt(2 * Nk)
        tg.tdagw_set_channel_factors(c.h, U, np.full((P, P, rank), 1e-2), U)
    return c


CASES = [(12, 1, tg.FULL, 0, tg.C64), (12, 1, tg.LOWRANK, 29, tg.C64), (9, 1, tg.CHANNEL, 4, tg.C64),
         (6, 2, tg.FULL, 0, tg.C64), (12, 1, tg.FULL, 0, tg.C128), (23, 1, tg.LOWRANK, 40, tg.C128)]
IDS = ["dense", "lowrank", "channel", "nb4-dense", "dense-c128", "lowrank-c128"]


@pytest.mark.parametrize("L,nc,mode,rank,dtype", CASES, ids=IDS)
@pytest.mark.parametrize("T", [2, 31, 101])
def test_graph_replay_and_direct_launches_agree(L, nc, mode, rank, dtype, T):
    c = _ctx(L, nc, mode, rank, dtype)
    flags = tg.FLAG_RESET | tg.FLAG_STAGEWISE
    a = c.propagate(PULSE, T, 0.2, mode, flags)
    b = c.propagate(PULSE, T, 0.2, mode, flags | tg.FLAG_NO_GRAPH)
    assert np.abs(a[:, 0]).max() > 0
    np.testing.assert_array_equal(a, b)
    c.close()


@pytest.mark.parametrize("L,nc,mode,rank,dtype", CASES, ids=IDS)
def test_resume_on_the_stagewise_kernels_is_bitwise(L, nc, mode, rank, dtype):
    c = _ctx(L, nc, mode, rank, dtype)
    full = c.propagate(PULSE, 80, 0.2, mode, tg.FLAG_RESET | tg.FLAG_STAGEWISE)
    first = c.propagate(PULSE, 37, 0.2, mode, tg.FLAG_RESET | tg.FLAG_STAGEWISE)
    np.testing.assert_array_equal(first, full[:38])
    if dtype == tg.C64:
        # through a saved state, exact in complex64 (sum and carry of 32 bits in 64); in complex128 the
        # saved sum is rounded to 64 bits, so the run goes on in its context
        drho, carry, step = tg.tdagw_get_state(c.h)
        c.close()
        c = _ctx(L, nc, mode, rank, dtype)
        tg.tdagw_set_state(c.h, drho, carry, step)
    second = c.propagate(PULSE, 43, 0.2, mode, tg.FLAG_STAGEWISE)
    np.testing.assert_array_equal(second, full[37:])
    c.close()


@pytest.mark.parametrize("L,nc,rank,kblocks", [(12, 1, 29, 0), (12, 1, 29, 1), (36, 2, 830, 0)],
                         ids=["on-chip", "streamed", "streamed-with-prefetch"])
def test_lowrank_timeout_is_reported_and_context_survives(L, nc, rank, kblocks):
    """The grid barrier waits for a block that does not exist: every wait gives up after its budget
    (the streaming kernel's copies in flight are awaited), the call reports TDAGW_ERR_TIMEOUT and
    the same context then propagates normally."""
    c = _ctx(L, nc, tg.LOWRANK, rank, kblocks=kblocks)
    tg.tdagw_propagate(c.h, [tg.make_field(PULSE)], [20], 0.2, tg.LOWRANK, tg.FLAG_RESET | tg.FLAG_TEST_TIMEOUT)
    with pytest.raises(tg.TdagwError) as e:
        tg.tdagw_sync(c.h)
    assert e.value.code == tg.ERR_TIMEOUT
    good = c.propagate(PULSE, 20, 0.2, tg.LOWRANK)
    ref = c.propagate(PULSE, 20, 0.2, tg.LOWRANK, tg.FLAG_RESET | tg.FLAG_STAGEWISE)
    assert op.rel_l2(good[:, 0], ref[:, 0]) < 1e-6
    c.close()


@pytest.mark.parametrize("L,nc,rank", [(23, 1, 500), (30, 1, 511), (36, 1, 320), (17, 2, 400), (24, 2, 190)])
def test_onchip_lowrank_with_long_exchange(L, nc, rank):
    """Up to 152 partial vectors of up to 512 columns per stage; tolerances of the on-chip kernel's
    other tests (the same sums)."""
    p = wl.small_model(L, nc)
    U, S, V, d = wl.random_factors(p.N, rank, seed=rank + L)
    _run(p, tg.LOWRANK, lambda m: (lambda v: olr.apply_lowrank(d, U, S, V, v)),
         lambda c: tg.tdagw_set_factors(c.h, U, S, V, d), T=12)
