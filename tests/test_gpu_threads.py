"""Four threads, each with a context and a stream of its own, with models of two sizes through
the same single-launch kernel: the launches' shared-memory sizes differ, and neither thread may
change what another one launches with.  Every call has to succeed and repeat its thread's first
result bit for bit."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2502_05635_gb300 as tg  # noqa: E402
import workloads as wl  # noqa: E402

PULSE = wl.Pulse(E0=5e-3, omega=0.12, t0=0.4, sigma=0.8)


def _factors(c, p, mode, rank, kblocks):
    P, Nk = p.Nb ** 2, p.N // p.Nb ** 2
    if mode == tg.LOWRANK:
        U, S, V, d = wl.random_factors(p.N, rank, seed=rank)
        tg.tdagw_set_kdiag_blocks(c.h, kblocks)
        tg.tdagw_set_factors(c.h, U, S, V, np.zeros((Nk, P, P), complex) if kblocks else d)
    elif mode == tg.CHANNEL:
        rng = np.random.default_rng(rank)
        U = (rng.standard_normal((P, P, Nk, rank)) + 1j * rng.standard_normal((P, P, Nk, rank))) / np.sqrt(2 * Nk)
        tg.tdagw_set_channel_factors(c.h, U, np.full((P, P, rank), 1e-2), U)


@pytest.mark.parametrize("mode,sizes,kblocks", [(tg.FULL, ((9, 0), (12, 0)), 0), (tg.FULL, ((14, 0), (19, 0)), 0),
                                                (tg.LOWRANK, ((12, 20), (12, 200)), 0),
                                                (tg.LOWRANK, ((23, 100), (23, 235)), 0),
                                                (tg.LOWRANK, ((8, 3), (24, 100)), 1),
                                                (tg.CHANNEL, ((5, 1), (23, 30)), 0)],
                         ids=["dense-cluster", "dense-grid", "lowrank-cluster", "lowrank-grid", "streamed", "channel"])
def test_two_sizes_from_four_threads(mode, sizes, kblocks):
    errors = []

    def work(L, rank, start):
        try:
            p = wl.small_model(L, 1)
            st = torch.cuda.Stream()
            c = tg.Context(p, tg.C64, stream=st.cuda_stream)
            _factors(c, p, mode, rank, kblocks)
            first = c.propagate(PULSE, 2, 0.2, mode)
            start.wait(120)
            f = [tg.make_field(PULSE)]
            for n in range(4000):  # launches follow one another: only every eighth result is read
                tg.tdagw_propagate(c.h, f, [2], 0.2, mode)
                if n % 8 == 7:
                    np.testing.assert_array_equal(tg.tdagw_observables(c.h), first)
            c.close()
        except Exception as e:  # noqa: BLE001
            errors.append(e)
            start.abort()

    start = threading.Barrier(4)
    ts = [threading.Thread(target=work, args=(L, r, start)) for L, r in sizes * 2]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not errors, errors
