"""The stage-wise single-trajectory kernels at the edges of their sums, against the FP64 oracle: the
last block's sum of the blocks' observables (one block, 31 to 34 of them, and more; 256 threads in
complex64, 32 in complex128), and the sum of the V pass's partial vectors (one per 16 rows: 1, 3 to
5, 15 to 17 and more).  Tolerances: those of the propagation tests, 1e-5 and 1e-10 relative L2 for
the two precisions, and of the application tests, 2e-6 and 1e-12 of the largest entry."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2502_05635_gb300 as tg  # noqa: E402
import workloads as wl  # noqa: E402
from oracle import channel as oc  # noqa: E402
from oracle import lowrank as olr  # noqa: E402
from oracle import model as om  # noqa: E402
from oracle import propagate as op  # noqa: E402

PULSE = wl.Pulse(E0=5e-3, omega=0.12, t0=1.0, sigma=0.8, dir_x=0.6, dir_y=0.8)


def _ctx(p, dtype=tg.C64):
    return tg.Context(p, dtype, stream=torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("L,nc,dtype,tol", [(2, 1, tg.C128, 1e-10), (3, 1, tg.C128, 1e-10), (15, 1, tg.C128, 1e-10),
                                            (16, 1, tg.C128, 1e-10), (17, 1, tg.C128, 1e-10), (8, 2, tg.C128, 1e-10),
                                            (8, 1, tg.C64, 1e-5), (9, 1, tg.C64, 1e-5), (22, 2, tg.C64, 1e-5),
                                            (45, 1, tg.C64, 1e-5), (23, 2, tg.C64, 1e-5)])
def test_observables_over_block_counts(L, nc, dtype, tol):
    p = wl.small_model(L, nc)
    mdl = om.Model(p)
    U, S, V, d = wl.random_factors(p.N, 3, seed=L)
    ref, _ = op.rk4(mdl, lambda v: olr.apply_lowrank(d, U, S, V, v), op.half_step_samples(PULSE, 0.2, 8), 0.2, 8,
                    direction=(0.6, 0.8))
    c = _ctx(p, dtype)
    tg.tdagw_set_factors(c.h, U, S, V, d)
    got = c.propagate(PULSE, 8, 0.2, tg.LOWRANK, tg.FLAG_RESET | tg.FLAG_STAGEWISE)
    c.close()
    for j in range(3):
        assert op.rel_l2(got[1:, j], ref[1:, j]) < tol, j


@pytest.mark.parametrize("dtype,tol", [(tg.C64, 2e-6), (tg.C128, 1e-12)], ids=["c64", "c128"])
@pytest.mark.parametrize("L,nc", [(1, 1), (3, 1), (4, 1), (5, 1), (2, 2), (8, 1), (4, 2), (9, 1), (17, 1), (5, 2)])
def test_partial_vector_counts(L, nc, dtype, tol):
    p = wl.small_model(L, nc)
    P, Nk, r = p.Nb ** 2, L * L, min(3, L * L)
    rng = np.random.default_rng(L)
    g = lambda *s: (rng.standard_normal(s) + 1j * rng.standard_normal(s)) / np.sqrt(2 * Nk)
    U, V, D, S = g(P, P, Nk, r), g(P, P, Nk, r), g(P, Nk, Nk), rng.uniform(0.1, 1.0, (P, P, r))
    for q in range(P):
        U[q, q] = V[q, q] = 0
        S[q, q] = 0
    Ul, Sl, Vl, dl = wl.random_factors(p.N, min(5, p.N), seed=L)
    c = _ctx(p, dtype)
    tg.tdagw_set_channel_factors(c.h, U, S, V, D)
    tg.tdagw_set_factors(c.h, Ul, Sl, Vl, dl)
    x = wl.random_state(p.N, 3)
    tx = torch.from_numpy(x).to("cuda", torch.complex64 if dtype == tg.C64 else torch.complex128)
    for mode, ref in ((tg.CHANNEL, oc.apply_channel(D, U, S, V, x)), (tg.LOWRANK, olr.apply_lowrank(dl, Ul, Sl, Vl, x))):
        y = torch.full_like(tx, float("nan"))
        tg.tdagw_apply(c.h, mode, tx, y)
        assert np.abs(y.cpu().numpy() - ref).max() < tol * np.abs(ref).max(), mode
    c.close()
