"""Low-rank applications at the edges of their kernels, against the same product in FP64 (numpy)
on the same factors: the one-launch cluster kernel and the three-launch path on both sides of
the line between them, odd and tiny ranks, fewer rows than CTAs or warps, both precisions, and
the allocation-free entry point.

Tolerance: relative L2 of y, 1e-6 in complex64 (inputs exact in FP32, sums of at most a few
thousand terms of one sign-random product each: below 16 x 2^-24) and 1e-13 in complex128."""
import numpy as np
import pytest

import workloads as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2502_05635_gb300 as tg  # noqa: E402

CASES = [(1, 1, 1), (1, 2, 3), (2, 1, 16), (5, 1, 7), (12, 1, 29), (12, 1, 113), (12, 1, 114), (12, 1, 513),
         (8, 2, 64), (17, 2, 231), (24, 1, 256), (30, 1, 2)]


def _factors(N, r):
    U, S, V, d = wl.random_factors(N, r, seed=N + r)
    f32 = lambda a: a.astype(np.complex64 if np.iscomplexobj(a) else np.float32)
    return f32(U), f32(S), f32(V), f32(d)


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("dtype,tol", [(tg.C64, 1e-6), (tg.C128, 1e-13)], ids=["c64", "c128"])
@pytest.mark.parametrize("L,nc,rank", CASES)
def test_apply_lowrank_edges(L, nc, rank, dtype, tol):
    p = wl.small_model(L, nc)
    rank = min(rank, p.N)
    U, S, V, d = _factors(p.N, rank)
    x = wl.random_state(p.N, 5).astype(np.complex64)
    ref = d.astype(complex) * x + U.astype(complex) @ (S.astype(float) * (V.astype(complex).conj().T @ x.astype(complex)))
    ctx = tg.Context(p, dtype, stream=torch.cuda.current_stream().cuda_stream)
    tg.tdagw_set_factors(ctx.h, U, S, V, d)
    tdt = torch.complex64 if dtype == tg.C64 else torch.complex128
    xd = torch.from_numpy(x).to("cuda", tdt)
    y = torch.full_like(xd, float("nan"))
    tg.tdagw_apply(ctx.h, tg.LOWRANK, xd, y)
    assert _rel(y.cpu().numpy(), ref) < tol


@pytest.mark.parametrize("N,rank,ld", [(1, 1, 2), (7, 3, 4), (576, 29, 32), (576, 114, 114), (2304, 255, 256),
                                       (4000, 513, 514)])
def test_noalloc_edges(N, rank, ld):
    U, S, V, d = _factors(N, rank)
    x = wl.random_state(N, 6).astype(np.complex64)
    ref = d.astype(complex) * x + U.astype(complex) @ (S.astype(float) * (V.astype(complex).conj().T @ x.astype(complex)))
    pad = lambda a: torch.from_numpy(np.pad(a, ((0, 0), (0, ld - rank)), constant_values=np.nan)).cuda()
    y = torch.full((N,), float("nan"), dtype=torch.complex64, device="cuda")
    tg.tdagw_apply_lowrank_noalloc(pad(U), pad(V), torch.from_numpy(S).cuda(), torch.from_numpy(d).cuda(),
                                   torch.from_numpy(x).cuda(), y, stream=torch.cuda.current_stream().cuda_stream)
    assert _rel(y.cpu().numpy(), ref) < 1e-6
