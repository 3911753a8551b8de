"""Small calls on kernels whose work split is made for large ones: results against the FP64
oracle where few trajectories or columns leave most threads without work, and that a call is not
slower than one that has many times its work (best of several passes)."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2502_05635_gb300 as tg  # noqa: E402
import test_gpu_channel_tc as ctc  # noqa: E402
import workloads as wl  # noqa: E402


def _best(f, n=15):
    for _ in range(3):
        f()
    torch.cuda.synchronize()
    best = 1e30
    for _ in range(n):
        t0 = time.perf_counter()
        f()
        torch.cuda.synchronize()
        best = min(best, time.perf_counter() - t0)
    return best


def _gauss(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / np.sqrt(2 * shape[-2])


@pytest.mark.parametrize("L,nc,B", [(12, 1, 1), (13, 1, 2), (5, 2, 3), (9, 2, 5), (9, 2, 1)])
def test_split_channel_few_trajectories_vs_oracle(L, nc, B):
    """k-points fewer, as many and more than the CTAs, one to five trajectories of uneven
    lengths; the bar of the split-FP16 paths (1e-4)."""
    p = wl.small_model(L, nc)
    mdl, fac, _ = ctc._factors(p, 5)
    c = ctc._ctx(p)
    tg.tdagw_set_channel_factors(c.h, fac[1], fac[2], fac[3], fac[0])
    pulses, steps = ctc._pulses(B, 7 * L + B), [40 - 7 * b for b in range(B)]
    got = c.propagate_batch(pulses, steps, 0.2, tg.CHANNEL, ctc.SPLIT).reshape(41, B, 3)
    c.close()
    ctc._check_vs_oracle(mdl, fac, got, pulses, steps)


def test_split_channel_one_trajectory_not_slower_than_64():
    p = wl.small_model(20, 2)
    P, Nk, z = p.Nb ** 2, 400, 4
    rng = np.random.default_rng(3)
    U = _gauss(rng, P, P, Nk, z)
    S = 1e-2 * np.exp(-4.0 * np.arange(z) / z) * np.ones((P, P, 1))
    c = ctc._ctx(p)
    tg.tdagw_set_channel_factors(c.h, U, S, U)
    pulses = ctc._pulses(64, 1)
    one = _best(lambda: c.propagate_batch(pulses[:1], [40], 0.2, tg.CHANNEL, ctc.SPLIT))
    many = _best(lambda: c.propagate_batch(pulses, [40] * 64, 0.2, tg.CHANNEL, ctc.SPLIT))
    c.close()
    print(f"one {one * 1e3:.3f} ms, 64 {many * 1e3:.3f} ms")
    assert one < many, (one, many)


@pytest.mark.parametrize("L,nc,kblocks", [(12, 1, 0), (23, 1, 0), (36, 1, 0), (13, 2, 0), (23, 1, 1)],
                         ids=["cluster", "grid", "large-grid", "nb4-grid", "streamed"])
def test_lowest_ranks_not_slower_than_sixteen(L, nc, kblocks):
    """One trajectory at ranks 1 and 2 (on-chip kernel; with k-block diagonals the streaming one):
    the sums of the row subsets may not outgrow the products.  At rank 16 there are at most 64 of
    them, at ranks 1 and 2 as many as a CTA has rows: half as much again is allowed."""
    p = wl.small_model(L, nc)
    P, t = p.Nb ** 2, {}
    for rank in (1, 2, 16):
        U, S, V, d = wl.random_factors(p.N, rank, seed=rank)
        c = ctc._ctx(p)
        tg.tdagw_set_kdiag_blocks(c.h, kblocks)
        tg.tdagw_set_factors(c.h, U, S, V, np.zeros((L * L, P, P), complex) if kblocks else d)
        t[rank] = _best(lambda: c.propagate(wl.Pulse(E0=1e-3), 100, 0.2, tg.LOWRANK))
        c.close()
    print({k: round(v * 1e6, 1) for k, v in t.items()})
    assert max(t[1], t[2]) < 1.5 * t[16], t


def test_apply_of_a_low_rank_not_slower_than_of_four_times_the_rank():
    """N = 20736: the rules by N r may not send a low rank of a large model to a kernel for small
    models."""
    p = wl.small_model(36, 2)
    c, t = ctc._ctx(p), {}
    x = torch.randn(p.N, dtype=torch.complex64, device="cuda")
    y = torch.empty_like(x)
    for rank in (3, 12):
        U, S, V, d = wl.random_factors(p.N, rank, seed=rank)
        tg.tdagw_set_factors(c.h, U, S, V, d)
        t[rank] = _best(lambda: [tg.tdagw_apply(c.h, tg.LOWRANK, x, y) for _ in range(50)])
    c.close()
    print({k: round(v * 2e4, 1) for k, v in t.items()})
    assert t[3] < 1.1 * t[12], t


@pytest.mark.parametrize("L,nc,rank", [(13, 2, 24), (27, 1, 22), (28, 1, 20), (14, 2, 20)])
def test_apply_on_both_sides_of_the_cluster_kernels_largest_model(L, nc, rank):
    """N = 2704, 2916 | 3136, 3136 (the line is 3072), N rank within its bound on both sides; bound as
    in the tests of the application's edges."""
    import test_gpu_apply_edges as edges
    edges.test_apply_lowrank_edges(L, nc, rank, tg.C64, 1e-6)
