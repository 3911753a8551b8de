"""The work that a user of this framework has it do, as measurable cases.

Every case goes through the public entry points of `paper_2502_05635_gb300` (the names of
the C ABI): kernel applications, propagations of one trajectory, batched propagations,
value and gradients of a batch, spectra of recorded currents.  Model sizes, ranks, batch
sizes and pulse distributions are those of this repository's workloads; runs are shortened
to a few dozen steps with pulses that peak inside them (t0 = 6, sigma 1.5 - 3), because the
cost of a step does not depend on the step.

Kinds of cases and what `run` returns:
  apply    y = K x on device vectors: y
  single   one trajectory from equilibrium: the observables (P, J, occupation per step) and,
           with "state", the final density matrix that a user saves to resume
  batch    B trajectories of different pulses and lengths in one launch: their observables
  adjoint  checkpointed batch, then gradients with respect to every field sample and to the
           pulse parameters: observables and both gradients
  hhg      spectra of recorded currents (host arrays in and out)
A complex64 context computes in 32 bits and hands its observables out widened; they are
returned here in 32 bits, the type they were computed in.  complex128 contexts and spectra
stay in 64 bits.

Low-rank factors are seeded Gaussian columns of norm about one with geometrically decaying
singular values (the recipe of the repository's large-size parity runs), Hermitian like the
kernel they stand for (V = U up to signs); channel-wise factors likewise per channel, with
the dense diagonal channels of the built kernel.  All factors are exact in 32 bits, so a
64-bit evaluation works on the same numbers.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

import paper_2502_05635_gb300 as tg

DT = 0.2
MODES = {"full": tg.FULL, "lowrank": tg.LOWRANK, "channel": tg.CHANNEL}


# ------------------------------------------------------------------ the cases ----------

def listed():
    return [
        # one K~ x inside a user's own iterative solver, smallest model: launch latency
        dict(name="apply_lowrank_l12", kind="apply", mode="lowrank", L=12, copies=1, rank=29),
        # the parity workload (12 x 12, dense kernel), a tenth of its length
        dict(name="full_l12", kind="single", mode="full", L=12, copies=1, rank=0, steps=200),
        # an ordinary single run at about the field sweep's size, odd grid and odd rank
        dict(name="lowrank_l23_odd", kind="single", mode="lowrank", L=23, copies=1, rank=235, steps=150),
        # the benchmark: MoS2-size model at rank 1024, state saved to resume
        dict(name="lowrank_l36", kind="single", mode="lowrank", L=36, copies=2, rank=1024, steps=60, state=True),
        # the same size with the channel-wise kernel (rank 5 % of Nk)
        dict(name="channel_l36", kind="single", mode="channel", L=36, copies=2, rank=65, steps=60),
        # the same size with the full dense kernel
        dict(name="full_l36", kind="single", mode="full", L=36, copies=2, rank=0, steps=12),
        # a validation run in double precision, odd four-band grid
        dict(name="lowrank_l17_c128", kind="single", mode="lowrank", L=17, copies=2, rank=231, steps=40, c128=True,
             state=True),
        # the field sweep: 256 pulses of uneven length in one launch, FP32 factors
        dict(name="sweep_l24", kind="batch", mode="lowrank", L=24, copies=1, rank=256, B=256, steps_lo=20,
             steps_hi=160),
        # the precision study: largest model, split-FP16 factors
        dict(name="precision_l48_split", kind="batch", mode="lowrank", L=48, copies=2, rank=2048, B=64, steps_lo=12,
             steps_hi=12, split=True),
        # channel-wise kernel, 64 pulses in one launch, split-FP16 segments
        dict(name="channel_l36_b64_split", kind="batch", mode="channel", L=36, copies=2, rank=65, B=64, steps_lo=30,
             steps_hi=30, split=True),
        # pulse optimisation: value and gradients of 32 trajectories
        dict(name="adjoint_l36", kind="adjoint", mode="lowrank", L=36, copies=1, rank=512, B=32, steps_lo=40,
             steps_hi=49),
        # spectra of an angle sweep's currents
        dict(name="hhg_b60", kind="hhg", B=60, steps_lo=2000, steps_hi=2000, nfreq=512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _steps_for(rng, per_step, cap, lo, hi):
    """A step count in [lo, hi], spread over its logarithm, of at most cap work in all."""
    return max(lo, min(_log(rng, lo, hi), int(cap / max(per_step, 1.0))))


def draw(rng):
    kind = rng.choice(["apply", "single", "single", "single", "batch", "batch", "batch", "adjoint", "hhg"])
    if kind == "hhg":
        s = _log(rng, 200, 2000)
        return dict(kind="hhg", B=_log(rng, 1, 60), steps_lo=max(1, s // 2), steps_hi=s, nfreq=_log(rng, 33, 512))
    copies = rng.choice([1, 2])
    if kind in ("apply", "single"):
        L = _log(rng, 6, 36)
        N, Nk = 4 * copies * copies * L * L, L * L
        mode = rng.choice(["full", "lowrank", "channel"])
        c = dict(kind=kind, mode=mode, L=L, copies=copies, rank=_rank(rng, mode, N, Nk))
        if kind == "single":
            c128 = rng.random() < 0.25 and N <= 5000
            per = _stage_bytes(c) * 4 * (4 if c128 else 1)
            c["steps"] = _steps_for(rng, per + 4 * 2e7, 5e10, 8, 200)
            c["state"] = rng.random() < 0.3
            if c128:
                c["c128"] = True
        return c
    L = _log(rng, 6, 24) if copies == 1 else _log(rng, 6, 20)
    N, Nk = 4 * copies * copies * L * L, L * L
    B = _log(rng, 2, 256)
    if kind == "adjoint":
        c = dict(kind=kind, mode="lowrank", L=L, copies=copies, rank=_rank(rng, "lowrank", N, Nk), B=min(B, 64))
        if rng.random() < 0.3:
            c["split"] = True
        hi = _steps_for(rng, 3 * 4 * _stage_flops(c) * c["B"], 3e11, 8, 64)
    else:
        mode = rng.choice(["lowrank", "lowrank", "channel", "full"])
        c = dict(kind=kind, mode=mode, L=L, copies=copies, rank=_rank(rng, mode, N, Nk), B=B)
        if mode != "full" and rng.random() < 0.5:
            c["split"] = True
        hi = _steps_for(rng, 4 * _stage_flops(c) * B, 3e11, 8, 160)
    c["steps_hi"] = hi
    c["steps_lo"] = max(1, hi // 4) if rng.random() < 0.7 else hi
    return c


def _rank(rng, mode, N, Nk):
    if mode == "full":
        return 0
    if mode == "channel":
        return max(1, min(Nk, int(rng.uniform(0.03, 0.12) * Nk)))
    return max(2, min(1024, int(rng.uniform(0.03, 0.15) * N)))


# ------------------------------------------------------------------ inputs -------------

def _params(case):
    return types.SimpleNamespace(L=case["L"], nb_copies=case["copies"],
                                 offsets=(0.0, 0.03, 0.0, 0.0) if case["copies"] == 2 else (0.0,) * 4,
                                 Delta=0.08, t=0.05, m=0.1, a=6.0, r0=20.0)


def _sizes(case):
    Nb, Nk = 2 * case["copies"], case["L"] ** 2
    return Nb, Nk, Nb * Nb * Nk


def _generator(seed, what):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + what)
    return g


def _gauss(shape, g, scale):
    """complex64 Gaussian entries with E|z|^2 = 2 scale^2, on the GPU."""
    z = torch.randn(tuple(shape) + (2,), generator=g, device="cuda", dtype=torch.float32)
    return torch.view_as_complex(z.mul_(scale))


def _lowrank(case, seed):
    """U, S, V, diag on the GPU (complex64 / float32): U of column norm about one, V = U with
    random column signs (mostly attractive, like the kernel), S from 0.05 down by e^-3."""
    _, _, N = _sizes(case)
    r = case["rank"]
    g = _generator(seed, 1)
    U = _gauss((N, r), g, 1.0 / math.sqrt(2 * N))
    sgn = torch.where(torch.rand(r, generator=g, device="cuda") < 0.85, -1.0, 1.0)
    S = (0.05 * torch.exp(-3.0 * torch.arange(r, device="cuda", dtype=torch.float64) / r)).float()
    diag = torch.full((N,), -0.0134, device="cuda", dtype=torch.float32).to(torch.complex64)
    return U, S, U * sgn, diag


def _channel_pairs(case):
    """Off-diagonal channels (p, q), p < q, that do not vanish: the bands alternate between the
    copies, and a kernel entry needs n1, n3 and n2, n4 in the same copy."""
    Nb = 2 * case["copies"]
    P = Nb * Nb
    c = (lambda n: n % 2) if case["copies"] == 2 else (lambda n: 0)
    return [(p, q) for p in range(P) for q in range(p + 1, P)
            if c(p // Nb) == c(q // Nb) and c(p % Nb) == c(q % Nb)]


def _channels(case, seed):
    """Per nonvanishing channel p -> q, p < q: U, V (Nk x z) and S; q -> p is its adjoint."""
    _, Nk, _ = _sizes(case)
    z = case["rank"]
    pairs = _channel_pairs(case)
    g = _generator(seed, 2)
    U = _gauss((len(pairs), Nk, z), g, 1.0 / math.sqrt(2 * Nk))
    V = _gauss((len(pairs), Nk, z), g, 1.0 / math.sqrt(2 * Nk))
    S = (0.02 * torch.exp(-4.0 * torch.arange(z, device="cuda", dtype=torch.float64) / z)).float()
    return pairs, U, S, V


def _pulses(case, seed):
    """Seeded pulses and lengths: amplitudes 1e-4 .. 1e-2 (log-uniform), frequencies 0.06 - 0.16,
    directions over the plane, peaking within the first 12 time units."""
    B = case.get("B", 1)
    rng = np.random.default_rng([int(seed), 3])
    E0 = 10.0 ** rng.uniform(-4.0, -2.0, B)
    om, sg, an = rng.uniform(0.06, 0.16, B), rng.uniform(1.5, 3.0, B), rng.uniform(0.0, np.pi, B)
    ps = [types.SimpleNamespace(kind=tg.FIELD_GAUSS_COS, E0=float(E0[b]), omega=float(om[b]), t0=6.0,
                                sigma=float(sg[b]), T_pulse=0.0, dir_x=float(np.cos(an[b])),
                                dir_y=float(np.sin(an[b]))) for b in range(B)]
    if "steps" in case:
        return ps, [case["steps"]]
    st = rng.integers(case["steps_lo"], case["steps_hi"] + 1, B)
    st[int(rng.integers(B))] = case["steps_hi"]
    return ps, [int(s) for s in st]


def _objective(case, seed):
    """dJ/d(observables) of a user's objective, (steps + 1) x B x 3."""
    rng = np.random.default_rng([int(seed), 4])
    return rng.standard_normal((case["steps_hi"] + 1, case["B"], 3))


def _vector(case, seed):
    _, _, N = _sizes(case)
    return _gauss((N,), _generator(seed, 5), 1e-2)


def _currents(case, seed):
    """Recorded observables of B driven trajectories (rows x B x 3, J in column 1): a few
    harmonics of the drive under its envelope, NaN after each trajectory's end."""
    rng = np.random.default_rng([int(seed), 6])
    rows, B = case["steps_hi"] + 1, case["B"]
    st = rng.integers(case["steps_lo"], case["steps_hi"] + 1, B).astype(np.int32)
    st[0] = case["steps_hi"]
    t = DT * np.arange(rows)
    env = np.sin(np.pi * np.arange(rows) / rows) ** 2
    obs = np.zeros((rows, B, 3))
    for b in range(B):
        for h, a in ((1, 1.0), (3, 1e-2), (5, 1e-4)):
            obs[:, b, 1] += a * env * np.sin(0.1 * h * t + rng.uniform(0, 2 * np.pi))
        obs[:, b, 0] = rng.standard_normal(rows)
        obs[st[b] + 1:, b] = np.nan
    w = 0.1 * np.linspace(0.3, 9.0, case["nfreq"]) * rng.uniform(0.95, 1.05)
    return obs, st, w


def prepare(case, seed):
    if case["kind"] == "hhg":
        obs, st, w = _currents(case, seed)
        return dict(case=case, obs=obs, steps=st, omega=w)
    ctx = tg.Context(_params(case), tg.C128 if case.get("c128") else tg.C64,
                     stream=torch.cuda.current_stream().cuda_stream)
    if case["mode"] == "lowrank":
        U, S, V, d = _lowrank(case, seed)
        host = [t.to(torch.complex128).cpu().numpy() for t in (U, V, d)]
        tg.tdagw_set_factors(ctx.h, host[0], S.double().cpu().numpy(), host[1], host[2])
    elif case["mode"] == "channel":
        Nb, Nk, _ = _sizes(case)
        P, z = Nb * Nb, case["rank"]
        pairs, U, S, V = _channels(case, seed)
        Uh, Vh = np.zeros((P, P, Nk, z), np.complex128), np.zeros((P, P, Nk, z), np.complex128)
        Sh, rk = np.zeros((P, P, z)), np.zeros((P, P), np.int32)
        Un, Vn, Sn = U.cpu().numpy(), V.cpu().numpy(), S.double().cpu().numpy()
        for e, (p, q) in enumerate(pairs):
            Uh[p, q], Vh[p, q] = Un[e], Vn[e]
            Uh[q, p], Vh[q, p] = Vn[e], Un[e]
            Sh[p, q] = Sh[q, p] = Sn
            rk[p, q] = rk[q, p] = z
        tg.tdagw_set_channel_factors(ctx.h, Uh, Sh, Vh, None, rk)
    st = dict(case=case, ctx=ctx)
    if case["kind"] == "apply":
        st["x"] = _vector(case, seed)
        st["y"] = torch.empty_like(st["x"])
        return st
    pulses, steps = _pulses(case, seed)
    st["pulses"], st["steps"] = pulses, steps
    if case["kind"] == "adjoint":
        st["dJ"] = _objective(case, seed)
    return st


# ------------------------------------------------------------------ one pass -----------

def run(st):
    case = st["case"]
    if case["kind"] == "hhg":
        return tg.tdagw_hhg_spectrum(st["obs"], st["steps"], DT, st["omega"], component=1)
    ctx, mode = st["ctx"], MODES[case["mode"]]
    if case["kind"] == "apply":
        tg.tdagw_apply(ctx.h, mode, st["x"], st["y"])
        return st["y"]
    flags = tg.FLAG_RESET | (tg.FLAG_SPLIT_F16 if case.get("split") else 0)
    if case["kind"] == "single":
        obs = ctx.propagate(st["pulses"][0], st["steps"][0], DT, mode, flags)
        out = {"obs": obs}
        if case.get("state"):
            out["drho"] = tg.tdagw_get_state(ctx.h)[0]
        if not case.get("c128"):
            out = {k: v.astype(np.complex64 if np.iscomplexobj(v) else np.float32) for k, v in out.items()}
        return out
    if case["kind"] == "batch":
        return ctx.propagate_batch(st["pulses"], st["steps"], DT, mode, flags).astype(np.float32)
    B = case["B"]
    tg.tdagw_propagate(ctx.h, [tg.make_field(p) for p in st["pulses"]], st["steps"], DT, mode,
                       flags | tg.FLAG_CHECKPOINT)
    obs = tg.tdagw_observables(ctx.h, B=B)
    dE, dp = tg.tdagw_adjoint(ctx.h, st["dJ"], case["steps_hi"], B)
    return {"obs": obs.astype(np.float32), "dJdE": dE.astype(np.float32), "dJdp": dp.astype(np.float32)}


# ------------------------------------------------------------------ unavoidable work ---

def _kernel_elems(case):
    Nb, Nk, N = _sizes(case)
    if case["mode"] == "full":
        return N * N
    if case["mode"] == "lowrank":
        return 2 * N * case["rank"] + N
    return Nb * Nb * Nk * Nk + 4 * len(_channel_pairs(case)) * Nk * case["rank"]


def _stage_bytes(case):
    return 8 * _kernel_elems(case)


def _stage_flops(case):
    """One kernel application and the Nb x Nb commutators of one trajectory."""
    Nb, Nk, _ = _sizes(case)
    return 8 * _kernel_elems(case) + 16 * Nk * Nb ** 3


def work(case):
    if case["kind"] == "hhg":
        n, f = case["B"] * (case["steps_hi"] + 1), case["nfreq"]
        return {"bytes": 8 * (n + f + f * case["B"]), "flops": 4 * n * f}
    _, _, N = _sizes(case)
    el = 16 if case.get("c128") else 8
    kernel = el * _kernel_elems(case)
    if case["kind"] == "apply":
        return {"bytes": kernel + 2 * el * N, "flops": _stage_flops(case)}
    if case["kind"] == "single":
        T = case["steps"]
        out = 24 * (T + 1) + (el * N if case.get("state") else 0)
        return {"bytes": kernel + 6 * el * N + out, "flops": 4 * T * _stage_flops(case)}
    B, T = case["B"], (case["steps_lo"] + case["steps_hi"]) / 2
    fwd = 4 * T * B * _stage_flops(case)
    out = 24 * (case["steps_hi"] + 1) * B
    if case["kind"] == "batch":
        return {"bytes": kernel + 6 * el * N + out, "flops": fwd}
    # reverse stages: the kernel's adjoint once and three commutator-like products per stage
    return {"bytes": kernel + 6 * el * N + 3 * out, "flops": 2 * fwd}


# ------------------------------------------------------------------ the same in 64 bits -

class _Model:
    """Bands, dipoles, velocity and screened interaction of the lattice model (FP64)."""

    def __init__(self, case):
        p = _params(case)
        self.Nb, self.Nk, self.N = _sizes(case)
        L, nc, Nb, Nk, a = p.L, p.nb_copies, self.Nb, self.Nk, p.a
        k = np.stack(np.divmod(np.arange(Nk), L), 1) * (2 * np.pi / L)      # k a
        hx, hy = p.t * np.sin(k[:, 0]), p.t * np.sin(k[:, 1])
        hz = p.Delta + p.m * (2 - np.cos(k[:, 0]) - np.cos(k[:, 1]))
        d = np.sqrt(hx ** 2 + hy ** 2 + hz ** 2)
        # eigenvectors of one copy (columns: lower, upper), largest component real positive
        big, off = (d + hz) / np.sqrt(2 * d * (d + hz)), (hx + 1j * hy) / np.sqrt(2 * d * (d + hz))
        u = np.empty((Nk, 2, 2), complex)
        u[:, 0, 0], u[:, 1, 0] = -off.conj(), big
        u[:, 0, 1], u[:, 1, 1] = big, off
        sx, sy, sz = (np.array(s, complex) for s in ([[0, 1], [1, 0]], [[0, -1j], [1j, 0]], [[1, 0], [0, -1]]))
        dh = [a * (p.t * np.cos(k[:, i])[:, None, None] * s + p.m * np.sin(k[:, i])[:, None, None] * sz)
              for i, s in ((0, sx), (1, sy))]
        vel = [u.conj().transpose(0, 2, 1) @ h @ u for h in dh]
        eps = np.empty((Nk, Nb))
        U, V, D = np.zeros((Nk, Nb, Nb), complex), np.zeros((Nk, Nb, Nb), complex), np.zeros((2, Nk, Nb, Nb), complex)
        e2 = np.stack([-d, d], 1)
        ec = np.concatenate([e2 + p.offsets[c] for c in range(nc)], 1)        # copy-major
        order = np.argsort(ec, axis=1, kind="stable")
        for n in range(Nb):
            cn, bn = np.divmod(order[:, n], 2)
            kk = np.arange(Nk)
            eps[:, n] = ec[kk, order[:, n]]
            for o in range(2):
                U[kk, 2 * cn + o, n] = u[kk, o, bn]
            for m in range(Nb):
                cm, bm = np.divmod(order[:, m], 2)
                same = cn == cm
                V[:, n, m] = np.where(same, vel[0][kk, bn, bm], 0)
                gap = e2[kk, bm] - e2[kk, bn]
                for i in range(2):
                    x = 1j * vel[i][kk, bn, bm] / np.where(gap == 0, 1.0, gap)
                    D[i, :, n, m] = np.where(same & (bn != bm), x, 0)
        gx, gw = np.polynomial.legendre.leggauss(64)
        th = np.pi / 8 * (gx + 1)
        A, h = Nk * a * a, np.pi / (L * a)
        w0 = 8 * 2 * np.pi / (A * p.r0) * np.sum(np.pi / 8 * gw * np.log1p(p.r0 * h / np.cos(th))) / (4 * h * h)
        i = np.arange(L)
        i = np.where(i >= (L + 1) // 2, i - L, i)
        q = 2 * np.pi / (L * a) * np.hypot(i[:, None], i[None, :])
        with np.errstate(divide="ignore"):
            W = 2 * np.pi / (A * q * (1 + p.r0 * q))
        W[0, 0] = w0
        ii, jj = np.divmod(np.arange(Nk), L)
        self.W = torch.from_numpy(W[(ii[:, None] - ii) % L, (jj[:, None] - jj) % L]).cuda()
        self.U, self.vx, self.dx, self.dy = (torch.from_numpy(x).cuda() for x in (U, V, D[0], D[1]))
        self.gap = torch.from_numpy(eps[:, :, None] - eps[:, None, :]).cuda()
        self.occ = torch.tensor([1.0] * (Nb // 2) + [0.0] * (Nb // 2), dtype=torch.float64, device="cuda")

    def overlaps(self):
        """O[k, k', n, n'] = (U_k^+ U_k')_{n n'}"""
        return torch.einsum("kon,lop->klnp", self.U.conj(), self.U)

    def dense(self):
        O = self.overlaps()
        Nk, Nb = self.Nk, self.Nb
        K = torch.empty((Nk, Nb, Nb, Nk, Nb, Nb), dtype=torch.complex128, device="cuda")
        for n in range(Nb):
            for m in range(Nb):
                x = O[:, :, n, :, None] * O[:, :, m, None, :].conj()
                K[:, n, m] = -self.W[:, :, None, None] * x
        return K.reshape(self.N, self.N)

    def diagonal_channels(self):
        O = self.overlaps()
        on = torch.diagonal(O, dim1=2, dim2=3)                                 # k, k', n
        D = -self.W[:, :, None, None] * on[:, :, :, None] * on[:, :, None, :].conj()
        return D.permute(2, 3, 0, 1).reshape(self.Nb ** 2, self.Nk, self.Nk)


def _apply64(case, seed, mdl):
    """X (N x B, complex128) -> K X, plain torch."""
    if case["mode"] == "full":
        K = mdl.dense()
        return lambda X: K @ X
    if case["mode"] == "lowrank":
        U, S, V, d = (t.to(torch.complex128) for t in _lowrank(case, seed))
        return lambda X: d[:, None] * X + U @ (S[:, None] * (V.conj().T @ X))
    pairs, U, S, V = _channels(case, seed)
    U, S, V = U.to(torch.complex128), S.to(torch.complex128), V.to(torch.complex128)
    D, P, Nk = mdl.diagonal_channels(), mdl.Nb ** 2, mdl.Nk
    ps, qs = (torch.tensor([x[i] for x in pairs], device="cuda") for i in (0, 1))

    def apply(X):
        Xp = X.reshape(Nk, P, -1).transpose(0, 1)
        Y = D @ Xp
        Y = Y.index_add(0, ps, U @ (S[:, None] * (V.mH @ Xp[qs])))
        Y = Y.index_add(0, qs, V @ (S[:, None] * (U.mH @ Xp[ps])))
        return Y.transpose(0, 1).reshape(X.shape)

    return apply


def _fields64(pulses, T, params=None):
    """E(j DT / 2) of every pulse, (2 T + 1) x B; params (B x 4: E0, omega, t0, sigma) if given."""
    if params is None:
        params = torch.tensor([[p.E0, p.omega, p.t0, p.sigma] for p in pulses], dtype=torch.float64, device="cuda")
    t = 0.5 * DT * torch.arange(2 * T + 1, dtype=torch.float64, device="cuda")[:, None]
    E0, om, t0, sg = params.unbind(1)
    return E0 * torch.exp(-((t - t0) ** 2) / (2 * sg ** 2)) * torch.cos(om * t)


def _rk4(mdl, apply, E, pulses, T):
    """Observables ((T + 1) x B x 3) and the final state of classical RK4 from equilibrium."""
    Nk, Nb, B = mdl.Nk, mdl.Nb, len(pulses)
    dirs = torch.tensor([[p.dir_x, p.dir_y] for p in pulses], dtype=torch.complex128, device="cuda")
    dip = dirs[:, 0, None, None, None] * mdl.dx + dirs[:, 1, None, None, None] * mdl.dy    # B, Nk, Nb, Nb
    rho0 = torch.diag(mdl.occ).to(torch.complex128)

    def f(j, X):
        Xk = X.T.reshape(B, Nk, Nb, Nb)
        M = apply(X).T.reshape(B, Nk, Nb, Nb) + E[j].to(torch.complex128)[:, None, None, None] * dip
        rho = Xk + rho0
        return (-1j * (mdl.gap * Xk + M @ rho - rho @ M)).reshape(B, -1).T

    def obs(X):
        rho = X.T.reshape(B, Nk, Nb, Nb) + rho0
        P = (rho * mdl.dx.conj()).real.sum((1, 2, 3)) / Nk
        J = (rho * mdl.vx.conj()).real.sum((1, 2, 3)) / Nk
        return torch.stack([P, J, rho[:, :, Nb // 2, Nb // 2].real.mean(1)], 1)

    x = torch.zeros((mdl.N, B), dtype=torch.complex128, device="cuda")
    rec = [obs(x)]
    for n in range(T):
        k1 = f(2 * n, x)
        k2 = f(2 * n + 1, x + 0.5 * DT * k1)
        k3 = f(2 * n + 1, x + 0.5 * DT * k2)
        k4 = f(2 * n + 2, x + DT * k3)
        x = x + DT / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
        rec.append(obs(x))
    return torch.stack(rec), x


def exact(case, seed):
    if case["kind"] == "hhg":
        obs, st, w = _currents(case, seed)
        J = torch.from_numpy(np.nan_to_num(obs[:, :, 1])).cuda().to(torch.complex128)
        t = DT * torch.arange(J.shape[0], dtype=torch.float64, device="cuda")
        om = torch.from_numpy(w).cuda()
        F = torch.polar(torch.ones((), dtype=torch.float64, device="cuda"), -om[:, None] * t) @ J
        return ((om[:, None] * DT) ** 2 * F.abs() ** 2).cpu().numpy()
    mdl = _Model(case)
    apply = _apply64(case, seed, mdl)
    if case["kind"] == "apply":
        return apply(_vector(case, seed).to(torch.complex128)[:, None])[:, 0]
    pulses, steps = _pulses(case, seed)
    T = max(steps)
    if case["kind"] != "adjoint":
        rec, x = _rk4(mdl, apply, _fields64(pulses, T), pulses, T)
        if case["kind"] == "single":
            out = {"obs": rec[:, 0].cpu().numpy()}
            if case.get("state"):
                out["drho"] = x[:, 0].cpu().numpy()
            return out
        return _ended(rec, steps).cpu().numpy()
    par = torch.tensor([[p.E0, p.omega, p.t0, p.sigma] for p in pulses], dtype=torch.float64, device="cuda",
                       requires_grad=True)
    E = _fields64(pulses, T, par)
    leaf = E.detach().requires_grad_(True)
    rec, _ = _rk4(mdl, apply, leaf, pulses, T)
    dJ = torch.from_numpy(_objective(case, seed)).cuda()
    for b, s in enumerate(steps):
        dJ[s + 1:, b] = 0
    rec.backward(dJ)
    E.backward(leaf.grad)
    return {"obs": _ended(rec.detach(), steps).cpu().numpy(), "dJdE": leaf.grad.cpu().numpy(),
            "dJdp": par.grad.cpu().numpy()}


def _ended(rec, steps):
    """NaN after each trajectory's last step."""
    rec = rec.clone()
    for b, s in enumerate(steps):
        rec[s + 1:, b] = float("nan")
    return rec
