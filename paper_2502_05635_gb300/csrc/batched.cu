// Batched TD-aGW propagation: B trajectories (different pulses and lengths) in one
// persistent cooperative launch (complex64).  Across trajectories the contraction of Eq.
// sigma-from-k becomes a matrix product: with the states as columns of X (N x B),
//   low rank (Eq. svd_acc):  Y = S o (V^H X)  (r x B),   dSigma = K^diag o X + U Y
//   dense:                   dSigma = K X
// followed by the per-k commutator and RK4 stage update of Eq. tdagw for every column.
//
// Work split: CTA (rg, tg) owns the pair elements of a k-aligned row group rg and the
// trajectories of group tg; trajectories are sorted by length (longest first), so the
// active ones at step n are a prefix of length B_act(n) and each group takes an equal
// share of that prefix -- finished trajectories cost nothing (compaction by sorting); the
// numbers of row and trajectory groups follow the active count (step_plan).
// Per low-rank stage:
//   A  P[rg] = V[rows(rg)]^H X[rows(rg), tg]        (partial over the row group)
//   -- grid barrier --
//   C  Y[j, tg] = S_j sum_rg P[rg][j, tg]            (each CTA: a slice of j)
//   -- grid barrier --
//   D  dSigma[rows(rg), tg] = U[rows(rg)] Y[:, tg] + K^diag o X
//   E  commutator + RK4 for k in rg, trajectories in tg (rows this CTA just computed)
// Dense stages: grid barrier (X complete), dSigma[rows(rg), tg] = K[rows(rg)] X[:, tg], E.
// The matrix products are register-tiled (8 x 4 complex outputs per thread) FP32 FMAs
// through shared memory (block_gemm).  Grid barriers are bounded waits (as in the single-trajectory
// persistent kernel); on expiry the kernel sets an error word and returns.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "batched_common.cuh"

namespace tdagw {

using namespace batched;

namespace {

// Commutator + RK4 stage update of one (k, trajectory) block, all NB^2 elements in
// registers (the same arithmetic as stage_element, Eq. tdagw).  The observables (last
// stage) are added to ob in double-float (FP64 arithmetic is slow on this GPU).
template <int NB>
__device__ void stage_kb(const BatchArgs& a, int k, int b, int st, float E, float2 dr, ObsDF& ob) {
    constexpr int NB2 = NB * NB;
    const int64_t Bp = a.Bp;
    float2 X[NB2], M[NB2];
#pragma unroll
    for (int g = 0; g < NB2; ++g) {
        const int64_t i = (int64_t)k * NB2 + g;
        X[g] = __ldcg(a.X + i * Bp + b);
        const float2 d1 = a.dx[i], d2 = a.dy[i];
        const float2 ds = __ldcg(a.dS + i * Bp + b);
        M[g] = make_float2(ds.x + E * (dr.x * d1.x + dr.y * d2.x), ds.y + E * (dr.x * d1.y + dr.y * d2.y));
    }
#pragma unroll
    for (int n = 0; n < NB; ++n)
#pragma unroll
        for (int m = 0; m < NB; ++m) {
            const int g = n * NB + m;
            const int64_t i = (int64_t)k * NB2 + g;
            float2 comm = cscale(M[g], a.occ[m] - a.occ[n]);
#pragma unroll
            for (int l = 0; l < NB; ++l) {
                comm = cfma(M[n * NB + l], X[l * NB + m], comm);
                comm = csub(comm, cmul(X[n * NB + l], M[l * NB + m]));
            }
            const float2 h0 = gap_times(a.gap[i], X[g]);
            const float2 s = cadd(h0, comm);
            const float2 kv = make_float2(s.y, -s.x);
            const int64_t e = i * Bp + b;
            const float2 xs = __ldcg(a.Ssum + e), xc = __ldcg(a.Ccomp + e);
            float2 Xn;
            if (st < 3) {
                const float2 ac = st == 0 ? kv : cadd(__ldcg(a.acc + e), cscale(kv, 2.f));
                a.acc[e] = ac;
                const float cn = st == 2 ? a.dt : 0.5f * a.dt;
                Xn = cadd(xs, cadd(xc, cscale(kv, cn)));
            } else {
                const float2 ac = cadd(__ldcg(a.acc + e), kv);
                const float2 inc = cscale(ac, a.dt / 6.f);
                float2 ns, nc;
                if (a.kahan) {
                    float ex, ey;
                    ns.x = two_sum(xs.x, inc.x, ex);
                    ns.y = two_sum(xs.y, inc.y, ey);
                    nc = make_float2(xc.x + ex, xc.y + ey);
                } else {
                    ns = cadd(xs, inc);
                    nc = xc;
                }
                a.Ssum[e] = ns;
                a.Ccomp[e] = nc;
                Xn = cadd(ns, nc);
                const float2 rho = (n == m) ? make_float2(Xn.x + a.occ[n], Xn.y) : Xn;
                const float2 d1 = a.dx[i], v1 = a.vx[i];
                ob.p.add_prod(rho.x, d1.x);
                ob.p.add_prod(rho.y, d1.y);
                ob.j.add_prod(rho.x, v1.x);
                ob.j.add_prod(rho.y, v1.y);
                if (n == m && n == a.c1) ob.o.add(rho.x);
            }
            a.X[e] = Xn;
        }
}

// A: partial V^H X over this row group (channel-wise: one product per input pair q, its V
// segment's rows of this row group with the rows k P + q of X)
template <int NB, bool CH>
__device__ __noinline__ void phase_vhx() {
    BatchShared& bs = batch_shared();
    const BatchArgs& a = bs.a;
    const StepShared& sh = bs.s;
    constexpr int NB2 = NB * NB;
    if constexpr (!CH) {
        const int64_t ra = (int64_t)sh.ka * NB2;
        if (sh.nb > 0)
            block_gemm<true>(a.V + ra * a.ldu, a.ldu, a.r, sh.nrows, a.X + ra * a.Bp + sh.b0, a.Bp, sh.nb,
                             a.P + (int64_t)blockIdx.x * a.r * kTileB, kTileB, false, nullptr, nullptr);
    } else if (sh.nb > 0) {
        // channel-wise: q-major row shares as in D below (rows q Nk + k' of the
        // V segments, one or two input pairs per row group); the group writes the
        // partials of those pairs' columns only
        for (int q = sh.u0 / a.Nk; q < NB2 && q * a.Nk < sh.u1; ++q) {
            const int ldv = a.chm->ldv[q];
            const int k0 = max(sh.u0 - q * a.Nk, 0), k1 = min(sh.u1 - q * a.Nk, a.Nk);
            if (ldv == 0 || k1 <= k0) continue;
            block_gemm<true>(a.Vch + a.chm->vbase[q] + (int64_t)k0 * ldv, ldv, ldv, k1 - k0,
                             a.X + ((int64_t)k0 * NB2 + q) * a.Bp + sh.b0, (int64_t)NB2 * a.Bp, sh.nb,
                             a.P + ((int64_t)blockIdx.x * a.r + a.chm->sbase[q]) * kTileB, kTileB, false,
                             nullptr, nullptr);
        }
    }
}

// C: Y[j][b] = S_j sum over row groups, j in this CTA's slice (channel-wise: over the row
// groups whose share touches the input pair of column j)
template <int NB, bool CH>
__device__ __noinline__ void phase_sy() {
    BatchShared& bs = batch_shared();
    const BatchArgs& a = bs.a;
    const StepShared& sh = bs.s;
    constexpr int NB2 = NB * NB;
    if (sh.nb > 0) {
        const int Rg = sh.Rg;
        auto range = [&](int j, int& g0, int& g1) {
            g0 = 0;
            g1 = Rg - 1;
            if constexpr (CH) {
                int q = 0;
                while (q + 1 < NB2 && a.chm->sbase[q + 1] <= j) ++q;
                const int64_t NR = a.N, RG = Rg, lo = (int64_t)q * a.Nk;
                g0 = max(0, (int)(((lo + 1) * RG + NR - 1) / NR) - 1);
                g1 = min(Rg - 1, (int)(((lo + a.Nk) * RG + NR - 1) / NR) - 1);
            }
        };
        // partials of the row groups of this trajectory group
        reduce_partials(a.P + (int64_t)sh.tg * Rg * a.r * kTileB, (int64_t)a.r * kTileB, sh.jr0, sh.jr1,
                        sh.nb, a.S, a.Y + sh.b0, a.Bp, range, reinterpret_cast<float2*>(bs.obs));
    }
}

template <int NB, bool CH>
__device__ __noinline__ void phase_uy() {
    BatchShared& bs = batch_shared();
    const BatchArgs& a = bs.a;
    const StepShared& sh = bs.s;
    constexpr int NB2 = NB * NB;
    if constexpr (!CH) {
        // D: dSigma = U Y + K^diag X for this row group (the strict diagonal fused
        // into the product, or the k = k' blocks added after it)
        const int64_t ra = (int64_t)sh.ka * NB2, x0 = ra * a.Bp + sh.b0;
        if (sh.nb > 0)
            block_gemm<false>(a.U + ra * a.ldu, a.ldu, sh.nrows, a.r, a.Y + sh.b0, a.Bp, sh.nb, a.dS + x0,
                              a.Bp, false, a.kblk ? nullptr : a.diag + ra, a.X + x0);
        if (a.kblk) {
            __syncthreads();  // this CTA's U Y rows are written
            if (sh.nb > 0)
                kblock_term<NB, false>(a.kblk, a.X, a.dS, a.Bp, (int64_t)sh.ka * NB2, sh.nrows, sh.b0, sh.nb);
        }
    } else {
        // D (channel-wise) by p-major shares: row group rg takes the rows
        // [u0, u1) of the order p Nk + k (one or two output pairs), so each pair
        // is one product over many k-points instead of the group's few: the dense
        // diagonal channel with x_p over all k, then each off-diagonal channel's
        // U^pq with its block of S o Y added.  The rows reach their k-point's
        // owner through global memory across the barrier below.
        const int64_t ldo = (int64_t)NB2 * a.Bp;
        if (sh.nb > 0)
            for (int p = sh.u0 / a.Nk; p < NB2 && p * a.Nk < sh.u1; ++p) {
                const int k0 = max(sh.u0 - p * a.Nk, 0), k1 = min(sh.u1 - p * a.Nk, a.Nk);
                if (k1 <= k0) continue;
                const int ldw = a.chm->ldw[p];
                const float2* Ub = a.Uch + a.chm->ubase[p] + (int64_t)k0 * ldw;
                float2* o = a.dS + ((int64_t)k0 * NB2 + p) * a.Bp + sh.b0;
                block_gemm<false>(Ub + a.chm->nlr[p], ldw, k1 - k0, a.Nk, a.X + (int64_t)p * a.Bp + sh.b0,
                                  ldo, sh.nb, o, ldo, false, nullptr, nullptr);
                for (int q = 0; q < NB2; ++q) {
                    const int z = a.choff[2 * NB2 * NB2 + p * NB2 + q];
                    if (q == p || z == 0) continue;
                    const int64_t yrow = a.chm->sbase[q] + a.choff[NB2 * NB2 + q * NB2 + p];
                    block_gemm<false>(Ub + a.choff[p * NB2 + q], ldw, k1 - k0, z,
                                      a.Y + yrow * a.Bp + sh.b0, a.Bp, sh.nb, o, ldo, true, nullptr,
                                      nullptr);
                }
            }
    }
}

// dense mode: dSigma rows of this row group
template <int NB>
__device__ __noinline__ void phase_dense() {
    BatchShared& bs = batch_shared();
    const BatchArgs& a = bs.a;
    const StepShared& sh = bs.s;
    constexpr int NB2 = NB * NB;
    const int64_t ra = (int64_t)sh.ka * NB2;
    if (sh.nb > 0)
        block_gemm<false>(a.K + ra * a.N, a.N, sh.nrows, (int)a.N, a.X + sh.b0, a.Bp, sh.nb,
                          a.dS + ra * a.Bp + sh.b0, a.Bp, false, nullptr, nullptr);
}

// Records, commutator + RK4 stage update and observables partials of this CTA's block (k in
// [ka, kb), trajectories [b0, b0 + nb)), stage gs of the launch.
template <int NB>
__device__ __forceinline__ void epilogue(const BatchArgs& a, BatchShared& bs, int gs) {
    constexpr int NB2 = NB * NB;
    volatile StepShared& sh = bs.s;
    const int tid = threadIdx.x, n = gs >> 2, st = gs & 3;
    const int nb = sh.nb, b0 = sh.b0, ka = sh.ka, kb = sh.kb;
    if (a.recX) {
        // stage input and dSigma of this stage, for the adjoint's backward sweep
        const int64_t slot = (int64_t)(n * 4 + st) * a.N * a.Bp, ra = (int64_t)ka * NB2;
        for (int e = threadIdx.x; e < (kb - ka) * NB2 * nb; e += kBThreads) {
            const int64_t off = (ra + e / nb) * a.Bp + b0 + e % nb;
            a.recX[slot + off] = __ldcg(a.X + off);
            a.recDS[slot + off] = __ldcg(a.dS + off);
        }
    }
    // E: commutator + RK4 for (k in [ka, kb), b in [b0, b1))
    const int eoff = st == 0 ? 0 : (st == 3 ? 2 : 1);
    {
        const int bl = tid % kTileB, kg = tid / kTileB;  // 16 k-groups x 32 trajectories
        ObsDF ob;
        if (bl < nb) {
            const int b = b0 + bl;
            const float E = (float)a.Etab[(int64_t)b * a.ldE + 2 * (a.n0 + n) + eoff];
            const float2 dr = a.dir[b];
            for (int k = ka + kg; k < kb; k += kBThreads / kTileB) stage_kb<NB>(a, k, b, st, E, dr, ob);
        }
        if (st == 3) {
            bs.obs[(kg * kTileB + bl) * 3] = ob.p.value();
            bs.obs[(kg * kTileB + bl) * 3 + 1] = ob.j.value();
            bs.obs[(kg * kTileB + bl) * 3 + 2] = ob.o.value();
        }
    }
    __syncthreads();
    if (st == 3)
        for (int bl = tid; bl < nb; bl += kBThreads) {
            double s0 = 0.0, s1 = 0.0, s2 = 0.0;
            for (int kg = 0; kg < kBThreads / kTileB; ++kg) {
                s0 += bs.obs[(kg * kTileB + bl) * 3];
                s1 += bs.obs[(kg * kTileB + bl) * 3 + 1];
                s2 += bs.obs[(kg * kTileB + bl) * 3 + 2];
            }
            double* rr = a.red + ((int64_t)sh.rg * a.Bp + b0 + bl) * 3;
            rr[0] = s0;
            rr[1] = s1;
            rr[2] = s2;
        }
    __syncthreads();
}

// CH: the channel-wise mode (a separate instantiation, so the other modes' code is unchanged)
template <int NB, bool CH>
__global__ void __launch_bounds__(kBThreads, 1) batched_kernel(BatchArgs a) {
    BatchShared& bs = batch_shared();
    volatile StepShared& sh = bs.s;
    const int tid = threadIdx.x;
    constexpr int NB2 = NB * NB;
    if (tid == 0) {
        bs.abort_s = 0;
        bs.gen = 0;
        bs.n = 0;
        sh.Bact = -1;
    }
    copy_args(bs.a, a);
    __syncthreads();
    // observables of step n - 1's end (row n), from the split of that step
    auto last_observables = [&](int n) {
        const StepPlan pp = step_plan(a.act[a.n0 + n - 1], gridDim.x, a.Nk);
        if (blockIdx.x / pp.Rg < (unsigned)pp.Tg)
            reduce_observables_row(a, n, pp, blockIdx.x / pp.Rg, blockIdx.x % pp.Rg);
    };
    // stage counter (4 step + stage), read from shared memory so that no register holds it
    // across the calls
    volatile int& gs = bs.n;
    while (gs < 4 * a.Tmax) {
        const int n = gs >> 2, st = gs & 3;
        if (st == 0) {
            // this step's block of the split
            if (tid == 0) {
                bs.prev_act = sh.Bact;
                set_step(a, a.act[a.n0 + n], NB2, sh);
            }
            __syncthreads();
        }
        // the dense product and the channel-wise row shares read every CTA's rows of X
        const bool need_x_barrier = (a.mode == TDAGW_FULL || CH) ? !(n == 0 && st == 0)
                                                                 : (st == 0 && sh.Bact != *(volatile int*)&bs.prev_act && n > 0);
        if (need_x_barrier && !bgrid_sync(a, bs)) return;
        if (st == 0 && a.ckS && (a.n0 + n) % a.ck_period == 0) {
            // checkpoint of the compensated state at the start of step n0 + n (own block,
            // complete: a barrier precedes every change of the split)
            const int64_t slot = (int64_t)((a.n0 + n) / a.ck_period) * a.N * a.Bp;
            const int nb = sh.nb, b0 = sh.b0, nrows = sh.nrows;
            const int64_t ra = (int64_t)sh.ka * NB2;
            for (int e = threadIdx.x; e < nrows * nb; e += kBThreads) {
                const int64_t off = (ra + e / nb) * a.Bp + b0 + e % nb;
                a.ckS[slot + off] = __ldcg(a.Ssum + off);
                a.ckC[slot + off] = __ldcg(a.Ccomp + off);
            }
        }
        // observables of step n-1
        if (st == 0 && n > 0 && a.mode == TDAGW_FULL) last_observables(n);
        if (a.mode != TDAGW_FULL) {
            phase_vhx<NB, CH>();
            if (!bgrid_sync(a, bs)) return;
            if ((gs & 3) == 0 && gs > 0) last_observables(gs >> 2);
            phase_sy<NB, CH>();
            if (!bgrid_sync(a, bs)) return;
            phase_uy<NB, CH>();
            // channel-wise: every CTA has read all rows of X (and written its dSigma rows)
            // before any CTA rewrites its rows
            if (CH && !bgrid_sync(a, bs)) return;
        } else {
            phase_dense<NB>();
            // every CTA has read all rows of X before any CTA rewrites its rows
            if (!bgrid_sync(a, bs)) return;
        }
        __syncthreads();
        epilogue<NB>(a, bs, gs);
        if (tid == 0) gs = gs + 1;
        __syncthreads();
    }
    // observables of the last step
    if (a.Tmax > 0 && bgrid_sync(a, bs)) last_observables(a.Tmax);
}

}  // namespace

}  // namespace tdagw

namespace tdagw {

namespace {

__global__ void replicate_rows_kernel(const double* __restrict__ row, double* __restrict__ obs, int B) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < B) {
        obs[3 * b] = row[0];
        obs[3 * b + 1] = row[1];
        obs[3 * b + 2] = row[2];
    }
}

// obs_out[n][perm[b]] = obs_sorted[n][b]
__global__ void unpermute_kernel(const double* __restrict__ src, double* __restrict__ dst,
                                 const int* __restrict__ perm, int B, int64_t rows) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= rows * B) return;
    const int64_t n = e / B;
    const int b = (int)(e % B);
    for (int q = 0; q < 3; ++q) dst[(n * B + perm[b]) * 3 + q] = src[e * 3 + q];
}

}  // namespace

// Host driver of the batched path (complex64 contexts).  Trajectories are sorted by length
// (longest first); the split into row and trajectory groups follows the active count step by
// step (step_plan), so no call has to be tuned first.
BatchSetup prepare_batch(Ctx& c, const tdagw_field* fields, int B, const int* steps, double dt) {
    const HostModel& h = c.hm;
    cudaStream_t s = c.stream;
    const int64_t N = h.N;
    BatchSetup bs;
    std::vector<int>& perm = bs.perm;
    perm.resize(B);
    for (int b = 0; b < B; ++b) perm[b] = b;
    std::stable_sort(perm.begin(), perm.end(), [&](int x, int y) { return steps[x] > steps[y]; });
    const int Tmax = steps[perm[0]];
    const int Bp = (B + 3) / 4 * 4;
    const int64_t ldE = 2 * (int64_t)Tmax + 1;
    std::vector<int>& act = bs.act;
    act.assign(std::max(Tmax, 1), 0);
    for (int n = 0; n < Tmax; ++n) {
        int cnt = 0;
        for (int b = 0; b < B; ++b) cnt += steps[b] > n ? 1 : 0;
        act[n] = cnt;
    }
    // per-trajectory inputs in sorted order
    c.bEtab.ensure((size_t)B * ldE * sizeof(double));
    TDAGW_CUDA(cudaMemsetAsync(c.bEtab.p, 0, (size_t)B * ldE * sizeof(double), s));
    std::vector<float2> dir(B);
    std::vector<FieldParams> fp(B);
    for (int q = 0; q < B; ++q) {
        const tdagw_field& f = fields[perm[q]];
        const int64_t ns = 2 * (int64_t)steps[perm[q]] + 1;
        if (f.kind == TDAGW_FIELD_TABLE)
            TDAGW_CUDA(cudaMemcpyAsync(c.bEtab.as<double>() + (int64_t)q * ldE, f.table, ns * sizeof(double),
                                       cudaMemcpyHostToDevice, s));
        fp[q] = FieldParams{f.E0, f.omega, f.t0, f.sigma, f.T_pulse, f.kind, ns};
        dir[q] = make_float2((float)f.dir_x, (float)f.dir_y);
    }
    // analytic tables of all trajectories in one launch
    c.bfield.ensure(B * sizeof(FieldParams));
    TDAGW_CUDA(cudaMemcpyAsync(c.bfield.p, fp.data(), B * sizeof(FieldParams), cudaMemcpyHostToDevice, s));
    launch_field_tables(c.bfield.as<FieldParams>(), B, ldE, ldE, dt, c.bEtab.as<double>(), s);
    c.bdir.ensure(B * sizeof(float2));
    TDAGW_CUDA(cudaMemcpyAsync(c.bdir.p, dir.data(), B * sizeof(float2), cudaMemcpyHostToDevice, s));
    c.bact.ensure(act.size() * sizeof(int));
    TDAGW_CUDA(cudaMemcpyAsync(c.bact.p, act.data(), act.size() * sizeof(int), cudaMemcpyHostToDevice, s));
    c.bperm.ensure(B * sizeof(int));
    TDAGW_CUDA(cudaMemcpyAsync(c.bperm.p, perm.data(), B * sizeof(int), cudaMemcpyHostToDevice, s));
    // state
    const size_t sbytes = (size_t)N * Bp * sizeof(float2);
    for (DevBuf* b : {&c.bX, &c.bS, &c.bC, &c.bA, &c.bdS}) b->ensure(sbytes);
    // observables: row 0 is the equilibrium value for every trajectory
    const int64_t rows = Tmax + 1;
    c.bobs.ensure((size_t)rows * B * 3 * sizeof(double));
    TDAGW_CUDA(cudaMemsetAsync(c.bobs.p, 0xFF, (size_t)rows * B * 3 * sizeof(double), s));  // NaN
    c.obs.ensure((size_t)std::max<int64_t>(rows * B, 1) * 3 * sizeof(double));
    TDAGW_CUDA(cudaMemsetAsync(c.X.p, 0, N * sizeof(float2), s));
    launch_observables_row<float>(c, c.X.p, 0, s);
    replicate_rows_kernel<<<(B + 127) / 128, 128, 0, s>>>(c.obs.as<double>(), c.bobs.as<double>(), B);
    check_launch("replicate_rows_kernel");
    bs.Tmax = Tmax;
    bs.Bp = Bp;
    bs.ldE = ldE;
    bs.rows = rows;
    return bs;
}

void reset_batch_observables(Ctx& c, const BatchSetup& bs, int B) {
    TDAGW_CUDA(cudaMemsetAsync(c.bobs.p, 0xFF, (size_t)bs.rows * B * 3 * sizeof(double), c.stream));
    replicate_rows_kernel<<<(B + 127) / 128, 128, 0, c.stream>>>(c.obs.as<double>(), c.bobs.as<double>(), B);
    check_launch("replicate_rows_kernel");
}

void launch_batched(Ctx& c, const void* fn, dim3 grid, dim3 block, size_t smem, const void* args,
                    size_t args_size, const std::vector<ResetOp>& resets, bool use_graph) {
    cudaStream_t s = c.stream;
    void* kargs[] = {const_cast<void*>(args)};
    auto direct = [&](cudaStream_t st) {
        for (const ResetOp& r : resets) TDAGW_CUDA(cudaMemsetAsync(r.p, 0, r.bytes, st));
        TDAGW_CUDA(cudaLaunchCooperativeKernel(fn, grid, block, kargs, smem, st));
    };
    if (!use_graph || c.batch_graphs_off) {
        direct(s);
        return;
    }
    // key: kernel, geometry, shared memory, the argument bytes and the reset list
    std::vector<unsigned char> key;
    auto put = [&](const void* p, size_t n) {
        const unsigned char* b = static_cast<const unsigned char*>(p);
        key.insert(key.end(), b, b + n);
    };
    put(&fn, sizeof(fn));
    put(&grid, sizeof(grid));
    put(&block, sizeof(block));
    put(&smem, sizeof(smem));
    put(args, args_size);
    for (const ResetOp& r : resets) put(&r, sizeof(r));
    for (size_t i = 0; i < c.batch_graphs.size(); ++i)
        if (c.batch_graphs[i].key == key) {
            TDAGW_CUDA(cudaGraphLaunch(c.batch_graphs[i].exec, s));
            return;
        }
    if (!c.cap) TDAGW_CUDA(cudaStreamCreateWithFlags(&c.cap, cudaStreamNonBlocking));
    cudaGraph_t g = nullptr;
    cudaGraphExec_t ge = nullptr;
    bool ok = cudaStreamBeginCapture(c.cap, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
        for (const ResetOp& r : resets) ok = ok && cudaMemsetAsync(r.p, 0, r.bytes, c.cap) == cudaSuccess;
        cudaLaunchAttribute attr;
        attr.id = cudaLaunchAttributeCooperative;
        attr.val.cooperative = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = grid;
        cfg.blockDim = block;
        cfg.dynamicSmemBytes = smem;
        cfg.stream = c.cap;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        ok = ok && cudaLaunchKernelExC(&cfg, fn, kargs) == cudaSuccess;
        const bool ended = cudaStreamEndCapture(c.cap, &g) == cudaSuccess;
        ok = ok && ended && g && cudaGraphInstantiate(&ge, g, 0) == cudaSuccess;
        if (g) cudaGraphDestroy(g);
    }
    if (!ok) {
        // capture of a cooperative launch unavailable: direct launches from now on
        cudaGetLastError();
        if (ge) cudaGraphExecDestroy(ge);
        c.batch_graphs_off = true;
        direct(s);
        return;
    }
    if (c.batch_graphs.size() >= 8) {
        cudaGraphExecDestroy(c.batch_graphs.front().exec);
        c.batch_graphs.erase(c.batch_graphs.begin());
    }
    c.batch_graphs.push_back({key, ge});
    TDAGW_CUDA(cudaGraphLaunch(ge, s));
}

void finish_batch(Ctx& c, const BatchSetup& bs, int B) {
    const int64_t rows = bs.rows;
    c.obs.ensure((size_t)rows * B * 3 * sizeof(double));
    unpermute_kernel<<<(unsigned)((rows * B + 255) / 256), 256, 0, c.stream>>>(
        c.bobs.as<double>(), c.obs.as<double>(), c.bperm.as<int>(), B, rows);
    check_launch("unpermute_kernel");
    c.obs_rows = rows;
    c.obs_B = B;
}

// Partial products, S o Y and observables partials of a launch over G CTAs.
static void batch_buffers(Ctx& c, BatchArgs& a, int G, int r, int Bp) {
    c.bP.ensure((size_t)G * std::max(r, 1) * kTileB * sizeof(float2));
    c.bY.ensure((size_t)std::max(r, 1) * Bp * sizeof(float2));
    c.bred.ensure((size_t)std::min(G, c.hm.Nk) * Bp * 3 * sizeof(double));
    a.P = c.bP.as<float2>();
    a.Y = c.bY.as<float2>();
    a.red = c.bred.as<double>();
}

void propagate_batched(Ctx& c, const tdagw_field* fields, int B, const int* steps, double dt,
                       int mode, int flags) {
    TDAGW_REQUIRE(c.dtype == TDAGW_C64, TDAGW_ERR_UNSUPPORTED, "batched propagation needs a complex64 context");
    TDAGW_REQUIRE(flags & TDAGW_FLAG_RESET, TDAGW_ERR_UNSUPPORTED,
                  "batched propagation starts from drho = 0 (TDAGW_FLAG_RESET)");
    const HostModel& h = c.hm;
    cudaStream_t s = c.stream;
    const int64_t N = h.N;
    const BatchSetup bs = prepare_batch(c, fields, B, steps, dt);
    const std::vector<int>& perm = bs.perm;
    const int Tmax = bs.Tmax;
    const int Bp = bs.Bp;
    const int64_t ldE = bs.ldE;
    const size_t sbytes = (size_t)N * Bp * sizeof(float2);
    // channel-wise mode: S, the partials and Y span the stot columns of the V segments
    const int r = mode == TDAGW_LOWRANK ? c.rank : (mode == TDAGW_CHANNEL ? (int)c.ch.m.stot : 0);
    const int ldu = r + (r & 1);

    int dev = 0, nsm = 0;
    TDAGW_CUDA(cudaGetDevice(&dev));
    TDAGW_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const size_t smem = kBatchSmem;
    const bool ch = mode == TDAGW_CHANNEL;
    const void* fn = h.Nb == 2 ? (ch ? (const void*)batched_kernel<2, true> : (const void*)batched_kernel<2, false>)
                               : (ch ? (const void*)batched_kernel<4, true> : (const void*)batched_kernel<4, false>);
    TDAGW_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    TDAGW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kBThreads, smem));
    TDAGW_REQUIRE(per_sm >= 1, TDAGW_ERR_UNSUPPORTED, "batched kernel does not fit on this device");

    BatchArgs a{};
    a.U = c.U.as<float2>();
    a.V = c.V.as<float2>();
    a.S = mode == TDAGW_CHANNEL ? c.ch.S.as<float>() : c.S.as<float>();
    a.diag = c.diagF.as<float2>();
    if (mode == TDAGW_CHANNEL) {
        // layout tables on the device: ChMeta, then uoff, voff and z (P x P each)
        const int P = h.Nb * h.Nb;
        std::vector<int> tab(3 * P * P);
        for (int e = 0; e < P * P; ++e) {
            tab[e] = c.ch.uoff[e];
            tab[P * P + e] = c.ch.voff[e];
            tab[2 * P * P + e] = c.ch.z[e];
        }
        c.bchm.ensure(sizeof(ChMeta) + tab.size() * sizeof(int));
        TDAGW_CUDA(cudaMemcpyAsync(c.bchm.p, &c.ch.m, sizeof(ChMeta), cudaMemcpyHostToDevice, s));
        TDAGW_CUDA(cudaMemcpyAsync(static_cast<char*>(c.bchm.p) + sizeof(ChMeta), tab.data(), tab.size() * sizeof(int),
                                   cudaMemcpyHostToDevice, s));
        a.Vch = c.ch.V.as<float2>();
        a.Uch = c.ch.U.as<float2>();
        a.chm = c.bchm.as<ChMeta>();
        a.choff = reinterpret_cast<const int*>(static_cast<char*>(c.bchm.p) + sizeof(ChMeta));
    }
    a.kblk = c.kdiag ? c.kblkF.as<float2>() : nullptr;
    a.K = c.K.as<float2>();
    a.dx = c.dx.as<float2>();
    a.dy = c.dy.as<float2>();
    a.vx = c.vx.as<float2>();
    a.gap = c.gap.as<float2>();
    a.X = c.bX.as<float2>();
    a.Ssum = c.bS.as<float2>();
    a.Ccomp = c.bC.as<float2>();
    a.acc = c.bA.as<float2>();
    a.dS = c.bdS.as<float2>();
    a.Etab = c.bEtab.as<double>();
    a.dir = c.bdir.as<float2>();
    a.act = c.bact.as<int>();
    a.obs = c.bobs.as<double>();
    a.N = N;
    a.ldE = ldE;
    a.Nk = h.Nk;
    a.Nb = h.Nb;
    a.r = r;
    a.ldu = ldu;
    a.Bp = Bp;
    a.B = B;
    a.mode = mode;
    a.kahan = (flags & TDAGW_FLAG_NO_KAHAN) ? 0 : 1;
    a.c1 = h.c1;
    for (int q = 0; q < 4; ++q) a.occ[q] = (float)h.occ[q];
    a.dt = (float)dt;
    a.wait_ns = 2000000000ull;
    c.sync.ensure(4 * sizeof(unsigned));
    a.bar = reinterpret_cast<unsigned long long*>(c.sync.p);
    a.err = reinterpret_cast<int*>(c.sync.as<unsigned>() + 2);

    const int G = nsm;  // one CTA per SM (the staging memory fills it)
    TDAGW_REQUIRE((B + kTileB - 1) / kTileB <= G, TDAGW_ERR_UNSUPPORTED, "too many trajectories for one launch");
    batch_buffers(c, a, G, r, Bp);
    a.Tmax = Tmax;
    const bool ckpt = (flags & TDAGW_FLAG_CHECKPOINT) != 0;
    c.adj.valid = false;
    if (ckpt) {
        // compensated state every ceil(sqrt(Tmax)) steps for the adjoint's recomputes
        const int period = std::max(1, (int)std::ceil(std::sqrt((double)Tmax)));
        const int nck = (Tmax + period - 1) / period;
        c.ckS.ensure((size_t)nck * sbytes);
        c.ckC.ensure((size_t)nck * sbytes);
        a.ckS = c.ckS.as<float2>();
        a.ckC = c.ckC.as<float2>();
        a.ck_period = period;
    }
    const bool test_timeout = (flags & TDAGW_FLAG_TEST_TIMEOUT) != 0;
    if (test_timeout) {
        a.extra_arrivals = 1;
        a.wait_ns = 20000000ull;
    }
    launch_batched(c, fn, dim3(G), dim3(kBThreads), smem, &a, sizeof(a),
                   {{c.bX.p, sbytes}, {c.bS.p, sbytes}, {c.bC.p, sbytes}, {c.sync.p, 4 * sizeof(unsigned)}},
                   !(flags & TDAGW_FLAG_NO_GRAPH) && !test_timeout);
    c.persistent_launched = true;
    a.extra_arrivals = 0;
    a.wait_ns = 2000000000ull;
    if (ckpt) {
        AdjointState& st = c.adj;
        st.valid = true;
        st.B = B;
        st.Bp = Bp;
        st.Tmax = Tmax;
        st.period = a.ck_period;
        st.G = G;
        st.mode = mode;
        st.dt = dt;
        st.perm = perm;
        st.steps.assign(steps, steps + B);
        st.fields.assign(fields, fields + B);
        for (tdagw_field& f : st.fields) f.table = nullptr;
        st.fwd_args.resize(sizeof(BatchArgs));
        std::memcpy(st.fwd_args.data(), &a, sizeof(BatchArgs));
        st.fwd_fn = fn;
    }
    // observables in the caller's trajectory order
    finish_batch(c, bs, B);
}

}  // namespace tdagw

namespace tdagw {

// The backward sweep of the adjoint after a checkpointed split-FP16 (tensor-core) forward
// run uses the FP32 batched kernels' split (step_plan).  Fills c.adj like a checkpointed FP32 run; the caller adds the tensor-core fields.
void prepare_adjoint_fp32(Ctx& c, const BatchSetup& bs, const tdagw_field* fields, int B, const int* steps,
                          double dt, int flags) {
    const HostModel& h = c.hm;
    const int64_t N = h.N;
    const int Bp = bs.Bp;
    const int r = c.rank, ldu = r + (r & 1);
    int dev = 0, nsm = 0;
    TDAGW_CUDA(cudaGetDevice(&dev));
    TDAGW_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    const size_t smem = kBatchSmem;
    const void* fn = h.Nb == 2 ? (const void*)batched_kernel<2, false> : (const void*)batched_kernel<4, false>;
    TDAGW_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int per_sm = 0;
    TDAGW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kBThreads, smem));
    TDAGW_REQUIRE(per_sm >= 1, TDAGW_ERR_UNSUPPORTED, "batched kernel does not fit on this device");
    const int G = nsm;
    TDAGW_REQUIRE((B + kTileB - 1) / kTileB <= G, TDAGW_ERR_UNSUPPORTED, "too many trajectories for one launch");
    BatchArgs a{};
    a.U = c.U.as<float2>();
    a.V = c.V.as<float2>();
    a.S = c.S.as<float>();
    a.diag = c.diagF.as<float2>();
    a.kblk = c.kdiag ? c.kblkF.as<float2>() : nullptr;
    a.K = c.K.as<float2>();
    a.dx = c.dx.as<float2>();
    a.dy = c.dy.as<float2>();
    a.vx = c.vx.as<float2>();
    a.gap = c.gap.as<float2>();
    a.X = c.bX.as<float2>();
    a.Ssum = c.bS.as<float2>();
    a.Ccomp = c.bC.as<float2>();
    a.acc = c.bA.as<float2>();
    a.dS = c.bdS.as<float2>();
    a.Etab = c.bEtab.as<double>();
    a.dir = c.bdir.as<float2>();
    a.act = c.bact.as<int>();
    a.obs = c.bobs.as<double>();
    a.N = N;
    a.ldE = bs.ldE;
    a.Nk = h.Nk;
    a.Nb = h.Nb;
    a.r = r;
    a.ldu = ldu;
    a.Bp = Bp;
    a.B = B;
    a.mode = TDAGW_LOWRANK;
    a.kahan = (flags & TDAGW_FLAG_NO_KAHAN) ? 0 : 1;
    a.c1 = h.c1;
    for (int q = 0; q < 4; ++q) a.occ[q] = (float)h.occ[q];
    a.dt = (float)dt;
    a.wait_ns = 2000000000ull;
    c.sync.ensure(4 * sizeof(unsigned));
    a.bar = reinterpret_cast<unsigned long long*>(c.sync.p);
    a.err = reinterpret_cast<int*>(c.sync.as<unsigned>() + 2);
    a.Tmax = bs.Tmax;
    batch_buffers(c, a, G, r, Bp);
    AdjointState& st = c.adj;
    st = AdjointState{};
    st.valid = true;
    st.B = B;
    st.Bp = Bp;
    st.Tmax = bs.Tmax;
    st.G = G;
    st.mode = TDAGW_LOWRANK;
    st.dt = dt;
    st.perm = bs.perm;
    st.steps.assign(steps, steps + B);
    st.fields.assign(fields, fields + B);
    for (tdagw_field& f : st.fields) f.table = nullptr;
    st.fwd_args.resize(sizeof(BatchArgs));
    std::memcpy(st.fwd_args.data(), &a, sizeof(BatchArgs));
    st.fwd_fn = fn;
}

}  // namespace tdagw
