// Shared pieces of the batched kernels (forward propagation and adjoint): launch
// arguments, the bounded grid barrier, trajectory grouping and the register-tiled complex
// matrix product through shared memory.
#pragma once

#include "common.cuh"
#include "persist.cuh"
#include "stage.cuh"

namespace tdagw {
namespace batched {

constexpr int kBThreads = 512;
constexpr int kTileB = 32;      // trajectories per CTA block (max)
constexpr int kDepth = 8;       // reduction depth of one staged chunk (per slice)
constexpr int kStages = 3;      // staged chunks in flight (cp.async groups)
constexpr int kSplitMax = 8;    // reduction-dimension split of block_gemm for small M
// One stage of block_gemm's shared memory (floats): the A chunk (kSplit x kDepth rows of 512 /
// kSplit complex and 4 of padding) and the B chunk (kSplit x kDepth x kTileB complex).
constexpr int kStageA = kDepth * 2 * (512 + 4 * kSplitMax);
constexpr int kStageB = kSplitMax * kDepth * kTileB * 2;
constexpr int kStageFloats = kStageA + kStageB;
constexpr int kGemmFloats = kStages * kStageFloats;
// partial sums of block_gemm's slices reuse the staging memory
static_assert(kGemmFloats >= 512 * kTileB * 2, "slice partials fit the staging memory");
struct BatchArgs {
    // factors / kernel
    const float2* U;      // N x ldu
    const float2* V;      // N x ldu
    const float* S;       // r
    const float2* diag;   // N
    const float2* kblk;   // k-block reading of K^diag (Nk x P x P, (k P + p) P + q) or nullptr
    const float2* K;      // N x N (dense mode)
    // channel-wise mode (Eq. svd-channel-wise): V and U segments, the layout, and the P x P
    // tables uoff [p P + q], voff [q P + p], z [p P + q] (S, P, Y then span m->stot columns)
    const float2* Vch;
    const float2* Uch;
    const ChMeta* chm;
    const int* choff;
    // model (per pair element)
    const float2* dx;
    const float2* dy;
    const float2* vx;
    const float2* gap;
    // batched state, N x Bp row-major (column b = trajectory b in sorted order)
    float2* X;
    float2* Ssum;
    float2* Ccomp;
    float2* acc;
    float2* dS;
    // low-rank intermediates
    float2* P;            // CTAs x r x kTileB: partial products of every CTA
    float2* Y;            // r x Bp
    // per trajectory (sorted order)
    const double* Etab;   // B x ldE
    const float2* dir;    // B (dir_x, dir_y)
    const int* act;       // T_max: active trajectories during step n
    double* red;          // row groups (max) x Bp x 3 observables partials
    double* obs;          // (T_max + 1) x B x 3 (sorted order)
    unsigned long long* bar;
    int* err;
    int64_t N, ldE;
    int Nk, Nb, r, ldu, Bp, B, Tmax, mode, kahan, c1;
    float occ[4];
    float dt;
    unsigned long long wait_ns;
    // adjoint support: global step offset of this launch, checkpoints of the compensated
    // state every ck_period steps, and per-stage records of (X_s, dSigma_s) for the steps
    // of this launch (layout [step * 4 + stage][N][Bp])
    int n0, ck_period;
    float2* ckS;
    float2* ckC;
    float2* recX;
    float2* recDS;
    int extra_arrivals;  // > 0 only for the timeout test: the grid barrier can never complete
};

// One product of block_gemm: C (+)= op(A) B (see there).
struct GemmArgs {
    const float2 *A, *Bm, *diag, *xd;
    float2* out;
    int64_t lda, ldb, ldo;
    int M, Q, nb, acc;
};

// The calling CTA's block of a step: trajectories [b0, b0 + nb) of group tg (none when the
// split leaves the CTA idle), k-points [ka, kb) and their nrows pair elements, columns
// [jr0, jr1) of the S o Y sum, rows [u0, u1) of the pair-major order (channel-wise mode).
struct StepShared {
    int Bact, Rg, rg, tg, ka, kb, nrows, b0, nb, jr0, jr1, u0, u1;
};
// Dynamic shared memory of the batched kernels: the staging memory of block_gemm, the partial
// sums of the observables (16 x kTileB x 3 doubles; also the partial sums of S o Y), and the
// arguments of the product and of the phases (they are calls that need the registers, so
// their arguments go through shared memory).
constexpr int kObsDoubles = (kBThreads / kTileB) * kTileB * 3;
struct BatchShared {
    float gemm[kGemmFloats];
    double obs[kObsDoubles];
    GemmArgs g;
    BatchArgs a;
    StepShared s;
    int abort_s, prev_act, n;
    unsigned gen;
};
static_assert(kBThreads * sizeof(float2) <= kObsDoubles * sizeof(double), "partial sums of S o Y");
constexpr size_t kBatchSmem = sizeof(BatchShared);
// taken from the symbol and not passed to the calls, so that they know it for shared memory
extern __shared__ __align__(16) unsigned char batch_smem[];
__device__ __forceinline__ BatchShared& batch_shared() { return *reinterpret_cast<BatchShared*>(batch_smem); }

// launch arguments -> shared memory, a word per thread
template <typename T> __device__ __forceinline__ void copy_args(T& dst, const T& src) {
    static_assert(sizeof(T) % 4 == 0 && sizeof(T) / 4 <= kBThreads, "one word per thread");
    if (threadIdx.x < sizeof(T) / 4) reinterpret_cast<int*>(&dst)[threadIdx.x] = reinterpret_cast<const int*>(&src)[threadIdx.x];
}

// grid barrier with a monotonic arrival counter (see persist::grid_sync); all threads call
static __device__ bool bgrid_sync(const BatchArgs& a, BatchShared& bs) {
    int* abort_s = &bs.abort_s;
    __syncthreads();
    if (threadIdx.x == 0 && !*abort_s) {
        const unsigned gen = bs.gen;
        const unsigned long long target = (unsigned long long)(gen + 1) * gridDim.x + a.extra_arrivals;
        persist::red_release_add64(a.bar, 1ull);
        const uint64_t t0 = persist::gtimer();
        while (persist::ld_acquire64(a.bar) < target) {
            if (persist::gtimer() - t0 > a.wait_ns || *(volatile int*)a.err) {
                atomicExch(a.err, 1);
                *abort_s = 1;
                break;
            }
            __nanosleep(32);
        }
        bs.gen = gen + 1;
    }
    __syncthreads();
    return !*(volatile int*)abort_s;
}

// Work split of one step with Bact active trajectories over G CTAs: the fewest trajectory
// groups of at most kTileB (a group's products cost a full 32-column tile however few
// columns are live, so splitting further only adds row traffic), and as many k-aligned row
// groups as the CTAs left to each.  Recomputed when the active count changes, so that the
// CTAs of finished trajectories take rows of the remaining ones: the field sweep (B = 256,
// N = 2304, rank 256, uneven lengths) keeps its tiles full to the end.
struct StepPlan {
    int Rg, Tg;
};
__host__ __device__ __forceinline__ StepPlan step_plan(int Bact, int G, int Nk) {
    StepPlan p;
    p.Tg = (Bact + kTileB - 1) / kTileB;
    if (p.Tg < 1) p.Tg = 1;
    p.Rg = G / p.Tg;
    if (p.Rg > Nk) p.Rg = Nk;
    return p;
}

// trajectories [b0, b1) of group tg among the B_act active ones
__device__ __forceinline__ void group_range(int Bact, int Tg, int tg, int& b0, int& b1) {
    b0 = (int)((int64_t)tg * Bact / Tg);
    b1 = (int)((int64_t)(tg + 1) * Bact / Tg);
}

__device__ __forceinline__ void set_step(const BatchArgs& a, int Bact, int NB2, volatile StepShared& s) {
    const StepPlan pl = step_plan(Bact, gridDim.x, a.Nk);
    const int rg = blockIdx.x % pl.Rg, tg = blockIdx.x / pl.Rg;
    const int ka = (int)((int64_t)rg * a.Nk / pl.Rg), kb = (int)((int64_t)(rg + 1) * a.Nk / pl.Rg);
    int b0 = 0, b1 = 0;
    if (tg < pl.Tg) group_range(Bact, pl.Tg, tg, b0, b1);
    s.Bact = Bact;
    s.Rg = pl.Rg;
    s.rg = rg;
    s.tg = tg;
    s.ka = ka;
    s.kb = kb;
    s.nrows = (kb - ka) * NB2;
    s.b0 = b0;
    s.nb = b1 - b0;
    s.jr0 = (int)((int64_t)rg * a.r / pl.Rg);
    s.jr1 = (int)((int64_t)(rg + 1) * a.r / pl.Rg);
    s.u0 = (int)((int64_t)rg * a.N / pl.Rg);
    s.u1 = (int)((int64_t)(rg + 1) * a.N / pl.Rg);
}

// asynchronous copies global -> shared of n bytes, zero-filled up to 8 or 16
__device__ __forceinline__ void cp8(float2* dst, const float2* src, int n) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(n)
                 : "memory");
}
__device__ __forceinline__ void cp16(float2* dst, const float2* src, int n) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((unsigned)__cvta_generic_to_shared(dst)),
                 "l"(src), "r"(n)
                 : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// C[m][b] (+)= sum_q opA(q, m) Bm[q][b] for m in [0, M), b in [0, nb) (nb <= 32),
// q in [0, Q).  opA(q, m) = conj(A[q lda + m]) (TRANS: A is Q x M, rows q) or
// A[m lda + q] (NN: A is M x Q, rows m).  Bm rows q at Bm + q ldb.
//
// Bound by the FP32 pipes (each CTA reuses a staged A element 32 times).  Register tile:
// TM rows x 4 columns complex per thread, 8 column groups x tyc row groups x ks slices of the
// reduction dimension (tyc ks = 64): 256 FMAs for six 16-byte shared-memory loads at TM = 8.
// The loads read 64 or 128 contiguous bytes per 8 lanes (the former tile's 32-byte stride
// cost twice the wavefronts).  Scalar FMAs: the packed two-FMA instruction reaches 39 TFLOP/s
// on an outer product, against 64 for scalar FMAs (measured, 152 SMs, register operands only).
// Chunks of kDepth rows per slice arrive by cp.async, kStages deep, with one barrier per
// chunk.  A CTA's few rows (the U Y and K X products: 15 to 130 rows) are covered by narrow
// tiles with the reduction split over up to 8 slices, whose partial tiles are added in a
// fixed order through the idle staging memory: results are deterministic.  acc adds to out.
// Measured alone on 152 SMs, 32 columns: 52 TFLOP/s at 512 x 512, 42 at 256 x 121 and
// 121 x 256, 34 at 36 x 512 (64 is the FMA ceiling above).  With step_plan, against the
// former 4 x 4 single-buffered tile and fixed split: the field sweep 55.5 -> 34.0 ms (256
// uneven trajectories of 20-160 steps, N = 2304, rank 256), checkpointed forward and gradients
// of 32 trajectories 56.6 -> 31.5 ms (49 steps, N = 5184, rank 512).
template <bool TRANS, int TM, int LKS>
__device__ __noinline__ void block_gemm_tile() {
    BatchShared& bs = batch_shared();
    float* smem = bs.gemm;
    const GemmArgs* g = &bs.g;
    const float2 *__restrict__ A = g->A, *__restrict__ Bm = g->Bm;
    const int64_t lda = g->lda, ldb = g->ldb;
    const int M = g->M, Q = g->Q, nb = g->nb;
    constexpr int ks = 1 << LKS;               // slices of the reduction dimension
    constexpr int ng = kBThreads / ks;         // threads per slice
    constexpr int tyc = ng / 8;                // row groups
    constexpr int Mt = TM * tyc;               // rows per pass
    constexpr int ldq = Mt + 4;                // complex per staged A row
    // rows of a thread: TM / 2 pairs 2 ty + 2 tyc u, + 1, and one more when TM is odd
    constexpr int TP = TM / 2;
    static_assert(ks * kDepth * ldq * 2 <= kStageA && ks * kDepth * kTileB * 2 <= kStageB, "stage size");
    const int tid = threadIdx.x;
    const int slice = tid / ng, tl = tid % ng;
    const int tx = tl % 8, ty = tl / 8;
    auto row_of = [&](int u) { return u < 2 * TP ? 2 * ty + 2 * tyc * (u >> 1) + (u & 1) : 2 * tyc * TP + ty; };
    for (int m0 = 0; m0 < M; m0 += Mt) {
        const int mrows = min(Mt, M - m0);
        float2 c[TM][4];
#pragma unroll
        for (int u = 0; u < TM; ++u)
#pragma unroll
            for (int v = 0; v < 4; ++v) c[u][v] = make_float2(0.f, 0.f);
        const int nfull = (Q + ks * kDepth - 1) / (ks * kDepth);
        // depth of chunk c (the last one is spread evenly over the slices)
        auto depth = [&](int ch) { return min(kDepth, (Q - ch * ks * kDepth + ks - 1) / ks); };
        // this thread's share of a full chunk: fixed places, so that a full chunk costs one
        // address and one copy per element pair (TRANS: consecutive threads copy consecutive
        // pairs along m, rows start on 16 bytes (even lda); NN: 8 consecutive threads copy the
        // kDepth columns of a row)
        const int fr = TRANS ? tid / (Mt / 2) : tid / kDepth, fm = TRANS ? 2 * (tid % (Mt / 2)) : 0;
        const float2* fa = TRANS ? A + (int64_t)fr * lda + m0 + fm : A + (int64_t)m0 * lda + tid % kDepth;
        const int fn = TRANS ? 8 * max(0, min(2, mrows - fm)) : 0;
        const int bb = tid % kTileB, br = tid / kTileB;
        const float2* fb = Bm + (int64_t)br * ldb + bb;
        auto stage = [&](int ch) {
            if (ch < nfull) {
                float2* sA = reinterpret_cast<float2*>(smem + (ch % kStages) * kStageFloats);
                float2* sB = sA + kStageA / 2;
                const int q0 = ch * ks * kDepth, kc = depth(ch);
                if (q0 + ks * kDepth <= Q) {
                    if (TRANS) {
                        constexpr int rs = 2 * kBThreads / Mt;  // rows per copy of the CTA
                        const float2* p = fa + (int64_t)q0 * lda;
                        float2* d = sA + fr * ldq + fm;
#pragma unroll
                        for (int i = 0; i < ks * kDepth / rs; ++i) {
                            cp16(d + i * rs * ldq, fn ? p : A, fn);
                            p += (int64_t)rs * lda;
                        }
                    } else {
                        constexpr int rs = kBThreads / kDepth;  // (slice, m) rows per copy of the CTA
                        const float2* p = fa + q0;
                        const int q = tid % kDepth;
#pragma unroll
                        for (int i = 0; i < ks * Mt / rs; ++i) {
                            const int m = (fr + i * rs) % Mt, sl = (fr + i * rs) / Mt;
                            const bool in = m < mrows;
                            cp8(sA + (sl * kDepth + q) * ldq + m, in ? p + (int64_t)m * lda + sl * kDepth : A, in ? 8 : 0);
                        }
                    }
                    constexpr int rb = kBThreads / kTileB;
                    const float2* p = fb + (int64_t)q0 * ldb;
                    const int n = bb < nb ? 8 : 0;
#pragma unroll
                    for (int i = 0; i < (ks * kDepth + rb - 1) / rb; ++i) {
                        if (ks * kDepth >= rb || br < ks * kDepth) cp8(sB + tid + i * kBThreads, n ? p : Bm, n);
                        p += (int64_t)rb * ldb;
                    }
                } else {
                    for (int e = tid; e < ks * kDepth * Mt; e += kBThreads) {
                        const int q = e % kDepth, r = e / kDepth, m = r % Mt, s = r / Mt;
                        if (q < kc) {
                            const int qg = q0 + s * kc + q;
                            const bool in = qg < Q && m < mrows;
                            cp8(sA + (s * kDepth + q) * ldq + m,
                                !in ? A : (TRANS ? A + (int64_t)qg * lda + m0 + m : A + (int64_t)(m0 + m) * lda + qg),
                                in ? 8 : 0);
                        }
                    }
                    for (int e = tid; e < ks * kDepth * kTileB; e += kBThreads) {
                        const int b = e % kTileB, r = e / kTileB, s = r / kDepth, q = r % kDepth;
                        if (q < kc) {
                            const int qg = q0 + s * kc + q;
                            const bool in = qg < Q && b < nb;
                            cp8(sB + e, in ? Bm + (int64_t)qg * ldb + b : Bm, in ? 8 : 0);
                        }
                    }
                }
            }
            cp_commit();
        };
#pragma unroll
        for (int ch = 0; ch < kStages - 1; ++ch) stage(ch);
        for (int ch = 0; ch < nfull; ++ch) {
            cp_wait<kStages - 2>();
            __syncthreads();  // chunk ch has landed for every thread; chunk ch - 1 is consumed
            stage(ch + kStages - 1);
            const float2* sA = reinterpret_cast<const float2*>(smem + (ch % kStages) * kStageFloats);
            const float2* sB = sA + kStageA / 2 + slice * kDepth * kTileB;
            sA += slice * kDepth * ldq;
            const int kc = depth(ch);
            auto fma_row = [&](int q) {
                float4 av[TP + (TM & 1)], bv[2];
                // columns 2 tx, 2 tx + 1, 16 + 2 tx, 17 + 2 tx
                bv[0] = *reinterpret_cast<const float4*>(sB + q * kTileB + 2 * tx);
                bv[1] = *reinterpret_cast<const float4*>(sB + q * kTileB + 16 + 2 * tx);
#pragma unroll
                for (int u = 0; u < TP; ++u) av[u] = *reinterpret_cast<const float4*>(sA + q * ldq + 2 * ty + 2 * tyc * u);
                if (TM & 1) {
                    const float2 z = sA[q * ldq + 2 * tyc * TP + ty];
                    av[TM / 2] = make_float4(z.x, z.y, 0.f, 0.f);
                }
#pragma unroll
                for (int u = 0; u < TM; ++u) {
                    const float4 a4 = av[u / 2];
                    const float ax = (u & 1) ? a4.z : a4.x;
                    const float ay = (u & 1) ? a4.w : a4.y;
#pragma unroll
                    for (int v = 0; v < 4; ++v) {
                        const float4 b4 = bv[v / 2];
                        const float bx = (v & 1) ? b4.z : b4.x;
                        const float by = (v & 1) ? b4.w : b4.y;
                        c[u][v].x = fmaf(ax, bx, c[u][v].x);
                        c[u][v].y = fmaf(ax, by, c[u][v].y);
                        // conj(a) b or a b
                        c[u][v].x = fmaf(TRANS ? ay : -ay, by, c[u][v].x);
                        c[u][v].y = fmaf(TRANS ? -ay : ay, bx, c[u][v].y);
                    }
                }
            };
            // not unrolled: 2 or 4 rows gain nothing (four warps per scheduler cover the loads)
            // and cost registers
#pragma unroll 1
            for (int q = 0; q < kc; ++q) fma_row(q);
        }
        const float2 *diag = g->diag, *xd = g->xd;
        float2* out = g->out;
        const int64_t ldo = g->ldo;
        const bool acc_out = g->acc != 0;
        auto finish = [&](int m, int b, float2 r) {
            if (diag) r = cfma(diag[m], __ldcg(xd + (int64_t)m * ldb + b), r);
            float2* o = out + (int64_t)m * ldo + b;
            if (acc_out) r = cadd(r, *o);
            *o = r;
        };
        if (ks == 1) {
#pragma unroll
            for (int u = 0; u < TM; ++u)
#pragma unroll
                for (int v = 0; v < 4; ++v) {
                    const int b = (v >> 1) * 16 + 2 * tx + (v & 1), m = row_of(u);
                    if (b < nb && m < mrows) finish(m0 + m, b, c[u][v]);
                }
            __syncthreads();  // the staging memory is reused
        } else {
            __syncthreads();  // the last chunk is consumed
            float2* red = reinterpret_cast<float2*>(smem);  // [slice][m][32]
#pragma unroll
            for (int u = 0; u < TM; ++u)
#pragma unroll
                for (int h = 0; h < 2; ++h)
                    *reinterpret_cast<float4*>(red + (slice * Mt + row_of(u)) * kTileB + 16 * h + 2 * tx) =
                        make_float4(c[u][2 * h].x, c[u][2 * h].y, c[u][2 * h + 1].x, c[u][2 * h + 1].y);
            __syncthreads();
            for (int e = tid; e < mrows * kTileB; e += kBThreads) {
                const int b = e % kTileB;
                float2 r = red[e];
#pragma unroll
                for (int s = 1; s < ks; ++s) r = cadd(r, red[s * Mt * kTileB + e]);
                if (b < nb) finish(m0 + e / kTileB, b, r);
            }
            __syncthreads();
        }
    }
}

// k-block reading of K^diag: out[row][b] += sum_q B_k[p][q] x[k P + q][b] (CT: the conjugate
// transpose, conj(B_k[q][p]), for K^H) for rows [ra, ra + nrows) (whole k-points) and columns
// [b0, b0 + nb); row = k P + p, B_k[p][q] at kblk[(k P + p) P + q].
template <int NB, bool CT>
static __device__ void kblock_term(const float2* __restrict__ kblk, const float2* __restrict__ x,
                                   float2* __restrict__ out, int64_t ld, int64_t ra, int nrows, int b0, int nb) {
    constexpr int P = NB * NB;
    for (int e = threadIdx.x; e < nrows * nb; e += kBThreads) {
        const int64_t row = ra + e / nb;
        const int b = b0 + e % nb;
        const int64_t k0 = row - row % P;
        const int p = (int)(row % P);
        float2 s = __ldcg(out + row * ld + b);
#pragma unroll
        for (int q = 0; q < P; ++q) {
            const float2 bq = CT ? cconj(kblk[(k0 + q) * P + p]) : kblk[row * P + q];
            s = cfma(bq, __ldcg(x + (k0 + q) * ld + b), s);
        }
        out[row * ld + b] = s;
    }
}

// The product with the tile of those built that pads M least: the cost of a pass is that of its Mt
// rows (512 threads x TM rows / slices), whatever the split.  Heights 3 and 7 (17 to 24 and 49 to 56
// rows) are not built; 4 and 8 take those.
template <bool TRANS>
static __device__ __forceinline__ void block_gemm(const float2* __restrict__ A, int64_t lda, int M, int Q,
                                  const float2* __restrict__ Bm, int64_t ldb, int nb,
                                  float2* __restrict__ out, int64_t ldo, bool acc_out,
                                  const float2* __restrict__ diag, const float2* __restrict__ xd) {
    if (threadIdx.x == 0) batch_shared().g = GemmArgs{A, Bm, diag, xd, out, lda, ldb, ldo, M, Q, nb, acc_out ? 1 : 0};
    __syncthreads();
    if (TRANS) {  // V^H X: M is the rank
        if (M > 256) block_gemm_tile<TRANS, 8, 0>();
        else if (M > 128) block_gemm_tile<TRANS, 8, 1>();
        else if (M > 64) block_gemm_tile<TRANS, 8, 2>();
        else block_gemm_tile<TRANS, 8, 3>();
    } else {      // U Y, K X: M is the CTA's rows
        if (M > 128) block_gemm_tile<TRANS, 8, 1>();
        else if (M > 64) block_gemm_tile<TRANS, 8, 2>();
        else if (M > 48) block_gemm_tile<TRANS, 8, 3>();
        else if (M > 40) block_gemm_tile<TRANS, 6, 3>();
        else if (M > 32) block_gemm_tile<TRANS, 5, 3>();
        else if (M > 16) block_gemm_tile<TRANS, 4, 3>();
        else block_gemm_tile<TRANS, 2, 3>();
    }
}

// Sum over c in [0, n) of src[c stride] (complex) by the calling thread, eight loads in flight,
// fixed order.
static __device__ __forceinline__ float2 strided_sum(const float2* __restrict__ src, int64_t stride, int n) {
    float2 s8[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) s8[u] = make_float2(0.f, 0.f);
    int c = 0;
    for (; c + 8 <= n; c += 8) {
#pragma unroll
        for (int u = 0; u < 8; ++u) s8[u] = cadd(s8[u], __ldcg(src + (c + u) * stride));
    }
#pragma unroll
    for (int u = 0; u < 7; ++u)
        if (c + u < n) s8[u] = cadd(s8[u], __ldcg(src + (c + u) * stride));
    return cadd(cadd(cadd(s8[0], s8[1]), cadd(s8[2], s8[3])), cadd(cadd(s8[4], s8[5]), cadd(s8[6], s8[7])));
}

// Y[j][b] = S_j sum_g part[g][j][b] for the columns j of [jr0, jr1) and this group's nb
// trajectories: partials of the row groups [g0(j), g1(j)] at P + g pstride + j kTileB + bl.
// With few columns per CTA the sum over the row groups is split over the CTA's threads
// (subsets combined in a fixed order through scr, 512 float2), so that it is one or two
// batches of loads instead of a serial chain.
template <class RANGE>
static __device__ void reduce_partials(const float2* __restrict__ P, int64_t pstride, int jr0, int jr1, int nb,
                                       const float* __restrict__ S, float2* __restrict__ Y, int64_t ldy, RANGE range,
                                       float2* scr) {
    const int ne = (jr1 - jr0) * kTileB;
    for (int base = 0; base < ne; base += kBThreads) {
        const int w = min(ne - base, kBThreads);          // elements of this pass (a multiple of 32)
        const int nsub = kBThreads / w;                   // threads per element
        const int sub = threadIdx.x / w, e = base + threadIdx.x % w;
        const int j = jr0 + e / kTileB, bl = e % kTileB;
        float2 s = make_float2(0.f, 0.f);
        if (sub < nsub && bl < nb) {
            int g0, g1;
            range(j, g0, g1);
            const int first = g0 + sub;
            if (first <= g1)
                s = strided_sum(P + (int64_t)first * pstride + (int64_t)j * kTileB + bl, pstride * nsub,
                                (g1 - first) / nsub + 1);
        }
        if (nsub > 1) {
            __syncthreads();
            if (sub < nsub) scr[sub * w + threadIdx.x % w] = s;
            __syncthreads();
            if (sub == 0)
                for (int u = 1; u < nsub; ++u) s = cadd(s, scr[u * w + threadIdx.x]);
        }
        if (sub == 0 && bl < nb) Y[(int64_t)j * ldy + bl] = cscale(s, S[j]);
    }
}

// Observables of step n (rows of a.obs) of the trajectories of group tg at that step from the
// row groups' partials: one warp per trajectory, lanes over the row groups, fixed order.  The
// trajectories are dealt to the last warps of the group's CTAs (rg of Rg): one CTA alone held
// up the next barrier by 4 us.
static __device__ void reduce_observables_row(const BatchArgs& a, int n, const StepPlan& pl, int tg, int rg) {
    if ((threadIdx.x >> 5) != kBThreads / 32 - 1) return;
    int p0, p1;
    group_range(a.act[a.n0 + n - 1], pl.Tg, tg, p0, p1);
    const int lane = threadIdx.x & 31;
    for (int b = p0 + rg; b < p1; b += pl.Rg) {
        double s0 = 0, s1 = 0, s2 = 0;
        for (int g = lane; g < pl.Rg; g += 32) {
            const double* rr = a.red + ((int64_t)g * a.Bp + b) * 3;
            s0 += __ldcg(rr);
            s1 += __ldcg(rr + 1);
            s2 += __ldcg(rr + 2);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            s0 += __shfl_xor_sync(0xffffffffu, s0, o);
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        if (lane == 0) {
            double* o = a.obs + ((int64_t)n * a.B + b) * 3;
            o[0] = s0 / a.Nk;
            o[1] = s1 / a.Nk;
            o[2] = s2 / a.Nk;
        }
    }
}

}  // namespace batched
}  // namespace tdagw
