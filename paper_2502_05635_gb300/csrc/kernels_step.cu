// Per-stage kernels of the propagation: the kernel contraction dSigma = K . X as a
// streaming complex GEMV (dense form of Eq. sigma-from-k, and the two passes of the
// truncated-SVD form of Eq. svd_acc), and the fused per-k commutator + RK4 stage update +
// observables kernel (Eq. tdagw).
#include <cooperative_groups.h>

#include "common.cuh"
#include "stage.cuh"

namespace tdagw {

namespace {

// threads per block of the stage and observables kernels: in FP64 small blocks, which spread a
// few thousand elements over the SMs (bound by the few FP64 pipes of each)
template <typename R> constexpr int kStageThreads = sizeof(R) == 8 ? 32 : 256;

// ---------------------------------------------------------------- vector loads -------

// Two consecutive complex elements; streaming (evict-first) loads for matrix operands
// that are read once per stage, cached loads for the vector operand.
__device__ __forceinline__ void ld2_stream(const float2* p, float2& a, float2& b) {
    const float4 v = __ldcs(reinterpret_cast<const float4*>(p));
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ld2_stream(const double2* p, double2& a, double2& b) {
    a = __ldcs(p);
    b = __ldcs(p + 1);
}
__device__ __forceinline__ void ld2_plain(const float2* p, float2& a, float2& b) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ld2_plain(const double2* p, double2& a, double2& b) {
    a = p[0];
    b = p[1];
}
__device__ __forceinline__ void ld2_cached(const float2* p, float2& a, float2& b) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(p));
    a = make_float2(v.x, v.y);
    b = make_float2(v.z, v.w);
}
__device__ __forceinline__ void ld2_cached(const double2* p, double2& a, double2& b) {
    a = __ldg(p);
    b = __ldg(p + 1);
}

// ---------------------------------------------------------------- GEMV ---------------

// out[row] = sum_c A[row, c] x[c] for ROWS rows per block.  Each thread walks the columns two
// complex at a time (16 B per row per step for c64) so that a warp covers 512 contiguous
// bytes of each row per load; the ROWS accumulators share every load of x.  Bound by HBM:
// 0.487 ms = 7.06 TB/s at N = 20736 in complex64 (0.541 while the kernel also had a split of
// the columns, which no call used).
template <typename R, int ROWS, int THREADS>
__global__ void __launch_bounds__(THREADS)
gemv_kernel(const cplx_t<R>* __restrict__ A, int64_t lda, int64_t nrows, int64_t ncols,
            const cplx_t<R>* __restrict__ x, cplx_t<R>* __restrict__ out) {
    using C = cplx_t<R>;
    const int64_t r0 = (int64_t)blockIdx.x * ROWS;
    C acc[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) acc[r] = mk((R)0, (R)0);
    const int tid = threadIdx.x;
    bool valid[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) valid[r] = (r0 + r) < nrows;

    int64_t c = 2 * tid;
#pragma unroll 2
    for (; c + 1 < ncols; c += 2 * THREADS) {
        C x0, x1;
        ld2_cached(x + c, x0, x1);
        C a0[ROWS], a1[ROWS];
#pragma unroll
        for (int r = 0; r < ROWS; ++r) {
            if (valid[r]) ld2_stream(A + (r0 + r) * lda + c, a0[r], a1[r]);
            else a0[r] = a1[r] = mk((R)0, (R)0);
        }
#pragma unroll
        for (int r = 0; r < ROWS; ++r) acc[r] = cfma(a1[r], x1, cfma(a0[r], x0, acc[r]));
    }
    if ((ncols & 1) && tid == 0) {
        const int64_t cl = ncols - 1;
        const C xl = x[cl];
#pragma unroll
        for (int r = 0; r < ROWS; ++r)
            if (valid[r]) acc[r] = cfma(A[(r0 + r) * lda + cl], xl, acc[r]);
    }
    // block reduction: warp shuffles, then across warps in shared memory
#pragma unroll
    for (int r = 0; r < ROWS; ++r)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[r] = cadd(acc[r], shfl_xor(acc[r], o));
    constexpr int NW = THREADS / 32;
    __shared__ C red[NW][ROWS];
    const int lane = tid & 31, warp = tid >> 5;
    if (lane == 0)
#pragma unroll
        for (int r = 0; r < ROWS; ++r) red[warp][r] = acc[r];
    __syncthreads();
    if (tid < ROWS && valid[tid]) {
        C s = red[0][tid];
#pragma unroll
        for (int w = 1; w < NW; ++w) s = cadd(s, red[w][tid]);
        out[r0 + tid] = s;
    }
}

// y = V^H x with V stored N x ldu row-major: block (b, cb) accumulates
//   part[b][c] = sum_{i in rows of b} conj(V[i][c]) x_i
// for its 512 columns c (two per thread), streaming the rows of V (16 B per thread per
// row, so a warp reads 256 contiguous bytes).
template <typename R>
__global__ void __launch_bounds__(256)
vcols_kernel(const cplx_t<R>* __restrict__ V, int64_t ldv, int64_t N, int r,
             const cplx_t<R>* __restrict__ x, cplx_t<R>* __restrict__ part, int64_t rpb) {
    using C = cplx_t<R>;
    const int64_t i0 = blockIdx.x * rpb, i1 = min(N, i0 + rpb);
    const int64_t c = (int64_t)blockIdx.y * 512 + 2 * threadIdx.x;
    if (c >= ldv) return;
    C a0 = mk((R)0, (R)0), a1 = a0;
#pragma unroll 4
    for (int64_t i = i0; i < i1; ++i) {
        C v0, v1;
        ld2_stream(V + i * ldv + c, v0, v1);
        const C xi = __ldg(x + i);
        a0 = cfmac(v0, xi, a0);
        a1 = cfmac(v1, xi, a1);
    }
    if (c < r) part[(int64_t)blockIdx.x * r + c] = a0;
    if (c + 1 < r) part[(int64_t)blockIdx.x * r + c + 1] = a1;
}

// ytil[j] = S[j] * sum_s part[s][j]: finishes y = S o (V^H x) of Eq. svd_acc.  kYCols columns
// per block (128 or 256 contiguous bytes), the partials split over the rest of the threads (four
// loads in flight each) and combined in a fixed order: one thread per column took a chain of
// up to 304 loads (about 50 us).  Narrow blocks in FP64, whose additions would otherwise queue
// at the pipes of a few SMs.  subs: threads per column; a few partials (small models) get as many
// as they need and one barrier, not the halvings of a full block (N = 144, channel-wise stage by
// stage, us per stage with one thread per column, a full block and this: 17.2, 17.9, 17.2 in complex64,
// 21.9, 22.8, 20.2 in complex128).
constexpr int kYThreads = 512;
template <typename R> constexpr int kYCols = sizeof(R) == 8 ? 8 : 32;
template <typename R> constexpr int kYSubs = kYThreads / kYCols<R>;
template <typename R, int subs>
__device__ __forceinline__ void yreduce(const cplx_t<R>* __restrict__ part, int nsplit, int r, const R* __restrict__ S,
                                        cplx_t<R>* __restrict__ ytil) {
    using C = cplx_t<R>;
    constexpr int cols = kYCols<R>;
    const int col = threadIdx.x % cols, sub = threadIdx.x / cols;
    const int j = blockIdx.x * cols + col;
    const int q0 = (int)((int64_t)sub * nsplit / subs), q1 = (int)((int64_t)(sub + 1) * nsplit / subs);
    __shared__ C red[subs][cols];
    C s[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) s[u] = mk((R)0, (R)0);
    if (j < r) {
        int q = q0;
        for (; q + 4 <= q1; q += 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) s[u] = cadd(s[u], part[(int64_t)(q + u) * r + j]);
        }
        if (subs <= 4) {
#pragma unroll
            for (int u = 0; u < 3; ++u)
                if (q + u < q1) s[u] = cadd(s[u], part[(int64_t)(q + u) * r + j]);
        } else {
            for (; q < q1; ++q) s[0] = cadd(s[0], part[(int64_t)q * r + j]);
        }
    }
    C t = cadd(cadd(s[0], s[1]), cadd(s[2], s[3]));
    red[sub][col] = t;
    if (subs <= 4) {
        __syncthreads();
        if (sub == 0) {
#pragma unroll
            for (int u = 1; u < subs; ++u) t = cadd(t, red[u][col]);
        }
    } else {
#pragma unroll
        for (int o = subs / 2; o > 0; o >>= 1) {
            __syncthreads();
            if (sub < o) red[sub][col] = cadd(red[sub][col], red[sub + o][col]);
        }
        t = red[sub][col];
    }
    if (sub == 0 && j < r) ytil[j] = cscale(t, S[j]);
}
template <typename R>
__global__ void __launch_bounds__(kYThreads)
yreduce_kernel(const cplx_t<R>* __restrict__ part, int nsplit, int r, const R* __restrict__ S,
               cplx_t<R>* __restrict__ ytil) {
    yreduce<R, kYSubs<R>>(part, nsplit, r, S, ytil);
}
template <typename R, int subs>
__global__ void __launch_bounds__(subs * kYCols<R>)
yreduce_few_kernel(const cplx_t<R>* __restrict__ part, int nsplit, int r, const R* __restrict__ S,
                   cplx_t<R>* __restrict__ ytil) {
    yreduce<R, subs>(part, nsplit, r, S, ytil);
}

// Sums of W rows held one partial per lane: W 2^k halvings across the lanes, then plain
// butterflies, so that four rows cost 6 complex additions per lane instead of 20 (FP64
// additions are as dear as FMAs here).  The sum of row (lane >> (5 - log2 W)) is in every lane
// of its group.
template <int W, typename C> __device__ __forceinline__ C warp_rows_sum(C (&v)[W], int lane) {
    int o = 16;
#pragma unroll
    for (int w = W; w > 1; w >>= 1, o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int q = 0; q < w / 2; ++q) {
            const C keep = up ? v[q + w / 2] : v[q], send = up ? v[q] : v[q + w / 2];
            v[q] = cadd(keep, shfl_xor(send, o));
        }
    }
    C s = v[0];
#pragma unroll
    for (; o > 0; o >>= 1) s = cadd(s, shfl_xor(s, o));
    return s;
}

// one warp's dot products of W consecutive rows of A (row stride lda) with x over ncols
// columns, two complex per lane and step (rows and x start on 16 bytes)
template <typename R, int W>
__device__ __forceinline__ void row_dots(const cplx_t<R>* __restrict__ A, int64_t lda, int nrows, int ncols,
                                         const cplx_t<R>* x, int lane, cplx_t<R> (&acc)[W]) {
    using C = cplx_t<R>;
#pragma unroll
    for (int w = 0; w < W; ++w) acc[w] = mk((R)0, (R)0);
    int c = 2 * lane;
#pragma unroll 2
    for (; c + 1 < ncols; c += 64) {
        C x0, x1;
        ld2_plain(x + c, x0, x1);
#pragma unroll
        for (int w = 0; w < W; ++w)
            if (w < nrows) {
                C a0, a1;
                ld2_stream(A + w * lda + c, a0, a1);
                acc[w] = cfma(a1, x1, cfma(a0, x0, acc[w]));
            }
    }
    if (c < ncols) {
        const C x0 = x[c];
#pragma unroll
        for (int w = 0; w < W; ++w)
            if (w < nrows) acc[w] = cfma(A[w * lda + c], x0, acc[w]);
    }
}

// out[row] = sum_c A[row, c] x[c] (+ diag[row] xd[row]), one warp per W rows: the U pass, whose
// rows are short (a block of 256 threads per four rows left most of them idle below 512
// columns and spent more on its reduction than on the products).
template <typename R, int W>
__global__ void __launch_bounds__(128)
urows_kernel(const cplx_t<R>* __restrict__ A, int64_t lda, int64_t nrows, int ncols, const cplx_t<R>* __restrict__ x,
             cplx_t<R>* __restrict__ out, const cplx_t<R>* __restrict__ diag, const cplx_t<R>* __restrict__ xd) {
    using C = cplx_t<R>;
    const int lane = threadIdx.x & 31;
    const int64_t r0 = (blockIdx.x * (int64_t)4 + (threadIdx.x >> 5)) * W;
    if (r0 >= nrows) return;
    C acc[W];
    row_dots<R, W>(A + r0 * lda, lda, (int)min((int64_t)W, nrows - r0), ncols, x, lane, acc);
    C s = warp_rows_sum<W>(acc, lane);
    const int64_t row = r0 + lane / (32 / W);
    if (lane % (32 / W) == 0 && row < nrows) {
        if (diag) s = cfma(diag[row], xd[row], s);
        out[row] = s;
    }
}

// ---------------------------------------------------------------- small apply --------

// The whole low-rank application y = diag o x + U (S o (V^H x)) in one launch: one cluster of
// eight CTAs, each with a contiguous share of the rows.  V^H x over the share (column pairs x
// row subsets, subsets added in order), the eight partial vectors through distributed shared
// memory, then the share's rows of U.  Bound by the three launches it replaces (small N r).
constexpr int kClThreads = 512, kClCtas = 8, kClMaxRank = 512;
// N r at most: N = 576, rank 29 takes 7.2 us a call (14.4 with three launches and the former
// reductions), rank 110 10.3 (rank 120 with three launches 14.4); N = 2304, rank 28 12.3 (rank
// 30 15.4).  And N at most: eight CTAs walk all rows, 256 a pass, so a low rank does not make a
// large model cheap.  us per call of a series, one cluster against three launches, at ranks 3
// and 12: N = 1296 10.3 and 14.4, 8.4 and 14.4; N = 2704 14.5 and 14.5, 12.4 and 16.5; N = 3600 16.6
// and 15.5, 15.5 and 16.5; N = 5184 22.4 and 15.5, 20.5 and 16.5; N = 20736 rank 3 67.7 and 23.7.
// Complex64 only: in complex128 eight SMs' FP64 pipes are slower than three launches.
constexpr int64_t kClMaxElems = 65536, kClMaxN = 3072;
__global__ void __cluster_dims__(kClCtas, 1, 1) __launch_bounds__(kClThreads)
lr_cluster_kernel(const float2* __restrict__ U, const float2* __restrict__ V, int64_t ld, int N, int r,
                  const float* __restrict__ S, const float2* __restrict__ diag, const float2* __restrict__ x,
                  float2* __restrict__ y) {
    using R = float;
    using C = float2;
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    __shared__ __align__(16) C sub[2 * kClThreads];
    __shared__ __align__(16) C part[kClMaxRank], ys[kClMaxRank];
    const int tid = threadIdx.x, lane = tid & 31, cta = (int)cl.block_rank();
    const int i0 = (int)((int64_t)cta * N / kClCtas), i1 = (int)((int64_t)(cta + 1) * N / kClCtas);
    const int ncp = (r + 1) / 2, nsub = kClThreads / ncp;
    const int cp = tid % ncp, sb = tid / ncp;
    C a0 = mk((R)0, (R)0), a1 = a0;
    const bool two = 2 * cp + 1 < r;
    if (sb < nsub) {
#pragma unroll 4
        for (int i = i0 + sb; i < i1; i += nsub) {
            const C* v = V + i * ld + 2 * cp;
            const C xi = x[i];
            if (two) {
                C v0, v1;
                ld2_stream(v, v0, v1);
                a0 = cfmac(v0, xi, a0);
                a1 = cfmac(v1, xi, a1);
            } else {
                a0 = cfmac(v[0], xi, a0);
            }
        }
        sub[2 * tid] = a0;
        sub[2 * tid + 1] = a1;
    }
    __syncthreads();
    for (int j = tid; j < r; j += kClThreads) {
        C s = sub[j];
        for (int u = 1; u < nsub; ++u) s = cadd(s, sub[2 * u * ncp + j]);
        part[j] = s;
    }
    cl.sync();
    for (int j = tid; j < r; j += kClThreads) {
        C s = cl.map_shared_rank(part, 0)[j];
#pragma unroll
        for (int c = 1; c < kClCtas; ++c) s = cadd(s, cl.map_shared_rank(part, c)[j]);
        ys[j] = cscale(s, S[j]);
    }
    cl.sync();  // the partials are read before any CTA exits; ys is complete
    constexpr int W = 2;
    for (int r0 = i0 + W * (tid >> 5); r0 < i1; r0 += W * (kClThreads / 32)) {
        C acc[W];
        row_dots<R, W>(U + r0 * ld, ld, min(W, i1 - r0), r, ys, lane, acc);
        C s = warp_rows_sum<W>(acc, lane);
        const int row = r0 + lane / (32 / W);
        if (lane % (32 / W) == 0 && row < i1) {
            if (diag) s = cfma(diag[row], x[row], s);
            y[row] = s;
        }
    }
}

// ---------------------------------------------------------------- stage --------------

// Block partial sums of (P_x, J_x, occ_c1) in FP64, then the last block to arrive adds
// the partials in a fixed order and stores row `row` of obs.  Up to 32 blocks one warp does it: the
// full block's two levels of shuffles and its barriers cost more than one thread's sum did (dense,
// N = 256, 100 steps: 2.40 ms with one thread, 2.49 with the block, 2.34 with one warp).
__device__ void reduce_observables(double v0, double v1, double v2, double* red,
                                   unsigned* counter, double* obs_row, double inv_nk,
                                   int64_t* step_to_bump, int64_t new_step) {
    for (int o = 16; o > 0; o >>= 1) {
        v0 += __shfl_xor_sync(0xffffffffu, v0, o);
        v1 += __shfl_xor_sync(0xffffffffu, v1, o);
        v2 += __shfl_xor_sync(0xffffffffu, v2, o);
    }
    __shared__ double sred[32][3];
    __shared__ bool last;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) {
        sred[warp][0] = v0;
        sred[warp][1] = v1;
        sred[warp][2] = v2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0, b = 0, c = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            a += sred[w][0];
            b += sred[w][1];
            c += sred[w][2];
        }
        red[blockIdx.x * 3 + 0] = a;
        red[blockIdx.x * 3 + 1] = b;
        red[blockIdx.x * 3 + 2] = c;
        __threadfence();
        const unsigned t = atomicAdd(counter, 1u);
        last = (t == gridDim.x - 1);
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double a = 0, b = 0, c = 0;
    if (gridDim.x <= 32) {
        // one warp, one partial per lane, as many halvings as there are partials
        if (warp == 0) {
            if (lane < (int)gridDim.x) {
                a = __ldcg(red + lane * 3 + 0);
                b = __ldcg(red + lane * 3 + 1);
                c = __ldcg(red + lane * 3 + 2);
            }
            for (int o = 16; o > 0; o >>= 1)
                if (o < (int)gridDim.x) {
                    a += __shfl_xor_sync(0xffffffffu, a, o);
                    b += __shfl_xor_sync(0xffffffffu, b, o);
                    c += __shfl_xor_sync(0xffffffffu, c, o);
                }
        }
    } else {
        // the block's threads share the blocks' partials (fixed order)
        for (unsigned q = threadIdx.x; q < gridDim.x; q += blockDim.x) {
            a += __ldcg(red + q * 3 + 0);
            b += __ldcg(red + q * 3 + 1);
            c += __ldcg(red + q * 3 + 2);
        }
        for (int o = 16; o > 0; o >>= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            b += __shfl_xor_sync(0xffffffffu, b, o);
            c += __shfl_xor_sync(0xffffffffu, c, o);
        }
        if (lane == 0) {
            sred[warp][0] = a;
            sred[warp][1] = b;
            sred[warp][2] = c;
        }
        __syncthreads();
        if (threadIdx.x == 0)
            for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
                a += sred[w][0];
                b += sred[w][1];
                c += sred[w][2];
            }
    }
    if (threadIdx.x == 0) {
        obs_row[0] = a * inv_nk;
        obs_row[1] = b * inv_nk;
        obs_row[2] = c * inv_nk;
        *counter = 0u;
        if (step_to_bump) *step_to_bump = new_step;
    }
}

// One RK4 stage for all k: k_s = -i [diag(eps) + E(t_s).d + dSigma, rho0 + X_s] per k
// (Eq. tdagw with dSigma from Eq. sigma-from-k), accumulated into the classical RK4
// combination; the next stage input X_{s+1} = drho_n + c_{s+1} dt k_s is written directly.
// On the last stage the state is advanced with a compensated (TwoSum) accumulation and
// the observables of the new state are reduced.  One thread per pair element (k, n, m);
// the Nb^2 threads of one k are adjacent lanes of a warp and exchange the Nb x Nb blocks
// by shuffles.
template <typename R, int NB>
__global__ void __launch_bounds__(kStageThreads<R>) stage_kernel(StageParams<R> p) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int64_t nstep = *p.step;
    const int eoff = p.stage == 0 ? 0 : (p.stage == 3 ? 2 : 1);
    const R E = (R)p.Etab[2 * nstep + eoff];
    Obs3 ob{0.0, 0.0, 0.0};
    stage_element<R, NB>(p, i, i < p.N, threadIdx.x & 31, p.stage, E, ob);
    if (p.stage == 3)
        reduce_observables(ob.p, ob.j, ob.o, p.red, p.counter, p.obs + (nstep + 1) * 3,
                           1.0 / (double)p.Nk, p.step, nstep + 1);
}

// Observables of rho0 + X into obs row `row` (used for the initial row of a run).
template <typename R, int NB>
__global__ void __launch_bounds__(kStageThreads<R>)
observables_kernel(const cplx_t<R>* __restrict__ X, const cplx_t<R>* __restrict__ dx,
                   const cplx_t<R>* __restrict__ vx, int64_t N, int Nk, int c1, R o0_, R o1_,
                   R o2_, R o3_, double* red, unsigned* counter, double* obs_row) {
    using C = cplx_t<R>;
    constexpr int NB2 = NB * NB;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int g = (threadIdx.x & 31) % NB2, n = g / NB, m = g % NB;
    const R occ[4] = {o0_, o1_, o2_, o3_};
    double a = 0, b = 0, c = 0;
    if (i < N) {
        C rho = X[i];
        if (n == m) rho.x += occ[n];
        const C d = dx[i], v = vx[i];
        a = (double)rho.x * (double)d.x + (double)rho.y * (double)d.y;
        b = (double)rho.x * (double)v.x + (double)rho.y * (double)v.y;
        c = (n == m && n == c1) ? (double)rho.x : 0.0;
    }
    reduce_observables(a, b, c, red, counter, obs_row, 1.0 / (double)Nk, nullptr, 0);
}

// the k = k' blocks of K: out[(k P + p) P + q] = K[(k P + p) N + k P + q]
template <typename R>
__global__ void gather_kblocks_kernel(const cplx_t<R>* __restrict__ K, int64_t N, int Nk, int P,
                                      cplx_t<R>* __restrict__ out) {
    const int64_t n = (int64_t)Nk * P * P;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t k = e / (P * P), r = e % (P * P);
        const int p = (int)(r / P), q = (int)(r % P);
        out[e] = K[(k * P + p) * N + k * P + q];
    }
}

// y[k P + p] += sum_q B[k][p][q] x[k P + q]: the k-block reading of K^diag x
template <typename R>
__global__ void kblock_add_kernel(const cplx_t<R>* __restrict__ B, const cplx_t<R>* __restrict__ x,
                                  cplx_t<R>* __restrict__ y, int Nk, int P) {
    using C = cplx_t<R>;
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= (int64_t)Nk * P) return;
    const int64_t k = i / P;
    const int p = (int)(i % P);
    const C* b = B + (k * P + p) * P;
    const C* xk = x + k * P;
    C s = y[i];
    for (int q = 0; q < P; ++q) s = cfma(b[q], xk[q], s);
    y[i] = s;
}

}  // namespace

template <typename R>
void launch_gather_kblocks(const Ctx& c, void* dst, cudaStream_t s) {
    const HostModel& h = c.hm;
    gather_kblocks_kernel<R><<<152 * 4, 256, 0, s>>>(c.K.as<cplx_t<R>>(), h.N, h.Nk, h.Nb * h.Nb,
                                                     static_cast<cplx_t<R>*>(dst));
    check_launch("gather_kblocks_kernel");
}

template <typename R>
void launch_kblock_add(const void* B, const void* x, void* y, int Nk, int P, cudaStream_t s) {
    using C = cplx_t<R>;
    const int64_t n = (int64_t)Nk * P;
    kblock_add_kernel<R><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(
        static_cast<const C*>(B), static_cast<const C*>(x), static_cast<C*>(y), Nk, P);
    check_launch("kblock_add_kernel");
}

template <typename R>
void launch_gemv(const void* A, int64_t lda, int64_t nrows, int64_t ncols, const void* x,
                 void* out, cudaStream_t s) {
    using C = cplx_t<R>;
    constexpr int ROWS = 4, THREADS = 256;
    gemv_kernel<R, ROWS, THREADS><<<(unsigned)((nrows + ROWS - 1) / ROWS), THREADS, 0, s>>>(
        static_cast<const C*>(A), lda, nrows, ncols, static_cast<const C*>(x), static_cast<C*>(out));
    check_launch("gemv_kernel");
}

template <typename R>
void launch_vcols(const void* V, int64_t ldv, int64_t N, int r, const void* x, void* part,
                  int nblocks, cudaStream_t s) {
    using C = cplx_t<R>;
    const int64_t rpb = (N + nblocks - 1) / nblocks;
    dim3 grid((unsigned)nblocks, (unsigned)((ldv + 511) / 512));
    vcols_kernel<R><<<grid, 256, 0, s>>>(static_cast<const C*>(V), ldv, N, r,
                                          static_cast<const C*>(x), static_cast<C*>(part), rpb);
    check_launch("vcols_kernel");
}

template <typename R>
void launch_yreduce(const void* part, int nsplit, int r, const void* S, void* ytil,
                    cudaStream_t s) {
    using C = cplx_t<R>;
    const int subs = nsplit <= 4 ? 1 : (nsplit <= 16 ? 4 : kYSubs<R>);
    auto k = subs == 1 ? yreduce_few_kernel<R, 1> : (subs == 4 ? yreduce_few_kernel<R, 4> : yreduce_kernel<R>);
    k<<<(r + kYCols<R> - 1) / kYCols<R>, subs * kYCols<R>, 0, s>>>(static_cast<const C*>(part), nsplit, r,
                                                                 static_cast<const R*>(S), static_cast<C*>(ytil));
    check_launch("yreduce_kernel");
}

template <typename R>
void launch_urows(const void* A, int64_t lda, int64_t nrows, int ncols, const void* x, void* out, const void* diag,
                  const void* xd, cudaStream_t s) {
    using C = cplx_t<R>;
    // one row per warp while that leaves SMs without a block
    const bool few = nrows < 4 * 4 * 152;
    const int64_t rpb = few ? 4 : 16;
    auto k = few ? urows_kernel<R, 1> : urows_kernel<R, 4>;
    k<<<(unsigned)((nrows + rpb - 1) / rpb), 128, 0, s>>>(static_cast<const C*>(A), lda, nrows, ncols,
                                                          static_cast<const C*>(x), static_cast<C*>(out),
                                                          static_cast<const C*>(diag), static_cast<const C*>(xd));
    check_launch("urows_kernel");
}

template <typename R>
void launch_lowrank_apply(const void* U, const void* V, int64_t ld, int64_t N, int r, const void* S, const void* diag,
                          const void* x, void* y, void* part, int nblocks, void* ytil, cudaStream_t s) {
    using C = cplx_t<R>;
    if constexpr (sizeof(R) == 4) {
        if (r <= kClMaxRank && N <= kClMaxN && N * r <= kClMaxElems) {
            lr_cluster_kernel<<<kClCtas, kClThreads, 0, s>>>(
                static_cast<const C*>(U), static_cast<const C*>(V), ld, (int)N, r, static_cast<const R*>(S),
                static_cast<const C*>(diag), static_cast<const C*>(x), static_cast<C*>(y));
            check_launch("lr_cluster_kernel");
            return;
        }
    }
    launch_vcols<R>(V, ld, N, r, x, part, nblocks, s);
    launch_yreduce<R>(part, nblocks, r, S, ytil, s);
    launch_urows<R>(U, ld, N, r, ytil, y, diag, x, s);
}

template <typename R>
void launch_stage(Ctx& c, int stage, double dt, double dirx, double diry, bool kahan,
                  cudaStream_t s) {
    using C = cplx_t<R>;
    StageParams<R> p;
    p.X = c.X.as<C>();
    p.dS = c.dS.as<C>();
    p.dx = c.dx.as<C>();
    p.dy = c.dy.as<C>();
    p.vx = c.vx.as<C>();
    p.gap = c.gap.as<typename GapT<R>::type>();
    p.acc = c.acc.as<C>();
    p.Ssum = c.Ssum.as<C>();
    p.Ccomp = c.Ccomp.as<C>();
    p.Xnext = c.X.as<C>();  // in place: each thread reads X[i] before writing it
    p.Etab = c.Etab.as<double>();
    p.step = c.stepctr.as<int64_t>();
    p.obs = c.obs.as<double>();
    p.red = c.red.as<double>();
    p.counter = c.counter.as<unsigned>();
    p.N = c.hm.N;
    p.Nk = c.hm.Nk;
    p.c1 = c.hm.c1;
    for (int q = 0; q < 4; ++q) p.occ[q] = (R)c.hm.occ[q];
    p.dt = (R)dt;
    p.dirx = (R)dirx;
    p.diry = (R)diry;
    p.stage = stage;
    p.kahan = kahan ? 1 : 0;
    const unsigned blocks = (unsigned)((c.hm.N + kStageThreads<R> - 1) / kStageThreads<R>);
    if (c.hm.Nb == 2) stage_kernel<R, 2><<<blocks, kStageThreads<R>, 0, s>>>(p);
    else stage_kernel<R, 4><<<blocks, kStageThreads<R>, 0, s>>>(p);
    check_launch("stage_kernel");
}

template <typename R>
void launch_observables_row(Ctx& c, const void* X, int64_t row, cudaStream_t s) {
    using C = cplx_t<R>;
    const unsigned blocks = (unsigned)((c.hm.N + kStageThreads<R> - 1) / kStageThreads<R>);
    const HostModel& h = c.hm;
    double* orow = c.obs.as<double>() + row * 3;
    if (h.Nb == 2)
        observables_kernel<R, 2><<<blocks, kStageThreads<R>, 0, s>>>(
            static_cast<const C*>(X), c.dx.as<C>(), c.vx.as<C>(), h.N, h.Nk, h.c1, (R)h.occ[0],
            (R)h.occ[1], (R)h.occ[2], (R)h.occ[3], c.red.as<double>(), c.counter.as<unsigned>(), orow);
    else
        observables_kernel<R, 4><<<blocks, kStageThreads<R>, 0, s>>>(
            static_cast<const C*>(X), c.dx.as<C>(), c.vx.as<C>(), h.N, h.Nk, h.c1, (R)h.occ[0],
            (R)h.occ[1], (R)h.occ[2], (R)h.occ[3], c.red.as<double>(), c.counter.as<unsigned>(), orow);
    check_launch("observables_kernel");
}

#define INST(R)                                                                            \
    template void launch_gemv<R>(const void*, int64_t, int64_t, int64_t, const void*, void*, cudaStream_t); \
    template void launch_yreduce<R>(const void*, int, int, const void*, void*, cudaStream_t); \
    template void launch_vcols<R>(const void*, int64_t, int64_t, int, const void*, void*, int, \
                                  cudaStream_t);                                          \
    template void launch_lowrank_apply<R>(const void*, const void*, int64_t, int64_t, int, const void*, const void*, \
                                          const void*, void*, void*, int, void*, cudaStream_t); \
    template void launch_stage<R>(Ctx&, int, double, double, double, bool, cudaStream_t);   \
    template void launch_observables_row<R>(Ctx&, const void*, int64_t, cudaStream_t);
INST(float)
INST(double)
template void launch_gather_kblocks<float>(const Ctx&, void*, cudaStream_t);
template void launch_gather_kblocks<double>(const Ctx&, void*, cudaStream_t);
template void launch_kblock_add<float>(const void*, const void*, void*, int, int, cudaStream_t);
template void launch_kblock_add<double>(const void*, const void*, void*, int, int, cudaStream_t);
#undef INST

}  // namespace tdagw
