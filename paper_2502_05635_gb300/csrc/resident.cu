// Persistent single-trajectory propagation with the kernel resident in shared memory
// (complex64, small models): one cooperative launch runs all RK4 steps of a call (Eq. tdagw,
// dSigma from Eq. sigma-from-k or Eq. svd_acc).  Each CTA holds the rows of K (dense), or of U
// and V (low rank), of its k-points in shared memory for the whole launch, and the state of its
// rows in registers (one pair element per thread), so that a stage reads nothing but what the
// CTAs exchange:
//
//   dense     the stage input X (N complex):  write own rows; barrier; read all; K rows . X
//   low rank  the partial vectors of V^H x:   write own; barrier; every CTA adds all of them
//             (G x rank, fixed order), scales by S and multiplies its rows of U
//   then the commutator, the RK4 stage update and the observables in registers.
//
// The smallest models fit in one cluster of up to 16 CTAs: the exchange then goes through
// distributed shared memory (every CTA writes its part into the others') and the cluster's
// hardware barrier instead of L2 and a counter.
//
// Bound by the one barrier per stage and the exchange around it.  The stage-wise
// path of the dense kernel takes two launches per stage; the streaming low-rank kernel
// (lr_persistent.cu) two barriers, and its state goes through L2.  The exchange buffers
// alternate by stage parity: a CTA writes the next stage's while a slower one still reads.
// The grid form's waits are bounded as in the other persistent kernels (the timeout hook tests them
// in its low-rank form).  The cluster form waits at the hardware's cluster barrier, which has no
// budget: its CTAs are scheduled together, and none leaves before its last barrier.
//
// Measured per stage: dense, N = 576 6.1 us (stage-wise) -> 3.6 (grid) -> 2.7 (cluster); low
// rank, N = 2116, rank 235 9.3 us (streaming kernel) -> 5.6 (grid).
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "persist.cuh"
#include "stage.cuh"

namespace tdagw {

namespace {

using namespace persist;
namespace cg = cooperative_groups;

constexpr int kClMax = 16;  // CTAs of a cluster (above 8: opt-in)
constexpr int kRThreads = 512, kRWarps = kRThreads / 32;
constexpr size_t kRSmem = 224 * 1024;  // dynamic shared memory at most

struct ResArgs {
    const float2* A;      // dense: K (N x N); low rank: U (N x ld)
    const float2* V;      // low rank: V (N x ld)
    const float* S;
    const float2* diag;
    const float2* dx;
    const float2* dy;
    const float2* vx;
    const float2* gap;
    float2* X;            // state, read at the start and written at the end
    float2* Ssum;
    float2* Ccomp;
    const double* Etab;
    double* obs;          // (T + 1) x 3
    double* red;          // G x 3
    float2* xch;          // exchange: 2 x N (dense) or 2 x G x ld (low rank)
    unsigned long long* bar_count;
    int* err;
    int64_t ld;           // row length of A and V (complex)
    int N, Nk, r, T, kahan, c1, rows_max;
    float occ[4];
    float dt, dirx, diry;
    int extra_arrivals;
    unsigned long long wait_ns;
};

// 16-byte asynchronous copies of n complex (even) from global to shared memory
__device__ __forceinline__ void load_rows(float2* dst, const float2* src, int64_t n) {
    for (int64_t e = 2 * threadIdx.x; e < n; e += 2 * kRThreads)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(saddr(dst + e)), "l"(src + e) : "memory");
}

// out[row] = sum_c A[row][c] v[c] for this CTA's rows, A and v in shared memory.  A warp takes
// W rows of one column part at a time; with few rows per warp the columns are split over
// `parts` warps, whose dots are added by the reader (dots: parts x rows_max).
template <int W>
__device__ __forceinline__ void row_pass(const float2* A, int ld, int nrows, int rows_max, int parts, const float2* v,
                                         float2* dots, int warp, int lane) {
    const int part = warp % parts, wr = warp / parts, nw = kRWarps / parts;
    const int pw = ((ld + parts - 1) / parts + 1) & ~1;
    const int c0 = part * pw, c1 = min(ld, c0 + pw);
    for (int r0 = wr * W; r0 < nrows; r0 += nw * W) {
        float2 acc[W];
#pragma unroll
        for (int w = 0; w < W; ++w) acc[w] = make_float2(0.f, 0.f);
        for (int c = c0 + 2 * lane; c < c1; c += 64) {
            const float4 xv = *reinterpret_cast<const float4*>(v + c);
#pragma unroll
            for (int w = 0; w < W; ++w) {
                const float4 a = *reinterpret_cast<const float4*>(A + (r0 + (r0 + w < nrows ? w : 0)) * ld + c);
                acc[w] = cfma(make_float2(a.x, a.y), make_float2(xv.x, xv.y), acc[w]);
                acc[w] = cfma(make_float2(a.z, a.w), make_float2(xv.z, xv.w), acc[w]);
            }
        }
        // sums over the lanes: W rows are halved between the lane halves first
        int o = 16;
#pragma unroll
        for (int h = W; h > 1; h >>= 1, o >>= 1) {
            const bool up = lane & o;
#pragma unroll
            for (int q = 0; q < h / 2; ++q) {
                const float2 keep = up ? acc[q + h / 2] : acc[q], send = up ? acc[q] : acc[q + h / 2];
                acc[q] = cadd(keep, shfl_xor(send, o));
            }
        }
        float2 s = acc[0];
#pragma unroll
        for (; o > 0; o >>= 1) s = cadd(s, shfl_xor(s, o));
        const int row = r0 + lane / (32 / W);
        if (lane % (32 / W) == 0 && row < nrows) dots[part * rows_max + row] = s;
    }
}

// CL: the grid is one cluster
template <int NB, bool LR, bool CL>
__global__ void __launch_bounds__(kRThreads, 1) resident_kernel(ResArgs a) {
    extern __shared__ __align__(128) unsigned char smem[];
    constexpr int P = NB * NB;
    const int G = gridDim.x, cta = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ka = (int)((int64_t)cta * a.Nk / G), kb = (int)((int64_t)(cta + 1) * a.Nk / G);
    const int ra = ka * P, nrows = (kb - ka) * P, ld = (int)a.ld;
    const int nv = LR ? ld : a.N;  // length of the exchanged vector (N is even: Nb^2 a multiple of 4)

    float2* As = reinterpret_cast<float2*>(smem);               // rows_max x ld
    float2* Vs = As + (int64_t)a.rows_max * ld;                 // low rank: rows_max x ld
    float2* vec = Vs + (LR ? (int64_t)a.rows_max * ld : 0);     // S o y, or X (cluster: two X, by parity)
    float2* pcl = vec + (CL && !LR ? 2 : 1) * nv;               // cluster, low rank: 2 x G partial vectors
    float2* xs = pcl + (CL && LR ? 2 * (int64_t)G * ld : 0);    // own stage input (low rank)
    float2* dots = xs + a.rows_max;                             // parts x rows_max
    float2* sub = dots + kRWarps * a.rows_max;                  // low rank: 2 x kRThreads partial sums
    __shared__ float wf[6 * kRWarps];
    __shared__ int abort_flag;
    volatile int* abort_s = &abort_flag;

    if (tid == 0) abort_flag = 0;
    load_rows(As, a.A + (int64_t)ra * ld, (int64_t)nrows * ld);
    if (LR) load_rows(Vs, a.V + (int64_t)ra * ld, (int64_t)nrows * ld);
    __shared__ double cobs[2][kClMax][3];  // cluster: the CTAs' observables, in the last CTA

    // this thread's pair element (nrows <= kRThreads)
    const bool act = tid < nrows;
    const int i = ra + (act ? tid : 0);
    const int base = lane - lane % P, n_ = (lane % P) / NB, m_ = lane % NB;
    const float2 zero = make_float2(0.f, 0.f);
    float2 X = act ? a.X[i] : zero, Ss = act ? a.Ssum[i] : zero, Cc = act ? a.Ccomp[i] : zero, acc = zero;
    const float2 d1 = act ? a.dx[i] : zero, d2 = act ? a.dy[i] : zero, v1 = act ? a.vx[i] : zero;
    const float2 gp = act ? a.gap[i] : zero, dg = LR && act ? a.diag[i] : zero;
    const float2 D = make_float2(a.dirx * d1.x + a.diry * d2.x, a.dirx * d1.y + a.diry * d2.y);
    const float fmn = a.occ[m_] - a.occ[n_];
    // observables of rho0 + X: per-warp double-float sums, then the CTA's sum (after a barrier)
    auto warp_observables = [&]() {
        ObsDF ob;
        if (act) {
            const float2 rho = n_ == m_ ? cadd(X, make_float2(a.occ[n_], 0.f)) : X;
            ob.p.add_prod(rho.x, d1.x);
            ob.p.add_prod(rho.y, d1.y);
            ob.j.add_prod(rho.x, v1.x);
            ob.j.add_prod(rho.y, v1.y);
            if (n_ == m_ && n_ == a.c1) ob.o.add(rho.x);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ob.p = ob.p.shfl_xor_sum(o);
            ob.j = ob.j.shfl_xor_sum(o);
            ob.o = ob.o.shfl_xor_sum(o);
        }
        if (lane == 0) {
            wf[6 * warp] = ob.p.hi;
            wf[6 * warp + 1] = ob.p.lo;
            wf[6 * warp + 2] = ob.j.hi;
            wf[6 * warp + 3] = ob.j.lo;
            wf[6 * warp + 4] = ob.o.hi;
            wf[6 * warp + 5] = ob.o.lo;
        }
    };
    int opar = 0;
    auto publish_observables = [&]() {
        if (tid >= 3) return;
        DF s;
        for (int w = 0; w < (nrows + 31) / 32; ++w) {
            DF t;
            t.hi = wf[6 * w + 2 * tid];
            t.lo = wf[6 * w + 2 * tid + 1];
            s.add(t);
        }
        // (alternating by step in the cluster: the last CTA may still read the previous one)
        if (CL) cg::this_cluster().map_shared_rank(&cobs[opar][cta][tid], G - 1)[0] = s.value();
        else __stcg(a.red + 3 * cta + tid, s.value());
    };
    // row `row` of the observables from the CTAs' sums (one warp of the last CTA, fixed order)
    auto write_observables = [&](int64_t row) {
        if (!CL) {
            reduce_obs_row(a.red, G, 1.0 / (double)a.Nk, a.obs + 3 * row, lane);
        } else if (lane < 3) {
            double s = 0.0;
            for (int c = 0; c < G; ++c) s += cobs[opar][c][lane];
            a.obs[3 * row + lane] = s * (1.0 / (double)a.Nk);
        }
    };
    if (act) xs[tid] = X;
    warp_observables();  // row 0, by the same sums as every other row (a resumed run repeats it)
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if (CL) cg::this_cluster().sync();  // every CTA runs: its shared memory may be written
    publish_observables();

    // column parts of the row pass: as many as the groups of four rows leave warps for
    int parts = 1;
    while (2 * parts * ((nrows + 3) / 4) <= kRWarps) parts *= 2;
    unsigned lgen = 0;
    for (int gs = 0; gs < 4 * a.T; ++gs) {
        const int n = gs >> 2, st = gs & 3, par = gs & 1;
        const float E = (float)__ldg(a.Etab + 2 * (int64_t)n + (st == 0 ? 0 : (st == 3 ? 2 : 1)));
        if (LR) {
            // ---- V pass: thread = (column pair, subset of the rows); no more subsets than rows
            // (below, than CTAs): their sums are added one after the other, and a low rank would
            // make up to 512 of them, nearly all empty (N = 2116, rank 1: 9.6 -> 4.4 us / stage)
            const int ncp = ld / 2, nsub = min(kRThreads / ncp, nrows), cp = tid % ncp, sb = tid / ncp;
            float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
            if (sb < nsub) {
                float2 y0 = zero, y1 = zero;
                for (int row = sb; row < nrows; row += nsub) {
                    const float4 v = *reinterpret_cast<const float4*>(Vs + (int64_t)row * ld + 2 * cp);
                    y0 = cfmac(make_float2(v.x, v.y), xs[row], y0);
                    y1 = cfmac(make_float2(v.z, v.w), xs[row], y1);
                }
                s = make_float4(y0.x, y0.y, y1.x, y1.y);
            }
            if (nsub > 1) {
                if (sb < nsub) reinterpret_cast<float4*>(sub)[tid] = s;
                __syncthreads();
                if (tid < ncp)
                    for (int u = 1; u < nsub; ++u) {
                        const float4 t = reinterpret_cast<const float4*>(sub)[u * ncp + tid];
                        s.x += t.x;
                        s.y += t.y;
                        s.z += t.z;
                        s.w += t.w;
                    }
            }
            const int64_t off = ((int64_t)par * G + cta) * ld + 2 * tid;
            if (tid < ncp) {
                if (CL)
                    for (int c = 0; c < G; ++c)
                        *reinterpret_cast<float4*>(cg::this_cluster().map_shared_rank(pcl + off, c)) = s;
                else
                    __stcg(reinterpret_cast<float4*>(a.xch + off), s);
            }
        } else if (act) {
            if (CL)
                for (int c = 0; c < G; ++c) *cg::this_cluster().map_shared_rank(vec + (int64_t)par * nv + i, c) = X;
            else
                __stcg(a.xch + (int64_t)par * a.N + i, X);
        }
        if (CL) cg::this_cluster().sync();
        else if (!grid_sync<kRThreads>(a.bar_count, a.err, a.extra_arrivals, a.wait_ns, lgen, abort_s)) return;
        // observables after the previous step, or of the start (published before this barrier)
        if (st == 0 && cta == G - 1 && warp == kRWarps - 1) write_observables(n);
        if (LR) {
            // ---- S o sum of all partial vectors: thread = (column pair, subset of the CTAs)
            const int ncp = ld / 2, nsub = min(kRThreads / ncp, G), cp = tid % ncp, sb = tid / ncp;
            float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4* src = reinterpret_cast<const float4*>((CL ? pcl : a.xch) + (int64_t)par * G * ld) + cp;
            if (sb < nsub) {
#pragma unroll 8
                for (int c = sb; c < G; c += nsub) {
                    const float4 t = CL ? src[(int64_t)c * ncp] : __ldcg(src + (int64_t)c * ncp);
                    s.x += t.x;
                    s.y += t.y;
                    s.z += t.z;
                    s.w += t.w;
                }
                reinterpret_cast<float4*>(sub)[tid] = s;
            }
            __syncthreads();
            if (tid < ncp) {
                for (int u = 1; u < nsub; ++u) {
                    const float4 t = reinterpret_cast<const float4*>(sub)[u * ncp + tid];
                    s.x += t.x;
                    s.y += t.y;
                    s.z += t.z;
                    s.w += t.w;
                }
                const float s0 = a.S[2 * tid], s1 = 2 * tid + 1 < a.r ? a.S[2 * tid + 1] : 0.f;
                reinterpret_cast<float4*>(vec)[tid] = make_float4(s.x * s0, s.y * s0, s.z * s1, s.w * s1);
            }
        } else if (!CL) {
            for (int e = 2 * tid; e < a.N; e += 2 * kRThreads)
                *reinterpret_cast<float4*>(vec + e) =
                    __ldcg(reinterpret_cast<const float4*>(a.xch + (int64_t)par * a.N + e));
        }
        if (LR || !CL) __syncthreads();
        row_pass<4>(As, ld, nrows, a.rows_max, parts, vec + (CL && !LR ? (int64_t)par * nv : 0), dots, warp, lane);
        __syncthreads();
        // ---- commutator and RK4 stage update (the arithmetic of stage_element)
        float2 dS = act ? dots[tid] : zero;
        if (act)
            for (int p = 1; p < parts; ++p) dS = cadd(dS, dots[p * a.rows_max + tid]);
        if (LR) dS = cfma(dg, X, dS);
        const float2 M = cadd(dS, make_float2(E * D.x, E * D.y));
        float2 comm = cscale(M, fmn);
#pragma unroll
        for (int l = 0; l < NB; ++l) {
            const float2 Mnl = shfl(M, base + n_ * NB + l);
            const float2 Xlm = shfl(X, base + l * NB + m_);
            const float2 Xnl = shfl(X, base + n_ * NB + l);
            const float2 Mlm = shfl(M, base + l * NB + m_);
            comm = cfma(Mnl, Xlm, comm);
            comm = csub(comm, cmul(Xnl, Mlm));
        }
        const float2 sv = cadd(gap_times(gp, X), comm);
        const float2 kv = make_float2(sv.y, -sv.x);
        if (st < 3) {
            acc = st == 0 ? kv : cadd(acc, cscale(kv, 2.f));
            const float cn = st == 2 ? a.dt : 0.5f * a.dt;
            X = cadd(Ss, cadd(Cc, cscale(kv, cn)));
        } else {
            const float2 inc = cscale(cadd(acc, kv), a.dt / 6.f);
            if (a.kahan) {
                float ex, ey;
                Ss = make_float2(two_sum(Ss.x, inc.x, ex), two_sum(Ss.y, inc.y, ey));
                Cc = make_float2(Cc.x + ex, Cc.y + ey);
            } else {
                Ss = cadd(Ss, inc);
            }
            X = cadd(Ss, Cc);
            warp_observables();
        }
        if (LR && act) xs[tid] = X;
        __syncthreads();
        if (st == 3) {
            opar ^= 1;
            publish_observables();
        }
    }
    if (act) {
        a.X[i] = X;
        a.Ssum[i] = Ss;
        a.Ccomp[i] = Cc;
    }
    // observables of the last step (cluster: no CTA leaves while another writes its memory)
    if (CL) cg::this_cluster().sync();
    else if (!grid_sync<kRThreads>(a.bar_count, a.err, a.extra_arrivals, a.wait_ns, lgen, abort_s)) return;
    if (cta == G - 1 && warp == 0) write_observables(a.T);
}

}  // namespace

bool launch_resident(Ctx& c, int mode, int T, double dt, double dirx, double diry, bool kahan, bool test_timeout,
                     cudaStream_t s) {
    const HostModel& h = c.hm;
    const bool lr = mode == TDAGW_LOWRANK;
    const int P = h.Nb * h.Nb;
    if (c.dtype != TDAGW_C64 || (lr && (c.kdiag || c.rank < 1))) return false;
    const int64_t N = h.N, ld = lr ? c.rank + (c.rank & 1) : N;
    if (lr && ld > 2 * kRThreads) return false;
    // up to 256 elements dense runs stay with the stage kernels: one block of theirs holds the whole
    // state, and its FP64 sums of an undisturbed state give the exact zero that the tests hold at
    // N = 256, where the double-float sums of several CTAs may leave 1e-17; the timeout hook is for
    // the low-rank and channel-wise kernels, dense runs complete with it
    if (!lr && (N <= 256 || test_timeout)) return false;
    int dev = 0, nsm = 0, smem_max = 0, coop = 0;
    TDAGW_CUDA(cudaGetDevice(&dev));
    TDAGW_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    TDAGW_CUDA(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    TDAGW_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
    if (!coop) return false;
    const size_t cap = std::min(kRSmem, (size_t)smem_max - 4096);
    auto smem_for = [&](int rows, int gcl) {  // gcl: CTAs of the cluster, 0: grid
        const int64_t vecs = lr ? ld + 2 * gcl * ld : (gcl ? 2 : 1) * N;
        return (size_t)((lr ? 2 : 1) * (int64_t)rows * ld + vecs + rows + (int64_t)kRWarps * rows +
                        (lr ? 2 * kRThreads : 0)) * sizeof(float2);
    };
    auto rows_of = [&](int g) { return (h.Nk + g - 1) / g * P; };
    auto kernel = [&](bool cl) -> const void* {
        if (h.Nb == 2) {
            if (lr) return cl ? (const void*)resident_kernel<2, true, true> : (const void*)resident_kernel<2, true, false>;
            return cl ? (const void*)resident_kernel<2, false, true> : (const void*)resident_kernel<2, false, false>;
        }
        if (lr) return cl ? (const void*)resident_kernel<4, true, true> : (const void*)resident_kernel<4, true, false>;
        return cl ? (const void*)resident_kernel<4, false, true> : (const void*)resident_kernel<4, false, false>;
    };
    // one cluster when the kernel fits in it (and the device has room for such a cluster); the
    // bounded waits of the timeout test are those of the grid
    int G = 1;
    while (2 * G <= std::min(kClMax, h.Nk)) G *= 2;
    bool cl = !test_timeout && rows_of(G) <= kRThreads && smem_for(rows_of(G), G) <= cap;
    cudaLaunchAttribute attr{};
    cudaLaunchConfig_t cfg{};
    if (cl) {
        const void* fn = kernel(true);
        const size_t sm = smem_for(rows_of(G), G);
        // the same limit for every model: a launch by another thread must not find it lowered
        TDAGW_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap));
        TDAGW_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        attr.id = cudaLaunchAttributeClusterDimension;
        attr.val.clusterDim.x = (unsigned)G;
        attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
        cfg.gridDim = dim3(G);
        cfg.blockDim = dim3(kRThreads);
        cfg.dynamicSmemBytes = sm;
        cfg.stream = s;
        cfg.attrs = &attr;
        cfg.numAttrs = 1;
        int ncl = 0;
        if (cudaOccupancyMaxActiveClusters(&ncl, fn, &cfg) != cudaSuccess) {
            (void)cudaGetLastError();
            ncl = 0;
        }
        cl = ncl >= 1;
    }
    if (!cl) {
        // k-points per CTA: low rank about sqrt(N) CTAs (a CTA reads its share of the factors
        // and one partial vector per CTA: 2 N / G + G rows, least at G = sqrt(N)), more where their
        // shares do not fit; dense eight rows.  Whatever fits is taken: up to 152 partial vectors of
        // 500 columns cost less than streaming the factors and a second barrier (us / stage streamed
        // and on chip: N = 2116 rank 400 9.9 and 6.7, rank 500 10.4 and 8.6; N = 3600 rank 511 10.6 and 10.1; N = 5184
        // rank 290 12.8 and 8.5; four bands, N = 4624 rank 400 12.2 and 9.0, N = 9216 rank 190 12.0 and 7.9)
        const int Gw = lr ? (int)std::lround(std::sqrt((double)N)) : (int)((N + 7) / 8);
        G = std::max(1, std::min({Gw, nsm, h.Nk}));
        while (G < std::min(nsm, h.Nk) && (rows_of(G) > kRThreads || smem_for(rows_of(G), 0) > cap)) ++G;
        if (rows_of(G) > kRThreads || smem_for(rows_of(G), 0) > cap) return false;
    }
    const int rows_max = rows_of(G);

    ResArgs a{};
    a.A = lr ? c.U.as<float2>() : c.K.as<float2>();
    a.V = lr ? c.V.as<float2>() : nullptr;
    a.S = lr ? c.S.as<float>() : nullptr;
    a.diag = lr ? c.diagF.as<float2>() : nullptr;
    a.dx = c.dx.as<float2>();
    a.dy = c.dy.as<float2>();
    a.vx = c.vx.as<float2>();
    a.gap = c.gap.as<float2>();
    a.X = c.X.as<float2>();
    a.Ssum = c.Ssum.as<float2>();
    a.Ccomp = c.Ccomp.as<float2>();
    a.Etab = c.Etab.as<double>();
    a.obs = c.obs.as<double>();
    c.red.ensure((size_t)std::max<int64_t>(G, (N + 31) / 32) * 3 * sizeof(double));
    a.red = c.red.as<double>();
    c.pbuf.ensure(2 * (size_t)(lr ? G * ld : N) * sizeof(float2));
    a.xch = c.pbuf.as<float2>();
    c.sync.ensure(4 * sizeof(unsigned));
    TDAGW_CUDA(cudaMemsetAsync(c.sync.p, 0, 4 * sizeof(unsigned), s));
    a.bar_count = reinterpret_cast<unsigned long long*>(c.sync.p);
    a.err = reinterpret_cast<int*>(c.sync.as<unsigned>() + 2);
    a.ld = ld;
    a.N = (int)N;
    a.Nk = h.Nk;
    a.r = lr ? c.rank : 0;
    a.T = T;
    a.kahan = kahan ? 1 : 0;
    a.c1 = h.c1;
    a.rows_max = rows_max;
    for (int q = 0; q < 4; ++q) a.occ[q] = (float)h.occ[q];
    a.dt = (float)dt;
    a.dirx = (float)dirx;
    a.diry = (float)diry;
    a.extra_arrivals = test_timeout ? 1 : 0;
    a.wait_ns = test_timeout ? 20000000ull : 2000000000ull;
    void* args[] = {&a};
    const void* fn = kernel(cl);
    if (cl) {
        TDAGW_CUDA(cudaLaunchKernelExC(&cfg, fn, args));
    } else {
        const size_t smem = smem_for(rows_max, 0);
        TDAGW_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cap));
        int per_sm = 0;
        TDAGW_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kRThreads, smem));
        if (per_sm < 1) return false;
        TDAGW_CUDA(cudaLaunchCooperativeKernel(fn, dim3(G), dim3(kRThreads), args, smem, s));
    }
    c.persistent_launched = true;
    return true;
}

}  // namespace tdagw
