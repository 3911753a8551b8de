// High-harmonic spectrum of recorded currents (Sec. "SVD acceleration of TD-aGW"):
//   HHG_b(w) = | w sum_{n=0..T_b} J_b(t_n) e^{-i w t_n} dt |^2,   t_n = n dt,
// for B trajectories (an angle or frequency sweep) at nfreq angular frequencies, FP64
// throughout.
//
// Bound by the FP64 pipes (two FMAs per sample, frequency and trajectory cannot be avoided;
// this GPU does about two per SM and clock).  A thread takes one frequency and TB trajectories,
// so that the phasor e^{-i w t_n} is advanced once for all of them: 2 + 4 / TB operations per
// sample instead of 6.  A block takes chunks of at most kHhgChunk samples, staged in shared
// memory (zero past a trajectory's end), with the phasor computed exactly at each chunk's start,
// so rounding does not accumulate over long runs; a second kernel adds the blocks' sums along
// time in order.  60 trajectories x 2001 steps x 512 frequencies, whole call with its copies:
// 1.11 -> 0.56 ms; one trajectory x 201 steps x 33 frequencies 0.22 -> 0.17 ms.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "hhg_plan.h"

namespace tdagw {

namespace {

// part[(z nfreq + f) B + b]: the sum over the samples of block z's cpb chunks; with one block
// along z the spectrum itself goes to out
template <int TB>
__global__ void __launch_bounds__(kHhgThreads)
hhg_kernel(const double* __restrict__ J, int64_t stride, int B, const int* __restrict__ steps, double dt,
           const double* __restrict__ omega, int nfreq, int clen, int cpb, double2* __restrict__ part, double* __restrict__ out) {
    __shared__ double js[kHhgChunk][TB];
    const int b0 = blockIdx.y * TB;
    const int f = blockIdx.x * kHhgThreads + threadIdx.x;
    int tmax = -1;  // last sample of this block's trajectories
#pragma unroll
    for (int u = 0; u < TB; ++u)
        if (b0 + u < B) tmax = max(tmax, steps[b0 + u]);
    const double w = f < nfreq ? omega[f] : 0.0;
    double sdt, cdt;
    sincos(w * dt, &sdt, &cdt);
    double re[TB], im[TB];
#pragma unroll
    for (int u = 0; u < TB; ++u) re[u] = im[u] = 0.0;
    for (int c = 0; c < cpb; ++c) {
        const int64_t n0 = ((int64_t)blockIdx.z * cpb + c) * clen;
        const int cnt = (int)min((int64_t)clen, (int64_t)tmax + 1 - n0);
        if (cnt <= 0) break;
        __syncthreads();
        for (int e = threadIdx.x; e < cnt * TB; e += kHhgThreads) {
            const int u = e % TB, b = b0 + u;
            const int64_t n = n0 + e / TB;
            js[e / TB][u] = b < B && n <= steps[b] ? J[(n * B + b) * stride] : 0.0;
        }
        __syncthreads();
        double s0, c0;
        sincos(w * ((double)n0 * dt), &s0, &c0);
        double cr = c0, ci = -s0;  // e^{-i w t_n}
        for (int e = 0; e < cnt; ++e) {
#pragma unroll
            for (int u = 0; u < TB; ++u) {
                re[u] = fma(js[e][u], cr, re[u]);
                im[u] = fma(js[e][u], ci, im[u]);
            }
            const double nr = cr * cdt + ci * sdt;  // times e^{-i w dt}
            const double ni = ci * cdt - cr * sdt;
            cr = nr;
            ci = ni;
        }
    }
    if (f >= nfreq) return;
    const double a = w * dt;
#pragma unroll
    for (int u = 0; u < TB; ++u)
        if (b0 + u < B) {
            if (gridDim.z == 1) out[(int64_t)f * B + b0 + u] = a * a * (re[u] * re[u] + im[u] * im[u]);
            else part[((int64_t)blockIdx.z * nfreq + f) * B + b0 + u] = make_double2(re[u], im[u]);
        }
}

__global__ void __launch_bounds__(kHhgThreads)
hhg_power_kernel(const double2* __restrict__ part, int nchunk, double dt, const double* __restrict__ omega, int nfreq,
                 int B, double* __restrict__ out) {
    const int64_t e = blockIdx.x * (int64_t)kHhgThreads + threadIdx.x;
    if (e >= (int64_t)nfreq * B) return;
    double re = 0.0, im = 0.0;
    for (int c = 0; c < nchunk; ++c) {
        const double2 p = part[(int64_t)c * nfreq * B + e];
        re += p.x;
        im += p.y;
    }
    const double a = omega[e / B] * dt;
    out[e] = a * a * (re * re + im * im);
}

}  // namespace

void hhg_spectrum(const double* J, int64_t rows, int64_t stride, int B, const int* steps, double dt,
                  const double* omega, int nfreq, double* out, cudaStream_t s) {
    int tmax = 0;
    for (int b = 0; b < B; ++b) tmax = std::max(tmax, steps[b]);
    TDAGW_REQUIRE(rows >= (int64_t)tmax + 1, TDAGW_ERR_INVALID_ARG, "fewer rows than steps + 1");
    // the rows used (the last element read is (tmax B + B - 1) stride)
    const size_t nJ = (((size_t)tmax + 1) * B - 1) * stride + 1;
    const HhgPlan pl = hhg_plan(tmax, B, nfreq);
    const int64_t per = (int64_t)nfreq * B;
    const int nz = pl.nz;
    // one allocation: the partial sums, the result, omega, J, the step counts
    const size_t nO = (size_t)per, nP = nz > 1 ? 2 * nO * nz : 0;
    DevBuf buf;
    buf.ensure((nP + nO + (size_t)nfreq + nJ) * sizeof(double) + (size_t)B * sizeof(int));
    double2* dP = buf.as<double2>();
    double *dO = buf.as<double>() + nP, *dW = dO + nO, *dJ = dW + nfreq;
    int* dS = reinterpret_cast<int*>(dJ + nJ);
    TDAGW_CUDA(cudaMemcpyAsync(dJ, J, nJ * sizeof(double), cudaMemcpyHostToDevice, s));
    TDAGW_CUDA(cudaMemcpyAsync(dS, steps, (size_t)B * sizeof(int), cudaMemcpyHostToDevice, s));
    TDAGW_CUDA(cudaMemcpyAsync(dW, omega, (size_t)nfreq * sizeof(double), cudaMemcpyHostToDevice, s));
    const dim3 grid((unsigned)pl.gx, (unsigned)pl.gy, (unsigned)nz);
    auto kern = pl.tb == 8 ? hhg_kernel<8> : (pl.tb == 4 ? hhg_kernel<4> : hhg_kernel<1>);
    kern<<<grid, kHhgThreads, 0, s>>>(dJ, stride, B, dS, dt, dW, nfreq, pl.clen, pl.cpb, dP, dO);
    check_launch("hhg_kernel");
    if (nz > 1) {
        hhg_power_kernel<<<(unsigned)((per + kHhgThreads - 1) / kHhgThreads), kHhgThreads, 0, s>>>(dP, nz, dt, dW, nfreq,
                                                                                                  B, dO);
        check_launch("hhg_power_kernel");
    }
    TDAGW_CUDA(cudaMemcpyAsync(out, dO, nO * sizeof(double), cudaMemcpyDeviceToHost, s));
    TDAGW_CUDA(cudaStreamSynchronize(s));
}

}  // namespace tdagw
