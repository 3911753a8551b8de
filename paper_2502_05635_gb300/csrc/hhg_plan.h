// Launch geometry of the HHG spectra (hhg.cu): host arithmetic only, without CUDA headers, so
// that it can be checked on its own for runs that are too long to execute.
#pragma once

#include <algorithm>
#include <cstdint>

namespace tdagw {

constexpr int kHhgThreads = 128, kHhgChunk = 256;
constexpr int kHhgMaxZ = 65535;  // the largest z extent of a grid

struct HhgPlan {
    int tb;         // trajectories per thread
    int clen, cpb;  // samples per chunk, consecutive chunks per block
    int gx, gy, nz; // blocks along frequencies, trajectory groups and time
};

// Geometry for B trajectories of at most tmax steps (tmax + 1 samples) at nfreq frequencies.
inline HhgPlan hhg_plan(int tmax, int B, int nfreq) {
    HhgPlan p;
    // trajectories per thread, and chunks short enough to fill the GPU (a short run of a few
    // trajectories is bound by the length of one thread's chain, not by the pipes)
    p.tb = B >= 8 ? 8 : (B >= 4 ? 4 : 1);
    p.gx = (nfreq + kHhgThreads - 1) / kHhgThreads;
    p.gy = (B + p.tb - 1) / p.tb;
    const int64_t per = (int64_t)nfreq * B;
    const int64_t blocks = (int64_t)p.gx * p.gy;
    p.clen = kHhgChunk;
    while (p.clen > 32 && blocks * (tmax / p.clen + 1) < 2 * 152) p.clen /= 2;
    // blocks along time: one per chunk while the partial sums stay below 64 MB and the grid
    // within its limit (from 65535 chunks on, 16776960 samples, a block takes several chunks)
    const int nchunk = tmax / p.clen + 1;
    const int64_t most = std::min<int64_t>({nchunk, (int64_t)(1 << 22) / per, kHhgMaxZ});
    const int want = (int)std::max<int64_t>(1, most);
    p.cpb = (nchunk + want - 1) / want;
    p.nz = (nchunk + p.cpb - 1) / p.cpb;
    return p;
}

}  // namespace tdagw
