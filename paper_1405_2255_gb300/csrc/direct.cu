// direct.cu -- direct summation of eq. (1) (and f_b of eq. 6) on the GPU in FP64:
// the truth generator for large N and the "GPU FP64 direct summation" baseline.
#include <cooperative_groups.h>

#include "kernels.cuh"

namespace gb3 {

// What bounds it: the FP64 pipe, at 18 operations a pair (3 differences, 3 for r^2, 5 in
// rsqrt(), 7 for the sums) and 2 lanes a cycle and SM; an instruction costs the same however many
// of its lanes are active, and four warps saturate an SM.  So the sinks times the slices of the
// sources have to fill every SM evenly: a block takes S <= 32 sinks and one of CL slices of the
// sources, each of its warps a part of that slice, and the 32 / S replicas of a sink within a warp
// take its sources in turn.  The CL blocks of one sink group are a cluster and add their sums
// through distributed shared memory, so the call needs no scratch in global memory.
// 4096 sinks of 3e5 particles: 200.7 ms with one thread per sink and all sources (32 blocks of 128
// on 152 SMs), 44.1 ms so (27.9e9 pairs/s, 0.95 of the pipe's 0.528e12 operations/s).
constexpr int kDirWarps = 8;
constexpr int kDirThreads = 32 * kDirWarps;

// r2 > 0 and not NaN, by its bits (a comparison of doubles takes the FP64 pipe)
__device__ __forceinline__ bool positive_bits(double r2) {
    return (unsigned long long)__double_as_longlong(r2) - 1ull < 0x7ff0000000000000ull;
}

template <bool WANT_F>
__global__ void __launch_bounds__(kDirThreads) k_direct(const double* __restrict__ x, const double* __restrict__ mu,
                                                        int n, double G, const int64_t* __restrict__ sinks,
                                                        int nsinks, int S, int CL, double* __restrict__ psi,
                                                        double* __restrict__ acc, double* __restrict__ f) {
    constexpr int NV = WANT_F ? 5 : 4;
    __shared__ d4 tile_all[kDirWarps][32];
    __shared__ double red[kDirWarps][32][NV];
    __shared__ double bsum[32][NV];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    d4* tile = tile_all[w];
    const int rank = (int)(blockIdx.x % (unsigned)CL);
    const long long t0 = (long long)(blockIdx.x / (unsigned)CL) * S;
    const int slot = lane & (S - 1), rep = lane / S, R = 32 / S;
    const bool active = t0 + slot < nsinks;
    const long long bi = active ? (sinks ? sinks[t0 + slot] : t0 + slot) : 0;
    const double bx = x[3 * bi], by = x[3 * bi + 1], bz = x[3 * bi + 2];
    double v[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = 0.0;
    // the warp's slice of the sources
    const long long ns = (long long)CL * kDirWarps, sl = (long long)rank * kDirWarps + w;
    const int jb = (int)((long long)n * sl / ns), je = (int)((long long)n * (sl + 1) / ns);
    for (int j0 = jb; j0 < je; j0 += 32) {
        const int j = j0 + lane;
        __syncwarp();
        if (j < je) tile[lane] = mk4(x[3 * (long long)j], x[3 * (long long)j + 1], x[3 * (long long)j + 2], mu[j]);
        __syncwarp();
        const int nt = min(32, je - j0);
#pragma unroll 2
        for (int k = rep; k < nt; k += R) {
            const d4 q = tile[k];
            const double dx = q.x - bx, dy = q.y - by, dz = q.z - bz;
            const double r2 = dx * dx + dy * dy + dz * dz;
            if (positive_bits(r2)) {
                const double rinv = rsqrt(r2);
                // (mu / r, mu / r^2, mu / r^3 in this order: 1 / r^2 alone overflows for a subnormal r^2,
                // and a massless source would give NaN)
                const double qm = q.w * rinv;
                const double q2 = qm * rinv;
                const double q3 = q2 * rinv;
                v[0] += qm;
                v[1] = fma(q3, dx, v[1]);
                v[2] = fma(q3, dy, v[2]);
                v[3] = fma(q3, dz, v[3]);
                if (WANT_F) v[NV - 1] += q2;
            }
        }
    }
    // replicas, then warps, then the blocks of the cluster, each in order
#pragma unroll
    for (int q = 0; q < NV; ++q) {
        for (int o = S; o < 32; o <<= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
        if (rep == 0) red[w][slot][q] = v[q];
    }
    __syncthreads();
    const int c = threadIdx.x / 32, sk = lane;  // component c of sink sk (kDirWarps >= NV)
    if (c < NV && sk < S) {
        double s = 0.0;
        for (int k = 0; k < kDirWarps; ++k) s += red[k][sk][c];
        bsum[sk][c] = s;
    }
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    if (CL > 1) cl.sync();
    if (rank == 0 && c < NV && sk < S && t0 + sk < nsinks) {
        double s = bsum[sk][c];
        for (int r = 1; r < CL; ++r) s += *cl.map_shared_rank(&bsum[sk][c], r);
        const long long t = t0 + sk;
        if (c == 0) psi[t] = G * s;
        else if (c < 4) acc[3 * t + c - 1] = G * s;
        else f[t] = G * s;
    }
    if (CL > 1) cl.sync();  // the peers' sums stay until they are read
}

void launch_direct(const double* x, const double* mu, int n, double G, const int64_t* sinks, int nsinks,
                   double* psi, double* acc, double* f, cudaStream_t s) {
    if (nsinks <= 0) return;
    // at least eight blocks per SM, so that the last one costs little: first more slices of the
    // sources (CL), while a warp has more than 14 of them, then fewer sinks a block (their sources
    // are read from L2 once per block).  (Slices of fewer sources cost a cluster's barriers and give nothing:
    // n sinks of n sources, always 8 slices and so: 33 10.3 and 6.2 us, 200 43.8 and 14.4, 300 63.5 and
    // 34.8, from 400 the same)
    const long long want = 8LL * sm_count();
    auto groups = [&](int S) { return ((long long)nsinks + S - 1) / S; };
    int S = 32, CL = 1;
    while (CL < 8 && groups(S) * CL < want && n > 14 * kDirWarps * CL) CL *= 2;
    while (S > 1 && groups(S) * CL < want) S /= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(groups(S) * CL));
    cfg.blockDim = dim3(kDirThreads);
    cfg.stream = s;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = (unsigned)CL;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = CL > 1 ? 1 : 0;
    if (f) cudaLaunchKernelEx(&cfg, k_direct<true>, x, mu, n, G, sinks, nsinks, S, CL, psi, acc, f);
    else cudaLaunchKernelEx(&cfg, k_direct<false>, x, mu, n, G, sinks, nsinks, S, CL, psi, acc, f);
    note_launch();
}

}  // namespace gb3
