// upward.cu -- A5-A6 of the path (M2M eq. 4, multipole power eq. 14; P2M eq. 3c: p2m_split.cu)
// and the per-cell minimum of the acceleration scale used by eqs. (18a,b).
#include <cooperative_groups.h>

#include <vector>
#include <algorithm>

#include "harmonics.cuh"
#include "kernels.cuh"

namespace gb3 {

namespace cg = cooperative_groups;

// ---------------------------------------------------------------- M2M
// M_n^m(z') = sum_{k<=n} sum_l Upsilon_k^l(z - z') M_{n-k}^{m-l}(z): a cluster of eight blocks per parent, a
// block per daughter: a thread per output, the outputs with the most terms in the first warps, the terms of
// an output dealt out to four warps.  The daughters' contributions are added in daughter order.
// What bounds it: the FP64 pipe, of which a warp has a quarter of an SM's, and whose instructions cost the
// same however many lanes are active; at p = 14 a parent with eight daughters has some 70 us of it on one SM.
// A level with few parents is as long as one parent, hence the cluster.  13 levels of a cusp of 6e4 at p = 14:
// 8.1 ms with the daughters one after another in one warp, 1.9 ms with a warp per daughter, 0.61 ms so.
// (On levels that fill the device the empty blocks of missing daughters cost less than the even shares give:
// 2072 parents at p = 10 128 us with a block per parent, 88 us so.)
constexpr int kM2MWarps64 = 8;
constexpr int kM2MParts = 4;
__global__ void __launch_bounds__(kM2MWarps64 * 32) k_m2m(Cells c, const d4* __restrict__ cen, int lev_begin,
                                                          int p, double* __restrict__ M) {
    extern __shared__ cd csm[];
    constexpr int T = kM2MWarps64 * 32;
    const int t = threadIdx.x, wid = t >> 5, lane = t & 31;
    const int nco = ncoef(p), nout = out_count(p);
    cd* Yw = csm;
    cd* Mw = Yw + nco;
    cd* res = Mw + nco;  // [kM2MParts][nout]
    const cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)(blockIdx.x & 7), cell = lev_begin + (int)(blockIdx.x >> 3);
    const int nch = c.nchild[cell];
    if (nch == 0) return;  // (the whole cluster)
    if (rank < nch) {
        const int d = c.child[cell] + rank;
        const int t1 = (2 * (p + 1) + 31) & ~31;  // the warps after the columns' take the moments
        if (t < t1) {
            const d4 zp = cen[cell], z = cen[d];
            upsilon_columns2(p, t, z.x - zp.x, z.y - zp.y, z.z - zp.z, Yw, false);
        } else {
            expand_real(p, M + (size_t)d * nco, Mw, false, t - t1, T - t1);
        }
        __syncthreads();
        // (warp w takes part w % 4, so that the four parts of the SM's pipe have the same)
        for (int u = wid; u < kM2MParts * ((nout + 31) / 32); u += kM2MWarps64) {
            const int q = u % kM2MParts, o = nout - 1 - (u / kM2MParts * 32 + lane);
            if (o < 0) continue;
            const int n = out_order(o), m = o - n * (n + 1) / 2;
            cd4 s{0.0, 0.0, 0.0, 0.0};
            for (int k = q; k <= n; k += kM2MParts) {
                const int nn = n - k;
                const int lmin = max(-k, m - nn), lmax = min(k, m + nn);
                const cd *y = Yw + k * k + k, *x = Mw + nn * nn + nn + m;
#pragma unroll 4
                for (int l = lmin; l <= lmax; ++l) s.add(y[l], x[-l]);
            }
            res[q * nout + o] = s.sum();
        }
        __syncthreads();
        for (int o = t; o < nout; o += T)
            res[o] = ((res[o] + res[nout + o]) + res[2 * nout + o]) + res[3 * nout + o];
    }
    cl.sync();
    double* out = M + (size_t)cell * nco;
    for (int o = rank * T + t; o < nout; o += 8 * T) {
        const int n = out_order(o), m = o - n * (n + 1) / 2;
        cd v = mkc(0.0, 0.0);
        for (int j = 0; j < nch; ++j) v = v + *cl.map_shared_rank(res + o, j);
        out[cix(n, m)] = v.re;
        if (m) out[cix(n, -m)] = v.im;
    }
    cl.sync();  // the sums are read before their block ends
}

void launch_m2m_level(Cells c, const d4* cen, int lev_begin, int lev_end, int p, double* M, cudaStream_t s) {
    int ncl = lev_end - lev_begin;
    if (ncl <= 0) return;
    init_rec_tables();
    const size_t sm = (size_t)(2 * ncoef(p) + kM2MParts * out_count(p)) * sizeof(cd);
    launch_cluster8(k_m2m, 8 * ncl, kM2MWarps64 * 32, sm, s, c, cen, lev_begin, p, M);
    note_launch();
}

// ---------------------------------------------------------------- power
// weight of |M_n^m|^2 in P_n^2 (m and -m together) at n (n + 1) / 2 + m: (2 - delta_m0) (n-m)! (n+m)!
__device__ double g_power_w[(kMaxP + 1) * (kMaxP + 2) / 2];

// Two cells per warp: the terms of every (n, m) by all lanes, then lane n of each half adds up order n.
// (A thread per cell waited for 225 dependent steps: 70 us for the 1,027 cells of a 1e4 tree, 83 us for
// 49,616; a half warp per cell with a lane per order held the FP64 pipe with idle lanes, 134 us.)
constexpr int kPowWarps = 4;
__global__ void __launch_bounds__(kPowWarps * 32) k_power(const double* __restrict__ M, int ncells, int p,
                                                          double* __restrict__ P) {
    __shared__ double term_all[kPowWarps][2][(kMaxP + 1) * (kMaxP + 2) / 2];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nt = (p + 1) * (p + 2) / 2;
    const int cell0 = 2 * (blockIdx.x * kPowWarps + w);
    if (cell0 >= ncells) return;
    const int nc = min(2, ncells - cell0);
    for (int t = lane; t < nc * nt; t += 32) {
        const int k = t >= nt, o = k ? t - nt : t;
        int n = (int)((sqrtf(8.f * (float)o + 1.f) - 1.f) * 0.5f);
        while (n * (n + 1) / 2 > o) --n;
        while ((n + 1) * (n + 2) / 2 <= o) ++n;
        const int m = o - n * (n + 1) / 2;
        const double* R = M + (size_t)(cell0 + k) * ncoef(p);
        const double re = R[cix(n, m)], im = m ? R[cix(n, -m)] : 0.0;
        term_all[w][k][o] = __ldg(&g_power_w[o]) * (re * re + im * im);
    }
    __syncwarp();
    for (int t = lane; t < 2 * 16 * ((p + 16) / 16); t += 32) {
        const int k = (t >> 4) & 1, n = (t & 15) + 16 * (t >> 5);
        if (k >= nc || n > p) continue;
        const double* q = term_all[w][k] + n * (n + 1) / 2;
        double s = q[0];
        for (int m = 1; m <= n; ++m) s += q[m];
        P[(size_t)(cell0 + k) * (p + 1) + n] = sqrt(s);
    }
}

void launch_power(const double* M, int ncells, int p, double* P, cudaStream_t s) {
    static DeviceOnce once;
    once_per_device(once, [] {
        double f[2 * kMaxP + 1], wt[(kMaxP + 1) * (kMaxP + 2) / 2];
        f[0] = 1;
        for (int i = 1; i <= 2 * kMaxP; ++i) f[i] = f[i - 1] * i;
        for (int n = 0; n <= kMaxP; ++n)
            for (int m = 0; m <= n; ++m) wt[n * (n + 1) / 2 + m] = (m ? 2.0 : 1.0) * f[n - m] * f[n + m];
        cudaMemcpyToSymbol(g_power_w, wt, sizeof wt);
    });
    if (ncells > 0) {
        const int per = 2 * kPowWarps;
        k_power<<<(ncells + per - 1) / per, kPowWarps * 32, 0, s>>>(M, ncells, p, P);
        note_launch();
    }
}

// ---------------------------------------------------------------- min scale
__global__ void k_minscale_leaves(const double* __restrict__ sc, Cells c, const int* __restrict__ leaves,
                                  int nleaves) {
    const int lane = threadIdx.x & 31, nw = (gridDim.x * blockDim.x) >> 5;
    for (int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < nleaves; t += nw) {
        const int cell = leaves[t];
        double m = INFINITY;
        for (int i = c.first[cell] + lane, e = c.first[cell] + c.count[cell]; i < e; i += 32)
            if (!c.pact || c.pact[i]) m = fmin(m, sc[i]);  // over the active sinks only (Sec. 7.1)
        m = warp_min(m);
        if (lane == 0) c.minscale[cell] = m;
    }
}
// the internal cells, bottom-up: one cluster whose blocks meet at its barrier between the levels (a launch
// per level took 4 us each, 11 of them for a Plummer sphere of 1e6)
struct Levels {
    int n, start[kMaxLevel + 2];
};
constexpr int kMinThreads = 1024;
__global__ void __launch_bounds__(kMinThreads) k_minscale_levels(const __grid_constant__ Cells c,
                                                                 const __grid_constant__ Levels lv) {
        cg::cluster_group cl = cg::this_cluster();
    for (int L = lv.n - 1; L >= 0; --L) {
        for (int cell = lv.start[L] + blockIdx.x * blockDim.x + threadIdx.x; cell < lv.start[L + 1];
             cell += gridDim.x * blockDim.x) {
            const int nch = c.nchild[cell], ch = c.child[cell];
            if (!nch) continue;
            double m = INFINITY;
            for (int j = 0; j < nch; ++j) m = fmin(m, __ldcg(c.minscale + ch + j));  // (other blocks wrote them)
            c.minscale[cell] = m;
        }
        cl.sync();
    }
}
void launch_minscale(const double* scale_sorted, Cells c, const int* leaves, int nleaves, const int* lev_start, int nlev,
                     cudaStream_t s) {
    if (nleaves <= 0) return;
    k_minscale_leaves<<<grid_for((long long)nleaves * 32, 256, 16), 256, 0, s>>>(scale_sorted, c, leaves, nleaves);
    note_launch();
    Levels lv;
    lv.n = nlev - 1;  // the deepest level holds leaves only
    for (int L = 0; L < nlev; ++L) lv.start[L] = lev_start[L];
    if (lv.n <= 0) return;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 8;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.gridDim = dim3(8);
    cfg.blockDim = dim3(kMinThreads);
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, k_minscale_levels, c, lv);
    note_launch();
}
// the caller's scale (an acceleration, ~ mu / x^2) in the working units (e nullable)
__global__ void k_scale_from_caller(const double* __restrict__ scale, const int* __restrict__ perm, int n,
                                    double* __restrict__ out, const int* __restrict__ e) {
    const int ks = e ? 2 * e[0] - e[1] : 0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        out[i] = ldexp(scale[perm[i]], ks);
}
void launch_scale_from_caller(const double* scale, const int* perm, int n, double* scale_sorted, cudaStream_t s,
                              const int* e) {
    if (n > 0) k_scale_from_caller<<<grid_for(n, 256), 256, 0, s>>>(scale, perm, n, scale_sorted, e); note_launch();
}

}  // namespace gb3

namespace gb3 {
// ---------------------------------------------------------------- active subsets (Sec. 7.1)
__global__ void k_active_sorted(const unsigned char* __restrict__ active, const int* __restrict__ perm, int n,
                                unsigned char* __restrict__ pact, int* __restrict__ ai) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const unsigned char a = active[perm[i]] != 0;
        pact[i] = a;
        ai[i] = a;
    }
}
__global__ void k_active_cells(const int* __restrict__ first, const int* __restrict__ count, int ncells,
                               const int* __restrict__ scan, const int* __restrict__ total, int n,
                               unsigned char* __restrict__ act) {
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncells; c += gridDim.x * blockDim.x) {
        const int f = first[c], e = f + count[c];
        const int hi = e < n ? scan[e] : *total;
        act[c] = hi - scan[f] > 0;
    }
}
void launch_active_flags(const unsigned char* active, const int* perm, int n, const int* first, const int* count,
                         int ncells, unsigned char* pact, unsigned char* act, int* ai, int* scan, int* scan_tmp,
                         cudaStream_t s) {
    if (n <= 0) return;
    k_active_sorted<<<grid_for(n, 256), 256, 0, s>>>(active, perm, n, pact, ai);
    note_launch();
    int* total = ai + n;  // ai holds n + 1 ints
    scan_exclusive_i32(ai, scan, n, total, scan_tmp, s);
    k_active_cells<<<grid_for(ncells, 256), 256, 0, s>>>(first, count, ncells, scan, total, n, act);
    note_launch();
}
}  // namespace gb3

namespace gb3 {
// ---------------------------------------------------------------- individual accuracy (Sec. 7, opening)
// scale_sorted[i] *= eps_b[perm[i]] / eps, so that eps * min_B(scale) = min_B(eps_b a_b);
// a non-positive or non-finite eps_b sets kStatInvalid
__global__ void k_scale_eps(const double* __restrict__ eps_b, const int* __restrict__ perm, int n, double eps,
                            double* __restrict__ scale_sorted, unsigned* __restrict__ status) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        const double e = eps_b[perm[i]];
        if (!(e > 0) || !isfinite(e)) atomicOr(status, kStatInvalid);
        scale_sorted[i] *= e / eps;
    }
}
void launch_scale_eps(const double* eps_b, const int* perm, int n, double eps, double* scale_sorted, unsigned* status,
                      cudaStream_t s) {
    if (n > 0) k_scale_eps<<<grid_for(n, 256), 256, 0, s>>>(eps_b, perm, n, eps, scale_sorted, status); note_launch();
}
}  // namespace gb3
