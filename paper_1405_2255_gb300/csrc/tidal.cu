// tidal.cu -- the tidal tensor T = grad grad Psi (Sec. 7.4) as an optional output of an
// evaluation: the far part from the local expansion's Psi_2^m at each particle (eq. 7
// taken to n = 2), the near part as the direct Hessian over the P2P lists (the same
// sources as the particle's P2P), combined, multiplied by G and scattered like Psi and a.
// Reading: T_xy = +Im Psi_2^2 / 2 (with the harmonics of App. A.3, Psi_2^2 = (d_x + i d_y)^2
// Psi); the other entries as printed in Sec. 7.4.  T is stored as (xx, xy, xz, yy, yz, zz).
#include "harmonics.cuh"
#include "kernels.cuh"

namespace gb3 {

// far part (FP64).  Psi_2^m = sum_{k,l} conj(Upsilon_k^l) F_{k+2}^{m+l}, m = 0, 1, 2, at s - x.  With
// X_k^{-l} = (-1)^l conj(X_k^l) the terms of l and -l combine: for a coefficient pair A = F_{k+2}^{m+l},
// B = (-1)^l F_{k+2}^{m-l},
//   conj(Y) A + Y B = Y.re (A + B) + Y.im (i (B - A)),  Y = Upsilon_k^l,
// and for m = 0 the imaginary part cancels: ten multiply-adds per (k, l) with the combinations formed
// once per leaf.  The recurrence (k^2 - l^2) Y_k = (2k - 1) z Y_{k-1} - r^2 Y_{k-2} is run on W_k = Y_k /
// sigma_k with sigma_k = (2k - 1) / (k^2 - l^2) sigma_{k-1}, sigma_l = 1, so that z W_{k-1} needs no
// factor; sigma is folded into the combinations.
// What bounds it: the FP64 pipe, whose instructions cost the same however many lanes are active.  A
// block takes the particles of kTidLeaves leaves together, so that its warps are full.  150,001
// particles, p = 14: 2.00 ms with a block per leaf, eq. 7 term by term and a division per (k, l);
// 0.62 ms so.
constexpr int kTidThreads = 128;
constexpr int kTidLeaves = 8;

struct TidTab {
    double beta[kMaxP + 1][kMaxP + 1];   // 1 / (k^2 - l^2) sigma_{k-2} / sigma_k at [l][k]
    double sigma[kMaxP + 1][kMaxP + 1];  // [l][k]
    double inv2l[kMaxP + 1];
};
static __constant__ TidTab c_tid;
static void init_tid_tab() {
    static DeviceOnce once;
    once_per_device(once, [] {
        TidTab t;
        memset(&t, 0, sizeof t);
        for (int l = 0; l <= kMaxP; ++l) {
            t.sigma[l][l] = 1.0;
            for (int k = l + 1; k <= kMaxP; ++k) {
                const double inv = 1.0 / (double)(k * k - l * l);
                t.sigma[l][k] = (2.0 * k - 1.0) * inv * t.sigma[l][k - 1];
                t.beta[l][k] = k >= l + 2 ? inv * t.sigma[l][k - 2] / t.sigma[l][k] : 0.0;
            }
            t.inv2l[l] = l ? 1.0 / (2.0 * l) : 0.0;
        }
        cudaMemcpyToSymbol(c_tid, &t, sizeof t);
    });
}

// combinations of one (k, l), sigma_k folded in: m = 0: Y.re and Y.im weights of Psi_2^0; m = 1, 2:
// the complex weights of Y.re and Y.im
struct TidComb {
    double r0, i0, ar[2], ai[2], br[2], bi[2];
};

__global__ void __launch_bounds__(kTidThreads) k_l2p_tidal(const d4* __restrict__ xm, Cells c,
                                                           const d4* __restrict__ cen,
                                                           const int* __restrict__ leaves, int nleaves, int p,
                                                           const double* __restrict__ F, double* __restrict__ T) {
    extern __shared__ __align__(16) unsigned char tsm[];
    TidComb* comb_all = (TidComb*)tsm;  // [kTidLeaves][npair]
    __shared__ int s_cell[kTidLeaves], s_end[kTidLeaves];
    const int nco = ncoef(p), q = p - 2, npair = (q + 1) * (q + 2) / 2;
    for (int t0 = blockIdx.x * kTidLeaves; t0 < nleaves; t0 += gridDim.x * kTidLeaves) {
        __syncthreads();
        if (threadIdx.x == 0) {
            int sum = 0;
            for (int u = 0; u < kTidLeaves; ++u) {
                const int cell = t0 + u < nleaves ? leaves[t0 + u] : -1;
                const bool on = cell >= 0 && cell_active(c, cell);
                sum += on ? c.count[cell] : 0;
                s_cell[u] = cell;
                s_end[u] = sum;  // particles of the leaves up to this one
            }
        }
        __syncthreads();
        for (int i = threadIdx.x; i < kTidLeaves * npair; i += blockDim.x) {
            const int u = i / npair, r = i % npair;
            if (s_end[u] == (u ? s_end[u - 1] : 0)) continue;
            // r counts (l, k) with l <= k <= q, columns l one after another
            int l = 0, b = 0;
            while (r >= b + q + 1 - l) b += q + 1 - l++;
            const int k = l + r - b;
            const double* Fr = F + (size_t)s_cell[u] * nco;
            const double sg = (l & 1) ? -1.0 : 1.0, sc = c_tid.sigma[l][k];
            TidComb cb;
#pragma unroll
            for (int m = 0; m <= 2; ++m) {
                const cd A = load_real_storage(Fr, k + 2, m + l);
                cd Bq = mkc(0.0, 0.0);
                if (l) Bq = load_real_storage(Fr, k + 2, m - l);
                const cd B = mkc(sg * Bq.re, sg * Bq.im);
                const cd a = mkc(sc * (A.re + B.re), sc * (A.im + B.im));  // of Y.re
                const cd d = mkc(sc * (A.im - B.im), sc * (B.re - A.re));  // of Y.im: i (B - A)
                if (m == 0) {
                    cb.r0 = a.re;
                    cb.i0 = d.re;
                } else {
                    cb.ar[m - 1] = a.re;
                    cb.ai[m - 1] = a.im;
                    cb.br[m - 1] = d.re;
                    cb.bi[m - 1] = d.im;
                }
            }
            comb_all[i] = cb;
        }
        __syncthreads();
        const int total = s_end[kTidLeaves - 1];
        for (int j = threadIdx.x; j < total; j += blockDim.x) {
            int u = 0;
            while (j >= s_end[u]) ++u;
            const int cell = s_cell[u], at = c.first[cell] + j - (u ? s_end[u - 1] : 0);
            const d4 s = cen[cell], xb = xm[at];
            const double x = s.x - xb.x, y = s.y - xb.y, z = s.z - xb.z;
            const double r2 = x * x + y * y + z * z;
            double p20 = 0.0, r21 = 0.0, i21 = 0.0, r22 = 0.0, i22 = 0.0;
            cd d = mkc(1.0, 0.0);
            const TidComb* cb = comb_all + u * npair;
            for (int l = 0; l <= q; ++l) {
                if (l > 0) {
                    const double sc = c_tid.inv2l[l], sx = sc * x, sy = sc * y;
                    d = cd{sx * d.re - sy * d.im, sx * d.im + sy * d.re};
                }
                cd prev2 = mkc(0.0, 0.0), Y = d;
                for (int k = l; k <= q; ++k, ++cb) {
                    if (k > l) {
                        const double b = r2 * c_tid.beta[l][k];
                        const cd nx = cd{z * Y.re - b * prev2.re, z * Y.im - b * prev2.im};
                        prev2 = Y;
                        Y = nx;
                    }
                    p20 = fma(Y.re, cb->r0, fma(Y.im, cb->i0, p20));
                    r21 = fma(Y.re, cb->ar[0], fma(Y.im, cb->br[0], r21));
                    i21 = fma(Y.re, cb->ai[0], fma(Y.im, cb->bi[0], i21));
                    r22 = fma(Y.re, cb->ar[1], fma(Y.im, cb->br[1], r22));
                    i22 = fma(Y.re, cb->ai[1], fma(Y.im, cb->bi[1], i22));
                }
            }
            double* o = T + 6 * (size_t)at;
            o[0] = -0.5 * p20 + 0.5 * r22;
            o[1] = 0.5 * i22;
            o[2] = r21;
            o[3] = -0.5 * p20 - 0.5 * r22;
            o[4] = i21;
            o[5] = p20;
        }
    }
}

void launch_l2p_tidal(const d4* xm, Cells c, const d4* cen, const int* leaves, int nleaves, int p, const double* F,
                      double* T, cudaStream_t s) {
    if (nleaves <= 0) return;  // (p < 2: no terms and T_far = 0)
    init_tid_tab();
    auto smem = [](int order) { return sizeof(TidComb) * (size_t)kTidLeaves * (order >= 2 ? (order - 1) * order / 2 : 0); };
    const size_t sm = smem(p);
    static DeviceOnce once;
    allow_smem(once, k_l2p_tidal, smem(kMaxP));
    const unsigned g = grid_for(((long long)nleaves + kTidLeaves - 1) / kTidLeaves * kTidThreads, kTidThreads, 16);
    k_l2p_tidal<<<g, kTidThreads, sm, s>>>(xm, c, cen, leaves, nleaves, p, F, T);
    note_launch();
}

// near part without a work plan (FP64 mode; mixed mode where the planned form of p2p.cu has no room
// for its scratch): one warp per sink leaf, lane = sink (chunks of 32), the sources of the leaf's
// own P2P segment and of its ancestors' segments through shared-memory tiles of 32.
// FP32 = true: dx from the two-float position records (hi + lo), FP32 pair terms, two-float sums
// folded per tile; false: FP64 throughout.
constexpr int kTidWarps = 4;
template <bool FP32>
__global__ void __launch_bounds__(kTidWarps * 32) k_p2p_tidal(const d4* __restrict__ xm, const float4* __restrict__ xp,
                                                              int n, Cells c,
                                                              const int2* __restrict__ list,
                                                              const int* __restrict__ seg_start,
                                                              const int* __restrict__ seg_end,
                                                              const int* __restrict__ leaves, int nleaves,
                                                              double* __restrict__ T) {
    __shared__ d4 tile64[kTidWarps][32];
    __shared__ float tile32[kTidWarps][7][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int t = blockIdx.x * kTidWarps + wid; t < nleaves; t += gridDim.x * kTidWarps) {
        const int leaf = leaves[t];
        if (!cell_active(c, leaf)) continue;
        const int first = c.first[leaf], count = c.count[leaf];
        for (int s0 = 0; s0 < count; s0 += 32) {
            const int i = first + s0 + lane;
            const bool act = s0 + lane < count;
            d4 xb = mk4(0, 0, 0, 0);
            float bh[3] = {0.f, 0.f, 0.f}, bl[3] = {0.f, 0.f, 0.f};
            if (act) {
                if (FP32) {
                    const float4 h = xp[2 * (size_t)i], l = xp[2 * (size_t)i + 1];
                    bh[0] = h.x;
                    bh[1] = h.y;
                    bh[2] = h.z;
                    bl[0] = l.x;
                    bl[1] = l.y;
                    bl[2] = l.z;
                } else {
                    xb = xm[i];
                }
            }
            double S64[6] = {0, 0, 0, 0, 0, 0};
            ff S32[6];
            for (int k = 0; k < 6; ++k) S32[k] = ff{0.f, 0.f};
            for (int cell = leaf; cell >= 0; cell = c.parent[cell]) {
                for (int e = seg_start[cell]; e < seg_end[cell]; ++e) {
                    const int A = list[e].x;
                    const int af = c.first[A], an = c.count[A];
                    for (int j0 = 0; j0 < an; j0 += 32) {
                        const int nt = min(32, an - j0);
                        __syncwarp();
                        if (lane < nt) {
                            const int j = af + j0 + lane;
                            if (FP32) {
                                const float4 h = xp[2 * (size_t)j], l = xp[2 * (size_t)j + 1];
                                tile32[wid][0][lane] = h.x;
                                tile32[wid][1][lane] = h.y;
                                tile32[wid][2][lane] = h.z;
                                tile32[wid][3][lane] = h.w;
                                tile32[wid][4][lane] = l.x;
                                tile32[wid][5][lane] = l.y;
                                tile32[wid][6][lane] = l.z;
                            } else {
                                tile64[wid][lane] = xm[j];
                            }
                        }
                        __syncwarp();
                        if (FP32) {
                            float P[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
                            for (int jj = 0; jj < nt; ++jj) {
                                const float dx = (bh[0] - tile32[wid][0][jj]) + (bl[0] - tile32[wid][4][jj]);
                                const float dy = (bh[1] - tile32[wid][1][jj]) + (bl[1] - tile32[wid][5][jj]);
                                const float dz = (bh[2] - tile32[wid][2][jj]) + (bl[2] - tile32[wid][6][jj]);
                                const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
                                if (r2 > 0.f) {
                                    const float ri = rsqrtf(r2), ri2 = ri * ri;
                                    const float q5 = tile32[wid][3][jj] * ri * ri2 * ri2;
                                    const float q3 = 3.f * q5;
                                    const float qr = q5 * r2;
                                    P[0] = fmaf(q3 * dx, dx, P[0] - qr);
                                    P[1] = fmaf(q3 * dx, dy, P[1]);
                                    P[2] = fmaf(q3 * dx, dz, P[2]);
                                    P[3] = fmaf(q3 * dy, dy, P[3] - qr);
                                    P[4] = fmaf(q3 * dy, dz, P[4]);
                                    P[5] = fmaf(q3 * dz, dz, P[5] - qr);
                                }
                            }
                            for (int k = 0; k < 6; ++k) ff_acc(S32[k], P[k]);
                        } else {
                            for (int jj = 0; jj < nt; ++jj) {
                                const d4 q = tile64[wid][jj];
                                const double dx = xb.x - q.x, dy = xb.y - q.y, dz = xb.z - q.z;
                                const double r2 = dx * dx + dy * dy + dz * dz;
                                if (r2 > 0.0) {
                                    const double ri = rsqrt(r2), ri2 = ri * ri;
                                    const double q5 = q.w * ri * ri2 * ri2;
                                    const double q3 = 3.0 * q5, qr = q5 * r2;
                                    S64[0] += q3 * dx * dx - qr;
                                    S64[1] += q3 * dx * dy;
                                    S64[2] += q3 * dx * dz;
                                    S64[3] += q3 * dy * dy - qr;
                                    S64[4] += q3 * dy * dz;
                                    S64[5] += q3 * dz * dz - qr;
                                }
                            }
                        }
                    }
                }
            }
            if (act) {
                double* o = T + 6 * (size_t)i;
                for (int k = 0; k < 6; ++k) o[k] = FP32 ? (double)S32[k].hi + (double)S32[k].lo : S64[k];
            }
        }
    }
}

void launch_p2p_tidal(const d4* xm, const float4* xp, int n, bool fp32, Cells c, const int2* list,
                      const int* seg_start, const int* seg_end, const int* leaves, int nleaves, double* T,
                      cudaStream_t s) {
    if (nleaves <= 0) return;
    long long g = ((long long)nleaves + kTidWarps - 1) / kTidWarps;
    if (g > (long long)sm_count() * 32) g = (long long)sm_count() * 32;
    if (fp32) k_p2p_tidal<true><<<(unsigned)g, kTidWarps * 32, 0, s>>>(xm, xp, n, c, list, seg_start, seg_end,
                                                                      leaves, nleaves, T);
    else k_p2p_tidal<false><<<(unsigned)g, kTidWarps * 32, 0, s>>>(xm, xp, n, c, list, seg_start, seg_end, leaves,
                                                                   nleaves, T);
    note_launch();
}

// T_caller = G (far + near), active particles only
__global__ void k_finish_tidal(const double* __restrict__ Tf, const double* __restrict__ Tn,
                               const int* __restrict__ perm, int n, double G, const unsigned char* __restrict__ pact,
                               double* __restrict__ T, const int* __restrict__ e) {
    const int kt = e ? e[1] - 3 * e[0] : 0;  // the tidal tensor ~ mu / x^3 in the working units
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        if (pact && !pact[i]) continue;
        const int o = perm[i];
        for (int k = 0; k < 6; ++k)
            T[6 * (size_t)o + k] = ldexp(G * (Tf[6 * (size_t)i + k] + Tn[6 * (size_t)i + k]), kt);
    }
}
void launch_finish_tidal(const double* Tf, const double* Tn, const int* perm, int n, double G,
                         const unsigned char* pact, double* T, cudaStream_t s, const int* e) {
    if (n > 0) k_finish_tidal<<<grid_for(n, 256), 256, 0, s>>>(Tf, Tn, perm, n, G, pact, T, e); note_launch();
}

}  // namespace gb3
