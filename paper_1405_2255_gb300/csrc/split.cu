// split.cu -- mixed-mode M2M (eq. 4), L2L (eq. 5) and L2P (eqs. 3a, 7; P2M: p2m_split.cu) with the same order
// split as the M2L: the expansion orders n <= 2 are formed in FP64, the higher
// orders in FP32 on quantities scaled by the cell radius (Upsilon evaluated at
// (x - z)/rho, whose values are bounded by 1/n!), then rescaled in FP64.  The
// higher orders carry a fraction ~ theta^n of an expansion's contribution, so
// FP32 rounding there stays far below the targeted force error.
#include <cooperative_groups.h>

#include "harmonics.cuh"
#include "kernels.cuh"

namespace gb3 {

static __constant__ float c_inv_upf[kMaxP + 1][kMaxP + 1];  // 1 / (n^2 - m^2)
static __constant__ float c_twf2[kMaxP + 2];                // 2n - 1
static __constant__ float c_inv2jf[kMaxP + 1];              // 1 / (2j)

static void init_split_up_tables() {
    static DeviceOnce once;
    once_per_device(once, [] {
        float a[kMaxP + 1][kMaxP + 1], b[kMaxP + 2], c[kMaxP + 1];
        for (int n = 0; n <= kMaxP; ++n)
            for (int m = 0; m <= kMaxP; ++m) a[n][m] = (n * n != m * m) ? 1.0f / (float)(n * n - m * m) : 0.f;
        for (int n = 0; n <= kMaxP + 1; ++n) b[n] = (float)(2 * n - 1);
        c[0] = 0.f;
        for (int j = 1; j <= kMaxP; ++j) c[j] = 1.0f / (2.0f * j);
        cudaMemcpyToSymbol(c_inv_upf, a, sizeof a);
        cudaMemcpyToSymbol(c_twf2, b, sizeof b);
        cudaMemcpyToSymbol(c_inv2jf, c, sizeof c);
    });
}

// What bounds these kernels: the FP64 pipe (2 lanes a cycle and SM, an instruction costs the same
// however many lanes are active, and so does a conversion between FP64 and FP32).  So the powers of the
// radii are formed once per cell, every real coefficient is converted once (the entries of order -m are
// sign changes of those of order m), and the low orders are taken as real linear forms.

// pw[cell][k] = rho^k, pw[cell][p + 1 + k] = rho^-k (0 for k > 0 of a cell of radius 0), by repeated
// products; one thread per cell
__global__ void k_pow_tables(const d4* __restrict__ cen, int ncells, int p, double* __restrict__ pw) {
    const int cell = blockIdx.x * blockDim.x + threadIdx.x;
    if (cell >= ncells) return;
    const double rho = cen[cell].w, inv = rho > 0 ? 1.0 / rho : 0.0;
    double* t = pw + (size_t)cell * 2 * (p + 1);
    double v = 1.0, u = 1.0;
    for (int k = 0; k <= p; ++k) {
        t[k] = v;
        t[p + 1 + k] = u;
        v *= rho;
        u *= inv;
    }
}
void launch_pow_tables(const d4* cen, int ncells, int p, double* pw, cudaStream_t s) {
    if (ncells > 0) {
        k_pow_tables<<<(ncells + 127) / 128, 128, 0, s>>>(cen, ncells, p, pw);
        note_launch();
    }
}

__device__ inline int n_of(int i) {
    int n = (int)sqrtf((float)i);
    while (n * n > i) --n;
    while ((n + 1) * (n + 1) <= i) ++n;
    return n;
}
// out (full complex, FP32) = R (real storage) times sc[n] for the (p+1)^2 coefficients, by nt threads (t)
__device__ __forceinline__ void expand_scaled(const double* __restrict__ R, const double* __restrict__ sc, int nco,
                                              int t, int nt, float2* out) {
    for (int i = t; i < nco; i += nt) {
        const int n = n_of(i), c0 = n * n + n, m = i - c0, am = m < 0 ? -m : m;
        const float v = (float)(R[i] * sc[n]);
        const float w = (am & 1) ? -v : v;
        if (m >= 0) {
            out[c0 + am].x = v;
            out[c0 - am].x = w;
            if (m == 0) out[c0].y = 0.f;
        } else {
            out[c0 + am].y = v;
            out[c0 - am].y = -w;
        }
    }
}

constexpr int kSplitWarps = 4;

// ---------------------------------------------------------------- L2P
// Psi_0^0 = sum_{k,l} Upsilon_k^{l*} F_k^l and Psi_1^m = sum_{k,l} Upsilon_k^{l*} F_{k+1}^{m+l}
// (Upsilon at s_B - x_b): terms with k <= 2 in FP64; terms with k >= 3 in FP32 as
// Uhat_k^{l*} Fhat_k^l and Uhat_k^{l*} Fhat_{k+1}^{m+l} / rho with Uhat_k = Upsilon_k((s - x)/rho),
// Fhat_n = F_n rho^n.  One warp per leaf, lane = particle.
// The terms k <= 2 are linear in the nine real entries u of Upsilon (upsilon_low): with l and -l taken
// together (F^{-l} = (-1)^l conj(F^l)), psi and az take 2 Re and 2 Im of F_k^l and F_{k+1}^l, and ax, ay
// the parts of A + B (of Re Y) and i (B - A) (of Im Y), A = F_{k+1}^{1+l}, B = (-1)^l F_{k+1}^{1-l}:
// 36 multiply-adds per particle (some 90 when every complex term was taken by itself).
__global__ void __launch_bounds__(kSplitWarps * 32) k_l2p_split(const d4* __restrict__ xm, Cells c,
                                                                const d4* __restrict__ cen,
                                                                const double* __restrict__ pw,
                                                                const int* __restrict__ leaves, int nleaves, int p,
                                                                const double* __restrict__ F, double* __restrict__ psi,
                                                                double* __restrict__ acc) {
    extern __shared__ __align__(16) unsigned char sraw[];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nco = ncoef(p);
    const size_t per_warp = ((size_t)nco * sizeof(float2) + 36 * sizeof(double) + 15) & ~(size_t)15;
    double* C = (double*)(sraw + wid * per_warp);  // [9][4]: weights of u in psi, p10, Re p11, Im p11
    float2* Fh = (float2*)(C + 36);                // [nco] F_n rho^n
    const int t = blockIdx.x * kSplitWarps + wid;
    if (t >= nleaves) return;
    const int cell = leaves[t];
    if (!cell_active(c, cell)) return;
    const d4 s = cen[cell];
    const double rho = s.w;
    const double* Fr = F + (size_t)cell * nco;
    const double* pc = pw + (size_t)cell * 2 * (p + 1);
    expand_scaled(Fr, pc, nco, lane, 32, Fh);
    if (lane < 9) {
        const int k = lane < 1 ? 0 : (lane < 4 ? 1 : 2), m = lane - k * k - k, l = m < 0 ? -m : m;
        const cd f0 = load_real_storage(Fr, k, l), f1 = load_real_storage(Fr, k + 1, l);
        const cd A = load_real_storage(Fr, k + 1, 1 + l);
        cd B = mkc(0.0, 0.0);
        if (l) B = load_real_storage(Fr, k + 1, 1 - l);
        if (l & 1) B = mkc(-B.re, -B.im);
        double* w = C + 4 * lane;
        if (m >= 0) {
            w[0] = l ? f0.re + f0.re : f0.re;
            w[1] = l ? f1.re + f1.re : f1.re;
            w[2] = A.re + B.re;
            w[3] = A.im + B.im;
        } else {
            w[0] = f0.im + f0.im;
            w[1] = f1.im + f1.im;
            w[2] = A.im - B.im;
            w[3] = B.re - A.re;
        }
    }
    __syncwarp();
    const double rinv = pc[p + 2];
    const int first = c.first[cell], count = c.count[cell];
    for (int j = lane; j < count; j += 32) {
        const d4 xb = xm[first + j];
        const double vx = s.x - xb.x, vy = s.y - xb.y, vz = s.z - xb.z;
        // k <= 2 in FP64
        double u[9], q[4] = {0.0, 0.0, 0.0, 0.0};
        upsilon_low(vx, vy, vz, u);
        // the weights are read from shared memory here: kept in registers across the loop (127 of them)
        // they cost more warps than the reads (0.68 ms for the 43,413 leaves of a Plummer sphere of 1e6)
        const double* Cj = C;
        asm volatile("" : "+l"(Cj));
#pragma unroll
        for (int i = 0; i < 9; ++i)
#pragma unroll
            for (int d = 0; d < 4; ++d) q[d] = fma(u[i], Cj[4 * i + d], q[d]);
        // k >= 3 in FP32 on the scaled offset
        float h00 = 0.f;
        float2 h10 = make_float2(0.f, 0.f), h11 = make_float2(0.f, 0.f);
        if (rho > 0 && p >= 3) {
            const float x = (float)(vx * rinv), y = (float)(vy * rinv), z = (float)(vz * rinv);
            const float r2 = x * x + y * y + z * z;
            float2 d = make_float2(1.f, 0.f);
            for (int l = 0; l <= p; ++l) {
                if (l > 0) {
                    const float sc = c_inv2jf[l];
                    d = make_float2(sc * (x * d.x - y * d.y), sc * (x * d.y + y * d.x));
                }
                const float sg = (l & 1) ? -1.f : 1.f;
                float2 prev2 = make_float2(0.f, 0.f), prev = d;
                for (int k = l; k <= p; ++k) {
                    float2 Y;
                    if (k == l) Y = d;
                    else {
                        const float a = c_twf2[k] * z, iv = c_inv_upf[k][l];
                        Y = make_float2((a * prev.x - r2 * prev2.x) * iv, (a * prev.y - r2 * prev2.y) * iv);
                        prev2 = prev;
                        prev = Y;
                    }
                    if (k < 3) continue;
                    const float2 Xp = make_float2(Y.x, -Y.y);
                    const float2 Xn = make_float2(sg * Y.x, sg * Y.y);
                    const float2* Fk = Fh + k * k + k;
                    if (l == 0) h00 += Xp.x * Fk[0].x - Xp.y * Fk[0].y;
                    else h00 += 2.f * (Xp.x * Fk[l].x - Xp.y * Fk[l].y);
                    if (k < p) {
                        const float2* Fk1 = Fh + (k + 1) * (k + 1) + (k + 1);
                        cmacf(h10, Xp, Fk1[l]);
                        cmacf(h11, Xp, Fk1[1 + l]);
                        if (l > 0) {
                            cmacf(h10, Xn, Fk1[-l]);
                            cmacf(h11, Xn, Fk1[1 - l]);
                        }
                    }
                }
            }
        }
        const int i = first + j;
        psi[i] = q[0] + (double)h00;
        acc[3 * (size_t)i] = -(q[2] + (double)h11.x * rinv);
        acc[3 * (size_t)i + 1] = -(q[3] + (double)h11.y * rinv);
        acc[3 * (size_t)i + 2] = -(q[1] + (double)h10.x * rinv);
    }
}

void launch_l2p_split(const d4* xm, Cells c, const d4* cen, const double* pw, const int* leaves, int nleaves, int p,
                      const double* F, double* psi, double* acc, cudaStream_t s) {
    if (nleaves <= 0) return;
    if (p < 3) {
        launch_l2p(xm, c, cen, leaves, nleaves, p, F, psi, acc, s);
        return;
    }
    init_split_up_tables();
    const size_t per_warp = ((size_t)ncoef(p) * sizeof(float2) + 36 * sizeof(double) + 15) & ~(size_t)15;
    k_l2p_split<<<(nleaves + kSplitWarps - 1) / kSplitWarps, kSplitWarps * 32, kSplitWarps * per_warp, s>>>(
        xm, c, cen, pw, leaves, nleaves, p, F, psi, acc);
    note_launch();
}

// full complex Upsilon_k^l(v), k <= 2, from the closed forms (conj_out: conjugates)
__device__ inline void upsilon_low_full(double x, double y, double z, cd out[9], bool conj_out) {
    double u[9];
    upsilon_low(x, y, z, u);
    for (int k = 0; k <= 2; ++k)
        for (int l = 0; l <= k; ++l) {
            cd v = mkc(u[cix(k, l)], l ? u[cix(k, -l)] : 0.0);
            if (conj_out) v = conjc(v);
            out[cix(k, l)] = v;
            if (l) {
                // X^{-l} = (-1)^l conj(X^l) for both Upsilon and its conjugate
                out[cix(k, -l)] = (l & 1) ? mkc(-v.re, v.im) : mkc(v.re, -v.im);
            }
        }
}

// FP32 column m of Upsilon at a scaled offset (|v| <= 1), optionally conjugated
__device__ inline void upsilon_column_f(int p, int m, float x, float y, float z, float2* out, bool conj_out) {
    const float r2 = x * x + y * y + z * z;
    float2 d = make_float2(1.f, 0.f);
    for (int j = 1; j <= m; ++j) {
        const float s = c_inv2jf[j];
        d = make_float2(s * (x * d.x - y * d.y), s * (x * d.y + y * d.x));
    }
    float2 prev2 = make_float2(0.f, 0.f), prev = d;
    const float sg = (m & 1) ? -1.f : 1.f;
    for (int n = m; n <= p; ++n) {
        float2 v;
        if (n == m) v = d;
        else {
            const float a = c_twf2[n] * z, iv = __frcp_rn((float)(n * n - m * m));
            v = make_float2((a * prev.x - r2 * prev2.x) * iv, (a * prev.y - r2 * prev2.y) * iv);
            prev2 = prev;
            prev = v;
        }
        if (conj_out) v.y = -v.y;
        out[cix(n, m)] = v;
        if (m) out[cix(n, -m)] = make_float2(sg * v.x, -sg * v.y);
    }
}

// ---------------------------------------------------------------- M2M
// M_n^m(z') = sum_{k<=n} sum_l Upsilon_k^l(z - z') M_{n-k}^{m-l}(z): outputs n <= 2 in FP64,
// outputs n >= 3 in FP32 as Mhat_n = M_n / rho'^n = sum Uhat_k Mt_{n-k} with
// Uhat_k = Upsilon_k((z - z')/rho'), Mt_j = M_j(z) / rho'^j.  One block per parent, or a cluster of eight
// with a block per daughter (kCluster).  The threads first prepare the daughters' arrays, then the warps take
// (32 outputs, daughter) pairs, the outputs with the most terms first; the daughters' contributions are
// summed in daughter order.
// What bounds it: the chain of a level with few parents, which leaves the device idle (hence the clusters),
// and on the large levels the instructions of the sums.  p = 14: 32 us a level of a sphere of 1e4 and
// 0.68 ms for all levels of one of 1e6 with all outputs of a daughter in one warp, 13 us and
// 0.53 ms so.
constexpr int kM2MWarps = 8;
__host__ __device__ inline size_t m2m_child_bytes(int p) {
    return ((size_t)2 * ncoef(p) * sizeof(float2) + 18 * sizeof(cd) + 15) & ~(size_t)15;
}
__host__ __device__ inline size_t m2m_smem_bytes(int p) {  // per daughter of a block
    return m2m_child_bytes(p) + out_count(p) * sizeof(float2) + 6 * sizeof(cd);
}
template <bool kCluster>
__global__ void __launch_bounds__(kM2MWarps * 32) k_m2m_split(Cells c, const d4* __restrict__ cen,
                                                               const double* __restrict__ pw, int lev_begin,
                                                               int p, double* __restrict__ M) {
    extern __shared__ __align__(16) unsigned char sraw[];
    constexpr int S = kCluster ? 1 : 8;  // daughters of a block
    const int t = threadIdx.x, wid = t >> 5, lane = t & 31;
    const int nco = ncoef(p), nout = out_count(p);
    const size_t per_child = m2m_child_bytes(p);
    cd* r64 = (cd*)(sraw + S * per_child);  // [S][6]
    float2* r32 = (float2*)(r64 + S * 6);    // [S][nout]
    const int rank = kCluster ? (int)(blockIdx.x & 7) : 0;
    const int cell = lev_begin + (kCluster ? blockIdx.x >> 3 : blockIdx.x);
    const int nch = c.nchild[cell];
    if (nch == 0) return;  // leaves (the whole cluster)
    const int mine = kCluster ? (rank < nch ? 1 : 0) : nch, first = c.child[cell] + rank;
    const d4 zp = cen[cell];
    const double *pwr = pw + (size_t)cell * 2 * (p + 1), *pwi = pwr + p + 1;  // rho^n, rho^-n
    const double rho = zp.w;
    const int t1 = (S * (p + 1) + 31) & ~31;  // the warps after the columns' take the moments
    if (t < t1) {
        const int d = t % S, m = t / S;
        if (d < mine && m <= p) {
            const double inv = pwi[1];
            const d4 z = cen[first + d];
            const double vx = z.x - zp.x, vy = z.y - zp.y, vz = z.z - zp.z;
            float2* Yh = (float2*)((cd*)(sraw + d * per_child) + 18);
            upsilon_column_f(p, m, (float)(vx * inv), (float)(vy * inv), (float)(vz * inv), Yh, false);
        }
    } else {
        for (int d = 0; d < mine; ++d)
            expand_scaled(M + (size_t)(first + d) * nco, pwi, nco, t - t1, kM2MWarps * 32 - t1,
                          (float2*)((cd*)(sraw + d * per_child) + 18) + nco);
        if (wid == kM2MWarps - 1) {
            for (int i = lane; i < 9 * mine; i += 32) {
                const int d = i / 9, e = i - 9 * d, n = n_of(e);
                ((cd*)(sraw + d * per_child))[9 + e] = load_real_storage(M + (size_t)(first + d) * nco, n, e - n * n - n);
            }
            if (lane < mine) {
                const d4 z = cen[first + lane];
                upsilon_low_full(z.x - zp.x, z.y - zp.y, z.z - zp.z, (cd*)(sraw + lane * per_child), false);
            }
        }
    }
    __syncthreads();
    const int units = mine * ((nout + 31) / 32);
    for (int u = wid; u < units; u += kM2MWarps) {
        const int w = u / mine, d = u - w * mine, o = nout - 1 - (w * 32 + lane);
        if (o < 0) continue;
        const cd* Y64 = (const cd*)(sraw + d * per_child);
        const cd* M64 = Y64 + 9;
        const float2* Yh = (const float2*)(M64 + 9);
        const float2* Mt = Yh + nco;
        const int n = out_order(o), m = o - n * (n + 1) / 2;
        if (n <= 2) {
            cd sum = mkc(0.0, 0.0);
            for (int k = 0; k <= n; ++k) {
                const int nn = n - k;
                for (int l = max(-k, m - nn); l <= min(k, m + nn); ++l)
                    cmac(sum, Y64[cix(k, l)], M64[cix(nn, m - l)]);
            }
            r64[d * 6 + o] = sum;
        } else {
            float2 sum = make_float2(0.f, 0.f);
            if (rho > 0)
                for (int k = 0; k <= n; ++k) {
                    const int nn = n - k, lmin = max(-k, m - nn), lmax = min(k, m + nn);
                    const float2 *y = Yh + k * k + k, *x = Mt + nn * nn + nn + m;
#pragma unroll 4
                    for (int l = lmin; l <= lmax; ++l) cmacf(sum, y[l], x[-l]);
                }
            r32[d * nout + o] = sum;
        }
    }
    if (kCluster) cooperative_groups::this_cluster().sync();
    else __syncthreads();
    // the parent's moments: the daughters' terms summed in daughter order
    double* out = M + (size_t)cell * nco;
    for (int o = rank * (kM2MWarps * 32) + t; o < nout; o += S == 1 ? 8 * kM2MWarps * 32 : kM2MWarps * 32) {
        const int n = out_order(o), m = o - n * (n + 1) / 2;
        cd v;
        if (n <= 2) {
            v = mkc(0.0, 0.0);
            for (int j = 0; j < nch; ++j)
                v = v + (kCluster ? *cooperative_groups::this_cluster().map_shared_rank(r64 + o, j) : r64[j * 6 + o]);
        } else {
            float2 a = make_float2(0.f, 0.f);
            for (int j = 0; j < nch; ++j) {
                const float2 b = kCluster ? *cooperative_groups::this_cluster().map_shared_rank(r32 + o, j)
                                          : r32[j * nout + o];
                a.x += b.x;
                a.y += b.y;
            }
            const double sc = pwr[n];
            v = mkc((double)a.x * sc, (double)a.y * sc);
        }
        out[cix(n, m)] = v.re;
        if (m) out[cix(n, -m)] = v.im;
    }
    if (kCluster) cooperative_groups::this_cluster().sync();  // the sums are read before their block ends
}

void launch_m2m_split(Cells c, const d4* cen, const double* pw, int lev_begin, int lev_end, int p, double* M, cudaStream_t s) {
    const int ncl = lev_end - lev_begin;
    if (ncl <= 0) return;
    if (p < 3) {
        launch_m2m_level(c, cen, lev_begin, lev_end, p, M, s);
        return;
    }
    init_split_up_tables();
    const size_t per = m2m_smem_bytes(p);
    // (leaves of the level return at once)
    // a cluster per parent for up to six parents per SM: 944 parents at p = 14 take 43 us as blocks and 39 as
    // clusters, 2016 parents 49 and 73
    if (ncl <= 6 * sm_count()) {
        launch_cluster8(k_m2m_split<true>, 8 * ncl, kM2MWarps * 32, per, s, c, cen, pw, lev_begin, p, M);
    } else {
        static DeviceOnce once;
        allow_smem(once, k_m2m_split<false>, 8 * m2m_smem_bytes(kMaxP));
        k_m2m_split<false><<<(unsigned)ncl, kM2MWarps * 32, 8 * per, s>>>(c, cen, pw, lev_begin, p, M);
    }
    note_launch();
}

// ---------------------------------------------------------------- L2L
// F_n^m(s') += sum_{k<=p-n} sum_l Upsilon_k^{l*}(s - s') F_{n+k}^{m+l}(s): terms with n+k <= 2
// in FP64, the others in FP32 as rho^-n sum Uhat_k^{l*} Fhat_{n+k}^{m+l} with
// Uhat_k = Upsilon_k((s - s')/rho), Fhat_j = F_j(s) rho^j (rho: the parent's radius).
// W warps per cell, a thread per output, the outputs with the most terms first.  The FP64 terms of the six
// outputs n <= 2 are 20 products, one per lane of the last warp.
// What bounds it: as for the M2M.  p = 14: 31 us a level of a sphere of 1e4 and 0.61 ms for all levels of
// one of 1e6 with all outputs of a cell in one warp, 12.5 us and 0.585 ms so.
struct L2LTerm {
    signed char n, m, k, l;
};
__device__ constexpr L2LTerm kL2LTerm[20] = {
    {0, 0, 0, 0},  {0, 0, 1, -1}, {0, 0, 1, 0}, {0, 0, 1, 1},  {0, 0, 2, -2}, {0, 0, 2, -1}, {0, 0, 2, 0},
    {0, 0, 2, 1},  {0, 0, 2, 2},  {1, 0, 0, 0}, {1, 0, 1, -1}, {1, 0, 1, 0},  {1, 0, 1, 1},  {1, 1, 0, 0},
    {1, 1, 1, -1}, {1, 1, 1, 0},  {1, 1, 1, 1}, {2, 0, 0, 0},  {2, 1, 0, 0},  {2, 2, 0, 0}};
__device__ constexpr int kL2LStart[7] = {0, 9, 13, 17, 18, 19, 20};  // first product of output n (n + 1) / 2 + m
__host__ __device__ inline size_t l2l_cell_bytes(int p) {
    return ((size_t)2 * ncoef(p) * sizeof(float2) + (9 + 9 + 20 + 6) * sizeof(cd) + 15) & ~(size_t)15;
}
template <int W>
__global__ void __launch_bounds__(W == 1 ? 128 : W * 32) k_l2l_split(Cells c, const d4* __restrict__ cen,
                                                                     const double* __restrict__ pw, int lev_begin,
                                                                     int lev_end, int p, double* __restrict__ F) {
    extern __shared__ __align__(16) unsigned char sraw[];
    constexpr int kCells = W == 1 ? 4 : 1, T = W * 32;  // cells of a block, threads of a cell
    const int g = threadIdx.x / T, t = threadIdx.x % T, lane = threadIdx.x & 31;
    const int nco = ncoef(p), nout = out_count(p);
    cd* Y64 = (cd*)(sraw + g * l2l_cell_bytes(p));
    cd* F64 = Y64 + 9;
    cd* prod = F64 + 9;
    cd* low = prod + 20;
    float2* Yh = (float2*)(low + 6);
    float2* Fh = Yh + nco;
    const int cell = lev_begin + blockIdx.x * kCells + g;
    if (cell >= lev_end || !cell_active(c, cell)) return;  // (the same for all threads of a cell)
    const int par = c.parent[cell];
    const d4 s = cen[par], sp = cen[cell];
    const double rho = s.w;
    double* out = F + (size_t)cell * nco;
    const double* Fp = F + (size_t)par * nco;
    if (!(rho > 0)) {  // all particles at the parent's centre: the shift is the identity
        for (int i = t; i < nco; i += T) out[i] += Fp[i];
        return;
    }
    const double *pwr = pw + (size_t)par * 2 * (p + 1), *pwi = pwr + p + 1;  // rho^n, rho^-n
    const double inv = pwi[1];
    const double vx = s.x - sp.x, vy = s.y - sp.y, vz = s.z - sp.z;
    if (t <= p) upsilon_column_f(p, t, (float)(vx * inv), (float)(vy * inv), (float)(vz * inv), Yh, true);
    if (W == 1 || t >= 32) expand_scaled(Fp, pwr, nco, W == 1 ? t : t - 32, W == 1 ? 32 : T - 32, Fh);
    if (t >= T - 32) {
        if (lane < 9) {
            const int n = n_of(lane);
            F64[lane] = load_real_storage(Fp, n, lane - n * n - n);
        }
        if (lane == 31) upsilon_low_full(vx, vy, vz, Y64, true);
        __syncwarp();
        if (lane < 20) {
            const L2LTerm e = kL2LTerm[lane];
            prod[lane] = Y64[cix(e.k, e.l)] * F64[cix(e.n + e.k, e.m + e.l)];
        }
        __syncwarp();
        if (lane < 6) {
            cd v = mkc(0.0, 0.0);
            for (int i = kL2LStart[lane]; i < kL2LStart[lane + 1]; ++i) v = v + prod[i];
            low[lane] = v;
        }
    }
    if (W == 1) __syncwarp();
    else __syncthreads();
    for (int o = t; o < nout; o += T) {
        const int n = out_order(o), m = o - n * (n + 1) / 2;
        const double sc = pwi[n];
        double re = out[cix(n, m)], im = m ? out[cix(n, -m)] : 0.0;
        float2 v32 = make_float2(0.f, 0.f);
        for (int k = max(0, 3 - n); k <= p - n; ++k) {
            const float2* xk = Yh + k * k + k;
            const float2* yk = Fh + (n + k) * (n + k) + (n + k) + m;
#pragma unroll 4
            for (int l = -k; l <= k; ++l) cmacf(v32, xk[l], yk[l]);
        }
        if (n <= 2) {
            const cd v = low[o];
            re += v.re;
            im += v.im;
        }
        out[cix(n, m)] = fma((double)v32.x, sc, re);
        if (m) out[cix(n, -m)] = fma((double)v32.y, sc, im);
    }
}

template <int W>
static void go_l2l_split(Cells c, const d4* cen, const double* pw, int lev_begin, int lev_end, int p, double* F,
                         cudaStream_t s) {
    const int per = W == 1 ? 4 : 1;
    k_l2l_split<W><<<(unsigned)((lev_end - lev_begin + per - 1) / per), per * W * 32, per * l2l_cell_bytes(p), s>>>(
        c, cen, pw, lev_begin, lev_end, p, F);
    note_launch();
}
void launch_l2l_split(Cells c, const d4* cen, const double* pw, int lev_begin, int lev_end, int p, double* F, cudaStream_t s) {
    if (lev_end <= lev_begin) return;
    if (p < 3) {
        launch_l2l_level(c, cen, lev_begin, lev_end, p, F, s);
        return;
    }
    init_split_up_tables();
    switch ((out_count(p) + 31) / 32) {
        case 1: go_l2l_split<1>(c, cen, pw, lev_begin, lev_end, p, F, s); break;
        case 2: go_l2l_split<2>(c, cen, pw, lev_begin, lev_end, p, F, s); break;
        case 3: go_l2l_split<3>(c, cen, pw, lev_begin, lev_end, p, F, s); break;
        default: go_l2l_split<4>(c, cen, pw, lev_begin, lev_end, p, F, s); break;
    }
}

}  // namespace gb3
