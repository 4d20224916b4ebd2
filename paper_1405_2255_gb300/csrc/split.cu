// split.cu -- mixed-mode M2M (eq. 4), L2L (eq. 5) and L2P (eqs. 3a, 7; P2M: p2m_split.cu) with the same order
// split as the M2L: the expansion orders n <= 2 are formed in FP64, the higher
// orders in FP32 on quantities scaled by the cell radius (Upsilon evaluated at
// (x - z)/rho, whose values are bounded by 1/n!), then rescaled in FP64.  The
// higher orders carry a fraction ~ theta^n of an expansion's contribution, so
// FP32 rounding there stays far below the targeted force error.
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
// out (full complex, FP32) = R (real storage) times sc[n] for the (p+1)^2 coefficients, one warp
__device__ __forceinline__ void expand_scaled(const double* __restrict__ R, const double* __restrict__ sc, int nco,
                                              int lane, float2* out) {
    for (int i = lane; i < nco; i += 32) {
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
    expand_scaled(Fr, pc, nco, lane, Fh);
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
            const float a = c_twf2[n] * z, iv = c_inv_upf[n][m];
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
// Uhat_k = Upsilon_k((z - z')/rho'), Mt_j = M_j(z) / rho'^j.  One block per parent and one
// warp per daughter; the daughters' contributions are then summed in daughter order.
constexpr int kM2MWarps = 8;
__host__ __device__ inline size_t m2m_warp_bytes(int p) {
    return ((size_t)2 * ncoef(p) * sizeof(float2) + 18 * sizeof(cd) + 15) & ~(size_t)15;
}
__host__ __device__ inline size_t m2m_smem_bytes(int p) {
    const size_t nout = (size_t)(p + 1) * (p + 2) / 2;
    return kM2MWarps * m2m_warp_bytes(p) + kM2MWarps * nout * sizeof(float2) + kM2MWarps * 6 * sizeof(cd);
}
template <int MAXQ>
__global__ void __launch_bounds__(kM2MWarps * 32) k_m2m_split(Cells c, const d4* __restrict__ cen,
                                                               const double* __restrict__ pw, int lev_begin,
                                                               int lev_end, int p, double* __restrict__ M,
                                                               LaneSched sched) {
    extern __shared__ __align__(16) unsigned char sraw[];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nco = ncoef(p), nout = (p + 1) * (p + 2) / 2;
    const size_t per_warp = m2m_warp_bytes(p);
    float2* Yh = (float2*)(sraw + wid * per_warp);
    float2* Mt = Yh + nco;
    cd* Y64 = (cd*)(Mt + nco);
    cd* M64 = Y64 + 9;
    float2* r32 = (float2*)(sraw + kM2MWarps * per_warp);  // [kM2MWarps][nout]
    cd* r64 = (cd*)(r32 + kM2MWarps * nout);                // [kM2MWarps][6]
    const int cell = lev_begin + blockIdx.x;
    if (cell >= lev_end) return;
    const int nch = c.nchild[cell];
    if (nch == 0) return;  // leaves
    const d4 zp = cen[cell];
    const double *pwr = pw + (size_t)cell * 2 * (p + 1), *pwi = pwr + p + 1;  // rho^n, rho^-n
    const double rho = zp.w, inv = pwi[1];
    if (wid < nch) {
        const int cnt = sched.cnt[lane];
        const int d = c.child[cell] + wid;
        const d4 z = cen[d];
        const double vx = z.x - zp.x, vy = z.y - zp.y, vz = z.z - zp.z;
        if (lane <= p) upsilon_column_f(p, lane, (float)(vx * inv), (float)(vy * inv), (float)(vz * inv), Yh, false);
        const double* Md = M + (size_t)d * nco;
        expand_scaled(Md, pwi, nco, lane, Mt);
        if (lane < 9) {
            const int n = n_of(lane);
            M64[lane] = load_real_storage(Md, n, lane - n * n - n);
        }
        if (lane == 0) upsilon_low_full(vx, vy, vz, Y64, false);
        __syncwarp();
#pragma unroll
        for (int q = 0; q < MAXQ; ++q) {
            if (q < cnt) {
                const int n = sched.n[lane][q], m = sched.m[lane][q];
                const int o = n * (n + 1) / 2 + m;
                if (n <= 2) {
                    cd sum = mkc(0.0, 0.0);
                    for (int k = 0; k <= n; ++k) {
                        const int nn = n - k;
                        for (int l = max(-k, m - nn); l <= min(k, m + nn); ++l)
                            cmac(sum, Y64[cix(k, l)], M64[cix(nn, m - l)]);
                    }
                    r64[wid * 6 + o] = sum;
                } else {
                    float2 sum = make_float2(0.f, 0.f);
                    if (rho > 0)
                        for (int k = 0; k <= n; ++k) {
                            const int nn = n - k;
                            for (int l = max(-k, m - nn); l <= min(k, m + nn); ++l)
                                cmacf(sum, Yh[cix(k, l)], Mt[cix(nn, m - l)]);
                        }
                    r32[wid * nout + o] = sum;
                }
            }
        }
    }
    __syncthreads();
    // the parent's moments: the daughters' terms summed in daughter order
    double* out = M + (size_t)cell * nco;
    for (int o = threadIdx.x; o < nout; o += blockDim.x) {
        int n = 0;
        while ((n + 1) * (n + 2) / 2 <= o) ++n;
        const int m = o - n * (n + 1) / 2;
        cd v;
        if (n <= 2) {
            v = mkc(0.0, 0.0);
            for (int j = 0; j < nch; ++j) v = v + r64[j * 6 + o];
        } else {
            float2 a = make_float2(0.f, 0.f);
            for (int j = 0; j < nch; ++j) {
                a.x += r32[j * nout + o].x;
                a.y += r32[j * nout + o].y;
            }
            const double sc = pwr[n];
            v = mkc((double)a.x * sc, (double)a.y * sc);
        }
        out[cix(n, m)] = v.re;
        if (m) out[cix(n, -m)] = v.im;
    }
}

void launch_m2m_split(Cells c, const d4* cen, const double* pw, int lev_begin, int lev_end, int p, double* M, cudaStream_t s) {
    const int ncl = lev_end - lev_begin;
    if (ncl <= 0) return;
    if (p < 3) {
        launch_m2m_level(c, cen, lev_begin, lev_end, p, M, s);
        return;
    }
    init_split_up_tables();
    LaneSched sched = make_lane_sched(p, kSchedUp);
    int maxq = 0;
    for (int l = 0; l < 32; ++l) maxq = sched.cnt[l] > maxq ? sched.cnt[l] : maxq;
    const size_t sm = m2m_smem_bytes(p);
    const unsigned g = (unsigned)ncl;  // one block per cell of the level (leaves return at once)
    if (maxq <= 4) {
        cudaFuncSetAttribute(k_m2m_split<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        k_m2m_split<4><<<g, kM2MWarps * 32, sm, s>>>(c, cen, pw, lev_begin, lev_end, p, M, sched);
    } else if (maxq <= 8) {
        cudaFuncSetAttribute(k_m2m_split<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        k_m2m_split<8><<<g, kM2MWarps * 32, sm, s>>>(c, cen, pw, lev_begin, lev_end, p, M, sched);
    } else {
        cudaFuncSetAttribute(k_m2m_split<24>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
        k_m2m_split<24><<<g, kM2MWarps * 32, sm, s>>>(c, cen, pw, lev_begin, lev_end, p, M, sched);
    }
    note_launch();
}

// ---------------------------------------------------------------- L2L
// F_n^m(s') += sum_{k<=p-n} sum_l Upsilon_k^{l*}(s - s') F_{n+k}^{m+l}(s): terms with n+k <= 2
// in FP64, the others in FP32 as rho^-n sum Uhat_k^{l*} Fhat_{n+k}^{m+l} with
// Uhat_k = Upsilon_k((s - s')/rho), Fhat_j = F_j(s) rho^j (rho: the parent's radius).
// One warp per cell.  The FP64 terms of the six outputs n <= 2 are 20 products, one per lane.
struct L2LTerm {
    signed char n, m, k, l;
};
__device__ constexpr L2LTerm kL2LTerm[20] = {
    {0, 0, 0, 0},  {0, 0, 1, -1}, {0, 0, 1, 0}, {0, 0, 1, 1},  {0, 0, 2, -2}, {0, 0, 2, -1}, {0, 0, 2, 0},
    {0, 0, 2, 1},  {0, 0, 2, 2},  {1, 0, 0, 0}, {1, 0, 1, -1}, {1, 0, 1, 0},  {1, 0, 1, 1},  {1, 1, 0, 0},
    {1, 1, 1, -1}, {1, 1, 1, 0},  {1, 1, 1, 1}, {2, 0, 0, 0},  {2, 1, 0, 0},  {2, 2, 0, 0}};
__device__ constexpr int kL2LStart[7] = {0, 9, 13, 17, 18, 19, 20};  // first product of output n (n + 1) / 2 + m
__host__ __device__ inline size_t l2l_warp_bytes(int p) {
    return ((size_t)2 * ncoef(p) * sizeof(float2) + (9 + 9 + 20 + 6) * sizeof(cd) + 15) & ~(size_t)15;
}
__global__ void __launch_bounds__(128) k_l2l_split(Cells c, const d4* __restrict__ cen,
                                                   const double* __restrict__ pw, int lev_begin, int lev_end,
                                                   int p, double* __restrict__ F, LaneSched sched) {
    extern __shared__ __align__(16) unsigned char sraw[];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nco = ncoef(p);
    cd* Y64 = (cd*)(sraw + wid * l2l_warp_bytes(p));
    cd* F64 = Y64 + 9;
    cd* prod = F64 + 9;
    cd* low = prod + 20;
    float2* Yh = (float2*)(low + 6);
    float2* Fh = Yh + nco;
    const int cell = lev_begin + blockIdx.x * 4 + wid;
    if (cell >= lev_end || !cell_active(c, cell)) return;
    const int par = c.parent[cell];
    const d4 s = cen[par], sp = cen[cell];
    const double rho = s.w;
    double* out = F + (size_t)cell * nco;
    const double* Fp = F + (size_t)par * nco;
    if (!(rho > 0)) {  // all particles at the parent's centre: the shift is the identity
        for (int i = lane; i < nco; i += 32) out[i] += Fp[i];
        return;
    }
    const double *pwr = pw + (size_t)par * 2 * (p + 1), *pwi = pwr + p + 1;  // rho^n, rho^-n
    const double inv = pwi[1];
    const double vx = s.x - sp.x, vy = s.y - sp.y, vz = s.z - sp.z;
    if (lane <= p) upsilon_column_f(p, lane, (float)(vx * inv), (float)(vy * inv), (float)(vz * inv), Yh, true);
    expand_scaled(Fp, pwr, nco, lane, Fh);
    if (lane < 9) {
        const int n = n_of(lane);
        F64[lane] = load_real_storage(Fp, n, lane - n * n - n);
    }
    if (lane == 0) upsilon_low_full(vx, vy, vz, Y64, true);
    __syncwarp();
    if (lane < 20) {
        const L2LTerm t = kL2LTerm[lane];
        prod[lane] = Y64[cix(t.k, t.l)] * F64[cix(t.n + t.k, t.m + t.l)];
    }
    __syncwarp();
    if (lane < 6) {
        cd v = mkc(0.0, 0.0);
        for (int i = kL2LStart[lane]; i < kL2LStart[lane + 1]; ++i) v = v + prod[i];
        low[lane] = v;
    }
    __syncwarp();
    const int cnt = sched.cnt[lane];
    for (int q = 0; q < cnt; ++q) {
        const int n = sched.n[lane][q], m = sched.m[lane][q];
        float2 v32 = make_float2(0.f, 0.f);
        for (int k = max(0, 3 - n); k <= p - n; ++k) {
            const float2* xk = Yh + k * k + k;
            const float2* yk = Fh + (n + k) * (n + k) + (n + k) + m;
            for (int l = -k; l <= k; ++l) cmacf(v32, xk[l], yk[l]);
        }
        const double sc = pwi[n];
        double re = out[cix(n, m)], im = m ? out[cix(n, -m)] : 0.0;
        if (n <= 2) {
            const cd v = low[n * (n + 1) / 2 + m];
            re += v.re;
            im += v.im;
        }
        out[cix(n, m)] = fma((double)v32.x, sc, re);
        if (m) out[cix(n, -m)] = fma((double)v32.y, sc, im);
    }
}

void launch_l2l_split(Cells c, const d4* cen, const double* pw, int lev_begin, int lev_end, int p, double* F, cudaStream_t s) {
    const int ncl = lev_end - lev_begin;
    if (ncl <= 0) return;
    if (p < 3) {
        launch_l2l_level(c, cen, lev_begin, lev_end, p, F, s);
        return;
    }
    init_split_up_tables();
    LaneSched sched = make_lane_sched(p, kSchedDown);
    const size_t sm = 4 * l2l_warp_bytes(p);
    cudaFuncSetAttribute(k_l2l_split, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    k_l2l_split<<<(unsigned)((ncl + 3) / 4), 128, sm, s>>>(c, cen, pw, lev_begin, lev_end, p, F, sched);
    note_launch();
}

}  // namespace gb3
