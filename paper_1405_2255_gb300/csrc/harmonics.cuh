// harmonics.cuh -- device solid harmonics (eq. 2) and what the kernels of the expansions' shifts share
// (eqs. 3a, 4, 5, 7).
#pragma once
#include "common.cuh"

namespace gb3 {

// Recurrence coefficients as doubles (no integer-to-FP64 conversions in the loops):
// tw[n] = 2n - 1, inv_up[n][m] = 1 / (n^2 - m^2).
struct RecTables {
    double tw[kMaxP + 2];
    double inv_up[kMaxP + 1][kMaxP + 1];
    double up_a[kMaxP + 1][kMaxP + 1];  // (2n - 1) / (n^2 - m^2)
    double inv_2j[kMaxP + 1];  // 1 / (2j)
};
// one copy per translation unit (no relocatable device code); each unit that
// launches kernels using the recurrences calls init_rec_tables() first
static __constant__ RecTables c_rec;
static inline void init_rec_tables() {
    static DeviceOnce once;
    once_per_device(once, [] {
        RecTables t;
        memset(&t, 0, sizeof t);
        for (int n = 0; n <= kMaxP + 1; ++n) t.tw[n] = 2.0 * n - 1.0;
        for (int n = 0; n <= kMaxP; ++n)
            for (int m = 0; m <= kMaxP; ++m) {
                t.inv_up[n][m] = (n * n != m * m) ? 1.0 / (double)(n * n - m * m) : 0.0;
                t.up_a[n][m] = (n * n != m * m) ? (2.0 * n - 1.0) / (double)(n * n - m * m) : 0.0;
            }
        for (int j = 1; j <= kMaxP; ++j) t.inv_2j[j] = 1.0 / (2.0 * j);
        cudaMemcpyToSymbol(c_rec, &t, sizeof t);
    });
}

// 1 / (n^2 - m^2) for reads at a lane's own m (constant memory serves one address at a time)
struct InvUp {
    double v[kMaxP + 1][kMaxP + 1];
    constexpr InvUp() : v{} {
        for (int n = 0; n <= kMaxP; ++n)
            for (int m = 0; m <= kMaxP; ++m) v[n][m] = n != m ? 1.0 / (double)(n * n - m * m) : 0.0;
    }
};
static __device__ const InvUp g_inv_up = InvUp();

// The columns m >= 0 of the regular harmonics Upsilon_n^m(r), n = m..p, written to the full complex array
// out[cix(n, +-m)] (negative m by X_n^{-m} = (-1)^m X_n^{m*}).  Diagonal: Upsilon_m^m = prod_{j<=m}
// (x+iy)/(2j); then (n^2-m^2) Upsilon_n^m = (2n-1) z Upsilon_{n-1}^m - r^2 Upsilon_{n-2}^m (App. A.3.1).
// If conj_out, the conjugates are written instead.  Two threads per column (thread t of a block: column
// t / 2, t odd the imaginary parts), for t < 2 (p + 1) and the rest of their last warp (whole warps call
// it).  A warp that is alone on its part of the FP64 pipe takes 64 cycles per instruction, so the number of
// instructions per step counts.
__device__ inline void upsilon_columns2(int p, int t, double x, double y, double z, cd* out, bool conj_out) {
    const int m = min(t >> 1, p), last = min((t | 31) >> 1, p);
    const bool im = t & 1;
    const double r2 = x * x + y * y + z * z, ys = im ? y : -y;
    double d = im ? 0.0 : 1.0;
    for (int j = 1; j <= last; ++j) {
        const double other = __shfl_xor_sync(0xffffffffu, d, 1);
        const double v = c_rec.inv_2j[j] * (x * d + ys * other);
        if (j <= m) d = v;
    }
    if ((t >> 1) > p) return;
    const double cs = im && conj_out ? -1.0 : 1.0, sg = ((m & 1) ? -1.0 : 1.0) * (im ? -1.0 : 1.0);
    double prev2 = 0.0, prev = d;
    double* o = (double*)out + (im ? 1 : 0);
    for (int n = m; n <= p; ++n) {
        if (n > m) {
            const double v = ((c_rec.tw[n] * z) * prev - r2 * prev2) * g_inv_up.v[n][m];
            prev2 = prev;
            prev = v;
        }
        const double w = cs * prev;
        o[2 * cix(n, m)] = w;
        if (m) o[2 * cix(n, -m)] = sg * w;
    }
}

// the nine real-storage coefficients of Upsilon_n^m(d), n <= 2 (App. A.3.1 in closed form):
// U0 = 1, U1^0 = z, U1^1 = (x+iy)/2, U2^0 = (3z^2-r^2)/4, U2^1 = z(x+iy)/2, U2^2 = (x+iy)^2/8
__device__ inline void upsilon_low(double x, double y, double z, double u[9]) {
    const double r2 = x * x + y * y + z * z;
    u[cix(0, 0)] = 1.0;
    u[cix(1, -1)] = 0.5 * y;
    u[cix(1, 0)] = z;
    u[cix(1, 1)] = 0.5 * x;
    u[cix(2, -2)] = 0.25 * x * y;
    u[cix(2, -1)] = 0.5 * z * y;
    u[cix(2, 0)] = 0.25 * (3.0 * z * z - r2);
    u[cix(2, 1)] = 0.5 * z * x;
    u[cix(2, 2)] = 0.125 * (x * x - y * y);
}

// a sum of complex products as four chains (the latency of an FP64 addition, not the pipe, is what a warp
// that is alone waits for)
struct cd4 {
    double rr, ii, ri, ir;
    __device__ __forceinline__ void add(cd a, cd b) {
        rr = fma(a.re, b.re, rr);
        ii = fma(a.im, b.im, ii);
        ri = fma(a.re, b.im, ri);
        ir = fma(a.im, b.re, ir);
    }
    __device__ __forceinline__ cd sum() const { return cd{rr - ii, ri + ir}; }
};

// complex FP32 multiply-accumulate: acc += a * b
__device__ inline void cmacf(float2& acc, float2 a, float2 b) {
    acc.x = fmaf(a.x, b.x, acc.x);
    acc.x = fmaf(-a.y, b.y, acc.x);
    acc.y = fmaf(a.x, b.y, acc.y);
    acc.y = fmaf(a.y, b.x, acc.y);
}

// expand a real-storage expansion into a full complex array (optionally conjugated)
__device__ inline void expand_real(int p, const double* R, cd* out, bool conj_out, int lane, int nlanes) {
    const int nc = ncoef(p);
    for (int i = lane; i < nc; i += nlanes) {
        int n = (int)sqrtf((float)i);
        while (n * n > i) --n;
        while ((n + 1) * (n + 1) <= i) ++n;
        int m = i - n * n - n;
        cd v = load_real_storage(R, n, m);
        out[i] = conj_out ? conjc(v) : v;
    }
}

// Outputs (n, m), 0 <= m <= n, of an expansion by index o = n (n + 1) / 2 + m.  The kernels that form all
// outputs of one shift (M2M, L2L) give each thread one output, in the order of the outputs' terms, so that
// the lanes of a warp have about the same number of them: dealt out to the 32 lanes of one warp by a table
// of the longest first, a lane waited at each of its outputs for the longest of the others', 32 us for a
// level of any size at p = 14 (the sums themselves keep their order).
__host__ __device__ inline int out_count(int p) { return (p + 1) * (p + 2) / 2; }
__device__ __forceinline__ int out_order(int o) {
    int n = (int)((sqrtf(8.f * (float)o + 1.f) - 1.f) * 0.5f);
    while (n * (n + 1) / 2 > o) --n;
    while ((n + 1) * (n + 2) / 2 <= o) ++n;
    return n;
}

}  // namespace gb3
