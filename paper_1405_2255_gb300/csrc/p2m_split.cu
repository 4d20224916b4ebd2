// p2m_split.cu -- P2M (eq. 3c).  In mixed mode the orders n <= 2 in FP64, the higher orders in FP32 on the
// offsets scaled by the cell's radius (Upsilon_n^m((x - z)/rho), bounded by 1/n!), rescaled in FP64; in
// FP64 mode all orders in FP64.
//
// One warp per leaf, lane = particle; the columns of Upsilon come from their recurrences in registers
// and every coefficient is summed over the warp.  What bounds it is the number of instructions (ALU and
// shuffles; 0.55 ms for the 43,413 leaves of a Plummer sphere of 1e6 at p = 14 with five shuffles and
// additions per coefficient and a run-time order).  So the order is a compile-time constant and 32
// coefficients are summed together: at each step of a butterfly (xor 16, 8, 4, 2, 1) a lane passes on
// the half of the coefficients that it will not keep, 31 shuffles and additions for 32 sums that end in
// 32 lanes, in the order of the single butterflies: 0.21 ms.  In FP64 (bound by the FP64 pipe) the same,
// the reciprocals of the recurrence being constants: 1e5 particles at p = 10 took 0.84 ms with a division
// and ten additions per coefficient, 0.21 ms so.
#include <utility>

#include "harmonics.cuh"
#include "kernels.cuh"

namespace gb3 {
namespace {

constexpr int kWarps = 4;

// the sum of value j over the warp ends in lane j
template <int S, class T>
__device__ __forceinline__ void halve(T (&v)[32], int lane) {
    const bool hi = lane & S;
#pragma unroll
    for (int i = 0; i < S; ++i) {
        const T keep = hi ? v[i + S] : v[i], send = hi ? v[i] : v[i + S];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, S);
    }
}
template <class T>
__device__ __forceinline__ T sums32(T (&v)[32], int lane) {
    halve<16>(v, lane);
    halve<8>(v, lane);
    halve<4>(v, lane);
    halve<2>(v, lane);
    halve<1>(v, lane);
    return v[0];
}
// the same for the nine FP64 values of the low orders: value j ends in lane sum9_lane(j)
__device__ inline double sum9(const double (&v)[9], int lane) {
    double a[5], b[3];
    const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4, h2 = lane & 2;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const double keep = h16 ? v[i + 4] : v[i], send = h16 ? v[i] : v[i + 4];
        a[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
    }
    a[4] = v[8] + __shfl_xor_sync(0xffffffffu, v[8], 16);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const double keep = h8 ? a[i + 2] : a[i], send = h8 ? a[i] : a[i + 2];
        b[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
    }
    b[2] = a[4] + __shfl_xor_sync(0xffffffffu, a[4], 8);
    const double k1 = h4 ? b[1] : b[0], s1 = h4 ? b[0] : b[1];
    double c = k1 + __shfl_xor_sync(0xffffffffu, s1, 4);
    const double d = b[2] + __shfl_xor_sync(0xffffffffu, b[2], 4);
    const double k2 = h2 ? d : c, s2 = h2 ? c : d;  // lanes with bit 2 set go on with value 8
    c = k2 + __shfl_xor_sync(0xffffffffu, s2, 2);
    return c + __shfl_xor_sync(0xffffffffu, c, 1);
}
__device__ __forceinline__ int sum9_lane(int j) {
    return j == 8 ? 2 : ((j & 4) ? 16 : 0) + ((j & 2) ? 8 : 0) + ((j & 1) ? 4 : 0);
}

// places of the summed coefficients (n >= N0), column by column, real part before imaginary part
template <int P, int N0>
struct Slots {
    static constexpr int N = (P + 1) * (P + 1) - N0 * N0;
    short at[N > 0 ? N : 1];
    unsigned char n[N > 0 ? N : 1];
    constexpr Slots() : at{}, n{} {
        int k = 0;
        for (int m = 0; m <= P; ++m)
            for (int j = m > N0 ? m : N0; j <= P; ++j) {
                at[k] = (short)(j * j + j + m);
                n[k++] = (unsigned char)j;
                if (m) {
                    at[k] = (short)(j * j + j - m);
                    n[k++] = (unsigned char)j;
                }
            }
    }
};
template <int P, int N0>
__device__ constexpr Slots<P, N0> kSlots = Slots<P, N0>();

// values before coefficient (n, m), n >= N0, in that order
template <int P, int N0>
constexpr int value_index(int n, int m) {
    int k = 0;
    for (int j = 0; j < m; ++j) k += (j ? 2 : 1) * (P - (j > N0 ? j : N0) + 1);
    return k + (m ? 2 : 1) * (n - (m > N0 ? m : N0));
}
// coefficient (N, M) of the lane's particle and the rest of its column (compile-time recursion, so
// that every value has its register): (px, py) and (qx, qy) the two before it in its column, (dr, di)
// the diagonal.  Explicit operations, so that the rounding does not depend on how a compiler contracts them
__device__ __forceinline__ float mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul(double a, double b) { return __dmul_rn(a, b); }
template <int P, class T, int N0>
struct Columns {
    T x, y, z, r2, dr, di, px, py, qx, qy;
    T v[32];
    static constexpr int G = (Slots<P, N0>::N + 31) / 32 > 0 ? (Slots<P, N0>::N + 31) / 32 : 1;
    T acc[G];
    int lane;
    template <int K>
    __device__ __forceinline__ void put(T a) {
        v[K & 31] = a;
        if constexpr ((K & 31) == 31) acc[K / 32] += sums32(v, lane);
    }
    template <int M, int N>
    __device__ __forceinline__ void step() {
        if constexpr (N == M) {
            if constexpr (M > 0) {
                constexpr T s = T(1) / (T(2) * (T)M);
                const T re = mul(s, fma(x, dr, -mul(y, di)));
                di = mul(s, fma(x, di, mul(y, dr)));
                dr = re;
            }
            px = dr;
            py = di;
            qx = qy = T(0);
        } else {
            constexpr T iv = T(1) / (T)(N * N - M * M);
            const T a = mul((T)(2 * N - 1), z);
            const T vx = mul(fma(a, px, -mul(r2, qx)), iv);
            const T vy = mul(fma(a, py, -mul(r2, qy)), iv);
            qx = px;
            qy = py;
            px = vx;
            py = vy;
        }
        if constexpr (N >= N0) {
            put<value_index<P, N0>(N, M)>(px);
            if constexpr (M > 0) put<value_index<P, N0>(N, M) + 1>(py);
        }
        if constexpr (N < P) step<M, N + 1>();
    }
    template <int... M>
    __device__ __forceinline__ void columns(std::integer_sequence<int, M...>) {
        (step<M, M>(), ...);
    }
    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int i = 0; i < G; ++i) acc[i] = T(0);
    }
    __device__ __forceinline__ void run(T ax, T ay, T az, T mu) {
        x = ax;
        y = ay;
        z = az;
        r2 = fma(z, z, fma(x, x, mul(y, y)));
        dr = mu;
        di = T(0);
        columns(std::make_integer_sequence<int, P + 1>{});
        if constexpr (Slots<P, N0>::N & 31) {
#pragma unroll
            for (int k = Slots<P, N0>::N & 31; k < 32; ++k) v[k] = T(0);
            acc[Slots<P, N0>::N / 32] += sums32(v, lane);
        }
    }
};

template <int P>
__global__ void __launch_bounds__(kWarps * 32) k_p2m_split(const d4* __restrict__ xm, Cells c,
                                                           const d4* __restrict__ cen,
                                                           const double* __restrict__ pw,
                                                           const int* __restrict__ leaves, int nleaves,
                                                           double* __restrict__ M) {
    constexpr int NV = Slots<P, 3>::N, G = (NV + 31) / 32;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = blockIdx.x * kWarps + wid;
    if (t >= nleaves) return;
    const int cell = leaves[t];
    const d4 z = cen[cell];
    const double* pc = pw + (size_t)cell * 2 * (P + 1);
    const double rho = z.w, rinv = pc[P + 2];
    const int first = c.first[cell], count = c.count[cell];
    double lo[9];
    Columns<P, float, 3> col;
    col.lane = lane;
    col.clear();
#pragma unroll
    for (int i = 0; i < 9; ++i) lo[i] = 0.0;
    for (int b = 0; b < count; b += 32) {
        const int i = b + lane;
        double dx = 0, dy = 0, dz = 0, mu = 0;
        if (i < count) {
            const d4 q = xm[first + i];
            dx = q.x - z.x; dy = q.y - z.y; dz = q.z - z.z; mu = q.w;
        }
        double u[9];
        upsilon_low(dx, dy, dz, u);
#pragma unroll
        for (int k = 0; k < 9; ++k) lo[k] = fma(mu, u[k], lo[k]);
        // mu * Upsilon_n^m((x - z)/rho) in FP32, n >= 3 kept
        if (rho > 0 && P > 2) col.run((float)(dx * rinv), (float)(dy * rinv), (float)(dz * rinv), (float)mu);
    }
    const double low = sum9(lo, lane);
    double* out = M + (size_t)cell * ncoef(P);
#pragma unroll
    for (int j = 0; j < 9; ++j)
        if (lane == sum9_lane(j)) out[j] = low;
#pragma unroll
    for (int g = 0; g < G; ++g) {
        const int j = 32 * g + lane;
        if (j < NV) out[kSlots<P, 3>.at[j]] = (double)col.acc[g] * pc[kSlots<P, 3>.n[j]];
    }
}

template <int P>
__global__ void __launch_bounds__(kWarps * 32) k_p2m(const d4* __restrict__ xm, Cells c, const d4* __restrict__ cen,
                                                     const int* __restrict__ leaves, int nleaves,
                                                     double* __restrict__ M) {
    constexpr int NV = Slots<P, 0>::N;
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int t = blockIdx.x * kWarps + wid;
    if (t >= nleaves) return;
    const int cell = leaves[t];
    const d4 z = cen[cell];
    const int first = c.first[cell], count = c.count[cell];
    Columns<P, double, 0> col;
    col.lane = lane;
    col.clear();
    for (int b = 0; b < count; b += 32) {
        const int i = b + lane;
        double dx = 0, dy = 0, dz = 0, mu = 0;
        if (i < count) {
            const d4 q = xm[first + i];
            dx = q.x - z.x; dy = q.y - z.y; dz = q.z - z.z; mu = q.w;
        }
        col.run(dx, dy, dz, mu);
    }
    double* out = M + (size_t)cell * ncoef(P);
#pragma unroll
    for (int g = 0; g < Columns<P, double, 0>::G; ++g) {
        const int j = 32 * g + lane;
        if (j < NV) out[kSlots<P, 0>.at[j]] = col.acc[g];
    }
}

template <int P>
void go64(const d4* xm, Cells c, const d4* cen, const int* leaves, int nleaves, double* M, cudaStream_t s) {
    k_p2m<P><<<(nleaves + kWarps - 1) / kWarps, kWarps * 32, 0, s>>>(xm, c, cen, leaves, nleaves, M);
    note_launch();
}

template <int P>
void go(const d4* xm, Cells c, const d4* cen, const double* pw, const int* leaves, int nleaves, double* M,
        cudaStream_t s) {
    k_p2m_split<P><<<(nleaves + kWarps - 1) / kWarps, kWarps * 32, 0, s>>>(xm, c, cen, pw, leaves, nleaves, M);
    note_launch();
}
}  // namespace

void launch_p2m(const d4* xm, Cells c, const d4* cen, const int* leaves, int nleaves, int p, double* M,
                cudaStream_t s) {
    static_assert(kMaxP == 20, "one case per order");
    if (nleaves <= 0) return;
    switch (p) {
#define GB3_P2M(P) \
    case P: go64<P>(xm, c, cen, leaves, nleaves, M, s); break;
        GB3_P2M(0) GB3_P2M(1) GB3_P2M(2) GB3_P2M(3) GB3_P2M(4) GB3_P2M(5) GB3_P2M(6) GB3_P2M(7) GB3_P2M(8)
        GB3_P2M(9) GB3_P2M(10) GB3_P2M(11) GB3_P2M(12) GB3_P2M(13) GB3_P2M(14) GB3_P2M(15) GB3_P2M(16)
        GB3_P2M(17) GB3_P2M(18) GB3_P2M(19) GB3_P2M(20)
#undef GB3_P2M
    }
}

void launch_p2m_split(const d4* xm, Cells c, const d4* cen, const double* pw, const int* leaves, int nleaves, int p,
                      double* M, cudaStream_t s) {
    if (nleaves <= 0) return;
    switch (p) {
#define GB3_P2M(P) \
    case P: go<P>(xm, c, cen, pw, leaves, nleaves, M, s); break;
        GB3_P2M(2) GB3_P2M(3) GB3_P2M(4) GB3_P2M(5) GB3_P2M(6) GB3_P2M(7) GB3_P2M(8) GB3_P2M(9) GB3_P2M(10)
        GB3_P2M(11) GB3_P2M(12) GB3_P2M(13) GB3_P2M(14) GB3_P2M(15) GB3_P2M(16) GB3_P2M(17) GB3_P2M(18)
        GB3_P2M(19) GB3_P2M(20)
#undef GB3_P2M
        default: launch_p2m(xm, c, cen, leaves, nleaves, p, M, s); break;  // p < 2: nothing to split
    }
}

}  // namespace gb3
