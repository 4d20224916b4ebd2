// m2l_f64.cu -- A9 in FP64: the M2L of eq. (3b) through rotations into the frame of the interaction
// (App. A.5: eq. A31 along the z axis, the swap matrices of App. A.5.1), O(p^3) per pair.  The frames,
// the normalisation and the real storage are those of m2l_rot.cuh; every operation is IEEE FP64.
//
// What bounds it: the FP64 pipe (2 lanes a cycle and SM, an instruction costs the same however many
// of its lanes are active; 64 issue slots pass per FP64 instruction of a scheduler, so loads, indexing
// and shared-memory traffic are hidden behind it).  So the form with the fewest FP64 operations wins
// (p = 14: 5,774 multiply-adds a pair against 21,760 of eq. 3b term by term; p = 10: 2,564 against
// 6,864), in loops over the order (no code per order), and every lane has to hold a pair: lane = pair,
// a sink's list is cut into chunks of 32 pairs and the last, shorter chunks of several sinks share a
// warp in groups of 8 lanes.  A chunk's pairs are added in list order and a sink's chunks in chunk
// order, whatever shares their warp, so a system gives the same bits in an ensemble as alone.
// Shared memory holds, per warp, the rotated multipoles (entries |m| <= min(k, p - k) only, all that
// eq. A31 reads: 113 of 225 at p = 14) and work vectors of 4 p + 3 rows: five warps an SM at p = 14,
// eight at p = 10 (two more rows of 2 p + 1 left room for four and six, and for some of the latency:
// 5.0 and 3.5 ms below).  1e5 particles, p = 10 (598,127 pairs): 31.9 ms with eq. 3b term by term, 4.36 ms
// so (2.9 ms at the pipe's rate); 6e4 cusp, p = 14 (143,081 pairs): 30.7 -> 3.10 ms (1.6).
#include <vector>

#include "kernels.cuh"

namespace gb3 {
namespace {

constexpr int kOrd = kMaxP + 1;
constexpr int kPitch = 33;  // doubles per row of the work vectors (a row is read along and across lanes)
constexpr int kZm = kMaxP / 2 + 1;

struct F64Tab {
    double norm[kOrd * kOrd];           // N_n^|m| = sqrt((n-m)! (n+m)!) at n^2 + n + m
    int off[kOrd][2][2];                // sw offsets: [n][0 cosine, 1 sine block][row parity]
    double sw[3200];                    // nonzero entries of Bhat_n: [column][row], rows of one parity
    double z[kOrd * kZm * kOrd];        // (-1)^m (n+k)! / (N_k^m N_n^m) at (n * kZm + m) * kOrd + k
};
__device__ F64Tab g_tab;

// first row and column of a block: cosine entries have n + m + l even (m, l >= 0), sine entries
// n + m + l odd (m, l >= 1); a = parity of the rows m
__host__ __device__ inline int row0(int sine, int a) { return sine && a == 0 ? 2 : a; }
__host__ __device__ inline int col0(int n, int sine, int a) {
    const int par = (n + a + sine) & 1;
    return sine && par == 0 ? 2 : par;
}
__host__ __device__ inline int steps2(int first, int last) { return last < first ? 0 : (last - first) / 2 + 1; }

void init_tab() {
    static DeviceOnce once;
    once_per_device(once, [] {
        std::vector<F64Tab> hold(1);
        F64Tab& t = hold[0];
        memset(&t, 0, sizeof t);
        double fact[2 * kMaxP + 1];
        fact[0] = 1.0;
        for (int i = 1; i <= 2 * kMaxP; ++i) fact[i] = fact[i - 1] * i;
        auto nrm = [&](int n, int m) { return sqrt(fact[n - m] * fact[n + m]); };
        for (int n = 0; n <= kMaxP; ++n)
            for (int m = -n; m <= n; ++m) t.norm[cix(n, m)] = nrm(n, m < 0 ? -m : m);
        for (int n = 0; n <= kMaxP; ++n)
            for (int m = 0; m < kZm; ++m)
                for (int k = m; k + n <= kMaxP; ++k)
                    if (m <= n) t.z[(n * kZm + m) * kOrd + k] = ((m & 1) ? -1.0 : 1.0) * fact[n + k] / (nrm(k, m) * nrm(n, m));
        // B_n by the recurrences of App. A.5.1 (dyadic rationals, exact in FP64)
        constexpr int O = kMaxP + 1, W = 2 * O + 1;
        std::vector<double> b(W * W, 0.0), nb;
        auto at = [&](int m, int l) -> double { return b[(O + m) * W + O + l]; };
        b[O * W + O] = 1.0;
        int used = 0;
        for (int n = 0; n <= kMaxP; ++n) {
            for (int sine = 0; sine < 2; ++sine)
                for (int a = 0; a < 2; ++a) {
                    t.off[n][sine][a] = used;
                    for (int l = col0(n, sine, a); l <= n; l += 2)
                        for (int m = row0(sine, a); m <= n; m += 2) {
                            const double f = nrm(n, l) / nrm(n, m), sg = (l & 1) ? -1.0 : 1.0;
                            const double bp = at(m, l) * f, bm = at(m, -l) * f;
                            t.sw[used++] = sine ? bp - sg * bm : (l == 0 ? bp : bp + sg * bm);
                        }
                }
            if (n == kMaxP) break;
            nb.assign(W * W, 0.0);
            for (int l = -(n + 1); l <= n + 1; ++l) {
                for (int m = -n; m <= n; ++m) nb[(O + m) * W + O + l] = 0.5 * (at(m, l - 1) - at(m, l + 1));
                nb[(O + n + 1) * W + O + l] = 0.5 * (at(n, l - 1) + at(n, l + 1)) + at(n, l);
                nb[(O - n - 1) * W + O + l] = 0.5 * (at(-n, l - 1) + at(-n, l + 1)) - at(-n, l);
            }
            b.swap(nb);
        }
        cudaMemcpyToSymbol(g_tab, &t, sizeof t);
    });
}

// ---------------------------------------------------------------- one order of one pair, in shared memory
// Pointers are to the centre entry (m = 0) of the lane's column; Re X^m sits m rows above, Im X^m m
// rows below.

// NR rows of one parity: out^{m} = (sum_l C[l][m] in^{l}) * sc
template <int NR>
__device__ __forceinline__ void swap_rows(const double* __restrict__ C, int cstride, const double* in, int istep,
                                          int ncol, double* out, int ostep, double sc) {
    double acc[NR];
#pragma unroll
    for (int r = 0; r < NR; ++r) acc[r] = 0.0;
#pragma unroll 2
    for (int i = 0; i < ncol; ++i) {
        const double x = *in;
#pragma unroll
        for (int r = 0; r < NR; ++r) acc[r] = fma(__ldg(C + r), x, acc[r]);
        in += istep;
        C += cstride;
    }
#pragma unroll
    for (int r = 0; r < NR; ++r) out[r * ostep] = sc == 1.0 ? acc[r] : acc[r] * sc;
}
// out = Bhat_n in for the rows |m| <= RL, from the entries |l| <= CL
__device__ void swap_xz(int n, int RL, int CL, const double* in, int ip, double* out, int op, double sc) {
    for (int sine = 0; sine < 2; ++sine) {
        const int si = sine ? -ip : ip, so = sine ? -op : op;
        for (int a = 0; a < 2; ++a) {
            const int m0 = row0(sine, a), l0 = col0(n, sine, a);
            const int nr = steps2(m0, RL), nc = steps2(l0, CL), cs = steps2(m0, n);
            const double* C = g_tab.sw + g_tab.off[n][sine][a];
            const double* x = in + l0 * si;
            double* y = out + m0 * so;
            int r = 0;
            for (; r + 4 <= nr; r += 4) swap_rows<4>(C + r, cs, x, 2 * si, nc, y + 2 * r * so, 2 * so, sc);
            switch (nr - r) {
                case 3: swap_rows<3>(C + r, cs, x, 2 * si, nc, y + 2 * r * so, 2 * so, sc); break;
                case 2: swap_rows<2>(C + r, cs, x, 2 * si, nc, y + 2 * r * so, 2 * so, sc); break;
                case 1: swap_rows<1>(C + r, cs, x, 2 * si, nc, y + 2 * r * so, 2 * so, sc); break;
                default: break;
            }
        }
    }
}
// X^m *= (cr + i sg ci)[m]
__device__ __forceinline__ void zrot(int n, double* x, int p, const double* cr, const double* ci, bool conj) {
#pragma unroll 2
    for (int m = 1; m <= n; ++m) {
        const double re = x[m * p], im = x[-m * p], c = cr[m], s = conj ? -ci[m] : ci[m];
        x[m * p] = fma(re, c, -(im * s));
        x[-m * p] = fma(re, s, im * c);
    }
}

__host__ __device__ inline int rot_entries(int p) {  // sum over k of 2 min(k, p - k) + 1
    int t = 0;
    for (int k = 0; k <= p; ++k) t += 2 * (k < p - k ? k : p - k) + 1;
    return t;
}
__host__ inline size_t m2l_f64_smem(int p) {
    return ((size_t)rot_entries(p) * 32 + (size_t)(4 * p + 3) * kPitch) * sizeof(double);
}

// ---------------------------------------------------------------- work items
// A sink's list is cut into chunks of 32 pairs (kM2LChunk).  A chunk of more than 24 pairs has a warp
// to itself; the last chunks of up to 8, 16 and 24 pairs are collected by size and share warps: 24 with
// 8, 16 with 16, the remaining 8s by four.  counts[0] = whole, [1..3] = rest of 8, 16, 24; [4] the item
// counter.  The order of the lists does not matter for the results.
struct Items {
    int2* whole;    // (sink, chunk)
    int2* rest[3];  // the same: chunks of up to 8, 16, 24 pairs
    unsigned* counts;
};

__global__ void k_m2l_f64_count(const int* __restrict__ seg_start, const int* __restrict__ seg_end, int ncells,
                                int* __restrict__ cnt) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ncells; i += gridDim.x * blockDim.x)
        cnt[i] = (seg_end[i] - seg_start[i] + kM2LChunk - 1) / kM2LChunk;
}

// slots for `mine` entries of each lane from *counter (one atomic per warp)
__device__ inline unsigned warp_slots(unsigned mine, unsigned* counter) {
    const int lane = threadIdx.x & 31;
    unsigned x = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    unsigned b = 0;
    if (lane == 31 && x) b = atomicAdd(counter, x);
    return __shfl_sync(0xffffffffu, b, 31) + x - mine;
}

__global__ void k_m2l_f64_items(const int* __restrict__ seg_start, const int* __restrict__ seg_end, int ncells,
                                Items it) {
    for (int i0 = blockIdx.x * blockDim.x; i0 < ncells; i0 += gridDim.x * blockDim.x) {
        const int i = i0 + threadIdx.x;
        const int len = i < ncells ? seg_end[i] - seg_start[i] : 0;
        const int full = len / kM2LChunk, r = len % kM2LChunk;
        const int cls = r == 0 ? 0 : (r + 7) / 8;  // 4: more than 24, a warp to itself
        const int nw = full + (cls == 4 ? 1 : 0);
        unsigned at = warp_slots((unsigned)nw, &it.counts[0]);
        for (int k = 0; k < nw; ++k) it.whole[at + k] = make_int2(i, k);
#pragma unroll
        for (int q = 1; q <= 3; ++q) {
            at = warp_slots(cls == q ? 1u : 0u, &it.counts[q]);
            if (cls == q) it.rest[q - 1][at] = make_int2(i, full);
        }
    }
}

// Mn = N_n^m M_n^m, so that the swaps are the symmetric matrices of the normalised harmonics
__global__ void k_m2l_f64_norm(const double* __restrict__ M, long long total, int nco, double* __restrict__ Mn) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x)
        Mn[t] = M[t] * __ldg(&g_tab.norm[(int)(t % nco)]);
}

// a sink of several chunks: F = its chunks' expansions, added in chunk order
__global__ void k_m2l_f64_reduce(const int* __restrict__ cnt, const int* __restrict__ cstart, int ncells, int nco,
                                 const double* __restrict__ part, double* __restrict__ F) {
    const long long total = (long long)ncells * nco;
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
         t += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(t / nco), j = (int)(t % nco), n = cnt[i];
        if (n < 2) continue;
        const double* q = part + (size_t)cstart[i] * nco + j;
        double v = 0.0;
        for (int k = 0; k < n; ++k) v += q[(size_t)k * nco];
        F[t] = v;
    }
}

// One warp per block and item, lane = pair.  The expansion of a sink's only chunk goes to F (zero
// beforehand), that of one of several chunks to part.
__global__ void __launch_bounds__(32) k_m2l_f64(const int2* __restrict__ list, const int* __restrict__ seg_start,
                                                const int* __restrict__ seg_end, const int* __restrict__ cnt,
                                                const int* __restrict__ cstart, Items it,
                                                const d4* __restrict__ cen, const double* __restrict__ Mn, int p,
                                                double* __restrict__ part, double* __restrict__ F) {
    extern __shared__ double dsm[];
    __shared__ int s_c[kOrd];    // centre rows of the rotated multipoles' orders
    __shared__ int s_base[4], s_len[4];
    __shared__ double* s_dst[4];
    const int lane = threadIdx.x, nco = ncoef(p), g = lane >> 3;
    double* S = dsm + lane;
    double* const w0 = dsm + rot_entries(p) * 32;
    double* const w1 = w0 + (2 * p + 1) * kPitch;
    const unsigned n0 = it.counts[0], n1 = it.counts[1], n2 = it.counts[2], n3 = it.counts[3];
    const unsigned i2 = (n2 + 1) / 2, i1 = n1 > n3 ? (n1 - n3 + 3) / 4 : 0;
    for (;;) {
        unsigned w = 0;
        if (lane == 0) w = atomicAdd(&it.counts[4], 1u);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w >= n0 + n3 + i2 + i1) break;
        // the chunk of each group of 8 lanes and the lane it starts at
        int2 e = make_int2(-1, 0);
        int base = 0;
        if (w < n0) {
            e = it.whole[w];
        } else if ((w -= n0) < n3) {
            if (g < 3) e = it.rest[2][w];
            else {
                base = 24;
                if (w < n1) e = it.rest[0][w];
            }
        } else if ((w -= n3) < i2) {
            base = 16 * (g >> 1);
            if (2 * w + (g >> 1) < n2) e = it.rest[1][2 * w + (g >> 1)];
        } else {
            w -= i2;
            base = 8 * g;
            if (n3 + 4 * w + g < n1) e = it.rest[0][n3 + 4 * w + g];
        }
        const int B = e.x;
        int s0 = 0, len = 0;
        if (B >= 0) {
            s0 = seg_start[B] + e.y * kM2LChunk;
            len = min(kM2LChunk, seg_end[B] - s0);
        }
        const bool act = lane - base < len;
        const unsigned heads = __ballot_sync(0xffffffffu, B >= 0 && lane == base);
        const int nch = __popc(heads);
        if ((heads >> lane) & 1) {
            const int k = __popc(heads & ((1u << lane) - 1u));
            s_base[k] = base;
            s_len[k] = len;
            s_dst[k] = cnt[B] == 1 ? F + (size_t)B * nco : part + (size_t)(cstart[B] + e.y) * nco;
        }
        // the lane's pair: phases e^{-i m alpha}, e^{-i m beta} and the powers of 1 / R
        const int xe = act ? list[s0 + lane - base].x : 0;
        const int A = m2l_src(xe), q = act ? m2l_order(xe, p) : 0;
        int P = q;
        for (int o = 16; o > 0; o >>= 1) P = max(P, __shfl_xor_sync(0xffffffffu, P, o));
        const bool mask = __any_sync(0xffffffffu, act && q < P);  // pairs of lower order (adaptive walk)
        double Rinv = 1.0, wr = 1.0, wi = 0.0, ur = 1.0, ui = 0.0;
        if (act) {
            const d4 zA = cen[A], sB = cen[B];
            const double x = sB.x - zA.x, y = sB.y - zA.y, z = sB.z - zA.z;
            const double t2 = x * x + y * y, r2 = t2 + z * z;
            Rinv = rsqrt(r2);
            double t = 0.0;
            if (t2 > 1e-280 * r2) {  // below, the direction is the z axis to far more than FP64's digits
                const double ti = rsqrt(t2);
                t = t2 * ti;
                wr = y * ti;
                wi = x * ti;
            }
            ur = z * Rinv;
            ui = -t * Rinv;
        }
        double cwr[kOrd], cwi[kOrd], cur[kOrd], cui[kOrd];
        cwr[0] = cur[0] = 1.0;
        cwi[0] = cui[0] = 0.0;
        for (int m = 1; m <= P; ++m) {
            cwr[m] = cwr[m - 1] * wr - cwi[m - 1] * wi;
            cwi[m] = cwr[m - 1] * wi + cwi[m - 1] * wr;
            cur[m] = cur[m - 1] * ur - cui[m - 1] * ui;
            cui[m] = cur[m - 1] * ui + cui[m - 1] * ur;
        }
        // multipoles into the rotated frame, order by order, times R^-k
        double tk = 1.0;
        int row = 0;
        for (int k = 0; k <= P; ++k) {
            const int L = min(k, P - k);
            double *c0 = w0 + k * kPitch + lane, *c1 = w1 + k * kPitch + lane;
            const double* src = Mn + (size_t)A * nco + k * k + k;
#pragma unroll 4
            for (int j = -k; j <= k; ++j) c0[j * kPitch] = act ? src[j] : 0.0;
            zrot(k, c0, kPitch, cwr, cwi, false);
            swap_xz(k, k, k, c0, kPitch, c1, kPitch, 1.0);
            zrot(k, c1, kPitch, cur, cui, false);
            swap_xz(k, L, k, c1, kPitch, S + (row + L) * 32, 32, tk);
            if (lane == 0) s_c[k] = row + L;
            row += 2 * L + 1;
            tk *= Rinv;
        }
        __syncwarp();
        // F in the rotated frame (eq. A31) and back: orders n and P - n together, so that their
        // 2 P + 2 rows fill the lanes that then add up the chunks
        auto back = [&](int n, double* x) {
            const int L = min(n, P - n);
            double tn = Rinv;
            for (int i = 0; i < n; ++i) tn *= Rinv;
            double *cx = x + n * kPitch + lane, *ca = w0 + n * kPitch + lane;
            for (int m = 0; m <= L; ++m) {
                const double* z = g_tab.z + (n * kZm + m) * kOrd;
                double re = 0.0, im = 0.0;
#pragma unroll 2
                for (int k = m; k <= P - n; ++k) {
                    const double* v = S + s_c[k] * 32;
                    double a = v[m * 32], b = v[-m * 32];
                    if (mask && n + k > q) a = b = 0.0;
                    const double zc = __ldg(z + k);
                    re = fma(zc, a, re);
                    if (m) im = fma(zc, b, im);
                }
                cx[m * kPitch] = re * tn;
                if (m) cx[-m * kPitch] = im * tn;
            }
            swap_xz(n, n, L, cx, kPitch, ca, kPitch, 1.0);
            zrot(n, ca, kPitch, cur, cui, true);
            swap_xz(n, n, n, ca, kPitch, cx, kPitch, 1.0);
            zrot(n, cx, kPitch, cwr, cwi, true);
        };
        for (int n = 0; 2 * n <= P; ++n) {
            const int o = P - n;
            back(n, w1);  // (its 2 n + 1 rows and those of o together are 2 P + 2)
            if (o > n) back(o, w1 + (2 * n + 1) * kPitch);
            __syncwarp();
            const int ra = 2 * n + 1, rows = o > n ? 2 * P + 2 : ra;
            for (int r = lane; r < rows; r += 32) {
                const double* x = w1 + r * kPitch;
                const int i = r < ra ? n * n + r : o * o + r - ra;
                const double nm = __ldg(&g_tab.norm[i]);
                for (int k = 0; k < nch; ++k) {
                    const double* xb = x + s_base[k];
                    double s = 0.0;
                    for (int b = 0; b < s_len[k]; ++b) s += xb[b];
                    s_dst[k][i] = s * nm;
                }
            }
            __syncwarp();
        }
        for (int k = 0; k < nch; ++k)
            for (int i = ncoef(P) + lane; i < nco; i += 32) s_dst[k][i] = 0.0;
        __syncwarp();
    }
}

struct F64Layout {
    int2* whole;
    int2* rest[3];
    int *cnt, *cstart, *stmp;
    unsigned* counts;
    double *Mn, *part;
    size_t bytes;
};
F64Layout f64_layout(void* tmp, int ncells, int p, long long npairs) {
    F64Layout L;
    const size_t nc = (size_t)(ncells > 0 ? ncells : 1), items = (size_t)(npairs / kM2LChunk) + nc + 1;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        off = (off + 255) & ~(size_t)255;
        unsigned char* r = tmp ? (unsigned char*)tmp + off : nullptr;
        off += bytes;
        return r;
    };
    L.whole = (int2*)take(items * sizeof(int2));
    for (int i = 0; i < 3; ++i) L.rest[i] = (int2*)take(nc * sizeof(int2));
    L.cnt = (int*)take(nc * sizeof(int));
    L.cstart = (int*)take(nc * sizeof(int));
    L.stmp = (int*)take(scan_tmp_ints((long long)nc) * sizeof(int));
    L.counts = (unsigned*)take(8 * sizeof(unsigned));
    L.Mn = (double*)take(nc * (size_t)ncoef(p) * sizeof(double));
    L.part = (double*)take(items * (size_t)ncoef(p) * sizeof(double));
    L.bytes = off + 256;
    return L;
}

}  // namespace

size_t m2l_f64_tmp_bytes(int ncells, int p, long long npairs) { return f64_layout(nullptr, ncells, p, npairs).bytes; }

void launch_m2l_f64(const int2* list, const int* seg_start, const int* seg_end, void* tmp, int ncells, const d4* cen,
                    const double* M, int p, double* F, long long npairs, cudaStream_t s) {
    if (ncells <= 0) return;
    init_tab();
    const F64Layout L = f64_layout(tmp, ncells, p, npairs);
    const Items it{L.whole, {L.rest[0], L.rest[1], L.rest[2]}, L.counts};
    const long long total = (long long)ncells * ncoef(p);
    cudaMemsetAsync(L.counts, 0, 8 * sizeof(unsigned), s);
    k_m2l_f64_norm<<<grid_for(total, 256), 256, 0, s>>>(M, total, ncoef(p), L.Mn);
    note_launch();
    k_m2l_f64_count<<<grid_for(ncells, 256), 256, 0, s>>>(seg_start, seg_end, ncells, L.cnt);
    note_launch();
    scan_exclusive_i32(L.cnt, L.cstart, ncells, nullptr, L.stmp, s);
    k_m2l_f64_items<<<grid_for(ncells, 256), 256, 0, s>>>(seg_start, seg_end, ncells, it);
    note_launch();
    const size_t sm = m2l_f64_smem(p);
    static DeviceOnce once;
    allow_smem(once, k_m2l_f64, m2l_f64_smem(kMaxP));
    int bps = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_m2l_f64, 32, sm);
    k_m2l_f64<<<sm_count() * (bps > 0 ? bps : 1), 32, sm, s>>>(list, seg_start, seg_end, L.cnt, L.cstart, it, cen, L.Mn,
                                                               p, L.part, F);
    note_launch();
    k_m2l_f64_reduce<<<grid_for(total, 256), 256, 0, s>>>(L.cnt, L.cstart, ncells, ncoef(p), L.part, F);
    note_launch();
}

}  // namespace gb3
