// p2p.cu -- the mixed-precision P2P of eq. (1): for every sink leaf B, Psi_b += mu_a / r and
// a_b += mu_a (x_a - x_b) / r^3 over the particles a of its source cells (its own P2P segment
// and those of its ancestors), a != b and r > 0 (coincident pairs skipped).
//
// Pair terms are FP32; each lane's FP32 sums over one tile (at most 128 pairs) are added to
// two-float accumulators (TwoSum), so the sum over a sink's thousands of sources is compensated.
// What a pair needs in FP32 is an accurate difference dx = x_a - x_b.  Two forms:
//   near: dx = (h_a - h_b) + (l_a - l_b) from the two-float positions (hi = fl32(x),
//         lo = fl32(x - hi)), one FP32 rounding relative to |dx| itself however close the pair;
//   far:  every source of a tile is turned once into its FP32 offset from the sink leaf's centre
//         c, o_a = (h_a - c_h) + (l_a - c_l), the sink likewise, and dx = o_a - o_b: one FP32
//         operation per coordinate and pair instead of three.  o_a and o_b carry absolute errors
//         of about 2^-24 |o|, so dx is relatively accurate to about 2^-24 (1 + 2 rho_B / |dx|).
// A source cell A is near when some pair of A x B could be closer than rho_B (the sink leaf's
// radius): |s_A - s_B| < rho_A + 2 rho_B.  Far pairs are then at least rho_B apart and their dx
// is good to about 3 x 2^-24, the same order as the rsqrt.approx of every pair.
//
// Work plan, built once per evaluation (k_p2p_count, k_p2p_emit): per leaf, its sources as
// particle ranges with their class (consecutive source cells of one class whose particles are
// contiguous are merged), in a region sized by its number of source cells, near ranges from the
// front and far ones from the back; and the work items (leaf, sink chunk).  Every lane holds two
// sinks, so that each source read from shared memory serves two pairs: a leaf of c sinks is cut
// into k items of at most 2 S sinks (slot s of an item holds its sinks s and S + s), each item
// replicated R <= 8 times across a warp (lane = replica * S + slot; replica r takes every R-th
// group of four sources of a tile), with (k, R) the cheapest by a cost per item of the lanes'
// pair work (2 / R per source) and the staging of its sources.  Every item streams its leaf's
// ranges as tiles of up to 128 sources: 32-byte position records copied asynchronously into a
// raw tile while the previous tile is computed, then converted into the structure-of-arrays
// tile the pairs read (offsets from the leaf centre for far tiles); a tile holds one class.
// Items run in decreasing order of their length (source particles / R) from an atomic counter.
#include <algorithm>
#include <climits>

#include "kernels.cuh"

namespace gb3 {

constexpr int kP2PWarpsM = 4;        // warps per block
constexpr int kP2PTileM = 128;       // sources per staged tile at the largest replica count (4 x 32)
constexpr int kRangeCountBits = 29;  // a range record holds count | near << 30 | guard << 29
constexpr int kRangeMax = (1 << kRangeCountBits) - 1;

typedef unsigned long long f2;  // two packed floats
__device__ __forceinline__ f2 f2_pack(float a, float b) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_unpack(f2 v, float& a, float& b) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f2 f2_sub(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// the sink of a lane, its coordinates duplicated in both halves
struct SinkPk {
    f2 hx, hy, hz, lx, ly, lz;
};
struct AccPk {
    f2 ps, ax, ay, az;
};

// two sources against the sink; TWO_FLOAT: dx from the two-float parts, else from X, Y, Z alone
// (FP32 offsets, or the high parts for the low-order estimate); GUARD: skip r = 0
template <bool TWO_FLOAT, bool GUARD>
__device__ __forceinline__ void pair2(f2 X, f2 Y, f2 Z, f2 W, f2 XL, f2 YL, f2 ZL, const SinkPk& b, AccPk& a) {
    f2 dx = f2_sub(X, b.hx), dy = f2_sub(Y, b.hy), dz = f2_sub(Z, b.hz);
    if (TWO_FLOAT) {
        dx = f2_add(dx, f2_sub(XL, b.lx));
        dy = f2_add(dy, f2_sub(YL, b.ly));
        dz = f2_add(dz, f2_sub(ZL, b.lz));
    }
    const f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_mul(dz, dz)));
    float r2a, r2b;
    f2_unpack(r2, r2a, r2b);
    float ia = rsqrt_ftz(r2a), ib = rsqrt_ftz(r2b);
    if (GUARD) {
        ia = r2a > 0.f ? ia : 0.f;
        ib = r2b > 0.f ? ib : 0.f;
    }
    const f2 rinv = f2_pack(ia, ib);
    const f2 qm = f2_mul(W, rinv);
    const f2 q3 = f2_mul(qm, f2_mul(rinv, rinv));
    a.ps = f2_add(a.ps, qm);
    a.ax = f2_fma(q3, dx, a.ax);
    a.ay = f2_fma(q3, dy, a.ay);
    a.az = f2_fma(q3, dz, a.az);
}

// one group of four sources of the tile (index g) against the lane's two sinks
template <bool TWO_FLOAT, bool GUARD>
__device__ __forceinline__ void group4(const float* __restrict__ T, int g, const SinkPk& b0, const SinkPk& b1,
                                       AccPk& a0, AccPk& a1) {
    // 16-byte loads straight into packed pairs (sources 0, 1 and 2, 3 of the group)
    const ulonglong2 X = ((const ulonglong2*)(T + 0 * kP2PTileM))[g], Y = ((const ulonglong2*)(T + 1 * kP2PTileM))[g],
                     Z = ((const ulonglong2*)(T + 2 * kP2PTileM))[g], W = ((const ulonglong2*)(T + 3 * kP2PTileM))[g];
    ulonglong2 XL = make_ulonglong2(0ull, 0ull), YL = XL, ZL = XL;
    if (TWO_FLOAT) {
        XL = ((const ulonglong2*)(T + 4 * kP2PTileM))[g];
        YL = ((const ulonglong2*)(T + 5 * kP2PTileM))[g];
        ZL = ((const ulonglong2*)(T + 6 * kP2PTileM))[g];
    }
    const f2 x01 = X.x, y01 = Y.x, z01 = Z.x, w01 = W.x, x23 = X.y, y23 = Y.y, z23 = Z.y, w23 = W.y;
    const f2 l01 = XL.x, m01 = YL.x, n01 = ZL.x, l23 = XL.y, m23 = YL.y, n23 = ZL.y;
    pair2<TWO_FLOAT, GUARD>(x01, y01, z01, w01, l01, m01, n01, b0, a0);
    pair2<TWO_FLOAT, GUARD>(x01, y01, z01, w01, l01, m01, n01, b1, a1);
    pair2<TWO_FLOAT, GUARD>(x23, y23, z23, w23, l23, m23, n23, b0, a0);
    pair2<TWO_FLOAT, GUARD>(x23, y23, z23, w23, l23, m23, n23, b1, a1);
}

constexpr int kP2PRmax = 8;  // replicas of an item across a warp
// groups of four per replica in a full tile, and sources per full tile: 4 R (32 / R) <= 128
__host__ __device__ constexpr int p2p_groups(int R) { return 32 / R; }
__host__ __device__ constexpr int p2p_tile(int R) { return 4 * R * (32 / R); }

// replica r0 of R takes groups r0, r0 + R, ... of a tile of ng groups (one loop for every R,
// so that the four forms of the pair code stay small enough for the instruction cache)
template <bool TWO_FLOAT, bool GUARD>
__device__ __forceinline__ void tile_any(const float* __restrict__ T, int ng, int r0, int R, const SinkPk& b0,
                                         const SinkPk& b1, AccPk& a0, AccPk& a1) {
#pragma unroll 2
    for (int g = r0; g < ng; g += R) group4<TWO_FLOAT, GUARD>(T, g, b0, b1, a0, a1);
}

// s.hi += v with the rounding error of that addition (TwoSum) kept in s.lo; s.lo is not
// renormalised against s.hi (its own rounding, u |s.lo|, stays far below u |s.hi|)
__device__ __forceinline__ void acc2(ff& s, float v) {
    const ff t = two_sum(s.hi, v);
    s.hi = t.hi;
    s.lo = __fadd_rn(s.lo, t.lo);
}

// the FP32 partials of one sink folded into its two-float sums (4 per sink)
__device__ __forceinline__ void fold(AccPk& a, ff* sum) {
    float u0, u1;
    f2_unpack(a.ps, u0, u1);
    acc2(sum[0], u0 + u1);
    f2_unpack(a.ax, u0, u1);
    acc2(sum[1], u0 + u1);
    f2_unpack(a.ay, u0, u1);
    acc2(sum[2], u0 + u1);
    f2_unpack(a.az, u0, u1);
    acc2(sum[3], u0 + u1);
    const f2 zero = f2_pack(0.f, 0.f);
    a = AccPk{zero, zero, zero, zero};
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
    const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait0() { asm volatile("cp.async.wait_group 0;\n" ::: "memory"); }

// How a leaf of c sinks is cut into work items: k items of at most Q S sinks, each replicated R
// times across a warp (lane = replica * S + slot; slot s of an item holds its sinks s, S + s, ...,
// (Q - 1) S + s).  A source costs an item Q / R steps of the warp.
struct Chunk {
    int k, R, S, Q;
};
// The mixed P2P: two sinks per slot; the least cost k (2 / R + 0.6) per source over
// k >= ceil(c / 64) (the lanes' pair work and the staging of the sources, in units of a lane's
// pair), then k = ceil(c / (2 S)) so that no item is empty.  Items longer than piece_steps steps
// are split (see below).
struct PlanMixed {
    static constexpr bool budget = false;
    static constexpr unsigned piece_steps = 8192, sub_steps = 1024;
    static constexpr int sub_n = 16384;  // particles of the largest system whose pieces are shared
    static constexpr int max_pieces = 64;
    static constexpr bool merge = true;
    static constexpr int nv = 4;  // sums per sink
    __device__ static inline Chunk chunk(int c) {
        Chunk r{1, 1, 1, 2};
        if (c <= 0) return r;
        const int kmin = (c + 63) / 64;
        float best = 3.0e38f;
        for (int kk = kmin; kk < kmin + 12; ++kk) {
            const int SS = (c + 2 * kk - 1) / (2 * kk);
            const int RR = 32 / SS < kP2PRmax ? 32 / SS : kP2PRmax;
            const float cost = (float)kk * (2.0f / (float)RR + 0.6f);
            if (cost < best) {
                best = cost;
                r.k = kk;
                r.R = RR;
                r.S = SS;
            }
        }
        r.k = (c + 2 * r.S - 1) / (2 * r.S);
        return r;
    }
};
// The FP64 P2P is bound by the FP64 pipe alone (an instruction costs the same however many lanes
// are active, staging runs beside it): the fewest steps k Q / R per source over S <= 32 slots and
// Q <= 4 sinks per slot.  Short pieces (a step of 18 FP64 instructions holds a quarter of an SM for
// 1152 cycles, so 256 steps are 0.14 ms) keep every SM busy to the end; where there are many, longer
// ones do too (k_p2p_pieces).
struct PlanF64 {
    static constexpr bool budget = true;
    static constexpr unsigned piece_steps = 256, sub_steps = 0;
    static constexpr int sub_n = 0;
    static constexpr int max_pieces = 1024;
    static constexpr bool merge = true;
    static constexpr int nv = 4;
    // (all lanes of a warp together: lane S - 1 looks at S slots; the least cost, of equal ones the most
    // slots.  One lane through all 128 pairs took 20 us a call)
    __device__ static inline Chunk chunk(int c) {
        const int S = (int)(threadIdx.x & 31) + 1, R = min(32 / S, 16);
        float best = 3.0e38f;
        int bq = 1;
        if (S <= c)
            for (int Q = 1; Q <= 4; ++Q) {
                const int k = (c + Q * S - 1) / (Q * S);
                const float cost = (float)(k * Q) / (float)R + 0.02f * (float)k;
                if (cost < best) {
                    best = cost;
                    bq = Q;
                }
            }
        const int least = __reduce_min_sync(0xffffffffu, __float_as_int(best));  // positive: ordered as integers
        const int l = 31 - __clz(__ballot_sync(0xffffffffu, __float_as_int(best) == least));
        if (c <= 0) return Chunk{1, 1, 1, 1};
        Chunk r;
        r.S = l + 1;
        r.Q = __shfl_sync(0xffffffffu, bq, l);
        r.R = min(32 / r.S, 16);
        r.k = (c + r.Q * r.S - 1) / (r.Q * r.S);
        return r;
    }
};

// The mixed tidal P2P: a slot holds two sinks as the halves of packed operations, and the R groups of
// S lanes take shares of the source cells of their own: the fewest items k / R per source.
struct PlanTidal {
    static constexpr bool budget = true;
    static constexpr unsigned piece_steps = 1024, sub_steps = 0;
    static constexpr int sub_n = 0;
    static constexpr int max_pieces = 256;
    static constexpr bool merge = false;
    static constexpr int nv = 6;
    __device__ static inline Chunk chunk(int c) {
        Chunk r{1, 1, 1, 2};
        if (c <= 0) return r;
        const int slots = (c + 1) / 2, kmin = (slots + 31) / 32;
        float best = 3.0e38f;
        for (int k = kmin; k < kmin + 6; ++k) {
            const int S = (slots + k - 1) / k, R = min(32 / S, 4);
            const float cost = (float)k / (float)R * (1.0f + 0.05f * (float)R);
            if (cost < best) {
                best = cost;
                r = Chunk{(slots + S - 1) / S, R, S, 2};
            }
        }
        return r;
    }
};

// class of source cell A for sink leaf B (see the file comment); mode 1 only
__device__ inline bool p2p_near(const d4& a, const d4& b) {
    const double dx = a.x - b.x, dy = a.y - b.y, dz = a.z - b.z;
    const double lim = a.w + 2.0 * b.w;
    return dx * dx + dy * dy + dz * dz < lim * lim;
}

// Long items are split: a leaf whose item would take a lane more than piece_steps steps
// (Q sources / R) has its stream of source cells cut into P = ceil(steps / piece_steps) <=
// max_pieces pieces of about equal numbers of source cells, each with its own ranges, items
// and FP64 partial sums, which k_p2p_reduce adds in piece order.  The split depends on the leaf
// and its own system alone, so a system gives the same result in an ensemble as alone.
// PL::budget: the pieces are short where that fills the device, and longer where their partial sums
// would exceed the system's share of the workspace (k_p2p_pieces).
// A piece of the mixed P2P of a small system is shared by U = its steps / sub_steps warps: its stream of
// sources is cut at tile boundaries into U parts with ranges, items and partial sums of their own, so
// the tiles and their FP32 sums are those of the whole piece.  With few leaves the longest item sets
// the kernel's time: 1e4 particles (892 leaves) 0.37 ms with whole pieces, 0.18 ms with parts of 1024
// steps; with enough leaves the parts only cost (their starts and sums; 1e5: 1.71 and 1.89 ms, 1e6: 4.74
// and 5.03 ms), so systems of more than sub_n particles have none (counted is the leaf's own system: the
// same alone and in an ensemble).

// per leaf index t (one warp each): the number of its source cells nb[t] (the ranges it can need
// at most: its own and its ancestors' segment lengths), its pieces P and their parts U as np[t] =
// P | U << 16, its items per piece kc[t] and its sort key,
// descending in the length of a piece's items (a lane's steps, Q source particles / R; 0 for a leaf
// without active particles); tot[0] += nb.  work != nullptr: np[t] is the length of the leaf's items,
// root[t] its system's root and work[root] the sum of length x sinks over the system; k_p2p_pieces follows
template <class PL>
__global__ void k_p2p_count(Cells c, const int2* __restrict__ list, const int* __restrict__ seg_start,
                            const int* __restrict__ seg_end, const int* __restrict__ leaves, int nleaves, int sub_n,
                            int n, const int* __restrict__ off, int nsys, int* __restrict__ nb, int* __restrict__ np,
                            int* __restrict__ kc, uint64_t* __restrict__ keys, int* __restrict__ root,
                            unsigned long long* __restrict__ work, unsigned long long* __restrict__ tot) {
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    unsigned long long my = 0;
    for (int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < nleaves; t += nw) {
        const int leaf = leaves[t];
        long long e = 0, src = 0;
        int top = leaf;
        for (int cell = leaf; cell >= 0; cell = c.parent[cell]) {
            top = cell;
            const int s0 = seg_start[cell], s1 = seg_end[cell];
            e += s1 - s0;
            for (int i = s0 + lane; i < s1; i += 32) src += c.count[list[i].x];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) src += __shfl_xor_sync(0xffffffffu, src, o);
        const Chunk ch = PL::chunk(c.count[leaf]);  // (by the whole warp)
        if (lane == 0) {
            nb[t] = (int)e;
            my += (unsigned long long)e;
            kc[t] = ch.k;
            const unsigned long long l = (unsigned long long)ch.Q * (unsigned long long)src / (unsigned long long)ch.R + 1;
            const unsigned len = !cell_active(c, leaf) ? 0u : (l > 0xfffffffeull ? 0xfffffffeu : (unsigned)l);
            if (PL::budget && work) {
                np[t] = (int)len;
                root[t] = top;
                atomicAdd(&work[top], (unsigned long long)len * (unsigned)c.count[leaf]);
                continue;
            }
            int P = (int)(((unsigned long long)len + PL::piece_steps - 1) / PL::piece_steps);
            const int cap = e < PL::max_pieces ? (int)e : PL::max_pieces;
            P = P < 1 ? 1 : (P > cap ? (cap > 0 ? cap : 1) : P);
            const unsigned w32 = len ? (unsigned)(((unsigned long long)len + P - 1) / P) : 0u;
            unsigned U = 1;
            if constexpr (PL::sub_steps > 0) {
                int size = n;
                if (off) {
                    const int k = system_of(off, nsys, c.first[leaf]);
                    size = off[k + 1] - off[k];
                }
                if (size <= sub_n) U = min(max(min(w32 / PL::sub_steps, (unsigned)(e / P)), 1u), 255u);
            }
            np[t] = P | (int)(U << 16);
            keys[t] = ((uint64_t)(255u - qlen8((w32 + U - 1) / U)) << 32) | (unsigned)t;
        }
    }
    if (lane == 0 && my) atomicAdd(&tot[0], my);
}

// The pieces of PL::budget's leaves.  A piece costs nv partial sums per sink, so pieces of L steps of a system
// with the work A = sum of length x sinks take 8 nv A / L bytes: L is the shortest for which that is at most
// nv / 4 (base + per x the system's particles), and at least piece_steps.  (Of 256 steps in any system the FP64 plan's
// partial sums took up to 10 KB per particle, of 1024 steps the tidal plan's up to 9 KB: 13 times the bound of the
// whole workspace for leaves of 1024.)  A call takes 6 us longer, so it is left out where no system can
// need it (an item has at most 4 steps per particle; 4096 particles).
template <class PL>
__global__ void k_p2p_pieces(Cells c, int nleaves, const int* __restrict__ nb, const int* __restrict__ root,
                             const unsigned long long* __restrict__ work, PlanBudget bg, int* __restrict__ np,
                             uint64_t* __restrict__ keys) {
    for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nleaves; t += gridDim.x * blockDim.x) {
        const int r = root[t], e = nb[t];
        const double L = ceil(32.0 * (double)work[r] / (bg.base + bg.per * (double)c.count[r]));
        const unsigned len = (unsigned)np[t];
        unsigned P;
        if (L <= (double)PL::piece_steps) P = (unsigned)(((unsigned long long)len + PL::piece_steps - 1) / PL::piece_steps);
        else P = (unsigned)((double)len / L);  // (rounded down: the sum stays within the share)
        P = max(1u, min(P, (unsigned)max(1, min(e, PL::max_pieces))));
        np[t] = (int)(P | 1u << 16);
        keys[t] = ((uint64_t)(255u - qlen8((unsigned)(((unsigned long long)len + P - 1) / P))) << 32) | (unsigned)t;
    }
}

// the warp's sum of v, and *before = the sum over the lanes below
__device__ inline unsigned long long warp_total(unsigned long long v, unsigned long long* before) {
    const int lane = threadIdx.x & 31;
    unsigned long long x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    *before = x - v;
    return __shfl_sync(0xffffffffu, x, 31);
}

// per position q of the sorted order: its leaf index order[q], pieces npc[q] (their parts counted) and
// items nit[q] (pieces x items per piece; 0 for a leaf without active particles); a split leaf (more than one
// piece) takes the first of its partial-sum slots pbase[q] (pieces x sinks of them; -1: not split)
// and an entry (leaf index, first slot) of the split list; a leaf with parts also the first of its nb + 2
// npc places for their records, cbase[q].  tot[1] items, tot[2] those places, tot[3] pieces, tot[4]
// slots, tot[5] split leaves; one atomic per warp and counter (a thread each took 60 us for 43,000
// leaves).
__global__ void k_p2p_nitems(const uint64_t* __restrict__ keys, const int* __restrict__ leaves, int nleaves, Cells c,
                             const int* __restrict__ np, const int* __restrict__ nb, const int* __restrict__ kc,
                             int* __restrict__ order, int* __restrict__ nit, int* __restrict__ npc, int* __restrict__ pbase,
                             int* __restrict__ cbase, int2* __restrict__ split, unsigned long long* __restrict__ tot) {
    const int lane = threadIdx.x & 31;
    for (int q0 = blockIdx.x * blockDim.x; q0 < nleaves; q0 += gridDim.x * blockDim.x) {
        const int q = q0 + threadIdx.x;
        int t = 0, k = 0, P = 0, count = 0, places = 0;
        if (q < nleaves) {
            t = (int)(keys[q] & 0xffffffffu);
            order[q] = t;
            const int leaf = leaves[t];
            count = c.count[leaf];
            if (cell_active(c, leaf)) {
                k = kc[t];
                P = (np[t] & 0xffff) * (np[t] >> 16);
                if ((np[t] >> 16) > 1) places = nb[t] + 2 * P;
            }
            nit[q] = k * P;
            npc[q] = P;
        }
        const bool sp = P > 1;
        const unsigned long long slots = sp ? (unsigned long long)P * (unsigned long long)count : 0ull;
        unsigned long long ex, sbefore, lbefore, cbefore = 0, tc = 0, cb = 0;
        if (__any_sync(0xffffffffu, places)) tc = warp_total((unsigned long long)places, &cbefore);
        const unsigned long long ti = warp_total((unsigned long long)k * P, &ex), tp = warp_total(P, &ex);
        const unsigned long long ts = warp_total(slots, &sbefore), tl = warp_total(sp ? 1 : 0, &lbefore);
        unsigned long long sb = 0, lb = 0;
        if (lane == 0) {
            if (ti) atomicAdd(&tot[1], ti);
            if (tp) atomicAdd(&tot[3], tp);
            if (tc) cb = atomicAdd(&tot[2], tc);
            if (tl) {
                sb = atomicAdd(&tot[4], ts);
                lb = atomicAdd(&tot[5], tl);
            }
        }
        sb = __shfl_sync(0xffffffffu, sb, 0) + sbefore;
        lb = __shfl_sync(0xffffffffu, lb, 0) + lbefore;
        cb = __shfl_sync(0xffffffffu, cb, 0) + cbefore;
        if (q < nleaves) {
            if (places) cbase[q] = (int)cb;
            pbase[q] = sp ? (int)sb : -1;
            if (sp) split[lb] = make_int2(t, (int)sb);
        }
    }
}

// per piece v: its leaf index, its region of ranges [r0, r1) (near ranges from the front, far
// ones from the back), their numbers, and the first of its partial sums (-1: the piece is the
// whole leaf and writes psi and acc directly)
struct Pieces {
    int *leaf, *r0, *r1, *nnear, *nfar, *part;
};

// ranges and items of piece v, one warp per piece (the pieces of a long leaf side by side: with one
// warp per leaf the longest leaf set the kernel's time); with parts, one warp per piece and its parts
// (v the first of them).  Piece j of a leaf (sorted position q, the last with voff[q] <= v; j = (v -
// voff[q]) / U) takes the source cells j e / P .. (j + 1) e / P - 1 of
// the leaf's stream (its own segment, then each ancestor's; e cells in all) and owns that part of
// the leaf's region [roff[t], roff[t] + e).  Within a piece the sources are merged per class in
// stream order: an
// entry joins the open range of its class when its particles follow that range's directly.  The
// lanes take up to 32 entries at a time; each finds its class predecessor (the closest lower
// lane of its class, else the open range carried from the earlier entries), the entries that do
// not join start a run, a run's count and guard flag are summed in shared memory, and every run
// but the last of its class is written out; the last stays open until the piece ends.  This is
// the result of the sequential pass.
// Without PL::merge: one far record per source cell, in stream order from the front (the tidal P2P).
constexpr int kEmitWarps = 4;
template <class PL>
__global__ void __launch_bounds__(kEmitWarps * 32)
    k_p2p_emit(Cells c, const int2* __restrict__ list, const int* __restrict__ seg_start,
               const int* __restrict__ seg_end, const int* __restrict__ leaves, int nleaves, int mode,
               const int* __restrict__ order, const int* __restrict__ roff, const int* __restrict__ nb,
               const int* __restrict__ ioff, const int* __restrict__ nit, const int* __restrict__ voff,
               const int* __restrict__ npc, const int* __restrict__ np, const int* __restrict__ pbase,
               const int* __restrict__ cbase, int npieces, Pieces pc, int2* __restrict__ ranges, int2* __restrict__ cuts, int2* __restrict__ items) {
    constexpr bool MERGE = PL::merge;
    __shared__ int rsum_all[kEmitWarps][33], rg_all[kEmitWarps][33];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int* rsum = rsum_all[wid];  // [0]: the open range carried in; [1 + L]: the run starting at lane L
    int* rg = rg_all[wid];
    const unsigned below = (1u << lane) - 1u, upto = below | (1u << lane);
    const int nw = (gridDim.x * blockDim.x) >> 5;
    for (int v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < npieces; v += nw) {
        int q = 0;
        for (int hi = nleaves - 1; q < hi;) {
            const int mid = (q + hi + 1) >> 1;
            if (voff[mid] <= v) q = mid;
            else hi = mid - 1;
        }
        const int t = order[q], P = np[t] & 0xffff, U = np[t] >> 16;
        if ((v - voff[q]) % U) continue;  // a later part of a piece: its first part's warp makes it
        const int pj = (v - voff[q]) / U;
        const int kper = nit[q] / (P * U);  // items per piece or part
        const int leaf = leaves[t];
        const int count = c.count[leaf];
        for (int j = lane; j < kper * U; j += 32)
            items[ioff[q] + pj * kper * U + j] = make_int2(v + j / kper, j % kper);
        const d4 sb = c.sr[leaf];
        const long long b0 = c.first[leaf], b1 = b0 + count;
        const long long e = nb[t];
        const long long f0 = e * pj / P, f1 = e * (pj + 1) / P;
        const int r0 = roff[t] + (int)f0, r1 = roff[t] + (int)f1;
        // the cursor over the leaf's stream of source cells: cell, its list segment, position
        int cell = leaf, s1 = seg_end[leaf], at = seg_start[leaf];
        for (long long skip = f0; skip > 0;) {
            const long long len = s1 - at;
            if (len > skip) {
                at += (int)skip;
                break;
            }
            skip -= len;
            at = s1;
            if (skip > 0) {
                cell = c.parent[cell];
                at = seg_start[cell];
                s1 = seg_end[cell];
            }
        }
        int cf[2] = {0, 0}, cn[2] = {0, 0}, cnt[2] = {0, 0};  // open range and records written per class
        bool cg[2] = {false, false};
        auto put = [&](int k, int idx, int f, int n, bool g) {
            ranges[k ? r0 + idx : r1 - 1 - idx] = make_int2(f, n | (k << 30) | ((g ? 1 : 0) << kRangeCountBits));
        };
        for (long long fi = f0; fi < f1;) {
            while (at >= s1) {  // on to the next ancestor's segment
                cell = c.parent[cell];
                at = seg_start[cell];
                s1 = seg_end[cell];
            }
            const int m = (int)min((long long)min(32, s1 - at), f1 - fi);
            int f = 0, n = 0, kk = -1;
            if (lane < m) {
                const int A = list[at + lane].x;
                f = c.first[A];
                n = c.count[A];
                if (MERGE) kk = mode == 1 ? (p2p_near(c.sr[A], sb) ? 1 : 0) : (mode == 3 ? 1 : 0);
                else ranges[r0 + (int)(fi - f0) + lane] = make_int2(f, n);
                if (n <= 0) kk = -1;
            }
            at += m;
            fi += m;
            if (!MERGE) continue;
            const bool g = kk >= 0 && f < b1 && b0 < (long long)f + n;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const unsigned M = __ballot_sync(0xffffffffu, kk == k);
                if (!M) continue;
                const unsigned pm = M & below;
                const int pl = pm ? 31 - __clz(pm) : lane;
                const int pf = __shfl_sync(0xffffffffu, f, pl), pn = __shfl_sync(0xffffffffu, n, pl);
                const long long pe = pm ? (long long)pf + pn : (cn[k] > 0 ? (long long)cf[k] + cn[k] : -1);
                const bool mine = kk == k;
                const unsigned S = __ballot_sync(0xffffffffu, mine && pe != f);
                const unsigned sm = S & upto;
                const int rs = sm ? 31 - __clz(sm) : -1;  // the run this lane belongs to
                rsum[lane] = 0;
                rg[lane] = 0;
                if (lane == 0) rsum[32] = rg[32] = 0;
                __syncwarp();
                if (mine) {
                    atomicAdd(&rsum[rs + 1], n);
                    if (g) atomicOr(&rg[rs + 1], 1);
                }
                __syncwarp();
                if (!S) {  // every entry joins the open range
                    cn[k] += rsum[0];
                    cg[k] = cg[k] || rg[0];
                } else {
                    int base = cnt[k];
                    if (cn[k] > 0) {  // the open range closes at the first start
                        if (lane == 0) put(k, base, cf[k], cn[k] + rsum[0], cg[k] || rg[0]);
                        ++base;
                    }
                    const int last = 31 - __clz(S);
                    if (((S >> lane) & 1) && lane != last)
                        put(k, base + __popc(S & below), f, rsum[lane + 1], rg[lane + 1] != 0);
                    cnt[k] = base + __popc(S) - 1;
                    cf[k] = __shfl_sync(0xffffffffu, f, last);
                    cn[k] = rsum[last + 1];
                    cg[k] = rg[last + 1] != 0;
                }
                __syncwarp();
            }
        }
        if (lane == 0) {
            for (int k = 1; k >= 0; --k)
                if (cn[k] > 0) put(k, cnt[k]++, cf[k], cn[k], cg[k]);
            pc.leaf[v] = t;
            pc.r0[v] = r0;
            pc.r1[v] = r1;
            pc.nnear[v] = cnt[1];
            pc.nfar[v] = cnt[0];
            pc.part[v] = P * U > 1 ? pbase[q] + pj * U * count : -1;
        }
        __syncwarp();
        if (U == 1) continue;
        // The parts: the piece's tiles are cut (tiles of T sources of the near records, then of the far
        // ones); part u has the tiles u K .. (u + 1) K - 1, the last part the rest.  The records of a
        // class that overlap its interval of sources are copied, clipped, behind those of the part
        // before it (a record cut in two is in both, hence one place more per part and class).
        const int nr[2] = {__shfl_sync(0xffffffffu, cnt[1], 0), __shfl_sync(0xffffffffu, cnt[0], 0)};  // near, far
        const int rb[2] = {r0, r1 - nr[1]};
        int2* cut = cuts + (size_t)cbase[q] + (size_t)f0 + 2 * (size_t)pj * U;
        const int T = p2p_tile(PL::chunk(count).R), K = max(1, (int)PL::sub_steps * PL::chunk(count).R / (2 * T));
        long long total[2] = {0, 0};
        for (int k = 0; k < 2; ++k) {
            for (int i = lane; i < nr[k]; i += 32) total[k] += ranges[rb[k] + i].y & kRangeMax;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) total[k] += __shfl_xor_sync(0xffffffffu, total[k], o);
        }
        const long long ntl = (total[0] + T - 1) / T;  // near tiles
        for (int u = 0; u < U; ++u) {
            const long long t0 = (long long)u * K, t1 = u + 1 < U ? t0 + K : LLONG_MAX / T;
            int at2[2], num[2];
            for (int k = 0; k < 2; ++k) {
                // the part's interval [a, b) of the class's sources
                const long long s0 = k ? max(t0 - ntl, 0ll) : min(t0, ntl), s1 = k ? max(t1 - ntl, 0ll) : min(t1, ntl);
                const long long a = min(s0 * T, total[k]), b = s1 > total[k] / T ? total[k] : s1 * T;
                int2* dst = cut + (k ? nr[0] + U : 0);
                long long before = 0;
                int n = 0, firstrec = -1;
                for (int i0 = 0; i0 < nr[k] && a < b; i0 += 32) {
                    const int i = i0 + lane;
                    const int2 rec = i < nr[k] ? ranges[rb[k] + i] : make_int2(0, 0);
                    const int m = rec.y & kRangeMax;
                    int x = m;
#pragma unroll
                    for (int o = 1; o < 32; o <<= 1) {
                        const int y = __shfl_up_sync(0xffffffffu, x, o);
                        if (lane >= o) x += y;
                    }
                    const long long p0 = before + x - m;  // sources before this record
                    const long long lo = max(p0, a), hi = min(p0 + m, b);
                    const unsigned on = __ballot_sync(0xffffffffu, lo < hi);
                    if (on && firstrec < 0) firstrec = i0 + __ffs(on) - 1;
                    if (lo < hi)
                        dst[firstrec + u + n + __popc(on & below)] =
                            make_int2(rec.x + (int)(lo - p0), (int)(hi - lo) | (rec.y & ~kRangeMax));
                    n += __popc(on);
                    before += __shfl_sync(0xffffffffu, x, 31);
                    if (before >= b) break;
                }
                at2[k] = (int)(dst - ranges) + (firstrec < 0 ? 0 : firstrec + u);
                num[k] = n;
            }
            if (lane == 0) {
                pc.leaf[v + u] = t;
                pc.r0[v + u] = at2[0];
                pc.nnear[v + u] = num[0];
                pc.r1[v + u] = at2[1] + num[1];
                pc.nfar[v + u] = num[1];
                pc.part[v + u] = pbase[q] + (pj * U + u) * count;
            }
        }
        __syncwarp();
    }
}

// the FP64 partial sums of the split leaves added in piece order into psi and acc (NV = 4) or into
// the NV values per sink of acc: one warp per entry (t, first slot) of the split list, lanes over
// the leaf's sinks
template <int NV>
__global__ void k_p2p_reduce(Cells c, const int* __restrict__ leaves, const int* __restrict__ np,
                             const int2* __restrict__ split, int nsplit, const double* __restrict__ part,
                             double* __restrict__ psi, double* __restrict__ acc) {
    const int lane = threadIdx.x & 31;
    const int nw = (gridDim.x * blockDim.x) >> 5;
    for (int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < nsplit; w += nw) {
        const int2 sp = split[w];
        const int leaf = leaves[sp.x], P = (np[sp.x] & 0xffff) * (np[sp.x] >> 16);
        const int first = c.first[leaf], count = c.count[leaf];
        for (int sk = lane; sk < count; sk += 32) {
            double v[NV];
#pragma unroll
            for (int d = 0; d < NV; ++d) v[d] = 0.0;
            for (int j = 0; j < P; ++j) {
                const double* pp = part + NV * ((size_t)sp.y + (size_t)j * count + sk);
#pragma unroll
                for (int d = 0; d < NV; ++d) v[d] += pp[d];
            }
            const size_t i = (size_t)first + sk;
            if (NV == 4) {
                psi[i] = v[0];
                acc[3 * i] = v[1];
                acc[3 * i + 1] = v[2];
                acc[3 * i + 2] = v[3];
            } else {
#pragma unroll
                for (int d = 0; d < NV; ++d) acc[NV * i + d] = v[d];
            }
        }
    }
}

// The ranges of one item as a stream of tiles.  The item's records (its near segment, then
// its far segment) are read 32 at a time into a register window, lane j holding record
// w0 + j, and the next window is loaded as soon as the current one is taken.  A tile takes
// sources from consecutive ranges of one class; fill() copies their position records (two
// float4 each, one with LOADLO false) into the raw tile and returns their number (0 when the
// stream is exhausted) with the tile's class and guard flag.
struct RangeStream {
    int a0, na, b0, total;  // flattened record i: i < na ? a0 + i : b0 + i - na; total records
    int pos, w0;            // next record, first record of the window
    int2 win, nwin;         // the window and the one after it
    int af, an, off;        // the current range and the position in it
    bool near, guard;       // its class and guard flag
    __device__ int2 load(const int2* __restrict__ ranges, int w, int lane) const {
        const int i = w + lane;
        return i < total ? ranges[i < na ? a0 + i : b0 + (i - na)] : make_int2(0, 0);
    }
    __device__ void start(const int2* __restrict__ ranges, int lane, int r0, int r1, int s0, int s1) {
        a0 = r0;
        na = r1 - r0;
        b0 = s0;
        total = na + (s1 - s0);
        pos = w0 = 0;
        win = load(ranges, 0, lane);
        nwin = load(ranges, 32, lane);
        af = an = off = 0;
        near = guard = false;
    }
    template <bool LOADLO>
    __device__ int fill(const int2* __restrict__ ranges, const float4* __restrict__ xp, int lane, int T,
                        float4* raw, bool& tile_near, bool& tile_guard) {
        int m = 0;
        tile_guard = false;
        tile_near = near;
        while (m < T) {
            if (off == an) {  // next range
                if (pos >= total) break;
                if (pos - w0 >= 32) {  // on to the prefetched window
                    win = nwin;
                    w0 += 32;
                    nwin = load(ranges, w0 + 32, lane);
                }
                const int rx = __shfl_sync(0xffffffffu, win.x, pos - w0);
                const int ry = __shfl_sync(0xffffffffu, win.y, pos - w0);
                const bool nr = (ry >> 30) & 1;
                if (m > 0 && nr != tile_near) break;  // a tile holds one class
                ++pos;
                af = rx;
                an = ry & kRangeMax;
                off = 0;
                near = nr;
                guard = (ry >> kRangeCountBits) & 1;
                tile_near = nr;
                continue;
            }
            const int k = min(T - m, an - off);
            for (int q = lane; q < k; q += 32) {
                const float4* g = xp + 2 * ((size_t)af + off + q);
                float4* t = raw + 2 * (m + q);
                cp_async16(t, g);
                if (LOADLO) cp_async16(t + 1, g + 1);
            }
            tile_guard = tile_guard || guard;
            m += k;
            off += k;
        }
        return m;
    }
};

// MODE 0: dx from the FP32 high parts (the low-order estimate); 1: near ranges two-float,
// far ranges FP32 offsets from the leaf centre; 2: offsets for every range; 3: two-float for
// every range
template <int MODE>
__global__ void __launch_bounds__(kP2PWarpsM * 32, 4)
    k_p2p_mixed(const float4* __restrict__ xp, Cells c, const int* __restrict__ leaves,
                const int2* __restrict__ ranges, const Pieces pc, const int2* __restrict__ items, int nitems,
                unsigned* __restrict__ counter, double* __restrict__ psi, double* __restrict__ acc,
                double* __restrict__ part) {
    constexpr bool LOADLO = MODE >= 1;  // the tiles carry the low parts
    constexpr bool CENTRE = MODE == 1 || MODE == 2;
    constexpr int NA = LOADLO ? 7 : 4;  // arrays of the computed tile
    // per warp: the raw position records of the tile in flight, and the tile being computed
    // (structure of arrays X | Y | Z | W [| XL | YL | ZL], high parts or offsets)
    __shared__ __align__(16) float4 raws[kP2PWarpsM][2 * kP2PTileM];
    __shared__ __align__(16) float tiles[kP2PWarpsM][NA * kP2PTileM];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    float4* raw = raws[wid];
    float* tile = tiles[wid];
    const f2 zero = f2_pack(0.f, 0.f);
    for (;;) {
        unsigned w = 0;
        if (lane == 0) w = atomicAdd(counter, 1u);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w >= (unsigned)nitems) break;
        const int2 it = items[w];
        const int v = it.x, t = pc.leaf[v], leaf = leaves[t];
        const int first = c.first[leaf], count = c.count[leaf];
        const Chunk ch = PlanMixed::chunk(count);
        const int R = ch.R, S = ch.S;
        const int s0 = it.y * 2 * S, chunk = min(2 * S, count - s0);
        // lanes past S * R repeat replica 0's work; their sums are not used.  The lane's sinks
        // are s0 + slot and s0 + S + slot; a missing one repeats the item's first sink
        const int slot = lane % S, rep = lane / S < R ? lane / S : 0;
        const bool okA = lane < S * R && slot < chunk, okB = lane < S * R && S + slot < chunk;
        const int iA = first + s0 + (slot < chunk ? slot : 0);
        const int iB = first + s0 + (S + slot < chunk ? S + slot : 0);
        // the leaf centre as two floats; the sinks as FP32 offsets from it (CENTRE) or their
        // high parts
        float chx = 0.f, chy = 0.f, chz = 0.f, clx = 0.f, cly = 0.f, clz = 0.f;
        if (CENTRE) {
            const d4 sc = c.sr[leaf];
            chx = (float)sc.x;
            chy = (float)sc.y;
            chz = (float)sc.z;
            clx = (float)(sc.x - (double)chx);
            cly = (float)(sc.y - (double)chy);
            clz = (float)(sc.z - (double)chz);
        }
        auto far_sink = [&](int i) {
            const float4 h = xp[2 * (size_t)i];
            float ox = h.x, oy = h.y, oz = h.z;
            if (CENTRE) {
                const float4 l = xp[2 * (size_t)i + 1];
                ox = __fadd_rn(__fsub_rn(h.x, chx), __fsub_rn(l.x, clx));
                oy = __fadd_rn(__fsub_rn(h.y, chy), __fsub_rn(l.y, cly));
                oz = __fadd_rn(__fsub_rn(h.z, chz), __fsub_rn(l.z, clz));
            }
            return SinkPk{f2_pack(ox, ox), f2_pack(oy, oy), f2_pack(oz, oz), zero, zero, zero};
        };
        auto near_sink = [&](int i) {
            const float4 h = xp[2 * (size_t)i], l = xp[2 * (size_t)i + 1];
            return SinkPk{f2_pack(h.x, h.x), f2_pack(h.y, h.y), f2_pack(h.z, h.z),
                          f2_pack(l.x, l.x), f2_pack(l.y, l.y), f2_pack(l.z, l.z)};
        };
        const SinkPk fA = far_sink(iA), fB = far_sink(iB);
        AccPk aA{zero, zero, zero, zero}, aB{zero, zero, zero, zero};
        ff sA[4], sB[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) sA[q] = sB[q] = ff{0.f, 0.f};
        RangeStream cur;
        {
            const int r0 = pc.r0[v], r1 = pc.r1[v];
            cur.start(ranges, lane, r0, r0 + pc.nnear[v], r1 - pc.nfar[v], r1);
        }
        const int T = p2p_tile(R);  // sources per tile, shared by the replicas
        bool near = false, guard = false, near_next = false, guard_next = false;
        int nt = cur.fill<LOADLO>(ranges, xp, lane, T, raw, near, guard);
        cp_async_commit();
        while (nt > 0) {
            cp_async_wait0();
            __syncwarp();  // the raw tile has arrived; every lane is done with the previous tile
            const int ng = (nt + 3) >> 2;
            const bool two = MODE == 3 || (MODE == 1 && near);
            // the computed tile: offsets from the leaf centre (far, CENTRE) or the parts as they
            // are; padded to whole groups with massless sources far away
            for (int j = lane; j < 4 * ng; j += 32) {
                float x = 1e15f, y = 1e15f, z = 1e15f, wm = 0.f, xl = 0.f, yl = 0.f, zl = 0.f;
                if (j < nt) {
                    const float4 h = raw[2 * j];
                    wm = h.w;
                    if (LOADLO) {
                        const float4 l = raw[2 * j + 1];
                        if (CENTRE && !two) {
                            x = __fadd_rn(__fsub_rn(h.x, chx), __fsub_rn(l.x, clx));
                            y = __fadd_rn(__fsub_rn(h.y, chy), __fsub_rn(l.y, cly));
                            z = __fadd_rn(__fsub_rn(h.z, chz), __fsub_rn(l.z, clz));
                        } else {
                            x = h.x;
                            y = h.y;
                            z = h.z;
                            xl = l.x;
                            yl = l.y;
                            zl = l.z;
                        }
                    } else {
                        x = h.x;
                        y = h.y;
                        z = h.z;
                    }
                }
                tile[j] = x;
                tile[kP2PTileM + j] = y;
                tile[2 * kP2PTileM + j] = z;
                tile[3 * kP2PTileM + j] = wm;
                if (LOADLO && two) {
                    tile[4 * kP2PTileM + j] = xl;
                    tile[5 * kP2PTileM + j] = yl;
                    tile[6 * kP2PTileM + j] = zl;
                }
            }
            __syncwarp();  // the computed tile is complete and the raw tile free
            // the next tile's copies run while this one is computed
            const int nx = cur.fill<LOADLO>(ranges, xp, lane, T, raw, near_next, guard_next);
            cp_async_commit();
            if (two) {  // the sinks' two-float parts, read again for this tile
                const SinkPk nA = near_sink(iA), nB = near_sink(iB);
                if (guard) tile_any<true, true>(tile, ng, rep, R, nA, nB, aA, aB);
                else tile_any<true, false>(tile, ng, rep, R, nA, nB, aA, aB);
            } else {
                if (guard) tile_any<false, true>(tile, ng, rep, R, fA, fB, aA, aB);
                else tile_any<false, false>(tile, ng, rep, R, fA, fB, aA, aB);
            }
            // fold the FP32 partials (<= 128 pairs per sink) into the two-float sums
            fold(aA, sA);
            fold(aB, sB);
            nt = nx;
            near = near_next;
            guard = guard_next;
        }
        // add the replicas' partial sums into the lanes of replica 0 (a tree over the replicas:
        // at step h, replica r takes replica r + h when r is a multiple of 2 h)
        for (int h = 1; h < R; h *= 2) {
            const int src = min(lane + h * S, 31);
            const bool take = rep % (2 * h) == 0 && rep + h < R && lane < S * R;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                ff ta = sA[q], tb = sB[q];
                ff_add_lane(ta, src);
                ff_add_lane(tb, src);
                if (take) {
                    sA[q] = ta;
                    sB[q] = tb;
                }
            }
        }
        // a whole leaf writes psi and acc; a piece of a split leaf its partial-sum slots
        const int pslot = pc.part[v];
        auto out = [&](int i, const ff* sm) {
            double* o4 = pslot >= 0 ? part + 4 * ((size_t)pslot + (size_t)(i - first)) : nullptr;
            const double vv[4] = {(double)sm[0].hi + (double)sm[0].lo, (double)sm[1].hi + (double)sm[1].lo,
                                  (double)sm[2].hi + (double)sm[2].lo, (double)sm[3].hi + (double)sm[3].lo};
            if (o4) {
#pragma unroll
                for (int d = 0; d < 4; ++d) o4[d] = vv[d];
            } else {
                psi[i] = vv[0];
                acc[3 * (size_t)i] = vv[1];
                acc[3 * (size_t)i + 1] = vv[2];
                acc[3 * (size_t)i + 2] = vv[3];
            }
        };
        if (lane < S) {
            if (okA) out(iA, sA);
            if (okB) out(iB, sB);
        }
    }
}

// FP64: one warp per item, sinks and replicas as the plan lays them out (PlanF64), the item's ranges
// as tiles of up to 64 FP64 records in shared memory.  WANT_F: only sum mu / r^2 (the estimate of
// f, eq. 6), in place of psi.
constexpr int kP2PWarpsD = 4;
constexpr int kP2PTileD = 64;

// r2 > 0 by its bits (r2 is no NaN: positions are finite; a comparison of doubles takes the FP64 pipe)
__device__ __forceinline__ bool positive_bits(double r2) { return __double_as_longlong(r2) > 0; }

template <int Q, bool WANT_F>
__device__ __forceinline__ void tile_f64(const d4* __restrict__ tile, int nt, int rep, int R, const double (&b)[4][3],
                                         double (&v)[4][4]) {
    for (int j = rep; j < nt; j += R) {
        const d4 a = tile[j];
#pragma unroll
        for (int u = 0; u < Q; ++u) {
            const double dx = a.x - b[u][0], dy = a.y - b[u][1], dz = a.z - b[u][2];
            const double r2 = dx * dx + dy * dy + dz * dz;
            if (positive_bits(r2)) {
                // (no 1 / r^2 by itself: it overflows for a subnormal r^2, and a massless source would give NaN)
                const double rinv = rsqrt(r2), qm = a.w * rinv;
                if (WANT_F) {
                    v[u][0] = fma(qm, rinv, v[u][0]);
                } else {
                    const double q3 = qm * rinv * rinv;
                    v[u][0] += qm;
                    v[u][1] = fma(q3, dx, v[u][1]);
                    v[u][2] = fma(q3, dy, v[u][2]);
                    v[u][3] = fma(q3, dz, v[u][3]);
                }
            }
        }
    }
}

template <bool WANT_F>
__global__ void __launch_bounds__(kP2PWarpsD * 32)
    k_p2p_f64(const d4* __restrict__ xm, Cells c, const int* __restrict__ leaves, const int2* __restrict__ ranges,
              const Pieces pc, const int2* __restrict__ items, int nitems, unsigned* __restrict__ counter,
              double* __restrict__ psi, double* __restrict__ acc, double* __restrict__ part) {
    constexpr int NV = WANT_F ? 1 : 4;
    __shared__ __align__(32) d4 tiles[kP2PWarpsD][kP2PTileD];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    d4* tile = tiles[wid];
    for (;;) {
        unsigned w = 0;
        if (lane == 0) w = atomicAdd(counter, 1u);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w >= (unsigned)nitems) break;
        const int2 it = items[w];
        const int pv = it.x, leaf = leaves[pc.leaf[pv]];
        const int first = c.first[leaf], count = c.count[leaf];
        const Chunk ch = PlanF64::chunk(count);
        const int R = ch.R, S = ch.S, Q = ch.Q;
        const int s0 = it.y * Q * S, chunk = min(Q * S, count - s0);
        // lanes past S * R repeat replica 0's work; their sums are not used.  A missing sink repeats
        // the item's first one
        const int slot = lane % S, rep = lane / S < R ? lane / S : 0;
        double b[4][3], v[4][4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int k = u * S + slot;
            const d4 xb = xm[first + s0 + (u < Q && k < chunk ? k : 0)];
            b[u][0] = xb.x;
            b[u][1] = xb.y;
            b[u][2] = xb.z;
#pragma unroll
            for (int d = 0; d < 4; ++d) v[u][d] = 0.0;
        }
        RangeStream cur;
        {
            const int r0 = pc.r0[pv], r1 = pc.r1[pv];
            cur.start(ranges, lane, r0, r0 + pc.nnear[pv], r1 - pc.nfar[pv], r1);
        }
        const int T = R * (kP2PTileD / R);  // sources per tile, shared by the replicas
        for (;;) {
            bool near, guard;
            __syncwarp();  // every lane is done with the previous tile
            const int nt = cur.fill<true>(ranges, (const float4*)xm, lane, T, (float4*)tile, near, guard);
            if (nt == 0) break;
            cp_async_commit();
            cp_async_wait0();
            __syncwarp();
            switch (Q) {
                case 1: tile_f64<1, WANT_F>(tile, nt, rep, R, b, v); break;
                case 2: tile_f64<2, WANT_F>(tile, nt, rep, R, b, v); break;
                case 3: tile_f64<3, WANT_F>(tile, nt, rep, R, b, v); break;
                default: tile_f64<4, WANT_F>(tile, nt, rep, R, b, v); break;
            }
        }
        // the replicas' sums into the lanes of replica 0, in the order of a tree
        for (int h = 1; h < R; h *= 2) {
            const int src = min(lane + h * S, 31);
            const bool take = rep % (2 * h) == 0 && rep + h < R && lane < S * R;
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int d = 0; d < NV; ++d) {
                    const double o = __shfl_sync(0xffffffffu, v[u][d], src);
                    if (take) v[u][d] += o;
                }
        }
        const int pslot = pc.part[pv];
        if (lane < S) {
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const int k = u * S + slot;
                if (u >= Q || k >= chunk) continue;
                if (pslot >= 0) {
                    double* o = part + 4 * ((size_t)pslot + (size_t)(s0 + k));
#pragma unroll
                    for (int d = 0; d < 4; ++d) o[d] = v[u][d];
                } else {
                    const size_t i = (size_t)first + s0 + k;
                    psi[i] = v[u][0];
#pragma unroll
                    for (int d = 1; d < NV; ++d) acc[3 * i + d - 1] = v[u][d];
                }
            }
        }
    }
}

// The near tidal tensor in mixed precision (Sec. 7.4): dx from the two-float positions, FP32 pair terms
// summed over a tile (at most 32 sources of one source cell, in order), the tiles added as two-float
// sums.  30 packed FP32 operations and two rsqrt for the two pairs of a slot: bound by the FMA pipe.
// The R groups of S lanes take tiles of their own, all in step: the source cells are cut into tiles 32
// records at a time, the tiles ordered by length and dealt to the groups, so that the tiles of a round
// are about equally long.  The shorter ones are filled up with massless sources beside the leaf: its first
// particle moved by 4 units in x (the extent is below 2; of a system without extent, whose coordinates
// are not scaled, the low part holds the move), so that 1 / r^2 and r^2 stay in range wherever the
// leaf lies.  (A filler at a fixed place is no zero term: for a sink within 5e-20 of it 1 / r^2 overflows,
// for one farther than 1.8e19 r^2 does, and 0 times infinity is NaN.)  150,001 particles, 1.16e9 pairs:
// 19.0 ms with one warp per leaf and one sink per lane (the longest leaf ran on alone), 3.3 ms with
// groups that run through their tiles on their own (they diverge), 2.2 ms so.
constexpr int kTidWarps = 4;
constexpr int kTidTile = 32;
constexpr int kTidGroups = 4;  // PlanTidal's largest R
constexpr int kTidBatch = 64;  // tiles ordered together

struct TidAcc {
    f2 p[6];
};
// one source (h: high parts and mass, l: low parts) against the slot's two sinks
__device__ __forceinline__ void tid_pair(const float4& h, const float4& l, const f2 (&bh)[3], const f2 (&bl)[3],
                                         TidAcc& a) {
    const f2 dx = f2_add(f2_sub(bh[0], f2_pack(h.x, h.x)), f2_sub(bl[0], f2_pack(l.x, l.x)));
    const f2 dy = f2_add(f2_sub(bh[1], f2_pack(h.y, h.y)), f2_sub(bl[1], f2_pack(l.y, l.y)));
    const f2 dz = f2_add(f2_sub(bh[2], f2_pack(h.z, h.z)), f2_sub(bl[2], f2_pack(l.z, l.z)));
    const f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_mul(dz, dz)));
    float ra, rb;
    f2_unpack(r2, ra, rb);
    float ia = rsqrt_ftz(ra), ib = rsqrt_ftz(rb);
    if (fminf(ra, rb) < 0x1p-126f) {  // coincident (skipped) or subnormal
        if (ra < 0x1p-126f) ia = ra > 0.f ? rsqrtf(ra) : 0.f;
        if (rb < 0x1p-126f) ib = rb > 0.f ? rsqrtf(rb) : 0.f;
    }
    const f2 ri = f2_pack(ia, ib), ri2 = f2_mul(ri, ri);
    const f2 q5 = f2_mul(f2_mul(f2_mul(f2_pack(h.w, h.w), ri), ri2), ri2);
    const f2 q3 = f2_mul(f2_pack(3.f, 3.f), q5);
    const f2 nq5 = q5 ^ 0x8000000080000000ull;  // -q5
    const f2 qx = f2_mul(q3, dx), qy = f2_mul(q3, dy), qz = f2_mul(q3, dz);
    a.p[0] = f2_fma(qx, dx, f2_fma(nq5, r2, a.p[0]));
    a.p[1] = f2_fma(qx, dy, a.p[1]);
    a.p[2] = f2_fma(qx, dz, a.p[2]);
    a.p[3] = f2_fma(qy, dy, f2_fma(nq5, r2, a.p[3]));
    a.p[4] = f2_fma(qy, dz, a.p[4]);
    a.p[5] = f2_fma(qz, dz, f2_fma(nq5, r2, a.p[5]));
}
// sum += the tile's value (TwoSum, both halves)
__device__ __forceinline__ void tid_fold(f2& hi, f2& lo, f2 v) {
    const f2 s = f2_add(hi, v), bb = f2_sub(s, hi);
    const f2 e = f2_add(f2_sub(hi, f2_sub(s, bb)), f2_sub(v, bb));
    hi = s;
    lo = f2_add(lo, e);
}

__global__ void __launch_bounds__(kTidWarps * 32)
    k_p2p_tidal_mixed(const float4* __restrict__ xp, Cells c, const int* __restrict__ leaves,
                      const int2* __restrict__ ranges, const Pieces pc, const int2* __restrict__ items, int nitems,
                      unsigned* __restrict__ counter, double* __restrict__ T, double* __restrict__ part) {
    __shared__ __align__(16) float4 bufs[kTidWarps][2][kTidGroups][2 * kTidTile];
    __shared__ int2 tiles_all[kTidWarps][kTidBatch], sorted_all[kTidWarps][kTidBatch];
    __shared__ __align__(16) float4 fill_all[kTidWarps][2];  // the record of the fillers
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const f2 zero = f2_pack(0.f, 0.f);
    for (;;) {
        unsigned w = 0;
        if (lane == 0) w = atomicAdd(counter, 1u);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w >= (unsigned)nitems) break;
        const int2 it = items[w];
        const int pv = it.x, leaf = leaves[pc.leaf[pv]];
        const int first = c.first[leaf], count = c.count[leaf];
        const Chunk ch = PlanTidal::chunk(count);
        const int R = ch.R, S = ch.S;
        const int s0 = it.y * 2 * S, chunk = min(2 * S, count - s0);
        const int slot = lane % S, g = lane / S;
        const bool in = g < R;
        const int kA = slot < chunk ? slot : 0, kB = S + slot < chunk ? S + slot : 0;
        f2 bh[3], bl[3], sh[6], sl[6];
        {
            const size_t iA = (size_t)(first + s0 + kA), iB = (size_t)(first + s0 + kB);
            const float4 ah = xp[2 * iA], al = xp[2 * iA + 1], dh = xp[2 * iB], dl = xp[2 * iB + 1];
            bh[0] = f2_pack(ah.x, dh.x);
            bh[1] = f2_pack(ah.y, dh.y);
            bh[2] = f2_pack(ah.z, dh.z);
            bl[0] = f2_pack(al.x, dl.x);
            bl[1] = f2_pack(al.y, dl.y);
            bl[2] = f2_pack(al.z, dl.z);
        }
#pragma unroll
        for (int q = 0; q < 6; ++q) sh[q] = sl[q] = zero;
        int2 *tiles = tiles_all[wid], *sorted = sorted_all[wid];
        float4* fill = fill_all[wid];
        if (lane < 2) {
            fill[lane] = xp[2 * (size_t)first + lane];
            if (lane == 0) fill[0].w = 0.f;
            else fill[1].x += 4.f;
        }
        const int end = pc.r1[pv];
        int at = pc.r0[pv], off = 0;  // the next record and the tiles of it that are done
        while (at < end) {
            // the next records' tiles, as many as the batch holds
            const int2 rec = at + lane < end ? ranges[at + lane] : make_int2(0, 0);
            const int o = lane == 0 ? off : 0, nt = (rec.y + kTidTile - 1) / kTidTile - o;
            int incl = nt;
#pragma unroll
            for (int h = 1; h < 32; h <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, h);
                if (lane >= h) incl += y;
            }
            const unsigned fit = __ballot_sync(0xffffffffu, incl <= kTidBatch);
            const int nrec = fit ? __popc(fit & ~(fit + 1u)) : 0;  // records taken whole (a prefix)
            const int ntl = nrec ? __shfl_sync(0xffffffffu, incl, nrec - 1) : kTidBatch;
            const int take = nrec ? (lane < nrec ? nt : 0) : (lane == 0 ? kTidBatch : 0);
            for (int k = 0; k < take; ++k) {
                const int d = (o + k) * kTidTile;
                tiles[incl - nt + k] = make_int2(rec.x + d, min(kTidTile, rec.y - d));
            }
            if (nrec) {
                at += min(nrec, end - at);
                off = 0;
            } else {
                off += kTidBatch;
            }
            __syncwarp();
            // ordered by decreasing length
            for (int k = lane; k < ntl; k += 32) {
                const int2 mine = tiles[k];
                int r = 0;
                for (int j = 0; j < ntl; ++j) {
                    const int y = tiles[j].y;
                    r += y > mine.y || (y == mine.y && j < k);
                }
                sorted[r] = mine;
            }
            __syncwarp();
            // copy the tiles of round i (one per group), filled up to the longest of them
            auto fetch = [&](int i, int b) {
                if (i * R >= ntl || !in) return;
                const float4 fh = fill[0], fl = fill[1];  // (here, so that the copies' issue hides the reads)
                const int nmax = sorted[i * R].y, k = i * R + g;
                const int2 t = k < ntl ? sorted[k] : make_int2(0, 0);
                float4* buf = bufs[wid][b][g];
                const float4* src = xp + 2 * (size_t)t.x;
                for (int j = slot; j < 2 * t.y; j += S) cp_async16(buf + j, src + j);
                for (int j = t.y + slot; j < nmax; j += S) {
                    buf[2 * j] = fh;
                    buf[2 * j + 1] = fl;
                }
            };
            fetch(0, 0);
            cp_async_commit();
            for (int i = 0; i * R < ntl; ++i) {
                cp_async_wait0();
                __syncwarp();  // the round's tiles have arrived, and the other buffer is no longer read
                fetch(i + 1, (i + 1) & 1);
                cp_async_commit();
                const int n = sorted[i * R].y;
                const float4* t = bufs[wid][i & 1][in ? g : 0];
                TidAcc a;
#pragma unroll
                for (int q = 0; q < 6; ++q) a.p[q] = zero;
#pragma unroll 2
                for (int j = 0; j < n; ++j) tid_pair(t[2 * j], t[2 * j + 1], bh, bl, a);
#pragma unroll
                for (int q = 0; q < 6; ++q) tid_fold(sh[q], sl[q], a.p[q]);
            }
            cp_async_wait0();
            __syncwarp();
        }
        __syncwarp();
        // the groups' sums, in group order, as FP64
        const int pslot = pc.part[pv];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            float hA, hB, lA, lB;
            f2_unpack(sh[q], hA, hB);
            f2_unpack(sl[q], lA, lB);
            double vA = (double)hA + (double)lA, vB = (double)hB + (double)lB;
            double tA = vA, tB = vB;
            for (int r = 1; r < R; ++r) {
                tA += __shfl_sync(0xffffffffu, vA, min(slot + r * S, 31));
                tB += __shfl_sync(0xffffffffu, vB, min(slot + r * S, 31));
            }
            if (lane < S) {
                double* o = pslot >= 0 ? part + 6 * ((size_t)pslot + (size_t)s0) : T + 6 * ((size_t)first + s0);
                if (slot < chunk) o[6 * (size_t)slot + q] = tA;
                if (S + slot < chunk) o[6 * (size_t)(S + slot) + q] = tB;
            }
        }
    }
}

namespace {
// layout of the fixed part of the scratch (depends on the number of leaves only)
struct PlanLayout {
    uint64_t *k0, *k1;
    int *order, *nb, *roff, *np, *kc, *npc, *voff, *nit, *ioff, *pbase, *stmp, *rtmp;
    int2* split;
    unsigned long long* tot;  // [0] ranges, [1] items, [2] parts' records, [3] pieces, [4] partial slots,
                              // [5] split leaves
    unsigned* counter;
    size_t bytes;
};
PlanLayout plan_layout(void* base, int nleaves) {
    PlanLayout L;
    const size_t nl = (size_t)(nleaves > 0 ? nleaves : 1);
    unsigned char* p = (unsigned char*)base;
    size_t off = 0;
    auto take = [&](size_t bytes) {
        off = (off + 255) & ~(size_t)255;
        unsigned char* r = p ? p + off : nullptr;
        off += bytes;
        return r;
    };
    L.tot = (unsigned long long*)take(8 * 8);  // (tot, counter and k1 side by side: cleared together)
    L.counter = (unsigned*)take(4 * 4);
    L.k1 = (uint64_t*)take(nl * 8);
    L.k0 = (uint64_t*)take(nl * 8);
    L.order = (int*)take(nl * 4);
    L.nb = (int*)take(nl * 4);
    L.roff = (int*)take((nl + 1) * 4);
    L.np = (int*)take(nl * 4);
    L.kc = (int*)take(nl * 4);
    L.npc = (int*)take(nl * 4);
    L.voff = (int*)take((nl + 1) * 4);
    L.nit = (int*)take(nl * 4);
    L.ioff = (int*)take((nl + 1) * 4);
    L.pbase = (int*)take(nl * 4);
    L.split = (int2*)take(nl * 8);
    L.stmp = (int*)take(scan_tmp_ints((long long)nl + 1) * 4);
    L.rtmp = (int*)take(radix_tmp_ints((long long)nl) * 4);
    L.bytes = (off + 255) & ~(size_t)255;
    return L;
}

// the work plan of PL over the segments of list, then run(ranges, pieces, items, nitems, counter,
// part) and the sum of the split leaves' pieces into psi and acc; the return value as
// launch_p2p_mixed's
template <class PL, class RUN>
size_t plan_and_run(int n, Cells c, const int2* list, const int* seg_start, const int* seg_end, const int* leaves,
                    int nleaves, double* psi, double* acc, int mode, void* tmp, size_t tmp_bytes,
                    unsigned long long* h_tot, bool shares, const int* off, int nsys, PlanBudget bg, cudaStream_t s,
                    RUN run) {
    if (nleaves <= 0) return 0;
    if (n > kRangeMax) return ~(size_t)0;  // no range is ever cut: a leaf's region holds its source cells
    PlanLayout L = plan_layout(tmp, nleaves);
    if (tmp_bytes < L.bytes) return L.bytes;
    const bool cut = PL::budget && 32.0 * n * (4.0 * n + 1.0) > (double)PL::piece_steps * (bg.base + bg.per * n);
    unsigned long long* work = cut ? (unsigned long long*)L.k1 : nullptr;  // (k1 and voff have their own use later)
    int* root = L.voff;
    unsigned char* zero_end = cut ? (unsigned char*)(work + nleaves) : (unsigned char*)(L.counter + 4);  // (roots <= leaves)
    cudaMemsetAsync(L.tot, 0, (size_t)(zero_end - (unsigned char*)L.tot), s);
    k_p2p_count<PL><<<grid_for((long long)nleaves * 32, 128, 16), 128, 0, s>>>(
        c, list, seg_start, seg_end, leaves, nleaves, shares ? PL::sub_n : 0, n, off, nsys, L.nb, L.np, L.kc, L.k0, root, work,
        L.tot);
    note_launch();
    if constexpr (PL::budget) if (cut) {
        k_p2p_pieces<PL><<<grid_for(nleaves, 128), 128, 0, s>>>(c, nleaves, L.nb, root, work, bg, L.np, L.k0);
        note_launch();
    }
    scan_exclusive_i32(L.nb, L.roff, nleaves, L.roff + nleaves, L.stmp, s);
    // the low 32 bits are the leaf index, already in order: sort the 8 length bits only
    const int flip = radix_sort_pairs_bits(L.k0, nullptr, L.k1, nullptr, nleaves, L.rtmp, 32, 40, s);
    int* cbase = (int*)(flip ? L.k0 : L.k1);  // (the sort's other buffer is free)
    k_p2p_nitems<<<grid_for(nleaves, 256), 256, 0, s>>>(flip ? L.k1 : L.k0, leaves, nleaves, c, L.np, L.nb, L.kc,
                                                        L.order, L.nit, L.npc, L.pbase, cbase, L.split, L.tot);
    note_launch();
    scan_exclusive_i32(L.nit, L.ioff, nleaves, L.ioff + nleaves, L.stmp, s);
    scan_exclusive_i32(L.npc, L.voff, nleaves, L.voff + nleaves, L.stmp, s);
    cudaMemcpyAsync(h_tot, L.tot, 6 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, s);
    cudaStreamSynchronize(s);
    const unsigned long long nranges = h_tot[0], nitems = h_tot[1], ncuts = h_tot[2], npieces = h_tot[3],
                             nslots = h_tot[4], nsplit = h_tot[5], most = INT_MAX;
    // (a part's records are indexed from the ranges, with the items and pieces between them)
    if (nranges > most || nitems > most || nslots > most ||
        (ncuts && nranges + nitems + 3 * npieces + ncuts + 128 > most))
        return ~(size_t)0;
    auto a256 = [](unsigned long long b) { return (size_t)((b + 255) & ~255ull); };
    const size_t o_ranges = L.bytes, o_items = o_ranges + a256(nranges * sizeof(int2)),
                 o_pieces = o_items + a256(nitems * sizeof(int2)),
                 o_cuts = o_pieces + a256(npieces * 6 * sizeof(int)),
                 o_part = o_cuts + a256(ncuts * sizeof(int2)),
                 need = o_part + a256(nslots * PL::nv * sizeof(double)) + 256;
    if (tmp_bytes < need) return need;
    unsigned char* b = (unsigned char*)tmp;
    int2* ranges = (int2*)(b + o_ranges);
    int2* items = (int2*)(b + o_items);
    int* pv = (int*)(b + o_pieces);
    const size_t npv = (size_t)npieces;
    const Pieces pc{pv, pv + npv, pv + 2 * npv, pv + 3 * npv, pv + 4 * npv, pv + 5 * npv};
    double* part = (double*)(b + o_part);
    if (nitems == 0) return need;
    const unsigned g = grid_for((long long)npieces * 32, kEmitWarps * 32, 16);  // one warp per piece
    k_p2p_emit<PL><<<g, kEmitWarps * 32, 0, s>>>(c, list, seg_start, seg_end, leaves, nleaves, mode, L.order, L.roff,
                                             L.nb, L.ioff, L.nit, L.voff, L.npc, L.np, L.pbase, cbase, (int)npieces, pc, ranges,
                                             (int2*)(b + o_cuts), items);
    note_launch();
    run(ranges, pc, items, (int)nitems, L.counter, part);
    if (nsplit > 0) {
        k_p2p_reduce<PL::nv><<<grid_for((long long)nsplit * 32, 128, 16), 128, 0, s>>>(
            c, leaves, L.np, L.split, (int)nsplit, part, psi, acc);
        note_launch();
    }
    return need;
}
// persistent blocks of a kernel whose warps take the items: as many as are resident on the device at once
// (at most per_sm per SM), but no more than the items need, so that a few items are spread over the SMs
// (with every resident block some SMs' warps took several of the long items: the estimate of 4096
// particles in FP64 0.65 ms)
template <class K>
int item_blocks(K kern, int threads, int nitems, int per_sm = 32) {
    int bps = 1;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, kern, threads, 0);
    const int w = threads / 32;
    return std::min(sm_count() * std::min(bps < 1 ? 1 : bps, per_sm), (nitems + w - 1) / w);
}
}  // namespace

bool p2p_shares(int smallest_system) { return smallest_system <= PlanMixed::sub_n; }

size_t p2p_plan_fixed_bytes(int nleaves) { return plan_layout(nullptr, nleaves).bytes; }

size_t launch_p2p_mixed(const float4* xp, int n, Cells c, const int2* list, const int* seg_start,
                        const int* seg_end, const int* leaves, int nleaves, double* psi, double* acc, int mode,
                        void* tmp, size_t tmp_bytes, unsigned long long* h_tot, cudaStream_t s, bool shares,
                        const int* off, int nsys) {
    auto run = [&](const int2* ranges, const Pieces& pc, const int2* items, int nitems, unsigned* counter,
                   double* part) {
        auto go = [&](auto kern) {
            const int nblocks = item_blocks(kern, kP2PWarpsM * 32, nitems);
            mark_begin(s);
            kern<<<nblocks, kP2PWarpsM * 32, 0, s>>>(xp, c, leaves, ranges, pc, items, nitems, counter, psi, acc, part);
            mark_end(s);
        };
        if (mode == 1) go(k_p2p_mixed<1>);
        else if (mode == 2) go(k_p2p_mixed<2>);
        else if (mode == 3) go(k_p2p_mixed<3>);
        else go(k_p2p_mixed<0>);
        note_launch();
    };
    return plan_and_run<PlanMixed>(n, c, list, seg_start, seg_end, leaves, nleaves, psi, acc, mode, tmp, tmp_bytes,
                                   h_tot, shares, off, nsys, PlanBudget{0.0, 0.0}, s, run);
}

size_t launch_p2p_f64_plan(const d4* xm, int n, Cells c, const int2* list, const int* seg_start, const int* seg_end,
                           const int* leaves, int nleaves, double* psi, double* acc, bool want_f, PlanBudget bg,
                           void* tmp, size_t tmp_bytes, unsigned long long* h_tot, cudaStream_t s) {
    auto run = [&](const int2* ranges, const Pieces& pc, const int2* items, int nitems, unsigned* counter,
                   double* part) {
        auto go = [&](auto kern) {
            // Eight warps per SM keep the FP64 pipe busy, and with few items per warp more only take the long
            // ones early (both P2P kernels of 4096 particles 0.99 ms, 0.95 with two blocks per SM).  With many items every
            // resident block: two per SM crowd on the SMs that the M2L beside them leaves first (cusp of 6e4
            // 28.6 ms, 21.5 so).
            const bool few = nitems <= 4 * 2 * kP2PWarpsD * sm_count();
            const int nblocks = item_blocks(kern, kP2PWarpsD * 32, nitems, few ? 2 : 32);
            kern<<<nblocks, kP2PWarpsD * 32, 0, s>>>(xm, c, leaves, ranges, pc, items, nitems, counter, psi, acc, part);
        };
        if (want_f) go(k_p2p_f64<true>);
        else go(k_p2p_f64<false>);
        note_launch();
    };
    return plan_and_run<PlanF64>(n, c, list, seg_start, seg_end, leaves, nleaves, psi, acc, 0, tmp, tmp_bytes, h_tot,
                                 false, nullptr, 0, bg, s, run);
}

size_t launch_p2p_tidal_plan(const float4* xp, int n, Cells c, const int2* list, const int* seg_start,
                             const int* seg_end, const int* leaves, int nleaves, double* T, PlanBudget bg, void* tmp,
                             size_t tmp_bytes, unsigned long long* h_tot, cudaStream_t s) {
    auto run = [&](const int2* ranges, const Pieces& pc, const int2* items, int nitems, unsigned* counter,
                   double* part) {
        k_p2p_tidal_mixed<<<item_blocks(k_p2p_tidal_mixed, kTidWarps * 32, nitems), kTidWarps * 32, 0, s>>>(
            xp, c, leaves, ranges, pc, items, nitems, counter, T, part);
        note_launch();
    };
    return plan_and_run<PlanTidal>(n, c, list, seg_start, seg_end, leaves, nleaves, nullptr, T, 0, tmp, tmp_bytes,
                                   h_tot, false, nullptr, 0, bg, s, run);
}

}  // namespace gb3
