// sort.cu -- the device-wide exclusive scan and the stable LSD radix sorts (Morton keys, interaction
// lists by sink, work orders), each one kernel per pass over the data.
//
// Both use the chained scan with look-back (Merrill and Garland 2016): a block takes the next tile by
// a ticket, publishes the tile's counts, and adds up the counts of the tiles before it from their
// published words until it meets one that already holds a full prefix.  A tile only waits for tiles
// with lower tickets, whose blocks are running; a wait is limited all the same, and past the limit
// the block counts the items before its tile itself, so no wait decides the result.
//
// What bounds them: for the short arrays of small systems the launches (a pass was a histogram, a
// scan of one to three kernels and a scatter), for long ones the traffic (the keys were read twice a
// pass).  A 1e4 evaluation had 0.67 ms of sort and scan kernels in histogram, scan and scatter form and
// had 0.27 ms so; whole calls 2.52 -> 2.22 ms (1e4), 4.97 -> 4.44 (1e5).  Short sorts now run in one cluster.
#include <cooperative_groups.h>

#include "kernels.cuh"

namespace gb3 {
namespace cg = cooperative_groups;
namespace {

typedef unsigned long long u64;
constexpr int kPollLimit = 1 << 20;
// published word: count | flag << 56 (1 the tile's own count, 2 with all tiles before) | pass << 58
constexpr u64 kOwn = 1ull << 56, kAll = 2ull << 56, kCountMask = kOwn - 1;

__device__ __forceinline__ u64 load_word(const u64* p) { return *(const volatile u64*)p; }
__device__ __forceinline__ void store_word(u64* p, u64 v) { *(volatile u64*)p = v; }

// sum of the counts of the tiles before tile b (words at st + stride * tile); false past the limit.
// The words of kBack tiles are read at a time: while the first tiles run, the nearest full prefix is
// many tiles back.
constexpr int kBack = 4;
__device__ inline bool look_back(const u64* st, long long b, long long stride, u64 tag, u64& sum) {
    sum = 0;
    int polls = 0;
    for (long long t = b - 1; t >= 0;) {
        u64 v[kBack];
        const int m = t + 1 < kBack ? (int)(t + 1) : kBack;
#pragma unroll
        for (int i = 0; i < kBack; ++i) v[i] = i < m ? load_word(st + (t - i) * stride) : 0;
        bool wait = false;
#pragma unroll
        for (int i = 0; i < kBack; ++i) {
            if (i >= m || wait) continue;
            if ((v[i] >> 58) != tag || !(v[i] & (kOwn | kAll))) {
                wait = true;  // not published yet: read again from here
                continue;
            }
            sum += v[i] & kCountMask;
            if (v[i] & kAll) return true;
            --t;
        }
        if (wait && ++polls > kPollLimit) return false;
    }
    return true;
}

// ---------------------------------------------------------------- scan
constexpr int kScanThreads = 256;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;
constexpr int kScanOne = 1024 * 16;  // up to here one block does it all

// exclusive scan of v over the block (blockDim a multiple of 32); total: the block's sum
__device__ inline int block_scan(int v, int* sw, int& total) {
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) sw[w] = x;
    __syncthreads();
    if (w == 0) {
        int s = lane < nw ? sw[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < nw) sw[lane] = s;
    }
    __syncthreads();
    const int base = w ? sw[w - 1] : 0;
    total = sw[nw - 1];
    __syncthreads();
    return base + x - v;
}

template <int THREADS, int ITEMS>
__global__ void __launch_bounds__(THREADS) k_scan(const int* __restrict__ in, int* __restrict__ out, long long n,
                                                  int* __restrict__ d_total, u64* __restrict__ st,
                                                  unsigned* __restrict__ ticket) {
    __shared__ int sw[32];
    __shared__ unsigned s_b;
    __shared__ u64 s_pre;
    if (threadIdx.x == 0) s_b = ticket ? atomicAdd(ticket, 1u) : 0u;
    __syncthreads();
    const long long b = s_b, base = b * (THREADS * ITEMS), i0 = base + (long long)threadIdx.x * ITEMS;
    int v[ITEMS], local = 0;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        v[k] = i0 + k < n ? in[i0 + k] : 0;
        local += v[k];
    }
    int total;
    const int ex = block_scan(local, sw, total);
    int pre = 0;
    if (ticket) {
        if (threadIdx.x == 0) {
            u64 sum = 0;
            bool ok = true;
            if (b > 0) {
                store_word(st + b, (u64)(unsigned)total | kOwn);
                ok = look_back(st, b, 1, 0, sum);
            }
            s_pre = ok ? sum : ~0ull;
        }
        __syncthreads();
        if (s_pre == ~0ull) {  // past the waiting limit: add up the items before the tile
            int part = 0, all;
            for (long long i = threadIdx.x; i < base; i += THREADS) part += in[i];
            block_scan(part, sw, all);
            if (threadIdx.x == 0) s_pre = (u64)(unsigned)all;
            __syncthreads();
        }
        pre = (int)(unsigned)s_pre;
        if (threadIdx.x == 0) store_word(st + b, (u64)(unsigned)(pre + total) | kAll);
    }
    int run = pre + ex;
#pragma unroll
    for (int k = 0; k < ITEMS; ++k) {
        if (i0 + k < n) out[i0 + k] = run;
        run += v[k];
    }
    if (d_total && base + THREADS * ITEMS >= n && threadIdx.x == THREADS - 1) *d_total = run;
}

}  // namespace

size_t scan_tmp_ints(long long n) { return n > kScanOne ? 2 * (size_t)((n + kScanTile - 1) / kScanTile) + 6 : 1; }

void scan_exclusive_i32(const int* in, int* out, long long n, int* d_total, int* tmp, cudaStream_t s) {
    if (n <= 0) {
        if (d_total) cudaMemsetAsync(d_total, 0, sizeof(int), s);
        return;
    }
    if (n <= kScanTile) {
        k_scan<kScanThreads, kScanItems><<<1, kScanThreads, 0, s>>>(in, out, n, d_total, nullptr, nullptr);
    } else if (n <= kScanOne) {
        k_scan<1024, 16><<<1, 1024, 0, s>>>(in, out, n, d_total, nullptr, nullptr);
    } else {
        const long long tiles = (n + kScanTile - 1) / kScanTile;
        u64* st = (u64*)(((uintptr_t)tmp + 7) & ~(uintptr_t)7);
        unsigned* ticket = (unsigned*)(st + tiles);
        cudaMemsetAsync(st, 0, (size_t)tiles * sizeof(u64) + sizeof(unsigned), s);
        k_scan<kScanThreads, kScanItems><<<(unsigned)tiles, kScanThreads, 0, s>>>(in, out, n, d_total, st, ticket);
    }
    note_launch();
}

namespace {
// ---------------------------------------------------------------- radix sort
// 8 bits a pass.  A warp ranks its items of a tile in item order (match masks and a counter per digit
// in shared memory), the tile is put in digit order in shared memory and written out in runs.
constexpr int kRsThreads = 256;
constexpr int kRsWarps = kRsThreads / 32;
// items per thread: 8, or 16 for the keys-only sorts of more than kRsLong items, whose looking back
// takes more instructions than the ranking (2.86e6 32-bit keys: 46 us a pass with 8, 34 us with 16;
// 6.4e6: 82 and 62; below, the tiles of 16 are too few for the SMs)
constexpr int kRsItems = 8, kRsItemsLong = 16;
constexpr long long kRsLong = 1 << 19;
constexpr int kRsTile = kRsThreads * kRsItems;  // the smaller tile sizes the scratch
constexpr int kRsMaxPasses = 8;

// scratch: the words of every tile and digit (one array for all passes, told apart by their pass), a
// histogram and a ticket per pass; zero before the sort
struct RsTmp {
    u64* st;
    unsigned* hist;    // [kRsMaxPasses][256]
    unsigned* ticket;  // [kRsMaxPasses]
    size_t bytes;
    RsTmp(void* tmp, long long n) {
        const size_t tiles = (size_t)((n + kRsTile - 1) / kRsTile);
        st = (u64*)(((uintptr_t)tmp + 7) & ~(uintptr_t)7);
        hist = (unsigned*)(st + tiles * 256);
        ticket = hist + kRsMaxPasses * 256;
        bytes = (size_t)((unsigned char*)(ticket + kRsMaxPasses) - (unsigned char*)st);
    }
};

// the digit histograms of all passes; SRC(i) gives key i and may store it
template <class SRC>
__device__ __forceinline__ void histograms(SRC key_of, long long n, int shift0, int passes, unsigned* hist) {
    __shared__ unsigned h[kRsMaxPasses * 256];
    for (int i = threadIdx.x; i < passes * 256; i += blockDim.x) h[i] = 0;
    __syncthreads();
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
        const u64 k = key_of(i);
        for (int p = 0; p < passes; ++p) atomicAdd(&h[p * 256 + (int)((k >> (shift0 + 8 * p)) & 255)], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < passes * 256; i += blockDim.x)
        if (h[i]) atomicAdd(&hist[i], h[i]);
}
template <class K>
__global__ void __launch_bounds__(256) k_rs_hist(const K* __restrict__ keys, long long n, int shift0, int passes,
                                                 unsigned* __restrict__ hist) {
    histograms([&](long long i) { return (u64)keys[i]; }, n, shift0, passes, hist);
}
// key = (sink << xb) | first entry: the first entry (taken as unsigned) in the low xb bits
template <class K>
__global__ void __launch_bounds__(256) k_rs_pack(const int2* __restrict__ list, long long n, int xb, int passes,
                                                 K* __restrict__ keys, unsigned* __restrict__ hist) {
    histograms(
        [&](long long i) {
            const int2 v = list[i];
            const u64 k = ((u64)(unsigned)v.y << xb) | (u64)(unsigned)v.x;
            keys[i] = (K)k;
            return k;
        },
        n, 0, passes, hist);
}

// one pass: items by the digit at shift (VALS: with values; list != nullptr: keys are written as pairs)
template <class K, bool VALS, int ITEMS>
__global__ void __launch_bounds__(kRsThreads) k_rs_pass(const K* __restrict__ kin, const int* __restrict__ vin,
                                                        K* __restrict__ kout, int* __restrict__ vout, long long n,
                                                        int shift, int pass, u64* __restrict__ st,
                                                        const unsigned* __restrict__ hist,
                                                        unsigned* __restrict__ ticket, int2* __restrict__ list,
                                                        int xb) {
    constexpr int kTile = kRsThreads * ITEMS;
    __shared__ K s_key[kTile];
    __shared__ int s_val[VALS ? kTile : 1];
    __shared__ unsigned wc[kRsWarps][256];
    __shared__ long long gofs[256];
    __shared__ unsigned toff[256];
    __shared__ int sw[32];
    __shared__ unsigned s_b;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, d0 = threadIdx.x;
    if (threadIdx.x == 0) s_b = atomicAdd(ticket + pass, 1u);
#pragma unroll
    for (int k = 0; k < kRsWarps; ++k) wc[k][d0] = 0;
    __syncthreads();
    const long long b = s_b, base = b * kTile;
    const int cnt = (int)min((long long)kTile, n - base);
    // ranks within the warp's items, in item order
    K key[ITEMS];
    int val[VALS ? ITEMS : 1];
    unsigned rank[ITEMS];
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const int j = (w * ITEMS + i) * 32 + lane;
        key[i] = j < cnt ? kin[base + j] : (K)0;
        if (VALS) val[i] = j < cnt ? vin[base + j] : 0;
    }
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        const bool valid = (w * ITEMS + i) * 32 + lane < cnt;
        const int d = (int)((key[i] >> shift) & 255);
        // the lanes with the same digit, a bit at a time (__match_any_sync takes several times as long)
        unsigned peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const unsigned on = (d >> k) & 1 ? 0xffffffffu : 0u;
            peers &= ~(on ^ __ballot_sync(0xffffffffu, on != 0u));
        }
        const unsigned c = valid ? wc[w][d] : 0u;
        rank[i] = c + __popc(peers & ((1u << lane) - 1u));
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) wc[w][d] = c + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // digit d0: the warps' offsets, the tile's count, its place in the tile and in the output
    unsigned own = 0;
#pragma unroll
    for (int k = 0; k < kRsWarps; ++k) {
        const unsigned c = wc[k][d0];
        wc[k][d0] = own;
        own += c;
    }
    const u64 tag = (u64)pass + 1;
    u64* word = st + b * 256 + d0;
    if (b > 0) store_word(word, (u64)own | kOwn | tag << 58);
    int all;
    toff[d0] = (unsigned)block_scan((int)own, sw, all);
    // exclusive scan of the digits' totals (each below 2^31 and so their sum)
    const int gbase = block_scan((int)hist[pass * 256 + d0], sw, all);
    u64 before = 0;
    const bool ok = b == 0 || look_back(st + d0, b, 256, tag, before);
    if (__syncthreads_or(!ok)) {  // past the waiting limit: count the keys before the tile
        unsigned* h = (unsigned*)s_key;
        h[d0] = 0;
        __syncthreads();
        for (long long i = threadIdx.x; i < base; i += kRsThreads) atomicAdd(&h[(int)((kin[i] >> shift) & 255)], 1u);
        __syncthreads();
        before = h[d0];
        __syncthreads();
    }
    store_word(word, (before + own) | kAll | tag << 58);
    gofs[d0] = (long long)gbase + (long long)before - (long long)toff[d0];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
        if ((w * ITEMS + i) * 32 + lane < cnt) {
            const int d = (int)((key[i] >> shift) & 255);
            const unsigned at = toff[d] + wc[w][d] + rank[i];
            s_key[at] = key[i];
            if (VALS) s_val[at] = val[i];
        }
    }
    __syncthreads();
    const K mask = xb >= (int)(8 * sizeof(K)) ? ~(K)0 : (K)(((K)1 << xb) - 1);
    for (int j = threadIdx.x; j < cnt; j += kRsThreads) {
        const K k = s_key[j];
        const long long at = gofs[(int)((k >> shift) & 255)] + j;
        if (list) list[at] = make_int2((int)(unsigned)(k & mask), (int)(k >> xb));
        else kout[at] = k;
        if (VALS) vout[at] = s_val[j];
    }
}

template <class K, bool VALS>
int passes_of(K* keys, int* vals, K* keys_alt, int* vals_alt, long long n, const RsTmp& T, int begin_bit, int passes,
              int2* list, int xb, cudaStream_t s) {
    const bool lng = !VALS && sizeof(K) == 4 && n > kRsLong;
    const long long tile = (long long)kRsThreads * (lng ? kRsItemsLong : kRsItems);
    const unsigned tiles = (unsigned)((n + tile - 1) / tile);
    auto kern = k_rs_pass<K, VALS, kRsItems>;
    if constexpr (!VALS && sizeof(K) == 4)
        if (lng) kern = k_rs_pass<K, VALS, kRsItemsLong>;
    K *ka = keys, *kb = keys_alt;
    int *va = vals, *vb = vals_alt;
    for (int p = 0; p < passes; ++p) {
        kern<<<tiles, kRsThreads, 0, s>>>(ka, va, kb, vb, n, begin_bit + 8 * p, p, T.st, T.hist,
                                                        T.ticket, p == passes - 1 ? list : nullptr, xb);
        note_launch();
        std::swap(ka, kb);
        std::swap(va, vb);
    }
    return passes & 1;
}

// ---------------------------------------------------------------- sort in one cluster
// All passes of a short array in one cluster of eight blocks: the items stay in registers and shared
// memory, a pass exchanges the blocks' digit counts and then the items through distributed shared memory.
// lin != nullptr: the items are pairs, packed and unpacked as above; else kin (and vin).  Every index of
// kClBlocks * 1024 * ITEMS is held; those from n on have all bits set and stay last (the order is stable).
// What bounds it: the chain of a pass (ranking, two cluster barriers): 1e4 keys with values, eight passes,
// 44 us (as launches 68 and the histogram), lists of 5.3e4, 1.2e4 and 6e3 pairs, three passes, 31, 15 and 12 us
// (33, 27 and 27); calls of 1e4 particles 1.26 -> 1.21 ms, of 2000 without allocations 1.16 -> 1.07.  The lines:
// 6.1e4 keys with values 129 us in the cluster and 78 as launches, 5.3e4 pairs as above.
constexpr int kClBlocks = 8, kClThreads = 1024;
constexpr long long kClMax = (long long)kClBlocks * kClThreads * 8, kClMaxVals = kClMax / 2;
template <class K, bool VALS, int ITEMS>
__global__ void __launch_bounds__(kClThreads) k_sort_cluster(const int2* lin, const K* kin, const int* vin, int n,
                                                             int begin_bit, int passes, int xb, int2* lout, K* kout,
                                                             int* vout) {
    constexpr int kHold = kClThreads * ITEMS;  // items of a block (a power of two)
    extern __shared__ __align__(16) unsigned char csm[];
    K* buf = (K*)csm;
    int* vbuf = (int*)(buf + kHold);
    __shared__ unsigned wc[32][256], part[4][256], tot[256], at[256], sw[8];
    const cg::cluster_group cl = cg::this_cluster();
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, b = (int)blockIdx.x, d0 = t & 255, q = t >> 8;
    const int local = w * ITEMS * 32 + lane;  // the thread's items: local + 32 i
    K key[ITEMS];
    int val[VALS ? ITEMS : 1];
    unsigned rank[ITEMS];
    for (int p = 0; p < passes; ++p) {
        const int shift = begin_bit + 8 * p;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int j = local + 32 * i;
            if (p) {
                key[i] = buf[j];
                if (VALS) val[i] = vbuf[j];
            } else {
                const int g = b * kHold + j;
                key[i] = ~(K)0;
                if (VALS) val[i] = 0;
                if (g < n) {
                    if (lin) {
                        const int2 v = lin[g];
                        key[i] = (K)(((u64)(unsigned)v.y << xb) | (u64)(unsigned)v.x);
                    } else {
                        key[i] = kin[g];
                        if (VALS) val[i] = vin[g];
                    }
                }
            }
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) wc[8 * q + k][d0] = 0;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int d = (int)((key[i] >> shift) & 255);
            unsigned peers = 0xffffffffu;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const unsigned on = (d >> k) & 1 ? 0xffffffffu : 0u;
                peers &= ~(on ^ __ballot_sync(0xffffffffu, on != 0u));
            }
            const unsigned c = wc[w][d];
            rank[i] = c + __popc(peers & ((1u << lane) - 1u));
            __syncwarp();
            if (lane == __ffs(peers) - 1) wc[w][d] = c + __popc(peers);
            __syncwarp();
        }
        __syncthreads();
        // digit d0: the warps' offsets (8 warps per thread) and the block's count
        unsigned own = 0;
        unsigned c8[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            c8[k] = own;
            own += wc[8 * q + k][d0];
        }
        part[q][d0] = own;
        __syncthreads();
        unsigned off = 0;
        for (int k = 0; k < q; ++k) off += part[k][d0];
#pragma unroll
        for (int k = 0; k < 8; ++k) wc[8 * q + k][d0] = off + c8[k];
        if (q == 3) tot[d0] = off + own;
        cl.sync();  // all counts are there, and every block's items are in registers
        unsigned x = 0, before = 0, all = 0;
        if (t < 256) {
            for (int r = 0; r < kClBlocks; ++r) {
                const unsigned v = *cl.map_shared_rank(tot + d0, r);
                if (r < b) before += v;
                all += v;
            }
            x = all;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) sw[w] = x;
        }
        __syncthreads();
        if (t < 256) {
            for (int k = 0; k < w; ++k) x += sw[k];
            at[d0] = x - all + before;
        }
        __syncthreads();
        const bool last = p == passes - 1;
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
            const int d = (int)((key[i] >> shift) & 255);
            const unsigned pos = at[d] + wc[w][d] + rank[i];
            if (!last) {
                const int r = (int)(pos / kHold), j = (int)(pos % kHold);
                *cl.map_shared_rank(buf + j, r) = key[i];
                if (VALS) *cl.map_shared_rank(vbuf + j, r) = val[i];
            } else if (pos < (unsigned)n) {
                if (lout) {
                    const K mask = xb >= (int)(8 * sizeof(K)) ? ~(K)0 : (K)(((K)1 << xb) - 1);
                    lout[pos] = make_int2((int)(unsigned)(key[i] & mask), (int)(key[i] >> xb));
                } else {
                    kout[pos] = key[i];
                    if (VALS) vout[pos] = val[i];
                }
            }
        }
        cl.sync();  // the items of the next pass are there; the counts have been read
    }
}
template <class K, bool VALS, int ITEMS>
void go_cluster(int2* list, const K* kin, const int* vin, int n, int begin_bit, int passes, int xb, K* kout, int* vout,
                cudaStream_t s) {
    const size_t sm = (size_t)kClThreads * ITEMS * (sizeof(K) + (VALS ? sizeof(int) : 0));
    auto kern = k_sort_cluster<K, VALS, ITEMS>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    launch_cluster8(kern, kClBlocks, kClThreads, sm, s, (const int2*)list, kin, vin, n, begin_bit, passes, xb, list,
                    kout, vout);
    note_launch();
}
// n <= kClMax (with values kClMaxVals); pairs in place in list, or kin, vin to kout, vout (which may be the same arrays)
template <class K, bool VALS>
void sort_cluster(int2* list, const K* kin, const int* vin, int n, int begin_bit, int passes, int xb, K* kout,
                  int* vout, cudaStream_t s) {
    const int per = kClBlocks * kClThreads;
    if (n <= per) go_cluster<K, VALS, 1>(list, kin, vin, n, begin_bit, passes, xb, kout, vout, s);
    else if (n <= 2 * per) go_cluster<K, VALS, 2>(list, kin, vin, n, begin_bit, passes, xb, kout, vout, s);
    else if (n <= 4 * per) go_cluster<K, VALS, 4>(list, kin, vin, n, begin_bit, passes, xb, kout, vout, s);
    else if constexpr (!VALS) go_cluster<K, VALS, 8>(list, kin, vin, n, begin_bit, passes, xb, kout, vout, s);
}

int bits_for(long long v) {
    int b = 1;
    while ((1LL << b) < v) ++b;
    return b;
}
}  // namespace

size_t radix_tmp_ints(long long n) {
    const size_t tiles = (size_t)((n + kRsTile - 1) / kRsTile) + 1;
    return tiles * 512 + kRsMaxPasses * 257 + 2;
}

int radix_sort_pairs_bits(uint64_t* keys, int* idx, uint64_t* keys_alt, int* idx_alt, long long n, int* tmp,
                          int begin_bit, int end_bit, cudaStream_t s) {
    if (n <= 1) return 0;
    const int passes = (end_bit - begin_bit + 7) / 8;
    u64 *ka = (u64*)keys, *kb = (u64*)keys_alt;
    if (n <= (idx ? kClMaxVals : kClMax)) {
        u64* out = passes & 1 ? kb : ka;
        if (idx)
            sort_cluster<u64, true>(nullptr, ka, idx, (int)n, begin_bit, passes, 64, out, passes & 1 ? idx_alt : idx, s);
        else
            sort_cluster<u64, false>(nullptr, ka, nullptr, (int)n, begin_bit, passes, 64, out, nullptr, s);
        return passes & 1;
    }
    const RsTmp T(tmp, n);
    cudaMemsetAsync(T.st, 0, T.bytes, s);
    k_rs_hist<u64><<<grid_for(n, 256 * kRsItems, 4), 256, 0, s>>>(ka, n, begin_bit, passes, T.hist);
    note_launch();
    return idx ? passes_of<u64, true>(ka, idx, kb, idx_alt, n, T, begin_bit, passes, nullptr, 64, s)
               : passes_of<u64, false>(ka, nullptr, kb, nullptr, n, T, begin_bit, passes, nullptr, 64, s);
}

void radix_sort_pairs(uint64_t* keys, int* idx, uint64_t* keys_alt, int* idx_alt, int n, int* tmp,
                      cudaStream_t s) {
    // 8 passes over the 63 key bits: the result is back in (keys, idx)
    radix_sort_pairs_bits(keys, idx, keys_alt, idx_alt, n, tmp, 0, 64, s);
}

// ---------------------------------------------------------------- list sort
// bits of a key below the sink's, and all of them
static int list_key_bits(int ncells, bool wide, int& xb) {
    const int sb = bits_for(ncells);
    xb = wide ? 32 : sb;
    return xb + sb;
}
size_t list_sort_tmp_bytes(long long npairs, int ncells, bool wide) {
    const size_t n = (size_t)(npairs > 0 ? npairs : 1);
    int xb;
    const size_t key = list_key_bits(ncells, wide, xb) <= 32 ? sizeof(unsigned) : sizeof(u64);
    return n * 2 * key + radix_tmp_ints((long long)n) * sizeof(int) + 256;
}

// LSD passes over the keys alone (8 bits per pass over the xb + sb bits in use; 32-bit keys where they
// hold them), the last one writing pairs
template <class K>
static void sort_list(int2* list, long long npairs, int xb, int bits, void* tmp, cudaStream_t s) {
    const int passes = (bits + 7) / 8;
    if (npairs <= kClMax) {
        sort_cluster<K, false>(list, nullptr, nullptr, (int)npairs, 0, passes, xb, nullptr, nullptr, s);
        return;
    }
    K* k0 = (K*)tmp;
    K* k1 = k0 + npairs;
    const RsTmp T(k1 + npairs, npairs);
    cudaMemsetAsync(T.st, 0, T.bytes, s);
    k_rs_pack<K><<<grid_for(npairs, 256 * kRsItems, 4), 256, 0, s>>>(list, npairs, xb, passes, k0, T.hist);
    note_launch();
    passes_of<K, false>(k0, nullptr, k1, nullptr, npairs, T, 0, passes, list, xb, s);
}
void sort_pairs_by_sink(int2* list, long long npairs, int ncells, void* tmp, cudaStream_t s, bool wide) {
    if (npairs <= 1) return;
    int xb;
    const int bits = list_key_bits(ncells, wide, xb);
    if (bits <= 32) sort_list<unsigned>(list, npairs, xb, bits, tmp, s);
    else sort_list<u64>(list, npairs, xb, bits, tmp, s);
}

}  // namespace gb3
