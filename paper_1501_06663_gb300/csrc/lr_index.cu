// Suffix array, rank and lcp arrays on the device: the step before the
// longest-repeat query.  The paper builds them on the host and notes that
// they can be built in parallel on a GPU by prefix doubling (Sec. 4, citing
// Osipov 2012 and Deo and Keely 2013); this is a prefix-doubling build, for
// one string or for many strings packed back to back (string j owns
// positions [off[j], off[j+1])) in one pass.
//
//  * round 0: every suffix gets a key of its string index (most significant)
//    and its first c symbols, each in the bits its dense code needs (the
//    symbols that occur numbered 1 .. sigma, 0 past the end of its string;
//    c = 21 for DNA, 9 for 96 symbols, 7 for all 256, fewer when the string
//    index needs bits);
//    the keys are sorted with their positions (radix sort) and each
//    position's rank becomes the sorted index of the first key equal to its
//    own (a max-scan over group heads).  Strings occupy consecutive rank
//    ranges, [off[j], off[j+1]) for string j;
//  * round r >= 1, h = c * 2^(r-1): key(i) = (rank(i), rank(i + h) + 1, or 0
//    past the end of i's string), for the suffixes still in groups of two or
//    more only (the others keep their ranks), sorted again; ranks are equal
//    iff the strings and the first c * 2^r symbols are; a re-sorted suffix
//    takes the rank of its old group's start plus the offset of its new
//    group inside the old one;
//  * rounds stop when all ranks differ; the suffix array is kept from the
//    first sort on: a re-sorted group's members move only within its range
//    (flattened index g holds the suffix of local rank g - off[j]);
//  * lcp of each pair of sa neighbours: pairs with different round-0 keys
//    have it from the keys; of the others the round at which they parted
//    gives it within a factor of two (first c * 2^(r-1) symbols equal, fewer
//    than c * 2^r), binary lifting over the ranks of the earlier rounds
//    (equal ranks at round q mean c * 2^q equal symbols) and fewer than c
//    symbol comparisons give the rest.
//
// What bounds it: the radix sorts (CUB; two thirds of the time), then the
// scattered rank stores and the lookups of k_lcp.  2^25 + 1 positions of
// English take 7.3 ms and 2^28 70 ms; 10.5 and 89.7 ms with the suffix array
// sorted once more from the final ranks, round 0's ranks sorted back to
// position order at any size, separate marks, max-scans and updates, the
// actives selected from all positions every round, keys of 32 + 26 instead of
// 26 + 26 bits, and a thread per position coding all its symbols.
#include <cuda_runtime.h>
#include <cub/cub.cuh>
#include <thrust/iterator/counting_iterator.h>
#include <cstdint>
#include "lr_internal.h"

namespace lr {

namespace {

// The string holding flattened position g: the last j with off[j] <= g.
__device__ __forceinline__ long long string_of(const int64_t* __restrict__ off, long long num, long long g) {
    long long lo = 0, hi = num - 1;
    while (lo < hi) {
        const long long mid = (lo + hi + 1) >> 1;
        if (__ldg(off + mid) <= g) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The symbols that occur: seen[c] = 1 for every byte value c of the text.
__global__ void k_seen(const uint8_t* __restrict__ text, long long total, uint8_t* __restrict__ seen) {
    __shared__ uint8_t s[256];
    for (int t = threadIdx.x; t < 256; t += blockDim.x) s[t] = 0;
    __syncthreads();
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x)
        s[__ldg(text + i)] = 1;
    __syncthreads();
    for (int t = threadIdx.x; t < 256; t += blockDim.x)
        if (s[t]) seen[t] = 1;
}

// Dense codes 1 .. sigma of the symbols that occur (0: past the end of a
// string), bps bits each.
struct SymCodes {
    uint16_t code[256];
};

// Round-0 keys: a block's symbols are coded once into shared memory, a thread
// rolls the keys of eight consecutive positions out of them (one symbol in,
// one shifted out), and the keys leave through shared memory in order.  With
// one thread per position reading and coding all its symbols itself 2^25
// positions of English took 386 us.
constexpr int kKeyThreads = 256, kKeyPer = 8, kKeyTile = kKeyThreads * kKeyPer;
constexpr int kMaxSyms = 63;                             // one bit per symbol at least
constexpr int kKeySteps = 4;                             // strings a thread steps over before it searches
__global__ void __launch_bounds__(kKeyThreads)
k_keys0(const uint8_t* __restrict__ text, long long total, const int64_t* __restrict__ off, long long num, int csyms,
        int bps, SymCodes codes, uint64_t* __restrict__ key, int32_t* __restrict__ val, int32_t* __restrict__ end) {
    __shared__ uint16_t sc[256];
    __shared__ __align__(16) uint16_t cd[kKeyTile + ((kMaxSyms + 7) & ~7) + 8];
    __shared__ uint64_t out[kKeyTile + kKeyTile / kKeyPer];   // one word of padding per thread's keys
    const int tid = threadIdx.x;
    for (int t = tid; t < 256; t += kKeyThreads) sc[t] = codes.code[t];
    __syncthreads();
    const long long g0 = (long long)blockIdx.x * kKeyTile;
    const int need = kKeyTile + ((csyms + 7) & ~7) + 8;
    for (int t = tid; t < need; t += kKeyThreads) cd[t] = g0 + t < total ? sc[__ldg(text + g0 + t)] : (uint16_t)0;
    __syncthreads();
    const long long i = g0 + (long long)tid * kKeyPer;
    const int kbits = csyms * bps;
    const uint64_t mask = (1ull << kbits) - 1;           // kbits <= 63
    if (i < total) {
        long long j = string_of(off, num, i), e = __ldg(off + j + 1);
        uint64_t* o = out + tid * (kKeyPer + 1);
        if (num == 1 || i + kKeyPer + csyms <= e) {      // (past the end of the text the codes are 0)
            const uint64_t top = (uint64_t)j << kbits;
            uint64_t k = 0;
            for (int t0 = 0; t0 < csyms + kKeyPer - 1; t0 += 8) {
                const uint4 w = *reinterpret_cast<const uint4*>(cd + tid * kKeyPer + t0);
                const uint32_t c[8] = {w.x & 0xffffu, w.x >> 16, w.y & 0xffffu, w.y >> 16,
                                       w.z & 0xffffu, w.z >> 16, w.w & 0xffffu, w.w >> 16};
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    k = ((k << bps) | c[u]) & mask;
                    const int q = t0 + u - (csyms - 1);  // the symbol completes the key of position i + q
                    if (q >= 0 && q < kKeyPer) o[q] = top | k;
                }
            }
            if (end)
                for (int q = 0; q < kKeyPer; ++q)
                    if (i + q < total) end[i + q] = (int32_t)e;
        } else {
            // across strings: each position by itself; past a few empty
            // strings the next one is looked up (2^18 of them between two
            // strings of 50 000 positions: 17.3 ms walked, 0.30 searched)
            for (int q = 0; q < kKeyPer && i + q < total; ++q) {
                for (int t = 0; t < kKeySteps && i + q >= e; ++t) { ++j; e = __ldg(off + j + 1); }
                if (i + q >= e) { j = string_of(off, num, i + q); e = __ldg(off + j + 1); }
                uint64_t k = (uint64_t)j;
                for (int t = 0; t < csyms; ++t) k = (k << bps) | (i + q + t < e ? (uint64_t)cd[tid * kKeyPer + q + t] : 0ull);
                o[q] = k;
                if (end) end[i + q] = (int32_t)e;
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kKeyPer; ++u) {
        const int x = u * kKeyThreads + tid;
        if (g0 + x < total) {
            key[g0 + x] = out[x + x / kKeyPer];
            val[g0 + x] = (int32_t)(g0 + x);
        }
    }
}

// A rank word holds the rank in bits 0..30 and, in bit 31, whether the
// position is still in a group of two or more (then every member of its
// group is, so equal words still mean equal groups).
constexpr uint32_t kActiveBit = 0x80000000u;
constexpr uint32_t kRankMask = 0x7fffffffu;

// Round r >= 1 keys of the suffixes still in groups of two or more (act[0..A),
// ascending positions): (rank(i), rank(i + h) + 1, or 0 past the end of i's
// string).
// `end` (null for one string: `total`) holds the ends of the positions'
// strings; the halves take sb bits each.
__global__ void k_keys_act(const int32_t* __restrict__ act, long long A, const int32_t* __restrict__ rank,
                           long long h, const int32_t* __restrict__ end, long long total, int sb,
                           uint64_t* __restrict__ key, int32_t* __restrict__ val) {
    const long long a = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (a >= A) return;
    const long long i = __ldg(act + a);
    const long long e = end ? (long long)__ldg(end + i) : total;
    const uint32_t second = (i + h < e) ? ((uint32_t)__ldg(rank + i + h) & kRankMask) + 1u : 0u;
    key[a] = ((uint64_t)((uint32_t)__ldg(rank + i) & kRankMask) << sb) | second;
    val[a] = (int32_t)i;
}

// Selects position i when its rank word carries the active bit.
struct ActiveAt {
    const int32_t* rank;
    __device__ __forceinline__ bool operator()(int32_t i) const { return ((uint32_t)__ldg(rank + i) & kActiveBit) != 0; }
};

// Groups of equal sorted keys, a tile of kGrpTile per block: a bitmap of the
// elements that start one, the last start before each of its words, and the
// start of the group that runs into the tile (found from its first element by
// doubling steps back, then halving: a few steps for the usual group).
constexpr int kGrpThreads = 256, kGrpPer = 8, kGrpTile = kGrpThreads * kGrpPer;
struct GroupMap {
    unsigned bits[kGrpTile / 32 + 1];                    // the extra word: bit 0 = the element after the tile
    int32_t last[kGrpTile / 32];                         // last start before the word, -1: before the tile
    long long first;                                     // start of the group of the tile's first element
};

// The start of the run of elements equal (key >> shift) to element g.
__device__ __forceinline__ long long run_start(const uint64_t* __restrict__ key, long long g, int shift) {
    const uint64_t k = __ldg(key + g) >> shift;
    long long step = 1, lo = -1;                         // lo: an element known to differ (or -1)
    while (true) {
        if (g - step < 0) break;
        if ((__ldg(key + g - step) >> shift) != k) { lo = g - step; break; }
        g -= step;
        step *= 2;
    }
    while (g - lo > 1) {                                 // g is equal, lo is not
        const long long mid = lo + (g - lo) / 2;
        if ((__ldg(key + mid) >> shift) == k) g = mid; else lo = mid;
    }
    return g;
}

// One warp: last starts before the words.
__device__ __forceinline__ void group_lasts(GroupMap& m) {
    constexpr int kPer = kGrpTile / 32 / 32;             // 2
    const int lane = threadIdx.x & 31;
    int own[kPer], x = -1;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int w = lane * kPer + u;
        const unsigned b = m.bits[w];
        own[u] = b ? w * 32 + 31 - __clz(b) : -1;
        x = max(x, own[u]);
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x = max(x, y);
    }
    int run = __shfl_up_sync(0xffffffffu, x, 1);
    if (lane == 0) run = -1;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        m.last[lane * kPer + u] = run;
        run = max(run, own[u]);
    }
}

// The start of the group of element x of the tile at t0.
__device__ __forceinline__ long long group_start(const GroupMap& m, long long t0, int x) {
    const unsigned b = m.bits[x >> 5] & ((2u << (x & 31)) - 1u);
    const int at = b ? (x & ~31) + 31 - __clz(b) : m.last[x >> 5];
    return at >= 0 ? t0 + at : m.first;
}

__device__ __forceinline__ bool starts_group(const GroupMap& m, int x) { return (m.bits[x >> 5] >> (x & 31)) & 1u; }

// Round 0, over all sorted keys: the rank word of each suffix (the start of
// its group, with the active bit in groups of two or more) goes to its
// position (kScatter) or stays in sorted order, sa takes the sorted
// positions, sep is 0 where a group starts, and the lcp of neighbours in
// different groups is the number of equal leading symbols of their keys.
template <bool kScatter>
__global__ void __launch_bounds__(kGrpThreads)
k_rank0(const uint64_t* __restrict__ key, const int32_t* __restrict__ val, long long total, int kbits, int bps,
        int32_t* __restrict__ rank, int32_t* __restrict__ sa, uint8_t* __restrict__ sep, int32_t* __restrict__ lcp) {
    __shared__ GroupMap m;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long t0 = (long long)blockIdx.x * kGrpTile;
#pragma unroll
    for (int u = 0; u < kGrpPer; ++u) {
        const int x = u * kGrpThreads + tid;
        const long long g = t0 + x;
        const uint64_t k = g < total ? __ldg(key + g) : 0;
        uint64_t p = __shfl_up_sync(0xffffffffu, k, 1);
        if (lane == 0 && g > 0 && g < total) p = __ldg(key + g - 1);
        const bool head = g < total && (g == 0 || k != p);
        const unsigned b = __ballot_sync(0xffffffffu, head || g >= total);
        if (lane == 0) m.bits[u * (kGrpThreads / 32) + warp] = b;
        if (head) {
            const long long j = (long long)(k >> kbits);
            const bool same = g > 0 && (long long)(p >> kbits) == j;
            lcp[g + j] = same ? __clzll((long long)((k ^ p) << (64 - kbits))) / bps : 0;
        }
        if (g < total) sep[g] = head ? 0 : 0xff;
    }
    if (tid == 0) {
        const long long g = t0 + kGrpTile;
        m.bits[kGrpTile / 32] = g >= total || __ldg(key + g) != __ldg(key + g - 1);
    }
    __syncthreads();
    if (warp == 0) group_lasts(m);
    if (tid == 32) m.first = (m.bits[0] & 1u) ? t0 : run_start(key, t0, 0);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kGrpPer; ++u) {
        const int x = u * kGrpThreads + tid;
        const long long g = t0 + x;
        if (g >= total) break;
        const bool act = !(starts_group(m, x) && starts_group(m, x + 1));
        const int32_t word = (int32_t)((uint32_t)group_start(m, t0, x) | (act ? kActiveBit : 0u));
        const int32_t v = __ldg(val + g);
        if (kScatter) rank[v] = word; else rank[g] = word;
        sa[g] = v;
    }
}

// rank[val[i]] = word[i] for i < count, window by window of 2^kWinPos positions
// (blocks in window order, each reading the pairs once more and storing those
// of its window), so that the stores merge in L2: 2^25 stores into one
// 134 MB array run at 45 G/s, into 64 MB of it at 130.
constexpr int kWinPos = 24;
__global__ void __launch_bounds__(kGrpThreads)
k_scatter_words(const int32_t* __restrict__ val, const int32_t* __restrict__ word, long long count,
                int32_t* __restrict__ rank, unsigned per_window) {
    const int w = (int)(blockIdx.x / per_window);
    const long long i0 = (long long)(blockIdx.x % per_window) * kGrpTile;
    if (i0 + kGrpTile <= count) {
        int4 v[2], x[2];
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const long long i = i0 / 4 + u * kGrpThreads + threadIdx.x;
            v[u] = __ldcs(reinterpret_cast<const int4*>(val) + i);
            x[u] = __ldcs(reinterpret_cast<const int4*>(word) + i);
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            if ((v[u].x >> kWinPos) == w) rank[v[u].x] = x[u].x;
            if ((v[u].y >> kWinPos) == w) rank[v[u].y] = x[u].y;
            if ((v[u].z >> kWinPos) == w) rank[v[u].z] = x[u].z;
            if ((v[u].w >> kWinPos) == w) rank[v[u].w] = x[u].w;
        }
    } else {
        for (long long i = i0 + threadIdx.x; i < count; i += kGrpThreads) {
            const int32_t v = __ldcs(val + i);
            if ((v >> kWinPos) == w) rank[v] = __ldcs(word + i);
        }
    }
}

// Round r >= 1, over the re-sorted keys key[0..A) (halves of sb bits): an old
// group (rank g0 = its first sorted index) holds its re-sorted members at
// a0 .. a0 + size - 1, so member a sits at sorted index g0 + a - a0 and its
// new rank is the index of its new group's first member, g0 + ah - a0, with
// the active bit when the new group has two or more members.  New group
// starts inside an old group take sep = r.  The rank words go to their
// positions (kScatter) or stay in key order.
template <bool kScatter>
__global__ void __launch_bounds__(kGrpThreads)
k_update(const uint64_t* __restrict__ key, const int32_t* __restrict__ val, long long A, int sb,
         int32_t* __restrict__ rank, int32_t* __restrict__ sa, uint8_t* __restrict__ sep, int round) {
    __shared__ GroupMap nm, om;                          // new and old groups
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const long long t0 = (long long)blockIdx.x * kGrpTile;
    uint32_t old[kGrpPer];
#pragma unroll
    for (int u = 0; u < kGrpPer; ++u) {
        const long long a = t0 + u * kGrpThreads + tid;
        const uint64_t k = a < A ? __ldg(key + a) : 0;
        uint64_t p = __shfl_up_sync(0xffffffffu, k, 1);
        if (lane == 0 && a > 0 && a < A) p = __ldg(key + a - 1);
        const bool nh = a >= A || a == 0 || k != p, oh = a >= A || a == 0 || (k >> sb) != (p >> sb);
        const unsigned nb = __ballot_sync(0xffffffffu, nh), ob = __ballot_sync(0xffffffffu, oh);
        if (lane == 0) {
            nm.bits[u * (kGrpThreads / 32) + warp] = nb;
            om.bits[u * (kGrpThreads / 32) + warp] = ob;
        }
        old[u] = (uint32_t)(k >> sb);
    }
    if (tid == 0) {
        const long long a = t0 + kGrpTile;
        nm.bits[kGrpTile / 32] = a >= A || __ldg(key + a) != __ldg(key + a - 1);
    }
    __syncthreads();
    if (warp == 0) group_lasts(nm);
    if (warp == 1) group_lasts(om);
    if (tid == 64) nm.first = (nm.bits[0] & 1u) ? t0 : run_start(key, t0, 0);
    if (tid == 96) om.first = (om.bits[0] & 1u) ? t0 : run_start(key, t0, sb);
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kGrpPer; ++u) {
        const int x = u * kGrpThreads + tid;
        const long long a = t0 + x;
        if (a >= A) break;
        const long long g0 = old[u], s0 = group_start(om, t0, x), hh = group_start(nm, t0, x);
        const bool nh = starts_group(nm, x), act = !(nh && starts_group(nm, x + 1));
        const int32_t v = __ldg(val + a);
        const int32_t word = (int32_t)((uint32_t)(g0 + (hh - s0)) | (act ? kActiveBit : 0u));
        if (kScatter) rank[v] = word; else rank[a] = word;
        sa[g0 + (a - s0)] = v;
        if (nh && s0 != a) sep[g0 + (a - s0)] = (uint8_t)round;
    }
}

// String-local suffix array of a batch: index g lies in string j's range.
__global__ void k_local_sa(int32_t* __restrict__ sa, long long total, const int64_t* __restrict__ off, long long num) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g < total) sa[g] -= (int32_t)__ldg(off + string_of(off, num, g));
}

// lcp of sorted neighbours g - 1, g that share their round-0 key, written in
// the layout the queries take (string j's n_j + 1 entries at off[j] + j), and
// the string-local rank.  The two suffixes parted at round r = sep[g] >= 1
// (k_rank0 wrote the others): their first csyms * 2^(r-1) symbols are equal
// and fewer than csyms * 2^r are; the rest is found by binary
// lifting over the ranks of rounds r - 2 .. 0 (equal ranks at round q mean
// csyms * 2^q more equal symbols, longest first), then fewer than csyms
// symbol comparisons.
__global__ void k_lcp(const uint8_t* __restrict__ text, long long total, const int64_t* __restrict__ off,
                      long long num, const int32_t* __restrict__ sorted, const int32_t* __restrict__ levels,
                      int rounds, int csyms, const uint8_t* __restrict__ sep, const int32_t* __restrict__ frank,
                      int32_t* __restrict__ rank, int32_t* __restrict__ lcp) {
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= total) return;
    const long long j = string_of(off, num, g);
    const long long a = __ldg(off + j), e = __ldg(off + j + 1);
    rank[g] = (int32_t)(frank[g] - a);
    int r = sep[g];
    if (r == 0) return;
    r = r < rounds ? r : rounds - 1;                       // every index parts by the last round
    long long l = (long long)csyms << (r - 1);
    long long x = sorted[g - 1] + l, y = sorted[g] + l;
    for (int q = r - 2; q >= 0; --q) {
        const long long len = (long long)csyms << q;
        const int32_t* R = levels + (size_t)q * (size_t)total;
        if (x < e && y < e && __ldg(R + x) == __ldg(R + y)) { l += len; x += len; y += len; }
    }
    for (int t = 0; t < csyms && x < e && y < e && __ldg(text + x) == __ldg(text + y); ++t) { ++l; ++x; ++y; }
    lcp[g + j] = (int32_t)l;
}

// The closing sentinel lcp[n_j] = 0 of every string (and the only entry of
// an empty one).
__global__ void k_lcp_tails(const int64_t* __restrict__ off, long long num, int32_t* __restrict__ lcp) {
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j < num) lcp[__ldg(off + j + 1) + j] = 0;
}

// Sets *bad unless off[0] = 0, off[num] = total and off never decreases.
__global__ void k_check_off(const int64_t* __restrict__ off, long long num, long long total,
                            unsigned long long* __restrict__ bad) {
    const long long j = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (j > num) return;
    const long long v = __ldg(off + j);
    bool b = v < 0 || v > total || (j == 0 && v != 0) || (j == num && v != total);
    if (j < num && __ldg(off + j + 1) < v) b = true;
    if (b) atomicOr(bad, 1ull);
}

inline unsigned blocks(long long n, int t) { return (unsigned)((n + t - 1) / t); }

size_t sort_temp_bytes(long long n) {
    size_t a = 0, c = 0;
    cub::DoubleBuffer<uint64_t> keys(nullptr, nullptr);
    cub::DoubleBuffer<int32_t> vals(nullptr, nullptr), pos(nullptr, nullptr);
    cub::DeviceRadixSort::SortPairs(nullptr, a, keys, vals, (int)n, 0, 64, (cudaStream_t)0);
    cub::DeviceRadixSort::SortPairs(nullptr, c, pos, vals, (int)n, 0, 32, (cudaStream_t)0);
    size_t d = 0;
    cub::DeviceSelect::If(nullptr, d, thrust::counting_iterator<int32_t>(0), (int32_t*)nullptr,
                          (unsigned long long*)nullptr, (int)n, ActiveAt{nullptr}, (cudaStream_t)0);
    if (d > a) a = d;
    d = 0;
    cub::DeviceSelect::If(nullptr, d, (const int32_t*)nullptr, (int32_t*)nullptr, (unsigned long long*)nullptr, (int)n,
                          ActiveAt{nullptr}, (cudaStream_t)0);
    if (d > a) a = d;
    return (c > a ? c : a) + 256;
}

// Which way rank words go to position order: straight while their array
// (kDirectPos positions) stays in the 129 MB L2, or for few of them; else
// window by window, W windows of 2^kWinPos positions, up to kScatterWins
// (kUpdateWins after round 0); above, round 0's by a radix sort keyed by
// position and later ones straight.  Per word the windows cost 1.2 ps each
// (reading the pairs again) and 8 ps for the stores, the sort 24 ps, stores
// past L2 30 ps.  The build of 2^25 + 1 positions of English takes 7.29 ms
// with windows and 7.85 straight, of 30 M mixed positions 6.52 and 6.32; 10^8
// positions of English 22.0 and (with the sort) 25.0.  Just below the line
// (31 352 422 positions, straight) and on its other side (31 457 281, windows):
// English 7.45 and 6.99, DNA 6.36 and 6.08, protein 5.09 and 4.77, binary 3.47
// and 3.13 ms, so it lies too high for these texts rather than too low.
constexpr long long kDirectPos = 30LL << 20, kDirectWords = 1LL << 18;
constexpr long long kScatterWins = 13, kUpdateWins = 19;

inline size_t al(size_t v) { return (v + 255) & ~(size_t)255; }

}  // namespace

// Layout of the work memory for n positions and `rounds` rank levels.
size_t index_work_bytes(long long n, int rounds) {
    const size_t nn = (size_t)n;
    return al(nn * 8) * 2 + al(nn * 4) * 5 + al(nn) + al((size_t)rounds * nn * 4) + al(64) + al(sort_temp_bytes(n));
}

cudaError_t IndexWork::alloc(long long n, int rounds) {
    release();
    const size_t nn = (size_t)n;
    bytes = index_work_bytes(n, rounds);
    cudaError_t e = cudaMalloc((void**)&base, bytes);
    if (e != cudaSuccess) { cudaGetLastError(); base = nullptr; bytes = 0; return cudaErrorMemoryAllocation; }
    unsigned char* p = base;
    k0 = (uint64_t*)p; p += al(nn * 8);
    k1 = (uint64_t*)p; p += al(nn * 8);
    v0 = (int32_t*)p; p += al(nn * 4);
    v1 = (int32_t*)p; p += al(nn * 4);
    head = (int32_t*)p; p += al(nn * 4);
    hp = (int32_t*)p; p += al(nn * 4);
    end = (int32_t*)p; p += al(nn * 4);
    sep = (uint8_t*)p; p += al(nn);
    levels = (int32_t*)p; p += al((size_t)rounds * nn * 4);
    misc = (unsigned long long*)p; p += al(64);
    tmp = p;
    tmp_bytes = sort_temp_bytes(n);
    cap_n = n;
    cap_rounds = rounds;
    return cudaSuccess;
}

void IndexWork::release() {
    if (base) cudaFree(base);
    base = nullptr;
    bytes = 0;
    cap_n = 0;
    cap_rounds = 0;
}

// Builds sa, rank (string-local, at the strings' offsets) and lcp (n_j + 1
// entries per string at off[j] + j) of text[0..total) split by the device
// offset table off[0..num]; `w` must hold `total` positions.  When more
// rounds are needed than w holds and `grow` is set, w is reallocated (which
// waits for the device); otherwise cudaErrorMemoryAllocation.
cudaError_t build_arrays_batch(const uint8_t* text, long long total, const int64_t* off, long long num, int32_t* sa,
                               int32_t* rank, int32_t* lcp, IndexWork& w, bool grow, cudaStream_t stream,
                               int* rounds_out) {
    if (total > w.cap_n) return cudaErrorMemoryAllocation;
    // every kernel below trusts the offset table: check it first
    cudaError_t e = cudaMemsetAsync(w.misc, 0, 16, stream);
    if (e != cudaSuccess) return e;
    k_check_off<<<blocks(num + 1, 256), 256, 0, stream>>>(off, num, total, w.misc + 1);
    e = cudaMemcpyAsync(&w.groups_host, w.misc + 1, 8, cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return e;
    if (w.groups_host != 0) return cudaErrorInvalidValue;
    k_lcp_tails<<<blocks(num, 256), 256, 0, stream>>>(off, num, lcp);
    if (total == 0) {
        if (rounds_out) *rounds_out = 0;
        return cudaGetLastError();
    }
    const size_t nn = (size_t)total;
    // the alphabet that occurs, coded densely: more symbols per round-0 key
    // for a small alphabet (21 for DNA, 9 for 96 symbols, 7 for all 256)
    uint8_t* seen = reinterpret_cast<uint8_t*>(w.head);
    e = cudaMemsetAsync(seen, 0, 256, stream);
    if (e != cudaSuccess) return e;
    k_seen<<<(unsigned)(total < (1 << 22) ? blocks(total, 256) : 1216), 256, 0, stream>>>(text, total, seen);
    uint8_t seen_h[256];
    e = cudaMemcpyAsync(seen_h, seen, 256, cudaMemcpyDeviceToHost, stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) return e;
    SymCodes codes;
    int sigma = 0;
    for (int c = 0; c < 256; ++c) codes.code[c] = seen_h[c] ? (uint16_t)++sigma : (uint16_t)0;
    int bps = 1;
    while ((1 << bps) <= sigma) ++bps;                     // codes 0 .. sigma
    int jobbits = 0;
    while (jobbits < 40 && (1ll << jobbits) < num) ++jobbits;
    const int csyms = (63 - jobbits) / bps;
    int bits = 1;
    while (bits < 31 && (1ll << bits) <= total) ++bits;
    cub::DoubleBuffer<uint64_t> keys(w.k0, w.k1);
    cub::DoubleBuffer<int32_t> vals(w.v0, w.v1);
    // round 0: every suffix by its string and first csyms symbols
    const bool one = num == 1;
    k_keys0<<<blocks(total, kKeyTile), kKeyThreads, 0, stream>>>(text, total, off, num, csyms, bps, codes, keys.Current(),
                                                                vals.Current(), one ? nullptr : w.end);
    size_t tb = w.tmp_bytes;
    e = cub::DeviceRadixSort::SortPairs(w.tmp, tb, keys, vals, (int)total, 0, jobbits + bps * csyms, stream);
    if (e != cudaSuccess) return e;
    // The suffix array is kept in sa (flattened) from here on
    const long long wins = (total + (1LL << kWinPos) - 1) >> kWinPos;
    auto scatter_words = [&](const int32_t* val, const int32_t* word, long long count, int32_t* rank_out) {
        const unsigned per = blocks(count, kGrpTile);
        k_scatter_words<<<(unsigned)(wins * per), kGrpThreads, 0, stream>>>(val, word, count, rank_out, per);
    };
    const bool direct = total <= kDirectPos;
    if (direct) {
        k_rank0<true><<<blocks(total, kGrpTile), kGrpThreads, 0, stream>>>(keys.Current(), vals.Current(), total,
                                                                          bps * csyms, bps, w.levels, sa, w.sep, lcp);
    } else {
        int32_t* words = wins <= kScatterWins ? reinterpret_cast<int32_t*>(keys.Alternate()) : w.hp;
        k_rank0<false><<<blocks(total, kGrpTile), kGrpThreads, 0, stream>>>(keys.Current(), vals.Current(), total,
                                                                           bps * csyms, bps, words, sa, w.sep, lcp);
        if (wins <= kScatterWins) {
            scatter_words(vals.Current(), words, total, w.levels);
        } else {
            cub::DoubleBuffer<int32_t> pos(vals.Current(), vals.Alternate());
            cub::DoubleBuffer<int32_t> rnk(w.hp, w.levels);
            tb = w.tmp_bytes;
            e = cub::DeviceRadixSort::SortPairs(w.tmp, tb, pos, rnk, (int)total, 0, bits, stream);
            if (e == cudaSuccess && rnk.Current() != w.levels)
                e = cudaMemcpyAsync(w.levels, rnk.Current(), nn * 4, cudaMemcpyDeviceToDevice, stream);
            if (e != cudaSuccess) return e;
        }
    }
    // the active positions, ascending (their rank words are then read in
    // order); only the suffixes in groups of two or more are sorted again
    int32_t *act = w.head, *spare = w.hp;
    tb = w.tmp_bytes;
    e = cub::DeviceSelect::If(w.tmp, tb, thrust::counting_iterator<int32_t>(0), act, w.misc + 2, (int)total,
                              ActiveAt{w.levels}, stream);
    if (e != cudaSuccess) return e;
    int rounds = 1;
    for (int r = 1;; ++r) {
        e = cudaMemcpyAsync(&w.groups_host, w.misc + 2, 8, cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        if (e != cudaSuccess) return e;
        const long long A = (long long)w.groups_host;
        if (A == 0) { rounds = r; break; }
        if (r >= 40 || A > total) return cudaErrorUnknown;
        if (r >= w.cap_rounds) {                          // more rounds than the level store holds
            if (!grow) return cudaErrorMemoryAllocation;
            IndexWork bigger;
            e = bigger.alloc(w.cap_n, w.cap_rounds * 2);
            if (e != cudaSuccess) return e;
            e = cudaMemcpyAsync(bigger.levels, w.levels, (size_t)w.cap_rounds * nn * 4, cudaMemcpyDeviceToDevice,
                                stream);
            if (e == cudaSuccess && !one) e = cudaMemcpyAsync(bigger.end, w.end, nn * 4, cudaMemcpyDeviceToDevice, stream);
            if (e == cudaSuccess) e = cudaMemcpyAsync(bigger.sep, w.sep, nn, cudaMemcpyDeviceToDevice, stream);
            if (e == cudaSuccess) e = cudaMemcpyAsync(bigger.head, act, (size_t)A * 4, cudaMemcpyDeviceToDevice,
                                                      stream);
            if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
            if (e != cudaSuccess) { bigger.release(); return e; }
            w.release();
            w = bigger;
            bigger.base = nullptr;                        // owned by w now
            keys = cub::DoubleBuffer<uint64_t>(w.k0, w.k1);
            vals = cub::DoubleBuffer<int32_t>(w.v0, w.v1);
            act = w.head;
            spare = w.hp;
        }
        const int32_t* prev = w.levels + (size_t)(r - 1) * nn;
        int32_t* level = w.levels + (size_t)r * nn;
        e = cudaMemcpyAsync(level, prev, nn * 4, cudaMemcpyDeviceToDevice, stream);   // settled ranks stay
        if (e != cudaSuccess) return e;
        const long long h = (long long)csyms << (r - 1);
        k_keys_act<<<blocks(A, 256), 256, 0, stream>>>(act, A, prev, h, one ? nullptr : w.end, total, bits,
                                                       keys.Current(), vals.Current());
        tb = w.tmp_bytes;
        e = cub::DeviceRadixSort::SortPairs(w.tmp, tb, keys, vals, (int)A, 0, 2 * bits, stream);
        if (e != cudaSuccess) return e;
        if (direct || A <= kDirectWords || wins > kUpdateWins) {
            k_update<true><<<blocks(A, kGrpTile), kGrpThreads, 0, stream>>>(keys.Current(), vals.Current(), A, bits, level,
                                                                            sa, w.sep, r);
        } else {
            int32_t* words = reinterpret_cast<int32_t*>(keys.Alternate());
            k_update<false><<<blocks(A, kGrpTile), kGrpThreads, 0, stream>>>(keys.Current(), vals.Current(), A, bits, words,
                                                                             sa, w.sep, r);
            scatter_words(vals.Current(), words, A, level);
        }
        tb = w.tmp_bytes;
        e = cub::DeviceSelect::If(w.tmp, tb, (const int32_t*)act, spare, w.misc + 2, (int)A, ActiveAt{level}, stream);
        if (e != cudaSuccess) return e;
        int32_t* t = act;
        act = spare;
        spare = t;
    }
    k_lcp<<<blocks(total, 256), 256, 0, stream>>>(text, total, off, num, sa, w.levels, rounds, csyms, w.sep,
                                                  w.levels + (size_t)(rounds - 1) * nn, rank, lcp);
    if (!one) k_local_sa<<<blocks(total, 256), 256, 0, stream>>>(sa, total, off, num);
    if (rounds_out) *rounds_out = rounds;
    return cudaGetLastError();
}

}  // namespace lr
