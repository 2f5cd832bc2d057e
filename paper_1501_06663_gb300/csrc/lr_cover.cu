// The cover kernel of the longest-repeat query (Tian and Xu, arXiv
// 1501.06663, Algorithms 2 and 4, GPU kernel of Sec. 4.2.2): from the compact
// LLR array LLRc to the longest repeats of every position.
//
// Starts and ends of LLRc strictly increase (Sec. 3.2), so the compact LLR's
// covering a position k form a contiguous window of LLRc, and entry v is a
// longest one (a holder) exactly at the positions
//     [max(s_v, e_PG + 1), min(e_v, s_NG - 1)],
// PG / NG its nearest strictly longer neighbours in LLRc.  The set of holders
// therefore changes only where such an interval begins or ends, and the
// kernel works per entry (0.2 to 0.75 of them per position on the texts
// measured), not per position.  Per tile of 2048, 4096 or 8192 positions
// (tiles in order by an atomic ticket):
//
//  * the entries that reach the tile, LLRc[lo, cb1), are staged in shared
//    memory: the tile's own [cb0, cb1) plus the carry before them;
//  * one thread per entry looks left and right over the overlapping entries
//    for PG and NG, counting those of its own length on the way: this gives
//    the interval, the holders where it begins and the holders left where it
//    ends, and so a record (leftmost holder, number of holders) for every
//    position where the set of holders changes, and the tile's number of
//    LR starts, which is published for the look-back at once (the leftmost
//    query needs no counts and stops at the first entry as long);
//  * a position finds its record by one bit scan over a bitmap of those
//    positions: longest length and leftmost start are the holder's
//    (Algorithm 2), the tie count is in the record;
//  * for the all-LR query the tie counts are scanned into CSR offsets
//    (byte prefixes of eight positions per lane, or ballots per run of 32
//    where a count exceeds 15, the tile is cut off or offsets[] is not aligned
//    to 32 bytes; warp totals; decoupled look-back over the tiles), and every
//    holder's start is written, ascending, by following the links to the next
//    entry of the same length (Algorithm 4's second walk).
//
// A tile whose carry is longer than kSpec entries (more than kSpec compact
// LLR's over one position) walks LLRc in place instead (cover_long_carry).
//
// A lane owns one position of each run of 32 for lengths and leftmost starts
// (a warp stores 128 contiguous bytes) and eight consecutive ones for offsets
// (two whole sectors each).
//
// What bounds it: instruction issue (71 to 79 % of the slots) and the waits
// between its phases, of which the look-back is the longest; DRAM runs at
// half its rate.  The form before it worked per position (a range-maximum
// table over the window of each run of 32) and took 2.18 ms for 2^28
// positions of English (0.21 entries per position), 2.77 ms for 258 M of
// mixed DNA and protein (0.52); this one takes 1.55 and 2.31 ms.  It has 166
// instead of 240 instructions per run of 32 positions (English); per-entry
// work pays as long as entries are fewer than positions, which they are by
// construction (at most one starts at each).  Four consecutive positions per
// lane with vector stores were slower (1.69 against 1.58 ms then).  Persistent
// CTAs that take the next ticket early were slower (2.24 ms): a tile taken
// early publishes late, and every later tile waits for it; so were look-back
// steps over 128 or 256 words (1.88, 2.12 ms).
#include <cuda_runtime.h>
#include <cstdint>
#include "lr_device.cuh"
#include "lr_internal.h"

namespace lr {

namespace {

constexpr int32_t kSpec = 64;                     // carry entries staged with the tile's own

// Shape of a cover tile of kTile x TP positions run by kThreads x TP threads;
// every warp owns 8 consecutive runs of 32 positions.  kMinBlocks fills all
// warp slots of an SM in every shape (27.5 KB of shared memory per 2048
// positions, 32 registers; 6 instead of 8 CTAs with 40 registers: 3 % slower).
template <int TP>
struct Cfg {
    static constexpr int kTileC = kTile * TP;
    static constexpr int kThr = kThreads * TP;
    static constexpr int kWarps = kThr / kWarp;
    static constexpr int kChunks = kTileC / kWarp;
    static constexpr int kChunksPerWarp = kChunks / kWarps;
    static constexpr int kMinBlocks = TP == 1 ? 8 : (TP == 2 ? 4 : 2);
    static constexpr int kCap = kTileC + kSpec;   // the tile's own entries and the carry always fit
    static_assert(kCap + 2 < (1 << 16), "record indices must fit 16 bits");
};

template <int TP>
struct __align__(16) CoverSmem {
    static constexpr int kChunks = Cfg<TP>::kChunks;
    // Staged entry i at ent[i + 1]: start, length.  ent[0] has length 0 and
    // start -1: it stops the scans to the left and is the "no holder" entry;
    // the one after the last starts after everything and stops the scans to
    // the right.
    int2 ent[Cfg<TP>::kCap + 2];
    alignas(16) uint32_t rec[Cfg<TP>::kTileC];   // at a boundary: ent index of the leftmost holder | number of holders << 16
    unsigned bmap[kChunks];          // bit x: the set of holders changes at position x (bit 0 always set)
    // distance to the next entry of the same length with no longer one
    // between (0: none that overlaps; 255: that or more)
    static constexpr int kNxWords = (Cfg<TP>::kCap + 2 + 3) / 4;
    uint32_t nx[kNxWords];
    int32_t wtot[Cfg<TP>::kWarps];   // tie counts per warp
    long long tile;
    long long obase;
    int32_t lo;
    int32_t nlow;                    // staged carry candidates that end before the tile
    int32_t ttot;                    // the tile's total of tie counts
    int32_t far;                     // a distance does not fit nx
};

// The words cover_long_carry keeps in place of the staged entries.
template <int TP>
struct LongSmem {
    static constexpr int kChunks = Cfg<TP>::kChunks;
    unsigned smap[kChunks];          // bit x: an entry starts at k0 + x
    unsigned emap[kChunks];          // bit x: an entry ends at k0 + x
    int32_t spre[kChunks];           // exclusive prefix popcounts of the bitmap words
    int32_t epre[kChunks];
    int32_t chunk[kChunks];          // run totals of the tie counts
};

// Exclusive prefix popcounts of the kChunks bitmap words, by one warp.
template <int kChunks>
__device__ __forceinline__ void popc_prefix(const unsigned* map, int32_t* pre) {
    constexpr int kPer = kChunks / kWarp;
    const int lane = lane_id();
    int c[kPer], sum = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) { c[i] = __popc(map[kPer * lane + i]); sum += c[i]; }
    int run = warp_incl_scan(sum) - sum;
#pragma unroll
    for (int i = 0; i < kPer; ++i) { pre[kPer * lane + i] = run; run += c[i]; }
}

// Exclusive scan of the kChunks ints of a[] by one warp; returns the total.
template <int kChunks>
__device__ __forceinline__ int scan_chunks(int32_t* a) {
    constexpr int kPer = kChunks / kWarp;
    const int lane = lane_id();
    int c[kPer], sum = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) { c[i] = a[kPer * lane + i]; sum += c[i]; }
    const int incl = warp_incl_scan(sum);
    int run = incl - sum;
#pragma unroll
    for (int i = 0; i < kPer; ++i) { a[kPer * lane + i] = run; run += c[i]; }
    return __shfl_sync(kFull, incl, kWarp - 1);
}

// Exclusive prefix of the tie counts c of a warp's 32 positions; *tot their
// sum.  Counts are almost always below 4: two ballots over their bit planes.
__device__ __forceinline__ int ties_prefix(int c, unsigned below, int* tot) {
    if (__ballot_sync(kFull, c > 3) == 0u) {
        const unsigned b0 = __ballot_sync(kFull, c & 1), b1 = __ballot_sync(kFull, c & 2);
        *tot = __popc(b0) + 2 * __popc(b1);
        return __popc(b0 & below) + 2 * __popc(b1 & below);
    }
    const int incl = warp_incl_scan(c);
    *tot = __shfl_sync(kFull, incl, kWarp - 1);
    return incl - c;
}

// Four consecutive CSR offsets at a 32-byte-aligned address: a whole sector.
__device__ __forceinline__ void store_offsets(int64_t* p, long long a, long long b, long long c, long long d) {
    asm volatile("st.global.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(p), "l"(a), "l"(b), "l"(c), "l"(d) : "memory");
}

// The tile's place in starts[] (whole warp): look back over the earlier
// tiles, publish the inclusive prefix, write offsets[n] from the last tile.
__device__ __forceinline__ long long place_tile(const Scratch& s, long long tile, long long ntiles, int32_t n, int tot,
                                                int64_t* __restrict__ offsets) {
    const long long ex = (tile == 0) ? 0 : lookback(s.status_o, tile, s.err, s.spin_limit);
    if (lane_id() == 0) {
        if (tile != 0 && tile != s.hold_tile) publish(s.status_o, tile, kPrefix, ex + tot);
        if (tile == ntiles - 1) {
            offsets[n] = ex + tot;
            if (s.total_out) *s.total_out = ex + tot;
        }
    }
    return ex;
}

// A tile with a carry too long to stage: the window of each position from
// bitmaps of starts and ends (popcounts), its entries walked in LLRc.
// Called by the whole CTA.
template <bool kAll, int TP>
__device__ __noinline__ void cover_long_carry(CoverSmem<TP>& sm, int32_t n, const Scratch& s, long long tile, int32_t cb0,
                                              int32_t cb1, int32_t* __restrict__ lr_len, int32_t* __restrict__ lr_start,
                                              int64_t* __restrict__ offsets, int32_t* __restrict__ starts,
                                              long long capacity) {
    constexpr int kCoverTile = Cfg<TP>::kTileC, kCoverThreads = Cfg<TP>::kThr;
    constexpr int kChunks = Cfg<TP>::kChunks, kChunksPerWarp = Cfg<TP>::kChunksPerWarp;
    static_assert(sizeof(LongSmem<TP>) <= sizeof(sm.ent), "the bitmaps replace the staged entries");
    LongSmem<TP>& lm = *reinterpret_cast<LongSmem<TP>*>(sm.ent);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int32_t k0 = (int32_t)(tile * kCoverTile);
    if (tid < kChunks) { lm.smap[tid] = 0; lm.emap[tid] = 0; }
    if (warp == 0) {                                  // the first entry that reaches the tile (ends increase)
        int32_t t = cb0;
        while (t > 0) {
            const int32_t idx = t - 1 - lane;
            const bool reach = idx >= 0 && s.cend[idx] >= k0;
            const unsigned m = __ballot_sync(kFull, reach);
            if (m == kFull) { t -= kWarp; continue; }
            t -= __ffs(~m) - 1;
            break;
        }
        if (lane == 0) sm.lo = t;
    }
    __syncthreads();
    const int32_t lo = sm.lo, C = cb0 - lo, M = cb1 - lo;
    for (int i = tid; i < M; i += kCoverThreads) {
        const int32_t cs = s.cstart[lo + i], ce = s.cend[lo + i];
        const uint32_t xs = (uint32_t)(cs - k0), xe = (uint32_t)(ce - k0);
        if (i >= C && xs < (uint32_t)kCoverTile) atomicOr(&lm.smap[xs >> 5], 1u << (xs & 31));
        if (xe < (uint32_t)kCoverTile) atomicOr(&lm.emap[xe >> 5], 1u << (xe & 31));
    }
    __syncthreads();
    if (warp == 0) popc_prefix<kChunks>(lm.smap, lm.spre);
    if (warp == 1) popc_prefix<kChunks>(lm.emap, lm.epre);
    __syncthreads();
    const int32_t* gcs = s.cstart + lo;
    const int32_t* gce = s.cend + lo;
    const unsigned below = (1u << lane) - 1u;
    // window [lw, hi] of this lane's position in run c
    auto window = [&](int c, int32_t& lw, int32_t& hi) {
        hi = C + lm.spre[c] + __popc(lm.smap[c] & (below | (1u << lane))) - 1;
        lw = lm.epre[c] + __popc(lm.emap[c] & below);
    };
    // longest length b over the window, its leftmost holder vb, the number of holders ct
    auto best_of = [&](int32_t lw, int32_t hi, int32_t& b, int32_t& vb, int32_t& ct) {
        b = 0; vb = -1; ct = 0;
        for (int32_t v = lw; v <= hi; ++v) {
            const int32_t len = gce[v] - gcs[v] + 1;
            const bool gt = len > b;
            ct = gt ? 1 : ct + (len == b);
            vb = gt ? v : vb;
            b = gt ? len : b;
        }
    };
    int32_t pk[kChunksPerWarp], pre[kChunksPerWarp];  // tie counts and their prefixes within the run
#pragma unroll
    for (int q = 0; q < kChunksPerWarp; ++q) {
        const int c = warp * kChunksPerWarp + q;
        const int32_t k = k0 + c * kWarp + lane;
        int32_t lw, hi, b, vb, ct;
        window(c, lw, hi);
        best_of(lw, hi, b, vb, ct);
        if (k < n) {
            __stcs(lr_len + k, b);
            __stcs(lr_start + k, b > 0 ? gcs[vb] : -1);
        }
        pk[q] = k < n ? ct : 0;
        if constexpr (kAll) {
            int tot;
            pre[q] = ties_prefix(pk[q], below, &tot);
            if (lane == 0) lm.chunk[c] = tot;
        }
    }
    if constexpr (kAll) {
        __syncthreads();
        if (warp == 0) {
            const int tot = scan_chunks<kChunks>(lm.chunk);
            if (lane == 0 && tile != s.hold_tile) publish(s.status_o, tile, tile == 0 ? kPrefix : kAggregate, tot);
            const long long ex = place_tile(s, tile, num_cover_tiles(n, TP), n, tot, offsets);
            if (lane == 0) sm.obase = ex;
        }
        __syncthreads();
        const long long obase = sm.obase;
        for (int q = 0; q < kChunksPerWarp; ++q) {
            const int c = warp * kChunksPerWarp + q;
            const int32_t k = k0 + c * kWarp + lane;
            long long o = obase + lm.chunk[c] + pre[q];
            if (k < n) __stcs(reinterpret_cast<long long*>(offsets) + k, o);
            if (pk[q] == 0) continue;
            int32_t lw, hi, b, vb, ct;
            window(c, lw, hi);
            best_of(lw, hi, b, vb, ct);
            for (int32_t v = vb; v <= hi; ++v) {
                if (gce[v] - gcs[v] + 1 != b) continue;
                if (o < capacity) __stcs(starts + o, gcs[v]);
                ++o;
            }
        }
    }
}

// From the staged entries to the outputs of the tile (whole CTA, after the
// barrier that completes the staging; sm.bmap, rec[0], nx, ttot and far are
// initialised).  Staged entries nlow + 1 .. MS of sm.ent reach the tile.
// kOne: the tile is the whole string, so there is nothing to look back to.
template <bool kAll, int TP, bool kOne>
__device__ __forceinline__ void cover_entries(CoverSmem<TP>& sm, int32_t n, const Scratch& s, long long tile, int32_t k0,
                                              int32_t MS, int32_t nlow, int32_t* __restrict__ lr_len,
                                              int32_t* __restrict__ lr_start, int64_t* __restrict__ offsets,
                                              int32_t* __restrict__ starts, long long capacity, int vec) {
    constexpr int kCoverTile = Cfg<TP>::kTileC;
    constexpr int kCoverThreads = Cfg<TP>::kThr;
    constexpr int kChunksPerWarp = Cfg<TP>::kChunksPerWarp;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // Per entry: the positions of the tile [hs, he) where it is a holder, the
    // holders where they begin and those left where it ends.
    uint8_t* const nx = reinterpret_cast<uint8_t*>(sm.nx);
    const int32_t k1 = k0 > 0x7fffffff - kCoverTile ? 0x7fffffff : k0 + kCoverTile;   // the tile's end (no entry ends past n)
    int32_t held = 0;                                         // positions x holders of this thread's entries
    for (int v0 = nlow + 1 + warp * kWarp; v0 <= MS; v0 += kCoverThreads) {
        const int v = v0 + lane;
        const bool in = v <= MS;                              // other lanes take the outer entries and stop at once
        const int2 me = sm.ent[in ? v : 0];
        const int32_t L = me.y, e1 = me.x + L;                // one past its end
        const int32_t a = me.x > k0 ? me.x : k0;
        const int32_t b1 = e1 < k1 ? e1 : k1;
        if constexpr (!kAll) {
            // Leftmost only: v is the answer from where the nearest entry
            // before it that is as long has ended, unless a longer one has
            // begun by then.  Neither scan passes over more than that: the
            // kernel takes 148 us for 2^26 positions of English, 244 for DNA
            // and, where 24 entries of one length cover every position, 360
            // for 2^25; 168, 336 and 741 with the scans of the all-LR query.
            int32_t qe;
            bool go;
            int u = in ? v : 1;
            do {
                const int2 q = sm.ent[--u];
                qe = q.x + q.y;
                go = (qe > a) & (q.y < L);
            } while (go);
            const int32_t hs = qe > a ? qe : a;
            if (hs < b1) {
                u = v;
                int2 q;
                do {
                    q = sm.ent[++u];
                    go = (q.x <= hs) & (q.y <= L);
                } while (go);
                if (q.x > hs) {
                    const int32_t x = hs - k0;
                    sm.rec[x] = (uint32_t)v;
                    atomicOr(&sm.bmap[x >> 5], 1u << (x & 31));
                    // nothing covers the position after v where the next
                    // entry starts later; else what is best there begins there
                    if (sm.ent[v + 1].x > e1 && e1 < k1) {
                        const int32_t y = e1 - k0;
                        sm.rec[y] = 0u;
                        atomicOr(&sm.bmap[y >> 5], 1u << (y & 31));
                    }
                }
            }
            __syncwarp();
            continue;
        }
        // to the left, over the entries that still cover a: those of length L
        // before a longer one are holders wherever v begins to be one
        int32_t left = v, eq = 1, qe;
        bool go;
        int u = in ? v : 1;
        do {
            const int2 q = sm.ent[--u];
            qe = q.x + q.y;
            go = (qe > a) & (q.y <= L);
            if (go & (q.y == L)) { ++eq; left = u; }
        } while (go);
        const int32_t hs = qe > a ? qe : a;
        // to the right, over the entries that start by e1, up to a longer one
        // (unless v is never the longest in this tile)
        int32_t first = MS + 1, feq = 0, qs;
        u = hs < b1 ? v : MS;
        do {
            const int2 q = sm.ent[++u];
            qs = q.x;
            go = (qs <= e1) & (q.y <= L);
            if (go & (q.y == L)) { first = min(first, u); ++feq; }
        } while (go);
        const int32_t he = qs < b1 ? qs : b1;
        if (hs < he) {
            held += he - hs;
            if (feq > 0) {
                nx[v] = (uint8_t)(first - v < 255 ? first - v : 255);
                if (first - v >= 255) sm.far = 1;
            }
            if (sm.ent[first].x > hs) {                       // else the next of length L begins at hs too
                const int32_t x = hs - k0;
                sm.rec[x] = (uint32_t)left | ((uint32_t)eq << 16);
                atomicOr(&sm.bmap[x >> 5], 1u << (x & 31));
            }
            // where v ends with no longer entry begun: the remaining holders
            // of length L, if any; nothing, if no entry starts by then; else
            // the best shorter entry begins there
            if (qs > e1 && e1 < k1 && (feq > 0 || u == v + 1)) {
                const int32_t x = e1 - k0;
                sm.rec[x] = feq > 0 ? ((uint32_t)first | ((uint32_t)feq << 16)) : 0u;
                atomicOr(&sm.bmap[x >> 5], 1u << (x & 31));
            }
        }
        __syncwarp();
    }
    if constexpr (kAll) {
        held = (int32_t)__reduce_add_sync(kFull, (unsigned)held);
        if (lane == 0 && held) atomicAdd(&sm.ttot, held);
    }
    __syncthreads();
    if constexpr (kAll) {
        if (!kOne && tid == 0 && tile != s.hold_tile) publish(s.status_o, tile, tile == 0 ? kPrefix : kAggregate, sm.ttot);
    }

    // Per position: its record is the one of the last boundary at or before it.
    const unsigned below = (1u << lane) - 1u;
    const unsigned upto = below | (1u << lane);
    const int c0 = warp * kChunksPerWarp;
    int pb = 0;                                               // last boundary before the warp's current run
    for (int w0 = c0; w0 > 0; w0 -= kWarp) {
        const int w = w0 - 1 - lane;
        const unsigned word = w >= 0 ? sm.bmap[w] : 0u;
        const unsigned m = __ballot_sync(kFull, word != 0u);
        if (m) {
            const int l = __ffs(m) - 1;
            pb = (w0 - 1 - l) * kWarp + 31 - __clz(__shfl_sync(kFull, word, l));
            break;
        }
    }
    uint32_t pk[kChunksPerWarp];                              // the positions' records
    uint32_t all_r = 0;                                       // their bitwise or: bounds the counts
    int32_t sum = 0;
#pragma unroll
    for (int q = 0; q < kChunksPerWarp; ++q) {
        const int x0 = (c0 + q) * kWarp;
        const unsigned word = sm.bmap[c0 + q];
        const unsigned m = word & upto;
        const uint32_t r = sm.rec[m ? x0 + 31 - __clz(m) : pb];
        if (word) pb = x0 + 31 - __clz(word);
        const int2 h = sm.ent[r & 0xffffu];
        const int32_t k = k0 + x0 + lane;
        pk[q] = r;
        if (k < n) {
            __stcs(lr_len + k, h.y);
            __stcs(lr_start + k, h.x);
            sum += (int32_t)(r >> 16);
            all_r |= r;
        } else {
            pk[q] = 0;
        }
    }
    if constexpr (kAll) {
        sum = (int32_t)__reduce_add_sync(kFull, (unsigned)sum);
        if (lane == 0) sm.wtot[warp] = sum;
        if (kOne) {
            if (tid == 0) {
                sm.obase = 0;
                offsets[n] = sm.ttot;
                if (s.total_out) *s.total_out = sm.ttot;
            }
        } else if (warp == Cfg<TP>::kWarps - 1) {
            const long long ex = place_tile(s, tile, num_cover_tiles(n, TP), n, sm.ttot, offsets);
            if (lane == 0) sm.obase = ex;
        }
        __syncthreads();
        long long o0 = sm.obase;
        {
            const int32_t t = lane < warp ? sm.wtot[lane] : 0;
            o0 += (int32_t)__reduce_add_sync(kFull, (unsigned)t);
        }
        // starts[o0 ..]: 32-bit indices from here; entries past the capacity are not written
        const long long room = capacity - o0;
        const int32_t lim = room < 0 ? 0 : (room > 0x7fffffff ? 0x7fffffff : (int32_t)room);
        int32_t* const out = starts + o0;
        const bool far = sm.far != 0;
        // every compact LLR of the longest length over a position (its record
        // r, its first start at out[o]), ascending
        auto emit = [&](uint32_t r, int32_t o) {
            int32_t left = min((int32_t)(r >> 16), lim - o);
            if (left <= 0) return;
            int v = (int)(r & 0xffffu);
            int32_t* p = out + o;
            __stcs(p, sm.ent[v].x);
            if (!far) {
                while (--left > 0) {
                    v += nx[v];
                    __stcs(++p, sm.ent[v].x);
                }
            } else {
                while (--left > 0) {
                    const int32_t d = nx[v], L = sm.ent[v].y;
                    v += d;
                    if (d == 255)
                        while (v <= MS && sm.ent[v].y != L) ++v;
                    __stcs(++p, sm.ent[v].x);
                }
            }
        };
        // Prefixes of the counts, eight consecutive positions per lane, where
        // every count of the warp fits four bits, an index twelve, and the
        // tile is whole: the records go through shared memory as 16-bit words
        // (the warp's part of rec, which nobody reads any more), one
        // multiplication makes the prefixes of four counts, a lane stores
        // eight offsets, and the loop over the runs needs no registers for
        // them and is not unrolled.  English 2^28 1.58 -> 1.55 ms, DNA 2^26
        // 608 -> 577 us, mixed batch 2.40 -> 2.31 ms; with the loop unrolled
        // the code no longer fits the instruction cache (1.80 ms).
        const bool whole = vec && k0 <= n - kCoverTile;
        if (Cfg<TP>::kCap + 2 <= 0x1000 && whole && !__any_sync(kFull, all_r >= (16u << 16))) {
            uint16_t* const rb = reinterpret_cast<uint16_t*>(sm.rec + c0 * kWarp);   // records as index | count << 12
            uint16_t* const ob = rb + kChunksPerWarp * kWarp;
#pragma unroll
            for (int q = 0; q < kChunksPerWarp; ++q)
                rb[q * kWarp + lane] = (uint16_t)((pk[q] & 0xfffu) | ((pk[q] >> 4) & 0xf000u));
            __syncwarp();
            const uint4 r8 = *reinterpret_cast<const uint4*>(rb + lane * 8);
            // counts of four positions, a byte each
            const uint32_t cx = ((r8.x >> 12) & 0xfu) | ((r8.x >> 20) & 0xf00u) | ((r8.y << 4) & 0xf0000u) | ((r8.y >> 4) & 0xf000000u);
            const uint32_t cy = ((r8.z >> 12) & 0xfu) | ((r8.z >> 20) & 0xf00u) | ((r8.w << 4) & 0xf0000u) | ((r8.w >> 4) & 0xf000000u);
            const uint32_t sx = cx * 0x01010101u, sy = cy * 0x01010101u;   // inclusive prefixes, a byte each
            const uint32_t tx = sx >> 24;
            const uint32_t px = sx << 8, py = (sy << 8) + tx * 0x01010101u;  // exclusive ones of the eight
            const int32_t mine = (int32_t)(tx + (sy >> 24));
            const uint32_t ex = (uint32_t)(warp_incl_scan(mine) - mine);
            const uint32_t e2 = ex * 0x10001u;                               // below 2^16: 256 counts of at most 15
            uint4 w;
            w.x = __byte_perm(px, 0, 0x4140) + e2;
            w.y = __byte_perm(px, 0, 0x4342) + e2;
            w.z = __byte_perm(py, 0, 0x4140) + e2;
            w.w = __byte_perm(py, 0, 0x4342) + e2;
            *reinterpret_cast<uint4*>(ob + lane * 8) = w;
            int64_t* const po = offsets + k0 + c0 * kWarp + lane * 8;
            const long long base = o0 + ex;
            store_offsets(po, base, base + ((px >> 8) & 0xffu), base + ((px >> 16) & 0xffu), base + (px >> 24));
            store_offsets(po + 4, base + (py & 0xffu), base + ((py >> 8) & 0xffu), base + ((py >> 16) & 0xffu),
                          base + (py >> 24));
            __syncwarp();
#pragma unroll 1
            for (int q = 0; q < kChunksPerWarp; ++q) {
                const uint32_t r = rb[q * kWarp + lane];
                emit((r & 0xfffu) | ((r >> 12) << 16), (int32_t)ob[q * kWarp + lane]);
                __syncwarp();
            }
            return;
        }
        int32_t run = 0;
#pragma unroll
        for (int q = 0; q < kChunksPerWarp; ++q) {
            const int32_t k = k0 + (c0 + q) * kWarp + lane;
            int tot;
            const int32_t o = run + ties_prefix((int)(pk[q] >> 16), below, &tot);
            run += tot;
            if (k < n) __stcs(reinterpret_cast<long long*>(offsets) + k, o0 + o);
            emit(pk[q], o);
            __syncwarp();
        }
    }
}

}  // namespace

template <bool kAll, int TP>
__global__ void __launch_bounds__(Cfg<TP>::kThr, Cfg<TP>::kMinBlocks)
k_cover(int32_t n, Scratch s, int32_t* __restrict__ lr_len, int32_t* __restrict__ lr_start,
        int64_t* __restrict__ offsets, int32_t* __restrict__ starts, long long capacity, int vec) {
    begin_last();
    constexpr int kCoverTile = Cfg<TP>::kTileC;
    constexpr int kCoverThreads = Cfg<TP>::kThr;
    constexpr int kCoverTilesPer = TP;
    constexpr int kChunks = Cfg<TP>::kChunks;
    extern __shared__ __align__(16) unsigned char cover_smem[];
    CoverSmem<TP>& sm = *reinterpret_cast<CoverSmem<TP>*>(cover_smem);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        if constexpr (kAll) sm.tile = atomicAdd(&s.tickets[2], 1u);
        sm.nlow = 0;
        sm.ttot = 0;
        sm.far = 0;
        sm.rec[0] = 0;                                       // no holder at the tile's start, unless an entry writes it
    }
    if (tid < kChunks) sm.bmap[tid] = tid == 0 ? 1u : 0u;
    if constexpr (kAll) {
        for (int i = tid; i < CoverSmem<TP>::kNxWords; i += kCoverThreads) sm.nx[i] = 0;
    }
    __syncthreads();
    // leftmost only: no look-back, so no order of the tiles to keep (1.2 x 10^4
    // positions by rank 31.5 -> 29.8 us without the ticket)
    const long long tile = kAll ? sm.tile : (long long)blockIdx.x;
    const int32_t k0 = (int32_t)(tile * kCoverTile);         // n < 2^31: positions fit 32 bits
    // LLRc entries [cb0, cb1) start inside this tile; clamped so that a
    // corrupted front end (already reported) cannot send reads out of bounds
    const long long ft = tile * kCoverTilesPer;               // first front-end tile
    const long long ft1 = (ft + kCoverTilesPer < s.ntiles) ? ft + kCoverTilesPer : s.ntiles;
    int32_t cb0 = s.tile_cbase[ft], cb1 = s.tile_cbase[ft1];
    cb0 = cb0 < 0 ? 0 : (cb0 > n ? n : cb0);
    cb1 = cb1 < cb0 ? cb0 : (cb1 > n ? n : cb1);
    if (cb1 - cb0 > kCoverTile) cb1 = cb0 + kCoverTile;

    // Stage LLRc[cb0 - kSpec, cb1): the tile's own entries and, in the same
    // round trip, the kSpec entries before them, which hold the carry (the
    // entries whose end reaches k0: a suffix, ends increase) unless it is
    // longer than kSpec.
    const int32_t sbase = cb0 > kSpec ? cb0 - kSpec : 0;
    const int32_t MS = cb1 - sbase;
    const int32_t nspec = cb0 - sbase;
    constexpr int kBatch = 2;                                 // entries a thread has in flight (one: 4 % slower)
    for (int i0 = 0; i0 < MS; i0 += kBatch * kCoverThreads) {
        int32_t cs[kBatch], ce[kBatch];
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int i = i0 + u * kCoverThreads + tid;
            cs[u] = i < MS ? __ldcg(s.cstart + sbase + i) : 0;
            ce[u] = i < MS ? __ldcg(s.cend + sbase + i) : 0;
        }
        if (i0 == 0 && warp < kSpec / kWarp) {
            const unsigned m = __ballot_sync(kFull, tid < nspec && ce[0] < k0);
            if (lane == 0 && m) atomicAdd(&sm.nlow, __popc(m));
        }
#pragma unroll
        for (int u = 0; u < kBatch; ++u) {
            const int i = i0 + u * kCoverThreads + tid;
            // entries inside [0, n): whatever a failed front end (already
            // reported) left here, the scans below end at the outer entries
            if ((uint32_t)cs[u] >= (uint32_t)n) cs[u] = k0;
            if (ce[u] < cs[u] || ce[u] >= n) ce[u] = cs[u];
            if (i < MS) sm.ent[i + 1] = make_int2(cs[u], ce[u] - cs[u] + 1);
        }
    }
    if (tid == 0) {
        sm.ent[0] = make_int2(-1, 0);
        sm.ent[MS + 1] = make_int2(0x7fffffff, 0);
    }
    __syncthreads();
    // every staged candidate reaches k0 with more LLRc before them: the carry
    // may be longer than what is staged
    const int32_t nlow = sm.nlow;
    if (sbase > 0 && nlow == 0) {
        __syncthreads();
        cover_long_carry<kAll, TP>(sm, n, s, tile, cb0, cb1, lr_len, lr_start, offsets, starts, capacity);
        return;
    }
    cover_entries<kAll, TP, false>(sm, n, s, tile, k0, MS, nlow, lr_len, lr_start, offsets, starts, capacity, vec);
}

// A string of at most one tile of 8192 positions: the whole query in one CTA
// and one launch (Lemma 1 from sa or rank into shared memory by position,
// flags, compaction, cover), with nothing to clear before it.  What bounds a
// query of this size is launches and the chains between them: 4099
// positions of DNA took 74 us with five launches, and 42 us with this one (33 us
// since the results of a query come back in one copy).
constexpr int kOneTP = 4;
static_assert(Cfg<kOneTP>::kTileC == kOneTileMax, "one-tile strings");

template <bool kAll, bool kSa>
__global__ void __launch_bounds__(Cfg<kOneTP>::kThr, 1)
k_one_tile(const int32_t* __restrict__ in, const int32_t* __restrict__ lcp, int32_t n, Scratch s,
           int32_t* __restrict__ lr_len, int32_t* __restrict__ lr_start, int64_t* __restrict__ offsets,
           int32_t* __restrict__ starts, long long capacity) {
    constexpr int TP = kOneTP, kThr = Cfg<TP>::kThr, kChunks = Cfg<TP>::kChunks, kPer = Cfg<TP>::kTileC / kThr;
    extern __shared__ __align__(16) unsigned char cover_smem[];
    CoverSmem<TP>& sm = *reinterpret_cast<CoverSmem<TP>*>(cover_smem);
    int32_t* const D = reinterpret_cast<int32_t*>(cover_smem + sizeof(CoverSmem<TP>));   // L by position, -1 where none came
    __shared__ int32_t wsum[kThr / kWarp];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) {
        sm.ttot = 0;
        sm.far = 0;
        sm.rec[0] = 0;
    }
    if (tid < kChunks) sm.bmap[tid] = tid == 0 ? 1u : 0u;
    if constexpr (kAll) {
        for (int i = tid; i < CoverSmem<TP>::kNxWords; i += kThr) sm.nx[i] = 0;
    }
    // all loads in flight before the first is used
    int32_t v[kPer], a[kPer], b[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int r = j * kThr + tid;
        v[j] = r < n ? __ldg(in + r) : 0;
        if (kSa) { a[j] = r < n ? __ldg(lcp + r) : 0; b[j] = r < n ? __ldg(lcp + r + 1) : 0; }
        D[r] = -1;
    }
    bool bad = false;
    if (tid == 0 && (__ldg(lcp) != 0 || __ldg(lcp + n) != 0)) bad = true;
    if (!kSa) {
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const int k = j * kThr + tid;
            if (k < n && (uint32_t)v[j] >= (uint32_t)n) { bad = true; v[j] = 0; }
            a[j] = k < n ? __ldg(lcp + v[j]) : 0;
            b[j] = k < n ? __ldg(lcp + v[j] + 1) : 0;
        }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        const int r = j * kThr + tid;
        if (r >= n) continue;
        const uint32_t p = kSa ? (uint32_t)v[j] : (uint32_t)r;
        if (p >= (uint32_t)n) { bad = true; continue; }
        int32_t L = a[j] > b[j] ? a[j] : b[j];
        if ((uint32_t)L > (uint32_t)n - p) { bad = true; L = 0; }   // negative ones too
        D[p] = L;
    }
    __syncthreads();
    // flags and compaction: eight consecutive positions per thread
    static_assert(kPer == 8, "positions per thread");
    const int x = tid * kPer;
    int32_t l[kPer], prev = x > 0 ? max(D[x - 1], 0) : 0;
    unsigned f = 0;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
        l[j] = D[x + j];
        if (x + j < n && l[j] < 0) bad = true;                // sa gave another position twice
        l[j] = max(l[j], 0);
        if (l[j] > 0 && l[j] >= prev) f |= 1u << j;           // 0 past the end
        prev = l[j];
    }
    if (bad) atomicOr(s.err, kErrInput);
    const int c = __popc(f), incl = warp_incl_scan(c);
    if (lane == kWarp - 1) wsum[warp] = incl;
    __syncthreads();
    const int w = wsum[lane];                                 // kThr / kWarp = 32 totals
    static_assert(kThr / kWarp == kWarp, "one total per lane");
    int o = incl - c + (int)__reduce_add_sync(kFull, lane < warp ? (unsigned)w : 0u);
    const int32_t m = (int32_t)__reduce_add_sync(kFull, (unsigned)w);
#pragma unroll
    for (int j = 0; j < kPer; ++j)
        if ((f >> j) & 1u) sm.ent[++o] = make_int2(x + j, l[j]);
    if (tid == 0) {
        sm.ent[0] = make_int2(-1, 0);
        sm.ent[m + 1] = make_int2(0x7fffffff, 0);
        s.tile_cbase[s.ntiles] = m;
    }
    __syncthreads();
    cover_entries<kAll, TP, true>(sm, n, s, 0, 0, m, 0, lr_len, lr_start, offsets, starts, capacity, 0);
}

namespace {

template <bool kAll, int TP>
void launch_cover_t(int32_t n, const Scratch& s, int32_t* lr_len, int32_t* lr_start, int64_t* offsets,
                    int32_t* starts, long long capacity, cudaStream_t stream) {
    const unsigned grid = (unsigned)num_cover_tiles(n, TP);
    const int vec = ((uintptr_t)offsets & 31u) == 0 ? 1 : 0;   // whole-sector stores (tiles start at multiples of 2048)
    launch_after(k_cover<kAll, TP>, grid, Cfg<TP>::kThr, sizeof(CoverSmem<TP>), stream, n, s, lr_len, lr_start, offsets, starts,
                 capacity, vec);
}

template <int TP>
cudaError_t set_cover_smem() {
    cudaError_t e = cudaFuncSetAttribute(k_cover<true, TP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sizeof(CoverSmem<TP>));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_cover<false, TP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(CoverSmem<TP>));
    return e;
}

}  // namespace

namespace {
constexpr size_t kOneSmem = sizeof(CoverSmem<kOneTP>) + (size_t)Cfg<kOneTP>::kTileC * 4;

template <bool kAll, bool kSa>
cudaError_t set_one_smem() {
    return cudaFuncSetAttribute(k_one_tile<kAll, kSa>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kOneSmem);
}

template <bool kAll, bool kSa>
void launch_one_t(const int32_t* in, const int32_t* lcp, int32_t n, const Scratch& s, int32_t* lr_len, int32_t* lr_start,
                  int64_t* offsets, int32_t* starts, long long capacity, cudaStream_t stream) {
    k_one_tile<kAll, kSa><<<1, Cfg<kOneTP>::kThr, kOneSmem, stream>>>(in, lcp, n, s, lr_len, lr_start, offsets, starts,
                                                                      capacity);
}
}  // namespace

void launch_one_tile(const int32_t* sa, const int32_t* rank, const int32_t* lcp, int32_t n, const Scratch& s,
                     int32_t* lr_len, int32_t* lr_start, int64_t* offsets, int32_t* starts, long long capacity, bool all,
                     cudaStream_t stream) {
    if (!all) { offsets = nullptr; starts = nullptr; capacity = 0; }
    if (sa) {
        if (all) launch_one_t<true, true>(sa, lcp, n, s, lr_len, lr_start, offsets, starts, capacity, stream);
        else launch_one_t<false, true>(sa, lcp, n, s, lr_len, lr_start, offsets, starts, capacity, stream);
    } else {
        if (all) launch_one_t<true, false>(rank, lcp, n, s, lr_len, lr_start, offsets, starts, capacity, stream);
        else launch_one_t<false, false>(rank, lcp, n, s, lr_len, lr_start, offsets, starts, capacity, stream);
    }
}

cudaError_t configure_cover() {
    cudaError_t e = set_one_smem<true, true>();
    if (e == cudaSuccess) e = set_one_smem<true, false>();
    if (e == cudaSuccess) e = set_one_smem<false, true>();
    if (e == cudaSuccess) e = set_one_smem<false, false>();
    if (e == cudaSuccess) e = set_cover_smem<1>();
    if (e == cudaSuccess) e = set_cover_smem<2>();
    if (e == cudaSuccess) e = set_cover_smem<4>();
    return e;
}

void launch_cover(int32_t n, const Scratch& s, int32_t* lr_len, int32_t* lr_start, int64_t* offsets,
                  int32_t* starts, long long capacity, bool all, int tiles_per, cudaStream_t stream) {
    if (!all) { offsets = nullptr; starts = nullptr; capacity = 0; }
    switch (tiles_per) {
        case 2:
            if (all) launch_cover_t<true, 2>(n, s, lr_len, lr_start, offsets, starts, capacity, stream);
            else launch_cover_t<false, 2>(n, s, lr_len, lr_start, offsets, starts, capacity, stream);
            break;
        case 4:
            if (all) launch_cover_t<true, 4>(n, s, lr_len, lr_start, offsets, starts, capacity, stream);
            else launch_cover_t<false, 4>(n, s, lr_len, lr_start, offsets, starts, capacity, stream);
            break;
        default:
            if (all) launch_cover_t<true, 1>(n, s, lr_len, lr_start, offsets, starts, capacity, stream);
            else launch_cover_t<false, 1>(n, s, lr_len, lr_start, offsets, starts, capacity, stream);
    }
}

}  // namespace lr
