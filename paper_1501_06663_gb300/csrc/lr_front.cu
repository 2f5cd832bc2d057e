// Front ends of the longest-repeat query: they turn the input arrays into
// the compact LLR array LLRc (Sec. 3.2 / Sec. 4.2.1 of Tian and Xu, arXiv
// 1501.06663): every position i with L_i > 0 and L_i >= L_{i-1}, in
// ascending i, as cstart[t] = i, cend[t] = i + L_i - 1, where
// L_i = max(lcp[rank[i]], lcp[rank[i]+1]) (Lemma 1).  They also record, for
// every tile of kTile positions and every segment of kSeg positions, the
// index of its first LLRc entry (tile_cbase, seg_cbase), which the cover
// kernels start from.
//
// Three front ends compute the same LLRc:
//
//  * rank-order (the default when the suffix array is given).  Lemma 1 read
//    in rank order is L_{sa[r]} = max(lcp[r], lcp[r+1]): sa and lcp are then
//    read once, coalesced, instead of one random lcp sector per position.
//    k_part1 and k_part2 radix-partition the pairs <sa[r], L_{sa[r]}> by
//    the position, first into super-buckets of 2^20 positions, then into
//    buckets of 2^15 (packed 4-byte entries; a length of 4095 or more goes
//    to lbig).  k_bucket_llr then loads one bucket per
//    CTA, scatters its lengths into shared memory by position, and flags
//    and compacts them.
//
//  * dense (the suffix array given, up to a few million positions): the
//    lengths are stored straight at their positions (k_scatter) and compacted
//    tile by tile (k_compact).
//
//  * rank gather (when only rank is given, as in the paper's data flow of
//    Sec. 4): k_gather reads rank coalesced, gathers the two lcp words of each
//    position and stores the lengths in the same dense array.
//
// All place their entries in LLRc with a decoupled look-back over the
// per-CTA counts (tiles handed out in order by an atomic ticket).
#include <cuda_runtime.h>
#include <cstdint>
#include "lr_device.cuh"
#include "lr_internal.h"

namespace lr {

namespace {

constexpr int kSms = 152;                // of a GB300: grids of the kernels whose CTAs stay

// The same pointer, its origin hidden from the compiler.  The stage areas of the
// partition kernels are reached through such pointers: measured with events,
// at 2^28 positions of English, the partition phase takes 1.39 ms with both
// (generic addresses), 1.42 with k_part1's alone and 1.50 with neither; in
// the bucket kernel and for the counters the same change made no difference.
template <class T>
__device__ __forceinline__ T* opaque(T* p) { asm volatile("" : "+l"(p)); return p; }

__device__ __forceinline__ void report(const Scratch& s, unsigned bits) { atomicOr(s.err, bits); }

// The strings of a batched query that overlap one CTA's flattened range
// [g0, g1), with their offsets staged in shared memory when there are at
// most kSegCap of them (else looked up in global memory).
struct SegView {
    const int64_t* off;      // global, num + 1 entries
    long long* sh;           // shared, kSegCap + 1 entries
    long long j0, j1;        // first and last string overlapping the range
    bool staged;

    // Called by the whole CTA (contains a barrier).
    __device__ void stage(const Segs& segs, const Scratch& s, long long g0, long long g1, long long* smem) {
        off = segs.off;
        sh = smem;
        // j1: the string holding the start of the tile after the range,
        // which is at or after the string holding g1 - 1
        const long long t0 = g0 / kTile, t1 = (g1 - 1) / kTile + 1;
        j0 = s.tile_seg[t0];
        j1 = (t1 < s.ntiles) ? s.tile_seg[t1] : segs.num - 1;
        if (j1 < j0) j1 = j0;                          // only after a reported bad offset table
        staged = (j1 - j0 + 2) <= kSegCap + 1;
        if (staged)
            for (long long i = threadIdx.x; i < j1 - j0 + 2; i += blockDim.x) sh[i] = __ldg(off + j0 + i);
        __syncthreads();
    }
    __device__ __forceinline__ long long at(long long j) const { return staged ? sh[j - j0] : __ldg(off + j); }
    // the string holding position g (j0 <= result <= j1); `hint` only moves forward
    __device__ __forceinline__ long long find(long long g, long long hint) const {
        if (staged) {
            long long j = hint;
            while (j < j1 && sh[j + 1 - j0] <= g) ++j;
            return j;
        }
        long long lo = hint, hi = j1;                 // last j with off[j] <= g
        while (lo < hi) {
            const long long mid = (lo + hi + 1) >> 1;
            if (__ldg(off + mid) <= g) lo = mid; else hi = mid - 1;
        }
        return lo;
    }
};

// For every tile of kTile flattened positions, the string holding its first
// position (the last j with off[j] <= tile start); the offset table is
// checked on the way, by all `step` threads.  With the strings dealt to the
// threads of the tiles alone, a query of 4.5 M strings of one symbol took 2.77
// ms by rank and 1.06 ms by sa, most of it here; now 0.16 ms.
__device__ __forceinline__ void seg_index(int32_t n, const Scratch& s, const Segs& segs, long long first, long long step) {
    for (long long t = first; t < s.ntiles; t += step) {
        const long long g = t * kTile;
        long long lo = 0, hi = segs.num - 1;
        while (lo < hi) {
            const long long mid = (lo + hi + 1) >> 1;
            if (__ldg(segs.off + mid) <= g) lo = mid; else hi = mid - 1;
        }
        s.tile_seg[t] = (int32_t)lo;
    }
    if (first == 0 && (__ldg(segs.off) != 0 || __ldg(segs.off + segs.num) != n)) report(s, kErrInput);
    // offsets must not decrease
    for (long long j = first; j < segs.num; j += step)
        if (__ldg(segs.off + j) > __ldg(segs.off + j + 1)) report(s, kErrInput);
}

// Blocks of 256 threads for `work` items of a kernel that also runs
// seg_index: four items or strings per thread, a few blocks per SM at most.
unsigned index_grid(long long work, const Segs& segs) {
    const long long most = work > segs.num ? work : segs.num, blocks = (most + 1023) / 1024;
    return (unsigned)(blocks < 8 * kSms ? blocks : 8 * kSms);
}

__global__ void k_seg_index(int32_t n, Scratch s, Segs segs) {
    begin_after();
    seg_index(n, s, segs, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
}

}  // namespace

void launch_seg_index(int32_t n, const Scratch& s, const Segs& segs, cudaStream_t stream) {
    k_seg_index<<<index_grid(4 * s.ntiles, segs), 256, 0, stream>>>(n, s, segs);
}

// ---------------------------------------------------------------------------
// rank-order front end
// ---------------------------------------------------------------------------

// Shared memory of a partition CTA: per-bucket counters and the round's
// entries staged in bucket order, so that each warp store writes one
// contiguous run.  An entry and its bucket id are staged side by side, by one
// 8-byte store: with the ids in an array of their own, two stores to random
// banks per entry, the partition phase of English 2^28 took 1.51 ms instead
// of 1.42, now 1.39 (shared-memory wavefronts are what bounds it).
struct PartSmem {
    uint32_t* hist;      // nb: entries of the round per bucket, then slot counters
    uint32_t* loff;      // nb + 1: exclusive prefix of hist (staging offsets), in
                         // place of hist (the scan reads hist before it writes)
    uint32_t* base;      // nb: where the round's entries of a bucket go, minus loff: staged
                         // entry i of bucket b belongs at index base[b] + i of all buckets
    uint32_t* stage;     // kPartRound entries with their bucket ids (8 bytes, from the next 8-byte boundary), in
                         // bucket order
};

__host__ __device__ inline size_t part_stage_offset(int nb) { return (size_t)(2 * nb + 2) * 4; }

__device__ __forceinline__ PartSmem part_smem(unsigned char* raw, int nb) {
    PartSmem p;
    p.hist = reinterpret_cast<uint32_t*>(raw);
    p.loff = p.hist;
    p.base = p.loff + nb + 1;
    p.stage = p.base + nb;
    return p;
}

// Bulk-copy staging of a level-1 round: sa[r0, r0 + kPartRound) and the
// round's lcp slice (kPartRound + 1 entries from a 16-byte-aligned start,
// rounded out to 16-byte multiples: at most kPartRound + 8 entries), at a
// 16-byte-aligned offset after the counters; it overlaps the stage area,
// which is written only after every thread has read its entries.
constexpr int kPartLcpCap = kPartRound + 8;
constexpr int kPartLoadBytes = kPartRound * 4 + kPartLcpCap * 4;
__host__ __device__ inline size_t part_load_offset(int nb) { return ((size_t)(2 * nb + 1) * 4 + 15) & ~(size_t)15; }

size_t part_smem_bytes(int nb) {
    const size_t a = part_stage_offset(nb) + (size_t)kPartRound * 8;
    const size_t b = part_load_offset(nb) + kPartLoadBytes;
    return a > b ? a : b;
}

// Room for c entries in bucket b (of 2^log entries) by one global atomic:
// the index base of PartSmem.  More entries than the bucket holds (the
// positions are not a permutation) set *over; the caller then checks every
// index before it writes.
__device__ __forceinline__ uint32_t part_room(unsigned* cursor, int b, uint32_t c, uint32_t loff, int log, int* over) {
    const uint32_t at = atomicAdd(cursor + (size_t)b * kCursorStride, c);
    if (at + c > (1u << log)) *over = 1;
    return ((uint32_t)b << log) + at - loff;
}

// Exclusive scan of hist[0..nb) into loff[0..nb] by the whole CTA
// (kPartThreads threads, R consecutive buckets each, nb <= R * kPartThreads),
// and one global atomic per non-empty bucket to reserve the round's room.
template <int R>
__device__ __forceinline__ void part_reserve_r(const PartSmem& p, int nb, unsigned* cursor, int log, int* over) {
    __shared__ uint32_t wsum[kPartThreads / kWarp];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    uint32_t a[R], sum = 0;
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int b = R * tid + u;
        a[u] = (b < nb) ? p.hist[b] : 0u;
        sum += a[u];
    }
    const int incl = warp_incl_scan((int)sum);
    if (lane == kWarp - 1) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        const int v = (lane < kPartThreads / kWarp) ? (int)wsum[lane] : 0;
        const int wi = warp_incl_scan(v);
        if (lane < kPartThreads / kWarp) wsum[lane] = wi - v;
        if (lane == kWarp - 1) p.loff[nb] = wi;
    }
    __syncthreads();
    uint32_t ex = wsum[warp] + incl - sum;
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int b = R * tid + u;
        if (b < nb) {
            p.loff[b] = ex;
            if (a[u]) p.base[b] = part_room(cursor, b, a[u], ex, log, over);
        }
        ex += a[u];
    }
}

// The same by warp 0 alone, for at most kWarp * R buckets (R consecutive
// buckets per lane); the other warps wait at the caller's next barrier.
// Each lane writes the staging offsets of its own buckets in place of their
// counts after reading them.  Buckets from `last` on get no room.
template <int R>
__device__ __forceinline__ void part_reserve_w(const PartSmem& p, int nb, int last, unsigned* cursor, int log,
                                               int* over) {
    if (threadIdx.x >= kWarp) return;
    const int lane = threadIdx.x;
    uint32_t a[R], sum = 0;
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int b = R * lane + u;
        a[u] = (b < nb) ? p.hist[b] : 0u;
        sum += a[u];
    }
    const int incl = warp_incl_scan((int)sum);
    uint32_t ex = (uint32_t)incl - sum;
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int b = R * lane + u;
        if (b < nb) {
            p.loff[b] = ex;
            if (a[u] && b < last) p.base[b] = part_room(cursor, b, a[u], ex, log, over);
        }
        ex += a[u];
    }
    if (lane == kWarp - 1) p.loff[nb] = (uint32_t)incl;
}

// The exclusive scan of hist[0..nb) into loff[0..nb] alone, by warp 0, for
// at most kWarp * R buckets: k_part1 then reserves each bucket's room with
// one thread per bucket, in the same phase as its staging writes.
template <int R>
__device__ __forceinline__ void part_scan_w(const PartSmem& p, int nb) {
    if (threadIdx.x >= kWarp) return;
    const int lane = threadIdx.x;
    uint32_t a[R], sum = 0;
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int b = R * lane + u;
        a[u] = (b < nb) ? p.hist[b] : 0u;
        sum += a[u];
    }
    const int incl = warp_incl_scan((int)sum);
    uint32_t ex = (uint32_t)incl - sum;
#pragma unroll
    for (int u = 0; u < R; ++u) {
        const int b = R * lane + u;
        if (b < nb) p.loff[b] = ex;
        ex += a[u];
    }
    if (lane == kWarp - 1) p.loff[nb] = (uint32_t)incl;
}

// up to 2048 super-buckets (n <= 2^31 positions in super-buckets of 2^20)
__device__ __forceinline__ void part_reserve(const PartSmem& p, int nb, unsigned* cursor, int log, int* over) {
    static_assert(4 * kPartThreads >= 2048, "partition CTAs too small for 2048 super-buckets");
    if (nb <= 2 * kPartThreads) part_reserve_r<2>(p, nb, cursor, log, over);
    else part_reserve_r<4>(p, nb, cursor, log, over);
}

// The level-1 entries of a round whose counts are complete: staging offsets,
// room in the super-buckets, the entries staged in bucket order and written
// out (a warp store is one run per bucket it touches).  key: bucket << 16 |
// slot, or ~0u for none; `over` is zero before.  Returns 1 when a
// super-bucket gets more than 2^20 entries.  Called by the whole CTA after
// the barrier that completes the counts.
__device__ __forceinline__ unsigned level1_write(const PartSmem& P, int nb, const Scratch& s,
                                                 const uint32_t (&ent)[kPartPer], const uint32_t (&key)[kPartPer],
                                                 bool all_valid, int* over) {
    // 8-byte aligned; formed from the address, so a generic pointer (see opaque)
    uint2* const stage = reinterpret_cast<uint2*>(((uintptr_t)P.stage + 7u) & ~(uintptr_t)7u);
    const bool wscan = nb <= 8 * kWarp;
    if (wscan) part_scan_w<8>(P, nb);
    else part_reserve(P, nb, s.cursor1, kSuperLog, over);
    __syncthreads();
    if (wscan) {
        for (int b = threadIdx.x; b < nb; b += kPartThreads) {
            const uint32_t o = P.loff[b], c = P.loff[b + 1] - o;
            if (c) P.base[b] = part_room(s.cursor1, b, c, o, kSuperLog, over);
        }
    }
#pragma unroll
    for (int j = 0; j < kPartPer; ++j) {
        if (!all_valid && key[j] == 0xffffffffu) continue;
        const uint32_t b1 = key[j] >> 16;
        const uint32_t o = P.loff[b1] + (key[j] & 0xffffu);
        stage[o] = make_uint2(ent[j], b1);
    }
    __syncthreads();
    unsigned bad = 0;
    if (all_valid && *over == 0) {                      // kPartRound entries, all with room
#pragma unroll
        for (int j = 0; j < kPartPer; ++j) {
            const uint32_t i = j * kPartThreads + threadIdx.x;
            const uint2 v = stage[i];
            s.ent1[P.base[v.y] + i] = v.x;
        }
    } else {
        const uint32_t total = P.loff[nb];
        for (uint32_t i = threadIdx.x; i < total; i += kPartThreads) {
            const uint2 v = stage[i];
            const uint32_t b1 = v.y, idx = P.base[b1] + i;
            if (idx - (b1 << kSuperLog) < (uint32_t)kSuper) s.ent1[idx] = v.x;
            else bad = 1;                               // more than 2^20 positions: not a permutation
        }
    }
    return bad;
}

// Slot of this lane's entry in bucket b among the entries counted so far,
// with one shared atomic per run of lanes (in lane order) that carry the
// same b: entries that arrive clustered by bucket would otherwise serialise
// on one counter.  All lanes of the warp call it; a lane with !valid gets
// no slot (and b is ignored).
__device__ __forceinline__ uint32_t run_slot(uint32_t* hist, uint32_t b, bool valid) {
    const int lane = lane_id();
    const uint32_t bk = valid ? b : 0xffffffffu;
    const uint32_t pb = __shfl_up_sync(kFull, bk, 1);
    const bool head = lane == 0 || bk != pb;
    const unsigned heads = __ballot_sync(kFull, head);
    const unsigned upto = (2u << lane) - 1u;           // lanes 0 .. lane
    const int h = 31 - __clz(heads & upto);            // head of this lane's run
    const unsigned after = heads & ~upto;
    const int next = after ? __ffs(after) - 1 : kWarp; // head of the next run
    uint32_t base = 0;
    if (head && valid) base = atomicAdd(hist + b, (uint32_t)(next - lane));
    base = __shfl_sync(kFull, base, h);
    return base + (uint32_t)(lane - h);
}

// The level-1 partition of one round's <position p[j], length L[j]> pairs
// (entry j of each thread, at round index j * kPartThreads + thread, when
// that index is below cnt), as k_part1 does it for its rank-order pairs,
// for the rank-window front end: counted per super-bucket in shared memory
// (one atomic per run of lanes with the same super-bucket, run_slot: the
// rank-window pairs come in such runs), room reserved with one global
// atomic per touched super-bucket (cursors one cache line apart), staged in
// bucket order and written out as <position mod 2^20, min(L, 4095)>.  A length of 4095 or
// more is stored in lbig (field 4095); the length of the last position of
// every bucket goes to halo (the next bucket's predecessor).  Returns 1
// after an input error (a position out of range, or more than 2^20 of them
// in a super-bucket: the positions are not a permutation).
__device__ __forceinline__ unsigned level1_scatter(const PartSmem& P, int nb, const Scratch& s, int32_t n,
                                                   const uint32_t (&p)[kPartPer], const int32_t (&L)[kPartPer],
                                                   int cnt, int* over) {
    unsigned bad = 0;
    uint32_t ent[kPartPer], key[kPartPer];          // key: bucket << 16 | slot, or ~0u
#pragma unroll
    for (int j = 0; j < kPartPer; ++j) {
        const bool in = j * kPartThreads + (int)threadIdx.x < cnt;
        const uint32_t pj = p[j];
        const bool ok = in && pj < (uint32_t)n;
        if (in && !ok) bad = 1;
        uint32_t b1 = 0;
        if (ok) {
            const int32_t Lj = L[j];
            uint32_t field = (uint32_t)Lj;
            if (field >= kEsc12) { field = kEsc12; s.lbig[pj] = Lj; }
            if ((pj & (kBucket - 1)) == kBucket - 1) s.halo[(pj >> kBucketLog) + 1] = Lj;
            b1 = pj >> kSuperLog;
            ent[j] = ((pj & (kSuper - 1)) << 12) | field;
        }
        const uint32_t slot = run_slot(P.hist, b1, ok);     // the pairs come in runs of one super-bucket
        key[j] = ok ? ((b1 << 16) | slot) : 0xffffffffu;
    }
    const bool all_valid = __syncthreads_and(cnt == kPartRound && !bad) != 0;
    return bad | level1_write(P, nb, s, ent, key, all_valid, over);
}

// Level 1: Lemma 1 in rank order.  Each CTA takes kPartRound consecutive
// ranks r, forms <sa[r], max(lcp[r], lcp[r+1])> and partitions these pairs
// into super-buckets of 2^20 positions (level1_write).  What bounds it:
// shared-memory wavefronts (84 % of the load/store pipe's rate: the counting
// atomics, the staging stores and the look-ups of staging offsets hit random
// banks).  2^26 positions of English take 207 us (2.6 instructions per
// position); 231 us with every entry checked, 4-byte shared loads and the
// bucket ids in an array of their own.
template <bool kBatch>
__global__ void __launch_bounds__(kPartThreads, kPartBlocks)
k_part1(const int32_t* __restrict__ sa, const int32_t* __restrict__ lcp, int32_t n, Scratch s, Segs segs, int tma) {
    begin_after();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned long long load_bar, load_bar2;
    const int nb = (int)s.nsupers;                    // <= 2048
    const PartSmem P = part_smem(smem_raw, nb);
    const long long r0 = (long long)blockIdx.x * kPartRound;
    // Full rounds (16-byte-aligned inputs) arrive by two bulk copies issued
    // before anything else: of a single string, every round but the last.
    // Of a batch, every full round's sa slice (flattened like the positions)
    // at once, on its own barrier, and then the lcp slice of a round that
    // lies inside one string, copied from the 16-byte boundary at or below
    // its first entry (shift entries earlier).  Other rounds load per thread.
    const int32_t* Ssa = reinterpret_cast<const int32_t*>(smem_raw + part_load_offset(nb));
    const int32_t* Slcp = Ssa + kPartRound;
    __shared__ int bulk_s, shift_s, sab_s, over_s;
    __shared__ long long bbase_s, bnj_s;          // batch round: its string's offset and length
    if (threadIdx.x == 0) {
        int bk = 0, shift = 0, sab = 0;
        long long lsrc = r0, cnt = kPartRound + 4;    // lcp entries copied
        if constexpr (!kBatch) {
            bk = tma && r0 + kPartRound + 4 <= (long long)n + 1;
            if (bk) {
                mbar_init(&load_bar, 1);
                mbar_fence_init();
                mbar_arrive_tx(&load_bar, (unsigned)(kPartRound * 4 + cnt * 4));
                bulk_g2s(const_cast<int32_t*>(Ssa), sa + r0, kPartRound * 4, &load_bar);
                bulk_g2s(const_cast<int32_t*>(Slcp), lcp + lsrc, (unsigned)(cnt * 4), &load_bar);
            }
        } else if (tma && r0 + kPartRound <= (long long)n) {
            sab = 1;
            mbar_init(&load_bar, 1);
            mbar_init(&load_bar2, 1);
            mbar_fence_init();
            mbar_arrive_tx(&load_bar, (unsigned)(kPartRound * 4));
            bulk_g2s(const_cast<int32_t*>(Ssa), sa + r0, kPartRound * 4, &load_bar);
            if (r0 + kPartRound < (long long)n) {
                // the round lies inside one string when the string holding
                // its first position also holds the next round's first
                // position (two independent loads; the string's offsets come
                // from warp 1)
                const long long t0 = r0 / kTile;
                const long long j = s.tile_seg[t0], jn = s.tile_seg[t0 + kPartRound / kTile];
                const long long l0 = r0 + j;          // the round's first lcp entry
                lsrc = l0 & ~3LL;
                cnt = (l0 + kPartRound + 1 - lsrc + 3) & ~3LL;
                if (j >= 0 && j < segs.num && jn == j && lsrc >= 0 && lsrc + cnt <= (long long)n + segs.num) {
                    bk = 1;
                    shift = (int)(l0 - lsrc);
                    mbar_arrive_tx(&load_bar2, (unsigned)(cnt * 4));
                    bulk_g2s(const_cast<int32_t*>(Slcp), lcp + lsrc, (unsigned)(cnt * 4), &load_bar2);
                }
            }
        }
        over_s = 0;
        bulk_s = bk;
        shift_s = shift;
        sab_s = sab;
    }
    if constexpr (kBatch) {
        // the string of a round that may arrive by bulk copies: its offset
        // and length, zero when the offset table contradicts the round (every
        // entry then fails its checks below)
        if (threadIdx.x == kWarp && tma && r0 + kPartRound < (long long)n) {
            const long long j = s.tile_seg[r0 / kTile];
            long long b0 = 0, b1 = 0;
            if (j >= 0 && j < segs.num) { b0 = __ldg(segs.off + j); b1 = __ldg(segs.off + j + 1); }
            const bool ok = b0 >= 0 && b0 <= r0 && b1 > r0 + kPartRound && b1 <= (long long)n;
            bbase_s = ok ? b0 : 0;
            bnj_s = ok ? b1 - b0 : 0;
        }
    }
    for (int b = threadIdx.x; b < nb; b += kPartThreads) P.hist[b] = 0;
    // a round across strings copies no lcp slice: its string offsets use
    // the lcp part of the bulk-copy area (read only before the stage area is
    // written)
    static_assert((kSegCap + 1) * 8 <= kPartLcpCap * 4, "string offsets must fit the lcp copy area");
    long long* seg_sh = reinterpret_cast<long long*>(const_cast<int32_t*>(Slcp));
    SegView sv{};
    __syncthreads();
    const bool bulk = bulk_s != 0;
    const int shift = shift_s;
    // a round across string boundaries looks its strings up per entry
    if constexpr (kBatch) {
        if (!bulk) sv.stage(segs, s, r0, (r0 + kPartRound < n) ? r0 + kPartRound : n, seg_sh);
    }
    // bulk round of a batch: its string's offset and length (the string
    // goes on past the round, so only its first rank can lie in the round)
    uint32_t bbase = 0, bnj = 0;
    if constexpr (kBatch) {
        if (bulk) { bbase = (uint32_t)bbase_s; bnj = (uint32_t)bnj_s; }
    }
    unsigned bad = 0;
    if (!kBatch && blockIdx.x == 0 && threadIdx.x == 0 && (__ldg(lcp) != 0 || __ldg(lcp + n) != 0)) bad = 1;
    // In a batch, flattened rank index r of string j is local rank
    // r - off[j]; its suffix starts at off[j] + sa[r] and its lcp pair is at
    // lcp[off[j] + j + (r - off[j]) ..].  Positions are flattened.
    uint32_t p[kPartPer];
    int32_t L[kPartPer];
    long long hint = kBatch ? sv.j0 : 0;
    const bool sab = kBatch ? sab_s != 0 : bulk;      // sa of the round in shared memory
    bool landed = true;                               // false: the copies never landed (reported; load nothing)
    if (sab && !mbar_wait(&load_bar, 0)) landed = false;
    if (kBatch && bulk && landed && !mbar_wait(&load_bar2, 0)) landed = false;
    if (!landed && threadIdx.x == 0) report(s, kErrTimeout);
    if (bulk) {
        // four consecutive ranks per thread and group: sa by one 16-byte
        // load, the five lcp words from the two 16-byte loads around them
        const uint32_t lim = kBatch ? bnj : (uint32_t)n;      // positions of the round's string
#pragma unroll
        for (int g = 0; g < kPartPer / 4; ++g) {
            const int x = (g * kPartThreads + (int)threadIdx.x) * 4;
            const int4 sv = *reinterpret_cast<const int4*>(Ssa + x);
            const int4 wa = *reinterpret_cast<const int4*>(Slcp + x);
            int32_t w0 = wa.x, w1 = wa.y, w2 = wa.z, w3 = wa.w, w4;
            if constexpr (!kBatch) {                          // the next lane's first word
                w4 = __shfl_down_sync(kFull, wa.x, 1);
                if ((threadIdx.x & 31) == 31) w4 = Slcp[x + 4];
            } else {
                const int4 wb = *reinterpret_cast<const int4*>(Slcp + x + 4);
                w4 = wb.x;
                if (shift == 1) { w0 = wa.y; w1 = wa.z; w2 = wa.w; w3 = wb.x; w4 = wb.y; }
                else if (shift == 2) { w0 = wa.z; w1 = wa.w; w2 = wb.x; w3 = wb.y; w4 = wb.z; }
                else if (shift == 3) { w0 = wa.w; w1 = wb.x; w2 = wb.y; w3 = wb.z; w4 = wb.w; }
                if (x == 0 && (long long)bbase == r0 && bnj != 0 && w0 != 0) bad = 1;   // lcp sentinel
            }
            const uint32_t pl[4] = {(uint32_t)sv.x, (uint32_t)sv.y, (uint32_t)sv.z, (uint32_t)sv.w};
            const int32_t Lv[4] = {max(w0, w1), max(w1, w2), max(w2, w3), max(w3, w4)};
#pragma unroll
            for (int c = 0; c < 4; ++c) {
                // negative lengths are too long as unsigned ones
                const bool in = landed && pl[c] < lim, fit = (uint32_t)Lv[c] <= lim - pl[c];
                if (!(in && fit)) bad = 1;
                p[g * 4 + c] = in ? bbase + pl[c] : 0xffffffffu;
                L[g * 4 + c] = fit ? Lv[c] : 0;
            }
        }
    } else {
#pragma unroll
        for (int j = 0; j < kPartPer; ++j) {
            const long long r = r0 + (long long)j * kPartThreads + threadIdx.x;
            p[j] = 0xffffffffu;
            L[j] = 0;
            if (r >= n) continue;
            if (sab && !landed) continue;
            uint32_t pl = sab ? (uint32_t)Ssa[j * kPartThreads + (int)threadIdx.x] : (uint32_t)__ldcs(sa + r);
            long long base = 0, nj = n, lidx = r;
            if constexpr (kBatch) {
                hint = sv.find(r, hint);
                base = sv.at(hint);
                nj = sv.at(hint + 1) - base;
                lidx = r + hint;
                if (base < 0 || nj < 1 || base + nj > n || r < base) { bad = 1; continue; }   // bad offset table
            }
            const int32_t a = __ldcs(lcp + lidx), c = __ldg(lcp + lidx + 1);
            if (kBatch && ((r == base && a != 0) || (r == base + nj - 1 && c != 0))) bad = 1;   // lcp sentinels
            int32_t Lj = a > c ? a : c;
            if (pl >= (uint32_t)nj) { bad = 1; continue; }
            if (Lj < 0 || (long long)Lj > nj - pl) { bad = 1; Lj = 0; }
            p[j] = (uint32_t)(base + pl);
            L[j] = Lj;
        }
    }
    // the steps of level1_scatter, with one shared atomic per entry (pairs in
    // rank order come in no runs)
    uint32_t ent[kPartPer], key[kPartPer];          // key: bucket << 16 | slot, or ~0u
    bool valid = true;
#pragma unroll
    for (int j = 0; j < kPartPer; ++j) {
        const uint32_t pj = p[j];
        key[j] = 0xffffffffu;
        if (pj >= (uint32_t)n) { valid = false; continue; }
        const int32_t Lj = L[j];
        uint32_t field = (uint32_t)Lj;
        if (field >= kEsc12) { field = kEsc12; s.lbig[pj] = Lj; }
        if ((pj & (kBucket - 1)) == kBucket - 1) s.halo[(pj >> kBucketLog) + 1] = Lj;
        const uint32_t b1 = pj >> kSuperLog;
        ent[j] = (pj << 12) | field;
        key[j] = (b1 << 16) | atomicAdd(&P.hist[b1], 1u);
    }
    const bool all_valid = __syncthreads_and(valid) != 0;
    bad |= level1_write(P, nb, s, ent, key, all_valid, &over_s);
    if (bad) report(s, kErrInput);
}

// Rank-window front end (rank without sa, one string of 2^24 positions or
// more).  Lemma 1 in text order, max(lcp[rank[i]], lcp[rank[i] + 1]), makes
// k_gather read one random lcp sector per position from HBM.  Here
// k_rank_win first partitions the pairs <rank[i], i> by rank into windows
// of 2^22 ranks (8-byte entries rank << 32 | i, in the compact LLR region,
// which is idle until k_bucket_llr).  k_part1_win then takes kPartRound
// pairs of one window per CTA, gathers their two lcp words from the
// window's 16 MB slice of lcp (CTAs run in window order, so the slice stays
// in L2 while its window is processed) and partitions <i, L_i> into the
// level-1 super-buckets like k_part1.  k_part2 and k_bucket_llr follow
// unchanged.  2^26 positions of English: k_rank_win 226 us (245 with window
// ids staged beside the pairs, shared-memory wavefronts 72 %), k_part1_win
// 490 us (waits on the scattered L2 reads of lcp).
__host__ __device__ inline size_t win_stage_offset(int nw) { return ((size_t)(2 * nw + 1) * 4 + 15) & ~(size_t)15; }
size_t rank_win_smem_bytes(int nw) { return win_stage_offset(nw) + (size_t)kPartRound * 8; }
size_t part_scatter_smem_bytes(int nb) { return part_stage_offset(nb) + (size_t)kPartRound * 8; }

__global__ void __launch_bounds__(kPartThreads, kPartBlocks)
k_rank_win(const int32_t* __restrict__ rank, int32_t n, Scratch s, int tma) {
    begin_after();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned long long load_bar;
    __shared__ int over_s;                            // not read: every window index is checked below
    const int nw = (int)s.nwins;                      // <= kMaxWins
    const PartSmem P = part_smem(smem_raw, nw);       // counters; the stage area is the 8-byte one below
    unsigned long long* stage = reinterpret_cast<unsigned long long*>(smem_raw + win_stage_offset(nw));
    // a full round's ranks arrive by one bulk copy into the stage area,
    // which is written only after every thread has read its ranks
    const int32_t* Srk = reinterpret_cast<const int32_t*>(stage);
    const long long i0 = (long long)blockIdx.x * kPartRound;
    const bool bulk = tma && i0 + kPartRound <= (long long)n;
    if (threadIdx.x == 0 && bulk) {
        mbar_init(&load_bar, 1);
        mbar_fence_init();
        mbar_arrive_tx(&load_bar, (unsigned)(kPartRound * 4));
        bulk_g2s(const_cast<int32_t*>(Srk), rank + i0, kPartRound * 4, &load_bar);
    }
    for (int b = threadIdx.x; b < nw; b += kPartThreads) P.hist[b] = 0;
    __syncthreads();
    unsigned bad = 0;
    bool landed = true;                               // false: the copy never landed (reported; load nothing)
    if (bulk && !mbar_wait(&load_bar, 0)) {
        landed = false;
        if (threadIdx.x == 0) report(s, kErrTimeout);
    }
    uint32_t rk[kPartPer], key[kPartPer];             // key: window << 16 | slot, or ~0u
#pragma unroll
    for (int j = 0; j < kPartPer; ++j) {
        const long long i = i0 + (long long)j * kPartThreads + threadIdx.x;
        key[j] = 0xffffffffu;
        rk[j] = 0;
        if (i >= n || !landed) continue;
        const uint32_t r = bulk ? (uint32_t)Srk[j * kPartThreads + threadIdx.x] : (uint32_t)__ldcs(rank + i);
        if (r >= (uint32_t)n) { bad = 1; continue; }
        const uint32_t w = r >> kWinLog;
        rk[j] = r;
        key[j] = (w << 16) | atomicAdd(&P.hist[w], 1u);
    }
    __syncthreads();
    if (nw <= 2 * kWarp) part_reserve_w<2>(P, nw, nw, s.cursor_w, kWinLog, &over_s);
    else part_reserve(P, nw, s.cursor_w, kWinLog, &over_s);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < kPartPer; ++j) {
        if (key[j] == 0xffffffffu) continue;
        const uint32_t w = key[j] >> 16;
        const uint32_t o = P.loff[w] + (key[j] & 0xffffu);
        stage[o] = ((unsigned long long)rk[j] << 32) | (uint32_t)(i0 + j * kPartThreads + threadIdx.x);
    }
    __syncthreads();
    const uint32_t total = P.loff[nw];
    for (uint32_t t = threadIdx.x; t < total; t += kPartThreads) {
        const unsigned long long e = stage[t];
        const uint32_t w = (uint32_t)(e >> 32) >> kWinLog, idx = P.base[w] + t;
        if (idx - (w << kWinLog) < (1u << kWinLog) && idx < (uint32_t)n) s.went[idx] = e;
        else bad = 1;                                 // a window overflows: rank is not a permutation
    }
    if (bad) report(s, kErrInput);
}

// The pair lcp[i], lcp[i + 1] of a random i by one 16-byte load where both lie
// in one 16-byte word of memory (three of four i) that ends inside the array
// (`last`: its last index), else by two 4-byte loads (rank-window phase at
// 8 x 10^7 positions of English 1.116 against 1.155 ms).
__device__ __forceinline__ void lcp_pair(const int32_t* __restrict__ lcp, long long i, long long last, int32_t& a, int32_t& b) {
    const int32_t* p = lcp + i;
    const int q = (int)(((uintptr_t)p >> 2) & 3u);    // word of the 16 bytes p lies in
    if (q < 3 && i - q >= 0 && i - q + 3 <= last) {
        const int4 v = __ldg(reinterpret_cast<const int4*>(p - q));
        a = q == 0 ? v.x : (q == 1 ? v.y : v.z);
        b = q == 0 ? v.y : (q == 1 ? v.z : v.w);
    } else {
        a = __ldg(p);
        b = __ldg(p + 1);
    }
}

__global__ void __launch_bounds__(kPartThreads, kPartBlocks)
k_part1_win(const int32_t* __restrict__ lcp, int32_t n, Scratch s) {
    begin_after();
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int nb = (int)s.nsupers;
    const PartSmem P = part_smem(smem_raw, nb);
    constexpr int kRoundsPerWin = (1 << kWinLog) / kPartRound;
    const long long w = blockIdx.x / kRoundsPerWin;
    const int q = blockIdx.x % kRoundsPerWin;
    const uint32_t fill = __ldcg(s.cursor_w + (size_t)w * kCursorStride);
    const long long wsize = ((long long)n - (w << kWinLog) < (1LL << kWinLog)) ? (long long)n - (w << kWinLog)
                                                                                : (1LL << kWinLog);
    __shared__ int over_s;
    if (threadIdx.x == 0) over_s = 0;
    for (int b = threadIdx.x; b < nb; b += kPartThreads) P.hist[b] = 0;
    unsigned bad = 0;
    if (q == 0 && threadIdx.x == 0) {
        if ((long long)fill != wsize) bad = 1;                  // rank is not a permutation
        if (w == 0 && (__ldg(lcp) != 0 || __ldg(lcp + n) != 0)) bad = 1;   // lcp sentinels
    }
    __syncthreads();
    const long long lim = (long long)fill < wsize ? (long long)fill : wsize;
    const long long e0 = (long long)q * kPartRound;
    if (e0 >= lim) {                                  // uniform over the CTA
        if (bad) report(s, kErrInput);
        return;
    }
    const int cnt = (int)(lim - e0 < kPartRound ? lim - e0 : kPartRound);
    const unsigned long long* src = s.went + (w << kWinLog) + e0;
    uint32_t p[kPartPer];
    int32_t L[kPartPer];
#pragma unroll
    for (int j = 0; j < kPartPer; ++j) {              // all pairs in flight first: p = i, L = rank
        const int x = j * kPartThreads + (int)threadIdx.x;
        const unsigned long long e = (x < cnt) ? __ldcs(src + x) : 0xffffffffull;
        p[j] = (uint32_t)e;
        L[j] = (int32_t)(e >> 32);
    }
#pragma unroll
    for (int j = 0; j < kPartPer; ++j) {
        const int x = j * kPartThreads + (int)threadIdx.x;
        if (x >= cnt) continue;
        const uint32_t i = p[j], r = (uint32_t)L[j];
        if (i >= (uint32_t)n || r >= (uint32_t)n) { bad = 1; p[j] = 0xffffffffu; L[j] = 0; continue; }
        int32_t a, c;
        lcp_pair(lcp, r, n, a, c);
        int32_t Lj = a > c ? a : c;
        if (Lj < 0 || (long long)Lj > (long long)n - i) { bad = 1; Lj = 0; }
        L[j] = Lj;
    }
    bad |= level1_scatter(P, nb, s, n, p, L, cnt, &over_s);
    if (bad) report(s, kErrInput);
}

// Level 2: rounds of kPartRound entries of one super-bucket, split into its
// kSubPerSuper buckets the same way.  The entries stay as they are: a
// bucket's CTA reads the position mod 2^15 from them.  CTAs stay and take
// every gridDim.x-th round; the next round's entries arrive by a bulk copy
// while this one is counted, staged and written.  Bound by shared-memory
// wavefronts like k_part1 (81 %): 2^26 positions of English take 117 us (0.93
// instructions per entry), 151 with every entry checked and the ids staged.
// kRuns: slots by run_slot, for level-1 entries that come clustered by
// bucket (those of the rank-window front end).
template <bool kRuns>
__global__ void __launch_bounds__(kPartThreads, kPartBlocks)
k_part2(int32_t n, Scratch s, int rounds) {
    begin_after();
    __shared__ __align__(16) uint32_t load[kPartRound];
    __shared__ __align__(16) uint32_t stage_s[kPartRound];
    uint32_t* const stage = opaque(stage_s);
    __shared__ uint32_t cnt_s[2][kSubPerSuper + 1];     // counts, then staging offsets, of this round and the next
    __shared__ uint32_t base_s[kSubPerSuper];
    __shared__ int over_s;
    __shared__ unsigned long long load_bar;
    constexpr int kChunksPerSuper = kSuper / kPartRound;
    const int tid = threadIdx.x;
    int c = blockIdx.x;
    if (c >= rounds) return;
    uint32_t fill = __ldcg(s.cursor1 + (size_t)(c / kChunksPerSuper) * kCursorStride);
    if (tid == 0) {
        mbar_init(&load_bar, 1);
        mbar_fence_init();
        mbar_arrive_tx(&load_bar, kPartRound * 4);
        bulk_g2s(load, s.ent1 + (size_t)c * kPartRound, kPartRound * 4, &load_bar);
    }
    if (tid < 2 * (kSubPerSuper + 1)) cnt_s[0][tid] = 0;
    __syncthreads();
    unsigned bad = 0;
    for (int it = 0; c < rounds; ++it) {
        const int b1 = c / kChunksPerSuper, q = c % kChunksPerSuper, next = c + (int)gridDim.x;
        const long long bb = (long long)b1 * kSubPerSuper;
        const int nsub = (int)((s.nbuckets - bb < kSubPerSuper) ? s.nbuckets - bb : kSubPerSuper);
        const uint32_t i0 = (uint32_t)q * kPartRound;
        const bool full = i0 + kPartRound <= fill;
        if (q == 0 && tid == 0) {
            const long long want = ((long long)n - (long long)b1 * kSuper < kSuper) ? (long long)n - (long long)b1 * kSuper : kSuper;
            if ((long long)fill != want) bad = 1;
        }
        PartSmem P;
        P.hist = P.loff = cnt_s[it & 1];
        P.base = base_s;
        const bool landed = mbar_wait(&load_bar, it & 1);
        uint32_t ent[kPartPer], slot[kPartPer];
        if (full) {                                     // four consecutive entries per load
#pragma unroll
            for (int g = 0; g < kPartPer / 4; ++g) {
                const uint4 v = reinterpret_cast<const uint4*>(load)[g * kPartThreads + tid];
                ent[4 * g] = v.x; ent[4 * g + 1] = v.y; ent[4 * g + 2] = v.z; ent[4 * g + 3] = v.w;
            }
#pragma unroll
            for (int j = 0; j < kPartPer; ++j)
                slot[j] = kRuns ? run_slot(P.hist, ent[j] >> 27, true) : atomicAdd(&P.hist[ent[j] >> 27], 1u);
        } else {
#pragma unroll
            for (int j = 0; j < kPartPer; ++j) {
                const uint32_t i = j * kPartThreads + tid;
                const bool in = i0 + i < fill;
                ent[j] = in ? load[i] : 0u;
                const bool ok = in && (int)(ent[j] >> 27) < nsub;   // a position at or past the last bucket: reported
                if (in && !ok) bad = 1;
                slot[j] = 0xffffffffu;
                if (kRuns) {
                    const uint32_t t = run_slot(P.hist, ent[j] >> 27, ok);
                    if (ok) slot[j] = t;
                } else if (ok) {
                    slot[j] = atomicAdd(&P.hist[ent[j] >> 27], 1u);
                }
            }
        }
        if (__syncthreads_or(!landed)) {                // the copy never landed: reported, nothing more is loaded
            if (tid == 0) report(s, kErrTimeout);
            break;
        }
        if (tid == kPartThreads - 1 && next < rounds) {
            fence_proxy_async_smem();
            mbar_arrive_tx(&load_bar, kPartRound * 4);
            bulk_g2s(load, s.ent1 + (size_t)next * kPartRound, kPartRound * 4, &load_bar);
        }
        if (next < rounds) fill = __ldcg(s.cursor1 + (size_t)(next / kChunksPerSuper) * kCursorStride);
        if (tid < kWarp) {
            if (tid == 0) over_s = 0;
            __syncwarp();
            if (full && tid >= nsub && P.hist[tid]) over_s = 1;
        }
        part_reserve_w<1>(P, kSubPerSuper, nsub, s.cursor2 + (size_t)bb * kCursorStride, kBucketLog, &over_s);
        __syncthreads();
        if (tid <= kSubPerSuper) cnt_s[(it & 1) ^ 1][tid] = 0;
#pragma unroll
        for (int j = 0; j < kPartPer; ++j)
            if (full || slot[j] != 0xffffffffu) stage[P.loff[ent[j] >> 27] + slot[j]] = ent[j];
        const uint32_t total = P.loff[kSubPerSuper];
        __syncthreads();
        uint32_t* dst = s.ent2 + ((size_t)bb << kBucketLog);
        if (full && over_s == 0) {
#pragma unroll
            for (int j = 0; j < kPartPer; ++j) {
                const uint32_t i = j * kPartThreads + tid;
                const uint32_t e = stage[i];
                dst[P.base[e >> 27] + i] = e;
            }
        } else {
            for (uint32_t i = tid; i < total; i += kPartThreads) {
                const uint32_t e = stage[i], b2 = e >> 27, idx = P.base[b2] + i;
                if ((int)b2 < nsub && idx - (b2 << kBucketLog) < (uint32_t)kBucket) dst[idx] = e;
                else bad = 1;
            }
        }
        c = next;
    }
    if (bad) report(s, kErrInput);
}

// K1 (Sec. 4.2.1) on 2-byte length words: each warp owns kPerWarp chunks of
// 256 consecutive positions from position x0 on, eight consecutive positions
// per lane.  One 16-byte load gives a lane its words, the flags are sign bits
// shifted together (first position in the top bit).  W gives plain words:
// load8(q, x) for positions x .. x + 7 of a lane in its warp's chunk q, and
// at(x); below W::kEsc a word is the length, W::kEsc itself stands for a longer
// one (in lbig), anything above for a position that got no length (reported:
// sa gave another one twice).
// `halo`: the length of the position before 0 (used where x0 is 0).
constexpr int kBktChunk = 256;                                   // = kSeg: seg_cbase falls out of the chunk counts
static_assert(kBktChunk == kSeg, "chunk and segment sizes");

// L of position x of a tile, 0 <= x < cnt, whose word is f; a position without a length counts as 0
template <class W>
__device__ __forceinline__ int32_t word_len(uint32_t f, int x, const int32_t* lbig) {
    return f < W::kEsc ? (int32_t)f : (f == W::kEsc ? __ldcg(lbig + x) : 0);
}
template <class W>
__device__ __forceinline__ int32_t llr_len(const W& words, int x, const int32_t* lbig) {
    return word_len<W>(words.at(x), x, lbig);
}

template <int kPerWarp, class W>
__device__ __forceinline__ void llr_flags(const W& words, int x0, int cnt, int32_t halo, const int32_t* lbig,
                                          uint32_t (&flags)[(kPerWarp + 3) / 4], int32_t* counts, unsigned& bad) {
    const int lane = lane_id();
    uint32_t last = 0;                                       // word of the position before the chunk
    if (x0 == 0) last = min((uint32_t)halo, W::kEsc);
    else if (x0 - 1 < cnt) last = min(words.at(x0 - 1), W::kEsc);
#pragma unroll
    for (int q = 0; q < kPerWarp; ++q) {
        const int x = x0 + q * kBktChunk + lane * 8;
        const uint4 w = words.load8(q, x);
        const uint32_t m = __vmaxu2(__vmaxu2(w.x, w.y), __vmaxu2(w.z, w.w));
        const bool odd = (m & 0xffffu) >= W::kEsc || (m >> 16) >= W::kEsc;
        uint32_t prev = __shfl_up_sync(kFull, w.w >> 16, 1);
        if (lane == 0) prev = last;
        last = min(__shfl_sync(kFull, w.w >> 16, kWarp - 1), W::kEsc);
        uint32_t f = 0;
        if (__any_sync(kFull, odd || x + 8 > cnt)) {
            // a length from lbig, a position without one or past the end
            int32_t before = x > 0 ? (x - 1 < cnt ? llr_len(words, x - 1, lbig) : 0) : halo;
            for (int j = 0; j < 8; ++j) {
                const bool in = x + j < cnt;
                if (in && words.at(x + j) > W::kEsc) bad = 1;
                const int32_t l = in ? llr_len(words, x + j, lbig) : 0;
                f = 2 * f + (l > 0 && l >= before);
                before = l;
            }
        } else {
            const uint32_t l[8] = {w.x & 0xffffu, w.x >> 16, w.y & 0xffffu, w.y >> 16,
                                   w.z & 0xffffu, w.z >> 16, w.w & 0xffffu, w.w >> 16};
#pragma unroll
            for (int j = 0; j < 8; ++j) {                     // sign of l - max(prev, 1): 1 = dropped
                f = __funnelshift_l(l[j] - max(prev, 1u), f, 1);
                prev = l[j];
            }
            f ^= 0xffu;
        }
        flags[q / 4] |= (f & 0xffu) << (8 * (q % 4));
        const int c = (int)__reduce_add_sync(kFull, (unsigned)__popc(f & 0xffu));
        if (lane == 0) counts[q] = c;
    }
}

// K3: a chunk's kept positions are listed in shared memory (mine, kBktChunk
// entries per warp) and then written to LLRc in one run.  W::List holds the
// position, or the position << 16 | its word where the words are not in shared
// memory (5 x 10^4 positions: k_compact 8.7 us; 10.4 where it read each word
// again before the entry's stores).
template <int kPerWarp, class W>
__device__ __forceinline__ void llr_write(const W& words, int x0, long long k0, const int32_t* lbig,
                                          const uint32_t (&flags)[(kPerWarp + 3) / 4], const int32_t* offs, long long base,
                                          typename W::List* mine, const Scratch& s) {
    constexpr bool kListed = sizeof(typename W::List) == 4;
    const int lane = lane_id();
#pragma unroll
    for (int q = 0; q < kPerWarp; ++q) {
        const int x = x0 + q * kBktChunk + lane * 8;
        const uint32_t f = (flags[q / 4] >> (8 * (q % 4))) & 0xffu;
        const int c = __popc(f);
        const int incl = warp_incl_scan(c);
        int o = incl - c;
        uint4 w = make_uint4(0, 0, 0, 0);
        if constexpr (kListed) w = words.load8(q, x);
        const uint32_t l[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int j = 0; j < 8; ++j)
            if (f & (0x80u >> j))
                mine[o++] = (typename W::List)(kListed ? ((uint32_t)(x + j) << 16) | ((l[j / 2] >> (16 * (j & 1))) & 0xffffu)
                                                       : (uint32_t)(x + j));
        const int tot = __shfl_sync(kFull, incl, kWarp - 1);
        __syncwarp();
        const long long to = base + offs[q];
        for (int i = lane; i < tot; i += kWarp) {
            const uint32_t e = mine[i];
            const int y = (int)(kListed ? e >> 16 : e);
            const int32_t k = (int32_t)(k0 + y);
            s.cstart[to + i] = k;
            s.cend[to + i] = k + word_len<W>(kListed ? e & 0xffffu : words.at(y), y, lbig) - 1;
        }
        __syncwarp();
    }
}

// Exclusive scan of a tile's kChunks chunk counts and the tile's place in
// LLRc (K2, look-back), by one warp; *total the tile's count.
template <int kChunks>
__device__ __forceinline__ long long llr_place(int32_t* counts, unsigned long long* status, long long tile,
                                               const Scratch& s, int32_t* total) {
    const int lane = lane_id();
    constexpr int kPer = (kChunks + kWarp - 1) / kWarp;
    int a[kPer], sum = 0;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int i = lane * kPer + u;
        a[u] = i < kChunks ? counts[i] : 0;
        sum += a[u];
    }
    const int incl = warp_incl_scan(sum);
    int ex = incl - sum;
#pragma unroll
    for (int u = 0; u < kPer; ++u) {
        const int i = lane * kPer + u;
        if (i < kChunks) counts[i] = ex;
        ex += a[u];
    }
    *total = __shfl_sync(kFull, incl, kWarp - 1);
    return lookback_exclusive(status, tile, *total, s.err, s.spin_limit);
}

// First LLRc entry of each tile of kTile positions and of each segment of
// kSeg positions of a tile of kChunks chunks (whole CTA).
template <int kChunks>
__device__ __forceinline__ void llr_bases(long long tile, const int32_t* offs, long long base, int32_t total,
                                          const Scratch& s) {
    const int i = threadIdx.x;
    if (i >= kChunks) return;
    const long long sg = tile * kChunks + i;
    const int32_t at = (int32_t)(base + offs[i]);
    if (sg < s.nsegs) s.seg_cbase[sg] = at;
    if (sg == s.nsegs - 1) s.seg_cbase[s.nsegs] = (int32_t)(base + total);
    constexpr int kPerTile = kTile / kBktChunk;
    if (i % kPerTile == 0) {
        const long long t = sg / kPerTile;
        if (t < s.ntiles) s.tile_cbase[t] = at;
        if (t == s.ntiles - 1) s.tile_cbase[s.ntiles] = (int32_t)(base + total);
    }
}

// One bucket of kBucket positions per CTA: lengths scattered into shared
// memory by position, then flags (K1), compaction (K2) and the bucket's place
// in LLRc by look-back (K3).
//
// A position's word is the low half of its entry: the 12-bit length field
// under the low four bits of the position.  XOR with those four bits (a
// constant pattern per eight positions) leaves the plain field, and anything
// else above bit 11 means that the position was never written (the words
// start with the four bits inverted).
//
// 2^26 positions of English take 114 us (67 M warp instructions); with a
// ballot per run of 32 positions and one store per flagged lane it was 190 us
// (156 M).  With the first entries loaded while the words are preset, 2^28
// positions take 421 us instead of 436.
__device__ __forceinline__ uint32_t bucket_pattern(int x, int pair) {   // position bits of words x + 2 pair, x + 2 pair + 1
    const uint32_t lo = (uint32_t)((x & 8) + 2 * pair);
    return (lo << 12) | ((lo + 1) << 28);
}
struct BucketWords {
    static constexpr uint32_t kEsc = kEsc12;
    using List = uint16_t;
    const uint16_t* sL;
    __device__ __forceinline__ uint32_t at(int x) const { return (uint32_t)sL[x] ^ ((uint32_t)(x & 15) << 12); }
    __device__ __forceinline__ uint4 load8(int, int x) const {
        uint4 w = *reinterpret_cast<const uint4*>(sL + x);
        w.x ^= bucket_pattern(x, 0);
        w.y ^= bucket_pattern(x, 1);
        w.z ^= bucket_pattern(x, 2);
        w.w ^= bucket_pattern(x, 3);
        return w;
    }
};

__global__ void __launch_bounds__(kBucketThreads, 3)
k_bucket_llr(int32_t n, Scratch s) {
    begin_after();
    constexpr int kChunks = kBucket / kBktChunk;             // 128
    constexpr int kWarps = kBucketThreads / kWarp;           // 16
    constexpr int kPerWarp = kChunks / kWarps;               // 8
    extern __shared__ __align__(16) unsigned char smem_raw[];
    uint16_t* sL = reinterpret_cast<uint16_t*>(smem_raw);                        // kBucket words
    uint16_t* list = reinterpret_cast<uint16_t*>(smem_raw + kBucket * 2);        // kBktChunk kept positions per warp
    __shared__ int32_t ccnt[kChunks];
    __shared__ long long b_s, base_s;
    __shared__ int32_t total_s;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) b_s = atomicAdd(&s.tickets[1], 1u);
    __syncthreads();
    const long long b = b_s;
    const long long k0 = b * kBucket;
    const int cnt = (int)(((long long)n - k0 < kBucket) ? (long long)n - k0 : kBucket);
    // the bucket's first entries are on their way while its words are preset
    // (they are used only if the bucket is full)
    const uint32_t* ent = s.ent2 + ((size_t)b << kBucketLog);
    const uint32_t fill = __ldcg(s.cursor2 + (size_t)b * kCursorStride);
    constexpr int kUnroll = 2;                               // loads of four entries per batch; two batches in flight
    constexpr int kBatches = kBucket / 4 / (kBucketThreads * kUnroll);
    const uint4* src = reinterpret_cast<const uint4*>(ent) + tid;
    uint4 e[2][kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) e[0][u] = __ldcs(src + u * kBucketThreads);
    for (int i = tid; i < kBucket / 8; i += kBucketThreads) {
        uint4 u;
        u.x = bucket_pattern(8 * i, 0) ^ 0xf000f000u;
        u.y = bucket_pattern(8 * i, 1) ^ 0xf000f000u;
        u.z = bucket_pattern(8 * i, 2) ^ 0xf000f000u;
        u.w = bucket_pattern(8 * i, 3) ^ 0xf000f000u;
        reinterpret_cast<uint4*>(sL)[i] = u;
    }
    __syncthreads();

    // scatter the bucket's lengths into shared memory by position
    unsigned bad = fill != (uint32_t)cnt;
    const int nent = (int)(fill < (uint32_t)cnt ? fill : (uint32_t)cnt);
    if (nent == kBucket) {
#pragma unroll 2
        for (int t = 0; t < kBatches; ++t) {
            if (t + 1 < kBatches) {
#pragma unroll
                for (int u = 0; u < kUnroll; ++u) e[(t + 1) & 1][u] = __ldcs(src + ((t + 1) * kUnroll + u) * kBucketThreads);
            }
#pragma unroll
            for (int u = 0; u < kUnroll; ++u) {
                const uint4 v = e[t & 1][u];
                sL[(v.x >> 12) & (kBucket - 1)] = (uint16_t)v.x;
                sL[(v.y >> 12) & (kBucket - 1)] = (uint16_t)v.y;
                sL[(v.z >> 12) & (kBucket - 1)] = (uint16_t)v.z;
                sL[(v.w >> 12) & (kBucket - 1)] = (uint16_t)v.w;
            }
        }
    } else {
        for (int i = tid; i < nent; i += kBucketThreads) {
            const uint32_t v = __ldcs(ent + i), low = (v >> 12) & (kBucket - 1);
            if (low < (uint32_t)cnt) sL[low] = (uint16_t)v;
            else bad = 1;
        }
    }
    __syncthreads();
    const BucketWords words{sL};
    const int32_t* lbig = s.lbig + k0;
    const int x0 = warp * kPerWarp * kBktChunk;
    const int32_t halo = (x0 == 0 && k0 > 0) ? __ldcg(s.halo + b) : 0;
    uint32_t flags[(kPerWarp + 3) / 4] = {};
    llr_flags<kPerWarp>(words, x0, cnt, halo, lbig, flags, ccnt + warp * kPerWarp, bad);
    if (bad) report(s, kErrInput);
    __syncthreads();
    if (warp == 0) {
        int32_t total;
        const long long at = llr_place<kChunks>(ccnt, s.status_b, b, s, &total);
        if (lane == 0) { base_s = at; total_s = total; }
    }
    __syncthreads();
    llr_bases<kChunks>(b, ccnt, base_s, total_s, s);
    llr_write<kPerWarp>(words, x0, k0, lbig, flags, ccnt + warp * kPerWarp, base_s, list + warp * kBktChunk, s);
}

// ---------------------------------------------------------------------------
// dense front end
// ---------------------------------------------------------------------------

// Up to kDenseMaxN positions with sa, the lengths go straight to a 2-byte
// array in text order: k_scatter stores L_{sa[r]} at sa[r] (scattered stores
// into an array that stays in L2, where partial writes merge), k_compact reads
// it back tile by tile, flags and compacts it.  The array is preset (k_prep) to
// kDenseNone; a position that still has it afterwards means that sa gave
// another one twice.
constexpr uint32_t kDenseEsc = 0xfffeu;           // longer: the length is in lbig
constexpr uint32_t kDenseNone = 0xffffu;

// What must be clear before k_compact and the cover kernel: the tickets and
// the look-back words of this n (those of tile t).
__device__ __forceinline__ void clear_tickets(const Scratch& s) {
    for (int i = 0; i < 4; ++i) s.tickets[i] = 0;
}
__device__ __forceinline__ void clear_status(int32_t n, const Scratch& s, long long t) {
    s.status_g[t] = 0;
    s.status_o[t] = 0;
    if (t < num_seg_tiles(n)) s.status_w[t] = 0;
}

// The above and the dense array (kDenseNone); a batch's tile index as well.
// One launch instead of two memsets and k_seg_index.
__global__ void __launch_bounds__(256) k_prep(int32_t n, Scratch s, Segs segs, int fill) {
    begin_after();
    const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x, step = (long long)gridDim.x * blockDim.x;
    if (i0 == 0) clear_tickets(s);
    for (long long i = i0; i < s.ntiles; i += step) clear_status(n, s, i);
    constexpr uint32_t kTwo = kDenseNone | (kDenseNone << 16);
    const uint4 none = make_uint4(kTwo, kTwo, kTwo, kTwo);
    if (fill)
        for (long long i = i0; i < ((long long)n + 7) / 8; i += step) reinterpret_cast<uint4*>(s.dense)[i] = none;
    if (segs.num > 0) seg_index(n, s, segs, i0, step);
}

void launch_prep(int32_t n, const Scratch& s, const Segs& segs, bool fill, cudaStream_t stream) {
    k_prep<<<index_grid(fill ? ((long long)n + 7) / 8 : s.ntiles, segs), 256, 0, stream>>>(n, s, segs, fill ? 1 : 0);
}

template <bool kBatch>
__global__ void __launch_bounds__(kThreads) k_scatter(const int32_t* __restrict__ sa, const int32_t* __restrict__ lcp,
                                                      int32_t n, Scratch s, Segs segs) {
    begin_after();
    constexpr int kPer = kTile / kThreads;
    __shared__ long long seg_sh[kBatch ? kSegCap + 1 : 1];
    const int tid = threadIdx.x;
    const long long r0 = (long long)blockIdx.x * kTile;
    // the round's string, where it lies inside one (else looked up per entry)
    long long base = 0, nj = n, lbase = 0, hint = 0;
    bool direct = true;
    SegView sv{};
    if constexpr (kBatch) {
        const long long r1 = (r0 + kTile < n) ? r0 + kTile : n;
        sv.stage(segs, s, r0, r1, seg_sh);
        hint = sv.find(r0, sv.j0);
        base = sv.at(hint);
        const long long end = sv.at(hint + 1);
        nj = end - base;
        lbase = hint;
        direct = base >= 0 && base <= r0 && r1 <= end && end <= (long long)n;
    }
    unsigned bad = 0;
    if (!kBatch && blockIdx.x == 0 && tid == 0 && (__ldg(lcp) != 0 || __ldg(lcp + n) != 0)) bad = 1;
    auto put = [&](uint32_t pl, int32_t a, int32_t b, long long at, long long len) {
        int32_t L = a > b ? a : b;
        if ((long long)pl >= len) { bad = 1; return; }
        if (L < 0 || (long long)L > len - (long long)pl) { bad = 1; L = 0; }
        const long long p = at + pl;
        uint32_t w = (uint32_t)L;
        if (w >= kDenseEsc) { w = kDenseEsc; s.lbig[p] = L; }
        s.dense[p] = (uint16_t)w;
    };
    if (direct) {
        uint32_t v[kPer];
        int32_t a[kPer], b[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const long long r = r0 + j * kThreads + tid;
            v[j] = r < n ? (uint32_t)__ldcs(sa + r) : 0u;
            a[j] = r < n ? __ldg(lcp + lbase + r) : 0;
            b[j] = r < n ? __ldg(lcp + lbase + r + 1) : 0;
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const long long r = r0 + j * kThreads + tid;
            if (r >= n) continue;
            if (kBatch && ((r == base && a[j] != 0) || (r == base + nj - 1 && b[j] != 0))) bad = 1;   // lcp sentinels
            put(v[j], a[j], b[j], base, nj);
        }
    } else {
        for (int j = 0; j < kPer; ++j) {
            const long long r = r0 + j * kThreads + tid;
            if (r >= n) continue;
            hint = sv.find(r, hint);
            const long long at = sv.at(hint), len = sv.at(hint + 1) - at;
            if (at < 0 || len < 1 || at + len > n || r < at) { bad = 1; continue; }   // bad offset table
            const int32_t a = __ldg(lcp + r + hint), b = __ldg(lcp + r + hint + 1);
            if ((r == at && a != 0) || (r == at + len - 1 && b != 0)) bad = 1;        // lcp sentinels
            put((uint32_t)__ldcs(sa + r), a, b, at, len);
        }
    }
    if (bad) report(s, kErrInput);
}

// Lemma 1 in text order into the dense array (rank alone): rank is streamed,
// the two lcp words of each position are gathered, all loads of a thread in
// flight before the first is used; a tile across strings looks each
// position's string up.  What bounds it is the rate of scattered sector reads
// (1.1 per position).  6 x 10^6 positions of protein take 40 us here and 25 in
// k_compact; in one kernel that also flagged, compacted and looked back per
// 2048 positions, with 25 KB of shared memory, it was 71 us, and 180 instead
// of 154 us for 1.6 x 10^7.
template <bool kBatch>
__global__ void __launch_bounds__(kThreads) k_gather(const int32_t* __restrict__ rank, const int32_t* __restrict__ lcp,
                                                     int32_t n, Scratch s, Segs segs) {
    begin_after();
    constexpr int kPer = kTile / kThreads;
    __shared__ long long seg_sh[kBatch ? kSegCap + 1 : 1];
    const int tid = threadIdx.x;
    const long long k0 = (long long)blockIdx.x * kTile;
    // One string has no tile index to wait for, and what must be clear is
    // clear before the next kernel: each CTA clears its tile's status words,
    // without k_prep (2^20 positions, leftmost: 45 us, 48 with it).
    if (!kBatch && tid == 0) {
        const long long t = blockIdx.x;
        clear_status(n, s, t);
        if (t == 0) clear_tickets(s);
    }
    long long base = 0, nj = n, lbase = 0, hint = 0;
    bool direct = true;
    SegView sv{};
    if constexpr (kBatch) {
        const long long k1 = (k0 + kTile < n) ? k0 + kTile : n;
        sv.stage(segs, s, k0, k1, seg_sh);
        hint = sv.find(k0, sv.j0);
        base = sv.at(hint);
        const long long end = sv.at(hint + 1);
        nj = end - base;
        lbase = base + hint;
        direct = base >= 0 && base <= k0 && k1 <= end && end <= (long long)n;
    }
    // Invalid input is reported and clamped so every access stays in bounds.
    unsigned bad = 0;
    if (!kBatch && blockIdx.x == 0 && tid == 0 && (__ldg(lcp) != 0 || __ldg(lcp + n) != 0)) bad = 1;
    auto put = [&](long long k, int32_t a, int32_t b, long long at, long long len) {
        int32_t L = a > b ? a : b;
        if (L < 0 || (long long)L > len - (k - at)) { bad = 1; L = 0; }
        uint32_t w = (uint32_t)L;
        if (w >= kDenseEsc) { w = kDenseEsc; s.lbig[k] = L; }
        s.dense[k] = (uint16_t)w;
    };
    if (direct) {
        uint32_t r[kPer];
        int32_t a[kPer], b[kPer];
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const long long k = k0 + j * kThreads + tid;
            r[j] = (k < n) ? (uint32_t)__ldcs(rank + k) : 0u;
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const long long k = k0 + j * kThreads + tid;
            if (k < n && (long long)r[j] >= nj) { bad = 1; r[j] = 0; }
            a[j] = (k < n) ? __ldg(lcp + lbase + r[j]) : 0;
            b[j] = (k < n) ? __ldg(lcp + lbase + r[j] + 1) : 0;
        }
#pragma unroll
        for (int j = 0; j < kPer; ++j) {
            const long long k = k0 + j * kThreads + tid;
            if (k >= n) continue;
            if (kBatch && ((r[j] == 0 && a[j] != 0) || ((long long)r[j] == nj - 1 && b[j] != 0))) bad = 1;   // lcp sentinels
            put(k, a[j], b[j], base, nj);
        }
    } else {
        // across strings: kTogether positions at a time, each one's string
        // beside its rank (all eight: 70 registers instead of 40, and 3 % more
        // time where tiles lie inside strings)
        constexpr int kTogether = 2;
#pragma unroll 1
        for (int j0 = 0; j0 < kPer; j0 += kTogether) {
            uint32_t r[kTogether];
            int32_t str[kTogether], a[kTogether], b[kTogether];   // string, or -1: no position, or a bad offset table
#pragma unroll
            for (int j = 0; j < kTogether; ++j) {
                const long long k = k0 + (j0 + j) * kThreads + tid;
                if (k < n) hint = sv.find(k, hint);
                str[j] = k < n ? (int32_t)hint : -1;
                r[j] = k < n ? (uint32_t)__ldcs(rank + k) : 0u;
            }
#pragma unroll
            for (int j = 0; j < kTogether; ++j) {
                const long long k = k0 + (j0 + j) * kThreads + tid;
                a[j] = b[j] = 0;
                if (str[j] < 0) continue;
                const long long at = sv.at(str[j]), len = sv.at(str[j] + 1) - at;
                if (at < 0 || len < 1 || at + len > n || k < at) { bad = 1; s.dense[k] = 0; str[j] = -1; continue; }
                if ((long long)r[j] >= len) { bad = 1; r[j] = 0; }
                a[j] = __ldg(lcp + at + str[j] + r[j]);
                b[j] = __ldg(lcp + at + str[j] + r[j] + 1);
            }
#pragma unroll
            for (int j = 0; j < kTogether; ++j) {
                if (str[j] < 0) continue;
                const long long at = sv.at(str[j]), len = sv.at(str[j] + 1) - at;
                if ((r[j] == 0 && a[j] != 0) || ((long long)r[j] == len - 1 && b[j] != 0)) bad = 1;   // lcp sentinels
                put(k0 + (j0 + j) * kThreads + tid, a[j], b[j], at, len);
            }
        }
    }
    if (bad) report(s, kErrInput);
}

template <int kPerWarp>
struct DenseWords {
    static constexpr uint32_t kEsc = kDenseEsc;
    using List = uint32_t;
    const uint16_t* d;                            // of the tile's first position
    uint4 w[kPerWarp];                            // the lane's own words, kept from the one load of them
    __device__ __forceinline__ uint32_t at(int x) const { return __ldcg(d + x); }
    __device__ __forceinline__ uint4 load8(int q, int) const { return w[q]; }
};

constexpr int kCompactThreads = 512;
__global__ void __launch_bounds__(kCompactThreads) k_compact(int32_t n, Scratch s) {
    begin_after();
    constexpr int kChunks = kCompactTile / kBktChunk;        // 32
    constexpr int kWarps = kCompactThreads / kWarp;          // 16
    constexpr int kPerWarp = kChunks / kWarps;               // 2
    __shared__ uint32_t list[kWarps * kBktChunk];
    __shared__ int32_t ccnt[kChunks];
    __shared__ long long t_s, base_s;
    __shared__ int32_t total_s;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    if (tid == 0) t_s = atomicAdd(&s.tickets[1], 1u);
    __syncthreads();
    const long long t = t_s, k0 = t * kCompactTile;
    const int cnt = (int)(((long long)n - k0 < kCompactTile) ? (long long)n - k0 : kCompactTile);
    const int32_t* lbig = s.lbig + k0;
    const int x0 = warp * kPerWarp * kBktChunk;
    DenseWords<kPerWarp> words{s.dense + k0, {}};
#pragma unroll
    for (int q = 0; q < kPerWarp; ++q)
        words.w[q] = __ldcg(reinterpret_cast<const uint4*>(words.d + x0 + q * kBktChunk + lane * 8));
    const int32_t halo = (x0 == 0 && k0 > 0) ? llr_len(words, -1, lbig) : 0;
    unsigned bad = 0;
    uint32_t flags[1] = {};
    llr_flags<kPerWarp>(words, x0, cnt, halo, lbig, flags, ccnt + warp * kPerWarp, bad);
    if (bad) report(s, kErrInput);
    __syncthreads();
    if (warp == 0) {
        int32_t total;
        const long long at = llr_place<kChunks>(ccnt, s.status_g, t, s, &total);
        if (lane == 0) { base_s = at; total_s = total; }
    }
    __syncthreads();
    llr_bases<kChunks>(t, ccnt, base_s, total_s, s);
    llr_write<kPerWarp>(words, x0, k0, lbig, flags, ccnt + warp * kPerWarp, base_s, list + warp * kBktChunk, s);
}

void launch_scatter(const int32_t* sa, const int32_t* lcp, int32_t n, const Scratch& s, const Segs& segs,
                    cudaStream_t stream) {
    launch_after(segs.num > 0 ? k_scatter<true> : k_scatter<false>, (unsigned)s.ntiles, kThreads, 0, stream, sa, lcp, n, s,
                 segs);
}

void launch_gather(const int32_t* rank, const int32_t* lcp, int32_t n, const Scratch& s, const Segs& segs,
                   cudaStream_t stream) {
    if (segs.num > 0) launch_after(k_gather<true>, (unsigned)s.ntiles, kThreads, 0, stream, rank, lcp, n, s, segs);
    else k_gather<false><<<(unsigned)s.ntiles, kThreads, 0, stream>>>(rank, lcp, n, s, segs);   // the first kernel
}

void launch_compact(int32_t n, const Scratch& s, cudaStream_t stream) {
    const unsigned grid = (unsigned)(((long long)n + kCompactTile - 1) / kCompactTile);
    launch_after(k_compact, grid, kCompactThreads, 0, stream, n, s);
}

size_t bucket_smem_bytes() { return (size_t)kBucket * 2 + (size_t)(kBucketThreads / kWarp) * kBktChunk * 2; }

template <bool kRuns>
void launch_part2(int32_t n, const Scratch& s, cudaStream_t stream) {
    const int rounds = (int)(((long long)n + kPartRound - 1) / kPartRound);   // the entries of every super-bucket but the last fill it
    const int grid = rounds < kSms * kPartBlocks ? rounds : kSms * kPartBlocks;
    launch_after(k_part2<kRuns>, grid, kPartThreads, 0, stream, n, s, rounds);
}

void launch_partition(const int32_t* sa, const int32_t* lcp, int32_t n, const Scratch& s, const Segs& segs,
                      cudaStream_t stream) {
    const unsigned g1 = (unsigned)(((long long)n + kPartRound - 1) / kPartRound);
    // bulk copies need 16-byte-aligned sources
    const int tma = (((uintptr_t)sa | (uintptr_t)lcp) & 15u) == 0 ? 1 : 0;
    const size_t smem = part_smem_bytes((int)s.nsupers);
    if (segs.num > 0) launch_after(k_part1<true>, g1, kPartThreads, smem, stream, sa, lcp, n, s, segs, tma);
    else k_part1<false><<<g1, kPartThreads, smem, stream>>>(sa, lcp, n, s, segs, tma);
    launch_part2<false>(n, s, stream);
}

void launch_rank_window_front(const int32_t* rank, const int32_t* lcp, int32_t n, const Scratch& s,
                              cudaStream_t stream) {
    const unsigned g0 = (unsigned)(((long long)n + kPartRound - 1) / kPartRound);
    const int tma = ((uintptr_t)rank & 15u) == 0 ? 1 : 0;   // bulk copies need a 16-byte-aligned source
    k_rank_win<<<g0, kPartThreads, rank_win_smem_bytes((int)s.nwins), stream>>>(rank, n, s, tma);
    const unsigned g1 = (unsigned)(s.nwins * ((1 << kWinLog) / kPartRound));
    // not launch_after: with an early start the phase takes 1.116 instead of
    // 1.054 ms at 8 x 10^7 positions of English
    k_part1_win<<<g1, kPartThreads, part_scatter_smem_bytes((int)s.nsupers), stream>>>(lcp, n, s);
    launch_part2<true>(n, s, stream);
}

void launch_bucket_front(int32_t n, const Scratch& s, cudaStream_t stream) {
    launch_after(k_bucket_llr, (unsigned)s.nbuckets, kBucketThreads, bucket_smem_bytes(), stream, n, s);
}

cudaError_t configure_front() {
    cudaError_t e = cudaFuncSetAttribute(k_bucket_llr, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)bucket_smem_bytes());
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_part1<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)part_smem_bytes(2048));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_part1<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)part_smem_bytes(2048));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_rank_win, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)rank_win_smem_bytes(kMaxWins));
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(k_part1_win, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)part_scatter_smem_bytes(2048));
    return e;
}

}  // namespace lr
