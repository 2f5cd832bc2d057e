// Launch sequence of one longest-repeat query on a stream: clear the
// per-query status words, run a front end (lr_front.cu) that builds the
// compact LLR array (with sa, a dense array up to a few million positions and
// the rank-order partition above; rank windows from rank alone for
// one long string; else the rank gather), then a cover kernel (the tile
// cover of lr_cover.cu by default, or the warp-segment cover of
// lr_cover_w.cu when the shape asks for it).  A short string takes one kernel
// instead (k_one_tile).
#include <cuda_runtime.h>
#include <cstdint>
#include "lr_internal.h"

namespace lr {

cudaError_t configure_front();
cudaError_t configure_cover();
cudaError_t configure_cover_w();

cudaError_t configure_kernels() {
    cudaError_t e = configure_front();
    if (e == cudaSuccess) e = configure_cover();
    return e == cudaSuccess ? configure_cover_w() : e;
}

cudaError_t launch_query(const int32_t* sa, const int32_t* rank, const int32_t* lcp, int32_t n, const Scratch& s,
                         int32_t* lr_len, int32_t* lr_start, int64_t* offsets, int32_t* starts,
                         long long capacity, bool all, cudaStream_t stream, int* launches,
                         PhaseEvents* events, const Segs& segs, const Shape& shape) {
    const bool timed = events && events->enabled;
    int k = 0;
    auto mark = [&]() { if (timed) cudaEventRecord(events->ev[k], stream); ++k; };
    if (s.one_tile && segs.num == 0 && n <= kOneTileMax) {
        mark();
        launch_one_tile(sa, rank, lcp, n, s, lr_len, lr_start, offsets, starts, capacity, all, stream);
        if (timed) cudaEventRecord(events->ev[k], stream);
        if (launches) *launches = 1;
        if (events) events->count = k;
        return cudaGetLastError();
    }
    const bool rankwin = !sa && segs.num == 0 && s.cursor_w && (long long)n >= kRankWinMinN;
    const bool dense = sa ? (long long)n <= (segs.num > 0 ? kDenseMaxBatch : kDenseMaxN) : !rankwin;
    mark();
    if (dense) {
        if (sa || segs.num > 0) launch_prep(n, s, segs, sa != nullptr, stream);   // k_prep
        if (sa) launch_scatter(sa, lcp, n, s, segs, stream);        // k_scatter
        else launch_gather(rank, lcp, n, s, segs, stream);          // k_gather
        mark();
        launch_compact(n, s, stream);                               // k_compact
    } else {
        cudaError_t e = cudaMemsetAsync(s.zero_base, 0, s.zero_bytes, stream);
        if (e != cudaSuccess) return e;
        if (segs.num > 0) launch_seg_index(n, s, segs, stream);     // k_seg_index
        if (sa) launch_partition(sa, lcp, n, s, segs, stream);      // k_part1, k_part2
        else launch_rank_window_front(rank, lcp, n, s, stream);     // k_rank_win, k_part1_win, k_part2
        mark();
        launch_bucket_front(n, s, stream);                          // k_bucket_llr
    }
    mark();
    if (shape.tile_cover)
        launch_cover(n, s, lr_len, lr_start, offsets, starts, capacity, all, shape.cover_tiles_per, stream);
    else
        launch_cover_w(n, s, lr_len, lr_start, offsets, starts, capacity, all, stream);
    if (timed) cudaEventRecord(events->ev[k], stream);
    if (launches) *launches = dense ? (sa || segs.num > 0 ? 4 : 3) : (sa ? 4 : 5) + (segs.num > 0 ? 1 : 0);
    if (events) events->count = k;
    return cudaGetLastError();
}

}  // namespace lr
