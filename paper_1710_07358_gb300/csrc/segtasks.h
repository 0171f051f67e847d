// The list of long segments that k_seg_group makes for k_seg_long: how long a
// segment has to be, what a chunk of one is, and which of its records fit.
// Plain integer arithmetic, for host and device.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define PR_HD __host__ __device__ __forceinline__
#else
#define PR_HD inline
#endif

namespace pr {

// A segment of more than `most` elements is left to k_seg_long, in chunks of
// `chunk`.  Both grow with the elements so that the tasks fit: at most half
// of them long segments (unless there are that few segments at all), the
// other half the further chunks of those.
constexpr int64_t kLongSeg = 2048;
constexpr int64_t kLongChunk = 8192;

struct SegSplit {
    int64_t most, chunk;
};
PR_HD SegSplit seg_split_lengths(int64_t total, int64_t nseg, unsigned tasks) {
    const int64_t share = total / (tasks / 2) + 1;
    const int64_t most = nseg <= tasks / 2 || share < kLongSeg ? kLongSeg : share;
    const int64_t chunk = share < kLongChunk ? kLongChunk : share;
    return {most, chunk < most ? most : chunk};
}
PR_HD unsigned seg_chunks(int64_t len, const SegSplit& sp) { return (unsigned)((len + sp.chunk - 1) / sp.chunk); }

// Tasks asked for so far.  Segments of well-formed offsets ask for at most
// `tasks` in all; malformed ones may overlap, each asking for up to half of
// that, so that the sum over nseg of them passes 32 bits: with a 32-bit count
// it wrapped, later segments were listed over earlier records, and a chunk's
// index less its segment's first task pointed far outside the list.
using SegCount = unsigned long long;

// Records of a segment's n tasks, from `first` on, that lie in the list.
PR_HD unsigned seg_listed(SegCount first, unsigned n, unsigned tasks) {
    if (first >= tasks) return 0u;
    const SegCount room = tasks - first;
    return n < room ? n : (unsigned)room;
}

}  // namespace pr
