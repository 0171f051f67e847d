// Reduction kernels.  Included by the per-dtype instantiation units only.
//
// k_reduce     plain reduction of x[0..n) in ONE launch:
//   Step 1 (Section 2.3 / Section 3, "Unrolling the step 1"): a persistent grid
//     (Section 2.5) strides over the input in VB-byte vectors; each thread keeps
//     U independent accumulators and issues its U loads before accumulating,
//     so U*VB bytes per thread are in flight.  Elements before the first VB
//     boundary and after the last full vector are read as scalars (no access
//     outside [x, x+n); the identity is never needed as a load mask).
//   Step 3: the U accumulators are combined, then the warp (shuffle butterfly
//     or redux.sync), then the block (one value per warp in shared memory).
//   Large inputs (the TAIL variant): the grid-stride part stops at a
//     multiple of the grid's stride near nine tenths of the vectors, and the
//     rest is cut into tiles of whole rounds of blockDim x TL vectors (about
//     128 KiB) that blocks claim from an atomic counter, a claim ahead.  SMs
//     stream at unequal rates (their finishing times spread over a few
//     microseconds), so a static split ends when the slowest SM does;
//     claimed tiles let the fast SMs take the slow ones' share of the end.
//     An exact trait adds the tiles to its accumulators; any other reduces
//     each tile like a block partial, stored in a slot indexed by the tile,
//     so the result does not depend on which block took which tile.
//   Stage 2 (Section 2.3), fused: every block stores its partial; the last
//     block to finish (atomic ticket after a fence) combines all partials in
//     block-index order, then the tile partials in tile order, writes the
//     result and re-arms the ticket and claim counters.  A launch of one
//     block (small inputs) finishes with the same combine and no ticket.
//
// k_segmented  many reductions (segments of a CSR offsets array, or equal rows)
//   in one launch.  The element range [offsets[0], offsets[nseg]) is cut into
//   tiles of blockDim*U*VB bytes, and runs of tiles form chunks.  With many
//   segments per block there are two chunks per block, claimed dynamically
//   from an atomic counter so that blocks delayed by many segment boundaries
//   do not hold up the launch; with few, one static chunk per block.
//   Inside a tile that lies in one segment the block streams exactly like
//   k_reduce; a tile containing segment boundaries emits the finished
//   segment, reduces the segments that lie wholly inside the tile (short ones
//   one per warp, long ones with the whole block) and starts the next one.
//   A segment that crosses chunk boundaries leaves one partial per chunk it
//   touches (its first chunk's "tail" slot, later chunks' "head" slots); the
//   last of those chunks to finish (per-segment ticket) combines them in chunk
//   order.  Partials are indexed by chunk, not by block, so results are
//   deterministic for a fixed launch configuration whatever the claim order.
//
// k_seg_group, k_seg_long  segments of a CSR offsets array when there are many
//   (kSegGroupMin): a tile of k_segmented costs its block several barriers and
//   a search, which hundreds of short segments a tile do not pay for.  The
//   first kernel takes up to 32 neighbouring segments a warp, through shared
//   memory where they are short; the second shares the long ones among all
//   warps, chunk by chunk.  fp32 sum on GB300: 10^6 segments of 24 elements on
//   average (96 MB) 840 -> 52 us (0.30 of a 6.8 TB/s copy; launches repeated on
//   one input, a call through the binding takes 56), 65536 of 1000 231 -> 70,
//   10^5 log-uniform to 16384 317 -> 212, 8192 of 40000 205 -> 207; maximum with
//   index of the first 976 -> 105, of the last 538 -> 243.  Short
//   segments are bound by instructions, about 24 warp instructions a segment
//   of 24 (ncu: issue slots 60 % busy, no one stall dominant), long ones by HBM.
//
// k_rows       equal rows of `cols` elements (cols a multiple of the vector
//   width, x aligned to it): the flattened vectors are split into one run of
//   whole tiles per block; a block streams its run exactly like k_reduce and
//   finishes a row each time the run crosses a row end.  The first vectors of
//   the next row are loaded before that row's block combine, so loads stay in
//   flight through it.  A row shared by several blocks leaves one partial per
//   block (the first block's "tail" slot, later blocks' "head" slots); the
//   last of them to finish (per-row ticket) combines them in block order, so
//   results are deterministic for a fixed launch configuration.
//
// k_rows_group  equal rows of any length and alignment, short ones above all:
//   a row goes to a group of 2^gl neighbouring lanes of a warp (gl <= 5) or
//   to a whole block, and ends with a combine across those lanes only.  k_rows
//   and k_segmented end every row with a combine of the whole block, about
//   1.2 us during which the block streams nothing: a row of a megabyte hides
//   it, one of a few kilobytes does not.  Bound by HBM from a few kilobytes a
//   row (fp32 sum of [32768, 1000] 174 -> 22.6 us, 0.86 of a 6.8 TB/s copy;
//   [8192, 4096] 47 -> 22.6), by the latency of each row's short chain below
//   ([200000, 120] 968 -> 18.2 us, 0.78; maximum with index of [32768, 1000]
//   397 -> 26.7).  No grid loop: a block per 256 threads of work, so that the
//   hardware evens out the rows.
//
// k_combine_parts  one block combining an array of partials in order.
#pragma once
#include <type_traits>
#include "segtasks.h"
#include "traits.cuh"

namespace pr {

constexpr int kSlot = 64;      // bytes per partial slot (>= sizeof(Part) of every trait)
constexpr int kSmallSeg = 512; // segments up to this length are reduced by one warp
// Segmented launches of this many segments and more take k_seg_group and
// k_seg_long; smaller ones k_segmented, which hands segments over to groups of
// lanes itself when their mean is at most kGroupMean and none is longer than
// kGroupMost elements (which every block sees for itself: no second launch).
// Measured on GB300 (us, fp32 sum, k_segmented before / k_segmented with the
// hand-over / k_seg_group + k_seg_long): 1000 segments of 24 on average 72 /
// 6.4 / 8.5, 4096 log-uniform to 4096 22.5 / 12.7 / 18.5, 10^4 of 24 98 / 25 /
// 8.5; k_segmented splits few and long ones best (64 log-uniform to 2^20 16 /
// 16 / 25, 4096 to 2^20 183 / 183 / 189) unless the accumulator is heavy
// (maximum with index: 4096 to 2^20 416 / 417 / 218, 877 to 380 000 76 / 76 /
// 50, 64 to 2^20 31 / 32 / 30).
constexpr int64_t kSegGroupMin = 8192;
constexpr int64_t kSegGroupMinHeavy = 512;   // kernels with an index or product state
constexpr int64_t kGroupMean = 4096;
constexpr int64_t kGroupMost = 8192;
constexpr int kGroupBlock = 256;   // threads per block of the group kernels
constexpr int kGroupVec = 32;      // bytes per vector load
enum : int { kErrInvalid = 1, kErrTimeout = 4 };

// One task of k_seg_group's shared part: a long segment, or a chunk of one
// that is longer than a chunk.  A segment's tasks follow one another; its
// partials and its count of finished chunks go by task index.
struct SegTask {
    int64_t seg;
    unsigned first;      // the segment's first task
    unsigned finished;   // in the first task: chunks whose partials are stored
};

// Tasks that a launch lists at most, as far as the partial slots suffice.
constexpr unsigned kSegTasks = 65536;

struct Workspace {
    char* partials;      // gmax slots (k_reduce)
    char* head;          // gmax slots (k_segmented: first-segment partial of a block; k_reduce: tile partials)
    char* tail;          // gmax slots (k_segmented: last-segment partial of a block)
    unsigned* seg_cnt;   // gmax tickets (k_segmented), zero between launches
    unsigned* counter;   // 1 ticket (k_reduce), zero between launches
    unsigned* chunk_ctr; // next chunk (k_segmented) or tile (k_reduce) to claim, zero between launches
    unsigned* blk_done;  // blocks finished (k_segmented), zero between launches
    int* err;            // device error word
    int gmax;
    SegTask* tasks = nullptr;       // kSegTasks (k_seg_group)
    SegCount* task_count = nullptr; // tasks asked for, zero between launches
};

struct ReduceArgs {
    const void* x;
    int64_t n;
    int64_t head;        // elements before the first VB-aligned element (< VE, <= n)
    void* out;
    void* part_out;      // non-null: store the final Part here instead of a result
    int out_f64;
    Workspace ws;
    int64_t* argidx;     // arg-extremum traits: index of the first extremum (may be null)
    int64_t stat = 0;      // tile_vec > 0: vectors (after the head) of the grid-stride part,
                           // a multiple of U x threads
    int64_t tile_vec = 0;  // > 0: the vectors past `stat` are claimed in tiles of about this
                           // many vectors (partials in ws.head); 0: no claimed tail
};

struct SegArgs {
    const void* x;
    const int64_t* off;  // nseg+1 CSR offsets, or null for equal rows of `cols`
    int64_t cols;
    int64_t nseg;
    int64_t shift;       // x's element offset from the previous VB boundary
    void* out;
    int64_t* argidx;
    pr_prod_aux* aux;
    int out_f64;
    int chunks_per_block;  // chunks (contiguous tile runs) per block
    int dynamic_chunks;    // 1: blocks claim chunks from an atomic counter; 0: chunk c -> block c mod grid
    Workspace ws;
};

struct RowArgs {
    const void* x;       // aligned to the vector width
    int64_t rows, cols;  // cols > 0, a multiple of the elements per vector
    void* out;
    int64_t* argidx;
    pr_prod_aux* aux;
    int out_f64;
    Workspace ws;
};

struct SegGroupArgs {
    const void* x;
    const int64_t* off;  // nseg+1 CSR offsets
    int64_t nseg;
    int shift;           // x's element offset from the previous 32-byte boundary
    unsigned tasks;      // tasks that may be listed: kSegTasks, or what the partial slots hold
    void* out;
    int64_t* argidx;
    pr_prod_aux* aux;
    Workspace ws;
};

struct RowGroupArgs {
    const void* x;
    int64_t rows, cols;  // 0 < cols < 2^30
    int shift;           // x's element offset from the previous 32-byte boundary
    int gl;              // log2 of the lanes per row: 0..5, or 8 (a block per row)
    void* out;
    int64_t* argidx;
    pr_prod_aux* aux;
};

struct BwdArgs {
    const void* x;
    const void* g;
    const int64_t* argidx;
    const pr_prod_aux* aux;
    void* gi;
    int64_t rows, cols;
    int64_t shift;           // grad_in's element offset from the previous VB boundary
    int64_t chunks_per_row;
    int op;
};


// The value that crosses blocks: the trait's Part, combined with the trait's
// combine (the same one the warp and block stages use).
template <class T>
struct GridR {
    using Part = typename T::Part;
    __device__ __forceinline__ static Part up(const typename T::Part& p) { return p; }
    __device__ __forceinline__ static Part part_init() { return T::part_init(); }
    __device__ __forceinline__ static Part combine(const Part& a, const Part& b) { return T::combine(a, b); }
    __device__ __forceinline__ static Part warp_reduce(Part p) { return T::warp_reduce(p); }
    __device__ __forceinline__ static void store(void* out, int64_t i, const Part& p, bool f64) { T::store(out, i, p, f64); }
    __device__ __forceinline__ static void store_aux(int64_t* ai, pr_prod_aux* ax, int64_t i, const Part& p, int64_t sb) {
        T::store_aux(ai, ax, i, p, sb);
    }
};

// Largest block a trait's kernels are compiled for (a trait with a large
// per-thread state declares kMaxBlock to get more registers per thread); the
// host clamps launch configurations to it.
template <class T, class = void>
struct MaxBlock {
    static constexpr int value = 1024;
};
template <class T>
struct MaxBlock<T, std::void_t<decltype(T::kMaxBlock)>> {
    static constexpr int value = T::kMaxBlock;
};

// Blocks of the plain reduction that must fit on one SM at once (a trait
// declares kMinBlocks to cap its registers per thread; default 1).
template <class T, class = void>
struct MinBlocks {
    static constexpr int value = 1;
};
template <class T>
struct MinBlocks<T, std::void_t<decltype(T::kMinBlocks)>> {
    static constexpr int value = T::kMinBlocks;
};

// A trait whose combine is exact and independent of order (integer,
// bitwise, max / min and arg-extremum) declares kExact: claimed tail tiles
// then join its running accumulators, with no partial per tile.
template <class T, class = void>
struct Exact {
    static constexpr bool value = false;
};
template <class T>
struct Exact<T, std::void_t<decltype(T::kExact)>> {
    static constexpr bool value = T::kExact;
};

// Vectors a thread loads per round of a claimed tile: four for a float trait
// whose accumulator is one or two words and whose registers are not capped,
// U otherwise (exact traits add tiles to their running accumulators).
template <class T, int U, class = void>
struct TileLoads {
    static constexpr int value =
        (!Exact<T>::value && MinBlocks<T>::value == 1 && sizeof(typename T::Acc) <= 8 && U < 4) ? 4 : U;
};
template <class T, int U>
struct TileLoads<T, U, std::void_t<decltype(T::kTileLoads)>> {   // a trait's own choice
    static constexpr int value = T::kTileLoads;
};

// Claimed tail tiles a block of k_reduce holds partials for: one value per
// warp and tile in shared memory, up to 16 KiB (64 tiles of fp32 partials).
// Exact traits keep no tile partials.
template <class T>
struct TileSlots {
    static constexpr int kBytes = (MaxBlock<T>::value / 32) * (int)sizeof(typename T::Part);
    static constexpr int value = Exact<T>::value ? (1 << 20)
                               : (16384 / kBytes > 64 ? 64 : (16384 / kBytes < 4 ? 4 : 16384 / kBytes));
};

template <class T>
__device__ __forceinline__ typename T::Part* slot(char* base, int64_t i) {
    return reinterpret_cast<typename T::Part*>(base + i * kSlot);
}

// Combine a thread's U accumulators into one Part.
template <class T, int U>
__device__ __forceinline__ typename T::Part fold(typename T::Acc (&acc)[U]) {
    typename T::Part p = T::to_part(acc[0]);
#pragma unroll
    for (int u = 1; u < U; u++) p = T::combine(p, T::to_part(acc[u]));
    return p;
}

// ------------------------------------------------------------------------
// Plain reduction
// ------------------------------------------------------------------------

template <class T, int U, int VB, bool TAIL>
__device__ __forceinline__ void reduce_body(const ReduceArgs& a) {
    using Ld = typename T::Ld;
    using In = typename Ld::In;
    using E = typename Ld::E;
    using Part = typename T::Part;
    constexpr int VE = VB / Ld::ES;
    const In* x = static_cast<const In*>(a.x);

    typename T::Acc acc[U];
#pragma unroll
    for (int u = 0; u < U; u++) acc[u] = T::init();

    const int64_t nth = (int64_t)gridDim.x * blockDim.x;
    const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t head = a.head;
    const int64_t nvec = (a.n - head) / VE;
    const bool dyn = TAIL && a.tile_vec > 0;
    int64_t nstat = nvec;                           // vectors of the grid-stride part
    if constexpr (TAIL) nstat = dyn ? a.stat : nvec;
    const char* xv = reinterpret_cast<const char*>(x + head);
    using GR = GridR<T>;
    using G = typename GR::Part;
    // claimed tiles: thread 0 makes the block's first two claims while the
    // loads of its last grid-stride step travel (claims made earlier would
    // hand out tiles by start order rather than by progress), keeps them in
    // shared memory, and then at each tile publishes the claim it made a
    // tile earlier and makes the next, so no warp waits for a claim's round
    // trip
    __shared__ unsigned s_claim[2], s_claim1;
    bool claimed = false;
    auto claim_first = [&]() {
        if constexpr (TAIL)
            if (dyn && !claimed && threadIdx.x == 0) {
                s_claim[0] = atomicAdd(a.ws.chunk_ctr, 1u);
                s_claim1 = atomicAdd(a.ws.chunk_ctr, 1u);
                claimed = true;
            }
    };

    int64_t i = tid;
    for (; i + (int64_t)(U - 1) * nth < nstat; i += (int64_t)U * nth) {
        Words<VB> w[U];
#pragma unroll
        for (int u = 0; u < U; u++) w[u] = ldv<VB>(xv + (i + u * nth) * VB);
        if (i + (int64_t)(2 * U - 1) * nth >= nstat) claim_first();   // the last step
#pragma unroll
        for (int u = 0; u < U; u++) {
            E e[VE];
            Ld::template dec<VB>(w[u], e);
            T::add_vec(acc[u], e, head + (i + u * nth) * VE);
        }
    }
    for (; i < nstat; i += nth) {
        Words<VB> w = ldv<VB>(xv + i * VB);
        E e[VE];
        Ld::template dec<VB>(w, e);
        T::add_vec(acc[0], e, head + i * VE);
    }
    if (tid < head) T::add(acc[0], Ld::one(x, tid), tid);
    for (int64_t j = head + nvec * VE + tid; j < a.n; j += nth) T::add(acc[0], Ld::one(x, j), j);
    claim_first();   // (a grid-stride part too short for the loop)
    unsigned c_next = ~0u;

    // claimed tiles: vectors [nstat, nvec) in tiles of R rounds of blockDim x
    // TL vectors (R from the requested tile size), the next claim issued with
    // a tile's first loads.  An exact trait adds them to its accumulators
    // (each still sees its vectors in increasing index order: tiles lie past
    // the grid-stride part and a block's claims increase), with U loads a
    // thread.  Any other trait reduces each tile like a block partial into a
    // slot indexed by the tile, with four loads a thread where its
    // accumulator is one or two words and its registers are not capped (U
    // where four would spill).
    constexpr bool EX = Exact<T>::value;
    constexpr int TL = TileLoads<T, U>::value;
    const int64_t round_vec = (int64_t)blockDim.x * TL;
    const int rounds = dyn && a.tile_vec > round_vec ? (int)(a.tile_vec / round_vec) : 1;
    const int64_t tile = round_vec * rounds;
    const int64_t ntiles = dyn ? (nvec - nstat + tile - 1) / tile : 0;
    // one tile into accumulators ac; with its first loads thread 0 publishes
    // the next tile (claimed a tile earlier) and claims the one after (if
    // `more`: a block of a float trait stops claiming when its TileSlots
    // partial slots are full)
    auto run_tile = [&](typename T::Acc (&ac)[U], unsigned t, int k, bool more) {
        const int64_t v0 = nstat + (int64_t)t * tile + threadIdx.x;   // this thread's first vector
        const char* p0 = xv + v0 * VB;
        const int64_t left = nvec - v0;                               // vectors from v0 to the end
        const bool full = left >= tile;                               // every tile but the last
        for (int r = 0; r < rounds; r++) {
            const int64_t o = (int64_t)r * round_vec;
            Words<VB> w[TL];
#pragma unroll
            for (int q = 0; q < TL; q++)
                if (full || o + q * (int)blockDim.x < left) w[q] = ldv<VB>(p0 + (o + q * (int)blockDim.x) * VB);
            if (r == 0 && threadIdx.x == 0) {
                s_claim[(k + 1) & 1] = c_next;
                c_next = more ? atomicAdd(a.ws.chunk_ctr, 1u) : ~0u;
            }
#pragma unroll
            for (int q = 0; q < TL; q++) {
                const int64_t oq = o + q * (int)blockDim.x;
                if (full || oq < left) {
                    E e[VE];
                    Ld::template dec<VB>(w[q], e);
                    T::add_vec(ac[q % U], e, head + (v0 + oq) * VE);
                }
            }
        }
    };
    if constexpr (TAIL && EX) {
        if (dyn) {
            __syncthreads();   // the first claims, in shared memory
            unsigned t = s_claim[0];
            if (threadIdx.x == 0) c_next = s_claim1;
            for (int k = 0; (int64_t)t < ntiles; k++) {
                run_tile(acc, t, k, true);
                __syncthreads();
                t = s_claim[(k + 1) & 1];
            }
        }
    }

    const Part p = block_combine<T>(fold<T, U>(acc));

    int ktiles = 0;   // tiles this block reduced (float traits)
    if constexpr (TAIL && !EX) if (dyn) {
        // a tile's partial: each warp's value in a shared slot (no combine
        // across warps inside the loop, so no warp falls behind the others
        // between barriers); after the block's last tile, thread j combines
        // its tile j's warp values in warp order and stores them in the
        // tile's slot
        constexpr int NW = MaxBlock<T>::value / 32;
        constexpr int NS = TileSlots<T>::value;
        __shared__ Part s_tp[NS][NW];
        __shared__ unsigned s_tid[NS];
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        const int nwarps = (blockDim.x + 31) >> 5;
        unsigned t = s_claim[0];   // written before block_combine's barriers
        if (threadIdx.x == 0) c_next = s_claim1;
        int k = 0;
        while ((int64_t)t < ntiles) {
            typename T::Acc ta[U];
#pragma unroll
            for (int u = 0; u < U; u++) ta[u] = T::init();
            run_tile(ta, t, k, k + 2 < NS);
            const Part tp = T::warp_reduce(fold<T, U>(ta));
            if (lane == 0) s_tp[k][warp] = tp;
            if (threadIdx.x == 0) s_tid[k] = t;
            __syncthreads();
            t = s_claim[(k + 1) & 1];
            k++;
        }
        if ((int)threadIdx.x < k) {
            Part q = s_tp[threadIdx.x][0];
            for (int w = 1; w < nwarps; w++) q = T::combine(q, s_tp[threadIdx.x][w]);
            *slot<GR>(a.ws.head, s_tid[threadIdx.x]) = GR::up(q);
        }
        ktiles = k;
    }

    // the result (valid in thread 0) to out, or as a Part to part_out
    auto finish = [&](const G& q) {
        if (a.part_out) {
            *static_cast<G*>(a.part_out) = q;
        } else {
            GR::store(a.out, 0, q, a.out_f64 != 0);
            GR::store_aux(a.argidx, nullptr, 0, q, 0);
        }
    };
    // one block (small inputs): its partial is the only one, so it finishes
    // at once, with the same combine the last block would make, and no
    // round trip through memory, fence or ticket
    if constexpr (!TAIL) {
        if (gridDim.x == 1) {
            G q = threadIdx.x == 0 ? GR::combine(GR::part_init(), GR::up(p)) : GR::part_init();
            q = block_combine<GR>(q);
            if (threadIdx.x == 0) finish(q);
            return;
        }
    }

    // every thread that wrote a partial (thread 0 the block's, and with a
    // claimed tail of a float trait the first threads their tiles') fences;
    // a barrier then orders those writes before thread 0's ticket
    __shared__ unsigned s_last;
    if constexpr (TAIL && !EX) {
        if (threadIdx.x == 0) *slot<GR>(a.ws.partials, blockIdx.x) = GR::up(p);
        if (threadIdx.x == 0 || (int)threadIdx.x < ktiles) __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) s_last = (atomicAdd(a.ws.counter, 1u) == gridDim.x - 1);
    } else if (threadIdx.x == 0) {
        *slot<GR>(a.ws.partials, blockIdx.x) = GR::up(p);
        __threadfence();
        const unsigned ticket = atomicAdd(a.ws.counter, 1u);
        s_last = (ticket == gridDim.x - 1);
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    G q = GR::part_init();
    if constexpr (TAIL && !EX) {
        // block partials, then tile partials in tile order; the tile loop is
        // unrolled so that a thread's loads of several slots travel together
        for (int j = threadIdx.x; j < (int)gridDim.x; j += blockDim.x)
            q = GR::combine(q, ld_cg_any(slot<GR>(a.ws.partials, j)));
        const int nt = (int)ntiles;
        int j = threadIdx.x;
        for (; j + 3 * (int)blockDim.x < nt; j += 4 * blockDim.x) {
            G v[4];
#pragma unroll
            for (int r = 0; r < 4; r++) v[r] = ld_cg_any(slot<GR>(a.ws.head, j + r * (int)blockDim.x));
#pragma unroll
            for (int r = 0; r < 4; r++) q = GR::combine(q, v[r]);
        }
        for (; j < nt; j += blockDim.x) q = GR::combine(q, ld_cg_any(slot<GR>(a.ws.head, j)));
    } else {
        for (int j = threadIdx.x; j < (int)gridDim.x; j += blockDim.x)
            q = GR::combine(q, ld_cg_any(slot<GR>(a.ws.partials, j)));
    }
    q = block_combine<GR>(q);
    if (threadIdx.x == 0) {
        finish(q);
        *a.ws.counter = 0u;
        if constexpr (TAIL)
            if (dyn) *a.ws.chunk_ctr = 0u;
    }
}

// The plain reduction's kernel.  A trait that declares kMinBlocks gets the
// two-argument launch bound (a register cap); the others keep the one-argument
// bound, with which the compiler chooses their registers freely (an explicit
// minimum of one block makes it take more, and so halves some traits'
// occupancy).
// TAIL: the variant with claimed tail tiles (large inputs; its tile loads
// take registers the grid-stride kernel does not need).
template <class T, int U, int VB, bool TAIL>
__global__ void __launch_bounds__(MaxBlock<T>::value) k_reduce(ReduceArgs a) {
    reduce_body<T, U, VB, TAIL>(a);
}
template <class T, int U, int VB, bool TAIL>
__global__ void __launch_bounds__(MaxBlock<T>::value, MinBlocks<T>::value) k_reduce_occ(ReduceArgs a) {
    reduce_body<T, U, VB, TAIL>(a);
}
template <class T, int U, int VB, bool TAIL = false>
constexpr auto reduce_kernel() {
    if constexpr (MinBlocks<T>::value > 1) return &k_reduce_occ<T, U, VB, TAIL>;
    else return &k_reduce<T, U, VB, TAIL>;
}

// One block: out = parts[0] (x) parts[1] (x) ... in index order (slot stride kSlot).
template <class T>
__global__ void __launch_bounds__(256) k_combine_parts(const char* parts, int count, void* out, int out_f64) {
    using GR = GridR<T>;
    using G = typename GR::Part;
    G q = GR::part_init();
    for (int j = threadIdx.x; j < count; j += blockDim.x)
        q = GR::combine(q, *reinterpret_cast<const G*>(parts + (int64_t)j * kSlot));
    q = block_combine<GR>(q);
    if (threadIdx.x == 0) GR::store(out, 0, q, out_f64 != 0);
}

// ------------------------------------------------------------------------
// Row reduction
// ------------------------------------------------------------------------

template <class T, int U, int VB>
__global__ void __launch_bounds__(MaxBlock<T>::value) k_rows(RowArgs a) {
    using Ld = typename T::Ld;
    using E = typename Ld::E;
    using Acc = typename T::Acc;
    using Part = typename T::Part;
    using GR = GridR<T>;
    using G = typename GR::Part;
    constexpr int VE = VB / Ld::ES;
    const char* xv = static_cast<const char*>(a.x);
    const bool f64 = a.out_f64 != 0;
    const int B = blockDim.x;
    const int64_t cv = a.cols / VE;                 // vectors per row
    const int64_t nv = a.rows * cv;                 // vectors in all
    const int64_t TILE = (int64_t)B * U;            // vectors per tile
    const int64_t ntile = (nv + TILE - 1) / TILE;
    const int64_t R = (ntile + gridDim.x - 1) / gridDim.x * TILE;  // vectors per block run
    const int64_t vlo = (int64_t)blockIdx.x * R < nv ? (int64_t)blockIdx.x * R : nv;
    const int64_t vhi = vlo + R < nv ? vlo + R : nv;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    (void)lane;
    (void)warp;
    __shared__ int s_fin;

    Words<VB> pre[U];   // this thread's first U vectors of the next row piece
    bool have = false;
    for (int64_t v = vlo; v < vhi;) {
        const int64_t r = v / cv;
        const int64_t pend = (r + 1) * cv < vhi ? (r + 1) * cv : vhi;
        Acc acc[U];
#pragma unroll
        for (int u = 0; u < U; u++) acc[u] = T::init();
        int64_t i = v + threadIdx.x;
        if (have) {
#pragma unroll
            for (int u = 0; u < U; u++) {
                E e[VE];
                Ld::template dec<VB>(pre[u], e);
                T::add_vec(acc[u], e, (i + (int64_t)u * B) * VE);
            }
            i += TILE;
        }
        for (; i + (int64_t)(U - 1) * B < pend; i += TILE) {
            Words<VB> w[U];
#pragma unroll
            for (int u = 0; u < U; u++) w[u] = ldv<VB>(xv + (i + (int64_t)u * B) * VB);
#pragma unroll
            for (int u = 0; u < U; u++) {
                E e[VE];
                Ld::template dec<VB>(w[u], e);
                T::add_vec(acc[u], e, (i + (int64_t)u * B) * VE);
            }
        }
        for (; i < pend; i += B) {
            const Words<VB> w = ldv<VB>(xv + i * VB);
            E e[VE];
            Ld::template dec<VB>(w, e);
            T::add_vec(acc[0], e, i * VE);
        }
        // load the next piece's first vectors now, so that they arrive during the combine
        have = false;
        if (pend < vhi) {
            const int64_t nend = pend + cv < vhi ? pend + cv : vhi;
            const int64_t j = pend + threadIdx.x;
            if (j + (int64_t)(U - 1) * B < nend) {
#pragma unroll
                for (int u = 0; u < U; u++) pre[u] = ldv<VB>(xv + (j + (int64_t)u * B) * VB);
                have = true;
            }
        }
        // finish this block's piece of row r
        const Part p = block_combine<T>(fold<T, U>(acc));
        const int64_t sb = r * a.cols;
        const int64_t ba = (r * cv) / R, bb = ((r + 1) * cv - 1) / R;
        if (ba == bb) {
            if (threadIdx.x == 0) {
                const G g = GR::up(p);
                GR::store(a.out, r, g, f64);
                GR::store_aux(a.argidx, a.aux, r, g, sb);
            }
        } else {
            if (threadIdx.x == 0) {
                *slot<GR>(v > r * cv ? a.ws.head : a.ws.tail, blockIdx.x) = GR::up(p);
                __threadfence();
                const unsigned old = atomicAdd(a.ws.seg_cnt + ba, 1u);
                s_fin = (old == (unsigned)(bb - ba));
            }
            __syncthreads();
            if (s_fin) {
                __threadfence();
                G q = GR::part_init();
                for (int64_t k = threadIdx.x; k <= bb - ba; k += B)
                    q = GR::combine(q, ld_cg_any(k == 0 ? slot<GR>(a.ws.tail, ba) : slot<GR>(a.ws.head, ba + k)));
                q = block_combine<GR>(q);
                if (threadIdx.x == 0) {
                    GR::store(a.out, r, q, f64);
                    GR::store_aux(a.argidx, a.aux, r, q, sb);
                    a.ws.seg_cnt[ba] = 0u;
                }
            }
        }
        v = pend;
    }
}

// ------------------------------------------------------------------------
// Runs of x reduced by groups of lanes
// ------------------------------------------------------------------------

// Accumulators a lane keeps: one per load in flight where an accumulator is
// one or two words (shorter chains of dependent operations, and a smaller sum
// of rounding errors), else one.
template <class T, int U, class = void>
struct GroupAccs {
    static constexpr int value = sizeof(typename T::Acc) <= 8 ? U : 1;
};
template <class T, int U>
struct GroupAccs<T, U, std::void_t<decltype(T::kGroupAccs)>> {
    static constexpr int value = T::kGroupAccs;
};

// A trait with a neutral element (pad) takes a vector that a run's end cuts as
// a whole one, in the order of a tree: added one by one, the elements of such
// vectors made up most of the rounding error of short runs.
template <class T, class = void>
struct HasPad : std::false_type {};
template <class T>
struct HasPad<T, std::void_t<decltype(&T::pad)>> : std::true_type {};

// Elements combined as a tree.
template <class T, int K>
__device__ __forceinline__ typename T::Part tree(const typename T::Ld::E (&e)[K]) {
    typename T::Part t[K];
#pragma unroll
    for (int k = 0; k < K; k++) t[k] = e[k];
#pragma unroll
    for (int s = 1; s < K; s <<= 1)
#pragma unroll
        for (int k = 0; k + s < K; k += 2 * s) t[k] = T::combine(t[k], t[k + s]);
    return t[0];
}

// Rounds of loads after which a lane's accumulator joins its total: an fp64
// sum takes no more additions than elements (the fp64 pipe bounds it), but as a
// tree over a round's vectors and in short chains of those.
template <class T, class = void>
struct GroupSteps {
    static constexpr int value = 0;
};
template <class T>
struct GroupSteps<T, std::void_t<decltype(T::kGroupSteps)>> {
    static constexpr int value = T::kGroupSteps;
};

// Accumulators combined as a tree.
template <class T, int N>
__device__ __forceinline__ typename T::Part fold_tree(const typename T::Acc (&acc)[N]) {
    typename T::Part p[N];
#pragma unroll
    for (int u = 0; u < N; u++) p[u] = T::to_part(acc[u]);
#pragma unroll
    for (int s = 1; s < N; s <<= 1)
#pragma unroll
        for (int u = 0; u + s < N; u += 2 * s) p[u] = T::combine(p[u], p[u + s]);
    return p[0];
}

// The elements [p0, p0 + len) of x that lane t of G neighbours takes, combined
// into one Part (the trait is given indices relative to p0, plus i0).  The run is
// covered by 32-byte vectors on the 32-byte grid of memory, lane t taking
// vectors t, t + G, ..., U of them in flight; of the vectors that hold the
// run's ends the elements outside it are dropped, and one that is not wholly
// inside [X0, X1), the elements the caller vouches for, is read element by
// element.
template <class T, int U>
__device__ __forceinline__ typename T::Part group_part(const typename T::Ld::In* x, int64_t p0, int len, int shift,
                                                       int64_t X0, int64_t X1, int t, int G, int64_t i0 = 0) {
    using Ld = typename T::Ld;
    using E = typename Ld::E;
    constexpr int VE = kGroupVec / Ld::ES;
    constexpr int NA = GroupAccs<T, U>::value;
    typename T::Acc acc[NA];
#pragma unroll
    for (int u = 0; u < NA; u++) acc[u] = T::init();
    const int mis = (int)((p0 + shift) & (VE - 1));       // elements of the first vector before the run
    const int nv = len > 0 ? (len + mis + VE - 1) / VE : 0;
    const char* base = reinterpret_cast<const char*>(x) + (p0 - mis) * Ld::ES;
    // run-relative element range that whole vectors may be read from
    const int64_t s0 = X0 - p0, s1 = X1 - p0;
    const int c_lo = s0 < -VE ? -VE : (int)s0, c_hi = s1 < (int64_t)len + VE ? (int)s1 : len + VE;
    constexpr int kSteps = GroupSteps<T>::value;
    E t_u[U];
    typename T::Part total = T::part_init();
    int step = 0;
    for (int j = t; j < nv; j += U * G) {
        Words<kGroupVec> w[U];
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int v = j + u * G, c = v * VE - mis;
            if (v < nv && c >= c_lo && c + VE <= c_hi) w[u] = ldv<kGroupVec>(base + (int64_t)v * kGroupVec);
        }
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int v = j + u * G, c = v * VE - mis;
            typename T::Acc& a = acc[u % NA];
            if constexpr (kSteps > 0) t_u[u] = T::pad();
            if (v >= nv) continue;
            const bool whole = c >= 0 && c + VE <= len;
            if (whole || (HasPad<T>::value && c >= c_lo && c + VE <= c_hi)) {
                E e[VE];
                Ld::template dec<kGroupVec>(w[u], e);
                if constexpr (HasPad<T>::value) {
                    if (!whole) {   // bit k: element c + k belongs to the run
                        asm volatile("");   // (a branch: selects in every vector cost whole rows a tenth)
                        const int lo = c < 0 ? -c : 0, hi = len - c < VE ? len - c : VE;
                        const unsigned m = ((1u << hi) - 1u) >> lo << lo;
#pragma unroll
                        for (int k = 0; k < VE; k++) e[k] = m >> k & 1u ? e[k] : T::pad();
                    }
                }
                if constexpr (kSteps > 0) t_u[u] = tree<T>(e);
                else T::add_vec(a, e, i0 + c);
            } else if (!HasPad<T>::value && c >= c_lo && c + VE <= c_hi) {
                E e[VE];
                Ld::template dec<kGroupVec>(w[u], e);
#pragma unroll
                for (int k = 0; k < VE; k++)
                    if ((unsigned)(c + k) < (unsigned)len) T::add(a, e[k], i0 + c + k);
            } else {
                const int e1 = c + VE < len ? c + VE : len;
                for (int i = c > 0 ? c : 0; i < e1; i++) T::add(a, Ld::one(x, p0 + i), i0 + i);
            }
        }
        if constexpr (kSteps > 0) {
            T::add_tree(acc[0], tree<T>(t_u));
            if (++step == kSteps) {
                total = T::combine(total, fold_tree<T, NA>(acc));
#pragma unroll
                for (int u = 0; u < NA; u++) acc[u] = T::init();
                step = 0;
            }
        }
    }
    if constexpr (kSteps > 0) return T::combine(total, fold_tree<T, NA>(acc));
    else return fold_tree<T, NA>(acc);
}

// Combine across the lanes of each group of 2^gl neighbours (gl <= 5; all 32
// lanes call); every lane of a group gets its result.
template <class T>
__device__ __forceinline__ typename T::Part group_combine(typename T::Part p, int gl) {
    if (gl == 5) return T::warp_reduce(p);
    for (int m = (1 << gl) >> 1; m >= 1; m >>= 1) p = T::combine(p, shfl_xor_any(p, m));
    return p;
}

// Lanes per segment (log2) for segments of `mean` elements on average: two
// loads a lane for half as many vectors again as such a segment touches, so
// that most segments of a spread of lengths need one round of loads.
template <class Ld>
__device__ __forceinline__ int group_lanes(int64_t mean) {
    const int64_t nv = mean / (kGroupVec / Ld::ES) + 1;
    int gl = 0;
    while (gl < 5 && ((int64_t)2 << gl) < nv + nv / 2) gl++;
    return gl;
}

// The result of segment s, from the lane that holds it.
template <class T>
__device__ __forceinline__ void store_segment(const typename T::Part& p, int64_t s, void* out, int64_t* argidx,
                                              pr_prod_aux* aux) {
    using GR = GridR<T>;
    const typename GR::Part g = GR::up(p);
    GR::store(out, s, g, false);
    GR::store_aux(argidx, aux, s, g, 0);
}

// One warp reduces up to 32 neighbouring segments s0, s0 + 1, ...: lane i
// holds segment s0 + i's first element b and its length (0: none; the segment
// lies in [X0, X1)).  Groups of 2^gl lanes take a segment each, in rounds,
// two loads a lane at a time; the vectors that hold a segment's ends are
// masked.  A segment of more than four loads a lane would hold the other
// groups up and waits for the whole warp, after the rounds; so do all where
// a vector might not lie in [X0, X1).
template <class T>
__device__ __forceinline__ void warp_segments(const typename T::Ld::In* x, int shift, int64_t X0, int64_t X1, int64_t s0,
                                              int64_t b, int len, int gl, void* out, int64_t* argidx,
                                              pr_prod_aux* aux) {
    using Ld = typename T::Ld;
    using E = typename Ld::E;
    using Part = typename T::Part;
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int VE = kGroupVec / Ld::ES;
    constexpr int U = 2;
    const int lane = threadIdx.x & 31, lanes = 1 << gl, t = lane & (lanes - 1);
    const int per = 32 >> gl;                                // segments a round
    const bool one = len > 0 && len <= (4 * VE << gl) && b - VE >= X0 && b + len + VE <= X1;
    unsigned rounds = gl < 5 ? __ballot_sync(kAll, one) : 0u;
    unsigned rest = __ballot_sync(kAll, len > 0) & ~rounds;
    const int small = rounds >> lane & 1u ? len : 0;
    for (int k = 0; rounds >> k; k += per) {
        const int i = k + (lane >> gl);
        const int64_t p0 = __shfl_sync(kAll, b, i);
        const int n = __shfl_sync(kAll, small, i);
        const int mis = (int)((p0 + shift) & (VE - 1));
        const int nv = n > 0 ? (n + mis + VE - 1) / VE : 0;
        const typename Ld::In* base = x + (p0 - mis);
        typename T::Acc acc = T::init();
        for (int j = t; __any_sync(kAll, j < nv); j += U * lanes) {
            Words<kGroupVec> w[U];
#pragma unroll
            for (int u = 0; u < U; u++)
                if (j + u * lanes < nv) w[u] = ldv<kGroupVec>(base + (j + u * lanes) * VE);
#pragma unroll
            for (int u = 0; u < U; u++) {
                if (j + u * lanes >= nv) continue;
                const int c = (j + u * lanes) * VE - mis;
                E e[VE];
                Ld::template dec<kGroupVec>(w[u], e);
                // bit i: element c + i belongs to the segment
                const int lo = c < 0 ? -c : 0, hi = n - c;
                const unsigned m = (hi >= VE ? (unsigned)((1ull << VE) - 1) : (1u << hi) - 1u) >> lo << lo;
                if constexpr (HasPad<T>::value) {
                    if (c < 0 || hi < VE) {
                        asm volatile("");   // (a branch)
#pragma unroll
                        for (int q = 0; q < VE; q++) e[q] = m >> q & 1u ? e[q] : T::pad();
                    }
                    if constexpr (T::kIdx) T::add_vec(acc, e, c);
                    else T::add_tree(acc, tree<T>(e));
                } else if (c >= 0 && hi >= VE) {
                    T::add_vec(acc, e, c);
                } else {
#pragma unroll
                    for (int q = 0; q < VE; q++)
                        if (m >> q & 1u) T::add(acc, e[q], c + q);
                }
            }
        }
        const Part p = group_combine<T>(T::to_part(acc), gl);
        if (t == 0 && n > 0) store_segment<T>(p, s0 + i, out, argidx, aux);
        if (k + per >= 32) break;
    }
    for (; rest; rest &= rest - 1) {
        const int i = __ffs(rest) - 1;
        const Part p = T::warp_reduce(
            group_part<T, 2>(x, __shfl_sync(kAll, b, i), __shfl_sync(kAll, len, i), shift, X0, X1, lane, 32));
        if (lane == 0) store_segment<T>(p, s0 + i, out, argidx, aux);
    }
}

template <class T>
__device__ __forceinline__ void rows_group_body(const RowGroupArgs& a) {
    using GR = GridR<T>;
    using G = typename GR::Part;
    const auto* x = static_cast<const typename T::Ld::In*>(a.x);
    const int lanes = 1 << a.gl;
    const int t = threadIdx.x & (lanes - 1);
    const int64_t r = ((int64_t)blockIdx.x * kGroupBlock + threadIdx.x) >> a.gl;
    const bool has = r < a.rows;
    typename T::Part p = group_part<T, 4>(x, has ? r * a.cols : 0, has ? (int)a.cols : 0, a.shift, 0, a.rows * a.cols,
                                          t, lanes);
    p = a.gl > 5 ? block_combine<T>(p) : group_combine<T>(p, a.gl);
    if (t == 0 && has) {
        const G g = GR::up(p);
        GR::store(a.out, r, g, false);
        GR::store_aux(a.argidx, a.aux, r, g, 0);
    }
}

// A trait that declares kGroupBlocks has that many blocks an SM at least (64
// registers at four: the sums and products of fp32 would take 72, three
// blocks, [32768, 1000] 24.6 us instead of 22.6).
template <class T, class = void>
struct GroupBlocks {
    static constexpr int value = 0;
};
template <class T>
struct GroupBlocks<T, std::void_t<decltype(T::kGroupBlocks)>> {
    static constexpr int value = T::kGroupBlocks;
};
template <class T>
__global__ void __launch_bounds__(kGroupBlock) k_rows_group(RowGroupArgs a) {
    rows_group_body<T>(a);
}
template <class T>
__global__ void __launch_bounds__(kGroupBlock, GroupBlocks<T>::value) k_rows_group_occ(RowGroupArgs a) {
    rows_group_body<T>(a);
}
template <class T>
constexpr auto rows_group_kernel() {
    if constexpr (GroupBlocks<T>::value > 0) return &k_rows_group_occ<T>;
    else return &k_rows_group<T>;
}

// ------------------------------------------------------------------------
// Segmented reduction
// ------------------------------------------------------------------------

struct Segs {
    const int64_t* off;
    int64_t cols, nseg, P0, P1;
    __device__ __forceinline__ int64_t raw(int64_t s) const { return off ? __ldg(off + s) : s * cols; }
    // segment bounds clamped to [P0, P1]: malformed offsets cannot move a read
    // outside the range the caller vouches for
    __device__ __forceinline__ int64_t clamp(int64_t b) const { return b < P0 ? P0 : (b > P1 ? P1 : b); }
    __device__ __forceinline__ int64_t begin(int64_t s) const { return clamp(raw(s)); }
    __device__ __forceinline__ int64_t end(int64_t s) const { return begin(s + 1); }
    // Largest s in [lo, nseg) with begin(s) <= p (requires begin(lo) <= p),
    // found by one warp (all 32 lanes call; every lane gets the answer).
    // begin() is non-decreasing, so {s : begin(s) <= p} is a prefix of
    // [lo, nseg): one coalesced probe of the next 32 segments settles the
    // common case (the answer is near lo), else a 32-ary search narrows the
    // interval 32-fold per round.
    __device__ int64_t find(int64_t lo, int64_t p, int lane) const {
        if (!off) {
            int64_t s = p / cols;
            s = s < lo ? lo : s;
            return s > nseg - 1 ? nseg - 1 : s;
        }
        int64_t hi = nseg - 1;
        {
            const int64_t q = lo + 1 + lane;
            const unsigned m = __ballot_sync(0xffffffffu, q <= hi && begin(q) <= p);
            if (m != 0xffffffffu) return lo + __popc(m);
            lo += 32;
        }
        while (lo < hi) {
            const int64_t step = (hi - lo + 32) / 32;
            const int64_t q = lo + (int64_t)lane * step;
            const unsigned m = __ballot_sync(0xffffffffu, q <= hi && begin(q) <= p);
            const int last = 31 - __clz(m);
            lo = lo + (int64_t)last * step;
            hi = lo + step - 1 < hi ? lo + step - 1 : hi;
        }
        return lo;
    }
};

// Batches q, q + nwarp, ... of 2^batch neighbouring segments, one a warp at a
// time (batch <= 5), none longer than `most`.  Empty segments get the
// identity, malformed offsets raise the error word.
template <class T>
__device__ __forceinline__ void segment_batches(const Segs& sg, const typename T::Ld::In* x, int shift, int batch,
                                                int64_t q, int64_t nwarp, int64_t most, void* out, int64_t* argidx,
                                                pr_prod_aux* aux, int* err) {
    const int lane = threadIdx.x & 31;
    const int64_t nbatch = (sg.nseg + ((int64_t)1 << batch) - 1) >> batch;
    int gl = group_lanes<typename T::Ld>((sg.P1 - sg.P0) / sg.nseg);
    if (gl < 5 - batch) gl = 5 - batch;          // a short batch has lanes to spare
    for (; q < nbatch; q += nwarp) {
        const int64_t s = (q << batch) + lane;
        const bool mine = lane < (1 << batch) && s < sg.nseg;
        const int64_t rb = mine ? sg.raw(s) : 0, re = mine ? sg.raw(s + 1) : 0;
        if (mine && (rb > re || rb < 0)) atomicOr(err, kErrInvalid);
        const int64_t b = sg.clamp(rb), len = mine ? sg.clamp(re) - b : 0;
        if (mine && len == 0) T::store_empty(out, s, false, argidx, aux);
        warp_segments<T>(x, shift, sg.P0, sg.P1, q << batch, b, len > 0 && len <= most ? (int)len : 0, gl, out, argidx,
                         aux);
    }
}

template <class T, int U, int VB>
struct SegCtx {
    using Ld = typename T::Ld;
    using In = typename Ld::In;
    using E = typename Ld::E;
    static constexpr int VE = VB / Ld::ES;
    const In* x;
    Segs sg;
    int64_t P0, P1;

    // Accumulate the elements with position in [lo, hi) among the U vectors
    // this thread owns in the tile starting at position tlo.
    __device__ __forceinline__ void masked(typename T::Acc (&acc)[U], int64_t tlo, int64_t lo, int64_t hi) const {
        if (lo >= hi) return;
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t vp = tlo + ((int64_t)u * blockDim.x + threadIdx.x) * VE;
            if (vp + VE <= lo || vp >= hi) continue;
            if (vp >= P0 && vp + VE <= P1) {
                const Words<VB> w = ldv<VB>(x + vp);
                E e[VE];
                Ld::template dec<VB>(w, e);
#pragma unroll
                for (int k = 0; k < VE; k++)
                    if (vp + k >= lo && vp + k < hi) T::add(acc[u], e[k], vp + k);
            } else {
                const int64_t a0 = vp > lo ? vp : lo;
                const int64_t a1 = vp + VE < hi ? vp + VE : hi;
                for (int64_t p = a0; p < a1; p++) T::add(acc[u], Ld::one(x, p), p);
            }
        }
    }
};

// Same as SegCtx::masked, from vectors already loaded for an interior tile.
template <class T, int U, int VB>
__device__ __forceinline__ void masked_words(typename T::Acc (&acc)[U], const Words<VB> (&w)[U], int64_t tlo,
                                             int64_t lo, int64_t hi) {
    using Ld = typename T::Ld;
    using E = typename Ld::E;
    constexpr int VE = VB / Ld::ES;
    if (lo >= hi) return;
#pragma unroll
    for (int u = 0; u < U; u++) {
        const int64_t vp = tlo + ((int64_t)u * blockDim.x + threadIdx.x) * VE;
        if (vp + VE <= lo || vp >= hi) continue;
        E e[VE];
        Ld::template dec<VB>(w[u], e);
#pragma unroll
        for (int k = 0; k < VE; k++)
            if (vp + k >= lo && vp + k < hi) T::add(acc[u], e[k], vp + k);
    }
}

template <class T, int U, int VB>
__global__ void __launch_bounds__(512) k_segmented(SegArgs a) {
    using Ld = typename T::Ld;
    using In = typename Ld::In;
    using E = typename Ld::E;
    using Acc = typename T::Acc;
    using Part = typename T::Part;
    constexpr int VE = VB / Ld::ES;
    const In* x = static_cast<const In*>(a.x);
    const int64_t nseg = a.nseg;
    const bool f64 = a.out_f64 != 0;
    const int64_t gtid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t nth = (int64_t)gridDim.x * blockDim.x;
    if (nseg <= 0) return;

    Segs sg{a.off, a.cols, nseg, 0, 0};
    const int64_t raw0 = sg.raw(0), rawN = sg.raw(nseg);
    const int64_t P0 = raw0 < 0 ? 0 : raw0;
    const int64_t P1 = rawN < P0 ? P0 : rawN;
    sg.P0 = P0;
    sg.P1 = P1;

    // Segments that are all short go to groups of lanes (see k_seg_group; this
    // kernel has the launches of fewer than kSegGroupMin of them, where every
    // block can look at all lengths for itself).
    if (a.off && nseg < kSegGroupMin && P1 - P0 <= nseg * kGroupMean) {
        bool longer = false;
        for (int64_t s = threadIdx.x; s < nseg; s += blockDim.x) longer |= sg.end(s) - sg.begin(s) > kGroupMost;
        if (!__syncthreads_or(longer)) {
            const int64_t nwarp = nth >> 5;
            int batch = 5;
            while (batch > 0 && (nseg >> batch) < nwarp) batch--;
            segment_batches<typename GroupTrait<T>::type>(sg, x, (int)(reinterpret_cast<uintptr_t>(x) % kGroupVec) / Ld::ES, batch, gtid >> 5,
                               nwarp, kGroupMost, a.out, a.argidx, a.aux, a.ws.err);
            return;
        }
    }

    // Empty segments get the identity; malformed offsets raise the error word.
    for (int64_t s = gtid; s < nseg; s += nth) {
        const int64_t rb = sg.raw(s), re = sg.raw(s + 1);
        if (rb > re || rb < 0) atomicOr(a.ws.err, kErrInvalid);
        if (sg.begin(s) == sg.end(s)) T::store_empty(a.out, s, f64, a.argidx, a.aux);
    }
    if (P1 <= P0) return;

    const int B = blockDim.x;
    const int64_t TILE = (int64_t)B * VE * U;
    const int64_t shift = a.shift;
    const int64_t J0 = ((P0 + shift) / VE) * VE;  // first VB boundary at or before P0
    const int64_t ntiles = (P1 + shift - J0 + TILE - 1) / TILE;
    // chunks: a few per block, at most one slot pair per chunk
    int64_t nchunk = (int64_t)a.chunks_per_block * gridDim.x;
    nchunk = nchunk < a.ws.gmax ? nchunk : a.ws.gmax;
    nchunk = nchunk < ntiles ? nchunk : ntiles;
    const int64_t K = (ntiles + nchunk - 1) / nchunk;  // tiles per chunk
    nchunk = (ntiles + K - 1) / K;                      // chunks that hold tiles
    const int64_t CB = K * TILE;

    SegCtx<T, U, VB> ctx{x, sg, P0, P1};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = B >> 5;

    __shared__ int64_t s_i64;
    __shared__ int s_fin;
    __shared__ unsigned s_chunk;
    using GR = GridR<T>;
    using G = typename GR::Part;

    for (int64_t iter = 0;; iter++) {
        int64_t c;
        if (a.dynamic_chunks) {
            __syncthreads();  // s_chunk / s_i64 of the previous chunk are consumed
            if (threadIdx.x == 0) s_chunk = atomicAdd(a.ws.chunk_ctr, 1u);
            __syncthreads();
            c = s_chunk;
        } else {
            c = blockIdx.x + iter * gridDim.x;
        }
        if (c >= nchunk) break;
        const int64_t t0 = c * K;
        const int64_t t1 = t0 + K < ntiles ? t0 + K : ntiles;
        const int64_t blk_lo = (J0 + t0 * TILE - shift) > P0 ? (J0 + t0 * TILE - shift) : P0;
        const int64_t blk_hi = (J0 + t1 * TILE - shift) < P1 ? (J0 + t1 * TILE - shift) : P1;

        // Finish this chunk's piece of segment s (all threads call).
        auto emit = [&](int64_t s, Acc (&acc)[U]) {
            const Part p = block_combine<T>(fold<T, U>(acc));
#pragma unroll
            for (int u = 0; u < U; u++) acc[u] = T::init();
            const int64_t sb = sg.begin(s), se = sg.end(s);
            if (sb >= blk_lo && se <= blk_hi) {
                if (threadIdx.x == 0) {
                    const G g = GR::up(p);
                    GR::store(a.out, s, g, f64);
                    GR::store_aux(a.argidx, a.aux, s, g, sb);
                }
                return;
            }
            const int64_t ba = (sb + shift - J0) / CB, bb = (se - 1 + shift - J0) / CB;
            if (threadIdx.x == 0) {
                *slot<GR>(sb < blk_lo ? a.ws.head : a.ws.tail, c) = GR::up(p);
                __threadfence();
                const unsigned old = atomicAdd(a.ws.seg_cnt + ba, 1u);
                s_fin = (old == (unsigned)(bb - ba));
            }
            __syncthreads();
            if (s_fin) {
                // the whole block combines the segment's chunk partials (a
                // segment can span every chunk of the launch)
                __threadfence();
                G q = GR::part_init();
                for (int64_t k = threadIdx.x; k <= bb - ba; k += B)
                    q = GR::combine(q, ld_cg_any(k == 0 ? slot<GR>(a.ws.tail, ba) : slot<GR>(a.ws.head, ba + k)));
                q = block_combine<GR>(q);
                if (threadIdx.x == 0) {
                    GR::store(a.out, s, q, f64);
                    GR::store_aux(a.argidx, a.aux, s, q, sb);
                    a.ws.seg_cnt[ba] = 0u;
                }
            }
            __syncthreads();
        };

        // Tiles lying wholly inside [P0, P1) are "interior": their vectors are
        // loaded one tile ahead, so loads stay in flight through the block
        // combines at segment boundaries (and through the search below).
        auto interior = [&](int64_t t) {
            const int64_t l = J0 + t * TILE - shift;
            return l >= P0 && l + TILE <= P1;
        };
        auto load_tile = [&](int64_t t, Words<VB> (&w)[U]) {
            const int64_t l = J0 + t * TILE - shift;
#pragma unroll
            for (int u = 0; u < U; u++) w[u] = ldv<VB>(x + l + ((int64_t)u * B + threadIdx.x) * VE);
        };
        Words<VB> wn[U];
        bool have = t0 < t1 && interior(t0);
        if (have) load_tile(t0, wn);

        if (warp == 0) {
            const int64_t r = sg.find(0, blk_lo, lane);
            if (lane == 0) s_i64 = r;
        }
        __syncthreads();
        int64_t cs = s_i64;
        int64_t cend = sg.end(cs);

        Acc acc[U];
#pragma unroll
        for (int u = 0; u < U; u++) acc[u] = T::init();

        for (int64_t t = t0; t < t1; t++) {
            const int64_t tlo = J0 + t * TILE - shift, thi = tlo + TILE;
            Words<VB> w[U];
#pragma unroll
            for (int u = 0; u < U; u++) w[u] = wn[u];
            const bool cur = have;
            have = t + 1 < t1 && interior(t + 1);
            if (have) load_tile(t + 1, wn);
            if (cur && cend >= thi) {
                // the whole tile lies inside segment cs: stream it
#pragma unroll
                for (int u = 0; u < U; u++) {
                    E e[VE];
                    Ld::template dec<VB>(w[u], e);
                    T::add_vec(acc[u], e, tlo + ((int64_t)u * B + threadIdx.x) * VE);
                }
                continue;
            }
            // accumulate positions [p0, p1) of this tile into ac
            auto part = [&](Acc (&ac)[U], int64_t p0, int64_t p1) {
                if (cur) masked_words<T, U, VB>(ac, w, tlo, p0, p1);
                else ctx.masked(ac, tlo, p0, p1);
            };
            const int64_t lo = tlo > P0 ? tlo : P0, hi = thi < P1 ? thi : P1;
            if (cend >= hi) {
                part(acc, lo, hi);
                continue;
            }
            // segment cs ends inside this tile
            part(acc, lo, cend);
            emit(cs, acc);
            __syncthreads();
            if (warp == 0) {
                const int64_t r = sg.find(cs + 1, hi - 1, lane);
                if (lane == 0) s_i64 = r;
            }
            __syncthreads();
            const int64_t ns = s_i64;
            // segments lying wholly inside the tile: short ones one per warp ...
            for (int64_t s = cs + 1 + warp; s < ns; s += nwarps) {
                const int64_t sb = sg.begin(s), se = sg.end(s);
                if (se == sb || se - sb > kSmallSeg) continue;
                Acc wa = T::init();
                int64_t p = sb + lane;
                for (; p + 96 < se; p += 128) {
                    const E v0 = Ld::one(x, p), v1 = Ld::one(x, p + 32), v2 = Ld::one(x, p + 64), v3 = Ld::one(x, p + 96);
                    T::add(wa, v0, p);
                    T::add(wa, v1, p + 32);
                    T::add(wa, v2, p + 64);
                    T::add(wa, v3, p + 96);
                }
                for (; p < se; p += 32) T::add(wa, Ld::one(x, p), p);
                const Part q = T::warp_reduce(T::to_part(wa));
                if (lane == 0) {
                    const G g = GR::up(q);
                    GR::store(a.out, s, g, f64);
                    GR::store_aux(a.argidx, a.aux, s, g, sb);
                }
            }
            // ... long ones with the whole block
            for (int64_t s = cs + 1; s < ns; s++) {
                const int64_t sb = sg.begin(s), se = sg.end(s);
                if (se - sb <= kSmallSeg) continue;
                Acc ba_[U];
#pragma unroll
                for (int u = 0; u < U; u++) ba_[u] = T::init();
                part(ba_, sb, se);
                const Part q = block_combine<T>(fold<T, U>(ba_));
                if (threadIdx.x == 0) {
                    const G g = GR::up(q);
                    GR::store(a.out, s, g, f64);
                    GR::store_aux(a.argidx, a.aux, s, g, sb);
                }
            }
            cs = ns;
            cend = sg.end(cs);
            part(acc, sg.begin(ns), hi);
        }
        emit(cs, acc);
    }
    // the last block out re-arms the chunk counter for the next launch
    if (a.dynamic_chunks && threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(a.ws.blk_done, 1u) == gridDim.x - 1) {
            *a.ws.chunk_ctr = 0u;
            *a.ws.blk_done = 0u;
        }
    }
}

// ------------------------------------------------------------------------
// Many segments
// ------------------------------------------------------------------------

__device__ __forceinline__ Segs seg_bounds(const int64_t* off, int64_t nseg) {
    Segs sg{off, 0, nseg, 0, 0};
    const int64_t raw0 = sg.raw(0), rawN = sg.raw(nseg);
    sg.P0 = raw0 < 0 ? 0 : raw0;
    sg.P1 = rawN < sg.P0 ? sg.P0 : rawN;
    return sg;
}

// 1. All but the long segments, up to 32 neighbours a warp at a time; the
// long ones are listed as tasks of at most a chunk.
//
// Short segments (at most kStageMean bytes on average) are staged: a batch of
// neighbours is one contiguous run, copied to the warp's shared memory, so
// that loads are whole and coalesced whatever the lengths, and a group's
// lanes read their segment element by element, with no vector cut by a
// segment's end.  A batch that does not fit (or reaches the ends of x, or
// holds a long segment) is reduced from x directly.  One stage a warp: the
// other warps of the SM cover its wait, and a second stage would take the
// shared memory that the L1 cache needs for the loads in flight of the direct
// path and of k_seg_long (measured: 8192 segments of 40000 254 us with two
// stages, 207 with one).  Five blocks an SM: 96 registers, the most that no
// trait of 32-bit types spills at (10^6 segments of 24, summed plainly: 50 us; six
// blocks 53, eight 53; 105 against 107 and 118 for the maximum with index; the
// maximum with index of 16-bit types spills 80 bytes).
constexpr int kSegBlock = 128;
constexpr int kStageBytes = 4096;    // a warp's stage: one batch
constexpr int kStageMean = 512;

template <class T>
__global__ void __launch_bounds__(kSegBlock, 5) k_seg_group(SegGroupArgs a) {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // k_seg_long may take its place as blocks leave
    using Ld = typename T::Ld;
    using In = typename Ld::In;
    using Part = typename T::Part;
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int VE = kGroupVec / Ld::ES, CAP = kStageBytes / Ld::ES, PE = 16 / Ld::ES;
    __shared__ __align__(32) unsigned char s_stage[kSegBlock / 32][kStageBytes];
    const In* x = static_cast<const In*>(a.x);
    const Segs sg = seg_bounds(a.off, a.nseg);
    const SegSplit sp = seg_split_lengths(sg.P1 - sg.P0, a.nseg, a.tasks);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nwarp = (int64_t)gridDim.x * (kSegBlock / 32);
    const int64_t mean = (sg.P1 - sg.P0) / a.nseg;
    const bool stage = mean * Ld::ES <= kStageMean;
    int batch = 5;
    while (batch > 0 && (a.nseg >> batch) < nwarp) batch--;
    if (stage)
        while (batch > 1 && mean << batch > CAP * 3 / 4) batch--;   // (mean <= CAP / 8)
    const int64_t nbatch = (a.nseg + ((int64_t)1 << batch) - 1) >> batch;
    int gl = group_lanes<Ld>(mean);
    if (gl < 5 - batch) gl = 5 - batch;          // a short batch has lanes to spare
    const In* v = reinterpret_cast<const In*>(s_stage[warp]);
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(s_stage[warp]);

    // this lane's segment of batch w (raw bounds)
    auto load = [&](int64_t w, int64_t& b, int64_t& e) {
        const int64_t s = (w << batch) + lane;
        const bool mine = lane < (1 << batch) && s < a.nseg && w < nbatch;
        b = mine ? sg.raw(s) : 0;
        e = mine ? sg.raw(s + 1) : 0;
    };
    int64_t q = (int64_t)blockIdx.x * (kSegBlock / 32) + warp;
    int64_t nb, ne;
    load(q, nb, ne);
    for (; q < nbatch; q += nwarp) {
        const int64_t rb = nb, re = ne, s0 = q << batch;
        const bool mine = lane < (1 << batch) && s0 + lane < a.nseg;
        const unsigned in = __ballot_sync(kAll, mine);
        if (stage) {
            // well-formed, inside [P0, P1) with the vectors around it, and
            // short enough: 32-bit places from the first staged element on
            const int64_t p0 = __shfl_sync(kAll, rb, 0);
            const int mis = (int)((p0 + a.shift) & (VE - 1));
            const int64_t base = p0 - mis;
            const uint64_t ob = (uint64_t)(rb - base), oe = (uint64_t)(re - base);
            const bool ok = !mine || (ob <= oe && oe <= (uint64_t)(CAP - VE));
            const int n = __shfl_sync(kAll, (int)oe, 31 - __clz(in));
            const int pieces = (n + PE - 1) / PE;                                  // 16 bytes each
            if (__all_sync(kAll, ok) && base >= sg.P0 && base + pieces * PE <= sg.P1) {
                const char* src = reinterpret_cast<const char*>(x + base);
                for (int i = lane; i < pieces; i += 32)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i * 16), "l"(src + i * 16) : "memory");
                load(q + nwarp, nb, ne);
                asm volatile("cp.async.wait_all;" ::: "memory");
                __syncwarp();
                const int lanes = 1 << gl, t = lane & (lanes - 1);
                const int r0 = (int)ob, n0 = mine ? (int)oe - r0 : 0;
                if (mine && n0 == 0) T::store_empty(a.out, s0 + lane, false, a.argidx, a.aux);
                for (int k = 0; k < 1 << batch; k += 32 >> gl) {
                    const int i = k + (lane >> gl);
                    const In* run = v + __shfl_sync(kAll, r0, i);
                    const int len = __shfl_sync(kAll, n0, i);
                    typename T::Acc acc = T::init();
                    int j = t;
                    // four a step, as a tree where the trait has no index: a
                    // shorter chain of operations and of roundings
                    for (; j + 3 * lanes < len; j += 4 * lanes) {
                        const typename Ld::E e[4] = {Ld::lone(run[j]), Ld::lone(run[j + lanes]),
                                                     Ld::lone(run[j + 2 * lanes]), Ld::lone(run[j + 3 * lanes])};
                        if constexpr (HasPad<T>::value && !T::kIdx) {
                            T::add_tree(acc, tree<T>(e));
                        } else if constexpr (!T::kIdx) {
                            T::add_vec(acc, e, 0);
                        } else {
#pragma unroll
                            for (int q = 0; q < 4; q++) T::add(acc, e[q], j + q * lanes);
                        }
                    }
                    if constexpr (HasPad<T>::value && !T::kIdx) {
                        typename Ld::E e[3];
#pragma unroll
                        for (int q = 0; q < 3; q++) e[q] = j + q * lanes < len ? Ld::lone(run[j + q * lanes]) : T::pad();
                        T::add_rest(acc, tree<T>(e));
                    } else {
#pragma unroll
                        for (int q = 0; q < 3; q++)
                            if (j + q * lanes < len) T::add(acc, Ld::lone(run[j + q * lanes]), j + q * lanes);
                    }
                    const Part p = group_combine<T>(T::to_part(acc), gl);
                    if (t == 0 && len > 0) store_segment<T>(p, s0 + i, a.out, a.argidx, a.aux);
                }
                __syncwarp();
                continue;
            }
        }
        load(q + nwarp, nb, ne);
        if (mine && (rb > re || rb < 0)) atomicOr(a.ws.err, kErrInvalid);
        const int64_t b = sg.clamp(rb), len = mine ? sg.clamp(re) - b : 0;
        if (mine && len == 0) T::store_empty(a.out, s0 + lane, false, a.argidx, a.aux);
        unsigned big = __ballot_sync(kAll, len > sp.most);
        if (big) {
            const unsigned n = big >> lane & 1u ? seg_chunks(len, sp) : 0u;
            const SegCount first = n ? atomicAdd(a.ws.task_count, (SegCount)n) : 0u;
            // (malformed offsets may ask for more tasks than there are: the
            // segments past the end of the list stay unset)
            const unsigned listed = seg_listed(first, n, a.tasks);
            if (listed < n) atomicOr(a.ws.err, kErrInvalid);
            for (; big; big &= big - 1) {
                const int i = __ffs(big) - 1;
                const unsigned f = __shfl_sync(kAll, (unsigned)first, i), c = __shfl_sync(kAll, listed, i);
                for (unsigned k = lane; k < c; k += 32) a.ws.tasks[f + k] = SegTask{s0 + i, f, 0u};
            }
        }
        warp_segments<T>(x, a.shift, sg.P0, sg.P1, s0, b, len > 0 && len <= sp.most ? (int)len : 0, gl, a.out, a.argidx,
                         a.aux);
    }
}

// 2. The long segments: tasks claimed from a counter by warps, which wait for
// nobody: the next claim, then the next task's record, then its offsets load
// while a task's elements travel.  A segment's partials go by task index;
// the warp that stores the last one of 64 neighbours combines them, and the
// one that finishes the last 64 combines those, in order both times.
constexpr unsigned kTaskGroup = 64;

template <class T>
__device__ __forceinline__ void seg_long_body(const SegGroupArgs& a) {
    using Part = typename T::Part;
    constexpr unsigned kAll = 0xffffffffu;
    const auto* x = static_cast<const typename T::Ld::In*>(a.x);
    const Segs sg = seg_bounds(a.off, a.nseg);
    const SegSplit sp = seg_split_lengths(sg.P1 - sg.P0, a.nseg, a.tasks);
    const int lane = threadIdx.x & 31;
    asm volatile("griddepcontrol.wait;" ::: "memory");   // k_seg_group is done and its list visible
    const SegCount asked = __ldcg(a.ws.task_count);
    const unsigned ntask = asked < a.tasks ? (unsigned)asked : a.tasks;
    Part* parts = reinterpret_cast<Part*>(a.ws.head);
    auto claim = [&]() { return lane == 0 ? atomicAdd(a.ws.chunk_ctr, 1u) : 0u; };
    auto record = [&](unsigned k, int64_t& s, unsigned& first) {
        s = k < ntask ? __ldcg(reinterpret_cast<const long long*>(&a.ws.tasks[k].seg)) : 0;
        first = k < ntask ? __ldcg(&a.ws.tasks[k].first) : 0u;
    };
    if (ntask) {
        unsigned k = __shfl_sync(kAll, claim(), 0), first;
        int64_t s;
        record(k, s, first);
        int64_t b = sg.begin(s), e = sg.end(s);
        unsigned k1 = claim();
        while (k < ntask) {
            k1 = __shfl_sync(kAll, k1, 0);
            const unsigned k2 = claim();
            int64_t s1;
            unsigned first1;
            record(k1, s1, first1);
            const unsigned c = k - first;                    // this chunk of the segment
            const int64_t len = e - b, c0 = (int64_t)c * sp.chunk, left = len - c0;
            const unsigned chunks = seg_chunks(len, sp);
            Part p = group_part<T, 4>(x, b + c0, (int)(left < sp.chunk ? left : sp.chunk), a.shift, sg.P0, sg.P1, lane,
                                      32, c0);
            const int64_t b1 = sg.begin(s1), e1 = sg.end(s1);
            p = T::warp_reduce(p);
            if (chunks == 1) {
                if (lane == 0) store_segment<T>(p, s, a.out, a.argidx, a.aux);
            } else {
                // c's group of chunks [g0, g0 + n), counted in its first task
                const unsigned g0 = c / kTaskGroup * kTaskGroup;
                const unsigned n = chunks - g0 < kTaskGroup ? chunks - g0 : kTaskGroup;
                unsigned done = 0u;
                if (lane == 0) {
                    parts[k] = p;
                    __threadfence();
                    done = atomicAdd(&a.ws.tasks[first + g0].finished, 1u) == n - 1;
                }
                if (__shfl_sync(kAll, done, 0)) {
                    __threadfence();
                    auto gather = [&](unsigned from, unsigned count, unsigned step) {
                        Part q = T::part_init();
                        for (unsigned i = lane; i < count && from + i * step < a.tasks; i += 32)
                            q = T::combine(q, ld_cg_any(parts + from + i * step));
                        return T::warp_reduce(q);
                    };
                    Part q = gather(first + g0, n, 1);
                    const unsigned groups = (chunks + kTaskGroup - 1) / kTaskGroup;
                    bool last = groups == 1;
                    if (!last) {
                        // the groups of a segment are counted in its second task
                        done = 0u;
                        if (lane == 0) {
                            parts[first + g0] = q;
                            __threadfence();
                            done = atomicAdd(&a.ws.tasks[first + 1].finished, 1u) == groups - 1;
                        }
                        last = __shfl_sync(kAll, done, 0) != 0u;
                        if (last) {
                            __threadfence();
                            q = gather(first, groups, kTaskGroup);
                        }
                    }
                    if (last && lane == 0) store_segment<T>(q, s, a.out, a.argidx, a.aux);
                }
            }
            k = k1;
            k1 = k2;
            s = s1;
            first = first1;
            b = b1;
            e = e1;
        }
    }
    // The last block out clears the counters for the next launch.
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(a.ws.blk_done, 1u) == gridDim.x - 1) {
            *a.ws.chunk_ctr = 0u;
            *a.ws.task_count = 0;
            *a.ws.blk_done = 0u;
        }
    }
}

// A trait that declares kLongBlocks has that many blocks an SM at least (80
// registers at three: the sums and products of 16-bit types would take 92,
// two blocks, 8192 segments of 40000 bf16 137 us instead of 120).
template <class T, class = void>
struct LongBlocks {
    static constexpr int value = 0;
};
template <class T>
struct LongBlocks<T, std::void_t<decltype(T::kLongBlocks)>> {
    static constexpr int value = T::kLongBlocks;
};
template <class T>
__global__ void __launch_bounds__(kGroupBlock) k_seg_long(SegGroupArgs a) {
    seg_long_body<T>(a);
}
template <class T>
__global__ void __launch_bounds__(kGroupBlock, LongBlocks<T>::value) k_seg_long_occ(SegGroupArgs a) {
    seg_long_body<T>(a);
}
template <class T>
constexpr auto seg_long_kernel() {
    if constexpr (LongBlocks<T>::value > 0) return &k_seg_long_occ<T>;
    else return &k_seg_long<T>;
}

}  // namespace pr
