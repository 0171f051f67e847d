// Reduction along the middle axis of a contiguous row-major [outer, n, inner]
// array: out[p, q] = x[p, 0, q] (x) x[p, 1, q] (x) ... (x) x[p, n-1, q].  With
// outer = the product of the leading sizes and inner = the product of the
// trailing ones this is the reduction of any one axis of a contiguous tensor
// (Section 1.1's reduction, applied to every column of every [n, inner] slab).
//
// k_axis    one warp per (slab p, group of column vectors, split of the rows).
//   A lane owns one column vector (VB bytes; VB = 0: one element) and keeps
//   one accumulator per element of it.  When a row holds fewer than 32 column
//   vectors, a warp covers 32/bx rows per step (bx lanes per row), so every
//   load instruction still touches 32 neighbouring vectors.  Each lane issues
//   U rows' loads before accumulating any of them.  The lanes that share a
//   column then combine by an xor butterfly over the row bits of the lane
//   index, in a fixed order.  Where tiles alone leave warps idle, the warps of
//   a block share a tile's rows first and combine through shared memory (as a
//   tree), and only then are the rows split over blocks: a partial per
//   warp and output cost more traffic than the input where the axis is short
//   ([64, 577, 768] fp32 maximum with index: 49 splits wrote and read 38 MB
//   each of 16-byte partials for 113 MB of input; with shared splits 77 -> 27
//   us, 0.62 of a 6.8 TB/s copy: one wave of blocks, bound by latency).  A lane
//   then takes more rows of a column than a split's lane did, so sums and
//   products take the AxisTrait form, which keeps what they round off (error
//   of the fp32 sum of [1, 5000, 4096] 1.2e-7 with splits of a warp, 1.5e-7 by
//   plain chains, 7.8e-8 now; fp64 2.1e-16, 2.8e-16, 2.0e-16).  With one split
//   the outputs are written; with more, the partials, and k_axis_finish combines each output's
//   partials in a fixed order (one thread per output folding the splits as
//   trees of eight, or with many splits one warp per output and a fixed tree), so
//   results are deterministic for a fixed launch shape.
// k_axis_backward  gradient of an axis reduction: grad_in[p, i, q] from
//   grad_out[p, q] and the per-output state, one streaming write.
#pragma once
#include "kernels.cuh"

namespace pr {

struct AxisArgs {
    const void* x;
    int64_t outer, n, inner;
    int64_t qv;               // column vectors per row: inner / VE
    int bx;                   // lanes per row (power of two, <= 32)
    int64_t groups;           // column groups per row: ceil(qv / bx)
    int64_t splits;           // row splits that leave a partial each (one warp's, or a block's)
    int coop;                 // warps of a block that share a split (k_axis COOP; else 1)
    int64_t rows_per_split;   // rows of one warp
    void* out;
    int64_t* argidx;
    pr_prod_aux* aux;
    int out_f64;
    char* scratch;            // splits > 1: partials of GridR<T>::Part, [split][output] when
                              // splits <= kAxisThreadFinish, else [output][split]
};

// Up to this many splits the finishing pass takes one thread per output
// (coalesced over outputs); beyond it, one warp per output.
constexpr int kAxisThreadFinish = 64;
// Most warps of a block that share a split (their partials meet in shared memory).
constexpr int kAxisCoop = 8;

// A column's elements reach its accumulator in increasing index order, so a
// trait may take them with a cheaper in-order step (add_ordered).
template <class T, class = void>
struct HasOrdered : std::false_type {};
template <class T>
struct HasOrdered<T, std::void_t<decltype(&T::add_ordered)>> : std::true_type {};

// A trait whose in-order step runs on a caller's (value, row) register pair
// (kOrderedPair: the arg-extremum of floats).
template <class T, class = void>
struct HasOrderedPair : std::false_type {};
template <class T>
struct HasOrderedPair<T, std::void_t<decltype(T::kOrderedPair)>> : std::true_type {};

template <class T>
__device__ __forceinline__ void add_in_order(typename T::Acc& a, typename T::Ld::E v, int64_t i) {
    if constexpr (HasOrdered<T>::value) T::add_ordered(a, v, i);
    else T::add(a, v, i);
}

// What the warps that share a split exchange: Parts, or a trait's accumulators
// where it can merge them (no rounding lost, and no fp64 operation a warp).
template <class T, class = void>
struct ColPart {
    using P = typename T::Part;
    __device__ __forceinline__ static P from(const typename T::Acc& a) { return T::to_part(a); }
    __device__ __forceinline__ static P combine(const P& a, const P& b) { return T::combine(a, b); }
    __device__ __forceinline__ static typename T::Part part(const P& p) { return p; }
};
template <class T>
struct ColPart<T, std::void_t<decltype(&T::merge)>> {
    using P = typename T::Acc;
    __device__ __forceinline__ static P from(const typename T::Acc& a) { return a; }
    __device__ __forceinline__ static P combine(const P& a, const P& b) { return T::merge(a, b); }
    __device__ __forceinline__ static typename T::Part part(const P& p) { return T::to_part(p); }
};

// Column elements (a divisor of VE) whose partials of kAxisCoop warps meet in
// shared memory at a time: up to 16 KB.
template <class T, int VE>
struct AxisPhase {
    static constexpr int kBytes = kAxisCoop * 32 * (int)sizeof(typename ColPart<T>::P);
    static constexpr int fit(int k) { return k > 1 && k * kBytes > 16384 ? fit(k / 2) : k; }
    static constexpr int value = fit(VE);
};

template <int VB, class Ld>
__device__ __forceinline__ void axis_load(const typename Ld::In* x, int64_t e0, typename Ld::E (&e)[VB ? VB / Ld::ES : 1]) {
    if constexpr (VB == 0) {
        e[0] = Ld::one(x, e0);
    } else {
        const Words<VB> w = ldv<VB>(x + e0);
        Ld::template dec<VB>(w, e);
    }
}

// COOP: the variant whose blocks' warps share a split (a.coop of them, the
// whole block).  It is compiled apart because its shared memory and registers
// cost the other resident warps ([4096, 16, 512] fp64 minimum with index 79 us
// without it in the kernel, 91 with).  Its sums spill a little at the compiler's
// choice of registers (fp32 16 bytes at 64, 16-bit 12 at 80, where the fp64
// product's state spills 12 too).
template <class T, int U, int VB, bool COOP>
__global__ void __launch_bounds__(COOP ? 32 * kAxisCoop : MaxBlock<T>::value) k_axis(AxisArgs a) {
    using Ld = typename T::Ld;
    using In = typename Ld::In;
    using E = typename Ld::E;
    using Acc = typename T::Acc;
    using Part = typename T::Part;
    using GR = GridR<T>;
    using G = typename GR::Part;
    constexpr int VE = VB ? VB / Ld::ES : 1;
    const In* x = static_cast<const In*>(a.x);
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // k_axis_finish waits for this grid's end
    const int lane = threadIdx.x & 31;
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t tiles = a.outer * a.groups;
    const int64_t wsplits = a.splits * a.coop;                   // warps per tile
    if (wid >= tiles * wsplits) return;  // whole warps (blockDim is a multiple of 32); none where warps share a split
    const int64_t tile = wid / wsplits, ws = wid - tile * wsplits;
    const int64_t s = ws / a.coop;
    const int64_t p = tile / a.groups, grp = tile - p * a.groups;
    const int bx = a.bx, ry = 32 / bx;
    const int tx = lane & (bx - 1), ty = lane / bx;
    const int64_t col = grp * bx + tx;
    const bool has = col < a.qv;
    const int64_t r0 = ws * a.rows_per_split;
    const int64_t r1 = r0 + a.rows_per_split < a.n ? r0 + a.rows_per_split : a.n;
    const int64_t slab = p * a.n * a.inner + col * VE;  // element offset of (p, row 0, this column)

    Acc acc[VE];
#pragma unroll
    for (int k = 0; k < VE; k++) acc[k] = T::init();
    if constexpr (HasOrderedPair<T>::value) {
        // per element the running extremum and its row relative to r0 (a
        // split holds fewer than 2^31 rows): three operations an element
        // (pick, compare of bits, select) instead of the accumulator's
        // 64-bit index and its "none yet" test; started at this lane's first
        // row, picked against itself so that a NaN has the bits that later
        // picks give it (any other payload would read as a change, and take
        // the index of the next row), then the same steps as add_ordered
        if (has && r0 + ty < r1) {
            float sv[VE];
            int so[VE];
            int64_t r = r0 + ty;
            {
                E e[VE];
                axis_load<VB, Ld>(x, slab + r * a.inner, e);
#pragma unroll
                for (int k = 0; k < VE; k++) {
                    sv[k] = T::ordered_pick(e[k], e[k]);
                    so[k] = (int)(r - r0);
                }
            }
            r += ry;
            for (; r + (int64_t)(U - 1) * ry < r1; r += (int64_t)U * ry) {
                E e[U][VE];
#pragma unroll
                for (int u = 0; u < U; u++) axis_load<VB, Ld>(x, slab + (r + (int64_t)u * ry) * a.inner, e[u]);
#pragma unroll
                for (int u = 0; u < U; u++) {
                    const int rel = (int)(r + (int64_t)u * ry - r0);
#pragma unroll
                    for (int k = 0; k < VE; k++) {
                        const float m = T::ordered_pick(sv[k], e[u][k]);
                        so[k] = __float_as_uint(m) != __float_as_uint(sv[k]) ? rel : so[k];
                        sv[k] = m;
                    }
                }
            }
            for (; r < r1; r += ry) {
                E e[VE];
                axis_load<VB, Ld>(x, slab + r * a.inner, e);
                const int rel = (int)(r - r0);
#pragma unroll
                for (int k = 0; k < VE; k++) {
                    const float m = T::ordered_pick(sv[k], e[k]);
                    so[k] = __float_as_uint(m) != __float_as_uint(sv[k]) ? rel : so[k];
                    sv[k] = m;
                }
            }
#pragma unroll
            for (int k = 0; k < VE; k++) acc[k] = T::from_ordered(sv[k], r0 + so[k]);
        }
    } else if (has) {
        int64_t r = r0 + ty;
        // sums and products take the rows of a step as a tree (an fp64 sum
        // four: a shorter chain for the same additions)
        if constexpr (COOP && HasPad<T>::value && !T::kIdx) {
            constexpr int R = sizeof(E) == 8 ? 4 : U;
            for (; r + (int64_t)(R - 1) * ry < r1; r += (int64_t)R * ry) {
                E e[R][VE];
#pragma unroll
                for (int u = 0; u < R; u++) axis_load<VB, Ld>(x, slab + (r + (int64_t)u * ry) * a.inner, e[u]);
#pragma unroll
                for (int k = 0; k < VE; k++) {
                    E t[R];
#pragma unroll
                    for (int u = 0; u < R; u++) t[u] = e[u][k];
                    T::add_vec(acc[k], t, r);
                }
            }
        }
        for (; r + (int64_t)(U - 1) * ry < r1; r += (int64_t)U * ry) {
            E e[U][VE];
#pragma unroll
            for (int u = 0; u < U; u++) axis_load<VB, Ld>(x, slab + (r + (int64_t)u * ry) * a.inner, e[u]);
#pragma unroll
            for (int u = 0; u < U; u++)
#pragma unroll
                for (int k = 0; k < VE; k++) add_in_order<T>(acc[k], e[u][k], r + (int64_t)u * ry);
        }
        for (; r < r1; r += ry) {
            E e[VE];
            axis_load<VB, Ld>(x, slab + r * a.inner, e);
#pragma unroll
            for (int k = 0; k < VE; k++) add_in_order<T>(acc[k], e[k], r);
        }
    }
    const bool f64 = a.out_f64 != 0;
    auto result = [&](int k, const Part& q) {
        if (ty != 0 || !has) return;
        const int64_t o = p * a.inner + col * VE + k;
        const G g = GR::up(q);
        if (a.splits == 1) {
            GR::store(a.out, o, g, f64);
            GR::store_aux(a.argidx, a.aux, o, g, 0);
        } else {
            const int64_t nout = a.outer * a.inner;
            reinterpret_cast<G*>(a.scratch)[a.splits <= kAxisThreadFinish ? s * nout + o : o * a.splits + s] = g;
        }
    };
    // a warp's column elements combine across its rows' lanes; then (COOP),
    // KP elements at a time, across the block's warps as a tree, each element
    // by one of the warps
    if constexpr (COOP) {
        constexpr int KP = AxisPhase<T, VE>::value;
        using CP = ColPart<T>;
        using P = typename CP::P;
        __shared__ P s_part[KP][kAxisCoop][32];
        const int warp = threadIdx.x >> 5;
#pragma unroll
        for (int k = 0; k < VE; k++) {
            P q = CP::from(acc[k]);
            for (int m = 16; m >= bx; m >>= 1) q = CP::combine(q, shfl_xor_any(q, m));
            s_part[k % KP][warp][lane] = q;
            if (k % KP == KP - 1) {
                __syncthreads();
                for (int j = warp; j < KP; j += a.coop) {
                    // as a tree: coop is a power of two of at most eight
                    auto pair = [&](int w) { return CP::combine(s_part[j][w][lane], s_part[j][w + 1][lane]); };
                    auto quad = [&](int w) { return CP::combine(pair(w), pair(w + 2)); };
                    q = a.coop == 8 ? CP::combine(quad(0), quad(4))
                                    : (a.coop == 4 ? quad(0) : (a.coop == 2 ? pair(0) : s_part[j][0][lane]));
                    result(k - (KP - 1) + j, CP::part(q));
                }
                if (k < VE - 1) __syncthreads();   // before the slots are written again
            }
        }
    } else {
#pragma unroll
        for (int k = 0; k < VE; k++) {
            Part q = T::to_part(acc[k]);
            for (int m = 16; m >= bx; m >>= 1) q = T::combine(q, shfl_xor_any(q, m));
            result(k, q);
        }
    }
}

// Few splits: one thread per output folds its splits in order, as trees of eight.  Many: one
// warp per output, the lanes taking the splits in order (lane, lane + 32, ...)
// and combining by a fixed butterfly.
template <class T>
__global__ void __launch_bounds__(256) k_axis_finish(AxisArgs a) {
    using GR = GridR<T>;
    using G = typename GR::Part;
    asm volatile("griddepcontrol.wait;" ::: "memory");   // launched as k_axis' programmatic dependent
    const int64_t nout = a.outer * a.inner;
    const G* part = reinterpret_cast<const G*>(a.scratch);
    if (a.splits <= kAxisThreadFinish) {
        const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
        if (o >= nout) return;
        auto at = [&](int64_t s) { return s < a.splits ? part[s * nout + o] : GR::part_init(); };
        auto pair = [&](int64_t s) { return GR::combine(at(s), at(s + 1)); };
        auto quad = [&](int64_t s) { return GR::combine(pair(s), pair(s + 2)); };
        auto eight = [&](int64_t s) { return s + 4 < a.splits ? GR::combine(quad(s), quad(s + 4)) : quad(s); };
        G q = eight(0);
        for (int64_t s = 8; s < a.splits; s += 8) q = GR::combine(q, eight(s));
        GR::store(a.out, o, q, a.out_f64 != 0);
        GR::store_aux(a.argidx, a.aux, o, q, 0);
        return;
    }
    const int lane = threadIdx.x & 31;
    const int64_t o = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (o >= nout) return;
    const G* src = part + o * a.splits;
    G q = GR::part_init();
    for (int64_t s = lane; s < a.splits; s += 32) q = GR::combine(q, src[s]);
    q = GR::warp_reduce(q);
    if (lane == 0) {
        GR::store(a.out, o, q, a.out_f64 != 0);
        GR::store_aux(a.argidx, a.aux, o, q, 0);
    }
}

// Empty axis (n == 0): every output is the identity.
template <class T>
__global__ void __launch_bounds__(256) k_axis_empty(AxisArgs a) {
    const int64_t nout = a.outer * a.inner;
    for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < nout; o += (int64_t)gridDim.x * blockDim.x)
        T::store_empty(a.out, o, a.out_f64 != 0, a.argidx, a.aux);
}

// One vector store of VB bytes.
template <class F, int VB>
__device__ __forceinline__ void st_vec(F* p, const F (&v)[VB / sizeof(F)]);

template <>
__device__ __forceinline__ void st_vec<float, 16>(float* p, const float (&v)[4]) {
    asm volatile("st.global.v4.f32 [%0], {%1,%2,%3,%4};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
template <>
__device__ __forceinline__ void st_vec<float, 32>(float* p, const float (&v)[8]) {
    asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
                 "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7]) : "memory");
}
template <>
__device__ __forceinline__ void st_vec<double, 16>(double* p, const double (&v)[2]) {
    asm volatile("st.global.v2.f64 [%0], {%1,%2};" ::"l"(p), "d"(v[0]), "d"(v[1]) : "memory");
}
template <>
__device__ __forceinline__ void st_vec<double, 32>(double* p, const double (&v)[4]) {
    asm volatile("st.global.v4.f64 [%0], {%1,%2,%3,%4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3]) : "memory");
}

struct AxisBwdArgs {
    const void* x;            // PROD only
    const void* g;            // grad_out [outer, inner]
    const int64_t* argidx;    // MAX / MIN: [outer, inner]
    const pr_prod_aux* aux;   // PROD: [outer, inner]
    void* gi;                 // grad_in [outer, n, inner]
    int64_t outer, n, inner;
    int64_t qv;               // vectors per row: inner / VE
    int op;
};

// grad_in viewed as rows (p, i) of qv vectors; a thread walks the flattened
// vectors with a grid stride, advancing (p, i, column) by carries instead of
// dividing per vector.  OPK: 0 sum (broadcast), 1 max/min (one-hot at argidx),
// 2 prod (zero-count aware).  With VB > 0, grad_out (and argidx) are read as
// vectors of the same columns.
template <class F, int VB, int OPK>
__global__ void __launch_bounds__(256) k_axis_backward(AxisBwdArgs a) {
    constexpr int VE = VB ? VB / (int)sizeof(F) : 1;
    const F* g = static_cast<const F*>(a.g);
    const F* x = static_cast<const F*>(a.x);
    F* gi = static_cast<F*>(a.gi);
    const int64_t total = a.outer * a.n * a.qv;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= total) return;
    int64_t R = v / a.qv, cq = v - R * a.qv;
    int64_t p = R / a.n, i = R - p * a.n;
    const int64_t dR = stride / a.qv, dq = stride - dR * a.qv;
    const int64_t dp = dR / a.n, di = dR - dp * a.n;
    for (; v < total; v += stride) {
        const int64_t o0 = p * a.inner + cq * VE;        // first output of this vector's columns
        const int64_t e0 = (p * a.n + i) * a.inner + cq * VE;
        F gv[VE];
        if constexpr (VB == 0) {
            gv[0] = g[o0];
        } else {
            const Words<VB> w = ldv<VB>(g + o0);
            memcpy(gv, w.w, VB);
        }
        F vals[VE];
        if constexpr (OPK == 0) {
#pragma unroll
            for (int k = 0; k < VE; k++) vals[k] = gv[k];
        } else if constexpr (OPK == 1) {
#pragma unroll
            for (int k = 0; k < VE; k++) vals[k] = __ldg(a.argidx + o0 + k) == i ? gv[k] : (F)0;
        } else {
#pragma unroll
            for (int k = 0; k < VE; k++) {
                const pr_prod_aux ax = a.aux[o0 + k];
                const F gp = (F)((double)gv[k] * ax.p_nz);
                vals[k] = ax.zero_count == 0 ? gp / x[e0 + k]
                          : (ax.zero_count == 1 && ax.first_zero == i ? gp : (F)0);
            }
        }
        if constexpr (VB == 0) {
            gi[e0] = vals[0];
        } else {
            st_vec<F, VB>(gi + e0, vals);
        }
        // advance by the stride: columns, then rows, then slabs
        cq += dq;
        const int64_t c1 = cq >= a.qv ? 1 : 0;
        cq -= c1 * a.qv;
        i += di + c1;
        const int64_t c2 = i >= a.n ? 1 : 0;
        i -= c2 * a.n;
        p += dp + c2;
    }
}

// The same gradient with each column's grad_out and state held in registers:
// a warp takes a group of column vectors of one slab (lanes as in k_axis: bx
// per row, 32 / bx rows a step) and writes every `splits`-th step of its rows,
// so that the warps of a slab write one moving window of neighbouring rows.
// k_axis_backward re-reads them for every row, 96 bytes per 32 written for
// the extrema; it keeps inputs too small for two steps a warp, and rows that
// leave lanes without a column.  Bound by the write: fp32 maximum of [64, 577,
// 768] 62 -> 20.7 us (0.80 of a 6.8 TB/s copy), of [16, 4096, 4096] 528 -> 146
// (1.08), its sum 156 -> 147, product of [64, 577, 768] 170 -> 57 (0.58, with
// x read; the divisions).
template <class F, int VB, int OPK>
__global__ void __launch_bounds__(256) k_axis_backward_cols(AxisBwdArgs a, int bx, int64_t groups, int64_t splits,
                                                            int xvec) {
    constexpr int VE = VB ? VB / (int)sizeof(F) : 1;
    const int lane = threadIdx.x & 31, ry = 32 / bx;
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t tile = wid / splits, s = wid - tile * splits;
    const int64_t p = tile / groups, col = (tile - p * groups) * bx + (lane & (bx - 1));
    if (p >= a.outer || col >= a.qv) return;
    const int64_t o0 = p * a.inner + col * VE;
    const F* x = static_cast<const F*>(a.x);
    F* gi = static_cast<F*>(a.gi);
    int64_t i = s * ry + lane / bx;
    // the product's factors of row r, loaded a row ahead of their use
    F xe[VE];
    auto load_x = [&](int64_t r) {
        if (OPK != 2 || r >= a.n) return;
        const int64_t e0 = (p * a.n + r) * a.inner + col * VE;
        if constexpr (VB != 0) {
            if (xvec) {
                const Words<VB> w = ldv<VB>(x + e0);
                memcpy(xe, w.w, VB);
                return;
            }
        }
#pragma unroll
        for (int k = 0; k < VE; k++) xe[k] = __ldg(x + e0 + k);
    };
    load_x(i);
    F gv[VE];
    int64_t hot[VE];      // the row that gets gv, -1: none, -2: every row, -3: every row, divided by x
    if constexpr (VB == 0) {
        gv[0] = __ldg(static_cast<const F*>(a.g) + o0);
    } else {
        const Words<VB> w = ldv<VB>(static_cast<const F*>(a.g) + o0);
        memcpy(gv, w.w, VB);
    }
#pragma unroll
    for (int k = 0; k < VE; k++) {
        hot[k] = -2;
        if constexpr (OPK == 1) {
            hot[k] = __ldg(a.argidx + o0 + k);
        } else if constexpr (OPK == 2) {
            const pr_prod_aux ax = a.aux[o0 + k];
            gv[k] = (F)((double)gv[k] * ax.p_nz);
            hot[k] = ax.zero_count == 0 ? -3 : (ax.zero_count == 1 ? ax.first_zero : -1);
        }
    }
    for (; i < a.n; i += splits * ry) {
        const int64_t e0 = (p * a.n + i) * a.inner + col * VE;
        F vals[VE];
        if constexpr (OPK == 2) {
            F xc[VE];
#pragma unroll
            for (int k = 0; k < VE; k++) xc[k] = xe[k];
            load_x(i + splits * ry);
#pragma unroll
            for (int k = 0; k < VE; k++) vals[k] = hot[k] == -3 ? gv[k] / xc[k] : (hot[k] == i ? gv[k] : (F)0);
        } else {
#pragma unroll
            for (int k = 0; k < VE; k++) vals[k] = OPK == 0 || hot[k] == i ? gv[k] : (F)0;
        }
        if constexpr (VB == 0) gi[e0] = vals[0];
        else st_vec<F, VB>(gi + e0, vals);
    }
}

}  // namespace pr
