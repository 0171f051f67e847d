// Backward kernels of a row reduction y[r] = (x) over x[r, 0..cols):
//   SUM      dy/dx[r,c] = 1
//   MAX/MIN  1 at the first arg-extremum, 0 elsewhere
//   PROD     prod_{j != c} x[r,j]: with no zero in the row P_nz / x[r,c];
//            with one zero, P_nz at the zero and 0 elsewhere; with two or
//            more zeros, 0 everywhere (P_nz = product of the non-zero elements)
// times grad_out[r].  The work is one streaming write of grad_in (plus a read
// of x for product rows without zeros): rows are cut into chunks of
// blockDim*U vectors, each thread writes U vectors of VB bytes.  The grid is
// several times what is resident and chunk t goes to block t mod grid, so the
// blocks in flight always write one window of neighbouring chunks and the
// hardware hands the remaining blocks to whichever SMs finish first (no tail of
// SMs still writing fixed shares).  Row-uniform values (grad_out, argidx, aux)
// are re-read only when a block's row changes.  Rows of at most 32768 elements
// take the flat form, k_backward_flat.
#include "registry.h"
#include "kernels.cuh"
#include "axis.cuh"

namespace pr {

constexpr int kFlatBlock = 256;

// Row-uniform description of the gradient: value gv at column `hot` (or at
// every column when hot == -2), 0 elsewhere; div: gv / x[c] at every column.
template <class F>
struct RowGrad {
    F gv;
    int64_t hot;
    bool div;
};

template <class F>
__device__ __forceinline__ RowGrad<F> row_grad(const BwdArgs& a, int64_t r) {
    const F g = static_cast<const F*>(a.g)[r];
    RowGrad<F> rg{g, -2, false};
    if (a.op == PR_MAX || a.op == PR_MIN) {
        rg.hot = a.argidx[r];
        if (rg.hot < 0) rg.hot = -1;
    } else if (a.op == PR_PROD) {
        const pr_prod_aux ax = a.aux[r];
        const F gp = (F)((double)g * ax.p_nz);
        if (ax.zero_count == 0) { rg.gv = gp; rg.div = true; }
        else if (ax.zero_count == 1) { rg.gv = gp; rg.hot = ax.first_zero; }
        else { rg.gv = (F)0; rg.hot = -1; }
    }
    return rg;
}

template <class F>
__device__ __forceinline__ F elem_grad(const RowGrad<F>& rg, const F* xrow, int64_t c) {
    if (rg.div) return rg.gv / xrow[c];
    if (rg.hot == -2) return rg.gv;
    return c == rg.hot ? rg.gv : (F)0;
}

template <class F, int U, int VB>
__global__ void __launch_bounds__(1024) k_backward(BwdArgs a) {
    constexpr int VE = VB / sizeof(F);
    F* gi = static_cast<F*>(a.gi);
    const F* x = static_cast<const F*>(a.x);
    const int64_t ntiles = a.rows * a.chunks_per_row;
    const int64_t CV = (int64_t)blockDim.x * U;  // vectors per chunk
    int64_t rc = -1;
    RowGrad<F> rg{};
    for (int64_t t = blockIdx.x; t < ntiles; t += gridDim.x) {
        const int64_t r = t / a.chunks_per_row, c = t - r * a.chunks_per_row;
        if (r != rc) {
            rg = row_grad<F>(a, r);
            rc = r;
        }
        const int64_t base = r * a.cols;
        const int64_t mis = (base + a.shift) % VE;
        int64_t head = (VE - mis) % VE;
        head = head < a.cols ? head : a.cols;
        const int64_t nvec = (a.cols - head) / VE;
        F* grow = gi + base;
        const F* xrow = x ? x + base : nullptr;
#pragma unroll
        for (int u = 0; u < U; u++) {
            const int64_t v = c * CV + (int64_t)u * blockDim.x + threadIdx.x;
            if (v < nvec) {
                const int64_t c0 = head + v * VE;
                F vals[VE];
                // row-uniform branches: the broadcast and one-hot rows cost no
                // per-element arithmetic beyond one compare
                if (rg.div) {
#pragma unroll
                    for (int k = 0; k < VE; k++) vals[k] = rg.gv / xrow[c0 + k];
                } else if (rg.hot == -2) {
#pragma unroll
                    for (int k = 0; k < VE; k++) vals[k] = rg.gv;
                } else {
                    const int64_t h = rg.hot - c0;
                    const int hk = (h >= 0 && h < VE) ? (int)h : -1;
#pragma unroll
                    for (int k = 0; k < VE; k++) vals[k] = hk == k ? rg.gv : (F)0;
                }
                st_vec<F, VB>(grow + c0, vals);
            }
        }
        if (c == 0) {
            // unaligned head and the tail after the last full vector
            const int64_t tail0 = head + nvec * VE;
            const int64_t nscalar = head + (a.cols - tail0);
            for (int64_t j = threadIdx.x; j < nscalar; j += blockDim.x) {
                const int64_t col = j < head ? j : tail0 + (j - head);
                grow[col] = elem_grad(rg, xrow, col);
            }
        }
    }
}

// Flat form: gi as one array of vectors whatever the rows, for rows too short
// to fill a chunk of k_backward (which gives a block of 512 threads to every
// row, however short).  A block takes kFlatU vectors a thread of neighbouring
// memory; one 64-bit division places the block's first element, a 32-bit
// multiply-high each vector's (row_inv: floor((2^32 - 1) / cols), whose
// estimate is at most one short).  A vector that lies in one row takes that
// row's gradient as k_backward does; one that crosses row ends is filled
// element by element.  OPK: 0 sum, 1 max/min, 2 prod.
constexpr int kFlatU = 4;
constexpr int kFlatVec = 32;

template <class F, int OPK>
__device__ __forceinline__ RowGrad<F> flat_row(const BwdArgs& a, int64_t r) {
    const F g = __ldg(static_cast<const F*>(a.g) + r);
    RowGrad<F> rg{g, -2, false};
    if constexpr (OPK == 1) {
        rg.hot = __ldg(a.argidx + r);
        if (rg.hot < 0) rg.hot = -1;
    } else if constexpr (OPK == 2) {
        const pr_prod_aux ax = a.aux[r];
        rg.gv = ax.zero_count >= 2 ? (F)0 : (F)((double)g * ax.p_nz);
        rg.div = ax.zero_count == 0;
        rg.hot = ax.zero_count == 1 ? ax.first_zero : -1;
    }
    return rg;
}

template <class F, int OPK>
__global__ void __launch_bounds__(kFlatBlock) k_backward_flat(BwdArgs a, unsigned row_inv, int xvec) {
    constexpr int VE = kFlatVec / (int)sizeof(F);
    F* gi = static_cast<F*>(a.gi);
    const F* x = static_cast<const F*>(a.x);
    const int64_t total = a.rows * a.cols;
    const int cols = (int)a.cols;
    const int64_t b0 = (int64_t)blockIdx.x * (kFlatBlock * kFlatU * VE) - a.shift;   // block's first element
    const int64_t R0 = b0 > 0 ? b0 / a.cols : 0;
    const int C0 = (int)(b0 - R0 * a.cols);            // its column (negative before gi's first element)
#pragma unroll
    for (int u = 0; u < kFlatU; u++) {
        const int off = (u * kFlatBlock + (int)threadIdx.x) * VE;
        const int64_t e0 = b0 + off;
        if (e0 >= total) break;
        const int ce = C0 + off;
        int q = ce > 0 ? (int)__umulhi((unsigned)ce, row_inv) : 0;
        if (ce - q * cols >= cols) q++;
        int64_t r = R0 + q;
        int c = ce - q * cols;
        F vals[VE];
        if (c >= 0 && c + VE <= cols) {
            const RowGrad<F> rg = flat_row<F, OPK>(a, r);
            if constexpr (OPK == 0) {
#pragma unroll
                for (int k = 0; k < VE; k++) vals[k] = rg.gv;
            } else {
                if (OPK == 2 && rg.div) {
                    F xe[VE];
                    if (xvec) {
                        const Words<kFlatVec> w = ldv<kFlatVec>(x + e0);
                        memcpy(xe, w.w, kFlatVec);
                    } else {
#pragma unroll
                        for (int k = 0; k < VE; k++) xe[k] = __ldg(x + e0 + k);
                    }
#pragma unroll
                    for (int k = 0; k < VE; k++) vals[k] = rg.gv / xe[k];
                } else {
                    const int64_t h = rg.hot - c;
                    const int hk = (h >= 0 && h < VE) ? (int)h : -1;
#pragma unroll
                    for (int k = 0; k < VE; k++) vals[k] = hk == k ? rg.gv : (F)0;
                }
            }
            st_vec<F, kFlatVec>(gi + e0, vals);
            continue;
        }
        RowGrad<F> rg{};
        bool have = false;
#pragma unroll
        for (int k = 0; k < VE; k++) {
            vals[k] = (F)0;
            if (c == cols) {
                c = 0;
                r++;
                have = false;
            }
            if (c >= 0 && r < a.rows) {
                if (!have) rg = flat_row<F, OPK>(a, r);
                have = true;
                vals[k] = OPK == 0 ? rg.gv : (rg.div ? rg.gv / __ldg(x + e0 + k) : (rg.hot == c ? rg.gv : (F)0));
            }
            c++;
        }
        if (e0 >= 0 && e0 + VE <= total) {
            st_vec<F, kFlatVec>(gi + e0, vals);
        } else {
#pragma unroll
            for (int k = 0; k < VE; k++)
                if (e0 + k >= 0 && e0 + k < total) gi[e0 + k] = vals[k];
        }
    }
}

template <class F, int OPK>
static void flat_go(const BwdArgs& a, int64_t grid, bool xvec, cudaStream_t st) {
    k_backward_flat<F, OPK><<<(unsigned)grid, kFlatBlock, 0, st>>>(a, 0xffffffffu / (unsigned)a.cols, xvec ? 1 : 0);
}

// shift in a is gi's element offset from the previous 32-byte boundary
template <class F>
static cudaError_t launch_flat(const BwdArgs& a, cudaStream_t st) {
    constexpr int64_t VE = kFlatVec / (int)sizeof(F);
    const int64_t per = kFlatBlock * kFlatU * VE;
    const int64_t grid = (a.rows * a.cols + a.shift + per - 1) / per;
    if (grid > 0x7fffffff) return cudaErrorInvalidConfiguration;
    const bool xvec = ((uintptr_t)a.x - (uintptr_t)a.gi) % kFlatVec == 0;
    if (a.op == PR_SUM) flat_go<F, 0>(a, grid, xvec, st);
    else if (a.op == PR_PROD) flat_go<F, 2>(a, grid, xvec, st);
    else flat_go<F, 1>(a, grid, xvec, st);
    return cudaGetLastError();
}

cudaError_t launch_backward_flat(const BwdArgs& a, bool f64, cudaStream_t st) {
    return f64 ? launch_flat<double>(a, st) : launch_flat<float>(a, st);
}

template <class F, int U, int VB>
cudaError_t launch_backward(const BwdArgs& a, int grid, int block, cudaStream_t st) {
    k_backward<F, U, VB><<<grid, block, 0, st>>>(a);
    return cudaGetLastError();
}

template <class F, int U, int VB>
static void reg_bwd(uint8_t dtype) {
    reg_add(KernelKey{K_BACKWARD, dtype, 0, 0, 0, (uint8_t)U, (uint8_t)VB},
            KernelEntry{reinterpret_cast<const void*>(&k_backward<F, U, VB>),
                        reinterpret_cast<void*>(&launch_backward<F, U, VB>)});
}

template <class F, int VB, int OPK>
cudaError_t launch_axis_backward(const AxisBwdArgs& a, int grid, int block, cudaStream_t st) {
    k_axis_backward<F, VB, OPK><<<grid, block, 0, st>>>(a);
    return cudaGetLastError();
}

// Column form (k_axis_backward_cols): lanes per row, column groups and row
// splits as in its comment.
template <class F, int VB>
static void axis_cols_go(const AxisBwdArgs& a, int bx, int64_t groups, int64_t splits, cudaStream_t st) {
    const int64_t grid = (a.outer * groups * splits + 7) / 8;
    const int xvec = VB && a.op == PR_PROD && reinterpret_cast<uintptr_t>(a.x) % VB == 0 ? 1 : 0;
    const unsigned g = (unsigned)grid;
    if (a.op == PR_SUM) k_axis_backward_cols<F, VB, 0><<<g, 256, 0, st>>>(a, bx, groups, splits, xvec);
    else if (a.op == PR_PROD) k_axis_backward_cols<F, VB, 2><<<g, 256, 0, st>>>(a, bx, groups, splits, xvec);
    else k_axis_backward_cols<F, VB, 1><<<g, 256, 0, st>>>(a, bx, groups, splits, xvec);
}

cudaError_t launch_axis_backward_cols(const AxisBwdArgs& a, bool f64, int vb, int bx, int64_t groups, int64_t splits,
                                      cudaStream_t st) {
    if (f64) {
        if (vb == 32) axis_cols_go<double, 32>(a, bx, groups, splits, st);
        else if (vb == 16) axis_cols_go<double, 16>(a, bx, groups, splits, st);
        else axis_cols_go<double, 0>(a, bx, groups, splits, st);
    } else {
        if (vb == 32) axis_cols_go<float, 32>(a, bx, groups, splits, st);
        else if (vb == 16) axis_cols_go<float, 16>(a, bx, groups, splits, st);
        else axis_cols_go<float, 0>(a, bx, groups, splits, st);
    }
    return cudaGetLastError();
}

// Keyed by (dtype, op kind in the op field: 0 sum, 1 max/min, 2 prod, vector width).
template <class F, int VB>
static void reg_axis_bwd(uint8_t dtype) {
    reg_add(KernelKey{K_AXIS_BACKWARD, dtype, 0, 0, 0, 0, (uint8_t)VB},
            KernelEntry{reinterpret_cast<const void*>(&k_axis_backward<F, VB, 0>),
                        reinterpret_cast<void*>(&launch_axis_backward<F, VB, 0>)});
    reg_add(KernelKey{K_AXIS_BACKWARD, dtype, 1, 0, 0, 0, (uint8_t)VB},
            KernelEntry{reinterpret_cast<const void*>(&k_axis_backward<F, VB, 1>),
                        reinterpret_cast<void*>(&launch_axis_backward<F, VB, 1>)});
    reg_add(KernelKey{K_AXIS_BACKWARD, dtype, 2, 0, 0, 0, (uint8_t)VB},
            KernelEntry{reinterpret_cast<const void*>(&k_axis_backward<F, VB, 2>),
                        reinterpret_cast<void*>(&launch_axis_backward<F, VB, 2>)});
}

void register_backward() {
    reg_axis_bwd<float, 0>(PR_F32);
    reg_axis_bwd<float, 16>(PR_F32);
    reg_axis_bwd<float, 32>(PR_F32);
    reg_axis_bwd<double, 0>(PR_F64);
    reg_axis_bwd<double, 16>(PR_F64);
    reg_axis_bwd<double, 32>(PR_F64);
    reg_bwd<float, 2, 16>(PR_F32);
    reg_bwd<float, 2, 32>(PR_F32);
    reg_bwd<float, 4, 16>(PR_F32);
    reg_bwd<float, 4, 32>(PR_F32);
    reg_bwd<double, 2, 16>(PR_F64);
    reg_bwd<double, 2, 32>(PR_F64);
    reg_bwd<double, 4, 16>(PR_F64);
    reg_bwd<double, 4, 32>(PR_F64);
}

}  // namespace pr
