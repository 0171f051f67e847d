// Host-side table of compiled kernel variants.  Every instantiation unit
// registers, per (kind, dtype, combiner, precision, aux output), one entry per
// (unroll, vector width); the API picks the entry named by the launch
// configuration.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

namespace pr {

struct ReduceArgs;
struct SegArgs;
struct RowArgs;
struct RowGroupArgs;
struct SegGroupArgs;
struct AxisArgs;
struct AxisBwdArgs;
struct ScanArgs;
struct BwdArgs;

enum Kind : uint8_t {
    K_REDUCE = 0, K_SEGMENTED = 1, K_BACKWARD = 2, K_COMBINE = 3, K_ROWS = 4,
    K_AXIS = 5, K_AXIS_FINISH = 6, K_AXIS_EMPTY = 7, K_AXIS_BACKWARD = 8, K_SCAN = 9,
    K_REDUCE_TAIL = 10, // k_reduce with claimed tail tiles (large inputs)
    K_ROWS_GROUP = 11,  // a group of lanes per row (short rows, any alignment)
    K_SEG_GROUP = 12,   // many segments: the short ones,
    K_SEG_LONG = 13,    // and the long ones
    K_AXIS_COOP = 14    // k_axis whose blocks' warps share a split
};
enum Aux : uint8_t { AUX_NONE = 0, AUX_ARG = 1, AUX_PROD = 2 };

struct KernelKey {
    uint8_t kind, dtype, op, prec, aux, unroll, vb;
};

using ReduceLaunch = cudaError_t (*)(const ReduceArgs&, int grid, int block, cudaStream_t);
using SegLaunch = cudaError_t (*)(const SegArgs&, int grid, int block, cudaStream_t);
using RowLaunch = cudaError_t (*)(const RowArgs&, int grid, int block, cudaStream_t);
using SegGroupLaunch = cudaError_t (*)(const SegGroupArgs&, int grid, int block, cudaStream_t);
using RowGroupLaunch = cudaError_t (*)(const RowGroupArgs&, int grid, int block, cudaStream_t);
using AxisLaunch = cudaError_t (*)(const AxisArgs&, int grid, int block, cudaStream_t);
using AxisBwdLaunch = cudaError_t (*)(const AxisBwdArgs&, int grid, int block, cudaStream_t);
using ScanLaunch = cudaError_t (*)(const ScanArgs&, int grid, int block, size_t smem, cudaStream_t);
using BwdLaunch = cudaError_t (*)(const BwdArgs&, int grid, int block, cudaStream_t);
using CombineLaunch = cudaError_t (*)(const char* parts, int count, void* out, int out_f64, cudaStream_t);

struct KernelEntry {
    const void* fn;      // the __global__ function (occupancy queries)
    void* launch;        // one of the *Launch types above, by kind
    int part_bytes = 0;  // K_AXIS, K_AXIS_COOP, K_SEG_GROUP: bytes of one partial
    int tile_slots = 0;  // K_REDUCE_TAIL: claimed tiles a block holds partials for
    int tile_loads = 0;  // K_REDUCE_TAIL: vectors a thread loads per round of a tile
};

void reg_add(const KernelKey& k, const KernelEntry& e);
const KernelEntry* reg_find(const KernelKey& k);

// Unroll factors and vector widths compiled for every family.
constexpr int kUnrolls[] = {2, 4};
constexpr int kVecBytes[] = {16, 32};

// Flat gradient of a row reduction (backward.cu); a.shift counts from the previous 32-byte boundary.
cudaError_t launch_backward_flat(const BwdArgs& a, bool f64, cudaStream_t st);
// Axis gradient by columns (backward.cu).
cudaError_t launch_axis_backward_cols(const AxisBwdArgs& a, bool f64, int vb, int bx, int64_t groups, int64_t splits,
                                      cudaStream_t st);

void register_f32();
void register_f32_seg();
void register_f16();
void register_bf16();
void register_f64();
void register_i32();
void register_u32();
void register_i64();
void register_backward();
void register_scan();

// Registers every family above exactly once (thread-safe).
void ensure_registered();

}  // namespace pr
