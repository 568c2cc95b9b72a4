// FP64 fused step (2D and 3D).  Built with --fmad=false so that its rounding
// follows the plain multiply-then-add order.  Also holds the variant table.
#include "dispatch.h"

namespace tlbm {

cudaError_t launch_step_f64(int dim, int vec, bool trt, int rows, const void* src, void* dst, const KParams& p, dim3 grid,
                            dim3 block, cudaStream_t s) {
    if (dim == 2) {
        TLBM_STEP_CASE(2, double, 2, true)
        TLBM_STEP_CASE(2, double, 1, true)
        TLBM_STEP_CASE(2, double, 2, false)
        TLBM_AA_CASE(2, double, 2, true)
        TLBM_AA_CASE(2, double, 2, false)
    } else {
        TLBM_STEP_CASE(3, double, 1, true)
        TLBM_STEP_CASE(3, double, 2, true)
        TLBM_STEP_CASE(3, double, 1, false)
        TLBM_AA_CASE(3, double, 1, true)
        TLBM_AA_CASE(3, double, 1, false)
    }
    return cudaErrorInvalidValue;
}

const void* func_step_f64(int dim, int vec, bool trt, int rows) {
    if (dim == 2) {
        TLBM_STEP_FUNC(2, double, 2, true)
        TLBM_STEP_FUNC(2, double, 1, true)
        TLBM_STEP_FUNC(2, double, 2, false)
        TLBM_AA_FUNC(2, double, 2, true)
        TLBM_AA_FUNC(2, double, 2, false)
    } else {
        TLBM_STEP_FUNC(3, double, 1, true)
        TLBM_STEP_FUNC(3, double, 2, true)
        TLBM_STEP_FUNC(3, double, 1, false)
        TLBM_AA_FUNC(3, double, 1, true)
        TLBM_AA_FUNC(3, double, 1, false)
    }
    return nullptr;
}

// One thread per node, nodes in their order in memory.  The FP64 pipe spends as
// much on an idle lane as on a busy one, and warps that end with their row idle
// on its rest: 14 % of the lanes at 193 nodes,
// 20 % at 129.  us per step, warps inside rows -> this kernel: 193^3 3415 -> 2904,
// 129^3 1097 -> 877, 65^3 174 -> 125; 129^2 13.3 -> 8.1, 513^2 76 -> 63, 2049^2
// 944 -> 925, 4097^2 3682 -> 3681; in place the same.  (With the wall rules face by
// face and nine blocks per SM in 2D: 129^2 7.0, 513^2 61.5, 2049^2 909, 4097^2 3621.)
template <int DIM>
static cudaError_t launch_flat_f64(int mode, const void* src, void* dst, const KParams& p, cudaStream_t s) {
    if (mode == PULL) return launch_flat_as<DIM, double, PULL>(src, dst, p, s);
    if (mode == AA_EVEN) return launch_flat_as<DIM, double, AA_EVEN>(src, dst, p, s);
    return launch_flat_as<DIM, double, AA_ODD>(src, dst, p, s);
}

cudaError_t launch_flat(int dim, int prec, int mode, const void* src, void* dst, const KParams& p, cudaStream_t s) {
    if (prec == 0) return dim == 2 ? launch_flat_f64<2>(mode, src, dst, p, s) : launch_flat_f64<3>(mode, src, dst, p, s);
    return launch_flat_3d_f16(prec, mode, src, dst, p, s);
}

const void* step_function(int dim, int prec, int vec, bool trt, int rows) {
    if (prec == 0) return func_step_f64(dim, vec, trt, rows);
    if (dim == 2) return prec == 1 ? func_step_2d_f32(vec, trt, rows) : func_step_2d_f16(prec, vec, trt, rows);
    return prec == 1 ? func_step_3d_f32(vec, trt, rows) : func_step_3d_f16(prec, vec, trt, rows);
}

bool step_variant_available(int dim, int prec, int vec, bool trt, int rows) {
    return step_function(dim, prec, vec, trt, rows) != nullptr;
}

cudaError_t launch_step(int dim, int prec, int vec, bool trt, int rows, const void* src, void* dst,
                        const KParams& p, dim3 grid, dim3 block, cudaStream_t s) {
    if (!step_variant_available(dim, prec, vec, trt, rows)) return cudaErrorInvalidValue;
    if (prec == 0) return launch_step_f64(dim, vec, trt, rows, src, dst, p, grid, block, s);
    if (dim == 2) {
        if (prec == 1) return launch_step_2d_f32(vec, trt, rows, src, dst, p, grid, block, s);
        return launch_step_2d_f16(prec, vec, trt, rows, src, dst, p, grid, block, s);
    }
    if (prec == 1) return launch_step_3d_f32(vec, trt, rows, src, dst, p, grid, block, s);
    return launch_step_3d_f16(prec, vec, trt, rows, src, dst, p, grid, block, s);
}

}  // namespace tlbm
