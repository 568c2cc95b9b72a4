// Host-side launch entry points of the step kernels.  Each translation unit
// instantiates the variants of one (dimension, storage) family; the FP64 unit
// is built without FMA contraction.
#pragma once
#include <cuda_runtime.h>

#include "kernels.cuh"
#include "staged.cuh"

namespace tlbm {

// prec: 0 FP64, 1 FP32, 2 FP16-offset, 3 BF16-offset (enum tlbm_prec).
// vec: nodes per thread.  trt: two-relaxation-time form of the collision.
// Returns cudaErrorInvalidValue if the variant is not compiled.
// rows: consecutive rows per thread (1, or 2 / 4 for the software-pipelined kernel);
// -AA_EVEN / -AA_ODD select the two halves of an in-place step pair, which read
// and write `dst` only.
cudaError_t launch_step(int dim, int prec, int vec, bool trt, int rows, const void* src, void* dst,
                        const KParams& p, dim3 grid, dim3 block, cudaStream_t s);
bool step_variant_available(int dim, int prec, int vec, bool trt, int rows);
// device function of a compiled variant (for cudaFuncGetAttributes), or nullptr
const void* step_function(int dim, int prec, int vec, bool trt, int rows);

// step with one thread per node in memory order, TRT form: FP64, and the halves of
// a 16-bit 3D in-place pair (mode: PULL, or a half of an in-place pair, which reads
// and writes dst).  Cells of up to FLAT_NODES nodes (32-bit thread numbers).
constexpr double FLAT_NODES = 4e9;
cudaError_t launch_flat(int dim, int prec, int mode, const void* src, void* dst, const KParams& p, cudaStream_t s);
template <int DIM, class S, int MODE>
cudaError_t launch_flat_as(const void* src, void* dst, const KParams& p, cudaStream_t s) {
    const long long n = (long long)p.L.nx * p.L.ny * p.L.nz;
    const unsigned grid = (unsigned)((n + FLAT_THREADS - 1) / FLAT_THREADS);
    step_flat_kernel<DIM, S, MODE><<<grid, FLAT_THREADS, 0, s>>>((const S*)src, (S*)dst, p);
    return cudaGetLastError();
}
cudaError_t launch_flat_3d_f16(int prec, int mode, const void* src, void* dst, const KParams& p, cudaStream_t s);

// shared-memory staged (TMA bulk copy) step, TRT form, FP32/FP16/BF16 storage,
// nc = 4 or 8 consumer warps
const void* staged_function(int dim, int prec, int nc);
cudaError_t launch_staged(int dim, int prec, int nc, const void* src, void* dst, const KParams& p,
                          const StagedInfo& si, int grid, size_t smem, cudaStream_t s);

// several steps of a 2D cell per launch (step_multi.cu), TRT form
struct MultiGeo {
    int tw, th;  // nodes of a block's tile
    int m;       // nodes its region has around the tile: most steps per launch - 1
    int W, H;    // region: W >= tw + 2 m columns, H = th + 2 m rows
    int RS;      // elements of a region row in shared memory
    int steps;   // steps of this launch, 1 <= steps <= m + 1
};
// choose the tile and the steps per launch for a cell; false if the kernel cannot be used
bool multi_setup(int prec, const KParams& p, MultiGeo& g);
cudaError_t launch_multi(int prec, const void* src, void* dst, const KParams& p, const MultiGeo& g, cudaStream_t s);

// MARCH_STEPS steps of a 2D FP32, FP16 or BF16 cell with walls on every side in one pass over
// memory, in segments of `rows` rows (step_march.cu), TRT form
constexpr int MARCH_STEPS = 3;
constexpr int MARCH_COLUMNS = 56;  // columns a warp stores
int march_rows(int prec, const KParams& p);  // rows of a segment, 0: the device cannot be asked
cudaError_t launch_march(int prec, const void* src, void* dst, const KParams& p, int rows, cudaStream_t s);

// the same for the cells of a batch: what the kernel reads of a cell in its hot
// path (members as in KParams), all of a launch's cells by value
struct MarchCell {
    Layout L;
    int heat_axis, strips, block0;  // block0: its first block of the launch
    float gbetaf, omegaf, Thf, Tcf, bodyf[3], spf, smf, shpf, shmf, qpf, qmf, scale, inv_scale;
    decltype(KParams::tf) tf;
    int loff[14], soff[14];
    void* buf[2];
    const KParams* full;  // all parameters, in device memory
};
constexpr int MARCH_MANY = 64;  // most cells of a launch (kernel parameters hold 32 KB)
struct MarchBatch {
    MarchCell cell[MARCH_MANY];
    int n, rows;
};
static_assert(sizeof(MarchBatch) <= 32000, "kernel parameters");
MarchCell march_cell(const KParams& p, const void* buf0, const void* buf1, const KParams* full);
int march_cell_blocks(const MarchCell& c, int rows);
int march_batch_rows(int prec, const long long* strips_ny, int n);  // (strips, ny) of each cell; 0: the device cannot be asked
cudaError_t launch_march_batch(int prec, const MarchBatch& b, int grid, int parity, cudaStream_t s);

// per-unit entry points
cudaError_t launch_step_2d_f32(int vec, bool trt, int rows, const void*, void*, const KParams&, dim3, dim3,
                               cudaStream_t);
cudaError_t launch_step_2d_f16(int prec, int vec, bool trt, int rows, const void*, void*, const KParams&, dim3, dim3,
                               cudaStream_t);
cudaError_t launch_step_3d_f32(int vec, bool trt, int rows, const void*, void*, const KParams&, dim3, dim3,
                               cudaStream_t);
cudaError_t launch_step_3d_f16(int prec, int vec, bool trt, int rows, const void*, void*, const KParams&, dim3, dim3,
                               cudaStream_t);
cudaError_t launch_step_f64(int dim, int vec, bool trt, int rows, const void*, void*, const KParams&, dim3, dim3,
                            cudaStream_t);
const void* func_step_2d_f32(int vec, bool trt, int rows);
const void* func_step_2d_f16(int prec, int vec, bool trt, int rows);
const void* func_step_3d_f32(int vec, bool trt, int rows);
const void* func_step_3d_f16(int prec, int vec, bool trt, int rows);
const void* func_step_f64(int dim, int vec, bool trt, int rows);

}  // namespace tlbm

// Instantiate-and-launch helper: one case of a (vec, trt) switch.
#define TLBM_STEP_CASE(DIM, S, VEC, TRT)                                                            \
    if (vec == VEC && trt == TRT && rows == 1) {                                                    \
        tlbm::step_kernel<DIM, S, VEC, TRT><<<grid, block, 0, s>>>((const S*)src, (S*)dst, p);      \
        return cudaGetLastError();                                                                  \
    }

#define TLBM_STEP_FUNC(DIM, S, VEC, TRT) \
    if (vec == VEC && trt == TRT && rows == 1) return (const void*)&tlbm::step_kernel<DIM, S, VEC, TRT>;

// software-pipelined multi-row variants (two-relaxation-time form)
#define TLBM_ROWS_CASE(DIM, S, VEC, ROWS)                                                             \
    if (vec == VEC && trt && rows == ROWS) {                                                        \
        tlbm::step_kernel_rows<DIM, S, VEC, true, ROWS><<<grid, block, 0, s>>>((const S*)src, (S*)dst, p); \
        return cudaGetLastError();                                                                  \
    }
#define TLBM_ROWS_FUNC(DIM, S, VEC, ROWS) \
    if (vec == VEC && trt && rows == ROWS) return (const void*)&tlbm::step_kernel_rows<DIM, S, VEC, true, ROWS>;

// variants held to REGS registers
#define TLBM_STEPCAP_CASE(DIM, S, VEC, TRT, REGS)                                                          \
    if (vec == VEC && trt == TRT && rows == 1) {                                                    \
        tlbm::step_kernel_cap<DIM, S, VEC, TRT, REGS><<<grid, block, 0, s>>>((const S*)src, (S*)dst, p);  \
        return cudaGetLastError();                                                                  \
    }
#define TLBM_STEPCAP_FUNC(DIM, S, VEC, TRT, REGS) \
    if (vec == VEC && trt == TRT && rows == 1) return (const void*)&tlbm::step_kernel_cap<DIM, S, VEC, TRT, REGS>;
#define TLBM_AACAP_CASE(DIM, S, VEC, TRT, REGS)                                                                     \
    if (vec == VEC && trt == TRT && rows == -tlbm::AA_EVEN) {                                               \
        tlbm::step_kernel_aa_cap<DIM, S, VEC, TRT, tlbm::AA_EVEN, REGS><<<grid, block, 0, s>>>((S*)dst, p);       \
        return cudaGetLastError();                                                                          \
    }                                                                                                       \
    if (vec == VEC && trt == TRT && rows == -tlbm::AA_ODD) {                                                \
        tlbm::step_kernel_aa_cap<DIM, S, VEC, TRT, tlbm::AA_ODD, REGS><<<grid, block, 0, s>>>((S*)dst, p);        \
        return cudaGetLastError();                                                                          \
    }
#define TLBM_AACAP_FUNC(DIM, S, VEC, TRT, REGS)                                                                     \
    if (vec == VEC && trt == TRT && rows == -tlbm::AA_EVEN)                                                 \
        return (const void*)&tlbm::step_kernel_aa_cap<DIM, S, VEC, TRT, tlbm::AA_EVEN, REGS>;                     \
    if (vec == VEC && trt == TRT && rows == -tlbm::AA_ODD)                                                  \
        return (const void*)&tlbm::step_kernel_aa_cap<DIM, S, VEC, TRT, tlbm::AA_ODD, REGS>;

#define TLBM_ROWSCAP_CASE(DIM, S, VEC, ROWS, REGS)                                                    \
    if (vec == VEC && trt && rows == ROWS) {                                                        \
        tlbm::step_kernel_rows_cap<DIM, S, VEC, true, ROWS, REGS><<<grid, block, 0, s>>>((const S*)src, (S*)dst, p); \
        return cudaGetLastError();                                                                  \
    }
#define TLBM_ROWSCAP_FUNC(DIM, S, VEC, ROWS, REGS) \
    if (vec == VEC && trt && rows == ROWS) return (const void*)&tlbm::step_kernel_rows_cap<DIM, S, VEC, true, ROWS, REGS>;

// in-place (AA) halves
#define TLBM_AA_CASE(DIM, S, VEC, TRT)                                                                       \
    if (vec == VEC && trt == TRT && rows == -tlbm::AA_EVEN) {                                               \
        tlbm::step_kernel_aa<DIM, S, VEC, TRT, tlbm::AA_EVEN><<<grid, block, 0, s>>>((S*)dst, p);           \
        return cudaGetLastError();                                                                          \
    }                                                                                                       \
    if (vec == VEC && trt == TRT && rows == -tlbm::AA_ODD) {                                                \
        tlbm::step_kernel_aa<DIM, S, VEC, TRT, tlbm::AA_ODD><<<grid, block, 0, s>>>((S*)dst, p);            \
        return cudaGetLastError();                                                                          \
    }
#define TLBM_AA_FUNC(DIM, S, VEC, TRT)                                                                       \
    if (vec == VEC && trt == TRT && rows == -tlbm::AA_EVEN)                                                 \
        return (const void*)&tlbm::step_kernel_aa<DIM, S, VEC, TRT, tlbm::AA_EVEN>;                         \
    if (vec == VEC && trt == TRT && rows == -tlbm::AA_ODD)                                                  \
        return (const void*)&tlbm::step_kernel_aa<DIM, S, VEC, TRT, tlbm::AA_ODD>;
