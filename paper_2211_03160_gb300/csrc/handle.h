// Host-side state of a tlbm handle (private to the library).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/tlbm.h"
#include "dispatch.h"

struct tlbm_s {
    int nx, ny, nz, dim, lattice, prec;
    int qf, qg;
    double Ra, Pr, Ma;
    tlbm_params prm;
    double U, H, nu, alpha, gbeta, a_T, omega;
    double S[tlbm::MAXQ], Q[7];
    tlbm::KParams kp;
    int vec, trt, bx, by;      // step kernel variant and block shape
    int rows;                  // consecutive rows per thread (software-pipelined when > 1)
    int aa;                    // 1: in-place (AA) streaming in one population buffer
    int nbuf;                  // population buffers: 2, or 1 in place
    int graph_chosen;          // set by tlbm_set_graph: launch single steps as the caller asked
    int graph_steps;           // steps per CUDA graph replay in tlbm_step (0: plain launches)
    cudaGraphExec_t graph;     // captured block of graph_steps steps starting from buffer 0
    cudaStream_t capture_stream;
    int multi;                 // > 1: steps per launch of calls of MULTI_CALL steps or more
    int march;                 // > 0: by step_march.cu in segments of this many rows, else by step_multi.cu
    tlbm::MultiGeo mg;         // tile of the latter
    int flat;                  // 1: the kernel with one thread per node in memory order
    int staged;                // 1: shared-memory staged (TMA bulk copy) kernel
    int variant_chosen;        // 2: tlbm_set_variant / tlbm_set_staged chose the kernel; 1: the register kernels, as the library chooses
    int staged_tw, staged_nc, staged_stages, staged_grid;
    unsigned long long wait_ns;  // staged kernel: give up on a copy after this long
    size_t staged_smem;
    size_t elem;               // bytes per stored value
    size_t popset_bytes;       // one population buffer (f planes then g planes)
    size_t red_off, res_off, stage_off, total_bytes;
    size_t status_off;         // device status word of the staged kernel
    char* mem;                 // bound device block
    size_t mem_bytes;
    void* buf[2];
    int cur;                   // buffer holding the current state (in place: 0 natural, 1 swapped order)
    int64_t t;
    cudaStream_t stream;
    int64_t launches;
    char err[256];
};

namespace tlbm {
// Calls of at least this many steps advance several steps per launch where the
// handle or batch does that at all (shorter calls keep one launch per step).
constexpr int MULTI_CALL = 16;

// The reductions of many handles at once (api.cu); the first handle that
// failed in *failed.
int reduce_many(tlbm_t* hs, int n, const KParams* d_kp, cudaStream_t stream, double* nu, int* diverged,
                int* failed);
}  // namespace tlbm
