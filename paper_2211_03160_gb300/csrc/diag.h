// Host-side entry points of the diagnostic kernels (diag.cu).
#pragma once
#include <cuda_runtime.h>

#include "kernels.cuh"

namespace tlbm {

constexpr int RED_FIELDS = 6;    // sum u_h T, sum 1/2 rho u^2, sum rho, max u^2, bad, sum T
constexpr int RED_BLOCKS = 608;  // most blocks of one state's reduction
constexpr int RED_MANY = 64;     // most states of one reduction launch

// rho, u, T of the state into dense arrays of doubles (f64) or floats; null
// arrays are left out.
cudaError_t launch_macros(int dim, int prec, const void* buf, const KParams& p, void* rho, void* ux, void* uy,
                          void* uz, void* T, bool f64, cudaStream_t s);

// The reductions of `count` <= RED_MANY states of one lattice and storage in
// two launches.  State i: its population buffer, parameters (device address,
// or null with count = 1 to use *p), nodes, scratch of RED_BLOCKS * RED_FIELDS
// doubles, and status word.  out[8 i .. 8 i + 6): its RED_FIELDS results,
// out[8 i + 6]: its status word as a double.  All in device memory.
struct RedState {
    const void* buf;
    const KParams* kp;
    double* partials;
    const int* status;
    int block0, blocks;  // its blocks of the flattened grid (set by launch_reduce)
    bool flat;           // walked in memory order (set by launch_reduce)
};
struct RedStates {
    RedState s[RED_MANY];
};
cudaError_t launch_reduce(int dim, int prec, RedStates& st, int count, const KParams* const* host_kp, double* out,
                          cudaStream_t s);

}  // namespace tlbm
