// Diagnostics of a state: macroscopic fields and the FP64 reductions (a6)
// behind tlbm_nusselt, tlbm_energy and tlbm_status, one state or many at once.
//
// Both kernels walk segments of 32 nodes: a warp takes a segment, lane by lane,
// so that every population is one coalesced 32-element load at an offset known
// per launch (no division or address table per node and value).  A segment is a
// stretch of one row, or of the cell's nodes in memory order (walks_flat).
#include <algorithm>

#include "diag.cuh"
#include "diag.h"

namespace tlbm {

namespace {

constexpr int THREADS = 256;
constexpr int WARPS = THREADS / 32;

// segment k of a state: row (y, z) and first column
__device__ __forceinline__ void segment(unsigned k, unsigned segs, const Layout& L, int& x0, int& y, int& z) {
    const unsigned r = k / segs;
    x0 = 32 * (int)(k - r * segs);
    const unsigned zz = L.nz > 1 ? r / (unsigned)L.ny : 0u;
    z = (int)zz;
    y = (int)(r - zz * (unsigned)L.ny);
}

// this lane's node of segment k in memory order, across row ends, so that only the
// cell's last segment is not full; false if it has none
__device__ __forceinline__ bool flat_segment(unsigned k, const Layout& L, int& x, int& y, int& z) {
    const unsigned n = 32u * k + (threadIdx.x & 31u), r = n / (unsigned)L.nx;
    const unsigned zz = L.nz > 1 ? r / (unsigned)L.ny : 0u;
    x = (int)(n - r * (unsigned)L.nx);
    y = (int)(r - zz * (unsigned)L.ny);
    z = (int)zz;
    return r < (unsigned)L.ny * (unsigned)L.nz;
}

// segments of a state
__host__ __device__ inline unsigned segments(const Layout& L, bool flat) {
    const unsigned rows = (unsigned)L.ny * (unsigned)L.nz;
    return flat ? ((unsigned)L.nx * rows + 31u) / 32u : (unsigned)(L.nx + 31) / 32u * rows;
}

// Whether a state is walked in memory order.  FP64 arithmetic: always, the FP64
// pipe spends as much on an idle lane as on a busy one.  FP32 arithmetic, bound by
// HBM and the latency of its loads: where over a quarter of the lanes would idle,
// else a division less per node is worth more.  us, rows -> memory order: FP64
// fields of an FP16 state 161^3 882 -> 744, 385^3 10797 -> 9994, 3 x 300^2 517 ->
// 55, 256^3 2945 both ways; FP32 fields of an FP32 state, 2D, 33 nodes a row 31 ->
// 27, 65 32.2 -> 29.9, 129 49.8 and 51.1, 8193^2 869 and 1009.
bool walks_flat(const Layout& L, bool fp64) {
    const int lanes = (L.nx + 31) / 32 * 32;
    return fp64 || 4 * (lanes - L.nx) > lanes;
}

template <int DIM, class S>
__device__ __noinline__ void macros_node_d(const S* own, const KParams& p, const int* off, double* m) {
    double u[3];
    diag_macros_d<DIM, S>(own, p, off, m[0], u, m[4]);
    m[1] = u[0];
    m[2] = u[1];
    m[3] = u[2];
}

// Bound by HBM for FP32 fields (the state read once, the fields written once)
// and by the FP64 pipe for FP64 ones.  40 registers for the FP32 fields of 2D
// 16-bit and 3D FP32 states: the compiler's own 32 send too few of a node's loads
// out together (8193^2 FP16 799 -> 758 us), its 42 leave five blocks on an SM
// (385^3 FP32 1339 -> 1246).
template <int DIM, class S, class O>
constexpr int MACRO_BLOCKS = sizeof(O) == 4 && sizeof(S) == (DIM == 2 ? 2 : 4) ? 6 : 0;  // per SM, 0: as it comes
template <int DIM, class S, class O, bool FLAT>
__global__ void __launch_bounds__(THREADS, (MACRO_BLOCKS<DIM, S, O>))
    macros_kernel(const S* __restrict__ buf, const KParams p, const DiagOff k, unsigned segs, unsigned n,
                  O* __restrict__ rho, O* __restrict__ ux, O* __restrict__ uy, O* __restrict__ uz,
                  O* __restrict__ T) {
    const Layout& L = p.L;
    const unsigned nw = gridDim.x * WARPS;
    for (unsigned i = blockIdx.x * WARPS + (threadIdx.x >> 5); i < n; i += nw) {
        int x, y, z;
        if constexpr (FLAT) {
            if (!flat_segment(i, L, x, y, z)) continue;
        } else {
            segment(i, segs, L, x, y, z);
            x += threadIdx.x & 31;
            if (x >= L.nx) continue;
        }
        const S* own = buf + L.slot(x, y, z);
        O m[5];
        if constexpr (std::is_same<O, float>::value && !std::is_same<S, double>::value) {
            float f[Lat<DIM>::F::Q], g[Lat<DIM>::G::Q], u[3];
            diag_load<DIM, S, float>(own, p, k.off, f, g);
            if (diag_macros_f<DIM>(f, g, k, m[0], u, m[4])) {
                m[1] = u[0];
                m[2] = u[1];
                m[3] = u[2];
            } else {
                double d[5];
                macros_node_d<DIM, S>(own, p, k.off, d);
#pragma unroll
                for (int c = 0; c < 5; ++c) m[c] = (O)d[c];
            }
        } else {
            double u[3], r, t;
            diag_macros_d<DIM, S>(own, p, k.off, r, u, t);
            m[0] = (O)r;
            m[1] = (O)u[0];
            m[2] = (O)u[1];
            m[3] = (O)u[2];
            m[4] = (O)t;
        }
        const long long at = ((long long)z * L.ny + y) * L.nx + x;
        if (rho) rho[at] = m[0];
        if (ux) ux[at] = m[1];
        if (uy) uy[at] = m[2];
        if (DIM == 3 && uz) uz[at] = m[3];
        if (T) T[at] = m[4];
    }
}

// A thread's running sums.  FP32 terms go into double-FP32 sums of GROUP terms
// (exact to about 2^-47 of the group) that are then added to the FP64 sums: two
// conversions and two additions per GROUP terms instead of one of each per
// term, the FP64 pipe being 1/64 as fast as the FP32 one.  Eight terms: the sum
// of an 8193^2 FP32 state 2.0 ms without the groups, 0.98 with them.
template <class C>
struct Sums {
    static constexpr int GROUP = 8;
    double a[RED_FIELDS] = {0, 0, 0, 0, 0, 0};
    Df d[4] = {{0, 0}, {0, 0}, {0, 0}, {0, 0}};
    C mx = C(0);
    bool bad = false;
    int in = 0;
    __device__ static constexpr int field(int k) { return k == 3 ? 5 : k; }
    __device__ __forceinline__ void flush() {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            a[field(k)] += (double)d[k].h + (double)d[k].l;
            d[k] = {0, 0};
        }
        in = 0;
    }
    __device__ __forceinline__ void add(const C (&t)[5]) {
        const C v[4] = {t[0], t[1], t[2], t[4]};
        if (!isfinite(t[2]) || !isfinite(t[4]) || !isfinite(t[3])) bad = true;
        if constexpr (std::is_same<C, double>::value) {
            mx = fmax(mx, t[3]);
#pragma unroll
            for (int k = 0; k < 4; ++k) a[field(k)] += v[k];
        } else {
            mx = fmaxf(mx, t[3]);
            // a sum of such terms cannot overflow FP32 (false for a NaN too)
            if (fabsf(v[0]) + fabsf(v[1]) + fabsf(v[2]) + fabsf(v[3]) < 1e30f) {
#pragma unroll
                for (int k = 0; k < 4; ++k) df_add(d[k], v[k]);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) a[field(k)] += (double)v[k];
            }
            if (++in == GROUP) flush();
        }
    }
    __device__ __forceinline__ void close() {
        if constexpr (!std::is_same<C, double>::value) flush();
        a[3] = (double)mx;
        a[4] = bad ? 1.0 : 0.0;
    }
};

// FP64 reduction, pass 1: a state's blocks sum its segments in a fixed order
// (warp w of the state's W warps takes segments w, w + W, ..., then a fixed
// shuffle tree and a fixed cross-warp order) into one row of partials each.
// The grid of a state depends on its size only, so its sums are the same bits
// whether it is reduced alone or with others.  ONE: a single state whose
// parameters come by value.
template <int DIM, class S, bool ONE>
__global__ void __launch_bounds__(THREADS)
    reduce_kernel(const __grid_constant__ RedStates st, int count, const __grid_constant__ KParams p1,
                  const __grid_constant__ DiagOff k1) {
    using C = typename Storage<S>::C;
    using LF = typename Lat<DIM>::F;
    using LG = typename Lat<DIM>::G;
    __shared__ int soff[MAXQ + 7];
    __shared__ double sm[WARPS][RED_FIELDS];
    int i = 0;
    if constexpr (!ONE)
        while (i + 1 < count && st.s[i + 1].block0 <= (int)blockIdx.x) ++i;
    const RedState& q = st.s[i];
    const KParams& p = ONE ? p1 : *q.kp;
    if constexpr (!ONE) {
        static_for<LF::Q + LG::Q>([&](auto jj) {
            constexpr int j = decltype(jj)::value;
            constexpr int ex = j < LF::Q ? LF::e(j < LF::Q ? j : 0, 0) : LG::e(j < LF::Q ? 0 : j - LF::Q, 0);
            if (threadIdx.x == j) soff[j] = p.loff[j] - ex;  // the two-buffer order
        });
        __syncthreads();
    }
    const int* off = ONE ? k1.off : soff;
    const Layout L = p.L;
    const S* buf = static_cast<const S*>(q.buf);
    const unsigned segs = (unsigned)(L.nx + 31) / 32u, n = segments(L, q.flat);
    const unsigned W = (unsigned)q.blocks * WARPS;
    const unsigned k0 = ((unsigned)blockIdx.x - (unsigned)q.block0) * WARPS + (threadIdx.x >> 5);
    Sums<C> sum;
    if (q.flat) {
        for (unsigned k = k0; k < n; k += W) {
            int x, y, z;
            if (flat_segment(k, L, x, y, z)) {
                C t[5];
                node_terms<DIM, S>(buf + L.slot(x, y, z), p, off, t);
                sum.add(t);
            }
        }
    } else if constexpr (!std::is_same<C, double>::value) {
        for (unsigned k = k0; k < n; k += W) {
            int x, y, z;
            segment(k, segs, L, x, y, z);
            x += threadIdx.x & 31;
            if (x < L.nx) {
                C t[5];
                node_terms<DIM, S>(buf + L.slot(x, y, z), p, off, t);
                sum.add(t);
            }
        }
    }
    sum.close();
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int f = 0; f < RED_FIELDS; ++f) {
            const double v = __shfl_down_sync(0xffffffffu, sum.a[f], o);
            sum.a[f] = (f == 3 || f == 4) ? fmax(sum.a[f], v) : sum.a[f] + v;
        }
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0)
        for (int f = 0; f < RED_FIELDS; ++f) sm[w][f] = sum.a[f];
    __syncthreads();
    if (threadIdx.x < RED_FIELDS) {
        const int f = threadIdx.x;
        double v = sm[0][f];
        for (int j = 1; j < WARPS; ++j) v = (f == 3 || f == 4) ? fmax(v, sm[j][f]) : v + sm[j][f];
        q.partials[(long long)((int)blockIdx.x - q.block0) * RED_FIELDS + f] = v;
    }
}

// Pass 2: block i combines state i's partials, warp f the field f (each lane
// every 32nd row in order, then a fixed shuffle tree).
__global__ void __launch_bounds__(32 * RED_FIELDS)
    reduce_final_kernel(const __grid_constant__ RedStates st, double* __restrict__ out) {
    const RedState& q = st.s[blockIdx.x];
    const int f = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const bool is_max = f == 3 || f == 4;
    double v = 0.0;
    for (int b = lane; b < q.blocks; b += 32) {
        const double t = q.partials[b * RED_FIELDS + f];
        v = is_max ? fmax(v, t) : v + t;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const double t = __shfl_down_sync(0xffffffffu, v, o);
        v = is_max ? fmax(v, t) : v + t;
    }
    if (lane == 0) out[8 * blockIdx.x + f] = v;
    if (threadIdx.x == 0) out[8 * blockIdx.x + 6] = (double)*q.status;
}

// blocks of one state's reduction: a few segments per warp, at most four blocks
// on each of 152 SMs (a constant, so that the sums do not depend on the device)
int red_blocks(const KParams& p, bool flat) {
    const long long n = segments(p.L, flat);
    return (int)std::max<long long>(1, std::min<long long>(RED_BLOCKS, (n + 4 * WARPS - 1) / (4 * WARPS)));
}

template <int DIM, class S, class O, bool FLAT>
cudaError_t macros_as(const void* buf, const KParams& p, void* rho, void* ux, void* uy, void* uz, void* T, cudaStream_t s) {
    const unsigned n = segments(p.L, FLAT), grid = std::min(16384u, (n + WARPS - 1) / WARPS);
    macros_kernel<DIM, S, O, FLAT><<<grid, THREADS, 0, s>>>((const S*)buf, p, diag_offsets<DIM>(p), (unsigned)(p.L.nx + 31) / 32u,
                                                            n, (O*)rho, (O*)ux, (O*)uy, (O*)uz, (O*)T);
    return cudaGetLastError();
}
template <int DIM, class S>
cudaError_t macros_t(const void* buf, const KParams& p, void* rho, void* ux, void* uy, void* uz, void* T, bool f64,
                     cudaStream_t s) {
    if (f64) return macros_as<DIM, S, double, true>(buf, p, rho, ux, uy, uz, T, s);
    if constexpr (!std::is_same<S, double>::value)
        if (!walks_flat(p.L, false)) return macros_as<DIM, S, float, false>(buf, p, rho, ux, uy, uz, T, s);
    return macros_as<DIM, S, float, true>(buf, p, rho, ux, uy, uz, T, s);
}

template <int DIM, class S>
cudaError_t reduce_t(const RedStates& st, int count, unsigned grid, const KParams* p1, cudaStream_t s) {
    if (p1) reduce_kernel<DIM, S, true><<<grid, THREADS, 0, s>>>(st, count, *p1, diag_offsets<DIM>(*p1));
    else reduce_kernel<DIM, S, false><<<grid, THREADS, 0, s>>>(st, count, KParams{}, DiagOff{});
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_macros(int dim, int prec, const void* buf, const KParams& p, void* rho, void* ux, void* uy,
                          void* uz, void* T, bool f64, cudaStream_t s) {
    if (dim == 2) {
        if (prec == 0) return macros_t<2, double>(buf, p, rho, ux, uy, uz, T, f64, s);
        if (prec == 1) return macros_t<2, float>(buf, p, rho, ux, uy, uz, T, f64, s);
        if (prec == 2) return macros_t<2, __half>(buf, p, rho, ux, uy, uz, T, f64, s);
        return macros_t<2, __nv_bfloat16>(buf, p, rho, ux, uy, uz, T, f64, s);
    }
    if (prec == 0) return macros_t<3, double>(buf, p, rho, ux, uy, uz, T, f64, s);
    if (prec == 1) return macros_t<3, float>(buf, p, rho, ux, uy, uz, T, f64, s);
    if (prec == 2) return macros_t<3, __half>(buf, p, rho, ux, uy, uz, T, f64, s);
    return macros_t<3, __nv_bfloat16>(buf, p, rho, ux, uy, uz, T, f64, s);
}

cudaError_t launch_reduce(int dim, int prec, RedStates& st, int count, const KParams* const* host_kp, double* out,
                          cudaStream_t s) {
    int grid = 0;
    for (int i = 0; i < count; ++i) {
        st.s[i].block0 = grid;
        st.s[i].flat = walks_flat(host_kp[i]->L, prec == 0);
        st.s[i].blocks = red_blocks(*host_kp[i], st.s[i].flat);
        grid += st.s[i].blocks;
    }
    const KParams* p1 = count == 1 && !st.s[0].kp ? host_kp[0] : nullptr;
    cudaError_t e;
    if (dim == 2) {
        if (prec == 0) e = reduce_t<2, double>(st, count, grid, p1, s);
        else if (prec == 1) e = reduce_t<2, float>(st, count, grid, p1, s);
        else if (prec == 2) e = reduce_t<2, __half>(st, count, grid, p1, s);
        else e = reduce_t<2, __nv_bfloat16>(st, count, grid, p1, s);
    } else {
        if (prec == 0) e = reduce_t<3, double>(st, count, grid, p1, s);
        else if (prec == 1) e = reduce_t<3, float>(st, count, grid, p1, s);
        else if (prec == 2) e = reduce_t<3, __half>(st, count, grid, p1, s);
        else e = reduce_t<3, __nv_bfloat16>(st, count, grid, p1, s);
    }
    if (e != cudaSuccess) return e;
    reduce_final_kernel<<<count, 32 * RED_FIELDS, 0, s>>>(st, out);
    return cudaGetLastError();
}

}  // namespace tlbm
