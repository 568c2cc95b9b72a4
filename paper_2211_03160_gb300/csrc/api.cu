// C ABI of the thermal lattice Boltzmann library (declared in include/tlbm.h):
// handle lifecycle, parameter mapping, memory binding, launches of the fused
// step, and the initial-state, population transfer, macro and reduction kernels.
#include <cuda_runtime.h>

#include <cmath>
#include <cstddef>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>

#include "../../include/tlbm.h"
#include "diag.h"
#include "dispatch.h"
#include "handle.h"

using namespace tlbm;

namespace {

constexpr int RED_ROWS = 1024;     // rows of reduction partials in the bound block's scratch
static_assert(RED_ROWS >= RED_BLOCKS, "scratch of the reductions");
constexpr long long STAGE_NODES = 1ll << 21;  // FP64 staging chunk for population transfers

thread_local char g_create_error[256] = "";

size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

}  // namespace



// ------------------------------------------------------------------ errors

static int fail(tlbm_t h, int code, const char* fmt, ...) {
    char* dst = h ? h->err : g_create_error;
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(dst, 256, fmt, ap);
    va_end(ap);
    return code;
}

static int cuda_fail(tlbm_t h, cudaError_t e, const char* what) {
    return fail(h, TLBM_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

static void drop_graph(tlbm_t h);
static int set_staged(tlbm_t h, int tile_width, int stages);
static void pick_16bit(tlbm_t h);
static void pick_multi(tlbm_t h);

// The buffer (two-buffer pull) or the order (in place: 0 natural, 1 swapped)
// of the current state, and the matching state order for the diagnostic and
// transfer kernels.
static void set_cur(tlbm_t h, int c) {
    h->cur = c;
    h->kp.state = h->aa ? (c ? 2 : 1) : 0;
}

#define TLBM_CHECK_HANDLE(h)                                   \
    do {                                                       \
        if (!(h)) return fail(nullptr, TLBM_ERR_ARG, "NULL handle"); \
        (h)->err[0] = 0;                                       \
    } while (0)

#define TLBM_CHECK_BOUND(h)                                                         \
    do {                                                                            \
        if (!(h)->mem) return fail((h), TLBM_ERR_UNBOUND, "device memory not bound"); \
    } while (0)

// ------------------------------------------------------------------ kernels

namespace {

// splitmix64 output function (Steele, Lea & Flood 2014).
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
    uint64_t z = x + 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// A box of nodes [x0, x0 + wx) x [y0, y0 + wy) x [z0, z0 + wz), enumerated x fastest.
struct Window {
    int x0, y0, z0, wx, wy, wz;
};

__device__ __forceinline__ void window_xyz(long long k, const Window& w, int& x, int& y, int& z) {
    x = w.x0 + (int)(k % w.wx);
    long long r = k / w.wx;
    y = w.y0 + (int)(r % w.wy);
    z = w.z0 + (int)(r / w.wy);
}

__device__ __forceinline__ void node_xyz(long long n, const Layout& L, int& x, int& y, int& z) {
    x = (int)(n % L.nx);
    long long r = n / L.nx;
    y = (int)(r % L.ny);
    z = (int)(r / L.ny);
}

// Initial state: f = w (rho = 1, u = 0), g = g_eq(T, 0) with the conductive
// profile plus seeded uniform noise.  Every pre-collision value f_i(x) is
// written where the state order p.state keeps it (pre_index).
template <int DIM, class S>
__global__ void init_kernel(S* __restrict__ buf, const KParams p, uint64_t seed, double amp) {
    using LF = typename Lat<DIM>::F;
    using LG = typename Lat<DIM>::G;
    using C = typename Storage<S>::C;
    const Layout& L = p.L;
    const long long N = (long long)L.nx * L.ny * L.nz;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        node_xyz(n, L, x, y, z);
        const int c = p.heat_axis == 0 ? x : (p.heat_axis == 1 ? y : z);
        const int len = p.heat_axis == 0 ? L.nx : (p.heat_axis == 1 ? L.ny : L.nz);
        const double r = (double)(splitmix64(seed ^ splitmix64((uint64_t)n)) >> 11) * 0x1.0p-53;
        double T = __dadd_rn(p.Th, __dmul_rn(p.Tc - p.Th, __ddiv_rn((double)c + 0.5, (double)len)));
        T = __dadd_rn(T, __dmul_rn(amp, 2.0 * r - 1.0));
        double nm[LG::Q];
        for (int k = 0; k < LG::Q; ++k) nm[k] = 0.0;
        nm[0] = T;
        nm[DIM == 2 ? 3 : 4] = p.a_T * T;
        double gq[LG::Q];
        populations<LG, double>(nm, gq);
        const C scale = (C)p.scale;
        static_for<LF::Q>([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            *TLBM_DBG(p, (buf + pre_index<LF, i>(p, x, y, z)), 0, 1) = enc_f<LF, S, C>(C(0), i, scale);
        });
        S* gb = buf + (long long)LF::Q * L.plane;
        static_for<LG::Q>([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            *TLBM_DBG(p, (gb + pre_index<LG, i>(p, x, y, z)), 0, 1) = enc_g<S, C>((C)gq[i], scale);
        });
    }
}

// Initial state from given fields (warm start): f = f_eq(rho = 1, u) and
// g = g_eq(T, u) at every node, written where p.state keeps them.
template <int DIM, class S>
__global__ void init_fields_kernel(S* __restrict__ buf, const KParams p, const float* __restrict__ Tf,
                                   const float* __restrict__ uxf, const float* __restrict__ uyf,
                                   const float* __restrict__ uzf) {
    using LF = typename Lat<DIM>::F;
    using LG = typename Lat<DIM>::G;
    using C = typename Storage<S>::C;
    const Layout& L = p.L;
    const long long N = (long long)L.nx * L.ny * L.nz;
    for (long long n = blockIdx.x * (long long)blockDim.x + threadIdx.x; n < N;
         n += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        node_xyz(n, L, x, y, z);
        const double T = Tf[n];
        const double u[3] = {uxf ? (double)uxf[n] : 0.0, uyf ? (double)uyf[n] : 0.0,
                             (DIM == 3 && uzf) ? (double)uzf[n] : 0.0};
        const double uu = u[0] * u[0] + u[1] * u[1] + u[2] * u[2];
        double nm[LG::Q];
        for (int k = 0; k < LG::Q; ++k) nm[k] = 0.0;
        nm[0] = T;
        nm[1] = u[0] * T;
        nm[2] = u[1] * T;
        if (DIM == 3) nm[3] = u[2] * T;
        nm[DIM == 2 ? 3 : 4] = p.a_T * T;
        double gq[LG::Q];
        populations<LG, double>(nm, gq);
        const C scale = (C)p.scale;
        static_for<LF::Q>([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            const double eu = LF::e(i, 0) * u[0] + LF::e(i, 1) * u[1] + LF::e(i, 2) * u[2];
            const double dev = (LF::w36(i) / 36.0) * (3.0 * eu + 4.5 * eu * eu - 1.5 * uu);
            *TLBM_DBG(p, (buf + pre_index<LF, i>(p, x, y, z)), 0, 1) = enc_f<LF, S, C>((C)dev, i, scale);
        });
        S* gb = buf + (long long)LF::Q * L.plane;
        static_for<LG::Q>([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            *TLBM_DBG(p, (gb + pre_index<LG, i>(p, x, y, z)), 0, 1) = enc_g<S, C>((C)gq[i], scale);
        });
    }
}

// Host FP64 populations (one plane, nodes [n0, n0 + cnt)) -> the state's slots.
// dev: offset storage takes flow values as deviations f_i - w_i (the exact
// FP64 image of what it stores; checkpoints), otherwise as f_i.
template <int DIM, class S>
__global__ void scatter_kernel(S* __restrict__ buf, const double* __restrict__ stage, int pop, long long n0,
                               long long cnt, const Window w, const KParams p, bool dev) {
    using LF = typename Lat<DIM>::F;
    using LG = typename Lat<DIM>::G;
    using C = typename Storage<S>::C;
    const Layout& L = p.L;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < cnt;
         k += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        window_xyz(n0 + k, w, x, y, z);
        const double v = stage[k];
        static_for<LF::Q>([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            if (pop == i) {
                S s;
                if constexpr (Storage<S>::offset) s = from_c<S>((C)((dev ? v : v - LF::w36(i) / 36.0) * p.scale));
                else s = (S)v;
                *TLBM_DBG(p, (buf + pre_index<LF, i>(p, x, y, z)), 0, 1) = s;
            }
        });
        static_for<LG::Q>([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            if (pop == LF::Q + i) {
                S s;
                if constexpr (Storage<S>::offset) s = from_c<S>((C)(v * p.scale));
                else s = (S)v;
                *TLBM_DBG(p, (buf + ((long long)LF::Q * L.plane + pre_index<LG, i>(p, x, y, z))), 0, 1) = s;
            }
        });
    }
}

// The state's slots -> canonical FP64 populations (one plane, nodes [n0, n0 + cnt)).
// dev: offset storage hands out flow deviations f_i - w_i (exact) instead.
template <int DIM, class S>
__global__ void gather_kernel(const S* __restrict__ buf, double* __restrict__ stage, int pop, long long n0,
                              long long cnt, const Window w, const KParams p, bool dev) {
    using LF = typename Lat<DIM>::F;
    using LG = typename Lat<DIM>::G;
    const Layout& L = p.L;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < cnt;
         k += (long long)gridDim.x * blockDim.x) {
        int x, y, z;
        window_xyz(n0 + k, w, x, y, z);
        double v = 0.0;
        static_for<LF::Q>([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            if (pop == i) {
                const double raw = to_c<double>(*TLBM_DBG(p, (buf + pre_index<LF, i>(p, x, y, z)), 0, 1));
                if constexpr (Storage<S>::offset) v = (dev ? 0.0 : LF::w36(i) / 36.0) + raw * (double)p.inv_scale;
                else v = raw;
            }
        });
        static_for<LG::Q>([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            if (pop == LF::Q + i) {
                const double raw =
                    to_c<double>(*TLBM_DBG(p, (buf + ((long long)LF::Q * L.plane + pre_index<LG, i>(p, x, y, z))), 0, 1));
                if constexpr (Storage<S>::offset) v = raw * (double)p.inv_scale;
                else v = raw;
            }
        });
        stage[k] = v;
    }
}

template <int DIM, class S>
struct DiagKernels {
    static cudaError_t init(void* buf, const KParams& p, uint64_t seed, double amp, cudaStream_t s) {
        init_kernel<DIM, S><<<2048, 256, 0, s>>>((S*)buf, p, seed, amp);
        return cudaGetLastError();
    }
    static cudaError_t init_fields(void* buf, const KParams& p, const float* T, const float* ux, const float* uy,
                                   const float* uz, cudaStream_t s) {
        init_fields_kernel<DIM, S><<<2048, 256, 0, s>>>((S*)buf, p, T, ux, uy, uz);
        return cudaGetLastError();
    }
    static cudaError_t scatter(void* buf, const double* st, int pop, long long n0, long long cnt, const Window& w,
                               const KParams& p, cudaStream_t s, bool dev = false) {
        scatter_kernel<DIM, S><<<1024, 256, 0, s>>>((S*)buf, st, pop, n0, cnt, w, p, dev);
        return cudaGetLastError();
    }
    static cudaError_t gather(const void* buf, double* st, int pop, long long n0, long long cnt, const Window& w,
                              const KParams& p, cudaStream_t s, bool dev = false) {
        gather_kernel<DIM, S><<<1024, 256, 0, s>>>((const S*)buf, st, pop, n0, cnt, w, p, dev);
        return cudaGetLastError();
    }
};

// dispatch a diagnostic call over (dim, precision)
template <class F>
cudaError_t with_types(int dim, int prec, F&& f) {
    if (dim == 2) {
        switch (prec) {
        case TLBM_FP64: return f(DiagKernels<2, double>{});
        case TLBM_FP32: return f(DiagKernels<2, float>{});
        case TLBM_FP16_OFFSET: return f(DiagKernels<2, __half>{});
        default: return f(DiagKernels<2, __nv_bfloat16>{});
        }
    }
    switch (prec) {
    case TLBM_FP64: return f(DiagKernels<3, double>{});
    case TLBM_FP32: return f(DiagKernels<3, float>{});
    case TLBM_FP16_OFFSET: return f(DiagKernels<3, __half>{});
    default: return f(DiagKernels<3, __nv_bfloat16>{});
    }
}

}  // namespace

// ------------------------------------------------------------------ setup

extern "C" void tlbm_default_params(tlbm_params* p) {
    if (!p) return;
    memset(p, 0, sizeof(*p));
    p->walls = TLBM_RB;
    const double nan = std::nan("");
    p->a_T = p->nu = p->alpha = p->gbeta = nan;
    p->s_rho = p->s_e = p->s_eps = p->s_j = p->s_q = p->s_pi = p->s_m = nan;
    p->q_e = p->q_v = nan;
    p->Th = p->Tc = nan;
    p->store_scale = nan;
}

static double pick(double v, double d) { return std::isnan(v) ? d : v; }

// Default step variant per (dimension, storage): nodes per thread and block
// shape, from a sweep on GB300 at 8193^2 (2D) and 385^3 (3D).
struct VariantDefault {
    int vec, bx, by, rows;
};
static VariantDefault default_variant(int dim, int prec) {
    if (dim == 2) {
        switch (prec) {
        case TLBM_FP64: return {2, 64, 1, 1};
        case TLBM_FP32: return {4, 32, 4, 2};
        default: return {4, 32, 1, 1};
        }
    }
    switch (prec) {
    case TLBM_FP64: return {1, 32, 4, 1};
    case TLBM_FP32: return {1, 32, 2, 1};
    default: return {2, 32, 1, 1};
    }
}
static int default_vec(int dim, int prec) { return default_variant(dim, prec).vec; }

// FP64 cells with two-relaxation-time rates: one thread per node in memory order
static int flat_fp64(tlbm_t h) {
    return h->prec == TLBM_FP64 && h->kp.trt && (double)h->nx * h->ny * h->nz <= FLAT_NODES;
}

extern "C" int tlbm_create(tlbm_t* out, int nx, int ny, int nz, int lattice, double Ra, double Pr, double Ma,
                           int precision, const tlbm_params* pin) {
    g_create_error[0] = 0;
    if (!out) return fail(nullptr, TLBM_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (lattice != TLBM_D2Q9_D2Q5 && lattice != TLBM_D3Q19_D3Q7)
        return fail(nullptr, TLBM_ERR_ARG, "unknown lattice %d", lattice);
    if (precision < TLBM_FP64 || precision > TLBM_BF16_OFFSET)
        return fail(nullptr, TLBM_ERR_UNSUPPORTED, "unknown precision %d", precision);
    const int dim = lattice == TLBM_D2Q9_D2Q5 ? 2 : 3;
    if (dim == 2) nz = 1;
    if (nx < 3 || ny < 3 || (dim == 3 && nz < 3))
        return fail(nullptr, TLBM_ERR_ARG, "grid %d x %d x %d too small (each extent >= 3)", nx, ny, nz);
    if (nx > (1 << 24) || ny > 65535 || nz > 65535 || (double)nx * ny * nz > 4e10)
        return fail(nullptr, TLBM_ERR_ARG, "grid too large (nx <= 2^24, ny and nz <= 65535)");
    if (!(Ra > 0) || !(Pr > 0) || !(Ma > 0))
        return fail(nullptr, TLBM_ERR_ARG, "Ra, Pr and Ma must be > 0");
    tlbm_params prm;
    if (pin) prm = *pin;
    else tlbm_default_params(&prm);
    if (prm.walls != TLBM_RB && prm.walls != TLBM_SIDE_HEATED)
        return fail(nullptr, TLBM_ERR_ARG, "unknown walls %d", prm.walls);
    if (prm.periodic_mask < 0 || prm.periodic_mask > 7)
        return fail(nullptr, TLBM_ERR_ARG, "periodic_mask out of range");
    if (prm.streaming != TLBM_STREAM_PULL && prm.streaming != TLBM_STREAM_INPLACE)
        return fail(nullptr, TLBM_ERR_ARG, "unknown streaming %d", prm.streaming);

    tlbm_s* h = new (std::nothrow) tlbm_s();
    if (!h) return fail(nullptr, TLBM_ERR_OOM, "host allocation failed");
    h->nx = nx; h->ny = ny; h->nz = nz; h->dim = dim; h->lattice = lattice; h->prec = precision;
    h->qf = dim == 2 ? 9 : 19;
    h->qg = dim == 2 ? 5 : 7;
    h->Ra = Ra; h->Pr = Pr; h->Ma = Ma;
    h->prm = prm;

    // free-fall scaling, Eqs. (2)-(4)
    h->prm.Th = pick(prm.Th, 0.5);
    h->prm.Tc = pick(prm.Tc, -0.5);
    const double dT = h->prm.Th - h->prm.Tc;
    h->U = prm.u_is_ma ? Ma : Ma / std::sqrt(3.0);
    h->H = dim == 2 ? ny : nz;
    h->nu = pick(prm.nu, h->U * h->H * std::sqrt(Pr / Ra));
    h->alpha = pick(prm.alpha, h->U * h->H / std::sqrt(Pr * Ra));
    h->gbeta = pick(prm.gbeta, h->U * h->U / (h->H * dT));
    h->a_T = pick(prm.a_T, dim == 2 ? -2.0 / 3.0 : -0.75);
    h->omega = dim == 2 ? (4.0 + h->a_T) / 10.0 : (6.0 + h->a_T) / 21.0;
    if (!(3.0 * h->nu > 1e-6) || !(h->alpha > 0) || !(h->omega > 0) || !(dT != 0)) {
        delete h;
        return fail(nullptr, TLBM_ERR_ARG, "relaxation time out of range (3 nu = %g, alpha = %g)", 3.0 * h->nu,
                    h->alpha);
    }
    const double snu = 1.0 / (3.0 * h->nu + 0.5);
    const double sq = 8.0 * (2.0 - snu) / (8.0 - snu);
    const double s_rho = pick(prm.s_rho, 1.0), s_e = pick(prm.s_e, snu), s_eps = pick(prm.s_eps, snu);
    const double s_j = pick(prm.s_j, 1.0), s_q = pick(prm.s_q, sq), s_pi = pick(prm.s_pi, snu);
    const double s_m = pick(prm.s_m, sq);
    if (dim == 2) {
        const double S[9] = {s_rho, s_e, s_eps, s_j, s_q, s_j, s_q, snu, snu};
        memcpy(h->S, S, sizeof(S));
    } else {
        const double S[19] = {s_rho, s_e, s_eps, s_j, s_q, s_j, s_q, s_j, s_q, snu,
                              s_pi,  snu, s_pi,  snu, snu, snu, s_m, s_m, s_m};
        memcpy(h->S, S, sizeof(S));
    }
    const double qj = 1.0 / (h->alpha / h->omega + 0.5);
    const double qeven = 1.0 / (0.5 + 0.25 / (1.0 / qj - 0.5));
    const double q_e = pick(prm.q_e, qeven), q_v = pick(prm.q_v, qeven);
    if (dim == 2) {
        const double Q[5] = {1.0, qj, qj, q_e, q_v};
        memcpy(h->Q, Q, sizeof(Q));
    } else {
        const double Q[7] = {1.0, qj, qj, qj, q_e, q_v, q_v};
        memcpy(h->Q, Q, sizeof(Q));
    }

    // device layout
    KParams& kp = h->kp;
    memset(&kp, 0, sizeof(kp));
    kp.L.nx = nx; kp.L.ny = ny; kp.L.nz = nz; kp.L.dim = dim;
    kp.L.zg = dim == 3 ? 1 : 0;
    kp.L.P = (int)align_up((size_t)nx + 16, ROW_ALIGN);
    const long long rows = (long long)(ny + 2) * (dim == 3 ? nz + 2 : 1);
    kp.L.plane = (long long)align_up((size_t)(SLOT_OFF + rows * kp.L.P + TAIL), 64);
    kp.periodic = prm.periodic_mask;
    kp.grav_axis = dim - 1;
    kp.heat_axis = prm.walls == TLBM_RB ? dim - 1 : 0;
    // two-relaxation-time form applies when the even / odd non-conserved rates coincide
    {
        const int ev2[] = {1, 2, 7, 8}, od2[] = {4, 6};
        const int ev3[] = {1, 2, 9, 10, 11, 12, 13, 14, 15}, od3[] = {4, 6, 8, 16, 17, 18};
        const int* ev = dim == 2 ? ev2 : ev3;
        const int* od = dim == 2 ? od2 : od3;
        const int nev = dim == 2 ? 4 : 9, nod = dim == 2 ? 2 : 6;
        bool ok = true;
        for (int k = 1; k < nev; ++k) ok = ok && h->S[ev[k]] == h->S[ev[0]];
        for (int k = 1; k < nod; ++k) ok = ok && h->S[od[k]] == h->S[od[0]];
        const int tev = dim == 2 ? 3 : 4;  // first even non-conserved thermal moment
        for (int k = tev + 1; k < h->qg; ++k) ok = ok && h->Q[k] == h->Q[tev];
        for (int k = 2; k < tev; ++k) ok = ok && h->Q[k] == h->Q[1];
        kp.trt = ok ? 1 : 0;
        kp.sp = h->S[ev[0]];
        kp.sm = h->S[od[0]];
        kp.shp = 1.0 - 0.5 * kp.sp;
        kp.shm = 1.0 - 0.5 * kp.sm;
        kp.qp = h->Q[tev];
        kp.qm = h->Q[1];
        kp.spf = (float)kp.sp; kp.smf = (float)kp.sm; kp.shpf = (float)kp.shp; kp.shmf = (float)kp.shm;
        kp.qpf = (float)kp.qp; kp.qmf = (float)kp.qm;
    }
    h->trt = kp.trt;
    h->flat = flat_fp64(h);
    {
        // per-population pull / store offsets (elements, relative to a node's own
        // slot in plane 0): plane j, shifted back by the population's e_y, e_z
        // (the x-shift is taken by the kernel's loads)
        const long long P = kp.L.P, RP = (long long)(ny + 2) * kp.L.P;
        const int qf = h->qf;
        for (int j = 0; j < h->qf + h->qg; ++j) {
            int ey, ez;
            if (dim == 2) {
                ey = j < qf ? D2Q9::e(j, 1) : D2Q5::e(j - qf, 1);
                ez = 0;
            } else {
                ey = j < qf ? D3Q19::e(j, 1) : D3Q7::e(j - qf, 1);
                ez = j < qf ? D3Q19::e(j, 2) : D3Q7::e(j - qf, 2);
            }
            kp.soff[j] = (int)((long long)j * kp.L.plane);
            kp.loff[j] = (int)((long long)j * kp.L.plane - ey * P - ez * RP);
        }
        kp.plane32 = (int)kp.L.plane;
        kp.rp = (int)RP;
    }
    h->wait_ns = TILE_WAIT_NS;
    h->vec = default_variant(dim, precision).vec;
    h->bx = default_variant(dim, precision).bx;
    h->by = default_variant(dim, precision).by;
    h->rows = default_variant(dim, precision).rows;
    kp.xmax_load = kp.L.P - h->vec;
    kp.gbeta = h->gbeta; kp.omega = h->omega; kp.Th = h->prm.Th; kp.Tc = h->prm.Tc; kp.a_T = h->a_T;
    kp.wTh = kp.omega * kp.Th;
    kp.wTc = kp.omega * kp.Tc;
    for (int a = 0; a < 3; ++a) {
        kp.body[a] = prm.body_force[a];
        kp.bodyf[a] = (float)prm.body_force[a];
    }
    for (int k = 0; k < MAXQ; ++k) {
        const double s = k < h->qf ? h->S[k] : 0.0;
        kp.S[k] = s;
        kp.Sh[k] = 1.0 - 0.5 * s;
        kp.Sf[k] = (float)s;
        kp.Shf[k] = (float)(1.0 - 0.5 * s);
    }
    for (int k = 0; k < 7; ++k) {
        const double q = k < h->qg ? h->Q[k] : 0.0;
        kp.Q[k] = q;
        kp.Qf[k] = (float)q;
    }
    kp.gbetaf = (float)h->gbeta; kp.omegaf = (float)h->omega; kp.Thf = (float)h->prm.Th;
    kp.Tcf = (float)h->prm.Tc; kp.a_Tf = (float)h->a_T;
    double scale = pick(prm.store_scale, precision == TLBM_FP16_OFFSET ? 1024.0 : 1.0);
    if (precision <= TLBM_FP32) scale = 1.0;
    int scale_exp = 0;
    if (!(scale > 0) || std::frexp(scale, &scale_exp) != 0.5) {
        delete h;
        return fail(nullptr, TLBM_ERR_ARG, "store_scale must be a power of two");
    }
    kp.scale = (float)scale;
    kp.inv_scale = (float)(1.0 / scale);
    {
        // FP32 constants of the two-relaxation-time collision (KParams::tf):
        // the in-kernel expressions, one operation per statement, so that the
        // host compiler forms each exactly as the kernel does
        const float sc = kp.scale;
        const int w0i = dim == 2 ? D2Q9::w36(0) : D3Q19::w36(0);
        const int wai = dim == 2 ? D2Q9::w36(1) : D3Q19::w36(1);
        const int wbi = dim == 2 ? D2Q9::w36(D2Q9::Q - 1) : D3Q19::w36(D3Q19::Q - 1);
        const float w0 = (float)w0i / 36.0f, wa = (float)wai / 36.0f, wb = (float)wbi / 36.0f;
        const float sp = kp.spf, sm = kp.smf, shp = kp.shpf, shm = kp.shmf, qp = kp.qpf, qm = kp.qmf;
        auto& t = kp.tf;
        t.m3shp = -3.0f * shp;
        t.r1 = 4.5f * sp;
        t.r3 = 3.0f * sm;
        const float spm = sp + sm;        // (sp + sm) / 2 and (sm - sp) / 2 are exact halvings
        t.c1 = 1.0f - 0.5f * spm;
        const float dsm = sm - sp;
        t.c2 = 0.5f * dsm;
        t.omsp = 1.0f - sp;
        t.w0s = w0 * sc;                  // sc is a power of two: exact
        t.was = wa * sc;
        t.wbs = wb * sc;
        const float s9 = 9.0f * shp, s3 = 3.0f * shm;
        t.f9a = s9 * t.was;
        t.f9b = s9 * t.wbs;
        t.f3a = s3 * t.was;
        t.f3b = s3 * t.wbs;
        const float wT = 0.5f * kp.omegaf;
        const float qpm = qp + qm;
        t.t1 = 1.0f - 0.5f * qpm;
        const float dq = qm - qp;
        t.t2 = 0.5f * dq;
        t.qpwT = qp * wT;
        t.hqm = 0.5f * qm;
        t.omqp = 1.0f - qp;
        const float rest = std::fma(-(float)(h->qg - 1), wT, 1.0f);
        t.g0c = qp * rest;
    }

    {
        // FP64 constants of the two-relaxation-time collision (KParams::td)
        auto& t = kp.td;
        t.hsp = 0.5 * (1.0 - kp.sp);
        t.hsm = 0.5 * (1.0 - kp.sm);
        t.osp = 1.0 - kp.sp;
        t.sp = kp.sp;
        t.k15 = -1.5 * kp.sp;
        t.k6 = -6.0 * kp.shp;
        t.b1 = 4.5 * kp.sp;
        t.b2 = 18.0 * kp.shp;
        t.a1 = 3.0 * kp.sm;
        t.a2 = 6.0 * kp.shm;
        t.hgb = 0.5 * kp.gbeta;
        for (int a = 0; a < 3; ++a) t.hb[a] = 0.5 * kp.body[a];
        const double wT = 0.5 * kp.omega;
        t.hqp = 0.5 * (1.0 - kp.qp);
        t.hqm = 0.5 * (1.0 - kp.qm);
        t.oqp = 1.0 - kp.qp;
        t.qpwT = kp.qp * wT;
        t.hq = 0.5 * kp.qm;
        t.g0c = kp.qp * (1.0 - (h->qg - 1) * wT);
    }

    if ((long long)(h->qf + h->qg) * kp.L.plane + kp.L.P >= (1ll << 31)) {
        delete h;
        return fail(nullptr, TLBM_ERR_ARG, "cell too large: a population set must hold fewer than 2^31 elements");
    }
    h->elem = precision == TLBM_FP64 ? 8 : (precision == TLBM_FP32 ? 4 : 2);
    h->popset_bytes = align_up((size_t)(h->qf + h->qg) * (size_t)kp.L.plane * h->elem, 256);
    h->aa = prm.streaming == TLBM_STREAM_INPLACE;
    h->nbuf = h->aa ? 1 : 2;
    if (h->aa) {
        h->rows = 1;  // the in-place halves have no multi-row variant
        if (dim == 2 && precision == TLBM_FP32) h->by = 1;  // 57.4 vs 56.0 GLUPS with 32 x 4 at 8193^2
    }
    h->red_off = h->nbuf * h->popset_bytes;
    h->res_off = h->red_off + align_up((size_t)RED_ROWS * RED_FIELDS * sizeof(double), 256);
    h->status_off = h->res_off + 128;
    h->stage_off = h->res_off + 256;
    const long long N = (long long)nx * ny * nz;
    h->total_bytes = h->stage_off + align_up((size_t)std::min<long long>(N, STAGE_NODES) * sizeof(double), 256);
    h->stream = nullptr;
    set_cur(h, 0);
    h->t = 0;
    h->graph_steps = 16;
    *out = h;
    return TLBM_OK;
}

extern "C" int tlbm_required_bytes(tlbm_t h, size_t* bytes) {
    TLBM_CHECK_HANDLE(h);
    if (!bytes) return fail(h, TLBM_ERR_ARG, "bytes is NULL");
    *bytes = h->total_bytes;
    return TLBM_OK;
}

extern "C" int tlbm_bind_memory(tlbm_t h, void* dev_ptr, size_t bytes) {
    TLBM_CHECK_HANDLE(h);
    if (!dev_ptr) return fail(h, TLBM_ERR_ARG, "dev_ptr is NULL");
    if (((uintptr_t)dev_ptr) % 256) return fail(h, TLBM_ERR_ARG, "dev_ptr must be 256-byte aligned");
    if (bytes < h->total_bytes)
        return fail(h, TLBM_ERR_OOM, "bound block has %zu bytes, %zu needed", bytes, h->total_bytes);
    cudaPointerAttributes a;
    cudaError_t e = cudaPointerGetAttributes(&a, dev_ptr);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaPointerGetAttributes");
    if (a.type != cudaMemoryTypeDevice && a.type != cudaMemoryTypeManaged)
        return fail(h, TLBM_ERR_ARG, "dev_ptr is not device memory");
    // the staged kernel's status word starts cleared
    e = cudaMemset((char*)dev_ptr + h->status_off, 0, sizeof(int));
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaMemset");
    drop_graph(h);
    h->mem = (char*)dev_ptr;
    h->mem_bytes = bytes;
    h->buf[0] = h->mem;
    h->buf[1] = h->aa ? h->mem : h->mem + h->popset_bytes;
#ifdef TLBM_DEBUG_BOUNDS
    h->kp.dbg_lo = h->mem;
    h->kp.dbg_hi = h->mem + h->nbuf * h->popset_bytes;
    h->kp.dbg_count = (unsigned long long*)(h->mem + h->status_off + 64);
    e = cudaMemset(h->kp.dbg_count, 0, sizeof(unsigned long long));
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaMemset");
#endif
    set_cur(h, 0);
    pick_16bit(h);
    pick_multi(h);
    return TLBM_OK;
}

extern "C" int tlbm_set_stream(tlbm_t h, void* s) {
    TLBM_CHECK_HANDLE(h);
    h->stream = (cudaStream_t)s;
    return TLBM_OK;
}

extern "C" int tlbm_init(tlbm_t h, uint64_t seed, double noise_amp) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    if (!std::isfinite(noise_amp) || noise_amp < 0) return fail(h, TLBM_ERR_ARG, "noise_amp must be finite, >= 0");
    cudaError_t e = cudaMemsetAsync(h->mem, 0, h->nbuf * h->popset_bytes, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaMemsetAsync");
    e = cudaMemsetAsync(h->mem + h->status_off, 0, sizeof(int), h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaMemsetAsync");
    set_cur(h, 0);
    e = with_types(h->dim, h->prec, [&](auto K) { return decltype(K)::init(h->buf[0], h->kp, seed, noise_amp, h->stream); });
    if (e != cudaSuccess) return cuda_fail(h, e, "init kernel");
    h->launches += 1;
    h->t = 0;
    return TLBM_OK;
}

extern "C" int tlbm_init_fields(tlbm_t h, const float* T, const float* ux, const float* uy, const float* uz) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    if (!T) return fail(h, TLBM_ERR_ARG, "T is required");
    cudaError_t e = cudaMemsetAsync(h->mem, 0, h->nbuf * h->popset_bytes, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->mem + h->status_off, 0, sizeof(int), h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaMemsetAsync");
    set_cur(h, 0);
    e = with_types(h->dim, h->prec, [&](auto K) {
        return decltype(K)::init_fields(h->buf[0], h->kp, T, ux, uy, uz, h->stream);
    });
    if (e != cudaSuccess) return cuda_fail(h, e, "init_fields kernel");
    h->launches += 1;
    h->t = 0;
    return TLBM_OK;
}

// Launch one step reading buffer `parity` and writing the other, on stream s
// (no bookkeeping).
static cudaError_t launch_step_raw(tlbm_t h, int parity, cudaStream_t s) {
    const KParams& kp = h->kp;
    const void* src = h->buf[parity];
    void* dst = h->buf[parity ^ 1];
    if (h->staged) {
        StagedInfo si;
        si.tw = h->staged_tw;
        si.tiles_per_row = (h->nx + si.tw - 1) / si.tw;
        si.tiles = h->ny * h->nz * si.tiles_per_row;
        si.stages = h->staged_stages;
        si.status = (int*)(h->mem + h->status_off);
        si.wait_ns = h->wait_ns;
        return launch_staged(h->dim, h->prec, h->staged_nc, src, dst, kp, si, h->staged_grid, h->staged_smem, s);
    }
    if (h->flat) return launch_flat(h->dim, h->prec, h->aa ? (parity ? AA_ODD : AA_EVEN) : PULL, src, h->aa ? h->buf[0] : dst, kp, s);
    const int vec = h->vec;
    const int bx = h->bx, by = h->by, rows = h->rows;
    const int threads_x = (h->nx + vec - 1) / vec;
    dim3 block(bx, by, 1);
    dim3 grid((threads_x + bx - 1) / bx, (h->ny + by * rows - 1) / (by * rows), h->dim == 3 ? h->nz : 1);
    // in place: natural order -> the AA_EVEN half, swapped -> AA_ODD, one buffer
    if (h->aa) return launch_step(h->dim, h->prec, vec, h->trt != 0, parity ? -AA_ODD : -AA_EVEN, src, h->buf[0], kp,
                                  grid, block, s);
    return launch_step(h->dim, h->prec, vec, h->trt != 0, rows, src, dst, kp, grid, block, s);
}

static void drop_graph(tlbm_t h) {
    if (h->graph) {
        cudaGraphExecDestroy(h->graph);
        h->graph = nullptr;
    }
}

constexpr int MULTI_GRAPH = 8;  // launches of a graph block (even: it ends in the buffer it began in)

// Launch `steps` <= h->multi steps (with march: h->multi or 1) reading buffer
// `parity` and writing the other.
static cudaError_t launch_multi_raw(tlbm_t h, int parity, int steps, cudaStream_t s) {
    if (h->march && steps == 1) return launch_step_raw(h, parity, s);
    if (h->march) return launch_march(h->prec, h->buf[parity], h->buf[parity ^ 1], h->kp, h->march, s);
    MultiGeo g = h->mg;
    g.steps = steps;
    return launch_multi(h->prec, h->buf[parity], h->buf[parity ^ 1], h->kp, g, s);
}

// Capture a block of launches starting from buffer 0 into a CUDA graph (on a
// private stream; the graph is replayed on the handle's stream): graph_steps
// single steps, or MULTI_GRAPH launches of several steps.
static int build_graph(tlbm_t h) {
    drop_graph(h);
    cudaError_t e = cudaSuccess;
    if (!h->capture_stream) e = cudaStreamCreateWithFlags(&h->capture_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaStreamCreate");
    e = cudaStreamBeginCapture(h->capture_stream, cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaStreamBeginCapture");
    cudaError_t le = cudaSuccess;
    const int count = h->multi ? MULTI_GRAPH : h->graph_steps;
    for (int k = 0; k < count && le == cudaSuccess; ++k)
        le = h->multi ? launch_multi_raw(h, k & 1, h->multi, h->capture_stream) : launch_step_raw(h, k & 1, h->capture_stream);
    cudaGraph_t g = nullptr;
    e = cudaStreamEndCapture(h->capture_stream, &g);
    if (le != cudaSuccess || e != cudaSuccess) {
        if (g) cudaGraphDestroy(g);
        return cuda_fail(h, le != cudaSuccess ? le : e, "step graph capture");
    }
    e = cudaGraphInstantiate(&h->graph, g, 0);
    cudaGraphDestroy(g);
    if (e != cudaSuccess) {
        h->graph = nullptr;
        return cuda_fail(h, e, "cudaGraphInstantiate");
    }
    return TLBM_OK;
}

static cudaError_t launch_one_step(tlbm_t h) {
    cudaError_t e = launch_step_raw(h, h->cur, h->stream);
    if (e == cudaSuccess) {
        set_cur(h, h->cur ^ 1);
        h->t += 1;
        h->launches += 1;
    }
    return e;
}

// n steps, several per launch: graph blocks, then single launches, the last ones
// of fewer steps.
// The state ends in the buffer that n single steps would leave it in (readers of
// the bound block and batches go by that): up to two single-step launches first
// make the number of launches as odd as n (three steps a launch always are).
static int step_multi(tlbm_t h, int64_t n) {
    const int k = h->multi;
    int ones = 0;
    if (!h->march)
        while ((ones + (n - ones + k - 1) / k - n) % 2) ++ones;
    while (n > 0) {
        if (ones == 0 && h->cur == 0 && n >= (int64_t)k * MULTI_GRAPH) {
            if (!h->graph) {
                int rc = build_graph(h);
                if (rc != TLBM_OK) return rc;
            }
            cudaError_t e = cudaGraphLaunch(h->graph, h->stream);
            if (e != cudaSuccess) return cuda_fail(h, e, "cudaGraphLaunch");
            h->t += (int64_t)k * MULTI_GRAPH;
            h->launches += MULTI_GRAPH;
            n -= (int64_t)k * MULTI_GRAPH;
        } else {
            const int now = ones > 0 ? 1 : (n >= k ? k : (h->march ? 1 : (int)n));
            ones -= ones > 0;
            cudaError_t e = launch_multi_raw(h, h->cur, now, h->stream);
            if (e != cudaSuccess) return cuda_fail(h, e, "step kernel");
            set_cur(h, h->cur ^ 1);
            h->t += now;
            h->launches += 1;
            n -= now;
        }
    }
    return TLBM_OK;
}

extern "C" int tlbm_step(tlbm_t h, int64_t n) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    if (n < 0) return fail(h, TLBM_ERR_ARG, "n must be >= 0");
    if (h->multi && n >= MULTI_CALL) return step_multi(h, n);
    while (n > 0) {
        if (!h->multi && h->graph_steps >= 2 && h->cur == 0 && n >= h->graph_steps) {
            if (!h->graph) {
                int rc = build_graph(h);
                if (rc != TLBM_OK) return rc;
            }
            cudaError_t e = cudaGraphLaunch(h->graph, h->stream);
            if (e != cudaSuccess) return cuda_fail(h, e, "cudaGraphLaunch");
            h->t += h->graph_steps;  // an even number of steps: the state is back in buffer 0
            h->launches += h->graph_steps;
            n -= h->graph_steps;
        } else {
            cudaError_t e = launch_one_step(h);
            if (e != cudaSuccess) return cuda_fail(h, e, "step kernel");
            n -= 1;
        }
    }
    return TLBM_OK;
}

extern "C" int tlbm_set_graph(tlbm_t h, int steps) {
    TLBM_CHECK_HANDLE(h);
    if (steps < 0 || steps % 2 || steps > 4096) return fail(h, TLBM_ERR_ARG, "steps must be even, in [0, 4096]");
    drop_graph(h);
    h->graph_steps = steps;
    h->graph_chosen = 1;  // the caller chose how single steps are launched
    h->multi = 0;
    return TLBM_OK;
}

extern "C" int tlbm_macros(tlbm_t h, void* rho, void* ux, void* uy, void* uz, void* T, int out_dtype) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    if (out_dtype != TLBM_OUT_F64 && out_dtype != TLBM_OUT_F32) return fail(h, TLBM_ERR_ARG, "bad out_dtype");
    if (h->dim == 2) uz = nullptr;
    cudaError_t e = launch_macros(h->dim, h->prec, h->buf[h->cur], h->kp, rho, ux, uy, uz, T,
                                  out_dtype == TLBM_OUT_F64, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "macros kernel");
    h->launches += 1;
    return TLBM_OK;
}

// the reduction's view of a handle's current state (parameters by value)
static RedState red_state(tlbm_t h) {
    return {h->buf[h->cur], nullptr, (double*)(h->mem + h->red_off), (const int*)(h->mem + h->status_off), 0, 0, false};
}

// runs the two-pass reduction and copies the six results to the host
static int run_reduce(tlbm_t h, double* res) {
    double* out = (double*)(h->mem + h->res_off);
    RedStates st;
    st.s[0] = red_state(h);
    const KParams* kp = &h->kp;
    cudaError_t e = launch_reduce(h->dim, h->prec, st, 1, &kp, out, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "reduction kernel");
    h->launches += 2;
    double r[8];
    e = cudaMemcpyAsync(r, out, sizeof(r), cudaMemcpyDeviceToHost, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaMemcpyAsync");
    e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaStreamSynchronize");
    memcpy(res, r, RED_FIELDS * sizeof(double));
    if (r[6] != 0.0) return fail(h, TLBM_ERR_TIMEOUT, "a staged step gave up waiting for its copies");
    return TLBM_OK;
}

// the reduction found a non-finite value or |u| > 0.5 (|u|^2 > 0.25)
static bool reduce_diverged(const double* r) { return r[4] != 0.0 || !(r[3] <= 0.25); }

static double nusselt_of(tlbm_t h, const double* r) {
    const double N = (double)h->nx * h->ny * h->nz;
    const int ax = h->kp.heat_axis;
    const double L = ax == 0 ? h->nx : (ax == 1 ? h->ny : h->nz);
    return 1.0 + L * (r[0] / N) / (h->alpha * (h->prm.Th - h->prm.Tc));
}

// The reductions of n bound two-buffer handles of one lattice and storage whose
// work is all on `stream`, RED_MANY at a time in two launches and one copy (a
// reduction on its own costs about 20 us of launches, copy and wait whatever
// its size).  d_kp[i]: handle i's parameters in device memory.  nu (may be
// null) and diverged as tlbm_nusselt and tlbm_status give them.
int tlbm::reduce_many(tlbm_t* hs, int n, const KParams* d_kp, cudaStream_t stream, double* nu, int* diverged,
                      int* failed) {
    for (int i0 = 0; i0 < n; i0 += RED_MANY) {
        const int count = std::min(RED_MANY, n - i0);
        RedStates st;
        const KParams* kp[RED_MANY];
        for (int i = 0; i < count; ++i) {
            st.s[i] = red_state(hs[i0 + i]);
            st.s[i].kp = d_kp + i0 + i;
            kp[i] = &hs[i0 + i]->kp;
        }
        // results behind the first handle's partials
        static_assert((RED_ROWS - RED_BLOCKS) * RED_FIELDS >= 8 * RED_MANY, "scratch of the results");
        tlbm_t h = hs[i0];
        double* out = (double*)(h->mem + h->red_off) + RED_BLOCKS * RED_FIELDS;
        double r[8 * RED_MANY];
        cudaError_t e = launch_reduce(h->dim, h->prec, st, count, kp, out, stream);
        if (e == cudaSuccess) e = cudaMemcpyAsync(r, out, count * 8 * sizeof(double), cudaMemcpyDeviceToHost, stream);
        if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
        *failed = i0;
        if (e != cudaSuccess) return cuda_fail(h, e, "reduction");
        h->launches += 2;
        for (int i = 0; i < count; ++i) {
            tlbm_t q = hs[i0 + i];
            const double* v = r + 8 * i;
            *failed = i0 + i;
            q->err[0] = 0;
            if (v[6] != 0.0) return fail(q, TLBM_ERR_TIMEOUT, "a staged step gave up waiting for its copies");
            diverged[i0 + i] = reduce_diverged(v) ? 1 : 0;
            if (nu) {
                nu[i0 + i] = nusselt_of(q, v);
                if (diverged[i0 + i]) fail(q, TLBM_ERR_DIVERGED, "the state has diverged (the value is written)");
            }
        }
    }
    return TLBM_OK;
}

extern "C" int tlbm_nusselt(tlbm_t h, double* nu) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    if (!nu) return fail(h, TLBM_ERR_ARG, "nu is NULL");
    double r[RED_FIELDS];
    int rc = run_reduce(h, r);
    if (rc) return rc;
    *nu = nusselt_of(h, r);
    if (reduce_diverged(r)) return fail(h, TLBM_ERR_DIVERGED, "the state has diverged (the value is written)");
    return TLBM_OK;
}

extern "C" int tlbm_energy(tlbm_t h, double* ekin, double* mass) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    double r[RED_FIELDS];
    int rc = run_reduce(h, r);
    if (rc) return rc;
    if (ekin) *ekin = r[1];
    if (mass) *mass = r[2];
    if (reduce_diverged(r)) return fail(h, TLBM_ERR_DIVERGED, "the state has diverged (the values are written)");
    return TLBM_OK;
}

extern "C" int tlbm_status(tlbm_t h, int* diverged, int64_t* step) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    double r[RED_FIELDS];
    int rc = run_reduce(h, r);
    if (rc) return rc;
    if (diverged) *diverged = reduce_diverged(r) ? 1 : 0;
    if (step) *step = h->t;
    return TLBM_OK;
}

static int get_window(tlbm_t h, const Window& w, double* host_f, double* host_g) {
    const long long N = (long long)w.wx * w.wy * w.wz;
    double* stage = (double*)(h->mem + h->stage_off);
    for (int pop = 0; pop < h->qf + h->qg; ++pop) {
        double* dst = pop < h->qf ? (host_f ? host_f + (long long)pop * N : nullptr)
                                  : (host_g ? host_g + (long long)(pop - h->qf) * N : nullptr);
        if (!dst) continue;
        for (long long n0 = 0; n0 < N; n0 += STAGE_NODES) {
            const long long cnt = std::min(STAGE_NODES, N - n0);
            cudaError_t e = with_types(h->dim, h->prec, [&](auto K) {
                return decltype(K)::gather(h->buf[h->cur], stage, pop, n0, cnt, w, h->kp, h->stream);
            });
            if (e != cudaSuccess) return cuda_fail(h, e, "gather kernel");
            h->launches += 1;
            e = cudaMemcpyAsync(dst + n0, stage, cnt * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
            if (e != cudaSuccess) return cuda_fail(h, e, "cudaMemcpyAsync D2H");
            e = cudaStreamSynchronize(h->stream);
            if (e != cudaSuccess) return cuda_fail(h, e, "cudaStreamSynchronize");
        }
    }
    return TLBM_OK;
}

extern "C" int tlbm_get_populations(tlbm_t h, double* host_f, double* host_g) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    const Window w = {0, 0, 0, h->nx, h->ny, h->nz};
    return get_window(h, w, host_f, host_g);
}

extern "C" int tlbm_get_populations_window(tlbm_t h, int x0, int y0, int z0, int wx, int wy, int wz,
                                           double* host_f, double* host_g) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    if (h->dim == 2) {
        z0 = 0;
        wz = 1;
    }
    if (x0 < 0 || y0 < 0 || z0 < 0 || wx < 1 || wy < 1 || wz < 1 || x0 + wx > h->nx || y0 + wy > h->ny ||
        z0 + wz > h->nz)
        return fail(h, TLBM_ERR_ARG, "window out of the cell");
    const Window w = {x0, y0, z0, wx, wy, wz};
    return get_window(h, w, host_f, host_g);
}

// Replace the state by FP64 populations delivered chunk by chunk: src(pop, n0,
// cnt, chunk) points chunk at nodes n0 .. n0 + cnt of population pop (flow
// planes first) and returns TLBM_OK or an error code.  reuse: src hands out
// one host buffer again and again, so each chunk's copy must finish before the
// next call.  Synchronises.
template <class Src>
static int put_state(tlbm_t h, Src src, bool reuse, bool dev = false) {
    const long long N = (long long)h->nx * h->ny * h->nz;
    const Window full = {0, 0, 0, h->nx, h->ny, h->nz};
    double* stage = (double*)(h->mem + h->stage_off);
    cudaError_t e = cudaMemsetAsync(h->mem, 0, h->nbuf * h->popset_bytes, h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaMemsetAsync");
    e = cudaMemsetAsync(h->mem + h->status_off, 0, sizeof(int), h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaMemsetAsync");
    set_cur(h, 0);
    for (int pop = 0; pop < h->qf + h->qg; ++pop) {
        for (long long n0 = 0; n0 < N; n0 += STAGE_NODES) {
            const long long cnt = std::min(STAGE_NODES, N - n0);
            const double* chunk = nullptr;
            const int rc = src(pop, n0, cnt, chunk);
            if (rc != TLBM_OK) return rc;
            e = cudaMemcpyAsync(stage, chunk, cnt * sizeof(double), cudaMemcpyHostToDevice, h->stream);
            if (e != cudaSuccess) return cuda_fail(h, e, "cudaMemcpyAsync H2D");
            e = with_types(h->dim, h->prec, [&](auto K) {
                return decltype(K)::scatter(h->buf[0], stage, pop, n0, cnt, full, h->kp, h->stream, dev);
            });
            if (e != cudaSuccess) return cuda_fail(h, e, "scatter kernel");
            h->launches += 1;
            if (reuse) {
                e = cudaStreamSynchronize(h->stream);
                if (e != cudaSuccess) return cuda_fail(h, e, "cudaStreamSynchronize");
            }
        }
    }
    e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaStreamSynchronize");
    h->t = 0;
    return TLBM_OK;
}

extern "C" int tlbm_set_populations(tlbm_t h, const double* host_f, const double* host_g) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    if (!host_f || !host_g) return fail(h, TLBM_ERR_ARG, "host_f and host_g are required");
    const long long N = (long long)h->nx * h->ny * h->nz;
    return put_state(h, [&](int pop, long long n0, long long, const double*& chunk) {
        chunk = (pop < h->qf ? host_f + (long long)pop * N : host_g + (long long)(pop - h->qf) * N) + n0;
        return (int)TLBM_OK;
    }, false);
}

// ------------------------------------------------------------------ checkpoint files

namespace {
// File header of tlbm_save: native byte order, checked by `order`.
struct CkptHeader {
    char magic[8];          // "TLBMCKP1"
    uint32_t order;         // 0x01020304 as written
    int32_t version;        // 1
    int32_t lattice, nx, ny, nz, precision, walls, periodic_mask, nderived;
    int32_t flow_dev;       // 1: flow planes hold f_i - w_i (offset storage), 0: f_i
    int32_t pad;
    double Ra, Pr, Ma, Th, Tc, scale;
    double body[3];
    double derived[7 + MAXQ + 7];  // tlbm_derived: U, H, nu, alpha, gbeta, a_T, omega, S, Q
    int64_t t;              // steps taken since the initial state
    int64_t nodes;          // nx * ny * nz
};
}  // namespace

static void ckpt_fill(tlbm_t h, CkptHeader& c) {
    memset(&c, 0, sizeof(c));
    memcpy(c.magic, "TLBMCKP1", 8);
    c.order = 0x01020304u;
    c.version = 1;
    c.lattice = h->lattice;
    c.nx = h->nx;
    c.ny = h->ny;
    c.nz = h->nz;
    c.precision = h->prec;
    c.walls = h->prm.walls;
    c.periodic_mask = h->prm.periodic_mask;
    c.Ra = h->Ra;
    c.Pr = h->Pr;
    c.Ma = h->Ma;
    c.Th = h->prm.Th;
    c.Tc = h->prm.Tc;
    c.scale = h->kp.scale;
    for (int a = 0; a < 3; ++a) c.body[a] = h->prm.body_force[a];
    int n = 0;
    tlbm_derived(h, c.derived, 7 + MAXQ + 7, &n);
    c.nderived = n;
    c.flow_dev = h->prec == TLBM_FP64 ? 0 : 1;  // offset storage (FP32, FP16, BF16)
    c.t = h->t;
    c.nodes = (int64_t)h->nx * h->ny * h->nz;
}

extern "C" int tlbm_save(tlbm_t h, const char* path) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    if (!path) return fail(h, TLBM_ERR_ARG, "path is NULL");
    FILE* fp = fopen(path, "wb");
    if (!fp) return fail(h, TLBM_ERR_ARG, "cannot open %s for writing", path);
    CkptHeader c;
    ckpt_fill(h, c);
    int rc = TLBM_OK;
    if (fwrite(&c, sizeof(c), 1, fp) != 1) rc = fail(h, TLBM_ERR_ARG, "write to %s failed", path);
    const long long N = c.nodes;
    const Window full = {0, 0, 0, h->nx, h->ny, h->nz};
    double* stage = (double*)(h->mem + h->stage_off);
    double* buf = rc == TLBM_OK ? (double*)malloc((size_t)std::min(STAGE_NODES, N) * sizeof(double)) : nullptr;
    if (rc == TLBM_OK && !buf) rc = fail(h, TLBM_ERR_OOM, "host buffer");
    for (int pop = 0; rc == TLBM_OK && pop < h->qf + h->qg; ++pop) {
        for (long long n0 = 0; rc == TLBM_OK && n0 < N; n0 += STAGE_NODES) {
            const long long cnt = std::min(STAGE_NODES, N - n0);
            cudaError_t e = with_types(h->dim, h->prec, [&](auto K) {
                return decltype(K)::gather(h->buf[h->cur], stage, pop, n0, cnt, full, h->kp, h->stream, true);
            });
            h->launches += 1;
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(buf, stage, cnt * sizeof(double), cudaMemcpyDeviceToHost, h->stream);
            if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
            if (e != cudaSuccess) rc = cuda_fail(h, e, "checkpoint gather");
            else if (fwrite(buf, sizeof(double), (size_t)cnt, fp) != (size_t)cnt)
                rc = fail(h, TLBM_ERR_ARG, "write to %s failed", path);
        }
    }
    free(buf);
    if (fclose(fp) != 0 && rc == TLBM_OK) rc = fail(h, TLBM_ERR_ARG, "closing %s failed", path);
    return rc;
}

extern "C" int tlbm_load(tlbm_t h, const char* path) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    if (!path) return fail(h, TLBM_ERR_ARG, "path is NULL");
    FILE* fp = fopen(path, "rb");
    if (!fp) return fail(h, TLBM_ERR_ARG, "cannot open %s", path);
    CkptHeader c, mine;
    ckpt_fill(h, mine);
    int rc = TLBM_OK;
    if (fread(&c, sizeof(c), 1, fp) != 1 || memcmp(c.magic, "TLBMCKP1", 8) != 0 || c.order != 0x01020304u ||
        c.version != 1)
        rc = fail(h, TLBM_ERR_ARG, "%s is not a checkpoint of this format", path);
    else if (c.lattice != mine.lattice || c.nx != mine.nx || c.ny != mine.ny || c.nz != mine.nz ||
             c.precision != mine.precision)
        rc = fail(h, TLBM_ERR_ARG, "checkpoint lattice / size / storage differ from the handle's");
    else if (c.walls != mine.walls || c.periodic_mask != mine.periodic_mask || c.nderived != mine.nderived ||
             c.flow_dev != mine.flow_dev ||
             memcmp(&c.Ra, &mine.Ra, offsetof(CkptHeader, t) - offsetof(CkptHeader, Ra)) != 0)
        rc = fail(h, TLBM_ERR_ARG, "checkpoint parameters differ from the handle's");
    const long long N = c.nodes;
    double* buf = rc == TLBM_OK ? (double*)malloc((size_t)std::min(STAGE_NODES, N) * sizeof(double)) : nullptr;
    if (rc == TLBM_OK && !buf) rc = fail(h, TLBM_ERR_OOM, "host buffer");
    if (rc == TLBM_OK) {
        rc = put_state(h, [&](int, long long, long long cnt, const double*& chunk) {
            if (fread(buf, sizeof(double), (size_t)cnt, fp) != (size_t)cnt)
                return fail(h, TLBM_ERR_ARG, "%s is shorter than its header says", path);
            chunk = buf;
            return (int)TLBM_OK;
        }, true, true);
        if (rc == TLBM_OK) {
            char extra;
            if (fread(&extra, 1, 1, fp) != 0) rc = fail(h, TLBM_ERR_ARG, "%s is longer than its header says", path);
        }
        if (rc == TLBM_OK) {
            h->t = c.t;
            // 16-bit storage: the step counter the time steps keep in word 0 of
            // the current buffer (their stochastic rounding salt), as the
            // uninterrupted run had it
            if (h->elem == 2) {
                const uint32_t t32 = (uint32_t)c.t;
                cudaError_t e = cudaMemcpyAsync(h->buf[0], &t32, sizeof(t32), cudaMemcpyHostToDevice, h->stream);
                if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
                if (e != cudaSuccess) rc = cuda_fail(h, e, "cudaMemcpyAsync (step counter)");
            }
        }
    }
    free(buf);
    fclose(fp);
    return rc;
}

extern "C" int tlbm_set_variant(tlbm_t h, int vec, int form, int block_x, int block_y, int rows) {
    TLBM_CHECK_HANDLE(h);
    const int v = vec > 0 ? vec : default_vec(h->dim, h->prec);
    if (form < 0 || form > 2) return fail(h, TLBM_ERR_ARG, "form must be 0 (auto), 1 (MRT) or 2 (TRT)");
    if (form == 2 && !h->kp.trt)
        return fail(h, TLBM_ERR_ARG, "the relaxation rates are not of two-relaxation-time form");
    const int trt = form == 1 ? 0 : h->kp.trt;
    const int bx = block_x > 0 ? block_x : default_variant(h->dim, h->prec).bx;
    const int by = block_y > 0 ? block_y : default_variant(h->dim, h->prec).by;
    if (bx % 32 || bx * by > 1024) return fail(h, TLBM_ERR_ARG, "block_x must be a multiple of 32, bx*by <= 1024");
    const int nr = rows > 0 ? rows : 1;
    if (h->aa && nr != 1) return fail(h, TLBM_ERR_UNSUPPORTED, "in-place streaming has no multi-row variant");
    // the in-place scheme alternates two kernels; both must exist
    const int kinds[2] = {h->aa ? -AA_EVEN : nr, h->aa ? -AA_ODD : nr};
    for (int kind : kinds) {
        if (!step_variant_available(h->dim, h->prec, v, trt != 0, kind))
            return fail(h, TLBM_ERR_UNSUPPORTED, "step variant (vec %d, %s, %d rows%s) not built", v,
                        trt ? "TRT" : "MRT", nr, h->aa ? ", in place" : "");
        cudaFuncAttributes fa;
        cudaError_t e = cudaFuncGetAttributes(&fa, step_function(h->dim, h->prec, v, trt != 0, kind));
        if (e != cudaSuccess) return cuda_fail(h, e, "cudaFuncGetAttributes");
        if (bx * by > fa.maxThreadsPerBlock)
            return fail(h, TLBM_ERR_ARG, "block of %d threads exceeds the variant's limit of %d", bx * by,
                        fa.maxThreadsPerBlock);
    }
    h->vec = v;
    h->trt = trt;
    h->bx = bx;
    h->by = by;
    h->rows = nr;
    h->staged = 0;
    h->flat = 0;
    h->multi = 0;
    h->kp.xmax_load = h->kp.L.P - v;
    if (vec > 0 || form > 0 || block_x > 0 || block_y > 0 || rows > 0) {
        h->variant_chosen = 2;
    } else {
        // every argument 0: the library's choice among the register kernels
        h->variant_chosen = 1;
        h->flat = flat_fp64(h);
        pick_16bit(h);
        pick_multi(h);
    }
    drop_graph(h);
    return TLBM_OK;
}

static int set_staged(tlbm_t h, int tile_width, int stages) {
    if (h->aa) return fail(h, TLBM_ERR_UNSUPPORTED, "the staged kernel uses two buffers (no in-place variant)");
    if (h->prec == TLBM_FP64) return fail(h, TLBM_ERR_UNSUPPORTED, "the staged kernel has no FP64 variant");
    if (!h->kp.trt) return fail(h, TLBM_ERR_UNSUPPORTED, "the staged kernel needs two-relaxation-time rates");
    const int A = 16 / (int)h->elem;
    const int nx_a = (h->nx + A - 1) / A * A;
    // default: whole rows up to the widest tile (512 nodes in 2D, 448 in 3D),
    // else segments of that width
    const int twmax = h->dim == 3 ? 448 : 512;
    int tw = tile_width > 0 ? tile_width : std::min(twmax, nx_a);
    if (tw % A || tw < A || tw > twmax)
        return fail(h, TLBM_ERR_ARG, "tile_width must be a multiple of %d in [%d, %d]", A, A, twmax);
    if (tw > nx_a) tw = nx_a;
    // consumer warps (one pair of nodes per thread): 4 for tiles up to 256
    // nodes, else 8 in 2D and 7 in 3D
    const int nc = tw > 256 ? (h->dim == 3 ? 7 : 8) : 4;
    const int lw = 64 * nc + 2 * A;   // shared row length per population (elements)
    const size_t stage_bytes = (size_t)(h->qf + h->qg) * lw * h->elem;
    const void* fn = staged_function(h->dim, h->prec, nc);
    if (!fn) return fail(h, TLBM_ERR_UNSUPPORTED, "staged kernel not built for this precision");
    int dev = 0, optin = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaDeviceGetAttribute");
    // allow the device's full opt-in shared memory for this kernel, so that
    // handles with different tile shapes can share it
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaFuncSetAttribute (shared memory size)");
    const int threads = 32 * (nc + 1);
    int ns = stages;
    if (ns <= 0) {
        // the most tiles in flight per SM (blocks per SM x stages) up to six,
        // more blocks first (else the fewest stages that fit): on GB300 2 x 3
        // was best for 96-register consumers, 3 x 2 for 72-register ones, and
        // more in flight was slower
        int first = 0, best_in = 0, best_b = 0;
        for (int k = 2; k <= TILE_MAX_STAGES; ++k) {
            int b = 0;
            const size_t sm = 512 + (size_t)k * stage_bytes;
            if (sm > (size_t)optin) break;
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, fn, threads, sm);
            if (e != cudaSuccess) return cuda_fail(h, e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
            if (b < 1) break;
            if (!first) first = k;
            const int in = b * k;
            if (in <= 6 && (in > best_in || (in == best_in && b > best_b))) {
                ns = k;
                best_in = in;
                best_b = b;
            }
        }
        if (ns == 0) ns = first;
        if (ns == 0) return fail(h, TLBM_ERR_ARG, "two stages of %zu bytes do not fit in shared memory", stage_bytes);
    }
    if (ns < 2 || ns > TILE_MAX_STAGES) return fail(h, TLBM_ERR_ARG, "stages must be in [2, %d]", TILE_MAX_STAGES);
    const size_t smem = 512 + (size_t)ns * stage_bytes;
    if (smem > (size_t)optin) return fail(h, TLBM_ERR_ARG, "%zu bytes of shared memory per block exceed %d", smem, optin);
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, threads, smem);
    if (e != cudaSuccess) return cuda_fail(h, e, "cudaOccupancyMaxActiveBlocksPerMultiprocessor");
    if (per_sm < 1) return fail(h, TLBM_ERR_ARG, "%zu bytes of shared memory per block do not fit", smem);
    const long long tiles = (long long)h->ny * h->nz * ((h->nx + tw - 1) / tw);
    if (tiles >= (1ll << 31)) return fail(h, TLBM_ERR_ARG, "too many tiles for the staged kernel");
    h->staged = 1;
    h->staged_tw = tw;
    h->staged_nc = nc;
    h->staged_stages = ns;
    h->staged_smem = smem;
    h->staged_grid = (int)std::min<long long>(tiles, (long long)per_sm * sms);
    drop_graph(h);
    return TLBM_OK;
}

// Step kernel of an FP16 or BF16 cell with two-relaxation-time rates whose
// launches the caller has not chosen.
// 2D, two buffers: the staged kernel, 512-node tiles with the stages chosen as
// above (2 stages and three blocks per SM on GB300, the fastest there).
// 3D, two buffers: the staged kernel (2 stages, two blocks per SM) takes a row per
// tile and seven warps, so it is for rows that nearly fill those.  us per step,
// staged and node pairs in rows: 385^3 1110 and 1283, 448 x 385^2 1160 and 1305, 385 x
// 129^2 133 and 150, 416 x 129^2 134 and 150, 448 x 129^2 137 and 153; at the border 384
// x 129^2 136 and 132, 383 x 129^2 143 and 141, 449 x 129^2 254 and 170; 321^3 782 and
// 791, 193^3 208 and 193, 65^3 26 and 14.  (Cells too small to fill the GPU lose: 385 x
// 33^2 15.5 and 12.7.)  Else warps inside rows: one node a thread up to 4 M nodes,
// where a second one in flight per thread is worth less than twice the warps, then
// node pairs (one node and pairs: 33^3 5.0 and 6.4, 65^3 13.0 and 14.0, 145^3 95 and
// 94, 161^3 129 and 116; between, 97^3 36 and 34, 129^3 75 and 72).
// 3D, in place: one thread per node in memory order for small cells and where
// pairs leave over 1/16 of a row's last warps idle (step_3d_f16.cu).  With none
// idle it was pairs' gain before the wall rules went face by face (192^3 196 us
// against 206, 320^3 821 and 919).
static void pick_16bit(tlbm_t h) {
    if (h->elem != 2 || !h->kp.trt || h->variant_chosen > 1) return;
    const double nodes = (double)h->nx * h->ny * h->nz;
    const long long lanes = (h->nx + 63) / 64 * 64ll;
    if (h->aa) {
        h->flat = h->dim == 3 && nodes <= FLAT_NODES && (nodes <= 4e6 || 16ll * h->nx < 15 * lanes);
        return;
    }
    if (!h->variant_chosen && (h->dim == 2 || (h->nx >= 384 && h->nx <= 448))) {
        // (the register kernel stays if the device cannot host the staged one)
        if (set_staged(h, 0, h->dim == 3 ? 2 : 0) == TLBM_OK) return;
        h->staged = 0;
        h->err[0] = 0;
    }
    if (h->dim == 3 && nodes <= 4e6) {
        h->vec = 1;
        h->bx = 32;
        h->by = 2;
        h->kp.xmax_load = h->kp.L.P - 1;
    }
}

// Several steps per launch: 2D two-buffer cells with two-relaxation-time rates
// whose launches the caller has not chosen.  FP32 and 16-bit cells with walls all
// around go through step_march.cu from 250,000 / 270,000 nodes unless their width
// would leave more than a quarter of its strips' columns idle (513^2 when the line
// was drawn, FP32: 6.7 us per step, 7.1 in tiles, 10.5 singly; FP16: 7.6, 7.4 and
// 12.3; now 5.7 against 7.4 singly and 6.8 against 8.9).  Else tiles
// (step_multi.cu) up to the size where one step fills the GPU.  FP32, FP16 and BF16:
// 300,000 nodes (a 513^2 cell gains 1.5x, a 1025^2 one 1.1x in FP32 and loses a
// quarter in FP16), the 16-bit ones not with rows of over 2048 nodes, which suit
// the staged kernel's tiles (4000 x 70: 8.5 us per step staged, 8.8 here); FP64,
// bound by its pipe, 30,000 (65^2 6.9 -> 5.4 us against one thread per node, 129^2
// 7.0 and 7.2, 193^2 12.2 both ways).
static void pick_multi(tlbm_t h) {
    h->multi = h->march = 0;
    if (h->dim != 2 || h->aa || !h->kp.trt || h->variant_chosen > 1 || h->graph_chosen) return;
    const long long nodes = (long long)h->nx * h->ny;
    const int strips = (h->nx + MARCH_COLUMNS - 1) / MARCH_COLUMNS;
    if (h->prec != TLBM_FP64 && !h->kp.periodic && nodes >= (h->prec == TLBM_FP32 ? 250000 : 270000) && 4 * h->nx >= 3 * strips * MARCH_COLUMNS) {
        h->march = march_rows(h->prec, h->kp);
        if (h->march) h->multi = MARCH_STEPS;
        return;
    }
    if (nodes > (h->prec == TLBM_FP64 ? 30000 : 300000)) return;
    if (h->elem == 2 && h->nx > 2048) return;
    // a region wraps around a periodic axis at most once
    if (((h->kp.periodic & 1) && h->nx < 16) || ((h->kp.periodic & 2) && h->ny < 16)) return;
    if (multi_setup(h->prec, h->kp, h->mg)) h->multi = h->mg.m + 1;
}

extern "C" int tlbm_set_staged(tlbm_t h, int tile_width, int stages) {
    TLBM_CHECK_HANDLE(h);
    const int rc = set_staged(h, tile_width, stages);
    if (rc == TLBM_OK) {
        h->variant_chosen = 2;
        h->multi = 0;
    }
    return rc;
}

extern "C" int tlbm_set_wait_limit(tlbm_t h, double seconds) {
    TLBM_CHECK_HANDLE(h);
    if (!(seconds >= 0.0 && seconds <= 10.0)) return fail(h, TLBM_ERR_ARG, "seconds must be in [0, 10]");
    h->wait_ns = (unsigned long long)(seconds * 1e9);
    drop_graph(h);
    return TLBM_OK;
}

extern "C" int tlbm_get_staged(tlbm_t h, int* tile_width, int* stages, int* blocks) {
    TLBM_CHECK_HANDLE(h);
    if (tile_width) *tile_width = h->staged ? h->staged_tw : 0;
    if (stages) *stages = h->staged ? h->staged_stages : 0;
    if (blocks) *blocks = h->staged ? h->staged_grid : 0;
    return TLBM_OK;
}

extern "C" int tlbm_get_variant(tlbm_t h, int* vec, int* form, int* block_x, int* block_y, int* rows) {
    TLBM_CHECK_HANDLE(h);
    if (rows) *rows = h->rows;
    if (vec) *vec = h->staged ? 0 : h->vec;
    if (form) *form = h->trt ? 2 : 1;
    if (block_x) *block_x = h->bx;
    if (block_y) *block_y = h->by;
    return TLBM_OK;
}

extern "C" int tlbm_derived(tlbm_t h, double* out, int cap, int* count) {
    TLBM_CHECK_HANDLE(h);
    if (!out && cap > 0) return fail(h, TLBM_ERR_ARG, "out is NULL");
    double v[7 + MAXQ + 7];
    int n = 0;
    v[n++] = h->U; v[n++] = h->H; v[n++] = h->nu; v[n++] = h->alpha;
    v[n++] = h->gbeta; v[n++] = h->a_T; v[n++] = h->omega;
    for (int k = 0; k < h->qf; ++k) v[n++] = h->S[k];
    for (int k = 0; k < h->qg; ++k) v[n++] = h->Q[k];
    for (int i = 0; i < n && i < cap; ++i) out[i] = v[i];
    if (count) *count = n < cap ? n : cap;
    return TLBM_OK;
}

extern "C" int tlbm_bounds_violations(tlbm_t h, int64_t* count) {
    TLBM_CHECK_HANDLE(h);
    TLBM_CHECK_BOUND(h);
    if (!count) return fail(h, TLBM_ERR_ARG, "count is NULL");
#ifdef TLBM_DEBUG_BOUNDS
    unsigned long long c = 0;
    cudaError_t e = cudaMemcpyAsync(&c, h->kp.dbg_count, sizeof(c), cudaMemcpyDeviceToHost, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) return cuda_fail(h, e, "reading the violation counter");
    *count = (int64_t)c;
    return TLBM_OK;
#else
    *count = 0;
    return fail(h, TLBM_ERR_UNSUPPORTED, "this library is built without bounds checks (TLBM_DEBUG_BOUNDS)");
#endif
}

extern "C" const char* tlbm_last_error(tlbm_t h) { return h ? h->err : g_create_error; }

extern "C" int tlbm_launch_count(tlbm_t h, int64_t* count) {
    TLBM_CHECK_HANDLE(h);
    if (!count) return fail(h, TLBM_ERR_ARG, "count is NULL");
    *count = h->launches;
    return TLBM_OK;
}

extern "C" void tlbm_destroy(tlbm_t h) {
    if (!h) return;
    drop_graph(h);
    if (h->capture_stream) cudaStreamDestroy(h->capture_stream);
    delete h;
}
