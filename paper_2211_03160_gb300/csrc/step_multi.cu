// Several time steps of a 2D cell in one launch, for cells too small to fill the
// GPU with one step (two-relaxation-time collision, two-buffer streaming).
//
// A block owns a tile of the cell and steps a region that is wider than it by
// K - 1 nodes on every side.  Step 1 pulls the region's populations from global
// memory; after every step but the last the post-collision values go to shared
// memory, where the next step pulls them, and the region that is still correct
// shrinks by one node a side; the last step stores the tile.  Nothing is
// exchanged between blocks inside a launch, the nodes around a tile are stepped
// by its neighbours as well.
//
// What bounds it: a one-step launch of such a cell costs 6 to 20 us, nearly all
// of it launch, instruction fetch and one pass through memory latency.  K steps a
// launch pay that once and run the collision from a warm instruction cache, for
// the price of (1 + 2 (K - 1) / tile)^2 redundant updates.  us per step on GB300,
// one-step launches in a CUDA graph -> this kernel: FP32 65^2 5.1 -> 1.7, 129^2
// 4.8 -> 1.9, 257^2 4.8 -> 2.4; FP16 129^2 4.5 -> 2.2, 257^2 4.9 -> 2.7, 500^2 8.7 ->
// 6.5; FP64, whose pipe the redundant updates keep busy, 65^2 6.9 -> 5.4 and 129^2
// 7.0 and 7.2.  (Launching the next block of steps early, with
// programmatic stream serialization, gained at most 2 % and lost 20 % in FP64.)
//
// Every node gets bitwise the values of the one-step kernels: the same
// collision, wall rules and storage rounding (values in shared memory are in
// the storage type), with the step counter's salt of its own step.
#include <algorithm>

#include "dispatch.h"

namespace tlbm {

namespace {

template <class S>
struct Multi {
    static constexpr int VEC = sizeof(S) == 8 ? 1 : 2;         // nodes per thread
    static constexpr int THREADS = sizeof(S) == 8 ? 256 : 512;  // most threads of a block
    static constexpr int PAD = 16;                              // elements before and after the planes
};

// Place of region node (r, x) in a shared plane with rows of RS elements.
// Populations that move along x are pulled by a thread's node pair as two values
// of different alignment; FP32 keeps those planes' even and odd columns apart,
// so that a warp's loads fall on neighbouring words.
template <class S, int EX>
__device__ __forceinline__ int multi_at(int r, int x, int RS) {
    if constexpr (sizeof(S) == 4 && EX != 0) return r * RS + (x & 1) * (RS >> 1) + (x >> 1);
    else return r * RS + x;
}

// A thread's VEC values of one population, written to or pulled from (at
// columns x - EX) its shared plane.
template <class S, int VEC, int EX>
__device__ __forceinline__ void multi_put(S* pl, int r, int x, int RS, const S (&v)[VEC], const bool (&in)[VEC]) {
    if constexpr (VEC == 2 && (EX == 0 || sizeof(S) == 2)) {
        if (in[0] && in[1]) {
            using W = typename std::conditional<sizeof(S) == 2, uint32_t, float2>::type;
            W w;
            memcpy(&w, v, sizeof(W));
            *reinterpret_cast<W*>(pl + r * RS + x) = w;
            return;
        }
    }
#pragma unroll
    for (int k = 0; k < VEC; ++k)
        if (in[k]) pl[multi_at<S, EX>(r, x + k, RS)] = v[k];
}
template <class S, int VEC, int EX, class C>
__device__ __forceinline__ void multi_get(const S* pl, int r, int x, int RS, C (&v)[VEC]) {
    if constexpr (VEC == 2 && EX == 0) {
        using W = typename std::conditional<sizeof(S) == 2, uint32_t, float2>::type;
        const W w = *reinterpret_cast<const W*>(pl + r * RS + x);
        S t[2];
        memcpy(t, &w, sizeof(W));
        v[0] = to_c<C>(t[0]);
        v[1] = to_c<C>(t[1]);
    } else {
#pragma unroll
        for (int k = 0; k < VEC; ++k) v[k] = to_c<C>(pl[multi_at<S, EX>(r, x + k - EX, RS)]);
    }
}

// The wall rules for the post-collision value `val` (unscaled) of population i
// of the node at (x, y), region node (r, c): half-way bounce-back into the
// ghost slot that the node pulls from in the next step (ghost_write's rule, in
// shared memory).  Faces crossed periodically need nothing: the region holds
// the images as nodes.
template <class LS, bool THERMAL, int i, int P0, class S, class C, bool RAW>
__device__ __forceinline__ void multi_ghost(S* sm, const KParams& p, const MultiGeo& g, int x, int y, int r, int c,
                                            C val, uint32_t salt) {
    constexpr int ex = LS::e(i, 0), ey = LS::e(i, 1), o = LS::opp(i);
    if constexpr (ex != 0 || ey != 0) {
        const bool ox = ex != 0 && !(p.periodic & 1) && (x + ex < 0 || x + ex >= p.L.nx);
        const bool oy = ey != 0 && !(p.periodic & 2) && (y + ey < 0 || y + ey >= p.L.ny);
        if (!(ox || oy)) return;
        const int rr = r + ey, cc = c + ex;
        if (rr < 0 || rr >= g.H || cc < 0 || cc >= g.W) return;  // outside: pulled by no node of this block
        const C scale = ScaleOf<C>::s(p);
        C out = val;
        if constexpr (THERMAL)  // axis-aligned: its direction names the face
            if (p.heat_axis == (ex != 0 ? 0 : 1)) out = anti_bounce_back<(ex + ey > 0)>(val, p);
        S v;
        if constexpr (THERMAL) v = enc_g_step<S, C>(out, scale, salt);
        else v = enc_f_step<LS, S, C, RAW>(out, o, scale, salt);
        sm[(P0 + o) * g.RS * g.H + multi_at<S, LS::e(o, 0)>(rr, cc, g.RS)] = v;
    }
}

template <class S>
__global__ void __launch_bounds__(Multi<S>::THREADS, 1)
    step_multi_kernel(const S* __restrict__ src, S* __restrict__ dst, const KParams p, const MultiGeo g) {
    using LF = D2Q9;
    using LG = D2Q5;
    using C = typename Storage<S>::C;
    constexpr int QF = LF::Q, QG = LG::Q, VEC = Multi<S>::VEC;
    constexpr bool KS = true, RAW = !Storage<S>::offset;
    extern __shared__ __align__(16) unsigned char multi_raw[];
    S* sm = reinterpret_cast<S*>(multi_raw) + Multi<S>::PAD;
    const Layout& L = p.L;
    const int RS = g.RS, plane = RS * g.H;
    const int cx0 = blockIdx.x * g.tw, cy0 = blockIdx.y * g.th;
    const int cx1 = min(cx0 + g.tw, L.nx), cy1 = min(cy0 + g.th, L.ny);
    const int X0 = cx0 - g.m, Y0 = cy0 - g.m;  // the region's corner
    const bool px = p.periodic & 1, py = p.periodic & 2;
    const C scale = ScaleOf<C>::s(p), inv_scale = ScaleOf<C>::inv(p);
    const C un = Storage<S>::offset ? inv_scale : C(1);  // the wall rules take unscaled values

    const uint32_t tcount = step_count<S>(src, 0);
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) advance_count<S>(dst, 0, tcount + (uint32_t)g.steps - 1u, true);

    int r = (int)threadIdx.x / (g.W / VEC), c = ((int)threadIdx.x - r * (g.W / VEC)) * VEC;
    for (int j = 1;; ++j) {
        // nodes still needed: the tile and `rem` nodes around it, inside the
        // cell along every axis that is not periodic.  FP64 threads take them
        // row by row anew each step, so that no warp is left half empty (the
        // FP64 pipe spends as much on an idle lane)
        const int rem = g.steps - j;
        const int ax0 = px ? cx0 - rem : max(cx0 - rem, 0), ax1 = px ? cx1 + rem : min(cx1 + rem, L.nx);
        const int ay0 = py ? cy0 - rem : max(cy0 - rem, 0), ay1 = py ? cy1 + rem : min(cy1 + rem, L.ny);
        if constexpr (VEC == 1) {
            const int wp = ax1 - ax0, row = (int)threadIdx.x / wp;
            r = ay0 - Y0 + row;
            c = ax0 - X0 + (int)threadIdx.x - row * wp;
        }
        const int x0 = X0 + c, y = Y0 + r;
        const bool need = y >= ay0 && y < ay1 && x0 + VEC > ax0 && x0 < ax1;
        const uint32_t salt = step_salt(tcount + (uint32_t)j - 1u);
        C f[QF][VEC], t[QG][VEC];
        bool in[VEC];
#pragma unroll
        for (int k = 0; k < VEC; ++k) in[k] = px || (x0 + k >= 0 && x0 + k < L.nx);
        if (need) {
            if (j == 1) {
                // from global memory: periodic images by their own coordinates,
                // a pair's node outside the cell somewhere harmless
                const int gy = y < 0 ? y + L.ny : (y >= L.ny ? y - L.ny : y);
                const S* rowp = src + L.row(gy, 0);
#pragma unroll
                for (int k = 0; k < VEC; ++k) {
                    int gx = x0 + k;
                    if (px) gx = gx < 0 ? gx + L.nx : (gx >= L.nx ? gx - L.nx : gx);
                    gx = min(max(gx, 0), L.nx - 1);
                    const S* own = rowp + gx;
                    static_for<QF>([&](auto ii) {
                        constexpr int i = decltype(ii)::value;
                        f[i][k] = to_c<C>(ld_one<S, false>(TLBM_DBG(p, (own + (p.loff[i] - LF::e(i, 0))), 0, 1)));
                    });
                    static_for<QG>([&](auto ii) {
                        constexpr int i = decltype(ii)::value;
                        t[i][k] = to_c<C>(ld_one<S, false>(TLBM_DBG(p, (own + (p.loff[QF + i] - LG::e(i, 0))), 0, 1)));
                    });
                }
            } else {
                static_for<QF>([&](auto ii) {
                    constexpr int i = decltype(ii)::value;
                    multi_get<S, VEC, LF::e(i, 0), C>(sm + i * plane, r - LF::e(i, 1), c, RS, f[i]);
                });
                static_for<QG>([&](auto ii) {
                    constexpr int i = decltype(ii)::value;
                    multi_get<S, VEC, LG::e(i, 0), C>(sm + (QF + i) * plane, r - LG::e(i, 1), c, RS, t[i]);
                });
            }
            static_for<QF>([&](auto ii) {
                constexpr int i = decltype(ii)::value;
#pragma unroll
                for (int k = 0; k < VEC; ++k) f[i][k] = raw_to_dev_k<LF, S, C, KS>(f[i][k], i, inv_scale);
            });
            static_for<QG>([&](auto ii) {
                constexpr int i = decltype(ii)::value;
#pragma unroll
                for (int k = 0; k < VEC; ++k) t[i][k] = raw_to_g_k<S, C, KS>(t[i][k], inv_scale);
            });
            collide_vec<2, true, C, collide_scaled<S, true>, VEC, true>(f, t, p);
        }
        if (rem == 0) {
            if (!need) return;
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                const int x = x0 + k;
                if (x < cx0 || x >= cx1) continue;
                S* own = dst + L.row(y, 0) + x;
                C f1[QF][1], t1[QG][1];
                static_for<QF>([&](auto ii) {
                    constexpr int i = decltype(ii)::value;
                    f1[i][0] = f[i][k];
                    *TLBM_DBG(p, (own + p.soff[i]), 0, 1) = enc_f_k<LF, S, C, KS>(f[i][k], i, scale, salt);
                });
                static_for<QG>([&](auto ii) {
                    constexpr int i = decltype(ii)::value;
                    t1[i][0] = t[i][k];
                    *TLBM_DBG(p, (own + p.soff[QF + i]), 0, 1) = enc_g_k<S, C, KS>(t[i][k], scale, salt);
                });
                wall_writes<2, S, 1, C, KS>(dst, p, x, y, 0, f1, t1, salt);
            }
            return;
        }
        if (j > 1) __syncthreads();  // everyone has pulled the previous step's values
        if (need) {
            static_for<QF>([&](auto ii) {
                constexpr int i = decltype(ii)::value;
                S v[VEC];
                enc_vec<LF, S, C, KS, VEC>(f[i], i, scale, salt, v);
                multi_put<S, VEC, LF::e(i, 0)>(sm + i * plane, r, c, RS, v, in);
            });
            static_for<QG>([&](auto ii) {
                constexpr int i = decltype(ii)::value;
                S v[VEC];
                enc_vec<LF, S, C, KS, VEC>(t[i], -1, scale, salt, v);
                multi_put<S, VEC, LG::e(i, 0)>(sm + (QF + i) * plane, r, c, RS, v, in);
            });
            const bool yface = y == 0 || y == L.ny - 1;
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                if (!in[k] || !(yface || x0 + k == 0 || x0 + k == L.nx - 1)) continue;
                static_for<QF>([&](auto ii) {
                    constexpr int i = decltype(ii)::value;
                    multi_ghost<LF, false, i, 0, S, C, RAW>(sm, p, g, x0 + k, y, r, c + k, f[i][k] * un, salt);
                });
                static_for<QG>([&](auto ii) {
                    constexpr int i = decltype(ii)::value;
                    multi_ghost<LG, true, i, QF, S, C, RAW>(sm, p, g, x0 + k, y, r, c + k, t[i][k] * un, salt);
                });
            }
        }
        __syncthreads();
    }
}

template <class S>
size_t multi_smem(const MultiGeo& g) {
    return ((size_t)14 * g.RS * g.H + 2 * Multi<S>::PAD) * sizeof(S);
}

// Rows of an odd number of half bank lines, so that two rows of a warp's pairs
// fall on different banks (FP64: one node per thread, any row).
template <class S>
int multi_row(int W) {
    constexpr int U = sizeof(S) == 8 ? 1 : 128 / (int)sizeof(S);  // elements of a line of the 32 banks
    return U == 1 ? W : (W + U / 2 - 1) / U * U + U / 2;
}

// Tile and steps per launch by a model of a launch's time in us on one SM, its
// constants fitted to the measurements above: a launch costs START; a step of a
// block costs STEP and BUSY for each warp of the SM's blocks (FP64: the FP64
// pipe's time for a warp's 114 instructions per node), the blocks of an SM
// beyond those resident at once add rounds.  The model only ranks: it is within
// 15 % of the measured times at 65^2 to 513^2.
template <class S>
bool multi_best(const KParams& p, int sms, MultiGeo& best) {
    constexpr bool F64 = sizeof(S) == 8;
    constexpr int VEC = Multi<S>::VEC;
    constexpr double START = F64 ? 3.4 : 3.0, STEP = F64 ? 0.5 : 1.3, BUSY = F64 ? 1.05 : 0.07;
    static constexpr int TILES[][2] = {{26, 26}, {26, 18}, {22, 22}, {22, 14}, {18, 10}, {14, 9}, {12, 12},
                                       {11, 11}, {10, 12}, {10, 8}, {8, 8}, {8, 4}, {7, 7}};
    double least = 1e30;
    for (const auto& t : TILES)
        for (int k = 2; k <= 8; ++k) {
            MultiGeo g{t[0], t[1], k - 1, 0, t[1] + 2 * (k - 1), 0, k};
            g.W = (t[0] + 2 * (k - 1) + VEC - 1) / VEC * VEC;
            g.RS = multi_row<S>(g.W);
            const int threads = (g.W / VEC * g.H + 31) / 32 * 32;
            const size_t smem = multi_smem<S>(g);
            if (threads > Multi<S>::THREADS || smem > 200 * 1024) continue;
            const long long blocks = (long long)((p.L.nx + g.tw - 1) / g.tw) * ((p.L.ny + g.th - 1) / g.th);
            // blocks an SM holds: registers (at most 128 a thread) and shared memory
            const long long held = std::max<long long>(1, std::min<long long>(65536 / (128 * threads), 220 * 1024 / (long long)smem));
            const long long mine = (blocks + sms - 1) / sms, at_once = std::min(mine, held);
            const long long rounds = (mine + at_once - 1) / at_once;
            double time = START + k * STEP;
            if (F64) {
                int warps = 0;
                for (int m = 0; m < k; ++m) warps += ((t[0] + 2 * m) * (t[1] + 2 * m) + 31) / 32;
                time = rounds * time + mine * BUSY * warps;
            } else {
                time = rounds * (time + k * BUSY * (double)(at_once * threads / 32));
            }
            if (time / k < least) {
                least = time / k;
                best = g;
            }
        }
    return least < 1e30;
}

template <class S>
cudaError_t multi_launch(const void* src, void* dst, const KParams& p, const MultiGeo& g, cudaStream_t s) {
    const int threads = (g.W / Multi<S>::VEC * g.H + 31) / 32 * 32;
    const size_t smem = g.steps > 1 ? multi_smem<S>(g) : 0;
    const dim3 grid((p.L.nx + g.tw - 1) / g.tw, (p.L.ny + g.th - 1) / g.th);
    step_multi_kernel<S><<<grid, threads, smem, s>>>((const S*)src, (S*)dst, p, g);
    return cudaGetLastError();
}

template <class S>
cudaError_t multi_allow(size_t most) {
    return cudaFuncSetAttribute(step_multi_kernel<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
}

}  // namespace

bool multi_setup(int prec, const KParams& p, MultiGeo& g) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return false;
    switch (prec) {
    case 0: return multi_best<double>(p, sms, g) && multi_allow<double>(200 * 1024) == cudaSuccess;
    case 1: return multi_best<float>(p, sms, g) && multi_allow<float>(200 * 1024) == cudaSuccess;
    case 2: return multi_best<__half>(p, sms, g) && multi_allow<__half>(200 * 1024) == cudaSuccess;
    default: return multi_best<__nv_bfloat16>(p, sms, g) && multi_allow<__nv_bfloat16>(200 * 1024) == cudaSuccess;
    }
}

cudaError_t launch_multi(int prec, const void* src, void* dst, const KParams& p, const MultiGeo& g, cudaStream_t s) {
    switch (prec) {
    case 0: return multi_launch<double>(src, dst, p, g, s);
    case 1: return multi_launch<float>(src, dst, p, g, s);
    case 2: return multi_launch<__half>(src, dst, p, g, s);
    default: return multi_launch<__nv_bfloat16>(src, dst, p, g, s);
    }
}

}  // namespace tlbm
