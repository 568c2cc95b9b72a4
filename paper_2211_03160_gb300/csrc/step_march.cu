// Three time steps of a 2D cell in one pass over memory, FP32, FP16 and BF16 storage
// (two-relaxation-time collision, two-buffer streaming, walls on every side).
//
// A one-step kernel of a large cell reads and writes the state once per step and
// is bound by HBM (62 GLUPS at 8193^2, 102 % of the copy rate).  Here a warp owns
// a strip of MARCH_OUT = 56 columns and marches up a segment of rows: it pulls
// row r from memory (two nodes per lane, 64 columns) and collides it (step 1);
// from the post-collision values of rows r - 2, r - 1 and r, which it holds in
// registers, it pulls and collides row r - 1 again (step 2), in the same way row
// r - 2 a third time (step 3), and stores that.  The state is read and written
// once per three steps.  The values a node needs from the columns next to it
// come by shuffles.  A strip's outer columns are stepped by its neighbours as
// well (64 / 56 redundant updates), and a segment steps two extra rows at either
// end.  No barrier: every warp is on its own.  The rows on their way from memory
// go through shared memory (asynchronous copies of each lane's own pairs): held
// in registers instead they spilled, and a spilled load waits for its data.
//
// Of a row's post-collision values only those are kept that a later row pulls:
// the populations with e_y = 0 for one row, those with e_y = +1 for two; those
// with e_y = -1 are pulled at once (28 registers a lane and step).  Wall rules of
// the inner steps: a node's half-way bounce-back value is its own post-collision
// value of the opposite population, so it is put in place of the shuffled one
// at the side walls, and in place of the missing row's values at the bottom and
// top.
//
// What bounds it now: instruction issue and latency at twelve warps an SM (167
// registers a thread; at 4097^2 issue slots 59 % used, 173 instructions per node and
// step, 210 in FP16); HBM moves 37 of the 112 bytes per update.  GLUPS on GB300
// by steps per pass (blocks of four warps per SM) at 8193^2: 2 (3) 111, 3 (3)
// 132, 3 (4, spilling) 80, 4 (2) 124; 2 (5, at 96 registers) 75.  us per step,
// one-step kernel -> this: 513^2 7.4 -> 5.7, 1025^2 22.2 -> 12.4, 2049^2 75.5 ->
// 38.1, 4097^2 279 -> 135, 8193^2 1081 -> 493 (136 GLUPS).  16-bit storage rounds (and
// hashes) every value of every step, so its steps cost more instructions and its
// one-step kernel was further from the HBM rate: FP16 1025^2 17.3 -> 15.7, 2049^2 47.5
// -> 44.8, 4097^2 173 -> 157, 8193^2 620 -> 564 (119 GLUPS).
//
// Every node gets bitwise the values of the one-step kernels.
#include <algorithm>

#include "dispatch.h"

namespace tlbm {

namespace {

constexpr int MARCH_W = 64;       // columns a warp steps
constexpr int MARCH_SIDE = 4;     // columns a side that it does not store: >= MARCH_STEPS, even (aligned pairs)
constexpr int MARCH_OUT = MARCH_W - 2 * MARCH_SIDE;
static_assert(MARCH_OUT == MARCH_COLUMNS, "columns a warp stores");
constexpr int MARCH_WARPS = 4;    // warps of a block
// Blocks per SM: 168 registers a thread; the 16-bit forms keep their rows packed
// and nearly fit in 128 (FP16 8193^2 563 us per step, 587 with three blocks).
template <class S>
struct MarchCfg {
    static constexpr int BLOCKS = sizeof(S) == 4 ? 3 : 4;
};
constexpr int MARCH_AHEAD = 1;    // rows whose copies are in flight

// A lane's pair of stored values: two floats, or two 16-bit values in a word.
template <class S>
using MarchPair = typename std::conditional<sizeof(S) == 4, float2, uint32_t>::type;

template <class S>
__device__ __forceinline__ float2 march_unpack(MarchPair<S> w) {
    if constexpr (sizeof(S) == 4) {
        return w;
    } else {
        typename Pair<S>::T t;
        memcpy(&t, &w, 4);
        return Pair<S>::unpack(t);
    }
}
// the storage rounding of a step (stochastic for 16-bit values)
template <class S>
__device__ __forceinline__ MarchPair<S> march_pack(float2 v, uint32_t salt) {
    if constexpr (sizeof(S) == 4) return v;
    else return cvt_rs2<S>(v.y, v.x, salt);
}
// A single stored value: a float, or a 16-bit value in both halves of a word.
template <class S>
using MarchOne = typename std::conditional<sizeof(S) == 4, float, uint32_t>::type;
template <class S>
__device__ __forceinline__ MarchOne<S> march_pack1(float v, uint32_t salt) {
    if constexpr (sizeof(S) == 4) return v;
    else return __byte_perm(cvt_rs2<S>(0.0f, v, salt), 0u, 0x1010);
}
// the lower / upper value of a pair
__device__ __forceinline__ float march_one(float2 v, bool upper) { return upper ? v.y : v.x; }
__device__ __forceinline__ uint32_t march_one(uint32_t v, bool upper) { return __byte_perm(v, v, upper ? 0x3232 : 0x1010); }

// value of column x - EX for the lane's two columns
template <int EX>
__device__ __forceinline__ float2 march_shift(float2 v) {
    if constexpr (EX == 1) return make_float2(__shfl_up_sync(0xffffffffu, v.y, 1), v.x);
    else if constexpr (EX == -1) return make_float2(v.y, __shfl_down_sync(0xffffffffu, v.x, 1));
    else return v;
}
template <int EX>
__device__ __forceinline__ uint32_t march_shift(uint32_t v) {
    if constexpr (EX == 1) return __byte_perm(__shfl_up_sync(0xffffffffu, v, 1), v, 0x5432);
    else if constexpr (EX == -1) return __byte_perm(v, __shfl_down_sync(0xffffffffu, v, 1), 0x5432);
    else return v;
}
// w with its lower / upper value taken from the lower / upper place of v, or from one value
__device__ __forceinline__ float2 march_lo(float2 w, float v) { return make_float2(v, w.y); }
__device__ __forceinline__ float2 march_hi(float2 w, float v) { return make_float2(w.x, v); }
__device__ __forceinline__ float2 march_lo(float2 w, float2 v) { return make_float2(v.x, w.y); }
__device__ __forceinline__ float2 march_hi(float2 w, float2 v) { return make_float2(w.x, v.y); }
__device__ __forceinline__ uint32_t march_lo(uint32_t w, uint32_t v) { return __byte_perm(w, v, 0x3254); }
__device__ __forceinline__ uint32_t march_hi(uint32_t w, uint32_t v) { return __byte_perm(w, v, 0x7610); }
// The thermal wall rule of the lower / upper (HI) wall for a post-collision value (scaled as it is stored,
// not yet rounded): anti-bounce-back at a wall of temperature Tw, bounce-back at
// an adiabatic one.
template <bool HI, class PT>
__device__ __forceinline__ float march_rule(float v, bool iso, const PT& p) {
    const float val = v * ScaleOf<float>::inv(p);
    return (iso ? anti_bounce_back<HI>(val, p) : val) * ScaleOf<float>::s(p);
}
template <bool HI, class PT>
__device__ __forceinline__ float2 march_rule(float2 v, bool iso, const PT& p) {
    return make_float2(march_rule<HI>(v.x, iso, p), march_rule<HI>(v.y, iso, p));
}

// copy the stored pairs a lane pulls for one row (before the shift along x) to
// the lane's places in shared memory, as one group of its asynchronous copies
template <class S, class PT>
__device__ __forceinline__ void march_fetch(const S* __restrict__ own, const PT& p, const KParams& full, uint32_t to) {
#pragma unroll
    for (int j = 0; j < 14; ++j)
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(to + j * MARCH_W * (int)sizeof(S)),
                     "l"(TLBM_DBG(full, (own + p.loff[j]), 0, 2)), "n"(2 * (int)sizeof(S))
                     : "memory");
}

// What a strip keeps of one step's post-collision values, as they would be
// stored: e_y = 0 of the last row (flow 0, 1, 3, thermal 0, 1, 3), e_y = +1 (flow
// 2, 5, 6, thermal 2) of the last row and of the one before; at a side wall the
// last row's diagonal with e_y = -1 that meets it and the
// value its thermal rule returns.
template <class S>
struct MarchKept {
    MarchPair<S> z[6], u1[4], u0[4];
    MarchOne<S> wd, wg;
};

// f, g: the post-collision values of row r, or anything if r = ny.  Keeps what
// later rows pull of them and turns f, g into what row r - 1 pulls.
template <int DIM, class S, class PT>
__device__ __forceinline__ void march_pull(MarchKept<S>& k, float2 (&f)[9], float2 (&g)[5], const PT& p, int r, int x,
                                           bool wall_strip, bool heat_y, uint32_t salt) {
    using W = MarchPair<S>;
    const Layout& L = p.L;
    W F[9], G[5];
#pragma unroll
    for (int i = 0; i < 9; ++i) F[i] = march_pack<S>(f[i], salt);
#pragma unroll
    for (int i = 0; i < 5; ++i) G[i] = march_pack<S>(g[i], salt);
    W n[9], m[5];  // what row r - 1 pulls
    n[0] = k.z[0];
    n[1] = march_shift<1>(k.z[1]);
    n[2] = k.u0[0];
    n[3] = march_shift<-1>(k.z[2]);
    n[5] = march_shift<1>(k.u0[1]);
    n[6] = march_shift<-1>(k.u0[2]);
    m[0] = k.z[3];
    m[1] = march_shift<1>(k.z[4]);
    m[2] = k.u0[3];
    m[3] = march_shift<-1>(k.z[5]);
    if (r < L.ny) {
        n[4] = F[4];
        n[7] = march_shift<-1>(F[7]);
        n[8] = march_shift<1>(F[8]);
        m[4] = G[4];
    } else {
        // past the top wall: what row ny - 1 pulls from there is its own (the
        // thermal one already as the wall returns it, see below)
        n[4] = k.u1[0];
        n[7] = k.u1[1];
        n[8] = k.u1[2];
        m[4] = k.u1[3];
    }
    if (wall_strip) {
        if (x == 0) {
            n[1] = march_lo(n[1], k.z[2]);
            n[5] = march_lo(n[5], k.wd);
            n[8] = march_lo(n[8], k.u1[2]);
            m[1] = march_lo(m[1], k.wg);
        }
        if (x == L.nx - 1) {
            n[3] = march_lo(n[3], k.z[1]);
            n[6] = march_lo(n[6], k.wd);
            n[7] = march_lo(n[7], k.u1[1]);
            m[3] = march_lo(m[3], k.wg);
        }
        if (x + 1 == L.nx - 1) {
            n[3] = march_hi(n[3], k.z[1]);
            n[6] = march_hi(n[6], k.wd);
            n[7] = march_hi(n[7], k.u1[1]);
            m[3] = march_hi(m[3], k.wg);
        }
        // keep what row r's node at a side wall gets back
        const bool upper = x + 1 == L.nx - 1;
        k.wd = march_one(x == 0 ? F[7] : F[8], upper);
        const float t = x == 0 ? march_rule<false>(g[3].x, !heat_y, p)
                               : march_rule<true>(upper ? g[1].y : g[1].x, !heat_y, p);
        k.wg = march_pack1<S>(t, salt);
    }
    // keep row r
#pragma unroll
    for (int q = 0; q < 4; ++q) k.u0[q] = k.u1[q];
    k.u1[0] = F[2];
    k.u1[1] = F[5];
    k.u1[2] = F[6];
    k.u1[3] = G[2];
    k.z[0] = F[0];
    k.z[1] = F[1];
    k.z[2] = F[3];
    k.z[3] = G[0];
    k.z[4] = G[1];
    k.z[5] = G[3];
    if (r == 0) {
        // below the bottom wall: what row 0 pulls from there is its own
        // (shifted back, as the next pull shifts it)
        k.u0[0] = F[4];
        k.u0[1] = march_shift<-1>(F[7]);
        k.u0[2] = march_shift<1>(F[8]);
        k.u0[3] = march_pack<S>(march_rule<false>(g[4], heat_y, p), salt);
    }
    if (r == L.ny - 1) k.u1[3] = march_pack<S>(march_rule<true>(g[2], heat_y, p), salt);
#pragma unroll
    for (int i = 0; i < 9; ++i) f[i] = march_unpack<S>(n[i]);
#pragma unroll
    for (int i = 0; i < 5; ++i) g[i] = march_unpack<S>(m[i]);
}

// One warp's strip and segment.  p: the parameters of the hot path; full: all of
// them, for the wall rules of the last step (the same object for a single cell).
template <int DIM, class S, class PT>
__device__ __forceinline__ void march_strip(const S* __restrict__ src, S* __restrict__ dst, const PT& p,
                                            const KParams& full, int strip, int sg, int seg) {
    static_assert(MARCH_SIDE >= MARCH_STEPS && MARCH_SIDE % 2 == 0, "valid columns");
    using LF = typename Lat<DIM>::F;
    using LG = typename Lat<DIM>::G;
    constexpr int QF = LF::Q, QG = LG::Q, Q = QF + QG;
    constexpr int LV = MARCH_STEPS, SIDE = MARCH_SIDE, OUT = MARCH_OUT;
    constexpr bool SC = collide_scaled<S, true>;
    using W = MarchPair<S>;
    const Layout& L = p.L;
    const int lane = threadIdx.x & 31;
    const int x = strip * OUT - SIDE + 2 * lane;  // the lane's first column
    const int y0 = sg * seg, y1 = min(y0 + seg, L.ny);
    const bool wall_strip = strip == 0 || strip * OUT + OUT + SIDE >= L.nx;
    const bool store = lane >= SIDE / 2 && lane < 32 - SIDE / 2 && x < L.nx;
    const bool heat_y = p.heat_axis == 1;
    const int xld = min(x, L.P - 2);

    // rows on their way from memory: a ring of MARCH_AHEAD + 1 rows per warp,
    // every lane's pairs in places of its own
    __shared__ __align__(16) S ring[MARCH_WARPS][MARCH_AHEAD + 1][Q][MARCH_W];
    constexpr int ROWB = Q * MARCH_W * (int)sizeof(S);
    S* mine = &ring[threadIdx.x >> 5][0][0][2 * lane];
    const uint32_t mine_at = smem_addr(mine);
    MarchKept<S> kept[LV - 1] = {};
    // the step counter of 16-bit storage (the salt of its stochastic rounding)
    const uint32_t tcount = step_count<S>(src, 0);
    if (strip == 0 && sg == 0 && lane == 0) advance_count<S>(dst, 0, tcount + (uint32_t)(LV - 1), true);

    const int r0 = max(y0 - (LV - 1), 0);
    const int rl = min(y1 + LV - 2, L.ny - 1);  // last row to pull
    const S* from = src + L.row(r0, 0) + xld;
#pragma unroll
    for (int k = 0; k < MARCH_AHEAD; ++k) {
        if (r0 + k <= rl) march_fetch(from + (long long)k * L.P, p, full, mine_at + k * ROWB);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    from += (long long)MARCH_AHEAD * L.P;
    int slot = 0, ahead = MARCH_AHEAD;
    for (int r = r0; r <= y1 + LV - 2; ++r) {
        float2 f[QF], g[QG];
        if (r < L.ny) {
            if (r + MARCH_AHEAD <= rl) march_fetch(from, p, full, mine_at + ahead * ROWB);
            asm volatile("cp.async.commit_group;" ::: "memory");
            asm volatile("cp.async.wait_group %0;" ::"n"(MARCH_AHEAD) : "memory");
            from += L.P;
            const S* row = mine + slot * (Q * MARCH_W);
            slot = slot == MARCH_AHEAD ? 0 : slot + 1;
            ahead = ahead == MARCH_AHEAD ? 0 : ahead + 1;
            static_for<QF>([&](auto ii) {
                constexpr int i = decltype(ii)::value;
                f[i] = march_unpack<S>(march_shift<LF::e(i, 0)>(*reinterpret_cast<const W*>(row + i * MARCH_W)));
            });
            static_for<QG>([&](auto ii) {
                constexpr int i = decltype(ii)::value;
                g[i] = march_unpack<S>(march_shift<LG::e(i, 0)>(*reinterpret_cast<const W*>(row + (QF + i) * MARCH_W)));
            });
            collide_trt_v<DIM, float2, SC, true>(f, g, p);
        }
        // step l + 2 of row r - 1 - l; rows past the top wall hold anything, and
        // so do rows too close to the segment's first one
#pragma unroll
        for (int l = 0; l < LV - 1; ++l) {
            march_pull<DIM, S>(kept[l], f, g, p, r - l, x, wall_strip, heat_y, step_salt(tcount + (uint32_t)l));
            if (r - l > r0) collide_trt_v<DIM, float2, SC, true>(f, g, p);
        }
        const int y = r - (LV - 1);
        if (y < y0 || !store) continue;
        S* own = dst + L.row(y, 0) + x;
        const uint32_t salt = step_salt(tcount + (uint32_t)(LV - 1));
        static_for<Q>([&](auto jj) {
            constexpr int j = decltype(jj)::value;
            const W w = march_pack<S>(j < QF ? f[j < QF ? j : 0] : g[j < QF ? 0 : j - QF], salt);
            if (x + 1 < L.nx) {
                __stwb(reinterpret_cast<W*>(TLBM_DBG(full, (own + p.soff[j]), 0, 2)), w);
            } else {
                S one[2];
                memcpy(one, &w, sizeof(W));
                *TLBM_DBG(full, (own + p.soff[j]), 0, 1) = one[0];
            }
        });
        if (y == 0 || y == L.ny - 1 || x == 0 || x + 2 >= L.nx) {
            float fw[QF][2], gw[QG][2];
#pragma unroll
            for (int i = 0; i < QF; ++i) { fw[i][0] = f[i].x; fw[i][1] = f[i].y; }
#pragma unroll
            for (int i = 0; i < QG; ++i) { gw[i][0] = g[i].x; gw[i][1] = g[i].y; }
            wall_writes<2, S, 2, float, true, PULL, true>(dst, full, x, y, 0, fw, gw, salt);
        }
    }
}

template <int DIM, class S>
__global__ void __launch_bounds__(32 * MARCH_WARPS, MarchCfg<S>::BLOCKS)
    step_march_kernel(const S* __restrict__ src, S* __restrict__ dst, const KParams p, int strips, int seg) {
    const int item = blockIdx.x * MARCH_WARPS + (threadIdx.x >> 5), sg = item / strips;
    if (sg * seg < p.L.ny) march_strip<DIM, S>(src, dst, p, p, item - sg * strips, sg, seg);
}

// The cells of a batch: a block's warps all march in one cell, whose parameters
// it reads from the launch's parameters (constant memory) at an index that is
// the same for the block.
template <int DIM, class S>
__global__ void __launch_bounds__(32 * MARCH_WARPS, MarchCfg<S>::BLOCKS)
    step_march_batch_kernel(const __grid_constant__ MarchBatch b, int parity) {
    int lo = 0, hi = b.n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if (b.cell[mid].block0 <= (int)blockIdx.x) lo = mid;
        else hi = mid - 1;
    }
    const MarchCell& c = b.cell[lo];
    const int item = ((int)blockIdx.x - c.block0) * MARCH_WARPS + (threadIdx.x >> 5), sg = item / c.strips;
    if (sg * b.rows < c.L.ny)
        march_strip<DIM, S>((const S*)c.buf[parity], (S*)c.buf[parity ^ 1], c, *c.full, item - sg * c.strips, sg, b.rows);
}

}  // namespace

// Rows of a segment.  Every segment costs 2 (MARCH_STEPS - 1) rows more than it
// stores, so as few segments as fill the GPU: one round of resident warps where
// that gives segments of up to 64 rows, else the fewest whole rounds that do
// (longer segments end too unevenly).  us per step at 2049^2 with 42 rows (one
// round) 42.0, 21 (two) 42.7, 48 47.2; at 8193^2 with 61 500, 84 509, 168 520,
// 683 621.
static int march_resident(int prec) { return (prec == 1 ? MarchCfg<float>::BLOCKS : MarchCfg<__half>::BLOCKS) * MARCH_WARPS; }

int march_rows(int prec, const KParams& p) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    const int strips = (p.L.nx + MARCH_OUT - 1) / MARCH_OUT, resident = sms * march_resident(prec);
    for (int rounds = 1;; ++rounds) {
        const long long segs = std::max<long long>(1, (long long)rounds * resident / strips);
        const int rows = (int)((p.L.ny + segs - 1) / segs);
        if (rows <= 64) return rows;
    }
}

template <class S>
static cudaError_t march_launch(const void* src, void* dst, const KParams& p, int rows, cudaStream_t s) {
    const int strips = (p.L.nx + MARCH_OUT - 1) / MARCH_OUT;
    const int items = strips * ((p.L.ny + rows - 1) / rows), grid = (items + MARCH_WARPS - 1) / MARCH_WARPS;
    step_march_kernel<2, S><<<grid, 32 * MARCH_WARPS, 0, s>>>((const S*)src, (S*)dst, p, strips, rows);
    return cudaGetLastError();
}
cudaError_t launch_march(int prec, const void* src, void* dst, const KParams& p, int rows, cudaStream_t s) {
    if (prec == 1) return march_launch<float>(src, dst, p, rows, s);
    if (prec == 2) return march_launch<__half>(src, dst, p, rows, s);
    return march_launch<__nv_bfloat16>(src, dst, p, rows, s);
}

int march_batch_rows(int prec, const long long* strips_ny, int n) {
    int dev = 0, sms = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
        return 0;
    // march_rows for all cells together
    const long long resident = (long long)sms * march_resident(prec);
    for (int rows = 4;; rows += rows < 16 ? 1 : 4) {
        long long items = 0;
        for (int i = 0; i < n; ++i) items += strips_ny[2 * i] * ((strips_ny[2 * i + 1] + rows - 1) / rows);
        if (items <= resident || rows >= 64) return rows;
    }
}

MarchCell march_cell(const KParams& p, const void* buf0, const void* buf1, const KParams* full) {
    MarchCell c{};
    c.L = p.L;
    c.heat_axis = p.heat_axis;
    c.gbetaf = p.gbetaf;
    c.omegaf = p.omegaf;
    c.Thf = p.Thf;
    c.Tcf = p.Tcf;
    for (int a = 0; a < 3; ++a) c.bodyf[a] = p.bodyf[a];
    c.spf = p.spf;
    c.smf = p.smf;
    c.shpf = p.shpf;
    c.shmf = p.shmf;
    c.qpf = p.qpf;
    c.qmf = p.qmf;
    c.tf = p.tf;
    c.scale = p.scale;
    c.inv_scale = p.inv_scale;
    for (int j = 0; j < 14; ++j) {
        c.loff[j] = p.loff[j];
        c.soff[j] = p.soff[j];
    }
    c.buf[0] = const_cast<void*>(buf0);
    c.buf[1] = const_cast<void*>(buf1);
    c.full = full;
    c.strips = (p.L.nx + MARCH_OUT - 1) / MARCH_OUT;
    return c;
}

int march_cell_blocks(const MarchCell& c, int rows) {
    return (c.strips * ((c.L.ny + rows - 1) / rows) + MARCH_WARPS - 1) / MARCH_WARPS;
}

cudaError_t launch_march_batch(int prec, const MarchBatch& b, int grid, int parity, cudaStream_t s) {
    if (prec == 1) step_march_batch_kernel<2, float><<<grid, 32 * MARCH_WARPS, 0, s>>>(b, parity);
    else if (prec == 2) step_march_batch_kernel<2, __half><<<grid, 32 * MARCH_WARPS, 0, s>>>(b, parity);
    else step_march_batch_kernel<2, __nv_bfloat16><<<grid, 32 * MARCH_WARPS, 0, s>>>(b, parity);
    return cudaGetLastError();
}

}  // namespace tlbm
