// The warm-start network's training path on channels-last activations.
//
// The layer kernels of conv.cu take NCHW tensors and turn each tile's input into
// the tensor cores' channel-contiguous operand with 2-byte loads; that staging,
// and for the weight gradient the patch matrix built from it, took most of their
// time.  Between the layers of one network the layout is free, so this path
// keeps activations and gradients "cl": BF16 [B][H][W][Cp] with Cp = 16 ceil(C /
// 16), channels past C zero.  A position's eight channels are then one 16-byte
// asynchronous copy straight into the operand, for the weight gradient too:
// its contraction runs over positions, and a K-major operand's shift along K is
// out of a descriptor's reach, but read "MN-major" (channels contiguous, the
// positions the strided index) a shift by one position is 16 bytes.
//
// Tiles, strips and virtual positions are conv.cu's: image columns in strips of
// Wt, a strip plus one halo column a side a virtual image of width Wv in which
// a 3x3 neighbour is a constant shift.  Both kernels are persistent and copy the
// tiles to come while the tensor cores work on the current one.
//
// us on GB300 for the 32 -> 32 layer at 48 x 65 x 65, NCHW kernels -> these:
// forward 36.4 -> 16.5, data gradient with mask and bias sums 35.1 (no mask, no
// sums) -> 24.6, weight gradient with its reduction 100.7 -> 30.8; the training
// iteration of that network 787 -> 297.  What bounds them now: issue and latency of
// the copies (a tile's 16-byte pieces, 40 to 120 cp.async a thread) and the barriers
// around them; the tensor pipe is 11 to 15 % active and what they write stays in L2.
// Included by conv.cu, whose geometry and descriptor helpers it uses.
#pragma once

namespace {

constexpr int CL_THREADS = 128;  // forward / data gradient: one thread per position

__host__ __device__ constexpr int groups_of(int C) { return 2 * ((C + 15) / 16); }  // 8-channel groups, an even number
// rows of a staged plane (16 bytes each), = 2 mod 8: the groups of a position fall on different banks
__host__ __device__ inline int pad_rows(int r) { return r + ((2 - (r & 7)) & 7); }

__device__ __forceinline__ void copy16(uint32_t to, const void* from, bool in) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(from), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void wait_copies() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// A CTA's tiles, blockIdx.x and every gridDim.x-th from there: image, strip and
// tile of the strip, advanced by the digits of gridDim.x (the divisions once).
struct Walk {
    long long tile, left;  // tile number and tiles in all
    int b, s, k, db, ds, dk, strips, tps;
    __device__ explicit Walk(const TcGeom& geo)
        : tile(blockIdx.x), left(geo.tiles), strips(geo.strips), tps(geo.tps) {
        const long long q = tile / tps, dq = (long long)gridDim.x / tps;
        k = (int)(tile - q * tps);
        b = (int)(q / strips);
        s = (int)(q - (long long)b * strips);
        dk = (int)(gridDim.x - dq * tps);
        db = (int)(dq / strips);
        ds = (int)(dq - (long long)db * strips);
    }
    __device__ bool valid() const { return tile < left; }
    __device__ void next() {
        tile += gridDim.x;
        k += dk;
        const int c = k >= tps;
        k -= c * tps;
        s += ds + c;
        const int d = s >= strips;
        s -= d * strips;
        b += db + d;
    }
};

// Copy `rows` virtual positions of tile q from v on, G groups each, into planes
// at `to`; COPIES > 1: that many times, copy d into the planes d G .. as shifted
// by d positions.  A thread takes one group of every (NT / G)-th position.  halo:
// the halo columns' image columns too (else zero).
template <int G, int NT, int COPIES>
__device__ __forceinline__ void stage(uint32_t to, int plane, const bf16* __restrict__ x, const Walk& q, int v, int rows,
                                      const TcGeom& geo, int H, int W, bool halo) {
    constexpr int STEP = NT / G;
    const int g = (int)threadIdx.x % G, r0 = (int)threadIdx.x / G, Wv = geo.Wv;
    const int u = v + Wv + r0, dq = STEP / Wv, dr = STEP - dq * Wv;  // v >= -1
    int i = u / Wv - 2, jj = u - (i + 2) * Wv - 1;
    const bf16* xb = x + (long long)q.b * H * W * (8 * G) + 8 * g;
    uint32_t at = to + g * plane + r0 * 16;
    for (int r = r0; r < rows + COPIES - 1; r += STEP) {
        const int j = q.s * geo.Wt + jj;
        const bool in = (unsigned)i < (unsigned)H && (unsigned)j < (unsigned)W && (halo || (unsigned)jj < (unsigned)geo.Wt);
        const bf16* from = xb + (in ? (long long)(i * W + j) * (8 * G) : 0);
#pragma unroll
        for (int d = 0; d < COPIES; ++d)
            if (COPIES == 1 || (r >= d && r - d < rows)) copy16(at + d * (G * plane - 16), from, in);
        at += STEP * 16;
        jj += dr;
        i += dq;
        if (jj >= Wv - 1) {
            jj -= Wv;
            ++i;
        }
    }
}

__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool add) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(idesc), "r"((uint32_t)add)
        : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc_smem(bar)) : "memory");
}
// 32 columns of tensor memory, this warp's lanes
__device__ __forceinline__ void tmem_ld32(uint32_t (&r)[32], uint32_t addr) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, "
        "%13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, "
        "[%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
          "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 48 columns, added to acc
__device__ __forceinline__ void tmem_add48(float (&acc)[48], uint32_t addr) {
    uint32_t r[48];
#pragma unroll
    for (int q = 0; q < 48; q += 16)
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
            "[%16];"
            : "=r"(r[q]), "=r"(r[q + 1]), "=r"(r[q + 2]), "=r"(r[q + 3]), "=r"(r[q + 4]), "=r"(r[q + 5]), "=r"(r[q + 6]),
              "=r"(r[q + 7]), "=r"(r[q + 8]), "=r"(r[q + 9]), "=r"(r[q + 10]), "=r"(r[q + 11]), "=r"(r[q + 12]),
              "=r"(r[q + 13]), "=r"(r[q + 14]), "=r"(r[q + 15])
            : "r"(addr + q));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int i = 0; i < 48; ++i) acc[i] += __uint_as_float(r[i]);
}

// ------------------------------------------------------------------ forward and data gradient

// acc[m] = bias[m] + sum over taps and input channels, as conv3x3_tc_kernel; G:
// 8-channel groups of the input.  Forward: y (FP32 NCHW) and act (cl,
// relu'd if relu) where given.  Data gradient (mask: the cl activation whose
// relu the gradient passes back through): act = acc where mask > 0, and the sums
// of those FP32 values over the CTA's positions to sums[cta][32].
template <int G, bool GRAD>
__global__ void __launch_bounds__(CL_THREADS, GRAD ? 4 : 6) conv_cl_kernel(const bf16* __restrict__ A, int M, const bf16* __restrict__ x,
                                                          int H, int W, const float* __restrict__ bias, int relu,
                                                          float* __restrict__ y, bf16* __restrict__ act,
                                                          const bf16* __restrict__ mask, float* __restrict__ sums,
                                                          TcGeom geo) {
    extern __shared__ __align__(1024) uint8_t cl_sm[];
    constexpr int CH = G / 2;
    const int Wv = geo.Wv, rows = tc_rows(Wv), plane = pad_rows(rows) * 16;
    uint8_t* sW = cl_sm;
    uint8_t* sX = cl_sm + 9 * CH * 1024;  // two input tiles
    float* red = reinterpret_cast<float*>(sX + (size_t)2 * G * plane);  // forward: the biases; gradient: 4 warps x 32 sums
    uint64_t* bar = reinterpret_cast<uint64_t*>(red + 128);
    uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 1);
    const int tid = threadIdx.x, warp = tid >> 5;
    const uint32_t xs = tc_smem(sX), ws = tc_smem(sW);
    const long long HW = (long long)H * W;
    const int Go = groups_of(M);  // groups of a cl output

    Walk q(geo), n = q;  // the current tile and the next one
    {
        for (int e = tid; e < 9 * CH * 64; e += CL_THREADS) copy16(ws + e * 16, reinterpret_cast<const uint8_t*>(A) + e * 16, true);
        stage<G, CL_THREADS, 1>(xs, plane, x, q, q.k * TC_PIX - 1, rows, geo, H, W, true);
        commit();
        n.next();
    }
    if (!GRAD && tid < 32) red[tid] = bias && tid < M ? bias[tid] : 0.f;
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(bar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 32;" ::"r"(tc_smem(tslot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t taddr = *tslot;
    const uint32_t idesc =
        (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TC_N >> 3) << 17) | ((uint32_t)(TC_PIX >> 4) << 24);
    float dsum[32];
#pragma unroll
    for (int m = 0; m < 32; ++m) dsum[m] = 0.f;

    bool ok = true;
    for (uint32_t it = 0; q.valid(); q = n, n.next(), ++it) {
        wait_copies<0>();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the copied tile becomes visible to the tensor cores
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (tid == 0) {
            // descriptors differ in their start address (16-byte units, low bits) only
            const uint64_t a0 = tc_desc(xs + (it & 1u) * G * plane, plane, 128), b0 = tc_desc(ws, 512, 128);
#pragma unroll
            for (int t = 0; t < 9; ++t) {
                const uint32_t shift = (uint32_t)((t / 3) * Wv + (t % 3));
#pragma unroll
                for (int h = 0; h < CH; ++h)
                    mma_f16(taddr, a0 + shift + h * (uint32_t)(plane >> 3), b0 + (t * CH + h) * 64, idesc, t + h > 0);
            }
            mma_commit(bar);
        }
        // the next tile, into the buffer whose MMAs the last iteration waited for
        if (n.valid())
            stage<G, CL_THREADS, 1>(xs + ((it & 1u) ^ 1u) * G * plane, plane, x, n, n.k * TC_PIX - 1, rows, geo, H, W, true);
        commit();
        const int v = Wv + q.k * TC_PIX + tid, i = v / Wv - 1, jj = v - (i + 1) * Wv - 1, j = q.s * geo.Wt + jj;
        const bool in = i < H && jj >= 0 && jj < geo.Wt && j < W;
        const long long pos = (long long)q.b * HW + (long long)i * W + j;
        uint4 mk[4];
        if (GRAD && in)
#pragma unroll
            for (int g = 0; g < 4; ++g)
                if (g < Go) mk[g] = reinterpret_cast<const uint4*>(mask)[pos * Go + g];
        ok = tc_wait(bar, it & 1u);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (__syncthreads_or(!ok)) {
            ok = false;
            break;
        }
        uint32_t r[32];
        tmem_ld32(r, taddr + ((uint32_t)(32 * warp) << 16));
        if (in) {
            if constexpr (GRAD) {
#pragma unroll
                for (int m = 0; m < 32; ++m) {
                    const uint32_t w = m < 8 * Go ? reinterpret_cast<const uint32_t*>(mk)[m >> 1] : 0u;
                    const float a = __uint_as_float(m & 1 ? w & 0xffff0000u : w << 16);
                    const float g = a > 0.f ? __uint_as_float(r[m]) : 0.f;
                    r[m] = __float_as_uint(g);
                    dsum[m] += g;
                }
            } else {
#pragma unroll
                for (int m = 0; m < 32; ++m) r[m] = __float_as_uint(__uint_as_float(r[m]) + red[m]);
                if (y) {
                    float* yp = y + (long long)q.b * M * HW + (long long)i * W + j;
#pragma unroll
                    for (int m = 0; m < 32; ++m)
                        if (m < M) yp[m * HW] = __uint_as_float(r[m]);
                }
                if (relu)
#pragma unroll
                    for (int m = 0; m < 32; ++m) r[m] = __float_as_uint(fmaxf(__uint_as_float(r[m]), 0.f));
            }
            if (act)
#pragma unroll
                for (int g = 0; g < 4; ++g)
                    if (g < Go) {
                        uint32_t w[4];
#pragma unroll
                        for (int u = 0; u < 4; ++u)
                            w[u] = pack2(__float2bfloat16_rn(__uint_as_float(r[8 * g + 2 * u])),
                                         __float2bfloat16_rn(__uint_as_float(r[8 * g + 2 * u + 1])));
                        reinterpret_cast<uint4*>(act)[pos * Go + g] = make_uint4(w[0], w[1], w[2], w[3]);
                    }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    wait_copies<0>();
    __syncthreads();
    if (!ok && tid == 0) atomicAdd(&g_conv_timeouts, 1ull);
    if constexpr (GRAD) {
#pragma unroll
        for (int m = 0; m < 32; ++m) {
            float s = dsum[m];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
            if ((tid & 31) == 0) red[warp * 32 + m] = s;
        }
        __syncthreads();
        if (tid < 32)
            sums[(long long)blockIdx.x * 32 + tid] = ok ? (red[tid] + red[32 + tid]) + (red[64 + tid] + red[96 + tid]) : __int_as_float(0x7fc00000);
    }
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 32;" ::"r"(taddr) : "memory");
}

size_t conv_cl_smem(int G, int Wv) {
    return (size_t)9 * (G / 2) * 1024 + (size_t)2 * G * pad_rows(tc_rows(Wv)) * 16 + 128 * sizeof(float) + 16;
}

// db[m] = sum over CTAs, in a fixed order: warp w adds every 32nd row, eight
// loads ahead of their sums, and a tree adds the warps.  (Lanes along the rows
// instead of along m: 11.1 us for 608 rows, 2.4 now.)
__global__ void __launch_bounds__(1024) sum_rows_kernel(const float* __restrict__ sums, int n, int M, float* __restrict__ db) {
    __shared__ float sm[32][33];
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    float s = 0.f;
    for (int k = w; k < n; k += 256) {
        float v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = k + 32 * u < n ? sums[(k + 32 * u) * 32 + l] : 0.f;
#pragma unroll
        for (int u = 0; u < 8; ++u) s += v[u];
    }
    sm[w][l] = s;
    __syncthreads();
    s = sm[l][w];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (l == 0 && w < M) db[w] = s;
}

// ------------------------------------------------------------------ weight gradient

// dW[n][c][di][dj] = sum over positions of dy[n][pos] x[c][pos + (di - 1, dj - 1)]:
// D[(dj, c)][n] for each di, M = 128 rows (3 x 8 GX of them used), N = 8 GY,
// K = the tile's 128 positions.  Both operands are MN-major: core matrix = 8
// positions x 8 channels (16 bytes a position), the next 8 positions 128 bytes
// on, the next 8 channels a plane on.  The planes of dj are the input shifted by
// dj positions, copied three times; di shifts the start address by Wv positions.
// Rows past 24 GX read planes that follow in shared memory and are never used.
// The tensor core truncates as it accumulates, an error that grows with the
// length of the sum, so a tile starts new accumulators (two sets of 96 columns in
// turn) and the tiles add up in registers: relative error 1.3e-6 -> 1.6e-7 at
// 48 x 65^2 and 4.4e-6 -> 1.8e-7 at 64 x 97^2 (NCHW kernel: 6.5e-7 and 2.1e-6), at no
// cost in time: the sums of one tile run beside the MMAs of the next.
// NS: tiles in shared memory.
// part[cta][32 di + n][row].
template <int GX, int GY, int NS>
__global__ void __launch_bounds__(WG_THREADS) wgrad_cl_kernel(const bf16* __restrict__ dy, int M, const bf16* __restrict__ x,
                                                              int C, int H, int W, TcGeom geo, float* __restrict__ part) {
    extern __shared__ __align__(1024) uint8_t cl_sm[];
    const int Wv = geo.Wv, rows = TC_PIX + 2 * Wv, plane = pad_rows(rows) * 16;
    constexpr int YPLANE = (TC_PIX + 2) * 16, NB = 8 * GY;
    const int xbytes = 3 * GX * plane, sbytes = xbytes + GY * YPLANE;
    uint64_t* bar = reinterpret_cast<uint64_t*>(cl_sm);  // two, used in turn
    uint32_t* tslot = reinterpret_cast<uint32_t*>(bar + 2);
    const uint32_t s0 = tc_smem(cl_sm) + 1024;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

    Walk n(geo);  // the next tile to copy
    auto load = [&](int st) {
        const uint32_t at = s0 + st * sbytes;
        if (n.valid()) {
            stage<GX, WG_THREADS, 3>(at, plane, x, n, n.k * TC_PIX - 1, rows, geo, H, W, true);
            stage<GY, WG_THREADS, 1>(at + xbytes, YPLANE, dy, n, n.k * TC_PIX + Wv, TC_PIX, geo, H, W, false);
        }
        commit();
        n.next();
    };

    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(bar)) : "memory");
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(tc_smem(bar + 1)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(tc_smem(tslot)) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t taddr = *tslot;
    // a warp sums half of its quadrant's columns
    const uint32_t own = taddr + ((uint32_t)(32 * (warp & 3)) << 16) + 48 * (warp >> 2);
    float acc[48];
#pragma unroll
    for (int i = 0; i < 48; ++i) acc[i] = 0.f;
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(NB >> 3) << 17) |
                           ((uint32_t)(128 >> 4) << 24);

    long long tile = blockIdx.x;
    const long long G = gridDim.x;
#pragma unroll
    for (int k = 0; k < NS - 1; ++k) load(k);
    bool ok = true;
    uint32_t it = 0;
    int st = 0;
    for (; tile < geo.tiles; tile += G, ++it) {
        wait_copies<NS - 2>();
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (tid == 0) {
            const uint64_t a0 = tc_desc(s0 + st * sbytes, 128, plane), b0 = tc_desc(s0 + st * sbytes + xbytes, 128, YPLANE);
#pragma unroll
            for (int di = 0; di < 3; ++di)
#pragma unroll
                for (int kk = 0; kk < TC_PIX / 16; ++kk)
                    mma_f16(taddr + 128 * (it & 1u) + 32 * di, a0 + (uint32_t)(di * Wv + 16 * kk), b0 + 16 * kk, idesc, kk > 0);
            mma_commit(bar + (it & 1u));
        }
        // the stage of the previous tile takes the tile NS - 1 ahead
        if (it > 0) ok = tc_wait(bar + ((it - 1) & 1u), ((it - 1) >> 1) & 1u);
        if (__syncthreads_or(!ok)) {
            ok = false;
            break;
        }
        const int free_st = st == 0 ? NS - 1 : st - 1;
        load(free_st);
        if (it > 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            tmem_add48(acc, own + 128 * ((it - 1) & 1u));
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        }
        st = st + 1 == NS ? 0 : st + 1;
    }
    if (ok && it > 0) ok = tc_wait(bar + ((it - 1) & 1u), ((it - 1) >> 1) & 1u);
    wait_copies<0>();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    ok = !__syncthreads_or(!ok);
    if (ok && it > 0) tmem_add48(acc, own + 128 * ((it - 1) & 1u));
    float* out = part + ((long long)blockIdx.x * 96 + 48 * (warp >> 2)) * 128 + 32 * (warp & 3) + lane;
#pragma unroll
    for (int i = 0; i < 48; ++i) out[i * 128] = ok ? acc[i] : __int_as_float(0x7fc00000);
    if (!ok && tid == 0) atomicAdd(&g_conv_timeouts, 1ull);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(taddr) : "memory");
}

// dw[n][c][di][dj] = the sum of the S partials in wgrad_reduce_kernel's order
__global__ void __launch_bounds__(32 * WR_SPLIT) wgrad_cl_reduce_kernel(const float* __restrict__ part, int S, int M, int C,
                                                                       int GX, float* __restrict__ dw) {
    const int idx = blockIdx.x * 32 + threadIdx.x, R = idx & 127, col = idx >> 7;
    const int dj = R / (8 * GX), c = R - dj * 8 * GX, di = col >> 5, n = col & 31;
    const bool used = dj < 3 && c < C && n < M;
    const float s = split_sum(part + idx, S, 96 * 128, used);
    if (threadIdx.y == 0 && used) dw[(n * C + c) * 9 + 3 * di + dj] = s;
}

size_t wgrad_cl_smem(int GX, int GY, int Wv, int NS) {
    const size_t plane = (size_t)pad_rows(TC_PIX + 2 * Wv) * 16, stage = 3 * GX * plane + (size_t)GY * (TC_PIX + 2) * 16;
    // the MMAs read 16 planes of the last stage from its highest start on
    const size_t reach = (size_t)(NS - 1) * stage + 16 * plane;
    const size_t all = (size_t)NS * stage;
    return 1024 + (reach > all ? reach : all);
}
// three tiles in shared memory where they fit (strips of up to 88 columns at 32 channels), else two
constexpr size_t WGRAD_CL_SMEM3 = 220 * 1024;
int wgrad_cl_stages(int GX, int GY, int Wv) { return wgrad_cl_smem(GX, GY, Wv, 3) <= WGRAD_CL_SMEM3 ? 3 : 2; }
// the most that any shape takes of a kernel with ns tiles
size_t wgrad_cl_smem_limit(int GX, int GY, int ns) { return ns == 3 ? WGRAD_CL_SMEM3 : wgrad_cl_smem(GX, GY, TC_WT + 2, 2); }

// ------------------------------------------------------------------ layout

__global__ void to_cl_kernel(const bf16* __restrict__ x, int C, int G, long long HW, long long n, bf16* __restrict__ out) {
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n * G; e += (long long)gridDim.x * blockDim.x) {
        const int g = (int)(e % G);
        const long long pos = e / G, b = pos / HW, p = pos - b * HW;
        const bf16* q = x + (b * C) * HW + p;
        uint32_t w[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int c = 8 * g + 2 * u;
            const bf16 zero = __float2bfloat16_rn(0.f);
            w[u] = pack2(c < C ? q[c * HW] : zero, c + 1 < C ? q[(c + 1) * HW] : zero);
        }
        reinterpret_cast<uint4*>(out)[e] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

// ------------------------------------------------------------------ optimiser

struct AdamLayers {
    tlbm_conv_layer l[TLBM_CONV_MAX_LAYERS];
};

// Adam (Kingma & Ba 2015) on every layer's FP32 weights and biases, and the new
// weights into the packed operands: one launch for the network (block.y = layer).
__global__ void adam_layers_kernel(const __grid_constant__ AdamLayers a, float lr, float b1, float b2, float eps, float c1,
                                   float c2) {
    const tlbm_conv_layer& q = a.l[blockIdx.y];
    const int nw = q.cout * q.cin * 9, n = nw + q.cout;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const bool isw = i < nw;
    const int k = isw ? i : i - nw;
    float* w = isw ? q.w : q.b;
    float* m = isw ? q.mw : q.mb;
    float* v = isw ? q.vw : q.vb;
    const float g = (isw ? q.gw : q.gb)[k];
    const float mi = b1 * m[k] + (1.f - b1) * g;
    const float vi = b2 * v[k] + (1.f - b2) * g * g;
    m[k] = mi;
    v[k] = vi;
    const float wn = w[k] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    w[k] = wn;
    if (isw) {
        const int o = k / (q.cin * 9), r = k - o * q.cin * 9, c = r / 9, t = r - c * 9;
        const int CH = (q.cin + 15) / 16, h = c >> 4, cc = c & 15;
        static_cast<bf16*>(q.a)[512 * (t * CH + h) + 256 * (cc >> 3) + 64 * (o >> 3) + 8 * (o & 7) + (cc & 7)] = __float2bfloat16_rn(wn);
    }
}

int launch_conv_cl(const bf16* A, int M, const bf16* x, int B, int C, int H, int W, const float* bias, int relu, float* y,
                   bf16* act, const bf16* mask, float* sums, long long grid, cudaStream_t s) {
    const TcGeom geo = tc_geometry(B, H, W);
    const int G = groups_of(C);
    const size_t smem = conv_cl_smem(G, geo.Wv);
    auto* fn = mask ? (G == 2 ? conv_cl_kernel<2, true> : conv_cl_kernel<4, true>)
                    : (G == 2 ? conv_cl_kernel<2, false> : conv_cl_kernel<4, false>);
    // (the limit belongs to the kernel, not to the launch: that of the widest strip,
    // whatever the shape, so that threads with other shapes never lower it)
    if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)conv_cl_smem(G, TC_WT + 2)) != cudaSuccess)
        return TLBM_ERR_CUDA;
    fn<<<(unsigned)grid, CL_THREADS, smem, s>>>(A, M, x, H, W, bias, relu, y, act, mask, sums, geo);
    return status_of(cudaGetLastError());
}

int conv_cl_grid(bool grad, int B, int C, int H, int W, long long* grid) {
    const TcGeom geo = tc_geometry(B, H, W);
    // as many CTAs as an SM's registers hold
    return persistent_grid(geo.tiles, conv_cl_smem(groups_of(C), geo.Wv), grad ? 4 : 6, grid);
}

int wgrad_cl_grid(int B, int cin, int cout, int H, int W, long long* grid) {
    const TcGeom geo = tc_geometry(B, H, W);
    const int GX = groups_of(cin), GY = groups_of(cout);
    return persistent_grid(geo.tiles, wgrad_cl_smem(GX, GY, geo.Wv, wgrad_cl_stages(GX, GY, geo.Wv)), 2, grid);
}

}  // namespace

extern "C" int tlbm_conv_channels_last(const void* x, int B, int C, int H, int W, void* out, void* stream) {
    if (!x || !out || !aligned16(out) || !conv_shape_ok(B, C, C, H, W)) return TLBM_ERR_ARG;
    const long long n = (long long)B * H * W;
    const int G = groups_of(C);
    to_cl_kernel<<<grid_for(n * G, 256), 256, 0, (cudaStream_t)stream>>>((const bf16*)x, C, G, (long long)H * W, n, (bf16*)out);
    return status_of(cudaGetLastError());
}

extern "C" int tlbm_conv3x3_forward_cl(const void* x, const void* a, const float* bias, float* y, void* act, int B, int cin,
                                       int cout, int H, int W, int relu, void* stream) {
    if (!x || !a || (!y && !act) || !aligned16(x) || !aligned16(a) || !aligned16(act) || !conv_shape_ok(B, cin, cout, H, W))
        return TLBM_ERR_ARG;
    long long grid = 0;
    if (conv_cl_grid(false, B, cin, H, W, &grid) != TLBM_OK) return TLBM_ERR_CUDA;
    return launch_conv_cl((const bf16*)a, cout, (const bf16*)x, B, cin, H, W, bias, relu, y, (bf16*)act, nullptr, nullptr,
                          grid, (cudaStream_t)stream);
}

extern "C" int tlbm_conv3x3_cl_workspace_bytes(int B, int cin, int cout, int H, int W, size_t* bytes) {
    if (!bytes || !conv_shape_ok(B, cin, cout, H, W)) return TLBM_ERR_ARG;
    long long S = 0, Gd = 0;
    if (wgrad_cl_grid(B, cin, cout, H, W, &S) != TLBM_OK || conv_cl_grid(true, B, cout, H, W, &Gd) != TLBM_OK) return TLBM_ERR_CUDA;
    const size_t wg = (size_t)S * 96 * 128 * sizeof(float);
    const size_t dg = (size_t)32 * 288 * sizeof(bf16) + (size_t)Gd * 32 * sizeof(float);
    *bytes = wg > dg ? wg : dg;
    return TLBM_OK;
}

extern "C" int tlbm_conv3x3_backward_data_cl(const void* dy, const float* w, const void* act, void* g, float* db, int B,
                                             int cin, int cout, int H, int W, void* workspace, size_t workspace_bytes,
                                             void* stream) {
    if (!dy || !w || !act || !g || !db || !workspace || !aligned16(dy) || !aligned16(act) || !aligned16(g) ||
        !aligned16(workspace) || !conv_shape_ok(B, cout, cin, H, W))
        return TLBM_ERR_ARG;
    size_t need = 0;
    tlbm_conv3x3_cl_workspace_bytes(B, cin, cout, H, W, &need);
    if (workspace_bytes < need) return TLBM_ERR_OOM;
    long long grid = 0;
    if (conv_cl_grid(true, B, cout, H, W, &grid) != TLBM_OK) return TLBM_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    bf16* at = (bf16*)workspace;
    float* sums = (float*)((char*)workspace + (size_t)32 * 288 * sizeof(bf16));
    int rc = flip_weights(w, cout, cin, at, s);
    if (rc == TLBM_OK)
        rc = launch_conv_cl(at, cin, (const bf16*)dy, B, cout, H, W, nullptr, 0, nullptr, (bf16*)g, (const bf16*)act, sums,
                            grid, s);
    if (rc != TLBM_OK) return rc;
    sum_rows_kernel<<<1, 1024, 0, s>>>(sums, (int)grid, cin, db);
    return status_of(cudaGetLastError());
}

extern "C" int tlbm_conv3x3_backward_weight_cl(const void* x, const void* dy, float* dw, int B, int cin, int cout, int H,
                                               int W, void* workspace, size_t workspace_bytes, void* stream) {
    if (!x || !dy || !dw || !workspace || !aligned16(x) || !aligned16(dy) || !conv_shape_ok(B, cin, cout, H, W))
        return TLBM_ERR_ARG;
    size_t need = 0;
    tlbm_conv3x3_cl_workspace_bytes(B, cin, cout, H, W, &need);
    if (workspace_bytes < need) return TLBM_ERR_OOM;
    const TcGeom geo = tc_geometry(B, H, W);
    const int GX = groups_of(cin), GY = groups_of(cout);
    const int ns = wgrad_cl_stages(GX, GY, geo.Wv);
    const size_t smem = wgrad_cl_smem(GX, GY, geo.Wv, ns);
    using Fn = void (*)(const bf16*, int, const bf16*, int, int, int, TcGeom, float*);
    static const Fn fns[2][2][2] = {{{wgrad_cl_kernel<2, 2, 2>, wgrad_cl_kernel<2, 2, 3>},
                                     {wgrad_cl_kernel<2, 4, 2>, wgrad_cl_kernel<2, 4, 3>}},
                                    {{wgrad_cl_kernel<4, 2, 2>, wgrad_cl_kernel<4, 2, 3>},
                                     {wgrad_cl_kernel<4, 4, 2>, wgrad_cl_kernel<4, 4, 3>}}};
    const Fn fn = fns[GX == 4][GY == 4][ns == 3];
    long long S = 0;
    if (wgrad_cl_grid(B, cin, cout, H, W, &S) != TLBM_OK ||
        cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wgrad_cl_smem_limit(GX, GY, ns)) != cudaSuccess)
        return TLBM_ERR_CUDA;
    cudaStream_t s = (cudaStream_t)stream;
    fn<<<(unsigned)S, WG_THREADS, smem, s>>>((const bf16*)dy, cout, (const bf16*)x, cin, H, W, geo, (float*)workspace);
    if (cudaGetLastError() != cudaSuccess) return TLBM_ERR_CUDA;
    wgrad_cl_reduce_kernel<<<96 * 128 / 32, dim3(32, WR_SPLIT), 0, s>>>((const float*)workspace, (int)S, cout, cin, GX, dw);
    return status_of(cudaGetLastError());
}

extern "C" int tlbm_conv_adam_layers(const tlbm_conv_layer* layers, int n, float lr, float b1, float b2, float eps, int t,
                                     void* stream) {
    if (!layers || n < 1 || n > TLBM_CONV_MAX_LAYERS || t < 1) return TLBM_ERR_ARG;
    AdamLayers a{};
    int most = 0;
    for (int i = 0; i < n; ++i) {
        const tlbm_conv_layer& q = layers[i];
        if (!q.w || !q.gw || !q.mw || !q.vw || !q.b || !q.gb || !q.mb || !q.vb || !q.a || q.cout < 1 || q.cout > 32 ||
            q.cin < 1 || q.cin > 32)
            return TLBM_ERR_ARG;
        a.l[i] = q;
        const int e = q.cout * q.cin * 9 + q.cout;
        most = e > most ? e : most;
    }
    const float c1 = 1.f - powf(b1, (float)t), c2 = 1.f - powf(b2, (float)t);
    adam_layers_kernel<<<dim3((most + 127) / 128, n), 128, 0, (cudaStream_t)stream>>>(a, lr, b1, b2, eps, c1, c2);
    return status_of(cudaGetLastError());
}
