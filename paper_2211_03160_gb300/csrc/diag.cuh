// Macroscopic fields and reduction terms of a state's nodes (§2.2: rho = sum f,
// T = sum g, u = (sum e f + F/2) / rho), shared by the diagnostic kernels.
#pragma once
#include "kernels.cuh"

namespace tlbm {

// Per-call constants of the diagnostic kernels, formed on the host: the element
// offset, relative to a node's own slot in plane 0, of each population's
// pre-collision value in the state's order (flow planes first), and gbeta / 2
// and body / 2 as unevaluated sums of two FP32 values.
struct DiagOff {
    int off[MAXQ + 7];
    float gh, gl, bh[3], bl[3];
};
template <int DIM>
inline DiagOff diag_offsets(const KParams& p) {
    using LF = typename Lat<DIM>::F;
    using LG = typename Lat<DIM>::G;
    DiagOff o{};
    o.gh = (float)(0.5 * p.gbeta);
    o.gl = (float)(0.5 * p.gbeta - (double)o.gh);
    for (int a = 0; a < 3; ++a) {
        o.bh[a] = (float)(0.5 * p.body[a]);
        o.bl[a] = (float)(0.5 * p.body[a] - (double)o.bh[a]);
    }
    auto one = [&](int plane, int opp, int ex, int ey, int ez) {
        if (p.state == 1) return (int)(plane * p.L.plane);
        return (int)((p.state == 2 ? opp : plane) * p.L.plane - ez * (long long)p.rp - ey * p.L.P - ex);
    };
    for (int i = 0; i < LF::Q; ++i) o.off[i] = one(i, LF::opp(i), LF::e(i, 0), LF::e(i, 1), LF::e(i, 2));
    for (int i = 0; i < LG::Q; ++i)
        o.off[LF::Q + i] = one(LF::Q + i, LF::Q + LG::opp(i), LG::e(i, 0), LG::e(i, 1), LG::e(i, 2));
    return o;
}

// The stored values of one node: flow as the storage keeps it (deviations in offset
// storage, f_i in FP64), in FP32 unscaled.  FP64 leaves the storage scale to the
// sums (a power of two: the same bits), one multiplication each instead of one
// per value.
template <int DIM, class S, class C>
__device__ __forceinline__ void diag_load(const S* __restrict__ own, const KParams& p, const int* off,
                                          C (&f)[Lat<DIM>::F::Q], C (&g)[Lat<DIM>::G::Q]) {
    constexpr int QF = Lat<DIM>::F::Q, QG = Lat<DIM>::G::Q;
#pragma unroll
    for (int i = 0; i < QF; ++i) f[i] = to_c<C>(ld_one<S, false>(TLBM_DBG(p, (own + off[i]), 0, 1)));
#pragma unroll
    for (int i = 0; i < QG; ++i) g[i] = to_c<C>(ld_one<S, false>(TLBM_DBG(p, (own + off[QF + i]), 0, 1)));
    if constexpr (Storage<S>::scaled && std::is_same<C, float>::value) {
        const C inv = ScaleOf<C>::inv(p);
#pragma unroll
        for (int i = 0; i < QF; ++i) f[i] *= inv;
#pragma unroll
        for (int i = 0; i < QG; ++i) g[i] *= inv;
    }
}

// FP64 macros.  The antisymmetric and symmetric parts of each pair are formed
// once and shared by the density and the momenta: 34 (2D) / 68 (3D) FP64
// operations and, for the other storages, the conversions.
template <int DIM, class S>
__device__ __forceinline__ void diag_macros_d(const S* __restrict__ own, const KParams& p, const int* off, double& rho,
                                              double (&u)[3], double& T) {
    using LF = typename Lat<DIM>::F;
    using LG = typename Lat<DIM>::G;
    double f[LF::Q], g[LG::Q];
    diag_load<DIM, S, double>(own, p, off, f, g);
    constexpr bool raw = !Storage<S>::offset;  // f_i rather than deviations
    double drho = raw ? dsub(f[0], weight<LF, double>(0)) : f[0];
    double j[3] = {0.0, 0.0, 0.0};
    static_for<LF::Q>([&](auto ii) {
        constexpr int i = decltype(ii)::value, o = LF::opp(i);
        if constexpr (i != 0 && i < o) {
            const double a = dsub(f[i], f[o]);
            drho = dadd(drho, dadd(raw ? dsub(f[i], 2.0 * weight<LF, double>(i)) : f[i], f[o]));
            static_for<DIM>([&](auto aa) {
                constexpr int ax = decltype(aa)::value;
                if constexpr (i == axis_pop<LF>(ax)) j[ax] = a;  // the axis pairs come first
                else if constexpr (LF::e(i, ax) == 1) j[ax] = dadd(j[ax], a);
                else if constexpr (LF::e(i, ax) == -1) j[ax] = dsub(j[ax], a);
            });
        }
    });
    T = g[0];
#pragma unroll
    for (int i = 1; i < LG::Q; ++i) T = dadd(T, g[i]);
    if constexpr (Storage<S>::scaled) {
        const double inv = ScaleOf<double>::inv(p);
        drho = dmul(drho, inv);
        T = dmul(T, inv);
#pragma unroll
        for (int ax = 0; ax < DIM; ++ax) j[ax] = dmul(j[ax], inv);
    }
    rho = dadd(1.0, drho);
    // the fast reciprocal within FP32's range, IEEE division outside it
    const double ir = rho > 1e-30 && rho < 1e30 ? drcp(rho) : 1.0 / rho;
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) u[ax] = 0.0;
#pragma unroll
    for (int ax = 0; ax < DIM; ++ax) {
        const double b = ax == DIM - 1 ? dfma(p.gbeta, T, p.body[ax]) : p.body[ax];
        u[ax] = dmul(dfma(0.5, dmul(rho, b), j[ax]), ir);
    }
}

// An unevaluated sum h + l of two FP32 values (about 48 bits).
struct Df {
    float h, l;
};
// a + b exactly (Knuth's two-sum)
__device__ __forceinline__ Df two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ void df_add(Df& a, float b) {
    const Df t = two_sum(a.h, b);
    a.h = t.h;
    a.l = __fadd_rn(a.l, t.l);
}
__device__ __forceinline__ float df_val(Df a) { return __fadd_rn(a.h, a.l); }

// FP32 fields of a node of FP32 / FP16 / BF16 storage, rounded from double-FP32
// arithmetic: the sums are exact to the last bits of the low words (about
// 2^-46), so the results are those of FP64 arithmetic rounded to FP32, except
// where a rounding boundary falls between the two (a few nodes in a million, each
// within 0.5001 units).  The same in FP64 took 51 FP64-pipe operations
// (conversions included) per node in 2D: the fields of an 8193^2 FP32 state 7.36
// ms, now 0.88 (5.5 TB/s); of a 385^3 FP16 state 11.5 ms, now 1.26.
// false: some value is outside the range where this holds (the caller then
// evaluates the node in FP64).
template <int DIM>
__device__ __forceinline__ bool diag_macros_f(const float (&f)[Lat<DIM>::F::Q], const float (&g)[Lat<DIM>::G::Q],
                                              const DiagOff& k, float& rho, float (&u)[3], float& T) {
    using LF = typename Lat<DIM>::F;
    using LG = typename Lat<DIM>::G;
    Df dr = {f[0], 0.0f}, j[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}}, t = {g[0], 0.0f};
    static_for<LF::Q>([&](auto ii) {
        constexpr int i = decltype(ii)::value;
        if constexpr (i > 0) df_add(dr, f[i]);
        static_for<DIM>([&](auto aa) {
            constexpr int ax = decltype(aa)::value;
            if constexpr (i == axis_pop<LF>(ax)) j[ax].h = f[i];
            else if constexpr (LF::e(i, ax) == 1) df_add(j[ax], f[i]);
            else if constexpr (LF::e(i, ax) == -1) df_add(j[ax], -f[i]);
        });
    });
    static_for<LG::Q>([&](auto ii) {
        constexpr int i = decltype(ii)::value;
        if constexpr (i > 0) df_add(t, g[i]);
    });
    // where terms cancel, much of a sum may stand in its low word, whose 24 bits then
    // decide: bring it up (always doing so took 8 % longer in 3D FP32)
    bool low = fabsf(t.l) > 0x1p-12f * fabsf(t.h);
#pragma unroll
    for (int ax = 0; ax < DIM; ++ax) low |= fabsf(j[ax].l) > 0x1p-12f * fabsf(j[ax].h);
    if (low) {
#pragma unroll
        for (int ax = 0; ax < DIM; ++ax) j[ax] = two_sum(j[ax].h, j[ax].l);
        t = two_sum(t.h, t.l);
    }
    Df r = two_sum(1.0f, dr.h);
    r.l = __fadd_rn(r.l, dr.l);
    rho = df_val(r);
    T = df_val(t);
    constexpr float BIG = 1e15f;
    if (!(rho > 1e-15f && rho < BIG && fabsf(T) < BIG && fabsf(j[0].h) < BIG && fabsf(j[1].h) < BIG &&
          fabsf(j[2].h) < BIG))
        return false;
    const float ir = __frcp_rn(r.h);
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) u[ax] = 0.0f;
#pragma unroll
    for (int ax = 0; ax < DIM; ++ax) {
        // q + c = j / rho: one Newton correction of the FP32 quotient
        const float q = __fmul_rn(j[ax].h, ir);
        const float rem = __fadd_rn(__fmaf_rn(-q, r.h, j[ax].h), __fmaf_rn(-q, r.l, j[ax].l));
        float c = __fmul_rn(rem, ir);
        // + F / (2 rho) = (gbeta T + body) / 2
        Df b = {k.bh[ax], k.bl[ax]};
        if (ax == DIM - 1) {
            const float m = __fmul_rn(k.gh, t.h);
            const float ml = __fadd_rn(__fmaf_rn(k.gh, t.h, -m), __fmaf_rn(k.gh, t.l, __fmul_rn(k.gl, t.h)));
            const float l0 = b.l;
            b = two_sum(m, b.h);
            b.l = __fadd_rn(b.l, __fadd_rn(l0, ml));
        }
        const Df v = two_sum(q, b.h);
        c = __fadd_rn(c, __fadd_rn(b.l, v.l));
        u[ax] = __fadd_rn(v.h, c);
    }
    return true;
}

// Per-node terms of the reductions (a6): u_h T, 1/2 rho |u|^2, rho, |u|^2, T,
// formed in the storage's collision precision (FP64 storage: FP64; otherwise
// FP32, the precision the state was computed in, with operations the compiler
// does not contract, so that every kernel forms the same terms).
template <int DIM, class S>
__device__ __forceinline__ void node_terms(const S* __restrict__ own, const KParams& p, const int* off,
                                           typename Storage<S>::C (&t)[5]) {
    using C = typename Storage<S>::C;
    if constexpr (std::is_same<C, double>::value) {
        double rho, u[3], T;
        diag_macros_d<DIM, S>(own, p, off, rho, u, T);
        const double u2 = dfma(u[0], u[0], dfma(u[1], u[1], dmul(u[2], u[2])));
        t[0] = dmul(p.heat_axis == 0 ? u[0] : u[DIM - 1], T);
        t[1] = dmul(dmul(0.5, rho), u2);
        t[2] = rho;
        t[3] = u2;
        t[4] = T;
    } else {
        using LF = typename Lat<DIM>::F;
        using LG = typename Lat<DIM>::G;
        float f[LF::Q], g[LG::Q];
        diag_load<DIM, S, float>(own, p, off, f, g);
        float drho = f[0], j[3] = {0.0f, 0.0f, 0.0f}, T = g[0], u[3] = {0.0f, 0.0f, 0.0f};
        static_for<LF::Q>([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            if constexpr (i > 0) drho = vadd(drho, f[i]);
            static_for<DIM>([&](auto aa) {
                constexpr int ax = decltype(aa)::value;
                if constexpr (i == axis_pop<LF>(ax)) j[ax] = f[i];
                else if constexpr (LF::e(i, ax) == 1) j[ax] = vadd(j[ax], f[i]);
                else if constexpr (LF::e(i, ax) == -1) j[ax] = vsub(j[ax], f[i]);
            });
        });
        static_for<LG::Q>([&](auto ii) {
            constexpr int i = decltype(ii)::value;
            if constexpr (i > 0) T = vadd(T, g[i]);
        });
        const float rho = vadd(1.0f, drho), ir = vrcp(rho);
#pragma unroll
        for (int ax = 0; ax < DIM; ++ax) {
            const float b = ax == DIM - 1 ? vfma(p.gbetaf, T, p.bodyf[ax]) : p.bodyf[ax];
            u[ax] = vmul(vfma(0.5f, vmul(rho, b), j[ax]), ir);
        }
        const float u2 = vfma(u[0], u[0], vfma(u[1], u[1], vmul(u[2], u[2])));
        t[0] = vmul(p.heat_axis == 0 ? u[0] : u[DIM - 1], T);
        t[1] = vmul(vmul(0.5f, rho), u2);
        t[2] = rho;
        t[3] = u2;
        t[4] = T;
    }
}

}  // namespace tlbm
