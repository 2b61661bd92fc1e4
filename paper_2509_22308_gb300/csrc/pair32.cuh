// The FP32 site update on two sites at once (one lane's pair of adjacent columns), with the
// packed FP32 instructions of sm_100 and later (add, sub, mul and fma on f32x2: two independent,
// separately rounded FP32 operations per instruction).
//
// They run at the scalar instructions' lane rate (measured on GB300: 125 against 124 operations
// per clock and SM) but take half the issue slots, and the FP32 kernels that use them are bound by how
// many instructions a warp has to get through one after the other, not by the pipe.  Pairs stay in 64-bit registers throughout: with float2 structs the compiler
// moved halves about (one update in a loop: 46 instructions and 135 clocks of latency as float2,
// 39 and 94 as below; 72 clocks of the FP32 pipe either way; scalar: 73 instructions, 171 clocks).
// Each half is rounded as the scalar operation, and every expression below is the one of
// moments() / collide() (common.cuh) in the same order, so the results are the scalar kernels' bits.
#pragma once

#include "common.cuh"

namespace lbmem {

struct alignas(8) f2 {
    unsigned long long v;
};
__device__ __forceinline__ f2 pack2(float x, float y) {
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ float lo2(f2 a) {
    return __uint_as_float((unsigned)a.v);
}
__device__ __forceinline__ float hi2(f2 a) {
    return __uint_as_float((unsigned)(a.v >> 32));
}
__device__ __forceinline__ f2 both(float v) { return pack2(v, v); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 sub2(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}

// quot() of common.cuh for both halves; nden = -den (the product (-q) den is exactly q (-den)).
__device__ __forceinline__ f2 quot2(f2 num, f2 nden, f2 inv) {
    const f2 q = mul2(num, inv);
    return fma2(fma2(q, nden, num), inv, q);
}

// max(|m|, |a|, |b|), NaN if any of them is one.
__device__ __forceinline__ float amax3(float m, float a, float b) {
    float r;
    asm("max.NaN.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(m), "f"(a), "f"(b));
    return r;
}

// Material constants of the two sites: MatT<float> with -c3.
struct PairMat {
    f2 inv3, cd, inv, nc3;
};
__device__ __forceinline__ PairMat pair_mat(const MatT<float> &a, const MatT<float> &b) {
    return PairMat{pack2(a.inv_eps3, b.inv_eps3), pack2(a.c_d, b.c_d), pack2(a.inv_eps, b.inv_eps),
                   pack2(-a.c3, -b.c3)};
}

// moments() (TM) of both sites.
__device__ __forceinline__ void moments_pair(const Pop<f2> &p, const PairMat &m, f2 &E3, f2 &Hx, f2 &Hy, f2 &d) {
    const f2 two = both(2.0f);
    d = add2(add2(add2(fma2(m.cd, p.ez, p.epx), p.emx), p.epy), p.emy);
    E3 = quot2(d, m.nc3, m.inv3);
    Hx = add2(fma2(two, p.hxz, add2(p.hxpx, p.hxmx)), sub2(p.epy, p.emy));
    Hy = add2(fma2(two, p.hyz, add2(p.hypy, p.hymy)), sub2(p.emx, p.epx));
}

// Moments and collision of both sites.  e3: per site the field (of TE the larger one) whose
// exponent field decides the runaway test; the exponent field of a maximum over many of them
// (amax3) is field_runaway() over each.  F3: the field triple of update_site() in FP32 to f3.
template <int POL, bool F3>
__device__ __forceinline__ void update_pair(Pop<f2> &p, const PairMat &m, f2 &e3, f2 *f3) {
    const f2 third = both(1.0f / 3.0f), n3 = both(-3.0f), two = both(2.0f);
    if constexpr (POL == POL_TM) {
        f2 E3, Hx, Hy, d;
        moments_pair(p, m, E3, Hx, Hy, d);
        e3 = E3;
        if (F3) {
            f3[0] = mul2(d, m.inv);
            f3[1] = Hx;
            f3[2] = Hy;
        }
        const f2 hx3 = quot2(Hx, n3, third), hy3 = quot2(Hy, n3, third);
        p.ez = sub2(E3, p.ez);
        p.epx = sub2(sub2(E3, hy3), p.epx);
        p.emx = sub2(add2(E3, hy3), p.emx);
        p.epy = sub2(add2(E3, hx3), p.epy);
        p.emy = sub2(sub2(E3, hx3), p.emy);
        p.hxpx = sub2(hx3, p.hxpx);
        p.hxmx = sub2(hx3, p.hxmx);
        p.hxz = sub2(hx3, p.hxz);
        p.hypy = sub2(hy3, p.hypy);
        p.hymy = sub2(hy3, p.hymy);
        p.hyz = sub2(hy3, p.hyz);
    } else {
        const f2 d = add2(add2(add2(fma2(m.cd, p.ez, p.epx), p.emx), p.epy), p.emy);
        const f2 E3 = quot2(d, m.nc3, m.inv3);
        const f2 dx = add2(add2(add2(fma2(m.cd, p.hxz, p.hxpx), p.hxmx), p.hypy), p.hymy);
        const f2 Ex3 = quot2(dx, m.nc3, m.inv3);
        const f2 Hz = add2(fma2(two, p.hyz, sub2(p.epx, p.emx)), sub2(p.hymy, p.hypy));
        e3 = pack2(amax3(0.f, lo2(E3), lo2(Ex3)), amax3(0.f, hi2(E3), hi2(Ex3)));
        if (F3) {
            f3[0] = Hz;
            f3[1] = mul2(dx, m.inv);
            f3[2] = mul2(d, m.inv);
        }
        const f2 hz3 = quot2(Hz, n3, third);
        p.epx = sub2(add2(E3, hz3), p.epx);
        p.emx = sub2(sub2(E3, hz3), p.emx);
        p.hypy = sub2(sub2(Ex3, hz3), p.hypy);
        p.hymy = sub2(add2(Ex3, hz3), p.hymy);
        p.hyz = sub2(hz3, p.hyz);
        p.ez = sub2(E3, p.ez);
        p.epy = sub2(E3, p.epy);
        p.emy = sub2(E3, p.emy);
        p.hxpx = sub2(Ex3, p.hxpx);
        p.hxmx = sub2(Ex3, p.hxmx);
        p.hxz = sub2(Ex3, p.hxz);
    }
}

}  // namespace lbmem
