// Double-float arithmetic (df32.cuh) on two sites at once with packed FP32 instructions: the operations,
// their order and so the results are df's (up to the sign of zeros).  A packed instruction works
// through the pipe at the scalar rate per site but takes one issue slot for two; a double-float
// update is 536 of them (TM; the scalar form's expressions 652) and hardly anything else, so the scalar
// kernel was bound by issue.
#pragma once

#include "common.cuh"
#include "pair32.cuh"

namespace lbmem {

struct df2 {
    f2 hi, lo;
};
__device__ __forceinline__ df2 pack_df(df a, df b) { return df2{pack2(a.hi, b.hi), pack2(a.lo, b.lo)}; }
__device__ __forceinline__ df first(df2 v) { return df(lo2(v.hi), lo2(v.lo)); }
__device__ __forceinline__ df second(df2 v) { return df(hi2(v.hi), hi2(v.lo)); }

__device__ __forceinline__ df2 two_sum(f2 a, f2 b) {
    const f2 s = add2(a, b), bb = sub2(s, a);
    return df2{s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ df2 two_diff(f2 a, f2 b) {  // two_sum(a, -b)
    const f2 s = sub2(a, b), bb = sub2(s, a);
    return df2{s, sub2(sub2(a, sub2(s, bb)), add2(b, bb))};
}
__device__ __forceinline__ df2 fast_two_sum(f2 a, f2 b) {
    const f2 s = add2(a, b);
    return df2{s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ df2 join(df2 s, df2 t) {
    const df2 v = fast_two_sum(s.hi, add2(s.lo, t.hi));
    return fast_two_sum(v.hi, add2(t.lo, v.lo));
}
__device__ __forceinline__ df2 operator+(df2 a, df2 b) { return join(two_sum(a.hi, b.hi), two_sum(a.lo, b.lo)); }
__device__ __forceinline__ df2 operator-(df2 a, df2 b) { return join(two_diff(a.hi, b.hi), two_diff(a.lo, b.lo)); }
__device__ __forceinline__ df2 operator*(df2 a, df2 b) {
    const f2 ch = mul2(a.hi, b.hi), cl1 = fma2(a.hi, b.hi, f2{ch.v ^ 0x8000000080000000ull});
    return fast_two_sum(ch, add2(cl1, fma2(a.lo, b.hi, mul2(a.hi, b.lo))));
}
__device__ __forceinline__ df2 twice(df2 a) { return df2{add2(a.hi, a.hi), add2(a.lo, a.lo)}; }  // exact

// Moments and collision of both sites (moments, collide, moments_te, collide_te of common.cuh for df).
// A product with -1/3 is the negated product with 1/3, and one with 2 is exact, so each H/3 is
// formed once.  Returns whether site A's or (with_b) site B's field ran away; F3: the field triple of
// update_site() to f3.
template <int POL, bool F3 = false>
__device__ __forceinline__ bool update_pair(Pop<df2> &p, const MatT<df> &ma, const MatT<df> &mb, bool with_b,
                                            unsigned rthr, df2 *f3 = nullptr) {
    const df2 cd = pack_df(ma.c_d, mb.c_d), inv3 = pack_df(ma.inv_eps3, mb.inv_eps3);
    const df t3((double)(1.0 / 3.0));
    const df2 third = pack_df(t3, t3);
    if constexpr (POL == POL_TM) {
        const df2 d = cd * p.ez + p.epx + p.emx + p.epy + p.emy;
        const df2 E = d * inv3;
        const df2 Hx = (twice(p.hxz) + (p.hxpx + p.hxmx)) + (p.epy - p.emy);
        const df2 Hy = (twice(p.hyz) + (p.hypy + p.hymy)) + (p.emx - p.epx);
        if (F3) f3[0] = d * pack_df(ma.inv_eps, mb.inv_eps), f3[1] = Hx, f3[2] = Hy;
        const df2 hx3 = Hx * third, hy3 = Hy * third;
        p.ez = E - p.ez;
        p.epx = (E - hy3) - p.epx;
        p.emx = (E + hy3) - p.emx;
        p.epy = (E + hx3) - p.epy;
        p.emy = (E - hx3) - p.emy;
        p.hxpx = hx3 - p.hxpx;
        p.hxmx = hx3 - p.hxmx;
        p.hxz = hx3 - p.hxz;
        p.hypy = hy3 - p.hypy;
        p.hymy = hy3 - p.hymy;
        p.hyz = hy3 - p.hyz;
        return field_runaway(first(E), rthr) || (with_b && field_runaway(second(E), rthr));
    } else {
        const df2 dy = cd * p.ez + p.epx + p.emx + p.epy + p.emy;
        const df2 dx = cd * p.hxz + p.hxpx + p.hxmx + p.hypy + p.hymy;
        const df2 Ey = dy * inv3, Ex = dx * inv3;
        const df2 Hz = (twice(p.hyz) + (p.epx - p.emx)) + (p.hymy - p.hypy), hz3 = Hz * third;
        if (F3) {
            const df2 inv = pack_df(ma.inv_eps, mb.inv_eps);
            f3[0] = Hz, f3[1] = dx * inv, f3[2] = dy * inv;
        }
        p.epx = (Ey + hz3) - p.epx;
        p.emx = (Ey - hz3) - p.emx;
        p.hypy = (Ex - hz3) - p.hypy;
        p.hymy = (Ex + hz3) - p.hymy;
        p.hyz = hz3 - p.hyz;
        p.ez = Ey - p.ez;
        p.epy = Ey - p.epy;
        p.emy = Ey - p.emy;
        p.hxpx = Ex - p.hxpx;
        p.hxmx = Ex - p.hxmx;
        p.hxz = Ex - p.hxz;
        return field_runaway(first(Ey), rthr) || field_runaway(first(Ex), rthr) ||
               (with_b && (field_runaway(second(Ey), rthr) || field_runaway(second(Ex), rthr)));
    }
}

// f(packed, a's, b's) for the eleven populations.
template <typename P, typename A, typename F>
__device__ __forceinline__ void each_of_pair(P &p, A &a, A &b, F f) {
    f(p.ez, a.ez, b.ez);
    f(p.epx, a.epx, b.epx);
    f(p.emx, a.emx, b.emx);
    f(p.epy, a.epy, b.epy);
    f(p.emy, a.emy, b.emy);
    f(p.hxpx, a.hxpx, b.hxpx);
    f(p.hxmx, a.hxmx, b.hxmx);
    f(p.hxz, a.hxz, b.hxz);
    f(p.hypy, a.hypy, b.hypy);
    f(p.hymy, a.hymy, b.hymy);
    f(p.hyz, a.hyz, b.hyz);
}

}  // namespace lbmem
