// Two samples of one ray at a time, in Blackwell's packed float32 arithmetic
// (fma.rn.f32x2 and the like: one instruction, two results, each rounded as the
// scalar instruction rounds it).  leaf_cost2 gives the bits of two leaf_cost
// calls (series form of the rise) with about half the instructions: the packed
// operations, floors by round-down additions (exact for |x| < 2^22) whose integer
// parts are read off the sum's bits, and one test for the clamps at the tile's
// border, which almost no sample needs.  (A packed multiplication that feeds a packed
// addition may be fused with it, .rn or not: wherever a rounded product is added to
// something, the sum, or the product, is formed with scalar instructions, which are not.
// j * a_hi is exact, fused or not, and the addend of an fma cannot be.)
#pragma once

#include "ss_device.cuh"

namespace ss {

struct F2 {
    unsigned long long v;
};

__device__ __forceinline__ F2 f2(float x, float y) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ F2 f2(float x) { return f2(x, x); }
__device__ __forceinline__ void f2_get(F2 a, float& x, float& y) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(a.v));
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_add_rm(F2 a, F2 b) {   // rounded down
    F2 r;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) { return f2_fma(b, f2(-1.0f), a); }   // exact product

// 1.5 * 2^23: x + kFloorBias rounded down is floor(x) + kFloorBias for |x| < 2^22
constexpr float kFloorBias = 12582912.0f;
constexpr uint32_t kFloorBits = 0x4B400000u;

// axis_pos for two samples, before the clamp: integer parts ia, ib, fractions f.
template <bool kGrid, bool kStereo>
__device__ __forceinline__ F2 axis_pos2(int32_t i0, float u0, float a_hi, float a_lo, float a, F2 corr,
                                        F2 jf, int32_t& ia, int32_t& ib) {
    const F2 bias = f2(kFloorBias);
    const F2 p = f2_mul(jf, f2(a_hi));
    const F2 kb = f2_add_rm(p, bias);
    const F2 fp = f2_sub(p, f2_add(kb, f2(-kFloorBias)));
    const F2 tail = f2_fma(jf, f2(a_lo), f2_mul(f2(kStereo ? -1.0f : -a), corr));
    const F2 s = kGrid ? f2_add(fp, tail)
                       : f2_add(f2_add(f2(__fsub_rn(u0, (float)i0)), fp), tail);
    const F2 sb = f2_add_rm(s, bias);
    const F2 f = f2_sub(s, f2_add(sb, f2(-kFloorBias)));
    float ka, kb2, sa, sb2;
    f2_get(kb, ka, kb2);
    f2_get(sb, sa, sb2);
    const uint32_t z = (uint32_t)i0 - 2u * kFloorBits;   // (modulo 2^32)
    ia = (int32_t)(__float_as_uint(ka) + __float_as_uint(sa) + z);
    ib = (int32_t)(__float_as_uint(kb2) + __float_as_uint(sb2) + z);
    return f;
}

__device__ __forceinline__ void clamp_cell(int32_t& i, float& f, int32_t n) {   // as in axis_pos
    const int32_t c = min(max(i, 0), n - 2);
    f = __fadd_rn(f, (float)(i - c));
    i = c;
}

template <bool kGrid, bool kStereo>
__device__ __forceinline__ void leaf_cost2(const Tile& T, const RayF& r, int32_t ja, int32_t jb,
                                           float& ca, float& cb) {
    const float fa = (float)ja, fb = (float)jb;
    const F2 jf = f2(fa, fb), one = f2(1.0f);
    const F2 t = f2_mul(jf, f2(T.delta_f));
    // rise (rise_of<true>)
    float t0, t1;
    f2_get(t, t0, t1);
    const F2 w = f2_mul(t, f2(__fadd_rn(r.B, t0), __fadd_rn(r.B, t1)));
    const F2 x = f2_mul(w, f2(r.inv_rho2));
    F2 q = f2_fma(x, f2(0.0546875f), f2(-0.078125f));
    q = f2_fma(x, q, f2(0.125f));
    q = f2_fma(x, q, f2(-0.25f));
    q = f2_fma(x, q, one);
    const F2 rise = f2_mul(f2_mul(w, f2(r.inv_2rho)), q);
    // offsets of the image (axis_corr)
    F2 cu, cv;
    if (!kStereo) {
        const F2 jb2 = f2_mul(jf, f2(r.b));
        float n0, n1, d0, d1;
        f2_get(f2_mul(jf, jb2), n0, n1);
        f2_get(jb2, d0, d1);
        cu = cv = f2(__fdividef(n0, __fadd_rn(1.0f, d0)), __fdividef(n1, __fadd_rn(1.0f, d1)));
    } else {
        float n0, n1, d0, d1;
        f2_get(rise, n0, n1);
        n0 = __fadd_rn(n0, __fmul_rn(t0, T.sz_f));
        n1 = __fadd_rn(n1, __fmul_rn(t1, T.sz_f));
        const F2 ws = f2(n0, n1);
        f2_get(f2_fma(ws, f2(r.b), one), d0, d1);
        const F2 k = f2(__fdividef(n0, d0), __fdividef(n1, d1));
        cu = f2_mul(k, f2_fma(f2_mul(jf, f2(r.au)), f2(r.b), f2(r.bu)));
        cv = f2_mul(k, f2_fma(f2_mul(jf, f2(r.av)), f2(r.b), f2(r.bv)));
    }
    int32_t ua, ub, va, vb;
    F2 fu = axis_pos2<kGrid, kStereo>(r.iu0, r.u0, r.au_hi, r.au_lo, r.au, cu, jf, ua, ub);
    F2 fv = axis_pos2<kGrid, kStereo>(r.iv0, r.v0, r.av_hi, r.av_lo, r.av, cv, jf, va, vb);
    const uint32_t mu = (uint32_t)(T.nx - 2), mv = (uint32_t)(T.ny - 2);
    if (max((uint32_t)ua, (uint32_t)ub) > mu || max((uint32_t)va, (uint32_t)vb) > mv) {
        float a, b;
        f2_get(fu, a, b);
        clamp_cell(ua, a, T.nx);
        clamp_cell(ub, b, T.nx);
        fu = f2(a, b);
        f2_get(fv, a, b);
        clamp_cell(va, a, T.ny);
        clamp_cell(vb, b, T.ny);
        fv = f2(a, b);
    }
    const uint32_t pitch = (uint32_t)T.pitch;
    const float* pa = cell_ptr(T.h, pitch, ua, va);
    const float* pb = cell_ptr(T.h, pitch, ub, vb);
    const F2 nh = f2(-r.href);
    const F2 d00 = f2_add(f2(__ldg(pa), __ldg(pb)), nh);
    const F2 d10 = f2_add(f2(__ldg(pa + 1), __ldg(pb + 1)), nh);
    const F2 d01 = f2_add(f2(__ldg(pa + pitch), __ldg(pb + pitch)), nh);
    const F2 d11 = f2_add(f2(__ldg(pa + pitch + 1), __ldg(pb + pitch + 1)), nh);
    const F2 top = f2_fma(fu, f2_sub(d10, d00), d00);
    const F2 bot = f2_fma(fu, f2_sub(d11, d01), d01);
    const F2 hb = f2_fma(fv, f2_sub(bot, top), top);
    float h0, h1;
    f2_get(rise, h0, h1);
    const F2 h = kGrid ? rise : f2(__fadd_rn(r.X, h0), __fadd_rn(r.X, h1));
    const F2 it = f2_mul(f2(T.inv_delta_f), f2(rcp_approx(fa), rcp_approx(fb)));
    f2_get(f2_mul(f2_sub(h, hb), it), ca, cb);
}

}  // namespace ss
