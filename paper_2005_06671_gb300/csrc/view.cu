// View rays of a camera against the bilinear terrain: the terrain points a
// camera sees, which are the origins of the shadow rays (Sec. 4: view rays are
// intersected with the displaced terrain, and the maximum mipmap lets a ray
// skip what it passes above).
//
// Per pixel:
//   d = unit(forward + a right + b up), x(tau) = C + tau d, samples tau_k = k step;
//   the hit is the first sample whose texel image is in the tile and lies on or
//   below the terrain (|x| - R - h <= 0, decided in FP64); when the sample
//   before it is in the tile too the crossing between the two is refined:
//   bisection until the bracket lies in one bilinear cell, then the single root of
//   the quadratic F there (see refine_crossing).
// Blocks of 2^k samples are walked near-to-far in float32, each about as long as
// the ray takes to lose the clearance the one before left (16 blocks and 3 groups
// of 4 samples per pixel of the polar view): a block is skipped when the ray's
// lowest height over it exceeds the maximum-mipmap value over its texel footprint
// by more than the float32 rounding, or when the footprint misses the tile, and
// halved otherwise.  A sample that float32 does not show clearly above or below
// the terrain or off the tile is decided in float-float arithmetic, and in FP64
// where that leaves a doubt: the first sample found below the terrain is the same
// one as an FP64 march finds.
//
// A second pass gathers the hits and refines them with full warps: F at the two samples
// in float-float, the root between them in float32 relative to those, one Newton step in
// float-float where the coordinates' rounding needs it, FP64 where they do not settle it.
// Then the hits are compacted in pixel order (per-block counts, one scan block,
// a scatter), so the ray list is deterministic.
//
// What bounds it: the FP64 pipe (77% / 86% busy, GB300 runs it at 1/64 of the float32
// rate) while setup, doubtful samples and refinement were FP64; now instruction
// issue in the march (75% of slots, 21 of 32 lanes: rays differ in length), and in the
// refinement the few hits that FP64 settles (issue 31%, FP64 pipe 61%, waits at barriers).  3840 x 2160 over
// 16384^2, 6.2 M hits: 18.55 -> 4.22 ms; 1920 x 1080 over 8192^2 4.83 -> 1.37 ms;
// 640 x 360 over 2048^2 of 20 m 1.26 -> 0.40 ms.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <cmath>

#include "ss_launch.h"

namespace ss {

namespace {

constexpr int kViewBlock = 256;
constexpr int kViewLeaf = 2;          // blocks of 4 samples are tested sample by sample

struct Cam {
    double C[3], f[3], r[3], u[3];
    double tan_x, tan_y;
    int32_t W, H;
    // per launch (host): 2/W, 2/H; |C|^2, |C|; the float32 ray state's camera terms
    double inv_w2, inv_h2, cc, cn;
    float cxf, cyf, czf, alt, zsum, inv_2cn, two_r_g;
    // float-float copies: C - P0 (P0 = (0, 0, R)), |C| - R, |C|, |C|^2, |C| + R, R, the image
    // scale, the pixel directions' terms
    DF rel[3], dalt, dcn, dcc, dzsum, dR, dk, df[3], dr[3], du[3], diw, dih;
    // their error bounds: positions (texels) pos0 + pos_t tau, heights (m) height0 + height_t tau
    float pos0, pos_t, height0, height_t;
};

struct ViewArgs {
    Tile T;
    Pyramid P;
    Cam cam;
    double step;
    DF dstep;
    float step_f, inv_step;
    float guard;              // float32 march: heights (view_guard)
    float pos_margin, pos_base, pos_t;   // texel positions (view_margin)
    int64_t K;
    int32_t pool;             // pixels of a march warp
    const float* stats;       // (global max, global min) of the heights
    float2* pix_uv;           // per pixel: hit texel coords, NaN when none
    int32_t* hit_k;           // per pixel: first sample below the terrain, -1 when none
    int32_t* block_count;     // per block of kViewBlock pixels
    int64_t* block_off;       // exclusive prefix of block_count
    int32_t n_blocks;
    int32_t groups;           // groups of kViewBlock pixels of a refine block
    float* uv_out;
    int32_t* pixel_out;
    int64_t* count_out;
};

// sample at distance tau: in-tile flag, and whether it is on or below the terrain
__device__ __forceinline__ bool below(const Tile& T, const double C[3], const double d[3],
                                      double tau, bool& inside, double& u, double& v) {
    const double x[3] = { C[0] + tau * d[0], C[1] + tau * d[1], C[2] + tau * d[2] };
    inside = texel_image64(T, x, u, v) && in_tile64(T, u, v);
    if (!inside) return false;
    int32_t i0, j0;
    double w[4];
    const double hb = fetch_bilinear64(T.h, T.pitch, T.nx, T.ny, u, v, &i0, &j0, w);
    const double H = sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]) - T.R;
    return H - hb <= 0.0;
}

// below() for the bisection of the crossing: one square root and one division
// (|x| serves both the height and the stereographic image; 1/g folded into the
// scale).  Its roundings differ from below()'s only at the 1e-16 relative
// level, and the bisection stops at a bracket of 2^-kViewHalvings of the step,
// below the FP64 resolution of |x| - R at the lunar radius (~1e-10 m), so the
// float32 hit coordinates are those of the full 48-halving bisection.
constexpr int kViewHalvings = 36;

__device__ __forceinline__ bool below_fast(const Tile& T, const double C[3], const double d[3],
                                           double tau) {
    const double x[3] = { C[0] + tau * d[0], C[1] + tau * d[1], C[2] + tau * d[2] };
    const double m = sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
    double k;
    if (T.proj == 0) {
        if (!(x[2] > 0.0)) return false;
        k = (T.R * T.inv_g) / x[2];
    } else {
        const double den = m + x[2];
        if (!(den > 0.0)) return false;
        k = (2.0 * T.R * T.inv_g) / den;
    }
    const double u = x[0] * k + T.cx, v = x[1] * k + T.cy;
    if (!in_tile64(T, u, v)) return false;
    int32_t i0, j0;
    double w[4];
    const double hb = fetch_bilinear64(T.h, T.pitch, T.nx, T.ny, u, v, &i0, &j0, w);
    return (m - T.R) - hb <= 0.0;
}

// below_fast's arithmetic, keeping the value F = (|x| - R) - h and the texel
// image: below_fast(tau) == (in && f <= 0), bit for bit.
struct ViewPt {
    double tau, f, u, v;
    bool in;
};

__device__ __forceinline__ ViewPt view_pt(const Tile& T, const double C[3], const double d[3],
                                          double tau) {
    ViewPt p;
    p.tau = tau;
    p.f = 0.0;
    p.u = p.v = 0.0;
    p.in = false;
    const double x[3] = { C[0] + tau * d[0], C[1] + tau * d[1], C[2] + tau * d[2] };
    const double m = sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]);
    double k;
    if (T.proj == 0) {
        if (!(x[2] > 0.0)) return p;
        k = (T.R * T.inv_g) / x[2];
    } else {
        const double den = m + x[2];
        if (!(den > 0.0)) return p;
        k = (2.0 * T.R * T.inv_g) / den;
    }
    p.u = x[0] * k + T.cx;
    p.v = x[1] * k + T.cy;
    if (!in_tile64(T, p.u, p.v)) return p;
    p.in = true;
    int32_t i0, j0;
    double w[4];
    const double hb = fetch_bilinear64(T.h, T.pitch, T.nx, T.ny, p.u, p.v, &i0, &j0, w);
    p.f = (m - T.R) - hb;
    return p;
}

// the bilinear cell fetch_bilinear64 reads for in-tile point p
__device__ __forceinline__ bool same_cell(const Tile& T, const ViewPt& a, const ViewPt& b) {
    const int32_t ia = min(max((int32_t)floor(a.u), 0), T.nx - 2);
    const int32_t ib = min(max((int32_t)floor(b.u), 0), T.nx - 2);
    const int32_t ja = min(max((int32_t)floor(a.v), 0), T.ny - 2);
    const int32_t jb = min(max((int32_t)floor(b.v), 0), T.ny - 2);
    return ia == ib && ja == jb;
}

// unit direction of pixel pix's view ray
__device__ __forceinline__ void pixel_dir(const Cam& cm, int64_t pix, double d[3]) {
    const int64_t i = pix % cm.W, j = pix / cm.W;
    const double aa = (((double)i + 0.5) * cm.inv_w2 - 1.0) * cm.tan_x;
    const double bb = (1.0 - ((double)j + 0.5) * cm.inv_h2) * cm.tan_y;
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] = cm.f[k] + aa * cm.r[k] + bb * cm.u[k];
    const double idn = 1.0 / sqrt(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) d[k] *= idn;
}

// ------------------------------------------------ float-float along a view ray
// Heights and texel positions to ~1e-13 of their size (2^-44 per operation),
// on the float32 pipes: GB300 runs FP64 at 1/64 of their rate.
struct ViewDir {
    DF d[3], cd2;   // unit direction, 2 C.d
};

// unit direction of pixel pix's view ray
__device__ __forceinline__ ViewDir view_dir(const Cam& cm, uint32_t pix) {
    const uint32_t j = pix / (uint32_t)cm.W, i = pix - j * (uint32_t)cm.W;
    const DF one = { 1.0f, 0.0f };
    // 2 (i + 1/2) / W - 1 (the tangents are in dr, du); the pixel index is below 2^31: exact as two floats
    const DF fi = df_two_sum((float)(i & ~0xffffu), (float)(i & 0xffffu) + 0.5f);
    const DF fj = df_two_sum((float)(j & ~0xffffu), (float)(j & 0xffffu) + 0.5f);
    const DF a = df_add(df_mul(cm.diw, fi), df_neg(one));
    const DF b = df_add(one, df_neg(df_mul(cm.dih, fj)));
    ViewDir v;
#pragma unroll
    for (int k = 0; k < 3; ++k)
        v.d[k] = df_add(cm.df[k], df_add(df_mul(a, cm.dr[k]), df_mul(b, cm.du[k])));
    const DF n2 = df_add(df_add(df_mul(v.d[0], v.d[0]), df_mul(v.d[1], v.d[1])),
                         df_mul(v.d[2], v.d[2]));
    const DF in = df_div(one, df_sqrt(n2));
#pragma unroll
    for (int k = 0; k < 3; ++k) v.d[k] = df_mul(v.d[k], in);
    const DF cd = df_add(df_add(df_mul(cm.rel[0], v.d[0]), df_mul(cm.rel[1], v.d[1])),
                         df_add(df_mul(cm.rel[2], v.d[2]), df_mul(cm.dR, v.d[2])));
    v.cd2 = DF{ 2.0f * cd.hi, 2.0f * cd.lo };
    return v;
}

// The point at tau: F = |x| - R - h, its texel image, its bilinear cell, and
// bounds of the rounding errors of F (err) and of the image (pos).  state: 1 in the tile,
// 0 off it, -1 in doubt (within the rounding of an edge, or no image).
// The bounds: about 2^-42 of the terms, the distances from the tile centre's point and
// along the ray among them.  Replayed against 64-bit mantissas (tiles up to 0.8 radii wide,
// cameras 0.1 to 300,000 km up): at most 0.32 of pos and 0.21 of err used.
struct ViewPtDF {
    DF f, u, v, rise;
    int32_t i0, j0;
    float err, pos;
    int state;
};

__device__ __forceinline__ void view_image_df(const Tile& T, const Cam& cm, const ViewDir& r, DF tau,
                                              DF& rise, DF& u, DF& v, float& den) {
    // rise = |C + tau d| - |C| = w / (|C| + sqrt(|C|^2 + w)), w = tau (2 C.d + tau)
    const DF w = df_mul(tau, df_add(r.cd2, tau));
    rise = df_div(w, df_add(cm.dcn, df_sqrt(df_add(cm.dcc, w))));
    const DF x = df_add(cm.rel[0], df_mul(tau, r.d[0])), y = df_add(cm.rel[1], df_mul(tau, r.d[1]));
    const DF z = df_add(cm.rel[2], df_mul(tau, r.d[2]));   // x_z - R
    const DF dd = T.proj == 0 ? df_add(cm.dR, z) : df_add(cm.dzsum, df_add(rise, z));
    den = dd.hi;
    const DF k = df_div(cm.dk, dd);
    u = df_add(df_mul(x, k), DF{ T.cx_f, 0.0f });
    v = df_add(df_mul(y, k), DF{ T.cy_f, 0.0f });
}

__device__ __forceinline__ ViewPtDF view_pt_df(const Tile& T, const Cam& cm, const ViewDir& r, DF tau) {
    ViewPtDF p;
    float den;
    view_image_df(T, cm, r, tau, p.rise, p.u, p.v, den);
    const DF rise = p.rise;
    const float um = (float)(T.nx - 1), vm = (float)(T.ny - 1);
    p.pos = cm.pos0 + cm.pos_t * tau.hi + 2e-14f * (fabsf(p.u.hi) + fabsf(p.v.hi));
    const float e = 1e-6f + 1e-11f * (fabsf(p.u.hi) + fabsf(p.v.hi)) + 1e-10f * (um + vm) + p.pos;
    const float inside = fminf(fminf(p.u.hi, um - p.u.hi), fminf(p.v.hi, vm - p.v.hi));
    p.f = DF{ 0.0f, 0.0f };
    p.err = 0.0f;
    p.i0 = p.j0 = 0;
    // (float32 of a value within e of an edge is within 2 e of it, or its ulp)
    const float edge = 2.0f * e + 2.5e-7f * fmaxf(fabsf(p.u.hi), fabsf(p.v.hi));
    p.state = !(den > 1.0f) || !(fabsf(inside) > edge) ? -1 : inside > 0.0f ? 1 : 0;
    if (p.state != 1) return p;
    p.i0 = min(df_floor(p.u), T.nx - 2);
    p.j0 = min(df_floor(p.v), T.ny - 2);
    const DF fu = df_add(p.u, DF{ -(float)p.i0, 0.0f }), fv = df_add(p.v, DF{ -(float)p.j0, 0.0f });
    const float* q = T.h + (int64_t)p.j0 * T.pitch + p.i0;
    const float h00 = __ldg(q), h10 = __ldg(q + 1), h01 = __ldg(q + T.pitch), h11 = __ldg(q + T.pitch + 1);
    const DF top = df_add(df_mul(fu, df_two_sum(h10, -h00)), DF{ h00, 0.0f });
    const DF bot = df_add(df_mul(fu, df_two_sum(h11, -h01)), DF{ h01, 0.0f });
    const DF hb = df_add(df_mul(fv, df_add(bot, df_neg(top))), top);
    p.f = df_add(df_add(cm.dalt, rise), df_neg(hb));
    const float rng = fmaxf(fmaxf(h00, h10), fmaxf(h01, h11)) - fminf(fminf(h00, h10), fminf(h01, h11));
    p.err = cm.height0 + cm.height_t * tau.hi + 2e-13f * (fabsf(rise.hi) + fabsf(hb.hi)) +
            2.0f * p.pos * rng;
    return p;
}

// k step as float-float (k < 2^31)
__device__ __forceinline__ DF view_tau(const ViewArgs& a, int32_t k) {
    const DF kk = df_two_sum((float)(k & ~0xffff), (float)(k & 0xffff));
    return df_mul(kk, a.dstep);
}

// Whether sample k of pixel pix lies on or below the terrain in the tile: in
// float-float, in FP64 (below()) where that is within 1000 x its error bound.
__device__ __noinline__ bool view_decide(const ViewArgs& a, uint32_t pix, int32_t k) {
    const ViewDir r = view_dir(a.cam, pix);
    const ViewPtDF p = view_pt_df(a.T, a.cam, r, view_tau(a, k));
    if (p.state == 0) return false;
    if (p.state == 1 && fabsf(p.f.hi) > 1000.0f * p.err + 1e-9f) return p.f.hi < 0.0f;
    double d[3], u, v;
    bool ins;
    pixel_dir(a.cam, pix, d);
    return below(a.T, a.cam.C, d, (double)k * a.step, ins, u, v);
}

// ------------------------------------------------------------ float32 march
// float32 state of one view ray.  The camera is taken relative to the tile
// centre's point on the sphere, P0 = (0, 0, R) (a few km, so float32 keeps it
// to a few mm); the ray height over the sphere is the camera altitude plus
// rise(tau) = |C + tau d| - |C| in the cancellation-free form of the shadow
// rays, so heights carry ~1e-2 m of rounding and texel positions
// ~2e-3 texel (5 m texels) over the ray's 150 km.
struct ViewRayF {
    float dx, dy, dz;        // unit direction
    float B;                 // 2 C.d
    float inv8r;             // stereographic: 1/(8 r) of the image circle (texels^-1)
    float tv, rise_tv;       // closest approach to the centre, and the rise there
};

__device__ __forceinline__ float sqrt_approx(float x) {   // 2^-22 relative, one instruction
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float view_rise(const Cam& cm, const ViewRayF& q, float t) {
    const float w = t * (q.B + t);
    const float x = 4.0f * w * cm.inv_2cn * cm.inv_2cn;
    return __fdividef(2.0f * w * cm.inv_2cn, 1.0f + sqrt_approx(fmaxf(0.0f, 1.0f + x)));
}

// texel coordinates of the ray point at tau (rise = rise(tau)); false when the
// point has no image (gnomonic: not in front of the plane; stereographic: near
// the antipode)
__device__ __forceinline__ bool view_image_f(const Tile& T, const Cam& cm, const ViewRayF& q,
                                             float tau, float rise, float& u, float& v) {
    const float z = cm.czf + tau * q.dz;
    const float den = T.proj == 0 ? T.R_f + z : cm.zsum + (rise + z);
    const float k = __fdividef(cm.two_r_g, den);
    u = (cm.cxf + tau * q.dx) * k + T.cx_f;
    v = (cm.cyf + tau * q.dy) * k + T.cy_f;
    return den > 1.0f;
}

struct ViewLevels {
    const float* ptr[kMaxLevels];
    uint32_t pitch[kMaxLevels];
};

// maximum of the heights over texel box [x0, x1] x [y0, y1] (inclusive, clamped
// to the tile), read as <= 2x2 cells of the coarsest level whose cells cover it
__device__ __forceinline__ float box_max(const ViewLevels& L, int32_t levels, int32_t x0, int32_t x1,
                                         int32_t y0, int32_t y1) {
    const int32_t ext = max(x1 - x0, y1 - y0);
    int32_t m = ext <= 1 ? 0 : 31 - __clz(ext);
    m += (((x1 >> m) - (x0 >> m)) > 1 || ((y1 >> m) - (y0 >> m)) > 1) ? 1 : 0;
    m = min(m, levels - 1);
    const uint32_t pm = L.pitch[m];
    const float* p = cell_ptr(L.ptr[m], pm, x0 >> m, y0 >> m);
    const uint32_t dx = (uint32_t)((x1 >> m) - (x0 >> m));
    const uint32_t dy = (uint32_t)((y1 >> m) - (y0 >> m)) * pm;
    return fmaxf(fmaxf(__ldg(p), __ldg(p + dx)), fmaxf(__ldg(p + dy), __ldg(p + dy + dx)));
}

struct ViewEnd {
    float t, rise, u, v;
    bool ok;
};

// Bound of the error of a float32 texel position at distance t (see launch_view_rays).
__device__ __forceinline__ float view_margin(const ViewArgs& a, float t) {
    return fmaxf(a.pos_margin, fmaf(a.pos_t, t, a.pos_base));
}

// And of a float32 height (m).
__device__ __forceinline__ float view_guard(const ViewArgs& a, float t) {
    return fmaf(2e-7f, t, a.guard);
}

__device__ __forceinline__ ViewEnd view_end(const ViewArgs& a, const ViewRayF& q, float j) {
    ViewEnd e;
    e.t = j * a.step_f;
    e.rise = view_rise(a.cam, q, e.t);
    e.ok = view_image_f(a.T, a.cam, q, e.t, e.rise, e.u, e.v);
    return e;
}

// How far the ray clears the terrain between two of its points: its lowest height
// there minus the maximum height under its footprint, less the guard.  Positive: no
// sample between them is below the terrain; +inf where the footprint misses the tile.
__device__ __forceinline__ float view_clear(const ViewArgs& a, const ViewLevels& L, const ViewRayF& q,
                                            const ViewEnd& x, const ViewEnd& y) {
    const Tile& T = a.T;
    const float du = y.u - x.u, dv = y.v - x.v;
    const float e = view_margin(a, y.t) + arc_bulge(du * du + dv * dv, q.inv8r);
    const float lo_u = fminf(x.u, y.u) - e, hi_u = fmaxf(x.u, y.u) + e;
    const float lo_v = fminf(x.v, y.v) - e, hi_v = fmaxf(x.v, y.v) + e;
    const float nxm = (float)(T.nx - 1), nym = (float)(T.ny - 1);
    // (no image at an end, or a NaN: not ruled out)
    if (!(x.ok && y.ok && hi_u - lo_u < 1e7f && hi_v - lo_v < 1e7f)) return -INFINITY;
    if (hi_u < 0.0f || lo_u > nxm || hi_v < 0.0f || lo_v > nym) return INFINITY;
    const int32_t x0 = max(__float2int_rd(lo_u), 0);
    const int32_t x1 = min(__float2int_rd(hi_u) + 1, T.nx - 1);
    const int32_t y0 = max(__float2int_rd(lo_v), 0);
    const int32_t y1 = min(__float2int_rd(hi_v) + 1, T.ny - 1);
    const float M = box_max(L, a.P.levels, x0, x1, y0, y1);
    const bool dip = q.tv > x.t && q.tv < y.t;
    const float Hmin = a.cam.alt + (dip ? q.rise_tv : fminf(x.rise, y.rise));
    return Hmin - M - view_guard(a, y.t);
}

// Samples j0 .. j0 + 3 (up to `last`) of pixel pix: the first on or below the
// terrain, 0 when none is.  clear: the last sample's height over the terrain.
__device__ __forceinline__ uint32_t view_leaf(const ViewArgs& a, const ViewRayF& q, uint32_t pix,
                                              uint32_t j0, uint32_t last, float& clear) {
    const Tile& T = a.T;
    const float nxm = (float)(T.nx - 1), nym = (float)(T.ny - 1);
    unsigned hit = 0, doubt = 0;
#pragma unroll
    for (int i = 0; i < 1 << kViewLeaf; ++i) {
        const ViewEnd e = view_end(a, q, (float)(j0 + i));
        const float pm = view_margin(a, e.t);
        const bool out = e.ok && (e.u < -pm || e.u > nxm + pm || e.v < -pm || e.v > nym + pm);
        const bool in = e.ok && e.u >= pm && e.u <= nxm - pm && e.v >= pm && e.v <= nym - pm;
        const int32_t i0 = min(max(__float2int_rd(e.u), 0), T.nx - 2);
        const int32_t k0 = min(max(__float2int_rd(e.v), 0), T.ny - 2);
        const float fu = e.u - (float)i0, fv = e.v - (float)k0;
        const float* p = cell_ptr(T.h, (uint32_t)T.pitch, i0, k0);
        const float h00 = __ldg(p), h10 = __ldg(p + 1);
        const float h01 = __ldg(p + (uint32_t)T.pitch), h11 = __ldg(p + (uint32_t)T.pitch + 1);
        const float top = h00 + fu * (h10 - h00);
        const float bot = h01 + fu * (h11 - h01);
        const float hb = top + fv * (bot - top);
        const float rng = fmaxf(fmaxf(h00, h10), fmaxf(h01, h11)) - fminf(fminf(h00, h10), fminf(h01, h11));
        const float gap = (a.cam.alt + e.rise) - hb, gd = view_guard(a, e.t) + pm * rng;
        // a sample below by more than the guard is a hit, above by more is none;
        // the others, and those near the tile's border, are decided exactly
        const bool mine = j0 + i <= last;
        clear = e.ok && !out ? gap : INFINITY;
        hit |= mine && in && gap < -gd ? 1u << i : 0u;
        doubt |= mine && !out && !(in && (gap > gd || gap < -gd)) ? 1u << i : 0u;
    }
    unsigned c = hit | doubt;
    while (c) {
        const int i = __ffs(c) - 1;
        if (((hit >> i) & 1u) || view_decide(a, pix, (int32_t)(j0 + i))) return j0 + i;
        c &= c - 1u;
    }
    return 0;
}

constexpr float kViewBeta = 0.7f;   // share of the clearance the next block may lose
constexpr int kViewFirst = 11;   // level of a ray's first block
__device__ __forceinline__ float exp2_int(int k) { return __int_as_float((127 + k) << 23); }   // |k| < 127
// floor(log2 x) of a positive normal x (+inf: 128)
__device__ __forceinline__ int ilog2_f(float x) { return (__float_as_int(x) >> 23) - 127; }

// Setup of pixel pix's ray: its float32 state and the samples b0 + 1 .. b0 + n that
// can hold the hit (n = 0: none), parked in the warp's queue at `slot`.
__device__ __noinline__ void view_park(const ViewArgs& a, uint32_t pix, uint32_t (*w)[32], int slot) {
    const Cam& cm = a.cam;
    const ViewDir r = view_dir(cm, pix);
    ViewRayF q;
    q.dx = r.d[0].hi;
    q.dy = r.d[1].hi;
    q.dz = r.d[2].hi;
    q.B = r.cd2.hi;
    // samples that can reach the highest height: tau^2 + 2 cd tau + E <= 0 with
    // E = |C|^2 - (R + hmax)^2; the margins cover the roundings (tau to 1e-6)
    const DF hm = { a.stats[0], 0.0f };
    const DF E = df_mul(df_add(cm.dalt, df_neg(hm)), df_add(cm.dzsum, hm));
    const DF cd = { 0.5f * r.cd2.hi, 0.5f * r.cd2.lo };
    const DF disc = df_add(df_mul(cd, cd), df_neg(E));
    const float slack = 1e-11f * (cd.hi * cd.hi + fabsf(E.hi));
    uint32_t b0 = 0, n = 0;
    if (disc.hi >= -slack) {
        const float sq = sqrtf(fmaxf(disc.hi, 0.0f) + slack);
        float tin, tout;   // -cd -/+ sq without cancellation
        if (cd.hi <= 0.0f) {
            tout = sq - cd.hi;
            tin = tout > 0.0f ? E.hi / tout : 0.0f;
        } else {
            tin = -cd.hi - sq;
            tout = E.hi / tin;
        }
        if (tout >= 0.0f) {
            const float f0 = floorf(tin * a.inv_step * 0.99999f) - 2.0f;
            const float f1 = ceilf(tout * a.inv_step * 1.00001f) + 2.0f;
            const int64_t k0 = f0 > 1.0f ? (int64_t)fminf(f0, 2.2e9f) : 1;
            const int64_t k1 = f1 < 2.2e9f ? min((int64_t)f1, a.K) : a.K;
            if (k0 <= k1) {
                b0 = (uint32_t)(k0 - 1);
                n = (uint32_t)(k1 - k0 + 1);
            }
        }
    }
    // image circle of the ray (stereographic): 1/(8 r) in texels^-1
    float inv8r = 0.0f;
    if (a.T.proj != 0) {
        const float Cz = a.T.R_f + cm.czf;
        const float Nx = cm.cyf * q.dz - Cz * q.dy, Ny = Cz * q.dx - cm.cxf * q.dz;
        const float Nz = cm.cxf * q.dy - cm.cyf * q.dx;
        const float nn = sqrtf(Nx * Nx + Ny * Ny + Nz * Nz);
        // (rounding of N_z: 1e-6 of its terms)
        const float nz = fabsf(Nz) + 1e-6f * (fabsf(cm.cxf) + fabsf(cm.cyf));
        inv8r = nn > 0.0f ? 1.0001f * nz / nn * a.T.g_f / (16.0f * a.T.R_f) : 0.0f;
    }
    w[0][slot] = __float_as_uint(q.dx);
    w[1][slot] = __float_as_uint(q.dy);
    w[2][slot] = __float_as_uint(q.dz);
    w[3][slot] = __float_as_uint(q.B);
    w[4][slot] = __float_as_uint(inv8r);
    w[5][slot] = b0;
    w[6][slot] = n;
}

// Lanes at a leaf block wait for kViewLeaves of them (or for the walks to end), lanes
// without a ray for kViewIdle.  (3840 x 2160 view: 4.35 ms; leaves at 6: 4.87, at 16: 4.29
// but 3% more on the smaller view; idle at 8, 12, 16: 1%, 7%, 9% more; beta 0.35, 0.5, 1:
// 17%, 5%, 1% more; first block 2^9, 2^13: 1% more; groups of 8 samples: 25% more.)
constexpr int kViewLeaves = 12, kViewIdle = 4;
constexpr int kViewHitBlock = 128;

// Pass 1: per pixel, the first sample below the terrain (hit_k, -1 when none).
// A warp owns a.pool consecutive pixels.  It sets up 32 of their rays at a time,
// with all lanes, and parks them in shared memory; each lane walks one ray and
// takes the next parked one when it is done.
__global__ void __launch_bounds__(kViewHitBlock, 8) view_hit_kernel(const __grid_constant__ ViewArgs a) {
    __shared__ ViewLevels s_lev;
    __shared__ uint32_t s_q[kViewHitBlock / 32][7][32];
    if (threadIdx.x < kMaxLevels) {
        s_lev.ptr[threadIdx.x] = a.P.ptr[threadIdx.x];
        s_lev.pitch[threadIdx.x] = (uint32_t)a.P.pitch[threadIdx.x];
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    uint32_t (*w)[32] = s_q[threadIdx.x >> 5];
    const uint64_t npix = (uint64_t)a.cam.W * (uint64_t)a.cam.H;
    uint64_t next = ((uint64_t)blockIdx.x * (kViewHitBlock / 32) + (threadIdx.x >> 5)) * (uint32_t)a.pool;
    const uint64_t end = min(next + (uint64_t)a.pool, npix);
    uint32_t qpix = 0;           // pixel of the queue's first slot
    int qpos = 0, qend = 0;      // parked rays not taken yet
    uint32_t pix = 0;            // the lane's ray
    bool busy = false;
    ViewRayF q;
    uint32_t b0 = 0, n = 0, s = 0, hit = 0;   // the current block: samples s + 1 .. s + 2^k after b0
    int k = 0, kk = 0;
    float drop = 1.0f;           // height lost per sample
    while (true) {
        if (busy && s >= n) {    // done: first sample found, or none
            a.hit_k[pix] = hit ? (int32_t)hit : -1;
            busy = false;
        }
        const unsigned mi = __ballot_sync(0xffffffffu, !busy);
        const bool more = qpos < qend || next < end;
        if (more && (mi == 0xffffffffu || __popc(mi) >= kViewIdle)) {
            if (qpos == qend) {
                __syncwarp();
                qend = (int)min((uint64_t)32, end - next);
                if (lane < qend) view_park(a, (uint32_t)next + lane, w, lane);
                qpix = (uint32_t)next;
                next += qend;
                qpos = 0;
                __syncwarp();
            }
            const int slot = qpos + __popc(mi & ((1u << lane) - 1u));
            if (!busy && slot < qend) {
                busy = true;
                pix = qpix + slot;
                q.dx = __uint_as_float(w[0][slot]);
                q.dy = __uint_as_float(w[1][slot]);
                q.dz = __uint_as_float(w[2][slot]);
                q.B = __uint_as_float(w[3][slot]);
                q.inv8r = __uint_as_float(w[4][slot]);
                b0 = w[5][slot];
                n = w[6][slot];
                q.tv = -0.5f * q.B;
                q.rise_tv = view_rise(a.cam, q, q.tv);
                kk = max(kViewLeaf, n <= 1u ? 0 : 32 - __clz(n - 1u));   // 2^kk >= n
                k = min(kk, kViewFirst);
                s = hit = 0;
            }
            qpos = min(qend, qpos + __popc(mi));
            continue;
        }
        if (mi == 0xffffffffu) break;
        const bool leaf = busy && k == kViewLeaf;
        const unsigned ml = __ballot_sync(0xffffffffu, leaf);
        float clear = -INFINITY;   // of the block; positive: go on behind it
        bool moved = false;
        if (ml == ~mi || __popc(ml) >= kViewLeaves) {
            if (leaf) {
                hit = view_leaf(a, q, pix, b0 + s + 1u, b0 + n, clear);
                clear = fmaxf(clear, 1e-6f);
                moved = true;
            }
        } else if (busy && !leaf) {
            const ViewEnd x = view_end(a, q, (float)(b0 + s + 1u));
            const ViewEnd y = view_end(a, q, (float)(b0 + s + min(1u << k, n - s)));
            clear = view_clear(a, s_lev, q, x, y);
            drop = (x.rise - y.rise) * exp2_int(-k);
            moved = true;
        }
        if (moved) {
            if (clear > 0.0f) {
                s = hit ? n : s + min(1u << k, n - s);
                // the next block: about as long as the ray takes to lose that clearance
                const float len = __fdividef(kViewBeta * clear, fmaxf(drop, 1e-6f));
                const int kn = min(ilog2_f(len), k + 2);
                k = max(min(kn, kk), kViewLeaf);
            } else {
                --k;
            }
        }
    }
}

// The crossing of F in [lo, hi] (F(lo) > 0 in the tile, F(hi) <= 0): the upper
// end of a bracket of the crossing.  The halvings of the bisection run until
// both ends lie in one bilinear cell: up to there the choices are the
// bisection's own (below_fast's arithmetic).  Inside one cell the terrain
// along the ray is a quadratic in tau (bilinear along a line; the image arc
// bends by ~1e-8 texel over a cell) and so is the ray's height (to ~1e-12 m),
// so F has exactly one root in a bracket where it changes sign: F at the
// midpoint and the quadratic through the three values place it, and one more
// value confirms a bracket [r - eps, r] or [r, r + eps] around the estimate r,
// eps = 8 x the FP64 rounding of F (2e-9 m) over the slope |F'| (at least
// 2^-36 of the step, the bisection's own bracket).  The upper end then lies
// within eps of the crossing, below 1/3 of a float32 step of texel
// coordinates >= 0.25.  Near-tangent crossings (eps above 2^-22 of the step),
// points near the tile's low edges and failed confirmations finish with
// halvings to 2^-kViewHalvings of the step, as before.
__device__ __noinline__ double refine_crossing(const Tile& T, const double C[3], const double d[3],
                                               ViewPt lo, double hi_t, double step) {
    double lo_t = lo.tau;
    ViewPt hi = view_pt(T, C, d, hi_t);
    const double tol = ldexp(step, -kViewHalvings);
    if (!(lo.in && lo.f > 0.0 && hi.in && hi.f <= 0.0)) {
        // (below()'s and below_fast's roundings disagree at an end): plain halvings
        for (int it = 0; it < kViewHalvings; ++it) {
            const double mid = lo_t + 0.5 * (hi_t - lo_t);
            if (below_fast(T, C, d, mid))
                hi_t = mid;
            else
                lo_t = mid;
        }
        return hi_t;
    }
    int it = 0;
    for (; it < kViewHalvings && !same_cell(T, lo, hi); ++it) {
        const ViewPt m = view_pt(T, C, d, lo.tau + 0.5 * (hi.tau - lo.tau));
        if (m.in && m.f <= 0.0)
            hi = m;
        else
            lo = m;
        if (!lo.in) break;   // (the ray left the tile between samples)
    }
    if (it < kViewHalvings && lo.in && same_cell(T, lo, hi)) {
        const double t0 = lo.tau, h = hi.tau - lo.tau;
        const ViewPt m = view_pt(T, C, d, t0 + 0.5 * h);
        // quadratic F(t0 + s h) = A + B s + Cq s^2 through s = 0, 1/2, 1
        const double A = lo.f, Cq = 2.0 * (lo.f + hi.f - 2.0 * m.f), B = hi.f - lo.f - Cq;
        if (m.in && same_cell(T, lo, m)) {
            if (m.f <= 0.0)
                hi = m;
            else
                lo = m;
        }
        const double l0 = (lo.tau - t0) / h, l1 = (hi.tau - t0) / h;   // bracket in s
        double s = -1.0;
        if (fabs(Cq) <= 1e-12 * fabs(B)) {
            if (B != 0.0) s = -A / B;
        } else {
            const double disc = B * B - 4.0 * A * Cq;
            if (disc >= 0.0) {
                const double q = -0.5 * (B + copysign(sqrt(disc), B));
                const double s1 = q / Cq, s2 = q != 0.0 ? A / q : -1.0;
                s = (s1 >= l0 && s1 <= l1) ? s1 : s2;
            }
        }
        const double r = t0 + s * h;
        const double slope = fabs((B + 2.0 * Cq * s) / h);
        const double eps = fmax(tol, 1.6e-8 / slope);
        const bool low_edge = fmin(lo.u, lo.v) < 0.25 || fmin(hi.u, hi.v) < 0.25;
        if (s >= l0 && s <= l1 && r > lo.tau && r <= hi.tau && slope > 0.0 &&
            eps <= ldexp(step, -22) && !low_edge) {
            const ViewPt pr = view_pt(T, C, d, r);
            if (pr.in && same_cell(T, lo, pr)) {
                if (pr.f <= 0.0) {           // crossing in (lo, r]
                    hi = pr;
                    if (r - eps <= lo.tau) return hi.tau;
                    const ViewPt pc = view_pt(T, C, d, r - eps);
                    if (pc.in && pc.f > 0.0) return hi.tau;
                    if (pc.in) hi = pc;
                } else {                     // crossing in (r, hi]
                    lo = pr;
                    if (r + eps >= hi.tau) return hi.tau;
                    const ViewPt pc = view_pt(T, C, d, r + eps);
                    if (pc.in && pc.f <= 0.0) return pc.tau;
                    if (pc.in) lo = pc;
                }
            }
        }
    }
    // halvings of whatever bracket is left, down to the bisection's resolution
    double a_t = lo.tau, b_t = hi.tau;
    for (int k = 0; k < 2 * kViewHalvings && b_t - a_t > tol; ++k) {
        const double mid = a_t + 0.5 * (b_t - a_t);
        if (below_fast(T, C, d, mid))
            b_t = mid;
        else
            a_t = mid;
    }
    return b_t;
}

// Texel coordinates of the hit of pixel pix in FP64: the crossing between the
// sample before the hit, when that is in the tile, and the hit.
__device__ __noinline__ float2 view_point64(const ViewArgs& a, uint32_t pix, int32_t hit_k) {
    const Tile& T = a.T;
    double d[3];
    pixel_dir(a.cam, pix, d);
    const double* C = a.cam.C;
    double hi = (double)hit_k * a.step;
    if (hit_k > 1) {
        const ViewPt lo = view_pt(T, C, d, (double)(hit_k - 1) * a.step);
        if (lo.in) hi = refine_crossing(T, C, d, lo, hi, a.step);
    }
    const double xh[3] = { C[0] + hi * d[0], C[1] + hi * d[1], C[2] + hi * d[2] };
    double hu, hv;
    // the point lies between two samples of the tile: it has an image
    texel_image64(T, xh, hu, hv);
    return make_float2((float)hu, (float)hv);
}

// The same from two float-float points, the samples before and at the hit.  A step
// is a fraction of a cell long, so between them, to 1e-7 of the step, the texel
// image is a line, the rise a parabola and the terrain bilinear cell by cell:
// F relative to its value at the first point is a quadratic in each cell the step
// crosses, in float32; the step is halved until both ends lie in one cell (the
// choices of refine_crossing), whose root is the hit.  The coordinates are the float32
// nearest to the crossing's: where the error of that root could move their rounding
// (kViewDoubt: a fifth of the rays at 20 m texels, 1% at 5 m), view_newton takes one step from it.  kViewUnsettled: a
// point within rounding of the tile's border or of the terrain, a step of more than one cell
// line per axis, a tangent ray, coordinates below 4.
// (With roots whose error stayed below a quarter of the rounding instead, 1.8e-3 of the
// coordinates of 1280 x 720 over 2048^2 of 20 m were one float32 step off; FP64 had 1.7e-5,
// these have 1.7e-6.)
enum { kViewUnsettled, kViewDoubt, kViewDone };
struct ViewRoot {
    float s, du, dv, slope, a2, err, off;   // root, image of the step, F there, error bounds
};

__device__ __forceinline__ int view_point_df(const ViewArgs& a, uint32_t pix, int32_t hit_k,
                                             float2& out, ViewRoot& root) {
    const Tile& T = a.T;
    const Cam& cm = a.cam;
    const ViewDir r = view_dir(cm, pix);
    const ViewPtDF hi = view_pt_df(T, cm, r, view_tau(a, hit_k));
    if (hi.state != 1) return kViewUnsettled;
    out = make_float2(hi.u.hi, hi.v.hi);
    if (!(fminf(hi.u.hi, hi.v.hi) >= 4.0f)) return kViewUnsettled;
    const int sure = df_hi_is_nearest(hi.u, hi.pos) && df_hi_is_nearest(hi.v, hi.pos) ? kViewDone
                                                                                      : kViewUnsettled;
    if (hit_k <= 1) return sure;
    const ViewPtDF lo = view_pt_df(T, cm, r, view_tau(a, hit_k - 1));
    if (lo.state == 0) return sure;     // the sample before the hit is off the tile
    if (lo.state < 0 || !(lo.f.hi > 4.0f * lo.err) || !(hi.f.hi < -4.0f * hi.err)) return kViewUnsettled;
    if (abs(hi.i0 - lo.i0) > 1 || abs(hi.j0 - lo.j0) > 1) return kViewUnsettled;
    const float du = df_add(hi.u, df_neg(lo.u)).hi, dv = df_add(hi.v, df_neg(lo.v)).hi;
    const float dr = df_add(hi.rise, df_neg(lo.rise)).hi, h = a.step_f;
    // rise(s) = s dr - K s (1 - s), K = h^2 (1 - (dr/h)^2) / 2 |x|
    const float ir = __fdividef(1.0f, cm.dcn.hi + lo.rise.hi);   // 1/|x|
    const float K = 0.5f * ir * fmaxf(0.0f, (h - dr) * (h + dr));
    const float u0 = df_add(lo.u, DF{ -(float)lo.i0, 0.0f }).hi;   // position in the first cell
    const float v0 = df_add(lo.v, DF{ -(float)lo.j0, 0.0f }).hi;
    // F(s) = a0 + a1 s + a2 s^2 in cell (i, j) (relative to the first point's)
    float base = 0.0f, href = 0.0f, relief = 0.0f, a0, a1, a2;
    auto cell = [&](int32_t i, int32_t j, bool first) {
        const float* p = cell_ptr(T.h, (uint32_t)T.pitch, lo.i0 + i, lo.j0 + j);
        const float h00 = __ldg(p), h10 = __ldg(p + 1);
        const float h01 = __ldg(p + (uint32_t)T.pitch), h11 = __ldg(p + (uint32_t)T.pitch + 1);
        const float p0 = u0 - (float)i, q0 = v0 - (float)j;   // position in the cell at s = 0
        const float d10 = h10 - h00, d01 = h01 - h00, dx = (h11 - h01) - d10;
        const float hb = d10 * p0 + d01 * q0 + dx * p0 * q0;
        if (first) {
            href = h00;
            base = hb;                                        // h(0) - href
        }
        relief = fmaxf(relief, fabsf(d10) + fabsf(d01) + fabsf(dx) + fabsf(h00 - href));
        a0 = lo.f.hi + (base - ((h00 - href) + hb));
        a1 = dr - K - d10 * du - d01 * dv - dx * (p0 * dv + q0 * du);
        a2 = K - dx * du * dv;
    };
    cell(0, 0, true);
    // halved until both ends lie in one cell
    float beg = 0.0f, fin = 1.0f;
    int32_t bi = 0, bj = 0, fi = hi.i0 - lo.i0, fj = hi.j0 - lo.j0;
    for (int it = 0; bi != fi || bj != fj; ++it) {
        const float m = 0.5f * (beg + fin);
        // (clamped to the cells of the two ends: the line crosses no other)
        const int32_t mi = min(max((int32_t)floorf(u0 + m * du), min(bi, fi)), max(bi, fi));
        const int32_t mj = min(max((int32_t)floorf(v0 + m * dv), min(bj, fj)), max(bj, fj));
        cell(mi, mj, false);
        const float f = a0 + m * (a1 + m * a2);
        if (it == 20 || !(fabsf(f) > 1e-6f * (fabsf(lo.f.hi) + relief))) return kViewUnsettled;
        if (f > 0.0f) {
            beg = m;
            bi = mi;
            bj = mj;
        } else {
            fin = m;
            fi = mi;
            fj = mj;
        }
    }
    cell(bi, bj, false);
    const float q = -0.5f * (a1 + copysignf(sqrtf(fmaxf(a1 * a1 - 4.0f * a0 * a2, 0.0f)), a1));
    const float r1 = q / a2, r2 = a0 / q;
    float s = r2 >= beg && r2 <= fin ? r2 : r1;
    const float slope = a1 + 2.0f * a2 * s;
    if (!(s >= beg && s <= fin)) s = -1.0f;
    // float32 of F's terms; what the parabola and the line leave out over a step h: the
    // next orders of the rise and of the image, h/|x| of the last one kept
    const float len = fmaxf(fabsf(du), fabsf(dv)), hr = h * ir;
    const float far = fmaxf(fabsf(lo.u.hi - T.cx_f), fabsf(lo.v.hi - T.cy_f));
    const float off = 0.3f * len * hr + 0.5f * far * hr * hr;   // texels
    const float err = 4e-7f * (fabsf(lo.f.hi) + fabsf(dr) + relief) + lo.err + hi.err + K * hr + off * relief;
    if (!(s >= 0.0f)) return kViewUnsettled;
    // errors of the coordinates: the root's, along the step, the line's, the first point's and
    // the float32 roundings of s du and s dv
    const DF u = df_add(lo.u, DF{ s * du, 0.0f }), v = df_add(lo.v, DF{ s * dv, 0.0f });
    const float e = (__fdividef(err, fabsf(slope)) + 3e-7f) * len + off + lo.pos;
    out = make_float2(u.hi, v.hi);
    if (!(fminf(out.x, out.y) >= 4.0f)) return kViewUnsettled;
    if (df_hi_is_nearest(u, e) && df_hi_is_nearest(v, e)) return kViewDone;
    root = ViewRoot{ s, du, dv, slope, a2, err, off };
    return kViewDoubt;
}

// One Newton step from a root of view_point_df, from F there in float-float.  Where the
// rounding of the coordinates is in doubt still, one more from F in FP64 (good to its
// rounding, 2e-9 m, over the slope: what refine_crossing takes seven values of F for).
__device__ __noinline__ float2 view_newton(const ViewArgs& a, uint32_t pix, int32_t hit_k,
                                           const ViewRoot& q) {
    const ViewDir r = view_dir(a.cam, pix);
    const ViewPtDF p = view_pt_df(a.T, a.cam, r,
                                  df_add(view_tau(a, hit_k - 1), df_mul_f(a.dstep, q.s)));
    const float ds = -p.f.hi / q.slope, rcp = 1.0f / fabsf(q.slope);
    const DF u = df_add(p.u, DF{ ds * q.du, 0.0f }), v = df_add(p.v, DF{ ds * q.dv, 0.0f });
    // (the slope is good to what the root's own error and 1e-6 move it)
    const float es = (p.err + fabsf(ds) * (fabsf(2.0f * q.a2 * ds) + q.err)) * rcp + 1e-6f * fabsf(ds);
    const float len = fmaxf(fabsf(q.du), fabsf(q.dv));
    const float e = (es + 2.5e-7f * fabsf(ds)) * len + q.off * fabsf(ds) + p.pos;
    if (p.state != 1 || !(fabsf(ds) <= 1e-3f) || !(fminf(u.hi, v.hi) >= 4.0f))
        return view_point64(a, pix, hit_k);
    if (df_hi_is_nearest(u, e) && df_hi_is_nearest(v, e)) return make_float2(u.hi, v.hi);
    double d[3];
    pixel_dir(a.cam, pix, d);
    const double tau = ((double)(hit_k - 1) + ((double)q.s + (double)ds)) * a.step;
    const ViewPt w = view_pt(a.T, a.cam.C, d, tau);
    const double dw = -w.f / (double)q.slope;
    if (!w.in || !(fabs(dw) <= 1e-6)) return view_point64(a, pix, hit_k);
    return make_float2((float)(w.u + dw * (double)q.du), (float)(w.v + dw * (double)q.dv));
}

// Pass 2: the hits of kViewBlock pixels at a time, gathered in shared memory so that
// full warps refine them (a pass-1 warp has a hit in only some of its lanes).  Those
// whose rounding is in doubt wait until a block is full of them, or the last group is
// done, for view_newton.  (3840 x 2160: 4.22 ms; one group per block 4.33; hits left to FP64
// waiting as well 4.34.)  Writes every pixel's texel coordinates (NaN without a hit) and
// the groups' hit counts.
__global__ void __launch_bounds__(kViewBlock, 4) view_refine_kernel(const __grid_constant__ ViewArgs a) {
    __shared__ int32_t s_pix[kViewBlock];
    __shared__ uint32_t s_doubt[2 * kViewBlock];
    __shared__ ViewRoot s_root[2 * kViewBlock];
    __shared__ int32_t s_cnt, s_cnt2;
    const int64_t npix = (int64_t)a.cam.W * a.cam.H;
    const int32_t first = blockIdx.x * a.groups, last = min(first + a.groups, a.n_blocks);
    if (threadIdx.x == 0) s_cnt2 = 0;
    for (int32_t g = first; g < last; ++g) {
        const int64_t base = (int64_t)g * kViewBlock;
        const int64_t pix = base + threadIdx.x;
        if (threadIdx.x == 0) s_cnt = 0;
        __syncthreads();
        const bool mine = pix < npix && a.hit_k[pix] >= 0;
        if (pix < npix && !mine) a.pix_uv[pix] = make_float2(NAN, NAN);
        if (mine) s_pix[atomicAdd(&s_cnt, 1)] = threadIdx.x;
        __syncthreads();
        const int cnt = s_cnt;
        if (threadIdx.x == 0) a.block_count[g] = cnt;
        if ((int)threadIdx.x < cnt) {
            const uint32_t p = (uint32_t)(base + s_pix[threadIdx.x]);
            const int32_t hit_k = a.hit_k[p];
            float2 uv;
            ViewRoot root;
            const int st = view_point_df(a, p, hit_k, uv, root);
            if (st == kViewDoubt) {
                const int i = atomicAdd(&s_cnt2, 1);   // (< kViewBlock waited)
                s_doubt[i] = p;
                s_root[i] = root;
            } else {
                if (st == kViewUnsettled) uv = view_point64(a, p, hit_k);
                a.pix_uv[p] = uv;
            }
        }
        __syncthreads();
        const int cnt2 = s_cnt2;
        if (cnt2 < kViewBlock && g + 1 < last) continue;
        for (int i = threadIdx.x; i < cnt2; i += kViewBlock) {
            const uint32_t p = s_doubt[i];
            a.pix_uv[p] = view_newton(a, p, a.hit_k[p], s_root[i]);
        }
        __syncthreads();
        if (threadIdx.x == 0) s_cnt2 = 0;
    }
}

// exclusive prefix of the per-block counts (one block of 1024 threads)
__global__ void __launch_bounds__(1024) view_scan_kernel(const ViewArgs a) {
    __shared__ int64_t part[1024];
    const int t = threadIdx.x;
    const int per = (a.n_blocks + 1023) / 1024;
    const int lo = min(t * per, a.n_blocks), hi = min(lo + per, a.n_blocks);
    int64_t s = 0;
    for (int b = lo; b < hi; ++b) s += a.block_count[b];
    part[t] = s;
    __syncthreads();
    for (int o = 1; o < 1024; o <<= 1) {   // inclusive Hillis-Steele scan
        const int64_t v = t >= o ? part[t - o] : 0;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    int64_t run = t > 0 ? part[t - 1] : 0;
    for (int b = lo; b < hi; ++b) {
        a.block_off[b] = run;
        run += a.block_count[b];
    }
    if (t == 1023) *a.count_out = part[1023];
}

// scatter the hits of each block to their place in pixel order
__global__ void __launch_bounds__(kViewBlock) view_compact_kernel(const ViewArgs a) {
    __shared__ int32_t warp_base[kViewBlock / 32];
    const int64_t npix = (int64_t)a.cam.W * a.cam.H;
    const int64_t pix = (int64_t)blockIdx.x * kViewBlock + threadIdx.x;
    float2 uv = make_float2(NAN, NAN);
    if (pix < npix) uv = a.pix_uv[pix];
    const bool hit = !isnan(uv.x);
    const unsigned m = __ballot_sync(0xffffffffu, hit);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) warp_base[w] = __popc(m);
    __syncthreads();
    if (threadIdx.x == 0) {
        int32_t s = 0;
        for (int k = 0; k < kViewBlock / 32; ++k) {
            const int32_t c = warp_base[k];
            warp_base[k] = s;
            s += c;
        }
    }
    __syncthreads();
    if (hit) {
        const int64_t o = a.block_off[blockIdx.x] + warp_base[w] +
                          __popc(m & ((1u << lane) - 1u));
        a.uv_out[2 * o] = uv.x;
        a.uv_out[2 * o + 1] = uv.y;
        if (a.pixel_out) a.pixel_out[o] = (int32_t)pix;
    }
}

}  // namespace

int64_t view_blocks(int32_t width, int32_t height) {
    return ((int64_t)width * height + kViewBlock - 1) / kViewBlock;
}

size_t view_workspace_bytes(int32_t width, int32_t height) {
    const int64_t npix = (int64_t)width * height, nb = view_blocks(width, height);
    return (size_t)(npix * 8 + nb * 4 + 256 + nb * 8 + 256 + npix * 4 + 256);
}

cudaError_t launch_view_rays(const Tile& T, const Pyramid& P, const ViewCamera& vc, double step,
                             int64_t K, const float* stats, float* uv, int32_t* pixel,
                             int64_t* count, void* workspace, cudaStream_t s) {
    ViewArgs a{};
    a.T = T;
    a.P = P;
    for (int k = 0; k < 3; ++k) {
        a.cam.C[k] = vc.pos[k];
        a.cam.f[k] = vc.forward[k];
        a.cam.r[k] = vc.right[k];
        a.cam.u[k] = vc.up[k];
    }
    a.cam.tan_x = vc.tan_x;
    a.cam.tan_y = vc.tan_y;
    a.cam.W = vc.width;
    a.cam.H = vc.height;
    a.cam.inv_w2 = 2.0 / (double)vc.width;
    a.cam.inv_h2 = 2.0 / (double)vc.height;
    a.cam.cc = vc.pos[0] * vc.pos[0] + vc.pos[1] * vc.pos[1] + vc.pos[2] * vc.pos[2];
    a.cam.cn = std::sqrt(a.cam.cc);
    a.cam.cxf = (float)vc.pos[0];
    a.cam.cyf = (float)vc.pos[1];
    a.cam.czf = (float)(vc.pos[2] - T.R);
    a.cam.alt = (float)(a.cam.cn - T.R);
    a.cam.zsum = (float)(a.cam.cn + T.R);
    a.cam.inv_2cn = (float)(0.5 / a.cam.cn);
    a.cam.two_r_g = (float)((T.proj == 0 ? 1.0 : 2.0) * T.R / T.g);
    auto split = [](double x) {
        DF d;
        d.hi = (float)x;
        d.lo = (float)(x - (double)d.hi);
        return d;
    };
    // (directions are normalised: any scale serves, one that keeps float32 in range)
    double scale = 0.0;
    for (int k = 0; k < 3; ++k)
        scale = std::fmax(scale, std::fmax(std::fabs(vc.forward[k]),
                                           std::fmax(std::fabs(vc.right[k] * vc.tan_x),
                                                     std::fabs(vc.up[k] * vc.tan_y))));
    if (!(scale > 0.0)) scale = 1.0;
    for (int k = 0; k < 3; ++k) {
        a.cam.rel[k] = split(vc.pos[k] - (k == 2 ? T.R : 0.0));
        a.cam.df[k] = split(vc.forward[k] / scale);
        a.cam.dr[k] = split(vc.right[k] * vc.tan_x / scale);
        a.cam.du[k] = split(vc.up[k] * vc.tan_y / scale);
    }
    a.cam.dalt = split(a.cam.cn - T.R);
    a.cam.dcn = split(a.cam.cn);
    a.cam.dcc = split(a.cam.cc);
    a.cam.dzsum = split(a.cam.cn + T.R);
    a.cam.dR = split(T.R);
    a.cam.dk = split((T.proj == 0 ? 1.0 : 2.0) * T.R / T.g);
    a.cam.diw = split(a.cam.inv_w2);
    a.cam.dih = split(a.cam.inv_h2);
    a.step = step;
    a.dstep = split(step);
    a.step_f = (float)step;
    a.inv_step = (float)(1.0 / step);
    // Float32 heights: the camera's own altitude and, seen from beyond a few radii, the root
    // in rise() near its zero (1e-6 each, replayed as below: at most 1.1 with half of it), plus
    // 2e-7 of the distance for the direction's and tau's roundings (0.5 of it used).  By the
    // sample's own distance: with the largest one allowed, max_dist_m = 2e9 took 1.64 ms
    // instead of 0.39 at 640 x 360.
    a.guard = (float)(0.03 + 1e-6 * std::fabs(a.cam.cn - T.R) * std::fmax(1.0, 0.5 * a.cam.cn / T.R));
    // Float32 texel positions err by the roundings of the coordinates (1.5e-7 (nx + ny))
    // and of the point relative to the tile centre's, 2^-24 of its terms, the camera's
    // distance D0 and tau, times the image's scale (its largest on the tile, heights above
    // -R/5) and 1 + q for the denominator's.  Replayed against 64-bit mantissas (tiles up to 0.8 radii
    // wide, cameras 0.1 to 30,000 km up and to 2.5 radii away, texels of 0.2 to 300 m): at
    // most 1.4 units where the bound takes 4 x 1.25.
    const double qt = std::hypot((double)(T.nx - 1), (double)(T.ny - 1)) * 0.5 * T.g / T.R;
    const double scale_max = 1.25 / T.g * (T.proj == 0 ? std::sqrt(1.0 + qt * qt) : 1.0 + 0.25 * qt * qt);
    const double d0 = std::sqrt(vc.pos[0] * vc.pos[0] + vc.pos[1] * vc.pos[1] +
                                (vc.pos[2] - T.R) * (vc.pos[2] - T.R));
    a.pos_margin = (float)std::fmax(0.01, 3e-7 * (double)(T.nx + T.ny));
    a.pos_t = (float)(2.384185791015625e-07 * scale_max * (1.0 + qt));   // 2^-22
    a.pos_base = (float)(1.5e-7 * (double)(T.nx + T.ny) + (double)a.pos_t * d0);
    a.cam.pos_t = (float)(2.5e-13 * scale_max * (1.0 + qt));
    a.cam.pos0 = (float)((double)a.cam.pos_t * d0 + 2e-14 * (double)(T.nx + T.ny));
    a.cam.height_t = (float)(2e-13 * std::fmax(1.0, 0.5 * a.cam.cn / T.R));
    a.cam.height0 = (float)(2e-13 * std::fabs(a.cam.cn - T.R) + 4e-16 * a.cam.cn);
    a.K = K;
    a.stats = stats;
    const int64_t npix = (int64_t)vc.width * vc.height, nb = view_blocks(vc.width, vc.height);
    unsigned char* ws = static_cast<unsigned char*>(workspace);
    a.pix_uv = reinterpret_cast<float2*>(ws);
    size_t off = (size_t)npix * 8;
    a.block_count = reinterpret_cast<int32_t*>(ws + off);
    off += (size_t)nb * 4;
    off = (off + 255) & ~(size_t)255;
    a.block_off = reinterpret_cast<int64_t*>(ws + off);
    off += (size_t)nb * 8;
    off = (off + 255) & ~(size_t)255;
    a.hit_k = reinterpret_cast<int32_t*>(ws + off);
    a.n_blocks = (int32_t)nb;
    a.uv_out = uv;
    a.pixel_out = pixel;
    a.count_out = count;
    // pixels of a march warp: 256, fewer when the image would not fill the GPU
    const int64_t fill = npix / ((int64_t)device_sm_count() * 32 * 4) / 32 * 32;
    a.pool = (int32_t)(fill < 32 ? 32 : fill > 256 ? 256 : fill);
    const int64_t per_block = (int64_t)a.pool * (kViewHitBlock / 32);
    view_hit_kernel<<<(unsigned)((npix + per_block - 1) / per_block), kViewHitBlock, 0, s>>>(a);
    // groups of a refine block: up to 8 while two waves of resident blocks remain
    const int64_t groups = nb / ((int64_t)device_sm_count() * 8);
    a.groups = (int32_t)(groups < 1 ? 1 : groups > 8 ? 8 : groups);
    view_refine_kernel<<<(unsigned)((nb + a.groups - 1) / a.groups), kViewBlock, 0, s>>>(a);
    view_scan_kernel<<<1, 1024, 0, s>>>(a);
    view_compact_kernel<<<(unsigned)nb, kViewBlock, 0, s>>>(a);
    return cudaGetLastError();
}

}  // namespace ss
