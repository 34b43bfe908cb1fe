// Exact descent over packets of rays (the default of ss_shadow_forward).
//
// A warp takes 32 neighbouring rays at once.  Their sample blocks at the same
// distance cover nearly the same terrain, so the coarse part of the descent is
// shared: blocks of 256 samples, then blocks of 8, are bounded for all 32 rays
// with one maximum M over the union of their footprints (each lane computes the
// M of another block, so a batch of 32 blocks costs one set of gathers), and
// what is left per ray and block is
//
//   prune  <=>  min over the block of  h + rise(t) - best t  >  M + guard,
//
// two fused multiply-adds at each block boundary (below), with no position, no
// gather and no division.  A ray's blocks of 8 samples that survive become
// tasks: a lane takes one (of any ray), bounds its two halves with the ray's
// own footprint, and each half that survives becomes a leaf task, 4 samples
// evaluated by one lane.  Every stage runs with full warps, whatever rays the
// work belongs to.  The running minimum of a ray is the 64-bit key of
// ss_leaftask.cuh (cost bits over sample index) in shared memory, so the
// result is the smallest cost and its smallest index in whatever order the
// samples are evaluated: the same bits as the single-lane walk and uniform
// stepping.
//
// The test.  A sample of the block wins only if (H(t) - h(t)) / t <= best with
// h(t) <= M, that is f(t) = H(t) - best t <= M.  H(t) = h_p + rise(t) is at
// least h_p + c t (B + t) with c a little below 1/(2 rho) (rise_floor below),
// so f is at least a convex quadratic, whose minimum over [ta, tb] is at least
// min(f(ta), f(tb)) - c (tb - ta)^2 / 4.
//
// Listed rays need not be neighbours, so their blocks are tasks from the whole
// ray down (pk_descend_list); the rest is the same.
//
// What bounds it: instruction issue (76% of slots at 2048^2, 30 of 32 lanes active,
// the ALU pipe 52% busy, shared and L1 wavefronts 65%, DRAM 0.1%); per packet of 32
// rays 11.5 k instructions: 12 leaf passes 3.8 k, 13 node passes ~3 k, tests 1 k,
// setup 0.6 k, unions 0.4 k.  Measured (GB300, pass with the mipmap) against the task
// descent of ss_task.cuh: 4096^2 15.3 -> 6.8 ms, 1531 x 1021 2.49 -> 0.72 ms, 256^2
// 1.15 -> 0.063 ms, 1200 x 1000 stereographic 3.59 -> 0.84 ms, 1.04 M view points
// 9.8 -> 1.9 ms, 100 k scattered points 3.2 -> 0.19 ms (the task descent's
// blocks of 6,144 or 3,072 rays leave most SMs idle on all but the first).
// Scalar leaves, tests and one push per node of the packet took 8.0 ms at 4096^2;
// tasks of 16 samples bounded in quarters 7.0 (against 7.1 then), but light-only passes
// 9% and view points 16% more.
#pragma once

#include "ss_forward.cuh"
#include "ss_leaf2.cuh"
#include "ss_leaftask.cuh"

namespace ss {

constexpr int kPkTopLog = 8;       // samples of a top block (log2)
constexpr int kPkNodeLog = 3;      // samples of a node; a top block has 32
constexpr int kPkTop = 1 << kPkTopLog, kPkNode = 1 << kPkNodeLog;
constexpr int kPkNodeRing = 64;    // < 32 tasks wait when up to 32 are added
// Stack of block tasks (listed rays).  A pass takes m tasks off its top and puts
// at most 2 m blocks of half the length back.  m = 32 while at most kPkStackFull
// wait, so entries stay below kPkStackFull + 32; above that m = 8: a block of
// level k then lies below kPkStackFull + 32 + 15 (16 - k), and k >= 3.
constexpr int kPkStackFull = 128, kPkStack = 384;
static_assert(kPkStackFull + 32 + 15 * 13 <= kPkStack, "stack of block tasks");
constexpr int kPkLeafRing = 128;   // < 32 wait when up to 64 are added
constexpr uint32_t kPkSparse = 0x80000000u;   // leaf task of samples j, 6j, 11j, 16j
constexpr float kPkSpread = 512.0f;   // listed rays: neighbours' minima serve as seeds
// Blocks of 4 warps (nothing is shared between warps but the level table; 2 warps
// measure the same), 8 of them per SM: 64 registers.  Three suns at 4096^2: 20.2 ms
// with 8, 20.9 with 6.
#ifndef SS_PK_MIN_BLOCKS
#define SS_PK_MIN_BLOCKS 8
#endif
constexpr int kPkThreads = 128;

// Shared memory of one warp.  ray: what the samples and bounds of a ray read.
template <bool kCount, bool kGrid, bool kLight, bool kStereo>
struct PkWarp {
    static constexpr bool kTexel = kGrid;               // origins at texel centres
    static constexpr bool kShort = kGrid && !kStereo;   // and straight images
    static constexpr int kWords = kShort ? 4 : 5;
    float4 ray[kWords][32];           // word-major: neighbouring slots in different banks
    unsigned long long key[32];
    float M[kGrid ? 32 : 1];          // maxima of a batch of blocks
    uint32_t node[kGrid ? kPkNodeRing : kPkStack];   // (k << 18) | (first / 8 << 5) | slot
    uint32_t leaf[kPkLeafRing];       // (first sample << 5) | slot
    float csat[kLight ? 32 : 1];      // the cost that saturates (negated: umbra)
    int32_t cnt[2][kCount ? 32 : 1];  // probes and samples (counting builds)
};

// A ray's bound test (see the top of this file): f(t) = (c t + cB - best) t + hg
// with hg = h_p - guards, compared with terrain maxima.
struct PkTest {
    float c, cB, hg;
};

// rise(t) = (w / 2 rho) k(x), w = t (B + t), x = w / rho^2, k(x) = 2/(1 + sqrt(1 + x)),
// which falls with x.  So rise >= c w with c = k(x_max) / 2 rho while w >= 0; where
// w < 0 (a sun below the horizon of p) c w exceeds rise by at most
// |w_min| (k(x_min) - k(x_max)) / 2 rho, w_min = -B^2 / 4.
// The guard takes the float32 roundings of the samples and of f: 32 unit
// roundoffs of every magnitude in them, twice (the samples use half of one).
template <bool kGrid>
__device__ __forceinline__ PkTest pk_test(const Tile& T, const RayF& r, float span) {
    PkTest q;
    const float tm = (float)max(r.j_hi, 1) * T.delta_f;
    const float xm = fmaxf(tm * (r.B + tm), 0.0f) * r.inv_rho2;
    const float k = __fdividef(2.0f, 1.0f + sqrtf(1.0f + xm)) * 0.999998f;
    q.c = r.inv_2rho * k;
    q.cB = q.c * r.B;
    float g = 2.0f * r.gconst + kGuardRel * (span + fabsf(r.href) + fabsf(r.X));
    if (r.B < 0.0f) {
        const float w = 0.250001f * r.B * r.B;
        const float kn = __fdividef(2.0f, 1.0f + sqrtf(fmaxf(0.0f, 1.0f - w * r.inv_rho2)));
        g += w * r.inv_2rho * (kn - k + 4e-6f);
    }
    q.hg = (kGrid ? r.href : r.href + r.X) - g;
    return q;
}

__device__ __forceinline__ float pk_f(float c, float p, float hg, float t) {
    return __fmaf_rn(__fmaf_rn(c, t, p), t, hg);
}

template <class Warp>
__device__ __forceinline__ void pk_store(Warp& W, int slot, const RayF& r,
                                         const PkTest& q) {
    const float jr = __uint_as_float((uint32_t)r.j_lo | ((uint32_t)r.j_hi << 16));
    W.ray[0][slot] = make_float4(r.au_hi, r.au_lo, r.av_hi, r.av_lo);
    W.ray[1][slot] = make_float4(r.b, r.href, r.B, r.inv_2rho);
    W.ray[2][slot] = make_float4(r.pos_eps, q.c, q.cB, q.hg);
    if constexpr (Warp::kShort) {
        W.ray[3][slot] = make_float4(jr, r.u0, r.v0, r.inv_rho2);
    } else {
        W.ray[3][slot] = make_float4(jr, r.u0, r.v0, r.inv_rho2);
        W.ray[4][slot] = make_float4(r.bu, r.bv, r.inv8r, r.X);
    }
}

// The ray of a task; jl, jh: its usable samples.
template <class Warp>
__device__ __forceinline__ void pk_load(const Warp& W, int slot, RayF& r, int32_t& jl,
                                        int32_t& jh) {
    const float4 p = W.ray[0][slot], q = W.ray[1][slot], s = W.ray[3][slot];
    r.au_hi = p.x;
    r.au_lo = p.y;
    r.av_hi = p.z;
    r.av_lo = p.w;
    r.b = q.x;
    r.href = q.y;
    r.B = q.z;
    r.inv_2rho = q.w;
    const uint32_t jr = __float_as_uint(s.x);
    jl = (int32_t)(jr & 0xffffu);
    jh = (int32_t)(jr >> 16);
    r.u0 = s.y;
    r.v0 = s.z;
    r.inv_rho2 = s.w;
    if constexpr (Warp::kTexel) {
        r.iu0 = (int32_t)s.y;
        r.iv0 = (int32_t)s.z;
    } else {
        r.iu0 = __float2int_rd(s.y);
        r.iv0 = __float2int_rd(s.z);
    }
    if constexpr (Warp::kShort) {
        r.bu = r.bv = r.inv8r = r.X = 0.0f;
    } else {
        const float4 t = W.ray[4][slot];
        r.bu = t.x;
        r.bv = t.y;
        r.inv8r = t.z;
        r.X = t.w;
    }
    r.au = __fadd_rn(r.au_hi, r.au_lo);
    r.av = __fadd_rn(r.av_hi, r.av_lo);
}

// Maximum height over the texels of the box (bilinear cells of every point in
// it), as <= 2x2 cells of the coarsest level whose cells cover it.
__device__ __forceinline__ float pk_box_max(const Tile& T, const LevelTab& L, int32_t levels,
                                            float xlo, float xhi, float ylo, float yhi) {
    // (clamped so that a box off the tile reads cells of the tile's border)
    const int32_t ax = __vimin_s32_relu(__float2int_rd(xlo), T.nx - 1);
    const int32_t bx = __vimin_s32_relu(__float2int_rd(xhi), T.nx - 2) + 1;
    const int32_t ay = __vimin_s32_relu(__float2int_rd(ylo), T.ny - 1);
    const int32_t by = __vimin_s32_relu(__float2int_rd(yhi), T.ny - 2) + 1;
    const int32_t ext = max(bx - ax, by - ay);
    int32_t m = ext <= 1 ? 0 : 31 - __clz(ext);
    m += (((bx >> m) - (ax >> m)) > 1 || ((by >> m) - (ay >> m)) > 1) ? 1 : 0;
    m = min(m, levels - 1);
    const uint32_t pm = L.pitch[m];
    const float* p = cell_ptr(L.ptr[m], pm, ax >> m, ay >> m);
    const uint32_t dx = (uint32_t)((bx >> m) - (ax >> m));
    const uint32_t dy = (uint32_t)((by >> m) - (ay >> m)) * pm;
    return fmaxf(fmaxf(__ldg(p), __ldg(p + dx)), fmaxf(__ldg(p + dy), __ldg(p + dy + dx)));
}

// What the footprints of a packet's blocks need: ranges over its rays.
template <bool kStereo>
struct PkUnion {
    float u0[2], v0[2], au[2], av[2], b[2], e;
    float B[kStereo ? 2 : 1], i2[kStereo ? 2 : 1], bu[kStereo ? 2 : 1], bv[kStereo ? 2 : 1];
    float inv8r;
};

__device__ __forceinline__ float pk_min(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}
__device__ __forceinline__ float pk_max(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFull, v, o));
    return v;
}
__device__ __forceinline__ void pk_range(float v, float (&o)[2]) {
    o[0] = pk_min(v);
    o[1] = pk_max(v);
}

// rise from w' = t (B + t) and i2 = 1/(2 rho) (relative error ~1e-6)
__device__ __forceinline__ float pk_rise(float w, float i2) {
    return __fdividef(2.0f * w * i2, 1.0f + sqrtf(fmaxf(0.0f, 1.0f + 4.0f * w * i2 * i2)));
}

// Maximum over the union of the rays' footprints of samples [ja, jb].  Interval
// arithmetic over the packet's ranges: gnomonic u = u0 + au tau, tau = j/(1 + b j)
// (increasing in j); stereographic u = u0 + (au j - w bu)/(1 + w b), w = rise +
// t s_z, the image between two samples within the sagitta of their chord.  +inf
// (nothing is pruned) where a denominator may come near zero.
template <bool kStereo>
__device__ __forceinline__ float pk_union_max(const Tile& T, const LevelTab& L, int32_t levels,
                                              const PkUnion<kStereo>& U, int32_t ja, int32_t jb) {
    const float fa = (float)ja, fb = (float)jb;
    float xlo, xhi, ylo, yhi, e = U.e;
    if constexpr (!kStereo) {
        const float da = __fmaf_rn(fa, U.b[1], 1.0f), db = __fmaf_rn(fb, U.b[0], 1.0f);
        if (!(fminf(da, db) > 0.25f)) return INFINITY;
        const float ta = __fdividef(fa, da), tb = __fdividef(fb, db);
        xlo = U.u0[0] + fminf(U.au[0] * ta, U.au[0] * tb);
        xhi = U.u0[1] + fmaxf(U.au[1] * ta, U.au[1] * tb);
        ylo = U.v0[0] + fminf(U.av[0] * ta, U.av[0] * tb);
        yhi = U.v0[1] + fmaxf(U.av[1] * ta, U.av[1] * tb);
    } else {
        xlo = ylo = INFINITY;
        xhi = yhi = -INFINITY;
#pragma unroll
        for (int k = 0; k < 2; ++k) {
            const float f = k ? fb : fa, t = f * T.delta_f;
            // rise grows with w' = t (B + t) and, where w' > 0, falls with rho
            const float w0 = t * (U.B[0] + t), w1 = t * (U.B[1] + t);
            const float r0 = pk_rise(w0, w0 >= 0.0f ? U.i2[0] : U.i2[1]);
            const float r1 = pk_rise(w1, w1 >= 0.0f ? U.i2[1] : U.i2[0]);
            const float ts = t * T.sz_f, pad = 2e-6f * (fabsf(ts) + fabsf(r0) + fabsf(r1));
            const float wl = r0 + ts - pad, wh = r1 + ts + pad;
            const float dl = 1.0f + fminf(wl * U.b[0], wl * U.b[1]);
            const float dh = 1.0f + fmaxf(wh * U.b[0], wh * U.b[1]);
            if (!(dl > 0.25f)) return INFINITY;
            const float il = 1.0f / dl, ih = 1.0f / dh;
            const float pu0 = wl * U.bu[0], pu1 = wl * U.bu[1], pu2 = wh * U.bu[0], pu3 = wh * U.bu[1];
            const float pv0 = wl * U.bv[0], pv1 = wl * U.bv[1], pv2 = wh * U.bv[0], pv3 = wh * U.bv[1];
            const float nul = f * U.au[0] - fmaxf(fmaxf(pu0, pu1), fmaxf(pu2, pu3));
            const float nuh = f * U.au[1] - fminf(fminf(pu0, pu1), fminf(pu2, pu3));
            const float nvl = f * U.av[0] - fmaxf(fmaxf(pv0, pv1), fmaxf(pv2, pv3));
            const float nvh = f * U.av[1] - fminf(fminf(pv0, pv1), fminf(pv2, pv3));
            xlo = fminf(xlo, U.u0[0] + fminf(nul * il, nul * ih));
            xhi = fmaxf(xhi, U.u0[1] + fmaxf(nuh * il, nuh * ih));
            ylo = fminf(ylo, U.v0[0] + fminf(nvl * il, nvl * ih));
            yhi = fmaxf(yhi, U.v0[1] + fmaxf(nvh * il, nvh * ih));
        }
        const float dx = xhi - xlo, dy = yhi - ylo;
        e += arc_bulge(dx * dx + dy * dy, U.inv8r);
    }
    // (a NaN or an overflow in the ranges prunes nothing)
    if (!(xhi - xlo < 1e7f && yhi - ylo < 1e7f)) return INFINITY;
    return pk_box_max(T, L, levels, xlo - e, xhi + e, ylo - e, yhi + e);
}

// The rings of a warp (the same values in every lane).
struct PkRings {
    int32_t nh, nc, lh, lc;
};

// One pass over up to 32 leaf tasks: a lane evaluates 4 samples of one ray.
// (Samples outside the usable range are replaced by the nearest usable one.)
template <bool kCount, bool kGrid, bool kPoly, bool kStereo, class Warp>
__device__ __forceinline__ void pk_leaf_pass(const Tile& T, Warp& W, PkRings& Q, int lane) {
    const int n = min(32, Q.lc);
    if (lane < n) {
        const uint32_t t = W.leaf[(Q.lh + lane) & (kPkLeafRing - 1)];
        const int slot = (int)(t & 31u);
        const int32_t j0 = (int32_t)((t & ~kPkSparse) >> 5);
        const bool sparse = (t & kPkSparse) != 0u;
        RayF q;
        int32_t jl, jh;
        pk_load(W, slot, q, jl, jh);
        const int32_t d = sparse ? 5 * j0 : 1;
        int32_t j[4];
        float c[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            j[i] = min(j0 + i * d, jh);
            if (!kGrid || kStereo) j[i] = max(j[i], jl);
        }
#pragma unroll
        for (int i = 0; i < 4; i += 2) {
            if constexpr (kPoly) {
                leaf_cost2<kGrid, kStereo>(T, q, j[i], j[i + 1], c[i], c[i + 1]);
            } else {
                float rise;
                c[i] = leaf_cost<kGrid, kPoly, kStereo>(T, q, j[i], rise);
                c[i + 1] = leaf_cost<kGrid, kPoly, kStereo>(T, q, j[i + 1], rise);
            }
        }
        const float best = fminf(fminf(c[0], c[1]), fminf(c[2], c[3]));   // (NaN costs drop out)
        // (a stale key is only larger: no better minimum is lost)
        if (best < INFINITY && best <= key_cost(W.key[slot])) {
            const int32_t bj = c[0] == best ? j[0] : c[1] == best ? j[1] : c[2] == best ? j[2] : j[3];
            atomicMin(&W.key[slot], pack_key(best, bj));
        }
        if (kCount) atomicAdd(&W.cnt[1][slot], 1 + (j[1] != j[0]) + (j[2] != j[1]) + (j[3] != j[2]));
    }
    Q.lh = (Q.lh + n) & (kPkLeafRing - 1);
    Q.lc -= n;
    __syncwarp();
}

// One pass over up to 32 block tasks: a lane bounds the two halves of one block
// of one ray.  The halves that may hold the minimum become leaf tasks (blocks
// of 8 samples) or block tasks (longer ones: listed rays only).
template <bool kCount, bool kGrid, bool kPoly, bool kLight, bool kStereo, class Warp>
__device__ __forceinline__ void pk_node_pass(const Tile& T, const LevelTab& L, int32_t levels,
                                             Warp& W, PkRings& Q, int lane) {
    // a gnomonic grid ray's usable samples start at 1.  (A stereographic one's image is an
    // arc: from a texel on the tile's border it can bulge out and come in again.)
    constexpr bool kFirst = kGrid && !kStereo;
    const int n = kGrid || Q.nc <= kPkStackFull ? min(32, Q.nc) : 8;
    bool pa = false, pb = false;
    int32_t s = 0, k = kPkNodeLog;
    int slot = 0;
    // (the children take the places of the tasks read here, and a vote alone orders no
    // memory: the barrier does)
    uint32_t task = 0;
    if (lane < n)
        task = kGrid ? W.node[(Q.nh + lane) & (kPkNodeRing - 1)] : W.node[Q.nc - n + lane];
    if (!kGrid) __syncwarp();
    if (lane < n) {
        slot = (int)(task & 31u);
        if (!kGrid) k = (int32_t)(task >> 18);
        s = (int32_t)((kGrid ? task : task & 0x3ffffu) >> 5) << kPkNodeLog;
        RayF r;
        int32_t jl, jh;
        pk_load(W, slot, r, jl, jh);
        const float4 q = W.ray[2][slot];
        const float best = key_cost(W.key[slot]);
        if (kLight && best <= -W.csat[slot]) jh = 0;   // in full umbra: nothing more to find
        const int32_t half = kGrid ? kPkNode / 2 : 1 << (k - 1);
        // (ends clipped to the usable samples: beyond them the image may leave the plane,
        // 1 + b j <= 0, or pass the antipode, and a box to there would miss the samples)
        const float fs = (float)s, fh = (float)half, fj = (float)jh;
        const float fl = kFirst ? 1.0f : (float)jl;
        const float j0 = kFirst ? fs + 1.0f : fmaxf(fs + 1.0f, fl);
        const float j1 = fmaxf(fminf(fs + (fh + 0.5f), fj), fl);
        const float j2 = fmaxf(fminf(fs + 2.0f * fh, fj), fl);
        const float t0 = j0 * T.delta_f, t1 = j1 * T.delta_f, t2 = j2 * T.delta_f;
        float x0, y0, x1, y1, x2, y2;
        block_end<kStereo>(T, r, j0, t0, kStereo ? rise_of<kPoly>(r, t0) : 0.0f, x0, y0);
        block_end<kStereo>(T, r, j1, t1, kStereo ? rise_of<kPoly>(r, t1) : 0.0f, x1, y1);
        block_end<kStereo>(T, r, j2, t2, kStereo ? rise_of<kPoly>(r, t2) : 0.0f, x2, y2);
        float ea = q.x, eb = q.x;
        if (kStereo) {
            ea += arc_bulge((x1 - x0) * (x1 - x0) + (y1 - y0) * (y1 - y0), r.inv8r);
            eb += arc_bulge((x2 - x1) * (x2 - x1) + (y2 - y1) * (y2 - y1), r.inv8r);
        }
        const float Ma = pk_box_max(T, L, levels, fminf(x0, x1) - ea, fmaxf(x0, x1) + ea,
                                    fminf(y0, y1) - ea, fmaxf(y0, y1) + ea);
        const float Mb = pk_box_max(T, L, levels, fminf(x1, x2) - eb, fmaxf(x1, x2) + eb,
                                    fminf(y1, y2) - eb, fmaxf(y1, y2) + eb);
        const float p = q.z - best, dt = fh * T.delta_f;
        const float hg = __fmaf_rn(-0.2503f * q.y * dt, dt, q.w);
        const float f0 = pk_f(q.y, p, hg, t0), f1 = pk_f(q.y, p, hg, t1);
        const float f2 = pk_f(q.y, p, hg, t2);
        pa = !(fminf(f0, f1) > Ma) && s + 1 <= jh && (kFirst || s + half >= jl);
        pb = !(fminf(f1, f2) > Mb) && s + half + 1 <= jh && (kFirst || s + 2 * half >= jl);
        if (kCount) atomicAdd(&W.cnt[0][slot], 2);
    }
    if (kGrid) Q.nh = (Q.nh + n) & (kPkNodeRing - 1);
    Q.nc -= n;
    const bool leaf = k == kPkNodeLog;
    {
        const unsigned ma = __ballot_sync(kFull, pa && leaf), mb = __ballot_sync(kFull, pb && leaf);
        const int32_t base = Q.lh + Q.lc, na = __popc(ma);
        const uint32_t t = ((uint32_t)(s + 1) << 5) | (uint32_t)slot;
        if (pa && leaf) W.leaf[(base + __popc(ma & lanemask_lt())) & (kPkLeafRing - 1)] = t;
        if (pb && leaf)
            W.leaf[(base + na + __popc(mb & lanemask_lt())) & (kPkLeafRing - 1)] =
                t + (uint32_t)(kPkNode / 2 << 5);
        Q.lc += na + __popc(mb);
    }
    if (!kGrid) {   // far halves first: the near ones are taken off first
        const unsigned mb = __ballot_sync(kFull, pb && !leaf), ma = __ballot_sync(kFull, pa && !leaf);
        const uint32_t t = ((uint32_t)(k - 1) << 18) | ((uint32_t)(s >> kPkNodeLog) << 5) | (uint32_t)slot;
        if (pb && !leaf)
            W.node[Q.nc + __popc(mb & lanemask_lt())] =
                t + ((1u << (k - 1) >> kPkNodeLog) << 5);
        Q.nc += __popc(mb);
        if (pa && !leaf) W.node[Q.nc + __popc(ma & lanemask_lt())] = t;
        Q.nc += __popc(ma);
    }
    __syncwarp();
}

// Node tasks of the lanes in `mine`: node n of ray `slot`.
template <class Warp>
__device__ __forceinline__ void pk_push_nodes(Warp& W, PkRings& Q, bool mine, int32_t n, int slot) {
    const unsigned mk = __ballot_sync(kFull, mine);
    if (mine)
        W.node[(Q.nh + Q.nc + __popc(mk & lanemask_lt())) & (kPkNodeRing - 1)] =
            ((uint32_t)n << 5) | (uint32_t)slot;
    Q.nc += __popc(mk);
    __syncwarp();
}

// The descent of one packet whose rays are in W and whose seeds wait as leaf
// tasks.  jh: the last usable sample of the lane's own ray (0: no ray).  On return
// every sample that could win has been evaluated.  One loop with one copy of each stage: unrolled into
// its callers the code outgrew the instruction cache (the top stall).
template <bool kCount, bool kPoly, bool kLight, bool kStereo, class Warp>
__device__ __forceinline__ void pk_descend(const Tile& T, const LevelTab& L, int32_t levels,
                                           Warp& W, const PkUnion<kStereo>& U, int32_t jh,
                                           PkRings& Q, int lane) {
    const float d = T.delta_f;
    const int32_t jmax = __reduce_max_sync(kFull, jh);
    int32_t s = 0, sn = 0;              // next batch of top blocks; the current top block
    uint32_t tops = 0, any = 0;         // the lane's / the packet's top blocks left
    uint32_t nodes = 0, un = 0;         // nodes left of the current top block / lanes with some
    int32_t st = 0;                     // first sample of the current batch of top blocks
    bool flush = true;                  // drain the rings (first: the seeds)
    while (true) {
        if (Q.lc >= 32 || (flush && Q.nc == 0 && Q.lc > 0)) {
            pk_leaf_pass<kCount, true, kPoly, kStereo>(T, W, Q, lane);
            continue;
        }
        if (Q.nc >= 32 || (flush && Q.nc > 0)) {
            pk_node_pass<kCount, true, kPoly, kLight, kStereo>(T, L, levels, W, Q, lane);
            continue;
        }
        if (un) {                       // each lane's next surviving node becomes a task
            const int n = __ffs(nodes) - 1;
            pk_push_nodes(W, Q, nodes != 0u, (sn >> kPkNodeLog) + n, lane);
            nodes &= nodes - 1u;
            un = __ballot_sync(kFull, nodes != 0u);
            continue;
        }
        flush = false;
        int32_t base, log;
        if (any) {                      // the nodes of the next surviving top block
            const int i = __ffs(any) - 1;
            any &= any - 1u;
            sn = base = st + i * kPkTop;
            log = kPkNodeLog;
            nodes = (tops >> i) & 1u;   // the lane's ray takes part
        } else if (s < jmax) {          // the next 32 top blocks
            st = base = s;
            s += 32 * kPkTop;
            log = kPkTopLog;
            nodes = 1u;
        } else {
            if (Q.nc + Q.lc == 0) break;
            flush = true;
            continue;
        }
        const int32_t a = base + (lane << log);
        float M = -INFINITY;
        if (a < jmax) {
            M = pk_union_max<kStereo>(T, L, levels, U, a + 1, min(a + (1 << log), jmax));
            if (kCount) atomicAdd(&W.cnt[0][lane], 1);
        }
        const float dt = (float)(1 << log) * d;
        // (the lane's own test is read back here: kept in registers across the loop it was
        // spilled, and one build got it wrong)
        const float4 qv = W.ray[2][lane];
        const PkTest q = { qv.y, qv.z, qv.w };
        // curvature term of the block length (0.1%: the roundings of t)
        const float hg = __fmaf_rn(-0.2503f * q.c * dt, dt, q.hg);
        const float best = key_cost(W.key[lane]);
        const float p = q.cB - best;
        uint32_t mask = 0;
        W.M[lane] = M;
        __syncwarp();
        // blocks that hold usable samples of the lane's ray
        if (kLight && best <= -W.csat[lane]) jh = 0;
        const int32_t nv = nodes && jh > base ? min((jh - base + (1 << log) - 1) >> log, 32) : 0;
        const int32_t ng = min((jmax - base + (1 << log) - 1) >> log, 32);   // of any ray's
        const float tb = (float)base * d;
        const F2 c2 = f2(q.c), p2 = f2(p), hg2 = f2(hg), dt2 = f2(dt);
        float f0 = pk_f(q.c, p, hg, tb);
#pragma unroll 2
        for (int g = 0; g < ng; g += 4) {
            const float4 M4 = *reinterpret_cast<const float4*>(&W.M[g]);
            const F2 tg = f2(__fmaf_rn((float)g, dt, tb));
            const F2 ta = f2_fma(f2(1.0f, 2.0f), dt2, tg), tc = f2_fma(f2(3.0f, 4.0f), dt2, tg);
            float f1, f2v, f3, f4;
            f2_get(f2_fma(f2_fma(c2, ta, p2), ta, hg2), f1, f2v);
            f2_get(f2_fma(f2_fma(c2, tc, p2), tc, hg2), f3, f4);
            uint32_t b = !(fminf(f0, f1) > M4.x) ? 1u : 0u;
            b |= !(fminf(f1, f2v) > M4.y) ? 2u : 0u;
            b |= !(fminf(f2v, f3) > M4.z) ? 4u : 0u;
            b |= !(fminf(f3, f4) > M4.w) ? 8u : 0u;
            mask |= b << g;
            f0 = f4;
        }
        mask &= nv >= 32 ? kFull : (1u << nv) - 1u;
        if (log == kPkNodeLog) {
            nodes = mask;
            un = __ballot_sync(kFull, mask != 0u);
        } else {
            tops = mask;
            any = __reduce_or_sync(kFull, mask);
            nodes = 0;
        }
        __syncwarp();                   // W.M is reused by the next batch
    }
}

// The descent of a packet of listed rays, which need not be neighbours: every
// ray's blocks are tasks from its root down (a block of 2^k >= j_hi samples),
// taken last in, first out, the near half of a block first.
template <bool kCount, bool kPoly, bool kLight, bool kStereo, class Warp>
__device__ __forceinline__ void pk_descend_list(const Tile& T, const LevelTab& L, int32_t levels,
                                                Warp& W, int32_t jh, PkRings& Q, int lane) {
    const int32_t k = jh <= kPkNode ? kPkNodeLog : 32 - __clz(jh - 1);
    pk_push_nodes(W, Q, jh > 0, k << 13, lane);
    while (true) {
        if (Q.lc >= 32 || (Q.nc == 0 && Q.lc > 0))
            pk_leaf_pass<kCount, false, kPoly, kStereo>(T, W, Q, lane);
        else if (Q.nc > 0)
            pk_node_pass<kCount, false, kPoly, kLight, kStereo>(T, L, levels, W, Q, lane);
        else
            break;
    }
}

// One packet: setup, seeds, descent, results.  ray: the lane's ray id (a valid
// one in every lane), live: whether it is the lane's to do.  prev_j, pu, pv: a
// finished neighbour's argmin and origin (prev_j < 1: none); on return the
// lane's own.
template <bool kCount, bool kGrid, bool kPoly, bool kLight, bool kStereo, class Warp>
__device__ __forceinline__ void pk_packet(const Tile& T, const LevelTab& L, int32_t levels,
                                          const Rays& R, const Outputs& O, int64_t ray, bool live,
                                          float span, Warp& W, int lane,
                                          int32_t& prev_j, float& pu, float& pv) {
    PkUnion<kStereo> U;
    int32_t jh, jc = -1;
    float csat = INFINITY, u0, v0, au, av;
    {
        RayF rf;
        setup_ray<kGrid, kLight, kStereo>(T, R, ray, span, rf);
        pk_store(W, lane, rf, pk_test<kGrid>(T, rf, span));
        jh = live && rf.j_lo <= rf.j_hi ? rf.j_hi : 0;
        if (kLight) csat = rf.c_sat;
        if (prev_j > 0)
            jc = seed_centre_of(rf.au, rf.av, prev_j, pu - rf.u0, pv - rf.v0);
        u0 = rf.u0;
        v0 = rf.v0;
        au = rf.au;
        av = rf.av;
        if constexpr (kGrid) {   // (a rectangle: the last lane's is the far corner)
            U.u0[0] = __shfl_sync(kFull, rf.u0, 0);
            U.v0[0] = __shfl_sync(kFull, rf.v0, 0);
            U.u0[1] = __shfl_sync(kFull, rf.u0, 31);
            U.v0[1] = __shfl_sync(kFull, rf.v0, 31);
        } else {
            pk_range(rf.u0, U.u0);
            pk_range(rf.v0, U.v0);
        }
        if constexpr (kGrid) {
            pk_range(rf.au, U.au);
            pk_range(rf.av, U.av);
            pk_range(rf.b, U.b);
            U.e = pk_max(rf.pos_eps) * 1.5f + 1e-3f;
            U.inv8r = 0.0f;
        }
        if constexpr (kGrid && kStereo) {
            pk_range(rf.B, U.B);
            pk_range(rf.inv_2rho, U.i2);
            pk_range(rf.bu, U.bu);
            pk_range(rf.bv, U.bv);
            U.inv8r = pk_max(rf.inv8r);
        }
    }
    // (light-only: a sample has to be below the saturated cost; index 0: none was)
    W.key[lane] = kLight ? pack_key(csat, 0) : kKeyNone;
    if (kLight) W.csat[lane] = csat;
    if (kCount) W.cnt[0][lane] = W.cnt[1][lane] = 0;
    PkRings Q = { 0, 0, 0, 0 };
    // seeds: samples around where the neighbour's argmin lies along this ray, else
    // samples 1, 6, 11, 16, 96, ... 2^16 (at most 4 tasks per lane: the ring holds them)
    const auto push_seed = [&](bool mine, uint32_t first) {
        const unsigned m = __ballot_sync(kFull, mine);
        if (mine)
            W.leaf[(Q.lh + Q.lc + __popc(m & lanemask_lt())) & (kPkLeafRing - 1)] =
                (first << 5) | (uint32_t)lane;
        Q.lc += __popc(m);
    };
    const auto near_seed = [&](bool mine, int32_t j) {
        push_seed(mine && j >= 0, (uint32_t)min(max(j - 1, 1), max(jh, 1)));
    };
    const auto sparse_seeds = [&](bool mine) {
        for (int32_t j = 1; j <= 4096; j <<= 4)
            push_seed(mine && j <= jh, (kPkSparse >> 5) | (uint32_t)j);
    };
    if constexpr (kGrid) {
        near_seed(jh > 0, jc);
        sparse_seeds(!kLight && jh > 0 && jc < 0);
        __syncwarp();
        pk_descend<kCount, kPoly, kLight, kStereo>(T, L, levels, W, U, jh, Q, lane);
    } else {
        // Listed rays that are neighbours (a view's): every fourth ray first, seeded as
        // above and around each other's minima, then the others around the minima of
        // the two nearest of those.
        const bool close = fmaxf(U.u0[1] - U.u0[0], U.v0[1] - U.v0[0]) <= kPkSpread;
        const bool two = close && !kLight;
        for (int phase = 0; phase < (two ? 2 : 1); ++phase) {
            const bool go = jh > 0 && (!two || ((lane & 3) == 0) == (phase == 0));
            const int rounds = !two ? 1 : phase == 0 ? 4 : 2;
            for (int r = 0; r < rounds; ++r) {
                if (r == 0 && phase == 0) {
                    near_seed(go && close, jc);
                    sparse_seeds(!kLight && go && !(close && jc >= 0));
                } else {
                    const int src = phase == 0 ? lane ^ (32 >> r)
                                    : r == 0 ? lane & 28 : (lane & 28) + (lane < 28 ? 4 : -4);
                    const int32_t jo = key_j(W.key[src]);
                    const float4 o = W.ray[3][src];
                    near_seed(go && jo > 0, seed_centre_of(au, av, jo, o.y - u0, o.z - v0));
                }
                __syncwarp();
                while (Q.lc > 0) pk_leaf_pass<kCount, kGrid, kPoly, kStereo>(T, W, Q, lane);
            }
            pk_descend_list<kCount, kPoly, kLight, kStereo>(T, L, levels, W, go ? jh : 0, Q, lane);
        }
    }
    if (kCount) {   // shared bounds counted in lanes without a ray: to the packet's first ray
        const unsigned mine = __ballot_sync(kFull, live);
        const unsigned lost = __reduce_add_sync(kFull, live ? 0u : (unsigned)W.cnt[0][lane]);
        if (mine && lane == __ffs(mine) - 1) W.cnt[0][lane] += (int32_t)lost;
    }
    const unsigned long long key = W.key[lane];
    const int32_t bj = kLight && key_j(key) == 0 ? -1 : key_j(key);
    if (live)
        finish_ray<kStereo, kRefineLater>(T, R, O, ray, key_cost(key), bj, kCount ? W.cnt[0][lane] : 0,
                                  kCount ? W.cnt[1][lane] : 0);
    prev_j = bj;
    pu = u0;
    pv = v0;
    __syncwarp();
}

// A strip of k.len grid packets of 8 columns, one below the other; the last row of
// one seeds the next.  Strips run row by row over the tile.  Lanes without a ray
// repeat one of the packet's.
template <bool kCount, bool kPoly, bool kLight, bool kStereo, class Warp>
__device__ __forceinline__ void pk_grid_strip(const Tile& T, const LevelTab& L, int32_t levels,
                                              const Rays& R, const Outputs& O, uint32_t strip,
                                              PkShape sh, float span, Warp& W, int lane) {
    const uint32_t nbx = (uint32_t)(T.nx + kPkCols - 1) / kPkCols;
    const uint32_t band = strip / nbx;
    const int32_t x = (int32_t)(strip - band * nbx) * kPkCols + (lane & (kPkCols - 1));
    const int32_t rows = sh.rays / kPkCols, row = min(lane / kPkCols, rows - 1);
    const int64_t y0 = (int64_t)band * sh.len * rows;
    int32_t prev_j = -1;
    float pu = 0.0f, pv = 0.0f;
    for (int k = 0; k < sh.len && y0 + k * rows < T.ny; ++k) {
        const int32_t y = (int32_t)y0 + k * rows + row;
        const bool live = lane < sh.rays && x < T.nx && y < T.ny;
        const int64_t ray = (int64_t)min(y, T.ny - 1) * T.nx + min(x, T.nx - 1);
        pk_packet<kCount, true, kPoly, kLight, kStereo>(T, L, levels, R, O, ray, live, span, W,
                                                        lane, prev_j, pu, pv);
        const int below = sh.rays - kPkCols + (lane & (kPkCols - 1));   // the last row's column
        prev_j = __shfl_sync(kFull, prev_j, below);
        pu = __shfl_sync(kFull, pu, below);
        pv = __shfl_sync(kFull, pv, below);
    }
}

// Each warp takes a strip of a.pk.len packets (listed rays: a.pk.rays consecutive
// ids each).
template <bool kCount, bool kGrid, bool kPoly, bool kLight, bool kStereo>
__global__ void __launch_bounds__(kPkThreads, SS_PK_MIN_BLOCKS)
dp_packet_kernel(const __grid_constant__ FwdArgs a) {
    __shared__ LevelTab s_lev;
    __shared__ PkWarp<kCount, kGrid, kLight, kStereo> s_w[kPkThreads / 32];
    if (threadIdx.x < kMaxLevels) {
        s_lev.ptr[threadIdx.x] = a.P.ptr[threadIdx.x];
        s_lev.pitch[threadIdx.x] = (uint32_t)a.P.pitch[threadIdx.x];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) report_nonfinite_heights(a.stats, a.O.status);
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const uint32_t strip = blockIdx.x * (kPkThreads / 32) + (threadIdx.x >> 5);
    const float span = a.stats[0] - a.stats[1];
    auto& W = s_w[threadIdx.x >> 5];
    if constexpr (kGrid) {
        pk_grid_strip<kCount, kPoly, kLight, kStereo>(a.T, s_lev, a.P.levels, a.R, a.O, strip,
                                                      a.pk, span, W, lane);
    } else {
        int32_t prev_j = -1;
        float pu = 0.0f, pv = 0.0f;
        const int32_t m = a.pk.rays, own = min(lane, m - 1);
        const int64_t first = (int64_t)strip * a.pk.len * m;
        for (int k = 0; k < a.pk.len && first + k * m < a.R.n; ++k) {
            const int64_t id = first + k * m + own;
            pk_packet<kCount, kGrid, kPoly, kLight, kStereo>(
                a.T, s_lev, a.P.levels, a.R, a.O, min(id, a.R.n - 1), lane < m && id < a.R.n,
                span, W, lane, prev_j, pu, pv);
        }
    }
}

template <bool C, bool G, bool P, bool L, bool S>
static void launch_packet(const FwdArgs& a, cudaStream_t s) {
    const int64_t n = a.R.mode == 0 ? (int64_t)a.T.nx * a.T.ny : a.R.n;
    const int64_t per = (int64_t)a.pk.rays * a.pk.len;
    const int64_t strips = a.R.mode == 0 ? pk_grid_strips(a.T.nx, a.T.ny, a.pk) : (n + per - 1) / per;
    const int64_t grid = (strips + kPkThreads / 32 - 1) / (kPkThreads / 32);
    dp_packet_kernel<C, G, P, L, S><<<(unsigned)grid, kPkThreads, 0, s>>>(a);
}

}  // namespace ss
