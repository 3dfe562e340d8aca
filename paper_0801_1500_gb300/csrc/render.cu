// Render kernels, wavefront style, for one frame or a batch of frames:
//   k_patch_grids  (frames whose grid was rebuilt on the device) copies the
//              rebuilt geometry into the frame descriptors;
//   k_primary  persistent; each warp pulls a 32-pixel tile of some frame from
//              an atomic queue, walks the primary rays (nearest hit), refines
//              the winner in its object's frame and appends the hit (AO
//              origin, normal) to its frame's hit list; the last CTA to
//              finish lays out the AO pass (prefix sums of hits and AO rays
//              per frame);
//   k_ao_near  (frames with rays enough) tests the AO rays of a tile
//              against the balls around it before they walk;
//   k_ao_walk  persistent; each lane holds one AO (or direct-light shadow)
//              ray; a warp refills its idle lanes together from its ray pool
//              once fewer than `refill` lanes still hold a ray, walks all of
//              them in lockstep (several cells per iteration), expands the
//              (ray, object) pairs over the lanes and tests them 32 at a
//              time; k_ao_walk64 walks the rays of FP64 frames one a lane,
//              settling in FP32 every pair that FP32 error bounds decide;
//   k_shade    one thread per hit: Phong + skylight with V = escaped / spp;
//   k_resolve  (supersampled frames) box-filters the finer raster.
// Plus the AO probe and the raw Philox kernel.
#include <string.h>

#include <algorithm>
#include <cmath>
#include <functional>
#include <type_traits>
#include <vector>

#include "gbrt_device.cuh"
#include "gbrt_internal.h"

namespace gbrt {

constexpr unsigned FULL = 0xffffffffu;

// A kernel launched as a programmatic dependent of the previous one in its
// stream (launch_dependent) starts while that kernel drains; it waits here,
// before reading anything the previous kernel wrote, until the previous grid
// has finished and its writes are visible. Without that launch attribute the
// wait returns at once.
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Largest f with off[f] <= x (off nondecreasing, x < off[n]).
template <class T>
__device__ __forceinline__ int find_frame(const T* off, int n, T x) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) >> 1;
        if (off[mid] <= x) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Primary ray of pixel (i, j), in FP64 (both paths derive their ray from it).
// 1/W, 1/H and the unit view direction come precomputed with the frame.
__device__ __forceinline__ void primary_ray64(const FrameDev& f, int i, int j, V3<double>& o, V3<double>& d) {
    double u = f.half_w * fma((double)(2 * i + 1), f.inv_w, -1.0);
    double v = f.half_h * fma(-(double)(2 * j + 1), f.inv_h, 1.0);
    V3<double> up = ld3(f.up), right = ld3(f.right);
    if (f.cam_kind == GBRT_CAMERA_ORTHO) {
        o = madd(madd(ld3(f.eye), u, right), v, up);
        d = ld3(f.dir_unit);
    } else {
        o = ld3(f.eye);
        V3<double> q = madd(madd(ld3(f.dir_unit), u, right), v, up);
        d = rsqrt(dot(q, q)) * q;
    }
}

// View direction of pixel q in FP32 (shading only).
__device__ __forceinline__ V3<float> view_dir_f(const FrameDev& f, uint32_t q) {
    V3<float> d = v3(f.dir_f[0], f.dir_f[1], f.dir_f[2]);
    if (f.cam_kind == GBRT_CAMERA_ORTHO) return d;
    const int i = (int)(q % (uint32_t)f.W), j = (int)(q / (uint32_t)f.W);
    float u = f.half_w_f * fmaf((float)(2 * i + 1), f.inv_w_f, -1.0f);
    float v = f.half_h_f * fmaf(-(float)(2 * j + 1), f.inv_h_f, 1.0f);
    d = madd(madd(d, u, v3(f.right_f[0], f.right_f[1], f.right_f[2])), v, v3(f.up_f[0], f.up_f[1], f.up_f[2]));
    return rsqrtf(dot(d, d)) * d;
}

// Float-float arithmetic (Dekker 1971, Knuth's TwoSum): a value held as an
// unevaluated sum hi + lo of two floats, about 48 bits. The float path forms
// its primary ray and the two points it rounds from that ray this way, on the
// FP32 pipe, instead of in FP64 (a GB300 SM runs FP64 at 1/64 of the FP32
// rate). Products and sums use the _rn intrinsics so that no step is fused.
struct Ff3 {
    V3<float> hi, lo;
};

// s + e = a + b exactly (s the rounded sum)
__device__ __forceinline__ void two_sum(float a, float b, float& s, float& e) {
    s = __fadd_rn(a, b);
    const float bb = __fsub_rn(s, a);
    e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// round(x + t d - p), one component: x and d float pairs, t and p floats
__device__ __forceinline__ float ff_point(float xh, float xl, float t, float dh, float dl, float p) {
    float s1, e1, s2, e2;
    two_sum(xh, -p, s1, e1);
    const float pr = __fmul_rn(t, dh);
    const float ep = __fmaf_rn(t, dh, -pr);  // t dh - pr exactly
    two_sum(s1, pr, s2, e2);
    return __fadd_rn(s2, __fadd_rn(__fadd_rn(xl, e1), __fadd_rn(__fadd_rn(e2, ep), __fmul_rn(t, dl))));
}

// x + t d - p rounded to float, per component
__device__ __forceinline__ V3<float> ff_point3(const Ff3& x, float t, const Ff3& d, V3<float> p) {
    return v3(ff_point(x.hi.x, x.lo.x, t, d.hi.x, d.lo.x, p.x), ff_point(x.hi.y, x.lo.y, t, d.hi.y, d.lo.y, p.y),
              ff_point(x.hi.z, x.lo.z, t, d.hi.z, d.lo.z, p.z));
}

// round(x + t d) and what the rounding left out (x + t d = point + rest to
// about 2^-48 of the point), one component
__device__ __forceinline__ float ff_entry(float xh, float xl, float t, float dh, float dl, float& rest) {
    const float pr = __fmul_rn(t, dh);
    const float ep = __fmaf_rn(t, dh, -pr);
    float s, e;
    two_sum(xh, pr, s, e);
    const float l = __fadd_rn(__fadd_rn(xl, e), __fadd_rn(ep, __fmul_rn(t, dl)));
    const float pt = __fadd_rn(s, l);
    rest = __fsub_rn(l, __fsub_rn(pt, s));
    return pt;
}

// a0 + i ai + j aj as a float pair (i, j below 2^24, so i ai_hi and j aj_hi
// are split exactly by an FMA)
__device__ __forceinline__ void ff_affine(float a0h, float a0l, float fi, float aih, float ail, float fj, float ajh,
                                          float ajl, float& hi, float& lo) {
    const float p1 = __fmul_rn(fi, aih), e1 = __fmaf_rn(fi, aih, -p1);
    const float p2 = __fmul_rn(fj, ajh), e2 = __fmaf_rn(fj, ajh, -p2);
    float s1, r1, s2, r2;
    two_sum(a0h, p1, s1, r1);
    two_sum(s1, p2, s2, r2);
    const float l = __fadd_rn(__fadd_rn(__fadd_rn(a0l, __fmul_rn(fi, ail)), __fadd_rn(e1, e2)),
                              __fadd_rn(__fadd_rn(r1, r2), __fmul_rn(fj, ajl)));
    hi = __fadd_rn(s2, l);  // |l| is far below |s2|: a fast two-sum renormalises
    lo = __fsub_rn(l, __fsub_rn(hi, s2));
}

// a.hi + a.lo times b.hi + b.lo, as a pair (the lo * lo term dropped)
__device__ __forceinline__ void ff_mul(float ah, float al, float bh, float bl, float& hi, float& lo) {
    const float p = __fmul_rn(ah, bh);
    const float e = __fadd_rn(__fmaf_rn(ah, bh, -p), __fadd_rn(__fmul_rn(ah, bl), __fmul_rn(al, bh)));
    hi = __fadd_rn(p, e);
    lo = __fsub_rn(e, __fsub_rn(hi, p));
}

// q / |q| as float pairs. 1/|q| starts from the hardware rsqrtf of |q|^2's
// high part and takes one Newton-Raphson step for the reciprocal square root,
// y1 = y0 + y0 (1 - n y0^2) / 2, with the residual 1 - n y0^2 formed from
// exact products; the step leaves about twice the seed's bits.
__device__ __forceinline__ void ff_normalise(Ff3& q) {
    float n, ne;  // |q|^2 = n + ne
    {
        float sq, se;
        ff_mul(q.hi.x, q.lo.x, q.hi.x, q.lo.x, n, ne);
        ff_mul(q.hi.y, q.lo.y, q.hi.y, q.lo.y, sq, se);
        float s, e;
        two_sum(n, sq, s, e);
        n = s;
        ne = __fadd_rn(__fadd_rn(ne, se), e);
        ff_mul(q.hi.z, q.lo.z, q.hi.z, q.lo.z, sq, se);
        two_sum(n, sq, s, e);
        n = s;
        ne = __fadd_rn(__fadd_rn(ne, se), e);
    }
    const float y0 = rsqrtf(n);
    float a, b;  // y0^2 = a + b exactly
    a = __fmul_rn(y0, y0);
    b = __fmaf_rn(y0, y0, -a);
    float c, cd;  // n a = c + cd exactly
    c = __fmul_rn(n, a);
    cd = __fmaf_rn(n, a, -c);
    // 1 - (n + ne)(a + b); 1 - c is exact (c is within a few ulp of 1)
    const float r = __fsub_rn(__fsub_rn(__fsub_rn(1.0f, c), cd), __fadd_rn(__fmul_rn(n, b), __fmul_rn(ne, a)));
    const float yl = __fmul_rn(__fmul_rn(0.5f, y0), r);
    ff_mul(q.hi.x, q.lo.x, y0, yl, q.hi.x, q.lo.x);
    ff_mul(q.hi.y, q.lo.y, y0, yl, q.hi.y, q.lo.y);
    ff_mul(q.hi.z, q.lo.z, y0, yl, q.hi.z, q.lo.z);
}

// The float path's primary ray of pixel (i, j) as float pairs, with no FP64:
// the orthographic origin, or the pinhole direction before normalisation, is
// affine in (i, j).
__device__ __forceinline__ void primary_ray_ff(const FrameDev& f, int i, int j, Ff3& o, Ff3& d) {
    const float fi = (float)i, fj = (float)j;
    Ff3 v;
    ff_affine(f.a0_hi[0], f.a0_lo[0], fi, f.ai_hi[0], f.ai_lo[0], fj, f.aj_hi[0], f.aj_lo[0], v.hi.x, v.lo.x);
    ff_affine(f.a0_hi[1], f.a0_lo[1], fi, f.ai_hi[1], f.ai_lo[1], fj, f.aj_hi[1], f.aj_lo[1], v.hi.y, v.lo.y);
    ff_affine(f.a0_hi[2], f.a0_lo[2], fi, f.ai_hi[2], f.ai_lo[2], fj, f.aj_hi[2], f.aj_lo[2], v.hi.z, v.lo.z);
    if (f.cam_kind == GBRT_CAMERA_ORTHO) {
        o = v;
        d.hi = v3(f.dir_hi[0], f.dir_hi[1], f.dir_hi[2]);
        d.lo = v3(f.dir_lo[0], f.dir_lo[1], f.dir_lo[2]);
    } else {
        o.hi = v3(f.eye_hi[0], f.eye_hi[1], f.eye_hi[2]);
        o.lo = v3(f.eye_lo[0], f.eye_lo[1], f.eye_lo[2]);
        ff_normalise(v);
        d = v;
    }
}

// Refinement of an FP32 root in the object's own frame. The FP32 walk's root t
// (along the ray x + t d, x its grid-entry point) is turned into the hit's
// offset from the object's base point p0 -- the point x + t d - p0 formed from
// float pairs (p0 is a float: the scene's coordinates are) and rounded to
// FP32; it has the size of the object (|w| <= r + L), so FP32 holds it to
// ~1e-7 of that -- and Newton steps in FP32 then move it along the ray by s to
// the surface: F(s) = |w_p + s d_p|^2 - r^2 (w_p, d_p: the parts perpendicular
// to the axis a; all of w and d for a sphere). The result is the offset w + s d
// (the re-projection then needs no more precision than FP32) and the root
// t + s, exactly, as a float pair for ranking near-ties. False when the steps
// do not settle (a grazing ray): the offset then stays at the FP32 root's
// point.
struct LocalHit {
    V3<float> w;     // hit point - p0
    float t, t_lo;   // root along the ray from its grid entry: t + t_lo exactly
};

// x = (oe, rest): the ray's grid-entry point and what its rounding left out;
// t: the FP32 root measured from oe along d (d.hi: the walk's direction)
__device__ __forceinline__ bool local_root(const SceneDev& sc, uint32_t id, const Ff3& x, const Ff3& d, float t,
                                           LocalHit& lh) {
    const V3<float> df = d.hi;
    V3<float> p0f, a;
    float L, r;
    Obj<float>::load(sc.obj, id, p0f, a, L, r);
    const V3<float> w = ff_point3(x, t, d, p0f);
    const float wa = dot_zyx(w, a), da = dot(df, a);
    const V3<float> wp = madd(w, -wa, a), dp = madd(df, -da, a);
    const float A = dot(dp, dp), B = dot(wp, dp), C = fmaf(-r, r, dot(wp, wp));
    float s = 0.0f, corr = 0.0f;
#pragma unroll
    for (int it = 0; it < 2; ++it) {
        const float As = A * s;
        corr = __fdividef(fmaf(As + 2.0f * B, s, C), 2.0f * (As + B));
        s -= corr;
    }
    const bool ok = fabsf(corr) <= 1e-4f * (fabsf(s) + r) && isfinite(s);
    if (!ok) s = 0.0f;
    lh.w = madd(w, s, df);
    two_sum(t, s, lh.t, lh.t_lo);
    return ok;
}

// The ray's grid-entry point at te0, rounded once (x.hi), and what the
// rounding left out (x.lo).
__device__ __forceinline__ void entry_point(const Ff3& o, const Ff3& d, float te0, Ff3& x) {
    x.hi.x = ff_entry(o.hi.x, o.lo.x, te0, d.hi.x, d.lo.x, x.lo.x);
    x.hi.y = ff_entry(o.hi.y, o.lo.y, te0, d.hi.y, d.lo.y, x.lo.y);
    x.hi.z = ff_entry(o.hi.z, o.lo.z, te0, d.hi.z, d.lo.z, x.lo.z);
}

// FP32 path: nearest hit in FP32 from the float-float ray re-based at its
// grid entry te0 (one rounding, so coordinates stay small relative to the
// scene).
template <bool SPLIT>
__device__ __forceinline__ void nearest_fp32(const FrameDev& f, int i, int j, bool on, int sub, int parts, float& te0,
                                             Nearest& h, bool& overflow) {
    if (!SPLIT && !on) return;
    const float inf = Num<float>::inf();
    Ff3 o, d, x;
    primary_ray_ff(f, i, j, o, d);
    float te1;
    if (!clip_grid(f.grid, o.hi, d.hi, 0.0f, inf, te0, te1)) {
        if (!SPLIT) return;
        on = false;
    }
    // the walk starts at the entry point rounded once
    entry_point(o, d, te0, x);
    trace_nearest<SPLIT>(f.grid, f.scene, x.hi, d.hi, on, sub, parts, h, overflow);
    // the lanes' hits, merged
    for (int y = 1; SPLIT && y < parts; y <<= 1) {
        const float t1 = __shfl_xor_sync(FULL, h.t1, y), t2 = __shfl_xor_sync(FULL, h.t2, y);
        const uint32_t k1 = __shfl_xor_sync(FULL, h.id1, y), k2 = __shfl_xor_sync(FULL, h.id2, y);
        if (k1 != GBRT_MISS) nearest_consider(h, k1, t1);
        if (k2 != GBRT_MISS) nearest_consider(h, k2, t2);
    }
}

// The winner -- and a runner-up within a relative 1e-4 band -- refined in its
// object's frame (local_root); the nearer refined root wins.
__device__ __forceinline__ void refine_fp32(const FrameDev& f, int i, int j, float te0, const Nearest& h,
                                            uint32_t& id, LocalHit& lh) {
    // the refinement needs what the rounding left out: the ray and its entry
    // point are formed again (the same steps give the same floats), which is
    // cheaper than holding their low parts in registers through the walk
    // (the copies of i and j keep the compiler from reusing the first ones)
    Ff3 o, d, x;
    int i2, j2;
    asm volatile("mov.b32 %0, %1;" : "=r"(i2) : "r"(i));
    asm volatile("mov.b32 %0, %1;" : "=r"(j2) : "r"(j));
    primary_ray_ff(f, i2, j2, o, d);
    entry_point(o, d, te0, x);
    local_root(f.scene, h.id1, x, d, h.t1, lh);
    id = h.id1;
    if (h.id2 != GBRT_MISS && (h.t2 - h.t1) <= 1e-4f * (h.t1 + te0)) {
        LocalHit l2;
        local_root(f.scene, h.id2, x, d, h.t2, l2);
        // t + t_lo pairs are normalised, so comparing them in order compares
        // the exact roots
        const bool nearer = l2.t < lh.t || (l2.t == lh.t && l2.t_lo < lh.t_lo);
        const bool same = l2.t == lh.t && l2.t_lo == lh.t_lo;
        if (nearer || (same && h.id2 < h.id1)) {
            id = h.id2;
            lh = l2;
        }
    }
}

// ---------------------------------------------------------------- FP32 filters of FP64 decisions

// The object filter. Every candidate of a cell is first tested, in FP32, as a
// ball: a sphere itself, or the sphere around a tube (SceneDev::bs, tubes
// marked by a negative radius). With b = w.d / d.d the ray's parameter at the
// ball's centre (w = o - centre), m = w - b d the ray's offset there and
// x = |m|^2 + max(b, 0)^2 - r^2, a ray that starts outside or inside the ball
// meets it ahead exactly when x <= 0 (b > 0: the centre lies behind, and
// |m|^2 + b^2 = |w|^2). filter_margin bounds the rounding of x ten times over:
// |m| is wrong by at most ~4e-7 (|b| + r) -- w is one rounding of exact floats,
// b's error only moves m along the ray -- and so is the reference test's own |m|;
// the square of that counts for a ball that is tiny against its distance (1e-9
// of it: without the square, 188 of 1,600 pixels were wrong). So x > margin is a
// miss and, for a sphere, x < -margin a hit that the reference test (hit_prim, or
// any_hit_object64 in FP64) decides the same way; what lies between is left to
// that test. A miss, nine candidates in ten, costs ~20 instructions instead of
// ~45, and in the FP64 path no FP64 instruction.
// reach: |b| + r, and for coordinates relative to a grid what their rounding adds.
__device__ __forceinline__ float filter_margin(float r, float reach) {
    return reach * fmaf(2e-12f, reach, 1e-5f * r);
}

// What a filter says of one (ray, object) pair.
enum : int { PAIR_MISS = 0, PAIR_HIT = 1, PAIR_OPEN = 2 };

// A tube in FP32, with error bounds. The arithmetic is hit_prim's; em bounds
// the error of the offset m (ten times over), et that of a root's t. On PAIR_HIT t is the nearest root in (0, tmax] and et its error.
// tlim: a root up to tlim - et is surely within tmax.
__device__ __forceinline__ int tube_root32(V3<float> o, V3<float> d, V3<float> p0, V3<float> a, float L, float r,
                                           float tlim, float tmax, float om, float& t, float& et) {
    const V3<float> w = o - p0;
    const float wa = dot(w, a), da = dot(d, a);
    const V3<float> wp = madd(w, -wa, a), dp = madd(d, -da, a);
    const float A = dot(dp, dp);
    if (!(A > 1e-3f)) return PAIR_OPEN;
    const float inv = 1.0f / A;
    const float tc = -dot(wp, dp) * inv;
    const V3<float> m = madd(wp, tc, dp);
    const float em = 4e-6f * (fabsf(tc) + L + r + om);
    const float disc = r * r - dot(m, m), md = 2.0f * (r + em) * em;
    if (disc < -md) return PAIR_MISS;
    if (!(disc > md)) return PAIR_OPEN;
    const float half = sqrtf(disc * inv);
    et = em * inv + md * inv / half;
    const float es = et + em;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        t = k ? tc + half : tc - half;
        const float s = wa + t * da;
        if (t > et && t < tlim - et && s > es && s < L - es) return PAIR_HIT;
        // a root that may count leaves the pair open, one that cannot is passed
        if (t > -et && t < tmax + et && s > -es && s < L + es) return PAIR_OPEN;
    }
    return PAIR_MISS;
}

// A sphere's nearest root ahead, from the filter's values: the ray's parameter
// tc at the centre, |m|^2 - r^2 and the margin of the latter.
__device__ __forceinline__ int sphere_root32(float tc, float x, float mg, float r, float om, float& t, float& et) {
    if (!(-x > mg)) return PAIR_OPEN;
    const float half = sqrtf(-x);
    et = 1e-6f * (fabsf(tc) + r + om) + mg / half;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        t = k ? tc + half : tc - half;
        if (t > et) return PAIR_HIT;
        if (t > -et) return PAIR_OPEN;
    }
    return PAIR_MISS;
}

// The exact root of pixel (i, j)'s FP64 ray with object id (infinity: none).
__device__ __noinline__ double exact_root64(const FrameDev& f, int i, int j, uint32_t id) {
    V3<double> o, d;
    double t;
    primary_ray64(f, i, j, o, d);
    return hit_object<double>(f.scene, id, o, d, 0.0, Num<double>::inf(), t) ? t : Num<double>::inf();
}

// FP64 path: the nearest object of pixel (i, j)'s ray. The walk and the roots
// are FP32, relative to the grid's lower corner, along the float-float ray from
// just before it enters the objects' bounds; each root carries its error, and
// FP64 roots (exact_root64) decide where the bounds do not: a pair too close
// to grazing, to the tube's end or to the ray's start, and two roots closer
// than their errors; the walk ends where the nearest root, with its error, lies
// before the cell's exit. The object is the one an FP64 walk finds; its FP64 root
// is formed by the caller, once per hit pixel instead of once per candidate
// (965 x 1137 frame, this kernel: 2.40 -> 0.205 ms; 256 x 256: 0.39 ->
// 0.049 ms. The FP64 pipe was the bound; now the walk's load latency and the
// winners' ~140 FP64 instructions are).
struct Near64 {
    uint32_t id;    // GBRT_MISS: none
    float t, e;     // its root from the grid entry, and that root's error
    uint32_t pend;  // a candidate that only FP64 can place (GBRT_MISS: none)
    float lo;       // which has no root before this
};

__device__ __forceinline__ void near64_settle(const FrameDev& f, int i, int j, float te0, Near64& h, uint32_t cand) {
    const double t64 = exact_root64(f, i, j, cand);
    if (t64 == Num<double>::inf()) return;
    const double b64 = h.id == GBRT_MISS ? Num<double>::inf() : exact_root64(f, i, j, h.id);
    if (t64 < b64 || (t64 == b64 && cand < h.id)) {
        h.id = cand;
        h.t = (float)(t64 - (double)te0);
        h.e = 2e-7f * fabsf(h.t);
    }
}

// A candidate's root (or, open, a candidate that may have one from lo on) joins
// h. What FP64 has to decide waits, one candidate a lane, for the end of the walk:
// most are behind the hit by then, and the warp's lanes settle theirs together (an
// FP64 instruction occupies the SM's pipe as long for one lane as for 32).
// Settled at once instead: 0.213 and 0.057 ms.
__device__ __forceinline__ void near64_consider(const FrameDev& f, int i, int j, float te0, Near64& h, uint32_t cand,
                                                bool open, float t, float et, float lo) {
    if (!open) {
        if (t + et < h.t - h.e) {
            h.id = cand;
            h.t = t;
            h.e = et;
            return;
        }
        lo = t - et;
    }
    if (lo > h.t + h.e || cand == h.pend) return;
    if (h.pend == GBRT_MISS || h.lo > h.t + h.e) {
        h.pend = cand;
        h.lo = lo;
    } else {
        near64_settle(f, i, j, te0, h, cand);
    }
}

__device__ __forceinline__ void near64_finish(const FrameDev& f, int i, int j, float te0, Near64& h) {
    if (h.pend != GBRT_MISS && !(h.lo > h.t + h.e)) near64_settle(f, i, j, te0, h, h.pend);
    h.pend = GBRT_MISS;
}

template <bool SPLIT>
__device__ __forceinline__ void nearest_filtered64(const FrameDev& f, int i, int j, bool on, int sub, int parts,
                                                   Near64& h, bool& overflow) {
    if (!SPLIT && !on) return;
    const GridDev& g = f.grid;
    const float inf = Num<float>::inf();
    Ff3 o, d, x;
    primary_ray_ff(f, i, j, o, d);
    // start the walk short of the bounding sphere (its own clip is then exact
    // enough however far the camera is)
    const V3<float> c = o.hi - v3(g.bs[0], g.bs[1], g.bs[2]);
    const float te0 = fmaxf(0.0f, -dot(c, d.hi) * (1.0f - 1e-6f) - 1.1f * g.bs[3]);
    entry_point(o, d, te0, x);
    const V3<float> lo = v3(g.lo[0], g.lo[1], g.lo[2]);
    const V3<float> xr = (x.hi - lo) + x.lo;
    const V3<float> df = d.hi;
    Walk w;
    on = on && walk_start_rel(g, xr, df, 0.0f, inf, w);
    if (!SPLIT && !on) return;
    const float om = 0.1f * fmaxf(g.hi[0] - lo.x, fmaxf(g.hi[1] - lo.y, g.hi[2] - lo.z));
    const float idd = __fdividef(-1.0f, dot(df, df));
    auto visit = [&] {
        const uint2 cr = __ldg(g.cells + GBRT_INDEX(w.cell, g.ncells));
        for (uint32_t k = cr.x, e = cr.x + cr.y; k < e; ++k) {
            const uint32_t cand = GBRT_INDEX(__ldg(g.items + GBRT_INDEX(k, g.nitems)), f.scene.S + f.scene.C);
            if (cand == h.id) continue;
            const float4 s = __ldg(f.scene.bs + cand);
            const V3<float> wv = xr - v3(s.x - lo.x, s.y - lo.y, s.z - lo.z);
            const float tc = dot(wv, df) * idd;
            const V3<float> m = madd(wv, tc, df);
            const float r = fabsf(s.w), bp = fminf(tc, 0.0f), x2 = fmaf(-r, r, dot(m, m));
            const float mg = filter_margin(r, fabsf(tc) + r + om);
            if (!(fmaf(bp, bp, x2) <= mg)) continue;
            float t, et;
            int what;
            if (s.w > 0.0f) {
                what = sphere_root32(tc, x2, mg, r, om, t, et);
            } else {
                V3<float> p0, a;
                float L, rr;
                Obj<float>::load(f.scene.obj, cand, p0, a, L, rr);
                what = tube_root32(xr, df, p0 - lo, a, L, rr, inf, inf, om, t, et);
            }
            // (no root of what lies in the ball comes before the ball)
            const float front = tc - 1.001f * sqrt_pos(mg - x2) - 1e-5f * (fabsf(tc) + r + om);
            if (what != PAIR_MISS) near64_consider(f, i, j, te0, h, cand, what == PAIR_OPEN, t, et, front);
        }
    };
    auto next = [&] { return walk_next_rel(w, g, xr, df, overflow); };
    if (!SPLIT) {
        do {
            visit();
            if (h.id != GBRT_MISS && h.t + h.e <= walk_cell_exit(w)) break;
        } while (next());
        near64_finish(f, i, j, te0, h);
        return;
    }
    split_walk(w, on, sub, parts, h, next, visit, [&] { return h.t + h.e; });
    near64_finish(f, i, j, te0, h);
    // the lanes' hits, merged
    for (int x = 1; x < parts; x <<= 1) {
        const uint32_t k = __shfl_xor_sync(FULL, h.id, x);
        const float t = __shfl_xor_sync(FULL, h.t, x), e = __shfl_xor_sync(FULL, h.e, x);
        if (k != GBRT_MISS && k != h.id) near64_consider(f, i, j, te0, h, k, false, t, e, t);
        near64_finish(f, i, j, te0, h);
    }
}

// Hit records: (AO origin xyz, pixel) and (normal xyz, object id).
template <class R>
struct HitIO;

template <>
struct HitIO<float> {
    static __device__ __forceinline__ void store_f(void* hits, int64_t slot, V3<float> o, V3<float> n, uint32_t q,
                                                   uint32_t id) {
        float4* H = (float4*)hits + 2 * slot;
        H[0] = make_float4(o.x, o.y, o.z, __uint_as_float(q));
        H[1] = make_float4(n.x, n.y, n.z, __uint_as_float(id));
    }
    static __device__ __forceinline__ void load(const void* hits, int64_t slot, V3<float>& o, V3<float>& n,
                                                uint32_t& q, uint32_t& id) {
        const float4* H = (const float4*)hits + 2 * slot;
        float4 a = H[0], b = H[1];
        o = v3(a.x, a.y, a.z);
        q = __float_as_uint(a.w);
        n = v3(b.x, b.y, b.z);
        id = __float_as_uint(b.w);
    }
};

template <>
struct HitIO<double> {
    static __device__ __forceinline__ void store(void* hits, int64_t slot, V3<double> o, V3<double> n, uint32_t q,
                                                 uint32_t id) {
        double2* H = (double2*)hits + 4 * slot;
        H[0] = make_double2(o.x, o.y);
        H[1] = make_double2(o.z, __longlong_as_double((long long)q));
        H[2] = make_double2(n.x, n.y);
        H[3] = make_double2(n.z, __longlong_as_double((long long)id));
    }
    static __device__ __forceinline__ void load(const void* hits, int64_t slot, V3<double>& o, V3<double>& n,
                                                uint32_t& q, uint32_t& id) {
        const double2* H = (const double2*)hits + 4 * slot;
        double2 a = H[0], b = H[1], c = H[2], e = H[3];
        o = v3(a.x, a.y, b.x);
        q = (uint32_t)__double_as_longlong(b.y);
        n = v3(c.x, c.y, e.x);
        id = (uint32_t)__double_as_longlong(e.y);
    }
};

template <class R>
__device__ __forceinline__ R ao_maxdist(const FrameDev& f);
template <>
__device__ __forceinline__ float ao_maxdist<float>(const FrameDev& f) { return f.ao_maxdist_f; }
template <>
__device__ __forceinline__ double ao_maxdist<double>(const FrameDev& f) { return f.ao_maxdist; }

// ---------------------------------------------------------------- primary pass

// AO rays a warp claims from the global queue at once (its local pool): 64, and
// fewer, down to 8, where 64 would leave warps without any. A small frame's AO
// pass is one round of such claims, bound by the latency of one warp's rays:
// 41 -> 30 us at 256 x 256, 4 samples; 33 -> 21 us at 128 x 96 (64 at once
// against this; shares of a half or a quarter: 34 us at 256 x 256).
__device__ __forceinline__ unsigned ao_claim(unsigned long long rays, int warps) {
    const unsigned long long share = rays / (unsigned)warps + 1ull;
    return share >= 64ull ? 64u : share <= 8ull ? 8u : (unsigned)(share + 7ull) & ~7u;
}

// Prefix sums of hits and AO rays per frame; resets the AO and shading queues.
// Run by one thread of the primary pass's last CTA once every CTA's hits are
// counted (the counts are read through L2: other CTAs added them atomically).
__device__ __forceinline__ void ao_plan(const BatchDev& b) {
    unsigned long long jobs = 0, hits = 0;
    b.job_off[0] = 0;
    b.hit_off[0] = 0;
    for (int f = 0; f < b.nframes; ++f) {
        unsigned long long h = __ldcg(b.hit_count + f);
        hits += h;
        jobs += h * (unsigned long long)b.frames[f].jobs_per_hit;
        b.hit_off[f + 1] = hits;
        b.job_off[f + 1] = jobs;
    }
    b.queue[1] = 0;
    b.queue[2] = 0;
    b.queue[3] = ao_claim(jobs, b.ao_warps);
}

// SPLIT: b.parts lanes share a primary ray (ray_parts).
template <int MODE, bool SPLIT>
__global__ void __launch_bounds__(256) k_primary(const __grid_constant__ BatchDev b) {
    const int lane = threadIdx.x & 31;
    const int parts = SPLIT ? b.parts : 1, sub = lane & (parts - 1);
    const long long total = b.tile_off[b.nframes] * parts;
    bool overflow = false;
    while (true) {
        long long item = 0;
        if (lane == 0) item = (long long)atomicAdd(b.queue, 1ull);
        item = __shfl_sync(FULL, item, 0);
        if (item >= total) break;
        int px = lane;  // the lane's pixel of the tile
        if (SPLIT) {    // (an item is 32 / parts pixels)
            px = ((int)(item & (parts - 1)) * 32 + lane) / parts;
            item /= parts;
        }
        const int f = find_frame(b.tile_off, b.nframes, item);
        const FrameDev& F = b.frames[f];
        const long long t = item - b.tile_off[f];
        const int tx = (int)(t % F.tiles_x), ty = (int)(t / F.tiles_x);
        const int i = tx * b.tile_w + px % b.tile_w;
        const int j = F.row0 + ty * b.tile_h + px / b.tile_w;
        const bool inside = i < F.W && j < F.row0 + F.rows;
        const bool mine = inside && sub == 0;  // the lane that writes the pixel
        uint32_t id = GBRT_MISS;
        LocalHit lh;
        bool hit = false;
        if (MODE == GBRT_FP32) {
            float te0 = 0.0f;
            Nearest h;
            h.t1 = h.t2 = Num<float>::inf();
            h.id1 = h.id2 = GBRT_MISS;
            nearest_fp32<SPLIT>(F, i, j, inside, sub, parts, te0, h, overflow);
            hit = mine && h.id1 != GBRT_MISS;
            if (hit) refine_fp32(F, i, j, te0, h, id, lh);
        } else {
            Near64 h;
            h.id = h.pend = GBRT_MISS;
            h.t = Num<float>::inf();
            h.e = h.lo = 0.0f;
            nearest_filtered64<SPLIT>(F, i, j, inside, sub, parts, h, overflow);
            id = h.id;
            hit = mine && id != GBRT_MISS;
        }
        // warp-aggregated append to this frame's hit list
        const unsigned hm = __ballot_sync(FULL, hit);
        unsigned base = 0;
        if (hm) {
            const int leader = __ffs(hm) - 1;
            if (lane == leader) base = atomicAdd(b.hit_count + f, (unsigned)__popc(hm));
            base = __shfl_sync(FULL, base, leader);
        }
        if (b.tiles && hm && lane == 0) {  // (the near pass's frames are not split into parts)
            unsigned long long at =
                atomicAdd(b.ntiles, (unsigned long long)((F.mask_words + F.rec_words - 1) / F.rec_words));
            for (int w = 0; w < F.mask_words; w += F.rec_words, ++at) {
                TileRec& rec = b.tiles[GBRT_INDEX(at, b.tile_cap)];
                rec.slot = F.hit_base + (int64_t)base;
                rec.n = __popc(hm);
                rec.frame = f;
                rec.word = w;
            }
        }
        if (!mine) continue;
        const uint32_t q = (uint32_t)j * (uint32_t)F.W + (uint32_t)i;
        if (hit) {
            const int64_t slot = GBRT_INDEX(F.hit_base + base + __popc(hm & ((1u << lane) - 1u)), b.hit_cap);
            if (MODE == GBRT_FP32) {
                // the refined offset w from p0 splits into its foot on the
                // generator (centre or axis), p0 + (w.a) a, and w_p, the
                // radial part (length r at the refined root); the re-projected
                // surface point plus eps along the normal facing the ray is
                // p0 + (w.a) a + (r +- eps) w_p/|w_p|, formed in FP32 relative
                // to p0 and rounded once when p0 is added
                V3<float> p0, a;
                float L, r;
                Obj<float>::load(F.scene.obj, id, p0, a, L, r);
                const float wa = dot(lh.w, a);
                const V3<float> wp = madd(lh.w, -wa, a);
                const float inv = rsqrtf(dot(wp, wp));
                V3<float> nf = inv * wp;
                const bool flip = dot(view_dir_f(F, q), nf) > 0.0f;
                const V3<float> off = madd(wa * a, flip ? r - F.eps_f : r + F.eps_f, nf);
                const V3<float> ao_o = p0 + off;
                if (flip) nf = v3(-nf.x, -nf.y, -nf.z);
                HitIO<float>::store_f(b.hits, slot, ao_o, nf, q, id);
            } else {
                V3<double> o64, d64, p, n;
                double t64;
                primary_ray64(F, i, j, o64, d64);
                hit_object<double>(F.scene, id, o64, d64, 0.0, Num<double>::inf(), t64);
                reproject64(F.scene, id, o64, d64, t64, p, n);
                const V3<double> ao_o = madd(p, F.eps, n);
                HitIO<double>::store(b.hits, slot, ao_o, n, q, id);
                HitIO<float>::store_f(b.hits32, slot, to_f(ao_o - ld3(F.grid.lo64)), to_f(n), q, id);
            }
            b.vis[slot] = 0u;
            b.lmask[slot] = 0u;
            if (F.out_ids) F.out_ids[q] = id;
        } else {
            if (MODE == GBRT_FP32) {
                float* out = (float*)F.out_rgb + 3 * (size_t)(q - F.rgb_q0);
                out[0] = F.bg_f[0];
                out[1] = F.bg_f[1];
                out[2] = F.bg_f[2];
            } else {
                double* out = (double*)F.out_rgb + 3 * (size_t)(q - F.rgb_q0);
                out[0] = F.bg[0];
                out[1] = F.bg[1];
                out[2] = F.bg[2];
            }
            if (F.out_ids) F.out_ids[q] = GBRT_MISS;
            if (F.out_vis) F.out_vis[q] = 0u;
        }
    }
    if (overflow) atomicOr(b.err, ERR_DDA_STEPS);
    // the last CTA to finish lays out the AO pass (queue[3] counts finished
    // CTAs; it starts at zero with the batch's counters)
    __shared__ bool last_cta;
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        last_cta = atomicAdd(b.queue + 3, 1ull) == (unsigned long long)gridDim.x - 1ull;
    }
    __syncthreads();
    if (last_cta && threadIdx.x == 0) {
        __threadfence();
        ao_plan(b);
    }
}

// ---------------------------------------------------------------- AO pass

// One AO job -- AO sample or direct-light shadow ray -- of frame F: its index
// jl among the frame's jobs (hits x jobs per hit) names the hit slot whose
// count or light bit it settles and the sample.
__device__ __forceinline__ void ao_split(const FrameDev& F, unsigned long long jl, uint32_t& h, uint32_t& smp) {
    const uint32_t jph = (uint32_t)F.jobs_per_hit;
    if (jl >= 0xFFFFFFFFull) {
        h = (uint32_t)(jl / jph);
    } else if (jph > 1u) {
        // jl / jph by the multiplier ceil(2^32 / jph): the product's high word
        // is the quotient or one more
        h = __umulhi((uint32_t)jl, F.jph_magic);
        if ((unsigned long long)h * jph > jl) --h;
    } else {
        h = (uint32_t)jl;
    }
    smp = (uint32_t)(jl - (unsigned long long)h * jph);
}

// Direction of job smp of a hit with normal n and pixel q, and whether a ray
// is cast at all (a light behind the surface needs none: its bit stays clear).
// lbit: 0 for an AO sample, 1 << l for the shadow ray toward light l.
template <class R>
__device__ __forceinline__ bool ao_direction(const FrameDev& F, uint32_t q, uint32_t smp, V3<R> n, V3<R>& d, R& tmax,
                                             uint32_t& lbit, bool facing_slack = false) {
    if (smp < (uint32_t)F.spp) {
        uint32_t b1, b2;
        ao_uniforms(q, smp, F.frame, F.seed_lo, F.seed_hi, b1, b2);
        d = cosine_dir(n, b1, b2);
        tmax = ao_maxdist<R>(F);
        lbit = 0u;
        return true;
    }
    const int l = (int)(smp - (uint32_t)F.spp);
    d = ShadeP<R>::ldir(F, l);
    tmax = Num<R>::inf();
    lbit = 1u << l;
    // FP64 frames ask in FP32 (the AO walk): a light within rounding of the
    // horizon gets its ray, and shading decides in FP64 whether it counts
    return dot(n, d) > (facing_slack ? R(-1e-5) : R(0));
}

// A ray that leaves the objects' bounds unoccluded: one more escaped AO
// sample, or its light's bit.
__device__ __forceinline__ void ao_escape(const BatchDev& b, int64_t vslot, uint32_t lbit) {
    if (lbit) atomicOr(b.lmask + vslot, lbit);
    else atomicAdd(b.vis + vslot, 1u);
}

// ---- near pass

__device__ __forceinline__ float max3(float a, float b, float c) {
    float m;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(a), "f"(b), "f"(c));
    return m;
}
// floats as integers of the same order, for the warp's integer reductions
__device__ __forceinline__ int ord_i(float x) {
    const int i = __float_as_int(x);
    return i ^ ((i >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float warp_min(float x) {
    const int m = __reduce_min_sync(FULL, ord_i(x));
    return __int_as_float(m ^ ((m >> 31) & 0x7fffffff));
}
__device__ __forceinline__ float warp_max(float x) { return -warp_min(-x); }
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(FULL, x, o);
    return x;
}

// Candidates of a work item (balls); the directions of eight samples on their
// way into registers; during the gather, where each row's balls lie.
constexpr int NEAR_SPHERES = 160, NEAR_TUBES = 128;
struct NearWarp {
    float4 sph[NEAR_SPHERES], tub[NEAR_TUBES];
    union {
        float dir[8][3][32];
        struct {
            uint32_t off[32];    // ball of position p: p + off[row]
            uint32_t owner[32];  // row whose balls start at this position of the chunk
        } rows;
    };
};
// Largest number of jobs a hit may have for its frame to have a near pass
// (bounds the masks to 64 bytes a hit).
constexpr int NEAR_MAX_JOBS = 256;
constexpr int NEAR_MIN_JOBS = 8;
// The pass pays where what it saves (near_work) is above these: its launch, the
// latency of its records (some 40 us a warp) and the walk's coarser units cost a
// frame the same however little that is. FP64 rays walk slower, and one a lane.
constexpr double NEAR_MIN_WORK = 28500, NEAR_MIN_WORK64 = 16000;
// With fewer records than this a tile's job words, which share its gather, are
// dealt to several records.
constexpr double NEAR_FULL_RECS = 12288;

// Largest b - q over the n candidates at c, for each of the NS directions: b =
// w.d with w = centre - o, q = sqrt(|w|^2 - r^2). The ray meets a ball ahead of
// an outside origin exactly when b >= q. w and q are per (hit, ball), so a
// (ray, ball) pair costs three FMAs and half a three-input maximum. An origin
// inside or within 5e-5 r of a ball sets bad (q would be too rough there),
// unless it is the ball of the object that the hit lies on (skip): rays from the
// outer side of a sphere or a tube do not meet it again. An FP64 origin is o + ol
// (float pairs: w then has FP32's relative error however large the coordinates).
//
// The object is known by its ball. A ball with the same centre and radius may
// still be another object's (the arms of a cross, a tube drawn twice), but the
// gather takes equal balls together or not at all: of several such candidates
// one is passed over and the next sets bad.
struct NearSkip {
    int kind;  // 0: a sphere, 1: a tube, -1: nothing is passed over
    V3<float> c;
    float r;
};
__device__ __forceinline__ float near_q(float4 A, float q2, const NearSkip& skip, bool& left, bool& bad) {
    if (q2 < 1e-4f * A.w * A.w) {
        if (left && A.x == skip.c.x && A.y == skip.c.y && A.z == skip.c.z && A.w == skip.r) {
            left = false;
            return Num<float>::inf();
        }
        bad = true;
    }
    return sqrt_pos(q2);
}
template <int NS, bool F64>
__device__ __forceinline__ void near_scan(const float4* c, int n, V3<float> o, V3<float> ol, const float (&d)[NS][3],
                                          float (&m)[NS], const NearSkip& skip, bool left, bool& bad) {
#pragma unroll 1
    for (int k = 0; k < n; k += 2) {
        const float4 A = c[k], B = c[k + 1 < n ? k + 1 : k];
        float ax = A.x - o.x, ay = A.y - o.y, az = A.z - o.z;
        float bx = B.x - o.x, by = B.y - o.y, bz = B.z - o.z;
        if (F64) {
            ax -= ol.x, ay -= ol.y, az -= ol.z;
            bx -= ol.x, by -= ol.y, bz -= ol.z;
        }
        const float qa = fmaf(ax, ax, fmaf(ay, ay, fmaf(az, az, -A.w * A.w)));
        const float qb = fmaf(bx, bx, fmaf(by, by, fmaf(bz, bz, -B.w * B.w)));
        const float na = -near_q(A, qa, skip, left, bad);
        const bool more = k + 1 < n;  // else B is A again, not one more candidate (an own tube there only walks)
        bool twin = false;
        const float nb = -near_q(B, qb, skip, left, twin);
        bad |= twin && more;
#pragma unroll
        for (int s = 0; s < NS; ++s)
            m[s] = max3(m[s], fmaf(ax, d[s][0], fmaf(ay, d[s][1], fmaf(az, d[s][2], na))),
                        fmaf(bx, d[s][0], fmaf(by, d[s][1], fmaf(bz, d[s][2], nb))));
    }
}

// Directions of cnt <= 8 jobs from j0 on, one hit a lane; which of them are rays.
// Not unrolled, like the scan's loop: the kernel was short of instruction cache
// (0.35 -> 0.31 ms at 965 x 1137; the figure with two lights, 16 + 2 jobs a hit,
// which goes from one width of near_jobs to the other, 1.62 -> 1.16 ms).
template <bool F64>
__device__ __forceinline__ uint32_t near_dirs(const FrameDev& F, NearWarp& S, int lane, int j0, int cnt, V3<float> nrm,
                                           uint32_t q) {
    uint32_t valid = 0u;
#pragma unroll 1
    for (int s = 0; s < cnt; ++s) {
        V3<float> dir = nrm;
        if (j0 + s < F.jobs_per_hit) {
            float tmax;
            uint32_t lbit;
            if (ao_direction<float>(F, q, (uint32_t)(j0 + s), nrm, dir, tmax, lbit, F64)) valid |= 1u << s;
        }
        S.dir[s][0][lane] = dir.x;
        S.dir[s][1][lane] = dir.y;
        S.dir[s][2][lane] = dir.z;
    }
    return valid;
}

// NS jobs (from j0) of a work item's hits, one hit a lane: which are occluded
// by a near sphere, which have to walk, which of those from the start, which
// leave the objects' bounds before the near pass's reach.
template <int NS, bool F64>
__device__ __forceinline__ void near_jobs(const FrameDev& F, NearWarp& S, int lane, int j0, V3<float> o, V3<float> ol,
                                          V3<float> nrm, uint32_t q, const NearSkip& skip, int ns, int nt, float rho,
                                          float delta, uint32_t& todo, uint32_t& start, uint32_t& escaped) {
    float d[NS][3], m[NS];
    uint32_t valid = 0u;
    constexpr int W = NS < 8 ? NS : 8;
    static_assert(NS <= 2 * W, "two calls fill the directions");
    // (two calls, not a loop: in a loop that it did not unroll, nvcc 13.0 lost the
    // first eight directions)
    auto fill = [&](auto at) {
        constexpr int h = decltype(at)::value;
        valid |= near_dirs<F64>(F, S, lane, j0 + h, W, nrm, q) << h;
#pragma unroll
        for (int s = 0; s < W; ++s)
#pragma unroll
            for (int k = 0; k < 3; ++k) d[h + s][k] = S.dir[s][k][lane];
    };
    fill(std::integral_constant<int, 0>());
    if constexpr (NS > W) fill(std::integral_constant<int, W>());
    // spheres, then tubes, through the same code (it has to stay in the
    // instruction cache): what a sphere's ball surely stops is hit, what comes
    // close to one or meets a tube's stays open
    bool bad = false;
    uint32_t hit = 0u, open = 0u;
    const float4* list = S.sph;
    int n = ns;
#pragma unroll 1
    for (int kind = 0; kind < 2; ++kind) {
#pragma unroll
        for (int s = 0; s < NS; ++s) m[s] = -Num<float>::inf();
        near_scan<NS, F64>(list, n, o, ol, d, m, skip, skip.kind == kind, bad);
        const float sure = kind == 0 ? delta : Num<float>::inf();
#pragma unroll
        for (int s = 0; s < NS; ++s) {
            hit |= m[s] > sure ? 1u << s : 0u;
            open |= m[s] >= -delta ? 1u << s : 0u;
        }
        list = S.tub;
        n = nt;
    }
    const V3<float> f = v3(o.x - F.grid.bs[0], o.y - F.grid.bs[1], o.z - F.grid.bs[2]);
    const float ff = dot(f, f) - F.grid.bs[3] * F.grid.bs[3];
    escaped = 0u;
#pragma unroll
    for (int s = 0; s < NS; ++s) {
        // f.f + 2 t f.d + t^2 - r^2 > 0 at t = reach, from inside: the ray left
        const float fd = f.x * d[s][0] + f.y * d[s][1] + f.z * d[s][2];
        escaped |= fmaf(rho, fmaf(2.0f, fd, rho), ff) > 0.0f ? 1u << s : 0u;
    }
    todo = valid & ~hit;
    start = todo & open;
    if (bad) todo = start = valid;
    escaped = ff < 0.0f ? escaped & todo & ~start : 0u;
    todo &= ~escaped;
}

// The near pass of an AO batch, one warp per tile (the <= 32 hits of a primary
// work item, one a lane). The hits of a tile lie close together, so their
// rays share the objects that they can meet within rho of the hits: the warp
// gathers those balls once, from the objects sorted by cell, drops the ones
// behind all of the hits, and tests every ray of the tile against every ball
// in registers (near_scan) instead of walking each ray through its first
// cells. Rays a sphere surely stops are done; the others go on to the walk, at
// distance rho. A ray too close to a silhouette to tell (delta), or that meets
// a tube's ball, walks from its start: tubes are cut to what sticks out of
// their atoms, so that is one ray in a hundred. The decisions are those of the
// walk's own test (delta is ten times the rounding of both).
// Measured (965 x 1137, 16 samples, 9.0 M AO rays): 140 balls a tile; 37% of the
// rays hit, 13% left the bounds, 1% open; 258 M warp instructions (some 40 M of the
// gather, 50 M of the directions, 160 M of the scan) in 0.31 ms, and the walk
// 1.00 -> 0.45 ms. 3860 x 4548: frame 15.8 -> 10.2 ms. Instruction issue (16 warps an SM, for the
// directions in registers) and the instruction cache bound it. Tried: the scan as f16-pair
// m16n8k16 mma.sync (13.7 cycles a 128 pairs, no faster than the FMAs), packed
// f32x2 FMAs (20% fewer instructions, 10% slower), a row of cells per lane in
// the gather (55 dependent rounds of loads instead of 16: 0.44 ms).
// F64: the same for FP64 frames, whose decisions delta covers as well (the
// directions are the FP32 ones the walk filters with, the origins float pairs):
// 0.33 ms, and the walk 1.53 -> 0.80 (965 x 1137, frame 1.87 -> 1.46 ms).
template <bool F64>
__global__ void __launch_bounds__(128, 4) k_ao_near(const __grid_constant__ BatchDev b) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    NearWarp& S = reinterpret_cast<NearWarp*>(smem_raw)[threadIdx.x >> 5];
    grid_dependency_wait();
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const unsigned long long total = *b.ntiles;
    while (true) {
        unsigned long long tile = 0;
        if (lane == 0) tile = atomicAdd(b.queue + 2, 1ull);
        tile = __shfl_sync(FULL, tile, 0);
        if (tile >= total) break;
        TileRec& rec = b.tiles[GBRT_INDEX(tile, b.tile_cap)];
        const int n = rec.n;
        const FrameDev& F = b.frames[GBRT_INDEX(rec.frame, b.nframes)];
        const int64_t slot = GBRT_INDEX(rec.slot + (lane < n ? lane : 0), b.hit_cap);
        V3<float> o, nrm, ol = v3(0.0f, 0.0f, 0.0f);
        uint32_t q, own;
        HitIO<float>::load(b.hits32, slot, o, nrm, q, own);
        if (F64) {  // hits32 holds the origin relative to the grid's corner
            V3<double> o64, n64;
            HitIO<double>::load(b.hits, slot, o64, n64, q, own);
            o = to_f(o64);
            ol = to_f(o64 - to_d(o));
        }
        float rho = F.near_pass ? F.grid.rho : 0.0f, delta = 0.0f;
        int ns = 0, nt = 0;
        NearSkip skip;
        skip.kind = -1;
        skip.r = 0.0f;
        if (rho > 0.0f) {
            // The hit's own ball, passed over where the object surely lies behind
            // the plane through the origin that the rays start from: a tube's
            // ball may hold the origin, and with a small eps it is closer to a
            // sphere than bad allows (1e-6 r keeps clear of the rounding here and
            // in the walk's own test). Outside alone is not enough: far from the
            // coordinates' zero an origin is rounded by more than eps, one on the
            // inner wall of an open tube to the outside or one on a thin object
            // aside of its normal, and its rays do meet the object.
            V3<float> p0, a;
            float L, r;
            own = GBRT_INDEX(own, F.scene.S + F.scene.C);
            Obj<float>::load(F.scene.obj, own, p0, a, L, r);
            const float4 c = __ldg(F.grid.cut + own);
            const V3<float> w = (o - p0) + ol, v = (o - v3(c.x, c.y, c.z)) + ol;
            const V3<float> wp = madd(w, -dot(w, a), a);  // (a sphere's axis is 0)
            skip.c = v3(c.x, c.y, c.z);
            skip.r = fabsf(c.w);
            if (c.w != 0.0f && dot(wp, nrm) > (L > 0.0f ? 1.0001f : 1.000001f) * r) skip.kind = L > 0.0f ? 1 : 0;
            // where the own ball keeps most of the hits from being looked at (an
            // eps of next to nothing, a view from inside) the pass is left out
            const bool kept = skip.kind < 0 && dot(v, v) - c.w * c.w < 1e-4f * c.w * c.w;
            if (2 * __popc(__ballot_sync(FULL, lane < n && kept)) > n) rho = 0.0f;
        }
        if (rho > 0.0f) {
            // the hits' box, its centre, and the cone of their normals
            const V3<float> mn = v3(warp_min(o.x), warp_min(o.y), warp_min(o.z));
            const V3<float> mx = v3(warp_max(o.x), warp_max(o.y), warp_max(o.z));
            const V3<float> ctr = 0.5f * (mn + mx), ext = 0.5f * (mx - mn);
            const float spread = sqrtf(dot(ext, ext));
            V3<float> ax = v3(warp_sum(nrm.x), warp_sum(nrm.y), warp_sum(nrm.z));
            ax = rsqrtf(fmaxf(dot(ax, ax), 1e-20f)) * ax;
            const float ca = warp_min(dot(ax, nrm)), sa = sqrtf(fmaxf(0.0f, 1.0f - ca * ca));
            const float rmax = F.grid.rmax * 1.001f;
            delta = 2.5e-4f * F.grid.rmax + 4e-6f * (rho + 2.0f * spread);
            // look less far, or not at all, where the hits' box with that
            // reach around it would hold more balls than pay (a pass of a
            // job word costs 70 instructions a ball, a walk about 95 a ray)
            const float most = 8.0f * (float)min(F.jobs_per_hit, 16);
            for (int t = 0;; ++t) {
                const float v = (ext.x + rho) * (ext.y + rho) * (ext.z + rho);
                if (8.0f * v * F.grid.density <= most) break;
                rho *= 0.75f;
                if (t == 2) {
                    rho = 0.0f;
                    break;
                }
            }
            for (int t = 0; t < 2 && rho > 0.0f; ++t) {
                ns = nt = 0;
                const float R = rho + rmax;
                int c0[3], c1[3];
                const float l[3] = {mn.x - R, mn.y - R, mn.z - R}, h[3] = {mx.x + R, mx.y + R, mx.z + R};
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    c0[k] = cell_of(F.grid, k, l[k]) >> 1;
                    c1[k] = cell_of(F.grid, k, h[k]) >> 1;
                }
                const int ny = c1[1] - c0[1] + 1, rows = ny * (c1[2] - c0[2] + 1);
                for (int r0 = 0; r0 < rows; r0 += 32) {
                    // one row of cells a lane: a run of balls; the runs are
                    // laid end to end and read 32 balls at a time
                    uint32_t k = 0, cnt = 0;
                    if (r0 + lane < rows) {
                        const int y = c0[1] + (r0 + lane) % ny, z = c0[2] + (r0 + lane) / ny;
                        const int64_t row = ((int64_t)z * F.grid.bn[1] + y) * F.grid.bn[0];
                        [[maybe_unused]] const int64_t starts = (int64_t)F.grid.bn[0] * F.grid.bn[1] * F.grid.bn[2] + 1;
                        k = __ldg(F.grid.bstart + GBRT_INDEX(row + c0[0], starts));
                        cnt = __ldg(F.grid.bstart + GBRT_INDEX(row + c1[0] + 1, starts)) - k;
                    }
                    uint32_t incl = cnt;
#pragma unroll
                    for (int off = 1; off < 32; off <<= 1) {
                        const uint32_t y = __shfl_up_sync(FULL, incl, off);
                        if (lane >= off) incl += y;
                    }
                    const uint32_t T = __shfl_sync(FULL, incl, 31), ex = incl - cnt;
                    S.rows.off[lane] = k - ex;
                    for (uint32_t base = 0; base < T; base += 32) {
                        const uint32_t u = ex > base ? ex : base, pos = u - base;
                        const bool mine = pos < 32u && incl > u;
                        __syncwarp();
                        if (mine) S.rows.owner[pos] = (uint32_t)lane;
                        const unsigned starts = __reduce_or_sync(FULL, mine ? 1u << pos : 0u);
                        __syncwarp();
                        const uint32_t p = base + lane;
                        bool sph = false, tub = false;
                        float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                        if (p < T) {
                            const unsigned r = S.rows.owner[31 - __clz(starts & (0xFFFFFFFFu >> (31 - lane)))];
                            s = __ldg(F.grid.balls + GBRT_INDEX(p + S.rows.off[r], (uint32_t)F.grid.nballs));
                            const float rad = fabsf(s.w);
                            const V3<float> v = v3(s.x, s.y, s.z) - ctr;
                            const float ex2 = fmaxf(fabsf(v.x) - ext.x, 0.0f), ey2 = fmaxf(fabsf(v.y) - ext.y, 0.0f),
                                        ez2 = fmaxf(fabsf(v.z) - ext.z, 0.0f), far = 1.001f * (rho + rad);
                            // behind every hit's tangent plane: the normals
                            // lie within the cone (ca) about ax
                            const float along = dot(v, ax), off = sqrt_pos(dot(v, v) - along * along);
                            const bool in = ex2 * ex2 + ey2 * ey2 + ez2 * ez2 <= far * far && s.w != 0.0f &&
                                            !(ca > 0.0f && along * ca + off * sa + spread <
                                                               -1.001f * rad - 1e-5f * (fabsf(along) + off));
                            sph = in && s.w > 0.0f;
                            tub = in && s.w < 0.0f;
                        }
                        const unsigned ms = __ballot_sync(FULL, sph), mt = __ballot_sync(FULL, tub);
                        const int is = ns + __popc(ms & lt), it = nt + __popc(mt & lt);
                        if (sph && is < NEAR_SPHERES) S.sph[is] = s;
                        if (tub && it < NEAR_TUBES) S.tub[it] = make_float4(s.x, s.y, s.z, -s.w);
                        ns += __popc(ms);
                        nt += __popc(mt);
                    }
                    __syncwarp();
                }
                if (ns <= NEAR_SPHERES && nt <= NEAR_TUBES) break;
                rho = t == 0 ? 0.6f * rho : 0.0f;  // the lists overflowed
            }
            __syncwarp();
        }
        if (lane == 0) rec.rho = rho;
        const int w0 = rec.word, w1 = min(w0 + F.rec_words, F.mask_words);
        for (int w = w0; w < w1; ++w) {
            const int j0 = 16 * w, cnt = F.jobs_per_hit - j0 < 16 ? F.jobs_per_hit - j0 : 16;
            uint32_t todo, start, esc = 0u;
            if (rho > 0.0f) {
                if (cnt > 8) {
                    near_jobs<16, F64>(F, S, lane, j0, o, ol, nrm, q, skip, ns, nt, rho, delta, todo, start, esc);
                } else {
                    todo = start = 0u;
                    for (int k = 0; k < cnt; k += 4) {
                        uint32_t t4, s4, e4;
                        near_jobs<4, F64>(F, S, lane, j0 + k, o, ol, nrm, q, skip, ns, nt, rho, delta, t4, s4, e4);
                        todo |= t4 << k;
                        start |= s4 << k;
                        esc |= e4 << k;
                    }
                }
            } else {
                todo = start = (1u << cnt) - 1u;
            }
            if (lane >= n) todo = start = esc = 0u;
            // escaped jobs: AO samples come first, then the lights
            const int sp = F.spp - j0 > 0 ? (F.spp - j0 < 16 ? F.spp - j0 : 16) : 0;
            const uint32_t vis = __popc(esc & ((1u << sp) - 1u));
            if (vis) atomicAdd(b.vis + slot, vis);
            if (esc >> sp) atomicOr(b.lmask + slot, (esc >> sp) << (j0 + sp - F.spp));
            if (lane < n) {
                const int64_t mask = F.mask_base + (slot - F.hit_base) * F.mask_words + w;
                b.masks[GBRT_INDEX(mask, b.mask_cap)] = todo | start << 16;
            }
            const uint32_t any = __reduce_or_sync(FULL, todo);
            const uint32_t groups = ((any & 0xFu) != 0u) | ((any & 0xF0u) != 0u) << 1 | ((any & 0xF00u) != 0u) << 2 |
                                    ((any & 0xF000u) != 0u) << 3;
            if (groups && lane == 0) {
                unsigned long long at = atomicAdd(b.nunits, (unsigned long long)__popc(groups));
                for (int g = 0; g < 4; ++g)
                    if ((groups >> g) & 1u) {
                        b.units[GBRT_INDEX(at, b.unit_cap)] = tile << 8 | (unsigned)(4 * w + g);
                        ++at;
                    }
            }
        }
        __syncwarp();
    }
}

// ---- FP32 frames

// Ray record in shared memory: (origin, tmax) and (direction, -) -- two
// 128-bit loads per test.
struct __align__(16) AoRay {
    V3<float> o;
    float tmax;
    V3<float> d;
    float pad;
};

// Per-warp shared state of the cooperative AO walk.
//   ray[lane]      the lane's ray (origin, tmax, direction)
//   sd             where each ray's pairs of the current iteration find their
//                  items (one range per cell taken)
//   owner          the ray whose pairs start at a position of the current chunk
//   obj, items     the ray's scene records and grid item list (batches mix
//                  scenes)
//   fifo[lane]     cells the ray has stepped to and loaded but not yet taken
// cells each active ray takes per lockstep iteration: further cells while it
// holds fewer than AO_MIN_PAIRS candidates, at most AO_CELLS
constexpr int AO_CELLS = 4;
// Pairs are tested where they were mapped, one per lane, with no mailbox of
// tested ids: a re-test of a missed object misses again, and the hit's own
// object cannot be met behind a convex outer side, so testing either is exact.
constexpr unsigned AO_MIN_PAIRS = 8;  // 6: 0.5% slower, 12: 1.5% slower

// per ray: its scene records and grid item list, when a batch mixes scenes
// (UNI: every frame of the batch has the same scene and grid -- the pointers
// are then kernel-wide)
template <bool UNI>
struct AoPtrs {
    const float4* obj[32];
    const uint32_t* items[32];
#ifdef GBRT_CHECKED
    int64_t nitems[32];  // the lengths the checked build tests indices against
    int64_t nobj[32];
#endif
};
template <>
struct AoPtrs<true> {};

// 4 KB a warp at most: four resident CTAs of 8 warps fit the
// 132 KB shared-memory configuration, leaving 124 KB of the SM's 256 KB to the
// L1 that caches the walk's cell, item and object loads. Measured: 5.25 KB a
// warp (60 KB of L1) 2.5% slower, 5 KB (92 KB of L1, with an 8-slot mailbox
// and a test queue) 1% slower.
static_assert(AO_CELLS == 4, "the pair segments of a ray are kept as one uint4 of starts and one of offsets");
// The unit of the near pass that a warp is taking rays from: 4 jobs of a work
// item's hits. b[s], z[s]: hits whose job s has to walk, has to walk from its
// start; used, rem: rays taken and left.
struct AoUnit {
    uint32_t b[4], z[4];
    int64_t slot;
    const FrameDev* F;
    int job;
    float tmin;
    uint32_t used, rem;
};
template <bool NEAR>
struct AoUnits {
    AoUnit unit;
};
template <>
struct AoUnits<false> {};

// Position of the n-th (from 0) set bit of m.
__device__ __forceinline__ int nth_bit(uint32_t m, unsigned n) {
    int at = 0;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) {
        const unsigned c = __popc((m >> at) & ((1u << w) - 1u));
        const bool up = n >= c;
        n -= up ? c : 0u;
        at += up ? w : 0;
    }
    return at;
}

// Hands `need` rays of the near pass's units to the idle lanes (free; i: a
// lane's rank among them): the hit slot, job, frame and start of each. The
// warp's unit is kept in U; sets exhausted when no unit is left.
__device__ __forceinline__ void unit_take(const BatchDev& b, AoUnit& U, int lane, unsigned long long total,
                                          unsigned need, unsigned i, bool free, bool& exhausted, int64_t& vslot,
                                          uint32_t& smp, float& tmin, const FrameDev*& Fp) {
    for (unsigned done = 0; done < need;) {
        unsigned rem = U.rem;
        if (rem == 0u) {
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd(b.queue + 1, 1ull);
            at = __shfl_sync(FULL, at, 0);
            if (at >= total) {
                exhausted = true;
                break;
            }
            const unsigned long long unit = b.units[GBRT_INDEX(at, b.unit_cap)];
            const int g = (int)(unit & 0xFFu), sh = 4 * (g & 3);
            const TileRec T = b.tiles[GBRT_INDEX(unit >> 8, b.tile_cap)];
            const FrameDev& N = b.frames[GBRT_INDEX(T.frame, b.nframes)];
            uint32_t m = 0u;
            if (lane < T.n) {
                const int64_t mask = N.mask_base + (T.slot - N.hit_base + lane) * N.mask_words + (g >> 2);
                m = b.masks[GBRT_INDEX(mask, b.mask_cap)] >> sh;
            }
            __syncwarp();
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const unsigned todo = __ballot_sync(FULL, (m >> s) & 1u);
                const unsigned start = __ballot_sync(FULL, (m >> (16 + s)) & 1u);
                U.b[s] = todo;
                U.z[s] = start;
                rem += __popc(todo);
            }
            U.slot = T.slot;
            U.F = &N;
            U.job = 4 * g;
            U.tmin = T.rho * (1.0f - 1e-4f);
            U.used = 0u;
            __syncwarp();
        }
        const unsigned take = rem < need - done ? rem : need - done;
        if (free && i >= done && i < done + take) {
            unsigned k = U.used + (i - done);
            int s = 0;
#pragma unroll
            for (int t = 0; t < 3; ++t) {
                const unsigned c = __popc(U.b[t]);
                const bool up = s == t && k >= c;
                k -= up ? c : 0u;
                s += up ? 1 : 0;
            }
            const int hit = nth_bit(U.b[s], k);
            vslot = GBRT_INDEX(U.slot + hit, b.hit_cap);
            smp = (uint32_t)(U.job + s);
            tmin = (U.z[s] >> hit) & 1u ? 0.0f : U.tmin;
            Fp = U.F;
        }
        __syncwarp();
        if (lane == 0) {
            U.used += take;
            U.rem = rem - take;
        }
        __syncwarp();
        done += take;
    }
}

template <bool UNI, bool NEAR>
struct AoWarp : AoPtrs<UNI>, AoUnits<NEAR> {
    AoRay ray[32];
    // item index of pair p of ray r: p + sdo[r][g] for the last cell g whose
    // pairs start at or before p (sds[r][g])
    uint4 sds[32];
    uint4 sdo[32];
    uint32_t owner[32];  // ray whose pairs start at this position of the current chunk
    // cells a ray has loaded but not yet taken, oldest first: an iteration takes
    // at least one of its at most AO_CELLS cells, so AO_CELLS - 1 wait at most
    uint2 fifo[32][AO_CELLS - 1];
};
static_assert(sizeof(AoWarp<false, true>) <= 4096, "the FP32 AO walk's per-warp state outgrew its 4 KB");

template <bool UNI, bool NEAR>
__device__ __forceinline__ const float4* ao_obj(const AoWarp<UNI, NEAR>& S, unsigned r, const float4* uni) {
    if constexpr (UNI) return uni;
    else return S.obj[r];
}
template <bool UNI, bool NEAR>
__device__ __forceinline__ const uint32_t* ao_items(const AoWarp<UNI, NEAR>& S, unsigned r, const uint32_t* uni) {
    if constexpr (UNI) return uni;
    else return S.items[r];
}
#ifdef GBRT_CHECKED
// ray r's item-buffer length and object count (the checked build's bounds)
template <bool UNI, bool NEAR>
__device__ __forceinline__ int64_t ao_nitems(const AoWarp<UNI, NEAR>& S, unsigned r, int64_t uni) {
    if constexpr (UNI) return uni;
    else return S.nitems[r];
}
template <bool UNI, bool NEAR>
__device__ __forceinline__ int64_t ao_nobj(const AoWarp<UNI, NEAR>& S, unsigned r, int64_t uni) {
    if constexpr (UNI) return uni;
    else return S.nobj[r];
}
#define GBRT_AO_ITEM(idx, r) GBRT_INDEX(idx, ao_nitems(S, r, unitems))
#define GBRT_AO_OBJ(id, r) GBRT_INDEX(id, ao_nobj(S, r, unobj))
#else
#define GBRT_AO_ITEM(idx, r) (idx)
#define GBRT_AO_OBJ(id, r) (id)
#endif

// Lockstep cooperative walk: every iteration each active ray takes its next
// one to AO_CELLS cells (all lanes run the same step code); the warp lays the
// (ray, item) pairs of those cells out densely with a scan and tests them 32
// at a time, one pair per lane. UNI: every frame of the batch has the same scene and grid.
// NEAR: the rays are those the near pass left, from its units.
template <bool UNI, bool NEAR>
__global__ void __launch_bounds__(256) k_ao_walk(const __grid_constant__ BatchDev b) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    AoWarp<UNI, NEAR>& S = reinterpret_cast<AoWarp<UNI, NEAR>*>(smem_raw)[threadIdx.x >> 5];
    grid_dependency_wait();
    if constexpr (NEAR) {
        S.unit.rem = 0u;
        __syncwarp();
    }
    const float4* uobj = nullptr;
    const uint32_t* uitems = nullptr;
    const uint2* ucells = nullptr;
    if constexpr (UNI) {
        uobj = b.frames[0].scene.obj;
        uitems = b.frames[0].grid.items;
        ucells = b.frames[0].grid.cells;
    }
#ifdef GBRT_CHECKED
    const int64_t unitems = b.frames[0].grid.nitems;
    const int64_t unobj = (int64_t)b.frames[0].scene.S + b.frames[0].scene.C;
#endif
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    const unsigned long long total = NEAR ? *b.nunits : b.job_off[b.nframes];
    const int refill = b.refill;
    bool has = false, exhausted = false, overflow = false;
    Walk w;
    unsigned nf = 0;      // cells waiting in this lane's fifo
    bool wend = false;    // the walk has no further cells
    uint32_t lbit = 0;  // 0: an AO sample; 1 << l: the shadow ray toward light l
    int64_t vslot = 0;
    const uint2* cells = nullptr;
    // the warp's pool of claimed rays [pool, pool_end) (warp-uniform)
    unsigned long long pool = 0, pool_end = 0;
    while (true) {
        // 1. compaction of rays: idle lanes take the next rays together, from
        //    the warp's pool, which claims ao_claim more rays from the global
        //    queue when it runs short
        const unsigned act = __ballot_sync(FULL, has);
        if (!exhausted && __popc(act) < refill) {
            const unsigned idle = ~act;
            const unsigned need = __popc(idle);
            // sets the lane up on job smp of hit vslot, from distance tmin on
            auto set_up = [&](const FrameDev& F, uint32_t smp, float tmin) {
                uint32_t q, own;
                V3<float> o, n, d;
                float tmax;
                HitIO<float>::load(b.hits32, vslot, o, n, q, own);
                if (!ao_direction<float>(F, q, smp, n, d, tmax, lbit)) {
                    // the light cannot reach this side: its bit stays clear
                } else if (walk_start(F.grid, o, d, tmin, tmax, w)) {
                    if constexpr (UNI) {
                        cells = ucells;
                    } else {
                        cells = F.grid.cells;
                        S.obj[lane] = F.scene.obj;
                        S.items[lane] = F.grid.items;
#ifdef GBRT_CHECKED
                        S.nitems[lane] = F.grid.nitems;
                        S.nobj[lane] = (int64_t)F.scene.S + F.scene.C;
#endif
                    }
                    AoRay ray;
                    ray.o = o;
                    ray.tmax = tmax;
                    ray.d = d;
                    ray.pad = 0.0f;
                    S.ray[lane] = ray;
                    // the walk stands on its first cell: its record waits in
                    // the fifo, so every later cell comes from a step
                    S.fifo[lane][0] = __ldg(cells + GBRT_INDEX(w.cell, w.ncells));
                    nf = 1;
                    wend = false;
                    has = true;
                } else {
                    ao_escape(b, vslot, lbit);  // misses the objects' bounds: escapes
                }
            };
            if constexpr (NEAR) {
                const FrameDev* Fp = nullptr;  // the frame of the ray this lane takes
                uint32_t smp = 0;
                float tmin = 0.0f;
                unit_take(b, S.unit, lane, total, need, __popc(idle & lt), !has, exhausted, vslot, smp, tmin, Fp);
                if (Fp) set_up(*Fp, smp, tmin);
            } else {
                const unsigned long long rem = pool_end - pool;
                unsigned long long fresh_base = 0;
                unsigned claim = 0;
                if (rem < need) {
                    claim = (unsigned)b.queue[3];
                    if (lane == 0) fresh_base = atomicAdd(b.queue + 1, (unsigned long long)claim);
                    fresh_base = __shfl_sync(FULL, fresh_base, 0);
                    if (fresh_base >= total) exhausted = true;
                }
                const unsigned n = rem + claim < need ? (unsigned)rem + claim : need;
                const unsigned i = __popc(idle & lt);
                if (!has && i < n) {
                    const unsigned long long jj = i < rem ? pool + i : fresh_base + (i - rem);
                    if (jj < total) {
                        const int f = b.nframes == 1 ? 0 : find_frame(b.job_off, b.nframes, jj);
                        const FrameDev& F = b.frames[f];
                        uint32_t h, smp;
                        ao_split(F, jj - b.job_off[f], h, smp);
                        vslot = GBRT_INDEX(F.hit_base + (int64_t)h, b.hit_cap);
                        set_up(F, smp, 0.0f);
                    }
                }
                if (rem >= need) {
                    pool += need;
                } else {
                    pool = fresh_base + (n - rem);
                    pool_end = fresh_base + claim;
                }
            }
        }
        if (exhausted && __ballot_sync(FULL, has) == 0) break;
        // 2. every active ray takes its next cells: its first, and further ones
        //    while it holds fewer than min_pairs candidates (an any-hit
        //    query may test objects past its first hit, so taking several at
        //    once is exact). The ray's fifo is first topped up to AO_CELLS
        //    loaded cells -- the new cells' loads are independent and overlap
        //    -- and the cells it does not take wait there for the next iteration
        // the walk's bound, counted per iteration rather than per step (every
        // iteration takes at least one cell or ends the ray, so a walk of the
        // grid's nx + ny + nz + 1 cells never reaches it; one whose crossing
        // times are not numbers ends here)
        if (has && --w.left <= 0) {
            overflow = true;
            wend = true;
            nf = 0;
        }
        bool ending = false;
        unsigned kg[AO_CELLS], ng[AO_CELLS];
        unsigned avail = 0u;
#pragma unroll
        for (int g = 0; g < AO_CELLS; ++g) {
            uint2 cr = make_uint2(0u, 0u);
            const bool queued = has && g < AO_CELLS - 1 && (unsigned)g < nf;
            if (queued) cr = S.fifo[lane][g];
            if (has && !queued && !wend) {
                if (walk_step(w)) cr = __ldg(cells + GBRT_INDEX(w.cell, w.ncells));
                else wend = true;
            }
            if (has && (queued || !wend)) avail = (unsigned)g + 1u;
            kg[g] = cr.x;
            ng[g] = cr.y;
        }
        if (has) {
            // take cells 0..m-1; the rest go back to the fifo
            // m = 1 + the number of prefixes (cells 0..g-1, g < avail) still
            // below min_pairs candidates: both conditions only turn false
            // (m = 0 when the walk has no cell left: the ray escapes below)
            const unsigned c1 = ng[0], c2 = c1 + ng[1], c3 = c2 + ng[2];
            constexpr unsigned MP = AO_MIN_PAIRS;
            const unsigned m = (avail > 0u) + (avail > 1u && c1 < MP) + (avail > 2u && c2 < MP) + (avail > 3u && c3 < MP);
#pragma unroll
            for (int g = 1; g < AO_CELLS; ++g) {
                if ((unsigned)g >= m && (unsigned)g < avail) S.fifo[lane][g - m] = make_uint2(kg[g], ng[g]);
                ng[g] = (unsigned)g >= m ? 0u : ng[g];
            }
            nf = avail - m;
            ending = wend && nf == 0u;  // escapes unless this iteration's tests hit
        }
        // 3. lay the warp's (ray, item) pairs out densely
        unsigned cnt = 0u;
#pragma unroll
        for (int g = 0; g < AO_CELLS; ++g) cnt += ng[g];
        unsigned incl = cnt;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            unsigned y = __shfl_up_sync(FULL, incl, off);
            if (lane >= off) incl += y;
        }
        const unsigned T = __shfl_sync(FULL, incl, 31);
        unsigned hitbits = 0;
        if (T > 0) {
            const unsigned ex = incl - cnt;
            const unsigned s1 = ex + ng[0], s2 = s1 + ng[1], s3 = s2 + ng[2];
            S.sds[lane] = make_uint4(ex, s1, s2, s3);
            S.sdo[lane] = make_uint4(kg[0] - ex, kg[1] - s1, kg[2] - s2, kg[3] - s3);
            // 4. map pairs to (ray, object) 32 at a time and test them in place
            //    (lanes past the last pair redo it, so the test runs without
            //    branches)
            for (unsigned base = 0; base < T; base += 32) {
                // rays mark where their pairs start inside this chunk; a pair's
                // ray is the last start at or before it. A ray takes part when its
                // pairs [ex, incl) are not empty and meet [base, base + 32).
                const unsigned u = ex > base ? ex : base;
                const unsigned pos = u - base;
                const bool mine = pos < 32u && incl > u;
                if (mine) S.owner[pos] = (uint32_t)lane;
                const unsigned starts = __reduce_or_sync(FULL, mine ? (1u << pos) : 0u);
                __syncwarp();
                const unsigned p = base + lane < T ? base + lane : T - 1u;
                const unsigned r = S.owner[31 - __clz(starts & (0xFFFFFFFFu >> (31 - lane)))];
                const uint4 st = S.sds[r], so = S.sdo[r];
                unsigned di = so.x;
                di = p >= st.y ? so.y : di;
                di = p >= st.z ? so.z : di;
                di = p >= st.w ? so.w : di;
                const uint32_t id = GBRT_AO_OBJ(__ldg(ao_items(S, r, uitems) + GBRT_AO_ITEM(p + di, r)), r);
                const AoRay ray = S.ray[r];
                float t;
                const bool hit = hit_object<float>(ao_obj(S, r, uobj), id, ray.o, ray.d, 0.0f, ray.tmax, t);
                hitbits |= hit ? (1u << r) : 0u;  // OR-ed over the warp after the last chunk
                __syncwarp();
            }
            hitbits = __reduce_or_sync(FULL, hitbits);
        }
        // 5. any hit occludes the ray; a ray whose walk ended escapes
        const bool occluded = (hitbits >> lane) & 1u;
        if (has && (occluded || ending)) {
            if (!occluded) ao_escape(b, vslot, lbit);
            has = false;
        }
        __syncwarp();
    }
    if (overflow) atomicOr(b.err, ERR_DDA_STEPS);
}

// ---- FP64 frames

// The ray a lane walks, and what settles it.
//   o        origin; of an FP64 ray: relative to the grid's lower corner
//            (formed in FP64, rounded once)
//   idd      -1 / d.d
//   slot     the hit (or the probe's point) it belongs to
//   lbit     0, or the bit of the light it goes to
//   f, smp   frame and sample: the exact FP64 ray is formed again where a test
//            needs it
struct LaneRay {
    V3<float> o, d;
    float idd, tmax;
    uint32_t lbit;
    int64_t slot;
    int f;
    uint32_t smp;
};
// a hit whose roots lie within this is within tmax
__device__ __forceinline__ float sure_within(float tmax) { return tmax * (1.0f - 1e-5f); }

// The scene and grid that a warp's rays in flight belong to (warp-uniform);
// lo and om: origin of an FP64 ray's coordinates, and the filter's margin for
// their rounding.
struct LaneScene {
    const float4* bs;
    const uint2* cells;
    const uint32_t* items;
    int64_t nitems;  // the checked build's bounds
    int32_t nobj;
    V3<float> lo;
    float om;
    // The balls a frame's rays are tested with: tubes cut to what sticks out of
    // their spheres (a ray without a limit that meets the rest meets the sphere
    // as well), unless the cut is of another geometry.
    static __device__ __forceinline__ const float4* balls(const FrameDev& F) {
        return isinf(F.ao_maxdist_f) && !F.stale ? F.grid.cut : F.scene.bs;
    }
    __device__ __forceinline__ bool is(const FrameDev& F) const { return F.grid.cells == cells && balls(F) == bs; }
    __device__ __forceinline__ void set(const FrameDev& F) {
        bs = balls(F);
        nobj = F.scene.S + F.scene.C;
        cells = F.grid.cells;
        items = F.grid.items;
        nitems = F.grid.nitems;
        lo = v3(F.grid.lo[0], F.grid.lo[1], F.grid.lo[2]);
        om = 0.1f * fmaxf(F.grid.hi[0] - lo.x, fmaxf(F.grid.hi[1] - lo.y, F.grid.hi[2] - lo.z));
    }
};

// What the filter left open: one pair through the reference test.
template <class Src>
__device__ __forceinline__ bool lane_settle(const Src& src, const LaneScene& A, const LaneRay& ray, uint32_t id) {
    V3<float> p0, a;
    float L, r, t, et;
    Obj<float>::load(src.frame(ray).scene.obj, id, p0, a, L, r);
    if constexpr (Src::F64) {
        if (L > 0.0f) {
            const int c = tube_root32(ray.o, ray.d, p0 - A.lo, a, L, r, sure_within(ray.tmax), ray.tmax, A.om, t, et);
            if (c != PAIR_OPEN) return c == PAIR_HIT;
        }
        return src.exact(ray, id);
    } else {
        return hit_prim(ray.o, ray.d, p0, a, L, r, 0.0f, ray.tmax, t);
    }
}

enum : int { LANES_GO = 0, LANES_AGAIN = 1, LANES_END = 2 };

// Any-hit walk, one ray per lane, over the rays that `src` hands out. A lane
// holds its walk, the rest of its current cell's item range [k, e), the record
// of the cell after it (already loaded) and the id of its next candidate
// (already loaded), so that an iteration -- one candidate through the filter,
// or one step into the next cell -- waits for one load. Candidates the filter
// leaves open wait in `pend` (a second one in `pend2`) and are settled
// together: when a lane has a second, when half the warp has one, and before
// lanes are refilled. A lane whose walk ended with an open candidate waits for
// that.
// Once fewer than `refill` lanes walk, src.refill gives the idle lanes rays.
template <class Src>
__device__ __forceinline__ void lane_walk(Src& src, LaneScene& A, int refill, uint32_t* err) {
    const int lane = threadIdx.x & 31;
    bool active = false, exhausted = false, overflow = false;
    LaneRay ray;
    Walk w;
    uint32_t k = 0, e = 0;         // items left of the lane's cell
    uint2 nxt = make_uint2(0, 0);  // the next cell's record, when more
    bool more = false;
    uint32_t id = 0;               // the candidate at k, when k < e
    uint32_t pend = GBRT_MISS, pend2 = GBRT_MISS;  // candidates the filter left open
    bool flush = false;            // settle them at the next turn (uniform)
    bool waiting = false;          // walk over, pend not settled yet
    while (true) {
        // settle what is open; finish the lanes that waited for it
        unsigned act = __ballot_sync(FULL, active);
        const bool low = exhausted ? act == 0u : __popc(act) < refill;
        if (low || flush) {
            flush = false;
            bool hit = false;
            if (pend != GBRT_MISS) hit = lane_settle(src, A, ray, GBRT_INDEX(pend, A.nobj));
            pend = hit ? GBRT_MISS : pend2;
            pend2 = GBRT_MISS;
            active = active && !hit;
            if (waiting && pend == GBRT_MISS) {
                if (!hit) src.escape(ray);
                waiting = false;
            }
            act = __ballot_sync(FULL, active);
            if (low && __any_sync(FULL, pend != GBRT_MISS)) continue;
        }
        if (low) {
            if (exhausted) {
                if (act == 0u) break;
                continue;
            }
            bool fresh = false;
            const int what = src.refill(A, lane, act, !active, ray, w, fresh);
            if (fresh) {
                ray.idd = __fdividef(-1.0f, dot(ray.d, ray.d));
                k = e = 0;
                nxt = __ldg(A.cells + GBRT_INDEX(w.cell, w.ncells));
                more = active = true;
            }
            exhausted = what == LANES_END;
            if (what != LANES_GO) continue;
        }
        // one candidate, or one cell
        bool ask = false;
        const uint32_t cur = id;
        const bool test = active && k < e;
        float4 s = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (test) {
            s = __ldg(A.bs + GBRT_INDEX(cur, A.nobj));
            ++k;
        }
        if (active && k >= e) {
            if (more) {
                k = nxt.x;
                e = nxt.x + nxt.y;
                if constexpr (Src::F64) more = walk_next_rel(w, src.frame(ray).grid, ray.o, ray.d, overflow);
                else more = walk_next(w, overflow);
                if (more) nxt = __ldg(A.cells + GBRT_INDEX(w.cell, w.ncells));
            } else if (!test) {
                // walk over: nothing left to test
                active = false;
                waiting = pend != GBRT_MISS;
                if (!waiting) src.escape(ray);
            }
        }
        if (active && k < e) id = __ldg(A.items + GBRT_INDEX(k, A.nitems));
        if (test) {
            V3<float> wv;
            if constexpr (Src::F64) wv = ray.o - v3(s.x - A.lo.x, s.y - A.lo.y, s.z - A.lo.z);
            else wv = ray.o - v3(s.x, s.y, s.z);
            const float bb = dot(wv, ray.d) * ray.idd;  // -b
            const V3<float> m = madd(wv, bb, ray.d);
            const float r = fabsf(s.w), bp = fminf(bb, 0.0f), reach = fabsf(bb) + r;
            const float x = fmaf(-r, r, fmaf(bp, bp, dot(m, m)));
            const float mg = filter_margin(r, Src::F64 ? reach + A.om : reach);
            if (x <= mg) {
                if (s.w > 0.0f && x < -mg && reach <= sure_within(ray.tmax)) {
                    active = false;  // occluded
                    pend = pend2 = GBRT_MISS;
                } else {
                    ask = true;
                }
            }
        }
        const unsigned asks = __ballot_sync(FULL, ask);
        if (asks) {
            const unsigned full = __ballot_sync(FULL, pend != GBRT_MISS);
            flush = (asks & full) != 0u || __popc(full) >= 16;
            if (ask && pend != GBRT_MISS) pend2 = cur;
            else if (ask) pend = cur;
        }
    }
    if (overflow) atomicOr(err, ERR_DDA_STEPS);
}

// The reference test of one (ray, object) pair of an FP64 frame, from the
// hit's FP64 record: any_hit_object64 on the ray that the sample defines.
__device__ __forceinline__ bool ao_exact64(const BatchDev& b, int f, int64_t vslot, uint32_t smp, uint32_t id) {
    const FrameDev& F = b.frames[f];
    V3<double> o, n, d;
    uint32_t q, own, lbit;
    double tmax;
    HitIO<double>::load(b.hits, vslot, o, n, q, own);
    ao_direction<double>(F, q, smp, n, d, tmax, lbit);
    return any_hit_object64(F.scene.obj64, id, o, d, tmax);
}

// The rays of a batch's FP64 frames: the warp's pool claims ao_claim jobs at a
// time. The rays in flight belong to one scene and grid; a warp whose pool
// moves on to another scene lets its lanes drain first. NEAR: the rays that the
// near pass left instead, from its units (every frame has the same scene and
// grid, and no AO limit).
template <bool NEAR>
struct FrameRays {
    static constexpr bool F64 = true;
    const BatchDev& b;
    AoUnit* const U;
    // the warp's claimed jobs [next, end) and the frame they belong to (uniform)
    unsigned long long next = 0, end = 0, f_lo = 0, f_hi = 0;
    int f = 0;

    __device__ __forceinline__ FrameRays(const BatchDev& batch, AoUnit* unit) : b(batch), U(unit) {}

    __device__ __forceinline__ void escape(const LaneRay& ray) const { ao_escape(b, ray.slot, ray.lbit); }

    __device__ __forceinline__ const FrameDev& frame(const LaneRay& ray) const { return b.frames[ray.f]; }

    __device__ __forceinline__ bool exact(const LaneRay& ray, uint32_t id) const {
        return ao_exact64(b, ray.f, ray.slot, ray.smp, id);
    }

    // Job smp of the hit in `slot`, from distance tmin on.
    __device__ __forceinline__ void set_up(const FrameDev& F, int fi, int64_t slot, uint32_t smp, float tmin,
                                           LaneRay& ray, Walk& w, bool& fresh) {
        uint32_t q, own;
        V3<float> nrm;
        ray.slot = slot;
        ray.smp = smp;
        ray.f = fi;
        HitIO<float>::load(b.hits32, slot, ray.o, nrm, q, own);
        if (ao_direction<float>(F, q, smp, nrm, ray.d, ray.tmax, ray.lbit, true)) {
            fresh = walk_start_rel(F.grid, ray.o, ray.d, tmin, ray.tmax, w);
            if (!fresh) ao_escape(b, slot, ray.lbit);  // misses the objects' bounds
        }
    }

    __device__ __forceinline__ int refill(LaneScene& A, int lane, unsigned act, bool free, LaneRay& ray, Walk& w,
                                          bool& fresh) {
        if constexpr (NEAR) {
            if (!A.cells) A.set(b.frames[0]);
            const unsigned idle = ~act;
            const FrameDev* Fp = nullptr;
            int64_t slot = 0;
            uint32_t smp = 0;
            float tmin = 0.0f;
            bool done = false;
            unit_take(b, *U, lane, *b.nunits, __popc(idle), __popc(idle & ((1u << lane) - 1u)), free, done, slot, smp,
                      tmin, Fp);
            if (Fp) set_up(*Fp, (int)(Fp - b.frames), slot, smp, tmin, ray, w, fresh);
            return done ? LANES_END : LANES_GO;
        }
        const unsigned long long total = b.job_off[b.nframes];
        if (next == end) {
            unsigned long long c = 0;
            const unsigned claim = (unsigned)b.queue[3];
            if (lane == 0) c = atomicAdd(b.queue + 1, (unsigned long long)claim);
            next = __shfl_sync(FULL, c, 0);
            if (next >= total) return LANES_END;
            end = next + claim < total ? next + claim : total;
        }
        if (next >= f_hi) {
            const int nf = b.nframes == 1 ? 0 : find_frame(b.job_off, b.nframes, next);
            const FrameDev& N = b.frames[nf];
            const bool same = A.is(N);
            if (!same && act != 0u) return LANES_GO;  // another scene: the lanes in flight drain first
            f = nf;
            f_lo = b.job_off[f];
            f_hi = b.job_off[f + 1];
            if (!same) A.set(N);
        }
        const FrameDev& F = b.frames[f];
        const unsigned idle = ~act, i = __popc(idle & ((1u << lane) - 1u));
        const unsigned long long left = (end < f_hi ? end : f_hi) - next;
        const unsigned n = left < (unsigned long long)__popc(idle) ? (unsigned)left : __popc(idle);
        if (free && i < n) {
            uint32_t h, smp;
            ao_split(F, next + i - f_lo, h, smp);
            set_up(F, f, GBRT_INDEX(F.hit_base + (int64_t)h, b.hit_cap), smp, 0.0f, ray, w, fresh);
        }
        next += n;
        return n < __popc(idle) && next < total ? LANES_AGAIN : LANES_GO;  // the rest from the next claim or frame
    }
};

// AO walk of FP64 frames, persistent. With every test and step in FP64 (1/64
// of the FP32 rate) the FP64 pipe was 87% busy and the walk took 15.5 of a
// 965 x 1137 frame's 17.9 ms; the filter leaves FP64 to one pair in some ten
// thousand (walk 1.53 ms; 256 x 256 frame at 8 samples 0.57 -> 0.11 ms). One
// ray a lane rather than the FP32 frames' pair expansion: with a filter this
// cheap the expansion costs more than the idle lanes (walk 3.8 ms with pairs
// queued in shared memory). Bound now by instruction issue and load
// latency. NEAR: after a near pass, over the rays it left (0.80 ms).
template <bool NEAR>
__global__ void __launch_bounds__(256, 3) k_ao_walk64(const __grid_constant__ BatchDev b) {
    __shared__ AoUnit units[NEAR ? 8 : 1];
    AoUnit* const unit = units + (NEAR ? threadIdx.x >> 5 : 0);
    grid_dependency_wait();
    if (NEAR) {
        unit->rem = 0u;
        __syncwarp();
    }
    FrameRays<NEAR> src(b, unit);
    LaneScene A;
    A.cells = nullptr;
    A.bs = nullptr;
    lane_walk(src, A, b.refill, b.err);
}

// ---------------------------------------------------------------- shading

template <class R>
__global__ void __launch_bounds__(256) k_shade(const __grid_constant__ BatchDev b) {
    grid_dependency_wait();
    const unsigned long long total = b.hit_off[b.nframes];
    for (unsigned long long g = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; g < total;
         g += (unsigned long long)gridDim.x * blockDim.x) {
        const int f = find_frame(b.hit_off, b.nframes, g);
        const FrameDev& F = b.frames[f];
        const int64_t slot = GBRT_INDEX(F.hit_base + (int64_t)(g - b.hit_off[f]), b.hit_cap);
        V3<R> o, n;
        uint32_t q, id;
        HitIO<R>::load(b.hits, slot, o, n, q, id);
        q = GBRT_INDEX(q, (uint32_t)F.W * (uint32_t)F.H);
        id = GBRT_INDEX(id, F.scene.S + F.scene.C);
        const uint32_t vis = b.vis[slot];
        V3<R> d;
        if (std::is_same<R, float>::value) {
            V3<float> df = view_dir_f(F, q);
            d = v3((R)df.x, (R)df.y, (R)df.z);
        } else {
            V3<double> o64, d64;
            primary_ray64(F, (int)(q % (uint32_t)F.W), (int)(q / (uint32_t)F.W), o64, d64);
            d = v3((R)d64.x, (R)d64.y, (R)d64.z);
        }
        R V = F.spp > 0 ? (R)vis / (R)F.spp : R(1);
        const uint32_t lit = F.shadows ? b.lmask[slot] : 0xFFFFFFFFu;
        R rgb[3];
        shade<R>(F, id, n, d, V, lit, rgb);
        // the colour buffer holds pixels [rgb_q0, ...): the whole image (rgb_q0 = 0)
        // or, for a supersampled frame, the finer raster's band (rgb_q0 = row0 W);
        // either way the band's pixels end at (row0 + rows) W
        R* out = (R*)F.out_rgb +
                 3 * (size_t)GBRT_INDEX((int64_t)q - F.rgb_q0, (int64_t)(F.row0 + F.rows) * F.W - F.rgb_q0);
        out[0] = rgb[0];
        out[1] = rgb[1];
        out[2] = rgb[2];
        if (F.out_vis) F.out_vis[q] = vis;
    }
}

// ---------------------------------------------------------------- grids rebuilt on the device

// Frames whose grid was rebuilt on the device take its current geometry
// before the frame's kernels run (their descriptors were written on the host).
__global__ void k_patch_grids(const __grid_constant__ BatchDev b) {
    FrameDev* frames = const_cast<FrameDev*>(b.frames);
    for (int f = blockIdx.x * blockDim.x + threadIdx.x; f < b.nframes; f += gridDim.x * blockDim.x)
        if (frames[f].grid_src) frames[f].grid = *frames[f].grid_src;
}

// ---------------------------------------------------------------- supersampling

// Box filter of supersampled frames: output pixel (i, j) is the mean of the
// m x m finer-raster colours (m i + a, m j + b), summed sub-row by sub-row.
// Frames are strided over blockIdx.y; frames without supersampling are skipped.
template <class R>
__global__ void __launch_bounds__(256) k_resolve(const __grid_constant__ BatchDev b) {
    grid_dependency_wait();
    for (int f = blockIdx.y; f < b.nframes; f += gridDim.y) {
        const FrameDev& F = b.frames[f];
        const int m = F.aa;
        if (m <= 1) continue;
        const int w = F.W / m;
        const int j0 = F.row0 / m;
        const long long n = (long long)w * (F.rows / m);
        const R mm = (R)(m * m);
        const R* fine = (const R*)F.out_rgb;
        R* out = (R*)F.out_final;
        for (long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x; k < n;
             k += (long long)gridDim.x * blockDim.x) {
            const int i = (int)(k % w), j = j0 + (int)(k / w);
            R acc[3] = {R(0), R(0), R(0)};
            for (int sb = 0; sb < m; ++sb) {
                const R* row = fine + 3 * ((long long)(m * j + sb) * F.W + (long long)m * i - F.rgb_q0);
                for (int sa = 0; sa < m; ++sa) {
                    acc[0] += row[3 * sa];
                    acc[1] += row[3 * sa + 1];
                    acc[2] += row[3 * sa + 2];
                }
            }
            R* o = out + 3 * ((long long)j * w + i);
            o[0] = acc[0] / mm;
            o[1] = acc[1] / mm;
            o[2] = acc[2] / mm;
        }
    }
}

// ---------------------------------------------------------------- probe, Philox

// The FP64 ray of sample smp of a probe's point pt. From far outside the objects
// it starts shortly before them instead (true): FP32 coordinates and crossings
// that grow with the distance would miss the cells, and an FP64 test loses its
// digits.
__device__ __forceinline__ bool probe_ray64(const FrameDev& F, const double* pts, const double* nrm, int64_t pt,
                                            uint32_t smp, V3<double>& o, V3<double>& d, double& tmax) {
    const V3<double> n = ld3(nrm + 3 * pt);
    o = madd(ld3(pts + 3 * pt), F.eps, n);
    uint32_t lbit;
    ao_direction<double>(F, (uint32_t)pt, smp, n, d, tmax, lbit);
    const double rb = F.grid.bs64[3], te = dot(ld3(F.grid.bs64) - o, d) - 1.1 * rb;
    if (!(te > rb)) return false;
    o = madd(o, te, d);
    tmax -= te;
    return true;
}

// That ray in FP32 where it is one from far outside (out of line: it is rare, and
// the probe's registers are the walk's).
struct FarRay {
    V3<float> o, d;
    float tmax;
    bool on;
};
__device__ __noinline__ FarRay probe_far_ray(const FrameDev& F, const double* pts, const double* nrm, int64_t pt,
                                             uint32_t smp) {
    V3<double> o, d;
    double tmax;
    FarRay r;
    r.on = probe_ray64(F, pts, nrm, pt, smp, o, d, tmax);
    r.o = to_f(o - ld3(F.grid.lo64));
    r.d = to_f(d);
    r.tmax = (float)tmax;
    return r;
}

// The rays of a probe's points: each warp takes a run of jobs (point, sample)
// of its own, so nothing is shared but the counts. A count is a float that
// escaped samples add 1 to: exact up to 2^24, the sample bound is 2^20.
template <bool FP64>
struct ProbeRays {
    static constexpr bool F64 = FP64;
    const FrameDev& F;
    const double* pts;
    const double* nrm;
    float* out;
    unsigned long long pool, pool_end;
    // the last point whose FP32 origin and normal were formed
    unsigned long long cached;
    V3<float> co, cn;

    __device__ __forceinline__ void escape(const LaneRay& ray) const { atomicAdd(out + ray.slot, 1.0f); }

    __device__ __forceinline__ const FrameDev& frame(const LaneRay&) const { return F; }

    __device__ __forceinline__ bool exact(const LaneRay& ray, uint32_t id) const {
        V3<double> o, d;
        double tmax;
        probe_ray64(F, pts, nrm, ray.slot, ray.smp, o, d, tmax);
        return any_hit_object64(F.scene.obj64, id, o, d, tmax);
    }

    __device__ __forceinline__ int refill(LaneScene&, int lane, unsigned act, bool free, LaneRay& ray, Walk& w,
                                          bool& fresh) {
        if (pool == pool_end) return LANES_END;
        const unsigned idle = ~act, i = __popc(idle & ((1u << lane) - 1u));
        const unsigned long long left = pool_end - pool;
        const unsigned n = left < (unsigned long long)__popc(idle) ? (unsigned)left : __popc(idle);
        const bool mine = free && i < n;
        const unsigned long long j = pool + i, spp = (unsigned long long)F.spp, pt = j / spp;
        const uint32_t smp = (uint32_t)(j - pt * spp);
        // origins are formed in FP64: once per point, not per refill
        V3<float> n0 = cn;
        if (mine) ray.o = co;
        if (__any_sync(FULL, mine && pt != cached)) {
            if (mine) {
                const V3<double> nn = ld3(nrm + 3 * pt), oo = madd(ld3(pts + 3 * pt), F.eps, nn);
                ray.o = co = to_f(FP64 ? oo - ld3(F.grid.lo64) : oo);
                n0 = cn = to_f(nn);
            }
            const unsigned last = 31u - __clz(__ballot_sync(FULL, mine));
            cached = __shfl_sync(FULL, pt, last);
            co = v3(__shfl_sync(FULL, co.x, last), __shfl_sync(FULL, co.y, last), __shfl_sync(FULL, co.z, last));
            cn = v3(__shfl_sync(FULL, cn.x, last), __shfl_sync(FULL, cn.y, last), __shfl_sync(FULL, cn.z, last));
        }
        if (mine) {
            float tmax;
            uint32_t lbit;
            ao_direction<float>(F, (uint32_t)pt, smp, n0, ray.d, tmax, lbit);
            if constexpr (FP64) {
                const GridDev& g = F.grid;
                const V3<float> q = ray.o - v3(g.bs[0] - g.lo[0], g.bs[1] - g.lo[1], g.bs[2] - g.lo[2]);
                if (dot(q, q) > 4.0f * g.bs[3] * g.bs[3]) {
                    const FarRay far = probe_far_ray(F, pts, nrm, (int64_t)pt, smp);
                    if (far.on) {
                        ray.o = far.o;
                        ray.d = far.d;
                        tmax = far.tmax;
                    }
                }
                fresh = walk_start_rel(g, ray.o, ray.d, 0.0f, tmax, w);
            } else {
                fresh = walk_start(F.grid, ray.o, ray.d, 0.0f, tmax, w);
            }
            ray.slot = (int64_t)pt;
            ray.tmax = tmax;
            ray.smp = smp;
            if (!fresh) escape(ray);
        }
        pool += n;
        return LANES_GO;
    }
};

// AO probe, counting pass: job (point, sample) runs of `run` a warp. One ray a
// lane through the filter (lane_walk) with all samples of a point spread over
// lanes; one thread a point before walked its samples one after another with
// the general test: 8,192 points x 64 samples 1.58 -> 0.13 ms.
template <int MODE>
__global__ void __launch_bounds__(256, 3) k_ao_probe(const __grid_constant__ FrameDev f, const double* pts,
                                                     const double* nrm, unsigned long long jobs,
                                                     unsigned long long run, float* out, uint32_t* err) {
    const unsigned long long warp = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const unsigned long long lo = warp * run;
    if (lo >= jobs) return;
    ProbeRays<MODE == GBRT_FP64> src{f, pts, nrm, out, lo, lo + run < jobs ? lo + run : jobs, ~0ull};
    LaneScene A;
    A.set(f);
    lane_walk(src, A, 16, err);
}

// Escaped samples -> visibility (1 where nothing was sampled).
__global__ void k_probe_share(float* out, int64_t n, int spp) {
    for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
        out[k] = spp > 0 ? out[k] / (float)spp : 1.0f;
}

__global__ void k_philox(const uint4* ctr, const uint2* key, int64_t n, uint4* out) {
    int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (k < n) out[k] = philox4x32_10(ctr[k], key[k]);
}

// ---------------------------------------------------------------- host side

namespace {

int err_of(cudaError_t e) {
    if (e == cudaSuccess) return GBRT_OK;
    return e == cudaErrorMemoryAllocation ? GBRT_ENOMEM : GBRT_EDEVICE;
}

template <class K>
int persistent_grid(Ctx* ctx, K kernel, int block, size_t smem = 0) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, smem) != cudaSuccess || per_sm < 1)
        per_sm = 1;
    if (ctx->tuning.ctas_per_sm > 0) per_sm = std::min(per_sm, ctx->tuning.ctas_per_sm);
    return per_sm * ctx->num_sms;
}

}  // namespace

int grow(Ctx* ctx, void** p, size_t* cap, size_t need) {
    if (*cap >= need) return GBRT_OK;
    cudaStreamSynchronize(ctx->stream);
    cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    size_t want = std::max(need, (size_t)4096);
    int rc = err_of(cudaMalloc(p, want));
    if (rc == GBRT_OK) *cap = want;
    ctx->graph_valid = false;
    return rc;
}

// Lay out one batch (all frames of one precision), upload its descriptors and
// enqueue memsets + the four kernels on `stream`.
struct Grids {
    int primary, near, ao, shade, resolve;  // near: 0 without a near pass
};

// Launch `kernel` as a programmatic dependent of the kernel before it in
// `stream`: its CTAs may be scheduled while that kernel drains, and they wait
// (grid_dependency_wait) for its results before reading them.
static cudaError_t launch_dependent(void (*kernel)(BatchDev), dim3 grid, dim3 block, size_t smem,
                                    cudaStream_t stream, const BatchDev& bd) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, bd);
}

template <bool UNI, bool NEAR>
static size_t ao_smem(int block) {
    return (size_t)(block / 32) * sizeof(AoWarp<UNI, NEAR>);
}
constexpr int NEAR_BLOCK = 128;
constexpr size_t NEAR_SMEM = NEAR_BLOCK / 32 * sizeof(NearWarp);
static_assert(NEAR_SMEM <= 48 * 1024, "above this a kernel has to ask for its shared memory");

// Shared-memory share of the SM asked for an AO walk whose CTAs of 256 threads
// use `smem` bytes: just enough for four of them (and the driver's per-CTA
// reservation), so the rest of the SM's 256 KB serves as L1 for the walk's
// cell, item and object loads (FP32: the 100 KB configuration instead of the
// 132 KB one the driver picks by default: AO walk 1.185 -> 1.176 ms on the
// paper frame).
template <class K>
static cudaError_t prefer_small_carveout(K kernel, size_t smem) {
    int dev = 0, per_sm = 0, reserved = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    if (e != cudaSuccess || per_sm <= 0) return e;
    const long long need = 4ll * ((long long)smem + reserved);
    const int pct = (int)std::min<long long>(100, (need * 100 + per_sm - 1) / per_sm);
    return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
}

// A refused preference leaves the driver's choice (and its error is cleared
// here, so it is not taken for a later launch's).
static void configure_ao() {
    if (prefer_small_carveout(k_ao_walk<true, false>, ao_smem<true, false>(256)) != cudaSuccess ||
        prefer_small_carveout(k_ao_walk<false, false>, ao_smem<false, false>(256)) != cudaSuccess ||
        prefer_small_carveout(k_ao_walk<true, true>, ao_smem<true, true>(256)) != cudaSuccess ||
        prefer_small_carveout(k_ao_walk<false, true>, ao_smem<false, true>(256)) != cudaSuccess ||
        prefer_small_carveout(k_ao_walk64<false>, 0) != cudaSuccess ||
        prefer_small_carveout(k_ao_walk64<true>, 8 * sizeof(AoUnit)) != cudaSuccess)
        (void)cudaGetLastError();
}

// uni: one scene and grid for the whole batch; near > 0: with a near pass of
// that many CTAs
template <class R>
static void launch_ao(const BatchDev& bd, bool uni, int near, int grid, int block, cudaStream_t stream) {
    if (std::is_same<R, double>::value) {
        if (near > 0) {
            launch_dependent(k_ao_near<true>, near, NEAR_BLOCK, NEAR_SMEM, stream, bd);
            launch_dependent(k_ao_walk64<true>, grid, block, 0, stream, bd);
        } else {
            launch_dependent(k_ao_walk64<false>, grid, block, 0, stream, bd);
        }
    } else if (near > 0) {
        launch_dependent(k_ao_near<false>, near, NEAR_BLOCK, NEAR_SMEM, stream, bd);
        if (uni) launch_dependent(k_ao_walk<true, true>, grid, block, ao_smem<true, true>(block), stream, bd);
        else launch_dependent(k_ao_walk<false, true>, grid, block, ao_smem<false, true>(block), stream, bd);
    } else {
        if (uni) launch_dependent(k_ao_walk<true, false>, grid, block, ao_smem<true, false>(block), stream, bd);
        else launch_dependent(k_ao_walk<false, false>, grid, block, ao_smem<false, false>(block), stream, bd);
    }
}

template <int MODE>
static void launch_primary(const BatchDev& bd, int grid, int block, cudaStream_t stream) {
    if (bd.parts > 1) k_primary<MODE, true><<<grid, block, 0, stream>>>(bd);
    else k_primary<MODE, false><<<grid, block, 0, stream>>>(bd);
}

// The passes after the primary one: AO walk, shading, and the box filter of
// supersampled frames (the AO plan runs in the primary kernel's last CTA).
template <class R>
static void launch_after_primary(const BatchDev& bd, bool uni, int near, int ao_grid, int block, int shade_grid,
                                 int resolve_grid, bool resolve, cudaStream_t stream,
                                 const std::function<void(int)>& mark) {
    launch_ao<R>(bd, uni, near, ao_grid, block, stream);
    mark(3);
    launch_dependent(k_shade<R>, shade_grid, 256, 0, stream, bd);
    if (resolve) launch_dependent(k_resolve<R>, dim3(resolve_grid, std::min(bd.nframes, 65535)), 256, 0, stream, bd);
}

static Grids grids_for(Ctx* ctx, int precision, bool uni, bool near) {
    const int block = ctx->tuning.block;
    if (!ctx->smem_configured) {
        configure_ao();
        ctx->smem_configured = true;
    }
    Grids g;
    g.near = !near ? 0
             : precision == GBRT_FP32 ? persistent_grid(ctx, k_ao_near<false>, NEAR_BLOCK, NEAR_SMEM)
                                      : persistent_grid(ctx, k_ao_near<true>, NEAR_BLOCK, NEAR_SMEM);
    if (precision == GBRT_FP32) {
        g.primary = persistent_grid(ctx, k_primary<GBRT_FP32, false>, block);
        if (near)
            g.ao = uni ? persistent_grid(ctx, k_ao_walk<true, true>, block, ao_smem<true, true>(block))
                       : persistent_grid(ctx, k_ao_walk<false, true>, block, ao_smem<false, true>(block));
        else
            g.ao = uni ? persistent_grid(ctx, k_ao_walk<true, false>, block, ao_smem<true, false>(block))
                       : persistent_grid(ctx, k_ao_walk<false, false>, block, ao_smem<false, false>(block));
    } else {
        g.primary = persistent_grid(ctx, k_primary<GBRT_FP64, false>, block);
        g.ao = near ? persistent_grid(ctx, k_ao_walk64<true>, block) : persistent_grid(ctx, k_ao_walk64<false>, block);
    }
    g.shade = ctx->num_sms * 8;
    g.resolve = ctx->num_sms * 4;
    return g;
}

// Every frame of the batch reads the same scene and grid (device-side rebuilt
// grids: the same rebuilt grid).
static bool one_scene(const FrameDev* frames, int n) {
    for (int f = 1; f < n; ++f) {
        const FrameDev& a = frames[0];
        const FrameDev& c = frames[f];
        if (c.scene.obj != a.scene.obj || c.scene.obj64 != a.scene.obj64 || c.grid.items != a.grid.items ||
            c.grid.cells != a.grid.cells || c.grid_src != a.grid_src)
            return false;
    }
    return true;
}

// Whether a near pass suits a frame's AO rays: enough of them a hit to share its
// per-hit work, no limit on their length (the pass takes a hit at any distance
// for one), and objects small enough (grid.rho); the grid's balls have to be the
// scene's.
static bool near_pass_suits(const FrameDev& f) {
    return f.grid.rho > 0.0f && !f.stale && std::isinf(f.ao_maxdist_f) &&
           f.jobs_per_hit >= NEAR_MIN_JOBS && f.jobs_per_hit <= NEAR_MAX_JOBS;
}

// Lanes that share a primary ray (split_walk). A frame with fewer tiles than the
// kernel has warps is bound by the latency of its slowest warp, a chain of
// dependent loads and tests (cell, item, object): 128 x 96 pixels, 36 us of
// which the mean warp is busy for 7. Then 2, 4 or 8 lanes walk a ray between
// them: 25 us with 8 at 128 x 96 (a frame of 520 atoms 66.7 -> 54), a 256 x 256
// frame 79.8 -> 71.9 with 2, FP64 184 -> 179. With more lanes than keep every
// tile resident at once the cells visited past the hit cost more than they hide
// in FP32 (256 x 256: 4 lanes 74, 8 lanes 84; FP64 171 and 192).
static int ray_parts(long long tiles, int warps) {
    int parts = 1;
    while (parts < 8 && 2 * parts * tiles <= warps) parts *= 2;
    return parts;
}

// Share of a frame's pixels that the objects' bounding sphere covers, roughly
// (a disc against the window; 1 from inside).
static double hit_share(const FrameDev& f) {
    double along = 0.0, r = f.grid.bs64[3], scale = 1.0;
    for (int k = 0; k < 3; ++k) along += (f.grid.bs64[k] - f.eye[k]) * f.dir_unit[k];
    if (f.cam_kind == GBRT_CAMERA_PINHOLE) {
        if (along <= r) return 1.0;
        scale = along;
    }
    return 0.785 * std::min(1.0, r / (f.half_w * scale)) * std::min(1.0, r / (f.half_h * scale));
}

// What the near pass saves a frame with that many tiles that are hit, in rays of a
// tile. A word of 16 jobs pays for its gather and scan with some 5 of them; a
// later word of 8 or fewer, scanned in fours, with all. The larger a tile is
// against the objects' distance, the more balls stand around it and the less far
// the pass looks, sooner with few jobs a hit. Fitted to 1,600 pairs of frames
// with and without the pass (orthographic; 1,014 to 249,990 objects; 200 to 1,300
// pixels a side; 8 to 64 jobs; the whole molecule or a third of it; FP32 and
// FP64): of the frames that get the pass, three lose by it, 2% at most; of those
// that do not, none would gain more than 11%. A line at a number of records (4,608
// and 3,072), as before, let frames of 8 jobs lose up to 16%: 26,318 objects at
// 560 x 560, 0.293 ms without and 0.318 with the pass; 250,000 objects at 330 x
// 330 and 48 samples, 0.547 and 0.599.
static double near_work(const FrameDev& f, double hit_tiles) {
    const int words = (f.jobs_per_hit + 15) / 16;
    double jobs = 0.0;
    for (int w = 0; w < words; ++w) {
        const int n = std::min(16, f.jobs_per_hit - 16 * w);
        if (w == 0 || n > 8) jobs += std::max(0, n - 5);
    }
    // a tile's linear size in mean distances of the objects, where they are
    double scale = 1.0;
    if (f.cam_kind == GBRT_CAMERA_PINHOLE) {
        double along = 0.0;
        for (int k = 0; k < 3; ++k) along += (f.grid.bs64[k] - f.eye[k]) * f.dir_unit[k];
        scale = std::max(along, 0.5 * f.grid.bs64[3]);
    }
    const double pixel = 2.0 * scale * std::sqrt(f.half_w * f.half_h * f.inv_w * f.inv_h);
    const double tile = std::sqrt(32.0) * pixel * std::cbrt((double)f.grid.density);
    const double full = std::min(f.jobs_per_hit, 16) / 16.0;
    const double reach = tile / (f.precision == GBRT_FP64 ? 0.2 + 0.2 * full : 0.3 * full);
    return hit_tiles * jobs / (1.0 + reach * reach);
}

// optional passes of a batch, and its scene layout
enum : int { EXTRA_RESOLVE = 1, EXTRA_PATCH = 2, EXTRA_UNI = 4 };

static int enqueue_batch(Ctx* ctx, cudaStream_t stream, int precision, const BatchDev& bd, size_t desc_bytes,
                         const Grids& gr, int extra) {
    const bool resolve = (extra & EXTRA_RESOLVE) != 0;
    cudaError_t e = cudaMemcpyAsync(ctx->d_desc, ctx->h_desc, desc_bytes, cudaMemcpyHostToDevice, stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(ctx->d_counters, 0, ctx->counters_bytes_used, stream);
    if (e != cudaSuccess) return err_of(e);
    const int block = ctx->tuning.block;
    if (extra & EXTRA_PATCH) {
        k_patch_grids<<<1, 128, 0, stream>>>(bd);
        ctx->launches++;
    }
    // events between the kernels when timing (never inside a graph capture);
    // the AO-walk mode records only events 2 and 3, around the AO walk
    const int tm = stream == ctx->stream ? ctx->profiling : 0;
    auto mark = [&](int k) {
        if (tm == GBRT_PROFILE_ALL || (tm == GBRT_PROFILE_AO_WALK && (k == 2 || k == 3)))
            cudaEventRecord(ctx->ev[k], stream);
    };
    mark(0);
    const bool uni = (extra & EXTRA_UNI) != 0;
    if (precision == GBRT_FP32) {
        launch_primary<GBRT_FP32>(bd, gr.primary, block, stream);
        mark(1);
        mark(2);
        launch_after_primary<float>(bd, uni, gr.near, gr.ao, block, gr.shade, gr.resolve, resolve, stream, mark);
    } else {
        launch_primary<GBRT_FP64>(bd, gr.primary, block, stream);
        mark(1);
        mark(2);
        launch_after_primary<double>(bd, uni, gr.near, gr.ao, block, gr.shade, gr.resolve, resolve, stream, mark);
    }
    mark(4);
    if (tm) ctx->timed = tm;
    ctx->launches += 3 + (resolve ? 1 : 0) + (gr.near ? 1 : 0);
    return err_of(cudaGetLastError());
}

int render_frames(Ctx* ctx, FrameDev* frames, int n, bool use_graph) {
    if (n == 0) return GBRT_OK;
    const int precision = frames[0].precision;
    for (int f = 1; f < n; ++f)
        if (frames[f].precision != precision) return GBRT_EINVAL;
    const int tw = ctx->tuning.tile_w, th = ctx->tuning.tile_h;
    // hit records: FP32, or FP64 and the AO walk's FP32 ones behind them
    const size_t rec64 = precision == GBRT_FP32 ? 0 : 4 * sizeof(double2);
    const size_t rec = rec64 + 2 * sizeof(float4);
    // descriptors: frames, then tile_off (n + 1)
    const size_t frames_bytes = ((size_t)n * sizeof(FrameDev) + 255) & ~(size_t)255;
    const size_t desc_bytes = frames_bytes + (size_t)(n + 1) * sizeof(long long);
    // counters: queue [4], near units, near tiles, hit_count [n], job_off [n + 1],
    // hit_off [n + 1]
    const size_t counters_bytes = 6 * sizeof(unsigned long long) + (size_t)n * sizeof(unsigned) +
                                  2 * (size_t)(n + 1) * sizeof(unsigned long long) + 64;
    int64_t px = 0;
    long long tiles = 0;
    int64_t near_rays = 0;  // rays of the frames that a near pass suits, if every pixel hits
    bool many = false;      // a frame with too many jobs a hit for masks
    double near_gain = 0;   // and what the pass saves them (near_work)
    int64_t mask_words = 0, recs = 0, words = 0, all_rays = 0;  // recs, words: tile records, and their job words
    size_t fine_bytes = 0;  // finer-raster colours of the supersampled frames' bands
    bool resolve = false;
    int extra = 0;
    const size_t rgb_px = 3 * (precision == GBRT_FP32 ? sizeof(float) : sizeof(double));
    for (int f = 0; f < n; ++f) {
        frames[f].tiles_x = (frames[f].W + tw - 1) / tw;
        frames[f].tiles_y = (frames[f].rows + th - 1) / th;
        frames[f].hit_base = px;
        const int64_t fpx = (int64_t)frames[f].W * frames[f].rows;
        const long long ftiles = (long long)frames[f].tiles_x * frames[f].tiles_y;
        px += fpx;
        tiles += ftiles;
        frames[f].near_pass = near_pass_suits(frames[f]) ? 1 : 0;
        frames[f].mask_words = std::min((frames[f].jobs_per_hit + 15) / 16, (NEAR_MAX_JOBS + 15) / 16);
        frames[f].mask_base = mask_words;
        // a record takes all of its tile's words (they share the gather) unless
        // that leaves too few records
        const double hit_tiles = std::max(1.0, (double)ftiles * hit_share(frames[f]));
        const int per_tile = (int)std::min<double>(std::ceil(NEAR_FULL_RECS / hit_tiles),
                                                   (double)std::max(frames[f].mask_words, 1));
        frames[f].rec_words = std::max(1, (frames[f].mask_words + per_tile - 1) / per_tile);
        if (frames[f].near_pass) {
            near_rays += fpx * frames[f].jobs_per_hit;
            near_gain += near_work(frames[f], hit_tiles);
        }
        all_rays += fpx * frames[f].jobs_per_hit;
        many = many || frames[f].jobs_per_hit > NEAR_MAX_JOBS;
        mask_words += fpx * frames[f].mask_words;
        recs += ftiles * ((frames[f].mask_words + frames[f].rec_words - 1) / frames[f].rec_words);
        words += ftiles * frames[f].mask_words;
        if (frames[f].grid_src) extra |= EXTRA_PATCH;
        if (frames[f].aa > 1) {
            resolve = true;
            extra |= EXTRA_RESOLVE;
            fine_bytes += ((size_t)frames[f].W * frames[f].rows * rgb_px + 255) & ~(size_t)255;
        }
    }
    int rc;
    if (resolve) {
        if ((rc = grow(ctx, &ctx->d_fine, &ctx->fine_cap, fine_bytes)) != GBRT_OK) return rc;
        size_t off = 0;
        for (int f = 0; f < n; ++f) {
            if (frames[f].aa <= 1) continue;
            frames[f].out_rgb = (char*)ctx->d_fine + off;
            frames[f].rgb_q0 = (int64_t)frames[f].row0 * frames[f].W;
            off += ((size_t)frames[f].W * frames[f].rows * rgb_px + 255) & ~(size_t)255;
        }
    }
    if ((rc = grow(ctx, &ctx->d_hits, &ctx->hits_cap, (size_t)px * rec)) != GBRT_OK) return rc;
    if ((rc = grow(ctx, (void**)&ctx->d_vis, &ctx->vis_cap, (size_t)px * sizeof(unsigned))) != GBRT_OK) return rc;
    if ((rc = grow(ctx, (void**)&ctx->d_lmask, &ctx->lmask_cap, (size_t)px * sizeof(unsigned))) != GBRT_OK)
        return rc;
    // enough of them to pay for one more kernel, and at least half of the batch's
    // rays
    const bool uni = one_scene(frames, n);
    bool near = precision == GBRT_FP32
                    ? near_gain >= NEAR_MIN_WORK && 2 * near_rays >= all_rays && !many
                    : near_gain >= NEAR_MIN_WORK64 && near_rays == all_rays && !many && uni;
    const size_t units_at = (size_t)recs * sizeof(TileRec);
    const size_t masks_at = units_at + 4 * (size_t)words * sizeof(unsigned long long);
    if (near) {
        rc = grow(ctx, &ctx->d_near, &ctx->near_cap, masks_at + (size_t)mask_words * sizeof(unsigned));
        if (rc == GBRT_ENOMEM) {  // without memory for it, the frame does without the pass
            (void)cudaGetLastError();
            near = false;
        } else if (rc != GBRT_OK) {
            return rc;
        }
    }
    if ((rc = grow(ctx, &ctx->d_desc, &ctx->desc_cap, desc_bytes)) != GBRT_OK) return rc;
    if ((rc = grow(ctx, &ctx->d_counters, &ctx->counters_cap, counters_bytes)) != GBRT_OK) return rc;
    if (ctx->h_desc_cap < desc_bytes) {
        if (ctx->staging_pending) cudaEventSynchronize(ctx->staging_done);
        cudaFreeHost(ctx->h_desc);
        ctx->h_desc = nullptr;
        ctx->h_desc_cap = 0;
        if (cudaMallocHost(&ctx->h_desc, desc_bytes) != cudaSuccess) return GBRT_ENOMEM;
        ctx->h_desc_cap = desc_bytes;
        ctx->graph_valid = false;
    }
    // the pinned staging buffer is read by the previous batch's copy: wait for it
    if (ctx->staging_pending) cudaEventSynchronize(ctx->staging_done);
    memcpy(ctx->h_desc, frames, (size_t)n * sizeof(FrameDev));
    long long* toff = (long long*)((char*)ctx->h_desc + frames_bytes);
    toff[0] = 0;
    for (int f = 0; f < n; ++f) toff[f + 1] = toff[f] + (long long)frames[f].tiles_x * frames[f].tiles_y;

    BatchDev bd;
    bd.frames = (const FrameDev*)ctx->d_desc;
    bd.tile_off = (const long long*)((char*)ctx->d_desc + frames_bytes);
    char* cb = (char*)ctx->d_counters;
    bd.queue = (unsigned long long*)cb;
    bd.nunits = bd.queue + 4;
    bd.ntiles = bd.queue + 5;
    bd.job_off = bd.queue + 6;
    bd.hit_off = bd.job_off + (n + 1);
    bd.hit_count = (unsigned*)(bd.hit_off + (n + 1));
    bd.hits = ctx->d_hits;
    bd.hits32 = (char*)ctx->d_hits + (size_t)px * rec64;
    bd.vis = ctx->d_vis;
    bd.lmask = ctx->d_lmask;
    bd.err = ctx->d_err;
    bd.tiles = near ? (TileRec*)ctx->d_near : nullptr;
    bd.units = near ? (unsigned long long*)((char*)ctx->d_near + units_at) : nullptr;
    bd.masks = near ? (unsigned*)((char*)ctx->d_near + masks_at) : nullptr;
    bd.hit_cap = (int64_t)px;
    bd.tile_cap = near ? recs : 0;
    bd.mask_cap = near ? mask_words : 0;
    bd.unit_cap = near ? 4 * words : 0;
    bd.nframes = n;
    bd.tile_w = tw;
    bd.tile_h = th;
    bd.refill = ctx->tuning.refill;
    ctx->counters_bytes_used = counters_bytes;

    if (uni) extra |= EXTRA_UNI;
    const Grids gr = grids_for(ctx, precision, uni, near);
    bd.ao_warps = gr.ao * (ctx->tuning.block / 32);
    bd.parts = near ? 1 : ray_parts(tiles, gr.primary * (ctx->tuning.block / 32));
    if (!use_graph) {
        rc = enqueue_batch(ctx, ctx->stream, precision, bd, desc_bytes, gr, extra);
    } else {
        // replay a captured graph of {copy, memset, 4 kernels} when the batch
        // layout (buffers, counts, launch shape) is unchanged
        const long long key = ((long long)n << 40) ^ ((long long)precision << 36) ^ ((long long)gr.primary << 18) ^
                              (long long)gr.ao ^ ((long long)desc_bytes << 1);
        if (!ctx->graph_valid || ctx->graph_key != key || ctx->graph_extra != extra ||
            memcmp(&ctx->graph_bd, &bd, sizeof(bd)) != 0) {
            if (ctx->graph_exec) cudaGraphExecDestroy(ctx->graph_exec);
            ctx->graph_exec = nullptr;
            ctx->graph_valid = false;
            if (!ctx->capture_stream &&
                cudaStreamCreateWithFlags(&ctx->capture_stream, cudaStreamNonBlocking) != cudaSuccess)
                return GBRT_EDEVICE;
            cudaGraph_t graph;
            if (cudaStreamBeginCapture(ctx->capture_stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess)
                return GBRT_EDEVICE;
            int64_t launches0 = ctx->launches;
            int crc = enqueue_batch(ctx, ctx->capture_stream, precision, bd, desc_bytes, gr, extra);
            ctx->launches = launches0;
            cudaError_t ce = cudaStreamEndCapture(ctx->capture_stream, &graph);
            if (crc != GBRT_OK || ce != cudaSuccess) return crc != GBRT_OK ? crc : GBRT_EDEVICE;
            ce = cudaGraphInstantiate(&ctx->graph_exec, graph, 0);
            cudaGraphDestroy(graph);
            if (ce != cudaSuccess) return GBRT_EDEVICE;
            ctx->graph_valid = true;
            ctx->graph_key = key;
            ctx->graph_extra = extra;
            ctx->graph_bd = bd;
        }
        rc = err_of(cudaGraphLaunch(ctx->graph_exec, ctx->stream));
        ctx->launches += 3 + (resolve ? 1 : 0) + (gr.near ? 1 : 0) + ((extra & EXTRA_PATCH) ? 1 : 0);
    }
    if (rc != GBRT_OK) return rc;
    cudaEventRecord(ctx->staging_done, ctx->stream);
    ctx->staging_pending = true;
    return GBRT_OK;
}

void configure_render_kernels() { configure_ao(); }

int enqueue_prepared(BatchDev bd, int precision, long long tiles, cudaStream_t stream, int block, int num_sms,
                     bool patch) {
    auto grid_of = [&](auto kernel, size_t smem = 0) {
        int per_sm = 0;
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, block, smem) != cudaSuccess || per_sm < 1)
            per_sm = 1;
        return per_sm * num_sms;
    };
    // one frame: one scene and grid
    if (patch) k_patch_grids<<<1, 128, 0, stream>>>(bd);
    const auto none = [](int) {};
    const int ao = precision == GBRT_FP32 ? grid_of(k_ao_walk<true, false>, ao_smem<true, false>(block))
                                          : grid_of(k_ao_walk64<false>);
    bd.ao_warps = ao * (block / 32);
    const int primary = precision == GBRT_FP32 ? grid_of(k_primary<GBRT_FP32, false>)
                                               : grid_of(k_primary<GBRT_FP64, false>);
    bd.parts = ray_parts(tiles, primary * (block / 32));
    if (precision == GBRT_FP32) {
        launch_primary<GBRT_FP32>(bd, primary, block, stream);
        launch_after_primary<float>(bd, true, 0, ao, block, num_sms * 8, 0, false, stream, none);
    } else {
        launch_primary<GBRT_FP64>(bd, primary, block, stream);
        launch_after_primary<double>(bd, true, 0, ao, block, num_sms * 8, 0, false, stream, none);
    }
    return err_of(cudaGetLastError());
}

int launch_ao_probe(Ctx* ctx, const FrameDev& f, const double* pts, const double* nrm, int64_t n, float* out) {
    if (n == 0) return GBRT_OK;
    const unsigned long long jobs = (unsigned long long)n * (unsigned long long)f.spp;
    if (cudaMemsetAsync(out, 0, (size_t)n * sizeof(float), ctx->stream) != cudaSuccess) return GBRT_EDEVICE;
    if (jobs > 0) {
        // runs of at least a warp's width, at most one resident wave of warps
        const unsigned long long warps = (unsigned long long)ctx->num_sms * 24;
        const unsigned long long run = (std::max<unsigned long long>((jobs + warps - 1) / warps, 1) + 31) / 32 * 32;
        const int blocks = (int)(((jobs + run - 1) / run + 7) / 8);
        if (f.precision == GBRT_FP32)
            k_ao_probe<GBRT_FP32><<<blocks, 256, 0, ctx->stream>>>(f, pts, nrm, jobs, run, out, ctx->d_err);
        else
            k_ao_probe<GBRT_FP64><<<blocks, 256, 0, ctx->stream>>>(f, pts, nrm, jobs, run, out, ctx->d_err);
        ctx->launches++;
    }
    k_probe_share<<<(int)std::min<int64_t>((n + 255) / 256, 65535), 256, 0, ctx->stream>>>(out, n, f.spp);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? GBRT_OK : GBRT_EDEVICE;
}

int launch_philox(Ctx* ctx, const uint32_t* ctr, const uint32_t* key, int64_t n, uint32_t* out) {
    if (n == 0) return GBRT_OK;
    int blocks = (int)((n + 255) / 256);
    k_philox<<<blocks, 256, 0, ctx->stream>>>((const uint4*)ctr, (const uint2*)key, n, (uint4*)out);
    ctx->launches++;
    return cudaGetLastError() == cudaSuccess ? GBRT_OK : GBRT_EDEVICE;
}

#ifdef GBRT_CHECKED
// Indices the checked build found outside their buffers since the last call
// (the render kernels' counter), cleared as it is read.
unsigned long long checked_violations_render() {
    unsigned long long v = 0, z = 0;
    if (cudaMemcpyFromSymbol(&v, g_oob, sizeof(v)) != cudaSuccess) return 0;
    cudaMemcpyToSymbol(g_oob, &z, sizeof(z));
    return v;
}
#endif

}  // namespace gbrt
