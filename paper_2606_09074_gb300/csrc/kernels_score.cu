// The N x V importance kernel (Eq. 7, Eq. 20), plain and batched.
#include <math.h>

#include "internal.h"

namespace refine {

// ---------------------------------------------------------------------
// The N x V importance kernel.
//
// The lanes of a warp hold 64 consecutive primitives of the processing order,
// two each, or 32 (a "tile"; score_plan), and walk the cameras of the pass, or
// of an item of 64 views where the tile is split (TilePart); the camera records
// are staged once per CTA into shared memory by
// a TMA bulk copy.  For primitive i and view v (Eq. 13-14, Eq. 17, Eq. 20):
//   (U, V, z) = P mu + p                  homogeneous pixel, u = U / z
//   d_u z = max(-U, U - w z)              distance of the centre outside
//   d_v z = max(-V, V - h z)              [0,w] x [0,h], times z
//   in range: znear < z < zfar
//   3-sigma box meets the image  <=>  (max(d_u z, 0) z)^2 <= Qx  and
//                                     (max(d_v z, 0) z)^2 <= Qy
//     with g0 = z P0 - U P2, g1 = z P1 - V P2 (the rows of z^2 J W) and
//     Qx = |L g0|^2 = 9 z^4 S_xx, Qy = |L g1|^2 = 9 z^4 S_yy, L = 3 diag(s)
//     R(q)^T, i.e. Sigma2D = J W Sigma W^T J^T formed through the square
//     root of Sigma (well conditioned in float).
//   det Sigma2D = |L g0 x L g1|^2 / (81 z^8) > 0 whenever all three scales
//     are nonzero (L invertible, g0 and g1 independent); a warp holding a
//     primitive with an underflowed scale evaluates it on every pair.
//   term = vis / (z^2 + eta)              (Eq. 17, one MUFU reciprocal)
//
// Work is skipped only where the outcome is already implied, so every
// decision equals the full test's, bit for bit:
//  * per tile (the bounding box of its centres) and view, a lane classifies
//    one view (32 views at a time) with interval bounds of the linear forms z,
//    U, V, U - w z and V - h z over the box, widened by a slack that covers
//    float32 rounding (2^-17 of the largest magnitude for z, 2^-16 for the
//    others; classify):
//      IN   every centre is in range and inside the image: vis = 1 for all
//      OUT  every centre is out of range, or outside an image edge by more
//           than the footprint bound: vis = 0, the view is skipped
//      MIXED otherwise: decided pair by pair, on the axes left open;
//  * pair by pair (mixed_view) a centre inside the image is visible whatever
//    Sigma2D, and one outside is tested against the footprint bound, d_u <=
//    3 s_max K with the tile's K, or d_u (z - 3 s_max) <= 3 s_max E z with the
//    depth range open (classify; s_max inflated by 2^-11, K and E by 2^-8).
//    Only a pair within it needs Qx and Qy: a warp-uniform stage per axis,
//    entered when some lane does.
// Views are summed in blocks of 32, in view order (an invisible or skipped
// view adds +0, which changes nothing), and the block sums are added to the
// primitive's total with Kahan compensation, so a primitive's sum does not
// depend on the tile it is in and its rounding error does not grow with V.
// The epilogue forms D_i = alpha_i S_i / |V| * sum_k lambda^k G~_i^k (Eq. 7).
// ---------------------------------------------------------------------
// Floor of PairIn::s3: with it, and E > 1e-3 and z > 1e-6 (classify), s3 K is
// above every du whose (du z)^2 underflows, which the exact test would pass.
constexpr float kMinS3 = 1e-12f;
// From here on the square of du z may be infinite, which the exact test passes
// when its other side is too: the footprint bound then excludes nothing.
constexpr float kMaxDz = 1e18f;

struct PairIn {
    float mx, my, mz;
    float L[9];
    float s3;  // 3 s_max (1 + 2^-11), the square root of the record's footprint bound factor
};

struct __align__(16) TileBox {
    float cx, cy, cz;  // centre of the box of the tile's centres
    float hx, hy, hz;  // half extents
    float l1;          // sum over the axes of |centre| + half extent (magnitude bound)
    float s3;          // max over the tile of PairIn::s3
};

// A warp's shared-memory slot.  The tile box lives there while the tile's
// views are scored and is read back for each classification, so that it
// holds no registers across the view loop (the loads are volatile: never
// hoisted); k holds the footprint reach (classify) of the 32 views being
// scored, one per classifying lane; run holds every lane's running (sum,
// compensation) of its primitives, touched once in 32 views.
struct __align__(16) WarpSlot {
    TileBox box;
    float2 k[32];
    float2 run[2][32];
};

__device__ __forceinline__ TileBox load_box(const TileBox *s)
{
    TileBox t;
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(s);
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(t.cx), "=f"(t.cy), "=f"(t.cz), "=f"(t.hx) : "r"(a));
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(t.hy), "=f"(t.hz), "=f"(t.l1), "=f"(t.s3) : "r"(a + 16));
    return t;
}

struct Range {
    float lo, hi;
};

// [lo, hi] of a . mu + a0 over the tile box, widened by the slack sl.
__device__ __forceinline__ Range form_range(const float4 &a, const TileBox &t, float sl)
{
    const float mid = fmaf(a.x, t.cx, fmaf(a.y, t.cy, fmaf(a.z, t.cz, a.w)));
    const float rad = fmaf(fabsf(a.x), t.hx, fmaf(fabsf(a.y), t.hy, fmaf(fabsf(a.z), t.hz, sl)));
    return {mid - rad, mid + rad};
}

// Class of one view for one tile: kClsMixed, kClsIn or kClsOut in the low two
// bits; for MIXED also the axes whose test some centre of the tile may fail
// (kAxX: 0 < u < w, kAxY: 0 < v < h, kAxZ: znear < z < zfar) above them.  An
// axis that is not flagged holds for every centre of the tile, with the same
// float32 slack as the IN class, so a pair's test on it needs no evaluation.
//
// The slack of a range is at least 8 times the float32 rounding of its form
// evaluated pair by pair plus that of the range itself (together under 14 x
// 2^-24 of the sum of the terms' magnitudes, counted operation by operation).
// One slack serves U, V, U - w z and V - h z of a camera: 2^-16 times (its
// largest coefficient or w |R2| x the tile's l1 + its largest constant or w
// |t2|), twice the largest magnitude at 2^-17.
//
// The footprint bound.  The exact test passes an extent only if du^2 <= 9
// s_max^2 (fx^2 + (u - cx)^2), as |g0|^2 = fx^2 (x^2 + z^2).  Outside the image
// by du = max(-U, U - w z) > 0, |u - cx| <= e + du / z with e the larger
// distance of an edge from cx, so with E = sqrt(fx^2 + e^2)
//   du <= 3 s_max (E + du / z),  i.e.  du (z - s3) <= s3 E z,  s3 = 3 s_max,
// and over a box with z >= z_lo: du <= s3 K, K = min(E z_lo / (z_lo - max s3)
// (if z_lo > max s3), E + max du / z_lo).  *reach (MIXED) is (Kx, Ky), infinite
// (nothing is excluded) where a square of the exact test could overflow or
// underflow; with the depth range open (Ex, Ey), infinite where one could
// overflow.
enum { kClsMixed = 0, kClsIn = 1, kClsOut = 2 };
enum { kAxX = 4, kAxY = 8, kAxZ = 16 };

__device__ __forceinline__ float4 edge_form(const float4 &a, const float4 &c2, float w)
{
    return make_float4(fmaf(-w, c2.x, a.x), fmaf(-w, c2.y, a.y), fmaf(-w, c2.z, a.z), fmaf(-w, c2.w, a.w));
}

__device__ __forceinline__ int classify(const CamRec &c, const TileBox &t, float2 *reach)
{
    const float4 c2 = c.r2, lim = c.lim;
    const float zmax = fmaxf(fabsf(c2.x), fmaxf(fabsf(c2.y), fabsf(c2.z)));
    const Range z = form_range(c2, t, kTileSlack * fmaf(zmax, t.l1, fabsf(c2.w)));
    if (z.hi < lim.z || z.lo > lim.w) return kClsOut;
    const float4 k = c.k, c0 = c.r0, c1 = c.r1;
    const float sl = fmaf(k.z, t.l1, k.w);
    const Range U = form_range(c0, t, sl), V = form_range(c1, t, sl);
    const Range UW = form_range(edge_form(c0, c2, lim.x), t, sl), VH = form_range(edge_form(c1, c2, lim.y), t, sl);
    const bool zin = z.lo > lim.z && z.hi < lim.w;
    const bool xin = U.lo > 0.f && UW.hi < 0.f, yin = V.lo > 0.f && VH.hi < 0.f;
    if (zin && xin && yin) return kClsIn;
    const int mixed = kClsMixed | (xin ? 0 : kAxX) | (yin ? 0 : kAxY) | (zin ? 0 : kAxZ);
    const float dx = fmaxf(-U.lo, UW.hi), dy = fmaxf(-V.lo, VH.hi);  // largest du, dv of the box
    const float zs = z.lo - t.s3;
    const float iz = rcp_approx_ftz(z.lo), q = zs > 0.f ? z.lo * rcp_approx_ftz(zs) : INFINITY;
    const bool finite = fmaxf(dx, dy) * z.hi < kMaxDz;
    const bool safe = z.lo > 1e-6f && fminf(k.x, k.y) > 1e-3f && finite;
    const float kx = safe ? fminf(k.x * q, fmaf(fmaxf(dx, 0.f), iz, k.x)) * 1.00390625f : INFINITY;
    const float ky = safe ? fminf(k.y * q, fmaf(fmaxf(dy, 0.f), iz, k.y)) * 1.00390625f : INFINITY;
    const bool edge = !zin & finite;  // (kx and ky are infinite when not finite)
    *reach = make_float2(edge ? k.x : kx, edge ? k.y : ky);
    // the whole box beyond an edge by more than the reach of its largest primitive
    if (fmaxf(-U.hi, UW.lo) > t.s3 * kx || fmaxf(-V.hi, VH.lo) > t.s3 * ky) return kClsOut;
    return mixed;
}

// Projection term of a visible (primitive, view) pair.  PM (projection
// mode): 0 = Eq. 17, 1/(z^2 + eta); 1 = Table 3 "w/o P", 1; 2 = Eq. 14 before
// the simplification of Eq. 16, the Jacobian energy Tr(J^T J) = (fx^2 +
// fy^2)/z^2 + ((fx x)^2 + (fy y)^2)/z^4, with fx x and fy y from the camera's
// fx R0 and fy R1 rows (the same arithmetic on every path, so the weight does
// not depend on the tile's classification).
template <int PM>
__device__ __forceinline__ float weight(const CamExt *e, float z, float eta, float mx, float my, float mz)
{
    if (PM == kProjNone) return 1.f;
    // z^2 + eta >= eta >= 2^-126 (checked on the host), so the operand is
    // never subnormal; weights below 2^-126 (z beyond 9.2e18) flush to zero
    if (PM == kProjEq17) return rcp_approx_ftz(fmaf(z, z, eta));
    const float4 tx = e->tx, ty = e->ty, k = e->f;
    const float fxx = fmaf(tx.x, mx, fmaf(tx.y, my, fmaf(tx.z, mz, tx.w)));
    const float fyy = fmaf(ty.x, mx, fmaf(ty.y, my, fmaf(ty.z, mz, ty.w)));
    // explicit rounding intrinsics: never contracted into a neighbouring
    // add, so every path (IN, MIXED, plain, batched) rounds identically
    const float iz2 = rcp_approx(__fmul_rn(z, z));
    return __fmul_rn(fmaf(fmaf(fxx, fxx, __fmul_rn(fyy, fyy)), iz2, __fadd_rn(k.x, k.y)), iz2);
}

// A view of a tile that holds an underflowed scale: every pair in the depth
// range runs the whole test, the determinant included.
template <int PM, bool COUNT, int GPT>
__device__ __forceinline__ void mixed_view_det(const CamRec &c, const CamExt *e, float eta, const PairIn (&p)[GPT],
                                               const bool (&valid)[GPT], float (&part)[GPT],
                                               unsigned long long (&cnt)[kCountSlots])
{
    const float4 c0 = c.r0, c1 = c.r1, c2 = c.r2, lim = c.lim;
#pragma unroll
    for (int g = 0; g < GPT; ++g) {
        const float U = fmaf(c0.x, p[g].mx, fmaf(c0.y, p[g].my, fmaf(c0.z, p[g].mz, c0.w)));
        const float V = fmaf(c1.x, p[g].mx, fmaf(c1.y, p[g].my, fmaf(c1.z, p[g].mz, c1.w)));
        const float z = fmaf(c2.x, p[g].mx, fmaf(c2.y, p[g].my, fmaf(c2.z, p[g].mz, c2.w)));
        const float du = fmaxf(-U, fmaf(-lim.x, z, U)), dv = fmaxf(-V, fmaf(-lim.y, z, V));
        const bool inz = (z > lim.z) & (z < lim.w);
        const float ex = fmaxf(du, 0.f) * z, ey = fmaxf(dv, 0.f) * z;
        const float ex2 = ex * ex, ey2 = ey * ey;
        const float g0x = fmaf(-U, c2.x, z * c0.x), g0y = fmaf(-U, c2.y, z * c0.y), g0z = fmaf(-U, c2.z, z * c0.z);
        const float g1x = fmaf(-V, c2.x, z * c1.x), g1y = fmaf(-V, c2.y, z * c1.y), g1z = fmaf(-V, c2.z, z * c1.z);
        const float a0 = fmaf(p[g].L[0], g0x, fmaf(p[g].L[1], g0y, p[g].L[2] * g0z));
        const float a1 = fmaf(p[g].L[3], g0x, fmaf(p[g].L[4], g0y, p[g].L[5] * g0z));
        const float a2 = fmaf(p[g].L[6], g0x, fmaf(p[g].L[7], g0y, p[g].L[8] * g0z));
        const float b0 = fmaf(p[g].L[0], g1x, fmaf(p[g].L[1], g1y, p[g].L[2] * g1z));
        const float b1 = fmaf(p[g].L[3], g1x, fmaf(p[g].L[4], g1y, p[g].L[5] * g1z));
        const float b2 = fmaf(p[g].L[6], g1x, fmaf(p[g].L[7], g1y, p[g].L[8] * g1z));
        const float Qx = fmaf(a0, a0, fmaf(a1, a1, a2 * a2));
        const float Qy = fmaf(b0, b0, fmaf(b1, b1, b2 * b2));
        const float x0 = a1 * b2 - a2 * b1, x1 = a2 * b0 - a0 * b2, x2 = a0 * b1 - a1 * b0;
        const bool vis = inz & (ex2 <= Qx) & (ey2 <= Qy) & ((x0 != 0.f) | (x1 != 0.f) | (x2 != 0.f));
        part[g] += vis ? weight<PM>(e, z, eta, p[g].mx, p[g].my, p[g].mz) : 0.f;
        if (COUNT && valid[g]) {
            const bool o = inz & !((du <= 0.f) & (dv <= 0.f));
            cnt[kCntMixedPairs] += 1;
            cnt[kCntOpenX] += 1;
            cnt[kCntOpenY] += 1;
            cnt[kCntOpenZ] += 1;
            cnt[kCntBoundPairs] += o ? 1 : 0;
            cnt[kCntBoundX] += o ? 1 : 0;
            cnt[kCntBoundY] += o ? 1 : 0;
            cnt[kCntExactPairs] += inz ? 1 : 0;
            cnt[kCntExactX] += inz ? 1 : 0;
            cnt[kCntExactY] += inz ? 1 : 0;
            cnt[kCntVisMixed] += vis ? 1 : 0;
        }
        if (COUNT && (threadIdx.x & 31) == 0) cnt[kCntExactWarpAxes] += 2;
    }
}

// One extent of the exact footprint test: |L g|^2 with g = z r - W c2 (r the
// camera row of U or V, W its value).
__device__ __forceinline__ float extent2(const float4 &r, const float4 &c2, float W, float z, const PairIn &p)
{
    const float gx = fmaf(-W, c2.x, z * r.x), gy = fmaf(-W, c2.y, z * r.y), gz = fmaf(-W, c2.z, z * r.z);
    const float a0 = fmaf(p.L[0], gx, fmaf(p.L[1], gy, p.L[2] * gz));
    const float a1 = fmaf(p.L[3], gx, fmaf(p.L[4], gy, p.L[5] * gz));
    const float a2 = fmaf(p.L[6], gx, fmaf(p.L[7], gy, p.L[8] * gz));
    return fmaf(a0, a0, fmaf(a1, a1, a2 * a2));
}

// A MIXED view of a tile without underflowed scales, evaluated only on the
// axes its classification left open (NX: 0 < u < w, NY: 0 < v < h, NZ: the
// depth range); an axis that holds for every centre of the tile contributes
// d = 0 to the box test, which it then passes for every Sigma2D, so leaving
// it out changes no decision.  First the centre test and, for centres
// outside, a footprint bound; then the exact footprint test, entered per
// primitive slot g and per axis only when some lane of the warp needs it (a
// lane whose bound failed, or whose centre lies within that axis's interval,
// fails or passes it without evaluation).
//
// The bound (classify) with the depth range closed: du <= s3 Kx, the tile's
// reach, one multiply and one compare a pair; with the depth range open a pair
// forms its own, du (z - s3) <= s3 E z.  Both exclude only pairs that the exact
// test fails.
template <int PM, bool COUNT, int GPT, bool NX, bool NY, bool NZ>
__device__ __forceinline__ void mixed_view(const CamRec &c, const CamExt *e, const float2 &reach, float eta, const PairIn (&p)[GPT],
                                           const bool (&valid)[GPT], float (&part)[GPT],
                                           unsigned long long (&cnt)[kCountSlots])
{
    const float4 c2 = c.r2, lim = c.lim;
    const float2 K = reach;
    float z[GPT], U[GPT], V[GPT], du[GPT], dv[GPT];
    bool vis[GPT], nq[GPT];
#pragma unroll
    for (int g = 0; g < GPT; ++g) {
        z[g] = fmaf(c2.x, p[g].mx, fmaf(c2.y, p[g].my, fmaf(c2.z, p[g].mz, c2.w)));
        const bool inz = NZ ? (z[g] > lim.z) & (z[g] < lim.w) : true;
        bool inside = inz, reaches = inz;
        if (NX) {
            const float4 c0 = c.r0;
            U[g] = fmaf(c0.x, p[g].mx, fmaf(c0.y, p[g].my, fmaf(c0.z, p[g].mz, c0.w)));
            du[g] = fmaxf(-U[g], fmaf(-lim.x, z[g], U[g]));
            inside &= du[g] <= 0.f;
            if (!NZ) reaches &= du[g] <= p[g].s3 * K.x;
        }
        if (NY) {
            const float4 c1 = c.r1;
            V[g] = fmaf(c1.x, p[g].mx, fmaf(c1.y, p[g].my, fmaf(c1.z, p[g].mz, c1.w)));
            dv[g] = fmaxf(-V[g], fmaf(-lim.y, z[g], V[g]));
            inside &= dv[g] <= 0.f;
            if (!NZ) reaches &= dv[g] <= p[g].s3 * K.y;
        }
        if (NZ) {
            const float zs = z[g] - p[g].s3, t = p[g].s3 * z[g] * 1.00390625f;
            reaches &= (du[g] * zs <= K.x * t) & (dv[g] * zs <= K.y * t);
        }
        vis[g] = inside;
        nq[g] = !inside & reaches;
        if (COUNT && valid[g]) {
            const bool o = inz & !inside;
            cnt[kCntMixedPairs] += 1;
            cnt[kCntOpenX] += NX ? 1 : 0;
            cnt[kCntOpenY] += NY ? 1 : 0;
            cnt[kCntOpenZ] += NZ ? 1 : 0;
            cnt[kCntBoundPairs] += o ? 1 : 0;
            cnt[kCntBoundX] += (NX && o) ? 1 : 0;
            cnt[kCntBoundY] += (NY && o) ? 1 : 0;
            cnt[kCntExactPairs] += nq[g] ? 1 : 0;
            cnt[kCntExactX] += (NX && nq[g] && du[g] > 0.f) ? 1 : 0;
            cnt[kCntExactY] += (NY && nq[g] && dv[g] > 0.f) ? 1 : 0;
        }
    }
    // with one axis open, a centre outside is outside on that axis
    constexpr bool kOne = NX != NY;
#pragma unroll
    for (int g = 0; g < GPT; ++g) {
        bool ok = nq[g];
        if (NX && __any_sync(0xffffffffu, kOne ? nq[g] : nq[g] & (du[g] > 0.f))) {
            const float ex = (kOne ? du[g] : fmaxf(du[g], 0.f)) * z[g];
            ok &= ex * ex <= extent2(c.r0, c2, U[g], z[g], p[g]);
            if (COUNT && (threadIdx.x & 31) == 0) cnt[kCntExactWarpAxes] += 1;
        }
        if (NY && __any_sync(0xffffffffu, kOne ? nq[g] : nq[g] & (dv[g] > 0.f))) {
            const float ey = (kOne ? dv[g] : fmaxf(dv[g], 0.f)) * z[g];
            ok &= ey * ey <= extent2(c.r1, c2, V[g], z[g], p[g]);
            if (COUNT && (threadIdx.x & 31) == 0) cnt[kCntExactWarpAxes] += 1;
        }
        vis[g] |= ok;
    }
#pragma unroll
    for (int g = 0; g < GPT; ++g) {
        part[g] += vis[g] ? weight<PM>(e, z[g], eta, p[g].mx, p[g].my, p[g].mz) : 0.f;
        if (COUNT) cnt[kCntVisMixed] += (valid[g] && vis[g]) ? 1 : 0;
    }
}

// Kahan-compensated sum of the 32-view block sums.
__device__ __forceinline__ void kahan_add(float2 &run, float x)
{
    const float2 r = run;
    const float y = x - r.y;
    const float t = r.x + y;
    run = make_float2(t, (t - r.x) - y);
}

// Views [v0, vend) of the pass (v0 a multiple of 32) for one tile: added to
// the slot's running sums, or with pp their block sums stored at pp.  take_next() runs
// once, before the last block.
template <int PM, bool DET, bool COUNT, int GPT, typename F>
__device__ __forceinline__ void view_loop(const CamRec *cs, const CamExt *ce, int v0, int vend, float *pp, float eta,
                                          const PairIn (&p)[GPT], const bool (&valid)[GPT], WarpSlot *slot, F &&take_next,
                                          unsigned long long (&cnt)[kCountSlots])
{
    const int lane = threadIdx.x & 31;
    int nvalid = 0;
#pragma unroll
    for (int g = 0; g < GPT; ++g) nvalid += __popc(__ballot_sync(0xffffffffu, valid[g]));
    for (int vb = v0; vb < vend; vb += 32) {
        const int nv = min(32, vend - vb);
        if (vb + 32 >= vend) take_next();
        const unsigned vmask = nv == 32 ? 0xffffffffu : ((1u << nv) - 1u);
        unsigned in_m = 0u, out_m = 0u, ux_m = 0u, uy_m = 0u, uz_m = 0u;
        if (!DET) {
            const TileBox tb = load_box(&slot->box);
            float2 reach = make_float2(0.f, 0.f);
            const int cls = lane < nv ? classify(cs[vb + lane], tb, &reach) : (kAxX | kAxY | kAxZ);
            __syncwarp();  // every lane is done with the reaches of the views before
            slot->k[lane] = reach;
            __syncwarp();
            in_m = __ballot_sync(0xffffffffu, (cls & 3) == kClsIn);
            out_m = __ballot_sync(0xffffffffu, (cls & 3) == kClsOut);
            ux_m = __ballot_sync(0xffffffffu, (cls & kAxX) != 0);
            uy_m = __ballot_sync(0xffffffffu, (cls & kAxY) != 0);
            uz_m = __ballot_sync(0xffffffffu, (cls & kAxZ) != 0);
            if (COUNT && lane == 0) {
                cnt[kCntTiles] += nv;
                cnt[kCntInPairs] += (unsigned long long)__popc(in_m & vmask) * nvalid;
                cnt[kCntOutPairs] += (unsigned long long)__popc(out_m & vmask) * nvalid;
            }
        }
        {
            float part[GPT];
#pragma unroll
            for (int g = 0; g < GPT; ++g) part[g] = 0.f;
            // the single open axes first among the MIXED views: most of them
            const unsigned x_m = ux_m & ~uy_m & ~uz_m, y_m = uy_m & ~ux_m & ~uz_m;
            unsigned todo = vmask & ~out_m;
            while (todo) {
                const unsigned bit = todo & (0u - todo);
                const int b = 31 - __clz(bit);
                todo ^= bit;
                const CamRec &c = cs[vb + b];
                const CamExt *ext = PM == kProjFullJ ? ce + vb + b : nullptr;
                if (in_m & bit) {
                    const float4 c2 = c.r2;
#pragma unroll
                    for (int g = 0; g < GPT; ++g) {
                        const float z = fmaf(c2.x, p[g].mx, fmaf(c2.y, p[g].my, fmaf(c2.z, p[g].mz, c2.w)));
                        part[g] += weight<PM>(ext, z, eta, p[g].mx, p[g].my, p[g].mz);
                    }
                } else if (DET) {
                    mixed_view_det<PM, COUNT, GPT>(c, ext, eta, p, valid, part, cnt);
                } else {
                    const float2 &reach = slot->k[b];
                    if (y_m & bit)
                        mixed_view<PM, COUNT, GPT, false, true, false>(c, ext, reach, eta, p, valid, part, cnt);
                    else if (x_m & bit)
                        mixed_view<PM, COUNT, GPT, true, false, false>(c, ext, reach, eta, p, valid, part, cnt);
                    else if (uz_m & bit)
                        mixed_view<PM, COUNT, GPT, true, true, true>(c, ext, reach, eta, p, valid, part, cnt);
                    else
                        mixed_view<PM, COUNT, GPT, true, true, false>(c, ext, reach, eta, p, valid, part, cnt);
                }
            }
            if (pp) {  // a part of the tile's views: its block sums are added by the tile's last item
#pragma unroll
                for (int g = 0; g < GPT; ++g) pp[(vb >> 5) * (32 * GPT) + g * 32 + lane] = part[g];
            } else {
#pragma unroll
                for (int g = 0; g < GPT; ++g) kahan_add(slot->run[g][lane], part[g]);
            }
        }
    }
}

// Smallest and largest value of the warp (one instruction each on sm_103a;
// a NaN is passed over).
__device__ __forceinline__ float warp_min(float v)
{
    float r;
    asm volatile("redux.sync.min.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ float warp_max(float v)
{
    float r;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ void prefetch_l2(const void *p)
{
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// Scores one warp tile: the 32 * GPT primitives of the processing order
// starting at `base`; `take_next` runs before the last block of views (the
// warp draws its next item there).  `slot` is the warp's shared-memory slot.
//
// With `tp.parts` the item is only the views [tp.v0, tp.vend) of the tile: it
// stores their 32-view block sums, and whichever of the tile's tp.items items
// ends last (tp.done counts them, no waiting) adds the block sums of the pass
// in view order and finishes the tile, so the sum has the same bits as a
// whole tile's.
struct TilePart {
    int v0, vend;
    float *parts;    // the tile's block sums, [blocks of the pass][32 * GPT], or NULL for a whole tile
    unsigned *done;  // the tile's count of finished items, zero before the launch
    int items;
};

template <int PM, bool COUNT, int GPT, typename F>
__device__ __forceinline__ void score_tile(const ScoreLaunch &a, const CamRec *cs, const CamExt *ce,
                                           int64_t base, const TilePart &tp, WarpSlot *slot, F &&take_next,
                                           unsigned long long (&cnt)[kCountSlots])
{
    const int lane = threadIdx.x & 31;
    PairIn p[GPT];
    bool valid[GPT];
    bool degen = false;
    float lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY}, s3 = 0.f;
#pragma unroll
    for (int g = 0; g < GPT; ++g) {
        const int64_t j = base + g * 32 + lane;
        float4 ra = make_float4(0.f, 0.f, 0.f, 0.f), rb = ra, rc = ra, rd = ra;
        float2 run = make_float2(0.f, 0.f);
        valid[g] = j < a.n;
        if (valid[g]) {
            const int64_t i = __ldg(a.perm + j);
            const PrimRec *r = a.recs + i;
            ra = __ldg(&r->a); rb = __ldg(&r->b); rc = __ldg(&r->c); rd = __ldg(&r->d);
            if (!a.first) run = a.running[i];
        }
        slot->run[g][lane] = run;  // read and written by this lane only
        p[g].mx = ra.x; p[g].my = ra.y; p[g].mz = ra.z;
        p[g].s3 = fmaxf(sqrt_approx_ftz(fabsf(ra.w)), kMinS3);
        p[g].L[0] = rb.x; p[g].L[1] = rb.y; p[g].L[2] = rb.z; p[g].L[3] = rb.w;
        p[g].L[4] = rc.x; p[g].L[5] = rc.y; p[g].L[6] = rc.z; p[g].L[7] = rc.w;
        p[g].L[8] = rd.x;
        degen |= ra.w < 0.f;
        if (valid[g]) {
            lo[0] = fminf(lo[0], p[g].mx); hi[0] = fmaxf(hi[0], p[g].mx);
            lo[1] = fminf(lo[1], p[g].my); hi[1] = fmaxf(hi[1], p[g].my);
            lo[2] = fminf(lo[2], p[g].mz); hi[2] = fmaxf(hi[2], p[g].mz);
            s3 = fmaxf(s3, p[g].s3);
        }
    }
    if (!__any_sync(0xffffffffu, valid[0])) return;  // warp past the end

    {
        const float l0 = warp_min(lo[0]), l1 = warp_min(lo[1]), l2 = warp_min(lo[2]);
        const float h0 = warp_max(hi[0]), h1 = warp_max(hi[1]), h2 = warp_max(hi[2]);
        const float ts3 = warp_max(s3);
        __syncwarp();  // every lane is done with the previous tile's box
        if (lane == 0) {
            TileBox tb;
            tb.s3 = ts3;
            tb.cx = 0.5f * (l0 + h0); tb.hx = 0.5f * (h0 - l0);
            tb.cy = 0.5f * (l1 + h1); tb.hy = 0.5f * (h1 - l1);
            tb.cz = 0.5f * (l2 + h2); tb.hz = 0.5f * (h2 - l2);
            tb.l1 = (fabsf(tb.cx) + tb.hx) + (fabsf(tb.cy) + tb.hy) + (fabsf(tb.cz) + tb.hz);
            slot->box = tb;
        }
        __syncwarp();
    }

    if (__any_sync(0xffffffffu, degen))
        view_loop<PM, true, COUNT, GPT>(cs, ce, tp.v0, tp.vend, tp.parts, a.eta, p, valid, slot, take_next, cnt);
    else
        view_loop<PM, false, COUNT, GPT>(cs, ce, tp.v0, tp.vend, tp.parts, a.eta, p, valid, slot, take_next, cnt);

    if (tp.parts) {
        __threadfence();
        __syncwarp();
        unsigned before = 0;
        if (lane == 0) before = atomicAdd(tp.done, 1u);
        if (__shfl_sync(0xffffffffu, before, 0) != (unsigned)(tp.items - 1)) return;
        __threadfence();
        for (int b = 0; b < (a.vcount + 31) >> 5; ++b)
#pragma unroll
            for (int g = 0; g < GPT; ++g) kahan_add(slot->run[g][lane], __ldcg(tp.parts + b * (32 * GPT) + g * 32 + lane));
    }

#pragma unroll
    for (int g = 0; g < GPT; ++g) {
        if (!valid[g]) continue;
        const int64_t i = __ldg(a.perm + base + g * 32 + lane);
        const float2 run = slot->run[g][lane];
        if (!a.last) {
            a.running[i] = run;
            continue;
        }
        const float Ssum = run.x - run.y;
        if (a.view_sum) a.view_sum[i] = Ssum;
        const float4 rd = __ldg(&a.recs[i].d);  // (L8, alpha, m_gem, m_col)
        const SceneConsts sc = *a.consts;       // read here: no registers across the views
        const float coupled = fmaf(sc.kappa[0], rd.z, fmaf(sc.kappa[1], rd.w, sc.kappa[2] * rd.y));
        const float A = ((a.flags & REFINE_FLAG_NO_VIS) ? 1.f : rd.y) * (Ssum * a.inv_views);
        a.scores[i] = A * coupled;
    }
}

// A camera block may be staged by bulk copies only if its sources are 16-byte
// aligned and it fits the launch's dynamic shared memory.
__device__ __forceinline__ int cams_stageable(const ScoreLaunch &a)
{
    uint32_t dyn;
    asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(dyn));
    const bool full_j = proj_mode(a.flags) == kProjFullJ;
    return a.vcount >= 1 && (reinterpret_cast<uintptr_t>(a.cams) & 15u) == 0 &&
           (!full_j || (a.ext != nullptr && (reinterpret_cast<uintptr_t>(a.ext) & 15u) == 0)) &&
           (uint64_t)cams_smem(a.vcount, a.flags) <= (uint64_t)dyn;
}

__device__ __forceinline__ void bulk_g2s_chunks(unsigned char *dst, const void *src, uint32_t bytes, uint64_t *bar)
{
    for (uint32_t off = 0; off < bytes; off += 16384u) {
        const uint32_t len = bytes - off < 16384u ? bytes - off : 16384u;
        bulk_g2s(dst + off, static_cast<const unsigned char *>(src) + off, len, bar);
    }
}

// The camera records of a pass, then (FULL_JACOBIAN) their extensions.
__device__ __forceinline__ void stage_cams(const ScoreLaunch &a, unsigned char *smem, uint64_t *bar)
{
    const uint32_t bytes = (uint32_t)a.vcount * (uint32_t)sizeof(CamRec);
    mbar_expect_tx(bar, (uint32_t)cams_smem(a.vcount, a.flags));
    bulk_g2s_chunks(smem, a.cams, bytes, bar);
    if (proj_mode(a.flags) == kProjFullJ)
        bulk_g2s_chunks(smem + bytes, a.ext, (uint32_t)a.vcount * (uint32_t)sizeof(CamExt), bar);
}

template <int PM, bool COUNT, int GPT>
__global__ void __launch_bounds__(kScoreThreads, COUNT ? 1 : 4) k_score(ScoreLaunch a)
{
    const int64_t zero = pdl_wait();
    after(zero, a.perm);  // (the records are older than the kernel before this one)
    after(zero, a.consts);
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ WarpSlot s_slot[kScoreThreads / 32];
    CamRec *cs = reinterpret_cast<CamRec *>(smem_raw);

    // Stage this pass's cameras once per CTA (TMA bulk copy, mbarrier).
    __shared__ int s_ok;
    const CamExt *ce = reinterpret_cast<const CamExt *>(smem_raw + (size_t)a.vcount * sizeof(CamRec));
    if (threadIdx.x == 0) {
        s_ok = cams_stageable(a) && a.tiles_taken != nullptr;
        if (s_ok) {
            mbar_init(&bar, 1);
            stage_cams(a, smem_raw, &bar);
        } else {
            set_status(a.status, kEinval);
        }
    }
    __syncthreads();
    if (!s_ok) return;
    if (!mbar_wait_bounded(&bar, 0)) {
        set_status(a.status, kEtimeout);
        mbar_wait_bounded(&bar, 0);  // give the copy a second bound before leaving
        return;
    }

    unsigned long long cnt[kCountSlots];
#pragma unroll
    for (int k = 0; k < kCountSlots; ++k) cnt[k] = 0;
    // Every warp takes its own items from a counter: warps that draw cheap
    // tiles take more of them, and no warp waits for the others of its CTA.  A
    // warp draws its next item before the last block of views of the current
    // one (drawn any earlier, it could hold a whole tile back while the others
    // run out of work) and pulls that tile's records towards L2.  Tiles of
    // 32 * GPT primitives are taken from the end of the processing order, where
    // the large primitives are (the tiles with the most pairs to decide); the
    // last a.split_tiles tiles taken are split into items of kSplitViews
    // views.  Item indices stay below 2^31 (n <= INT32_MAX, and only a wave's
    // worth of tiles is split).
    const int lane = threadIdx.x & 31;
    WarpSlot *slot = &s_slot[__shfl_sync(0xffffffffu, threadIdx.x >> 5, 0)];  // a uniform address
    const int ntiles = (int)((a.n + 32 * GPT - 1) / (32 * GPT));
    const int whole = ntiles - a.split_tiles;
    const int per = a.split_tiles > 0 ? (a.vcount + kSplitViews - 1) / kSplitViews : 1;
    const int items = whole + a.split_tiles * per;
    auto draw = [&]() {
        int i = 0;
        if (lane == 0) i = (int)min((unsigned long long)items, atomicAdd(a.tiles_taken, 1ull));
        return __shfl_sync(0xffffffffu, i, 0);
    };
    auto tile_of = [&](int i) { return ntiles - 1 - (i < whole ? i : whole + (i - whole) / per); };
    for (int cur = draw(); cur < items;) {
        const int tile = tile_of(cur);
        TilePart tp = {0, a.vcount, nullptr, nullptr, 1};
        if (cur >= whole) {  // here tile = ntiles - 1 - whole - (cur - whole) / per, in [0, split_tiles)
            const int k = (cur - whole) % per, blocks = (a.vcount + 31) >> 5;
            tp = {k * kSplitViews, min(a.vcount, (k + 1) * kSplitViews),
                  a.parts + (size_t)tile * blocks * (32 * GPT), a.parts_done + tile, per};
        }
        int nxt = 0;
        auto take_next = [&]() {
            nxt = draw();
            if (nxt >= items || tile_of(nxt) == tile) return;
#pragma unroll
            for (int g = 0; g < GPT; ++g) {
                const int64_t j = (int64_t)tile_of(nxt) * (32 * GPT) + g * 32 + lane;
                if (j < a.n) prefetch_l2(a.recs + __ldg(a.perm + j));
            }
        };
        score_tile<PM, COUNT, GPT>(a, cs, ce, (int64_t)tile * (32 * GPT), tp, slot, take_next,
                                   cnt);
        cur = nxt;
    }
    if (COUNT) {
#pragma unroll
        for (int k = 0; k < kCountSlots; ++k) {
            unsigned long long v = cnt[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
            if (lane == 0 && v) atomicAdd(&a.need[k], v);
        }
    }
}

// The scene that a CTA of the batched kernel is scoring, in shared memory.
struct __align__(8) BatchScene {
    ScoreLaunch a;
    unsigned *next;  // tiles drawn so far
    unsigned tiles;
};

// The scene's tiles for the warps of the CTA: each draws its next tile from
// the scene's counter before the last view block of the current one, as in
// k_score.
template <int PM, int GPT>
__device__ __forceinline__ void score_scene(const BatchScene &sc, const CamRec *cs, WarpSlot *slot)
{
    const int lane = threadIdx.x & 31;
    const ScoreLaunch &a = sc.a;
    unsigned long long cnt[kCountSlots];  // not counted
    auto draw = [&]() {
        unsigned t = 0;
        if (lane == 0) t = atomicAdd(sc.next, 1u);
        return __shfl_sync(0xffffffffu, t, 0);
    };
    for (unsigned cur = draw(); cur < sc.tiles;) {
        unsigned nxt = 0;
        auto take_next = [&]() {
            nxt = draw();
            if (nxt >= sc.tiles) return;
#pragma unroll
            for (int g = 0; g < GPT; ++g) {
                const int64_t j = (int64_t)(sc.tiles - 1 - nxt) * (32 * GPT) + g * 32 + lane;
                if (j < a.n) prefetch_l2(a.recs + __ldg(a.perm + j));
            }
        };
        const CamExt *ce = PM == kProjFullJ ? reinterpret_cast<const CamExt *>(cs + a.vcount) : nullptr;
        const TilePart tp = {0, a.vcount, nullptr, nullptr, 1};
        score_tile<PM, false, GPT>(a, cs, ce, (int64_t)(sc.tiles - 1 - cur) * (32 * GPT), tp, slot, take_next, cnt);
        cur = nxt;
    }
}

// The batched form: one persistent launch over the tiles of many scenes.  A
// CTA stays with a scene, its cameras staged once by TMA, while the scene has
// tiles left: its warps draw them one by one, with no barrier in between, and
// the CTAs' first scenes are dealt in proportion to their work (tiles x
// views).  Then it goes on to the next scene that has tiles left.  So a CTA
// meets barriers a few times a launch, where items of up to 32 tiles had its
// warps wait for the slowest at every item's end: 12 scenes of 0.09-1.9M
// primitives (bfloat16, 81-298 views) 1.55 -> 1.36 ms a score launch.
// Every tile is scored by score_tile exactly as in k_score, so a scene's
// scores are the same alone and in a batch; scenes may differ in storage type
// (the records are float32) and in flags.  PM: the projection mode when every
// scene has the Eq. 17 one (the other two's code would cost registers), or
// kProjAny.
constexpr int kProjAny = -1;

template <int PM, int GPT, int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) k_score_batch(BatchLaunch b)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ __align__(8) uint64_t bar;
    __shared__ BatchScene s_sc;
    __shared__ int s_first, s_off, s_ok;
    __shared__ WarpSlot s_slot[THREADS / 32];
    CamRec *cs = reinterpret_cast<CamRec *>(smem_raw);
    WarpSlot *slot = &s_slot[__shfl_sync(0xffffffffu, threadIdx.x >> 5, 0)];  // a uniform address
    if (threadIdx.x == 0) {
        mbar_init(&bar, 1);
        const long long at = (long long)((double)b.work[b.n_scenes] * (blockIdx.x + 0.5) / gridDim.x);
        int lo = 0, hi = b.n_scenes - 1;  // last scene whose work begins at or before this CTA's share
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if (b.work[mid] <= at) lo = mid; else hi = mid - 1;
        }
        s_first = lo;
    }
    __syncthreads();
    int scene = s_first;
    uint32_t phase = 0;
    for (;;) {
        // the nearest scene from here on that has tiles left
        if (threadIdx.x == 0) s_off = b.n_scenes;
        __syncthreads();
        for (int k = threadIdx.x; k < b.n_scenes; k += THREADS) {
            const int s = scene + k < b.n_scenes ? scene + k : scene + k - b.n_scenes;
            if ((int64_t)__ldcg(b.next + s) * (32 * GPT) < b.scenes[s].n) {
                atomicMin(&s_off, k);
                break;
            }
        }
        __syncthreads();
        if (s_off >= b.n_scenes) break;  // every tile of every scene has been drawn
        scene = scene + s_off < b.n_scenes ? scene + s_off : scene + s_off - b.n_scenes;
        for (int k = threadIdx.x; k < (int)(sizeof(ScoreLaunch) / 8); k += THREADS)
            reinterpret_cast<uint64_t *>(&s_sc.a)[k] = reinterpret_cast<const uint64_t *>(b.scenes + scene)[k];
        __syncthreads();
        const ScoreLaunch &a = s_sc.a;
        if (threadIdx.x == 0) {
            s_sc.next = b.next + scene;
            s_sc.tiles = (unsigned)((a.n + 32 * GPT - 1) / (32 * GPT));
            s_ok = cams_stageable(a);
            if (s_ok) {
                fence_proxy_async_shared();
                stage_cams(a, smem_raw, &bar);
            } else {
                set_status(a.status, kEinval);
                atomicMax(b.next + scene, 0x7fffffffu);  // the scene is left unscored
            }
        }
        __syncthreads();
        if (!s_ok) continue;
        if (!mbar_wait_bounded(&bar, phase)) {
            // the tiles left unscored belong to this scene: its own status
            // word carries the error, and so does the launch's
            set_status(a.status, kEtimeout);
            set_status(b.status, kEtimeout);
            mbar_wait_bounded(&bar, phase);
            return;
        }
        phase ^= 1u;
        const int pm = PM == kProjAny ? proj_mode(a.flags) : PM;
        if (pm == kProjEq17)
            score_scene<kProjEq17, GPT>(s_sc, cs, slot);
        else if (pm == kProjNone)
            score_scene<kProjNone, GPT>(s_sc, cs, slot);
        else
            score_scene<kProjFullJ, GPT>(s_sc, cs, slot);
        __syncthreads();  // the cameras and s_sc are free again
    }
}

// Self-test of the bounded wait that guards the camera staging above: one
// thread stages `bytes` by a bulk copy while the barrier expects `bytes +
// missing` bytes.  With missing > 0 the phase cannot complete; the wait gives
// up after `limit` cycles (long after the copy itself has landed) and the
// kernel reports kEtimeout through the status word and returns.
__global__ void k_wait_selftest(const unsigned char *src, uint32_t bytes, uint32_t missing, long long limit,
                                int *status)
{
    __shared__ __align__(16) unsigned char buf[kSelftestMaxBytes];
    __shared__ __align__(8) uint64_t bar;
    if (threadIdx.x != 0) return;
    mbar_init(&bar, 1);
    mbar_expect_tx(&bar, bytes + missing);
    bulk_g2s(buf, src, bytes, &bar);
    if (!mbar_wait_bounded(&bar, 0, limit)) {
        set_status(status, kEtimeout);
        mbar_wait_bounded(&bar, 0, limit);
    }
}

cudaError_t launch_wait_selftest(const void *src, uint32_t bytes, uint32_t missing, long long limit, int *status,
                                 cudaStream_t s)
{
    k_wait_selftest<<<1, 32, 0, s>>>(static_cast<const unsigned char *>(src), bytes, missing, limit, status);
    return cudaGetLastError();
}

using ScoreFn = void (*)(ScoreLaunch);

template <int PM, bool COUNT, int GPT>
static ScoreFn score_fn()
{
    return &k_score<PM, COUNT, GPT>;
}

template <int PM, int GPT>
static ScoreFn pick_score_pg(bool count)
{
    return count ? score_fn<PM, true, GPT>() : score_fn<PM, false, GPT>();
}

template <int GPT>
static ScoreFn pick_score_g(int pm, bool count)
{
    if (pm == kProjNone) return pick_score_pg<kProjNone, GPT>(count);
    if (pm == kProjFullJ) return pick_score_pg<kProjFullJ, GPT>(count);
    return pick_score_pg<kProjEq17, GPT>(count);
}

static ScoreFn pick_score(int pm, bool count, int gpt)
{
    return gpt == 1 ? pick_score_g<1>(pm, count) : pick_score_g<2>(pm, count);
}

bool shape_valid(const ScoreShape &sh)
{
    return (sh.gpt == 1 || sh.gpt == 2) && (sh.threads == 128 || sh.threads == 256) && sh.ctas_per_sm >= 0 &&
           sh.views_per_pass >= 32 && sh.views_per_pass <= kViewsPerPass && sh.views_per_pass % 32 == 0;
}

// Opt-in to the shared memory of a camera block.  A launch may take 48 KB
// without it, static part included (kStaticBound).  The limit set is one
// constant for every launch: the attribute belongs to the function, so a
// smaller value set for one thread's launch would refuse another's larger one.
constexpr size_t kStaticBound = 8 * 1024;
static_assert(sizeof(WarpSlot) * (kScoreThreads / 32) + 1024 <= kStaticBound, "static shared memory of the score kernels");
constexpr size_t kMaxCamsSmem = (size_t)kViewsPerPass * (sizeof(CamRec) + sizeof(CamExt));

template <class Fn>
static cudaError_t allow_cams_smem(Fn fn, size_t smem)
{
    if (smem + kStaticBound <= 48 * 1024) return cudaSuccess;
    return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxCamsSmem);
}

// Persistent grid: as many CTAs as fit per SM, capped by the items.
//
// Split tiles.  A tile's views are one serial chain of a few tens of
// microseconds, so a launch of whole tiles ends on a ragged last wave, and one
// with fewer tiles than warp slots leaves the others idle.  The last wave of
// tiles (all of them, when there are no more) is therefore split into items of
// kSplitViews = 64 views, which costs a reload of the records per item and 4
// bytes per primitive and 32 views.  Measured (k_score, whole tiles against
// the split, each with the late draw of the next item): 1M x 150 (3.2 waves of
// tiles) 189 -> 156 us, 3.5M x 250 (11 waves) 660 -> 615 us, 150k x 1100 (half
// a wave) 610 -> 288 us.  Items of 32 views: 160, 625 and 307 us; of 96: 159,
// 616 and 293 us.  Two waves split instead of one cost 2-5 us, half a wave 0-6.
// Views of one or two blocks are not split: 77k x 61 takes 28.6 us whole and
// 32 us in single blocks.
// When all the blocks of 64-primitive tiles fill less than two waves, tiles of
// 32 primitives are taken (more instructions per pair but twice the warps).
ScorePlan score_plan(int num_sms, int64_t n, int vcount, int flags, bool split, const ScoreShape &sh)
{
    ScorePlan pl;
    const size_t smem = cams_smem(vcount, flags);
    const int64_t blocks = (vcount + 31) / 32;
    pl.gpt = sh.gpt;
    int per_sm = 0;
    const ScoreFn fn = pick_score(proj_mode(flags), false, pl.gpt);
    (void)allow_cams_smem(fn, smem);
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kScoreThreads, smem) != cudaSuccess ||
        per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    constexpr int kWarps = kScoreThreads / 32;
    const int64_t slots = (int64_t)num_sms * per_sm * kWarps;
    if (split && pl.gpt == 2 && (n + 63) / 64 * blocks < 2 * slots) pl.gpt = 1;
    const int64_t tiles = (n + 32 * pl.gpt - 1) / (32 * pl.gpt);
    int64_t items = tiles;
    if (split && vcount > kSplitViews) {
        pl.split_tiles = (int)(tiles < slots ? tiles : slots);
        items += pl.split_tiles * (int64_t)((vcount - 1) / kSplitViews);
    }
    int64_t g = (int64_t)num_sms * per_sm;
    if (g > (items + kWarps - 1) / kWarps) g = (items + kWarps - 1) / kWarps;
    if (g < 1) g = 1;
    pl.grid = (int)g;
    return pl;
}

cudaError_t launch_score(const ScoreLaunch &a, int gpt, const Chain &s)
{
    const ScoreFn fn = pick_score(proj_mode(a.flags), a.need != nullptr, gpt);
    const size_t smem = cams_smem(a.vcount, a.flags);
    const cudaError_t e = allow_cams_smem(fn, smem);
    if (e != cudaSuccess) return e;
    return launch_chained(fn, a.grid, kScoreThreads, smem, s, a);
}

using BatchFn = void (*)(BatchLaunch);

template <int PM>
static BatchFn batch_fn_pm(const ScoreShape &sh)
{
    if (sh.threads == 128) return sh.gpt == 1 ? &k_score_batch<PM, 1, 128> : &k_score_batch<PM, 2, 128>;
    return sh.gpt == 1 ? &k_score_batch<PM, 1, 256> : &k_score_batch<PM, 2, 256>;
}

static BatchFn batch_fn(const ScoreShape &sh, bool eq17)
{
    return eq17 ? batch_fn_pm<kProjEq17>(sh) : batch_fn_pm<kProjAny>(sh);
}

int score_batch_grid(int num_sms, size_t smem, bool eq17, const ScoreShape &sh)
{
    const BatchFn fn = batch_fn(sh, eq17);
    (void)allow_cams_smem(fn, smem);
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, sh.threads, smem) != cudaSuccess || per_sm < 1) {
        cudaGetLastError();
        per_sm = 1;
    }
    if (sh.ctas_per_sm > 0 && sh.ctas_per_sm < per_sm) per_sm = sh.ctas_per_sm;
    return num_sms * per_sm;
}

cudaError_t launch_score_batch(const BatchLaunch &b, size_t smem, int grid, const ScoreShape &sh, cudaStream_t s)
{
    const BatchFn fn = batch_fn(sh, b.eq17);
    const cudaError_t e = allow_cams_smem(fn, smem);
    if (e != cudaSuccess) return e;
    fn<<<grid, sh.threads, smem, s>>>(b);
    return cudaGetLastError();
}

}  // namespace refine
