// O(N^2) pair passes of the GB hot path on sm_103a.
//
// Every replica's atoms are cut into 32-atom tiles.  A warp owns runs of
// blocks of the upper triangle: 64 or 128 atoms ("i", two or four a lane, one
// FP32x2 register pair per two of them) against the 32 atoms of tile J ("j"),
// which a lane meets one after the other while their FP32 partial sums rotate
// one lane per step with warp shuffles.  Each step evaluates two or four
// pairs per lane with packed FP32x2 arithmetic, and every unordered pair is
// evaluated exactly once (Newton's third law).  The tiles on the diagonal are
// masked.  After each tile the j partials are folded into int64 fixed point
// with one global atomic per atom and component; the i partials go to int64
// sums in shared memory, flushed when the task ends.  FP32 partials never span
// more than one block and integer sums are associative, so results are the
// same for every run, task split and launch order.
//
// Pass 1 (Born integrals), pass 2 (GB + Coulomb energy, direct forces, dE/dR,
// optional dE/dq and soft repulsion) and pass 3 (Born-radius chain rule)
// share the walk (walk_task).  Blocks run one of the forms under "blocks by
// distance"; the general code of pass 2 (Energy) serves blocks that straddle
// the pair cutoff and evaluations that want energies or dE/dq.
#pragma once

#include "common.cuh"
#include "internal.h"
#include "poly_coeffs.h"

namespace gbk {

// Disjoint spheres (r >= a + s) with x = s/r <= 0.6: H = 1/2 s^3 r^-4 g(x^2) and
// -(dH/dr)/r = 1/2 s^3 r^-6 h(x^2), with g, h the fitted polynomials: no
// cancellation and no MUFU.
__device__ __forceinline__ bool far_ok(float r, float lim, float y) { return (r >= lim) && (y <= GB_POLY_YMAX); }

// --- packed FP32x2 helpers ----------------------------------------------------------
typedef float2 f2;
__device__ __forceinline__ f2 F2(float v) { return make_float2(v, v); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }

// MUFU reciprocal square root and base-2 exponential; inputs here are never
// denormal, so the flush-to-zero forms need no fix-up instructions.
__device__ __forceinline__ float rsqrt_ftz(float x) {
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float ex2_ftz(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ f2 rsqrt2(f2 x) { return make_float2(rsqrt_ftz(x.x), rsqrt_ftz(x.y)); }
__device__ __forceinline__ f2 ex22(f2 x) { return make_float2(ex2_ftz(x.x), ex2_ftz(x.y)); }
// 1/sqrt(x) refined by one Newton step y (3 - x y^2) / 2
__device__ __forceinline__ f2 rsqrt2_nr(f2 x) {
    const f2 y = rsqrt2(x);
    return mul2(y, fma2(F2(-0.5f), mul2(x, mul2(y, y)), F2(1.5f)));
}

constexpr float SQRT_LOG2E = 1.2011224087864498f;  // sqrt(log2(e))
constexpr float LN2 = 0.69314718055994531f;
constexpr float LOG2E = 1.4426950408889634f;
constexpr float FAR_R2 = 1.0e30f;                  // r^2 given to masked-off lanes

__device__ __forceinline__ void set2(f2& v, int half, float x) {
    if (half) v.y = x;
    else v.x = x;
}
__device__ __forceinline__ float get2(f2 v, int half) { return half ? v.y : v.x; }
__device__ __forceinline__ f2 neg2(f2 v) { return make_float2(-v.x, -v.y); }
// Compensated summation (Kahan): sum + c carries the running total, with c
// the negated rounding error of the additions so far.
__device__ __forceinline__ void kahan_add(f2& sum, f2& c, f2 term) {
    const f2 y = add2(term, neg2(c));
    const f2 t = add2(sum, y);
    c = add2(add2(t, neg2(sum)), neg2(y));
    sum = t;
}
// Reciprocal: MUFU estimate (flush-to-zero; arguments here are O(1) lengths)
// and one Newton step y + y (1 - x y), which brings it to about half an ulp.
__device__ __forceinline__ float rcp_ftz(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ f2 rcp2(f2 x) {
    const f2 y = make_float2(rcp_ftz(x.x), rcp_ftz(x.y));
    return fma2(y, fma2(neg2(x), y, F2(1.0f)), y);
}
// the bare MUFU reciprocal (1 ulp), for the distant forms in 1/r^2
__device__ __forceinline__ f2 rcp2_approx(f2 x) { return make_float2(rcp_ftz(x.x), rcp_ftz(x.y)); }
__device__ __forceinline__ f2 logv(f2 x) { return make_float2(logf(x.x), logf(x.y)); }

// --- HCT descreening integral H(r; a, s), closed form -----------------------------
// H = (1/4pi) * volume integral of |y - x_i|^-4 over the part of the sphere
// (centre x_j, radius s) that lies outside the sphere (x_i, a).  Closed form
// from spherical shells about x_i between L = max(a, |r - s|) and U = r + s:
//   H = 1/2 [1/L - 1/U + (r - s^2/r)/4 (1/U^2 - 1/L^2) + ln(L/U) / (2r)],
// plus 1/a - 1/L inside the bracket when x_i is engulfed (a < s - r), and 0
// when sphere j lies inside sphere i (a >= r + s).  It serves only pairs whose
// spheres overlap or nearly touch (chain neighbours and contacts), where its
// O(1) terms cancel to about a tenth of their size: the reciprocals and the
// logarithm are kept to FP32 rounding.  Both pairs of a lane (x and y halves)
// are evaluated at once, branch-free.
__device__ __forceinline__ f2 hct_closed2(f2 r, f2 rinv, f2 a, f2 s) {
    const f2 U = add2(r, s);
    const f2 rs = add2(r, neg2(s));
    const f2 L = make_float2(fmaxf(a.x, fabsf(rs.x)), fmaxf(a.y, fabsf(rs.y)));
    const f2 iU = rcp2(U), iL = rcp2(L);
    const f2 dU2 = add2(mul2(iU, iU), neg2(mul2(iL, iL)));        // 1/U^2 - 1/L^2
    const f2 w = fma2(neg2(mul2(s, s)), rinv, r);                 // r - s^2/r
    f2 b = fma2(mul2(F2(0.25f), w), dU2, add2(iL, neg2(iU)));
    b = fma2(mul2(F2(0.5f), rinv), logv(mul2(L, iU)), b);        // ln(L/U) / (2r)
    const f2 eng = mul2(F2(2.0f), add2(rcp2(a), neg2(iL)));       // engulfed: 2 (1/a - 1/L)
    b.x += (a.x < -rs.x) ? eng.x : 0.0f;
    b.y += (a.y < -rs.y) ? eng.y : 0.0f;
    return make_float2(a.x >= U.x ? 0.0f : 0.5f * b.x, a.y >= U.y ? 0.0f : 0.5f * b.y);
}

// -(dH/dr) / r of the closed form, for both pairs of a lane.  With dL = dL/dr
// (0 while L = a, sign(r - s) while L = |r - s|) and w = r - s^2/r:
//   dB/dr = -dL/L^2 + 1/U^2 + (1 + s^2/r^2)/4 (1/U^2 - 1/L^2)
//           + w/2 (dL/L^3 - 1/U^3) - ln(L/U) / (2 r^2) + (dL/L - 1/U) / (2r)
// plus 2 dL/L^2 when engulfed; -(dH/dr)/r = -dB/dr / (2r).
__device__ __forceinline__ f2 hct_closed_fr2(f2 r, f2 rinv, f2 a, f2 s) {
    const f2 U = add2(r, s);
    const f2 rs = add2(r, neg2(s));
    const bool on_x = a.x > fabsf(rs.x), on_y = a.y > fabsf(rs.y);   // L = a
    const f2 L = make_float2(on_x ? a.x : fabsf(rs.x), on_y ? a.y : fabsf(rs.y));
    const f2 dL = make_float2(on_x ? 0.0f : (rs.x > 0.0f ? 1.0f : -1.0f),
                              on_y ? 0.0f : (rs.y > 0.0f ? 1.0f : -1.0f));
    const f2 iU = rcp2(U), iL = rcp2(L);
    const f2 iU2 = mul2(iU, iU), iL2 = mul2(iL, iL);
    const f2 s2r2 = mul2(mul2(s, s), mul2(rinv, rinv));           // s^2 / r^2
    const f2 w = fma2(neg2(s2r2), r, r);                          // r - s^2/r
    const f2 dLiL = mul2(dL, iL);
    f2 db = fma2(neg2(dLiL), iL, iU2);                            // -dL/L^2 + 1/U^2
    db = fma2(mul2(F2(0.25f), add2(F2(1.0f), s2r2)), add2(iU2, neg2(iL2)), db);
    db = fma2(mul2(F2(0.5f), w), add2(mul2(dLiL, iL2), neg2(mul2(iU2, iU))), db);
    const f2 hr = mul2(F2(0.5f), rinv);
    db = fma2(neg2(mul2(hr, rinv)), logv(mul2(L, iU)), db);
    db = fma2(hr, add2(dLiL, neg2(iU)), db);
    db.x += (a.x < -rs.x) ? 2.0f * dLiL.x * iL.x : 0.0f;
    db.y += (a.y < -rs.y) ? 2.0f * dLiL.y * iL.y : 0.0f;
    const f2 fr = mul2(mul2(F2(-0.5f), db), rinv);
    return make_float2(a.x >= U.x ? 0.0f : fr.x, a.y >= U.y ? 0.0f : fr.y);
}

// J(z) = int_0^z t^2/(1-t) dt = -ln(1 - z) - z - z^2/2 = z^3 q(z): the fitted series
// of positive terms of poly_coeffs.h (gb_poly_q for z <= 1/2, gb_poly_q_hi for
// z <= 3/4), and beyond that the logarithm (UL = 1 / (1 - z)), where its terms
// cancel by less than a factor 10; each range behind a warp vote over the lanes
// that use the result.
__device__ __forceinline__ f2 shell_J(f2 z, f2 UL, bool use0, bool use1) {
    const f2 z2 = mul2(z, z), z3 = mul2(z2, z);
    f2 J = mul2(z3, gb_poly_q2(z));
    if (__any_sync(0xffffffffu, (use0 && z.x > GB_POLY_ZJ) || (use1 && z.y > GB_POLY_ZJ))) {
        const f2 Jh = mul2(z3, gb_poly_q_hi2(add2(z, F2(-GB_POLY_ZMID))));
        J = make_float2(z.x > GB_POLY_ZJ ? Jh.x : J.x, z.y > GB_POLY_ZJ ? Jh.y : J.y);
        if (__any_sync(0xffffffffu, (use0 && z.x > GB_POLY_ZJ2) || (use1 && z.y > GB_POLY_ZJ2))) {
            const f2 Jl = add2(logv(UL), neg2(fma2(F2(0.5f), z2, z)));
            J = make_float2(z.x > GB_POLY_ZJ2 ? Jl.x : J.x, z.y > GB_POLY_ZJ2 ? Jl.y : J.y);
        }
    }
    return J;
}

// --- the same integral restricted to the ball |y - x_i| < rc (Born-radius cutoff) ---
// Shells about x_i now run from L to U' = min(U, rc): the bracket of
// hct_closed2 with U' in place of U when L < U' (else no shell term), and the
// engulfed part 2 (1/a - 1/min(L, rc)) when a < s - r and a < rc.  irc = 1/rc.
// With z = (U' - L) / U' the bracket is
//   { z [s^2 - (r - L)^2] / L^2 + z^2 [r^2 - L^2 - s^2] / (2 L^2) - J(z) } / (2r),
// whose terms do not cancel as 1/L - 1/U' and the logarithm do: a pair's error
// is 1.2e-7 rms of the mean integral of overlapping pairs against 3.3e-7, and
// with rgbmax = 2.6 A, where nearly every bonded pair is cut, that decides R.
// It is exact (to rounding) for every geometry: any pair may take it.
__device__ __forceinline__ f2 hct_cut2(f2 r, f2 rinv, f2 a, f2 s, float rc, float irc) {
    const f2 U = add2(r, s);
    const f2 Up = make_float2(fminf(U.x, rc), fminf(U.y, rc));
    const f2 rs = add2(r, neg2(s));
    const f2 L = make_float2(fmaxf(a.x, fabsf(rs.x)), fmaxf(a.y, fabsf(rs.y)));
    const bool in0 = L.x < Up.x, in1 = L.y < Up.y;
    const f2 iU = rcp2(Up), iL = rcp2(L), iL2 = mul2(iL, iL);
    const f2 z = mul2(add2(Up, neg2(L)), iU), J = shell_J(z, mul2(Up, iL), in0, in1);
    const f2 d = add2(r, neg2(L));
    const f2 c1 = mul2(mul2(add2(s, neg2(d)), add2(s, d)), iL2);
    const f2 c2 = mul2(fma2(d, add2(r, L), neg2(mul2(s, s))), iL2);
    f2 b = mul2(mul2(F2(0.5f), rinv), fma2(z, fma2(mul2(F2(0.5f), z), c2, c1), neg2(J)));
    b.x = in0 ? b.x : 0.0f;
    b.y = in1 ? b.y : 0.0f;
    const f2 iLc = make_float2(L.x < rc ? iL.x : irc, L.y < rc ? iL.y : irc);
    const f2 eng = mul2(F2(2.0f), add2(rcp2(a), neg2(iLc)));
    b.x += (a.x < -rs.x && a.x < rc) ? eng.x : 0.0f;
    b.y += (a.y < -rs.y && a.y < rc) ? eng.y : 0.0f;
    return mul2(F2(0.5f), b);
}

// -(dH/dr)/r of hct_cut2.  As hct_closed_fr2 with dU = dU'/dr (1 while
// U < rc, 0 once U' = rc) in the terms that came from the upper limit:
//   dB/dr = -dL/L^2 + dU/U'^2 + (1 + s^2/r^2)/4 (1/U'^2 - 1/L^2)
//           + w/2 (dL/L^3 - dU/U'^3) - ln(L/U') / (2 r^2) + (dL/L - dU/U') / (2r)
// (0 when L >= U'), plus 2 dL/L^2 when engulfed with L < rc.
// (out of line: only overlapping pairs near the cutoff take it)
static __device__ __noinline__ f2 hct_cut_fr2(f2 r, f2 rinv, f2 a, f2 s, float rc) {
    const f2 U = add2(r, s);
    const bool cx = U.x > rc, cy = U.y > rc;
    const f2 Up = make_float2(cx ? rc : U.x, cy ? rc : U.y);
    const f2 rs = add2(r, neg2(s));
    const bool on_x = a.x > fabsf(rs.x), on_y = a.y > fabsf(rs.y);
    const f2 L = make_float2(on_x ? a.x : fabsf(rs.x), on_y ? a.y : fabsf(rs.y));
    const f2 dL = make_float2(on_x ? 0.0f : (rs.x > 0.0f ? 1.0f : -1.0f),
                              on_y ? 0.0f : (rs.y > 0.0f ? 1.0f : -1.0f));
    const f2 iU = rcp2(Up), iL = rcp2(L);
    const f2 iUd = make_float2(cx ? 0.0f : iU.x, cy ? 0.0f : iU.y);   // dU / U'
    const f2 iU2 = mul2(iU, iU), iL2 = mul2(iL, iL);
    const f2 s2r2 = mul2(mul2(s, s), mul2(rinv, rinv));
    const f2 w = fma2(neg2(s2r2), r, r);
    const f2 dLiL = mul2(dL, iL);
    f2 db = fma2(neg2(dLiL), iL, mul2(iUd, iU));
    db = fma2(mul2(F2(0.25f), add2(F2(1.0f), s2r2)), add2(iU2, neg2(iL2)), db);
    db = fma2(mul2(F2(0.5f), w), add2(mul2(dLiL, iL2), neg2(mul2(iUd, iU2))), db);
    const f2 hr = mul2(F2(0.5f), rinv);
    db = fma2(neg2(mul2(hr, rinv)), logv(mul2(L, iU)), db);
    db = fma2(hr, add2(dLiL, neg2(iUd)), db);
    db.x = (L.x < Up.x) ? db.x : 0.0f;
    db.y = (L.y < Up.y) ? db.y : 0.0f;
    db.x += (a.x < -rs.x && a.x < rc && L.x < rc) ? 2.0f * dLiL.x * iL.x : 0.0f;
    db.y += (a.y < -rs.y && a.y < rc && L.y < rc) ? 2.0f * dLiL.y * iL.y : 0.0f;
    return mul2(mul2(F2(-0.5f), db), rinv);
}

// Disjoint spheres (r >= a + s) reaching past rc: the shells run from
// L = r - s to U' = min(r + s, rc), and with w = U' - L, z = w / U' the
// integral takes a form without cancelling O(1/L) terms,
//   H = 1/(4r) [ (s/L) z^2 - J(z) ].
// w is formed as min((rc - r) + s, 2s): rc - r is exact for the pairs near the
// cutoff, so w carries one rounding.  Lanes with w <= 0 (sphere j wholly past
// rc, masked lanes) give 0.
struct CutFar {
    f2 z, w, iL, iU, B;
    bool cx, cy;                      // U' = rc (the cutoff limits the shells)
};
__device__ __forceinline__ CutFar hct_cut_far_terms(f2 r, f2 s, float rc, bool use0 = true, bool use1 = true) {
    CutFar c;
    const f2 L = add2(r, neg2(s));
    c.iL = rcp2(L);
    const f2 wc = add2(add2(F2(rc), neg2(r)), s);
    const f2 s2 = add2(s, s);
    c.cx = wc.x < s2.x;
    c.cy = wc.y < s2.y;
    c.w = make_float2(fmaxf(0.0f, c.cx ? wc.x : s2.x), fmaxf(0.0f, c.cy ? wc.y : s2.y));
    const f2 U = add2(L, c.w);
    c.iU = rcp2(U);
    c.z = mul2(c.w, c.iU);
    const f2 z2 = mul2(c.z, c.z), J = shell_J(c.z, mul2(U, c.iL), use0, use1);
    c.B = fma2(mul2(s, c.iL), z2, neg2(J));
    return c;
}
__device__ __forceinline__ f2 hct_cut_far2(f2 r, f2 rinv, f2 s, float rc, bool use0, bool use1) {
    return mul2(mul2(F2(0.25f), rinv), hct_cut_far_terms(r, s, rc, use0, use1).B);
}
// -(dH/dr)/r of hct_cut_far2: with z' = -1/U' while the cutoff limits the
// shells and -z/U' otherwise (dJ/dz = z^2/(1-z), z/(1-z) = w/L),
//   dB/dr = -(s/L^2) z^2 + z' z (2s - w) / L,   dH/dr = (dB/dr - B/r) / (4r),
// where no two terms cancel.
__device__ __forceinline__ f2 hct_cut_far_fr2(f2 r, f2 rinv, f2 s, float rc, bool use0, bool use1) {
    const CutFar c = hct_cut_far_terms(r, s, rc, use0, use1);
    const f2 zp = neg2(make_float2(c.cx ? c.iU.x : c.z.x * c.iU.x, c.cy ? c.iU.y : c.z.y * c.iU.y));
    const f2 t = mul2(mul2(zp, c.z), mul2(fma2(F2(2.0f), s, neg2(c.w)), c.iL));
    const f2 dB = fma2(neg2(mul2(s, mul2(c.iL, c.iL))), mul2(c.z, c.z), t);
    const f2 dH = mul2(mul2(F2(0.25f), rinv), fma2(neg2(c.B), rinv, dB));
    return mul2(neg2(dH), rinv);
}
// One direction (descreened atom radius a, descreening sphere s) per half of
// a queued pair near rc (see BornCut): disjoint spheres take the restricted form above (the whole sphere while it lies inside the ball, 0
// once it lies wholly past rc), overlapping ones the general restricted
// closed form behind a vote.
__device__ __forceinline__ f2 hct_cut_dir2(f2 r, f2 rinv, f2 a, f2 s, float rc) {
    const bool d0 = r.x >= a.x + s.x, d1 = r.y >= a.y + s.y;
    f2 h = hct_cut_far2(r, rinv, s, rc, d0, d1);
    if (__any_sync(0xffffffffu, !(d0 && d1))) {
        const f2 g = hct_cut2(r, rinv, a, s, rc, 1.0f / rc);
        h = make_float2(d0 ? h.x : g.x, d1 ? h.y : g.y);
    }
    return h;
}
__device__ __forceinline__ f2 hct_cut_dir_fr2(f2 r, f2 rinv, f2 a, f2 s, float rc) {
    const bool d0 = r.x >= a.x + s.x, d1 = r.y >= a.y + s.y;
    f2 h = hct_cut_far_fr2(r, rinv, s, rc, d0, d1);
    if (__any_sync(0xffffffffu, !(d0 && d1))) {
        const f2 g = hct_cut_fr2(r, rinv, a, s, rc);
        h = make_float2(d0 ? h.x : g.x, d1 ? h.y : g.y);
    }
    return h;
}

__device__ __forceinline__ long long warp_sum_ll(long long v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// --- diagonal masks -------------------------------------------------------------------
// Step k pairs lane l's i atoms with tile atom (l + k) mod 32.  A tile that
// holds the same atoms as an i half ("diagonal") keeps steps 1..15 and the
// lower half of step 16, which visit each unordered pair once.  Mode DX: the
// tile is the x half's own tile and the y half is below the diagonal (off);
// mode DY: the tile is the y half's own tile (x half fully on).
enum { M_FULL = 0, M_DX = 1, M_DY = 2 };
// Per-block bounds of the general energy code (see block_info).
struct BlockInfo {
    bool far;         // no pair within the soft repulsion's range
    float skip2;      // EF_STRADDLE blocks: a step whose pairs all have r^2 > skip2 adds nothing
};
struct Mask {
    bool x, y;
};
template <int MODE>
__device__ __forceinline__ Mask step_mask(int k, int lane) {
    const bool diag = (k >= 1 && k <= 15) || (k == 16 && lane < 16);
    Mask m;
    m.x = (MODE == M_DX) ? diag : true;
    m.y = (MODE == M_FULL) ? true : (MODE == M_DY ? diag : false);
    return m;
}
template <int MODE>
__device__ __forceinline__ f2 keep(f2 v, Mask m) {
    if (MODE == M_FULL) return v;
    return make_float2(m.x ? v.x : 0.0f, m.y ? v.y : 0.0f);
}
template <int MODE>
__device__ __forceinline__ f2 safe_r2(f2 r2, Mask m) {
    if (MODE == M_FULL) return r2;
    return make_float2(m.x ? r2.x : FAR_R2, m.y ? r2.y : FAR_R2);
}

__device__ __forceinline__ f2 sel2(f2 v, Mask m) { return make_float2(m.x ? v.x : 0.0f, m.y ? v.y : 0.0f); }

// Lanes past a replica's end hold ghost atoms (see ghost_x): zero charge,
// zero descreening radius, zero chain factor, parked far away.
__device__ __forceinline__ void load_xas(const PairArgs& A, int64_t base, int n, int i, float& x,
                                         float& y, float& z, float& a, float& s) {
    if (i < n) {
        const float4 p = __ldcg(&A.xyzq[base + i]);
        const float2 rs = A.rad[base + i];
        x = p.x; y = p.y; z = p.z;
        a = rs.x - A.offset;
        s = rs.y * a;
    } else {
        x = ghost_x(i - n); y = 0.0f; z = 0.0f; a = 1.0f; s = 0.0f;
    }
}

// --- pass 1: Born integrals I_i = sum_j H(r_ij; a_i, s_j) -----------------------
struct Born {
    static constexpr int NQ = 1;      // int64 i-side accumulators per atom (shared memory)
    static constexpr int NJ = 1;      // j-side ones that close pairs add to
    static constexpr bool RADIUS_CUT = true;   // EF_CUT: the cutoff is rgbmax
    static constexpr bool CHAIN = false;
    static __device__ __forceinline__ void flush_i(const PairArgs& A, int64_t base, int n, int i0, int lane,
                                                   long long* sa) {
        if (i0 + lane < n) red_add(&A.I_acc[base + i0 + lane], sa[lane]);
        if (i0 + 32 + lane < n) red_add(&A.I_acc[base + i0 + 32 + lane], sa[32 + lane]);
    }
};

// --- pass 2: GB + Coulomb pair energy, direct forces, dE/dR, dE/dq --------------
// Pair (i, j), both orderings of the double sum together:
//   e_GB = -tau k_e q_i q_j / f,  f^2 = r^2 + R_i R_j exp(-D),  D = r^2 / (4 R_i R_j)
//   e_C  =  k_c q_i q_j / r
//   -(de/dr)/r = k_c q_i q_j / r^3 - tau k_e q_i q_j (1 - exp(-D)/4) / f^3
//   R_i de/dR_i = tau k_e q_i q_j exp(-D)(R_i R_j + r^2/4) / (2 f^3)   (and i <-> j:
//                 (1 + D) R_i R_j = R_i R_j + r^2/4, the same value on both sides)
//   de/dq_i = (-tau k_e / f + k_c / r) q_j                  (and i <-> j)
// Each atom carries h = sqrt(log2 e) / (2R) (negated for i), so that
// exp(-D) = 2^(r^2 (-h_i) h_j) is two multiplies and one ex2.
struct Energy {
    static constexpr int NQ = 5;      // fx, fy, fz, R dE/dR, dE/dq (shared memory)
    static constexpr int NJ = 3;
    static constexpr bool RADIUS_CUT = false;  // EF_CUT: the cutoff is `cut`
    static constexpr bool CHAIN = false;
    struct IState {
        f2 nx, ny, nz, q, R, nh;
        f2 qa, qk;                    // q tau k_e / 2 and q k_c (unscreened pair factors)
        long long egb, ec, er;
    };
    struct JState { float x, y, z, q, R, h, fx, fy, fz, dR, phi; };
    struct Part {
        f2 sx, sy, sz, dR, phi, egb, ec, er;   // s* = sum of fr d (the i force is -s)
        f2 kgb, kc, kr;                        // compensation terms of the energy sums
        __device__ __forceinline__ void zero() {
            sx = sy = sz = dR = phi = egb = ec = er = kgb = kc = kr = F2(0.0f);
        }
    };
    static __device__ __forceinline__ void load_one(const PairArgs& A, int64_t base, int n, int i, float& x,
                                                    float& y, float& z, float& q, float& R, float& h) {
        if (i < n) {
            const float4 p = __ldcg(&A.xyzq[base + i]);
            const float2 rh = __ldcg(&A.Rh[base + i]);
            x = p.x; y = p.y; z = p.z; q = p.w; R = rh.x; h = rh.y * SQRT_LOG2E;
        } else {
            x = ghost_x(i - n); y = 0.0f; z = 0.0f; q = 0.0f; R = 1.0f; h = 0.5f * SQRT_LOG2E;
        }
    }
    static __device__ __forceinline__ void load_i(const PairArgs& A, int64_t base, int n, int i0, int lane, IState& st) {
        float x0, y0, z0, q0, R0, h0, x1, y1, z1, q1, R1, h1;
        load_one(A, base, n, i0 + lane, x0, y0, z0, q0, R0, h0);
        load_one(A, base, n, i0 + 32 + lane, x1, y1, z1, q1, R1, h1);
        st.nx = make_float2(-x0, -x1); st.ny = make_float2(-y0, -y1); st.nz = make_float2(-z0, -z1);
        st.q = make_float2(q0, q1); st.R = make_float2(R0, R1); st.nh = make_float2(-h0, -h1);
        st.qa = mul2(st.q, F2(0.5f * A.tau_ke));
        st.qk = mul2(st.q, F2(A.kc));
        st.egb = st.ec = st.er = 0;
    }
    static __device__ __forceinline__ void load_j(const PairArgs& A, int64_t base, int n, int j, JState& st) {
        load_one(A, base, n, j, st.x, st.y, st.z, st.q, st.R, st.h);
        st.fx = st.fy = st.fz = st.dR = st.phi = 0.0f;
    }
    template <int FLAGS, int MODE, bool FAR>
    static __device__ __forceinline__ void pair(const PairArgs& A, const IState& i, JState& j, Part& p, Mask m,
                                                const BlockInfo&, int i0, int jbase, int k) {
        const f2 dx = add2(F2(j.x), i.nx), dy = add2(F2(j.y), i.ny), dz = add2(F2(j.z), i.nz);
        const f2 r2 = safe_r2<MODE>(fma2(dx, dx, fma2(dy, dy, mul2(dz, dz))), m);
        // energies are sums of large terms that cancel: when they are wanted,
        // one Newton step takes the MUFU reciprocal square roots to FP32 rounding
        const f2 rinv = (FLAGS & EF_ENERGY) ? rsqrt2_nr(r2) : rsqrt2(r2);
        const f2 rinv2 = mul2(rinv, rinv);
        const f2 qq = mul2(i.q, F2(j.q));
        const f2 nDl = mul2(r2, mul2(i.nh, F2(j.h)));                 // -D log2(e)
        const f2 e = ex22(nDl);                                       // exp(-D)
        const f2 RR = mul2(i.R, F2(j.R));
        const f2 fsq = fma2(RR, e, r2);
        const f2 finv = (FLAGS & EF_ENERGY) ? rsqrt2_nr(fsq) : rsqrt2(fsq);
        const f2 finv3 = mul2(mul2(finv, finv), finv);
        // solvent factors: tE in the energy (-tE q q / f), tF in its f-derivative;
        // both (1/eps_in - 1/eps_out) k_e without salt, screened by
        // exp(-kappa f) with it (Debye-Hueckel)
        f2 tE = F2(A.tau_ke), w;
        if (FLAGS & EF_SALT) {
            const f2 f = mul2(fsq, finv);
            const f2 ekv = mul2(F2(A.ke_out), ex22(mul2(F2(-A.kappa * LOG2E), f)));   // k_e e^{-kappa f} / eps_out
            tE = add2(F2(A.kc), neg2(ekv));
            const f2 tF = fma2(neg2(ekv), mul2(F2(A.kappa), f), tE);
            w = mul2(mul2(qq, F2(0.5f)), mul2(tF, finv3));           // tF q q / (2 f^3)
        } else {
            w = mul2(mul2(i.qa, F2(j.q)), finv3);
        }
        const f2 nu = fma2(F2(0.5f), e, F2(-2.0f));                   // -2 (1 - e/4)
        const f2 qc = mul2(i.qk, F2(j.q));
        f2 fr = fma2(qc, mul2(rinv2, rinv), mul2(w, nu));
        f2 G = mul2(mul2(w, e), fma2(r2, F2(0.25f), RR));              // w e (1 + D) R_i R_j
        Mask cm{true, true};          // pair within the cutoff (EF_STRADDLE blocks test it)
        if (FLAGS & EF_STRADDLE) {
            cm.x = r2.x <= A.cut2;
            cm.y = r2.y <= A.cut2;
            fr = sel2(fr, cm);
            G = sel2(G, cm);
        }
        f2 er = F2(0.0f);
        if ((FLAGS & EF_REP) && !FAR) {
            const float sig2 = A.rep_sigma * A.rep_sigma;
            const bool n0 = r2.x < sig2, n1 = r2.y < sig2;
            if (__any_sync(0xffffffffu, n0 || n1)) {
                const int jj = jbase + ((threadIdx.x + k) & 31);
                const int ia = i0 + (threadIdx.x & 31), ib = ia + 32;
                if (n0 && (ia - jj > 1 || jj - ia > 1)) {
                    const float dd = A.rep_sigma - r2.x * rinv.x;
                    fr.x = fmaf(2.0f * A.rep_k * dd, rinv.x, fr.x);
                    er.x = A.rep_k * dd * dd;
                }
                if (n1 && (ib - jj > 1 || jj - ib > 1)) {
                    const float dd = A.rep_sigma - r2.y * rinv.y;
                    fr.y = fmaf(2.0f * A.rep_k * dd, rinv.y, fr.y);
                    er.y = A.rep_k * dd * dd;
                }
            }
        }
        fr = keep<MODE>(fr, m);
        G = keep<MODE>(G, m);
        p.sx = fma2(fr, dx, p.sx); p.sy = fma2(fr, dy, p.sy); p.sz = fma2(fr, dz, p.sz);
        j.fx = fmaf(fr.y, dx.y, fmaf(fr.x, dx.x, j.fx));
        j.fy = fmaf(fr.y, dy.y, fmaf(fr.x, dy.x, j.fy));
        j.fz = fmaf(fr.y, dz.y, fmaf(fr.x, dz.x, j.fz));
        p.dR = add2(p.dR, G);
        j.dR += G.x + G.y;
        if (FLAGS & EF_PHI) {
            f2 P = keep<MODE>(fma2(neg2(tE), finv, mul2(F2(A.kc), rinv)), m);
            if (FLAGS & EF_STRADDLE) P = sel2(P, cm);
            p.phi = fma2(P, F2(j.q), p.phi);
            j.phi = fmaf(P.y, i.q.y, fmaf(P.x, i.q.x, j.phi));
        }
        if (FLAGS & EF_ENERGY) {
            // the pair energies are large terms that cancel: compensated
            // (Kahan) FP32 sums within the block
            f2 eg = keep<MODE>(mul2(neg2(tE), mul2(qq, finv)), m), ecl = keep<MODE>(mul2(qc, rinv), m);
            if (FLAGS & EF_STRADDLE) {
                eg = sel2(eg, cm);
                ecl = sel2(ecl, cm);
            }
            kahan_add(p.egb, p.kgb, eg);
            kahan_add(p.ec, p.kc, ecl);
            if (FLAGS & EF_REP) kahan_add(p.er, p.kr, keep<MODE>(er, m));
        }
    }
    static __device__ __forceinline__ void rotate_data(JState& j, int src) {
        j.x = shfl(j.x, src); j.y = shfl(j.y, src); j.z = shfl(j.z, src);
        j.q = shfl(j.q, src); j.R = shfl(j.R, src); j.h = shfl(j.h, src);
    }
    template <int FLAGS>
    static __device__ __forceinline__ void rotate_acc_f(JState& j, int src) {
        j.fx = shfl(j.fx, src); j.fy = shfl(j.fy, src); j.fz = shfl(j.fz, src);
        j.dR = shfl(j.dR, src);
        if (FLAGS & EF_PHI) j.phi = shfl(j.phi, src);
    }
    static __device__ __forceinline__ void take_data(JState& j, const JState& d) {
        j.x = d.x; j.y = d.y; j.z = d.z; j.q = d.q; j.R = d.R; j.h = d.h;
    }
    template <int FLAGS>
    static __device__ __forceinline__ void fold_i_f(IState& i, long long* sa, int lane, const Part& p) {
        sa[lane] -= fix(p.sx.x); sa[32 + lane] -= fix(p.sx.y);
        sa[64 + lane] -= fix(p.sy.x); sa[96 + lane] -= fix(p.sy.y);
        sa[128 + lane] -= fix(p.sz.x); sa[160 + lane] -= fix(p.sz.y);
        sa[192 + lane] += fix(p.dR.x); sa[224 + lane] += fix(p.dR.y);
        if (FLAGS & EF_PHI) {
            sa[256 + lane] += fix(p.phi.x);
            sa[288 + lane] += fix(p.phi.y);
        }
        if (FLAGS & EF_ENERGY) {
            i.egb += (fix(p.egb.x) + fix(p.egb.y)) - (fix(p.kgb.x) + fix(p.kgb.y));
            i.ec += (fix(p.ec.x) + fix(p.ec.y)) - (fix(p.kc.x) + fix(p.kc.y));
            if (FLAGS & EF_REP) i.er += (fix(p.er.x) + fix(p.er.y)) - (fix(p.kr.x) + fix(p.kr.y));
        }
    }
    template <int FLAGS>
    static __device__ __forceinline__ void flush_j_f(const PairArgs& A, int64_t base, int n, int j, const JState& st) {
        if (j < n) {
            const int64_t g = base + j;
            red_add(&A.F_acc[g], fix(st.fx));
            red_add(&A.F_acc[A.N + g], fix(st.fy));
            red_add(&A.F_acc[2 * A.N + g], fix(st.fz));
            red_add(&A.dR_acc[g], fix(st.dR));
            if (FLAGS & EF_PHI) red_add(&A.phi_acc[g], fix(st.phi));
        }
    }
    template <int FLAGS>
    static __device__ __forceinline__ void flush_i_f(const PairArgs& A, int64_t base, int n, int i0, int lane,
                                                     long long* sa) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = i0 + 32 * h + lane;
            if (i < n) {
                const int64_t g = base + i;
                const int o = 32 * h + lane;
                red_add(&A.F_acc[g], sa[o]);
                red_add(&A.F_acc[A.N + g], sa[64 + o]);
                red_add(&A.F_acc[2 * A.N + g], sa[128 + o]);
                red_add(&A.dR_acc[g], sa[192 + o]);
                if (FLAGS & EF_PHI) red_add(&A.phi_acc[g], sa[256 + o]);
            }
        }
    }
    template <int FLAGS>
    static __device__ __forceinline__ void flush_sums_f(const PairArgs& A, int r, int lane, const IState& st) {
        if (FLAGS & EF_ENERGY) {
            const long long egb = warp_sum_ll(st.egb), ec = warp_sum_ll(st.ec);
            const long long er = (FLAGS & EF_REP) ? warp_sum_ll(st.er) : 0;
            if (lane == 0) {
                red_add(&A.E_acc[4 * r + 0], egb);
                red_add(&A.E_acc[4 * r + 1], ec);
                if (FLAGS & EF_REP) red_add(&A.E_acc[4 * r + 2], er);
            }
        }
    }
};

// --- pass 3: Born-radius chain rule -------------------------------------------
// E depends on R_i(psi_i), psi_i = a_i sum_j H(r_ij; a_i, s_j).  With
// c_i = dE/dR_i * dR_i/dpsi_i * a_i the pair (i, j) carries
//   -(dE/dr)/r = c_i * (-(dH(r; a_i, s_j)/dr)/r) + c_j * (-(dH(r; a_j, s_i)/dr)/r).
struct Chain {
    static constexpr int NQ = 3;      // fx, fy, fz (shared memory)
    static constexpr int NJ = 3;
    static constexpr bool RADIUS_CUT = true;   // EF_CUT: the cutoff is rgbmax
    static constexpr bool CHAIN = true;
    static __device__ __forceinline__ void load_one(const PairArgs& A, int64_t base, int n, int i, float& x,
                                                    float& y, float& z, float& a, float& s, float& c) {
        load_xas(A, base, n, i, x, y, z, a, s);
        c = (i < n) ? __ldcg(&A.cc[base + i]) : 0.0f;
    }
    static __device__ __forceinline__ void flush_i(const PairArgs& A, int64_t base, int n, int i0, int lane,
                                                   long long* sa) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int i = i0 + 32 * h + lane;
            if (i < n) {
                const int64_t g = base + i;
                const int o = 32 * h + lane;
                red_add(&A.F_acc[g], sa[o]);
                red_add(&A.F_acc[A.N + g], sa[64 + o]);
                red_add(&A.F_acc[2 * A.N + g], sa[128 + o]);
            }
        }
    }
};

// Energy's helpers carry the flag set; adapt them to the walker's interface.
template <int FLAGS>
struct EnergyF : Energy {
    static __device__ __forceinline__ void rotate_acc(JState& j, int src) { rotate_acc_f<FLAGS>(j, src); }
    static __device__ __forceinline__ void fold_i(IState& i, long long* sa, int lane, const Part& p) {
        fold_i_f<FLAGS>(i, sa, lane, p);
    }
    static __device__ __forceinline__ void flush_j(const PairArgs& A, int64_t b, int n, int j, const JState& s) {
        flush_j_f<FLAGS>(A, b, n, j, s);
    }
    static __device__ __forceinline__ void flush_i(const PairArgs& A, int64_t b, int n, int i0, int lane,
                                                   long long* sa) {
        flush_i_f<FLAGS>(A, b, n, i0, lane, sa);
    }
    static __device__ __forceinline__ void flush_sums(const PairArgs& A, int r, int lane, const IState& s) {
        flush_sums_f<FLAGS>(A, r, lane, s);
    }
};

// --- the warp walker ------------------------------------------------------------
// The steps of one (super-row, tile) block: after 32 rotations every j value is
// back in its home lane.
template <class P, int FLAGS, int MODE, bool FAR>
__device__ __forceinline__ void run_tile(const PairArgs& A, const typename P::IState& is, typename P::JState& js,
                                         typename P::Part& ip, const BlockInfo& bi, int i0, int jbase, int lane,
                                         int next) {
    // a DX block pairs the x half with its own tile: only steps 1 .. 16 carry
    // pairs (js enters rotated by one and leaves rotated by 17)
    constexpr int K0 = (MODE == M_DX) ? 1 : 0, K1 = (MODE == M_DX) ? 17 : 32;
    // with steps left out the loop is not worth unrolling
    constexpr int U = (FLAGS & EF_STRADDLE) ? 1 : 2;
#pragma unroll U
    for (int k = K0; k < K1; ++k) {
        // the next step's j data are fetched before this step's arithmetic, so
        // that only the short accumulator chain is serial between steps
        typename P::JState nx = js;
        P::rotate_data(nx, next);
        const Mask m = step_mask<MODE>(k, lane);
        bool busy = true;
        if (FLAGS & EF_STRADDLE) {   // every pair of this step wholly past the cutoff's reach
            const float dx0 = js.x + is.nx.x, dy0 = js.y + is.ny.x, dz0 = js.z + is.nz.x;
            const float dx1 = js.x + is.nx.y, dy1 = js.y + is.ny.y, dz1 = js.z + is.nz.y;
            const float q0 = fmaf(dx0, dx0, fmaf(dy0, dy0, dz0 * dz0));
            const float q1 = fmaf(dx1, dx1, fmaf(dy1, dy1, dz1 * dz1));
            busy = __any_sync(0xffffffffu, fminf(q0, q1) <= bi.skip2);
        }
        if (busy) P::template pair<FLAGS, MODE, FAR>(A, is, js, ip, m, bi, i0, jbase, k);
        P::rotate_acc(js, next);
        P::take_data(js, nx);
    }
}

// Bounds between the box of super-row K (tiles 2K, 2K+1) and the box of tile
// J: least and greatest distance squared, largest a and largest s of both.
struct BoxPair {
    float rmin2, rmax2, amax, smax;
};
__device__ __forceinline__ float4 row_box_lo(const PairArgs& A, int t0, int K, int nb, float4* hi) {
    float4 il = __ldcg(&A.boxes[2 * (t0 + 2 * K)]), ih = __ldcg(&A.boxes[2 * (t0 + 2 * K) + 1]);
    if (2 * K + 1 < nb) {
        const float4 l1 = __ldcg(&A.boxes[2 * (t0 + 2 * K + 1)]), h1 = __ldcg(&A.boxes[2 * (t0 + 2 * K + 1) + 1]);
        il = make_float4(fminf(il.x, l1.x), fminf(il.y, l1.y), fminf(il.z, l1.z), fmaxf(il.w, l1.w));
        ih = make_float4(fmaxf(ih.x, h1.x), fmaxf(ih.y, h1.y), fmaxf(ih.z, h1.z), fmaxf(ih.w, h1.w));
    }
    *hi = ih;
    return il;
}
__device__ __forceinline__ BoxPair box_pair(float4 il, float4 ih, float4 jl, float4 jh) {
    BoxPair b;
    const float gx = fmaxf(0.0f, fmaxf(il.x - jh.x, jl.x - ih.x));
    const float gy = fmaxf(0.0f, fmaxf(il.y - jh.y, jl.y - ih.y));
    const float gz = fmaxf(0.0f, fmaxf(il.z - jh.z, jl.z - ih.z));
    const float mx = fmaxf(ih.x - jl.x, jh.x - il.x);
    const float my = fmaxf(ih.y - jl.y, jh.y - il.y);
    const float mz = fmaxf(ih.z - jl.z, jh.z - il.z);
    b.rmin2 = gx * gx + gy * gy + gz * gz;
    b.rmax2 = mx * mx + my * my + mz * mz;
    b.amax = fmaxf(il.w, jl.w);
    b.smax = fmaxf(ih.w, jh.w);
    return b;
}

// Cutoff classes of a block from its box bounds (rmin / rmax the least /
// greatest distance between the boxes, smax the largest screened radius):
//   Born-radius cutoff (Born and chain passes): in range when
//     rmin < rgbmax + smax (some sphere j reaches into the ball about some
//     i), straddling when rmax + smax > rgbmax (some sphere reaches past it);
//   pair cutoff (energy pass): in range when rmin <= max(cut, rep_sigma),
//     straddling when rmax > cut.
// The bounds carry a 0.1 % margin, so that FP32 rounding of a pair's r^2 can
// never move it across a decision taken for its block.  A block that is not
// straddling needs no per-pair test; one out of range adds nothing.
__device__ __forceinline__ void cut_class(const PairArgs& A, bool radius_cut, const BoxPair& b, bool& in,
                                          bool& st) {
    if (radius_cut) {
        const float reach = A.rgbmax + b.smax, inner = A.rgbmax - b.smax;
        in = b.rmin2 <= 1.001f * reach * reach;
        st = inner <= 0.0f || b.rmax2 >= 0.999f * inner * inner;
    } else {
        in = b.rmin2 <= 1.001f * A.e_range2;
        st = b.rmax2 >= 0.999f * A.cut2;
    }
}

// Bounds of a block from the bounding boxes of its tiles (lo.xyz with max a,
// hi.xyz with max s, from k_tile_boxes); without boxes nothing is proven.
__device__ __forceinline__ BlockInfo block_info(const PairArgs& A, int r, int K, int J, int nb) {
    BlockInfo bi;
    bi.far = A.rep_k == 0.0f;
    bi.skip2 = A.boxes ? 1.001f * A.e_range2 : INFINITY;
    if (!bi.far && A.boxes) {
        const int t0 = A.tile_off[r];
        const float4 jl = __ldcg(&A.boxes[2 * (t0 + J)]), jh = __ldcg(&A.boxes[2 * (t0 + J) + 1]);
        float4 ih;
        const float4 il = row_box_lo(A, t0, K, nb, &ih);
        bi.far = box_pair(il, ih, jl, jh).rmin2 >= A.rep_sigma * A.rep_sigma;
    }
    return bi;
}

// --- blocks by distance ---------------------------------------------------------------
// Every 64 x 32 block is classified from the tile boxes (row_tier).  For the
// Born and chain passes
//   near (0):     some pair may overlap or have (s/r)^2 > GB_POLY_YFAR;
//                 polynomials in y = (s/r)^2 up to GB_POLY_YNEAR;
//   far (1):      none has: polynomials in y of degree 4 and 5;
//   distant (2, 3): polynomials of degree 3 or 2 in u = 1/r^2 with the powers
//                 of s folded into per-atom coefficients,
//                   H(r; a, s) = u^2 (A_0 + A_1 u + ...),  A_k = 1/2 s^3 g_k s^2k
//                   -(dH/dr)/r = u^3 (B_0 + B_1 u + ...),  B_k = 1/2 s^3 h_k s^2k
//                 (GB_Y_*: the largest (s/r)^2 for which such a fit is as good
//                 as the FP32 form that nearer blocks use).
// The integrals contain even powers of r only, so 1/r^2 is one MUFU
// reciprocal and no square root is taken.  The energy pass has one form; its
// near blocks are those inside the soft repulsion's range.
//
// Where both rows of a row pair are far from a tile the block is evaluated
// 128 x 32: lane l holds the four atoms 128 P + 32 q + l (NW = 2 FP32x2
// pairs), so that one load of the j atom and one rotation of its partial sums
// serve four pairs a lane.  A pair step costs issue slots for everything it
// executes -- an FP32x2 instruction takes two, three when it reads three
// different register pairs -- so shuffles and moves count in full: at two
// atoms a lane with the j atoms rotated by shuffles they were a third of the
// 72 / 110 / 104 slots of a Born / energy / chain step of 64 pairs, which now
// takes 36 to 41 / 79 / 57 to 62.
//
// Near and diagonal blocks (64 x 32, NW = 1) run the far form for every pair,
// without votes or branches; pairs closer than the block's bound t are left
// out (r^2 set to FAR_R2) and noted in a bit mask.  After the tile those are
// gathered and evaluated 32 at a time, exactly (close_pairs): two pairs of a
// hundred, which otherwise made every second step of a near block run the
// closed form for all its lanes.

// r^2 of a step's pairs: masked-off pairs (diagonal blocks) read as far; with
// NEAR, pairs below t set bit `bit` of the lane's masks and, with DROP, read
// as far too.
template <int MODE, bool NEAR, bool DROP>
__device__ __forceinline__ f2 screen_r2(f2 r2, Mask m, float t, unsigned bit, unsigned& mx, unsigned& my) {
    if (MODE == M_FULL && !NEAR) return r2;
    const bool cx = NEAR && r2.x < t && m.x, cy = NEAR && r2.y < t && m.y;
    if (NEAR) {
        mx |= cx ? bit : 0u;
        my |= cy ? bit : 0u;
    }
    return make_float2((DROP && cx) || !m.x ? FAR_R2 : r2.x, (DROP && cy) || !m.y ? FAR_R2 : r2.y);
}

// Bounds on r^2 in a block that straddles the Born-radius cutoff: pairs from
// close to in are as without a cutoff, pairs from out on add exact zeros.
struct Ring { float close, in, out; };
__device__ __forceinline__ Ring ring_of(const PairArgs& A, float close, float smax) {
    const float outer = A.rgbmax + smax, inner = fmaxf(A.rgbmax - smax, 0.0f);
    return Ring{close, 0.999f * inner * inner, 1.001f * outer * outer};
}
// The same screen with a ring: the other pairs read as far, and those before
// out (or NaN) set their bit.
template <int MODE, bool NEAR, bool DROP>
__device__ __forceinline__ f2 screen_r2(f2 r2, Mask m, Ring g, unsigned bit, unsigned& mx, unsigned& my) {
    const bool kx = r2.x >= g.close && r2.x < g.in, ky = r2.y >= g.close && r2.y < g.in;
    mx |= !kx && !(r2.x >= g.out) && m.x ? bit : 0u;
    my |= !ky && !(r2.y >= g.out) && m.y ? bit : 0u;
    return make_float2(kx && m.x ? r2.x : FAR_R2, ky && m.y ? r2.y : FAR_R2);
}

// The staged tile of a warp: j atoms (twice, see walk_far), what close pairs
// need of both sides, their j sums and their queue.
constexpr int CLOSE_CAP = 512;
template <class W>
struct Slot {
    long long* sa;        // [2][NQ][64] i-side sums of both rows
    float4* j4;           // [64] x, y, z and a fourth value of the j atoms
    typename W::B* jb;    // [64] further values
    float2* ja;           // [32] a, s of the j atoms
    long long* jac;       // [NJ][32] j-side sums of close pairs
    float4* i4;           // [64] x, y, z, c of the i atoms
    float2* i2;           // [64] a, s of the i atoms
    unsigned short* queue;
    __device__ __forceinline__ explicit Slot(int slot) {
        extern __shared__ __align__(16) unsigned char s_mem[];
        unsigned char* p = s_mem + slot;
        sa = (long long*)p;
        j4 = (float4*)(p + 2 * W::NQ * 64 * 8);
        jb = (typename W::B*)(j4 + 64);
        ja = (float2*)(j4 + 96);
        jac = (long long*)(ja + 32);
        i4 = (float4*)(jac + 32 * W::NJ);
        i2 = (float2*)(i4 + 64);
        queue = (unsigned short*)(i2 + 64);
    }
};
// Shared memory of a warp: i-side sums of two rows, then the larger of the
// staged tile of 128 x 32 blocks (two float4 arrays of 64) and a Slot.
template <class P>
constexpr int WARP_SMEM = 2 * P::NQ * 64 * 8 + 1024 + 512 + 256 + P::NJ * 256 + 1024 + 512 + 2 * CLOSE_CAP;
// Warps per block a pass can run within the 48 KB that need no opt-in.
template <class P>
inline int fit_warps(int wpb) { return wpb * WARP_SMEM<P> <= 49152 ? wpb : 49152 / WARP_SMEM<P>; }

// Exact sums into N shared 64-bit words by two 32-bit atomics each (there is no
// native 64-bit one): the carry follows from the low word's old value.  All
// low words first, so that their latencies overlap.
template <int N>
__device__ __forceinline__ void shared_add(long long* const (&p)[N], const long long (&v)[N]) {
    unsigned old[N];
#pragma unroll
    for (int k = 0; k < N; ++k) old[k] = atomicAdd((unsigned*)p[k], (unsigned)v[k]);
#pragma unroll
    for (int k = 0; k < N; ++k)
        atomicAdd((unsigned*)p[k] + 1, (unsigned)((u64)v[k] >> 32) + (old[k] + (unsigned)v[k] < old[k] ? 1u : 0u));
}

// The r^2 below which a pair of a near block is close: above it the spheres
// are disjoint in both directions and (s/r)^2 <= GB_POLY_YNEAR.  Rounded up a
// little, so that rounding in r^2 cannot admit a pair that is neither.
__device__ __forceinline__ float close_bound(float amax, float smax) {
    const float as = amax + smax;
    return 1.0001f * fmaxf(as * as, smax * smax * (1.0f / GB_POLY_YNEAR));
}
// The same from the staged atoms, where there are no tile boxes.
template <class W>
__device__ __forceinline__ float staged_bound(const Slot<W>& S, int lane) {
    const float2 a = S.i2[lane], b = S.i2[32 + lane], c = S.ja[lane];
    float am = fmaxf(a.x, fmaxf(b.x, c.x)), sm = fmaxf(a.y, fmaxf(b.y, c.y));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
        sm = fmaxf(sm, __shfl_xor_sync(0xffffffffu, sm, o));
    }
    return close_bound(am, sm);
}

// --- Born integrals --------------------------------------------------------------------
template <int NW>
struct BornY {
    static constexpr bool CUT = false;
    static constexpr int ATOMS = 64 * NW, NQ = Born::NQ, NJ = Born::NJ, UNROLL = NW == 2 ? 2 : 4;
    struct I { f2 nx[NW], ny[NW], nz[NW], s2[NW], hs3[NW]; };
    typedef float B;                                   // staged j values: x, y, z, s^2 | s^3 / 2
    struct J { float acc; };
    struct Part { f2 s[NW]; };
    static __device__ __forceinline__ void load(const PairArgs& A, int64_t base, int n, int i, float4& v, B& b, float2& as) {
        load_xas(A, base, n, i, v.x, v.y, v.z, as.x, as.y);
        v.w = as.y * as.y;
        b = 0.5f * v.w * as.y;
    }
    static __device__ __forceinline__ void load_i(const PairArgs& A, int64_t base, int n, int i0, int lane, I& st,
                                                  float4* i4 = nullptr, float2* i2 = nullptr) {
#pragma unroll
        for (int q = 0; q < 2 * NW; ++q) {
            float4 v;
            float b;
            float2 as;
            load(A, base, n, i0 + 32 * q + lane, v, b, as);
            set2(st.nx[q >> 1], q & 1, -v.x); set2(st.ny[q >> 1], q & 1, -v.y); set2(st.nz[q >> 1], q & 1, -v.z);
            set2(st.s2[q >> 1], q & 1, v.w); set2(st.hs3[q >> 1], q & 1, b);
            if (i4) {
                i4[32 * q + lane] = v;
                i2[32 * q + lane] = as;
            }
        }
    }
    static __device__ __forceinline__ void load_j(const PairArgs& A, int64_t base, int n, int j, float4& v, B& b) {
        float2 as;
        load(A, base, n, j, v, b, as);
    }
    static __device__ __forceinline__ void zero(J& j, Part& p) {
        j.acc = 0.0f;
#pragma unroll
        for (int q = 0; q < NW; ++q) p.s[q] = F2(0.0f);
    }
    template <int MODE = M_FULL, bool NEAR = false, class T = float>
    static __device__ __forceinline__ void step(const PairArgs&, const I& i, float4 v, B b, J& j, Part& p,
                                                Mask m = Mask{true, true}, T t = T(), unsigned bit = 0,
                                                unsigned* mk = nullptr) {
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const f2 dx = add2(F2(v.x), i.nx[q]), dy = add2(F2(v.y), i.ny[q]), dz = add2(F2(v.z), i.nz[q]);
            f2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
            if (MODE != M_FULL || NEAR) r2 = screen_r2<MODE, NEAR, true>(r2, m, t, bit, mk[0], mk[1]);
            const f2 u = rcp2_approx(r2);
            const f2 u2 = mul2(u, u);
            const f2 yj = mul2(F2(v.w), u), yi = mul2(i.s2[q], u);
            p.s[q] = fma2(F2(b), mul2(u2, NW == 1 ? gb_poly_gn2(yj) : gb_poly_gf2(yj)), p.s[q]);
            const f2 h = mul2(u2, NW == 1 ? gb_poly_gn2(yi) : gb_poly_gf2(yi));
            j.acc = fmaf(i.hs3[q].y, h.y, fmaf(i.hs3[q].x, h.x, j.acc));
        }
    }
    static __device__ __forceinline__ void rotate_acc(J& j, int src) { j.acc = shfl(j.acc, src); }
    static __device__ __forceinline__ void fold_i(const PairArgs&, long long* sa, int lane, const Part& p) {
#pragma unroll
        for (int q = 0; q < 2 * NW; ++q) sa[32 * q + lane] += fix_i(get2(p.s[q >> 1], q & 1));
    }
    // Two atoms at the same position (r = 0; masked pairs read as far) give a
    // NaN through r = r^2 / r; a NaN coordinate gives one in every sum it
    // enters.  Both are recorded before the fixed-point conversion would
    // hide them: here and where close pairs are evaluated.
    static __device__ __forceinline__ void flush_j(const PairArgs& A, int64_t base, int n, int j, const J& st,
                                                   const long long* jac = nullptr, int at = 0) {
        if (!isfinite(st.acc) && A.err) atomicCAS(A.err, 0, GB_ERR_NONFINITE);
        if (j < n) red_add(&A.I_acc[base + j], fix_i(st.acc) + (jac ? jac[at] : 0));
    }
    static __device__ __forceinline__ void flush_close(const PairArgs& A, int64_t g, const long long* jac, int j) {
        red_add(&A.I_acc[g], jac[j]);
    }
    static __device__ __forceinline__ float bound(const PairArgs&, const Slot<BornY>& S, int lane) { return staged_bound(S, lane); }
    // One close pair a lane, both directions as the halves of a pair.
    static __device__ __forceinline__ void close(const PairArgs& A, const Slot<BornY>& S, long long* sa, int i, int j,
                                                 bool valid, int, int) {
        const float4 xi = S.i4[i], xj = S.j4[j];
        const float2 ai = S.i2[i], aj = S.ja[j];
        const float dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
        const f2 r2 = F2(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        const f2 rinv = rsqrt2_nr(r2), r = mul2(r2, rinv), rinv2 = mul2(rinv, rinv);
        const f2 a = make_float2(ai.x, aj.x), s = make_float2(aj.y, ai.y), s2 = mul2(s, s);
        const f2 y = mul2(s2, rinv2);
        f2 h = mul2(mul2(mul2(F2(0.5f), s2), s), mul2(mul2(rinv2, rinv2), gb_poly_g2(y)));
        const bool c0 = !far_ok(r.x, a.x + s.x, y.x), c1 = !far_ok(r.y, a.y + s.y, y.y);
        if (__any_sync(0xffffffffu, c0 || c1)) {
            const f2 hc = hct_closed2(r, rinv, a, s);
            h = make_float2(c0 ? hc.x : h.x, c1 ? hc.y : h.y);
        }
        if (!valid) return;
        if (!isfinite(h.x + h.y) && A.err) atomicCAS(A.err, 0, GB_ERR_NONFINITE);
        long long* const to[2] = {&sa[i], &S.jac[j]};
        const long long v[2] = {fix_i(h.x), fix_i(h.y)};
        shared_add(to, v);
    }
};

template <int NW, int DEG>
struct BornU {
    static constexpr int ATOMS = 64 * NW, NQ = Born::NQ, UNROLL = 2;
    struct I { f2 nx[NW], ny[NW], nz[NW], A[NW][DEG + 1]; };
    typedef float4 B;                                  // staged j values: x, y, z, A_0 | A_1 ...
    struct J { float acc; };
    struct Part { f2 s[NW]; };
    static __device__ __forceinline__ void load_j(const PairArgs& A, int64_t base, int n, int j, float4& v, B& b) {
        constexpr float g3[] = GB_G3, g2[] = GB_G2;
        float a, s, c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        load_xas(A, base, n, j, v.x, v.y, v.z, a, s);
        float h = 0.5f * s * s * s;
#pragma unroll
        for (int k = 0; k <= DEG; ++k) {
            c[k] = h * (DEG == 3 ? g3[k] : g2[k]);
            h *= s * s;
        }
        v.w = c[0];
        b = make_float4(c[1], c[2], c[3], 0.0f);
    }
    static __device__ __forceinline__ void load_i(const PairArgs& A, int64_t base, int n, int i0, int lane, I& st) {
#pragma unroll
        for (int q = 0; q < 2 * NW; ++q) {
            float4 v;
            B b;
            load_j(A, base, n, i0 + 32 * q + lane, v, b);
            const float c[4] = {v.w, b.x, b.y, b.z};
            set2(st.nx[q >> 1], q & 1, -v.x); set2(st.ny[q >> 1], q & 1, -v.y); set2(st.nz[q >> 1], q & 1, -v.z);
#pragma unroll
            for (int k = 0; k <= DEG; ++k) set2(st.A[q >> 1][k], q & 1, c[k]);
        }
    }
    static __device__ __forceinline__ void zero(J& j, Part& p) {
        j.acc = 0.0f;
#pragma unroll
        for (int q = 0; q < NW; ++q) p.s[q] = F2(0.0f);
    }
    static __device__ __forceinline__ void step(const PairArgs&, const I& i, float4 v, B b, J& j, Part& p) {
        const float c[4] = {v.w, b.x, b.y, b.z};
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const f2 dx = add2(F2(v.x), i.nx[q]), dy = add2(F2(v.y), i.ny[q]), dz = add2(F2(v.z), i.nz[q]);
            const f2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
            const f2 u = rcp2_approx(r2);
            const f2 u2 = mul2(u, u);
            f2 pj = F2(c[DEG]), pi = i.A[q][DEG];
#pragma unroll
            for (int k = DEG - 1; k >= 0; --k) {
                pj = fma2(u, pj, F2(c[k]));
                pi = fma2(u, pi, i.A[q][k]);
            }
            p.s[q] = fma2(u2, pj, p.s[q]);
            j.acc = fmaf(u2.y, pi.y, fmaf(u2.x, pi.x, j.acc));
        }
    }
    static __device__ __forceinline__ void rotate_acc(J& j, int src) { j.acc = shfl(j.acc, src); }
    static __device__ __forceinline__ void fold_i(const PairArgs&, long long* sa, int lane, const Part& p) {
#pragma unroll
        for (int q = 0; q < 2 * NW; ++q) sa[32 * q + lane] += fix_i(get2(p.s[q >> 1], q & 1));
    }
    static __device__ __forceinline__ void flush_j(const PairArgs& A, int64_t base, int n, int j, const J& st) {
        if (!isfinite(st.acc) && A.err) atomicCAS(A.err, 0, GB_ERR_NONFINITE);
        if (j < n) red_add(&A.I_acc[base + j], fix_i(st.acc));
    }
};

// --- chain rule ------------------------------------------------------------------------
// Force sums of a pass whose blocks add fr d to j and -fr d to i.
template <int NW>
struct ForceSums {
    struct J { float fx, fy, fz; };
    struct Part { f2 x[NW], y[NW], z[NW]; };
    static __device__ __forceinline__ void zero(J& j, Part& p) {
        j.fx = j.fy = j.fz = 0.0f;
#pragma unroll
        for (int q = 0; q < NW; ++q) p.x[q] = p.y[q] = p.z[q] = F2(0.0f);
    }
    static __device__ __forceinline__ void add(f2 fr, f2 dx, f2 dy, f2 dz, int q, J& j, Part& p) {
        p.x[q] = fma2(fr, dx, p.x[q]); p.y[q] = fma2(fr, dy, p.y[q]); p.z[q] = fma2(fr, dz, p.z[q]);
        j.fx = fmaf(fr.y, dx.y, fmaf(fr.x, dx.x, j.fx));
        j.fy = fmaf(fr.y, dy.y, fmaf(fr.x, dy.x, j.fy));
        j.fz = fmaf(fr.y, dz.y, fmaf(fr.x, dz.x, j.fz));
    }
    static __device__ __forceinline__ void rotate_acc(J& j, int src) {
        j.fx = shfl(j.fx, src); j.fy = shfl(j.fy, src); j.fz = shfl(j.fz, src);
    }
    template <int NQ>
    static __device__ __forceinline__ void fold(long long* sa, int lane, const Part& p) {
#pragma unroll
        for (int q = 0; q < 2 * NW; ++q) {
            long long* o = sa + (q >> 1) * 64 * NQ + 32 * (q & 1) + lane;
            o[0] -= fix(get2(p.x[q >> 1], q & 1));
            o[64] -= fix(get2(p.y[q >> 1], q & 1));
            o[128] -= fix(get2(p.z[q >> 1], q & 1));
        }
    }
    static __device__ __forceinline__ void flush(const PairArgs& A, int64_t g, const J& st, const long long* jac, int at) {
        red_add(&A.F_acc[g], fix(st.fx) + (jac ? jac[at] : 0));
        red_add(&A.F_acc[A.N + g], fix(st.fy) + (jac ? jac[32 + at] : 0));
        red_add(&A.F_acc[2 * A.N + g], fix(st.fz) + (jac ? jac[64 + at] : 0));
    }
    static __device__ __forceinline__ void flush_close(const PairArgs& A, int64_t g, const long long* jac, int j) {
        red_add(&A.F_acc[g], jac[j]);
        red_add(&A.F_acc[A.N + g], jac[32 + j]);
        red_add(&A.F_acc[2 * A.N + g], jac[64 + j]);
    }
    // a close pair's force fr d, exactly
    static __device__ __forceinline__ void add_close(long long* sa, long long* jac, int i, int j, float fr, float dx,
                                                     float dy, float dz) {
        const long long fx = fix(fr * dx), fy = fix(fr * dy), fz = fix(fr * dz);
        long long* const to[6] = {&sa[i], &sa[64 + i], &sa[128 + i], &jac[j], &jac[32 + j], &jac[64 + j]};
        const long long v[6] = {-fx, -fy, -fz, fx, fy, fz};
        shared_add(to, v);
    }
};

template <int NW>
struct ChainY : ForceSums<NW> {
    typedef ForceSums<NW> F;
    static constexpr bool CUT = false;
    static constexpr int ATOMS = 64 * NW, NQ = Chain::NQ, NJ = Chain::NJ, UNROLL = NW == 2 ? 1 : 4;
    struct I { f2 nx[NW], ny[NW], nz[NW], s2[NW], hs3[NW], c[NW]; };
    typedef float2 B;                                  // staged j values: x, y, z, s^2 | s^3 / 2, c
    static __device__ __forceinline__ void load(const PairArgs& A, int64_t base, int n, int i, float4& v, B& b, float2& as) {
        Chain::load_one(A, base, n, i, v.x, v.y, v.z, as.x, as.y, b.y);
        v.w = as.y * as.y;
        b.x = 0.5f * v.w * as.y;
    }
    static __device__ __forceinline__ void load_i(const PairArgs& A, int64_t base, int n, int i0, int lane, I& st,
                                                  float4* i4 = nullptr, float2* i2 = nullptr) {
#pragma unroll
        for (int q = 0; q < 2 * NW; ++q) {
            float4 v;
            B b;
            float2 as;
            load(A, base, n, i0 + 32 * q + lane, v, b, as);
            set2(st.nx[q >> 1], q & 1, -v.x); set2(st.ny[q >> 1], q & 1, -v.y); set2(st.nz[q >> 1], q & 1, -v.z);
            set2(st.s2[q >> 1], q & 1, v.w); set2(st.hs3[q >> 1], q & 1, b.x); set2(st.c[q >> 1], q & 1, b.y);
            if (i4) {
                i4[32 * q + lane] = make_float4(v.x, v.y, v.z, b.y);
                i2[32 * q + lane] = as;
            }
        }
    }
    static __device__ __forceinline__ void load_j(const PairArgs& A, int64_t base, int n, int j, float4& v, B& b) {
        float2 as;
        load(A, base, n, j, v, b, as);
    }
    template <int MODE = M_FULL, bool NEAR = false, class T = float>
    static __device__ __forceinline__ void step(const PairArgs&, const I& i, float4 v, B b, typename F::J& j,
                                                typename F::Part& p, Mask m = Mask{true, true}, T t = T(),
                                                unsigned bit = 0, unsigned* mk = nullptr) {
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const f2 dx = add2(F2(v.x), i.nx[q]), dy = add2(F2(v.y), i.ny[q]), dz = add2(F2(v.z), i.nz[q]);
            f2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
            if (MODE != M_FULL || NEAR) r2 = screen_r2<MODE, NEAR, true>(r2, m, t, bit, mk[0], mk[1]);
            const f2 u = rcp2_approx(r2);
            const f2 yj = mul2(F2(v.w), u), yi = mul2(i.s2[q], u);
            const f2 t1 = fma2(mul2(i.c[q], F2(b.x)), NW == 1 ? gb_poly_hn2(yj) : gb_poly_hf2(yj),
                               mul2(mul2(F2(b.y), i.hs3[q]), NW == 1 ? gb_poly_hn2(yi) : gb_poly_hf2(yi)));
            F::add(mul2(t1, mul2(u, mul2(u, u))), dx, dy, dz, q, j, p);
        }
    }
    static __device__ __forceinline__ void fold_i(const PairArgs&, long long* sa, int lane, const typename F::Part& p) {
        F::template fold<NQ>(sa, lane, p);
    }
    static __device__ __forceinline__ void flush_j(const PairArgs& A, int64_t base, int n, int j, const typename F::J& st,
                                                   const long long* jac = nullptr, int at = 0) {
        if (j < n) F::flush(A, base + j, st, jac, at);
    }
    static __device__ __forceinline__ float bound(const PairArgs&, const Slot<ChainY>& S, int lane) { return staged_bound(S, lane); }
    static __device__ __forceinline__ void close(const PairArgs& A, const Slot<ChainY>& S, long long* sa, int i, int j,
                                                 bool valid, int, int) {
        const float4 xi = S.i4[i], xj = S.j4[j];
        const float2 ai = S.i2[i], aj = S.ja[j];
        const float dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
        const f2 r2 = F2(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        const f2 rinv = rsqrt2_nr(r2), r = mul2(r2, rinv), rinv2 = mul2(rinv, rinv);
        const f2 a = make_float2(ai.x, aj.x), s = make_float2(aj.y, ai.y), s2 = mul2(s, s);
        const f2 y = mul2(s2, rinv2);
        f2 h = mul2(mul2(mul2(F2(0.5f), s2), s), mul2(mul2(rinv2, mul2(rinv2, rinv2)), gb_poly_h2(y)));
        const bool c0 = !far_ok(r.x, a.x + s.x, y.x), c1 = !far_ok(r.y, a.y + s.y, y.y);
        if (__any_sync(0xffffffffu, c0 || c1)) {
            const f2 hc = hct_closed_fr2(r, rinv, a, s);
            h = make_float2(c0 ? hc.x : h.x, c1 ? hc.y : h.y);
        }
        if (valid) F::add_close(sa, S.jac, i, j, fmaf(xi.w, h.x, S.jb[j].y * h.y), dx, dy, dz);
    }
};

template <int NW, int DEG>
struct ChainU : ForceSums<NW> {
    typedef ForceSums<NW> F;
    static constexpr int ATOMS = 64 * NW, NQ = Chain::NQ, UNROLL = NW == 2 ? 1 : 2;
    struct I { f2 nx[NW], ny[NW], nz[NW], c[NW], Bk[NW][DEG + 1]; };
    typedef float4 B;                                  // staged j values: x, y, z, c | B_k
    static __device__ __forceinline__ void load_j(const PairArgs& A, int64_t base, int n, int j, float4& v, B& b) {
        constexpr float h3[] = GB_H3, h2[] = GB_H2;
        float a, s, c[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        Chain::load_one(A, base, n, j, v.x, v.y, v.z, a, s, v.w);
        float h = 0.5f * s * s * s;
#pragma unroll
        for (int k = 0; k <= DEG; ++k) {
            c[k] = h * (DEG == 3 ? h3[k] : h2[k]);
            h *= s * s;
        }
        b = make_float4(c[0], c[1], c[2], c[3]);
    }
    static __device__ __forceinline__ void load_i(const PairArgs& A, int64_t base, int n, int i0, int lane, I& st) {
#pragma unroll
        for (int q = 0; q < 2 * NW; ++q) {
            float4 v;
            B b;
            load_j(A, base, n, i0 + 32 * q + lane, v, b);
            const float c[4] = {b.x, b.y, b.z, b.w};
            set2(st.nx[q >> 1], q & 1, -v.x); set2(st.ny[q >> 1], q & 1, -v.y); set2(st.nz[q >> 1], q & 1, -v.z);
            set2(st.c[q >> 1], q & 1, v.w);
#pragma unroll
            for (int k = 0; k <= DEG; ++k) set2(st.Bk[q >> 1][k], q & 1, c[k]);
        }
    }
    static __device__ __forceinline__ void step(const PairArgs&, const I& i, float4 v, B b, typename F::J& j, typename F::Part& p) {
        const float c[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const f2 dx = add2(F2(v.x), i.nx[q]), dy = add2(F2(v.y), i.ny[q]), dz = add2(F2(v.z), i.nz[q]);
            const f2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
            const f2 u = rcp2_approx(r2);
            f2 pj = F2(c[DEG]), pi = i.Bk[q][DEG];
#pragma unroll
            for (int k = DEG - 1; k >= 0; --k) {
                pj = fma2(u, pj, F2(c[k]));
                pi = fma2(u, pi, i.Bk[q][k]);
            }
            const f2 t = fma2(i.c[q], pj, mul2(F2(v.w), pi));
            F::add(mul2(t, mul2(u, mul2(u, u))), dx, dy, dz, q, j, p);
        }
    }
    static __device__ __forceinline__ void fold_i(const PairArgs&, long long* sa, int lane, const typename F::Part& p) {
        F::template fold<NQ>(sa, lane, p);
    }
    static __device__ __forceinline__ void flush_j(const PairArgs& A, int64_t base, int n, int j, const typename F::J& st) {
        if (j < n) F::flush(A, base + j, st, nullptr, 0);
    }
};

// --- GB + Coulomb forces and R dE/dR (no energies, no dE/dq) ----------------------------
// With Q = k_c q_i q_j, W = Q / f^3 (times the screened factor with salt) and
// E = exp(-D),
//   -(de/dr)/r = Q / r^3 + W (en_a E + en_b),   R de/dR = en_g W E (R_i R_j + r^2/4):
// the solvent constants sit in two uniform factors of the bracket and in one
// factor applied when a block's sums are folded.
template <int NW, int FLAGS>
struct EnergyW : ForceSums<NW> {
    typedef ForceSums<NW> F;
    static constexpr bool CUT = false;
    static constexpr int ATOMS = 64 * NW, NQ = Energy::NQ, NJ = Energy::NJ, UNROLL = NW == 2 ? 1 : 4;
    struct I { f2 nx[NW], ny[NW], nz[NW], Q[NW], R[NW], nh[NW]; };
    typedef float2 B;                                  // staged j values: x, y, z, q | R, h
    struct J : F::J { float dR; };
    struct Part : F::Part { f2 dR[NW]; };
    static __device__ __forceinline__ void load_j(const PairArgs& A, int64_t base, int n, int j, float4& v, B& b) {
        Energy::load_one(A, base, n, j, v.x, v.y, v.z, v.w, b.x, b.y);
    }
    static __device__ __forceinline__ void load(const PairArgs& A, int64_t base, int n, int i, float4& v, B& b, float2& as) {
        load_j(A, base, n, i, v, b);
        as = F2(0.0f);
    }
    static __device__ __forceinline__ void load_i(const PairArgs& A, int64_t base, int n, int i0, int lane, I& st,
                                                  float4* i4 = nullptr, float2* = nullptr) {
#pragma unroll
        for (int q = 0; q < 2 * NW; ++q) {
            float4 v;
            B b;
            load_j(A, base, n, i0 + 32 * q + lane, v, b);
            set2(st.nx[q >> 1], q & 1, -v.x); set2(st.ny[q >> 1], q & 1, -v.y); set2(st.nz[q >> 1], q & 1, -v.z);
            set2(st.Q[q >> 1], q & 1, v.w * A.kc);
            set2(st.R[q >> 1], q & 1, b.x);
            set2(st.nh[q >> 1], q & 1, -b.y);
            if (i4) i4[32 * q + lane] = v;
        }
    }
    static __device__ __forceinline__ void zero(J& j, Part& p) {
        F::zero(j, p);
        j.dR = 0.0f;
#pragma unroll
        for (int q = 0; q < NW; ++q) p.dR[q] = F2(0.0f);
    }
    template <int MODE = M_FULL, bool NEAR = false>
    static __device__ __forceinline__ void step(const PairArgs& A, const I& i, float4 v, B b, J& j, Part& p,
                                                Mask m = Mask{true, true}, float t = 0.0f, unsigned bit = 0,
                                                unsigned* mk = nullptr) {
#pragma unroll
        for (int q = 0; q < NW; ++q) {
            const f2 dx = add2(F2(v.x), i.nx[q]), dy = add2(F2(v.y), i.ny[q]), dz = add2(F2(v.z), i.nz[q]);
            f2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
            // pairs inside the repulsion's range keep their GB and Coulomb terms here
            if (MODE != M_FULL || NEAR) r2 = screen_r2<MODE, NEAR, false>(r2, m, t, bit, mk[0], mk[1]);
            const f2 rinv = rsqrt2(r2);
            const f2 e = ex22(mul2(r2, mul2(i.nh[q], F2(b.y))));          // exp(-D)
            const f2 RR = mul2(i.R[q], F2(b.x));
            const f2 fsq = fma2(RR, e, r2);
            const f2 finv = rsqrt2(fsq);
            const f2 Q = mul2(i.Q[q], F2(v.w));
            f2 W = mul2(mul2(Q, finv), mul2(finv, finv));
            if (FLAGS & EF_SALT) {
                // tF / k_c = 1 - (1 + kappa f) k, k = (eps_in / eps_out) exp(-kappa f)
                const f2 kf = mul2(F2(A.kappa), mul2(fsq, finv));
                const f2 k = ex22(fma2(F2(-LOG2E), kf, F2(A.salt_l2)));
                W = mul2(W, fma2(neg2(k), kf, add2(F2(1.0f), neg2(k))));
            }
            const f2 fr = fma2(W, fma2(F2(A.en_a), e, F2(A.en_b)), mul2(mul2(Q, rinv), mul2(rinv, rinv)));
            const f2 We = mul2(W, e), X = fma2(r2, F2(0.25f), RR);
            F::add(fr, dx, dy, dz, q, j, p);
            p.dR[q] = fma2(We, X, p.dR[q]);
            j.dR = fmaf(We.y, X.y, fmaf(We.x, X.x, j.dR));
        }
    }
    static __device__ __forceinline__ void rotate_acc(J& j, int src) {
        F::rotate_acc(j, src);
        j.dR = shfl(j.dR, src);
    }
    static __device__ __forceinline__ void fold_i(const PairArgs& A, long long* sa, int lane, const Part& p) {
        F::template fold<NQ>(sa, lane, p);
#pragma unroll
        for (int q = 0; q < 2 * NW; ++q)
            sa[(q >> 1) * 64 * NQ + 192 + 32 * (q & 1) + lane] += fix(A.en_g * get2(p.dR[q >> 1], q & 1));
    }
    static __device__ __forceinline__ void flush_j(const PairArgs& A, int64_t base, int n, int j, const J& st,
                                                   const long long* jac = nullptr, int at = 0) {
        if (j >= n) return;
        F::flush(A, base + j, st, jac, at);
        red_add(&A.dR_acc[base + j], fix(A.en_g * st.dR));
    }
    static __device__ __forceinline__ float bound(const PairArgs& A, const Slot<EnergyW>&, int) { return A.rep_sigma * A.rep_sigma; }
    // Soft repulsion of a pair more than one position apart in the chain.
    static __device__ __forceinline__ void close(const PairArgs& A, const Slot<EnergyW>& S, long long* sa, int i, int j,
                                                 bool valid, int i0, int jbase) {
        const float4 xi = S.i4[i], xj = S.j4[j];
        const float dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz)), rinv = rsqrt_ftz(r2);
        const int gap = i0 + i - (jbase + j);
        if (valid && (gap > 1 || gap < -1))
            F::add_close(sa, S.jac, i, j, 2.0f * A.rep_k * (A.rep_sigma - r2 * rinv) * rinv, dx, dy, dz);
    }
};

// --- walking the blocks -------------------------------------------------------------
// Tiles J0 + (set bits of `mask`) against the W::ATOMS atoms from i0 (a row or
// a row pair), every block far.  The tile's j data stand in shared memory, the tile twice, so that
// lane l reads atom (l + k) mod 32 of step k at a fixed offset from its own
// address: two vector loads a step, free of bank conflicts, in place of six to
// eight shuffles.  Only the partial sums rotate by shuffles.  A function of
// its own: inlined into the walk its loop carried a dozen register moves a
// step (registers of the other paths), 10 to 15 % of its time.  The shuffles
// at its head tell the compiler that the arguments are the warp's, not the lane's.
template <class W>
__device__ __noinline__ void walk_far(const PairArgs& A, int r, int i0, int J0, unsigned mask, int slot) {
    extern __shared__ __align__(16) unsigned char s_mem[];
    const int lane = threadIdx.x & 31;
    slot = __shfl_sync(0xffffffffu, slot, 0);
    r = __shfl_sync(0xffffffffu, r, 0);
    i0 = __shfl_sync(0xffffffffu, i0, 0);
    J0 = __shfl_sync(0xffffffffu, J0, 0);
    mask = __ballot_sync(0xffffffffu, (mask >> lane) & 1u);
    const int64_t base = A.atom_off[r];
    const int n = (int)(A.atom_off[r + 1] - base);
    long long* sa = (long long*)(s_mem + slot);
    float4* sj = (float4*)(sa + 2 * W::NQ * 64);
    if (W::ATOMS == 64) sa += ((i0 >> 6) & 1) * 64 * W::NQ;
    typename W::B* sb = (typename W::B*)(sj + 64);
    typename W::I is;
    float4 v;
    typename W::B b;
    int j = 32 * (J0 + __ffs(mask) - 1) + lane;
    W::load_j(A, base, n, j, v, b);                // before the i atoms: one memory latency for both
    W::load_i(A, base, n, i0, lane, is);
    const int next = (lane + 1) & 31;
    for (;;) {
        mask &= mask - 1;
        __syncwarp();
        sj[lane] = sj[32 + lane] = v;
        sb[lane] = sb[32 + lane] = b;
        __syncwarp();
        typename W::J js;
        typename W::Part p;
        W::zero(js, p);
#pragma unroll W::UNROLL
        for (int k = 0; k < 32; ++k) {
            W::step(A, is, sj[lane + k], sb[lane + k], js, p);
            W::rotate_acc(js, next);
        }
        W::fold_i(A, sa, lane, p);
        W::flush_j(A, base, n, j, js);
        if (!mask) break;
        j = 32 * (J0 + __ffs(mask) - 1) + lane;
        W::load_j(A, base, n, j, v, b);
    }
}

// Pairs b0 .. b0 + CLOSE_CAP - 1 of those noted in the lanes' masks (bit k of
// mx / my: the x / y half's atom against tile atom (lane + k) mod 32) into the
// warp's queue; before: pairs of the lanes below.
template <class W>
__device__ __forceinline__ void queue_close(const Slot<W>& S, unsigned mx, unsigned my, int before, int b0, int lane) {
    int pos = before - b0;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        unsigned m = h ? my : mx;
        while (m) {
            const int k = __ffs(m) - 1;
            m &= m - 1;
            if (pos >= 0 && pos < CLOSE_CAP) S.queue[pos] = (unsigned short)((32 * h + lane) | (((lane + k) & 31) << 6));
            ++pos;
        }
    }
    __syncwarp();
}
// Entries e .. e + 31 of a queue of cnt.
template <class W>
__device__ __forceinline__ void run_close(const PairArgs& A, const Slot<W>& S, int row, int e, int cnt, int i0, int jbase,
                                          int lane) {
    const int q = S.queue[min(e + lane, cnt - 1)];
    W::close(A, S, S.sa + row * 64 * W::NQ, q & 63, q >> 6, e + lane < cnt, i0, jbase);
}
// The pairs noted in the lanes' masks, 32 at a time.  Returns their number;
// with DEFER the last CLOSE_CAP of them at most stay in the queue, and the
// number of those is returned (see round_pass in fused.cu).
template <class W, bool DEFER>
__device__ __noinline__ int close_pairs(const PairArgs& A, int slot, int row, unsigned mx, unsigned my, int i0, int jbase) {
    const int lane = threadIdx.x & 31;
    slot = __shfl_sync(0xffffffffu, slot, 0);
    row = __shfl_sync(0xffffffffu, row, 0);
    const Slot<W> S(slot);
    const int own = __popc(mx) + __popc(my);
    int at = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, at, o);
        if (lane >= o) at += v;
    }
    const int total = __shfl_sync(0xffffffffu, at, 31);
    if (total == 0) return 0;
#pragma unroll
    for (int q = 0; q < W::NJ; ++q) S.jac[32 * q + lane] = 0;
    for (int b0 = 0; b0 < total; b0 += CLOSE_CAP) {
        queue_close(S, mx, my, at - own, b0, lane);
        const int cnt = min(CLOSE_CAP, total - b0);
        if (DEFER && b0 + CLOSE_CAP >= total) return cnt;
        for (int e = 0; e < cnt; e += 32) run_close(A, S, row, e, cnt, i0, jbase, lane);
        __syncwarp();
    }
    return total;
}

// The bound of a near tile: that of its boxes, or from the staged atoms.
template <class W, bool CUT = W::CUT>
struct NearBound { typedef float T; };
template <class W>
struct NearBound<W, true> { typedef Ring T; };
template <class W>
__device__ __forceinline__ typename NearBound<W>::T near_bound(const PairArgs& A, const Slot<W>& S, float t, float smax, int lane) {
    if constexpr (W::CUT) {
        if (!A.boxes) {
            t = staged_bound(S, lane);
            smax = fmaxf(S.ja[lane].y, fmaxf(S.i2[lane].y, S.i2[32 + lane].y));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) smax = fmaxf(smax, __shfl_xor_sync(0xffffffffu, smax, o));
        }
        return ring_of(A, t, smax);
    } else {
        return A.boxes ? t : W::bound(A, S, lane);
    }
}
template <class W, int MODE, bool NEAR, class T>
__device__ __forceinline__ void near_tile(const PairArgs& A, const typename W::I& is, const Slot<W>& S,
                                          typename W::J& js, typename W::Part& p, T t, unsigned* mk, int lane) {
    // a DX block pairs the x half with its own tile: only steps 1 .. 16 carry pairs
    constexpr int K0 = (MODE == M_DX) ? 1 : 0, K1 = (MODE == M_DX) ? 17 : 32;
    const int next = (lane + 1) & 31;
#pragma unroll W::UNROLL
    for (int k = K0; k < K1; ++k) {
        W::template step<MODE, NEAR>(A, is, S.j4[lane + k], S.jb[lane + k], js, p, step_mask<MODE>(k, lane), t, 1u << k, mk);
        W::rotate_acc(js, next);
    }
}

// Row K (64 atoms) against tiles J0 + (set bits of `todo`), near or diagonal;
// t: of lane c the bound below which pairs of column J0 + c are close.  DEFER
// (one column): the close pairs stay in the queue, their number is returned.
template <class W, bool CLOSE, bool DEFER = false>
__device__ __noinline__ int walk_near(const PairArgs& A, int r, int K, int J0, unsigned todo, float t, int slot,
                                      float smax = 0.0f) {
    const int lane = threadIdx.x & 31;
    slot = __shfl_sync(0xffffffffu, slot, 0);
    r = __shfl_sync(0xffffffffu, r, 0);
    K = __shfl_sync(0xffffffffu, K, 0);
    J0 = __shfl_sync(0xffffffffu, J0, 0);
    todo = __ballot_sync(0xffffffffu, (todo >> lane) & 1u);
    const int64_t base = A.atom_off[r];
    const int n = (int)(A.atom_off[r + 1] - base);
    const Slot<W> S(slot);
    long long* sa = S.sa + (K & 1) * 64 * W::NQ;
    typename W::I is;
    float4 v;
    typename W::B b;
    float2 as;
    W::load(A, base, n, 32 * (J0 + __ffs(todo) - 1) + lane, v, b, as);
    W::load_i(A, base, n, 64 * K, lane, is, S.i4, S.i2);
    for (;;) {
        const int c = __ffs(todo) - 1, J = J0 + c;
        todo &= todo - 1;
        __syncwarp();
        S.j4[lane] = S.j4[32 + lane] = v;
        S.jb[lane] = S.jb[32 + lane] = b;
        S.ja[lane] = as;
        __syncwarp();
        typename NearBound<W>::T tc = near_bound(A, S, __shfl_sync(0xffffffffu, t, c), __shfl_sync(0xffffffffu, smax, c), lane);
        typename W::J js;
        typename W::Part p;
        W::zero(js, p);
        unsigned mk[2] = {0u, 0u};
        int shift = 0;
        if (J >= 2 * K + 2) {
            near_tile<W, M_FULL, CLOSE>(A, is, S, js, p, tc, mk, lane);
        } else if (J == 2 * K) {
            near_tile<W, M_DX, CLOSE>(A, is, S, js, p, tc, mk, lane);
            shift = 17;                    // sums start at atom lane + 1 and leave rotated by 17
        } else {
            near_tile<W, M_DY, CLOSE>(A, is, S, js, p, tc, mk, lane);
        }
        W::fold_i(A, sa, lane, p);
        __syncwarp();
        const int n_close = CLOSE ? close_pairs<W, DEFER>(A, slot, K & 1, mk[0], mk[1], 64 * K, 32 * J) : 0;
        const int at = (lane + shift) & 31;
        W::flush_j(A, base, n, 32 * J + at, js, !DEFER && n_close ? S.jac : nullptr, at);
        if (DEFER) return n_close;
        if (!todo) return 0;
        W::load(A, base, n, 32 * (J0 + __ffs(todo) - 1) + lane, v, b, as);
    }
}

// The same row by the general pair code of the energy pass: blocks that
// straddle the pair cutoff (EF_STRADDLE), and passes that want energies or dE/dq.
template <class P, int FLAGS>
__device__ __noinline__ void walk_general(const PairArgs& A, int r, int K, int J0, unsigned todo, int slot) {
    extern __shared__ __align__(16) unsigned char s_mem[];
    const int lane = threadIdx.x & 31, next = (lane + 1) & 31;
    const int64_t base = A.atom_off[r];
    const int n = (int)(A.atom_off[r + 1] - base), nb = (n + 31) >> 5;
    long long* sa = (long long*)(s_mem + slot) + (K & 1) * 64 * P::NQ;
    typename P::IState is;
    P::load_i(A, base, n, 64 * K, lane, is);
    while (todo) {
        const int J = J0 + __ffs(todo) - 1;
        todo &= todo - 1;
        const bool dx = (J == 2 * K);      // see run_tile: entry / exit rotation of a DX block
        typename P::JState js;
        P::load_j(A, base, n, 32 * J + ((lane + (dx ? 1 : 0)) & 31), js);
        typename P::Part ip;
        ip.zero();
        const BlockInfo bi = block_info(A, r, K, J, nb);
        if (J >= 2 * K + 2) {
            if (!(FLAGS & EF_STRADDLE) && bi.far) run_tile<P, FLAGS, M_FULL, true>(A, is, js, ip, bi, 64 * K, 32 * J, lane, next);
            else run_tile<P, FLAGS, M_FULL, false>(A, is, js, ip, bi, 64 * K, 32 * J, lane, next);
        } else if (dx) {
            run_tile<P, FLAGS, M_DX, false>(A, is, js, ip, bi, 64 * K, 32 * J, lane, next);
        } else {
            run_tile<P, FLAGS, M_DY, false>(A, is, js, ip, bi, 64 * K, 32 * J, lane, next);
        }
        P::fold_i(is, sa, lane, ip);
        P::flush_j(A, base, n, 32 * J + ((lane + (dx ? 17 : 0)) & 31), js);
    }
    P::flush_sums(A, r, lane, is);
}

// --- blocks that straddle the Born-radius cutoff --------------------------------------
// Pairs wholly inside the cutoff take the near form, pairs past its reach are
// left out, and the close ones and those whose sphere may cross it (see Ring)
// are queued and evaluated exactly, 32 at a time.  The restricted integrals
// cost ten times the near form and the sphere about the cutoff is thin (two
// times the largest s), but nearly every step of 64 pairs has a pair in it:
// taking the restricted form for all lanes of such steps bound the Born and
// chain passes, 641 and 980 us at 100,000 atoms and 12 A against 483 and 733
// now (25 A: 1600 and 2550 against 1186 and 1759).  Queueing all pairs in
// reach and none in the near form: 767 and 965 (25 A: 1856 and 2668).
struct BornCut : BornY<1> {
    static constexpr bool CUT = true;
    static __device__ __forceinline__ void close(const PairArgs& A, const Slot<BornCut>& S, long long* sa, int i, int j,
                                                 bool valid, int, int) {
        const float4 xi = S.i4[i], xj = S.j4[j];
        const float2 ai = S.i2[i], aj = S.ja[j];
        const float dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
        const f2 r2 = F2(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        const f2 rinv = rsqrt2_nr(r2), r = mul2(r2, rinv);
        const f2 h = hct_cut_dir2(r, rinv, make_float2(ai.x, aj.x), make_float2(aj.y, ai.y), A.rgbmax);
        if (!valid) return;
        if (!isfinite(h.x + h.y) && A.err) atomicCAS(A.err, 0, GB_ERR_NONFINITE);
        long long* const to[2] = {&sa[i], &S.jac[j]};
        const long long v[2] = {fix_i(h.x), fix_i(h.y)};
        shared_add(to, v);
    }
};
struct ChainCut : ChainY<1> {
    static constexpr bool CUT = true;
    static __device__ __forceinline__ void close(const PairArgs& A, const Slot<ChainCut>& S, long long* sa, int i, int j,
                                                 bool valid, int, int) {
        const float4 xi = S.i4[i], xj = S.j4[j];
        const float2 ai = S.i2[i], aj = S.ja[j];
        const float dx = xj.x - xi.x, dy = xj.y - xi.y, dz = xj.z - xi.z;
        const f2 r2 = F2(fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        const f2 rinv = rsqrt2_nr(r2), r = mul2(r2, rinv);
        const f2 h = hct_cut_dir_fr2(r, rinv, make_float2(ai.x, aj.x), make_float2(aj.y, ai.y), A.rgbmax);
        if (valid) F::add_close(sa, S.jac, i, j, fmaf(xi.w, h.x, S.jb[j].y * h.y), dx, dy, dz);
    }
};
template <class P>
struct CutForm { typedef BornCut W; };
template <>
struct CutForm<Chain> { typedef ChainCut W; };

// Form of a block (see above) from the bounds of its boxes.
template <class P, int FLAGS>
__device__ __forceinline__ int row_tier(const PairArgs& A, const BoxPair& b) {
    if (P::RADIUS_CUT) {
        const float as = b.amax + b.smax, s2 = b.smax * b.smax;
        if (b.rmin2 < as * as || s2 > GB_POLY_YFAR * b.rmin2) return 0;
        const float y3 = P::CHAIN ? GB_Y_H3 : GB_Y_G3, y2 = P::CHAIN ? GB_Y_H2 : GB_Y_G2;
        return s2 <= y2 * b.rmin2 ? 3 : (s2 <= y3 * b.rmin2 ? 2 : 1);
    }
    return (!(FLAGS & EF_REP) || b.rmin2 >= A.rep_sigma * A.rep_sigma) ? 1 : 0;
}

// Far tiles of a row (NW 1) or a row pair (NW 2).
template <class P, int FLAGS, int NW>
__device__ __forceinline__ void run_far(int tier, const PairArgs& A, int r, int i0, int J0, unsigned mask, int slot) {
    if constexpr (!P::RADIUS_CUT) {
        walk_far<EnergyW<NW, FLAGS & EF_SALT>>(A, r, i0, J0, mask, slot);
    } else if constexpr (P::CHAIN) {
        if (NW == 2 && tier == 3) walk_far<ChainU<2, 2>>(A, r, i0, J0, mask, slot);
        else if (tier >= 2) walk_far<ChainU<NW, 3>>(A, r, i0, J0, mask, slot);
        else walk_far<ChainY<NW>>(A, r, i0, J0, mask, slot);
    } else {
        if (NW == 2 && tier == 3) walk_far<BornU<2, 2>>(A, r, i0, J0, mask, slot);
        else if (tier >= 2) walk_far<BornU<NW, 3>>(A, r, i0, J0, mask, slot);
        else walk_far<BornY<NW>>(A, r, i0, J0, mask, slot);
    }
}
// The form of a pass's near blocks, and whether it has close pairs at all.
template <class P, int FLAGS>
struct NearForm {
    typedef EnergyW<1, FLAGS & EF_SALT> W;
    static constexpr bool CLOSE = (FLAGS & EF_REP) != 0;
};
template <int FLAGS>
struct NearForm<Born, FLAGS> {
    typedef BornY<1> W;
    static constexpr bool CLOSE = true;
};
template <int FLAGS>
struct NearForm<Chain, FLAGS> {
    typedef ChainY<1> W;
    static constexpr bool CLOSE = true;
};
template <class P, int FLAGS, bool DEFER = false>
__device__ __forceinline__ int run_near(const PairArgs& A, int r, int K, int J0, unsigned todo, float t, int slot) {
    return walk_near<typename NearForm<P, FLAGS>::W, NearForm<P, FLAGS>::CLOSE, DEFER>(A, r, K, J0, todo, t, slot);
}

// Work of replica r is walked as row pairs P = 0 .. ceil(nb/4) - 1 (nb tiles
// of 32 atoms; 128 atoms each, rows K = 2P and 2P + 1), each over the tiles
// (columns) J = 4P .. nb-1.  A warp task is (replica, 4P + rows, J, columns):
// rows is 1 or 2 for one row of the pair alone, 3 for both.  Columns where
// both rows are far (and inside every cutoff) are evaluated 128 x 32 by
// the task that holds row 0, the others row by row in 64 x 32 blocks.  Replicas
// of up to SMALL_TILES tiles run every block 64 x 32: their pass ends with the
// slowest warps, and half the block halves what the last ones still do.  Every
// choice depends on the replica and the block alone, so that results do not
// depend on how the work is cut or on what else is in the batch.  SMALL: the
// kernel for batches of small replicas alone (no 128 x 32 code, fewer registers).
//
// The tile boxes of 32 columns are classified at once, one column a lane.
// slot is the byte offset of the warp's shared memory (see Slot).  Loads of
// data that kernels rewrite (coordinates, radii, chain factors, boxes) go
// through L2 (ld.global.cg): a persistent launch reads them again after other
// SMs changed them, and L1 is not coherent.
template <class P, int FLAGS, bool SMALL = false>
__device__ __forceinline__ void walk_task(const PairArgs& A, const int4 t, int slot, int lane) {
    extern __shared__ __align__(16) unsigned char s_mem[];
    long long* sa = (long long*)(s_mem + slot);
#pragma unroll
    for (int q = 0; q < 4 * P::NQ; ++q) sa[32 * q + lane] = 0;
    __syncwarp();
    // energies and dE/dq have the general pair code alone, blocks that
    // straddle a cutoff too (without tile boxes every block counts as one)
    constexpr bool GENERAL = !P::RADIUS_CUT && (FLAGS & (EF_ENERGY | EF_PHI)) != 0;
    constexpr bool CUT = (FLAGS & EF_CUT) != 0;
    const int r = t.x, PR = t.y >> 2, sel = t.y & 3;
    const int64_t base = A.atom_off[r];
    const int n = (int)(A.atom_off[r + 1] - base);
    const int nb = (n + 31) >> 5;
    unsigned used = 0;
    for (int s0 = 0; s0 < t.w; s0 += 32) {
        const int J0 = t.z + s0, m = min(32, t.w - s0), J = J0 + lane;
        int tier[2] = {0, 0};
        bool in[2] = {true, true}, straddle[2] = {CUT, CUT};
        float bound[2] = {0.0f, 0.0f}, smax[2] = {0.0f, 0.0f};
        if (A.boxes && lane < m) {
            const int t0 = A.tile_off[r];
            const float4 jl = __ldcg(&A.boxes[2 * (t0 + J)]), jh = __ldcg(&A.boxes[2 * (t0 + J) + 1]);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (4 * PR + 2 * h >= nb) continue;
                float4 ih;
                const float4 il = row_box_lo(A, t0, 2 * PR + h, nb, &ih);
                const BoxPair b = box_pair(il, ih, jl, jh);
                tier[h] = row_tier<P, FLAGS>(A, b);
                bound[h] = P::RADIUS_CUT ? close_bound(b.amax, b.smax) : A.rep_sigma * A.rep_sigma;
                if (CUT) cut_class(A, P::RADIUS_CUT, b, in[h], straddle[h]);
                smax[h] = b.smax;
            }
        }
        const unsigned all = m == 32 ? 0xffffffffu : (1u << m) - 1u;
        unsigned wide = 0;
        if (!GENERAL && !SMALL && nb > SMALL_TILES) {
            const int both = (J >= 4 * PR + 4 && (!CUT || (in[0] && in[1] && !straddle[0] && !straddle[1])))
                                 ? min(tier[0], tier[1]) : 0;
#pragma unroll
            for (int k = P::RADIUS_CUT ? 3 : 1; k > 0; --k) {
                const unsigned w = __ballot_sync(0xffffffffu, both == k) & all;
                if (w && (sel & 1)) run_far<P, FLAGS, 2>(k, A, r, 128 * PR, J0, w, slot);
                wide |= w;
            }
            if (wide && (sel & 1)) used |= 3;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int K = 2 * PR + h;
            unsigned todo = all & ~wide;
            if (CUT) todo &= __ballot_sync(0xffffffffu, in[h]);
            if (J0 < 2 * K) todo &= ~((1u << (2 * K - J0)) - 1u);      // tiles before the row's diagonal
            if (!((sel >> h) & 1) || 2 * K >= nb || !todo) continue;
            used |= 1u << h;
            const unsigned st = CUT ? todo & __ballot_sync(0xffffffffu, straddle[h]) : 0u, rest = todo & ~st;
            if constexpr (CUT && P::RADIUS_CUT) {
                if (st) walk_near<typename CutForm<P>::W, true>(A, r, K, J0, st, bound[h], slot, smax[h]);
            } else if constexpr (CUT) {
                if (st) walk_general<P, FLAGS | EF_STRADDLE>(A, r, K, J0, st, slot);
            }
            if constexpr (GENERAL) {
                if (rest) walk_general<P, FLAGS>(A, r, K, J0, rest, slot);
            } else {
                const bool diag = J < 2 * K + 2;
                const unsigned near = rest & __ballot_sync(0xffffffffu, diag || tier[h] == 0);
                const unsigned far1 = rest & __ballot_sync(0xffffffffu, !diag && tier[h] == 1), far2 = rest & ~(near | far1);
                if (near) run_near<P, FLAGS>(A, r, K, J0, near, bound[h], slot);
                if (far1) run_far<P, FLAGS, 1>(1, A, r, 64 * K, J0, far1, slot);
                if (far2) run_far<P, FLAGS, 1>(2, A, r, 64 * K, J0, far2, slot);
            }
        }
    }
    __syncwarp();
#pragma unroll
    for (int h = 0; h < 2; ++h)
        if ((used >> h) & 1) P::flush_i(A, base, n, 128 * PR + 64 * h, lane, sa + h * 64 * P::NQ);
}


// --- the pair-pass kernel --------------------------------------------------------
// One warp per task.  MINB caps the registers so that two, three or four
// 256-thread blocks fit on an SM (128, 80, 64 a thread: more warps, more spills).
template <class P, int FLAGS, int MINB, bool SMALL>
__global__ void __launch_bounds__(256, MINB) k_pairs(const __grid_constant__ PairArgs A, const int4* __restrict__ tasks, int n_tasks) {
    pdl_enter();
    const int lane = threadIdx.x & 31;
    // the shuffle tells the compiler that the task is the same for the whole
    // warp: uniform loops and addresses, 3 to 5 % of a distant block
    const int w = __shfl_sync(0xffffffffu, (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)), 0);
    if (w >= n_tasks) return;
    walk_task<P, FLAGS, SMALL>(A, tasks[w], (threadIdx.x >> 5) * WARP_SMEM<P>, lane);
}

// The same pass over a task list built on the device (cutoff passes: the
// in-range blocks of k_block_list): the number of tasks is ctr[count_idx],
// and warps take tasks one at a time from the queue head ctr[head_idx] until
// it runs dry, so the grid only needs to fill the GPU.
template <class P, int FLAGS, int MINB>
__global__ void __launch_bounds__(256, MINB) k_pairs_dyn(const __grid_constant__ PairArgs A, const int4* __restrict__ tasks, int* ctr,
                                                         int count_idx, int head_idx) {
    pdl_enter();
    const int lane = threadIdx.x & 31, slot = (threadIdx.x >> 5) * WARP_SMEM<P>;
    const int n_tasks = __ldcg(&ctr[count_idx]);
    for (;;) {
        int w = 0;
        if (lane == 0) w = atomicAdd(&ctr[head_idx], 1);
        w = __shfl_sync(0xffffffffu, w, 0);
        if (w >= n_tasks) break;
        walk_task<P, FLAGS>(A, __ldcg(&tasks[w]), slot, lane);
    }
}

// Launch of pass policy P over a task list.
template <class P, int FLAGS, bool SMALL>
cudaError_t launch_pass_cap(const PairArgs& a, const TaskList& t, int cap, int wpb, cudaStream_t s) {
    wpb = fit_warps<P>(wpb);
    const size_t smem = (size_t)wpb * WARP_SMEM<P>;
    const dim3 g((t.n_tasks + wpb - 1) / wpb), b(32 * wpb);
    if (cap >= 4) return launch_pdl(k_pairs<P, FLAGS, 4, SMALL>, g, b, smem, s, a, t.d_tasks, t.n_tasks);
    if (cap >= 3) return launch_pdl(k_pairs<P, FLAGS, 3, SMALL>, g, b, smem, s, a, t.d_tasks, t.n_tasks);
    return launch_pdl(k_pairs<P, FLAGS, 2, SMALL>, g, b, smem, s, a, t.d_tasks, t.n_tasks);
}
template <class P, int FLAGS>
cudaError_t launch_pass(const PairArgs& a, const TaskList& t, int cap, int wpb, cudaStream_t s) {
    if (t.n_tasks == 0) return cudaSuccess;
    if constexpr (P::RADIUS_CUT || !(FLAGS & (EF_ENERGY | EF_PHI))) {
        if (t.small) return launch_pass_cap<P, FLAGS, true>(a, t, cap, wpb, s);
    }
    return launch_pass_cap<P, FLAGS, false>(a, t, cap, wpb, s);
}

// Bounding boxes of every 32-atom tile (one warp per tile): lo.xyz with the
// largest a = rho - offset, hi.xyz with the largest screened radius s.
__device__ __forceinline__ void tile_box_warp(const PairArgs& A, int M, int t, int lane) {
    int lo = 0, hi = M;               // replica r with tile_off[r] <= t < tile_off[r+1]
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (A.tile_off[mid] <= t) lo = mid;
        else hi = mid;
    }
    const int r = lo;
    const int64_t base = A.atom_off[r];
    const int n = (int)(A.atom_off[r + 1] - base);
    const int i = 32 * (t - A.tile_off[r]) + lane;
    float x = 0.0f, y = 0.0f, z = 0.0f, q = 0.0f, am = 0.0f, sm = 0.0f;
    if (i < n) {
        const float4 p = __ldcg(&A.xyzq[base + i]);
        const float2 rs = A.rad[base + i];
        x = p.x; y = p.y; z = p.z; q = p.w;
        am = rs.x - A.offset;
        sm = rs.y * am;
    }
    tile_box_store(A.boxes, t, i < n, x, y, z, am, sm, q, A.err);
}


}  // namespace gbk
