// iod_ff_cost.cuh -- one epoch's angle residuals in split FP32 arithmetic.
//
// The FP64 form (arctangent, arcsine, square root and division of Eqs. 5-9) takes about
// 300 FP64 warp instructions at 64 cycles, as much as two FP64 RK4 steps and, once the
// steps run in split words, as all the steps of a paper-scale interval together.  Here
// the line of sight is turned by the observed angles, whose sines and cosines are tabled
// in two words, so that each residual is the angle of a vector:
//     b_alpha = atan2(sin a~ rho_x - cos a~ rho_y, cos a~ rho_x + sin a~ rho_y),
//     b_beta  = atan2(sin b~ rho_xy - cos b~ rho_z, cos b~ rho_xy + sin b~ rho_z),
// already reduced to [-pi, pi].  Both angles go through one two-word arctangent in packed
// pairs: with c = i/128 nearest to the ratio of the smaller to the larger component,
// atan = atan(c) + atan(t), t = (a - c b)/(b + c a) at most 1/256, a short series.  The
// result is within 2.6e-14 rad, and for residuals below 0.1 rad within 1.5e-14, 1.4e-15 root
// mean square (the line of sight itself, at FP64's positions 1e-4 to 1e-3 LU apart: 1e-13 to
// 1e-12 rad).
#pragma once

#include "iod_ff.cuh"

namespace iod {
namespace ff {

// One epoch: sines and cosines of the observed angles, and the chief's position as the
// split step carries it (three words; x from the Moon; NaN where it holds FP64 values
// instead: the FP64 form decides there).  ok = 0: the observed elevation
// lies outside [-pi/2, pi/2], where the difference of Eq. 8 is not that angle.
struct alignas(16) Epoch {
    float2 ka, kal;        // (cos a~, sin a~): leading and low words
    float2 kb, kbl;        // (cos b~, sin b~)
    float2 ph, pl, pc;     // chief x, y
    float zh, zl, zc;      // chief z
    int ok;
    float far2;            // squared length of the line of sight up to which the split residuals are taken
    float pad;
};
static_assert(sizeof(Epoch) == 80, "Epoch layout");

// far2 of an epoch that FP64 propagation reaches in n steps.  The split residuals err by 1.4e-15
// rad (root mean square, up to 0.1 rad; the FP64 form by 7e-17, growing as the elevation's
// secant), which the rounding of the positions hides for near deputies only: one rounding of
// the deputy's and the chief's is 1.4e-15 rad at 1/32 LU, and n steps' at least sqrt(n) times
// that.
IOD_HD float far_limit(float n) { return mul(add(1.0f, n), 1.0f / 1024.0f); }

// atan(i / 128), i = 0..128, in two words
struct AtanTable {
    float h[129], l[129];
};

constexpr double atan_series(double x)      // |x| < 0.42
{
    double s = 0.0, p = x;
    for (int k = 0; k < 60; ++k) {
        s += (k & 1 ? -p : p) / (2 * k + 1);
        p *= x * x;
    }
    return s;
}

constexpr AtanTable make_atan_table()
{
    AtanTable T{};
    for (int i = 0; i <= 128; ++i) {
        const double c = i / 128.0;
        const double a = c < 0.42 ? atan_series(c) : 0.78539816339744830962 - atan_series((1.0 - c) / (1.0 + c));
        T.h[i] = (float)a;
        T.l[i] = (float)(a - (double)T.h[i]);
    }
    return T;
}

#ifdef __CUDACC__
static __device__ const AtanTable kAtan = make_atan_table();
IOD_HD float atan_h(int i) { return __ldg(&kAtan.h[i]); }
IOD_HD float atan_l(int i) { return __ldg(&kAtan.l[i]); }
// the hardware's estimate of 1/x
IOD_HD float rcp_est(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
IOD_HD float fabs1(float x) { return fabsf(x); }
IOD_HD int nearest(float x) { return __float2int_rn(x); }
#else
static const AtanTable kAtan = make_atan_table();
IOD_HD float atan_h(int i) { return kAtan.h[i]; }
IOD_HD float atan_l(int i) { return kAtan.l[i]; }
IOD_HD float rcp_est(float x) { return IOD_RCP_EST(x); }
IOD_HD float fabs1(float x) { return fabsf(x); }
IOD_HD int nearest(float x) { return (int)lrintf(x); }
#endif

// One vector's smaller component a and larger one m, both made positive, the nearest
// tabled ratio c with its arctangent, and what that is taken from or added to (base).
struct AngleParts {
    float a, al, m, ml, c, th, tl, base, basel, sg;
};

IOD_HD AngleParts angle_parts(float u, float ul, float v, float vl)
{
    AngleParts r;
    const float au = fabs1(u), av = fabs1(v);
    const bool neg = u < 0.0f, sw = av > au;
    const float aul = neg ? -ul : ul, avl = v < 0.0f ? -vl : vl;
    r.a = sw ? au : av;
    r.al = sw ? aul : avl;
    r.m = sw ? av : au;
    r.ml = sw ? avl : aul;
    int i = nearest(mul(mul(r.a, rcp_est(r.m)), 128.0f));
    i = i < 0 ? 0 : (i > 128 ? 128 : i);
    r.c = mul((float)i, 0.0078125f);
    r.th = atan_h(i);
    r.tl = atan_l(i);
    r.base = sw ? 0x1.921fb6p+0f : (neg ? 0x1.921fb6p+1f : 0.0f);          // pi/2, pi
    r.basel = sw ? -0x1.777a5cp-25f : (neg ? -0x1.777a5cp-24f : 0.0f);
    r.sg = sw != neg ? -1.0f : 1.0f;
    return r;
}

// Magnitude of the angle of (u, v), two words each, for two vectors at once.
IOD_HD void angle2(float2 uh, float2 ul, float2 vh, float2 vl, float2 &bh, float2 &bl)
{
    const AngleParts A = angle_parts(uh.x, ul.x, vh.x, vl.x), B = angle_parts(uh.y, ul.y, vh.y, vl.y);
    const float2 ah = mk2(A.a, B.a), al = mk2(A.al, B.al), mh = mk2(A.m, B.m), ml = mk2(A.ml, B.ml);
    const float2 c = mk2(A.c, B.c), th = mk2(A.th, B.th), tl = mk2(A.tl, B.tl), sg = mk2(A.sg, B.sg);
    const float2 base = mk2(A.base, B.base), basel = mk2(A.basel, B.basel);
    // t = (a - c m) / (m + c a); a - c mh is exact (c mh lies within a factor of two of it)
    const float2 p = mul2(c, mh), pe = fma2(c, mh, neg2(p)), nc = neg2(c);
    float2 nh, nl, dh, dl;
    fast_two_sum2(sub2(ah, p), sub2(fma2(nc, ml, al), pe), nh, nl);
    const float2 q = mul2(c, ah), qe = fma2(c, al, fma2(c, ah, neg2(q)));
    fast_two_sum2(mh, q, dh, dl);
    dl = add2(dl, add2(qe, ml));
    const float2 r = mk2(rcp_est(dh.x), rcp_est(dh.y));
    const float2 t0 = mul2(nh, r), nt = neg2(t0);
    const float2 t1 = mul2(r, add2(fma2(nt, dh, nh), fma2(nt, dl, nl)));
    float2 t, tlo;
    fast_two_sum2(t0, t1, t, tlo);
    // atan(t) = t - t^3/3 + t^5/5 - t^7/7
    const float2 z = mul2(t, t);
    float2 s = fma2(z, bc2(-0.14285715f), bc2(0.2f));
    s = mul2(z, fma2(z, s, bc2(-0.33333334f)));
    const float2 lo = fma2(t, s, add2(tl, tlo));
    float2 e, f, g;
    fast_two_sum2(th, t, e, f);
    f = add2(f, lo);
    // quadrant: base +- that
    fast_two_sum2(base, mul2(sg, e), bh, g);
    bl = add2(g, fma2(sg, f, basel));
}

// (k.x p + k.y q, k.y p - k.x q): the vector (p, q) turned by the angle of k
IOD_HD void turn(float2 k, float2 kl, float ph, float pl, float qh, float ql, float2 &h, float2 &l)
{
    const float2 m = mk2(k.y, -k.x), ml = mk2(kl.y, -kl.x);
    const float2 a = mul2(k, bc2(ph)), b = mul2(m, bc2(qh));
    float2 al = fma2(k, bc2(ph), neg2(a)), bl = fma2(m, bc2(qh), neg2(b));
    al = fma2(kl, bc2(ph), fma2(k, bc2(pl), al));
    bl = fma2(ml, bc2(qh), fma2(m, bc2(ql), bl));
    float2 s, e;
    two_sum2(a, b, s, e);
    two_sum2(s, add2(e, add2(al, bl)), h, l);      // the leading words may have cancelled
}

// sqrt(ah + al) in two words
IOD_HD void sqrt2w(float ah, float al, float &h, float &l)
{
    float y = rsqrt_est(ah);
    y = ffma(mul(0.5f, y), ffma(mul(-ah, y), y, 1.0f), y);
    const float g = mul(ah, y);
    const float d = mul(mul(0.5f, y), add(ffma(-g, g, ah), al));
    fast_two_sum(g, d, h, l);
}

// Residual magnitudes of the epoch for the line of sight (x, y packed; z), two words each:
// ba, bb in two words, and rho_xy.  r2: |rho|^2 (one word).  False where the split form
// does not apply (a line of sight along the pole or out of FP32's range, an observed
// elevation beyond the poles) or is the less exact one (far2 of the epoch, and less than
// 83 degrees from the equator): the FP64 form decides there.
IOD_HD bool residuals(const Epoch &E, float2 h, float2 l, float zh, float zl, float2 &bh, float2 &bl, float &rxyh,
                      float &rxyl)
{
    const float2 q = mul2(h, h), qe = fma2(add2(h, h), l, fma2(h, h, neg2(q)));
    float s, se;
    two_sum(q.x, q.y, s, se);
    se = add(se, add(qe.x, qe.y));
    const float r2 = ffma(zh, zh, s);
    if (!(s >= 1e-28f && r2 <= 1e28f) || !E.ok || (r2 > E.far2 && mul(64.0f, s) >= r2)) return false;
    sqrt2w(s, se, rxyh, rxyl);
    float2 ah, al, ch, cl;
    turn(E.ka, E.kal, h.x, l.x, h.y, l.y, ah, al);
    turn(E.kb, E.kbl, rxyh, rxyl, zh, zl, ch, cl);
    angle2(mk2(ah.x, ch.x), mk2(al.x, cl.x), mk2(ah.y, ch.y), mk2(al.y, cl.y), bh, bl);
    return true;
}

// The line of sight of a state in flight from the epoch's chief, two words.
IOD_HD void sight(const Epoch &E, const State &S, float2 &h, float2 &l, float &zh, float &zl)
{
    float2 d, e, f, g, r;
    two_sum2(S.ph, neg2(E.ph), d, e);
    two_sum2(S.pl, neg2(E.pl), f, g);
    two_sum2(d, f, h, r);
    l = add2(add2(r, e), add2(g, sub2(S.pc, E.pc)));
    float dz, ez, fz, gz, rz;
    two_sum(S.zh, -E.zh, dz, ez);
    two_sum(S.zl, -E.zl, fz, gz);
    two_sum(dz, fz, zh, rz);
    zl = add(add(rz, ez), add(gz, sub(S.zc, E.zc)));
}

// |rho| in two words from rho_xy and z.
IOD_HD void range2w(float rh, float rl, float zh, float zl, float &h, float &l)
{
    const float2 v = mk2(rh, zh), vl = mk2(rl, zl);
    const float2 q = mul2(v, v), qe = fma2(add2(v, v), vl, fma2(v, v, neg2(q)));
    float s, se;
    two_sum(q.x, q.y, s, se);
    sqrt2w(s, add(se, add(qe.x, qe.y)), h, l);
}

}  // namespace ff
}  // namespace iod
