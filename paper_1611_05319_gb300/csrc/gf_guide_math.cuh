// The guide field's value of one pixel in pairs of FP32 numbers.
//
// The value is defined in FP64, (t̂ * exp(-d^2 / (2 eta^2))) * w rounded once to FP32
// (so that a CPU in FP64 gives the same field), but FP64 runs at a 64th of the FP32
// rate here, and about 60 FP64 operations a pixel bound the kernel.  guide_value forms the same value as an
// unevaluated sum of two FP32 numbers (error-free transformations: Knuth's two-sum,
// the FMA two-product; Dekker, Numer. Math. 18, 1971) with a bound on its relative
// error, about 2^-37, and says so when the bound leaves the rounding to FP32 open: about
// one pixel in 2,800 (and none of 40 million random ones was rounded differently), which is then evaluated in FP64.  Every pixel therefore gets
// the FP64 evaluation's FP32 value, bit for bit.
#pragma once

#include <math.h>
#include <stdint.h>

#ifdef __CUDACC__
#define GM_FN __host__ __device__ __forceinline__
#else
#define GM_FN static inline
#endif

namespace gf {

// exp(-j / 32) for j = 0 .. GUIDE_EXP - 1, as pairs: d <= 3 eta keeps the exponent
// below 4.5 (and a little, where FP32 decides the cut)
constexpr int GUIDE_EXP = 148;
struct GuideExp {
    float h[GUIDE_EXP], l[GUIDE_EXP];
};

// One segment: start a, v = b - a, 1/|v|^2, v/|v|, all but a as pairs, and the spline's
// weight.  The search for the nearest segment reads the first five numbers (its 1/|v|^2
// is formed in FP32, il32; -1 at points that start no segment).
struct alignas(16) SegPair {
    float ax, ay, vxh, vyh;
    float il32, vxl, vyl, ilh;
    float ill, txh, txl, tyh;
    float tyl, sw, pad[2];
};

struct Pair {
    float h, l;
};

GM_FN float gm_fma(float a, float b, float c) { return fmaf(a, b, c); }
#ifdef __CUDA_ARCH__
GM_FN float gm_add(float a, float b) { return __fadd_rn(a, b); }
GM_FN float gm_mul(float a, float b) { return __fmul_rn(a, b); }
#else
GM_FN float gm_add(float a, float b) { return a + b; }
GM_FN float gm_mul(float a, float b) { return a * b; }
#endif
GM_FN float gm_sub(float a, float b) { return gm_add(a, -b); }

// a + b exactly
GM_FN Pair two_sum(float a, float b)
{
    Pair r;
    r.h = gm_add(a, b);
    const float t = gm_sub(r.h, a);
    r.l = gm_add(gm_sub(a, gm_sub(r.h, t)), gm_sub(b, t));
    return r;
}
// a + b exactly for |a| >= |b|
GM_FN Pair quick_sum(float a, float b)
{
    Pair r;
    r.h = gm_add(a, b);
    r.l = gm_sub(b, gm_sub(r.h, a));
    return r;
}
// (a.h + a.l) (b.h + b.l) to about 2^-46 relative
GM_FN Pair pair_mul(Pair a, Pair b)
{
    const float p = gm_mul(a.h, b.h);
    const float e = gm_fma(a.h, b.h, -p);
    return quick_sum(p, gm_add(e, gm_fma(a.h, b.l, gm_mul(a.l, b.h))));
}
GM_FN Pair pair_add(Pair a, Pair b)
{
    const Pair s = two_sum(a.h, b.h);
    return quick_sum(s.h, gm_add(s.l, gm_add(a.l, b.l)));
}
GM_FN Pair pair_neg(Pair a)
{
    Pair r;
    r.h = -a.h;
    r.l = -a.l;
    return r;
}
// the FP64 number as a pair
GM_FN Pair pair_of(double v)
{
    Pair r;
    r.h = (float)v;
    r.l = (float)(v - (double)r.h);
    return r;
}

// Rounds the pair to FP32 when every value within rel * |o| of it rounds alike.
GM_FN bool pair_round(Pair o, float rel, float &out)
{
    const float m = gm_mul(fabsf(o.h), rel);
    const float a = gm_add(o.h, gm_add(o.l, m)), b = gm_add(o.h, gm_sub(o.l, m));
    out = a;
    return a == b && fabsf(a) > 1e-25f;
}

// The value at pixel (x, y) of segment s; k2 = 1 / (2 eta^2) as a pair, ieta = 1 / eta.
// False when the FP64 evaluation has to decide.
GM_FN bool guide_value(float x, float y, const SegPair &s, Pair k2, float ieta, const GuideExp &T, float &ox, float &oy)
{
    const Pair wx = two_sum(x, -s.ax), wy = two_sum(y, -s.ay);  // exact
    const Pair vx = {s.vxh, s.vxl}, vy = {s.vyh, s.vyl}, il = {s.ilh, s.ill};
    const float far = fabsf(wx.h) + fabsf(wy.h);
    // which part of the segment is nearest: FP32 is off by at most 2^-21 |w| / |v| here,
    // and on either side of an end the two forms differ by (that |v|)^2 at most
    const float t = gm_mul(gm_fma(wx.h, vx.h, gm_mul(wy.h, vy.h)), il.h);
    const float band = 4.8e-7f * gm_fma(far, sqrtf(il.h), 1.0f);
    Pair d2;
    if (t > 0.0f && t < 1.0f) {
        // distance to the line: |w x v| / |v|
        const Pair c = pair_add(pair_mul(wx, vy), pair_neg(pair_mul(wy, vx)));
        d2 = pair_mul(pair_mul(c, c), il);
    } else {
        Pair ux = wx, uy = wy;
        if (t >= 1.0f) {
            ux = pair_add(wx, pair_neg(vx));
            uy = pair_add(wy, pair_neg(vy));
        }
        d2 = pair_add(pair_mul(ux, ux), pair_mul(uy, uy));
    }
    const Pair e = pair_mul(d2, k2);  // minus the exponent
    // exp(-e) = exp(-j / 32) exp(r), |r| <= 1 / 64 and a little
    const float jf = gm_sub(gm_fma(e.h, 32.0f, 12582912.0f), 12582912.0f);
    const int j = (int)jf;
    if (!(jf >= 0.0f && jf < (float)GUIDE_EXP)) return false;
    const Pair r = two_sum(gm_fma(jf, 0.03125f, -e.h), -e.l);  // the first difference is exact
    const float p = gm_mul(r.h, r.h), pe = gm_fma(r.h, r.h, -p);
    const float q = gm_mul(gm_mul(r.h, p), gm_fma(r.h, gm_fma(r.h, 1.0f / 120.0f, 1.0f / 24.0f), 1.0f / 6.0f));
    const float lo = gm_add(r.l, gm_fma(0.5f, pe, gm_fma(r.h, r.l, q)));
    Pair u = quick_sum(r.h, gm_mul(0.5f, p));  // exp(r) - 1
    u = quick_sum(u.h, gm_add(u.l, lo));
    const Pair th = {T.h[j], T.l[j]};
    const Pair tu = pair_mul(th, u);
    Pair ev = quick_sum(th.h, tu.h);
    ev = quick_sum(ev.h, gm_add(ev.l, gm_add(th.l, tu.l)));
    // relative error: 2^-38 for the chain above, the distance's 2^-45 |w| px times the
    // exponent's slope d / eta^2 <= 3 / eta, and near an end of the segment the other
    // form's difference
    float rel = gm_fma(gm_mul(far, ieta), 3.0f * 2.85e-14f, 7.3e-12f);
    if (fabsf(t) < band || fabsf(gm_sub(t, 1.0f)) < band) rel = gm_fma(gm_mul(far, far), k2.h * 9.2e-13f, rel);
    const Pair tx = {s.txh, s.txl}, ty = {s.tyh, s.tyl};
    Pair gx = pair_mul(tx, ev), gy = pair_mul(ty, ev);
    if (s.sw != 1.0f) {
        const Pair w = {s.sw, 0.0f};
        gx = pair_mul(gx, w);
        gy = pair_mul(gy, w);
    }
    // lengths for which the products' errors may leave FP32's range go the other way
    bool sure = il.h > 1e-10f && il.h < 1e10f && rel < 1e-8f;
    // an axis-parallel segment: a zero component stays the zero that FP64 gives
    if (s.txh == 0.0f) ox = gm_mul(s.txh, s.sw);
    else sure = pair_round(gx, rel, ox) && sure;
    if (s.tyh == 0.0f) oy = gm_mul(s.tyh, s.sw);
    else sure = pair_round(gy, rel, oy) && sure;
    return sure;
}

}  // namespace gf
