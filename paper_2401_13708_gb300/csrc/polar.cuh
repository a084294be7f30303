// polar.cuh -- the quantised polar coordinates of a key in float32 pairs.
//
// A key needs floor(u 2^29) of a radial and an angular coordinate that are
// defined by float64 operations (square root, atan2, divisions).  The float64
// pipe runs two lanes a cycle per SM, so those operations bounded the key
// kernels (make_keys 113 us at N = 1M); here the coordinates are computed in
// float32 hi/lo pairs to about 2^-44 and read off in fixed point, and where
// one lies within 2^-13 of a quantisation step the caller evaluates the
// float64 definition instead, so the keys are the same.  Compiles for the
// host too.
#pragma once

#include "bits.cuh"

namespace hts {

#ifdef __CUDA_ARCH__
#define HTS_TABLE static __device__ const
#else
#define HTS_TABLE static const
#endif

// atan(k / 64) in turns, times 2^52
HTS_TABLE long long kAtanTable[65] = {
    0ll, 11198622188162ll, 22391779856454ll, 33574024467030ll,
    44739939329418ll, 55884155234104ll, 67001365742401ll, 78086342025269ll,
    89133947149786ll, 100139149719183ll, 111097036780798ll, 122002825925530ll,
    132851876512487ll, 143639699963097ll, 154361969079894ll, 165014526356345ll,
    175593391255098ll, 186094766442951ll, 196515042981259ll, 206850804480476ll,
    217098830236791ll, 227256097377358ll, 237319782048240ll, 247287259686024ll,
    257156104419798ll, 266924087655091ll, 276589175895242ll, 286149527858622ll,
    295603490952174ll, 304949597162959ll, 314186558429756ll, 323313261556491ll,
    332328762728241ll, 341232281689067ll, 350023195638838ll, 358701032903775ll,
    367265466432638ll, 375716307167393ll, 384053497333959ll, 392277103695211ll,
    400387310804930ll, 408384414297927ll, 416268814248049ll, 424041008622372ll,
    431701586856582ll, 439251223573313ll, 446690672462190ll, 454020760337434ll,
    461242381386143ll, 468356491617896ll, 475364103523931ll, 482266280952042ll,
    489064134201383ll, 495758815339580ll, 502351513742990ll, 508843451859526ll,
    515235881192220ll, 521530078500619ll, 527727342216161ll, 533828989066887ll,
    539836350906148ll, 545750771739455ll, 551573604943114ll, 557306210667968ll,
    562949953421312ll,
};

struct Pair32 {  // hi + lo
    float h, l;
};

__host__ __device__ __forceinline__ long long float_to_ll(float x)  // to nearest; |x| < 2^62
{
#ifdef __CUDA_ARCH__
    return __float2ll_rn(x);
#else
    return llrintf(x);
#endif
}

__host__ __device__ __forceinline__ float rcp_near(float x)  // 1 / x within 2^-22
{
#ifdef __CUDA_ARCH__
    return __frcp_rn(x);
#else
    return 1.0f / x;
#endif
}

// a b rounded, whatever is done with it: a product whose rounding error is taken
// off elsewhere must not be fused into a sum
__host__ __device__ __forceinline__ float product(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    volatile float p = a * b;
    return p;
#endif
}

__host__ __device__ __forceinline__ Pair32 pair_of(double x)
{
    Pair32 p;
    split_f32(x, p.h, p.l);
    return p;
}

// The top kLevels bits of a fixed-point coordinate v (52 fraction bits, [0, 1)):
// false within 2^-13 of a step (and outside [0, 1)).
__host__ __device__ __forceinline__ bool quantise_fixed(long long v, int levels, uint64_t &q)
{
    const int drop = 52 - levels;
    const long long part = v & ((1ll << drop) - 1ll), margin = 1ll << (drop - 13);
    q = (uint64_t)(v >> drop);
    return v >= 0 && v < (1ll << 52) && part >= margin && part <= (1ll << drop) - margin;
}

// floor(u 2^levels) of u = (atan2(y, x) in [0, 2 pi)) / 2 pi.
//   t = min / max of |x|, |y|; c = k / 64 next to t; atan t = atan c + atan z with
//   z = (min - c max) / (max + c min), |z| < 2^-6.9; atan z = z (1 + s), s =
//   -z^2 / 3 + z^4 / 5 - z^6 / 7 in float32.  Errors in turns: z and its sums
//   2^-51, s 2^-47, the table 2^-53; a step's margin is 2^-42.
__host__ __device__ __forceinline__ bool quantise_angle(double x, double y, int levels, uint64_t &q)
{
    const Pair32 px = pair_of(x), py = pair_of(y);
    const bool nx = px.h < 0.0f, ny = py.h < 0.0f;
    const Pair32 ax{nx ? -px.h : px.h, nx ? -px.l : px.l}, ay{ny ? -py.h : py.h, ny ? -py.l : py.l};
    const bool swap = ay.h > ax.h;
    const Pair32 mx = swap ? ay : ax, mn = swap ? ax : ay;
    if (!(mx.h > 1e-25f && mx.h < 1e25f)) return false;
    const float t0 = mn.h * rcp_near(mx.h);
    const int k = (int)(t0 * 64.0f + 0.5f);  // 0 .. 64
    const float c = (float)k * (1.0f / 64.0f);
    // numerator min - c max (the first difference is exact: c max is within half of min, or 0)
    const float p = product(c, mx.h), pe = fmaf(c, mx.h, -p);
    const float a = mn.h - p, b = mn.l - pe - c * mx.l;
    const float nh = a + b, nl = b - (nh - a);
    // denominator max + c min
    const float p2 = product(c, mn.h), p2e = fmaf(c, mn.h, -p2);
    const float dh = mx.h + p2, dl = ((mx.h - dh) + p2) + p2e + mx.l + c * mn.l;
    const float rc = rcp_near(dh);
    const float q0 = nh * rc;
    const float q1 = (fmaf(-q0, dh, nh) + (nl - q0 * dl)) * rc;
    const float w = q0 * q0;
    const float s = w * fmaf(w, fmaf(w, -1.0f / 7.0f, 0.2f), -1.0f / 3.0f);
    // z (1 + s) / 2 pi
    constexpr float kInvH = 0.15915493667125702f, kInvL = 6.4206382432985265e-09f;  // 1 / 2 pi
    const float g = q0 * kInvH;
    const float ge = fmaf(q0, kInvH, -g) + q0 * kInvL + q1 * kInvH + g * s;
    constexpr float kOne = 4503599627370496.0f;  // 2^52
#ifdef __CUDA_ARCH__
    long long v = __ldg(kAtanTable + k);
#else
    long long v = kAtanTable[k];
#endif
    v += float_to_ll(g * kOne) + float_to_ll(ge * kOne);
    constexpr long long kTurn = 1ll << 52;
    if (swap) v = kTurn / 4 - v;
    if (nx) v = kTurn / 2 - v;
    if (ny) v = kTurn - v;
    return quantise_fixed(v, levels, q);
}

// The radial coordinate c of |y|^2 = n2 (its square root, or (1 + n2) / (1 - n2)
// for equal areas) as a pair, to about 2^-44 of itself; false outside its range.
__host__ __device__ __forceinline__ bool radial_pair(double n2, bool area, Pair32 &c)
{
    if (!area) {
        const Pair32 p = pair_of(n2);
        if (!(p.h > 1e-25f && p.h < 1.0f)) return false;
        const float s = sqrtf(p.h);                                         // rounded to nearest
        const float e = (fmaf(-s, s, p.h) + p.l) * (0.5f * rcp_near(s));    // the rest, to 2^-22 of itself
        c.h = s + e;
        c.l = e - (c.h - s);
        return true;
    }
    const Pair32 num = pair_of(1.0 + n2), den = pair_of(1.0 - n2);
    if (!(den.h > 1e-12f)) return false;
    const float r = rcp_near(den.h);
    const float q0 = num.h * r;
    const float q1 = (fmaf(-q0, den.h, num.h) + (num.l - q0 * den.l)) * r;
    c.h = q0 + q1;
    c.l = q1 - (c.h - q0);
    return true;
}

// Bounds of the radial coordinate for quantise_radius: the lower one and
// 2^52 / (hi - lo) as pairs; usable where hi - lo >= hi / 4 (the error of
// (c - lo) / (hi - lo), about 2^-45 hi / (hi - lo), then stays below half of a
// step's margin of 2^-42).
struct RadialBounds {
    Pair32 lo, scale;
    bool usable;
};

__host__ __device__ __forceinline__ RadialBounds radial_bounds(double lo, double hi)
{
    RadialBounds b;
    const double span = hi - lo;
    b.usable = span > 0.0 && span >= hi * 0.25 && span < 1e12 && span > 1e-12;
    b.lo = pair_of(lo);
    b.scale = pair_of(b.usable ? 4503599627370496.0 / span : 0.0);
    return b;
}

// floor(u 2^levels) of u = (c - lo) / (hi - lo).
__host__ __device__ __forceinline__ bool quantise_radius(double n2, bool area, const RadialBounds &b, int levels,
                                                         uint64_t &q)
{
    Pair32 c;
    if (!b.usable || !radial_pair(n2, area, c)) return false;
    const float d = c.h - b.lo.h, t = d - c.h;  // two-sum of c.h and -lo.h
    const float de = (c.h - (d - t)) + (-b.lo.h - t) + (c.l - b.lo.l);
    const float g = d * b.scale.h;
    const float ge = fmaf(d, b.scale.h, -g) + d * b.scale.l + de * b.scale.h;
    return quantise_fixed(float_to_ll(g) + float_to_ll(ge), levels, q);
}

#undef HTS_TABLE

}  // namespace hts
