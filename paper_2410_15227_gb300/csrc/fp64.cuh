// FP64 primitives of the closed form (k_map_fp64, k_map_fp64_flagged) with few
// FP64 instructions.  GB300 issues an FP64 warp instruction every ~20 cycles
// per SM, 1/64 of the FP32 rate, so the closed form is bound by their number:
// range reduction and table look-up run on the integer pipe, and the tail of
// each series, whose relative weight is below 2^-28 of the result's scale, in
// FP32.  Each function is within about 2 ulp of its largest argument's scale
// (absolute for the angle and the logarithm, which enter the weight as terms
// of size up to 1): counted in FP64 instructions, sqrt64 6, log_ratio 15,
// angle64 13.
//
// Method: table-driven argument reduction (P. T. P. Tang, "Table-driven
// implementation of the logarithm function in IEEE floating-point arithmetic",
// ACM TOMS 16, 1990) with the Taylor series of log(1 + f) and atan(d) on the
// reduced argument; square root and quotients by Newton's iteration from the
// hardware's approximate reciprocal (square root) of an FP64 number (PTX
// rcp/rsqrt.approx.ftz.f64, about 20 bits).
#pragma once

#include <cuda_runtime.h>

#include "split.cuh"

namespace em {

// atan(k/64), k = 0..64
__device__ const double kAtanTab[65] = {
    0.0, 0.015623728620476831, 0.031239833430268277, 0.046840712915969654,
    0.06241880999595735, 0.0779666338315423, 0.09347678115858947, 0.10894195698986579,
    0.12435499454676144, 0.13970887428916365, 0.15499674192394097, 0.1702119252854744,
    0.18534794999569476, 0.2003985538258785, 0.21535769969773805, 0.23021958727684372,
    0.24497866312686414, 0.2596296294082575, 0.2741674511196588, 0.2885873618940774,
    0.3028848683749714, 0.31705575320914703, 0.3310960767041321, 0.34500217720710513,
    0.35877067027057225, 0.3723984466767542, 0.38588266939807375, 0.39922076957525254,
    0.4124104415973873, 0.42544963737004227, 0.43833655985795783, 0.4510696559885235,
    0.4636476090008061, 0.4760693303227612, 0.48833395105640554, 0.5004408131472942,
    0.5123894603107377, 0.5241796287829132, 0.5358112379604637, 0.5472843809874369,
    0.5585993153435624, 0.5697564534829784, 0.5807563535676704, 0.5915997103351114,
    0.6022873461349642, 0.6128202021652414, 0.6231993299340659, 0.6334258829691446,
    0.6435011087932844, 0.6534263411807619, 0.6632029927060933, 0.6728325475937632,
    0.6823165548747481, 0.6916566218531999, 0.7008544078844502, 0.7099116184635249,
    0.7188299996216245, 0.7276113326265107, 0.7362574289814281, 0.7447701257160751,
    0.7531512809621944, 0.7614027698055784, 0.7695264804056583, 0.7775243103733478,
    0.7853981633974483};
// {r, -log(r)} with r = 1/(1 + (2i + 1)/128) rounded to 24 fraction bits:
// |m r - 1| < 1/128 for m in [1 + i/64, 1 + (i + 1)/64]
__device__ const double kLogTab[64][2] = {
    {0.9922480583190918, 0.007782144167345254}, {0.9770992398262024, 0.02316705602190537},
    {0.9624060392379761, 0.0383188391564274}, {0.9481481313705444, 0.053244532213941355},
    {0.9343065619468689, 0.06795066982474966}, {0.9208633303642273, 0.08244364639367177},
    {0.9078013896942139, 0.09672965812351915}, {0.8951048851013184, 0.11081437751616108},
    {0.882758617401123, 0.12470348222624754}, {0.8707482814788818, 0.138402343348216},
    {0.8590604066848755, 0.15191603736922912}, {0.8476821184158325, 0.16524957382662975},
    {0.8366013169288635, 0.17840764583128618}, {0.8258064389228821, 0.19139486836645206},
    {0.8152866363525391, 0.2042155265275298}, {0.805031418800354, 0.21687397275955023},
    {0.7950310707092285, 0.22937408243839452}, {0.7852760553359985, 0.2417199601702098},
    {0.7757575511932373, 0.2539152416459315}, {0.7664670944213867, 0.2659635112442357},
    {0.7573964595794678, 0.2778684379649404}, {0.7485380172729492, 0.2896332851324621},
    {0.7398843765258789, 0.3012613529299038}, {0.7314285635948181, 0.31275572071410657},
    {0.7231638431549072, 0.32411946679156683}, {0.7150837779045105, 0.33535557125779936},
    {0.7071823477745056, 0.3464667286963225}, {0.6994535326957703, 0.3574559163958201},
    {0.6918919086456299, 0.368325536944321}, {0.6844919919967651, 0.3790783333771956},
    {0.6772486567497253, 0.38971678140800936}, {0.6701570749282837, 0.40024315388246445},
    {0.6632124185562134, 0.4106599501309782}, {0.656410276889801, 0.4209692634448239},
    {0.6497461795806885, 0.4311734853074682}, {0.643216073513031, 0.44127457151508487},
    {0.6368159055709839, 0.4512746674225232}, {0.6305418610572815, 0.46117573235163795},
    {0.6243902444839478, 0.47097971428746843}, {0.6183574795722961, 0.48068854284992935},
    {0.6124401688575745, 0.49030402483243624}, {0.6066350936889648, 0.49982783230354705},
    {0.6009389758110046, 0.5092618873543081}, {0.5953488349914551, 0.518607767933336},
    {0.5898617506027222, 0.527867090552165}, {0.5844748616218567, 0.5370415073407391},
    {0.5791855454444885, 0.5461323942916368}, {0.573991060256958, 0.5551414572490838},
    {0.5688889026641846, 0.5640701140704163}, {0.5638766288757324, 0.5729197945399797},
    {0.5589519739151001, 0.5816917238021388}, {0.5541125535964966, 0.5903874475334989},
    {0.54935622215271, 0.5990081915087285}, {0.5446808338165283, 0.6075552818895098},
    {0.5400843620300293, 0.616029925644289}, {0.5355648398399353, 0.6244333136232646},
    {0.5311203598976135, 0.6327666169513138}, {0.5267489552497864, 0.6410312096889155},
    {0.5224489569664001, 0.6492279899316105}, {0.5182186365127563, 0.6573580475626508},
    {0.5140562057495117, 0.6654226697979941}, {0.5099601745605469, 0.6734226454098448},
    {0.5059288740158081, 0.6813591847610332}, {0.501960813999176, 0.6892332220998273}};

__device__ __forceinline__ double rcp_seed(double x)
{
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}

__device__ __forceinline__ double rsqrt_seed(double x)
{
    double r;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    return r;
}

// x cut to FP32 (towards zero) on the bits; 0 below FP32's normal range,
// its largest binade above it.  For seeds, tables' indexes and series' tails.
__device__ __forceinline__ float f32_cut(double x)
{
    const unsigned h = (unsigned)__double2hiint(x), e = (h >> 20) & 0x7ffu;
    const unsigned m = __funnelshift_l((unsigned)__double2loint(x), h & 0x7fffffffu, 3) - 0x40000000u;
    const unsigned v = e < 897u ? 0u : (e > 1150u ? 0x7f000000u : (m & 0x7fffffffu));
    return __uint_as_float(v | (h & 0x80000000u));
}

// sqrt(x), x >= 0 (0 below 2^-1000)
__device__ __forceinline__ double sqrt64(double x)
{
    const double y = rsqrt_seed(x);
    double g = x * y;
    double h = __hiloint2double(__double2hiint(y) - 0x100000, __double2loint(y));   // y / 2
    const double r = fma(-g, h, 0.5);
    g = fma(g, r, g);
    h = fma(h, r, h);
    g = fma(fma(-g, g, x), h, g);
    return __double2hiint(x) < (23 << 20) ? 0.0 : g;
}

// log(num / den) for normal num, den > 0: with their significands n, d in
// [1, 2), n/d = x / (1 + e), x = n s, 1 + e = d s, s the approximate
// reciprocal of d (|e| below about 2^-17), and log x = k log 2 - log r + log(1 + f) with
// m r = 1 + f from the table.
__device__ __forceinline__ double log_ratio(double num, double den, const double (*tab)[2])
{
    const int hn = __double2hiint(num), hd = __double2hiint(den);
    const double sn = __hiloint2double((hn & 0xfffff) | 0x3ff00000, __double2loint(num));
    const double sd = __hiloint2double((hd & 0xfffff) | 0x3ff00000, __double2loint(den));
    const double s = rcp_seed(sd);
    const double x = sn * s, e = fma(sd, s, -1.0);
    const double l1 = fma(-0.5 * e, e, e);
    const int hx = __double2hiint(x), i = (hx >> 14) & 63;
    const double m = __hiloint2double((hx & 0xfffff) | 0x3ff00000, __double2loint(x));
    const double f = fma(m, tab[i][0], -1.0);
    const float ff = f32_cut(f);
    const double t = f64_of(fmaf(ff, fmaf(ff, fmaf(ff, 1.f / 7.f, -1.f / 6.f), 0.2f), -0.25f));
    const double p = fma(f * f, fma(f, fma(f, t, 1.0 / 3.0), -0.5), f);
    const double k = f64_of((float)((hx >> 20) - 1023 + (hn >> 20) - (hd >> 20)));   // (float)0 becomes 2^-127, far below the sum
    // log 2 to FP64 and the rest
    return fma(k, 0.69314718055994530942, tab[i][1]) + fma(k, 2.3190468138462996e-17, p - l1);
}

// The angle of the vector (x, y) in [-pi, pi] (0 for the zero vector): with
// t = min/max of |x|, |y| and c = k/64 the nearest such fraction (from FP32),
// atan t = atan c + atan d, d = (min - c max)/(max + c min).
__device__ __forceinline__ double angle64(double y, double x, const double *tab)
{
    const int hx = __double2hiint(x), hy = __double2hiint(y);
    const int ux = hx & 0x7fffffff, uy = hy & 0x7fffffff;
    const bool swap = uy > ux;   // on the high words: t may exceed 1 by 2^-20
    const double ax = __hiloint2double(ux, __double2loint(x)), ay = __hiloint2double(uy, __double2loint(y));
    const double lo = swap ? ax : ay, hi = swap ? ay : ax;
    const int ulo = swap ? ux : uy, uhi = swap ? uy : ux;
    // t to FP32 from the high words: significands in [1, 2), the exponents' difference applied to the quotient's
    const int de = (ulo >> 20) - (uhi >> 20);   // <= 0
    const float sl = __int_as_float(((ulo & 0xfffff) << 3) | 0x3f800000), sh = __int_as_float(((uhi & 0xfffff) << 3) | 0x3f800000);
    const float kf = de < -20 ? 0.f : rintf(64.f * __int_as_float((127 + de) << 23) * __fdividef(sl, sh));
    const int k = min((int)kf, 64);
    const double c = f64_of(fminf(kf, 64.f) * 0.015625f);   // 0 becomes 2^-127: no effect
    const double nn = fma(-c, hi, lo), dd = fma(c, lo, hi);
    double r = rcp_seed(dd);
    r = fma(fma(-dd, r, 1.0), r, r);
    const double q = nn * r;
    const double d = fma(fma(-dd, q, nn), r, q);
    const double w = d * d;
    const float wf = f32_cut(w);
    const double t = f64_of(fmaf(wf, fmaf(wf, 1.f / 9.f, -1.f / 7.f), 0.2f));
    const double a = tab[k] + fma(d * w, fma(w, t, -1.0 / 3.0), d);
    const bool neg = (hx < 0) != swap;   // the angle from the nearer axis is subtracted
    const double base = swap ? 1.57079632679489661923 : (hx < 0 ? 3.14159265358979323846 : 0.0);
    // first quadrant: a, pi/2 - a; second: pi - a, pi/2 + a
    const double v = base + __hiloint2double(__double2hiint(a) ^ ((neg ? 1 : 0) << 31), __double2loint(a));
    const double s = __hiloint2double(__double2hiint(v) ^ (hy & 0x80000000), __double2loint(v));
    return uhi == 0 ? 0.0 : s;
}

}  // namespace em
