// FP64 arithmetic counted in pipe slots.  A warp's FP64 instruction (conversions to and from FP32 and
// comparisons among them) holds a sub-partition's FP64 pipe for 64 cycles on GB300, so the functions
// here trade FP64 instructions for integer ones, table look-ups and the hardware's approximations.
#pragma once

#include <cuda_runtime.h>

namespace scivr {

__device__ __constant__ const double2 kExp2Table[64] = {   // 2^(j / 64), leading and trailing word
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.02c9a3e778061p+0, -0x1.19083535b085dp-56},
    {0x1.059b0d3158574p+0, 0x1.d73e2a475b465p-55}, {0x1.0874518759bc8p+0, 0x1.186be4bb284ffp-57},
    {0x1.0b5586cf9890fp+0, 0x1.8a62e4adc610bp-54}, {0x1.0e3ec32d3d1a2p+0, 0x1.03a1727c57b53p-59},
    {0x1.11301d0125b51p+0, -0x1.6c51039449b3ap-54}, {0x1.1429aaea92de0p+0, -0x1.32fbf9af1369ep-54},
    {0x1.172b83c7d517bp+0, -0x1.19041b9d78a76p-55}, {0x1.1a35beb6fcb75p+0, 0x1.e5b4c7b4968e4p-55},
    {0x1.1d4873168b9aap+0, 0x1.e016e00a2643cp-54}, {0x1.2063b88628cd6p+0, 0x1.dc775814a8495p-55},
    {0x1.2387a6e756238p+0, 0x1.9b07eb6c70573p-54}, {0x1.26b4565e27cddp+0, 0x1.2bd339940e9d9p-55},
    {0x1.29e9df51fdee1p+0, 0x1.612e8afad1255p-55}, {0x1.2d285a6e4030bp+0, 0x1.0024754db41d5p-54},
    {0x1.306fe0a31b715p+0, 0x1.6f46ad23182e4p-55}, {0x1.33c08b26416ffp+0, 0x1.32721843659a6p-54},
    {0x1.371a7373aa9cbp+0, -0x1.63aeabf42eae2p-54}, {0x1.3a7db34e59ff7p+0, -0x1.5e436d661f5e3p-56},
    {0x1.3dea64c123422p+0, 0x1.ada0911f09ebcp-55}, {0x1.4160a21f72e2ap+0, -0x1.ef3691c309278p-58},
    {0x1.44e086061892dp+0, 0x1.89b7a04ef80d0p-59}, {0x1.486a2b5c13cd0p+0, 0x1.3c1a3b69062f0p-56},
    {0x1.4bfdad5362a27p+0, 0x1.d4397afec42e2p-56}, {0x1.4f9b2769d2ca7p+0, -0x1.4b309d25957e3p-54},
    {0x1.5342b569d4f82p+0, -0x1.07abe1db13cadp-55}, {0x1.56f4736b527dap+0, 0x1.9bb2c011d93adp-54},
    {0x1.5ab07dd485429p+0, 0x1.6324c054647adp-54}, {0x1.5e76f15ad2148p+0, 0x1.ba6f93080e65ep-54},
    {0x1.6247eb03a5585p+0, -0x1.383c17e40b497p-54}, {0x1.6623882552225p+0, -0x1.bb60987591c34p-54},
    {0x1.6a09e667f3bcdp+0, -0x1.bdd3413b26456p-54}, {0x1.6dfb23c651a2fp+0, -0x1.bbe3a683c88abp-57},
    {0x1.71f75e8ec5f74p+0, -0x1.16e4786887a99p-55}, {0x1.75feb564267c9p+0, -0x1.0245957316dd3p-54},
    {0x1.7a11473eb0187p+0, -0x1.41577ee04992fp-55}, {0x1.7e2f336cf4e62p+0, 0x1.05d02ba15797ep-56},
    {0x1.82589994cce13p+0, -0x1.d4c1dd41532d8p-54}, {0x1.868d99b4492edp+0, -0x1.fc6f89bd4f6bap-54},
    {0x1.8ace5422aa0dbp+0, 0x1.6e9f156864b27p-54}, {0x1.8f1ae99157736p+0, 0x1.5cc13a2e3976cp-55},
    {0x1.93737b0cdc5e5p+0, -0x1.75fc781b57ebcp-57}, {0x1.97d829fde4e50p+0, -0x1.d185b7c1b85d1p-54},
    {0x1.9c49182a3f090p+0, 0x1.c7c46b071f2bep-56}, {0x1.a0c667b5de565p+0, -0x1.359495d1cd533p-54},
    {0x1.a5503b23e255dp+0, -0x1.d2f6edb8d41e1p-54}, {0x1.a9e6b5579fdbfp+0, 0x1.0fac90ef7fd31p-54},
    {0x1.ae89f995ad3adp+0, 0x1.7a1cd345dcc81p-54}, {0x1.b33a2b84f15fbp+0, -0x1.2805e3084d708p-57},
    {0x1.b7f76f2fb5e47p+0, -0x1.5584f7e54ac3bp-56}, {0x1.bcc1e904bc1d2p+0, 0x1.23dd07a2d9e84p-55},
    {0x1.c199bdd85529cp+0, 0x1.11065895048ddp-55}, {0x1.c67f12e57d14bp+0, 0x1.2884dff483cadp-54},
    {0x1.cb720dcef9069p+0, 0x1.503cbd1e949dbp-56}, {0x1.d072d4a07897cp+0, -0x1.cbc3743797a9cp-54},
    {0x1.d5818dcfba487p+0, 0x1.2ed02d75b3707p-55}, {0x1.da9e603db3285p+0, 0x1.c2300696db532p-54},
    {0x1.dfc97337b9b5fp+0, -0x1.1a5cd4f184b5cp-54}, {0x1.e502ee78b3ff6p+0, 0x1.39e8980a9cc8fp-55},
    {0x1.ea4afa2a490dap+0, -0x1.e9c23179c2893p-54}, {0x1.efa1bee615a27p+0, 0x1.dc7f486a4b6b0p-54},
    {0x1.f50765b6e4540p+0, 0x1.9d3e12dd8a18bp-54}, {0x1.fa7c1819e90d8p+0, 0x1.74853f3a5931ep-55},
};

// e^x = 2^(k / 64) e^r, |r| <= ln 2 / 128, by table and polynomial (P. T. P. Tang, ACM TOMS 15, 1989):
// twelve FP64 instructions (CUDA's exp: 18), within 0.52 ulp: half an ulp for the last addition, the other
// roundings a hundred times smaller, the series' remainder r^7 / 5040 below 2^-64.  (Without the table's
// trailing words and the series' last term it took ten, and was up to 1.26 ulp off.)  Outside
// |x| < 704, NaN included, CUDA's function.
__device__ __forceinline__ double exp_t(double x, const double2 *tab)
{
    if ((__double2hiint(x) & 0x7fffffff) >= 0x40860000) return exp(x);
    const double magic = 6755399441055744.0;                  // 1.5 * 2^52: the sum's low word is rint(64 x / ln 2)
    const double t = fma(x, 0x1.71547652b82fep+6, magic);
    const int k = __double2loint(t);
    const double kd = t - magic;
    double r = fma(kd, -0x1.62e42fefa39efp-7, x);
    r = fma(kd, -0x1.abc9e3b39803fp-62, r);
    const double r2 = r * r;
    double p = fma(r, 1.0 / 720.0, 1.0 / 120.0);
    p = fma(p, r, 1.0 / 24.0);
    p = fma(p, r, 1.0 / 6.0);
    p = fma(p, r, 0.5);
    p = fma(p, r2, r);
    const double2 v = tab[k & 63];
    const double s = v.x + fma(v.x, p, v.y);
    return __hiloint2double(__double2hiint(s) + ((k >> 6) << 20), __double2loint(s));
}

// 1/x from the hardware's approximation r (about 2^-20) by one cubically converging step,
// r (1 + e + e^2) with e = 1 - x r: within 0.51 ulp (e^3 is up to 2^-60), a division's result but for three
// numbers in ten thousand.  An FP64 division outside the exponents where r and e are exact enough (zero, denormal,
// near overflow, non-finite).
__device__ __forceinline__ double recip(double x)
{
    const int ex = (__double2hiint(x) >> 20) & 0x7ff;
    if ((unsigned)(ex - 64) > 1900u) return 1.0 / x;
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
    double e = fma(-x, r, 1.0);
    e = fma(e, e, e);
    return fma(r, e, r);
}

// (cos, sin)(E c dt) for a whole number c.  The phase is 2^-53 of itself off its exact value (2e-13 at 2000
// radians); where many samples share the factor, that error does not average out as it does with a
// phase for each, so it is put back to first order: E (c dt) = x + d, d from the products' exact remainders.
__device__ __forceinline__ double2 unit_phase(double E, double c, double dt)
{
    const double t = c * dt, x = E * t;
    const double d = fma(E, fma(c, dt, -t), fma(E, t, -x));
    double s, co;
    sincos(x, &s, &co);
    return make_double2(fma(-s, d, co), fma(co, d, s));
}

// Order of magnitudes as integers (comparisons run on the FP64 pipe otherwise).
__device__ __forceinline__ int mag_key(double x) { return __double2hiint(x) & 0x7fffffff; }
__device__ __forceinline__ bool finite_bits(double x) { return mag_key(x) < 0x7ff00000; }

// An FP32 value as FP64 by its bits; denormals become zero.
__device__ __forceinline__ double widen_normal(float x)
{
    const int b = __float_as_int(x), e = b & 0x7f800000, s = b & 0x80000000;
    const int hi = ((b & 0x7fffffff) >> 3) + (e == 0x7f800000 ? 0x70000000 : 0x38000000);
    return __hiloint2double(e ? hi | s : s, e ? b << 29 : 0);
}

// The same with denormals, by conversion (a branch: loads behind it do not move ahead of it).
__device__ __forceinline__ double widen(float x)
{
    if ((unsigned)((__float_as_int(x) & 0x7fffffff) - 1) < 0x7fffffu) return (double)x;
    return widen_normal(x);
}

__device__ const double2 kAngleTable[33] = {   // (cos, sin)(k pi / 64)
    {0x1.0000000000000p+0, 0x0.0p+0}, {0x1.ff621e3796d7ep-1, 0x1.91f65f10dd814p-5},
    {0x1.fd88da3d12526p-1, 0x1.917a6bc29b42cp-4}, {0x1.fa7557f08a517p-1, 0x1.2c8106e8e613ap-3},
    {0x1.f6297cff75cb0p-1, 0x1.8f8b83c69a60bp-3}, {0x1.f0a7efb9230d7p-1, 0x1.f19f97b215f1bp-3},
    {0x1.e9f4156c62ddap-1, 0x1.294062ed59f06p-2}, {0x1.e212104f686e5p-1, 0x1.58f9a75ab1fddp-2},
    {0x1.d906bcf328d46p-1, 0x1.87de2a6aea963p-2}, {0x1.ced7af43cc773p-1, 0x1.b5d1009e15cc0p-2},
    {0x1.c38b2f180bdb1p-1, 0x1.e2b5d3806f63bp-2}, {0x1.b728345196e3ep-1, 0x1.073879922ffeep-1},
    {0x1.a9b66290ea1a3p-1, 0x1.1c73b39ae68c8p-1}, {0x1.9b3e047f38741p-1, 0x1.30ff7fce17035p-1},
    {0x1.8bc806b151741p-1, 0x1.44cf325091dd6p-1}, {0x1.7b5df226aafafp-1, 0x1.57d69348ceca0p-1},
    {0x1.6a09e667f3bcdp-1, 0x1.6a09e667f3bcdp-1}, {0x1.57d69348ceca0p-1, 0x1.7b5df226aafafp-1},
    {0x1.44cf325091dd6p-1, 0x1.8bc806b151741p-1}, {0x1.30ff7fce17035p-1, 0x1.9b3e047f38741p-1},
    {0x1.1c73b39ae68c8p-1, 0x1.a9b66290ea1a3p-1}, {0x1.073879922ffeep-1, 0x1.b728345196e3ep-1},
    {0x1.e2b5d3806f63bp-2, 0x1.c38b2f180bdb1p-1}, {0x1.b5d1009e15cc0p-2, 0x1.ced7af43cc773p-1},
    {0x1.87de2a6aea963p-2, 0x1.d906bcf328d46p-1}, {0x1.58f9a75ab1fddp-2, 0x1.e212104f686e5p-1},
    {0x1.294062ed59f06p-2, 0x1.e9f4156c62ddap-1}, {0x1.f19f97b215f1bp-3, 0x1.f0a7efb9230d7p-1},
    {0x1.8f8b83c69a60bp-3, 0x1.f6297cff75cb0p-1}, {0x1.2c8106e8e613ap-3, 0x1.fa7557f08a517p-1},
    {0x1.917a6bc29b42cp-4, 0x1.fd88da3d12526p-1}, {0x1.91f65f10dd814p-5, 0x1.ff621e3796d7ep-1},
    {0x0.0p+0, 0x1.0000000000000p+0},
};

// arg(x + i y) for a number whose larger part has a magnitude in [1, 2) (or is zero: 0; NaN: NaN), xf
// and yf its parts in FP32: the nearest multiple k pi / 64 is turned away, which leaves a tangent
// |t| <= tan(pi / 128), and atan t = t - t^3 / 3 + t^5 / 5 - t^7 / 7 + t^9 / 9 (the remainder is below
// 2^-56 t).  15 FP64 instructions against 42 of atan2; absolute error below 5e-16.
__device__ __forceinline__ double arg_normal(double x, double y, float xf, float yf)
{
    const double ax = fabs(x), ay = fabs(y);
    const int k = __float2int_rn(atan2f(fabsf(yf), fabsf(xf)) * 20.371833f);
    const double2 cs = kAngleTable[min(max(k, 0), 32)];
    const double u = fma(ax, cs.x, ay * cs.y), v = fma(ay, cs.x, -ax * cs.y);
    const double t = v * recip(u);
    const double t2 = t * t;
    double p = fma(t2, 1.0 / 9.0, -1.0 / 7.0);
    p = fma(p, t2, 0.2);
    p = fma(p, t2, -1.0 / 3.0);
    const double a = fma(t * t2, p, t);
    // k pi / 64 from the integer's bits: 2^52 + k less 2^52
    const double kd = __hiloint2double(0x43300000, k) - 4503599627370496.0;
    double r = fma(kd, 0x1.921fb54442d18p-5, a);
    if (xf < 0.0f) r = 3.14159265358979323846 - r;
    if (xf == 0.0f && yf == 0.0f) r = 0.0;
    return __hiloint2double(__double2hiint(r) ^ (__float_as_int(yf) & 0x80000000), __double2loint(r));
}

}  // namespace scivr
