// FP64 functions of the cell integrals' closed form.
//
// GB300 issues two FP64 operations per SM and clock, so the closed form's cost
// is its count of FP64 instructions, and most of them were in its square
// roots, divisions, logarithms and arc tangent.  These versions take a first
// approximation from the FP32 units or from the bits and finish in FP64: Newton
// steps for 1/x and sqrt(x), ln(a/b) as 2 artanh((a - b)/(a + b)) of the
// mantissas without a division before it, the arc tangent as its series after a
// rotation by a multiple of pi/16.  Each is accurate to a few units of 1e-16;
// arguments outside the FP32 range take the library's
// functions.
#pragma once
#include <math.h>
#include <stdint.h>

#ifdef __CUDA_ARCH__
#define CF_RSQRT(x) rsqrtf(x)
#define CF_HI(x) __double2hiint(x)
#define CF_MAKE(h, x) __hiloint2double(h, __double2loint(x))
#else
#include <string.h>
#define CF_RSQRT(x) (1.0f / sqrtf(x))
static inline int cf_hi_host(double x) { uint64_t u; memcpy(&u, &x, 8); return (int)(u >> 32); }
static inline double cf_make_host(int h, double x)
{
    uint64_t u;
    memcpy(&u, &x, 8);
    u = (u & 0xffffffffull) | ((uint64_t)(uint32_t)h << 32);
    memcpy(&x, &u, 8);
    return x;
}
#define CF_HI(x) cf_hi_host(x)
#define CF_MAKE(h, x) cf_make_host(h, x)
#endif

// biased exponent of |x| within 2^-100 .. 2^100 (finite, normal, its square
// and its FP32 image too)
__host__ __device__ __forceinline__ bool cf_in_range(double x)
{
    const int e = (CF_HI(x) >> 20) & 0x7ff;
    return e > 1023 - 100 && e < 1023 + 100;
}

// 1/x: an FP32 reciprocal and two Newton steps
__host__ __device__ __forceinline__ double cf_rcp(double x)
{
    double y = (double)(1.0f / (float)x);
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
}

__host__ __device__ __forceinline__ double cf_sqrt(double x)
{
    if (!cf_in_range(x) || CF_HI(x) < 0) return sqrt(x);
    const double y = (double)CF_RSQRT((float)x), h = 0.5 * y;
    double r = x * y;
    r = fma(fma(-r, r, x), h, r);
    return fma(fma(-r, r, x), h, r);
}

// ln(a / b), a, b >= 0: exponents apart, mantissas brought within a factor of
// sqrt 2, then 2 artanh(s) with |s| <= 0.172 (ten terms: 2e-17 relative)
__host__ __device__ __forceinline__ double cf_log_ratio(double a, double b)
{
    const int ha = CF_HI(a), hb = CF_HI(b);
    int ea = ha >> 20, eb = hb >> 20;                       // sign 0: the biased exponents
    if (ea <= 0 || ea >= 0x7ff || eb <= 0 || eb >= 0x7ff) return log(a) - log(b);
    const int fa = (ha & 0xfffff) | 0x100000, fb = (hb & 0xfffff) | 0x100000;
    // 99/70 = sqrt 2 to 5e-5
    const int da = 70 * (fa >> 4) > 99 * (fb >> 4), db = 70 * (fb >> 4) > 99 * (fa >> 4);
    const double ma = CF_MAKE((ha & 0xfffff) | ((1023 - da) << 20), a), mb = CF_MAKE((hb & 0xfffff) | ((1023 - db) << 20), b);
    const double s = (ma - mb) * cf_rcp(ma + mb), t = s * s;
    double p = 1.0 / 19.0;
    p = fma(p, t, 1.0 / 17.0);
    p = fma(p, t, 1.0 / 15.0);
    p = fma(p, t, 1.0 / 13.0);
    p = fma(p, t, 1.0 / 11.0);
    p = fma(p, t, 1.0 / 9.0);
    p = fma(p, t, 1.0 / 7.0);
    p = fma(p, t, 1.0 / 5.0);
    p = fma(p, t, 1.0 / 3.0);
    p = fma(p, t, 1.0);
    return fma((double)(ea + da - eb - db), 0.69314718055994530942, 2.0 * s * p);
}

// cos and sin of k pi / 16, k = 0 .. 16
#ifdef __CUDACC__
static __device__ const double cf_cs_dev[17][2] = {
    {1.0, 0.0}, {0.98078528040323044913, 0.19509032201612826785}, {0.92387953251128675613, 0.38268343236508977173},
    {0.83146961230254523708, 0.55557023301960222474}, {0.70710678118654752440, 0.70710678118654752440},
    {0.55557023301960222474, 0.83146961230254523708}, {0.38268343236508977173, 0.92387953251128675613},
    {0.19509032201612826785, 0.98078528040323044913}, {0.0, 1.0},
    {-0.19509032201612826785, 0.98078528040323044913}, {-0.38268343236508977173, 0.92387953251128675613},
    {-0.55557023301960222474, 0.83146961230254523708}, {-0.70710678118654752440, 0.70710678118654752440},
    {-0.83146961230254523708, 0.55557023301960222474}, {-0.92387953251128675613, 0.38268343236508977173},
    {-0.98078528040323044913, 0.19509032201612826785}, {-1.0, 0.0}};
#endif

__host__ __device__ __forceinline__ double cf_atan2(double y, double x)
{
    // the larger of the two decides the scale; the other may vanish in FP32
    const int ey = (CF_HI(y) >> 20) & 0x7ff, ex = (CF_HI(x) >> 20) & 0x7ff;
    const int em = ey > ex ? ey : ex;
    if (em <= 1023 - 100 || em >= 1023 + 100) return atan2(y, x);
    const float k = rintf(atan2f((float)y, (float)x) * 5.0929581789406507f);      // 16 / pi
    const int q = k < 0.f ? (int)-k : (int)k;
#ifdef __CUDA_ARCH__
    const double c = cf_cs_dev[q][0], s0 = cf_cs_dev[q][1];
#else
    const double c = cos(q * (M_PI / 16)), s0 = sin(q * (M_PI / 16));
#endif
    const double s = k < 0.f ? -s0 : s0;
    const double xr = fma(x, c, y * s), yr = fma(y, c, -(x * s));
    const double t = yr * cf_rcp(xr), u = t * t;                                    // |t| <= 0.0985
    double p = 1.0 / 15.0;
    p = fma(-p, u, 1.0 / 13.0);
    p = fma(-p, u, 1.0 / 11.0);
    p = fma(-p, u, 1.0 / 9.0);
    p = fma(-p, u, 1.0 / 7.0);
    p = fma(-p, u, 1.0 / 5.0);
    p = fma(-p, u, 1.0 / 3.0);
    p = fma(-p, u, 1.0);
    return fma((double)k, 0.19634954084936207740, t * p);
}
