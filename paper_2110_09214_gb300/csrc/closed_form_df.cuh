// The closed form of a cell's integrals in pairs of floats (x = h + l, 48 bits).
//
// GB300 issues 64 FP32 instructions for one of FP64, and what leaves the closed
// form is a sum of binary32 terms: a pair of floats carries each of its numbers
// to about 2^-46, so that after the cancellations of the near field the rounded
// terms are those of the FP64 form but for one in thousands (measured against
// it on the CPU, tests/test_closed_form_df_host.py).  About 1800 FP32
// instructions where tri_closed_form_g takes 260 of FP64 at 16 clocks each: near
// cells of a field map 5.9 to 3.0 ms, of 64 chambers 2.1 to 1.05 ms, the assembly of
// 59,968 cells 21.5 to 16.5 ms.
// Where 48 bits do not decide the result (a point on an edge or a vertex, or, of a
// cell that is not axis-parallel, in its plane to 1e-12 of the distance)
// tri_closed_df returns false and the caller takes the FP64 form.
//
// Arithmetic: T. J. Dekker, "A floating-point technique for extending the
// available precision", 1971 (sums and products with their errors); functions
// from an FP32 value and one correction, ln(a/b) as 2 artanh((a - b)/(a + b)), the
// arc tangent as its series after a rotation by a multiple of pi/16.
#pragma once
#include <math.h>
#include <stdint.h>

#ifdef __CUDA_ARCH__
#define DF_ADD(a, b) __fadd_rn(a, b)
#define DF_SUB(a, b) __fsub_rn(a, b)
#define DF_MUL(a, b) __fmul_rn(a, b)
#define DF_FMA(a, b, c) __fmaf_rn(a, b, c)
#define DF_BITS(x) __float_as_int(x)
#define DF_FROM(i) __int_as_float(i)
#define DF_RSQRT(x) rsqrtf(x)
#define DF_RCP(x) __frcp_rn(x)
#else
#include <string.h>
#define DF_ADD(a, b) ((a) + (b))
#define DF_SUB(a, b) ((a) - (b))
#define DF_MUL(a, b) ((a) * (b))
#define DF_FMA(a, b, c) fmaf(a, b, c)
static inline int df_bits_host(float x) { int i; memcpy(&i, &x, 4); return i; }
static inline float df_from_host(int i) { float x; memcpy(&x, &i, 4); return x; }
#define DF_BITS(x) df_bits_host(x)
#define DF_FROM(i) df_from_host(i)
#define DF_RSQRT(x) (1.0f / sqrtf(x))
#define DF_RCP(x) (1.0f / (x))
#endif
#define DF_FN static __host__ __device__ __forceinline__

struct Dbf { float h, l; };

DF_FN Dbf df_norm(float a, float b)                     // |a| >= |b| (or a = 0)
{
    const float s = DF_ADD(a, b);
    return Dbf{s, DF_SUB(b, DF_SUB(s, a))};
}
DF_FN Dbf df_sum(Dbf a, Dbf b)
{
    const float s = DF_ADD(a.h, b.h), v = DF_SUB(s, a.h);
    const float e = DF_ADD(DF_SUB(a.h, DF_SUB(s, v)), DF_SUB(b.h, v));
    return df_norm(s, DF_ADD(e, DF_ADD(a.l, b.l)));
}
DF_FN Dbf df_neg(Dbf a) { return Dbf{-a.h, -a.l}; }
DF_FN Dbf df_dif(Dbf a, Dbf b) { return df_sum(a, df_neg(b)); }
DF_FN Dbf df_mul(Dbf a, Dbf b)
{
    const float p = DF_MUL(a.h, b.h);
    return df_norm(p, DF_FMA(a.l, b.h, DF_FMA(a.h, b.l, DF_FMA(a.h, b.h, -p))));
}
DF_FN Dbf df_mulf(Dbf a, float b)
{
    const float p = DF_MUL(a.h, b);
    return df_norm(p, DF_FMA(a.l, b, DF_FMA(a.h, b, -p)));
}
DF_FN Dbf df_div(Dbf a, Dbf b)
{
    const float y = DF_RCP(b.h), q = DF_MUL(a.h, y);
    const float p = DF_MUL(q, b.h), e = DF_FMA(q, b.h, -p);
    const float r = DF_FMA(-q, b.l, DF_ADD(DF_SUB(DF_SUB(a.h, p), e), a.l));
    return df_norm(q, DF_MUL(r, y));
}
DF_FN Dbf df_sqrt(Dbf x)
{
    const float y = DF_RSQRT(x.h), r = DF_MUL(x.h, y);
    const float p = DF_MUL(r, r), e = DF_FMA(r, r, -p);
    const float d = DF_ADD(DF_SUB(DF_SUB(x.h, p), e), x.l);
    return df_norm(r, DF_MUL(d, DF_MUL(0.5f, y)));
}
DF_FN Dbf df_dot(const Dbf *a, const Dbf *b) { return df_sum(df_sum(df_mul(a[0], b[0]), df_mul(a[1], b[1])), df_mul(a[2], b[2])); }
DF_FN Dbf df_scale(Dbf a, float p2) { return Dbf{DF_MUL(a.h, p2), DF_MUL(a.l, p2)}; }      // p2 a power of two
DF_FN Dbf df_sel(bool c, Dbf a, Dbf b) { return Dbf{c ? a.h : b.h, c ? a.l : b.l}; }

// ln(a / b), a, b > 0 within 2^-100 .. 2^100 of one another's exponents
DF_FN Dbf df_log_ratio(Dbf a, Dbf b)
{
    int k = (DF_BITS(a.h) >> 23) - (DF_BITS(b.h) >> 23);
    float bh = DF_MUL(b.h, DF_FROM((127 + k) << 23));
    if (a.h > 1.41421356f * bh) ++k;
    else if (bh > 1.41421356f * a.h) --k;
    b = df_scale(b, DF_FROM((127 + k) << 23));
    const Dbf z = df_div(df_dif(a, b), df_sum(a, b));                 // |z| <= 0.172
    const Dbf t = df_mul(z, z);
    const float u = t.h;
    float q = 1.0f / 19.0f;
    q = DF_FMA(q, u, 1.0f / 17.0f);
    q = DF_FMA(q, u, 1.0f / 15.0f);
    q = DF_FMA(q, u, 1.0f / 13.0f);
    q = DF_FMA(q, u, 1.0f / 11.0f);
    q = DF_FMA(q, u, 1.0f / 9.0f);
    q = DF_FMA(q, u, 1.0f / 7.0f);
    const Dbf fifth = {0.2f, (float)(0.2 - (double)0.2f)}, third = {1.0f / 3.0f, (float)(1.0 / 3.0 - (double)(1.0f / 3.0f))};
    const Dbf A = df_sum(fifth, df_mulf(t, q));
    const Dbf B = df_sum(third, df_mul(t, A));
    const Dbf s = df_sum(z, df_mul(z, df_mul(t, B)));
    const Dbf ln2 = {0.69314718055994530942f, (float)(0.69314718055994530942 - (double)0.69314718055994530942f)};
    return df_sum(df_mulf(ln2, (float)k), df_scale(s, 2.0f));
}

// cos and sin of k pi / 16, k = 0 .. 16, as pairs
#ifdef __CUDACC__
#define DF_CS(c, s) {(float)(c), (float)((c) - (double)(float)(c)), (float)(s), (float)((s) - (double)(float)(s))}
static __device__ const float df_cs_dev[17][4] = {
    DF_CS(1.0, 0.0), DF_CS(0.98078528040323044913, 0.19509032201612826785),
    DF_CS(0.92387953251128675613, 0.38268343236508977173), DF_CS(0.83146961230254523708, 0.55557023301960222474),
    DF_CS(0.70710678118654752440, 0.70710678118654752440), DF_CS(0.55557023301960222474, 0.83146961230254523708),
    DF_CS(0.38268343236508977173, 0.92387953251128675613), DF_CS(0.19509032201612826785, 0.98078528040323044913),
    DF_CS(0.0, 1.0), DF_CS(-0.19509032201612826785, 0.98078528040323044913),
    DF_CS(-0.38268343236508977173, 0.92387953251128675613), DF_CS(-0.55557023301960222474, 0.83146961230254523708),
    DF_CS(-0.70710678118654752440, 0.70710678118654752440), DF_CS(-0.83146961230254523708, 0.55557023301960222474),
    DF_CS(-0.92387953251128675613, 0.38268343236508977173), DF_CS(-0.98078528040323044913, 0.19509032201612826785),
    DF_CS(-1.0, 0.0)};
#endif

DF_FN Dbf df_atan2(Dbf y, Dbf x)
{
    const float k = rintf(atan2f(y.h, x.h) * 5.0929581789406507f);        // 16 / pi
    const int q = k < 0.f ? (int)-k : (int)k;
#ifdef __CUDA_ARCH__
    const Dbf c = {df_cs_dev[q][0], df_cs_dev[q][1]};
    Dbf s = {df_cs_dev[q][2], df_cs_dev[q][3]};
#else
    const double cd = q == 8 ? 0.0 : cos(q * (M_PI / 16)), sd = q == 16 ? 0.0 : sin(q * (M_PI / 16));
    const Dbf c = {(float)cd, (float)(cd - (double)(float)cd)};
    Dbf s = {(float)sd, (float)(sd - (double)(float)sd)};
#endif
    if (k < 0.f) s = df_neg(s);
    const Dbf xr = df_sum(df_mul(x, c), df_mul(y, s)), yr = df_dif(df_mul(y, c), df_mul(x, s));
    const Dbf t = df_div(yr, xr), u = df_mul(t, t);                        // |t| <= 0.0985
    float p = -1.0f / 13.0f;
    p = DF_FMA(p, u.h, 1.0f / 11.0f);
    p = DF_FMA(p, u.h, -1.0f / 9.0f);
    p = DF_FMA(p, u.h, 1.0f / 7.0f);
    const Dbf fifth = {0.2f, (float)(0.2 - (double)0.2f)}, third = {-1.0f / 3.0f, (float)(-1.0 / 3.0 - (double)(-1.0f / 3.0f))};
    const Dbf A = df_sum(fifth, df_mulf(u, -p));
    const Dbf B = df_sum(third, df_mul(u, A));
    const Dbf pi16 = {0.19634954084936207740f, (float)(0.19634954084936207740 - (double)0.19634954084936207740f)};
    return df_sum(df_mulf(pi16, k), df_sum(t, df_mul(t, df_mul(u, B))));
}

// Numbers of a cell for tri_closed_df, as pairs: its 9 vertex coordinates and the
// 22 of tri_closed_form_g's geometry (normal, twice the area, edges)
#define DF_TINY 1e-12f          // of the distance: where the FP64 form decides

// phi and F (tri_closed_form_g) at r; false: not decided in 48 bits.  want_f:
// false leaves F's part along the normal undecided in the cell's plane (phi is
// not affected there).
static __host__ __device__ __noinline__ bool tri_closed_df(const float2 *g2, Dbf rx, Dbf ry, Dbf rz, bool want_f, Dbf &phi,
                                                           Dbf &Fx, Dbf &Fy, Dbf &Fz)
{
    auto num = [&](int i) { return Dbf{g2[i].x, g2[i].y}; };
    const Dbf n[3] = {num(9), num(10), num(11)}, a2 = num(12);
    Dbf a[3][3], R[3];
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        a[i][0] = df_dif(num(3 * i), rx);
        a[i][1] = df_dif(num(3 * i + 1), ry);
        a[i][2] = df_dif(num(3 * i + 2), rz);
        const Dbf s = df_dot(a[i], a[i]);
        ok = ok && s.h > 1e-22f && s.h < 1e12f;      // (products of three below 1e-33 lose their low parts)
        R[i] = df_sqrt(s);
    }
    const Dbf h = df_neg(df_dot(a[0], n)), h2 = df_mul(h, h);
    // in the plane of an axis-parallel cell h is exactly 0 in either arithmetic
    const bool flat = a[0][0].h * n[0].h == 0.f && a[0][1].h * n[1].h == 0.f && a[0][2].h * n[2].h == 0.f;
    Dbf ps = {0.f, 0.f}, f[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    Dbf D = df_mul(df_mul(R[0], R[1]), R[2]);
    // the edges one after the other in one copy of the code, vertices rotated
    // (unrolled, the warps of a block waited for instructions)
#pragma unroll 1
    for (int i = 0; i < 3; ++i) {
        const Dbf d[3] = {num(13 + 6 * i), num(14 + 6 * i), num(15 + 6 * i)},
                  u[3] = {num(16 + 6 * i), num(17 + 6 * i), num(18 + 6 * i)};
        const Dbf lm = df_dot(a[0], d), lp = df_dot(a[1], d), p0 = df_dot(a[0], u);
        const bool fwd = lm.h >= 0.f, bwd = lp.h <= 0.f;
        const Dbf m = df_sum(df_mul(p0, p0), h2);
        const Dbf ej = df_sum(R[1], df_sel(bwd && !fwd, df_neg(lp), lp)), ei = df_sum(R[0], df_sel(fwd, lm, df_neg(lm)));
        // fwd: ej / ei; bwd: ei / ej; between the ends: ej ei / m
        const bool mid = !fwd && !bwd;
        const Dbf top = df_sel(fwd, ej, df_sel(bwd, ei, df_mul(ej, ei))), bot = df_sel(fwd, ei, df_sel(bwd, ej, m));
        ok = ok && (!mid || m.h > DF_TINY * R[0].h * R[0].h);
        const Dbf L = df_log_ratio(top, bot);
        ps = df_sum(ps, df_mul(p0, L));
#pragma unroll
        for (int c = 0; c < 3; ++c) f[c] = df_sum(f[c], df_mul(u[c], L));
        D = df_sum(D, df_mul(df_dot(a[0], a[1]), R[2]));
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const Dbf t = a[0][c];
            a[0][c] = a[1][c];
            a[1][c] = a[2][c];
            a[2][c] = t;
        }
        const Dbf t = R[0];
        R[0] = R[1];
        R[1] = R[2];
        R[2] = t;
    }
    ok = ok && !(want_f && !flat && D.h <= 0.f && fabsf(h.h) < DF_TINY * R[0].h);
    const Dbf Om = flat ? Dbf{0.f, 0.f} : df_scale(df_atan2(df_mul(a2, h), D), 2.0f);
    phi = df_dif(ps, df_mul(h, Om));
    Fx = df_sum(f[0], df_mul(Om, n[0]));
    Fy = df_sum(f[1], df_mul(Om, n[1]));
    Fz = df_sum(f[2], df_mul(Om, n[2]));
    return ok;
}
