// Double-float arithmetic for the exact dust-emission solve: a value is an
// unevaluated sum hi + lo of two IEEE binary32 numbers (|lo| <= ulp(hi)/2),
// about 48 significant bits, computed on the FP32 pipe.  GB300 retires an
// FP64 warp instruction far more slowly than an FP32 one, so the per-term
// work of the solve (the Planck factor 1/expm1(x) of every wavelength and
// population) runs in this arithmetic and only the per-population steps stay
// in FP64.
//
// Methods (all published, none taken from a math library):
//  * error-free transformations: Knuth's two-sum, Dekker's fast two-sum (for
//    |a| >= |b|), and the exact product a*b = p + e with e = fma(a, b, -p)
//    (Dekker 1971; Ogita, Rump and Oishi 2005);
//  * double-float sums and products built on them in the usual way
//    (Dekker 1971; Hida, Li and Bailey 2001);
//  * expm1(x), 0 <= x <= 88, from z = x EXP_N / ln 2 (the caller folds the
//    factor into its constants): z = k + f, |f| <= 1/2, k = 256 n + j;
//    e^x = 2^n (1 + s_j) (1 + p) with s_j = 2^(j/256) - 1 from a table of
//    double-float pairs (Tang's table-driven exponential, 1989/1992) and
//    p = expm1(r), r = f ln 2 / 256, |r| < 0.00136, from r + r^2/2 + r^3/6 + r^4/24
//    (the first omitted term is below 4e-17): the first two terms in
//    double-float, the rest in binary32.  About 60 operations, against some 150
//    of a Taylor series over |r| <= ln 2 / 2, and the same accuracy (rms
//    1.4e-15 relative over 7e-3 <= x <= 70, against 1.2e-15);
//  * 1/a: the binary32 reciprocal refined by one Newton step,
//    y' = y + y (1 - a y), with the residual formed exactly.
//
// The operations are spelled with round-to-nearest intrinsics on the device
// (nothing may be contracted into an FMA); on the host the same code is plain
// binary32 arithmetic and gives identical results when compiled without
// floating-point contraction (-ffp-contract=off).
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define DF_FN __host__ __device__ __forceinline__
#else
#define DF_FN static inline
#endif

#ifdef __CUDA_ARCH__
#define DF_ADD(a, b) __fadd_rn((a), (b))
#define DF_SUB(a, b) __fsub_rn((a), (b))
#define DF_MUL(a, b) __fmul_rn((a), (b))
#define DF_RCP(a) __frcp_rn(a)
#else
#define DF_ADD(a, b) ((a) + (b))
#define DF_SUB(a, b) ((a) - (b))
#define DF_MUL(a, b) ((a) * (b))
#define DF_RCP(a) (1.0f / (a))
#endif

namespace dfl {

struct df2 {
    float hi, lo;
};

DF_FN df2 make(float hi, float lo)
{
    df2 r;
    r.hi = hi;
    r.lo = lo;
    return r;
}

// s + e = a + b exactly
DF_FN void two_sum(float a, float b, float& s, float& e)
{
    s = DF_ADD(a, b);
    const float bb = DF_SUB(s, a);
    e = DF_ADD(DF_SUB(a, DF_SUB(s, bb)), DF_SUB(b, bb));
}

// s + e = a + b exactly, for |a| >= |b| (or a == 0)
DF_FN void fast_two_sum(float a, float b, float& s, float& e)
{
    s = DF_ADD(a, b);
    e = DF_SUB(b, DF_SUB(s, a));
}

// p + e = a * b exactly (barring underflow)
DF_FN void two_prod(float a, float b, float& p, float& e)
{
    p = DF_MUL(a, b);
    e = fmaf(a, b, -p);
}

DF_FN df2 renorm(float hi, float lo)
{
    df2 r;
    fast_two_sum(hi, lo, r.hi, r.lo);
    return r;
}

// a + b, for operands of the same sign (no cancellation between the high parts)
DF_FN df2 add(df2 a, df2 b)
{
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    e = DF_ADD(e, DF_ADD(a.lo, b.lo));
    return renorm(s, e);
}

DF_FN df2 mul(df2 a, df2 b)
{
    float p, e;
    two_prod(a.hi, b.hi, p, e);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return renorm(p, e);
}

// 1/a for a > 0 (binary32 normal range)
DF_FN df2 recip(df2 a)
{
    const float y = DF_RCP(a.hi);
    float p, e;
    two_prod(a.hi, y, p, e);            // a.hi y = p + e, p within an ulp of 1
    float r = DF_SUB(1.0f, p);          // exact
    r = DF_SUB(r, e);
    r = fmaf(-a.lo, y, r);              // r = 1 - a y to ~2^-48
    return renorm(y, DF_MUL(y, r));
}

// intervals of one binade in the exponential's table
#define DF_EXP_N 256
// DF_EXP_N / ln 2 (the factor from x to z), and ln 2 / DF_EXP_N in two binary32 pieces
#define DF_Z_PER_X 369.32993046757463
#define DF_X_PER_Z_0 0x1.62e430p-9f
#define DF_X_PER_Z_1 -0x1.05c610p-37f

// entry j of the table: 2^(j / DF_EXP_N) - 1
static inline df2 exp_table_entry(int j)
{
    const double v = ::expm1(j * (0.693147180559945309417232 / DF_EXP_N));
    const float h = (float)v;
    return make(h, (float)(v - (double)h));
}

// e^x - 1 for x = (k + f + fe) / DF_Z_PER_X, 0 <= x <= 88, |f| <= 1/2, as hi + lo
// with lo a few ulp of hi at most; tab(j) fetches the table's entry j
template <typename Tab>
DF_FN df2 expm1_reduced(int k, float f, float fe, const Tab& tab)
{
    // r = (f + fe) ln 2 / 256
    float p, e, rh, rl;
    two_prod(f, DF_X_PER_Z_0, p, e);
    fast_two_sum(p, fmaf(fe, DF_X_PER_Z_0, fmaf(f, DF_X_PER_Z_1, e)), rh, rl);
    // expm1(r) = ph + pl
    float q, qe, ph, pl;
    two_prod(rh, rh, q, qe);
    const float tail = DF_MUL(DF_MUL(rh, q), fmaf(rh, 1.0f / 24.0f, 1.0f / 6.0f));
    const float lo = DF_ADD(fmaf(0.5f, qe, fmaf(rh, rl, rl)), tail);
    fast_two_sum(rh, DF_MUL(0.5f, q), ph, pl);
    pl = DF_ADD(pl, lo);
    // m = s + p + s p = 2^(z/256 - n) - 1
    const df2 s = tab(k & (DF_EXP_N - 1));
    float u, ue, w, we, sp, spe;
    two_prod(s.hi, ph, sp, spe);
    spe = fmaf(s.lo, ph, fmaf(s.hi, pl, spe));
    fast_two_sum(s.hi, ph, u, ue);
    fast_two_sum(u, sp, w, we);
    const float ml = DF_ADD(DF_ADD(DF_ADD(s.lo, pl), DF_ADD(ue, we)), spe);
    // 2^n (1 + m) - 1 (m itself for n = 0)
    const int n = k >> 8;
    union {
        int i;
        float v;
    } c;
    c.i = (127 + n) << 23;
    float a, ae, b, be;
    fast_two_sum(c.v, DF_MUL(c.v, w), a, ae);
    fast_two_sum(a, -1.0f, b, be);
    const float l = fmaf(c.v, ml, DF_ADD(ae, be));
    return n == 0 ? make(w, ml) : make(b, l);
}

// e^x - 1 for x = z / DF_Z_PER_X
template <typename Tab>
DF_FN df2 expm1_z(df2 z, const Tab& tab)
{
    // k = z rounded to an integer through the 1.5 2^23 offset
    union {
        float v;
        int i;
    } c;
    c.v = DF_ADD(z.hi, 12582912.0f);
    float f, fe;
    two_sum(DF_SUB(z.hi, DF_SUB(c.v, 12582912.0f)), z.lo, f, fe);
    return expm1_reduced(c.i & 0x3FFFFF, f, fe, tab);
}

#ifndef __CUDACC__
// the host's form, of x itself, with the table computed at first use
struct host_exp_table {
    df2 t[DF_EXP_N];
    host_exp_table()
    {
        for (int j = 0; j < DF_EXP_N; ++j) t[j] = exp_table_entry(j);
    }
    df2 operator()(int j) const { return t[j]; }
};

static inline df2 expm1(df2 x)
{
    static const host_exp_table tab;
    const double z = ((double)x.hi + (double)x.lo) * DF_Z_PER_X, k = rint(z), r = z - k;
    const float h = (float)r;
    const df2 v = expm1_reduced((int)k, h, (float)(r - (double)h), tab);
    return renorm(v.hi, v.lo);
}
#endif

}  // namespace dfl
