// FP64 reconstruction on the integer pipe: the MC half slopes, the PPM interface values
// and limits, and the edge states they give, in block fixed point.
//
// GB300 issues an FP64 add every 16 cycles per SM and warp, an integer instruction every
// half cycle: reconstruction is additions and comparisons only, so its 64-bit integer
// form (2 instructions per addition) costs a fraction of the FP64 one, and it runs beside
// the FP64 arithmetic of the fluxes, which bounds the stencil kernels.
//
// The cell values x_i of a window share one exponent E: x_i is held as the 64-bit integer
// X_i = x_i 2^(1075 + kFxShift - E), |X_i| < 2^(53 + kFxShift).  Where every nonzero x_i
// lies within 2^kFxSpread of the largest, the X_i are exact multiples of 4, so the
// differences, the quarter of the central difference, their minmod and the sums x_i +- h
// are exact; each state is then rounded once, to nearest even.  That is at most the error
// of the FP64 sequence, which rounds the differences too.
//
// MC takes any finite window (mc_cell): a neighbour that is far above the other two values
// (2^5 and more) only bounds the slope from above, so it is replaced by one of the same
// sign 2^5 above them, and what lies below the last place, 2^-56 of the larger of the two
// others, is dropped; the FP64 sequence rounds their difference at 2^-54.  A slope of zero
// returns the cell value itself.  PPM takes the FP64 sequence in a window wider than
// kFxSpread.  A window with an infinity, a NaN or whose largest value, the far neighbour
// replaced, is nonzero and below 2^-943 takes the FP64 sequence too.  Denormals count as
// zero: a cell that is zero like one of its neighbours is flat.
#pragma once

#include <stdint.h>

namespace grmhd {

constexpr int kFxShift = 9;               // |X| < 2^62: a difference of two fits 63 bits
constexpr unsigned kFxSpread = 7u << 20;  // kFxShift - 2, in place in the high word
constexpr unsigned kFxMinE = 80u << 20;   // every shift below stays above the denormals

#ifdef __CUDA_ARCH__
__device__ __forceinline__ unsigned fx_hi(double x) { return (unsigned)__double2hiint(x); }
__device__ __forceinline__ unsigned fx_lo(double x) { return (unsigned)__double2loint(x); }
__device__ __forceinline__ double fx_double(unsigned long long b) { return __longlong_as_double((long long)b); }
__device__ __forceinline__ unsigned fx_shl(unsigned hi, unsigned lo, unsigned s) { return __funnelshift_l(lo, hi, s); }
// a shift count past 63 gives 0 (the PTX shift clamps)
__device__ __forceinline__ unsigned long long fx_shr(unsigned long long v, unsigned s)
{
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return r;
}
__device__ __forceinline__ int fx_clz(unsigned long long v) { return __clzll((long long)v); }
__device__ __forceinline__ long long fx_mulhi(long long a, long long b) { return __mul64hi(a, b); }
#else
#include <string.h>
inline unsigned long long fx_bits(double x)
{
    unsigned long long b;
    memcpy(&b, &x, 8);
    return b;
}
inline unsigned fx_hi(double x) { return (unsigned)(fx_bits(x) >> 32); }
inline unsigned fx_lo(double x) { return (unsigned)fx_bits(x); }
inline double fx_double(unsigned long long b)
{
    double x;
    memcpy(&x, &b, 8);
    return x;
}
inline unsigned fx_shl(unsigned hi, unsigned lo, unsigned s)
{
    s &= 31u;
    return s ? (hi << s) | (lo >> (32 - s)) : hi;
}
inline unsigned long long fx_shr(unsigned long long v, unsigned s) { return s > 63u ? 0ull : v >> s; }
inline int fx_clz(unsigned long long v) { return v ? __builtin_clzll(v) : 64; }
inline long long fx_mulhi(long long a, long long b) { return (long long)(((__int128)a * b) >> 64); }
#endif

#ifndef __CUDACC__
#define GRMHD_HD inline
#else
#define GRMHD_HD __host__ __device__ __forceinline__
#endif

// exponent field of x, in place in the high word
GRMHD_HD unsigned fx_exp(double x) { return fx_hi(x) & 0x7ff00000u; }

GRMHD_HD unsigned fx_max(unsigned a, unsigned b) { return a > b ? a : b; }

// x is zero or within the spread below the block exponent E
GRMHD_HD bool fx_near(double x, unsigned E)
{
    return E - fx_exp(x) <= kFxSpread || ((fx_hi(x) & 0x7fffffffu) | fx_lo(x)) == 0u;
}

// block exponent of three values: the largest of theirs, at least kFxMinE (a window of
// zeros has that one; smaller values are then not near it)
GRMHD_HD unsigned fx_block(double a, double b, double c)
{
    return fx_max(fx_max(fx_exp(a), fx_exp(b)), fx_max(fx_exp(c), kFxMinE));
}

GRMHD_HD bool fx_finite(unsigned E) { return E < 0x7ff00000u; }

// x as a fixed-point number of a block whose values are near E (fx_near)
GRMHD_HD long long fx_of(double x, unsigned E)
{
    const unsigned hi = fx_hi(x), lo = fx_lo(x), e = hi & 0x7ff00000u;
    const unsigned m = (hi & 0xfffffu) | (e < 0x100000u ? e : 0x100000u);   // 0 for a zero
    const unsigned s = kFxShift - ((E - e) >> 20);
    const long long v = (long long)(((unsigned long long)fx_shl(m, lo, s) << 32) | fx_shl(lo, 0u, s));
    const long long n = (long long)(int)hi >> 31;
    return (v ^ n) - n;
}

// the number with the sign and significand of x and the exponent field e <= E (normally
// that of x), in a block of exponent E >= kFxMinE: bits below the block's last place are
// dropped (toward zero); a zero or denormal (e = 0) gives 0
GRMHD_HD long long fx_cut(double x, unsigned e, unsigned E)
{
    const unsigned hi = fx_hi(x);
    const unsigned m = (hi & 0xfffffu) | 0x100000u;
    const unsigned long long w = (((unsigned long long)m << 32) | fx_lo(x)) << kFxShift;
    const long long v = (long long)fx_shr(w, (E - e) >> 20);
    const long long n = (long long)(int)hi >> 31;
    return (v ^ n) - n;
}

// back to FP64, rounded to nearest even (|v| < 2^63)
GRMHD_HD double fx_to(long long v, unsigned E)
{
    const long long n = v >> 63;
    const unsigned long long u = (unsigned long long)((v ^ n) - n);
    const int lz = fx_clz(u | 1ull);
    const unsigned long long y = u << lz;
    const unsigned long long q = y >> 11;                              // 53 bits, the leading one at 52
    const unsigned inc = (((unsigned)y & 0x7ffu) + ((unsigned)q & 1u)) > 0x400u ? 1u : 0u;
    // value 2^(lz position): the biased exponent is that of E plus 2 - lz; the leading one
    // adds one more to the field
    const unsigned long long e = (unsigned long long)(E + ((unsigned)(10 - kFxShift - lz) << 20)) << 32;
    const unsigned long long b = (q + inc + e) | ((unsigned long long)n & 0x8000000000000000ull);
    return fx_double(u ? b : 0ull);
}

// minmod(dm, c, dp) for c = (dm + dp) / 4: c lies between zero and the smaller of two
// agreeing differences, or is cut to it
GRMHD_HD long long fx_minmod(long long dm, long long c, long long dp)
{
    const long long mn = dm < dp ? dm : dp, mx = dm < dp ? dp : dm;
    const long long top = mn & ~(mn >> 63), bot = mx & (mx >> 63);   // max(mn, 0), min(mx, 0)
    const long long r = c < bot ? bot : c;
    return r > top ? top : r;
}

// the MC half slope of b from its neighbours, fixed point
GRMHD_HD long long fx_half_slope(long long a, long long b, long long x)
{
    return fx_minmod(b - a, (x - a) >> 2, x - b);
}

// PPM interface value between p and q with the full slopes sp, sq
GRMHD_HD long long fx_iface(long long p, long long q, long long sp, long long sq)
{
    return p + ((q - p) >> 1) - fx_mulhi(sq - sp, 0x2AAAAAAAAAAAAAABll);   // 2^64 / 6
}

// Colella & Woodward's limits of the parabola through l, c, r, as in ppm_limit: with
// p = r - c and q = c - l, flat unless p and q agree in sign, else neither overshoots
// twice the other (3c - 2r = c - 2p, 3c - 2l = c + 2q)
GRMHD_HD void fx_limit(long long c, long long& l, long long& r)
{
    const long long p = r - c, q = c - l;
    const long long n = p >> 63;
    const long long ap = (p ^ n) - n, aq = (q ^ n) - n;   // |p|, and q with p's sign taken out
    const bool same = aq > 0 && ap > 0;
    const unsigned long long up = (unsigned long long)ap, uq = (unsigned long long)aq;   // read where same
    const long long p1 = up > 2 * uq ? 2 * aq : ap, q1 = uq > 2 * up ? 2 * ap : aq;
    r = same ? c + ((p1 ^ n) - n) : c;
    l = same ? c - ((q1 ^ n) - n) : c;
}

// The edge states lo = b - h, hi = b + h of cell b with its MC half slope h; false (and
// no valid states) where the window needs the FP64 sequence.  Branch-free, so that the
// independent quantities of a march interleave.
GRMHD_HD bool fx_mc_cell(double a, double b, double x, double& lo, double& hi)
{
    const unsigned ea = fx_exp(a), eb = fx_exp(b), ex = fx_exp(x);
    const unsigned top = fx_max(ea, fx_max(eb, ex));
    const unsigned la = fx_max(eb, ex) + (5u << 20), lx = fx_max(ea, eb) + (5u << 20);
    const unsigned fa = ea < la ? ea : la, f = ex < lx ? ex : lx;
    const unsigned E0 = fx_max(fx_max(fa, f), eb), E = fx_max(E0, kFxMinE);
    const long long c = fx_cut(b, eb, E), h = fx_half_slope(fx_cut(a, fa, E), c, fx_cut(x, f, E));
    lo = h ? fx_to(c - h, E) : b;
    hi = h ? fx_to(c + h, E) : b;
    return top < 0x7ff00000u && (E0 >= kFxMinE || (eb | (ea < ex ? ea : ex)) == 0u);
}

// PPM at cell a0 with the next two cells a1, x, the slope s0 of a0 and the interface value
// ip below it: the limited edge states lo, hi of a0, the interface value `in` between a0
// and a1 and the slope s1 of a1.  ip and s0 enter to the block's last place, 2^-9 ulp of
// its largest value.  False where the window needs the FP64 sequence.  Branch-free.
GRMHD_HD bool fx_ppm_cell(double a0, double a1, double x, double s0, double ip, double& lo, double& hi, double& in,
                          double& s1)
{
    const unsigned es = fx_exp(s0), ei = fx_exp(ip);
    const unsigned E = fx_max(fx_block(a0, a1, x), fx_max(es, ei));
    const bool ok = fx_finite(E) && fx_near(a0, E) && fx_near(a1, E) && fx_near(x, E);
    const long long c0 = fx_of(a0, E), c1 = fx_of(a1, E);
    const long long h1 = fx_half_slope(c0, c1, fx_of(x, E));
    const long long f = fx_iface(c0, c1, fx_cut(s0, es, E), 2 * h1);
    long long l = fx_cut(ip, ei, E), r = f;
    fx_limit(c0, l, r);
    lo = fx_to(l, E);
    hi = fx_to(r, E);
    in = fx_to(f, E);
    s1 = fx_to(2 * h1, E);
    return ok;
}

}  // namespace grmhd
