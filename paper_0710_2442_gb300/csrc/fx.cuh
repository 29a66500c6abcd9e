// fx.cuh -- FP64 products on the integer pipe: block fixed point.
//
// GB300 runs two FP64 operations per SM and clock (measured 1.88 DFMA lanes
// per clock), but 64 lanes of IMAD.WIDE (32 x 32 + 64 -> 64 bits).  A link times
// a half spinor needs no exponent per term where no component is far below the others:
// the half spinor is scaled by its own largest exponent, the link by 1 (SU(3): |U_ij| <= 1), and
// both become integers of 58 bits below the scale, in two limbs of one sign, v = h 2^29 + l.
// A real product is three IMAD.WIDE: hh += u.h v.h and mid += u.h v.l + u.l v.h; the l l term is
// below 2^-58 of the scale and is dropped (it vanishes where the link is exact in one limb).
//
// Precision.  Operands are cut at 2^-58 of the scale, and a sum of eight hops, kept in
// 64-bit integers at 2^-56, is off by about 2^-55.6 of the scale (root mean square) before it is
// rounded to FP64 once.  That is an absolute error: a component whose terms are all small against the
// scale (fields graded within a site, sparse or nearly diagonal links) would come out
// worse than from FP64 arithmetic, whose error follows the terms.  So a hop adds up, for each
// component, the moduli of its eight contributions, a lower bound of its terms', and where
// they are below 5/32 of the scale (kFxGuard) the site is done over in FP64.  Between 5/32 and
// 3/16 the error is 0.9 to 1.0 of the FP64 stencil's (root mean square; the worst inputs tried: unit
// links, components graded by up to 2^30), above it smaller, 0.35 to 0.4 where the eight hops
// contribute alike; between 4/32 and 5/32 it would be 1.06 to 1.14.  Gaussian fields fall
// below the line at one to two sites in a million.
//
// Ranges, with the unit of a term at 2^58 = scale: |v.h| <= 2^29, |v.l| < 2^29 for
// a component, twice that after the projection's one addition; a boundary phase makes the
// limbs of their product again, |v.h| <= 2 sqrt(2) 2^29, |v.l| < 2^29.  Link entries
// |u.h| <= 1.25 2^29, |u.l| < 2^29 (SU(3), and SU(3) over a mean link of 0.8 or more).  Of six terms
// each, |hh| <= 6 1.25 2 sqrt(2) 2^58 = 21.3 2^58, to which the rounding adds at most 8 2^58, and
// |mid| <= 6 (1.25 2 + 2) 2^58 = 27 2^58 without a phase, 6 (1.25 + 2 sqrt(2)) 2^58 = 24.5 2^58 with one: below
// 2^63 = 32 2^58.  A row of a hop sums three products of moduli 1.25 sqrt(2) and 2 sqrt(2) at most,
// 15 scales, so eight hops give at most 120 2^56 < 2^63 = 128 2^56.
// Fields outside the ranges (a link entry above 1.25, exponents below 2^-423 or above 2^477,
// Inf, NaN) are reported to the caller, who does the site in FP64.
#pragma once

#include "common.cuh"

namespace wl {

// exponents (biased) of half spinors that the fixed-point path takes
constexpr int kFxEmin = 600, kFxEmax = 1500;
// |hi word| << 1 of a link's largest entry, below 1.25 + 2^-20
constexpr unsigned kFxLinkHi = 0x3FF40000u << 1;
constexpr int kFxLimb = 29;                            // bits of the low limb
constexpr int kFxLow = (1 << kFxLimb) - 1;
constexpr int kFxLinkLimb = 5 << (kFxLimb - 2);        // 1.25
constexpr double kFxU = (kFxLinkLimb + 1.0) / (1 << kFxLimb), kFx2Sqrt2 = 2.8285;
static_assert(6 * kFxU * kFx2Sqrt2 + 8 < 32, "hh");
static_assert(6 * (2 * kFxU + 2) < 32 && 6 * (kFxU + kFx2Sqrt2) < 32, "mid");
static_assert(8 * 3 * kFxU * kFx2Sqrt2 / 2 * kFx2Sqrt2 < 128, "eight hops");
// The guard: the contributions' moduli are counted in 256ths of the scale.
constexpr unsigned kFxGuard = 40;

// Right shifts that give 0 for counts of the word length and more.
__host__ __device__ __forceinline__ unsigned fx_shr32(unsigned v, unsigned s) {
#ifdef __CUDA_ARCH__
    unsigned r;
    asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(v), "r"(s));
    return r;
#else
    return s >= 32 ? 0u : v >> s;
#endif
}
__host__ __device__ __forceinline__ unsigned fx_shr64_lo(unsigned long long v, unsigned s) {
#ifdef __CUDA_ARCH__
    unsigned long long r;
    asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(s));
    return (unsigned)r;
#else
    return s >= 64 ? 0u : (unsigned)(v >> s);
#endif
}
// arithmetic, d in 0..63
__host__ __device__ __forceinline__ long long fx_sar(long long v, int d) { return v >> d; }

struct FxMag {
    int h, l;  // magnitude, h 2^29 + l, 0 <= l < 2^29
};
struct FxReal {
    int h, l;  // signed limbs
};
struct FxCplx {
    FxReal re, im;
};

// A double's exponent against a scale: both come as |hi word| << 1, the scale
// word with ones below its exponent e, so that the difference is that of the
// exponents.  fx_scale_word(e + OFF) gives the right shift of fx_mag.
__host__ __device__ __forceinline__ unsigned fx_scale_word(int e) { return (unsigned)e << 21 | 0x1FFFFFu; }
__host__ __device__ __forceinline__ unsigned fx_shift(unsigned scale, unsigned hi2) { return (scale - hi2) >> 21; }

// The magnitude of the double (hi, lo), its mantissa shifted right by t >= 5
// from the top of 64 bits.  t = 6 + e - exponent puts an exponent equal to the
// scale's below 2^58 (spinors), t = 5 + 1023 - exponent puts 1.0 at 2^58 (links).
// Zeros and denormals have t so large that nothing is left.
constexpr int kFxOffSpinor = 6, kFxOffLink = 5;
__host__ __device__ __forceinline__ FxMag fx_mag(unsigned hi, unsigned lo, unsigned t) {
    const unsigned mh = (hi & 0xFFFFFu) | 0x100000u;
    const unsigned long long M = ((unsigned long long)mh << 32 | lo) << 11;
    return FxMag{(int)fx_shr32((unsigned)(M >> 32), t + kFxLimb - 32), (int)(fx_shr64_lo(M, t) & (unsigned)kFxLow)};
}
// sg times the double's sign
__host__ __device__ __forceinline__ int fx_sign(unsigned hi, int sg) { return sg - 2 * sg * (int)(hi >> 31); }

// sg times a link entry.
__host__ __device__ __forceinline__ FxReal fx_link(unsigned hi, unsigned lo, int sg = 1) {
    const FxMag m = fx_mag(hi, lo, fx_shift(fx_scale_word(1023 + kFxOffLink), hi << 1));
    const int s = fx_sign(hi, sg);
    return FxReal{m.h * s, m.l * s};
}

// One accumulating sum of products; hh 2^58 + mid 2^29 in units of the product
// of the two 2^58 scales.  mid starts at half of its last kept bit, hh at
// the half that rounds the sum when it is shifted right by d + 2 (fx_align).
struct FxAcc {
    long long hh, mid;
};
__host__ __device__ __forceinline__ FxAcc fx_zero(long long half = 0) { return FxAcc{half, 1LL << (kFxLimb - 1)}; }
constexpr int kFxMaxShift = 60;  // of d: what is shifted further vanishes all the same
__host__ __device__ __forceinline__ void fx_mac(FxAcc& a, const FxReal& u, const FxReal& v) {
    a.hh += (long long)u.h * v.h;
    a.mid += (long long)u.h * v.l;
    a.mid += (long long)u.l * v.h;
}
// The sum with the scale at 2^58, and (with the half for d) at 2^56 of a scale 2^d larger.
__host__ __device__ __forceinline__ long long fx_sum(const FxAcc& a) { return a.hh + (a.mid >> kFxLimb); }
__host__ __device__ __forceinline__ long long fx_half(int d) { return 2LL << d; }
__host__ __device__ __forceinline__ long long fx_align(long long w, int d) { return fx_sar(w, d + 2); }
__host__ __device__ __forceinline__ FxReal fx_neg(const FxReal& a) { return FxReal{-a.h, -a.l}; }

// Links stored in this form (four 32-bit words an entry: re.h, re.l, im.h,
// im.l) mark a link out of range by re.h of their first entry.
constexpr unsigned kFxBadLink = 0x80000000u;

// n + the modulus of a contribution at 2^56, in 2^-24 of the scale: eight stay below 2^31.
__host__ __device__ __forceinline__ unsigned fx_modulus(long long w, unsigned n) {
    const int x = (int)(w >> 32);
#ifdef __CUDA_ARCH__
    return __sad(x, 0, n);
#else
    return (unsigned)(x < 0 ? -x : x) + n;
#endif
}
// Two of them in 256ths of the scale, rounded down, a in the low half.
__host__ __device__ __forceinline__ unsigned fx_count(unsigned a, unsigned b) {
#ifdef __CUDA_ARCH__
    return __byte_perm(a, b, 0x7632);
#else
    return a >> 16 | b >> 16 << 16;
#endif
}
__host__ __device__ __forceinline__ unsigned fx_swap(unsigned c) { return c >> 16 | c << 16; }
__host__ __device__ __forceinline__ bool fx_below(unsigned c) { return (c & 0xFFFFu) < kFxGuard || (c >> 16) < kFxGuard; }

#ifdef __CUDACC__
// v 2^k as a double, rounded once, with two FP64 additions (the conversion
// instruction takes five): v = h 2^32 + l; the words of h (biased to unsigned)
// and l under the exponents of 2^84 and 2^52 are 2^84 + 2^63 + h 2^32 and
// 2^52 + l, and the exponent fields take k.  bias = fx_bias(k).
struct FxBias {
    int a, b;   // high words of 2^(84 + k), 2^(52 + k)
    double c;   // (2^84 + 2^63 + 2^52) 2^k
};
__device__ __forceinline__ FxBias fx_bias(int k) {
    const int s = k * (1 << 20);
    return FxBias{0x45300000 + s, 0x43300000 + s, __hiloint2double(0x45300000 + s, (int)0x80100000)};
}
__device__ __forceinline__ double fx_double(long long v, const FxBias& b) {
    const int h = (int)((unsigned)(v >> 32) ^ 0x80000000u), l = (int)(unsigned)v;
    return (__hiloint2double(b.a, h) - b.c) + __hiloint2double(b.b, l);
}
// The same, bit for bit, in integer instructions, for results that are normal or zero (kFxEmin): where
// several warps of a sub-partition convert at a time, the two additions of each wait for
// the FP64 pipe (64 cycles an instruction).
__device__ __forceinline__ double fx_double_int(long long v, int k) {
    const unsigned sg = (unsigned)(v >> 32) & 0x80000000u;
    unsigned long long m = (unsigned long long)(v < 0 ? -v : v);
    const int n = __clzll((long long)m);
    m <<= n & 63;
    const unsigned long long q = m >> 11;  // 53 bits; the others round, to nearest even
    const unsigned up = ((unsigned)m & 0x7FFu) + ((unsigned)q & 1) > 0x400u;
    // the leading bit of q adds 1 to the exponent field, a carry of the rounding another
    const unsigned long long w = q + up + ((unsigned long long)(unsigned)(1023 + 63 - 1 + k - n) << 52);
    return m ? __hiloint2double((int)((unsigned)(w >> 32) | sg), (int)(unsigned)w) : 0.0;
}
#endif

// A sum of products of link-like numbers back to limbs at 2^58, l in [0, 2^29).
__host__ __device__ __forceinline__ FxReal fx_requant(long long hh, long long mid) {
    const long long n = hh + ((mid + (1LL << (kFxLimb - 1))) >> kFxLimb);
    return FxReal{(int)(n >> kFxLimb), (int)n & kFxLow};
}
// re, im of a b - c d, for the third row of a 12-real link (conjugated by the caller)
__host__ __device__ __forceinline__ FxCplx fx_cross(const FxCplx& a, const FxCplx& b, const FxCplx& c, const FxCplx& d) {
    FxAcc r{0, 0}, i{0, 0};
    fx_mac(r, a.re, b.re);
    fx_mac(r, fx_neg(a.im), b.im);
    fx_mac(r, fx_neg(c.re), d.re);
    fx_mac(r, c.im, d.im);
    fx_mac(i, a.re, b.im);
    fx_mac(i, a.im, b.re);
    fx_mac(i, fx_neg(c.re), d.im);
    fx_mac(i, fx_neg(c.im), d.re);
    return FxCplx{fx_requant(r.hh, r.mid), fx_requant(i.hh, i.mid)};
}
// Whether the high limb of such an entry is in the links' range.  A component can reach 6.25, and wraps from 4 on
// to -4 .. -1.75: still out of it.
__host__ __device__ __forceinline__ bool fx_limb_fits(int h) { return (unsigned)h + kFxLinkLimb <= 2u * kFxLinkLimb; }
__host__ __device__ __forceinline__ void fx_recon_row2(FxCplx U[3][3]) {
#pragma unroll
    for (int q = 0; q < 3; q++) {
        const int a = (q + 1) % 3, b = (q + 2) % 3;
        U[2][q] = fx_cross(U[0][a], U[1][b], U[0][b], U[1][a]);
        U[2][q].im = fx_neg(U[2][q].im);
    }
}
// eta h (a boundary phase on a projected component)
__host__ __device__ __forceinline__ FxCplx fx_phase(const FxCplx& eta, const FxCplx& h) {
    FxAcc r{0, 0}, i{0, 0};
    fx_mac(r, eta.re, h.re);
    fx_mac(r, fx_neg(eta.im), h.im);
    fx_mac(i, eta.re, h.im);
    fx_mac(i, eta.im, h.re);
    return FxCplx{fx_requant(r.hh, r.mid), fx_requant(i.hh, i.mid)};
}

}  // namespace wl
