// fx.cuh - 64-bit fixed-point arithmetic of the FP64 transforms.
//
// This GPU issues 2 FP64 operations per SM and clock, but 64 two-word additions and 28 32 x 32 + 64-bit
// multiply-adds (measured lane-operations per SM and clock at 2.07 GHz: fma.f64 1.9, add.cc + addc 51,
// product-and-sum 28.5).  A Fourier transform of one line has a known range (|X| <= the number of its
// inputs times their largest modulus), so its FP64 transforms run here on integers: the line is
// scaled by a power of two that leaves exactly that headroom, every butterfly addition is exact, and
// only products round, to one unit of the last place.  The results' unit is 2^-57 (L = 16) to 2^-53
// (inverse transforms of L = 512) of the line's largest input; the first step, and half of the
// 32-point DFT, work in units 4 to 16 times finer.  (FP64's own unit is 2^-53 of each value.)  Against
// longdouble a line's rms error is 0.2 to 1.0 of that of the same plan in FP64, in the worst of six
// kinds of fields 0.88 on inverse lines at L = 512 (tests/test_fixed_point_lines.py).  Inputs and
// outputs stay FP64 in memory.
// Measured at 128^3, one system: FP64 apply 9.05 -> 2.13 ms (z pass 5.21 -> 0.93, y passes 1.05 -> 0.175
// each, inverse x 0.57 -> 0.12, contrast source and forward x 0.76 -> 0.31).
//
// Numbers.  A value is a signed 64-bit integer v standing for v 2^E, E shared by its line.
// Twiddles and constants are two signed words W = W1 2^-w + W0 2^-2w, w = 31 or 32; a product splits
// v = h 2^w + l and keeps h W1 + (l W1 + h W0 + 2^(w-1)) 2^-w, dropping only l W0 2^-2w (below half a
// unit).  Summing the middle words in 32 bits by mad.hi was no faster (z pass 1.55 ms either way, before
// fx_mad had its present form) and its truncations cost accuracy.
//
// Two units.  The first step of a two-step transform grows its inputs by far less than the whole, so
// it runs in a unit 2^-K of the second's (fx_prescale; the twiddles between the steps carry the
// factor 2^-K): what the inputs lose to rounding is then negligible, and a line's error is that of
// the twiddled values and the last butterflies' constants.
#pragma once
#include "common.cuh"
#include <cmath>

namespace lsm {

// A 64-bit value as its two words.  Kept as words: the assembler then spends two instructions on a
// sum or a difference (3.3 when the same sums are written on 64-bit operands).
struct fxr {
    unsigned l;
    int h;
};
struct __align__(16) fxc {   // complex fixed-point value
    fxr x, y;
};
template <> struct real_of<fxc> { typedef fxr type; };

__host__ __device__ __forceinline__ long long fx_ll(fxr a) { return (long long)((unsigned long long)(unsigned)a.h << 32 | a.l); }
__host__ __device__ __forceinline__ fxr fx_r(long long v) {
    fxr r;
    r.l = (unsigned)v;
    r.h = (int)(v >> 32);
    return r;
}
#ifdef __CUDACC__
#define FX_RANGE(ok)
__device__ __forceinline__ fxr fx_add(fxr a, fxr b) {
    fxr r;
    asm("add.cc.u32 %0, %2, %4; addc.u32 %1, %3, %5;" : "=r"(r.l), "=r"(r.h) : "r"(a.l), "r"(a.h), "r"(b.l), "r"(b.h));
    return r;
}
__device__ __forceinline__ fxr fx_sub(fxr a, fxr b) {
    fxr r;
    asm("sub.cc.u32 %0, %2, %4; subc.u32 %1, %3, %5;" : "=r"(r.l), "=r"(r.h) : "r"(a.l), "r"(a.h), "r"(b.l), "r"(b.h));
    return r;
}
// a b + c.  As a product and a sum the assembler makes one multiply-add of it (28 per SM and clock, on
// the FMA pipe alone); mad.wide.s32 came out as 2.5 instructions (23 per clock), and C as a 64 x 64
// bit product where it knows an operand to be non-negative.
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) {
    long long r;
    asm("{.reg .s64 t; mul.wide.s32 t, %1, %2; add.s64 %0, t, %3;}" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
__device__ __forceinline__ long long fx_pack(unsigned l, int h) {
    long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(l), "r"(h));
    return r;
}
__device__ __forceinline__ fxr fx_words(long long v) {
    fxr r;
    asm("mov.b64 {%0, %1}, %2;" : "=r"(r.l), "=r"(r.h) : "l"(v));
    return r;
}
#else
// Host form, for tests of this arithmetic on the CPU: the same results, with every sum and every
// factor's range checked.
static long fx_range_errors = 0;
#define FX_RANGE(ok) (fx_range_errors += !(ok))
inline fxr fx_add(fxr a, fxr b) {
    long long r;
    FX_RANGE(!__builtin_add_overflow(fx_ll(a), fx_ll(b), &r));
    return fx_r(r);
}
inline fxr fx_sub(fxr a, fxr b) {
    long long r;
    FX_RANGE(!__builtin_sub_overflow(fx_ll(a), fx_ll(b), &r));
    return fx_r(r);
}
inline long long fx_mad(int a, int b, long long c) {
    long long r;
    FX_RANGE(!__builtin_add_overflow((long long)a * b, c, &r));
    return r;
}
inline long long fx_pack(unsigned l, int h) { return fx_ll(fxr{l, h}); }
inline fxr fx_words(long long v) { return fx_r(v); }
#endif
__device__ __forceinline__ fxr fx_neg(fxr a) { return fx_sub(fxr{0u, 0}, a); }
__device__ __forceinline__ long long fx_sext(int h) { return fx_pack((unsigned)h, h >> 31); }
template <> __device__ __forceinline__ fxc cadd<fxc>(fxc a, fxc b) { return fxc{fx_add(a.x, b.x), fx_add(a.y, b.y)}; }
template <> __device__ __forceinline__ fxc csub<fxc>(fxc a, fxc b) { return fxc{fx_sub(a.x, b.x), fx_sub(a.y, b.y)}; }
template <> __device__ __forceinline__ fxc czero<fxc>() { return fxc{fxr{0u, 0}, fxr{0u, 0}}; }
// a + S i b and a - S i b
template <int S> __device__ __forceinline__ fxc fx_addi(fxc a, fxc b) {
    return S > 0 ? fxc{fx_sub(a.x, b.y), fx_add(a.y, b.x)} : fxc{fx_add(a.x, b.y), fx_sub(a.y, b.x)};
}
template <int S> __device__ __forceinline__ fxc fx_subi(fxc a, fxc b) { return fx_addi<-S>(a, b); }
template <int S> __device__ __forceinline__ fxc cmul_si(fxc a) {
    return S > 0 ? fxc{fx_neg(a.y), a.x} : fxc{a.y, fx_neg(a.x)};
}
// bits 31 .. 62 of v, and v >> 31
__device__ __forceinline__ int fx_sr31w(fxr v) { return (int)__funnelshift_l(v.l, (unsigned)v.h, 1); }
__device__ __forceinline__ long long fx_sr31(long long t) {
    const fxr v = fx_words(t);
    return fx_pack((unsigned)fx_sr31w(v), v.h >> 31);
}

// 2^62 times a butterfly constant, looked up by its FP64 value (callers pass literals, so the
// lookup folds at compile time)
__host__ __device__ __forceinline__ constexpr long long fx_const_abs(double c) {
    return c == 0.92387953251128675613 ? 4260642322793532497LL    // cos(pi/8)
         : c == 0.38268343236508977173 ? 1764815834521887442LL    // sin(pi/8)
         : c == 0.70710678118654752440 ? 3260954456333195553LL    // 1/sqrt(2)
         : c == 0.98078528040323044913 ? 4523073764714963030LL    // cos(pi/16)
         : c == 0.19509032201612826785 ? 899695310372275547LL     // sin(pi/16)
         : c == 0.83146961230254523708 ? 3834476785802888710LL    // cos(3 pi/16)
         : c == 0.55557023301960222474 ? 2562115475870945497LL    // sin(3 pi/16)
         : c == 0.86602540378443864676 ? 3993837246235628775LL    // sqrt(3)/2
         : c == 0.30901699437494742410 ? 1425089352415399811LL    // cos(2 pi/5)
         : c == 0.80901699437494742410 ? 3730932361629093763LL    // -cos(4 pi/5)
         : c == 0.95105651629515357212 ? 4385974038932618941LL    // sin(2 pi/5)
         : c == 0.58778525229247312917 ? 2710681029835013083LL    // sin(4 pi/5)
                                       : 0x7fffffffffffffffLL;    // not a constant of the butterflies
}
__host__ __device__ __forceinline__ constexpr long long fx_const(double c) {
    return c < 0 ? -fx_const_abs(-c) : fx_const_abs(c);
}

// v = h 2^32 + l with l signed
__device__ __forceinline__ void fx_split(fxr v, int& h, int& l) {
    FX_RANGE(fx_ll(v) < 0x7fffffff80000000LL);
    l = (int)v.l;
    h = v.h + (int)(v.l >> 31);
}
__host__ __device__ __forceinline__ constexpr int fx_w1(long long k) { return (int)((k + (1LL << 30)) >> 31); }
__host__ __device__ __forceinline__ constexpr int fx_w0(long long k) {
    return (int)(k - ((long long)fx_w1(k) << 31));
}
// v k 2^-62 (|v| < 2^62)
__device__ __forceinline__ fxr fx_scale(fxr v, long long k) {
    FX_RANGE(fx_ll(v) >> 62 == fx_ll(v) >> 63);
    const int v1 = fx_sr31w(v), v0 = (int)(v.l & 0x7fffffffu);
    const int w1 = fx_w1(k), w0 = fx_w0(k);
    const long long t = fx_mad(v1, w0, fx_mad(v0, w1, 1LL << 30));
    return fx_words(fx_mad(v1, w1, fx_sr31(t)));
}
// a (re + i im), re = r1 2^-31 + r0 2^-62 and so im (|a| < 2^60.67)
__device__ __forceinline__ fxc fx_cmul(fxc a, int r1, int r0, int i1, int i0) {
    FX_RANGE(fx_ll(a.x) >> 62 == fx_ll(a.x) >> 63 && fx_ll(a.y) >> 62 == fx_ll(a.y) >> 63);
    const int x1 = fx_sr31w(a.x), x0 = (int)(a.x.l & 0x7fffffffu);
    const int y1 = fx_sr31w(a.y), y0 = (int)(a.y.l & 0x7fffffffu);
    const long long tr = fx_mad(y1, -i0, fx_mad(y0, -i1, fx_mad(x1, r0, fx_mad(x0, r1, 1LL << 30))));
    const long long ti = fx_mad(y1, r0, fx_mad(y0, r1, fx_mad(x1, i0, fx_mad(x0, i1, 1LL << 30))));
    return fxc{fx_words(fx_mad(y1, -i1, fx_mad(x1, r1, fx_sr31(tr)))), fx_words(fx_mad(y1, r1, fx_mad(x1, i1, fx_sr31(ti))))};
}
// a (re + i im), re = r1 2^-32 + r0 2^-64 and so im, both at most 1/4 (the two-step plans' scaled
// twiddles; |a| < 2^62): the split falls on the words and the shift of the middle sum costs one
// instruction
__device__ __forceinline__ fxc fx_cmul32(fxc a, int r1, int r0, int i1, int i0) {
    int xh, xl, yh, yl;
    fx_split(a.x, xh, xl);
    fx_split(a.y, yh, yl);
    const fxr tr = fx_words(fx_mad(yh, -i0, fx_mad(yl, -i1, fx_mad(xh, r0, fx_mad(xl, r1, 1LL << 31)))));
    const fxr ti = fx_words(fx_mad(yh, r0, fx_mad(yl, r1, fx_mad(xh, i0, fx_mad(xl, i1, 1LL << 31)))));
    return fxc{fx_words(fx_mad(yh, -i1, fx_mad(xh, r1, fx_sext(tr.h)))), fx_words(fx_mad(yh, r1, fx_mad(xh, i1, fx_sext(ti.h))))};
}
// v k 2^-62 for |v| < 2^63, one more multiply-add (k < 2^62 a constant whose low word is below 2^30)
__device__ __forceinline__ fxr fx_scale_wide(fxr v, long long k) {
    int h, l;
    fx_split(v, h, l);
    const int k1 = fx_w1(k), k0 = 2 * fx_w0(k);
    const long long t = fx_mad(h, k0, fx_mad(l, k1, 1LL << 30));
    return fx_words(fx_mad(h, k1, fx_mad(h, k1, fx_sr31(t))));
}
// a (re + i im) / 4, re = kr 2^-62 and so im, |re + i im| = 1 (|a| < 2^62.7)
__device__ __forceinline__ fxc fx_cmul_quarter(fxc a, long long kr, long long ki) {
    const int r1 = (int)((kr + (1LL << 31)) >> 32), i1 = (int)((ki + (1LL << 31)) >> 32);
    return fx_cmul32(a, r1, (int)(kr - ((long long)r1 << 32)), i1, (int)(ki - ((long long)i1 << 32)));
}
// v 2^-sh, rounded to nearest, for sh of either sign; 64 or more shifts any value out
__device__ __forceinline__ fxr fx_shift(fxr v, int sh) {
    if (sh > 0) return fx_r(((fx_ll(v) >> min(sh - 1, 63)) + 1) >> 1);
    return fx_r((long long)((unsigned long long)fx_ll(v) << min(-sh, 63)));
}
// high words of the components' moduli (less one for negative ones), or-ed
__device__ __forceinline__ unsigned fx_hibits(fxc v) {
    return (unsigned)((v.x.h ^ (v.x.h >> 31)) | (v.y.h ^ (v.y.h >> 31)));
}
// +-a +-b
__device__ __forceinline__ fxr fx_pm(fxr a, bool pa, fxr b, bool pb) {
    return pa ? (pb ? fx_add(a, b) : fx_sub(a, b)) : (pb ? fx_sub(b, a) : fx_neg(fx_add(a, b)));
}
template <int S> __device__ __forceinline__ fxc cmul_const(fxc a, double re, double im_s) {
    const double im = S * im_s;
    if (re == im || re == -im) {
        // (x + i y) c (p + i q), p, q = +-1: two real products of (p x - q y) and (q x + p y)
        const long long k = fx_const(re < 0 ? -re : re);
        const bool p = re > 0, q = im > 0;
        return fxc{fx_scale(fx_pm(a.x, p, a.y, !q), k), fx_scale(fx_pm(a.x, q, a.y, p), k)};
    }
    const long long kr = fx_const(re), ki = fx_const(im);
    return fx_cmul(a, fx_w1(kr), fx_w0(kr), fx_w1(ki), fx_w0(ki));
}

// a tw[k] (S < 0) or a conj(tw[k]) (S > 0); a fixed-point entry is (W1, W0) of the real part, then
// of the imaginary part, scaled for fx_cmul32
template <int S, typename C> __device__ __forceinline__ C tw_mul(C a, const C* __restrict__ tw, int k) {
    C w = __ldg(&tw[k]);
    if (S > 0) w.y = -w.y;
    return cmul(a, w);
}
template <int S> __device__ __forceinline__ fxc tw_mul32(fxc a, const int4* __restrict__ tw, int k) {
#ifdef __CUDACC__
    // volatile: 15 entries fetched ahead of their use would spill
    int4 w;
    asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(w.x), "=r"(w.y), "=r"(w.z), "=r"(w.w) : "l"(tw + k));
#else
    const int4 w = tw[k];
#endif
    return S > 0 ? fx_cmul32(a, w.x, w.y, -w.z, -w.w) : fx_cmul32(a, w.x, w.y, w.z, w.w);
}
// v (|v| <= 1/4) as the two-word fixed-point number v1 2^-32 + v0 2^-64, v0 within +-(2^31 - 1) so
// that either sign can be negated
inline void fx_table_words(long double v, int* v1, int* v0) {
    const long double f = 4294967296.0L, lim = 2147483647.0L;
    const long double a = nearbyintl(v * f);
    const long double b = nearbyintl((v * f - a) * f);
    *v1 = (int)a;
    *v0 = (int)(b > lim ? lim : (b < -lim ? -lim : b));
}
// K of the two-step plan of length L, and the part of it that the twiddles between the steps carry
// (L = 512: the second step is the 32-point DFT in two units, which carries the other 2)
__host__ __device__ constexpr int fx_prescale(int L) { return L == 16 ? 2 : (L == 512 ? 4 : 3); }
__host__ __device__ constexpr int fx_twiddle_k(int L) { return L == 16 || L == 512 ? 2 : 3; }

// twiddles between the steps of a two-step transform of length L: v[k1] tw[t k1].  Row t = 0 has
// none; in fixed point every entry also passes to the second step's unit (the table's entries carry
// the factor, k1 = 0 is shifted).
template <int S, int L, int A, typename C> __device__ __forceinline__ void tw_row(C* v, const C* __restrict__ tw, int t) {
    if (t) {
#pragma unroll
        for (int k1 = 1; k1 < A; ++k1) v[k1] = tw_mul<S>(v[k1], tw, t * k1);
    }
}
template <int S, int L, int A> __device__ __forceinline__ void tw_row(fxc* v, const int4* __restrict__ tw, int t) {
    constexpr int K = fx_twiddle_k(L);
    v[0].x = fx_r((fx_ll(v[0].x) + (1 << (K - 1))) >> K);
    v[0].y = fx_r((fx_ll(v[0].y) + (1 << (K - 1))) >> K);
#pragma unroll
    for (int k1 = 1; k1 < A; ++k1) v[k1] = tw_mul32<S>(v[k1], tw, t * k1);
}

// ---------------------------------------------------------------------------------------------
// FP64 <-> fixed point
// ---------------------------------------------------------------------------------------------
// high word of |v|: its maximum over a line gives the line's largest exponent
__device__ __forceinline__ unsigned fx_mag(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// Scale of a line whose largest magnitude word is mag: its values are below 2^(eb - 1022).
struct FxScale {
    int eb;       // largest biased exponent, 1 .. 2047
    bool small;   // subnormal inputs count (beside larger values they shift out to zero)
    bool bad;     // the line holds an infinity or a NaN: all its outputs are NaN
    __host__ __device__ __forceinline__ FxScale(unsigned mag) {
        eb = (int)(mag >> 20);
        bad = eb == 2047;
        small = eb < 128;
        eb = eb > 1 ? eb : 1;
    }
    // exponent of the unit of the fixed-point values when they are scaled to below 2^bits
    __host__ __device__ __forceinline__ int unit(int bits) const { return eb - 1022 - bits; }
};

// v as a multiple of the line's unit, rounded towards zero: |result| < 2^bits.  No FP64 instruction:
// the rare cases are branches the compiler must not turn into always-executed FP64 selects.
__device__ __forceinline__ fxr fx_from(double v, const FxScale& s, int bits) {
    const int hi = __double2hiint(v);
    const unsigned lo = (unsigned)__double2loint(v), a = (unsigned)hi & 0x7fffffffu;
    // shift from a leading bit at 62 to bits - 1: 63 - bits + eb - e
    unsigned sh = (((unsigned)(63 - bits + s.eb) << 20 | 0xfffffu) - a) >> 20;
    unsigned mh = (__funnelshift_l(lo, (unsigned)hi, 10) & 0x3fffffffu) | 0x40000000u;
    if (s.small && a < 0x100000u) {   // subnormal or zero: no implicit bit, exponent 1
        mh &= 0x3fffffffu;
        sh -= 1;
    }
    sh = sh < 63u ? sh : 63u;
    const fxr m = fx_r((long long)((unsigned long long)mh << 32 | (lo << 10)) >> sh);
    const int sg = hi >> 31;
    return fx_sub(fxr{m.l ^ (unsigned)sg, m.h ^ sg}, fxr{(unsigned)sg, sg});
}
__device__ __forceinline__ fxc fx_from(double2 v, const FxScale& s, int bits) {
    return fxc{fx_from(v.x, s, bits), fx_from(v.y, s, bits)};
}

// v 2^E rounded to FP64 (to nearest), with gradual underflow; results above the range are infinite.  Ties
// go towards zero: either constant costs one addition where ties to even take two instructions more,
// and the rms error of a line is the same under the three rules (mean ratio over 444 sets of lines
// 0.999, 0.999).
struct FxUnit {
    int e;       // E + 1085: one below the biased exponent of a value with no leading zeros
    bool odd;    // some v gives no normal number, or the line is bad or zero: fx_to_odd
    bool bad;
    __device__ __forceinline__ FxUnit(int E, bool nan, bool zero) {
        e = E + 1085;
        bad = nan;
        odd = nan || zero || E < -1021 || E > 960;
    }
};
__device__ __forceinline__ double fx_to(fxr v, const FxUnit& u) {
    const int sg = v.h >> 31;
    const fxr m = fx_sub(fxr{v.l ^ (unsigned)sg, v.h ^ sg}, fxr{(unsigned)sg, sg});   // < 2^63
    const bool small = m.h == 0;
    const int lz = __clz(small ? (int)m.l : m.h) + (small ? 31 : -1);   // one less than the leading zeros: leading bit to 62
    const unsigned long long n = ((unsigned long long)fx_ll(m) << lz) + 0x1ff;
    const unsigned h = (unsigned)(n >> 42) + ((unsigned)(u.e - 1 - lz) << 20);   // a carry goes into the exponent
    return __hiloint2double(small && m.l == 0 ? 0 : (int)(h | ((unsigned)sg & 0x80000000u)), (int)(unsigned)(n >> 10));
}
__device__ __forceinline__ double2 fx_to(fxc v, const FxUnit& u) { return make_double2(fx_to(v.x, u), fx_to(v.y, u)); }
__device__ __forceinline__ double fx_to_odd(fxr v, const FxUnit& u) {
    if (u.bad) return __hiloint2double(0x7ff80000, 0);
    const int sg = v.h >> 31;
    const fxr m = fx_sub(fxr{v.l ^ (unsigned)sg, v.h ^ sg}, fxr{(unsigned)sg, sg});
    if ((m.h | (int)m.l) == 0) return 0.0;
    const int be = u.e + 1 - (m.h ? __clz(m.h) : 32 + __clz((int)m.l));   // biased exponent
    if (be >= 1 && be <= 2046) return fx_to(v, u);
    const fxr q = be < 1 ? fx_shift(m, 11 - u.e) : fxr{0u, 0x7ff00000};   // below the normal range: in units of 2^-1074
    return __hiloint2double(q.h | (sg & (int)0x80000000), (int)q.l);
}
__device__ __forceinline__ double2 fx_to_odd(fxc v, const FxUnit& u) { return make_double2(fx_to_odd(v.x, u), fx_to_odd(v.y, u)); }

// Bits of a line's inputs, in the unit of the outputs: a line with at most nin nonzero inputs, each
// component below 2^bits in modulus, keeps its outputs below 2^62.6 (log2(nin) + 1/2 bits of growth).
// last: radix of the last step's DFT; 8 multiplies just before its final additions, so one bit less
// keeps those products' factors in range.  nz: nonzero inputs of a first-step DFT, whose outputs, 2^K
// finer, stay below 2^61.9.
inline int fx_bits(int L, int nin, int nz, int last) {
    const double one = 4611686018427387904.0;   // 2^62
    int b = 62;
    while (b > 0 && (double)nin * (double)(1ull << b) > 1.0717734625362931 * one) --b;   // 2^62.1
    if (last == 8) --b;
    while (b > 0 && (double)nz * (double)(1ull << b) * (1 << fx_prescale(L)) > 0.6597539553864471 * one) --b;   // 2^61.4
    return b;
}

// Spectrum entry pair for the multiply: G = (G1 2^-31 + G0 2^-61) 2^eG, one exponent for the six
// components of a point, every component below 1/2 before it.
struct FxG {
    static constexpr int ZERO_EXP = -4000;    // all six components zero
    static constexpr int BAD_EXP = 1 << 20;   // a component is not finite
};

}  // namespace lsm
