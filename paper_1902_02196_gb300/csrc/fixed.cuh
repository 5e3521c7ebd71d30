// 64-bit fixed-point complex numbers for the FP64 transforms.
//
// sm_103a issues two FP64 operations per clock and SM and many times as many integer ones, so an FFT whose values
// are 64-bit integers on one common power-of-two scale (block floating point) runs several times faster than the
// same FFT in FP64: a complex sum is four integer additions, a complex product with a 62-bit factor twelve
// 32 x 32 -> 64 bit multiply-adds.
//
// Error.  A value keeps up to 61 bits below its block's bound, however small it is itself; FP64 keeps 53 of its own.  The
// integers are the better ones while a block's values are within eight bits of its largest, as the values of one
// transform are, and lose where small values have nothing to do with the large ones.  So a block is a line (or
// the lines of a component that go together), and its scale is renewed before every pass.
//
// Scale.  The caller picks the scale from the largest input (block floating point) so that no
// partial sum of a transform can overflow: with n non-zero inputs of components below 2^T every
// modulus stays below sqrt(2) n 2^T, which has to be at most 2^61 (fx_room).
#pragma once

#include "common.cuh"

struct __align__(16) fx2 {
    long long x, y;
};

__device__ __forceinline__ fx2 cadd(fx2 a, fx2 b) { return fx2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ fx2 csub(fx2 a, fx2 b) { return fx2{a.x - b.x, a.y - b.y}; }
__device__ __forceinline__ fx2 cmul_i(fx2 a, int dir) { return dir < 0 ? fx2{a.y, -a.x} : fx2{-a.y, a.x}; }

// A factor c in [-1, 1] as c = hi 2^-30 + lo 2^-62 (two signed words of q = c 2^62)
__host__ __device__ __forceinline__ int fx_hi(long long q) { return (int)((q + (1LL << 31)) >> 32); }
__host__ __device__ __forceinline__ int fx_lo(long long q) { return (int)(q - ((long long)fx_hi(q) << 32)); }

// a = high 2^32 + low, both signed
__device__ __forceinline__ int fx_low(long long a) { return (int)a; }
__device__ __forceinline__ int fx_high(long long a) { return (int)(a >> 32) + (int)((unsigned)(int)a >> 31); }
__device__ __forceinline__ long long fx_mad(int a, int b, long long c) { return (long long)a * b + c; }

// a (c + i s), w = (hi c, lo c, hi s, lo s), |a| < 2^61; the low x low products are dropped (below one
// unit), the rest is rounded once.  12 wide multiply-adds.
__device__ __forceinline__ fx2 cmul(fx2 a, int4 w) {
    const int xh = fx_high(a.x), xl = fx_low(a.x), yh = fx_high(a.y), yl = fx_low(a.y);
    const int nyh = -yh, ns = -w.z;  // (yl may be -2^31, which has no negative)
    const long long hr = fx_mad(nyh, w.z, (long long)xh * w.x);
    const long long hi = fx_mad(yh, w.x, (long long)xh * w.z);
    long long lr = fx_mad(xl, w.x, 1LL << 29);
    long long li = fx_mad(xl, w.z, 1LL << 29);
    lr = fx_mad(xh, w.y, lr);
    li = fx_mad(xh, w.w, li);
    lr = fx_mad(yl, ns, lr);
    li = fx_mad(yl, w.x, li);
    lr = fx_mad(nyh, w.w, lr);
    li = fx_mad(yh, w.y, li);
    return fx2{(hr << 2) + (lr >> 30), (hi << 2) + (li >> 30)};
}
// (the twiddle table has no lo = -2^31)
__device__ __forceinline__ int4 fx_conj(int4 w) { return make_int4(w.x, w.y, -w.z, -w.w); }

// a c for a real factor q = c 2^62
__device__ __forceinline__ long long fx_scale(long long a, long long q) {
    const int ah = fx_high(a), al = fx_low(a);
    const long long l = fx_mad(ah, fx_lo(q), fx_mad(al, fx_hi(q), 1LL << 29));
    return ((long long)ah * fx_hi(q) << 2) + (l >> 30);
}

// 2^62 times the cosine or sine of a multiple of pi/16; c is one of fft2.cuh's constants (folded at compile time)
__device__ __forceinline__ constexpr long long fx_constant(double c) {
    const double m = c < 0 ? -c : c;
    const long long q = m > 0.95   ? 4523073764714963030LL
                        : m > 0.9  ? 4260642322793532497LL
                        : m > 0.8  ? 3834476785802888710LL
                        : m > 0.6  ? 3260954456333195553LL
                        : m > 0.5  ? 2562115475870945497LL
                        : m > 0.3  ? 1764815834521887442LL
                                   : 899695310372275547LL;
    return c < 0 ? -q : q;
}

// a (c + i s) with constants: the transforms of fft2.cuh on fixed-point values come through here.
// An eighth of a turn takes two real products of the sum and difference.
__device__ __forceinline__ fx2 rot(fx2 a, double c, double s) {
    const long long qc = fx_constant(c), qs = fx_constant(s);
    if (qc == qs) return fx2{fx_scale(a.x - a.y, qc), fx_scale(a.x + a.y, qc)};
    if (qc == -qs) return fx2{fx_scale(a.x + a.y, qc), fx_scale(a.y - a.x, qc)};
    return cmul(a, make_int4(fx_hi(qc), fx_lo(qc), fx_hi(qs), fx_lo(qs)));
}

// log2 of a power of two
__host__ __device__ constexpr int fx_log2(int n) { return n <= 1 ? 0 : 1 + fx_log2(n / 2); }
// bits T of the input components of a transform with n non-zero inputs (sqrt(2) n 2^T <= 2^60.5)
__host__ __device__ constexpr int fx_room(int n) { return 60 - fx_log2(n); }

// ---------------------------------------------------------------------------
// double <-> fixed point
// ---------------------------------------------------------------------------
// magnitude key of a double: exponent and leading mantissa bits; the largest key of a block gives
// the block's biased exponent E = key >> 20 (2047: an Inf or a NaN is among them)
__device__ __forceinline__ unsigned fx_key(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }
__device__ __forceinline__ unsigned fx_key(double2 v) { return max(fx_key(v.x), fx_key(v.y)); }
// the same for integers: the high word of |v| (or of |v| - 1); keys are collected by OR, which has
// the leading bit of the largest
__device__ __forceinline__ unsigned fx_key(long long v) {
    const int h = (int)(v >> 32);
    return (unsigned)(h ^ (h >> 31));
}
__device__ __forceinline__ unsigned fx_key(fx2 v) { return fx_key(v.x) | fx_key(v.y); }
// bits b with |v| <= 2^b for every v of a block with these keys
__device__ __forceinline__ int fx_bits(unsigned key) { return 64 - __clz((int)key); }
// bits that a line whose values have these keys has to drop before a pass of n points
__device__ __forceinline__ int excess(unsigned key, int n) { return max(fx_bits(key) - fx_room(n), 0); }

// A block's scale: v -> v 2^(T + 1022 - E).  Blocks below 2^-958 are raised by 2^512 first, so
// that no value of theirs is subnormal.
struct FxScale {
    int sh;      // 62 - T + E, the shift of a mantissa at bit 61 whose exponent is 0
    int ex;      // v = fixed 2^ex
    bool tiny;
    __device__ __forceinline__ FxScale(unsigned key, int T) {
        const int E0 = (int)(key >> 20);
        tiny = E0 < 64;
        const int E = tiny ? max(E0, 1) + 512 : E0;
        sh = 62 - T + E;
        ex = E - 1022 - T - (tiny ? 512 : 0);
    }
    __device__ __forceinline__ long long operator()(double v) const {
        if (tiny) v *= 0x1p512;
        const int hi = __double2hiint(v), lo = __double2loint(v);
        const unsigned long long m =
            ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)lo) << 9;
        const int r = min(sh - ((hi >> 20) & 0x7ff), 63) - 1;
        const long long a = (long long)(((m >> r) + 1) >> 1), sg = hi >> 31;
        return (a ^ sg) - sg;
    }
    __device__ __forceinline__ fx2 operator()(double2 v) const { return fx2{(*this)(v.x), (*this)(v.y)}; }
};

// v 2^ex, rounded to nearest (to a subnormal number where it is one); out of range to infinity.  INRANGE: fx_in_range(ex),
// where no v gives either
__device__ __forceinline__ bool fx_in_range(int ex) { return ex >= -1022 && ex <= 960; }
template <bool INRANGE = false>
__device__ __forceinline__ double fx_double(long long v, int ex) {
    const long long sg = v >> 63;
    const unsigned long long a = (unsigned long long)((v ^ sg) - sg);
    const int lz = __clzll((long long)a);
    const int e = 1085 - lz + ex;  // biased exponent, the leading bit of m counts as one
    const unsigned long long m = (((a << (lz & 63)) >> (INRANGE ? 10 : min(max(10 - e, 10), 63))) + 1) >> 1;
    unsigned long long bits = ((unsigned long long)(unsigned)(INRANGE ? e : max(e, 0)) << 52) + m;
    if (!INRANGE && e >= 2046) bits = 0x7ff0000000000000ull;
    if (a == 0) bits = 0;
    return __longlong_as_double((long long)(bits | ((unsigned long long)sg & 0x8000000000000000ull)));
}
template <bool INRANGE = false>
__device__ __forceinline__ double2 fx_double(fx2 v, int ex) {
    return make_double2(fx_double<INRANGE>(v.x, ex), fx_double<INRANGE>(v.y, ex));
}

// v 2^-k, rounded to nearest
__device__ __forceinline__ fx2 fx_shift(fx2 v, int k) {
    const long long h = (1LL << k) >> 1;
    return fx2{(v.x + h) >> k, (v.y + h) >> k};
}
