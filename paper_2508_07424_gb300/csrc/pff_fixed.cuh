// 64-bit fixed-point complex arithmetic for the FP64 transforms (sm_103a).
//
// What bounds an FP64 transform on this part is the FP64 pipe: 1.97 FMA per clock and SM, against
// 114 32-bit integer adds, 57 64-bit adds and 24-32 wide integer multiply-adds (measured). A line is
// therefore transformed in 64-bit integers with one power-of-two scale per line: a complex add
// costs 0.035 clk per SM instead of 1.0, a twiddle multiply about 0.55 instead of 2.0.
//
// Precision. Every intermediate of an FFT network is a sum of inputs times unit twiddles, so it is
// bounded by the L1 norm of the line (sum of |re| + |im|). The line is scaled so that this norm
// lies in [2^61, 2^62): no stage can overflow and none needs a shift. One unit is then at most 2^-61 of the
// L1 norm, each twiddle multiply rounds to half a unit, and the twiddles carry 61 fraction bits.
// Forward and inverse transforms of 4 to 1024 points against long double, mean relative error in the
// 2-norm, fixed point / FP64 (radix-4 Stockham): white noise 0.9e-16 / 1.9e-16 at 512 points and
// 1.6e-16 / 2.0e-16 at 1024 (the worst ratio); fields with crack-tip peaks 0.5e-16 / 1.7e-16; 8 decades of
// magnitude 0.5e-16 / 1.6e-16. A line with an infinity or a NaN gives NaN throughout; subnormal
// inputs count as zero.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pff {

struct __align__(16) fx2 { long long x, y; };
// Twiddle w = re + i im, each as hi 2^-30 + lo 2^-61 with |hi| <= 2^30, |lo| <= 2^30.
struct __align__(16) fxw { int rh, rl, ih, il; };

__device__ __forceinline__ fx2 cadd(fx2 a, fx2 b) { return fx2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ fx2 csub(fx2 a, fx2 b) { return fx2{a.x - b.x, a.y - b.y}; }

// Split x = hi 2^31 + lo, 0 <= lo < 2^31 (|x| < 2^62, so hi fits 32 bits).
__device__ __forceinline__ void fx_split(long long x, int &hi, int &lo) {
    hi = (int)(x >> 31);
    lo = (int)x & 0x7fffffff;
}
// a w: twice the products of the high parts (units of 2^31 2^-30), plus the cross products shifted by
// 30 bits and rounded; the product of the low parts (at most half a unit) is dropped. With |w| = 1
// and |a| < 2^62 the sum of the high products stays below 2^61 and the cross sum below 2^63.
__device__ __forceinline__ fx2 cmul(fx2 a, fxw w) {
    int xh, xl, yh, yl;
    fx_split(a.x, xh, xl);
    fx_split(a.y, yh, yl);
    const int nh = -w.ih, nl = -w.il;
    long long cr = 1 << 29, ci = 1 << 29;
    cr += (long long)xh * w.rl;
    cr += (long long)xl * w.rh;
    cr += (long long)yh * nl;
    cr += (long long)yl * nh;
    ci += (long long)xh * w.il;
    ci += (long long)xl * w.ih;
    ci += (long long)yh * w.rl;
    ci += (long long)yl * w.rh;
    const long long hr = (long long)xh * w.rh + (long long)yh * nh;
    const long long hi = (long long)xh * w.ih + (long long)yh * w.rh;
    return fx2{(cr >> 30) + 2 * hr, (ci >> 30) + 2 * hi};
}
// x sqrt(1/2), the factor as hi 2^-30 + lo 2^-61
constexpr int kR2h = 759250125, kR2l = -12858223;
__device__ __forceinline__ long long fx_mul_r2(long long x) {
    int xh, xl;
    fx_split(x, xh, xl);
    long long c = 1 << 29;
    c += (long long)xh * kR2l;
    c += (long long)xl * kR2h;
    return (c >> 30) + 2 * ((long long)xh * kR2h);
}

// ---- conversion of a line ------------------------------------------------------------------------
// Scale of a line: value = integer * 2^-k. mx: the largest high word (sign cleared) of the line,
// l1: its L1 norm in units of 2^(E - 1023 - 63), E = mx >> 20 (fx_l1_term).
__device__ __forceinline__ unsigned fx_hi_abs(double d) { return (unsigned)__double2hiint(d) & 0x7fffffffu; }
// |d| as a float relative to the exponent of the largest value: the exponent field is rebased so
// that E becomes 190 (values 2^-190 below the largest count as zero), the 20 high mantissa bits kept.
__device__ __forceinline__ float fx_l1_term(unsigned ha, unsigned base) {
    const int t = (int)ha - (int)base;
    return __int_as_float((t > 0 ? t : 0) << 3);
}
__device__ __forceinline__ unsigned fx_l1_base(unsigned mx) { return (mx & 0x7ff00000u) - (190u << 20); }
// k with l1 2^k in [2^61, 2^62) (l1 raised by the truncation of its terms); 0 for a zero line
__device__ __forceinline__ int fx_scale(unsigned mx, float l1) {
    if (mx < 0x00100000u) return 0;
    const int fl = (int)(__float_as_uint(l1 * 1.0001f) >> 23) - 127;  // floor(log2)
    return 61 - (fl + (int)(mx >> 20) - 1023 - 63);
}
// d 2^k rounded to an integer. The mantissa sits at bits 10..62 and is shifted down by
// 1085 - e - k >= 1 bits, at most 64: from there on the value is below half a unit and (m >> 63) + 1 rounds to
// zero (at 63 it would give one unit to every value however small, and the tails of a line would add up).
__device__ __forceinline__ long long fx_in(double d, int k) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d);
    const int hi = (int)(b >> 32);
    const int e = (hi >> 20) & 0x7ff;
    int s = 1085 - e - k;
    s = s < 64 ? s : 64;
    const unsigned long long m = (((b & 0xfffffffffffffull) | 0x10000000000000ull) << 10);
    unsigned long long u = (m >> (s - 1)) + 1;
    u >>= 1;
    if (e == 0) u = 0;
    const long long sg = (long long)(hi >> 31);
    return (long long)((u ^ (unsigned long long)sg) - (unsigned long long)sg);
}
// x 2^-k as a double, rounded half up; e0 = 1086 - k (biased exponent of bit 63). Results below the
// normal range are zero.
__device__ __forceinline__ double fx_out(long long x, int e0) {
    const long long sg = x >> 63;
    unsigned long long u = (unsigned long long)((x ^ sg) - sg);
    const int lz = __clzll((long long)u);
    u <<= (lz & 63);
    const unsigned long long m = (u >> 11) + ((u >> 10) & 1);
    const int e = e0 - lz;
    unsigned long long b = m + ((unsigned long long)(unsigned)(e - 1) << 52);
    if (x == 0 || e < 1) b = 0;
    return __longlong_as_double((long long)(b | ((unsigned long long)sg & 0x8000000000000000ull)));
}
__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000LL); }

// Host side: the twiddle exp(-2 pi i m / L) in fxw form.
static inline fxw fx_twiddle_host(long long m, long long L) {
    const long double a = -2.0L * 3.14159265358979323846264338327950288L * (long double)m / (long double)L;
    auto put = [](long double v, int &h, int &l) {
        const long double s = v * 1073741824.0L;
        h = (int)llrintl(s);
        l = (int)llrintl((s - (long double)h) * 2147483648.0L);
    };
    fxw w;
    put(cosl(a), w.rh, w.rl);
    put(sinl(a), w.ih, w.il);
    return w;
}

}  // namespace pff
