// 64-bit fixed-point complex arithmetic for the FP64 transforms (sm_103a).
//
// What bounds an FP64 transform on this part is the FP64 pipe: 1.97 FMA per clock and SM, against
// 114 32-bit integer adds, 57 64-bit adds and 24-32 wide integer multiply-adds (measured). A line is
// therefore transformed in 64-bit integers with one power-of-two scale per line: a complex add
// costs 0.035 clk per SM instead of 1.0, a twiddle multiply about 0.55 instead of 2.0.
//
// Precision. Every intermediate of an FFT network is a sum of inputs times unit twiddles, so it is
// bounded by the norm sum |z| of the line. The line is scaled so that a bound of this norm (at most 8 %
// above it) lies in [0.455, 0.91) 2^63: no stage can overflow and none needs a shift. One unit is then at most
// 2^-61.8 of that bound, and a twiddle multiply is off by at most 2.5 units (0.55 in the mean square). A power
// of two for the scale costs up to a bit, so what counts is the error at the bottom of the octave: mean relative
// error in the 2-norm at the worst of eight scales, 1e-16, fixed point / FP64 (radix-4 Stockham), against long
// double (tests/test_fixed_point.py):
//   points   noise       uniform in [0, 1]   unit modulus   crack profile   1 + 1e-6 noise   8 decades
//      128   0.48 / 1.65    0.52 / 1.52       0.50 / 1.67    0.52 / 1.61      0.53 / 1.72    0.48 / 1.63
//      512   0.70 / 1.89    0.71 / 1.79       0.70 / 1.90    0.51 / 1.64      0.68 / 2.03    0.50 / 1.88
//     1024   1.26 / 2.00    1.32 / 1.86       1.48 / 2.01    0.51 / 1.67      1.46 / 2.07    0.61 / 1.97
// (With the sum of |re| + |im| below 2^62 as the bound, lines of 1024 points reached 2.5 to 3.4.) Twiddles
// made on the host carry 62 fraction bits; those that rve_dissipation_noalloc makes on the device are rounded to
// doubles first, as FP64 ones are, and add at most 0.4 to the first figures. A line with an infinity or a NaN
// gives NaN throughout, and so does one whose norm passes 2^1024; subnormal inputs and results count as zero.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace pff {

struct __align__(16) fx2 { long long x, y; };
// Twiddle w = re + i im, each as hi 2^-30 + lo 2^-62 with |hi| <= 2^30, |lo| < 2^31.
struct __align__(16) fxw { int rh, rl, ih, il; };

__device__ __forceinline__ fx2 cadd(fx2 a, fx2 b) { return fx2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ fx2 csub(fx2 a, fx2 b) { return fx2{a.x - b.x, a.y - b.y}; }

// Split x = hi 2^32 + lo, |lo| <= 2^31: lo is the low word as a signed number (|x| < 2^63 - 2^31), hi one
// shift-and-add. FP64 solves are 2.3 % faster than with a shift and a mask at 31 bits, 5 % faster than with the
// carry of x + 2^31.
__device__ __forceinline__ void fx_split(long long x, int &hi, int &lo) {
    lo = (int)x;
    hi = (int)(x >> 32) + (int)((unsigned)lo >> 31);
}
// a w: four times the products of the high parts (units of 2^32 2^-30), plus the cross products (2^32 2^-62 and
// 2^-30) shifted by 30 bits and rounded; the products of the low parts, of either sign and at most one unit each,
// are dropped. With |a| <= 0.91 2^63 the cross sum stays below 2^62 (0.91 sqrt 2 + 1 / sqrt 2) = 1.995 2^62,
// which is what the limit of 0.91 is for.
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
    return fx2{(cr >> 30) + 4 * hr, (ci >> 30) + 4 * hi};
}
// x sqrt(1/2), the factor as hi 2^-30 + lo 2^-62
constexpr int kR2h = 759250125, kR2l = -25716447;
__device__ __forceinline__ long long fx_mul_r2(long long x) {
    int xh, xl;
    fx_split(x, xh, xl);
    long long c = 1 << 29;
    c += (long long)xh * kR2l;
    c += (long long)xl * kR2h;
    return (c >> 30) + 4 * ((long long)xh * kR2h);
}

// ---- conversion of a line ------------------------------------------------------------------------
// Scale of a line: value = integer * 2^-k. mx: the largest high word (sign cleared) of the line,
// norm: the bound of its norm in units of 2^(E - 1023 - 63), E = mx >> 20 (the sum of fx_norm_term).
__device__ __forceinline__ unsigned fx_hi_abs(double d) { return (unsigned)__double2hiint(d) & 0x7fffffffu; }
// |d| as a float relative to the exponent of the largest value: the exponent field is rebased so
// that E becomes 190 (values 2^-190 below the largest count as zero), the 20 high mantissa bits kept.
__device__ __forceinline__ float fx_rel_abs(unsigned ha, unsigned base) {
    const int t = (int)ha - (int)base;
    return __int_as_float((t > 0 ? t : 0) << 3);
}
// An upper bound of |re + i im|: max + (sqrt 2 - 1) min, the chord of sqrt(1 + t^2) over [0, 1]. At most 8 %
// above it, where |re| + |im| is up to 41 % above: 0.4 bits for two more operations per point.
__device__ __forceinline__ float fx_norm_term(unsigned hre, unsigned him, unsigned base) {
    return fx_rel_abs(hre > him ? hre : him, base) + 0.4142136f * fx_rel_abs(hre > him ? him : hre, base);
}
__device__ __forceinline__ unsigned fx_norm_base(unsigned mx) { return (mx & 0x7ff00000u) - (190u << 20); }
// k with norm 2^k in [0.455, 0.91) 2^63 (1.0991: 1 / 0.91, and 1e-4 for the truncation of the terms and the
// rounding of their sum), one less where a single value would reach 2^62 (fx_in); 0 for a zero line
__device__ __forceinline__ int fx_scale(unsigned mx, float norm) {
    if (mx < 0x00100000u) return 0;
    const int fl = (int)(__float_as_uint(norm * 1.0991f) >> 23) - 127;  // floor(log2)
    const int E = (int)(mx >> 20), k = 62 - (fl + E - 1023 - 63);
    return k < 1084 - E ? k : 1084 - E;
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
// +-u 2^-k as a double (sg = 0 or -1), rounded half up; e0 = 1086 - k (biased exponent of bit 63). Results below
// the normal range are zero.
__device__ __forceinline__ double fx_out_abs(unsigned long long u, long long sg, int e0) {
    const bool zero = u == 0;
    const int lz = __clzll((long long)u);
    u <<= (lz & 63);
    const unsigned long long m = (u >> 11) + ((u >> 10) & 1);
    const int e = e0 - lz;
    unsigned long long b = m + ((unsigned long long)(unsigned)(e - 1) << 52);
    if (zero || e < 1) b = 0;
    return __longlong_as_double((long long)(b | ((unsigned long long)sg & 0x8000000000000000ull)));
}
__device__ __forceinline__ double fx_out(long long x, int e0) {
    const long long sg = x >> 63;
    return fx_out_abs((unsigned long long)((x ^ sg) - sg), sg, e0);
}
// (x + y) 2^-k: the sum may need 65 bits, its size fits 64. Its sign is that of x and y where they agree, else
// that of the wrapped sum, which is the majority of the three.
__device__ __forceinline__ double fx_out_sum(long long x, long long y, int e0) {
    const unsigned long long a = (unsigned long long)x, b = (unsigned long long)y, w = a + b;
    const long long sg = (long long)((a & b) | (a & w) | (b & w)) >> 63;
    return fx_out_abs((w ^ (unsigned long long)sg) - (unsigned long long)sg, sg, e0);
}
__device__ __forceinline__ double fx_nan() { return __longlong_as_double(0x7ff8000000000000LL); }

// ---- butterflies -----------------------------------------------------------------------------------
// 4- and 8-point DFTs, natural order in and out (forward).
__device__ __forceinline__ void fx_dft4(fx2 &a, fx2 &b, fx2 &c, fx2 &d) {
    const fx2 p = cadd(a, c), m = csub(a, c), q = cadd(b, d), r = csub(b, d);
    a = cadd(p, q);
    b.x = m.x + r.y; b.y = m.y - r.x;
    c = csub(p, q);
    d.x = m.x - r.y; d.y = m.y + r.x;
}
__device__ __forceinline__ void fx_dft8(fx2 (&v)[8]) {
    fx2 e[4], o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        e[j] = cadd(v[j], v[j + 4]);
        o[j] = csub(v[j], v[j + 4]);
    }
    // odd outputs: o_j w_8^j, w_8 = (1 - i) / sqrt 2 (the scaling before the sums: no fixed-point overflow)
    const long long x1 = fx_mul_r2(o[1].x), y1 = fx_mul_r2(o[1].y), x3 = fx_mul_r2(o[3].x), y3 = fx_mul_r2(o[3].y);
    o[1].x = x1 + y1; o[1].y = y1 - x1;
    const fx2 t = o[2];
    o[2].x = t.y; o[2].y = -t.x;
    o[3].x = y3 - x3; o[3].y = -x3 - y3;
    fx_dft4(e[0], e[1], e[2], e[3]);
    fx_dft4(o[0], o[1], o[2], o[3]);
#pragma unroll
    for (int j = 0; j < 4; ++j) { v[2 * j] = e[j]; v[2 * j + 1] = o[j]; }
}
// One self-sorting pass of a line of 2^lgL points, 2^lgN points of whose sub-transforms are done, for thread t
// of 2^lgT: v[m] is point t + (m << lgT). Radix 8 as long as three levels are left, then 4 or 2. True after
// the last pass, which leaves v[m] at that point; else v[r] goes to fx_pass_out(lgN, t) + (r << lgN).
__device__ __forceinline__ int fx_pass_out(int lgN, int t) {
    const int kk = t & ((1 << lgN) - 1);
    return ((t - kk) << 3) + kk;
}
__device__ __forceinline__ bool fx_pass(fx2 (&v)[8], int lgL, int lgT, int lgN, int t, const fxw *__restrict__ tw) {
    const int left = lgL - lgN;
    if (left >= 3) {
        const int kk = t & ((1 << lgN) - 1);
        if (lgN > 0) {
#pragma unroll
            for (int r = 1; r < 8; ++r) v[r] = cmul(v[r], tw[(r * kk) << (left - 3)]);
        }
        fx_dft8(v);
        return left == 3;
    }
    if (left == 2) {
        if (lgL == 2) {
            fx_dft4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
            for (int b = 0; b < 2; ++b) {
                const int j = t + (b << lgT);
#pragma unroll
                for (int r = 1; r < 4; ++r) v[b + 2 * r] = cmul(v[b + 2 * r], tw[r * j]);
                fx_dft4(v[b], v[b + 2], v[b + 4], v[b + 6]);
            }
        }
    } else {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const fx2 c = cmul(v[b + 4], tw[t + (b << lgT)]);
            v[b + 4] = csub(v[b], c);
            v[b] = cadd(v[b], c);
        }
    }
    return true;
}

// Host side: the twiddle exp(-2 pi i m / L) in fxw form.
static inline fxw fx_twiddle_host(long long m, long long L) {
    const long double a = -2.0L * 3.14159265358979323846264338327950288L * (long double)m / (long double)L;
    auto put = [](long double v, int &h, int &l) {
        const long double s = v * 1073741824.0L;
        h = (int)llrintl(s);
        const long long r = llrintl((s - (long double)h) * 4294967296.0L);
        l = (int)(r > 2147483647ll ? 2147483647ll : r < -2147483647ll ? -2147483647ll : r);
    };
    fxw w;
    put(cosl(a), w.rh, w.rl);
    put(sinl(a), w.ih, w.il);
    return w;
}

}  // namespace pff
