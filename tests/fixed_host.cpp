// The 64-bit fixed-point arithmetic of the FP64 transforms on the host, for tests/test_fixed_point.py.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <complex>
#include <cstring>
#include <vector>

static inline int __double2hiint(double d) {
    long long b;
    std::memcpy(&b, &d, 8);
    return (int)(b >> 32);
}
static inline long long __double_as_longlong(double d) {
    long long b;
    std::memcpy(&b, &d, 8);
    return b;
}
static inline double __longlong_as_double(long long b) {
    double d;
    std::memcpy(&d, &b, 8);
    return d;
}
static inline float __int_as_float(int b) {
    float f;
    std::memcpy(&f, &b, 4);
    return f;
}
static inline unsigned __float_as_uint(float f) {
    unsigned b;
    std::memcpy(&b, &f, 4);
    return b;
}
static inline int __clzll(long long v) { return v ? __builtin_clzll((unsigned long long)v) : 64; }

#include "../paper_2508_07424_gb300/csrc/pff_fixed.cuh"

typedef std::complex<long double> cl;
static const long double kTau = 6.28318530717958647692528676655900577L;

static std::vector<pff::fxw> twiddles(int L, bool from_double) {
    std::vector<pff::fxw> w(L);
    for (int m = 0; m < L; ++m) {
        w[m] = pff::fx_twiddle_host(m, L);
        if (!from_double) continue;
        auto put = [](double v, int &h, int &l) {  // as the device does it from sincospi
            v *= 1073741824.0;
            h = (int)std::rint(v);
            l = (int)std::fmin(std::fmax(std::rint((v - (double)h) * 4294967296.0), -2147483647.0), 2147483647.0);
        };
        put((double)cosl(-kTau * m / L), w[m].rh, w[m].rl);
        put((double)sinl(-kTau * m / L), w[m].ih, w[m].il);
    }
    return w;
}
// One line: the scale, the conversions and the passes of the kernels, thread after thread.
static void line(double *x, int lgL, const std::vector<pff::fxw> &tw) {
    const int L = 1 << lgL, lgT = lgL > 3 ? lgL - 3 : 0, T = 1 << lgT;
    unsigned mx = 0;
    for (int i = 0; i < 2 * L; ++i) mx = std::max(mx, pff::fx_hi_abs(x[i]));
    const unsigned base = pff::fx_norm_base(mx);
    float norm = 0.f;
    for (int i = 0; i < L; ++i) norm += pff::fx_norm_term(pff::fx_hi_abs(x[2 * i]), pff::fx_hi_abs(x[2 * i + 1]), base);
    const int k = pff::fx_scale(mx, norm);
    std::vector<pff::fx2> a(std::max(L, 8)), b(a);
    for (int i = 0; i < L; ++i) a[i] = pff::fx2{pff::fx_in(x[2 * i], k), pff::fx_in(x[2 * i + 1], k)};
    bool last = false;
    for (int lgN = 0; !last; lgN += 3) {
        for (int t = 0; t < T; ++t) {
            pff::fx2 v[8];
            for (int m = 0; m < 8; ++m) v[m] = a[t + (m << lgT)];
            last = pff::fx_pass(v, lgL, lgT, lgN, t, tw.data());
            for (int m = 0; m < 8; ++m) b[last ? t + (m << lgT) : pff::fx_pass_out(lgN, t) + (m << lgN)] = v[m];
        }
        a = b;
    }
    for (int i = 0; i < L; ++i) {
        x[2 * i] = pff::fx_out(a[i].x, 1086 - k);
        x[2 * i + 1] = pff::fx_out(a[i].y, 1086 - k);
    }
}
// The same in FP64: a radix-4 self-sorting network with fused multiply-adds.
static void line_fp64(double *xy, int lgL, const std::vector<std::complex<double>> &w) {
    typedef std::complex<double> cd;
    const int L = 1 << lgL;
    std::vector<cd> x(L), y(L);
    for (int i = 0; i < L; ++i) x[i] = cd(xy[2 * i], xy[2 * i + 1]);
    auto mul = [](cd a, cd b) {
        return cd(std::fma(a.real(), b.real(), -(a.imag() * b.imag())), std::fma(a.real(), b.imag(), a.imag() * b.real()));
    };
    int Ns = 1;
    if (lgL & 1) {
        for (int j = 0; j < L / 2; ++j) {
            y[2 * j] = x[j] + x[j + L / 2];
            y[2 * j + 1] = x[j] - x[j + L / 2];
        }
        x.swap(y);
        Ns = 2;
    }
    for (; Ns < L; Ns *= 4) {
        for (int t = 0; t < L / 4; ++t) {
            const int k = t & (Ns - 1), s = k * (L / (4 * Ns)), o = 4 * (t - k) + k;
            const cd a0 = x[t], a1 = mul(x[t + L / 4], w[s]), a2 = mul(x[t + L / 2], w[2 * s]), a3 = mul(x[t + 3 * L / 4], w[3 * s]);
            const cd p = a0 + a2, m = a0 - a2, q = a1 + a3, r = cd(a1.imag() - a3.imag(), a3.real() - a1.real());
            y[o] = p + q;
            y[o + Ns] = m + r;
            y[o + 2 * Ns] = p - q;
            y[o + 3 * Ns] = m - r;
        }
        x.swap(y);
    }
    for (int i = 0; i < L; ++i) {
        xy[2 * i] = x[i].real();
        xy[2 * i + 1] = x[i].imag();
    }
}
static void exact(std::vector<cl> &a) {
    const size_t n = a.size();
    if (n == 1) return;
    std::vector<cl> e(n / 2), o(n / 2);
    for (size_t i = 0; i < n / 2; ++i) {
        e[i] = a[2 * i];
        o[i] = a[2 * i + 1];
    }
    exact(e);
    exact(o);
    for (size_t k = 0; k < n / 2; ++k) {
        const cl t = cl(cosl(-kTau * k / n), sinl(-kTau * k / n)) * o[k];
        a[k] = e[k] + t;
        a[k + n / 2] = e[k] - t;
    }
}

extern "C" {

void sum_from_fixed(int n, const long long *x, const long long *y, int k, double *out) {
    for (int i = 0; i < n; ++i) out[i] = pff::fx_out_sum(x[i], y[i], 1086 - k);
}

void to_fixed(int n, const double *d, int k, long long *out) {
    for (int i = 0; i < n; ++i) out[i] = pff::fx_in(d[i], k);
}

// Relative errors in the 2-norm of the transforms of n lines of 2^lgL complex points: fixed point with
// twiddles of full length, with twiddles rounded to doubles, and FP64.
void line_errors(int n, int lgL, const double *x, double *fixed, double *fixed_noalloc, double *fp64) {
    const int L = 1 << lgL;
    const std::vector<pff::fxw> tw = twiddles(L, false), twd = twiddles(L, true);
    std::vector<std::complex<double>> w(L);
    for (int m = 0; m < L; ++m) w[m] = std::complex<double>((double)cosl(-kTau * m / L), (double)sinl(-kTau * m / L));
    for (int i = 0; i < n; ++i, x += 2 * L) {
        std::vector<cl> r(L);
        for (int j = 0; j < L; ++j) r[j] = cl(x[2 * j], x[2 * j + 1]);
        exact(r);
        auto err = [&](const std::vector<double> &y) {
            long double d = 0, s = 0;
            for (int j = 0; j < L; ++j) {
                d += std::norm(r[j] - cl(y[2 * j], y[2 * j + 1]));
                s += std::norm(r[j]);
            }
            return (double)sqrtl(d / s);
        };
        std::vector<double> y(x, x + 2 * L);
        line(y.data(), lgL, tw);
        fixed[i] = err(y);
        y.assign(x, x + 2 * L);
        line(y.data(), lgL, twd);
        fixed_noalloc[i] = err(y);
        y.assign(x, x + 2 * L);
        line_fp64(y.data(), lgL, w);
        fp64[i] = err(y);
    }
}

// The largest error, in units, of a w (w as it is held, in exact arithmetic) over every twiddle w of L points and
// directions of a that make the partial sums largest, at the largest |a| that the scale allows.
double multiply_error(int L) {
    const long double lim = 0.91L * 9223372036854775808.0L;
    double worst = 0.0;
    for (int m = 0; m < L; ++m) {
        const pff::fxw w = pff::fx_twiddle_host(m, L);
        const cl lo(w.rl, w.il);
        const __int128 re = ((__int128)w.rh << 32) + w.rl, im = ((__int128)w.ih << 32) + w.il;  // units of 2^-62
        for (int d = 0; d < 16; ++d) {
            const long double ph = kTau * d / 16;
            cl u(cosl(ph), sinl(ph));
            if (d & 1) u = std::abs(lo) > 0 ? std::conj(lo) / std::abs(lo) * (d & 2 ? 1.0L : -1.0L) : u;
            long long ax = llrintl(lim * u.real()), ay = llrintl(lim * u.imag());
            if (d & 4) ax = (ax & ~0xffffffffll) + (w.rh < 0 ? -0x80000000ll : 0x7fffffffll);  // largest low words
            if (d & 4) ay = (ay & ~0xffffffffll) + (w.ih > 0 ? -0x80000000ll : 0x7fffffffll);
            const pff::fx2 p = pff::cmul(pff::fx2{ax, ay}, w);
            const __int128 ex = ((__int128)p.x << 62) - (ax * re - ay * im), ey = ((__int128)p.y << 62) - (ax * im + ay * re);
            worst = std::max(worst, (double)std::max(ex < 0 ? -ex : ex, ey < 0 ? -ey : ey) / 4611686018427387904.0);
        }
    }
    return worst;
}

}  // extern "C"
