// Fused spectral passes of the FFT phase-field-fracture solver (sm_103a).
//
// A spectral operator  v -> F^-1[ Op(xi) F[ pro(v) ] ]  is applied as
//   k_x_fwd   : per pair of x-rows, evaluate the prologue (e.g. the stress C_phi : p of a CG
//               direction) for NC components, pack the two real rows as one complex line, FFT
//               along x, split into the two half spectra, store [c][z][y][kx];
//   k_axis    : per tile of CW adjacent kx columns, FFT along y (2D) or y then z (3D), apply the
//               per-frequency operator (projection, gradient, divergence, preconditioner), inverse
//               FFT, store;
//   k_x_inv   : rebuild the packed line from two half spectra, inverse FFT along x, evaluate the
//               epilogue (CG vector update, residual, dot products) with a deterministic
//               reduction finalised by the last CTA.
//   k_x_mid   : inverse x pass, a pointwise map (damage flux Gc l A grad phi), forward x pass.
// All kernels of one solve read their scalars (alpha, beta, done flag) from a device Scal block,
// so a whole CG iteration is launched without host synchronisation.
#pragma once

#include <algorithm>
#include <type_traits>

#include "pff_common.cuh"
#include "pff_fixed.cuh"
#include "pff_host.cuh"

namespace pff {

enum { AX_FWD = 0, AX_INV = 1, AX_FWD_OP_INV = 2 };

// Epilogues that define FACC = true also provide apply_f(v, val, float *acc), used on the FP32
// path to accumulate a thread's partial sums in FP32.
template <class E, class = void> struct facc_of : std::false_type {};
template <class E> struct facc_of<E, std::void_t<decltype(E::FACC)>> : std::integral_constant<bool, E::FACC> {};

// ---- transform of lines ----------------------------------------------------------------------------
// FP64 lines are transformed in 64-bit fixed point (fx_lines; pff_fixed.cuh), FP32 lines in float2:
// shared-memory Stockham (fft_lines) in the x passes, warps in registers (warp_lines) in the column passes.
// The FP32 forms were measured against fx_lines instantiated for float2: 128^3 column pass 48 against
// 58 us, 1024^2 column pass 25 against 42 us, x passes equal or slower.
// `line_c` is the type that the butterflies work on, `line_w` that of the twiddles.
template <typename T> struct line_of;
template <> struct line_of<float> { typedef float2 c; typedef float2 w; };
template <> struct line_of<double> { typedef fx2 c; typedef fxw w; };
template <typename T> using line_c = typename line_of<T>::c;
template <typename T> using line_w = typename line_of<T>::w;

__device__ __forceinline__ int ilog2(int v) { return 31 - __clz(v); }

// Twiddle table of a line of L points (host side), in the form that the butterflies use.
static inline void axis_twiddle(int m, int L, fxw &w) { w = fx_twiddle_host(m, L); }
static inline void axis_twiddle(int m, int L, float2 &w) {
    const long double a = -2.0L * 3.14159265358979323846264338327950288L * (long double)m / (long double)L;
    w = make_float2((float)cosl(a), (float)sinl(a));
}

// Shared-memory index of point p of a line. FP64 lines skip one element after every eight, so that
// the strided writes of the first exchange of fx_lines (8 t + q) hit distinct banks.
template <typename T> __host__ __device__ __forceinline__ constexpr int lpos(int p) {
    return sizeof(T) == 8 ? p + (p >> 3) : p;
}
// Elements of shared memory that an FP64 line of L points needs, a multiple of 16.
__host__ __device__ constexpr int fx_line_room(int L) { return (L + L / 8 + 15) / 16 * 16; }
// Stride of the lines of an x pass.
template <typename T> __host__ __device__ constexpr int x_line_stride(int L) {
    return sizeof(T) == 8 ? fx_line_room(L) + 4 : L;
}


// e0 of a line that holds an infinity or a NaN, or whose norm leaves the FP64 range.
constexpr int kBadLine = 1 << 20;

// Transform FP64 lines held in dynamic shared memory: line i < nlines starts at element
// (i / NL NG + i mod NL) LS (groups of NG lines of which the first NL are transformed), point p at
// lpos<double>(p), natural order in and out. A line of L points is worked on by T = L / 8 threads with 8
// points each: radix-8 self-sorting passes and a last one of radix 2 or 4, each reading
// x[t + m T] and exchanging through the line itself. 8 points per thread rather than 16: the grids
// of this library have few lines per SM, so the work has to be spread over threads (512^2: 771 column
// lines of 64 threads on 152 SMs). The inverse is the forward network on swapped real and
// imaginary parts. Converts to fixed point on the way in; on the way out back to FP64 scaled by
// 2^-osh, or leaves integers with their e0 (fx_out) in the int array at ke0 when ke0 >= 0.
// A function of its own, called once or twice per kernel, for the build time and because one
// instance serves every length. Every thread of the CTA calls it; blockDim is a multiple of T and of 32.
// SOME: there may be warps without a line (x passes: three lines of 512 points for 256 threads). They
// leave, and a line that spans several warps synchronises its own T threads by a named barrier (512^2
// damage passes 18.7 / 30.7 -> 14.8 / 26.5 us). The column passes have a line for every thread; there
// the CTA barrier is the faster one (36.6 against 38.2 us).
template <bool SOME> __device__ __forceinline__ void line_sync(int lgT, int group) {
    if (lgT <= 5) __syncwarp();
    else if constexpr (SOME) asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(1 << lgT) : "memory");
    else __syncthreads();
}
template <bool SOME>
static __device__ __noinline__ void fx_lines(int nlines, int LS, int lgL, const fxw *__restrict__ tw, bool inv, int osh,
                                             int ke0, int NL, int NG) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ unsigned wmx[32];
    __shared__ float wnorm[32];
    const int lgT = lgL > 3 ? lgL - 3 : 0, TH = 1 << lgT;
    const int t = threadIdx.x & (TH - 1), gpc = blockDim.x >> lgT, nv = lgL < 3 ? 1 << lgL : 8;
    const bool wide = TH > 32;  // a line spans several warps
    const int group = threadIdx.x >> lgT;  // at most 8 groups of more than a warp (512 threads)
    for (int first = 0; first < nlines; first += gpc) {
        if (SOME && first + ((int)(threadIdx.x & ~31u) >> lgT) >= nlines) break;  // no line in this warp
        const int line = first + group;
        const bool valid = line < nlines;
        const int at = NL == NG ? line : line / NL * NG + line % NL;
        double2 *p = reinterpret_cast<double2 *>(smem_raw) + (valid ? at * LS : 0);
        fx2 *q = reinterpret_cast<fx2 *>(p);
        double2 d[8];
        fx2 v[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
            double2 z = make_double2(0.0, 0.0);
            if (valid && m < nv) z = p[lpos<double>(t + (m << lgT))];
            d[m] = inv ? make_double2(z.y, z.x) : z;
        }
        // scale of the line, from its largest value and a bound of its norm
        unsigned mx = 0;
#pragma unroll
        for (int m = 0; m < 8; ++m) mx = max(mx, max(fx_hi_abs(d[m].x), fx_hi_abs(d[m].y)));
        const int sw = wide ? 32 : TH;
        for (int o = sw >> 1; o; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const unsigned base = fx_norm_base(mx);
        float norm = 0.f;
#pragma unroll
        for (int m = 0; m < 8; ++m) norm += fx_norm_term(fx_hi_abs(d[m].x), fx_hi_abs(d[m].y), base);
        for (int o = sw >> 1; o; o >>= 1) norm += __shfl_xor_sync(0xffffffffu, norm, o);
        if (wide) {
            if ((threadIdx.x & 31) == 0) {
                wmx[threadIdx.x >> 5] = mx;
                wnorm[threadIdx.x >> 5] = norm;
            }
            line_sync<SOME>(lgT, group);
            const int w0 = group << (lgT - 5), nw = 1 << (lgT - 5);
            for (int w = 0; w < nw; ++w) mx = max(mx, wmx[w0 + w]);
            norm = 0.f;
            for (int w = 0; w < nw; ++w) {
                const int dE = (int)(mx >> 20) - (int)(wmx[w0 + w] >> 20);
                norm += dE < 126 ? wnorm[w0 + w] * __int_as_float((127 - dE) << 23) : 0.f;
            }
        }
        const int k = fx_scale(mx, norm);
        const int e0 = mx >= 0x7ff00000u || k <= -963 ? kBadLine : 1086 - k;
#pragma unroll
        for (int m = 0; m < 8; ++m) v[m] = fx2{fx_in(d[m].x, k), fx_in(d[m].y, k)};
        for (int lgN = 0; !fx_pass(v, lgL, lgT, lgN, t, tw); lgN += 3) {
            const int at8 = fx_pass_out(lgN, t);
            line_sync<SOME>(lgT, group);
            if (valid) {
#pragma unroll
                for (int r = 0; r < 8; ++r) q[lpos<double>(at8 + (r << lgN))] = v[r];
            }
            line_sync<SOME>(lgT, group);
#pragma unroll
            for (int m = 0; m < 8; ++m) v[m] = q[lpos<double>(t + (m << lgT))];
        }
        if (valid) {
            if (ke0 >= 0) {
#pragma unroll
                for (int m = 0; m < 8; ++m)
                    if (m < nv) q[lpos<double>(t + (m << lgT))] = v[m];
                if (t == 0) (reinterpret_cast<int *>(smem_raw) + ke0)[at] = e0;
            } else {
#pragma unroll
                for (int m = 0; m < 8; ++m) {
                    double x = fx_out(v[m].x, e0 - osh), y = fx_out(v[m].y, e0 - osh);
                    if (e0 == kBadLine) x = y = fx_nan();
                    if (m < nv) p[lpos<double>(t + (m << lgT))] = inv ? make_double2(y, x) : make_double2(x, y);
                }
            }
        }
    }
}

// ---- FP32 lines of the column passes, one lane group or warp per line, in registers ------------------
template <int R> struct log2_of { static constexpr int v = R == 1 ? 0 : 1 + log2_of<R / 2>::v; };
template <> struct log2_of<1> { static constexpr int v = 0; };

// Points per lane of the warp transform of a line of L points (S = L / R lanes, S <= 32), and
// whether the line takes the two-pass form (L >= 256, one line per warp) or the single-pass form
// (a lane group of S lanes per line). Up to 128 points, 16 per lane keep most butterflies in
// registers: a 128-point line has 3 lane stages instead of the 5 that 4 per lane would need.
__host__ __device__ constexpr int axis_points_per_lane(int L) {
    return L < 16 ? 4 : (L <= 128 ? 16 : (L == 256 ? 8 : (L == 512 ? 16 : 32)));
}
__host__ __device__ constexpr bool axis_two_pass(int L) { return L >= 256; }
__device__ __forceinline__ int brev_bits(int v, int bits) {
    return bits == 0 ? 0 : (int)(__brev((unsigned)v) >> (32 - bits));
}
// Frequency index held at storage position p of a line of L points after the forward transform.
// Single pass (wfft_fwd): p = l + S m holds brev_R(m) + R brev_S(l). Two-pass (wfft2_fwd, S = 32
// lanes in G = 32 / R groups): p = l + 32 c holds brev_R(l / G) + R brev_R(c) + R^2 brev_G(l mod G).
template <typename T> __device__ __forceinline__ int axis_freq(int p, int L) {
    if (sizeof(T) == 8) return p;  // FP64 lines are in natural order
    const int R = axis_points_per_lane(L);
    const int lgR = ilog2(R), lgS = ilog2(L) - lgR;
    if (!axis_two_pass(L)) {
        const int m = p >> lgS, l = p & ((1 << lgS) - 1);
        return brev_bits(m, lgR) + (brev_bits(l, lgS) << lgR);
    }
    const int lgG = 5 - lgR;
    const int lp = p & 31, c = p >> 5;
    const int j = lp >> lgG, gg = lp & ((1 << lgG) - 1);
    return brev_bits(j, lgR) + (brev_bits(c, lgR) << lgR) + (brev_bits(gg, lgG) << (2 * lgR));
}

__device__ __forceinline__ float2 shfl_xor_c(float2 v, int m) {
    return make_float2(__shfl_xor_sync(0xffffffffu, v.x, m), __shfl_xor_sync(0xffffffffu, v.y, m));
}
template <typename C> __device__ __forceinline__ C conj_c(C a) { a.y = -a.y; return a; }

// w_32^t = exp(-2 pi i t / 32), t < 32: the twiddles of the in-register stages (R <= 32), at
// offsets known at compile time, so they are read from the constant bank. Each translation unit
// that includes this header has its own copy; axis_twiddles_init() fills it on the current device.
static __constant__ float2 c_w32f[32];
template <typename C> __device__ __forceinline__ C w32(int t);
template <> __device__ __forceinline__ float2 w32<float2>(int t) { return c_w32f[t]; }

// d w_32^t and d conj(w_32^t) for a t known at compile time (the unrolled stages): t = 8 is -i,
// a swap and a sign change instead of a complex multiply.
template <typename C> __device__ __forceinline__ C mul_w32(const C &d, int t) {
    if (t == 8) { C r; r.x = d.y; r.y = -d.x; return r; }
    return cmul(d, w32<C>(t));
}
template <typename C> __device__ __forceinline__ C mul_w32c(const C &d, int t) {
    if (t == 8) { C r; r.x = -d.y; r.y = d.x; return r; }
    return cmul(d, conj_c(w32<C>(t)));
}

static inline cudaError_t axis_twiddles_init() {
    float2 f[32];
    for (int t = 0; t < 32; ++t) {
        const long double a = -2.0L * 3.14159265358979323846264338327950288L * (long double)t / 32.0L;
        f[t] = make_float2((float)cosl(a), (float)sinl(a));
    }
    return cudaMemcpyToSymbol(c_w32f, f, sizeof(f));
}

// Forward lane stage h over the R values of each lane: the lower lane of a pair keeps a + b, the
// upper one (a - b) w. Both are t w~ with t = o + sgn v (sgn = -1 on the upper lane) and w~ = 1 on
// the lower lane, so every lane runs the same instructions (no divergent halves). TW = false for
// h = 1, whose twiddle is w_L^0 = 1 on both lanes. tsh = log2(L / (2 h)) (the twiddle stride).
template <typename C, int R, bool TW>
__device__ __forceinline__ void lane_stage_fwd(C (&v)[R], int l, int h, int tsh, const C *__restrict__ tw) {
    typedef typename real_of<C>::type Rt;
    const bool upper = (l & h) != 0;
    const Rt sg = upper ? (Rt)-1 : (Rt)1;
    C w;
    if (TW) {
        w = tw[(l & (h - 1)) << tsh];
        if (!upper) { w.x = (Rt)1; w.y = (Rt)0; }
    }
#pragma unroll
    for (int m = 0; m < R; ++m) {
        const C o = shfl_xor_c(v[m], h);
        C t;
        t.x = fma(sg, v[m].x, o.x);
        t.y = fma(sg, v[m].y, o.y);
        v[m] = TW ? cmul(t, w) : t;
    }
}
// Inverse lane stage h: the upper lane sends u = conj(w) b', the lower one a'; the lower lane keeps
// a' + u, the upper one a' - u, i.e. o + sgn send with sgn = -1 on the upper lane.
template <typename C, int R, bool TW>
__device__ __forceinline__ void lane_stage_inv(C (&v)[R], int l, int h, int tsh, const C *__restrict__ tw) {
    typedef typename real_of<C>::type Rt;
    const bool upper = (l & h) != 0;
    const Rt sg = upper ? (Rt)-1 : (Rt)1;
    C w;
    if (TW) {
        w = conj_c(tw[(l & (h - 1)) << tsh]);
        if (!upper) { w.x = (Rt)1; w.y = (Rt)0; }
    }
#pragma unroll
    for (int m = 0; m < R; ++m) {
        const C send = TW ? cmul(v[m], w) : v[m];
        const C o = shfl_xor_c(send, h);
        v[m].x = fma(sg, send.x, o.x);
        v[m].y = fma(sg, send.y, o.y);
    }
}

// Forward transform of one line: v[m] = x[l + S m] on entry, v[m] = X[axis_freq(l + S m)] on
// exit (unnormalised, w_L = exp(-2 pi i / L), tw[j] = w_L^j). Every lane of the warp must call it.
template <typename C, int R>
__device__ __forceinline__ void wfft_fwd(C (&v)[R], int l, int S, int L, const C *__restrict__ tw) {
    constexpr int lgR = log2_of<R>::v;
#pragma unroll
    for (int h = R / 2; h >= 1; h >>= 1) {
#pragma unroll
        for (int b = 0; b < R; b += 2 * h) {
#pragma unroll
            for (int j = 0; j < h; ++j) {
                const C a = v[b + j], c = v[b + j + h];
                v[b + j] = cadd(a, c);
                const C d = csub(a, c);
                v[b + j + h] = j == 0 ? d : mul_w32(d, j * (16 / h));
            }
        }
    }
#pragma unroll
    for (int m = 1; m < R; ++m) {
        const int k1 = (int)(__brev((unsigned)m) >> (32 - lgR));
        v[m] = cmul(v[m], tw[(l * k1) & (L - 1)]);
    }
    const int lgL = ilog2(L);
    int lgh = ilog2(S) - 1;
    for (int h = S >> 1; h >= 2; h >>= 1, --lgh) lane_stage_fwd<C, R, true>(v, l, h, lgL - 1 - lgh, tw);
    if (S >= 2) lane_stage_fwd<C, R, false>(v, l, 1, 0, tw);
}

// Inverse of wfft_fwd up to the factor L: storage order in, natural order out (unnormalised
// inverse DFT). Every lane of the warp must call it.
template <typename C, int R>
__device__ __forceinline__ void wfft_inv(C (&v)[R], int l, int S, int L, const C *__restrict__ tw) {
    constexpr int lgR = log2_of<R>::v;
    const int lgL = ilog2(L);
    if (S >= 2) lane_stage_inv<C, R, false>(v, l, 1, 0, tw);
    int lgh = 1;
    for (int h = 2; h < S; h <<= 1, ++lgh) lane_stage_inv<C, R, true>(v, l, h, lgL - 1 - lgh, tw);
#pragma unroll
    for (int m = 1; m < R; ++m) {
        const int k1 = (int)(__brev((unsigned)m) >> (32 - lgR));
        v[m] = cmul(v[m], conj_c(tw[(l * k1) & (L - 1)]));
    }
#pragma unroll
    for (int h = 1; h < R; h <<= 1) {
#pragma unroll
        for (int b = 0; b < R; b += 2 * h) {
#pragma unroll
            for (int j = 0; j < h; ++j) {
                const C t = j == 0 ? v[b + j + h] : mul_w32c(v[b + j + h], j * (16 / h));
                const C a = v[b + j];
                v[b + j] = cadd(a, t);
                v[b + j + h] = csub(a, t);
            }
        }
    }
}

// In-register radix-2 stages over R values (compile-time twiddles w_{2h}^j = w_32^(16 j / h)).
template <typename C, int R> __device__ __forceinline__ void regs_dif(C (&v)[R]) {
#pragma unroll
    for (int h = R / 2; h >= 1; h >>= 1) {
#pragma unroll
        for (int b = 0; b < R; b += 2 * h) {
#pragma unroll
            for (int j = 0; j < h; ++j) {
                const C a = v[b + j], c = v[b + j + h];
                v[b + j] = cadd(a, c);
                const C d = csub(a, c);
                v[b + j + h] = j == 0 ? d : mul_w32(d, j * (16 / h));
            }
        }
    }
}
template <typename C, int R> __device__ __forceinline__ void regs_dit(C (&v)[R]) {
#pragma unroll
    for (int h = 1; h < R; h <<= 1) {
#pragma unroll
        for (int b = 0; b < R; b += 2 * h) {
#pragma unroll
            for (int j = 0; j < h; ++j) {
                const C t = j == 0 ? v[b + j + h] : mul_w32c(v[b + j + h], j * (16 / h));
                const C a = v[b + j];
                v[b + j] = cadd(a, t);
                v[b + j + h] = csub(a, t);
            }
        }
    }
}

// Two-pass warp transform of a line of L = 32 R points (R >= 8), one line per warp: the lane
// dimension (32 points) is split as 32 = G x R (G = 32 / R) so that most butterflies run in
// registers instead of across lanes. Pass A: lane l holds x[l + 32 m]; R-point DFT over m,
// twiddle w_L^(l k1). Transpose through the line's shared memory (rows of 32 + G elements, so
// that the gathers hit distinct banks): lane (j, g) = (l / G, l mod G) takes the R values of
// row j at columns g + G t. Pass B: R-point DFT over t, twiddle w_32^(g c), then log2 G stages
// across the G lanes of a group. The result is in the order of axis_freq; `line` must have room
// for L + 32 elements. Every lane of the warp must call it.
template <typename C, int R>
__device__ __forceinline__ void wfft2_fwd(C (&v)[R], C *line, int l, int L, const C *__restrict__ tw) {
    constexpr int G = 32 / R, lgR = log2_of<R>::v, rs = 32 + G;
    regs_dif<C, R>(v);
#pragma unroll
    for (int m = 1; m < R; ++m) {
        const int k1 = (int)(__brev((unsigned)m) >> (32 - lgR));
        v[m] = cmul(v[m], tw[(l * k1) & (L - 1)]);
    }
    __syncwarp();
#pragma unroll
    for (int m = 0; m < R; ++m) line[m * rs + l] = v[m];
    __syncwarp();
    const int j = l / G, gg = l & (G - 1);
#pragma unroll
    for (int t = 0; t < R; ++t) v[t] = line[j * rs + gg + G * t];
    regs_dif<C, R>(v);
    if (G > 1) {
#pragma unroll
        for (int c = 1; c < R; ++c) {
            const int cc = (int)(__brev((unsigned)c) >> (32 - lgR));
            v[c] = cmul(v[c], tw[(gg * cc * R) & (L - 1)]);
        }
        // lanes of a group differ in their low log2 G bits (gg), so the stages index by l
#pragma unroll
        for (int h = G >> 1; h >= 2; h >>= 1) lane_stage_fwd<C, R, true>(v, l, h, ilog2(L) - 1 - ilog2(h), tw);
        lane_stage_fwd<C, R, false>(v, l, 1, 0, tw);
    }
}
template <typename C, int R>
__device__ __forceinline__ void wfft2_inv(C (&v)[R], C *line, int l, int L, const C *__restrict__ tw) {
    constexpr int G = 32 / R, lgR = log2_of<R>::v, rs = 32 + G;
    const int j = l / G, gg = l & (G - 1);
    if (G > 1) {
        lane_stage_inv<C, R, false>(v, l, 1, 0, tw);
#pragma unroll
        for (int h = 2; h < G; h <<= 1) lane_stage_inv<C, R, true>(v, l, h, ilog2(L) - 1 - ilog2(h), tw);
#pragma unroll
        for (int c = 1; c < R; ++c) {
            const int cc = (int)(__brev((unsigned)c) >> (32 - lgR));
            v[c] = cmul(v[c], conj_c(tw[(gg * cc * R) & (L - 1)]));
        }
    }
    regs_dit<C, R>(v);
    __syncwarp();
#pragma unroll
    for (int t = 0; t < R; ++t) line[j * rs + gg + G * t] = v[t];
    __syncwarp();
#pragma unroll
    for (int m = 0; m < R; ++m) v[m] = line[m * rs + l];
#pragma unroll
    for (int m = 1; m < R; ++m) {
        const int k1 = (int)(__brev((unsigned)m) >> (32 - lgR));
        v[m] = cmul(v[m], conj_c(tw[(l * k1) & (L - 1)]));
    }
    regs_dit<C, R>(v);
}

// Transform the lines [0, nlines) of the tile, one line per lane group of S lanes, looping over
// groups of lines when there are more lines than warps. INV selects the inverse network.
// Lines of a tile of CW columns start 16 / CW elements apart modulo the 16 elements of a shared-memory
// phase. The 16 / S lines that a half-warp works on together are taken dist = S CW / 16 apart, so that
// they start S elements apart and their accesses fall on distinct banks (adjacent lines overlapped:
// two-way conflicts on 128 points; 128^3 projection pass 45.2 -> 43.3 us).
template <typename C, int R, bool TWO, bool INV>
__device__ __forceinline__ void warp_lines(C *s, int nlines, int LS, int L, int lgCW, const C *__restrict__ tw) {
    const int lgS = ilog2(L) - log2_of<R>::v, S = 1 << lgS;
    const int lpw = 32 >> lgS;  // lines per warp
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
    const int l = lane & (S - 1);
    for (int grp = warp; grp * lpw < nlines; grp += nwarps) {  // uniform across the warp
        int line = grp * lpw + (lane >> lgS);
        const bool valid = line < nlines;
        const int lgd = lgS + lgCW - 4;  // log2 dist
        if (!TWO && lgS < 4 && lgd > 0) {
            const int r = line & ((1 << lgCW) - 1);
            line = line - r + ((r & ((1 << (4 - lgS)) - 1)) << lgd) + (r >> (4 - lgS));
        }
        C *p = s + (size_t)(valid ? line : 0) * LS;
        C v[R];
#pragma unroll
        for (int m = 0; m < R; ++m) v[m] = p[l + S * m];
        if constexpr (TWO) {  // S = 32: one line per warp, every lane of it valid or not
            if constexpr (INV) wfft2_inv<C, R>(v, p, l, L, tw);
            else wfft2_fwd<C, R>(v, p, l, L, tw);
        } else {
            if constexpr (INV) wfft_inv<C, R>(v, l, S, L, tw);
            else wfft_fwd<C, R>(v, l, S, L, tw);
        }
        __syncwarp();
        if (valid) {
#pragma unroll
            for (int m = 0; m < R; ++m) p[l + S * m] = v[m];
        }
        __syncwarp();
    }
}

// Stride of the lines of a column tile of CW columns. Consecutive threads read CW columns of a row, so
// lines that differ by one start (128 bytes / CW) apart modulo the 128-byte bank period and the
// transposing accesses of one phase hit distinct banks; FP32 lines of the two-pass form have room for
// their transposition.
template <typename T> __host__ __device__ constexpr int axis_line_stride(int L, int CW) {
    return sizeof(T) == 8 ? fx_line_room(L) + 8 / CW : L + 16 / CW + (axis_two_pass(L) ? 32 : 0);
}

// Threads per CTA at most: 512, or 256 where an FP32 lane holds 16 or more values (more registers each).
template <typename T> __host__ __device__ constexpr int axis_max_threads(int R) {
    return sizeof(T) == 4 && R >= 16 ? 256 : 512;
}
// Dispatch key of the column-pass instances: points per lane and form.
enum { AXK_4 = 0, AXK_16 = 1, AXK_8T = 2, AXK_16T = 3, AXK_32T = 4 };
__host__ __device__ constexpr int axis_form(int L) {
    return axis_two_pass(L) ? (L == 256 ? AXK_8T : (L == 512 ? AXK_16T : AXK_32T)) : (L < 16 ? AXK_4 : AXK_16);
}
template <int K> struct axis_form_of {
    static constexpr int R = K == AXK_4 ? 4 : (K == AXK_8T ? 8 : (K == AXK_32T ? 32 : 16));
    static constexpr bool TWO = K >= AXK_8T;
};
// FP32 lines of 16 to 128 points: 80 registers, 3 CTAs of 256 threads per SM (128^3 projection pass 49.4 -> 45.1 us).
// The bound spills 40 to 68 bytes in every operator, which pays where there are more than two CTAs per SM and costs
// where there are not. FP32R solves with the bound against without: 128^3 3 % (equilibrium) and 6 % (damage) faster,
// 128x128x64 3.5 %, 64^3 1 and 2.6 %, 64x64x16 1.5 and 2.6 %; 128^2 and 64^2 1 to 1.7 % slower, 128x64x1 1 and 3 %;
// 256^2 and more in 2D equal (those lines take the two-pass form). A second instance for small grids would double
// the compilation of the column passes for those few percent.
template <typename T, int K> __host__ __device__ constexpr int axis_min_blocks() { return sizeof(T) == 4 && K == AXK_16 ? 3 : 0; }

// ---- x passes ------------------------------------------------------------------------------------
// A CTA owns RP pairs of x-rows; each pair is one packed complex line Z = a + i b per component.
// Pointwise work runs over the RP nx columns of the pairs with every thread, at most 256. The FP32
// passes are bound by the latency of their loads, so the registers of the forward and inverse passes are
// bounded for occupancy: 64 up to three components (the 512 CTAs of 256 threads of a 1024^2 pass fit the 608
// slots in one wave instead of two, 43.6 -> 31.8 us per CG forward launch), 72 with six (the 2048 CTAs of
// 128 threads of a 128^3 pass in two waves instead of three: CG forward 154 -> 131 us, inverse
// 66 -> 59 us; 85 registers gain no wave and measured 5-10 % slower). FP64: two CTAs per SM. The rule goes by the
// number of components; with it and the fixed-point residual passes the FP32R equilibrium is 1.02 to 1.40 times
// as fast on all of 17 grids (2D 64^2 to 1024^2 and 1024x64, 3D 16^3 to 128^3, plates).
template <typename T, int NC> __host__ __device__ constexpr int x_max_regs() { return sizeof(T) == 8 ? 128 : (NC <= 3 ? 64 : 72); }
template <typename T> __host__ __device__ constexpr int x_mid_threads() { return sizeof(T) == 8 ? 256 : 512; }

// Launch shape. FP32: 128 threads of 4 columns. FP64: 256 columns, a thread per column up to 256 (half the
// threads left 7 warps per SM and two rounds of lines: 64x64x32 CG passes 35.1 / 28.3 -> 31.1 / 23.4 us); on
// small grids an FP64 pass is bound by the FP64 work of the few SMs that hold a CTA, so there a CTA
// takes as few row pairs as give a whole warp, until there are two CTAs per SM (64^2 with the
// split: 4 -> 32 CTAs, 66 -> 24 us per forward pass; FP32 passes gained nothing from it).
constexpr int kSmCount = 152;  // GB300
struct XShape { int threads, blocks, RP; };
template <typename T> inline XShape x_shape(int nx, long long pairs) {
    constexpr bool fx = sizeof(T) == 8;
    const int unit = fx ? nx : nx / 4;  // FP64: columns, FP32: threads of a row pair
    const int full = fx ? 256 : 128;
    int RP = full / unit > 1 ? full / unit : 1;
    while (RP > 1 && (RP > pairs || (fx && pairs / RP < 2 * kSmCount && RP / 2 * unit >= 32))) RP >>= 1;
    XShape x;
    x.RP = RP;
    x.blocks = (int)(pairs / RP);
    x.threads = !fx ? RP * unit : std::max(32, std::min(256, RP * nx));
    return x;
}
// Dynamic shared memory: the lines, then (FP64) one exponent per line.
template <typename T> inline size_t x_smem(int nx, int RP, int NC) {
    return (size_t)RP * NC * (x_line_stride<T>(nx) * 2 * sizeof(T) + (sizeof(T) == 8 ? 4 : 0));
}
template <typename T> __device__ __forceinline__ int x_ke0(int nlines, int LS) {
    return sizeof(T) == 8 ? nlines * LS * 4 : -1;
}
// Transform the first NL of the NG lines of each of the RP row pairs of the CTA.
template <typename T, int NL, int NG>
__device__ __forceinline__ void x_lines(typename cplx_of<T>::type *s, const Geom &g, int RP, int LS,
                                        const line_w<T> *__restrict__ tw, bool inv, int ke0) {
    if constexpr (sizeof(T) == 8) fx_lines<true>(RP * NL, LS, g.lx, tw, inv, inv ? g.lx + g.ly + g.lz : 0, ke0, NL, NG);
    else fft_lines<float2, NL>(s, g.nx, g.lx, NL, NG, 1, tw, inv);
}

// Call f(row pair, x, voxel of the first row) for the columns of the CTA's row pairs that this thread
// handles: FP32, four columns nx / 4 apart, unrolled so that their loads are in flight together; FP64, a
// strided loop.
template <typename T, class F>
__device__ __forceinline__ void x_columns(const Geom &g, long long pair0, int RP, const F &f) {
    if constexpr (sizeof(T) == 4) {
        const int TL = g.nx >> 2, rp = threadIdx.x / TL, t = threadIdx.x - rp * TL;
        const long long row0 = 2 * (pair0 + rp) * g.nx;
#pragma unroll
        for (int q = 0; q < 4; ++q) f(rp, t + q * TL, row0 + t + q * TL);
    } else {
#pragma unroll 2
        for (int i = threadIdx.x; i < RP * g.nx; i += blockDim.x) {
            const int rp = i >> g.lx, x = i & (g.nx - 1);
            f(rp, x, 2 * (pair0 + rp) * g.nx + x);
        }
    }
}

// Store the two half spectra of each packed line of the CTA, Xa = (Z(k) + conj Z(-k)) / 2,
// Xb = (Z(k) - conj Z(-k)) / 2i. FP64 lines are still integers here: the sums are exact and the halving
// goes into the exponent of the conversion.
template <typename T, int NC, int NG>
__device__ __forceinline__ void store_split(const Geom &g, typename cplx_of<T>::type *__restrict__ spec, long long pair0,
                                            int RP, const typename cplx_of<T>::type *s, int LS, const int *ke) {
    typedef typename cplx_of<T>::type C;
    const int nx = g.nx, lh = g.lx - 1, h = 1 << lh;
    if constexpr (sizeof(T) == 4) {
        const int TL = nx >> 2, rp = threadIdx.x / TL, t = threadIdx.x - rp * TL;
        for (int k = t; k <= h; k += TL) {
            const int km = (nx - k) & (nx - 1);
#pragma unroll
            for (int c = 0; c < NC; ++c) {
                const C *line = s + (rp * NG + c) * LS;
                const C Z = line[k], Zm = line[km];
                C *dst = spec + (size_t)c * g.Nh + 2 * (pair0 + rp) * g.Px + k;
                dst[0] = make_float2(0.5f * (Z.x + Zm.x), 0.5f * (Z.y - Zm.y));
                dst[g.Px] = make_float2(0.5f * (Z.y + Zm.y), -0.5f * (Z.x - Zm.x));
            }
        }
    } else {
        for (int i = threadIdx.x; i < RP * NC * h; i += blockDim.x) {
            const int ln = i >> lh, k0 = i & (h - 1);
            const int rp = ln / NC, c = ln - rp * NC, at = rp * NG + c;
            const fx2 *line = reinterpret_cast<const fx2 *>(s + at * LS);
            C *dst = spec + (size_t)c * g.Nh + 2 * (pair0 + rp) * g.Px;
            const int e0 = ke[at];
            for (int k = k0; k <= h; k += h) {  // k0 = 0 also stores the Nyquist column
                const fx2 Z = line[lpos<T>(k)], Zm = line[lpos<T>((nx - k) & (nx - 1))];
                C Xa = make_double2(fx_out_sum(Z.x, Zm.x, e0 - 1), fx_out_sum(Z.y, -Zm.y, e0 - 1));
                C Xb = make_double2(fx_out_sum(Z.y, Zm.y, e0 - 1), fx_out_sum(Zm.x, -Z.x, e0 - 1));
                if (e0 == kBadLine) Xa.x = Xa.y = Xb.x = Xb.y = fx_nan();
                dst[k] = Xa;
                dst[g.Px + k] = Xb;
                if (k0 != 0) break;
            }
        }
    }
}
// Load the packed lines Z = Xa + i Xb of the CTA from the half spectra, into storage order.
template <typename T, int NC>
__device__ __forceinline__ void load_packed(const Geom &g, const typename cplx_of<T>::type *__restrict__ spec,
                                            long long pair0, int RP, typename cplx_of<T>::type *s, int LS) {
    typedef typename cplx_of<T>::type C;
    const int nx = g.nx, lh = g.lx - 1, h = 1 << lh;
    if constexpr (sizeof(T) == 4) {
        // k = t, t + nx / 4 and (t = 0 only) nx / 2: a fixed trip count lets the loads be issued together
        const int TL = nx >> 2, rp = threadIdx.x / TL, t = threadIdx.x - rp * TL;
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            C *line = s + (rp * NC + c) * nx;
            const C *src = spec + (size_t)c * g.Nh + 2 * (pair0 + rp) * g.Px;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const int k = t + q * TL;
                if (k > h) break;
                C Xa = src[k], Xb = src[g.Px + k];
                if (k == 0 || k == h) { Xa.y = 0; Xb.y = 0; }
                line[k] = make_float2(Xa.x - Xb.y, Xa.y + Xb.x);
                if (k > 0 && k < h) line[nx - k] = make_float2(Xa.x + Xb.y, -Xa.y + Xb.x);
            }
        }
    } else {
#pragma unroll 4
        for (int i = threadIdx.x; i < RP * NC * h; i += blockDim.x) {
            const int ln = i >> lh, k = i & (h - 1);
            const int rp = ln / NC, c = ln - rp * NC;
            C *line = s + ln * LS;
            const C *src = spec + (size_t)c * g.Nh + 2 * (pair0 + rp) * g.Px;
            const C Xa = src[k], Xb = src[g.Px + k];
            C Z = make_double2(Xa.x - Xb.y, Xa.y + Xb.x), Zc = make_double2(Xa.x + Xb.y, Xb.x - Xa.y);
            if (k == 0) {  // the columns k = 0 and nx / 2 are real
                Z = make_double2(Xa.x, Xb.x);
                Zc = make_double2(src[h].x, src[g.Px + h].x);
            }
            line[lpos<T>(k)] = Z;
            line[lpos<T>(k == 0 ? h : nx - k)] = Zc;
        }
    }
}

// ---- x-axis forward (r2c) pass ------------------------------------------------------------------
template <typename T, int NC, class Pro>
__device__ __forceinline__ void x_fwd_body(const Geom &g, int RP, const Pro &pro,
                                           typename cplx_of<T>::type *__restrict__ spec,
                                           const line_w<T> *__restrict__ tw, double *partials, Scal *sc) {
    typedef typename cplx_of<T>::type C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *s = reinterpret_cast<C *>(smem_raw);
    if (pro.skip_if_done && sc->done) return;
    const int nx = g.nx, LS = x_line_stride<T>(nx);
    const long long pair0 = (long long)blockIdx.x * RP;
    double acc[Pro::NR > 0 ? Pro::NR : 1];
#pragma unroll
    for (int k = 0; k < (Pro::NR > 0 ? Pro::NR : 1); ++k) acc[k] = 0.0;
    x_columns<T>(g, pair0, RP, [&](int rp, int x, long long v) {
        T va[NC], vb[NC];
        pro.eval(v, va, acc);
        pro.eval(v + nx, vb, acc);
        C *line = s + rp * NC * LS + lpos<T>(x);
#pragma unroll
        for (int c = 0; c < NC; ++c) line[c * LS] = cmk<C>(va[c], vb[c]);
    });
    __syncthreads();
    const int ke0 = x_ke0<T>(RP * NC, LS);
    x_lines<T, NC, NC>(s, g, RP, LS, tw, false, ke0);
    __syncthreads();
    store_split<T, NC, NC>(g, spec, pair0, RP, s, LS, reinterpret_cast<int *>(smem_raw) + ke0);
    if constexpr (Pro::NR > 0) reduce_finalize<Pro::NR>(acc, partials, sc, pro.fin(sc));
}

template <typename T, int NC, class Pro>
__global__ void __maxnreg__((x_max_regs<T, NC>()))
    k_x_fwd(Geom g, int RP, Pro pro, typename cplx_of<T>::type *__restrict__ spec, const line_w<T> *__restrict__ tw,
            double *partials, Scal *sc) {
    x_fwd_body<T, NC>(g, RP, pro, spec, tw, partials, sc);
}

// ---- batched launches: several RVEs of one grid in one launch -----------------------------------
// blockIdx.z selects the RVE; each carries its own functor, spectral buffer, reduction partials
// and scalar block (the per-RVE reductions see gridDim.x * gridDim.y blocks, as unbatched).
constexpr int kMaxBatch = 16;
template <class F> struct SlotArg {
    F f;
    void *spec;
    double *partials;
    Scal *sc;
};
template <class F> struct SlotArgs {
    SlotArg<F> a[kMaxBatch];
};

template <typename T, int NC, class Pro>
__global__ void __maxnreg__((x_max_regs<T, NC>()))
    k_x_fwd_b(Geom g, int RP, SlotArgs<Pro> args, const line_w<T> *__restrict__ tw) {
    typedef typename cplx_of<T>::type C;
    const SlotArg<Pro> &a = args.a[blockIdx.z];
    x_fwd_body<T, NC>(g, RP, a.f, (C *)a.spec, tw, a.partials, a.sc);
}

// Condition of the while node whose body a kernel ends: set by the thread that has just updated the
// solve's scalars (or by a kernel that skips because the solve is done), so that an iteration needs no
// kernel of its own for it. 0: not in such a graph.
__device__ __forceinline__ void loop_cond(cudaGraphConditionalHandle cond, const Scal *sc) {
    if (cond) cudaGraphSetConditional(cond, sc->done ? 0u : 1u);
}
template <class F> struct FinCond {  // the finalizer of a reduction, then the loop condition
    F fin;
    cudaGraphConditionalHandle cond;
    const Scal *sc;
    __device__ void operator()(const double *t) const {
        fin(t);
        loop_cond(cond, sc);
    }
};

// ---- x-axis inverse (c2r) pass with a fused epilogue --------------------------------------------
template <typename T, int NC, class Epi>
__device__ __forceinline__ void x_inv_body(const Geom &g, int RP, const typename cplx_of<T>::type *__restrict__ spec,
                                           const Epi &epi, const line_w<T> *__restrict__ tw, double *partials,
                                           Scal *sc, cudaGraphConditionalHandle cond) {
    typedef typename cplx_of<T>::type C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *s = reinterpret_cast<C *>(smem_raw);
    if (epi.skip_if_done && sc->done) {
        if (blockIdx.x == 0 && threadIdx.x == 0) loop_cond(cond, sc);
        return;
    }
    const int nx = g.nx, LS = x_line_stride<T>(nx);
    const long long pair0 = (long long)blockIdx.x * RP;
    load_packed<T, NC>(g, spec, pair0, RP, s, LS);
    __syncthreads();
    // the scale 1/N is a power of two: in the exponent of the FP64 conversion, a factor in FP32
    x_lines<T, NC, NC>(s, g, RP, LS, tw, true, -1);
    __syncthreads();
    constexpr int NR1 = Epi::NR > 0 ? Epi::NR : 1;
    double acc[NR1];
#pragma unroll
    for (int k = 0; k < NR1; ++k) acc[k] = 0.0;
    const T sN = sizeof(T) == 8 ? (T)1 : (T)g.invN;
    // FP32 path with an epilogue that supports it: the thread's voxels are summed in FP32 and
    // converted once (FP64 issues at 1/64 of the FP32 rate on this part); the reduction across
    // threads and CTAs stays FP64
    constexpr bool F32ACC = sizeof(T) == 4 && facc_of<Epi>::value;
    float accf[NR1];
#pragma unroll
    for (int k = 0; k < NR1; ++k) accf[k] = 0.f;
    x_columns<T>(g, pair0, RP, [&](int rp, int x, long long v) {
        const C *line = s + rp * NC * LS + lpos<T>(x);
        T va[NC], vb[NC];
#pragma unroll
        for (int c = 0; c < NC; ++c) {
            const C z = line[c * LS];
            va[c] = sizeof(T) == 8 ? z.x : z.x * sN;
            vb[c] = sizeof(T) == 8 ? z.y : z.y * sN;
        }
        if constexpr (F32ACC) {
            epi.apply_f(v, va, accf);
            epi.apply_f(v + nx, vb, accf);
        } else {
            epi.apply(v, va, acc);
            epi.apply(v + nx, vb, acc);
        }
    });
    if constexpr (F32ACC) {
#pragma unroll
        for (int k = 0; k < NR1; ++k) acc[k] = (double)accf[k];
    }
    if constexpr (Epi::NR > 0)
        reduce_finalize<Epi::NR>(acc, partials, sc, FinCond<typename Epi::Fin>{epi.fin(sc), cond, sc});
}

template <typename T, int NC, class Epi>
__global__ void __maxnreg__((x_max_regs<T, NC>()))
    k_x_inv(Geom g, int RP, const typename cplx_of<T>::type *__restrict__ spec, Epi epi,
            const line_w<T> *__restrict__ tw, double *partials, Scal *sc, cudaGraphConditionalHandle cond) {
    x_inv_body<T, NC>(g, RP, spec, epi, tw, partials, sc, cond);
}

template <typename T, int NC, class Epi>
__global__ void __maxnreg__((x_max_regs<T, NC>()))
    k_x_inv_b(Geom g, int RP, SlotArgs<Epi> args, const line_w<T> *__restrict__ tw) {
    typedef typename cplx_of<T>::type C;
    const SlotArg<Epi> &a = args.a[blockIdx.z];
    x_inv_body<T, NC>(g, RP, (const C *)a.spec, a.f, tw, a.partials, a.sc, 0);
}

// ---- x-axis inverse, pointwise map, x-axis forward ----------------------------------------------
// Inverse x pass of NCI components, mid.apply(v, in[NCI], out[NCO]) per voxel (NCO <= NCI), forward
// x pass of the NCO outputs.
template <typename T, int NCI, int NCO, class Mid>
__device__ __forceinline__ void x_mid_body(const Geom &g, int RP, typename cplx_of<T>::type *__restrict__ spec,
                                           const Mid &mid, const line_w<T> *__restrict__ tw, Scal *sc) {
    typedef typename cplx_of<T>::type C;
    static_assert(NCO <= NCI, "k_x_mid maps NCI components to at most NCI");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *s = reinterpret_cast<C *>(smem_raw);
    if (mid.skip_if_done && sc->done) return;
    const int nx = g.nx, LS = x_line_stride<T>(nx);
    const long long pair0 = (long long)blockIdx.x * RP;
    load_packed<T, NCI>(g, spec, pair0, RP, s, LS);
    __syncthreads();
    x_lines<T, NCI, NCI>(s, g, RP, LS, tw, true, -1);
    __syncthreads();
    const T sN = sizeof(T) == 8 ? (T)1 : (T)g.invN;
    x_columns<T>(g, pair0, RP, [&](int rp, int x, long long v) {
        C *line = s + rp * NCI * LS + lpos<T>(x);
        T va[NCI], vb[NCI], oa[NCO], ob[NCO];
#pragma unroll
        for (int c = 0; c < NCI; ++c) {
            const C z = line[c * LS];
            va[c] = sizeof(T) == 8 ? z.x : z.x * sN;
            vb[c] = sizeof(T) == 8 ? z.y : z.y * sN;
        }
        mid.apply(v, va, oa);
        mid.apply(v + nx, vb, ob);
#pragma unroll
        for (int c = 0; c < NCO; ++c) line[c * LS] = cmk<C>(oa[c], ob[c]);
    });
    __syncthreads();
    const int ke0 = x_ke0<T>(RP * NCI, LS);
    x_lines<T, NCO, NCI>(s, g, RP, LS, tw, false, ke0);
    __syncthreads();
    store_split<T, NCO, NCI>(g, spec, pair0, RP, s, LS, reinterpret_cast<int *>(smem_raw) + ke0);
}

template <typename T, int NCI, int NCO, class Mid>
__global__ void __launch_bounds__(x_mid_threads<T>(), sizeof(T) == 8 ? 2 : 0)
    k_x_mid(Geom g, int RP, typename cplx_of<T>::type *__restrict__ spec, Mid mid, const line_w<T> *__restrict__ tw,
            Scal *sc) {
    x_mid_body<T, NCI, NCO>(g, RP, spec, mid, tw, sc);
}

template <typename T, int NCI, int NCO, class Mid>
__global__ void __launch_bounds__(x_mid_threads<T>(), sizeof(T) == 8 ? 2 : 0)
    k_x_mid_b(Geom g, int RP, SlotArgs<Mid> args, const line_w<T> *__restrict__ tw) {
    typedef typename cplx_of<T>::type C;
    const SlotArg<Mid> &a = args.a[blockIdx.z];
    x_mid_body<T, NCI, NCO>(g, RP, (C *)a.spec, a.f, tw, a.sc);
}

// ---- y / z axis pass ----------------------------------------------------------------------------
// axis = 1 (y) or 2 (z). A CTA owns CW adjacent kx columns of one plane (z for axis y, y for
// axis z) and all L points along the axis, for every component. MODE: AX_FWD, AX_INV or
// AX_FWD_OP_INV (forward, the per-frequency operator mapping NCI -> NCO components, inverse).
// The tile is read from global memory with consecutive threads on consecutive kx (coalesced runs
// of CW complex values per row) into shared memory, one line of L points per (component, column).
template <typename T, int K, bool INV>
__device__ __forceinline__ void axis_lines(typename cplx_of<T>::type *s, int nlines, int LS, int lgL, int lgCW,
                                           const line_w<T> *__restrict__ tw) {
    if constexpr (sizeof(T) == 8) fx_lines<false>(nlines, LS, lgL, tw, INV, 0, -1, 1, 1);
    else warp_lines<float2, axis_form_of<K>::R, axis_form_of<K>::TWO, INV>(s, nlines, LS, 1 << lgL, lgCW, tw);
}

template <typename T, int NCI, int NCO, int MODE, int K, class Op>
__device__ __forceinline__ void axis_body(const Geom &g, int axis, int CW,
                                          const typename cplx_of<T>::type *__restrict__ spec_in,
                                          typename cplx_of<T>::type *spec_out, const Op &op,
                                          const line_w<T> *__restrict__ tw, Scal *sc) {
    typedef typename cplx_of<T>::type C;
    constexpr int NOUT = (MODE == AX_FWD_OP_INV) ? NCO : NCI;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C *s = reinterpret_cast<C *>(smem_raw);
    if (op.skip_if_done && sc->done) return;
    const int L = axis == 1 ? g.ny : g.nz;
    const int lgL = axis == 1 ? g.ly : g.lz;
    const int lgCW = ilog2(CW);
    const int LS = axis_line_stride<T>(L, CW);
    const int kx0 = blockIdx.x * CW;
    const int other = blockIdx.y;
    // element offsets in 32 bits: every spectrum of a valid configuration (at most 2^24 voxels,
    // x padded to Px <= max(16, nx/2 + 16)) has fewer than 2^29 elements over all its components
    const unsigned Nh = (unsigned)g.Nh;
    const unsigned lstride = axis == 1 ? (unsigned)g.Px : (unsigned)g.Px * g.ny;
    const unsigned base = (axis == 1 ? (unsigned)other * g.ny * g.Px : (unsigned)other * g.Px) + kx0;
    const int nth = blockDim.x;
    const int npt = L * CW;  // points of one component in the tile
    // 1. coalesced load: i = (c, pos, cc), cc fastest. Each thread issues UB loads before it
    //    stores any of them, so that many loads are in flight. The tile belongs to this CTA alone
    //    and is read before any of it is written back, so the read-only path is safe in place.
    //    (Asynchronous 8-byte copies straight to shared memory measured 1.3-2x slower.)
    constexpr int UB = 8;
    for (int i0 = threadIdx.x; i0 < NCI * npt; i0 += nth * UB) {
        C tmp[UB];
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int i = i0 + u * nth;
            if (i < NCI * npt) {
                const int c = i >> (lgL + lgCW);
                const int rem = i & (npt - 1);
                const int pos = rem >> lgCW, cc = rem & (CW - 1);
                tmp[u] = __ldg(spec_in + (c * Nh + base + pos * lstride + cc));
            }
        }
#pragma unroll
        for (int u = 0; u < UB; ++u) {
            const int i = i0 + u * nth;
            if (i < NCI * npt) {
                const int c = i >> (lgL + lgCW);
                const int rem = i & (npt - 1);
                const int pos = rem >> lgCW, cc = rem & (CW - 1);
                s[((c << lgCW) + cc) * LS + lpos<T>(pos)] = tmp[u];
            }
        }
    }
    __syncthreads();
    // 2. transforms (and the operator between them)
    axis_lines<T, K, MODE == AX_INV>(s, NCI * CW, LS, lgL, lgCW, tw);
    if constexpr (MODE == AX_FWD_OP_INV) {
        __syncthreads();
        for (int i = threadIdx.x; i < npt; i += nth) {
            const int cc = i >> lgL, p = i & (L - 1);
            const int kk = axis_freq<T>(p, L);
            const int kx = kx0 + cc;
            const int ky = axis == 1 ? kk : axis_freq<T>(other, g.ny);
            const int kz = axis == 1 ? (g.nz > 1 ? other : 0) : kk;
            C in[NCI], out[NCO];
#pragma unroll
            for (int c = 0; c < NCI; ++c) in[c] = s[((c << lgCW) + cc) * LS + lpos<T>(p)];
            op.apply(g, kx, ky, kz, in, out);
#pragma unroll
            for (int c = 0; c < NCO; ++c) s[((c << lgCW) + cc) * LS + lpos<T>(p)] = out[c];
        }
        __syncthreads();
        axis_lines<T, K, true>(s, NCO * CW, LS, lgL, lgCW, tw);
    }
    __syncthreads();
    // 3. coalesced store
    for (int i = threadIdx.x; i < NOUT * npt; i += nth) {
        const int c = i >> (lgL + lgCW);
        const int rem = i & (npt - 1);
        const int pos = rem >> lgCW, cc = rem & (CW - 1);
        spec_out[c * Nh + base + pos * lstride + cc] = s[((c << lgCW) + cc) * LS + lpos<T>(pos)];
    }
}

template <typename T, int NCI, int NCO, int MODE, int K, class Op>
__global__ void __launch_bounds__(axis_max_threads<T>(axis_form_of<K>::R), axis_min_blocks<T, K>())
    k_axis(Geom g, int axis, int CW, const typename cplx_of<T>::type *__restrict__ spec_in,
           typename cplx_of<T>::type *spec_out, Op op, const line_w<T> *__restrict__ tw, Scal *sc) {
    axis_body<T, NCI, NCO, MODE, K>(g, axis, CW, spec_in, spec_out, op, tw, sc);
}

template <typename T, int NCI, int NCO, int MODE, int K, class Op>
__global__ void __launch_bounds__(axis_max_threads<T>(axis_form_of<K>::R), axis_min_blocks<T, K>())
    k_axis_b(Geom g, int axis, int CW, SlotArgs<Op> args, const line_w<T> *__restrict__ tw) {
    typedef typename cplx_of<T>::type C;
    const SlotArg<Op> &a = args.a[blockIdx.z];
    axis_body<T, NCI, NCO, MODE, K>(g, axis, CW, (const C *)a.spec, (C *)a.spec, a.f, tw, a.sc);
}

// Launch shape of k_axis for an axis of L points, NM components and CW columns per CTA: the threads of
// every line (FP64: L / 8 per line, FP32: a lane group of S = L / R) up to 16 warps, which loop over the
// lines beyond, and the padded lines in dynamic shared memory.
template <typename T> inline void axis_shape(int L, int NM, int CW, int &threads, size_t &smem, int wcap = 16) {
    constexpr bool fx = sizeof(T) == 8;
    const int R = fx ? 8 : axis_points_per_lane(L), S = L > R ? L / R : 1;
    const long long lanes = (long long)NM * CW * S;
    int w = (int)std::min<long long>((lanes + 31) / 32, axis_max_threads<T>(R) / 32);
    w = std::max(1, std::min(w, std::max(1, wcap)));
    if (fx && S > 32) w = std::max(1, w / (S / 32)) * (S / 32);  // whole lines
    threads = 32 * w;
    smem = (size_t)NM * CW * (size_t)axis_line_stride<T>(L, CW) * 2 * sizeof(T);
}

template <typename T, class Op>
using axis_kernel_t = void (*)(Geom, int, int, const typename cplx_of<T>::type *__restrict__, typename cplx_of<T>::type *,
                               Op, const line_w<T> *__restrict__, Scal *);

// The instance of k_axis for the points per lane of an axis of L points.
template <typename T, int NCI, int NCO, int MODE, class Op> inline axis_kernel_t<T, Op> axis_kernel(int L) {
    if constexpr (sizeof(T) == 8) return k_axis<T, NCI, NCO, MODE, AXK_4, Op>;  // one instance for every length
    else switch (axis_form(L)) {
    case AXK_4: return k_axis<T, NCI, NCO, MODE, AXK_4, Op>;
    case AXK_16: return k_axis<T, NCI, NCO, MODE, AXK_16, Op>;
    case AXK_8T: return k_axis<T, NCI, NCO, MODE, AXK_8T, Op>;
    case AXK_16T: return k_axis<T, NCI, NCO, MODE, AXK_16T, Op>;
    default: return k_axis<T, NCI, NCO, MODE, AXK_32T, Op>;
    }
}

template <typename T, class Op>
using axis_kernel_b_t = void (*)(Geom, int, int, SlotArgs<Op>, const line_w<T> *__restrict__);
template <typename T, int NCI, int NCO, int MODE, class Op> inline axis_kernel_b_t<T, Op> axis_kernel_b(int L) {
    if constexpr (sizeof(T) == 8) return k_axis_b<T, NCI, NCO, MODE, AXK_4, Op>;  // one instance for every length
    else switch (axis_form(L)) {
    case AXK_4: return k_axis_b<T, NCI, NCO, MODE, AXK_4, Op>;
    case AXK_16: return k_axis_b<T, NCI, NCO, MODE, AXK_16, Op>;
    case AXK_8T: return k_axis_b<T, NCI, NCO, MODE, AXK_8T, Op>;
    case AXK_16T: return k_axis_b<T, NCI, NCO, MODE, AXK_16T, Op>;
    default: return k_axis_b<T, NCI, NCO, MODE, AXK_32T, Op>;
    }
}

// ---- pointwise kernel with deterministic reductions ---------------------------------------------
template <class F>
__global__ void __launch_bounds__(256) k_pointwise_b(long long N, SlotArgs<F> args) {
    const SlotArg<F> &a = args.a[blockIdx.z];
    const F &f = a.f;
    Scal *sc = a.sc;
    if (f.skip_if_done && sc->done) return;
    double acc[F::NR > 0 ? F::NR : 1];
#pragma unroll
    for (int k = 0; k < (F::NR > 0 ? F::NR : 1); ++k) acc[k] = 0.0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < N; v += stride) f.apply(v, acc);
    if constexpr (F::NR > 0) reduce_finalize<F::NR>(acc, a.partials, sc, f.fin(sc), F::MAXRED);
}

template <class F>
__global__ void __launch_bounds__(256) k_pointwise(long long N, F f, double *partials, Scal *sc,
                                                   cudaGraphConditionalHandle cond) {
    if (f.skip_if_done && sc->done) {
        if (blockIdx.x == 0 && threadIdx.x == 0) loop_cond(cond, sc);
        return;
    }
    double acc[F::NR > 0 ? F::NR : 1];
#pragma unroll
    for (int k = 0; k < (F::NR > 0 ? F::NR : 1); ++k) acc[k] = 0.0;
    const long long stride = (long long)gridDim.x * blockDim.x;
    for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < N; v += stride) f.apply(v, acc);
    if constexpr (F::NR > 0)
        reduce_finalize<F::NR>(acc, partials, sc, FinCond<typename F::Fin>{f.fin(sc), cond, sc}, F::MAXRED);
}

}  // namespace pff
