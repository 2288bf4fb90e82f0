// Allocation-free evaluation of the dissipation functional D(phi) and crack surface Gamma(phi).
//
// Some callers cannot allocate device memory at the moment they need this value: code running
// inside a host framework that owns the whole device memory through its own pool, code that
// must not trigger the implicit device synchronisation of cudaMalloc/cudaFree in a latency-
// critical loop, or embedded callers with a fixed memory budget reserved up front. For them this
// file provides rve_dissipation_noalloc: the caller passes device inputs and a device output,
// and every intermediate (half spectra, reduction partials, solver scalars, FFT twiddles) lives
// in one file-scope __device__ array of fixed size that each GPU loading the library holds
// until the process exits.
//
// One launch sets up the call's tables; the computation is the same three fused passes the engine uses for D and Gamma:
// the forward r2c FFT of phi, the spectral gradient i xi~ phi^ (frequency tables built in the
// scratch array), and the inverse c2r FFT with
// the reduction of sum Gc (phi^2/(2l) + l/2 grad phi . A grad phi).
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>

#include "../../include/pff_rve.h"
#include "pff_common.cuh"
#include "pff_functors.cuh"
#include "pff_kernels.cuh"

using namespace pff;

namespace pffnoalloc {

// 8 MiB of scratch: enough for 2D grids up to 512 x 512 and 3D grids up to 32^3, or any other
// shape whose layout (scalars, partial sums, twiddles, half spectra; computed per call) fits.
constexpr size_t kScratchBytes = 8u << 20;
static __device__ __align__(256) unsigned char g_scratch[kScratchBytes];

constexpr int kMaxDevices = 64;
static void *g_scratch_addr[kMaxDevices] = {nullptr};

static size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

struct Layout {
    size_t scal, partials, tw, xi, spec, total;
};

static int cw_of(int L) {
    const int TL = L / 4;
    int cw = 256 / (TL > 0 ? TL : 1);
    if (cw > 16) cw = 16;
    if (cw < 2) cw = 2;
    return cw;
}

// Set-up of a call in one launch (latency is all there is to it: 8 separate launches and clears took
// half of the call's 67 us at 128^2): the solver scalars (the reduction counter must start at zero; state
// left by an earlier call is not trusted), the twiddles of the three axes in the fixed-point form of the
// FP64 transforms, and the frequencies xi~ = 2 pi k / n (FFT order, Nyquist set to zero; the x axis covers
// the padded half-spectrum columns, whose padding gets zero). The padding columns of the spectra are
// not cleared: every column is transformed by itself and the inverse x pass reads none of them.
__global__ void k_setup(Scal *sc, fxw *tw, double *xi, int nx, int ny, int nz, int Px) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0) *sc = Scal{};
    const int nt = nx + ny + nz;
    if (i < nt) {
        const int L = i < nx ? nx : (i < nx + ny ? ny : nz), m = i < nx ? i : (i < nx + ny ? i - nx : i - nx - ny);
        double s, c;
        sincospi(-2.0 * (double)m / (double)L, &s, &c);
        auto put = [](double v, int &h, int &l) {
            v *= 1073741824.0;
            h = (int)rint(v);
            l = (int)fmin(fmax(rint((v - (double)h) * 4294967296.0), -2147483647.0), 2147483647.0);
        };
        fxw w;
        put(c, w.rh, w.rl);
        put(s, w.ih, w.il);
        tw[i] = w;
        return;
    }
    i -= nt;
    if (i >= Px + ny + nz) return;
    const bool x = i < Px;
    const int n = x ? nx : (i < Px + ny ? ny : nz), k = x ? i : (i < Px + ny ? i - Px : i - Px - ny);
    double v = 0.0;
    if (k < (x ? n / 2 + 1 : n) && 2 * k != n) {
        const int kk = k <= n / 2 ? k : k - n;
        v = 6.283185307179586476925286766559 * (double)kk / (double)n;
    }
    xi[i] = v;
}

// Epilogue of the last pass: the dissipation density of Eq. (CrackLenght_ani) summed with and
// without Gc, as the engine's, but with the grain ids checked against n_grains before they index
// the caller's tables. The ids come from caller memory that this entry point cannot validate on
// the host, so an id outside [0, n_grains) reads no table entry and turns both sums into NaN.
template <int D>
struct EpiDissChecked {
    static constexpr int NR = 2;
    bool skip_if_done;
    const double *phi;
    const double *GcTab, *Atab;
    const int *gid;
    int n_grains;
    double ell;
    double *result;  // D and Gamma, the caller's
    __device__ void apply(long long v, const double *gr, double *acc) const {
        const int gg = gid[v];
        if (gg < 0 || gg >= n_grains) {
            const double nan = __longlong_as_double(0x7ff8000000000000LL);
            acc[0] += nan;
            acc[1] += nan;
            return;
        }
        const double *A = Atab + (size_t)gg * 6;
        double q;
        if constexpr (D == 2) {
            q = gr[0] * (A[0] * gr[0] + A[2] * gr[1]) + gr[1] * (A[2] * gr[0] + A[1] * gr[1]);
        } else {
            q = gr[0] * (A[0] * gr[0] + A[5] * gr[1] + A[4] * gr[2]) +
                gr[1] * (A[5] * gr[0] + A[1] * gr[1] + A[3] * gr[2]) +
                gr[2] * (A[4] * gr[0] + A[3] * gr[1] + A[2] * gr[2]);
        }
        const double p = phi[v];
        const double dens = p * p / (2.0 * ell) + 0.5 * ell * q;
        acc[0] += GcTab[gg] * dens;
        acc[1] += dens;
    }
    struct Fin {
        double *result;
        __device__ void operator()(const double *t) const { result[0] = t[0]; result[1] = t[1]; }
    };
    __device__ Fin fin(Scal *) const { return Fin{result}; }
};

}  // namespace pffnoalloc

using namespace pffnoalloc;

extern "C" int rve_dissipation_noalloc(int dim, const int n[3], double ell, int n_grains, const int32_t *grain_id,
                                       const double *Gc, const double *A, const double *phi, double *out,
                                       void *stream) {
    if (!n || !grain_id || !Gc || !A || !phi || !out || n_grains <= 0 || !(ell > 0)) return RVE_EINVAL;
    if (dim != 2 && dim != 3) return RVE_EINVAL;
    auto pow2 = [](int v) { return v >= 4 && v <= 1024 && (v & (v - 1)) == 0; };
    const int nx = n[0], ny = n[1], nz = dim == 2 ? 1 : n[2];
    // 3D plates one voxel thick (nz = 1) are accepted as by rve_create: no z transform
    if (!pow2(nx) || !pow2(ny) || (dim == 2 ? n[2] != 1 : (nz != 1 && !pow2(nz)))) return RVE_EINVAL;

    Geom g{};
    g.d = dim; g.ns = dim == 2 ? 3 : 6;
    g.nx = nx; g.ny = ny; g.nz = nz;
    auto lg = [](int v) { int l = 0; while ((1 << l) < v) ++l; return l; };
    g.lx = lg(nx); g.ly = lg(ny); g.lz = lg(nz);
    const int cwy = cw_of(ny), cwz = nz > 1 ? cw_of(nz) : 2, cw = cwy > cwz ? cwy : cwz;
    g.Px = ((nx / 2 + 1 + cw - 1) / cw) * cw;
    g.N = (long long)nx * ny * nz;
    g.Nh = (long long)g.Px * ny * nz;
    g.invN = 1.0 / (double)g.N;

    // launch shape of the x passes (same rule as the engine); grids too small for one warp of row
    // pairs of nx / 4 columns are refused, as by rve_create
    const int TL = nx / 4;
    const long long pairs = (long long)ny * nz / 2;
    if ((long long)TL * (128 / TL < 1 ? 1 : (128 / TL < pairs ? 128 / TL : pairs)) < 32) return RVE_EINVAL;
    const XShape xs = x_shape<double>(nx, pairs);

    // scratch layout; reject grids whose requirement exceeds the static array
    Layout lay;
    lay.scal = 0;
    lay.partials = align256(sizeof(Scal));
    lay.tw = lay.partials + align256(sizeof(double) * 2 * (size_t)xs.blocks);
    lay.xi = lay.tw + align256(sizeof(double2) * (size_t)(nx + ny + nz));
    lay.spec = lay.xi + align256(sizeof(double) * (size_t)(g.Px + ny + nz));
    lay.total = lay.spec + align256(sizeof(double2) * (size_t)dim * (size_t)g.Nh);
    if (lay.total > kScratchBytes) {
        std::fprintf(stderr,
                     "rve_dissipation_noalloc: grid %dx%dx%d needs %zu bytes of scratch, more than the fixed %zu\n",
                     nx, ny, nz, lay.total, kScratchBytes);
        return RVE_EINVAL;
    }

    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return RVE_ECUDA;
    if (!g_scratch_addr[dev]) {
        // one-time set-up on this device (the device is current): the host-side name of
        // g_scratch is not a device address, so look the address up and keep it.
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_scratch) != cudaSuccess || !p) return RVE_ECUDA;
        g_scratch_addr[dev] = p;
    }
    unsigned char *base = (unsigned char *)g_scratch_addr[dev];
    Scal *sc = (Scal *)(base + lay.scal);
    double *partials = (double *)(base + lay.partials);
    fxw *twx = (fxw *)(base + lay.tw);
    fxw *twy = twx + nx;
    fxw *twz = twy + ny;
    double *xix = (double *)(base + lay.xi);
    double *xiy = xix + g.Px;
    double *xiz = xiy + ny;
    const XiTab<double> xi{xix, xiy, xiz};
    double2 *spec = (double2 *)(base + lay.spec);
    cudaStream_t st = (cudaStream_t)stream;

    {
        const int n_el = (nx + ny + nz) + (g.Px + ny + nz);
        k_setup<<<(n_el + 127) / 128, 128, 0, st>>>(sc, twx, xix, nx, ny, nz, g.Px);
        if (cudaGetLastError() != cudaSuccess) return RVE_ECUDA;
    }
    auto launch = [&](auto kernel, dim3 grid, int threads, size_t sm, auto... args) -> cudaError_t {
        const cudaError_t e = smem_raise((const void *)kernel, sm);
        if (e != cudaSuccess) return e;
        kernel<<<grid, threads, sm, st>>>(args...);
        return cudaGetLastError();
    };
    auto axis_launch = [&](auto kernel, int ax, int NM, const auto &op, const fxw *tw) -> cudaError_t {
        const int L = ax == 1 ? ny : nz;
        const int CW = ax == 1 ? cwy : cwz;
        int threads;
        size_t sm;
        axis_shape<double>(L, NM, CW, threads, sm);
        return launch(kernel, dim3(g.Px / CW, ax == 1 ? nz : ny), threads, sm, g, ax, CW, (const double2 *)spec, spec, op, tw, sc);
    };
    // forward x pass of phi
    if (launch(k_x_fwd<double, 1, ProField<double>>, dim3(xs.blocks), xs.threads, x_smem<double>(nx, xs.RP, 1), g, xs.RP,
               ProField<double>{false, phi}, spec, (const fxw *)twx, partials, sc) != cudaSuccess)
        return RVE_ECUDA;
    const int32_t *gid = grain_id;
    if (dim == 2) {
        if (axis_launch(axis_kernel<double, 1, 2, AX_FWD_OP_INV, OpGrad<double2, 2>>(ny), 1, 2, OpGrad<double2, 2>{false, xi}, twy))
            return RVE_ECUDA;
        if (launch(k_x_inv<double, 2, EpiDissChecked<2>>, dim3(xs.blocks), xs.threads, x_smem<double>(nx, xs.RP, 2), g,
                   xs.RP, (const double2 *)spec, EpiDissChecked<2>{false, phi, Gc, A, gid, n_grains, ell, out},
                   (const fxw *)twx, partials, sc, (cudaGraphConditionalHandle)0) != cudaSuccess)
            return RVE_ECUDA;
    } else {
        if (nz == 1) {
            // plate: xi_z = 0, so the gradient is taken in the y pass, as in 2D
            if (axis_launch(axis_kernel<double, 1, 3, AX_FWD_OP_INV, OpGrad<double2, 3>>(ny), 1, 3, OpGrad<double2, 3>{false, xi},
                            twy))
                return RVE_ECUDA;
        } else {
            if (axis_launch(axis_kernel<double, 1, 1, AX_FWD, OpGrad<double2, 3>>(ny), 1, 1, OpGrad<double2, 3>{false, xi}, twy))
                return RVE_ECUDA;
            if (axis_launch(axis_kernel<double, 1, 3, AX_FWD_OP_INV, OpGrad<double2, 3>>(nz), 2, 3, OpGrad<double2, 3>{false, xi},
                            twz))
                return RVE_ECUDA;
            if (axis_launch(axis_kernel<double, 3, 3, AX_INV, OpGrad<double2, 3>>(ny), 1, 3, OpGrad<double2, 3>{false, xi}, twy))
                return RVE_ECUDA;
        }
        if (launch(k_x_inv<double, 3, EpiDissChecked<3>>, dim3(xs.blocks), xs.threads, x_smem<double>(nx, xs.RP, 3), g,
                   xs.RP, (const double2 *)spec, EpiDissChecked<3>{false, phi, Gc, A, gid, n_grains, ell, out},
                   (const fxw *)twx, partials, sc, (cudaGraphConditionalHandle)0) != cudaSuccess)
            return RVE_ECUDA;
    }
    return RVE_OK;
}
