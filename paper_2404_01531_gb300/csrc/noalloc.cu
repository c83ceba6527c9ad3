// FD-subcell right-hand side without any device allocation.
//
// Who needs this: callers that cannot call cudaMalloc -- a host application
// that hands the library memory from its own pool and forbids allocations
// behind its back, or a latency-critical path where a first-touch allocation
// would stall.  ffe_create allocates everything a context needs, so those
// callers cannot use ffe_rhs; this entry point computes the FD right-hand side
// of caller-built extended blocks from caller-owned inputs and outputs, and
// keeps its intermediate data (the current J~ at every extended cell and the
// face fluxes) in one file-scope device array of fixed size,
// FFE_NOALLOC_SCRATCH_DOUBLES doubles (8 MiB).  Every GPU that loads the
// library holds that array until the process exits.
//
// Unlike the context path, the current J~ of every ghost cell is computed here
// from that cell's state: a context gives the ghosts across a DG neighbour's
// face that neighbour's nodal current instead (evaluated like its state), so
// the two agree on ghosts from FD neighbours and boundary states only.
#include <cmath>
#include <cstdio>
#include <mutex>

#include "ffe_internal.h"
#include "fd_common.cuh"
#include "physics.cuh"

namespace {

using namespace ffe;

constexpr long long kScratchDoubles = 1LL << 20;   // FFE_NOALLOC_SCRATCH_DOUBLES
constexpr int kMaxDevices = 64;

static __device__ __align__(256) double g_scratch[kScratchDoubles];

std::mutex g_mu;
double* g_scratch_ptr[kMaxDevices] = {};

struct NA {
    int n, nc, ne;
    int64_t ext, nface;         // doubles per element block: extended cells, faces of one direction
    double eta, eps, sc[3];     // sc[k] = (2/h_k) (nc/2)
    int corr;
    const double* Uext;         // [9][n][ext]
    double* J;                  // scratch [3][n][ext]
    double* F;                  // scratch [3][9][n][nface]
    double* out;                // [9][n][nc^3]
};

__global__ void k_na_current(NA a) {
    const int64_t total = (int64_t)a.n * a.ext;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        double u[NV], jd[3], jf[3];
        for (int v = 0; v < NV; ++v) u[v] = a.Uext[(int64_t)v * total + q];
        current_flat(u, a.eta, jd, jf);
        for (int k = 0; k < 3; ++k) a.J[(int64_t)k * total + q] = jf[k];
    }
}

// One thread per (element, direction, flux pair, line of cells), as k_fd_flux of the
// context path does (fd_common.cuh).  Single-warp CTAs: a call holds at most 19
// elements at P = 5, 1078 warps, and the FP64 pipe wants them spread evenly over
// the SMs.  19 elements: 0.49 -> 0.16 ms for the three kernels, against a thread
// per face with four divisions per value, and 0.091 ms with indicators and weights in
// integers.
__global__ void __launch_bounds__(32) k_na_flux(NA a) {
    const int nc = a.nc, nl = nc * nc, per = 3 * FLUX_PAIRS * nl;
    const int64_t cells = (int64_t)a.n * a.ext;
    for (int t = blockIdx.x * 32 + threadIdx.x; t < a.n * per; t += gridDim.x * 32) {
        const int w = t / per, r = t % per, line = r % nl, kp = r / nl;
        const int k = kp / FLUX_PAIRS, pr = kp % FLUX_PAIRS;
        int qa, qb;
        bool neg;
        flux_pair(k, pr, qa, qb, neg);
        int64_t stride;
        const int64_t base = w * a.ext + line_start(k, line % nc, line / nc, nc, stride);
        const double* pa = a.Uext + qa * cells + base;
        const double* pb = (qb < NV ? a.Uext + qb * cells : a.J + (qb - NV) * cells) + base;
        const unsigned long long sb = neg ? 0x8000000000000000ULL : 0ULL;
        double* fa = a.F + (((int64_t)k * NV + qa) * a.n + w) * a.nface + line;
        double* fb = pr < 4 ? a.F + (((int64_t)k * NV + qb) * a.n + w) * a.nface + line : nullptr;
        recon_lines<Weno5zLine>(pa, pb, stride, sb, nc, a.eps,
                                [&](int m, double La, double Ra, double Sa, double Lb, double Rb, double Sb) {
                                    double Fa, Fb;
                                    rusanov_pair(La, Ra, Sa, Lb, Rb, Sb, a.corr, Fa, Fb);
                                    fa[m * nl] = Fa;
                                    if (fb) fb[m * nl] = __longlong_as_double((long long)(fbits(Fb) ^ sb));
                                });
    }
}

__global__ void k_na_update(NA a) {
    const int nc = a.nc, ne = a.ne, ncell = nc * nc * nc;
    const int64_t total = (int64_t)a.n * ncell, cells = (int64_t)a.n * a.ext;
    for (int64_t q = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x) {
        const int w = (int)(q / ncell), c = (int)(q % ncell);
        const int cc[3] = {c % nc, (c / nc) % nc, c / (nc * nc)};
        const int64_t o = (int64_t)w * a.ext + (cc[0] + GH) + (int64_t)ne * ((cc[1] + GH) + (int64_t)ne * (cc[2] + GH));
        double u[NV], jd[3], jf[3], du[NV];
        for (int v = 0; v < NV; ++v) u[v] = a.Uext[(int64_t)v * cells + o];
        current_flat(u, a.eta, jd, jf);
        du[0] = -jd[0]; du[1] = -jd[1]; du[2] = -jd[2];
        du[3] = du[4] = du[5] = 0.0;
        du[6] = u[8];
        du[7] = du[8] = 0.0;
        for (int k = 0; k < 3; ++k) {
            const int t1 = k == 0 ? 1 : 0, t2 = k == 2 ? 1 : 2;
            const int f0 = face_index(nc, cc[k], cc[t1], cc[t2]), f1 = f0 + nc * nc;
            for (int v = 0; v < NV; ++v) {
                const double* fl = a.F + (((int64_t)k * NV + v) * a.n + w) * a.nface;
                du[v] = fma(-a.sc[k], fl[f1] - fl[f0], du[v]);
            }
        }
        for (int v = 0; v < NV; ++v) a.out[(int64_t)v * total + q] = du[v];
    }
}

}  // namespace

namespace ffe {
void set_last_error(const char* msg);
}

extern "C" ffe_status ffe_fd_rhs_noalloc(int P, int n_elem, const double* h_host, double eta, double weno_eps,
                                         int fd_corrector, const double* Uext_dev, double* dUdt_dev,
                                         void* cuda_stream) try {
    char msg[256];
    if (P < 3 || P > 6 || n_elem < 0 || !h_host || (n_elem > 0 && (!Uext_dev || !dUdt_dev))) {
        ffe::set_last_error("ffe_fd_rhs_noalloc: need 3 <= P <= 6, n_elem >= 0, h and buffers non-null");
        return FFE_EINVAL;
    }
    for (int k = 0; k < 3; ++k)
        if (!(h_host[k] > 0.0) || !std::isfinite(h_host[k])) {
            ffe::set_last_error("ffe_fd_rhs_noalloc: element widths must be positive and finite");
            return FFE_EINVAL;
        }
    if (!(eta >= 0.0) || !std::isfinite(eta) || !(weno_eps > 0.0) || !std::isfinite(weno_eps)) {
        ffe::set_last_error("ffe_fd_rhs_noalloc: need finite eta >= 0 and weno_eps > 0");
        return FFE_EINVAL;
    }
    const int nc = 2 * P + 1, ne = nc + 2 * GH;
    const long long per_elem = 3LL * ne * ne * ne + 3LL * NV * (nc + 1) * nc * nc;
    const long long cap = kScratchDoubles / per_elem;
    if (n_elem > cap) {
        snprintf(msg, sizeof msg,
                 "ffe_fd_rhs_noalloc: %d elements need %lld scratch doubles; the fixed scratch holds %lld "
                 "(at most %lld elements of order %d per call)",
                 n_elem, per_elem * n_elem, kScratchDoubles, cap, P);
        ffe::set_last_error(msg);
        return FFE_EINVAL;
    }
    if (n_elem == 0) return FFE_OK;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) {
        snprintf(msg, sizeof msg, "ffe_fd_rhs_noalloc: cudaGetDevice: %s", cudaGetErrorString(e));
        ffe::set_last_error(msg);
        return FFE_ECUDA;
    }
    if (dev < 0 || dev >= kMaxDevices) {
        snprintf(msg, sizeof msg, "ffe_fd_rhs_noalloc: device %d is beyond the %d devices this entry point serves",
                 dev, kMaxDevices);
        ffe::set_last_error(msg);
        return FFE_EINVAL;
    }
    double* scratch = nullptr;
    {
        // first call on this device: resolve the device address of the static array
        std::lock_guard<std::mutex> lk(g_mu);
        if (!g_scratch_ptr[dev]) {
            void* p = nullptr;
            e = cudaGetSymbolAddress(&p, g_scratch);
            if (e != cudaSuccess) {
                snprintf(msg, sizeof msg, "ffe_fd_rhs_noalloc: cudaGetSymbolAddress: %s", cudaGetErrorString(e));
                ffe::set_last_error(msg);
                return FFE_ECUDA;
            }
            g_scratch_ptr[dev] = (double*)p;
        }
        scratch = g_scratch_ptr[dev];
    }
    NA a;
    a.n = n_elem;
    a.nc = nc;
    a.ne = ne;
    a.ext = (int64_t)ne * ne * ne;
    a.nface = (int64_t)(nc + 1) * nc * nc;
    a.eta = eta;
    a.eps = weno_eps;
    for (int k = 0; k < 3; ++k) a.sc[k] = (2.0 / h_host[k]) * (0.5 * nc);
    a.corr = fd_corrector;
    a.Uext = Uext_dev;
    a.J = scratch;                                   // every entry written before it is read
    a.F = scratch + 3LL * n_elem * a.ext;            // likewise: nothing needs clearing
    a.out = dUdt_dev;
    cudaStream_t st = (cudaStream_t)cuda_stream;
    int nsm = 0;
    if (cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || nsm < 1) nsm = 1;
    k_na_current<<<nsm * 4, 256, 0, st>>>(a);
    k_na_flux<<<nsm * 16, 32, 0, st>>>(a);
    k_na_update<<<nsm * 4, 256, 0, st>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        snprintf(msg, sizeof msg, "ffe_fd_rhs_noalloc: launch: %s", cudaGetErrorString(e));
        ffe::set_last_error(msg);
        return FFE_ECUDA;
    }
    return FFE_OK;
} catch (...) {
    // a host exception (the mutex, an allocation inside the runtime) must not
    // cross the C ABI
    ffe::set_last_error("ffe_fd_rhs_noalloc: host resources exhausted");
    return FFE_ENOMEM;
}
