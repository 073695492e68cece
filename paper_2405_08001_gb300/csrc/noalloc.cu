// sim_pHp_noalloc: an allocation-free variant of the p^T H p reduction, for callers that cannot allocate device
// memory themselves (a host application that owns the whole device-memory budget through its own allocator, such
// as a game engine or a renderer loading this library as a plugin, or a real-time thread that must never block
// in the driver's allocator).  The caller passes its own device buffers for the inputs and the output; the
// kernel's scratch (one partial sum per block and the arrival ticket of the last-block finish) lives in a
// file-scope __device__ array that every GPU loading the library holds until the process exits.
#include <mutex>
#include <string>

#include "../../include/pncg.h"
#include "common.cuh"
#include "geometry.cuh"

namespace {

constexpr int NA_THREADS = 256;
constexpr int NA_MAX_BLOCKS = 1 << 16;                                // 512 KiB of partial sums
constexpr long long NA_MAX_ITEMS = (long long)NA_THREADS * NA_MAX_BLOCKS;  // 16,777,216 tets or vertices
constexpr int NA_MAX_DEVICES = 64;

struct NoAllocScratch {
    double partial[NA_MAX_BLOCKS];
    unsigned int ticket;
};

// The scratch: shared by every call on a device, it keeps the last call's contents.
static __device__ __align__(256) NoAllocScratch g_noalloc_scratch;

std::mutex g_setup_mutex;
NoAllocScratch *g_scratch_ptr[NA_MAX_DEVICES] = {};
thread_local std::string g_noalloc_err;

struct Mat3 { double m[3][3]; };   // columns are edge vectors
__device__ inline Mat3 edges(const double *x, const int v[4])
{
    Mat3 d;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        const double x0 = x[3 * v[0] + a];
#pragma unroll
        for (int c = 0; c < 3; ++c) d.m[a][c] = x[3 * v[c + 1] + a] - x0;
    }
    return d;
}
// columns d1 x d2, d2 x d0, d0 x d1
__device__ inline Mat3 cofactors(const Mat3 &d)
{
    Mat3 c;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const int p = (b + 1) % 3, q = (b + 2) % 3;
        c.m[0][b] = d.m[1][p] * d.m[2][q] - d.m[2][p] * d.m[1][q];
        c.m[1][b] = d.m[2][p] * d.m[0][q] - d.m[0][p] * d.m[2][q];
        c.m[2][b] = d.m[0][p] * d.m[1][q] - d.m[1][p] * d.m[0][q];
    }
    return c;
}

// p^T M p + h^2 sum_e V_e [mu |dF|^2 + Psi_33 (cof F : dF)^2 + Psi_3 d2det(F)[dF, dF]] in double precision, one
// thread per tet (and per vertex for the inertia term).  With the edge vectors of the rest, current and direction
// values Dm, Ds, Dp (columns): J = det Ds / det Dm, cof F : dF = cof(Ds) : Dp / det Dm, d2det(F)[dF, dF] = 2 cof(Dp) : Ds /
// det Dm and dF = Dp cof(Dm)^T / det Dm, so that neither D_m^-1 nor F is formed.  Bound by FP64 issue (1.68 lanes per
// clock and SM): about 175 operations a tet with two divisions, where the form on F took about 400 with nine.  998,250 tets:
// on F 768 us, on edge vectors 411, with det_forms and log_tab 354.
__global__ void __launch_bounds__(NA_THREADS) k_pHp_noalloc(NoAllocScratch *scr, int nv, int nt, const double *x,
                                                             const double *p, const double *X, const int *tets,
                                                             const double *mass, double mu, double lam, double h2,
                                                             double *out)
{
    __shared__ double sh[32];
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double s[1] = {0.0};
    if (i < nv) {
        const double px = p[3 * i], py = p[3 * i + 1], pz = p[3 * i + 2];
        s[0] += mass[i] * (px * px + py * py + pz * pz);
    }
    if (i < nt) {
        const int v[4] = {tets[4 * i], tets[4 * i + 1], tets[4 * i + 2], tets[4 * i + 3]};
        const Mat3 A = edges(X, v), Ds = edges(x, v), Dp = edges(p, v);
        const Mat3 ca = cofactors(A);
        const double det = A.m[0][0] * ca.m[0][0] + A.m[1][0] * ca.m[1][0] + A.m[2][0] * ca.m[2][0];
        double ds = 0.0, g3, h3;
#pragma unroll
        for (int a = 0; a < 3; ++a)     // s_1 . (s_2 x s_0), whose cross product det_forms has too
            ds += Ds.m[a][1] * (Ds.m[(a + 1) % 3][2] * Ds.m[(a + 2) % 3][0] - Ds.m[(a + 2) % 3][2] * Ds.m[(a + 1) % 3][0]);
        pncg::det_forms<double>(Ds.m, Dp.m, g3, h3);
        if (ds > 0.0 && det > 0.0) {
            const double idet = 1.0 / det, J = ds * idet, iJ = det / ds;
            const double L = pncg::log_tab(J);
            const double Psi3 = (lam * L - mu) * iJ, Psi33 = (mu + lam * (1.0 - L)) * iJ * iJ;
            double n2 = 0.0;
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int b = 0; b < 3; ++b) {
                    const double f = Dp.m[a][0] * ca.m[b][0] + Dp.m[a][1] * ca.m[b][1] + Dp.m[a][2] * ca.m[b][2];
                    n2 += f * f;
                }
            g3 *= idet;
            h3 *= 2.0 * idet;
            s[0] += h2 * (det * (1.0 / 6.0)) * (mu * (n2 * idet * idet) + Psi33 * (g3 * g3) + Psi3 * h3);
        } else {
            s[0] = nan("");     // an inverted current tet, or a rest tet of non-positive volume
        }
    }
    pncg::block_sum<1>(s, sh);
    if (pncg::publish_partials<1>(s, scr->partial, &scr->ticket)) {
        double t[1];
        pncg::finish_sums<1>(t, scr->partial, sh);
        if (threadIdx.x == 0) *out = t[0];
    }
}

} // namespace

extern "C" {

const char *sim_noalloc_last_error(void) { return g_noalloc_err.c_str(); }

sim_status sim_pHp_noalloc(int32_t n_verts, int32_t n_tets, const double *x, const double *p, const double *rest_x,
                           const int32_t *tets, const double *mass, double youngs, double poisson, double dt,
                           double *out, void *cuda_stream)
{
    if (n_verts <= 0 || n_tets <= 0 || !x || !p || !rest_x || !tets || !mass || !out || !(dt > 0) ||
        !(poisson > -1.0 && poisson < 0.5)) {
        g_noalloc_err = "sim_pHp_noalloc: invalid argument";
        return SIM_ERR_INVALID_ARG;
    }
    if ((long long)n_verts > NA_MAX_ITEMS || (long long)n_tets > NA_MAX_ITEMS) {
        g_noalloc_err = "sim_pHp_noalloc: at most " + std::to_string(NA_MAX_ITEMS) +
                        " tets and vertices per call (the static scratch holds " + std::to_string(NA_MAX_BLOCKS) +
                        " block partial sums)";
        return SIM_ERR_INVALID_ARG;
    }
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || dev < 0 || dev >= NA_MAX_DEVICES) {
        g_noalloc_err = "sim_pHp_noalloc: no usable CUDA device";
        return SIM_ERR_CUDA;
    }
    NoAllocScratch *scr;
    {
        // first call on this device: the scratch's device address (the symbol's host name is only a stand-in)
        std::lock_guard<std::mutex> lock(g_setup_mutex);
        if (!g_scratch_ptr[dev]) {
            void *ptr = nullptr;
            e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);
            if (e != cudaSuccess || !ptr) {
                g_noalloc_err = std::string("sim_pHp_noalloc: cudaGetSymbolAddress failed: ") + cudaGetErrorString(e);
                return SIM_ERR_CUDA;
            }
            g_scratch_ptr[dev] = (NoAllocScratch *)ptr;
        }
        scr = g_scratch_ptr[dev];
    }
    cudaStream_t s = (cudaStream_t)cuda_stream;
    // the arrival ticket must start at zero (the finishing block also resets it)
    e = cudaMemsetAsync(&scr->ticket, 0, sizeof(unsigned int), s);
    if (e != cudaSuccess) {
        g_noalloc_err = std::string("sim_pHp_noalloc: ") + cudaGetErrorString(e);
        return SIM_ERR_CUDA;
    }
    const double mu = youngs / (2.0 * (1.0 + poisson)), lam = youngs * poisson / ((1.0 + poisson) * (1.0 - 2.0 * poisson));
    const int n = n_verts > n_tets ? n_verts : n_tets;
    const int blocks = (n + NA_THREADS - 1) / NA_THREADS;
    k_pHp_noalloc<<<blocks, NA_THREADS, 0, s>>>(scr, n_verts, n_tets, x, p, rest_x, tets, mass, mu, lam, dt * dt, out);
    e = cudaGetLastError();
    if (e != cudaSuccess) {
        g_noalloc_err = std::string("sim_pHp_noalloc: launch failed: ") + cudaGetErrorString(e);
        return SIM_ERR_CUDA;
    }
    return SIM_OK;
}

} // extern "C"
