// noalloc.cu -- diagnostics of a caller-owned population array without any
// device allocation.
//
// Some callers cannot call cudaMalloc at the point where they need these
// numbers: hosts whose device memory is handed out by their own pool or held to a
// fixed budget, which a library must not grow or fragment behind their back, and
// latency-bound loops where the implicit device synchronisation an allocation can
// cause is not acceptable.  For them, vlbm_diagnostics_noalloc reduces a
// population array the caller already owns, using a fixed scratch array compiled
// into the library instead of memory from cudaMalloc.
//
// The scratch is a file-scope __device__ array of VLBM_NOALLOC_MAX_ROWS x 6
// doubles (768 KiB, six partial sums per CTA of at most VLBM_NOALLOC_MAX_ROWS); every GPU that loads the library holds it until the
// process exits.  Host code cannot use the array's name as a device address, so
// the first call on each device looks its address up with cudaGetSymbolAddress
// (with that device current) and caches it; that first call should therefore
// come before any stream capture, and the cached address does not survive a
// cudaDeviceReset of that device.  All calls share the one array: calls whose
// kernels overlap on the GPU (on different streams) race on it.  The per-CTA
// partial sums are fully rewritten by every call, so nothing in the scratch has
// to start at zero.
#include <mutex>
#include <string>

#include "../../include/vlbm.h"
#include "vlbm_internal.h"

namespace {

constexpr int NOALLOC_THREADS = 128;
constexpr int NQ = 6;   // mass, momentum x/y/z, energy, non-finite count
constexpr int MAX_DEVICES = 64;

static __device__ __align__(256) double g_noalloc_scratch[(size_t)VLBM_NOALLOC_MAX_ROWS * NQ];

std::mutex g_mu;
double *g_scratch_ptr[MAX_DEVICES] = {};
thread_local std::string g_noalloc_error;

struct VelNA { double v2, v3; };   // the positive velocities (v[2], v[3]); v[0] = -v[3], v[1] = -v[2]

// Sums of a dense [16][nt][np] FP64 population array.  Bound: GB300's FP64 pipe (one warp
// instruction per 64 cycles and scheduler), so the work per cell is kept to 40 FP64 instructions:
// the sums of each k_theta row and k_phi column of the 4 x 4 populations (24 additions) give
// density, momenta (the velocities come in +- pairs) and energy, a thread keeps one column for all
// its rows so that cos(phi), sin(phi) enter once per column, and the row factors are formed once per
// CTA.  (One thread per cell with its own sincos took 170 FP64 instructions a cell: 177 us for
// 512 x 1024.)  Non-finite values are found on the exponent bits in the integer pipe.
// Thread: column 32 chunk + lane, rows blockIdx.y rows .. + rows - 1; a CTA's four warps take
// consecutive column chunks.
constexpr int NA_ROWS_MAX = 64;

__device__ __forceinline__ void na_load(const double *f, size_t plane, size_t cell, double (&v)[16])
{
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __ldg(f + k * plane + cell);
}

__global__ void __launch_bounds__(NOALLOC_THREADS) noalloc_sums_kernel(const double *f, int nt, int np, double radius,
                                                                        VelNA c, int rows, double *part)
{
    __shared__ double rs[NA_ROWS_MAX], rc[NA_ROWS_MAX];   // sin(theta), cos(theta) of the CTA's rows
    __shared__ double ls[32], lc[32];                      // sin, cos of a lane's offset in its chunk of columns
    __shared__ double bs[NOALLOC_THREADS / 32], bc[NOALLOC_THREADS / 32];   // ... of the warps' first chunks
    __shared__ double red[NQ][NOALLOC_THREADS / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int i0 = blockIdx.y * rows, n = min(rows, nt - i0);
    const double pi = 3.14159265358979323846;
    const double area = radius * radius * (pi / nt) * (2.0 * pi / np);
    // one sincos per thread, in warps of their own: the rows (threads 0 .. 63), the lane offsets and the chunks
    if ((int)threadIdx.x < NA_ROWS_MAX) {
        const int i = i0 + min((int)threadIdx.x, n - 1), m = nt - 1 - i;
        double st, ct;
        sincospi(((i <= m ? i : m) + 0.5) / nt, &st, &ct);
        if (i == m) ct = 0.0;
        if (i > m) ct = -ct;
        rs[threadIdx.x] = st;
        rc[threadIdx.x] = ct;
    } else if (warp == 2) {
        sincospi((2.0 * lane + 1.0) / np, &ls[lane], &lc[lane]);
    } else if (lane < NOALLOC_THREADS / 32) {
        sincospi(64.0 * (blockIdx.x * (NOALLOC_THREADS / 32) + lane) / np, &bs[lane], &bc[lane]);
    }
    __syncthreads();
    const size_t plane = (size_t)nt * np;
    const int chunks = (np + 31) / 32;
    double acc[NQ] = {0, 0, 0, 0, 0, 0};
    int bad = 0;
    for (int ch = blockIdx.x * (NOALLOC_THREADS / 32) + warp; ch < chunks; ch += gridDim.x * (NOALLOC_THREADS / 32)) {
        const int j = 32 * ch + lane;
        const bool in = j < np;
        const size_t cell0 = (size_t)i0 * np + (in ? j : np - 1);
        // sums over the rows, weighted by the row's sine: populations of |v_theta| = v[3] and v[2], of
        // |v_phi| = v[3], j_theta cos(theta), j_phi, j_theta sin(theta)
        double so = 0.0, si = 0.0, sp = 0.0, a = 0.0, b = 0.0, z = 0.0;
        double v[16];
        na_load(f, plane, cell0, v);
        for (int r = 0; r < n; ++r) {
            double w[16];
            if (r + 1 < n) na_load(f, plane, cell0 + (size_t)(r + 1) * np, w);
            int top = 0;
#pragma unroll
            for (int k = 0; k < 16; ++k) top = max(top, __double2hiint(v[k]) & 0x7fffffff);
            if (in && top >= 0x7ff00000) ++bad;
            double R[4], C[4];
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                R[m] = (v[4 * m] + v[4 * m + 1]) + (v[4 * m + 2] + v[4 * m + 3]);
                C[m] = (v[m] + v[m + 4]) + (v[m + 8] + v[m + 12]);
            }
            const double jt = fma(c.v3, R[3] - R[0], c.v2 * (R[2] - R[1]));
            const double jp = fma(c.v3, C[3] - C[0], c.v2 * (C[2] - C[1]));
            const double s = rs[r], sj = s * jt;
            so = fma(s, R[0] + R[3], so);
            si = fma(s, R[1] + R[2], si);
            sp = fma(s, C[0] + C[3], sp);
            a = fma(rc[r], sj, a);
            b = fma(s, jp, b);
            z = fma(s, sj, z);
            if (r + 1 < n) {
#pragma unroll
                for (int k = 0; k < 16; ++k) v[k] = w[k];
            }
        }
        if (!in) continue;
        // phi_j = 2 pi (32 ch) / np + (2 lane + 1) pi / np
        double sb = bs[warp], cb = bc[warp];
        if (ch >= (int)(gridDim.x * (NOALLOC_THREADS / 32))) sincospi(64.0 * ch / np, &sb, &cb);
        const double sph = fma(sb, lc[lane], cb * ls[lane]), cph = fma(cb, lc[lane], -(sb * ls[lane]));
        // sum |v|^2 f = v3^2 (so + sp) + v2^2 (si + the populations of |v_phi| = v[2]: the others of the mass;
        // an infinite sp is in so or si as well, and infinities of both signs meet there)
        const double mass = so + si, rest = isinf(sp) ? 0.0 : mass - sp;
        acc[0] += mass;
        acc[1] += fma(a, cph, -(b * sph));
        acc[2] += fma(a, sph, b * cph);
        acc[3] -= z;
        acc[4] += fma(c.v3 * c.v3, so + sp, c.v2 * c.v2 * (si + rest));
    }
    acc[5] = bad;
    // warps by a butterfly whose first steps also halve the sums that a lane carries (9 additions, not 30):
    // after them lane l has sum l / 4 of its group of 8 quantities, over all lanes
    double h4[4], h2[2];
    const bool u16 = lane & 16, u8 = lane & 8, u4 = lane & 4;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const double up = q + 4 < NQ ? acc[q + 4 < NQ ? q + 4 : 0] : 0.0;
        h4[q] = (u16 ? up : acc[q]) + __shfl_xor_sync(0xffffffffu, u16 ? acc[q] : up, 16);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
        h2[q] = (u8 ? h4[q + 2] : h4[q]) + __shfl_xor_sync(0xffffffffu, u8 ? h4[q] : h4[q + 2], 8);
    double h = (u4 ? h2[1] : h2[0]) + __shfl_xor_sync(0xffffffffu, u4 ? h2[0] : h2[1], 4);
    h += __shfl_xor_sync(0xffffffffu, h, 2);
    h += __shfl_xor_sync(0xffffffffu, h, 1);
    if ((lane & 3) == 0 && lane / 4 < NQ) red[lane / 4][warp] = h;
    __syncthreads();
    if (threadIdx.x < NQ) {
        const int q = threadIdx.x;
        static_assert(NOALLOC_THREADS == 128, "four warps");
        const double t = (red[q][0] + red[q][1]) + (red[q][2] + red[q][3]);
        const double scale = (q < 4) ? area : (q == 4 ? 0.5 * area : 1.0);
        part[(size_t)q * gridDim.x * gridDim.y + (size_t)blockIdx.y * gridDim.x + blockIdx.x] = t * scale;
    }
}

// One warp per quantity adds the n CTA partials in a fixed order: four chains a lane, then a tree.  (One chain
// was up to 40 additions long, the longest of the whole sum.  Emulated against extended precision over ten grids
// of 16 x 20 to 800 x 1500, the root mean square errors relative to those of the form with one block per row:
// momentum vector 0.42 to 0.93, mass 0.64 to 1.21 (0.90 on the average), energy 0.48 to 1.26 (0.85).)
__global__ void __launch_bounds__(32 * NQ) noalloc_final_kernel(const double *part, int n, double *out)
{
    const int lane = threadIdx.x & 31, q = threadIdx.x >> 5;
    double t[4] = {0.0, 0.0, 0.0, 0.0};
    for (int b = lane; b < n; b += 128)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (b + 32 * k < n) t[k] += part[(size_t)q * n + b + 32 * k];
    double s = (t[0] + t[2]) + (t[1] + t[3]);
#pragma unroll
    for (int m = 16; m > 0; m >>= 1) s += __shfl_xor_sync(0xffffffffu, s, m);
    if (lane == 0) out[q] = s;
}

int na_fail(int code, const std::string &m)
{
    g_noalloc_error = m;
    return code;
}

// Device address of the scratch array for the current device (looked up once per device).
int scratch_for_current_device(double **out)
{
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return na_fail(VLBM_ERR_CUDA, std::string("cudaGetDevice: ") + cudaGetErrorString(e));
    if (dev < 0 || dev >= MAX_DEVICES) return na_fail(VLBM_ERR_UNSUPPORTED, "device ordinal beyond 63");
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_scratch_ptr[dev]) {
        double *p = nullptr;
        e = cudaGetSymbolAddress((void **)&p, g_noalloc_scratch);
        if (e != cudaSuccess || !p)
            return na_fail(VLBM_ERR_CUDA, std::string("cudaGetSymbolAddress: ") + cudaGetErrorString(e));
        g_scratch_ptr[dev] = p;
    }
    *out = g_scratch_ptr[dev];
    return VLBM_OK;
}

}  // namespace

extern "C" {

int vlbm_diagnostics_noalloc(const double *f_dev, int n_theta, int n_phi, double radius, double *out_dev,
                             void *stream)
{
    if (!f_dev || !out_dev) return na_fail(VLBM_ERR_ARG, "NULL device pointer");
    if (n_theta < 1 || n_phi < 1 || !(radius > 0.0)) return na_fail(VLBM_ERR_ARG, "bad grid or radius");
    if (n_theta > VLBM_NOALLOC_MAX_ROWS)
        return na_fail(VLBM_ERR_ARG, "n_theta = " + std::to_string(n_theta) + " exceeds the scratch limit of " +
                                         std::to_string(VLBM_NOALLOC_MAX_ROWS) + " rows");
    double *part = nullptr;
    int rc = scratch_for_current_device(&part);
    if (rc) return rc;
    const VelNA c{sqrt(3.0 - sqrt(6.0)), sqrt(3.0 + sqrt(6.0))};
    cudaStream_t s = (cudaStream_t)stream;
    // rows per CTA: two warps per scheduler (608 of them) where the grid is large enough, which
    // saturates the FP64 pipe; within the shared row tables and the scratch's count of CTAs
    const int chunks = (n_phi + 31) / 32, cx = (chunks + NOALLOC_THREADS / 32 - 1) / (NOALLOC_THREADS / 32);
    const long long want = ((long long)n_theta * chunks + 1215) / 1216;
    const int rows = (int)(want < 1 ? 1 : want > NA_ROWS_MAX ? NA_ROWS_MAX : want);
    const int gy = (n_theta + rows - 1) / rows, gx = cx < VLBM_NOALLOC_MAX_ROWS / gy ? cx : VLBM_NOALLOC_MAX_ROWS / gy;
    noalloc_sums_kernel<<<dim3(gx, gy), NOALLOC_THREADS, 0, s>>>(f_dev, n_theta, n_phi, radius, c, rows, part);
    noalloc_final_kernel<<<1, 32 * NQ, 0, s>>>(part, gx * gy, out_dev);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return na_fail(VLBM_ERR_CUDA, std::string("launch: ") + cudaGetErrorString(e));
    return VLBM_OK;
}

const char *vlbm_noalloc_last_error(void) { return g_noalloc_error.c_str(); }

}  // extern "C"
