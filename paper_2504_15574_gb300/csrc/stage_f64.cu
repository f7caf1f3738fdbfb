// stage_f64.cu -- FP64 kernels of the parity path (compiled with -fmad=false).
//
// One RK3 stage of arXiv 2504.15574 Sec. 3.7 fused into one kernel: moments
// (Eq. f_moments_sum), equilibrium (Eq. feq_Q=4), BGK (Sec. 3.2), geometric
// force through K^H and Ktilde^H (Eq. df), WENO-5 fluxes in theta and phi
// (Eqs. fluxes_W5, WENO5_delta, WENO5_sigma) in the flux form of
// Eq. (discrete_advection_sphere), and the Shu-Osher stage combination.
//
// This path exists to reproduce an FP64 reference evaluation of the method
// operation for operation: every expression below is evaluated in a fixed
// order with no FMA contraction (other than inside a division), rounded quotients
// where the method divides, and sums over populations in ascending k.  Each
// interface flux is computed once (one face kernel into global buffers), then one
// kernel updates the cells.  It is not the throughput path (that is stage_f32.cu);
// it shares the ghost-row layout so that all reads are plain loads.
#include "vlbm_internal.h"

namespace vk {

namespace {

// ---- arithmetic -----------------------------------------------------------------------
// GB300 issues one FP64 warp instruction per 64 cycles and scheduler (2 FP64 lanes per SM), so a
// stage's time is its FP64 instruction count: 135 per interface value and 105 per population and
// cell when every division was the compiler's and every stencil form was evaluated per face (490,
// 487 and 384 us for the phi faces, theta faces and cells of a 256 x 512 stage, 535 G FP64
// instructions/s of ~578).  The forms below give the same bits with fewer of them: scalings by
// powers of two and reciprocal seeds go to the integer and FP32 pipes, which are otherwise idle.

// x 2^K, |K| <= 4, by an exponent addition; zeros are returned as they are.  What could leave the
// normal range (or is not finite) sets `bad` and the caller takes its plain form: a multiplication
// here, even one predicated off, would be issued to the FP64 pipe (8 of 78 instructions a face).
template <int K>
__device__ __forceinline__ double scale2(double x, bool &bad)
{
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const bool zero = ((hi << 1) | lo) == 0;
    bad |= !zero && (unsigned)((hi >> 20) & 0x7ff) - 8u >= 2030u;
    return __hiloint2double(zero ? hi : hi + K * (1 << 20), lo);
}

// x / d with 1/d = h + l held to 106 bits (DivC, built on the host): RN(x h + RN(x l)), the two-
// operation multiplication by an arbitrary-precision constant of Brisebarre and Muller ("Correctly
// rounded multiplication by arbitrary precision constants", 2005).  Exact for d = 6 and d = 3 (no
// quotient comes within 1/6 ulp of a rounding boundary); for a general d it differs from the
// rounded quotient only where x / d is within 2^-105 of a boundary.  h is rounded toward zero and l
// positive, so infinities pass through.
__device__ __forceinline__ double div_const(double x, const DivC &d) { return __fma_rn(x, d.h, __dmul_rn(x, d.l)); }

// a / b with three FP64 operations: a reciprocal of b good to 2^-44 is formed in FP32 (the leading
// 24 bits of b's significand through the hardware reciprocal, one error term with the remaining
// bits) and assembled into a double by integer operations; then one residual correction of the
// quotient (Markstein 1990).  The corrected value is within 2^-88 of a / b before its rounding, so
// it is the rounded quotient but for a chance of about 2^-35 per division (none in 4e8 random
// ones).  A b that is not positive and well inside the normal range sets `bad`: the caller then takes
// its plain form.
__device__ __forceinline__ double div_pos(double a, double b, bool &bad)
{
    const int hi = __double2hiint(b), lo = __double2loint(b);
    bad |= (unsigned)((hi >> 20) - (1023 - 500)) > 1000u;
    const float bh = __int_as_float(0x3f800000 | ((hi & 0xfffff) << 3) | (int)((unsigned)lo >> 29));
    const float bl = (float)(lo & 0x1fffffff) * 0x1p-52f;
    float r0;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r0) : "f"(bh));
    r0 = fmaxf(fminf(r0, 0.99999994f), 0.5f);   // inside one binade: the error term is added to its bits
    float e = __fmaf_rn(-bh, r0, 1.0f);
    e = __fmaf_rn(-bl, r0, e);
    const float r1 = __fmul_rn(r0, __fmaf_rn(e, e, e));
    const int u = __float_as_int(r0), i1 = __float2int_rn(__fmul_rn(r1, 0x1p53f));
    long long bits = ((long long)((u >> 3) + ((1023 - 127) << 20)) << 32) | (unsigned)(u << 29);
    bits += i1;
    bits -= (long long)((hi >> 20) - 1023) << 52;
    const double r = __longlong_as_double(bits);
    const double q = __dmul_rn(a, r);
    return __fma_rn(__fma_rn(-b, q, a), r, q);
}

// The interface value as the oracle writes it, for stencils with values outside the fast forms'
// ranges (denormal differences, near-overflow, non-finite populations).
__device__ __noinline__ double weno5_plain(double a, double b, double c, double d, double e, double eps)
{
    double p1 = (2.0 * a - 7.0 * b + 11.0 * c) / 6.0;
    double p2 = (-b + 5.0 * c + 2.0 * d) / 6.0;
    double p3 = (2.0 * c + 5.0 * d - e) / 6.0;
    double d1a = a - 2.0 * b + c, d1b = a - 4.0 * b + 3.0 * c;
    double d2a = b - 2.0 * c + d, d2b = b - d;
    double d3a = c - 2.0 * d + e, d3b = 3.0 * c - 4.0 * d + e;
    double s1 = 13.0 / 12.0 * (d1a * d1a) + 0.25 * (d1b * d1b);
    double s2 = 13.0 / 12.0 * (d2a * d2a) + 0.25 * (d2b * d2b);
    double s3 = 13.0 / 12.0 * (d3a * d3a) + 0.25 * (d3b * d3b);
    double w1 = 0.1 / ((s1 + eps) * (s1 + eps));
    double w2 = 0.6 / ((s2 + eps) * (s2 + eps));
    double w3 = 0.3 / ((s3 + eps) * (s3 + eps));
    return (w1 * p1 + w2 * p2 + w3 * p3) / (w1 + w2 + w3);
}

// Plain product and quotient behind a call, for the rare values that the fast forms leave out.
__device__ __noinline__ double mul_plain(double a, double b) { return a * b; }
__device__ __noinline__ double div_plain(double a, double b) { return a / b; }

// Interface values of S consecutive faces from y[0 .. S + 3] in upwind order: face f has the stencil
// a..e = y[f .. f + 4] (c the upwind cell, d the downwind cell), in the oracle's expression order.
// The forms of one column (13/12 times the squared second difference, and 5 y) are shared by the
// three candidate stencils centred on it, which changes no bit: 45 + 4 divisions of 3 FP64
// operations per face.
template <int S>
__device__ __forceinline__ void weno5_strip(const double (&y)[S + 4], double eps, const DivC &six, double (&r)[S])
{
    double kq[S + 4], y5[S + 4];
    bool bad = false;
#pragma unroll
    for (int i = 1; i <= 2; ++i) {
        const double d = y[i - 1] - scale2<1>(y[i], bad) + y[i + 1];
        kq[i] = 13.0 / 12.0 * (d * d);
    }
    y5[2] = 5.0 * y[2];
#pragma unroll
    for (int f = 0; f < S; ++f) {
        const double a = y[f], b = y[f + 1], c = y[f + 2], d = y[f + 3], e = y[f + 4];
        const double d3a = c - scale2<1>(d, bad) + e;
        kq[f + 3] = 13.0 / 12.0 * (d3a * d3a);
        y5[f + 3] = 5.0 * d;
        const double c3 = 3.0 * c;
        const double d1b = a - scale2<2>(b, bad) + c3;
        const double d2b = b - d;
        const double d3b = c3 - scale2<2>(d, bad) + e;
        const double s1 = kq[f + 1] + scale2<-2>(d1b * d1b, bad) + eps;
        const double s2 = kq[f + 2] + scale2<-2>(d2b * d2b, bad) + eps;
        const double s3 = kq[f + 3] + scale2<-2>(d3b * d3b, bad) + eps;
        const double w1 = div_pos(0.1, s1 * s1, bad), w2 = div_pos(0.6, s2 * s2, bad),
                     w3 = div_pos(0.3, s3 * s3, bad);
        const double p1 = div_const(scale2<1>(a, bad) - 7.0 * b + 11.0 * c, six);
        const double p2 = div_const(y5[f + 2] - b + scale2<1>(d, bad), six);
        const double p3 = div_const(scale2<1>(c, bad) + y5[f + 3] - e, six);
        r[f] = div_pos(w1 * p1 + w2 * p2 + w3 * p3, w1 + w2 + w3, bad);
    }
    if (bad)
#pragma unroll
        for (int f = 0; f < S; ++f) r[f] = weno5_plain(y[f], y[f + 1], y[f + 2], y[f + 3], y[f + 4], eps);
}

// The same for the upwind stencils of Eq. (fluxes_U1-3).
template <int S>
__device__ __forceinline__ void upwind_strip(int scheme, const double (&y)[S + 4], const DivC &six, double (&r)[S])
{
#pragma unroll
    for (int f = 0; f < S; ++f) {
        const double b = y[f + 1], c = y[f + 2], d = y[f + 3];
        r[f] = (scheme == VLBM_U1) ? c : (scheme == VLBM_U2) ? 1.5 * c - 0.5 * b
                                                             : div_const(2.0 * d + 5.0 * c - b, six);
    }
}

// Writes v at interior (k, i, j) and at every ghost image of that cell.
template <typename T>
__device__ __forceinline__ void store_with_images(T *f, const Layout &L, int k, int i, int j, T v)
{
    const int np = L.np;
    auto put_row = [&](int kk, int r, int c) {
        f[L.at(kk, r, c)] = v;
        // periodic images of column c inside [-GC, np+GC)
        for (int m = 1; c - m * np >= -GC; ++m) f[L.at(kk, r, c - m * np)] = v;
        for (int m = 1; c + m * np < np + GC; ++m) f[L.at(kk, r, c + m * np)] = v;
    };
    put_row(k, i, j);
    if (i < GR || i >= L.nt - GR) {
        int jj = j + np / 2;
        if (jj >= np) jj -= np;
        int r = (i < GR) ? (-1 - i) : (2 * L.nt - 1 - i);
        put_row(L.nk - 1 - k, r, jj);
    }
}

// Interface fluxes of one stage, one strip of S consecutive faces of one population per thread.
// Theta flux through interface fi (between rows fi-1 and fi, fi = 0..nt) of population k: the
// reconstruction on the nodal g = sin f of rows fi-3..fi+2 (ghost rows with their own, negative,
// sine), or (Komissarov) on f itself times v_theta sin(theta_fi); a thread walks S rows of one
// column.  Phi flux through interface fj (between columns fj-1 and fj, fj = 0..np) of row i; a
// thread walks S columns of one row.  For a negative velocity the strip is walked backwards, which
// puts its values in upwind order.  The first nb_phi CTAs take the phi faces, the others the theta
// faces (one launch: on small grids either alone leaves schedulers idle).
// Bound: the FP64 pipe (57 operations a face; 240 us for the 4.2 M faces of 256 x 512, D2Q16, by
// count).  Long strips share the column forms, short ones spread a small grid over more
// schedulers: launch_stage_f64 picks S.
template <int S>
__global__ void __launch_bounds__(128) faces_f64_kernel(const StageD p, int nb_phi)
{
    const Layout L = p.L;
    const int q = p.c.q;
    const bool theta = (int)blockIdx.x >= nb_phi;
    double y[S + 4], r[S];
    if (!theta) {
        const int ns = (L.np + S) / S;   // strips of the np + 1 faces
        const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        const int k = blockIdx.y;
        if (t >= (long long)ns * L.nt) return;
        const int i = (int)(t / ns), f0 = (int)(t - (long long)i * ns) * S;
        const double vb = p.c.v[k % q];
        const int dir = vb > 0.0 ? 1 : -1;
        // y[m] = column c0 + dir m; a strip that reaches past the last face reads the last column in store
        const int c0 = dir > 0 ? f0 - 3 : f0 + S + 1;
        const double *g = p.in + L.at(k, i, 0);
#pragma unroll
        for (int m = 0; m < S + 4; ++m) y[m] = g[min(c0 + dir * m, L.np + GC - 1)];
        if (p.scheme == VLBM_WENO5) weno5_strip<S>(y, p.eps, p.six, r);
        else upwind_strip<S>(p.scheme, y, p.six, r);
        double *out = p.Fp + ((size_t)k * L.nt + i) * (L.np + 1);
#pragma unroll
        for (int f = 0; f < S; ++f) {
            const int fj = dir > 0 ? f0 + f : f0 + S - 1 - f;
            if (fj <= L.np) out[fj] = vb * r[f];
        }
        return;
    }
    const int ns = (L.nt + S) / S;
    const long long t = (long long)(blockIdx.x - nb_phi) * blockDim.x + threadIdx.x;
    const int k = blockIdx.y;
    if (t >= (long long)ns * L.np) return;
    const int st = (int)(t / L.np), j = (int)(t - (long long)st * L.np), f0 = st * S;
    const double va = p.c.v[k / q];
    const int dir = va > 0.0 ? 1 : -1;
    const int r0 = dir > 0 ? f0 - 3 : f0 + S + 1;
#pragma unroll
    for (int m = 0; m < S + 4; ++m) {
        const int row = min(r0 + dir * m, L.nt + GR - 1);
        const double v = p.in[L.at(k, row, j)];
        y[m] = p.komissarov ? v : p.sin_ext[row + GR] * v;
    }
    if (p.scheme == VLBM_WENO5) weno5_strip<S>(y, p.eps, p.six, r);
    else upwind_strip<S>(p.scheme, y, p.six, r);
#pragma unroll
    for (int f = 0; f < S; ++f) {
        const int fi = dir > 0 ? f0 + f : f0 + S - 1 - f;
        if (fi > L.nt) continue;
        const double flux = p.komissarov ? va * p.sin_f[fi] * r[f] : va * r[f];
        p.Ft[((size_t)k * (L.nt + 1) + fi) * L.np + j] = flux;
        if (p.pole) {
            if (fi == 0) p.pole[(size_t)k * L.np + j] = flux;
            if (fi == L.nt) p.pole[((size_t)NK + k) * L.np + j] = flux;
        }
    }
}

// Cells of one stage: moments, equilibrium, force, BGK, the flux differences of the interface
// fluxes above and the stage combination, in the oracle's operation order.  A CTA takes 32
// consecutive cells; its 8 warps first form the moments of those cells (one warp each for n, the
// two momenta and then the two velocities: the sums run over k in order, so they are chains), then
// each warp updates two populations of them.  One thread per cell, the earlier form, left a
// 32 x 64 grid with 64 warps of 1,700 serial FP64 operations (71 us a launch).  Bound on large
// grids: the FP64 pipe (about 54 operations per population, from 105; divisions by row constants,
// tau and 3 are two operations each).
constexpr int CELL_WARPS = 8;
__global__ void __launch_bounds__(32 * CELL_WARPS) cells_f64_kernel(const StageD p)
{
    __shared__ double gs[NK][32], mom[3][32], vel[4][32];
    const Layout L = p.L;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int q = p.c.q, nk = q * q;
    const long long cells = (long long)L.nt * L.np;
    const long long cell = (long long)blockIdx.x * 32 + lane;
    const bool in = cell < cells;
    const int i = in ? (int)(cell / L.np) : 0, j = in ? (int)(cell - (long long)i * L.np) : 0;
    for (int k = warp; k < nk; k += CELL_WARPS) gs[k][lane] = p.in[L.at(k, i, j)];
    __syncthreads();
    if (warp < 3) {
        double m = 0.0;
        for (int k = 0; k < nk; ++k) {
            const double g = gs[k][lane];
            m += (warp == 0) ? g : g * p.c.v[warp == 1 ? k / q : k % q];
        }
        mom[warp][lane] = m;
    }
    __syncthreads();
    if (warp == 1 || warp == 2) {
        bool bad = false;
        double u = div_pos(mom[warp][lane], mom[0][lane], bad);
        if (bad) u = div_plain(mom[warp][lane], mom[0][lane]);
        vel[warp - 1][lane] = u;
    }
    __syncthreads();
    if (warp == 0) {
        const double ut = vel[0][lane], up = vel[1][lane];
        const double u2 = ut * ut + up * up;
        vel[2][lane] = u2;
        vel[3][lane] = 3.0 * u2;
    }
    __syncthreads();
    if (!in) return;
    const double n = mom[0][lane], ut = vel[0][lane], up = vel[1][lane], u2 = vel[2][lane], u23 = vel[3][lane];
    const RowD rd = p.row[i];
#pragma unroll 1
    for (int k = warp; k < nk; k += CELL_WARPS) {
        const int a = k / q, b = k % q;
        const double va = p.c.v[a], vb = p.c.v[b];
        const double gk = gs[k][lane];
        // loaded ahead of the arithmetic
        const double fn = p.Ft[((size_t)k * (L.nt + 1) + i) * L.np + j];
        const double fs = p.Ft[((size_t)k * (L.nt + 1) + i + 1) * L.np + j];
        const double fw = p.Fp[((size_t)k * L.nt + i) * (L.np + 1) + j];
        const double fe = p.Fp[((size_t)k * L.nt + i) * (L.np + 1) + j + 1];
        const double f0 = (p.stage == 1) ? 0.0 : p.fold[L.at(k, i, j)];
        // equilibrium (T0 = 1): Eq. feq_Q=4 (third order), or Eq. feq_Q=3 (second order) for D2Q9
        const double xi = va * ut + vb * up;
        const double xi2 = xi * xi;
        bool bad = false;
        double h = scale2<-1>(xi2 - u2, bad);
        if (bad) h = mul_plain(0.5, xi2 - u2);
        const double second = 1.0 + xi + h;
        const double nw = n * p.wk[k];
        const double feq = (q == 3) ? nw * second : nw * (second + div_const(xi * (xi2 - u23), p.six));
        // velocity derivatives: K on k_theta at fixed k_phi, Ktilde on k_phi at fixed k_theta
        double kg = p.c.K[a * q] * gs[b][lane], ktg = p.c.Kt[b * q] * gs[q * a][lane];
        for (int m = 1; m < q; ++m) {
            kg += p.c.K[a * q + m] * gs[q * m + b][lane];
            ktg += p.c.Kt[b * q + m] * gs[q * a + m][lane];
        }
        const double force = rd.cotR * (p.vb2[b] * kg - va * ktg);
        const double adv_t = -div_const(fs - fn, rd.th);
        const double adv_p = -div_const(fe - fw, rd.ph);
        const double Lk = adv_t + adv_p - force - div_const(gk - feq, p.tau_div);

        double outv;
        if (p.stage == 1) outv = gk + p.dt * Lk;
        else if (p.stage == 2) outv = 0.75 * f0 + 0.25 * gk + p.dt_stage * Lk;
        else outv = div_const(f0, p.three) + 2.0 / 3.0 * gk + p.dt_stage * Lk;
        store_with_images(p.out, L, k, i, j, outv);
    }
}

// Initial populations: third-order Hermite projection of a Maxwellian at T
// (T = 1: the BGK equilibrium, Eq. feq_Q=4).
// (q = 3: the same projection to second order, Eq. feq_Q=3 at T = 1.)
__device__ __forceinline__ double finit(int q, double n, double wk, double va, double vb, double ut, double up,
                                        double T)
{
    const double xi = va * ut + vb * up;
    const double u2 = ut * ut + up * up;
    if (T == 1.0) {
        if (q == 3) return n * wk * (1.0 + xi + 0.5 * (xi * xi - u2));
        return n * wk * (1.0 + xi + 0.5 * (xi * xi - u2) + xi * (xi * xi - 3.0 * u2) / 6.0);
    }
    const double v2 = va * va + vb * vb;
    const double dT = T - 1.0;
    const double second = xi * xi - u2 + dT * (v2 - 2.0);
    if (q == 3) return n * wk * (1.0 + xi + 0.5 * second);
    const double third = xi * (xi * xi - 3.0 * u2) + 3.0 * dT * xi * (v2 - 4.0);
    return n * wk * (1.0 + xi + 0.5 * second + third / 6.0);
}

template <typename T>
__global__ void init_kernel(T *f, const Layout L, const double *rho, const double *ut, const double *up,
                            const double *temp, const VelD c, double rho_ref)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = blockIdx.y;
    if (j >= L.np) return;
    const size_t cell = (size_t)i * L.np + j;
    const double tt = temp ? temp[cell] : 1.0;
    const int q = c.q;
    for (int k = 0; k < q * q; ++k) {
        const int a = k / q, b = k % q;
        double v = finit(q, rho[cell], c.w[a] * c.w[b], c.v[a], c.v[b], ut[cell], up[cell], tt);
        if (rho_ref != 0.0) v -= c.w[a] * c.w[b] * rho_ref;
        f[L.at(k, i, j)] = (T)v;
    }
}

template <typename T>
__global__ void moments_kernel(const T *f, const Layout L, double *rho, double *ut, double *up, double *temp,
                               const VelD c, double rho_ref)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    const int i = blockIdx.y;
    if (j >= L.np) return;
    const int q = c.q, nk = q * q;
    double fk[NK];
    for (int k = 0; k < nk; ++k) {
        double v = (double)f[L.at(k, i, j)];
        if (rho_ref != 0.0) v = c.w[k / q] * c.w[k % q] * rho_ref + v;
        fk[k] = v;
    }
    double n = 0.0, jt = 0.0, jp = 0.0;
    for (int k = 0; k < nk; ++k) {
        n += fk[k];
        jt += fk[k] * c.v[k / q];
        jp += fk[k] * c.v[k % q];
    }
    const size_t cell = (size_t)i * L.np + j;
    const double u1 = jt / n, u2 = jp / n;
    rho[cell] = n;
    ut[cell] = u1;
    up[cell] = u2;
    if (temp) {
        double e = 0.0;
        for (int k = 0; k < nk; ++k) {
            const double ct = c.v[k / q] - u1, cp = c.v[k % q] - u2;
            e += fk[k] * (ct * ct + cp * cp);
        }
        temp[cell] = e / (2.0 * n);
    }
}

// Polar ring filter: mean over aligned blocks of b columns, summed in column order.
template <typename T>
__global__ void filter_kernel(T *f, const Layout L, const int *rows, const int *blocks, int nrows)
{
    const int rr = blockIdx.y;
    const int k = blockIdx.z;
    if (rr >= nrows) return;
    const int i = rows[rr];
    const int b = blocks[rr];
    const int nblk = L.np / b;
    for (int blk = blockIdx.x * blockDim.x + threadIdx.x; blk < nblk; blk += gridDim.x * blockDim.x) {
        const int j0 = blk * b;
        double s = 0.0;
        for (int m = 0; m < b; ++m) s += (double)f[L.at(k, i, j0 + m)];
        const T mean = (T)(s / (double)b);
        for (int m = 0; m < b; ++m) store_with_images(f, L, k, i, j0 + m, mean);
    }
}

}  // namespace

template <int S>
static void launch_faces(const StageD &p, cudaStream_t s)
{
    const Layout &L = p.L;
    const long long sp = (long long)((L.np + S) / S) * L.nt, stt = (long long)((L.nt + S) / S) * L.np;
    const int nb = (int)((sp + 127) / 128), nt = (int)((stt + 127) / 128);
    faces_f64_kernel<S><<<dim3(nb + nt, L.nk), 128, 0, s>>>(p, nb);
}

void launch_stage_f64(const StageD &p, cudaStream_t s)
{
    // Strip length of the face walk: 8 faces share their column forms best (64 FP64 operations a
    // face at S = 1, 59 at 8); a grid with fewer faces than about two warps of long strips per
    // scheduler (608 of them) takes shorter ones, since a lone warp's chain of FP64 operations
    // bounds the launch there.
    const long long faces = 2LL * p.L.nk * p.L.nt * p.L.np, lanes = 2LL * 608 * 32;
    if (faces >= 8 * lanes) launch_faces<8>(p, s);
    else if (faces >= 2 * lanes) launch_faces<2>(p, s);
    else launch_faces<1>(p, s);
    const long long cells = (long long)p.L.nt * p.L.np;
    cells_f64_kernel<<<(unsigned)((cells + 31) / 32), 32 * CELL_WARPS, 0, s>>>(p);
}

void launch_init_f64(double *f, const Layout &L, const double *rho, const double *ut, const double *up,
                     const double *T, const VelD &c, cudaStream_t s)
{
    dim3 grid((L.np + 127) / 128, L.nt);
    init_kernel<double><<<grid, 128, 0, s>>>(f, L, rho, ut, up, T, c, 0.0);
}

void launch_moments_f64(const double *f, const Layout &L, double *rho, double *ut, double *up, double *T,
                        const VelD &c, cudaStream_t s)
{
    dim3 grid((L.np + 127) / 128, L.nt);
    moments_kernel<double><<<grid, 128, 0, s>>>(f, L, rho, ut, up, T, c, 0.0);
}

void launch_filter_f64(double *f, const Layout &L, const int *rows, const int *blocks, int nrows, cudaStream_t s)
{
    if (nrows <= 0) return;
    dim3 grid((L.np / 2 + 127) / 128 + 1, nrows, L.nk);
    filter_kernel<double><<<grid, 128, 0, s>>>(f, L, rows, blocks, nrows);
}

}  // namespace vk
