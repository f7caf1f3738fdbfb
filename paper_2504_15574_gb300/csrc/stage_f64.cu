// stage_f64.cu -- FP64 kernels of the parity path (compiled with -fmad=false).
//
// One RK3 stage of arXiv 2504.15574 Sec. 3.7 in two kernels (faces, cells): moments
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
// instructions/s of ~610).  The forms below give the same bits with fewer of them: most products go
// to the integer pipe (f64_int.cuh; issue slots were 11 % used), scalings by powers of two become
// exponent additions, and reciprocal seeds come from the FP32 pipe.

// Interface flux v r of a stencil with values outside the fast forms' range (beyond [2^-400, 2^100)
// and not zero, or not finite) or with a quotient that a fast division missed, with the interface value r as
// the oracle writes it.
__device__ __noinline__ double weno5_plain(double a, double b, double c, double d, double e, double eps, double v)
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
    return v * ((w1 * p1 + w2 * p2 + w3 * p3) / (w1 + w2 + w3));
}

// Walks n consecutive WENO-5 faces from the values load(0), load(1), ... in upwind order: face f has the
// stencil a..e = values f .. f + 4 (c the upwind cell, d the downwind cell), in the oracle's
// expression order, and gives its flux to store(f, flux), v times the interface value (store_r: the
// value itself, for the Komissarov factor).  The forms of one column (13/12 times the squared second
// difference, and 5 y) are shared by the three candidate stencils centred on it, which changes no
// bit.  30 FP64 instructions a face, four of which check its quotients: with every value zero or in
// [2^-400, 2^100), differences are zero or multiples of the smallest ulp, so no product leaves the
// normal range.
template <class Load, class Store>
__device__ __forceinline__ void weno5_walk(int n, bool plain, double eps, double v, const DivC &six, Load load,
                                           Store store)
{
    double a = load(0), b = load(1), c = load(2), d = load(3), e = load(4);
    const double vb = a - scale2<1>(b) + c, vc = b - scale2<1>(c) + d;
    const double c1312 = 13.0 / 12.0;
    double k1 = mul_int_z(sq_int(vb), c1312), k2 = mul_int_z(sq_int(vc), c1312), c5 = mul_small<5>(c);
    // values still to be walked over that are outside the range keep the next faces on the plain form
    int out = 0;
    if (!(f64_within<400, 100>(a))) out = 1;
    if (!(f64_within<400, 100>(b))) out = 2;
    if (!(f64_within<400, 100>(c))) out = 3;
    if (!(f64_within<400, 100>(d))) out = 4;
#pragma unroll 1
    for (int f = 0; f < n; ++f) {
        const double next = load(min(f + 5, n + 3));
        if (!(f64_within<400, 100>(e))) out = 5;
        const double d3a = c - scale2<1>(d) + e;
        const double k3 = mul_int_z(sq_int(d3a), c1312);
        const double d5 = mul_small<5>(d), c3 = mul_small<3>(c);
        const double d1b = a - scale2<2>(b) + c3;
        const double d2b = b - d;
        const double d3b = c3 - scale2<2>(d) + e;
        const double s1 = add_pos(add_pos(k1, scale2<-2>(sq_int(d1b))), eps);
        const double s2 = add_pos(add_pos(k2, scale2<-2>(sq_int(d2b))), eps);
        const double s3 = add_pos(add_pos(k3, scale2<-2>(sq_int(d3b))), eps);
        bool miss = plain || out > 0;
        const double w1 = div_pos(0.1, mul_int(s1, s1), miss), w2 = div_pos(0.6, mul_int(s2, s2), miss),
                     w3 = div_pos(0.3, mul_int(s3, s3), miss);
        const double p1 = div_const_int(scale2<1>(a) - mul_small<7>(b) + mul_small<11>(c), six);
        const double p2 = div_const_int(c5 - b + scale2<1>(d), six);
        const double p3 = div_const_int(scale2<1>(c) + d5 - e, six);
        const double num = mul_int_z(p1, w1) + mul_int_z(p2, w2) + mul_int_z(p3, w3);
        const double r = div_pos(num, add_pos(add_pos(w1, w2), w3), miss);
        double flux = mul_int_zz(r, v);   // (v = 0: a D2Q9 population at rest along the axis)
        if (miss || !f64_within<500, 500>(num)) flux = weno5_plain(a, b, c, d, e, eps, v);
        store(f, flux);
        --out;
        a = b;
        b = c;
        c = d;
        d = e;
        e = next;
        k1 = k2;
        k2 = k3;
        c5 = d5;
    }
}

// The same for the upwind stencils of Eq. (fluxes_U1-3).
template <class Load, class Store>
__device__ __forceinline__ void upwind_walk(int n, int scheme, double v, const DivC &six, Load load, Store store)
{
    double b = load(1), c = load(2), d = load(3);
#pragma unroll 1
    for (int f = 0; f < n; ++f) {
        const double next = load(min(f + 4, n + 3));
        const double r = (scheme == VLBM_U1) ? c : (scheme == VLBM_U2) ? 1.5 * c - 0.5 * b
                                                                       : div_const(2.0 * d + 5.0 * c - b, six);
        store(f, v * r);
        b = c;
        c = d;
        d = next;
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
// faces (one launch: on small grids either alone leaves schedulers idle).  The walk is a rolled
// loop: unrolled, its 1,000 instructions a face would not stay in the instruction cache.  256 x 512: 298 us a
// launch, the FP64 pipe 76 % and the integer pipe 69 % busy.  (82 registers, five CTAs per SM: held to 80 or
// 72 for six or seven, a step took 1,479 and 1,422 us instead of 1,405.)
__global__ void __launch_bounds__(128) faces_f64_kernel(const StageD p, int nb_phi, int S)
{
    const Layout L = p.L;
    const int q = p.c.q, k = blockIdx.y;
    if ((int)blockIdx.x < nb_phi) {
        const int ns = (L.np + S) / S;   // strips of the np + 1 faces
        const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
        if (t >= (long long)ns * L.nt) return;
        const int i = (int)(t / ns), f0 = (int)(t - (long long)i * ns) * S, n = min(S, L.np + 1 - f0);
        const double vb = p.c.v[k % q];
        const int dir = vb > 0.0 ? 1 : -1;
        // value m is column f0 - 3 + m, or (backwards) column f0 + n + 1 - m
        const double *g = p.in + L.at(k, i, dir > 0 ? f0 - 3 : f0 + n + 1);
        double *out = p.Fp + ((size_t)k * L.nt + i) * (L.np + 1) + (dir > 0 ? f0 : f0 + n - 1);
        auto load = [&](int m) { return g[dir * m]; };
        auto store = [&](int f, double flux) { out[dir * f] = flux; };
        if (p.scheme == VLBM_WENO5) weno5_walk(n, p.plain, p.eps, vb, p.six, load, store);
        else upwind_walk(n, p.scheme, vb, p.six, load, store);
        return;
    }
    const int ns = (L.nt + S) / S;
    const long long t = (long long)(blockIdx.x - nb_phi) * blockDim.x + threadIdx.x;
    if (t >= (long long)ns * L.np) return;
    const int st = (int)(t / L.np), j = (int)(t - (long long)st * L.np), f0 = st * S, n = min(S, L.nt + 1 - f0);
    const double va = p.c.v[k / q];
    const int dir = va > 0.0 ? 1 : -1;
    const int r0 = dir > 0 ? f0 - 3 : f0 + n + 1;
    auto load = [&](int m) {
        const int row = r0 + dir * m;
        const double x = p.in[L.at(k, row, j)];
        return p.komissarov ? x : p.sin_ext[row + GR] * x;
    };
    auto store = [&](int f, double flux) {
        const int fi = dir > 0 ? f0 + f : f0 + n - 1 - f;
        p.Ft[((size_t)k * (L.nt + 1) + fi) * L.np + j] = flux;
        if (p.pole) {
            if (fi == 0) p.pole[(size_t)k * L.np + j] = flux;
            if (fi == L.nt) p.pole[((size_t)NK + k) * L.np + j] = flux;
        }
    };
    // (Komissarov: the walk gives the value itself, the flux is v_theta sin(theta_fi) times it)
    auto store_kom = [&](int f, double r) {
        const int fi = dir > 0 ? f0 + f : f0 + n - 1 - f;
        store(f, va * p.sin_f[fi] * r);
    };
    if (p.scheme == VLBM_WENO5) {
        if (p.komissarov) weno5_walk(n, p.plain, p.eps, 1.0, p.six, load, store_kom);
        else weno5_walk(n, p.plain, p.eps, va, p.six, load, store);
    } else if (p.komissarov) {
        upwind_walk(n, p.scheme, 1.0, p.six, load, store_kom);
    } else {
        upwind_walk(n, p.scheme, va, p.six, load, store);
    }
}

// One population's update of one cell.  FAST: products on the integer pipe, for populations that are
// zero or in [2^-40, 2^100) and a positive density (then every product here is zero or normal).  PLAIN: real
// divisions, for a run whose constants are no numbers of ordinary size (in a kernel of its own: the code of
// these divisions beside the other forms cost 2.5 %, 256 x 512).
template <bool FAST, bool PLAIN, int CELLS>
__device__ __forceinline__ void cell_update(const StageD &p, const Layout &L, const RowD &rd,
                                            const double (*gs)[CELLS], int lane, int i, int j, int k, double n,
                                            double ut, double up, double u2, double u23)
{
    auto mul = [](double a, double b) { return FAST ? mul_int_zz(a, b) : a * b; };
    auto div = [](double a, const DivC &d) { return PLAIN ? a / d.d : div_const(a, d); };   // (a of any size)
    auto divc = [=](double a, const DivC &d) { return FAST ? div_const_int(a, d) : div(a, d); };
    const int q = p.c.q, a = k / q, b = k % q;
    const double va = p.c.v[a], vb = p.c.v[b];
    const double gk = gs[k][lane];
    // loaded ahead of the arithmetic
    const double fn = p.Ft[((size_t)k * (L.nt + 1) + i) * L.np + j];
    const double fs = p.Ft[((size_t)k * (L.nt + 1) + i + 1) * L.np + j];
    const double fw = p.Fp[((size_t)k * L.nt + i) * (L.np + 1) + j];
    const double fe = p.Fp[((size_t)k * L.nt + i) * (L.np + 1) + j + 1];
    const double f0 = (p.stage == 1) ? 0.0 : p.fold[L.at(k, i, j)];
    // equilibrium (T0 = 1): Eq. feq_Q=4 (third order), or Eq. feq_Q=3 (second order) for D2Q9
    const double xi = mul(va, ut) + mul(vb, up);
    const double xi2 = mul(xi, xi);
    const double half = xi2 - u2;
    const double second = 1.0 + xi + (FAST ? scale2<-1>(half) : 0.5 * half);
    const double nw = mul(n, p.wk[k]);
    const double feq = (q == 3) ? mul(nw, second) : mul(nw, second + divc(mul(xi, xi2 - u23), p.six));
    // velocity derivatives: K on k_theta at fixed k_phi, Ktilde on k_phi at fixed k_theta
    double kg = mul(p.c.K[a * q], gs[b][lane]), ktg = mul(p.c.Kt[b * q], gs[q * a][lane]);
#pragma unroll 1
    for (int m = 1; m < q; ++m) {
        kg += mul(p.c.K[a * q + m], gs[q * m + b][lane]);
        ktg += mul(p.c.Kt[b * q + m], gs[q * a + m][lane]);
    }
    const double force = mul(rd.cotR, mul(p.vb2[b], kg) - mul(va, ktg));
    const double adv_t = -div(fs - fn, rd.th);
    const double adv_p = -div(fe - fw, rd.ph);
    const double Lk = adv_t + adv_p - force - divc(gk - feq, p.tau_div);

    double outv;
    if (p.stage == 1) outv = gk + p.dt * Lk;
    else if (p.stage == 2) outv = 0.75 * f0 + (FAST ? scale2<-2>(gk) : 0.25 * gk) + p.dt_stage * Lk;
    else outv = div(f0, p.three) + mul(2.0 / 3.0, gk) + p.dt_stage * Lk;
    store_with_images(p.out, L, k, i, j, outv);
}

// Pole mass-flux budget of one step, by the threads of one CTA: budget += dt (m1/6 + m2/6 + 2 m3/3),
// m_s = -R dph sum_{k,j} (F_south - F_north) of stage s.
__device__ __forceinline__ void pole_budget_f64(const StageD &p)
{
    constexpr int NT = 256;
    __shared__ double red[3][NT];
    const int np = p.L.np;
    const size_t per = (size_t)NK * np;
    double acc[3] = {0, 0, 0};
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        const double *pn = p.pole_all + (size_t)s * 2 * per, *ps = pn + per;
#pragma unroll 4
        for (size_t x = threadIdx.x; x < per; x += NT) acc[s] += ps[x] - pn[x];
    }
    for (int s = 0; s < 3; ++s) red[s][threadIdx.x] = acc[s];
    __syncthreads();
    for (int w = NT / 2; w > 0; w >>= 1) {
        if ((int)threadIdx.x < w)
            for (int s = 0; s < 3; ++s) red[s][threadIdx.x] += red[s][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double m1 = -p.R * p.dph * red[0][0], m2 = -p.R * p.dph * red[1][0], m3 = -p.R * p.dph * red[2][0];
        *p.budget += p.dt * (m1 / 6.0 + m2 / 6.0 + 2.0 * m3 / 3.0);
    }
}

// Cells of one stage: moments, equilibrium, force, BGK, the flux differences of the interface
// fluxes above and the stage combination, in the oracle's operation order.  A CTA of 256 threads
// takes CELLS consecutive cells (32 or 16): thread = cell and slot.  Slots 0, 1, 2 first form the
// moments (the sums run over k in order, so they are chains), 1 and 2 then the velocities; then
// each slot updates the populations slot, slot + 256 / CELLS, ....  One thread per cell, the earlier
// form, left a 32 x 64 grid with 64 warps of 1,700 serial FP64 operations (71 us a launch).  Bound
// on large grids: the FP64 pipe (37 instructions per population, from 105).  16 cells per CTA where
// 32 would leave SMs without one.  In stage 3 one more CTA adds the step's pole budget (a launch
// of its own was 3-10 us a step).  256 x 512: 169 us a launch, the FP64 pipe 77 % busy.
template <int CELLS, bool PLAIN>
__global__ void __launch_bounds__(256) cells_f64_kernel(const StageD p, int nblocks)
{
    constexpr int SLOTS = 256 / CELLS;
    __shared__ double gs[NK][CELLS], mom[3][CELLS], vel[4][CELLS];
    if ((int)blockIdx.x == nblocks) {
        pole_budget_f64(p);
        return;
    }
    const Layout L = p.L;
    const int c = threadIdx.x % CELLS, slot = threadIdx.x / CELLS;
    const int q = p.c.q, nk = q * q;
    const long long cells = (long long)L.nt * L.np;
    const long long cell = (long long)blockIdx.x * CELLS + c;
    const bool in = cell < cells;
    const int i = in ? (int)(cell / L.np) : 0, j = in ? (int)(cell - (long long)i * L.np) : 0;
    bool out = PLAIN;
    for (int k = slot; k < nk; k += SLOTS) {
        const double g = p.in[L.at(k, i, j)];
        out |= !f64_within<40, 100>(g);
        gs[k][c] = g;
    }
    const bool plain = __syncthreads_or(out);
    if (slot < 3) {
        double m = 0.0;
        for (int k = 0; k < nk; ++k) {
            const double g = gs[k][c], v = slot == 0 ? 1.0 : p.c.v[slot == 1 ? k / q : k % q];
            m += plain ? g * v : mul_int_zz(g, v);
        }
        mom[slot][c] = m;
    }
    __syncthreads();
    // (a density that is not positive takes the plain forms: its velocities may be of any size)
    const double n = mom[0][c];
    const bool slow = plain || !(n > 0.0) || !f64_within<110, 110>(n);
    if (slot == 1 || slot == 2) {
        const double m = mom[slot][c];
        bool miss = slow;
        double u = div_pos(m, n, miss);
        if (miss) u = f64_zero(m) && !slow ? m : m / n;
        vel[slot - 1][c] = u;
    }
    __syncthreads();
    if (slot == 0) {
        const double ut = vel[0][c], up = vel[1][c];
        const double u2 = ut * ut + up * up;
        vel[2][c] = u2;
        vel[3][c] = 3.0 * u2;
    }
    __syncthreads();
    if (!in) return;
    const double ut = vel[0][c], up = vel[1][c], u2 = vel[2][c], u23 = vel[3][c];
    const RowD rd = p.row[i];
#pragma unroll 1
    for (int k = slot; k < nk; k += SLOTS) {
        if (PLAIN || slow) cell_update<false, PLAIN, CELLS>(p, L, rd, gs, c, i, j, k, n, ut, up, u2, u23);
        else cell_update<true, false, CELLS>(p, L, rd, gs, c, i, j, k, n, ut, up, u2, u23);
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

void launch_stage_f64(const StageD &p, cudaStream_t s)
{
    // Strip length of the face walk: long strips share their column forms best (the first face of a
    // strip forms two columns more); a grid with fewer faces than about two warps of long strips per
    // scheduler (608 of them) takes shorter ones, since a lone warp's chain of operations bounds
    // the launch there.
    const Layout &L = p.L;
    const long long faces = 2LL * L.nk * L.nt * L.np, lanes = 2LL * 608 * 32;
    const int S = faces >= 16 * lanes ? 16 : faces >= 8 * lanes ? 8 : faces >= 4 * lanes ? 4 : faces >= 2 * lanes ? 2 : 1;
    const long long sp = (long long)((L.np + S) / S) * L.nt, stt = (long long)((L.nt + S) / S) * L.np;
    const int nb = (int)((sp + 127) / 128), nt = (int)((stt + 127) / 128);
    faces_f64_kernel<<<dim3(nb + nt, L.nk), 128, 0, s>>>(p, nb, S);
    const long long cells = (long long)p.L.nt * p.L.np;
    const int extra = (p.stage == 3 && p.budget) ? 1 : 0;
    auto launch = [&](auto *kernel, int per) {
        const unsigned nb = (unsigned)((cells + per - 1) / per);
        kernel<<<nb + extra, 256, 0, s>>>(p, (int)nb);
    };
    if (p.plain) launch(cells_f64_kernel<32, true>, 32);
    else if (cells <= 32LL * 152 * 2) launch(cells_f64_kernel<16, false>, 16);   // 32: fewer than two CTAs per SM
    else launch(cells_f64_kernel<32, false>, 32);
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
