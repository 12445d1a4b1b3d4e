// step_kernels.cu -- pointwise kernels of the quasi-static projection step
// (section 3.3): stress predictor with the STZ rate, effective temperature,
// right-hand side of the projection system, stress correction (alone, or
// fused with the next step's predictor), wall fill, and the optional stress
// advection; the explicit method of section 3.2 (ENO advection, Eq. 33); and
// the adjoint kernels of the reverse mode.
//
// Cell arrays (nz, ny, nx); stress (6, nz, ny, nx) in the order xx, yy, zz,
// yz, xz, xy; corner arrays (3, nz+1, ny, nx).  x and y are periodic.
#include "qsmg_impl.h"

namespace qsmg {
namespace {

// 32 x 8 threads over (i, j), grid.z over planes: no flat-index division
constexpr int BX = 32, BY = 8;
const dim3 kBlock(BX, BY);
inline dim3 cell_grid(int nx, int ny, int nplanes) {
    return dim3((nx + BX - 1) / BX, (ny + BY - 1) / BY, nplanes);
}

__device__ __forceinline__ bool cell_ijk(int nx, int ny, int &i, int &j, int &k) {
    i = blockIdx.x * BX + threadIdx.x;
    j = blockIdx.y * BY + threadIdx.y;
    k = blockIdx.z;
    return i < nx && j < ny;
}

// Launch of a kernel that marches columns in z: blocks of `threads` over the
// columns of a plane in linear order (the FP64 pipe is paid for by the warp
// instruction, so lanes are packed whatever nx is), grid.y over chunks of
// `chunk` planes.  A chunk repeats one plane's partial sums, so chunks are as
// long as leaves the chip about four blocks an SM; then blocks shrink.
struct March {
    dim3 grid;
    int threads, chunk;
};
inline March march(long columns, int planes) {
    March m;
    m.threads = 128;
    m.chunk = 16;
    auto blocks = [&] {
        return ((columns + m.threads - 1) / m.threads) * ((planes + m.chunk - 1) / m.chunk);
    };
    while (m.chunk > 1 && blocks() < 608) m.chunk /= 2;
    while (m.threads > 32 && blocks() < 608) m.threads /= 2;
    m.grid = dim3((unsigned)((columns + m.threads - 1) / m.threads),
                  (planes + m.chunk - 1) / m.chunk);
    return m;
}

struct StzConst {
    double half_eDT_over_tau0;  // exp(-Delta/(kB T)) / (2 tau0)
    double beta;                // Omega eps0 / (kB T)
    double sY, ez_K;
};

__host__ StzConst stz_const(const StepParams &p) {
    StzConst c;
    c.half_eDT_over_tau0 = 0.5 * exp(-p.Delta_K / p.T) / p.tau0;
    c.beta = p.Omega * p.eps0 / (p.kB * p.T);
    c.sY = p.sY;
    c.ez_K = p.ez_K;
    return c;
}

// exp(x + y) + exp(y - x), x > 0.  FP64 runs at 1/64 of the FP32 rate, and for
// x > 13.8 (at Table 1's constants every cell above yield) the second term is
// below exp(-27.6) = 1.1e-12 of the first: there its ratio exp(-2 x) is taken in
// FP32 (relative error 4e-6 at most: the rounding of 2 x <= 87, expf's own),
// which changes the sum by less than 0.02 units of its last place.  Errors of
// 2^20 sums against quad precision, x in 13.85..25, y in -36..-30: 3.238339 units
// rms and 16.92 at most, from the rounding of x + y; with both terms in FP64
// 3.238348 and 16.92.
__device__ __forceinline__ double exp_pair(double x, double y) {
    const double ep = exp(x + y);
    const float x2 = -2.0f * (float)x;
    if (x2 < -27.6f) {
        const float r = expf(x2);
        return r > 0.0f ? fma(ep, (double)r, ep) : ep;  // (no inf * 0)
    }
    return ep + exp(y - x);
}

// athermal STZ rate magnitude, Eqs. (20)-(22):
//   D = exp(-e_z/(kB chi)) exp(-Delta/(kB T)) cosh(Omega eps0 sbar/(kB T)) (1 - s_Y/sbar) / tau0,
// 0 at or below yield (or for chi <= 0).  The product exp(-e_z/chi) cosh(beta
// sbar) is taken as (exp(beta sbar - e_z/chi) + exp(-beta sbar - e_z/chi)) / 2
// and 1/sbar is computed once by the caller.
__device__ __forceinline__ double stz_rate(const StzConst &c, double sbar, double inv_sbar,
                                           double chi) {
    if (!(sbar > c.sY) || !(chi > 0.0)) return 0.0;
    const double y = -c.ez_K / chi, x = c.beta * sbar;
    return exp_pair(x, y) * c.half_eDT_over_tau0 * (1.0 - c.sY * inv_sbar);
}

// 1/2 sigma0 : sigma0, given the mean stress m
__device__ __forceinline__ double j2_of(const double s[6], double m) {
    const double d0 = s[0] - m, d1 = s[1] - m, d2 = s[2] - m;
    return 0.5 * (d0 * d0 + d1 * d1 + d2 * d2) + (s[3] * s[3] + s[4] * s[4] + s[5] * s[5]);
}

// sbar = sqrt(q) and its reciprocal (0 for q = 0) from the reciprocal square
// root, each corrected once: equal to sqrt(q) and 1 / sqrt(q) in 3 million q from
// 2^-1000 to 2^1000, for about half their FP64 instructions
__device__ __forceinline__ void sbar_inv(double q, double &sb, double &inv) {
    const int hi = __double2hiint(q);
    if (hi >= 0x00100000 && hi < 0x7ff00000) {  // positive, normal and finite
        inv = rsqrt(q);
        sb = q * inv;
        sb = fma(fma(-sb, sb, q), 0.5 * inv, sb);
        inv = fma(fma(-sb, inv, 1.0), inv, inv);
    } else {
        sb = sqrt(q);
        inv = sb > 0.0 ? 1.0 / sb : 0.0;
    }
}

// sbar with sbar^2 = 1/2 sigma0 : sigma0
__device__ __forceinline__ double sbar_of(const double s[6]) {
    return sqrt(j2_of(s, (s[0] + s[1] + s[2]) * (1.0 / 3.0)));
}

// Eq. (31): G[a][b] = d v_a / d x_b at the centre of cell (i, j, k), from its
// 8 corners; each derivative averages the 4 edge differences along its axis.
// Computed for a column of cells marching up in z: each corner plane's
// contributions -- x-differences, y-differences and the sum over the 2 x 2
// corners around the column -- are formed once and shared by the cells
// below and above the plane.  The x- and y-differences come from the two
// diagonals (their sum and difference): 39 FP64 operations a cell with the
// scaling, instead of 72.
struct GradPlane {
    double X[3], Y[3], Z[3];
};

__device__ __forceinline__ GradPlane grad_plane(const double *__restrict__ v, long cs, long off,
                                                long r0, long r1, int i, int i1) {
    GradPlane P;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const double *g = v + a * cs + off;
        const double c00 = g[r0 + i], c10 = g[r0 + i1], c01 = g[r1 + i], c11 = g[r1 + i1];
        const double d1 = c11 - c00, d2 = c10 - c01;
        P.X[a] = d1 + d2;
        P.Y[a] = d1 - d2;
        P.Z[a] = (c00 + c10) + (c01 + c11);
    }
    return P;
}

// gradient of the cell between corner planes lo (k) and hi (k+1)
__device__ __forceinline__ void grad_cell(const GradPlane &lo, const GradPlane &hi, double inv4h,
                                          double G[3][3]) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
        G[a][0] = (lo.X[a] + hi.X[a]) * inv4h;
        G[a][1] = (lo.Y[a] + hi.Y[a]) * inv4h;
        G[a][2] = (hi.Z[a] - lo.Z[a]) * inv4h;
    }
}

// column (i, j) of a chunk of cells; false if outside the grid
struct CellColumn {
    int i, j, i1, k0, k1;
    long pl, cs, r0, r1;
};
__device__ __forceinline__ bool cell_column(int nx, int ny, int nz, int chunk, CellColumn &C) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    C.j = m / nx;
    C.i = m - C.j * nx;
    if (C.j >= ny) return false;
    C.i1 = C.i + 1 < nx ? C.i + 1 : 0;
    const int j1 = C.j + 1 < ny ? C.j + 1 : 0;
    C.k0 = blockIdx.y * chunk;
    C.k1 = C.k0 + chunk < nz ? C.k0 + chunk : nz;
    C.pl = (long)nx * ny;
    C.cs = (long)(nz + 1) * C.pl;
    C.r0 = (long)C.j * nx;
    C.r1 = (long)j1 * nx;
    return true;
}

// constants of the predictor and the corrector: G of a cell enters both only
// as dt G, so the scale of the gradient carries the time step
struct CellConst {
    double dt4h, dt2h;  // dt / (4 h), dt / (2 h)
    double lam, mu, mu2, mu2dt;
};
CellConst cell_const(const StepParams &p) {
    return CellConst{p.dt * (0.25 / p.h), p.dt * (0.5 / p.h), p.lam, p.mu, 2.0 * p.mu, 2.0 * p.mu * p.dt};
}

// Eq. (27) at cell q: sigma* = sigma + dt (L sigma + sigma L^T - tr(L) sigma
// - 2 mu D^pl sigma0 / sbar) from dt times the cell-centre gradient of v^n (G)
// and the cell's sigma^n (s6) and chi^n; also stores D^pl and sbar.  Its
// increment (objective_increment): with
// P = 2 mu dt D^pl / sbar and H = dt L - (tr(dt L) + P) / 2 I the update is
// sigma + (H sigma + sigma H^T + P m I), m the mean stress: 49 instructions
// where the terms one by one take 68.  The increment is summed before it is
// added to sigma, which rounds the result once.
__device__ __forceinline__ void objective_increment(const CellConst &w, const StzConst &c,
                                                    const double (&G)[3][3],
                                                    const double (&s6)[6], double chi_q,
                                                    double (&inc)[6], double &D, double &sb) {
    const double S[3][3] = {{s6[0], s6[5], s6[4]}, {s6[5], s6[1], s6[3]}, {s6[4], s6[3], s6[2]}};
    const double m = (s6[0] + s6[1] + s6[2]) * (1.0 / 3.0);
    double inv_sb;
    sbar_inv(j2_of(s6, m), sb, inv_sb);
    D = stz_rate(c, sb, inv_sb, chi_q);
    const double P = w.mu2dt * D * inv_sb;
    const double tr = 0.5 * (G[0][0] + G[1][1] + G[2][2] + P);
    double H[3][3];
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) H[a][b] = a == b ? G[a][b] - tr : G[a][b];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        double t = H[a][0] * S[0][a];
        t = fma(H[a][1], S[1][a], t);
        t = fma(H[a][2], S[2][a], t);
        inc[a] = fma(2.0, t, P * m);
    }
    const int ia[3] = {1, 0, 0}, ib[3] = {2, 2, 1};
#pragma unroll
    for (int n = 0; n < 3; n++) {
        const int a = ia[n], b = ib[n];
        double t = H[a][0] * S[0][b];
#pragma unroll
        for (int e = 0; e < 3; e++) {
            if (e > 0) t = fma(H[a][e], S[e][b], t);
            t = fma(S[a][e], H[b][e], t);
        }
        inc[3 + n] = t;
    }
}
__device__ __forceinline__ void predict_cell(const CellConst &w, const StzConst &c,
                                             const double (&G)[3][3], const double (&s6)[6],
                                             double chi_q, long q, long nc,
                                             double *__restrict__ sig_star,
                                             double *__restrict__ dpl,
                                             double *__restrict__ sbar_out) {
    double inc[6], D, sb;
    objective_increment(w, c, G, s6, chi_q, inc, D, sb);
#pragma unroll
    for (int n = 0; n < 6; n++) sig_star[n * nc + q] = s6[n] + inc[n];
    dpl[q] = D;
    sbar_out[q] = sb;
}

// Eq. (29) at one cell: sigma = sigma* + dt (lam tr(D) I + 2 mu D), D = sym G
// (G: dt times the gradient)
__device__ __forceinline__ void correct_cell(const CellConst &w, const double (&G)[3][3],
                                             const double (&ss)[6], double (&s6)[6]) {
    const double lt = w.lam * (G[0][0] + G[1][1] + G[2][2]);
#pragma unroll
    for (int a = 0; a < 3; a++) s6[a] = fma(w.mu2, G[a][a], ss[a] + lt);
    s6[3] = fma(w.mu, G[1][2] + G[2][1], ss[3]);
    s6[4] = fma(w.mu, G[0][2] + G[2][0], ss[4]);
    s6[5] = fma(w.mu, G[0][1] + G[1][0], ss[5]);
}

// Eq. (27) over a column chunk of cells.  FP64 instructions bound it (its 144
// bytes a cell take 0.36 ms at 256^3): 4.36 ms there, 5.94 with the gradient
// unshifted, both exponentials in FP64 and 32 x 8 thread blocks.
__global__ void __launch_bounds__(128)
    k_stress_predict(StepParams p, CellConst w, StzConst c, int chunk, const double *__restrict__ v,
                     const double *__restrict__ sig, const double *__restrict__ chi,
                     double *__restrict__ sig_star, double *__restrict__ dpl,
                     double *__restrict__ sbar_out, long nc) {
    CellColumn C;
    if (!cell_column(p.nx, p.ny, p.nz, chunk, C)) return;
    GradPlane lo = grad_plane(v, C.cs, C.k0 * C.pl, C.r0, C.r1, C.i, C.i1);
    for (int k = C.k0; k < C.k1; k++) {
        const GradPlane hi = grad_plane(v, C.cs, (k + 1) * C.pl, C.r0, C.r1, C.i, C.i1);
        const long q = k * C.pl + C.r0 + C.i;
        double G[3][3];
        grad_cell(lo, hi, w.dt4h, G);
        lo = hi;
        double s6[6];
#pragma unroll
        for (int a = 0; a < 6; a++) s6[a] = sig[a * nc + q];
        predict_cell(w, c, G, s6, chi[q], q, nc, sig_star, dpl, sbar_out);
    }
}

// Eq. (26): chi' = chi + (dt/c0)[ (2 D sbar / s_Y)(chi_inf - chi) + l^2 div(D grad chi) ]
// diffusion: sum over the 6 faces of (D_P + D_N)/2 (chi_N - chi_P) / h^2;
// z ghost cells carry linearly extrapolated sigma and chi, and their D is
// the STZ rate of those extrapolated values
// A thread marches a column in z: a z face's flux serves the cells below and
// above it.  The products of constants are formed on the host -- three FP64
// divisions a cell were half of this kernel: 0.72 ms at 256^3, 1.73 before.
struct ChiConst {
    double grow, diff;  // 2 dt / (c0 s_Y);  dt l^2 / (2 c0 h^2)
    double chi_inf;
};
__global__ void __launch_bounds__(128)
    k_chi_update(StepParams p, StzConst c, ChiConst w, int chunk, const double *__restrict__ sig,
                 const double *__restrict__ chi, const double *__restrict__ dpl,
                 const double *__restrict__ sbar, double *__restrict__ chi_new, long nc) {
    CellColumn C;
    if (!cell_column(p.nx, p.ny, p.nz, chunk, C)) return;
    const int nz = p.nz;
    const long pl = C.pl;
    const long rm = (long)(C.j ? C.j - 1 : p.ny - 1) * p.nx + C.i, rp = C.r1 + C.i;
    const long xm = C.r0 + (C.i ? C.i - 1 : p.nx - 1), xp = C.r0 + C.i1;
    // (D_P + D_N) (chi_N - chi_P) of the z face on side +-1 of a wall cell q:
    // the ghost's values are 2 * (this layer) - (next layer inward)
    auto wall_flux = [&](long q, long in, double cP, double DP) {
        double s6[6];
#pragma unroll
        for (int a = 0; a < 6; a++) s6[a] = 2.0 * sig[a * nc + q] - sig[a * nc + q + in];
        const double cn = 2.0 * cP - chi[q + in], sbn = sbar_of(s6);
        return (DP + stz_rate(c, sbn, sbn > 0.0 ? 1.0 / sbn : 0.0, cn)) * (cn - cP);
    };
    long q = C.k0 * pl + C.r0 + C.i;
    double c0 = chi[q], D0 = dpl[q];
    // flux across the face below the current cell, from the cell below
    double below = C.k0 == 0 ? -wall_flux(q, pl, c0, D0)
                             : (D0 + dpl[q - pl]) * (c0 - chi[q - pl]);
    for (int k = C.k0; k < C.k1; k++, q += pl) {
        const long kp = k * pl;
        double above, c1 = 0.0, D1 = 0.0;
        if (k + 1 < nz) {
            c1 = chi[q + pl];
            D1 = dpl[q + pl];
            above = (D0 + D1) * (c1 - c0);
        } else {
            above = wall_flux(q, -pl, c0, D0);
        }
        double acc = above - below;
        const long nb[4] = {xp, xm, rp, rm};
#pragma unroll
        for (int n = 0; n < 4; n++) acc = fma(D0 + dpl[kp + nb[n]], chi[kp + nb[n]] - c0, acc);
        const double growth = D0 * sbar[q] * (w.chi_inf - c0);
        chi_new[q] = c0 + fma(w.grow, growth, w.diff * acc);
        below = above;
        c0 = c1;
        D0 = D1;
    }
}

// b = (h^2/(mu dt)) div sigma* at interior corners; the corner derivative is
// Eq. (31) shifted by half a cell: cells (i-1..i, j-1..j, k-1..k).
// Corner divergence, marching up one (i, j) corner column: each cell layer's
// contributions -- the x-differences of sigma_a0 plus the y-differences of
// sigma_a1, and the layer sum of sigma_a2 over the 2 x 2 cells around the
// column -- are formed once and shared by the corners below and above the
// layer (FP64 is add-bound here: 40 instructions a corner instead of 72);
// 1.33 ms at 256^3, 1.49 with one z chunk length and 32 x 8 blocks
struct DivLayer {
    double XY[3], Z[3];
};

// over the 2 x 2 cells f[y][x]
__device__ __forceinline__ double sum4(const double (&f)[2][2]) {
    return (f[0][0] + f[0][1]) + (f[1][0] + f[1][1]);
}
__device__ __forceinline__ double dif_x(const double (&f)[2][2]) {
    return (f[0][1] - f[0][0]) + (f[1][1] - f[1][0]);
}
__device__ __forceinline__ double dif_y(const double (&f)[2][2]) {
    return (f[1][0] - f[0][0]) + (f[1][1] - f[0][1]);
}

// the layer's x-y part, and the 2 x 2 cells of the components whose z
// derivative enters (xz, yz, zz)
__device__ __forceinline__ void div_parts(const double *__restrict__ ss, long nc, long base,
                                          long rj0, long rj1, int im, int i, double (&xy)[3],
                                          double (&fz)[3][2][2]) {
    auto cells = [&](int n, double (&f)[2][2]) {
        const double *g = ss + n * nc + base;
        f[0][0] = g[rj0 + im];
        f[0][1] = g[rj0 + i];
        f[1][0] = g[rj1 + im];
        f[1][1] = g[rj1 + i];
    };
    double f[2][2];
    cells(5, f);  // xy: its x- and y-differences from the two diagonals
    const double d1 = f[1][1] - f[0][0], d2 = f[0][1] - f[1][0];
    xy[1] = d1 + d2;
    xy[0] = d1 - d2;
    cells(0, f);
    xy[0] += dif_x(f);
    cells(1, f);
    xy[1] += dif_y(f);
    cells(4, fz[0]);
    cells(3, fz[1]);
    cells(2, fz[2]);
    xy[2] = dif_x(fz[0]) + dif_y(fz[1]);
}

__device__ __forceinline__ DivLayer div_layer(const double *__restrict__ ss, long nc, long base,
                                              long rj0, long rj1, int im, int i) {
    DivLayer L;
    double f[3][2][2];
    div_parts(ss, nc, base, rj0, rj1, im, i, L.XY, f);
#pragma unroll
    for (int a = 0; a < 3; a++) L.Z[a] = sum4(f[a]);
    return L;
}

// (its wall planes, not part of the system, are zeroed)
__global__ void __launch_bounds__(128)
    k_div_rhs(StepParams p, int chunk, const double *__restrict__ ss, double *__restrict__ b,
              double scale) {
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int m = blockIdx.x * blockDim.x + threadIdx.x, j = m / nx, i = m - j * nx;
    if (j >= ny) return;
    const int k0 = 1 + blockIdx.y * chunk;
    const int k1 = k0 + chunk < nz ? k0 + chunk : nz;  // corners k0 .. k1-1
    const int im = i ? i - 1 : nx - 1, jm = j ? j - 1 : ny - 1;
    const long nc = (long)nx * ny * nz, pl = (long)nx * ny;
    const long rj0 = (long)jm * nx, rj1 = (long)j * nx;
    const long cs = (long)(nz + 1) * pl;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        if (k0 == 1) b[a * cs + m] = 0.0;
        if (k1 == nz) b[a * cs + nz * pl + m] = 0.0;
    }
    DivLayer lo = div_layer(ss, nc, (long)(k0 - 1) * pl, rj0, rj1, im, i);
    for (int k = k0; k < k1; k++) {
        const DivLayer hi = div_layer(ss, nc, (long)k * pl, rj0, rj1, im, i);
        const long node = (long)k * pl + m;
#pragma unroll
        for (int a = 0; a < 3; a++)
            b[a * cs + node] = scale * ((lo.XY[a] + hi.XY[a]) + (hi.Z[a] - lo.Z[a]));
        lo = hi;
    }
}

// Eq. (29) over a column chunk of cells; chi_dst <- chi_src on the way
// (the step's new chi, when chi_dst is not null)
__global__ void __launch_bounds__(128)
    k_stress_correct(StepParams p, CellConst w, int chunk, const double *__restrict__ v,
                     const double *__restrict__ ss, double *__restrict__ sig,
                     const double *__restrict__ chi_src, double *__restrict__ chi_dst, long nc) {
    CellColumn C;
    if (!cell_column(p.nx, p.ny, p.nz, chunk, C)) return;
    GradPlane lo = grad_plane(v, C.cs, C.k0 * C.pl, C.r0, C.r1, C.i, C.i1);
    for (int k = C.k0; k < C.k1; k++) {
        const GradPlane hi = grad_plane(v, C.cs, (k + 1) * C.pl, C.r0, C.r1, C.i, C.i1);
        const long q = k * C.pl + C.r0 + C.i;
        double G[3][3];
        grad_cell(lo, hi, w.dt4h, G);
        lo = hi;
        double s6[6], ss6[6];
#pragma unroll
        for (int a = 0; a < 6; a++) ss6[a] = ss[a * nc + q];
        correct_cell(w, G, ss6, s6);
#pragma unroll
        for (int a = 0; a < 6; a++) sig[a * nc + q] = s6[a];
        if (chi_dst) chi_dst[q] = chi_src[q];
    }
}

// Eq. (29) of step n and Eq. (27) of step n+1 in one pass: both use the
// gradient of the same velocity v^{n+1}, so it is formed once, and sigma^{n+1}
// goes from the correction straight into the predictor without a round trip
// through memory.  sig_star holds sigma* of step n on entry and of step n+1
// on return (each cell reads and writes only its own entries); sig receives
// sigma^{n+1}, chi_dst the step's new chi (chi_src).
__global__ void __launch_bounds__(128)
    k_correct_predict(StepParams p, CellConst w, StzConst c, int chunk,
                      const double *__restrict__ v, double *__restrict__ sig_star,
                      double *__restrict__ sig, const double *__restrict__ chi_src,
                      double *__restrict__ chi_dst, double *__restrict__ dpl,
                      double *__restrict__ sbar_out, long nc) {
    CellColumn C;
    if (!cell_column(p.nx, p.ny, p.nz, chunk, C)) return;
    GradPlane lo = grad_plane(v, C.cs, C.k0 * C.pl, C.r0, C.r1, C.i, C.i1);
    for (int k = C.k0; k < C.k1; k++) {
        const GradPlane hi = grad_plane(v, C.cs, (k + 1) * C.pl, C.r0, C.r1, C.i, C.i1);
        const long q = k * C.pl + C.r0 + C.i;
        double G[3][3];
        grad_cell(lo, hi, w.dt4h, G);
        lo = hi;
        double s6[6], ss6[6];
#pragma unroll
        for (int a = 0; a < 6; a++) ss6[a] = sig_star[a * nc + q];
        correct_cell(w, G, ss6, s6);
#pragma unroll
        for (int a = 0; a < 6; a++) sig[a * nc + q] = s6[a];
        const double chi_q = chi_src[q];
        chi_dst[q] = chi_q;
        predict_cell(w, c, G, s6, chi_q, q, nc, sig_star, dpl, sbar_out);
    }
}

// wall velocities of section 4 (simple shear with ramp) and section 5 (disc)
__global__ void k_wall_fill(WallParams w, double *__restrict__ v) {
    const int i = blockIdx.x * BX + threadIdx.x, j = blockIdx.y * BY + threadIdx.y;
    if (i >= w.nx || j >= w.ny) return;
    const long pl = (long)w.nx * w.ny;
    const long t = (long)j * w.nx + i;
    double top[3] = {0.0, 0.0, 0.0}, bot[3] = {0.0, 0.0, 0.0};
    if (w.kind == 0) {
        const double U = (w.t < w.t_ramp) ? w.U_B * w.t / w.t_ramp : w.U_B;
        top[0] = U;
        bot[0] = -U;
    } else {
        const double L = 0.5 * w.nx * w.h;
        const double x = -L + i * w.h, y = -0.5 * w.ny * w.h + j * w.h;
        const double r2 = (x * x + y * y) / (L * L), R2 = w.R * w.R;
        const double f = (r2 < R2) ? 1.0 : exp(-w.lambda_w * (r2 - R2) * (r2 - R2));
        top[0] = -w.omega * y * f;
        top[1] = w.omega * x * f;
        const double sgn = (w.kind == 2) ? 1.0 : (w.kind == 3 ? -1.0 : 0.0);
        bot[0] = sgn * top[0];
        bot[1] = sgn * top[1];
    }
    const long cs = (long)(w.nz + 1) * pl;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        v[a * cs + t] = bot[a];
        v[a * cs + (long)w.nz * pl + t] = top[a];
    }
}

// ------------------------------------------------------------ explicit method
// (section 3.2): forward Euler of Eqs. (24)-(26) with ENO advection (Eq. 33)

// ENO first derivative, Eq. (33), times 2 h, from the values at offsets -2..2
// along one axis and the velocity component u along it: the one-sided
// three-point stencil on the upwind side where that side is smoother than the
// centre, else the centred difference.  The smoothness test compares the
// magnitudes of the undivided second differences: the curvatures of Eq. (33)
// are those divided by the same h^2 > 0, which cannot reorder them.  With f1
// the neighbour on the upwind side and c_up the second difference about it the
// one-sided stencil 3 f0 - 4 f1 + f2 is c_up + 2 (f0 - f1); values are chosen
// and magnitudes compared with integer instructions, which leaves 7 FP64
// instructions (they set the pace: 19 clocks of an SM each) of about 20.  c0 returns the centred second
// difference.
__device__ __forceinline__ double eno_2h(double fm2, double fm1, double f0, double fp1, double fp2,
                                         double u, double &c0) {
    const bool neg = u < 0.0;
    const double f1 = neg ? fp1 : fm1;
    // (explicit fma: a doubling would otherwise become an addition of its own)
    const double cu = fma(-2.0, f1, neg ? fp2 : f0) + (neg ? f0 : fm2);
    c0 = fma(-2.0, f0, fp1) + fm1;
    const double one = fma(2.0, f0 - f1, cu), mid = fp1 - fm1;
    // |c0| > |cu|, false for a NaN on either side
    const long long m0 = __double_as_longlong(c0) & 0x7fffffffffffffffLL,
                    mu = __double_as_longlong(cu) & 0x7fffffffffffffffLL;
    const bool smoother = m0 > mu && m0 <= 0x7ff0000000000000LL;
    const double side = __longlong_as_double(__double_as_longlong(one) ^
                                             (neg ? (long long)0x8000000000000000ULL : 0LL));
    return smoother && (neg || u > 0.0) ? side : mid;
}

// offsets along an axis of n entries, -2 .. 2 around i, periodic
__device__ __forceinline__ void around(int i, int n, int (&o)[5]) {
#pragma unroll
    for (int m = 0; m < 5; m++) {
        const int a = i + m - 2;
        o[m] = a < 0 ? a + n : (a >= n ? a - n : a);
    }
}

// 2 h (u.grad) sigma_n at cell (i, j, k) for the 6 stored components: ENO
// derivatives (Eq. 33) along x and y (wrapping) and z, where cell fields two
// layers beyond the z boundaries are extrapolated linearly from the two
// layers next to them; u is the cell's advecting velocity
__device__ __forceinline__ void stress_advection(const double *__restrict__ sig, long nc, int nx,
                                                 long pl, int nz, int j, int k, long col,
                                                 const int (&ix)[5], const int (&jy)[5],
                                                 const double (&u)[3], double (&adv)[6]) {
    const long rx = k * pl + (long)j * nx, cy = k * pl + (col - (long)j * nx);
    const bool inner = k >= 2 && k < nz - 2;
#pragma unroll
    for (int n = 0; n < 6; n++) {
        const double *f = sig + n * nc;
        double fx[5], fy[5], fz[5], c0;
#pragma unroll
        for (int m = 0; m < 5; m++) {
            fx[m] = f[rx + ix[m]];
            fy[m] = f[cy + (long)jy[m] * nx];
        }
        if (inner) {
#pragma unroll
            for (int m = 0; m < 5; m++) fz[m] = f[(k + m - 2) * pl + col];
        } else {
#pragma unroll
            for (int m = 0; m < 5; m++) {
                const int kk = k + m - 2;
                if (kk < 0)
                    fz[m] = f[col] + kk * (f[pl + col] - f[col]);
                else if (kk > nz - 1)
                    fz[m] = f[(nz - 1) * pl + col] +
                            (kk - (nz - 1)) * (f[(nz - 1) * pl + col] - f[(nz - 2) * pl + col]);
                else
                    fz[m] = f[kk * pl + col];
            }
        }
        double t = u[0] * eno_2h(fx[0], fx[1], fx[2], fx[3], fx[4], u[0], c0);
        t = fma(u[1], eno_2h(fy[0], fy[1], fy[2], fy[3], fy[4], u[1], c0), t);
        adv[n] = fma(u[2], eno_2h(fz[0], fz[1], fz[2], fz[3], fz[4], u[2], c0), t);
    }
}

// the mean of a cell's 8 corner velocities, from the plane sums below and above
__device__ __forceinline__ void mean_velocity(const GradPlane &lo, const GradPlane &hi,
                                              double (&u)[3]) {
#pragma unroll
    for (int a = 0; a < 3; a++) u[a] = 0.125 * (lo.Z[a] + hi.Z[a]);
}

// Eq. (25) at cell centres: sigma' = sigma + dt (-(u.grad) sigma + L sigma +
// sigma L^T - tr(L) sigma + C:(D - D^pl sigma0 / sbar)), L the Eq. (31)
// gradient of v, u the mean of the cell's 8 corner velocities; the ENO
// stencils reach two cells out, z ghost cells extrapolate each component
// linearly from the two layers next to the wall; D^pl and sbar of the state
// are written for the chi update.  Columns march in z as in the predictor;
// bound by FP64 instructions: 124 us at 64 x 64 x 32, 219 with a thread a cell
// and both one-sided derivatives formed.
__global__ void __launch_bounds__(128)
    k_explicit_stress(StepParams p, CellConst w, StzConst c, int chunk,
                      const double *__restrict__ v, const double *__restrict__ sig,
                      const double *__restrict__ chi, double *__restrict__ sig_new,
                      double *__restrict__ dpl, double *__restrict__ sbar_out, long nc) {
    CellColumn C;
    if (!cell_column(p.nx, p.ny, p.nz, chunk, C)) return;
    const long col = C.r0 + C.i;
    int ix[5], jy[5];
    around(C.i, p.nx, ix);
    around(C.j, p.ny, jy);
    GradPlane lo = grad_plane(v, C.cs, C.k0 * C.pl, C.r0, C.r1, C.i, C.i1);
    for (int k = C.k0; k < C.k1; k++) {
        const GradPlane hi = grad_plane(v, C.cs, (k + 1) * C.pl, C.r0, C.r1, C.i, C.i1);
        const long q = k * C.pl + col;
        double G[3][3], u[3], adv[6], s6[6], rate[6], D, sb;
        grad_cell(lo, hi, w.dt4h, G);
        mean_velocity(lo, hi, u);
        lo = hi;
        stress_advection(sig, nc, p.nx, C.pl, p.nz, C.j, k, col, ix, jy, u, adv);
#pragma unroll
        for (int a = 0; a < 6; a++) s6[a] = sig[a * nc + q];
        objective_increment(w, c, G, s6, chi[q], rate, D, sb);
        const double lt = w.lam * (G[0][0] + G[1][1] + G[2][2]);
#pragma unroll
        for (int a = 0; a < 3; a++) rate[a] += fma(w.mu2, G[a][a], lt);
        rate[3] = fma(w.mu, G[1][2] + G[2][1], rate[3]);
        rate[4] = fma(w.mu, G[0][2] + G[2][0], rate[4]);
        rate[5] = fma(w.mu, G[0][1] + G[1][0], rate[5]);
#pragma unroll
        for (int n = 0; n < 6; n++) sig_new[n * nc + q] = s6[n] + fma(-w.dt2h, adv[n], rate[n]);
        dpl[q] = D;
        sbar_out[q] = sb;
    }
}

// the stress advection of the general constitutive law (section 2), which
// Eq. (27) drops, as an option of the quasi-static step: sigma* -= dt (u.grad)
// sigma^n, u the mean of the cell's 8 corner velocities of v^n (the
// explicit method's advection, Eq. 33 and its ghosts); bound by the 18 ENO
// derivatives a cell: 391 us at 96^3, 810 with a thread a cell
__global__ void __launch_bounds__(128)
    k_stress_advect(StepParams p, CellConst w, int chunk, const double *__restrict__ v,
                    const double *__restrict__ sig, double *__restrict__ sig_star, long nc) {
    CellColumn C;
    if (!cell_column(p.nx, p.ny, p.nz, chunk, C)) return;
    const long col = C.r0 + C.i;
    int ix[5], jy[5];
    around(C.i, p.nx, ix);
    around(C.j, p.ny, jy);
    auto corner_sum = [&](int k, double (&z)[3]) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const double *g = v + a * C.cs + k * C.pl;
            z[a] = (g[C.r0 + C.i] + g[C.r0 + C.i1]) + (g[C.r1 + C.i] + g[C.r1 + C.i1]);
        }
    };
    double lo[3], hi[3];
    corner_sum(C.k0, lo);
    for (int k = C.k0; k < C.k1; k++) {
        corner_sum(k + 1, hi);
        double u[3], adv[6], ss[6];
#pragma unroll
        for (int a = 0; a < 3; a++) {
            u[a] = 0.125 * (lo[a] + hi[a]);
            lo[a] = hi[a];
        }
        stress_advection(sig, nc, p.nx, C.pl, p.nz, C.j, k, col, ix, jy, u, adv);
        const long q = k * C.pl + col;
#pragma unroll
        for (int n = 0; n < 6; n++) ss[n] = sig_star[n * nc + q];
#pragma unroll
        for (int n = 0; n < 6; n++) sig_star[n * nc + q] = fma(-w.dt2h, adv[n], ss[n]);
    }
}

// Eq. (24) at interior corners (k = 1 .. nz-1):
//   v' = v + dt (-(v.grad) v + div sigma / rho + kappa lap v),
// the divergence the corner version of Eq. (31) over the 8 cells around the
// corner, the Laplacian Eq. (32) along each axis (the second differences the
// ENO test forms anyway), ENO advection with the corner's own velocity;
// corners up to two planes beyond a wall reflect v through the wall value,
// v(-m) = 2 v(0) - v(m).  Marches in z; 59 us at 64 x 64 x 32 against 102 with
// a thread a corner.
struct VelConst {
    double div, lap, adv;  // dt / (4 h rho);  dt kappa / h^2;  dt / (2 h)
};
__global__ void __launch_bounds__(128)
    k_explicit_velocity(StepParams p, VelConst w, int chunk, const double *__restrict__ v,
                        const double *__restrict__ sig, double *__restrict__ v_new, long nc) {
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int col = blockIdx.x * blockDim.x + threadIdx.x, j = col / nx, i = col - j * nx;
    if (j >= ny) return;
    const int k0 = 1 + blockIdx.y * chunk;
    const int k1 = k0 + chunk < nz ? k0 + chunk : nz;
    const long pl = (long)nx * ny, cs = (long)(nz + 1) * pl;
    const int im = i ? i - 1 : nx - 1, jm = j ? j - 1 : ny - 1;
    const long rj0 = (long)jm * nx, rj1 = (long)j * nx;
    int ix[5], jy[5];
    around(i, nx, ix);
    around(j, ny, jy);
    // the z differences are taken column by column (the layer sums of the
    // right-hand side would cost 9 instructions less and 3% more rounding)
    double flo[3][2][2], fhi[3][2][2], xlo[3], xhi[3];
    div_parts(sig, nc, (long)(k0 - 1) * pl, rj0, rj1, im, i, xlo, flo);
    for (int k = k0; k < k1; k++) {
        div_parts(sig, nc, (long)k * pl, rj0, rj1, im, i, xhi, fhi);
        const long node = (long)k * pl + col;
        const double u[3] = {v[node], v[cs + node], v[2 * cs + node]};
        const bool inner = k >= 2 && k <= nz - 2;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const double *g = v + a * cs;
            double fx[5], fy[5], fz[5], cx, cy, cz;
#pragma unroll
            for (int m = 0; m < 5; m++) {
                fx[m] = g[k * pl + rj1 + ix[m]];
                fy[m] = g[k * pl + (long)jy[m] * nx + i];
            }
            if (inner) {
#pragma unroll
                for (int m = 0; m < 5; m++) fz[m] = g[(k + m - 2) * pl + col];
            } else {
#pragma unroll
                for (int m = 0; m < 5; m++) {
                    const int kk = k + m - 2;
                    if (kk < 0)
                        fz[m] = 2.0 * g[col] - g[-kk * pl + col];
                    else if (kk > nz)
                        fz[m] = 2.0 * g[nz * pl + col] - g[(2 * nz - kk) * pl + col];
                    else
                        fz[m] = g[kk * pl + col];
                }
            }
            double t = u[0] * eno_2h(fx[0], fx[1], fx[2], fx[3], fx[4], u[0], cx);
            t = fma(u[1], eno_2h(fy[0], fy[1], fy[2], fy[3], fy[4], u[1], cy), t);
            t = fma(u[2], eno_2h(fz[0], fz[1], fz[2], fz[3], fz[4], u[2], cz), t);
            const double div = (xlo[a] + xhi[a]) +
                               (((fhi[a][0][0] - flo[a][0][0]) + (fhi[a][0][1] - flo[a][0][1])) +
                                ((fhi[a][1][0] - flo[a][1][0]) + (fhi[a][1][1] - flo[a][1][1])));
            const double lap = (cx + cy) + cz;
            v_new[a * cs + node] =
                fx[2] + fma(w.lap, lap, fma(w.div, div, -w.adv * t));
        }
#pragma unroll
        for (int a = 0; a < 3; a++) {
            xlo[a] = xhi[a];
#pragma unroll
            for (int y = 0; y < 2; y++)
#pragma unroll
                for (int e = 0; e < 2; e++) flo[a][y][e] = fhi[a][y][e];
        }
    }
}

}  // namespace

cudaError_t stress_predict(const StepParams &p, const double *v, const double *sig,
                           const double *chi, double *sig_star, double *dpl, double *sbar,
                           cudaStream_t s) {
    const long nc = (long)p.nx * p.ny * p.nz;
    const March m = march((long)p.nx * p.ny, p.nz);
    k_stress_predict<<<m.grid, m.threads, 0, s>>>(p, cell_const(p), stz_const(p), m.chunk, v, sig,
                                                  chi, sig_star, dpl, sbar, nc);
    count_launch();
    return cudaGetLastError();
}

cudaError_t chi_update(const StepParams &p, const double *sig, const double *chi,
                       const double *dpl, const double *sbar, double *chi_new, cudaStream_t s) {
    const long nc = (long)p.nx * p.ny * p.nz;
    const March m = march((long)p.nx * p.ny, p.nz);
    const ChiConst w{2.0 * p.dt / (p.c0 * p.sY),
                     0.5 * (p.dt / p.c0) * ((p.l * p.l) / (p.h * p.h)), p.chi_inf};
    k_chi_update<<<m.grid, m.threads, 0, s>>>(p, stz_const(p), w, m.chunk, sig, chi, dpl, sbar,
                                              chi_new, nc);
    count_launch();
    return cudaGetLastError();
}

cudaError_t div_rhs(const StepParams &p, const double *sig_star, double *b, cudaStream_t s) {
    const double scale = p.h * p.h / (p.mu * p.dt) * (0.25 / p.h);
    const March m = march((long)p.nx * p.ny, p.nz - 1);
    k_div_rhs<<<m.grid, m.threads, 0, s>>>(p, m.chunk, sig_star, b, scale);
    count_launch();
    return cudaGetLastError();
}

cudaError_t stress_correct(const StepParams &p, const double *v, const double *sig_star,
                           double *sig, const double *chi_src, double *chi_dst, cudaStream_t s) {
    const long nc = (long)p.nx * p.ny * p.nz;
    const March m = march((long)p.nx * p.ny, p.nz);
    k_stress_correct<<<m.grid, m.threads, 0, s>>>(p, cell_const(p), m.chunk, v, sig_star, sig,
                                                  chi_src, chi_dst, nc);
    count_launch();
    return cudaGetLastError();
}

cudaError_t stress_advect(const StepParams &p, const double *v, const double *sig,
                          double *sig_star, cudaStream_t s) {
    const long nc = (long)p.nx * p.ny * p.nz;
    const March m = march((long)p.nx * p.ny, p.nz);
    k_stress_advect<<<m.grid, m.threads, 0, s>>>(p, cell_const(p), m.chunk, v, sig, sig_star, nc);
    count_launch();
    return cudaGetLastError();
}

cudaError_t correct_predict(const StepParams &p, const double *v, double *sig_star, double *sig,
                            const double *chi_src, double *chi_dst, double *dpl, double *sbar,
                            cudaStream_t s) {
    const long nc = (long)p.nx * p.ny * p.nz;
    const March m = march((long)p.nx * p.ny, p.nz);
    k_correct_predict<<<m.grid, m.threads, 0, s>>>(p, cell_const(p), stz_const(p), m.chunk, v,
                                                   sig_star, sig, chi_src, chi_dst, dpl, sbar, nc);
    count_launch();
    return cudaGetLastError();
}

cudaError_t wall_fill(const WallParams &w, double *v, cudaStream_t s) {
    k_wall_fill<<<cell_grid(w.nx, w.ny, 1), kBlock, 0, s>>>(w, v);
    count_launch();
    return cudaGetLastError();
}

cudaError_t explicit_stress(const StepParams &p, const double *v, const double *sig,
                            const double *chi, double *sig_new, double *dpl, double *sbar,
                            cudaStream_t s) {
    const long nc = (long)p.nx * p.ny * p.nz;
    const March m = march((long)p.nx * p.ny, p.nz);
    k_explicit_stress<<<m.grid, m.threads, 0, s>>>(p, cell_const(p), stz_const(p), m.chunk, v, sig,
                                                   chi, sig_new, dpl, sbar, nc);
    count_launch();
    return cudaGetLastError();
}

cudaError_t explicit_velocity(const StepParams &p, double rho, double kappa, const double *v,
                              const double *sig, double *v_new, cudaStream_t s) {
    const long nc = (long)p.nx * p.ny * p.nz;
    if (p.nz < 2) return cudaSuccess;
    const March m = march((long)p.nx * p.ny, p.nz - 1);
    const VelConst w{p.dt * (0.25 / p.h) / rho, p.dt * kappa / (p.h * p.h), p.dt * (0.5 / p.h)};
    k_explicit_velocity<<<m.grid, m.threads, 0, s>>>(p, w, m.chunk, v, sig, v_new, nc);
    count_launch();
    return cudaGetLastError();
}

}  // namespace qsmg

// ------------------------------------------------------------------ adjoint
//
// Reverse of one projection step for the gradient of an objective through
// the step: given the adjoints (vbar, sigbar, chibar) of the state after the
// step, the adjoints of the state before it.  Each kernel is the transpose
// of one forward equation (Eqs. 26, 27, 29, 31 and the right-hand side of
// Eq. 30); the projection solve is its own transpose (the scaled operator is
// symmetric) and runs through the multigrid solver.  Stored stress adjoints
// follow the stored components: for an off-diagonal component the adjoint is
// the sum of the two full-matrix entries, so the full-matrix adjoint is half
// of it.

namespace qsmg {
namespace {

// STZ rate (as stz_rate) with its partial derivatives in sbar and chi
__device__ __forceinline__ void stz_rate_d(const StzConst &c, double sbar, double inv_sbar,
                                           double chi, double &D, double &Ds, double &Dc) {
    if (!(sbar > c.sY) || !(chi > 0.0)) {
        D = Ds = Dc = 0.0;
        return;
    }
    const double y = -c.ez_K / chi, x = c.beta * sbar;
    const double ep = exp(x + y), em = exp(y - x);
    const double f = 1.0 - c.sY * inv_sbar;
    D = (ep + em) * c.half_eDT_over_tau0 * f;
    Ds = c.half_eDT_over_tau0 * (c.beta * (ep - em) * f + (ep + em) * c.sY * inv_sbar * inv_sbar);
    Dc = D * c.ez_K / (chi * chi);
}

// deviatoric part and sbar of a stored stress
__device__ __forceinline__ void dev_of(const double s[6], double S0[3][3], double &sb,
                                       double &inv_sb) {
    const double m = (s[0] + s[1] + s[2]) * (1.0 / 3.0);
    S0[0][0] = s[0] - m;
    S0[1][1] = s[1] - m;
    S0[2][2] = s[2] - m;
    S0[1][2] = S0[2][1] = s[3];
    S0[0][2] = S0[2][0] = s[4];
    S0[0][1] = S0[1][0] = s[5];
    sb = sbar_of(s);
    inv_sb = sb > 0.0 ? 1.0 / sb : 0.0;
}

// stored adjoint of a symmetric full-matrix adjoint X (added, times w)
__device__ __forceinline__ void add_stored(double out[6], const double X[3][3], double w) {
    out[0] += w * X[0][0];
    out[1] += w * X[1][1];
    out[2] += w * X[2][2];
    out[3] += w * (X[1][2] + X[2][1]);
    out[4] += w * (X[0][2] + X[2][0]);
    out[5] += w * (X[0][1] + X[1][0]);
}

// Transpose of the chi diffusion at one z-wall ghost face.  Cell P (boundary
// layer) has a ghost neighbour with chi_g = 2 chi_P - chi_Q and sigma_g =
// 2 sigma_P - sigma_Q (Q the next layer inward); its face term in P's update
// is a (D_P + D_g)/2 (chi_g - chi_P), a = chibar'_P dt l^2 / (c0 h^2).
// Returns the adjoint contributions: to chi_P (cP), chi_Q (cQ), D_P (dP) and
// the full-matrix stress adjoint Sg of the ghost (P receives 2 Sg, Q -Sg).
struct GhostAdj {
    double cP, cQ, dP;
    double Sg[3][3];
};
__device__ __forceinline__ GhostAdj ghost_adj(const StzConst &c, const double *__restrict__ sig,
                                              const double *__restrict__ chi,
                                              const double *__restrict__ dpl, long nc, long qP,
                                              long qQ, double a) {
    GhostAdj G;
    double sg[6];
#pragma unroll
    for (int n = 0; n < 6; n++) sg[n] = 2.0 * sig[n * nc + qP] - sig[n * nc + qQ];
    const double cP = chi[qP], cg = 2.0 * cP - chi[qQ], DP = dpl[qP];
    double S0[3][3], sb, inv;
    dev_of(sg, S0, sb, inv);
    double Dg, Dgs, Dgc;
    stz_rate_d(c, sb, inv, cg, Dg, Dgs, Dgc);
    const double half_gap = 0.5 * (cg - cP);
    // d/dchi_g = a (D_P + D_g)/2 + a (chi_g - chi_P)/2 dD_g/dchi_g; chi_g = 2 chi_P - chi_Q
    const double dg = a * 0.5 * (DP + Dg) + a * half_gap * Dgc;
    G.cP = -a * 0.5 * (DP + Dg) + 2.0 * dg;
    G.cQ = -dg;
    G.dP = a * half_gap;
    const double w = a * half_gap * Dgs * 0.5 * inv;  // Dbar_g dD_g/dsbar_g / (2 sbar_g)
#pragma unroll
    for (int r = 0; r < 3; r++)
#pragma unroll
        for (int s = 0; s < 3; s++) G.Sg[r][s] = w * S0[r][s];
    return G;
}

// Transpose of Eq. (26) in gather form, per cell P: chib (adjoint of chi^n
// through the chi update), Db and sbb (adjoints of D^pl_P and sbar_P), and
// sgb (stress adjoint from the z-wall ghosts, stored; zero away from the two
// outer layers on each side)
__global__ void k_adj_chi(StepParams p, StzConst c, const double *__restrict__ sig,
                          const double *__restrict__ chi, const double *__restrict__ dpl,
                          const double *__restrict__ sbar, const double *__restrict__ cb1,
                          double *__restrict__ chib, double *__restrict__ Db,
                          double *__restrict__ sbb, double *__restrict__ sgb, long nc) {
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    int i, j, k;
    if (!cell_ijk(nx, ny, i, j, k)) return;
    const long pl = (long)nx * ny;
    const long q = (long)k * pl + (long)j * nx + i;
    const double kap = p.dt / p.c0, kd = kap * (p.l * p.l) / (p.h * p.h);
    const double bP = cb1[q], cP = chi[q], DP = dpl[q], sP = sbar[q];
    double cb = bP - bP * kap * 2.0 * DP * sP / p.sY;
    double db = bP * kap * 2.0 * sP / p.sY * (p.chi_inf - cP);
    const double sbv = bP * kap * 2.0 * DP / p.sY * (p.chi_inf - cP);
    const int ip = (i + 1 < nx) ? i + 1 : 0, im = i ? i - 1 : nx - 1;
    const int jp = (j + 1 < ny) ? j + 1 : 0, jm = j ? j - 1 : ny - 1;
    long nb[6];
    int nn = 0;
    nb[nn++] = (long)k * pl + (long)j * nx + ip;
    nb[nn++] = (long)k * pl + (long)j * nx + im;
    nb[nn++] = (long)k * pl + (long)jp * nx + i;
    nb[nn++] = (long)k * pl + (long)jm * nx + i;
    if (k + 1 < nz) nb[nn++] = q + pl;
    if (k > 0) nb[nn++] = q - pl;
    for (int n = 0; n < nn; n++) {
        const double bN = cb1[nb[n]], DN = dpl[nb[n]], cN = chi[nb[n]];
        cb += kd * 0.5 * (DP + DN) * (bN - bP);
        db += kd * 0.5 * (cN - cP) * (bP - bN);
    }
    double sg[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    // this cell's own ghost faces
    if (k == nz - 1) {
        const GhostAdj G = ghost_adj(c, sig, chi, dpl, nc, q, q - pl, bP * kd);
        cb += G.cP;
        db += G.dP;
        add_stored(sg, G.Sg, 2.0);
    }
    if (k == 0) {
        const GhostAdj G = ghost_adj(c, sig, chi, dpl, nc, q, q + pl, bP * kd);
        cb += G.cP;
        db += G.dP;
        add_stored(sg, G.Sg, 2.0);
    }
    // this cell as the inner layer of a neighbour's ghost
    if (k == nz - 2) {
        const GhostAdj G = ghost_adj(c, sig, chi, dpl, nc, q + pl, q, cb1[q + pl] * kd);
        cb += G.cQ;
        add_stored(sg, G.Sg, -1.0);
    }
    if (k == 1) {
        const GhostAdj G = ghost_adj(c, sig, chi, dpl, nc, q - pl, q, cb1[q - pl] * kd);
        cb += G.cQ;
        add_stored(sg, G.Sg, -1.0);
    }
    chib[q] = cb;
    Db[q] = db;
    sbb[q] = sbv;
#pragma unroll
    for (int n = 0; n < 6; n++) sgb[n * nc + q] = sg[n];
}

// Transpose of Eq. (27) (with the work term and the right-hand side of
// Eq. 30 folded in), per cell: from the stored adjoint of sigma^{n+1}
// (sb1, which is also that of sigma*), the gradient of the adjoint solve
// (lam), and the chi-update adjoints, the adjoints of sigma^n (written over
// sb1), chi^n (chib_out) and of the velocity gradient L (Lb, 9 per cell,
// row-major).  w_work weighs the step's plastic work 2 D^pl sbar dt h^3.
__global__ void k_adj_predict(StepParams p, StzConst c, const double *__restrict__ v,
                              const double *__restrict__ lam, const double *__restrict__ sig,
                              const double *__restrict__ chi, double *__restrict__ sb1,
                              const double *__restrict__ chib, const double *__restrict__ Db_in,
                              const double *__restrict__ sbb_in, const double *__restrict__ sgb,
                              double *__restrict__ chib_out, double *__restrict__ Lb,
                              double w_work, long nc, int chunk) {
    CellColumn C;
    if (!cell_column(p.nx, p.ny, p.nz, chunk, C)) return;
    const double inv4h = 0.25 / p.h, dt = p.dt, mu = p.mu;
    const double rhs_scale = p.h * p.h / (p.mu * dt);  // (h^2/(mu dt)) / (4h) * 4h
    const double work = w_work * 2.0 * dt * p.h * p.h * p.h;
    GradPlane vlo = grad_plane(v, C.cs, C.k0 * C.pl, C.r0, C.r1, C.i, C.i1);
    GradPlane llo = grad_plane(lam, C.cs, C.k0 * C.pl, C.r0, C.r1, C.i, C.i1);
    for (int k = C.k0; k < C.k1; k++) {
        const GradPlane vhi = grad_plane(v, C.cs, (k + 1) * C.pl, C.r0, C.r1, C.i, C.i1);
        const GradPlane lhi = grad_plane(lam, C.cs, (k + 1) * C.pl, C.r0, C.r1, C.i, C.i1);
        const long q = k * C.pl + C.r0 + C.i;
        double L[3][3], Gl[3][3];
        grad_cell(vlo, vhi, inv4h, L);
        grad_cell(llo, lhi, inv4h, Gl);
        vlo = vhi;
        llo = lhi;
        double s6[6], ss[6];
#pragma unroll
        for (int n = 0; n < 6; n++) {
            s6[n] = sig[n * nc + q];
            ss[n] = sb1[n * nc + q];
        }
        // right-hand side b = (h^2/(mu dt)) corner-div sigma*: its transpose
        // is -(h^2/(mu dt)) times the cell gradient of the solve's adjoint
        ss[0] -= rhs_scale * Gl[0][0];
        ss[1] -= rhs_scale * Gl[1][1];
        ss[2] -= rhs_scale * Gl[2][2];
        ss[3] -= rhs_scale * (Gl[1][2] + Gl[2][1]);
        ss[4] -= rhs_scale * (Gl[0][2] + Gl[2][0]);
        ss[5] -= rhs_scale * (Gl[0][1] + Gl[1][0]);
        // full-matrix adjoint of sigma*
        const double B[3][3] = {{ss[0], 0.5 * ss[5], 0.5 * ss[4]},
                                {0.5 * ss[5], ss[1], 0.5 * ss[3]},
                                {0.5 * ss[4], 0.5 * ss[3], ss[2]}};
        const double S[3][3] = {{s6[0], s6[5], s6[4]}, {s6[5], s6[1], s6[3]}, {s6[4], s6[3], s6[2]}};
        double S0[3][3], sb, inv;
        dev_of(s6, S0, sb, inv);
        double D, Ds, Dc;
        stz_rate_d(c, sb, inv, chi[q], D, Ds, Dc);
        double db = Db_in[q] + work * sb;
        double sbv = sbb_in[q] + work * D;
        const double trL = L[0][0] + L[1][1] + L[2][2];
        const double P = 2.0 * mu * dt * D * inv;
        const double trB = (B[0][0] + B[1][1] + B[2][2]) * (1.0 / 3.0);
        double Sb[3][3], Lbar[3][3];
        double BdotS = 0.0, BdotS0 = 0.0;
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int b = 0; b < 3; b++) {
                BdotS += B[a][b] * S[a][b];
                BdotS0 += B[a][b] * S0[a][b];
            }
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int b = 0; b < 3; b++) {
                double ltb = 0.0, bl = 0.0, bs = 0.0;
#pragma unroll
                for (int e = 0; e < 3; e++) {
                    ltb += L[e][a] * B[e][b];
                    bl += B[a][e] * L[e][b];
                    bs += B[a][e] * S[e][b];
                }
                Sb[a][b] = B[a][b] + dt * (ltb + bl - trL * B[a][b]) -
                           P * (B[a][b] - (a == b ? trB : 0.0));
                Lbar[a][b] = dt * (2.0 * bs - (a == b ? BdotS : 0.0));
            }
        const double Pb = -BdotS0;
        db += Pb * 2.0 * mu * dt * inv;
        sbv -= Pb * 2.0 * mu * dt * D * inv * inv;
        sbv += db * Ds;
        chib_out[q] = chib[q] + db * Dc;
        double out[6];
#pragma unroll
        for (int n = 0; n < 6; n++) out[n] = sgb[n * nc + q];
        const double w = sbv * 0.5 * inv;
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int b = 0; b < 3; b++) Sb[a][b] += w * S0[a][b];
        add_stored(out, Sb, 1.0);
#pragma unroll
        for (int n = 0; n < 6; n++) sb1[n * nc + q] = out[n];
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int b = 0; b < 3; b++) Lb[(a * 3 + b) * nc + q] = Lbar[a][b];
    }
}

// cell tensors read as full 3 x 3 matrices: the stored adjoint of
// sigma^{n+1} mapped through C (C:Sigmabar, symmetric), or a general one
// stored row-major in 9 arrays
struct LoadCSym {
    const double *sb;
    long nc;
    double lam, mu;
    __device__ __forceinline__ void operator()(long q, double T[3][3]) const {
        const double s0 = sb[q], s1 = sb[nc + q], s2 = sb[2 * nc + q];
        const double tr = s0 + s1 + s2;
        T[0][0] = lam * tr + 2.0 * mu * s0;
        T[1][1] = lam * tr + 2.0 * mu * s1;
        T[2][2] = lam * tr + 2.0 * mu * s2;
        T[1][2] = T[2][1] = mu * sb[3 * nc + q];
        T[0][2] = T[2][0] = mu * sb[4 * nc + q];
        T[0][1] = T[1][0] = mu * sb[5 * nc + q];
    }
};
struct LoadFull {
    const double *t;
    long nc;
    __device__ __forceinline__ void operator()(long q, double T[3][3]) const {
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int b = 0; b < 3; b++) T[a][b] = t[(a * 3 + b) * nc + q];
    }
};

// the corner divergence of k_div_rhs for a general cell tensor T (row a =
// output component): the 4 cells (jm..j, im..i) of one cell layer
template <class Load>
__device__ __forceinline__ DivLayer tensor_layer(const Load &ld, long base, long rj0, long rj1,
                                                 int im, int i) {
    double T00[3][3], T01[3][3], T10[3][3], T11[3][3];
    ld(base + rj0 + im, T00);
    ld(base + rj0 + i, T01);
    ld(base + rj1 + im, T10);
    ld(base + rj1 + i, T11);
    DivLayer L;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        L.XY[a] = ((T01[a][0] - T00[a][0]) + (T11[a][0] - T10[a][0])) +
                  ((T10[a][1] - T00[a][1]) + (T11[a][1] - T01[a][1]));
        L.Z[a] = (T00[a][2] + T01[a][2]) + (T10[a][2] + T11[a][2]);
    }
    return L;
}

// out = add + scale * corner-div T at the interior corners, zero on the wall
// planes; the transpose of the cell gradient of Eq. (31) is -1/(4h) times this
// divergence
template <class Load>
__global__ void __launch_bounds__(128)
    k_corner_div(StepParams p, Load ld, int chunk, const double *__restrict__ add,
                 double *__restrict__ out, double scale) {
    const int nx = p.nx, ny = p.ny, nz = p.nz;
    const int m = blockIdx.x * blockDim.x + threadIdx.x, j = m / nx, i = m - j * nx;
    if (j >= ny) return;
    const int k0 = 1 + blockIdx.y * chunk;
    const int k1 = k0 + chunk < nz ? k0 + chunk : nz;
    const int im = i ? i - 1 : nx - 1, jm = j ? j - 1 : ny - 1;
    const long pl = (long)nx * ny, cs = (long)(nz + 1) * pl;
    const long rj0 = (long)jm * nx, rj1 = (long)j * nx;
#pragma unroll
    for (int a = 0; a < 3; a++) {
        if (k0 == 1) out[a * cs + m] = 0.0;
        if (k1 == nz) out[a * cs + nz * pl + m] = 0.0;
    }
    DivLayer lo = tensor_layer(ld, (long)(k0 - 1) * pl, rj0, rj1, im, i);
    for (int k = k0; k < k1; k++) {
        const DivLayer hi = tensor_layer(ld, (long)k * pl, rj0, rj1, im, i);
        const long node = (long)k * pl + m;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const double d = (lo.XY[a] + hi.XY[a]) + (hi.Z[a] - lo.Z[a]);
            out[a * cs + node] = (add ? add[a * cs + node] : 0.0) + scale * d;
        }
        lo = hi;
    }
}

// sum over cells of a * b into partials[kRedBlocks] (fixed geometry, so the
// total is bitwise reproducible)
__global__ void __launch_bounds__(kRedThreads)
    k_dot_cells(const double *__restrict__ a, const double *__restrict__ b, long n,
                double *__restrict__ partials) {
    __shared__ double red[kRedThreads / 32];
    double acc = 0.0;
    for (long t = (long)blockIdx.x * kRedThreads + threadIdx.x; t < n;
         t += (long)gridDim.x * kRedThreads)
        acc += a[t] * b[t];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < kRedThreads / 32; w++) s += red[w];
        partials[blockIdx.x] = s;
    }
}

}  // namespace

cudaError_t adj_correct(const StepParams &p, const double *sb1, const double *vb1,
                        double *rhs_out, cudaStream_t s) {
    const long nc = (long)p.nx * p.ny * p.nz;
    const LoadCSym ld{sb1, nc, p.lam, p.mu};
    const March m = march((long)p.nx * p.ny, p.nz - 1);
    k_corner_div<LoadCSym><<<m.grid, m.threads, 0, s>>>(p, ld, m.chunk, vb1, rhs_out,
                                                        -p.dt * 0.25 / p.h);
    count_launch();
    return cudaGetLastError();
}

cudaError_t adj_chi(const StepParams &p, const double *sig, const double *chi, const double *dpl,
                    const double *sbar, const double *cb1, double *chib, double *Db, double *sbb,
                    double *sgb, cudaStream_t s) {
    const long nc = (long)p.nx * p.ny * p.nz;
    k_adj_chi<<<cell_grid(p.nx, p.ny, p.nz), kBlock, 0, s>>>(p, stz_const(p), sig, chi, dpl, sbar,
                                                              cb1, chib, Db, sbb, sgb, nc);
    count_launch();
    return cudaGetLastError();
}

cudaError_t adj_predict(const StepParams &p, const double *v, const double *lam,
                        const double *sig, const double *chi, double *sb1, const double *chib,
                        const double *Db, const double *sbb, const double *sgb, double *chib_out,
                        double *Lb, double w_work, cudaStream_t s) {
    const long nc = (long)p.nx * p.ny * p.nz;
    const March m = march((long)p.nx * p.ny, p.nz);
    k_adj_predict<<<m.grid, m.threads, 0, s>>>(p, stz_const(p), v, lam, sig, chi, sb1, chib, Db,
                                               sbb, sgb, chib_out, Lb, w_work, nc, m.chunk);
    count_launch();
    return cudaGetLastError();
}

cudaError_t adj_grad_transpose(const StepParams &p, const double *Lb, double *vb,
                               cudaStream_t s) {
    const long nc = (long)p.nx * p.ny * p.nz;
    const LoadFull ld{Lb, nc};
    const March m = march((long)p.nx * p.ny, p.nz - 1);
    k_corner_div<LoadFull><<<m.grid, m.threads, 0, s>>>(p, ld, m.chunk, nullptr, vb, -0.25 / p.h);
    count_launch();
    return cudaGetLastError();
}

cudaError_t dot_cells(const double *a, const double *b, long n, double *partials,
                      cudaStream_t s) {
    k_dot_cells<<<kRedBlocks, kRedThreads, 0, s>>>(a, b, n, partials);
    count_launch();
    return cudaGetLastError();
}

}  // namespace qsmg
