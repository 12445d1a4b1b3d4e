// strip64.cu -- FP64 Gauss-Seidel sweeps (and coarse residuals) on row strips of
// one plane, for levels whose rows are short enough for shared memory.
//
// The FP64 pipe takes a warp instruction every 16 clocks of an SM and every 64
// clocks of one scheduler, however many lanes are active, so an FP64 sweep is
// bound by the number of full-lane FP64 instructions and by how evenly they
// are dealt to the 608 schedulers.  Eight colour launches of one thread a node
// leave most schedulers idle on levels of 64^3 and below and evaluate every
// sum of a node from scratch.  Here a sweep is two launches (planes of one
// k-parity, then of the other, as in smoother_fast.cu); a CTA owns TY rows of
// a plane:
//   - the sums S = up + down and differences D = up - down of the two
//     neighbour planes are formed once per node and shared;
//   - coarse levels: the dz = +-1 part is applied row by row (small_cycle.cu
//     has the same form), 96 FP64 instructions a node instead of 154;
//   - the 4 in-plane colours run on shared rows, lanes packed by colour.
// Measured per phase launch (before: four colour launches): fine 32^3 6.3 us
// (29), 64^3 19 us (30), coarse 32^3 9.5 us (57), 64^3 37.6 us (57).  What
// bounds it now: at 64^3 two waves of 256 strips on 152 SMs, at 32^3 the
// latency of the loads, the four passes and the single-warp FP64 rate.
//
// Window rows jj = 0 .. TY+2 are y = y0 - 1 - F + jj; the odd ones have
// y-parity F and are updated first (rows 1 .. TY+1), then the even ones
// (2 .. TY); rows 1+F .. TY+F are the strip's own.  So each strip repeats one
// row of its neighbour's work (and two rows of S, D), which is what it costs
// not to synchronise between strips; the sweep is out of place.
#include "qsmg_impl.h"

namespace qsmg {
namespace {

constexpr int NT = 256;
constexpr int kStripSmem = 200 * 1024;

__device__ __forceinline__ int fdiv(int t, unsigned m) {
    return m ? (int)__umulhi((unsigned)t, m) : t;
}
inline unsigned magic(int d) { return d == 1 ? 0u : (unsigned)((1ull << 32) / (unsigned)d + 1); }

// column offset in a shared row: parity-split, three components a node
__device__ __forceinline__ int scol(int i, int hx) { return 3 * ((i & 1) * hx + (i >> 1)); }

struct StripGeo {
    int nx, ny, nz, hx, w, ty;  // w: row pitch (elements)
    unsigned mnx, mhx;
    long ps, cs;
};

// Finest level: P, D and R (right-hand side plus the sums of the z pairs).
struct FineStrip {
    static constexpr int kArrays = 3;
    Fine<double> f;
};
// Coarse levels: P, R, then S, D and the row parts U, V of the fold.
struct CoarseStrip {
    static constexpr int kArrays = 6;
    Coarse<double> c;
};

// residual of the node at window row jj, columns xm, x0, xp (offsets)
__device__ __forceinline__ void resid(const CoarseStrip &op, const double *P, const double *,
                                      const double *R, const double *U, const double *V, int w,
                                      int jj, int xm, int x0, int xp, double o[3]) {
    const int col[3] = {xm, x0, xp};
    auto u = [&](int b, int dx, int dy) -> double { return P[(jj + dy) * w + col[dx + 1] + b]; };
    double t[3];
    coarse_plane_terms(op.c, u, t);
    const int q = jj * w + x0;
#pragma unroll
    for (int a = 0; a < 3; a++)
        o[a] = R[q + a] - (op.c.cd[a][0] * P[q + a] + ((U[q - w + a] + V[q + w + a]) + t[a]));
}
// numerator of component a of a node's update (the right-hand side minus every
// off-centre term): the passes give every component a thread, so that a pass
// over a few rows occupies all four schedulers (one warp instruction holds its
// scheduler's FP64 pipe for 64 clocks)
__device__ __forceinline__ double numer_c(const FineStrip &op, const double *P, const double *D,
                                          const double *R, const double *, const double *, int w,
                                          int jj, int xm, int x0, int xp, int a) {
    const double lp = op.f.lp, kq = op.f.kq;
    const double *p = P + jj * w + a, *d = D + jj * w;
    const double sx = p[xm] + p[xp], sy = p[x0 - w] + p[x0 + w];
    const double r = R[jj * w + x0 + a];
    if (a == 2) return r + sx + sy + kq * ((d[xp] - d[xm]) + (d[x0 + w + 1] - d[x0 - w + 1]));
    const double *o = P + jj * w + 1 - a;  // the other in-plane component
    const double dz = a ? d[x0 + w + 2] - d[x0 - w + 2] : d[xp + 2] - d[xm + 2];
    const double mx = ((o[xp + w] - o[xp - w]) - (o[xm + w] - o[xm - w])) + dz;
    return r + lp * (a ? sy : sx) + (a ? sx : sy) + kq * mx;
}
__device__ __forceinline__ double numer_c(const CoarseStrip &op, const double *P, const double *,
                                          const double *R, const double *U, const double *V, int w,
                                          int jj, int xm, int x0, int xp, int a) {
    const Coarse<double> &c = op.c;
    const double *p = P + jj * w + a;
    double o = c.cd[a][1] * (p[xm] + p[xp]) + c.cd[a][2] * (p[x0 - w] + p[x0 + w]) +
               c.cd[a][3] * ((p[xm - w] + p[xp + w]) + (p[xp - w] + p[xm + w]));
    if (a < 2) {
        const double *u = P + jj * w + 1 - a;
        o += c.g[2][0] * ((u[xp + w] - u[xp - w]) - (u[xm + w] - u[xm - w]));
    }
    const int q = jj * w + x0 + a;
    return R[q] - ((U[q - w] + V[q + w]) + o);
}
__device__ __forceinline__ double dinv(const FineStrip &op, int) { return op.f.dinv; }
__device__ __forceinline__ double dinv(const CoarseStrip &op, int a) { return op.c.dinv[a]; }

// what a node contributes besides S and D: nothing on coarse levels, the
// right-hand side with the z sums on the finest one
__device__ __forceinline__ double rhs(const FineStrip &op, int a, double b, double s) {
    return a == 2 ? b + op.f.lp * s : b + s;
}
__device__ __forceinline__ double rhs(const CoarseStrip &, int, double b, double) { return b; }

// the row parts of the coarse fold (see z_row in small_cycle.cu) at one node:
// R -= A, and U, V for the rows above and below
__device__ __forceinline__ void row_parts(const CoarseStrip &op, const double *S, const double *D,
                                          double *R, double *U, double *V, int row, int xm, int x0,
                                          int xp) {
    const Coarse<double> &c = op.c;
    const double *s = S + row, *d = D + row;
    double A[3], B[3], G[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const double sx = s[xm + a] + s[xp + a], s0 = s[x0 + a];
        A[a] = c.cd[a][4] * s0 + c.cd[a][5] * sx;
        B[a] = c.cd[a][6] * s0 + c.cd[a][7] * sx;
    }
    const double d0 = d[xp] - d[xm], d2 = d[xp + 2] - d[xm + 2];
    A[0] += c.g[1][0] * d2;
    B[0] += c.g[1][1] * d2;
    A[2] += c.g[1][0] * d0;
    B[2] += c.g[1][1] * d0;
    G[0] = c.g[2][1] * (s[xp + 1] - s[xm + 1]);
    G[1] = c.g[2][1] * (s[xp] - s[xm]) +
           (c.g[0][0] * d[x0 + 2] + c.g[0][1] * (d[xm + 2] + d[xp + 2]));
    G[2] = c.g[0][0] * d[x0 + 1] + c.g[0][1] * (d[xm + 1] + d[xp + 1]);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        R[row + x0 + a] -= A[a];
        U[row + x0 + a] = B[a] - G[a];
        V[row + x0 + a] = B[a] + G[a];
    }
}
__device__ __forceinline__ void row_parts(const FineStrip &, const double *, const double *,
                                          double *, double *, double *, int, int, int, int) {}

// One phase of a sweep on planes k = kbase + 2 blockIdx.y, or with RES (F = 0)
// the residual of every plane k = 1 + blockIdx.y into vout, whose wall planes
// are zeroed.  zsrc: the z-neighbour planes; wall: the array with the walls.
template <class OP, int F, bool RES>
__global__ void __launch_bounds__(NT, 2)
    k_gs_strip(StripGeo g, OP op, const double *__restrict__ b, const double *__restrict__ vin,
               const double *zsrc, const double *wall, double *vout, int kbase) {
    extern __shared__ __align__(16) double sms[];
    const int TY = g.ty, rows = TY + 3, w = g.w, size = rows * w;
    double *P = sms, *D = P + size, *R = D + size;
    double *S = OP::kArrays == 6 ? R + size : nullptr, *U = S + size, *V = U + size;
    const int tid = threadIdx.x, nx = g.nx, hx = g.hx;
    const int k = RES ? 1 + blockIdx.y : kbase + 2 * blockIdx.y;
    const int y0 = blockIdx.x * TY;
    const double *own = vin + k * g.ps, *bk = b + k * g.ps;
    const double *lo = (k == 1 ? wall : zsrc) + (k - 1) * g.ps;
    const double *hi = (k + 1 == g.nz ? wall : zsrc) + (k + 1) * g.ps;
    for (int e = tid; e < rows * nx; e += NT) {
        const int jj = fdiv(e, g.mnx), i = e - jj * nx;
        int y = y0 - 1 - F + jj;
        while (y < 0) y += g.ny;
        while (y >= g.ny) y -= g.ny;
        const long q = (long)y * nx + i;
        const int s = jj * w + scol(i, hx);
        double l[3], h[3], p[3], r[3];
#pragma unroll
        for (int a = 0; a < 3; a++) {
            l[a] = lo[q + a * g.cs];
            h[a] = hi[q + a * g.cs];
            p[a] = __ldg(own + q + a * g.cs);
            r[a] = __ldg(bk + q + a * g.cs);
        }
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const double sum = h[a] + l[a];
            P[s + a] = p[a];
            D[s + a] = h[a] - l[a];
            R[s + a] = rhs(op, a, r[a], sum);
            if (OP::kArrays == 6) S[s + a] = sum;
        }
    }
    __syncthreads();
    if (OP::kArrays == 6) {
        for (int e = tid; e < rows * nx; e += NT) {
            const int jj = fdiv(e, g.mnx), i = e - jj * nx;
            row_parts(op, S, D, R, U, V, jj * w, scol(i ? i - 1 : nx - 1, hx), scol(i, hx),
                      scol(i + 1 < nx ? i + 1 : 0, hx));
        }
        __syncthreads();
    }
    if constexpr (RES) {
        double *out = vout + k * g.ps;
        for (int e = tid; e < TY * nx; e += NT) {
            const int jt = fdiv(e, g.mnx), i = e - jt * nx, jj = 1 + jt, y = y0 + jt;
            if (y >= g.ny) continue;
            const int x0 = scol(i, hx);
            double o[3];
            resid(op, P, D, R, U, V, w, jj, scol(i ? i - 1 : nx - 1, hx), x0,
                  scol(i + 1 < nx ? i + 1 : 0, hx), o);
            const long q = (long)y * nx + i;
#pragma unroll
            for (int a = 0; a < 3; a++) {
                out[q + a * g.cs] = o[a];
                if (k == 1) vout[q + a * g.cs] = 0.0;
                if (k + 1 == g.nz) vout[q + a * g.cs + (long)g.nz * g.ps] = 0.0;
            }
        }
        return;
    }
    // colours (F,F), (1-F,F), (F,1-F), (1-F,1-F) in (x, y) parity
#pragma unroll 1
    for (int pass = 0; pass < 4; pass++) {
        const int pi = (pass & 1) ? 1 - F : F, even = pass >> 1;
        const int n = (TY / 2 + 1 - even) * hx;
        for (int e3 = tid; e3 < 3 * n; e3 += NT) {
            const int a = (e3 >= n) + (e3 >= 2 * n), e = e3 - a * n;
            const int jr = fdiv(e, g.mhx), ih = e - jr * hx, jj = 2 * jr + 1 + even;
            const int i = 2 * ih + pi;
            const int x0 = scol(i, hx);
            P[jj * w + x0 + a] =
                dinv(op, a) * numer_c(op, P, D, R, U, V, w, jj, scol(i ? i - 1 : nx - 1, hx), x0,
                                      scol(i + 1 < nx ? i + 1 : 0, hx), a);
        }
        __syncthreads();
    }
    double *out = vout + k * g.ps;
    for (int e = tid; e < TY * nx; e += NT) {
        const int jt = fdiv(e, g.mnx), i = e - jt * nx, y = y0 + jt;
        if (y >= g.ny) continue;
        const long q = (long)y * nx + i;
#pragma unroll
        for (int a = 0; a < 3; a++) out[q + a * g.cs] = P[(jt + 1 + F) * w + scol(i, hx) + a];
    }
}

// strip height: 8 rows keep the repeated row at 1/8 of the work, 4 give a
// small level enough CTAs; 0 if the rows are too long for shared memory
int strip_rows(const Dims &d, int arrays, int nplanes) {
    for (int ty = 8; ty >= 4; ty -= 4) {
        if ((size_t)arrays * (ty + 3) * 3 * d.nx * sizeof(double) > kStripSmem) continue;
        if (ty == 8 && (long)((d.ny + 7) / 8) * nplanes < 152) continue;
        return ty;
    }
    return 0;
}

template <class OP, int F, bool RES>
cudaError_t launch(const Dims &d, const OP &op, const double *b, const double *vin,
                   const double *zsrc, const double *wall, double *vout, int kbase, int nplanes,
                   cudaStream_t s) {
    if (nplanes <= 0) return cudaSuccess;
    StripGeo g;
    g.nx = d.nx;
    g.ny = d.ny;
    g.nz = d.nz;
    g.hx = d.nx / 2;
    g.w = 3 * d.nx;
    g.ty = strip_rows(d, OP::kArrays, nplanes);
    if (g.ty == 0) return cudaErrorNotSupported;
    g.mnx = magic(d.nx);
    g.mhx = magic(g.hx);
    g.ps = (long)d.nx * d.ny;
    g.cs = d.cs;
    const size_t smem = (size_t)OP::kArrays * (g.ty + 3) * g.w * sizeof(double);
    const dim3 grid((d.ny + g.ty - 1) / g.ty, nplanes);
    k_gs_strip<OP, F, RES><<<grid, NT, smem, s>>>(g, op, b, vin, zsrc, wall, vout, kbase);
    count_launch();
    return cudaGetLastError();
}

template <class OP>
cudaError_t sweep(const Dims &d, const OP &op, const double *b, const double *vin,
                  const double *wall, double *vout, bool descending, cudaStream_t s) {
    const int ne = d.nz / 2 - 1, no = d.nz / 2;
    cudaError_t e;
    if (!descending) {  // even planes with colours 0-3, then odd ones with 4-7
        e = launch<OP, 0, false>(d, op, b, vin, vin, wall, vout, 2, ne, s);
        if (e != cudaSuccess) return e;
        return launch<OP, 0, false>(d, op, b, vin, vout, wall, vout, 1, no, s);
    }
    e = launch<OP, 1, false>(d, op, b, vin, vin, wall, vout, 1, no, s);
    if (e != cudaSuccess) return e;
    return launch<OP, 1, false>(d, op, b, vin, vout, wall, vout, 2, ne, s);
}

template <class K>
cudaError_t allow(K kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kStripSmem);
}

}  // namespace

cudaError_t strip_init() {
    cudaError_t e = allow(k_gs_strip<FineStrip, 0, false>);
    if (e == cudaSuccess) e = allow(k_gs_strip<FineStrip, 1, false>);
    if (e == cudaSuccess) e = allow(k_gs_strip<CoarseStrip, 0, false>);
    if (e == cudaSuccess) e = allow(k_gs_strip<CoarseStrip, 1, false>);
    return e == cudaSuccess ? allow(k_gs_strip<CoarseStrip, 0, true>) : e;
}

bool strip_fits(const Dims &d, bool finest) {
    return d.nx <= (finest ? kStripFineNx : kStripCoarseNx) && d.nx % 2 == 0 && d.ny % 2 == 0 &&
           strip_rows(d, finest ? FineStrip::kArrays : CoarseStrip::kArrays, d.nz / 2) > 0;
}

cudaError_t gs_sweep_strip(const Dims &d, const Fine<double> &f, const double *b,
                           const double *vin, const double *wall, double *vout, bool descending,
                           cudaStream_t s) {
    return sweep(d, FineStrip{f}, b, vin, wall, vout, descending, s);
}
cudaError_t gs_sweep_strip(const Dims &d, const Coarse<double> &c, const double *b,
                           const double *vin, const double *wall, double *vout, bool descending,
                           cudaStream_t s) {
    return sweep(d, CoarseStrip{c}, b, vin, wall, vout, descending, s);
}
cudaError_t residual_strip(const Dims &d, const Coarse<double> &c, const double *b,
                           const double *x, double *r, cudaStream_t s) {
    return launch<CoarseStrip, 0, true>(d, CoarseStrip{c}, b, x, x, x, r, 1, d.nz - 1, s);
}
}  // namespace qsmg
