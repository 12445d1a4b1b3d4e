// strip.cu -- Gauss-Seidel sweeps (and coarse residuals) on row strips of one
// plane, for levels whose rows are short enough for shared memory.
//
// FP64: the pipe takes a warp instruction every 16 clocks of an SM and every 64
// clocks of one scheduler, however many lanes are active, so an FP64 sweep is
// bound by the number of full-lane FP64 instructions and by how evenly they
// are dealt to the 608 schedulers.  Eight colour launches of one thread a node
// leave most schedulers idle on levels of 64^3 and below and evaluate every
// sum of a node from scratch.  Here, as in smoother_rows.cu, a sweep is two
// launches: colours 0-3 (colour (i&1) + 2 (j&1) + 4 (k&1)) live on the even
// planes, 4-7 on the odd ones, and the stencil couples a plane only to its two
// neighbours, so the planes of one k-parity are updated in the order of their 4
// colours from the old neighbour planes, then the others from the new ones:
// every node sees the values of eight colour passes, and v is read and written
// about twice a sweep.  A CTA owns TY rows of a plane:
//   - the sums S = up + down and differences D = up - down of the two
//     neighbour planes are formed once per node and shared;
//   - coarse levels: the dz = +-1 part is applied row by row (small_cycle.cu
//     has the same form), 96 FP64 instructions a node instead of 154;
//   - the 4 in-plane colours run on shared rows, lanes packed by colour.
// FP32 takes the same kernel, a node a thread, on levels too small for the
// persistent row strips (smoother_rows.cu) or of rows these do not take: the z
// sums are evaluated once instead of in every pass.
// Measured per phase launch in FP64 (before: four colour launches): fine 32^3 6.3 us
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
template <typename T>
struct FineStrip {
    static constexpr int kArrays = 3;
    Fine<T> f;
};
// Coarse levels: P, R, then S, D and the row parts U, V of the fold.
template <typename T>
struct CoarseStrip {
    static constexpr int kArrays = 6;
    Coarse<T> c;
};

// sum of the terms of the node at window row jj, columns xm, x0, xp (offsets)
// that its own value does not enter: the numerators of its update
template <typename T>
__device__ __forceinline__ void numer(const FineStrip<T> &op, const T *P, const T *D, const T *R,
                                      const T *, const T *, int w, int jj, int xm, int x0, int xp,
                                      T o[3]) {
    const T lp = op.f.lp, kq = op.f.kq;
    const T *p = P + jj * w, *pm = p - w, *pp = p + w, *d = D + jj * w, *dm = d - w, *dp = d + w,
            *r = R + jj * w + x0;
    const T m01 =
        ((pp[xp + 1] - pm[xp + 1]) - (pp[xm + 1] - pm[xm + 1])) + (d[xp + 2] - d[xm + 2]);
    const T m10 = ((pp[xp] - pm[xp]) - (pp[xm] - pm[xm])) + (dp[x0 + 2] - dm[x0 + 2]);
    const T m2 = (d[xp] - d[xm]) + (dp[x0 + 1] - dm[x0 + 1]);
    o[0] = r[0] + lp * (p[xm] + p[xp]) + (pm[x0] + pp[x0]) + kq * m01;
    o[1] = r[1] + lp * (pm[x0 + 1] + pp[x0 + 1]) + (p[xm + 1] + p[xp + 1]) + kq * m10;
    o[2] = r[2] + (p[xm + 2] + p[xp + 2]) + (pm[x0 + 2] + pp[x0 + 2]) + kq * m2;
}
template <typename T>
__device__ __forceinline__ void numer(const CoarseStrip<T> &op, const T *P, const T *, const T *R,
                                      const T *U, const T *V, int w, int jj, int xm, int x0, int xp,
                                      T o[3]) {
    const int col[3] = {xm, x0, xp};
    auto u = [&](int b, int dx, int dy) -> T { return P[(jj + dy) * w + col[dx + 1] + b]; };
    T t[3];
    coarse_plane_terms(op.c, u, t);
    const int q = jj * w + x0;
#pragma unroll
    for (int a = 0; a < 3; a++) o[a] = R[q + a] - ((U[q - w + a] + V[q + w + a]) + t[a]);
}
// component a alone: in FP64 the passes give every component a thread, so that
// a pass over a few rows occupies all four schedulers (one warp instruction
// holds its scheduler's FP64 pipe for 64 clocks)
template <typename T>
__device__ __forceinline__ T numer_c(const FineStrip<T> &op, const T *P, const T *D, const T *R,
                                     const T *, const T *, int w, int jj, int xm, int x0, int xp,
                                     int a) {
    const T lp = op.f.lp, kq = op.f.kq;
    const T *p = P + jj * w + a, *d = D + jj * w;
    const T sx = p[xm] + p[xp], sy = p[x0 - w] + p[x0 + w];
    const T r = R[jj * w + x0 + a];
    if (a == 2) return r + sx + sy + kq * ((d[xp] - d[xm]) + (d[x0 + w + 1] - d[x0 - w + 1]));
    const T *o = P + jj * w + 1 - a;  // the other in-plane component
    const T dz = a ? d[x0 + w + 2] - d[x0 - w + 2] : d[xp + 2] - d[xm + 2];
    const T mx = ((o[xp + w] - o[xp - w]) - (o[xm + w] - o[xm - w])) + dz;
    return r + lp * (a ? sy : sx) + (a ? sx : sy) + kq * mx;
}
template <typename T>
__device__ __forceinline__ T numer_c(const CoarseStrip<T> &op, const T *P, const T *, const T *R,
                                     const T *U, const T *V, int w, int jj, int xm, int x0, int xp,
                                     int a) {
    const Coarse<T> &c = op.c;
    const T *p = P + jj * w + a;
    T o = c.cd[a][1] * (p[xm] + p[xp]) + c.cd[a][2] * (p[x0 - w] + p[x0 + w]) +
          c.cd[a][3] * ((p[xm - w] + p[xp + w]) + (p[xp - w] + p[xm + w]));
    if (a < 2) {
        const T *u = P + jj * w + 1 - a;
        o += c.g[2][0] * ((u[xp + w] - u[xp - w]) - (u[xm + w] - u[xm - w]));
    }
    const int q = jj * w + x0 + a;
    return R[q] - ((U[q - w] + V[q + w]) + o);
}
template <typename T>
__device__ __forceinline__ T dinv(const FineStrip<T> &op, int) { return op.f.dinv; }
template <typename T>
__device__ __forceinline__ T dinv(const CoarseStrip<T> &op, int a) { return op.c.dinv[a]; }

// what a node contributes besides S and D: nothing on coarse levels, the
// right-hand side with the z sums on the finest one
template <typename T>
__device__ __forceinline__ T rhs(const FineStrip<T> &op, int a, T b, T s) {
    return a == 2 ? b + op.f.lp * s : b + s;
}
template <typename T>
__device__ __forceinline__ T rhs(const CoarseStrip<T> &, int, T b, T) { return b; }

// the row parts of the coarse fold (see z_row in small_cycle.cu) at one node:
// R -= A, and U, V for the rows above and below
template <typename T>
__device__ __forceinline__ void row_parts(const CoarseStrip<T> &op, const T *S, const T *D, T *R,
                                          T *U, T *V, int row, int xm, int x0, int xp) {
    const Coarse<T> &c = op.c;
    const T *s = S + row, *d = D + row;
    T A[3], B[3], G[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const T sx = s[xm + a] + s[xp + a], s0 = s[x0 + a];
        A[a] = c.cd[a][4] * s0 + c.cd[a][5] * sx;
        B[a] = c.cd[a][6] * s0 + c.cd[a][7] * sx;
    }
    const T d0 = d[xp] - d[xm], d2 = d[xp + 2] - d[xm + 2];
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
template <typename T>
__device__ __forceinline__ void row_parts(const FineStrip<T> &, const T *, const T *, T *, T *,
                                          T *, int, int, int, int) {}

// column of x index i in the global arrays (parity-split or natural)
__device__ __forceinline__ int gcol(int i, int hx, int split) {
    return split ? (i & 1) * hx + (i >> 1) : i;
}

// One phase of a sweep on planes k = kbase + 2 blockIdx.y, or with RES (F = 0)
// the residual of every plane k = 1 + blockIdx.y into vout, whose wall planes
// are zeroed.  zsrc: the z-neighbour planes; wall: the array with the walls;
// split: the arrays are in parity-split column order.
template <typename T, class OP, int F, bool RES>
__global__ void __launch_bounds__(NT, 2)
    k_gs_strip(StripGeo g, OP op, const T *__restrict__ b, const T *__restrict__ vin,
               const T *zsrc, const T *wall, T *vout, int kbase, int split) {
    extern __shared__ __align__(16) unsigned char strip_smem[];
    const int TY = g.ty, rows = TY + 3, w = g.w, size = rows * w;
    T *P = reinterpret_cast<T *>(strip_smem), *D = P + size, *R = D + size;
    T *S = R + size, *U = S + size, *V = U + size;  // coarse levels only
    const int tid = threadIdx.x, nx = g.nx, hx = g.hx;
    const int k = RES ? 1 + blockIdx.y : kbase + 2 * blockIdx.y;
    const int y0 = blockIdx.x * TY;
    const T *own = vin + k * g.ps, *bk = b + k * g.ps;
    const T *lo = (k == 1 ? wall : zsrc) + (k - 1) * g.ps;
    const T *hi = (k + 1 == g.nz ? wall : zsrc) + (k + 1) * g.ps;
    for (int e = tid; e < rows * nx; e += NT) {
        const int jj = fdiv(e, g.mnx), i = e - jj * nx;
        int y = y0 - 1 - F + jj;
        while (y < 0) y += g.ny;
        while (y >= g.ny) y -= g.ny;
        // i counts columns in the array's own order
        const long q = (long)y * nx + i;
        const int s = jj * w + (split ? 3 * i : scol(i, hx));
        T l[3], h[3], p[3], r[3];
#pragma unroll
        for (int a = 0; a < 3; a++) {
            l[a] = lo[q + a * g.cs];
            h[a] = hi[q + a * g.cs];
            p[a] = __ldg(own + q + a * g.cs);
            r[a] = RES ? T(0) : __ldg(bk + q + a * g.cs);
        }
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const T sum = h[a] + l[a];
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
    T *out = vout + k * g.ps;
    if constexpr (RES) {
        for (int e = tid; e < TY * nx; e += NT) {
            const int jt = fdiv(e, g.mnx), i = e - jt * nx, jj = 1 + jt, y = y0 + jt;
            if (y >= g.ny) continue;
            const int x0 = scol(i, hx);
            T o[3];
            numer(op, P, D, R, U, V, w, jj, scol(i ? i - 1 : nx - 1, hx), x0,
                  scol(i + 1 < nx ? i + 1 : 0, hx), o);
            const long q = (long)y * nx + gcol(i, hx, split);
#pragma unroll
            for (int a = 0; a < 3; a++) {
                // the right-hand side last: it would lose digits to the
                // neighbour sums, which cancel with the centre term first
                out[q + a * g.cs] = (o[a] - op.c.cd[a][0] * P[jj * w + x0 + a]) +
                                    __ldg(bk + q + a * g.cs);
                if (k == 1) vout[q + a * g.cs] = T(0);
                if (k + 1 == g.nz) vout[q + a * g.cs + (long)g.nz * g.ps] = T(0);
            }
        }
    } else {
        // colours (F,F), (1-F,F), (F,1-F), (1-F,1-F) in (x, y) parity
#pragma unroll 1
        for (int pass = 0; pass < 4; pass++) {
            const int pi = (pass & 1) ? 1 - F : F, even = pass >> 1;
            const int n = (TY / 2 + 1 - even) * hx, nc = sizeof(T) == 8 ? 3 : 1;
            for (int e3 = tid; e3 < nc * n; e3 += NT) {
                const int a = nc == 1 ? 0 : (e3 >= n) + (e3 >= 2 * n), e = e3 - a * n;
                const int jr = fdiv(e, g.mhx), ih = e - jr * hx, jj = 2 * jr + 1 + even;
                const int i = 2 * ih + pi, x0 = scol(i, hx), xm = scol(i ? i - 1 : nx - 1, hx),
                          xp = scol(i + 1 < nx ? i + 1 : 0, hx);
                if constexpr (sizeof(T) == 8) {
                    P[jj * w + x0 + a] =
                        dinv(op, a) * numer_c(op, P, D, R, U, V, w, jj, xm, x0, xp, a);
                } else {
                    T o[3];
                    numer(op, P, D, R, U, V, w, jj, xm, x0, xp, o);
#pragma unroll
                    for (int c = 0; c < 3; c++) P[jj * w + x0 + c] = dinv(op, c) * o[c];
                }
            }
            __syncthreads();
        }
        for (int e = tid; e < TY * nx; e += NT) {
            const int jt = fdiv(e, g.mnx), i = e - jt * nx, y = y0 + jt;
            if (y >= g.ny) continue;
            const long q = (long)y * nx + i;
            const int s = (jt + 1 + F) * w + (split ? 3 * i : scol(i, hx));
#pragma unroll
            for (int a = 0; a < 3; a++) out[q + a * g.cs] = P[s + a];
        }
    }
}

// strip height: 8 rows keep the repeated row at 1/8 of the work, 4 give a
// small level enough CTAs; 0 if the rows are too long for shared memory
int strip_rows(const Dims &d, size_t node_bytes, int nplanes) {
    for (int ty = 8; ty >= 4; ty -= 4) {
        if (node_bytes * (ty + 3) * d.nx > (size_t)kStripSmem) continue;
        if (ty == 8 && (long)((d.ny + 7) / 8) * nplanes < 152) continue;
        return ty;
    }
    return 0;
}

template <int F, bool RES, typename T, class OP>
cudaError_t launch(const Dims &d, const OP &op, const T *b, const T *vin, const T *zsrc,
                   const T *wall, T *vout, int kbase, int nplanes, cudaStream_t s, int split) {
    if (nplanes <= 0) return cudaSuccess;
    const size_t node = 3 * OP::kArrays * sizeof(T);
    StripGeo g;
    g.nx = d.nx;
    g.ny = d.ny;
    g.nz = d.nz;
    g.hx = d.nx / 2;
    g.w = 3 * d.nx;
    g.ty = strip_rows(d, node, nplanes);
    if (g.ty == 0) return cudaErrorNotSupported;
    g.mnx = magic(d.nx);
    g.mhx = magic(g.hx);
    g.ps = (long)d.nx * d.ny;
    g.cs = d.cs;
    const dim3 grid((d.ny + g.ty - 1) / g.ty, nplanes);
    k_gs_strip<T, OP, F, RES>
        <<<grid, NT, node * (g.ty + 3) * d.nx, s>>>(g, op, b, vin, zsrc, wall, vout, kbase, split);
    count_launch();
    return cudaGetLastError();
}

template <typename T, class OP>
cudaError_t sweep(const Dims &d, const OP &op, const T *b, const T *vin, const T *wall, T *vout,
                  bool descending, cudaStream_t s, int split) {
    const int ne = d.nz / 2 - 1, no = d.nz / 2;
    cudaError_t e;
    if (!descending) {  // even planes with colours 0-3, then odd ones with 4-7
        e = launch<0, false>(d, op, b, vin, vin, wall, vout, 2, ne, s, split);
        if (e != cudaSuccess) return e;
        return launch<0, false>(d, op, b, vin, vout, wall, vout, 1, no, s, split);
    }
    e = launch<1, false>(d, op, b, vin, vin, wall, vout, 1, no, s, split);
    if (e != cudaSuccess) return e;
    return launch<1, false>(d, op, b, vin, vout, wall, vout, 2, ne, s, split);
}

template <class K>
cudaError_t allow(K kernel) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kStripSmem);
}
template <typename T>
cudaError_t allow_all() {
    cudaError_t e = allow(k_gs_strip<T, FineStrip<T>, 0, false>);
    if (e == cudaSuccess) e = allow(k_gs_strip<T, FineStrip<T>, 1, false>);
    if (e == cudaSuccess) e = allow(k_gs_strip<T, CoarseStrip<T>, 0, false>);
    if (e == cudaSuccess) e = allow(k_gs_strip<T, CoarseStrip<T>, 1, false>);
    return e == cudaSuccess ? allow(k_gs_strip<T, CoarseStrip<T>, 0, true>) : e;
}

}  // namespace

cudaError_t strip_init() {
    const cudaError_t e = allow_all<double>();
    return e == cudaSuccess ? allow_all<float>() : e;
}

template <typename T>
bool strip_fits(const Dims &d, bool finest) {
    const size_t node = 3 * sizeof(T) * (finest ? 3 : 6);
    if (d.nx % 2 || d.ny % 2 || strip_rows(d, node, d.nz / 2) == 0) return false;
    if (sizeof(T) == 8) return d.nx <= (finest ? kStripFineNx : kStripCoarseNx);
    return finest ? !fine_rows_fit(d) : !coarse_rows_fit(d);
}

template <typename T>
cudaError_t gs_sweep_strip(const Dims &d, const Fine<T> &f, const T *b, const T *vin,
                           const T *wall, T *vout, bool descending, cudaStream_t s, int split) {
    return sweep(d, FineStrip<T>{f}, b, vin, wall, vout, descending, s, split);
}
template <typename T>
cudaError_t gs_sweep_strip(const Dims &d, const Coarse<T> &c, const T *b, const T *vin,
                           const T *wall, T *vout, bool descending, cudaStream_t s) {
    return sweep(d, CoarseStrip<T>{c}, b, vin, wall, vout, descending, s, 0);
}
template <typename T>
cudaError_t residual_strip(const Dims &d, const Coarse<T> &c, const T *b, const T *x, T *r,
                           cudaStream_t s) {
    return launch<0, true>(d, CoarseStrip<T>{c}, b, x, x, x, r, 1, d.nz - 1, s, 0);
}

// FP32: the persistent rows where they take the level, else the strips (which a
// caller's arrays at any word suit); every level of even sizes that mg_setup
// accepts suits one of them
cudaError_t gs_sweep_fine32(const Dims &d, const Fine<float> &f, const float *b, const float *vin,
                            float *vout, bool descending, cudaStream_t s, int split,
                            const SweepSync *sync) {
    if (!sync && strip_fits<float>(d, true))
        return gs_sweep_strip(d, f, b, vin, vin, vout, descending, s, split);
    return gs_sweep_fine_rows(d, f, b, vin, vout, descending, s, split, sync);
}
cudaError_t gs_sweep_coarse32(const Dims &d, const Coarse<float> &c, const float *b,
                              const float *vin, float *vout, bool descending, cudaStream_t s) {
    if (strip_fits<float>(d, false))
        return gs_sweep_strip(d, c, b, vin, vin, vout, descending, s);
    return gs_sweep_coarse_rows(d, c, b, vin, vout, descending, s);
}

#define INSTANTIATE(T)                                                                           \
    template bool strip_fits<T>(const Dims &, bool);                                             \
    template cudaError_t gs_sweep_strip<T>(const Dims &, const Fine<T> &, const T *, const T *,  \
                                           const T *, T *, bool, cudaStream_t, int);             \
    template cudaError_t gs_sweep_strip<T>(const Dims &, const Coarse<T> &, const T *, const T *, \
                                           const T *, T *, bool, cudaStream_t);                  \
    template cudaError_t residual_strip<T>(const Dims &, const Coarse<T> &, const T *, const T *, \
                                           T *, cudaStream_t);
INSTANTIATE(double)
INSTANTIATE(float)
#undef INSTANTIATE

}  // namespace qsmg
