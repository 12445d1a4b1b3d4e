// residual64.cu -- the finest level's FP64 residual, marching in z.
//
// r = b - A x of the 19-point operator (scaled Eq. 30), stored in FP64 or
// reduced to its norm with an FP32 copy for the refinement step.  FP64
// instructions set the pace (19 clocks of an SM a warp instruction), so the
// kernel is built to issue few: with P = u(x+1) - u(x-1), Q = v(y+1) - v(y-1), W = w(z+1) - w(z-1)
// the mixed terms are kq times the differences of A = Q + W along x, B = P + W
// along y and C = P + Q along z, each formed once a node and shared through
// shared memory (A, B) or along the march (C), and the FP32 copy is scaled by a
// power of two in its exponent: 38 instructions a node with the norm, where
// one thread a node took 45.  256^3: 1470 us with the FP32 copy (1720), FP64 pipe
// 82% busy; two to four blocks an SM make no difference.
//
// A block owns a TX x TY tile of columns and marches over a chunk of planes
// with a ring of three haloed planes of x in shared memory; the loads of the
// plane after next are in flight while a plane is computed.
#include "qsmg_impl.h"

namespace qsmg {
namespace {

constexpr int NT = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// fixed-order sum over the block, valid in thread 0
__device__ double block_sum(double v) {
    __shared__ double sh[NT / 32];
    v = warp_sum(v);
    const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
    __syncthreads();
    if (l == 0) sh[w] = v;
    __syncthreads();
    v = threadIdx.x < (unsigned)(blockDim.x >> 5) ? sh[threadIdx.x] : 0.0;
    return w == 0 ? warp_sum(v) : 0.0;
}

// Block `block` of `blocks` adds its sum to the reduction: the last one to
// arrive adds all partial sums in a fixed order into *out and rearms the
// counter, which saves the launch of a kernel for it
__device__ void finish_sum(double acc, int block, int blocks, const NormBuf &nb, double *out) {
    __shared__ bool last;
    const double s = block_sum(acc);
    if (threadIdx.x == 0) {
        nb.partials[block] = s;
        __threadfence();
        last = atomicAdd(nb.count, 1u) == (unsigned)blocks - 1;
    }
    __syncthreads();
    if (!last) return;
    __threadfence();
    double t = 0.0;
    for (int i = threadIdx.x; i < blocks; i += blockDim.x) t += __ldcg(nb.partials + i);
    t = block_sum(t);
    if (threadIdx.x == 0) {
        *out = t;
        *nb.count = 0u;
    }
}

// float(r 2^-e) by exponent arithmetic (no FP64 multiplication); values whose
// exponent falls below the normal range vanish in FP32 anyway, those above it
// are infinite
__device__ __forceinline__ float scaled32(double r, int e) {
    const int hi = __double2hiint(r), ex = (hi >> 20) & 0x7ff;
    if (ex == 0x7ff) return (float)r;
    if (ex - e <= 0 || ex == 0) return 0.0f;
    if (ex - e >= 0x7ff) return __int_as_float(hi < 0 ? 0xff800000 : 0x7f800000);
    return (float)__hiloint2double(hi - e * (1 << 20), __double2loint(r));
}

enum { kStore = 0, kNorm = 1 };

// MODE kStore: r (walls zeroed).  MODE kNorm: sum of squares into *sum and, if
// r32, float(r 2^-norm_exponent(*scale2)) in parity-split column order (split)
template <int TX, int MODE>
__global__ void __launch_bounds__(NT, 2)
    k_res_march(Dims d, Fine<double> f, int chunk, const double *__restrict__ b,
                const double *__restrict__ x, double *__restrict__ r, float *__restrict__ r32,
                int split, const double *scale2, NormBuf nb, double *sum) {
    constexpr int TY = NT / TX, PX = TX + 2, PY = TY + 2, PL = PX * PY, HALO = 2 * PX + 2 * TY;
    __shared__ double T[3][3][PL];  // [plane mod 3][component][row][column]
    __shared__ double A[TY][PX], B[PY][TX];
    const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
    const int nx = d.nx, ny = d.ny, nz = d.nz;
    const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
    const int k0 = 1 + blockIdx.z * chunk, k1 = k0 + chunk < nz ? k0 + chunk : nz;
    const long ps = (long)nx * ny, cs = d.cs;
    const int i = x0 + tx, j = y0 + ty;
    const bool act = i < nx && j < ny;  // the others work on wrapped columns
    const long col = (long)(j % ny) * nx + i % nx;
    const int own = (ty + 1) * PX + tx + 1;
    // this thread's halo column, if it has one: rows -1 and TY, columns -1 and TX
    const bool halo = tid < HALO;
    int hpos = 0;
    long hcol = 0;
    if (halo) {
        int hr, hc;
        if (tid < 2 * PX) {
            hr = tid < PX ? 0 : PY - 1;
            hc = tid < PX ? tid : tid - PX;
        } else {
            const int e = tid - 2 * PX;
            hr = 1 + (e < TY ? e : e - TY);
            hc = e < TY ? 0 : PX - 1;
        }
        hpos = hr * PX + hc;
        hcol = (long)((y0 - 1 + hr + ny) % ny) * nx + (x0 - 1 + hc + nx) % nx;
    }
    double n[3], h[3], bn[3];
    auto fetch = [&](int k) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            n[a] = __ldg(x + a * cs + k * ps + col);
            if (halo) h[a] = __ldg(x + a * cs + k * ps + hcol);
        }
    };
    auto put = [&](int k) {
#pragma unroll
        for (int a = 0; a < 3; a++) {
            T[k % 3][a][own] = n[a];
            if (halo) T[k % 3][a][hpos] = h[a];
        }
    };
    int e = 0;
    if (MODE == kNorm && r32) e = norm_exponent(*scale2);
    // planes k0-1, k0, k0+1 in the ring; C of the first two
    fetch(k0 - 1);
    put(k0 - 1);
    fetch(k0);
    put(k0);
    fetch(k0 + 1);
    __syncthreads();
    const double lp = f.lp, kq = f.kq, d0 = f.d0;
    auto pq = [&](int k, double &P, double &Q) {
        const double *u = T[k % 3][0], *v = T[k % 3][1];
        P = u[own + 1] - u[own - 1];
        Q = v[own + PX] - v[own - PX];
    };
    double P, Q, Cm, C;
    pq(k0 - 1, P, Q);
    Cm = P + Q;
    pq(k0, P, Q);
    C = P + Q;
    double um[3], uc[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        um[a] = T[(k0 - 1) % 3][a][own];
        uc[a] = T[k0 % 3][a][own];
    }
    double acc = 0.0;
    for (int k = k0; k < k1; k++) {
        double un[3];
#pragma unroll
        for (int a = 0; a < 3; a++) un[a] = n[a];
        put(k + 1);
#pragma unroll
        for (int a = 0; a < 3; a++) bn[a] = act ? __ldg(b + a * cs + k * ps + col) : 0.0;
        if (k + 1 < k1) fetch(k + 2);
        __syncthreads();
        const double *u = T[k % 3][0], *v = T[k % 3][1], *w = T[k % 3][2];
        const double *wp = T[(k + 1) % 3][2], *wm = T[(k + 2) % 3][2];  // k - 1 = k + 2 mod 3
        const double W = un[2] - um[2];
        A[ty][tx + 1] = Q + W;
        B[ty + 1][tx] = P + W;
        if (tid < 2 * TY) {  // A on the columns beside the tile
            const int row = 1 + (tid < TY ? tid : tid - TY), c = tid < TY ? 0 : PX - 1;
            const int q = row * PX + c;
            A[row - 1][c] = (v[q + PX] - v[q - PX]) + (wp[q] - wm[q]);
        } else if (tid < 2 * TY + 2 * TX) {  // B on the rows beside it
            const int g = tid - 2 * TY, c = g < TX ? g : g - TX, row = g < TX ? 0 : PY - 1;
            const int q = row * PX + c + 1;
            B[row][c] = (u[q + 1] - u[q - 1]) + (wp[q] - wm[q]);
        }
        double Pn, Qn;
        pq(k + 1, Pn, Qn);
        const double Cn = Pn + Qn;
        // the neighbour sums cancel with the centre term first; the right-hand
        // side, added to them, would lose digits
        double o[3];
        o[0] = fma(-d0, uc[0], fma(lp, u[own - 1] + u[own + 1],
                                   (u[own - PX] + u[own + PX]) + (um[0] + un[0])));
        o[1] = fma(-d0, uc[1], fma(lp, v[own - PX] + v[own + PX],
                                   (v[own - 1] + v[own + 1]) + (um[1] + un[1])));
        o[2] = fma(-d0, uc[2], fma(lp, um[2] + un[2],
                                   (w[own - 1] + w[own + 1]) + (w[own - PX] + w[own + PX])));
        __syncthreads();
        o[0] = fma(kq, A[ty][tx + 2] - A[ty][tx], o[0]) + bn[0];
        o[1] = fma(kq, B[ty + 2][tx] - B[ty][tx], o[1]) + bn[1];
        o[2] = fma(kq, Cn - Cm, o[2]) + bn[2];
        if (act) {
            const long row = (long)k * ps + (long)j * nx;
#pragma unroll
            for (int a = 0; a < 3; a++) {
                if (MODE == kStore) {
                    r[a * cs + row + i] = o[a];
                    if (k == 1) r[a * cs + col] = 0.0;
                    if (k == nz - 1) r[a * cs + nz * ps + col] = 0.0;
                } else {
                    acc = fma(o[a], o[a], acc);
                    if (r32)
                        r32[a * cs + row + (split ? (i & 1) * (nx >> 1) + (i >> 1) : i)] =
                            scaled32(o[a], e);
                }
            }
        }
        // the next plane is put over plane k - 1, which was last read before
        // the barrier above
        P = Pn;
        Q = Qn;
        Cm = C;
        C = Cn;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            um[a] = uc[a];
            uc[a] = un[a];
        }
    }
    if (MODE == kNorm)
        finish_sum(acc, blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z),
                   gridDim.x * gridDim.y * gridDim.z, nb, sum);
}

// sum of squares of the lifted right-hand side b - A (walls of x): b itself
// but on the planes beside the walls
__global__ void __launch_bounds__(NT)
    k_lifted_norm(Dims d, Fine<double> f, int chunk, const double *__restrict__ b,
                  const double *__restrict__ x, NormBuf nb, double *sum) {
    const int nx = d.nx, ny = d.ny, nz = d.nz;
    const long ps = (long)nx * ny, m = blockIdx.x * (long)NT + threadIdx.x;
    const int k0 = 1 + blockIdx.y * chunk, k1 = k0 + chunk < nz ? k0 + chunk : nz;
    double acc = 0.0;
    if (m < ps) {
        const int j = (int)(m / nx), i = (int)(m - (long)j * nx);
        const long row = (long)j * nx;
        const long im = row + (i ? i - 1 : nx - 1), ip = row + (i + 1 < nx ? i + 1 : 0);
        const long jm = (long)(j ? j - 1 : ny - 1) * nx + i, jp = (long)(j + 1 < ny ? j + 1 : 0) * nx + i;
        for (int k = k0; k < k1; k++) {
            double o[3];
#pragma unroll
            for (int a = 0; a < 3; a++) o[a] = b[a * d.cs + k * ps + m];
#pragma unroll
            for (int side = 0; side < 2; side++) {
                if (k != (side ? nz - 1 : 1)) continue;
                const double *q = x + (side ? (long)nz * ps : 0L), s = side ? f.kq : -f.kq;
                const double *u = q, *v = q + d.cs, *w = q + 2 * d.cs;
                o[0] += u[m] + s * (w[ip] - w[im]);
                o[1] += v[m] + s * (w[jp] - w[jm]);
                o[2] += f.lp * w[m] + s * ((u[ip] - u[im]) + (v[jp] - v[jm]));
            }
#pragma unroll
            for (int a = 0; a < 3; a++) acc = fma(o[a], o[a], acc);
        }
    }
    finish_sum(acc, blockIdx.x + gridDim.x * blockIdx.y, gridDim.x * gridDim.y, nb, sum);
}

// 32-wide tiles where they fill their rows, else 16-wide ones
inline bool wide(const Dims &d) { return d.nx % 32 == 0 || d.nx > 256; }

// chunks of 32 planes, shorter while the chip has fewer than two blocks an SM
// (a chunk repeats the loads of two planes and three instructions a node)
dim3 march_grid(const Dims &d, int &chunk) {
    const int tx = wide(d) ? 32 : 16, ty = NT / tx;
    const int gx = (d.nx + tx - 1) / tx, gy = (d.ny + ty - 1) / ty;
    chunk = 32;
    while (chunk > 1 && (long)gx * gy * ((d.nz - 2) / chunk + 1) < 304) chunk /= 2;
    return dim3(gx, gy, (d.nz - 2) / chunk + 1);
}
dim3 lifted_grid(const Dims &d, int &chunk) {
    const long g = ((long)d.nx * d.ny + NT - 1) / NT;
    chunk = 16;
    while (chunk > 1 && g * ((d.nz - 2) / chunk + 1) < 304) chunk /= 2;
    return dim3((unsigned)g, (d.nz - 2) / chunk + 1);
}

template <int MODE>
cudaError_t launch(const Dims &d, const Fine<double> &f, const double *b, const double *x,
                   double *r, float *r32, int split, const double *scale2, const NormBuf &nb,
                   double *sum, cudaStream_t s) {
    int chunk;
    const dim3 g = march_grid(d, chunk);
    if (wide(d))
        k_res_march<32, MODE><<<g, NT, 0, s>>>(d, f, chunk, b, x, r, r32, split, scale2, nb, sum);
    else
        k_res_march<16, MODE><<<g, NT, 0, s>>>(d, f, chunk, b, x, r, r32, split, scale2, nb, sum);
    count_launch();
    return cudaGetLastError();
}

}  // namespace

long norm_blocks(const Dims &d) {
    int chunk;
    const dim3 a = march_grid(d, chunk), b = lifted_grid(d, chunk);
    const long na = (long)a.x * a.y * a.z, nb = (long)b.x * b.y;
    return na > nb ? na : nb;
}

cudaError_t residual_march(const Dims &d, const Fine<double> &f, const double *b, const double *x,
                           double *r, cudaStream_t s) {
    return launch<kStore>(d, f, b, x, r, nullptr, 0, nullptr, NormBuf{}, nullptr, s);
}
cudaError_t residual_norm(const Dims &d, const Fine<double> &f, const double *b, const double *x,
                          float *r32, int split, const double *scale2, const NormBuf &nb,
                          double *sum, cudaStream_t s) {
    return launch<kNorm>(d, f, b, x, nullptr, r32, split, scale2, nb, sum, s);
}
cudaError_t lifted_norm(const Dims &d, const Fine<double> &f, const double *b, const double *x,
                        const NormBuf &nb, double *sum, cudaStream_t s) {
    int chunk;
    const dim3 g = lifted_grid(d, chunk);
    k_lifted_norm<<<g, NT, 0, s>>>(d, f, chunk, b, x, nb, sum);
    count_launch();
    return cudaGetLastError();
}

}  // namespace qsmg
