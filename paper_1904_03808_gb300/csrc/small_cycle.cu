// small_cycle.cu -- the V-cycle of the small levels in one launch.
//
// On a level of 32^3 nodes or fewer a sweep, a residual or a transfer is a
// few hundred nanoseconds of arithmetic, and a V-cycle of separate launches
// spends its time on launches and on waiting for the first loads of each.
// Here one cluster of 16 CTAs walks the whole V-cycle (section 3.6) from a
// given level down to the dense coarsest solve and back up:
//   - a CTA owns `ppc` consecutive interior planes of every level and keeps
//     their x and b in shared memory for the whole launch, with copies (halos)
//     of the plane below and the plane above them; only the top level's
//     arrays are read from and written to global memory;
//   - an update is stored (FP64: an updated plane is copied) through distributed
//     shared memory to the halos that mirror it too, and a cluster barrier (0.2 us measured, against
//     1.2 us for a grid-wide one) takes the place of a launch boundary;
//   - a sweep is the two phases of strip.cu, planes of one k-parity
//     and then of the other: the dz = +-1 part of the 27-point operator is
//     folded into the right-hand side, then the 4 in-plane colours run on the
//     plane, so every node sees the neighbour values of the sequential order.
//     The halos written in a phase are not those read in it;
//   - one thread a node in FP32 (up to kMaxNodes of them on the largest
//     planes), one a node component in FP64.
// Levels start from x = 0 below the top, so the first phase of their first
// pre-sweep has no neighbour planes to fold.  Every level's operator, the
// finest included, is used in its parity-class form (Coarse<T>).
//
// What bounds it: latency.  At 16^3 a phase is about 2.5 k clocks -- 600 for
// the folded rows, 4 x 250 for the passes, 900 for the barrier and the copies
// before it -- and at 32^3 the shared-memory loads add to that.  One FP32
// V-cycle from 32^3 (32^3, 16^3, 8^3 and the 4^3 solve) takes 75 us against
// about 250 us as 40 launches in a CUDA graph, one from 16^3 28 against
// 150 us.  FP64 is bound by the pipe besides (kSmallNodes64): the cycle from
// 16^3 takes 127 us (176 with three components a thread) against 780 us.  Slower forms measured on the way, per cycle
// from 32^3: three words a node instead of one 16-byte access 78 us,
// neighbour planes read remotely at the start of a phase 89 us,
// one thread per component with the 116-operation form of the fold 123 us,
// halos written by the single updates 92 us.
//
// Shared planes are [row][column][component] with the columns in parity-split
// order and a row pitch by which the nodes of a warp, which threads own in
// colour-major order, fall into different banks.
#include <cooperative_groups.h>

#include <vector>

#include "qsmg_impl.h"

namespace qsmg {
namespace {

namespace cg = cooperative_groups;

constexpr int kCta = 16;          // CTAs of the cluster
constexpr int kMaxNodes = 4;
constexpr size_t kSmallSmem = 220 * 1024;

// quotient of t / d for t * d < 2^32, from m = 2^32 / d + 1 (0 for d = 1)
__device__ __forceinline__ int fdiv(int t, unsigned m) {
    return m ? (int)__umulhi((unsigned)t, m) : t;
}

// Elements of a node in a shared plane: in FP32 its three components and one
// more, so that a node is one 16-byte load or store (8 loads of a node's
// neighbours instead of 24, 6 instead of 18 for the fold)
template <typename T>
constexpr int kNode = sizeof(T) == 4 ? 4 : 3;

__device__ __forceinline__ void load3(const float *p, float (&v)[3]) {
    const float4 q = *reinterpret_cast<const float4 *>(p);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
}
__device__ __forceinline__ void load3(const double *p, double (&v)[3]) {
#pragma unroll
    for (int a = 0; a < 3; a++) v[a] = p[a];
}
__device__ __forceinline__ void store3(float *p, const float (&v)[3]) {
    *reinterpret_cast<float4 *>(p) = make_float4(v[0], v[1], v[2], 0.f);
}
__device__ __forceinline__ void store3(double *p, const double (&v)[3]) {
#pragma unroll
    for (int a = 0; a < 3; a++) p[a] = v[a];
}

// A node of a plane, in the colour-major order in which threads own nodes
// (colour, then row, then column of the colour's quarter of the plane: a warp
// works on one colour), with the element offsets of its columns and rows at
// -1, 0, +1 (periodic)
struct Node {
    int c[3], r[3];
    int colour;  // -1: no node
};

// offset of column i in a row of level L (parity-split where it is smoothed)
template <typename T>
__device__ __forceinline__ int col_of(const SmallLevel &L, int i) {
    return kNode<T> * (L.hx ? (i & 1) * L.hx + (i >> 1) : i);
}

// The dz = +-1 part of the 27-point operator (coarse_z_terms) is separable
// row by row: with S = up + down and D = up - down, row y' contributes
//   A(y) + U(y - 1) + V(y + 1)
// to row y, each of A, U, V three components formed from columns x - 1, x,
// x + 1 of one row only: 46 operations a node instead of 116.
// SHARES: of S - 2 p, p the node between up and down (plane_residual_at).
template <bool SHARES, typename T>
__device__ __forceinline__ void z_row(const Coarse<T> &c, const T *lo, const T *P, const T *hi,
                                      const Node &n, T A[3], T U[3], T V[3]) {
    T S[3][3], D[3][3];  // [column][component]
#pragma unroll
    for (int x = 0; x < 3; x++) {
        T l[3], h[3], p[3];
        load3(lo + n.r[1] + n.c[x], l);
        load3(hi + n.r[1] + n.c[x], h);
        if (SHARES) load3(P + n.r[1] + n.c[x], p);
#pragma unroll
        for (int a = 0; a < 3; a++) {
            S[x][a] = h[a] + l[a];
            if (SHARES) S[x][a] -= T(2) * p[a];
            D[x][a] = h[a] - l[a];
        }
    }
    T B[3], G[3];
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const T sx = S[0][a] + S[2][a];
        A[a] = c.cd[a][4] * S[1][a] + c.cd[a][5] * sx;
        B[a] = c.cd[a][6] * S[1][a] + c.cd[a][7] * sx;
    }
    const T d0 = D[2][0] - D[0][0], d2 = D[2][2] - D[0][2];
    A[0] += c.g[1][0] * d2;
    B[0] += c.g[1][1] * d2;
    A[2] += c.g[1][0] * d0;
    B[2] += c.g[1][1] * d0;
    G[0] = c.g[2][1] * (S[2][1] - S[0][1]);
    G[1] = c.g[2][1] * (S[2][0] - S[0][0]) +
           (c.g[0][0] * D[1][2] + c.g[0][1] * (D[0][2] + D[2][2]));
    G[2] = c.g[0][0] * D[1][1] + c.g[0][1] * (D[0][1] + D[2][1]);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        U[a] = B[a] - G[a];
        V[a] = B[a] + G[a];
    }
}

// sum over the 8 in-plane offsets at node n of plane P
template <typename T>
__device__ __forceinline__ void plane_at(const Coarse<T> &c, const T *P, const Node &n, T o[3]) {
    T v[3][3][3];  // [row][column][component]
#pragma unroll
    for (int y = 0; y < 3; y++)
#pragma unroll
        for (int x = 0; x < 3; x++)
            if (x != 1 || y != 1) load3(P + n.r[y] + n.c[x], v[y][x]);
    auto u = [&](int b, int dx, int dy) -> T { return v[dy + 1][dx + 1][b]; };
    coarse_plane_terms(c, u, o);
}

// A x at node n of plane P but for z_row's terms of S - 2 p.  The rows of A sum to
// zero, so the centre term is the shares of the 26 others: with S - 2 p above,
// each class of in-plane neighbours has the sum of its weights over the three
// planes and gives up its share of the centre before it is weighted, and no sum of
// the size of the centre term is rounded.  (A sweep rounds such sums, and a
// residual that rounds the same ones does not see what its fixed point lost.)
template <typename T>
__device__ __forceinline__ void plane_residual_at(const Coarse<T> &c, const T *P, const Node &n,
                                                  T o[3]) {
    T v[3][3][3];  // [row][column][component]
#pragma unroll
    for (int y = 0; y < 3; y++)
#pragma unroll
        for (int x = 0; x < 3; x++) load3(P + n.r[y] + n.c[x], v[y][x]);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        const T p = v[1][1][a];
        const T sx = (v[1][0][a] + v[1][2][a]) - T(2) * p, sy = (v[0][1][a] + v[2][1][a]) - T(2) * p;
        const T sd = ((v[0][0][a] + v[2][2][a]) + (v[0][2][a] + v[2][0][a])) - T(4) * p;
        o[a] = (c.cd[a][1] + T(2) * c.cd[a][5]) * sx + (c.cd[a][2] + T(2) * c.cd[a][6]) * sy +
               (c.cd[a][3] + T(2) * c.cd[a][7]) * sd;
    }
    const T g = c.g[2][0] + T(2) * c.g[2][1];
    o[0] += g * ((v[2][2][1] - v[0][2][1]) - (v[2][0][1] - v[0][0][1]));
    o[1] += g * ((v[2][2][0] - v[0][2][0]) - (v[2][0][0] - v[0][0][0]));
}

// Component a alone of z_row and of plane_at: in FP64 a warp instruction takes
// 64 clocks of its scheduler however few lanes it has, so three threads a node
// (one a component) finish a pass over a small plane in a third of the time,
// for a few repeated sums.  a = 0 and 1 share the code with x and y exchanged
// (the warps of a component stay together, so the branch on a = 2 is uniform
// but for one warp).
template <typename T>
__device__ __forceinline__ void z_row_c(const Coarse<T> &c, const T *lo, const T *hi,
                                        const Node &n, int a, T &A, T &U, T &V) {
    auto S = [&](int x, int b) { const int q = n.r[1] + n.c[x] + b; return hi[q] + lo[q]; };
    auto D = [&](int x, int b) { const int q = n.r[1] + n.c[x] + b; return hi[q] - lo[q]; };
    const T s0 = S(1, a), sx = S(0, a) + S(2, a);
    A = c.cd[a][4] * s0 + c.cd[a][5] * sx;
    T B = c.cd[a][6] * s0 + c.cd[a][7] * sx, G;
    if (a == 1) {
        G = c.g[2][1] * (S(2, 0) - S(0, 0)) + (c.g[0][0] * D(1, 2) + c.g[0][1] * (D(0, 2) + D(2, 2)));
    } else {
        const int b = 2 - a;  // the component whose x-difference couples
        const T d = D(2, b) - D(0, b);
        A += c.g[1][0] * d;
        B += c.g[1][1] * d;
        if (a == 0)
            G = c.g[2][1] * (S(2, 1) - S(0, 1));
        else
            G = c.g[0][0] * D(1, 1) + c.g[0][1] * (D(0, 1) + D(2, 1));
    }
    U = B - G;
    V = B + G;
}
template <typename T>
__device__ __forceinline__ T plane_at_c(const Coarse<T> &c, const T *P, const Node &n, int a) {
    auto u = [&](int dx, int dy, int b) { return P[n.r[dy + 1] + n.c[dx + 1] + b]; };
    T o = c.cd[a][1] * (u(-1, 0, a) + u(1, 0, a)) + c.cd[a][2] * (u(0, -1, a) + u(0, 1, a)) +
          c.cd[a][3] * ((u(-1, -1, a) + u(1, 1, a)) + (u(1, -1, a) + u(-1, 1, a)));
    if (a < 2) {
        const int b = 1 - a;
        o += c.g[2][0] * ((u(1, 1, b) - u(1, -1, b)) - (u(-1, 1, b) - u(-1, -1, b)));
    }
    return o;
}

// COMP: a thread owns one component of its nodes, else all three
template <typename T, int NODES, bool COMP>
struct Walker {
    static constexpr int NC = COMP ? 1 : 3;
    const SmallPlan<T> &g;
    T *sm;
    cg::cluster_group cl;
    int rank, tid, nt;
    Node node[NODES];
    int comp[NODES];  // the component owned (COMP), else 0
    int act;          // threads that own nodes on the current level (whole warps)

    // own planes of level l: [first, last)
    __device__ __forceinline__ int first(int l) const {
        const int k = 1 + rank * g.lev[l].ppc;
        return k < g.lev[l].nz ? k : g.lev[l].nz;
    }
    __device__ __forceinline__ int last(int l) const {
        const int k = 1 + (rank + 1) * g.lev[l].ppc;
        return k < g.lev[l].nz ? k : g.lev[l].nz;
    }
    // own plane k of an array of level l; x has its halos around the own
    // planes, so that plane k0 - 1 and plane k1 are addressed alike
    __device__ __forceinline__ T *own(int l, int off, int k) const {
        return sm + off + (k - 1 - rank * g.lev[l].ppc) * g.lev[l].pl;
    }
    // plane k (1 <= k < nz) of an array of level l with planes of `size`
    // elements, at its owner
    __device__ __forceinline__ T *plane(int l, int off, int k, int size) const {
        const int o = fdiv(k - 1, g.lev[l].mppc);
        T *p = sm + off + (k - 1 - o * g.lev[l].ppc) * size;
        return o == rank ? p : cl.map_shared_rank(p, o);
    }
    // the halo of the CTA before (side 0) or after (side 1) this one that
    // copies this one's first or last plane, or null
    __device__ __forceinline__ T *halo(int l, int side) const {
        const SmallLevel &L = g.lev[l];
        if (side == 0)
            return rank > 0 ? cl.map_shared_rank(sm + L.x + L.ppc * L.pl, rank - 1) : nullptr;
        return 1 + (rank + 1) * L.ppc < L.nz ? cl.map_shared_rank(sm + L.x - L.pl, rank + 1)
                                             : nullptr;
    }
    // barrier over the threads that own nodes
    __device__ __forceinline__ void sync_act() const {
        asm volatile("bar.sync 1, %0;" ::"r"(act) : "memory");
    }

    // this thread's nodes on level l
    __device__ __forceinline__ void enter(int l) {
        const SmallLevel &L = g.lev[l];
        const int nh = L.np >> 2;
        const int own = (3 / NC) * L.np;
        act = own < nt ? (own + 31) & ~31 : nt;
#pragma unroll
        for (int u = 0; u < NODES; u++) {
            const int t = tid + u * nt;
            comp[u] = COMP && t < own ? fdiv(t, L.mnp) : 0;
            const int m = t - comp[u] * L.np;
            const int q = fdiv(m, L.mnh), h = m - q * nh, jh = fdiv(h, L.mhx), ih = h - jh * L.hx;
            const int i = 2 * ih + (q & 1), j = 2 * jh + (q >> 1);
            Node &n = node[u];
            n.colour = t < own ? q : -1;
            n.c[0] = col_of<T>(L, i ? i - 1 : L.nx - 1);
            n.c[1] = col_of<T>(L, i);
            n.c[2] = col_of<T>(L, i + 1 < L.nx ? i + 1 : 0);
            n.r[0] = L.w * (j ? j - 1 : L.ny - 1);
            n.r[1] = L.w * j;
            n.r[2] = L.w * (j + 1 < L.ny ? j + 1 : 0);
        }
    }

    // r = right-hand side of plane P (RES: zero) minus the dz = +-1 terms (SHARES:
    // less their shares of the centre term), at own nodes
    template <bool RES = false, bool SHARES = false>
    __device__ __forceinline__ void fold(const Coarse<T> &c, const T *b, const T *P,
                                         T (&r)[NODES][NC], int pl) const {
        const T *lo = P - pl, *hi = P + pl;
        T *U = sm + g.scratch, *V = U + g.plmax;
#pragma unroll
        for (int u = 0; u < NODES; u++) {
            if (node[u].colour < 0) continue;
            T up[NC], vp[NC], bp[NC] = {};
            const int o = node[u].r[1] + node[u].c[1] + comp[u];
            if constexpr (COMP)
                z_row_c(c, lo, hi, node[u], comp[u], r[u][0], up[0], vp[0]);
            else
                z_row<SHARES>(c, lo, P, hi, node[u], r[u], up, vp);
            put(U + o, up);
            put(V + o, vp);
            if (!RES) get(b + o, bp);
#pragma unroll
            for (int a = 0; a < NC; a++) r[u][a] = bp[a] - r[u][a];
        }
        sync_act();
#pragma unroll
        for (int u = 0; u < NODES; u++) {
            if (node[u].colour < 0) continue;
            const int om = node[u].r[0] + node[u].c[1] + comp[u],
                      op = node[u].r[2] + node[u].c[1] + comp[u];
            T up[NC], vp[NC];
            get(U + om, up);
            get(V + op, vp);
#pragma unroll
            for (int a = 0; a < NC; a++) r[u][a] -= up[a] + vp[a];
        }
    }
    // the owned components of a node
    __device__ __forceinline__ static void get(const T *p, T (&v)[NC]) {
        if constexpr (COMP)
            v[0] = p[0];
        else
            load3(p, v);
    }
    __device__ __forceinline__ static void put(T *p, const T (&v)[NC]) {
        if constexpr (COMP)
            p[0] = v[0];
        else
            store3(p, v);
    }
    // the in-plane terms at own node u
    __device__ __forceinline__ void in_plane(const Coarse<T> &c, const T *P, int u,
                                             T (&o)[NC]) const {
        if constexpr (COMP)
            o[0] = plane_at_c(c, P, node[u], comp[u]);
        else
            plane_at(c, P, node[u], o);
    }

    // n sweeps on the level entered; zero: its x is still zero everywhere
    __device__ __forceinline__ void sweeps(int l, int n, int F, bool zero) {
        const SmallLevel &L = g.lev[l];
        const Coarse<T> &c = g.op[l];
        const int k0 = first(l), nk = last(l) - k0, pl = L.pl, ppc = L.ppc;
        T *const X0 = sm + L.x, *const B0 = sm + L.b;
        T *const below = halo(l, 0), *const above = halo(l, 1);
#pragma unroll 1
        for (int s = 0; s < 2 * n; s++) {
            const int par = (s & 1) ? 1 - F : F;
            if (tid < act)
#pragma unroll 1
                for (int q = (k0 ^ par) & 1; q < nk; q += 2) {
                    T r[NODES][NC];
                    T *const P = X0 + q * pl;
                    T *const h0 = q == 0 ? below : nullptr, *const h1 = q == ppc - 1 ? above : nullptr;
                    const T *b = B0 + q * pl;
                    if (zero && s == 0) {
#pragma unroll
                        for (int u = 0; u < NODES; u++)
                            if (node[u].colour >= 0)
                                get(b + node[u].r[1] + node[u].c[1] + comp[u], r[u]);
                    } else {
                        fold(c, b, P, r, pl);
                    }
                    // colours (F,F), (1-F,F), (F,1-F), (1-F,1-F) in (x, y) parity
#pragma unroll 1
                    for (int pass = 0; pass < 4; pass++) {
                        if (pass) sync_act();
                        const int colour = pass ^ (3 * F);
#pragma unroll
                        for (int u = 0; u < NODES; u++) {
                            if (node[u].colour != colour) continue;
                            T o[NC];
                            in_plane(c, P, u, o);
                            const int e = node[u].r[1] + node[u].c[1] + comp[u];
#pragma unroll
                            for (int a = 0; a < NC; a++)
                                o[a] = c.dinv[comp[u] + a] * (r[u][a] - o[a]);
                            put(P + e, o);
                            if constexpr (!COMP) {
                                if (h0) put(h0 + e, o);
                                if (h1) put(h1 + e, o);
                            }
                        }
                    }
                    // FP64: 16 bytes at a time after the passes, which takes less
                    // than scattered stores of the single components
                    if (COMP && (h0 || h1)) {
                        sync_act();
                        const float4 *src = reinterpret_cast<const float4 *>(P);
                        for (int e = tid; e < pl * (int)sizeof(T) / 16; e += act) {
                            const float4 v = src[e];
                            if (h0) reinterpret_cast<float4 *>(h0)[e] = v;
                            if (h1) reinterpret_cast<float4 *>(h1)[e] = v;
                        }
                    }
                    // the next plane's fold overwrites U and V: every thread
                    // is past reading them (three barriers ago)
                }
            cl.sync();
        }
    }

    // b of level l+1 = T^T (b - A x) of level l, and its x = 0
    __device__ __forceinline__ void restrict_residual(int l) {
        const SmallLevel &L = g.lev[l], &C = g.lev[l + 1];
        const Coarse<T> &c = g.op[l];
        const int nc3 = 3 * C.np, k0 = first(l), k1 = last(l);
        // on the finest level, whose residual limits what the cycles reach
        const bool shares = !COMP && g.fine && l == 0;
        T *R = sm + g.scratch;  // in place of U
        if (tid < act)
#pragma unroll 1
            for (int k = k0; k < k1; k++) {
                T r[NODES][NC];
                const T *P = own(l, L.x, k), *B = own(l, L.b, k);
                // the right-hand side last: it would lose digits to the
                // neighbour sums, which cancel with the centre term first
                if (shares)
                    fold<true, true>(c, B, P, r, L.pl);
                else
                    fold<true>(c, B, P, r, L.pl);
                sync_act();
#pragma unroll
                for (int u = 0; u < NODES; u++) {
                    if (node[u].colour < 0) continue;
                    T o[NC], b[NC];
                    const int q = node[u].r[1] + node[u].c[1] + comp[u];
                    if (shares) {
                        if constexpr (!COMP) plane_residual_at(c, P, node[u], o);
                    } else {
                        T x[NC];
                        in_plane(c, P, u, o);
                        get(P + q, x);
#pragma unroll
                        for (int a = 0; a < NC; a++) o[a] += c.cd[comp[u] + a][0] * x[a];
                    }
                    get(B + q, b);
#pragma unroll
                    for (int a = 0; a < NC; a++) o[a] = (r[u][a] - o[a]) + b[a];
                    put(R + q, o);
                }
                sync_act();
                // x and y parts of the full weighting
                T *p = sm + L.p + (k - k0) * C.pl;
                for (int e = tid; e < nc3; e += act) {
                    const int m = e / 3, a = e - 3 * m;
                    const int J = fdiv(m, C.mnx), I = m - J * C.nx;
                    constexpr int N = kNode<T>;
                    const int im = N * (L.hx + (I ? I - 1 : L.hx - 1)) + a, i0 = N * I + a,
                              ip = i0 + N * L.hx;
                    const T *r0 = R + 2 * J * L.w, *rm = R + (J ? 2 * J - 1 : L.ny - 1) * L.w,
                            *rp = r0 + L.w;
                    const T tm = (T(0.5) * rm[im] + rm[i0]) + T(0.5) * rm[ip];
                    const T t0 = (T(0.5) * r0[im] + r0[i0]) + T(0.5) * r0[ip];
                    const T tp = (T(0.5) * rp[im] + rp[i0]) + T(0.5) * rp[ip];
                    p[J * C.w + col_of<T>(C, I) + a] = (T(0.5) * tm + t0) + T(0.5) * tp;
                }
                sync_act();
            }
        cl.sync();
        // z part, gathered by the owner of each coarse plane (row padding
        // included: it is never used)
        for (int K = first(l + 1); K < last(l + 1); K++) {
            const T *p0 = plane(l, L.p, 2 * K - 1, C.pl), *p1 = plane(l, L.p, 2 * K, C.pl),
                    *p2 = plane(l, L.p, 2 * K + 1, C.pl);
            T *b = own(l + 1, C.b, K);
            for (int e = tid; e < C.pl; e += nt)
                b[e] = (T(0.5) * p0[e] + p1[e]) + T(0.5) * p2[e];
        }
        __syncthreads();
    }

    // x of level l, halos included, to zero: before a cycle reaches it, with
    // a cluster barrier between this and any store into its halos
    __device__ __forceinline__ void clear(int l) {
        const SmallLevel &L = g.lev[l];
        T *x = sm + L.x - L.pl;
        for (int e = tid; e < (L.ppc + 2) * L.pl; e += nt) x[e] = T(0);
    }

    // x of level l += T x of level l+1
    __device__ __forceinline__ void prolong(int l) {
        const SmallLevel &L = g.lev[l], &C = g.lev[l + 1];
        const int k0 = first(l), k1 = last(l);
        T *Z = sm + g.scratch;  // the coarse planes averaged to each own plane's z
        for (int k = k0; k < k1; k++) {
            const int K = k >> 1;
            const T *lo = K > 0 ? plane(l + 1, C.x, K, C.pl) : nullptr;
            const T *hi = (k & 1) ? (K + 1 < C.nz ? plane(l + 1, C.x, K + 1, C.pl) : nullptr) : lo;
            for (int e = tid; e < C.pl; e += nt)
                Z[(k - k0) * C.pl + e] = T(0.5) * ((lo ? lo[e] : T(0)) + (hi ? hi[e] : T(0)));
        }
        __syncthreads();
        T *const below = halo(l, 0), *const above = halo(l, 1);
        for (int e = tid; e < (k1 - k0) * L.np; e += nt) {
            const int p = fdiv(e, L.mnp), m = e - p * L.np;
            const int j = fdiv(m, L.mnx), i = m - j * L.nx;
            const int I = i >> 1, J = j >> 1;
            const int c0 = col_of<T>(C, I),
                      c1 = (i & 1) ? col_of<T>(C, I + 1 < C.nx ? I + 1 : 0) : c0;
            const T *z0 = Z + p * C.pl + J * C.w,
                    *z1 = (j & 1) ? Z + p * C.pl + (J + 1 < C.ny ? J + 1 : 0) * C.w : z0;
            const int q = j * L.w + col_of<T>(L, i);
            T *X = sm + L.x + p * L.pl + q;
            T v[3], z00[3], z01[3], z10[3], z11[3];
            load3(X, v);
            load3(z0 + c0, z00);
            load3(z0 + c1, z01);
            load3(z1 + c0, z10);
            load3(z1 + c1, z11);
#pragma unroll
            for (int a = 0; a < 3; a++)
                v[a] += T(0.25) * ((z00[a] + z01[a]) + (z10[a] + z11[a]));
            store3(X, v);
            if (below && p == 0) store3(below + q, v);
            if (above && p == L.ppc - 1) store3(above + q, v);
        }
        cl.sync();
        clear(l + 1);  // for the next cycle
    }

    // x = Ainv b on the coarsest level (x = 0 before): every CTA gathers b
    // and takes every 16th row, 16 lanes a row, FP64 sums in a fixed order.
    // The unknowns are ordered plane, node, component.
    __device__ __forceinline__ void coarsest() {
        const int l = g.nlev - 1;
        const SmallLevel &L = g.lev[l];
        const int n3 = 3 * L.np, lane = tid & 15, ng = nt >> 4, n = g.ncoarse;
        auto at = [](int m3) { return kNode<T> == 3 ? m3 : m3 + m3 / 3; };  // place in a plane
        double *v = reinterpret_cast<double *>(sm + g.scratch);
        // the first row's leading entries, loaded while b is on its way
        constexpr int PRE = 9;
        double pre[PRE];
        const int u0 = rank + kCta * (tid >> 4);
#pragma unroll
        for (int t = 0; t < PRE; t++) {
            const int q = lane + 16 * t;
            pre[t] = u0 < n && q < n ? __ldg(g.Ainv + (long)u0 * n + q) : 0.0;
        }
        cl.sync();
        for (int e = tid; e < n; e += nt) {
            const int K1 = fdiv(e, L.mn3);
            v[e] = (double)plane(l, L.b, K1 + 1, L.pl)[at(e - K1 * n3)];
        }
        __syncthreads();
        for (int t0 = 0; t0 < n; t0 += kCta * ng) {  // uniform: the shuffles need whole warps
            const int u = t0 + u0;
            const double *row = g.Ainv + (long)u * n;
            double acc = 0.0;
            if (u < n) {
                int q = lane;
                if (t0 == 0)
#pragma unroll
                    for (int t = 0; t < PRE; t++, q += 16)
                        if (q < n) acc += pre[t] * v[q];
#pragma unroll 4
                for (; q < n; q += 16) acc += __ldg(row + q) * v[q];
            }
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o, 16);
            if (lane == 0 && u < n) {
                const int K1 = fdiv(u, L.mn3);
                plane(l, L.x, K1 + 1, L.pl)[at(u - K1 * n3)] = (T)acc;
            }
        }
        cl.sync();
    }
};

template <typename T, int NODES, int MAXT>
__global__ void __launch_bounds__(MAXT, 1)
    k_small_cycle(const __grid_constant__ SmallPlan<T> g, const T *__restrict__ b, T *x,
                  int from_zero, int cycles) {
    extern __shared__ __align__(16) unsigned char smem_small[];
    Walker<T, NODES, sizeof(T) == 8> w{g, reinterpret_cast<T *>(smem_small), cg::this_cluster(),
                                       (int)cg::this_cluster().block_rank(), (int)threadIdx.x,
                                       (int)blockDim.x};
    const SmallLevel &L = g.lev[0];
    const long ps = L.np, cs = (long)(L.nz + 1) * ps;
    const int n3 = 3 * L.np, k0 = w.first(0), k1 = w.last(0);
    // b of the own planes; x of the own planes and of those around them
    for (int e = w.tid; e < (k1 > k0 ? k1 - k0 + 2 : 0) * n3; e += w.nt) {
        const int t = fdiv(e, L.mnp), m = e - t * L.np, q = t / 3, a = t - 3 * q;
        const int j = fdiv(m, L.mnx), i = m - j * L.nx, k = k0 - 1 + q;
        const int s = j * L.w + col_of<T>(L, i) + a;
        const long gq = a * cs + k * ps + m;
        w.own(0, L.x, k)[s] = from_zero ? T(0) : x[gq];
        if (k >= k0 && k < k1) w.own(0, L.b, k)[s] = b[gq];
    }
    for (int l = 1; l < g.nlev; l++) w.clear(l);
    w.cl.sync();
#pragma unroll 1
    for (int n = 0; n < cycles; n++) {
        // down (s < nlev - 1), then up: one code path for every level
        const int down = g.nlev - 1;
#pragma unroll 1
        for (int s = 0; s < 2 * down; s++) {
            const bool up = s >= down;
            const int l = up ? 2 * down - 1 - s : s;
            if (s == down) w.coarsest();
            if (up) w.prolong(l);
            w.enter(l);
            // below the top (and at the top of a first cycle from zero) x = 0
            const bool zero = !up && (l > 0 || (from_zero && n == 0));
            w.sweeps(l, up ? g.nu2 : g.nu1, up ? 1 : 0, zero);
            if (!up) w.restrict_residual(l);
        }
    }
    for (int e = w.tid; e < (k1 - k0) * n3; e += w.nt) {
        const int t = fdiv(e, L.mnp), m = e - t * L.np, q = t / 3, a = t - 3 * q;
        const int j = fdiv(m, L.mnx), i = m - j * L.nx;
        x[a * cs + (k0 + q) * ps + m] = w.own(0, L.x, k0 + q)[j * L.w + col_of<T>(L, i) + a];
    }
    // no CTA leaves while another may still store into its shared memory
    w.cl.sync();
}

inline unsigned magic(int d) { return d == 1 ? 0u : (unsigned)((1ull << 32) / (unsigned)d + 1); }

template <typename T>
void configure(const SmallPlan<T> &g, cudaLaunchConfig_t &cfg, cudaLaunchAttribute *attr,
               cudaStream_t s) {
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3(kCta);
    cfg.blockDim = dim3(g.threads);
    cfg.dynamicSmemBytes = g.smem;
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kCta;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
}

// The kernel's instantiations, smallest planes first: `most` is the largest
// plane (FP32: nodes, FP64: node components) and `nodes` of them go to a
// thread.  Few threads leave each more registers, which hold a level's
// constants and node offsets across its phases (16^3 step: 796 us with 128 of
// them against 870 with 64; steps whose top level here has planes of 40 x 20 and
// 24 x 24 nodes gain 1 and 2% from bounds of 832 and 640 instead of 1024); on
// 32 x 32 planes 512 threads with two nodes each also pass barriers sooner
// (64^3 solve 2.83 against 2.92 ms), on the smaller ones one node a thread
// stays faster.
template <typename T>
using SmallFn = void (*)(SmallPlan<T>, const T *, T *, int, int);
template <typename T>
struct SmallKernel {
    SmallFn<T> f;
    int most, nodes;
};
template <typename T>
const std::vector<SmallKernel<T>> &small_kernels();
template <>
const std::vector<SmallKernel<float>> &small_kernels() {
    static const std::vector<SmallKernel<float>> k = {
        {k_small_cycle<float, 1, 256>, 256, 1},
        {k_small_cycle<float, 1, 512>, 512, 1},
        {k_small_cycle<float, 1, 640>, 640, 1},
        {k_small_cycle<float, 1, 832>, 832, 1},
        {k_small_cycle<float, 2, 512>, 1024, 2},
        {k_small_cycle<float, kMaxNodes, 640>, 640 * kMaxNodes, kMaxNodes}};
    return k;
}
template <>
const std::vector<SmallKernel<double>> &small_kernels() {
    static const std::vector<SmallKernel<double>> k = {
        {k_small_cycle<double, 1, 256>, 256, 1},
        {k_small_cycle<double, 1, 768>, 768, 1}};
    return k;
}

// shared-memory layout of the plan; false if it does not fit
template <typename T>
bool small_layout(const Dims *d, const Coarse<T> *op, int nlev, SmallPlan<T> &g) {
    long off = 0;
    constexpr int N = kNode<T>;
    // nodes a shared-memory wavefront serves: eight of 16 bytes in FP32, the
    // banks of 16 elements three apart in FP64
    const int unit = N == 4 ? 8 : 16;
    for (int l = 0; l < nlev; l++) {
        SmallLevel &L = g.lev[l];
        g.op[l] = op[l];
        L.nx = d[l].nx;
        L.ny = d[l].ny;
        L.nz = d[l].nz;
        L.np = L.nx * L.ny;
        L.ppc = (L.nz - 1 + kCta - 1) / kCta;
        L.mnx = magic(L.nx);
        L.mnp = magic(L.np);
        L.mppc = magic(L.ppc);
        L.mn3 = magic(3 * L.np);
        L.w = N * L.nx;
        if (l + 1 < nlev) {
            L.hx = L.nx / 2;
            L.mhx = magic(L.hx);
            L.mnh = magic(L.np / 4);
            // two rows of a colour apart, as if its lanes went on in one row
            if (N == 4)
                while ((2 * (L.w / N) - L.hx) % unit > 1) L.w += N;
            else
                while ((2 * L.w - N * L.hx) % unit > 1) L.w++;
        }
        L.pl = L.ny * L.w;
        if (l + 1 < nlev) L.pl = (L.pl + 3) & ~3;  // planes are copied 16 bytes at a time
    }
    for (int l = 0; l < nlev; l++) {
        SmallLevel &L = g.lev[l];
        off = (off + 3) & ~3L;
        off += L.pl;  // the halo below the own planes
        L.x = (int)off;
        off += (long)(L.ppc + 1) * L.pl;  // and the one above
        L.b = (int)off;
        off += (long)L.ppc * L.pl;
        if (l + 1 < nlev) {
            L.p = (int)off;
            off += (long)L.ppc * g.lev[l + 1].pl;
        }
    }
    off = (off + 3) & ~3L;
    g.scratch = (int)off;
    g.plmax = g.lev[0].pl;
    for (int l = 1; l < nlev; l++) g.plmax = g.plmax < g.lev[l].pl ? g.lev[l].pl : g.plmax;
    long sc = 2L * g.plmax;  // U and V
    const long need_v = (long)g.ncoarse * (long)(sizeof(double) / sizeof(T));
    sc = sc < need_v ? need_v : sc;
    for (int l = 0; l + 1 < nlev; l++) {
        const long need_z = (long)g.lev[l].ppc * g.lev[l + 1].pl;
        sc = sc < need_z ? need_z : sc;
    }
    g.smem = (size_t)(off + sc) * sizeof(T);
    return g.smem <= kSmallSmem;
}

}  // namespace

// The plan for levels d[0 .. nlev-1] (d[nlev-1] solved densely), or false if
// they do not suit the kernel: at most kSmallCoarse unknowns on the coarsest
// level (a CTA takes every 16th row of its dense solve), planes that fit the
// cluster's shared memory and its threads (up to 32x32x48 nodes, planes of up to
// 2560), and at most `max_nodes` nodes on the top level (beyond it, the whole
// chip is faster than 16 SMs).
template <typename T>
bool small_plan(const Dims *d, const Coarse<T> *op, int nlev, int ncoarse, const double *Ainv,
                int nu1, int nu2, long max_nodes, SmallPlan<T> &g) {
    if (nlev < 2 || nlev > kSmallLevels || ncoarse > kSmallCoarse) return false;
    if ((long)d[0].nx * d[0].ny * d[0].nz > max_nodes) return false;
    g = SmallPlan<T>{};
    g.nlev = nlev;
    g.nu1 = nu1;
    g.nu2 = nu2;
    g.ncoarse = ncoarse;
    g.Ainv = Ainv;
    if (!small_layout(d, op, nlev, g)) return false;
    const int np = g.lev[0].np * (sizeof(T) == 8 ? 3 : 1);  // FP64: a thread a component
    g.nodes = 0;
    for (const SmallKernel<T> &k : small_kernels<T>()) {
        if (np > k.most) continue;
        g.kernel = (const void *)k.f;
        g.nodes = k.nodes;
        const int per = (np + k.nodes - 1) / k.nodes;
        g.threads = per < 128 ? 128 : (per + 31) / 32 * 32;
        break;
    }
    if (!g.nodes) return false;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    configure(g, cfg, attr, nullptr);
    int nc = 0;
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&nc, (SmallFn<T>)g.kernel, &cfg);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return nc > 0;
}

template <typename T>
cudaError_t small_cycle(const SmallPlan<T> &g, const T *b, T *x, bool from_zero, int cycles,
                        cudaStream_t s) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[1];
    configure(g, cfg, attr, s);
    const cudaError_t e =
        cudaLaunchKernelEx(&cfg, (SmallFn<T>)g.kernel, g, b, x, from_zero ? 1 : 0, cycles);
    count_launch();
    return e;
}

template bool small_plan<float>(const Dims *, const Coarse<float> *, int, int, const double *, int,
                                int, long, SmallPlan<float> &);
template bool small_plan<double>(const Dims *, const Coarse<double> *, int, int, const double *,
                                 int, int, long, SmallPlan<double> &);
template cudaError_t small_cycle<float>(const SmallPlan<float> &, const float *, float *, bool,
                                        int, cudaStream_t);
template cudaError_t small_cycle<double>(const SmallPlan<double> &, const double *, double *, bool,
                                         int, cudaStream_t);

template <typename T>
static cudaError_t small_attrs() {
    for (const SmallKernel<T> &k : small_kernels<T>()) {
        cudaError_t e =
            cudaFuncSetAttribute(k.f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k.f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)kSmallSmem);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t small_init() {
    const cudaError_t e = small_attrs<float>();
    return e == cudaSuccess ? small_attrs<double>() : e;
}

}  // namespace qsmg
