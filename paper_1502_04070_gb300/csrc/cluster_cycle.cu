// cluster_cycle.cu -- the multigrid cycle below a small level (Sec. 3) in one launch of one thread-block
// cluster, every array of those levels in the cluster's shared memory.
//
// A V-cycle visits a level in 21 dependent phases (three per Uzawa step, defect, restriction,
// prolongation) of a few thousand cells at most, so its time is the latency of a phase, not its
// arithmetic.  One launch per phase or step costs 9-15 us each; one CTA with all levels in its shared
// memory costs 3.4 us a phase (barriers of 1024 threads, one SM's shared-memory pipe).  Here the cell
// rows of the larger levels are split over the CTAs of a cluster (16 on levels with N >= 32, one cell a
// thread pair on N = 64), a CTA writes the rows its neighbours need straight into their shared memory, and
// the phases meet at the cluster's hardware barrier.  Levels with few cells are held and computed by
// every CTA alike, which needs the CTA's own barrier only.
//
// float64 runs the same code: an SM executes 2 float64 FMA per clock, so there the split also brings 16
// times the float64 units to a level, and only levels with N <= 8 are held by every CTA.
//
// What a thread computes: one velocity node (both components) or one vertex, as a list of (coefficient,
// offset) pairs that the host writes per level and stencil class from the merged stencils, zeros
// dropped: in every class, mid-lines included, 17 + 9 + 9 + 7 entries of A for the cell's nodes, 0 + 4 + 4 +
// 4 of B^T and 12 of B (a few more in the one cell at the centre); the transfers likewise (25 + 9 + 9 + 9 and at
// most 5).  One short loop serves all cells: straight-line code per class ran at the rate at which the
// instructions of its dozen kilobytes arrive (2,200 clocks for a phase of 16 cells against 900), and in
// float64 a warp instruction occupies its pipe for 64 clocks, so the work has to be spread over many
// warps.  Items are ordered node by node: the warps of a phase have the same number of entries.
//
// Measured (GB300, whole calls) against a launch per phase, or levels 0-4 in one CTA where that served: by this kernel
// alone a float64 V(3,3) cycle at h = 1/32 264 us against 1752 us and a mixed-precision solve with W-cycles at h = 1/512
// 37.6 against 64.0 ms; with what changed since 231 us and 34.2 ms, three implicit Euler steps there 25.7 against 51.6 ms.
// The float32 levels 1-5 take 91 us a V-cycle (105 phases; before, 283 us for levels 1-4 alone), the float64 levels 1-4
// 176 us (float64 pipe).
//
// A launch executes a list of operations that the host recursion writes: V- or W-cycle,
// coarsest level 0 (27 x 27 inverse), 1 or 2 (dense inverse, rows over the cluster).  With coarsest level
// 3 the dense solve needs the whole GPU (5 M float64 FMA): the list is cut there and the pieces pass
// the levels' state through global memory (L2).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include <cooperative_groups.h>

#include "cellops.cuh"
#include "cluster_cycle.cuh"
#include "elements.h"
#include "kernels.cuh"

namespace smg {
namespace {

constexpr int kNT = 512;                 // threads per CTA
constexpr int kNW = kNT / 32;
// smooth() gives a thread kNodes velocity nodes and one vertex of a level, the launch one entry of Shat^{-1}
constexpr int kNodes = 2;
static_assert(4 * 4 * 64 <= kNodes * kNT && 5 * 65 <= kNT && 4 * 16 * 16 <= kNodes * kNT && 17 * 17 <= kNT,
              "N = 64 in 16 parts, N = 16 whole");

// ---- placement: cell rows of a level in a CTA, and the byte offsets of its arrays
template <typename T>
__host__ __device__ constexpr int rep_n() { return sizeof(T) == 4 ? 16 : 8; }   // levels with N <= this: every CTA alike

struct Place {
    int n, rp;                           // cells per side; cell rows per CTA (the last CTA also holds row n)
    bool dist;
    int WH, RS, VW;                      // pairs per plane row, per lattice row; vertices per row
    unsigned u, th, f, p, dp, g, s, end; // byte offsets
};
template <typename T>
__host__ __device__ inline Place place(int l, int P, unsigned base) {
    Place L;
    L.n = 2 << l;
    L.dist = P > 1 && L.n > rep_n<T>();
    L.rp = L.dist ? L.n / P : L.n;
    L.WH = L.n + 3;
    L.RS = 2 * L.WH;
    L.VW = L.n + 3;
    const unsigned z2 = 2 * (unsigned)sizeof(T), z = (unsigned)sizeof(T);
    auto al = [](unsigned b) { return (b + 15u) & ~15u; };
    L.u = base;
    L.th = L.u + al(z2 * 2 * (L.rp + 3) * L.RS);
    L.p = L.th + al(z2 * 2 * (L.rp + 4) * L.RS);
    L.dp = L.p + al(z * (L.rp + 3) * L.VW);
    L.f = L.dp + al(z * (L.rp + 3) * L.VW);
    L.g = L.f + al(z2 * 2 * L.rp * 2 * L.n);
    L.s = L.g + al(z * (L.rp + 1) * (L.n + 1));
    L.end = L.s + al(z * (L.rp + 1) * (L.n + 1));
    return L;
}
// shared memory: the dense solve's right-hand side, the level-0 inverse, the transfers' lists, the lists of
// levels lo + 1 .. top, then the levels' arrays
constexpr unsigned kOffInv = 8u * (unsigned)kClusterMaxNb, kOffXfer = kOffInv + 8u * 27 * 27 + 8u;
static_assert(kOffXfer % 16 == 0, "the lists are copied in 16-byte units");
template <typename T>
__host__ __device__ inline unsigned fixed_bytes(int lo, int top) {
    return kOffXfer + (unsigned)sizeof(XferLists<T>) + (unsigned)sizeof(LevelLists<T>) * (unsigned)(top - lo);
}
template <typename T>
unsigned smem_bytes(int lo, int top, int P) {
    unsigned b = fixed_bytes<T>(lo, top);
    for (int l = lo; l <= top; ++l) b = place<T>(l, P, b).end;
    return b;
}

template <typename T>
struct Args {
    const ClusterTables<T>* tab;         // device
    T *u[kClusterTopMax + 1], *p[kClusterTopMax + 1], *f[kClusterTopMax + 1], *g[kClusterTopMax + 1];
    const T* sinv[kClusterTopMax + 1];
    const double* inv0;                  // level-0 bordered inverse (27 x 27)
    const double* cinv;                  // coarsest level c > 0: its bordered inverse, cnb x cnb
    int cnb;
    T sigma;
    int top, lo, dom;
    unsigned ld_x, ld_f, st_x, st_f;     // levels whose (u, p) / (f, g) are read at the start / written at the end
    Place pl[kClusterTopMax + 1];
    int nu_pre, nu_post, nops;
    unsigned char ops[kClusterMaxOps];   // operation | level << 4
};

// ---- cluster primitives
__device__ __forceinline__ unsigned cl_rank() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ unsigned cl_size() {
    unsigned r;
    asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
    return r;
}
// every thread of every CTA of the cluster; orders shared (and global) writes before it with reads after
__device__ __forceinline__ void cl_sync() { cooperative_groups::this_cluster().sync(); }
__device__ __forceinline__ unsigned cl_map(unsigned a, unsigned rank) {
    unsigned r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void st_cl(unsigned a, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ void st_cl(unsigned a, double v) { asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory"); }
__device__ __forceinline__ void st_cl(unsigned a, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void st_cl(unsigned a, double2 v) {
    asm volatile("st.shared::cluster.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}

// ---- pairs (x, y)
__device__ __forceinline__ float2 mk(float x, float y) { return make_float2(x, y); }
__device__ __forceinline__ double2 mk(double x, double y) { return make_double2(x, y); }
__device__ __forceinline__ float2 pfma(float c, float2 v, float2 s) { return __ffma2_rn(make_float2(c, c), v, s); }
__device__ __forceinline__ double2 pfma(double c, double2 v, double2 s) { return make_double2(fma(c, v.x, s.x), fma(c, v.y, s.y)); }

// One level as the phases see it.  Arrays: velocity pairs by lattice row and column parity, lattice
// point (X, Y) at (Y - 2 row0) RS + (X & 1) WH + (X >> 1) + 1, with a zero column on each side and, from cell
// row r0 - 1 (th: r0 - 2), the neighbours' rows; vertex arrays likewise; f, g, Shat^{-1} own rows only.
template <typename T>
struct Lev {
    using P2 = typename Vec2<T>::type;
    int n, lgh, rp, r0, r1, rv, WH, RS, VW;   // own cell rows [r0, r1), of which rv hold unknown nodes
    bool dist;
    int rank, P, dom;
    T sigma;
    P2 *u, *th, *f;
    T *p, *dp, *g, *s;
    const LevelLists<T>* q;
    const XferLists<T>* x;
    __device__ __forceinline__ P2* uat(int i, int j) const { return u + (2 * (j - r0 + 1)) * RS + i + 1; }   // cell (i, j)
    __device__ __forceinline__ P2* that(int i, int j) const { return th + (2 * (j - r0 + 2)) * RS + i + 1; }
    __device__ __forceinline__ T* pat(int i, int j) const { return p + (j - r0 + 1) * VW + i + 1; }
    __device__ __forceinline__ T* dpat(int i, int j) const { return dp + (j - r0 + 1) * VW + i + 1; }
    __device__ __forceinline__ P2* fat(int i, int j) const { return f + (j - r0) * 4 * n + i; }   // then plane +n, row +2n
    __device__ __forceinline__ int gat(int i, int j) const { return (j - r0) * (n + 1) + i; }
    __device__ __forceinline__ void sync() const {
        if (dist) cl_sync();
        else __syncthreads();
    }
    // v at d (an entry of cell row j) and in the neighbours' copies of that row: HI rows above, LO below;
    // rows are `rowb` bytes apart and a neighbour numbers the same row rp rows away
    template <int LO, typename V>
    __device__ __forceinline__ void put(V* d, int j, int rowb, V v) const {
        *d = v;
        if (dist) {
            const unsigned a = (unsigned)__cvta_generic_to_shared(d);
            if (j == r0 && rank > 0) st_cl(cl_map(a + rp * rowb, rank - 1), v);
            if (j >= r1 - LO && rank + 1 < P) st_cl(cl_map(a - rp * rowb, rank + 1), v);
            if (LO == 2 && rp == 1 && rank + 2 < P) st_cl(cl_map(a - 2 * rp * rowb, rank + 2), v);
        }
    }
};

// acc + sum over N list entries of coefficient times the value at its offset from c
template <int N, typename T, typename P2>
__device__ __forceinline__ P2 list_sum(const E1<T>* e, const P2* c, P2 acc) {
    E1<T> t[N];
#pragma unroll
    for (int w = 0; w < N; ++w) t[w] = e[w];
    P2 v[N];
#pragma unroll
    for (int w = 0; w < N; ++w) v[w] = c[t[w].o];
#pragma unroll
    for (int w = 0; w < N; ++w) acc = pfma(t[w].c, v[w], acc);
    return acc;
}
// the A row of node s: 18 entries of V (and 3 more in the one cell at the centre: a branch of its own, so
// that the other lanes' sum stays one straight line), 9 of the others
template <typename T, typename P2>
__device__ __forceinline__ P2 a_sum(const E1<T>* e, int s, bool centre, const P2* c) {
    P2 acc = list_sum<9, T, P2>(e, c, mk(T(0), T(0)));
    if (s == 0) {
        acc = list_sum<9, T, P2>(e + 9, c, acc);
        if (centre) acc = list_sum<3, T, P2>(e + 18, c, acc);
    }
    return acc;
}
template <int N, typename T, typename P2>
__device__ __forceinline__ void b_sum(const E2<T>* e, const P2* c, T& bx, T& by) {
    E2<T> t[N];
#pragma unroll
    for (int w = 0; w < N; ++w) t[w] = e[w];
#pragma unroll
    for (int w = 0; w < N; ++w) {
        const P2 v = c[t[w].o];
        bx = fma(t[w].cx, v.x, bx);
        by = fma(t[w].cy, v.y, by);
    }
}
// B u at the vertex of a cell of class k (c: the cell's entry of u)
template <typename T, typename P2>
__device__ __forceinline__ T bu_sum(const E2<T>* e, bool centre, const P2* c) {
    T bx = T(0), by = T(0);
    b_sum<6>(e, c, bx, by);
    b_sum<6>(e + 6, c, bx, by);
    if (centre) b_sum<4>(e + 12, c, bx, by);
    return bx + by;
}
template <typename T>
__device__ __forceinline__ typename Vec2<T>::type bt_sum(const E2<T>* e, const T* p) {
    typename Vec2<T>::type acc = mk(T(0), T(0));
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const E2<T> t = e[v];
        const T q = p[t.o];
        acc = mk(fma(t.cx, q, acc.x), fma(t.cy, q, acc.y));
    }
    return acc;
}
// Velocity work items of a level: node s of cell (i, j), all V first, then H, E, C (the cell rows and
// columns are powers of two); false for nodes that are not unknowns.
template <typename T>
__device__ __forceinline__ bool item_node(const Lev<T>& L, int it, int lc, int& i, int& j, int& s) {
    s = it >> lc;
    const int r = it & ((1 << lc) - 1);
    i = r & (L.n - 1);
    j = L.r0 + (r >> (L.lgh + 1));
    const int X = 2 * i + (s & 1), Y = 2 * j + (s >> 1);
    return X > 0 && Y > 0 && !(L.dom == kDomL && l_masked_node(X, Y, L.n));
}
// vertices of the own rows: columns 0 .. N - 1, then column N
template <typename T>
__device__ __forceinline__ void item_vertex(const Lev<T>& L, int it, int rows, int& i, int& j) {
    const int cells = rows * L.n;
    const bool edge = it >= cells;
    i = edge ? L.n : it & (L.n - 1);
    j = L.r0 + (edge ? it - cells : it >> (L.lgh + 1));
}
template <typename T>
__device__ __forceinline__ int log_cells(const Lev<T>& L) { return 31 - __clz(L.rv * L.n); }

// ---- `steps` Uzawa steps (zero: from u = 0, p = 0, whatever the arrays hold).  A thread owns the same
// nodes (at most kNodes) and the same vertex in every phase and step: its right-hand side, u, u^{m-1/2} and p stay in
// registers.
template <typename T>
__device__ __forceinline__ void smooth(const Lev<T>& L, int steps, bool zero) {
    using P2 = typename Vec2<T>::type;
    const int lc = log_cells(L), rowb = 2 * L.RS * (int)sizeof(P2), vrowb = L.VW * (int)sizeof(T);
    struct Node {
        bool live, centre;
        int s, j;
        P2 *u, *th;          // the node's own entries
        const P2* cu;        // the cell's
        const T *p, *dp;
        const E1<T>* a;
        const E2<T>* bt;
        P2 f, x, h;          // right-hand side, u, u^{m-1/2}
        T ti;
    } nd[kNodes];
#pragma unroll
    for (int q = 0; q < kNodes; ++q) {
        const int it = threadIdx.x + q * kNT;
        int i, j, s;
        nd[q].live = it < 4 << lc && item_node(L, it, lc, i, j, s);
        if (!nd[q].live) continue;
        const int k = stencil_class(i, j, L.n), off = (s & 1) * L.WH + (s >> 1) * L.RS;
        nd[q].centre = k == 6;
        nd[q].s = s;
        nd[q].j = j;
        nd[q].cu = L.uat(i, j);
        nd[q].u = L.uat(i, j) + off;
        nd[q].th = L.that(i, j) + off;
        nd[q].p = L.pat(i, j);
        nd[q].dp = L.dpat(i, j);
        nd[q].a = L.q->A[k] + list_start(s);
        nd[q].bt = L.q->BT[k] + 4 * (s - 1);
        nd[q].f = L.fat(i, j)[(s & 1) * L.n + (s >> 1) * 2 * L.n];
        nd[q].ti = L.q->ti[k][s];
        nd[q].x = *nd[q].u;
    }
    const int rows = L.r1 - L.r0;
    const bool vlive = (int)threadIdx.x < rows * (L.n + 1);
    int vi = 0, vj = L.r0;
    if (vlive) item_vertex(L, threadIdx.x, rows, vi, vj);
    const int vk = stencil_class(vi, vj, L.n), vg = L.gat(vi, vj);
    const T ss = L.sigma * L.s[vg], g = L.g[vg];
    T p = zero ? T(0) : *L.pat(vi, vj);
    for (int m = 0; m < steps; ++m) {
        // u^{m-1/2} = u + tau Ahat^{-1} (f - A u - B^T p)
#pragma unroll
        for (int q = 0; q < kNodes; ++q) {
            if (!nd[q].live) continue;
            if (zero && m == 0) {
                nd[q].h = mk(nd[q].ti * nd[q].f.x, nd[q].ti * nd[q].f.y);
            } else {
                P2 t = a_sum<T, P2>(nd[q].a, nd[q].s, nd[q].centre, nd[q].cu);
                if (nd[q].s > 0) {
                    const P2 b = bt_sum<T>(nd[q].bt, nd[q].p);
                    t = mk(t.x + b.x, t.y + b.y);
                }
                nd[q].h = pfma(nd[q].ti, mk(nd[q].f.x - t.x, nd[q].f.y - t.y), nd[q].x);
            }
            L.template put<1>(nd[q].th, nd[q].j, rowb, nd[q].h);
        }
        L.sync();
        // dp = sigma Shat^{-1} (B u^{m-1/2} - g), p += dp
        if (vlive) {
            const T d = ss * (bu_sum<T, P2>(L.q->B[vk], vk == 6, L.that(vi, vj)) - g);
            p += d;
            L.template put<1>(L.dpat(vi, vj), vj, vrowb, d);
            L.template put<1>(L.pat(vi, vj), vj, vrowb, p);
        }
        L.sync();
        // u = u^{m-1/2} - tau Ahat^{-1} B^T dp
#pragma unroll
        for (int q = 0; q < kNodes; ++q) {
            if (!nd[q].live) continue;
            nd[q].x = nd[q].s > 0 ? pfma(-nd[q].ti, bt_sum<T>(nd[q].bt, nd[q].dp), nd[q].h) : nd[q].h;
            L.template put<1>(nd[q].u, nd[q].j, rowb, nd[q].x);
        }
        L.sync();
    }
}

// ---- the defect: r_u = f - A u - B^T p into th, g - B u into dp (no synchronisation inside)
template <typename T>
__device__ __forceinline__ void defect_phase(const Lev<T>& L) {
    using P2 = typename Vec2<T>::type;
    const int lc = log_cells(L);
    for (int it = threadIdx.x; it < 4 << lc; it += kNT) {
        int i, j, s;
        if (!item_node(L, it, lc, i, j, s)) continue;
        const int k = stencil_class(i, j, L.n);
        const P2 f = L.fat(i, j)[(s & 1) * L.n + (s >> 1) * 2 * L.n];
        P2 t = a_sum<T, P2>(L.q->A[k] + list_start(s), s, k == 6, L.uat(i, j));
        if (s > 0) {
            const P2 b = bt_sum<T>(L.q->BT[k] + 4 * (s - 1), L.pat(i, j));
            t = mk(t.x + b.x, t.y + b.y);
        }
        L.template put<2>(L.that(i, j) + (s & 1) * L.WH + (s >> 1) * L.RS, j, 2 * L.RS * (int)sizeof(P2),
                          mk(f.x - t.x, f.y - t.y));
    }
    const int rows = L.r1 - L.r0, items = rows * (L.n + 1);
    for (int it = kNT - 1 - (int)threadIdx.x; it < items; it += kNT) {
        int i, j;
        item_vertex(L, it, rows, i, j);
        const int k = stencil_class(i, j, L.n);
        const T bu = bu_sum<T, P2>(L.q->B[k], k == 6, L.uat(i, j));
        const bool live = !(L.dom == kDomL && l_masked_vertex(i, j, L.n));
        L.template put<1>(L.dpat(i, j), j, L.VW * (int)sizeof(T), live ? L.g[L.gat(i, j)] - bu : T(0));
    }
}

// Restriction of the defect (th, dp of F) into (f, g) of C; the CTA that holds the fine row 2J forms
// coarse row J, for every CTA if C is held by all of them.
template <int N, typename T, typename P2>
__device__ __forceinline__ P2 xfer_sum(const E1<T>* e, int WH, const P2* c, P2 acc) {
#pragma unroll
    for (int w = 0; w < N; ++w) {
        const E1<T> t = e[w];
        acc = pfma(t.c, c[xfer_off(t.o, WH)], acc);
    }
    return acc;
}
template <typename T, typename V>
__device__ __forceinline__ void store_coarse(const Lev<T>& F, const Lev<T>& C, V* d, V v) {
    if (F.dist && !C.dist) {
        const unsigned a = (unsigned)__cvta_generic_to_shared(d);
        for (int r = 0; r < F.P; ++r) st_cl(cl_map(a, r), v);
    } else {
        *d = v;
    }
}
template <typename T>
__device__ __forceinline__ void restrict_phase(const Lev<T>& F, const Lev<T>& C) {
    using P2 = typename Vec2<T>::type;
    const int nc = C.n;
    const int ja = F.dist ? (F.r0 + 1) >> 1 : 0, jb = F.dist ? (F.r1 + 1) >> 1 : nc + 1;   // coarse rows [ja, jb)
    const int cells = (min(jb, nc) - ja) * nc;                                             // 0 or a power of two
    const int lc = cells > 0 ? 31 - __clz(cells) : 0;
    for (int it = threadIdx.x; it < 4 * cells; it += kNT) {
        const int s = it >> lc, r = it & (cells - 1);
        const int I = r & (nc - 1), J = ja + (r >> (C.lgh + 1));
        const int X = 2 * I + (s & 1), Y = 2 * J + (s >> 1);
        if (X == 0 || Y == 0 || (F.dom == kDomL && l_masked_node(X, Y, nc))) continue;
        const int k = stencil_class(I, J, nc);
        const E1<T>* e = F.x->R[k] + (s == 0 ? 0 : 27 + 9 * s);
        const P2* c = F.that(2 * I, 2 * J);
        P2 acc = xfer_sum<9, T, P2>(e, F.WH, c, mk(T(0), T(0)));
        if (s == 0) {
            acc = xfer_sum<9, T, P2>(e + 9, F.WH, c, acc);
            acc = xfer_sum<9, T, P2>(e + 18, F.WH, c, acc);
            if (k == 6) acc = xfer_sum<9, T, P2>(e + 27, F.WH, c, acc);
        }
        store_coarse(F, C, C.fat(I, J) + (s & 1) * nc + (s >> 1) * 2 * nc, acc);
    }
    // P1: the fine vertex at the coarse one, and halves of those halfway along the coarse edges through it
    const int nv = (jb - ja) * (nc + 1);
    for (int it = kNT - 1 - (int)threadIdx.x; it < nv; it += kNT) {
        const int J = ja + it / (nc + 1), I = it % (nc + 1);
        const T* r = F.dpat(2 * I, 2 * J);
        T half = r[-1] + r[1] + r[-F.VW] + r[F.VW];   // zero outside the domain
        if (I < nc && J < nc && orient(I, J, nc) == 0) half += r[F.VW + 1];
        if (I > 0 && J > 0 && orient(I - 1, J - 1, nc) == 0) half += r[-F.VW - 1];
        if (I < nc && J > 0 && orient(I, J - 1, nc) == 1) half += r[-F.VW + 1];
        if (I > 0 && J < nc && orient(I - 1, J, nc) == 1) half += r[F.VW - 1];
        const T v = (F.dom == kDomL && l_masked_vertex(I, J, nc)) ? T(0) : fma(T(0.5), half, r[0]);
        store_coarse(F, C, C.g + C.gat(I, J), v);
    }
}

// Prolongation and correction: (u, p) of F += I (u, p) of C, one fine node or vertex a thread (nodes by
// their place in the coarse square).
template <typename T>
__device__ __forceinline__ void prolong_phase(const Lev<T>& F, const Lev<T>& C) {
    using P2 = typename Vec2<T>::type;
    const int nc = C.n, n = F.n;
    const bool one = F.rv == 1;                       // a single fine row: half of a row of coarse squares
    const int ls = 31 - __clz((one ? 1 : F.rv >> 1) * nc);
    for (int it = threadIdx.x; it < (one ? 8 : 16) << ls; it += kNT) {
        const int pt = it >> ls, r = it & ((1 << ls) - 1);
        const int fa = pt & 3, fb = (pt >> 2) + (one ? 2 * (F.r0 & 1) : 0);
        const int I = r & (nc - 1), J = (F.r0 >> 1) + (r >> (C.lgh + 1));
        const int X = 4 * I + fa, Y = 4 * J + fb;
        if (X == 0 || Y == 0 || (F.dom == kDomL && l_masked_node(X, Y, n))) continue;
        const E1<T>* e = F.x->P[orient(I, J, nc)][4 * fb + fa];
        const P2* z = C.uat(I, J);
        const P2 acc = xfer_sum<5, T, P2>(e, C.WH, z, mk(T(0), T(0)));
        P2* d = F.uat(X >> 1, Y >> 1) + (X & 1) * F.WH + (Y & 1) * F.RS;
        const P2 o = *d;
        F.template put<1>(d, Y >> 1, 2 * F.RS * (int)sizeof(P2), mk(o.x + acc.x, o.y + acc.y));
    }
    const int rows = F.r1 - F.r0, items = rows * (n + 1);
    for (int it = kNT - 1 - (int)threadIdx.x; it < items; it += kNT) {
        int x, y;
        item_vertex(F, it, rows, x, y);
        if (F.dom == kDomL && l_masked_vertex(x, y, n)) continue;
        const int I = x >> 1, J = y >> 1;
        const T* c = C.pat(I, J);
        T v;
        if (!(x & 1)) v = (y & 1) ? T(0.5) * (c[0] + c[C.VW]) : c[0];
        else if (!(y & 1)) v = T(0.5) * (c[0] + c[1]);
        else v = T(0.5) * (orient(I, J, nc) == 0 ? c[0] + c[C.VW + 1] : c[1] + c[C.VW]);
        T* d = F.pat(x, y);
        F.template put<1>(d, y, F.VW * (int)sizeof(T), *d + v);
    }
}

// ---- exact solves on the coarsest level (float64)
template <typename T>
__device__ __forceinline__ T* u_entry(const Lev<T>& L, int c, int X, int Y) {
    return reinterpret_cast<T*>(L.uat(X >> 1, Y >> 1) + (X & 1) * L.WH + (Y & 1) * L.RS) + c;
}
template <typename T>
__device__ __forceinline__ T f_entry(const Lev<T>& L, int c, int X, int Y) {
    return reinterpret_cast<const T*>(L.fat(X >> 1, Y >> 1) + (X & 1) * L.n + (Y & 1) * 2 * L.n)[c];
}
// level 0: 27 unknowns (see elements.cpp), the same in every CTA
template <typename T>
__device__ __forceinline__ void coarse0_phase(const Lev<T>& L, const double* inv, double* b) {
    const int t = threadIdx.x;
    if (t < 27) b[t] = t < 18 ? (double)f_entry(L, t / 9, 1 + t % 9 % 3, 1 + t % 9 / 3) : (double)L.g[t - 18];
    __syncthreads();
    if (t < 27) {
        double x = 0.0;
#pragma unroll
        for (int s = 0; s < 27; ++s) x = fma(inv[t * 27 + s], b[s], x);
        if (t < 18) *u_entry(L, t / 9, 1 + t % 9 % 3, 1 + t % 9 / 3) = (T)x;
        else *L.pat((t - 18) % 3, (t - 18) / 3) = (T)x;
    }
    __syncthreads();
}
// levels 1, 2 (held by every CTA): one warp per row of the dense inverse, rows over the whole cluster,
// each result written to every CTA
template <typename T>
__device__ __forceinline__ void dense_phase(const Lev<T>& L, const double* __restrict__ inv, int nb, double* b) {
    const int nm = 2 * L.n - 1, nv = nm * nm, nunk = nb - 1, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int t = threadIdx.x; t < nunk; t += kNT) {
        const int c = t / nv, r = t - c * nv;
        b[t] = c < 2 ? (double)f_entry(L, c, 1 + r % nm, 1 + r / nm) : (double)L.g[t - 2 * nv];
    }
    cl_sync();   // and no CTA reads the previous solution any more
    for (int row = L.rank * kNW + warp; row < nunk; row += L.P * kNW) {
        const double* m = inv + (size_t)row * nb;
        double x = 0.0;
        for (int t = lane; t < nunk; t += 32) x = fma(__ldg(m + t), b[t], x);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        const int c = row / nv, r = row - c * nv;
        T* d = c < 2 ? u_entry(L, c, 1 + r % nm, 1 + r / nm) : L.pat((row - 2 * nv) % (L.n + 1), (row - 2 * nv) / (L.n + 1));
        const unsigned a = (unsigned)__cvta_generic_to_shared(d);
        for (int k = lane; k < L.P; k += 32) st_cl(cl_map(a, k), (T)x);
    }
    cl_sync();
}

template <typename T>
__device__ __forceinline__ Lev<T> level(const Args<T>& A, const Place* pl, unsigned char* sm, int l, int rank, int P) {
    using P2 = typename Vec2<T>::type;
    const Place& q = pl[l];
    Lev<T> L;
    L.n = q.n;
    L.lgh = l;                           // N / 2 = 2^l
    L.rp = q.rp;
    L.dist = q.dist;
    L.r0 = q.dist ? rank * q.rp : 0;
    L.r1 = (!q.dist || rank == P - 1) ? q.n + 1 : L.r0 + q.rp;
    L.rv = q.rp;
    L.WH = q.WH;
    L.RS = q.RS;
    L.VW = q.VW;
    L.rank = rank;
    L.P = P;
    L.dom = A.dom;
    L.sigma = A.sigma;
    L.u = reinterpret_cast<P2*>(sm + q.u);
    L.th = reinterpret_cast<P2*>(sm + q.th);
    L.f = reinterpret_cast<P2*>(sm + q.f);
    L.p = reinterpret_cast<T*>(sm + q.p);
    L.dp = reinterpret_cast<T*>(sm + q.dp);
    L.g = reinterpret_cast<T*>(sm + q.g);
    L.s = reinterpret_cast<T*>(sm + q.s);
    L.x = reinterpret_cast<const XferLists<T>*>(sm + kOffXfer);
    L.q = reinterpret_cast<const LevelLists<T>*>(sm + kOffXfer + sizeof(XferLists<T>)) + (l - A.lo - 1);   // none for level lo
    return L;
}

template <typename T>
__global__ void __launch_bounds__(kNT, 1) k_cluster_cycle(const __grid_constant__ Args<T> A) {
    using P2 = typename Vec2<T>::type;
    extern __shared__ __align__(16) unsigned char sm[];
    __shared__ Place pl[kClusterTopMax + 1];
    const int rank = (int)cl_rank(), P = (int)cl_size(), tid = threadIdx.x;
    double* rhs = reinterpret_cast<double*>(sm);
    double* inv0 = reinterpret_cast<double*>(sm + kOffInv);
    // what does not depend on earlier launches: the zero borders, the coefficients, Shat^{-1}
    const unsigned fixed = fixed_bytes<T>(A.lo, A.top);
    for (int k = tid; k < (int)(sizeof(pl) / 4); k += kNT) reinterpret_cast<int*>(pl)[k] = reinterpret_cast<const int*>(A.pl)[k];
    {
        // the lists (the transfers', then those of levels lo + 1 .. top), all loads in flight at once
        constexpr int xw = (int)(sizeof(XferLists<T>) / 16), lw = (int)(sizeof(LevelLists<T>) / 16);
        const int nw = xw + lw * (A.top - A.lo);
        const uint4 *xs = reinterpret_cast<const uint4*>(&A.tab->x), *ls = reinterpret_cast<const uint4*>(&A.tab->L[A.lo + 1]);
        uint4* dst = reinterpret_cast<uint4*>(sm + kOffXfer);
#pragma unroll 8
        for (int k = tid; k < nw; k += kNT) dst[k] = __ldg(k < xw ? xs + k : ls + (k - xw));
        const unsigned words = (A.pl[A.top].end - fixed) / 16;
        uint4* z = reinterpret_cast<uint4*>(sm + fixed);
        for (unsigned k = tid; k < words; k += kNT) z[k] = make_uint4(0u, 0u, 0u, 0u);
        T sv[kClusterTopMax];                // at most one vertex per thread and level
#pragma unroll
        for (int m = 0; m < kClusterTopMax; ++m) {
            const int l = A.lo + 1 + m;
            if (l <= A.top) {
                const int n = A.pl[l].n, r0 = A.pl[l].dist ? rank * A.pl[l].rp : 0;
                const int rows = (!A.pl[l].dist || rank == P - 1) ? n + 1 - r0 : A.pl[l].rp;
                if (tid < rows * (n + 1)) sv[m] = __ldg(A.sinv[l] + r0 * (n + 1) + tid);
            }
        }
        if (A.lo == 0)
            for (int k = tid; k < 27 * 27; k += kNT) inv0[k] = __ldg(A.inv0 + k);
        __syncthreads();
#pragma unroll
        for (int m = 0; m < kClusterTopMax; ++m) {
            const int l = A.lo + 1 + m;
            if (l <= A.top) {
                const int n = pl[l].n, r0 = pl[l].dist ? rank * pl[l].rp : 0;
                const int rows = (!pl[l].dist || rank == P - 1) ? n + 1 - r0 : pl[l].rp;
                if (tid < rows * (n + 1)) reinterpret_cast<T*>(sm + pl[l].s)[tid] = sv[m];
            }
        }
    }
    pdl_wait();
    for (int l = A.lo; l <= A.top; ++l) {
        const Lev<T> L = level(A, pl, sm, l, rank, P);
        const int n = L.n, ld = 2 * n + 1, n2 = ld * ld;
        if ((A.ld_f >> l) & 1u) {
            const int cnt = L.rv * 2 * 2 * n;     // own lattice rows, columns 0 .. 2N - 1
            for (int k = tid; k < cnt; k += kNT) {
                const int X = k & (2 * n - 1), y = k / (2 * n), s = (2 * L.r0 + y) * ld + X;
                L.f[y * 2 * n + (X & 1) * n + (X >> 1)] = mk(A.f[l][s], A.f[l][n2 + s]);
            }
            const int vc = (L.r1 - L.r0) * (n + 1);
            for (int k = tid; k < vc; k += kNT) L.g[k] = A.g[l][L.r0 * (n + 1) + k];
        }
        if ((A.ld_x >> l) & 1u) {
            const int cnt = (L.rp + 3) * 2 * 2 * n;   // the neighbours' rows too; off the boundary only
            for (int k = tid; k < cnt; k += kNT) {
                const int X = k & (2 * n - 1), y = k / (2 * n), Y = 2 * (L.r0 - 1) + y, s = Y * ld + X;
                if (Y > 0 && Y < 2 * n && Y < 2 * (L.r1 + 1) && X > 0)
                    L.u[y * L.RS + (X & 1) * L.WH + (X >> 1) + 1] = mk(A.u[l][s], A.u[l][n2 + s]);
            }
            const int vc = (L.rp + 3) * (n + 1);
            for (int k = tid; k < vc; k += kNT) {
                const int J = L.r0 - 1 + k / (n + 1), I = k % (n + 1);
                if (J >= 0 && J <= n && J <= L.r1) *L.pat(I, J) = A.p[l][J * (n + 1) + I];
            }
        }
    }
    cl_sync();

    for (int k = 0; k < A.nops; ++k) {
        const int op = A.ops[k] & 15, l = A.ops[k] >> 4;
        const Lev<T> L = level(A, pl, sm, l, rank, P);
        if (op <= kOpPost) {
            smooth(L, op == kOpPost ? A.nu_post : A.nu_pre, op == kOpPreZero);
        } else if (op == kOpRestrict) {
            const Lev<T> C = level(A, pl, sm, l - 1, rank, P);
            defect_phase(L);
            L.sync();
            restrict_phase(L, C);
            L.sync();
        } else if (op == kOpProlong) {
            const Lev<T> C = level(A, pl, sm, l - 1, rank, P);
            prolong_phase(L, C);
            L.sync();
        } else if (op == kOpClear) {
            for (int t = tid; t < (L.rp + 3) * 2 * L.RS; t += kNT) L.u[t] = mk(T(0), T(0));
            for (int t = tid; t < (L.rp + 3) * L.VW; t += kNT) L.p[t] = T(0);
            L.sync();
        } else if (l == 0) {
            coarse0_phase(L, inv0, rhs);
        } else {
            dense_phase(L, A.cinv, A.cnb, rhs);
        }
    }

    for (int l = A.lo; l <= A.top; ++l) {
        const Lev<T> L = level(A, pl, sm, l, rank, P);
        if (!L.dist && rank > 0) continue;
        const int n = L.n, ld = 2 * n + 1, n2 = ld * ld;
        const int rows = 2 * L.rv + (L.r1 == n + 1 ? 1 : 0);   // lattice rows, the last one with row 2N
        if ((A.st_x >> l) & 1u) {
            for (int k = tid; k < rows * ld; k += kNT) {
                const int y = k / ld, X = k - y * ld;
                const P2 v = L.u[(y + 2) * L.RS + (X & 1) * L.WH + (X >> 1) + 1];
                A.u[l][2 * L.r0 * ld + k] = v.x;
                A.u[l][n2 + 2 * L.r0 * ld + k] = v.y;
            }
            for (int k = tid; k < (L.r1 - L.r0) * (n + 1); k += kNT)
                A.p[l][L.r0 * (n + 1) + k] = *L.pat(k % (n + 1), L.r0 + k / (n + 1));
        }
        if ((A.st_f >> l) & 1u) {
            for (int k = tid; k < 2 * L.rv * 2 * n; k += kNT) {
                const int X = k & (2 * n - 1), y = k / (2 * n);
                const P2 v = L.f[y * 2 * n + (X & 1) * n + (X >> 1)];
                A.f[l][(2 * L.r0 + y) * ld + X] = v.x;
                A.f[l][n2 + (2 * L.r0 + y) * ld + X] = v.y;
            }
            for (int k = tid; k < (L.r1 - L.r0) * (n + 1); k += kNT) A.g[l][L.r0 * (n + 1) + k] = L.g[k];
        }
    }
    pdl_trigger();
}

}  // namespace

namespace {
constexpr int kClusterCTAs = 16;         // beyond the portable 8: twice the SMs per level, one GPC per cluster
}

template <typename T>
cudaError_t launch_cluster_ops(cudaStream_t s, const ClusterHost<T>& h, const std::vector<unsigned char>& ops, unsigned ld_x,
                               unsigned ld_f, unsigned st_x, unsigned st_f) {
    if (h.top > cluster_top<T>() || h.lo < 0 || h.lo >= h.top || (int)ops.size() > kClusterMaxOps)
        return cudaErrorInvalidValue;
    for (unsigned char o : ops)   // the dense inverse of a larger level is not this kernel's
        if ((o & 15) == kOpCoarse && h.lo > 0 && h.cnb - 1 > kClusterMaxNb) return cudaErrorInvalidValue;
    static_assert(sizeof(Args<T>) <= 4096, "kernel parameters");
    Args<T> A{};
    A.tab = h.tab;
    for (int l = h.lo; l <= h.top; ++l) {
        A.u[l] = h.u[l];
        A.p[l] = h.p[l];
        A.f[l] = h.f[l];
        A.g[l] = h.g[l];
        A.sinv[l] = h.sinv[l];
    }
    A.inv0 = h.inv0;
    A.cinv = h.cinv;
    A.cnb = h.cnb;
    A.sigma = h.sigma;
    A.top = h.top;
    A.lo = h.lo;
    A.dom = h.dom;
    A.ld_x = ld_x;
    A.ld_f = ld_f;
    A.st_x = st_x;
    A.st_f = st_f;
    A.nu_pre = h.nu_pre;
    A.nu_post = h.nu_post;
    A.nops = (int)ops.size();
    std::memcpy(A.ops, ops.data(), ops.size());
    // every level small enough to be held by every CTA: one CTA
    const int P = (2 << h.top) > rep_n<T>() ? kClusterCTAs : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(P);
    cfg.blockDim = dim3(kNT);
    unsigned end = fixed_bytes<T>(h.lo, h.top);
    for (int l = h.lo; l <= h.top; ++l) {
        A.pl[l] = place<T>(l, P, end);
        end = A.pl[l].end;
    }
    cfg.dynamicSmemBytes = end;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = P;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl_enabled() ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, k_cluster_cycle<T>, A);
}

template <typename T>
bool prepare_cluster_cycle() {
    unsigned bytes = smem_bytes<T>(0, cluster_top<T>(), kClusterCTAs);
    // (coarsest levels above 0 hold fewer levels, one-CTA launches only the small ones)
    for (int lo = 0; lo < cluster_top<T>(); ++lo)
        for (int top = lo + 1; top <= cluster_top<T>(); ++top)
            bytes = std::max(bytes, smem_bytes<T>(lo, top, (2 << top) > rep_n<T>() ? kClusterCTAs : 1));
    bool ok = cudaFuncSetAttribute(k_cluster_cycle<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
              cudaFuncSetAttribute(k_cluster_cycle<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess;
    if (ok) {
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(kClusterCTAs);
        cfg.blockDim = dim3(kNT);
        cfg.dynamicSmemBytes = bytes;
        cudaLaunchAttribute at[1];
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = kClusterCTAs;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        cfg.attrs = at;
        cfg.numAttrs = 1;
        int clusters = 0;
        ok = cudaOccupancyMaxActiveClusters(&clusters, k_cluster_cycle<T>, &cfg) == cudaSuccess && clusters > 0;
    }
    if (!ok) cudaGetLastError();
    return ok;
}

template <typename T>
bool fill_cluster_level(LevelLists<T>& q, int n, const OpCoef<T>& c, T tau) {
    const int WH = n + 3, RS = 2 * WH, VW = n + 3;   // as in place()
    const ListStructure& S = list_structure();
    q = LevelLists<T>{};
    auto off = [&](int w) {
        const int dx = w % 5 - 2, dy = w / 5 - 2;
        return dy * RS + (dx & 1) * WH + (dx >> 1);
    };
    for (int k = 0; k < kStencilClasses; ++k) {
        for (int s = 0; s < 4; ++s) {
            q.ti[k][s] = tau * c.MIdg[k][s];
            for (int m = list_start(s); m < (s < 3 ? list_start(s + 1) : kListA); ++m)
                if (const int w = S.A[k][m]; w >= 0) q.A[k][m] = E1<T>{c.MA[k][s][w], off(w)};
            for (int m = 4 * (s - 1); s > 0 && m < 4 * s; ++m)
                if (const int v = S.BT[k][m]; v >= 0)
                    q.BT[k][m] = E2<T>{c.MBTx[k][s][v], c.MBTy[k][s][v], (v / 3 - 1) * VW + v % 3 - 1};
        }
        for (int m = 0; m < kListB; ++m)
            if (const int w = S.B[k][m]; w >= 0) q.B[k][m] = E2<T>{c.MBx[k][w], c.MBy[k][w], off(w)};
    }
    return S.ok;
}

template <typename T>
bool fill_cluster_xfer(XferLists<T>& x) {
    x = XferLists<T>{};
    auto pack = [](int dx, int dy) { return ((2 * dy + (dx & 1)) << 16) | ((dx >> 1) & 0xffff); };
    const TransferWeights t = transfer_weights();
    for (int k = 0; k < kStencilClasses; ++k)
        for (int s = 0; s < 4; ++s) {
            int m = 0;
            const int cap = s == 0 ? 36 : 9;
            for (int dy = -4; dy < 4; ++dy)
                for (int dx = -4; dx < 4; ++dx) {   // fine point (4I + dx, 4J + dy), owned by one coarse square
                    const int SQ = (dx < 0 ? 1 : 0) + (dy < 0 ? 2 : 0), L = sq_local(SQ, s);
                    if (L < 0) continue;
                    const double w = t.P2[sq_orient(k, SQ)][L][dy + 4 * (SQ >> 1)][dx + 4 * (SQ & 1)];
                    if (w == 0.0) continue;
                    if (m == cap) return false;
                    x.R[k][(s == 0 ? 0 : 27 + 9 * s) + m++] = E1<T>{(T)w, pack(dx, dy)};
                }
            if (s == 0 && k != 6 && m > 27) return false;
        }
    for (int o = 0; o < 2; ++o)
        for (int pt = 0; pt < 16; ++pt) {
            int m = 0;
            for (int L = 0; L < 9; ++L) {
                const double w = t.P2[o][L][pt / 4][pt % 4];
                if (w == 0.0) continue;
                if (m == 5) return false;
                x.P[o][pt][m++] = E1<T>{(T)w, pack(L % 3, L / 3)};
            }
        }
    return true;
}

template cudaError_t launch_cluster_ops<float>(cudaStream_t, const ClusterHost<float>&, const std::vector<unsigned char>&,
                                               unsigned, unsigned, unsigned, unsigned);
template cudaError_t launch_cluster_ops<double>(cudaStream_t, const ClusterHost<double>&, const std::vector<unsigned char>&,
                                                unsigned, unsigned, unsigned, unsigned);
template bool prepare_cluster_cycle<float>();
template bool prepare_cluster_cycle<double>();
template bool fill_cluster_level<float>(LevelLists<float>&, int, const OpCoef<float>&, float);
template bool fill_cluster_level<double>(LevelLists<double>&, int, const OpCoef<double>&, double);
template bool fill_cluster_xfer<float>(XferLists<float>&);
template bool fill_cluster_xfer<double>(XferLists<double>&);

}  // namespace smg
