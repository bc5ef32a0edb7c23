// stencil_tables.cuh -- the merged stencils as their kernels use them: the compile-time structure of the orientation
// classes 0 and 1 and the values that a level fills it with (uzawa_reg.cu, coefficients in registers), the weights of
// the canonical embedding (uzawa_reg.cu, kernels.cu), and the entries of every class as lists (cluster_cycle.cu and the
// mid-line tiles of uzawa_reg.cu).
#pragma once
#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace smg {

// ---------------------------------------------------------------------------------------------
// Structure of the merged stencils of the orientation classes 0 and 1 (common.cuh), by window
// point w = (dy + 2) * 5 + dx + 2 of the 5 x 5 lattice window around the cell's vertex (2i, 2j)
// and owned node s (0 V, 1 H, 2 E, 3 C):
//   kGid[cls][s][w]  group of the A coefficient (-1: zero); every group holds one value
//   kBx / kBy[cls][w]  the vertex's B row in units of b/2 (values 0, +-1, +-2)
//   kBTx / kBTy[cls][s][v]  the B^T rows over the 3 x 3 vertex window v = (dj + 1) * 3 + di + 1,
//                           in units of b/2
constexpr int kGroups = 8;
constexpr int kGidDiagV = 4, kGidDiagE = 7;   // groups of the diagonal of the V row and of the H, E, C rows
constexpr signed char kGid[2][4][25] = {
    {{0, 1, 2, -1, -1, 1, -1, 3, 1, -1, 2, 3, 4, 3, 2, -1, 1, 3, -1, 1, -1, -1, 2, 1, 0},
     {-1, -1, 1, -1, -1, -1, -1, 5, 6, -1, -1, -1, 3, 7, 3, -1, -1, -1, 6, 5, -1, -1, -1, -1, 1},
     {-1, -1, -1, -1, -1, -1, -1, -1, -1, -1, 1, 5, 3, -1, -1, -1, 6, 7, 6, -1, -1, -1, 3, 5, 1},
     {-1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, 6, 1, -1, -1, 6, 7, 6, -1, -1, 1, 6, -1}},
    {{-1, -1, 0, 1, 2, -1, 1, 3, -1, 1, 0, 3, 4, 3, 0, 1, -1, 3, 1, -1, 2, 1, 0, -1, -1},
     {-1, -1, -1, -1, 1, -1, -1, -1, 5, 6, -1, -1, 3, 7, 3, -1, -1, 6, 5, -1, -1, -1, 1, -1, -1},
     {-1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, 3, 6, 1, -1, 5, 7, 5, -1, 1, 6, 3, -1, -1},
     {-1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, -1, 1, 5, -1, -1, -1, 5, 7, 5, -1, -1, -1, 5, 1}}};
constexpr signed char kBx[2][25] = {
    {0, 0, 0, 0, 0, -1, -1, 1, 1, 0, 0, -2, 0, 2, 0, 0, -1, -1, 1, 1, 0, 0, 0, 0, 0},
    {0, 0, 0, 0, 0, 0, -1, -1, 1, 1, 0, -2, 0, 2, 0, -1, -1, 1, 1, 0, 0, 0, 0, 0, 0}};
constexpr signed char kBy[2][25] = {
    {0, -1, 0, 0, 0, 0, -1, -2, -1, 0, 0, 1, 0, -1, 0, 0, 1, 2, 1, 0, 0, 0, 0, 1, 0},
    {0, 0, 0, -1, 0, 0, -1, -2, -1, 0, 0, -1, 0, 1, 0, 0, 1, 2, 1, 0, 0, 1, 0, 0, 0}};
constexpr signed char kBTx[2][4][9] = {
    {{0, 0, 0, 0, 0, 0, 0, 0, 0}, {0, 0, 0, 0, 2, -2, 0, 0, 0}, {0, 0, 0, 1, -1, 0, 0, 1, -1}, {0, 0, 0, 0, 1, -1, 0, 1, -1}},
    {{0, 0, 0, 0, 0, 0, 0, 0, 0}, {0, 0, 0, 0, 2, -2, 0, 0, 0}, {0, 0, 0, 0, 1, -1, 1, -1, 0}, {0, 0, 0, 0, 1, -1, 0, 1, -1}}};
constexpr signed char kBTy[2][4][9] = {
    {{0, 0, 0, 0, 0, 0, 0, 0, 0}, {0, 1, 0, 0, -1, 1, 0, 0, -1}, {0, 0, 0, 0, 2, 0, 0, -2, 0}, {0, 0, 0, 0, 1, 1, 0, -1, -1}},
    {{0, 0, 0, 0, 0, 0, 0, 0, 0}, {0, 0, 1, 0, 1, -1, 0, -1, 0}, {0, 0, 0, 0, 2, 0, 0, -2, 0}, {0, 0, 0, 0, 1, 1, 0, -1, -1}}};

__host__ __device__ constexpr bool a_win(int C, int w) {
    return kGid[C][0][w] >= 0 || kGid[C][1][w] >= 0 || kGid[C][2][w] >= 0 || kGid[C][3][w] >= 0;
}
__host__ __device__ constexpr bool bt_vwin(int C, int v) {
    for (int s = 0; s < 4; ++s)
        if (kBTx[C][s][v] != 0 || kBTy[C][s][v] != 0) return true;
    return false;
}

// Values of the structure above for one level
struct RegVals {
    float a[2][kGroups];   // A group values, per class
    float ti[2][2];        // tau / diag A: [class][0 = V row, 1 = H, E, C rows]
    float b;               // B = (b / 2) x (the integer tables)
};

// Fills q from the level's merged stencils and checks that they have exactly the compile-time
// structure (zeros, equal groups, B entries +-b, +-b/2) up to rounding; false if not (the caller then
// uses kernels that take the stencils as they are).
inline bool make_reg_vals(const OpCoef<float>& c, float tau, RegVals& q) {
    constexpr double tol = 1e-6;
    double amax = 0.0, bmax = 0.0;
    for (int C = 0; C < 2; ++C) {
        for (int s = 0; s < 4; ++s)
            for (int w = 0; w < 25; ++w) amax = std::max(amax, std::fabs((double)c.MA[C][s][w]));
        for (int w = 0; w < 25; ++w) bmax = std::max({bmax, std::fabs((double)c.MBx[C][w]), std::fabs((double)c.MBy[C][w])});
    }
    if (!(amax > 0.0) || !(bmax > 0.0)) return false;
    const double b = bmax;
    for (int C = 0; C < 2; ++C) {
        bool set[kGroups] = {};
        for (int s = 0; s < 4; ++s)
            for (int w = 0; w < 25; ++w) {
                const double v = c.MA[C][s][w];
                const int gid = kGid[C][s][w];
                if (gid < 0) {
                    if (std::fabs(v) > tol * amax) return false;
                    continue;
                }
                if (!set[gid]) {
                    q.a[C][gid] = (float)v;
                    set[gid] = true;
                } else if (std::fabs(v - (double)q.a[C][gid]) > tol * std::fabs(v) + 0.1 * tol * amax) {
                    return false;
                }
            }
        for (int g = 0; g < kGroups; ++g)
            if (!set[g]) return false;
        for (int w = 0; w < 25; ++w)
            if (std::fabs(c.MBx[C][w] - 0.5 * b * kBx[C][w]) > tol * b ||
                std::fabs(c.MBy[C][w] - 0.5 * b * kBy[C][w]) > tol * b)
                return false;
        for (int s = 0; s < 4; ++s)
            for (int v = 0; v < 9; ++v)
                if (std::fabs(c.MBTx[C][s][v] - 0.5 * b * kBTx[C][s][v]) > tol * b ||
                    std::fabs(c.MBTy[C][s][v] - 0.5 * b * kBTy[C][s][v]) > tol * b)
                    return false;
        // the diagonal groups are the stored inverse diagonals
        if (std::fabs(1.0 / q.a[C][kGidDiagV] - c.MIdg[C][0]) > tol * std::fabs(c.MIdg[C][0])) return false;
        for (int s = 1; s < 4; ++s)
            if (std::fabs(1.0 / q.a[C][kGidDiagE] - c.MIdg[C][s]) > tol * std::fabs(c.MIdg[C][s])) return false;
        q.ti[C][0] = tau * c.MIdg[C][0];
        q.ti[C][1] = tau * c.MIdg[C][1];
    }
    q.b = (float)b;
    return true;
}

// acc += (k / 2) v with a compile-time k in {0, +-1, +-2}
template <int K>
__device__ __forceinline__ void addk(float& acc, float v) {
    if constexpr (K == 2) acc += v;
    else if constexpr (K == -2) acc -= v;
    else if constexpr (K == 1) acc = fmaf(0.5f, v, acc);
    else if constexpr (K == -1) acc = fmaf(-0.5f, v, acc);
}

// ---- the canonical embedding (Sec. 3)
// the two triangles of a coarse square of orientation o (the split of tri_mask), vertices in coarse
// lattice units (0 or 2)
struct EmbedTri {
    int x[3], y[3];
};
__host__ __device__ constexpr EmbedTri embed_tri(int o, int t) {
    return o == 0 ? (t == 0 ? EmbedTri{{0, 2, 2}, {0, 0, 2}} : EmbedTri{{0, 2, 0}, {0, 2, 2}})
                  : (t == 0 ? EmbedTri{{0, 2, 0}, {0, 0, 2}} : EmbedTri{{2, 2, 0}, {0, 2, 2}});
}
// Value at the fine lattice point (fa / 2, fb / 2), fa, fb in [0, 4), of the coarse P2 basis
// function of local node L (lattice offset (L % 3, L / 3)): in the triangle that holds the point,
// with barycentric coordinates l, l_i (2 l_i - 1) at vertex i and 4 l_j l_k at the midpoint of the
// edge (j, k); zero where L is no node of that triangle.  Evaluated at compile time.
__host__ __device__ constexpr double embed_weight(int o, int L, int fa, int fb) {
    const double px = 0.5 * fa, py = 0.5 * fb;
    const int lx = L % 3, ly = L / 3;
    for (int t = 0; t < 2; ++t) {
        const EmbedTri T = embed_tri(o, t);
        const double twoA = (T.x[1] - T.x[0]) * (T.y[2] - T.y[0]) - (T.x[2] - T.x[0]) * (T.y[1] - T.y[0]);
        double l[3] = {0.0, 0.0, 0.0};
        bool inside = true;
        for (int i = 0; i < 3; ++i) {
            const int j = (i + 1) % 3, k = (i + 2) % 3;
            l[i] = ((T.x[j] - px) * (T.y[k] - py) - (T.x[k] - px) * (T.y[j] - py)) / twoA;
            if (l[i] < 0.0) inside = false;
        }
        if (!inside) continue;
        for (int i = 0; i < 3; ++i)
            if (T.x[i] == lx && T.y[i] == ly) return l[i] * (2.0 * l[i] - 1.0);
        for (int i = 0; i < 3; ++i) {
            const int j = (i + 1) % 3, k = (i + 2) % 3;
            if (T.x[j] + T.x[k] == 2 * lx && T.y[j] + T.y[k] == 2 * ly) return 4.0 * l[j] * l[k];
        }
        return 0.0;
    }
    return 0.0;
}
__host__ __device__ constexpr bool embed_partition_of_unity() {
    for (int o = 0; o < 2; ++o)
        for (int f = 0; f < 16; ++f) {
            double s = 0.0;
            for (int L = 0; L < 9; ++L) s += embed_weight(o, L, f % 4, f / 4);
            if (s != 1.0) return false;
        }
    return true;
}
static_assert(embed_partition_of_unity(), "the coarse basis functions sum to one at every fine point");
static_assert(embed_weight(0, 0, 1, 0) == 0.375 && embed_weight(0, 1, 1, 0) == 0.75 && embed_weight(0, 2, 1, 0) == -0.125,
              "on a coarse edge the embedding is the quadratic through its three nodes");
static_assert(embed_weight(1, 4, 2, 2) == 1.0 && embed_weight(0, 3, 2, 2) == 0.0, "a coarse node keeps its value");

// ---- the merged stencils of every class as lists (for kernels that sum them entry by entry)
template <typename T>
struct alignas(2 * sizeof(T)) E1 {   // coefficient and an offset
    T c;
    int o;
};
template <typename T>
struct alignas(16) E2 {              // the x and the y coefficient and an offset
    T cx, cy;
    int o;
};
// In every class, mid-lines included, the nodes V, H, E, C of a cell have 17 + 9 + 9 + 7 entries of A and 0 + 4 + 4 + 4
// of B^T, its vertex has 12 of B; the one cell at the centre (class 6) has 21 of A at V and 16 of B.
__host__ __device__ constexpr int list_start(int s) { return s == 0 ? 0 : 18 + 9 * s; }
constexpr int kListA = 54, kListBT = 12, kListB = 16;   // per class: 27 + 9 + 9 + 9, 4 + 4 + 4, 16

// Which entries there are (window points, -1: none), from the masks of common.cuh.  (Not from a level's own
// coefficients: at small beta h^2 the entries that only the mass has are tiny, and yet they count; leaving them
// out below 1e-6 of the largest made float32 W-cycles a hundred times less accurate.)
struct ListStructure {
    signed char A[kStencilClasses][kListA], BT[kStencilClasses][kListBT], B[kStencilClasses][kListB];
    bool ok = true;
};
inline const ListStructure& list_structure() {
    static const ListStructure S = [] {
        ListStructure r;
        for (int k = 0; k < kStencilClasses; ++k) {
            for (auto& v : r.A[k]) v = -1;
            for (auto& v : r.BT[k]) v = -1;
            for (auto& v : r.B[k]) v = -1;
            for (int s = 0; s < 4; ++s) {
                int m = 0;
                for (int w = 0; w < 25; ++w)
                    if (nz_MA(k, s, w)) {
                        if (m == (s == 0 ? (k == 6 ? 21 : 18) : 9)) r.ok = false;
                        else r.A[k][list_start(s) + m++] = (signed char)w;
                    }
                m = 0;
                for (int v = 0; v < 9; ++v)
                    if (nz_MBT(k, s, v)) {
                        if (s == 0 || m == 4) r.ok = false;
                        else r.BT[k][4 * (s - 1) + m++] = (signed char)v;
                    }
            }
            int m = 0;
            for (int w = 0; w < 25; ++w)
                if (nz_MB(k, w)) {
                    if (m == (k == 6 ? 16 : 12)) r.ok = false;
                    else r.B[k][m++] = (signed char)w;
                }
        }
        return r;
    }();
    return S;
}

}  // namespace smg
