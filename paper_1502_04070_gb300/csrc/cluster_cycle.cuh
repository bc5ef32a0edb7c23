// cluster_cycle.cuh -- host interface of the cluster cycle of the small levels (cluster_cycle.cu).
#pragma once
#include <vector>

#include <cuda_runtime.h>

#include "common.cuh"
#include "stencil_tables.cuh"

namespace smg {

constexpr int kClusterTopMax = 5;        // highest level any precision takes (N = 64)
constexpr int kClusterMaxOps = 256;
constexpr int kClusterMaxNb = 532;       // bordered system of coarsest level 2
// highest level whose arrays fit the cluster's shared memory: N = 64 in float32, N = 32 in float64
template <typename T>
constexpr int cluster_top() { return sizeof(T) == 4 ? 5 : 4; }

// operations of a cycle: the pre-smoothing steps from an iterate known to be zero or from any, the
// post-smoothing steps, defect and restriction to the level below, the exact coarsest solve,
// prolongation from the level below, iterate := 0
enum : unsigned char { kOpPreZero = 0, kOpPre = 1, kOpPost = 2, kOpRestrict = 3, kOpCoarse = 4, kOpProlong = 5, kOpClear = 6 };
inline unsigned char cluster_op(int op, int level) { return (unsigned char)(op | level << 4); }

// What the kernel's threads sum (stencil_tables.cuh): offsets are those of the value from the cell's own in
// the level's arrays; unused entries are zero.
template <typename T>
struct alignas(16) LevelLists {
    E1<T> A[kStencilClasses][kListA];    // from list_start(s): 18 entries of V (21 at the centre), 9 of H, E, C
    E2<T> BT[kStencilClasses][kListBT];  // 4 of H, E, C (the V rows of B^T vanish)
    E2<T> B[kStencilClasses][kListB];    // 12 (16 at the centre)
    T ti[kStencilClasses][4];            // tau / diag A
};
template <typename T>
struct alignas(16) XferLists {           // offsets packed (xfer_off): they depend on the level's row length
    E1<T> R[kStencilClasses][63];        // restriction, by class of the coarse cell: 27 of V (36 at the centre), 9 each
    E1<T> P[2][16][5];                   // prolongation, by orientation of the coarse square and fine point 4 fb + fa
};
__host__ __device__ __forceinline__ int xfer_off(int o, int WH) { return (o >> 16) * WH + (int)(short)(o & 0xffff); }
template <typename T>
struct ClusterTables {
    XferLists<T> x;
    LevelLists<T> L[kClusterTopMax + 1]; // index = level
};
// host: the lists of a level with N = n, and of the transfers; false if a stencil has more entries than
// they hold (no level does)
template <typename T>
bool fill_cluster_level(LevelLists<T>& q, int n, const OpCoef<T>& c, T tau);
template <typename T>
bool fill_cluster_xfer(XferLists<T>& x);

template <typename T>
struct ClusterHost {
    T *u[kClusterTopMax + 1], *p[kClusterTopMax + 1], *f[kClusterTopMax + 1], *g[kClusterTopMax + 1];
    const T* sinv[kClusterTopMax + 1];
    const ClusterTables<T>* tab;         // device
    const double* inv0;                  // coarsest level 0: its 27 x 27 inverse
    const double* cinv;                  // coarsest level 1, 2: its dense inverse (cnb x cnb)
    int cnb;
    T sigma;
    int nu_pre, nu_post;
    int top, lo, dom;                    // levels lo (the coarsest of the iteration) .. top
};
// One launch of operations `ops` (at most kClusterMaxOps) on the levels' compact arrays; ld_x, ld_f,
// st_x, st_f: bit masks of the levels whose (u, p) / (f, g) are read before and written after.  An error
// if the arguments are out of range.
template <typename T>
cudaError_t launch_cluster_ops(cudaStream_t s, const ClusterHost<T>& h, const std::vector<unsigned char>& ops, unsigned ld_x,
                               unsigned ld_f, unsigned st_x, unsigned st_f);
// raises the kernel's limits on the current device; false: the device cannot hold one cluster
template <typename T>
bool prepare_cluster_cycle();
}  // namespace smg
