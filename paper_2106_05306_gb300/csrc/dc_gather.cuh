// Element and node kernels by component: helpers shared by the forward local step and the
// adjoint's operator.
#pragma once

#include "dc_internal.h"

// Meshes of at most this many triangles / nodes take three lanes for each in the element
// and node kernels (Lane3), larger ones one thread.  The split halves a lane's chain of
// FP64 instructions and triples the lanes, so it pays while the chip's schedulers have at
// most about one warp each.  Measured, one thread -> three lanes (us): local step 256 nodes
// 11.7 -> 6.0, 3721 nodes 8.1 -> 8.0, 161000 nodes 102 -> 109; right-hand side 11.9 -> 8.1,
// 12.4 -> 9.1, 31.7 -> 39.8; 10000 nodes (triangles on one thread) 15.0 -> 13.3 and 13.2 ->
// 9.6; the adjoint's element and node kernels 9.3 -> 6.4 and 12.9 -> 9.8 at 256 nodes, 7.0 ->
// 6.9 and 13.3 -> 10.2 at 3721.
constexpr int DC_SPLIT_TRIS = 8000;
constexpr int DC_SPLIT_NODES = 20000;
// Threads for n items, three lanes or one thread each (whole warps).
inline int dc_group_threads(int n, bool split) { return split ? (n + 9) / 10 * 32 : (n + 31) / 32 * 32; }

// Element and node kernels on groups of three lanes, one per component, ten groups to a
// warp (lanes 30 and 31 idle).  A warp's FP64 instruction takes its scheduler 64 cycles
// whatever its lanes do, so a lane's chain of instructions is its time while the chip is
// not full: a component per lane cuts the chain to what the components share.
struct Lane3 {
    int group, c, base;                // item within the warp, component, first lane of the group
    bool on;
    __device__ __forceinline__ Lane3() {
        const int lane = threadIdx.x & 31;
        group = lane / 3;
        c = lane - 3 * group;
        base = 3 * group;
        on = lane < 30;
    }
    // the group's three values of x
    __device__ __forceinline__ void all(double x, double v[3]) const {
#pragma unroll
        for (int k = 0; k < 3; ++k) v[k] = __shfl_sync(0xffffffffu, x, (base + k) & 31);
    }
};
__device__ __forceinline__ double comp(const d4* p, int i, int c) {
    return reinterpret_cast<const double*>(p)[4 * (long)i + c];
}
__device__ __forceinline__ double& comp(d4* p, int i, int c) { return reinterpret_cast<double*>(p)[4 * (long)i + c]; }

// Row sum over a list, one component: sum_k val[k] v[idx[k]].c in list order, the entries
// of four terms loaded together.
template <class F>
__device__ __forceinline__ void list4(int lo, int hi, const int* __restrict__ idx, const double* __restrict__ val, F f) {
    for (int k = lo; k < hi; k += 4) {
        int j[4];
        double l[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int e = min(k + q, hi - 1);
            j[q] = idx[e];
            l[q] = val[e];
        }
        f(k, j, l);
    }
}

// Component c of the element pass's contributions to node i, added to r in list order:
// the triangles' columns (vertex 0: minus the sum of the two stored ones), then the
// bending rows.  Four entries at a time, their loads together: a node's list is two
// dependent loads per entry, which is what a small mesh's gather waits for.
__device__ __forceinline__ double dc_gather_elements(const DevMesh& dm, int i, int c, double r,
                                                     const d4* __restrict__ c1, const d4* __restrict__ c2,
                                                     const d4* __restrict__ bu) {
    const int lo = dm.iptr[i], hi = dm.iptr[i + 1], blo = dm.tbptr[i], bhi = dm.tbptr[i + 1];
    for (int k = lo; k < hi; k += 4) {
        int a[4];
        double x[4], y[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) a[q] = dm.iidx[min(k + q, hi - 1)];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int t = a[q] / 3;
            a[q] -= 3 * t;
            x[q] = a[q] != 2 ? comp(c1, t, c) : 0.0;
            y[q] = a[q] != 1 ? comp(c2, t, c) : 0.0;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (k + q < hi) {
                const double z = x[q] + y[q];
                r += a[q] == 0 ? -z : z;
            }
    }
    list4(blo, bhi, dm.tbidx, dm.tbval, [&](int k, const int j[4], const double l[4]) {
        double u[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) u[q] = comp(bu, j[q], c);
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (k + q < bhi) r += l[q] * u[q];
    });
    return r;
}
