// Numeric factorisation of the adjoint preconditioner's fronts (single precision
// LDL^T, see dc_frontal.cu for the matrix and the solves), one tree level at a
// time, leaves first.
//
// What bounds it: an SM does about 0.5 TFLOP/s of FP32, and a front's pivot
// columns are a serial chain, so a front on one CTA is slow however wide the CTA
// (the 1200-unknown root of a 200x200 cloth took 65 ms that way).  Each level is
// therefore a sequence of launches over tiles of all its fronts:
//   extend   -- adds the children's update blocks into the level's fronts, one CTA
//               per 64 x 64 tile of the parent's lower triangle;
//   panel k  -- 32 pivot columns of every front that has them: each CTA factorises
//               and inverts the 32 x 32 diagonal block (again: it is small, and
//               recomputing it is cheaper than a launch or a wait between CTAs) and
//               solves FF_ROWS of the rows below it, one row per thread in registers;
//   update k -- the rank-32 update of the trailing lower triangle: 128 x 64 tiles on
//               the tensor cores (tcgen05, TF32 split in three passes, FP32
//               accumulation) on levels with fronts of 160 unknowns or more while 64
//               rows are left, else 64 x 64 tiles of FP32 FMAs;
//   inverse  -- X = L_ss^-1 of every pivot block (the solves multiply by it), one CTA
//               per 32 columns (fewer for pivot blocks of more than 1536 unknowns).
// The tile lists depend only on the fronts' sizes and are laid out once by
// ff_plan.  Every entry's arithmetic depends only on its own front and its level's
// choice of update, and its order is that of one CTA per front taking the panels in
// turn.
//
// Measured (device time of one factorisation, the launches one by one and cold under the
// profiler; before: one CTA per front): one 200x200 cloth 118 ms -> 6.0 ms, one 61x61
// cloth 4.1 -> 1.3 ms, 96 cloths of 16x16..64x64 9.5 -> 5.4 ms.
#include <algorithm>
#include <cstdlib>
#include <mutex>
#include <string>
#include <vector>

#include "dc_adjoint.h"
#include "dc_internal.h"
#include "dc_tc.cuh"

namespace {

constexpr int PB = 32;                     // panel width
constexpr int FF_PT = 160;                 // threads of a panel CTA: one warp on the diagonal block, one on its inverse
constexpr int FF_ROWS = FF_PT - 64;        // rows below it per CTA
constexpr int FF_TILE = 64;                // tile of the extend-add and of the updates
constexpr int LSS = 36;                    // row stride of the diagonal block in shared memory (16-byte rows)
// Tensor-core update: 128 x TC_N accumulator tiles in TMEM, operands in shared memory
// (A: 128 rows, B: TC_N rows, each as TF32 hi and lo parts).
constexpr int TC_M = 128;
constexpr int TC_N = 64;
constexpr uint32_t TC_COLS = 64;                          // TMEM columns per CTA
constexpr int TC_A_BYTES = TC_M * TC_K * 4;               // one part of A
constexpr int TC_B_BYTES = TC_N * TC_K * 4;               // one part of B
constexpr int TC_BYTES = 2 * TC_A_BYTES + 2 * TC_B_BYTES;
constexpr int TC_MIN_N2 = 64;                             // smaller trailing blocks: FMA tiles
constexpr int TC_MIN_F = 160;                             // levels with smaller fronts: FMA tiles
constexpr int TC_WAIT = 1 << 22;                          // polls of an MMA completion

// Adds the children's update blocks into one tile of a front (children in
// order).  A tile's rows and columns are looked up in the child's position map
// (increasing), which is staged in shared memory.
__global__ void __launch_bounds__(256) k_ff_extend(FrontDev fd, const int2* __restrict__ tasks) {
    extern __shared__ int smap[];
    __shared__ int idx[2][FF_TILE];        // child index of each tile row / column, -1: none
    const int2 task = tasks[blockIdx.x];
    const int s = task.x, r0 = (task.y >> 16) * FF_TILE, c0 = (task.y & 0xffff) * FF_TILE;
    const int f = fd.f[s];
    const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
    float* F = fd.pool + fd.off[s];
    float acc[2][8];
    bool touched = false;
    for (int q = fd.cptr[s]; q < fd.cptr[s + 1]; ++q) {
        const int c = fd.child[q];
        const int fc = fd.f[c], pc = fd.p[c], nn = (fc - pc) / 3;
        const int* map = fd.cmap + fd.uptr[c];
        __syncthreads();                   // the previous child's tables are no longer read
        for (int k = tid; k < nn; k += 256) smap[k] = map[k];
        __syncthreads();
        bool hit = false;
        if (tid < 2 * FF_TILE) {
            const int side = tid / FF_TILE, t = tid % FF_TILE;
            const int pos = (side ? c0 : r0) + t, node = pos / 3;
            int lo = 0, hi = nn;           // first entry >= node
            while (lo < hi) {
                const int mid = (lo + hi) >> 1;
                if (smap[mid] < node) lo = mid + 1;
                else hi = mid;
            }
            hit = pos < f && lo < nn && smap[lo] == node;
            idx[side][t] = hit ? pc + 3 * lo + pos % 3 : -1;
        }
        const int rows_hit = __syncthreads_or(tid < FF_TILE && hit);
        const int cols_hit = __syncthreads_or(tid >= FF_TILE && hit);
        if (!rows_hit || !cols_hit) continue;
        const float* Fc = fd.pool + fd.off[c];
        if (!touched) {
            touched = true;
#pragma unroll
            for (int u = 0; u < 2; ++u)
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                    const int r = r0 + tx + 32 * u, cc = c0 + ty + 8 * v;
                    acc[u][v] = (r < f && cc <= r) ? F[(long)cc * f + r] : 0.0f;
                }
        }
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int ri = idx[0][tx + 32 * u];
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const int ci = idx[1][ty + 8 * v];
                if (ri >= ci && ci >= 0) acc[u][v] += Fc[(long)ci * fc + ri];
            }
        }
    }
    if (!touched) return;
#pragma unroll
    for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int v = 0; v < 8; ++v) {
            const int r = r0 + tx + 32 * u, cc = c0 + ty + 8 * v;
            if (r < f && cc <= r) F[(long)cc * f + r] = acc[u][v];
        }
}

// One strip of eight pivot columns in the diagonal block's rows (one per lane), and its
// share of the columns after it.  (Templates, so that every index into a row's registers
// is a constant.)
template <int C0>
__device__ __forceinline__ void ff_strip(float (&a)[PB], float* Ls, float* Dd, int lane, float tau) {
#pragma unroll
    for (int cc = 0; cc < 8; ++cc) {
        const int c = C0 + cc;
        float d = __shfl_sync(0xffffffffu, a[c], c);
        if (fabsf(d) < tau) d = (d < 0.0f) ? -tau : tau;
        const float id = 1.0f / d;
        const float u = lane > c ? a[c] : 0.0f;                // l d in the lanes below c
#pragma unroll
        for (int j = cc + 1; j < 8; ++j) {
            const float lj = __shfl_sync(0xffffffffu, a[c], C0 + j) * id;
            a[C0 + j] -= u * lj;
        }
        Ls[lane * LSS + c] = lane > c ? u * id : (lane == c ? 1.0f : 0.0f);
        if (lane == c) Dd[c] = d;
    }
}
template <int C0>
__device__ __forceinline__ void ff_strip_rest(float (&a)[PB], const float* Ls, int lane) {
#pragma unroll
    for (int j = C0 + 8; j < PB; ++j) {
        const float4 l0 = *reinterpret_cast<const float4*>(Ls + j * LSS + C0);
        const float4 l1 = *reinterpret_cast<const float4*>(Ls + j * LSS + C0 + 4);
        const float lj[8] = {l0.x, l0.y, l0.z, l0.w, l1.x, l1.y, l1.z, l1.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) a[j] -= (lane > C0 + q ? a[C0 + q] : 0.0f) * lj[q];
    }
}
// Rows C0 + 1 .. C0 + 8 of the block's inverse, column `lane` (a lane reads only what it
// wrote itself, and published columns of L).
__device__ __forceinline__ void ff_inverse_rows(int c0, const float* Ls, float* Xs, int lane, int kb) {
    for (int i = c0 + 1; i < c0 + 9 && i < PB; ++i) {
        float acc = 0.0f;
#pragma unroll 8
        for (int q = 0; q < i; ++q) acc += Ls[i * LSS + q] * Xs[q * LSS + lane];
        const float x = i > lane ? -acc : (i == lane ? 1.0f : 0.0f);
        Xs[i * LSS + lane] = (lane < kb && i < kb) ? x : (i == lane ? 1.0f : 0.0f);
    }
}
// Columns [CL, CL + 8) of l = D^-1 L_kk^-1 a for one row below the block.
template <int CL>
__device__ __forceinline__ void ff_solve(const float (&a)[PB], const float* Xs, const float* Dd, float* dst, int f,
                                         int kb, bool valid) {
#pragma unroll
    for (int c = (CL > 0 ? CL : 0); c < CL + 8 && c < PB; ++c) {
        float sum = 0.0f;
#pragma unroll
        for (int j = 0; j <= c; ++j) sum += Xs[c * LSS + j] * a[j];
        if (valid && c < kb) dst[(long)c * f] = sum / Dd[c];
    }
}

// Panel k of one front, a pipeline over strips of eight columns: warp 0 holds the rows of
// the diagonal block, one per lane, eliminates a strip in them (shuffles only),
// publishes it and subtracts its share from its remaining columns; warp 1 forms the
// rows of the block's inverse that the published columns complete; the other warps hold
// FF_ROWS rows below the block, one per thread, all 32 columns in registers, and form
// l = D^-1 L_kk^-1 a for the columns whose inverse rows are there.
// The factorised block waits in the diagonal block of the front's inverse (its place in
// the front is still being read by the other CTAs) and its inverse in its binv slot.
__global__ void __launch_bounds__(FF_PT) k_ff_panel(FrontDev fd, const int2* __restrict__ tasks, int k) {
    __shared__ __align__(16) float Ls[PB * LSS];   // unit-lower L of the block, row-major
    __shared__ __align__(16) float Xs[PB * LSS];   // its inverse
    __shared__ float Dd[PB];
    const int2 task = tasks[blockIdx.x];
    const int s = task.x, rb = task.y;
    const int f = fd.f[s], p = fd.p[s], k0 = k * PB, kb = min(PB, p - k0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool diag = warp == 0, below = warp >= 2;
    float* F = fd.pool + fd.off[s];
    const int row = diag ? k0 + lane : k0 + kb + rb * FF_ROWS + tid - 64;
    const bool valid = diag ? lane < kb : below && row < f;
    float* const col0 = F + (long)k0 * f + row;
    float a[PB];
#pragma unroll
    for (int c = 0; c < PB; ++c) a[c] = (valid && c < kb && (!diag || c <= lane)) ? col0[(long)c * f] : 0.0f;
    // columns past a partial last panel: the identity (their factors are 1 and 0)
    if (diag && lane >= kb)
#pragma unroll
        for (int c = 0; c < PB; ++c)
            if (c == lane) a[c] = 1.0f;
    const float tau = fd.tau[s];
    if (warp == 1) Xs[lane] = lane == 0 ? 1.0f : 0.0f;
    // strip C0: publish it, then every warp's share of the work that it completes
#define FF_STRIP(C0)                                                                                    \
    if (diag) ff_strip<C0>(a, Ls, Dd, lane, tau);                                                       \
    __syncthreads();                                                                                    \
    if (diag) ff_strip_rest<C0>(a, Ls, lane);                                                           \
    else if (warp == 1) ff_inverse_rows(C0, Ls, Xs, lane, kb);                                          \
    else ff_solve<C0 - 7>(a, Xs, Dd, col0, f, kb, valid);   /* inverse rows up to C0 are complete */
    FF_STRIP(0)
    FF_STRIP(8)
    FF_STRIP(16)
    FF_STRIP(24)
#undef FF_STRIP
    __syncthreads();
    if (diag) {
        if (rb == 0 && lane < kb) {
            float* W = fd.linv + fd.linv_off[s] + (long)k0 * p + k0;
            float* Bi = fd.binv + fd.binv_off[s] + (long)k * PB * PB;   // column-major
#pragma unroll
            for (int c = 0; c < PB; ++c)
                if (c <= lane) W[(long)c * p + lane] = lane == c ? Dd[c] : Ls[lane * LSS + c];
#pragma unroll
            for (int c = 0; c < PB; ++c) Bi[c * PB + lane] = Xs[lane * LSS + c];
        }
    } else if (below) {
        ff_solve<PB - 7>(a, Xs, Dd, col0, f, kb, valid);
    }
}

// The pivots of panel k (k_ff_panel keeps the factorised block in the inverse).
__device__ __forceinline__ float ff_pivot(const FrontDev& fd, int s, int p, int k0, int c) {
    return fd.linv[fd.linv_off[s] + (long)(k0 + c) * p + k0 + c];
}

// Rank-32 update k of one 64 x 64 tile of the trailing lower triangle, T -= L D L^T,
// in FP32 FMAs.
__global__ void __launch_bounds__(256) k_ff_update(FrontDev fd, const int2* __restrict__ tasks, int k) {
    __shared__ __align__(16) float As[PB][FF_TILE];
    __shared__ __align__(16) float Bs[PB][FF_TILE + 4];
    const int2 task = tasks[blockIdx.x];
    const int s = task.x;
    const int r0 = (task.y >> 16) * FF_TILE, c0 = (task.y & 0xffff) * FF_TILE;
    const int f = fd.f[s], p = fd.p[s], k0 = k * PB, kb = min(PB, p - k0), n2 = f - k0 - kb;
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float* Fp = fd.pool + fd.off[s] + (long)k0 * f + k0 + kb;          // L's rows below the block
    float* C = Fp + (long)kb * f;
#pragma unroll
    for (int e = tid; e < PB * FF_TILE; e += 256) {
        const int r = e % FF_TILE, c = e / FF_TILE;
        As[c][r] = (c < kb && r0 + r < n2) ? Fp[(long)c * f + r0 + r] : 0.0f;
        Bs[c][r] = (c < kb && c0 + r < n2) ? Fp[(long)c * f + c0 + r] * ff_pivot(fd, s, p, k0, c) : 0.0f;
    }
    float old[4][4], acc[4][4];
    bool on[4][4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int c = c0 + 4 * ty + v;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = r0 + tx + 16 * u;
            on[u][v] = r < n2 && c <= r;
            old[u][v] = on[u][v] ? C[(long)c * f + r] : 0.0f;
            acc[u][v] = 0.0f;
        }
    }
    __syncthreads();
#pragma unroll 8
    for (int c = 0; c < PB; ++c) {
        const float4 b = *reinterpret_cast<const float4*>(&Bs[c][4 * ty]);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const float x = As[c][tx + 16 * u];
            acc[u][0] += x * b.x;
            acc[u][1] += x * b.y;
            acc[u][2] += x * b.z;
            acc[u][3] += x * b.w;
        }
    }
#pragma unroll
    for (int v = 0; v < 4; ++v)
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (on[u][v]) C[(long)(c0 + 4 * ty + v) * f + r0 + tx + 16 * u] = old[u][v] - acc[u][v];
}

// Rows [g0, g0 + ROWS) of L below the block (column c of row g at Lp[c f + g]), times
// the pivots when SCALED, split into TF32 hi/lo parts in the operand layout; rows at or
// beyond n2 and columns at or beyond kb are zero.
template <int ROWS, bool SCALED>
__device__ __forceinline__ void tc_stage(const float* __restrict__ Lp, int f, int g0, int n2, int kb,
                                         const float* __restrict__ D, int p, unsigned char* hi, unsigned char* lo) {
#pragma unroll
    for (int e0 = 0; e0 < ROWS * (TC_K / 4); e0 += 256) {
        const int e = e0 + threadIdx.x, r = e % ROWS, k4 = e / ROWS, g = g0 + r;
        float v[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int k = 4 * k4 + j;
            const bool on = g < n2 && k < kb;
            v[j] = on ? Lp[(long)k * f + g] : 0.0f;
            if (SCALED && on) v[j] *= D[(long)k * p + k];
        }
        float4 h, l;
        tc_split(v[0], h.x, l.x);
        tc_split(v[1], h.y, l.y);
        tc_split(v[2], h.z, l.z);
        tc_split(v[3], h.w, l.w);
        *reinterpret_cast<float4*>(hi + tc_off(r, 4 * k4)) = h;
        *reinterpret_cast<float4*>(lo + tc_off(r, 4 * k4)) = l;
    }
}

// The same update of one 128 x TC_N tile on the tensor cores: stage L's rows (A) and
// L D's rows (B), issue the three TF32 passes (hi hi, hi lo, lo hi; K = 32 in four slices
// each) from one thread into TMEM, and subtract the accumulator from T's lower entries
// (thread = row, coalesced down a column).  A tile is a chain of latencies (its loads, the
// MMAs, the read-back), so four CTAs share an SM: 64 registers a thread, 48 KB of
// operands and 64 of the 512 TMEM columns each.  An MMA that does not complete within
// TC_WAIT polls sets the fault word; the CTA waits once more for it, frees its TMEM and
// leaves.
__global__ void __launch_bounds__(256, 4) k_ff_update_tc(FrontDev fd, const int2* __restrict__ tasks, int k) {
    extern __shared__ __align__(1024) unsigned char tcs[];
    __shared__ uint64_t bar;
    __shared__ uint32_t slot;
    unsigned char* a_hi = tcs;
    unsigned char* a_lo = a_hi + TC_A_BYTES;
    unsigned char* b_hi = a_lo + TC_A_BYTES;
    unsigned char* b_lo = b_hi + TC_B_BYTES;
    constexpr uint32_t idesc = tc_idesc_tf32(TC_M, TC_N);
    const int2 task = tasks[blockIdx.x];
    const int s = task.x;
    const int r0 = (task.y >> 16) * TC_M, q0 = (task.y & 0xffff) * TC_N;
    const int f = fd.f[s], p = fd.p[s], k0 = k * PB, kb = min(PB, p - k0), n2 = f - k0 - kb;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, wg = warp >> 2, lq = warp & 3;
    const float* Lp = fd.pool + fd.off[s] + (long)k0 * f + k0 + kb;
    const float* D = fd.linv + fd.linv_off[s] + (long)k0 * p + k0;
    float* T = fd.pool + fd.off[s] + (long)(k0 + kb) * f + k0 + kb;
    if (tid == 0) {
        tc_mbar_init(&bar, 1);
        tc_mbar_init_fence();
    }
    if (warp == 0) tc_alloc(&slot, TC_COLS);
    tc_stage<TC_M, false>(Lp, f, r0, n2, kb, D, p, a_hi, a_lo);
    tc_stage<TC_N, true>(Lp, f, q0, n2, kb, D, p, b_hi, b_lo);
    tc_fence_async_smem();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    const uint32_t tmem = slot;
    if (tid == 0) {
        const uint32_t ah = tc_smem_u32(a_hi), al = tc_smem_u32(a_lo);
        const uint32_t bh = tc_smem_u32(b_hi), bl = tc_smem_u32(b_lo);
#pragma unroll
        for (int pass = 0; pass < 3; ++pass) {
            const uint32_t a = pass == 2 ? al : ah, b = pass == 1 ? bl : bh;
#pragma unroll
            for (int kk = 0; kk < TC_K / 8; ++kk)
                tc_mma_tf32(tmem, tc_desc(a + kk * 2 * TC_CORE_K_BYTES), tc_desc(b + kk * 2 * TC_CORE_K_BYTES), idesc,
                            (pass | kk) ? 1u : 0u);
        }
        tc_commit(&bar);
    }
    // this thread's row; the current values of a 16-column chunk are loaded while the
    // tensor core (or the other chunk) works
    const int r = r0 + 32 * lq + lane;
    float old[16];
    auto load = [&](int h) {
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            const int col = q0 + 16 * (wg + 2 * h) + c;
            old[c] = (r < n2 && col <= r) ? T[(long)col * f + r] : 0.0f;
        }
    };
    load(0);
    const bool done = tc_mbar_wait(&bar, 0, TC_WAIT);
    if (!__syncthreads_or(!done)) {
        tc_fence_after_sync();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            if (h) load(1);
            float v[16];
            tc_ld16(tmem + ((uint32_t)(32 * lq) << 16) + 16u * (wg + 2 * h), v);
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const int col = q0 + 16 * (wg + 2 * h) + c;
                if (r < n2 && col <= r) T[(long)col * f + r] = old[c] - v[c];
            }
        }
    } else {
        if (tid == 0) atomicExch(fd.fault, 1ull);
        tc_mbar_wait(&bar, 0, TC_WAIT);
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 0) tc_dealloc(tmem, TC_COLS);
}

// CW columns [32 J + CW h, ...) of the inverse X of a front's unit-lower pivot block, by
// block rows: X_JJ = B_J, X_IJ = -B_I sum_{K=J}^{I-1} L_IK X_KJ; the factorised diagonal
// block J goes back into the front first.  Lane = row, a warp CW / 8 columns; L's block
// row streams through shared memory 64 columns at a time, the columns of X stay there
// (SX) or, for pivot blocks too large for that, are read back through L1.
constexpr int FF_KT = 64;
template <int CW, bool SX>
__global__ void __launch_bounds__(256) k_ff_inverse(FrontDev fd, const int2* __restrict__ tasks) {
    extern __shared__ __align__(16) float xsm[];   // SX: X rows k1 .. p, [k - k1][CW]
    __shared__ float Lt[2][FF_KT][PB];
    __shared__ float Tm[CW][PB + 1];
    constexpr int NC = CW / 8;
    const int2 task = tasks[blockIdx.x];
    const int s = task.x, J = task.y >> 8, ch = (task.y & 0xff) * CW;
    const int f = fd.f[s], p = fd.p[s], k1 = J * PB, nb = (p + PB - 1) / PB, jb = min(PB, p - k1);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const float* binv = fd.binv + fd.binv_off[s];
    float* F = fd.pool + fd.off[s];
    float* X = fd.linv + fd.linv_off[s] + (long)(k1 + ch) * p;          // this task's first column
    const int ncol = min(CW, jb - ch);
    for (int e = tid; e < PB * CW; e += 256) {
        const int r = e % PB, c = e / PB;
        if (c < ncol && r < jb) {
            float* w = X + (long)c * p + k1 + r;
            const float b = binv[(long)J * PB * PB + (ch + c) * PB + r];
            if (r >= ch + c) {
                F[(long)(k1 + ch + c) * f + k1 + r] = *w;
                *w = b;
            } else if (!SX) {
                *w = 0.0f;                 // (read back with the column's other rows)
            }
            if (SX) xsm[r * CW + c] = b;
        } else if (SX && r < jb) {
            xsm[r * CW + c] = 0.0f;
        }
    }
    for (int I = J + 1; I < nb; ++I) {
        const int i0 = I * PB, ib = min(PB, p - i0);
        const int nk = i0 - k1;
        float acc[NC];
#pragma unroll
        for (int v = 0; v < NC; ++v) acc[v] = 0.0f;
        // row `lane` of B_I, wanted at the end of this block row
        const float* Bi = binv + (long)I * PB * PB + lane;
        float br[PB];
#pragma unroll
        for (int q = 0; q < PB; ++q) br[q] = q < ib ? Bi[q * PB] : 0.0f;
        float nx[FF_KT / 8];
        auto fetch = [&](int t0) {
#pragma unroll
            for (int m = 0; m < FF_KT / 8; ++m) {
                const int q = t0 + warp + 8 * m;
                nx[m] = (q < nk && lane < ib) ? F[(long)(k1 + q) * f + i0 + lane] : 0.0f;
            }
        };
        fetch(0);
        __syncthreads();                   // X rows of the previous block are in place
        for (int t0 = 0, b = 0; t0 < nk; t0 += FF_KT, b ^= 1) {
#pragma unroll
            for (int m = 0; m < FF_KT / 8; ++m) Lt[b][warp + 8 * m][lane] = nx[m];
            __syncthreads();
            if (t0 + FF_KT < nk) fetch(t0 + FF_KT);
            const int n = min(FF_KT, nk - t0);
#pragma unroll 8
            for (int q = 0; q < n; ++q) {
                const float l = Lt[b][q][lane];
                if (NC == 4) {
                    const float4 x = *reinterpret_cast<const float4*>(xsm + (t0 + q) * CW + 4 * warp);
                    acc[0] += l * x.x;
                    acc[NC > 1 ? 1 : 0] += l * x.y;
                    acc[NC > 2 ? 2 : 0] += l * x.z;
                    acc[NC > 2 ? 3 : 0] += l * x.w;
                    continue;
                }
#pragma unroll
                for (int v = 0; v < NC; ++v) {
                    const int c = warp * NC + v;
                    acc[v] += l * (SX ? xsm[(t0 + q) * CW + c] : (c < ncol ? X[(long)c * p + k1 + t0 + q] : 0.0f));
                }
            }
        }
#pragma unroll
        for (int v = 0; v < NC; ++v) Tm[warp * NC + v][lane] = acc[v];
        __syncwarp();                      // a warp's columns of Tm are its own
#pragma unroll
        for (int v = 0; v < NC; ++v) {
            const int c = warp * NC + v;
            float x = 0.0f;
#pragma unroll
            for (int q = 0; q < PB; ++q)
                if (q < ib) x -= br[q] * Tm[c][q];
            if (lane < ib) {
                if (c < ncol) X[(long)c * p + i0 + lane] = x;
                if (SX) xsm[(i0 - k1 + lane) * CW + c] = c < ncol ? x : 0.0f;
            }
        }
    }
}

inline int cdiv(int a, int b) { return (a + b - 1) / b; }

}  // namespace

// The columns of X a k_ff_inverse CTA takes for a pivot block of p unknowns: 32, 16 or 8 (at
// most `most`) while they fit its shared memory, else 8 without (returns 0).
static int ff_inverse_cols(int p, int most) {
    for (int cw = most; cw >= 8; cw /= 2)
        if ((size_t)cw * p * sizeof(float) <= 192 * 1024) return cw;
    return 0;
}

// Whether a level whose largest front has max_f unknowns uses the tensor-core updates
// (off for every level when DC_FRONT_FMA=1 is in the environment).
static bool ff_level_tc(int max_f) {
    static const bool off = [] {
        const char* e = std::getenv("DC_FRONT_FMA");
        return e && e[0] == '1';
    }();
    return !off && max_f >= TC_MIN_F;
}

// Tile lists of every level's launches, in launch order.  tc: -1 by the level's largest
// front, 0 / 1 forced; cols: the most columns of an inverse task, 0 for its form without
// shared memory (both for tests).
void ff_plan(const HostFronts& fr, FrontPlan& pl, std::vector<int2>& tasks, int tc, int cols) {
    pl = FrontPlan();
    tasks.clear();
    const int nl = (int)fr.lvl_ptr.size() - 1;
    for (int l = 0; l < nl; ++l) {
        const int q0 = fr.lvl_ptr[l], q1 = fr.lvl_ptr[l + 1];
        auto close = [&](int kind, int k) {
            const int begin = pl.launches.empty() ? 0 : pl.launches.back().begin + pl.launches.back().count;
            if ((int)tasks.size() > begin) pl.launches.push_back(FrontLaunch{kind, k, l, begin, (int)tasks.size() - begin});
        };
        int mp = 0, mf = 0;
        for (int q = q0; q < q1; ++q) {
            const int s = fr.lvl_sn[q];
            mp = std::max(mp, fr.p[s]);
            mf = std::max(mf, fr.f[s]);
            if (fr.cptr[s] == fr.cptr[s + 1]) continue;
            const int n = cdiv(fr.f[s], FF_TILE);
            for (int i = 0; i < n; ++i)
                for (int j = 0; j <= i; ++j) tasks.push_back(make_int2(s, (i << 16) | j));
        }
        close(FF_EXTEND, 0);
        const bool ltc = tc < 0 ? ff_level_tc(mf) : tc != 0;
        for (int k = 0; k * PB < mp; ++k) {
            const int k0 = k * PB;
            for (int q = q0; q < q1; ++q) {
                const int s = fr.lvl_sn[q];
                if (k0 >= fr.p[s]) continue;
                const int below = fr.f[s] - k0 - std::min(PB, fr.p[s] - k0);
                for (int rb = 0; rb < std::max(1, cdiv(below, FF_ROWS)); ++rb) tasks.push_back(make_int2(s, rb));
            }
            close(FF_PANEL, k);
            for (int pass = 0; pass < 2; ++pass) {   // FMA tiles, then tensor-core tiles
                for (int q = q0; q < q1; ++q) {
                    const int s = fr.lvl_sn[q];
                    if (k0 >= fr.p[s]) continue;
                    const int n2 = fr.f[s] - k0 - std::min(PB, fr.p[s] - k0);
                    if ((ltc && n2 >= TC_MIN_N2) != (pass == 1)) continue;
                    const int tm = pass ? TC_M : FF_TILE, tn = pass ? TC_N : FF_TILE;
                    for (int i = 0; i < cdiv(n2, tm); ++i)
                        for (int j = 0; j * tn < std::min((i + 1) * tm, n2); ++j)
                            tasks.push_back(make_int2(s, (i << 16) | j));
                }
                close(pass ? FF_UPDATE_TC : FF_UPDATE, k);
            }
        }
        // the inverse: the tasks of one launch share its column count
        for (int cw : {32, 16, 8, 0}) {
            for (int q = q0; q < q1; ++q) {
                const int s = fr.lvl_sn[q], p = fr.p[s];
                if (ff_inverse_cols(p, cols) != cw) continue;
                const int w = std::max(cw, 8);
                for (int J = 0; J * PB < p; ++J)
                    for (int c = 0; c * w < std::min(PB, p - J * PB); ++c) tasks.push_back(make_int2(s, (J << 8) | c));
            }
            close(FF_INVERSE, cw);
            if (!pl.launches.empty() && pl.launches.back().kind == FF_INVERSE && pl.launches.back().level == l &&
                pl.launches.back().k == cw) {
                int p = 0;
                for (int q = q0; q < q1; ++q)
                    if (ff_inverse_cols(fr.p[fr.lvl_sn[q]], cols) == cw) p = std::max(p, fr.p[fr.lvl_sn[q]]);
                pl.launches.back().smem = cw * p * (int)sizeof(float);
            }
        }
    }
}

// Shared-memory limits of the factorisation kernels (per function, set once).
cudaError_t ff_configure() {
    static std::mutex mu;
    static bool done = false;
    std::lock_guard<std::mutex> lock(mu);
    if (done) return cudaSuccess;
    cudaError_t e = cudaFuncSetAttribute(k_ff_update_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_BYTES);
    for (const void* k : {(const void*)k_ff_inverse<32, true>, (const void*)k_ff_inverse<16, true>,
                          (const void*)k_ff_inverse<8, true>})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 192 * 1024);
    done = e == cudaSuccess;
    return e;
}

// One factorisation: the launches of the plan on stream s.
void ff_factorize(const FrontDev& fd, const FrontPlan& pl, cudaStream_t s, KTimer* kt) {
    const size_t map_bytes = sizeof(int) * (size_t)(fd.max_f / 3 + 1);
    int level = -1;
    for (const FrontLaunch& a : pl.launches) {
        if (kt && a.level != level) {
            if (level >= 0) kt->end(DC_KT_FRONT);
            kt->begin(DC_KT_FRONT);
        }
        level = a.level;
        const int2* t = fd.tasks + a.begin;
        dc_note_launch();
        if (a.kind == FF_EXTEND) k_ff_extend<<<a.count, 256, map_bytes, s>>>(fd, t);
        else if (a.kind == FF_PANEL) k_ff_panel<<<a.count, FF_PT, 0, s>>>(fd, t, a.k);
        else if (a.kind == FF_UPDATE) k_ff_update<<<a.count, 256, 0, s>>>(fd, t, a.k);
        else if (a.kind == FF_UPDATE_TC) k_ff_update_tc<<<a.count, 256, TC_BYTES, s>>>(fd, t, a.k);
        else if (a.k == 32) k_ff_inverse<32, true><<<a.count, 256, a.smem, s>>>(fd, t);
        else if (a.k == 16) k_ff_inverse<16, true><<<a.count, 256, a.smem, s>>>(fd, t);
        else if (a.k == 8) k_ff_inverse<8, true><<<a.count, 256, a.smem, s>>>(fd, t);
        else k_ff_inverse<8, false><<<a.count, 256, 0, s>>>(fd, t);
    }
    if (kt && level >= 0) kt->end(DC_KT_FRONT);
}

// One dense front through the factorisation: the test hook behind
// dc_debug_front_factor (synchronous; allocates and frees its own buffers).
dc_status ff_debug_factor(int n, int p, const float* A, float* out, float* linv_out, int tc, int cols,
                          std::string* err) {
    if (!A || !out) {
        *err = "dc_debug_front_factor: null A or out";
        return DC_ERR_INVALID;
    }
    HostFronts fr;
    fr.S = 1;
    fr.f = {n};
    fr.p = {p};
    fr.cptr = {0, 0};
    fr.lvl_ptr = {0, 1};
    fr.lvl_sn = {0};
    FrontPlan pl;
    std::vector<int2> tasks;
    ff_plan(fr, pl, tasks, tc != 0, cols);
    const int nbk = cdiv(p, PB);
    // device image: ints [f, p, cptr0, cptr1], long longs [off, binv_off, linv_off]
    int hi[4] = {n, p, 0, 0};
    long long hl[3] = {0, 0, 0};
    float tau = 1e-30f;
    int* di = nullptr;
    long long* dl = nullptr;
    int2* dt = nullptr;
    float *pool = nullptr, *binv = nullptr, *linv = nullptr, *dtau = nullptr;
    unsigned long long *fault = nullptr, fl = 0;
    cudaError_t e = ff_configure();
    if (e == cudaSuccess) do {
        if ((e = cudaMalloc(&fault, sizeof(fl))) || (e = cudaMemset(fault, 0, sizeof(fl))) || (e = cudaMalloc(&di, sizeof(hi))) || (e = cudaMalloc(&dl, sizeof(hl))) ||
            (e = cudaMalloc(&dt, sizeof(int2) * tasks.size())) ||
            (e = cudaMalloc(&pool, sizeof(float) * (size_t)n * n)) ||
            (e = cudaMalloc(&binv, sizeof(float) * (size_t)nbk * PB * PB)) ||
            (e = cudaMalloc(&linv, sizeof(float) * (size_t)p * p)) || (e = cudaMalloc(&dtau, sizeof(float))) ||
            (e = cudaMemcpy(di, hi, sizeof(hi), cudaMemcpyHostToDevice)) ||
            (e = cudaMemcpy(dl, hl, sizeof(hl), cudaMemcpyHostToDevice)) ||
            (e = cudaMemcpy(dt, tasks.data(), sizeof(int2) * tasks.size(), cudaMemcpyHostToDevice)) ||
            (e = cudaMemcpy(dtau, &tau, sizeof(float), cudaMemcpyHostToDevice)) ||
            (e = cudaMemcpy(pool, A, sizeof(float) * (size_t)n * n, cudaMemcpyHostToDevice)) ||
            (e = cudaMemset(linv, 0xff, sizeof(float) * (size_t)p * p)))   // NaNs: nothing there may be read
            break;
        FrontDev fd{};
        fd.S = 1;
        fd.max_f = n;
        fd.tau = dtau;
        fd.f = di;
        fd.p = di + 1;
        fd.cptr = di + 2;
        fd.off = dl;
        fd.binv_off = dl + 1;
        fd.linv_off = dl + 2;
        fd.pool = pool;
        fd.binv = binv;
        fd.linv = linv;
        fd.tasks = dt;
        fd.fault = fault;
        ff_factorize(fd, pl, nullptr, nullptr);
        if ((e = cudaGetLastError()) || (e = cudaDeviceSynchronize())) break;
        if ((e = cudaMemcpy(&fl, fault, sizeof(fl), cudaMemcpyDeviceToHost)) ||
            (e = cudaMemcpy(out, pool, sizeof(float) * (size_t)n * n, cudaMemcpyDeviceToHost)))
            break;
        if (linv_out) {
            e = cudaMemcpy(linv_out, linv, sizeof(float) * (size_t)p * p, cudaMemcpyDeviceToHost);
            for (int c = 0; c < p; ++c) std::fill(linv_out + (size_t)c * p, linv_out + (size_t)c * p + c, 0.0f);
        }
    } while (false);
    cudaFree(di);
    cudaFree(dl);
    cudaFree(dt);
    cudaFree(pool);
    cudaFree(binv);
    cudaFree(linv);
    cudaFree(dtau);
    cudaFree(fault);
    if (e == cudaSuccess && fl) {
        *err = "dc_debug_front_factor: a tensor-core wait gave up";
        return DC_ERR_TIMEOUT;
    }
    if (e != cudaSuccess) {
        *err = std::string("dc_debug_front_factor: ") + cudaGetErrorString(e);
        return DC_ERR_CUDA;
    }
    return DC_OK;
}
