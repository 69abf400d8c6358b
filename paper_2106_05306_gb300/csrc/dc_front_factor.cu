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
//               the 32 x 32 diagonal block (again: it is small, and recomputing it
//               is cheaper than a launch or a wait between CTAs) and solves FF_ROWS
//               of the rows below it, one row per thread in registers;
//   update k -- the rank-32 update of the trailing lower triangle, one CTA per
//               64 x 64 tile, and of the inverse of the pivot block (below);
//   finish   -- the diagonal blocks go back into the fronts, and the inverse's
//               block rows are completed.
// The tile lists depend only on the fronts' sizes and are laid out once by
// ff_plan.  Every entry's arithmetic depends only on its own front, so an
// instance gives the same bits alone and in a batch.
//
// The inverse X of the unit-lower pivot block (the solves multiply by it) grows
// with the panels: X = B_k W_k by block rows, with B_k the inverse of diagonal
// block k and W_IJ = -sum_{J <= k < I} L_Ik B_k W_kJ.  Panel k writes its own
// block column W_Ik = -L_Ik B_k, and update k adds W_Ik W_kJ to the columns left
// of it, a rank-32 update like the trailing one; finish multiplies by B_k.
//
// Measured (device time of one factorisation, the launches one by one under the
// profiler; before: one CTA per front with its panel in shared memory and the
// trailing updates as three TF32 passes on the tensor cores): one 200x200 cloth
// 118 ms -> 4.5 ms, one 61x61 cloth 4.1 -> 0.95 ms, 96 cloths of 16x16..64x64
// 9.5 -> 4.7 ms.  The tile updates are bound by the traffic of the trailing block
// (32 columns per pass), so FP32 FMAs keep up and nothing is split to TF32.
#include <algorithm>
#include <string>
#include <vector>

#include "dc_adjoint.h"
#include "dc_internal.h"

namespace {

constexpr int PB = 32;                     // panel width
constexpr int FF_PT = 128;                 // threads of a panel CTA: one warp on the diagonal block
constexpr int FF_ROWS = FF_PT - 32;        // rows below it per CTA
constexpr int FF_TILE = 64;                // tile of the extend-add and of the updates
constexpr int FF_FCOLS = 128;              // inverse columns per finish CTA
constexpr int LSS = 36;                    // row stride of the diagonal block in shared memory (16-byte rows)

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

// Panel k of one front: warp 0 holds the rows of the diagonal block, one per lane,
// the other warps FF_ROWS rows below it, one per thread, all 32 columns in
// registers.  Eight columns at a time: warp 0 eliminates them in its rows
// (shuffles only) and publishes that strip of L, then every row subtracts its
// share from its remaining columns.  The factorised diagonal block goes to the
// front's binv slot (its place in the front is still being read by the other
// CTAs); rows inside the pivot block also give W_Ik = -L_Ik B_k.
__global__ void __launch_bounds__(FF_PT) k_ff_panel(FrontDev fd, const int2* __restrict__ tasks, int k) {
    __shared__ __align__(16) float Ls[PB * LSS];   // unit-lower L of the block, row-major
    __shared__ float rd[PB];
    const int2 task = tasks[blockIdx.x];
    const int s = task.x, rb = task.y;
    const int f = fd.f[s], p = fd.p[s], k0 = k * PB, kb = min(PB, p - k0);
    const int tid = threadIdx.x, lane = tid & 31;
    const bool diag = tid < 32;
    float* F = fd.pool + fd.off[s];
    const int row = diag ? k0 + lane : k0 + kb + rb * FF_ROWS + tid - 32;
    const bool valid = diag ? lane < kb : row < f;
    float a[PB];
    {
        const float* src = F + (long)k0 * f + row;
#pragma unroll
        for (int c = 0; c < PB; ++c) a[c] = (valid && c < kb && (!diag || c <= lane)) ? src[(long)c * f] : 0.0f;
    }
    // columns past a partial last panel: the identity (their factors are 1 and 0)
    if (diag && lane >= kb)
#pragma unroll
        for (int c = 0; c < PB; ++c)
            if (c == lane) a[c] = 1.0f;
    const float tau = fd.tau[s];
    float dl = 1.0f;                       // this lane's pivot (diagonal warp)
#pragma unroll
    for (int c0 = 0; c0 < PB; c0 += 8) {
        if (diag) {
#pragma unroll
            for (int cc = 0; cc < 8; ++cc) {
                const int c = c0 + cc;
                float d = __shfl_sync(0xffffffffu, a[c], c);
                if (fabsf(d) < tau) d = (d < 0.0f) ? -tau : tau;
                const float id = 1.0f / d;
                const float u = a[c];                          // l d in the lanes below c
                const float l = lane > c ? u * id : 0.0f;
#pragma unroll
                for (int j = cc + 1; j < 8; ++j) a[c0 + j] -= l * __shfl_sync(0xffffffffu, u, c0 + j);
                Ls[lane * LSS + c] = lane == c ? 1.0f : l;
                if (lane == c) {
                    dl = d;
                    rd[c] = id;
                }
            }
        }
        __syncthreads();
        if (!diag) {
#pragma unroll
            for (int cc = 1; cc < 8; ++cc) {
                float t = a[c0 + cc];
#pragma unroll
                for (int q = 0; q < cc; ++q) t -= a[c0 + q] * Ls[(c0 + cc) * LSS + c0 + q];
                a[c0 + cc] = t;
            }
        }
#pragma unroll
        for (int j = c0 + 8; j < PB; ++j) {
            const float4 x = *reinterpret_cast<const float4*>(Ls + j * LSS + c0);
            const float4 y = *reinterpret_cast<const float4*>(Ls + j * LSS + c0 + 4);
            a[j] -= a[c0] * x.x + a[c0 + 1] * x.y + a[c0 + 2] * x.z + a[c0 + 3] * x.w + a[c0 + 4] * y.x +
                    a[c0 + 5] * y.y + a[c0 + 6] * y.z + a[c0 + 7] * y.w;
        }
    }
    if (diag) {
        if (rb == 0) {
            float* Bi = fd.binv + fd.binv_off[s] + (long)k * PB * PB;   // column-major
#pragma unroll
            for (int c = 0; c < PB; ++c) Bi[c * PB + lane] = lane == c ? dl : (lane > c ? Ls[lane * LSS + c] : 0.0f);
        }
        return;
    }
    if (!valid) return;
    float* dst = F + (long)k0 * f + row;
#pragma unroll
    for (int c = 0; c < PB; ++c) {
        a[c] *= rd[c];
        if (c < kb) dst[(long)c * f] = a[c];
    }
    if (row >= p) return;
    // L_Ik B_k by back substitution against the block (x B = l  <=>  x = l L^-1)
#pragma unroll
    for (int j = PB - 1; j > 0; --j)
#pragma unroll
        for (int c = 0; c < j; ++c) a[c] -= a[j] * Ls[j * LSS + c];
    float* W = fd.linv + fd.linv_off[s] + (long)k0 * p + row;
#pragma unroll
    for (int c = 0; c < PB; ++c)
        if (c < kb) W[(long)c * p] = -a[c];
}

// Rank-32 update k of one 64 x 64 tile: of the trailing lower triangle,
// T -= L D L^T, or (bit 30 of task.y) of the pivot block's inverse,
// W_IJ += W_Ik W_kJ for the columns left of panel k.
__global__ void __launch_bounds__(256) k_ff_update(FrontDev fd, const int2* __restrict__ tasks, int k) {
    __shared__ __align__(16) float As[PB][FF_TILE];
    __shared__ __align__(16) float Bs[PB][FF_TILE + 4];
    const int2 task = tasks[blockIdx.x];
    const int s = task.x;
    const bool inv = (task.y >> 30) & 1;
    const int r0 = ((task.y >> 15) & 0x7fff) * FF_TILE, c0 = (task.y & 0x7fff) * FF_TILE;
    const int f = fd.f[s], p = fd.p[s], k0 = k * PB, kb = min(PB, p - k0);
    const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
    float* C;                              // the tile's matrix, column-major
    int ld, nr, nc;
    if (!inv) {
        const int n2 = f - k0 - kb;
        float* Fp = fd.pool + fd.off[s] + (long)k0 * f + k0 + kb;      // L's rows below the block
        const float* D = fd.binv + fd.binv_off[s] + (long)k * PB * PB;
        C = Fp + (long)kb * f;
        ld = f;
        nr = nc = n2;
#pragma unroll
        for (int e = tid; e < PB * FF_TILE; e += 256) {
            const int r = e % FF_TILE, c = e / FF_TILE;
            const bool on = c < kb;
            As[c][r] = (on && r0 + r < n2) ? Fp[(long)c * f + r0 + r] : 0.0f;
            Bs[c][r] = (on && c0 + r < n2) ? -Fp[(long)c * f + c0 + r] * D[c * PB + c] : 0.0f;
        }
    } else {
        float* X = fd.linv + fd.linv_off[s];
        const int rows = p - k0 - kb;
        C = X + k0 + kb;
        ld = p;
        nr = rows;
        nc = k0;
#pragma unroll
        for (int e = tid; e < PB * FF_TILE; e += 256) {
            const int r = e % FF_TILE, c = e / FF_TILE;
            As[c][r] = r0 + r < rows ? X[(long)(k0 + c) * p + k0 + kb + r0 + r] : 0.0f;
            const int j = e % PB, cc = e / PB;
            Bs[j][cc] = c0 + cc < k0 ? X[(long)(c0 + cc) * p + k0 + j] : 0.0f;
        }
    }
    float acc[4][4];
    bool on[4][4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
        const int c = c0 + 4 * ty + v;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int r = r0 + tx + 16 * u;
            on[u][v] = r < nr && c < nc && (inv || c <= r);
            acc[u][v] = on[u][v] ? C[(long)c * ld + r] : 0.0f;
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
            if (on[u][v]) C[(long)(c0 + 4 * ty + v) * ld + r0 + tx + 16 * u] = acc[u][v];
}

// Block row k of one front: writes the factorised diagonal block into the front,
// inverts it (B_k, column per lane) and completes X_kJ = B_k W_kJ for FF_FCOLS
// columns (one per thread).
__global__ void __launch_bounds__(FF_PT) k_ff_finish(FrontDev fd, const int2* __restrict__ tasks) {
    __shared__ __align__(16) float Ls[PB * LSS];
    __shared__ __align__(16) float Bs[PB * LSS];
    const int2 task = tasks[blockIdx.x];
    const int s = task.x, k = task.y >> 16, ch = task.y & 0xffff;
    const int f = fd.f[s], p = fd.p[s], k0 = k * PB, kb = min(PB, p - k0);
    const int tid = threadIdx.x, lane = tid & 31;
    const float* blk = fd.binv + fd.binv_off[s] + (long)k * PB * PB;
    float* F = fd.pool + fd.off[s] + (long)k0 * f + k0;
    float* X = fd.linv + fd.linv_off[s];
    for (int e = tid; e < PB * PB; e += FF_PT) {
        const int r = e % PB, c = e / PB;
        const float v = blk[e];
        if (ch == 0 && r >= c && r < kb) F[(long)c * f + r] = v;
        Ls[r * LSS + c] = r > c ? v : 0.0f;
    }
    __syncthreads();
    if (tid < 32) {
        float x[PB];                       // column `lane` of L^-1
#pragma unroll
        for (int i = 0; i < PB; ++i) {
            float t = i == lane ? 1.0f : 0.0f;
#pragma unroll
            for (int q = 0; q < i; ++q) t -= Ls[i * LSS + q] * x[q];
            x[i] = i >= lane ? t : 0.0f;
            Bs[i * LSS + lane] = x[i];
        }
        if (ch == 0 && lane < kb)
#pragma unroll
            for (int i = 0; i < PB; ++i)
                if (i >= lane && i < kb) X[(long)(k0 + lane) * p + k0 + i] = x[i];
    }
    __syncthreads();
    const int c = ch * FF_FCOLS + tid;
    if (c >= k0) return;
    float* col = X + (long)c * p + k0;
    float w[PB];
#pragma unroll
    for (int q = 0; q < PB; ++q) w[q] = q < kb ? col[q] : 0.0f;
#pragma unroll
    for (int r = PB - 1; r > 0; --r) {     // in place, last row first
        float t = w[r];
#pragma unroll
        for (int q = 0; q < r; ++q) t += Bs[r * LSS + q] * w[q];
        w[r] = t;
    }
#pragma unroll
    for (int q = 0; q < PB; ++q)
        if (q < kb) col[q] = w[q];
}

inline int cdiv(int a, int b) { return (a + b - 1) / b; }

}  // namespace

// Tile lists of every level's launches, in launch order.
void ff_plan(const HostFronts& fr, FrontPlan& pl, std::vector<int2>& tasks) {
    pl = FrontPlan();
    tasks.clear();
    const int nl = (int)fr.lvl_ptr.size() - 1;
    for (int l = 0; l < nl; ++l) {
        const int q0 = fr.lvl_ptr[l], q1 = fr.lvl_ptr[l + 1];
        auto close = [&](int kind, int k) {
            const int begin = pl.launches.empty() ? 0 : pl.launches.back().begin + pl.launches.back().count;
            if ((int)tasks.size() > begin) pl.launches.push_back(FrontLaunch{kind, k, l, begin, (int)tasks.size() - begin});
        };
        int mp = 0;
        for (int q = q0; q < q1; ++q) {
            const int s = fr.lvl_sn[q];
            mp = std::max(mp, fr.p[s]);
            if (fr.cptr[s] == fr.cptr[s + 1]) continue;
            const int n = cdiv(fr.f[s], FF_TILE);
            for (int i = 0; i < n; ++i)
                for (int j = 0; j <= i; ++j) tasks.push_back(make_int2(s, (i << 16) | j));
        }
        close(FF_EXTEND, 0);
        for (int k = 0; k * PB < mp; ++k) {
            for (int q = q0; q < q1; ++q) {
                const int s = fr.lvl_sn[q], k0 = k * PB;
                if (k0 >= fr.p[s]) continue;
                const int below = fr.f[s] - k0 - std::min(PB, fr.p[s] - k0);
                for (int rb = 0; rb < std::max(1, cdiv(below, FF_ROWS)); ++rb) tasks.push_back(make_int2(s, rb));
            }
            close(FF_PANEL, k);
            for (int q = q0; q < q1; ++q) {
                const int s = fr.lvl_sn[q], k0 = k * PB;
                if (k0 >= fr.p[s]) continue;
                const int kb = std::min(PB, fr.p[s] - k0);
                const int n = cdiv(fr.f[s] - k0 - kb, FF_TILE);
                for (int i = 0; i < n; ++i)
                    for (int j = 0; j <= i; ++j) tasks.push_back(make_int2(s, (i << 15) | j));
                const int ni = cdiv(fr.p[s] - k0 - kb, FF_TILE), nj = cdiv(k0, FF_TILE);
                for (int i = 0; i < ni; ++i)
                    for (int j = 0; j < nj; ++j) tasks.push_back(make_int2(s, (1 << 30) | (i << 15) | j));
            }
            close(FF_UPDATE, k);
        }
        for (int q = q0; q < q1; ++q) {
            const int s = fr.lvl_sn[q];
            for (int k = 0; k * PB < fr.p[s]; ++k)
                for (int ch = 0; ch < std::max(1, cdiv(k * PB, FF_FCOLS)); ++ch)
                    tasks.push_back(make_int2(s, (k << 16) | ch));
        }
        close(FF_FINISH, 0);
    }
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
        else k_ff_finish<<<a.count, FF_PT, 0, s>>>(fd, t);
    }
    if (kt && level >= 0) kt->end(DC_KT_FRONT);
}

// One dense front through the factorisation: the test hook behind
// dc_debug_front_factor (synchronous; allocates and frees its own buffers).
dc_status ff_debug_factor(int n, int p, const float* A, float* out, float* linv_out, std::string* err) {
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
    ff_plan(fr, pl, tasks);
    const int nbk = cdiv(p, PB);
    // device image: ints [f, p, cptr0, cptr1], long longs [off, binv_off, linv_off]
    int hi[4] = {n, p, 0, 0};
    long long hl[3] = {0, 0, 0};
    float tau = 1e-30f;
    int* di = nullptr;
    long long* dl = nullptr;
    int2* dt = nullptr;
    float *pool = nullptr, *binv = nullptr, *linv = nullptr, *dtau = nullptr;
    cudaError_t e = cudaSuccess;
    do {
        if ((e = cudaMalloc(&di, sizeof(hi))) || (e = cudaMalloc(&dl, sizeof(hl))) ||
            (e = cudaMalloc(&dt, sizeof(int2) * tasks.size())) ||
            (e = cudaMalloc(&pool, sizeof(float) * (size_t)n * n)) ||
            (e = cudaMalloc(&binv, sizeof(float) * (size_t)nbk * PB * PB)) ||
            (e = cudaMalloc(&linv, sizeof(float) * (size_t)p * p)) || (e = cudaMalloc(&dtau, sizeof(float))) ||
            (e = cudaMemcpy(di, hi, sizeof(hi), cudaMemcpyHostToDevice)) ||
            (e = cudaMemcpy(dl, hl, sizeof(hl), cudaMemcpyHostToDevice)) ||
            (e = cudaMemcpy(dt, tasks.data(), sizeof(int2) * tasks.size(), cudaMemcpyHostToDevice)) ||
            (e = cudaMemcpy(dtau, &tau, sizeof(float), cudaMemcpyHostToDevice)) ||
            (e = cudaMemcpy(pool, A, sizeof(float) * (size_t)n * n, cudaMemcpyHostToDevice)) ||
            (e = cudaMemset(linv, 0, sizeof(float) * (size_t)p * p)))
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
        ff_factorize(fd, pl, nullptr, nullptr);
        if ((e = cudaGetLastError()) || (e = cudaDeviceSynchronize())) break;
        if ((e = cudaMemcpy(out, pool, sizeof(float) * (size_t)n * n, cudaMemcpyDeviceToHost))) break;
        if (linv_out) e = cudaMemcpy(linv_out, linv, sizeof(float) * (size_t)p * p, cudaMemcpyDeviceToHost);
    } while (false);
    cudaFree(di);
    cudaFree(dl);
    cudaFree(dt);
    cudaFree(pool);
    cudaFree(binv);
    cudaFree(linv);
    cudaFree(dtau);
    if (e != cudaSuccess) {
        *err = std::string("dc_debug_front_factor: ") + cudaGetErrorString(e);
        return DC_ERR_CUDA;
    }
    return DC_OK;
}
