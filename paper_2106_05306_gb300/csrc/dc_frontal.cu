// Per-step single-precision multifrontal LDL^T of the constrained adjoint
// matrix, used as the preconditioner of the FP64 adjoint Krylov solve.
//
// The matrix factorised is H^ = T H T + (I - T T) with H = P - Delta P - Delta R
// (Sec. 4, Eq. ppr_adjoint) and a per-node T: the identity for free nodes, 0 for
// stick nodes, the tangent-plane projector I - n n^T for slip nodes.  It differs
// from the exact constrained operator only by the obliqueness of the slip
// constraint and by single-precision rounding; the outer FP64 GMRES removes both.
// No pivoting beyond the supernode order; a pivot below tau is replaced by
// +-tau (the preconditioner stays usable, GMRES corrects).
//
// Fronts are dense column-major f x f blocks (DOF granularity, 3 per node) in
// one pool; only their lower triangles are used.  Their numeric factorisation is
// in dc_front_factor.cu; this file has the assembly and the solves.
#include <mutex>

#include "dc_adjoint.h"
#include "dc_internal.h"
#include "dc_wait.cuh"

namespace {

constexpr int FT = 1024;      // threads per solve CTA

__device__ __forceinline__ d4 ld(const d4* p) {
    const double2* q = reinterpret_cast<const double2*>(p);
    double2 a = q[0], b = q[1];
    d4 r;
    r.x = a.x; r.y = a.y; r.z = b.x; r.w = b.y;
    return r;
}
__device__ __forceinline__ void st(d4* p, double x, double y, double z, double w = 0.0) {
    double2* q = reinterpret_cast<double2*>(p);
    q[0] = make_double2(x, y);
    q[1] = make_double2(z, w);
}
inline int nblk(long n, int b) { return (int)((n + b - 1) / b); }

// Node transform of the constraint: 0 free, 1 stick, 2 slip (normal n).
__device__ __forceinline__ void node_T(int type, const double n[3], double T[9]) {
    for (int r = 0; r < 3; ++r)
        for (int c = 0; c < 3; ++c) {
            double v = (r == c) ? 1.0 : 0.0;
            if (type == 1) v = 0.0;
            else if (type == 2) v -= n[r] * n[c];
            T[3 * r + c] = v;
        }
}

// One 3x3 block H^_ij of the constrained matrix, written into its front.
__global__ void k_pairs(DevMesh dm, AdjDev ad, FrontDev fd) {
    int id = blockIdx.x * blockDim.x + threadIdx.x;
    if (id >= fd.NP) return;
    const int i = fd.pr_i[id], j = fd.pr_j[id];
    const double h2 = ad.h * ad.h;
    double H[9] = {0, 0, 0, 0, 0, 0, 0, 0, 0};
    for (int k = fd.pr_cptr[id]; k < fd.pr_cptr[id + 1]; ++k) {
        int code = fd.pr_code[k];
        if (code >= 0) {
            int t = code / 9, a = (code / 3) % 3, b = code % 3;
            d4 g = ld(dm.G + t);
            double ga0, ga1, gb0, gb1;
            if (a == 1) { ga0 = g.x; ga1 = g.y; } else if (a == 2) { ga0 = g.z; ga1 = g.w; }
            else { ga0 = -(g.x + g.z); ga1 = -(g.y + g.w); }
            if (b == 1) { gb0 = g.x; gb1 = g.y; } else if (b == 2) { gb0 = g.z; gb1 = g.w; }
            else { gb0 = -(g.x + g.z); gb1 = -(g.y + g.w); }
            const d4 A0 = ld(ad.tr0 + t), A1 = ld(ad.tr1 + t), A2 = ld(ad.tr2 + t);
            const double s00 = A0.w, s01 = A1.w, s11 = A2.x, itr = A2.y;
            // the triangle's a_a, a_b and projector P, formed once per triangle
            const d4 va = ld(ad.tav + 4 * (long)t + a), vb = ld(ad.tav + 4 * (long)t + b);
            const d4 pp = ld(ad.tav + 4 * (long)t + 3);
            const double aa[3] = {va.x, va.y, va.z}, ab[3] = {vb.x, vb.y, vb.z};
            const double P[9] = {pp.x, pp.y, pp.z, pp.y, pp.w, A2.z, pp.z, A2.z, A2.w};
            double w = h2 * dm.wt[t];
            double gg = ga0 * gb0 + ga1 * gb1;
            double gam = ga0 * gb0 * s00 + (ga0 * gb1 + ga1 * gb0) * s01 + ga1 * gb1 * s11;
            double trS = itr > 0.0 ? 1.0 / itr : 0.0;   // 0 for a collapsed triangle (a_a = a_b = 0)
            // block = w ((g_a.g_b) I - trS a_a a_b^T - gam P)
            for (int r = 0; r < 3; ++r)
                for (int c = 0; c < 3; ++c) {
                    double dl = (r == c) ? 1.0 : 0.0;
                    H[3 * r + c] += w * (gg * dl - trS * aa[r] * ab[c] - gam * P[3 * r + c]);
                }
        } else {
            int b = -code - 1;
            d4 q = ld(ad.bq + b);
            double w = h2 * dm.wb[b] * fd.pr_coef[k];
            double qh[3] = {q.x, q.y, q.z};
            for (int r = 0; r < 3; ++r)
                for (int c = 0; c < 3; ++c)
                    H[3 * r + c] += w * (((r == c) ? (1.0 - q.w) : 0.0) + q.w * qh[r] * qh[c]);
        }
    }
    int ti = ad.type[i], tj = ad.type[j];
    if (i == j) {
        double mi = dm.mass[i];
        H[0] += mi; H[4] += mi; H[8] += mi;
        if (ti == 2) {
            d4 sl = ld(ad.slip + i), nb = ld(ad.nb + i);
            double th[3] = {sl.x, sl.y, sl.z}, n[3] = {nb.x, nb.y, nb.z};
            double bh[3] = {n[1] * th[2] - n[2] * th[1], n[2] * th[0] - n[0] * th[2], n[0] * th[1] - n[1] * th[0]};
            for (int r = 0; r < 3; ++r)
                for (int c = 0; c < 3; ++c) H[3 * r + c] += sl.w * bh[r] * bh[c];
        }
    }
    double Hc[9];
    if (ti == 0 && tj == 0) {
        for (int q = 0; q < 9; ++q) Hc[q] = H[q];
    } else {
        double ni[3] = {0, 0, 0}, nj[3] = {0, 0, 0};
        if (ti == 2) { d4 nb = ld(ad.nb + i); ni[0] = nb.x; ni[1] = nb.y; ni[2] = nb.z; }
        if (tj == 2) { d4 nb = ld(ad.nb + j); nj[0] = nb.x; nj[1] = nb.y; nj[2] = nb.z; }
        double Ti[9], Tj[9], M1[9];
        node_T(ti, ni, Ti);
        node_T(tj, nj, Tj);
        for (int r = 0; r < 3; ++r)
            for (int c = 0; c < 3; ++c) {
                double s = 0;
                for (int q = 0; q < 3; ++q) s += H[3 * r + q] * Tj[3 * q + c];
                M1[3 * r + c] = s;
            }
        for (int r = 0; r < 3; ++r)
            for (int c = 0; c < 3; ++c) {
                double s = 0;
                for (int q = 0; q < 3; ++q) s += Ti[3 * r + q] * M1[3 * q + c];
                Hc[3 * r + c] = s;
            }
        if (i == j)   // + (I - T): identity on the constrained directions
            for (int q = 0; q < 9; ++q) Hc[q] += ((q % 4) == 0 ? 1.0 : 0.0) - Ti[q];
    }
    float* F = fd.pool + fd.pr_dst[id];
    const long ldf = fd.pr_ld[id];
    for (int c = 0; c < 3; ++c)
        for (int r = 0; r < 3; ++r) F[c * ldf + r] = (float)Hc[3 * r + c];
}

// Issues L2 prefetches for [p, p + bytes) (128-byte lines, spread over the CTA),
// so that a front's blocks stream in from HBM while the CTA gathers its inputs.
__device__ __forceinline__ void prefetch_l2(const void* p, size_t bytes) {
    const char* c = static_cast<const char*>(p);
    for (size_t o = (size_t)threadIdx.x * 128; o < bytes; o += (size_t)blockDim.x * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(c + o));
}

// Column-major matrix-vector product on one CTA: t_i = sum_k A[k * lda + i] v_k for
// rows i < nrows and k < K (k <= i when tri).  Rows go in passes of GV_ROWS; the
// k range is cut into G contiguous chunks with G a function of K alone, every
// (row, chunk) partial sum is one work item (consecutive items take consecutive
// rows: coalesced), and a row's partial sums are added in chunk order.  The
// arithmetic thus depends only on (nrows, K), never on the CTA size, so a front
// gives the same bits whatever else shares its level.  fin(i, t_i) stores.
constexpr int GV_ROWS = 128;
constexpr int GV_MAXG = 8;
__host__ __device__ constexpr int gv_groups(int K) { return K <= 8 ? 1 : (K + 7) / 8 < GV_MAXG ? (K + 7) / 8 : GV_MAXG; }

template <class Fin>
__device__ __forceinline__ void cm_gemv(const float* __restrict__ A, long lda, int nrows, int K, bool tri,
                                        const float* __restrict__ v, float* __restrict__ red, Fin fin) {
    const int nt = blockDim.x, tid = threadIdx.x;
    const int G = gv_groups(K);
    const int C = (K + G - 1) / G;
    for (int i0 = 0; i0 < nrows; i0 += GV_ROWS) {
        for (int item = tid; item < GV_ROWS * G; item += nt) {
            const int r = item % GV_ROWS, g = item / GV_ROWS, i = i0 + r;
            float acc = 0.0f;
            if (i < nrows) {
                const int k0 = g * C;
                int k1 = min(K, k0 + C);
                if (tri) k1 = min(k1, i + 1);
                const float* a = A + i;
#pragma unroll 4
                for (int k = k0; k < k1; ++k) acc += a[(long)k * lda] * v[k];
            }
            red[g * GV_ROWS + r] = acc;
        }
        __syncthreads();
        if (tid < GV_ROWS && i0 + tid < nrows) {
            float t = 0.0f;
            for (int q = 0; q < G; ++q) t += red[q * GV_ROWS + tid];
            fin(i0 + tid, t);
        }
        __syncthreads();
    }
}

// The blocks a front's solves read, fetched into L2 ahead of use.
__device__ __forceinline__ void msolve_prefetch(const FrontDev& fd, int s) {
    const int f = fd.f[s], p = fd.p[s];
    prefetch_l2(fd.linv + fd.linv_off[s], sizeof(float) * p * p);
    prefetch_l2(fd.pool + fd.off[s], sizeof(float) * (size_t)p * f);
}

// Forward substitution L y = r for front s (one CTA), then z = D^-1 y.  y_s =
// L_ss^-1 w_s with the stored explicit inverse; the rows below accumulate
// -L_Us y_s into the front's update vector, which the parent adds in.  The
// children's update vectors are read through L2 (other CTAs of a tree-scheduled
// launch write them).
__device__ __forceinline__ void msolve_fwd_front(const FrontDev& fd, int s, float* __restrict__ w) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const float* F = fd.pool + fd.off[s];
    const float* X = fd.linv + fd.linv_off[s];
    const int f = fd.f[s], p = fd.p[s];
    const int base = 3 * fd.begin[s];
    float* y = w + f;
    float* red = y + f;                // [GV_MAXG][GV_ROWS] partial sums
    // w = the children's update entries (pull lists: children in order), then r
    // on the pivots -- the sums of a child-by-child scatter into zeroed storage
    const int* pp = fd.pull_ptr + fd.pull_off[s];
    for (int t = tid; t < f; t += nt) {
        const int node = t / 3, comp = t - 3 * node;
        float a = 0.0f;
        for (int e = pp[node]; e < pp[node + 1]; ++e) a += __ldcg(fd.acc + fd.pull_idx[e] + comp);
        if (t < p) a += fd.rvec[base + t];
        w[t] = a;
    }
    __syncthreads();
    cm_gemv(X, p, p, p, true, w, red, [&](int i, float t) { y[i] = t; });
    float* acc = fd.acc + fd.acc_off[s];
    cm_gemv(F + p, f, f - p, p, false, y, red, [&](int i, float t) { acc[i] = w[p + i] - t; });
    for (int t = tid; t < p; t += nt) fd.zvec[base + t] = y[t] / F[(long)t * f + t];
}

// Forward substitution over one level (CTA per front of sn_list).
__global__ void __launch_bounds__(FT) k_msolve_fwd(FrontDev fd, const int* __restrict__ sn_list,
                                                    const double* __restrict__ mask) {
    extern __shared__ float w[];
    const int s = sn_list[blockIdx.x];
    if (mask && mask[fd.sn_inst[s]] == 0.0) return;
    msolve_prefetch(fd, s);
    msolve_fwd_front(fd, s, w);
}

// Backward substitution L^T x = z for front s (one CTA), top-down: x_s =
// L_ss^-T (z_s - L_Us^T x_U).  One warp per row (lanes along the row), two rows
// per warp at a time; a row's sum does not depend on the CTA size.  x_U is read
// through L2 (the ancestors' CTAs of a tree-scheduled launch write it).
__device__ __forceinline__ void msolve_bwd_front(const FrontDev& fd, int s, float* __restrict__ sm) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const float* F = fd.pool + fd.off[s];
    const float* X = fd.linv + fd.linv_off[s];
    const int f = fd.f[s], p = fd.p[s], nu = f - p;
    const int base = 3 * fd.begin[s];
    float* w = sm;
    float* xu = sm + p;
    const int* un = fd.unode + fd.uptr[s];
    for (int t = tid; t < p; t += nt) w[t] = fd.zvec[base + t];
    for (int k = tid; k < nu; k += nt) xu[k] = __ldcg(fd.xvec + 3 * un[k / 3] + k % 3);
    __syncthreads();
    const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
    for (int t = warp; t < p; t += 2 * nw) {
        const int t2 = t + nw;
        const bool two = t2 < p;
        const float* r1 = F + (long)t * f + p;
        const float* r2 = F + (long)(two ? t2 : t) * f + p;
        float s1 = 0.0f, s2 = 0.0f;
        for (int k = lane; k < nu; k += 32) {
            const float x = xu[k];
            s1 += r1[k] * x;
            s2 += r2[k] * x;
        }
        for (int o = 16; o > 0; o >>= 1) {
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        if (lane == 0) {
            w[t] -= s1;
            if (two) w[t2] -= s2;
        }
    }
    __syncthreads();
    for (int i = warp; i < p; i += 2 * nw) {
        const int i2 = i + nw;
        const bool two = i2 < p;
        const float* c1 = X + (long)i * p;   // column i of L_ss^-1 = row i of L_ss^-T
        const float* c2 = X + (long)(two ? i2 : i) * p;
        float s1 = 0.0f, s2 = 0.0f;
        for (int k = i + lane; k < p; k += 32) s1 += c1[k] * w[k];
        if (two)
            for (int k = i2 + lane; k < p; k += 32) s2 += c2[k] * w[k];
        for (int o = 16; o > 0; o >>= 1) {
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        if (lane == 0) {
            fd.xvec[base + i] = s1;
            if (two) fd.xvec[base + i2] = s2;
        }
    }
}

// Backward substitution over one level (CTA per front of sn_list).
__global__ void __launch_bounds__(FT) k_msolve_bwd(FrontDev fd, const int* __restrict__ sn_list,
                                                    const double* __restrict__ mask) {
    extern __shared__ float sm[];
    const int s = sn_list[blockIdx.x];
    if (mask && mask[fd.sn_inst[s]] == 0.0) return;
    msolve_prefetch(fd, s);
    msolve_bwd_front(fd, s, sm);
}

// Tree-scheduled solves: one launch per sweep.  Persistent CTAs take the fronts
// of items[0 .. n_items) (a topological order, children first) from a ticket
// counter; the backward sweep takes them in reverse.  Before a front a CTA waits
// (bounded, dc_wait.cuh) for its children's done flags (forward) or its
// parent's (backward).  A front is only ever waited on by fronts of its own
// instance, and an instance is masked whole, so a masked front is skipped
// without a flag.  An item waits only on items with smaller tickets, held by
// CTAs already running, so the launch completes whatever the number resident.
// Threads per CTA of a tree-scheduled solve: the fronts on the dependency chain
// are the large ones, so wide CTAs pay (measured on the 256-cloth batch: 128
// threads 1.50 s, 256 threads 1.09 s, 512 threads 1.02 s of solves per bench step).
constexpr int MT = 512;

__device__ __forceinline__ int ms_take(const FrontDev& fd, int* ticket, int n_items, int* s_item) {
    if (threadIdx.x == 0) *s_item = dc_fault_set(fd.fault) ? n_items : atomicAdd(ticket, 1);
    __syncthreads();
    const int t = *s_item;
    __syncthreads();   // every thread has read the ticket before it is rewritten
    return t;
}

__global__ void __launch_bounds__(MT) k_msolve_fwd_tree(FrontDev fd, const int* __restrict__ items, int n_items,
                                                        const double* __restrict__ mask) {
    extern __shared__ float w[];
    __shared__ int s_item, s_ok;
    int* ticket = fd.sched;
    int* done = fd.sched + 1;
    for (;;) {
        const int t = ms_take(fd, ticket, n_items, &s_item);
        if (t >= n_items) return;
        const int s = items[t];
        if (mask && mask[fd.sn_inst[s]] == 0.0) continue;
        msolve_prefetch(fd, s);
        if (threadIdx.x == 0) {
            bool ok = true;
            for (int q = fd.cptr[s]; ok && q < fd.cptr[s + 1]; ++q) ok = dc_wait_flag(done + fd.child[q], fd.fault);
            s_ok = ok;
        }
        __syncthreads();
        if (!s_ok) return;
        msolve_fwd_front(fd, s, w);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) dc_st_release(done + s, 1);
    }
}

__global__ void __launch_bounds__(MT) k_msolve_bwd_tree(FrontDev fd, const int* __restrict__ items, int n_items,
                                                        const double* __restrict__ mask) {
    extern __shared__ float sm[];
    __shared__ int s_item, s_ok;
    int* ticket = fd.sched + fd.S + 1;
    int* done = fd.sched + fd.S + 2;
    for (;;) {
        const int t = ms_take(fd, ticket, n_items, &s_item);
        if (t >= n_items) return;
        const int s = items[n_items - 1 - t];
        if (mask && mask[fd.sn_inst[s]] == 0.0) continue;
        msolve_prefetch(fd, s);
        if (threadIdx.x == 0) {
            const int par = fd.parent[s];
            s_ok = par < 0 || dc_wait_flag(done + par, fd.fault);
        }
        __syncthreads();
        if (!s_ok) return;
        msolve_bwd_front(fd, s, sm);
        __threadfence();
        __syncthreads();
        if (threadIdx.x == 0) dc_st_release(done + s, 1);
    }
}

// r = Pi_B w in single precision (DOF order 3*node + c).
__global__ void k_pre_in(int n, const int* __restrict__ type, const d4* __restrict__ nb, const d4* __restrict__ w,
                         float* __restrict__ r, const int* __restrict__ node_inst, const double* __restrict__ mask) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    if (mask && mask[node_inst[j]] == 0.0) return;
    d4 a = ld(w + j);
    double v[3] = {a.x, a.y, a.z};
    int ty = type[j];
    if (ty == 1) {
        v[0] = v[1] = v[2] = 0.0;
    } else if (ty == 2) {
        d4 q = ld(nb + j);
        double s = q.x * v[0] + q.y * v[1] + q.z * v[2];
        v[0] -= s * q.x; v[1] -= s * q.y; v[2] -= s * q.z;
    }
    r[3 * j] = (float)v[0];
    r[3 * j + 1] = (float)v[1];
    r[3 * j + 2] = (float)v[2];
}

// out = S_C x in double precision: stick -> 0, slip -> x - n ((n - mu t).x).
__global__ void k_pre_out(int n, const double* __restrict__ mu, const int* __restrict__ type, const d4* __restrict__ nb,
                          const d4* __restrict__ slip, const float* __restrict__ x, d4* __restrict__ out,
                          const int* __restrict__ node_inst, const double* __restrict__ mask) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    if (mask && mask[node_inst[j]] == 0.0) return;
    double v[3] = {(double)x[3 * j], (double)x[3 * j + 1], (double)x[3 * j + 2]};
    int ty = type[j];
    if (ty == 1) {
        v[0] = v[1] = v[2] = 0.0;
    } else if (ty == 2) {
        d4 q = ld(nb + j), sl = ld(slip + j);
        const double mj = mu[j];
        double cz = (q.x - mj * sl.x) * v[0] + (q.y - mj * sl.y) * v[1] + (q.z - mj * sl.z) * v[2];
        v[0] -= cz * q.x; v[1] -= cz * q.y; v[2] -= cz * q.z;
    }
    st(out + j, v[0], v[1], v[2]);
}

}  // namespace

size_t frontal_solve_smem(int max_f) { return (2 * (size_t)max_f + GV_ROWS * GV_MAXG) * sizeof(float) + 64; }

// The dynamic shared-memory limit of the solve kernels is a per-function
// attribute shared by every context of the process, so it only ever grows.
cudaError_t frontal_configure(int max_f) {
    static std::mutex mu;
    static size_t solve_bytes = 48 * 1024;
    std::lock_guard<std::mutex> lock(mu);
    const size_t sb = frontal_solve_smem(max_f);
    if (sb > solve_bytes) {
        for (const void* k : {(const void*)k_msolve_fwd, (const void*)k_msolve_bwd, (const void*)k_msolve_fwd_tree,
                              (const void*)k_msolve_bwd_tree}) {
            cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sb);
            if (e != cudaSuccess) return e;
        }
        solve_bytes = sb;
    }
    return cudaSuccess;
}

cudaError_t frontal_tree_grid(int max_f, int* grid_f, int* grid_b, size_t* smem_out) {
    const size_t smem = frontal_solve_smem(max_f);
    *smem_out = smem;
    int dev = 0, sms = 0, nf = 0, nb = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nf, k_msolve_fwd_tree, MT, smem);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k_msolve_bwd_tree, MT, smem);
    if (e != cudaSuccess) return e;
    *grid_f = sms * (nf > 0 ? nf : 1);
    *grid_b = sms * (nb > 0 ? nb : 1);
    return cudaSuccess;
}

static int solve_threads(int mf) { return mf <= 64 ? 128 : (mf <= 128 ? 256 : (mf <= 256 ? 512 : FT)); }

void frontal_factorize(const DevMesh& dm, const AdjDev& ad, const FrontDev& fd, const FrontPlan& plan, cudaStream_t s,
                       KTimer* kt) {
    if (kt) kt->begin(DC_KT_ASSEMBLE);
    cudaMemsetAsync(fd.pool, 0, sizeof(float) * fd.pool_size, s);
    dc_note_launch();
    k_pairs<<<nblk(fd.NP, 128), 128, 0, s>>>(dm, ad, fd);
    if (kt) kt->end(DC_KT_ASSEMBLE);
    ff_factorize(fd, plan, s, kt);
}

void frontal_precond(const AdjDev& ad, const FrontDev& fd, const int* lvl_ptr, int nlev, const int* lvl_maxf,
                     int n_free, const d4* w, d4* out, cudaStream_t s, KTimer* kt, const int* act_sn,
                     const int* act_ptr, const int* act_tq, int n_act_tq) {
    dc_note_launch();
    k_pre_in<<<nblk(n_free, 128), 128, 0, s>>>(n_free, ad.type, ad.nb, w, fd.rvec, ad.node_inst, ad.mask);
    if (fd.tree) {
        const int* items = act_tq ? act_tq : fd.tq;
        const int n = act_tq ? n_act_tq : fd.S;
        if (n > 0) {
            cudaMemsetAsync(fd.sched, 0, sizeof(int) * 2 * ((size_t)fd.S + 1), s);
            if (kt) kt->begin(DC_KT_MSOLVE);
            dc_note_launch();
            k_msolve_fwd_tree<<<n < fd.tree_grid_f ? n : fd.tree_grid_f, MT, fd.tree_smem, s>>>(fd, items, n, ad.mask);
            dc_note_launch();
            k_msolve_bwd_tree<<<n < fd.tree_grid_b ? n : fd.tree_grid_b, MT, fd.tree_smem, s>>>(fd, items, n, ad.mask);
            if (kt) kt->end(DC_KT_MSOLVE);
        }
        dc_note_launch();
        k_pre_out<<<nblk(n_free, 128), 128, 0, s>>>(n_free, ad.mu, ad.type, ad.nb, ad.slip, fd.xvec, out,
                                                      ad.node_inst, ad.mask);
        return;
    }
    // level l's fronts: the compacted list of the active instances' fronts, or all of them
    auto level = [&](int l, int& cnt) -> const int* {
        if (act_sn) {
            cnt = act_ptr[l + 1] - act_ptr[l];
            return act_sn + act_ptr[l];
        }
        cnt = lvl_ptr[l + 1] - lvl_ptr[l];
        return fd.lvl_sn + lvl_ptr[l];
    };
    for (int l = 0; l < nlev; ++l) {
        int cnt;
        const int* sn = level(l, cnt);
        if (cnt > 0) {
            const int mf = lvl_maxf[l];
            dc_note_launch();
            if (kt) kt->begin(DC_KT_MSOLVE);
            k_msolve_fwd<<<cnt, solve_threads(mf), frontal_solve_smem(mf), s>>>(fd, sn, ad.mask);
            if (kt) kt->end(DC_KT_MSOLVE);
        }
    }
    for (int l = nlev - 1; l >= 0; --l) {
        int cnt;
        const int* sn = level(l, cnt);
        if (cnt > 0) {
            const int mf = lvl_maxf[l];
            dc_note_launch();
            if (kt) kt->begin(DC_KT_MSOLVE);
            k_msolve_bwd<<<cnt, solve_threads(mf), frontal_solve_smem(mf), s>>>(fd, sn, ad.mask);
            if (kt) kt->end(DC_KT_MSOLVE);
        }
    }
    dc_note_launch();
    k_pre_out<<<nblk(n_free, 128), 128, 0, s>>>(n_free, ad.mu, ad.type, ad.nb, ad.slip, fd.xvec, out,
                                                  ad.node_inst, ad.mask);
}
