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
#include <algorithm>
#include <mutex>
#include <utility>
#include <vector>

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

// One 3x3 block H^_ij of the constrained matrix, written into its front.  A thread's FP64
// chain bounds it; the pairs come sorted by the length of their sums, 1/(1/tr S) is formed
// per triangle and flat bending adds only its diagonal: 2308 -> 377 us for 96 cloths
// (161000 nodes).
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
            const double s00 = A0.w, s01 = A1.w, s11 = A2.x;
            // the triangle's a_a, a_b and projector P, formed once per triangle
            const d4 va = ld(ad.tav + 4 * (long)t + a), vb = ld(ad.tav + 4 * (long)t + b);
            const d4 pp = ld(ad.tav + 4 * (long)t + 3);
            const double aa[3] = {va.x, va.y, va.z}, ab[3] = {vb.x, vb.y, vb.z};
            const double P[9] = {pp.x, pp.y, pp.z, pp.y, pp.w, A2.z, pp.z, A2.z, A2.w};
            double w = h2 * dm.wt[t];
            double gg = ga0 * gb0 + ga1 * gb1;
            double gam = ga0 * gb0 * s00 + (ga0 * gb1 + ga1 * gb0) * s01 + ga1 * gb1 * s11;
            const double trS = va.w;
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
            if (q.w == 0.0) {               // constant projection (q_hat = 0): w I
                H[0] += w; H[4] += w; H[8] += w;
                continue;
            }
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

// Column-major matrix-vector product on one CTA: t_i = sum_k A[k * lda + i] v_k for rows
// r_lo <= i < r_hi and k < K (k <= i when TRI).  Rows go in passes of GV_ROWS; the k range
// is cut into at most GV_MAXG contiguous chunks, their number a function of K alone, every
// (row, chunk) partial sum is one work item (consecutive items take consecutive rows:
// coalesced), and a row's partial sums are added in chunk order.  A row's arithmetic
// thus depends only on (i, K), never on the CTA size or on the rows that share its CTA.
// PAD: items of a pass are numbered for GV_ROWS rows (whole fronts), else for the rows
// there are (short row blocks).  fin(i, t_i) stores.
constexpr int GV_ROWS = 128;
constexpr int GV_MAXG = 8;
__host__ __device__ constexpr int gv_groups(int K) { return K <= 8 ? 1 : (K + 7) / 8 < GV_MAXG ? (K + 7) / 8 : GV_MAXG; }

// PRE: the first GV_PRE entries of a thread's first two items come from its registers
// (GemvPre, loaded before the vector was there); after() runs once the products of the first
// pass are formed.
constexpr int GV_PRE = 10;
struct GemvPre {
    float a[2][GV_PRE];
    template <bool TRI, bool PAD>
    __device__ __forceinline__ void load(const float* __restrict__ A, long lda, int r_lo, int r_hi, int K) {
        const int G = gv_groups(K), C = (K + G - 1) / G;
        const int R = min(GV_ROWS, r_hi - r_lo), Rp = PAD ? GV_ROWS : R;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int item = threadIdx.x + j * blockDim.x, g = item / Rp, r = item - g * Rp, i = r_lo + r;
            const int k0 = g * C;
            int k1 = item < Rp * G && r < R ? min(K, k0 + C) : 0;
            if (TRI) k1 = min(k1, i + 1);
            const float* p = A + i + (long)k0 * lda;
#pragma unroll
            for (int q = 0; q < GV_PRE; ++q) {
                a[j][q] = k0 + q < k1 ? *p : 0.0f;
                p += lda;
            }
        }
    }
};
struct GvNone {
    __device__ __forceinline__ void operator()() const {}
};

template <bool TRI, bool PAD, bool PRE = false, class Fin, class After = GvNone>
__device__ __forceinline__ void cm_gemv(const float* __restrict__ A, long lda, int r_lo, int r_hi, int K,
                                        const float* __restrict__ v, float* __restrict__ red, Fin fin,
                                        const GemvPre* pre = nullptr, After after = After()) {
    const int nt = blockDim.x, tid = threadIdx.x;
    const int G = gv_groups(K), C = (K + G - 1) / G;
    for (int i0 = r_lo; i0 < r_hi; i0 += GV_ROWS) {
        const int R = min(GV_ROWS, r_hi - i0), Rp = PAD ? GV_ROWS : R;
        int first = tid;
        if (PRE && i0 == r_lo) {
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int item = tid + j * nt, g = item / Rp, r = item - g * Rp, i = i0 + r;
                if (item >= Rp * G) break;
                float acc = 0.0f;
                if (r < R) {
                    const int k0 = g * C;
                    int k1 = min(K, k0 + C);
                    if (TRI) k1 = min(k1, i + 1);
#pragma unroll
                    for (int q = 0; q < GV_PRE; ++q)
                        if (k0 + q < k1) acc += pre->a[j][q] * v[k0 + q];
                    const float* a = A + i;
#pragma unroll 8
                    for (int k = k0 + GV_PRE; k < k1; ++k) acc += a[(long)k * lda] * v[k];
                }
                red[g * GV_ROWS + r] = acc;
            }
            after();
            first = tid + 2 * nt;
        }
        for (int item = first; item < Rp * G; item += nt) {
            const int g = item / Rp, r = item - g * Rp, i = i0 + r;
            float acc = 0.0f;
            if (r < R) {
                const int k0 = g * C;
                int k1 = min(K, k0 + C);
                if (TRI) k1 = min(k1, i + 1);
                const float* a = A + i;
#pragma unroll 4
                for (int k = k0; k < k1; ++k) acc += a[(long)k * lda] * v[k];
            }
            red[g * GV_ROWS + r] = acc;
        }
        __syncthreads();
        if (tid < R) {
            float t = 0.0f;
            for (int q = 0; q < G; ++q) t += red[q * GV_ROWS + tid];
            fin(i0 + tid, t);
        }
        __syncthreads();
    }
}

// Forward substitution L y = r for front s, then z = D^-1 y, in two halves: half A is
// y_s = L_ss^-1 w_s with the stored explicit inverse (and z_s), half B the update vector
// w_U - L_Us y_s that the parent adds in, each over rows [r_lo, r_hi).  w is the children's
// update entries (pull lists: children in order), then r on the pivots -- the sums of a
// child-by-child scatter into zeroed storage.  Vectors that other CTAs of a launch write
// are read through L2.
__device__ __forceinline__ float ms_pull(const FrontDev& fd, const int* __restrict__ pp, int t) {
    const int node = t / 3, comp = t - 3 * node;
    float a = 0.0f;
    for (int e = pp[node]; e < pp[node + 1]; ++e) a += __ldcg(fd.acc + fd.pull_idx[e] + comp);
    return a;
}
// The lookups of a position's pull list, and its value from them.
struct MsPull {
    int e0, e1, i0, i1;
};
__device__ __forceinline__ MsPull ms_pull_begin(const FrontDev& fd, const int* __restrict__ pp, int t) {
    const int node = t / 3;
    MsPull q{pp[node], pp[node + 1], 0, 0};
    if (q.e0 < q.e1) q.i0 = fd.pull_idx[q.e0];
    if (q.e0 + 1 < q.e1) q.i1 = fd.pull_idx[q.e0 + 1];
    return q;
}
__device__ __forceinline__ float ms_pull_end(const FrontDev& fd, const MsPull& q, int t) {
    const int comp = t % 3;
    const float x = q.e0 < q.e1 ? __ldcg(fd.acc + q.i0 + comp) : 0.0f;
    const float y = q.e0 + 1 < q.e1 ? __ldcg(fd.acc + q.i1 + comp) : 0.0f;
    float a = 0.0f;
    if (q.e0 < q.e1) a += x;
    if (q.e0 + 1 < q.e1) a += y;
    for (int e = q.e0 + 2; e < q.e1; ++e) a += __ldcg(fd.acc + fd.pull_idx[e] + comp);
    return a;
}
template <bool FEW, class Wait>
__device__ __forceinline__ bool ms_fwd_a(const FrontDev& fd, int s, int r_lo, int r_hi, float* __restrict__ w,
                                         Wait wait) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int f = fd.f[s], p = fd.p[s], base = 3 * fd.begin[s];
    const float* F = fd.pool + fd.off[s];
    float* red = w + p;                // [GV_MAXG][GV_ROWS] partial sums
    const int* pp = fd.pull_ptr + fd.pull_off[s];
    // the pivot of this thread's row of the first pass, ahead of the wait
    const float d0 = r_lo + tid < r_hi ? F[(long)(r_lo + tid) * f + r_lo + tid] : 1.0f;
    const float* X = fd.linv + fd.linv_off[s];
    GemvPre pre;
    MsPull pull{0, 0, 0, 0};
    float rv = 0.0f;
    if (FEW) {
        pre.load<true, false>(X, p, r_lo, r_hi, p);
        if (tid < r_hi) {
            pull = ms_pull_begin(fd, pp, tid);
            rv = fd.rvec[base + tid];
        }
    }
    if (!wait()) return false;
    if (FEW && tid < r_hi) w[tid] = ms_pull_end(fd, pull, tid) + rv;
    for (int t = FEW ? tid + nt : tid; t < r_hi; t += nt) w[t] = ms_pull(fd, pp, t) + fd.rvec[base + t];
    __syncthreads();
    cm_gemv<true, false, FEW>(X, p, r_lo, r_hi, p, w, red, [&](int i, float t) {
        fd.yvec[base + i] = t;
        fd.zvec[base + i] = t / (i == r_lo + tid ? d0 : F[(long)i * f + i]);
    }, &pre);
    return true;
}
template <bool FEW, class Wait>
__device__ __forceinline__ bool ms_fwd_b(const FrontDev& fd, int s, int r_lo, int r_hi, float* __restrict__ y,
                                         Wait wait) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int f = fd.f[s], p = fd.p[s], base = 3 * fd.begin[s], nr = r_hi - r_lo;
    float* w = y + p;                  // [nr]
    float* red = w + nr;               // [GV_MAXG][GV_ROWS]
    const int* pp = fd.pull_ptr + fd.pull_off[s];
    float* acc = fd.acc + fd.acc_off[s];
    const float* A = fd.pool + fd.off[s] + p;
    GemvPre pre;
    MsPull pull{0, 0, 0, 0};
    if (FEW) {
        pre.load<false, false>(A, f, r_lo, r_hi, p);
        if (tid < nr) pull = ms_pull_begin(fd, pp, p + r_lo + tid);
    }
    if (!wait()) return false;
    for (int t = tid; t < p; t += nt) y[t] = __ldcg(fd.yvec + base + t);
    if (FEW && tid < nr) w[tid] = ms_pull_end(fd, pull, p + r_lo + tid);
    for (int t = FEW ? tid + nt : tid; t < nr; t += nt) w[t] = ms_pull(fd, pp, p + r_lo + t);
    __syncthreads();
    cm_gemv<false, false, FEW>(A, f, r_lo, r_hi, p, y, red,
                               [&](int i, float t) { acc[i] = w[i - r_lo] - t; }, &pre);
    return true;
}

// Rows [r_lo, r_hi) of a row-major product, one warp per row (lanes along the row), two
// rows per warp at a time: t_i = sum_{k_lo(i) <= k < K} A[i * lda + k] v_k.  A row's sum does
// not depend on the CTA size.
template <bool UPPER, class Fin>
__device__ __forceinline__ void rm_gemv(const float* __restrict__ A, long lda, int r_lo, int r_hi, int K,
                                        const float* __restrict__ v, Fin fin) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int i = r_lo + warp; i < r_hi; i += 2 * nw) {
        const int i2 = i + nw;
        const bool two = i2 < r_hi;
        const float* r1 = A + (long)i * lda;
        const float* r2 = A + (long)(two ? i2 : i) * lda;
        float s1 = 0.0f, s2 = 0.0f;
        if (UPPER) {
#pragma unroll 4
            for (int k = i + lane; k < K; k += 32) s1 += r1[k] * v[k];
            if (two)
#pragma unroll 4
                for (int k = i2 + lane; k < K; k += 32) s2 += r2[k] * v[k];
        } else if (two) {
#pragma unroll 4
            for (int k = lane; k < K; k += 32) {
                const float x = v[k];
                s1 += r1[k] * x;
                s2 += r2[k] * x;
            }
        } else {
#pragma unroll 4
            for (int k = lane; k < K; k += 32) s1 += r1[k] * v[k];
        }
        for (int o = 16; o > 0; o >>= 1) {
            s1 += __shfl_xor_sync(0xffffffffu, s1, o);
            s2 += __shfl_xor_sync(0xffffffffu, s2, o);
        }
        if (lane == 0) {
            fin(i, s1);
            if (two) fin(i2, s2);
        }
    }
}

// Backward substitution L^T x = z for front s: half A is w_s = z_s - L_Us^T x_U (kept in
// yvec, which the forward sweep is done with), half B x_s = L_ss^-T w_s.
template <class Wait>
__device__ __forceinline__ bool ms_bwd_a(const FrontDev& fd, int s, int r_lo, int r_hi, float* __restrict__ xu,
                                         Wait wait) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int f = fd.f[s], p = fd.p[s], nu = f - p, base = 3 * fd.begin[s];
    const float* A = fd.pool + fd.off[s] + p;
    const int* un = fd.unode + fd.uptr[s];
    for (int i = r_lo + (tid >> 5); i < r_hi; i += nt >> 5)
        for (int k = 32 * (tid & 31); k < nu; k += 1024)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(A + (long)i * f + k));
    if (!wait()) return false;
    for (int k = tid; k < nu; k += nt) xu[k] = __ldcg(fd.xvec + 3 * un[k / 3] + k % 3);
    __syncthreads();
    rm_gemv<false>(A, f, r_lo, r_hi, nu, xu,
                   [&](int i, float t) { fd.yvec[base + i] = __ldcg(fd.zvec + base + i) - t; });
    __syncthreads();
    return true;
}
template <class Wait>
__device__ __forceinline__ bool ms_bwd_b(const FrontDev& fd, int s, int r_lo, int r_hi, float* __restrict__ w,
                                         Wait wait) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int p = fd.p[s], base = 3 * fd.begin[s];
    const float* X = fd.linv + fd.linv_off[s];   // column i of L_ss^-1 = row i of L_ss^-T
    for (int i = r_lo + (tid >> 5); i < r_hi; i += nt >> 5)
        for (int k = i + 32 * (tid & 31); k < p; k += 1024)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(X + (long)i * p + k));
    if (!wait()) return false;
    const float* src = fd.f[s] > p ? fd.yvec : fd.zvec;   // (a root has no half A)
    for (int t = r_lo + tid; t < p; t += nt) w[t] = __ldcg(src + base + t);
    __syncthreads();
    rm_gemv<true>(X, p, r_lo, r_hi, p, w, [&](int i, float t) { fd.xvec[base + i] = t; });
    __syncthreads();
    return true;
}

// The whole of front s on one CTA: both halves with the vectors kept in shared memory (the
// same sums in the same order).
template <bool FEW, class Wait>
__device__ __forceinline__ bool ms_fwd_whole(const FrontDev& fd, int s, float* __restrict__ w, Wait wait) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int f = fd.f[s], p = fd.p[s], base = 3 * fd.begin[s];
    const float* F = fd.pool + fd.off[s];
    float* y = w + f;
    float* red = y + p;                // [GV_MAXG][GV_ROWS]
    const int* pp = fd.pull_ptr + fd.pull_off[s];
    const float* X = fd.linv + fd.linv_off[s];
    GemvPre pre;
    MsPull pull{0, 0, 0, 0};
    float rv = 0.0f, d = 1.0f;
    if (FEW) {
        pre.load<true, true>(X, p, 0, p, p);
        if (tid < f) pull = ms_pull_begin(fd, pp, tid);
        if (tid < p) {
            rv = fd.rvec[base + tid];
            d = F[(long)tid * f + tid];
        }
    }
    if (!wait()) return false;
    if (FEW && tid < f) w[tid] = ms_pull_end(fd, pull, tid) + rv;
    for (int t = FEW ? tid + nt : tid; t < f; t += nt)
        w[t] = ms_pull(fd, pp, t) + (t < p ? fd.rvec[base + t] : 0.0f);
    __syncthreads();
    cm_gemv<true, true, FEW>(X, p, 0, p, p, w, red, [&](int i, float t) { y[i] = t; }, &pre,
                             [&]() { pre.load<false, true>(F + p, f, 0, f - p, p); });
    float* acc = fd.acc + fd.acc_off[s];
    cm_gemv<false, true, FEW>(F + p, f, 0, f - p, p, y, red, [&](int i, float t) { acc[i] = w[p + i] - t; }, &pre);
    for (int t = tid; t < p; t += nt) fd.zvec[base + t] = y[t] / (FEW && t == tid ? d : F[(long)t * f + t]);
    return true;
}
template <bool FEW, class Wait>
__device__ __forceinline__ bool ms_bwd_whole(const FrontDev& fd, int s, float* __restrict__ w, Wait wait) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int f = fd.f[s], p = fd.p[s], nu = f - p, base = 3 * fd.begin[s];
    const float* F = fd.pool + fd.off[s];
    float* xu = w + p;
    const int* un = fd.unode + fd.uptr[s];
    // zvec is the forward launch's
    int src = 0;
    if (FEW) {
        if (tid < nu) src = un[tid / 3];
        for (int t = tid; t < p; t += nt) w[t] = __ldcg(fd.zvec + base + t);
    }
    if (!wait()) return false;
    if (!FEW)
        for (int t = tid; t < p; t += nt) w[t] = __ldcg(fd.zvec + base + t);
    if (FEW && tid < nu) xu[tid] = __ldcg(fd.xvec + 3 * src + tid % 3);
    for (int k = FEW ? tid + nt : tid; k < nu; k += nt) xu[k] = __ldcg(fd.xvec + 3 * un[k / 3] + k % 3);
    __syncthreads();
    if (nu > 0) {
        rm_gemv<false>(F + p, f, 0, p, nu, xu, [&](int i, float t) { w[i] -= t; });
        __syncthreads();
    }
    rm_gemv<true>(fd.linv + fd.linv_off[s], p, 0, p, p, w, [&](int i, float t) { fd.xvec[base + i] = t; });
    __syncthreads();
    return true;
}

// A task of front s: rows of one half, or all of it (MS_AB).
template <bool fwd, bool FEW, class Wait>
__device__ __forceinline__ bool ms_front(const FrontDev& fd, int s, int phase, int r_lo, int r_hi,
                                         float* __restrict__ sm, Wait wait) {
    if (phase == MS_AB) return fwd ? ms_fwd_whole<FEW>(fd, s, sm, wait) : ms_bwd_whole<FEW>(fd, s, sm, wait);
    if (fwd)
        return phase == MS_A ? ms_fwd_a<FEW>(fd, s, r_lo, r_hi, sm, wait) : ms_fwd_b<FEW>(fd, s, r_lo, r_hi, sm, wait);
    return phase == MS_A ? ms_bwd_a(fd, s, r_lo, r_hi, sm, wait) : ms_bwd_b(fd, s, r_lo, r_hi, sm, wait);
}

// Substitution over one level (CTA per front of sn_list).
__global__ void __launch_bounds__(FT) k_msolve_fwd(FrontDev fd, const int* __restrict__ sn_list,
                                                    const double* __restrict__ mask) {
    extern __shared__ float sm[];
    const int s = sn_list[blockIdx.x];
    if (mask && mask[fd.sn_inst[s]] == 0.0) return;
    ms_front<true, false>(fd, s, MS_AB, 0, 0, sm, []() { return true; });
}
__global__ void __launch_bounds__(FT) k_msolve_bwd(FrontDev fd, const int* __restrict__ sn_list,
                                                    const double* __restrict__ mask) {
    extern __shared__ float sm[];
    const int s = sn_list[blockIdx.x];
    if (mask && mask[fd.sn_inst[s]] == 0.0) return;
    ms_front<false, false>(fd, s, MS_AB, 0, 0, sm, []() { return true; });
}

// Tree-scheduled solves, one launch per sweep.  Persistent CTAs take tasks -- a front, or
// some rows of one half of a large one -- from a ticket counter in a topological order
// (forward: children first; backward: parents first), and before a task wait (bounded,
// dc_wait.cuh) for what it reads: its front's children (forward), its parent (backward),
// or its own half A (half B).  A front is only ever waited on by fronts of its own
// instance, and an instance is masked whole, so a masked front is skipped without
// counting.  A task waits only on tasks with smaller tickets, held by CTAs already
// running, so a launch completes whatever the number resident.
// Why large fronts are split: one CTA reads the factor at about 0.1 TB/s, so the chain of
// the top fronts set the time while the chip waited (one 200 x 200 cloth: 2.35 ms for the
// two sweeps over a 0.5 GB factor).
// Threads per CTA and CTAs per SM: a front is a chain of latencies, so many CTAs share an SM
// where there are many fronts (96 cloths, the gradient call: forward at 3 CTAs 53.3 ms,
// at 4 51.2), and the fronts on the dependency chain are the large ones, so wide CTAs pay.
// FEW (at most MS_FEW fronts, 24 per SM): the time is the chain of fronts, each of them a
// chain of loads after its wait, so a thread loads its pull lists, right-hand side, pivots
// and the first entries of its rows before the wait and the second product's during the
// first.  That takes 64 registers, two CTAs an SM, which many fronts cannot spare.
// Measured, without -> with (us, gradient calls): 256-node cloth 14400 -> 13500, 61 x 61 nodes
// 21400 -> 20000, 200 x 200 nodes 49800 -> 47300; batches of 8 cloths of 16 x 16 nodes 6255 ->
// 6090, 4 of 32 x 32 9720 -> 9330, 16 of 24 x 24 9210 -> 9130, 12 of 40 x 40 15450 both; 96 cloths
// 47600 -> 49200.
constexpr int MT = 512;

template <bool FWD, bool FEW>
__global__ void __launch_bounds__(MT, FEW ? 2 : FWD ? 4 : 3) k_msolve_tree(FrontDev fd, const int* __restrict__ list, int n,
                                                       const double* __restrict__ mask) {
    extern __shared__ float sm[];
    __shared__ int s_item, s_ok;
    int* ticket = fd.sched + (FWD ? 0 : 2 * fd.S + 1);
    int* done = ticket + 1;                        // ends, then half-A ends
    for (;;) {
        if (threadIdx.x == 0) s_item = dc_fault_set(fd.fault) ? n : atomicAdd(ticket, 1);
        __syncthreads();
        const int t = s_item;
        if (t >= n) return;
        const int4 task = (FWD ? fd.ftask : fd.btask)[list ? list[t] : t];
        const int s = task.x, phase = task.y;
        if (mask && mask[fd.sn_inst[s]] == 0.0) {
            __syncthreads();                       // every thread has read the ticket
            continue;
        }
        if (phase == MS_AB) {
            const int f = fd.f[s], p = fd.p[s];
            prefetch_l2(fd.linv + fd.linv_off[s], sizeof(float) * p * p);
            prefetch_l2(fd.pool + fd.off[s], sizeof(float) * (size_t)p * f);
        }
        auto wait = [&]() {
            if (threadIdx.x == 0) {
                bool ok = true;
                if (phase == MS_B && fd.parent[s] >= 0) {
                    ok = dc_wait_count(done + fd.S + s, FWD ? fd.need[s].y : fd.need[s].w, fd.fault);
                } else if (FWD) {
                    for (int q = fd.cptr[s]; ok && q < fd.cptr[s + 1]; ++q)
                        ok = dc_wait_count(done + fd.child[q], fd.cneed[q], fd.fault);
                } else {
                    const int par = fd.parent[s];
                    ok = par < 0 || dc_wait_count(done + par, fd.need[par].z, fd.fault);
                }
                s_ok = ok;
            }
            __syncthreads();
            return s_ok != 0;
        };
        if (!ms_front<FWD, FEW>(fd, s, phase, task.z, task.w, sm, wait)) return;
        __syncthreads();
        if (threadIdx.x == 0) {
            const bool mid = phase == MS_A && fd.parent[s] >= 0;   // (a root's forward ends with half A)
            dc_add_release(done + (mid ? fd.S : 0) + s, 1);
        }
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
        for (const void* k : {(const void*)k_msolve_fwd, (const void*)k_msolve_bwd, (const void*)k_msolve_tree<true, false>,
                              (const void*)k_msolve_tree<false, false>, (const void*)k_msolve_tree<true, true>,
                              (const void*)k_msolve_tree<false, true>}) {
            cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sb);
            if (e != cudaSuccess) return e;
        }
        solve_bytes = sb;
    }
    return cudaSuccess;
}

cudaError_t frontal_tree_grid(int max_f, bool few, int* grid, size_t* smem_out) {
    const size_t smem = frontal_solve_smem(max_f);
    *smem_out = smem;
    int dev = 0, sms = 0, n = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = few ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_msolve_tree<true, true>, MT, smem)
                                 : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_msolve_tree<true, false>, MT, smem);
    if (e != cudaSuccess) return e;
    *grid = sms * (n > 0 ? n : 1);
    return cudaSuccess;
}

// Tasks of the tree-scheduled solve (FrontDev::ftask, btask, need): fronts farthest from
// their root first (backward: nearest first), those of one depth together: half A and
// whole fronts, then half B, so that a CTA waiting for a half A seldom holds up a task
// that is ready.  A front whose two products have at most `target` entries is one task;
// else each half is cut into row blocks of about that many, in multiples of eight rows (a
// 32-byte sector of every column): 16 tasks per SM and sweep, within [4096, 65536]
// entries (4096 entries, 16 KB, take an SM about 0.2 us, well below the cost of starting
// a task).  No split changes a bit of the result.
void ms_plan(const HostFronts& fr, const std::vector<int>& order, std::vector<int4>& ftask, std::vector<int4>& btask,
             std::vector<int4>& need) {
    long long total = 0;
    for (int s = 0; s < fr.S; ++s) total += (long long)fr.p[s] * (fr.p[s] + 1) / 2 + (long long)fr.p[s] * (fr.f[s] - fr.p[s]);
    const long long target = std::min<long long>(65536, std::max<long long>(4096, total / (DC_SMS * 16)));
    need.assign(fr.S, make_int4(1, 0, 1, 0));
    ftask.clear();
    btask.clear();
    auto blocks = [&](std::vector<int4>& out, int s, int phase, int rows, auto work) {
        int n = 0;
        for (int r = 0; r < rows; ++n) {
            long long w = 0;
            int e = r;
            while (e < rows && (w < target || e % 8)) w += work(e++);
            out.push_back(make_int4(s, phase, r, e));
            r = e;
        }
        return n;
    };
    std::vector<int> depth(fr.S, 0);
    for (int s = fr.S - 1; s >= 0; --s) depth[s] = fr.parent[s] >= 0 ? depth[fr.parent[s]] + 1 : 0;
    std::vector<std::pair<int, int>> span;   // fronts of one depth
    for (int q = 0; q < fr.S;) {
        int e = q;
        while (e < fr.S && depth[order[e]] == depth[order[q]]) ++e;
        span.push_back({q, e});
        q = e;
    }
    auto emit = [&](std::vector<int4>& out, const std::pair<int, int>& sp, bool fwd) {
        for (int second = 0; second < 2; ++second)
            for (int q = sp.first; q < sp.second; ++q) {
                const int s = order[q];
                const long long p = fr.p[s], nu = fr.f[s] - p;
                if (p * (p + 1) / 2 + p * nu <= target) {
                    if (!second) out.push_back(make_int4(s, MS_AB, 0, 0));
                } else if (fwd && !second) {
                    (nu > 0 ? need[s].y : need[s].x) = blocks(out, s, MS_A, (int)p, [&](int i) { return (long long)i + 1; });
                } else if (fwd && nu > 0) {
                    need[s].x = blocks(out, s, MS_B, (int)nu, [&](int) { return p; });
                } else if (!fwd && !second && nu > 0) {
                    need[s].w = blocks(out, s, MS_A, (int)p, [&](int) { return nu; });
                } else if (!fwd && second) {
                    need[s].z = blocks(out, s, MS_B, (int)p, [&](int i) { return p - i; });
                }
            }
    };
    for (const auto& sp : span) emit(ftask, sp, true);
    for (size_t k = span.size(); k-- > 0;) emit(btask, span[k], false);
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
                     const int* act_ptr, const int* act_f, int n_act_f, const int* act_b, int n_act_b) {
    dc_note_launch();
    k_pre_in<<<nblk(n_free, 128), 128, 0, s>>>(n_free, ad.type, ad.nb, w, fd.rvec, ad.node_inst, ad.mask);
    if (fd.tree) {
        const int nf = act_f ? n_act_f : fd.n_ftask, nb = act_f ? n_act_b : fd.n_btask;
        if (nf > 0) {
            cudaMemsetAsync(fd.sched, 0, sizeof(int) * (4 * (size_t)fd.S + 2), s);
            if (kt) kt->begin(DC_KT_MSOLVE);
            dc_note_launch();
            (fd.few ? k_msolve_tree<true, true> : k_msolve_tree<true, false>)<<<std::min(nf, fd.tree_grid), MT, fd.tree_smem, s>>>(fd, act_f, nf, ad.mask);
            dc_note_launch();
            (fd.few ? k_msolve_tree<false, true> : k_msolve_tree<false, false>)<<<std::min(nb, fd.tree_grid), MT, fd.tree_smem, s>>>(fd, act_b, nb, ad.mask);
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
