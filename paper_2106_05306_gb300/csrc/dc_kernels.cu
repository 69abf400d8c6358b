// Forward-step kernels of libdc (FP64, sm_103a).
//
// One PD iteration (Sec. 3.1-3.2) is four launches:
//   local   -- per triangle: polar projection of F (stretch) and its right-hand
//              side contribution; per vertex: bending projection;
//   gather  -- per free node: b = M (v_n + h g) + h sum_i w_i A_i^T (p_i - A_i x_n)
//              + h f   (Eq. pd_velocity / pd_velocity_with_contact, expanded so
//              that the O(h^2 |L x|) terms never cancel);
//   solve_fwd / solve_bwd -- v_half = L^-T L^-1 b with the explicit inverse
//              factor, and the per-node Signorini-Coulomb update fused into the
//              backward sweep (Eq. contact_all).
// Every reduction is a fixed-order gather (no atomics), so a launch is bitwise
// repeatable and independent of what else runs on the GPU.
#include <algorithm>
#include <atomic>
#include <mutex>

#include "dc_internal.h"
#include "dc_obstacle.cuh"
#include "dc_gather.cuh"
#include "dc_polar.cuh"
#include "dc_wait.cuh"

namespace {
std::atomic<long long> g_launches{0};
}  // namespace

void dc_note_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
void dc_add_launches(long long n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
long long dc_launch_count() { return g_launches.load(std::memory_order_relaxed); }

namespace {

__device__ __forceinline__ d4 ld(const d4* p) {
    const double2* q = reinterpret_cast<const double2*>(p);
    double2 a = q[0], b = q[1];
    d4 r;
    r.x = a.x; r.y = a.y; r.z = b.x; r.w = b.y;
    return r;
}
// a load through L2 only, for data that other CTAs of the same launch write
__device__ __forceinline__ d4 ld_cg(const d4* p) {
    const double2* q = reinterpret_cast<const double2*>(p);
    double2 a = __ldcg(q), b = __ldcg(q + 1);
    d4 r;
    r.x = a.x; r.y = a.y; r.z = b.x; r.w = b.y;
    return r;
}
__device__ __forceinline__ void st(d4* p, double x, double y, double z, double w = 0.0) {
    double2* q = reinterpret_cast<double2*>(p);
    q[0] = make_double2(x, y);
    q[1] = make_double2(z, w);
}

// Signed distance and its gradient for one analytic obstacle (reading R4).
__device__ double sdf(const DevParams& P, int o, double x, double y, double z, double* n) {
    const double* q = P.oprm + 8 * o;
    const int kind = P.okind[o];
    if (kind == DC_MESH) {
        const double xx[3] = {x, y, z};
        return dc_mesh_sdf(P.mesh, (int)q[0], (int)q[1], xx, n, nullptr);
    }
    if (kind == DC_PLANE) {
        if (n) { n[0] = q[0]; n[1] = q[1]; n[2] = q[2]; }
        return q[0] * x + q[1] * y + q[2] * z - q[3];
    }
    double cx, cy, cz, r;
    if (kind == DC_SPHERE) {
        cx = q[0]; cy = q[1]; cz = q[2]; r = q[3];
    } else {
        double abx = q[3] - q[0], aby = q[4] - q[1], abz = q[5] - q[2];
        double t = ((x - q[0]) * abx + (y - q[1]) * aby + (z - q[2]) * abz) /
                   (abx * abx + aby * aby + abz * abz);
        t = fmin(fmax(t, 0.0), 1.0);
        cx = q[0] + t * abx; cy = q[1] + t * aby; cz = q[2] + t * abz; r = q[6];
    }
    double dx = x - cx, dy = y - cy, dz = z - cz;
    double d = sqrt(dx * dx + dy * dy + dz * dz);
    if (n) { n[0] = dx / d; n[1] = dy / d; n[2] = dz / d; }
    return d - r;
}

// Boundary arrays: component c of caller node e sits at ext[e * cs + c * ns]
// with (cs, ns) = (3, 1) node-major ([m][3]) or (1, m) component-major ([3][m]).
__global__ void k_permute_in(const double* __restrict__ ext, d4* __restrict__ out,
                             const int* __restrict__ int2ext, int m, int cs, long ns) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const long e = (long)int2ext[i] * cs;
    st(out + i, ext[e], ext[e + ns], ext[e + 2 * ns]);
}

__global__ void k_permute_out(const d4* __restrict__ in, double* __restrict__ ext,
                              const int* __restrict__ int2ext, int m, int cs, long ns) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const long e = (long)int2ext[i] * cs;
    d4 a = ld(in + i);
    ext[e] = a.x; ext[e + ns] = a.y; ext[e + 2 * ns] = a.z;
}

__global__ void k_zero_range(d4* v, int lo, int hi) {
    int i = lo + blockIdx.x * blockDim.x + threadIdx.x;
    if (i < hi) st(v + i, 0.0, 0.0, 0.0);
}

// Contact set, normal and bias for the step (reading R4); resets the impulse.
__global__ void k_detect(DevMesh dm, DevParams P, const d4* __restrict__ x_n, const d4* __restrict__ v_n,
                         int* __restrict__ contact, d4* __restrict__ nb, d4* __restrict__ f,
                         d4* __restrict__ ind) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= dm.m_free) return;
    d4 x = ld(x_n + i), v = ld(v_n + i);
    double px = x.x + P.h * v.x, py = x.y + P.h * v.y, pz = x.z + P.h * v.z;
    double best = 1e300;
    int bo = -1;
    const int inst = P.node_inst[i];
    for (int o = P.optr[inst]; o < P.optr[inst + 1]; ++o) {
        double ph = sdf(P, o, px, py, pz, nullptr);
        if (ph < best) { best = ph; bo = o; }
    }
    st(f + i, 0.0, 0.0, 0.0);
    if (bo >= 0 && best <= P.delta) {
        double n[3];
        double ph0 = sdf(P, bo, x.x, x.y, x.z, n);
        contact[i] = bo;
        st(nb + i, n[0], n[1], n[2], ph0 / P.h);
        st(ind + i, 1.0, 1.0, 1.0);
    } else {
        contact[i] = -1;
        st(ind + i, 0.0, 0.0, 0.0);
    }
}

// Polar factor R of a 3x2 F (reading R1): the closed form, or the fixed rule
// for a triangle collapsed onto a line (dc_polar.cuh).
__device__ __forceinline__ void polar3x2(const double F[6], double R[6]) {
    double sinv[3], itr;
    dc_polar3x2(F, R, sinv, &itr);
}

// Local step, triangles then bending vertices.  ST: a triangle on three lanes (150 FP64
// instructions become 80 a lane), SN: a vertex on three lanes; else one thread each.
// Where a vertex's rest shape is flat (s_b = 0) its projection is 0 and the velocity part
// of A_b x is not needed (but by the mass splitting).
template <bool ST, bool SN>
__global__ void k_local(DevMesh dm, DevParams P, const d4* __restrict__ x_n, const d4* __restrict__ v,
                        d4* __restrict__ c1, d4* __restrict__ c2, d4* __restrict__ bu, int n_tri_threads) {
    const int tid = blockIdx.x * blockDim.x + threadIdx.x;
    const double h = P.h;
    if (tid < n_tri_threads) {
        if (ST) {
            const Lane3 L;
            const int id = min((tid >> 5) * 10 + L.group, dm.T - 1);
            const bool on = L.on && (tid >> 5) * 10 + L.group < dm.T;
            const int c = L.c;
            const int4 tr = dm.tri[id];
            const d4 g = ld(dm.G + id);
            const double w = dm.wt[id] * h;
            const double x0 = comp(x_n, tr.x, c), x1 = comp(x_n, tr.y, c), x2 = comp(x_n, tr.z, c);
            const double v0 = comp(v, tr.x, c), v1 = comp(v, tr.y, c), v2 = comp(v, tr.z, c);
            const double e1 = x1 - x0, e2 = x2 - x0, f1 = v1 - v0, f2 = v2 - v0;
            const double Fn0 = e1 * g.x + e2 * g.z, Fn1 = e1 * g.y + e2 * g.w;
            const double F0 = Fn0 + h * (f1 * g.x + f2 * g.z), F1 = Fn1 + h * (f1 * g.y + f2 * g.w);
            double F[6], R[6], sinv[3], itr;
            L.all(F0, F);
            L.all(F1, F + 3);
            double R0, R1;
            if (dc_polar3x2(F, R, sinv, &itr)) {
                R0 = c == 0 ? R[0] : c == 1 ? R[1] : R[2];
                R1 = c == 0 ? R[3] : c == 1 ? R[4] : R[5];
            } else {
                R0 = sinv[0] * F0 + sinv[1] * F1;
                R1 = sinv[1] * F0 + sinv[2] * F1;
            }
            const double D0 = w * (R0 - (P.mass_split ? F0 : Fn0)), D1 = w * (R1 - (P.mass_split ? F1 : Fn1));
            if (on) {
                comp(c1, id, c) = D0 * g.x + D1 * g.y;
                comp(c2, id, c) = D0 * g.z + D1 * g.w;
            }
            return;
        }
        const int id = tid;
        if (id >= dm.T) return;
        int4 tr = dm.tri[id];
        d4 g = ld(dm.G + id);
        double w = dm.wt[id] * h;
        d4 x0 = ld(x_n + tr.x), x1 = ld(x_n + tr.y), x2 = ld(x_n + tr.z);
        d4 v0 = ld(v + tr.x), v1 = ld(v + tr.y), v2 = ld(v + tr.z);
        double e1[3] = {x1.x - x0.x, x1.y - x0.y, x1.z - x0.z};
        double e2[3] = {x2.x - x0.x, x2.y - x0.y, x2.z - x0.z};
        double f1[3] = {v1.x - v0.x, v1.y - v0.y, v1.z - v0.z};
        double f2[3] = {v2.x - v0.x, v2.y - v0.y, v2.z - v0.z};
        double Fn[6], F[6], R[6];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            Fn[c] = e1[c] * g.x + e2[c] * g.z;          // column 0
            Fn[3 + c] = e1[c] * g.y + e2[c] * g.w;      // column 1
            F[c] = Fn[c] + h * (f1[c] * g.x + f2[c] * g.z);
            F[3 + c] = Fn[3 + c] + h * (f1[c] * g.y + f2[c] * g.w);
        }
        polar3x2(F, R);
        // p - A x_n (Eq. pd_velocity), or p - A x^k for the mass splitting
        const double* Fr = P.mass_split ? F : Fn;
        double D[6];
#pragma unroll
        for (int k = 0; k < 6; ++k) D[k] = w * (R[k] - Fr[k]);
        st(c1 + id, D[0] * g.x + D[3] * g.y, D[1] * g.x + D[4] * g.y, D[2] * g.x + D[5] * g.y);
        st(c2 + id, D[0] * g.z + D[3] * g.w, D[1] * g.z + D[4] * g.w, D[2] * g.z + D[5] * g.w);
        return;
    }
    if (!SN) {
        const int b = tid - n_tri_threads;
        if (b >= dm.m) return;
        const double s = dm.sb[b];
        const bool moving = s > 0.0 || P.mass_split;
        double qn[3] = {0, 0, 0}, qv[3] = {0, 0, 0};
        for (int k = dm.bptr[b]; k < dm.bptr[b + 1]; ++k) {
            int j = dm.bidx[k];
            double l = dm.bval[k];
            d4 xj = ld(x_n + j);
            qn[0] += l * xj.x; qn[1] += l * xj.y; qn[2] += l * xj.z;
            if (moving) {
                d4 vj = ld(v + j);
                qv[0] += l * vj.x; qv[1] += l * vj.y; qv[2] += l * vj.z;
            }
        }
        double q[3] = {qn[0] + h * qv[0], qn[1] + h * qv[1], qn[2] + h * qv[2]};
        double p[3] = {0, 0, 0};
        if (s > 0.0) {
            double nq = sqrt(q[0] * q[0] + q[1] * q[1] + q[2] * q[2]);
            if (nq > 1e-14 * s) {
                double k = s / nq;
                p[0] = k * q[0]; p[1] = k * q[1]; p[2] = k * q[2];
            } else {
                d4 qr = ld(dm.qrest + b);
                p[0] = qr.x; p[1] = qr.y; p[2] = qr.z;
            }
        }
        double w = dm.wb[b] * h;
        const double* qr = P.mass_split ? q : qn;
        st(bu + b, w * (p[0] - qr[0]), w * (p[1] - qr[1]), w * (p[2] - qr[2]));
        return;
    }
    const Lane3 L;
    const int item = ((tid - n_tri_threads) >> 5) * 10 + L.group;
    if (((tid - n_tri_threads) >> 5) * 10 >= dm.m) return;   // (whole warps)
    const int b = min(item, dm.m - 1), c = L.c;
    const double s = dm.sb[b];
    const bool moving = s > 0.0 || P.mass_split;
    double qn = 0.0, qv = 0.0;
    list4(dm.bptr[b], dm.bptr[b + 1], dm.bidx, dm.bval, [&](int k, const int j[4], const double l[4]) {
        const int n = dm.bptr[b + 1] - k;
        double x[4], u[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            x[q] = comp(x_n, j[q], c);
            u[q] = moving ? comp(v, j[q], c) : 0.0;
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (q < n) {
                qn += l[q] * x[q];
                if (moving) qv += l[q] * u[q];
            }
    });
    const double q = qn + h * qv;
    double qa[3];
    L.all(q, qa);
    double p = 0.0;
    if (s > 0.0) {
        double nq = sqrt(qa[0] * qa[0] + qa[1] * qa[1] + qa[2] * qa[2]);
        if (nq > 1e-14 * s) {
            double k = s / nq;
            p = k * q;
        } else {
            p = comp(dm.qrest, b, c);
        }
    }
    const double w = dm.wb[b] * h;
    if (L.on && item < dm.m) comp(bu, b, c) = w * (p - (P.mass_split ? q : qn));
}

// Right-hand side.  SN: a free node on three lanes, else one thread.
template <bool SN>
__global__ void k_gather_rhs(DevMesh dm, DevParams P, const d4* __restrict__ v_n, const d4* __restrict__ c1,
                             const d4* __restrict__ c2, const d4* __restrict__ bu, const d4* __restrict__ f,
                             d4* __restrict__ b) {
    if (!SN) {
        int i = blockIdx.x * blockDim.x + threadIdx.x;
        if (i >= dm.m_free) return;
        d4 vn = ld(v_n + i);
        double mi = dm.mass[i];
        double r0 = mi * (vn.x + P.h * P.g[0]);
        double r1 = mi * (vn.y + P.h * P.g[1]);
        double r2 = mi * (vn.z + P.h * P.g[2]);
        for (int k = dm.iptr[i]; k < dm.iptr[i + 1]; ++k) {
            int e = dm.iidx[k];
            int t = e / 3, a = e - 3 * t;
            if (a == 1) {
                d4 c = ld(c1 + t);
                r0 += c.x; r1 += c.y; r2 += c.z;
            } else if (a == 2) {
                d4 c = ld(c2 + t);
                r0 += c.x; r1 += c.y; r2 += c.z;
            } else {
                d4 ca = ld(c1 + t), cb = ld(c2 + t);
                r0 -= ca.x + cb.x; r1 -= ca.y + cb.y; r2 -= ca.z + cb.z;
            }
        }
        for (int k = dm.tbptr[i]; k < dm.tbptr[i + 1]; ++k) {
            double l = dm.tbval[k];
            d4 u = ld(bu + dm.tbidx[k]);
            r0 += l * u.x; r1 += l * u.y; r2 += l * u.z;
        }
        d4 fi = ld(f + i);
        st(b + i, r0 + P.h * fi.x, r1 + P.h * fi.y, r2 + P.h * fi.z);
        return;
    }
    const int id = blockIdx.x * blockDim.x + threadIdx.x, i = id / 3, c = id - 3 * i;
    if (i >= dm.m_free) return;
    const double mi = dm.mass[i];
    double r = mi * (comp(v_n, i, c) + P.h * (c == 0 ? P.g[0] : c == 1 ? P.g[1] : P.g[2]));
    r = dc_gather_elements(dm, i, c, r, c1, c2, bu);
    comp(b, i, c) = r + P.h * comp(f, i, c);
}

// Butterfly sums of three values over a warp (the sums of three separate butterflies):
// once half of the lanes hold copies they take another value's adds, 8 FP64 instructions
// instead of 15.  Lane 0 returns the three sums.
__device__ __forceinline__ void warp_sum3(double& s0, double& s1, double& s2) {
    const int lane = threadIdx.x & 31;
    s0 += __shfl_xor_sync(0xffffffffu, s0, 16);
    s1 += __shfl_xor_sync(0xffffffffu, s1, 16);
    s2 += __shfl_xor_sync(0xffffffffu, s2, 16);
    double a = lane & 16 ? s1 : s0;
    a += __shfl_xor_sync(0xffffffffu, a, 8);
    s2 += __shfl_xor_sync(0xffffffffu, s2, 8);
    a = lane & 8 ? s2 : a;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    s0 = a;
    s1 = __shfl_sync(0xffffffffu, a, 16);
    s2 = __shfl_sync(0xffffffffu, a, 8);
}

// Forward substitution with the explicit inverse factor, y = L^-1 b.  Rows with
// more than LONG_ROW nonzeros (separator rows near the top of the elimination
// tree) get a whole CTA each; the other rows one warp each.  Both reductions
// run in a fixed order, so the result is bitwise repeatable.  CONTIG: every row's
// columns are consecutive and end at the row itself (in a postordered elimination tree a
// row of L^-1 is its node's subtree), so no index is read.
template <bool CONTIG>
__global__ void __launch_bounds__(256) k_solve_fwd(DevMesh dm, const d4* __restrict__ b, d4* __restrict__ y) {
    __shared__ double red[3][8];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool wide = (int)blockIdx.x < dm.n_long;
    const int q = ((int)blockIdx.x - dm.n_long) * 8 + warp;
    if (!wide && q >= dm.n_short) return;
    const int row = wide ? dm.long_rows[blockIdx.x] : dm.short_rows[q];
    const int lo = dm.fptr[row], hi = dm.fptr[row + 1];
    const int stride = wide ? 256 : 32;
    double s0 = 0, s1 = 0, s2 = 0;
    auto at = [&](int k) { return ld(b + (CONTIG ? row - (hi - 1 - k) : dm.fidx[k])); };
    int k = lo + (wide ? threadIdx.x : lane);
    for (; k + stride < hi; k += 2 * stride) {
        const double a0 = dm.fval[k], a1 = dm.fval[k + stride];
        const d4 u0 = at(k), u1 = at(k + stride);
        s0 += a0 * u0.x + a1 * u1.x; s1 += a0 * u0.y + a1 * u1.y; s2 += a0 * u0.z + a1 * u1.z;
    }
    if (k < hi) {
        const double a = dm.fval[k];
        const d4 u = at(k);
        s0 += a * u.x; s1 += a * u.y; s2 += a * u.z;
    }
    warp_sum3(s0, s1, s2);
    if (!wide) {
        if (lane == 0) st(y + row, s0, s1, s2);
        return;
    }
    if (lane == 0) { red[0][warp] = s0; red[1][warp] = s1; red[2][warp] = s2; }
    __syncthreads();
    if (threadIdx.x < 3) {
        double t = 0;
        for (int w = 0; w < 8; ++w) t += red[threadIdx.x][w];
        comp(y, row, threadIdx.x) = t;
    }
}

// Per-node Signorini-Coulomb solve (Eq. contact_1-3, reading R5) in world
// frame: v = vt + c f, u_N = n.v + beta, u_T = v - (n.v) n.
__device__ __forceinline__ int coulomb(double mu, double c, const double n[3], double beta,
                                       const double vt[3], double v[3], double f[3]) {
    double vn = n[0] * vt[0] + n[1] * vt[1] + n[2] * vt[2];
    double uN = vn + beta;
    if (uN >= 0.0) {                                        // take off
        v[0] = vt[0]; v[1] = vt[1]; v[2] = vt[2];
        f[0] = f[1] = f[2] = 0.0;
        return 0;
    }
    double uT[3] = {vt[0] - vn * n[0], vt[1] - vn * n[1], vt[2] - vn * n[2]};
    double nt = sqrt(uT[0] * uT[0] + uT[1] * uT[1] + uT[2] * uT[2]);
    if (nt <= mu * (-uN)) {                                 // stick
        for (int k = 0; k < 3; ++k) {
            v[k] = -beta * n[k];
            f[k] = (v[k] - vt[k]) / c;
        }
        return 1;
    }
    double fN = -uN / c;                                    // slip
    double ft = mu * fN / nt;
    for (int k = 0; k < 3; ++k) {
        f[k] = fN * n[k] - ft * uT[k];
        v[k] = vt[k] + c * f[k];
    }
    return 2;
}

// The contact update of one node (out of line: few nodes take it, and inlined it sets
// the register count of every kernel that ends in finish_row).
__device__ __noinline__ void contact_row(double s0, double s1, double s2, double mu, double c, const d4* nb, d4* f,
                                         d4* out, int* case_) {
    const d4 q = ld(nb), fo = ld(f);
    const double n[3] = {q.x, q.y, q.z};
    const double vt[3] = {s0 - c * fo.x, s1 - c * fo.y, s2 - c * fo.z};
    double v[3], fn[3];
    *case_ = coulomb(mu, c, n, q.w, vt, v, fn);
    st(f, fn[0], fn[1], fn[2]);
    st(out, v[0], v[1], v[2]);
}

// Output of one row of the backward substitution: mode 0 stores it; mode 1
// applies the node's Signorini-Coulomb update (contact nodes) and stores v; mode 2
// stores the compliance c_j = h s0.
__device__ __forceinline__ void finish_row(const DevParams& P, int row, double s0, double s1, double s2,
                                           d4* __restrict__ out, int mode, const int* __restrict__ contact,
                                           const d4* __restrict__ nb, const double* __restrict__ cc,
                                           d4* __restrict__ f, int* __restrict__ case_, double* __restrict__ c_out) {
    if (mode == 2) {
        c_out[row] = P.h * s0;
        return;
    }
    if (mode == 1 && contact[row] >= 0) {
        contact_row(s0, s1, s2, P.node_mu[row], cc[row], nb + row, f + row, out + row, case_ + row);
        return;
    }
    st(out + row, s0, s1, s2);
}

__global__ void k_solve_bwd(DevMesh dm, DevParams P, const d4* __restrict__ y, d4* __restrict__ out, int mode,
                            const int* __restrict__ contact, const d4* __restrict__ nb,
                            const double* __restrict__ cc, d4* __restrict__ f, int* __restrict__ case_,
                            double* __restrict__ c_out) {
    int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (row >= dm.m_free) return;
    double s0 = 0, s1 = 0, s2 = 0;
    const int hi = dm.kptr[row + 1];
#pragma unroll 4
    for (int k = dm.kptr[row] + (threadIdx.x & 31); k < hi; k += 32) {
        const double a = dm.kval[k];
        const d4 u = ld(y + dm.kidx[k]);
        s0 += a * u.x; s1 += a * u.y; s2 += a * u.z;
    }
    warp_sum3(s0, s1, s2);
    if ((threadIdx.x & 31) != 0) return;
    finish_row(P, row, s0, s1, s2, out, mode, contact, nb, cc, f, case_, c_out);
}

// ---- supernodal substitution (global_solver 1): leaves-first for L y = b and
// root-first for L^T x = y, three right-hand sides.  Per front, with w its gathered
// right-hand side:
//   forward   half A  y_s = L_ss^-1 w_s             half B  acc = w_U - L_Us y_s
//   backward  half A  w_s = y_s - L_Us^T x_U        half B  x_s = L_ss^-T w_s.

// Fronts of at most PS_SMALL nodes sum a row in plain k order, one lane per (row,
// column of the right-hand side); larger fronts cut the k range of a row into at most
// GV_MAXG chunks, their number a function of its length K alone, and add the chunks in
// order.  A row's result depends only on its front, never on which CTA, warp, lane or
// rows share its task.
constexpr int PS_SMALL = DC_PS_SMALL;
constexpr int PS_WARPS = DC_PS_WARPS;      // small fronts per CTA when they go in groups
constexpr int PS_LD = PS_SMALL + 1;        // shared-memory column stride of a small front (no bank conflicts)
constexpr int GV_ROWS = 128;               // rows of one pass
constexpr int GV_MAXG = 8;
__host__ __device__ constexpr int gv_groups(int K) { return K <= 8 ? 1 : (K + 7) / 8 < GV_MAXG ? (K + 7) / 8 : GV_MAXG; }

// The entries of the children's update vectors that add into position t of a front
// (pull list pp, children in order), then b_t for a pivot (bt not null): the three columns go
// to w[0], w[stride], w[2 stride].  The sums are those of a child-by-child scatter into zeroed
// storage, in the same order; the first two entries are loaded together.
__device__ __forceinline__ void ps_pull(const PSolveDev& ps, const int* __restrict__ pp, int t,
                                        const d4* __restrict__ bt, double* __restrict__ w, int stride) {
    const int e0 = pp[t], e1 = pp[t + 1];
    const int i0 = e0 < e1 ? ps.pull_idx[e0] : 0, i1 = e0 + 1 < e1 ? ps.pull_idx[e0 + 1] : 0;
    double x = 0.0, y = 0.0, z = 0.0;
    d4 b;
    if (bt) b = ld(bt);
    if (e0 < e1) {
        const d4 a = ld_cg(ps.acc + i0);
        const bool two = e0 + 1 < e1;
        d4 c;
        if (two) c = ld_cg(ps.acc + i1);
        x += a.x; y += a.y; z += a.z;
        if (two) { x += c.x; y += c.y; z += c.z; }
        for (int e = e0 + 2; e < e1; ++e) {
            const d4 d = ld_cg(ps.acc + ps.pull_idx[e]);
            x += d.x; y += d.y; z += d.z;
        }
    }
    if (bt) { x += b.x; y += b.y; z += b.z; }
    w[0] = x;
    w[stride] = y;
    w[2 * stride] = z;
}

// Rows of one pass of a CTA (its partial sums' shared memory; no bit depends on it).
__host__ __device__ constexpr int ps_pass_rows(int threads) { return threads > 128 ? GV_ROWS : GV_ROWS / 2; }

// Column-major product on one CTA with three right-hand sides: t_c,i = sum_k
// A[k * lda + i] v[c * ldv + k] for rows r_lo <= i < r_hi and k < K (TRI 1: only
// k <= i; TRI 2: only k >= i).  Work items are the (row, chunk) pairs with a nonempty k range,
// numbered chunk by chunk (the row fastest: coalesced loads), so that the empty half of a
// triangle takes no lanes.  fin(i, t0, t1, t2) stores.
template <int TRI, class Fin>
__device__ __forceinline__ void ps_rows(const double* __restrict__ A, long lda, int r_lo, int r_hi, int K,
                                        const double* __restrict__ v, int ldv, double* __restrict__ red, Fin fin) {
    const int nt = blockDim.x, tid = threadIdx.x;
    const int G = gv_groups(K), C = (K + G - 1) / G;
    const int ROWS = ps_pass_rows(nt);         // rows of a pass
    const int RS = ROWS * GV_MAXG;             // stride between the three columns' partial sums
    for (int i0 = r_lo; i0 < r_hi; i0 += ROWS) {
        const int R = min(ROWS, r_hi - i0);
        // rows [lo(g), hi(g)) of this pass have entries in chunk g
        auto lo = [&](int g) { return TRI == 1 ? min(R, max(0, g * C - i0)) : 0; };
        auto hi = [&](int g) { return TRI == 2 ? max(0, min(R, (g + 1) * C - i0)) : R; };
        int n_items = R * G;
        if (TRI != 0) {
            n_items = 0;
#pragma unroll 1
            for (int g = 0; g < G; ++g) n_items += max(0, hi(g) - lo(g));
        }
        for (int item = tid; item < n_items; item += nt) {
            int g = 0, r = item;
            if (TRI == 0) {
                g = item / R;
                r = item - g * R;
            } else {
#pragma unroll 1
                for (;; ++g) {
                    const int m = max(0, hi(g) - lo(g));
                    if (r < m) break;
                    r -= m;
                }
                r += lo(g);
            }
            int k0 = g * C, k1 = min(K, k0 + C);
            if (TRI == 1) k1 = min(k1, i0 + r + 1);
            if (TRI == 2) k0 = max(k0, i0 + r);
            const double* col = A + (long)k0 * lda + i0 + r;
            double a0 = 0.0, a1 = 0.0, a2 = 0.0;
#pragma unroll 4
            for (int k = k0; k < k1; ++k) {
                const double x = *col;
                col += lda;
                a0 += x * v[k];
                a1 += x * v[ldv + k];
                a2 += x * v[2 * ldv + k];
            }
            red[g * ROWS + r] = a0;
            red[RS + g * ROWS + r] = a1;
            red[2 * RS + g * ROWS + r] = a2;
        }
        __syncthreads();
        if (tid < R) {                         // (ROWS <= nt) the row's chunks with entries, in order
            const int i = i0 + tid, gl = TRI == 2 ? i / C : 0, gh = TRI == 1 ? i / C + 1 : G;
            double t0 = 0.0, t1 = 0.0, t2 = 0.0;
            for (int g = gl; g < gh; ++g) {
                t0 += red[g * ROWS + tid];
                t1 += red[RS + g * ROWS + tid];
                t2 += red[2 * RS + g * ROWS + tid];
            }
            fin(i, t0, t1, t2);
        }
        __syncthreads();
    }
}
// Nodes [lo, hi) of src, component-major with stride n, into dst (through L2: other CTAs of
// the launch may have written them).
__device__ __forceinline__ void ps_load(const d4* __restrict__ src, int lo, int hi, int n, double* __restrict__ dst) {
    for (int t = lo + threadIdx.x; t < hi; t += blockDim.x) {
        const d4 a = ld_cg(src + t);
        dst[t] = a.x;
        dst[n + t] = a.y;
        dst[2 * n + t] = a.z;
    }
}
__device__ __forceinline__ void ps_load_nodes(const d4* __restrict__ src, const int* __restrict__ node, int n,
                                              double* __restrict__ dst) {
    for (int t = threadIdx.x; t < n; t += blockDim.x) {
        const d4 a = ld_cg(src + node[t]);
        dst[t] = a.x;
        dst[n + t] = a.y;
        dst[2 * n + t] = a.z;
    }
}

// A task of a large front: rows [r_lo, r_hi) of one half (PS_A, PS_B), or all of it (PS_AB),
// with the vectors between the halves in shared memory; the same sums in the same order.
// wait() blocks until the inputs are there and returns false to give up.
template <class Wait>
__device__ __forceinline__ bool ps_fwd_cta(const PSolveDev& ps, int s, int phase, int r_lo, int r_hi,
                                           const d4* __restrict__ b, d4* __restrict__ y, double* __restrict__ smd,
                                           Wait wait) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int begin = ps.begin[s], ns = ps.p[s] / 3, fs = ps.f[s] / 3, nu = fs - ns;
    const int* pp = ps.pull_ptr + ps.pull_off[s];
    const bool whole = phase == PS_AB;
    if (!wait()) return false;
    double* yv = smd;                          // [3][ns]
    double* w = yv + 3 * ns;                   // [3][nw] gathered right-hand side, positions from w0
    if (phase == PS_B) {
        const int nr = r_hi - r_lo;
        ps_load(y + begin, 0, ns, ns, yv);
        for (int t = tid; t < nr; t += nt) ps_pull(ps, pp + ns + r_lo, t, nullptr, w + t, nr);
        __syncthreads();
    } else {
        const int n = whole ? fs : r_hi;
        for (int t = tid; t < n; t += nt) ps_pull(ps, pp, t, t < ns ? b + begin + t : nullptr, w + t, n);
        __syncthreads();
        ps_rows<1>(ps.xinv + ps.xoff[s], ns, whole ? 0 : r_lo, whole ? ns : r_hi, ns, w, n, w + 3 * n,
                   [&](int i, double t0, double t1, double t2) {
                       yv[i] = t0;
                       yv[ns + i] = t1;
                       yv[2 * ns + i] = t2;
                       st(y + begin + i, t0, t1, t2);
                   });
        if (!whole) return true;
    }
    // update vector: w_U - L_Us y_s
    const int r0 = whole ? 0 : r_lo, r1 = whole ? nu : r_hi, ldw = whole ? fs : r_hi - r_lo;
    const double* wu = whole ? w + ns : w - r_lo;
    d4* acc = ps.acc + ps.aoff[s];
    ps_rows<0>(ps.panel + ps.poff[s] + ns, fs, r0, r1, ns, yv, ns, w + 3 * ldw,
               [&](int i, double t0, double t1, double t2) {
                   const double* q = wu + i;
                   st(acc + i, q[0] - t0, q[ldw] - t1, q[2 * ldw] - t2);
               });
    return true;
}

// Backward; half A leaves w_s in ps.wbuf (a root has no half A, and reads y).
template <class Wait>
__device__ __forceinline__ bool ps_bwd_cta(const PSolveDev& ps, const DevParams& P, int s, int phase, int r_lo,
                                           int r_hi, const d4* __restrict__ y, d4* __restrict__ out, int mode,
                                           const int* __restrict__ contact, const d4* __restrict__ nb,
                                           const double* __restrict__ cc, d4* __restrict__ f, int* __restrict__ case_,
                                           double* __restrict__ c_out, double* __restrict__ smd, Wait wait) {
    const int begin = ps.begin[s], ns = ps.p[s] / 3, nu = ps.f[s] / 3 - ns;
    const bool whole = phase == PS_AB;
    if (!wait()) return false;
    double* w = smd;                           // [3][ns]
    double* xu = w + 3 * ns;                   // [3][nu]
    double* red = xu + 3 * nu;                 // [3][GV_MAXG * GV_ROWS]
    ps_load((phase == PS_B && nu > 0 ? ps.wbuf : y) + begin, whole ? 0 : r_lo, phase == PS_A ? r_hi : ns, ns, w);
    if (phase != PS_B) ps_load_nodes(ps.xint, ps.unode + ps.uptr[s], nu, xu);
    __syncthreads();
    if (phase != PS_B && nu > 0)
        ps_rows<0>(ps.pant + ps.toff[s], ns, whole ? 0 : r_lo, whole ? ns : r_hi, nu, xu, nu, red,
                   [&](int i, double t0, double t1, double t2) {
                       const double w0 = w[i] - t0, w1 = w[ns + i] - t1, w2 = w[2 * ns + i] - t2;
                       if (!whole) {
                           st(ps.wbuf + begin + i, w0, w1, w2);
                           return;
                       }
                       w[i] = w0;
                       w[ns + i] = w1;
                       w[2 * ns + i] = w2;
                   });
    if (phase == PS_A) return true;
    ps_rows<2>(ps.xinvt + ps.xoff[s], ns, whole ? 0 : r_lo, whole ? ns : r_hi, ns, w, ns, red,
               [&](int i, double t0, double t1, double t2) {
                   const int row = begin + i;
                   st(ps.xint + row, t0, t1, t2);
                   finish_row(P, row, t0, t1, t2, out, mode, contact, nb, cc, f, case_, c_out);
               });
    return true;
}

// Small fronts, on nt lanes (sync: their barrier): one lane
// per (row, column) pair, so that a front of ns or nu rows keeps 3 ns or 3 nu lanes
// busy; a pair's sum runs over k in ascending order.  w: [6][PS_LD].
template <class Sync>
__device__ __forceinline__ void ps_fwd_small(const PSolveDev& ps, int s, const d4* __restrict__ b,
                                             d4* __restrict__ y, double* __restrict__ w, int lane, int nt, Sync sync) {
    constexpr int L = PS_LD;
    const int begin = ps.begin[s], ns = ps.p[s] / 3, fs = ps.f[s] / 3, nu = fs - ns;
    double* yv = w + 3 * L;
    const int* pp = ps.pull_ptr + ps.pull_off[s];
    for (int t = lane; t < fs; t += nt)
        ps_pull(ps, pp, t, t < ns ? b + begin + t : nullptr, w + t, L);
    sync();
    // y_s = L_ss^-1 w_s (lower triangle)
    const double* X = ps.xinv + ps.xoff[s];
    for (int q = lane; q < 3 * ns; q += nt) {
        const int i = q / 3, col = q - 3 * i;
        const double* wc = w + col * L;
        double a = 0.0;
#pragma unroll 4
        for (int k = 0; k <= i; ++k) a += X[(long)k * ns + i] * wc[k];
        yv[col * L + i] = a;
    }
    sync();
    // update vector: w_U - L_Us y_s
    const double* Pn = ps.panel + ps.poff[s] + ns;
    double* acc = reinterpret_cast<double*>(ps.acc + ps.aoff[s]);
    for (int q = lane; q < 3 * nu; q += nt) {
        const int i = q / 3, col = q - 3 * i;
        const double* yc = yv + col * L;
        double a = 0.0;
#pragma unroll 4
        for (int k = 0; k < ns; ++k) a += Pn[(long)k * fs + i] * yc[k];
        acc[4 * i + col] = w[col * L + ns + i] - a;
    }
    for (int t = lane; t < ns; t += nt) st(y + begin + t, yv[t], yv[L + t], yv[2 * L + t]);
}

template <class Sync>
__device__ __forceinline__ void ps_bwd_small(const PSolveDev& ps, const DevParams& P, int s, const d4* __restrict__ y,
                                             d4* __restrict__ out, int mode, const int* __restrict__ contact,
                                             const d4* __restrict__ nb, const double* __restrict__ cc,
                                             d4* __restrict__ f, int* __restrict__ case_, double* __restrict__ c_out,
                                             double* __restrict__ w, int lane, int nt, Sync sync) {
    constexpr int L = PS_LD;
    const int begin = ps.begin[s], ns = ps.p[s] / 3, fs = ps.f[s] / 3, nu = fs - ns;
    double* xu = w + 3 * L;                // x_U, later x_s
    const int* un = ps.unode + ps.uptr[s];
    for (int t = lane; t < fs; t += nt) {
        const d4 a = ld_cg(t < ns ? y + begin + t : ps.xint + un[t - ns]);
        double* p = t < ns ? w + t : xu + t - ns;
        p[0] = a.x;
        p[L] = a.y;
        p[2 * L] = a.z;
    }
    sync();
    // w_s -= L_Us^T x_U (the transposed update block is ns x nu column-major)
    const double* T = ps.pant + ps.toff[s];
    for (int q = lane; q < 3 * ns; q += nt) {
        const int i = q / 3, col = q - 3 * i;
        const double* xc = xu + col * L;
        double a = 0.0;
#pragma unroll 4
        for (int k = 0; k < nu; ++k) a += T[(long)k * ns + i] * xc[k];
        w[col * L + i] -= a;
    }
    sync();
    // x_s = L_ss^-T w_s (upper triangle of the transposed inverse), into xu
    const double* XT = ps.xinvt + ps.xoff[s];
    for (int q = lane; q < 3 * ns; q += nt) {
        const int i = q / 3, col = q - 3 * i;
        const double* wc = w + col * L;
        double a = 0.0;
#pragma unroll 4
        for (int k = i; k < ns; ++k) a += XT[(long)k * ns + i] * wc[k];
        xu[col * L + i] = a;
    }
    sync();
    for (int t = lane; t < ns; t += nt) {
        const double a0 = xu[t], a1 = xu[L + t], a2 = xu[2 * L + t];
        const int row = begin + t;
        st(ps.xint + row, a0, a1, a2);
        finish_row(P, row, a0, a1, a2, out, mode, contact, nb, cc, f, case_, c_out);
    }
}

// Level kernels: CTAs [0, n_big) take one large front each, the others PS_WARPS small
// fronts each (one per warp).
__global__ void __launch_bounds__(256) k_ps_fwd(PSolveDev ps, const int* __restrict__ big, int n_big,
                                                const int* __restrict__ small, int n_small,
                                                const d4* __restrict__ b, d4* __restrict__ y) {
    extern __shared__ double smd[];
    if ((int)blockIdx.x < n_big) {
        const int s = big[blockIdx.x];
        ps_fwd_cta(ps, s, PS_AB, 0, 0, b, y, smd, []() { return true; });
        return;
    }
    const int warp = threadIdx.x >> 5;
    const int q = ((int)blockIdx.x - n_big) * PS_WARPS + warp;
    if (q < n_small)
        ps_fwd_small(ps, small[q], b, y, smd + warp * 6 * PS_LD, threadIdx.x & 31, 32, []() { __syncwarp(); });
}

__global__ void __launch_bounds__(256) k_ps_bwd(PSolveDev ps, DevParams P, const int* __restrict__ big, int n_big,
                                                const int* __restrict__ small, int n_small, const d4* __restrict__ y,
                                                d4* __restrict__ out, int mode, const int* __restrict__ contact,
                                                const d4* __restrict__ nb, const double* __restrict__ cc,
                                                d4* __restrict__ f, int* __restrict__ case_,
                                                double* __restrict__ c_out) {
    extern __shared__ double smd[];
    if ((int)blockIdx.x < n_big) {
        const int s = big[blockIdx.x];
        ps_bwd_cta(ps, P, s, PS_AB, 0, 0, y, out, mode, contact, nb, cc, f, case_, c_out, smd,
                   []() { return true; });
        return;
    }
    const int warp = threadIdx.x >> 5;
    const int q = ((int)blockIdx.x - n_big) * PS_WARPS + warp;
    if (q < n_small)
        ps_bwd_small(ps, P, small[q], y, out, mode, contact, nb, cc, f, case_, c_out, smd + warp * 6 * PS_LD,
                     threadIdx.x & 31, 32, []() { __syncwarp(); });
}

// ---- tree-scheduled sweeps: one launch for both sweeps of a global step (or one
// for each).  CTAs take tasks from a ticket counter in a topological order: a
// group of small fronts (32 to 128 threads each), one front as a whole, or some rows of one
// half of a large front.  Before a task a CTA waits until what it reads is complete:
//   forward, whole or half A   every child's forward tasks
//   backward, whole or half A  the parent's backward tasks (the parent's own wait
//                              covers the ancestors above it)
//   half B                     the front's own half-A tasks
//   backward at a root         its own forward tasks
// Each front counts its finished tasks in four counters (forward, forward half A,
// backward, backward half A) whose targets are ps.need.  A task waits only on tasks
// with smaller tickets, which CTAs already running hold, and the smallest unfinished
// ticket never waits, so a launch makes progress whatever the number of resident CTAs.
// A row's arithmetic is that of the level kernels, so the results are the same bits.
// Every wait is bounded (dc_wait.cuh): one that gives up sets the sticky fault word,
// and every CTA stops taking tasks once the word is set.
//
// Why large fronts are split by rows: an SM does one FP64 warp instruction in 16
// cycles at its measured peak (a warp alone one in 64), so the top fronts of one large cloth (400
// pivots, an 80,000-entry triangle at 200 x 200 nodes) kept one CTA busy for tens of
// microseconds each while the rest of the chip waited for them.

// The task's dependencies (one thread); false when a wait gave up.
__device__ __forceinline__ bool ps_wait(const PSolveDev& ps, bool fwd, bool fused, int s, int phase) {
    int* f = ps.sched + 1;                         // forward, forward half A
    int* b = ps.sched + 2 * ps.S + 2;              // backward, backward half A
    if (fwd) {
        if (phase == PS_B) return dc_wait_count(f + ps.S + s, ps.need[s].y, ps.fault);
        bool ok = true;
        for (int q = ps.cptr[s]; ok && q < ps.cptr[s + 1]; ++q) {
            const int c = ps.child[q];
            ok = dc_wait_count(f + c, ps.need[c].x, ps.fault);
        }
        return ok;
    }
    const int par = ps.parent[s];
    if (par < 0) return !fused || dc_wait_count(f + s, ps.need[s].x, ps.fault);
    if (phase == PS_B) return dc_wait_count(b + ps.S + s, ps.need[s].w, ps.fault);
    return dc_wait_count(b + par, ps.need[par].z, ps.fault);
}
// The counter a finished task adds to.
__device__ __forceinline__ int* ps_counter(const PSolveDev& ps, bool fwd, int s, int phase) {
    int* base = fwd ? ps.sched + 1 : ps.sched + 2 * ps.S + 2;
    const bool mid = phase == PS_A && ps.parent[s] >= 0;   // (a root's forward ends with half A)
    return base + (mid ? ps.S : 0) + s;
}

constexpr int ps_tree_threads(int kind) { return kind == PS_KIND_MANY ? 128 : 256; }
constexpr int ps_tree_ctas(int kind) { return kind == PS_KIND_NARROW ? 3 : kind == PS_KIND_WIDE ? 4 : 8; }
// kernel instance of a kind
#define PS_PICK(k, kind) ((kind) == PS_KIND_NARROW ? k<PS_KIND_NARROW> : (kind) == PS_KIND_WIDE ? k<PS_KIND_WIDE> : k<PS_KIND_MANY>)

// FWD / BWD: which sweeps this launch runs (both: the backward tasks follow the
// forward ones in ticket order).
template <bool FWD, bool BWD>
__device__ __forceinline__ void ps_run(const PSolveDev& ps, const DevParams& P, const d4* __restrict__ b,
                                       d4* __restrict__ y, d4* __restrict__ out, int mode,
                                       const int* __restrict__ contact, const d4* __restrict__ nb,
                                       const double* __restrict__ cc, d4* __restrict__ f, int* __restrict__ case_,
                                       double* __restrict__ c_out, double* __restrict__ smd) {
    __shared__ int s_item, s_ok, s_grp[PS_WARPS];
    int* ticket = FWD ? ps.sched : ps.sched + 2 * ps.S + 1;
    const int nf = FWD ? ps.n_ftask : 0, n = nf + (BWD ? ps.n_btask : 0);
    const int tid = threadIdx.x;
    for (;;) {
        if (tid == 0) s_item = dc_fault_set(ps.fault) ? n : atomicAdd(ticket, 1);
        __syncthreads();
        const int t = s_item;
        if (t >= n) return;
        const bool fwd = FWD && (!BWD || t < nf);
        const int4 task = fwd ? ps.ftask[t] : ps.btask[t - nf];
        if (task.y != PS_GROUP) {
            const int s = task.x;
            auto wait = [&]() {
                if (tid == 0) s_ok = ps_wait(ps, fwd, FWD, s, task.y);
                __syncthreads();
                return s_ok != 0;
            };
            if (task.y == PS_FRONT) {
                if (!wait()) return;
                auto sync = []() { __syncthreads(); };
                if (fwd) ps_fwd_small(ps, s, b, y, smd, tid, blockDim.x, sync);
                else ps_bwd_small(ps, P, s, y, out, mode, contact, nb, cc, f, case_, c_out, smd, tid, blockDim.x, sync);
            } else if (fwd) {
                if (!ps_fwd_cta(ps, s, task.y, task.z, task.w, b, y, smd, wait)) return;
            } else {
                if (!ps_bwd_cta(ps, P, s, task.y, task.z, task.w, y, out, mode, contact, nb, cc, f, case_, c_out, smd,
                                wait))
                    return;
            }
            __syncthreads();
            if (tid == 0) dc_add_release(ps_counter(ps, fwd, s, task.y), 1);
        } else {
            const int nt = task.w, sub = tid / nt, ln = tid - sub * nt;   // (whole warps)
            if (sub < task.z) {
                const int s = ps.tq_sn[task.x + sub];
                // barrier of a front's threads: nt >= 64 leaves at most four fronts to the CTA
                auto sync = [&]() {
                    if (nt == 32) __syncwarp();
                    else if (sub == 0) asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory");
                    else if (sub == 1) asm volatile("bar.sync 2, %0;" ::"r"(nt) : "memory");
                    else if (sub == 2) asm volatile("bar.sync 3, %0;" ::"r"(nt) : "memory");
                    else asm volatile("bar.sync 4, %0;" ::"r"(nt) : "memory");
                };
                if (ln == 0) s_grp[sub] = ps_wait(ps, fwd, FWD, s, PS_AB);
                sync();                    // the leader's acquire orders every lane's reads
                if (s_grp[sub]) {
                    double* w = smd + sub * 6 * PS_LD;
                    if (fwd) ps_fwd_small(ps, s, b, y, w, ln, nt, sync);
                    else ps_bwd_small(ps, P, s, y, out, mode, contact, nb, cc, f, case_, c_out, w, ln, nt, sync);
                    sync();
                    if (ln == 0) dc_add_release(ps_counter(ps, fwd, s, PS_AB), 1);
                }
            }
            __syncthreads();   // every warp has read s_item before it is rewritten
        }
    }
}

template <int KIND>
__global__ void __launch_bounds__(ps_tree_threads(KIND), ps_tree_ctas(KIND)) k_ps_fwd_tree(PSolveDev ps, const d4* __restrict__ b,
                                                                    d4* __restrict__ y) {
    extern __shared__ double smd[];
    const DevParams none{};
    ps_run<true, false>(ps, none, b, y, nullptr, 0, nullptr, nullptr, nullptr, nullptr, nullptr, nullptr, smd);
}

template <int KIND>
__global__ void __launch_bounds__(ps_tree_threads(KIND), ps_tree_ctas(KIND))
    k_ps_bwd_tree(PSolveDev ps, DevParams P, d4* __restrict__ y, d4* __restrict__ out, int mode,
                  const int* __restrict__ contact, const d4* __restrict__ nb, const double* __restrict__ cc,
                  d4* __restrict__ f, int* __restrict__ case_, double* __restrict__ c_out) {
    extern __shared__ double smd[];
    ps_run<false, true>(ps, P, nullptr, y, out, mode, contact, nb, cc, f, case_, c_out, smd);
}

// Both sweeps of one global step as one launch: the backward work of small trees
// runs while the forward sweeps of large ones are still in their upper levels.
template <int KIND>
__global__ void __launch_bounds__(ps_tree_threads(KIND), ps_tree_ctas(KIND))
    k_ps_sweeps_tree(PSolveDev ps, DevParams P, const d4* __restrict__ b, d4* __restrict__ y, d4* __restrict__ out,
                     int mode, const int* __restrict__ contact, const d4* __restrict__ nb,
                     const double* __restrict__ cc, d4* __restrict__ f, int* __restrict__ case_,
                     double* __restrict__ c_out) {
    extern __shared__ double smd[];
    ps_run<true, true>(ps, P, b, y, out, mode, contact, nb, cc, f, case_, c_out, smd);
}

__global__ void k_finalize(int m, double h, const d4* __restrict__ x_n, const d4* __restrict__ v,
                           d4* __restrict__ x1, unsigned long long* __restrict__ nonfinite) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    d4 a = ld(x_n + i), b = ld(v + i);
    const double x = a.x + h * b.x, y = a.y + h * b.y, z = a.z + h * b.z;
    st(x1 + i, x, y, z);
    if (!(isfinite(x) && isfinite(y) && isfinite(z) && isfinite(b.x) && isfinite(b.y) && isfinite(b.z)))
        atomicExch(nonfinite, 1ull);
}

// Instances that have taken their own number of steps keep their state.
__global__ void k_freeze(int m, int m_free, const int* __restrict__ node_inst, const int* __restrict__ inst_steps,
                         int step, const int* __restrict__ step_base, const d4* __restrict__ xin,
                         const d4* __restrict__ vin, d4* __restrict__ xout, d4* __restrict__ vout,
                         int* __restrict__ contact) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m || inst_steps[node_inst[i]] > step + (step_base ? *step_base : 0)) return;
    const d4 x = ld(xin + i), v = ld(vin + i);
    st(xout + i, x.x, x.y, x.z);
    st(vout + i, v.x, v.y, v.z);
    if (i < m_free) contact[i] = -1;
}

__global__ void k_set_int(int* p, int v) { *p = v; }

__global__ void k_pass_adjoint(int m, const int* __restrict__ node_inst, const int* __restrict__ inst_steps,
                               int step, const d4* __restrict__ gv_in, d4* __restrict__ gv_out) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m || inst_steps[node_inst[i]] > step) return;
    const d4 g = ld(gv_in + i);
    st(gv_out + i, g.x, g.y, g.z);
}

// Global step of the mass splitting (Eq. ly_et_al_govrningEq as printed):
// v_half = M^-1 b per free node, then the node's contact update.
__global__ void k_mass_solve(DevMesh dm, DevParams P, const d4* __restrict__ b, d4* __restrict__ v,
                             const int* __restrict__ contact, const d4* __restrict__ nb,
                             const double* __restrict__ cc, d4* __restrict__ f, int* __restrict__ case_) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= dm.m_free) return;
    const d4 q = ld(b + i);
    const double mi = dm.mass[i];
    finish_row(P, i, q.x / mi, q.y / mi, q.z / mi, v, 1, contact, nb, cc, f, case_, nullptr);
}

__global__ void k_count_cases(const int* __restrict__ contact, const int* __restrict__ case_, int n,
                              unsigned long long* counters) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n || contact[i] < 0) return;
    atomicAdd(counters + case_[i], 1ull);
}

inline int nblk(long n, int b) { return (int)((n + b - 1) / b); }

}  // namespace

void launch_permute_in(const double* ext, d4* out, const int* int2ext, int m, int layout, cudaStream_t s) {
    dc_note_launch();
    const bool cm = layout == DC_LAYOUT_COMPONENT_MAJOR;
    k_permute_in<<<nblk(m, 256), 256, 0, s>>>(ext, out, int2ext, m, cm ? 1 : 3, cm ? (long)m : 1L);
}
void launch_permute_out(const d4* in, double* ext, const int* int2ext, int m, int layout, cudaStream_t s) {
    dc_note_launch();
    const bool cm = layout == DC_LAYOUT_COMPONENT_MAJOR;
    k_permute_out<<<nblk(m, 256), 256, 0, s>>>(in, ext, int2ext, m, cm ? 1 : 3, cm ? (long)m : 1L);
}
void launch_zero_pins(d4* v, int m_free, int m, cudaStream_t s) {
    if (m > m_free) {
        dc_note_launch();
        k_zero_range<<<nblk(m - m_free, 256), 256, 0, s>>>(v, m_free, m);
    }
}
void launch_detect(const DevMesh& dm, const DevParams& P, const d4* x_n, const d4* v_n, int* contact,
                   d4* nb, d4* f, d4* ind, cudaStream_t s) {
    dc_note_launch();
    k_detect<<<nblk(dm.m_free, dm.bs_node), dm.bs_node, 0, s>>>(dm, P, x_n, v_n, contact, nb, f, ind);
}
void launch_local(const DevMesh& dm, const DevParams& P, const d4* x_n, const d4* v, d4* c1, d4* c2,
                  d4* bu, cudaStream_t s) {
    dc_note_launch();
    const bool st = dm.T <= DC_SPLIT_TRIS, sn = dm.m <= DC_SPLIT_NODES;
    const int nt = dc_group_threads(dm.T, st);
    auto k = st ? (sn ? k_local<true, true> : k_local<true, false>) : (sn ? k_local<false, true> : k_local<false, false>);
    k<<<nblk((long)nt + dc_group_threads(dm.m, sn), dm.bs_local), dm.bs_local, 0, s>>>(dm, P, x_n, v, c1, c2, bu, nt);
}
void launch_gather_rhs(const DevMesh& dm, const DevParams& P, const d4* v_n, const d4* c1, const d4* c2,
                       const d4* bu, const d4* f, d4* b, cudaStream_t s) {
    dc_note_launch();
    if (dm.m <= DC_SPLIT_NODES)
        k_gather_rhs<true><<<nblk(3L * dm.m_free, dm.bs_gather), dm.bs_gather, 0, s>>>(dm, P, v_n, c1, c2, bu, f, b);
    else
        k_gather_rhs<false><<<nblk(dm.m_free, dm.bs_gather), dm.bs_gather, 0, s>>>(dm, P, v_n, c1, c2, bu, f, b);
}
namespace {
size_t ps_smem(int fs) { return (6 * (size_t)fs + 3 * (size_t)GV_ROWS * GV_MAXG) * sizeof(double); }
// CTA-path fronts get 128 threads up to 96 nodes, else 256; the warp path needs 256
int ps_threads(int big_fs, int n_small) { return (n_small > 0 || big_fs > 96) ? 256 : 128; }
size_t ps_level_smem(int big_fs, int n_small) {
    const size_t a = big_fs > 0 ? ps_smem(big_fs) : 0;
    const size_t b = n_small > 0 ? (size_t)PS_WARPS * 6 * PS_LD * sizeof(double) : 0;
    return a > b ? a : b;
}
}  // namespace

// The level kernels' dynamic shared-memory limit is shared by every context of
// the process: it only ever grows.
cudaError_t psolve_configure(int max_fs) {
    static std::mutex mu;
    static size_t configured = 48 * 1024;
    std::lock_guard<std::mutex> lock(mu);
    const size_t need = ps_level_smem(max_fs, 1);
    if (need <= configured) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    for (const void* k :
         {(const void*)k_ps_fwd, (const void*)k_ps_bwd, (const void*)k_ps_fwd_tree<PS_KIND_NARROW>,
          (const void*)k_ps_fwd_tree<PS_KIND_WIDE>, (const void*)k_ps_fwd_tree<PS_KIND_MANY>,
          (const void*)k_ps_bwd_tree<PS_KIND_NARROW>, (const void*)k_ps_bwd_tree<PS_KIND_WIDE>,
          (const void*)k_ps_bwd_tree<PS_KIND_MANY>, (const void*)k_ps_sweeps_tree<PS_KIND_NARROW>,
          (const void*)k_ps_sweeps_tree<PS_KIND_WIDE>, (const void*)k_ps_sweeps_tree<PS_KIND_MANY>})
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)need);
    if (e == cudaSuccess) configured = need;
    return e;
}

// CTAs of a launch: as many as the widest stage of the tree has tasks for (`width`), beyond 128
// three quarters of that, and of the places on the chip where there are more.  A CTA without a
// ready task polls and keeps its part of an SM from other streams' kernels.  Measured against
// every CTA that fits: three 45 x 45 cloths on streams of their own (a stage has at most 48
// fronts), two steps 5.28 -> 2.44 ms each, one of them alone 6.8 -> 7.0; three batches of 64 cloths
// of 40 x 40 nodes 13.7 -> 9.8, one of them 15.3 -> 15.5.  A stage of twice the places or more
// takes them all: 256 cloths of 40 x 40 nodes, three quarters -> all, one batch 39.1 -> 36.1 ms, three
// 33.2 -> 34.6 ms each.
cudaError_t psolve_tree_grid(int max_fs, int kind, int width, int* grid, size_t* smem_out) {
    const int nt = ps_tree_threads(kind);
    const size_t smem = std::max((6 * (size_t)max_fs + 3 * (size_t)ps_pass_rows(nt) * GV_MAXG) * sizeof(double),
                                 (size_t)(nt / 32) * 6 * PS_LD * sizeof(double));
    *smem_out = smem;
    int dev = 0, sms = 0, n = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, PS_PICK(k_ps_sweeps_tree, kind), nt, smem);
    if (e != cudaSuccess) return e;
    const int fit = sms * std::max(1, n);
    const int wide = kind == PS_KIND_NARROW || width >= 2 * fit ? fit : fit / 4 * 3;
    *grid = std::max(1, std::min(wide, width <= 128 ? width : std::max(128, width / 4 * 3)));
    return cudaSuccess;
}

static void run_fwd_tree(const PSolveDev& ps, const d4* b, d4* y, cudaStream_t s) {
    const int grid = std::min(ps.tree_grid, ps.n_ftask);
    auto k = PS_PICK(k_ps_fwd_tree, ps.kind);
    k<<<grid, ps_tree_threads(ps.kind), ps.tree_smem, s>>>(ps, b, y);
}

void launch_solve_fwd(const DevMesh& dm, const d4* b, d4* y, cudaStream_t s) {
    if (dm.solver == 1) {
        const PSolveDev& ps = dm.ps;
        if (ps.tree) {
            if (ps.n_ftask == 0) return;
            cudaMemsetAsync(ps.sched, 0, sizeof(int) * (2 * (size_t)ps.S + 1), s);
            dc_note_launch();
            run_fwd_tree(ps, b, y, s);
            return;
        }
        for (int l = 0; l < ps.nlev; ++l) {
            const int nb = ps.nbig_h[l], nsm = ps.nsmall_h[l];
            if (nb + nsm <= 0) continue;
            const int* big = ps.sn + ps.lvl_ptr_h[l];
            const int grid = nb + (nsm + PS_WARPS - 1) / PS_WARPS;
            dc_note_launch();
            k_ps_fwd<<<grid, ps_threads(ps.maxbig_h[l], nsm), ps_level_smem(ps.maxbig_h[l], nsm), s>>>(
                ps, big, nb, big + nb, nsm, b, y);
        }
        return;
    }
    dc_note_launch();
    const int grid = dm.n_long + nblk(dm.n_short, 8);
    if (dm.fwd_contig)
        k_solve_fwd<true><<<grid, 256, 0, s>>>(dm, b, y);
    else
        k_solve_fwd<false><<<grid, 256, 0, s>>>(dm, b, y);
}
void launch_solve_fwd_skip(const DevMesh& dm, const d4* b, d4* y, int skip, cudaStream_t s) {
    const PSolveDev& ps = dm.ps;
    cudaMemsetAsync(ps.sched, 0, sizeof(int) * (2 * (size_t)ps.S + 1), s);
    const int ticket = skip;   // pageable source: copied before the call returns
    cudaMemcpyAsync(ps.sched, &ticket, sizeof(int), cudaMemcpyHostToDevice, s);
    dc_note_launch();
    run_fwd_tree(ps, b, y, s);
}
void launch_solve_bwd(const DevMesh& dm, const DevParams& P, const d4* y, d4* out, int mode, const int* contact,
                      const d4* nb, const double* c, d4* f, int* case_, double* c_out, cudaStream_t s) {
    if (dm.solver == 1) {
        const PSolveDev& ps = dm.ps;
        if (ps.tree) {
            if (ps.n_btask == 0) return;
            cudaMemsetAsync(ps.sched + 2 * (size_t)ps.S + 1, 0, sizeof(int) * (2 * (size_t)ps.S + 1), s);
            dc_note_launch();
            const int grid = std::min(ps.tree_grid, ps.n_btask);
            auto k = PS_PICK(k_ps_bwd_tree, ps.kind);
            k<<<grid, ps_tree_threads(ps.kind), ps.tree_smem, s>>>(ps, P, const_cast<d4*>(y), out, mode, contact, nb, c, f, case_, c_out);
            return;
        }
        for (int l = ps.nlev - 1; l >= 0; --l) {
            const int nbg = ps.nbig_h[l], nsm = ps.nsmall_h[l];
            if (nbg + nsm <= 0) continue;
            const int* big = ps.sn + ps.lvl_ptr_h[l];
            const int grid = nbg + (nsm + PS_WARPS - 1) / PS_WARPS;
            dc_note_launch();
            k_ps_bwd<<<grid, ps_threads(ps.maxbig_h[l], nsm), ps_level_smem(ps.maxbig_h[l], nsm), s>>>(
                ps, P, big, nbg, big + nbg, nsm, y, out, mode, contact, nb, c, f, case_, c_out);
        }
        return;
    }
    dc_note_launch();
    k_solve_bwd<<<nblk((long)dm.m_free * 32, 256), 256, 0, s>>>(dm, P, y, out, mode, contact, nb, c, f, case_,
                                                                c_out);
}
bool launch_solve_sweeps(const DevMesh& dm, const DevParams& P, const d4* b, d4* y, d4* out, int mode,
                         const int* contact, const d4* nb, const double* c, d4* f, int* case_, double* c_out,
                         cudaStream_t s) {
    const PSolveDev& ps = dm.ps;
    if (dm.solver != 1 || !ps.tree || !ps.fused) return false;
    if (ps.n_ftask == 0) return true;
    cudaMemsetAsync(ps.sched, 0, sizeof(int) * 2 * (2 * (size_t)ps.S + 1), s);
    dc_note_launch();
    const int grid = std::min(ps.tree_grid, ps.n_ftask + ps.n_btask);
    auto k = PS_PICK(k_ps_sweeps_tree, ps.kind);
    k<<<grid, ps_tree_threads(ps.kind), ps.tree_smem, s>>>(ps, P, b, y, out, mode, contact, nb, c, f, case_, c_out);
    return true;
}
void launch_finalize(const DevMesh& dm, const DevParams& P, const d4* x_n, const d4* v, d4* x_np1,
                     unsigned long long* nonfinite, cudaStream_t s) {
    dc_note_launch();
    k_finalize<<<nblk(dm.m, dm.bs_node), dm.bs_node, 0, s>>>(dm.m, P.h, x_n, v, x_np1, nonfinite);
}
void launch_freeze(const DevMesh& dm, const DevParams& P, const int* inst_steps, int step, const int* step_base,
                   const d4* xin, const d4* vin, d4* xout, d4* vout, int* contact, cudaStream_t s) {
    dc_note_launch();
    k_freeze<<<nblk(dm.m, 256), 256, 0, s>>>(dm.m, dm.m_free, P.node_inst, inst_steps, step, step_base, xin, vin,
                                             xout, vout, contact);
}
void launch_set_int(int* p, int v, cudaStream_t s) {
    dc_note_launch();
    k_set_int<<<1, 1, 0, s>>>(p, v);
}
void launch_pass_adjoint(const DevMesh& dm, const DevParams& P, const int* inst_steps, int step, const d4* gv_in,
                         d4* gv_out, cudaStream_t s) {
    dc_note_launch();
    k_pass_adjoint<<<nblk(dm.m, 256), 256, 0, s>>>(dm.m, P.node_inst, inst_steps, step, gv_in, gv_out);
}
void launch_mass_solve(const DevMesh& dm, const DevParams& P, const d4* b, d4* v, const int* contact, const d4* nb,
                       const double* c, d4* f, int* case_, cudaStream_t s) {
    dc_note_launch();
    k_mass_solve<<<nblk(dm.m_free, dm.bs_node), dm.bs_node, 0, s>>>(dm, P, b, v, contact, nb, c, f, case_);
}
void launch_count_cases(const int* contact, const int* case_, int m_free, unsigned long long* counters,
                        cudaStream_t s) {
    dc_note_launch();
    k_count_cases<<<nblk(m_free, 256), 256, 0, s>>>(contact, case_, m_free, counters);
}
