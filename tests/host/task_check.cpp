// Host-only check of the tree-scheduled sweeps' tasks (dc_build_ps_tasks), for k copies of an n x n
// grid cloth: every front's rows are taken once, the targets are the numbers of tasks, a task
// waits only on smaller tickets, no depth and phase has more tasks than `width`, and the small
// fronts of a wide depth share CTAs.  Arguments: pairs k n.  Prints "ok" or the first broken rule.
#include <cstdio>
#include <cstdlib>
#include <map>
#include <string>
#include <vector>

#include "dc_internal.h"

static std::string fronts(int n, HostFronts& fr) {
    std::vector<double> pos;
    std::vector<int> tri;
    for (int v = 0; v < n * n; ++v) {
        const double x[3] = {v % n / double(n - 1), 0.5, v / n / double(n - 1)};
        pos.insert(pos.end(), x, x + 3);
    }
    for (int j = 0; j + 1 < n; ++j)
        for (int i = 0; i + 1 < n; ++i) {
            const int a = j * n + i;
            tri.insert(tri.end(), {a, a + 1, a + n + 1, a, a + n + 1, a + n});
        }
    HostMesh hm;
    std::string e = dc_build_mesh(hm, n * n, pos.data(), (int)tri.size() / 3, tri.data(), 0, nullptr);
    if (!e.empty()) return e;
    dc_params p{};
    p.k_stretch = 1e3;
    p.k_bend = 1e-3;
    p.h = 1.0 / 120.0;
    std::vector<double> mass(hm.m);
    for (int i = 0; i < hm.m; ++i) mass[i] = 0.1 * hm.abar[i];
    HostFactor hf;
    dc_build_factor(hm, p, mass, hf, e, false);
    return e.empty() ? dc_build_fronts(hm, hf, fr) : e;
}

// k copies side by side: what the task lists are built from
static HostFronts copies(const HostFronts& fr, int k) {
    HostFronts o;
    o.S = k * fr.S;
    o.cptr.assign(1, 0);
    for (int c = 0; c < k; ++c)
        for (int s = 0; s < fr.S; ++s) {
            o.f.push_back(fr.f[s]);
            o.p.push_back(fr.p[s]);
            o.parent.push_back(fr.parent[s] < 0 ? -1 : fr.parent[s] + c * fr.S);
            for (int q = fr.cptr[s]; q < fr.cptr[s + 1]; ++q) o.child.push_back(fr.child[q] + c * fr.S);
            o.cptr.push_back((int)o.child.size());
        }
    return o;
}

static const char* check(const HostFronts& fr) {
    std::vector<int> tq_ptr, tq_sn;
    std::vector<int4> task[2], need;
    int kind = 0, width = 0;
    dc_build_tree_items(fr, tq_ptr, tq_sn);
    dc_build_ps_tasks(fr, tq_ptr, tq_sn, task[0], task[1], need, kind, width);
    std::vector<int> depth(fr.S, 0);
    for (int s = fr.S - 1; s >= 0; --s) depth[s] = fr.parent[s] < 0 ? 0 : depth[fr.parent[s]] + 1;
    const int threads = kind == PS_KIND_MANY ? 128 : 256;
    int widest = 0;
    for (int way = 0; way < 2; ++way) {                       // forward, backward
        std::vector<int> a(fr.S, 0), b(fr.S, 0), na(fr.S, 0), nb(fr.S, 0), done(fr.S, 0);
        std::vector<int> ends(fr.S, -1), half(fr.S, -1);      // last ticket of each phase
        std::map<std::pair<int, int>, int> stage;             // tasks of a depth and phase
        std::map<int, int> small_tasks, small_fronts;
        for (int t = 0; t < (int)task[way].size(); ++t) {
            const int4 q = task[way][t];
            const bool group = q.y == PS_GROUP;
            const int n = group ? q.z : 1;
            if (group && (q.w < 32 || q.w * n > threads)) return "threads of a group";
            for (int k = 0; k < n; ++k) {
                const int s = group ? tq_sn[q.x + k] : q.x, ns = fr.p[s] / 3, nu = fr.f[s] / 3 - ns;
                const bool large = fr.f[s] / 3 > DC_PS_SMALL, root = fr.parent[s] < 0;
                if (large != (q.y != PS_GROUP && q.y != PS_FRONT)) return "kind of task";
                if (k && depth[s] != depth[tq_sn[q.x]]) return "one depth per group";
                if (!large) small_fronts[depth[s]]++, small_tasks[depth[s]] += k == 0;
                if (k == 0) stage[{depth[s], q.y == PS_B && !root}]++;
                // what it waits for has smaller tickets only
                if (q.y == PS_B && !root) {
                    if (a[s] != ns) return "half A before half B";
                } else if (way == 0) {
                    for (int c = fr.cptr[s]; c < fr.cptr[s + 1]; ++c)
                        if (done[fr.child[c]] != need[fr.child[c]].x) return "children before parents";
                } else if (!root && done[fr.parent[s]] != need[fr.parent[s]].z) {
                    return "parents before children";
                }
                const int rows_b = way == 0 ? nu : ns;
                if (q.y == PS_A) {
                    if (a[s] != q.z || q.w <= q.z || q.w > ns) return "rows of half A";
                    a[s] = q.w;
                    ++na[s];
                    if (way == 0 && root) ++done[s];
                } else if (q.y == PS_B) {
                    if (b[s] != q.z || q.w <= q.z || q.w > rows_b) return "rows of half B";
                    b[s] = q.w;
                    ++nb[s];
                    ++done[s];
                } else {
                    if (done[s]) return "a whole front twice";
                    a[s] = ns;
                    b[s] = rows_b;
                    ++done[s];
                }
            }
        }
        for (int s = 0; s < fr.S; ++s) {
            const int ns = fr.p[s] / 3, nu = fr.f[s] / 3 - ns;
            if (a[s] != ns && !(way == 1 && nu == 0)) return "every row of half A";
            if (b[s] != (way == 0 ? nu : ns)) return "every row of half B";
            if (done[s] != (way == 0 ? need[s].x : need[s].z)) return "targets";
            if (na[s] && nu > 0 && na[s] != (way == 0 ? need[s].y : need[s].w)) return "half-A targets";
        }
        for (const auto& e : stage) widest = std::max(widest, e.second);
        for (const auto& e : small_tasks) {
            const int n = small_fronts[e.first], least = (n + threads / 32 - 1) / (threads / 32);
            if (e.second > 256 && e.second > least) return "a wide depth's small fronts share CTAs";
            if (n <= 96 && e.second != n) return "few small fronts take a CTA each";
        }
    }
    return widest == width ? "" : "width";
}

int main(int argc, char** argv) {
    for (int i = 1; i + 1 < argc; i += 2) {
        HostFronts fr;
        const std::string e = fronts(atoi(argv[i + 1]), fr);
        const char* bad = e.empty() ? check(copies(fr, atoi(argv[i]))) : e.c_str();
        if (*bad) {
            printf("%s cloths of %s: %s\n", argv[i], argv[i + 1], bad);
            return 1;
        }
    }
    puts("ok");
    return 0;
}
