// Elimination schedules of the local problems (front_plan.h), on the host.
#include "front_plan.h"

#include <algorithm>
#include <array>
#include <set>

namespace mhm {

std::vector<FrontStep> front_schedule(const std::vector<std::vector<int>>& adj, const std::vector<int>& order,
                                      int* slots) {
    const int n = (int)order.size();
    std::vector<int> pidx(n), need(n), ent(n), when(n), slot(n, -1), enter_at(n, -1);
    for (int p = 0; p < n; ++p) pidx[order[p]] = p;
    for (int v = 0; v < n; ++v) {   // the first step that touches v
        need[v] = pidx[v] - 1;
        for (int u : adj[v]) need[v] = std::min(need[v], pidx[u]);
        ent[v] = v;
    }
    std::sort(ent.begin(), ent.end(), [&](int a, int b) {
        return need[a] != need[b] ? need[a] < need[b] : pidx[a] < pidx[b];
    });
    for (int k = n - 1, next = 1 << 30; k >= 0; --k) when[k] = next = std::min(need[ent[k]], next - 1);
    std::vector<FrontStep> out;
    std::set<int> used;
    for (int k = 0; k < n; ++k) {
        if (when[k] >= 0) {
            enter_at[when[k]] = ent[k];
            continue;
        }
        FrontStep s;   // the front before the first elimination
        s.enter = ent[k];
        s.zs = slot[ent[k]] = (int)used.size();
        used.insert(s.zs);
        s.m = (int)used.size();
        out.push_back(s);
    }
    *slots = (int)used.size();
    for (int p = 0; p < n; ++p) {
        FrontStep s;
        s.pivot = order[p];
        s.ps = slot[s.pivot];
        s.m = *used.rbegin() + 1;
        const int v = enter_at[p];
        if (v >= 0) {   // the lowest free slot, or the pivot's own: the front stays packed
            int z = 0;
            while (z != s.ps && used.count(z)) ++z;
            s.enter = v;
            s.zs = slot[v] = z;
            s.m = std::max(s.m, z + 1);
        }
        used.erase(s.ps);
        if (v >= 0) used.insert(s.zs);
        *slots = std::max(*slots, s.m);
        out.push_back(s);
    }
    return out;
}

FrontPlan front_plan_2d(int P, int N) {
    FrontPlan plan;
    const int PN = P * N;
    auto dof = [&](int x, int y) { return y * (PN + 1) - y * (y - 1) / 2 + x; };
    const int n = (PN + 1) * (PN + 2) / 2;
    std::vector<std::array<int, 2>> xy(n);
    for (int y = 0; y <= PN; ++y)
        for (int x = 0; x <= PN - y; ++x) xy[dof(x, y)] = {x, y};
    // nodes of the fine triangles in kappa order (row by row, up then down), local order
    // A, B, C and for P2 the midpoints of BC, CA, AB
    const int nb = P == 1 ? 3 : 6;
    struct Inc { int tri, a, up; };
    std::vector<std::vector<Inc>> inc(n);
    std::vector<std::array<int, 6>> tri;
    std::vector<int> tup;
    for (int j = 0; j < N; ++j)
        for (int up = 1; up >= 0; --up)
            for (int i = 0; i < (up ? N - j : N - 1 - j); ++i) {
                const int ax = up ? i : i + 1, ay = j, bx = i + 1, by = up ? j : j + 1, cx = i, cy = j + 1;
                std::array<int, 6> d{};
                d[0] = dof(P * ax, P * ay), d[1] = dof(P * bx, P * by), d[2] = dof(P * cx, P * cy);
                if (P == 2) d[3] = dof(bx + cx, by + cy), d[4] = dof(cx + ax, cy + ay), d[5] = dof(ax + bx, ay + by);
                for (int a = 0; a < nb; ++a) inc[d[a]].push_back({(int)tri.size(), a, up});
                tri.push_back(d);
                tup.push_back(up);
            }
    std::vector<std::vector<int>> adj(n);
    for (int v = 0; v < n; ++v) {
        for (const Inc& q : inc[v])
            for (int b = 0; b < nb; ++b)
                if (tri[q.tri][b] != v) adj[v].push_back(tri[q.tri][b]);
        std::sort(adj[v].begin(), adj[v].end());
        adj[v].erase(std::unique(adj[v].begin(), adj[v].end()), adj[v].end());
    }
    // P1: lattice rows in turn.  P2: the four nodes of each fine square together, so that the
    // front holds one row of vertices and edge midpoints (35 slots at N = 16) and not two
    // whole lattice rows (65).
    std::vector<int> order(n);
    for (int v = 0; v < n; ++v) order[v] = v;
    if (P == 2)
        std::sort(order.begin(), order.end(), [&](int a, int b) {
            const std::array<int, 4> ka{xy[a][1] / 2, xy[a][0] / 2, xy[a][1] % 2, xy[a][0]};
            const std::array<int, 4> kb{xy[b][1] / 2, xy[b][0] / 2, xy[b][1] % 2, xy[b][0]};
            return ka < kb;
        });
    int slots = 0;
    const std::vector<FrontStep> steps = front_schedule(adj, order, &slots);
    if (slots > kMaxSlots || (int)tri.size() >= 0xffff) return plan;
    plan.steps = (int)steps.size();
    plan.slots = slots;
    plan.ncp = P == 1 ? 8 : 16;
    plan.cp.assign((size_t)plan.steps * plan.ncp * 2, 0);
    std::vector<int> slot(n, -1);   // where a node in the front sits
    for (int s = 0; s < plan.steps; ++s) {
        const FrontStep& st = steps[s];
        const int v = st.enter;
        int mass = 0;
        if (v >= 0)
            for (const Inc& q : inc[v]) mass += P == 1 || q.a >= 3;
        if (v >= 0) mass |= (xy[v][0] + xy[v][1] == PN) << 8 | (xy[v][0] == 0) << 9 | (xy[v][1] == 0) << 10;
        plan.ev.push_back(st.ps | st.zs << 8 | st.m << 16);
        plan.ev.push_back(v >= 0 ? xy[v][0] | xy[v][1] << 16 : 0);
        plan.ev.push_back(mass);
        plan.ev.push_back(st.pivot >= 0 ? xy[st.pivot][0] | xy[st.pivot][1] << 16 : -1);
        uint32_t* cp = &plan.cp[(size_t)s * plan.ncp * 2];
        for (int k = 0; k < plan.ncp; ++k) cp[2 * k] = kNoSlot, cp[2 * k + 1] = 0xffff0000u;
        if (v >= 0) {
            int k = 0;
            for (int u : adj[v]) {
                const int sl = u == st.pivot ? kPivotSlot : slot[u];
                if (sl < 0) continue;   // not in the front (yet)
                uint32_t e[2] = {0, 0}, t[2] = {0xffff, 0xffff};
                int c = 0;
                for (const Inc& q : inc[v])
                    for (int b = 0; b < nb; ++b)
                        if (tri[q.tri][b] == u) {
                            e[c] = 36 * !q.up + nb * q.a + b;
                            t[c++] = q.tri;
                        }
                if (k >= plan.ncp - 3) return FrontPlan{};
                cp[2 * k] = sl | e[0] << 8 | e[1] << 16;
                cp[2 * k + 1] = t[0] | t[1] << 16;
                ++k;
            }
            for (size_t q = 0; q < inc[v].size(); ++q) {   // the diagonal, two terms per entry
                uint32_t* d = cp + 2 * (plan.ncp - 3 + q / 2);
                const uint32_t e = 36 * !inc[v][q].up + (nb + 1) * inc[v][q].a, t = inc[v][q].tri;
                if (q % 2 == 0) d[0] = kDiagSlot | e << 8, d[1] = t | 0xffff0000u;
                else d[0] |= e << 16, d[1] = (d[1] & 0xffff) | t << 16;
            }
        }
        if (st.pivot >= 0) slot[st.pivot] = -1;
        if (v >= 0) slot[v] = st.zs;
    }
    return plan;
}

FrontPlan3 front_plan_3d(int n, int nb, const std::vector<int32_t>& dofs, const std::vector<int8_t>& cls,
                         const std::vector<int32_t>& xyz, int R) {
    FrontPlan3 plan;
    const int nt = (int)cls.size(), n1 = n - 1;
    std::vector<int> deg(n, 0);
    for (int s = 0; s < nt * nb; ++s) ++deg[dofs[s]];
    const int pin = (int)(std::max_element(deg.begin(), deg.end()) - deg.begin());
    plan.pin = pin;
    auto dof = [&](int v) { return v + (v >= pin); };
    auto node = [&](int d) { return d == pin ? -1 : d - (d > pin); };
    std::vector<std::vector<int>> inc(n1), adj(n1);   // slots t nb + a; neighbours
    for (int s = 0; s < nt * nb; ++s)
        if (dofs[s] != pin) inc[node(dofs[s])].push_back(s);
    int top = 0;
    for (int v = 0; v < n1; ++v) {
        for (int s : inc[v])
            for (int b = 0; b < nb; ++b) {
                const int u = node(dofs[s / nb * nb + b]);
                if (u >= 0 && u != v) adj[v].push_back(u);
            }
        std::sort(adj[v].begin(), adj[v].end());
        adj[v].erase(std::unique(adj[v].begin(), adj[v].end()), adj[v].end());
        top = std::max(top, xyz[3 * dof(v)]);
    }
    std::vector<FrontStep> steps;
    double best = 0.0;
    for (int kind = 0; kind < 3; ++kind) {
        auto key = [&](int v) -> std::array<int, 6> {
            const int A = xyz[3 * dof(v)], B = xyz[3 * dof(v) + 1], C = xyz[3 * dof(v) + 2];
            if (kind == 0) return {C, B, A, 0, 0, 0};
            if (kind == 1) return {C / 2, B / 2, A / 2, C, B, A};
            return {top - B, top - A, B - C, 0, 0, 0};
        };
        std::vector<int> order(n1);
        for (int v = 0; v < n1; ++v) order[v] = v;
        std::sort(order.begin(), order.end(), [&](int a, int b) { return key(a) < key(b); });
        int slots = 0;
        const std::vector<FrontStep> st = front_schedule(adj, order, &slots);
        double work = 0.0;
        for (const FrontStep& q : st)
            if (q.pivot >= 0) work += (double)(R + q.m) * (R + q.m);
        if (steps.empty() || work < best) steps = st, best = work, plan.slots = slots;
    }
    if (plan.slots > kMaxSlots) return FrontPlan3{};
    plan.steps = (int)steps.size();
    while (steps[plan.first_pivot].pivot < 0) ++plan.first_pivot;
    std::vector<int> slot(n1, -1);
    std::vector<uint32_t> diag(n1, 0);
    std::vector<std::vector<std::array<int, 2>>> rows(n1);
    for (const FrontStep& st : steps) {
        const int v = st.enter, first = (int)plan.ent.size();
        if (v >= 0) {
            diag[v] = (uint32_t)plan.con.size() | (uint32_t)inc[v].size() << 16;
            for (int part = 0; part < 8; ++part) {   // the diagonal: every eighth incident tetrahedron
                const size_t c0 = plan.con.size();
                for (size_t k = part; k < inc[v].size(); k += 8) {
                    const int t = inc[v][k] / nb, a = inc[v][k] % nb;
                    plan.con.push_back(t | (uint32_t)((cls[t] * nb + a) * nb + a) << 16);
                }
                plan.ent.push_back(kDiagSlot | (uint32_t)(plan.con.size() - c0) << 8 | (uint32_t)c0 << 16);
            }
            for (int u : adj[v]) {
                const int sl = u == st.pivot ? kPivotSlot : slot[u];
                if (sl < 0) continue;
                const size_t c0 = plan.con.size();
                for (int s : inc[v])
                    for (int b = 0; b < nb; ++b)
                        if (node(dofs[s / nb * nb + b]) == u) {
                            const int t = s / nb, a = s % nb;
                            plan.con.push_back(t | (uint32_t)((cls[t] * nb + a) * nb + b) << 16);
                        }
                plan.ent.push_back(sl | (uint32_t)(plan.con.size() - c0) << 8 | (uint32_t)c0 << 16);
                rows[v].push_back({u, (int)plan.val.size()});
                rows[u].push_back({v, (int)plan.val.size()});
                plan.val.push_back((uint32_t)c0 | (uint32_t)(plan.con.size() - c0) << 16);
                plan.rc.push_back(v | (uint32_t)u << 16);
            }
        }
        plan.ev.push_back(st.ps | st.zs << 8 | st.m << 16);
        plan.ev.push_back(v >= 0 ? dof(v) : -1);
        plan.ev.push_back(first);
        plan.ev.push_back(((int)plan.ent.size() - first) | (st.pivot >= 0 ? st.pivot << 16 : 0));
        if (st.pivot >= 0) slot[st.pivot] = -1;
        if (v >= 0) slot[v] = st.zs;
    }
    if (plan.con.size() > 0xffff) return FrontPlan3{};
    plan.off = (int)plan.val.size();
    for (int v = 0; v < n1; ++v) {
        rows[v].push_back({v, plan.off + v});
        std::sort(rows[v].begin(), rows[v].end());
        plan.rp.push_back((int)plan.col.size());
        for (const auto& q : rows[v]) plan.col.push_back(q[0] | (uint32_t)q[1] << 16);
        plan.val.push_back(diag[v]);
    }
    plan.rp.push_back((int)plan.col.size());
    return plan;
}

}  // namespace mhm
