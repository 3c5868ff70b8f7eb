// Elimination schedules of the local problems (front_plan.h), on the host.
#include "front_plan.h"

#include <algorithm>
#include <array>

namespace mhm {

std::vector<FrontStep> front_schedule(const std::vector<int>& cliques, int nb, const std::vector<int>& order,
                                      int* slots) {
    const int n = (int)order.size();
    std::vector<int> pidx(n), need(n);
    for (int p = 0; p < n; ++p) pidx[order[p]] = p, need[order[p]] = p - 1;
    for (size_t c = 0; c < cliques.size(); c += nb) {   // the first step that touches v
        int first = n;
        for (int a = 0; a < nb; ++a)
            if (cliques[c + a] >= 0) first = std::min(first, pidx[cliques[c + a]]);
        for (int a = 0; a < nb; ++a) {
            const int v = cliques[c + a];
            if (v >= 0) need[v] = std::min(need[v], first);   // (no nodes before the clique's own first: p - 1 < p)
        }
    }
    // in the order of need, then of elimination (counted into place); then no two at one step
    std::vector<int> at(n + 2, 0), ent(n), when(n);
    for (int v = 0; v < n; ++v) ++at[need[v] + 2];
    for (int k = 1; k < n + 2; ++k) at[k] += at[k - 1];
    for (int p = 0; p < n; ++p) ent[at[need[order[p]] + 1]++] = order[p];
    for (int k = n - 1, next = 1 << 30; k >= 0; --k) when[k] = next = std::min(need[ent[k]], next - 1);
    int k = 0;
    while (k < n && when[k] < 0) ++k;   // the front before the first elimination
    std::vector<FrontStep> out;
    if (k > kMaxSlots) return out;
    out.reserve(n + k);
    std::vector<int> slot(n, -1);
    uint64_t used[(kMaxSlots + 64) / 64] = {};   // slots in use
    int top = k;                                 // the highest of them + 1
    for (int e = 0; e < k; ++e) {
        FrontStep s;
        s.enter = ent[e];
        s.zs = slot[ent[e]] = e;
        s.m = e + 1;
        used[e >> 6] |= 1ull << (e & 63);
        out.push_back(s);
    }
    *slots = k;
    for (int p = 0; p < n; ++p) {
        FrontStep s;
        s.pivot = order[p];
        s.ps = slot[s.pivot];
        s.m = top;
        used[s.ps >> 6] &= ~(1ull << (s.ps & 63));
        if (k < n && when[k] == p) {   // the lowest free slot, or the pivot's own: the front stays packed
            int w = 0;
            while (!~used[w]) ++w;
            const int z = 64 * w + __builtin_ctzll(~used[w]);
            if (z >= kMaxSlots) return {};
            s.enter = ent[k++];
            s.zs = slot[s.enter] = z;
            s.m = std::max(s.m, z + 1);
            used[w] |= 1ull << (z & 63);
        }
        top = s.m;
        while (top > 0 && !(used[(top - 1) >> 6] >> ((top - 1) & 63) & 1)) --top;
        *slots = std::max(*slots, s.m);
        out.push_back(s);
    }
    return out;
}

FrontPlan front_plan_2d(int P, int N) {
    FrontPlan plan;
    const int PN = P * N;
    if (PN + 2 * P - 1 > kMaxSlots || N * N >= 0xffff) return plan;   // slots of the orders below
    auto dof = [&](int x, int y) { return y * (PN + 1) - y * (y - 1) / 2 + x; };
    const int n = (PN + 1) * (PN + 2) / 2;
    // nodes of the fine triangles in kappa order (row by row, up then down), local order
    // A, B, C and for P2 the midpoints of BC, CA, AB; the triangles around every node
    const int nb = P == 1 ? 3 : 6;
    std::vector<int> tri((size_t)N * N * nb), inc((size_t)n * 6), ninc(n, 0);   // inc: t * 16 + 8 up + a
    int nt = 0;
    for (int j = 0; j < N; ++j)
        for (int up = 1; up >= 0; --up)
            for (int i = 0; i < (up ? N - j : N - 1 - j); ++i, ++nt) {
                const int ax = up ? i : i + 1, ay = j, bx = i + 1, by = up ? j : j + 1, cx = i, cy = j + 1;
                int* d = &tri[(size_t)nt * nb];
                d[0] = dof(P * ax, P * ay), d[1] = dof(P * bx, P * by), d[2] = dof(P * cx, P * cy);
                if (P == 2) d[3] = dof(bx + cx, by + cy), d[4] = dof(cx + ax, cy + ay), d[5] = dof(ax + bx, ay + by);
                for (int a = 0; a < nb; ++a) inc[6 * d[a] + ninc[d[a]]++] = nt * 16 + 8 * up + a;
            }
    // P1: lattice rows in turn.  P2: the four nodes of each fine square together, so that the
    // front holds one row of vertices and edge midpoints (35 slots at N = 16) and not two
    // whole lattice rows (65).
    std::vector<int> order, px(n), py(n);   // and the nodes' lattice points
    order.reserve(n);
    for (int y = 0; y <= PN; y += P)
        for (int x = 0; x <= PN - y; x += P)
            for (int v = y; v < y + P; ++v)
                for (int u = x; u < x + P && u + v <= PN; ++u) {
                    const int d = dof(u, v);
                    px[d] = u, py[d] = v;
                    order.push_back(d);
                }
    int slots = 0;
    const std::vector<FrontStep> steps = front_schedule(tri, nb, order, &slots);
    if (steps.empty()) return plan;
    plan.steps = (int)steps.size();
    plan.slots = slots;
    plan.ncp = P == 1 ? 8 : 16;
    plan.tab.assign((size_t)plan.steps * (4 + 2 * plan.ncp), 0);
    std::vector<int> slot(n, -1);   // where a node in the front sits
    for (int s = 0; s < plan.steps; ++s) {
        const FrontStep& st = steps[s];
        const int v = st.enter;
        uint32_t* ev = &plan.tab[4 * (size_t)s];
        uint32_t* cp = &plan.tab[4 * (size_t)plan.steps + (size_t)s * plan.ncp * 2];
        ev[0] = st.ps | st.zs << 8 | st.m << 16;
        ev[3] = st.pivot >= 0 ? px[st.pivot] | py[st.pivot] << 16 : -1;
        for (int k = 0; k < plan.ncp; ++k) cp[2 * k] = kNoSlot, cp[2 * k + 1] = 0xffff0000u;
        if (v >= 0) {
            int mass = 0, k = 0, node[18];   // the couplings in ascending order of the other node
            for (int q = 0; q < ninc[v]; ++q) {
                const int id = inc[6 * v + q], t = id >> 4, a = id & 7, up = id >> 3 & 1;
                mass += P == 1 || a >= 3;
                for (int b = 0; b < nb; ++b) {
                    const int u = tri[(size_t)t * nb + b], sl = u == st.pivot ? kPivotSlot : slot[u];
                    if (u == v || sl < 0) continue;   // (not in the front yet)
                    const uint32_t e = 36 * !up + nb * a + b;
                    int i = k;
                    while (i > 0 && node[i - 1] >= u) --i;
                    if (i < k && node[i] == u) {   // the second triangle of an edge
                        cp[2 * i] |= e << 16;
                        cp[2 * i + 1] = (cp[2 * i + 1] & 0xffff) | (uint32_t)t << 16;
                        continue;
                    }
                    if (k >= plan.ncp - 3) return FrontPlan{};
                    for (int c = k; c > i; --c) node[c] = node[c - 1], cp[2 * c] = cp[2 * c - 2], cp[2 * c + 1] = cp[2 * c - 1];
                    node[i] = u;
                    cp[2 * i] = sl | e << 8;
                    cp[2 * i + 1] = t | 0xffff0000u;
                    ++k;
                }
                uint32_t* d = cp + 2 * (plan.ncp - 3 + q / 2);   // the diagonal, two terms per entry
                const uint32_t e = 36 * !up + (nb + 1) * a;
                if (q % 2 == 0) d[0] = kDiagSlot | e << 8, d[1] = t | 0xffff0000u;
                else d[0] |= e << 16, d[1] = (d[1] & 0xffff) | (uint32_t)t << 16;
            }
            ev[1] = px[v] | py[v] << 16;
            ev[2] = mass | (px[v] + py[v] == PN) << 8 | (px[v] == 0) << 9 | (py[v] == 0) << 10;
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
    std::vector<int> cliques(nt * nb);
    for (int v = 0; v < n1; ++v) {
        inc[v].reserve(deg[dof(v)]);
        adj[v].reserve(32);
    }
    for (int s = 0; s < nt * nb; ++s) {
        cliques[s] = node(dofs[s]);
        if (dofs[s] != pin) inc[cliques[s]].push_back(s);
    }
    int top = 0;
    std::vector<int> seen(n1, -1);
    for (int v = 0; v < n1; ++v) {
        seen[v] = v;
        for (int s : inc[v])
            for (int b = 0; b < nb; ++b) {
                const int u = cliques[s / nb * nb + b];
                if (u < 0 || seen[u] == v) continue;
                seen[u] = v;
                adj[v].push_back(u);
            }
        std::sort(adj[v].begin(), adj[v].end());
        top = std::max(top, xyz[3 * dof(v)]);
    }
    std::vector<FrontStep> steps;
    double best = 0.0;
    for (int kind = 0; kind < 3; ++kind) {
        // the nodes by their keys, six numbers below 256 (A >= B >= C)
        std::vector<std::pair<uint64_t, int>> keys(n1);
        for (int v = 0; v < n1; ++v) {
            const int A = xyz[3 * dof(v)], B = xyz[3 * dof(v) + 1], C = xyz[3 * dof(v) + 2];
            const int q[3][6] = {{C, B, A, 0, 0, 0}, {C / 2, B / 2, A / 2, C, B, A}, {top - B, top - A, B - C, 0, 0, 0}};
            keys[v] = {0, v};
            for (int i = 0; i < 6; ++i) keys[v].first = keys[v].first << 8 | (uint64_t)q[kind][i];
        }
        std::sort(keys.begin(), keys.end());
        std::vector<int> order(n1);
        for (int k = 0; k < n1; ++k) order[k] = keys[k].second;
        int slots = 0;
        const std::vector<FrontStep> st = front_schedule(cliques, nb, order, &slots);
        if (st.empty()) continue;
        double work = 0.0;
        for (const FrontStep& q : st)
            if (q.pivot >= 0) work += (double)(R + q.m) * (R + q.m);
        if (steps.empty() || work < best) steps = st, best = work, plan.slots = slots;
    }
    if (steps.empty()) return FrontPlan3{};
    plan.steps = (int)steps.size();
    while (steps[plan.first_pivot].pivot < 0) ++plan.first_pivot;
    std::vector<int> slot(n1, -1), at(n1);
    std::vector<std::vector<uint32_t>> terms;
    std::vector<uint32_t> diag(n1, 0);
    std::vector<std::vector<std::array<int, 2>>> rows(n1);
    for (int v = 0; v < n1; ++v) rows[v].reserve(adj[v].size() + 1);
    plan.con.reserve((size_t)nt * nb * (nb + 1) / 2);
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
            // v's terms by neighbour, in the order of its incidences
            for (size_t k = 0; k < adj[v].size(); ++k) at[adj[v][k]] = (int)k;
            if (terms.size() < adj[v].size()) terms.resize(adj[v].size());
            for (auto& q : terms) q.clear();
            for (int s : inc[v]) {
                const int t = s / nb, a = s - t * nb;
                for (int b = 0; b < nb; ++b) {
                    const int u = cliques[t * nb + b];
                    if (u >= 0 && u != v) terms[at[u]].push_back(t | (uint32_t)((cls[t] * nb + a) * nb + b) << 16);
                }
            }
            for (size_t k = 0; k < adj[v].size(); ++k) {
                const int u = adj[v][k], sl = u == st.pivot ? kPivotSlot : slot[u];
                if (sl < 0) continue;
                const size_t c0 = plan.con.size();
                plan.con.insert(plan.con.end(), terms[k].begin(), terms[k].end());
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
