// Loads (f, phi_w)_K of a source that is not constant (Sec. 4.2, Eq. "source_term"), node by
// node: the collapsed 4 x 4 Gauss rule on every fine triangle around the node.
//
// sin sin: the fine triangles of one orientation are translates, so with the node at
// (x, y) and a point of the rule at (x, y) + d the addition theorem splits
//   sin(k (x + dx)) sin(k (y + dy)) = sum of four products of a factor of the node and one
// of d alone.  The sums over the 16 points of w phi_a times the factors of d are four
// numbers per orientation and local node a, computed once per element; sin and cos at the
// nodes come from two tables over the lattice directions.  A load is then about 40 FP64
// operations per node (16 points x 2 sinpi x every local node of every triangle before:
// 8.8 M FP64 operations per element at P1 r = 5, more than its factorisation).
// Values: 16 multiply-adds per triangle and local node with w phi_a from a table.
//
// F_K = (f, 1)_K is the sum of the loads (the basis sums to one).
#pragma once

#include "local_common.cuh"

namespace mhm {

// Calls fn(up, i, j, a) for the fine triangles around lattice point (X, Y) (degree P),
// a the point's local index in each: up to 6 at a vertex, 2 at a P2 edge midpoint.
template <class F>
__device__ __forceinline__ void for_incident(int P, int N, int X, int Y, F&& fn) {
    auto add = [&](bool up, int i, int j, int a) {
        if (i >= 0 && j >= 0 && i + j <= N - (up ? 1 : 2)) fn(up, i, j, a);
    };
    if (P == 1 || ((X & 1) == 0 && (Y & 1) == 0)) {
        const int x = P == 1 ? X : X >> 1, y = P == 1 ? Y : Y >> 1;
        add(true, x, y, 0);
        add(true, x - 1, y, 1);
        add(true, x, y - 1, 2);
        add(false, x - 1, y - 1, 1);
        add(false, x - 1, y, 0);
        add(false, x, y - 1, 2);
        return;
    }
    const int x = X >> 1, y = Y >> 1;   // the fine square of an edge midpoint
    if (!(Y & 1)) {                     // horizontal edge
        add(true, x, y, 5);
        add(false, x, y - 1, 3);
    } else if (!(X & 1)) {              // vertical edge
        add(true, x, y, 4);
        add(false, x - 1, y, 5);
    } else {                            // diagonal edge
        add(true, x, y, 3);
        add(false, x, y, 4);
    }
}

// doubles of the tables: sin sin: 48 sums, then sin and cos of both coordinates per lattice
// column and row; values: w phi_a (6 x 16)
__host__ __device__ inline int source_table_doubles(int kind, int PN) {
    return kind == MHM_SRC_CONST ? 0 : (kind == MHM_SRC_QUAD ? 96 : 48 + 8 * (PN + 1));
}

// Fills the tables of the element with vertices X (all threads of the group, a multiple of
// 32; tid the index in it).  No barrier.
__device__ inline void source_tables(const DeviceMesh& dm, int kind, double value, double freq, int P, int N,
                                     const double X[3][2], double* tab, int tid, int nthr) {
    if (kind == MHM_SRC_CONST) return;
    const double* gx = dm.gauss_x + 3 * kMaxGauss;
    const double* gw = dm.gauss_w + 3 * kMaxGauss;
    const int nb = P == 1 ? 3 : 6, PN = P * N;
    const double e1[2] = {(X[1][0] - X[0][0]) / N, (X[1][1] - X[0][1]) / N};
    const double e2[2] = {(X[2][0] - X[0][0]) / N, (X[2][1] - X[0][1]) / N};
    const double adet = fabs(e1[0] * e2[1] - e2[0] * e1[1]);
    const double kk = freq * M_PI;
    const double amp = kind == MHM_SRC_SINSIN ? 2.0 * kk * kk * value : 1.0;
    // one point of one (orientation, local node) per thread; 16 lanes sum up
    const int items = 16 * nb * (kind == MHM_SRC_SINSIN ? 2 : 1);   // (whole warps)
    for (int it = tid; it < items; it += nthr) {
        const int k = it & 15, o = it >> 4, dn = o >= nb, a = dn ? o - nb : o;
        const double xi = gx[k >> 2], eta = gx[k & 3] * (1.0 - xi);
        const double l[3] = {1.0 - xi - eta, xi, eta};
        double phi;
        if (P == 1) phi = l[a];
        else if (a < 3) phi = l[a] * (2.0 * l[a] - 1.0);
        else phi = 4.0 * (a == 3 ? l[1] * l[2] : a == 4 ? l[2] * l[0] : l[0] * l[1]);
        const double w = gw[k >> 2] * gw[k & 3] * (1.0 - xi) * adet * amp * phi;
        if (kind == MHM_SRC_QUAD) {
            tab[it] = w;
            continue;
        }
        // offset of the point from node a in the lattice directions: vertices A, B, C at
        // (0,0), (1,0), (0,1) (up) or (1,0), (1,1), (0,1) (down)
        double u = dn ? 1.0 - l[2] : l[1], v = dn ? 1.0 - l[0] : l[2];
        const double nu[3] = {dn ? 1.0 : 0.0, 1.0, 0.0}, nv[3] = {0.0, dn ? 1.0 : 0.0, 1.0};
        if (a < 3) u -= nu[a], v -= nv[a];
        else {
            const int p = a == 3 ? 1 : a == 4 ? 2 : 0, q = a == 3 ? 2 : a == 4 ? 0 : 1;
            u -= 0.5 * (nu[p] + nu[q]);
            v -= 0.5 * (nv[p] + nv[q]);
        }
        double sx, cx, sy, cy;
        sincospi(freq * (u * e1[0] + v * e2[0]), &sx, &cx);
        sincospi(freq * (u * e1[1] + v * e2[1]), &sy, &cy);
        double m[4] = {w * cx * cy, w * cx * sy, w * sx * cy, w * sx * sy};
#pragma unroll
        for (int q = 0; q < 4; ++q)
            for (int s = 8; s > 0; s >>= 1) m[q] += __shfl_xor_sync(0xffffffffu, m[q], s);
        if (k < 4) tab[4 * o + k] = k == 0 ? m[0] : k == 1 ? m[1] : k == 2 ? m[2] : m[3];
    }
    if (kind != MHM_SRC_SINSIN) return;
    for (int it = tid; it < 4 * (PN + 1); it += nthr) {   // (column, row) x (x, y)
        const int d = it & 1, row = (it >> 1) & 1, i = it >> 2;
        const double p = row ? X[0][d] + i * (e2[d] / P) : i * (e1[d] / P);
        double s, c;
        sincospi(freq * p, &s, &c);
        double* t = tab + 48 + (row ? 4 * (PN + 1) : 0) + 4 * i + 2 * d;
        t[0] = s;
        t[1] = c;
    }
}

// (f, phi_w)_K of lattice point (x, y); vals: the element's point values (MHM_SRC_QUAD).
__device__ __forceinline__ double source_node(int kind, int P, int N, int x, int y, const double* tab,
                                              const double* vals) {
    double s = 0.0;
    if (kind == MHM_SRC_QUAD) {
        for_incident(P, N, x, y, [&](bool up, int i, int j, int a) {
            const double* f = vals + 16 * (j * (2 * N - j) + (up ? i : N - j + i));
            const double* w = tab + 16 * a;
#pragma unroll
            for (int k = 0; k < 16; ++k) s = fma(w[k], f[k], s);
        });
        return s;
    }
    const int nb = P == 1 ? 3 : 6;
    double m0 = 0.0, m1 = 0.0, m2 = 0.0, m3 = 0.0;
    for_incident(P, N, x, y, [&](bool up, int, int, int a) {
        const double* m = tab + 4 * (up ? a : nb + a);
        m0 += m[0], m1 += m[1], m2 += m[2], m3 += m[3];
    });
    const double* ti = tab + 48 + 4 * x;
    const double* tj = tab + 48 + 4 * (P * N + 1) + 4 * y;
    const double sx = fma(ti[0], tj[1], ti[1] * tj[0]), cx = fma(ti[1], tj[1], -(ti[0] * tj[0]));
    const double sy = fma(ti[2], tj[3], ti[3] * tj[2]), cy = fma(ti[3], tj[3], -(ti[2] * tj[2]));
    return fma(sx, fma(sy, m0, cy * m1), cx * fma(sy, m2, cy * m3));
}

// The integrals f phi_a of every fine triangle by the element's point values, tri[nb t + a]
// (nthr threads, whole warps; a barrier before they are read).  Four lanes read a triangle's 16
// values side by side: node by node, a thread reads six triangles of 128 bytes one after the
// other, a quarter of a sector per load
// (1702 elements P1 r = 4 with 10 columns: 0.710 -> 0.692 ms).
__device__ inline void source_triangles(int P, int N, const double* tab, const double* vals, double* tri, int tid,
                                        int nthr) {
    const int nb = P == 1 ? 3 : 6, q = tid & 3;
    for (int t0 = 0; t0 < N * N; t0 += nthr >> 2) {
        const int t = t0 + (tid >> 2);
        const bool in = t < N * N;
        double f[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) f[k] = in ? vals[16 * (size_t)t + 4 * k + q] : 0.0;
        for (int a = 0; a < nb; ++a) {
            double m = 0.0;
#pragma unroll
            for (int k = 0; k < 4; ++k) m = fma(tab[16 * a + 4 * k + q], f[k], m);
            m += __shfl_xor_sync(0xffffffffu, m, 1);
            m += __shfl_xor_sync(0xffffffffu, m, 2);
            if (in && q == (a & 3)) tri[(size_t)nb * t + a] = m;
        }
    }
}

// source_node from source_triangles
__device__ __forceinline__ double source_node_of_triangles(int P, int N, int x, int y, const double* tri) {
    const int nb = P == 1 ? 3 : 6;
    double s = 0.0;
    for_incident(P, N, x, y, [&](bool up, int i, int j, int a) { s += tri[nb * (j * (2 * N - j) + (up ? i : N - j + i)) + a]; });
    return s;
}

}  // namespace mhm
