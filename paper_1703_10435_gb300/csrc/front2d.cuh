// Set-up of one coarse triangle for the frontal kernels (local_fp64.cu, reconstruct.cu).
#pragma once

#include "front.cuh"
#include "local_common.cuh"
#include "source_loads.cuh"

namespace mhm {

struct FrontCtx {
    double X[3][2];
    double area, flen[3], FK;
    int sgn[3], rev[3], la1[3], bad, pin, scale;   // pin: lattice point x | y << 16; scale: front_scale
};

// The pinned node, by one warp: the first node (in DOF order) of the first fine triangle of
// largest kappa, as x | y << 16; DOF 0 when kappa is uniform.  Pinned in the stiffest region
// the solution carries no large constant over it, which the face integrals would cancel in
// rounding; any node of the element can be pinned here (a window over two levels takes only
// those of its first two).  On channels of 1e3 the blocks of levels 3..7 come out
// 1e-11 to 3e-11 of their norm off the exact ones (1e-10 to 3e-10 pinned in the first two levels).
// *scale: the matrix's (front_scale).
__device__ inline int choose_pin_warp(int P, int N, const double* kap, int* scale) {
    const int lane = threadIdx.x & 31, PN = P * N;
    long long best = -1;   // (kappa > 0 orders like its bits)
    int at = 0, least = 0x7fffffff;
#pragma unroll 4
    for (int t = lane; t < N * N; t += 32) {
        const long long k = __double_as_longlong(kap[t]);
        if (k > best) best = k, at = t;
        if (k > 0) least = min(least, (int)(k >> 32));
    }
    for (int o = 16; o > 0; o >>= 1) {
        const long long k = __shfl_xor_sync(0xffffffffu, best, o);
        const int t = __shfl_xor_sync(0xffffffffu, at, o);
        if (k > best || (k == best && t < at)) best = k, at = t;
    }
    *scale = front_scale((int)(best >> 32), __reduce_min_sync(0xffffffffu, least));
    int j = 0, t = at;
    while (t >= 2 * (N - j) - 1) t -= 2 * (N - j) - 1, ++j;
    int nx[6], ny[6], px = 0, py = 0, bd = 1 << 30;
    element_nodes(P, t < N - j, t < N - j ? t : t - (N - j), j, nx, ny);
    for (int a = 0; a < (P == 1 ? 3 : 6); ++a) {
        const int d = ny[a] * (PN + 1) - ny[a] * (ny[a] - 1) / 2 + nx[a];
        if (d < bd) bd = d, px = nx[a], py = ny[a];
    }
    return px | py << 16;
}

// Geometry, pin, scaled element matrices (Ke, 72), mass of a node on k fine triangles (mass, 8) and
// source tables of element K; all threads of the block, ends with a barrier.
__device__ __forceinline__ void front_element(const DeviceMesh& dm, int64_t K, const double* kap, int P, int N,
                                              int src_kind, double src_value, double src_freq, FrontCtx& c,
                                              double* Ke, double* mass, double* tab) {
    const int tid = threadIdx.x, nthr = blockDim.x;
    if (tid < 6) c.X[tid >> 1][tid & 1] = dm.geom[6 * K + tid];
    if (tid < 3) {
        c.sgn[tid] = dm.sign[3 * K + tid];
        c.rev[tid] = dm.rev[3 * K + tid];
        c.la1[tid] = face_la1(dm, K, tid);
    }
    if (tid < 32) {
        int scale;
        const int pin = choose_pin_warp(P, N, kap, &scale);
        if (tid == 0) c.pin = pin, c.scale = scale, c.bad = 0;
    }
    __syncthreads();
    if (tid < 3) {
        const double* P0 = c.X[(tid + 1) % 3];
        const double* Q0 = c.X[(tid + 2) % 3];
        c.flen[tid] = sqrt((Q0[0] - P0[0]) * (Q0[0] - P0[0]) + (Q0[1] - P0[1]) * (Q0[1] - P0[1]));
    }
    const double area = 0.5 * fabs((c.X[1][0] - c.X[0][0]) * (c.X[2][1] - c.X[0][1]) -
                                   (c.X[2][0] - c.X[0][0]) * (c.X[1][1] - c.X[0][1]));
    if (tid == 0) c.area = area;
    if (tid < 8) mass[tid] = tid * (area / ((double)N * N) / 3.0);
    element_stiffness_pair(P, N, c.X, Ke, Ke + 36, tid, nthr, exp2_of(c.scale));
    source_tables(dm, src_kind, src_value, src_freq, P, N, c.X, tab, tid, nthr);
    __syncthreads();
}

// Source loads of all nodes to src (dof order) and their sum F_K to c.FK (a constant source:
// c.FK alone); ends with a barrier.
__device__ __forceinline__ void front_source(int kind, double value, int P, int N, const double* tab,
                                             const double* vals, FrontCtx& c, double* src) {
    const int tid = threadIdx.x, nthr = blockDim.x, PN = P * N, n = (PN + 1) * (PN + 2) / 2;
    if (kind == MHM_SRC_CONST) {
        if (tid == 0) c.FK = value * c.area;
    } else {
        int x = tid, y = 0;
        for (int u = tid; u < n; u += nthr, x += nthr) {
            while (x > PN - y) x -= PN + 1 - y, ++y;
            src[u] = source_node(kind, P, N, x, y, tab, vals);
        }
        __syncthreads();
        if (tid < 32) {
            double s = 0.0;
            for (int u = tid; u < n; u += 32) s += src[u];
            for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (tid == 0) c.FK = s;
        }
    }
    __syncthreads();
}

}  // namespace mhm
