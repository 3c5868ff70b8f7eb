// Three-dimensional local problems (the paper's experiment, Sec. 5) on the GPU:
// solveLocalProblem for every coarse tetrahedron (Sec. 3, Eqs. "etaf", "etai") in FP64
// or mixed precision, and the gather of the skeleton system (Eq. "mat_global").
// Conventions in mhm3d.h.
//
// No atomics anywhere, every sum in a fixed order: repeated calls are bit-identical.
//   k_local3d (FP64): frontal elimination of the pinned matrix bordered by the projected loads
//     g - (1^T g / |K|) m (front.cuh): class matrices of the six congruence classes of
//     sub-tetrahedra (closed forms, per element type), couplings gathered per DOF, multiplier
//     loads from the face table (a fine face triangle puts a third of its area on each load
//     node); the face integrals are what the elimination leaves in the border;
//   k_local3d_mixed: an FP32 factor of the diagonally scaled matrix, FP64 refinement against
//     the matrix-free residual, and the corrected bilinear form (see the kernel).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>

#include "front.cuh"
#include "mhm3d_internal.h"

namespace mhm3 {

namespace {

struct Local3DArgs {
    const double* geom;
    const int8_t* signs;
    const int8_t* perm;
    const int8_t* sub_cls;
    const int8_t* sub_base;
    const int32_t* inc_off;   // per local DOF, its slots t nb + a (ascending)
    const int32_t* inc_ent;
    const int32_t* ftab_off;
    const int16_t* ftab_node;
    const int8_t* ftab_cnt;
    const double* kappa;
    double src_value, src_freq;
    int64_t K0, K1;
    int N, n, nb, nsub, m, NI, R;
    double* AK;
    double* EK;
    double* BK;
    double* FK;
    int32_t* status;
    int32_t* iters;       // may be NULL
    int only_failed;      // FP64 kernel: solve only the elements whose status is nonzero (iters -1)
    int it_max;           // mixed kernel: refinement passes
    double tol;           // mixed kernel: scaled residual target per column
    // frontal elimination (front.cuh): step tables; per type of element (K mod 24: translates)
    // the six class matrices and vol, area_a / (3 N^2); mass of a DOF on a unit volume; fine
    // face triangles of subface q that load DOF w, per local face and permutation (x n x m)
    const int4* ev;
    const uint32_t *ent, *con;
    int steps, slots;
    const double *cls24, *geo24, *mass1;
    const uint8_t* fcnt;
    int source;           // 1: sin sin sin, by Source3; 0: constant
    // mixed kernel: values and rows of the matrix (FrontPlan3)
    const uint32_t *val, *rc, *col;
    const int32_t* rp;
    int first, off, pin;
};

constexpr int kPath[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};

// Source tables (sin sin sin by the collapsed Gauss rule).  With a sub-tetrahedron's first vertex at
// x and a point of the rule at x + d, the addition theorem splits f(x + d) into eight products of
// sines and cosines of x and of d,
//   load of local DOF a = sum_b prod_c (b_c ? cos : sin)(k x_c) M[a][b],
//   M[a][b] = sum over the points of w phi_a prod_c (b_c ? sin : cos)(k d_c),
// so an element needs 3 sincos per sub-tetrahedron where the rule has 3 sines at each of its 64
// points.  The sub-tetrahedra of a class are translates, and the 24 types of element (K mod 24) are
// images of type 0 under permutations and reflections of the axes, so the M of the six classes
// of type 0 serve all: 480 values (P2) that the host forms for every call (source_tables) and the
// kernels take as a parameter: the call allocates nothing and has one launch.  (1536 elements of P2
// r = 1, m = 4, whole call: 0.285 ms with tables of all types formed by a kernel in memory from the
// stream-ordered pool, 0.465 formed by every block for itself, 0.197 as a parameter.)
struct Source3 {
    double M[6 * 10 * 8];    // per class, local DOF, b
    uint8_t axis[24][4];     // per type: axis that type 0's x, y, z goes to, + 4 if reflected
};

__device__ __forceinline__ double warp_sum(double v) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Source loads of element K per DOF (src, n) through the loads of every sub-tetrahedron (PL,
// nsub x nb), summed per DOF in the fixed order of its incidence list.  All threads; ends
// with a barrier.
__device__ __forceinline__ void source_loads3(const Local3DArgs& g, const Source3& q, int64_t K, double* PL, double* src) {
    const int nb = g.nb, N = g.N;
    const double* V = g.geom + 12 * K;
    const uint8_t* axis = q.axis[K % 24];
    for (int t = threadIdx.x; t < g.nsub; t += blockDim.x) {
        double s[3], c[3], T[8];   // along type 0's axes
        for (int y = 0; y < 3; ++y) {
            const int x = axis[y] & 3;
            const double p = V[x] + ((V[3 + x] - V[x]) * g.sub_base[3 * t] + (V[6 + x] - V[3 + x]) * g.sub_base[3 * t + 1] +
                                     (V[9 + x] - V[6 + x]) * g.sub_base[3 * t + 2]) / N;
            sincospi(g.src_freq * p, &s[y], &c[y]);
            if (axis[y] & 4) c[y] = -c[y];   // (the cosine goes with the sine of d)
        }
#pragma unroll
        for (int b = 0; b < 8; ++b) T[b] = (b & 1 ? c[0] : s[0]) * (b & 2 ? c[1] : s[1]) * (b & 4 ? c[2] : s[2]);
        const int m0 = g.sub_cls[t] * 8 * nb;
        for (int a = 0; a < nb; ++a) {
            double v = 0.0;
#pragma unroll
            for (int b = 0; b < 8; ++b) v = fma(T[b], q.M[m0 + 8 * a + b], v);
            PL[t * nb + a] = v;
        }
    }
    __syncthreads();
    for (int w = threadIdx.x; w < g.n; w += blockDim.x) {
        double v = 0.0;
        for (int e = g.inc_off[w]; e < g.inc_off[w + 1]; ++e) v += PL[g.inc_ent[e]];
        src[w] = v;
    }
    __syncthreads();
}

// Entering rows of the frontal elimination (front_plan_3d's tables): couplings from kappa
// and the class matrices S, loads -s (psi_j, phi_w) - (1^T g / |K|) m_w from the face counts.
template <int VEC>
struct FrontRows3D {
    static constexpr int C = VEC / 32;
    const Local3DArgs& g;
    const double *kap, *S, *src;   // src NULL: constant source
    double vol;
    double cp[C], cf[C];           // projection coefficient x |K|; -s area / (3 N^2)
    int base[C];                   // first face count of the column, -1: no face
    __device__ __forceinline__ void prep(int, const int4& v, double* nb, double* wnew) {
        const int lane = threadIdx.x & 31, zs = (v.x >> 8) & 255, R = g.R;
        if (zs == mhm::kNoSlot) return;
        const double mt = g.mass1[v.y];
        mhm::static_for<C>([&](auto k) {
            const int q = lane + 32 * k;
            double x = 0.0;
            if (q < R) {
                x = -cp[k] * mt;
                if (q == g.NI) {
                    x = src ? x + src[v.y] : fma(g.src_value * vol, mt, x);
                } else {
                    const int cnt = g.fcnt[base[k] + v.y * g.m];
                    // (cnt as a double without a conversion: 2^52 + cnt - 2^52)
                    if (cnt) x = fma(cf[k], __hiloint2double(0x43300000, cnt) - 4503599627370496.0, x);
                }
            }
            nb[q] = x;
        });
        if (lane == 0) *wnew = 0.0;
        __syncwarp();
        const int count = v.w & 0xffff;
        for (int q = lane; q < ((count + 31) & ~31); q += 32) {
            const uint32_t en = q < count ? g.ent[v.z + q] : mhm::kNoSlot;
            const int sl = en & 255, terms = (en >> 8) & 255;
            const uint32_t* con = g.con + (en >> 16);
            double x = 0.0;
            for (int i = 0; i < terms; ++i) x = fma(kap[con[i] & 0xffff], S[con[i] >> 16], x);
            if (q < 32) {   // the first eight: the diagonal
                double d = sl == mhm::kDiagSlot ? x : 0.0;
                d += __shfl_xor_sync(0xffffffffu, d, 1);
                d += __shfl_xor_sync(0xffffffffu, d, 2);
                d += __shfl_xor_sync(0xffffffffu, d, 4);
                if (lane == 0) nb[R + zs] = d;
            }
            if (sl < mhm::kDiagSlot) nb[R + sl] = x;
            else if (sl == mhm::kPivotSlot) *wnew = x;
        }
    }
};

struct Front3Smem {
    int S, kap, src, PL, total;   // doubles
};
__host__ __device__ inline Front3Smem front3_smem(int vec, int n, int nb, int nsub, bool source) {
    Front3Smem l;
    int o = (int)mhm::front_shared_values(vec);
    l.S = o, o += 6 * nb * nb;
    l.kap = o, o += nsub;
    l.src = o, o += source ? n : 0;
    l.PL = o, o += source ? nsub * nb : 0;
    l.total = o;
    return l;
}

// FP64: one block per coarse tetrahedron at a time eliminates the pinned matrix bordered by
// its R loads from a front of at most 41 slots (P2, r = 2: 165 DOFs) held in registers
// (front.cuh); what is left of the border are the face integrals.  Bound by the FP64 pipe
// (84 % busy at m = 4, 12.4 k warp instructions per element; 81 % at m = 16).  12288 elements,
// m = 4, sin sin sin: 9.4 ms (79.5 ms with the dense matrix in shared memory, one element per SM);
// 1536 elements, m = 16: 4.0 ms (14.6 ms).
template <class T, int MINB>
__global__ void __launch_bounds__(T::threads, MINB) k_local3d(const __grid_constant__ Local3DArgs g,
                                                             const __grid_constant__ Source3 source) {
    extern __shared__ double sm[];
    __shared__ int bad, scales;
    __shared__ double FKs;
    const int tid = threadIdx.x, nthr = blockDim.x, n = g.n, nb = g.nb, NI = g.NI, R = g.R, m = g.m;
    const Front3Smem L = front3_smem(T::vec, n, nb, g.nsub, g.source != 0);
    const mhm::FrontShared<double> sh = mhm::front_shared(sm, T::vec);
    double *S = sm + L.S, *kap = sm + L.kap, *src = sm + L.src;
    for (int64_t K = g.K0 + blockIdx.x; K < g.K1; K += gridDim.x) {
        if (g.only_failed && g.status[K] == MHM_OK) continue;   // (the whole block)
        const double* geo = g.geo24 + 8 * (K % 24);
        const double vol = geo[0];
        for (int t = tid; t < 6 * nb * nb; t += nthr) S[t] = g.cls24[(size_t)(K % 24) * 6 * nb * nb + t];
        for (int t = tid; t < g.nsub; t += nthr) kap[t] = g.kappa[K * (int64_t)g.nsub + t];
        if (tid == 0) bad = 0;
        if (g.source) source_loads3(g, source, K, sm + L.PL, src);
        if (tid < 32) {
            double f = 0.0;
            if (g.source) {
                for (int w = tid; w < n; w += 32) f += src[w];
                f = warp_sum(f);
            } else {
                f = g.src_value * vol;
            }
            int most = -1, least = 0x7fffffff;
            for (int t = tid; t < g.nsub; t += 32) {
                const long long k = __double_as_longlong(g.kappa[K * (int64_t)g.nsub + t]);
                if (k > 0) most = max(most, (int)(k >> 32)), least = min(least, (int)(k >> 32));
            }
            most = __reduce_max_sync(0xffffffffu, most);
            least = __reduce_min_sync(0xffffffffu, least);
            if (tid == 0) FKs = f, scales = mhm::front_scale(most, least);
        }
        __syncthreads();
        const int scale = scales;
        if (scale != 0) {
            for (int t = tid; t < 6 * nb * nb; t += nthr) S[t] *= mhm::exp2_of(scale);
            __syncthreads();
        }
        // (psi_j, 1)_{dK} of column j: s |subface|; the projection is its negative over |K|
        auto moment = [&](int j) {
            const int a = j / m, q = j % m, b0 = (a * 6 + g.perm[4 * K + a]) * (m + 1) + q;
            int c = 0;
            for (int e = g.ftab_off[b0]; e < g.ftab_off[b0 + 1]; ++e) c += g.ftab_cnt[e];
            return (double)g.signs[4 * K + a] * geo[1 + a] * c;
        };
        FrontRows3D<T::vec> rows{g, kap, S, g.source ? src : nullptr, vol};
        mhm::static_for<T::vec / 32>([&](auto k) {
            const int q = (tid & 31) + 32 * k;
            rows.cp[k] = rows.cf[k] = 0.0;
            rows.base[k] = 0;
            if (q < NI) {
                const int a = q / m;
                rows.cp[k] = -moment(q);
                rows.cf[k] = -(double)g.signs[4 * K + a] * geo[1 + a];
                rows.base[k] = (a * 6 + g.perm[4 * K + a]) * n * m + q % m;
            } else if (q == NI) {
                rows.cp[k] = FKs;
            }
        });
        double A[T::NT];
        mhm::front_eliminate<T>(rows, g.ev, g.steps, R, sh, A, &bad, (double*)nullptr, 0);
        double* AK = g.AK + K * (int64_t)NI * NI;
        mhm::front_result<T>(R, A, [&](int i, int j, double v) {
            if (scale != 0) v *= mhm::exp2_of(scale);
            if (i < NI) {
                AK[i * NI + j] = v;
                AK[j * NI + i] = v;
            } else if (j < NI) {
                g.EK[K * NI + j] = -v;
            }
        });
        for (int j = tid; j < NI; j += nthr) g.BK[K * NI + j] = moment(j);
        if (tid == 0) {
            g.FK[K] = FKs;
            g.status[K] = bad ? MHM_ERR_INVALID_ARG : MHM_OK;
            if (g.iters) g.iters[K] = g.only_failed ? -1 : 1;
        }
        __syncthreads();
    }
}

// The frontal kernel of a bordered matrix of M rows.
struct Front3Kernel {
    void (*kern)(const Local3DArgs, const Source3) = nullptr;
    int threads = 0, vec = 0;
};
template <class T, int MINB>
void front3_try(int M, Front3Kernel* k) {
    if (k->kern || M > T::rows) return;
    k->kern = k_local3d<T, MINB>;
    k->threads = T::threads;
    k->vec = T::vec;
}
// few: no more elements than three per SM: 4 warps (and one for the rows) share an element, which
// shortens a step where a single warp's latency is what counts (24 elements, m = 4: 0.86 -> 0.48
// ms; 0.37 without the source tables' own kernel); the same results bit for bit.
Front3Kernel front3_kernel(int M, bool few) {
    Front3Kernel k;
    if (few) {
        front3_try<mhm::FrontTiles<4, 1, 2>, 4>(M, &k);
        front3_try<mhm::FrontTiles<4, 1, 4>, 4>(M, &k);
    }
    front3_try<mhm::FrontTiles<1, 1, 8>, 12>(M, &k);
    front3_try<mhm::FrontTiles<1, 1, 12>, 12>(M, &k);
    front3_try<mhm::FrontTiles<1, 1, 15>, 8>(M, &k);
    front3_try<mhm::FrontTiles<4, 1, 7>, 2>(M, &k);
    return k;
}

// Entering rows of the FP32 factor: the scaled off-diagonal values, counted off in the order
// of the entries (each entering node has 8 diagonal entries in front).
struct FrontRowsScaled {
    const Local3DArgs& g;
    const float *off, *diag;
    int vec, entered = 0;
    __device__ __forceinline__ void prep(int, const int4& v, float* nb, float* wnew) {
        const int lane = threadIdx.x & 31, zs = (v.x >> 8) & 255;
        if (zs == mhm::kNoSlot) return;
        ++entered;
        for (int q = lane; q < vec; q += 32) nb[q] = 0.0f;
        if (lane == 0) *wnew = 0.0f;
        __syncwarp();
        for (int q = 8 + lane; q < (v.w & 0xffff); q += 32) {
            const int sl = g.ent[v.z + q] & 255;
            const float x = off[v.z + q - 8 * entered];
            if (sl == mhm::kPivotSlot) *wnew = x;
            else nb[sl] = x;
        }
        if (lane == 0) nb[zs] = diag[v.y - (v.y > g.pin)];
    }
};

using FrontTilesMixed = mhm::FrontTiles<1, 1, 11>;   // fronts of at most 44 slots
constexpr int kMaxMixedR = 17;                       // three columns for each of 8 warps (m <= 4)

struct Mixed3Smem {   // offsets in doubles
    int S, kap, A, Z, Rr, W, Lc, inv, sc, src, cp, cf, gn, red, mz, front, total;
};
__host__ __device__ inline Mixed3Smem mixed3_smem(int n, int R, int nb, int nsub, int off, int slots) {
    const int n1 = n - 1, pl = nsub * nb;
    Mixed3Smem l;
    int o = 0;
    l.S = o, o += 6 * nb * nb;
    l.kap = o, o += nsub;
    l.A = o, o += off + n1;                                   // values of the pinned matrix
    l.Z = o, o += n1 * R;
    l.Rr = o, o += n1 * R > pl ? n1 * R : pl;                 // residuals (before: loads per sub-tetrahedron)
    l.W = o, o += ((n1 * R > off + n1 ? n1 * R : off + n1) + 1) / 2 + R * R;   // FP32 solves (before: scaled values); outputs
    l.Lc = o, o += (n1 * slots + 1) / 2;                      // FP32 pivot columns
    l.inv = o, o += (n1 + 1) / 2;
    l.sc = o, o += n1;
    l.src = o, o += n;
    l.cp = o, o += R;
    l.cf = o, o += R;
    l.gn = o, o += R;
    l.red = o, o += R;
    l.mz = o, o += R;
    l.front = o, o += ((int)mhm::front_shared_values(FrontTilesMixed::vec) + 1) / 2;
    l.total = o;
    return l;
}

// Mixed precision (Sec. 3: the local matrix is factored once and each further solve is
// only products with the factor): the pinned matrix, scaled by its diagonal, is factored
// in FP32 by the frontal elimination (one warp, the pivot columns kept in shared memory);
// the N_I + 1 solutions are refined in FP64 against the FP64 residual r = g~ - A z (rows of
// the assembled matrix), each pass one FP32 forward and backward sweep over the pivots (a warp
// takes up to three columns, a lane the front's slots), until every column's scaled
// residual |S r| <= tol |S g~| or it_max passes.  The face integrals use the corrected
// bilinear form
//   (s psi_j, eta_i)_{dK} = -(g~_j . z_i + z_j . r_i),
// whose error is the product of the two solution errors in the energy norm (second order),
// averaged with its transpose.  An element whose FP32 factor breaks down or that does not
// converge gets MHM_ERR_NOT_CONVERGED (the host then re-solves it in FP64 unless asked not to).
//
// Bound by issued instructions and their latencies: 0.74 M warp instructions per element (two
// passes), most of them the FP32 sweeps, 11 k of them FP64 (20 % of that pipe on 192 elements); two elements per SM
// (110 KB of shared memory each) hide one another's chains.  12288 elements, m = 4: 24.6 ms
// (91.3 ms with a dense packed factor, 512 threads and one element per SM).  The FP64 kernel
// takes 9.4 ms, so meshes of 512 elements or more come here only with it_max 1 or no re-solve.
__global__ void __launch_bounds__(kThreads, 2) k_local3d_mixed(const __grid_constant__ Local3DArgs g,
                                                               const __grid_constant__ Source3 source) {
    extern __shared__ double sm[];
    __shared__ int bad;
    __shared__ double FKs;
    const int n = g.n, n1 = n - 1, nb = g.nb, NI = g.NI, R = g.R, m = g.m, off = g.off, slots = g.slots;
    const Mixed3Smem L = mixed3_smem(n, R, nb, g.nsub, off, slots);
    double *S = sm + L.S, *kap = sm + L.kap, *A = sm + L.A, *Z = sm + L.Z, *Rr = sm + L.Rr, *sc = sm + L.sc;
    double *src = sm + L.src, *cp = sm + L.cp, *cf = sm + L.cf, *gn = sm + L.gn, *red = sm + L.red, *mz = sm + L.mz;
    float* W = reinterpret_cast<float*>(sm + L.W);
    float* Lc = reinterpret_cast<float*>(sm + L.Lc);
    float* inv = reinterpret_cast<float*>(sm + L.inv);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    constexpr int NWARP = kThreads / 32;
    for (int64_t K = g.K0 + blockIdx.x; K < g.K1; K += gridDim.x) {
        const double* geo = g.geo24 + 8 * (K % 24);
        const double vol = geo[0];
        // ---- class matrices, kappa, source loads; projection and face coefficients per column
        for (int t = tid; t < 6 * nb * nb; t += kThreads) S[t] = g.cls24[(size_t)(K % 24) * 6 * nb * nb + t];
        for (int t = tid; t < g.nsub; t += kThreads) kap[t] = g.kappa[K * (int64_t)g.nsub + t];
        if (tid == 0) bad = 0;
        if (g.source) source_loads3(g, source, K, Rr, src);
        if (warp == 0) {
            double f = 0.0;
            if (g.source) {
                for (int w = lane; w < n; w += 32) f += src[w];
                f = warp_sum(f);
            } else {
                f = g.src_value * vol;
            }
            if (lane == 0) FKs = cp[NI] = f;
        }
        auto moment = [&](int j) {   // (psi_j, 1)_{dK}
            const int a = j / m, q = j % m, b0 = (a * 6 + g.perm[4 * K + a]) * (m + 1) + q;
            int c = 0;
            for (int e = g.ftab_off[b0]; e < g.ftab_off[b0 + 1]; ++e) c += g.ftab_cnt[e];
            return (double)g.signs[4 * K + a] * geo[1 + a] * c;
        };
        for (int j = tid; j < NI; j += kThreads) {
            cp[j] = -moment(j);
            cf[j] = -(double)g.signs[4 * K + j / m] * geo[1 + j / m];
        }
        __syncthreads();
        // projected load of column c at node w
        auto load = [&](int w, int c) {
            const int d = w + (w >= g.pin);
            const double mt = g.mass1[d];
            double x = -cp[c] * mt;
            if (c == NI) return g.source ? x + src[d] : fma(g.src_value * vol, mt, x);
            const int a = c / m, cnt = g.fcnt[((a * 6 + g.perm[4 * K + a]) * n + d) * m + c % m];
            // (cnt as a double without a conversion: 2^52 + cnt - 2^52)
            if (cnt) x = fma(cf[c], __hiloint2double(0x43300000, cnt) - 4503599627370496.0, x);
            return x;
        };
        // ---- values of the pinned matrix, the scaling S = diag^-1/2, the scaled values in FP32
        for (int q = tid; q < off + n1; q += kThreads) {
            const uint32_t v = g.val[q];
            const uint32_t* con = g.con + (v & 0xffff);
            double x = 0.0;
            for (int i = 0; i < (int)(v >> 16); ++i) x = fma(kap[con[i] & 0xffff], S[con[i] >> 16], x);
            A[q] = x;
        }
        __syncthreads();
        for (int w = tid; w < n1; w += kThreads) {
            const double d = A[off + w];
            if (!(d > 0.0)) bad = 1;
            sc[w] = d > 0.0 ? 1.0 / sqrt(d) : 1.0;
        }
        __syncthreads();
        for (int q = tid; q < off + n1; q += kThreads) {
            const uint32_t rc = q < off ? g.rc[q] : (uint32_t)(q - off) * 0x10001u;
            W[q] = (float)(A[q] * sc[rc & 0xffff] * sc[rc >> 16]);
        }
        __syncthreads();
        // ---- FP32 factor: warp 0; the others prepare z = 0, r = g~ and |S g~|^2 per column
        if (warp == 0) {
            const mhm::FrontShared<float> sh = mhm::front_shared(reinterpret_cast<float*>(sm + L.front), FrontTilesMixed::vec);
            FrontRowsScaled rows{g, W, W + off, FrontTilesMixed::vec};
            float F[FrontTilesMixed::NT];
            mhm::front_eliminate<FrontTilesMixed>(rows, g.ev, g.steps, 0, sh, F, &bad, Lc, slots, inv, g.first);
        } else {
            for (int c = warp - 1; c < R; c += NWARP - 1) {
                double s = 0.0;
                for (int w = lane; w < n1; w += 32) {
                    const double r = load(w, c), x = sc[w] * r;
                    Rr[w * R + c] = r;
                    Z[w * R + c] = 0.0;
                    s = fma(x, x, s);
                }
                s = warp_sum(s);
                if (lane == 0) gn[c] = s;
            }
        }
        __syncthreads();
        // ---- refinement
        int passes = 0;
        bool converged = false;
        const double tol2 = g.tol * g.tol;
        for (int pass = 0; pass < g.it_max && !bad; ++pass) {
            for (int it = tid; it < n1 * R; it += kThreads) W[it] = (float)(sc[it / R] * Rr[it]);
            __syncthreads();
            if (warp < R) {
                // columns warp, warp + 8, warp + 16; a lane holds slots lane and lane + 32
                const int nc = (R - warp + NWARP - 1) / NWARP;
                float v0[3] = {0, 0, 0}, v1[3] = {0, 0, 0};
                int4 e = g.ev[0];
                for (int st = 0; st < g.steps; ++st) {
                    const int ps = e.x & 255, zs = (e.x >> 8) & 255, used = e.x >> 16, pn = e.w >> 16, en = e.y - (e.y > g.pin);
                    if (st + 1 < g.steps) e = g.ev[st + 1];
                    const bool pivot = ps != mhm::kNoSlot;
                    const float* lc = Lc + (st - g.first) * slots;
                    const float l0 = pivot && lane < used ? lc[lane] : 0.0f;
                    const float l1 = pivot && lane + 32 < used ? lc[lane + 32] : 0.0f;
                    const float di = pivot ? inv[st - g.first] : 0.0f;
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        if (k < nc) {
                            const int c = warp + NWARP * k;
                            const float y = pivot ? __shfl_sync(0xffffffffu, ps >= 32 ? v1[k] : v0[k], ps & 31) : 0.0f;
                            if (zs != mhm::kNoSlot) {
                                const float x = W[en * R + c];
                                if (zs == lane) v0[k] = x;
                                if (zs == lane + 32) v1[k] = x;
                            }
                            v0[k] = fmaf(-l0, y, v0[k]);
                            v1[k] = fmaf(-l1, y, v1[k]);
                            if (pivot && lane == 0) W[pn * R + c] = y * di;
                        }
                }
#pragma unroll
                for (int k = 0; k < 3; ++k) v0[k] = v1[k] = 0.0f;
                __syncwarp();
                for (int st = g.steps - 1; st >= g.first; --st) {
                    const int4 b = g.ev[st];
                    const int ps = b.x & 255, used = b.x >> 16, pn = b.w >> 16;
                    const float* lc = Lc + (st - g.first) * slots;
                    const float l0 = lane < used ? lc[lane] : 0.0f, l1 = lane + 32 < used ? lc[lane + 32] : 0.0f;
                    float t[3], y[3];
#pragma unroll
                    for (int k = 0; k < 3; ++k) {
                        y[k] = k < nc ? W[pn * R + warp + NWARP * k] : 0.0f;
                        t[k] = fmaf(l0, v0[k], l1 * v1[k]);
                    }
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
                        for (int k = 0; k < 3; ++k) t[k] += __shfl_xor_sync(0xffffffffu, t[k], o);
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        if (k < nc) {
                            const float x = y[k] - t[k];
                            if (ps == lane) v0[k] = x;
                            if (ps == lane + 32) v1[k] = x;
                            if (lane == 0) W[pn * R + warp + NWARP * k] = x;
                        }
                }
            }
            __syncthreads();
            // z += S w; then r = g~ - A z on the pinned rows (z vanishes on the pinned DOF)
            for (int it = tid; it < n1 * R; it += kThreads) Z[it] = fma(sc[it / R], (double)W[it], Z[it]);
            __syncthreads();
            for (int it = tid; it < n1 * R; it += kThreads) {
                const int w = it / R, c = it - w * R;
                double s = load(w, c);
                for (int q = g.rp[w]; q < g.rp[w + 1]; ++q) {
                    const uint32_t e = g.col[q];
                    s = fma(-A[e >> 16], Z[(e & 0xffff) * R + c], s);
                }
                Rr[it] = s;
            }
            __syncthreads();
            // converged when every column's |S r|^2 <= tol^2 |S g~|^2
            for (int c = warp; c < R; c += NWARP) {
                double s = 0.0;
                for (int w = lane; w < n1; w += 32) {
                    const double x = sc[w] * Rr[w * R + c];
                    s = fma(x, x, s);
                }
                s = warp_sum(s);
                if (lane == 0) red[c] = s;
            }
            __syncthreads();
            passes = pass + 1;
            converged = true;
            for (int c = 0; c < R; ++c) converged = converged && red[c] <= tol2 * gn[c];
            if (converged) break;   // (the same in every thread)
            __syncthreads();
        }
        converged = converged && !bad;

        // ---- corrected face integrals X_ji = g~_j . z_i + z_j . r_i, averaged with X_ij; the
        // multiplier loads live on their subface: g~_j . z = N_j . z - c_j m . z
        double* X = sm + L.W;   // (the FP32 solves are done)
        for (int c = warp; c < R; c += NWARP) {
            double s = 0.0;
            for (int w = lane; w < n1; w += 32) s = fma(g.mass1[w + (w >= g.pin)], Z[w * R + c], s);
            s = warp_sum(s);
            if (lane == 0) mz[c] = s;
        }
        __syncthreads();
        for (int it = tid; it < R * R; it += kThreads) {
            const int j = it / R, i = it - j * R;
            double s = -cp[j] * mz[i];
            if (j < NI) {
                const int a = j / m, b0 = (a * 6 + g.perm[4 * K + a]) * (m + 1) + j % m;
                double t = 0.0;
                for (int e = g.ftab_off[b0]; e < g.ftab_off[b0 + 1]; ++e) {
                    const int d = g.ftab_node[e], w = d - (d > g.pin);
                    if (d != g.pin) t = fma(__hiloint2double(0x43300000, g.ftab_cnt[e]) - 4503599627370496.0, Z[w * R + i], t);
                }
                s = fma(cf[j], t, s);
            } else if (g.source) {
                for (int w = 0; w < n1; ++w) s = fma(src[w + (w >= g.pin)], Z[w * R + i], s);
            } else {
                s = fma(g.src_value * vol, mz[i], s);
            }
            for (int w = 0; w < n1; ++w) s = fma(Z[w * R + j], Rr[w * R + i], s);
            X[it] = s;
        }
        __syncthreads();
        double* AK = g.AK + K * (int64_t)NI * NI;
        for (int it = tid; it < NI * NI; it += kThreads) {
            const int j = it / NI, i = it - j * NI;
            AK[it] = -0.5 * (X[j * R + i] + X[i * R + j]);
        }
        for (int j = tid; j < NI; j += kThreads) {
            g.EK[K * NI + j] = 0.5 * (X[j * R + NI] + X[NI * R + j]);
            g.BK[K * NI + j] = moment(j);
        }
        if (tid == 0) {
            g.FK[K] = FKs;
            g.status[K] = converged ? MHM_OK : MHM_ERR_NOT_CONVERGED;
            if (g.iters) g.iters[K] = passes;
        }
        __syncthreads();
    }
}

// skeleton values: one thread per entry of a neighbour block
__global__ void k_skeleton3d_A(const Nbr3* nbrs, int64_t nblocks, const int32_t* rowptr, int m, int NI,
                               const double* AK, double* vals) {
    const int64_t mm = (int64_t)m * m;
    for (int64_t it = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; it < nblocks * mm;
         it += (int64_t)gridDim.x * blockDim.x) {
        const Nbr3 b = nbrs[it / mm];
        const int q = (int)((it % mm) / m), q2 = (int)(it % m);
        double v = AK[((int64_t)b.K0 * NI + b.a0 * m + q) * NI + b.b0 * m + q2];
        if (b.K1 >= 0) v += AK[((int64_t)b.K1 * NI + b.a1 * m + q) * NI + b.b1 * m + q2];
        vals[rowptr[(int64_t)b.f * m + q] + b.col_off + q2] = v;
    }
}

__global__ void k_skeleton3d_E(const int32_t* face_ka, int64_t nlam, int m, int NI, const double* EK, double* E) {
    for (int64_t l = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; l < nlam; l += (int64_t)gridDim.x * blockDim.x) {
        const int64_t f = l / m;
        const int q = (int)(l % m);
        const int32_t* k = face_ka + 4 * f;
        double v = EK[(int64_t)k[0] * NI + k[1] * m + q];
        if (k[2] >= 0) v += EK[(int64_t)k[2] * NI + k[3] * m + q];
        E[l] = v;
    }
}

template <typename T>
mhm_status upload3(const std::vector<T>& h, T** d) {
    if (h.empty()) {
        *d = nullptr;
        return MHM_OK;
    }
    cudaError_t e = cudaMalloc((void**)d, h.size() * sizeof(T));
    if (e == cudaErrorMemoryAllocation) return mhm::fail(MHM_ERR_OOM, "cudaMalloc failed for 3-D mesh tables");
    if (e != cudaSuccess) return mhm::cuda_fail(e, "cudaMalloc");
    e = cudaMemcpy(*d, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return mhm::cuda_fail(e, "cudaMemcpy");
    return MHM_OK;
}

// sin and cos of pi x; x mod 2 is exact, so the argument of sin is rounded once.
void sincospi_host(double x, double* s, double* c) {
    const double y = M_PI * (x - 2.0 * std::rint(0.5 * x));
    *s = std::sin(y);
    *c = std::cos(y);
}

// Source3 for f = value 3 k^2 sin sin sin, k = freq pi.  Type 0 of h = 1 / nc has the edge vectors
// h (-1/2, 0, 0), h (0, -1/2, -1/2), h (0, 1, 0), and a point of class (p0, p1, p2) takes steps
// r0 >= r1 >= r2 along edges p0, p1, p2, so d = h / N (-t0 / 2, t2 - t1 / 2, -t1 / 2) with t[p_k] = r_k:
// three arguments t0, t1 and six pairs (t1, t2) per point for the six classes.
void source_tables(const mhm_mesh3d* m, double value, double freq, Source3* out) {
    const int nb = m->nb;
    const double h = 1.0 / m->desc.nc / m->N, kf = freq * M_PI;
    const double amp = h * h * h / 4.0 * value * 3.0 * kf * kf;   // 6 |sub-tetrahedron| = h^3 / 4
    double f[6][8];
    std::fill(out->M, out->M + 6 * 8 * nb, 0.0);
    for (int q = 0; q < kQuad; ++q) {
        const double* qp = &m->quad[4 * q];
        const double* phi = &m->quad[4 * kQuad + (size_t)q * nb];
        const double r[3] = {qp[0] + qp[1] + qp[2], qp[1] + qp[2], qp[2]};
        double sx[3], cx[3];
        for (int k = 0; k < 3; ++k) sincospi_host(freq * (-0.5 * h * r[k]), &sx[k], &cx[k]);
        for (int cls = 0; cls < 6; ++cls) {
            int at[3];   // step along each edge
            for (int k = 0; k < 3; ++k) at[kPath[cls][k]] = k;
            double sy, cy;
            sincospi_host(freq * (h * (r[at[2]] - 0.5 * r[at[1]])), &sy, &cy);
            for (int b = 0; b < 8; ++b)
                f[cls][b] = qp[3] * amp * (b & 1 ? sx[at[0]] : cx[at[0]]) * (b & 2 ? sy : cy) * (b & 4 ? sx[at[1]] : cx[at[1]]);
            double* M = out->M + cls * 8 * nb;
            for (int a = 0; a < nb; ++a)
                for (int b = 0; b < 8; ++b) M[8 * a + b] += phi[a] * f[cls][b];
        }
    }
    std::copy(&m->axis[0][0], &m->axis[0][0] + 24 * 4, &out->axis[0][0]);
}

// The mesh's small tables, gathered into one allocation and one copy (a cudaMalloc and a copy each
// take longer than the tables' contents).
struct Pack3 {
    std::vector<char> bytes;
    std::vector<std::pair<void**, size_t>> at;
    template <typename T, typename D>
    void add(const std::vector<T>& h, D** d) {
        at.emplace_back((void**)d, bytes.size());
        const char* p = reinterpret_cast<const char*>(h.data());
        bytes.insert(bytes.end(), p, p + h.size() * sizeof(T));
        bytes.resize((bytes.size() + 255) & ~(size_t)255);
    }
    mhm_status upload(char** base) {
        const mhm_status st = upload3(bytes, base);
        for (const auto& q : at) *q.first = st ? nullptr : *base + q.second;
        return st;
    }
};

// Tables of the frontal elimination: step tables; per element type (the 24 tetrahedra of a
// cube: every other element is a translate) the class matrices in closed form, |K| and the
// face areas; mass per DOF; face counts per local face, permutation, DOF and subface.
void add_front_tables(mhm_mesh3d* m, Pack3* pack) {
    const int nb = m->nb, n = (int)m->n, N = m->N, mm = m->desc.m, P = m->desc.degree;
    const mhm::FrontPlan3 plan = mhm::front_plan_3d(n, nb, m->sub_dofs, m->sub_cls, m->nodes, (int)m->NI + 1);
    m->fsteps = plan.steps;
    m->fslots = plan.slots;
    m->ffirst = plan.first_pivot;
    m->fpin = plan.pin;
    m->foff = plan.off;
    std::vector<double> cls((size_t)24 * 6 * nb * nb), geo(24 * 8, 0.0), mass(n, 0.0);
    for (int t = 0; t < 24; ++t) {
        const double* V = &m->geom[12 * t];
        double E[3][3];   // edge vectors along the path of the Freudenthal simplex
        for (int k = 0; k < 3; ++k)
            for (int c = 0; c < 3; ++c) E[k][c] = V[3 * (k + 1) + c] - V[3 * k + c];
        auto cross = [](const double* u, const double* v, double* w) {
            w[0] = u[1] * v[2] - u[2] * v[1], w[1] = u[2] * v[0] - u[0] * v[2], w[2] = u[0] * v[1] - u[1] * v[0];
        };
        double x[3];
        cross(E[1], E[2], x);
        geo[8 * t] = std::fabs(E[0][0] * x[0] + E[0][1] * x[1] + E[0][2] * x[2]) / 6.0;
        for (int a = 0; a < 4; ++a) {
            int b[3], k = 0;
            for (int v = 0; v < 4; ++v)
                if (v != a) b[k++] = v;
            double u[3], w[3];
            for (int c = 0; c < 3; ++c) u[c] = V[3 * b[1] + c] - V[3 * b[0] + c], w[c] = V[3 * b[2] + c] - V[3 * b[0] + c];
            cross(u, w, x);
            geo[8 * t + 1 + a] = 0.5 * std::sqrt(x[0] * x[0] + x[1] * x[1] + x[2] * x[2]) / ((double)N * N) / 3.0;
        }
        // edges 0 and 2 are the images of type 0's along -x and y, edge 1 of -(y + z) / 2
        const double sign[3] = {-1.0, 1.0, -1.0};
        const int edge[3] = {0, 2, 1};
        for (int y = 0; y < 3; ++y) {
            int x = 0;
            for (int c = 1; c < 3; ++c)
                if (y < 2 ? std::fabs(E[edge[y]][c]) > std::fabs(E[edge[y]][x]) : c != m->axis[t][0] % 4 && c != m->axis[t][1] % 4) x = c;
            m->axis[t][y] = (uint8_t)(x + (sign[y] * E[edge[y]][x] < 0.0 ? 4 : 0));
        }
        const double Vs = geo[8 * t] / ((double)N * N * N);
        for (int c = 0; c < 6; ++c) {
            double J[3][3], G[4][3];   // vertices of the class's path from its first; gradients of the barycentrics
            for (int v = 0; v < 3; ++v)
                for (int k = 0; k < 3; ++k) J[v][k] = (v ? J[v - 1][k] : 0.0) + E[kPath[c][v]][k] / N;
            const double* e[3] = {J[0], J[1], J[2]};
            for (int v = 0; v < 3; ++v) {
                cross(e[(v + 1) % 3], e[(v + 2) % 3], x);
                const double d = e[v][0] * x[0] + e[v][1] * x[1] + e[v][2] * x[2];
                for (int k = 0; k < 3; ++k) G[v + 1][k] = x[k] / d;
            }
            for (int k = 0; k < 3; ++k) G[0][k] = -(G[1][k] + G[2][k] + G[3][k]);
            auto d = [&](int i, int j) { return G[i][0] * G[j][0] + G[i][1] * G[j][1] + G[i][2] * G[j][2]; };
            // int grad phi_a . grad phi_b from int l_a l_b = Vs (1 + [a = b]) / 20 (P2 edges 4 l_a l_b)
            static const int ed[6][2] = {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}};
            double* S = &cls[((size_t)t * 6 + c) * nb * nb];
            for (int a = 0; a < nb; ++a)
                for (int b = 0; b < nb; ++b) {
                    double v;
                    if (P == 1) {
                        v = d(a, b);
                    } else if (a < 4 && b < 4) {
                        v = d(a, b) * (a == b ? 0.6 : -0.2);
                    } else if (a < 4 || b < 4) {
                        const int q = std::min(a, b), j = ed[std::max(a, b) - 4][0], k = ed[std::max(a, b) - 4][1];
                        v = 4.0 * (d(q, k) * (q == j ? 0.15 : -0.05) + d(q, j) * (q == k ? 0.15 : -0.05));
                    } else {
                        const int i = ed[a - 4][0], j = ed[a - 4][1], k = ed[b - 4][0], l = ed[b - 4][1];
                        v = 0.8 * (d(j, l) * (1 + (i == k)) + d(j, k) * (1 + (i == l)) + d(i, l) * (1 + (j == k)) +
                                   d(i, k) * (1 + (j == l)));
                    }
                    S[a * nb + b] = Vs * v;
                }
        }
    }
    const double per[2] = {P == 1 ? 0.25 : -0.05, 0.2};   // int phi over a tetrahedron of unit volume: vertices, edges
    for (int w = 0; w < n; ++w)
        for (int e = m->inc_off[w]; e < m->inc_off[w + 1]; ++e) mass[w] += per[m->inc_ent[e] % nb >= 4] / ((double)N * N * N);
    std::vector<uint8_t> cnt((size_t)24 * n * mm, 0);
    for (int b = 0; b < 24; ++b)
        for (int q = 0; q < mm; ++q)
            for (int e = m->ftab_off[b * (mm + 1) + q]; e < m->ftab_off[b * (mm + 1) + q + 1]; ++e)
                cnt[((size_t)b * n + m->ftab_node[e]) * mm + q] = (uint8_t)m->ftab_cnt[e];
    pack->add(plan.ev, &m->d_fev);
    pack->add(plan.ent, &m->d_fent);
    pack->add(plan.con, &m->d_fcon);
    pack->add(plan.val, &m->d_fval);
    pack->add(plan.rc, &m->d_frc);
    pack->add(plan.rp, &m->d_frp);
    pack->add(plan.col, &m->d_fcol);
    pack->add(cls, &m->d_cls24);
    pack->add(geo, &m->d_geo24);
    pack->add(mass, &m->d_mass1);
    pack->add(cnt, &m->d_fcnt);
}

void free_device(mhm_mesh3d* m) {
    void* ptrs[] = {m->d_geom, m->d_signs, m->d_perm, m->d_rowptr, m->d_nbrs, m->d_face_ka, m->d_tables};
    for (void* p : ptrs)
        if (p) cudaFree(p);
}

}  // namespace

}  // namespace mhm3

using namespace mhm3;

extern "C" mhm_status mhm3d_create_mesh(const mhm3d_mesh_desc* desc, int32_t device, mhm3d_mesh** out) {
    if (!desc || !out) return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_create_mesh: NULL argument");
    *out = nullptr;
    const mhm3d_mesh_desc d = *desc;
    if (d.nc < 1 || d.nc > 64 || d.r < 0 || d.r > 4 || (d.degree != 1 && d.degree != 2))
        return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_create_mesh: need 1 <= nc <= 64, 0 <= r <= 4, degree 1 or 2");
    int s = 0;
    while ((1 << (2 * s)) < d.m && s < 8) ++s;
    if (d.m < 1 || (1 << (2 * s)) != d.m || s > d.r)
        return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_create_mesh: m must be 4^s with s <= r");
    if (d.degree == 1 && (1 << d.r) < 2 * (1 << s))
        return mhm::fail(MHM_ERR_INVALID_ARG,
                         "mhm3d_create_mesh: degree 1 needs 2^r >= 2 sqrt(m) (the local traces must outnumber "
                         "the multipliers, else A_K is singular)");
    const int PN = d.degree << d.r;
    const int64_t n = (int64_t)(PN + 1) * (PN + 2) * (PN + 3) / 6;
    const int64_t nK = 24LL * d.nc * d.nc * d.nc;
    if (nK * 16LL * d.m * d.m > (1LL << 34))   // A_K alone: n_K N_I^2 doubles
        return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_create_mesh: the per-element blocks would exceed 2^34 values");
    if (device >= 0) {
        if (!mhm::device_supported(device))
            return mhm::fail(MHM_ERR_UNSUPPORTED, "mhm3d_create_mesh: device is not an sm_103 GPU");
        if (n > kMaxLocal || d.m > kMaxM)
            return mhm::fail(MHM_ERR_UNSUPPORTED,
                             "mhm3d_create_mesh: more local DOFs or multipliers than the kernels take "
                             "(degree 2: r <= 2, degree 1: r <= 3, m <= 16)");
    }
    mhm_mesh3d* m = new mhm_mesh3d();
    m->device = device;
    m->desc = d;
    m->s = s;
    const std::string err = build_mesh3d_host(m);
    if (!err.empty()) {
        delete m;
        return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_create_mesh: " + err);
    }
    if (device >= 0) {
        cudaError_t ce = cudaSetDevice(device);
        if (ce != cudaSuccess) {
            delete m;
            return mhm::cuda_fail(ce, "cudaSetDevice");
        }
        mhm_status st = MHM_OK;
        if (!st) st = upload3(m->geom, &m->d_geom);
        if (!st) st = upload3(m->signs, &m->d_signs);
        if (!st) st = upload3(m->perm, &m->d_perm);
        if (!st) st = upload3(m->rowptr, &m->d_rowptr);
        if (!st) st = upload3(m->nbrs, &m->d_nbrs);
        if (!st) st = upload3(m->face_ka, &m->d_face_ka);
        Pack3 pack;
        pack.add(m->sub_cls, &m->d_sub_cls);
        pack.add(m->sub_base, &m->d_sub_base);
        pack.add(m->inc_off, &m->d_inc_off);
        pack.add(m->inc_ent, &m->d_inc_ent);
        pack.add(m->ftab_off, &m->d_ftab_off);
        pack.add(m->ftab_node, &m->d_ftab_node);
        pack.add(m->ftab_cnt, &m->d_ftab_cnt);
        add_front_tables(m, &pack);
        if (!st) st = pack.upload(&m->d_tables);
        if (st) {
            free_device(m);
            delete m;
            return st;
        }
    }
    *out = m;
    return MHM_OK;
}

extern "C" void mhm3d_destroy_mesh(mhm3d_mesh* mesh) {
    if (!mesh) return;
    if (mesh->device >= 0) {
        cudaSetDevice(mesh->device);
        free_device(mesh);
    }
    delete mesh;
}

extern "C" mhm_status mhm3d_mesh_query(const mhm3d_mesh* m, int32_t what, void* host_out, size_t bytes) {
    if (!m || !host_out) return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_mesh_query: NULL argument");
    auto copy = [&](const void* src, size_t n) -> mhm_status {
        if (bytes < n) return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_mesh_query: output buffer too small");
        if (n) std::memcpy(host_out, src, n);
        return MHM_OK;
    };
    switch (what) {
        case MHM3D_Q_SIZES: {
            const int64_t s[8] = {m->nK, m->nf, m->nv, m->nlam, m->n, m->NI, m->nsub, m->nnz};
            return copy(s, sizeof(s));
        }
        case MHM3D_Q_TETS: return copy(m->tets.data(), m->tets.size() * 4);
        case MHM3D_Q_TET_FACES: return copy(m->tet_faces.data(), m->tet_faces.size() * 4);
        case MHM3D_Q_TET_SIGNS: return copy(m->signs.data(), m->signs.size());
        case MHM3D_Q_FACES: return copy(m->faces.data(), m->faces.size() * 4);
        case MHM3D_Q_VERTICES: return copy(m->verts.data(), m->verts.size() * 8);
        case MHM3D_Q_NORMALS: return copy(m->normals.data(), m->normals.size() * 8);
        case MHM3D_Q_CSR_ROWPTR: return copy(m->rowptr.data(), m->rowptr.size() * 4);
        case MHM3D_Q_CSR_COLS: return copy(m->cols.data(), m->cols.size() * 4);
        case MHM3D_Q_SUB_DOFS: return copy(m->sub_dofs.data(), m->sub_dofs.size() * 4);
        case MHM3D_Q_NODES: return copy(m->nodes.data(), m->nodes.size() * 4);
        case MHM3D_Q_FACE_PERM: return copy(m->perm.data(), m->perm.size());
        case MHM3D_Q_FTAB_OFF: return copy(m->ftab_off.data(), m->ftab_off.size() * 4);
        case MHM3D_Q_FTAB_NODE: return copy(m->ftab_node.data(), m->ftab_node.size() * 2);
        case MHM3D_Q_FTAB_COUNT: return copy(m->ftab_cnt.data(), m->ftab_cnt.size());
        case MHM3D_Q_QUAD: return copy(m->quad.data(), m->quad.size() * 8);
        default: return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_mesh_query: unknown query");
    }
}

extern "C" mhm_status mhm3d_local_solve_batch(const mhm3d_mesh* m, const double* kappa, const mhm3d_source* f,
                                              int32_t precision, const mhm3d_opts* opts, int64_t K0, int64_t K1,
                                              double* AK, double* EK, double* BK, double* FK, int32_t* status,
                                              int32_t* iters, void* stream) {
    // every argument is checked before the device: a host-only mesh reports argument errors too
    if (!m) return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_local_solve_batch: NULL mesh");
    if (!kappa || !f || !AK || !EK || !BK || !FK || !status)
        return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_local_solve_batch: NULL pointer argument");
    if (f->kind != MHM3D_SRC_CONST && f->kind != MHM3D_SRC_SINSINSIN)
        return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_local_solve_batch: unknown source kind");
    if (precision != MHM_FP64 && precision != MHM_MIXED)
        return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_local_solve_batch: precision must be MHM_FP64 or MHM_MIXED");
    mhm3d_opts o{8, 1e-9, 0};
    if (opts) o = *opts;
    if (o.it_max < 1 || !(o.tol > 0.0))
        return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_local_solve_batch: it_max >= 1 and tol > 0 required");
    if (K1 <= 0) K1 = m->nK;
    if (K0 < 0 || K1 > m->nK || K0 > K1) return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_local_solve_batch: K range");
    if (m->device < 0) return mhm::fail(MHM_ERR_UNSUPPORTED, "mhm3d_local_solve_batch: host-only mesh");
    if (K1 == K0) return MHM_OK;
    MHM_CUDA_TRY(cudaSetDevice(m->device));
    Local3DArgs g{};
    g.geom = m->d_geom, g.signs = m->d_signs, g.perm = m->d_perm;
    g.sub_cls = m->d_sub_cls, g.sub_base = m->d_sub_base;
    g.inc_off = m->d_inc_off, g.inc_ent = m->d_inc_ent;
    g.ftab_off = m->d_ftab_off, g.ftab_node = m->d_ftab_node, g.ftab_cnt = m->d_ftab_cnt;
    g.kappa = kappa;
    g.src_value = f->value, g.src_freq = f->freq;
    g.K0 = K0, g.K1 = K1;
    g.N = m->N, g.n = (int)m->n, g.nb = m->nb, g.nsub = (int)m->nsub, g.m = m->desc.m;
    g.NI = (int)m->NI, g.R = (int)m->NI + 1;
    g.AK = AK, g.EK = EK, g.BK = BK, g.FK = FK, g.status = status, g.iters = iters;
    g.it_max = o.it_max, g.tol = o.tol;
    g.ev = m->d_fev, g.ent = m->d_fent, g.con = m->d_fcon, g.steps = m->fsteps, g.slots = m->fslots, g.pin = m->fpin;
    g.cls24 = m->d_cls24, g.geo24 = m->d_geo24, g.mass1 = m->d_mass1, g.fcnt = m->d_fcnt;
    g.val = m->d_fval, g.rc = m->d_frc, g.rp = m->d_frp, g.col = m->d_fcol, g.first = m->ffirst, g.off = m->foff;
    cudaStream_t s = (cudaStream_t)stream;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->device);
    const Front3Kernel k = front3_kernel(g.R + m->fslots, K1 - K0 <= 3 * (int64_t)sms);
    if (!k.kern) return mhm::fail(MHM_ERR_UNSUPPORTED, "mhm3d_local_solve_batch: front too large");
    Source3 source{};
    g.source = f->kind == MHM3D_SRC_SINSINSIN;
    if (g.source) source_tables(m, f->value, f->freq, &source);
    cudaError_t e = cudaSuccess;
    // one wave of blocks that share the elements out evenly
    auto launch = [&](void (*kern)(const Local3DArgs, const Source3), int threads, size_t smem) {
        int per_sm = 0;
        cudaError_t c = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (c == cudaSuccess) c = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
        if (c != cudaSuccess) return c;
        const int64_t each = (K1 - K0 + sms - 1) / sms, rounds = (each + std::max(per_sm, 1) - 1) / std::max(per_sm, 1);
        kern<<<(unsigned)std::min<int64_t>(K1 - K0, sms * ((each + rounds - 1) / rounds)), threads, smem, s>>>(g, source);
        return cudaGetLastError();
    };
    // MIXED with room to refine and the FP64 re-solve allowed ends with FP64-quality blocks on
    // either kernel, and the FP64 one is the faster (12288 elements, m = 4: 9.4 against 24.6 ms,
    // 1536: 1.5 against 3.6; m = 1: 6.6 against 17.7, 0.9 against 2.6; P1 r = 3: 10.6 against 23.3,
    // 1.6 against 3.4; 192 elements: 0.43 against 0.65).  The line was drawn where the two met with
    // one warp per element in FP64; with four it is the faster below 512 too, where the refinement
    // stays for the sake of tol and iters.  The rule goes by the mesh and not by the call's range:
    // a range gives the full call's bits.
    const bool direct = o.it_max >= 2 && !o.no_fallback && m->nK >= 512;
    const bool mixed = precision == MHM_MIXED && !direct && g.R <= kMaxMixedR && m->fslots <= FrontTilesMixed::rows;
    if (mixed)
        e = launch(k_local3d_mixed, kThreads,
                   (size_t)mixed3_smem(g.n, g.R, g.nb, g.nsub, g.off, g.slots).total * sizeof(double));
    if (e == cudaSuccess && !(mixed && o.no_fallback)) {
        g.only_failed = mixed;   // the elements the refinement could not finish, again in FP64
        e = launch(k.kern, k.threads,
                   (size_t)front3_smem(k.vec, g.n, g.nb, g.nsub, g.source != 0).total * sizeof(double));
    }
    if (e != cudaSuccess) return mhm::cuda_fail(e, "mhm3d_local_solve_batch: launch");
    return MHM_OK;
}

extern "C" mhm_status mhm3d_assemble_skeleton(const mhm3d_mesh* m, const double* AK, const double* EK,
                                              double* A_vals, double* E, void* stream) {
    if (!m) return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_assemble_skeleton: NULL mesh");
    if (!AK || !EK || !A_vals || !E) return mhm::fail(MHM_ERR_INVALID_ARG, "mhm3d_assemble_skeleton: NULL pointer");
    if (m->device < 0) return mhm::fail(MHM_ERR_UNSUPPORTED, "mhm3d_assemble_skeleton: host-only mesh");
    MHM_CUDA_TRY(cudaSetDevice(m->device));
    const int64_t nblocks = (int64_t)m->nbrs.size();
    const int64_t items = nblocks * m->desc.m * m->desc.m;
    const int threads = 256;
    int sms = 152;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->device);
    const int64_t want = (items + threads - 1) / threads;
    const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * 8));
    k_skeleton3d_A<<<grid, threads, 0, (cudaStream_t)stream>>>(m->d_nbrs, nblocks, m->d_rowptr, m->desc.m,
                                                               (int)m->NI, AK, A_vals);
    MHM_CUDA_TRY(cudaGetLastError());
    const int64_t want_e = (m->nlam + threads - 1) / threads;
    const unsigned grid_e = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want_e, (int64_t)sms * 8));
    k_skeleton3d_E<<<grid_e, threads, 0, (cudaStream_t)stream>>>(m->d_face_ka, m->nlam, m->desc.m, (int)m->NI, EK, E);
    MHM_CUDA_TRY(cudaGetLastError());
    return MHM_OK;
}
