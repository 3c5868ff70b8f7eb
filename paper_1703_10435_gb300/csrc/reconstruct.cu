// computeSolution (Alg. 1; Sec. 2, Eq. "u_Hh"; Sec. 3): on every coarse
// triangle K,  u_{H,h} = u0_K + sum_i k_i eta_i + eta_f.  By linearity this is
// one zero-mean Neumann solve per K with the combined load
//     g = sum_i k_i N~_i + f~      (k_i: global multipliers of K's local basis),
// done here in FP64: the frontal elimination of the FP64 local solves (front.cuh) with that
// load as its one border row, which keeps every step's scaled pivot column w / d in scratch,
// and a backward sweep over the steps by one warp, x_p = g_p / d - sum_j (w_j / d) x_j over
// the front.  Optional per-K squared L2 and broken-H1 errors against an exact solution by the
// collapsed 4 x 4 Gauss rule per fine triangle.
// Levels whose front is too large (P2 r = 7) are refused.
//
// Bound by the FP64 pipe (85 % busy): 16.6 k FP64 warp instructions per element of P1 r = 5,
// of which the update of the front takes 8 k, a step's fixed part (reciprocal, scaling,
// couplings, the backward sum) the rest.  32768 elements: 32.2 ms (182.6 ms with a window
// over two levels and a dense backward sweep).
#include <cuda_runtime.h>

#include <algorithm>

#include "front2d.cuh"
#include "local_common.cuh"

namespace mhm {

namespace {

struct RecArgs {
    DeviceMesh dm;
    const double* kappa;
    const double* lambda;
    const double* u0;
    const int32_t* k_lambda;    // n_K * N_I global multiplier ids
    int P, N, PN, dpf, NI, nloc;
    int src_kind;
    const double* src_vals;   // MHM_SRC_QUAD: 16 values per fine triangle, laid out like kappa
    double src_value, src_freq;
    int ex_kind;                // 0 none, 1 sin sin, 2 quadratic polynomial
    double ex[6];
    char* ws;
    size_t slot_bytes;
    int64_t nK;                 // launch indices of this level
    const int64_t* nod_off;     // first nodal value of each K in u_out (NULL: K * nloc)
    double* u_out;              // n_K * nloc (per-K levels: at nod_off)
    double* err_out;            // n_K * 2 (squared L2, squared H1 seminorm) or NULL
    const int4* ev;             // frontal elimination: the level's step tables
    const uint2* cp;
    int steps, slots;
};

__device__ __forceinline__ void fine_xy(const double Xc[3][2], int N, bool up, int i, int j, double X[3][2]) {
    const double e1x = (Xc[1][0] - Xc[0][0]) / N, e1y = (Xc[1][1] - Xc[0][1]) / N;
    const double e2x = (Xc[2][0] - Xc[0][0]) / N, e2y = (Xc[2][1] - Xc[0][1]) / N;
    int a[3][2];
    if (up) { a[0][0] = i; a[0][1] = j; a[1][0] = i + 1; a[1][1] = j; a[2][0] = i; a[2][1] = j + 1; }
    else    { a[0][0] = i + 1; a[0][1] = j; a[1][0] = i + 1; a[1][1] = j + 1; a[2][0] = i; a[2][1] = j + 1; }
    for (int v = 0; v < 3; ++v) {
        X[v][0] = Xc[0][0] + a[v][0] * e1x + a[v][1] * e2x;
        X[v][1] = Xc[0][1] + a[v][0] * e1y + a[v][1] * e2y;
    }
}

__device__ __forceinline__ void basis_eval(int P, double l0, double l1, double l2, double* phi, double* dxi,
                                           double* deta) {
    if (P == 1) {
        phi[0] = l0; phi[1] = l1; phi[2] = l2;
        dxi[0] = -1; dxi[1] = 1; dxi[2] = 0;
        deta[0] = -1; deta[1] = 0; deta[2] = 1;
        return;
    }
    phi[0] = l0 * (2 * l0 - 1); phi[1] = l1 * (2 * l1 - 1); phi[2] = l2 * (2 * l2 - 1);
    phi[3] = 4 * l1 * l2; phi[4] = 4 * l2 * l0; phi[5] = 4 * l0 * l1;
    dxi[0] = -(4 * l0 - 1); deta[0] = -(4 * l0 - 1);
    dxi[1] = 4 * l1 - 1;    deta[1] = 0;
    dxi[2] = 0;             deta[2] = 4 * l2 - 1;
    dxi[3] = 4 * l2;        deta[3] = 4 * l1;
    dxi[4] = -4 * l2;       deta[4] = 4 * (l0 - l2);
    dxi[5] = 4 * (l0 - l1); deta[5] = -4 * l1;
}

__device__ void exact_eval(const RecArgs& g, double x, double y, double* u, double* ux, double* uy) {
    if (g.ex_kind == 1) {
        const double f = g.ex[0], amp = g.ex[1];
        const double sx = sinpi(f * x), sy = sinpi(f * y), cx = cospi(f * x), cy = cospi(f * y);
        *u = amp * sx * sy;
        *ux = amp * f * M_PI * cx * sy;
        *uy = amp * f * M_PI * sx * cy;
    } else {
        const double* c = g.ex;
        *u = c[0] + c[1] * x + c[2] * y + c[3] * x * x + c[4] * x * y + c[5] * y * y;
        *ux = c[1] + 2 * c[3] * x + c[4] * y;
        *uy = c[2] + c[4] * x + 2 * c[5] * y;
    }
}

__device__ double block_sum(double v, double* red) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];   // same order in every thread
    __syncthreads();
    return s;
}

// Squared L2 and H1 errors of u = zs + shift on element K (vertices Xc); all threads.
__device__ void element_errors(const RecArgs& g, int64_t K, const double Xc[3][2], const double* zs, double shift,
                               double* red) {
    const double* gx = g.dm.gauss_x + 3 * kMaxGauss;
    const double* gw = g.dm.gauss_w + 3 * kMaxGauss;
    const int nb = g.P == 1 ? 3 : 6;
    double e2 = 0.0, h2 = 0.0;
    for (int t = threadIdx.x; t < g.N * g.N; t += blockDim.x) {
        int j = 0, rs = 0;
        while (rs + 2 * (g.N - j) - 1 <= t) { rs += 2 * (g.N - j) - 1; ++j; }
        const int o = t - rs;
        const bool up = o < g.N - j;
        const int i = up ? o : o - (g.N - j);
        int nx[6], ny[6];
        element_nodes(g.P, up, i, j, nx, ny);
        double X[3][2];
        fine_xy(Xc, g.N, up, i, j, X);
        const double j00 = X[1][0] - X[0][0], j10 = X[1][1] - X[0][1];
        const double j01 = X[2][0] - X[0][0], j11 = X[2][1] - X[0][1];
        const double det = j00 * j11 - j01 * j10;
        double uv[6];
        for (int a = 0; a < nb; ++a)
            uv[a] = zs[ny[a] * (g.PN + 1) - ny[a] * (ny[a] - 1) / 2 + nx[a]] + shift;
        for (int qi = 0; qi < 4; ++qi)
            for (int qj = 0; qj < 4; ++qj) {
                const double xi = gx[qi], eta = gx[qj] * (1.0 - gx[qi]);
                const double w = gw[qi] * gw[qj] * (1.0 - gx[qi]) * fabs(det);
                double phi[6], dxi[6], deta[6];
                basis_eval(g.P, 1.0 - xi - eta, xi, eta, phi, dxi, deta);
                double uh = 0.0, gxi = 0.0, geta = 0.0;
                for (int a = 0; a < nb; ++a) {
                    uh += phi[a] * uv[a];
                    gxi += dxi[a] * uv[a];
                    geta += deta[a] * uv[a];
                }
                // grad_x = J^{-T} grad_ref
                const double ux = (j11 * gxi - j10 * geta) / det, uy = (-j01 * gxi + j00 * geta) / det;
                const double x = X[0][0] + xi * j00 + eta * j01, y = X[0][1] + xi * j10 + eta * j11;
                double ue, uex, uey;
                exact_eval(g, x, y, &ue, &uex, &uey);
                e2 += w * (uh - ue) * (uh - ue);
                h2 += w * ((ux - uex) * (ux - uex) + (uy - uey) * (uy - uey));
            }
    }
    const double E2 = block_sum(e2, red), H2 = block_sum(h2, red);
    if (threadIdx.x == 0) {
        g.err_out[2 * K] = E2;
        g.err_out[2 * K + 1] = H2;
    }
}

// Load of a node: the combined load of the nodes in dof order.
struct RecLoad {
    const double* gl;
    int PN;
    __device__ __forceinline__ void node(int) {}
    __device__ __forceinline__ double operator()(int x, int y, int, int) const {
        return gl[y * (PN + 1) - y * (y - 1) / 2 + x];
    }
};

struct RecSmem {
    int Ke, mass, lamc, xs, red, tab, z, total;   // doubles
};
__host__ __device__ inline RecSmem rec_smem(int vec, int NI, int kind, int P, int N) {
    const int PN = P * N;
    RecSmem l;
    int o = (int)front_shared_values(vec);
    l.Ke = o, o += 72;
    l.mass = o, o += 8;
    l.lamc = o, o += NI;     // k_i (-s |F|) per local multiplier
    l.xs = o, o += vec;      // solution at the front's slots
    l.red = o, o += 32;
    l.tab = o, o += source_table_doubles(kind, PN);
    l.z = o, o += (PN + 1) * (PN + 2) / 2;   // load, then solution, per node
    l.total = o;
    return l;
}

// One block per coarse triangle at a time (front.cuh); SL: slots per lane of the backward sweep.
template <class T, int NCP, int SL, int MINB>
__global__ void __launch_bounds__(T::threads, MINB) k_reconstruct(const __grid_constant__ RecArgs g) {
    extern __shared__ double smem[];
    __shared__ FrontCtx c;
    const int P = g.P, N = g.N, PN = g.PN, NI = g.NI, tid = threadIdx.x, nthr = blockDim.x, stride = g.slots + 1;
    const RecSmem L = rec_smem(T::vec, NI, g.src_kind, P, N);
    const FrontShared<double> sh = front_shared(smem, T::vec);
    double *Ke = smem + L.Ke, *lamc = smem + L.lamc, *xs = smem + L.xs, *z = smem + L.z;
    double* keep = reinterpret_cast<double*>(g.ws + (size_t)blockIdx.x * g.slot_bytes);
    for (int64_t ki = blockIdx.x; ki < g.nK; ki += gridDim.x) {
        const int64_t K = g.dm.klist ? (int64_t)g.dm.klist[ki] : ki;
        const double* kap = g.kappa + (g.dm.kap_off ? g.dm.kap_off[K] : K * (int64_t)N * N);
        front_element(g.dm, K, kap, P, N, g.src_kind, g.src_value, g.src_freq, c, Ke, smem + L.mass, smem + L.tab);
        front_source(g.src_kind, g.src_value, P, N, smem + L.tab,
                     g.src_vals ? g.src_vals + 16 * (kap - g.kappa) : nullptr, c, z);
        if (tid < 32) {   // k_i N_i's coefficients and sum_i k_i (1^T N_i) / |K|
            double cl = 0.0;
            for (int i = tid; i < NI; i += 32) {
                const int a = i / g.dpf, row = face_row(i - a * g.dpf, c.la1[a], g.dm.fm, g.dm.lmax1);
                lamc[i] = row < 0 ? 0.0 : g.lambda[g.k_lambda[K * NI + i]] * (-c.sgn[a] * c.flen[a]);
                if (row >= 0) cl = fma(lamc[i], g.dm.btab_sum[row], cl);
            }
            for (int o = 16; o > 0; o >>= 1) cl += __shfl_xor_sync(0xffffffffu, cl, o);
            if (tid == 0) smem[L.red] = (cl + c.FK) / c.area;   // coefficient of the mass vector
        }
        __syncthreads();
        const double cm = smem[L.red], area_fine = c.area / ((double)N * N);
        {
            int x = tid, y = 0;
            for (int u = tid; u < g.nloc; u += nthr, x += nthr) {
                while (x > PN - y) x -= PN + 1 - y, ++y;
                const double m = node_mass(P, N, x, y, area_fine);
                double v = g.src_kind == MHM_SRC_CONST ? (g.src_value - cm) * m : fma(-cm, m, z[u]);
                for (int a = 0; a < 3; ++a) {
                    const int kl = face_position(PN, x, y, a);
                    if (kl < 0) continue;
                    const int kk = c.rev[a] ? PN - kl : kl;
                    for (int jf = 0; jf < g.dpf; ++jf) {
                        const int row = face_row(jf, c.la1[a], g.dm.fm, g.dm.lmax1);
                        if (row >= 0) v = fma(lamc[a * g.dpf + jf], g.dm.btab[row * (PN + 1) + kk], v);
                    }
                }
                z[u] = v;
            }
        }
        __syncthreads();
        FrontRows2D<NCP, RecLoad> rows{g.cp, kap, Ke, g.steps, 1, T::vec, c.pin, RecLoad{z, PN}};
        if (T::NW == 1 || (tid >> 5) == T::NW) rows.start();
        {
            double A[T::NT];
            front_eliminate<T>(rows, g.ev, g.steps, 1, sh, A, &c.bad, keep, stride);
        }
        __syncthreads();
        // backward sweep; two steps' columns are in flight
        if (tid < 32) {
            for (int q = tid; q < T::vec; q += 32) xs[q] = 0.0;
            struct Col { double s[SL], y; int4 v; };
            auto fetch = [&](int e) {
                Col k;
                k.v = make_int4(kNoSlot | kNoSlot << 8, 0, 0, 0);
                if (e >= 0) k.v = g.ev[e];
                const bool on = (k.v.x & 255) != kNoSlot;
                const int m = on ? (k.v.x >> 16) & 255 : 0;
                const double* r = keep + (size_t)max(e, 0) * stride;
                k.y = on ? r[0] : 0.0;
#pragma unroll
                for (int q = 0; q < SL; ++q) k.s[q] = tid + 32 * q < m ? r[1 + tid + 32 * q] : 0.0;
                return k;
            };
            Col k0 = fetch(g.steps - 1), k1 = fetch(g.steps - 2);
            __syncwarp();
            for (int e = g.steps - 1; (k0.v.x & 255) != kNoSlot; --e) {
                const Col k2 = fetch(e - 2);
                double t = k0.s[0] * xs[tid];
#pragma unroll
                for (int q = 1; q < SL; ++q) t = fma(k0.s[q], xs[tid + 32 * q], t);
                for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
                t = k0.y - t;
                __syncwarp();
                if (tid == 0) {
                    const int x = k0.v.w & 0xffff, y = k0.v.w >> 16;
                    xs[k0.v.x & 255] = t;
                    z[y * (PN + 1) - y * (y - 1) / 2 + x] = t;
                }
                __syncwarp();
                k0 = k1;
                k1 = k2;
            }
        }
        __syncthreads();
        // zero mean, then u0
        double mz = 0.0;
        {
            int x = tid, y = 0;
            for (int u = tid; u < g.nloc; u += nthr, x += nthr) {
                while (x > PN - y) x -= PN + 1 - y, ++y;
                mz = fma(node_mass(P, N, x, y, area_fine), z[u], mz);
            }
        }
        const double mean = block_sum(mz, smem + L.red) / c.area;
        double shift = g.u0[K] - mean;
        if (c.scale != 0) {   // (the mean in the scaled range: mass times z can underflow in the other)
            for (int u = tid; u < g.nloc; u += nthr) z[u] = (z[u] - mean) * exp2_of(c.scale);
            __syncthreads();
            shift = g.u0[K];
        }
        double* uK = g.u_out + (g.nod_off ? g.nod_off[K] : K * (int64_t)g.nloc);
        for (int w = tid; w < g.nloc; w += nthr) uK[w] = z[w] + shift;
        if (g.err_out) element_errors(g, K, c.X, z, shift, smem + L.red);
        __syncthreads();
    }
}

// The frontal kernel of a level (one border row); NULL if the front is too large.
struct RecKernel {
    void (*kern)(const RecArgs) = nullptr;
    int threads = 0, vec = 0;
};
template <class T, int SL, int MINB>
void rec_try(const Level& lv, RecKernel* k) {
    if (k->kern || lv.fsteps == 0 || lv.fslots + 1 > T::rows || lv.fslots > 32 * SL) return;
    k->kern = lv.fncp == 8 ? k_reconstruct<T, 8, SL, MINB> : k_reconstruct<T, 16, SL, MINB>;
    k->threads = T::threads;
    k->vec = T::vec;
}
// (few: no more elements than three per SM, which four warps each finish sooner: front.cuh)
RecKernel rec_kernel(const Level& lv, bool few) {
    RecKernel k;
    if (few) {
        rec_try<FrontTiles<4, 1, 2>, 1, 4>(lv, &k);
        rec_try<FrontTiles<4, 1, 3>, 2, 4>(lv, &k);
    }
    rec_try<FrontTiles<1, 1, 5>, 1, 16>(lv, &k);
    rec_try<FrontTiles<1, 1, 9>, 2, 16>(lv, &k);
    rec_try<FrontTiles<4, 1, 5>, 3, 3>(lv, &k);
    rec_try<FrontTiles<4, 2, 9>, 5, 1>(lv, &k);
    return k;
}

}  // namespace

}  // namespace mhm

using namespace mhm;

extern "C" mhm_status mhm_reconstruct(const mhm_mesh* mesh, const double* kappa, const mhm_source* f,
                                      const double* lambda, const double* u0, const mhm_exact* exact,
                                      double* u_nodal, double* err_sq, void* stream) {
    if (!mesh) return fail(MHM_ERR_INVALID_ARG, "mhm_reconstruct: NULL mesh");
    if (mesh->device < 0) return fail(MHM_ERR_UNSUPPORTED, "mhm_reconstruct: mesh was created without a device");
    if (!kappa || !f || !lambda || !u0 || !u_nodal) return fail(MHM_ERR_INVALID_ARG, "mhm_reconstruct: NULL pointer argument");
    if (err_sq && !exact) return fail(MHM_ERR_INVALID_ARG, "mhm_reconstruct: err_sq needs an exact solution");
    {
        const mhm_status sst = check_source(f, "mhm_reconstruct");
        if (sst) return sst;
    }
    if (exact && exact->kind != MHM_EXACT_SINSIN && exact->kind != MHM_EXACT_POLY)
        return fail(MHM_ERR_INVALID_ARG, "mhm_reconstruct: unknown exact-solution kind");
    MHM_CUDA_TRY(cudaSetDevice(mesh->device));
    cudaStream_t s = (cudaStream_t)stream;
    // one launch per refinement level, in stream order
    for (const Level& lv : mesh->levels) {
        RecArgs g;
        g.dm = mesh->dev(lv);
        g.kappa = kappa;
        g.lambda = lambda;
        g.u0 = u0;
        g.k_lambda = mesh->d_k_lambda;
        g.P = mesh->desc.degree;
        g.N = lv.N;
        g.PN = lv.PN;
        g.dpf = mesh->dpf;
        g.NI = (int)mesh->NI;
        g.nloc = (int)lv.nloc;
        g.src_kind = f->kind;
        g.src_vals = f->kind == MHM_SRC_QUAD ? f->values_dev : nullptr;
        g.src_value = f->value;
        g.src_freq = f->freq;
        g.ex_kind = exact ? (exact->kind == MHM_EXACT_SINSIN ? 1 : 2) : 0;
        for (int i = 0; i < 6; ++i) g.ex[i] = exact ? exact->c[i] : 0.0;
        g.nK = lv.nK;
        g.nod_off = mesh->d_nod_off;
        g.u_out = u_nodal;
        g.err_out = err_sq;
        int sms = 0, occ = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, mesh->device);
        const RecKernel front = rec_kernel(lv, lv.nK <= 3 * (int64_t)sms);
        g.ev = lv.d_fev;
        g.cp = lv.d_fcp;
        g.steps = lv.fsteps;
        g.slots = lv.fslots;
        if (!front.kern) return fail(MHM_ERR_UNSUPPORTED, "mhm_reconstruct: front too large (r too large)");
        void (*kern)(const RecArgs) = front.kern;
        const int threads = front.threads;
        g.slot_bytes = ((size_t)g.steps * (g.slots + 1) * sizeof(double) + 255) & ~(size_t)255;
        const size_t smem = (size_t)rec_smem(front.vec, g.NI, f->kind, g.P, g.N).total * sizeof(double);
        MHM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem);
        // one wave, the elements shared out evenly
        const int64_t each = (lv.nK + sms - 1) / sms, rounds = (each + std::max(occ, 1) - 1) / std::max(occ, 1);
        const int64_t grid = std::min(lv.nK, sms * ((each + rounds - 1) / rounds));
        char* ws = nullptr;
        cudaError_t e = cudaMallocAsync((void**)&ws, (size_t)grid * g.slot_bytes, s);
        if (e != cudaSuccess) return cuda_fail(e, "mhm_reconstruct: cudaMallocAsync");
        g.ws = ws;
        kern<<<(unsigned)grid, threads, smem, s>>>(g);
        e = cudaGetLastError();
        cudaFreeAsync(ws, s);
        if (e != cudaSuccess) return cuda_fail(e, "mhm_reconstruct: launch");
    }
    return MHM_OK;
}
