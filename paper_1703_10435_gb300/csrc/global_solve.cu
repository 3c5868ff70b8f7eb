// reduceLocalProblems' solve (Alg. 1; Sec. 3, Eq. "mat_global"):
//     [ A  B^T ] [lambda]   [E]
//     [ B  0   ] [u0    ] = [F]
// in FP64 on the GPU, by a multifrontal LDL^T factorisation in a nested-dissection order
// of the structured coarse mesh (the paper solves this system with a direct sparse solver,
// Pardiso or PaStiX, Sec. 4.1).
//
// Ordering.  The coarse squares [i0, i1) x [j0, j1) are bisected along their longer side
// down to blocks of at most 2 x 2 squares.  A cut along a grid line owns the faces on that
// line (its separator); a leaf owns the faces inside its block (and those on the domain
// boundary) and the u0 of its elements.  The elements of a leaf touch only its own faces
// and the faces on its block's boundary, which belong to ancestors' separators, so the
// factorisation of a node touches only its front: its own unknowns and the boundary
// faces of its block (the update unknowns).
//
// Pivoting.  A is negative definite, so eliminating a node's multipliers before its u0
// gives negative pivots and then positive ones (the Schur complement B (-A)^-1 B^T is
// positive definite on the u0 a block can fix: see "constant modes" at dissect).  So an
// LDL^T without pivoting is stable in this order and the fronts keep a fixed structure.  Large
// fronts check the sign of their multipliers' pivots (kSignedPanel).
//
// Storage.  Every node has an F x F front (column-major, lower triangle) in one buffer:
// after its factorisation its first k columns hold L (unit lower triangle, diagonal entries
// replaced by D) and its trailing (F - k) x (F - k) block the update matrix its parent adds
// in.  All fronts of a depth are factored together, 32 pivots at a time: k_nd_panel factors the
// diagonal block and solves the rows below it, k_nd_update subtracts L D L^T from the trailing
// tiles.  (Library factorisations, one front after the other, took 93 of 132 ms at 128 x 128
// squares with 6 multipliers per face; 5.0 G multiply-adds are 8.0 ms of the FP64 pipe;
// the whole solve now takes 25.8 ms there.)
// Forward and backward substitution take 32 pivots at a time too, one block per front.  One
// step of iterative refinement against the assembled system follows the solve.
#include <cuda_runtime.h>

#include <algorithm>
#include <functional>
#include <map>
#include <string>
#include <vector>

#include "front.cuh"
#include "mhm_internal.h"

namespace mhm {

struct NDNode {
    int depth = 0, parent = -1, child[2] = {-1, -1};
    int64_t k = 0, F = 0;               // own unknowns, front size
    int64_t front_off = 0, vec_off = 0;  // offsets (doubles) in the front and vector buffers
    int64_t map_off[2] = {0, 0};         // children's update positions in this front
    std::vector<int32_t> idx;            // the front's unknowns: own (elimination order), then update
    int32_t deferred = -1;               // a u0 passed up to the parent (see dissect)
};

struct NDPlan {
    std::vector<NDNode> nodes;              // post-order (children before parents)
    std::vector<std::vector<int>> by_depth;
    struct Depth {              // the nodes of one depth in the list of all, and their largest sizes
        int64_t first = 0, count = 0, k = 0, F = 0, child = 0;
    };
    std::vector<Depth> depth;
    int64_t n = 0, front_doubles = 0, vec_doubles = 0;
    // device
    double* fronts = nullptr;
    double* vecs = nullptr;
    double* x = nullptr;       // solution
    double* dx = nullptr;      // correction of the refinement step
    double* b = nullptr;       // right-hand side
    double* r = nullptr;       // residual
    double* diag = nullptr;    // factored 32 x 32 diagonal blocks of the depth at hand, by node
    int* list = nullptr;       // nodes by depth
    double* vals = nullptr;    // values of the assembled saddle-point CSR (refinement)
    int64_t* dst = nullptr;    // per saddle-point entry: its place in a front (lower triangle), or -1
    int32_t* maps = nullptr;   // children's update -> parent front positions
    int32_t* idx = nullptr;    // all fronts' unknowns
    // per node: k, F, front_off, vec_off, map_off[0..1], child[0..1], idx offset, size of the first
    // child's update, pivots that have to be negative
    int64_t* node_info = nullptr;
    int* dinfo = nullptr;           // per node: a pivot was refused (k_nd_panel)
};

void free_nd_plan(NDPlan* p) {
    if (!p) return;
    for (void* q : {(void*)p->fronts, (void*)p->vecs, (void*)p->x, (void*)p->dx, (void*)p->b, (void*)p->r,
                    (void*)p->diag, (void*)p->list, (void*)p->vals, (void*)p->dst, (void*)p->maps, (void*)p->idx,
                    (void*)p->node_info, (void*)p->dinfo})
        if (q) cudaFree(q);
    delete p;
}

namespace {

constexpr int kNodeInfo = 11;   // int64 fields per node on the device
constexpr int kNdThreads = 256;
constexpr int kNdPanel = 32;    // pivots per step
// Fronts with a larger F x k panel (doubles) are refused if a multiplier's pivot is not negative:
// A is then not negative definite, and an indefinite front of hundreds of unknowns is not
// stable without pivoting.  In smaller ones only pivots that cannot be divided by are refused.
constexpr int64_t kSignedPanel = 20 * 1024;

// ---------------------------------------------------------------- symbolic ---

struct Grid {
    int nx, ny;
    std::map<std::pair<int32_t, int32_t>, int32_t> face_of;   // (vertex, vertex) -> face
    int32_t face(int i0, int j0, int i1, int j1) const {     // face between grid vertices
        const int32_t a = j0 * (nx + 1) + i0, b = j1 * (nx + 1) + i1;
        auto it = face_of.find({std::min(a, b), std::max(a, b)});
        return it == face_of.end() ? -1 : it->second;
    }
};

// Builds the dissection tree of the rectangle [i0, i1) x [j0, j1); returns the node id.
//
// Constant modes.  Inside a block that does not touch the domain boundary, the flux
// balance of the block as a whole involves only the faces on its boundary: the rows of B
// restricted to the faces the block eliminates are a signed incidence matrix of the
// connected graph of its elements, of rank (elements - 1), so the last u0 pivot would be
// zero.  Such a block therefore passes one u0 up as an update unknown; a parent eliminates
// the u0 its children pass up after its separator, passes one of them on unless its own
// block touches the domain boundary, and the root eliminates what is left.
int dissect(const mhm_mesh* m, const Grid& g, NDPlan& P, int i0, int i1, int j0, int j1, int depth) {
    const int w = i1 - i0, h = j1 - j0;
    const bool touches = i0 == 0 || j0 == 0 || i1 == g.nx || j1 == g.ny;
    NDNode node;
    node.depth = depth;
    std::vector<int32_t> own;
    auto add_face = [&](std::vector<int32_t>& v, int32_t f) {
        if (f < 0) return;   // (every grid line segment is a face of the structured mesh)
        for (int64_t j = m->lam_off[f]; j < m->lam_off[f + 1]; ++j) v.push_back((int32_t)j);
    };
    int c0 = -1, c1 = -1;
    if (w <= 2 && h <= 2) {
        // leaf: faces inside the block and on the domain boundary, then the u0 of its elements
        for (int j = j0; j <= j1; ++j)
            for (int i = i0; i < i1; ++i)
                if ((j > j0 && j < j1) || j == 0 || j == g.ny) add_face(own, g.face(i, j, i + 1, j));
        for (int i = i0; i <= i1; ++i)
            for (int j = j0; j < j1; ++j)
                if ((i > i0 && i < i1) || i == 0 || i == g.nx) add_face(own, g.face(i, j, i, j + 1));
        for (int j = j0; j < j1; ++j)
            for (int i = i0; i < i1; ++i) add_face(own, g.face(i, j, i + 1, j + 1));
        for (int j = j0; j < j1; ++j)
            for (int i = i0; i < i1; ++i) {
                const int64_t K = 2 * ((int64_t)j * g.nx + i);
                own.push_back((int32_t)(m->nlam + K));
                own.push_back((int32_t)(m->nlam + K + 1));
            }
        if (!touches) {
            node.deferred = own.back();
            own.pop_back();
        }
    } else if (w >= h) {
        const int im = i0 + w / 2;
        c0 = dissect(m, g, P, i0, im, j0, j1, depth + 1);
        c1 = dissect(m, g, P, im, i1, j0, j1, depth + 1);
        for (int j = j0; j < j1; ++j) add_face(own, g.face(im, j, im, j + 1));
    } else {
        const int jm = j0 + h / 2;
        c0 = dissect(m, g, P, i0, i1, j0, jm, depth + 1);
        c1 = dissect(m, g, P, i0, i1, jm, j1, depth + 1);
        for (int i = i0; i < i1; ++i) add_face(own, g.face(i, jm, i + 1, jm));
    }
    if (c0 >= 0) {
        bool any = false;
        for (int c : {c0, c1})
            if (P.nodes[c].deferred >= 0) {
                own.push_back(P.nodes[c].deferred);
                any = true;
            }
        if (!touches && any) {
            node.deferred = own.back();
            own.pop_back();
        }
    }
    // update unknowns: the faces on the block's boundary that are not on the domain boundary
    std::vector<int32_t> upd;
    if (j0 > 0)
        for (int i = i0; i < i1; ++i) add_face(upd, g.face(i, j0, i + 1, j0));
    if (j1 < g.ny)
        for (int i = i0; i < i1; ++i) add_face(upd, g.face(i, j1, i + 1, j1));
    if (i0 > 0)
        for (int j = j0; j < j1; ++j) add_face(upd, g.face(i0, j, i0, j + 1));
    if (i1 < g.nx)
        for (int j = j0; j < j1; ++j) add_face(upd, g.face(i1, j, i1, j + 1));
    if (node.deferred >= 0) upd.push_back(node.deferred);
    node.k = (int64_t)own.size();
    node.idx = own;
    node.idx.insert(node.idx.end(), upd.begin(), upd.end());
    node.F = (int64_t)node.idx.size();
    node.child[0] = c0;
    node.child[1] = c1;
    P.nodes.push_back(std::move(node));
    const int id = (int)P.nodes.size() - 1;
    if (c0 >= 0) P.nodes[c0].parent = id;
    if (c1 >= 0) P.nodes[c1].parent = id;
    return id;
}

}  // namespace

mhm_status build_nd_plan(const mhm_mesh* m, NDPlan** out) {
    NDPlan* P = new NDPlan();
    Grid g;
    g.nx = m->desc.nx;
    g.ny = m->desc.ny;
    for (int64_t e = 0; e < m->ne; ++e) g.face_of[{m->face_v[2 * e], m->face_v[2 * e + 1]}] = (int32_t)e;
    dissect(m, g, *P, 0, g.nx, 0, g.ny, 0);
    P->n = m->nlam + m->nK;
    // every unknown owned by exactly one node
    std::vector<int32_t> node_of(P->n, -1), pos_of(P->n, -1);
    for (size_t id = 0; id < P->nodes.size(); ++id) {
        const NDNode& nd = P->nodes[id];
        for (int64_t t = 0; t < nd.k; ++t) {
            if (node_of[nd.idx[t]] >= 0) {
                free_nd_plan(P);
                return fail(MHM_ERR_INVALID_ARG, "mhm_solve_global: an unknown owned twice by the dissection");
            }
            node_of[nd.idx[t]] = (int32_t)id;
            pos_of[nd.idx[t]] = (int32_t)t;
        }
    }
    for (int64_t u = 0; u < P->n; ++u)
        if (node_of[u] < 0) {
            free_nd_plan(P);
            return fail(MHM_ERR_INVALID_ARG, "mhm_solve_global: an unknown owned by no node of the dissection");
        }
    int maxd = 0;
    for (NDNode& nd : P->nodes) maxd = std::max(maxd, nd.depth);
    P->by_depth.assign(maxd + 1, {});
    for (size_t id = 0; id < P->nodes.size(); ++id) {
        NDNode& nd = P->nodes[id];
        nd.front_off = P->front_doubles;
        P->front_doubles += nd.F * nd.F;
        nd.vec_off = P->vec_doubles;
        P->vec_doubles += nd.F;
        P->by_depth[nd.depth].push_back((int)id);
    }
    std::vector<int32_t> list;
    size_t widest = 1;
    for (const std::vector<int>& ids : P->by_depth) {
        NDPlan::Depth d;
        d.first = (int64_t)list.size();
        d.count = (int64_t)ids.size();
        widest = std::max(widest, ids.size());
        for (int id : ids) {
            const NDNode& nd = P->nodes[id];
            list.push_back(id);
            d.k = std::max(d.k, nd.k);
            d.F = std::max(d.F, nd.F);
            for (int c : nd.child)
                if (c >= 0) d.child = std::max(d.child, P->nodes[c].F - P->nodes[c].k);
        }
        P->depth.push_back(d);
    }
    // children's update positions in the parent's front
    std::vector<int32_t> maps;
    for (NDNode& nd : P->nodes) {
        std::map<int32_t, int32_t> pos;
        for (int64_t t = 0; t < nd.F; ++t) pos[nd.idx[t]] = (int32_t)t;
        for (int s = 0; s < 2; ++s) {
            nd.map_off[s] = (int64_t)maps.size();
            if (nd.child[s] < 0) continue;
            const NDNode& c = P->nodes[nd.child[s]];
            for (int64_t t = c.k; t < c.F; ++t) {
                auto it = pos.find(c.idx[t]);
                if (it == pos.end()) {
                    free_nd_plan(P);
                    return fail(MHM_ERR_INVALID_ARG, "mhm_solve_global: a child's update unknown outside its parent");
                }
                maps.push_back(it->second);
            }
        }
    }
    // each saddle-point entry (r, c) goes to the front of whichever of r, c is eliminated
    // first (post-order of the nodes, then the order inside the node), lower triangle only
    std::vector<int64_t> dst(m->aug_nnz, -1);
    auto rank = [&](int32_t u) { return ((int64_t)node_of[u] << 32) | pos_of[u]; };
    for (int64_t r = 0; r < P->n; ++r) {
        for (int32_t t = m->aug_rowptr[r]; t < m->aug_rowptr[r + 1]; ++t) {
            const int32_t c = m->aug_cols[t];
            const int32_t first = rank((int32_t)r) <= rank(c) ? (int32_t)r : c;
            const NDNode& nd = P->nodes[node_of[first]];
            // positions of r and c in that front
            auto find = [&](int32_t u) -> int64_t {
                if (node_of[u] == node_of[first]) return pos_of[u];
                for (int64_t q = nd.k; q < nd.F; ++q)
                    if (nd.idx[q] == u) return q;
                return -1;
            };
            const int64_t pr = find((int32_t)r), pc = find(c);
            if (pr < 0 || pc < 0) {
                free_nd_plan(P);
                return fail(MHM_ERR_INVALID_ARG, "mhm_solve_global: a matrix entry outside the fronts");
            }
            if (pr >= pc) dst[t] = nd.front_off + pr + pc * nd.F;
        }
    }
    std::vector<int64_t> info(P->nodes.size() * kNodeInfo);
    std::vector<int32_t> idx_all;
    for (size_t id = 0; id < P->nodes.size(); ++id) {
        const NDNode& nd = P->nodes[id];
        idx_all.insert(idx_all.end(), nd.idx.begin(), nd.idx.end());
        int64_t* q = &info[id * kNodeInfo];
        q[0] = nd.k;
        q[1] = nd.F;
        q[2] = nd.front_off;
        q[3] = nd.vec_off;
        q[4] = nd.map_off[0];
        q[5] = nd.map_off[1];
        q[6] = nd.child[0];
        q[7] = nd.child[1];
        q[8] = (int64_t)idx_all.size() - nd.F;
        q[9] = nd.child[0] >= 0 ? P->nodes[nd.child[0]].F - P->nodes[nd.child[0]].k : 0;
        q[10] = 0;   // pivots that have to be negative: the own multipliers, which come first
        while (nd.F * nd.k > kSignedPanel && q[10] < nd.k && nd.idx[q[10]] < m->nlam) ++q[10];
    }
    // device
    auto up = [](const auto& v, auto** d) -> cudaError_t {
        using T = typename std::decay<decltype(v[0])>::type;
        cudaError_t e = cudaMalloc((void**)d, std::max<size_t>(1, v.size()) * sizeof(T));
        if (e == cudaSuccess && !v.empty()) e = cudaMemcpy(*d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
        return e;
    };
    cudaError_t e = cudaMalloc((void**)&P->fronts, P->front_doubles * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&P->vecs, P->vec_doubles * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&P->x, P->n * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&P->dx, P->n * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&P->b, P->n * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&P->r, P->n * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&P->diag, widest * kNdPanel * kNdPanel * sizeof(double));
    if (e == cudaSuccess) e = cudaMalloc((void**)&P->vals, std::max<int64_t>(1, m->aug_nnz) * sizeof(double));
    if (e == cudaSuccess) e = up(dst, &P->dst);
    if (e == cudaSuccess) e = up(maps, &P->maps);
    if (e == cudaSuccess) e = up(idx_all, &P->idx);
    if (e == cudaSuccess) e = up(list, &P->list);
    if (e == cudaSuccess) e = up(info, &P->node_info);
    if (e == cudaSuccess) e = cudaMalloc((void**)&P->dinfo, std::max<size_t>(1, P->nodes.size()) * sizeof(int));
    if (e != cudaSuccess) {
        free_nd_plan(P);
        return cuda_fail(e, "mhm_solve_global: device memory of the factorisation");
    }
    *out = P;
    return MHM_OK;
}

namespace {

// ----------------------------------------------------------------- kernels ---

__global__ void k_fill_saddle(int64_t nnz, const int64_t* src, const double* A_vals, const double* BK, double* out) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= nnz) return;
    const int64_t s = src[t];
    out[t] = s >= 0 ? A_vals[s] : BK[-s - 1];
}

__global__ void k_nd_assemble(int64_t nnz, const int64_t* dst, const double* vals, double* fronts) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < nnz && dst[t] >= 0) fronts[dst[t]] = vals[t];
}

// The update block of child slot s of every node in `list` added into the node's front
// (lower triangles on both sides); grid (nodes, groups of the child's columns).
__global__ void k_nd_extend_add(const int* list, int slot, const int64_t* info, const int32_t* maps, double* fronts) {
    const int64_t* q = info + (int64_t)list[blockIdx.x] * kNodeInfo;
    const int64_t c = q[6 + slot];
    if (c < 0) return;
    const int64_t* qc = info + c * kNodeInfo;
    const int64_t kc = qc[0], Fc = qc[1], Fp = q[1];
    const int nu = (int)(Fc - kc);
    const int32_t* map = maps + q[4 + slot];
    const double* C = fronts + qc[2];
    double* Pf = fronts + q[2];
    // a warp per column
    for (int j = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5); j < nu; j += gridDim.y * (blockDim.x >> 5)) {
        const int64_t pj = map[j];
        for (int i = j + (threadIdx.x & 31); i < nu; i += 32) {
            const int64_t pi = map[i], hi = pi > pj ? pi : pj, lo = pi > pj ? pj : pi;
            Pf[hi + lo * Fp] += C[(kc + i) + (kc + j) * Fc];
        }
    }
}

// One step of the LDL^T without pivoting of every front of a depth: the diagonal block of the
// (up to) 32 pivots from p0 on and the rows below it, l = w / d with w_q = a_q - sum_{r<q}
// w_r L_qr.  Grid (nodes, groups of blockDim rows): one warp of every block factors the
// diagonal block for itself (a lane a row, in registers; the pivot column through shared
// memory), then a thread solves one row in registers.  A block of four warps takes 15 us of
// the FP64 pipe for its rows, one of a single warp 4: depths with few fronts use single warps.
// (The diagonal block by four warps with a barrier and a division per pivot: 40 us.)  The
// factored diagonal block goes to `diag` (the other blocks of the front still read the old
// one); k_nd_update puts it in place.
__global__ void __launch_bounds__(128) k_nd_panel(const int* list, const int64_t* info, double* fronts, int p0,
                                                  double* diag, int* bad) {
    __shared__ double L[kNdPanel][kNdPanel + 1];
    __shared__ double dinv[kNdPanel], col[2][kNdPanel];
    const int id = list[blockIdx.x];
    const int64_t* q = info + (int64_t)id * kNodeInfo;
    const int k = (int)q[0], F = (int)q[1];
    const int nb = min(kNdPanel, k - p0);
    const int row0 = p0 + nb + blockIdx.y * blockDim.x;
    if (nb <= 0 || (blockIdx.y > 0 && row0 >= F)) return;
    double* Fr = fronts + q[2];
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        double a[kNdPanel];   // row `lane`; rows and columns past nb: unit
#pragma unroll
        for (int j = 0; j < kNdPanel; ++j)
            a[j] = lane >= j && lane < nb ? Fr[(p0 + lane) + (int64_t)(p0 + j) * F] : (lane == j ? 1.0 : 0.0);
#pragma unroll
        for (int p = 0; p < kNdPanel; ++p) {   // column p keeps w = l d until its turn is over
            if (p < nb) {
                double* w = col[p & 1];
                w[lane] = a[p];
                __syncwarp();
                const double d = w[p], inv = front_rcp(d);
                if (lane == 0) {
                    dinv[p] = inv;
                    // zero, not finite or where front_rcp does not hold; of the wrong sign
                    const int h = __double2hiint(d);
                    if (blockIdx.y == 0 && (!front_positive(fabs(d)) || (p0 + p < q[10] && h >= 0))) bad[id] = 1;
                }
                const double l = a[p] * inv;
#pragma unroll
                for (int j = p + 1; j < kNdPanel; ++j) a[j] = fma(-l, w[j], a[j]);   // (j > lane: not used)
                if (lane > p) a[p] = l;
            } else if (lane == p) {
                dinv[p] = 1.0;
            }
        }
#pragma unroll
        for (int j = 0; j < kNdPanel; ++j) {
            L[lane][j] = a[j];
            if (blockIdx.y == 0) diag[((int64_t)blockIdx.x * kNdPanel + j) * kNdPanel + lane] = a[j];
        }
    }
    __syncthreads();
    const int i = row0 + threadIdx.x;
    if (i >= F) return;
    double w[kNdPanel];
#pragma unroll
    for (int c = 0; c < kNdPanel; ++c) w[c] = c < nb ? Fr[i + (int64_t)(p0 + c) * F] : 0.0;
#pragma unroll
    for (int r = 0; r < kNdPanel; ++r)
#pragma unroll
        for (int c = r + 1; c < kNdPanel; ++c) w[c] = fma(-w[r], L[c][r], w[c]);
#pragma unroll
    for (int c = 0; c < kNdPanel; ++c)
        if (c < nb) Fr[i + (int64_t)(p0 + c) * F] = w[c] * dinv[c];
}

// The step's update of the trailing lower triangle, U -= L21 D L21^T, in TS x TS tiles (grid
// (nodes, tiles)), a thread 4 x 4 entries; tile 0 also puts the factored diagonal block in place.
template <int TS>
__global__ void __launch_bounds__(TS * TS / 16) k_nd_update(const int* list, const int64_t* info, double* fronts, int p0,
                                                            const double* diag) {
    __shared__ double Ls[kNdPanel][TS], Ws[kNdPanel][TS];
    constexpr int TH = TS / 4, NT = TH * TH;
    const int64_t* q = info + (int64_t)list[blockIdx.x] * kNodeInfo;
    const int k = (int)q[0], F = (int)q[1];
    const int nb = min(kNdPanel, k - p0);
    if (nb <= 0) return;
    double* Fr = fronts + q[2];
    const double* dg = diag + (int64_t)blockIdx.x * kNdPanel * kNdPanel;
    if (blockIdx.y == 0)
        for (int t = threadIdx.x; t < nb * kNdPanel; t += NT) {
            const int j = t / kNdPanel, i = t % kNdPanel;
            if (i >= j && i < nb) Fr[(p0 + i) + (int64_t)(p0 + j) * F] = dg[j * kNdPanel + i];
        }
    const int pe = p0 + nb, nt = (F - pe + TS - 1) / TS;
    int ti = (int)((sqrtf(8.0f * blockIdx.y + 1.0f) - 1.0f) * 0.5f);   // tile row of the lower triangle
    while (ti * (ti + 1) / 2 > (int)blockIdx.y) --ti;
    while ((ti + 1) * (ti + 2) / 2 <= (int)blockIdx.y) ++ti;
    const int tj = (int)blockIdx.y - ti * (ti + 1) / 2;
    if (ti >= nt) return;
    const int r0 = pe + ti * TS, c0 = pe + tj * TS;
    for (int t = threadIdx.x; t < kNdPanel * TS; t += NT) {
        const int c = t / TS, i = t % TS;
        const double d = c < nb ? dg[c * kNdPanel + c] : 0.0;
        Ls[c][i] = c < nb && r0 + i < F ? Fr[(r0 + i) + (int64_t)(p0 + c) * F] : 0.0;
        Ws[c][i] = c < nb && c0 + i < F ? d * Fr[(c0 + i) + (int64_t)(p0 + c) * F] : 0.0;
    }
    __syncthreads();
    const int tx = threadIdx.x % TH, ty = threadIdx.x / TH;   // rows tx + TH a, columns ty + TH b
    double acc[4][4] = {};
    for (int c = 0; c < nb; ++c) {
        double l[4], w[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) l[a] = Ls[c][tx + TH * a], w[a] = Ws[c][ty + TH * a];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = fma(l[a], w[b], acc[a][b]);
    }
#pragma unroll
    for (int b = 0; b < 4; ++b)
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const int i = r0 + tx + TH * a, j = c0 + ty + TH * b;
            if (i < F && j <= i) Fr[i + (int64_t)j * F] -= acc[a][b];
        }
}

// Forward elimination and diagonal scaling of one depth (one block per node): the front
// vector (shared memory, F values) takes the own right-hand sides and the children's update
// vectors; 32 own pivots at a time, solved by one warp against the diagonal block, then
// subtracted from the rows below; then z = y / d on the own part.  The update part stays for
// the parent.
__global__ void __launch_bounds__(kNdThreads) k_nd_forward(const int* list, const int64_t* info, const int32_t* maps,
                                                           const int32_t* idx, const double* fronts, double* vecs,
                                                           const double* b) {
    extern __shared__ double v[];
    __shared__ double L[kNdPanel][kNdPanel + 1];
    const int64_t* q = info + (int64_t)list[blockIdx.x] * kNodeInfo;
    const int k = (int)q[0], F = (int)q[1], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double* Fr = fronts + q[2];
    const int32_t* ix = idx + q[8];
    for (int i = threadIdx.x; i < F; i += kNdThreads) v[i] = i < k ? b[ix[i]] : 0.0;
    __syncthreads();
    for (int s = 0; s < 2; ++s) {   // children in a fixed order
        const int64_t c = q[6 + s];
        if (c < 0) continue;
        const int64_t* qc = info + c * kNodeInfo;
        const int64_t kc = qc[0], nu = qc[1] - kc;
        const double* vc = vecs + qc[3];
        const int32_t* map = maps + q[4 + s];
        for (int64_t i = threadIdx.x; i < nu; i += kNdThreads) v[map[i]] += vc[kc + i];
        __syncthreads();
    }
    for (int p0 = 0; p0 < k; p0 += kNdPanel) {
        const int nb = min(kNdPanel, k - p0);
        for (int j = warp; j < nb; j += kNdThreads / 32)
            if (lane < nb) L[lane][j] = Fr[(p0 + lane) + (int64_t)(p0 + j) * F];
        __syncthreads();
        if (warp == 0) {
            double y = lane < nb ? v[p0 + lane] : 0.0;
            for (int r = 0; r < nb; ++r) {
                const double yr = __shfl_sync(0xffffffffu, y, r);
                if (lane > r && lane < nb) y = fma(-L[lane][r], yr, y);
            }
            if (lane < nb) v[p0 + lane] = y;
        }
        __syncthreads();
        for (int i = p0 + nb + threadIdx.x; i < F; i += kNdThreads) {
            const double* col = Fr + i + (int64_t)p0 * F;
            double s = v[i];
            if (nb == kNdPanel) {   // (all loads in flight)
#pragma unroll
                for (int c = 0; c < kNdPanel; ++c) s = fma(-col[(int64_t)c * F], v[p0 + c], s);
            } else {
                for (int c = 0; c < nb; ++c) s = fma(-col[(int64_t)c * F], v[p0 + c], s);
            }
            v[i] = s;
        }
        __syncthreads();
    }
    double* out = vecs + q[3];
    for (int i = threadIdx.x; i < F; i += kNdThreads) out[i] = i < k ? v[i] / Fr[i + (int64_t)i * F] : v[i];
}

// Back substitution of one depth (one block per node, parents before children): x at the
// update unknowns comes from the solution vector (ancestors); x_p = z_p - sum_{i > p}
// L[i][p] x_i for the own pivots from last to first, 32 at a time (a warp per column for the
// rows below the diagonal block, then one warp inside it); the own x go to the solution vector.
__global__ void __launch_bounds__(kNdThreads) k_nd_backward(const int* list, const int64_t* info, const int32_t* idx,
                                                            const double* fronts, const double* vecs, double* x) {
    extern __shared__ double v[];
    __shared__ double L[kNdPanel][kNdPanel + 1];
    __shared__ double sum[kNdPanel];
    const int64_t* q = info + (int64_t)list[blockIdx.x] * kNodeInfo;
    const int k = (int)q[0], F = (int)q[1], lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double* Fr = fronts + q[2];
    const double* z = vecs + q[3];
    const int32_t* ix = idx + q[8];
    for (int i = threadIdx.x; i < F; i += kNdThreads) v[i] = i < k ? z[i] : x[ix[i]];
    __syncthreads();
    for (int p0 = (k - 1) / kNdPanel * kNdPanel; p0 >= 0; p0 -= kNdPanel) {
        const int nb = min(kNdPanel, k - p0);
        {   // a warp takes columns warp, warp + 8, .. together
            constexpr int W = kNdThreads / 32, C = kNdPanel / W;
            const double* col[C];
            double s[C];
#pragma unroll
            for (int c = 0; c < C; ++c) {
                const int j = min(warp + W * c, nb - 1);   // (past nb: the last column again, not kept)
                col[c] = Fr + (int64_t)(p0 + j) * F;
                s[c] = 0.0;
                if (lane < nb) L[lane][j] = col[c][p0 + lane];
            }
#pragma unroll 4
            for (int i = p0 + nb + lane; i < F; i += 32) {
                const double x = v[i];
#pragma unroll
                for (int c = 0; c < C; ++c) s[c] = fma(col[c][i], x, s[c]);
            }
#pragma unroll
            for (int c = 0; c < C; ++c) {
                for (int o = 16; o > 0; o >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], o);
                if (lane == 0 && warp + W * c < nb) sum[warp + W * c] = s[c];
            }
        }
        __syncthreads();
        if (warp == 0) {
            double t = lane < nb ? v[p0 + lane] - sum[lane] : 0.0;
            for (int r = nb - 1; r > 0; --r) {
                const double xr = __shfl_sync(0xffffffffu, t, r);
                if (lane < r) t = fma(-L[r][lane], xr, t);
            }
            if (lane < nb) v[p0 + lane] = t;
        }
        __syncthreads();
    }
    for (int p = threadIdx.x; p < k; p += kNdThreads) x[ix[p]] = v[p];
}

// r = b - M x for the assembled saddle-point CSR (one warp per row, fixed summation order).
__global__ void k_nd_residual(int64_t n, const int32_t* rowptr, const int32_t* cols, const double* vals,
                              const double* x, const double* b, double* r) {
    const int64_t row = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (row >= n) return;
    double s = 0.0;
    for (int32_t t = rowptr[row] + lane; t < rowptr[row + 1]; t += 32) s = fma(vals[t], x[cols[t]], s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (lane == 0) r[row] = b[row] - s;
}

__global__ void k_rhs_saddle(int64_t L, int64_t nK, const double* E, const double* FK, double* rhs) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < L) rhs[t] = E[t];
    else if (t < L + nK) rhs[t] = FK[t - L];
}

__global__ void k_add_split(int64_t L, int64_t nK, const double* x, const double* dx, double* lam, double* u0) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < L) lam[t] = x[t] + dx[t];
    else if (t < L + nK) u0[t - L] = x[t] + dx[t];
}

unsigned blocks_for(int64_t n, int threads) { return (unsigned)std::max<int64_t>(1, (n + threads - 1) / threads); }

// Solves M x = rhs into x with the factors in the fronts, depth by depth.
mhm_status nd_solve(const NDPlan* P, const double* rhs, double* x, cudaStream_t s) {
    for (size_t d = P->depth.size(); d-- > 0;) {
        const NDPlan::Depth& q = P->depth[d];
        k_nd_forward<<<(unsigned)q.count, kNdThreads, q.F * sizeof(double), s>>>(P->list + q.first, P->node_info, P->maps,
                                                                                P->idx, P->fronts, P->vecs, rhs);
    }
    for (const NDPlan::Depth& q : P->depth)
        k_nd_backward<<<(unsigned)q.count, kNdThreads, q.F * sizeof(double), s>>>(P->list + q.first, P->node_info, P->idx,
                                                                                  P->fronts, P->vecs, x);
    MHM_CUDA_TRY(cudaGetLastError());
    return MHM_OK;
}

// Factors the fronts of one depth: children's updates, then 32 pivots at a time.
mhm_status nd_factor(const NDPlan* P, const NDPlan::Depth& q, cudaStream_t s) {
    const int* list = P->list + q.first;
    const unsigned n = (unsigned)q.count;
    if (q.child > 0)
        for (int slot = 0; slot < 2; ++slot)
            k_nd_extend_add<<<dim3(n, (unsigned)std::min<int64_t>(64, (q.child + 7) / 8)), kNdThreads, 0, s>>>(
                list, slot, P->node_info, P->maps, P->fronts);
    for (int64_t p0 = 0; p0 < q.k; p0 += kNdPanel) {
        const int64_t rest = std::max<int64_t>(q.F - p0 - 1, 1);
        const int rows = n >= 128 ? 128 : 32;   // (rows per block: k_nd_panel)
        k_nd_panel<<<dim3(n, (unsigned)((rest + rows - 1) / rows)), rows, 0, s>>>(list, P->node_info, P->fronts, (int)p0,
                                                                                 P->diag, P->dinfo);
        // small fronts: 32 x 32 tiles (a leaf's trailing block has 24 to 72 rows)
        const int64_t ts = q.F >= 256 ? 64 : 32, t = (rest + ts - 1) / ts;
        const dim3 grid(n, (unsigned)(t * (t + 1) / 2));
        if (ts == 64) k_nd_update<64><<<grid, 256, 0, s>>>(list, P->node_info, P->fronts, (int)p0, P->diag);
        else k_nd_update<32><<<grid, 64, 0, s>>>(list, P->node_info, P->fronts, (int)p0, P->diag);
    }
    MHM_CUDA_TRY(cudaGetLastError());
    return MHM_OK;
}

}  // namespace

}  // namespace mhm

using namespace mhm;

extern "C" mhm_status mhm_solve_global(const mhm_mesh* mesh, const double* A_vals, const double* E,
                                       const double* BK, const double* FK, double* lambda, double* u0,
                                       void* stream) {
    if (!mesh) return fail(MHM_ERR_INVALID_ARG, "mhm_solve_global: NULL mesh");
    if (mesh->device < 0) return fail(MHM_ERR_UNSUPPORTED, "mhm_solve_global: mesh was created without a device");
    if (!A_vals || !E || !BK || !FK || !lambda || !u0)
        return fail(MHM_ERR_INVALID_ARG, "mhm_solve_global: NULL pointer argument");
    MHM_CUDA_TRY(cudaSetDevice(mesh->device));
    cudaStream_t s = (cudaStream_t)stream;
    if (!mesh->nd) {
        NDPlan* P = nullptr;
        mhm_status st = build_nd_plan(mesh, &P);
        if (st) return st;
        mesh->nd = P;
    }
    NDPlan* P = mesh->nd;
    const int thr = 256;
    // assembled saddle-point values, fronts zeroed and filled with the original entries
    k_fill_saddle<<<blocks_for(mesh->aug_nnz, thr), thr, 0, s>>>(mesh->aug_nnz, mesh->d_aug_src, A_vals, BK, P->vals);
    MHM_CUDA_TRY(cudaMemsetAsync(P->fronts, 0, P->front_doubles * sizeof(double), s));
    MHM_CUDA_TRY(cudaMemsetAsync(P->dinfo, 0, P->nodes.size() * sizeof(int), s));
    k_nd_assemble<<<blocks_for(mesh->aug_nnz, thr), thr, 0, s>>>(mesh->aug_nnz, P->dst, P->vals, P->fronts);
    MHM_CUDA_TRY(cudaGetLastError());
    mhm_status st = MHM_OK;
    size_t vec_bytes = 0;   // a front vector in shared memory
    for (const NDPlan::Depth& d : P->depth) vec_bytes = std::max(vec_bytes, (size_t)d.F * sizeof(double));
    if (vec_bytes > 200 * 1024) return fail(MHM_ERR_UNSUPPORTED, "mhm_solve_global: a front vector exceeds shared memory");
    MHM_CUDA_TRY(cudaFuncSetAttribute(k_nd_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vec_bytes));
    MHM_CUDA_TRY(cudaFuncSetAttribute(k_nd_backward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)vec_bytes));
    // numeric factorisation, deepest level first; solve, then one step of refinement against
    // the assembled system
    for (size_t d = P->depth.size(); d-- > 0 && !st;) st = nd_factor(P, P->depth[d], s);
    if (!st) {
        k_rhs_saddle<<<blocks_for(P->n, thr), thr, 0, s>>>(mesh->nlam, mesh->nK, E, FK, P->b);
        st = nd_solve(P, P->b, P->x, s);
    }
    if (!st) {
        k_nd_residual<<<blocks_for(P->n * 32, thr), thr, 0, s>>>(P->n, mesh->d_aug_rowptr, mesh->d_aug_cols, P->vals, P->x,
                                                                 P->b, P->r);
        st = nd_solve(P, P->r, P->dx, s);
    }
    if (!st) k_add_split<<<blocks_for(P->n, thr), thr, 0, s>>>(mesh->nlam, mesh->nK, P->x, P->dx, lambda, u0);
    cudaError_t e = cudaGetLastError();
    if (!st && e != cudaSuccess) st = cuda_fail(e, "mhm_solve_global: solve");
    if (!st) {
        // a refused pivot means a singular or (in a large front) indefinite system: report it (synchronises)
        std::vector<int> bad(P->nodes.size());
        e = cudaMemcpyAsync(bad.data(), P->dinfo, bad.size() * sizeof(int), cudaMemcpyDeviceToHost, s);
        if (e == cudaSuccess) e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) return cuda_fail(e, "mhm_solve_global: status");
        for (int v : bad)
            if (v != 0) return fail(MHM_ERR_INVALID_ARG, "mhm_solve_global: singular saddle-point system (zero, non-finite or wrong-sign pivot)");
    }
    return st;
}
