// Frontal elimination of the local problems in FP64.
//
// What it computes.  The pinned matrix A_p of a local problem bordered by its R load columns,
//     [ 0  G^T ]
//     [ G  A_p ],
// is eliminated node by node; after all nodes the leading block holds -G^T A_p^{-1} G, the
// face integrals of Eq. "mat_global".  A node enters when the elimination first touches it
// (front_plan.h), so the matrix at hand is the R loads and the nodes in the front, at most
// M = R + slots rows: 33 slots for P1 at N = 32, 35 for P2 at N = 16 (an elimination level by
// level works on windows of two levels, 64 and 127 rows).
//
// How.  This GPU has two FP64 multiply-adds per clock and SM, half a lane per scheduler: a
// warp's FP64 instruction holds its scheduler's unit for 64 clocks, however many of its lanes
// work, and about 60 other instructions fit beside it.  So the layout is made for full FP64 instructions: the lower
// triangle lives in registers in tiles of 4 x 8 entries, one entry per lane, and a step is one
// multiply-add per tile of the rows in use, a_ij -= (w_i / d) w_j with w the pivot's column in
// shared memory.  The step's other FP64 work is the reciprocal (3), the scaling of w and the
// entering node's couplings and loads (about 6).  The entering node usually takes the pivot's
// slot in the same step.
// One warp per element while the triangle fits its registers (M <= 64).  Larger fronts take
// WR x WC warps: warp (r, c) owns rows 4 r .. 4 r + 3 and columns 8 c .. 8 c + 7 of every
// 4 WR x 8 WC block, so which of its registers hold a row or a column is known at compile
// time up to the block's index; a further warp prepares the entering rows.
#pragma once

#include <cmath>
#include <utility>

#include "front_plan.h"
#include "local_common.cuh"

namespace mhm {

// fn(integral_constant<int, 0>) .. fn(integral_constant<int, N - 1>): loops whose index must
// be a constant (entries of a register array).
template <class F, int... I>
__device__ __forceinline__ void static_for_seq(F&& fn, std::integer_sequence<int, I...>) {
    (fn(std::integral_constant<int, I>{}), ...);
}
template <int N, class F> __device__ __forceinline__ void static_for(F&& fn) {
    static_for_seq(fn, std::make_integer_sequence<int, N>{});
}

// fn(integral_constant<int, i>) for a run-time i in [LO, HI), by halving.
template <int LO, int HI, class F> __device__ __forceinline__ void static_select(int i, F&& fn) {
    if constexpr (HI - LO == 1) {
        fn(std::integral_constant<int, LO>{});
    } else {
        constexpr int M = (LO + HI) / 2;
        if (i < M) static_select<LO, M>(i, fn);
        else static_select<M, HI>(i, fn);
    }
}
// fn(0), fn(1), .. fn(n - 1) for a run-time n <= N, each index a constant.  The rest of the
// range hangs in one branch: under a loop of conditions the compiler issues every
// instruction with a predicate, and a switched-off FP64 instruction holds the scheduler for its 64 clocks too.
template <int I, int N, class F> __device__ __forceinline__ void static_upto(int n, F&& fn) {
    if constexpr (I < N) {
        if (n > I) {
            fn(std::integral_constant<int, I>{});
            static_upto<I + 1, N>(n, fn);
        }
    }
}

// The distribution of the triangle: AR rows of blocks of 4 WR x 8 WC entries.
template <int WR_, int WC_, int AR_>
struct FrontTiles {
    static constexpr int WR = WR_, WC = WC_, AR = AR_, NW = WR * WC;
    static constexpr int cols(int a) { return (4 * WR * a + 4 * WR - 1) / (8 * WC) + 1; }   // blocks of row a
    static constexpr int at(int a) { return a == 0 ? 0 : at(a - 1) + cols(a - 1); }
    static constexpr int NT = at(AR);        // entries per lane
    static constexpr int NB = cols(AR - 1);  // block columns
    static constexpr int rows = 4 * WR * AR;
    static constexpr int vec = (rows + 31) / 32 * 32;   // entries of a vector over the rows
    static constexpr int threads = NW == 1 ? 32 : 32 * (NW + 1);
    // first block row that holds entries of block column b
    static constexpr int first(int b) { return (8 * WC * b) / (4 * WR); }
};
// Shared memory of one element (F values): pivot column, scaled pivot column and entering row (two of
// each, used in turn), a row of zeros, the inverse pivots and the pivots' couplings.
template <class F>
struct FrontShared {
    F *w[2], *s[2], *nb[2], *zero, *piv;
};
__host__ __device__ constexpr size_t front_shared_values(int vec) { return 7 * (size_t)vec + 4; }
template <class F>
__device__ __forceinline__ FrontShared<F> front_shared(F* base, int v) {
    FrontShared<F> f;
    for (int k = 0; k < 2; ++k) f.w[k] = base + k * v, f.s[k] = base + (2 + k) * v, f.nb[k] = base + (4 + k) * v;
    f.zero = base + 6 * v;
    f.piv = base + 7 * v;   // inverse pivot per parity; then the pivot's coupling with the entering node
    return f;
}

// 1 / d for 2^-1022 <= |d| < 2^1021 (the estimate flushes subnormals, d or 1 / d): one step of the
// hyperpower iteration of order three (M. Altman, Pacific J. Math. 10, 1960), y (1 + e + e^2)
// with e = 1 - d y, from the hardware's estimate y.  The estimate reads and gives 20 bits of
// mantissa, so |e| <= 2^-19; 1 / d = y (1 + e + e^2 + e^3 + ..), so the step leaves out 2^-57, a
// sixteenth of an ulp at most, and with its roundings ends within 0.57 ulp: the division's value or
// the one next to it.  Three FP64 instructions after the estimate.
__device__ __forceinline__ double front_rcp(double d) {
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
    const double e = fma(-d, y, 1.0), t = fma(e, e, e);
    return fma(t, y, y);
}

__device__ __forceinline__ float front_rcp(float d) { return 1.0f / d; }

// d positive and where front_rcp holds (a double by its high word: no FP64 instruction)
__device__ __forceinline__ bool front_positive(double d) {
    return (unsigned)__double2hiint(d) - 0x00100000u < 0x7fc00000u - 0x00100000u;
}
__device__ __forceinline__ bool front_positive(float d) { return d > 0.0f && d < INFINITY; }

// Power of two by which an element's matrix is scaled, from the high words of its largest and
// smallest positive kappa.  1 unless one of them is beyond 2^+-900; then the largest goes to 2^800 (by
// 2^1000 at most), so that every pivot and its reciprocal stay normal numbers for a contrast of up to
// about 2^1700 (front_rcp takes 2^-1022 to 2^1021, and a pivot is a few kappa).  The loads are not
// scaled: what the border is left with has to be multiplied by the scale.  Exact, so results do
// not depend on it.  Returned as the exponent, so that asking for 0 takes no FP64 instruction.
__device__ __forceinline__ int front_scale(int kmax, int kmin) {
    const int emax = (kmax >> 20) - 1023, emin = (kmin >> 20) - 1023;
    return kmax < 0 || (emax <= 900 && emin >= -900) ? 0 : min(1000, 800 - emax);
}
__device__ __forceinline__ double exp2_of(int e) { return __hiloint2double((1023 + e) << 20, 0); }

template <int NW> __device__ __forceinline__ void front_sync() {
    if (NW == 1) __syncwarp();
    else __syncthreads();
}

// The elimination.  T: FrontTiles.  ev: the step table (front_plan.h).
// prob.prep(e, ev[e], nb, wnew) is called by one warp for every step in order: it fills nb
// (T::vec entries) with the row of step e's entering node against the loads and the front
// as the step leaves it, zero elsewhere, and *wnew with its coupling to the pivot.  keep (NULL: none) gets the scaled
// pivot column of every step, `stride` values apart, and kinv (NULL: none) the inverse pivots;
// both start at step e0, the first that has a pivot.  *bad: 1 if a pivot was not positive.
// A: the entries; the result is read with front_result.  All warps of the element call it;
// starts and ends with a barrier.
template <class T, class F, class Prob>
__device__ __forceinline__ void front_eliminate(Prob& prob, const int4* __restrict__ ev, int steps, int R,
                                                const FrontShared<F>& sh, F (&A)[T::NT], int* bad, F* keep, int stride,
                                                F* kinv = nullptr, int e0 = 0) {
    constexpr int WR = T::WR, WC = T::WC, NW = T::NW, AR = T::AR;
    const int tid = NW == 1 ? (int)(threadIdx.x & 31) : (int)threadIdx.x;
    const int warp = NW == 1 ? 0 : __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int row = 4 * (warp / WC) + (lane >> 3), col = 8 * (warp % WC) + (lane & 7);   // inside a block
#pragma unroll
    for (int q = 0; q < T::NT; ++q) A[q] = F(0);
    for (int t = tid; t < 7 * T::vec; t += T::threads) sh.w[0][t] = F(0);
    front_sync<NW>();
    int4 v = ev[0];
    if (NW > 1 && warp == NW) {
        int4 vn = ev[steps > 1];
        prob.prep(0, v, sh.nb[0], sh.piv + 2);
        __syncthreads();
        for (int e = 0; e < steps; ++e) {
            const bool pivot = (v.x & 255) != kNoSlot;
            v = vn;
            if (e + 2 < steps) vn = ev[e + 2];
            if (e + 1 < steps) prob.prep(e + 1, v, sh.nb[(e + 1) & 1], sh.piv + 2 + ((e + 1) & 1));
            __syncthreads();
            if (pivot) __syncthreads();
        }
        __syncthreads();
        return;
    }
    if (NW == 1) prob.prep(0, v, sh.nb[0], sh.piv + 2);
    front_sync<NW>();
    for (int e = 0; e < steps; ++e) {
        const int par = e & 1;
        const int ps = v.x & 255, zs = (v.x >> 8) & 255, mm = R + ((v.x >> 16) & 255);
        if (e + 1 < steps) v = ev[e + 1];
        const int P = ps == kNoSlot ? -1 : R + ps, Z = zs == kNoSlot ? -1 : R + zs;
        F* w = sh.w[par];
        F* s = sh.s[par];
        const F* nb = sh.nb[par];
        // the pivot's row and column to w, then those of the entering node from nb (a slot
        // left free goes to zero and stays there)
        auto cross = [&](int X, auto&& fn) {   // fn(entry, other index) on row and column X
            static_select<0, AR>(X / (4 * WR), [&](auto ca) {
                constexpr int a = ca;
                if (X - row == 4 * WR * a)
                    static_for<T::cols(a)>([&](auto cb) {
                        constexpr int b = cb;
                        if (8 * WC * b + col <= X) fn(A[T::at(a) + b], 8 * WC * b + col);
                    });
            });
            static_select<0, T::NB>(X / (8 * WC), [&](auto cb) {
                constexpr int b = cb;
                if (X - col == 8 * WC * b)
                    static_for<AR - T::first(b)>([&](auto ca) {
                        constexpr int a = ca + T::first(b);
                        const int i = 4 * WR * a + row;
                        if (a > T::first(b) + 2 * WC / WR || i > X) fn(A[T::at(a) + b], i);
                    });
            });
        };
        if (P >= 0) {
            const F* in = Z == P ? nb : sh.zero;
            F d = F(0);
            bool own = false;   // this lane holds the pivot
            cross(P, [&](F& x, int k) {
                w[k] = x;
                if (NW > 1 && k == P) d = x, own = true;
                x = in[k];
            });
            // (outside the row's loop: there the reciprocal would be issued for every entry)
            if (NW > 1 && own) {
                if (!front_positive(d)) *bad = 1;
                sh.piv[par] = front_rcp(d);
            }
        }
        if (Z >= 0 && Z != P) cross(Z, [&](F& x, int k) { x = nb[k]; });
        front_sync<NW>();
        F inv = F(0);
        if (NW == 1 && P >= 0) {   // (read by all lanes before w[P] changes)
            const F d = w[P];
            if (!front_positive(d)) *bad = 1;
            inv = front_rcp(d);
        }
        if (NW == 1 && e + 1 < steps) prob.prep(e + 1, v, sh.nb[par ^ 1], sh.piv + 2 + (par ^ 1));
        if (NW == 1) __syncwarp();
        if (P >= 0) {
            const F wnew = sh.piv[2 + par];
            if (NW > 1) inv = sh.piv[par];
            // whole blocks: rows past the ones in use get zeros
            const int top = (mm + 8 * WC - 1) / (8 * WC) * (8 * WC);
            for (int q = tid; q < top; q += 32 * NW) {
                F x = q == Z ? wnew : (q == P || q >= mm) ? F(0) : w[q];
                if (q == Z || q == P || q >= mm) w[q] = x;
                x *= inv;
                s[q] = x;
                if (keep && q < mm) keep[(size_t)(e - e0) * stride + q] = x;
            }
            if (kinv && tid == 0) kinv[e - e0] = inv;
        }
        if (NW == 1 || P >= 0) front_sync<NW>();
        if (P >= 0) {
            F wb[T::NB];
            static_for<T::NB>([&](auto b) { wb[b] = 8 * WC * b < mm ? w[8 * WC * b + col] : F(0); });
            // rows of blocks with this warp's rows in use
            static_upto<0, AR>((mm - 4 * (warp / WC) + 4 * WR - 1) / (4 * WR), [&](auto ca) {
                constexpr int a = ca;
                const F sa = s[4 * WR * a + row];
                static_for<T::cols(a)>([&](auto cb) {
                    constexpr int b = cb;
                    A[T::at(a) + b] = fma(-sa, wb[b], A[T::at(a) + b]);
                });
            });
        }
    }
    front_sync<NW>();
}

// Calls fn(i, j, value) for this thread's entries i >= j of the leading R x R block.
template <class T, class Fn>
__device__ __forceinline__ void front_result(int R, const double (&A)[T::NT], Fn&& fn) {
    const int tid = T::NW == 1 ? (int)(threadIdx.x & 31) : (int)threadIdx.x, warp = tid >> 5, lane = tid & 31;
    if (warp >= T::NW) return;
    const int row = 4 * (warp / T::WC) + (lane >> 3), col = 8 * (warp % T::WC) + (lane & 7);
    static_for<T::AR>([&](auto ca) {
        constexpr int a = ca;
        if (4 * T::WR * a < R)
            static_for<T::cols(a)>([&](auto cb) {
                constexpr int b = cb;
                const int i = 4 * T::WR * a + row, j = 8 * T::WC * b + col;
                if (i < R && j <= i) fn(i, j, A[T::at(a) + b]);
            });
    });
}

// Entering rows of the 2-D local problems (FrontPlan's tables): couplings from kappa and the
// two element matrices, ahead of their use by one batch of 32 / ncp steps (loads of the batch
// after it in flight).  load.node(info), then load(x, y, info,
// column) gives the node's load (info: mass count | faces << 8).  The pinned
// node is kept as a node coupled to nothing, with a unit pivot and no loads.
template <int NCP, class Load>
struct FrontRows2D {
    static constexpr int B = 32 / NCP;
    const uint2* cp;
    const double* kap;
    const double* Ke;
    int steps, R, vec, pin;   // vec: entries of a row; pin: lattice point x | y << 16
    Load load;
    int pin_slot = -1;
    uint2 cur, nxt, far;
    double val = 0.0, diag = 0.0, k0 = 0.0, k1 = 0.0;

    __device__ __forceinline__ uint2 entry(int batch) const {
        const int lane = threadIdx.x & 31, e = batch * B + lane / NCP;
        return e < steps ? cp[(size_t)e * NCP + lane % NCP] : make_uint2(kNoSlot, 0xffff0000u);
    }
    __device__ __forceinline__ void fetch(uint2 q) {
        const uint32_t t1 = q.y >> 16;
        const bool any = (q.x & 255) != kNoSlot;
        k0 = any ? kap[q.y & 0xffff] : 0.0;
        k1 = any && t1 != 0xffff ? kap[t1] : 0.0;
    }
    __device__ __forceinline__ void start() {
        nxt = entry(0);
        fetch(nxt);
        far = entry(1);
    }
    __device__ __forceinline__ void prep(int e, const int4& v, double* nb, double* wnew) {
        const int lane = threadIdx.x & 31, sub = lane % NCP;
        if (e % B == 0) {
            cur = nxt;
            val = fma(k1, Ke[(cur.x >> 16) & 255], k0 * Ke[(cur.x >> 8) & 255]);
            diag = val + __shfl_down_sync(0xffffffffu, val, 1) + __shfl_down_sync(0xffffffffu, val, 2);
            nxt = far;
            fetch(nxt);
            far = entry(e / B + 2);
        }
        const int ps = v.x & 255, zs = (v.x >> 8) & 255;
        if (zs != kNoSlot) {
            const bool pinned = v.y == pin;
            load.node(v.z);
            for (int q = lane; q < vec; q += 32) nb[q] = q < R && !pinned ? load(v.y & 0xffff, v.y >> 16, v.z, q) : 0.0;
            if (lane == 0) *wnew = 0.0;
            __syncwarp();
            if (lane / NCP == e % B) {
                const int sl = cur.x & 255;
                if (sub == NCP - 3) nb[R + zs] = pinned ? 1.0 : diag;
                else if (sl < kDiagSlot && !pinned && sl != pin_slot) nb[R + sl] = val;
                else if (sl == kPivotSlot && !pinned && ps != pin_slot) *wnew = val;
            }
            if (ps == pin_slot && ps != kNoSlot) pin_slot = -1;
            if (pinned) pin_slot = zs;
        } else if (ps == pin_slot && ps != kNoSlot) {
            pin_slot = -1;
        }
    }
};

}  // namespace mhm
