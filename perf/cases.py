"""The work that users of this package have it do, as cases that can be timed and checked:
local solves + skeleton gather of the 2-D pipeline (FP64 and mixed, P1 and P2, one level for
all elements or a level per element), the global solve, the reconstruction, and the 3-D
local solves + skeleton gather.

`listed()` names the cases, `draw(rng)` gives more of the same ranges, `prepare` makes the
inputs and the objects a program keeps, `run` is one pass, `work` what it cannot do without,
and `exact` the same outputs from plain numpy / torch in 64 bits (block elimination over
lattice rows with the zero row sums of the Neumann matrix restored at every level; dense
Cholesky for the tetrahedra; a dense LU for small skeleton systems)."""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_1703_10435_gb300 import mhm
from paper_1703_10435_gb300 import workloads as W
from paper_1703_10435_gb300.pipeline import Pipeline

F64 = torch.float64
DEV = "cuda" if torch.cuda.is_available() else "cpu"


# ------------------------------------------------------------------------------ the cases

def listed():
    return [
        # the first problem anybody runs: 32 coarse triangles, 45 DOFs each; latency only
        dict(name="step_p1_tiny_fp64", kind="step", nx=4, ny=4, r=3, degree=1, m=1, l=1,
             precision="fp64", source="sinsin", field="uniform", decades=0.5),
        # an ordinary heterogeneous problem, all FP64: 2048 elements, contrast 1e4 per triangle
        dict(name="step_p1_r5_fp64", kind="step", nx=32, ny=32, r=5, degree=1, m=2, l=2,
             precision="fp64", source="const", field="uniform", decades=2.0),
        # a ragged, odd-sized mesh at a coarser level in mixed precision, f given by values
        dict(name="step_p1_r4_ragged_mixed", kind="step", nx=37, ny=23, r=4, degree=1, m=1, l=2,
             precision="mixed", source="quad", field="grf", decades=2.0),
        # the benchmark's own workload: 32768 elements, mixed precision, random field
        dict(name="step_p1_r5_mixed", kind="step", nx=128, ny=128, r=5, degree=1, m=2, l=2,
             precision="mixed", source="const", field="grf", decades=2.0),
        # quadratic elements in mixed precision, contrast 1e6 (a quarter of the large instance)
        dict(name="step_p2_r4_mixed", kind="step", nx=128, ny=128, r=4, degree=2, m=3, l=1,
             precision="mixed", source="sinsin", field="grf", decades=3.0),
        # quadratic elements all in FP64
        dict(name="step_p2_r4_fp64", kind="step", nx=56, ny=40, r=4, degree=2, m=3, l=1,
             precision="fp64", source="const", field="grf", decades=3.0),
        # channels of 1e3 times the background: a level (3..7) per element and a multiplier degree
        # per face, mixed (at 1e4 the result itself is only fixed to about 1e-9 in 64 bits)
        dict(name="levels_mixed", kind="levels", nx=64, ny=64, precision="mixed", field_seed=0, channels=16),
        # the same in FP64 on a coarser T_H
        dict(name="levels_fp64", kind="levels", nx=40, ny=40, precision="fp64", field_seed=0, channels=10),
        # the skeleton's saddle-point system of the benchmark's mesh (0.33 M unknowns)
        dict(name="global_128", kind="global", nx=128, ny=128, m=2, l=2, decades=1.0),
        # u on every submesh of that mesh from its multipliers
        dict(name="reconstruct_p1_r5", kind="reconstruct", nx=128, ny=128, r=5, degree=1, m=2, l=2,
             source="const", field="grf", decades=2.0),
        # the paper's own experiment in 3-D: 12288 tetrahedra, m = 4, mixed precision
        dict(name="cube_m4_mixed", kind="cube", nc=8, r=2, degree=2, m=4, precision="mixed",
             source="sinsinsin", decades=1.0),
        # its finer multiplier space, m = 16, all FP64
        dict(name="cube_m16_fp64", kind="cube", nc=4, r=2, degree=2, m=16, precision="fp64",
             source="sinsinsin", decades=1.0),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _grid(rng, lo, hi):
    """nx, ny with nx ny spread over [lo, hi] on a log scale, not square in general."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    a = math.exp(rng.uniform(-0.7, 0.7))
    nx = max(2, int(round(math.sqrt(n * a))))
    return nx, max(2, min(int(round(n / nx)), hi // nx))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "levels", "global", "reconstruct", "cube", "cube"])
    if kind in ("step", "reconstruct"):
        degree = rng.choice([1, 1, 2])
        r = rng.choice([3, 4, 5]) if degree == 1 else rng.choice([2, 3, 4])
        space = [(1, 0), (1, 1), (2, 0), (1, 2), (2, 1), (3, 1), (2, 2), (1, 3)]
        m, l = rng.choice([s for s in space if 2 * s[0] * (s[1] + 1) <= degree << r])
        nx, ny = _grid(rng, 16, 16384 if degree == 1 else 8192)
        c = dict(kind=kind, nx=nx, ny=ny, r=r, degree=degree, m=m, l=l)
        if kind == "step":
            c["precision"] = rng.choice(["fp64", "mixed"])
        c["source"] = rng.choice(["const", "const", "sinsin"] + (["quad"] if nx * ny <= 4096 else []))
        c["field"] = rng.choice(["uniform", "grf"])
        c["decades"] = round(rng.uniform(0.5, 2.0 if c["field"] == "uniform" else 3.0), 3)
        return c
    if kind == "levels":
        nx, ny = _grid(rng, 64, 1600)
        return dict(kind=kind, nx=nx, ny=ny, precision=rng.choice(["fp64", "mixed"]),
                    field_seed=rng.randrange(1000), channels=rng.randint(4, 10))
    if kind == "global":
        nx, ny = _grid(rng, 16, 16384)
        m, l = rng.choice([(1, 1), (2, 1), (1, 2), (2, 2), (3, 1)])
        return dict(kind=kind, nx=nx, ny=ny, m=m, l=l, decades=round(rng.uniform(0.2, 2.0), 3))
    degree, r, m = rng.choice([(2, 2, 4), (2, 2, 4), (2, 2, 1), (2, 2, 16), (2, 1, 4), (2, 1, 1), (1, 3, 4), (1, 2, 4),
                               (1, 2, 1)])
    nc = _log_int(rng, 1, 8 if m < 16 else 4)
    return dict(kind=kind, nc=nc, r=r, degree=degree, m=m, precision=rng.choice(["fp64", "mixed"]),
                source=rng.choice(["const", "sinsinsin"]), decades=round(rng.uniform(0.3, 1.5), 3))


# ------------------------------------------------------------------------ inputs and passes

def _gen(seed, device=DEV):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _centroid_lattice(N):
    return torch.as_tensor(W.fine_centroid_lattice(N) / N)


def _verts(nx, ny):
    """(n_K, 3, 2) vertices of the coarse triangles."""
    j, i = np.divmod(np.arange(nx * ny), nx)
    p = lambda a, b: np.stack([(i + a) / nx, (j + b) / ny], -1)
    lo, up = np.stack([p(0, 0), p(1, 0), p(1, 1)], 1), np.stack([p(0, 0), p(1, 1), p(0, 1)], 1)
    return np.stack([lo, up], 1).reshape(-1, 3, 2)


def _field(c, seed, device=DEV):
    """kappa, n_K x 4^r: 10^U per fine triangle, or an exponentiated random Fourier field of
    correlation length 0.02 at the fine centroids."""
    n_K, N, g = 2 * c["nx"] * c["ny"], 1 << c["r"], _gen(seed)
    if c["field"] == "uniform":
        e = torch.rand(n_K, N * N, generator=g, device=DEV, dtype=F64) * 2 - 1
        return (10.0 ** (c["decades"] * e)).to(device)
    F = 64
    om = torch.randn(2, F, generator=g, device=DEV) / 0.02
    ph = torch.rand(F, generator=g, device=DEV) * 2 * math.pi
    verts, lat = torch.as_tensor(_verts(c["nx"], c["ny"]), device=DEV), _centroid_lattice(N).to(DEV)
    out = torch.empty(n_K, N * N, dtype=F64, device=DEV)
    step = max(1, (1 << 21) // (N * N))
    for a in range(0, n_K, step):
        v = verts[a:a + step]
        xy = v[:, :1] + lat[None, :, :1] * (v[:, 1:2] - v[:, :1]) + lat[None, :, 1:] * (v[:, 2:] - v[:, :1])
        x, y = xy[..., 0].float(), xy[..., 1].float()
        s = torch.zeros_like(x)
        for k in range(F):
            s += torch.cos(x * om[0, k] + y * om[1, k] + ph[k])
        out[a:a + step] = 10.0 ** (c["decades"] * torch.clamp(s.double() * math.sqrt(2.0 / F) / 3.0, -1, 1))
    return out.to(device)


def _quad_fn(x, y):
    return torch.exp(x) * torch.cos(3 * y) + 1.0 / (1.0 + x + y)


_DUFFY = None


def _duffy():
    """(16, 2) points and (16,) weights of the collapsed 4 x 4 Gauss rule."""
    global _DUFFY
    if _DUFFY is None:
        a, w = np.polynomial.legendre.leggauss(4)
        a, w = 0.5 * (a + 1), 0.5 * w
        _DUFFY = (np.array([(a[i], a[j] * (1 - a[i])) for i in range(4) for j in range(4)]),
                  np.array([w[i] * w[j] * (1 - a[i]) for i in range(4) for j in range(4)]))
    return _DUFFY


def _source_points(v, N):
    """Physical positions (B, N^2, 16, 2) of the source points of coarse triangles v (B, 3, 2)."""
    lat = torch.as_tensor(W.fine_triangle_lattice(N) / N, device=v.device)
    ref = torch.as_tensor(_duffy()[0], device=v.device)
    b = lat[:, 0, None] + ref[None, :, :1] * (lat[:, 1] - lat[:, 0])[:, None] + ref[None, :, 1:] * (lat[:, 2] - lat[:, 0])[:, None]
    return v[:, 0, None, None] + b[None, ..., :1] * (v[:, 1] - v[:, 0])[:, None, None] + b[None, ..., 1:] * (v[:, 2] - v[:, 0])[:, None, None]


def _source(c, state):
    if c["source"] == "const":
        return mhm.Source(mhm.MHM_SRC_CONST, 1.0, 1.0)
    if c["source"] == "sinsin":
        return mhm.Source(mhm.MHM_SRC_SINSIN, 1.0, 2.0)
    N = 1 << c["r"]
    verts = torch.as_tensor(_verts(c["nx"], c["ny"]), device=DEV)
    vals = torch.empty(verts.shape[0], N * N, 16, dtype=F64, device=DEV)
    step = max(1, (1 << 20) // (N * N))
    for a in range(0, verts.shape[0], step):
        p = _source_points(verts[a:a + step], N)
        vals[a:a + step] = _quad_fn(p[..., 0], p[..., 1])
    state["values"] = vals
    return mhm.quad_source(vals.view(-1))


def _levels_of(c):
    """Refinement level of every K: by the distance of its centroid to the nearest channel."""
    f = W.ChannelField(c["field_seed"], n_channels=c["channels"])
    d, H = f.distance(_verts(c["nx"], c["ny"]).mean(1)), 1.0 / c["nx"]
    r = np.full(d.shape, 3, dtype=np.int8)
    for t, lev in ((4 * H, 4), (2 * H, 5), (H, 6), (0.5 * H, 7)):
        r[d < t] = lev
    return r


def _levels_kappa(c, seed):
    """kappa per K and fine triangle, flat: a background value and a value per channel (up to
    1e3 times it), both from the seed; and the first value of every K."""
    f, g = W.ChannelField(c["field_seed"], n_channels=c["channels"]), _gen(seed)
    rk, verts = _levels_of(c), torch.as_tensor(_verts(c["nx"], c["ny"]), device=DEV)
    bg = float(torch.rand((), generator=g, device=DEV, dtype=F64) * 0.5 + 0.75)
    hi = 1e3 * (torch.rand(f.n_channels, generator=g, device=DEV, dtype=F64) * 0.5 + 0.5)
    pt, dr = torch.as_tensor(f.points, device=DEV), torch.as_tensor(f.dirs, device=DEV)
    off = np.concatenate([[0], np.cumsum(4 ** rk.astype(np.int64))])
    out = torch.empty(int(off[-1]), dtype=F64, device=DEV)
    for r in sorted(set(rk.tolist())):
        N, Ks = 1 << r, np.nonzero(rk == r)[0]
        lat, step = _centroid_lattice(N).to(DEV), max(1, (1 << 21) // (N * N))
        for a in range(0, len(Ks), step):
            k = torch.as_tensor(Ks[a:a + step], device=DEV)
            v = verts[k]
            xy = v[:, :1] + lat[None, :, :1] * (v[:, 1:2] - v[:, :1]) + lat[None, :, 1:] * (v[:, 2:] - v[:, :1])
            near = torch.full(xy.shape[:2], math.inf, dtype=F64, device=DEV)
            val = torch.full_like(near, bg)
            for q in range(f.n_channels):
                d = ((xy[..., 1] - pt[q, 1]) * dr[q, 0] - (xy[..., 0] - pt[q, 0]) * dr[q, 1]).abs()
                val = torch.where((d < near) & (d <= f.half_width), hi[q], val)
                near = torch.minimum(near, d)
            at = torch.as_tensor(off[Ks[a:a + step]], device=DEV)[:, None] + torch.arange(N * N, device=DEV)
            out[at.reshape(-1)] = val.reshape(-1)
    return out, off


def _precision(c):
    return mhm.MHM_MIXED if c["precision"] == "mixed" else mhm.MHM_FP64


def prepare(case, seed):
    c, st = case, {"kind": case["kind"], "f": case.get("source", "const") != "const"}
    if c["kind"] == "step":
        st["pipe"] = Pipeline(c["nx"], c["ny"], c["r"], c["degree"], c["m"], c["l"], 0, _precision(c))
        st["kappa"], st["source"] = _field(c, seed), _source(c, st)
    elif c["kind"] == "levels":
        rk = _levels_of(c)
        lf = _face_degrees(c, rk)
        st["pipe"] = Pipeline(c["nx"], c["ny"], 3, 1, 1, 3, 0, _precision(c), rk, lf)
        st["kappa"], st["source"] = _levels_kappa(c, seed)[0], mhm.Source(mhm.MHM_SRC_CONST, 1.0, 1.0)
    elif c["kind"] == "global":
        st["mesh"] = mhm.Mesh(c["nx"], c["ny"], 3, 1, c["m"], c["l"], 0)
        b = _global_blocks(c, seed)
        st["in"] = [t.to(DEV) for t in (b["A_vals"], b["E"], b["BK"], b["FK"])]
        st["lam"] = torch.empty(st["mesh"].n_lambda, dtype=F64, device=DEV)
        st["u0"] = torch.empty(st["mesh"].n_K, dtype=F64, device=DEV)
    elif c["kind"] == "reconstruct":
        M = st["mesh"] = mhm.Mesh(c["nx"], c["ny"], c["r"], c["degree"], c["m"], c["l"], 0)
        st["kappa"], st["source"] = _field(c, seed), _source(c, st)
        st["lam"], st["u0"] = (t.to(DEV) for t in _multipliers(c, seed))
        st["u"] = torch.empty(int(M.nodal_offset[-1]), dtype=F64, device=DEV)
    else:
        M = st["mesh"] = mhm.Mesh3D(c["nc"], c["r"], c["degree"], c["m"], 0)
        st["precision"] = _precision(c)
        st["kappa"], st["source"] = _cube_kappa(c, seed), _cube_source(c)
        z = lambda *s: torch.zeros(*s, dtype=F64, device=DEV)
        st["out"] = dict(AK=z(M.n_K, M.n_I, M.n_I), EK=z(M.n_K, M.n_I), BK=z(M.n_K, M.n_I), FK=z(M.n_K),
                         status=torch.zeros(M.n_K, dtype=torch.int32, device=DEV), A_vals=z(M.nnz), E=z(M.n_lambda))
    return st


def run(state):
    if state["kind"] in ("step", "levels"):
        p = state["pipe"]
        p.step(state["kappa"], state["source"])
        return _results(state, dict(AK=p.AK, EK=p.EK, BK=p.BK, FK=p.FK, status=p.status, A_vals=p.A_vals, E=p.E))
    if state["kind"] == "global":
        mhm.mhm_solve_global(state["mesh"], *state["in"], state["lam"], state["u0"])
        return dict(lam=state["lam"], u0=state["u0"])
    if state["kind"] == "reconstruct":
        mhm.mhm_reconstruct(state["mesh"], state["kappa"], state["source"], state["lam"], state["u0"], None, state["u"])
        return dict(u=state["u"])
    o = state["out"]
    mhm.mhm3d_local_solve_batch(state["mesh"], state["kappa"], state["source"], o["AK"], o["EK"], o["BK"], o["FK"],
                                o["status"], precision=state["precision"])
    mhm.mhm3d_assemble_skeleton(state["mesh"], o["AK"], o["EK"], o["A_vals"], o["E"])
    return _results(state, o)


def _results(state, o):
    """A constant f is its own mean, so its compatible load, eta_f, E_K and E vanish: what is
    computed for them is rounding alone, and no result."""
    return {k: v for k, v in o.items() if state["f"] or k not in ("EK", "E")}


# ------------------------------------------------------------------------------ the work

def _elimination_fmas(P, N, R):
    """Multiply-adds of one element's block elimination by lattice levels with R loads:
    factor, coupling, Schur update, forward solve, its update, and the products of the loads."""
    PN, tot = P * N, 0.0
    size = lambda lev: sum(PN + 1 - j for j in range(P * lev, min(P * lev + P, PN + 1)))
    for lev in range(N + 1):
        b, bn = size(lev), size(lev + 1) if lev < N else 0
        tot += b ** 3 / 6 + bn * b * b / 2 + b * bn * bn / 2 + R * b * b / 2 + bn * R * b + b * R * R / 2
    return tot


def _dissection_flops(w, h, s):
    """Dense flops of a nested dissection of a w x h block of squares, s unknowns per face."""
    if w * h <= 4:
        f = s * (3 * w * h + w + h) + 2 * w * h
        return f ** 3 / 3
    a, b = max(w, h), min(w, h)
    sep, front = s * b, s * (b + 2 * (w + h))
    k = min(sep, front)
    own = 2 * (k ** 3 / 6 + k * k * (front - k) / 2 + k * (front - k) ** 2 / 2)
    return own + _dissection_flops(a // 2, b, s) + _dissection_flops(a - a // 2, b, s)


def work(case):
    c = case
    if c["kind"] == "cube":
        n = (c["degree"] << c["r"]) + 1
        n, NI, n_K = n * (n + 1) * (n + 2) // 6, 4 * c["m"], 24 * c["nc"] ** 3
        nf = 2 * n_K + 12 * c["nc"] ** 2
        nnz = (16 * n_K - (4 * n_K - nf)) * c["m"] ** 2
        by = 8 * n_K * (8 ** c["r"] + NI * NI + 2 * NI + 1.5) + 8 * (nnz + nf * c["m"])
        return {"bytes": by, "flops": 2.0 * n_K * (n ** 3 / 6 + n * n * (NI + 1) / 2 + n * NI * NI / 2)}
    nx, ny = c["nx"], c["ny"]
    n_K, nf = 2 * nx * ny, nx * (ny + 1) + ny * (nx + 1) + nx * ny
    if c["kind"] == "levels":
        rk, d = _levels_of(c).astype(int), 4
        fl = 2.0 * sum(_elimination_fmas(1, 1 << r, 3 * d + 1) * int((rk == r).sum()) for r in set(rk.tolist()))
        fine = int((4 ** rk.astype(np.int64)).sum())
    elif c["kind"] == "global":
        d, fine, fl = c["m"] * (c["l"] + 1), 0, float(_dissection_flops(nx, ny, c["m"] * (c["l"] + 1)))
    else:
        d, N = c["m"] * (c["l"] + 1), 1 << c["r"]
        R = 1 if c["kind"] == "reconstruct" else 3 * d + 1
        fine, fl = n_K * N * N * (17 if c["source"] == "quad" else 1), 2.0 * n_K * _elimination_fmas(c["degree"], N, R)
    NI, nnz = 3 * d, (9 * n_K - (3 * n_K - nf)) * d * d
    if c["kind"] == "global":
        return {"bytes": 8.0 * (nnz + 2 * nf * d + n_K * (NI + 2)), "flops": fl}
    if c["kind"] == "reconstruct":
        PN = c["degree"] << c["r"]
        return {"bytes": 8.0 * (fine + nf * d + n_K * (1 + (PN + 1) * (PN + 2) // 2)), "flops": fl}
    return {"bytes": 8.0 * (fine + n_K * (NI * NI + 2 * NI + 1.5) + nnz + nf * d), "flops": fl}


# ------------------------------------------------- the same in plain 64-bit numpy and torch

def _coarse(nx, ny):
    """(tri_faces n_K x 3, signs n_K x 3, n_faces): faces numbered by first encounter, local
    face a opposite vertex a; sign of the outward normal against the face's."""
    j, i = np.divmod(np.arange(nx * ny), nx)
    v = lambda a, b: (j + b) * (nx + 1) + i + a
    tri = np.stack([np.stack([v(0, 0), v(1, 0), v(1, 1)], 1), np.stack([v(0, 0), v(1, 1), v(0, 1)], 1)], 1).reshape(-1, 3)
    a, b = tri[:, [1, 2, 0]], tri[:, [2, 0, 1]]
    key = (np.minimum(a, b).astype(np.int64) * ((nx + 1) * (ny + 1)) + np.maximum(a, b)).ravel()
    u, first, inv, cnt = np.unique(key, return_index=True, return_inverse=True, return_counts=True)
    rank = np.empty(len(u), dtype=np.int64)
    rank[np.argsort(first)] = np.arange(len(u))
    inv = inv.reshape(-1)
    boundary = (cnt[inv] == 1).reshape(-1, 3)
    return rank[inv].reshape(-1, 3), np.where(boundary | (a < b), 1, -1), len(u)


def _face_degrees(c, rk):
    tf, _, nf = _coarse(c["nx"], c["ny"])
    rmax = np.zeros(nf, dtype=np.int64)
    np.maximum.at(rmax, tf.ravel(), np.repeat(rk.astype(np.int64), 3))
    return W.face_degree_from_levels(rmax)


def _face_table(PN, P, m, l):
    """(m (l+1), PN+1): integrals over [0, 1] of the multiplier basis times the face nodes' basis."""
    N = PN // P
    T = np.zeros((m * (l + 1), PN + 1))
    cuts = sorted({i / N for i in range(N + 1)} | {q / m for q in range(m + 1)})
    x, w = np.polynomial.legendre.leggauss((P + l) // 2 + 2)
    for a, b in zip(cuts[:-1], cuts[1:]):
        if b - a < 1e-13:
            continue
        s = a + (b - a) * 0.5 * (x + 1)
        e, q = min(N - 1, int((a + b) / 2 * N)), min(m - 1, int((a + b) / 2 * m))
        t = s * N - e
        phi = [1 - t, t] if P == 1 else [(1 - t) * (1 - 2 * t), 4 * t * (1 - t), t * (2 * t - 1)]
        xi = 2 * (s * m - q) - 1
        for p in range(l + 1):
            psi = np.polynomial.legendre.Legendre.basis(p)(xi)
            for k, f in enumerate(phi):
                T[q * (l + 1) + p, P * e + k] += 0.5 * (b - a) * (w * psi * f).sum()
    return T


def _stiffness2(X, P):
    """Stiffness of the triangle X (3, 2), nodes: vertices, then midpoints of (0,1), (1,2), (2,0)."""
    J = np.stack([X[1] - X[0], X[2] - X[0]], 1)
    area, g = abs(np.linalg.det(J)) / 2, np.linalg.inv(J)
    G = np.stack([-g[0] - g[1], g[0], g[1]])
    if P == 1:
        return area * G @ G.T
    S = np.zeros((6, 6))
    for lam in ((.5, .5, 0), (0, .5, .5), (.5, 0, .5)):
        D = [(4 * lam[a] - 1) * G[a] for a in range(3)]
        D += [4 * (lam[a] * G[b] + lam[b] * G[a]) for a, b in ((0, 1), (1, 2), (2, 0))]
        D = np.array(D)
        S += area / 3 * D @ D.T
    return S


def _dof(PN, i, j):
    return j * (PN + 1) - j * (j - 1) // 2 + i


class _Local2:
    """Block elimination of the local Neumann problems of one level r, degree P."""

    def __init__(self, nx, ny, r, P, m, l, device):
        self.N, self.P, self.dev = 1 << r, P, device
        N, PN = self.N, P << r
        self.PN, self.n = PN, (PN + 1) * (PN + 2) // 2
        tri = W.fine_triangle_lattice(N).astype(int)
        nodes = [P * tri[:, a] for a in range(3)]
        if P == 2:
            nodes += [tri[:, a] + tri[:, b] for a, b in ((0, 1), (1, 2), (2, 0))]
        self.dofs = np.stack([_dof(PN, p[:, 0], p[:, 1]) for p in nodes], 1)
        self.row = tri[:, :, 1].min(1)
        V = _verts(nx, ny)[:2]
        down = (tri[:, 0, 0] != tri[:, 2, 0]).astype(int)
        self.Ke = np.zeros((2, 2, self.dofs.shape[1], self.dofs.shape[1]))
        for par in range(2):
            e1, e2 = (V[par, 1] - V[par, 0]) / N, (V[par, 2] - V[par, 0]) / N
            for d, X in enumerate(([0 * e1, e1, e2], [e1, e1 + e2, e2])):
                self.Ke[par, d] = _stiffness2(np.array(X), P)
        self.down = down
        self.areaK = 0.5 / (nx * ny)
        at = self.areaK / (N * N)
        per = np.full(3, at / 3) if P == 1 else np.array([0, 0, 0] + [at / 3] * 3)
        self.mass = np.zeros(self.n)
        np.add.at(self.mass, self.dofs, np.broadcast_to(per, self.dofs.shape))
        # unsigned multiplier loads, per parity: -|F| int psi phi on the nodes of local face a
        T, d = _face_table(PN, P, m, l), m * (l + 1)
        corner = np.array([(0, 0), (1, 0), (0, 1)])
        self.load = np.zeros((2, 3 * d, self.n))
        for par in range(2):
            low_first = ((True, False, True), (False, False, True))[par]   # does v[a+1] have the lower id than v[a+2]?
            for a in range(3):
                p, q = (a + 1) % 3, (a + 2) % 3
                F = np.linalg.norm(V[par, q] - V[par, p])
                if not low_first[a]:
                    p, q = q, p
                ij = corner[p] * PN + np.arange(PN + 1)[:, None] * (corner[q] - corner[p])
                self.load[par, a * d:(a + 1) * d, _dof(PN, ij[:, 0], ij[:, 1])] -= F * T.T
        self.start = [_dof(PN, 0, min(P * lev, PN)) for lev in range(N + 1)] + [self.n]

    def source(self, c, verts):
        """(f, phi_w)_K for the elements with vertices verts (B, 3, 2)."""
        B, dev = verts.shape[0], self.dev
        if c["source"] == "const":
            return torch.as_tensor(self.mass, device=dev).expand(B, -1).clone()
        p = _source_points(verts, self.N)
        if c["source"] == "quad":
            f = _quad_fn(p[..., 0], p[..., 1])
        else:
            f = 2 * (2 * math.pi) ** 2 * torch.sin(2 * math.pi * p[..., 0]) * torch.sin(2 * math.pi * p[..., 1])
        pts, w = _duffy()
        lam = np.stack([1 - pts[:, 0] - pts[:, 1], pts[:, 0], pts[:, 1]], 1)
        phi = lam if self.P == 1 else np.concatenate(
            [lam * (2 * lam - 1)] + [(4 * lam[:, a] * lam[:, b])[:, None] for a, b in ((0, 1), (1, 2), (2, 0))], 1)
        area2 = 2 * self.areaK / self.N ** 2
        v = torch.einsum("btq,qa->bta", f, torch.as_tensor(phi * w[:, None] * area2, device=dev))
        out = torch.zeros(B, self.n, dtype=F64, device=dev)
        return out.index_add_(1, torch.as_tensor(self.dofs.ravel(), device=dev), v.reshape(B, -1))

    def solve(self, kappa, par, G, back=False):
        """G (B, n, R): (Gram of L^-1 g~, or with `back` the zero-mean solutions)."""
        B, R, dev, st = G.shape[0], G.shape[2], self.dev, self.start
        mass = torch.as_tensor(self.mass, device=dev)
        G = G - mass[None, :, None] * (G.sum(1, keepdim=True) / self.areaK)
        Ke = torch.as_tensor(self.Ke, device=dev)[par]
        gram, carry, kept = torch.zeros(B, R, R, dtype=F64, device=dev), None, []
        Gl = G[:, st[0]:st[1]]
        for lev in range(self.N):
            o, b, t = st[lev], st[lev + 1] - st[lev], st[lev + 2] - st[lev]
            el = np.nonzero(self.row == lev)[0]
            loc = self.dofs[el] - o
            wide = max(t, int(loc.max()) + 1)
            idx = torch.as_tensor((loc[:, :, None] * wide + loc[:, None, :]).ravel(), device=dev)
            vals = kappa[:, torch.as_tensor(el, device=dev), None, None] * Ke[:, torch.as_tensor(self.down[el], device=dev)]
            win = torch.zeros(B, wide * wide, dtype=F64, device=dev).index_add_(1, idx, vals.reshape(B, -1)).view(B, wide, wide)
            if carry is not None:
                win[:, :carry.shape[1], :carry.shape[1]] += carry
            S, C = win[:, :b, :b].clone(), win[:, b:t, :b]
            D = torch.diagonal(S, dim1=1, dim2=2)
            D -= S.sum(2) + C.sum(1)                       # rows of the Neumann matrix sum to zero
            L = torch.linalg.cholesky(S)
            Y = torch.linalg.solve_triangular(L, Gl, upper=False)
            X = torch.linalg.solve_triangular(L, C.transpose(1, 2), upper=False)
            gram += Y.transpose(1, 2) @ Y
            carry = win[:, b:t, b:t] - X.transpose(1, 2) @ X
            Gl = G[:, st[lev + 1]:st[lev + 2]] - X.transpose(1, 2) @ Y
            if back:
                kept.append((L, X, Y))
        if not back:
            return gram
        z = [torch.zeros(B, 1, R, dtype=F64, device=dev)]
        for L, X, Y in reversed(kept):
            z.append(torch.linalg.solve_triangular(L.transpose(1, 2), Y - X @ z[-1], upper=True))
        z = torch.cat(z[::-1], 1)
        return z - (mass[None, :, None] * z).sum(1, keepdim=True) / self.areaK

    def blocks(self, c, kappa, Ks, signs, device):
        """A_K, E_K, B_K, F_K of the elements Ks (all faces with the full multiplier space)."""
        par = torch.as_tensor(Ks % 2, device=device)
        NI = self.load.shape[1]
        s = torch.as_tensor(np.repeat(signs[Ks], NI // 3, axis=1).astype(float), device=device)
        N_ = torch.as_tensor(self.load, device=device)[par] * s[:, :, None]
        f = self.source(c, torch.as_tensor(_verts(c["nx"], c["ny"])[Ks], device=device))
        gram = self.solve(kappa, par, torch.cat([N_, f[:, None]], 1).transpose(1, 2))
        return -gram[:, :NI, :NI], gram[:, :NI, NI], -N_.sum(2), f.sum(1)


def _scatter(c, AK, EK, tf, deg):
    """Skeleton values in CSR order and right-hand side from the blocks; deg: multipliers per
    face (m (l_e + 1)), slots of stride N_I / 3."""
    NI, nf = AK.shape[1], len(deg)
    d = NI // tf.shape[1]
    off = np.concatenate([[0], np.cumsum(deg)])
    p = np.arange(d)
    gid = np.where(p[None, None, :] < deg[tf][..., None], off[tf][..., None] + p, -1).reshape(-1, NI)
    g = torch.as_tensor(gid, device=AK.device)
    ok = (g[:, :, None] >= 0) & (g[:, None, :] >= 0)
    n = int(off[-1])
    key = (g[:, :, None] * n + g[:, None, :])[ok]
    key, order = torch.sort(key, stable=True)
    vals = AK[ok][order]
    first = torch.ones_like(key, dtype=torch.bool)
    first[1:] = key[1:] != key[:-1]
    at = torch.nonzero(first).flatten()
    A = vals[at].clone()
    second = torch.nonzero(~first).flatten()
    A[torch.searchsorted(at, second, right=True) - 1] += vals[second]
    E = torch.zeros(n, dtype=F64, device=AK.device)
    e = g >= 0
    E.index_add_(0, g[e], EK[e])
    return A, E, gid, key[at]


def _global_blocks(c, seed):
    """Blocks and skeleton system of a constant kappa per coarse element (host, deterministic)."""
    nx, ny = c["nx"], c["ny"]
    tf, sg, nf = _coarse(nx, ny)
    n_K, d = 2 * nx * ny, c["m"] * (c["l"] + 1)
    loc = _Local2(nx, ny, 4, 1, c["m"], c["l"], "cpu")
    one = np.ones((n_K, 3), dtype=int)
    A2, E2, B2, F2 = loc.blocks(dict(c, source="const"), torch.ones(2, 256, dtype=F64), np.arange(2), one, "cpu")
    g = torch.Generator().manual_seed(int(seed) % (1 << 62))
    kap = 10.0 ** (c["decades"] * (2 * torch.rand(n_K, generator=g, dtype=F64) - 1))
    s = torch.as_tensor(np.repeat(sg, d, axis=1).astype(float))
    k = torch.arange(n_K) % 2
    AK = A2[k] * s[:, :, None] * s[:, None, :] / kap[:, None, None]
    EK, BK, FK = E2[k] * s / kap[:, None], B2[k] * s, F2[k].clone()
    A, E, gid, key = _scatter(c, AK, EK, tf, np.full(nf, d))
    return dict(A_vals=A, E=E, BK=BK.reshape(-1), FK=FK, gid=gid, key=key)


def _multipliers(c, seed):
    """Multipliers and means of a smooth u with the seed's amplitude, plus small higher moments."""
    nx, ny, d = c["nx"], c["ny"], c["m"] * (c["l"] + 1)
    tf, sg, nf = _coarse(nx, ny)
    g = torch.Generator().manual_seed(int(seed) % (1 << 62))
    amp = 0.5 + float(torch.rand((), generator=g, dtype=F64))
    V = _verts(nx, ny)
    mid, n = np.zeros((nf, 2)), np.zeros((nf, 2))
    for a in range(3):
        p, q = V[:, (a + 1) % 3], V[:, (a + 2) % 3]
        t = (q - p) / np.linalg.norm(q - p, axis=1, keepdims=True)
        mid[tf[:, a]] = 0.5 * (p + q)
        n[tf[:, a]] = sg[:, a, None] * np.stack([t[:, 1], -t[:, 0]], 1)
    x, y, pi = mid[:, 0], mid[:, 1], math.pi
    flux = -amp * pi * (n[:, 0] * np.cos(pi * x) * np.sin(pi * y) + n[:, 1] * np.sin(pi * x) * np.cos(pi * y))
    lam = 0.05 * torch.randn(nf, d, generator=g, dtype=F64)
    lam[:, ::c["l"] + 1] += torch.as_tensor(flux)[:, None]
    cen = V.mean(1)
    return lam.reshape(-1), torch.as_tensor(amp * np.sin(pi * cen[:, 0]) * np.sin(pi * cen[:, 1]))


def exact(case, seed):
    c = case
    if c["kind"] == "cube":
        return _exact_cube(c, seed)
    if c["kind"] == "global":
        return _exact_global(c, seed)
    nx, ny, dev = c["nx"], c["ny"], DEV
    tf, sg, nf = _coarse(nx, ny)
    n_K = 2 * nx * ny
    if c["kind"] == "reconstruct":
        kappa = _field(c, seed)
        lam, u0 = (t.to(DEV) for t in _multipliers(c, seed))
        loc, d = _Local2(nx, ny, c["r"], c["degree"], c["m"], c["l"], dev), c["m"] * (c["l"] + 1)
        u = torch.empty(n_K, loc.n, dtype=F64, device=dev)
        for Ks in np.array_split(np.arange(n_K), -(-n_K // 2048)):
            par, k = torch.as_tensor(Ks % 2, device=dev), torch.as_tensor(Ks, device=dev)
            s = torch.as_tensor(np.repeat(sg[Ks], d, axis=1).astype(float), device=dev)
            lk = lam.view(nf, d)[torch.as_tensor(tf[Ks], device=dev)].reshape(len(Ks), -1) * s
            G = torch.einsum("bi,bin->bn", lk, torch.as_tensor(loc.load, device=dev)[par])
            G = G + loc.source(c, torch.as_tensor(_verts(nx, ny)[Ks], device=dev))
            u[k] = loc.solve(kappa[k], par, G[:, :, None], back=True)[:, :, 0] + u0[k, None]
        return dict(u=u.reshape(-1))
    if c["kind"] == "levels":
        (kappa, off), rk = _levels_kappa(c, seed), _levels_of(c)
        ldeg, m, l, P = _face_degrees(c, rk).astype(int), 1, 3, 1
        c = dict(c, source="const")
    else:
        kappa, rk, ldeg = _field(c, seed).reshape(-1), np.full(n_K, c["r"]), np.full(nf, c["l"])
        off, m, l, P = np.arange(n_K + 1) * 4 ** c["r"], c["m"], c["l"], c["degree"]
    l = int(ldeg.max())
    NI = 3 * m * (l + 1)
    z = lambda *s: torch.zeros(*s, dtype=F64, device=dev)
    AK, EK, BK, FK = z(n_K, NI, NI), z(n_K, NI), z(n_K, NI), z(n_K)
    for r in sorted(set(rk.tolist())):
        loc, Kr = _Local2(nx, ny, r, P, m, l, dev), np.nonzero(rk == r)[0]
        for Ks in np.array_split(Kr, -(-len(Kr) // (2048 if r < 6 else 256))):
            k = torch.as_tensor(Ks, device=dev)
            kap = kappa[torch.as_tensor(off[Ks], device=dev)[:, None] + torch.arange(4 ** r, device=dev)]
            AK[k], EK[k], BK[k], FK[k] = loc.blocks(c, kap, Ks, sg, dev)
    if c["kind"] == "levels":   # slots past a face's own degree hold zeros
        on = (np.arange(NI // 3)[None, None] % (l + 1) <= ldeg[tf][..., None]).reshape(n_K, NI)
        on = torch.as_tensor(on.astype(float), device=dev)
        AK, EK, BK = AK * on[:, :, None] * on[:, None], EK * on, BK * on
    A, E, _, _ = _scatter(c, AK, EK, tf, m * (ldeg + 1))
    return _results({"f": c["source"] != "const"}, dict(AK=AK.reshape(-1), EK=EK.reshape(-1), BK=BK.reshape(-1), FK=FK,
                                                       status=None, A_vals=A, E=E))


def _exact_global(c, seed):
    b = _global_blocks(c, seed)
    nl, n_K = b["E"].numel(), b["FK"].numel()
    if nl + n_K > 14000:
        return None
    M = torch.zeros(nl + n_K, nl + n_K, dtype=F64)
    M[b["key"] // nl, b["key"] % nl] = b["A_vals"]
    k, g = torch.arange(n_K)[:, None].expand(-1, b["gid"].shape[1]), torch.as_tensor(b["gid"])
    M[nl + k, g] = M[g, nl + k] = b["BK"].view(n_K, -1)
    M, rhs = M.to(DEV), torch.cat([b["E"], b["FK"]]).to(DEV)
    LU, piv = torch.linalg.lu_factor(M)
    x = torch.linalg.lu_solve(LU, piv, rhs[:, None])
    for _ in range(2):
        x = x + torch.linalg.lu_solve(LU, piv, rhs[:, None] - M @ x)
    return dict(lam=x[:nl, 0].contiguous(), u0=x[nl:, 0].contiguous())


# ------------------------------------------------------------------------ the tetrahedra

_EDGES3 = list(itertools.combinations(range(4), 2))


def _cube_kappa(c, seed):
    e = torch.rand(24 * c["nc"] ** 3, 8 ** c["r"], generator=_gen(seed), device=DEV, dtype=F64) * 2 - 1
    return 10.0 ** (c["decades"] * e)


def _cube_source(c):
    if c["source"] == "const":
        return mhm.Source3D(mhm.MHM3D_SRC_CONST, 1.0, 1.0)
    return mhm.Source3D(mhm.MHM3D_SRC_SINSINSIN, 1.0, _cube_freq(c))


def _cube_freq(c):
    """The paper's source; on a single cube, whose elements it integrates to zero, half its frequency."""
    return 2.0 if c["nc"] > 1 else 1.0


def _cube_mesh(nc):
    """(vertex ids n_K x 4, coordinates): every cube cut by its centre and face centres."""
    corner = lambda i, j, k: i + (nc + 1) * (j + (nc + 1) * k)
    n0, n1 = (nc + 1) ** 3, nc ** 3
    X = [(i / nc, j / nc, k / nc) for k in range(nc + 1) for j in range(nc + 1) for i in range(nc + 1)]
    X += [((i + .5) / nc, (j + .5) / nc, (k + .5) / nc) for k in range(nc) for j in range(nc) for i in range(nc)]
    fid, tets = {}, []
    for ax in range(3):       # centres of the grid faces normal to axis ax
        dims = [nc + (a == ax) for a in range(3)]
        for k in range(dims[2]):
            for j in range(dims[1]):
                for i in range(dims[0]):
                    fid[(ax, i, j, k)] = len(X)
                    X.append(tuple((p + (0 if a == ax else .5)) / nc for a, p in enumerate((i, j, k))))
    for k in range(nc):
        for j in range(nc):
            for i in range(nc):
                centre = n0 + i + nc * (j + nc * k)
                for ax in range(3):
                    u, v = [a for a in range(3) if a != ax]
                    for side in range(2):
                        at = [i, j, k]
                        at[ax] += side
                        ring = []
                        for du, dv in ((0, 0), (1, 0), (1, 1), (0, 1)):
                            q = list(at)
                            q[u] += du
                            q[v] += dv
                            ring.append(corner(*q))
                        f = fid[(ax, *at)]
                        tets += [(centre, f, ring[e], ring[(e + 1) % 4]) for e in range(4)]
    return np.array(tets), np.array(X)


def _exact_cube(c, seed):
    N, P, m, dev = 1 << c["r"], c["degree"], c["m"], DEV
    tets, X = _cube_mesh(c["nc"])
    n_K, PN = len(tets), P * N
    # faces by first encounter, orientation signs
    ids = np.stack([np.sort(np.delete(tets, a, 1), 1) for a in range(4)], 1)
    key = (ids[..., 0].astype(np.int64) * len(X) + ids[..., 1]) * len(X) + ids[..., 2]
    u, first, inv, cnt = np.unique(key.ravel(), return_index=True, return_inverse=True, return_counts=True)
    rank = np.empty(len(u), dtype=np.int64)
    rank[np.argsort(first)] = np.arange(len(u))
    inv = inv.reshape(-1)
    tf, boundary = rank[inv].reshape(-1, 4), (cnt[inv] == 1).reshape(-1, 4)
    g = X[ids]
    nrm = np.cross(g[:, :, 1] - g[:, :, 0], g[:, :, 2] - g[:, :, 0])
    side = np.einsum("kac,kac->ka", nrm, X[tets] - g[:, :, 0])       # the vertex opposite face a
    sg = np.where(boundary | (side < 0), 1.0, -1.0)
    # submesh: nodes, sub-tetrahedra of six classes
    nodes = [(A, B, C) for C in range(PN + 1) for B in range(C, PN + 1) for A in range(B, PN + 1)]
    at = {p: i for i, p in enumerate(nodes)}
    n, sub, cls = len(nodes), [], []
    for z3, z2, z1 in itertools.product(range(N), repeat=3):
        for pi, perm in enumerate(itertools.permutations(range(3))):
            path = [np.array((z1, z2, z3))]
            for a in perm:
                path.append(path[-1] + np.eye(3, dtype=int)[a])
            if all(N >= q[0] >= q[1] >= q[2] >= 0 for q in path):
                sub.append(path)
                cls.append(pi)
    sub, cls = np.array(sub), np.array(cls)
    pts = [P * sub[:, a] for a in range(4)] + ([sub[:, a] + sub[:, b] for a, b in _EDGES3] if P == 2 else [])
    dofs = np.array([[at[tuple(p[t])] for p in pts] for t in range(len(sub))])
    nb = dofs.shape[1]
    # stiffness of the six classes of every K, from the barycentric gradients (translates of those at the origin)
    a4, w4 = np.polynomial.legendre.leggauss(4)
    a4, w4 = 0.5 * (a4 + 1), 0.5 * w4
    q3 = np.array([(a, b * (1 - a), d * (1 - a) * (1 - b)) for a in a4 for b in a4 for d in a4])
    wq = np.array([wa * wb * wd * (1 - a) ** 2 * (1 - b) for a, wa in zip(a4, w4) for b, wb in zip(a4, w4) for d, wd in zip(a4, w4)])
    lam = np.concatenate([1 - q3.sum(1, keepdims=True), q3], 1)
    if P == 1:
        phi, dphi = lam, np.broadcast_to(np.eye(4), (64, 4, 4))
    else:
        phi = np.stack([lam[:, a] * (2 * lam[:, a] - 1) for a in range(4)] + [4 * lam[:, a] * lam[:, b] for a, b in _EDGES3], 1)
        dphi = np.zeros((64, 10, 4))
        for a in range(4):
            dphi[:, a, a] = 4 * lam[:, a] - 1
        for e, (a, b) in enumerate(_EDGES3):
            dphi[:, 4 + e, a], dphi[:, 4 + e, b] = 4 * lam[:, b], 4 * lam[:, a]
    V = X[tets]
    bary = lambda L, s: np.stack([s - L[..., 0], L[..., 0] - L[..., 1], L[..., 1] - L[..., 2], L[..., 2]], -1) / s
    vol = np.abs(np.linalg.det(V[:, 1:] - V[:, :1])) / 6
    six = np.array([np.concatenate([np.zeros((1, 3), dtype=int), np.cumsum(np.eye(3, dtype=int)[list(p)], 0)])
                    for p in itertools.permutations(range(3))])
    XT = np.einsum("kvi,tav->ktai", V, bary(six, N))
    Ji = np.linalg.inv((XT[:, :, 1:] - XT[:, :, :1]))                   # columns: gradients of the barycentrics 1..3
    gb = np.concatenate([-Ji.sum(-1, keepdims=True), Ji], -1).transpose(0, 1, 3, 2)
    M4 = np.einsum("q,qai,qbj->abij", wq, dphi, dphi)
    gg = np.einsum("kcix,kcjx->kcij", gb, gb)
    Ke = np.einsum("abij,kcij->kcab", M4, gg) * (6 * vol / N ** 3)[:, None, None, None]
    # loads of the multipliers: a third of each fine face triangle per vertex (P1) or edge midpoint (P2)
    M = int(round(math.sqrt(m)))
    load = np.zeros((24, 4 * m, n))
    for K in range(24):
        for a in range(4):
            loc = [v for v in range(4) if v != a]
            srt = sorted(loc, key=lambda v: tets[K, v])
            # fine triangles of the sorted frame and the nodes they load
            co = np.array([(0, 0, 0), (1, 0, 0), (1, 1, 0), (1, 1, 1)])   # lattice direction of vertex v
            pos = lambda p, q, s: tuple(co[srt[0]] * (s - p - q) + co[srt[1]] * p + co[srt[2]] * q)
            for j in range(N):
                for i in range(N - j):
                    for up in (True, False):
                        if not up and i + j + 1 >= N:
                            continue
                        t = [(i, j), (i + 1, j), (i, j + 1)] if up else [(i + 1, j), (i + 1, j + 1), (i, j + 1)]
                        cx, cy = sum(p for p, _ in t) * M / (3 * N), sum(q for _, q in t) * M / (3 * N)
                        ci, cj = int(cx), int(cy)
                        big = cx - ci + cy - cj < 1
                        q = sum((M - jj) + (M - 1 - jj) for jj in range(cj)) + (ci if big else M - cj + ci)
                        ln = t if P == 1 else [(t[x][0] + t[y][0], t[x][1] + t[y][1]) for x, y in ((0, 1), (1, 2), (0, 2))]
                        for p in ln:
                            load[K, a * m + q, at[pos(p[0], p[1], PN)]] -= 1.0
    area = 0.5 * np.linalg.norm(nrm, axis=2) / N ** 2 / 3
    per = np.full(4, 0.25) if P == 1 else np.array([-.05] * 4 + [.2] * 6)
    mass1 = np.zeros(n)
    np.add.at(mass1, dofs, np.broadcast_to(per / N ** 3, dofs.shape))
    kap = _cube_kappa(c, seed)
    t_ = lambda x: torch.as_tensor(x, device=dev)
    NI = 4 * m
    z = lambda *s: torch.zeros(*s, dtype=F64, device=dev)
    AK, EK, BK, FK = z(n_K, NI, NI), z(n_K, NI), z(n_K, NI), z(n_K)
    idx = t_((dofs[:, :, None] * n + dofs[:, None, :]).ravel())
    for Ks in np.array_split(np.arange(n_K), -(-n_K // 1024)):
        k, B = t_(Ks), len(Ks)
        A = z(B, n * n).index_add_(1, idx, (kap[k][:, :, None, None] * t_(Ke[Ks])[:, t_(cls)]).reshape(B, -1)).view(B, n, n)
        s = t_(np.repeat(sg[Ks] * area[Ks], m, axis=1))
        N_ = t_(load)[t_(Ks % 24)] * s[:, :, None]
        mass = t_(mass1) * t_(vol[Ks])[:, None]
        if c["source"] == "const":
            f = mass.clone()
        else:
            xt = t_(bary(sub, N)) @ t_(V[Ks])[:, None]                    # (B, T, 4, 3)
            xq = torch.einsum("qa,btac->btqc", t_(lam), xt)
            kf = math.pi * _cube_freq(c)
            fv = 3 * kf ** 2 * torch.sin(kf * xq).prod(-1)
            fe = torch.einsum("btq,qa->bta", fv, t_(phi * wq[:, None])) * t_(6 * vol[Ks] / N ** 3)[:, None, None]
            f = z(B, n).index_add_(1, t_(dofs.ravel()), fe.reshape(B, -1))
        G = torch.cat([N_, f[:, None]], 1).transpose(1, 2)
        G = G - mass[:, :, None] * (G.sum(1, keepdim=True) / t_(vol[Ks])[:, None, None])
        L = torch.linalg.cholesky(A[:, 1:, 1:])
        Y = torch.linalg.solve_triangular(L, G[:, 1:], upper=False)
        gram = Y.transpose(1, 2) @ Y
        AK[k], EK[k], BK[k], FK[k] = -gram[:, :NI, :NI], gram[:, :NI, NI], -N_.sum(2), f.sum(1)
    A, E, _, _ = _scatter(c, AK, EK, tf, np.full(len(u), m))
    return _results({"f": c["source"] != "const"}, dict(AK=AK, EK=EK, BK=BK, FK=FK, status=None, A_vals=A, E=E))
