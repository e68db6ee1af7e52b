"""The work that a program using this library has it do, as cases that can be measured.

A program builds the H-matrix of a mesh (hm_efie_fill, hm_efie_far), factors the near-field
preconditioner (precond_setup), and then solves for many right-hand sides: one by one, in a
batch, or as a served stream.  Inside a solve the time goes to the preconditioned operator
(Eq. 28), the refinement residual and the Gram-Schmidt steps.  The cases are these calls, each
through its public entry point:

    near     near-field blocks of a mesh
    far      ACA factors of the admissible blocks
    setup    precond_setup, then the factors applied once (D^{-1} L^{-1} x)
    op       hm_apply of the preconditioned operator A
    residual hm_apply of Z itself (FP64), the refinement residual's operator
    solve    solve_device, right-hand sides and solutions on the device
    host     solve, right-hand sides and solutions in host memory
    serve    requests through the slots of a Batch

Meshes: a jittered lambda/10 plate of m x m squares (3 m^2 - 2 m unknowns) and an icosphere of
30 * 4^d edges whose vertices are moved by up to 5% of an edge (a regular icosphere has
exactly tied ACA pivots, which no real mesh has).  The H-matrix is an input of the solver calls:
it is kept per mesh, while vectors and right-hand sides come from the seed.  What the complex-FP32
operators and the mixed solves (asked for 1e-4 to 1e-5) return carries single precision, and is kept as
complex64; FP64 handles return complex128.
"""
import functools
import math

import numpy as np
import torch

import paper_2111_13483_gb300 as hm
from efie_problem import builder as _builder
from efie_problem import mesh as _mesh
from efie_problem import tree as _tree

H = hm.hmsolve
LEAF, ETA, JITTER = 64, 1.0, 0.1


def listed():
    return [
        # H-matrix build of a mid-size mesh: the dense near field, then the far-field factors
        dict(name="near_plate72", kind="near", mesh="plate", size=72),
        dict(name="far_plate48", kind="far", mesh="plate", size=48),
        # a new geometry's preconditioner: the 30,720-unknown benchmark sphere in the mixed
        # form with compressed fill-in, and the FP64 form without compression
        dict(name="setup_mixed_sphere30720", kind="setup", mesh="sphere", size=5, precision=1, fill_tol=1e-2,
             ordering=1, nrhs=8),
        dict(name="setup_fp64_plate40", kind="setup", mesh="plate", size=40, precision=0, fill_tol=0.0, ordering=1,
             nrhs=1),
        # the operator of one Arnoldi step: the benchmark's 64 columns; a ragged batch with
        # dense coefficients; one column of a small body; the FP64 form, one column
        dict(name="op_mixed_sphere30720_64", kind="op", mesh="sphere", size=5, precision=1, fill_tol=1e-2, ordering=1,
             nrhs=64),
        dict(name="op_mixed_plate87_23", kind="op", mesh="plate", size=87, precision=1, fill_tol=0.0, ordering=1,
             nrhs=23),
        dict(name="op_mixed_plate20_1", kind="op", mesh="plate", size=20, precision=1, fill_tol=0.0, ordering=1,
             nrhs=1),
        dict(name="op_fp64_sphere7680_1", kind="op", mesh="sphere", size=4, precision=0, fill_tol=0.0, ordering=1,
             nrhs=1),
        # the refinement residual of the benchmark's batch
        dict(name="residual_sphere30720_64", kind="residual", mesh="sphere", size=5, nrhs=64),
        # a monostatic sweep over the 10 x 10 lambda plate, 64 angles at once
        dict(name="solve_mixed_plate100_64", kind="solve", mesh="plate", size=100, precision=1, fill_tol=1e-2,
             ordering=1, nrhs=64, tol=1e-5, restart=50),
        # one plane wave on the 1920-unknown sphere, plain FP64, from host memory
        dict(name="host_fp64_sphere1920_1", kind="host", mesh="sphere", size=3, precision=0, fill_tol=0.0, ordering=1,
             nrhs=1, tol=1e-4, restart=30),
        # served requests: 40 angles through 16 slots that are refilled as solves end
        dict(name="serve_mixed_sphere7680_40", kind="serve", mesh="sphere", size=4, precision=1, fill_tol=1e-2,
             ordering=1, nrhs=40, slots=16, tol=1e-5, restart=30),
    ]


def _log_size(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["near", "far", "setup", "op", "op", "residual", "solve", "host", "serve"])
    c = dict(kind=kind, mesh="plate", size=_log_size(rng, 8, 72))
    if kind in ("near", "far"):
        c["size"] = _log_size(rng, 8, 72) if kind == "near" else _log_size(rng, 16, 48)
        return c
    if rng.random() < 0.3:
        c.update(mesh="sphere", size=rng.choice([2, 3, 4]))
    c["nrhs"] = _log_size(rng, 1, 64)
    if kind == "residual":
        return c
    c.update(precision=rng.choice([0, 1, 1]), fill_tol=rng.choice([0.0, 1e-3, 1e-2]), ordering=rng.choice([1, 1, 2]))
    if kind == "setup":
        c["nrhs"] = rng.choice([1, 8])
        if c["precision"] == 0:
            c["fill_tol"] = 0.0
    if c["precision"] == 0:   # the FP64 form is the smaller problems' and the narrow batches'
        c["size"] = c["size"] if c["mesh"] == "sphere" else min(c["size"], 40)
        c["nrhs"] = min(c["nrhs"], 16)
    if kind in ("solve", "host", "serve"):
        c.update(tol=rng.choice([1e-4, 1e-5]), restart=rng.choice([30, 50]))
        if kind == "host":
            c["nrhs"] = min(c["nrhs"], 8)
        if c["precision"] == 0:
            c["fill_tol"] = 0.0
            c["nrhs"] = min(c["nrhs"], 4)
            c["size"] = min(c["size"], 3) if c["mesh"] == "sphere" else min(c["size"], 32)
        if kind == "serve":
            c["slots"] = rng.choice([4, 8, 16])
    return c


# ---- geometry and H-matrix: what the program has read or built before ---------------------------
class _Geometry:
    def __init__(self, mesh, size):
        if mesh == "plate":
            V, T = _mesh.plate(size, 0.1 * size, JITTER, 0)
        else:
            V, T = _mesh.icosphere(size, 0.075 * 2 ** size)
            edge = np.linalg.norm(V[T[0, 0]] - V[T[0, 1]])
            V = V + np.random.default_rng(0).uniform(-0.05 * edge, 0.05 * edge, V.shape)
        rwg = self.rwg = _mesh.RWG(V, T)
        root, leaves, perm = _tree.build_tree(rwg.midpoints(), LEAF, vertices=V)
        _tree.attach_boxes(root, perm, *rwg.support_boxes())
        near, far = _tree.partition(root, ETA)
        lp = np.array([lf.lo for lf in leaves] + [leaves[-1].hi], dtype=np.int64)
        self.perm, self.leaf_ptr = perm.astype(np.int32), lp.astype(np.int32)
        self.near = sorted({(min(t, s), max(t, s)) for t, s in near})
        self.near_rows = [perm[lp[t]:lp[t + 1]] for t, _ in self.near]
        self.near_cols = [perm[lp[s]:lp[s + 1]] for _, s in self.near]
        fr = [(t, s) for t, s in far if t.lo < s.lo]
        fr.sort(key=lambda ts: (ts[0].lo, ts[1].lo, ts[0].hi, ts[1].hi))
        self.far = [(t.lo, t.hi, s.lo, s.hi) for t, s in fr]
        self.far_rows = [perm[t.lo:t.hi] for t, _ in fr]
        self.far_cols = [perm[s.lo:s.hi] for _, s in fr]
        self.mesh = H.Mesh(rwg.V, rwg.T, rwg.tri, rwg.free, _builder.K0, _builder.ETA0)


@functools.lru_cache(maxsize=4)
def _geometry(mesh, size):
    return _Geometry(mesh, size)


def _variant(G, kind, seed):
    """The mesh that a seed's build is called for, its vertices and its impedance: the near field of a slightly
    deformed body with the same blocks; the far field in another medium (a deformation would change the ranks, and
    with them the sizes of the outputs)."""
    rng = np.random.default_rng(seed)
    V, eta0 = G.rwg.V, _builder.ETA0
    if kind == "near":
        V = V + rng.uniform(-0.002, 0.002, V.shape) * (np.ptp(V, axis=0) > 0)
    else:
        eta0 *= rng.uniform(0.5, 1.0)
    return H.Mesh(V, G.rwg.T, G.rwg.tri, G.rwg.free, _builder.K0, eta0), V, eta0


@functools.lru_cache(maxsize=4)
def _problem(mesh, size):
    G = _geometry(mesh, size)
    P = _builder.Problem()
    P.rwg, P.k, P.eta0 = G.rwg, _builder.K0, _builder.ETA0
    P.perm, P.leaf_ptr = G.perm, G.leaf_ptr
    P.near_t = np.array([a for a, _ in G.near], dtype=np.int32)
    P.near_s = np.array([b for _, b in G.near], dtype=np.int32)
    P.near_data, off = H.hm_efie_fill(G.mesh, G.near_rows, G.near_cols, mirror=1)
    P.near_off = off[:-1].astype(np.int64)
    f = np.array(G.far, dtype=np.int32).reshape(-1, 4)
    P.far_r0, P.far_r1, P.far_c0, P.far_c1 = (np.ascontiguousarray(f[:, i]) for i in range(4))
    if G.far:
        P.far_rank, P.far_uoff, P.far_voff, P.far_U, P.far_V = H.hm_efie_far(G.mesh, G.far_rows, G.far_cols, 1e-3)
    else:
        P.far_rank, P.far_uoff, P.far_voff = np.zeros(0, np.int32), np.zeros(0, np.int64), np.zeros(0, np.int64)
        P.far_U, P.far_V = np.zeros(1, np.complex128), np.zeros(0, np.complex128)
    return P


@functools.lru_cache(maxsize=1)
def _stream():
    """The program's stream: the handles' and its own tensor work are ordered on it."""
    return torch.cuda.Stream()


def _handle(case):
    P = _problem(case["mesh"], case["size"])
    return P, hm.hmat_create(P, ordering=case.get("ordering", 1), fill_tol=case.get("fill_tol", 0.0),
                             precision=case.get("precision", 1), stream=_stream().cuda_stream)


# Radon's 7-point degree-5 rule on a triangle
_S15 = math.sqrt(15.0)
_QW = [9 / 40] + [(155 - _S15) / 1200] * 3 + [(155 + _S15) / 1200] * 3
_QB = [[1 / 3] * 3] + [[1 - 2 * a if i == j else a for j in range(3)] for a in ((6 - _S15) / 21, (6 + _S15) / 21)
                       for i in range(3)]


def _plane_waves(P, seed, count):
    """Right-hand sides <f_m, E_inc> of plane waves from random directions with random linear polarisation, original
    order: (count, n) on the device."""
    rng = np.random.default_rng(seed)
    z, phi, psi = rng.uniform(-1, 1, count), rng.uniform(0, 2 * np.pi, count), rng.uniform(0, 2 * np.pi, count)
    s = np.sqrt(1 - z * z)
    th = np.stack([z * np.cos(phi), z * np.sin(phi), -s], 1)
    ph = np.stack([-np.sin(phi), np.cos(phi), 0 * phi], 1)
    dev = dict(dtype=torch.float64, device="cuda")
    kh = torch.tensor(-np.stack([s * np.cos(phi), s * np.sin(phi), z], 1), **dev)
    pol = torch.tensor(np.cos(psi)[:, None] * th + np.sin(psi)[:, None] * ph, **dev)
    rwg = P.rwg
    V, T = torch.tensor(rwg.V, **dev), torch.tensor(rwg.T.astype(np.int64), device="cuda")
    Q = torch.einsum("qa,tad->tqd", torch.tensor(_QB, **dev), V[T])
    w = torch.tensor(_QW, **dev)
    tri, free = (torch.tensor(a.astype(np.int64), device="cuda") for a in (rwg.tri, rwg.free))
    length = torch.tensor(rwg.length, **dev)
    out = torch.zeros(count, rwg.n, dtype=torch.complex128, device="cuda")
    for c in range(count):
        a = -P.k * (Q @ kh[c])
        e = torch.complex(torch.cos(a), torch.sin(a)) * w
        for side, sign in ((0, 0.5), (1, -0.5)):
            t = tri[:, side]
            rho = (Q[t] - V[free[:, side]][:, None, :]) @ pol[c]
            out[c] += sign * length * (rho * e[t]).sum(1)
    return out


def _vectors(n, seed, count):
    """Unit vectors with the flat spectrum of Krylov vectors: (count, n) complex128 on the device."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.view_as_complex(torch.randn(count, n, 2, dtype=torch.float64, device="cuda", generator=g))
    return x / torch.linalg.vector_norm(x, dim=1, keepdim=True)


# ---- the calls ----------------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    if kind in ("near", "far"):
        G = _geometry(case["mesh"], case["size"])
        return dict(case=case, mesh=_variant(G, kind, seed)[0], rows=getattr(G, kind + "_rows"),
                    cols=getattr(G, kind + "_cols"))
    P, h = _handle(case)
    s = dict(case=case, h=h)
    if kind in ("op", "solve", "host", "serve"):
        hm.precond_setup(h)
    if kind in ("setup", "op", "residual"):
        s["x"] = _vectors(P.n, seed, case["nrhs"])
    else:
        s["V"] = _plane_waves(P, seed, case["nrhs"])
        if kind in ("host", "serve"):
            s["V"] = s["V"].cpu().numpy()
    if kind == "host":
        s["V"] = np.asfortranarray(s["V"].T)
    return s


def _kept(case, y):
    """What the program keeps of a result: single precision of the single-precision forms."""
    if case.get("precision", 0) == 0:
        return y
    return y.astype(np.complex64) if isinstance(y, np.ndarray) else y.to(torch.complex64)


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "near":
        return H.hm_efie_fill(s["mesh"], s["rows"], s["cols"], mirror=1)[0]
    if kind == "far":
        rank, uoff, voff, U, V = H.hm_efie_far(s["mesh"], s["rows"], s["cols"], 1e-3)
        return dict(rank=rank, U=U, V=V)
    h = s["h"]
    if kind == "host":
        return _kept(case, hm.solve(h, s["V"], tol=case["tol"], restart=case["restart"])[0])
    if kind == "serve":
        return _kept(case, _serve(h, s["V"], case))
    o32 = H.OP32 if case.get("precision") == 1 else 0
    with torch.cuda.stream(_stream()):
        if kind == "solve":
            I = torch.empty_like(s["V"])
            hm.solve_device(h, s["V"], I, tol=case["tol"], restart=case["restart"])
            return _kept(case, I)
        x = s["x"]
        y = torch.empty_like(x)
        if kind == "residual":
            hm.hm_apply(h, H.OP_Z, x, y)
            return y
        if kind == "op":
            hm.hm_apply(h, o32 + H.OP_A, x, y)
            return _kept(case, y)
        hm.precond_setup(h)
        z = torch.empty_like(x)
        hm.hm_apply(h, o32 + H.OP_LINV, x, y)
        hm.hm_apply(h, o32 + H.OP_DINV, y, z)
        return dict(linv=_kept(case, y), dinv=_kept(case, z))


def _serve(h, V, case):
    out = np.empty(V.shape, dtype=np.complex128)
    where, nxt, left = {}, 0, len(V)
    b = hm.Batch(h, min(case["slots"], len(V)), case["restart"])
    try:
        while left:
            while nxt < len(V):
                slot = b.submit(V[nxt], tol=case["tol"])
                if slot is None:
                    break
                where[slot] = nxt
                nxt += 1
            for slot in b.step():
                out[where.pop(slot)] = b.result(slot)[0]
                left -= 1
    finally:
        b.close()
    return out


# ---- the work a pass cannot do without ----------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _facts(key):
    """Stored entries of a case's H-matrix and factors, and the mean Arnoldi steps of its solves."""
    case = dict(key)
    P, h = _handle(case)
    if case["kind"] != "residual":
        hm.precond_setup(h)
    f = hm.hmat_stats(h)
    f["steps"] = 0.0
    if "tol" in case:
        V = _plane_waves(P, 1, 2)
        f["steps"] = float(np.mean(hm.solve_device(h, V, torch.empty_like(V), tol=case["tol"], restart=case["restart"])[0]))
    return f


def work(case):
    kind = case["kind"]
    if kind in ("near", "far"):
        G = _geometry(case["mesh"], case["size"])
        m = np.array([len(r) for r in getattr(G, kind + "_rows")], dtype=np.float64)
        n = np.array([len(c) for c in getattr(G, kind + "_cols")], dtype=np.float64)
        if kind == "near":
            # an entry needs four triangle pairs, a pair serves up to nine entries; 49 kernel
            # values a pair, about 40 operations each
            return dict(bytes=16.0 * float(m @ n), flops=float(m @ n) * 4 / 9 * 49 * 40)
        r = np.minimum(6.0, np.minimum(m, n) / 2)   # typical rank at 1e-3; a row of n entries: 4 n / 3 pairs
        return dict(bytes=16.0 * float(np.sum(np.minimum(r * (m + n), m * n))),
                    flops=float(np.sum(r * (m + n))) * 4 / 3 * 49 * 40)
    f = _facts(tuple(sorted((k, v) for k, v in case.items() if k not in ("name", "nrhs", "slots"))))
    n, B, e = f["n"], case["nrhs"], 8.0 if case.get("precision") == 1 else 16.0
    near, far, coef, diag = f["near_entries"], f["far_entries"], f["coef_entries"], f["diag_entries"]
    if kind == "residual":
        return dict(bytes=16.0 * (near + far) + 32.0 * n * B, flops=16.0 * B * (near + far))
    if kind == "setup":
        return dict(bytes=16.0 * near + e * (coef + 2 * diag) + 48.0 * n * B,
                    flops=1e9 * f["setup_gflop"] + 8.0 * B * (coef + diag))
    op_bytes, op_flops = e * (far + coef + 2 * diag), 16.0 * B * (coef + far + diag)
    if kind == "op":
        return dict(bytes=op_bytes + 32.0 * n * B, flops=op_flops)
    # a step: the operator, and two Gram-Schmidt passes over half a restart cycle's basis
    cols = min(B, case.get("slots", B), 64 if case["precision"] == 1 else 16)
    j = min(f["steps"], case["restart"]) / 2
    return dict(bytes=f["steps"] * math.ceil(B / cols) * (op_bytes + 16.0 * n * cols * (j + 3)) + 32.0 * n * B,
                flops=f["steps"] * (op_flops + 32.0 * B * n * j))


# ---- the results in 64 bits ---------------------------------------------------------------------
EXACT_N = 8000   # larger systems take a dense elimination too long


def exact(case, seed):
    kind = case["kind"]
    if kind == "near":
        G = _geometry(case["mesh"], case["size"])
        return _exact_near(G, *_variant(G, kind, seed)[1:])
    if kind == "far":
        return None      # the factors of a low-rank block are not unique
    if case.get("precision") == 0 and case["fill_tol"] > 0 or kind in ("op", "setup") and case["fill_tol"] > 0:
        return None      # depends on the ranks that the truncation chooses
    n = 3 * case["size"] ** 2 - 2 * case["size"] if case["mesh"] == "plate" else 30 * 4 ** case["size"]
    if n > EXACT_N:
        return None
    P = _problem(case["mesh"], case["size"])
    N, F = _dense(P)
    perm = torch.tensor(P.perm.astype(np.int64), device="cuda")
    if kind in ("residual", "solve", "host", "serve"):
        inv = torch.argsort(perm)
        Z = (N + F)[inv][:, inv]
        if kind == "residual":
            return _vectors(P.n, seed, case["nrhs"]) @ Z.T
        X = torch.linalg.solve(Z, _plane_waves(P, seed, case["nrhs"]).T)
        return X if kind == "host" else X.T
    # solve order: the leaves in the block order of Algorithm 1, an integer plan
    lp = P.leaf_ptr
    order = H.hm_plan_order_method(case["ordering"], len(lp) - 1, P.near_t, P.near_s)
    idx = torch.tensor(np.concatenate([np.arange(lp[l], lp[l + 1]) for l in order]), device="cuda")
    size = np.diff(lp)[order]
    U, Dk = _eliminate(N[idx][:, idx], size, order, P)
    F = F[idx][:, idx]
    X = _vectors(P.n, seed, case["nrhs"]).T
    tri = torch.linalg.solve_triangular
    off = np.concatenate([[0], np.cumsum(size)])

    def blocks(f, x):
        return torch.cat([f(Dk[k], x[off[k]:off[k + 1]]) for k in range(len(Dk))])

    def linv(x):
        return tri(U.T, x, upper=False, unitriangular=True)

    if kind == "setup":
        y = linv(X)
        return dict(linv=y.T, dinv=blocks(torch.linalg.solve, y).T)
    w = linv(F @ tri(U, X, upper=True, unitriangular=True))
    return blocks(torch.linalg.solve, blocks(torch.matmul, X) + w).T


def _dense(P):
    """Near and far part of Z, dense, in cluster order."""
    N, F = (torch.zeros(P.n, P.n, dtype=torch.complex128, device="cuda") for _ in range(2))
    lp = P.leaf_ptr
    data, fU, fV = (torch.tensor(a, device="cuda") for a in (P.near_data, P.far_U, P.far_V))

    def put(A, r0, r1, c0, c1, B):
        A[r0:r1, c0:c1] = B
        A[c0:c1, r0:r1] = B.T

    for t, s, o in zip(P.near_t, P.near_s, P.near_off):
        m, c = lp[t + 1] - lp[t], lp[s + 1] - lp[s]
        put(N, lp[t], lp[t + 1], lp[s], lp[s + 1], data[o:o + m * c].view(c, m).T)
    for b in range(len(P.far_rank)):
        r0, r1, c0, c1, r = (int(a[b]) for a in (P.far_r0, P.far_r1, P.far_c0, P.far_c1, P.far_rank))
        u, v = int(P.far_uoff[b]), int(P.far_voff[b])
        m, c = r1 - r0, c1 - c0
        B = fU[u:u + m * c].view(c, m).T if r < 0 else fU[u:u + m * r].view(r, m).T @ fV[v:v + c * r].view(r, c)
        put(F, r0, r1, c0, c1, B)
    return N, F


def _eliminate(A, size, order, P):
    """Block elimination of A (solve order): A = U^T diag(D_k) U with U unit upper triangular."""
    nb = len(size)
    off = np.concatenate([[0], np.cumsum(size)])
    pos = np.empty(nb, dtype=np.int64)
    pos[order] = np.arange(nb)
    reach = np.arange(nb)   # the last block coupled to block k or an earlier one
    for t, s in zip(pos[P.near_t], pos[P.near_s]):
        reach[min(t, s)] = max(reach[min(t, s)], t, s)
    reach = np.maximum.accumulate(reach)
    U, D = torch.eye(len(A), dtype=A.dtype, device=A.device), []
    for k in range(nb):
        a, b, e = off[k], off[k + 1], off[reach[k] + 1]
        D.append(A[a:b, a:b].clone())
        if e > b:
            W = torch.linalg.solve(D[k], A[a:b, b:e])
            U[a:b, b:e] = W
            A[b:e, b:e] -= A[b:e, a:b] @ W
    return U, D


def _exact_near(G, V, eta0):
    """The near-field blocks of Eq. 7 by the same 7 x 7 point rule and, for close triangles, the singular part in
    closed form (Wilton et al. 1984, Graglia 1993), in torch."""
    dev = dict(dtype=torch.float64, device="cuda")
    rwg, k = G.rwg, _builder.K0
    V, T = torch.tensor(V, **dev), torch.tensor(rwg.T.astype(np.int64), device="cuda")
    tri, free = (torch.tensor(a.astype(np.int64), device="cuda") for a in (rwg.tri, rwg.free))
    edge, nt = torch.tensor(rwg.edge.astype(np.int64), device="cuda"), len(rwg.T)
    length = torch.linalg.vector_norm(V[edge[:, 1]] - V[edge[:, 0]], dim=1)
    C = V[T]
    nrm = torch.linalg.cross(C[:, 1] - C[:, 0], C[:, 2] - C[:, 0])
    area = torch.linalg.vector_norm(nrm, dim=1) / 2
    nrm = nrm / (2 * area[:, None])
    cen = C.mean(1)
    hmax = torch.stack([torch.linalg.vector_norm(C[:, i] - C[:, j], dim=1) for i, j in ((0, 1), (0, 2), (1, 2))]).amax(0)
    w, Q = torch.tensor(_QW, **dev), torch.einsum("qa,tad->tqd", torch.tensor(_QB, **dev), C)
    rows = torch.tensor(np.concatenate([np.tile(r, len(c)) for r, c in zip(G.near_rows, G.near_cols)]).astype(np.int64),
                        device="cuda")
    cols = torch.tensor(np.concatenate([np.repeat(c, len(r)) for r, c in zip(G.near_rows, G.near_cols)]).astype(np.int64),
                        device="cuda")
    keys = torch.unique(torch.cat([tri[rows, s] * nt + tri[cols, t] for s in (0, 1) for t in (0, 1)]))

    def potential(q, r):   # int 1/R and int (r' - rho)/R over triangle q at the points r (np, 7, 3)
        n, P0 = nrm[q][:, None], C[q]
        h = ((r - P0[:, None, 0]) * n).sum(-1)
        rho, ah = r - h[..., None] * n, h.abs()
        S0, Sv = torch.zeros_like(h), torch.zeros_like(r)
        for i in range(3):
            a, b = P0[:, None, i], P0[:, None, (i + 1) % 3]
            le = torch.linalg.vector_norm(b - a, dim=-1, keepdim=True)
            l = (b - a) / le
            u = torch.linalg.cross(l, n)
            lp, lm, p0 = ((b - rho) * l).sum(-1), ((a - rho) * l).sum(-1), ((a - rho) * u).sum(-1)
            R0 = p0 * p0 + h * h
            Rp, Rm = (lp * lp + R0).sqrt(), (lm * lm + R0).sqrt()
            f = torch.where(lp + lm >= 0, ((Rp + lp) / (Rm + lm)).log(), ((Rm - lm) / (Rp - lp)).log())
            f = torch.where(R0 > 1e-24 * le[..., 0] ** 2, f, torch.zeros_like(f))
            S0 += p0 * f
            g = ah * (torch.atan(p0 * lp / (R0 + ah * Rp)) - torch.atan(p0 * lm / (R0 + ah * Rm)))
            S0 -= torch.where((ah > 0) & (p0 != 0), g, torch.zeros_like(g))
            Sv += (0.5 * (R0 * f + lp * Rp - lm * Rm))[..., None] * u
        return S0, Sv, rho

    vals = torch.empty(len(keys), 8, dtype=torch.complex128, device="cuda")   # <<G>>, <<G r>>, <<G r'>>, <<G r.r'>>
    for c0 in range(0, len(keys), 1 << 18):
        p, q = keys[c0:c0 + (1 << 18)] // nt, keys[c0:c0 + (1 << 18)] % nt
        rp, rq = Q[p], Q[q]
        R = torch.linalg.vector_norm(rp[:, :, None] - rq[:, None], dim=-1)
        far_g = torch.complex(torch.cos(k * R), -torch.sin(k * R)) / R
        sm = torch.complex(-2 * torch.sin(0.5 * k * R) ** 2 / R, -torch.sin(k * R) / R)
        sm = torch.where(R < 1e-14, torch.full_like(sm, -1j * k), sm)
        thr = (1.5 * (hmax[p] + hmax[q])).clamp_min(0.2)
        close = (p == q) | (torch.linalg.vector_norm(cen[p] - cen[q], dim=1) < thr)
        g = torch.where(close[:, None, None], sm, far_g) * w * area[q][:, None, None]
        s0, sv = g.sum(2), torch.einsum("pab,pbd->pad", g, rq.to(g.dtype))
        i = close.nonzero()[:, 0]
        S0, Sv, rho = potential(q[i], rp[i])
        s0[i] += S0
        sv[i] += Sv + rho * S0[..., None]
        s0, sv = s0 * w * area[p][:, None], sv * (w * area[p][:, None])[..., None]
        rc = rp.to(g.dtype)
        vals[c0:c0 + (1 << 18)] = torch.cat([s0.sum(1)[:, None], (s0[..., None] * rc).sum(1), sv.sum(1),
                                             (sv * rc).sum((1, 2))[:, None]], 1)
    out = torch.zeros(len(rows), dtype=torch.complex128, device="cuda")
    for c0 in range(0, len(rows), 1 << 21):
        m, n = rows[c0:c0 + (1 << 21)], cols[c0:c0 + (1 << 21)]
        z = torch.zeros(len(m), dtype=torch.complex128, device="cuda")
        for s in (0, 1):
            for t in (0, 1):
                p, q = tri[m, s], tri[n, t]
                v = vals[torch.searchsorted(keys, p * nt + q)]
                vm, vn = V[free[m, s]].to(v.dtype), V[free[n, t]].to(v.dtype)
                dot = v[:, 7] - (vn * v[:, 1:4]).sum(1) - (vm * v[:, 4:7]).sum(1) + (vm * vn).sum(1) * v[:, 0]
                z += (1 if s == t else -1) / (area[p] * area[q]) * (dot / 4 - v[:, 0] / (k * k))
        out[c0:c0 + (1 << 21)] = 1j * k * eta0 / (4 * math.pi) * length[m] * length[n] * z
    o = 0   # a leaf's own block: the upper triangle mirrored
    for (t, s), r, c in zip(G.near, G.near_rows, G.near_cols):
        if t == s:
            B = out[o:o + len(r) * len(c)].view(len(c), len(r)).T.clone()
            B = torch.triu(B) + torch.triu(B, 1).T
            out[o:o + len(r) * len(c)] = B.T.reshape(-1)
        o += len(r) * len(c)
    return out
