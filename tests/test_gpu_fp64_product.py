"""The FP64 product Z x (hm_apply ops 5 and 3) entry by entry, for factors, near field and vectors of any scale: the
digits on the tensor cores follow the largest entries near by, and an output they could give less accurately than FP64
FMAs comes from those.

Tolerance: an output is a sum of products n_ij x_j and u_il (v_jl x_j), whose FP64 FMAs (complex, so two a term) err by
at most u times twice the number of terms behind one another times S = |N| |x| + sum |U| (|V|^T |x|): at most n terms
of a row after at most n of a rank vector, and a few additions of partial sums.  The bound is sqrt(2) 2 (2 n + 32) u S.
"""
import copy

import numpy as np
import pytest
import torch

import paper_2111_13483_gb300 as hm
from test_gpu_setup_blocks import MIXED, problem

pytestmark = pytest.mark.gpu
H = hm.hmsolve


def apply(h, op, X):
    x = torch.from_numpy(np.ascontiguousarray(X)).cuda()
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    hm.hm_apply(h, op, x, y)
    return y.cpu().numpy()


def far_blocks(P):
    for b in range(len(P.far_rank)):
        r0, r1, c0, c1, r = (int(a[b]) for a in (P.far_r0, P.far_r1, P.far_c0, P.far_c1, P.far_rank))
        u, v, m, c = int(P.far_uoff[b]), int(P.far_voff[b]), r1 - r0, c1 - c0
        yield slice(r0, r1), slice(c0, c1), slice(u, u + m * (c if r < 0 else r)), slice(v, v + c * max(r, 0)), r


def exact(P, X, near=True):
    """Z X^T or Z_F X^T, transposed, and S of every entry; cluster order, 64-bit mantissas or more."""
    X = X.astype(np.clongdouble).T
    A = np.abs(X).astype(float)
    y, S = np.zeros_like(X), np.zeros_like(A)
    lp = P.leaf_ptr

    def add(i, j, B):
        y[i] += B @ X[j]
        S[i] += np.abs(B).astype(float) @ A[j]

    if near:
        for t, s, o in zip(P.near_t, P.near_s, P.near_off):
            i, j = slice(lp[t], lp[t + 1]), slice(lp[s], lp[s + 1])
            m, c = lp[t + 1] - lp[t], lp[s + 1] - lp[s]
            B = P.near_data[o:o + m * c].reshape(c, m).T.astype(np.clongdouble)
            add(i, j, B)
            if t != s:
                add(j, i, B.T)
    for i, j, u, v, r in far_blocks(P):
        if r == 0:
            continue
        m, c = i.stop - i.start, j.stop - j.start
        U = P.far_U[u].reshape(-1, m).T.astype(np.clongdouble)
        if r < 0:
            add(i, j, U)
            add(j, i, U.T)
            continue
        V = P.far_V[v].reshape(r, c).T.astype(np.clongdouble)
        for a, b, F, G in ((i, j, U, V), (j, i, V, U)):
            y[a] += F @ (G.T @ X[b])
            S[a] += np.abs(F).astype(float) @ (np.abs(G).T.astype(float) @ A[b])
    return y.T, S.T


def scaled(P, kind):
    """P with other scales, and the factor of each vector entry (cluster order)."""
    Q, d, rng = copy.copy(P), np.ones(P.n), np.random.default_rng(5)
    Q.far_U, Q.far_V, Q.near_data = P.far_U.copy(), P.far_V.copy(), P.near_data.copy()
    if kind.startswith("uv"):
        Q.far_V *= 2.0 ** -int(kind[2:])
        for _, _, u, _, r in far_blocks(P):
            Q.far_U[u] *= 2.0 ** (int(kind[2:]) if r > 0 else 0)
    elif kind == "blocks":   # every block its own
        for _, _, u, v, r in far_blocks(P):
            k = int(rng.integers(-50, 51)) if r > 0 else 0
            Q.far_U[u] *= 2.0 ** k
            Q.far_V[v] *= 2.0 ** -k
    elif kind.startswith("z"):
        Q.far_U *= 2.0 ** int(kind[1:])
        Q.near_data *= 2.0 ** int(kind[1:])
    elif kind.startswith("near"):
        Q.near_data *= 2.0 ** int(kind[4:])
    elif kind == "leaves":   # vectors graded from leaf to leaf, and within the leaves
        d = 2.0 ** -(3.0 * np.searchsorted(P.leaf_ptr, np.arange(P.n), side="right"))
    elif kind == "entries":
        d = 2.0 ** -rng.integers(0, 60, P.n).astype(float)
    elif kind == "rows":     # coefficients and vector graded the opposite way, within the blocks
        d = 2.0 ** -(np.arange(P.n) % 50.0)
        for t, s, o in zip(P.near_t, P.near_s, P.near_off):
            (a, m), (b, c) = ((int(P.leaf_ptr[l]), int(P.leaf_ptr[l + 1] - P.leaf_ptr[l])) for l in (t, s))
            g = 2.0 ** ((a + np.arange(m)) % 50)[None, :] * 2.0 ** ((b + np.arange(c)) % 50)[:, None]
            Q.near_data[o:o + m * c] *= g.ravel()
    return Q, d


CHECKED = [0, 3, 7]   # columns compared with the exact product
KINDS = ["uv0", "uv10", "uv20", "uv40", "uv-40", "blocks", "z-40", "z40", "near40", "near-40", "leaves", "entries", "rows"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("mesh", ["mixed", "sphere480"])
def test_entries_at_every_scale(kind, mesh, sphere480):
    P = problem(MIXED, 11)[0] if mesh == "mixed" else sphere480
    P, d = scaled(P, kind)
    h = hm.hmat_create(P, ordering=1)
    rng = np.random.default_rng(4)
    X = (rng.standard_normal((16, P.n)) + 1j * rng.standard_normal((16, P.n))) * d
    X[3] = 0
    X[3, P.n // 2] = 1      # one entry alone
    X[7, :P.n // 2] = 0
    new2orig = np.asarray(hm.hm_get_index_map(h))
    inv = np.argsort(np.asarray(P.perm))
    for op in (H.OP_Z, H.OP_ZF):
        want, S = exact(P, X[CHECKED], near=op == H.OP_Z)
        into = np.argsort(inv[new2orig]) if op == H.OP_ZF else np.asarray(P.perm)   # op 3: solve order, op 5: original
        x = np.zeros_like(X)
        if op == H.OP_Z:
            x[:, np.asarray(P.perm)] = X
        else:
            x = X[:, inv[new2orig]]
        ref = None
        for w in (16, 1, 4, 5):
            y = apply(h, op, x[:w])
            ref = y if ref is None else ref
            assert np.array_equal(y, ref[:w]), (op, w)
        got = (ref[:, np.asarray(P.perm)] if op == H.OP_Z else ref[:, into])[CHECKED]
        err = np.abs(got - want).astype(float)
        assert np.all(err <= np.sqrt(2) * 2 * (2 * P.n + 32) * 2.0 ** -53 * S), (op, float(np.max(err[S > 0] / S[S > 0])))


def test_small_entries_of_a_vector_keep_their_bits():
    """A product whose vector entries are all 2^-40 of the column's largest one, in a row the largest one is not coupled
    to: two bodies that do not see each other (far blocks of rank 0) beside each other in one vector."""
    P = problem([64, 64, 64, 33], 3)[0]
    P.far_rank = np.zeros_like(P.far_rank)
    P.near_data = P.near_data.copy()
    for t, s, o in zip(P.near_t, P.near_s, P.near_off):
        if (t < 2) != (s < 2):
            m, c = int(P.leaf_ptr[t + 1] - P.leaf_ptr[t]), int(P.leaf_ptr[s + 1] - P.leaf_ptr[s])
            P.near_data[o:o + m * c] = 0
    h = hm.hmat_create(P, ordering=1)
    rng = np.random.default_rng(4)
    X = rng.standard_normal((5, P.n)) + 1j * rng.standard_normal((5, P.n))
    X[:, P.leaf_ptr[2]:] *= 2.0 ** -40
    want, S = exact(P, X)
    err = np.abs(apply(h, H.OP_Z, X) - want).astype(float)
    assert np.all(err <= np.sqrt(2) * 2 * (2 * P.n + 32) * 2.0 ** -53 * S)


@pytest.mark.parametrize("w", [1, 16])
def test_results_below_the_normal_range(w):
    """A subnormal vector entry: products exact to a few units of the last place of the range."""
    P, _, Z = problem(MIXED, 11)
    h = hm.hmat_create(P, ordering=1)
    X = np.zeros((w, P.n), dtype=np.complex128)
    X[:, 40] = 2.0 ** -1040
    y = apply(h, H.OP_Z, X)
    near = np.abs(Z[:, 40]) > 1e-3
    assert np.all(np.abs(y - Z[:, 40] * 2.0 ** -1040)[:, near] <= 64 * 2.0 ** -1074)
