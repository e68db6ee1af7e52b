"""The factorisation, the near-field product and the solver's vector passes on block sizes the meshes do not have: 1 to 64
unknowns side by side (tiles, pieces and chunks of every kernel cut short somewhere), with steps whose next block is
and is not among their updates, and the look-ahead of the setup against the launches in one stream.

The matrices are symmetric, complex, with a dominant diagonal (growth below 2).  Tolerances: FP64 sums of at most
600 terms, 600 u < 7e-14, through explicit inverses of condition below 10: 1e-11.  Complex FP32: the same terms at
u = 6e-8, sqrt(600) u 10 < 1.5e-5, twice that for the panel behind it: 3e-5.
"""
from types import SimpleNamespace

import numpy as np
import pytest
import torch

import paper_2111_13483_gb300 as hm

pytestmark = pytest.mark.gpu
H = hm.hmsolve
MIXED = [1, 2, 3, 31, 32, 33, 63, 64, 4, 5, 7, 8, 9, 15, 16, 17, 24, 25, 29, 64]


def problem(sizes, seed):
    rng = np.random.default_rng(seed)
    lp = np.concatenate([[0], np.cumsum(sizes)])
    n, nl = int(lp[-1]), len(sizes)
    Z = np.zeros((n, n), dtype=np.complex128)
    nt, ns = [], []
    for t in range(nl):
        for s in range(t, nl):
            if not (t == s or (s == t + 1 and t % 3 != 2) or s == t + 4 or (s - t) % 7 == 6):
                continue
            nt.append(t)
            ns.append(s)
            B = rng.standard_normal((sizes[t], sizes[s])) + 1j * rng.standard_normal((sizes[t], sizes[s]))
            if t == s:
                B = (B + B.T) / 2
            Z[lp[t]:lp[t + 1], lp[s]:lp[s + 1]] = B
            Z[lp[s]:lp[s + 1], lp[t]:lp[t + 1]] = B.T
    near = {(t, s) for t, s in zip(nt, ns)}
    far, U, V, F = [], [], [], np.zeros((n, n), dtype=np.complex128)
    for t in range(nl):
        for s in range(t + 1, nl):   # the other pairs: ranks 0, 1, 2 and dense blocks (-1)
            if (t, s) in near:
                continue
            m, c = sizes[t], sizes[s]
            r = min([0, 1, 2, -1][(t + s) % 4], m, c)
            w = c if r < 0 else r
            u = rng.standard_normal((m, w)) + 1j * rng.standard_normal((m, w))
            v = np.eye(c) if r < 0 else rng.standard_normal((c, w)) + 1j * rng.standard_normal((c, w))
            far.append((lp[t], lp[t + 1], lp[s], lp[s + 1], r, sum(x.size for x in U), sum(x.size for x in V)))
            U.append(u.T.ravel())
            V.append(np.zeros(0, np.complex128) if r < 0 else v.T.ravel())
            F[lp[t]:lp[t + 1], lp[s]:lp[s + 1]] = u @ v.T
            F[lp[s]:lp[s + 1], lp[t]:lp[t + 1]] = v @ u.T
    np.fill_diagonal(Z, 2 * np.sum(np.abs(Z) + np.abs(F), axis=1))
    blocks = [Z[lp[t]:lp[t + 1], lp[s]:lp[s + 1]].T.ravel() for t, s in zip(nt, ns)]
    off = np.concatenate([[0], np.cumsum([b.size for b in blocks])[:-1]])
    far = np.array(far).reshape(-1, 7)
    flat = lambda x: np.concatenate(x + [np.zeros(0, np.complex128)])
    return SimpleNamespace(n=n, perm=np.arange(n), leaf_ptr=lp, near_t=np.array(nt), near_s=np.array(ns), near_off=off,
                           near_data=np.concatenate(blocks), far_r0=far[:, 0], far_r1=far[:, 1], far_c0=far[:, 2],
                           far_c1=far[:, 3], far_rank=far[:, 4], far_uoff=far[:, 5], far_voff=far[:, 6], far_U=flat(U),
                           far_V=flat(V)), Z, Z + F


def blocks_of(h, P):
    size = np.diff(P.leaf_ptr)[hm.hm_get_order(h)]
    ptr, idx = hm.hm_get_fill(h)
    out = []
    for k in range(len(size)):
        nk = int(size[k])
        for kind in (0, 1):
            out.append(hm.hm_get_block(h, kind, k, (nk, nk)))
        if ptr[k + 1] > ptr[k]:
            out.append(hm.hm_get_block(h, 2, k, (nk, int(size[idx[ptr[k]:ptr[k + 1]]].sum()))))
    return out


def factor(P, Z, order, ptr, idx):
    lp = P.leaf_ptr
    A = Z.copy()
    at = [np.arange(lp[l], lp[l + 1]) for l in order]
    out = []
    for k in range(len(order)):
        D = A[np.ix_(at[k], at[k])]
        out += [D, np.linalg.inv(D)]
        if ptr[k + 1] > ptr[k]:
            J = np.concatenate([at[j] for j in idx[ptr[k]:ptr[k + 1]]])
            W = np.linalg.solve(D, A[np.ix_(at[k], J)])
            out.append(W)
            A[np.ix_(J, J)] -= A[np.ix_(J, at[k])] @ W
    return out


@pytest.mark.parametrize("sizes", [MIXED, MIXED[::-1], [1] * 12, [64] * 5, [33, 1, 64, 2]])
@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("ordering", [1, 2])
def test_factor_of_uneven_blocks(sizes, prec, ordering):
    P, Z, _ = problem(sizes, 5)
    h = hm.hmat_create(P, ordering=ordering, precision=prec)
    hm.precond_setup(h)
    got = blocks_of(h, P)
    ref = factor(P, Z, hm.hm_get_order(h), *hm.hm_get_fill(h))
    tol = 3e-5 if prec else 1e-11
    for g, r in zip(got, ref):
        assert np.max(np.abs(g - r)) <= tol * np.max(np.abs(r))
    hm.hm_profile(h, 1)   # timed launches go to one stream
    hm.precond_setup(h)
    hm.hm_profile(h, 0)
    assert all(np.array_equal(a, b) for a, b in zip(got, blocks_of(h, P)))


@pytest.mark.parametrize("sizes", [MIXED, [64] * 8, [64] * 8 + [1], [1, 64, 2, 33]])
def test_products_and_solves_of_uneven_blocks(sizes):
    """The FP64 product at the widths where its kernels change (1 to 64 columns), each column with the bits of the others'
    widths, and solves of n around the 512 entries of one chunk of the vector passes."""
    P, _, Z = problem(sizes, 9)
    h = hm.hmat_create(P, ordering=1)
    hm.precond_setup(h)
    rng = np.random.default_rng(1)
    X = rng.standard_normal((64, P.n)) + 1j * rng.standard_normal((64, P.n))
    want = X @ Z.T   # this product takes and gives the original order
    ref = None
    for w in (64, 1, 3, 4, 5, 8, 16, 17):
        x = torch.from_numpy(X[:w]).cuda()
        y = torch.empty_like(x)
        hm.hm_apply(h, H.OP_Z, x, y)
        y = y.cpu().numpy()
        ref = y if ref is None else ref
        assert np.array_equal(y, ref[:w])
    assert np.max(np.abs(ref - want)) <= 1e-13 * np.max(np.abs(want))
    B = rng.standard_normal((P.n, 3)) + 1j * rng.standard_normal((P.n, 3))
    I, its, rr, code = hm.solve(h, B, tol=1e-10, restart=20)
    assert code == 0
    assert np.all(np.linalg.norm(B - Z @ I, axis=0) <= 2e-10 * np.linalg.norm(B, axis=0))


@pytest.mark.parametrize("sizes", [MIXED, [32] * 9, [33] * 9, [1, 64, 2, 33, 5, 6, 7, 8, 9, 10]])
def test_far_field_widths(sizes):
    """The complex-FP32 far field where its kernels change (16 / 17 columns, even and odd widths, blocks of one and of two
    row patches): the bits of every column at every width, and 1e-5 (600 terms, sqrt(600) u 5) of the exact product."""
    P, N, Z = problem(sizes, 3)
    h = hm.hmat_create(P, ordering=1, precision=1)
    hm.precond_setup(h)
    rng = np.random.default_rng(2)
    X = rng.standard_normal((64, P.n)) + 1j * rng.standard_normal((64, P.n))
    p = np.asarray(hm.hm_get_index_map(h))
    F = (Z - N)[np.ix_(p, p)]
    np.fill_diagonal(F, 0)
    ref = None
    for w in (64, 4, 16, 17, 18, 23, 32, 33, 48, 49, 63):
        x = torch.from_numpy(X[:w]).cuda()
        y = torch.empty_like(x)
        hm.hm_apply(h, H.OP32 + H.OP_ZF, x, y)
        y = y.cpu().numpy()
        ref = y if ref is None else ref
        assert np.array_equal(y, ref[:w])
    want = X @ F.T
    assert np.max(np.abs(ref - want)) <= 1e-5 * np.max(np.abs(want))


def apply_z(h, X, op=H.OP_Z):
    x = torch.from_numpy(X).cuda()
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    hm.hm_apply(h, op, x, y)
    torch.cuda.synchronize()
    return y.cpu().numpy()


@pytest.mark.parametrize("w", [1, 4, 5, 16])
def test_split_product_scales_exactly_and_keeps_columns_apart(w):
    """The digits of a column follow its largest exponent: a power of two in front comes out exactly, also far from 1, and a
    NaN or an infinity spoils its own column only."""
    P, _, Z = problem(MIXED, 11)
    h = hm.hmat_create(P, ordering=1)
    rng = np.random.default_rng(4)
    X = rng.standard_normal((w, P.n)) + 1j * rng.standard_normal((w, P.n))
    y = apply_z(h, X)
    for k in (-600, -60, 60, 600):
        assert np.array_equal(apply_z(h, np.ldexp(X.real, k) + 1j * np.ldexp(X.imag, k)),
                              np.ldexp(y.real, k) + 1j * np.ldexp(y.imag, k))
    assert np.all(apply_z(h, 0 * X) == 0)
    for bad in (np.nan, np.inf):
        B = X.copy()
        B[w - 1, 7] = bad
        z = apply_z(h, B)
        assert np.array_equal(z[:w - 1], y[:w - 1]) and not np.any(np.isfinite(z[w - 1].real))
    assert np.array_equal(apply_z(h, X), y)


@pytest.mark.parametrize("w", [1, 16])
def test_split_product_of_leaves_without_far_blocks(w):
    """Four leaves, the second of them in no far block but one of rank 0: its rows of the far product are 0, for every
    size of the vector, zero included."""
    P, N, Z = problem([33, 1, 64, 2], 11)
    h = hm.hmat_create(P, ordering=1)
    rng = np.random.default_rng(4)
    p = np.asarray(hm.hm_get_index_map(h))
    row = int(np.argwhere(p == 33)[0, 0])
    X = rng.standard_normal((w, P.n)) + 1j * rng.standard_normal((w, P.n))
    for scale in (0.0, 1e-280, 1.0, 1e280):
        y = apply_z(h, scale * X, H.OP_ZF)
        assert np.all(np.isfinite(y)) and np.all(y[:, row] == 0)
        assert scale != 0.0 or np.all(y == 0)
