"""The two-level sweeps (the default) against the one-row-per-CTA kind at the edges of their column
groups (1; 4; 8 columns), with dense and compressed coefficients, a ragged mesh and the Sloan order,
and their fallback when the handle's budget has no room for their data.

Tolerances: both sum the same products in another order, through the inverse of a super-row's unit
triangle.  FP64: 1e-12.  Complex FP32: each side is within sqrt(terms) u growth of the exact sweep,
about sqrt(3000) * 6e-8 * 5 = 1.6e-5; 5e-5 for their difference.
"""
import numpy as np
import pytest
import torch

import efie_problem as ep
import paper_2111_13483_gb300 as hm

pytestmark = pytest.mark.gpu
H = hm.hmsolve


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _apply(h, op, X):
    dx = torch.from_numpy(X).cuda()
    dy = torch.empty_like(dx)
    hm.hm_apply(h, op, dx, dy)
    return dy.cpu().numpy()


@pytest.mark.parametrize("mesh,ordering,fill_tol", [("plate_tiny", 1, 0.0), ("sphere1920", 1, 0.0), ("sphere1920", 2, 1e-2),
                                                    ("plate1160", 1, 1e-2)])
@pytest.mark.parametrize("prec", [0, 1])
def test_against_one_row_per_cta(mesh, ordering, fill_tol, prec):
    P = ep.build(mesh)
    h = hm.hmat_create(P, ordering=ordering, fill_tol=fill_tol, precision=prec)
    hm.precond_setup(h)
    rng = np.random.default_rng(3)
    X = rng.standard_normal((64, P.n)) + 1j * rng.standard_normal((64, P.n))
    off = H.OP32 if prec else 0
    for op in (H.OP_LINV, H.OP_LTINV):
        full = _apply(h, off + op, X)
        H.hm_set_sweep_schedule(h, 1, 1, 0)
        ref = _apply(h, off + op, X)
        H.hm_set_sweep_schedule(h, 0, 0)
        for c in range(64):
            assert rel(full[c], ref[c]) < (5e-5 if prec else 1e-12), (op, c)
        for n in (1, 2, 4, 5, 16, 17, 33):      # a column's bits do not depend on the batch
            assert np.array_equal(_apply(h, off + op, X[:n]), full[:n]), (op, n)


def test_budget_without_room_falls_back():
    # one super-row (8 leaves): its data are larger than the setup's workspace, so a budget between the two exists
    P = ep.build(dict(kind="sphere", d=2, a=0.3, leaf=64, eta=1.0, aca_eps=1e-3))
    g = hm.hmat_create(P, ordering=1)
    hm.precond_setup(g)
    full = hm.hmat_stats(g)["device_bytes"]
    H.hm_set_sweep_schedule(g, 1, 1, 0)
    rng = np.random.default_rng(4)
    X = rng.standard_normal((1, P.n)) + 1j * rng.standard_normal((1, P.n))
    ref = _apply(g, H.OP_LINV, X)
    h = hm.hmat_create(P, ordering=1, hbm_budget=full - 1)
    hm.precond_setup(h)
    assert hm.hmat_stats(h)["device_bytes"] < full - 1
    assert np.array_equal(_apply(h, H.OP_LINV, X), ref)
    # room at the setup, none left for the solve's workspace: the sweeps give theirs back
    h = hm.hmat_create(P, ordering=1, hbm_budget=full + 65536)
    hm.precond_setup(h)
    b = P.plane_wave([0.0, 0.0, -1.0], [1.0, 0.0, 0.0])
    x, it, rr, code = hm.solve(h, b, tol=1e-6)
    assert code == 0
    assert rel(x, hm.solve(g, b, tol=1e-6)[0]) < 1e-8
