"""hbm_budget and the two-level data of the sweeps: when there is room for them, and what a call that does not fit, and
one that fits only in their place, leave behind."""
import numpy as np
import pytest
import torch

import efie_problem as ep
import paper_2111_13483_gb300 as hm
from test_gpu_setup_blocks import problem

pytestmark = pytest.mark.gpu
H = hm.hmsolve
MESH = dict(kind="sphere", d=2, a=0.3, leaf=64, eta=1.0, aca_eps=1e-3)   # one super-row, larger than the elimination's workspace


def used(h):
    return hm.hmat_stats(h)["device_bytes"]


def sweep(h, prec, X):
    x = torch.from_numpy(X).cuda()
    y = torch.empty_like(x)
    hm.hm_apply(h, (H.OP32 if prec else 0) + H.OP_LINV, x, y)
    return y.cpu().numpy()


def sizes(P, prec, fill_tol=0.0):
    """Bytes after a setup and the operator's workspace of one column; a vector; L^{-1} of it by both sweeps."""
    g = hm.hmat_create(P, ordering=1, precision=prec, fill_tol=fill_tol)
    hm.precond_setup(g)
    full = used(g)
    rng = np.random.default_rng(4)
    X = rng.standard_normal((1, P.n)) + 1j * rng.standard_normal((1, P.n))
    two = sweep(g, prec, X)
    work = used(g) - full
    H.hm_set_sweep_schedule(g, 1, 1, 0)
    return full, work, X, two, sweep(g, prec, X)


@pytest.mark.parametrize("prec,fill_tol", [(0, 0.0), (1, 0.0), (1, 1e-2)])
def test_a_budget_of_the_steady_state_keeps_the_two_level_sweeps(prec, fill_tol):
    """What the handle holds after a setup is smaller than what the elimination takes on the way (its workspace); a budget
    that holds either has room for the sweeps' data, also in a second setup (which, with compressed coefficients, has
    their store beside the elimination)."""
    P = ep.build(dict(MESH, d=3, a=0.6))
    full, work, X, two, one = sizes(P, prec, fill_tol)
    assert not np.array_equal(two, one)
    g = hm.hmat_create(P, ordering=1, precision=prec, fill_tol=fill_tol)
    before = used(g)   # the elimination: its workspace beside the dense coefficients and the diagonal blocks, twice
    f = hm.hmat_stats(g)
    c, d = f["coef_entries_dense"], f["diag_entries"]
    elimination = before + (16 * (2 * c + 2 * d) if prec == 0 else 8 * (2 * c + 2 * d) + 16 * d)
    h = hm.hmat_create(P, ordering=1, precision=prec, fill_tol=fill_tol, hbm_budget=max(elimination, full) + work + 8192)
    for _ in range(1 if fill_tol else 2):
        hm.precond_setup(h)
        assert np.array_equal(sweep(h, prec, X), two)


@pytest.mark.parametrize("prec", [0, 1])
def test_refused_call_leaves_the_sweeps(prec):
    P = ep.build(MESH)
    full, work, X, two, one = sizes(P, prec)
    assert not np.array_equal(two, one)
    h = hm.hmat_create(P, ordering=1, precision=prec, hbm_budget=full + work + 4096)
    hm.precond_setup(h)
    assert np.array_equal(sweep(h, prec, X), two)
    before = used(h)
    with pytest.raises(Exception):
        hm.Batch(h, 1024, 50)
    V = np.zeros((P.n, 64), dtype=np.complex128)
    with pytest.raises(Exception):
        hm.solve(h, V, tol=1e-6, restart=2000)
    assert used(h) == before
    assert np.array_equal(sweep(h, prec, X), two)


@pytest.mark.parametrize("prec", [0, 1])
def test_sweeps_come_back_after_a_batch(prec):
    P = ep.build(MESH)
    full, work, X, two, one = sizes(P, prec)
    engine = hm.Batch.bytes(h := hm.hmat_create(P, ordering=1, precision=prec), 1, 5)
    hm.hmat_destroy(h)
    h = hm.hmat_create(P, ordering=1, precision=prec, hbm_budget=full + work + engine // 2)
    hm.precond_setup(h)
    assert np.array_equal(sweep(h, prec, X), two)
    before = used(h)
    b = hm.Batch(h, 1, 5)                      # fits only in the place of the two-level data
    assert np.array_equal(sweep(h, prec, X), one)
    V = P.plane_wave([0.0, 0.0, -1.0], [1.0, 0.0, 0.0])
    b.submit(V, tol=1e-4)
    fin = []
    while not fin:
        fin = b.step()
    assert b.result(fin[0])[3] == 0
    b.close()
    assert used(h) == before
    assert np.array_equal(sweep(h, prec, X), two)
    x, it, rr, code = hm.solve(h, V, tol=1e-4, restart=5)   # the same for a solve
    assert code == 0 and used(h) == before
    assert np.array_equal(sweep(h, prec, X), two)


@pytest.mark.parametrize("sizes_", [[64], [64, 33], [5, 40, 64, 17]])
def test_a_schedule_set_later_takes_the_place_of_the_two_level_data(sizes_):
    """A few blocks, whose two-level data are little more than their hand-over buffers: the words of the sweeps that are
    asked for fit in their place."""
    P = problem(sizes_, 3)[0]
    g = hm.hmat_create(P, ordering=1, precision=1)
    hm.precond_setup(g)
    rng = np.random.default_rng(4)
    X = rng.standard_normal((1, P.n)) + 1j * rng.standard_normal((1, P.n))
    two = sweep(g, 1, X)
    full = used(g)
    H.hm_set_sweep_schedule(g, 1, 1, 0)
    one = sweep(g, 1, X)
    h = hm.hmat_create(P, ordering=1, precision=1, hbm_budget=full)
    hm.precond_setup(h)
    assert np.array_equal(sweep(h, 1, X), two)
    H.hm_set_sweep_schedule(h, 1, 1, 0)
    assert np.array_equal(sweep(h, 1, X), one)
