"""Dense blocks whose tiles are joined, cut and dealt out in items: the entries against the input generator's host code
at the sizes where a tile starts or ends (128 rows, 64 columns, 256 joined columns, items of 256 entries)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,widths", [
    (1, [1, 1, 255, 1, 256, 257]),          # joined up to, and one past, 256 columns
    (16, [16, 16, 16, 64, 65, 128]),        # items of exactly 256 entries; a block cut into columns, then joined to
    (128, [64, 64, 128, 3]),                # the tallest block that joins
    (129, [64, 65, 1]),                     # one row more: cut, never joined
    (300, [5, 130]),
])
@pytest.mark.parametrize("scratch", [0, 1])
def test_joined_and_cut_tiles(sphere480, m, widths, scratch):
    """Blocks with the same rows next to each other, between blocks with others; scratch = 1 byte puts every block into
    a chunk of its own.  Both sides sum the same 49-point rule and closed forms in FP64: 1e-12 of the largest entry,
    the bound of the other fill tests."""
    import efie_problem.builder as B
    from paper_2111_13483_gb300 import hmsolve as H
    P = sphere480
    rng = np.random.default_rng(m)
    r0, r1 = rng.integers(0, P.n, m), rng.integers(0, P.n, m)
    rows, cols = [], []
    for r in (r0, r1, r0):
        for w in widths:
            rows.append(r)
            cols.append(rng.integers(0, P.n, w))
    mesh = H.Mesh(P.rwg.V, P.rwg.T, P.rwg.tri, P.rwg.free, B.K0, B.ETA0)
    out, off = H.hm_efie_fill(mesh, rows, cols, scratch_bytes=scratch)
    ref, roff = B.EntryEvaluator(P.rwg).blocks(rows, cols)
    assert np.array_equal(off, roff)
    assert np.max(np.abs(out - ref)) <= 1e-12 * np.max(np.abs(ref))


@pytest.mark.parametrize("k", [1e-3, 2.0, 4e5])
def test_phase_of_every_size(sphere480, k):
    """Wave numbers from kR << 1 (the limit of the extracted kernel) to kR > 1e5 (past the reduced argument).  The phase
    of an entry carries some eight roundings of coordinates up to 1 and distances up to 2 on either side, each 2^-53 k
    times that: 1e-12 + 2e-15 k of the largest."""
    import efie_problem.builder as B
    from paper_2111_13483_gb300 import hmsolve as H
    P = sphere480
    rng = np.random.default_rng(7)
    rows, cols = [rng.integers(0, P.n, 40)], [rng.integers(0, P.n, 40)]
    mesh = H.Mesh(P.rwg.V, P.rwg.T, P.rwg.tri, P.rwg.free, k, B.ETA0)
    out, _ = H.hm_efie_fill(mesh, rows, cols)
    ref, _ = B.EntryEvaluator(P.rwg, k=k).blocks(rows, cols)
    assert np.max(np.abs(out - ref)) <= (1e-12 + 2e-15 * k) * np.max(np.abs(ref))
