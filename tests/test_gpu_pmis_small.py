"""The C/F split of a level of at most 2048 rows (one block, csrc/setup.cu)
against the oracle's, exactly: row counts ragged against the block's sweeps,
at the line and one row past it (the launches of the general form), short and
long rows, rows without strong neighbours, and weights that need many rounds.
The coarse numbering is checked through P and the coarse operator."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amg():
    import paper_1512_04629_gb300.amg as m

    return m


def _chain(n):
    return sp.diags([-np.ones(n - 1), np.full(n, 2.0), -np.ones(n - 1)], [-1, 0, 1]).tocsr()


def _random(n, per_row, seed=0):
    """Symmetric M-matrix of about per_row entries a row."""
    rng = np.random.default_rng(seed)
    m = n * (per_row - 1) // 2
    i, j = rng.integers(0, n, m), rng.integers(0, n, m)
    w = rng.uniform(0.2, 1.0, m)
    B = sp.coo_matrix((w[i != j], (i[i != j], j[i != j])), shape=(n, n)).tocsr()
    B = B + B.T
    A = (sp.diags(np.asarray(B.sum(axis=1)).ravel() + 0.1) - B).tocsr()
    A.sort_indices()
    return A


def _isolated(n):
    """A chain with every fifth row on its own (no strong neighbour: F)."""
    A = _chain(n).tolil()
    for i in range(0, n, 5):
        for j in (i - 1, i + 1):
            if 0 <= j < n:
                A[i, j] = A[j, i] = -1e-9
    return A.tocsr()


CASES = {
    "chain_37": lambda: _chain(37),
    "chain_2047": lambda: _chain(2047),
    "chain_2048": lambda: _chain(2048),
    "chain_2049": lambda: _chain(2049),
    "isolated_513": lambda: _isolated(513),
    "random_257_6": lambda: _random(257, 6),
    "random_1025_14": lambda: _random(1025, 14),
    "random_129_100": lambda: _random(129, 100),
    "random_2048_30": lambda: _random(2048, 30),
    "random_2049_30": lambda: _random(2049, 30),
}


@pytest.mark.parametrize("case", list(CASES))
def test_small_level_split(amg, case):
    A = CASES[case]()
    A.sort_indices()
    opts = dict(max_size=16, max_levels=3, seed=11)
    ref = oracle.Hierarchy(A, **opts)
    h = amg.Hierarchy.setup(A, **opts)
    assert h.num_levels == ref.num_levels
    for l in range(h.num_levels - 1):
        np.testing.assert_array_equal(h.level_array(l, "cf"), ref.cf(l), err_msg=f"cf_{l}")
        got, want = h.export(l, "P"), ref.matrix(l, "P")
        np.testing.assert_array_equal(got.rowptr, want.rowptr)
        np.testing.assert_array_equal(got.col, want.col)
    last = h.num_levels - 1
    np.testing.assert_array_equal(h.export(last, "A").col, ref.matrix(last, "A").col)
