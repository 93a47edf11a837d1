"""Batched solves over rows of every length around the entries that a pass takes
together: 4 at a time, then 2, then 1."""
import numpy as np
import pytest
import scipy.sparse as sp

import amg_inputs as gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ring(n, length):
    """A circulant with `length` entries in every row: the diagonal, pairs of
    neighbours and, for even lengths, the entry opposite.  Strictly dominant,
    eigenvalues in [1, 2 length - 1]."""
    i = np.arange(n)
    offs = [0] + [s * k for k in range(1, (length - 1) // 2 + 1) for s in (1, -1)]
    if length % 2 == 0:
        offs.append(n // 2)
    rows = np.concatenate([i for _ in offs])
    cols = np.concatenate([(i + o) % n for o in offs])
    vals = np.concatenate([np.full(n, float(length) if o == 0 else -1.0) for o in offs])
    A = sp.csr_matrix((vals, (rows, cols)), shape=(n, n))
    A.sort_indices()
    assert (np.diff(A.indptr) == length).all()
    return A


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("length", [1, 2, 3, 4, 5, 6, 7, 8, 10])
def test_every_row_length(length, precision):
    """Against the dense solution: relative residuals of 1e-10 leave it within
    (2 length - 1) 1e-10."""
    import paper_1512_04629_gb300.amg as amg

    n, k = 500, 9
    A = _ring(n, length)
    B = np.stack([gen.rhs_uniform(n, 40 + c) for c in range(k)], 1)
    h = amg.Hierarchy.setup(A, max_size=20, precision=precision)
    X, infos = h.solve_batch(B, tol=1e-10)
    ref = np.linalg.solve(A.toarray(), B)
    for c in range(k):
        assert infos[c].status == 0
        assert np.linalg.norm(X[:, c] - ref[:, c]) <= 2 * length * 1e-10 * np.linalg.norm(ref[:, c])
