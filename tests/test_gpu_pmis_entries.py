"""Which small levels are split in one block: at most 2048 rows and at most
100,000 entries.  One block walks every entry of a sweep on one SM; levels of
more entries are split by launches over the whole device."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ring(n, length):
    """A circulant with `length` entries in every row (even: the opposite one too)."""
    i = np.arange(n)
    offs = [0] + [s * k for k in range(1, (length - 1) // 2 + 1) for s in (1, -1)]
    if length % 2 == 0:
        offs.append(n // 2)
    A = sp.csr_matrix((np.concatenate([np.full(n, float(length) if o == 0 else -1.0) for o in offs]),
                       (np.concatenate([i for _ in offs]), np.concatenate([(i + o) % n for o in offs]))), shape=(n, n))
    A.sort_indices()
    assert A.nnz == n * length
    return A


def test_entries_bound():
    import paper_1512_04629_gb300.amg as amg

    opts = dict(max_size=16, max_levels=2, seed=5)
    launched = []
    for length in (49, 50, 51, 52):  # 98,000 to 104,000 entries
        A = _ring(2000, length)
        before = amg.kernel_launches()
        h = amg.Hierarchy.setup(A, **opts)
        launched.append(amg.kernel_launches() - before)
        ref = oracle.Hierarchy(A, **opts)
        assert h.num_levels == ref.num_levels == 2
        np.testing.assert_array_equal(h.level_array(0, "cf"), ref.cf(0))
        np.testing.assert_array_equal(h.export(0, "P").col, ref.matrix(0, "P").col)
    # by launches: the weights, eight rounds of two, the C flags and their scan
    assert abs(launched[0] - launched[1]) <= 3 and abs(launched[2] - launched[3]) <= 3, launched
    assert min(launched[2:]) >= max(launched[:2]) + 12, launched
