"""Which finest operators are stored by row patterns, by the bytes that level 0
is charged -- a byte per row and npat * (width + 1) entries for a stored one,
its CSR arrays for any other -- and the stored form at sizes whose blocks take
more than one round of rows, ragged in the last, bit for bit against one lane
per row."""
import numpy as np
import pytest
import scipy.sparse as sp

import amg_inputs as gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
CSR1 = 7


@pytest.fixture(scope="module")
def amg():
    import paper_1512_04629_gb300.amg as m

    return m


def _two_level(amg, A, **opts):
    """A over 40 piecewise-constant aggregates: level 0 is all that relaxes."""
    n, nc = A.shape[0], 40
    P = sp.csr_matrix((np.ones(n), (np.arange(n), np.arange(n) * nc // n)), shape=(n, nc))
    Ac = (P.T @ A @ P).tocsr()
    Ac.sort_indices()
    cf = np.full(n, -1, np.int8)
    cf[:nc] = 1
    return amg.Hierarchy.assemble([A, Ac], [P], [cf], [None, np.zeros(Ac.nnz, np.uint8)], **opts)


def _classes(n, k):
    """Tridiagonal with k distinct interior diagonals: k + 2 distinct rows."""
    d = 4.0 + (np.arange(n) % k) * 2.0 ** -12
    d[0] = d[-1] = 4.0
    return sp.diags([-np.ones(n - 1), d, -np.ones(n - 1)], [-1, 0, 1]).tocsr()


def _band(n, half):
    offs = list(range(-half, half + 1))
    return sp.diags([np.full(n - abs(o), 2.0 * half + 1 if o == 0 else -1.0) for o in offs], offs).tocsr()


def _wide_classes(n, k, half):
    """A band with k distinct interior diagonals, half rows at either end of their own."""
    A = _band(n, half).tolil()
    d = 2.0 * half + 1 + (np.arange(n) % k) * 2.0 ** -12
    d[:half] = d[-half:] = 2.0 * half + 1
    A.setdiag(d)
    return A.tocsr()


def _distinct_rows(A):
    """(rows that differ in offsets or values, longest row), with numpy alone."""
    seen, width = set(), 0
    for i in range(A.shape[0]):
        p, q = A.indptr[i], A.indptr[i + 1]
        seen.add((A.indices[p:q] - i).tobytes() + A.data[p:q].tobytes())
        width = max(width, q - p)
    return len(seen), width


# name: (matrix, distinct rows when stored or 0)
CASES = {
    "2d5_71": (lambda: gen.poisson2d_5pt(71).to_scipy(), 9),
    "3d7_17": (lambda: gen.poisson3d_7pt(17).to_scipy(), 27),
    "3d27_33": (lambda: gen.poisson3d_27pt(33).to_scipy(), 27),
    "most_patterns": (lambda: _classes(8000, 253), 255),
    "one_pattern_too_many": (lambda: _classes(8000, 254), 0),
    "longest_row": (lambda: _band(32800, 15), 31),
    "rows_too_long": (lambda: _band(32800, 16), 0),
    # the FP64 table takes 12 (width + 1) bytes a pattern and may take 12,288: 85 rows of up to 11 entries
    "largest_table": (lambda: _wide_classes(33000, 75, 5), 85),
    "table_too_large": (lambda: _wide_classes(33000, 76, 5), 0),
    "long_rows_small_grid": (lambda: gen.poisson3d_27pt(13).to_scipy(), 0),
    "few_entries": (lambda: gen.poisson2d_5pt(60).to_scipy(), 0),
    "lognormal": (lambda: gen.fv7_lognormal(17, seed=3).to_scipy(), 0),
}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("case", sorted(CASES))
def test_what_is_stored(amg, case, precision):
    A = CASES[case][0]()
    stored = CASES[case][1]
    vb = 8 if precision == 0 else 4
    opts = dict(precision=precision, transfer_variant=CSR1)
    got = [_two_level(amg, A, spmv_variant=v, **opts).level_stats(0)["bytes_per_cycle"] for v in (-1, CSR1)]
    npat, width = _distinct_rows(A)
    if not stored:
        assert got[0] == got[1]
        return
    assert npat == stored
    csr = A.nnz * (vb + 4) + 4 * (A.shape[0] + 1)
    assert got[1] - got[0] == 2 * (csr - A.shape[0] - npat * (width + 1) * (vb + 4))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("make", [lambda: gen.poisson3d_7pt(79).to_scipy(),      # 493,039 rows: three rounds of a wave
                                  lambda: gen.poisson3d_27pt(63).to_scipy(),     # 250,047: two
                                  lambda: _classes(152 * 6 * 256 * 2 + 33, 200),  # a last round of one block and a warp's rest
                                  lambda: _classes(152 * 6 * 256 + 1, 7)], ids=["3d7_79", "3d27_63", "classes_2", "classes_1"])
def test_several_rounds_of_rows(amg, make, precision):
    A = make()
    n = A.shape[0]
    r = torch.from_numpy(gen.rhs_uniform(n, 4)).cuda()
    z = []
    for variant in (-1, CSR1):
        h = _two_level(amg, A, precision=precision, spmv_variant=variant, transfer_variant=CSR1)
        out = torch.zeros_like(r)
        h.precond_apply(r, out)
        z.append((out.cpu().numpy(), h.level_stats(0)["bytes_per_cycle"]))
    assert z[0][1] < z[1][1]  # stored
    np.testing.assert_array_equal(z[0][0], z[1][0])
