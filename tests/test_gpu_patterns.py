"""The finest operator stored by its distinct rows (csrc/patterns.cu) against
the one-lane CSR kernels, whose row sums run in the same order: one cycle is
the same bits, at sizes ragged against warps, blocks and grids, at the largest
number of patterns and row length, and for the operators just past them, which
keep the general layouts."""
import numpy as np
import pytest
import scipy.sparse as sp

import amg_inputs as gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
SELL32, CSR1 = 6, 7


@pytest.fixture(scope="module")
def amg():
    import paper_1512_04629_gb300.amg as m

    return m


def _classes(n, k, seed=0):
    """Tridiagonal, n rows, with k distinct interior diagonals: the two end
    rows add two patterns, so the operator has k + 2 distinct rows."""
    d = 4.0 + (np.arange(n) % k) * 2.0 ** -12
    d[0] = d[-1] = 4.0
    return sp.diags([-np.ones(n - 1), d, -np.ones(n - 1)], [-1, 0, 1]).tocsr()


def _band(n, half):
    """Rows of up to 2 half + 1 entries."""
    offs = list(range(-half, half + 1))
    return sp.diags([np.full(n - abs(o), 2.0 * half + 1 if o == 0 else -1.0) for o in offs], offs).tocsr()


CASES = {
    # name: (matrix, stored by patterns)
    "2d5_71": (lambda: gen.poisson2d_5pt(71).to_scipy(), True),
    "2d5_96": (lambda: gen.poisson2d_5pt(96).to_scipy(), True),
    "3d7_17": (lambda: gen.poisson3d_7pt(17).to_scipy(), True),
    "3d27_13": (lambda: gen.poisson3d_27pt(13).to_scipy(), False),  # long rows, few of them
    "3d27_33": (lambda: gen.poisson3d_27pt(33).to_scipy(), True),
    "q1_33": (lambda: gen.q1_laplace3d(33).to_scipy(), True),
    "aniso_67": (lambda: gen.rotated_aniso_q1(67).to_scipy(), True),
    "one_row_short_of_a_block": (lambda: _classes(8191, 3), True),
    "most_patterns": (lambda: _classes(8000, 253), True),
    "one_pattern_too_many": (lambda: _classes(8000, 254), False),
    "longest_row": (lambda: _band(32800, 15), True),
    "rows_too_long": (lambda: _band(32800, 16), False),
    "lognormal": (lambda: gen.fv7_lognormal(17, seed=3).to_scipy(), False),
}


def _two_level(amg, A, **opts):
    """A over 40 piecewise-constant aggregates: level 0 is all that relaxes."""
    n, nc = A.shape[0], 40
    P = sp.csr_matrix((np.ones(n), (np.arange(n), np.arange(n) * nc // n)), shape=(n, nc))
    Ac = (P.T @ A @ P).tocsr()
    Ac.sort_indices()
    cf = np.full(n, -1, np.int8)
    cf[:nc] = 1
    return amg.Hierarchy.assemble([A, Ac], [P], [cf], [None, np.zeros(Ac.nnz, np.uint8)], **opts)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("case", sorted(CASES))
def test_cycle_equals_one_lane_rows(amg, case, precision):
    make, stored = CASES[case]
    A = make()
    n = A.shape[0]
    r = torch.from_numpy(gen.rhs_uniform(n, 4)).cuda()
    z = []
    for variant in (-1, CSR1):
        h = _two_level(amg, A, precision=precision, spmv_variant=variant, transfer_variant=CSR1)
        if variant == -1 and stored:
            assert h.level_stats(0)["spmv_variant"] == SELL32
        out = torch.zeros_like(r)
        h.precond_apply(r, out)
        z.append(out.cpu().numpy())
    if stored:
        np.testing.assert_array_equal(z[0], z[1])
    else:  # whatever layout the trials chose: row sums in another order
        tol = 1e-13 if precision == 0 else 1e-5
        assert np.linalg.norm(z[0] - z[1]) <= tol * np.linalg.norm(z[1])


@pytest.mark.parametrize("krylov", [0, 1])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("case", ["2d5_71", "3d7_17", "most_patterns"])
def test_solve_matches_one_lane_rows(amg, case, precision, krylov):
    """The reducing kernels (A p with p . q, the true residual, the
    post-smoothing with r . z) by patterns: the same iterations and, to
    rounding, the same solution."""
    A = CASES[case][0]()
    b = gen.rhs_uniform(A.shape[0], 5)
    got = []
    for variant in (-1, CSR1):
        h = amg.Hierarchy.setup(A, gamma=[0.0, 0.1], precision=precision, krylov=krylov, spmv_variant=variant)
        x, info = h.solve(b, tol=1e-8)
        assert info.status == 0 and info.final_relres <= 1e-8
        got.append((x, info.iterations))
    assert got[0][1] == got[1][1]
    assert np.linalg.norm(got[0][0] - got[1][0]) <= 1e-9 * np.linalg.norm(got[1][0])
