"""The bytes charged to a finest operator stored by row patterns: what the cycle
streams (a byte per row and the table), not the CSR arrays that it does not
read."""
import numpy as np
import pytest

import amg_inputs as gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
CSR1 = 7


@pytest.fixture(scope="module")
def amg():
    import paper_1512_04629_gb300.amg as m

    return m


def _level0(amg, A, precision, variant):
    """(bytes per launch of the level-0 pre- and post-smoothing in precond_apply
    and of A p in a solve, level_stats)."""
    h = amg.Hierarchy.setup(A, gamma=[0.0, 0.1], precision=precision, spmv_variant=variant, transfer_variant=CSR1)
    r = torch.from_numpy(gen.rhs_uniform(A.n, 2)).cuda()
    z = torch.empty_like(r)
    h.timing_enable(True)
    h.precond_apply(r, z)
    got = [h.timing_get(kind, 0) for kind in (amg.K_PRE, amg.K_POST)]
    h.timing_reset()
    h.solve(r, tol=1e-2)
    got.append(h.timing_get(amg.K_AP, 0))
    return [nbytes / launches for launches, _, nbytes in got], h.level_stats(0)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("case,patterns,width", [("3d7_24", 27, 7), ("3d27_33", 27, 27), ("lognormal_24", 0, 0)])
def test_level0_bytes(amg, case, precision, patterns, width):
    A = {"3d7_24": lambda: gen.poisson3d_7pt(24), "3d27_33": lambda: gen.poisson3d_27pt(33),
         "lognormal_24": lambda: gen.fv7_lognormal(24, seed=3)}[case]()
    n, vb = A.n, 8 if precision == 0 else 4

    def operator(value_bytes, stored):
        if stored:
            return n + patterns * (width + 1) * (value_bytes + 4)
        return A.nnz * (value_bytes + 4) + 4 * (n + 1)

    auto, stats = _level0(amg, A, precision, -1)
    lanes, lanes_stats = _level0(amg, A, precision, CSR1)
    for got, stored in ((auto, patterns > 0), (lanes, False)):
        assert got[1] == operator(vb, stored) + 4 * n * vb  # x, b, 1 / diagonal, output
        assert got[2] == operator(8, stored) + 16 * n
        assert got[0] in (operator(vb, stored) + 3 * n * vb, operator(vb, stored) + 4 * n * vb)
    saved = 2 * (operator(vb, False) - operator(vb, patterns > 0))
    assert lanes_stats["bytes_per_cycle"] - stats["bytes_per_cycle"] == saved
