"""The batched passes where they can go wrong: row lengths around the number
of entries taken together, row counts ragged against blocks, every width, and
the FP32 <-> FP64 conversions at both ends of FP32's range."""
import numpy as np
import pytest
import scipy.sparse as sp

import amg_inputs as gen

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def amg():
    import paper_1512_04629_gb300.amg as m

    return m


def _band(n, half):
    """2 half + 1 entries a row (fewer at the ends), strictly dominant."""
    offs = range(-half, half + 1)
    return sp.diags([np.full(n - abs(o), 2.0 * half + 1.0 if o == 0 else -1.0) for o in offs], list(offs)).tocsr()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n,half,k", [(997, 1, 1), (997, 2, 8), (4099, 3, 9), (513, 4, 17), (2053, 3, 33), (300, 5, 64)])
def test_batch_matches_single_solves(amg, n, half, k, precision):
    """Every column equals its own single solve.  A's eigenvalues lie in
    [1, 4 half + 1], so relative residuals of 1e-10 leave the two solutions
    within 2 (4 half + 1) 1e-10 of each other."""
    A = _band(n, half)
    B = np.stack([gen.rhs_uniform(n, 20 + c) for c in range(k)], 1)
    h = amg.Hierarchy.setup(A, max_size=20, gamma=[0.0, 0.1], precision=precision)
    assert h.num_levels >= 3
    X, infos = h.solve_batch(B, tol=1e-10)
    for c in sorted({0, k // 2, k - 1}):
        x, info = h.solve(np.ascontiguousarray(B[:, c]), tol=1e-10)
        assert info.status == 0 and infos[c].status == 0 and infos[c].final_relres <= 1e-10
        assert np.linalg.norm(X[:, c] - x) <= 2 * (4 * half + 1) * 1e-10 * np.linalg.norm(x)


@pytest.mark.parametrize("k", [3, 16, 40])
def test_conversions_at_the_ends_of_fp32(amg, k):
    """A = I, one level: the FP32 cycle returns its rounded input, so one step
    gives a right-hand side that FP32 holds exactly -- subnormals, the smallest
    and the largest normal numbers, both zeros -- to the bit, and any other
    within its second step's rounding."""
    n = 64
    A = sp.identity(n, format="csr")
    rng = np.random.default_rng(3)
    tiny = float(np.finfo(np.float32).tiny)
    exact = [rng.integers(-5000, 5000, n) * 2.0 ** -149, np.where(np.arange(n) % 2, tiny, -tiny),
             np.where(np.arange(n) % 3, 3.0, -0.0), rng.standard_normal(n).astype(np.float32).astype(np.float64),
             np.full(n, 2.0 ** 60)]
    rounded = [rng.standard_normal(n) * s for s in (1e-20, 1.0, 1e20)]
    cols = [(exact + rounded)[c % 8] for c in range(k)]
    B = np.stack(cols, 1)
    h = amg.Hierarchy.setup(A, precision=1)
    X, infos = h.solve_batch(B, tol=1e-8)
    for c in range(k):
        assert infos[c].status == 0
        if c % 8 < len(exact):
            np.testing.assert_array_equal(X[:, c], B[:, c])
        else:
            assert np.linalg.norm(X[:, c] - B[:, c]) <= 1e-8 * np.linalg.norm(B[:, c])
