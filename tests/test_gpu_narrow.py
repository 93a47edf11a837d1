"""The rounding of the FP32 cycle's input (csrc/fp_convert.cuh: narrow) against
numpy's, at the ends of FP32's range.  With A = I on the finest of two levels the
pre-smooth is the rounded input and leaves no residual, so the cycle returns it."""
import numpy as np
import pytest
import scipy.sparse as sp

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TINY, MAX = float(np.finfo(np.float32).tiny), float(np.finfo(np.float32).max)


def _identity(n, precision):
    import paper_1512_04629_gb300.amg as amg

    A = sp.identity(n, format="csr")
    nc = 8
    P = sp.csr_matrix((np.ones(n), (np.arange(n), np.arange(n) * nc // n)), shape=(n, nc))
    Ac = (P.T @ P).tocsr()
    cf = np.full(n, -1, np.int8)
    cf[:nc] = 1
    return amg.Hierarchy.assemble([A, Ac], [P], [cf], [None, np.zeros(Ac.nnz, np.uint8)], precision=precision)


def _edges():
    v = [0.0, -0.0, MAX, np.nextafter(MAX, 0.0), np.nextafter(MAX, np.inf), MAX + 2.0 ** 102, TINY, TINY * (1 - 2.0 ** -25),
         TINY * (1 - 2.0 ** -24), TINY * (1 - 2.0 ** -23), TINY * (1 + 2.0 ** -24), TINY * (1 + 3 * 2.0 ** -24),
         2.0 ** -127, 2.0 ** -149, 2.0 ** -150, np.nextafter(2.0 ** -150, 1.0), 2.0 ** -151, 1.5 * 2.0 ** -149,
         2.5 * 2.0 ** -149, 1e-300, 5e-324]
    for e in (-126, -125, -64, -1, 0, 1, 63, 126):
        for m in (0.0, 2.0 ** -24, np.nextafter(2.0 ** -24, 0), np.nextafter(2.0 ** -24, 1), 2.0 ** -23, 3 * 2.0 ** -24,
                  0.5, 1.0 - 2.0 ** -23, 1.0 - 2.0 ** -24, 1.0 - 2.0 ** -25, np.nextafter(1.0, 0)):
            v.append((1.0 + m) * 2.0 ** e if 1.0 + m < 2.0 else 2.0 ** (e + 1))
            v.append(np.nextafter(2.0 ** (e + 1), 0))
    rng = np.random.default_rng(1)
    v += list(rng.standard_normal(500) * np.exp2(rng.integers(-155, 120, 500)))
    v = np.array(v)
    return np.concatenate([v, -v])


def test_finite_values():
    r = _edges()
    h = _identity(len(r), 1)
    z = torch.empty(len(r), dtype=torch.float64, device="cuda")
    h.precond_apply(torch.from_numpy(r).cuda(), z)
    want = r.astype(np.float32).astype(np.float64)
    assert np.isfinite(want).all()
    np.testing.assert_array_equal(z.cpu().numpy(), want)


@pytest.mark.parametrize("value", [MAX + 2.0 ** 103, 3.5e38, 1e300, np.inf, -np.inf, np.nan])
def test_what_fp32_cannot_hold_is_not_finite(value):
    """The halfway point above the largest number, and all beyond it, round to
    infinity; an infinity or a NaN stays what it is.  Either way the row's
    residual, and so its result, is not finite."""
    r = np.ones(64)
    r[5] = value
    z = torch.zeros(64, dtype=torch.float64, device="cuda")
    _identity(64, 1).precond_apply(torch.from_numpy(r).cuda(), z)
    assert not np.isfinite(z.cpu().numpy()[5])
