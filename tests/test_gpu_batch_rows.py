"""Batched solves where the passes' rows divide differently: rows of every
length around the entries taken together (4 at a time, then 2, then 1), and row
counts around the last size of one wave of blocks and the first of two."""
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


@pytest.mark.parametrize("precision,k", [(1, 64), (1, 33), (0, 64)])
@pytest.mark.parametrize("off", [-1, 0, 1, 517])
def test_row_counts_around_a_second_wave(precision, k, off):
    """Every column against its own single solve, at row counts around 15 steps
    of a wave's blocks, past which ranges of 15 steps in one wave become ranges of
    8 in two.  Eigenvalues of the operator lie in [1, 5]."""
    import paper_1512_04629_gb300.amg as amg

    sms = torch.cuda.get_device_properties(0).multi_processor_count
    # resident blocks times the rows of a step: 512 threads over K / 2 (FP64) or K / 4 lanes a row
    wave = sms * 2 * 16 if precision == 0 else sms * 3 * 32
    n = 15 * wave + off
    A = sp.diags([-np.ones(n - 1), np.full(n, 3.0), -np.ones(n - 1)], [-1, 0, 1]).tocsr()
    gen_b = torch.Generator(device="cuda").manual_seed(9)
    B = torch.rand(n, k, generator=gen_b, device="cuda", dtype=torch.float64) - 0.5
    h = amg.Hierarchy.setup(A, gamma=[0.0, 0.1], precision=precision)
    X, infos = h.solve_batch(B, tol=1e-10)
    for c in (0, k - 1):
        x, info = h.solve(B[:, c].contiguous(), tol=1e-10)
        assert info.status == 0 and infos[c].status == 0
        assert torch.linalg.norm(X[:, c] - x) <= 10 * 1e-10 * torch.linalg.norm(x)
        # and row by row: the residual of every row, the ranges' first and last among them
        r = B[:, c] - 3.0 * X[:, c]
        r[1:] += X[:-1, c]
        r[:-1] += X[1:, c]
        assert torch.linalg.norm(r) <= 2e-10 * torch.linalg.norm(B[:, c])
