"""Adaptive solves go through the captured step once a hierarchy has stopped
changing: a solve without reintroductions on a hierarchy that was solved with
before launches a few kernels a window from the host, not every kernel of
every step."""
import pytest

import amg_inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k_check", [1, 3, 4, 5])
@pytest.mark.parametrize("krylov", [0, 1])
def test_windows_without_resets_use_the_graph(krylov, k_check):
    """A step is some twenty kernels (four levels and the Krylov updates); a
    window's own -- residuals, restarts -- are at most ten."""
    from paper_1512_04629_gb300 import amg

    A = gen.poisson2d_5pt(64)
    b = gen.rhs_uniform(A.n, 3)
    h = amg.Hierarchy.setup(A, krylov=krylov, k_check=k_check)
    launched, steps, xs = [], [], []
    for _ in range(3):
        before = amg.kernel_launches()
        x, info = h.solve(b, tol=1e-8, adaptive=True)
        launched.append(amg.kernel_launches() - before)
        assert info.status == 0 and info.resets == 0
        steps.append(info.iterations)
        xs.append(x)
    assert steps[0] == steps[1] == steps[2]
    windows = -(-steps[0] // k_check)
    assert launched[1] <= 10 * windows + 10 and launched[2] <= 10 * windows + 10, (launched, windows)
    # the same kernels in the same order, with a graph or without one
    assert (xs[0] == xs[1]).all() and (xs[0] == xs[2]).all()
