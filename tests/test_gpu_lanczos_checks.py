"""The Lanczos checks change from waiting to running ahead at step 32: odd cycles
exhaust the Krylov space at (n - 1) / 2 steps, before, at and behind that step,
and their extreme eigenvalues are cos(2 pi / n) and -cos(pi / n); a limit on the
steps ends a run there."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [9, 17, 55, 61, 63, 65, 67, 71, 73, 75, 101, 131])
def test_odd_cycles(cuda_lib, n):
    from paper_2305_16086_gb300 import Graph

    g = gg.cycle(n)
    with Graph(g.row_ptr, g.col_idx) as G:
        lam = G.estimate_lambda()
    assert abs(lam["lambda_plus"] - np.cos(2 * np.pi / n)) < 1e-12
    assert abs(lam["lambda_minus"] + np.cos(np.pi / n)) < 1e-12
    assert lam["iterations"] == (n - 1) // 2


@pytest.mark.parametrize("steps", [1, 7, 8, 9, 31, 32, 33, 35, 36, 37, 40])
def test_a_limit_on_the_steps(cuda_lib, steps):
    from paper_2305_16086_gb300 import Graph

    g = gg.perturbed_grid(40, 41, 0.05, 2)  # far from converged at 40 steps
    with Graph(g.row_ptr, g.col_idx) as G:
        lam = G.estimate_lambda(max_iter=steps, allow_unconverged=True)
        again = G.estimate_lambda(max_iter=steps, allow_unconverged=True)
    assert lam["iterations"] == steps and lam == again
    assert -1.0 < lam["lambda_minus"] <= lam["lambda_plus"] < 1.0  # Ritz values
