"""GPU test of the exactly diagonalised sectors (k_ft_exact, csrc/ftlm.cu) with couplings near the square root of
binary64's smallest numbers: the rotations stay orthogonal, so the weights of a start vector sum to one."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("weak", [1e-150, 1e-154, 3e-158, 1e-160, 1e-161, 3e-162, 1e-170, 1e-300])
def test_weights_sum_to_one(weak):
    """One bond of 1 and a ring of weak ones: states without the strong bond's spins are degenerate to the last bit
    and coupled by weak elements alone.  The weights round as the exact sectors' test bounds them."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0706_3293_gb300 import api
    n, steps = 10, 50
    u = np.concatenate([[0], np.arange(n)])
    v = np.concatenate([[1], (np.arange(n) + 1) % n])
    J = np.concatenate([[-1.0], np.full(n, -weak)])
    run = api.ftlm_run(n, api.BondList.make(u, v, J), 4, steps, 3, [1.0])
    for A in range(n + 1):
        dim = math.comb(n, A)
        if dim > steps:
            continue
        tol = 160 * dim * np.finfo(float).eps
        for r in range(4):
            assert run.mlen[A, r] == dim
            assert abs(run.tau[A, r, :dim].sum() - 1.0) <= tol, (A, r)
            # levels: the strong bond's -1/4 J (triplet) and 3/4 J (singlet)
            levels = np.array([0.25, -0.75])
            assert np.abs(run.theta[A, r, :dim][:, None] - levels).min(1).max() <= tol
