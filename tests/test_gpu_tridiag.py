"""GPU tests of the tridiagonal eigensolvers (csrc/tridiag.cuh, the Ritz values of lanczos_run, and
the finite-temperature eigen-decomposition) at the edges of their 32-row chunks."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from paper_0706_3293_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0706_3293_gb300 import api
    return api


@pytest.mark.parametrize("m", [1, 2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 130])
def test_ritz_values_vs_lapack(hm, m):
    """Every Ritz value of T_m (up to 64 of them) against LAPACK on the returned alpha, beta, ghosts
    included.  Bound: the minors' rounding perturbs the entries of T by at most 7 eps of its
    Gershgorin bound, the bracket adds one eps, LAPACK's own error is at most m eps."""
    inst = W.small_ring(14, -1.0, -0.4)
    b = hm.Basis(inst.n_sites, inst.two_s, inst.two_m)
    r = hm.lanczos_run(b, hm.bonds_of(inst), m, seed=5, n_ritz=min(m + 2, 64))
    al, be = r.alpha, r.beta
    assert r.steps_done == m
    T = np.diag(al) + np.diag(be[: m - 1], 1) + np.diag(be[: m - 1], -1)
    ref = np.linalg.eigvalsh(T)
    n = min(m, 64)
    bound = np.abs(T).sum(1).max()
    assert np.abs(r.ritz[:n] - ref[:n]).max() <= (8 + m) * np.finfo(float).eps * bound
    assert np.isnan(r.ritz[n:]).all()                    # past the dimension of T


def test_ftlm_long_krylov_spaces(hm):
    """Many rows of T, most of them past convergence, so that the decomposition splits and deflates.  The
    quadrature over 32 vectors has converged long before, so Z and E agree with a shorter run up to the
    FP32 vectors' rounding, 430 steps of 2^-24."""
    inst = W.small_ring(12, -1.0, -0.3)
    T = [0.3, 1.0, 5.0]
    a = hm.ftlm_run(12, hm.bonds_of(inst), 32, 100, 9, T)
    c = hm.ftlm_run(12, hm.bonds_of(inst), 32, 430, 9, T)
    tol = 430 * 2.0**-24
    assert np.allclose(c.Z * np.exp(-(c.e_ref - a.e_ref) / np.array(T)), a.Z, rtol=tol)
    assert np.allclose(c.E, a.E, rtol=tol)
    k = int(np.argmax(a.mlen[:, 0]))
    assert abs(c.tau[k, 0, : c.mlen[k, 0]].sum() - 1.0) <= 430 * 16 * np.finfo(float).eps


@pytest.mark.parametrize("n,two_m,steps", [(11, 1, 7), (11, 1, 8), (12, 4, 33), (13, 1, 192), (13, 1, 200)])
def test_arnoldi_gram_schmidt_tiles(hm, n, two_m, steps):
    """Gram-Schmidt over row tiles (up to 192 vectors, then the untiled kernels) at row counts that are no
    multiple of a tile: H is tridiagonal to the double-float dots' rounding (dim terms of 2^-46 of the
    vectors' products, |v| = |w| / beta = 1, scaled by |H|), as a Hermitian H's Arnoldi matrix is, and
    its lowest eigenvalue is the sector's once the space holds it."""
    inst = W.small_ring(n, -1.0, -0.4, two_m=two_m)
    b = hm.Basis(inst.n_sites, inst.two_s, inst.two_m)
    r = hm.arnoldi_run(b, hm.bonds_of(inst), steps, seed=11, n_ritz=1)
    assert r.steps == steps
    H = r.H[:steps, :steps]
    scale = np.abs(r.H).max()
    off = H - np.triu(np.tril(H, 1), -1)
    assert np.abs(off).max() <= b.dim * 2.0**-46 * scale
    assert np.abs(np.diag(H, 1) - np.diag(H, -1)).max() <= b.dim * 2.0**-46 * scale
    if steps >= 192:
        eye = torch.eye(b.dim, dtype=torch.float64, device="cuda")
        dense = torch.stack([hm.matvec(b, hm.bonds_of(inst), eye[k].contiguous()) for k in range(b.dim)])
        e0 = np.linalg.eigvalsh(dense.cpu().numpy())[0]
        assert abs(r.ritz[0] - e0) <= 1e-11 * abs(e0)


@pytest.mark.parametrize("m", [3, 31, 32, 33, 64, 65, 96, 97, 130])
def test_ftlm_quadrature_moments(hm, m):
    """An m-step run and a 2-step run of the same vectors share alpha_0, beta_0 and alpha_1, so their moments
    sum_j tau_j theta_j^k, k <= 3, agree: the weights of interlacing values add up to one but for 16 roundings
    a factor, and the values lie within 10 eps of the norm of T's (bound: sum |J| 3/4).  Sectors of at most m
    states are diagonalised instead, without FP32 vectors."""
    inst = W.small_ring(12, -1.0, -0.3)
    bonds = hm.bonds_of(inst)
    two, run = (hm.ftlm_run(12, bonds, 2, k, 9, [1.0]) for k in (2, m))
    nrm = 0.75 * np.abs(inst.J).sum()
    for A in range(13):
        for r in range(2):
            n2, n = int(two.mlen[A, r]), int(run.mlen[A, r])
            if n2 < 2 or n < 3 or math.comb(12, A) <= m:
                continue
            t2, t = two.theta[A, r, :n2], run.theta[A, r, :n]
            assert (run.tau[A, r, :n] >= 0).all()
            for k in range(4):
                a, b = two.tau[A, r, :n2] @ t2**k, run.tau[A, r, :n] @ t**k
                assert abs(a - b) <= (16 * n + 10 * k + 64) * np.finfo(float).eps * nrm**k, (A, r, k)


@pytest.mark.parametrize("n,steps", [(10, 9), (11, 60), (12, 70), (12, 230)])
def test_ftlm_exact_sectors(hm, n, steps):
    """Sectors of at most `steps` states (one, odd and even sizes, in shared memory and beyond it), degenerate
    levels included, against LAPACK on H's columns: Jacobi stops at off-diagonals of 1e-15 of the norm, its
    rotations round each element at most 40 (dim - 1) times by 4 eps; the weights of a level sum
    to |P r|^2, and all of them to one."""
    inst = W.small_ring(n, -1.0, -0.5)
    bonds = hm.bonds_of(inst)
    run = hm.ftlm_run(n, bonds, 3, steps, 4, [1.0])
    for A in range(n + 1):
        dim = math.comb(n, A)
        if dim > steps:
            continue
        b = hm.Basis(n, 1, n - 2 * A)
        eye = torch.eye(dim, dtype=torch.float64, device="cuda")
        H = torch.stack([hm.matvec(b, bonds, eye[k].contiguous()) for k in range(dim)]).cpu().numpy()
        ref = np.linalg.eigvalsh(H)
        tol = 160 * dim * np.finfo(float).eps * max(np.abs(H).sum(1).max(), 1.0)
        for r in range(3):
            assert run.mlen[A, r] == dim
            assert np.abs(np.sort(run.theta[A, r, :dim]) - ref).max() <= tol
            assert abs(run.tau[A, r, :dim].sum() - 1.0) <= tol
            v = oracle.start_pm1(oracle.splitmix(4, (A << 20) + r), dim) / math.sqrt(dim)
            m1, m2 = (run.tau[A, r, :dim] @ run.theta[A, r, :dim] ** k for k in (1, 2))
            nrm = max(np.abs(H).sum(1).max(), 1.0)
            assert abs(m1 - v @ H @ v) <= 2 * tol and abs(m2 - v @ H @ (H @ v)) <= 4 * tol * nrm
