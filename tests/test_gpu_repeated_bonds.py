"""GPU tests of lists in which a bond comes twice or more, as on a torus two sites wide, with the same and with
different couplings: H is the sum over the list, against the oracle, on every path that takes s = 1/2 and s = 1
lists, with the bonds below, across and above the split of the block path."""
import math

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
from lattices import LATTICES
from paper_0706_3293_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0706_3293_gb300 import api
    return api


def case(hm, name):
    if name in LATTICES:
        (n, bonds, cls), _ = LATTICES[name]
        u, v = np.array(bonds).T
        J = np.array([-1.0, -0.625])[cls]
    else:
        n = int(name.split()[0])
        u, v, J = W.ring_bonds(n, -1.0, -0.375)
        again = {"low": [0, 1, n], "high": [n - 2, n - 3, 2 * n - 4], "all": list(range(len(u))), "thrice": [0, 0, 8, 8, n - 3, n - 3],
                 "mixed": [0, 8, n - 2], "bonds": [0, 8, n - 2]}[name.split()[1]]
        Ja = J[again]
        if "mixed" in name:                               # the pair again with the other class's coupling
            Ja = np.where(Ja == -1.0, -0.375, -1.0)
        u, v, J = np.concatenate([u, u[again]]), np.concatenate([v, v[again]]), np.concatenate([J, Ja])
        if "bonds" in name:
            J = np.random.default_rng(n).uniform(-1.2, -0.8, len(u))
    return n, hm.BondList.make(u, v, J), oracle.Bonds(u, v, J)


NAMES = [f"{n} {k}" for n in (12, 16) for k in ("low", "high", "all", "thrice", "mixed", "bonds")] + [
    "square 6x2 torus", "square 8x2 torus", "triangular 6x2 torus"]


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("row", ["table", "slots", "delta"])
@pytest.mark.parametrize("name", NAMES)
def test_products_and_runs(hm, name, row, monkeypatch):
    monkeypatch.setenv("HM_JIT_ROW", row)
    n, bl, obl = case(hm, name)
    b, ob = hm.Basis(n, 1, 0), oracle.Basis(n, 1, n // 2)
    x = oracle.start_uniform(3, b.dim)
    xd = torch.from_numpy(x).cuda()
    ref = ob.matvec(obl, x)
    assert rel(hm.matvec(b, bl, xd).cpu().numpy(), ref) <= 1e-12
    assert rel(hm.matvec(b, bl, xd.float()).double().cpu().numpy(), ref) <= 1e-5
    many = torch.stack([xd, -xd] * 4, 1).contiguous()
    assert rel(hm.matvec(b, bl, many)[:, 4].cpu().numpy(), ref) <= 1e-12
    assert rel(hm.matvec(b, bl, many.float())[:, 7].double().cpu().numpy(), -ref) <= 1e-5
    oal, obe = ob.lanczos(obl, x, 10)
    scale = np.abs(oal).max()
    for jit in ("1", "0"):                                # the whole-run kernel, and the generic kernels step by step
        monkeypatch.setenv("HM_JIT", jit)
        for dt, tol in ((torch.float64, 1e-11), (torch.float32, 2e-5)):
            r = hm.lanczos_run(b, bl, 10, v0=xd.to(dt), dtype=dt)
            assert np.abs(r.alpha - oal).max() <= tol * scale and np.abs(r.beta - obe).max() <= tol * scale
    monkeypatch.setenv("HM_JIT", "1")
    run = hm.LanczosRun(b, bl, 10, v0=xd)
    run.step(10)
    assert np.abs(run.read()[0] - oal).max() <= 1e-11 * scale
    g = oracle.start_uniform(4, b.dim)
    np.testing.assert_allclose(hm.bond_corr(b, bl, torch.from_numpy(g).cuda(), xd).cpu().numpy(), ob.bond_corr(obl, g, x),
                               rtol=0, atol=1e-11 * b.dim)


@pytest.mark.parametrize("parity", [1, -1])
@pytest.mark.parametrize("name", NAMES)                  # the triangular torus fits with its repeated bonds as one
def test_spin_flip_blocks(hm, name, parity):
    n, bl, obl = case(hm, name)
    b, ob = hm.Basis(n, 1, 0, parity=parity), oracle.Basis(n, 1, n // 2)
    x = oracle.start_uniform(3, b.dim)
    xd = torch.from_numpy(x).cuda()
    ref = oracle.flip_matvec(ob, obl, x, parity)
    assert rel(hm.matvec(b, bl, xd).cpu().numpy(), ref) <= 1e-12
    assert rel(hm.matvec(b, bl, xd.float()).double().cpu().numpy(), ref) <= 1e-5
    q = x / np.linalg.norm(x)
    first = q @ oracle.flip_matvec(ob, obl, q, parity)
    for dt, tol in ((torch.float64, 1e-11), (torch.float32, 2e-5)):
        assert abs(hm.lanczos_run(b, bl, 4, v0=xd.to(dt), dtype=dt).alpha[0] - first) <= tol * np.abs(bl.J).sum()


@pytest.mark.parametrize("name", [k for k in NAMES if k.split()[0] == "12" and "bonds" not in k] + ["square 6x2 torus"])
def test_finite_temperature(hm, name):
    """First moments <v|H|v> of each sector: FP32 rows of at most 3 n_bonds + 8 roundings."""
    n, bl, obl = case(hm, name)
    run = hm.ftlm_run(n, bl, 2, 12, 5, [1.0])
    tol = (3 * len(bl) + 8) * 2.0**-24 * 0.75 * np.abs(bl.J).sum()
    for A in range(n + 1):
        res = oracle.ftlm_sector(oracle.Basis(n, 1, A), obl, 5, 2, 12)
        for r in range(2):
            m = int(run.mlen[A, r])
            assert m == min(12, math.comb(n, A)) or m < 12
            assert abs(float(run.tau[A, r, :m] @ run.theta[A, r, :m]) - float(np.dot(res[r][1], res[r][0]))) <= tol


@pytest.mark.parametrize("kind", ["low", "thrice", "all"])
@pytest.mark.parametrize("n", [8, 10])
def test_spin_one(hm, n, kind):
    n, bl, obl = case(hm, f"{n} {kind}")
    b, ob = hm.Basis(n, 2, 0), oracle.Basis(n, 2, n)
    x = oracle.start_uniform(3, b.dim)
    xd = torch.from_numpy(x).cuda()
    ref = ob.matvec(obl, x)
    assert rel(hm.matvec(b, bl, xd).cpu().numpy(), ref) <= 1e-12
    assert rel(hm.matvec(b, bl, xd.float()).double().cpu().numpy(), ref) <= 1e-5
    oal, _ = ob.lanczos(obl, x, 8)
    for dt, tol in ((torch.float64, 1e-11), (torch.float32, 2e-5)):
        assert np.abs(hm.lanczos_run(b, bl, 8, v0=xd.to(dt), dtype=dt).alpha - oal).max() <= tol * np.abs(oal).max()
