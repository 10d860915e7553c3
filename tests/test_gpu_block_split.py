"""GPU tests of the block path on two-dimensional clusters, ladders and rings with far neighbours, whose bonds
fit its slots only from some split position on (csrc/blk_fit.h): the kernel taken, and products and
Lanczos runs against the oracle, in the whole sector and in both spin-flip blocks."""
import numpy as np
import pytest

import oracle
from lattices import LATTICES

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def hm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0706_3293_gb300 import api
    return api


SMALL = [k for k in LATTICES if LATTICES[k][0][0] <= 21 and LATTICES[k][1]]
J = [-1.0, -0.625]


def rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def lists(hm, name, kind):
    """The lattice's couplings by class, or a coupling for each bond."""
    (n, bonds, cls), _ = LATTICES[name]
    u, v = np.array(bonds).T
    Jb = np.array(J)[cls] if kind == "classes" else np.random.default_rng(n).uniform(-1.2, -0.8, len(u))
    return n, hm.BondList.make(u, v, Jb), oracle.Bonds(u, v, Jb)


@pytest.mark.parametrize("name", SMALL)
def test_products(hm, name):
    n, bl, obl = lists(hm, name, "classes")
    b, ob = hm.Basis(n, 1, n % 2), oracle.Basis(n, 1, n // 2)
    assert hm.matvec_kernel_name(b, bl) == "k_blk_matvec"
    x = oracle.start_uniform(3, b.dim)
    ref = ob.matvec(obl, x)
    assert rel(hm.matvec(b, bl, torch.from_numpy(x).cuda()).cpu().numpy(), ref) <= 1e-12
    y32 = hm.matvec(b, bl, torch.from_numpy(x.astype(np.float32)).cuda()).double().cpu().numpy()
    assert rel(y32, ref) <= 1e-5
    run = hm.LanczosRun(b, bl, 12, v0=torch.from_numpy(x).cuda())
    assert run.kernel_name().startswith("k_blk_lz64")
    run.step(12)
    al, be, _ = run.read()
    whole = hm.lanczos_run(b, bl, 12, v0=torch.from_numpy(x).cuda())
    oal, obe = ob.lanczos(obl, x, 12)
    for a, c in ((al, be), (whole.alpha, whole.beta)):
        np.testing.assert_allclose(a, oal, rtol=0, atol=1e-11 * np.abs(oal).max())
        np.testing.assert_allclose(c, obe, rtol=0, atol=1e-11 * np.abs(oal).max())


@pytest.mark.parametrize("parity", [1, -1])
@pytest.mark.parametrize("name,kind", [(k, kind) for k in SMALL if LATTICES[k][0][0] % 2 == 0 for kind in ("classes", "bonds")
                                       # with a coupling for each bond no split holds these
                                       if kind == "classes" or not ("ladder" in k or "J1-J2" in k)])
def test_spin_flip_blocks(hm, name, kind, parity):
    n, bl, obl = lists(hm, name, kind)
    b, ob = hm.Basis(n, 1, 0, parity=parity), oracle.Basis(n, 1, n // 2)
    x = oracle.start_uniform(5, b.dim)
    xd = torch.from_numpy(x).cuda()
    assert rel(hm.matvec(b, bl, xd).cpu().numpy(), oracle.flip_matvec(ob, obl, x, parity)) <= 1e-12
    run = hm.lanczos_run(b, bl, 8, v0=xd)
    q, prev, beta = x / np.linalg.norm(x), np.zeros(b.dim), 0.0
    for j in range(8):                                    # the recurrence with the oracle's product
        w = oracle.flip_matvec(ob, obl, q, parity) - beta * prev
        alpha = q @ w
        w -= alpha * q
        prev, beta = q, np.linalg.norm(w)
        q = w / beta
        scale = np.abs(run.alpha).max()
        assert abs(run.alpha[j] - alpha) <= 1e-11 * scale and abs(run.beta[j] - beta) <= 1e-11 * scale


@pytest.mark.parametrize("name", ["square 7x3", "ladder 10x2"])
def test_bond_correlations(hm, name):
    n, bl, obl = lists(hm, name, "classes")
    b, ob = hm.Basis(n, 1, n % 2), oracle.Basis(n, 1, n // 2)
    g, x = oracle.start_uniform(1, b.dim), oracle.start_uniform(2, b.dim)
    got = hm.bond_corr(b, bl, torch.from_numpy(g).cuda(), torch.from_numpy(x).cuda()).cpu().numpy()
    ref = ob.bond_corr(obl, g, x)
    np.testing.assert_allclose(got, ref, rtol=0, atol=1e-11 * np.abs(ref).max())
