"""GPU tests of per-bond plans whose couplings lie far apart (BlkParams::pb_wide): the matrix elements of the
weak bonds keep their bits.  Columns of H, whose off-diagonal elements J_b / 2 are single terms."""
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


def couplings(n, least):
    """Every bond of a J1-J2 ring its own coupling, sizes spread evenly in the logarithm down to least."""
    u, v, _ = W.ring_bonds(n, -1.0, -0.5)
    rng = np.random.default_rng(n)
    J = rng.permutation(np.geomspace(1.0, least, len(u))) * rng.uniform(0.6, 1.0, len(u)) * rng.choice([-1, 1], len(u))
    return u, v, J


def column(ob, u, v, J, i, flip=0):
    """Column i of H as {row: element} and the diagonal's terms; flip: of a spin-flip block."""
    d = [int(a) for a in ob.decode(i)]
    out, diag = {}, []
    for p, q, j in zip(u, v, J):
        if d[p] == d[q]:
            diag.append(-j / 4)
            continue
        diag.append(j / 4)
        t = list(d)
        t[p], t[q] = d[q], d[p]
        r, s = int(ob.encode(t)), 1
        if flip and r >= ob.dim // 2:
            r, s = ob.dim - 1 - r, flip
        out.setdefault(r, []).append(-s * j / 2)
    return out, diag


# C_b holds 56 bits below the largest coupling, its low part (at most 1/2) 24 more of it: 1e-3 is exact, 6e-10 (2^-31) keeps
# 2^-50 of itself, 6e-14 (2^-44) 2^-37
@pytest.mark.parametrize("least,tol", [(0.2, 0.0), (1e-3, 0.0), (1e-9, 2.0**-49), (1e-13, 2.0**-36)])
@pytest.mark.parametrize("row", ["table", "slots"])
@pytest.mark.parametrize("n,two_m,parity", [(14, 0, 0), (17, 3, 0), (14, 0, 1), (14, 0, -1)])
def test_columns_of_h(hm, n, two_m, parity, row, least, tol, monkeypatch):
    monkeypatch.setenv("HM_JIT_ROW", row)
    u, v, J = couplings(n, least)
    b = hm.Basis(n, 1, two_m, parity=parity)
    ob = oracle.Basis(n, 1, (n - two_m) // 2)
    bl = hm.BondList.make(u, v, J)
    assert hm.matvec_kernel_name(b, bl) == "k_blk_matvec_jit"
    for i in np.random.default_rng(1).integers(0, b.dim, 12):
        x = torch.zeros(b.dim, dtype=torch.float64, device="cuda")
        x[int(i)] = 1.0
        y = hm.matvec(b, bl, x).cpu().numpy()
        col, diag = column(ob, u, v, J, int(i), parity)
        for r, terms in col.items():
            if r != i:
                s = float(sum(np.array(terms, dtype=np.longdouble)))
                assert abs(y[r] - s) <= tol * abs(s) + (len(terms) - 1) * 2.0**-52 * abs(np.array(terms)).max(), r
                y[r] = 0.0
        extra = sum(col.get(int(i), []))
        assert abs(y[i] - sum(diag) - extra) <= len(u) * 2.0**-52 * (np.abs(J).sum() / 4 + abs(extra))
        y[i] = 0.0
        assert not y.any()


@pytest.mark.parametrize("n,two_m", [(12, 0), (16, 2), (19, 3)])
def test_runs(hm, n, two_m):
    """Whole run = step-wise run bit for bit, and both the oracle's."""
    u, v, J = couplings(n, 1e-4)
    b, ob = hm.Basis(n, 1, two_m + n % 2 - two_m % 2), oracle.Basis(n, 1, (n - (two_m + n % 2 - two_m % 2)) // 2)
    bl = hm.BondList.make(u, v, J)
    x = oracle.start_uniform(7, b.dim)
    xd = torch.from_numpy(x).cuda()
    whole = hm.lanczos_run(b, bl, 15, v0=xd)
    run = hm.LanczosRun(b, bl, 15, v0=xd)
    run.step(15)
    al, be, _ = run.read()
    assert np.array_equal(whole.alpha, al) and np.array_equal(whole.beta, be)
    oal, obe = ob.lanczos(oracle.Bonds(u, v, J), x, 15)
    np.testing.assert_allclose(al, oal, rtol=0, atol=1e-11 * np.abs(oal).max())
    np.testing.assert_allclose(be, obe, rtol=0, atol=1e-11 * np.abs(oal).max())
