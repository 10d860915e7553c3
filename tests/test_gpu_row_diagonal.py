"""GPU test of the row sweep's integer diagonal (row_plan, csrc/basis.cu) with couplings far apart: rows in which a
zero digit or opposite signs remove the large couplings keep the small ones' bits.  Each row against its own
bound, in extended precision."""
import itertools

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0706_3293_gb300 import api
    return api


def diagonal(n, two_s, A, u, v, J):
    """The states in index order, H_ii and sum_b |terms| in extended precision."""
    st = np.array(sorted((a for a in itertools.product(range(two_s + 1), repeat=n) if sum(a) == A), key=lambda a: a[::-1]))
    m = (two_s - 2 * st).astype(np.longdouble) / 2
    t = np.array([-np.longdouble(j) * m[:, p] * m[:, q] for p, q, j in zip(u, v, J)])
    return st, t.sum(0), np.abs(t).sum(0)


# ratios that the two parts of the integer hold, and beyond them (the table form)
@pytest.mark.parametrize("ratio", [0.3, 1e-4, 1e-6, 1e-9, 1e-12, 1e-200])
@pytest.mark.parametrize("n,two_s,two_m", [(7, 2, 0), (5, 4, 2), (9, 1, 1), (6, 3, 0)])
def test_small_couplings_keep_their_bits(hm, n, two_s, two_m, ratio):
    """Columns of H: the diagonal element, its terms rounded a few times, 2^-53 n_bonds of their sum; for integer
    spins many of them have terms of the small couplings alone."""
    u, v = (np.concatenate([np.arange(n), np.arange(n)]), np.concatenate([(np.arange(n) + 1) % n, (np.arange(n) + 2) % n]))
    rng = np.random.default_rng(n)
    J = np.concatenate([np.where(np.arange(n) % 2, -1.0, 1.0), ratio * rng.uniform(-1, 1, n)])
    b = hm.Basis(n, two_s, two_m)
    bl = hm.BondList.make(u, v, J)
    _, dg, mag = diagonal(n, two_s, b.A, u, v, J)
    rows = np.arange(b.dim) if b.dim <= 64 else rng.choice(b.dim, 64, replace=False)
    if two_s % 2 == 0:
        weak = np.nonzero((mag > 0) & (mag < 20 * ratio))[0]
        assert len(weak) > 0
        rows = np.concatenate([weak[:16], rows])[:64]
    for dtype, eps in ((torch.float64, 2.0**-53), (torch.float32, 2.0**-24)):
        x = torch.zeros((b.dim, 64), dtype=dtype, device="cuda")
        x[torch.from_numpy(rows), torch.arange(len(rows))] = 1.0
        y = hm.matvec(b, bl, x[:, : len(rows)].contiguous()).double().cpu().numpy()
        got = y[rows, np.arange(len(rows))].astype(np.longdouble)
        tiny = 0.0 if dtype == torch.float64 else 2.0**-140
        assert (np.abs(got - dg[rows]) <= (len(u) + 4) * eps * mag[rows] + tiny).all()


@pytest.mark.parametrize("ratio", [1e-3, 1e-7, 1e-11])
def test_momentum_rows(hm, ratio):
    """s = 1 ring, k = 0: the state of digits 0 1 2 1 repeated has zero digits between all neighbours, so its
    diagonal element is the second neighbours' alone, -J2 (-1) n / 2, and nothing else leads back to its orbit."""
    n = 8
    u = np.concatenate([np.arange(n), np.arange(n)])
    v = np.concatenate([(np.arange(n) + 1) % n, (np.arange(n) + 2) % n])
    j2 = -ratio * 0.7309167
    b = hm.Basis(n, 2, 0, momentum=0)
    bl = hm.BondList.make(u, v, np.concatenate([np.full(n, -1.0), np.full(n, j2)]))
    eye = torch.eye(b.dim, dtype=torch.float64, device="cuda")
    diag = np.array([float(hm.matvec(b, bl, eye[k].contiguous())[k]) for k in range(b.dim)])
    want = j2 * n / 2
    assert np.abs(diag - want).min() <= 4 * 2.0**-53 * abs(want)
