"""GPU tests of y = H x for several vectors (csrc/blk_multi.cu) against H itself, element by element."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_0706_3293_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0706_3293_gb300 import api
    return api


def lattice(n, kind):
    if kind == "complete":                                # four classes, more than six low ends of cross bonds
        u, v = np.triu_indices(n, 1)
        return u, v, np.array([-1.0, 0.6, -0.25, 0.1])[np.arange(len(u)) % 4]
    if kind == "far":                                     # no low bond in one class, none across in another
        return np.array([0, 0, n - 2, 3]), np.array([1, n - 1, n - 1, n - 2]), np.array([-1.0, 0.5, 0.25, 0.25])
    return W.ring_bonds(n, -1.0, None if kind == "ring" else -0.3)


def product(u, v, J, n, two_m, x):
    """H x in extended precision and sum_j |H_ij x_j|, from the states in index order."""
    A = (n - two_m) // 2
    w = np.array([s for s in range(1 << n) if bin(s).count("1") == A], dtype=np.int64)
    y, bound = np.zeros(x.shape, np.longdouble), np.zeros(x.shape, np.longdouble)
    xl = x.astype(np.longdouble)
    for p, q, j in zip(u, v, J):
        ne = ((w >> p) ^ (w >> q)) & 1
        y += -j * np.where(ne, -0.25, 0.25)[:, None] * xl
        bound += abs(j) * 0.25 * np.abs(xl)
        t = np.searchsorted(w, w ^ ((1 << int(p)) | (1 << int(q))))
        i = np.nonzero(ne)[0]
        y[i] += -j * 0.5 * xl[t[i]]
        bound[i] += abs(j) * 0.5 * np.abs(xl[t[i]])
    return y, bound


@pytest.mark.parametrize("n,two_m,kind", [(10, 0, "ring"), (10, 8, "j1j2"), (11, 1, "complete"), (12, -4, "far"),
                                          (13, 3, "j1j2"), (15, 1, "ring"), (10, 10, "ring")])
@pytest.mark.parametrize("nvec", [2, 3, 7, 8, 33, 64])
def test_several_vectors(hm, n, two_m, kind, nvec):
    """Couplings of J, sizes and numbers of vectors with idle lanes and a second launch.  FP64: a value is cut
    at 2^-54 of its row's largest, the class sums round a few times (2^-52 of sum |H x| a bond more than
    covers both); the exponents of x spread over 40 binades.  FP32: one rounding a bond and class."""
    b = hm.Basis(n, 1, two_m)
    u, v, J = lattice(n, kind)
    bl = hm.BondList.make(u, v, J)
    gen = np.random.default_rng(n * 100 + nvec)
    x = (gen.random((b.dim, nvec)) - 0.5) * 2.0 ** gen.integers(-20, 20, (b.dim, nvec))
    y, bound = product(u, v, J, n, two_m, x)
    got = hm.matvec(b, bl, torch.from_numpy(x).cuda()).cpu().numpy()
    assert (np.abs(got - y) <= (len(u) + 8) * 2.0**-52 * bound).all()
    x32 = x.astype(np.float32)
    y, bound = product(u, v, J, n, two_m, x32)
    got = hm.matvec(b, bl, torch.from_numpy(x32).cuda()).cpu().numpy()
    assert (np.abs(got - y) <= (len(u) + 16) * 3 * 2.0**-24 * bound).all()


def test_special_values(hm):
    """Rows with infinities and NaN, with zeros only, near the ends of binary64's range."""
    n = 12
    b = hm.Basis(n, 1, 0)
    u, v, J = lattice(n, "j1j2")
    bl = hm.BondList.make(u, v, J)
    gen = np.random.default_rng(5)
    x = gen.random((b.dim, 5)) - 0.5
    x[:, 1] *= 1e-300
    x[:, 2] = 0.0
    x[7, 2] = 5e-324
    x[:, 3] *= 1e306
    y, bound = product(u, v, J, n, 0, x)
    x[100, 0], x[200, 0], x[:, 4] = np.inf, np.nan, -0.0
    got = hm.matvec(b, bl, torch.from_numpy(x).cuda()).cpu().numpy()
    assert (np.abs(got[:, 1:4] - y[:, 1:4]) <= (len(u) + 8) * 2.0**-52 * bound[:, 1:4] + 1e-322).all()
    assert (got[:, 4] == 0).all()
    reach = np.zeros((b.dim, 1))
    reach[100] = reach[200] = 1.0
    hit = product(u, v, np.ones(len(u)), n, 0, reach)[1][:, 0] > 0
    assert (~np.isfinite(got[hit, 0])).all() and np.isfinite(got[~hit, 0]).all()
    assert (np.abs(got[~hit, 0] - y[~hit, 0]) <= (len(u) + 8) * 2.0**-52 * bound[~hit, 0]).all()
