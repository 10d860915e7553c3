"""GPU tests of the integer sums of several vectors (csrc/blk_multi.cu) on what their alignment has to bear:
couplings far apart, an own value far above its neighbours, rows and columns of zeros, many high sites.
Each row against its own bound sum_j |H_ij x_j|, in extended precision."""
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


def states(n, two_m):
    A = (n - two_m) // 2
    w = np.arange(1 << n, dtype=np.uint32)
    pop = sum((w >> k) & 1 for k in range(n))
    return w[pop == A].astype(np.int64)


def product(u, v, J, w, x):
    """H x and sum_j |H_ij x_j| (the diagonal element as one term) in extended precision."""
    xl = x.astype(np.longdouble)
    dg = np.zeros(len(w), np.longdouble)
    y, bound = np.zeros(x.shape, np.longdouble), np.zeros(x.shape, np.longdouble)
    for p, q, j in zip(u, v, J):
        ne = ((w >> p) ^ (w >> q)) & 1
        dg += -np.longdouble(j) * np.where(ne, -0.25, 0.25)
        i = np.nonzero(ne)[0]
        t = np.searchsorted(w, w[i] ^ ((1 << int(p)) | (1 << int(q))))
        y[i] += -np.longdouble(j) * 0.5 * xl[t]
        bound[i] += abs(j) * 0.5 * np.abs(xl[t])
    return y + dg[:, None] * xl, bound + np.abs(dg)[:, None] * np.abs(xl), dg


def rounding(u, J):
    """Every gathered value cut at 2^-53 of the largest term, sums floored twice a class, class sums and
    the diagonal rounded: below 2^-52 (n_bonds + 8) of the bound; the diagonal element itself is a binary64 sum
    over the classes, 4 2^-53 of sum_c |J_c| n_c / 4."""
    return (len(u) + 8) * 2.0**-52


@pytest.mark.parametrize("nvec", [2, 3, 8])
@pytest.mark.parametrize("ratio", [1e-3, 1e-8, 1e-17, 1e-40])
def test_couplings_far_apart(hm, ratio, nvec):
    """Neighbours across the weak bonds far larger than those across the strong ones, in half the columns the
    other way round; 1e-40 is beyond the integers' range."""
    n = 12
    b = hm.Basis(n, 1, 0)
    u, v, J = W.ring_bonds(n, -1.0, -0.3)
    J = np.where(np.arange(len(u)) < n, -1.0, -0.3 * ratio)
    gen = np.random.default_rng(nvec)
    w = states(n, 0)
    x = gen.random((b.dim, nvec)) - 0.5
    x *= np.where(gen.random((b.dim, 1)) < 0.1, 1.0 / ratio, 1.0) ** np.array([1 if k % 2 == 0 else 2 for k in range(nvec)])
    y, bound, _ = product(u, v, J, w, x)
    got = hm.matvec(b, hm.BondList.make(u, v, J), torch.from_numpy(x).cuda()).cpu().numpy()
    diag = 4 * 2.0**-53 * np.abs(J).sum() / 4 * np.abs(x)
    assert (np.abs(got - y) <= rounding(u, J) * bound + diag).all()


def test_own_value_without_weight(hm):
    """Rows whose diagonal element is exactly zero keep their neighbours' bits under an own value of 2^80."""
    n = 12
    b = hm.Basis(n, 1, 0)
    u, v, J = W.ring_bonds(n, -1.0)
    w = states(n, 0)
    _, _, dg = product(u, v, J, w, np.zeros((b.dim, 1)))
    zero = np.nonzero(dg == 0)[0]
    reach = {int(i) for i in zero}
    gen = np.random.default_rng(3)
    x = gen.random((b.dim, 4)) - 0.5
    mine = []
    for i in zero:                                        # rows no exchange apart, so that none is a neighbour of another
        near = {int(np.searchsorted(w, w[i] ^ ((1 << int(p)) | (1 << int(q))))) for p, q in zip(u, v)
                if ((w[i] >> p) ^ (w[i] >> q)) & 1}
        if not near & set(mine):
            mine.append(int(i))
    assert len(mine) >= 20 and set(mine) <= reach
    x[mine] = 2.0**80
    y, bound, _ = product(u, v, J, w, x)
    got = hm.matvec(b, hm.BondList.make(u, v, J), torch.from_numpy(x).cuda()).cpu().numpy()
    assert (np.abs(got - y) <= rounding(u, J) * bound)[mine].all()


def test_unit_vectors_are_columns_of_h(hm):
    n = 12
    b = hm.Basis(n, 1, 2)
    u, v, J = W.ring_bonds(n, -1.0, -0.3)
    cols = np.array([0, 1, 77, b.dim // 2, b.dim - 1])
    x = np.zeros((b.dim, len(cols)))
    x[cols, np.arange(len(cols))] = 1.0
    y, bound, _ = product(u, v, J, states(n, 2), x)
    got = hm.matvec(b, hm.BondList.make(u, v, J), torch.from_numpy(x).cuda()).cpu().numpy()
    assert (got[bound == 0] == 0).all()
    assert (np.abs(got - y) <= rounding(u, J) * bound + 4 * 2.0**-53 * np.abs(J).sum() / 4 * x).all()


@pytest.mark.parametrize("scale", [2.0**-1000, 2.0**-958, 2.0**-900, 2.0**900, 2.0**964, 2.0**1010])
def test_ends_of_the_range(hm, scale):
    """Around the exponents where the integers hand over to binary64, and beyond them."""
    n = 11
    b = hm.Basis(n, 1, 1)
    u, v, J = W.ring_bonds(n, -1.0, -0.25)
    gen = np.random.default_rng(8)
    x = (gen.random((b.dim, 6)) - 0.5) * 2.0 ** gen.integers(-8, 8, (b.dim, 6)) * scale
    y, bound, _ = product(u, v, J, states(n, 1), x)
    got = hm.matvec(b, hm.BondList.make(u, v, J), torch.from_numpy(x).cuda()).cpu().numpy()
    assert (np.abs(got - y) <= rounding(u, J) * bound + 4 * 2.0**-53 * np.abs(J).sum() / 4 * np.abs(x) + 1e-320).all()


@pytest.mark.parametrize("n,two_m,nvec", [(18, 0, 8), (20, 4, 3), (22, 10, 4)])
def test_many_high_sites(hm, n, two_m, nvec):
    """Five to nine sites above the split: high exchanges within and across classes."""
    b = hm.Basis(n, 1, two_m)
    u, v, J = W.ring_bonds(n, -1.0, -0.3)
    gen = np.random.default_rng(n)
    x = gen.random((b.dim, nvec)) - 0.5
    y, bound, _ = product(u, v, J, states(n, two_m), x)
    bl = hm.BondList.make(u, v, J)
    diag = 4 * 2.0**-53 * np.abs(J).sum() / 4 * np.abs(x)
    got = hm.matvec(b, bl, torch.from_numpy(x).cuda()).cpu().numpy()
    assert (np.abs(got - y) <= rounding(u, J) * bound + diag).all()
    x32 = x.astype(np.float32)
    y, bound, _ = product(u, v, J, states(n, two_m), x32)
    got = hm.matvec(b, bl, torch.from_numpy(x32).cuda()).cpu().numpy()
    assert (np.abs(got - y) <= (len(u) + 16) * 3 * 2.0**-24 * (bound + np.abs(J).sum() / 4 * np.abs(x32))).all()


@pytest.mark.parametrize("n,two_m,nvec", [(24, 0, 2), (30, 16, 32), (32, 20, 32), (32, 20, 2), (32, -22, 33)])
def test_up_to_nineteen_high_sites(hm, n, two_m, nvec):
    """Against the products of single vectors, exact sums rounded once: row sums of |H| are at most 3/4 sum |J|.
    The last two sectors have too few rows a block and take the general rows."""
    b = hm.Basis(n, 1, two_m)
    u, v, J = W.ring_bonds(n, -1.0, -0.3)
    bl = hm.BondList.make(u, v, J)
    x = torch.rand((b.dim, nvec), dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n)) - 0.5
    got = hm.matvec(b, bl, x)
    for k in {0, 1, nvec - 1}:
        ref = hm.matvec(b, bl, x[:, k].contiguous())
        assert (got[:, k] - ref).abs().max().item() <= rounding(u, J) * 0.75 * np.abs(J).sum() * 0.5
