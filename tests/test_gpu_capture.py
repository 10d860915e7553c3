"""GPU tests of products first made inside a stream capture: on a basis that has made none of several vectors,
and with a bond list whose split position is new to the basis.  Replays equal products outside a capture."""
import pytest

torch = pytest.importorskip("torch")

from lattices import LATTICES
from paper_0706_3293_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hm():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0706_3293_gb300 import api
    return api


def replay(hm, b, bl, x):
    y = torch.zeros_like(x)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        hm.matvec(b, bl, x, out=y)
    g.replay()
    torch.cuda.synchronize()
    return y


def lattice(hm, name, rand=False):
    (n, bonds, cls), _ = LATTICES[name]
    J = [[-1.0, -0.625][c] for c in cls]
    return n, hm.BondList.make(*zip(*bonds), [j * (1 + 0.01 * k) for k, j in enumerate(J)] if rand else J)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32], ids=["f64", "f32"])
@pytest.mark.parametrize("warm", [False, True])
def test_several_vectors_first(hm, warm, dtype):
    """warm: one vector before, whose split position is another."""
    n = 16
    bl = hm.BondList.make(*W.ring_bonds(n, -1.0, -0.5))
    b = hm.Basis(n, 1, 0)
    x = torch.rand((b.dim, 8), dtype=dtype, device="cuda") - 0.5
    if warm:
        hm.matvec(b, bl, x[:, 0].contiguous())
    y = replay(hm, b, bl, x)
    ref = torch.stack([hm.matvec(b, bl, x[:, k].double().contiguous()) for k in range(8)], 1)
    eps = 2.0**-52 if dtype == torch.float64 else 2.0**-23
    tol = 2 * len(bl) * eps * sum(abs(bl.J)) * 0.75       # row sums of |H| times |x| <= 1/2, n_bonds roundings
    assert (y.double() - ref).abs().max().item() <= tol
    assert (hm.matvec(b, bl, x).double() - ref).abs().max().item() <= tol


@pytest.mark.parametrize("parity", [0, 1])
def test_a_split_that_is_new_to_the_basis(hm, parity):
    """The ring's tables are of 10 low sites, the triangular cluster's of 12."""
    n, bl = lattice(hm, "triangular 4x4")
    b, fresh = hm.Basis(n, 1, 0, parity=parity), hm.Basis(n, 1, 0, parity=parity)
    x = torch.rand(b.dim, dtype=torch.float64, device="cuda") - 0.5
    hm.matvec(b, hm.BondList.make(*W.ring_bonds(n, -1.0)), x)
    assert torch.equal(replay(hm, b, bl, x), hm.matvec(fresh, bl, x))


def test_first_product_of_a_basis(hm):
    n, bl = lattice(hm, "square 4x4")
    b, fresh = hm.Basis(n, 1, 0), hm.Basis(n, 1, 0)
    x = torch.rand(b.dim, dtype=torch.float64, device="cuda") - 0.5
    assert torch.equal(replay(hm, b, bl, x), hm.matvec(fresh, bl, x))


def test_first_product_with_a_coupling_for_each_bond(hm):
    """The kernel compiled before, on another basis; tables of this one in the capture."""
    n, bl = lattice(hm, "square 4x4", rand=True)
    b, fresh = hm.Basis(n, 1, 0), hm.Basis(n, 1, 0)
    x = torch.rand(b.dim, dtype=torch.float64, device="cuda") - 0.5
    ref = hm.matvec(fresh, bl, x)
    assert torch.equal(replay(hm, b, bl, x), ref)
