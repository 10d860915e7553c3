"""GPU tests of the block path's y = H x with target tables (RowTable, csrc/blk_sweep.cuh) against the
generic rows, which HM_JIT_ROW = slots selects: the same exact integer sums in FP64."""
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
    if kind == "ring":
        return W.ring_bonds(n, -1.0)
    if kind == "j1j2":
        return W.ring_bonds(n, -1.0, -0.5)
    if kind == "three":                                   # three classes, second neighbours in two of them
        u, v, J = W.ring_bonds(n, -1.0, -0.3)
        J[n::2] = -0.7
        return u, v, J
    if kind == "graph":                                   # four classes on a random graph: no triangles to speak of
        u, v = W.random_regular_graph(n, 3 if n % 2 == 0 else 4, 7)
        return u, v, np.array([-1.0, 0.6, -0.25, 0.1])[np.arange(len(u)) % 4]
    u = np.array([0, 0, 0], dtype=np.int32)               # three bonds of one site, far apart
    return u, np.array([1, n // 2, n - 1], dtype=np.int32), np.array([-1.0, -1.0, 0.5])


@pytest.mark.parametrize("kind", ["ring", "j1j2", "three", "graph", "star"])
# (24, +-18), (22, 16): the largest block is far smaller than the class next to it, whose ranks the cross
# entries hold
@pytest.mark.parametrize("n,two_m", [(10, 0), (10, 8), (11, 1), (13, 5), (16, 0), (17, 1), (20, 2), (22, 0), (26, 12),
                                     (24, 18), (24, -18), (22, 16)])
def test_table_rows_equal_generic_rows(hm, n, two_m, kind, monkeypatch):
    b = hm.Basis(n, 1, two_m)
    bl = hm.BondList.make(*lattice(n, kind))
    gen = torch.Generator(device="cuda").manual_seed(n)
    x = torch.rand(b.dim + 1, dtype=torch.float64, device="cuda", generator=gen) - 0.5
    for xv in (x[:-1], x[1:]):                            # 16-byte aligned and not
        out = {}
        for row in ("table", "slots"):
            monkeypatch.setenv("HM_JIT_ROW", row)
            out[row] = (hm.matvec(b, bl, xv), hm.matvec(b, bl, xv.float()))
        assert torch.equal(out["table"][0], out["slots"][0])
        # FP32 rows: the same at most 3 n_bonds + 4 float terms, |x| <= 1/2, in another order
        tol = 2 * (3 * len(bl) + 4) * 2.0**-24 * 0.75 * np.abs(bl.J).sum() * 0.5
        assert (out["table"][1] - out["slots"][1]).abs().max().item() <= tol


@pytest.mark.parametrize("parity", [1, -1])
def test_table_rows_flip_basis(hm, parity, monkeypatch):
    b = hm.Basis(18, 1, 0, parity=parity)
    bl = hm.BondList.make(*lattice(18, "j1j2"))
    x = torch.rand(b.dim, dtype=torch.float64, device="cuda")
    out = {}
    for row in ("table", "slots"):
        monkeypatch.setenv("HM_JIT_ROW", row)
        out[row] = hm.matvec(b, bl, x)
    assert torch.equal(out["table"], out["slots"])


def test_capture_of_a_new_layout(hm):
    """A bond list first seen inside a stream capture: no table is built there, the product is the same."""
    b = hm.Basis(14, 1, 0)
    x = torch.rand(b.dim, dtype=torch.float64, device="cuda")
    hm.matvec(b, hm.BondList.make(*lattice(14, "ring")), x)
    bl = hm.BondList.make(*lattice(14, "j1j2"))
    y = torch.empty_like(x)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        hm.matvec(b, bl, x, out=y)
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(y, hm.matvec(b, bl, x))
