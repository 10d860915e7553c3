"""GPU tests of the whole-run kernel of small FP64 sectors (csrc/lz_small.cu): the same bits as the
step-wise runs, which HM_BLK_SPLIT = 1 selects for e0_grad."""
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


def bonds(n, kind):
    if kind == "j1j2":
        return W.ring_bonds(n, -1.0, -0.5)
    u, v, J = W.ring_bonds(n, -1.0, -0.5)
    if kind == "pairs":                                   # every coupling different: per-bond rows
        return u, v, np.linspace(-1.5, 0.7, len(u))
    if kind == "four":
        return u, v, np.array([-1.0, 0.6, -0.25, 0.1])[np.arange(len(u)) % 4]
    if kind == "inexact":                                 # ratios that are no small integers
        return u, v, np.array([-1.0, 0.6180339887498949])[np.arange(len(u)) % 2]
    return u[:1], v[:1], J[:1]                            # one bond: breaks down after two steps


# one block and one row, single blocks, a last warp with few rows, 924-row blocks, more blocks than fit (21, 22)
@pytest.mark.parametrize("n,two_m", [(10, 10), (10, -8), (10, 0), (11, 1), (13, 5), (16, 0), (17, -1), (19, 3),
                                     (20, 0), (20, 18), (21, 1), (22, -18)])
@pytest.mark.parametrize("kind", ["j1j2", "pairs", "four", "inexact", "one"])
def test_whole_run_equals_steps(hm, n, two_m, kind, monkeypatch):
    b = hm.Basis(n, 1, two_m)
    bl = hm.BondList.make(*bonds(n, kind))
    x = torch.rand(b.dim, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n)) - 0.25
    whole = hm.lanczos_run(b, bl, 25, v0=x)
    run = hm.LanczosRun(b, bl, 25, v0=x)
    run.step(25)
    al, be, rc = run.read()
    assert whole.status == rc and whole.steps_done == len(al)
    assert np.array_equal(whole.alpha, al) and np.array_equal(whole.beta, be)
    a = hm.e0_grad(b, bl, 25, v0=x, want_psi=True)
    monkeypatch.setenv("HM_BLK_SPLIT", "1")
    c = hm.e0_grad(b, bl, 25, v0=x, want_psi=True)
    assert a[0] == c[0] and a[3] == c[3] and torch.equal(a[2], c[2]) and np.array_equal(a[1], c[1])
