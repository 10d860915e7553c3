"""GPU test of the sweep form of the general row products against their table form (HM_ROW_RUN = 2
selects the table form), over spins, odd sizes, sectors, repeated pairs and couplings of every kind."""
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


CASES = [(2, 1, 0), (5, 1, 1), (9, 1, 3), (11, 2, 0), (7, 2, 2), (9, 3, 1), (10, 3, 0), (6, 4, 0), (7, 5, 3), (5, 6, 2),
         (5, 7, 1), (4, 7, 28), (40, 1, 34)]


def bonds(hm, n, kind, rng):
    u, v, J = W.ring_bonds(n, -1.0, None if n < 5 else -0.375)
    if kind == "random":                                       # every coupling its own class, mixed signs and sizes
        J = rng.uniform(-1.5, 1.5, len(u)) * 10.0 ** rng.integers(-3, 3, len(u))
    if kind == "many":                                         # repeated pairs: 128 terms, the most the form takes
        k = rng.integers(0, len(u), 128)
        u, v, J = u[k], v[k], rng.uniform(-1, 1, 128)
    return hm.BondList.make(u, v, J)


@pytest.mark.parametrize("kind", ["ring", "random", "many"])
@pytest.mark.parametrize("n,two_s,two_m", CASES, ids=str)
def test_sweep_form_equals_table_form(hm, n, two_s, two_m, kind, monkeypatch):
    """Both forms round a row's sum of T terms in binary64 (binary32): they differ by at most
    2 T eps sum |c x|, bounded here with the row sums of |H|."""
    rng = np.random.default_rng(n * 100 + two_s)
    b = hm.Basis(n, two_s, two_m)
    bl = bonds(hm, n, kind, rng)
    mag = hm.BondList.make(bl.u, bl.v, -np.abs(bl.J))          # exchange elements >= 0: bounds sum |c| off the diagonal
    diag = np.abs(bl.J).sum() * (two_s / 2.0) ** 2
    terms = 3 * len(bl) + 4
    for dtype, eps in ((torch.float64, 2.0**-53), (torch.float32, 2.0**-24)):
        for nvec in (1, 3):
            x = torch.from_numpy(rng.uniform(-1, 1, (b.dim, nvec))).to(dtype).cuda()
            x = x[:, 0].contiguous() if nvec == 1 else x
            one = torch.ones(b.dim, dtype=dtype, device="cuda")
            out = {}
            for run in ("1", "2"):
                monkeypatch.setenv("HM_ROW_RUN", run)
                monkeypatch.setenv("HM_BLK_K", "8")
                out[run] = hm.matvec(b, bl, x).double().cpu().numpy()
                bound = hm.matvec(b, mag, one).abs().max().item() + 2 * diag
            assert np.abs(out["1"] - out["2"]).max() <= 2 * terms * eps * bound
            assert np.abs(out["1"]).max() > 0 or len(bl) == 0 or b.dim == 1


@pytest.mark.parametrize("n,two_s,two_m", [(9, 1, 1), (8, 3, 0), (6, 5, 2)])
def test_sweep_form_lanczos(hm, n, two_s, two_m, monkeypatch):
    """The same alpha, beta from both forms over ten steps, which amplify a rounding by less than 1e3."""
    b = hm.Basis(n, two_s, two_m)
    bl = bonds(hm, n, "ring", None)
    res = {}
    for run in ("1", "2"):
        monkeypatch.setenv("HM_ROW_RUN", run)
        res[run] = hm.lanczos_run(b, bl, 10, seed=3)
    scale = np.abs(res["2"].alpha).max()
    assert np.abs(res["1"].alpha - res["2"].alpha).max() <= 1e3 * len(bl) * 2.0**-46 * scale
    assert np.abs(res["1"].beta - res["2"].beta).max() <= 1e3 * len(bl) * 2.0**-46 * scale


@pytest.mark.parametrize("k", ["0", "half"])
@pytest.mark.parametrize("n,two_s,two_m", [(6, 1, 0), (12, 1, 0), (13, 1, 1), (16, 1, 4), (8, 2, 0), (6, 3, 0), (6, 4, 2)])
def test_sweep_form_momentum(hm, n, two_s, two_m, k, monkeypatch):
    """Momentum blocks, orbits of short period among the targets: the sweep form against the table
    form, within the rounding of a row of T terms (x of size 1, row sums of |H| below sum |J| s (2s + 1),
    orbit factors below sqrt(N))."""
    if k == "half" and n % 2:
        pytest.skip("momentum pi needs an even ring")
    b = hm.Basis(n, two_s, two_m, momentum=0 if k == "0" else n // 2)
    u, v, J = W.ring_bonds(n, -1.0, -0.375)
    bl = hm.BondList.make(u, v, J)
    bound = np.abs(J).sum() * (two_s / 2.0) * (two_s + 1) * np.sqrt(n)
    rng = np.random.default_rng(n)
    for dtype, eps in ((torch.float64, 2.0**-53), (torch.float32, 2.0**-24)):
        x = torch.from_numpy(rng.uniform(-1, 1, b.dim)).to(dtype).cuda()
        out = {}
        for run in ("1", "2"):
            monkeypatch.setenv("HM_ROW_RUN", run)
            out[run] = hm.matvec(b, bl, x).double().cpu().numpy()
        assert np.abs(out["1"] - out["2"]).max() <= 2 * (3 * len(bl) + 4) * eps * bound
