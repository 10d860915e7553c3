"""GPU test of the bounded grid barriers of the whole-run kernel (csrc/lz_small.cu): with a limit of 0 ns no
CTA waits for another, every CTA returns, and the call reports HM_ETIMEOUT (no fault, no hang);
the next call on the same device is correct."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_0706_3293_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limits,call", [("0", "lanczos_run"), ("0", "e0_grad"), ("5000000000,0", "e0_grad")],
                         ids=["lanczos_run", "e0_grad pass 1", "e0_grad pass 2"])
def test_barrier_gives_up_and_device_stays_usable(limits, call, monkeypatch):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_0706_3293_gb300 import _capi, api
    b = api.Basis(16, 1, 0)
    bl = api.BondList.make(*W.ring_bonds(16, -1.0, -0.3))
    run = lambda: api.lanczos_run(b, bl, 30, seed=3) if call == "lanczos_run" else api.e0_grad(b, bl, 60, seed=3)
    ok = run()
    monkeypatch.setenv("HM_LZ_BARRIER_NS", limits)
    with pytest.raises(_capi.HMError) as ei:
        run()
    assert ei.value.code == _capi.HM_ETIMEOUT
    if "," in limits:                                     # the second limit is of e0_grad's second pass alone
        assert api.lanczos_run(b, bl, 30, seed=3).steps_done == 30
    monkeypatch.delenv("HM_LZ_BARRIER_NS")
    again = run()
    if call == "lanczos_run":
        assert np.array_equal(ok.alpha, again.alpha) and np.array_equal(ok.beta, again.beta)
    else:
        assert ok[0] == again[0] and np.array_equal(ok[1], again[1])
    torch.cuda.synchronize()
