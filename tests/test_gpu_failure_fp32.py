"""The bounded waits of the FP32 product, as tests/test_gpu_failure.py has it for the tensor-core
kernels: MHC_FLAG_TEST_STALL arms a CTA's first stage barrier for 16 bytes more than its copies
deliver, the waits run out (0.1 s), the CTAs wait for the copies in flight and return, and the host
reads MHC_ERR_TIMEOUT; after a reset the handle's results are the oracle's."""
import pytest

from tests.parity import TOL
from tests.test_gpu_parity import make_case, need_gpu, oracle_ref

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("direction", [False, True])
@pytest.mark.parametrize("N,M,K", [(8, 24, 3), (300, 900, 40)])   # one k-block a CTA and less; cut tiles
def test_fp32_wait_times_out_and_context_survives(N, M, K, direction):
    from paper_2102_03691_gb300.mhc import FLAG_TEST_STALL, MhcError, ModalHeatCurrent
    need_gpu()
    c = make_case(N=N, M=M, T=K, B=4, seed=9990)
    h = ModalHeatCurrent(precision="fp32", k_max=K, direction=direction)
    h.set_modes(c["E"], c["mass"], c["f"])
    h.set_bins_uniform(0.0, c["f_hi"], c["B"])
    v, W = torch.from_numpy(c["v"]).cuda(), torch.from_numpy(c["W"]).cuda()
    h.set_flags(FLAG_TEST_STALL)
    h.push(v, W)                     # asynchronous: OK
    with pytest.raises(MhcError) as err:
        h.sync()
    assert err.value.status == 4     # MHC_ERR_TIMEOUT
    h.set_flags(0)
    h.reset()                        # clears the sticky status
    h.push(v, W)
    oracle_ref(c, direction=direction).check_current(h.read_binned_current(), TOL["fp32"], "after the timeout")
    h.close()
