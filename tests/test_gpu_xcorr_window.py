"""The cross-correlation windows where their kernel changes: one step and one lag, blocks that go
through the ring's wrap-around, windows of whole and ragged 64-step rows, and one too long for
shared memory; against the oracle's sums of the library's own binned currents (split FP16 operands of
22 bits under a row scale, FP32 sums of 128 steps: inside the 1e-5 bar of the sum of absolute
values)."""
import numpy as np
import pytest

import oracle
from tests.parity import REL_TOL, check
from tests.test_gpu_parity import make_case, need_gpu, run_gpu

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,L,K,T", [(1, 1, 1, 9), (3, 40, 7, 33), (43, 9, 70, 150), (5, 33, 32, 100),
                                     (2, 65, 64, 200), (1, 12300, 20, 90)])
def test_bin_bin_stage_alone(B, L, K, T):
    need_gpu()
    c = make_case(N=40, M=120, T=T, B=B, seed=9900 + B, drive=2e-3)
    h, Jb, _ = run_gpu(c, "fp16x3", K=K, L=L, xcorr=True)
    X, cnt = h.read_xcorr()
    np.testing.assert_array_equal(cnt, np.maximum(T - np.arange(L), 0))
    o, S = oracle.gkma_xcorr(Jb, L), oracle.gkma_xcorr(np.abs(Jb), L)
    check(X, o, S, None, REL_TOL, f"bin-bin stage B={B} L={L} K={K}")
    h.close()
