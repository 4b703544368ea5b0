"""The lag correlation of many tiles (from 700: a CTA of few warps each, or clusters for blocks of 16
warps): one step, ragged bins and lags, one to sixteen warps of steps.  The stage is judged alone
(tests/test_gpu_lag_plan.py has the bound)."""
import numpy as np
import pytest

from tests.parity import REL_TOL, stage_corr_check
from tests.test_gpu_parity import make_case, need_gpu, run_gpu

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,B,L", [(1, 304, 310), (32, 301, 300), (33, 304, 310), (200, 280, 320), (390, 281, 318),
                                   (500, 70, 1250)])
def test_lag_stage_of_many_tiles(K, B, L):
    need_gpu()
    T = 2 * K + (K + 1) // 2
    c = make_case(N=16, M=48, T=T, B=B, seed=9050 + K, drive=2e-3)
    h, Jb, J = run_gpu(c, "fp16x3", K=K, L=L)
    C, cnt = h.read_corr()
    np.testing.assert_array_equal(cnt, np.maximum(T - np.arange(L), 0))
    stage_corr_check(C, Jb, J, L, REL_TOL, f"lag stage K={K} B={B} L={L}")
    h.close()
