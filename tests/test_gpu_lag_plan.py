"""The lag correlation's split of a block over warps and CTAs: one warp with one step, warps
without steps, one CTA a tile, clusters of two to four CTAs, ragged last ranks, bins and lags that
do not fill a tile.  The stage is judged alone, against the oracle's lag sums of the library's own
binned currents: FP32 partial sums over at most 64 steps err by at most 66 * 2^-24 = 4e-6 of the
sum of the absolute values of their terms, inside the 1e-5 bar."""
import numpy as np
import pytest

from tests.parity import REL_TOL, stage_corr_check
from tests.test_gpu_parity import make_case, need_gpu, run_gpu

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,B,L", [
    (1, 1, 1), (3, 5, 33), (7, 4, 40),      # one CTA a tile, fewer warps with steps than warps
    (32, 8, 8), (77, 37, 123),              # one CTA a tile, 8 and 16 warps
    (61, 301, 20), (64, 304, 32),           # 76 tiles: clusters (B % 4 != 0, and 16-byte copies)
    (250, 64, 200), (1000, 100, 200),       # clusters of four CTAs
    (1023, 3, 1000),                        # the largest block, 32 tiles
])
def test_lag_stage_alone(K, B, L):
    need_gpu()
    T = 2 * K + (K + 1) // 2   # two whole blocks and a ragged one
    c = make_case(N=16, M=48, T=T, B=B, seed=9000 + K, drive=2e-3)
    h, Jb, J = run_gpu(c, "fp16x3", K=K, L=L)
    C, cnt = h.read_corr()
    np.testing.assert_array_equal(cnt, np.maximum(T - np.arange(L), 0))
    stage_corr_check(C, Jb, J, L, REL_TOL, f"lag stage K={K} B={B} L={L}")
    h.close()
