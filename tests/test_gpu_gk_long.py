"""Green-Kubo reads where the warps of a row change: 256, 512 and 1024 lags and one more, lags that no
lane holds in registers, rows that do not fill a CTA, many rows of a few more lags, and tables built
by the CTAs and by a launch; held to the roundings of FP64 (tests/test_gpu_gk_precision.py)."""
import numpy as np
import pytest

from tests.test_gpu_gk_precision import DT, TK, V, held, reference
from tests.test_gpu_parity import make_case, need_gpu, run_gpu

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,B,T", [(256, 2, 300), (257, 3, 200), (512, 1, 90), (513, 3, 700), (1024, 1, 1100),
                                   (1025, 5, 400), (2049, 2, 2100), (3001, 1, 90), (700, 60, 90),
                                   (300, 169, 320)])
def test_reads_of_long_curves(L, B, T):
    need_gpu()
    c = make_case(N=12, M=36, T=T, B=B, seed=9400 + L, drive=2e-3)
    h, _, _ = run_gpu(c, "fp16x3", K=500, L=L, dt_ps=DT, T_K=TK, V_A3=V)
    lo, hi = 0.3 * (L - 1) * DT, 0.9 * (L - 1) * DT
    C, cnt = h.read_corr()
    kt, kw, skt, skw = reference(C, cnt, lo, hi)
    gt, gw = h.read_kappa_gk(lo, hi)
    n = min(L, T)          # lags with terms
    held(gt, kt, skt, 2 * n + 9, f"kappa(tau) L={L} B={B}")
    held(gw, kw, skw, 2 * n + L + 9, f"window beside kappa(tau) L={L} B={B}")
    held(h.read_kappa_window(lo, hi), kw, skw, 2 * n + 11, f"window alone L={L} B={B}")
    h.close()
