"""Green-Kubo read-outs at the sizes where their kernels change: lags a lane keeps in registers or
recomputes, tables that fit a CTA or come from a launch, rows that do not fill a CTA, runs shorter
than the lags, and the bin-bin window averages read straight from the float-pair state.  The
oracle's FP64 integral of the library's own sums is the reference: both sides add at most 2 L
positive-weight terms in FP64 or in float pairs of 46 bits, so 1e-11 of the integral over the
absolute values covers L up to 1e4 (1e4 * 2^-46 = 1.4e-10 would need every rounding to align; the
errors of the pairs' terms are independent, sqrt(L) 2^-46 = 1.4e-12)."""
import numpy as np
import pytest

import oracle
from tests.parity import check
from tests.test_gpu_parity import make_case, need_gpu, run_gpu

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DT, TK, V = 0.01, 300.0, 320.0
TOL = 1e-11


def window(L, lo=0.3, hi=0.9):
    return lo * (L - 1) * DT, hi * (L - 1) * DT


@pytest.mark.parametrize("L,B", [(1, 1), (31, 2), (33, 3), (256, 1), (257, 5), (6145, 1)])
def test_gkma_reads(L, B):
    need_gpu()
    c = make_case(N=12, M=36, T=90, B=B, seed=9600 + L, drive=2e-3)
    h, _, _ = run_gpu(c, "fp16x3", K=40, L=L, dt_ps=DT, T_K=TK, V_A3=V)
    lo, hi = window(L)
    kt, kw = h.read_kappa_gk(lo, hi)
    C, cnt = h.read_corr()
    okt, skt = oracle.gk_kappa(C, cnt, DT, TK, V), oracle.gk_kappa(np.abs(C), cnt, DT, TK, V)
    check(kt, okt, skt, None, TOL, f"kappa(tau) L={L}")
    pick = [l for l in range(L) if lo <= l * DT <= hi]
    okw = okt[..., pick].mean(-1) if pick else np.zeros(okt.shape[:-1])
    skw = skt[..., pick].mean(-1) if pick else np.zeros(okt.shape[:-1])
    check(kw, okw, skw, None, TOL, f"window beside kappa(tau) L={L}")
    check(h.read_kappa_window(lo, hi), okw, skw, None, TOL, f"window alone L={L}")
    h.close()


@pytest.mark.parametrize("L,B,T", [(1, 1, 20), (33, 7, 90), (40, 22, 17), (3073, 1, 90), (20, 3, 0)])
def test_bin_bin_window_alone(L, B, T):
    from paper_2102_03691_gb300.mhc import ModalHeatCurrent
    need_gpu()
    c = make_case(N=24, M=72, T=max(T, 1), B=B, seed=9700 + L, drive=2e-3)
    h = ModalHeatCurrent(precision="fp16x3", k_max=40, n_lags=L, xcorr=True, dt_ps=DT, T_K=TK, V_A3=V)
    h.set_modes(c["E"], c["mass"], c["f"])
    h.set_bins_uniform(0.0, c["f_hi"], B)
    for t0 in range(0, T, 40):
        h.push(np.ascontiguousarray(c["v"][t0:t0 + 40]), np.ascontiguousarray(c["W"][t0:t0 + 40]))
    lo, hi = window(L)
    _, kw = h.read_kappa_xcorr(lo, hi, with_tau=False)
    X, cnt = h.read_xcorr()
    X = X.reshape(B * B, 3, 3, L)
    okt, skt = oracle.gk_kappa(X, cnt, DT, TK, V), oracle.gk_kappa(np.abs(X), cnt, DT, TK, V)
    pick = [l for l in range(L) if lo <= l * DT <= hi]
    okw = okt[..., pick].mean(-1) if pick else np.zeros(okt.shape[:-1])
    skw = skt[..., pick].mean(-1) if pick else np.zeros(okt.shape[:-1])
    check(kw.reshape(okw.shape), okw, skw, None, TOL, f"bin-bin window L={L} B={B}")
    h.close()
