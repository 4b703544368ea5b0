"""The Green-Kubo read-outs hold FP64 precision beyond the sums they start from: with few lags each
result is a handful of FP64 roundings of the library's own sums, so it is held to those, against
extended precision.

kappa(tau_l) = (c dt / 2) sum_{1 <= m <= l} (C(m-1) + C(m)), C(m) = Csum(m) / (T - m): the division
(as a reciprocal and a product) is 2 roundings a term, the sums of up to 2 L terms in any order at
most 2 L, the prefactor 1 and the constant c dt / 2 of its own 6; an average 2 more.  Each is 2^-53 of
the sum of the absolute values."""
import numpy as np
import pytest

from tests.test_gpu_parity import make_case, need_gpu, run_gpu

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
DT, TK, V = 0.01, 300.0, 320.0
KB, WMK = 8.617333262145179e-5, 1602.176634
LD = np.longdouble


def reference(C, cnt, lo, hi):
    """(kappa(tau), window average, and both with the absolute values of C) in extended precision."""
    L = C.shape[-1]
    half = LD(0.5) * LD(WMK) / (LD(KB) * LD(TK) * LD(TK) * LD(V)) * LD(DT)
    out = []
    for X in (C, np.abs(C)):
        c = X.astype(LD) / np.maximum(cnt, 1).astype(LD) * (cnt > 0)
        kt = np.zeros(c.shape, LD)
        kt[..., 1:] = half * np.cumsum(c[..., :-1] + c[..., 1:], axis=-1)
        pick = [l for l in range(L) if lo <= l * DT <= hi]
        out += [kt, kt[..., pick].mean(-1) if pick else np.zeros(c.shape[:-1], LD)]
    return out


def held(got, want, scale, roundings, what):
    err = np.abs(got.astype(LD) - want)
    bar = roundings * LD(2.0) ** -53 * scale
    assert (err <= bar).all(), f"{what}: {float((err / np.where(bar > 0, bar, 1)).max()):.1f} of the bar"


@pytest.mark.parametrize("L", [2, 3, 5])
@pytest.mark.parametrize("T", [5, 11, 77, 331, 1000])
def test_gkma_reads_hold_fp64(L, T):
    need_gpu()
    c = make_case(N=12, M=36, T=T, B=3, seed=9500 + T, drive=2e-3)
    h, _, _ = run_gpu(c, "fp16x3", K=min(T, 500), L=L, dt_ps=DT, T_K=TK, V_A3=V)
    lo, hi = 0.5 * DT, (L - 1) * DT
    C, cnt = h.read_corr()
    kt, kw, skt, skw = reference(C, cnt, lo, hi)
    gt, gw = h.read_kappa_gk(lo, hi)
    held(gt, kt, skt, 2 * L + 9, f"kappa(tau) L={L} T={T}")
    held(gw, kw, skw, 2 * L + 11, f"window beside kappa(tau) L={L} T={T}")
    held(h.read_kappa_window(lo, hi), kw, skw, 2 * L + 11, f"window alone L={L} T={T}")
    h.close()


def bin_bin(B, L, T, scale=1.0):
    """A handle with T steps of bin-bin sums of L lags, its sums and its origin counts."""
    c = make_case(N=12, M=36, T=T, B=B, seed=9550 + T, drive=2e-3)
    c["v"], c["W"] = (c["v"] * scale).astype(np.float32), (c["W"] * scale).astype(np.float32)
    h, _, _ = run_gpu(c, "fp16x3", K=60, L=L, dt_ps=DT, T_K=TK, V_A3=V, xcorr=True)
    X, cnt = h.read_xcorr()
    return h, X, cnt


@pytest.mark.parametrize("L", [2, 3, 5])
@pytest.mark.parametrize("T", [5, 77, 331])
def test_bin_bin_window_holds_fp64(L, T):
    need_gpu()
    h, X, cnt = bin_bin(7, L, T)
    lo, hi = 0.5 * DT, (L - 1) * DT
    kt, kw, skt, skw = reference(X, cnt, lo, hi)
    _, gw = h.read_kappa_xcorr(lo, hi, with_tau=False)
    held(gw, kw, skw, 2 * L + 11, f"bin-bin window L={L} T={T}")
    gt, gw = h.read_kappa_xcorr(lo, hi)
    held(gt, kt, skt, 2 * L + 9, f"bin-bin kappa(tau) L={L} T={T}")
    held(gw, kw, skw, 2 * L + 11, f"bin-bin window beside kappa(tau) L={L} T={T}")
    h.close()


# sums near the ends of single precision's range, where its products leave it; many outputs and one,
# lags that a thread takes alone, in batches, and shared among threads; a table of a launch
@pytest.mark.parametrize("scale", [2.0 ** -26, 1.0, 2.0 ** 27])
@pytest.mark.parametrize("B,L,T", [(1, 1, 7), (7, 3, 77), (43, 40, 90), (2, 300, 331), (1, 3001, 90)])
def test_bin_bin_window_over_the_range_of_single_precision(B, L, T, scale):
    need_gpu()
    h, X, cnt = bin_bin(B, L, T, scale)
    assert np.isfinite(X).all() and (X != 0).any()
    lo, hi = 0.5 * DT, (L - 1) * DT
    _, kw, _, skw = reference(X, cnt, lo, hi)
    _, gw = h.read_kappa_xcorr(lo, hi, with_tau=False)
    held(gw, kw, skw, 2 * min(L, T) + 11, f"bin-bin window B={B} L={L} T={T} scale={scale}")
    h.close()


@pytest.mark.parametrize("B,L,T", [(7, 40, 90), (43, 40, 90), (2, 400, 331)])
@pytest.mark.parametrize("lo,hi", [(0.0, 0.1), (0.2, 0.5), (0.49, 0.493)])   # early, middle, at most one lag
def test_bin_bin_window_that_ends_early(B, L, T, lo, hi):
    need_gpu()
    h, X, cnt = bin_bin(B, L, T)
    lo, hi = lo * L * DT, hi * L * DT
    _, kw, _, skw = reference(X, cnt, lo, hi)
    _, gw = h.read_kappa_xcorr(lo, hi, with_tau=False)
    held(gw, kw, skw, 2 * L + 11, f"bin-bin window B={B} L={L} {lo}..{hi}")
    h.close()
