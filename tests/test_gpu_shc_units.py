"""The SHC tile reduction where its warps have no unit, one, and several (two tile pairs of one atom
range up to many of several ranges), with lags that do not fill a warp; against the oracle."""
import numpy as np
import pytest

from tests.parity import REL_TOL, check_shc_corr
from tests.test_gpu_parity import make_case, need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,T,nc,K", [(3, 5, 1, 5), (90, 512, 300, 256), (400, 90, 33, 45), (1500, 128, 250, 64)])
def test_shc_units(N, T, nc, K):
    from paper_2102_03691_gb300.mhc import SpectralHeatCurrent
    need_gpu()
    c = make_case(N=N, M=1, T=T, B=1, seed=9600 + N)
    s = SpectralHeatCurrent(N, nc, k_max=K, precision="fp16x3")
    for t in range(0, T, K):
        s.push(np.ascontiguousarray(c["v"][t:t + K]), np.ascontiguousarray(c["W"][t:t + K]))
    Kg, _ = s.read_corr()
    check_shc_corr(Kg, c["v"], c["W"], nc, REL_TOL, f"SHC units N={N} nc={nc} K={K}")
    s.close()
