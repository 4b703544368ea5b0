"""A group with a system beyond the cluster pack (32768 atoms) packs its systems one by one: bitwise the
solo pushes."""
import numpy as np
import pytest

from tests.test_gpu_parity import make_case, need_gpu

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_group_with_a_system_beyond_the_cluster_pack():
    from paper_2102_03691_gb300.mhc import ModalHeatCurrent, ModalHeatCurrentGroup
    need_gpu()
    K, L = 6, 3
    cs = [make_case(N=N, M=M, T=2 * K, B=4, seed=9700 + N) for N, M in ((200, 600), (32771, 24), (43, 129))]

    def handles():
        hs = []
        for c in cs:
            h = ModalHeatCurrent(precision="fp16x3", k_max=K, n_lags=L, split_d=1)
            h.set_modes(c["E"], c["mass"], c["f"])
            h.set_bins_uniform(0.0, c["f_hi"], c["B"])
            hs.append(h)
        return hs

    solo, grouped = handles(), handles()
    grp = ModalHeatCurrentGroup(grouped)
    for t in (0, K):
        vs, Ws = ([np.ascontiguousarray(c[x][t:t + K]) for c in cs] for x in ("v", "W"))
        for h, v, W in zip(solo, vs, Ws):
            h.push(v, W)
        grp.push(vs, Ws)
        for a, b in zip(solo, grouped):
            np.testing.assert_array_equal(a.read_binned_current(), b.read_binned_current())
            np.testing.assert_array_equal(a.read_total_current(), b.read_total_current())
    for a, b in zip(solo, grouped):
        np.testing.assert_array_equal(a.read_corr()[0], b.read_corr()[0])
        np.testing.assert_array_equal(a.read_hnema()[0], b.read_hnema()[0])
    grp.close()
