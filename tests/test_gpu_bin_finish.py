"""The bin finish: block lengths around its thread counts, bins of one and of many partial slots,
and the HNEMA sums of its binned currents, which it adds in FP64.

The inputs of a step are those of one fixed step times a factor in [1, 1.5) 2^(-3 j), j < 7, so a
bin's currents have one sign and lie within a factor 2^19 of each other: their 24-bit values and the
sums of up to 1024 of them (2^10) fit 24 + 19 + 10 = 53 bits, every FP64 addition is exact in any
order, and the mean must equal NumPy's bit for bit."""
import numpy as np
import pytest

from tests.test_gpu_parity import make_case, need_gpu, run_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def scaled_case(N, M, B, T, seed):
    c = make_case(N=N, M=M, T=1, B=B, seed=seed)
    k = np.arange(T)
    a = (1.0 + 0.5 * np.random.default_rng(seed).random(T)) * 2.0 ** (-3 * (k % 7))
    c["v"] = (c["v"] * a[:, None, None]).astype(np.float32)
    c["W"] = np.repeat(c["W"], T, axis=0)
    return c


def exact(Jb):
    """Elements whose FP64 sums over the steps are exact in any order."""
    a = np.abs(Jb.astype(np.float64))
    lo = a.min(axis=0)
    return (lo > 0) & (a.sum(axis=0) <= 2.0 ** 52 * np.spacing(lo.astype(np.float32)).astype(np.float64))


@pytest.mark.parametrize("K,N,M,B", [(1, 8, 24, 3), (127, 8, 24, 3), (128, 200, 600, 1), (129, 20, 60, 4),
                                     (256, 100, 300, 2), (257, 20, 60, 4), (769, 20, 60, 2),
                                     (1000, 20, 60, 5)])
@pytest.mark.parametrize("direction", [False, True])
def test_hnema_sums_are_fp64_sums(K, N, M, B, direction):
    need_gpu()
    c = scaled_case(N, M, B, K, 9900 + K)
    h, Jb, _ = run_gpu(c, "fp32", K=K, direction=direction)
    mean, _ = h.read_hnema()
    want = Jb.astype(np.float64).sum(axis=0) / K
    ok = exact(Jb)
    assert ok.mean() > 0.6, ok.mean()
    np.testing.assert_array_equal(mean[ok], want[ok])
    h.close()


def test_hnema_sums_do_not_depend_on_the_group():
    # a short and a long block in one grouped launch: bitwise the solo sums
    from paper_2102_03691_gb300.mhc import ModalHeatCurrent, ModalHeatCurrentGroup
    need_gpu()
    cs = [make_case(N=20, M=60, T=K, B=4, seed=9950 + K) for K in (100, 300)]

    def handles():
        hs = []
        for c in cs:
            h = ModalHeatCurrent(precision="fp16x3", k_max=300, split_d=1)
            h.set_modes(c["E"], c["mass"], c["f"])
            h.set_bins_uniform(0.0, c["f_hi"], c["B"])
            hs.append(h)
        return hs

    solo, grouped = handles(), handles()
    for h, c in zip(solo, cs):
        h.push(c["v"], c["W"])
    grp = ModalHeatCurrentGroup(grouped)
    grp.push([c["v"] for c in cs], [c["W"] for c in cs])
    for a, b in zip(solo, grouped):
        np.testing.assert_array_equal(a.read_binned_current(), b.read_binned_current())
        np.testing.assert_array_equal(a.read_hnema()[0], b.read_hnema()[0])
    grp.close()


@pytest.mark.parametrize("top", [2.0 ** 127, 2.0 ** 129])   # finite currents; some of them infinite
def test_hnema_sums_beyond_single_precision(top):
    need_gpu()
    T = 40
    c = make_case(N=8, M=24, T=1, B=60, seed=9960)   # a mode or none in most bins: infinities of one sign
    c["v"] = np.repeat(c["v"], T, axis=0)
    c["W"] = np.repeat(c["W"], T, axis=0)
    h, Jb, _ = run_gpu(c, "fp32", K=T)
    h.close()
    s = np.sqrt(top / float(np.abs(Jb).max()))
    c["v"], c["W"] = (c["v"] * s).astype(np.float32), (c["W"] * s).astype(np.float32)
    h, Jb, _ = run_gpu(c, "fp32", K=T)
    assert np.isinf(Jb).any() == (top > 2.0 ** 128)
    assert T * np.abs(Jb[np.isfinite(Jb)].astype(np.float64)).max() > 3.4e38
    mean, _ = h.read_hnema()
    with np.errstate(invalid="ignore"):
        want = Jb.astype(np.float64).sum(axis=0) / T
    np.testing.assert_allclose(mean, want, rtol=T * 2.0 ** -53)
    h.close()
