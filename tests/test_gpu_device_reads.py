"""Read-outs into device memory, which the kernels write directly, equal the host read-outs bit for
bit; a destination that no kernel may store doubles to (not 8-byte aligned) still works."""
import ctypes

import numpy as np
import pytest

from tests.test_gpu_parity import make_case, need_gpu, run_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("direction", [False, True])
@pytest.mark.parametrize("shift", [0, 4])
def test_device_reads_equal_host_reads(direction, shift):
    from paper_2102_03691_gb300.mhc import MEM_DEVICE
    need_gpu()
    L, B = 19, 5
    c = make_case(N=20, M=60, T=50, B=B, seed=9800, drive=2e-3)
    h, _, _ = run_gpu(c, "fp16x3", K=25, L=L, direction=direction, xcorr=True)
    lo, hi = 0.03, 0.15

    def dev(n):
        buf = torch.full((8 * n + 8,), 0x5A, dtype=torch.uint8, device="cuda")
        return buf, ctypes.c_void_p(buf.data_ptr() + shift)

    def got(buf, like):
        b = buf.cpu().numpy()
        assert (b[:shift] == 0x5A).all() and (b[shift + 8 * like.size:] == 0x5A).all()
        return np.frombuffer(b[shift:shift + 8 * like.size].tobytes()).reshape(like.shape)

    mean, kap = h.read_hnema()
    kt, kw = h.read_kappa_gk(lo, hi)
    X, _ = h.read_xcorr()
    _, xw = h.read_kappa_xcorr(lo, hi, with_tau=False)
    bm, pm = dev(mean.size)
    bk, pk = dev(kap.size)
    bt, pt = dev(kt.size)
    bw, pw = dev(kw.size)
    bx, px = dev(X.size)
    bv, pv = dev(xw.size)
    f = h._L
    h._check(f.mhc_read_hnema(h._h, pk, pm, MEM_DEVICE))
    h._check(f.mhc_read_kappa_gk(h._h, pt, lo, hi, pw, MEM_DEVICE))
    h._check(f.mhc_read_xcorr(h._h, px, None, MEM_DEVICE))
    h._check(f.mhc_read_kappa_xcorr(h._h, None, lo, hi, pv, MEM_DEVICE))
    torch.cuda.synchronize()
    for buf, like in ((bm, mean), (bk, kap), (bt, kt), (bw, kw), (bx, X), (bv, xw)):
        np.testing.assert_array_equal(got(buf, like), like)
    h.close()
