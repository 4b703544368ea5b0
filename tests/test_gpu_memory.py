"""Device memory that a handle holds beside what its results need: the FP32 product's tail pieces."""
import pytest

from tests.test_gpu_parity import make_case, need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def handle(c, precision, K, **kw):
    from paper_2102_03691_gb300.mhc import ModalHeatCurrent
    h = ModalHeatCurrent(precision=precision, k_max=K, **kw)
    h.set_modes(c["E"], c["mass"], c["f"])
    h.set_bins_uniform(0.0, c["f_hi"], c["B"])
    return h


@pytest.mark.parametrize("direction", [False, True])
def test_fp32_product_holds_one_plane_and_its_tail(direction):
    # E and B take the same bytes in both precisions (4 and 2 + 2), so the difference is the product:
    # a plane [4 K][M_pad] a direction, and second and later pieces of the last wave's tiles, fewer
    # than two of 128 x 128 a resident CTA
    need_gpu()
    N, K = 512, 1024
    c = make_case(N=N, M=3 * N, T=1, B=4, seed=9980)
    a, b = handle(c, "fp32", K, direction=direction), handle(c, "fp16x3", K, direction=direction, split_d=1)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    park = 2 * 96 * 256 * 4 * sms if direction else 0   # the other path's per-CTA direction sums
    plane = 4 * 4 * K * 3 * N * (3 if direction else 1)
    extra = a.info()["device_bytes"] - b.info()["device_bytes"] + park
    assert plane <= extra <= plane + 2 * (2 * sms) * 128 * 128 * 4 + (1 << 20), (extra, plane)
    a.close()
    b.close()
