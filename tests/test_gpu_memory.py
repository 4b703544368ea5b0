"""Device memory that a handle holds beside what its results need: the FP32 product's planes and
the split workspace of a tuned shape."""
import os
import subprocess
import sys

import numpy as np
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


_CHILD = r"""
import sys
sys.path.insert(0, sys.argv[1])
from tests.test_gpu_memory import handle
from tests.test_gpu_parity import make_case
from paper_2102_03691_gb300.mhc import ModalHeatCurrentGroup
import numpy as np
cs = [make_case(N=40, M=120, T=16, B=4, seed=9985 + j) for j in range(2)]
def members():
    return [handle(c, "fp16x3", 16) for c in cs]
hs = members()
before = [h.info()["device_bytes"] for h in hs]
g = ModalHeatCurrentGroup(hs)
after = [h.info()["device_bytes"] for h in hs]
g.push([c["v"] for c in cs], [c["W"] for c in cs])
grouped = [h.read_binned_current().copy() for h in hs]
for h in hs:
    h.reset()
for h, c, J in zip(hs, cs, grouped):      # a member pushed by itself gets its workspace back
    h.push(c["v"], c["W"])
    assert np.abs(h.read_binned_current() - J).max() <= 1e-5 * np.abs(J).max()
print("bytes", *before, *after, *[h.info()["device_bytes"] for h in hs])
"""


def test_group_members_hold_no_split_workspace(tmp_path):
    # grouped launches run unsplit: what the members' bins reserved for a tuned split is given back
    need_gpu()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    p = torch.cuda.get_device_properties(0)
    (tmp_path / "tune.txt").write_text(f"{p.multi_processor_count} 2 0 16 0 128 120 128 32 8 1 -1 {p.name}\n")
    (tmp_path / "child.py").write_text(_CHILD)
    r = subprocess.run([sys.executable, str(tmp_path / "child.py"), root],
                       env=dict(os.environ, MHC_TUNE_CACHE=str(tmp_path / "tune.txt")),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    b = list(map(int, r.stdout.split("bytes")[1].split()))
    # 128 columns x 256 modes x 4 bytes a plane, at least one
    assert all(x - y >= 128 * 256 * 4 for x, y in zip(b[:2], b[2:4])), b
    assert all(z >= x for x, z in zip(b[:2], b[4:])), b


def test_an_autotuned_split_that_does_not_fit_runs_unsplit():
    # the direction split's planes of the last wave (453 MB here) with 150 MB left on the device: the
    # push takes the unsplit kernel, and its currents are those of a handle that was told to
    need_gpu()
    from paper_2102_03691_gb300.mhc import ModalHeatCurrent
    N, M, K, B = 3000, 9000, 512, 5
    g = torch.Generator(device="cuda").manual_seed(9995)
    E = torch.randn((3 * N, M), generator=g, device="cuda") / (3 * N) ** 0.5
    v, W = (torch.randn((K, N, q), generator=g, device="cuda") for q in (3, 9))
    f, mass = torch.rand(M, generator=g, device="cuda").cpu().numpy() * 16.0, [28.085] * N

    def handle(split_d, tile_config):
        h = ModalHeatCurrent(precision="fp16x3", k_max=K, direction=True, split_d=split_d, tile_config=tile_config)
        h.set_modes(E, mass, f)
        h.set_bins_uniform(0.0, 16.0, B)
        return h

    ref, h = handle(1, 5), handle(0, 0)
    ref.push(v, W)
    want = ref.read_binned_current()
    warm = handle(1, 0)                       # every tile's kernel is loaded while there is room
    warm.push(v, W)
    warm.sync()
    warm.close()
    torch.cuda.synchronize()
    fill = torch.empty(torch.cuda.mem_get_info()[0] - (150 << 20), dtype=torch.uint8, device="cuda")
    try:
        for _ in range(3):
            h.push(v, W)
        got = h.read_binned_current()
        assert h.info()["tile_split"] == 1
    finally:
        del fill
        torch.cuda.empty_cache()
    np.testing.assert_array_equal(got, want)
    h.close()
    ref.close()
