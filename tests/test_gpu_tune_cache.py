"""The autotuner's results are kept apart for handles with and without cross-correlations, whose
projections run behind other traffic: in the process, in the tuning file, and read back from it.
The file is read once a process, so each case runs in a process of its own."""
import os
import subprocess
import sys

import pytest

from tests.test_gpu_parity import need_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

_CHILD = r"""
import sys
sys.path.insert(0, sys.argv[1])
from tests.test_gpu_parity import make_case, run_gpu
c = make_case(N=40, M=120, T=16, B=4, seed=9970)
for xcorr in map(int, sys.argv[2:]):
    h, _, _ = run_gpu(c, "fp16x3", K=16, L=8, xcorr=bool(xcorr))
    i = h.info()
    print("got", xcorr, i["tile_n"], i["tile_k"], i["stages"], i["tile_pair"], i["tile_split"])
    h.close()
"""


def child(tmp_path, order):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    (tmp_path / "child.py").write_text(_CHILD)
    r = subprocess.run([sys.executable, str(tmp_path / "child.py"), root] + list(map(str, order)),
                       env=dict(os.environ, MHC_TUNE_CACHE=str(tmp_path / "tune.txt")),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    return [tuple(map(int, l.split()[1:])) for l in r.stdout.splitlines() if l.startswith("got")]


@pytest.mark.parametrize("order", [(0, 1), (1, 0)])
def test_each_kind_of_handle_tunes_for_itself(tmp_path, order):
    need_gpu()
    child(tmp_path, order)
    flags = [int(l.split()[2]) for l in (tmp_path / "tune.txt").read_text().splitlines()]
    assert flags == [2 * x for x in order]      # bit 1: cross-correlations


def test_each_kind_of_handle_reads_its_own_line(tmp_path):
    need_gpu()
    p = torch.cuda.get_device_properties(0)
    # line: sm prec flags K split_req D_ld M_eff bn bk stages pair split device
    (tmp_path / "tune.txt").write_text("".join(
        f"{p.multi_processor_count} 2 {flags} 16 0 128 120 {cfg} {p.name}\n"
        for flags, cfg in ((0, "256 64 2 0 1"), (2, "128 32 8 1 1"))))
    assert child(tmp_path, (1, 0)) == [(1, 128, 32, 8, 1, 1), (0, 256, 64, 2, 0, 1)]
    assert len((tmp_path / "tune.txt").read_text().splitlines()) == 2
