"""Direction-resolved split with the last wave's tiles cut along d (each direction segment of a
tile by itself): every tile shape, several chunks a segment and one, a last range ragged in modes
and columns.  The autotuner alone chooses this plan, so a tuning-cache file with the plan written
in is given to a process of its own, and its currents are held to the oracle's bar."""
import os
import subprocess
import sys

import numpy as np
import pytest

from tests.parity import REL_TOL
from tests.test_gpu_parity import make_case, need_gpu, oracle_ref

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

_CHILD = r"""
import sys
sys.path.insert(0, sys.argv[1])
import numpy as np
from tests.test_gpu_parity import make_case, run_gpu
N, M = int(sys.argv[2]), int(sys.argv[3])
for K in map(int, sys.argv[5:]):
    c = make_case(N=N, M=M, T=2 * K, B=8, seed=9200 + N)
    h, Jb, _ = run_gpu(c, "fp16x3", K=K, direction=True)
    i = h.info()
    assert i["tile_split"] == -1, i
    np.save(f"{sys.argv[4]}/J{K}.npy", Jb)
    h.close()
"""

SHAPES = [(256, 64, 2, 0), (256, 32, 4, 0), (128, 64, 3, 0), (128, 32, 6, 0),
          (256, 64, 3, 1), (256, 32, 6, 1), (128, 64, 4, 1), (128, 32, 8, 1)]


@pytest.mark.parametrize("N,M,K0", [(300, 900, 143), (43, 129, 20), (1500, 4500, 60)])
def test_cut_tiles_of_every_shape(tmp_path, N, M, K0):
    need_gpu()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    shapes = SHAPES if N == 300 else [SHAPES[2], SHAPES[4]]
    props = torch.cuda.get_device_properties(0)
    npad = (N + 127) // 128 * 128
    # line: sm prec dir K split_req D_ld M_eff bn bk stages pair split device
    (tmp_path / "tune.txt").write_text("".join(
        f"{props.multi_processor_count} 2 1 {K0 + q} 0 {3 * npad} {M} {bn} {bk} {st} {pair} -1 {props.name}\n"
        for q, (bn, bk, st, pair) in enumerate(shapes)))
    Ks = [K0 + q for q in range(len(shapes))]
    (tmp_path / "child.py").write_text(_CHILD)
    r = subprocess.run([sys.executable, str(tmp_path / "child.py"), root, str(N), str(M), str(tmp_path)]
                       + list(map(str, Ks)), env=dict(os.environ, MHC_TUNE_CACHE=str(tmp_path / "tune.txt")),
                       capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    for K, shape in zip(Ks, shapes):
        c = make_case(N=N, M=M, T=2 * K, B=8, seed=9200 + N)
        oracle_ref(c, direction=True).check_current(np.load(tmp_path / f"J{K}.npy"), REL_TOL,
                                                    f"direction tail N={N} {shape}")
