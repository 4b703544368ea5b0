"""The FP32 path's tiles: whole waves, a last wave cut along d into planes that the bin epilogue
adds, the cap on the pieces of a tile, ragged modes, columns and d's, and the direction split's
three products in one launch; against the oracle with the FP32 path's bar (tests/parity.py)."""
import pytest

from tests.test_gpu_parity import TOL, make_case, need_gpu, oracle_ref, run_gpu

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,M,K,direction", [
    (1, 3, 1, False), (1, 3, 1, True),    # one tile of one chunk
    (43, 129, 33, False),                 # a last tile of one mode and of four columns
    (300, 900, 40, False),                # 16 tiles of 8 chunks: the cap of eight pieces
    (300, 900, 100, True),                # 96 tiles of three chunks, three directions
    (700, 2100, 300, False),              # 170 tiles: a whole wave and a cut tail
])
def test_fp32_tiles_against_the_oracle(N, M, K, direction):
    need_gpu()
    c = make_case(N=N, M=M, T=K, B=5, seed=9100 + N, drive=2e-3)
    h, Jb, _ = run_gpu(c, "fp32", K=K, direction=direction)
    oracle_ref(c, direction=direction).check_current(Jb, TOL["fp32"], f"fp32 tiles N={N} K={K}")
    h.close()
