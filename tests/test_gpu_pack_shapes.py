"""The cluster pack at the shapes where its copies and row ends change: atom counts that are not a
multiple of four (4-byte copies, a partial last group of values), one atom past a CTA and past the
portable cluster size, the widest cluster and the kernel beyond it, inputs in the middle of a
buffer; plain and direction-major rows; against the oracle, and bitwise against the aligned copies
of the same inputs."""
import numpy as np
import pytest

from tests.parity import REL_TOL
from tests.test_gpu_parity import TOL, make_case, need_gpu, oracle_ref, run_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp16x3", "fp32"])
@pytest.mark.parametrize("direction", [False, True])
@pytest.mark.parametrize("N", [2, 511, 513, 1025, 8193])
def test_ragged_atom_counts(N, direction, precision):
    need_gpu()
    c = make_case(N=N, M=min(3 * N, 40), T=3, B=2, seed=9300 + N)
    o = oracle_ref(c, direction=direction)
    h, Jb, J = run_gpu(c, precision, K=3, L=2, direction=direction)
    np.testing.assert_allclose(J, o.J, rtol=1e-12, atol=1e-9 * np.abs(o.J).max())
    o.check_current(Jb, TOL[precision], f"pack N={N} direction={direction}")
    h.close()


@pytest.mark.parametrize("N", [16385, 20000, 32767, 32769])
def test_large_systems(N):
    need_gpu()
    c = make_case(N=N, M=24, T=2, B=2, seed=9400)
    o = oracle_ref(c)
    h, Jb, J = run_gpu(c, "fp16x3", K=2)
    np.testing.assert_allclose(J, o.J, rtol=1e-12, atol=1e-9 * np.abs(o.J).max())
    o.check_current(Jb, REL_TOL, f"pack N={N}")
    h.close()


@pytest.mark.parametrize("N", [64, 1001])
def test_inputs_in_the_middle_of_a_buffer(N):
    from paper_2102_03691_gb300.mhc import ModalHeatCurrent
    need_gpu()
    c = make_case(N=N, M=60, T=4, B=3, seed=9500)
    h, Jb, J = run_gpu(c, "fp16x3", K=4)
    h.close()
    h = ModalHeatCurrent(precision="fp16x3", k_max=4)
    h.set_modes(c["E"], c["mass"], c["f"])
    h.set_bins_uniform(0.0, c["f_hi"], c["B"])

    def shifted(x):
        x = np.ascontiguousarray(x, dtype=np.float32)
        buf = torch.empty(x.size + 1, device="cuda")
        buf[1:] = torch.from_numpy(x.ravel()).cuda()
        return buf[1:].view(x.shape)
    h.push(shifted(c["v"]), shifted(c["W"]))
    np.testing.assert_array_equal(h.read_binned_current(), Jb)
    np.testing.assert_array_equal(h.read_total_current(), J)
    h.close()
