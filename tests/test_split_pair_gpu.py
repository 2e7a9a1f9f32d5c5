"""Both operands of a tensor-core contraction split by one launch, against a launch
per operand (row panels: planes over the cap): the same planes, so the same bits.
Operands of equal and of very different sizes, K below and above one 256-wide chunk,
one slice and a batch, an operand that all slices share."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libtnc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return libtnc


@pytest.mark.parametrize("mode", [1, 2, 3, 4])
@pytest.mark.parametrize("mb,nb,kb,sliced_a,sliced_b", [
    (8, 8, 6, 0, 0), (10, 8, 9, 0, 0), (8, 12, 7, 2, 2), (10, 9, 8, 2, 0), (9, 10, 8, 0, 2)])
def test_split_pair(lib, mode, mb, nb, kb, sliced_a, sliced_b):
    from paper_2205_00393_gb300 import Network
    rng = np.random.default_rng(100 * mb + 10 * nb + kb)

    def rnd(bits):
        x = rng.standard_normal((2, 1 << bits)).astype(np.float32)
        return (x[0] + 1j * x[1]).astype(np.complex64).reshape((2,) * bits)
    m, k, n = list(range(mb)), list(range(mb, mb + kb)), list(range(mb + kb, mb + kb + nb))
    s = list(range(mb + kb + nb, mb + kb + nb + max(sliced_a, sliced_b)))
    sa, sb = s[:sliced_a], s[:sliced_b]
    # sliced indices join two tensors: the operand's own and the last one, or both operands
    last = n + (s if sliced_a != sliced_b else [])
    A, B, D = rnd(mb + kb + len(sa)), rnd(kb + nb + len(sb)), rnd(len(last))
    net = Network([A, B, D], [tuple(k + sa + m), tuple(n + sb + k), tuple(last)], np.full(mb + kb + nb + len(s), 2), tuple(m))
    net.set_path([(0, 1), (2, 3)])
    net.set_slices(s)
    net.set_option("persistent", 0)
    out = {}
    for cap in (32, 16):
        net.set_option("tc_plane_cap_log2", cap)
        net.set_timing(True)
        out[cap] = net.contract(0, net.n_slices, mode).cpu().numpy()
        splits = [r["kind"] for r in net.last_timings()[0]].count(4)
        net.set_timing(False)
        net.check_device()
        assert splits == 1 if cap == 32 else splits >= 2
    assert np.array_equal(out[32], out[16])
