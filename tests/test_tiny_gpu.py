"""Networks that fit one CTA: the automatic executor's one-CTA path against the
persistent executor and the per-level launches, over the forms that it accepts:
levels of one item and of many, padded item groups, K of one and beyond one
64-term run, final contractions with fewer products than lanes, sliced and
unsliced, ragged and repeated ranges, more slices than CTAs at once, leaf
variants, a caller's workspace, capture; and that what is refused stays refused.

Bound: the FP32 sums of every contraction are the same in the same order on every
path; the FP64 sums over slices and lanes differ by their order at most: 2^12
terms of 2^-53 each are 5e-13 of the largest partial sum, 1e-10 of the largest
output with a cancellation of 200 (another FP32 order would show as 1e-7)."""

import numpy as np
import pytest

from tnc_inputs import bitstring_variants, circuit_to_network, grid_rqc, random_bitstrings

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libtnc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return libtnc


def _net(circuit, target):
    from paper_2205_00393_gb300 import Network
    net = Network.from_tn(circuit_to_network(circuit).as_complex64())
    net.set_path(net.greedy_path())
    if target:
        net.set_slices(net.find_slices(target, 7))
    return net


def _close(a, b):
    return np.all(np.abs(a - b) <= 1e-10 * max(np.abs(b).max(), 1e-300))


def _run(net, persistent, call):
    net.set_option("persistent", persistent)
    net.set_timing(True)
    out = call().cpu().numpy()
    records, launches = net.last_timings()
    net.set_timing(False)
    net.check_device()
    return out, [r["kind"] for r in records], launches


@pytest.mark.parametrize("r,c,cycles,n_open,target,mode", [
    (1, 2, 1, 0, 0, 0), (2, 2, 3, 4, 0, 0), (1, 5, 6, 1, 0, 3), (2, 3, 5, 2, 6, 0), (3, 3, 8, 6, 10, 4), (3, 4, 8, 0, 8, 2),
    (3, 4, 10, 5, 9, 0), (4, 5, 8, 1, 7, 0), (4, 5, 8, 3, 10, 1), (3, 5, 9, 6, 11, 0), (4, 4, 8, 4, 12, 0)])
def test_tiny_ranges(lib, r, c, cycles, n_open, target, mode):
    net = _net(grid_rqc(r, c, cycles, 3, n_open=n_open), target)
    n = min(net.n_slices, 1000)
    for lo, hi in {(0, 1), (0, n), (n // 3, n), (n - 1, n), (n // 2, n // 2)}:
        def call():
            return net.contract(lo, hi, mode, out=torch.full((net.n_out,), 7.0, dtype=torch.complex128, device="cuda"))
        got, kinds, launches = _run(net, 2, call)
        if hi > lo:
            assert kinds == [9] and launches == 2
        for persistent in (1, 0):
            assert _close(got, _run(net, persistent, call)[0])


@pytest.mark.parametrize("r,c,cycles,n_open,target,count", [(3, 3, 8, 5, 0, 5), (3, 4, 8, 0, 8, 23), (4, 4, 8, 2, 10, 7)])
def test_tiny_variants(lib, r, c, cycles, n_open, target, count):
    circuit = grid_rqc(r, c, cycles, 3, n_open=n_open)
    net = _net(circuit, target)
    net.set_leaf_variants(*bitstring_variants(circuit, random_bitstrings(circuit, count, 5)))
    for v, s in (((0, count), (0, net.n_slices)), ((1, count - 1), (net.n_slices // 2, net.n_slices)), ((2, 3), (0, 1))):
        def call():
            return net.contract_variants(*v, *s)
        got, kinds, launches = _run(net, 2, call)
        assert kinds == [9] and launches == 2
        for persistent in (1, 0):
            assert _close(got, _run(net, persistent, call)[0])


def test_tiny_workspace_and_capture(lib):
    from paper_2205_00393_gb300 import TNCError
    net = _net(grid_rqc(3, 4, 8, 1, n_open=2), 8)
    ref = net.contract().cpu().numpy()
    # a workspace that does not hold a slice stays an error, one that does is taken
    need = net.workspace_bytes(1)
    net.set_workspace(torch.empty(need - 256, dtype=torch.uint8, device="cuda"))
    with pytest.raises(TNCError) as e:
        net.contract()
    assert e.value.status == 2
    net.set_workspace(torch.empty(need, dtype=torch.uint8, device="cuda"))
    assert np.array_equal(net.contract().cpu().numpy(), ref)
    assert net.stats()["last_batch"] == 1
    net.set_workspace(None)
    # captured after a first call; the replay reads the leaves of its own time
    out = torch.zeros(net.n_out, dtype=torch.complex128, device="cuda")
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        net.contract(out=out)
    for _ in range(2):
        out.fill_(7.0)
        graph.replay()
        assert np.array_equal(out.cpu().numpy(), ref)
