"""What calls of a network that fits one CTA share (host_tiny.cpp): two streams with a
workspace each, and graphs that hold a call's tables and partial results while
other calls of the same network go on."""

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


def _net(r, c, cycles, n_open, target):
    from paper_2205_00393_gb300 import Network
    net = Network.from_tn(circuit_to_network(grid_rqc(r, c, cycles, 3, n_open=n_open)).as_complex64())
    net.set_path(net.greedy_path())
    net.set_slices(net.find_slices(target, 7))
    return net


def _one_cta(net, call):
    net.set_timing(True)
    out = call().cpu().numpy()
    kinds = [r["kind"] for r in net.last_timings()[0]]
    net.set_timing(False)
    return out, kinds == [9]


def test_two_streams_with_a_workspace_each(lib):
    net = _net(4, 5, 8, 3, 9)
    n = min(net.n_slices, 4096)
    assert n >= 64
    ranges = [(0, n), (n // 2, n)]
    want = []
    for lo, hi in ranges:
        out, tiny = _one_cta(net, lambda: net.contract(lo, hi))
        assert tiny
        want.append(out)
    streams = [torch.cuda.Stream() for _ in ranges]
    ws = [torch.empty(max(net.workspace_bytes(1), 16 * n * net.n_out + 256) // 256 * 256, dtype=torch.uint8, device="cuda")
          for _ in ranges]
    outs = [[torch.zeros(net.n_out, dtype=torch.complex128, device="cuda") for _ in range(20)] for _ in ranges]
    torch.cuda.synchronize()
    for i in range(20):  # both streams hold work at all times
        for q, (lo, hi) in enumerate(ranges):
            net.set_workspace(ws[q])
            net.contract(lo, hi, out=outs[q][i], stream=streams[q])
    torch.cuda.synchronize()
    net.set_workspace(None)
    for q in range(2):
        for o in outs[q]:
            assert np.array_equal(o.cpu().numpy(), want[q])


@pytest.mark.parametrize("r,c,cycles,n_open,target,lo,hi", [(4, 5, 8, 1, 7, 0, 4096), (4, 4, 8, 6, 9, 3, 511), (3, 5, 9, 6, 9, 0, 32)])
def test_partial_results_in_rounds(lib, r, c, cycles, n_open, target, lo, hi):
    """A caller's workspace of one slice, smaller than the call's partial results: rounds
    of them; the same up to the order of FP64 sums (bound of test_tiny_gpu.py)."""
    net = _net(r, c, cycles, n_open, target)
    want, tiny = _one_cta(net, lambda: net.contract(lo, hi))
    assert tiny
    size = net.workspace_bytes(1)
    assert 16 * net.n_out * (hi - lo) > size
    net.set_workspace(torch.empty(size + 256, dtype=torch.uint8, device="cuda")[:size])
    got, tiny = _one_cta(net, lambda: net.contract(lo, hi, out=torch.full((net.n_out,), 7.0, dtype=torch.complex128, device="cuda")))
    assert tiny
    assert np.all(np.abs(got - want) <= 1e-10 * np.abs(want).max())


@pytest.mark.parametrize("per_slice", [False, True])
def test_variants_in_rounds(lib, per_slice):
    """Rounds over whole variants, and (a workspace below one variant's partial results)
    over the slices of each."""
    circuit = grid_rqc(4, 4, 8, 3, n_open=6)
    net = _net(4, 4, 8, 6, 9 if per_slice else 11)
    net.set_leaf_variants(*bitstring_variants(circuit, random_bitstrings(circuit, 9, 5)))
    want, tiny = _one_cta(net, lambda: net.contract_variants(1, 9))
    assert tiny
    size, one = net.workspace_bytes(1), 16 * net.n_out * net.n_slices
    assert (one > size) if per_slice else (one <= size < 8 * one)
    net.set_workspace(torch.empty(size, dtype=torch.uint8, device="cuda"))
    got, tiny = _one_cta(net, lambda: net.contract_variants(1, 9))
    assert tiny
    assert np.all(np.abs(got - want) <= 1e-10 * np.abs(want).max())


def _captured(net, lo, hi, mode):
    """A graph of one call, after a call alike."""
    out = torch.zeros(net.n_out, dtype=torch.complex128, device="cuda")
    net.contract(lo, hi, mode, out=out)
    torch.cuda.synchronize()
    want = out.cpu().numpy()
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        net.contract(lo, hi, mode, out=out)
    return graph, out, want


def _replays(graph, out, want):
    out.fill_(7.0)
    graph.replay()
    torch.cuda.synchronize()
    return np.array_equal(out.cpu().numpy(), want)


def test_captured_call_outlives_larger_ones(lib):
    """The buffer of a captured call's partial results is not freed by a longer range."""
    net = _net(4, 5, 8, 1, 7)
    graphs = [_captured(net, lo, hi, 0) for lo, hi in ((1, 3), (0, 200))]
    net.contract(0, 4096)
    hold = [torch.full((1 << 18,), 3.0, dtype=torch.float64, device="cuda") for _ in range(8)]  # over what is free
    torch.cuda.synchronize()
    assert all(_replays(*g) for g in graphs)
    del hold


def test_captured_call_outlives_other_plans(lib):
    """Its tables are not freed by the plans of other calls that take their place."""
    net = _net(3, 4, 8, 2, 8)
    graph = _captured(net, 0, net.n_slices, 0)
    want = graph[2]
    for cap in range(16, 40):  # another plan key each
        net.set_option("tc_plane_cap_log2", cap)
        assert np.array_equal(net.contract().cpu().numpy(), want)
    hold = [torch.full((1 << 14,), 3.0, dtype=torch.float64, device="cuda") for _ in range(64)]
    assert _replays(*graph)
    del hold


def test_first_call_in_a_capture_falls_back(lib):
    """A longer range than any before it, captured: nothing is allocated on this path; the
    per-level launches, which have run alike, take the call."""
    net = _net(3, 4, 8, 2, 8)
    out = torch.zeros(net.n_out, dtype=torch.complex128, device="cuda")
    net.contract(0, 1)  # one CTA per slice
    net.set_option("persistent", 0)
    want = net.contract(out=out).cpu().numpy()
    net.set_option("persistent", 2)
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        net.contract(out=out)
    assert _replays(graph, out, want)


def test_statistics_of_a_one_cta_call(lib):
    """They name no layout and no executor that did not run; a workspace of two slices is
    still reported as one."""
    net = _net(3, 4, 8, 2, 8)
    net.set_option("persistent", 1)
    net.contract()
    st = net.stats()
    assert st["last_persist_deps"] == 1 and min(st["last_workspace"]) > 0
    net.set_option("persistent", 2)
    net.set_workspace(torch.empty(net.workspace_bytes(2), dtype=torch.uint8, device="cuda"))
    assert _one_cta(net, net.contract)[1]
    st = net.stats()
    assert st["last_persist_deps"] == 0 and st["last_workspace"] == [0, 0] and st["last_batch"] == 2
