"""The adjoint pass under stream capture: a first call of its kind runs node by node, whose
launches carry their parameters, into the caller's workspace; a repeated one by
levels, from tables that other calls of the network do not free."""

import numpy as np
import pytest

from tnc_inputs import circuit_to_network, grid_rqc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture()
def case(libtnc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_00393_gb300 import Network
    tn_ = circuit_to_network(grid_rqc(3, 4, 8, 68, n_open=2)).as_complex64()
    net = Network.from_tn(tn_)
    net.set_path(net.greedy_path())
    net.set_slices(net.find_slices(8, 7))
    rng = np.random.default_rng(3)
    grad = torch.from_numpy(rng.standard_normal(net.n_out) + 1j * rng.standard_normal(net.n_out)).cuda()
    return net, grad


def _capture(net, grad, **kw):
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        env = net.contract_backward(grad, **kw)
    return graph, env


def _replays(graph, env, want):
    env.fill_(7.0)
    graph.replay()
    torch.cuda.synchronize()
    return np.array_equal(env.cpu().numpy(), want)


def test_first_call_in_a_capture(case):
    net, grad = case
    net.contract()  # the leaves are on the device
    net.contract_backward(grad, 0, 1)  # (kernels are loaded)
    ws = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    net.set_workspace(ws)
    graph, env = _capture(net, grad, lo=0, hi=net.n_slices)
    want = net.contract_backward(grad).cpu().numpy()  # by levels
    got = [_replays(graph, env, want) for _ in range(2)]
    assert all(got)


def test_captured_tables_stay(case):
    net, grad = case
    ws = torch.empty(64 << 20, dtype=torch.uint8, device="cuda")
    net.set_workspace(ws)
    want = net.contract_backward(grad).cpu().numpy()
    net.set_timing(True)
    net.contract_backward(grad)
    by_levels = net.last_timings()[1]
    net.set_timing(False)
    net.set_option("backward_keep_every", 2)
    net.set_timing(True)
    net.contract_backward(grad)
    assert by_levels < net.last_timings()[1] / 2  # the level plan is what runs by default
    net.set_timing(False)
    net.set_option("backward_keep_every", 0)
    graph, env = _capture(net, grad)
    for leaf in range(8):  # other masks: other plans
        mask = np.ones(net.n_tensors, dtype=np.uint8)
        mask[leaf] = 0
        net.contract_backward(grad, leaf_mask=mask)
    hold = [torch.full((1 << 14,), 3.0, dtype=torch.float64, device="cuda") for _ in range(256)]  # over what is free
    assert _replays(graph, env, want)
    del hold
