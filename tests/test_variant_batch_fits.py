"""A batch of several variants fits the workspace it was chosen for, although a
smaller batch can need more bytes than a larger one (operands whose planes pass
"tc_plane_cap_log2" are cut into panels). On the CPU the choice is swept over
workspaces and counts by the library's own workspace plan; on the GPU a case whose
evened batch needs more than the workspace equals one variant per call, bit for
bit, and still shares launches."""

import numpy as np
import pytest

from tnc_inputs import bitstring_variants, circuit_to_network, grid_rqc, random_bitstrings


def _net(r, c, cycles, n_open, target, cap):
    from paper_2205_00393_gb300 import Network
    circuit = grid_rqc(r, c, cycles, 3, n_open=n_open)
    net = Network.from_tn(circuit_to_network(circuit).as_complex64())
    net.set_path(net.greedy_path())
    net.set_slices(net.find_slices(target, 7))
    if cap:
        net.set_option("tc_plane_cap_log2", cap)
    return circuit, net


@pytest.mark.parametrize("r,c,cycles,n_open,target,mode,cap", [
    (4, 5, 12, 2, 17, 2, 26), (4, 5, 12, 3, 19, 2, 25), (4, 5, 12, 4, 18, 1, 25), (4, 5, 12, 3, 17, 4, 24),
    (4, 6, 12, 3, 23, 2, 0), (5, 5, 12, 2, 23, 2, 0), (4, 5, 12, 3, 17, 0, 0)])
def test_batch_fits_its_workspace(libtnc, r, c, cycles, n_open, target, mode, cap):
    _, net = _net(r, c, cycles, n_open, target, cap)
    n = net.n_slices
    peak = {}

    def need(b):
        if b not in peak:
            peak[b] = net.arena(b, mode)["peak"]
        return peak[b]

    batched = 0
    for slices in list(range(2 * n, min(48 * n, 200), max(1, n // 3))) + [19, 43]:
        for count in (2, 3, 5, 7, 14, 28, 64):
            got = net.variants_batch(count, mode, need(slices))
            assert got == 0 or (got % n == 0 and got >= 2 * n and need(got) <= need(slices)), (slices, count)
            batched += got > 0
    assert batched
    for count in (2, 9, 40):
        got = net.variants_batch(count, mode)
        assert got == 0 or need(got) <= max(need(1), 1 << 30)


@pytest.mark.gpu
@pytest.mark.parametrize("n_open,target,mode,cap,slices,count", [
    (2, 17, 2, 26, 43, 14), (3, 19, 2, 25, 11, 5), (2, 17, 1, 25, 19, 3), (4, 18, 1, 26, 15, 7)])
def test_evened_batch_needs_more_than_the_workspace(libtnc, n_open, target, mode, cap, slices, count):
    """Workspaces that hold `slices` slices, but not the next smaller number of whole
    variants that evens the batches out."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    circuit, net = _net(4, 5, 12, n_open, target, cap)
    net.set_leaf_variants(*bitstring_variants(circuit, random_bitstrings(circuit, count, 5)))
    size = net.arena(slices, mode)["peak"]
    batch = net.variants_batch(count, mode, size)
    assert batch == 0 or net.arena(batch, mode)["peak"] <= size  # before anything runs
    ws = torch.empty(size, dtype=torch.uint8, device="cuda")
    net.set_workspace(ws)
    net.set_option("persistent", 0)
    net.set_timing(True)
    out = net.contract_variants(0, count, mode=mode).cpu().numpy()
    shared = net.last_timings()[1]
    net.check_device()
    if batch:
        assert net.stats()["last_batch"] == batch
    net.set_timing(True)
    one = np.concatenate([net.contract_variants(v, v + 1, mode=mode).cpu().numpy() for v in range(count)])
    alone = net.last_timings()[1]
    net.check_device()
    assert np.array_equal(out, one)
    assert shared < alone if batch else shared <= alone


@pytest.mark.gpu
def test_batch_that_cannot_be_had(libtnc):
    """On a full device the library's own workspace holds one variant's slices but not
    the batch's: the variants then run one after another."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    mode, count = 2, 20
    circuit, net = _net(4, 5, 12, 4, 18, 0)
    net.set_leaf_variants(*bitstring_variants(circuit, random_bitstrings(circuit, count, 5)))
    net.set_option("persistent", 0)
    out = torch.empty((count, net.n_out), dtype=torch.complex128, device="cuda")
    one = np.concatenate([net.contract_variants(v, v + 1, mode=mode).cpu().numpy() for v in range(count)])
    batch = net.variants_batch(count, mode)
    left = 400 << 20
    assert net.arena(net.n_slices, mode)["peak"] < left // 4 and net.arena(batch, mode)["peak"] > left + (200 << 20)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    full = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    net.contract_variants(0, count, mode=mode, out=out)
    net.check_device()
    del full
    torch.cuda.empty_cache()
    assert np.array_equal(out.cpu().numpy(), one)
    net.contract_variants(0, count, mode=mode, out=out)  # and in a batch again
    assert net.stats()["last_batch"] == batch and np.array_equal(out.cpu().numpy(), one)


@pytest.mark.gpu
def test_many_after_a_workspace_was_lost(libtnc):
    """contract_many replays a kept sequence in the networks' own workspaces. After a batch
    that could not be had, a network's workspace may be a smaller one (at the same
    address, perhaps): the sequence is built anew, and results stay the same."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_00393_gb300 import contract_many
    mode, count = 2, 20
    circuit, net = _net(4, 5, 12, 4, 18, 0)
    _, other = _net(3, 4, 8, 1, 8, 0)
    nets = [net, other]
    for q in nets:
        q.set_option("persistent", 0)
    net.set_leaf_variants(*bitstring_variants(circuit, random_bitstrings(circuit, count, 5)))
    ranges = [(0, 8 * net.n_slices), (0, other.n_slices)]  # (slices of eight variants)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        outs = [torch.empty(q.n_out, dtype=torch.complex128, device="cuda") for q in nets]
        out = torch.empty((count, net.n_out), dtype=torch.complex128, device="cuda")
        for _ in range(3):  # eager, captured, replayed
            contract_many(nets, ranges, mode, outs=outs, stream=stream)
        stream.synchronize()
        want = [o.cpu().numpy() for o in outs]
        torch.cuda.empty_cache()
        left = 400 << 20
        full = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
        net.contract_variants(0, count, mode=mode, out=out, stream=stream)
        net.check_device(stream)
        del full
        torch.cuda.empty_cache()
        for _ in range(2):
            for o in outs:
                o.fill_(float("nan"))
            contract_many(nets, ranges, mode, outs=outs, stream=stream)
            stream.synchronize()
            # (other numbers of slices per batch: bound of test_many_gpu.py)
            assert all(np.allclose(o.cpu().numpy(), w, rtol=1e-9, atol=1e-15) for o, w in zip(outs, want))
