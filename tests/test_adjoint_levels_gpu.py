"""The adjoint pass by tree levels against the node-by-node pass (which runs when
intermediates are recomputed from checkpoints): batches of slices with a
smaller last one, single slices, masked leaves, tensor-core contractions.

Both run the same contractions and add the slices in FP64; only how the FP64
sums are cut into batches may differ, which can move the final rounding to
complex64 by one unit in the last place (2^-23 of the value)."""

import numpy as np
import pytest

from tnc_inputs import circuit_to_network, grid_rqc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libtnc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return libtnc


@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("rows,cols,cycles,n_open,target,lo,hi,slices_per_batch,mode", [
    (2, 2, 4, 2, 2, 0, 3, 2, 0), (3, 3, 6, 1, 3, 1, 8, 2, 0), (3, 4, 8, 0, 8, 0, 16, 16, 0), (3, 4, 8, 3, 8, 5, 6, 1, 0),
    (4, 4, 10, 2, 60, 0, 1, 1, 0),      # no sliced index: every contraction but the last is slice-invariant
    (4, 5, 11, 2, 15, 3, 8, 2, 2), (4, 5, 11, 2, 16, 0, 4, 4, 4), (4, 5, 12, 4, 18, 0, 3, 2, 1)])
def test_levels_match_node_by_node(lib, rows, cols, cycles, n_open, target, lo, hi, slices_per_batch, mode, masked):
    from paper_2205_00393_gb300 import Network
    c = grid_rqc(rows, cols, cycles, 60 + cycles, n_open=n_open)
    tn_ = circuit_to_network(c).as_complex64()
    net = Network.from_tn(tn_)
    net.set_path(net.greedy_path())
    net.set_slices(net.find_slices(target, 7))
    assert hi <= net.n_slices
    rng = np.random.default_rng(hi)
    grad = torch.from_numpy(rng.standard_normal(net.n_out) + 1j * rng.standard_normal(net.n_out))
    mask = None
    if masked:
        mask = np.array([g >= 0 and c.gates[g].name == "fsim" for g in tn_.leaf_gate], dtype=np.uint8)
    net.contract_backward(grad, lo, lo + 1, mode, leaf_mask=mask)
    one = net.stats()["backward_workspace"]
    out = []
    for keep in (0, 2):
        net.set_option("backward_keep_every", keep)
        for _ in range(2):  # planned, then replayed
            env = net.contract_backward(grad, lo, hi, mode, leaf_mask=mask, budget_bytes=int(one * (slices_per_batch + 0.5)))
        net.check_device()
        out.append(env.cpu().numpy())
    rms = float(np.sqrt(np.mean(np.abs(out[1]) ** 2)))
    assert rms > 0
    tol = 2.0 ** -23 * np.maximum(np.abs(out[1]), 1e-3 * rms)
    if mode == 0:
        assert np.all(np.abs(out[0] - out[1]) <= tol)
    else:  # another batch may also split K of a tensor-core contraction differently
        assert float(np.max(np.abs(out[0] - out[1]))) <= 1e-4 * float(np.max(np.abs(out[1])))
