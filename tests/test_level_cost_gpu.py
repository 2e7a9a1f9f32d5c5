"""tnc_stats "level_cost" counts the launches that the per-level executor makes of a
batch: grouped and single FP32 contractions (large ones, and those of long K), fused
stem groups, tensor-core contractions with one or two split launches, panels and K
splits, and the final contraction."""

import pytest

from tnc_inputs import circuit_to_network, grid_rqc, stem_path

from .test_parity_tc_gpu import _three_leaf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _launches(net, slices, mode):
    net.set_option("persistent", 0)
    net.contract(0, slices, mode)
    assert net.stats()["last_batch"] == slices
    net.set_timing(True)
    net.contract(0, slices, mode)
    net.check_device()
    ran = net.last_timings()[1]
    net.set_timing(False)
    return ran, net.stats()["level_cost"][str(mode)][0]


@pytest.mark.parametrize("r,c,cycles,n_open,target,slices,options", [
    (3, 4, 8, 1, 8, 16, {}), (4, 5, 12, 3, 17, 8, {}), (4, 6, 12, 3, 20, 2, {}), (4, 6, 12, 3, 23, 1, {}),
    (4, 5, 12, 3, 18, 4, {"tc_plane_cap_log2": 22}), (4, 6, 12, 3, 23, 2, {"tc_plane_cap_log2": 24}),
    (4, 5, 10, 9, 0, 1, {})])
def test_level_cost_counts_launches(libtnc, r, c, cycles, n_open, target, slices, options):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_00393_gb300 import Network
    circuit = grid_rqc(r, c, cycles, 3, n_open=n_open)
    ref = circuit_to_network(circuit).as_complex64()
    net = Network.from_tn(ref)
    net.set_path(net.greedy_path() if target else stem_path(ref, circuit))
    net.set_slices(net.find_slices(target, 7) if target else [])
    for key, value in options.items():
        net.set_option(key, value)
    for mode in (0, 2, 4):
        ran, counted = _launches(net, min(slices, net.n_slices), mode)
        assert ran == counted, mode


def test_level_cost_counts_k_splits(libtnc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_00393_gb300 import Network
    net = Network.from_tn(_three_leaf(401, 7, 7, 16, False))
    net.set_path([(0, 1), (2, 3)])
    for mode in (0, 2, 4):
        ran, counted = _launches(net, 1, mode)
        assert ran == counted, mode
