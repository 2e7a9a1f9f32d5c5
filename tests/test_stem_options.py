"""Stem options that change after a network was used: plans kept by the options they
depend on must not serve the new ones. Tensors that a fused group keeps on chip have
no place in its workspace plan, so a plan of other groups has none for tensors that
are now stored."""

import numpy as np
import pytest

from tnc_inputs import circuit_to_network, grid_rqc, stem_path

OPTIONS = [("stem_coalesce_bits", 0), ("stem_coalesce_bits", 6), ("stem_min_outer_log2", 0), ("stem_min_outer_log2", 12),
           ("stem_cap_log2", 10), ("stem_cap_log2", 0)]


def _net():
    from paper_2205_00393_gb300 import Network
    c = grid_rqc(4, 4, 10, 3, n_open=2)
    t = circuit_to_network(c).as_complex64()
    net = Network.from_tn(t)
    net.set_path(stem_path(t, c))
    return net


@pytest.mark.parametrize("key,value", OPTIONS)
def test_plans_follow_the_options(libtnc, key, value):
    def stats(net):
        peak = net.arena(1)["peak"]  # (plans the groups)
        st = net.stats()
        assert st["workspace_batch1"] == net.workspace_bytes(1) == peak
        return st

    used, fresh = _net(), _net()
    before = stats(used)  # plans made with the defaults
    fresh.set_option(key, value)
    used.set_option(key, value)
    a, b = stats(used), stats(fresh)
    assert a["stem_groups"] == b["stem_groups"] != before["stem_groups"]
    assert a["level_cost"] == b["level_cost"] != before["level_cost"]


def test_first_statistics_are_those_of_the_groups(libtnc):
    """tnc_stats reports the workspace and the launches of the fused groups that it lists,
    also before anything else planned them."""
    first, later = _net(), _net()
    a = first.stats()
    later.workspace_bytes(1)
    assert a == later.stats() == first.stats()


@pytest.mark.gpu
@pytest.mark.parametrize("key,value", OPTIONS)
def test_results_follow_the_options(libtnc, key, value):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    net = _net()
    want = net.contract().cpu().numpy()
    net.set_option(key, value)
    got = net.contract().cpu().numpy()
    net.check_device()
    # (sums of at most 2^4 products per step may be ordered differently: 400 steps of 2^-24)
    assert np.max(np.abs(got - want)) <= 400 * 2.0 ** -24 * np.max(np.abs(want))


@pytest.mark.gpu
def test_scalar_branch_without_inner_modes(libtnc):
    """A branch of sliced modes only is a scalar in every slice; with "stem_coalesce_bits" 0
    no mode of the stem has to stay inner. Such a step is no fused group, and the call
    runs."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_00393_gb300 import Network
    from tnc_inputs.network import TensorNetwork
    rng = np.random.default_rng(7)

    def rnd(n):
        return (rng.standard_normal((2,) * n) + 1j * rng.standard_normal((2,) * n)).astype(np.complex64)
    # stem modes 0..13, the sliced mode 14 joins the stem and the branch
    t = TensorNetwork([rnd(8), rnd(7), rnd(1)], [tuple(range(7)) + (14,), tuple(range(7, 14)), (14,)],
                      np.full(15, 2, dtype=np.int64), tuple(range(14)), [-1, -1, -1])
    t2 = TensorNetwork(t.tensors + [rnd(2)], t.indices + [(0, 15)], np.full(16, 2, dtype=np.int64),
                       (15,) + tuple(range(1, 14)), [-1] * 4)
    net = Network.from_tn(t2)
    net.set_path([(0, 1), (4, 2), (5, 3)])
    net.set_slices([14])
    net.set_option("persistent", 0)
    net.set_option("stem_cap_log2", 0)
    want = net.contract().cpu().numpy()
    net.set_option("stem_cap_log2", 13)
    net.set_option("stem_min_outer_log2", 0)
    net.set_option("stem_coalesce_bits", 0)
    got = net.contract().cpu().numpy()
    net.check_device()
    assert all(g[3] > 0 for g in net.stats()["stem_groups"])
    assert np.array_equal(got, want)
