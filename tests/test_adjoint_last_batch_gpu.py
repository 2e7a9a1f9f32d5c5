"""The node-by-node adjoint pass with a smaller last batch that needs more workspace than
the others (its operand planes are not cut into panels): the workspace is sized for
both, and nothing is written past it. The circuits' last batches need up to 5% more."""

import numpy as np
import pytest

from tnc_inputs import circuit_to_network, grid_rqc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_open,target,cap,keep,hi,budget_mb", [
    (3, 18, 24, 2, 15, 100), (3, 18, 24, 4, 15, 100), (3, 18, 24, 2, 15, 85)])
def test_last_batch_stays_inside(libtnc, n_open, target, cap, keep, hi, budget_mb):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2205_00393_gb300 import Network
    net = Network.from_tn(circuit_to_network(grid_rqc(4, 5, 12, 3, n_open=n_open)).as_complex64())
    net.set_path(net.greedy_path())
    net.set_slices(net.find_slices(target, 7))
    net.set_option("tc_plane_cap_log2", cap)
    net.set_option("backward_keep_every", keep)
    rng = np.random.default_rng(hi)
    grad = torch.from_numpy(rng.standard_normal(net.n_out) + 1j * rng.standard_normal(net.n_out)).cuda()
    assert hi <= net.n_slices
    guard = torch.full((256 << 20,), 0x5A, dtype=torch.uint8, device="cuda")  # the workspace is its beginning

    def run():
        env = net.contract_backward(grad, 0, hi, 4, budget_bytes=budget_mb << 20)
        net.check_device()
        return env.cpu().numpy(), net.stats()["backward_workspace"]

    net.set_workspace(guard)
    want, size = run()
    assert size <= budget_mb << 20 and hi % net.stats()["last_batch"]
    assert bool((guard[size:] == 0x5A).all())
    guard.fill_(0x5A)
    net.set_workspace(guard[:(size + 255) // 256 * 256])
    got, again = run()
    assert again == size and np.array_equal(got, want)
    assert bool((guard[(size + 255) // 256 * 256:] == 0x5A).all())
