"""Several variants per launch (tnc_contract_variants over every slice) against one
variant per call: bit for bit, since every contraction, slice sum and final sum
keeps its terms and their order. Sliced and unsliced, stem groups, tensor cores,
final contractions and root tensors, one batch, uneven batches in a small
workspace, a workspace of one variant, and kept invariants."""

import numpy as np
import pytest

from tnc_inputs import bitstring_variants, circuit_to_network, grid_rqc, random_bitstrings, stem_path

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libtnc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return libtnc


@pytest.mark.parametrize("r,c,cycles,n_open,target,count,mode", [
    (4, 4, 10, 2, 0, 7, 0),    # stem groups, final contraction
    (4, 4, 9, 9, 0, 5, 0),     # stem, a root tensor of 512 outputs
    (3, 7, 10, 1, 12, 6, 2),   # sliced, FP32 contractions
    (4, 5, 12, 9, 17, 5, 0),   # sliced, a root tensor
    (4, 6, 12, 3, 19, 4, 3),   # sliced, tensor cores
    (4, 6, 12, 4, 20, 3, 4),   # (more slices than a batch: one variant after another)
    (4, 6, 12, 3, 23, 4, 2),   # tensor cores, few slices
    (4, 6, 12, 4, 23, 5, 4)])
def test_variant_batches(lib, r, c, cycles, n_open, target, count, mode):
    from paper_2205_00393_gb300 import Network
    circuit = grid_rqc(r, c, cycles, 3, n_open=n_open)
    ref = circuit_to_network(circuit).as_complex64()
    net = Network.from_tn(ref)
    net.set_path(net.greedy_path() if target else stem_path(ref, circuit))
    if target:
        net.set_slices(net.find_slices(target, 7))
    net.set_leaf_variants(*bitstring_variants(circuit, random_bitstrings(circuit, count, 5)))
    net.set_option("persistent", 0)
    n = net.n_slices

    def check(v0=0, v1=count):
        # (in the same workspace: how many slices share a batch decides the order of their sum)
        one = np.concatenate([net.contract_variants(v, v + 1, mode=mode).cpu().numpy().reshape(1, -1)
                              for v in range(v0, v1)])
        out = torch.full((v1 - v0, net.n_out), 7.0, dtype=torch.complex128, device="cuda")
        net.contract_variants(v0, v1, mode=mode, out=out)
        net.check_device()
        assert np.array_equal(out.cpu().numpy(), one)

    check()
    check(1, count - 1)
    for variants in (2, 1):
        ws = torch.empty(net.arena(min(n * variants, 1024), mode)["peak"] + 256, dtype=torch.uint8, device="cuda")
        net.set_workspace(ws[:ws.numel() // 256 * 256])
        check()
    net.set_workspace(None)
    net.set_option("cache_invariants", 1)
    check()
    check()
    net.set_option("cache_invariants", 0)
    # a part of the slices: their ids are not consecutive over the variants
    if n > 1:
        part = net.contract_variants(0, count, 1, n, mode=mode).cpu().numpy()
        for v in range(count):
            assert np.array_equal(part[v], net.contract_variants(v, v + 1, 1, n, mode=mode).cpu().numpy().reshape(-1))
