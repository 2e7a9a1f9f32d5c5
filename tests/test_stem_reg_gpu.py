"""Stem groups that run in registers: gates of one and two modes, projections and
steps that add modes, over sub-tensors of 2^9 to 2^12 elements, with and without
coalesced lowest modes (which decides whether the first and last pass load and
store on their own), sliced and in batches. Every output is the same sum in the
same order as in separate launches of the steps, so the results are equal."""

import numpy as np
import pytest

from oracle import tn
from tnc_inputs import circuit_to_network, grid_rqc, stem_path

from ._util import floored_rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libtnc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return libtnc


@pytest.mark.parametrize("rows,cols,cycles,n_open,cap,coalesce,sliced", [
    (4, 5, 9, 4, 12, 3, 0), (4, 5, 9, 0, 12, 0, 2), (4, 5, 8, 6, 11, 3, 1), (4, 5, 10, 1, 10, 2, 0),
    (3, 6, 10, 2, 10, 4, 2), (3, 6, 8, 3, 9, 1, 0), (2, 9, 9, 5, 9, 3, 1), (2, 10, 8, 2, 12, 5, 0)])
def test_groups_equal_separate_steps(lib, rows, cols, cycles, n_open, cap, coalesce, sliced):
    from paper_2205_00393_gb300 import FP32, Network
    c = grid_rqc(rows, cols, cycles, 17 + cap + cols, n_open=n_open)
    tn_ = circuit_to_network(c).as_complex64()
    path = stem_path(tn_, c)
    net = Network.from_tn(tn_)
    net.set_path(path)
    S = [int(e) for e in net.find_slices(c.n_qubits - 2, 7)[:sliced]]
    net.set_slices(S)
    net.set_option("persistent", 0)
    net.set_option("stem_min_outer_log2", 3)
    net.set_option("stem_coalesce_bits", coalesce)
    out = []
    for value in (cap, 0):
        net.set_option("stem_cap_log2", value)
        net.set_timing(True)
        out.append(net.contract(0, net.n_slices, FP32).cpu().numpy())
        kinds = [r["kind"] for r in net.last_timings()[0]]
        net.set_timing(False)
        net.check_device()
        assert (kinds.count(8) > 0) == (value > 0), kinds
    assert np.array_equal(out[0], out[1])
    assert floored_rel_err(out[0], tn.contract(tn_, path, S), c.n_qubits) <= 1e-5
