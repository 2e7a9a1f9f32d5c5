"""Tensor-core contractions on pairs of CTAs (256 x 128 tiles) at the edges of
their range: the smallest, fewer items than pairs, several items per pair, K of
one k-block, a K split, batches of slices with an operand common to all of them.

The persistent executor runs the same contractions on single-CTA tiles, with
the same products added in the same order: the results are equal bit for bit.
Against the FP64 oracle they hold the bounds of the split modes."""

import numpy as np
import pytest

from oracle import tn
from tnc_inputs.network import TensorNetwork

from ._util import floored_rel_err

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = {1: 1e-4, 2: 1e-4, 3: 1e-3, 4: 1e-4}


@pytest.fixture(scope="module")
def lib(libtnc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return libtnc


def _network(mb, nb, kb, n_sliced, seed):
    """A[m,k] B[k,n] D[n,s,o] with n_sliced closed indices s between A and D: the
    node A B varies with the slice through A only."""
    rng = np.random.default_rng(seed)

    def rnd(bits):
        x = rng.standard_normal((2, 1 << bits)).astype(np.float32)
        return (x[0] + 1j * x[1]).astype(np.complex64).reshape((2,) * bits)
    m, k, n = list(range(mb)), list(range(mb, mb + kb)), list(range(mb + kb, mb + kb + nb))
    s = list(range(mb + kb + nb, mb + kb + nb + n_sliced))
    o = [mb + kb + nb + n_sliced]
    a = [x for p in zip(k, m) for x in p] + k[len(m):] + m[len(k):] + s
    b = n[::-1] + k
    tensors = [rnd(len(a)), rnd(len(b)), rnd(nb + n_sliced + 1)]
    dims = np.full(mb + kb + nb + n_sliced + 1, 2, dtype=np.int64)
    return TensorNetwork(tensors, [tuple(a), tuple(b), tuple(n + s + o)], dims, tuple(m + o), [-1] * 3), s


@pytest.mark.parametrize("mode", [1, 2, 3, 4])
@pytest.mark.parametrize("mb,nb,kb,n_sliced", [
    (8, 7, 10, 0),    # one item
    (9, 8, 11, 0),    # 4 items on 76 pairs
    (12, 10, 5, 0),   # 128 items of one k-block (two for 32-bit parts)
    (12, 11, 8, 0),   # 256 items: 3 or 4 per pair, two chunks each
    (8, 7, 13, 0),    # K split over 2 CTA pairs
    (10, 9, 7, 2)])   # 4 slices, B common to them: 64 items (single CTAs) ...
def test_pair_equals_single_tiles(lib, mode, mb, nb, kb, n_sliced):
    from paper_2205_00393_gb300 import Network
    ref_net, s = _network(mb, nb, kb, n_sliced, 100 * mb + 10 * nb + kb)
    net = Network.from_tn(ref_net)
    path = [(0, 1), (2, 3)]
    net.set_path(path)
    net.set_slices(s)
    out = []
    for persistent in (0, 1):
        net.set_option("persistent", persistent)
        out.append(net.contract(0, net.n_slices, mode).cpu().numpy())
        net.check_device()
    assert np.array_equal(out[0], out[1])
    err = floored_rel_err(out[0], tn.contract(ref_net, path, s), 0)
    print("mode %d (%d, %d, %d) sliced %d: %.2e" % (mode, mb, nb, kb, n_sliced, err))
    assert err <= TOL[mode]


@pytest.mark.parametrize("mode", [2, 4])
def test_pair_batch_with_a_common_operand(lib, mode):
    """8 slices of (2^10, 2^9, 2^7) in one launch: 128 items, the planes of B once."""
    test_pair_equals_single_tiles(lib, mode, 10, 9, 7, 3)
