"""The FP32 contraction kernels at the edges of their tile choice: 64 x 64, 32 x
64 and 64 x 32 tiles, and clusters of 2, 4 and 8 CTAs that share the K of one
tile (few tiles, K >= 128).

Bound: a partial sum adds 64 complex products with FP32 FMAs (128 roundings
per component), and the compensated sum of the partials and the last rounding
add a few more, so each component is within (128 + 8) 2^-24 of the exact
result, relative to the sum of |a_k| |b_k| (a component's terms are at most
that, up to the factor sqrt(2) of |re| + |im|)."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libtnc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return libtnc


def _pair(mb, nb, kb, permuted, seed):
    rng = np.random.default_rng(seed)

    def rnd(bits):
        x = rng.standard_normal((2, 1 << bits)).astype(np.float32)
        return (x[0] + 1j * x[1]).astype(np.complex64).reshape((2,) * bits)
    m, k, n = list(range(mb)), list(range(mb, mb + kb)), list(range(mb + kb, mb + kb + nb))
    a, b = m + k, k + n
    if permuted:
        a = [x for p in zip(k, m) for x in p] + k[len(m):] + m[len(k):]
        b = n[::-1] + k
    A, B = rnd(mb + kb), rnd(kb + nb)
    Am = A.transpose([a.index(e) for e in m + k]).reshape(1 << mb, 1 << kb).astype(np.complex128)
    Bm = B.transpose([b.index(e) for e in k + n]).reshape(1 << kb, 1 << nb).astype(np.complex128)
    return [A, B], [tuple(a), tuple(b)], np.full(mb + kb + nb, 2), tuple(m + n), k, Am, Bm


@pytest.mark.parametrize("n_sliced", [0, 2])
@pytest.mark.parametrize("permuted", [False, True])
@pytest.mark.parametrize("mb,nb,kb", [
    (7, 0, 7), (2, 5, 9), (6, 2, 10),     # narrow: clusters of 2 and 8 on 64 x 32 tiles
    (6, 6, 7), (6, 6, 8), (5, 7, 11),     # clusters of 2, 4 and 8 on 32 x 64 tiles
    (10, 9, 8), (10, 9, 6),               # 256 tiles of 32 x 64, with and without clusters
    (11, 9, 7), (11, 9, 2), (14, 3, 4),   # more: 64 x 64 tiles, and narrow ones without clusters
    (7, 6, 0), (3, 4, 3), (6, 7, 5)])     # K below one k-tile, one, two
def test_pair_within_rounding(lib, mb, nb, kb, permuted, n_sliced):
    from paper_2205_00393_gb300 import FP32, Network
    if kb < n_sliced:
        pytest.skip("no contracted index to slice")
    tensors, indices, dims, open_ids, k, A, B = _pair(mb, nb, kb + n_sliced, permuted, 1000 + 64 * mb + 8 * nb + kb)
    net = Network(tensors, indices, dims, open_ids)
    net.set_path([(0, 1)])
    net.set_slices(k[:n_sliced])
    out = {}
    for persistent in (0, 1):
        net.set_option("persistent", persistent)
        out[persistent] = net.contract(0, net.n_slices, FP32).cpu().numpy().reshape(1 << mb, 1 << nb)
        net.check_device()
    ref, size = A @ B, np.abs(A) @ np.abs(B)
    err = np.maximum(np.abs((out[0] - ref).real), np.abs((out[0] - ref).imag))
    print("(%d, %d, %d) sliced %d: worst error %.2e of the sum of |a||b|" % (mb, nb, kb, n_sliced, np.max(err / size)))
    assert np.all(err <= (128 + 8) * 2.0 ** -24 * np.sqrt(2) * size)
    # every tile shape, and a cluster, adds the same partials in the same order
    assert np.array_equal(out[0], out[1])
