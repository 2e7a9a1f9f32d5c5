"""The final contraction's reductions at the edges of their ranges: K from one
element to several chunks (K = 256 / R: every lane one product), 1 to 64 outputs,
one slice and a batch, on both executors; and root tensors of more than 64
outputs, whose sums the persistent executor cuts into tasks of 1024 outputs.

Bound: products and runs of at most 16 of them are FP32 (each component within
(2 * 16 + 2) 2^-24 of its exact value relative to the sum of |a_k| |b_k|), all
else FP64. Root tensors are FP32 contractions of up to 8 terms."""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib(libtnc):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    return libtnc


@pytest.mark.parametrize("n_sliced", [0, 3])
@pytest.mark.parametrize("mb,nb,kb", [
    (0, 0, 0), (0, 0, 7), (0, 0, 8), (0, 0, 9), (1, 0, 7), (3, 3, 1), (3, 3, 2), (2, 1, 5), (0, 0, 15), (2, 2, 14),
    (3, 3, 16), (5, 5, 3), (6, 5, 2), (9, 5, 3)])
def test_final_contraction(lib, mb, nb, kb, n_sliced):
    from paper_2205_00393_gb300 import FP32, Network
    rng = np.random.default_rng(10000 + 256 * mb + 16 * nb + kb)

    def rnd(bits):
        x = rng.standard_normal((2, 1 << bits)).astype(np.float32)
        return (x[0] + 1j * x[1]).astype(np.complex64).reshape((2,) * bits)
    m, k, n = list(range(mb)), list(range(mb, mb + kb)), list(range(mb + kb, mb + kb + nb))
    s = list(range(mb + kb + nb, mb + kb + nb + n_sliced))
    A, B = rnd(mb + kb + n_sliced), rnd(kb + nb + n_sliced)
    net = Network([A, B], [tuple(k + m + s), tuple(s + n + k)], np.full(mb + kb + nb + n_sliced, 2), tuple(n + m))
    net.set_path([(0, 1)])
    net.set_slices(s)
    Am = A.reshape(1 << kb, 1 << mb, -1).astype(np.complex128)
    Bm = B.reshape(-1, 1 << nb, 1 << kb).astype(np.complex128)
    ref = np.einsum("kms,snk->nm", Am, Bm).reshape(-1)
    size = np.einsum("kms,snk->nm", np.abs(Am), np.abs(Bm)).reshape(-1)
    out = []
    for persistent in (0, 1):
        net.set_option("persistent", persistent)
        out.append(net.contract(0, net.n_slices, FP32).cpu().numpy())
        net.check_device()
    d = out[0] - ref
    err = np.maximum(np.abs(d.real), np.abs(d.imag))
    assert np.all(err <= (2 * 16 + 2) * 2.0 ** -24 * np.sqrt(2) * size)
    assert np.array_equal(out[0], out[1])
