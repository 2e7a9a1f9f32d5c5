"""Performance cases: the work that users of this library have it do, through
its public entry points (``Network``, ``contract_many``, ``CircuitAmplitudes``).

A case is a dict of plain values. Its ``kind`` is one of

* ``slices``: slices [lo, hi) of a grid circuit along the greedy path
  (``Network.contract``): amplitudes, from one launch-bound call to the
  30-qubit benchmark workload;
* ``stem``: the same along the time-ordered stem path, where every step is
  narrow;
* ``variants``: a batch of correlated bitstrings (``contract_variants``);
* ``many``: circuits of uneven size together (``contract_many``);
* ``gradient``: amplitudes and gate-parameter gradients of one training step
  (``CircuitAmplitudes``);
* ``environments``: the adjoint pass alone (``contract_backward``);
* ``pair``: one contraction of two tensors, its whole result read out;
* ``triple``: one contraction inside a network, A B, followed by a small D.

Inputs follow the seeded generators of ``tnc_inputs``: the seed draws the
gates, bitstrings and tensor entries; sizes come from the case alone, so that
every seed runs the same plan. ``exact`` simulates the circuits as state
vectors (sliced indices are projectors on their wire segments) or multiplies
the matrices, in complex128 with plain PyTorch.
"""

import math

import numpy as np
import torch

from paper_2205_00393_gb300 import (FP32, SPLIT_BF16, SPLIT_BF16X2, SPLIT_FP16X2, SPLIT_TF32, Network,
                                    contract_many)
from paper_2205_00393_gb300.torch_fn import CircuitAmplitudes
from tnc_inputs import bitstring_variants, circuit_to_network, grid_rqc, random_bitstrings, stem_path
from tnc_inputs.network import TensorNetwork

MODES = {"fp32": FP32, "tf32": SPLIT_TF32, "bf16": SPLIT_BF16, "bf16x2": SPLIT_BF16X2, "fp16x2": SPLIT_FP16X2}
SA_SEED = 7  # of the slice refiner, as in the benchmark


# ------------------------------------------------------------------- cases


def listed():
    return [
        # one amplitude of a small circuit, every slice: the shortest call, all launches and dependencies
        {"name": "slices-12q-fp32", "kind": "slices", "rows": 3, "cols": 4, "cycles": 8, "n_open": 0, "target": 8,
         "lo": 0, "hi": 16, "mode": "fp32"},
        # 16 amplitudes of a 20-qubit circuit in the most accurate tensor-core mode, every slice
        {"name": "slices-20q-bf16", "kind": "slices", "rows": 4, "cols": 5, "cycles": 12, "n_open": 4, "target": 16,
         "lo": 0, "hi": 16, "mode": "bf16"},
        # a block of slices of a 24-qubit circuit in the default arithmetic; an odd number of them
        {"name": "slices-24q-fp32", "kind": "slices", "rows": 4, "cols": 6, "cycles": 12, "n_open": 0, "target": 20,
         "lo": 5, "hi": 12, "mode": "fp32"},
        # all slices of a 25-qubit circuit in split TF32
        {"name": "slices-25q-tf32", "kind": "slices", "rows": 5, "cols": 5, "cycles": 14, "n_open": 4, "target": 22,
         "lo": 0, "hi": 32, "mode": "tf32"},
        # the benchmark workload: one call of 4 slices of the 30-qubit circuit
        {"name": "slices-30q-fp16x2", "kind": "slices", "rows": 5, "cols": 6, "cycles": 14, "n_open": 6,
         "target": 27, "lo": 8, "hi": 12, "mode": "fp16x2"},
        # the 28-qubit stem path (secondary slicing), a 2 GiB stem that absorbs one gate after another
        {"name": "stem-28q-fp32", "kind": "stem", "rows": 4, "cols": 7, "cycles": 12, "n_open": 4, "sliced": 0,
         "mode": "fp32"},
        # correlated samples: 23 bitstrings that share the state before their projections
        {"name": "variants-24q-fp32", "kind": "variants", "rows": 4, "cols": 6, "cycles": 10, "n_open": 6,
         "path": "stem", "target": 0, "count": 23, "mode": "fp32"},
        # the batched uneven workload: its first circuits, 2 slices each, replayed from a graph
        {"name": "many-20-bf16", "kind": "many", "first": 0, "circuits": 20, "slices": 2, "mode": "bf16"},
        # one training step on a 16-qubit circuit: amplitudes and all fSim gradients
        {"name": "gradient-16q-fp32", "kind": "gradient", "rows": 4, "cols": 4, "cycles": 10, "n_open": 2,
         "target": 12, "mode": "fp32"},
        # the adjoint pass of a 25-qubit circuit over every slice: environments of all fSim gates
        {"name": "environments-25q-bf16", "kind": "environments", "rows": 5, "cols": 5, "cycles": 12, "n_open": 2,
         "target": 22, "mode": "bf16"},
        # two tensors with permuted modes, FP32, M = 2^11, N = 2^10, K = 2^12
        {"name": "pair-fp32", "kind": "pair", "mb": 11, "nb": 10, "kb": 12, "permuted": True, "mode": "fp32"},
        # a large contraction in split FP16x2 (M = 2^12, N = 2^11, K = 2^12) and the 64 columns that follow it
        {"name": "triple-fp16x2", "kind": "triple", "mb": 12, "nb": 11, "kb": 12, "ob": 6, "permuted": True,
         "mode": "fp16x2"},
    ]


_GRIDS = [(3, 3), (3, 4), (3, 5), (4, 4), (4, 5), (3, 7), (4, 6), (5, 5), (5, 6)]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _draw_slices(rng):
    mode = rng.choice(["fp32", "fp32", "tf32", "bf16", "bf16", "bf16x2", "fp16x2", "fp16x2"])
    rows, cols = rng.choice(_GRIDS)
    n_open = rng.randint(0, 6)
    case = {"kind": "slices", "rows": rows, "cols": cols, "cycles": rng.randint(8, 14), "n_open": n_open,
            "target": 62, "lo": 0, "hi": 1, "mode": mode}
    net, _, _ = _plan(case, 0)
    width = net.stats()["max_log2_size"]
    case["target"] = int(max(n_open + 4, min(width - rng.randint(2, 7), 27)))
    net, tn, path = _plan(case, 0)
    # complex multiply-accumulates of the call: at most the listed calls'
    most = 2.0 ** 36 if mode == "fp32" else 2.0 ** 40
    budget = _log_uniform(rng, 2.0 ** 16, most)
    n = net.n_slices
    while n > 1 and _cmacs(tn, path, net.sliced, n) > budget:
        n //= 2
    if _cmacs(tn, path, net.sliced, n) > most:
        return None
    if n > 4 and rng.random() < 0.5:  # a ragged block
        n -= rng.randint(1, n // 2)
    n = min(n, 1024)
    case["lo"] = rng.randint(0, net.n_slices - n)
    case["hi"] = case["lo"] + n
    return case


def _draw_stem(rng):
    rows, cols = rng.choice([(4, 5), (3, 7), (4, 6), (5, 5), (4, 6), (2, 13)])
    return {"kind": "stem", "rows": rows, "cols": cols, "cycles": rng.randint(8, 12), "n_open": rng.randint(1, 6),
            "sliced": rng.randint(0, 2), "mode": "fp32"}


def _draw_variants(rng):
    stem = rng.random() < 0.6
    rows, cols = rng.choice([(4, 4), (4, 5), (3, 7), (4, 6)] if stem else [(3, 3), (3, 4), (4, 4), (4, 5)])
    return {"kind": "variants", "rows": rows, "cols": cols, "cycles": rng.randint(8, 10), "n_open": rng.randint(0, 6),
            "path": "stem" if stem else "greedy", "target": 0 if stem else rng.randint(10, 14),
            "count": round(_log_uniform(rng, 2, 40)), "mode": rng.choice(["fp32", "bf16", "fp16x2"])}


def _draw_many(rng):
    return {"kind": "many", "first": rng.randint(1, 160), "circuits": rng.randint(3, 10), "slices": rng.randint(1, 2),
            "mode": rng.choice(["fp32", "bf16", "fp16x2"]), "small": True}


def _draw_gradient(rng):
    rows, cols = rng.choice([(2, 3), (3, 3), (3, 4), (4, 4), (4, 5)])
    return {"kind": "gradient", "rows": rows, "cols": cols, "cycles": rng.randint(4, 10), "n_open": rng.randint(0, 4),
            "target": rng.randint(9, 14), "mode": rng.choice(["fp32", "fp32", "bf16", "fp16x2"])}


def _draw_environments(rng):
    rows, cols = rng.choice([(3, 4), (4, 4), (4, 5), (4, 6), (5, 5)])
    return {"kind": "environments", "rows": rows, "cols": cols, "cycles": rng.randint(8, 12),
            "n_open": rng.randint(0, 4), "target": rng.randint(17, 22),
            "mode": rng.choice(["fp32", "tf32", "bf16", "fp16x2"])}


def _draw_pair(rng):
    while True:
        mb, nb, kb = rng.randint(2, 13), rng.randint(0, 12), rng.randint(0, 13)
        if 8 <= mb + nb + kb <= 34 and max(mb + kb, nb + kb, mb + nb) <= 23:
            return {"kind": "pair", "mb": mb, "nb": nb, "kb": kb, "permuted": rng.random() < 0.7, "mode": "fp32"}


def _draw_triple(rng):
    while True:
        mb, nb, kb = rng.randint(7, 13), rng.randint(7, 12), rng.randint(5, 13)
        if mb + nb + kb <= 35 and max(mb + kb, nb + kb, mb + nb) <= 24:
            return {"kind": "triple", "mb": mb, "nb": nb, "kb": kb, "ob": rng.randint(1, 6),
                    "permuted": rng.random() < 0.7, "mode": rng.choice(["tf32", "bf16", "bf16x2", "fp16x2"])}


def draw(rng):
    makers = [_draw_slices] * 4 + [_draw_stem, _draw_variants, _draw_many, _draw_gradient, _draw_environments,
                                   _draw_pair, _draw_pair, _draw_triple, _draw_triple]
    while True:
        case = rng.choice(makers)(rng)
        if case is None:
            continue
        if case["kind"] == "many":  # not more than the listed batch
            if work(case)["flops"] > work(listed()[7])["flops"]:
                continue
        elif case["kind"] not in ("pair", "triple", "slices"):
            if work(case)["flops"] > 8 * 2.0 ** (36 if case["mode"] == "fp32" else 38):
                continue
        return case


# ------------------------------------------------------------------ inputs


def _circuit(case, seed):
    return grid_rqc(case["rows"], case["cols"], case["cycles"], int(seed), n_open=case["n_open"])


def _plan(case, seed, circuit=None):
    """The planned network of a circuit case, its (complex64) tensors and its path."""
    circuit = _circuit(case, seed) if circuit is None else circuit
    tn = circuit_to_network(circuit).as_complex64()
    net = Network.from_tn(tn)
    stem = case["kind"] == "stem" or case.get("path") == "stem"
    path = stem_path(tn, circuit) if stem else net.greedy_path()
    net.set_path(path)
    if case["kind"] == "stem":
        # the first of the slicer's indices: a stem cut into a few large slices
        width = net.stats()["max_log2_size"]
        net.set_slices(net.find_slices(width - 2, SA_SEED)[:case["sliced"]] if case["sliced"] else [])
    elif case["target"]:
        net.set_slices(net.find_slices(case["target"], SA_SEED))
    return net, tn, path


def _many_circuits(case, seed):
    """Circuits first, first + 1, ... of the batched uneven workload (the sizes
    of ``tnc_inputs.circuits.batched_workload``; gates from the seed). With
    "small" only those of at most 2^26 complex multiply-accumulates per slice."""
    rng = np.random.default_rng(1000)
    out = []
    for i in range(256):
        nq = int(rng.integers(20, 37))
        cycles = int(rng.integers(10, 17))
        n_open = int(rng.integers(0, 7))
        k = int(rng.integers(4, 13))
        if i < case["first"]:
            continue
        r = int(math.floor(math.sqrt(nq)))
        c = int(math.ceil(nq / r))
        removed = [(r - 1, cc) for cc in range(c - (r * c - nq), c)]
        circuit = grid_rqc(r, c, cycles, int(seed) * 1000 + i, n_open=n_open, removed=removed)
        tn = circuit_to_network(circuit).as_complex64()
        net = Network.from_tn(tn)
        path = net.greedy_path()
        net.set_path(path)
        width = net.stats()["max_log2_size"]
        net.set_slices(net.find_slices(max(min(width - k, 24), n_open + 4), SA_SEED))
        if case.get("small") and _cmacs(tn, path, net.sliced, 1) > 2.0 ** 26:
            continue
        out.append((circuit, net, tn, path))
        if len(out) == case["circuits"]:
            break
    return out


def _fsim_leaves(circuit, tn):
    return [i for i, g in enumerate(tn.leaf_gate) if g >= 0 and circuit.gates[g].name == "fsim"]


def _matrices(case, seed):
    """The tensors of a pair or triple case: binary modes as separate indices,
    interleaved (A) and reversed (B) in memory where the case is permuted."""
    rng = np.random.default_rng(int(seed))
    mb, nb, kb = case["mb"], case["nb"], case["kb"]

    def rnd(bits):
        x = rng.standard_normal((2, 1 << bits), dtype=np.float32) * np.float32(math.sqrt(0.5))
        return (x[0] + 1j * x[1]).reshape((2,) * bits)
    m, k, n = list(range(mb)), list(range(mb, mb + kb)), list(range(mb + kb, mb + kb + nb))
    a, b = m + k, k + n
    if case["permuted"]:
        a = [x for pair in zip(k, m) for x in pair] + k[len(m):] + m[len(k):]
        b = n[::-1] + k
    tensors, indices = [rnd(mb + kb), rnd(kb + nb)], [tuple(a), tuple(b)]
    if case["kind"] == "pair":
        return TensorNetwork(tensors, indices, np.full(mb + nb + kb, 2, dtype=np.int64), tuple(m + n), [-1] * 2), m, n
    o = list(range(mb + kb + nb, mb + kb + nb + case["ob"]))
    tensors.append(rnd(nb + case["ob"]))
    indices.append(tuple(n + o))
    return TensorNetwork(tensors, indices, np.full(mb + kb + nb + case["ob"], 2, dtype=np.int64), tuple(m + o),
                         [-1] * 3), m, n


# ----------------------------------------------------------- prepare and run


def prepare(case, seed):
    kind, mode = case["kind"], MODES[case["mode"]]
    state = {"kind": kind, "mode": mode}
    if kind in ("pair", "triple"):
        tn = _matrices(case, seed)[0]
        net = Network.from_tn(tn)
        net.set_path([(0, 1)] if kind == "pair" else [(0, 1), (2, 3)])
        state.update(net=net, lo=0, hi=1)
    elif kind == "slices":
        net, _, _ = _plan(case, seed)
        state.update(net=net, lo=case["lo"], hi=case["hi"])
        if case["target"] >= 24:  # as the benchmark does: a workspace for the whole block
            state["ws"] = torch.empty(net.workspace_bytes(min(case["hi"] - case["lo"], 4)), dtype=torch.uint8,
                                      device="cuda")
            net.set_workspace(state["ws"])
    elif kind == "stem":
        net, _, _ = _plan(case, seed)
        state.update(net=net, lo=0, hi=net.n_slices)
    elif kind == "variants":
        circuit = _circuit(case, seed)
        net, _, _ = _plan(case, seed, circuit)
        net.set_leaf_variants(*bitstring_variants(circuit, random_bitstrings(circuit, case["count"], int(seed) + 1)))
        state.update(net=net, count=case["count"])
    elif kind == "many":
        nets = [net for _, net, _, _ in _many_circuits(case, seed)]
        state.update(nets=nets, ranges=[(0, min(net.n_slices, case["slices"])) for net in nets],
                     outs=[torch.empty(net.n_out, dtype=torch.complex128, device="cuda") for net in nets],
                     stream=torch.cuda.Stream())
    elif kind == "gradient":
        circuit = _circuit(case, seed)
        tn = circuit_to_network(circuit)
        params = [circuit.gates[i].params for i in circuit.fsim_gates()]
        state.update(amp=CircuitAmplitudes(tn, _fsim_leaves(circuit, tn), target_log2=case["target"], seed=SA_SEED,
                                           mode=mode),
                     params=torch.tensor(params, dtype=torch.float64, requires_grad=True),
                     weight=_weights(case, seed).cuda())
    else:
        circuit = _circuit(case, seed)
        net, tn, _ = _plan(case, seed, circuit)
        mask = np.zeros(tn.n_tensors, dtype=np.uint8)
        mask[_fsim_leaves(circuit, tn)] = 1
        state.update(net=net, mask=mask, grad=_weights(case, seed).cuda())
    return state


def _weights(case, seed):
    """Weights of the outputs in the loss, complex128, one per amplitude."""
    x = np.random.default_rng(int(seed) + 2).standard_normal((2, 1 << case["n_open"]))
    return torch.from_numpy(x[0] + 1j * x[1])


def run(state):
    kind, mode = state["kind"], state["mode"]
    if kind == "variants":
        return state["net"].contract_variants(0, state["count"], mode=mode)
    if kind == "many":
        with torch.cuda.stream(state["stream"]):
            return contract_many(state["nets"], state["ranges"], mode, outs=state["outs"])
    if kind == "gradient":
        amps = state["amp"](state["params"])
        loss = (torch.conj(state["weight"]) * amps).real.sum()
        (grad,) = torch.autograd.grad(loss, state["params"])
        return {"amplitudes": amps.detach(), "grad": grad}
    if kind == "environments":
        return state["net"].contract_backward(state["grad"], mode=mode, leaf_mask=state["mask"])
    return state["net"].contract(state["lo"], state["hi"], mode)


# -------------------------------------------------------------------- work


def _cmacs(tn, path, sliced, n_slices, variant_leaves=(), n_variants=1, backward=None):
    """Complex multiply-accumulates of n_slices slices: contractions without a
    sliced index (or variant leaf) below them once, the others once per slice
    and variant. ``backward``: the leaves whose environments are asked for; the
    environments of the children on the way to them are added, and the final
    contraction's value is left out."""
    cut, dims = set(sliced), tn.dims
    n = tn.n_tensors
    legs = [frozenset(ix) for ix in tn.indices]
    varies = [bool(l & cut) or v in variant_leaves for v, l in enumerate(legs)]
    needs = [backward is not None and v in backward for v in range(n)]
    total = 0.0
    for step, (i, j) in enumerate(path):
        bits = sum(math.log2(dims[e]) for e in (legs[i] | legs[j]) - cut)
        last = step == len(path) - 1
        times = n_slices * n_variants if varies[i] or varies[j] or last else 1
        if backward is None:
            total += 2.0 ** bits * times
        else:
            total += 2.0 ** bits * times * (int(needs[i]) + int(needs[j]) + (0 if last else 1))
        legs.append(legs[i] ^ legs[j])
        varies.append(varies[i] or varies[j])
        needs.append(needs[i] or needs[j])
    return total


def work(case):
    kind = case["kind"]
    if kind in ("pair", "triple"):
        m, n, k = 1 << case["mb"], 1 << case["nb"], 1 << case["kb"]
        flops, elems, out = 8.0 * m * n * k, m * k + k * n, m * n
        if kind == "triple":
            o = 1 << case["ob"]
            flops, elems, out = flops + 8.0 * m * n * o, elems + n * o, m * o
        return {"bytes": 8.0 * elems + 16.0 * out, "flops": flops}
    if kind == "many":
        flops = nbytes = 0.0
        for _, net, tn, path in _many_circuits(case, 0):
            flops += 8.0 * _cmacs(tn, path, net.sliced, min(net.n_slices, case["slices"]))
            nbytes += net.leaf_bytes() + 16.0 * net.n_out
        return {"bytes": nbytes, "flops": flops}
    circuit = _circuit(case, 0)
    net, tn, path = _plan(case, 0, circuit)
    args = (tn, path, net.sliced)
    nbytes = net.leaf_bytes() + 16.0 * net.n_out
    if kind == "variants":
        leaves, data = bitstring_variants(circuit, random_bitstrings(circuit, case["count"], 1))
        return {"bytes": nbytes + 16.0 * len(leaves) * case["count"] + 16.0 * net.n_out * case["count"],
                "flops": 8.0 * _cmacs(*args, net.n_slices, set(leaves), case["count"])}
    if kind in ("gradient", "environments"):
        back = _cmacs(*args, net.n_slices, backward=set(_fsim_leaves(circuit, tn)))
        forward = _cmacs(*args, net.n_slices) if kind == "gradient" else 0.0
        return {"bytes": nbytes + net.leaf_bytes(), "flops": 8.0 * (forward + back)}
    count = case["hi"] - case["lo"] if kind == "slices" else net.n_slices
    return {"bytes": nbytes, "flops": 8.0 * _cmacs(*args, count)}


# ------------------------------------------------------------------- exact


def _apply(state, u, qubits, n):
    """Gate matrix u (2^k x 2^k) on the listed qubits (first = most significant) of a state of n qubits."""
    if len(qubits) == 2 and qubits[0] > qubits[1]:  # ascending qubits
        u = u.reshape(2, 2, 2, 2).permute(1, 0, 3, 2).reshape(4, 4)
        qubits = qubits[::-1]
    if len(qubits) == 1:
        x = state.reshape(1 << qubits[0], 2, 1, 1, -1)
    else:
        x = state.reshape(1 << qubits[0], 2, 1 << (qubits[1] - qubits[0] - 1), 2, -1)
    if u.requires_grad or state.requires_grad:
        if len(qubits) == 1:
            return torch.einsum("ij,ajbcd->aibcd", u, x).reshape(-1)
        y = x.permute(1, 3, 0, 2, 4).reshape(4, -1)
        y = (u @ y).reshape(2, 2, x.shape[0], x.shape[2], x.shape[4])
        return y.permute(2, 0, 3, 1, 4).reshape(-1)
    out = torch.zeros_like(x)
    rows = u.cpu().tolist()
    two = len(qubits) == 2
    for i, row in enumerate(rows):
        dst = out[:, i >> 1, :, i & 1] if two else out[:, i]
        for j, w in enumerate(row):
            if w != 0:
                dst.add_(x[:, j >> 1, :, j & 1] if two else x[:, j], alpha=w)
    return out.reshape(-1)


def _amplitudes(circuit, tn, fixed, leaves=None, projections=True):
    """The open amplitudes of the network: a state-vector run over its leaves
    (``leaves`` replaces them by tensors), every index in ``fixed`` held to its
    value. With projections=False the whole final state."""
    n = circuit.n_qubits

    def leaf(i):
        if leaves is not None and i in leaves:
            return leaves[i]
        return torch.from_numpy(np.asarray(tn.tensors[i], dtype=np.complex128)).cuda()

    def hold(u, wires):  # rows of u whose new wires are held to another value vanish
        for pos, e in enumerate(wires):
            if e in fixed:
                keep = torch.zeros(2, dtype=torch.complex128, device="cuda")
                keep[fixed[e]] = 1
                one = torch.ones(2, dtype=torch.complex128, device="cuda")
                rows = keep if len(wires) == 1 else torch.kron(*((keep, one) if pos == 0 else (one, keep)))
                u = rows[:, None] * u
        return u
    eye = torch.eye(2, dtype=torch.complex128, device="cuda")
    pending = [hold(eye, tn.indices[q]) for q in range(n)]
    state = torch.ones(1, dtype=torch.complex128, device="cuda")
    for q in range(n):
        state = torch.kron(state, leaf(q))
    for g, gate in enumerate(circuit.gates):
        k = len(gate.qubits)
        wires = tn.indices[n + g][:k]
        u = leaf(n + g).reshape(1 << k, 1 << k)
        if k == 1:
            q = gate.qubits[0]
            pending[q] = hold(u @ pending[q], wires)
            continue
        a, b = gate.qubits
        state = _apply(state, hold(u @ torch.kron(pending[a], pending[b]), wires), (a, b), n)
        pending[a] = pending[b] = eye
    for q in range(n):
        if pending[q] is not eye:
            state = _apply(state, pending[q], (q,), n)
    if not projections:
        return state
    at = n + len(circuit.gates)
    for q in range(n - len(circuit.open_qubits)):  # the closed qubits come first
        v = leaf(at + q)
        x = state.reshape(2, -1)
        state = v[0] * x[0] + v[1] * x[1]
    return state


def _blocks(lo, hi):
    """[lo, hi) as aligned power-of-two blocks (start, log2 size)."""
    while lo < hi:
        b = 0
        while lo % (2 << b) == 0 and lo + (2 << b) <= hi:
            b += 1
        yield lo, b
        lo += 1 << b


def _slice_sum(circuit, net, tn, lo, hi):
    total = 0
    ids = sorted(net.sliced)
    for start, free in _blocks(lo, hi):
        total = total + _amplitudes(circuit, tn, {e: (start >> j) & 1 if j < 62 else 0
                                                  for j, e in enumerate(ids) if j >= free})
    return total


def exact(case, seed):
    with torch.no_grad():
        kind = case["kind"]
        if kind in ("pair", "triple"):
            tn, m, n = _matrices(case, seed)
            mb, nb, kb = case["mb"], case["nb"], case["kb"]
            k = list(range(mb, mb + kb))

            def matrix(i, rows, cols):
                t = torch.from_numpy(tn.tensors[i]).cuda()
                at = {e: p for p, e in enumerate(tn.indices[i])}
                order = [at[e] for e in rows + cols]
                return t.permute(order).reshape(1 << len(rows), 1 << len(cols)).to(torch.complex128)
            c = matrix(0, m, k) @ matrix(1, k, n)
            if kind == "triple":
                c = c @ matrix(2, n, list(range(mb + kb + nb, mb + kb + nb + case["ob"])))
            return c.reshape(-1)
        if kind == "many":
            return [_slice_sum(circuit, net, tn, 0, min(net.n_slices, case["slices"])) if circuit.n_qubits <= 25
                    else None for circuit, net, tn, _ in _many_circuits(case, seed)]
        circuit = _circuit(case, seed)
        if kind == "slices":
            if circuit.n_qubits * len(list(_blocks(case["lo"], case["hi"]))) > 100:
                return None
            net, tn, _ = _plan(case, seed, circuit)
            return _slice_sum(circuit, net, tn, case["lo"], case["hi"])
        if kind == "stem":
            net, tn, _ = _plan(case, seed, circuit)
            return _amplitudes(circuit, tn, {})
        if kind == "variants":
            tn = circuit_to_network(circuit).as_complex64()
            final = _amplitudes(circuit, tn, {}, projections=False)
            bits = random_bitstrings(circuit, case["count"], int(seed) + 1).astype(np.int64)
            closed = circuit.n_qubits - case["n_open"]
            rows = [sum(int(b[q]) << (closed - 1 - q) for q in range(closed)) for b in bits]
            return final.reshape(1 << closed, -1)[torch.tensor(rows, device="cuda")]
    if kind == "gradient":
        params = torch.tensor([circuit.gates[i].params for i in circuit.fsim_gates()], dtype=torch.float64,
                              requires_grad=True)
        tn = circuit_to_network(circuit).as_complex64()
        leaves = {}
        for i, (theta, phi) in zip(_fsim_leaves(circuit, tn), params):
            c, s, one, zero = torch.cos(theta) + 0j, -1j * torch.sin(theta), torch.ones(()) + 0j, torch.zeros(()) + 0j
            u = torch.stack([one, zero, zero, zero, zero, c, s, zero, zero, s, c, zero, zero, zero, zero,
                             torch.exp(-1j * phi)]).to(torch.complex128)
            rounded = torch.from_numpy(np.asarray(tn.tensors[i], dtype=np.complex128)).reshape(-1)
            leaves[i] = (u + (rounded - u).detach()).cuda()  # the library's leaves are complex64
        amps = _amplitudes(circuit, tn, {}, leaves)
        (grad,) = torch.autograd.grad((torch.conj(_weights(case, seed).cuda()) * amps).real.sum(), params)
        return {"amplitudes": amps.detach(), "grad": grad}
    tn = circuit_to_network(circuit).as_complex64()
    n_two = sum(len(g.qubits) == 2 for g in circuit.gates)
    if 16.0 * 2 ** circuit.n_qubits * 3 * n_two > 220e9:
        return None
    which = _fsim_leaves(circuit, tn)
    leaves = {i: torch.from_numpy(np.asarray(tn.tensors[i], dtype=np.complex128)).cuda().requires_grad_(True)
              for i in which}
    value = (_weights(case, seed).cuda() * _amplitudes(circuit, tn, {}, leaves)).sum().real
    grads = dict(zip(which, torch.autograd.grad(value, [leaves[i] for i in which])))
    # PyTorch's gradient of a holomorphic value's real part is the conjugate of its derivative
    return torch.cat([torch.conj(grads[i]).reshape(-1) if i in grads
                      else torch.zeros(int(t.size), dtype=torch.complex128, device="cuda")
                      for i, t in enumerate(tn.tensors)])
