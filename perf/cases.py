"""Timed workloads of the contraction-tree executor, through its public entry points.

Each case is one pass that a program using this package makes: a contraction
of a circuit or spin network (``TensorNetwork.contract``, sliced or not,
open outputs or not), many copies or many networks per call
(``contract_instances``, ``Batch``), a gradient step (``autograd``), an
open-output sample (``sampling.OpenAmplitudes``) or a single pairwise
contraction (two tensors), which is what every node of a tree is.

Results come back in the network's own type (complex64 / float32): the value
mantissa * 2**exp2 as the caller's next single-precision step takes it.
Leaf values follow from the seed alone; the structure (labels, tree, sliced
labels) follows from the case and is planned once per process, as a program
that contracts many networks of one shape keeps its tree.
"""
import functools
import math
import random

import numpy as np
import torch

from paper_2002_01935_gb300 import autograd, binding, inputs, planner, sampling


def listed():
    return [
        # the smallest call: one amplitude of a 16-qubit, 8-cycle circuit, a
        # few hundred tiny nodes; launches and latency are all of it
        {"name": "amplitude_4x4", "kind": "circuit", "rows": 4, "cols": 4, "cycles": 8, "n_open": 0,
         "mode": "fp32", "target": 0, "slice_batch": 0, "host": False},
        # bitstring sampling: the 2^6 amplitudes over six open qubits for one
        # draw of the others after another, copied to the host each time
        {"name": "sampler_5x4", "kind": "sampler", "rows": 5, "cols": 4, "cycles": 12, "n_open": 6,
         "mode": "fp16_split", "draws": 4},
        # many bitstrings of one circuit in one launch sequence
        {"name": "amplitudes_5x5", "kind": "amplitudes", "rows": 5, "cols": 5, "cycles": 10, "copies": 32,
         "mode": "fp16_split"},
        # a circuit too wide for the memory given to it: every slice of a
        # sliced tree, eight side by side, some output qubits left open
        {"name": "sliced_5x5", "kind": "circuit", "rows": 5, "cols": 5, "cycles": 12, "n_open": 4,
         "mode": "tf32_split", "target": 20, "slice_batch": 8, "host": False},
        # two slices of the 49-qubit, 14-cycle amplitude (2^28-entry tensors):
        # the largest work that one GPU is given, repeated 2^23 times in a run
        {"name": "slices_7x7", "kind": "slices", "rows": 7, "cols": 7, "cycles": 14, "target": 28,
         "trials": 16, "count": 2, "mode": "fp16_split"},
        # free energy of a 100-spin model and its derivative by every bond
        # (forward and reverse sweep, real numbers)
        {"name": "ising_100_grad", "kind": "ising_grad", "n": 100, "graph": 0, "mode": "fp32"},
        # many partition functions of uneven size as one captured batch
        {"name": "ising_batch", "kind": "ising_batch", "nets": 48, "n_lo": 40, "n_hi": 100, "graph": 7000,
         "mode": "fp16_split"},
        # a training step of a parametrised circuit: loss over 64 bitstrings,
        # gradient by all angles
        {"name": "train_5x4", "kind": "train", "rows": 5, "cols": 4, "cycles": 12, "copies": 64,
         "mode": "fp16_split"},
        # one large complex node with 2^25 outputs on the tensor cores
        {"name": "node_large", "kind": "node", "m": "2," * 12 + "2", "n": "2," * 11 + "2", "k": "2," * 9 + "2",
         "b": "", "complex": True, "mode": "fp16_split"},
        # a mid-size complex node in plain single precision
        {"name": "node_fp32", "kind": "node", "m": "2," * 10 + "2", "n": "2," * 10 + "2", "k": "2," * 9 + "2",
         "b": "", "complex": True, "mode": "fp32"},
        # labels of other sizes than powers of two: one node ...
        {"name": "node_ragged", "kind": "node", "m": "3,5,6,3,2", "n": "7,3,2,5,3", "k": "3,6,5,2", "b": "3",
         "complex": True, "mode": "fp32"},
        # ... and a whole hyperedge network of three-valued labels on a random
        # 3-regular graph, some of them left open (marginals)
        {"name": "hyper_dim3", "kind": "hyper", "n": 54, "q": 3, "graph": 12, "n_open": 4, "mode": "fp32"},
    ]


MODES = ("fp32", "fp16_split", "tf32_split", "bf16_split", "tf32_3m")
GRIDS = ((3, 3), (4, 3), (4, 4), (5, 4), (5, 5))


def draw(rng: random.Random):
    kind = rng.choice(("circuit", "circuit", "node", "node", "node", "ragged", "hyper", "ising_grad", "ising_batch",
                       "train", "amplitudes", "sampler"))
    mode = rng.choice(MODES)
    rows, cols = rng.choice(GRIDS)
    if kind == "circuit":
        return {"kind": kind, "rows": rows, "cols": cols, "cycles": rng.randint(8, 11), "n_open": rng.randint(3, 6),
                "mode": mode, "target": rng.choice((0, 0, {9: 0, 12: 8, 16: 9, 20: 12, 25: 16}[rows * cols])),
                "slice_batch": rng.choice((0, 1, 4, 8)),
                "host": rng.random() < 0.3}
    if kind == "sampler":
        return {"kind": kind, "rows": rows, "cols": cols, "cycles": rng.randint(8, 10), "n_open": rng.randint(4, 7),
                "mode": mode, "draws": rng.randint(1, 6)}
    if kind == "amplitudes":
        return {"kind": kind, "rows": rows, "cols": cols, "cycles": rng.randint(8, 10), "copies": _log(rng, 9, 100),
                "mode": mode}
    if kind == "train":
        rows, cols = rng.choice(GRIDS[:4])
        return {"kind": kind, "rows": rows, "cols": cols, "cycles": rng.randint(8, 11), "copies": _log(rng, 9, 80),
                "mode": mode}
    if kind == "ising_grad":
        return {"kind": kind, "n": 2 * rng.randint(20, 50), "graph": rng.randint(0, 99), "mode": mode}
    if kind == "ising_batch":
        lo = 2 * rng.randint(20, 35)
        return {"kind": kind, "nets": _log(rng, 8, 100), "n_lo": lo, "n_hi": lo + 2 * rng.randint(2, 14),
                "graph": rng.randint(0, 9999), "mode": mode}
    if kind == "hyper":
        q = rng.choice((3, 3, 3, 4, 5))
        return {"kind": kind, "n": 2 * rng.randint(8, {3: 28, 4: 20, 5: 15}[q]), "q": q, "graph": rng.randint(0, 99),
                "n_open": rng.randint(2, 5), "mode": "fp32"}
    if kind == "ragged":
        group = lambda hi: ",".join(str(rng.choice((2, 3, 3, 5, 6, 7))) for _ in range(rng.randint(1, hi)))  # noqa: E731
        return {"kind": "node", "m": group(5), "n": group(5), "k": group(4), "b": rng.choice(("", "", "3", "5")),
                "complex": rng.random() < 0.6, "mode": rng.choice(("fp32", "fp16_split"))}
    # power-of-two node: 2^20 to 2^34 multiply-adds, squarish, narrow, outer
    # or inner; labels of size 2, 4 and 8 mixed
    work = rng.uniform(20, 34 if mode != "fp32" else 32)
    shape = [rng.uniform(0.4, 1.6) for _ in range(3)]
    m, n, k = (max(1, min(13, round(work * s / sum(shape)))) for s in shape)
    return {"kind": "node", "m": _bits(rng, m), "n": _bits(rng, n), "k": _bits(rng, k),
            "b": _bits(rng, rng.choice((0, 0, 1, 2))), "complex": rng.random() < 0.6, "mode": mode}


def _log(rng, lo, hi):
    return round(math.exp(rng.uniform(math.log(lo), math.log(hi))))


def _bits(rng, bits):
    """Sizes 2, 4, 8 whose product is 2^bits, as text."""
    out = []
    while bits > 0:
        j = min(bits, rng.choice((1, 1, 1, 2, 3)))
        out.append(str(2 ** j))
        bits -= j
    return ",".join(out)


# --------------------------------------------------------------------------
# structures (labels, trees), planned once per process
# --------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _circuit_plan(rows, cols, cycles, n_open, target, trials):
    """Labels and tree of a circuit network: they depend on the grid, the
    cycles and the open qubits, not on the gates."""
    net = inputs.circuit_network(inputs.random_circuit(rows, cols, cycles, seed=0), [0] * (rows * cols),
                                 open_qubits=range(rows * cols - n_open, rows * cols))
    if trials:
        pairs, sliced, info = planner.hyper_greedy(net.labels, net.dims, net.open, trials=trials, seed=0,
                                                   target_width=float(target) if target else None)
    else:
        pairs, sliced, info = planner.plan(net)
    return net, pairs, sliced, info


@functools.lru_cache(maxsize=None)
def _ising_plan(n, graph):
    edges = inputs.random_regular_graph(n, 3, graph)
    net = inputs.ising_network(n, edges, [1.0] * len(edges), 0.3)
    pairs, _, info = planner.plan(net)
    return edges, net, pairs, info


@functools.lru_cache(maxsize=None)
def _batch_sizes(nets, n_lo, n_hi, graph):
    """Spin counts and graphs of the networks of a batch: those whose greedy
    tree stays within 2^20 entries."""
    rng = np.random.default_rng(graph)
    got, j = [], 0
    while len(got) < nets:
        n = int(rng.choice(np.arange(n_lo, n_hi + 1, 2)))
        if _ising_plan(n, graph + j)[3].W <= 20:
            got.append((n, graph + j))
        j += 1
    return tuple(got)


@functools.lru_cache(maxsize=None)
def _hyper_plan(n, q, graph, n_open):
    """One label of size q per vertex of a random 3-regular graph, shared by
    the matrices of its edges; the first labels are open."""
    edges = inputs.random_regular_graph(n, 3, graph)
    labels = [[int(u), int(v)] for u, v in edges]
    net = inputs.Network([np.zeros((q, q))] * len(edges), labels, {v: q for v in range(n)}, list(range(n_open)))
    pairs, _, info = planner.plan(net)
    return net, pairs, info


def _node_labels(case):
    dims = {g: [int(x) for x in case[g].split(",") if x] for g in "mnkb"}
    ids, nxt = {}, 0
    for g in "mnkb":
        ids[g] = list(range(nxt, nxt + len(dims[g])))
        nxt += len(dims[g])
    size = dict(zip(range(nxt), dims["m"] + dims["n"] + dims["k"] + dims["b"]))
    m, n, k, b = (ids[g] for g in "mnkb")
    # summed labels interleaved with kept ones, as between nodes of a tree
    return b + k[::2] + m + k[1::2], n[:2] + k + b + n[2:], b + m + n, size


def _circuit(case, seed):
    """Gates, angles and bitstrings of this seed."""
    return inputs.random_circuit(case["rows"], case["cols"], case["cycles"], seed=seed)


def _to(tensors, dtype, host=False):
    ts = [torch.from_numpy(np.array(t, order="C")).to(dtype) for t in tensors]
    return [t.pin_memory() for t in ts] if host else [t.cuda() for t in ts]


def _couplings(case, n, seed):
    return inputs.ising_couplings(n, seed)


def _edge_matrices(J):
    """exp(0.3 J s s') as [edges, 2, 2]."""
    s = np.array([1.0, -1.0])
    return np.exp(0.3 * J[:, None, None] * np.outer(s, s))


# --------------------------------------------------------------------------
# what the program holds before the call
# --------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "node":
        la, lb, lo, size = _node_labels(case)
        g = torch.Generator(device="cuda").manual_seed(seed)
        dt = torch.complex64 if case["complex"] else torch.float32
        ts = [torch.randn([size[l] for l in ls], dtype=dt, device="cuda", generator=g) for ls in (la, lb)]
        return {"case": case, "tnw": binding.TensorNetwork([la, lb], size, lo, ts, complex_=case["complex"]),
                "pairs": [(0, 1)], "sliced": [], "leaves": ts}
    if kind in ("circuit", "slices"):
        net, pairs, sliced, _ = _circuit_plan(case["rows"], case["cols"], case["cycles"], case.get("n_open", 0),
                                              case["target"], case.get("trials", 16))
        nq = case["rows"] * case["cols"]
        no = case.get("n_open", 0)
        bits = inputs.random_bitstrings(nq, 1, seed)[0]
        mine = inputs.circuit_network(_circuit(case, seed), bits, open_qubits=range(nq - no, nq))
        ts = _to(mine.tensors, torch.complex64, case.get("host", False))
        return {"case": case, "tnw": binding.TensorNetwork(net.labels, net.dims, net.open, ts), "pairs": pairs,
                "sliced": sliced, "leaves": ts}
    if kind == "sampler":
        nq, no = case["rows"] * case["cols"], case["n_open"]
        _, pairs, _, _ = _circuit_plan(case["rows"], case["cols"], case["cycles"], no, 0, 0)
        amps = sampling.OpenAmplitudes(_circuit(case, seed), range(nq - no, nq), mode=case["mode"], pairs=pairs)
        return {"case": case, "amps": amps,
                "x": [list(map(int, b)) for b in inputs.random_bitstrings(nq - no, case["draws"], seed)]}
    if kind == "amplitudes":
        net, pairs, _, _ = _circuit_plan(case["rows"], case["cols"], case["cycles"], 0, 0, 16)
        nq, c = case["rows"] * case["cols"], case["copies"]
        mine = inputs.circuit_network(_circuit(case, seed), [0] * nq)
        bits = torch.from_numpy(inputs.random_bitstrings(nq, c, seed).astype(np.int64)).cuda()
        outs = torch.eye(2, dtype=torch.complex64, device="cuda")[bits]  # [copies, qubits, 2]
        ts = _to(mine.tensors[:-nq], torch.complex64) + [outs[:, q].contiguous() for q in range(nq)]
        return {"case": case, "tnw": binding.TensorNetwork(net.labels, net.dims, net.open, ts), "pairs": pairs,
                "strides": [0] * (net.n_tensors - nq) + [2] * nq, "leaves": ts}
    if kind == "train":
        net, pairs, _, _ = _circuit_plan(case["rows"], case["cols"], case["cycles"], 0, 0, 0)
        nq, c = case["rows"] * case["cols"], case["copies"]
        circ = _circuit(case, seed)
        mine = inputs.circuit_network(circ, [0] * nq)
        base = _to(mine.tensors, torch.complex64)
        bits = torch.from_numpy(inputs.random_bitstrings(nq, c, seed).astype(np.int64)).cuda()
        outs = torch.eye(2, dtype=torch.complex64, device="cuda")[bits]
        fs = circ.fsim_gates()
        angles = np.array([circ.gates[g].params for g in fs], dtype=np.float32)
        tnw = binding.TensorNetwork(net.labels, net.dims, net.open, base)
        return {"case": case, "tnw": tnw, "pairs": pairs, "base": base,
                "leaf_of": [mine.meta["gate_leaf"][g] for g in fs],
                "batch": {net.n_tensors - nq + q: outs[:, q].contiguous() for q in range(nq)},
                "angles": torch.from_numpy(angles).cuda()}
    if kind == "ising_grad":
        edges, net, pairs, _ = _ising_plan(case["n"], case["graph"])
        ts = _to(net.tensors, torch.float32)
        bonds = torch.from_numpy(_edge_matrices(_couplings(case, len(edges), seed))).float().cuda()
        return {"case": case, "tnw": binding.TensorNetwork(net.labels, net.dims, net.open, ts, complex_=False),
                "pairs": pairs, "copies": ts[:case["n"]], "bonds": bonds}
    if kind == "ising_batch":
        nets, trees, keep, sizes = [], [], [], []
        for j, (n, graph) in enumerate(_batch_sizes(case["nets"], case["n_lo"], case["n_hi"], case["graph"])):
            edges, net, pairs, _ = _ising_plan(n, graph)
            bonds = torch.from_numpy(_edge_matrices(_couplings(case, len(edges), seed + j))).float().cuda()
            ts = _to(net.tensors[:n], torch.float32) + list(bonds.unbind(0))
            nets.append(binding.TensorNetwork(net.labels, net.dims, net.open, ts, complex_=False))
            trees.append(pairs)
            keep.append(ts)
            sizes.append(n)
        return {"case": case, "batch": binding.Batch(nets, trees, mode=case["mode"]), "leaves": keep,
                "bits": torch.tensor(sizes, dtype=torch.int64, device="cuda")}
    if kind == "hyper":
        net, pairs, _ = _hyper_plan(case["n"], case["q"], case["graph"], case["n_open"])
        g = torch.Generator(device="cuda").manual_seed(seed)
        # Boltzmann factors of random pair couplings, of mean one per entry
        w = torch.exp(0.3 * torch.randn(len(net.labels), case["q"], case["q"], device="cuda", generator=g)) / case["q"]
        ts = list(w.unbind(0))
        return {"case": case, "tnw": binding.TensorNetwork(net.labels, net.dims, net.open, ts, complex_=False),
                "pairs": pairs, "sliced": [], "leaves": ts}
    raise ValueError(kind)


def _value(m, e, dtype):
    """mantissa * 2**exp2 in the network's own type."""
    return torch.ldexp(m, e).to(dtype)


def _fsim(angles):
    """fSim(theta, phi) leaves [n, 2, 2, 2, 2] from angles [n, 2]."""
    th, ph = angles.double().unbind(1)
    z, one = torch.zeros_like(th), torch.ones_like(th)
    re = torch.stack([one, z, z, z, z, th.cos(), z, z, z, z, th.cos(), z, z, z, z, ph.cos()], 1)
    im = torch.stack([z, z, z, z, z, z, -th.sin(), z, z, -th.sin(), z, z, z, z, z, -ph.sin()], 1)
    return torch.complex(re, im).view(-1, 2, 2, 2, 2)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "node":
        m, e = state["tnw"].contract(state["pairs"], [], case["mode"])
        return [m.to(torch.complex64 if case["complex"] else torch.float32), e]
    if kind in ("circuit", "slices", "hyper"):
        out = ex = None
        if case.get("host"):  # leaves and result in host memory
            out = torch.empty(state["tnw"].out_shape, dtype=torch.complex128)
            ex = torch.empty((), dtype=torch.int64)
        m, e = state["tnw"].contract(state["pairs"], state["sliced"], case["mode"], out=out, out_exp=ex,
                                     slice_count=case.get("count", 0), slice_batch=case.get("slice_batch", 0))
        return _value(m, e, torch.float32 if kind == "hyper" else torch.complex64)
    if kind == "sampler":
        return [state["amps"](x).astype(np.complex64) for x in state["x"]]
    if kind == "amplitudes":
        m, e = state["tnw"].contract_instances(state["pairs"], case["mode"], case["copies"], state["strides"])
        return _value(torch.view_as_complex(m), e, torch.complex64)
    if kind == "train":
        angles = state["angles"].detach().requires_grad_(True)
        gates = _fsim(angles).to(torch.complex64).unbind(0)
        leaves = list(state["base"])
        for v, t in zip(state["leaf_of"], gates):
            leaves[v] = t
        for v in state["batch"]:
            leaves[v] = None
        amp = autograd.contract_batch(state["tnw"], state["pairs"], case["mode"], leaves, state["batch"])
        loss = amp.abs().square().log().mean()
        loss.backward()
        return [amp.detach().to(torch.complex64), angles.grad]
    if kind == "ising_grad":
        bonds = state["bonds"].detach().requires_grad_(True)
        z = autograd.contract(state["tnw"], state["pairs"], [], case["mode"], *state["copies"], *bonds.unbind(0))
        free = z.log()
        free.backward()
        return [free.detach().float(), bonds.grad]
    if kind == "ising_batch":
        m, e, _ = state["batch"].contract()
        return _value(m[:, 0], e - state["bits"], torch.float32)  # Z / 2^N
    raise ValueError(kind)


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def work(case):
    kind = case["kind"]
    numel = lambda net: sum(math.prod(net.dims[l] for l in ls) for ls in net.labels)  # noqa: E731
    if kind == "node":
        la, lb, lo, size = _node_labels(case)
        vol = lambda ls: math.prod(size[l] for l in ls)  # noqa: E731
        c = case["complex"]
        return {"bytes": (8 if c else 4) * (vol(la) + vol(lb) + vol(lo)), "flops": (8.0 if c else 2.0) * vol(size)}
    if kind in ("circuit", "slices"):
        net, _, _, info = _circuit_plan(case["rows"], case["cols"], case["cycles"], case.get("n_open", 0),
                                        case["target"], case.get("trials", 16))
        slices = case.get("count") or info.d_sliced
        return {"bytes": 8 * (numel(net) + 2 ** case.get("n_open", 0)), "flops": 8.0 * info.C * slices}
    if kind == "sampler":
        net, _, _, info = _circuit_plan(case["rows"], case["cols"], case["cycles"], case["n_open"], 0, 0)
        return {"bytes": 8 * case["draws"] * (numel(net) + 2 ** case["n_open"]), "flops": 8.0 * info.C * case["draws"]}
    if kind == "amplitudes":
        net, _, _, info = _circuit_plan(case["rows"], case["cols"], case["cycles"], 0, 0, 16)
        return {"bytes": 8 * (numel(net) + case["copies"] * (1 + 2 * case["rows"] * case["cols"])),
                "flops": 8.0 * info.C * case["copies"]}
    if kind == "train":  # forward and two contractions per node back
        net, _, _, info = _circuit_plan(case["rows"], case["cols"], case["cycles"], 0, 0, 0)
        return {"bytes": 8 * (2 * numel(net) + case["copies"] * (1 + 2 * case["rows"] * case["cols"])),
                "flops": 24.0 * info.C * case["copies"]}
    if kind == "ising_grad":
        _, net, _, info = _ising_plan(case["n"], case["graph"])
        return {"bytes": 4 * (numel(net) + 6 * case["n"]), "flops": 6.0 * info.C}
    if kind == "ising_batch":
        plans = [_ising_plan(*p) for p in _batch_sizes(case["nets"], case["n_lo"], case["n_hi"], case["graph"])]
        return {"bytes": 4 * sum(numel(p[1]) + 1 for p in plans), "flops": sum(2.0 * p[3].C for p in plans)}
    if kind == "hyper":
        net, _, info = _hyper_plan(case["n"], case["q"], case["graph"], case["n_open"])
        return {"bytes": 4 * (numel(net) + case["q"] ** case["n_open"]), "flops": 2.0 * info.C}
    raise ValueError(kind)


# --------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# --------------------------------------------------------------------------

def _tree_sum(leaves, labels, pairs, open_labels):
    """Pairwise einsum in 64 bits along a tree (any order gives the same sum)."""
    left = {}
    for ls in labels:
        for l in ls:
            left[l] = left.get(l, 0) + 1
    for l in open_labels:
        left[l] += 1
    live = {v: (t, list(ls)) for v, (t, ls) in enumerate(zip(leaves, labels))}
    for i, (a, b) in enumerate(pairs):
        (ta, la), (tb, lb) = live.pop(a), live.pop(b)
        for l in la + lb:
            left[l] -= 1
        out = [l for l in dict.fromkeys(la + lb) if left[l] > 0]
        for l in out:
            left[l] += 1
        at = {l: j for j, l in enumerate(dict.fromkeys(la + lb))}
        live[len(labels) + i] = (torch.einsum(ta, [at[l] for l in la], tb, [at[l] for l in lb],
                                              [at[l] for l in out]), out)
    t, ls = live.popitem()[1]
    return t.permute([ls.index(l) for l in open_labels])


def _apply(psi, gate, qubits, nq):
    """gate [out..., in...] on the axes `qubits` of the state [2] * nq."""
    w = len(qubits)
    psi = torch.tensordot(gate, psi.reshape([2] * nq), dims=(list(range(w, 2 * w)), list(qubits)))
    return torch.movedim(psi, list(range(w)), list(qubits))


def _state(circ, gates):
    """Final state vector: gates[i] is gate i's matrix as a complex128 tensor."""
    nq = circ.n_qubits
    psi = torch.zeros(2 ** nq, dtype=torch.complex128, device="cuda")
    psi[0] = 1.0
    for g, m in zip(circ.gates, gates):
        psi = _apply(psi, m.reshape([2] * (2 * len(g.qubits))), g.qubits, nq)
    return psi.reshape([2] * nq)


def _stored(circ):
    """The gate matrices as stored in the leaves (complex64), widened."""
    return [torch.from_numpy(np.asarray(g.matrix).astype(np.complex64).astype(np.complex128)).cuda()
            for g in circ.gates]


def exact(case, seed):
    kind = case["kind"]
    if kind == "slices":
        return None  # minutes in 64 bits
    if kind == "node":
        la, lb, lo, size = _node_labels(case)
        vol = math.prod(size.values())
        if vol > 2 ** 36:
            return None
        ta, tb = (t.to(torch.complex128 if case["complex"] else torch.float64)
                  for t in prepare(case, seed)["leaves"])
        # mantissa and exponent: every operand is scaled by the frexp exponent
        # of its largest component
        e = 0
        for t in (ta, tb):
            big = float(torch.view_as_real(t).abs().max() if case["complex"] else t.abs().max())
            e += math.frexp(big)[1]
        group = lambda t, ls, order: t.permute([ls.index(l) for g in order for l in g]).reshape(  # noqa: E731
            [math.prod(size[l] for l in g) for g in order])
        ids = lambda g: [l for l in lo if l in g]  # noqa: E731
        b = ids(set(la) & set(lb))
        m, n = [l for l in lo if l in la and l not in b], [l for l in lo if l in lb and l not in b]
        k = [l for l in la if l not in lo]
        c = torch.bmm(group(ta, la, (b, m, k)), group(tb, lb, (b, k, n)))
        return [(c * 2.0 ** -e).reshape([size[l] for l in lo]), None]
    if kind in ("circuit", "sampler", "amplitudes"):
        nq = case["rows"] * case["cols"]
        circ = _circuit(case, seed)
        psi = _state(circ, _stored(circ))
        if kind == "sampler":
            return [psi[tuple(int(x) for x in b)].cpu().numpy()
                    for b in inputs.random_bitstrings(nq - case["n_open"], case["draws"], seed)]
        if kind == "amplitudes":
            bits = torch.from_numpy(inputs.random_bitstrings(nq, case["copies"], seed).astype(np.int64)).cuda()
            return psi[tuple(bits.unbind(1))]
        bits = inputs.random_bitstrings(nq, 1, seed)[0]
        v = psi[tuple(int(x) for x in bits[:nq - case["n_open"]])]
        return v.cpu() if case["host"] else v
    if kind == "train":
        nq = case["rows"] * case["cols"]
        circ = _circuit(case, seed)
        fs = circ.fsim_gates()
        angles = torch.tensor(np.array([circ.gates[g].params for g in fs], dtype=np.float32).astype(np.float64),
                              device="cuda", requires_grad=True)
        gates = _stored(circ)
        for g, m in zip(fs, _fsim(angles).unbind(0)):
            gates[g] = m
        bits = torch.from_numpy(inputs.random_bitstrings(nq, case["copies"], seed).astype(np.int64)).cuda()
        amp = _state(circ, gates)[tuple(bits.unbind(1))]
        amp.abs().square().log().mean().backward()
        return [amp.detach(), angles.grad]
    if kind == "ising_grad":
        edges, net, pairs, _ = _ising_plan(case["n"], case["graph"])
        bonds = torch.from_numpy(_edge_matrices(_couplings(case, len(edges), seed))).float().double().cuda()
        bonds.requires_grad_(True)
        free = _tree_sum(_to(net.tensors[:case["n"]], torch.float64) + list(bonds.unbind(0)), net.labels, pairs,
                         []).log()
        free.backward()
        return [free.detach(), bonds.grad]
    if kind == "ising_batch":
        z = []
        for j, (n, graph) in enumerate(_batch_sizes(case["nets"], case["n_lo"], case["n_hi"], case["graph"])):
            edges, net, pairs, _ = _ising_plan(n, graph)
            bonds = torch.from_numpy(_edge_matrices(_couplings(case, len(edges), seed + j))).float().double().cuda()
            z.append(_tree_sum(_to(net.tensors[:n], torch.float64) + list(bonds.unbind(0)), net.labels, pairs, [])
                     * 2.0 ** -n)
        return torch.stack(z)
    if kind == "hyper":
        net, pairs, _ = _hyper_plan(case["n"], case["q"], case["graph"], case["n_open"])
        return _tree_sum([t.double() for t in prepare(case, seed)["leaves"]], net.labels, pairs, net.open)
    raise ValueError(kind)
