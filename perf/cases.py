"""Workloads that stand for what a program has this engine do, each as one call of its public API.

A case is a dict of plain values; ``prepare`` builds what a program holds before the call (the
network on the device, the plan, an amplitude buffer to read), ``run`` makes the call, ``exact``
gives the same outputs from torch in 64 bits without this package's kernels, and ``work`` counts
what one call cannot do without.

Kinds of case:

* ``circuit``: amplitudes of a seeded Sycamore-shaped random circuit on its last ``open`` qubits
  (the other qubits closed on seeded bits) along a greedy or an annealed path, all slices.
  ``open_sliced`` of the open qubits enumerate amplitude batches;
* ``slices``: a range of slices of one of the stored paths (45 or 53 qubits), which is how a run
  over millions of slices is cut into calls;
* ``sparse``: amplitudes of a list of sampled bitstrings, every qubit open;
* ``step``: one pairwise contraction of two large tensors with shuffled label orders;
* ``readout``: the FP64 readout (sum p, sum p^2, linear XEB) of a vector of amplitudes.

Amplitudes are returned as complex64: the engine's arithmetic and storage between steps are
32 bits or less, the complex128 accumulator only keeps the sum over slices from adding to that,
and a program that goes on to sample or to store them keeps them in complex64.
"""
import functools
import json
import math
import os

import numpy as np
import torch

import paper_2310_03978_gb300
from paper_2310_03978_gb300 import tn
from paper_2310_03978_gb300 import workload as W
from paper_2310_03978_gb300.slice_support import supported_slices

PATHS = os.path.join(os.path.dirname(os.path.abspath(paper_2310_03978_gb300.__file__)), "paths")
# stored path: (rows, cols, cycles, removed sites, open qubits)
STORED = {
    "sycamore45_5x9_c14_open12": (5, 9, 14, (), 12),
    "sycamore53_6x9_c16_open12": (6, 9, 16, ((5, 8),), 12),
}
MODES = ("c64", "tf32", "split_tf32", "fp16_scaled", "bf16_scaled", "split_bf16", "split_fp16",
         "mixed")
# At theta = pi/2 fSim is a swap up to phases and nearly all slices of a closed circuit are exactly
# zero; a program that runs a range of slices meets both kinds.  Away from that angle many more
# contribute, so that a range has values that can be compared.
SLICE_THETA = 1.2


def _circuit(name, rows, cols, cycles, open_, mode, **more):
    c = {"kind": "circuit", "name": name, "rows": rows, "cols": cols, "cycles": cycles,
         "open": open_, "open_sliced": 0, "sliced": 0, "trials": 0, "anneal_cap": 0,
         "mode": mode, "eps_budget": 0.0, "host": False}
    c.update(more)
    return c


def listed():
    return [
        # the smallest: one batch of 64 amplitudes of a 12-qubit circuit, 147 steps of a few
        # elements each; a program that scans many small circuits pays this latency every time
        _circuit("circuit12", 3, 4, 8, 6, "c64"),
        # the same size with every qubit open, 64 batches of 64 amplitudes in one call, into a
        # host array
        _circuit("batches12", 3, 4, 8, 12, "c64", open_sliced=6, host=True),
        # a 20-qubit circuit in complex64: the ordinary validation run
        _circuit("circuit20", 4, 5, 14, 10, "c64"),
        # the whole state of 20 qubits in complex64: dense GEMMs on the CUDA cores
        _circuit("state20", 4, 5, 12, 20, "c64"),
        # 25 qubits, BF16 storage under its default error budget, two sliced bonds
        _circuit("circuit25_bf16", 5, 5, 12, 10, "bf16_scaled", sliced=2),
        # 30 qubits, 14 cycles, 16 slices on a greedy path: the benchmark's configuration
        _circuit("circuit30", 5, 6, 14, 10, "fp16_scaled", sliced=4, trials=20),
        # the same amplitudes along an annealed path under a 1e-3 error budget
        _circuit("circuit30_annealed", 5, 6, 14, 10, "fp16_scaled", anneal_cap=28,
                 eps_budget=1e-3),
        # 8 of the 2^13 slices of the 45-qubit 14-cycle path (the precision study's circuit)
        {"kind": "slices", "name": "slices45", "path": "sycamore45_5x9_c14_open12",
         "mode": "tf32", "count": 8, "flight": 8},
        # 2 of the 2^24 slices of the 53-qubit 16-cycle path
        {"kind": "slices", "name": "slices53", "path": "sycamore53_6x9_c16_open12",
         "mode": "fp16_scaled", "count": 2, "flight": 2},
        # 4096 sampled bitstrings of a 24-qubit 12-cycle circuit
        {"kind": "sparse", "name": "sparse24", "rows": 4, "cols": 6, "cycles": 12,
         "samples": 4096, "mode": "fp16_scaled"},
        # one dense pairwise contraction, m = n = 2^12, k = 2^11, compensated BF16
        {"kind": "step", "name": "step_dense", "lm": 12, "ln": 12, "lk": 11,
         "mode": "split_bf16"},
        # readout of 2^24 amplitudes gathered from all ranks
        {"kind": "readout", "name": "readout24", "count": 1 << 24, "qubits": 53, "plan": True},
    ]


# ------------------------------------------------------------------------------ paths (no data)
@functools.lru_cache(maxsize=None)
def _structure(rows, cols, cycles, open_, removed=()):
    """Labels and open labels of a circuit's network: they do not depend on the gates drawn."""
    circ = W.random_circuit(rows, cols, cycles, 1, removed)
    n = circ.n_qubits
    net = W.build_network(circ, range(n - open_, n), {q: 0 for q in range(n - open_)})
    return tuple(net.labels), tuple(net.open_labels)


@functools.lru_cache(maxsize=None)
def _circuit_path(rows, cols, cycles, open_, open_sliced, sliced, trials, anneal_cap):
    """(path, sliced labels) of a circuit case."""
    labels, opens = _structure(rows, cols, cycles, open_)
    if trials:
        path = W.best_random_greedy(labels, opens, (W.BASE_SEED + 1) ^ 0xFA7, trials, 0.05)
    else:
        path = W.greedy_path(labels, opens)
    if anneal_cap:
        path, cut, _ = tn.path_optimize(
            labels, opens, path, seed=7, sweeps=400, sweeps_per_slice=40, sweeps_final=200,
            t_start=0.03, t_end=0.001, max_log2_size=anneal_cap, chains=8, alpha=512.0,
            greedy_trials=10)
        return tuple(path), tuple(cut)
    cut = list(opens[:open_sliced])
    cut += W.greedy_slices(labels, opens, path, sliced) if sliced else []
    return tuple(path), tuple(cut)


@functools.lru_cache(maxsize=None)
def _stored_path(name):
    with open(os.path.join(PATHS, name + ".json")) as f:
        d = json.load(f)
    return tuple(tuple(p) for p in d["path"]), tuple(d["sliced"])


@functools.lru_cache(maxsize=None)
def _sparse_path(rows, cols, cycles):
    labels, opens = _structure(rows, cols, cycles, rows * cols)
    path = W.greedy_path(labels, opens)
    path, _, _ = tn.path_optimize(labels, opens, path, seed=7, sweeps=300, sweeps_final=0,
                                  t_start=0.03, t_end=0.001, chains=8)
    return tuple(path)


def _circuit_args(case):
    return (case["rows"], case["cols"], case["cycles"], case["open"], case["open_sliced"],
            case["sliced"], case["trials"], case["anneal_cap"])


@functools.lru_cache(maxsize=None)
def _cost(labels, opens, path, sliced):
    """(largest intermediate in log2 elements, T_cc of one slice in flops)."""
    ml, tcc, _ = W.path_cost(labels, opens, path, sliced)
    return ml, float(tcc)


def _circuit_cost(case):
    labels, opens = _structure(*_circuit_args(case)[:4])
    path, cut = _circuit_path(*_circuit_args(case))
    ml, tcc = _cost(labels, opens, path, cut)
    return ml, tcc * 2.0 ** len(cut)


# ------------------------------------------------------------------------------ drawn cases
# What the largest listed cases take: flops in the tensor-core modes (the 30-qubit greedy path)
# and on the CUDA cores, and the largest intermediate.
MOST_FLOPS, MOST_FLOPS_C64, MOST_LOG2 = 2.0 ** 47, 2.0 ** 42, 28


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_circuit(rng):
    while True:
        rows, cols = rng.randint(1, 5), rng.randint(2, 7)
        n = rows * cols
        if not 5 <= n <= 30:
            continue
        cycles, open_ = rng.randint(3, 16), rng.randint(1, min(n, 20))
        mode = rng.choice(MODES)
        host = rng.random() < 0.25
        if n > 20:  # annealed, as large circuits are run
            case = _circuit("", rows, cols, cycles, min(open_, 12), mode,
                            anneal_cap=rng.randint(22, MOST_LOG2), host=host)
        else:
            batches = rng.randint(0, min(6, open_ - 1)) if rng.random() < 0.4 else 0
            case = _circuit("", rows, cols, cycles, open_, mode, open_sliced=batches,
                            sliced=0 if batches else rng.randint(0, 4), host=host)
        if mode in ("fp16_scaled", "tf32") and rng.random() < 0.5:
            case["eps_budget"] = rng.choice((5e-4, 1e-3, 5e-3))
        ml, flops = _circuit_cost(case)
        if ml <= MOST_LOG2 and flops <= (MOST_FLOPS_C64 if mode == "c64" else MOST_FLOPS / 8):
            del case["name"]
            return case


def draw(rng):
    kind = rng.choice(("circuit", "circuit", "circuit", "slices", "sparse", "step", "readout"))
    if kind == "circuit":
        return _draw_circuit(rng)
    if kind == "slices":
        if rng.random() < 0.3:
            return {"kind": "slices", "path": "sycamore53_6x9_c16_open12",
                    "mode": rng.choice(("fp16_scaled", "mixed")), "count": 1, "flight": 1}
        flight = rng.randint(1, 8)
        return {"kind": "slices", "path": "sycamore45_5x9_c14_open12", "mode": rng.choice(MODES),
                "count": rng.randint(1, 12), "flight": flight}
    if kind == "sparse":
        while True:
            rows, cols = rng.randint(2, 4), rng.randint(3, 6)
            cycles = rng.randint(4, 12)
            case = {"kind": "sparse", "rows": rows, "cols": cols, "cycles": cycles,
                    "samples": _log_uniform(rng, 1, 4096),
                    "mode": rng.choice(("c64", "fp16_scaled", "split_bf16"))}
            labels, opens = _structure(rows, cols, cycles, rows * cols)
            if _cost(labels, opens, _sparse_path(rows, cols, cycles), ())[1] <= 2.0 ** 40:
                return case
    if kind == "step":
        while True:
            lm, ln, lk = rng.randint(0, 20), rng.randint(0, 14), rng.randint(1, 13)
            mode = rng.choice(MODES)
            if (lm + lk <= 23 and ln + lk <= 23 and lm + ln <= 24
                    and (mode != "c64" or lm + ln + lk <= 35)):
                return {"kind": "step", "lm": lm, "ln": ln, "lk": lk, "mode": mode}
    log2 = rng.uniform(0, 27)
    if rng.random() < 0.5:
        return {"kind": "readout", "count": 1 << min(25, int(log2)),
                "qubits": rng.randint(28, 53), "plan": True}
    return {"kind": "readout", "count": int(2.0 ** log2), "qubits": rng.randint(28, 53),
            "plan": False}


# ------------------------------------------------------------------------------ inputs
def _network(rows, cols, cycles, open_, seed, removed=(), theta=W.FSIM_THETA):
    circ = W.random_circuit(rows, cols, cycles, seed, removed, theta=theta)
    n = circ.n_qubits
    rng = W.Xoshiro256ss(seed ^ 0x5EED)
    closed = {q: rng.below(2) for q in range(n - open_)}
    return circ, W.build_network(circ, list(range(n - open_, n)), closed)


def _samples(case, seed):
    n = case["rows"] * case["cols"]
    return np.random.default_rng(seed).integers(0, 2, (case["samples"], n), dtype=np.uint8)


def _step_operands(case, seed):
    """Complex normal operands at an amplitude-like scale, with shuffled label orders."""
    lm, ln, lk = case["lm"], case["ln"], case["lk"]
    rng = np.random.default_rng(seed)
    M, N, K = list(range(lm)), list(range(100, 100 + ln)), list(range(200, 200 + lk))
    la = [int(x) for x in rng.permutation(M + K)]
    lb = [int(x) for x in rng.permutation(N + K)]
    out = [int(x) for x in rng.permutation(M + N)]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    scale = 2.0 ** (-(lm + ln + 2 * lk) / 4)
    A, B = (scale * torch.randn(1 << len(ls), dtype=torch.complex128, device="cuda",
                                generator=gen) for ls in (la, lb))
    return A, B, la, lb, out


def _readout_amps(case, seed):
    """Amplitudes as a deep random circuit gives them: complex normal, sum over 2^n of p = 1."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(case["count"], dtype=torch.complex128, device="cuda",
                       generator=gen) * 2.0 ** (-case["qubits"] / 2)


def _slice_begin(case, net, seed):
    """A range that starts at a slice no tensor forces to zero: the last fSim of two closed
    qubits fixes its input bonds when both bits are equal."""
    _, cut = _stored_path(case["path"])
    return min(supported_slices(net, cut, seed, 1)[0], (1 << len(cut)) - case["count"])


def prepare(case, seed):
    kind = case["kind"]
    if kind == "circuit":
        _, net = _network(case["rows"], case["cols"], case["cycles"], case["open"], seed)
        path, cut = _circuit_path(*_circuit_args(case))
        network = tn.Network.from_workload(net)
        plan = tn.Plan(network, path, cut, mode=case["mode"], eps_budget=case["eps_budget"],
                       use_graph=True)
        return {"kind": "contract", "plan": plan, "begin": 0, "end": 1 << len(cut),
                "amps": 1 << case["open"], "host": case["host"]}
    if kind == "slices":
        rows, cols, cycles, removed, open_ = STORED[case["path"]]
        _, net = _network(rows, cols, cycles, open_, seed, removed, SLICE_THETA)
        path, cut = _stored_path(case["path"])
        network = tn.Network.from_workload(net)
        plan = tn.Plan(network, path, cut, mode=case["mode"], use_graph=True,
                       max_slices_in_flight=case["flight"])
        begin = _slice_begin(case, net, seed)
        return {"kind": "contract", "plan": plan, "begin": begin, "end": begin + case["count"],
                "amps": 1 << open_, "host": False}
    if kind == "sparse":
        _, net = _network(case["rows"], case["cols"], case["cycles"],
                          case["rows"] * case["cols"], seed)
        network = tn.Network.from_workload(net)
        plan = tn.SparsePlan(network, _sparse_path(case["rows"], case["cols"], case["cycles"]),
                             _samples(case, seed), mode=case["mode"])
        return {"kind": "sparse", "plan": plan, "amps": case["samples"]}
    if kind == "step":
        A, B, la, lb, out = _step_operands(case, seed)
        network = tn.Network([A.cpu().numpy().reshape((2,) * len(la)),
                              B.cpu().numpy().reshape((2,) * len(lb))], [la, lb], out)
        plan = tn.Plan(network, [(0, 1)], mode=case["mode"], use_graph=True)
        return {"kind": "contract", "plan": plan, "begin": 0, "end": 1,
                "amps": 1 << len(out), "host": False}
    state = {"kind": "readout", "amps": _readout_amps(case, seed), "qubits": case["qubits"],
             "plan": None}
    if case["plan"]:
        # the plan of a rank that gathered the amplitudes: its network has as many open labels
        n = case["count"].bit_length() - 1
        net = W.build_network(W.hadamard_circuit(max(n, 1)), list(range(n)),
                              {} if n else {0: 0})
        state["plan"] = tn.Plan(tn.Network.from_workload(net),
                                W.greedy_path(net.labels, net.open_labels))
    return state


# ------------------------------------------------------------------------------ the call
def run(state):
    if state["kind"] == "readout":
        if state["plan"] is not None:
            return state["plan"].readout(state["amps"], state["qubits"])
        return tn.readout_noalloc(state["amps"], state["qubits"])
    if state["kind"] == "sparse":
        amps = torch.zeros(state["amps"], dtype=torch.complex128, device="cuda")
        state["plan"].contract(amps)
        return amps.to(torch.complex64)
    if state["host"]:
        return state["plan"].contract_host(state["begin"], state["end"]).astype(np.complex64)
    amps = torch.zeros(state["amps"], dtype=torch.complex128, device="cuda")
    state["plan"].contract(amps, state["begin"], state["end"])
    return amps.to(torch.complex64)


def work(case):
    """Flops of the pairwise contractions (8 per complex multiply-add); inputs and amplitudes as
    complex128, each once."""
    kind = case["kind"]
    if kind == "circuit":
        labels, opens = _structure(*_circuit_args(case)[:4])
        _, flops = _circuit_cost(case)
        return {"bytes": 16.0 * (sum(2.0 ** len(ls) for ls in labels) + 2.0 ** len(opens)),
                "flops": flops}
    if kind == "slices":
        rows, cols, cycles, removed, open_ = STORED[case["path"]]
        labels, opens = _structure(rows, cols, cycles, open_, removed)
        path, cut = _stored_path(case["path"])
        return {"bytes": 16.0 * (sum(2.0 ** len(ls) for ls in labels) + 2.0 ** open_),
                "flops": case["count"] * _cost(labels, opens, path, cut)[1]}
    if kind == "sparse":
        labels, opens = _structure(case["rows"], case["cols"], case["cycles"],
                                   case["rows"] * case["cols"])
        path = _sparse_path(case["rows"], case["cols"], case["cycles"])
        return {"bytes": 16.0 * (sum(2.0 ** len(ls) for ls in labels) + case["samples"]),
                "flops": _sparse_flops(labels, opens, path, case["samples"])}
    if kind == "step":
        lm, ln, lk = case["lm"], case["ln"], case["lk"]
        return {"bytes": 16.0 * (2.0 ** (lm + lk) + 2.0 ** (ln + lk) + 2.0 ** (lm + ln)),
                "flops": 8.0 * 2.0 ** (lm + ln + lk)}
    return {"bytes": 16.0 * case["count"], "flops": 6.0 * case["count"]}


def _sparse_flops(labels, opens, path, samples):
    """Pairwise flops with every open index restricted to at most ``samples`` configurations."""
    openset, total = set(opens), 0.0
    for s in W.replay_path(labels, opens, path):
        union = set(s.labels_a) | set(s.labels_b)
        conf = min(float(samples), 2.0 ** len(union & openset))
        total += 8.0 * conf * 2.0 ** len(union - openset)
    return total


# ------------------------------------------------------------------------------ 64 bits
def _apply(psi, gate, qubits, n):
    """One gate on a state vector (qubit 0 = most significant bit)."""
    u = torch.as_tensor(np.asarray(gate)).tolist()
    cuts, shape, left = sorted(qubits), [], 0
    for q in cuts:
        shape += [1 << (q - left), 2]
        left = q + 1
    x = psi.view(shape + [1 << (n - left)])
    out = torch.empty_like(x)

    def part(t, value):
        for i, q in enumerate(cuts):
            bit = (value >> (len(qubits) - 1 - qubits.index(q))) & 1
            t = t.select(i + 1, bit)
        return t

    for r, row in enumerate(u):
        y, first = part(out, r), True
        for c, v in enumerate(row):
            if v == 0:
                continue
            if first:
                torch.mul(part(x, c), v, out=y)
            else:
                y.add_(part(x, c), alpha=v)
            first = False
        if first:
            y.zero_()
    return out.view(-1)


def _state_vector(circ):
    n = circ.n_qubits
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda")
    psi[0] = 1.0
    waiting = {}  # one-qubit gates are multiplied into the next gate on their qubit
    for g in circ.gates:
        m = np.asarray(g.matrix, dtype=np.complex128)
        if len(g.qubits) == 1:
            waiting[g.qubits[0]] = m @ waiting.get(g.qubits[0], np.eye(2))
            continue
        a, b = g.qubits
        m = m @ np.kron(waiting.pop(a, np.eye(2)), waiting.pop(b, np.eye(2)))
        psi = _apply(psi, m, (a, b), n)
    for q, m in waiting.items():
        psi = _apply(psi, m, (q,), n)
    return psi


def _pair64(a, la, b, lb, keep):
    """One pairwise contraction as a permuted complex128 matrix product; ``keep``: labels still
    needed elsewhere."""
    shared = [l for l in la if l in set(lb)]
    k = [l for l in shared if l not in keep]
    if len(k) < len(shared):
        raise NotImplementedError("batch label")
    m, n = [l for l in la if l not in k], [l for l in lb if l not in k]
    at = a.permute([la.index(l) for l in m + k]).reshape(1 << len(m), 1 << len(k))
    bt = b.permute([lb.index(l) for l in k + n]).reshape(1 << len(k), 1 << len(n))
    return (at @ bt).view((2,) * (len(m) + len(n))), m + n


def _slices64(net, path, cut, begin, count):
    """Sum of a range of slices, contracted pair by pair in complex128."""
    total = 0
    for s in range(begin, begin + count):
        live = {}
        for i, (t, ls) in enumerate(zip(net.tensors, net.labels)):
            t = torch.as_tensor(t, device="cuda")
            fix = {l: (s >> j) & 1 for j, l in enumerate(cut)}
            for ax in range(len(ls) - 1, -1, -1):
                if ls[ax] in fix:
                    t = t.select(ax, fix[ls[ax]])
            live[i] = (t, [l for l in ls if l not in fix])
        opens = set(net.open_labels)
        for a, b in path:
            live[a] = _pair64(*live[a], *live.pop(b), opens)
        (t, ls), = live.values()
        total = total + t.permute([ls.index(l) for l in net.open_labels]).reshape(-1)
    return total


def exact(case, seed):
    kind = case["kind"]
    if kind == "circuit":
        rows, cols, n = case["rows"], case["cols"], case["rows"] * case["cols"]
        circ, net = _network(rows, cols, case["cycles"], case["open"], seed)
        psi = _state_vector(circ)
        bits = 0
        for q in range(n - case["open"]):
            bits = 2 * bits + net.closed_bits[q]
        amps = psi.view(1 << (n - case["open"]), -1)[bits].clone()
        return amps.cpu().numpy() if case["host"] else amps
    if kind == "slices":
        if "53" in case["path"]:
            return None  # 2^44 flops a slice: minutes in 64 bits
        rows, cols, cycles, removed, open_ = STORED[case["path"]]
        _, net = _network(rows, cols, cycles, open_, seed, removed, SLICE_THETA)
        path, cut = _stored_path(case["path"])
        return _slices64(net, path, cut, _slice_begin(case, net, seed), case["count"])
    if kind == "sparse":
        circ, _ = _network(case["rows"], case["cols"], case["cycles"],
                           case["rows"] * case["cols"], seed)
        smp = _samples(case, seed).astype(np.int64)
        n = smp.shape[1]
        index = (smp << np.arange(n - 1, -1, -1)).sum(axis=1)
        return _state_vector(circ)[torch.from_numpy(index).cuda()]
    if kind == "step":
        A, B, la, lb, out = _step_operands(case, seed)
        c, ls = _pair64(A.view((2,) * len(la)), la, B.view((2,) * len(lb)), lb, set())
        return c.permute([ls.index(l) for l in out]).reshape(-1)
    p = _readout_amps(case, seed).abs().square()
    s1, s2 = float(p.sum()), float(p.square().sum())
    d = 2.0 ** case["qubits"]
    return np.array([s1, s2, d * s1 / case["count"] - 1.0, d * s2 / s1 - 1.0])
