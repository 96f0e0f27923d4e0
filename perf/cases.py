"""What the framework is timed on: contraction calls as user programs make them.

A case is one call (or one captured batch of calls) of the public interface on a seeded random
circuit: the seed draws the gates and the bitstrings, the contraction plan belongs to the circuit's
shape (grid and depth) and is either the deterministic greedy one or one of the plans stored in
qxgen/plans.  Kinds of cases:

  contract  one Contractor call, host or device buffers, any precision form, a whole slice sum or a
            shard of its slices (what one process of dist.py contracts)
  serve     one asynchronous request on a serving lane: submitted, polled, amplitudes in pinned memory
  sample    one batch of candidates through qx_esup_sample (contraction, then the rejection tests)
  uneven    several uneven circuits in one captured CUDA graph (UnevenBatch)

The sizes are those of the repository's benchmark workloads (qxgen.workloads) and tests.
"""
import functools
import json
import math
import os

import numpy as np
import torch

from paper_2110_09894_gb300 import qx
from paper_2110_09894_gb300.batch import UnevenBatch
from qxgen import circuits as C
from qxgen import plan as P
from qxgen import workloads as W

PLANS = os.path.join(os.path.dirname(os.path.abspath(P.__file__)), "plans")
PRECISION = {"c64": qx.QX_PREC_C64, "3xtf32": qx.QX_PREC_3XTF32, "bf16x3": qx.QX_PREC_SPLIT_BF16,
             "fp16": qx.QX_PREC_FP16_SCALED}
LARGE = {"annealed": "grid6x6_d14_s10_open6_sa.json", "local-search": "grid6x6_d14_s10_open6_ls.json"}


def listed():
    return [
        # The first call of the README on the smallest benchmark workload: host bitstrings in, host
        # amplitudes out, every option at its default (complex64, the current stream).  Latency.
        contract("small_host_17", grid="3x4", depth=8, n_bits=17, entry="host"),
        # One amplitude of one circuit into a fresh output tensor: the paper's single-amplitude runs.
        contract("single_amplitude_4x4", grid="4x4", depth=12, n_bits=1, entry="device-fresh"),
        # The 64-slice, 256-bitstring workload in its default form: the benchmark's sliced workload.
        contract("sliced_checkpoint_3xtf32", grid="4x5", depth=12, plan="checkpoint", slices=6, n_bits=256,
                 precision="3xtf32", entry="device"),
        # The same workload under the plain greedy plan in the default precision, host to host.
        contract("sliced_greedy_c64_host", grid="4x5", depth=12, slices=6, n_bits=256, entry="host"),
        # ... and with an odd number of bitstrings in the scaled FP16 form.
        contract("sliced_greedy_fp16_201", grid="4x5", depth=12, slices=6, n_bits=201, precision="fp16",
                 entry="device"),
        # The headline workload: 36 qubits, 1024 slices, 64 open amplitudes, annealed plan.
        contract("large_annealed_3xtf32", plan="annealed", precision="3xtf32", entry="device"),
        # One process's shard of the same sum under the older local-search plan (large gathers and permutes).
        contract("large_local_search_shard", plan="local-search", precision="3xtf32", s_begin=64, s_end=160,
                 entry="device"),
        # A shard in the plain complex64 form, the accuracy reference users check the others against.
        contract("large_annealed_c64_shard", plan="annealed", precision="c64", s_begin=0, s_end=64,
                 entry="device"),
        # A ragged shard in the most accurate tensor-core form.
        contract("large_annealed_bf16x3_shard", plan="annealed", precision="bf16x3", s_begin=11, s_end=98,
                 entry="device"),
        # A serving request of 300 bitstrings on a resident 20-qubit circuit's lane.
        {"name": "serve_20q_300", "kind": "serve", "circuit": 7, "n_bits": 300, "precision": "3xtf32"},
        # A batch of candidates of the rejection sampler.
        {"name": "sample_20q_1024", "kind": "sample", "candidates": 1024, "precision": "3xtf32"},
        # 22 uneven circuits, light ones in the persistent launch and heavy ones batched, one graph.
        {"name": "uneven_22_circuits", "kind": "uneven", "first": 100, "count": 24, "precision": "3xtf32"},
    ]


def contract(name=None, grid="6x6", depth=14, plan="greedy", slices=0, n_open=0, n_bits=1, precision="c64",
             entry="device", s_begin=0, s_end=-1):
    case = {"kind": "contract", "grid": grid, "depth": depth, "plan": plan, "slices": slices, "n_open": n_open,
            "n_bits": n_bits, "precision": precision, "entry": entry, "s_begin": s_begin, "s_end": s_end}
    if name:
        case["name"] = name
    if plan in LARGE:  # 10 sliced bonds, qubits 30..35 open
        case |= {"slices": 10, "n_open": 6}
    return case


def draw(rng):
    kind = rng.choice(["grid", "grid", "grid", "large", "member", "serve", "sample", "uneven"])
    if kind == "large":
        precision = rng.choice(list(PRECISION))
        n = int(2 ** rng.uniform(0, 8 if precision != "c64" else 6))
        b = rng.randrange(1024 - n)
        return contract(plan=rng.choice(list(LARGE)), precision=precision, s_begin=b, s_end=b + n)
    if kind == "member":  # one of the uneven workload's circuits by itself
        js = [j for j, d in _member_plans().items() if d["estimated_s"] < 0.03]
        return {"kind": "member", "circuit": rng.choice(js), "precision": rng.choice(list(PRECISION))}
    if kind == "serve":
        js = [j for j, d in _serving_plans().items() if d["estimated_s"] < 0.03]
        return {"kind": "serve", "circuit": rng.choice(js), "n_bits": int(2 ** rng.uniform(0, 8.5)),
                "precision": rng.choice(["c64", "3xtf32"])}
    if kind == "sample":
        return {"kind": "sample", "candidates": int(2 ** rng.uniform(5, 11.5)),
                "precision": rng.choice(["c64", "3xtf32"])}
    if kind == "uneven":
        count = rng.randint(3, 14)
        return {"kind": "uneven", "first": rng.randrange(256 - count), "count": count,
                "precision": rng.choice(["3xtf32", "bf16x3"])}
    while True:
        rows = rng.randint(2, 5)
        cols = rng.randint(rows, 6 if rows < 4 else 5)
        case = contract(grid=f"{rows}x{cols}", depth=rng.randint(4, 14), slices=rng.randint(0, 6),
                        n_open=rng.choice([0, 0, 0, 1, 2, 5]), n_bits=int(2 ** rng.uniform(0, 8.6)),
                        precision=rng.choice(list(PRECISION)), entry=rng.choice(["host", "device", "device-fresh"]))
        try:
            n, rows, cols, depth, open_mask, order, sliced = _shape(_key(case))
        except ValueError:  # fewer bonds than slices asked for
            continue
        if work(case)["flops"] < 2e11 and P.plan_cost(_legs(n, rows, cols, depth, open_mask), order, sliced)[0] < 22:
            return case


# --- circuits and plans ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _stored(name):
    with open(os.path.join(PLANS, name)) as f:
        return json.load(f)


@functools.lru_cache(maxsize=None)
def _member_plans():
    plans = {d["j"]: d for d in _stored("batched_uneven.json")["plans"]}
    plans.update({d["j"]: d for d in _stored("batched_annealed.json")["plans"]})
    return plans


@functools.lru_cache(maxsize=None)
def _serving_plans():
    return {d["j"]: d for d in _stored("serving.json")["plans"]}


def _key(case):
    """What decides the plan of a case's circuit: the seed draws its gates, not its shape."""
    if case["kind"] in ("member", "serve"):
        return case["kind"], case["circuit"]
    if case["kind"] == "sample":
        return "contract", "4x5", 12, "checkpoint", 6, 0
    return "contract", case["grid"], case["depth"], case["plan"], case["slices"], case["n_open"]


@functools.lru_cache(maxsize=None)
def _shape(key):
    """(qubits, rows, columns, depth, open mask, order, sliced bonds)"""
    if key[0] in ("member", "serve"):
        n, depth = W.batched_specs()[key[1]][:2] if key[0] == "member" else W.serving_specs()[key[1]]
        d = (_member_plans() if key[0] == "member" else _serving_plans())[key[1]]
        rows, cols = C.near_square_shape(n)
        return n, rows, cols, depth, np.zeros(n, np.uint8), d["order"], d["sliced"]
    _, grid, depth, plan, slices, n_open = key
    rows, cols = (int(x) for x in grid.split("x"))
    n = rows * cols
    open_mask = np.zeros(n, np.uint8)
    open_mask[n - n_open:] = 1
    if plan != "greedy":
        d = _stored(LARGE.get(plan, "grid4x5_d12_s6_checkpoint.json"))
        return n, rows, cols, depth, open_mask, d["order"], d["sliced"]
    order, sliced, _, _ = W.make_plan(C.random_grid_circuit(rows, cols, depth, 0), open_mask, slices, 1)
    return n, rows, cols, depth, open_mask, order, sliced


def _legs(n, rows, cols, depth, open_mask):
    circ = C.random_grid_circuit(rows, cols, depth, 0, n=n)
    return P.network_legs(n, [g.qubits for g in circ.gates], open_mask)[0]


def _members(case):
    return [j for j in range(case["first"], case["first"] + case["count"])
            if _member_plans()[j]["estimated_s"] < 0.02]


class _Member:
    """One circuit of an uneven batch, as UnevenBatch takes it."""

    def __init__(self, j, seed):
        self.n_qubits, rows, cols, depth, self.open_mask, order, sliced = _shape(("member", j))
        self.circuit = C.random_grid_circuit(rows, cols, depth, seed + j, n=self.n_qubits)
        self.gates = C.gates_to_records(self.circuit)
        self.order, self.sliced = np.asarray(order, np.int64), np.asarray(sliced, np.int64)
        self.n_open = 0
        self.bitstrings = _bits(self.n_qubits, W.batched_specs()[j][3], seed + j)
        self.peak_rank = _peak(j)


@functools.lru_cache(maxsize=None)
def _peak(j):
    n, rows, cols, depth, open_mask, order, sliced = _shape(("member", j))
    return P.plan_cost(_legs(n, rows, cols, depth, open_mask), order, sliced)[0]


def _bits(n_qubits, count, seed):
    return np.random.default_rng(seed).integers(0, 2, size=(count, n_qubits), dtype=np.uint8)


def _n_bits(case):
    return {"member": lambda: W.batched_specs()[case["circuit"]][3],
            "sample": lambda: case["candidates"]}.get(case["kind"], lambda: case["n_bits"])()


def _slice_range(case):
    n_slices = 1 << len(_shape(_key(case))[6])
    return case.get("s_begin", 0), n_slices if case.get("s_end", -1) < 0 else case["s_end"]


# --- the calls ------------------------------------------------------------------------------------

def prepare(case, seed):
    dev = torch.device("cuda", 0)
    if case["kind"] == "uneven":
        batch = UnevenBatch([_Member(j, seed) for j in _members(case)], precision=PRECISION[case["precision"]],
                            mem_budget=16 << 30)
        batch.capture()
        return {"case": case, "batch": batch}
    n, rows, cols, depth, open_mask, order, sliced = _shape(_key(case))
    gates = C.gates_to_records(C.random_grid_circuit(rows, cols, depth, seed, n=n))
    n_bits = _n_bits(case)
    bits = _bits(n, n_bits, seed)
    # a program that keeps one circuit resident gives it a stream of its own; the shortest programs
    # (fresh outputs, host buffers) stay on the current one
    plain = case.get("entry") in ("host", "device-fresh")
    stream = torch.cuda.current_stream(dev) if plain else torch.cuda.Stream(dev)
    kw = {"precision": PRECISION[case["precision"]], "stream": stream}
    if case["kind"] == "contract" and case["plan"] in LARGE:
        kw["workspace_bytes"] = 24 << 30
    elif case["kind"] == "serve":
        kw["workspace_bytes"] = _workspace(case, kw["precision"], 4096)
    else:
        kw["workspace_bytes"] = _workspace(case, kw["precision"], (1 << len(sliced)) * n_bits)
    c = qx.Contractor(n, gates, open_mask, np.asarray(order, np.int64), np.asarray(sliced, np.int64), n_bits, **kw)
    state = {"case": case, "c": c, "bits": bits, "stream": stream, "range": _slice_range(case)}
    with torch.cuda.stream(stream):
        state["d_bits"] = torch.from_numpy(bits).to(dev)
        state["d_amps"] = torch.zeros((n_bits, 1 << c.n_open, 2), dtype=torch.float64, device=dev)
        if case["kind"] == "serve":  # as a server's lane: invariant tensors kept, launches in plan order
            qx.qx_set_memo(c.h, 1)
            qx.qx_set_streams(c.h, 1)
            state["h_amps"] = torch.zeros((n_bits, 1, 2), dtype=torch.float64).pin_memory()
        if case["kind"] == "sample":
            qx.qx_set_memo(c.h, 1)
            state["d_u"] = torch.from_numpy(np.random.default_rng(seed + 1).random(n_bits)).to(dev)
            state["d_acc"] = torch.zeros(n_bits, dtype=torch.int64, device=dev)
    torch.cuda.synchronize(dev)
    return state


def _workspace(case, precision, pairs):
    """Bytes for a batch of `pairs` (slice, bitstring) pairs, at most 24 GiB."""
    n, rows, cols, depth, open_mask, order, sliced = _shape(_key(case))
    h = qx.qx_create(-1, precision=precision)
    try:
        qx.qx_build_network(h, n, C.gates_to_records(C.random_grid_circuit(rows, cols, depth, 0, n=n)), open_mask)
        qx.qx_set_plan(h, order, sliced)
        one, want = (qx.qx_workspace_size(h, _n_bits(case), p) for p in (1, min(pairs, 65535)))
        return max(one, min(want, 24 << 30))
    finally:
        qx.qx_destroy(h)


def run(state):
    case = state["case"]
    if case["kind"] == "uneven":
        state["batch"].replay()
        return state["batch"].d_amps
    c, d_bits, (s0, s1) = state["c"], state["d_bits"], state["range"]
    if case["kind"] == "serve":
        req = qx.qx_submit(c.h, d_bits.data_ptr(), len(d_bits), s0, s1, state["d_amps"].data_ptr(),
                           state["h_amps"].data_ptr())
        while not qx.qx_poll(c.h, req):
            pass
        return state["h_amps"]
    if case["kind"] == "sample":
        n = len(d_bits)
        found, used, m = qx.qx_esup_sample(c.h, d_bits.data_ptr(), state["d_u"].data_ptr(), n, n // 8, n, 1.0,
                                           state["d_amps"].data_ptr(), state["d_acc"].data_ptr())
        return {"amps": state["d_amps"], "accepted": state["d_acc"], "found": found, "used": used, "bound": m}
    if case["kind"] == "contract" and case["entry"] == "host":
        return c.contract(state["bits"])
    if case["kind"] == "contract" and case["entry"] == "device-fresh":
        return c.contract_device(d_bits, None, s0, s1)
    with torch.cuda.stream(state["stream"]):
        return c.contract_device(d_bits, state["d_amps"], s0, s1)


def work(case):
    """Flops of the plan's products (8 M K N, each distinct one once) and the bytes of gates, bitstrings
    and amplitudes."""
    if case["kind"] == "uneven":
        ws = [work({"kind": "member", "circuit": j}) for j in _members(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    n, rows, cols, depth, open_mask, order, sliced = _shape(_key(case))
    s0, s1 = _slice_range(case)
    n_bits = _n_bits(case)
    once, per_slice, per_pair = _level_flops(_key(case))
    amps = n_bits << int(open_mask.sum())
    return {"bytes": 272 * len(_legs(n, rows, cols, depth, open_mask)) + n_bits * n + 16 * amps,
            "flops": once + (s1 - s0) * (per_slice + n_bits * per_pair)}


@functools.lru_cache(maxsize=None)
def _level_flops(key):
    """Flops of the steps that neither slices nor bitstrings reach, per slice, and per (slice, bitstring)."""
    n, rows, cols, depth, open_mask, order, sliced = _shape(key)
    legs, n_out = _legs(n, rows, cols, depth, open_mask), n - int(open_mask.sum())
    # executed_cost(b) = once + slices * (per_slice + b * per_pair)
    n_slices, once = 1 << len(sliced), _once_flops(legs, order, sliced, n_out)
    all_slices = P.executed_cost(legs, order, sliced, n_out, 0) - once
    per_pair = (P.executed_cost(legs, order, sliced, n_out, 1) - once - all_slices) // n_slices
    return once, all_slices // n_slices, per_pair


def _once_flops(legs, order, sliced, n_out):
    fixed = set(sliced) | {e for t in legs[len(legs) - n_out:] for e in t}
    sets, free = [frozenset(t) for t in legs], [not fixed & set(t) for t in legs]
    total = 0
    for a, b in order:
        free.append(free[a] and free[b])
        if free[-1]:
            total += 8 << len(sets[a] | sets[b])
        sets.append(sets[a] ^ sets[b])
    return total


# --- the same in 64 bits, with torch alone --------------------------------------------------------

def exact(case, seed):
    if case["kind"] == "uneven":
        out = []
        for j in _members(case):
            m = _Member(j, seed)
            out.append(_real(_state_amps(m.circuit, m.open_mask, m.bitstrings)))
        return out
    n, rows, cols, depth, open_mask, order, sliced = _shape(_key(case))
    circ = C.random_grid_circuit(rows, cols, depth, seed, n=n)
    bits = _bits(n, _n_bits(case), seed)
    s0, s1 = _slice_range(case)
    if n > 29 or s1 - s0 < 1 << len(sliced):
        if (s1 - s0) > 128:
            return None  # minutes of complex128 products
        return _real(_plan_amps(circ, open_mask, order, sliced, bits, s0, s1))
    amps = _state_amps(circ, open_mask, bits)
    if case["kind"] == "contract" and case["entry"] == "host":
        return amps.cpu().numpy()
    if case["kind"] == "sample":
        return {"amps": _real(amps), "accepted": None, "found": None, "used": None, "bound": None}
    return _real(amps)


def _real(amps):
    return torch.view_as_real(amps.contiguous())


def _device():
    return torch.device("cuda", 0) if torch.cuda.is_available() else torch.device("cpu")


def _state_amps(circ, open_mask, bits):
    """Amplitudes [bitstring][open assignment] by evolving the state vector gate by gate."""
    n, dev = circ.n_qubits, _device()
    psi = torch.zeros(1 << n, dtype=torch.complex128, device=dev)
    psi[0] = 1
    for g in circ.gates:
        m = torch.from_numpy(np.ascontiguousarray(g.matrix)).to(dev)
        if len(g.qubits) == 1:
            v = psi.view(1 << g.qubits[0], 2, -1)
            psi = torch.stack([m[r, 0] * v[:, 0] + m[r, 1] * v[:, 1] for r in (0, 1)], 1).reshape(-1)
        else:
            (a, b), m = g.qubits, m.view(2, 2, 2, 2)
            if a > b:
                (a, b), m = (b, a), m.permute(1, 0, 3, 2)
            v = psi.view(1 << a, 2, 1 << (b - a - 1), 2, -1)
            out = torch.zeros_like(v)
            for r in range(2):
                for s in range(2):
                    for x in range(2):
                        for y in range(2):
                            if m[r, s, x, y] != 0:
                                out[:, r, :, s] += m[r, s, x, y] * v[:, x, :, y]
            psi = out.view(-1)
    open_q = [q for q in range(n) if open_mask[q]]
    base = sum(torch.from_numpy(bits[:, q].astype(np.int64)) << (n - 1 - q) for q in range(n) if not open_mask[q])
    index = base[:, None] + torch.tensor([[sum(((o >> (len(open_q) - 1 - i)) & 1) << (n - 1 - q)
                                                for i, q in enumerate(open_q)) for o in range(1 << len(open_q))]])
    return psi[index.to(dev)]


def _plan_amps(circ, open_mask, order, sliced, bits, s0, s1):
    """The partial slice sum of one bitstring by the plan's products in complex128; a product is kept
    while the slice bits below it stay the same."""
    dev, n = _device(), circ.n_qubits
    legs, _, open_edges = P.network_legs(n, [g.qubits for g in circ.gates], open_mask)
    values = [torch.tensor([1, 0], dtype=torch.complex128)] * n
    values += [torch.from_numpy(np.ascontiguousarray(g.matrix)).reshape([2] * (2 * len(g.qubits))) for g in circ.gates]
    values += [torch.eye(2, dtype=torch.complex128)[int(bits[0, q])] for q in range(n) if not open_mask[q]]
    bit_of = {e: j for j, e in enumerate(sliced)}
    kept = [None] * (len(legs) + len(order))
    total = 0
    for s in range(s0, s1):
        made, labels = [], []
        for t, v in enumerate(values):
            cut = tuple((bit_of[e], (s >> bit_of[e]) & 1) for e in legs[t] if e in bit_of)
            made.append(cut)
            labels.append([e for e in legs[t] if e not in bit_of])
            if kept[t] is None or kept[t][0] != cut:
                kept[t] = (cut, v[tuple((s >> bit_of[e]) & 1 if e in bit_of else slice(None)
                                        for e in legs[t])].to(dev))
        for i, (a, b) in enumerate(order):
            t = len(legs) + i
            cut = tuple(sorted(set(made[a]) | set(made[b])))
            shared = [e for e in labels[a] if e in labels[b]]
            made.append(cut)
            labels.append([e for e in labels[a] if e not in shared] + [e for e in labels[b] if e not in shared])
            if kept[t] is None or kept[t][0] != cut:
                kept[t] = (cut, torch.tensordot(kept[a][1], kept[b][1], ([labels[a].index(e) for e in shared],
                                                                         [labels[b].index(e) for e in shared])))
        root = kept[-1][1].permute([labels[-1].index(e) for e in open_edges])
        total = total + root.reshape(1, -1)
    return total
