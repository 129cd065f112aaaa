"""Timed cases of the contraction engine: what a program asks of it through the public binding.

A case is a dict of plain values; `work` names its kind:

  amplitude     one <x|C|0> by tn_contract, the bitstring replaced before the call
  amplitudes    many bitstrings of one circuit as a resident batch (`call` = "resident": results stay on
                the device; "bitstrings": new bitstrings in and results read back in the pass)
  expectations  many <Z_i Z_j> of one circuit as a resident batch
  mixed         queries of several circuits of uneven size in one batch
  trace         tr(A B C) of dense matrices, `jobs` of them: one dense step and one long reduction
  permute       the axes of a device tensor in another order

`parts` is the number k of partitions and `anneal` the annealing iterations of the plan.

Circuits have a fixed structure per case; the gates, bitstrings, pairs, matrices and tensors come from the
seed.  The plan depends on the structure alone, so it is made once and kept, as a program would.
"""
import functools
import math
import random

import numpy as np
import torch

from paper_2507_20667_gb300 import inputs, tnsa

Z = np.diag([1.0, -1.0]).astype(np.complex128)


def listed():
    return [
        # a user's first amplitude, and the latency of a lone query: 10 qubits, Greedy tree, host in, host out
        dict(name="single_10q_c64", work="amplitude", layout="1d", qubits=10, depth=8, parts=1, anneal=0, precision="c64"),
        # sampling a small circuit: many short contractions that live wholly in on-chip programs
        dict(name="amps_10q_c64_512", work="amplitudes", layout="1d", qubits=10, depth=8, parts=1, anneal=0,
             precision="c64", jobs=512, call="resident"),
        # a small batch of a mid-sized circuit: too few jobs to fill the GPU, the longest chain counts
        dict(name="amps_24q_c64_64", work="amplitudes", layout="1d", qubits=24, depth=14, parts=4, anneal=600,
             precision="c64", jobs=64, call="resident"),
        # the benchmark's workload, end to end: new bitstrings from the host, every amplitude read back
        dict(name="amps_24q_c64_2432", work="amplitudes", layout="1d", qubits=24, depth=14, parts=4, anneal=600,
             precision="c64", jobs=2432, call="bitstrings"),
        # a 2D circuit in split precision: uneven partitions, some dense steps on the tensor cores
        dict(name="grid_4x5_bf16_256", work="amplitudes", layout="4x5", qubits=20, depth=8, parts=8, anneal=100,
             precision="bf16", jobs=256, call="resident"),
        # expectation values in the correctness precision
        dict(name="zz_12q_c128_64", work="expectations", layout="1d", qubits=12, depth=8, parts=2, anneal=100,
             precision="c128", jobs=64),
        # a server's launch: circuits of different size and layout, a few queries of each
        dict(name="mixed_bf16", work="mixed", circuits=8, queries=16, qubits_min=16, qubits_max=24, structure=100,
             anneal=100, precision="bf16"),
        # large dense steps: split precision at full tiles, ragged sizes in the finer split, plain complex64
        dict(name="trace_bf16_2048x1024x4096", work="trace", rows=2048, shared=1024, cols=4096, jobs=1,
             precision="bf16"),
        dict(name="trace_tf32_ragged", work="trace", rows=777, shared=1001, cols=1333, jobs=3, precision="tf32"),
        dict(name="trace_c64_1024x512x1536", work="trace", rows=1024, shared=512, cols=1536, jobs=2, precision="c64"),
        # the transposition of a large qubit tensor (every axis moves), and of a ragged complex128 one
        dict(name="permute_reversed_2p26", work="permute", dims=",".join(["2"] * 26), order="reversed", elem=8),
        dict(name="permute_ragged_c128", work="permute", dims="37,5,129,3,61", order="shuffled:3", elem=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["amplitude", "amplitudes", "amplitudes", "expectations", "mixed", "trace", "permute", "permute"])
    if kind == "permute":
        elem = rng.choice([4, 8, 8, 16])
        if rng.random() < 0.5:   # qubit tensors
            n = rng.randint(10, 26 if elem <= 8 else 25)
            dims = [2] * n
        else:                    # general bond dimensions, odd ones among them
            dims, total = [], _log_int(rng, 1 << 10, 1 << 25)
            while len(dims) < rng.randint(2, 7):
                d = _log_int(rng, 2, 200)
                if math.prod(dims) * d > total:
                    break
                dims.append(d)
            if len(dims) < 2:
                dims = [_log_int(rng, 16, 600), _log_int(rng, 16, 600)]
        order = rng.choice(["reversed", "shuffled:%d" % rng.randrange(1000), "legs:%d" % rng.randrange(1000)])
        return dict(work="permute", dims=",".join(map(str, dims)), order=order, elem=elem)
    if kind == "trace":
        precision = rng.choice(["bf16", "tf32", "c64"])
        top = 2048 if precision != "c64" else 1024
        m, k, n = (_log_int(rng, 64, top) for _ in range(3))
        return dict(work="trace", rows=m, shared=k, cols=n, jobs=rng.randint(1, 4), precision=precision)
    if kind == "mixed":
        return dict(work="mixed", circuits=rng.randint(2, 8), queries=rng.randint(2, 24), qubits_min=10,
                    qubits_max=rng.randint(12, 22), structure=rng.randrange(1000), anneal=rng.choice([60, 100, 200]),
                    precision=rng.choice(["c64", "bf16", "tf32"]))
    if kind == "expectations":
        return dict(work=kind, layout="1d", qubits=rng.randint(8, 12), depth=rng.randint(4, 8), parts=rng.choice([1, 2]),
                    anneal=rng.choice([30, 100]), precision=rng.choice(["c128", "c64"]), jobs=_log_int(rng, 8, 64))
    if kind == "amplitude":
        return dict(work=kind, layout="1d", qubits=rng.randint(6, 14), depth=rng.randint(4, 10), parts=rng.choice([1, 2]),
                    anneal=rng.choice([30, 100]), precision=rng.choice(["c64", "c64", "c128"]))
    if rng.random() < 0.7:
        case = dict(work=kind, layout="1d", qubits=rng.randint(8, 24), depth=rng.randint(6, 14))
    else:
        rows, cols = rng.choice([(3, 3), (3, 4), (3, 5), (4, 4), (4, 5)])
        case = dict(work=kind, layout="%dx%d" % (rows, cols), qubits=rows * cols, depth=rng.randint(6, 8))
    case.update(parts=rng.choice([1, 2, 4]), anneal=rng.choice([60, 100, 300]),
                precision=rng.choice(["c64", "c64", "bf16", "tf32"]), jobs=_log_int(rng, 16, 2432),
                call=rng.choice(["resident", "bitstrings"]))
    macs, _, mem = _counts(case)
    while (macs > 2e8 or mem > 2e7) and case["depth"] > 4:   # within one GPU and the largest listed case
        case["depth"] -= 1
        macs, _, mem = _counts(case)
    case["jobs"] = int(max(1, min(case["jobs"], 8e9 // macs, 2e9 // mem)))
    return case


# ---------------------------------------------------------------------- circuits, networks, plans
def _circuit(layout, qubits, depth, seed):
    if layout == "1d":
        return inputs.brickwork_1d(qubits, depth, seed)
    rows, cols = (int(v) for v in layout.split("x"))
    return inputs.grid_2d(rows, cols, depth, seed)


def _network(kind, circ):
    """(network, tensor ids a query replaces): the bra tensors, or the Z slots of <Z_i Z_j>."""
    if kind == "expectations":
        return inputs.zz_slots_tn(circ)
    net = inputs.amplitude_tn(circ, np.zeros(circ.n_qubits, np.int64))
    return net, inputs.bra_ids(net, circ.n_qubits)


@functools.lru_cache(maxsize=64)
def _plan_of(kind, layout, qubits, depth, parts, anneal):
    net, _ = _network(kind, _circuit(layout, qubits, depth, 0))
    h = tnsa.tn_build(net)
    if parts == 1:
        return tnsa.tn_plan_create(h, k=1)
    return tnsa.tn_plan_create(h, k=parts, iterations=anneal, steps_per_temp=8, seed=7, position=net.qubit)


def _plan(case):
    kind = "expectations" if case["work"] == "expectations" else "amplitudes"
    return _plan_of(kind, case["layout"], case["qubits"], case["depth"], case["parts"], case["anneal"])


def _counts(case):
    return tnsa.tn_plan_counts(_plan(case))


def _members(case):
    """The circuits of a mixed case: like a query pool, 1D and 2D in turn, 1 to 4 parts."""
    rng, out = random.Random(case["structure"]), []
    for i in range(case["circuits"]):
        n = rng.randint(case["qubits_min"], case["qubits_max"])
        if i % 2 == 0:
            layout, depth = "1d", rng.randint(8, 12)
        else:
            rows = int(math.sqrt(n))
            layout, depth = "%dx%d" % (rows, n // rows), rng.randint(6, 8)
            n = rows * (n // rows)
        out.append(dict(work="amplitudes", layout=layout, qubits=n, depth=depth, parts=(1, 2, 4)[i % 3],
                        anneal=case["anneal"]))
    return out


def _bits(rng, jobs, n):
    return rng.integers(0, 2, (jobs, n))


def _pairs(rng, jobs, n):
    return np.array([rng.choice(n, 2, replace=False) for _ in range(jobs)])


def _matrices(case, seed):
    rng = np.random.default_rng(seed)
    m, k, n = case["rows"], case["shared"], case["cols"]

    def normal(*shape):
        return (rng.standard_normal((*shape, 2)) * math.sqrt(0.5)).view(np.complex128)[..., 0]
    return [(normal(m, k), normal(k, n), normal(n, m)) for _ in range(case["jobs"])]


def _trace_network(mats):
    a, b, c = mats
    # A axis 1 - B axis 0, B axis 1 - C axis 0, C axis 1 - A axis 0
    return inputs.Network([a, b, c], np.array([[0, 1, 1, 0], [1, 1, 2, 0], [2, 1, 0, 0]], np.int32),
                          np.zeros(3, np.int32), ["dense"] * 3)


def _perm(case):
    dims = [int(d) for d in case["dims"].split(",")]
    how, _, num = case["order"].partition(":")
    axes = list(range(len(dims)))
    if how == "reversed":
        return dims, axes[::-1]
    rng = random.Random(int(num))
    if how == "shuffled":
        rng.shuffle(axes)
        return dims, axes
    # the operand of a pairwise step: a few legs (the shared ones) move to the end, the others keep their order
    shared = set(rng.sample(axes, max(1, len(axes) // 4)))
    return dims, [a for a in axes if a not in shared] + [a for a in axes if a in shared]


DTYPES = {4: torch.float32, 8: torch.complex64, 16: torch.complex128}


def _tensor(case, seed):
    dims, _ = _perm(case)
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(math.prod(dims), dtype=DTYPES[case["elem"]], device="cuda", generator=g)


# ---------------------------------------------------------------------- prepare and run
@functools.lru_cache(maxsize=1)
def _stream():
    """The one stream of the program: a context made without a stream would have its own."""
    return torch.cuda.Stream()


def _stage(batch, ids, values):
    """Arguments of tn_batch_set_tensors: job j's tensors `ids` take the rows of values[j]."""
    jobs = np.repeat(np.arange(len(values), dtype=np.int32), len(ids))
    tensors = np.tile(np.asarray(ids, dtype=np.int32), len(values))
    return batch, jobs, tensors, np.ascontiguousarray(values)


def prepare(case, seed):
    with torch.cuda.stream(_stream()):
        return _prepare(case, seed)


def _prepare(case, seed):
    kind = case["work"]
    if kind == "permute":
        x = _tensor(case, seed)
        dims, perm = _perm(case)
        out = torch.empty(math.prod(dims), dtype=x.dtype, device="cuda")
        ctx = tnsa.tn_ctx_create(0, stream=torch.cuda.current_stream().cuda_stream)
        return dict(kind=kind, ctx=ctx, x=x, out=out, elem=case["elem"], dims=dims, perm=perm)
    ctx = tnsa.tn_ctx_create(0, stream=torch.cuda.current_stream().cuda_stream)
    state = dict(kind=kind, ctx=ctx, precision=case["precision"],
                 dtype=torch.complex128 if case["precision"] == "c128" else torch.complex64)
    rng = np.random.default_rng([seed, 1])
    eye = np.eye(2, dtype=np.complex128)
    if kind == "amplitude":
        circ = _circuit(case["layout"], case["qubits"], case["depth"], seed)
        net, ids = _network(kind, circ)
        state.update(net=tnsa.tn_build(net), plan=_plan(case), ids=ids, bra=eye[_bits(rng, 1, circ.n_qubits)[0]])
        return state
    if kind == "trace":
        nets = [tnsa.tn_build(_trace_network(m)) for m in _matrices(case, seed)]
        plan = tnsa.tn_plan_import(nets[0], [(0, 1), (2, 3)])
        state["batch"] = tnsa.tn_batch_create(ctx, nets, [plan] * len(nets), case["precision"])
        jobs = len(nets)
    elif kind == "mixed":
        nets, plans, stage = [], [], []
        for m in _members(case):
            circ = _circuit(m["layout"], m["qubits"], m["depth"], seed)
            net, ids = _network(kind, circ)
            h = tnsa.tn_build(net)
            for x in _bits(rng, case["queries"], circ.n_qubits):
                stage.append((len(nets), ids, eye[x]))
                nets.append(h)
                plans.append(_plan(m))
        jobs = len(nets)
        state["batch"] = tnsa.tn_batch_create(ctx, nets, plans, case["precision"])
        tnsa.tn_batch_set_tensors(state["batch"], np.concatenate([[j] * len(ids) for j, ids, _ in stage]),
                                  np.concatenate([ids for _, ids, _ in stage]), np.concatenate([v for *_, v in stage]))
    else:
        circ = _circuit(case["layout"], case["qubits"], case["depth"], seed)
        net, ids = _network(kind, circ)
        jobs = case["jobs"]
        state["batch"] = tnsa.tn_batch_create(ctx, [tnsa.tn_build(net)] * jobs, [_plan(case)] * jobs, case["precision"])
        if kind == "expectations":
            values = np.broadcast_to(eye, (jobs, circ.n_qubits, 2, 2)).copy()
            for v, (i, j) in zip(values, _pairs(rng, jobs, circ.n_qubits)):
                v[i] = v[j] = Z
        else:
            values = eye[_bits(rng, jobs, circ.n_qubits)]
        state["stage"] = _stage(state["batch"], ids, values)
        if case.get("call") == "bitstrings":
            state["kind"] = "bitstrings"
        else:
            tnsa.tn_batch_set_tensors(*state["stage"])
    state["records"] = torch.zeros((jobs, 4), dtype=torch.float64, device="cuda")
    return state


def run(state):
    kind = state["kind"]
    if kind == "permute":
        tnsa.tn_permute(state["ctx"], state["x"].data_ptr(), state["out"].data_ptr(), state["elem"], state["dims"],
                        state["perm"])
        return state["out"]
    if kind == "amplitude":
        for t, v in zip(state["ids"], state["bra"]):
            tnsa.tn_net_set_tensor(state["net"], t, v)
        m, e, _ = tnsa.tn_contract(state["ctx"], state["net"], state["plan"], state["precision"])
        return np.array(tnsa.amplitude(m, e), np.complex128 if state["precision"] == "c128" else np.complex64)
    if kind == "bitstrings":
        tnsa.tn_batch_set_tensors(*state["stage"])
        tnsa.tn_batch_run(state["batch"])
        m, e, status = tnsa.tn_batch_results(state["batch"])
        return {"values": (m * np.exp2(e)).astype(np.complex64), "status": status}
    records = state["records"]   # per job: {double re, double im, int32 exp2, int32 status}
    tnsa.tn_batch_run(state["batch"], records.data_ptr())
    words = records.view(torch.int32)
    with torch.cuda.stream(_stream()):
        values = torch.view_as_complex(records[:, :2] * torch.exp2(words[:, 4:5].double())).to(state["dtype"])
    return {"values": values, "status": words[:, 5]}


# ---------------------------------------------------------------------- what a pass cannot do without
def work(case):
    kind = case["work"]
    if kind == "permute":
        n = math.prod(_perm(case)[0])
        return dict(bytes=2.0 * n * case["elem"], flops=0.0)
    if kind == "trace":
        m, k, n, jobs = case["rows"], case["shared"], case["cols"], case["jobs"]
        return dict(bytes=jobs * (16.0 * (m * k + k * n + n * m) + 32), flops=8.0 * jobs * (m * n * k + m * n))
    if kind == "mixed":
        parts = [work(dict(m, jobs=case["queries"])) for m in _members(case)]
        return {key: float(sum(p[key] for p in parts)) for key in ("bytes", "flops")}
    jobs = case.get("jobs", 1)
    net, _ = _network("expectations" if kind == "expectations" else "amplitudes",
                      _circuit(case["layout"], case["qubits"], case["depth"], 0))
    return dict(bytes=jobs * (16.0 * sum(t.size for t in net.tensors) + 32), flops=8.0 * jobs * _counts(case)[0])


# ---------------------------------------------------------------------- the same values in 64 bits
def _state_vector(circ):
    n = circ.n_qubits
    psi = torch.zeros(1 << n, dtype=torch.complex128, device="cuda" if torch.cuda.is_available() else "cpu")
    psi[0] = 1
    for g in circ.gates:
        if len(g.qubits) == 1:
            u = torch.from_numpy(g.matrix).to(psi.device)
            v = psi.view(1 << g.qubits[0], 2, -1)
            v0, v1 = v[:, 0], v[:, 1]
            psi = torch.stack((u[0, 0] * v0 + u[0, 1] * v1, u[1, 0] * v0 + u[1, 1] * v1), 1).reshape(-1)
        else:   # the only two-qubit gate of these circuits is CZ
            a, b = g.qubits
            psi.view(1 << a, 2, 1 << (b - a - 1), 2, -1)[:, 1, :, 1].mul_(-1)
    return psi


def _amplitudes(circ, bits):
    weights = 1 << np.arange(circ.n_qubits - 1, -1, -1)
    psi = _state_vector(circ)
    return psi[torch.from_numpy(bits @ weights).to(psi.device)].cpu()


def exact(case, seed):
    kind = case["work"]
    rng = np.random.default_rng([seed, 1])
    if kind == "permute":
        dims, perm = _perm(case)
        strides = [math.prod(dims[i + 1:]) for i in range(len(dims))]
        # flat source index of every output element (torch takes at most 25 axes)
        src = torch.zeros(1, dtype=torch.int64, device="cuda")
        for p in perm:
            src = (src[:, None] + strides[p] * torch.arange(dims[p], device="cuda")).reshape(-1)
        return _tensor(case, seed)[src]
    if kind == "trace":
        dev, out = "cuda" if torch.cuda.is_available() else "cpu", []
        for mats in _matrices(case, seed):
            a, b, c = (torch.from_numpy(np.ascontiguousarray(x)).to(dev) for x in mats)
            out.append(((a @ b) * c.T).sum().cpu())
        return {"values": torch.stack(out), "status": None}
    if kind == "mixed":
        values = []
        for m in _members(case):
            circ = _circuit(m["layout"], m["qubits"], m["depth"], seed)
            values.append(_amplitudes(circ, _bits(rng, case["queries"], circ.n_qubits)))
        return {"values": torch.cat(values), "status": None}
    circ = _circuit(case["layout"], case["qubits"], case["depth"], seed)
    n = circ.n_qubits
    if kind == "amplitude":
        return _amplitudes(circ, _bits(rng, 1, n))[0]
    if kind == "amplitudes":
        return {"values": _amplitudes(circ, _bits(rng, case["jobs"], n)), "status": None}
    weight = _state_vector(circ).abs().square().cpu().reshape((2,) * n)
    values = []
    for i, j in _pairs(rng, case["jobs"], n):
        w = weight.sum([a for a in range(n) if a not in (i, j)])
        values.append((w[0, 0] - w[0, 1] - w[1, 0] + w[1, 1]).to(torch.complex128))
    return {"values": torch.stack(values), "status": None}
