"""The optimizer steps this framework is used for, as cases to be timed and compared.

A case is one parameter-server step through the public interface: the n workers compress
their gradients, the server decodes, averages, updates and emits the next broadcast.  A
case says how the parameter vector is made up, how many workers there are, where Adam's
moments live, which quantizers are on and which options are set.  Shapes, worker counts and
gradient distributions are those of the repository's workloads (qadam_inputs), its smoke
test and its benchmark, or generic.

    shape     a workload's tensor list ("resnet18_qg", "bert_base"), "flat" (one tensor of `d`
              elements) or "tensors" (`d` elements split unevenly into `tensors` tensors)
    placement "server": the workers quantize g + e, the server keeps m and v
              "worker": the workers keep m and v and quantize their update (Algorithm 3)
    kg, grid  gradient quantizer: level parameter (-1: none) and grid; kx: weight quantizer (-1: none)
    decay     factor of the l2 term; block: > 0, one gradient scale per block of that many elements
    feedback  an error buffer for the weight broadcast
    call      "step": gradients on the GPU; "host": gradients in pinned host memory, the packed
              broadcast (or x) read back
"""
from __future__ import annotations

import random

import torch

import paper_2004_14180_b200 as qb
from qadam_inputs import Workload, get_workload, gradients, initial_weights

GRIDS = {"pow2": qb.GRID_POW2, "uniform": qb.GRID_UNIFORM, "stochastic": qb.GRID_STOCHASTIC}
PLACEMENTS = {"server": qb.PLACE_SERVER, "worker": qb.PLACE_WORKER}
WARM_STEPS = 3                    # steps before the timed ones: a run in progress has errors and moments
BATCHES = 4                       # gradient batches a state alternates between ...
BATCH_BYTES = 1 << 30             # ... unless one takes more than this


def _case(name, shape, n, d=0, tensors=1, placement="server", kg=0, grid="pow2", kx=-1, decay=0.0,
          block=0, feedback=False, grad="mixture", call="step"):
    c = dict(shape=shape, d=d, tensors=tensors, n=n, placement=placement, kg=kg, grid=grid, kx=kx,
             decay=decay, block=block, feedback=feedback, grad=grad, call=call)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The smallest problem anyone steps: a few ragged tensors (the smoke test's sizes); launches
        # and latency are all there is.
        _case("ragged_13k_n4", "tensors", 4, d=13290, tensors=3, kx=0, grad="gauss_tensor"),
        # A small flat vector, gradient quantizer only: the first configuration of the benchmark.
        _case("flat_1m_n4", "flat", 4, d=1 << 20, grad="gauss_worker"),
        # A convolutional network's tensors with 8 workers, as in the paper's experiments: gradients
        # at the coarsest level, full-precision weights.
        _case("resnet18_n8", "resnet18_qg", 8, grad="gauss_tensor"),
        # The same network as the paper prints the method: moments on the workers, both quantizers
        # at the next level (3-bit codes).
        _case("resnet18_n8_workers_k1", "resnet18_qg", 8, placement="worker", kg=1, kx=1, grad="gauss_tensor"),
        # The same with the 8-bit weights of the paper's size tables and its weight decay.
        _case("resnet18_n8_8bit_decay", "resnet18_qg", 8, kx=6, decay=5e-4, grad="gauss_tensor"),
        # The stochastic ternary operator the paper compares with, on the same network.
        _case("resnet18_n8_stochastic", "resnet18_qg", 8, grid="stochastic", grad="gauss_tensor"),
        # A training loop whose gradients arrive in host memory.
        _case("resnet18_n8_host", "resnet18_qg", 8, kx=0, grad="gauss_tensor", call="host"),
        # A finer gradient grid and 16-bit weights on a vector of odd length with an odd number of workers.
        _case("flat_10m_n5_levels", "flat", 5, d=10_000_019, kg=3, grid="uniform", kx=14),
        # A transformer's tensors (many of them, one very large) with 16 workers, both quantizers.
        _case("bert_n16", "bert_base", 16, kx=0, grad="student_t_tensor"),
        # The same with the moments on the workers and weight decay.
        _case("bert_n16_workers_decay", "bert_base", 16, placement="worker", kx=0, decay=5e-4,
              grad="student_t_tensor"),
        # One large vector with one scale, moments on the workers.
        _case("flat_67m_n16_workers", "flat", 16, d=1 << 26, placement="worker", kx=0),
        # The benchmark's headline: the largest vector, 16 workers.
        _case("flat_268m_n16", "flat", 16, d=1 << 28, kx=0),
    ]


def draw(rng):
    """Another case of the same ranges: vectors of 10^4 to 2^28 elements, 1 to 32 workers, every
    quantizer, placement and option; at most 2^32 gradient elements a step (fewer where a step moves
    more bytes per element)."""
    placement = rng.choice(["server", "server", "worker"])
    kind = rng.choices(["ternary", "five", "pow2", "uniform", "stochastic", "none"], [50, 15, 10, 10, 10, 5])[0]
    kg = {"ternary": 0, "five": 1, "stochastic": 0, "none": -1}.get(kind) if kind not in ("pow2", "uniform") \
        else rng.choice([2, 3, 4])
    grid = kind if kind in ("uniform", "stochastic") else "pow2"
    kx = rng.choice([-1, 0, 0, 1, 6, 14])
    n = rng.choice([1, 2, 3, 4, 5, 6, 8, 8, 12, 16, 16, 24, 32])
    decay = 5e-4 if rng.random() < 0.25 else 0.0
    feedback = kx >= 0 and rng.random() < 0.1
    call = "host" if rng.random() < 0.06 else "step"
    most = 1 << 32 if placement == "server" and kind in ("ternary", "five") and decay == 0.0 else 1 << 30
    if call == "host":
        most = 1 << 26
    top = min(1 << 28, most // n)
    shape = rng.choices(["flat", "tensors", "resnet18_qg", "bert_base"], [40, 30, 15, 15])[0]
    for name in ("bert_base", "resnet18_qg"):
        if shape == name and get_workload(name).d > top:
            shape = "flat"
    d, tensors, block = 0, 1, 0
    if shape in ("flat", "tensors"):
        d = int(10 ** 4 * (top / 10 ** 4) ** rng.random())
        if rng.random() < 0.3:
            d = d // 4096 * 4096
    if shape == "tensors":
        tensors = rng.randint(2, 200)
        d = max(d, 50 * tensors)
    elif shape == "flat" and rng.random() < 0.25:
        block = 1 << rng.randint(12, 22)
        while d // block > 20000:
            block *= 2
    grad = rng.choice(["gauss_tensor", "student_t_tensor", "mixture"])
    return _case(None, shape, n, d=d, tensors=tensors, placement=placement, kg=kg, grid=grid, kx=kx,
                 decay=decay, block=block, feedback=feedback, grad=grad, call=call)


def _workload(case, seed):
    if case["shape"] == "flat":
        lens = (case["d"],)
    elif case["shape"] == "tensors":
        # sizes log-uniform over three decades, fixed by the case; the last tensor takes what is left
        rng = random.Random(case["d"] * 1000 + case["tensors"])
        parts = [10 ** (3 * rng.random()) for _ in range(case["tensors"])]
        lens = [max(1, int(case["d"] * p / sum(parts))) for p in parts]
        lens[-1] += case["d"] - sum(lens)
        lens = tuple(lens)
    else:
        base = get_workload(case["shape"])
        return base.with_(n=case["n"], grad=case["grad"], scale_block=case["block"], seed=seed)
    return Workload(case["shape"], lens, (0,) * len(lens), (False,) * len(lens), n=case["n"], steps=1,
                    grad=case["grad"], w0="gauss:0.05", scale_block=case["block"], seed=seed)


def prepare(case, seed):
    w = _workload(case, int(seed))
    q = qb.QAdam(w.scale_seg_len, w.n, kg=case["kg"], kx=case["kx"], placement=PLACEMENTS[case["placement"]],
                 grid_g=GRIDS[case["grid"]], beta1=w.beta1, beta2=w.beta2, eps=w.eps, lr=w.lr,
                 x1=initial_weights(w, device="cuda"), seed=int(seed), want_wfeedback=case["feedback"])
    if case["decay"]:
        q.set_regularization(case["decay"])
    host = case["call"] == "host"
    batches = BATCHES if 4 * w.n * q.D <= BATCH_BYTES else 1
    pool = []
    row = torch.empty(w.d, dtype=torch.float32, device="cuda")
    for b in range(batches):
        g = torch.empty(w.n, q.D, dtype=torch.float32, device="cuda")
        for i in range(w.n):
            g[i].copy_(q.to_padded(gradients(w, b + 1, i, device="cuda", out=row)))
        pool.append(g.cpu().pin_memory() if host else g)
    state = {"q": q, "g": pool, "step": 0, "host": host}
    if host:
        state["stage"] = torch.empty(w.n, q.D, dtype=torch.float32, device="cuda")
        state["back"] = (torch.empty(q.wcode_bytes, dtype=torch.uint8) if case["kx"] >= 0
                         else torch.empty(q.D, dtype=torch.float32)).pin_memory()
    for _ in range(WARM_STEPS):
        run(state)
    return state


def run(state):
    q = state["q"]
    state["step"] += 1
    t = state["step"]
    g = state["g"][t % len(state["g"])]
    if state["host"]:
        q.step_host(t, g, state["stage"], state["back"])
    else:
        q.step(t, g)
    out = {"codes": q.gcodes, "scales": q.scales, "e": q.e, "x": q.x, "m": q.m, "v": q.v}
    if q.kx >= 0:
        out["weights"] = q.wcodes
    if q.wfeedback is not None:
        out["feedback"] = q.wfeedback
    if state["host"]:
        out["back"] = state["back"]
    return out


def work(case):
    """Bytes: gradients and state read once, state, codes and the broadcast written once (the codes
    pass from the workers to the server, so reading them back is not counted).  Operations: those
    of the method as it is written down, per gradient element and per weight."""
    w = _workload(case, 0)
    nd, d = w.n * w.d, w.d
    gbits = qb.qadam_grad_code_bits(case["kg"], GRIDS[case["grid"]])
    xbits = qb.qadam_weight_code_bits(case["kx"])
    on_workers = case["placement"] == "worker"
    moved = nd * (12 + gbits / 8) + 4 * w.n * w.num_segments + d * (8 + xbits / 8)
    moved += nd * 16 if on_workers else d * 16                  # m, v read and written
    if case["decay"]:
        moved += d * xbits / 8 if case["kx"] >= 0 else 0        # the held weights
    if case["feedback"]:
        moved += 8 * d
    adam = 12                                                   # moments, root, division, step
    ops = nd * (8 + (adam if on_workers else 0)) + d * (4 + (0 if on_workers else adam))
    return {"bytes": float(moved), "flops": float(ops)}


def tolerance(case):
    """Every operation is one rounded binary32 operation in a stated order, so that a code next to a
    threshold falls the same way everywhere: results are the same bits."""
    return "exact"
