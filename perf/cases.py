"""What is measured of this framework: calls as a user's program makes them,
through the Python binding of the C ABI, from the smallest graph to the
largest configuration.

Kinds of a case (``kind``):

* ``solve``: the whole machine (Alg. 1 / 2, or Alg. 3 / 4 with a pool) for a
  tick budget from fresh initialisations, then the best sets and the iterate;
* ``step``: plain projected momentum ascent from a given x (``init``,
  ``set_x``, ``step``), then the iterate, the momentum and the exact
  evaluation of the last rounded point;
* ``fb``: one training step on the differentiable f_B: forward, backward and
  an optimiser update;
* ``read``: the readouts of a given x and of given binary points: rounding,
  FP64 relaxed objective, exact integer evaluation.

Graph families (``family``): ``er`` member graphs G(n, p) packed into one
batch (``n_lo`` .. ``n_hi`` nodes each), ``sparse`` one large ER graph of a
mean degree, ``reg`` one random 3-regular graph, ``cl`` one Chung-Lu
power-law graph (exponent 2.5).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2605_06921_gb300 as mq

F32, BF16, F16 = mq.F32, mq.BF16, mq.F16
MIS, MAXCUT = mq.MIS, mq.MAXCUT

# hyperparameters of the two problems (the rows of the benchmark's workloads)
_HYPER = {
    MIS: dict(alpha=0.8, momentum=0.45, gamma=2.0, rho=0.6, t_gs=60, descent_cap=50, sigma=0.1),
    MAXCUT: dict(alpha=0.0025, momentum=0.8, lambda_=0.001, rho=0.8, t_gs=90, descent_cap=200, sigma=0.1),
}
_LAMBDA, _LR = 0.001, 0.001


def _er(name, kind, problem, graphs, n_lo, n_hi, p, batch, x, v, ticks, pool=0, init=1):
    return {"name": name, "kind": kind, "family": "er", "problem": problem, "graphs": graphs, "n_lo": n_lo,
            "n_hi": n_hi, "p": p, "batch": batch, "x": x, "v": v, "ticks": ticks, "pool": pool, "init": init}


def _one(name, kind, family, problem, n, degree, batch, x, v, ticks, signed=False):
    return {"name": name, "kind": kind, "family": family, "problem": problem, "n": n, "degree": degree,
            "signed": signed, "batch": batch, "x": x, "v": v, "ticks": ticks, "pool": 0, "init": 1}


def _fb(name, family, n, degree, batch, optimizer, signed=False):
    return {"name": name, "kind": "fb", "family": family, "n": n, "degree": degree, "signed": signed,
            "batch": batch, "optimizer": optimizer}


def listed():
    return [
        # the plain method: one small graph, one FP32 trajectory, 2000 ticks
        _er("mis_plain", "solve", MIS, 1, 200, 200, 0.05, 1, F32, F32, 2000, init=0),
        # a handful of small ragged graphs, plain steps: the smallest calls,
        # bound by launches and latency
        _er("cut_steps_small", "step", MAXCUT, 24, 30, 300, 0.1, 8, F32, F32, 32),
        # the batched MIS configuration: 512 uneven graphs, 16,384 BF16
        # trajectories, the whole machine
        _er("mis_batched_bf16", "solve", MIS, 512, 700, 800, 0.15, 32, BF16, BF16, 100),
        # the same batch in the plain FP32 storage, plain steps
        _er("mis_batched_f32_steps", "step", MIS, 512, 700, 800, 0.15, 32, F32, F32, 16),
        # the paper's ER shapes: few member graphs, many trajectories
        _er("er_mis_1000_100", "solve", MIS, 8, 1000, 1000, 0.1, 128, BF16, BF16, 200),
        # dense graphs, MaxCut, the shared top-K pool of pmQO
        _er("er_maxcut_1000_500_pool", "solve", MAXCUT, 8, 1000, 1000, 0.5, 128, BF16, BF16, 200, pool=8),
        # one large sparse graph, MaxCut, BF16
        _one("maxcut_regular_bf16", "solve", "reg", MAXCUT, 100_000, 3, 128, BF16, BF16, 100),
        # its +-1-weighted variant with FP32 momentum, plain steps
        _one("maxcut_signed_steps", "step", "reg", MAXCUT, 100_000, 3, 128, BF16, F32, 16, signed=True),
        # MIS at scale: ten million nodes, FP16
        _one("mis_scale_f16", "solve", "sparse", MIS, 10_000_000, 10.0, 16, F16, F16, 8),
        # training on the differentiable objective: power-law graph, FP32
        _fb("autograd_powerlaw", "cl", 1_000_000, 8.0, 64, "momentum"),
        # the same on a small graph with few columns, Adam
        _fb("autograd_small", "cl", 20_000, 8.0, 16, "adam"),
        # readouts of a batch: rounding, FP64 objective, exact evaluation
        _er("mis_readouts", "read", MIS, 64, 700, 800, 0.15, 32, BF16, BF16, 1),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    case = _draw(rng)
    del case["name"]
    return case


def _draw(rng):
    kind = rng.choice(["er", "er", "er", "one", "fb", "read"])
    x = rng.choice([F32, BF16, BF16, F16])
    v = rng.choice([F32, x])
    if kind in ("er", "read"):
        problem = rng.choice([MIS, MAXCUT])
        n_hi = int(_log(rng, 40, 1200))
        n_lo = max(20, int(n_hi * rng.uniform(0.5, 1.0)))
        p = round(min(0.5, max(4.0 / n_hi, _log(rng, 0.03, 0.5))), 4)
        batch = rng.choice([1, 4, 16, 32, 32, 64, 128])
        per = p * n_hi * n_hi * batch  # edge-updates of one member graph and tick
        graphs = max(1, min(512, int(_log(rng, 1, 512)), int(1.2e9 / per)))
        pool = rng.choice([0, 0, 4])
        if kind == "read":
            return _er("", "read", problem, min(graphs, 64), n_lo, n_hi, p, batch, x, v, 1)
        ticks = int(min(_log(rng, 20, 400), max(8, 1.2e11 / (per * graphs))))
        kind = rng.choice(["solve", "solve", "step"])
        return _er("", kind, problem, graphs, n_lo, n_hi, p, batch, x, v, ticks,
                   pool=pool if kind == "solve" else 0, init=rng.choice([0, 1]))
    if kind == "one":
        family = rng.choice(["reg", "sparse"])
        batch = rng.choice([16, 32, 64, 128])
        if family == "reg":
            n = 2 * int(_log(rng, 2_000, 60_000))
            problem, degree, signed = MAXCUT, 3, rng.random() < 0.5
        else:
            n = int(_log(rng, 20_000, 4_000_000))
            n = min(n, 80_000_000 // batch)
            problem, degree, signed = MIS, round(rng.uniform(4.0, 16.0), 1), False
        return _one("", rng.choice(["solve", "step"]), family, problem, n, degree, batch, x, v,
                    int(max(4, min(64, 4e7 / n))), signed=signed)
    batch = rng.choice([4, 16, 32, 64, 128])
    n = int(min(_log(rng, 2_000, 1_000_000), 64_000_000 // batch))
    family = rng.choice(["cl", "cl", "reg"])
    if family == "reg":
        return _fb("", "reg", n + n % 2, 3, batch, rng.choice(["momentum", "adam"]), signed=rng.random() < 0.5)
    return _fb("", "cl", n, round(rng.uniform(4.0, 12.0), 1), batch, rng.choice(["momentum", "adam"]))


# ------------------------------------------------------------------ graphs
class _Csr:
    """Host CSR arrays as the binding takes them."""

    def __init__(self, n, row_ptr, col_idx, weights=None, node_offsets=None):
        self.n, self.row_ptr, self.col_idx, self.weights = n, row_ptr, col_idx, weights
        self.node_offsets = np.array([0, n], dtype=np.int64) if node_offsets is None else node_offsets


def _gen(seed, salt):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * salt + seed)


def _sizes(case):
    rng = np.random.default_rng(10_000)  # the same sizes for every seed: outputs of one shape
    return [int(k) for k in rng.integers(case["n_lo"], case["n_hi"] + 1, size=case["graphs"])]


def _er_batch(case, seed):
    gen = _gen(seed, 1)
    offs, cols, counts = [0], [], []
    for n in _sizes(case):
        up = torch.triu(torch.rand((n, n), device="cuda", generator=gen) < case["p"], 1)
        a = up | up.t()
        counts.append(a.sum(1))
        cols.append((a.nonzero()[:, 1] + offs[-1]).to(torch.int32))
        offs.append(offs[-1] + n)
    row_ptr = torch.zeros(offs[-1] + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.cat(counts).cumsum(0)
    return _Csr(offs[-1], row_ptr.cpu().numpy(), torch.cat(cols).cpu().numpy(), None,
                np.array(offs, dtype=np.int64))


def _pairs(case, seed):
    """Endpoints of an undirected edge list (self loops and repeats included)."""
    n, gen = case["n"], _gen(seed, 2)
    if case["family"] == "reg":
        stubs = torch.randperm(3 * n, device="cuda", generator=gen) % n
        return stubs[0::2], stubs[1::2]
    m = int(n * case["degree"] / 2)
    if case["family"] == "sparse":
        return (torch.randint(0, n, (m,), device="cuda", generator=gen),
                torch.randint(0, n, (m,), device="cuda", generator=gen))
    w = torch.arange(1, n + 1, dtype=torch.float64, device="cuda") ** (-1.0 / 1.5)
    cdf = w.cumsum(0)
    cdf /= cdf[-1].clone()
    u, v = (torch.searchsorted(cdf, torch.rand(m, dtype=torch.float64, device="cuda", generator=gen), right=True)
            .clamp_(max=n - 1) for _ in range(2))
    return u, v


def _edge_list_graph(case, seed):
    n = case["n"]
    u, v = _pairs(case, seed)
    lo, hi = torch.minimum(u, v), torch.maximum(u, v)
    key = torch.unique((lo * n + hi)[lo != hi])
    lo, hi = key // n, key % n
    key, order = torch.sort(torch.cat([lo * n + hi, hi * n + lo]))
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    row_ptr[1:] = torch.bincount(key // n, minlength=n).cumsum(0)
    weights = None
    if case.get("signed"):
        w = torch.randint(0, 2, (lo.numel(),), device="cuda", generator=_gen(seed, 3)) * 2 - 1
        weights = torch.cat([w, w])[order].to(torch.int8).cpu().numpy()
    return _Csr(n, row_ptr.cpu().numpy(), (key % n).to(torch.int32).cpu().numpy(), weights)


def _graph(case, seed):
    return _er_batch(case, seed) if case["family"] == "er" else _edge_list_graph(case, seed)


def _shape(case):
    """Expected (nodes, CSR entries, member graphs)."""
    if case["family"] == "er":
        n = 0.5 * (case["n_lo"] + case["n_hi"])
        return case["graphs"] * n, case["graphs"] * case["p"] * n * n, case["graphs"]
    return case["n"], case["n"] * case["degree"], 1


# ------------------------------------------------------------------ inputs
_DTYPE = {F32: torch.float32, BF16: torch.bfloat16, F16: torch.float16}


def _x0(case, n, seed):
    """Points of the box as a descent meets them: most coordinates at a bound
    after the projection, the rest inside."""
    lo = 0.0 if case["problem"] == MIS else -1.0
    gen = _gen(seed, 4)
    x = torch.randn((n, case["batch"]), device="cuda", generator=gen) * 0.6 + (0.1 if lo == 0.0 else 0.0)
    return x.clamp_(lo, 1.0).to(_DTYPE[case["x"]])


def _bits(case, n, seed):
    """Binary points, node-major bit words; for MIS about 5 % of the nodes set."""
    words = (case["batch"] + 31) // 32
    gen = _gen(seed, 5)
    z = torch.rand((n, words * 32), device="cuda", generator=gen) < (0.05 if case["problem"] == MIS else 0.5)
    z[:, case["batch"]:] = False
    shift = torch.arange(32, device="cuda", dtype=torch.int64)
    w = (z.view(n, words, 32).to(torch.int64) << shift).sum(-1)
    return torch.where(w >= 2 ** 31, w - 2 ** 32, w).to(torch.int32).reshape(-1)


def _solver(case, seed, graph):
    p = mq.params(problem=case["problem"], batch=case["batch"], x_dtype=case["x"], v_dtype=case["v"],
                  init_kind=case["init"], seed=seed, pool_k=case["pool"], **_HYPER[case["problem"]])
    return mq.Solver(graph, p)


def _fb_x(case, seed):
    return torch.rand((case["n"], case["batch"]), device="cuda", generator=_gen(seed, 6)) * 2 - 1


def prepare(case, seed):
    csr = _graph(case, seed)
    graph = mq.Graph(csr)
    if case["kind"] == "fb":
        x = _fb_x(case, seed).requires_grad_(True)
        opt = (mq.PGAMomentum([x], lr=_LR, momentum=0.9) if case["optimizer"] == "momentum"
               else mq.PGAAdam([x], lr=_LR))
        return {"case": case, "graph": graph, "x": x, "opt": opt}
    state = {"case": case, "graph": graph, "solver": _solver(case, seed, graph)}
    if case["kind"] in ("step", "read"):
        state["x0"] = _x0(case, csr.n, seed)
    if case["kind"] == "read":
        state["bits"] = _bits(case, csr.n, seed)
        state["solver"].set_x(state["x0"])
    return state


# ------------------------------------------------------------------ one pass
def run(state):
    case = state["case"]
    if case["kind"] == "fb":
        x, opt = state["x"], state["opt"]
        opt.zero_grad(set_to_none=True)
        obj = mq.FbObjective.apply(x, state["graph"], _LAMBDA)
        obj.sum().backward()
        opt.step()
        return {"objective": obj.detach(), "grad": x.grad, "x": x.detach(), "state": opt.state[x][
            "v" if case["optimizer"] == "momentum" else "m"]}
    s = state["solver"]
    if case["kind"] == "solve":
        s.solve(case["ticks"])
        values, bits = s.best()
        return {"values": values, "bits": bits, "x": s.get_x()}
    if case["kind"] == "step":
        s.init()
        s.set_x(state["x0"])
        s.step(case["ticks"])
        value, a, b = s.step_stats()
        return {"x": s.get_x(), "v": s.get_v(), "value": value, "a": a, "b": b}
    value, a, b = s.evaluate(state["bits"])
    return {"value": value, "a": a, "b": b, "objective": s.objective_f64(), "rounded": s.round()}


def work(case):
    """Bytes: graph, inputs and outputs once (a tick budget's iterates need not
    leave the chip).  Flops: per edge-update one multiply and one add, per
    element and tick about a dozen operations of the update."""
    n, nnz, graphs = _shape(case)
    B = case["batch"]
    index = 4.0 * nnz + 8.0 * n
    if case["kind"] == "fb":
        state = 2 if case["optimizer"] == "momentum" else 4  # optimiser buffers read and written
        return {"bytes": index + 4.0 * n * B * (3 + state), "flops": 2.0 * nnz * B * 2 + 12.0 * n * B}
    sx, sv = (4 if case["x"] == F32 else 2), (4 if case["v"] == F32 else 2)
    words = n * ((B + 31) // 32) * 4.0
    flops = case["ticks"] * (2.0 * nnz * B + 12.0 * n * B)
    if case["kind"] == "solve":
        return {"bytes": index + words + n * B * sx, "flops": flops}
    if case["kind"] == "step":
        return {"bytes": index + n * B * (2.0 * sx + sv), "flops": flops}
    return {"bytes": index + 2 * words + n * B * sx, "flops": 4.0 * nnz * B}


# ------------------------------------------------------------------ 64-bit values
def _matvec(csr):
    """x -> A x in float64 on the GPU (weights of +-1 included)."""
    n = csr.n
    rp = torch.from_numpy(csr.row_ptr).cuda()
    col = torch.from_numpy(csr.col_idx).cuda().to(torch.int64)
    w = torch.ones(col.numel(), dtype=torch.float64, device="cuda") if csr.weights is None else \
        torch.from_numpy(csr.weights).cuda().to(torch.float64)
    a = torch.sparse_csr_tensor(rp, col, w, size=(n, n))
    return lambda x: a @ x


def _per_graph(csr, node_values):
    """Sums of (n, B) node values over every member graph, flattened to G*B."""
    offs = torch.from_numpy(csr.node_offsets).cuda()
    total = torch.zeros((csr.n + 1, node_values.shape[1]), dtype=torch.float64, device="cuda")
    total[1:] = node_values.cumsum(0)
    return (total[offs[1:]] - total[offs[:-1]]).reshape(-1)


def exact(case, seed):
    if case["kind"] == "solve":
        return None  # integer decisions feed back into the iterate: no 64-bit value of a whole run
    csr = _graph(case, seed)
    ax = _matvec(csr)
    if case["kind"] == "fb":
        x = _fb_x(case, seed).double()
        y = ax(x)
        obj = -_LAMBDA * x.sum(0) - (x * y).sum(0)
        g = -_LAMBDA - 2.0 * y
        if case["optimizer"] == "momentum":
            v, step = g, _LR * g
        else:
            v = 0.1 * g
            step = _LR * g / (g.abs() + 1e-8)
        return {"objective": obj, "grad": g, "x": (x + step).clamp(-1.0, 1.0), "state": v}
    h = _HYPER[case["problem"]]
    x = _x0(case, csr.n, seed).double()
    if case["kind"] == "read":
        y = x * ax(x)
        node = x - 0.5 * h["gamma"] * y if case["problem"] == MIS else -h["lambda_"] * x - y
        return {"value": None, "a": None, "b": None, "objective": _per_graph(csr, node), "rounded": None}
    n, nnz, _ = _shape(case)
    if case["problem"] == MIS or nnz > 40 * n or case["ticks"] > 32:
        return None  # a step is of the box's size, or there are many: roundings decide which bound a node meets
    v = torch.zeros_like(x)
    for _ in range(case["ticks"]):
        v = h["momentum"] * v + h["alpha"] * (-h["lambda_"] - 2.0 * ax(x))
        x = (x + v).clamp(-1.0, 1.0)
    return {"x": x, "v": v, "value": None, "a": None, "b": None}
