"""What is timed: the work that a program which selects parallel strategies has this library do.

A case says where the search tables come from (`source`), through which entry point the work goes (`entry`), which
tables are kept (`table`), and the sizes: B instances of at most L layers, S strategies, M memory bins.

source  "model"   the analytic cost model: a layer stack, a strategy table, per-instance rates
        "tables"  integer tables as a profiler measured them: nothing is known about their structure
entry   "step"    cost model (or given tables) -> search -> plan on device buffers (SearchBuffers.step)
        "host"    the same from pinned host buffers to host plans (HostSearch.run)
        "graph"   new rates copied in, then one replay of the captured step
        "switch"  the monitoring loop of a running job: re-evaluate, price the running plan, search with the price of
                  leaving it, decide
        "stages"  one instance per start layer, the optimum of every layer range, balanced pipeline stages
        "costs"   the cost model alone
table   "full"    every cell of C        "argmin"  the argmin table in its place      "none"  the optimum only

`draw` spreads the same kinds over their ranges.  Strategy counts follow from the axes: tensor-parallel degrees up to
the GPUs of a stage, 1 to 4 ZeRO stages, checkpointing on or off, sequence parallelism where it is considered;
`drop` takes single strategies out, as a program does that knows some to be unusable.
"""
import math

import numpy as np
import torch

from paper_2504_03662_b200 import binding as gb
from paper_2504_03662_b200 import inputs
from paper_2504_03662_b200.search import HostSearch, SearchBuffers, _dev_bytes

# layer kinds in turn, hidden size, sequence length, heads
STACKS = {
    "gpt": (("full",), 2048.0, 2048.0, 16.0),
    "175b": (("full",), 12288.0, 2048.0, 96.0),
    "hetero": (("attention", "ffn"), 8192.0, 4096.0, 64.0),
}
ZEROS = {1: (0,), 2: (0, 3), 3: (0, 2, 3), 4: (0, 1, 2, 3)}
PIPELINES = (1, 2, 4, 8, 16, 32, 64, 96)
TABLE_FLAGS = {"full": gb.STORE_C_FULL, "argmin": gb.STORE_ARGMIN, "none": 0}
TIME_MEDIAN = 5e5                 # measured tables: median layer time in ns


def _model(name, entry, stack, B, L, M, bin_mib, **kw):
    c = {"name": name, "entry": entry, "source": "model", "stack": stack, "B": B, "L": L, "M": M, "bin_mib": bin_mib, "gpus": 8, "zeros": 3,
         "sp": 1, "drop": 0, "b_max": 1, "pp": 1, "ragged": False, "table": "full"}
    c.update(kw)
    return c


def _tables(name, B, L, S, M, table, **kw):
    c = {"name": name, "entry": "step", "source": "tables", "B": B, "L": L, "S": S, "M": M, "table": table, "ragged": False, "per_layer": False,
         "trans_share": 0.1}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: a handful of measured layers and strategies; launches and the host path are all there is
        _tables("tiny_tables", 1, 4, 6, 64, "full", trans_share=0.05),
        # one running job looks at its own plan again: a single uniform decoder, 24 strategies, 180 GiB in 64 MiB bins
        _model("monitor_gpt", "switch", "gpt", 1, 24, 2880, 64, sp=0, b_max=16),
        # the same loop at one host call: half of a large decoder (two pipeline stages), rates of this minute, graph replay
        _model("replay_175b", "graph", "175b", 1, 48, 2880, 64, pp=2),
        # which micro-batch: sixteen candidates of the small decoder
        _model("sweep_micro_batch_gpt", "step", "gpt", 16, 24, 2880, 64, sp=0, b_max=16),
        # which micro-batch and pipeline degree: 64 candidates of the large decoder, 1 to 96 layers a stage, and the choice
        _model("sweep_pipeline_175b", "step", "175b", 64, 96, 2880, 64, b_max=8, ragged=True),
        # a long alternating stack under 64 measured rate pairs, all tables kept for later queries
        _model("hetero_full", "step", "hetero", 64, 160, 8192, 16, zeros=4),
        # the largest batch of it, optima only: what an outer loop over candidates asks
        _model("hetero_optima", "step", "hetero", 128, 160, 8192, 16, zeros=4, table="none"),
        # the largest call: the same batch from host descriptors to host plans
        _model("hetero_host", "host", "hetero", 128, 160, 8192, 16, zeros=4),
        # a thousand re-searches on measured tables: dense transition costs without any structure
        _tables("research_sweep", 1024, 48, 32, 2048, "full"),
        # measured transitions per layer, plans from the one-byte table, odd sizes
        _tables("argmin_per_layer", 96, 40, 44, 3001, "argmin", per_layer=True, ragged=True),
        # how to cut a 48-layer decoder into stages: every suffix of it searched, optima of all ranges
        _model("stages_gpt", "stages", "gpt", 48, 48, 2880, 64, sp=0, b_max=1, pp=8),
        # the cost model on its own over many measured rates
        _model("costs_bulk", "costs", "hetero", 8192, 160, 8192, 16, zeros=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    if rng.random() < 0.4:
        S, M, L = _log(rng, 5, 96), _log(rng, 60, 6000), _log(rng, 3, 96)
        # at most half of research_sweep's relaxations; the tables fit well below its 13 GB
        B = _log(rng, 1, max(1, min(1024, int(5e10 / (L * (M + 1) * S * S)), int(2.5e9 / (L * (M + 32) * S)))))
        per_layer = rng.random() < 0.25
        return {k: v for k, v in _tables("", B, L, S, M, rng.choice(("full", "full", "argmin", "none")), ragged=rng.random() < 0.4,
                                         per_layer=per_layer, trans_share=round(math.exp(rng.uniform(math.log(0.01), math.log(0.3))), 4)).items() if k != "name"}
    entry = rng.choice(("step", "step", "step", "host", "graph", "switch", "stages", "costs"))
    stack = rng.choice(tuple(STACKS))
    M, bin_mib = rng.choice(((2880, 64), (8192, 16), (rng.randrange(1200, 6000), 32)))
    zeros, sp = rng.choice((1, 2, 3, 4)), rng.choice((0, 1))
    gpus = rng.choice((4, 8, 8, 16))
    c = _model("", entry, stack, 1, _log(rng, 6, 160), M, bin_mib, gpus=gpus, zeros=zeros, sp=sp, pp=rng.choice((1, 2, 4, 8)), b_max=rng.choice((1, 2, 4, 8, 16)))
    del c["name"]
    c["drop"] = rng.choice((0, 0, rng.randrange(1, 4)))
    S = _strategies(c)
    if entry == "costs":
        c["B"] = _log(rng, 16, max(16, min(8192, int(8e7 / (c["L"] * S)))))
    elif entry == "stages":
        c["L"] = c["B"] = _log(rng, 12, 64)
    elif entry in ("step", "host"):
        c["table"] = rng.choice(("full", "full", "argmin", "none")) if entry == "step" else "full"
        c["B"] = _log(rng, 1, max(1, min(256, int(3e9 / (c["L"] * (M + 32) * S)))))
        c["ragged"] = entry == "step" and rng.random() < 0.4
    return c


# ------------------------------------------------------------------ inputs

def _degrees(case):
    return tuple(1 << k for k in range(int(math.log2(case["gpus"])) + 1))


def _strategies(case):
    if case["source"] == "tables":
        return case["S"]
    return len(_degrees(case)) * len(ZEROS[case["zeros"]]) * 2 * (2 if case["sp"] else 1) - case["drop"]


def _unit_ns(stack, b, L):
    """Nanoseconds per integer time unit, a power of ten that keeps a path sum over L layers well below 2^30."""
    kinds, h, seq, _ = STACKS[stack]
    worst = 0.0
    for k in kinds:
        c_lin, c_attn, p_coef, n_ar = inputs._KIND[k][:4]
        t = 4.0 * b * seq * h * (c_lin * h + c_attn * seq) / 0.8e15 + (2.0 * n_ar * b * seq * h * 2.0 + 3.0 * p_coef * h * h * 2.0 + 2.0 * b * seq * h * 2.0) / 360e9
        worst = max(worst, t)
    unit = 1.0
    while worst * L * 1e9 / unit > 2.0 ** 29:
        unit *= 10.0
    return unit


def _rates(w, rng):
    """Measured rates of every instance: compute and link within 20 % of the nominal ones."""
    u = rng.random((w.B, 2))
    w.inst["flops_rate"] = 1e15 * (0.8 + 0.4 * u[:, 0])
    w.inst["bw_tp"] = w.inst["bw_dp"] = 450e9 * (0.8 + 0.4 * u[:, 1])


def _model_workload(case, rng):
    kinds, h, seq, heads = STACKS[case["stack"]]
    B, L = case["B"], case["L"]
    layers = np.empty((1, L), inputs.LAYER_DESC)
    for l in range(L):
        layers[0, l] = inputs.layer_desc(kinds[l % len(kinds)], h, seq, heads)
    strat = inputs.strategy_table(_degrees(case), ZEROS[case["zeros"]], (0, 1), (0, 1) if case["sp"] else (0,), case["gpus"])
    if case["drop"]:
        gone = np.random.default_rng(case["drop"]).choice(len(strat), case["drop"], replace=False)
        strat = np.ascontiguousarray(np.delete(strat, gone))
    pp = np.full(B, float(case["pp"]))
    b = 1.0 + (np.arange(B) % case["b_max"]) if B > 1 else np.full(1, float(case["b_max"]))
    Ls = np.full(B, L, np.int32)
    if case["ragged"]:                                       # a stage of every pipeline degree: ceil(L / pp) layers, pp micro-batches in flight
        pp = np.array([PIPELINES[i % 8] for i in range(B)], np.float64)
        b = 1.0 + (np.arange(B) // 8) % case["b_max"]
        Ls = np.ceil(L / pp).astype(np.int32)
    if case["entry"] == "stages":                            # instance a: layers a, a+1, ...
        rows = np.repeat(layers, B, 0)
        for a in range(B):
            rows[a, :L - a] = layers[0, a:]
        layers, Ls = rows, (L - np.arange(B)).astype(np.int32)
    inst = inputs._inst(B, b=b, act_mult=pp, bin_bytes=case["bin_mib"] * 2.0 ** 20, time_unit_ns=_unit_ns(case["stack"], float(b.max()), L))
    w = inputs.Workload(case["stack"], B, L, len(strat), case["M"], Ls, layers=layers, strat=strat, inst=inst, meta={"pp": pp, "b": b})
    _rates(w, rng)
    if case["entry"] == "stages":                            # one model: every suffix under the same rates
        for f in ("flops_rate", "bw_tp", "bw_dp"):
            w.inst[f] = w.inst[f][0]
    return w


def _table_workload(case, rng):
    """Log-normal layer times around half a millisecond, memory of a few percent of the budget, dense transitions."""
    B, L, S, M = case["B"], case["L"], case["S"], case["M"]
    time = np.maximum(1, np.rint(TIME_MEDIAN * np.exp(0.5 * rng.standard_normal((B, L, S), np.float32)))).astype(np.int32)
    lo, hi = max(1, M // (6 * L)), max(2, 3 * M // L)        # on average a plan has to choose: the budget is neither empty nor free
    mem = rng.integers(lo, hi + 1, (B, L, S), np.int32)
    mats = (B, L, S, S) if case["per_layer"] else (B, S, S)
    trans = rng.integers(0, int(TIME_MEDIAN * case["trans_share"]) + 1, mats, np.int32)
    Ls = rng.integers(max(1, L // 3), L + 1, B).astype(np.int32) if case["ragged"] else np.full(B, L, np.int32)
    return inputs.Workload("tables", B, L, S, M, Ls, time, mem, trans)


def _workload(case, seed):
    rng = np.random.default_rng(seed)
    return _model_workload(case, rng) if case["source"] == "model" else _table_workload(case, rng)


_galv = None


def _library():
    """The one library context of this process."""
    global _galv
    if _galv is None:
        _galv = gb.Galv(torch.cuda.current_device())
    return _galv


def _plan_outputs(sb):
    out = {"opt_cost": sb.opt_cost, "plan": sb.plan, "mem_used": sb.mem_used, "status": sb.status, "C_last": sb.C_last}
    if sb.C is not None:
        out["C"] = sb.C
    if sb.A is not None:
        out["A"] = sb.A
    if sb.w.has_model:
        out.update(time_q=sb.time_q, mem_q=sb.mem_q, trans_q=sb.trans_q)
    return out


class _State:
    graph = None

    def __del__(self):
        if self.graph is not None:
            self.galv.galv_graph_destroy(self.graph)


def prepare(case, seed):
    galv = _library()
    w = _workload(case, seed)
    s = _State()
    s.case, s.galv, s.w = case, galv, w
    if case["entry"] == "host":
        s.host = HostSearch(galv, w, TABLE_FLAGS[case["table"]])
        return s
    dev = torch.device("cuda", galv.device)
    if case["entry"] == "costs":
        i32 = dict(dtype=torch.int32, device=dev)
        s.shape = gb.make_shape(w.B, w.Lmax, w.S, w.M, 0)
        s.L = torch.from_numpy(w.L).to(dev)
        s.layers, s.strat, s.inst = _dev_bytes(w.layers, dev), _dev_bytes(w.strat, dev), _dev_bytes(w.inst, dev)
        s.out = {"time_q": torch.empty(w.B, w.Lmax, w.S, **i32), "mem_q": torch.empty(w.B, w.Lmax, w.S, **i32),
                 "trans_q": torch.empty(w.B, w.S, w.S, **i32), "status": torch.empty(w.B, **i32)}
        return s
    s.sb = sb = SearchBuffers(galv, w, TABLE_FLAGS[case["table"]])
    if int(w.L.min()) < w.Lmax:                              # layers an instance does not have are never written
        for t in (sb.C, sb.A):
            if t is not None:
                t.zero_()
    i32 = dict(dtype=torch.int32, device=dev)
    if case["entry"] == "graph":
        s.new_inst = torch.from_numpy(w.inst.view(np.uint8).copy()).pin_memory()
        s.stream = torch.cuda.Stream()
        s.graph = galv.galv_graph_create(sb.shape, sb.L, sb.layers, sb.layer_stride_B, sb.strat, sb.inst, sb.time_q, sb.mem_q, sb.trans_q,
                                         sb.C, sb.A, sb.C_last, sb.workspace, None, sb.opt_cost, sb.plan, sb.mem_used, sb.status,
                                         s.stream.cuda_stream)
    elif case["entry"] == "switch":
        plan = np.random.default_rng(seed + 1).integers(0, w.S, (w.B, w.Lmax)).astype(np.int32)
        s.running = torch.from_numpy(plan).to(dev)
        s.horizon = torch.full((w.B,), 200, **i32)
        s.amended = torch.empty_like(sb.time_q)
        s.cost, s.mem = (torch.empty(w.B, dtype=torch.int64, device=dev) for _ in range(2))
        s.decision = torch.empty(w.B, **i32)
    elif case["entry"] == "stages":
        s.P = min(case["pp"], w.Lmax)
        s.opt_l = torch.empty(w.B, w.Lmax, **i32)
        s.cuts, s.bottleneck = torch.empty(s.P + 1, **i32), torch.empty(1, **i32)
    elif case["ragged"] and w.has_model:                     # the outer choice: 256 sequences a global batch
        s.n_micro = torch.from_numpy(np.maximum(1, 256 // w.meta["b"]).astype(np.int32)).to(dev)
        s.pp = torch.from_numpy(w.meta["pp"].astype(np.int32)).to(dev)
        s.group = torch.zeros(w.B, **i32)
        s.best_time, s.best_inst = torch.empty(1, dtype=torch.int64, device=dev), torch.empty(1, **i32)
    return s


def run(s):
    entry = s.case["entry"]
    if entry == "host":
        return s.host.run()
    if entry == "costs":
        s.galv.galv_eval_costs(s.shape, s.L, s.layers, 0, s.strat, s.inst, None, None, s.out["time_q"], s.out["mem_q"], s.out["trans_q"], s.out["status"])
        return s.out
    sb = s.sb
    if entry == "graph":
        sb.inst.copy_(s.new_inst, non_blocking=True)
        s.galv.galv_graph_launch(s.graph)
        return _plan_outputs(sb)
    if entry == "switch":
        sb.eval_costs()
        s.galv.galv_plan_cost(sb.shape, sb.L, sb.time_q, sb.mem_q, sb.trans_q, s.running, s.cost, s.mem)
        s.galv.galv_add_switch_cost(sb.shape, sb.L, sb.time_q, sb.trans_q, s.running, s.horizon, s.amended)
        s.galv.galv_dp_search(sb.shape, sb.L, s.amended, sb.mem_q, sb.trans_q, sb.C, sb.A, sb.C_last, sb.workspace, sb.status)
        s.galv.galv_backtrack(sb.shape, sb.L, s.amended, sb.mem_q, sb.trans_q, sb.C, sb.A, sb.C_last, None, sb.opt_cost, sb.plan, sb.mem_used, sb.status)
        s.galv.galv_switch_decision(s.w.B, s.cost, sb.opt_cost, sb.status, 50, s.decision)
        return dict(_plan_outputs(sb), amended=s.amended, cost=s.cost, mem=s.mem, decision=s.decision)
    sb.step()
    out = _plan_outputs(sb)
    if entry == "stages":
        s.galv.galv_layer_optima(sb.shape, sb.L, sb.C, None, sb.status, s.opt_l)
        s.galv.galv_stage_partition(s.w.Lmax, s.P, s.opt_l, s.cuts, s.bottleneck)
        out.update(opt_l=s.opt_l, cuts=s.cuts, bottleneck=s.bottleneck)
    elif hasattr(s, "best_time"):
        s.galv.galv_select_best(s.w.B, 1, sb.opt_cost, sb.status, s.n_micro, s.pp, s.group, s.best_time, s.best_inst)
        out.update(best_time=s.best_time, best_inst=s.best_inst)
    return out


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    """Bytes: descriptors or tables read once, results and kept tables written once.  Operations: one addition and one
    minimum per cell of the recurrence's table (how many of the S candidates of a cell have to be looked at depends on
    the data), a few dozen per element of the cost model."""
    w_L = case["L"]
    B, S, M = case["B"], _strategies(case), case["M"]
    P = (M + 1 + 31) // 32 * 32
    if case["entry"] == "stages":
        layers = w_L * (w_L + 1) // 2
    elif case["ragged"]:
        layers = sum(-(-w_L // PIPELINES[i % 8]) for i in range(B)) if case["source"] == "model" else int(B * w_L * 2 / 3)
    else:
        layers = B * w_L
    elements = layers * S
    if case["source"] == "model":
        mats = B
        nbytes = 80 * w_L + 32 * S + 64 * B
        flops = 40 * elements
        if case["entry"] == "costs":
            return {"bytes": nbytes + 8 * elements + 4 * B * S * S, "flops": flops}
        if case["entry"] != "host":
            nbytes += 8 * elements + 4 * B * S * S           # the integer tables are results too
    else:
        mats = layers if case["per_layer"] else B
        nbytes = 8 * elements + 4 * mats * S * S
        flops = 0
    nbytes += 4 * B * (w_L + 3)
    flops += 2 * elements * (M + 1)
    if case["entry"] != "host":
        nbytes += 4 * B * S * P
        nbytes += {"full": 4, "argmin": 1, "none": 0}[case["table"]] * elements * P
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Whole numbers throughout: tables, costs, plans and decisions are exact."""
    return "exact"
