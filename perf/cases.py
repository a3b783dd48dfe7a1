"""Performance cases of the what-if evaluator: what a program that plans frequencies has it do, through the calls of
include/emo.h as the binding offers them, from one policy on a packed graph to 16 384 policies on a 250 000-node trace.

The graphs are the named configurations of the workloads module, whole or scaled down; the levels, features and interval
policies are drawn from the seed.
"""
import functools
import math

import numpy as np
import torch

from paper_2607_12324_b200 import emo, workloads

PACK_NS = 5_000_000            # granularity bound of a pack (Sec. 4.4)
INTERVAL_NS = 20_000_000       # re-assignment period of time-interval policies


def listed():
    return [
        # one policy looked at closely (a tool shows the slack of every kernel): the smallest call, nothing but latency
        dict(name="one_packed", kind="slack_one", config="cfg2-packed", scale=1.0),
        # the same on a long trace, after the search has picked a policy
        dict(name="one_llm", kind="slack_one", config="cfg4-llm", scale=1.0),
        # a handful of candidates on a small graph: a control loop between two iterations
        dict(name="slack_tiny", kind="slack", config="cfg0-tiny", scale=1.0, B=64, out="slack"),
        # a training iteration, every output of the two passes (earliest and latest starts, slack, sums, critical counts)
        dict(name="all_train", kind="slack", config="cfg1-train", scale=1.0, B=4096, out="all"),
        # many policies on a packed graph, then the selection under a budget
        dict(name="slack_packed", kind="slack", config="cfg2-packed", scale=1.0, B=65536, out="slack"),
        # eight device timelines joined by collectives
        dict(name="slack_8dev", kind="slack", config="cfg3-8dev", scale=1.0, B=8192, out="slack"),
        # the headline batch: 250 000 nodes, 16 384 policies, the slack matrix materialised
        dict(name="slack_llm", kind="slack", config="cfg4-llm", scale=1.0, B=16384, out="slack"),
        # forward pass only with one level per pack (group_of) and an uneven number of policies: a sampling search
        dict(name="eval_llm_packs", kind="eval", config="cfg4-llm", scale=0.3, B=10001, grouped=True),
        # time-interval policies with idle energy (Alg. 1 as printed)
        dict(name="intervals_llm", kind="intervals", config="cfg4-llm", scale=0.3, B=16384),
        # the policy search of Alg. 2: a chain of batches, each decided on the host
        dict(name="search_llm", kind="search", config="cfg4-llm", scale=0.1, delta_ppm=50_000),
        # levels in host memory, five bits each, one call from bytes on the host to results on the host
        dict(name="host_llm", kind="host", config="cfg4-llm", scale=0.1, B=8192, bits=5),
        # tables of all packs of a trace from their features (Sec. 4.5)
        dict(name="model_packs", kind="model", packs=14694, metrics=16, benchmarks=12, levels=32),
    ]


def _log_int(rng, lo, hi):
    """Whole number between lo and hi, even over the logarithm, odd ones included."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# nodes of the whole configurations (for the bound on a drawn case's size)
_NODES = {"cfg0-tiny": 400, "cfg1-train": 10_000, "cfg2-packed": 1_013, "cfg3-8dev": 128_039, "cfg4-llm": 250_000}


def draw(rng):
    kind = rng.choice(["slack_one", "slack", "slack", "eval", "intervals", "search", "host", "model"])
    if kind == "model":
        return dict(kind=kind, packs=_log_int(rng, 500, 200_000), metrics=rng.randint(12, 20), benchmarks=rng.randint(6, 12),
                    levels=rng.choice([8, 16, 24, 32]))
    if kind == "search":
        config = rng.choice(["cfg1-train", "cfg4-llm"])
        return dict(kind=kind, config=config, scale=round(rng.uniform(0.3, 1.0) if config == "cfg1-train" else rng.uniform(0.02, 0.1), 3),
                    delta_ppm=rng.choice([20_000, 30_000, 50_000]))
    if kind in ("host", "intervals"):
        config = rng.choice(["cfg1-train", "cfg4-llm"])
    else:
        config = rng.choice(sorted(_NODES))
    scale = 1.0 if config == "cfg0-tiny" else round(math.exp(rng.uniform(math.log(0.05), math.log(0.5))), 3)
    case = dict(kind=kind, config=config, scale=scale)
    if kind == "slack_one":
        return case
    # at most a tenth of the largest listed case's nodes x policies
    most = int(250_000 * 16_384 / 10 / (_NODES[config] * scale))
    case["B"] = _log_int(rng, 16, max(16, min(65_536, most)))
    if kind == "slack":
        case["out"] = rng.choice(["slack", "slack", "all"])
    if kind == "eval":
        case["grouped"] = config in ("cfg1-train", "cfg4-llm") and rng.random() < 0.5
    if kind == "host":
        case["bits"] = rng.choice([5, 8])
    return case


# ---- inputs ------------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _trace(config, scale):
    """The execution graph of a recorded workload: host arrays that a program has read from its trace."""
    return workloads.make_graph(config, scale)


@functools.lru_cache(maxsize=None)
def _packs(config, scale):
    """Pack of every kernel (policy row), -1 for the other nodes."""
    g = _trace(config, scale)
    is_kernel = (g.kind == workloads.KIND_KERNEL).astype(np.uint8)
    stream = g.meta["node_timeline"] * 64 + np.maximum(g.meta["node_stream"], 0)
    _, pack_of, n_packs = emo.emo_pack_greedy(g.n, g.row_ptr, g.col, is_kernel, stream, g.lat[:, -1], PACK_NS)
    return pack_of, n_packs


@functools.lru_cache(maxsize=None)
def _default_time(config, scale):
    """Makespan at the default frequency (one pass over the trace on the host), for the grid of change points."""
    g = _trace(config, scale)
    t, rp, col = g.lat[:, -1].tolist(), g.row_ptr.tolist(), g.col.tolist()
    done = [0] * g.n
    for v in range(g.n):
        done[v] = max([done[k] for k in col[rp[v]:rp[v + 1]]], default=0) + t[v]
    return max(done, default=0)


def _intervals(case):
    T0 = _default_time(case["config"], case["scale"])
    return workloads.interval_breaks(T0, max(2, int(T0 * 1.05) // INTERVAL_NS + 1))


def _levels(seed, rows, L, B, mode, q_max):
    """Level matrix [rows][pitch of 16] on the device, drawn from the seed."""
    ldb = (B + 15) // 16 * 16
    out = torch.zeros((rows, ldb), dtype=torch.uint8, device="cuda")
    step = max(1, (1 << 26) // B)
    for r0 in range(0, rows, step):
        r1 = min(rows, r0 + step)
        workloads.policy_levels(seed, rows, L, B, mode, q_max, rows=(r0, r1), device="cuda", out=out[r0:r1, :B])
    return out


def _workspace(nbytes):
    return torch.empty(max(nbytes, 1 << 16), dtype=torch.uint8, device="cuda")


def _vec(n, dtype):
    return torch.zeros(n, dtype=dtype, device="cuda")


def prepare(case, seed):
    kind = case["kind"]
    if kind == "model":
        P, L = case["packs"], case["levels"]
        Bm, Tb, Eb = workloads.microbench_model(1, case["metrics"], case["benchmarks"], L)
        feat = workloads.pack_features(seed, Bm, P)
        cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
        return dict(case=case, B=cu(Bm), Tb=cu(Tb), Eb=cu(Eb), feat=cu(feat), x=_vec((P, case["benchmarks"]), torch.float64),
                    T=_vec((P, L), torch.float64), E=_vec((P, L), torch.float64), status=_vec(1, torch.int32))
    g = _trace(case["config"], case["scale"])
    policy_seed = 1000 + seed
    if kind in ("intervals", "search"):
        # every device timeline has its own row of interval policies
        G = emo.load_workload(g, emo.EMO_F_INTERVALS, group_of=workloads.device_of(g))
        breaks = _intervals(case)
        I = len(breaks)
        s = dict(case=case, G=G, breaks=breaks, idle=torch.from_numpy(workloads.idle_power(g.L)).cuda())
        if kind == "search":
            # the seed chooses the period (up to a tenth shorter) and the budget (up to a tenth tighter): another plan for the same trace
            u = workloads.rand_uniform(policy_seed, 90, np.arange(2))
            s["breaks"] = np.arange(I, dtype=np.int64) * int(breaks[1] * (1.0 - 0.1 * u[0]))
            s["T_max"] = emo.emo_target_from_delta(_default_time(case["config"], case["scale"]), int(case["delta_ppm"] * (1.0 - 0.1 * u[1])))
            s["ws"] = _workspace(emo.emo_workspace_bytes_search(G, I, 0, True))
            return s
        B = case["B"]
        s["F"] = workloads.interval_policies(policy_seed, G.info.rows, I, g.L, B, device="cuda")
        s.update(T=_vec(B, torch.int64), E=_vec(B, torch.float64), E_idle=_vec(B, torch.float64),
                 ws=_workspace(emo.emo_workspace_bytes_intervals(G, B, I, True)))
        return s
    group_of, rows = None, g.n
    if case.get("grouped"):
        group_of, rows = _packs(case["config"], case["scale"])
    G = emo.load_workload(g, group_of=group_of)
    s = dict(case=case, G=G)
    if kind == "slack_one":
        s["lvl"] = _levels(policy_seed, rows, g.L, 64, "mixed", g.meta["q_max"])[:, 40].contiguous()
        for k in ("ES", "LS", "slack"):
            s[k] = _vec(g.n, torch.int64)
        s.update(T=_vec(1, torch.int64), E=_vec(1, torch.float64), ws=_workspace(emo.emo_workspace_bytes(G, 1, 1)))
        return s
    B = case["B"]
    lvl = _levels(policy_seed, rows, g.L, B, g.meta["policy_mode"], g.meta["q_max"])
    if kind == "host":
        bits = case["bits"]
        ldp = (B + 7) // 8 * bits if bits < 8 else lvl.shape[1]
        packed = torch.zeros((rows, ldp), dtype=torch.uint8, device="cuda")
        if bits < 8:
            emo.emo_pack_levels(bits, rows, B, lvl, lvl.shape[1], packed, ldp)
        else:
            packed.copy_(lvl)
        s["host"] = torch.empty((rows, ldp), dtype=torch.uint8, pin_memory=True)
        s["host"].copy_(packed)
        s.update(packed=packed, lvl=torch.zeros_like(lvl), slack=_vec((g.n, B), torch.int64),
                 T=torch.zeros(B, dtype=torch.int64, pin_memory=True), E=torch.zeros(B, dtype=torch.float64, pin_memory=True),
                 sel=torch.zeros(4, dtype=torch.int64), ws=_workspace(emo.emo_workspace_bytes(G, B, 2)))
        s["packed"].zero_()
        return s
    s["lvl"] = lvl
    s.update(T=_vec(B, torch.int64), E=_vec(B, torch.float64), T0=_vec(1, torch.int64), E0=_vec(1, torch.float64),
             index=_vec(1, torch.int64), sel_T=_vec(1, torch.int64), sel_E=_vec(1, torch.float64))
    if kind == "slack":
        s["slack"] = _vec((g.n, B), torch.int64)
        if case["out"] == "all":
            s.update(ES=_vec((g.n, B), torch.int64), LS=_vec((g.n, B), torch.int64), sums=_vec(B, torch.int64), critical=_vec(B, torch.int32))
        s["ws"] = _workspace(emo.emo_workspace_bytes(G, B, 1))
    else:
        s["ws"] = _workspace(emo.emo_workspace_bytes(G, B, 0))
    return s


# ---- one pass ----------------------------------------------------------------------------------------------
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "model":
        emo.emo_pack_model(case["packs"], case["metrics"], case["benchmarks"], case["levels"], s["B"], s["feat"], s["Tb"], s["Eb"], s["x"],
                           s["T"], s["E"], status=s["status"])
        return {k: s[k] for k in ("x", "T", "E", "status")}
    G = s["G"]
    if kind == "slack_one":
        emo.emo_slack(G, s["lvl"], s["ES"], s["LS"], s["slack"], s["T"], s["E"], ws=s["ws"])
        return {k: s[k] for k in ("ES", "LS", "slack", "T", "E")}
    if kind == "search":
        r = emo.emo_search_dp(G, s["breaks"], s["idle"], s["T_max"], 1_000_000, s["ws"])
        return {k: r[k] for k in ("found", "F", "T", "E", "n_pred")}
    B = case["B"]
    if kind == "intervals":
        emo.emo_eval_intervals(G, B, s["F"], s["F"].shape[2], len(s["breaks"]), s["breaks"], s["idle"], s["T"], s["E"], s["E_idle"], s["ws"])
        return {k: s[k] for k in ("T", "E", "E_idle")}
    if kind == "host":
        emo.emo_slack_batch_host_packed(G, B, case["bits"], s["host"], s["host"].shape[1], s["packed"], s["lvl"], s["lvl"].shape[1],
                                        s["slack"], B, 50_000, s["T"], s["E"], None, None, s["sel"], s["ws"])
        return {"slack": s["slack"], "T": s["T"], "E": s["E"], "selected": s["sel"][:2], "T0": s["sel"][3:]}
    out = ["T", "E", "T0", "E0", "index", "sel_T", "sel_E"]
    if kind == "slack":
        emo.emo_slack_batch(G, B, s["lvl"], s["lvl"].shape[1], s.get("ES"), s.get("LS"), s["slack"], B, s["T"], s["E"], s.get("sums"),
                            s.get("critical"), ws=s["ws"], T0=s["T0"], E0=s["E0"])
        out += [k for k in ("slack", "ES", "LS", "sums", "critical") if k in s]
    else:
        emo.emo_eval_policies(G, B, s["lvl"], s["lvl"].shape[1], s["T"], s["E"], ws=s["ws"], T0=s["T0"], E0=s["E0"])
    emo.emo_select(B, s["T"], s["E"], 0, s["index"], s["sel_T"], s["sel_E"], ws=s["ws"], target_dev=s["T0"], delta_ppm=50_000)
    return {k: s[k] for k in out}


def work(case):
    """Bytes: levels, tables, edges and outputs once.  Operations: per node and policy the table sums, per edge the maximum."""
    if case["kind"] == "model":
        P, n, m, L = (case[k] for k in ("packs", "metrics", "benchmarks", "levels"))
        # features in; weights and tables out.  One projection (2nm), one triangular solve of full size, the two table sums.
        return {"bytes": 8 * P * (n + m + 2 * L), "flops": P * (2 * n * m + m ** 3 // 3 + 2 * m * m + 4 * m * L)}
    g = _trace(case["config"], case["scale"])
    graph = g.n * g.L * 12 + g.m * 4 + g.n * 8
    if case["kind"] == "slack_one":
        return {"bytes": graph // g.L + g.n * (1 + 24) + 16, "flops": 2 * (g.n + g.m) + 3 * g.n}
    if case["kind"] in ("intervals", "search"):
        rows, I = int(workloads.device_of(g).max()) + 1, len(_intervals(case))
        if case["kind"] == "search":
            B = I * g.L          # at least every level of every interval once
            return {"bytes": graph + B * (rows * I + 16), "flops": B * (2 * g.n + g.m)}
        return {"bytes": graph + case["B"] * (rows * I + 24), "flops": case["B"] * (2 * g.n + g.m)}
    B = case["B"]
    rows = _packs(case["config"], case["scale"])[1] if case.get("grouped") else g.n
    lvl = rows * B if case["kind"] != "host" or case["bits"] == 8 else rows * (B + 7) // 8 * case["bits"]
    if case["kind"] == "eval":
        return {"bytes": graph + lvl + 16 * B, "flops": B * (2 * g.n + g.m)}
    outs = 3 if case.get("out") == "all" else 1
    return {"bytes": graph + lvl + outs * 8 * g.n * B + 16 * B, "flops": B * (2 * (g.n + g.m) + 3 * g.n)}


def tolerance(case):
    """Times, slacks, levels and indices are whole numbers and exact.  Energies are fp64 sums of up to 250 000 terms: summed
    one by one in node order they differ by 4.7e-15 (75 000 nodes; two and a half times that for the largest graph by a
    random walk of roundings).  The packs' weights come from fp64 normal equations, 1.9e-15 from an active-set solver that
    works on the metric matrix itself; its condition number is 16, so another correct solver may lose 270 roundings."""
    return {"rel": 1e-13}
