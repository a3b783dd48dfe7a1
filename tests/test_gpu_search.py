"""Alg. 2 on the GPU evaluator (emo_search_dp) against the oracle's search: the same chosen policy, time and
number of predictions, energy within 1e-9 relative."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2607_12324_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch_cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a GPU")
    return torch


@pytest.fixture(scope="module")
def emo():
    from paper_2607_12324_b200 import build, emo as E
    build.build()
    return E


def run_search(torch, emo, g, dev_of, breaks, p_idle, T_max, bin_ns, max_batch=0, flags=0, kernels=None):
    """kernels: those that one policy and a full batch outside a search run (emo_call_intervals)."""
    h = emo.load_workload(g, flags, group_of=np.asarray(dev_of, np.int32))
    assert kernels is None or kernels == (emo.emo_call_intervals(h, 1, breaks), emo.emo_call_intervals(h, max_batch or 16384, breaks))
    pi = torch.from_numpy(np.asarray(p_idle, np.float64)).cuda() if p_idle is not None else None
    ws = torch.empty(emo.emo_workspace_bytes_search(h, len(breaks), max_batch, p_idle is not None), dtype=torch.uint8, device="cuda")
    r = emo.emo_search_dp(h, breaks, pi, T_max, bin_ns, ws, max_batch=max_batch)
    h.free()
    return r


def compare(a, b):
    assert a["found"] == b["found"]
    if a["found"]:
        assert a["T"] == b["T"]
        assert np.isclose(a["E"], b["E"], rtol=1e-9, atol=0)
        assert a["F"].tolist() == b["F"].tolist()
    assert a["n_pred"] == b["n_pred"]


@pytest.mark.parametrize("seed", range(4))
def test_random_dags(torch_cuda, emo, oracle_mod, seed):
    from tests.test_oracle_intervals import _random_case
    g, dev_of, breaks, _, p_idle = _random_case(60 + seed, n=50, L=4, D=2, I=5, B=1)
    dev_of[0] = 0
    t0 = int(oracle_mod.intervals(g, dev_of, breaks, np.full((2, 5, 1), g.L - 1, np.uint8), p_idle)["makespan"][0])
    for slack, bin_ns, mb in ((0.0, 1, 0), (0.1, 1, 0), (0.3, 5, 0), (0.3, 1, 7), (-0.5, 1, 0)):
        T_max = int(t0 * (1 + slack))
        compare(run_search(torch_cuda, emo, g, dev_of, breaks, p_idle, T_max, bin_ns, mb),
                oracle_mod.search_dp(g, dev_of, breaks, p_idle, T_max, bin_ns))
    compare(run_search(torch_cuda, emo, g, dev_of, breaks, None, int(t0 * 1.2), 1),
            oracle_mod.search_dp(g, dev_of, breaks, None, int(t0 * 1.2), 1))


def test_config_graph(torch_cuda, emo, oracle_mod):
    g = W.make_graph("cfg0-tiny", 0.5)
    dev_of = W.device_of(g)
    t0 = int(oracle_mod.batch(g, np.full((g.n, 1), g.L - 1, np.uint8))["makespan"][0])
    breaks = W.interval_breaks(t0, 6)
    p_idle = W.idle_power(g.L)
    T_max = t0 + t0 // 20
    a = run_search(torch_cuda, emo, g, dev_of, breaks, p_idle, T_max, 1000)
    b = oracle_mod.search_dp(g, dev_of, breaks, p_idle, T_max, 1000)
    compare(a, b)
    assert a["found"] and a["T"] <= T_max


@pytest.mark.parametrize("seed", range(4))
def test_a_thread_per_policy(torch_cuda, emo, oracle_mod, seed):
    """The kernel that gives every policy a thread, with nodes that outlast intervals (a level that no node starts at makes candidates
    equal: the first stays) and batches that split a round."""
    from tests.test_gpu_walk import weave
    g, dev_of = weave(70 + seed, 60, 2)
    dev_of[:2] = 0, 1
    t0 = int(oracle_mod.intervals(g, dev_of, np.zeros(1, np.int64), np.full((2, 1, 1), g.L - 1, np.uint8), None)["makespan"][0])
    breaks = np.arange(6, dtype=np.int64) * (t0 // 5)
    for p_idle in (W.idle_power(g.L), None):
        for slack, bin_ns, mb in ((0.1, 1, 0), (0.3, 5, 0), (0.3, t0 // 50, 7), (1.0, t0 // 20, 33)):
            T_max = int(t0 * (1 + slack))
            compare(run_search(torch_cuda, emo, g, dev_of, breaks, p_idle, T_max, bin_ns, mb, emo.EMO_F_INTERVALS, (2, 2)),
                    oracle_mod.search_dp(g, dev_of, breaks, p_idle, T_max, bin_ns))


@pytest.mark.parametrize("max_batch", [6000, 11000])
def test_one_kernel_for_all_of_a_round(torch_cuda, emo, oracle_mod, max_batch):
    """Many lanes, a last round of several batches: its full batches by themselves would run another kernel than the rest of it.  The search
    compares the energies of all of them, so they come from one kernel: that of the chosen policy (in a full batch of 6 000, in the rest
    of 2 824 behind a batch of 11 000) is, bit for bit, what a full batch gives."""
    torch = torch_cuda
    g = W.make_graph("cfg3-8dev", 0.01)
    dev_of = W.device_of(g)
    t0 = int(oracle_mod.batch(g, np.full((g.n, 1), g.L - 1, np.uint8))["makespan"][0])
    breaks, p_idle, T_max = np.arange(3, dtype=np.int64) * (t0 // 3), W.idle_power(g.L), t0 + t0 // 4
    a = run_search(torch, emo, g, dev_of, breaks, p_idle, T_max, 1, max_batch, emo.EMO_F_INTERVALS, (1, 2))
    assert a["n_pred"] == 1 + 24 + 24 ** 2 + 24 ** 3
    compare(a, oracle_mod.search_dp(g, dev_of, breaks, p_idle, T_max, 1))
    h = emo.load_workload(g, emo.EMO_F_INTERVALS, group_of=dev_of)
    assert emo.emo_call_intervals(h, 24 ** 3 % 11000, breaks) == 1
    F = torch.from_numpy(np.asarray(a["F"], np.uint8)).cuda()[None, :, None].repeat(int(dev_of.max()) + 1, 1, 6000).contiguous()
    T, E = torch.zeros(6000, dtype=torch.int64, device="cuda"), torch.zeros(6000, dtype=torch.float64, device="cuda")
    ws = torch.empty(emo.emo_workspace_bytes_intervals(h, 6000, 3, True), dtype=torch.uint8, device="cuda")
    emo.emo_eval_intervals(h, 6000, F, 6000, 3, breaks, torch.from_numpy(p_idle).cuda(), T, E, None, ws)
    assert bool((E == a["E"]).all()) and bool((T == a["T"]).all())
    h.free()
