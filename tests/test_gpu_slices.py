"""The slice kernels (calls with few policies: the graph cut into slices that are evaluated at the same time) against the oracle:
graphs of one, two and many slices (chained one by one and by groups), tiles with remainders, every output."""
import os

import numpy as np
import pytest

from paper_2607_12324_b200 import workloads as W
from tests.test_gpu_parity import assert_matches, emo, gpu_slack_batch, torch_cuda  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def levels(torch, rows, L, B, seed, pitch=0):
    """[rows][ldb] with bytes that no policy owns behind the batch."""
    ldb = pitch or (B + 15) // 16 * 16
    lv = np.full((rows, ldb), 0xFF, dtype=np.uint8)
    lv[:, :B] = np.random.RandomState(seed).randint(0, L, size=(rows, B))
    return lv[:, :B].copy(), torch.as_tensor(lv, device="cuda")


@pytest.mark.parametrize("name, scale, B", [("cfg0-tiny", 1.0, 64), ("cfg1-train", 0.02, 1), ("cfg1-train", 0.026, 9), ("cfg1-train", 0.3, 8), ("cfg1-train", 0.6, 31),
                                            ("cfg2-packed", 0.25, 33), ("cfg2-packed", 1.0, 257), ("cfg3-8dev", 0.02, 17), ("cfg3-8dev", 0.1, 7), ("cfg4-llm", 0.05, 40)])
def test_against_oracle(torch_cuda, emo, oracle_mod, name, scale, B):
    torch = torch_cuda
    g = W.make_graph(name, scale)
    lv, lv_dev = levels(torch, g.n, g.L, B, 5, pitch=B + 3 if B % 2 else 0)
    r_or = oracle_mod.batch(g, lv, want_arrays=True, threads=os.cpu_count() or 1)
    h = emo.load_workload(g)
    assert emo.emo_call_slices(h, B, True, emo.EMO_F_SLICE_KERNEL) > 0
    r = gpu_slack_batch(torch, emo, h, lv_dev, B, g.n, ldo=B + 2, base=True, flags=emo.EMO_F_SLICE_KERNEL)
    assert_matches(r, r_or, B)
    for k in ("ES", "LS", "slack"):
        assert (r[k][:, B:] == -7).all(), "padding columns of the outputs were written"
    base = oracle_mod.batch(g, np.full((g.n, 1), g.L - 1, dtype=np.uint8))
    assert r["T0"] == base["makespan"][0] and np.isclose(r["E0"], base["energy"][0], rtol=1e-12, atol=0)
    # forward only, and one policy alone
    T, E = torch.zeros(B, dtype=torch.int64, device="cuda"), torch.zeros(B, dtype=torch.float64, device="cuda")
    ws = torch.empty(emo.emo_workspace_bytes(h, B, 0, emo.EMO_F_SLICE_KERNEL), dtype=torch.uint8, device="cuda")
    emo.emo_eval_policies(h, B, lv_dev, lv_dev.stride(0), T, E, ws, flags=emo.EMO_F_SLICE_KERNEL)
    assert np.array_equal(T.cpu().numpy(), r_or["makespan"]) and np.allclose(E.cpu().numpy(), r_or["energy"], rtol=1e-12, atol=0)
    X = torch.zeros((3, g.n), dtype=torch.int64, device="cuda")
    ws = torch.empty(emo.emo_workspace_bytes(h, 1, 1), dtype=torch.uint8, device="cuda")
    emo.emo_slack(h, lv_dev[:, B - 1].contiguous(), X[0], X[1], X[2], T[:1], E[:1], ws)
    for k, x in zip(("ES", "LS", "slack"), X.cpu().numpy()):
        assert np.array_equal(x, r_or[k][:, B - 1]), k
    assert int(T[0]) == r_or["makespan"][B - 1]
    h.free()


def test_random_dags(torch_cuda, emo, oracle_mod):
    """Random graphs (ties, zero durations, several sources and terminal nodes, nodes outside every policy) of one to six slices."""
    torch = torch_cuda
    done = 0
    for seed in range(24):
        rs = np.random.RandomState(900 + seed)
        n, L, B = int(rs.choice([1, 40, 255, 256, 257, 400, 900])), int(rs.randint(1, 9)), int(rs.choice([1, 7, 8, 9, 40]))
        g = W.random_dag(40 + seed, n, float(rs.choice([1.0, 2.0, 4.0])) / n, L=L, max_dur=int(rs.choice([2, 40, 100000])))
        group = rs.randint(-1, 6, size=g.n).astype(np.int32) if seed % 3 == 0 else None
        rows = g.n if group is None else 6
        lv, lv_dev = levels(torch, rows, L, B, seed)
        r_or = oracle_mod.batch(g, lv, want_arrays=True, group_of=group)
        h = emo.load_workload(g, group_of=group)
        if emo.emo_call_slices(h, B, True, emo.EMO_F_SLICE_KERNEL) > 0:      # (not where too many values cross every cut)
            r = gpu_slack_batch(torch, emo, h, lv_dev, B, g.n, flags=emo.EMO_F_SLICE_KERNEL)
            assert_matches(r, r_or, B)
            done += 1
        h.free()
    assert done >= 12


def test_forward_calls_take_a_workspace_anywhere(torch_cuda, emo, oracle_mod):
    """A workspace at any address (a forward-only call needs none): the slice kernels, which move it in 16-byte pieces, leave the call to others."""
    torch = torch_cuda
    g, B = W.make_graph("cfg1-train", 0.3), 40
    lv, lv_dev = levels(torch, g.n, g.L, B, 7)
    want = oracle_mod.batch(g, lv)
    h = emo.load_workload(g)
    assert emo.emo_call_slices(h, B, False) > 8      # (fewer need no workspace either)
    buf = torch.zeros(emo.emo_workspace_bytes(h, B, 0) + 64, dtype=torch.uint8, device="cuda")
    for offset in (0, 1, 4, 8, 16):
        T, E = torch.zeros(B, dtype=torch.int64, device="cuda"), torch.zeros(B, dtype=torch.float64, device="cuda")
        buf.fill_(0xEE)
        emo.emo_eval_policies(h, B, lv_dev, lv_dev.stride(0), T, E, buf[offset:])
        assert np.array_equal(T.cpu().numpy(), want["makespan"]) and np.allclose(E.cpu().numpy(), want["energy"], rtol=1e-12, atol=0), offset
        assert bool((buf == 0xEE).all()) == (offset % 16 != 0), offset
    h.free()


def test_tiles_of_policies(torch_cuda, emo, oracle_mod):
    """A workspace that does not hold all policies at once: tiles of at least 64, with remainders, the baseline in the last one; less goes to the
    other kernels.  (A forward call touches its workspace on the slice kernels only.)"""
    torch = torch_cuda
    g, B = W.make_graph("cfg1-train", 0.4), 301
    lv, lv_dev = levels(torch, g.n, g.L, B, 8)
    want, base = oracle_mod.batch(g, lv, want_arrays=True), oracle_mod.batch(g, np.full((g.n, 1), g.L - 1, dtype=np.uint8))
    h = emo.load_workload(g)
    head = emo.emo_workspace_bytes(h, B, 0, emo.EMO_F_SPINE_KERNEL)
    per = (emo.emo_workspace_bytes(h, 160, 0) - emo.emo_workspace_bytes(h, 80, 0)) / 80.0
    assert emo.emo_call_slices(h, B, False) > 8 and per > 0
    for policies, takes in ((40, False), (81, True), (100, True), (200, True), (320, True)):
        ws = torch.full((head + int(per * policies) + 4096,), 0xEE, dtype=torch.uint8, device="cuda")
        T, E, T0, E0 = (torch.full((k,), -1, dtype=d, device="cuda") for k, d in ((B + 1, torch.int64), (B + 1, torch.float64), (1, torch.int64), (1, torch.float64)))
        emo.emo_eval_policies(h, B, lv_dev, lv_dev.stride(0), T, E, ws, T0=T0, E0=E0)
        assert np.array_equal(T.cpu().numpy(), np.r_[want["makespan"], -1]) and np.allclose(E.cpu().numpy(), np.r_[want["energy"], -1.0], rtol=1e-12, atol=0), policies
        assert int(T0) == base["makespan"][0] and np.isclose(float(E0), base["energy"][0], rtol=1e-12, atol=0)
        assert bool((ws != 0xEE).any()) == takes, policies
        if takes:
            ws = torch.zeros(head + int(2.1 * per * policies) + 8192, dtype=torch.uint8, device="cuda")
            X = torch.full((3, g.n, B + 1), -7, dtype=torch.int64, device="cuda")
            ss, nc = torch.full((B,), -1, dtype=torch.int64, device="cuda"), torch.full((B,), -1, dtype=torch.int32, device="cuda")
            emo.emo_slack_batch(h, B, lv_dev, lv_dev.stride(0), X[0], X[1], X[2], B + 1, T, E, ss, nc, ws, flags=emo.EMO_F_SLICE_KERNEL, T0=T0, E0=E0)
            for k, x in zip(("ES", "LS", "slack"), X.cpu().numpy()):
                assert np.array_equal(x[:, :B], want[k]) and (x[:, B:] == -7).all(), (k, policies)
            assert np.array_equal(ss.cpu().numpy(), want["slack"].sum(0)) and np.array_equal(nc.cpu().numpy(), (want["slack"] == 0).sum(0)) and int(T0) == base["makespan"][0]
    h.free()


def test_workspace_of_forward_calls(torch_cuda, emo):
    """One size for all batches up to the largest, bounded: 250 000 nodes, where all of 1 399 policies would take 0.76 GB."""
    torch = torch_cuda
    g, B = W.make_graph("cfg4-llm", 1.0), 700
    h = emo.load_workload(g)
    head = emo.emo_workspace_bytes(h, 1, 0, emo.EMO_F_SPINE_KERNEL)
    sizes = [emo.emo_workspace_bytes(h, b, 0) for b in (0, 1, 5, 16, 100, 700, 1399, 1400, 1401, 5000, 65536)]
    assert sizes == sorted(sizes) and sizes[-1] <= head + (1 << 28)
    lv = torch.randint(0, g.L, (g.n, 704), dtype=torch.uint8, device="cuda")
    out = []
    for ws in (None, torch.empty(sizes[-1], dtype=torch.uint8, device="cuda")):
        T, E = torch.zeros(B, dtype=torch.int64, device="cuda"), torch.zeros(B, dtype=torch.float64, device="cuda")
        emo.emo_eval_policies(h, B, lv, 704, T, E, ws)
        out.append((T, E))
    assert torch.equal(out[0][0], out[1][0]) and torch.allclose(out[0][1], out[1][1], rtol=1e-11, atol=0)
    h.free()


@pytest.mark.parametrize("name, scale, B", [("cfg2-packed", 0.2, 40), ("cfg0-tiny", 1.0, 40), ("cfg1-train", 0.3, 40)])
def test_pass_events(torch_cuda, emo, name, scale, B):
    """The forward events enclose the kernels of one slice, of a block per policy, of many slices; a forward call leaves the backward ones."""
    torch = torch_cuda
    g = W.make_graph(name, scale)
    h = emo.load_workload(g)
    assert emo.emo_call_slices(h, B, True) > 0
    lv, lv_dev = levels(torch, g.n, g.L, B, 9)
    ws = torch.empty(emo.emo_workspace_bytes(h, B, 1), dtype=torch.uint8, device="cuda")
    X, T, E = torch.zeros((g.n, B), dtype=torch.int64, device="cuda"), torch.zeros(B, dtype=torch.int64, device="cuda"), torch.zeros(B, dtype=torch.float64, device="cuda")
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(5)]
    for e in ev:
        e.record()
    busy = torch.zeros(1 << 28, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    emo.emo_set_pass_events(*ev[:4])
    try:
        emo.emo_slack_batch(h, B, lv_dev, lv_dev.stride(0), None, None, X, B, T, E, None, None, ws)
        torch.cuda.synchronize()
        forward, between, backward = (a.elapsed_time(b) for a, b in zip(ev, ev[1:4]))
        assert forward > 0.004 and between >= 0 and backward >= 0      # (no kernel of these takes less than 5 us)
        busy.fill_(1)
        emo.emo_eval_policies(h, B, lv_dev, lv_dev.stride(0), T, E, ws)
        torch.cuda.synchronize()
        assert ev[0].elapsed_time(ev[1]) > 0.004 and ev[3].elapsed_time(ev[0]) > 0
    finally:
        emo.emo_set_pass_events(None, None, None, None)
    h.free()


@pytest.mark.parametrize("streams, limit", [(8, 900), (12, 600)])
def test_matrices_of_12_and_16_columns(torch_cuda, emo, oracle_mod, streams, limit):
    """On both sides of the rule's line, every output."""
    from tests.test_host_programs import streams as graph
    torch = torch_cuda
    g, _ = graph(1, 2500, streams)
    h = emo.load_workload(g)
    for B in (limit - 1, limit):
        assert (emo.emo_call_slices(h, B, True) > 0) == (emo.emo_call_slices(h, B, False) > 0) == (B < limit)
        lv, lv_dev = levels(torch, g.n, g.L, B, 10)
        want = oracle_mod.batch(g, lv, want_arrays=True, threads=os.cpu_count() or 1)
        r = gpu_slack_batch(torch, emo, h, lv_dev, B, g.n, ldo=B + 1, base=True)
        assert_matches(r, want, B)
        T, E = torch.zeros(B, dtype=torch.int64, device="cuda"), torch.zeros(B, dtype=torch.float64, device="cuda")
        ws = torch.empty(emo.emo_workspace_bytes(h, B, 0), dtype=torch.uint8, device="cuda")
        emo.emo_eval_policies(h, B, lv_dev, lv_dev.stride(0), T, E, ws)
        assert np.array_equal(T.cpu().numpy(), want["makespan"]) and np.allclose(E.cpu().numpy(), want["energy"], rtol=1e-12, atol=0)
    h.free()


def test_sixteen_policies_a_block(torch_cuda, emo, oracle_mod):
    """Slack calls with plenty of blocks (nine and more per SM) of 16 policies each, the last one partly filled; every output."""
    torch = torch_cuda
    g, B = W.make_graph("cfg1-train", 1.0), 397
    h = emo.load_workload(g)
    assert emo.emo_call_slices(h, B, True) * ((B + 1 + 15) // 16) >= 9 * torch.cuda.get_device_properties(0).multi_processor_count
    lv, lv_dev = levels(torch, g.n, g.L, B, 11)
    want = oracle_mod.batch(g, lv, want_arrays=True, threads=os.cpu_count() or 1)
    r = gpu_slack_batch(torch, emo, h, lv_dev, B, g.n, ldo=B + 1, base=True)
    assert_matches(r, want, B)
    for k in ("ES", "LS", "slack"):
        assert (r[k][:, B:] == -7).all(), "padding columns of the outputs were written"
    h.free()


def test_long_paths(torch_cuda, emo, oracle_mod):
    """Slices of up to 2^30 ns: groups of fewer of them, so that their products stay 32-bit; times beyond 2^34."""
    from tests.test_host_programs import streams as graph
    torch = torch_cuda
    g, _ = graph(5, 7000, 3, dur=30_000_000)
    B = 21
    lv, lv_dev = levels(torch, g.n, g.L, B, 12)
    want = oracle_mod.batch(g, lv, want_arrays=True, threads=os.cpu_count() or 1)
    assert int(want["makespan"].max()) > 1 << 34
    h = emo.load_workload(g)
    assert emo.emo_call_slices(h, B, True) > 32
    assert_matches(gpu_slack_batch(torch, emo, h, lv_dev, B, g.n, base=True), want, B)
    h.free()


def test_slack_in_the_other_kernels_workspace(torch_cuda, emo, oracle_mod):
    """Wide matrices take more workspace than the kernels beside them: with what those need the call goes to them."""
    torch = torch_cuda
    g, B = W.make_graph("cfg3-8dev", 0.05), 16
    lv, lv_dev = levels(torch, g.n, g.L, B, 13)
    want = oracle_mod.batch(g, lv, want_arrays=True, threads=os.cpu_count() or 1)
    h = emo.load_workload(g)
    small = emo.emo_workspace_bytes(h, B, 1, emo.EMO_F_LANE_KERNEL)
    assert emo.emo_call_slices(h, B, True) > 0 and small < emo.emo_workspace_bytes(h, B, 1)
    X, T, E = torch.zeros((g.n, B), dtype=torch.int64, device="cuda"), torch.zeros(B, dtype=torch.int64, device="cuda"), torch.zeros(B, dtype=torch.float64, device="cuda")
    for size in (max(small, emo.emo_workspace_bytes(h, B, 1, emo.EMO_F_SPINE_KERNEL)), emo.emo_workspace_bytes(h, B, 1)):
        ws = torch.empty(size, dtype=torch.uint8, device="cuda")
        X.zero_()
        emo.emo_slack_batch(h, B, lv_dev, lv_dev.stride(0), None, None, X, B, T, E, None, None, ws)
        assert np.array_equal(X.cpu().numpy(), want["slack"]) and np.array_equal(T.cpu().numpy(), want["makespan"]), size
    h.free()


def test_slices_that_no_block_can_hold(torch_cuda, emo, oracle_mod):
    """Every node waits for the sixty before it: 150 KB of steps a slice and direction.  No call can use them, nothing of them stays on the
    device (33 MB here); the other kernels take the calls."""
    torch = torch_cuda
    n, k, rs = 16_000, 60, np.random.RandomState(1)
    rp = np.r_[0, np.cumsum(np.minimum(np.arange(n), k))].astype(np.int64)
    col = np.concatenate([np.arange(max(0, v - k), v) for v in range(n)]).astype(np.int32)
    lat, energy = np.stack([rs.randint(1, 100, n), rs.randint(10 ** 5, 10 ** 6, n)], 1).astype(np.int64), rs.rand(n, 2)
    used = []
    # (the same programs otherwise: a load that shapes the spine program compiles no slices, nor the program with the longer stages)
    for flags in (emo.EMO_F_LANES(2) | emo.EMO_F_SPINE_STAGE(16), emo.EMO_F_LANES(2) | emo.EMO_F_TEST_LONG_OOM):
        before = torch.cuda.mem_get_info()[0]
        h = emo.emo_graph_load(n, rp, col, None, 2, lat, energy, None, flags)
        used.append(before - torch.cuda.mem_get_info()[0])
        assert emo.emo_call_slices(h, 1, True, emo.EMO_F_SLICE_KERNEL) == emo.emo_call_slices(h, 1, False, emo.EMO_F_SLICE_KERNEL) == 0
        if len(used) == 2:
            lv = rs.randint(0, 2, size=(n, 16)).astype(np.uint8)
            T, E = torch.zeros(16, dtype=torch.int64, device="cuda"), torch.zeros(16, dtype=torch.float64, device="cuda")
            emo.emo_eval_policies(h, 16, torch.from_numpy(lv).cuda(), 16, T, E, None)
            g = W.Graph(n, rp, col, None, 2, lat, energy, None, "dense")
            assert np.array_equal(T.cpu().numpy(), oracle_mod.batch(g, lv)["makespan"])
        h.free()
    assert used[1] < used[0] + (16 << 20), used
