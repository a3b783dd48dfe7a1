"""Calls without outputs per node evaluate a contracted graph (chains of nodes that share a policy row, or have none, are one node): the
same makespans and energies as the oracle and as the kernels that walk every node, per-node and per-pack levels, random graphs with
nodes outside every policy and constant tables, and time intervals."""
import numpy as np
import pytest

from paper_2607_12324_b200 import workloads as W
from tests.test_gpu_parity import emo, torch_cuda  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def evaluate(torch, emo, h, lv, B, flags=0):
    T, E, T0, E0 = (torch.full((k,), -1, dtype=d, device="cuda") for k, d in ((B, torch.int64), (B, torch.float64), (1, torch.int64), (1, torch.float64)))
    ws = torch.empty(emo.emo_workspace_bytes(h, B, 0, flags), dtype=torch.uint8, device="cuda")
    emo.emo_eval_policies(h, B, lv, lv.stride(0), T, E, ws, flags=flags, T0=T0, E0=E0)
    return T.cpu().numpy(), E.cpu().numpy(), int(T0), float(E0)


def chains(seed, n, L):
    """A graph of long chains with a few cross edges; a third of the nodes have constant tables, some are in no group."""
    rs = np.random.RandomState(seed)
    last, edges = [-1] * 4, []
    for v in range(n):
        k = rs.randint(4)
        if last[k] >= 0:
            edges.append((last[k], v))
        if v and rs.rand() < 0.08:
            edges.append((int(rs.randint(v)), v))
        last[k] = v
    lat = rs.randint(0, 1000, size=(n, L)).astype(np.int64)
    en = rs.rand(n, L)
    const = rs.rand(n) < 0.33
    lat[const] = lat[const][:, :1]
    en[const] = en[const][:, :1]
    group = np.where(rs.rand(n) < 0.3, -1, (np.arange(n) // 9) % 17).astype(np.int32)
    return W.tiny_graph(n, sorted(set(edges)), lat, en, name=f"chains{seed}"), group


@pytest.mark.parametrize("B", [1, 33, 2000])
@pytest.mark.parametrize("seed", range(4))
def test_random_chains(torch_cuda, emo, oracle_mod, seed, B):
    torch = torch_cuda
    g, group = chains(seed, 2000 + 300 * seed, 3 + seed)
    rows = int(group.max()) + 1
    lv = np.random.RandomState(seed).randint(0, g.L, size=(rows, (B + 15) // 16 * 16)).astype(np.uint8)
    lv_dev = torch.from_numpy(lv).cuda()
    h = emo.load_workload(g, group_of=group)
    assert 0 < emo.emo_graph_contracted(h) <= g.n * 3 // 5
    want = oracle_mod.batch(g, lv[:, :B].copy(), group_of=group)
    base = oracle_mod.batch(g, np.full((rows, 1), g.L - 1, np.uint8), group_of=group)
    for flags in (0, emo.EMO_F_SLICE_KERNEL, emo.EMO_F_NO_STAGING):
        T, E, T0, E0 = evaluate(torch, emo, h, lv_dev, B, flags)
        assert np.array_equal(T, want["makespan"]) and T0 == base["makespan"][0], flags
        # sums of at most 2 900 non-negative terms in another order
        assert np.allclose(E, want["energy"], rtol=1e-12, atol=0) and np.isclose(E0, base["energy"][0], rtol=1e-12, atol=0), flags
    h.free()


@pytest.mark.parametrize("name, scale, B", [("cfg4-llm", 0.02, 4800), ("cfg3-8dev", 0.02, 300), ("cfg0-tiny", 1.0, 64)])
def test_workloads(torch_cuda, emo, oracle_mod, name, scale, B):
    """Per-kernel levels, per-pack levels (group_of of the greedy packing), and intervals."""
    torch = torch_cuda
    g = W.make_graph(name, scale)
    is_kernel = (g.kind == W.KIND_KERNEL).astype(np.uint8)
    stream = g.meta["node_timeline"] * 64 + np.maximum(g.meta["node_stream"], 0)
    _, packs, n_packs = emo.emo_pack_greedy(g.n, g.row_ptr, g.col, is_kernel, stream, g.lat[:, -1], 5_000_000)
    some = np.unique(np.r_[0, 1, B // 2, B - 1])
    for group, rows in ((None, g.n), (packs, n_packs)):
        lv = torch.randint(0, g.L, (rows, (B + 15) // 16 * 16), dtype=torch.uint8, device="cuda")
        h = emo.load_workload(g, group_of=group)
        assert (emo.emo_graph_contracted(h) > 0) == (g.n >= 2000 and (group is not None or name == "cfg3-8dev"))
        T, E, _, _ = evaluate(torch, emo, h, lv, B)
        T2, E2, _, _ = evaluate(torch, emo, h, lv, B, emo.EMO_F_FLOW_KERNEL)
        assert np.array_equal(T, T2) and np.allclose(E, E2, rtol=1e-12, atol=0)
        want = oracle_mod.batch(g, lv.cpu().numpy()[:, some], group_of=group)
        assert np.array_equal(T[some], want["makespan"]) and np.allclose(E[some], want["energy"], rtol=1e-12, atol=0)
        h.free()
    dev = W.device_of(g)
    h = emo.load_workload(g, emo.EMO_F_INTERVALS, group_of=dev)
    I = 9
    breaks = np.arange(I, dtype=np.int64) * max(1, int(h.info.T_worst // I))
    F = W.interval_policies(3, int(dev.max()) + 1, I, g.L, B, device="cuda")
    idle = W.idle_power(g.L)
    out = []
    for flags in (0, emo.EMO_F_NO_STAGING):
        T, E, Ei = (torch.zeros(B, dtype=d, device="cuda") for d in (torch.int64, torch.float64, torch.float64))
        ws = torch.empty(emo.emo_workspace_bytes_intervals(h, B, I, True), dtype=torch.uint8, device="cuda")
        emo.emo_eval_intervals(h, B, F, F.shape[2], I, breaks, torch.from_numpy(idle).cuda(), T, E, Ei, ws, flags=flags)
        out.append([x.cpu().numpy() for x in (T, E, Ei)])
    assert np.array_equal(out[0][0], out[1][0]) and np.allclose(out[0][2], out[1][2], rtol=1e-12, atol=0) and np.allclose(out[0][1], out[1][1], rtol=1e-12, atol=0)
    want = oracle_mod.intervals(g, dev, breaks, np.ascontiguousarray(F.cpu().numpy()[:, :, some]), idle)
    assert np.array_equal(out[0][0][some], want["makespan"]) and np.allclose(out[0][1][some], want["energy"], rtol=1e-12, atol=0)
    h.free()
