"""Time intervals, a thread per policy (graphs of few lanes): the oracle's times, busy times and energies and
those of the step-program kernel, at batches around a warp's and a block's policies, short and long intervals, nodes that outlast them."""
import numpy as np
import pytest

from paper_2607_12324_b200 import workloads as W
from tests.test_gpu_parity import emo, torch_cuda  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu


def weave(seed, n, rows):
    """Every node waits for the last one of its stream and, half of the time, for one of the streams beside it."""
    rs = np.random.RandomState(seed)
    last, edges = [-1] * 2, []
    for v in range(n):
        k = rs.randint(2)
        for u in {last[k], last[rs.randint(2)] if rs.rand() < 0.5 else -1}:
            if u >= 0:
                edges.append((u, v))
        last[k] = v
    lat = rs.randint(0, 1000, size=(n, 5)).astype(np.int64)
    lat[rs.rand(n) < 0.02] *= 60                      # outlasts an interval
    group = np.where(rs.rand(n) < 0.2, -1, rs.randint(0, rows, size=n)).astype(np.int32)
    return W.tiny_graph(n, sorted(set(edges)), lat, rs.rand(n, 5), name=f"weave{seed}"), group


@pytest.mark.parametrize("seed, n, rows, I, B", [(0, 40, 1, 2, 1), (1, 300, 1, 7, 5), (2, 700, 3, 40, 33), (3, 700, 2, 400, 129), (4, 1500, 1, 3, 2500), (5, 1500, 4, 26, 20000)])
def test_against_oracle_and_step_program(torch_cuda, emo, oracle_mod, seed, n, rows, I, B):
    torch = torch_cuda
    g, group = weave(seed, n, rows)
    rows = int(group.max()) + 1
    h = emo.load_workload(g, emo.EMO_F_INTERVALS, group_of=group)
    assert emo.emo_graph_flow(h, arrays=False)["lanes"] <= 3      # (the call takes a thread per policy)
    # a grid that ends before the schedule does, and one that outlasts it
    for span in (0.6, 1.5):
        breaks = np.arange(I, dtype=np.int64) * max(1, int(h.info.T_best * span / I))
        assert emo.emo_call_intervals(h, B, breaks) == 2 and emo.emo_call_intervals(h, B, breaks, emo.EMO_F_NO_STAGING) == 0
        F = np.random.RandomState(seed).randint(0, g.L, size=(rows, I, (B + 15) // 16 * 16)).astype(np.uint8)
        Fd, idle = torch.from_numpy(F).cuda(), torch.from_numpy(W.idle_power(g.L)).cuda()
        out = []
        for flags in (0, emo.EMO_F_NO_STAGING):
            T, E, Ei = (torch.zeros(B, dtype=d, device="cuda") for d in (torch.int64, torch.float64, torch.float64))
            ws = torch.empty(emo.emo_workspace_bytes_intervals(h, B, I, True), dtype=torch.uint8, device="cuda")
            emo.emo_eval_intervals(h, B, Fd, F.shape[2], I, breaks, idle, T, E, Ei, ws, flags=flags)
            out.append([x.cpu().numpy() for x in (T, E, Ei)])
        # busy times are whole numbers: the idle energies are the same sums; energies of at most 1 500 non-negative terms, in another order
        assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][2], out[1][2])
        assert np.allclose(out[0][1], out[1][1], rtol=1e-12, atol=0)
        some = np.unique(np.r_[0, B // 2, B - 1])
        want = oracle_mod.intervals(g, group, breaks, np.ascontiguousarray(F[:, :, some]), W.idle_power(g.L))
        assert np.array_equal(out[0][0][some], want["makespan"]) and np.allclose(out[0][1][some], want["energy"], rtol=1e-12, atol=0)
    h.free()


def test_energy_does_not_depend_on_the_policies_beside_it(torch_cuda, emo):
    """The same policy alone, among copies of itself and among policies whose nodes outlast whole intervals: the same energy, bit for bit (a
    search keeps the first of equal candidates)."""
    torch = torch_cuda
    n, rs = 400, np.random.RandomState(11)            # one chain: items of as many nodes as there can be, and some of four and fewer
    lat = rs.randint(1, 100, size=(n, 5)).astype(np.int64)
    lat[:, 0] *= 20                                   # level 0: an item of eight nodes outlasts the intervals below, elsewhere none does
    g = W.tiny_graph(n, [(v - 1, v) for v in range(1, n)], lat, rs.rand(n, 5))
    h = emo.load_workload(g, emo.EMO_F_INTERVALS, group_of=np.where(np.arange(n) < 300, 0, np.arange(n) // 4 % 2).astype(np.int32))
    I, rs = 600, np.random.RandomState(13)
    breaks = np.arange(I, dtype=np.int64) * 1500      # (and none is in the last one before the end)
    mine = rs.randint(1, 5, size=(2, I))
    assert emo.emo_call_intervals(h, 4, breaks) == 2

    def energies(F):
        B = F.shape[2]
        Fd = torch.from_numpy(np.ascontiguousarray(F.astype(np.uint8))).cuda()
        T, E = torch.zeros(B, dtype=torch.int64, device="cuda"), torch.zeros(B, dtype=torch.float64, device="cuda")
        ws = torch.empty(emo.emo_workspace_bytes_intervals(h, B, I, False), dtype=torch.uint8, device="cuda")
        emo.emo_eval_intervals(h, B, Fd, B, I, breaks, None, T, E, None, ws)
        return E.cpu().numpy()
    alone = energies(mine[:, :, None])[0]
    for B in (4, 16, 3000):
        assert (energies(np.repeat(mine[:, :, None], B, axis=2)) == alone).all()
        F = np.where(np.arange(B) % 3 == 0, mine[:, :, None], 0)
        assert (energies(F)[::3] == alone).all(), B
    h.free()


def test_many_lanes_in_several_waves(torch_cuda, emo, oracle_mod):
    """More than three lanes: the walk from the batch on whose lane-stream blocks come in two waves."""
    torch = torch_cuda
    g = W.make_graph("cfg3-8dev", 0.01)
    group = W.device_of(g)
    h = emo.load_workload(g, emo.EMO_F_INTERVALS, group_of=group)
    I, rows = 6, int(group.max()) + 1
    breaks = np.arange(I, dtype=np.int64) * max(1, int(h.info.T_worst // I))
    assert emo.emo_graph_flow(h, arrays=False)["lanes"] > 8
    idle = W.idle_power(g.L)
    for B, kernel in ((1000, 1), (4737, 2), (6000, 2)):
        assert emo.emo_call_intervals(h, B, breaks) == kernel
        F = W.interval_policies(3, rows, I, g.L, B, device="cuda")
        out = []
        for flags in (0, emo.EMO_F_FLOW_KERNEL):
            T, E, Ei = (torch.zeros(B, dtype=d, device="cuda") for d in (torch.int64, torch.float64, torch.float64))
            ws = torch.empty(emo.emo_workspace_bytes_intervals(h, B, I, True), dtype=torch.uint8, device="cuda")
            emo.emo_eval_intervals(h, B, F, F.shape[2], I, breaks, torch.from_numpy(idle).cuda(), T, E, Ei, ws, flags=flags)
            out.append([x.cpu().numpy() for x in (T, E, Ei)])
        # (busy times are whole numbers; energies are 1 300 terms in another order)
        assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][2], out[1][2]) and np.allclose(out[0][1], out[1][1], rtol=1e-12, atol=0)
        some = np.unique(np.r_[0, 31, 32, B // 2, B - 1])
        want = oracle_mod.intervals(g, group, breaks, np.ascontiguousarray(F.cpu().numpy()[:, :, some]), idle)
        assert np.array_equal(out[0][0][some], want["makespan"]) and np.allclose(out[0][1][some], want["energy"], rtol=1e-12, atol=0)
    h.free()
