"""Levels that change from call to call: the passes start ahead of their predecessors' end, but never read a level before its writer
has finished - also when that writer lets its successors start early (a kernel that releases its dependents on entry and writes
200 microseconds later).  Two sets of policies in turn in the same buffers; every result against the CPU oracle's."""
import os

import numpy as np
import pytest

from paper_2607_12324_b200 import workloads as W
from tests.test_gpu_parity import emo, torch_cuda  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu

LATE_COPY = r"""
extern "C" __global__ void late_copy(const unsigned char *src, unsigned char *dst, int n)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const long long t0 = clock64();
    while (clock64() - t0 < 400000) {}
    for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}
"""


@pytest.fixture(scope="module")
def late_copy(torch_cuda):  # noqa: F811
    k = torch_cuda.cuda._compile_kernel(LATE_COPY, "late_copy")
    return lambda dst, src: k((1, 1, 1), (1024, 1, 1), (src, dst, int(dst.numel())))


@pytest.mark.parametrize("name,scale,B", [("cfg0-tiny", 1.0, 64), ("cfg1-train", 0.1, 1), ("cfg1-train", 0.1, 333), ("cfg3-8dev", 0.01, 200)])
def test_levels_rewritten_between_calls(torch_cuda, emo, oracle_mod, late_copy, name, scale, B):  # noqa: F811
    torch = torch_cuda
    g = W.make_graph(name, scale)
    ldb = (B + 15) // 16 * 16
    rs = np.random.RandomState(B)
    host = [rs.randint(0, g.L, size=(g.n, ldb)).astype(np.uint8) for _ in range(2)]
    want = [oracle_mod.batch(g, x, B=B, want_arrays=True, threads=os.cpu_count() or 1) for x in host]
    src = [torch.as_tensor(x, device="cuda") for x in host]
    one = [torch.as_tensor(np.ascontiguousarray(x[:, 0]), device="cuda") for x in host]
    lvl, lvl_one = torch.zeros_like(src[0]), torch.zeros_like(one[0])
    h = emo.load_workload(g)
    ws = torch.empty(emo.emo_workspace_bytes(h, B, 1), dtype=torch.uint8, device="cuda")
    ws1 = torch.empty(emo.emo_workspace_bytes(h, 1, 1), dtype=torch.uint8, device="cuda")
    results = []
    for turn in range(6):
        k = turn % 2
        X = [torch.full((g.n, B), -7, dtype=torch.int64, device="cuda") for _ in range(2)]
        T, E = torch.zeros(B, dtype=torch.int64, device="cuda"), torch.zeros(B, dtype=torch.float64, device="cuda")
        O = [torch.full((g.n,), -7, dtype=torch.int64, device="cuda") for _ in range(6)]
        T1, E1 = torch.zeros(1, dtype=torch.int64, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
        late_copy(lvl, src[k])
        emo.emo_slack_batch(h, B, lvl, ldb, None, None, X[0], B, T, E, None, None, ws)
        late_copy(lvl, src[1 - k])
        emo.emo_slack_batch(h, B, lvl, ldb, X[1], None, None, B, T, E, None, None, ws)
        late_copy(lvl_one, one[k])
        emo.emo_slack(h, lvl_one, O[0], O[1], O[2], T1, E1, ws=ws1)
        late_copy(lvl_one, one[1 - k])
        emo.emo_slack(h, lvl_one, O[3], O[4], O[5], T1, E1, ws=ws1)
        results.append((k, X, T, O, T1))
    torch.cuda.synchronize()
    for k, X, T, O, T1 in results:
        assert np.array_equal(X[0].cpu().numpy(), want[k]["slack"])
        assert np.array_equal(X[1].cpu().numpy(), want[1 - k]["ES"]) and np.array_equal(T.cpu().numpy(), want[1 - k]["makespan"])
        for i, got in enumerate(O):
            assert np.array_equal(got.cpu().numpy(), want[k if i < 3 else 1 - k][("ES", "LS", "slack")[i % 3]][:, 0])
        assert int(T1.item()) == want[1 - k]["makespan"][0]
    h.free()


@pytest.mark.parametrize("name,scale,B", [("cfg2-packed", 0.2, 40), ("cfg0-tiny", 1.0, 64), ("cfg1-train", 0.3, 200), ("cfg1-train", 0.6, 1000)])
def test_selection_behind_rewritten_levels(torch_cuda, emo, oracle_mod, late_copy, name, scale, B):  # noqa: F811
    """Slice kernels of one slice, of a block per policy, of chained slices and of groups of them, then the one-block selection under the
    baseline's budget, levels rewritten before every call: each sees what its predecessor wrote."""
    torch = torch_cuda
    g = W.make_graph(name, scale)
    ldb = (B + 15) // 16 * 16
    rs = np.random.RandomState(B)
    host = [rs.randint(0, g.L, size=(g.n, ldb)).astype(np.uint8) for _ in range(2)]
    for x in host:
        x[:, 3::4] = g.L - 1 - (x[:, 3::4] == 0)      # (policies near the default one, inside the budget)
    want = [oracle_mod.batch(g, x, B=B, threads=os.cpu_count() or 1) for x in host]
    T0 = int(oracle_mod.batch(g, np.full((g.n, 1), g.L - 1, np.uint8))["makespan"][0])
    pick = [oracle_mod.select(r["makespan"], r["energy"], oracle_mod.target_from_delta(T0, 50_000)) for r in want]
    assert pick[0] != pick[1] and min(pick) >= 0
    src = [torch.as_tensor(x, device="cuda") for x in host]
    lvl = torch.zeros_like(src[0])
    h = emo.load_workload(g)
    assert emo.emo_call_slices(h, B, True) > 0
    ws = torch.empty(emo.emo_workspace_bytes(h, B, 1), dtype=torch.uint8, device="cuda")
    X = torch.zeros((g.n, B), dtype=torch.int64, device="cuda")
    T, E, base, base_E = (torch.zeros(k, dtype=d, device="cuda") for k, d in ((B, torch.int64), (B, torch.float64), (1, torch.int64), (1, torch.float64)))
    got = torch.full((12,), -7, dtype=torch.int64, device="cuda")
    for turn in range(12):
        late_copy(lvl, src[turn // 2 % 2])
        if turn % 2:
            emo.emo_eval_policies(h, B, lvl, ldb, T, E, ws, T0=base, E0=base_E)
        else:
            emo.emo_slack_batch(h, B, lvl, ldb, None, None, X, B, T, E, None, None, ws, T0=base, E0=base_E)
        emo.emo_select(B, T, E, 0, got[turn:turn + 1], None, None, ws=ws, target_dev=base, delta_ppm=50_000)
    torch.cuda.synchronize()
    assert got.cpu().tolist() == [pick[turn // 2 % 2] for turn in range(12)]
    h.free()
