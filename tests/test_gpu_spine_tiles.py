"""GPU parity of the spine kernels at the edges of their policy tiles: one, two, four and eight groups of 32 policies per block
(a worker thread then handles one, two or four policies), full and ragged last tiles, the baseline column in a tile of its own,
output pitches that allow and forbid vector stores, bundles of two (narrow graphs) and of four operations (wide graphs), with
and without folded tails, every output; against the CPU oracle: times bit-exact, energy within the reordering bound."""
from __future__ import annotations

import os

import numpy as np
import pytest

from paper_2607_12324_b200 import workloads as W
from tests.test_gpu_parity import E_RTOL, assert_matches, emo, gpu_slack_batch, torch_cuda  # noqa: F401  (fixtures)

pytestmark = pytest.mark.gpu

# policies per block with one block per SM, in groups of 32 (the widest graph's rows of slots leave no room for eight)
CASES = [("cfg1-train", 0.02, g, d) for g in (1, 2, 4, 8) for d in (-1, 0)] + \
        [("cfg4-llm", 0.002, g, d) for g in (1, 2, 4) for d in (-5, 0)] + \
        [("cfg3-8dev", 0.004, g, d) for g in (1, 2) for d in (-31, 0)]


# three groups for calls with ES, LS or the sums (one policy per worker thread), six (two)
CASES += [("cfg1-train", 0.02, g, d) for g in (3, 6) for d in (-1, 0, -33)] + [("cfg2-packed", 0.5, 6, -1), ("cfg4-llm", 0.002, 3, -1)]


@pytest.mark.parametrize("name,scale,groups,off", CASES)
def test_tiles(torch_cuda, emo, oracle_mod, name, scale, groups, off):
    torch = torch_cuda
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = W.make_graph(name, scale)
    B = sms * 32 * groups + off
    lv = W.policies_for(g, B=B, device="cuda")
    host = lv.cpu().numpy()
    r_or = oracle_mod.batch(g, host, B=B, want_arrays=True, threads=os.cpu_count() or 1)
    base = oracle_mod.batch(g, np.full((g.n, 1), g.L - 1, dtype=np.uint8))
    h = emo.load_workload(g)
    assert emo.emo_graph_spine(h)["ok"] == 1
    for ldo in (B, (B + 3) // 4 * 4 + 1):
        r = gpu_slack_batch(torch, emo, h, lv, B, g.n, want=("slack",), sums=False, base=True, flags=emo.EMO_F_SPINE_KERNEL, ldo=ldo)
        assert np.array_equal(r["makespan"], r_or["makespan"]) and r["T0"] == base["makespan"][0]
        np.testing.assert_allclose(r["energy"], r_or["energy"], rtol=E_RTOL, atol=0)
        assert r["E0"] == pytest.approx(base["energy"][0], rel=E_RTOL)
        assert np.array_equal(r["slack"][:, :B], r_or["slack"])
        assert (r["slack"][:, B:] == -7).all(), "padding columns of the slack matrix were written"
        r = gpu_slack_batch(torch, emo, h, lv, B, g.n, flags=emo.EMO_F_SPINE_KERNEL, ldo=ldo)
        assert_matches(r, r_or, B)
    h.free()


@pytest.mark.parametrize("name,scale", [("cfg3-8dev", 0.002), ("cfg3-8dev", 0.003), ("random", 38), ("random", 39)])
def test_programs_with_different_bundles(torch_cuda, emo, oracle_mod, name, scale):
    """Graphs whose program of long stages (batches of up to two groups per SM) has bundles of another size than the short one:
    default flags, every output, batches on both sides of the line."""
    torch = torch_cuda
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = W.make_graph(name, scale) if name != "random" else W.random_dag(*{38: (38, 253, 0.04348380468633499), 39: (39, 305, 0.03172406145819659)}[scale])
    h = emo.load_workload(g)
    bundles = set()
    for B in (1, 64, 4096, sms * 64 + 33):
        bundles.add(emo.emo_graph_spine_plan(h, B, True, True, sms)["bundle"])
        host = np.full((g.n, (B + 15) // 16 * 16), 0xFF, dtype=np.uint8)
        host[:, :B] = np.random.RandomState(B).randint(0, g.L, size=(g.n, B))
        lv = torch.as_tensor(host, device="cuda")
        r_or = oracle_mod.batch(g, host, B=B, want_arrays=True, threads=os.cpu_count() or 1)
        base = oracle_mod.batch(g, np.full((g.n, 1), g.L - 1, dtype=np.uint8))
        r = gpu_slack_batch(torch, emo, h, lv, B, g.n, want=("slack",), sums=False, base=True)
        assert np.array_equal(r["makespan"], r_or["makespan"]) and r["T0"] == base["makespan"][0]
        np.testing.assert_allclose(r["energy"], r_or["energy"], rtol=E_RTOL, atol=0)
        assert np.array_equal(r["slack"][:, :B], r_or["slack"])
        assert_matches(gpu_slack_batch(torch, emo, h, lv, B, g.n), r_or, B)
    assert bundles == {2, 4}
    h.free()


@pytest.mark.parametrize("name,scale", [("cfg1-train", 0.02), ("cfg3-8dev", 0.003)])
def test_one_workspace_for_smaller_batches_and_other_outputs(torch_cuda, emo, name, scale):
    """The workspace of a batch serves every smaller one, whichever tile and program that takes, and calls with more outputs."""
    torch = torch_cuda
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    g = W.make_graph(name, scale)
    h = emo.load_workload(g)
    most = 7 * 32 * sms + 1
    lv = W.policies_for(g, B=most, device="cuda")
    X = torch.zeros((3, g.n, most), dtype=torch.int64, device="cuda")
    T, E = torch.zeros(most, dtype=torch.int64, device="cuda"), torch.zeros(most, dtype=torch.float64, device="cuda")
    want = None
    for top in (most, 6 * 32 * sms, 4 * 32 * sms + 1, 3 * 32 * sms - 1, 2 * 32 * sms - 1, 32 * sms):
        ws = torch.empty(emo.emo_workspace_bytes(h, top, 1), dtype=torch.uint8, device="cuda")
        for B in sorted({top, top - 31, 5 * 32 * sms, 3 * 32 * sms, 2 * 32 * sms - 1, 32 * sms + 1, 32 * sms - 1, 7}, reverse=True):
            if B > top:
                continue
            T.zero_()
            emo.emo_slack_batch(h, B, lv, lv.stride(0), X[0], X[1], X[2], most, T, E, None, None, ws=ws)
            if want is None:
                want = T.clone()
            assert torch.equal(T[:B], want[:B])
    h.free()
