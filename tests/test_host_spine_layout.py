"""Host-side check of the layout that the spine kernels read (no GPU): both programs of a graph, the one with short and the one
with long stages, interpreted in numpy (tests/spine_layout_emulator.py) reproduce the oracle's makespan, energy, slack, ES and LS -
with the stores of a stage done at once and as late as the kernels allow, in both storing forms."""
from __future__ import annotations

import numpy as np
import pytest

from paper_2607_12324_b200 import workloads as W
from tests import spine_layout_emulator as LE
from tests.test_oracle_pins import TINY, all_policies


@pytest.fixture(scope="module")
def emo():
    from paper_2607_12324_b200 import build, emo as E
    build.build()
    return E


def compare(emo, oracle_mod, g, lv, flags=0):
    """Returns the bundle sizes of the programs that exist."""
    h = emo.load_workload(g, emo.EMO_F_HOST_ONLY | flags)
    r_or = oracle_mod.batch(g, lv, want_arrays=True)
    found = []
    for long_program in (False, True):
        v = emo.emo_graph_spine_layout(h, long_program)
        if not v["ok"]:
            continue
        found.append(v["bundle"])
        for late, extra in ((False, False), (False, True), (True, False), (True, True)):
            r = LE.run(v, g.n, lv, late, extra)
            assert np.array_equal(r["makespan"], r_or["makespan"]), (long_program, late, extra)
            np.testing.assert_allclose(r["energy"], r_or["energy"], rtol=1e-9)
            for k in ("slack", "ES", "LS") if extra else ("slack",):
                assert np.array_equal(r[k], r_or[k]), (k, long_program, late, extra)
    h.free()
    assert found
    return found


@pytest.mark.parametrize("gi", range(len(TINY)))
def test_layout_on_tiny_graphs(emo, oracle_mod, gi):
    g = TINY[gi]
    lv = all_policies(g.n, g.L)
    for lanes in (0, 1, 3):
        compare(emo, oracle_mod, g, lv[:, ::max(1, lv.shape[1] // 40)].copy(), emo.EMO_F_LANES(lanes))


@pytest.mark.parametrize("name,scale,k", [("cfg0-tiny", 1.0, 0), ("cfg1-train", 0.05, 0), ("cfg2-packed", 0.3, 0), ("cfg3-8dev", 0.002, 0),
                                            ("cfg3-8dev", 0.006, 0), ("cfg4-llm", 0.004, 0), ("cfg4-llm", 0.004, 8), ("cfg3-8dev", 0.006, 32)])
def test_layout_on_config_graphs(emo, oracle_mod, name, scale, k):
    g = W.make_graph(name, scale)
    lv = np.asarray(W.policies_for(g, B=16))[:, :16]
    compare(emo, oracle_mod, g, lv, emo.EMO_F_SPINE_STAGE(k) if k else 0)


def test_layout_on_random_dags(emo, oracle_mod):
    """Sparse graphs (long segments, programs with bundles of different sizes among them) and dense ones (merge operations)."""
    sizes = set()
    for seed in range(24):
        rs = np.random.RandomState(3000 + seed)
        n = int(rs.randint(30, 400))
        L = int(rs.randint(2, 9))
        p = float(rs.uniform(3, 12)) / n if seed % 2 else float(rs.choice([0.05, 0.12, 0.2]))
        g = W.random_dag(800 + seed, n, p, L=L, max_dur=int(rs.choice([5, 40, 100000])))
        h = emo.load_workload(g, emo.EMO_F_HOST_ONLY)
        ok = emo.emo_graph_spine(h)["ok"]
        h.free()
        if ok:
            sizes.add(tuple(compare(emo, oracle_mod, g, rs.randint(0, L, size=(g.n, 12)).astype(np.uint8))))
    assert {s for t in sizes for s in t} == {2, 4}
