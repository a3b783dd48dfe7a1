"""The compilers of the slice, contraction and walk programs on the host (no GPU): host_programs.cpp interprets what they build as the
kernels do and compares it with the plain recurrences."""
from __future__ import annotations

import ctypes
import os
import subprocess
import time

import numpy as np
import pytest

from paper_2607_12324_b200 import workloads as W
from tests.conftest import ROOT

SLICES, CONTRACT, WALK = 0, 1, 2


@pytest.fixture(scope="module")
def programs(tmp_path_factory):
    csrc = os.path.join(ROOT, "paper_2607_12324_b200", "csrc")
    lib = str(tmp_path_factory.mktemp("programs") / "programs.so")
    sources = ["emo_slice_compile.cpp", "emo_contract.cpp", "emo_walk_compile.cpp", "emo_flow_compile.cpp", "emo_spine_compile.cpp", "emo_compile.cpp"]
    subprocess.check_call(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-o", lib, os.path.join(ROOT, "tests", "host_programs.cpp")] + [os.path.join(csrc, s) for s in sources])
    so = ctypes.CDLL(lib)
    so.program_failure.restype = ctypes.c_char_p
    return so


def arguments(g, group):
    group = np.arange(g.n) if group is None else np.asarray(group)
    arrays = [np.ascontiguousarray(a, t) for a, t in ((g.row_ptr, np.int64), (g.col, np.int32), (group, np.int32), (g.lat, np.int64), (g.energy, np.float64))]
    rp, col, gr, lat, en = (a.ctypes.data_as(ctypes.c_void_p) for a in arrays)
    return arrays, (ctypes.c_int32(g.n), rp, col, gr, ctypes.c_int32(int(group.max(initial=-1)) + 1), ctypes.c_int32(g.L), lat, en)


def check(programs, kind, g, group=None, seed=0):
    """What the compiler reports, None where it leaves the graph to others."""
    keep, args = arguments(g, group)
    info = np.zeros(4, np.int32)
    rc = programs.program_check(kind, *args, ctypes.c_uint32(seed), info.ctypes.data_as(ctypes.c_void_p))
    assert rc >= 0, (programs.program_failure(), g.name, seed)
    return info.tolist() if rc else None


def random_graph(seed, longest=None):
    """Graphs of up to 1 500 nodes whose edges span up to 60, with sources, several ends, ties, nodes outside every policy, constant tables."""
    rs = np.random.RandomState(seed)
    n, L, most, span = 1 + rs.randint(1500 if seed % 7 == 0 else 300), 1 + rs.randint(9), 1 + rs.randint(4), 1 + rs.randint(60)
    edges = {(v - 1 - rs.randint(min(v, span)), v) for v in range(1, n) if rs.rand() > 0.2 for _ in range(1 + rs.randint(most))}
    dur = longest or (3 if rs.rand() < 0.3 else 100_000)
    lat, energy = rs.randint(0, dur, size=(n, L)).astype(np.int64), rs.rand(n, L)
    same = rs.rand(n) < (0.5 if rs.rand() < 0.5 else 0.0)
    lat[same], energy[same] = lat[same][:, :1], energy[same][:, :1]
    if seed % 11 == 0:
        lat[::17] *= 300
    group = None if rs.rand() < 0.5 else rs.randint(-1, 5, size=n)
    return W.tiny_graph(n, sorted(edges), lat, energy, name=f"random{seed}"), group


def test_slices(programs):
    """One slice, several, and (chains of three streams) more than are chained one by one."""
    kinds = {"one": 0, "several": 0, "groups": 0}
    for seed in range(160):
        g, group = random_graph(seed)
        info = check(programs, SLICES, g, group, seed)
        if info:
            kinds["one" if info[0] == 1 else "several"] += 1
    for seed in range(4):
        g, group = streams(seed, 7000, 3)
        info = check(programs, SLICES, g, group, seed)
        kinds["groups"] += info[2] > 1
    assert kinds["one"] > 20 and kinds["several"] > 20 and kinds["groups"] == 4


def streams(seed, n, k, dur=1000, L=4):
    """k streams in program order with a cross edge now and then."""
    rs = np.random.RandomState(seed)
    last, edges = [-1] * k, []
    for v in range(n):
        s = rs.randint(k)
        for u in {last[s], last[rs.randint(k)] if rs.rand() < 0.1 else -1}:
            if u >= 0:
                edges.append((u, v))
        last[s] = v
    return W.tiny_graph(n, edges, rs.randint(0, dur, size=(n, L)).astype(np.int64), rs.rand(n, L), name=f"streams{seed}"), None


def test_slices_of_long_paths(programs):
    """Slices of up to 2^30 ns: fewer of them in a group than their number alone would ask for, so that products stay 32-bit."""
    g, group = streams(5, 7000, 3, dur=30_000_000)
    plain, long = check(programs, SLICES, streams(5, 7000, 3)[0]), check(programs, SLICES, g, group)
    assert plain[2] > 1 and long[3] < plain[3] and long[0] > 32


def test_contraction(programs):
    smaller = 0
    for seed in range(160):
        g, group = random_graph(seed)
        smaller += check(programs, CONTRACT, g, group, seed)[0] < g.n
    assert smaller > 80


def test_walk(programs):
    done = 0
    for seed in range(160):
        g, group = random_graph(seed)
        done += check(programs, WALK, g, np.zeros(g.n, np.int64) if group is None else group, seed) is not None
    assert done > 150


@pytest.mark.parametrize("name, scale", [("cfg0-tiny", 1.0), ("cfg1-train", 0.3), ("cfg2-packed", 1.0), ("cfg3-8dev", 0.02), ("cfg4-llm", 0.03)])
def test_workloads(programs, name, scale):
    g = W.make_graph(name, scale)
    assert check(programs, SLICES, g) and check(programs, CONTRACT, g) and check(programs, WALK, g, W.device_of(g))


def wide_join(n, L, ends=False):
    """Arguments of program_compile: a chain whose every node one last node waits for, with an end behind every node or not."""
    chain = n // 2 if ends else n - 1
    edges = np.r_[np.c_[np.arange(chain - 1), np.arange(1, chain)], np.c_[np.arange(chain), np.full(chain, n - 1)]]
    if ends:
        edges = np.r_[edges, np.c_[np.arange(chain - 1), np.arange(chain, n - 1)]]
    edges = edges[np.lexsort((edges[:, 0], edges[:, 1]))]
    rp = np.r_[0, np.cumsum(np.bincount(edges[:, 1], minlength=n))].astype(np.int64)
    # (with several levels every operand can decide the last node's start: short nodes at one level, long ones at another)
    lat = np.repeat([[10 if L == 1 else 1000 * n] + [10] * (L - 1)], n, axis=0).astype(np.int64)
    lat[n - 1] = 10
    keep = [rp, np.ascontiguousarray(edges[:, 0], np.int32), np.arange(n, dtype=np.int32) % 2 if L > 1 else np.full(n, -1, np.int32), lat, np.ones((n, L))]
    a = [x.ctypes.data_as(ctypes.c_void_p) for x in keep]
    return keep, [ctypes.c_int32(n), a[0], a[1], a[2], ctypes.c_int32(2 if L > 1 else 0), ctypes.c_int32(L), a[3], a[4]]


@pytest.mark.parametrize("ends", [False, True])
def test_slices_of_a_wide_join(programs, ends):
    """A chain whose every node one last node waits for (a host sync), and the same with an end of its own behind every node: the slices'
    compiler looks at every edge a bounded number of times.  (Every operand looked up among its reader's, or a reader's operands counted
    again with each of them, is 4e9 steps here, more than two seconds.)"""
    keep, args = wide_join(180_000 if ends else 90_000, 1, ends)
    t = time.process_time()
    sliced = programs.program_compile(SLICES, *args)
    t = time.process_time() - t
    assert (ends or sliced == 1) and t < 1.0, t      # (with the ends every chain node is waited for across every cut: left to others)


@pytest.mark.parametrize("n, L", [(20_000, 4), (160_000, 4), (20_000, 200)])
def test_walk_programs_that_no_block_can_hold(programs, n, L):
    """A node with tens of thousands of operands, and more than 128 levels: refused, and nothing of the program is kept (0.9 GB for 160 000
    nodes, 61 MB for 200 levels)."""
    keep, args = wide_join(n, L) if L == 4 else arguments(streams(3, n, 2, L=L)[0], np.zeros(n, np.int32))
    assert programs.program_compile(WALK, *args) == 0
