"""Time-interval policies where whole runs of a lane are checked at once: runs of every length, packs that end exactly on a change
point, that cross one or several, lanes that serve two devices; times bit-exact, and equal policies with equal energies bit for
bit beside policies that leave the interval elsewhere.  Energy tolerance: both sides add n terms in fp64, at most n roundings."""
import numpy as np
import pytest

from paper_2607_12324_b200 import workloads as W
from tests.test_gpu_intervals import emo, run_gpu, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,B,step,devices", [(1, 1, 10, 1), (9, 33, 10, 1), (300, 70, 10, 1), (300, 64, 95, 1), (300, 33, 3, 2), (300, 129, 400, 2)])
def test_runs(torch_cuda, emo, oracle_mod, n, B, step, devices):  # noqa: F811
    rs = np.random.RandomState(n + B + step)
    L = 4
    lat = np.sort(rs.randint(1, 25, size=(n, L)), axis=1)[:, ::-1].astype(np.int64)
    lat[rs.rand(n) < 0.2] = 10                                  # ends on change points, and packs of no choice
    edges = [(i, i + 1) for i in range(n - 1)] + [(i, i + 3) for i in range(0, n - 3, 11)]
    g = W.tiny_graph(n, sorted(set(edges)), lat, rs.rand(n, L))
    dev = rs.randint(-1, devices, size=n)
    dev[0] = devices - 1
    I = 12
    F = rs.randint(0, L, size=(devices, I, B)).astype(np.uint8)
    F[:, :, ::7] = F[:, :, :1]
    T, E, Ei = run_gpu(torch_cuda, emo, g, dev, np.arange(I, dtype=np.int64) * step, F, [1.0, 2.0, 3.0, 4.0], flags=emo.EMO_F_INTERVALS)
    r = oracle_mod.intervals(g, dev, np.arange(I, dtype=np.int64) * step, F, [1.0, 2.0, 3.0, 4.0])
    assert np.array_equal(T, r["makespan"])
    assert np.allclose(E, r["energy"], rtol=(n + devices * I) * 2.3e-16, atol=0)
    assert np.allclose(Ei, r["e_idle"], rtol=(devices * I + 2) * 2.3e-16, atol=1e-30)
    assert (E[::7] == E[0]).all() and (T[::7] == T[0]).all()


@pytest.mark.parametrize("n,I,B", [(400, 4, 70), (400, 40, 33), (2000, 4, 300)])
def test_two_devices_that_lanes_seldom_change(torch_cuda, emo, oracle_mod, n, I, B):  # noqa: F811
    """The first half of the packs on one device, the second on the other: the interval at hand is kept across runs and given up
    where the device changes (with 40 intervals also the kernel that keeps none)."""
    rs = np.random.RandomState(n + I)
    L = 4
    lat = np.sort(rs.randint(1, 25, size=(n, L)), axis=1)[:, ::-1].astype(np.int64)
    edges = [(i, i + 1) for i in range(n - 1)] + [(i, i + 3) for i in range(0, n - 3, 11)]
    g = W.tiny_graph(n, sorted(set(edges)), lat, rs.rand(n, L))
    dev = (np.arange(n) >= n // 2).astype(np.int64)
    step = max(1, n * 10 // I)
    F = rs.randint(0, L, size=(2, I, B)).astype(np.uint8)
    T, E, Ei = run_gpu(torch_cuda, emo, g, dev, np.arange(I, dtype=np.int64) * step, F, [1.0, 2.0, 3.0, 4.0], flags=emo.EMO_F_INTERVALS)
    r = oracle_mod.intervals(g, dev, np.arange(I, dtype=np.int64) * step, F, [1.0, 2.0, 3.0, 4.0])
    assert np.array_equal(T, r["makespan"])
    assert np.allclose(E, r["energy"], rtol=(n + 2 * I) * 2.3e-16, atol=0)
    assert np.allclose(Ei, r["e_idle"], rtol=(2 * I + 2) * 2.3e-16, atol=1e-30)
