"""Pack modelling at the edges of its launch: one unknown and the most, odd numbers of packs (a warp takes two), more packs
than the blocks hold at once, levels that do not fill a half-warp, tables beyond 40 KB.

Tolerance: both sides solve the normal equations of the same free set in fp64, and a variable may be held whose gradient
component is below 1e-13 of the largest |B^T b|; either moves x by at most (1e-13 + rounding) cond(B)^2 of its largest entry."""
import numpy as np
import pytest

from paper_2607_12324_b200 import workloads as W
from tests.test_gpu_model import emo, run, torch_cuda  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,L,P", [(3, 1, 1, 1), (16, 16, 17, 2), (18, 16, 15, 33), (20, 15, 33, 16), (16, 12, 230, 5), (9, 6, 5, 8000)])
def test_edges(torch_cuda, emo, oracle_mod, n, m, L, P):  # noqa: F811
    B, Tb, Eb = W.microbench_model(21, n, m, L)
    feat = W.pack_features(22, B, P, noise=0.1)
    xo, To, Eo = oracle_mod.pack_model(B, feat, Tb, Eb)
    x, T, E = run(torch_cuda, emo, B, feat, Tb, Eb)
    tol = 4e-13 * np.linalg.cond(B) ** 2
    scale = np.abs(xo).max(axis=1, keepdims=True) + 1e-300
    assert (np.abs(x - xo) <= tol * scale).all()
    for got, want, tab in ((T, To, Tb), (E, Eo, Eb)):
        assert (np.abs(got - want) <= tol * scale * m * np.abs(tab).max()).all()
