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


def test_two_threads_with_tables_of_different_sizes(torch_cuda, emo):  # noqa: F811
    """Concurrent callers whose tables take 41 and 45 KB of shared memory: every call launches, with the results it has alone."""
    import threading
    n, m, P = 16, 12, 64
    jobs, errors = [], []
    for L in (212, 230):
        B, Tb, Eb = W.microbench_model(31, n, m, L)
        dev = [torch_cuda.as_tensor(np.ascontiguousarray(a), device="cuda") for a in (B, W.pack_features(32, B, P), Tb, Eb)]
        out = [torch_cuda.zeros(s, dtype=torch_cuda.float64, device="cuda") for s in ((P, m), (P, L), (P, L))]
        emo.emo_pack_model(P, n, m, L, *dev, *out)
        jobs.append((L, dev, out, [o.clone() for o in out], torch_cuda.cuda.Stream()))
    torch_cuda.cuda.synchronize()

    def call(L, dev, out, want, stream):
        try:
            for _ in range(2000):
                emo.emo_pack_model(P, n, m, L, *dev, *out, stream=stream)
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=call, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch_cuda.cuda.synchronize()
    assert not errors, errors[0]
    for _, _, out, want, _ in jobs:
        assert all(torch_cuda.equal(a, b) for a, b in zip(out, want))


@pytest.mark.parametrize("scale", [1.5, 2.0, 3.0, 6.5, 2.0 ** -3.3, 2.0 ** 40.5, 2.0 ** -61.4])
def test_gram_diagonals_with_odd_exponents(torch_cuda, emo, oracle_mod, scale):  # noqa: F811
    """Metric matrices whose Gram diagonal has odd exponents (columns of length `scale` and multiples of it): the unknowns' units
    are powers of two, so twice the metrics and features give the same weights bit for bit, whatever the exponent."""
    n, m, L, P = 12, 6, 5, 40
    B, Tb, Eb = W.microbench_model(41, n, m, L)
    B = B / np.linalg.norm(B, axis=0) * scale * np.array([1.0, 1.5, 1.0, 3.0, 1.0, 0.75])
    feat = W.pack_features(42, B, P, noise=0.1)
    xo, _, _ = oracle_mod.pack_model(B, feat, Tb, Eb)
    x, _, _ = run(torch_cuda, emo, B, feat, Tb, Eb)
    tol = 4e-13 * np.linalg.cond(B) ** 2
    assert (np.abs(x - xo) <= tol * (np.abs(xo).max(axis=1, keepdims=True) + 1e-300)).all()
    x2, _, _ = run(torch_cuda, emo, 2.0 * B, 2.0 * feat, Tb, Eb)
    assert np.array_equal(x2, x)
