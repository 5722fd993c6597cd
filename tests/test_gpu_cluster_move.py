"""The cluster march's re-sort when rings cross from any block to any other: fields and ring state of a
mixed wake on a cluster against the same wake in one block (its re-sort knows no other block), from the
same unsorted ring state.  Both take the same ring values in the same order; what differs is where the
float-float sums and the float matrix products are cut, a few units of 2^-24 of the largest value."""
import numpy as np
import pytest

from paper_2603_16623_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 1e-5  # norm-wise: up to 16 x 16 partial matrix products in float, 256 x 2^-24 = 1.5e-5 at worst, ~sqrt of that


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2603_16623_gb300 import wake
    wake.load()
    yield


def nerr(a, b):
    return float(np.max(np.abs(np.asarray(a, dtype=np.float64) - b)) / np.max(np.abs(b)))


def _radii(n, order, rng):
    c = (np.arange(n) + 0.5) * (6.0 / n)
    if order == "reversed":      # every ring leaves its block: more than a block's copies hold at once
        return c[::-1].copy()
    if order == "shuffled":
        return rng.permutation(c)
    if order == "ties":          # each radius twice, in different blocks
        return np.concatenate([c[:(n + 1) // 2], c[:n // 2]])
    c[[0, n - 1]] = c[[n - 1, 0]]  # "outliers": one ring crosses every block, each way
    c[n // 2], c[1] = c[1], c[n // 2]
    return c


# (rings, rings per thread, blocks): small blocks with a short last one, the automatic shapes' kinds, 8 per thread
@pytest.mark.parametrize("n,k,cl", [(300, 2, 5), (2100, 4, 3), (4000, 4, 6), (4000, 8, 2), (4096, 2, 16)])
@pytest.mark.parametrize("order", ["reversed", "shuffled", "ties", "outliers"])
def test_rings_cross_between_blocks(n, k, cl, order):
    from paper_2603_16623_gb300 import wake as wm
    rng = np.random.default_rng(n + cl)
    wk = W.Wake("move", W.edges_uniform(n, 6.0), [W.gaussian_beam(5_000, 0.02, 0.3, 0.2, 0.4, seed=n)], 0.01, 60,
                density=0.005)
    rho, u = _radii(n, order, rng), 0.05 * rng.standard_normal(n)
    q = rng.uniform(0.0, 6.5, 500)
    got = []
    for kw in (dict(rings_per_thread=k, cluster_ctas=cl), dict(rings_per_thread=8, cluster_ctas=1)):
        g = wm.Wake.from_workload(wk, precision="mixed", **kw)
        assert g.launch_config()[2] == kw["cluster_ctas"]
        g.set_ring_state(30, rho, u)
        f = g.fields_at(q)
        g.step_slices(6)
        assert g.progress()[:2] == (36, 0)
        got.append((f, g.ring_state()))
        g.close()
    for key in ("ez", "wr", "bt", "psi"):
        assert nerr(got[0][0][key], got[1][0][key]) < TOL, key
    for a, b in zip(got[0][1], got[1][1]):
        assert nerr(a, b) < TOL
