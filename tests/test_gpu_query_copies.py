"""Field queries answered by several blocks (or clusters), each solving the slice and taking its share
of the radii: the same values, bitwise, as radii asked a few at a time (one block), at the edges of
the shares, and a march that goes on as if nothing had been asked."""
import numpy as np
import pytest

from paper_2603_16623_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FIELDS = ("ez", "wr", "bt", "psi")


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2603_16623_gb300 import wake
    wake.load()
    yield


def _wake(n_rings):
    from paper_2603_16623_gb300 import wake as wm
    wk = W.Wake("q", W.edges_uniform(n_rings, 6.0), [W.gaussian_beam(20_000, 2.0, 0.3, 0.2, 0.8, seed=n_rings)],
                0.01, 120)
    return wm.Wake.from_workload(wk, precision="mixed")


# 200 rings: one block of 2 rings per thread; 2000: one of 4; 5000: clusters of five blocks
@pytest.mark.parametrize("n_rings", [200, 2000, 5000])
def test_radii_shared_over_blocks(n_rings):
    import torch
    g, h = _wake(n_rings), _wake(n_rings)
    threads = g.launch_config()[0]
    g.step_slices(70)
    h.step_slices(70)
    r = np.random.default_rng(n_rings).uniform(0.0, 7.0, 153 * threads + 1)
    r[:3] = (0.0, 1e-6, 6.0)
    few = [g.fields_at(r[i:i + 31]) for i in range(0, 8 * 31, 31)]
    few = {k: np.concatenate([f[k] for f in few]) for k in FIELDS}
    for n in (1, threads, threads + 1, r.size):
        got = g.fields_at(r[:n])
        out = {k: torch.full((n,), -7.0, dtype=torch.float32, device="cuda") for k in FIELDS}
        g.fields_at_device(torch.from_numpy(r[:n].copy()).cuda(), out)
        for k in FIELDS:
            assert np.array_equal(out[k].cpu().numpy(), got[k]), (n, k)
            m = min(n, few[k].size)
            assert np.array_equal(got[k][:m], few[k][:m]), (n, k)
    assert g.progress()[0] == 70
    g.step_slices(50)
    h.step_slices(50)
    for a, b in zip(g.ring_state(history=True), h.ring_state(history=True)):
        assert np.array_equal(a, b)
    g.close()
    h.close()
