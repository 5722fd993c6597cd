"""A ring history that a push turns into a radius without a number, while other rings cross from end to end in the same
push: every march sorts what there is (the places stay a permutation of the rings, NaN radii last) and the guard stops
the wake at that slice with WAKE_ENONFINITE; the other wake of the batch and the handle's next solve are untouched."""
import numpy as np
import pytest

from paper_2603_16623_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2603_16623_gb300 import wake
    wake.load()
    yield


# one block at 2, 4, 8 rings per thread; clusters at 4, 2, 8; FP64 on chip (one block, a cluster); the register and the
# global-memory marches of every kind
CASES = [
    ("ab2", "mixed", 200, {}), ("ab2", "mixed", 1500, {}), ("ab2", "mixed", 2000, dict(rings_per_thread=8, cluster_ctas=1)),
    ("ab2", "mixed", 3000, {}), ("ab2", "mixed", 2000, dict(rings_per_thread=2, cluster_ctas=4)),
    ("ab2", "mixed", 6000, dict(rings_per_thread=8, cluster_ctas=3)),
    ("ab2", "fp64", 300, {}), ("ab2", "fp64", 3000, {}), ("ab2", "fp64", 500, dict(block_threads=256)),
    ("ab2", "fp64", 500, dict(block_threads=64)),
    ("grid", "mixed", 1500, {}), ("grid", "mixed", 500, dict(block_threads=64, cluster_ctas=1)),
    ("ions", "mixed", 700, {}), ("ions", "mixed", 1500, {}), ("ions", "mixed", 300, dict(block_threads=64, cluster_ctas=1)),
    ("rk4", "mixed", 700, {}), ("rk4", "mixed", 2500, {}), ("rk4", "mixed", 500, dict(block_threads=64, cluster_ctas=1)),
    ("rk4", "fp64", 500, dict(block_threads=64, cluster_ctas=2)),
]


def _wake(march, n, seed):
    return W.Wake("h", W.edges_uniform(n, 4.0), [W.gaussian_beam(2000, 0.5, 0.3, 0.02, 0.04, seed=seed)], 0.01, 8,
                  ions=(1.0, 1836.0) if march == "ions" else None, integrator="rk4" if march == "rk4" else "ab2",
                  grid_nr=24 if march == "grid" else 0)


@pytest.mark.parametrize("march,precision,n,kw", CASES)
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_a_history_without_a_number_stops_the_wake(march, precision, n, kw, value):
    from paper_2603_16623_gb300 import wake as wm
    bad, good = (wm.Wake.from_workload(_wake(march, n, s), precision=precision, **kw) for s in (1, 2))
    good.step_slices(8)
    want, want_state = good.beam_fields(), good.ring_state()
    good.reset()
    bad.step_slices(8)
    whole = bad.beam_fields()

    e = bad.edges
    c = 0.5 * (e[1:] + e[:-1])
    rho = np.concatenate([c, c]) if march == "ions" else c
    ur, fr, fu = np.zeros_like(rho), np.zeros_like(rho), np.zeros_like(rho)
    dxi = 0.01
    for i, to in ((0, n - 1), (n - 1, 0), (n // 3, n // 2)):  # (rho moves by -0.5 dxi f)
        fr[i] = -2.0 * (c[to] - c[i]) / dxi
    hit = [n // 2, 5]
    fr[hit] = value
    if march == "rk4":  # (takes no history: a momentum whose square overflows leaves its stages without numbers)
        ur[hit] = 1e30 if precision == "mixed" else 1e200
    bad.set_ring_state(0, rho, ur, fr, fu)
    wm.wake_batch_step([bad, good], 8)
    at = 0 if march == "rk4" else 1
    assert bad.progress() == (at + 1, wm.WAKE_ENONFINITE, at)
    assert good.progress()[:2] == (8, 0)
    for k, v in good.beam_fields().items():
        assert np.array_equal(v, want[k]) or march == "grid", k  # (the grids' charges are summed in any order)
    if march != "grid":
        assert all(np.array_equal(a, b) for a, b in zip(good.ring_state(), want_state))
    bad.reset()
    bad.step_slices(8)
    assert bad.progress()[:2] == (8, 0)
    if march != "grid":
        assert all(np.array_equal(v, whole[k]) for k, v in bad.beam_fields().items())
    bad.close()
    good.close()
