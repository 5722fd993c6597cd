"""The double-precision on-chip march (march_f64.cuh) against the one-block
march that a given block size selects: ring counts at the edges of its shapes
(rings per thread 1, 2, 4; one block, full and ragged last blocks, the largest
cluster), from a scrambled ring state (ranks over long distances, radii at
equal values, a ring about to cross the axis), with a beam denser than its
staged radii and without one, field queries included.

Tolerance: the FP64 path's 1e-10 of the field's largest value.  Both marches
evaluate the same sums in another order; at 8192 rings a sum of n terms
differs by at most n 2^-53 = 1e-12 of its magnitude, three steps apart.  psi is
compared as psibar = 1 + psi: of an almost unperturbed plasma it is 1e-5, left
over from sums of order 10."""
import numpy as np
import pytest

from paper_2603_16623_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-10


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2603_16623_gb300 import wake
    wake.load()
    yield


def nerr(a, b):
    return np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300) if a.size else 0.0


@pytest.mark.parametrize("particles", [0, 6000])
@pytest.mark.parametrize("rings", [1, 2, 31, 32, 33, 127, 128, 129, 255, 257, 511, 512, 513, 769, 2000, 4095, 4096,
                                   4097, 5000, 8191, 8192])
def test_f64_march_matches_the_one_block_march(rings, particles):
    from paper_2603_16623_gb300 import wake as wm
    rng = np.random.Generator(np.random.PCG64(rings))
    edges = W.edges_uniform(rings, 4.0)
    beam = W.Beam(xi=rng.uniform(-0.01, 0.05, particles), r=0.4 * np.abs(rng.standard_normal(particles)),
                  w=np.full(particles, 0.2 / max(particles, 1)))
    wk = W.Wake("f64", edges, [beam], 0.02, 3)
    centre = 0.5 * (edges[1:] + edges[:-1])
    rho = centre + 0.2 * np.diff(edges) * rng.standard_normal(rings)
    rho = np.abs(rho[rng.permutation(rings)] if rings <= 1000 else rho)
    if rings > 2:
        rho[0] = rho[2]
    ur = 0.05 * rng.standard_normal(rings)
    i = int(np.argmin(rho))
    ur[i] = -2.0 * rho[i] / wk.dxi
    x = np.concatenate([[0.0], np.sort(rng.uniform(0.0, 5.0, 500))])
    out = []
    for threads in (0, 256):
        g = wm.Wake.from_workload(wk, precision="fp64", block_threads=threads, flags=wm.WAKE_DUMP_RING_FIELDS)
        assert g.launch_config()[2] == 1 or threads == 0
        g.set_ring_state(0, rho, ur)
        q = g.fields_at(x)
        g.step_slices(3)
        rings_ = dict(zip(("rho", "ur", "fr", "fu"), g.ring_state(history=True)))
        out.append({"progress": g.progress()[:2], "query": q, "state": rings_, "dump": g.ring_dumps(),
                    "beam": g.beam_fields()})
        g.close()
    a, b = out
    assert a["progress"] == b["progress"]
    for part in ("query", "state", "dump", "beam"):
        for k in a[part]:
            one = 1.0 if k == "psi" else 0.0  # psi as psibar = 1 + psi, the form the march takes it in
            assert nerr(one + a[part][k], one + b[part][k]) < TOL, (part, k)


def test_f64_shapes():
    """Blocks of at most 128 threads, at most 16 of them, none without a ring."""
    from paper_2603_16623_gb300 import wake as wm
    for rings in (1, 200, 512, 513, 2000, 4096, 4097, 8192):
        g = wm.Wake(W.edges_uniform(rings, 4.0), [], 0.01, 4, precision="fp64")
        t, k, cl = g.launch_config()
        assert t <= 128 and cl <= 16 and t * k * cl >= rings and (cl == 1 or t * k * (cl - 1) < rings)
        assert k == (1 if rings <= 512 else 2 if rings <= 4096 else 4)
        g.close()
