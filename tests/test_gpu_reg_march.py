"""The marches with a wake's rings in registers (march_reg.cuh: beam grids,
RK4, FP64 wakes of a given block size; march_reg_ions.cuh: two species) at
every number of rings per thread,
full and ragged last blocks, one block and clusters, against the
global-memory marches that serve more than 4 (2 of each species) rings per thread: from a
scrambled ring state with equal radii and a ring about to cross the axis,
two beams, field queries included.

Tolerance: the FP64 path's 1e-10 of the field's largest value (psi as
psibar = 1 + psi, the form the march takes it in): the same sums in another
association, n 2^-53 of their magnitude apart at most."""
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


def solve(march, rings, threads, cluster):
    from paper_2603_16623_gb300 import wake as wm
    rng = np.random.Generator(np.random.PCG64(rings))
    edges = W.edges_uniform(rings, 4.0)
    beams = [W.Beam(xi=rng.uniform(-0.01, 0.07, m), r=s * np.abs(rng.standard_normal(m)), w=np.full(m, 0.3 / m))
             for m, s in ((2500, 0.4), (300, 0.02))]
    wk = W.Wake("reg", edges, beams, 0.02, 4, integrator="rk4" if march == "rk4" else "ab2",
                ions=(1.0, 100.0) if march == "ions" else None,
                grid_nr=40 if march == "grid" else 600 if march == "wide grid" else 0)
    centre = np.tile(0.5 * (edges[1:] + edges[:-1]), 2 if march == "ions" else 1)
    rho = np.abs(centre + 0.3 * edges[1] * rng.standard_normal(centre.shape[0]))
    if rings > 2:
        rho[0] = rho[2]
    ur = 0.05 * rng.standard_normal(centre.shape[0])
    i = int(np.argmin(rho))
    ur[i] = -2.0 * rho[i] / wk.dxi
    kw = {} if march == "ab2" else {"cluster_ctas": cluster}
    g = wm.Wake.from_workload(wk, precision="fp64", block_threads=threads, flags=wm.WAKE_DUMP_RING_FIELDS, **kw)
    g.set_ring_state(0, rho, ur)
    q = g.fields_at(np.concatenate([[0.0], np.sort(rng.uniform(0.0, 5.0, 300))]))
    g.step_slices(2)
    g.step_slices(2)
    out = {"query": q, "state": dict(zip(("rho", "ur"), g.ring_state())), "dump": g.ring_dumps(),
           "beam": g.beam_fields(), "progress": {"slice, status": np.array(g.progress()[:2], dtype=np.float64)}}
    k = g.launch_config()[1]
    g.close()
    return k, out


@pytest.mark.parametrize("march", ["ab2", "grid", "wide grid", "rk4"])
@pytest.mark.parametrize("rings", [321, 512, 513, 1000, 1024])
def test_register_marches_match_the_global_memory_marches(march, rings):
    k, ref = solve(march, rings, 64, 1)
    assert k > 4
    seen = set()
    for threads, cluster in ((512, 1), (256, 1), (128, 2), (96, 3), (64, 8)):
        if march == "ab2" and cluster > 1:
            continue
        k, got = solve(march, rings, threads, cluster)
        seen.add(k)
        for part in got:
            for f in got[part]:
                one = 1.0 if f == "psi" else 0.0
                assert nerr(one + got[part][f], one + ref[part][f]) < TOL, (threads, cluster, part, f)
    assert seen <= {1, 2, 3, 4} or rings == 1024 and 4 in seen


@pytest.mark.parametrize("cells", [129, 192, 256, 257, 500, 512])
def test_register_two_species_march_matches_the_global_memory_march(cells):
    k, ref = solve("ions", cells, 64, 1)
    assert k > 4
    for threads, cluster in ((512, 1), (256, 1), (128, 2), (96, 3), (64, 8)):
        k, got = solve("ions", cells, threads, cluster)
        assert k <= 4  # (of both species)
        for part in got:
            for f in got[part]:
                one = 1.0 if f == "psi" else 0.0
                assert nerr(one + got[part][f], one + ref[part][f]) < TOL, (threads, cluster, part, f)


@pytest.mark.parametrize("march", ["ab2", "grid", "rk4"])
@pytest.mark.parametrize("rings", [1, 2, 31, 33, 64, 65, 127])
def test_register_marches_on_few_rings(march, rings):
    _, ref = solve(march, rings, 512, 1)
    for threads, cluster in ((64, 1), (64, 2), (64, 8)):
        if march == "ab2" and cluster > 1:
            continue
        _, got = solve(march, rings, threads, cluster)
        for part in got:
            for f in got[part]:
                one = 1.0 if f == "psi" else 0.0
                assert nerr(one + got[part][f], one + ref[part][f]) < TOL, (threads, cluster, part, f)
