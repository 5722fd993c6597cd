"""The binning's two chunk sizes give the same beam: particles outside the window carry a wake over the
line between them (152 x 256 x 16 particles) and change no field of the others, bitwise; equal radii,
radii of 0 and -0 among them."""
import numpy as np
import pytest

from paper_2603_16623_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LINE = 152 * 256 * 16


@pytest.fixture(scope="module", autouse=True)
def _gpu():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2603_16623_gb300 import wake
    wake.load()
    yield


@pytest.mark.parametrize("n_in", [1, 1023, 1025, 40_000])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_chunks_on_both_sides_of_the_line(n_in, precision):
    from paper_2603_16623_gb300 import wake as wm
    rng = np.random.default_rng(n_in)
    xi = rng.uniform(0.0, 0.49, n_in)
    r = np.round(rng.uniform(0.0, 1.0, n_in), 3)  # (many equal)
    r[::97] = 0.0
    r[::193] = -0.0
    got = []
    for n_out in (0, LINE - n_in, LINE + 1 - n_in):
        b = W.Beam(xi=np.concatenate([xi, np.full(n_out, 9.0)]), r=np.concatenate([r, np.full(n_out, 0.5)]),
                   w=np.full(n_in + n_out, 1e-7))
        g = wm.Wake.from_workload(W.Wake("bins", W.edges_uniform(64, 3.0), [b], 0.01, 50), precision=precision)
        g.step_slices(50)
        f = g.beam_fields()
        got.append({k: v[:n_in] for k, v in f.items()})
        assert all(not np.any(v[n_in:]) for v in f.values())
        g.close()
    for o in got[1:]:
        for k in got[0]:
            assert np.array_equal(got[0][k], o[k]), k
