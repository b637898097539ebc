"""The node classes that the raster leaves for the IBB update (read back as they are, completed with 0
in bricks without a particle) against the oracle, bit for bit: staged candidates and the unstaged
paths (more than 8 candidates, more than 192 control points, an overflowing list), walls, periodic
images, sizes that are no multiple of a brick or of 8 cells, both time parities, eager and captured
runs of one and of several steps, and after a read-back of counts, which rasters once more."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2308_05007_gb300 import inputs as I
from test_gpu_raster_pieces import CASES, _metaballs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("graphs", [True, False])
def test_step_classes_bit_exact(name, graphs):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_05007_gb300.rwmi import Simulation
    dims, walls, particles = CASES[name]
    w = I.Workload(name=name, dims=dims, tau=0.8, D=0.01, seed=1, wall_mask=walls, coupling=1,
                   metaballs=_metaballs(particles(np.random.default_rng(3))))
    with Simulation.from_workload(w, seed_walkers=False, use_graphs=graphs) as sim:
        ora = Oracle.from_workload(w, seed_walkers=False)
        for t in (0, 1, 2, 7, 12):
            sim.step(t - sim.t)
            got, want = sim.nodes().ravel(), ora.nodes(t).ravel()
            assert np.array_equal(got, want), (t, np.flatnonzero(got != want)[:10])
            assert (got > 0).any()
        sim.solid()
        assert np.array_equal(sim.nodes().ravel(), want)
