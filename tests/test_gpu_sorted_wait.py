"""The raster's wait for the resolve pass, which runs take once their walkers have been sorted: no bit
differs from one stream, with walkers that leave pass 1's resident grid (5 blocks of 256 per SM) one
block short, fill it, or loop in it, in captured and eager runs that begin before the first sort, and
in the branches of a batch."""
import numpy as np
import pytest

from paper_2308_05007_gb300 import inputs as I
from test_gpu_resolve import CASES, _metaballs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("blocks", [-1, 0, 3])
def test_sorted_runs_equal_one_stream(blocks):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_05007_gb300.rwmi import BATCH_BRANCHES, Batch, Simulation
    n = 256 * (5 * torch.cuda.get_device_properties(0).multi_processor_count + blocks) - 7
    dims, walls, particles = CASES["remainder"]
    w = I.Workload(name="grid", dims=dims, tau=0.8, D=0.01, seed=7, wall_mask=walls, n_walkers=n, sort_interval=4,
                   walker_box=((0.0, 0.0, 0.0), tuple(float(v) for v in dims)), metaballs=_metaballs(particles))
    runs = []
    for overlap, graphs in ((0, 1), (2, 1), (2, 0)):
        with Simulation.from_workload(w, overlap=overlap, use_graphs=graphs) as sim:
            for k in (3, 9, 16, 4):
                sim.step(k)
            runs.append((sim.walkers_by_id()[0], sim.velocity(), sim.solid()[0]))
    sims = [Simulation.from_workload(w) for _ in range(2)]
    with Batch(sims, mode=BATCH_BRANCHES) as batch:
        for k in (4, 12, 16):
            batch.step(k)
        batch.sync()
        runs += [(s.walkers_by_id()[0], s.velocity(), s.solid()[0]) for s in sims]
    for s in sims:
        s.close()
    for other in runs[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(runs[0], other))
