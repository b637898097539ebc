"""The resolve pass's warp-per-walker path (lanes over control points) against the oracle, with
walkers only in cells at a particle's surface: control points that fill no warp, exactly one, and
several with a remainder; brick lists of nine particles and lists that overflow; walls and periodic
images. Tolerance: at coordinates up to 32 a position carries 2e-6 (binary32) and a crossing
another 1e-6 / |grad f| ~ 2e-6, so 2e-5 per coordinate holds with a factor of five; a walker may
decide otherwise than the oracle when f lies within ~1e-6 of 1, i.e. within ~2e-6 cells of a surface
that steps of ~0.1 cells cross, about 2e-5 of the walkers: 1e-3 leaves a factor of fifty."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2308_05007_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _metaballs(particles):
    """particles: list of (origin, number of control points, spread, sum of k)."""
    rng = np.random.default_rng(5)
    P, n = len(particles), np.array([p[1] for p in particles])
    return I.Metaballs(
        center_offsets=np.concatenate([[0], np.cumsum(n)]).astype(np.int32),
        centers_body=np.concatenate([rng.normal(0.0, p[2], (p[1], 3)) for p in particles]).astype(np.float32),
        k=np.concatenate([np.full(p[1], p[3] / p[1]) for p in particles]).astype(np.float32),
        origin=np.array([p[0] for p in particles], np.float64), amplitude=np.tile([0.4, 0.2, 0.1], (P, 1)),
        period=np.full(P, 40.0), phase=np.full(P, 0.2), omega=np.tile([0.0, 0.0, 0.003], (P, 1)))


CASES = {   # dims, walls, particles
    "one_centre": ((13, 11, 9), 7, [((6.0, 5.0, 4.0), 1, 0.0, 5.0)]),
    "across_the_boundary": ((17, 15, 9), 0, [((1.0, 14.0, 4.0), 3, 0.8, 8.0)]),
    "one_warp": ((30, 28, 26), 4, [((15.0, 14.0, 13.0), 32, 2.0, 40.0)]),
    "remainder": ((30, 28, 26), 0, [((15.0, 14.0, 13.0), 33, 2.0, 40.0)]),
    "many_centres": ((30, 28, 26), 4, [((15.0, 14.0, 13.0), 193, 2.0, 40.0)]),
    "nine_in_a_brick": ((32, 32, 30), 4, [((13.0 + 0.7 * m, 16.0, 15.0), 2, 0.5, 6.0 + m) for m in range(9)]),
    "overflowing": ((32, 30, 30), 4, [((12.0 + 0.4 * m, 15.0, 15.0), 1, 0.3, 5.0 + m) for m in range(18)]),
}


@pytest.mark.parametrize("name", list(CASES))
def test_walkers_at_surfaces_match_the_oracle(name):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_05007_gb300.rwmi import Simulation
    dims, walls, particles = CASES[name]
    w = I.Workload(name=name, dims=dims, tau=0.8, D=0.01, seed=7, wall_mask=walls, n_walkers=200_000,
                   walker_box=((0.0, 0.0, 0.0), tuple(float(n) for n in dims)),
                   metaballs=_metaballs(particles))
    with Simulation.from_workload(w) as sim:
        x, _ = sim.walkers_by_id()
        ora = Oracle.from_workload(w, seed_walkers=False)
        count = np.asarray(sim.solid()[0]).ravel()
        x = np.ascontiguousarray(x[(lambda c: (c > 0) & (c < 64))(count[ora.bin_positions(x)])])
        assert len(x) > 1000
        sim.set_walkers(x)
        for _ in range(2):   # both time parities of the particles
            x_prev, _ = sim.walkers_by_id()
            t = sim.t
            sim.step(1)
            x_next, _ = sim.walkers_by_id()
            ora.set_velocity(sim.velocity().astype(np.float64))
            ora.set_time(t)
            xo = ora.walkers_advance(x_prev.astype(np.float64), np.arange(len(x_prev), dtype=np.uint32))
            d = np.abs(x_next - xo).max(1)
            assert (d > 2e-5).mean() <= 1e-3, np.sort(d)[-5:]


@pytest.mark.parametrize("blocks", [-1, 0, 3])
def test_raster_waits_for_resolve_pass(blocks):
    """Walkers that leave pass 1's resident grid (5 blocks of 256 per SM) one block short, fill it, or
    loop in it: the raster's wait for the resolve pass changes no bit against one stream, in
    captured and in eager runs of several steps."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_05007_gb300.rwmi import Simulation
    n = 256 * (5 * torch.cuda.get_device_properties(0).multi_processor_count + blocks) - 7
    dims, walls, particles = CASES["remainder"]
    w = I.Workload(name="grid", dims=dims, tau=0.8, D=0.01, seed=7, wall_mask=walls, n_walkers=n,
                   walker_box=((0.0, 0.0, 0.0), tuple(float(v) for v in dims)), metaballs=_metaballs(particles))
    runs = []
    for overlap, graphs in ((0, 1), (2, 1), (2, 0)):
        with Simulation.from_workload(w, overlap=overlap, use_graphs=graphs) as sim:
            for k in (9, 16, 5):
                sim.step(k)
            runs.append((sim.walkers_by_id()[0], sim.velocity(), sim.solid()[0]))
    for other in runs[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(runs[0], other))
