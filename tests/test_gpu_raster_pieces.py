"""The rasteriser's split of bricks into pieces (whole bricks, slices, parts of slices) and its staged
and unstaged candidate paths against the oracle: counts and owners are exact integers, so they are
compared bit for bit. The brick lists run from a handful (a brick in 64 pieces) to beyond four
per resident warp (whole bricks)."""
import numpy as np
import pytest

from oracle.oracle import Oracle
from paper_2308_05007_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _metaballs(particles):
    """particles: list of (origin, centres [n, 3], k [n]); all oscillate and spin slowly."""
    P = len(particles)
    off = np.cumsum([0] + [len(p[2]) for p in particles]).astype(np.int32)
    return I.Metaballs(
        center_offsets=off, centers_body=np.concatenate([np.reshape(p[1], (-1, 3)) for p in particles]).astype(np.float32),
        k=np.concatenate([np.asarray(p[2]) for p in particles]).astype(np.float32),
        origin=np.array([p[0] for p in particles], np.float64), amplitude=np.tile([0.4, 0.2, 0.1], (P, 1)),
        period=np.full(P, 40.0), phase=np.full(P, 0.2), omega=np.tile([0.0, 0.0, 0.003], (P, 1)))


def _ball(rng, origin, n, spread, ksum):
    return origin, rng.normal(0.0, spread, (n, 3)), np.full(n, ksum / n)


CASES = {   # dims, walls, particles; the comment gives the bricks and the pieces a brick is cut into
    "one_brick": ((7, 5, 8), 7, lambda r: [_ball(r, (3.0, 2.5, 4.0), 1, 0.0, 5.0)]),                     # 1: 64
    "odd_periodic": ((17, 15, 9), 0, lambda r: [_ball(r, (1.0, 14.0, 4.0), 3, 0.8, 8.0)]),               # 12: 64
    "small_walled": ((40, 35, 27), 4, lambda r: [_ball(r, (9.0, 9.0, 13.0), 5, 1.5, 30.0),
                                                  _ball(r, (21.0, 12.0, 13.0), 2, 1.0, 30.0)]),          # ~100: 64
    "touching": ((47, 46, 45), 0, lambda r: [_ball(r, (x, y, 22.5), 3, 2.0, 60.0)
                                             for x in (14.0, 26.0) for y in (12.0, 24.0)]),              # ~200: 32
    "slices_16": ((66, 59, 70), 0, lambda r: [_ball(r, (30.0, 30.0, 30.0), 4, 3.0, 500.0)]),             # ~600: 16 or 8
    "slices_4": ((100, 97, 104), 7, lambda r: [_ball(r, (20.0, 30.0, 40.0), 2, 3.0, 9000.0)]),           # ~2000: 4
    "slices_2": ((121, 119, 120), 7, lambda r: [_ball(r, (60.0, 60.0, 60.0), 1, 0.0, 7000.0)]),          # ~3300: 2
    "whole": ((137, 131, 136), 7, lambda r: [_ball(r, (70.0, 60.0, 70.0), 3, 4.0, 9000.0)]),             # ~5200: 1
    "many_centres": ((30, 28, 26), 4, lambda r: [_ball(r, (15.0, 14.0, 13.0), 193, 2.0, 40.0)]),         # not staged
    "nine_in_a_brick": ((32, 32, 30), 4, lambda r: [_ball(r, (13.0 + 0.7 * m, 16.0, 15.0), 2, 0.5, 6.0 + m)
                                                    for m in range(9)]),                                 # not staged
    "overflowing": ((32, 30, 30), 4, lambda r: [_ball(r, (12.0 + 0.4 * m, 15.0, 15.0), 1, 0.3, 5.0 + m)
                                                for m in range(18)]),                                    # list too long
}


@pytest.mark.parametrize("name", list(CASES))
def test_raster_pieces_bit_exact(name):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_05007_gb300.rwmi import Simulation
    dims, walls, particles = CASES[name]
    w = I.Workload(name=name, dims=dims, tau=0.8, D=0.01, seed=1, wall_mask=walls,
                   metaballs=_metaballs(particles(np.random.default_rng(3))))
    with Simulation.from_workload(w, seed_walkers=False) as sim:
        ora = Oracle.from_workload(w, seed_walkers=False)
        for t in (0, 1, 2):   # set-up's raster, then both time parities' rasters of the step
            if t:
                sim.step(1)
            cg, og = sim.solid()
            co, oo = ora.solid(t)
            assert np.array_equal(cg, co), (t, np.flatnonzero(cg != co)[:10])
            assert np.array_equal(og, oo)
