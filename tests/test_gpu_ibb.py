"""The paper's own coupling on the GPU (Section 2.4.3: IBB, Eqs. 23-25; Galilean-invariant
momentum exchange; refilling, Eq. 27) against the FP64 CPU oracle.

- Node classes (cell centre inside a particle, binary32 decision) are bit-exact, over a
  trajectory of moving, spinning particles between walls.
- One step from identical populations and velocities: q comes out of the same binary32 bisection
  on both sides, so the populations differ only by the update's arithmetic. Binary64 storage
  matches to 1e-12 of max|f|. Binary32-shifted storage matches to a few binary32 roundings of
  the update (2e-6 of max|f| and of max|f - w rho0| ~ 1e-3 of the link terms).
- Forces and torques from the momentum exchange agree to the same precision.
- The three step schedules and graph replay give identical results.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _need_gpu():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _ibb_workload(storage=1, q=15, walls=4, seed=9):
    from paper_2308_05007_gb300 import inputs as I
    return I.with_(I.ragged(q=q, storage=storage, walls=walls, seed=seed), coupling=1)


def test_ibb_nodes_bit_exact_along_a_trajectory():
    _need_gpu()
    from oracle.oracle import Oracle
    from paper_2308_05007_gb300.rwmi import Simulation
    w = _ibb_workload()
    ora = Oracle.from_workload(w, seed_walkers=False)
    with Simulation.from_workload(w, seed_walkers=False) as sim:
        for t in (0, 5, 17, 40):
            sim.step(t - sim.t)
            assert np.array_equal(sim.nodes(), ora.nodes(t)), f"t={t}"
        assert (sim.nodes() > 0).sum() > 50


def test_ibb_solid_counts_on_demand_equal_the_oracle_and_change_nothing():
    """IBB steps rasterise only bricks and walker masks; rwmi_solid forms the sub-sample counts of
    the current time on demand. They equal the oracle's raster bit for bit, and a run that reads
    them after every few steps keeps the same populations and walkers as one that never does."""
    _need_gpu()
    from oracle.oracle import Oracle
    from paper_2308_05007_gb300.rwmi import Simulation
    w = _ibb_workload(seed=21)
    ora = Oracle.from_workload(w, seed_walkers=False)
    with Simulation.from_workload(w) as a, Simulation.from_workload(w) as b:
        for t in (0, 3, 10, 17):
            a.step(t - a.t)
            b.step(t - b.t)
            ora.step_fluid(t - ora.t)
            cg, og = a.solid()
            co, oo = ora.solid(t)
            assert np.array_equal(cg, co), (t, np.flatnonzero(cg != co)[:10])
            assert np.array_equal(og, oo), t
            assert cg.max() == 64
        b.step(3)
        a.step(3)
        assert np.array_equal(a.populations(), b.populations())
        xa, _ = a.walkers_by_id()
        xb, _ = b.walkers_by_id()
        assert np.array_equal(xa, xb)


@pytest.mark.parametrize("storage,q", [(1, 15), (1, 19), (3, 15), (3, 19)])
def test_ibb_one_step_from_identical_state(storage, q):
    _need_gpu()
    from oracle.oracle import Oracle, lattice
    from paper_2308_05007_gb300.rwmi import Simulation
    w = _ibb_workload(storage=storage, q=q)
    with Simulation.from_workload(w, seed_walkers=False) as sim:
        eg, _ = sim.lattice()
        eo, wts = lattice(q)
        perm = np.array([int(np.where((eg == eo[i]).all(1))[0][0]) for i in range(q)])
        sim.step(11)
        t = sim.t
        f_prev = sim.populations()[perm]
        u_prev = sim.velocity().astype(np.float64)   # the previous update's velocity (u_f, u_ff)
        sim.step(1)
        f_gpu = sim.populations()[perm]
        F_gpu = sim.particle_forces()
        nodes_t = sim.nodes()   # classes of t + 1; the step used those of t
    ora = Oracle.from_workload(w, seed_walkers=False)
    ora.set_populations(f_prev)
    ora.set_velocity(u_prev)
    ora.set_time(t)
    fluid_t = ora.nodes(t) == 0
    ora.step_fluid(1)
    f_ora = ora.populations()
    F_ora = ora.forces()
    assert fluid_t.sum() < ora.n_cells and (ora.nodes(t) != ora.nodes(t - 1)).any()
    err = np.abs(f_gpu - f_ora)
    if storage == 3:
        tol = 1e-12 * np.abs(f_ora).max()
        ftol = 1e-9
    else:
        tol = 2e-6 * np.abs(f_ora).max()
        ftol = 2e-4
    assert err.max() <= tol, (err.max(), tol)
    scale = np.abs(F_ora).max()
    assert np.abs(F_gpu - F_ora).max() <= ftol * scale, (F_gpu, F_ora)
    del nodes_t


def test_ibb_schedules_and_graphs_agree():
    _need_gpu()
    from paper_2308_05007_gb300.rwmi import Simulation
    w = _ibb_workload()
    ref = None
    for overlap in (0, 1, 2):
        for graphs in (False, True):
            with Simulation.from_workload(w, seed_walkers=True, overlap=overlap, use_graphs=graphs) as s:
                s.step(13)
                pos, _ = s.walkers_by_id()
                st = (s.populations(), s.velocity(), pos, s.particle_forces())
            if ref is None:
                ref = st
            else:
                for a, b in zip(ref[:3], st[:3]):
                    assert np.array_equal(a, b), (overlap, graphs)
                np.testing.assert_allclose(ref[3], st[3], rtol=1e-12, atol=1e-12 * np.abs(ref[3]).max())


@pytest.mark.parametrize("storage,q", [(1, 15), (3, 19)])
def test_ibb_links_beyond_the_list_capacity_give_the_same_step(storage, q, monkeypatch):
    """A link list of 64 entries (RWMI_IBB_LINK_CAP) sends almost every link cell to the overflow
    slots: populations, velocities and walkers stay bit-identical to the full-size list, forces
    agree to the order of their FP64 atomics, and rwmi_sync reports no error."""
    _need_gpu()
    from paper_2308_05007_gb300.rwmi import Simulation
    w = _ibb_workload(storage=storage, q=q, seed=13)
    states = []
    for cap in (None, "64"):
        if cap is None:
            monkeypatch.delenv("RWMI_IBB_LINK_CAP", raising=False)
        else:
            monkeypatch.setenv("RWMI_IBB_LINK_CAP", cap)
        with Simulation.from_workload(w, seed_walkers=True) as s:
            s.step(17)
            pos, _ = s.walkers_by_id()
            states.append((s.populations(), s.velocity(), pos, s.particle_forces()))
            assert s.sync() == 0
    monkeypatch.delenv("RWMI_IBB_LINK_CAP", raising=False)
    for a, b in zip(states[0][:3], states[1][:3]):
        assert np.array_equal(a, b)
    F0, F1 = states[0][3], states[1][3]
    assert np.abs(F0).max() > 0
    np.testing.assert_allclose(F1, F0, rtol=1e-12, atol=1e-12 * np.abs(F0).max())


def test_ibb_rejects_other_storages():
    _need_gpu()
    from paper_2308_05007_gb300.rwmi import RwmiError, Simulation
    w = _ibb_workload(storage=2)
    with pytest.raises(RwmiError):
        Simulation.from_workload(w, seed_walkers=False)


@pytest.mark.parametrize("storage,tol", [(3, 1e-6), (1, 5e-5)])
def test_ibb_overlapping_pair_force_is_galilean_invariant(storage, tol):
    """The oracle's Galilean-invariance pin, run through the GPU's IBB path: two overlapping
    spheres co-moving with a uniform stream at U along their line of centres feel, on each
    particle, the force along U of the same pair at rest in still fluid (the pressure on the
    open piece of surface each particle owns, about 22). A plain momentum exchange would differ
    by rho U^2 A = 0.1 here. The fluid velocities u_f, u_ff reach the link update in binary32 in
    every storage (the velocity field is binary32), so u_f - u_w is not zero but about
    2^-24 U: over ~2000 links with terms of order w rho 3 (u_f - u_w) that leaves up to ~1e-6
    with binary64 storage (5e-8 measured). Binary32-shifted storage adds its rounding of the
    link terms: about 1e-8 per link of order 0.1, random in sign, ~5e-6 measured."""
    _need_gpu()
    from paper_2308_05007_gb300 import inputs as I
    from paper_2308_05007_gb300.rwmi import Simulation
    from test_oracle_ibb import _overlapping_pair
    forces = {}
    for U in (0.0, 0.04):
        w = I.with_(_overlapping_pair(U, q=15), storage=storage)
        with Simulation.from_workload(w, seed_walkers=False) as sim:
            sim.step(1)
            forces[U] = sim.particle_forces()[:, :3]
    fr, fm = forces[0.0], forces[0.04]
    print(f"IBB storage {storage}: |F_x(U) - F_x(0)| = {np.abs(fm[:, 0] - fr[:, 0]).max():.2e}")
    assert fr[0, 0] > 15.0 and fr[1, 0] < -15.0
    np.testing.assert_allclose(fm[:, 0], fr[:, 0], rtol=0, atol=tol)


def _shapes(name):
    """dims, walls and particles [(origin, centres, sigma, k range)] of a link test."""
    return {
        "one_centre": ((26, 24, 22), 4, [((13.2, 11.7, 11.1), 1, 0.0, (30.0, 30.0))]),
        "small_weights": ((24, 26, 28), 0, [((9.3, 12.2, 14.4), 5, 1.0, (0.4, 0.9)), ((18.4, 17.1, 8.2), 2, 0.6, (1.0, 2.0))]),
        "across_faces": ((22, 21, 20), 0, [((0.4, 20.6, 0.2), 4, 1.2, (3.0, 6.0))]),       # rows of 22 cells: refilled cell by cell
        "box_of_a_particle": ((15, 14, 16), 0, [((7.0, 7.0, 8.0), 3, 1.0, (4.0, 6.0))]),   # points near half the box
        "many_centres": ((44, 40, 36), 4, [((22.0, 20.0, 18.0), 40, 4.0, (0.5, 1.5))]),    # uneven surface, grazing links
        "long_box": ((600, 18, 16), 0, [((590.3, 9.2, 8.1), 3, 1.0, (4.0, 6.0)), ((300.6, 8.8, 7.9), 2, 1.0, (6.0, 9.0))]),
    }[name]


@pytest.mark.parametrize("name", ["one_centre", "small_weights", "across_faces", "box_of_a_particle", "many_centres",
                                  "long_box"])
@pytest.mark.parametrize("q", [15, 19])
def test_ibb_link_distances_over_shapes(name, q):
    """Binary64 storage, one step from the oracle's own state: the update depends on q of every link,
    and a q off by one bisection bracket (6e-8) would move a population by some 1e-9 of the largest,
    a thousand times the bound."""
    _need_gpu()
    from oracle.oracle import Oracle, lattice
    from paper_2308_05007_gb300 import inputs as I
    from paper_2308_05007_gb300.rwmi import Simulation
    dims, walls, parts = _shapes(name)
    rng = np.random.default_rng(4)
    cb = [rng.normal(0.0, s, (n, 3)).astype(np.float32) for _, n, s, _ in parts]
    k = [rng.uniform(*r, n).astype(np.float32) for _, n, _, r in parts]
    P = len(parts)
    mb = I.Metaballs(center_offsets=np.cumsum([0] + [len(v) for v in k]).astype(np.int32), centers_body=np.concatenate(cb),
                     k=np.concatenate(k), origin=np.array([p[0] for p in parts]), amplitude=np.tile([1.5, 0.7, 0.4], (P, 1)),
                     period=np.full(P, 150.0), phase=np.full(P, 0.3), omega=np.tile([0.002, 0.001, 0.004], (P, 1)))
    w = I.Workload(name=name, dims=dims, tau=0.75, D=0.02, seed=1, q=q, wall_mask=walls, body_force=(2e-5, 5e-6, 0.0),
                   metaballs=mb, storage=3, coupling=1)
    with Simulation.from_workload(w, seed_walkers=False) as sim:
        eg, _ = sim.lattice()
        eo, _ = lattice(q)
        perm = np.array([int(np.where((eg == eo[i]).all(1))[0][0]) for i in range(q)])
        for steps in (3, 4):
            sim.step(steps)
            t, f_prev, u_prev = sim.t, sim.populations()[perm], sim.velocity().astype(np.float64)
            sim.step(1)
            f_gpu, F_gpu = sim.populations()[perm], sim.particle_forces()
            ora = Oracle.from_workload(w, seed_walkers=False)
            ora.set_populations(f_prev)
            ora.set_velocity(u_prev)
            ora.set_time(t)
            ora.step_fluid(1)
            f_ora, F_ora = ora.populations(), ora.forces()
            assert np.abs(f_gpu - f_ora).max() <= 1e-12 * np.abs(f_ora).max()
            assert np.abs(F_gpu - F_ora).max() <= 1e-9 * np.abs(F_ora).max()
            assert np.abs(F_ora).max() > 0.0
