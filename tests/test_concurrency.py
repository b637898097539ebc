"""Contexts that step side by side share the GPU: the request loop tells each context how many there
are before it steps, and the results do not depend on it."""
import numpy as np
import pytest

from paper_2308_05007_gb300 import inputs as I
from paper_2308_05007_gb300.serve import Server
from test_serve_host import Clock, fake_backend, req


def test_loop_tells_each_context_how_many_there_are():
    clock = Clock()
    backend, log, _ = fake_backend(clock)
    told = []
    backend.share = lambda sim, contexts: told.append((sim.w.name, contexts, len(log)))
    srv = Server(backend, budget_bytes=1 << 40, max_active=3, chunk_cell_updates=1, clock=clock, sleep=clock.sleep)
    srv.run([req(0, 0.0, 8, 16), req(1, 0.0, 8, 32), req(2, 0.0, 8, 32), req(3, 0.0, 8, 16)])
    steps = [k for k, e in enumerate(log) if e[0] == "step"]
    assert [at for _, _, at in told] == steps                    # right before each step
    assert [n for n, _, _ in told] == [log[k][1] for k in steps]  # of the same context
    counts = [c for _, c, _ in told]
    assert counts[:3] == [3, 3, 3] and all(1 <= c <= 3 for c in counts) and len(counts) == 6


@pytest.mark.gpu
@pytest.mark.parametrize("coupling", [0, 1])
def test_results_do_not_depend_on_the_count(coupling):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2308_05007_gb300.rwmi import RwmiError, Simulation
    w = I.with_(I.ragged(dims=(67, 61, 58), n_particles=3, n_walkers=60_000, k_range=(9.0, 20.0), sigma=2.0),
                coupling=coupling)
    runs = []
    for counts in ((1,), (2,), (5, 16, 1000, 1)):
        with Simulation.from_workload(w) as sim:
            for k in range(8):
                sim.set_concurrency(counts[k % len(counts)])
                sim.step(16)
            runs.append((sim.walkers_by_id()[0], sim.velocity(), sim.solid()[0]))
            with pytest.raises(RwmiError):
                sim.set_concurrency(0)
    for other in runs[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(runs[0], other))
