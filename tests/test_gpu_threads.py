"""Simulations of different sizes driven from several host threads at once: the kernels they share
have one limit of dynamic shared memory, which no launch may lower under another."""
import threading

import pytest

import synth

ss = pytest.importorskip("paper_1808_06381_gb300")

pytestmark = pytest.mark.gpu


def _sim(n, precision):
    L = synth.box_length(n)
    pos = synth.uniform_positions(n, (L,) * 3, n)
    sim = ss.Simulation(n, (L,) * 3, ss.kappa_from_kappa_tau(0.5), seed=5, precision=precision, warm_start="none",
                        cg_tol=1e-8, positions=pos, use_torch_stream=False)
    sim.set_positions(pos, 0.3 * L)
    sim.build_neighbors()
    sim.assemble()
    return sim


def _run(jobs):
    """Each job in its own thread; the first exception, if any."""
    errors, barrier = [], threading.Barrier(len(jobs))

    def work(job):
        barrier.wait()
        try:
            job()
        except Exception as e:   # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    return errors


# sizes that take the same kernel with different shared-memory sizes
@pytest.mark.parametrize("precision,sizes", [("mixed", (3000, 60000)), ("fp64", (8000, 24000))])
def test_solves_of_different_sizes_from_several_threads(precision, sizes):
    sims = [_sim(n, precision) for n in sizes for _ in range(2)]

    def job(sim):
        def run():
            for _ in range(300):
                info = sim.solve_velocities()
                assert info["status"] == 0, info
        return run

    errors = _run([job(s) for s in sims])
    for s in sims:
        s.close()
    assert not errors, errors[0]


def test_structure_factors_of_different_grids_from_several_threads():
    sims = [_sim(3000, "mixed") for _ in range(4)]
    grids = (2048, 4096, 2048, 4096)

    def job(sim, grid):
        def run():
            for _ in range(200):
                sim.structure_factor(3, 3, grid=grid)
        return run

    errors = _run([job(s, g) for s, g in zip(sims, grids)])
    for s in sims:
        s.close()
    assert not errors, errors[0]
