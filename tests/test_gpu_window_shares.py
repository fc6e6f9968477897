"""Windows shared out by cost (streaming mixed solve, FP64 solve of large systems, batch): a
system whose first windows hold most of the entries, fewer windows than blocks, and one window."""
import numpy as np
import pytest

import oracle
import synth

ss = pytest.importorskip("paper_1808_06381_gb300")

pytestmark = pytest.mark.gpu


def _system(n, knot, seed):
    L = max(synth.box_length(n), 3.01)
    pos = synth.uniform_positions(n, (L,) * 3, seed)
    pos[:knot] = 0.5 * L + 0.5 * (pos[:knot] / L - 0.5)
    return pos, L


def _residual(n, pos, L, v, step=0):
    p = oracle.Params(n=n, L=(L,) * 3, kappa=oracle.kappa_from_kappa_tau(0.5), seed=9)
    sysr = oracle.assemble(p, pos, oracle.neighbors(p, pos, 0.0, "cells" if n > 5000 else "auto"),
                           oracle.noise(9, step, np.arange(n)), 0.0)
    return np.linalg.norm(sysr.b - sysr.matvec(v)) / np.linalg.norm(sysr.b)


# The solve meets tol on its own matrix; the oracle's differs by rounding (1e-13 of ||b||, FP64) or
# by the 2^-48 representation (~1e-12 relative entries, 2e-11 of ||b||).
@pytest.mark.parametrize("precision,n,knot", [("mixed", 200, 0), ("mixed", 257, 0), ("mixed", 40000, 900),
                                              ("mixed", 160000, 600), ("fp64", 90000, 600)])
def test_solve_with_unequal_windows(precision, n, knot):
    tol = 1e-11 if precision == "fp64" else 1e-10
    pos, L = _system(n, knot, 6)
    sim = ss.Simulation(n, (L,) * 3, ss.kappa_from_kappa_tau(0.5), seed=9, precision=precision, warm_start="none",
                        cg_tol=tol, cg_max_iter=5000, positions=pos)
    if precision == "mixed":
        sim.set_solver_config(0)
    sim.set_positions(pos, 0.0)
    sim.build_neighbors()
    sim.assemble()
    info = sim.solve_velocities()
    v = sim.get_velocities()
    sim.close()
    assert info["status"] == 0 and info["residual"] <= tol, info
    assert _residual(n, pos, L, v) <= tol + (1e-13 if precision == "fp64" else 2e-11)


def test_batch_of_unequal_replicas():
    shapes = [(300, 0), (20000, 500), (9000, 0)]
    made = [_system(n, knot, 7) for n, knot in shapes]
    batch = ss.Batch([{"n": n, "L": (m[1],) * 3, "kappa": ss.kappa_from_kappa_tau(0.5), "seed": 9, "cg_tol": 1e-8}
                      for (n, _), m in zip(shapes, made)], [m[0] for m in made])
    infos = batch.step(1)
    for k, ((n, _), (pos, L)) in enumerate(zip(shapes, made)):
        assert infos[k]["status"] == 0 and infos[k]["last_residual"] <= 1e-8, infos[k]
        assert _residual(n, pos, L, batch.sim(k).get_velocities()) <= 1e-8 + 2e-11
    batch.close()
