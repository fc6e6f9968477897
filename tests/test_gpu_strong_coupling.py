"""Solves at strong coupling (alpha up to 4,000; the condition number grows with it): every form of
the solve reaches its tolerance on the oracle's system, the pipelined ones through their change to
the standard recurrence."""
import numpy as np
import pytest

import oracle
import synth

ss = pytest.importorskip("paper_1808_06381_gb300")

pytestmark = pytest.mark.gpu


def _clustered(n, L, seed):
    """Positions of a density field with a correlation length of ~r_c, as a sheared run has them."""
    rng = np.random.Generator(np.random.PCG64(seed))
    k = 2 * np.pi / L * np.round(rng.normal(size=(64, 3)) / 0.95 * L / (2 * np.pi))
    ph = 2 * np.pi * rng.random(64)
    pos = np.empty((0, 3))
    while len(pos) < n:
        x = rng.random((4 * n, 3)) * L
        keep = rng.random(len(x)) < np.exp(0.72 * (np.sqrt(2 / 64) * np.cos(x @ k.T + ph).sum(1) - 2.5))
        pos = np.concatenate([pos, x[keep]])
    return pos[:n]


_systems = {}


def _system(n, alpha):
    if (n, alpha) not in _systems:
        L = synth.box_length(n)
        pos = _clustered(n, L, 3)
        p = oracle.Params(n=n, L=(L,) * 3, kappa=oracle.kappa_from_kappa_tau(0.5), seed=3, alpha=alpha)
        _systems.clear()
        _systems[n, alpha] = L, pos, oracle.assemble(p, pos, oracle.neighbors(p, pos, 0.3 * L, "cells"),
                                                     oracle.noise(3, 0, np.arange(n)), 0.3 * L)
    return _systems[n, alpha]


def _sim(n, alpha, precision, **kw):
    L, pos, _ = _system(n, alpha)
    sim = ss.Simulation(n, (L,) * 3, ss.kappa_from_kappa_tau(0.5), alpha=alpha, seed=3, precision=precision,
                        warm_start="none", cg_tol=1e-8, cg_max_iter=1000, positions=pos, **kw)
    sim.set_positions(pos, 0.3 * L)
    sim.build_neighbors()
    sim.assemble()
    return sim


# FP64: on chip (900; 20,011) and in memory (100,000).  Mixed: one row a thread (900; 20,011), two
# (100,000), and beyond the pipelined form (150,000).
@pytest.mark.parametrize("n", [900, 20011, 100000, 150000])
@pytest.mark.parametrize("alpha", [40.0, 150.0, 1000.0, 4000.0])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_solve_converges_at_strong_coupling(precision, alpha, n):
    if n == 150000 and precision == "fp64":
        pytest.skip("the form of 100,000 rows")
    sys = _system(n, alpha)[2]
    sim = _sim(n, alpha, precision)
    info = sim.solve_velocities()
    v = sim.get_velocities()
    sim.close()
    assert info["status"] == 0 and info["residual"] <= 1e-8, info
    # the oracle's matrix and the assembled one differ by ~1e-12 (mixed: double-float entries) and
    # 1e-15 (FP64) of an entry; a row's entries add up to less than twice its diagonal one
    slack = (1e-12 if precision == "mixed" else 1e-15) * 2 * np.linalg.norm(sys.diag[:, None] * v) / np.linalg.norm(sys.b)
    res = np.linalg.norm(sys.b - sys.matvec(v)) / np.linalg.norm(sys.b)
    assert res <= 1e-8 + slack, (res, slack)


def test_autotune_leaves_out_configurations_that_do_not_converge():
    """At alpha = 1,000 the pipelined form and the streaming one need different numbers of iterations: with
    a limit between the two, tuning keeps the one that converges; with one below both it returns
    their error and leaves the simulation as it was."""
    n, alpha = 20011, 1000.0
    L, pos, _ = _system(n, alpha)

    def sim_of(limit):
        sim = ss.Simulation(n, (L,) * 3, ss.kappa_from_kappa_tau(0.5), alpha=alpha, seed=3, precision="mixed",
                            warm_start="none", cg_tol=1e-8, cg_max_iter=limit, positions=pos)
        sim.set_positions(pos, 0.3 * L)
        sim.build_neighbors()
        sim.assemble()
        return sim

    sim = sim_of(1000)
    own = sim.solve_velocities()["iterations"]
    sim.set_solver_config(0)
    streaming = sim.solve_velocities()["iterations"]
    sim.close()
    assert abs(own - streaming) > 10   # else the limit below separates nothing
    sim = sim_of((own + streaming) // 2)
    info = sim.autotune(trials=1)
    assert (info["ms"][0] > 0) == (streaming < own) and (own > streaming or info["automatic"]), info
    assert sim.solve_velocities()["status"] == 0
    sim.close()
    sim = sim_of(20)
    with pytest.raises(ss.ShearsimError) as e:
        sim.autotune(trials=1)
    assert e.value.code == ss.SP_ERR_NOT_CONVERGED
    sim.set_positions(pos, 0.3 * L)   # the simulation stays usable
    assert sim.num_pairs() > 0
    sim.close()
