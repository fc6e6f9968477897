"""The on-chip pipelined solves (k64_cg_pipelined, k32_cg_pipelined) at the edges of their
ranges: one row or component per thread against two and four, strided chunks against runs,
the largest system, one chunk beyond it (the next form), ragged chunks, and chunks whose rows
are too long for shared memory."""
import numpy as np
import pytest

import oracle
import synth

ss = pytest.importorskip("paper_1808_06381_gb300")

pytestmark = pytest.mark.gpu

TOL = 1e-11
# The oracle forms b - A v in FP64 with its own sums: rounding of order n_partners * 2^-53 of
# the row's terms, below 1e-13 of ||b|| for these systems.  The mixed path solves the
# double-float system, whose entries agree with the FP64 ones to ~1e-12 relative.
SLACK = {"fp64": 1e-13, "mixed": 2e-11}


def _check(n, pos, L, warm, precision):
    tol = TOL if precision == "fp64" else 10 * TOL
    kappa = ss.kappa_from_kappa_tau(0.5)
    delta = 0.3 * L
    sim = ss.Simulation(n, (L,) * 3, kappa, seed=9, precision=precision, warm_start=warm, cg_tol=tol, cg_max_iter=5000,
                        positions=pos)
    p = oracle.Params(n=n, L=(L,) * 3, kappa=oracle.kappa_from_kappa_tau(0.5), seed=9)
    sim.set_positions(pos, delta)
    for step in range(2 if warm == "prev" else 1):   # the second solve starts from the first's velocities
        sim.set_step(step)
        sim.build_neighbors()
        sim.assemble()
        info = sim.solve_velocities()
        assert info["status"] == 0 and info["residual"] <= tol, info
        v = sim.get_velocities()
        sysr = oracle.assemble(p, pos, oracle.neighbors(p, pos, delta), oracle.noise(9, step, np.arange(n)),
                               delta)
        res = np.linalg.norm(sysr.b - sysr.matvec(v)) / np.linalg.norm(sysr.b)
        assert res <= tol + SLACK[precision], (step, res)
    sim.close()


# FP64, chunks of 32 rows per SM on 152 SMs: 1 up to 4,864 rows, 5 up to 24,320 (one component a
# thread), 10 up to 48,640 (two), 16 up to 77,824 (four); beyond, vectors in memory.  Mixed: 7 up
# to 34,048 (strided chunks), 15 up to 72,960 (one row a thread), 24 up to 116,736 (two); beyond,
# k32_cg_resident.
@pytest.mark.parametrize("precision,n,warm",
                         [("fp64", 33, "none"), ("fp64", 257, "prev"), ("fp64", 4865, "none"), ("fp64", 24320, "none"),
                          ("fp64", 24321, "prev"), ("fp64", 48641, "none"), ("fp64", 77824, "none"),
                          ("fp64", 77825, "none"),
                          ("mixed", 33, "none"), ("mixed", 257, "prev"), ("mixed", 4865, "none"),
                          ("mixed", 34048, "prev"), ("mixed", 34049, "none"), ("mixed", 72960, "none"),
                          ("mixed", 72961, "prev"), ("mixed", 116736, "none"), ("mixed", 116737, "prev")])
def test_on_chip_solve_meets_the_tolerance_on_the_oracles_system(precision, n, warm):
    L = max(synth.box_length(n), 2.01)
    _check(n, synth.uniform_positions(n, (L,) * 3, 3), L, warm, precision)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,knot", [(900, 300), (20011, 400)])
def test_rows_too_long_for_shared_memory(n, knot, precision):
    """A knot of particles within r_c of each other: rows of more entries than a chunk's share."""
    L = synth.box_length(n)
    pos = synth.uniform_positions(n, (L,) * 3, 4)
    pos[:knot] = 0.5 * L + 0.4 * (pos[:knot] / L - 0.5)
    _check(n, pos, L, "none", precision)
