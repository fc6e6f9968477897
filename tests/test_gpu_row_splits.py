"""The build and the stress where several threads share a row, on both sides of the sizes at
which one thread per row takes over, against the oracle: pairs exactly, the system and the
stress to the rounding of sums in another order; rows of more partners than the search keeps."""
import numpy as np
import pytest

import oracle
import synth

ss = pytest.importorskip("paper_1808_06381_gb300")

pytestmark = pytest.mark.gpu


def _compare(n, pos, L, precision, delta):
    kappa = ss.kappa_from_kappa_tau(0.5)
    sim = ss.Simulation(n, (L,) * 3, kappa, seed=7, precision=precision, warm_start="none",
                        cg_tol=1e-12 if precision == "fp64" else 1e-8, cg_max_iter=5000, positions=pos)
    p = oracle.Params(n=n, L=(L,) * 3, kappa=kappa, seed=7)
    sim.set_positions(pos, delta)
    sim.build_neighbors()
    sim.assemble()
    assert sim.solve_velocities()["status"] == 0
    diag, b, pairs, w = sim.system()
    v, stress = sim.get_velocities(), sim.stress_xy()
    sim.close()
    ref_pairs = oracle.neighbors(p, pos, delta, "cells" if n > 5000 else "auto")
    ref_pairs = ref_pairs[np.lexsort((ref_pairs[:, 1], ref_pairs[:, 0]))]
    assert np.array_equal(pairs, ref_pairs)
    sysr = oracle.assemble(p, pos, ref_pairs, oracle.noise(7, 0, np.arange(n)), delta)
    # FP64: sums of up to a few hundred terms in another order, 1e-14 each relative to the row's
    # terms; mixed: separations and weights of the 2^-48 representation, ~1e-12
    tol = 1e-12 if precision == "fp64" else 1e-10
    assert np.abs(diag - sysr.diag).max() <= tol * np.abs(sysr.diag).max()
    assert np.abs(b - sysr.b).max() <= tol * np.abs(sysr.b).max()
    # the pair terms of the virial cancel: rounding relative to the sum of their magnitudes is not
    # known here, so the bound is that of the solved state's parity (1e-10, 1e-4) widened by the
    # square root of the pairs beyond 4,096 particles' share (random signs)
    ref = oracle.stress_xy(p, pos, delta, ref_pairs, v)
    bound = (1e-10 if precision == "fp64" else 1e-4) * max(1.0, np.sqrt(n / 4096))
    assert abs(stress - ref) <= bound * abs(ref), (stress, ref)


# nine threads a row of the search below 48,000 rows, four warps a chunk of the assembly below
# 524,288, four lanes a row of the FP64 stress always, eight of the FP32 one below 130,000
@pytest.mark.parametrize("precision,n", [("fp64", 33), ("mixed", 33), ("fp64", 1025), ("fp64", 47999), ("mixed", 47999),
                                         ("fp64", 48000), ("mixed", 48000), ("mixed", 129999), ("mixed", 130000),
                                         ("mixed", 524287), ("mixed", 524288), ("fp64", 524288)])
def test_build_and_stress_across_the_splits(precision, n):
    L = max(synth.box_length(n), 3.01)
    _compare(n, synth.uniform_positions(n, (L,) * 3, 11), L, precision, 0.3 * L)


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("n,knot", [(800, 97), (800, 98), (3000, 400), (50000, 150)])
def test_rows_of_more_partners_than_the_search_keeps(precision, n, knot):
    """A knot of particles within r_c of each other: rows of 96 partners and of more."""
    L = synth.box_length(n)
    pos = synth.uniform_positions(n, (L,) * 3, 5)
    pos[:knot] = 0.5 * L + 0.4 * (pos[:knot] / L - 0.5)
    _compare(n, pos, L, precision, 0.4 * L)
