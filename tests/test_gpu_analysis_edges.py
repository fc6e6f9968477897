"""Edges of the analysis and training kernels: high Chebyshev degrees, ragged tiles of the
training step, one bin that takes every pair of the velocity correlation, more listed pairs than
a segment holds, and more than 128 tiles."""
import numpy as np
import pytest

import oracle
from oracle import mpnn
import synth

ss = pytest.importorskip("paper_1808_06381_gb300")

pytestmark = pytest.mark.gpu


def _solved(n, seed, precision):
    L = max(synth.box_length(n), 3.01)
    pos = synth.uniform_positions(n, (L,) * 3, seed)
    kappa = ss.kappa_from_kappa_tau(0.5)
    sim = ss.Simulation(n, (L,) * 3, kappa, seed=seed, positions=pos, precision=precision, warm_start="prev",
                        cg_tol=1e-12 if precision == "fp64" else 1e-8, cg_max_iter=5000)
    sim.set_positions(pos, 0.3 * L)
    sim.build_neighbors()
    sim.assemble()
    return sim, oracle.Params(n=n, L=(L,) * 3, kappa=kappa, seed=seed), pos, 0.3 * L


# p(A) is within rounding of A^(1/2), whose derivative is at most 1/2 on [1, lambda_max], so the
# matrices' difference (1e-14 FP64, 1e-12 mixed) enters by at most its half; the recurrence adds
# at most the degree times the unit rounding (2^-53, 2^-46) times sum |c_k|, below 1e-10 at 2,000.
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("mixed", 1e-9)])
@pytest.mark.parametrize("n,degree", [(300, 1), (129, 64), (200, 2000)])
def test_sqrt_apply_degrees(precision, tol, n, degree):
    sim, p, pos, delta = _solved(n, n, precision)
    sysr = oracle.assemble(p, pos, oracle.neighbors(p, pos, delta), np.zeros((n, 3)), delta)
    g = np.random.default_rng(n).standard_normal((n, 3))
    for _ in range(2):   # the second call finds the arrays of the first
        xi, lmax = sim.sqrt_apply(g, degree)
        ref, lref = oracle.sqrt_apply(sysr, g, degree)
        assert lmax == pytest.approx(lref, rel=1e-12)
        assert np.abs(xi - ref).max() <= tol * np.abs(ref).max()
        degree = max(1, degree // 3)
    sim.close()


# tiles of 128 rows: one short tile, a full one, one row more, and ragged tiles on every SM.
# BF16 rounding of weights and activations (relative 2^-9 through three layers): 3e-2 on the
# loss, 8e-2 on the gradients, as for whole tiles.
@pytest.mark.parametrize("n", [60, 128, 129, 20011])
def test_training_step_with_ragged_tiles(n):
    sim, _, _, _ = _solved(n, n, "fp64")
    sim.solve_velocities()
    W = mpnn.init_weights(11)
    W.o = np.random.Generator(np.random.PCG64(12)).normal(0, 0.6, W.o.shape)
    Wf = W.flat().astype(np.float32)
    sim.mpnn_enable(weights=Wf)
    vprev = sim.get_velocities()
    sim.set_step(1)
    sim.assemble()
    diag, b, pairs, w = sim.system()
    sim.mpnn_forward()
    sim.solve_velocities()
    vstar = sim.get_velocities()
    loss, grad = sim.mpnn_train_step(lr=0.0, want_grad=True)
    sim.close()
    rloss, rg = mpnn.loss_and_grad(mpnn.Weights.unflat(Wf), n, 4.0, pairs, w, diag, b, vprev, vstar)
    assert abs(loss - rloss) <= 3e-2 * rloss, (loss, rloss)
    g = mpnn.Weights.unflat(grad)
    for name in ("W1", "W2", "W3", "o"):
        a, r = getattr(g, name), getattr(rg, name)
        rel = np.linalg.norm(a - r) / np.linalg.norm(r)
        assert rel < 8e-2, (name, rel)


# Counts exactly; a product enters its bin rounded to 2^-20 max|u|^2 after FP32 rounding, so per
# bin |sum - oracle| <= count 2^-19 max|u|^2.
def _vcorr(pos, v, L, delta, nbins, rmax):
    p = oracle.Params(n=len(pos), L=L, kappa=0.3)
    rs, rc, rv = oracle.velocity_correlation(p, pos, delta, v, nbins, rmax)
    got = ss.velocity_correlation(pos, v, L, delta, 0.3, nbins, rmax)
    assert np.array_equal(got["counts"], rc)
    u = v.copy()
    u[:, 0] -= 0.3 * (pos[:, 1] - 0.5 * L[1])
    assert np.all(np.abs(got["sums"] - rs) <= rc * 2.0 ** -19 * float((u * u).sum(1).max()) + 1e-12)


def test_every_pair_in_one_bin():
    """A cluster far smaller than the only bin: every lane adds to one word, up to its capacity."""
    rng = np.random.default_rng(3)
    pos = 1.0 + 0.5 * rng.random((1500, 3))
    _vcorr(pos, 3.0 * np.ones((1500, 3)), (9.0, 9.0, 9.0), 1.2, 1, 4.0)


@pytest.mark.parametrize("delta", [0.0, 2.0, 7.5])
def test_more_listed_pairs_than_a_segment_holds(delta):
    """A lattice whose distances lie on bin edges and half-box ties: most pairs are listed."""
    g = np.stack(np.meshgrid(np.arange(16), np.arange(14), np.arange(12), indexing="ij"), -1).reshape(-1, 3)
    v = np.random.default_rng(5).standard_normal((len(g), 3))
    _vcorr(0.5 * g.astype(np.float64), v, (8.0, 7.0, 6.0), delta, 24, 3.0)


def test_more_than_128_tiles():
    n, L = 33025, (30.0, 28.0, 26.0)
    rng = np.random.default_rng(8)
    _vcorr(rng.random((n, 3)) * np.asarray(L), rng.standard_normal((n, 3)), L, 4.4, 50, 5.0)
