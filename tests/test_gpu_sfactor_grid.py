"""The grid form of S(q) (cloud-in-cell deposit and separable transform) against the same
estimate by numpy in FP64, for even and odd grids, the smallest and the largest, mode counts
from 0 to the limit, and rectangular mode sets."""
import numpy as np
import pytest

import synth

ss = pytest.importorskip("paper_1808_06381_gb300")

pytestmark = pytest.mark.gpu


def _reference(pos, L, delta, G, nkx, nky):
    n = pos.shape[0]
    xs = pos[:, 0] - delta / L * pos[:, 1]
    xs = (xs - L * np.floor(xs / L)) / L * G
    ys = pos[:, 1] / L * G
    i0, j0 = np.floor(xs).astype(int), np.floor(ys).astype(int)
    fx, fy = xs - i0, ys - j0
    rho = np.zeros((G, G))
    for di, wx in ((0, 1 - fx), (1, fx)):
        for dj, wy in ((0, 1 - fy), (1, fy)):
            np.add.at(rho, ((j0 + dj) % G, (i0 + di) % G), wx * wy)
    gx = np.arange(G)
    kx, ky = np.arange(-nkx, nkx + 1), np.arange(-nky, nky + 1)
    A = rho @ np.exp(-2j * np.pi * np.outer(gx, kx) / G)            # [gy][kx]
    F = np.exp(-2j * np.pi * np.outer(ky, gx) / G) @ A               # [ky][kx]
    win = np.outer(np.sinc(kx / G) ** 2, np.sinc(ky / G) ** 2)
    return np.abs(F.T) ** 2 / win ** 2 / n


# The deposit rounds each of 4 n weights to 2^-32 (error <= 2^-33 and the 2^-39 of the fixed
# point): |dF| <= 4 n 2^-32.9, so |dS| <= 2 sqrt(S / n) |dF| / w^2 + ..., w >= 0.65 in the
# allowed modes: below 1e-8 n^(1/2) sqrt(S) (1.3e-6 sqrt(S) at n = 17,000) plus the second order.
@pytest.mark.parametrize("G,nkx,nky,n,delta", [(8, 1, 1, 300, 0.0), (9, 2, 0, 500, 0.37), (64, 15, 15, 2000, 0.999),
                                               (255, 0, 20, 3000, 0.5), (256, 48, 48, 17000, 0.25),
                                               (1500, 33, 7, 4000, 0.61), (8192, 3, 2, 900, 0.1)])
def test_grid_structure_factor_matches_numpy(G, nkx, nky, n, delta):
    L = max(synth.box_length(n), 2.5)
    pos = synth.uniform_positions(n, (L,) * 3, G)
    pos[0], pos[1] = (0.0, 0.0, 0.0), (0.0, np.nextafter(L, 0.0), 0.0)   # corners of the fold
    sim = ss.Simulation(n, (L,) * 3, 1.0, seed=1, positions=pos)
    sim.set_positions(pos, delta * L)
    S, qx, qy = sim.structure_factor(nkx, nky, grid=G)
    sim.close()
    ref = _reference(pos, L, delta * L, G, nkx, nky)
    assert S.shape == ref.shape
    assert np.all(np.abs(S - ref) <= 1e-8 * np.sqrt(n) * (np.sqrt(ref) + 1e-4)), np.abs(S - ref).max()
    kx = np.arange(-nkx, nkx + 1)[:, None]
    ky = np.arange(-nky, nky + 1)[None, :]
    assert np.allclose(qx, 2 * np.pi * kx / L + 0 * ky, rtol=1e-14, atol=1e-14)
    assert np.allclose(qy, 2 * np.pi * ky / L - delta * 2 * np.pi * kx / L, rtol=1e-13, atol=1e-13)


def test_refused_positions_leave_the_call_usable():
    """Refused positions stay stored ("undefined until valid ones are set"): the deposit puts every
    value on the grid, and after valid positions the call gives what a new simulation gives."""
    n, G, k = 3000, 64, 8
    L = synth.box_length(n)
    pos = synth.uniform_positions(n, (L,) * 3, 2)
    ref = ss.Simulation(n, (L,) * 3, 1.0, seed=1, positions=pos)
    ref.set_positions(pos, 0.3 * L)
    want = ref.structure_factor(k, k, grid=G)[0]
    ref.close()
    bad = pos.copy()
    bad[:8, 1] = (-0.5 * L, -1e9, 3.7 * L, 1e12, 1e300, np.inf, -np.inf, np.nan)
    bad[8:14, 0] = (-2.5 * L, 9.0 * L, -1e300, np.inf, np.nan, L)
    sim = ss.Simulation(n, (L,) * 3, 1.0, seed=1, positions=pos)
    with pytest.raises(ss.ShearsimError):
        sim.set_positions(bad, 0.3 * L)
    assert np.all(np.isfinite(sim.structure_factor(k, k, grid=G)[0]))
    sim.set_positions(pos, 0.3 * L)
    assert np.array_equal(sim.structure_factor(k, k, grid=G)[0], want)
    sim.close()
