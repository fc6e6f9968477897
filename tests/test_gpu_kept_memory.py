"""Work arrays that a simulation keeps between calls are given back."""
import numpy as np
import pytest

import synth

ss = pytest.importorskip("paper_1808_06381_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,per_row", [("mixed", 160), ("fp64", 120)])
def test_the_vectors_of_sqrt_apply_are_given_back(precision, per_row):
    import torch
    n = 400000
    L = synth.box_length(n)
    pos = synth.uniform_positions(n, (L,) * 3, 3)
    sim = ss.Simulation(n, (L,) * 3, 1.0, seed=1, precision=precision, positions=pos)
    sim.build_neighbors()
    sim.assemble()
    g = np.random.Generator(np.random.PCG64(1)).standard_normal((n, 3))
    free = [torch.cuda.mem_get_info()[0]]
    xi = sim.sqrt_apply(g, 8)[0]
    free.append(torch.cuda.mem_get_info()[0])
    sim.set_fdt_noise(0)
    free.append(torch.cuda.mem_get_info()[0])
    assert free[0] - free[1] >= per_row * n                      # kept
    assert free[0] - free[2] <= 4 << 20                          # given back (allocations are rounded to 2 MB)
    assert np.array_equal(sim.sqrt_apply(g, 8)[0], xi)           # and allocated again
    sim.set_fdt_noise(8)
    sim.step(1)
    sim.set_fdt_noise(0)
    sim.step(1)
    sim.close()


@pytest.mark.parametrize("grid,nk,kept", [(2048, 3, True), (4096, 3, False), (0, 900, False)])
def test_large_arrays_of_the_structure_factor_are_not_kept(grid, nk, kept):
    import torch
    n = 2000
    L = synth.box_length(n)
    sim = ss.Simulation(n, (L,) * 3, 1.0, seed=1, precision="mixed", positions=synth.uniform_positions(n, (L,) * 3, 3))
    sim.step(1)
    sim.structure_factor(1, 1, grid=8)      # the call's kernels are loaded
    sim.structure_factor(1, 1, grid=0)
    before = torch.cuda.mem_get_info()[0]
    first = sim.structure_factor(nk, nk, grid=grid)[0]
    held = before - torch.cuda.mem_get_info()[0]
    assert (held > 30 << 20) == kept and held < 70 << 20, held
    assert np.array_equal(sim.structure_factor(nk, nk, grid=grid)[0], first)
    sim.close()
