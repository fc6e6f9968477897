"""Which form of the mixed solve a simulation without a chosen configuration takes."""
import pytest

import synth

ss = pytest.importorskip("paper_1808_06381_gb300")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [116737, 150000, 300000])
def test_beyond_the_pipelined_form_the_default_streams(n, monkeypatch):
    """k32_cg_resident, whose inner products use 18-bit weights, runs only where it was chosen: with
    a 40 KB budget it reports blocks whose entries did not fit, and the streaming form none."""
    monkeypatch.setenv("SHEARSIM_RESIDENT_SMEM", str(40 * 1024))
    L = synth.box_length(n)
    pos = synth.uniform_positions(n, (L,) * 3, 5)
    sim = ss.Simulation(n, (L,) * 3, ss.kappa_from_kappa_tau(0.5), seed=5, precision="mixed", warm_start="none",
                        cg_tol=1e-8, positions=pos)
    sim.set_positions(pos, 0.3 * L)
    sim.build_neighbors()
    sim.assemble()
    info = sim.solve_velocities()
    assert info["status"] == 0 and info["residual"] <= 1e-8 and info["offchip_blocks"] == 0, info
    sim.set_solver_config(9)
    info = sim.solve_velocities()
    assert info["status"] == 0 and info["offchip_blocks"] > 0, info
    sim.close()
