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


def _sim(n, seed=5):
    L = synth.box_length(n)
    pos = synth.uniform_positions(n, (L,) * 3, seed)
    sim = ss.Simulation(n, (L,) * 3, ss.kappa_from_kappa_tau(0.5), seed=seed, precision="mixed", warm_start="none",
                        cg_tol=1e-8, positions=pos)
    sim.set_positions(pos, 0.3 * L)
    return sim


@pytest.mark.parametrize("n", [777, 20011, 100000])
@pytest.mark.parametrize("config,threads", [(8, 1024), (9, 512)])
def test_a_chosen_on_chip_configuration_runs_at_every_size(n, config, threads):
    """Configurations 8 and 9 are k32_cg_resident for small systems too: its blocks are one per 256-row
    window and 256 threads (at most one per SM), the pipelined form's one per 32 n / SMs rows."""
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    sim = _sim(n)
    info = sim.set_solver_config(config)
    assert info["resident"] and info["block_threads"] == threads
    windows, groups = (n + 255) // 256, threads // 256
    blocks = min(sms, (windows + groups - 1) // groups)
    chunks = -(-n // 32)
    assert blocks != -(-chunks // -(-chunks // sms))   # what the pipelined form would take
    assert sim.profile_step()["persistent_blocks"] == blocks
    sim.close()


def test_autotune_reports_the_form_that_runs(tmp_path, monkeypatch):
    """Where the pipelined form is the fastest the simulation stays without a configuration: one block
    per 160 rows at n = 20,011, where the configurations run one per 256 rows or more.  A cached choice
    takes the same form, and one that was made without the second line keeps its configuration."""
    n = 20011
    cache = tmp_path / "tune.txt"
    monkeypatch.setenv("SHEARSIM_TUNE_CACHE", str(cache))
    for cached in (False, True):
        sim = _sim(n)
        info = sim.autotune(trials=2)
        assert info["from_cache"] == cached
        assert info["automatic"] == (sim.profile_step()["persistent_blocks"] > n // 256 + 1)
        sim.close()
    cache.write_text("".join(line for line in cache.read_text().splitlines(True) if "|automatic" not in line))
    sim = _sim(n)
    again = sim.autotune(trials=1)
    assert again["from_cache"] and not again["automatic"] and again["config"] == info["config"]
    assert sim.profile_step()["persistent_blocks"] <= n // 256 + 1
    sim.close()


@pytest.mark.parametrize("budget", ["0", "12288", "-1"])
@pytest.mark.parametrize("config", [8, 9])
def test_the_smallest_shared_memory_budget_holds_the_rows_records(config, budget, monkeypatch):
    """A budget below the rows' records (16 bytes each of up to 2048 rows) is raised to them: entries
    are gathered from memory, and the solve meets its tolerance."""
    monkeypatch.setenv("SHEARSIM_RESIDENT_SMEM", budget)
    sim = _sim(150000)
    sim.set_solver_config(config)
    sim.build_neighbors()
    sim.assemble()
    info = sim.solve_velocities()
    assert info["status"] == 0 and info["residual"] <= 1e-8 and info["offchip_blocks"] > 0, info
    sim.close()
