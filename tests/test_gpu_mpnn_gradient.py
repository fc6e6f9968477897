"""The gradient of a training step, to the rounding of its FP32 elements.

The tensor cores' FP32 accumulation truncates, so the order in which the backward's
accumulators take their tiles is part of the result: one accumulator per SM and weight takes
the tiles blockIdx + k gridDim in the order of k, the partial gradients are added in the order
of the blocks, and dY is rounded before its message pass.  The values below come from the
first form of these kernels (one tile at a time, transposed copies) on 152 SMs: the norm of the
gradient and eight sums of its elements with random signs."""
import numpy as np
import pytest

import synth

ss = pytest.importorskip("paper_1808_06381_gb300")

pytestmark = pytest.mark.gpu

VALUES = {   # (n, seed): loss, norm, signed sums
    (262144, 41): (0.7846663047043836, 2.836456969919854,
                   [1.588935872494, -0.6463316908048, 0.8886068082866, -1.250080601969,
                    1.575706763035, -1.35923599964, -0.4951740504166, 3.73530290575]),
    (70001, 43): (0.3628858677758569, 2.268903602673657,
                  [0.4583555687732, 0.9433875277009, -3.159270503764, -1.762460637119,
                   3.120119084078, -1.273733173335, 4.111281818759, -0.3671164996758]),
    (20011, 45): (4.658708511024924, 10.282441627171373,
                  [-10.15885090054, -12.09145982398, 3.741924956154, -16.30559245372,
                   -3.382358599803, -17.56425851992, -8.447910266677, -9.151031306537]),
}


@pytest.mark.parametrize("n,seed", list(VALUES))
def test_gradient_keeps_its_order_of_accumulation(n, seed):
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the partial gradients are one per SM; the values are for 152")
    L = synth.box_length(n)
    pos = synth.uniform_positions(n, (L,) * 3, seed)
    sim = ss.Simulation(n, (L,) * 3, ss.kappa_from_kappa_tau(0.5), seed=seed, precision="mixed", warm_start="prev",
                        cg_tol=1e-10, positions=pos)
    sim.set_positions(pos, 0.3 * L)
    sim.build_neighbors()
    sim.assemble()
    sim.solve_velocities()
    r = np.random.Generator(np.random.PCG64(seed))
    w = np.concatenate([r.normal(0, 6 ** -0.5, 384), r.normal(0, 0.125, 4096), r.normal(0, 0.125, 256),
                        r.normal(0, 0.6, 11)]).astype(np.float32)
    sim.mpnn_enable(weights=w)
    sim.set_step(1)
    sim.assemble()
    sim.mpnn_forward()
    sim.solve_velocities()
    loss, grad = sim.mpnn_train_step(lr=0.0, want_grad=True)
    sim.close()
    ref_loss, ref_norm, ref_sums = VALUES[n, seed]
    g = grad.astype(np.float64)
    signs = np.random.Generator(np.random.PCG64(7)).integers(0, 2, (8, g.size)) * 2.0 - 1.0
    # The target velocities agree to ~1e-10 (two solves to 1e-10), which moves a few FP32
    # roundings; an element's own rounding is 6e-8 of it.
    assert abs(loss - ref_loss) <= 1e-9 * ref_loss
    assert abs(np.linalg.norm(g) - ref_norm) <= 2e-7 * ref_norm
    assert np.abs(signs @ g - ref_sums).max() <= 2e-7 * ref_norm
