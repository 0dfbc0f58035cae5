"""FP64 step: dt_next is the Courant step of the new state (hydro_courant's, bit for bit) for every
gamma > 1, also just above 1, where an FP32 gamma - 1 would understate the sound speed, and for a
sound speed whose square is below FP32's normal range.  Gas at rest with pressures within 1% of
each other: whichever cell is looked at first, the one that sets the step lies only a little below
it, so an estimate of the signal speed that is low by more than its allowance drops it."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("extra", [0, 2])
@pytest.mark.parametrize("gamma,p0", [(1.0 + 2.0 ** -40, 1.0), (1.0 + 1.78e-7, 1.0), (1.0000002, 1.0), (1.0 + 4e-7, 1.0),
                                      (1.000001, 1.0), (1.0001, 1.0), (1.001, 1.0), (1.0 + 1e-12, 1e-40)])
def test_dt_next_is_the_minimum(gamma, p0, extra):
    from paper_2411_14631_gb300 import hydro as H, workloads as W
    lx = W.random_tree(4, extra, 11, p_refine=0.3) if extra else W.uniform_tree(5)
    tree = H.Octree(lx, 4 if extra else 5)
    r = np.random.default_rng(5)
    w = np.zeros((5, tree.ncell))
    w[0] = 1.0
    w[4] = p0 * r.uniform(1.0, 1.01, tree.ncell)
    for tiles_only in (False, True):
        prm = H.Params(gamma, cfl=0.4, p_floor=1e-60, tiles_only=tiles_only)
        sim = H.Simulation(tree, prm, w0=w)
        for _ in range(2):
            sim.step()
            dt = torch.zeros_like(sim.dt)
            H.hydro_courant(tree, prm, sim.u, dt)
            assert torch.equal(dt, sim.dt)
        assert 0.0 < float(sim.dt) < 1e30
