"""FP64 path: the CFL candidates left out by an FP32 estimate, and the arithmetic outside the middle
of the exponent range.

- dt_next of a step equals hydro_courant of the state it made, bit for bit: the same candidates,
  all of them formed there.  States where the estimate is weakest: cold hypersonic flow, pressures
  and densities at the floors, gas at rest, scales beyond FP32's range.
- Powers of two times the density and pressure (and the floors) scale the conserved state by the
  same power: 2^+-600 takes every reciprocal, division and sound speed through the IEEE operations.
  Both forms round each operation to within 1 ulp; a step has some 30 roundings in a row, so 1e-13
  of the largest value leaves an order of magnitude."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

STATES = {
    "turbulent": lambda r, n: (np.exp(r.normal(0, 1, n)), r.normal(0, 2, (3, n)), np.exp(r.normal(0, 1, n))),
    "hypersonic": lambda r, n: (np.exp(r.normal(0, 1, n)), 300 + r.normal(0, 20, (3, n)),
                                1e-3 * np.exp(r.normal(0, 2, n))),
    "floors": lambda r, n: (10.0 ** r.uniform(-12, 1, n), r.normal(0, 1e-3, (3, n)), 10.0 ** r.uniform(-24, -2, n)),
    "rest": lambda r, n: (np.ones(n), np.zeros((3, n)), np.where(r.random(n) < 0.1, 3.0, 1.0)),
    "large": lambda r, n: (1e45 * np.exp(r.normal(0, 1, n)), r.normal(0, 2, (3, n)), 1e45 * np.exp(r.normal(0, 1, n))),
}


def _prims(name, n, seed):
    rho, v, p = STATES[name](np.random.default_rng(seed), n)
    return np.concatenate([rho[None], v, p[None]])


@pytest.mark.parametrize("extra", [0, 2])
@pytest.mark.parametrize("name", sorted(STATES))
def test_step_dt_is_courant_of_the_new_state(name, extra):
    from paper_2411_14631_gb300 import hydro as H, workloads as W
    lx = W.random_tree(4, extra, 11, p_refine=0.3) if extra else W.uniform_tree(5)
    tree = H.Octree(lx, 4 if extra else 5)
    prm = H.Params(5.0 / 3.0, cfl=0.4)
    sim = H.Simulation(tree, prm, w0=_prims(name, tree.ncell, 3))
    for _ in range(2):
        sim.step()
        dt = torch.zeros_like(sim.dt)
        H.hydro_courant(tree, prm, sim.u, dt)
        assert torch.equal(dt, sim.dt)
    assert float(sim.dt) > 0.0


@pytest.mark.parametrize("tiles_only", [False, True])
@pytest.mark.parametrize("k", [600, -600])
def test_scaled_state_takes_ieee_operations(k, tiles_only):
    from paper_2411_14631_gb300 import hydro as H, workloads as W
    tree = H.Octree(W.uniform_tree(4), 4)
    w = _prims("turbulent", tree.ncell, 7)
    out = []
    for e in (0, k):
        s = 2.0 ** e
        ws = w.copy()
        ws[0] *= s
        ws[4] *= s
        prm = H.Params(1.4, cfl=0.4, rho_floor=1e-10 * s, p_floor=1e-20 * s, tiles_only=tiles_only)
        sim = H.Simulation(tree, prm, w0=ws)
        sim.step()
        out.append((sim.u.cpu().numpy() / s, sim.dt.cpu().numpy()))
    for v in range(5):
        assert np.abs(out[0][0][v] - out[1][0][v]).max() <= 1e-13 * np.abs(out[0][0][v]).max()
    assert abs(out[0][1][0] / out[1][1][0] - 1.0) <= 1e-14
