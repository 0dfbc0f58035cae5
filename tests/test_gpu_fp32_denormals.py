"""hydro_courant of the FP32 path (compiled without flushing denormals) reads state values and
parameters below FP32's normal range as zero: with every cell's pressure and the floor on it below
2^-126 no cell has a signal speed, and the step is that of zeros, bit for bit, with the octree, the
levels' and the batch form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("kind", ["box", "levels", "batch"])
def test_denormal_values_are_zeros(kind):
    from paper_2411_14631_gb300 import hydro as H, workloads as W
    tree = H.Octree.boxes(np.array([16, 24], dtype=np.int32)) if kind == "batch" else H.Octree(W.uniform_tree(4), 4)
    prm = H.Params(1.4, cfl=0.5, rho_floor=1e-30, p_floor=1e-39, precision=1)
    r = np.random.default_rng(7)
    out = []
    for tiny in (1e-38, 0.0):
        u = np.zeros((5, tree.ncell))
        u[0] = 1.0
        u[1:] = tiny * r.uniform(0.01, 1.0, (4, tree.ncell))
        dt = torch.zeros(max(1, tree.n_inst), dtype=torch.float64, device="cuda")
        (H.hydro_courant_levels if kind == "levels" else H.hydro_courant)(tree, prm, torch.as_tensor(u).cuda(), dt)
        out.append(dt)
    assert torch.equal(out[0], out[1]), out
    assert float(out[0].min()) > 1e300
