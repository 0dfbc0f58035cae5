"""Equal shares of z planes per CTA in the z-column kernels: CTAs that march through several columns
and, in a batch, several boxes (with their own dx, dt and next dt), against the tile kernel bit for
bit, states and time steps.  Where refined cells exist, a CTA crosses columns of the deepest
complete level.  The FP32 slab kernel takes short shares, and fixed segments beyond."""
import numpy as np
import pytest

from paper_2411_14631_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

# (precision, col_kernel, footprint side of the kernel that then runs)
KERNELS = {"pencil": (1, 2, 16), "slab32": (1, 1, 8), "slab64": (0, 0, 8)}


def _slots(side):
    """No fewer CTAs than are resident: 384-thread CTAs of the pencil kernel, 256 of the slab's."""
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    return sm * (2048 // (384 if side == 16 else 256))


def _run(tree, w0, precision, **kw):
    from paper_2411_14631_gb300 import hydro as H
    sim = H.Simulation(tree, H.Params(5 / 3, cfl=0.6, precision=precision, **kw), w0=w0)
    for _ in range(2):
        sim.step()
    assert sim.prm.read_status()[0] == 0
    return sim.u, sim.dt


def _state(n, seed):
    g = torch.Generator(device="cpu").manual_seed(seed)
    w = torch.rand((5, n), generator=g, dtype=torch.float64).numpy()
    w[0] += 1.0
    w[1:4] = 0.6 * (w[1:4] - 0.5)
    w[4] += 1.0
    return w


@pytest.mark.parametrize("few", [False, True])
@pytest.mark.parametrize("kernel", sorted(KERNELS))
def test_batch_shares_cross_boxes(kernel, few):
    from paper_2411_14631_gb300 import hydro as H
    precision, col, side = KERNELS[kernel]
    sizes = np.array([16] * 13 + [96, 16, 16, 80] + [16] * 9 + [112, 48, 16, 96] + [16] * 5 + [96], dtype=np.int32)
    if few:
        sizes = np.array([16] * 8 + [48, 16, 32] + [16] * 3 + [32], dtype=np.int32)
    tree = H.Octree.boxes(sizes, (1,) * 6)
    planes = int((sizes.astype(np.int64) ** 3).sum()) // side ** 2
    if few:
        # four CTAs per SM (64 registers a thread): shares of six planes
        share = planes / (4 * torch.cuda.get_device_properties(0).multi_processor_count)
        assert kernel != "slab32" or 4 < share <= 6, share
    else:
        share = planes / _slots(side)
        assert share > 16, share                   # longer than the small boxes' columns
    w0 = _state(tree.ncell, 1)
    # sound speeds, and so time steps, two decades apart between neighbouring boxes
    scale = 10.0 ** np.random.default_rng(2).uniform(-2, 2, sizes.size)
    for b in range(sizes.size):
        w0[4, tree.cell_off[b]:tree.cell_off[b + 1]] *= scale[b]
    ref = _run(tree, w0, precision, tiles_only=True)
    got = _run(tree, w0, precision, col_kernel=col)
    assert torch.equal(got[1], ref[1])
    assert torch.equal(got[0], ref[0])


@pytest.mark.parametrize("periodic", [True, False])
@pytest.mark.parametrize("kernel", sorted(KERNELS))
def test_level_shares_cross_columns_beside_refined_cells(kernel, periodic):
    from paper_2411_14631_gb300 import hydro as H
    precision, col, side = KERNELS[kernel]
    tree = H.Octree(W.random_tree(7, 1, 21, p_refine=0.03, periodic=periodic), 7, (0 if periodic else 1,) * 6)
    assert tree.t.grid_level == 7 and tree.levelmax == 8
    assert 128 ** 3 / side ** 2 / _slots(side) > 4      # several planes a CTA; 128 is no multiple of all shares
    w0 = _state(tree.ncell, 3)
    ref = _run(tree, w0, precision, tiles_only=True)
    got = _run(tree, w0, precision, col_kernel=col)
    assert torch.equal(got[1], ref[1])
    assert torch.equal(got[0], ref[0])
