"""The tile kernel's counters count every face of every tile of the levels it updates, also of tiles
in the middle of a finer level, where no cell is updated: the Newton solves of the exact solver in
both precisions, the surrogate's accepted and rejected faces, and the seeded solves.  A depth-1 tile
has 240 faces (4 x 4 x 5 per direction)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _tree(H, W):
    """Levels 1-4 complete, level 5 in one octant of the box, level 6 in one octant of that: tiles
    with every cell refined, with some and with none."""
    lx = [W.uniform_tree(4)]
    for level, m in ((5, 8), (6, 8)):
        k, j, i = np.meshgrid(*(np.arange(m),) * 3, indexing="ij")
        lx.append(np.stack([np.full(m ** 3, level), i.ravel(), j.ravel(), k.ravel()], axis=1))
    return H.Octree(np.concatenate(lx).astype(np.int32), 4, (1,) * 6)


@pytest.mark.parametrize("riemann,precision", [("EXACT", 0), ("EXACT", 1), ("MLP", 1), ("MLP_SEEDED", 1)])
def test_every_face_of_every_tile_is_counted(riemann, precision):
    from paper_2411_14631_gb300 import abi, hydro as H, workloads as W
    tree = _tree(H, W)
    assert tree.levelmax == 6 and tree.t.grid_level == 4
    refmask = tree.tables()["refmask"].cpu().numpy()
    octs = refmask[tree.lvl_off[4]:tree.lvl_off[5]]
    assert (octs == 0xFF).any() and (octs == 0).any()
    rng = np.random.default_rng(3)
    w = np.zeros((5, tree.ncell))
    w[0] = rng.uniform(1.0, 1.5, tree.ncell)
    w[1:4] = rng.uniform(-0.3, 0.3, (3, tree.ncell))
    w[4] = rng.uniform(1.0, 1.5, tree.ncell)
    prm = H.Params(1.4, cfl=0.4, riemann=getattr(abi, "RIEMANN_" + riemann), precision=precision, tiles_only=True)
    sur = H.Surrogate(seed=2)
    prm.c.mlp_weights = sur.packed.data_ptr()
    prm.c.mlp_resid_tol = 0.05
    sim = H.Simulation(tree, prm, w0=w)
    sim.step()
    status, cnt = prm.read_status()
    off = np.array(tree.t.tile_off[0][:])
    faces = 240 * int(off[tree.levelmax + 1] - off[4])
    assert status == 0
    if riemann == "EXACT":
        assert cnt[3] == faces and cnt[2] >= cnt[3]
    else:
        assert cnt[0] + cnt[1] == faces
        if riemann == "MLP_SEEDED":
            assert cnt[3] == faces
