"""The single-reduction form of the Poisson iteration (boxes of 700,000 cells and more, with the
preconditioner) against the oracle: tiles cut by the box, segments that do not divide it, equal
shares that meet two columns, both tile heights.

Tolerances: those of test_gpu_poisson.py (1e-10 of max|x|; Eq. 3 within 1e-11 and the oracle's own
sequential inner products, 2 n 2^-53 of themselves)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape,tile_y,seg", [((101, 83, 97), 0, 0), ((33, 150, 143), 16, 7), ((65, 129, 90), 8, 0),
                                              ((97, 31, 240), 8, 40), ((180, 141, 117), 0, 0)])
def test_single_reduction_matches_oracle(oracle, shape, tile_y, seg):
    from paper_2411_14631_gb300 import abi, poisson
    n = int(np.prod(shape))
    assert n >= 700000
    K = 12
    b = np.random.default_rng(2).standard_normal(n)
    x0 = 0.1 * np.random.default_rng(3).standard_normal(n)
    xo, eo, ito, sto = oracle.ppcg(shape, b, x0=x0, precond=1, tol=0.0, maxit=K)
    dev = [torch.tensor(a, device="cuda:0") for a in (b, x0)]
    s = poisson.PPCG(shape, precond=1, tol=0.0, max_iter=K, check_every=5, tile_y=tile_y, seg=seg)
    x, e, info = s.solve(*dev)
    assert info.status == abi.ENOCONV and info.iters == K == ito
    assert np.abs(x.cpu().numpy() - xo).max() <= 1e-10 * np.abs(xo).max()
    assert np.all(np.abs(e - eo) <= 1e-11 + 2 * n * 2.0 ** -53 * eo)
