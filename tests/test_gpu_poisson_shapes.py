"""Flat, narrow and long boxes above 700,000 cells, where the single-reduction form's tile height and
split of the planes differ from those of a cube: equal shares of few planes that meet many columns
(segments of one and two planes among them), one column of tiles, rows that 8 fits and 16 does not,
and boxes of too few planes for that form.  Against the oracle; tolerances of
test_gpu_poisson_forms.py."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("shape", [(300, 300, 9), (310, 470, 5), (1000, 140, 7), (16, 16, 3000), (9, 9, 9000), (24, 24, 1300),
                                   (1, 1, 800000), (33, 190, 190), (190, 33, 190), (17, 2900, 16), (9, 300, 300),
                                   (500, 500, 4), (1000, 800, 1), (600000, 2, 1)])
def test_matches_oracle(oracle, shape):
    from paper_2411_14631_gb300 import abi, poisson
    n = int(np.prod(shape))
    assert n >= 700000
    K = 12
    b = np.random.default_rng(2).standard_normal(n)
    x0 = 0.1 * np.random.default_rng(3).standard_normal(n)
    xo, eo, ito, sto = oracle.ppcg(shape, b, x0=x0, precond=1, tol=0.0, maxit=K)
    dev = [torch.tensor(a, device="cuda:0") for a in (b, x0)]
    s = poisson.PPCG(shape, precond=1, tol=0.0, max_iter=K, check_every=5)
    x, e, info = s.solve(*dev)
    assert info.status == abi.ENOCONV and info.iters == K == ito
    assert np.abs(x.cpu().numpy() - xo).max() <= 1e-10 * np.abs(xo).max()
    assert np.all(np.abs(e - eo) <= 1e-11 + 2 * n * 2.0 ** -53 * eo)
