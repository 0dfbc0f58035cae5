"""The end of a training step in one launch (gradient sum, Adam, packed weights): the packed block is
that of mlp_pack byte for byte (matrices, their transposes, padding, biases), the parameters and
moments are the oracle's Adam step on the step's own gradient, and that gradient is the oracle's,
for 12 CTAs with one chunk each (the sum's eight-wide loop and its tail) and for more chunks than
CTAs, both with a ragged last chunk.  Tolerances: those of test_gpu_mlp.py; the moments are those of
the middle of a run, so that a parameter's change does not hang on the sign of a vanishing gradient."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [64, 128, 1500, 20011])
def test_training_step(oracle, n):
    from paper_2411_14631_gb300 import hydro as H
    from paper_2411_14631_gb300.abi import lib
    sur = H.Surrogate(seed=6)
    rng = np.random.default_rng(n)
    x7 = np.concatenate([rng.normal(0, 1, (n, 6)), np.full((n, 1), 1.4)], axis=1)
    x8 = np.zeros((n, 8), dtype=np.float32)
    x8[:, :7] = x7
    x = torch.as_tensor(x8).cuda()
    y = torch.as_tensor(rng.normal(0, 1, (n, 2)).astype(np.float32)).cuda()
    th0 = sur.theta.cpu().numpy().astype(np.float64)
    dy = 2.0 * (sur.forward(x) - y) / n
    grad = torch.empty_like(sur.theta)
    scratch = torch.full((int(lib().mlp_scratch_bytes(n)) // 4 + 1,), float("nan"), dtype=torch.float32, device="cuda")
    H.mlp_grad(sur.packed, x, dy, grad, scratch)
    g = grad.cpu().numpy().astype(np.float64)
    g_o = oracle.mlp_backward(th0, x7, dy.cpu().numpy().astype(np.float64))
    assert np.linalg.norm(g - g_o) <= 3e-2 * np.linalg.norm(g_o)
    m, v = 1e-3 * rng.standard_normal(th0.size), 1e-5 * rng.uniform(0.5, 1.5, th0.size)
    sur.m.copy_(torch.as_tensor(m))
    sur.v.copy_(torch.as_tensor(v))
    loss = torch.zeros(1, device="cuda")
    scratch.fill_(float("nan"))
    H.mlp_train_step(sur.theta, sur.m, sur.v, sur.packed, x, y, 1e-3, 1000, loss, scratch)
    th = th0.copy()
    oracle.adam_step(th, m, v, g, 1e-3, 0.9, 0.999, 1e-8, 1000)
    assert np.abs(sur.m.cpu().numpy() - m).max() <= 1e-6 and np.abs(sur.v.cpu().numpy() - v).max() <= 1e-6
    assert np.abs(sur.theta.cpu().numpy() - th).max() <= 1e-6
    packed = sur.packed.clone()
    H.mlp_pack(sur.theta, packed)
    assert torch.equal(packed, sur.packed)
