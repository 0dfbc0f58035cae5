"""The hand-written device arithmetic of the update kernels against CUDA's own operations
(tests/device_math.cu, compiled like the FP32 kernels' file; its options change no FP64 operation).

Bounds: recip and divide are within 0.507 ulp, IEEE's results within 0.5, so the two are equal or
neighbours; sqrt_quot is within 1.0 ulp and sqrt of a rounded quotient within 0.85, so they are at
most two apart.  Out of the middle of the exponent range, and for the integer forms (MinMod, signs,
floors), the results are the same bits, up to the sign of a zero MinMod."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))
SPECIAL = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -np.nan, 5e-324, -5e-324, 2.0 ** -1022, 1e-310, -1e-310, 1.0, -1.0,
                    2.0 ** 500, 2.0 ** -500, np.nextafter(2.0 ** 500, 0), np.nextafter(2.0 ** -500, 0), -2.0 ** 500,
                    1.7e308, -1.7e308, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 3.0])


@pytest.fixture(scope="module")
def dm(tmp_path_factory):
    from paper_2411_14631_gb300 import build
    so = str(tmp_path_factory.mktemp("dm") / "device_math.so")
    cmd = [build.nvcc()] + build.ARCH + build.FLAGS + ["--use_fast_math", "-I" + build.CSRC, "-shared",
                                                       os.path.join(HERE, "device_math.cu"), "-o", so]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return C.CDLL(so)


def _dev(x):
    return torch.as_tensor(np.ascontiguousarray(x)).cuda()


def _call(fn, *args):
    torch.cuda.synchronize()
    assert fn(*args) == 0


def _p(t):
    return C.c_void_p(t.data_ptr())


def _pairs(seed, n=300000):
    """Ordinary magnitudes, the whole exponent range, the edge of the middle range, every pair of
    special values."""
    r = np.random.default_rng(seed)
    parts = []
    for lo, hi in ((-8, 8), (-1020, 1020), (-502, -498), (498, 502)):
        m = r.uniform(1.0, 2.0, (2, n)) * np.where(r.random((2, n)) < 0.5, -1.0, 1.0)
        parts.append(np.ldexp(m, r.integers(lo, hi, (2, n))))
    near = r.uniform(1.0, 2.0, n)               # quotients next to 1
    parts.append(np.stack([near, near * (1.0 + r.integers(-4, 5, n) * 2.0 ** -52)]))
    parts.append(np.stack([x.ravel() for x in np.meshgrid(SPECIAL, SPECIAL)]))
    return np.concatenate(parts, axis=1)


def _same(o, w):
    return (o.view(np.int64) == w.view(np.int64)) | (np.isnan(o) & np.isnan(w))


def _mid(x):
    e = (x.view(np.uint64) >> np.uint64(52)).astype(np.int64) & 0x7FF
    return (e >= 523) & (e < 1523)


def test_fp64_operations(dm):
    a, b = _pairs(1)
    n = a.size
    o, w = (torch.empty(6 * n, dtype=torch.float64, device="cuda") for _ in range(2))
    da, db = _dev(a), _dev(b)
    _call(dm.dm_ops, C.c_int64(n), _p(da), _p(db), _p(o), _p(w))
    o, w = o.cpu().numpy().reshape(6, n), w.cpu().numpy().reshape(6, n)
    mids = (_mid(b), _mid(b) & (_mid(a) | (a == 0)), _mid(a) & _mid(b) & (a > 0) & (b > 0))
    for k, (mid, ulps) in enumerate(zip(mids, (1, 1, 2))):
        assert mid.sum() > 100000 and (~mid).sum() > 100000
        assert _same(o[k][~mid], w[k][~mid]).all(), k
        x, y = o[k][mid], w[k][mid]
        # a quotient that leaves the normal range is rounded twice: no closer than its own grid
        ok = (np.abs(x.view(np.int64) - y.view(np.int64)) <= ulps) | ((x == 0) & (y == 0))
        assert ok.all(), (k, x[~ok][:4], y[~ok][:4])
    zero = (o[3] == 0) & (w[3] == 0)
    assert (zero | _same(o[3], w[3])).all()
    assert np.array_equal(o[4], w[4]) and np.array_equal(o[5], w[5])


def test_fp64_floor(dm):
    a, f = _pairs(2)
    f = np.abs(f)
    keep = np.isfinite(f) & (f > 0)
    a, f = a[keep], f[keep]
    a[::7] = f[::7]
    n = a.size
    o, w = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    da, df = _dev(a), _dev(f)
    _call(dm.dm_floor, C.c_int64(n), _p(da), _p(df), _p(o), _p(w))
    assert np.array_equal(o.cpu().numpy().view(np.int64), w.cpu().numpy().view(np.int64))


def test_fp32_reading_of_state_values(dm):
    """The update kernels' conversion and hydro_state_to_fp32's agree on every value but those
    within half a unit in the last place below 2^-126, which round up to it in the kernels."""
    x = _pairs(3).ravel()
    r = np.random.default_rng(4)
    tiny = np.ldexp(r.uniform(1.0, 2.0, 300000), r.integers(-160, -120, 300000)) * np.where(r.random(300000) < 0.5, -1, 1)
    edge = 2.0 ** -126 * (1.0 - r.integers(0, 2000, 20000) * 2.0 ** -34)
    x = np.concatenate([x, tiny, edge, -edge])
    n = x.size
    o, w = (torch.empty(n, dtype=torch.float32, device="cuda") for _ in range(2))
    dx = _dev(x)
    _call(dm.dm_read, C.c_int64(n), _p(dx), _p(o), _p(w))
    o, w = o.cpu().numpy(), w.cpu().numpy()
    up = (np.abs(x) < 2.0 ** -126) & (np.abs(x) >= 2.0 ** -126 * (1.0 - 2.0 ** -25))
    assert up.sum() > 1000
    assert np.all(w[up] == 0)
    nan = np.isnan(o) & np.isnan(w)
    assert (nan | (o.view(np.int32) == w.view(np.int32)))[~up].all()
    assert np.all(np.abs(o[up]) == 2.0 ** -126)


def test_fp32_increment(dm):
    """x + f in one multiply-add: the FP64 sum for every normal, zero, infinite or NaN f."""
    r = np.random.default_rng(5)
    n = 1000000
    f = (r.integers(0, 2 ** 32, n, dtype=np.uint64).astype(np.uint32)).view(np.float32).copy()
    f[:12] = [0.0, -0.0, np.inf, -np.inf, np.nan, 2.0 ** -126, -2.0 ** -126, 3.4028235e38, -3.4028235e38, 1.0, -1.0, 2.0 ** -125]
    den = (f != 0) & (np.abs(f) < 2.0 ** -126)
    f[den] = 0.0
    with np.errstate(over="ignore", invalid="ignore"):
        x = np.concatenate([f[: n // 2].astype(np.float64) * r.uniform(-2.0, 2.0, n // 2), r.standard_normal(n // 2)])
    x[np.isnan(x)] = 1.0
    o, w = (torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2))
    dx, df = _dev(x), _dev(f)
    _call(dm.dm_add, C.c_int64(n), _p(dx), _p(df), _p(o), _p(w))
    assert _same(o.cpu().numpy(), w.cpu().numpy()).all()


@pytest.mark.parametrize("cfl,dx", [(0.8, 2.0 ** -8), (0.4, 1.0 / 48.0)])
def test_cfl_step_falls_with_the_signal_speed(dm, cfl, dx):
    """Over every pair of neighbouring positive normal signal speeds: the smallest step of cells of
    one size is that of the largest signal speed."""
    rises = torch.zeros(1, dtype=torch.int64, device="cuda")
    _call(dm.dm_monotone, C.c_float(cfl), C.c_float(dx), _p(rises))
    assert int(rises.item()) == 0
