"""The start's FP64 -> FP32 rounding (to nearest, ties to even, by integer
operations in the normal range): u(t-1) as stored equals NumPy's conversion bit
for bit, on ties, their neighbours, both ends of the normal range, subnormals,
signed zeros, overflow and infinity. No tolerance."""
import numpy as np
import pytest

from paper_1904_12553_gb300 import workloads as W
from test_parity_gpu import _gpu  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def values(count):
    rng = np.random.default_rng(4)
    f = rng.integers(1, 0x7F800000, count, dtype=np.int64).astype(np.int32).view(np.float32)
    low, high = f.astype(np.float64), np.nextafter(f, np.float32(np.inf)).astype(np.float64)
    high[~np.isfinite(high)] = 2.0 ** 128
    v = np.where(np.arange(count) % 3 == 0, 0.5 * (low + high),
                 low + rng.random(count) * (high - low))
    v[1::5] = np.nextafter(0.5 * (low + high), 0)[1::5]
    v[2::5] = np.nextafter(0.5 * (low + high), np.inf)[2::5]
    edge = [0.0, 2.0 ** -126, np.nextafter(2.0 ** -126, 0), 2.0 ** -149, 2.0 ** -150, 5e-324,
            2.0 ** 128, np.nextafter(2.0 ** 128, 0), 2.0 ** 128 - 2.0 ** 103, 1e300, np.inf,
            np.float64(np.finfo(np.float32).max), 1.0, np.nextafter(2.0, 0)]
    v[:len(edge)] = edge
    return v * np.where(rng.random(count) < 0.5, -1.0, 1.0)


@pytest.mark.parametrize("precision", ["fp32", "bf16", "fp16"])
@pytest.mark.parametrize("nz", [0, 5])
def test_stored_velocity(precision, nz):
    from paper_1904_12553_gb300 import Solver
    nx, ny, D = 64, 21, 3 if nz else 2
    kw = dict(sigma=0.01, precision=precision)
    w = W.random_smooth3(3, 3, nx, ny, nz, **kw) if nz else W.random_smooth(3, 3, nx, ny, **kw)
    u = values(D * w.V).reshape((D,) + ((nz,) if nz else ()) + (ny, nx))
    s = Solver(w.params)
    s.init(w.c0, u)
    blob = s.get_state()[64:].numpy()
    s.close()
    planes = D + (0 if precision == "fp32" else 1)
    got = blob[-4 * planes * w.V:].view(np.float32)[:D * w.V]
    with np.errstate(over="ignore", under="ignore"):
        want = u.astype(np.float32).ravel()
    np.testing.assert_array_equal(got.view(np.int32), want.view(np.int32))
