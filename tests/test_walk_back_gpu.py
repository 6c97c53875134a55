"""States of 48 MB on, whose steps walk the tiles alternately forwards and
backwards: a periodic grid made of copies of a smaller one (whose steps always
walk forwards) evolves as copies of it, after an even and an odd number of steps,
with remainders in every axis.

The generic, the split D3Q15 and the 16-bit kernels are then the same code on the
same values: equal bits. The FP32 pipelined kernel sums an edge position's phi
from another box than an inner one's: within 1e-6 of the largest value, the bound
of its other comparisons."""
import os

import numpy as np
import pytest

from paper_1904_12553_gb300 import Solver, workloads as W
from test_parity_gpu import _gpu  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RHO = [1.0, 1.5, 2.0, 1.2, 1.8]


def run(params, c, u, steps, env):
    old = os.environ.pop("LBM_NPHASE_KERNEL", None)
    if env:
        os.environ["LBM_NPHASE_KERNEL"] = env
    try:
        s = Solver(params)
    finally:
        os.environ.pop("LBM_NPHASE_KERNEL", None)
        if old is not None:
            os.environ["LBM_NPHASE_KERNEL"] = old
    s.init(c, u)
    s.step(steps)
    m, k = s.moments(), s.kernels
    s.close()
    return m, k


def state_mb(N, V, prec, three):
    Q, D = (14, 3) if three else (8, 2)
    wide = 8 if prec == "fp64" else 4
    moving = 2 if prec in ("bf16", "fp16") else wide
    return V * (N * Q * moving + (2 * (N - 1) + D) * wide) / 2.0 ** 20


# phases, precision, unequal densities, Eq. N40, small grid, copies, kernels
CASES = [
    (3, "fp32", 1, 0, (235, 47), (3, 13), "generic", "tile_kernel"),
    (3, "fp32", 0, 1, (235, 47), (3, 13), "generic", "tile_kernel"),
    (5, "bf16", 1, 0, (121, 37), (5, 20), None, "tile_kernel"),
    (4, "bf16", 0, 0, (96, 48), (8, 16), None, "tile_kernel_tma"),
    (4, "fp16", 0, 0, (88, 37), (9, 19), None, "tile_kernel_tma"),
    (3, "fp32", 0, 0, (96, 45), (8, 13), "pipelined", "tile_kernel_tma"),
    (5, "fp32", 0, 0, (107, 43), (5, 13), "pipelined", "tile_kernel_tma"),
    (3, "bf16", 0, 0, (33, 13, 11), (3, 5, 7), None, "phi3_kernel + step3_kernel"),
    (3, "fp32", 1, 0, (33, 13, 11), (3, 5, 5), None, "phi3_kernel + pot3_kernel + step3_kernel"),
    (3, "fp64", 0, 0, (33, 13, 11), (2, 4, 4), None, "phi3_kernel + step3_kernel"),
    (5, "fp32", 0, 0, (33, 13, 11), (3, 5, 5), None, "phi3_kernel + step3_kernel"),
]


@pytest.mark.parametrize("steps", [6, 7])
@pytest.mark.parametrize("N,prec,nu,g40,shape,copies,env,kernels", CASES)
def test_copies_evolve_alike(N, prec, nu, g40, shape, copies, env, kernels, steps):
    three = len(shape) == 3
    kw = dict(rho=RHO[:N] if nu else None, sigma=1e-3, amp_u=0.01, precision=prec)
    if three:
        w = W.random_smooth3(N, N, *shape, **kw)
    else:
        w = W.random_smooth(N, N, *shape, grad_scheme=g40, **kw)
    big = tuple(a * b for a, b in zip(shape, copies))
    reps = (1,) + tuple(reversed(copies))
    params = {**w.params, "nx": big[0], "ny": big[1], **({"nz": big[2]} if three else {})}
    V = int(np.prod(big))
    assert state_mb(N, V, prec, three) >= 48
    assert state_mb(N, w.V, prec, three) < 48
    a, k = run(params, np.tile(w.c0, reps), np.tile(w.u0, reps), steps, None)
    assert k == kernels
    b, _ = run(w.params, w.c0, w.u0, steps, env)
    for f in ("phi", "u", "p"):
        x = a[f]
        y = np.tile(b[f], reps if b[f].ndim == len(reps) else reps[1:])
        assert np.isfinite(y).all()
        if kernels == "tile_kernel_tma" and prec == "fp32":
            assert np.abs(x - y).max() <= 1e-6 * np.abs(y).max(), f
        else:
            np.testing.assert_array_equal(x, y, err_msg=f)
