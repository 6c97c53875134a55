"""D3Q15 step kernels against the generic tile kernel where the z-marching
tests do not reach: unequal densities (phi, C_i and step kernels), the
TMA-staged z-marching kernel at sizes that take the split kernels by default,
and a box large enough to take it by rule.

FP32 and 16-bit: the same per-node arithmetic and stencil order, so the same
numbers. FP64: rounding differs where the compiler fuses differently; phi
(O(1)) to 1e-12 and u, p to 1e-11 of their largest value after 8 steps."""
import os

import numpy as np
import pytest

from paper_1904_12553_gb300 import workloads as W
from test_d3q15_gpu import _accept, _gpu, gpu3  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SHAPES = [(1, 1, 1), (5, 3, 2), (33, 5, 3), (40, 17, 9), (64, 8, 4)]
RHO = [3.0, 1.0, 2.0, 5.0, 4.0]


def same(a, b, prec):
    for k in ("phi", "u", "p"):
        if prec == "fp64":
            scale = 0.1 if k == "phi" else np.abs(b[k]).max() + 1e-30
            assert np.abs(a[k] - b[k]).max() <= 1e-11 * scale, k
        else:
            np.testing.assert_array_equal(a[k], b[k], err_msg=k)


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("N", [2, 3, 5])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "bf16", "fp16"])
@pytest.mark.parametrize("wall", [0, 1])
def test_unequal_densities_match_generic(N, prec, shape, wall):
    nx, ny, nz = shape
    w = W.random_smooth3(N + nx, N, nx, ny, nz, rho=RHO[:N], sigma=0.01, wall_y=wall,
                         amp_u=0.02, gravity=(1e-5, -2e-5, 3e-5))
    same(gpu3(w, 8, prec), gpu3(w, 8, prec, generic=True), prec)


def march(w, steps):
    from paper_1904_12553_gb300 import Solver
    os.environ["LBM_NPHASE_KERNEL"] = "pipelined"
    try:
        s = Solver(w.params)
    finally:
        os.environ.pop("LBM_NPHASE_KERNEL", None)
    assert s.step_kernel == "z-marching 3-D (TMA)"
    s.init(w.c0, w.u0)
    s.step(steps)
    m = s.moments()
    s.close()
    return m


@pytest.mark.parametrize("shape", [(40, 17, 23), (8, 8, 1), (64, 24, 70), (32, 16, 12)])
@pytest.mark.parametrize("N", [2, 3, 4])
@pytest.mark.parametrize("wall", [0, 1])
def test_march_at_every_size_matches_generic(N, shape, wall):
    nx, ny, nz = shape
    rng = np.random.default_rng(N + nx)
    w = W.random_smooth3(N + nx, N, nx, ny, nz, wall_y=wall, amp_u=0.02, precision="fp32",
                         sigma=W.sample_sigma(rng, N, accept=_accept()))
    same(march(w, 12), gpu3(w, 12, generic=True), "fp32")


@pytest.mark.parametrize("wall", [0, 1])
def test_march_by_rule_matches_generic(wall):
    rng = np.random.default_rng(9)
    w = W.random_smooth3(9, 3, 128, 128, 64, wall_y=wall, amp_u=0.02, precision="fp32",
                         sigma=W.sample_sigma(rng, 3, accept=_accept()))
    same(gpu3(w, 6), gpu3(w, 6, generic=True), "fp32")
