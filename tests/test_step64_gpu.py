"""The FP64 D2Q9 step kernels (one fused kernel; phi and C_i first, then the
collision, for unequal densities or Eq. N40) against the generic tile kernel:
grids smaller than a tile and its stencils, one node wide, tile edges and
remainders, more tiles than SMs.

Compared is what a step writes: the rest and moving populations, the NS
populations, phi(t-1) and u(t-1). Both sides round each of the ~1e3 operations
of a node-step once in FP64 (1.1e-16), in a different order; over 6 steps each
array agrees to 1e-11 of its largest value, and phi to 1e-12."""
import os

import numpy as np
import pytest

from paper_1904_12553_gb300 import workloads as W
from test_parity_gpu import _accept, _gpu  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [(1, 1), (2, 1), (1, 9), (3, 2), (16, 8), (17, 9), (15, 7), (64, 48), (150, 37),
         (203, 131)]
RHO = {2: [3.0, 1.0], 3: [10.0, 1.0, 5.0], 4: [2.0, 1.0, 3.0, 7.0],
       5: [6.0, 4.0, 1.0, 2.0, 3.0]}


def state_after(w, steps, generic):
    from paper_1904_12553_gb300 import Solver
    os.environ.pop("LBM_NPHASE_KERNEL", None)
    if generic:
        os.environ["LBM_NPHASE_KERNEL"] = "generic"
    try:
        s = Solver(w.params)
    finally:
        os.environ.pop("LBM_NPHASE_KERNEL", None)
    s.init(w.c0, w.u0)
    s.step(steps)
    v = s.get_state()[64:].numpy().view(np.float64).reshape(-1, w.V)
    s.close()
    n = w.params["N"] - 1
    cut = np.cumsum([n, 8 * n, 8, n, 2])
    return dict(zip(("h0", "hm", "gm", "phi", "u"), np.split(v, cut[:-1])))


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("N", [2, 3, 4, 5])
@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("unequal", [0, 1])
@pytest.mark.parametrize("scheme", [0, 1])
def test_step64_matches_generic(N, nx, ny, wall, unequal, scheme):
    seed = 11 * N + nx + 3 * ny + wall
    rng = np.random.default_rng(seed)
    rho = RHO[N] if unequal else None
    sigma = 0.01 if unequal else W.sample_sigma(rng, N, accept=_accept())
    w = W.random_smooth(seed, N, nx, ny, rho=rho, wall_y=wall, amp_u=0.02,
                        sigma=sigma, gravity=(1e-5, -2e-5), grad_scheme=scheme)
    a, b = state_after(w, 6, False), state_after(w, 6, True)
    for k in a:
        assert np.abs(a[k] - b[k]).max() <= 1e-11 * np.abs(b[k]).max(), k
    assert np.abs(a["phi"] - b["phi"]).max() <= 1e-12
