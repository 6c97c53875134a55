"""The FP32 step with halo-ring warps (grids of one wave: up to 152 or 304 tiles
of 32 x 8 nodes, by the phases) against the generic kernel without them: grids
smaller than a tile and its ring, tile edges and remainders, either side of
both lines.

The arithmetic is the same but for the compiler's contraction of products and
sums, so the two are equally rounded runs of one method: a field differs by no
more than the sum of their errors, taken as twice the generic run's difference
from the FP64 run, or by 1e-6 of its largest value (8 steps that each round a
stored value by 6e-8). Equal arrays need no bound: one of the inputs (N = 4,
608 x 128, unequal densities) diverges within the 8 steps in FP64 as well."""
import numpy as np
import pytest

from paper_1904_12553_gb300 import workloads as W
from test_parity_gpu import _accept, _gpu, gpu_run  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [(1, 1), (2, 3), (31, 9), (32, 8), (33, 17), (150, 37), (256, 152), (257, 152),
         (608, 128), (609, 128)]
RHO = {2: [3.0, 1.0], 3: [10.0, 1.0, 5.0], 4: [2.0, 1.0, 3.0, 7.0],
       5: [6.0, 4.0, 1.0, 2.0, 3.0]}


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("N", [2, 3, 4, 5])
@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("unequal", [0, 1])
def test_ring_warps_match_generic(N, nx, ny, wall, unequal):
    seed = 13 * N + nx + 3 * ny + wall
    rng = np.random.default_rng(seed)
    rho = RHO[N] if unequal else None
    sigma = 0.01 if unequal else W.sample_sigma(rng, N, accept=_accept())

    def case(precision):
        return W.random_smooth(seed, N, nx, ny, rho=rho, wall_y=wall, amp_u=0.02,
                               sigma=sigma, gravity=(1e-5, -2e-5), precision=precision)

    a = gpu_run(case("fp32"), 8)
    b = gpu_run(case("fp32"), 8, kernel="generic")
    e = gpu_run(case("fp64"), 8, kernel="generic")
    for k in ("phi", "u", "p"):
        x, y, z = (np.asarray(m[k]) for m in (a, b, e))
        if np.array_equal(x, y, equal_nan=True):
            continue
        bound = max(1e-6 * np.abs(y).max(), 2 * np.abs(y - z).max())
        assert np.abs(x - y).max() <= bound, k


@pytest.mark.parametrize("nx,ny", [(1, 1), (33, 9), (150, 37), (256, 152), (257, 152), (608, 128)])
@pytest.mark.parametrize("N", [2, 3, 4, 5])
@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("unequal", [0, 1])
def test_ring_warps_mixed_gradients(N, nx, ny, wall, unequal):
    """Eq. N40: rings of radius 2 and 3, by the same comparison."""
    seed = 17 * N + nx + 3 * ny + wall
    rho = [1.0 + 0.5 * k for k in range(N)] if unequal else None

    def case(precision):
        return W.random_smooth(seed, N, nx, ny, rho=rho, wall_y=wall, amp_u=0.01, sigma=1e-3,
                               grad_scheme=1, precision=precision)

    a = gpu_run(case("fp32"), 8)
    b = gpu_run(case("fp32"), 8, kernel="generic")
    e = gpu_run(case("fp64"), 8, kernel="generic")
    for k in ("phi", "u", "p"):
        x, y, z = (np.asarray(m[k]) for m in (a, b, e))
        if np.array_equal(x, y, equal_nan=True):
            continue
        bound = max(1e-6 * np.abs(y).max(), 2 * np.abs(y - z).max())
        assert np.abs(x - y).max() <= bound, k
