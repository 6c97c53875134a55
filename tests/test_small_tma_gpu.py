"""The TMA-pipelined FP32 kernel on grids that take the generic kernel by
default (LBM_NPHASE_KERNEL=pipelined), and both by rule on either side of the
line (608 tiles of 32 x 8 nodes), against the generic kernel: the same step and
arithmetic, within 1e-6 of the largest value (the bound of the pipelined
kernel's other comparisons)."""
import os

import numpy as np
import pytest

from paper_1904_12553_gb300 import workloads as W
from test_parity_gpu import _accept, _gpu, gpu_run, maxdiff  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def forced(w, steps):
    from paper_1904_12553_gb300 import Solver
    os.environ["LBM_NPHASE_KERNEL"] = "pipelined"
    try:
        s = Solver(w.params)
    finally:
        os.environ.pop("LBM_NPHASE_KERNEL", None)
    assert s.pipelined or w.params["nx"] % 8
    s.init(w.c0, w.u0)
    s.step(steps)
    m = s.moments()
    s.close()
    return m


def check(a, b):
    for k in ("phi", "u", "p"):
        assert maxdiff(a[k], b[k]) <= 1e-6 * (np.abs(b[k]).max() + 1e-30), k


def case(N, nx, ny, wall):
    seed = 7 * N + nx + ny + wall
    rng = np.random.default_rng(seed)
    return W.random_smooth(seed, N, nx, ny, wall_y=wall, amp_u=0.02, precision="fp32",
                           sigma=W.sample_sigma(rng, N, accept=_accept()))


@pytest.mark.parametrize("nx,ny", [(64, 48), (96, 40), (64, 16), (96, 45), (8, 8), (520, 300)])
@pytest.mark.parametrize("N", [2, 3, 4, 5])
@pytest.mark.parametrize("wall", [0, 1])
def test_pipelined_at_every_size(N, nx, ny, wall):
    w = case(N, nx, ny, wall)
    check(forced(w, 30), gpu_run(w, 30, kernel="generic"))


@pytest.mark.parametrize("nx,ny", [(512, 304), (512, 312)])  # 608 and 624 tiles
@pytest.mark.parametrize("N", [2, 5])
def test_either_side_of_the_line(N, nx, ny):
    w = case(N, nx, ny, 0)
    check(gpu_run(w, 20), gpu_run(w, 20, kernel="generic"))


# Rows padded to a multiple of 8 nodes: widths and heights of every remainder
# that moves the wrapped column and row (one tile and less, just over a tile,
# the column x = nx inside or beyond the last tile).
RAGGED = [(1, 1), (5, 3), (9, 20), (31, 9), (33, 8), (34, 17), (150, 37), (255, 10), (519, 301)]


@pytest.mark.parametrize("nx,ny", RAGGED)
@pytest.mark.parametrize("N", [2, 3, 5])
@pytest.mark.parametrize("wall", [0, 1])
def test_padded_rows(N, nx, ny, wall):
    w = case(N, nx, ny, wall)
    check(forced(w, 30), gpu_run(w, 30, kernel="generic"))


@pytest.mark.parametrize("nx,ny", [(37, 21), (1030, 700)])
@pytest.mark.parametrize("device", [False, True])
def test_padded_state_round_trip(nx, ny, device):
    """The blob holds dense rows: a run resumed from it (in another handle)
    continues bit for bit, and its size is that of nx x ny nodes."""
    from paper_1904_12553_gb300 import Solver
    w = case(3, nx, ny, 0)
    a, b = Solver(w.params), Solver(w.params)
    a.init(w.c0, w.u0)
    a.step(5)
    blob = a.get_state(device=device)
    assert blob.numel() == 64 + 4 * nx * ny * (2 * 9 + 8 + 2 + 2)
    a.step(5)
    b.set_state(blob)
    b.step(5)
    assert torch.equal(a.get_state()[64:], b.get_state()[64:])
    ma, mb = a.moments(), b.moments()
    for k in ma:
        np.testing.assert_array_equal(ma[k], mb[k])
    a.close()
    b.close()
