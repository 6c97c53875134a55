"""The start without a velocity, two phases in FP32 (a kernel of its own): the
state of a start with a zero velocity, value for value, and faster than it (1280 x
1024, us: 215 and 350; in one kernel 395 and 411). 0.9 times is allowed."""
import pytest

from paper_1904_12553_gb300 import Solver, workloads as W
from test_parity_gpu import _gpu  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def start(nx, ny, wall, p0=0.0):
    s = Solver(W.base_params(2, nx, ny, 1e-3, precision="fp32", wall_y=wall))
    g = torch.Generator(device="cuda").manual_seed(nx + ny)
    c = torch.rand((2, ny, nx), generator=g, device="cuda", dtype=torch.float64)
    c[:, : ny // 2] = torch.tensor([1.0, 0.0], device="cuda", dtype=torch.float64)[:, None, None]
    c = (c / c.sum(0)).contiguous()
    return s, c, torch.zeros((2, ny, nx), device="cuda", dtype=torch.float64)


@pytest.mark.parametrize("nx,ny", [(1, 1), (33, 9), (150, 37), (1501, 301)])
@pytest.mark.parametrize("wall", [0, 1])
@pytest.mark.parametrize("p0", [0.0, 1e-3])
def test_rest_start_is_a_zero_velocity_start(nx, ny, wall, p0):
    s, c, u = start(nx, ny, wall)
    s.init(c, None, p0)
    rest = s.get_state()[64:].view(torch.float32)
    s.init(c, u, p0)
    assert torch.equal(rest, s.get_state()[64:].view(torch.float32))
    s.close()


def test_rest_start_is_the_faster():
    s, c, u = start(1280, 1024, 0)

    def us(v):
        best = 1e9
        for _ in range(7):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            torch.cuda.synchronize()
            a.record()
            s.init(c, v)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 1e3)
        return best

    us(u)
    rest, moving = us(None), us(u)
    s.close()
    assert rest <= 0.9 * moving, (rest, moving)
