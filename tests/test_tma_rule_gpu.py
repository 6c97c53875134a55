"""FP32 grids on either side of the rules that choose the pipelined kernel and
its stages, against the generic kernel: the same step and arithmetic, within
1e-6 of the largest value (the bound of the pipelined kernel's other
comparisons)."""
import pytest

from paper_1904_12553_gb300 import binding, workloads as W
from test_parity_gpu import _gpu, gpu_run  # noqa: F401
from test_small_tma_gpu import case, check

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# 1216, 912, 1140, 912 tiles at N = 2..5: on the line, and just above
@pytest.mark.parametrize("N,nx,ny", [(2, 1024, 304), (2, 1024, 312), (3, 768, 304), (3, 773, 306),
                                     (4, 960, 304), (4, 955, 312), (5, 768, 304), (5, 771, 309)])
@pytest.mark.parametrize("wall", [0, 1])
def test_either_side_of_the_line(N, nx, ny, wall):
    w = case(N, nx, ny, wall)
    check(gpu_run(w, 12), gpu_run(w, 12, kernel="generic"))


# N = 3: two stages and two CTAs per SM, and from 5017 tiles three and one
@pytest.mark.parametrize("nx,ny", [(1216, 1056), (1248, 1040), (1504, 1000), (1501, 1003),
                                   (97, 10037)])
@pytest.mark.parametrize("wall", [0, 1])
def test_stages_of_three_phases(nx, ny, wall):
    w = case(3, nx, ny, wall)
    check(gpu_run(w, 6), gpu_run(w, 6, kernel="generic"))


# narrow grids, and grids with few lanes in use: the generic kernel on dense rows
@pytest.mark.parametrize("N,nx,ny", [(2, 1, 9001), (3, 9, 9003), (5, 57, 4099), (4, 65, 5001),
                                     (3, 20001, 9)])
def test_narrow_grids(N, nx, ny):
    w = case(N, nx, ny, 0)
    check(gpu_run(w, 8), gpu_run(w, 8, kernel="generic"))


def test_dense_workspace_is_enough():
    """A workspace without room for padded rows is accepted: the grid runs on
    the generic kernel, with its bits."""
    w = case(3, 1501, 301, 0)
    need = binding.lbm_nphase_workspace_bytes(w.params)
    dense = binding.lbm_nphase_workspace_bytes({**w.params, "rho": [3.0, 1.0, 2.0]})
    assert dense < need
    ws = torch.empty(dense, dtype=torch.uint8, device="cuda")
    h = binding.lbm_nphase_create(w.params, ws.data_ptr(), dense,
                                  torch.cuda.current_stream().cuda_stream)
    c = torch.from_numpy(w.c0).cuda()
    u = torch.from_numpy(w.u0).cuda()
    binding.lbm_nphase_init(h, c.data_ptr(), u.data_ptr(), w.p0)
    binding.lbm_nphase_step(h, 8)
    phi = torch.empty((2, 301, 1501), dtype=torch.float64, device="cuda")
    binding.lbm_nphase_moments(h, phi=phi.data_ptr())
    binding.lbm_nphase_destroy(h)
    want = gpu_run(w, 8, kernel="generic")["phi"]
    assert (phi.cpu().numpy() == want).all()
    with pytest.raises(binding.LbmError):
        binding.lbm_nphase_create(w.params, ws.data_ptr(), dense - 256,
                                  torch.cuda.current_stream().cuda_stream)
