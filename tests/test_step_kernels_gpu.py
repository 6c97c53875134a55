"""Solver.kernels names the kernels that a step launches, as the profiler sees
them, for every form, either side of the rules, and under both values of
LBM_NPHASE_KERNEL; the comparisons that force the TMA kernels do run them."""
import os
import re

import pytest

from paper_1904_12553_gb300 import Solver, workloads as W
from test_parity_gpu import PIPE, _gpu  # noqa: F401
from test_small_tma_gpu import RAGGED

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RHO = [3.0, 1.0, 2.0, 5.0, 4.0]


def solver(N, shape, prec, nu=0, g40=0, wall=0, env=None):
    old = os.environ.pop("LBM_NPHASE_KERNEL", None)
    if env:
        os.environ["LBM_NPHASE_KERNEL"] = env
    try:
        kw = dict(rho=RHO[:N] if nu else None, precision=prec, wall_y=wall)
        p = (W.base_params3(N, *shape, 0.01, **kw) if len(shape) == 3
             else W.base_params(N, *shape, 0.01, grad_scheme=g40, **kw))
        return Solver(p)
    finally:
        os.environ.pop("LBM_NPHASE_KERNEL", None)
        if old is not None:
            os.environ["LBM_NPHASE_KERNEL"] = old


def profiled(f):
    with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CUDA]) as p:
        f()
        torch.cuda.synchronize()
    return sorted(p.events(), key=lambda e: e.time_range.start)


@pytest.fixture(scope="module")
def profiler(_gpu):
    """The first profile of a process sees no kernels; a second one does, unless
    something else in the process holds the profiler."""
    x = torch.zeros(1024, device="cuda")
    profiled(lambda: x.add_(1))
    return any("elementwise" in e.name for e in profiled(lambda: x.add_(1)))


def launched(s):
    """Kernels of one step, in order, and whether a tile kernel has ring warps."""
    sh = (s.N,) + s.grid
    s.init(torch.full(sh, 1.0 / s.N, dtype=torch.float64, device="cuda"))
    s.step(1)
    torch.cuda.synchronize()
    out = []
    for e in profiled(lambda: s.step(1)):
        if "lbm::" not in e.name:
            continue
        m = re.search(r"lbm::(\w+)(?:<([^>]*)>)?", e.name)
        rw = m.group(1) == "tile_kernel" and m.group(2).split(",")[-1].strip() != "0"
        out.append(m.group(1) + (" (ring warps)" if rw else ""))
    return " + ".join(out)


CASES = [
    (3, (64, 48), "fp64", 0, 0, None, "step64_kernel"),
    (3, (64, 48), "fp64", 1, 0, None, "pot64_kernel + coll64_kernel"),
    (3, (64, 48), "fp64", 0, 1, None, "pot64_kernel + coll64_kernel"),
    (3, (64, 48), "fp64", 0, 0, "generic", "tile_kernel"),
    (3, (128, 128), "fp32", 0, 0, None, "tile_kernel (ring warps)"),
    (3, (128, 128), "fp32", 1, 1, None, "tile_kernel (ring warps)"),
    (5, (512, 304), "fp32", 0, 0, None, "tile_kernel"),
    (3, (128, 128), "fp32", 0, 0, "pipelined", "tile_kernel_tma"),
    (3, (130, 33), "fp32", 0, 0, "pipelined", "tile_kernel_tma"),
    (3, (1501, 997), "fp32", 0, 0, None, "tile_kernel_tma"),
    (3, (1501, 997), "fp32", 0, 0, "generic", "tile_kernel"),
    (3, (9, 20000), "fp32", 0, 0, None, "tile_kernel"),
    (5, (1024, 1024), "fp32", 1, 0, None, "tile_kernel"),
    (4, (64, 48), "bf16", 0, 0, None, "tile_kernel_tma"),
    (4, (65, 48), "fp16", 0, 0, None, "tile_kernel"),
    (3, (40, 17, 23), "fp64", 0, 0, None, "phi3_kernel + step3_kernel"),
    (3, (40, 17, 23), "bf16", 1, 0, None, "phi3_kernel + pot3_kernel + step3_kernel"),
    (3, (40, 17, 23), "fp32", 0, 0, None, "phi3_kernel + step3_kernel"),
    (3, (40, 17, 23), "fp32", 0, 0, "pipelined", "march3_tma_kernel"),
    (3, (128, 128, 64), "fp32", 0, 0, None, "march3_tma_kernel"),
    (3, (40, 17, 23), "fp32", 0, 0, "generic", "tile3_kernel"),
]
# either side of the pipelined kernel's line (1216, 912, 1140, 912 tiles)
CASES += [(N, sh, "fp32", 0, 0, None, k) for N, sh, k in [
    (2, (1024, 304), "tile_kernel"), (2, (1024, 312), "tile_kernel_tma"),
    (3, (768, 304), "tile_kernel"), (3, (773, 306), "tile_kernel_tma"),
    (4, (960, 304), "tile_kernel"), (4, (955, 312), "tile_kernel_tma"),
    (5, (768, 304), "tile_kernel"), (5, (771, 309), "tile_kernel_tma"),
    (4, (65, 5001), "tile_kernel"), (4, (20001, 12), "tile_kernel"), (3, (20001, 9), "tile_kernel"),
    (4, (20001, 17), "tile_kernel_tma")]]


@pytest.mark.parametrize("N,shape,prec,nu,g40,env,want", CASES)
def test_kernels_are_the_ones_launched(profiler, N, shape, prec, nu, g40, env, want):
    s = solver(N, shape, prec, nu, g40, env=env)
    try:
        assert s.kernels == want
        if not profiler:
            pytest.skip("no profiler in this process")
        assert launched(s) == want
    finally:
        s.close()


@pytest.mark.parametrize("wall", [0, 1])
def test_forced_comparisons_run_the_tma_kernels(wall):
    """The inputs of the pipelined and z-marching comparisons that set
    LBM_NPHASE_KERNEL=pipelined."""
    grids = {(N, (nx, ny)) for N, p, nx, ny, _ in PIPE if p == "fp32"}
    grids |= {(N, sh) for N in (2, 3, 5) for sh in RAGGED}
    for N, sh in sorted(grids):
        s = solver(N, sh, "fp32", wall=wall, env="pipelined")
        assert s.kernels == "tile_kernel_tma", (N, sh)
        s.close()
    for N in (2, 3, 4):
        for sh in ((40, 17, 23), (8, 8, 1), (64, 24, 70), (32, 16, 12)):
            s = solver(N, sh, "fp32", wall=wall, env="pipelined")
            assert s.kernels == "march3_tma_kernel", (N, sh)
            s.close()


def test_timeout_recovery_on_the_pipelined_kernel():
    """A wait that runs out, then a new start, on the kernel whose waits these
    are (the grid of the timeout test runs the generic one by rule)."""
    from paper_1904_12553_gb300 import LbmError, binding
    w = W.random_smooth(8, 3, 64, 40, precision="fp32", amp_u=0.01)
    runs = []
    for fail in (True, False):
        s = solver(3, (64, 40), "fp32", env="pipelined")
        assert s.kernels == "tile_kernel_tma"
        s.init(w.c0, w.u0)
        if fail:
            s.step(3)
            binding.lbm_nphase_selftest_wait_timeout(s.handle)
            with pytest.raises(LbmError) as e:
                s.diagnostics()
            assert e.value.status == 4  # LBM_ETIMEOUT
            with pytest.raises(LbmError):
                s.step(1)
            s.init(w.c0, w.u0)
        s.step(6)
        runs.append(s.get_state()[64:])
        s.close()
    assert torch.equal(*runs)
