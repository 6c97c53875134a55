"""Batches whose state is beyond 48 MB, where every other step walks the items
backwards: the single grids' bits under every schedule, and lists that stay
balanced on both kinds of step."""
import numpy as np
import pytest

from paper_1904_12553_gb300 import Batch, Solver, workloads as W
from test_parity_gpu import _accept, _gpu  # noqa: F401

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def grids(sizes):
    out = []
    for i, (N, nx, ny) in enumerate(sizes):
        rng = np.random.default_rng(i)
        out.append(W.random_smooth(i, N, nx, ny, wall_y=i % 2, amp_u=0.02, precision="fp32",
                                   sigma=W.sample_sigma(rng, N, accept=_accept())))
    return out


MIXED = [(2, 264, 203), (5, 256, 256), (3, 520, 131), (4, 128, 320), (5, 296, 299), (2, 512, 256)]


@pytest.fixture(scope="module")
def singles():
    out = []
    for w in grids(MIXED):
        s = Solver(w.params)
        s.init(w.c0, w.u0)
        per = {}
        for steps in (6, 7):
            s.step(steps - s.steps_taken)
            per[steps] = s.get_state()[64:]
        out.append(per)
        s.close()
    return out


@pytest.mark.parametrize("steps", [6, 7])
@pytest.mark.parametrize("sched,chunk", [(0, 1), (1, 1), (2, 1), (2, 4), (2, 16)])
def test_large_batch_matches_single_grids(singles, sched, chunk, steps):
    from paper_1904_12553_gb300 import binding
    ws = grids(MIXED)
    # read and written values of a node-step: 10 N in FP32
    assert sum(4 * 10 * w.params["N"] * w.V for w in ws) >= 48 << 20
    b = Batch([w.params for w in ws])
    b.set_schedule(8, sched, pipelined=True, chunk=chunk)
    for i, w in enumerate(ws):
        b.init(i, w.c0, w.u0)
    b.step(steps)
    for i, w in enumerate(ws):
        n = binding.lbm_nphase_state_bytes(b.case_handle(i))
        blob = torch.empty(n, dtype=torch.uint8)
        binding.lbm_nphase_get_state(b.case_handle(i), blob.data_ptr(), n)
        a, s = (x.view(torch.float32) for x in (blob[64:], singles[i][steps]))
        scale = s.abs().max()
        assert torch.isfinite(s).all() and (a - s).abs().max() <= 1e-6 * scale, i
    b.close()


def test_lists_stay_balanced_on_every_step():
    """24 grids of two and five phases: the dearest list is the same in both
    directions, so a step back takes about as long as a step forth; lists cut
    for other items took 1.5 times. 1.2 times is allowed."""
    ps = [W.base_params(2 if i % 2 else 5, 512, 512, 1e-3, precision="fp32") for i in range(24)]
    b = Batch(ps)
    b.set_schedule(8, 1, pipelined=True)
    for i, p in enumerate(ps):
        b.init(i, np.full((p["N"], 512, 512), 1.0 / p["N"]))
    b.step(4)
    took = [1e9, 1e9]
    for k in range(40):
        a, z = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record()
        b.step(1)
        z.record()
        torch.cuda.synchronize()
        took[k % 2] = min(took[k % 2], a.elapsed_time(z) * 1e3)
    b.close()
    assert max(took) <= 1.2 * min(took), took
