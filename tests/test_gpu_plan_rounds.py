"""Rounds of a batch plan by size: every round takes the kernel that
osiris_trace_batch takes for as many rays, from one round to the next of the
same plan, and small rounds are no slower than that."""
import pytest
import torch

import paper_2202_00086_gb300 as osr

pytestmark = pytest.mark.gpu

LANES = 152 * 256


def _setup(precision, q, side):
    cam = osr.Camera(0.9 if q is None else 0.0, 100.0, 60.0, (-8, 8, -8, 8), side, side, q=q)
    plan = osr.BatchPlan(2, precision=precision, tol=1e-7,
                         spacetime=osr.SPACETIME_KERR if q is None else osr.SPACETIME_QMETRIC,
                         workspace=torch.empty(osr.workspace_bytes(2), dtype=torch.uint8,
                                               device="cuda"))
    return cam, plan


@pytest.mark.parametrize("precision,q,large", [
    (osr.FP64, None, 5), (osr.DF64, None, 10), (osr.DF64, 0.5, 8), (osr.MIXED, None, 8),
    (osr.MIXED, 0.5, 5)])
def test_rounds_of_every_size_in_turn(precision, q, large):
    """From a few hundred rays to just above the line of the large kernels
    (a multiple of 256 lanes on each of 152 SMs), and back."""
    cam, plan = _setup(precision, q, 640)
    ref = osr.trace(cam, precision=precision, tol=1e-7)
    out = osr.alloc_outputs(cam.n_rays)
    for first, n in ((7, 500), (300, 20001), (0, large * LANES + 3), (11, 301),
                     (640, large * LANES), (5000, 4096), (9000, large * LANES - 1)):
        for t in out.values():
            t.fill_(77)
        cut = first + n // 3
        plan.launch([dict(camera=cam, out=out, first_ray=first, n_rays=cut - first),
                     dict(camera=cam, out=out, first_ray=cut, n_rays=first + n - cut)])
        torch.cuda.synchronize()
        for k in ref:
            assert torch.equal(out[k][first:first + n], ref[k][first:first + n]), (n, k)
            assert (out[k][:first] == 77).all() and (out[k][first + n:] == 77).all(), (n, k)
    plan.close()


def _least_ms(f):
    best = float("inf")
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        a.record()
        f()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("n", [500, 3000])
@pytest.mark.parametrize("precision,q", [(osr.DF64, None), (osr.DF64, 0.5), (osr.MIXED, None),
                                         (osr.MIXED, 0.5)])
def test_small_rounds_take_the_time_of_a_batch(precision, q, n):
    cam, plan = _setup(precision, q, 100)
    out = osr.alloc_outputs(cam.n_rays)
    ws = torch.empty(osr.workspace_bytes(1), dtype=torch.uint8, device="cuda")
    reqs = [dict(camera=cam, out=out, first_ray=3000, n_rays=n)]
    batch = _least_ms(lambda: osr.trace_batch(reqs, workspace=ws, precision=precision, tol=1e-7))
    assert _least_ms(lambda: plan.launch(reqs)) <= 1.2 * batch
    plan.close()
