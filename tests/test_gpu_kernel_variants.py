"""The register variants of the trace kernels: a launch of one ray less than the
line takes the small variant, one of as many rays as the line the large one,
and both give every ray the same bits (the same operations in the same order)."""
import pytest
import torch

import paper_2202_00086_gb300 as osr

pytestmark = pytest.mark.gpu

LANES = 152 * 256


@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("precision,integrator,q,lines", [
    (osr.FP64, osr.RKCK45, None, 5), (osr.FP64, osr.RKDP45, None, 5),
    (osr.DF64, osr.RKCK45, None, 10), (osr.DF64, osr.RKDP45, None, 10),
    (osr.DF64, osr.RKCK45, 0.5, 8), (osr.DF64, osr.RKDP45, 0.5, 8),
    (osr.MIXED, osr.RKCK45, None, 8), (osr.MIXED, osr.RKDP45, None, 8),
    (osr.MIXED, osr.RKCK45, 0.5, 5), (osr.MIXED, osr.RKDP45, 0.5, 5)])
def test_both_sides_of_the_line(precision, integrator, q, lines, persistent):
    line = lines * LANES
    g = torch.Generator().manual_seed(lines)
    st = torch.zeros(line, 6, dtype=torch.float64)
    st[:, 1] = 30.0
    st[:, 2] = 0.3 + 2.5 * torch.rand(line, generator=g, dtype=torch.float64)
    st[:, 4] = 0.5 - torch.rand(line, generator=g, dtype=torch.float64)
    E = torch.full((line,), 1.2, dtype=torch.float64)
    L = 8.0 * torch.rand(line, generator=g, dtype=torch.float64) - 4.0
    kw = dict(precision=precision, integrator=integrator, tol=1e-7, q=q, max_steps=200)
    if persistent:
        kw.update(persistent=True, workspace=torch.empty(osr.workspace_bytes(1),
                                                         dtype=torch.uint8, device="cuda"))
    got = []
    for n in (line - 1, line):
        out = osr.alloc_outputs(n)
        for t in out.values():
            t.fill_(77)
        osr.trace_states(0.0 if q is not None else 0.9, 100.0, st[:n].cuda(), E[:n].cuda(),
                         L[:n].cuda(), out=out, **kw)
        torch.cuda.synchronize()
        got.append(out)
    for k in got[0]:
        assert not (got[1][k] == 77).all(), k
        assert torch.equal(got[0][k].view(torch.uint8), got[1][k][:line - 1].view(torch.uint8)), k
