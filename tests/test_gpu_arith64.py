"""FP64 rays whose values leave the window of the products on the integer
pipes (arith64.cuh): their attempts run with plain FP64 instructions, beside
ordinary rays in the same warps, and both agree with the oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_2202_00086_gb300 as osr

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("integrator", [osr.RKCK45, osr.RKDP45])
@pytest.mark.parametrize("a", [0.0, 1e-170, 0.9])
def test_rays_outside_the_window(a, integrator):
    n = 96
    rng = np.random.default_rng(3)
    st = np.zeros((n, 6))
    st[:, 1] = rng.uniform(6.0, 60.0, n)
    st[:, 2] = rng.uniform(0.4, np.pi - 0.4, n)
    st[:, 5] = rng.uniform(-2.0, 2.0, n)
    E, L = np.full(n, 1.0), rng.uniform(-4.0, 4.0, n)
    st[:, 4] = rng.uniform(0.2, 1.0, n)
    st[::3, 4] = 0.0           # radial turning points
    st[1::6, 4] = 1e-25
    L[4::6] = 0.0
    st[5::12, 5] = 0.0
    s, e, l = (torch.tensor(v, device="cuda") for v in (st, E, L))
    out = osr.trace_states(a, 1000.0, s, e, l, integrator=integrator, max_steps=2000)
    torch.cuda.synchronize()
    ref = oracle.trace_states(a, 1000.0, st, E, L, max_steps=2000, integrator=integrator)
    # the bars of the parity suite: fates equal, positions within 1e-8 on a stopping surface
    # (not after 2,000 steps of a bound orbit, which ends at the step cap)
    assert np.array_equal(out["status"].cpu().numpy(), ref["status"])
    ends = (ref["status"] == osr.STATUS_CAPTURED) | (ref["status"] == osr.STATUS_ESCAPED)
    assert ends.sum() >= n // 2
    for key in ("r", "theta", "phi"):
        got = out[key].cpu().numpy()[ends]
        err = np.abs(got - ref[key][ends]) / np.maximum(1.0, np.abs(ref[key][ends]))
        assert err.max() <= 1e-8, (key, float(err.max()))
    # in warps of their own they give the same bits
    alone = osr.trace_states(a, 1000.0, s, e, l, integrator=integrator, max_steps=2000,
                             block_size=32, persistent=True,
                             workspace=torch.empty(osr.workspace_bytes(1), dtype=torch.uint8,
                                                   device="cuda"))
    for k in range(0, n, 7):
        one = osr.trace_states(a, 1000.0, s[k:k + 1].clone(), e[k:k + 1].clone(),
                               l[k:k + 1].clone(), integrator=integrator, max_steps=2000)
        for key in out:
            assert torch.equal(one[key][0], out[key][k]), (key, k)
            assert torch.equal(alone[key][k], out[key][k]), (key, k)
