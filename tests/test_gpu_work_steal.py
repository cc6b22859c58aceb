"""Plain FP64 and DF64 launches, whose blocks take over the indices of blocks
that have not started (csrc/work_steal.cuh): every ray is traced exactly once,
with the same bits as on a persistent grid, at ray counts around one chunk (32
rays), one block and the line where chunks change size (58,368 rays)."""
import pytest
import torch

import paper_2202_00086_gb300 as osr

pytestmark = pytest.mark.gpu


def _states(n):
    g = torch.Generator().manual_seed(n)
    st = torch.zeros(n, 6, dtype=torch.float64)
    st[:, 1] = 30.0
    st[:, 2] = 0.3 + 2.5 * torch.rand(n, generator=g, dtype=torch.float64)
    st[:, 4] = 0.5
    E = torch.full((n,), 1.2, dtype=torch.float64)
    L = 8.0 * torch.rand(n, generator=g, dtype=torch.float64) - 4.0
    return st.cuda(), E.cuda(), L.cuda()


@pytest.mark.parametrize("precision", [osr.FP64, osr.DF64])
@pytest.mark.parametrize("n,block,per_lane", [
    (1, 0, 0), (31, 32, 0), (33, 0, 0), (127, 0, 1), (129, 96, 0), (1000, 256, 3),
    (58367, 0, 0), (58368, 128, 0), (58369, 0, 0), (58400, 32, 0), (70001, 256, 2),
    (130000, 64, 0)])
def test_every_ray_once(precision, n, block, per_lane):
    st, E, L = _states(n)
    kw = dict(precision=precision, tol=1e-8, block_size=block, rays_per_lane=per_lane)
    stats = osr.new_stats()
    out = osr.alloc_outputs(n)
    for t in out.values():
        t.fill_(77)  # no status, and no valid step count of these rays
    osr.trace_states(0.9, 1000.0, st, E, L, out=out, stats=stats, **kw)
    ref = osr.trace_states(0.9, 1000.0, st, E, L, persistent=True,
                           workspace=torch.empty(osr.workspace_bytes(1), dtype=torch.uint8,
                                                 device="cuda"), **kw)
    torch.cuda.synchronize()
    assert osr.decode_stats(stats)["rays"] == n
    for k in out:
        assert torch.equal(out[k], ref[k]), k


@pytest.mark.parametrize("precision", [osr.FP64, osr.DF64])
def test_renders_on_two_streams_and_in_a_graph(precision):
    """Launches that run at the same time, and a captured launch replayed."""
    cam = osr.Camera(0.9, 1000.0, 60.0, (-8, 8, -8, 8), 301, 211)
    ref = osr.trace(cam, precision=precision, tol=1e-8)
    torch.cuda.synchronize()
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    a, b, c = (osr.alloc_outputs(cam.n_rays) for _ in range(3))
    torch.cuda.synchronize()
    osr.trace(cam, out=a, stream=s1, precision=precision, tol=1e-8)
    osr.trace(cam, out=b, stream=s2, precision=precision, tol=1e-8)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        osr.trace(cam, out=c, precision=precision, tol=1e-8)
    for _ in range(2):
        for t in c.values():
            t.zero_()
        graph.replay()
        torch.cuda.synchronize()
        for k in ref:
            assert torch.equal(c[k], ref[k]), k
    for k in ref:
        assert torch.equal(a[k], ref[k]) and torch.equal(b[k], ref[k]), k
