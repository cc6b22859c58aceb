"""Small DF64 rounds of the server wait for renders to share them: with a fake
backend and a clock moved by hand."""
import numpy as np
import pytest

import paper_2202_00086_gb300 as osr
from paper_2202_00086_gb300 import serve, workloads
from test_serve_host import FakeBackend


class Clock:
    t = 0.0

    def __call__(self):
        return self.t


def _server(clock, **kw):
    ref = [None]
    ref[0] = serve.RenderServer(backend=FakeBackend(ref), clock=clock, max_inflight=4,
                                round_rays=3000, min_chunk=500, **kw)
    return ref[0]


def _render(nx, ny, tol=1e-10):
    return workloads.render(0.5, 1000.0, 60.0, (-8, 8, -8, 8), nx, ny, tol=tol)


def test_small_rounds_share_launches():
    clock = Clock()
    srv = _server(clock, coalesce_s=0.003)
    srv.submit(_render(64, 66))  # 4,224 rays: a full round at once, 1,224 rays left
    srv.step()
    assert srv.round_entries == [1]
    clock.t = 0.002
    srv.submit(_render(24, 24))
    srv.step()
    assert srv.round_entries == [1]
    clock.t = 0.0031  # the rest of the first render and the second share a round
    srv.step()
    assert srv.round_entries == [1, 2]
    clock.t = 0.007  # long after the last round: at once
    srv.submit(_render(8, 8))
    srv.step()
    assert srv.round_entries == [1, 2, 1]
    clock.t = 0.008  # rays enough for a full round: at once
    srv.submit(_render(60, 50))
    srv.step()
    assert srv.round_entries == [1, 2, 1, 1]
    while not srv.idle():
        clock.t += 0.001
        srv.step()
    assert len(srv.done) == 4


@pytest.mark.parametrize("kw,tol", [(dict(coalesce_s=0.0), 1e-10),
                                    (dict(), 1e-10),  # a backend without a default
                                    (dict(coalesce_s=0.003, precision=osr.FP64), 1e-10),
                                    (dict(coalesce_s=0.003, loose_precision=osr.MIXED), 1e-8)])
def test_no_waiting(kw, tol):
    clock = Clock()
    srv = _server(clock, **kw)
    for k in range(3):
        srv.submit(_render(16, 16, tol))
        srv.step()
        assert srv.rounds == k + 1
        clock.t += 1e-4


def test_the_last_renders_of_a_stream_do_not_wait():
    clock = Clock()
    srv = _server(clock, coalesce_s=1e9)
    arrivals = [(0.0, _render(16, 16)) for _ in range(2)] + [(0.0, _render(70, 70))]
    summary = srv.run(arrivals, realtime=False, poll_s=0)
    assert summary["renders"] == 3
    assert np.array_equal([sum(n for _, n in r.chunks) for r in sorted(srv.done,
                                                                       key=lambda r: r.rid)],
                          [256, 256, 4900])
