"""A plain launch whose blocks wait in vain for work to take over
(csrc/work_steal.cuh): the real host library and hand-over around a stand-in
kernel, built with a short patience and with requests that are not sent, so
that no answer comes and nothing is in flight when a warp gives up. The launch
ends, counts its warps that gave up, and a ray that no block traced has
STATUS_NONE, not what its buffer held before."""
import subprocess

import pytest
import torch

import paper_2202_00086_gb300 as osr
from paper_2202_00086_gb300 import build as lib_build

pytestmark = pytest.mark.gpu

UNIT = r"""
#include <cuda_runtime.h>
#include "work_steal.cuh"
namespace osiris_impl {
// gives every ray that it is handed the status CAPTURED, but for each 64th: lost
__global__ void stand_in(const __grid_constant__ KernelArgs A) {
  steal_init(A);
  bool drained = false;
  unsigned turns = 0;
  for (;;) {
    int64_t ray = 0;
    bool over = false;
    const int got = steal_refill(A, !drained, false, ray, over);
    if (got && ray % 64 != 63) A.single.out.status[ray] = OSIRIS_STATUS_CAPTURED;
    drained |= over;
    if (!__any_sync(0xffffffffu, got)) {
      if (steal_waits(A, drained, turns)) continue;
      break;
    }
    turns = 0;
  }
}
const void* trace_kernel_fp64(Kernel, int, int, int64_t) { return (const void*)stand_in; }
const void* trace_kernel_mixed(Kernel, int, int, int64_t) { return (const void*)stand_in; }
const void* trace_kernel_df64(Kernel, int, int, int64_t) { return (const void*)stand_in; }
int launch_pipe_probe(int, int, int64_t, int, double*, void*) { return 1; }
int probe_resident_blocks(int, int, int*) { return 1; }
}  // namespace osiris_impl
"""


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    d = tmp_path_factory.mktemp("give_up")
    (d / "stand_in.cu").write_text(UNIT)
    lib = d / "libosiris_give_up.so"
    subprocess.run([lib_build._nvcc()] + lib_build.ARCH +
                   ["-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-shared",
                    "-DOSIRIS_STEAL_MUTE", "-DOSIRIS_STEAL_PATIENCE=1000u",
                    "-I" + lib_build.CSRC, "-I" + lib_build.ROOT + "/include",
                    lib_build.CSRC + "/osiris_api.cu", str(d / "stand_in.cu"), "-o", str(lib)],
                   check=True)
    return osr.load(str(lib))


@pytest.mark.parametrize("precision", [osr.FP64, osr.DF64])
@pytest.mark.parametrize("n,block", [(1, 32), (63, 64), (300, 128), (58369, 128)])
def test_untraced_rays_and_the_count(library, precision, n, block):
    chunk = 32 if n > 58368 else block
    blocks = (n + chunk - 1) // chunk  # none takes over another's index: all of them run
    st = torch.zeros(n, 6, dtype=torch.float64, device="cuda")
    E, L = torch.ones_like(st[:, 0]), torch.zeros_like(st[:, 0])
    out, stats = osr.alloc_outputs(n), osr.new_stats()
    out["status"].fill_(77)
    with osr.using_library(library):
        osr.trace_states(0.5, 1000.0, st, E, L, out=out, stats=stats, precision=precision,
                         block_size=block)
        torch.cuda.synchronize()
    want = torch.full((n,), osr.STATUS_CAPTURED, dtype=torch.uint8)
    want[63::64] = 0
    assert torch.equal(out["status"].cpu(), want)
    assert osr.decode_stats(stats)["gave_up"] == blocks * block // 32
