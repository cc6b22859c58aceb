"""A batch plan asks for the occupancy of its kernels when it is made and not
when it launches: the real host library around two stand-in kernels (for
launches of under and of at least 1,000 rays), with the query counted."""
import ctypes
import subprocess

import pytest
import torch

import paper_2202_00086_gb300 as osr
from paper_2202_00086_gb300 import build as lib_build

pytestmark = pytest.mark.gpu

UNIT = r"""
#include <cuda_runtime.h>
#include "osiris_internal.h"
extern "C" { int queries = 0; }
extern "C" cudaError_t counted_occupancy(int* blocks, const void*, int, size_t) {
  ++queries;
  *blocks = 2;
  return cudaSuccess;
}
namespace osiris_impl {
// the grid's blocks and a mark of the kernel, for the first request
template <int kMark>
__global__ void stand_in(const __grid_constant__ KernelArgs A) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    A.reqs[0].out.r[0] = gridDim.x;
    A.reqs[0].out.r[1] = kMark;
  }
}
template <bool kOne>
static const void* by_rays(int64_t rays) {
  return rays < 1000 || kOne ? (const void*)stand_in<1> : (const void*)stand_in<2>;
}
const void* trace_kernel_fp64(Kernel, int, int, int64_t rays) { return by_rays<true>(rays); }
const void* trace_kernel_mixed(Kernel, int, int, int64_t rays) { return by_rays<false>(rays); }
const void* trace_kernel_df64(Kernel, int, int, int64_t rays) { return by_rays<false>(rays); }
int launch_pipe_probe(int, int, int64_t, int, double*, void*) { return 1; }
int probe_resident_blocks(int, int, int*) { return 1; }
}  // namespace osiris_impl
"""


@pytest.fixture(scope="module")
def library(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan_create")
    (d / "stand_in.cu").write_text(UNIT)
    lib = d / "libosiris_plan_create.so"
    nvcc = [lib_build._nvcc()] + lib_build.ARCH
    flags = ["-O2", "-std=c++17", "-Xcompiler", "-fPIC", "-I" + lib_build.CSRC,
             "-I" + lib_build.ROOT + "/include"]
    rename = "-DcudaOccupancyMaxActiveBlocksPerMultiprocessor=counted_occupancy"
    for src, obj, more in ((lib_build.CSRC + "/osiris_api.cu", "api.o", [rename]),
                           (str(d / "stand_in.cu"), "stand_in.o", [])):
        subprocess.run(nvcc + flags + more + ["-c", src, "-o", str(d / obj)], check=True)
    subprocess.run(nvcc + ["-shared", "-o", str(lib), str(d / "api.o"), str(d / "stand_in.o")],
                   check=True)
    return osr.load(str(lib)), ctypes.c_int.in_dll(ctypes.CDLL(str(lib)), "queries")


@pytest.mark.parametrize("precision,kernels", [(osr.FP64, 1), (osr.DF64, 2), (osr.MIXED, 2)])
def test_occupancy_is_asked_for_at_creation(library, precision, kernels):
    lib, queries = library
    with osr.using_library(lib):
        cam = osr.Camera(0.5, 1000.0, 60.0, (-8, 8, -8, 8), 300, 300)
        out = osr.alloc_outputs(cam.n_rays)
        ws = torch.empty(osr.workspace_bytes(1), dtype=torch.uint8, device="cuda")
        before = queries.value
        plan = osr.BatchPlan(1, workspace=ws, precision=precision)
        assert queries.value == before + kernels
        sms = torch.cuda.get_device_properties(0).multi_processor_count
        for n in (100, 5000, 999, 1000, 90000, 1):
            plan.launch([dict(camera=cam, out=out, first_ray=0, n_rays=n)])
            torch.cuda.synchronize()
            got = out["r"][:2].tolist()
            assert got == [min((n + 127) // 128, 2 * sms), 2 if n >= 1000 and kernels == 2 else 1]
        assert queries.value == before + kernels
        plan.close()
