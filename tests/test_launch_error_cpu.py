"""A launch that CUDA refuses is reported by the library's return value alone: the runtime's last error is
clear afterwards, so that the caller's next check is about the caller's own calls.  (No GPU needed: the
runtime's two calls are stood in for.)"""
import os

import pytest
from host_build import host_lib

SOURCE = """
#include <cuda_runtime.h>
static cudaError_t outcome, last;
template <typename... K, typename... A>
cudaError_t fake_launch(const cudaLaunchConfig_t*, void (*)(K...), A&&...) {
  if (outcome != cudaSuccess) last = outcome;
  return outcome;
}
static cudaError_t fake_last() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
#define cudaLaunchKernelEx fake_launch
#define cudaGetLastError fake_last
#include "internal.h"
static void kernel(int) {}
extern "C" int launch(int result) {
  outcome = (cudaError_t)result;
  return (int)vp::launch_pdl(kernel, dim3(1), 32, 0, nullptr, 1);
}
extern "C" int set_last(int e) { return (int)(last = (cudaError_t)e); }
extern "C" int get_last() { return (int)last; }
"""


def test_refused_launch_leaves_no_last_error(tmp_path):
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not os.path.exists(os.path.join(cuda, "cuda_runtime.h")):
        pytest.skip("no CUDA headers")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    lib = host_lib(tmp_path, SOURCE, ("-O1", "-Wno-error", "-isystem", cuda, "-I", os.path.join(root, "include")))
    assert lib.launch(9) == 9 and lib.get_last() == 0  # cudaErrorInvalidConfiguration
    lib.set_last(1)  # an error of the caller's own, before a launch that succeeds, stays the caller's
    assert lib.launch(0) == 0 and lib.get_last() == 1
