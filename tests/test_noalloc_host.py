"""te_spmv_noalloc's host side without a GPU: its source compiled into a small
program whose CUDA runtime calls are fakes that count, fail on request and
record what the call does."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include <cuda_runtime.h>

static int n_sync, n_alloc, n_launched, fail_launch;
static cudaError_t fake_ok() { return cudaSuccess; }
static cudaError_t fake_sync(cudaStream_t) { ++n_sync; return cudaSuccess; }
// called once after every launch or pair of launches; the fail_launch-th fails
static cudaError_t fake_last_error() {
  return ++n_launched == fail_launch ? cudaErrorInvalidConfiguration : cudaSuccess;
}
static cudaError_t fake_host_alloc(void** p, size_t b) {
  ++n_alloc;
  *p = calloc(1, b);
  return cudaSuccess;
}
#define cudaGetDevice(d) (*(d) = 0, fake_ok())
#define cudaGetSymbolAddress(p, s) (*(p) = (void*)&n_sync, fake_ok())
#define cudaFuncSetAttribute(...) fake_ok()
#define cudaStreamSynchronize(s) fake_sync(s)
#define cudaGetLastError() fake_last_error()
#define cudaHostAlloc(p, b, f) fake_host_alloc(p, b)
#define cudaMalloc(p, b) fake_host_alloc((void**)(p), b)
#define cudaMallocHost(p, b) fake_host_alloc((void**)(p), b)
#define cudaHostGetDevicePointer(d, h, f) (*(d) = (h), fake_ok())
#define cudaFreeHost(p) fake_ok()
#include "te_noalloc.cu"
void te::set_last_error(const std::string&) {}
int* te::noalloc_status_words() {
  static int words[NA_DEVICES * NA_SLOTS * 2];
  return words;
}

int main(int argc, char** argv) {
  fail_launch = atoi(argv[1]);
  te_csr A = {};
  A.n = 10;
  A.nnz = 3;
  int64_t rp = 0;
  int32_t ci = 0;
  double v = 0;
  A.row_ptr = &rp;  // (never read: nothing runs)
  A.col_idx = &ci;
  A.values = &v;
  A.where = TE_DEVICE;
  te_precision p = {TE_F64, TE_F64, TE_F64};
  const te_status rc = te_spmv_noalloc(&A, p, &v, &v, nullptr);
  printf("rc %d sync %d alloc %d\n", (int)rc, n_sync, n_alloc);
  return 0;
}
"""


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    from paper_2201_07498_gb300 import _build
    d = tmp_path_factory.mktemp("noalloc")
    src = d / "harness.cu"
    src.write_text(HARNESS)
    exe = str(d / "harness")
    cmd = [_build.nvcc(), str(src), "-o", exe, "-I", _build.CSRC] + _build.NVCC_FLAGS
    cmd[cmd.index("-O3")] = "-O0"
    subprocess.run(cmd, check=True, capture_output=True)

    def run(fail_launch):
        out = subprocess.run([exe, str(fail_launch)], check=True, capture_output=True, text=True)
        w = out.stdout.split()
        return {w[i]: int(w[i + 1]) for i in (0, 2, 4)}
    return run


@pytest.mark.parametrize("fail_launch", [0, 1, 2])
def test_call_ends_after_what_it_queued(call, fail_launch):
    # with a launch that fails as without: the stream is waited for, so that no
    # kernel of this call is left to write its status words into a later call's
    r = call(fail_launch)
    assert (r["rc"] == 0) == (fail_launch == 0)
    assert r["sync"] == 1


def test_call_allocates_nothing(call):
    # neither on the device nor page-locked on the host, not even the first time
    assert call(0)["alloc"] == 0
