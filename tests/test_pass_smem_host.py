"""The basis passes' shared memory: a pass without digits keeps two stages, so that
copies run beside the sums, up to 54 binary64 columns and the pass vector; the
buffers of the digits and of the small coefficients are not taken from it.  The
source's own plan, compiled for the host."""
import os
import subprocess

import pytest

HARNESS = r"""
#include <cstdio>
#include "te_reorth.cu"
using namespace te;
int main() {
  const size_t cap = 227 * 1024;  // the most a CTA may have on this GPU
  const size_t stage = 55 * TILE_R * sizeof(double);
  for (int mode : {MODE_DOT, MODE_AXPY_DOT, MODE_AXPY_STORE, MODE_DCGS_DOT, MODE_DCGS_UPDATE})
    for (int digits = 0; digits < 2; ++digits) {
      const size_t fixed = smem_plan(mode, digits != 0, 0, 0).total + 128;
      const size_t region = (cap - fixed) / 128 * 128;
      const SmemPlan L = smem_plan(mode, digits != 0, region, 0);
      printf("%d %d %d %d\n", mode, digits, (int)(region / stage), (int)(L.total <= cap));
    }
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    from paper_2201_07498_gb300 import _build
    d = tmp_path_factory.mktemp("smem")
    (d / "harness.cu").write_text(HARNESS)
    flags = [f if f != "-O3" else "-O0" for f in _build.NVCC_FLAGS]
    subprocess.run([_build.nvcc(), str(d / "harness.cu"), "-o", str(d / "harness"), "-I",
                    _build.CSRC] + flags, check=True, capture_output=True)
    out = subprocess.run([str(d / "harness")], check=True, capture_output=True, text=True).stdout
    return [tuple(map(int, line.split())) for line in out.splitlines()]


def test_two_stages_without_digits(plans):
    assert len(plans) == 10
    for mode, digits, stages, fits in plans:
        assert fits
        assert stages >= (1 if digits else 2), (mode, digits, stages)
