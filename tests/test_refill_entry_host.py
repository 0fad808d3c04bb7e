"""Entries of the rigid kernels' refill list keep the record index, the slot and
the sub-warp of a stencil: indices of 32 bits in the instances of one record
kind, of any grid that fits a GPU in the other (2^32 records are a 16-bit
two-slot grid of 17 GB).  The device functions, compiled for the host."""
import subprocess

import pytest

from paper_2508_15522_gb300 import build

SOURCE = r"""
#include <cstdio>
#include "replica_common.cuh"
template <bool WIDE>
int check(long long r) {
  int bad = 0;
  for (int slot : {0, 1, 37, 127, 255})
    for (int sw = 0; sw < 4; ++sw) {
      const int2 e = refill_entry<WIDE>(r, slot, sw);
      bad += refill_record<WIDE>(e) != r || refill_slot(e) != slot || refill_sub<WIDE>(e) != sw;
    }
  return bad;
}
int main() {
  int bad = 0;
  for (long long r : {0LL, 1LL, 4095LL, (1LL << 31) - 1, 1LL << 31, (1LL << 32) - 1}) bad += check<false>(r) + check<true>(r);
  for (long long r : {1LL << 32, (1LL << 32) + 77, 71000000000LL, (1LL << 54) - 1}) bad += check<true>(r);
  printf("bad %d\n", bad);
  return bad != 0;
}
"""


def test_entries_keep_what_they_are_given(tmp_path):
    try:
        cc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "entry.cu", tmp_path / "entry"
    src.write_text(SOURCE)
    subprocess.run([cc, *build.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", build.INCLUDE, "-I", build.CSRC,
                    str(src), "-o", str(exe)], check=True, capture_output=True, text=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True)
    assert res.returncode == 0 and res.stdout.strip() == "bad 0", res.stdout
