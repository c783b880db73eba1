"""Rows of a gather tile near the largest map (N_G < 2^31 - 1): a block's 256
threads take the tile's rows in steps, four rows at a time in the staged form,
and a step past 2^31 - 1 must end the loop.  The kernels' own test of a row,
compiled on the host."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2009_10917_gb300", "csrc")

WRAP = r"""
#include "bs_check_pred.h"
/* rows that thread `tid` of 256 takes of [r0, r1), `step` apart; -1: more than `most` */
int w_rows(int32_t r0, int32_t r1, uint32_t tid, uint32_t step, uint32_t *out, int most) {
  int n = 0;
  for (uint32_t r = (uint32_t)r0 + tid; bs_row_before(r, r1); r += step) {
    if (n == most) return -1;
    out[n++] = r;
  }
  return n;
}
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    src, so = d / "wrap.c", d / "wrap.so"
    src.write_text(WRAP)
    subprocess.run(["gcc", "-std=c11", "-O2", "-Wall", "-Werror", "-shared", "-fPIC", "-I", CSRC,
                    str(src), "-o", str(so)], check=True)
    return ctypes.CDLL(str(so)).w_rows


@pytest.mark.parametrize("r0,r1", [(0, 1), (0, 700), (2**31 - 3, 2**31 - 2),
                                   (2**31 - 700, 2**31 - 2), (2**31 - 1026, 2**31 - 2)])
@pytest.mark.parametrize("step", [256, 1024])
def test_every_row_once_and_no_other(rows, r0, r1, step):
    out = (ctypes.c_uint32 * 16)()
    seen = []
    for tid in range(256):
        n = rows(r0, r1, tid, step, out, 16)
        assert n >= 0
        seen += out[:n]
    assert sorted(seen) == [r for r in range(r0, r1) if (r - r0) % step < 256]
