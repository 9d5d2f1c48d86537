"""CPU check of the move that puts BF16 rows staged one element to the right in
place: the functions the kernels call, compiled for the host, for every filter
size.  A row's words depend on that row alone (the next row belongs to another
warp), and every column in use moves by one."""
import os
import subprocess

import pytest

from paper_2504_01266_gb300 import build

SOURCE = r"""
#include <cstdio>
#include <vector>
#include "dw_kernels.cuh"
using namespace giga;

static int check(int K) {
  const int R = (K - 1) / 2, RP = geo_rp(K, 2), pitch = geo_pitch(K, 2, true);
  const int words = shift_words(R, RP), used = kTileW + RP + R;
  if (words > pitch / 2) return 1;  // writes stay in the row
  // two rows; the second differs between the runs
  std::vector<uint32_t> a(pitch), b(pitch);
  for (int k = 0; k < pitch; ++k) a[k] = b[k] = (uint32_t)(2 * k) | ((uint32_t)(2 * k + 1) << 16);
  for (int k = pitch / 2; k < pitch; ++k) b[k] = ~a[k];
  for (int k = 0; k < words; ++k) {
    const uint32_t v = shifted_word(a.data(), k, pitch / 2);
    if (v != shifted_word(b.data(), k, pitch / 2)) return 2;
    if (2 * k < used && (v & 0xffffu) != (uint32_t)(2 * k + 1)) return 3;
    if (2 * k + 1 < used && (v >> 16) != (uint32_t)(2 * k + 2)) return 4;
  }
  return 2 * words >= used ? 0 : 5;
}

int main() {
  for (int K = 1; K <= 31; K += 2)
    if (int e = check(K)) {
      std::printf("K = %d: check %d\n", K, e);
      return 1;
    }
  return 0;
}
"""


def test_shifted_rows_read_their_own_words_only(tmp_path):
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "shift.cu", tmp_path / "shift"
    src.write_text(SOURCE)
    r = subprocess.run([nvcc, *build.ARCH, *build.NVCC_FLAGS, str(src), "-o", str(exe)],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60,
                       env={**os.environ, "CUDA_VISIBLE_DEVICES": ""})
    assert r.returncode == 0, r.stdout
