"""The 32-bit words of the SGD stream at the largest sizes that the load accepts
(no GPU needed): place words, steps and replica offsets, in the arithmetic that
the kernels use, compiled for the host."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1410_8043_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "internal.h"
using namespace esspt;

int main() {
  // entries of users with one each (places per entry: per_step), up to the most
  // that a minibatch can hold; the groups of a warp side by side
  for (int gpw = 1; gpw <= 8; gpw *= 2)
    for (int per_step = 1; per_step <= 2; ++per_step) {
      const StreamGeometry g{gpw, per_step};
      for (int64_t step : {int64_t(0), int64_t(1) << 20, INT64_C(2147483646) / gpw, INT64_C(2147483646) / gpw + (1 << 22)})
        for (int grp = 0; grp < gpw; grp += gpw > 1 ? gpw - 1 : 1)
          for (int k = 0; k < 96; k += 5) {
            const int64_t want = ((step + k / per_step) * gpw + grp) * per_step + k % per_step;
            const int64_t at = record_place(g, place_word(g, step, grp), k);
            if (at != want || y_word(g, at) != want / per_step * 2 * per_step + want % per_step) {
              std::printf("gpw %d per_step %d step %lld: %lld, not %lld\n", gpw, per_step, (long long)step, (long long)at,
                          (long long)want);
              return 1;
            }
          }
    }
  // one step per entry (one group per warp) of nearly 2^31 entries, each warp's
  // first step aligned
  if (INT64_C(2147483646) + kStepAlign * INT64_C(152) * 7 * 4 > kMaxSteps) return 2;
  // item replicas held to 2^31 float4 in 32-byte sectors: the padded offset is a word
  for (int K = 4; K <= 512; K += 4) {
    const int64_t rows = (INT64_C(2147483647) - 1) / ((K + 7) / 8 * 2);
    if (rows * dR_stride4(K) >= (int64_t)kNoRecord || dR_stride4(K) * 4 < K || dR_stride4(K) % 2) return 3;
  }
  return 0;
}
"""


def test_words_at_the_largest_sizes(tmp_path):
    from paper_1410_8043_gb300 import build

    src, exe = tmp_path / "limits.cpp", tmp_path / "limits"
    src.write_text(PROGRAM)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc())))
    subprocess.check_call(["g++", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-I",
                           os.path.join(cuda, "include"), str(src), "-o", str(exe)])
    done = subprocess.run([str(exe)], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout


def test_kernels_use_that_arithmetic():
    """No other place arithmetic, and no signed step, in the sources."""
    fill = open(os.path.join(CSRC, "stream_layout.cu")).read()
    assert fill.count("record_place(") == 3 and "int32_t* total" not in fill
    kernel = open(os.path.join(CSRC, "mf_kernels.cu")).read()
    assert "uint32_t s0 = 0, s1 = 0;" in kernel and "int32_t s = s0" not in kernel.replace("uint32_t s = s0", "")
