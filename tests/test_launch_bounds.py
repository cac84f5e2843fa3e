"""Host checks of the integrator's launch rules.

The integrator's grid against the scratch through which particles move
between threads: a block's share is threads entries from blockIdx.x * threads
on, so no grid may have more threads than the scratch has entries, also where
the resident blocks were counted on a larger device than the context's.

The default shape against the SMs: from 128 particles per SM on there is work
for a block on every SM, and a shape of few large blocks must not leave more
than a tenth of the SMs without one."""
import subprocess

from paper_2311_08927_gb300 import build as B

PROGRAM = r"""
#include <cstdio>
#include "kernels.h"
using namespace chad;
int main() {
  const int64_t counts[] = {1, 31, 32, 33, 255, 256, 257, 5003, 19457, 38911, 60013, 311295, 311296,
                            311297, 1000000, 20000000};
  const int devices[] = {1, 18, 76, 148, 152, 160, 304};
  long long checked = 0;
  for (int64_t n : counts)
    for (int here : devices)
      for (int form = 0; form < 5; ++form)
        for (int v = 0; v < kNumVariants; ++v)
          for (int other : devices)
            for (int per_sm = 1; per_sm * kernel_variant(form, v).threads <= 2048; ++per_sm) {
              const int t = kernel_variant(form, v).threads;
              const int64_t cap = migrant_capacity(n, here), need = (n + t - 1) / t;
              const int64_t resident = (int64_t)other * per_sm, b = grid_blocks(n, t, resident, cap);
              ++checked;
              if (b < 1 || b > need || b > resident || b * t > cap) {
                std::printf("n %lld, %d of %d SMs, %d threads: %lld blocks, %lld entries\n", (long long)n,
                            other, here, t, (long long)b, (long long)cap);
                return 1;
              }
              // on the context's own device the scratch never cuts the grid
              if (other == here && b != (need < resident ? need : resident)) {
                std::printf("n %lld, %d SMs, %d threads: cut to %lld\n", (long long)n, here, t, (long long)b);
                return 2;
              }
            }
  std::printf("%lld\n", checked);
  return 0;
}
"""


FILLED = r"""
#include <cstdio>
#include "kernels.h"
using namespace chad;
int main() {
  long long checked = 0;
  for (int sms : {76, 148, 152, 160})
    for (int form = 0; form < 5; ++form)
      for (int64_t n = 128 * (int64_t)sms + 1; n <= 600 * (int64_t)sms; n += 97) {
        const int t = kernel_variant(form, default_variant(form, n, sms)).threads;
        ++checked;
        if (10 * ((n + t - 1) / t) < 9 * (int64_t)sms) {
          std::printf("form %d, n %lld, %d SMs: blocks of %d threads\n", form, (long long)n, sms, t);
          return 1;
        }
      }
  std::printf("%lld\n", checked);
  return 0;
}
"""


def _run(tmp_path, program):
    src, exe = tmp_path / "grid.cu", tmp_path / "grid"
    src.write_text(program)
    subprocess.run([B.nvcc(), *B.ARCH, *B.NVCC_FLAGS, "-o", str(exe), str(src)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 10_000


def test_no_grid_exceeds_the_migration_scratch(tmp_path):
    _run(tmp_path, PROGRAM)


def test_default_shape_puts_work_on_the_sms(tmp_path):
    _run(tmp_path, FILLED)
