"""Grid width of the adjoint and Pauli-sum passes: the few candidates against every width, on the host."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <chrono>
#include <cstdio>
#include "row_grid.h"

static long long every_width(long long n, long long batch, long long slots) {
  const long long most = std::max<long long>(1, std::min(n, (4 * slots + batch - 1) / batch));
  long long best = 1, best_cost = 0;
  for (long long gx = 1; gx <= most; ++gx) {
    const long long cost = ((n + gx - 1) / gx + 1) * ((gx * batch + slots - 1) / slots);
    if (gx == 1 || cost < best_cost) best = gx, best_cost = cost;
  }
  return best;
}

int main() {
  const long long batches[] = {1, 2, 3, 5, 7, 16, 63, 64, 100, 151, 152, 153, 300, 607, 608, 609, 1000, 2432, 2433, 65535, 1 << 20};
  const long long slots[] = {1, 2, 152, 304, 456, 608, 912};
  for (int lg = 0; lg <= 18; ++lg)
    for (long long s : slots)
      for (long long b : batches)
        for (long long n : {1ll << lg, (1ll << lg) + 1, 3ll << lg})
          if (tnq::best_row_grid(n, b, s) != every_width(n, b, s)) {
            std::printf("%lld tiles, batch %lld, %lld slots: %lld, not %lld\n", n, b, s, tnq::best_row_grid(n, b, s),
                        every_width(n, b, s));
            return 1;
          }
  const auto t0 = std::chrono::steady_clock::now();
  long long sum = 0;
  for (int i = 0; i < 10000; ++i) sum += tnq::best_row_grid((1ll << 18) + i, 1, 608);
  const double us = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count() * 1e6 / 10000;
  std::printf("%.3f us per call (%lld)\n", us, sum);
  return us < 1.0 ? 0 : 2;
}
"""


def test_candidates_give_the_best_width_in_no_time(tmp_path):
    src, exe = tmp_path / "row_grid.cpp", tmp_path / "row_grid"
    src.write_text(PROGRAM)
    csrc = os.path.join(ROOT, "paper_2108_06831_gb300", "csrc")
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", csrc, str(src), "-o", str(exe)], check=True)
    done = subprocess.run([str(exe)], capture_output=True, text=True)
    assert done.returncode == 0, done.stdout
    print(done.stdout)
