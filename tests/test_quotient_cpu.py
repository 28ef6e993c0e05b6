"""The corrected reciprocal of the quantiser (csrc/common.cuh, quot_window): for every pair of a bf16 weight's and
an fp32 scale's mantissa the two fused steps give the IEEE quotient. Exponents only shift both sides inside the
window. The same operations on the host, 2^7 x 2^23 pairs one by one (about a second on eight cores)."""
import subprocess

PROGRAM = r"""
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <thread>
#include <vector>
int main() {
  std::atomic<long> bad{0}, uncorrected{0};
  const uint32_t nt = std::max(1u, std::thread::hardware_concurrency());
  std::vector<std::thread> threads;
  for (uint32_t t = 0; t < nt; ++t)
    threads.emplace_back([&, t] {
      long b = 0, c = 0;
      for (uint32_t m = t; m < (1u << 23); m += nt) {
        const uint32_t bits = 0x3f800000u | m;
        float s;
        std::memcpy(&s, &bits, 4);
        const float r = 1.0f / s;
        for (int a = 128; a < 256; ++a) {
          const float w = (float)a, v0 = w * r;
          const float v = std::fma(std::fma(-v0, s, w), r, v0);
          b += v != w / s;
          c += v0 != w / s;
        }
      }
      bad += b;
      uncorrected += c;
    });
  for (auto& th : threads) th.join();
  std::printf("%ld %d\n", bad.load(), uncorrected.load() > 0);
}
"""


def test_corrected_reciprocal_is_the_quotient_for_every_mantissa_pair(tmp_path):
    src, exe = tmp_path / "quotient.cpp", tmp_path / "quotient"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-pthread", str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=300)
    assert r.stdout.split() == ["0", "1"], r.stdout
