"""The normalised moments' arithmetic, compiled for the host: the float32 nearest to float64's
quotient, and to its root."""
import os
import subprocess

from paper_2508_03911_gb300 import build

SOURCE = """
#include "quotient.h"
#include <cstdio>
#include <cstdint>
int main() {
  long bad = 0;
  auto check = [&](float a, float b) {
    const double r = double(a) / double(b);
    bad += hv::root_of_quotient(a, b) != float(sqrt(r > 0.0 ? r : 0.0));
    if (r > 1e-37 && r < 3e38) bad += hv::quotient(a, b) != float(r);
  };
  // pairs whose root lies so near the middle of two float32 that a step of the root by
  // float32 products picks the other one
  check(0x1.1cc67ep+25f, 0x1.15c1c2p+23f);
  check(0x1.8a1ab8p+64f, 0x1.cf0cbcp+23f);
  check(0x1.9a8fa6p+29f, 0x1.77d18p+23f);
  check(0x1.c7dd3ep+57f, 0x1.d5a646p+23f);
  check(0x1.e7916ap+68f, 0x1.ea4372p+23f);
  check(0x1.236958p+59f, 0x1.7331aep+23f);
  check(0x1.640df4p+45f, 0x1.d5a0eap+23f);
  // exact squares of 25 bits, halfway between two float32
  for (uint32_t m = (1u << 24) + 1; m < (1u << 25); m += 99998) check(float(double(m) * m), 1.f), check(float(m), float(m) / 4);
  for (float x : {0.f, 1e-44f, 1e-30f, 1e-25f, 1.f, 1e25f, 1e38f})
    for (float y : {1e-44f, 1e-30f, 1e-25f, 1.f, 1e25f, 1e38f}) check(x, y);
  uint64_t u = 88172645463325252ull;
  for (int i = 0; i < 3000000; ++i) {
    u ^= u << 13, u ^= u >> 7, u ^= u << 17;
    check(std::ldexp(float((u & 0xffffff) | 0x800000), int(u >> 58)), float(((u >> 24) & 0xffffff) | 0x800000));
  }
  std::printf("%ld\\n", bad);
}
"""


def test_normalised_moments_are_float64s(tmp_path):
    src, exe = tmp_path / "q.cpp", tmp_path / "q"
    src.write_text(SOURCE)
    cuda = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", f"-I{build.CSRC}", f"-I{cuda}", str(src), "-o", str(exe)],
                   check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split() == ["0"]
