"""The integer forms of the FP64 operations (gf_fp64.cuh) never overflow a
signed integer: their remainders are exact modulo 2^64 and have to be formed in
unsigned arithmetic, since a compiler may draw conclusions from a signed
difference's sign.  The host build of test_fp64_ops runs here as a program that
stops at the first signed overflow or undefined shift."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
MAIN = r"""
#include "fp64_shim.cpp"
#include <cstring>
#include <vector>
int main() {
  const int n = 200000;
  std::vector<double> a(n), b(n), o[4];
  for (auto& v : o) v.resize(n);
  std::vector<uint8_t> f(n);
  uint64_t s = 12345;
  auto bits = [&] {
    s = s * 6364136223846793005ull + 1442695040888963407ull;
    uint64_t x = s;
    s = s * 6364136223846793005ull + 1442695040888963407ull;
    return (x & 0xffffffff00000000ull) | (s >> 32);
  };
  for (int k = 0; k < n; ++k) {
    // any bits, then significands in [1, 2) with either sign
    uint64_t x = bits(), y = bits();
    if (k & 1) {
      x = (x & 0x800fffffffffffffull) | 0x3ff0000000000000ull;
      y = (y & 0x800fffffffffffffull) | 0x3ff0000000000000ull;
    }
    std::memcpy(&a[k], &x, 8);
    std::memcpy(&b[k], &y, 8);
  }
  for (double err : {0.0, 0x1p-22})
    fp64_ops(n, a.data(), b.data(), err, o[0].data(), o[1].data(), o[2].data(), o[3].data(),
             f.data());
  return 0;
}
"""


def test_no_signed_overflow(tmp_path):
    src, exe = tmp_path / "main.cpp", tmp_path / "main"
    src.write_text(MAIN)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-ffp-contract=off",
                           "-fsanitize=signed-integer-overflow,shift",
                           "-fsanitize-undefined-trap-on-error",
                           "-I", os.path.join(HERE, "..", "paper_2403_15435_gb300", "csrc"),
                           "-I", HERE, str(src), "-o", str(exe)])
    assert subprocess.run([str(exe)], timeout=120).returncode == 0
