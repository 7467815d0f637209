// The complex128 block kernel's scale on the CPU: for one-gate blocks with entries of a given size, whether
// f64_b_operand takes the block, and the smallest and largest exponent field that the kernel's addition
// can give for it.  usage: f64_scale_check size ..; prints "size taken lowest highest" per line.
// Built against the library by test_f64_range.py.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "block_f64.h"

using namespace qs;

int main(int argc, char** argv) {
  for (int i = 1; i < argc; ++i) {
    const double a = std::atof(argv[i]);
    qs_gate g;
    std::memset(&g, 0, sizeof g);
    g.kind = QS_MAT1;
    g.q[0] = 2;
    for (int k = 0; k < 4; ++k) g.m[2 * k] = k == 3 ? -a : a;
    Block b;
    for (int k = 0; k < 5; ++k) b.q[k] = k;
    b.gate_idx.push_back(0);
    std::vector<unsigned char> B(kF64B);
    int32_t vs = 0;
    const bool ok = f64_b_operand(&g, b, B.data(), &vs);
    const int lo = 1023 + 0 + (int)kF64MinExp - 1024 - vs, hi = 1023 + 62 + (int)kF64MaxExp - 1024 - vs;
    std::printf("%s %d %d %d\n", argv[i], (int)ok, lo, hi);
  }
  return 0;
}
