// Whether the complex128 blocks take one-block circuits of five rotations by an angle, and the largest relative
// error of the entries as their digits hold them.  usage: f64_entry_check angle ..; prints "angle taken error".
// Built against the library by test_f64_range.py.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "block_f64.h"

using namespace qs;

static double half_value(uint16_t h) {
  const int e = (h >> 10) & 31, m = h & 1023;
  const double v = e ? std::ldexp(1.0 + m / 1024.0, e - 15) : std::ldexp(m / 1024.0, -14);
  return h >> 15 ? -v : v;
}

int main(int argc, char** argv) {
  for (int i = 1; i < argc; ++i) {
    std::vector<qs_gate> g(5);
    Block b;
    for (int k = 0; k < 5; ++k) {
      std::memset(&g[k], 0, sizeof(qs_gate));
      g[k].kind = QS_RY;
      g[k].q[0] = b.q[k] = k;
      g[k].param[0] = std::atof(argv[i]);
      b.gate_idx.push_back((size_t)k);
    }
    std::vector<unsigned char> B(kF64B);
    int32_t vs = 0;
    const bool ok = f64_b_operand(g.data(), b, B.data(), &vs);
    double worst = 0;
    const long double c = std::cos(std::atof(argv[i]) / 2), s = std::sin(std::atof(argv[i]) / 2);
    for (int r = 0; r < 32 && ok; ++r)
      for (int col = 0; col < 32; ++col) {
        long double want = 1;   // RY: [c -s; s c] on every bit
        for (int k = 0; k < 5; ++k) {
          const int o = (r >> k) & 1, n = (col >> k) & 1;
          want *= o == n ? c : (o ? s : -s);
        }
        if (want == 0) continue;
        double got = 0;
        const int n = 16 * (r / 8) + 2 * (r % 8), k = 16 * (col / 8) + col % 8;
        for (int j = 0; j < kF64Slices; ++j) {
          uint16_t h;
          std::memcpy(&h, B.data() + j * 8192 + (n >> 3) * 1024 + (k >> 3) * 128 + (n & 7) * 16 + (k & 7) * 2, 2);
          got += std::ldexp(half_value(h), 45 - 9 * j);
        }
        worst = std::max(worst, (double)std::abs((std::ldexp((long double)got, -vs) - want) / want));
      }
    std::printf("%s %d %.3e\n", argv[i], (int)ok, worst);
  }
  return 0;
}
