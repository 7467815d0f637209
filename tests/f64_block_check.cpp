// The complex128 block kernel's layout and arithmetic on the CPU.  Reads gates and n, plans the
// 5-qubit blocks and, per block: checks that the tile's shared-memory map is one to one and puts
// every amplitude at its row and column; multiplies random rows by the block's digit slices
// in integers as the kernel does, against the block's gates applied to the row in long double.
// Prints the number of blocks, the largest error over the largest amplitude of the row, and the
// largest digit sum (exact in FP32 up to 2^24).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>

#include "block_f64.h"

using namespace qs;
using cl = std::complex<long double>;

static int fail(const char* what) {
  std::printf("%s\n", what);
  return 1;
}
static double half_value(uint16_t h) {
  const int e = (h >> 10) & 31, m = h & 1023;
  const double v = e ? std::ldexp(1.0 + m / 1024.0, e - 15) : std::ldexp(m / 1024.0, -14);
  return h >> 15 ? -v : v;
}

int main(int argc, char** argv) {
  if (argc < 3) return 2;
  const int n = std::atoi(argv[2]);
  std::vector<qs_gate> gates;
  FILE* f = std::fopen(argv[1], "rb");
  if (!f) return 2;
  for (qs_gate g; std::fread(&g, sizeof g, 1, f) == 1;) gates.push_back(g);
  std::fclose(f);
  std::vector<Block> blocks;
  plan_blocks(gates.data(), gates.size(), n, blocks, false);
  std::mt19937_64 rng(3);
  std::normal_distribution<double> normal;
  std::vector<unsigned char> B(kF64B);
  double worst = 0, big = 0;
  for (const Block& b : blocks) {
    F64Pass P;
    if (!f64_pass_desc(n, b.q, P)) return fail("descriptor");
    if (P.n_nt != n - 12 || kF64Low + P.g1 + P.g2 + P.n_oth != 12) return fail("tile positions");
    uint64_t mask = 0;
    for (int q : b.q) mask |= 1ull << q;
    std::vector<char> seen(1ull << n, 0);
    for (uint64_t t = 0; t < (1ull << (n - 12)); ++t) {
      uint64_t base = 0;
      for (int j = 0; j < P.n_nt; ++j) base |= ((t >> j) & 1) << P.nt_pos[j];
      std::vector<uint64_t> phys(4096);
      for (int q = 0; q < (1 << P.n_oth); ++q) {
        uint64_t a = base;
        for (int j = 0; j < P.n_oth; ++j) a |= (uint64_t)((q >> j) & 1) << P.oth_pos[j];
        const uint64_t c1 = (a >> kF64Low) & ((1ull << (P.a1 - kF64Low)) - 1);
        const uint64_t c3 = (a >> (P.a1 + P.g1)) & ((1ull << (P.b - P.a1 - P.g1)) - 1), c4 = a >> P.b;
        for (int e2 = 0; e2 < (1 << P.g2); ++e2)
          for (int e1 = 0; e1 < (1 << P.g1); ++e1)
            for (int e0 = 0; e0 < 8; ++e0) {
              const uint64_t ad = e0 + 8 * c1 + ((uint64_t)e1 << P.a1) + (c3 << (P.a1 + P.g1)) + ((c4 + e2) << P.b);
              uint32_t at = e0 + 8 * (e1 + ((e2 + (q << P.g2)) << P.g1));
              at ^= (at >> 3) & 7;   // the 128-byte swizzle
              if (ad >= seen.size() || seen[ad]++) return fail("box");
              phys[at] = ad;
            }
      }
      for (int m = 0; m < 128; ++m) {
        uint32_t r = 0;
        for (int j = 0; j < 7; ++j)
          if ((m >> j) & 1) r ^= P.row[j];
        if (phys[r] & mask) return fail("row");
        for (int c = 0; c < 32; ++c) {
          uint32_t a = r;
          uint64_t want = phys[r];
          for (int j = 0; j < 5; ++j)
            if ((c >> j) & 1) {
              a ^= P.col[j];
              want |= 1ull << b.q[j];
            }
          if (a >= 4096 || phys[a] != want) return fail("column");
        }
      }
    }
    int32_t vs = 0;
    if (!f64_b_operand(gates.data(), b, B.data(), &vs)) return fail("operand");
    for (int row = 0; row < 6; ++row) {
      std::complex<double> x[32];
      for (int c = 0; c < 32; ++c) {
        x[c] = {normal(rng), normal(rng)};
        if (row == 1 && c % 3) x[c] *= 1e-12;                          // wide range
        if (row == 2) x[c] = {1.0 - 1e-16 * c, c % 2 ? -1.0 : 1.0};    // digits near their limits
        if (row == 3 && c) x[c] = 0;
        if (row == 4) x[c] *= 1e-150;
      }
      cl y[32];
      for (int c = 0; c < 32; ++c) y[c] = cl(x[c].real(), x[c].imag());
      for (size_t gi : b.gate_idx) {
        cd m[16];
        int dim = 0, at[2] = {0, 0};
        gate_matrix(gates[gi], m, &dim);
        for (int k = 0; k < (dim == 4 ? 2 : 1); ++k)
          for (int i = 0; i < 5; ++i)
            if (b.q[i] == gates[gi].q[k]) at[k] = i;
        const int hi = 1 << at[0], lo = dim == 4 ? 1 << at[1] : 0;
        for (int r = 0; r < 32; ++r) {
          if ((r & hi) || (r & lo)) continue;
          const int idx[4] = {r, dim == 4 ? r | lo : r | hi, r | hi, r | hi | lo};
          cl v[4];
          for (int k = 0; k < dim; ++k) v[k] = y[idx[k]];
          for (int o = 0; o < dim; ++o) {
            cl s = 0;
            for (int k = 0; k < dim; ++k) s += cl(m[o * dim + k].real(), m[o * dim + k].imag()) * v[k];
            y[idx[o]] = s;
          }
        }
      }
      uint32_t top = 0;
      auto word = [](double v) {
        uint64_t w;
        std::memcpy(&w, &v, 8);
        return w;
      };
      for (int c = 0; c < 32; ++c)
        for (double v : {x[c].real(), x[c].imag()}) top = std::max(top, (uint32_t)(word(v) >> 32) & 0x7fffffffu);
      const int E = (int)(top >> 20);
      double dg[kF64Slices][64];
      for (int c = 0; c < 32; ++c)
        for (int p = 0; p < 2; ++p) {
          int64_t X = (int64_t)std::llrint(std::ldexp(p ? x[c].imag() : x[c].real(), 1076 - E));
          for (int i = kF64Slices - 1; i >= 0; --i) {
            const int64_t d = i ? ((X + 256) & 511) - 256 : X;
            X = (X - d) >> 9;
            if (std::llabs(d) > (i ? 256 : 512)) return fail("digit");
            dg[i][16 * (c / 8) + 8 * p + c % 8] = (double)d;
          }
        }
      for (int k = 0; k < 64; ++k) {
        double D[7] = {}, A[7] = {};
        for (int i = 0; i < kF64Slices; ++i)
          for (int j = 0; j < kF64Slices && i + j < 7; ++j)
            for (int c = 0; c < 64; ++c) {
              uint16_t h;
              std::memcpy(&h, B.data() + j * 8192 + (k >> 3) * 1024 + (c >> 3) * 128 + (k & 7) * 16 + (c & 7) * 2, 2);
              D[i + j] += dg[i][c] * half_value(h);
              A[i + j] = std::max(A[i + j], std::abs(D[i + j]));
            }
        for (int s = 0; s < 4; ++s) big = std::max(big, A[s]);
        int64_t Y = (int64_t)std::llrint(D[5] / 128 + D[6] / 65536);
        for (int s = 0; s < 5; ++s) Y += (int64_t)D[s] * (1ll << (38 - 9 * s));
        const double got = std::ldexp((double)Y, E - 1024 - vs);
        const cl w = y[8 * (k >> 4) + ((k & 15) >> 1)];
        const long double want = k & 1 ? w.imag() : w.real();
        worst = std::max(worst, (double)std::abs(got - want) / std::ldexp(1.0, E - 1023));
      }
    }
  }
  std::printf("%zu %.3e %.0f\n", blocks.size(), worst, big);
  return 0;
}
