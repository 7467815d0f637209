// Block chains on the CPU: reads gates (qs_gate records) and n, plans the passes, carries out
// every pass's data movement as its descriptor states it (tensor boxes, shared-memory maps) in
// double precision, and prints the largest difference from the gates applied one by one.
// Exits with 1 if a map is not one to one or a tile is not covered exactly once.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "chain.h"

using namespace qs;

static int fail(const char* what) {
  std::printf("%s\n", what);
  return 1;
}

int main(int argc, char** argv) {
  if (argc < 3) return 2;
  const int n = std::atoi(argv[2]);
  std::vector<qs_gate> gates;
  FILE* f = std::fopen(argv[1], "rb");
  if (!f) return 2;
  for (qs_gate g; std::fread(&g, sizeof g, 1, f) == 1;) gates.push_back(g);
  std::fclose(f);
  std::mt19937_64 rng(1);
  std::normal_distribution<double> normal;
  std::vector<cd> psi(1ull << n);
  for (cd& a : psi) a = cd(normal(rng), normal(rng));
  std::vector<cd> ref = psi;
  for (const qs_gate& g : gates) {
    cd m[16];
    int dim = 0;
    gate_matrix(g, m, &dim);
    const uint64_t a = 1ull << g.q[0], b = dim == 4 ? 1ull << g.q[1] : 0;
    for (uint64_t J = 0; J < ref.size(); ++J) {
      if ((J & a) || (J & b)) continue;
      const uint64_t at[4] = {J, dim == 4 ? J | b : J | a, J | a, J | a | b};
      cd v[4], o[4];
      for (int k = 0; k < dim; ++k) v[k] = ref[at[k]];
      for (int i = 0; i < dim; ++i) {
        o[i] = 0;
        for (int k = 0; k < dim; ++k) o[i] += m[i * dim + k] * v[k];
      }
      for (int i = 0; i < dim; ++i) ref[at[i]] = o[i];
    }
  }
  std::vector<ChainPlan> plan;
  plan_chains(gates.data(), gates.size(), n, plan);
  size_t blocks = 0, taken = 0;
  for (const ChainPlan& p : plan) {
    uint64_t mask[kChainMax] = {};
    for (size_t b = 0; b < p.blocks.size(); ++b) {
      for (int q : p.blocks[b].q) mask[b] |= 1ull << q;
      taken += p.blocks[b].gate_idx.size();
    }
    blocks += p.blocks.size();
    ChainPass P;
    if (!chain_pass_desc(n, p.tile, mask, (int)p.blocks.size(), P)) return fail("descriptor");
    if (P.n_nt != n - 12 || kChainLow + P.g1 + P.g2 + P.n_oth != 12) return fail("tile positions");
    std::vector<char> seen(1ull << n, 0);
    for (uint64_t t = 0; t < (1ull << (n - 12)); ++t) {
      uint64_t base = 0;
      for (int j = 0; j < P.n_nt; ++j) base |= ((t >> j) & 1) << P.nt_pos[j];
      std::vector<cd> slot(4096);
      std::vector<uint64_t> phys(4096);
      for (int q = 0; q < (1 << P.n_oth); ++q) {
        uint64_t a = base;
        for (int j = 0; j < P.n_oth; ++j) a |= (uint64_t)((q >> j) & 1) << P.oth_pos[j];
        const uint64_t c1 = (a >> kChainLow) & ((1ull << (P.a1 - kChainLow)) - 1);
        const uint64_t c3 = (a >> (P.a1 + P.g1)) & ((1ull << (P.b - P.a1 - P.g1)) - 1), c4 = a >> P.b;
        for (int e2 = 0; e2 < (1 << P.g2); ++e2)
          for (int e1 = 0; e1 < (1 << P.g1); ++e1)
            for (int e0 = 0; e0 < 16; ++e0) {
              const uint64_t ad = e0 + 16 * c1 + ((uint64_t)e1 << P.a1) + (c3 << (P.a1 + P.g1)) + ((c4 + e2) << P.b);
              uint32_t by = 8u * (e0 + 16 * (e1 + ((e2 + (q << P.g2)) << P.g1)));
              if (P.swizzle) by ^= ((by >> 7) & 7) << 4;
              if (ad >= psi.size() || seen[ad]++) return fail("box");
              slot[by / 8] = psi[ad];
              phys[by / 8] = ad;
            }
      }
      for (size_t b = 0; b < p.blocks.size(); ++b) {
        std::vector<cd> out(4096);
        std::vector<char> rd(4096, 0), wr(4096, 0);
        for (int m = 0; m < 128; ++m) {
          uint32_t r0 = 0, w0 = 0;
          for (int j = 0; j < 7; ++j)
            if ((m >> j) & 1) {
              r0 ^= P.rd[b].row[j];
              w0 ^= P.wr[b].row[j];
            }
          cd x[32];
          for (int c = 0; c < 32; ++c) {
            uint32_t a = r0;
            for (int j = 0; j < 5; ++j)
              if ((c >> j) & 1) a ^= P.rd[b].col[j];
            if ((a & 7) || a >= 32768 || rd[a / 8]++) return fail("read map");
            x[c] = slot[a / 8];
          }
          for (int c = 0; c < 32; ++c) {
            uint32_t a = w0;
            for (int j = 0; j < 5; ++j)
              if ((c >> j) & 1) a ^= P.wr[b].col[j];
            if ((a & 7) || a >= 32768 || wr[a / 8]++) return fail("write map");
            cd y = 0;
            for (int k = 0; k < 32; ++k) y += p.blocks[b].U[c * 32 + k] * x[k];
            out[a / 8] = y;
          }
        }
        slot = out;
      }
      for (int i = 0; i < 4096; ++i) psi[phys[i]] = slot[i];
    }
  }
  if (taken != gates.size()) return fail("gates");
  double err = 0;
  for (size_t i = 0; i < psi.size(); ++i) err = std::max(err, std::abs(psi[i] - ref[i]));
  std::printf("%zu %zu %.3e\n", plan.size(), blocks, err);
  return 0;
}
