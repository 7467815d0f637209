// Compares, for every block of a gate list, the density found from the gates' patterns (block_dense)
// with the one counted in the block's product, and the default method's choice made with either.
// usage: block_density_check gates.bin n.  Prints "blocks dense tiles"; exit 1 on a difference.
// Built against the library by test_block_density.py.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "auto_plan.h"
#include "chain.h"

using namespace qs;

int main(int argc, char** argv) {
  if (argc != 3) return 2;
  FILE* f = std::fopen(argv[1], "rb");
  if (!f) return 2;
  std::vector<qs_gate> g;
  qs_gate one;
  while (std::fread(&one, sizeof(qs_gate), 1, f) == 1) g.push_back(one);
  std::fclose(f);
  const int n = std::atoi(argv[2]);
  std::vector<Block> full, bare;
  plan_blocks(g.data(), g.size(), n, full);
  plan_blocks(g.data(), g.size(), n, bare, /*products=*/false);
  if (full.size() != bare.size()) return 1;
  std::vector<char> dense(bare.size());
  int count = 0;
  for (size_t i = 0; i < bare.size(); ++i) {
    dense[i] = block_dense(g.data(), bare[i]);
    count += dense[i];
    if (full[i].gate_idx != bare[i].gate_idx || (block_nonzeros(full[i]) > 512) != (bool)dense[i]) return 1;
  }
  std::vector<FOp> a, b;
  std::vector<int> va, vb;
  const bool x = auto_all_tiles(g.data(), g.size(), n, full, &a, &va);
  const bool y = auto_all_tiles(g.data(), g.size(), n, bare, dense, &b, &vb);
  std::printf("%zu %d %d\n", bare.size(), count, (int)y);
  return x == y && a.size() == b.size() && va == vb ? 0 : 1;
}
