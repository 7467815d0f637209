// Writes how many fused ops a circuit becomes, and how many of them are one-qubit ops with real matrices
// and diagonals: build_fused_ops, then the merge of one-qubit ops that lists for one CTA get.
// usage: fold_rule_dump gates.bin n relabel
// Built against the library by test_fold_rule.py.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "fuse_merge.h"
#include "internal.h"

using namespace qs;

int main(int argc, char** argv) {
  if (argc != 4) return 2;
  FILE* f = std::fopen(argv[1], "rb");
  if (!f) return 2;
  std::vector<qs_gate> g;
  qs_gate one;
  while (std::fread(&one, sizeof(qs_gate), 1, f) == 1) g.push_back(one);
  std::fclose(f);
  const int n = std::atoi(argv[2]);
  const bool relabel = std::atoi(argv[3]) != 0;
  std::vector<FOp> ops;
  std::vector<int> vmap;
  build_fused_ops(g.data(), g.size(), n, ops, vmap, true, relabel);
  if (!relabel) merge_one_qubit_ops(ops, n, nullptr);
  int real = 0, diag = 0;
  for (const FOp& o : ops) {
    diag += o.type == F_D;
    if (o.type != F_G1) continue;
    bool r = true;
    for (int k = 0; k < 4; ++k) r = r && o.m0[k].imag() == 0.0;
    real += r;
  }
  std::printf("%zu %d %d\n", ops.size(), real, diag);
  return 0;
}
