// Which pipeline of the chain kernel takes block b of tile `step - b`: "step nblk b pipeline" per line.
// Built against the library's headers by test_chain_order.py.
#include <cstdio>

#include "chain.h"

int main() {
  for (int nblk = 1; nblk <= qs::kChainMax; ++nblk)
    for (uint32_t step = 0; step < 64; ++step)
      for (int b = 0; b < nblk; ++b) std::printf("%u %d %d %u\n", step, nblk, b, qs::chain_group(step, nblk, b));
  return 0;
}
