// Passes of several 5-qubit blocks over one 12-qubit tile of the state.
#pragma once

#include <stdint.h>

#include <vector>

#include "internal.h"

namespace qs {

constexpr int kChainMax = 3;        // blocks in one pass
constexpr int kChainLow = 4;        // physical bits 0..3 are tile bits of every pass: 128-byte runs

// A pass: the tile (12 qubits, bits 0..3 among them) and its blocks in order, each on 5
// of the tile's qubits.  Applying the passes in order equals the circuit.
struct ChainPlan {
  uint64_t tile = 0;
  std::vector<Block> blocks;
};
// Plans gates[0..ngates) (n >= 12); products: also forms every block's matrix.
void plan_chains(const qs_gate* gates, size_t ngates, int n, std::vector<ChainPlan>& out, bool products = true);
// block_nonzeros(b) > 512, mostly from the gates' patterns (b.U is not needed)
bool block_dense(const qs_gate* gates, const Block& b);
// Whether the default method runs the whole circuit as this plan: at least three of its
// blocks are dense (more than 512 of 1024 entries nonzero) for each that is not.
bool chains_dense(const qs_gate* gates, const std::vector<ChainPlan>& plan);
// Whether enough gates make superpositions (neither diagonal nor a permutation) for that to
// be worth planning: a dense block holds at least five of them.
bool chains_likely(const qs_gate* gates, size_t ngates);

// Where the element of row m and column c of a block lies in the 32 KiB tile: byte
// offset = XOR of row[i] over the bits of m and col[i] over the bits of c.
struct ChainMap {
  uint16_t row[7];
  uint16_t col[5];
};

// What the kernel needs to know of a pass (a kernel parameter).
struct ChainPass {
  ChainMap rd[kChainMax], wr[kChainMax];
  int32_t nblk;                       // blocks
  int32_t nload, nstore;              // 32 KiB slots of loaded and of finished tiles
  int32_t n_nt, n_oth;                // positions outside the tile; tile positions outside the box
  uint8_t nt_pos[32];                 // ascending
  uint8_t oth_pos[8];
  // the box: amplitudes [bits 0..3 | run1 = bits a1 .. a1+g1-1 | run2 = bits b .. b+g2-1];
  // the other tile positions are one copy each for all their values
  int32_t a1, g1, b, g2;
  int32_t swizzle;                    // slots hold the box in the 128-byte swizzle
};
// blocks: qubit mask of each (within tile).  false if n or the masks do not fit.
bool chain_pass_desc(int n, uint64_t tile, const uint64_t* blocks, int nblk, ChainPass& P);

// The B operand of one block: three BF16 parts, kChainB bytes.
constexpr int kChainPart = 96 * 32 * 2;
constexpr int kChainB = 3 * kChainPart;
void chain_b_operand(const cd* U, unsigned char* out);

// Which of the kernel's two pipelines takes block b of tile `step - b`.  Alternating over all blocks of all steps,
// also those of tiles that are not there (before the first and after the last): a pipeline that takes
// a tile's last block then takes that of one of the next two tiles, and never reaches a barrier whose phase
// before last is still open.  (Counted over the items alone, the last tile of a pass of two blocks fell to the
// pipeline of the first blocks, which did not know how far the stores were: with slow stores it passed
// their barrier a phase early, wrote over a tile not yet stored and upset the count that the store waits for.)
#ifdef __CUDACC__
__host__ __device__
#endif
inline uint32_t chain_group(uint32_t step, int nblk, int b) {
  return (step * (uint32_t)nblk + (uint32_t)b) & 1u;
}

// once per call, before its passes
qs_status launch_chain_setup();
qs_status launch_chain_pass(State* st, const ChainPass& P, const void* b_dev, int* status_dev);

}  // namespace qs
