// Dense 5-qubit blocks of complex128 states on the tensor cores, in exact integer slices.
#pragma once

#include <stdint.h>

#include "internal.h"

namespace qs {

constexpr int kF64Low = 3;      // physical bits 0..2 are tile bits of every pass: 128-byte runs
constexpr int kF64Slices = 6;   // digits of an amplitude and of a matrix entry
constexpr int kF64B = kF64Slices * 64 * 64 * 2;
// The kernel moves a result into place by an addition to its exponent field: biased exponent
// 1023 + k of the integer sum (|sum| < 2^63, so k <= 62) plus E - 1024 - vs, E the biased exponent of
// the row's largest part.  With E and the block's largest entry within these bounds (vs = 55 minus that
// entry's exponent, -5 to 114) the field stays within 13 .. 2016.
constexpr uint32_t kF64MinExp = 128, kF64MaxExp = 1950;   // E; rows below are zero, above (and NaN) not a number
constexpr int kF64MaxEntryExp = 60;                       // largest entry within 2^-60 .. 2^60

// A pass of one block over the state (a kernel parameter).  The tile: the block's 5 qubits
// (columns c) and the 7 lowest others (rows m); 64 KiB in shared memory, element (m, c) at the
// XOR of row[i] over the bits of m and col[i] over the bits of c, in units of 16 bytes.
struct F64Pass {
  uint16_t row[7];
  uint16_t col[5];
  int32_t n_nt, n_oth;                // positions outside the tile; tile positions outside the box
  uint8_t nt_pos[32];                 // ascending
  uint8_t oth_pos[8];
  int32_t a1, g1, b, g2;              // the box (chain.h), on top of bits 0..2
  int32_t vs;                         // matrix entries are integers times 2^-vs
};
bool f64_pass_desc(int n, const int* q, F64Pass& P);
// The B operand of a block, kF64B bytes, and its scale: the product of its gates, formed in
// pairs of doubles (about 100 bits), so that one rounding per entry is left where the product
// in double would round once per gate.  false if a sum of digit products that has to be exact
// could exceed 2^24 (FP32 accumulation), or the largest entry is out of bounds (above) or not finite.
bool f64_b_operand(const qs_gate* gates, const Block& b, unsigned char* out, int32_t* vs);

qs_status launch_f64_setup();
qs_status launch_f64_pass(State* st, const F64Pass& P, const void* b_dev, int* status_dev);

}  // namespace qs
