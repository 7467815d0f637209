// Dense 5-qubit blocks of complex128 states on the tensor cores, in exact integer slices.
#pragma once

#include <stdint.h>

#include "internal.h"

namespace qs {

constexpr int kF64Low = 3;      // physical bits 0..2 are tile bits of every pass: 128-byte runs
constexpr int kF64Slices = 6;   // digits of an amplitude and of a matrix entry
constexpr int kF64B = kF64Slices * 64 * 64 * 2;
constexpr int kF64Op = kF64B + 32 * 32 * 16;   // a block in device memory: its B operand, then its matrix
// The kernel moves a result into place by an addition to its exponent field: biased exponent
// 1023 + k of the integer sum (|sum| < 2^63, so k <= 62) plus E - 1024 - vs, E the biased exponent of
// the row's largest part.  With E and the block's largest entry within these bounds (vs = 55 minus that
// entry's exponent, -5 to 114) the field stays within 13 .. 2016.
constexpr uint32_t kF64MinExp = 128, kF64MaxExp = 1950;   // E
// Rows outside these bounds (infinities and NaN among them) and rows with an amplitude, not zero, of less than
// 2^-kF64Spread of the largest are multiplied in FP64 arithmetic: on the largest's exponent an amplitude of
// 2^-k of it keeps 54 - k bits.  (Amplitudes below 2^-1042 count as zero.)  To look for them takes 2 % of a pass
// (25 qubits, 81 passes: 29.3 -> 30.1 ms); a pass with such rows in every tile takes 13.1 ms in place
// of 1.1, where its 48 gates take 10.7 one by one.  So the bound lies where states of layered circuits do
// not come: at 14 the same circuit met such rows in its first passes and took 36.3 ms in place of 32.7.
constexpr uint32_t kF64Spread = 20;
constexpr int kF64MaxEntryExp = 60;                       // largest entry within 2^-60 .. 2^60
// Entries are integers on the scale of the block's largest: one of 2^-k of it keeps 55 - k bits.  The
// rotations by small angles of a Trotter step make entries of their own size on the way to rare
// outcomes, so a block with an entry (that is not zero) below this runs on tile passes.
constexpr double kF64MinEntry = 1.0 / (1 << 20);

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
// could exceed 2^24 (FP32 accumulation), or the largest entry is out of bounds (above) or not finite, or
// another is too far below it.
// matrix (32x32, row-major; may be null): the product rounded to FP64.
bool f64_b_operand(const qs_gate* gates, const Block& b, unsigned char* out, int32_t* vs, cd* matrix = nullptr);

qs_status launch_f64_setup();
// b_dev: kF64Op bytes; status: page-locked host memory
qs_status launch_f64_pass(State* st, const F64Pass& P, const void* b_dev, int* status);

}  // namespace qs
