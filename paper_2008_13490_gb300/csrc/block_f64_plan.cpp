// Host side of the complex128 blocks: tile layout and the digit slices of a block's matrix.
#include <algorithm>
#include <cmath>
#include <cstring>

#include "block_f64.h"

namespace qs {

// Shared memory holds the tile as the tensor box lands: local bits 0..2 = physical bits 0..2,
// then the two longest runs of neighbouring tile positions (at most 8 long), then the rest (a
// copy each for all their values).  The 128-byte swizzle adds local bits 3..5 to the bank bits
// 0..2 of the 16-byte index; 16-byte accesses go 8 lanes at a time, so the rows that span the
// bank bits go to lane bits 0..2.
bool f64_pass_desc(int n, const int* q, F64Pass& P) {
  std::memset(&P, 0, sizeof(P));
  if (n < 12 || n > 36) return false;
  uint64_t block = 0;
  for (int i = 0; i < 5; ++i) {
    if (q[i] < 0 || q[i] >= n || (i && q[i] <= q[i - 1])) return false;
    block |= 1ull << q[i];
  }
  uint64_t tile = block;
  for (int p = 0, k = 0; k < 7; ++p)
    if (!((block >> p) & 1)) {
      tile |= 1ull << p;
      ++k;
    }
  std::pair<int, int> runs[9];
  int nr = 0;
  for (int p = kF64Low; p < n; ++p) {
    if (!((tile >> p) & 1)) {
      P.nt_pos[P.n_nt++] = (uint8_t)p;
      continue;
    }
    if (nr && runs[nr - 1].first + runs[nr - 1].second == p && runs[nr - 1].second < 8) ++runs[nr - 1].second;
    else runs[nr++] = {p, 1};
  }
  int r1 = 0, r2 = -1;
  for (int i = 1; i < nr; ++i)
    if (runs[i].second > runs[r1].second) r1 = i;
  for (int i = 0; i < nr; ++i)
    if (i != r1 && (r2 < 0 || runs[i].second > runs[r2].second)) r2 = i;
  if (r2 >= 0 && r2 < r1) std::swap(r1, r2);
  P.a1 = runs[r1].first;
  P.g1 = runs[r1].second;
  P.b = r2 >= 0 ? runs[r2].first : P.a1 + P.g1;
  P.g2 = r2 >= 0 ? runs[r2].second : 0;
  int local[12], nl = 0;
  for (int p = 0; p < kF64Low; ++p) local[nl++] = p;
  for (int i = 0; i < P.g1; ++i) local[nl++] = P.a1 + i;
  for (int i = 0; i < P.g2; ++i) local[nl++] = P.b + i;
  for (int r = 0; r < nr; ++r) {
    if (r == r1 || r == r2) continue;
    for (int i = 0; i < runs[r].second; ++i) {
      P.oth_pos[P.n_oth++] = (uint8_t)(runs[r].first + i);
      local[nl++] = runs[r].first + i;
    }
  }
  uint16_t box[12];
  for (int j = 0; j < 12; ++j) box[j] = (uint16_t)((1u << j) ^ (j >= 3 && j <= 5 ? 1u << (j - 3) : 0u));
  int nc = 0, rows[7], k = 0, rest[7], nrest = 0;
  uint32_t basis[3] = {0, 0, 0};
  for (int p = 0; p < n; ++p)
    for (int j = 0; j < 12; ++j)
      if (local[j] == p && ((block >> p) & 1)) P.col[nc++] = box[j];   // ascending positions
  for (int j = 0; j < 12; ++j) {
    if ((block >> local[j]) & 1) continue;
    uint32_t x = box[j] & 7u;
    bool fresh = false;
    for (int b = 2; b >= 0 && !fresh; --b)
      if ((x >> b) & 1) {
        if (!basis[b]) {
          basis[b] = x;
          fresh = true;
        } else {
          x ^= basis[b];
        }
      }
    if (fresh) rows[k++] = j;
    else rest[nrest++] = j;
  }
  for (int i = 0; i < nrest; ++i) rows[k++] = rest[i];
  for (int i = 0; i < 7; ++i) P.row[i] = box[rows[i]];
  return true;
}

namespace {

// FP16 bits of an integer of magnitude at most 2048
uint16_t half_of(int v) {
  if (v == 0) return 0;
  const uint32_t a = (uint32_t)(v < 0 ? -v : v);
  const int e = 31 - __builtin_clz(a);   // a = 2^e (1 + f)
  return (uint16_t)((v < 0 ? 0x8000u : 0u) | (uint32_t)(e + 15) << 10 | ((a << (10 - e > 0 ? 10 - e : 0)) & 0x3ffu));
}

}  // namespace

namespace {

// A 32x32 complex matrix in pairs of doubles (value = h + l), as planes: [row][column].
struct PairMatrix {
  double rh[32][32], rl[32][32], ih[32][32], il[32][32];
};

// (h, l) += g (xh + xl)
inline void mul_add(double g, double xh, double xl, double& h, double& l) {
  const double p = g * xh, e = std::fma(g, xh, -p);   // the product and its error
  const double s = h + p, z = s - h;                  // the sum and its error (Knuth)
  l += ((h - (s - z)) + (p - z)) + (e + g * xl);
  h = s;
}

// rows idx[0..dim) <- m (dim x dim) rows idx
template <int DIM>
void apply_rows(PairMatrix& U, const cd* m, const int* idx) {
  double rh[DIM][32], rl[DIM][32], ih[DIM][32], il[DIM][32];
  for (int o = 0; o < DIM; ++o)
    for (int c = 0; c < 32; ++c) {
      double a = 0, b = 0, p = 0, q = 0;
      for (int k = 0; k < DIM; ++k) {
        const int r = idx[k];
        const double gr = m[o * DIM + k].real(), gi = m[o * DIM + k].imag();
        mul_add(gr, U.rh[r][c], U.rl[r][c], a, b);
        mul_add(-gi, U.ih[r][c], U.il[r][c], a, b);
        mul_add(gr, U.ih[r][c], U.il[r][c], p, q);
        mul_add(gi, U.rh[r][c], U.rl[r][c], p, q);
      }
      rh[o][c] = a + b;
      rl[o][c] = b - (rh[o][c] - a);
      ih[o][c] = p + q;
      il[o][c] = q - (ih[o][c] - p);
    }
  for (int o = 0; o < DIM; ++o) {
    std::memcpy(U.rh[idx[o]], rh[o], sizeof(rh[o]));
    std::memcpy(U.rl[idx[o]], rl[o], sizeof(rl[o]));
    std::memcpy(U.ih[idx[o]], ih[o], sizeof(ih[o]));
    std::memcpy(U.il[idx[o]], il[o], sizeof(il[o]));
  }
}

void pair_product(const qs_gate* gates, const Block& b, PairMatrix& U) {
  std::memset(&U, 0, sizeof(U));
  for (int i = 0; i < 32; ++i) U.rh[i][i] = 1.0;
  for (size_t gi : b.gate_idx) {
    const qs_gate& g = gates[gi];
    cd m[16];
    int dim = 0, at[2] = {0, 0};
    gate_matrix(g, m, &dim);
    for (int k = 0; k < (dim == 4 ? 2 : 1); ++k)
      for (int i = 0; i < 5; ++i)
        if (b.q[i] == g.q[k]) at[k] = i;
    const int hi = 1 << at[0], lo = dim == 4 ? 1 << at[1] : 0;
    bool diag = true;
    for (int o = 0; o < dim; ++o)
      for (int k = 0; k < dim; ++k) diag = diag && (o == k || m[o * dim + k] == cd(0));
    for (int r = 0; r < 32; ++r) {
      if ((r & hi) || (r & lo)) continue;
      const int idx[4] = {r, dim == 4 ? r | lo : r | hi, r | hi, r | hi | lo};
      if (diag) {
        for (int k = 0; k < dim; ++k)
          if (m[k * dim + k] != cd(1)) apply_rows<1>(U, &m[k * dim + k], idx + k);
      } else if (dim == 2) {
        apply_rows<2>(U, m, idx);
      } else {
        apply_rows<4>(U, m, idx);
      }
    }
  }
}

}  // namespace

// Entry u = V 2^-vs with |V| <= 2^55: five balanced digits of 9 bits (|d| <= 256) from the
// bottom and a top one (|d| <= 1024), FP16 integers.  Row n = 16 q + 2 r + part is the real
// (part 0) or imaginary part of output 8 q + r; K = 16 j + k: the real parts of columns
// 8 j .. 8 j + 7, then the imaginary ones.  K-major core matrices, no swizzle.
bool f64_b_operand(const qs_gate* gates, const Block& b, unsigned char* out, int32_t* vs, cd* matrix) {
  PairMatrix U;
  pair_product(gates, b, U);
  for (int k = 0; matrix && k < 32 * 32; ++k)
    matrix[k] = cd(U.rh[k >> 5][k & 31] + U.rl[k >> 5][k & 31], U.ih[k >> 5][k & 31] + U.il[k >> 5][k & 31]);
  double big = 0;
  for (int r = 0; r < 32; ++r)
    for (int c = 0; c < 32; ++c) {
      if (!std::isfinite(U.rh[r][c]) || !std::isfinite(U.ih[r][c])) return false;
      big = std::max(big, std::max(std::abs(U.rh[r][c]), std::abs(U.ih[r][c])));
    }
  if (!(big > std::ldexp(1.0, -kF64MaxEntryExp) && big < std::ldexp(1.0, kF64MaxEntryExp))) return false;
  // an entry far below the largest would keep few digits of its own (kF64MinEntry)
  for (int r = 0; r < 32; ++r)
    for (int c = 0; c < 32; ++c) {
      const double a = std::max(std::abs(U.rh[r][c]), std::abs(U.ih[r][c]));
      if (a != 0 && a < big * kF64MinEntry) return false;
    }
  int e = 0;
  const double f = std::frexp(big, &e);   // big = f 2^e, 1/2 <= f < 1
  *vs = 55 - (f == 0.5 ? e - 1 : e);
  const double scale = std::ldexp(1.0, *vs);
  for (int n = 0; n < 64; ++n) {
    const int r = 8 * (n >> 4) + ((n & 15) >> 1), part = n & 1;
    double sum[kF64Slices] = {};   // of |digit| over the row, top first
    double l1 = 0;
    for (int k = 0; k < 64; ++k) {
      const int j = k >> 4, im = (k & 15) >> 3, c = 8 * j + (k & 7);
      const bool real = (part == 0) == (im == 0);   // [Re -Im; Im Re]
      const double xh = (real ? U.rh : U.ih)[r][c] * scale, xl = (real ? U.rl : U.il)[r][c] * scale;
      int64_t V = (int64_t)std::llrint(xh);
      V += (int64_t)std::llrint((xh - (double)V) + xl);
      if (part == 0 && im) V = -V;
      l1 += std::abs((double)V);
      for (int s = kF64Slices - 1; s >= 0; --s) {
        int d;
        if (s > 0) {
          d = (int)((V + 256) & 511) - 256;
          V = (V - d) >> 9;
        } else {
          d = (int)V;
        }
        sum[s] += std::abs((double)d);
        const uint16_t h = half_of(d);
        const int off = s * 8192 + (n >> 3) * 1024 + (k >> 3) * 128 + (n & 7) * 16 + (k & 7) * 2;
        std::memcpy(out + off, &h, 2);
      }
    }
    // the sums of order s take digits of amplitudes |d| <= 512 (top) or 256; from order 4 on a
    // unit is below 2^-56 of the row's largest amplitude, and a rounded sum does no harm
    for (int s = 0; s < 4; ++s) {
      double bound = 512 * sum[s];
      for (int j = 0; j < s; ++j) bound += 256 * sum[j];
      if (bound > 16777216.0) return false;
    }
    if (l1 > std::ldexp(1.0, 60)) return false;   // the 64-bit sums of the epilogue
  }
  return true;
}

}  // namespace qs
