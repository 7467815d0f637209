// Host side of the block chains: which gates go into which pass and block, and how a
// pass lays its tile out in shared memory.
#include <algorithm>
#include <cstring>

#include "chain.h"
#include "host_par.h"

namespace qs {

namespace {

int popc(uint64_t x) { return __builtin_popcountll(x); }

uint64_t mask_of(const qs_gate& g) {
  uint64_t m = 1ull << g.q[0];
  if (gate_is_two_qubit(g.kind)) m |= 1ull << g.q[1];
  return m;
}

// Number of gates that a set S takes in order: those on qubits of S that no skipped
// earlier gate on a shared qubit precedes.
int takes(const std::vector<uint64_t>& m, uint64_t S) {
  uint64_t blocked = 0;
  int cnt = 0;
  for (uint64_t q : m) {
    if ((q & blocked) | (q & ~S)) {
      blocked |= q;
      if ((blocked & S) == S) break;
      continue;
    }
    ++cnt;
  }
  return cnt;
}

// S grown to `size` qubits in circuit order from gate `start`, then by the lowest
// qubits of `within`
uint64_t grow(const std::vector<uint64_t>& m, size_t start, uint64_t S, int size, uint64_t within) {
  uint64_t blocked = 0;
  const size_t end = std::min(m.size(), start + 400);
  for (size_t i = start; i < end && popc(S) < size; ++i) {
    const uint64_t q = m[i];
    if ((q & blocked) | (q & ~within)) {
      blocked |= q;
      continue;
    }
    if (popc(S | q) <= size) S |= q;
    else blocked |= q;
  }
  for (uint64_t r = within & ~S; r && popc(S) < size; r &= r - 1) S |= r & (~r + 1);
  return S;
}

// Up to kChainMax blocks of 5 qubits of T for the gates that T takes, each the one (of the
// sets grown from the first gates left, and of 5 neighbouring qubits of T) that takes the
// most; returns the gates taken.
int split_tile(const std::vector<uint64_t>& m, uint64_t T, std::vector<uint64_t>& blocks) {
  std::vector<uint64_t> sub;
  uint64_t blocked = 0;
  for (uint64_t q : m) {
    if ((q & blocked) | (q & ~T)) {
      blocked |= q;
      if ((blocked & T) == T) break;
      continue;
    }
    sub.push_back(q);
  }
  uint64_t bit[12];
  int nb = 0;
  for (uint64_t r = T; r; r &= r - 1) bit[nb++] = r & (~r + 1);
  blocks.clear();
  int total = 0;
  while ((int)blocks.size() < kChainMax && !sub.empty()) {
    uint64_t best = 0;
    int best_cnt = -1;
    auto consider = [&](uint64_t S) {
      const int c = takes(sub, S);
      if (c > best_cnt) {
        best_cnt = c;
        best = S;
      }
    };
    for (size_t s = 0; s < 12 && s < sub.size(); ++s) consider(grow(sub, s, 0, 5, T));
    for (int a = 0; a + 5 <= nb; ++a) consider(bit[a] | bit[a + 1] | bit[a + 2] | bit[a + 3] | bit[a + 4]);
    blocks.push_back(best);
    total += best_cnt;
    blocked = 0;
    size_t w = 0;
    for (uint64_t q : sub)
      if ((q & blocked) | (q & ~best)) {
        blocked |= q;
        sub[w++] = q;
      }
    sub.resize(w);
  }
  return total;
}

}  // namespace

// Pass by pass: among tiles (those grown from each of the first gates left, and bits 0..3
// with every window of 8 neighbouring qubits) the kTry that take the most gates are split
// into blocks, and the one whose blocks take the most is kept.  40 layers of Haar + CZ at
// 30 qubits: 37 passes of 109 blocks.
void plan_chains(const qs_gate* gates, size_t ngates, int n, std::vector<ChainPlan>& out, bool products) {
  constexpr size_t kSeeds = 12, kTry = 4;
  const uint64_t low = (1ull << kChainLow) - 1, all = n >= 64 ? ~0ull : (1ull << n) - 1;
  out.clear();
  std::vector<uint64_t> m(ngates);
  std::vector<size_t> idx(ngates);
  for (size_t i = 0; i < ngates; ++i) {
    m[i] = mask_of(gates[i]);
    idx[i] = i;
  }
  std::vector<std::pair<int, uint64_t>> cand;
  std::vector<uint64_t> blocks, best;
  while (!m.empty()) {
    cand.clear();
    auto add = [&](uint64_t T) {
      for (const auto& c : cand)
        if (c.second == T) return;
      cand.push_back({takes(m, T), T});
    };
    for (size_t k = 0; k < kSeeds && k < m.size(); ++k) add(grow(m, k, low, 12, all));
    for (int a = kChainLow; a + 8 <= n; ++a) add(low | (255ull << a));
    std::stable_sort(cand.begin(), cand.end(), [](const auto& a, const auto& b) { return a.first > b.first; });
    int best_cnt = -1;
    ChainPlan p;
    for (size_t t = 0; t < kTry && t < cand.size() && cand[t].first > best_cnt; ++t) {
      const int c = split_tile(m, cand[t].second, blocks);
      if (c > best_cnt) {
        best_cnt = c;
        best = blocks;
        p.tile = cand[t].second;
      }
    }
    for (uint64_t S : best) {
      Block b;
      int i = 0;
      for (int q = 0; q < n; ++q)
        if ((S >> q) & 1) b.q[i++] = q;
      uint64_t blocked = 0;
      size_t w = 0;
      for (size_t j = 0; j < m.size(); ++j) {
        const uint64_t q = m[j];
        if ((q & blocked) | (q & ~S)) {
          blocked |= q;
          m[w] = q;
          idx[w++] = idx[j];
        } else {
          b.gate_idx.push_back(idx[j]);
        }
      }
      m.resize(w);
      idx.resize(w);
      b.ngates = (int)b.gate_idx.size();
      p.blocks.push_back(std::move(b));
    }
    out.push_back(std::move(p));
  }
  if (!products) return;
  std::vector<Block*> flat;
  for (ChainPlan& p : out)
    for (Block& b : p.blocks) flat.push_back(&b);
  parallel_for(flat.size(), 8, [&](size_t i) { block_product(gates, *flat[i]); });
}

namespace {

bool branches(const qs_gate& g) {
  switch (g.kind) {
    case QS_H: case QS_PX: case QS_MX: case QS_PY: case QS_MY: case QS_RX: case QS_RY: case QS_U2: case QS_U3:
    case QS_MAT1: case QS_MAT2:
      return true;
    default:
      return false;
  }
}
bool fixed_branch(const qs_gate& g) {
  return g.kind == QS_H || g.kind == QS_PX || g.kind == QS_MX || g.kind == QS_PY || g.kind == QS_MY;
}

}  // namespace

// block_nonzeros(b) > 512 without the product where its pattern decides: entry (r, c) can be
// nonzero only if a path of nonzero gate entries leads there.  A pattern that is sparse is
// certain; sums that cancel exactly come from the fixed gates (H H = 1), so a block with two
// of those is multiplied out.
bool block_dense(const qs_gate* gates, const Block& b) {
  uint32_t row[32];
  for (int r = 0; r < 32; ++r) row[r] = 1u << r;
  int fixed = 0;
  for (size_t gi : b.gate_idx) {
    const qs_gate& g = gates[gi];
    if (!branches(g) && g.kind < QS_CNOT && g.kind != QS_X && g.kind != QS_Y) continue;   // diagonal
    fixed += fixed_branch(g);
    cd m[16];
    int dim = 0, at[2] = {0, 0};
    gate_matrix(g, m, &dim);
    for (int k = 0; k < (dim == 4 ? 2 : 1); ++k)
      for (int i = 0; i < 5; ++i)
        if (b.q[i] == g.q[k]) at[k] = i;
    const int hi = 1 << at[0], lo = dim == 4 ? 1 << at[1] : 0;
    for (int r = 0; r < 32; ++r) {
      if ((r & hi) || (r & lo)) continue;
      const int idx[4] = {r, dim == 4 ? r | lo : r | hi, r | hi, r | hi | lo};
      uint32_t out[4] = {0, 0, 0, 0};
      for (int i = 0; i < dim; ++i)
        for (int k = 0; k < dim; ++k)
          if (m[i * dim + k] != cd(0)) out[i] |= row[idx[k]];
      for (int i = 0; i < dim; ++i) row[idx[i]] = out[i];
    }
  }
  int nz = 0;
  for (int r = 0; r < 32; ++r) nz += __builtin_popcount(row[r]);
  if (nz <= 512 || fixed < 2) return nz > 512;
  Block c = b;
  block_product(gates, c);
  return block_nonzeros(c) > 512;
}

bool chains_likely(const qs_gate* gates, size_t ngates) {
  size_t k = 0;
  for (size_t i = 0; i < ngates; ++i) k += branches(gates[i]);
  return 5 * k > ngates;
}

bool chains_dense(const qs_gate* gates, const std::vector<ChainPlan>& plan) {
  size_t total = 0, dense = 0, sparse = 0;
  for (const ChainPlan& p : plan) total += p.blocks.size();
  for (const ChainPlan& p : plan)
    for (const Block& b : p.blocks) {
      ++(block_dense(gates, b) ? dense : sparse);
      if (4 * dense >= 3 * total) return true;   // (decided: the rest need not be looked at)
      if (4 * sparse > total) return false;
    }
  return false;
}

namespace {

// Adds the bank bits (bits 0..3) of v to a reduced basis; true if they are new.
bool add_rank(uint32_t basis[4], uint32_t v) {
  uint32_t x = v & 15u;
  for (int b = 3; b >= 0; --b)
    if ((x >> b) & 1) {
      if (!basis[b]) {
        basis[b] = x;
        return true;
      }
      x ^= basis[b];
    }
  return false;
}

bool spans(const uint32_t* v, const int* rows) {
  uint32_t basis[4] = {0, 0, 0, 0};
  int r = 0;
  for (int i = 0; i < 4; ++i) r += add_rank(basis, v[rows[i]]);
  return r == 4;
}

}  // namespace

// A slot holds the tile as the tensor box lands: local bits 0..3 = physical bits 0..3,
// then run1, run2 and the other positions.  A warp reads or writes one column of 32 rows
// at a time, 8 bytes a lane and 16 lanes at a time, so the rows on lane bits 0..3 should
// span the four bank bits (bits 0..3 of the 8-byte index).  For the first read and the last
// write the layout is the box's: the 128-byte swizzle adds local bits 4..6 to bank bits
// 1..3, and the rows that give the largest rank go to the lanes.  Between two blocks the
// layout is free: local bit j >= 4 is also XORed into bank bits f[j], drawn until both the
// write and the read that follows are without conflicts.
bool chain_pass_desc(int n, uint64_t tile, const uint64_t* blocks, int nblk, ChainPass& P) {
  std::memset(&P, 0, sizeof(P));
  const uint64_t low = (1ull << kChainLow) - 1;
  if (n < 12 || n > 36 || nblk < 1 || nblk > kChainMax || popc(tile) != 12 || (tile >> n) || (tile & low) != low)
    return false;
  // runs of neighbouring tile positions above bit 3; the two longest go into the box
  std::vector<std::pair<int, int>> runs;   // (start, length)
  for (int p = kChainLow; p < n; ++p) {
    if (!((tile >> p) & 1)) {
      P.nt_pos[P.n_nt++] = (uint8_t)p;
      continue;
    }
    if (!runs.empty() && runs.back().first + runs.back().second == p) ++runs.back().second;
    else runs.push_back({p, 1});
  }
  std::vector<int> by((size_t)runs.size());
  for (size_t i = 0; i < by.size(); ++i) by[i] = (int)i;
  std::stable_sort(by.begin(), by.end(), [&](int a, int b) { return runs[a].second > runs[b].second; });
  int r1 = by[0], r2 = by.size() > 1 ? by[1] : -1;
  if (r2 >= 0 && r2 < r1) std::swap(r1, r2);
  P.a1 = runs[r1].first;
  P.g1 = runs[r1].second;
  P.b = r2 >= 0 ? runs[r2].first : P.a1 + P.g1;
  P.g2 = r2 >= 0 ? runs[r2].second : 0;
  int local[12], nl = 0;   // physical position of each local bit
  for (int p = 0; p < kChainLow; ++p) local[nl++] = p;
  for (int i = 0; i < P.g1; ++i) local[nl++] = P.a1 + i;
  for (int i = 0; i < P.g2; ++i) local[nl++] = P.b + i;
  for (size_t r = 0; r < runs.size(); ++r) {
    if ((int)r == r1 || (int)r == r2) continue;
    for (int i = 0; i < runs[r].second; ++i) {
      P.oth_pos[P.n_oth++] = (uint8_t)(runs[r].first + i);
      local[nl++] = runs[r].first + i;
    }
  }
  // (boxes of at least 1 KiB, so that each begins on the swizzle's 1 KiB pattern)
  P.swizzle = P.g1 + P.g2 >= 3 ? 1 : 0;
  uint32_t box[12];   // 8-byte index of each local bit in the box's layout
  for (int j = 0; j < 12; ++j) box[j] = (1u << j) ^ (P.swizzle && j >= 4 && j <= 6 ? 1u << (j - 3) : 0u);
  int rows[kChainMax][7], cols[kChainMax][5];
  for (int b = 0; b < nblk; ++b) {
    int free_rows[7], nr = 0, nc = 0;
    for (int p = 0; p < n; ++p) {
      if (!((blocks[b] >> p) & 1)) continue;
      int j = 0;
      while (j < 12 && local[j] != p) ++j;
      if (j == 12 || nc == 5) return false;
      cols[b][nc++] = j;   // ascending positions = the block's local index bits
    }
    if (nc != 5) return false;
    for (int j = 0; j < 12; ++j)
      if (std::find(cols[b], cols[b] + 5, j) == cols[b] + 5) free_rows[nr++] = j;
    // lane bits first: rows that raise the rank of the box layout's bank bits
    uint32_t basis[4] = {0, 0, 0, 0};
    int k = 0;
    bool used[7] = {};
    for (int i = 0; i < 7; ++i)
      if (add_rank(basis, box[free_rows[i]])) {
        rows[b][k++] = free_rows[i];
        used[i] = true;
      }
    for (int i = 0; i < 7; ++i)
      if (!used[i]) rows[b][k++] = free_rows[i];
  }
  auto fill = [&](ChainMap& M, int b, const uint32_t* v) {
    for (int i = 0; i < 7; ++i) M.row[i] = (uint16_t)(8u * v[rows[b][i]]);
    for (int i = 0; i < 5; ++i) M.col[i] = (uint16_t)(8u * v[cols[b][i]]);
  };
  fill(P.rd[0], 0, box);
  fill(P.wr[nblk - 1], nblk - 1, box);
  uint32_t seed = 0x9e3779b9u;
  for (int b = 0; b + 1 < nblk; ++b) {
    uint32_t v[12];
    for (int trial = 0; trial < 4096; ++trial) {
      for (int j = 0; j < 12; ++j) {
        v[j] = 1u << j;
        if (j < 4) continue;
        seed ^= seed << 13;
        seed ^= seed >> 17;
        seed ^= seed << 5;
        v[j] |= seed & 15u;
      }
      if (spans(v, rows[b]) && spans(v, rows[b + 1])) break;
    }
    fill(P.wr[b], b, v);
    fill(P.rd[b + 1], b + 1, v);
  }
  P.nblk = nblk;
  // as many as shared memory holds beside the blocks' operands: six slots with one block, five
  // with two (one of them between the blocks) or three (two between)
  P.nload = nblk == 1 ? 3 : 2;
  P.nstore = nblk == 1 ? 3 : nblk == 2 ? 2 : 1;
  return true;
}

// B, per BF16 part: 96 rows of K = 32, rows [-Im U | Re U | Im U] (row r of each = output r).
// The products with the real parts of a row read rows 32..95 and give (Re, Im) of the
// outputs in columns 0..31 and 32..63; those with the imaginary parts read rows 0..63.
// K-major core matrices of 8 rows x 16 bytes, no swizzle.
void chain_b_operand(const cd* U, unsigned char* out) {
  for (int row = 0; row < 32; ++row)
    for (int k0 = 0; k0 < 32; k0 += 8) {
      uint16_t re[3][8], im[3][8], neg[3][8];
      for (int k = 0; k < 8; ++k) {
        double a = U[row * 32 + k0 + k].real(), c = U[row * 32 + k0 + k].imag();
        for (int p = 0; p < 3; ++p) {
          re[p][k] = bf16_round_host((float)a);
          im[p][k] = bf16_round_host((float)c);
          neg[p][k] = im[p][k] ^ 0x8000u;
          a -= (double)bf16_to_float(re[p][k]);
          c -= (double)bf16_to_float(im[p][k]);
        }
      }
      unsigned char* at = out + (row >> 3) * 512 + (k0 >> 3) * 128 + (row & 7) * 16;
      for (int p = 0; p < 3; ++p, at += kChainPart) {
        std::memcpy(at, neg[p], 16);
        std::memcpy(at + 4 * 512, re[p], 16);
        std::memcpy(at + 8 * 512, im[p], 16);
      }
    }
}

}  // namespace qs
