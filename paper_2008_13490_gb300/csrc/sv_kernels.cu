// State-vector kernels for sm_103a.
//
//  tile_pass_kernel   one HBM read+write of the state applies every op of a
//                     pass: a CTA owns a tile of 2^12 amplitudes (12 qubits,
//                     any bit positions that include bits 0,1), lanes hold the 5
//                     lowest tile bits (gates there use warp shuffles), each
//                     thread holds 16 amplitudes in registers (4 tile bits),
//                     and shared memory transposes swap register and warp bits
//                     between stages.
//  plain_*_kernel     one launch per gate, the pair/quad update of the thesis's
//                     four-component loops (Eq. (psioft4componentupdates)) with
//                     the bit-insert index of its reduced loop, 64-bit indices.
//  small_state_kernel whole state in the registers of one CTA or a cluster (n < 12; the
//                     default method: n < 14).
//  remap_kernel       permutes bit positions inside a 12-bit tile (in place).
//  probs / marginal / loglik / reduce: Born rule p_J = |a_J|^2 with fp64
//                     accumulation of the sums.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstddef>
#include <cstring>

#include "dev_common.cuh"
#include "internal.h"
#include "tile_cp.h"

namespace qs {

// ------------------------------------------------------------------ tile pass

template <int J, typename R>
__device__ __forceinline__ void reg_gate(C2<R>* v, const C2<R>* m) {
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    if (r & (1 << J)) continue;
    const C2<R> a = v[r], b = v[r | (1 << J)];
    v[r] = cfma2(m[0], a, m[1], b);
    v[r | (1 << J)] = cfma2(m[2], a, m[3], b);
  }
}

template <int J, int K, typename R>
__device__ __forceinline__ void reg_gate_choice(C2<R>* v, const C2<R>* m0, const C2<R>* m1) {
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    if (r & (1 << J)) continue;
    const C2<R>* m = ((r >> K) & 1) ? m1 : m0;
    const C2<R> a = v[r], b = v[r | (1 << J)];
    v[r] = cfma2(m[0], a, m[1], b);
    v[r | (1 << J)] = cfma2(m[2], a, m[3], b);
  }
}

template <int K, typename R>
__device__ __forceinline__ void lane_gate_choice(C2<R>* v, int mask, C2<R> o0, C2<R> p0, C2<R> o1,
                                                 C2<R> p1) {
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const C2<R> q = shfl_xor_c(v[r], mask);
    if ((r >> K) & 1) v[r] = cfma2(o1, v[r], p1, q);
    else v[r] = cfma2(o0, v[r], p0, q);
  }
}

// ---- ops whose matrices are real (H, RY, X, CNOT): a product with each part, two packed FP32
// instructions per output amplitude in place of four; the values are those of cfma2

template <typename R>
__device__ __forceinline__ C2<R> rfma2(R m0, C2<R> a, R m1, C2<R> b) {
  return C2<R>{fma(m1, b.x, m0 * a.x), fma(m1, b.y, m0 * a.y)};
}
template <>
__device__ __forceinline__ C2<float> rfma2<float>(float m0, C2<float> a, float m1, C2<float> b) {
  const float2 r = __ffma2_rn(make_float2(m1, m1), make_float2(b.x, b.y),
                              __fmul2_rn(make_float2(m0, m0), make_float2(a.x, a.y)));
  return C2<float>{r.x, r.y};
}

// K < 0: the matrix m0; else m1 where register bit K is 1
template <int J, int K, typename R>
__device__ __forceinline__ void reg_gate_real(C2<R>* v, const R* m0, const R* m1) {
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    if (r & (1 << J)) continue;
    const R* m = K >= 0 && ((r >> (K < 0 ? 0 : K)) & 1) ? m1 : m0;
    const C2<R> a = v[r], b = v[r | (1 << J)];
    v[r] = rfma2(m[0], a, m[1], b);
    v[r | (1 << J)] = rfma2(m[2], a, m[3], b);
  }
}

// [1 1; 1 -1] (a Hadamard gate but for its factor, which the host gives to one op of several)
template <int J, typename R>
__device__ __forceinline__ void reg_butterfly(C2<R>* v) {
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    if (r & (1 << J)) continue;
    const C2<R> a = v[r], b = v[r | (1 << J)];
    v[r] = C2<R>{a.x + b.x, a.y + b.y};
    v[r | (1 << J)] = C2<R>{a.x - b.x, a.y - b.y};
  }
}

// ---- dense 4x4 ops on two qubits a (local index msb) and b: y = G x on each quad

template <typename R>
__device__ __forceinline__ C2<R> sel4(int o, C2<R> g0, C2<R> g1, C2<R> g2, C2<R> g3) {
  return csel(o >= 2, csel(o == 3, g3, g2), csel(o == 1, g1, g0));
}

// both qubits in register slots KA, KB: the quad of each r is in registers
template <int KA, int KB, typename R>
__device__ __forceinline__ void reg_g2(C2<R>* v, const C2<R>* g) {
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    if ((r >> KA) & 1 || (r >> KB) & 1) continue;
    C2<R> x[4];
#pragma unroll
    for (int l = 0; l < 4; ++l) x[l] = v[r | ((l >> 1) << KA) | ((l & 1) << KB)];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const C2<R> y0 = cfma2(g[4 * o], x[0], g[4 * o + 1], x[1]);
      const C2<R> y1 = cfma2(g[4 * o + 2], x[2], g[4 * o + 3], x[3]);
      v[r | ((o >> 1) << KA) | ((o & 1) << KB)] = C2<R>{y0.x + y1.x, y0.y + y1.y};
    }
  }
}

// one qubit on lane bit (mask), the other in register slot K; A_LANE: qubit a is
// the lane one.  Each lane holds two of a quad's amplitudes (register bit 0, 1),
// its partner lane the other two.
template <int K, bool A_LANE, typename R>
__device__ __forceinline__ void lane_reg_g2(C2<R>* v, const C2<R>* g, int mask, int u) {
  // quad index of (lane value w, register value c)
  auto q = [](int w, int c) { return A_LANE ? 2 * w + c : 2 * c + w; };
  C2<R> co[2][4];   // output c: coefficients of own c'=0, own 1, partner 0, partner 1
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int cc = j & 1, partner = j >> 1;
      // lane value of the input: own u or partner 1 - u; output at q(u, c)
      const C2<R> at0 = g[4 * q(0, c) + q(partner ? 1 : 0, cc)];   // u = 0
      const C2<R> at1 = g[4 * q(1, c) + q(partner ? 0 : 1, cc)];   // u = 1
      co[c][j] = csel(u != 0, at1, at0);
    }
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    if ((r >> K) & 1) continue;
    const C2<R> e0 = v[r], e1 = v[r | (1 << K)];
    const C2<R> p0 = shfl_xor_c(e0, mask), p1 = shfl_xor_c(e1, mask);
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const C2<R> y0 = cfma2(co[c][0], e0, co[c][1], e1);
      const C2<R> y1 = cfma2(co[c][2], p0, co[c][3], p1);
      v[r | (c << K)] = C2<R>{y0.x + y1.x, y0.y + y1.y};
    }
  }
}

// both qubits on lane bits: each lane holds one amplitude of every quad
template <typename R>
__device__ __forceinline__ void lane_lane_g2(C2<R>* v, const C2<R>* g, int ma, int mb, int o) {
  // o = own quad index 2 ua + ub; the amplitude at quad index o ^ f comes from lane ^ mask(f)
  const C2<R> c0 = sel4(o, g[0], g[5], g[10], g[15]);                    // f = 0: G[o][o]
  const C2<R> c1 = sel4(o, g[1], g[4], g[11], g[14]);                    // f = 1: G[o][o ^ 1]
  const C2<R> c2 = sel4(o, g[2], g[7], g[8], g[13]);                     // f = 2: G[o][o ^ 2]
  const C2<R> c3 = sel4(o, g[3], g[6], g[9], g[12]);                     // f = 3: G[o][o ^ 3]
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const C2<R> x = v[r];
    const C2<R> xb = shfl_xor_c(x, mb), xa = shfl_xor_c(x, ma), xab = shfl_xor_c(x, ma | mb);
    const C2<R> y0 = cfma2(c0, x, c1, xb);
    const C2<R> y1 = cfma2(c2, xa, c3, xab);
    v[r] = C2<R>{y0.x + y1.x, y0.y + y1.y};
  }
}

template <typename R>
__device__ __forceinline__ void apply_g2(C2<R>* v, const TileOp<R>* __restrict__ opp, int lane) {
  C2<R> g[16];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    g[i] = opp[0].m0[i];
    g[4 + i] = opp[0].m1[i];
    g[8 + i] = opp[1].m0[i];
    g[12 + i] = opp[1].m1[i];
  }
  const uint8_t sa = opp->csrc, ba = opp->cbit, sb = opp->dsrc, bb = opp->dbit;
  // the host orders the qubits: register slots ascending, a lane qubit first
  if (sa == CS_REG && sb == CS_REG) {
    switch (ba * 4 + bb) {
      case 1: reg_g2<0, 1>(v, g); break;
      case 2: reg_g2<0, 2>(v, g); break;
      case 3: reg_g2<0, 3>(v, g); break;
      case 6: reg_g2<1, 2>(v, g); break;
      case 7: reg_g2<1, 3>(v, g); break;
      default: reg_g2<2, 3>(v, g); break;
    }
    return;
  }
  if (sb == CS_LANE) {
    lane_lane_g2(v, g, 1 << ba, 1 << bb, 2 * ((lane >> ba) & 1) + ((lane >> bb) & 1));
    return;
  }
  const int mask = 1 << ba, u = (lane >> ba) & 1;   // a on the lane, b in register slot bb
  switch (bb) {
    case 0: lane_reg_g2<0, true>(v, g, mask, u); break;
    case 1: lane_reg_g2<1, true>(v, g, mask, u); break;
    case 2: lane_reg_g2<2, true>(v, g, mask, u); break;
    default: lane_reg_g2<3, true>(v, g, mask, u); break;
  }
}

template <typename R>
__device__ __forceinline__ int src_bit(uint8_t src, uint8_t bit, uint64_t tile, int lane, int warp) {
  switch (src) {
    case CS_TILE: return (int)((tile >> bit) & 1ull);
    case CS_LANE: return (lane >> bit) & 1;
    case CS_WARP: return (warp >> bit) & 1;
    default: return 0;
  }
}

// G2: the pass holds dense two-qubit ops (a kernel variant of its own, so that
// passes without them keep the leaner code)
// REAL: real matrices take their own path
template <typename R, bool G2, bool REAL = true>
__device__ __forceinline__ void apply_tile_op(C2<R>* v, const TileOp<R>* __restrict__ opp,
                                              uint64_t tile, int lane, int warp) {
  uint4 hdr = {};   // kind, slot, csrc, cbit | dsrc, dbit, term | pad[0..3] | pad[4..7]
  if (REAL) hdr = *reinterpret_cast<const uint4*>(opp);
  const uint8_t kind = opp->kind, slot = opp->slot, csrc = opp->csrc, cbit = opp->cbit;
  if constexpr (G2) {
    if (kind == TK_G2) {   // reads its continuation opp[1]
      apply_g2(v, opp, lane);
      return;
    }
  }
  if (REAL && (hdr.z & 0xff0000u)) {   // pad[2]: a real TK_REG or TK_LANE op
    R a[4], b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      a[i] = opp->m0[i].x;
      b[i] = opp->m1[i].x;
    }
    const bool in_reg = csrc == CS_REG;
    // [1 1; 1 -1] (beside the dense two-qubit code it costs registers, and with them a CTA per SM)
    if (!G2 && (hdr.z & 0xff0000u) == 0x20000u) {
      if (kind == TK_REG) {
        switch (slot) {
          case 0: reg_butterfly<0>(v); break;
          case 1: reg_butterfly<1>(v); break;
          case 2: reg_butterfly<2>(v); break;
          default: reg_butterfly<3>(v); break;
        }
        return;
      }
      const int mask = 1 << slot;
      const R sign = (lane & mask) ? R(-1) : R(1);
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const C2<R> q = shfl_xor_c(v[r], mask);
        v[r] = C2<R>{fma(sign, v[r].x, q.x), fma(sign, v[r].y, q.y)};
      }
      return;
    }
    if (!in_reg && csrc != CS_NONE && src_bit<R>(csrc, cbit, tile, lane, warp)) {
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = b[i];
    }
    if (kind == TK_REG) {
      switch (in_reg ? slot * 4 + cbit : 16 + slot) {
        case 1: reg_gate_real<0, 1>(v, a, b); break;
        case 2: reg_gate_real<0, 2>(v, a, b); break;
        case 3: reg_gate_real<0, 3>(v, a, b); break;
        case 4: reg_gate_real<1, 0>(v, a, b); break;
        case 6: reg_gate_real<1, 2>(v, a, b); break;
        case 7: reg_gate_real<1, 3>(v, a, b); break;
        case 8: reg_gate_real<2, 0>(v, a, b); break;
        case 9: reg_gate_real<2, 1>(v, a, b); break;
        case 11: reg_gate_real<2, 3>(v, a, b); break;
        case 12: reg_gate_real<3, 0>(v, a, b); break;
        case 13: reg_gate_real<3, 1>(v, a, b); break;
        case 14: reg_gate_real<3, 2>(v, a, b); break;
        case 16: reg_gate_real<0, -1>(v, a, a); break;
        case 17: reg_gate_real<1, -1>(v, a, a); break;
        case 18: reg_gate_real<2, -1>(v, a, a); break;
        default: reg_gate_real<3, -1>(v, a, a); break;
      }
      return;
    }
    const int mask = 1 << slot;
    const bool up = (lane >> slot) & 1;
    const R o0 = up ? a[3] : a[0], p0 = up ? a[2] : a[1], o1 = up ? b[3] : b[0], p1 = up ? b[2] : b[1];
    if (!G2 && !in_reg) {   // (registers, as above)
#pragma unroll
      for (int r = 0; r < 16; ++r) v[r] = rfma2(o0, v[r], p0, shfl_xor_c(v[r], mask));
      return;
    }
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const C2<R> q = shfl_xor_c(v[r], mask);
      const bool one = in_reg && ((r >> cbit) & 1);
      v[r] = rfma2(one ? o1 : o0, v[r], one ? p1 : p0, q);
    }
    return;
  }
  C2<R> m0[4], m1[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) m0[i] = opp->m0[i];
  if (csrc == CS_NONE && kind != TK_DIAG) {   // no choice bit: one matrix, no matrix selects
    if (kind == TK_REG) {
      switch (slot) {
        case 0: reg_gate<0>(v, m0); break;
        case 1: reg_gate<1>(v, m0); break;
        case 2: reg_gate<2>(v, m0); break;
        default: reg_gate<3>(v, m0); break;
      }
      return;
    }
    const int mask = 1 << slot;
    const bool b = (lane >> slot) & 1;
    const C2<R> o = csel(b, m0[3], m0[0]), p = csel(b, m0[2], m0[1]);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const C2<R> q = shfl_xor_c(v[r], mask);
      v[r] = cfma2(o, v[r], p, q);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) m1[i] = opp->m1[i];
  if (kind == TK_REG) {
    if (csrc == CS_REG) {
      switch (slot * 4 + cbit) {
        case 1: reg_gate_choice<0, 1>(v, m0, m1); break;
        case 2: reg_gate_choice<0, 2>(v, m0, m1); break;
        case 3: reg_gate_choice<0, 3>(v, m0, m1); break;
        case 4: reg_gate_choice<1, 0>(v, m0, m1); break;
        case 6: reg_gate_choice<1, 2>(v, m0, m1); break;
        case 7: reg_gate_choice<1, 3>(v, m0, m1); break;
        case 8: reg_gate_choice<2, 0>(v, m0, m1); break;
        case 9: reg_gate_choice<2, 1>(v, m0, m1); break;
        case 11: reg_gate_choice<2, 3>(v, m0, m1); break;
        case 12: reg_gate_choice<3, 0>(v, m0, m1); break;
        case 13: reg_gate_choice<3, 1>(v, m0, m1); break;
        case 14: reg_gate_choice<3, 2>(v, m0, m1); break;
        default: break;
      }
      return;
    }
    const bool s = (csrc != CS_NONE) && src_bit<R>(csrc, cbit, tile, lane, warp);
    C2<R> m[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) m[i] = csel(s, m1[i], m0[i]);
    switch (slot) {
      case 0: reg_gate<0>(v, m); break;
      case 1: reg_gate<1>(v, m); break;
      case 2: reg_gate<2>(v, m); break;
      default: reg_gate<3>(v, m); break;
    }
    return;
  }
  if (kind == TK_LANE) {
    const int mask = 1 << slot;
    const bool b = (lane >> slot) & 1;
    // out = own-coefficient * own + partner-coefficient * partner
    const C2<R> o0 = csel(b, m0[3], m0[0]), p0 = csel(b, m0[2], m0[1]);
    const C2<R> o1 = csel(b, m1[3], m1[0]), p1 = csel(b, m1[2], m1[1]);
    if (csrc == CS_REG) {
      switch (cbit) {
        case 0: lane_gate_choice<0>(v, mask, o0, p0, o1, p1); break;
        case 1: lane_gate_choice<1>(v, mask, o0, p0, o1, p1); break;
        case 2: lane_gate_choice<2>(v, mask, o0, p0, o1, p1); break;
        default: lane_gate_choice<3>(v, mask, o0, p0, o1, p1); break;
      }
      return;
    }
    const bool s = (csrc != CS_NONE) && src_bit<R>(csrc, cbit, tile, lane, warp);
    const C2<R> o = csel(s, o1, o0), p = csel(s, p1, p0);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const C2<R> q = shfl_xor_c(v[r], mask);
      v[r] = cfma2(o, v[r], p, q);
    }
    return;
  }
  // TK_DIAG ops go through DiagRun below.
}

// A run of consecutive diagonal ops (they commute) collapses, per thread, into a
// diagonal over the 4 register bits: a scalar s (ops whose bits are all lane,
// warp or tile-constant bits) times one 2-entry factor f[k] per register slot k
// (ops with one bit in a register).  An op with both bits in registers
// multiplies v directly.  flush() multiplies the collected diagonal into v once
// the run ends.  Per op this is 1-2 complex products per thread instead of 16.
// FLAG: a run that set no register-slot factor is multiplied by its scalar alone.  That saves FP64
// instructions and runs beside TK_RUN; in the lean FP32 code it cost registers for nothing (25 qubits, 20
// layers of Haar + CZ on tiles: 5.08 ms with it, 4.09 without).
template <typename R, bool FLAG>
struct DiagRun {
  C2<R> s, f0[2], f1[2], f2[2], f3[2];   // compile-time indices only (registers)
  bool slots;                            // a factor of a register slot was set (the same for the warp)

  __device__ __forceinline__ void reset() {
    const C2<R> one{R(1), R(0)};
    slots = false;
    s = one;
    f0[0] = f0[1] = f1[0] = f1[1] = f2[0] = f2[1] = f3[0] = f3[1] = one;
  }
  __device__ __forceinline__ void fold(int k, C2<R> e0, C2<R> e1) {
    slots = true;
    switch (k) {
      case 0: f0[0] = cmul(f0[0], e0); f0[1] = cmul(f0[1], e1); break;
      case 1: f1[0] = cmul(f1[0], e0); f1[1] = cmul(f1[1], e1); break;
      case 2: f2[0] = cmul(f2[0], e0); f2[1] = cmul(f2[1], e1); break;
      default: f3[0] = cmul(f3[0], e0); f3[1] = cmul(f3[1], e1); break;
    }
  }
  // d[2*bit_a + bit_b] (d[bit_a] for one-qubit diagonals); with TWO the
  // direct products go to v2 as well (the adjoint pass carries two states)
  template <bool TWO = false>
  __device__ __forceinline__ void add(C2<R>* v, const TileOp<R>* __restrict__ opp, uint64_t tile,
                                      int lane, int warp, C2<R>* v2 = nullptr) {
    const uint8_t csrc = opp->csrc, cbit = opp->cbit, dsrc = opp->dsrc, dbit = opp->dbit;
    C2<R> d[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) d[i] = opp->m0[i];
    const bool two = dsrc != CS_NONE;
    const bool ra = csrc == CS_REG, rb = dsrc == CS_REG;
    if (ra && rb) {
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const int idx = ((r >> cbit) & 1) * 2 + ((r >> dbit) & 1);
        const C2<R> f = csel(idx >= 2, csel(idx == 3, d[3], d[2]), csel(idx == 1, d[1], d[0]));
        v[r] = cmul(v[r], f);
        if (TWO) v2[r] = cmul(v2[r], f);
      }
      return;
    }
    const int ua = ra ? 0 : src_bit<R>(csrc, cbit, tile, lane, warp);
    const int ub = (two && !rb) ? src_bit<R>(dsrc, dbit, tile, lane, warp) : 0;
    if (ra) {   // entries for bit_a = 0 and 1 at this thread's bit_b
      if (two) fold(cbit, csel(ub, d[1], d[0]), csel(ub, d[3], d[2]));
      else fold(cbit, d[0], d[1]);
    } else if (rb) {   // entries for bit_b = 0 and 1 at this thread's bit_a
      fold(dbit, csel(ua, d[2], d[0]), csel(ua, d[3], d[1]));
    } else {
      const int idx = two ? (ua * 2 + ub) : ua;
      s = cmul(s, csel(idx >= 2, csel(idx == 3, d[3], d[2]), csel(idx == 1, d[1], d[0])));
    }
  }
  // TK_CP: one complex multiply into the factor of the register bit (or into
  // s), selected by the other bit; 16 selected multiplies when both bits are
  // register bits
  // (hdr = the op's first 16 bytes, read with one load: kind, slot, csrc,
  // cbit | dsrc, dbit, term | pad[0..3] | pad[4..7])
  __device__ __forceinline__ void add_cp(C2<R>* v, const TileOp<R>* __restrict__ opp, uint4 hdr,
                                         uint64_t ctx) {
    const uint32_t csrc = (hdr.x >> 16) & 0xffu, cbit = hdr.x >> 24, dsrc = hdr.y & 0xffu,
                   dbit = (hdr.y >> 8) & 0xffu, pa = hdr.z & 0xffu, pb = (hdr.z >> 8) & 0xffu;
    const C2<R> p = opp->m0[0], one{R(1), R(0)};
    const bool ra = csrc == CS_REG, rb = dsrc == CS_REG;
    if (ra && rb) {
#pragma unroll
      for (int r = 0; r < 16; ++r) v[r] = cmul(v[r], csel(((r >> cbit) & (r >> dbit) & 1) != 0, p, one));
      return;
    }
    const int ua = ra ? 1 : (int)((ctx >> pa) & 1ull);
    const int ub = rb ? 1 : (int)((ctx >> pb) & 1ull);
    const C2<R> e = csel((ua & ub) != 0, p, one);
    if (ra || rb) {
      slots = true;
      switch (ra ? cbit : dbit) {
        case 0: f0[1] = cmul(f0[1], e); break;
        case 1: f1[1] = cmul(f1[1], e); break;
        case 2: f2[1] = cmul(f2[1], e); break;
        default: f3[1] = cmul(f3[1], e); break;
      }
    } else {
      s = cmul(s, e);
    }
  }
  template <bool TWO = false>
  __device__ __forceinline__ void flush(C2<R>* v, C2<R>* v2 = nullptr) {
    if (FLAG && !slots) {
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        v[r] = cmul(v[r], s);
        if (TWO) v2[r] = cmul(v2[r], s);
      }
      reset();
      return;
    }
    // D(r) = s f0[r0] f1[r1] f2[r2] f3[r3] as (s f0 f1)[r & 3] * (f2 f3)[r >> 2]
    const C2<R> a0 = cmul(s, f0[0]), a1 = cmul(s, f0[1]);
    const C2<R> lo[4] = {cmul(a0, f1[0]), cmul(a1, f1[0]), cmul(a0, f1[1]), cmul(a1, f1[1])};
    const C2<R> hi[4] = {cmul(f2[0], f3[0]), cmul(f2[1], f3[0]), cmul(f2[0], f3[1]),
                         cmul(f2[1], f3[1])};
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const C2<R> D = cmul(lo[r & 3], hi[r >> 2]);
      v[r] = cmul(v[r], D);
      if (TWO) v2[r] = cmul(v2[r], D);
    }
    reset();
  }
};

// TK_RUN (tile_cp.h): a diagonal s prod_k f_k^(bit k of r) T[r] over the 16 register indices.
// U, W: the CTA's factors of the jobs and thread jobs; tabs: the (lane, warp) and register
// tables of the pass (lw = warp * 32 + lane).  Instruction issue bounds the pass, not HBM (30-qubit
// Fourier transform: 10.6 ms a pass for 2.5 ms of traffic): a run whose ops share a register slot,
// as those before a Hadamard on it do, touches the eight amplitudes where it is 1 and no others, and
// the rest of the diagonal is formed once from lo and hi parts (14.5 ms a pass with the general
// diagonal of DiagRun for each run, and the tile x thread phases one by one in each thread).
template <typename R>
__device__ __forceinline__ C2<R> run_entries(C2<R> f, const RunEntry<R>* __restrict__ e, int n, uint64_t ctx) {
  const C2<R> one{R(1), R(0)};
  for (int i = 0; i < n; ++i) {
    const RunEntry<R> x = e[i];
    f = cmul(f, csel(((ctx >> x.pa) & 1ull) != 0, x.p, one));
  }
  return f;
}
// every op has a bit in slot K: the amplitudes where it is 1
template <int K, typename R>
__device__ __forceinline__ void run_in_slot(C2<R>* v, C2<R> f, const C2<R>* __restrict__ T) {
  if (T) {
#pragma unroll
    for (int r = 0; r < 16; ++r)
      if (r & (1 << K)) v[r] = cmul(v[r], cmul(f, T[r]));
  } else {
#pragma unroll
    for (int r = 0; r < 16; ++r)
      if (r & (1 << K)) v[r] = cmul(v[r], f);
  }
}
template <typename R>
__device__ __forceinline__ void apply_cp_run(C2<R>* v, const TileOp<R>* __restrict__ opp, uint64_t ctx, int lw,
                                             const C2<R>* U, const C2<R>* W, const C2<R>* __restrict__ tabs) {
  // RunHeader, read as words: n_s, n_f[0] | n_f[1], n_f[2] | n_f[3], ubase | umask, tmask, - | toff | wbase, wmask, slot
  static_assert(offsetof(RunHeader, n_f) == 2 && offsetof(RunHeader, ubase) == 10 && offsetof(RunHeader, umask) == 12 &&
                offsetof(RunHeader, tmask) == 13 && offsetof(RunHeader, toff) == 16 && offsetof(RunHeader, wbase) == 20 &&
                offsetof(RunHeader, wmask) == 22 && offsetof(RunHeader, slot) == 23 && offsetof(TileOp<R>, m0) == 16);
  const uint4 w0 = *reinterpret_cast<const uint4*>(&opp->m0[0]);
  const uint2 w1 = *reinterpret_cast<const uint2*>(reinterpret_cast<const unsigned char*>(&opp->m0[0]) + 16);
  struct {
    uint32_t n_s, n_f[4], ubase, umask, tmask, toff, wbase, wmask, slot;
  } h = {w0.x & 0xffffu, {w0.x >> 16, w0.y & 0xffffu, w0.y >> 16, w0.z & 0xffffu}, w0.z >> 16, w0.w & 0xffu,
         (w0.w >> 8) & 0xffu, w1.x, w1.y & 0xffffu, (w1.y >> 16) & 0xffu, w1.y >> 24};
  const RunEntry<R>* __restrict__ e = reinterpret_cast<const RunEntry<R>*>(opp + 1);
  const C2<R>* __restrict__ T = tabs + h.toff;
  const C2<R> one{R(1), R(0)};
  if (h.slot) {
    const int k = (int)h.slot - 1;
    const int n_f = (int)(h.n_f[0] + h.n_f[1] + h.n_f[2] + h.n_f[3]);   // (only slot k's list is there)
    C2<R> f = one;
    if (n_f) f = run_entries(one, e, n_f, ctx);
    if (h.umask) f = cmul(f, U[h.ubase]);
    if (h.tmask & 31) {
      f = cmul(f, T[lw]);
      T += kRunTable;
    }
    if (!(h.tmask & 32)) T = nullptr;
    switch (k) {
      case 0: run_in_slot<0>(v, f, T); break;
      case 1: run_in_slot<1>(v, f, T); break;
      case 2: run_in_slot<2>(v, f, T); break;
      default: run_in_slot<3>(v, f, T); break;
    }
    return;
  }
  C2<R> s = one;
  if (h.wmask) {
    const C2<R>* w = W + h.wbase;
    const uint32_t bits = ((uint32_t)lw & 31u) | ((uint32_t)lw >> 5) << kLaneBits;   // lane, then warp bits
    for (uint32_t m = h.wmask; m; m &= m - 1) s = cmul(s, csel((bits & m & (0u - m)) != 0, *w++, one));
  } else {
    for (int i = 0; i < (int)h.n_s; ++i) {
      const RunEntry<R> x = e[i];
      s = cmul(s, csel(((ctx >> x.pa) & (ctx >> x.pb) & 1ull) != 0, x.p, one));
    }
  }
  e += h.n_s;
  int u = (int)h.ubase;
  if (h.umask & 1) s = cmul(s, U[u++]);
  if (h.tmask & 1) {
    s = cmul(s, T[lw]);
    T += kRunTable;
  }
  if (!((h.umask | h.tmask) & 30) && !(h.n_f[0] | h.n_f[1] | h.n_f[2] | h.n_f[3])) {
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = cmul(v[r], s);
  } else {
    C2<R> f[kRegBits];
#pragma unroll
    for (int k = 0; k < kRegBits; ++k) {
      f[k] = run_entries(one, e, h.n_f[k], ctx);
      e += h.n_f[k];
      if (h.umask & (2 << k)) f[k] = cmul(f[k], U[u++]);
      if (h.tmask & (2 << k)) {
        f[k] = cmul(f[k], T[lw]);
        T += kRunTable;
      }
    }
    // the products over slots 0 and 1, then over 2 and 3
    const C2<R> lo[4] = {s, cmul(s, f[0]), cmul(s, f[1]), cmul(cmul(s, f[0]), f[1])};
    const C2<R> f23 = cmul(f[2], f[3]);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      C2<R> d = lo[r & 3];
      if (r >= 4) d = cmul(d, r < 8 ? f[2] : (r < 12 ? f[3] : f23));
      v[r] = cmul(v[r], d);
    }
  }
  if (h.tmask & 32) {
#pragma unroll
    for (int r = 0; r < 16; ++r) v[r] = cmul(v[r], T[r]);
  }
}

// G2: the pass holds dense two-qubit ops; RUNS: it holds packed diagonal runs
// (TK_RUN); REAL: its real ops take their own path.  Each combination is its own
// instantiation, so that a pass without them keeps the leaner code and register allocation.
// FP32: three CTAs on an SM, 80 registers each (with two, 7 % slower); only the leanest has to be told.
template <typename R, bool G2, bool RUNS, bool REAL>
__global__ void __launch_bounds__(kTileThreads, sizeof(R) == 4 && !G2 && !RUNS && REAL ? 3 : 0)
    tile_pass_kernel(C2<R>* __restrict__ psi, const __grid_constant__ TileParams<R> P) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2<R>* sm = reinterpret_cast<C2<R>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t tile = blockIdx.x;

  __shared__ uint8_t s_pos[kTileBits];
  __shared__ uint64_t s_base;
  __shared__ C2<R> s_U[RUNS ? 2 * kMaxRunJobs : 1];   // the CTA's factors of jobs, then of thread jobs
  if (tid == 0) {
    const int n_nt = P.pass.n_nt;
    uint64_t base = 0;
    for (int j = 0; j < n_nt; ++j) base |= ((tile >> j) & 1ull) << P.pass.nt_pos[j];
    s_base = base;
  }
  if (tid < kTileBits) s_pos[tid] = P.pass.pos[tid];
  if constexpr (RUNS) {
    // one job per warp, an entry per lane: the product of its entries' phases at this
    // tile (bits below kCtxOne are tile bits, kCtxOne the constant 1)
    const uint64_t tctx = tile | (1ull << kCtxOne);
    const C2<R> one{R(1), R(0)};
    for (int j = warp; j < P.n_jobs + P.n_tjobs; j += kTileThreads / 32) {
      const bool tj = j >= P.n_jobs;
      RunJob jb;
      memcpy(&jb, tj ? P.tjobs + sizeof(RunJob) * (j - P.n_jobs) : P.jobs + sizeof(RunJob) * j, sizeof(jb));
      const RunEntry<R>* __restrict__ e = reinterpret_cast<const RunEntry<R>*>(P.ops + jb.op + 1) + jb.first;
      C2<R> u = one;
      for (int i = lane; i < jb.count; i += 32) {
        const RunEntry<R> x = e[i];
        const uint64_t b = jb.scalar ? ((tctx >> x.pa) & (tctx >> x.pb)) : (tctx >> x.pa);
        u = cmul(u, csel((b & 1ull) != 0, x.p, one));
      }
#pragma unroll
      for (int m = 16; m > 0; m >>= 1) u = cmul(u, shfl_xor_c(u, m));
      if (lane == 0) s_U[tj ? kMaxRunJobs + (j - P.n_jobs) : j] = u;
    }
  }
  __syncthreads();
  const uint64_t base = s_base;
  uint64_t loff = 0;
#pragma unroll
  for (int k = 0; k < kLaneBits; ++k)
    if ((lane >> k) & 1) loff |= 1ull << s_pos[k];

  const int nst = P.pass.n_stages;
  const TileStage* __restrict__ S = P.stages;
  const TileOp<R>* __restrict__ ops = P.ops;
  // context word of TK_CP bits: tile index, a constant 1 at bit 47, lane, warp
  const uint64_t ctx = tile | (1ull << kCtxOne) | ((uint64_t)lane << kCtxLane) | ((uint64_t)warp << kCtxWarp);
  C2<R> v[16];
  {
    const TileStage s0 = S[0];
    uint64_t g[kRegBits];
#pragma unroll
    for (int k = 0; k < kRegBits; ++k) g[k] = 1ull << s_pos[s0.reg[k]];
    uint64_t woff = 0;
#pragma unroll
    for (int k = 0; k < kWarpBits; ++k)
      if ((warp >> k) & 1) woff |= 1ull << s_pos[s0.warp[k]];
    const C2<R>* __restrict__ src = psi + (base | loff | woff);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      uint64_t o = 0;
#pragma unroll
      for (int k = 0; k < kRegBits; ++k)
        if ((r >> k) & 1) o |= g[k];
      v[r] = src[o];
    }
  }
  for (int s = 0; s < nst; ++s) {
    const TileStage cur = S[s];
    if (s > 0) {
      const TileStage prev = S[s - 1];
      int rb[kRegBits];
      int wo = lane;
#pragma unroll
      for (int k = 0; k < kRegBits; ++k) rb[k] = 1 << prev.reg[k];
#pragma unroll
      for (int k = 0; k < kWarpBits; ++k)
        if ((warp >> k) & 1) wo |= 1 << prev.warp[k];
      if (s > 1) __syncthreads();
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        int o = wo;
#pragma unroll
        for (int k = 0; k < kRegBits; ++k)
          if ((r >> k) & 1) o |= rb[k];
        sm[o] = v[r];
      }
      __syncthreads();
      int ro = lane;
#pragma unroll
      for (int k = 0; k < kRegBits; ++k) rb[k] = 1 << cur.reg[k];
#pragma unroll
      for (int k = 0; k < kWarpBits; ++k)
        if ((warp >> k) & 1) ro |= 1 << cur.warp[k];
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        int o = ro;
#pragma unroll
        for (int k = 0; k < kRegBits; ++k)
          if ((r >> k) & 1) o |= rb[k];
        v[r] = sm[o];
      }
    }
    for (int o = cur.op_begin; o < cur.op_end;) {
      const uint8_t k0 = ops[o].kind;
      if (RUNS && k0 == TK_RUN) {
        apply_cp_run<R>(v, ops + o, ctx, tid, s_U, s_U + kMaxRunJobs, P.tabs);
        o += 1 + ops[o].slot;   // the header and its entry slots
        continue;
      }
      if (k0 != TK_DIAG && k0 != TK_CP) {
        apply_tile_op<R, G2, REAL>(v, ops + o, tile, lane, warp);
        o += (G2 && k0 == TK_G2) ? 2 : 1;   // a dense two-qubit op spans two entries
        continue;
      }
      DiagRun<R, sizeof(R) == 8 || RUNS> dr;   // live only over the run
      dr.reset();
      uint4 hdr = *reinterpret_cast<const uint4*>(ops + o);
      do {
        if ((hdr.x & 0xffu) == TK_CP) dr.add_cp(v, ops + o, hdr, ctx);
        else dr.add(v, ops + o, tile, lane, warp);
        if (++o >= cur.op_end) break;
        hdr = *reinterpret_cast<const uint4*>(ops + o);
      } while ((hdr.x & 0xffu) == TK_DIAG || (hdr.x & 0xffu) == TK_CP);
      dr.flush(v);
    }
  }
  {
    const TileStage sl = S[nst - 1];
    uint64_t g[kRegBits];
#pragma unroll
    for (int k = 0; k < kRegBits; ++k) g[k] = 1ull << s_pos[sl.reg[k]];
    uint64_t woff = 0;
#pragma unroll
    for (int k = 0; k < kWarpBits; ++k)
      if ((warp >> k) & 1) woff |= 1ull << s_pos[sl.warp[k]];
    C2<R>* __restrict__ dst = psi + (base | loff | woff);
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      uint64_t o = 0;
#pragma unroll
      for (int k = 0; k < kRegBits; ++k)
        if ((r >> k) & 1) o |= g[k];
      dst[o] = v[r];
    }
  }
}

// ------------------------------------------------------------------ adjoint pass
//
// The backward sweep of the adjoint gradient over one tile pass.  With
// lambda = dL/dpsi^* propagated backwards, dL/dt of a gate's parameter is
// 2 Re <lambda_g | dU/dt | psi_{g-1}> = 2 Re <lambda_g | G psi_g> with
// G = (dU/dt) U^dagger, psi_g and lambda_g the states after the gate.  The host
// lists, from the last gate, runs of one-qubit gates on a qubit as one op: the inner
// products of TermRec, from which the derivatives of all the run's parameters
// follow, then the product of the run's U^dagger, applied to both states.  A diagonal
// gate has one op per parameter carrying G (TK_DIAG with term >= 0, not applied) and
// then U^dagger.  The tile planner keeps the order of ops that share a qubit, and a
// term op commutes with the U^dagger of a gate on other qubits (that unitary cancels
// from the inner product).  Here a tile of psi and one of lambda stay in registers
// through the pass; an op's sums over the tile go to s_term (warp sums, shared-memory
// atomics), written per tile to partial[tile][sum].
//
// The FP32 pipe bounds it (24 qubits, 20 layers of three rotations and CZs: 480 runs).  With a
// term op and a U^dagger per gate, three of each per run, and the CZs as diagonals of their own,
// the sweep took 40.1 ms in 11 passes; now 10.1 in 8.

// The sums over this thread's amplitudes that an op of a TermRec takes.
template <typename R>
struct CrossSum {
  R a0 = 0, a1 = 0, re = 0, im = 0;
  __device__ __forceinline__ void pair(C2<R> l0, C2<R> l1, C2<R> p0, C2<R> p1) {
    a0 = fma(l0.x, p0.y, a0);
    a0 = fma(-l0.y, p0.x, a0);
    a1 = fma(l1.x, p1.y, a1);
    a1 = fma(-l1.y, p1.x, a1);
    re = fma(l0.x, p1.x, re);
    re = fma(l0.y, p1.y, re);
    re = fma(-l1.x, p0.x, re);
    re = fma(-l1.y, p0.y, re);
    im = fma(l0.x, p1.y, im);
    im = fma(-l0.y, p1.x, im);
    im = fma(l1.x, p0.y, im);
    im = fma(-l1.y, p0.x, im);
  }
  // one amplitude of a qubit on a lane bit: own l and p, the partner lane's p (to be finished by lane_end)
  __device__ __forceinline__ void single(C2<R> l, C2<R> p, C2<R> q) {
    a0 = fma(l.x, p.y, a0);
    a0 = fma(-l.y, p.x, a0);
    re = fma(l.x, q.x, re);
    re = fma(l.y, q.y, re);
    im = fma(l.x, q.y, im);
    im = fma(-l.y, q.x, im);
  }
  __device__ __forceinline__ void lane_end(bool b) {
    a1 = b ? a0 : R(0);
    a0 = b ? R(0) : a0;
    re = b ? -re : re;
  }
  // adds the warp's sums to dst[0..3]: the four values are spread over lane pairs and quads, then
  // one value per lane (lane & 3) is summed over the lanes
  __device__ __forceinline__ void add_to(R* dst, int lane) const {
    const R z = lanes(lane);
    if (lane < 4) atomicAdd(dst + lane, z);
  }
  __device__ __forceinline__ R lanes(int lane) const {   // the sum lane & 3 of the warp
    const bool o = lane & 1, t = lane & 2;
    const R x = (o ? a1 : a0) + __shfl_xor_sync(0xffffffffu, o ? a0 : a1, 1);
    const R y = (o ? im : re) + __shfl_xor_sync(0xffffffffu, o ? re : im, 1);
    R z = (t ? y : x) + __shfl_xor_sync(0xffffffffu, t ? x : y, 2);
#pragma unroll
    for (int m = 4; m < 32; m <<= 1) z += __shfl_xor_sync(0xffffffffu, z, m);
    return z;
  }
};

template <int J, typename R>
__device__ __forceinline__ void reg_cross(const C2<R>* vp, const C2<R>* vl, CrossSum<R>& s) {
#pragma unroll
  for (int r = 0; r < 16; ++r)
    if (!(r & (1 << J))) s.pair(vl[r], vl[r | (1 << J)], vp[r], vp[r | (1 << J)]);
}

// lane qubit: the sums and the op (own and partner coefficients o0, p0, or o1, p1 where
// register bit K is 1; K < 0: one pair) on both states, psi's partner amplitudes fetched once
template <int K, typename R>
__device__ __forceinline__ void lane_cross(C2<R>* vp, C2<R>* vl, int mask, C2<R> o0, C2<R> p0, C2<R> o1, C2<R> p1,
                                           CrossSum<R>& s) {
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const C2<R> q = shfl_xor_c(vp[r], mask), k = shfl_xor_c(vl[r], mask);
    s.single(vl[r], vp[r], q);
    const bool one = K >= 0 && ((r >> (K < 0 ? 0 : K)) & 1);
    const C2<R> o = one ? o1 : o0, p = one ? p1 : p0;
    vp[r] = cfma2(o, vp[r], p, q);
    vl[r] = cfma2(o, vl[r], p, k);
  }
}

// a run's op (TK_REG or TK_LANE, term >= 0): its sums to dst, then the op on both states
template <typename R>
__device__ __forceinline__ void apply_run(C2<R>* vp, C2<R>* vl, const TileOp<R>* __restrict__ opp, uint64_t tile,
                                          int lane, int warp, R* dst) {
  CrossSum<R> s;
  if (opp->kind == TK_REG) {
    switch (opp->slot) {
      case 0: reg_cross<0>(vp, vl, s); break;
      case 1: reg_cross<1>(vp, vl, s); break;
      case 2: reg_cross<2>(vp, vl, s); break;
      default: reg_cross<3>(vp, vl, s); break;
    }
    s.add_to(dst, lane);
    apply_tile_op<R, false, false>(vp, opp, tile, lane, warp);
    apply_tile_op<R, false, false>(vl, opp, tile, lane, warp);
    return;
  }
  const int mask = 1 << opp->slot;
  const bool b = (lane & mask) != 0;
  const uint8_t csrc = opp->csrc, cbit = opp->cbit;
  const C2<R> o0 = csel(b, opp->m0[3], opp->m0[0]), p0 = csel(b, opp->m0[2], opp->m0[1]);
  const C2<R> o1 = csel(b, opp->m1[3], opp->m1[0]), p1 = csel(b, opp->m1[2], opp->m1[1]);
  if (csrc == CS_REG) {
    switch (cbit) {
      case 0: lane_cross<0>(vp, vl, mask, o0, p0, o1, p1, s); break;
      case 1: lane_cross<1>(vp, vl, mask, o0, p0, o1, p1, s); break;
      case 2: lane_cross<2>(vp, vl, mask, o0, p0, o1, p1, s); break;
      default: lane_cross<3>(vp, vl, mask, o0, p0, o1, p1, s); break;
    }
  } else {
    const bool c = csrc != CS_NONE && src_bit<R>(csrc, cbit, tile, lane, warp);
    lane_cross<-1>(vp, vl, mask, csel(c, o1, o0), csel(c, p1, p0), o1, p1, s);
  }
  s.lane_end(b);
  s.add_to(dst, lane);
}

// Re sum over this thread's 16 amplitudes of conj(l) (G p), G the diagonal d[2 bit_a + bit_b]
template <typename R>
__device__ __forceinline__ R term_of_diag(const C2<R>* vp, const C2<R>* vl, const TileOp<R>* __restrict__ opp,
                                          uint64_t tile, int lane, int warp) {
  C2<R> g[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) g[i] = opp->m0[i];
  R t = 0;
  auto dotre = [](C2<R> a, C2<R> b) { return fma(a.x, b.x, a.y * b.y); };   // Re conj(a) b
  const uint8_t csrc = opp->csrc, cbit = opp->cbit, dsrc = opp->dsrc, dbit = opp->dbit;
  const bool two = dsrc != CS_NONE;
  const int ua = csrc == CS_REG ? 0 : src_bit<R>(csrc, cbit, tile, lane, warp);
  const int ub = (two && dsrc != CS_REG) ? src_bit<R>(dsrc, dbit, tile, lane, warp) : 0;
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const int ba = csrc == CS_REG ? ((r >> cbit) & 1) : ua;
    const int bb = two ? (dsrc == CS_REG ? ((r >> dbit) & 1) : ub) : 0;
    const int idx = two ? ba * 2 + bb : ba;
    const C2<R> f = csel(idx >= 2, csel(idx == 3, g[3], g[2]), csel(idx == 1, g[1], g[0]));
    t += dotre(vl[r], cmul(f, vp[r]));
  }
  return t;
}

template <typename R, bool G2>
__global__ void __launch_bounds__(kTileThreads, sizeof(R) == 4 ? 2 : 1)
    adjoint_pass_kernel(C2<R>* __restrict__ psi, C2<R>* __restrict__ lam,
                        const __grid_constant__ TileParams<R> P, R* __restrict__ partial, int nsum) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2<R>* smp = reinterpret_cast<C2<R>*>(smem_raw);
  C2<R>* sml = smp + (1 << kTileBits);
  __shared__ R s_term[TileLimits<R>::kMaxOps];   // the state's precision
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint64_t tile = blockIdx.x;

  __shared__ uint8_t s_pos[kTileBits];
  __shared__ uint64_t s_base;
  if (tid == 0) {
    const int n_nt = P.pass.n_nt;
    uint64_t base = 0;
    for (int j = 0; j < n_nt; ++j) base |= ((tile >> j) & 1ull) << P.pass.nt_pos[j];
    s_base = base;
  }
  if (tid < kTileBits) s_pos[tid] = P.pass.pos[tid];
  for (int i = tid; i < nsum; i += kTileThreads) s_term[i] = R(0);
  __syncthreads();
  const uint64_t base = s_base;
  uint64_t loff = 0;
#pragma unroll
  for (int k = 0; k < kLaneBits; ++k)
    if ((lane >> k) & 1) loff |= 1ull << s_pos[k];

  const int nst = P.pass.n_stages;
  const TileStage* __restrict__ S = P.stages;
  const TileOp<R>* __restrict__ ops = P.ops;
  C2<R> vp[16], vl[16];
  {
    const TileStage s0 = S[0];
    uint64_t g[kRegBits];
#pragma unroll
    for (int k = 0; k < kRegBits; ++k) g[k] = 1ull << s_pos[s0.reg[k]];
    uint64_t woff = 0;
#pragma unroll
    for (int k = 0; k < kWarpBits; ++k)
      if ((warp >> k) & 1) woff |= 1ull << s_pos[s0.warp[k]];
    const uint64_t off0 = base | loff | woff;
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      uint64_t o = 0;
#pragma unroll
      for (int k = 0; k < kRegBits; ++k)
        if ((r >> k) & 1) o |= g[k];
      vp[r] = psi[off0 + o];
      vl[r] = lam[off0 + o];
    }
  }
  for (int s = 0; s < nst; ++s) {
    const TileStage cur = S[s];
    if (s > 0) {
      const TileStage prev = S[s - 1];
      int rb[kRegBits];
      int wo = lane;
#pragma unroll
      for (int k = 0; k < kRegBits; ++k) rb[k] = 1 << prev.reg[k];
#pragma unroll
      for (int k = 0; k < kWarpBits; ++k)
        if ((warp >> k) & 1) wo |= 1 << prev.warp[k];
      if (s > 1) __syncthreads();
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        int o = wo;
#pragma unroll
        for (int k = 0; k < kRegBits; ++k)
          if ((r >> k) & 1) o |= rb[k];
        smp[o] = vp[r];
        sml[o] = vl[r];
      }
      __syncthreads();
      int ro = lane;
#pragma unroll
      for (int k = 0; k < kRegBits; ++k) rb[k] = 1 << cur.reg[k];
#pragma unroll
      for (int k = 0; k < kWarpBits; ++k)
        if ((warp >> k) & 1) ro |= 1 << cur.warp[k];
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        int o = ro;
#pragma unroll
        for (int k = 0; k < kRegBits; ++k)
          if ((r >> k) & 1) o |= rb[k];
        vp[r] = smp[o];
        vl[r] = sml[o];
      }
    }
    for (int o = cur.op_begin; o < cur.op_end;) {
      const TileOp<R>* op = ops + o;
      if (op->term >= 0 && op->kind != TK_DIAG) {
        apply_run<R>(vp, vl, op, tile, lane, warp, s_term + op->term);
        ++o;
        continue;
      }
      if (op->term >= 0) {
        R t = term_of_diag<R>(vp, vl, op, tile, lane, warp);
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) t += __shfl_xor_sync(0xffffffffu, t, m);
        if (lane == 0) atomicAdd(&s_term[op->term], t);
        ++o;
        continue;
      }
      if (op->kind != TK_DIAG) {
        apply_tile_op<R, G2, false>(vp, op, tile, lane, warp);
        apply_tile_op<R, G2, false>(vl, op, tile, lane, warp);
        o += (G2 && op->kind == TK_G2) ? 2 : 1;   // a dense two-qubit op spans two entries
        continue;
      }
      DiagRun<R, true> dr;   // a run of diagonal U^dagger ops, on both states
      dr.reset();
      do {
        dr.template add<true>(vp, ops + o, tile, lane, warp, vl);
        ++o;
      } while (o < cur.op_end && ops[o].kind == TK_DIAG && ops[o].term < 0);
      dr.template flush<true>(vp, vl);
    }
  }
  {
    const TileStage sl = S[nst - 1];
    uint64_t g[kRegBits];
#pragma unroll
    for (int k = 0; k < kRegBits; ++k) g[k] = 1ull << s_pos[sl.reg[k]];
    uint64_t woff = 0;
#pragma unroll
    for (int k = 0; k < kWarpBits; ++k)
      if ((warp >> k) & 1) woff |= 1ull << s_pos[sl.warp[k]];
    const uint64_t off0 = base | loff | woff;
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      uint64_t o = 0;
#pragma unroll
      for (int k = 0; k < kRegBits; ++k)
        if ((r >> k) & 1) o |= g[k];
      psi[off0 + o] = vp[r];
      lam[off0 + o] = vl[r];
    }
  }
  __syncthreads();
  for (int i = tid; i < nsum; i += kTileThreads) partial[(size_t)tile * nsum + i] = s_term[i];
}

// the sums of a record over the tiles (FP64, one block per record) and the derivatives they give
template <typename R>
__global__ void __launch_bounds__(256)
    term_reduce_kernel(const R* __restrict__ partial, uint64_t tiles, int nsum, const TermRec* __restrict__ recs,
                       const TermPar* __restrict__ pars, double* __restrict__ dth) {
  const TermRec r = recs[blockIdx.x];
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  for (uint64_t t = threadIdx.x; t < tiles; t += blockDim.x) {
    const R* p = partial + t * nsum + r.sum;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < r.nsum) acc[k] += (double)p[k];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (k < r.nsum) acc[k] = block_sum(acc[k]);
  if (threadIdx.x) return;
  for (int i = r.par; i < r.par + r.npar; ++i) {
    const TermPar& q = pars[i];
    dth[q.slot] += 2.0 * (q.c[0] * acc[0] + q.c[1] * acc[1] + q.c[2] * acc[2] + q.c[3] * acc[3]);
  }
}

// ------------------------------------------------------------------ plain per-gate

template <typename R>
__global__ void plain_g1_kernel(C2<R>* __restrict__ psi, int n, PlainOp<R> op) {
  const uint64_t half = 1ull << (n - 1);
  const int t = op.t;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < half;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t i0 = insert_zero(i, t), i1 = i0 | (1ull << t);
    const C2<R>* m = op.m;
    if (op.type == F_G1C && ((i0 >> op.c) & 1ull)) m = op.m + 4;
    const C2<R> a = psi[i0], b = psi[i1];
    psi[i0] = cfma2(m[0], a, m[1], b);
    psi[i1] = cfma2(m[2], a, m[3], b);
  }
}

template <typename R>
__global__ void plain_diag_kernel(C2<R>* __restrict__ psi, int n, PlainOp<R> op) {
  const uint64_t N = 1ull << n;
  for (uint64_t J = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; J < N;
       J += (uint64_t)gridDim.x * blockDim.x) {
    const int ba = (int)((J >> op.a) & 1ull);
    const int idx = op.b >= 0 ? ba * 2 + (int)((J >> op.b) & 1ull) : ba;
    psi[J] = cmul(psi[J], op.m[idx]);
  }
}

template <typename R>
__global__ void plain_g2_kernel(C2<R>* __restrict__ psi, int n, PlainOp<R> op) {
  const uint64_t quarter = 1ull << (n - 2);
  const int lo = op.a < op.b ? op.a : op.b, hi = op.a < op.b ? op.b : op.a;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < quarter;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t base = insert_zero(insert_zero(i, lo), hi);
    uint64_t idx[4];
    C2<R> a[4];
#pragma unroll
    for (int l = 0; l < 4; ++l) {   // local index 2*bit_a + bit_b
      idx[l] = base | ((uint64_t)(l >> 1) << op.a) | ((uint64_t)(l & 1) << op.b);
      a[l] = psi[idx[l]];
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      C2<R> acc = cfma2(op.m[4 * r + 0], a[0], op.m[4 * r + 1], a[1]);
      const C2<R> acc2 = cfma2(op.m[4 * r + 2], a[2], op.m[4 * r + 3], a[3]);
      acc.x += acc2.x;
      acc.y += acc2.y;
      psi[idx[r]] = acc;
    }
  }
}

// ------------------------------------------------------------------ small states

// A small state: one amplitude per thread, kept in its register through the circuit, on one
// CTA or a cluster of CTAs (amplitude J of thread J mod T of CTA J / T, T threads).  An op on a lane
// bit takes its partner's amplitude by a shuffle, on a warp bit through shared memory, on a CTA bit
// from the other CTA's shared memory.  The ops are staged in shared memory.  Each kind of exchange
// writes two buffers in turn: who writes one again has passed the barrier of the exchange in
// between, which every reader reaches after it has used what it read.
//
// FP64 is bound by the FP64 pipe of the SMs it runs on, so it takes 128 threads on each of as many
// as 8 SMs (20 layers of Haar gates and CNOTs, kernel alone: 10 qubits 466 -> 95 us, 11 qubits
// 854 -> 135, against pairs in one SM's shared memory); FP32 by the latency of an op, so it stays on one SM
// while that holds the state (8 qubits, 47 ops: 34 -> 13.8 us; 11 qubits, 229 ops: 202 -> 72, where
// an op read its matrix from global memory and its pairs from shared memory, with a barrier each).
constexpr int kSmallOps = 256;   // ops staged at a time

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <typename R>
__device__ __forceinline__ C2<R> ld_cluster(const C2<R>* p, uint32_t rank) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(a), "r"(rank));
  C2<R> v;
  if constexpr (sizeof(R) == 8)
    asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
  else
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}

template <typename R>
__global__ void __launch_bounds__(1024)
    small_state_kernel(C2<R>* __restrict__ psi, int n, int tbits, const PlainOp<R>* __restrict__ ops, int nops) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const uint32_t T = 1u << tbits, tid = threadIdx.x;
  C2<R>* xb = reinterpret_cast<C2<R>*>(smem_raw);                 // exchanges in the CTA: 2 x blockDim.x
  C2<R>* cb = xb + 2 * blockDim.x;                                // in the cluster: 2 x blockDim.x
  PlainOp<R>* sop = reinterpret_cast<PlainOp<R>*>(cb + 2 * blockDim.x);
  const bool clustered = n > tbits;
  const uint32_t rank = clustered ? cluster_rank() : 0;
  const uint32_t J = (rank << tbits) | tid;
  const bool live = tid < T;                                      // (fewer than 32 amplitudes)
  C2<R> v{R(0), R(0)};
  if (live) v = psi[J];
  uint32_t xi = 0, ci = 0;                                        // the next buffer of either kind
  // after this the amplitude of J ^ mask is at buf[(tid ^ mask) mod T] of CTA rank ^ (mask / T)
  auto publish = [&](uint32_t mask) -> const C2<R>* {
    if (mask >= T) {
      C2<R>* buf = cb + ci * blockDim.x;
      ci ^= 1;
      buf[tid] = v;
      cluster_barrier();
      return buf;
    }
    C2<R>* buf = xb + xi * blockDim.x;
    xi ^= 1;
    buf[tid] = v;
    __syncthreads();
    return buf;
  };
  auto read = [&](const C2<R>* buf, uint32_t j) -> C2<R> {        // the amplitude of index j
    const uint32_t r = j >> tbits;
    const C2<R>* p = buf + (j & (T - 1));
    return r == rank ? *p : ld_cluster(p, r);
  };
  for (int k0 = 0; k0 < nops; k0 += kSmallOps) {
    const int cnt = min(kSmallOps, nops - k0);
    if (k0) __syncthreads();                                      // the last ones have been read
    const uint4* src = reinterpret_cast<const uint4*>(ops + k0);
    uint4* dst = reinterpret_cast<uint4*>(sop);
    for (uint32_t i = tid; i < cnt * (uint32_t)(sizeof(PlainOp<R>) / 16); i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    for (int k = 0; k < cnt; ++k) {
      const PlainOp<R>* op = sop + k;
      const int type = op->type;
      if (type == F_G1 || type == F_G1C) {
        const uint32_t mask = 1u << op->t;
        const C2<R>* m = op->m;
        if (type == F_G1C && ((J >> op->c) & 1u)) m += 4;
        const C2<R> q = mask < 32u ? shfl_xor_c(v, (int)mask) : read(publish(mask), J ^ mask);
        const bool up = (J & mask) != 0;
        if (up) m += 2;
        v = cfma2(m[0], csel(up, q, v), m[1], csel(up, v, q));
      } else if (type == F_D) {
        const uint32_t ba = (J >> op->a) & 1u;
        v = cmul(v, op->m[op->b >= 0 ? ba * 2 + ((J >> op->b) & 1u) : ba]);
      } else {
        const uint32_t ma = 1u << op->a, mb = 1u << op->b, base = J & ~(ma | mb);
        const C2<R>* buf = publish(ma | mb);
        const C2<R>* m = op->m + 4 * (((J & ma) ? 2 : 0) + ((J & mb) ? 1 : 0));
        // (a thread beyond the state, where there are fewer amplitudes than lanes, works on its own zeros)
        const C2<R> y0 = cfma2(m[0], live ? read(buf, base) : v, m[1], live ? read(buf, base | mb) : v);
        const C2<R> y1 = cfma2(m[2], live ? read(buf, base | ma) : v, m[3], live ? read(buf, base | ma | mb) : v);
        v = C2<R>{y0.x + y1.x, y0.y + y1.y};
      }
    }
  }
  if (live) psi[J] = v;
  if (clustered) cluster_barrier();                               // nobody reads this CTA's buffers any more
}

// The same for a state below a tile on one CTA of 256 threads that finds room on an SM beside a CTA of the
// packed kernel: amplitudes in shared memory, an op at a time (the code of that kernel).
template <typename R>
__global__ void __launch_bounds__(256)
    small_shared_kernel(C2<R>* __restrict__ psi, int n, const PlainOp<R>* __restrict__ ops, int nops) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2<R>* sm = reinterpret_cast<C2<R>*>(smem_raw);
  for (int J = threadIdx.x; J < 1 << n; J += blockDim.x) sm[J] = psi[J];
  __syncthreads();
  small_apply_ops(sm, n, ops, nops);
  for (int J = threadIdx.x; J < 1 << n; J += blockDim.x) psi[J] = sm[J];
}

// The adjoint sweep of a small state: psi and lambda as in small_state_kernel, an amplitude of each
// per thread, through the ops of a run list (PlainOp::pad[0] = 1 + the index of the op's first sum,
// 0: none).  A warp's sums go to partial[warp][sum], in the state's precision within a warp and FP64
// from there, as in the step per gate that it replaces: a launch of ≈ 4 us for each gate, where an
// op here takes ≈ 0.5 us (10 qubits, 12 layers of three rotations and CZs: 5.9 ms a training
// step, now 1.8).
template <typename R>
__global__ void __launch_bounds__(1024)
    adjoint_small_kernel(C2<R>* __restrict__ psi, C2<R>* __restrict__ lam, int n, int tbits,
                         const PlainOp<R>* __restrict__ ops, int nops, double* __restrict__ partial, int nsum) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const uint32_t T = 1u << tbits, tid = threadIdx.x;
  const int lane = (int)(tid & 31u);
  C2<R>* xb = reinterpret_cast<C2<R>*>(smem_raw);                 // exchanges in the CTA: 2 x 2 blockDim.x
  C2<R>* cb = xb + 4 * blockDim.x;                                // in the cluster: 2 x 2 blockDim.x
  PlainOp<R>* sop = reinterpret_cast<PlainOp<R>*>(cb + 4 * blockDim.x);
  const bool clustered = n > tbits;
  const uint32_t rank = clustered ? cluster_rank() : 0;
  const uint32_t J = (rank << tbits) | tid;
  const bool live = tid < T;
  double* const out = partial + (size_t)(rank * (blockDim.x >> 5) + (tid >> 5)) * nsum;
  C2<R> v{R(0), R(0)}, w{R(0), R(0)};
  if (live) {
    v = psi[J];
    w = lam[J];
  }
  uint32_t xi = 0, ci = 0;
  auto publish = [&](uint32_t mask) -> const C2<R>* {             // psi, then lambda blockDim.x further on
    const bool far = mask >= T;
    C2<R>* buf = far ? cb + 2 * ci * blockDim.x : xb + 2 * xi * blockDim.x;
    buf[tid] = v;
    buf[blockDim.x + tid] = w;
    if (far) {
      ci ^= 1;
      cluster_barrier();
    } else {
      xi ^= 1;
      __syncthreads();
    }
    return buf;
  };
  auto read = [&](const C2<R>* buf, uint32_t j) -> C2<R> {
    const uint32_t r = j >> tbits;
    const C2<R>* p = buf + (j & (T - 1));
    return r == rank ? *p : ld_cluster(p, r);
  };
  for (int k0 = 0; k0 < nops; k0 += kSmallOps) {
    const int cnt = min(kSmallOps, nops - k0);
    if (k0) __syncthreads();
    const uint4* src = reinterpret_cast<const uint4*>(ops + k0);
    uint4* dst = reinterpret_cast<uint4*>(sop);
    for (uint32_t i = tid; i < cnt * (uint32_t)(sizeof(PlainOp<R>) / 16); i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    for (int k = 0; k < cnt; ++k) {
      const PlainOp<R>* op = sop + k;
      const int type = op->type, sum = op->pad[0] - 1;
      if (type == F_G1 || type == F_G1C) {
        const uint32_t mask = 1u << op->t;
        const C2<R>* m = op->m;
        if (type == F_G1C && ((J >> op->c) & 1u)) m += 4;
        C2<R> qv, qw;
        if (mask < 32u) {
          qv = shfl_xor_c(v, (int)mask);
          qw = shfl_xor_c(w, (int)mask);
        } else {
          const C2<R>* buf = publish(mask);
          qv = read(buf, J ^ mask);
          qw = read(buf + blockDim.x, J ^ mask);
        }
        const bool up = (J & mask) != 0;
        if (sum >= 0) {
          CrossSum<R> s;
          s.single(w, v, qv);
          s.lane_end(up);
          const R z = s.lanes(lane);
          if (lane < 4) out[sum + lane] = (double)z;
        }
        if (up) m += 2;
        v = cfma2(m[0], csel(up, qv, v), m[1], csel(up, v, qv));
        w = cfma2(m[0], csel(up, qw, w), m[1], csel(up, w, qw));
      } else if (type == F_D) {
        const uint32_t ba = (J >> op->a) & 1u;
        const C2<R> d = op->m[op->b >= 0 ? ba * 2 + ((J >> op->b) & 1u) : ba];
        const C2<R> x = cmul(d, v);
        if (sum >= 0) {   // G on psi, not applied
          R z = fma(w.x, x.x, w.y * x.y);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xffffffffu, z, o);
          if (lane == 0) out[sum] = (double)z;
        } else {
          v = x;
          w = cmul(d, w);
        }
      } else {
        const uint32_t ma = 1u << op->a, mb = 1u << op->b, base = J & ~(ma | mb);
        const C2<R>* buf = publish(ma | mb);
        const C2<R>* m = op->m + 4 * (((J & ma) ? 2 : 0) + ((J & mb) ? 1 : 0));
        auto quad = [&](const C2<R>* b, C2<R> own) {
          const C2<R> y0 = cfma2(m[0], live ? read(b, base) : own, m[1], live ? read(b, base | mb) : own);
          const C2<R> y1 = cfma2(m[2], live ? read(b, base | ma) : own, m[3], live ? read(b, base | ma | mb) : own);
          return C2<R>{y0.x + y1.x, y0.y + y1.y};
        };
        v = quad(buf, v);
        w = quad(buf + blockDim.x, w);
      }
    }
  }
  if (live) {
    psi[J] = v;
    lam[J] = w;
  }
  if (clustered) cluster_barrier();
}

// ------------------------------------------------------------------ remap

__device__ __forceinline__ uint64_t tiles_of(const RemapDesc& d) { return 1ull << d.n_nt; }

template <typename R>
__global__ void __launch_bounds__(kTileThreads, sizeof(R) == 4 ? 3 : 2)
    remap_kernel(C2<R>* __restrict__ psi, const __grid_constant__ RemapDesc D) {
  const RemapDesc* d = &D;   // kernel parameter (constant bank)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C2<R>* sm = reinterpret_cast<C2<R>*>(smem_raw);
  // Every map below is linear over GF(2) in the bits of a 12-bit local index, so
  // each is the XOR of a table entry for the low 6 and one for the high 6 bits:
  //   address  local index -> offset in psi (deposit into the tile positions),
  //   slot     input index -> shared-memory slot (bank swizzle, below),
  //   gather   output index -> slot of the input amplitude it takes.
  // complex64 moves amplitude pairs (local bit 0 = position 0, which every remap
  // holds): one 16-byte global access per pair and one 16-byte shared store, the
  // two gathered amplitudes read separately.  The swizzle adds to every input
  // bit i >= kB a low slot bit, chosen so that the lanes of a wavefront hit
  // distinct banks both when the tile is written in input order and when it is
  // read in output order: kB = 4 bank-pair bits, output bits 1-4 over the lanes
  // of a half-warp (8-byte reads of complex64 pairs); kB = 3, output bits 0-2
  // over a quarter-warp (16-byte complex128 amplitudes).
  constexpr bool kPairs = sizeof(C2<R>) == 8;
  constexpr int kB = kPairs ? 4 : 3, kK0 = kPairs ? 1 : 0;
  __shared__ uint64_t s_alo[64], s_ahi[64];
  __shared__ uint16_t s_slo[64], s_shi[64], s_glo[64], s_ghi[64];
  __shared__ uint16_t s_m[kTileBits];
  const int tid = threadIdx.x;
  // the tile's bits outside the tile positions, deposited at nt_pos
  auto base_of = [&](uint64_t tile) {
    uint64_t base = 0;
    for (int j = 0; j < d->n_nt; ++j) base |= ((tile >> j) & 1ull) << d->nt_pos[j];
    return base;
  };
  if (tid == 0) {
    int used = 0;
    for (int k = kK0; k < kK0 + kB; ++k)
      if (d->src[k] < kB) used |= 1 << d->src[k];
    for (int i = 0; i < kTileBits; ++i) s_m[i] = (uint16_t)(1 << i);
    for (int k = kK0; k < kK0 + kB; ++k) {
      const int sk = d->src[k];
      if (sk < kB) continue;
      const int free_bits = ~used & ((1 << kB) - 1);
      const int j = free_bits & -free_bits;   // lowest unused bank bit
      used |= j;
      s_m[sk] = (uint16_t)(s_m[sk] ^ j);
    }
  }
  __syncthreads();
  if (tid < 128) {
    const int v = tid & 63, h = tid >> 6;   // entry v of the low (h = 0) or high table
    uint64_t a = 0;
    int slot = 0, gather = 0;
    for (int i = 0; i < 6; ++i)
      if ((v >> i) & 1) {
        a |= 1ull << d->pos[6 * h + i];
        slot ^= s_m[6 * h + i];
        gather ^= s_m[d->src[6 * h + i]];
      }
    (h ? s_ahi : s_alo)[v] = a;
    (h ? s_shi : s_slo)[v] = (uint16_t)slot;
    (h ? s_ghi : s_glo)[v] = (uint16_t)gather;
  }
  __syncthreads();
  // Persistent over tiles (grid = a few CTAs per SM): the next tile's loads are
  // issued into registers before the current tile is gathered and stored, so a
  // CTA keeps reads in flight through its exchange and store phases.
  const uint64_t tiles = tiles_of(D);
  uint64_t tile = blockIdx.x;
  if (tile >= tiles) return;
  if (kPairs && d->pos[0] == 0) {
    // slot(L ^ 1) = slot(L) ^ 1: a pair fills one aligned 16-byte slot pair.  A
    // thread's offsets, slots and gathers are the same for every tile: read from
    // the tables once, kept in registers.
    constexpr int kPer = (1 << kTileBits) / (2 * kTileThreads);
    float4* sm4 = reinterpret_cast<float4*>(smem_raw);
    const float* smf = reinterpret_cast<const float*>(smem_raw);
    float4* psi4 = reinterpret_cast<float4*>(psi);
    const int g1 = s_glo[1];   // gather(L ^ 1) = gather(L) ^ g1
    uint64_t ad[kPer];
    int sl[kPer], ga[kPer];
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      const int L = 2 * (tid + r * kTileThreads);
      ad[r] = (s_alo[L & 63] | s_ahi[L >> 6]) >> 1;
      sl[r] = s_slo[L & 63] ^ s_shi[L >> 6];
      ga[r] = s_glo[L & 63] ^ s_ghi[L >> 6];
    }
    uint64_t base = base_of(tile) >> 1;
    float4 q[kPer];
#pragma unroll
    for (int r = 0; r < kPer; ++r) q[r] = __ldcs(psi4 + (base | ad[r]));
    for (;;) {
#pragma unroll
      for (int r = 0; r < kPer; ++r)
        sm4[sl[r] >> 1] = (sl[r] & 1) ? make_float4(q[r].z, q[r].w, q[r].x, q[r].y) : q[r];
      __syncthreads();
      const uint64_t next = tile + gridDim.x;
      const uint64_t nbase = next < tiles ? base_of(next) >> 1 : 0;
      if (next < tiles) {
#pragma unroll
        for (int r = 0; r < kPer; ++r) q[r] = __ldcs(psi4 + (nbase | ad[r]));
      }
#pragma unroll
      for (int r = 0; r < kPer; ++r) {
        const float2 a0 = *reinterpret_cast<const float2*>(smf + 2 * ga[r]);
        const float2 a1 = *reinterpret_cast<const float2*>(smf + 2 * (ga[r] ^ g1));
        __stcs(psi4 + (base | ad[r]), make_float4(a0.x, a0.y, a1.x, a1.y));
      }
      if (next >= tiles) return;
      __syncthreads();   // the tile is gathered before the next one is written to shared memory
      tile = next;
      base = nbase;
    }
  }
  constexpr int kPer = (1 << kTileBits) / kTileThreads;
  uint64_t base = base_of(tile);
  C2<R> q[kPer];
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    const int L = tid + r * kTileThreads;
    q[r] = psi[base | s_alo[L & 63] | s_ahi[L >> 6]];
  }
  for (;;) {
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      const int L = tid + r * kTileThreads;
      sm[s_slo[L & 63] ^ s_shi[L >> 6]] = q[r];
    }
    __syncthreads();
    const uint64_t next = tile + gridDim.x;
    const uint64_t nbase = next < tiles ? base_of(next) : 0;
    if (next < tiles) {
#pragma unroll
      for (int r = 0; r < kPer; ++r) {
        const int L = tid + r * kTileThreads;
        q[r] = psi[nbase | s_alo[L & 63] | s_ahi[L >> 6]];
      }
    }
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      const int L = tid + r * kTileThreads;
      psi[base | s_alo[L & 63] | s_ahi[L >> 6]] = sm[s_glo[L & 63] ^ s_ghi[L >> 6]];
    }
    if (next >= tiles) return;
    __syncthreads();
    tile = next;
    base = nbase;
  }
}

// ------------------------------------------------------------------ reductions

// Per-thread sums of probabilities.  For an FP32 state each thread adds the
// probabilities of a chunk of kChunk of its elements in FP32 with Kahan
// compensation (the chunk sum is good to about one FP32 rounding), and only the
// chunk sums go into its FP64 accumulator: GB300's FP64 pipe is far slower
// than its FP32 pipe, and one FP64 add per element made this HBM-bound kernel
// FP64-bound.  The inner loop holds no FP64 instruction (a fold inside it is
// predicated into every iteration).  The reductions across threads and blocks
// are FP64.
constexpr int kChunk = 32;

struct Kahan32 {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float p) {
    const float y = p - c;
    const float t = s + y;
    c = (t - s) - y;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s - (double)c; }
};

template <typename R, typename O>
__global__ void __launch_bounds__(256)
    probs_kernel(const C2<R>* __restrict__ psi, O* __restrict__ out, uint64_t N,
                 double* __restrict__ partials) {
  double acc = 0.0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  if constexpr (sizeof(R) == 8) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < N; i += stride) {
      const C2<R> a = psi[i];
      const R p = a.x * a.x + a.y * a.y;
      if (out) out[i] = (O)p;
      acc += p;
    }
  } else {
    for (uint64_t i0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i0 < N; i0 += stride * kChunk) {
      Kahan32 k;
      for (int j = 0; j < kChunk; ++j) {
        const uint64_t i = i0 + (uint64_t)j * stride;
        if (i < N) {
          const C2<R> a = psi[i];
          const float p = a.x * a.x + a.y * a.y;
          if (out) out[i] = (O)p;
          k.add(p);
        }
      }
      acc += k.value();
    }
  }
  acc = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

// float specialisation: two amplitudes (16 bytes) per load, two floats per store
__global__ void __launch_bounds__(256)
    probs_kernel_f32x2(const float4* __restrict__ psi2, float2* __restrict__ out2, uint64_t N2,
                       double* __restrict__ partials) {
  double acc = 0.0;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  constexpr int kBatch = 8;   // loads in flight per thread
  for (uint64_t i0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i0 < N2; i0 += stride * kChunk) {
    Kahan32 k;
#pragma unroll
    for (int jb = 0; jb < kChunk; jb += kBatch) {
      float4 a[kBatch];
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const uint64_t i = i0 + (uint64_t)(jb + u) * stride;
        a[u] = i < N2 ? __ldcs(psi2 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < kBatch; ++u) {
        const uint64_t i = i0 + (uint64_t)(jb + u) * stride;
        float2 p;
        p.x = a[u].x * a[u].x + a[u].y * a[u].y;
        p.y = a[u].z * a[u].z + a[u].w * a[u].w;
        if (out2 && i < N2) __stcs(out2 + i, p);
        k.add(p.x);
        k.add(p.y);
      }
    }
    acc += k.value();
  }
  acc = block_sum(acc);
  if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

// A sum of FP32 numbers in three FP32 parts: an addition is split exactly into its rounded sum and its
// remainder (Knuth), the remainders are added in the same way, and only the sum of their remainders rounds,
// below FP64's unit.  (With the remainders summed plainly, 31 probabilities of 2^-25 beside one of 1 were off by
// up to 2^-42.)  An FP64 addition per number instead: 1.14 ms for the marginals below.
struct Sum32 {
  float s = 0.f, e = 0.f, f = 0.f;
  // a + b rounded; r: what that left out
  __device__ __forceinline__ static float two_sum(float a, float b, float& r) {
    const float t = a + b, v = t - a;
    r = (a - (t - v)) + (b - v);
    return t;
  }
  __device__ __forceinline__ void add(float p) {
    float r, q;
    s = two_sum(s, p, r);
    e = two_sum(e, r, q);
    f += q;
  }
  __device__ __forceinline__ bool finite() const { return fabsf(s) <= 3.402823466e38f; }
  __device__ __forceinline__ double value() const { return (double)s + ((double)e + (double)f); }
};

// Marginal over the bits of a mask.  A warp reads lines of 32 amplitudes (address bits 0..4)
// whose mask bits above are fixed, over a part of the remaining bits, so a lane's
// probabilities all go to one outcome: they are summed in registers (FP32 states in three FP32
// parts in chunks, then FP64; a chunk that leaves FP32's range is summed again in FP64), across the lanes
// whose mask bits agree, and added to the outcome once.  HBM bounds it.  One shared-memory FP64
// atomic per amplitude before: 28 qubits FP32, 10 low bits 1.86 ms, 10 high ones 18.9 ms; now
// 0.40 ms (0.61 when a batch was loaded after the last had been summed; reading 2 GiB at the copy rate: 0.32 ms).
struct MargPlan {
  uint8_t hi_pos[32];       // mask positions from 5 on, ascending
  int32_t n_hi, k_lo;       // of them; mask positions below 5
  uint32_t lane_mask;       // mask bits among the lane bits
  uint64_t rest;            // positions from 5 on outside the mask
  int32_t n_rest, chunk;    // of them; log2 of the lines of one unit
};
template <typename R>
__global__ void __launch_bounds__(256)
    marginal_kernel(const C2<R>* __restrict__ psi, int n, const __grid_constant__ MargPlan P,
                    double* __restrict__ acc_out, double* __restrict__ partials) {
  const int lane = threadIdx.x & 31;
  const bool live = n >= 5 || lane < (1 << n);
  const uint64_t units = 1ull << (P.n_hi + P.n_rest - P.chunk);
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x >> 5);
  uint32_t K_lo = 0;
  for (int b = 0, k = 0; b < 5; ++b)
    if ((P.lane_mask >> b) & 1u) K_lo |= (uint32_t)((lane >> b) & 1) << k++;
  double tot = 0.0;
  for (uint64_t u = (uint64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < units; u += warps) {
    const uint64_t K_hi = u & ((1ull << P.n_hi) - 1);
    uint64_t fixed = 0, a = 0;
    for (int b = 0; b < P.n_hi; ++b) fixed |= ((K_hi >> b) & 1ull) << P.hi_pos[b];
    {   // line number (u >> n_hi) << chunk of the rest, spread over its positions
      uint64_t r = (u >> P.n_hi) << P.chunk;
      for (uint64_t m = P.rest; m && r; m &= m - 1, r >>= 1)
        if (r & 1ull) a |= m & (~m + 1);
    }
    constexpr int kBatch = sizeof(R) == 8 ? 4 : 8;   // loads in flight
    const uint64_t lines = 1ull << P.chunk;
    double acc = 0.0;
    for (uint64_t r0 = 0; r0 < lines; r0 += kChunk) {
      const int cnt = (int)(lines - r0 < (uint64_t)kChunk ? lines - r0 : (uint64_t)kChunk);
      const uint64_t a0 = a;
      Sum32 k;
      C2<R> v[kBatch], nx[kBatch];   // a batch, and the next one on its way
      auto fetch = [&](int rb) {
#pragma unroll
        for (int r = 0; r < kBatch; ++r) {
          nx[r].x = nx[r].y = R(0);
          if (live && rb + r < cnt) nx[r] = psi[(fixed | a) + lane];
          a = ((a | ~P.rest) + 1) & P.rest;   // the next line
        }
      };
      fetch(0);
      for (int rb = 0; rb < cnt; rb += kBatch) {   // cnt: a power of two
#pragma unroll
        for (int r = 0; r < kBatch; ++r) v[r] = nx[r];
        if (rb + kBatch < cnt) fetch(rb + kBatch);
#pragma unroll
        for (int r = 0; r < kBatch; ++r) {
          const R p = v[r].x * v[r].x + v[r].y * v[r].y;
          if constexpr (sizeof(R) == 8) acc += p;
          else k.add(p);
        }
      }
      if constexpr (sizeof(R) == 4) {
        if (k.finite()) {
          acc += k.value();
        } else {
          a = a0;
          for (int r = 0; r < cnt; ++r) {
            const C2<R> v = psi[(fixed | a) + lane];   // not finite: a live lane
            acc += (double)(v.x * v.x + v.y * v.y);
            a = ((a | ~P.rest) + 1) & P.rest;
          }
        }
      }
    }
    tot += acc;
    for (int o = 1; o < 32; o <<= 1)
      if (!(P.lane_mask & (uint32_t)o)) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (live && (lane & ~P.lane_mask) == 0) atomicAdd(acc_out + ((K_hi << P.k_lo) | K_lo), acc);
  }
  tot = block_sum(tot);
  if (threadIdx.x == 0) partials[blockIdx.x] = tot;
}

template <typename O>
__global__ void convert_kernel(const double* __restrict__ in, O* __restrict__ out, uint64_t count) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < count;
       i += (uint64_t)gridDim.x * blockDim.x)
    out[i] = (O)in[i];
}

// sum_J n_J log p_J.  One FP64 logarithm per outcome held the kernel on the FP64 pipe (28 qubits:
// 16.6 ms; HBM: 0.48 ms), one FP64 product per count still did (1.98 ms).  For counts up to kMaxPower
// the terms are multiplied as integers: each thread keeps the product of the p_J^n_J as a 64-bit
// significand and an exponent, n_J products that are cut off at 2^-63 of a term of size 1 (a logarithm
// rounds at 2^-53 of |log p|), two 32-bit multiply-adds each, and takes one logarithm at the end:
// 0.75 ms with eight loads in flight (1.46 with the loads one by one).
constexpr uint32_t kMaxPower = 8;
struct LogProduct {
  double acc = 0.0;
  unsigned long long prod = 1ull << 63;   // the product's significand, prod / 2^63 in [1, 2)
  long long ex = 0;                       // and its exponent
  unsigned long long clamped = 0;
  // p small(): its exponent; its significand times 2^31 (FP32) or 2^63
  __device__ __forceinline__ static int exponent(float p) { return (int)(__float_as_uint(p) >> 23) - 127; }
  __device__ __forceinline__ static int exponent(double p) { return (int)((uint32_t)__double2hiint(p) >> 20) - 1023; }
  __device__ __forceinline__ static uint32_t significand(float p) { return __float_as_uint(p) << 8 | 0x80000000u; }
  __device__ __forceinline__ static unsigned long long significand(double p) {
    return (unsigned long long)__double_as_longlong(p) << 11 | 1ull << 63;
  }
  // Positive, not subnormal, and below 1/2.  An outcome from there on (one at most, of a distribution) takes
  // its logarithm alone: near 1 that is far smaller than the parts of a sum of a significand's and an
  // exponent's (of p = 1 - 1e-10 it had 34 bits).
  __device__ __forceinline__ static bool small(float p) { return (__float_as_uint(p) >> 23) - 1u < 125u; }
  __device__ __forceinline__ static bool small(double p) { return ((uint32_t)__double2hiint(p) >> 20) - 1u < 1021u; }
  // the upper 64 bits of prod * m: 2^62 or more
  __device__ __forceinline__ static unsigned long long high(unsigned long long a, uint32_t m) {
    return (a >> 32) * m + (((a & 0xffffffffull) * m) >> 32);
  }
  __device__ __forceinline__ static unsigned long long high(unsigned long long a, unsigned long long m) {
    return __umul64hi(a, m);
  }
  template <typename R>
  __device__ __forceinline__ void add(R p, uint32_t c) {
    if (c == 0) return;
    if (c <= kMaxPower && small(p)) {
      const auto m = significand(p);
      int e = (int)c * (exponent(p) + 1);
      for (uint32_t k = 0; k < c; ++k) {
        prod = high(prod, m);
        const int up = (long long)prod >= 0;   // below 2^63
        prod <<= up;
        e -= up;
      }
      ex += e;
      return;
    }
    double q = (double)p;
    if (!(q > 0.0)) {
      q = 1e-300;
      ++clamped;
    }
    acc += (double)c * log(q);
  }
  __device__ __forceinline__ double value() const {
    return acc + (log((double)prod * 0x1p-63) + (double)ex * 0.69314718055994530942);
  }
};
template <typename R>
__global__ void __launch_bounds__(256)
    loglik_kernel(const C2<R>* __restrict__ psi, const uint32_t* __restrict__ counts, uint64_t N,
                  double* __restrict__ partials, unsigned long long* __restrict__ clamps) {
  constexpr int kBatch = 8;   // loads in flight per thread
  // a small state takes as many blocks as have a batch for each thread: its logarithm costs more
  const uint64_t blocks = min((uint64_t)gridDim.x, max(N / (kBatch * blockDim.x), (uint64_t)1));
  if (blockIdx.x >= blocks) {
    if (threadIdx.x == 0) partials[blockIdx.x] = 0.0;
    return;
  }
  LogProduct l;
  const uint64_t stride = blocks * blockDim.x;
  uint64_t J = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  for (; J + (kBatch - 1) * stride < N; J += kBatch * stride) {
    C2<R> a[kBatch];
    uint32_t c[kBatch];
#pragma unroll
    for (int k = 0; k < kBatch; ++k) {
      a[k] = psi[J + k * stride];
      c[k] = counts[J + k * stride];
    }
#pragma unroll
    for (int k = 0; k < kBatch; ++k) l.add(a[k].x * a[k].x + a[k].y * a[k].y, c[k]);
  }
  for (; J < N; J += stride) l.add(psi[J].x * psi[J].x + psi[J].y * psi[J].y, counts[J]);
  const double acc = block_sum(l.value());
  if (threadIdx.x == 0) partials[blockIdx.x] = acc;
  if (l.clamped) atomicAdd(clamps, l.clamped);
}

__global__ void reduce_partials_kernel(const double* __restrict__ partials, int count,
                                       double* __restrict__ out) {
  double s = 0.0;
  for (int i = threadIdx.x; i < count; i += blockDim.x) s += partials[i];
  s = block_sum(s);
  if (threadIdx.x == 0) *out = s;
}

template <typename R>
__global__ void set_one_kernel(C2<R>* psi, uint64_t J) {
  C2<R> one;
  one.x = R(1);
  one.y = R(0);
  psi[J] = one;
}

// ------------------------------------------------------------------ launchers

namespace {
int grid_for(uint64_t work, int threads) {
  uint64_t g = (work + threads - 1) / threads;
  const uint64_t cap = 152ull * 16;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return (int)g;
}

template <typename F>
qs_status set_smem(F* f, size_t bytes) {
  if (bytes > 48 * 1024) {
    cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    if (e != cudaSuccess) return cuda_status(e, "cudaFuncSetAttribute");
  }
  return QS_OK;
}
}  // namespace

qs_status launch_set_basis(State* st, uint64_t J) {
  QS_CUDA(cudaMemsetAsync(st->data, 0, st->data_bytes, st->stream));
  if (st->prec == QS_C64) set_one_kernel<float><<<1, 1, 0, st->stream>>>((C2<float>*)st->data, J);
  else set_one_kernel<double><<<1, 1, 0, st->stream>>>((C2<double>*)st->data, J);
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

// does the pass (a host TileParams image) hold a dense two-qubit op?
template <typename R>
static bool pass_has_g2(const TileParams<R>& P) {
  const int nops = P.pass.n_stages > 0 ? P.stages[P.pass.n_stages - 1].op_end : 0;
  for (int o = 0; o < nops; ++o)
    if (P.ops[o].kind == TK_G2) return true;
  return false;
}

// which op kinds a forward pass holds, walking op headers only (a dense
// two-qubit op spans two slots; a TK_RUN header is followed by its entry slots,
// whose bytes are not op headers).  real: whether the code with a path of its own for real
// ops is the faster one.  FP64: always.  FP32: that code holds every complex op up by about a
// tenth, so real ops have to be the most.  25 qubits, kernels of a circuit, us, without / with it: Haar
// gates and CNOTs in equal numbers 6143 / 6866, RX and CNOT 3597 / 3959, Haar and CZ 4085 / 4083 (no
// real op), Hadamards and CNOTs 3649 / 2884, Fourier transform 1196 / 1120.  Beside dense
// two-qubit ops, whose code is large anyway, it wins from the first real op (300 mixed gates 2447 / 2346; SU(4)
// brickwork, none real, 2753 / 2787).
template <typename R>
static void pass_kinds(const TileParams<R>& P, bool* g2, bool* runs, bool* real) {
  *g2 = *runs = false;
  int n_real = 0, n_complex = 0;
  const int nops = P.pass.n_stages > 0 ? P.stages[P.pass.n_stages - 1].op_end : 0;
  for (int o = 0; o < nops;) {
    const uint8_t k = P.ops[o].kind;
    if (k == TK_RUN) {
      *runs = true;
      o += 1 + P.ops[o].slot;
    } else if (k == TK_G2) {
      *g2 = true;
      o += 2;
    } else {
      if (k == TK_REG || k == TK_LANE) ++(P.ops[o].pad[2] ? n_real : n_complex);
      ++o;
    }
  }
  *real = *g2 || n_real > n_complex;
}

template <typename R, bool G2, bool RUNS, bool REAL>
static qs_status tile_launch_t(State* st, const TileParams<R>& P) {
  const uint64_t tiles = 1ull << (st->n - kTileBits);
  const size_t smem = sizeof(C2<R>) << kTileBits;
  qs_status s = set_smem(tile_pass_kernel<R, G2, RUNS, REAL>, smem);
  if (s != QS_OK) return s;
  tile_pass_kernel<R, G2, RUNS, REAL><<<(unsigned)tiles, kTileThreads, smem, st->stream>>>((C2<R>*)st->data, P);
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

template <typename R, bool REAL>
static qs_status tile_launch_any(State* st, const TileParams<R>& P, bool g2, bool runs) {
  if constexpr (REAL)   // (a pass with dense two-qubit ops always takes it)
    if (g2) return runs ? tile_launch_t<R, true, true, REAL>(st, P) : tile_launch_t<R, true, false, REAL>(st, P);
  return runs ? tile_launch_t<R, false, true, REAL>(st, P) : tile_launch_t<R, false, false, REAL>(st, P);
}

qs_status launch_tile_pass(State* st, const void* params) {
  bool g2 = false, runs = false, real = false;
  if (st->prec == QS_C64) {
    const TileParams<float>& P = *(const TileParams<float>*)params;
    pass_kinds(P, &g2, &runs, &real);
    return real ? tile_launch_any<float, true>(st, P, g2, runs) : tile_launch_any<float, false>(st, P, g2, runs);
  }
  const TileParams<double>& P = *(const TileParams<double>*)params;
  pass_kinds(P, &g2, &runs, &real);
  return tile_launch_any<double, true>(st, P, g2, runs);
}

template <typename R, bool G2>
static qs_status adjoint_launch_t(State* st, void* lam, const TileParams<R>& P, void* partial, int nsum) {
  const uint64_t tiles = 1ull << (st->n - kTileBits);
  const size_t smem = 2 * (sizeof(C2<R>) << kTileBits);
  qs_status s = set_smem(adjoint_pass_kernel<R, G2>, smem);
  if (s != QS_OK) return s;
  adjoint_pass_kernel<R, G2><<<(unsigned)tiles, kTileThreads, smem, st->stream>>>(
      (C2<R>*)st->data, (C2<R>*)lam, P, (R*)partial, nsum);
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

qs_status launch_adjoint_pass(State* st, void* lam, const void* params, void* partial, int nsum) {
  if (st->prec == QS_C64) {
    const TileParams<float>& P = *(const TileParams<float>*)params;
    return pass_has_g2(P) ? adjoint_launch_t<float, true>(st, lam, P, partial, nsum)
                          : adjoint_launch_t<float, false>(st, lam, P, partial, nsum);
  }
  const TileParams<double>& P = *(const TileParams<double>*)params;
  return pass_has_g2(P) ? adjoint_launch_t<double, true>(st, lam, P, partial, nsum)
                        : adjoint_launch_t<double, false>(st, lam, P, partial, nsum);
}

qs_status launch_term_reduce(State* st, const void* partial, int nsum, const TermRec* recs, int nrec,
                             const TermPar* pars, double* dth) {
  if (nrec <= 0) return QS_OK;
  const uint64_t tiles = 1ull << (st->n - kTileBits);
  if (st->prec == QS_C64)
    term_reduce_kernel<float><<<nrec, 256, 0, st->stream>>>((const float*)partial, tiles, nsum, recs, pars, dth);
  else
    term_reduce_kernel<double><<<nrec, 256, 0, st->stream>>>((const double*)partial, tiles, nsum, recs, pars, dth);
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

template <typename R>
static qs_status plain_launch_t(State* st, const PlainOp<R>& op) {
  const int n = st->n;
  C2<R>* psi = (C2<R>*)st->data;
  if (op.type == F_G1 || op.type == F_G1C)
    plain_g1_kernel<R><<<grid_for(1ull << (n - 1), 256), 256, 0, st->stream>>>(psi, n, op);
  else if (op.type == F_D)
    plain_diag_kernel<R><<<grid_for(1ull << n, 256), 256, 0, st->stream>>>(psi, n, op);
  else
    plain_g2_kernel<R><<<grid_for(1ull << (n - 2), 256), 256, 0, st->stream>>>(psi, n, op);
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

qs_status launch_plain_op(State* st, const void* op_host, int /*type*/) {
  if (st->prec == QS_C64) return plain_launch_t<float>(st, *(const PlainOp<float>*)op_host);
  return plain_launch_t<double>(st, *(const PlainOp<double>*)op_host);
}

// FP64: 128 threads per SM (one warp on each of its FP64 pipes) on at most 8 SMs, the largest
// portable cluster; FP32: one SM up to 1024 amplitudes
static int small_tbits(const State* st) {
  return st->prec == QS_C128 ? std::max(std::min(st->n, 7), st->n - 3) : std::min(st->n, 10);
}
template <typename... P, typename... A>
static qs_status small_launch(State* st, void (*kernel)(P...), int tbits, size_t smem, A... args) {
  qs_status s = set_smem(kernel, smem);
  if (s != QS_OK) return s;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(1u << (st->n - tbits));
  cfg.blockDim = dim3(1u << std::max(tbits, 5));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cfg.gridDim.x;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  QS_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
  return QS_OK;
}

template <typename R>
static qs_status small_launch_t(State* st, const void* ops_dev, int nops) {
  const int tbits = small_tbits(st);
  const size_t smem =
      4 * sizeof(C2<R>) * (1u << std::max(tbits, 5)) + sizeof(PlainOp<R>) * (size_t)std::min(nops, kSmallOps);
  return small_launch(st, &small_state_kernel<R>, tbits, smem, (C2<R>*)st->data, st->n, tbits,
                      (const PlainOp<R>*)ops_dev, nops);
}

// A cluster waits until as many SMs of one GPC are free as it has CTAs: beside a persistent packed kernel
// (a CTA on each SM it holds, whatever is left there too little for one of 1024 threads) that can last
// until the kernel's end.  It certainly fits while the packed CTAs are fewer than the clusters that fit an empty
// device, one CTA to an SM, or leave more SMs than (cluster - 1) for each of these: some GPC then has
// `cluster` free.  (Every GPC holds a cluster of 8 here; 152 SMs in GPCs of 16 to 20.)
bool small_fits(const State* st) {
  const int held = packed_ctas();
  if (held == 0) return true;
  const int cluster = 1 << (st->n - small_tbits(st));
  int dev = 0, sms = 152, most = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cluster == 1) return held < sms;
  constexpr size_t kWhole = 160 * 1024;   // shared memory that two CTAs cannot have on an SM
  auto clusters = [&](auto kernel) {
    if (set_smem(kernel, kWhole) != QS_OK) return;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cluster);
    cfg.blockDim = dim3(1u << std::max(small_tbits(st), 5));
    cfg.dynamicSmemBytes = kWhole;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&most, kernel, &cfg) != cudaSuccess) {
      cudaGetLastError();
      most = 0;
    }
  };
  if (st->prec == QS_C64) clusters(&small_state_kernel<float>);
  else clusters(&small_state_kernel<double>);
  return held < std::max(most, sms - most * (cluster - 1));
}

int adjoint_small_warps(const State* st) {
  const int tbits = small_tbits(st);
  return (1 << (st->n - tbits)) * (1 << (std::max(tbits, 5) - 5));
}

template <typename R>
static qs_status adjoint_small_launch_t(State* st, void* lam, const void* ops_dev, int nops, double* partial, int nsum) {
  const int tbits = small_tbits(st);
  const size_t smem =
      8 * sizeof(C2<R>) * (1u << std::max(tbits, 5)) + sizeof(PlainOp<R>) * (size_t)std::min(nops, kSmallOps);
  return small_launch(st, &adjoint_small_kernel<R>, tbits, smem, (C2<R>*)st->data, (C2<R>*)lam, st->n, tbits,
                      (const PlainOp<R>*)ops_dev, nops, partial, nsum);
}

qs_status launch_adjoint_small(State* st, void* lam, const void* ops_dev, int nops, double* partial, int nsum,
                               const TermRec* recs, int nrec, const TermPar* pars, double* dth) {
  qs_status s = st->prec == QS_C64 ? adjoint_small_launch_t<float>(st, lam, ops_dev, nops, partial, nsum)
                                   : adjoint_small_launch_t<double>(st, lam, ops_dev, nops, partial, nsum);
  if (s != QS_OK || nrec <= 0) return s;
  term_reduce_kernel<double><<<nrec, 256, 0, st->stream>>>(partial, (uint64_t)adjoint_small_warps(st), nsum, recs, pars, dth);
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

template <typename R>
static qs_status small_shared_launch_t(State* st, const void* ops_dev, int nops) {
  const size_t smem = sizeof(C2<R>) << st->n;
  qs_status s = set_smem(small_shared_kernel<R>, smem);
  if (s != QS_OK) return s;
  small_shared_kernel<R><<<1, 256, smem, st->stream>>>((C2<R>*)st->data, st->n, (const PlainOp<R>*)ops_dev, nops);
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

qs_status launch_small(State* st, const void* ops_dev, int nops) {
  if (!small_fits(st))
    return st->prec == QS_C64 ? small_shared_launch_t<float>(st, ops_dev, nops) : small_shared_launch_t<double>(st, ops_dev, nops);
  return st->prec == QS_C64 ? small_launch_t<float>(st, ops_dev, nops) : small_launch_t<double>(st, ops_dev, nops);
}

qs_status launch_remap(State* st, const RemapDesc& d) {
  const uint64_t tiles = 1ull << (st->n - kTileBits);
  // persistent: as many CTAs as fit on the SMs (shared memory: one tile each)
  auto grid_for = [&](const void* kern, size_t smem) {
    int dev = 0, sms = 152, per = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, kTileThreads, smem);
    const uint64_t g = (uint64_t)sms * (uint64_t)(per < 1 ? 1 : per);
    return (unsigned)(g < tiles ? g : tiles);
  };
  if (st->prec == QS_C64) {
    const size_t smem = sizeof(C2<float>) << kTileBits;
    remap_kernel<float><<<grid_for((const void*)remap_kernel<float>, smem), kTileThreads, smem, st->stream>>>(
        (C2<float>*)st->data, d);
  } else {
    const size_t smem = sizeof(C2<double>) << kTileBits;
    qs_status s = set_smem(remap_kernel<double>, smem);
    if (s != QS_OK) return s;
    remap_kernel<double><<<grid_for((const void*)remap_kernel<double>, smem), kTileThreads, smem, st->stream>>>(
        (C2<double>*)st->data, d);
  }
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

qs_status launch_probs_range(State* st, uint64_t off, uint64_t count, void* out, int out_fp64,
                             double* partials) {
  if (st->prec == QS_C64 && !out_fp64 && (off % 2) == 0 && (count % 2) == 0) {
    probs_kernel_f32x2<<<kReduceBlocks, 256, 0, st->stream>>>((const float4*)((const C2<float>*)st->data + off),
                                                              (float2*)out, count / 2, partials);
  } else if (st->prec == QS_C64) {
    if (out_fp64)
      probs_kernel<float, double><<<kReduceBlocks, 256, 0, st->stream>>>(
          (const C2<float>*)st->data + off, (double*)out, count, partials);
    else
      probs_kernel<float, float><<<kReduceBlocks, 256, 0, st->stream>>>(
          (const C2<float>*)st->data + off, (float*)out, count, partials);
  } else if (out_fp64) {
    probs_kernel<double, double><<<kReduceBlocks, 256, 0, st->stream>>>(
        (const C2<double>*)st->data + off, (double*)out, count, partials);
  } else {
    probs_kernel<double, float><<<kReduceBlocks, 256, 0, st->stream>>>(
        (const C2<double>*)st->data + off, (float*)out, count, partials);
  }
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

qs_status launch_probs(State* st, void* out, int out_fp64, uint64_t mask, double* partials,
                       double* marg_acc) {
  const uint64_t N = 1ull << st->n;
  const uint64_t full = (st->n >= 64) ? ~0ull : ((1ull << st->n) - 1);
  const bool marginal = mask != 0 && (mask & full) != full;
  if (!marginal) {
    if (st->prec == QS_C64 && !out_fp64 && st->n >= 1) {
      probs_kernel_f32x2<<<kReduceBlocks, 256, 0, st->stream>>>((const float4*)st->data,
                                                                (float2*)out, N / 2, partials);
    } else if (st->prec == QS_C64) {
      probs_kernel<float, double><<<kReduceBlocks, 256, 0, st->stream>>>(
          (const C2<float>*)st->data, (double*)out, N, partials);
    } else if (out_fp64) {
      probs_kernel<double, double><<<kReduceBlocks, 256, 0, st->stream>>>(
          (const C2<double>*)st->data, (double*)out, N, partials);
    } else {
      probs_kernel<double, float><<<kReduceBlocks, 256, 0, st->stream>>>(
          (const C2<double>*)st->data, (float*)out, N, partials);
    }
    QS_CUDA(cudaGetLastError());
    return QS_OK;
  }
  // marginal over the bits of mask
  MargPlan P;
  std::memset(&P, 0, sizeof(P));
  int k = 0;
  for (int b = 0; b < st->n; ++b) {
    const bool in = (mask >> b) & 1;
    k += in;
    if (b < 5) {
      P.k_lo += in;
      P.lane_mask |= (uint32_t)in << b;
    } else if (in) {
      P.hi_pos[P.n_hi++] = (uint8_t)b;
    } else {
      P.rest |= 1ull << b;
      ++P.n_rest;
    }
  }
  // units of lines: about one per warp of the grid, of 16 lines at least while there are 256 units
  // (each ends in up to 32 atomic additions)
  const int want = 13 - P.n_hi;   // log2(kReduceBlocks * 8 warps)
  P.chunk = P.n_rest - std::max(0, std::min(P.n_rest, want));
  P.chunk = std::max(P.chunk, std::min({4, P.n_rest, std::max(0, P.n_hi + P.n_rest - 8)}));
  const uint64_t H = 1ull << k;
  QS_CUDA(cudaMemsetAsync(marg_acc, 0, H * sizeof(double), st->stream));
  if (st->prec == QS_C64)
    marginal_kernel<float><<<kReduceBlocks, 256, 0, st->stream>>>((const C2<float>*)st->data, st->n, P, marg_acc, partials);
  else
    marginal_kernel<double><<<kReduceBlocks, 256, 0, st->stream>>>((const C2<double>*)st->data, st->n, P, marg_acc, partials);
  QS_CUDA(cudaGetLastError());
  if (out) {
    if (out_fp64)
      QS_CUDA(cudaMemcpyAsync(out, marg_acc, H * sizeof(double), cudaMemcpyDeviceToDevice, st->stream));
    else {
      convert_kernel<float><<<grid_for(H, 256), 256, 0, st->stream>>>(marg_acc, (float*)out, H);
      QS_CUDA(cudaGetLastError());
    }
  }
  return QS_OK;
}

qs_status launch_reduce_partials(State* st, const double* partials, int count, double* out) {
  reduce_partials_kernel<<<1, 1024, 0, st->stream>>>(partials, count, out);
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

qs_status launch_loglik(State* st, const uint32_t* counts, double* partials,
                        unsigned long long* clamps) {
  const uint64_t N = 1ull << st->n;
  QS_CUDA(cudaMemsetAsync(clamps, 0, sizeof(unsigned long long), st->stream));
  if (st->prec == QS_C64)
    loglik_kernel<float><<<kReduceBlocks, 256, 0, st->stream>>>((const C2<float>*)st->data, counts, N,
                                                                partials, clamps);
  else
    loglik_kernel<double><<<kReduceBlocks, 256, 0, st->stream>>>((const C2<double>*)st->data, counts,
                                                                 N, partials, clamps);
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

}  // namespace qs
