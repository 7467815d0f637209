// Chains of 5-qubit blocks on the tcgen05 tensor cores: one sweep over the state applies
// up to three blocks to each 12-qubit tile.
//
// A block pass that applies one 32x32 unitary per sweep is bound by HBM (87 % of the copy
// bandwidth) with the tensor cores a third busy, so the way to more gates per second is
// fewer sweeps.  A tile of 2^12 amplitudes (physical bits 0..3, so that memory moves as
// 128-byte lines, and any 8 others) holds the light cone of several blocks: the 30-qubit
// circuit of 40 Haar + CZ layers takes 37 passes of 109 blocks, 153 ms,
// instead of 93 sweeps of one block (2.9 ms each) and 3 tile passes, 290 ms.  At 28 qubits a
// pass takes 0.69 ms with one block (HBM: 0.64 ms), 0.82 with two, 0.91 to 1.2 with three.
// Three is where shared memory (tile in and out, rows in and out of every block, B: about 1070
// cycles a block), the tensor cores (24 MMAs of 32 cycles a block) and HBM (2950 cycles a tile)
// come near each other; B of three blocks and five 32 KiB slots also just fill shared memory.
//
// Arithmetic: rows of 32 amplitudes are split into three BF16 parts (exact), the six part products down to 2^-24 are
// accumulated in FP32 in tensor memory.  One accumulator takes them all, the five corrections
// before A_0 B_0: they are added while the sum is small, so only the four steps of A_0 B_0
// round at full size.  The accumulation loses a little magnitude (it truncates); the blocks
// are unitary, so the pass's last epilogue scales the tile back to the squared norm that its
// first producer found (a block at a time and row by row, as in block_tc.cu, costs a tenth of
// the instructions and did not lower the error).
//
// Roles of the persistent CTA (one per SM; 20 warps), over items (tile t, block b).  Two equal
// pipelines take alternate items (chain_group), each with its own operand buffers, accumulator and warps:
//   warps 0-3, 4-7    producers: thread = row = tensor-memory lane; read the row from the
//                     tile's slot, split it, store the parts in tensor memory, a K half (16
//                     columns) at a time
//   warps 17, 19      MMA issuers (one elected lane)
//   warps 8-11, 12-15 epilogues: read the accumulators, write the row to the next slot, in the
//                     next block's layout or (rescaled) the box's
//   warp 16 loads tiles into slots (tensor boxes), warp 18 stores finished tiles (tensor boxes).
// An MMA warp is never more than a few MMAs ahead of the tensor cores, so what it waits
// between two items is lost there unless the other pipeline's MMAs fill it: with one issuer for
// all items they were half idle (1560 cycles an item of 768 cycles of MMAs).
// Items are ordered so that block b of tile t runs one step after block b - 1 of it: step k
// holds (k, 0), (k - 1, 1), (k - 2, 2), so an item's input was finished nblk items earlier.
// A 32 KiB slot is held only while its content waits for a reader: loaded tiles until the
// first producer has read them, the rows between blocks b and b + 1 in a slot of b's from the
// epilogue to the next producer, finished tiles in a slot until the store has read it.
// What bounds it: the chain of hand-offs from one block of a tile to the next (with the work
// of every role cut out they alone take 1090 cycles an item, of 1450 to 1600) and the
// producers' instructions (26 qubits, three blocks: issue slots 55 % busy, tensor pipe 49 %, HBM 46 %).  Three groups of warps that each took a tile through all its
// blocks ran at 2300 cycles an item.
// Every wait is bounded; a role that gives up sets a flag that ends the others' waits, and the
// kernel records QS_ETIMEOUT.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>

#include "chain.h"
#include "tc_ptx.cuh"

namespace qs {

namespace {

constexpr int kThreads = 640;
constexpr int kSlotBytes = 4096 * 8;
// Barriers of a kind are used in turn by the tiles (tile t: t mod kRing, use t / kRing),
// whatever the number of slots, and a role waits for a tile's only after it has passed one of the
// kRing - 1 tiles before (chain_group), so that no role can meet a phase two uses away.
constexpr uint32_t kRing = 4;
constexpr int kWarpLoad = 16, kWarpStore = 18;   // 17 and 19 issue MMAs
// tensor-memory columns: accumulator of pipeline g at 64 g (Re of the 32 outputs, then Im);
// operand A of its items in turn at 128 + 192 g + 96 (turn mod 2), a K half at +48, part p of
// it at +16 p (8 columns of real parts, two per column, then 8 of imaginary): the MMAs of a
// half start as soon as it is stored.
constexpr uint32_t kColA = 128, kHalfCols = 48;

// Dynamic shared memory: the blocks' B operands, then the slots from the next multiple of
// 32 KiB (element addresses are XORs of the slot's address and 15-bit offsets).  With the
// static arrays below (about 2 KiB) and one to three blocks the slots begin at 32 or 64 KiB
// and end at 224 KiB; the kernel checks that they fit.
constexpr int kDynSmem = 224 * 1024;

__device__ __forceinline__ void box_load5(uint32_t dst, const CUtensorMap* map, int c1, int c3, int c4,
                                          uint64_t* b) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, "
      "%4, %5, %6}], [%7];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(c1), "r"(0), "r"(c3), "r"(c4), "r"(smem_u32(b))
      : "memory");
}
__device__ __forceinline__ void box_store5(const CUtensorMap* map, int c1, int c3, int c4, uint32_t src) {
  asm volatile(
      "cp.async.bulk.tensor.5d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4, %5}], [%6];" ::"l"(
          reinterpret_cast<uint64_t>(map)),
      "r"(0), "r"(c1), "r"(0), "r"(c3), "r"(c4), "r"(src)
      : "memory");
}
__device__ __forceinline__ void bulk_wait_read_all() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }

// D (+)= A . B, A in tensor memory
template <bool ACC>
__device__ __forceinline__ void mma_bf16(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "n"(ACC ? 1 : 0));
}
// part product over one K half: the real parts meet B rows 32..95, the imaginary ones 0..63
template <bool FIRST>
__device__ __forceinline__ void mma_product(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc) {
  mma_bf16<!FIRST>(d, a, b + (2048 >> 4), idesc);
  mma_bf16<true>(d, a + 8, b, idesc);
}
// the corrections of one K half, smallest first (the first product overwrites the accumulator)
template <bool FIRST>
__device__ __forceinline__ void mma_corrections(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc) {
  constexpr uint32_t part = kChainPart >> 4;
  mma_product<FIRST>(d, a + 32, b, idesc);
  mma_product<false>(d, a, b + 2 * part, idesc);
  mma_product<false>(d, a + 16, b + part, idesc);
  mma_product<false>(d, a + 16, b, idesc);
  mma_product<false>(d, a, b + part, idesc);
}

// packed FP32x2
__device__ __forceinline__ uint64_t pack2(uint32_t a, uint32_t b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(uint64_t v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float sum8(const uint64_t* p) {
  const float2 v = unpack2(add2(add2(p[0], p[1]), add2(p[2], p[3])));
  return v.x + v.y;
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float2 lds64(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
  return v;
}
// v - b, b a BF16: one instruction, no conversion (mixed-precision fma)
__device__ __forceinline__ float minus_bf16(float v, uint16_t b) {
  float d;
  asm("fma.rn.f32.bf16 %0, %1, %2, %3;" : "=f"(d) : "h"(b), "h"((uint16_t)0xbf80), "f"(v));
  return d;
}
__device__ __forceinline__ void sts64(uint32_t a, float x, float y) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(x), "f"(y) : "memory");
}
// bit j of v at position pos[j]
__device__ __forceinline__ uint64_t spread_bits(const uint8_t* pos, int n, uint32_t v) {
  uint64_t a = 0;
  for (int j = 0; j < n; ++j) a |= (uint64_t)((v >> j) & 1u) << pos[j];
  return a;
}
// wait of a warp whose next instructions are warp-collective: one outcome for all lanes
__device__ __forceinline__ bool warp_wait(uint64_t* b, uint32_t parity, int* fail) {
  const bool ok = mbar_wait(b, parity, fail);
  if (__any_sync(0xffffffffu, !ok)) {
    atomicExch(fail, 1);
    return false;
  }
  return true;
}

__global__ void __launch_bounds__(kThreads, 1)
    chain_kernel(const __grid_constant__ ChainPass P, const __grid_constant__ CUtensorMap tmap,
                 const unsigned char* __restrict__ bmat, uint32_t ntiles, int* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[kRing], lread[kRing],             // tile loaded; read by the producers
      mfull[kChainMax - 1][kRing], mread[kChainMax - 1][kRing],           // rows between two blocks
      done[kRing], stored[kRing],                                         // finished; read by the store
      afull[2][2][2], aempty[2][2][2],   // operand halves, by pipeline, turn and half
      dfull[2], dempty[2], nsum[2], drain[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int s_fail;
  __shared__ float s_in[8][4];       // squared norms of loaded tiles, by tile and warp of rows
  __shared__ float s_out[2][2][4];   // squared norms of finished ones, by epilogue group and turn
  __shared__ uint16_t s_rd[kChainMax][128], s_wr[kChainMax][128];   // byte offset of row m, column 0
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int nblk = P.nblk;
  // slots: loads, one between each two blocks, stores
  const uint32_t nload = (uint32_t)P.nload, nstore = (uint32_t)P.nstore;
  const uint32_t S = nload + (uint32_t)nblk - 1u + nstore;
  unsigned char* const bptr = smem_raw + (-smem_u32(smem_raw) & 127u);
  const uint32_t slots = (smem_u32(bptr) + (uint32_t)(nblk * kChainB) + (kSlotBytes - 1u)) & ~(kSlotBytes - 1u);
  if (slots + S * (uint32_t)kSlotBytes > smem_u32(smem_raw) + (uint32_t)kDynSmem) {   // (the same for all threads)
    if (tid == 0) atomicExch(status, (int)QS_EUNSUPPORTED);
    return;
  }

  if (tid == 0) {
    s_fail = 0;
    for (uint32_t s = 0; s < kRing; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&lread[s], 128);
      for (int b = 0; b + 1 < kChainMax; ++b) {
        mbar_init(&mfull[b][s], 128);
        mbar_init(&mread[b][s], 128);
      }
      mbar_init(&done[s], 128);
      mbar_init(&stored[s], 1);
    }
    for (int g = 0; g < 2; ++g) {
      for (int k = 0; k < 4; ++k) {
        mbar_init(&afull[g][k >> 1][k & 1], 128);
        mbar_init(&aempty[g][k >> 1][k & 1], 1);
      }
      mbar_init(&dfull[g], 1);
      mbar_init(&dempty[g], 128);
      mbar_init(&nsum[g], 4);
      mbar_init(&drain[g], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  {
    const uint4* src = reinterpret_cast<const uint4*>(bmat);
    uint4* dst = reinterpret_cast<uint4*>(bptr);
    for (int i = tid; i < nblk * kChainB / 16; i += kThreads) dst[i] = src[i];
  }
  for (int i = tid; i < nblk * 128; i += kThreads) {
    const int b = i >> 7, m = i & 127;
    uint32_t r = 0, w = 0;
    for (int j = 0; j < 7; ++j)
      if ((m >> j) & 1) {
        r ^= P.rd[b].row[j];
        w ^= P.wr[b].row[j];
      }
    s_rd[b][m] = (uint16_t)r;
    s_wr[b][m] = (uint16_t)w;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_slot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // B is read by the MMAs
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  const uint32_t my_tiles = blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;
  const uint32_t steps = my_tiles ? my_tiles + (uint32_t)nblk - 1 : 0;

  if (warp < 8) {
    // ---------------- producers
    const uint32_t grp = (uint32_t)warp >> 2;
    const int m = tid & 127;
    const uint32_t acol = tmem + ((uint32_t)((warp & 3) * 32) << 16) + kColA + 192u * grp;
    uint32_t item = 0;
    bool ok = true;
    for (uint32_t step = 0; step < steps && ok; ++step) {
      for (int b = 0; b < nblk && ok; ++b) {
        if (step - (uint32_t)b >= my_tiles || chain_group(step, nblk, b) != grp) continue;
        const uint32_t it = item++;   // of this pipeline
        const uint32_t t = step - (uint32_t)b, ring = t % kRing, par = (t / kRing) & 1u;
        const uint32_t buf = it & 1u, apar = (it >> 1) & 1u;
        ok = warp_wait(b == 0 ? &full[ring] : &mfull[b - 1][ring], par, &s_fail);
        if (!ok) break;
        const uint32_t slot = b == 0 ? t % nload : nload + (uint32_t)b - 1u;
        // the row: column j at x[j], visited in Gray-code order (one XOR a step)
        float2 x[32];
        const uint32_t cb[5] = {P.rd[b].col[0], P.rd[b].col[1], P.rd[b].col[2], P.rd[b].col[3], P.rd[b].col[4]};
        uint32_t e = slots + slot * (uint32_t)kSlotBytes + s_rd[b][m];
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          if (k) e ^= cb[(k & 1) ? 0 : (k & 2) ? 1 : (k & 4) ? 2 : (k & 8) ? 3 : 4];
          x[k ^ (k >> 1)] = lds64(e);
        }
        if (b == 0) {
          uint64_t nr[4] = {0, 0, 0, 0};
#pragma unroll
          for (int j = 0; j < 32; ++j) {
            const uint64_t v = pack2(__float_as_uint(x[j].x), __float_as_uint(x[j].y));
            nr[j & 3] = fma2(v, v, nr[j & 3]);
          }
          const float nn = warp_sum(sum8(nr));
          if (lane == 0) s_in[t & 7u][warp & 3] = nn;
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {   // columns 16 h .. 16 h + 15
          // the MMAs have read this buffer's previous half
          ok = warp_wait(&aempty[grp][buf][h], apar ^ 1u, &s_fail);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          // each part is rounded from the running residual, which stays exact in FP32
#pragma unroll
          for (int p = 0; p < 3; ++p) {
            uint32_t w[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              float& v0 = j < 8 ? x[16 * h + 2 * j].x : x[16 * h + 2 * j - 16].y;
              float& v1 = j < 8 ? x[16 * h + 2 * j + 1].x : x[16 * h + 2 * j - 15].y;
              w[j] = bf16x2_bits(__floats2bfloat162_rn(v0, v1));
              if (p < 2) {
                v0 = minus_bf16(v0, (uint16_t)w[j]);
                v1 = minus_bf16(v1, (uint16_t)(w[j] >> 16));
              }
            }
            tmem_st16(acol + 96u * buf + kHalfCols * h + 16u * p, w);
          }
          tmem_wait_st();
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          mbar_arrive(&afull[grp][buf][h]);
        }
        // The slot may be overwritten.  Not before the whole row has been used: right after the
        // loads are issued the arrival can overtake them (with bank conflicts a refill did).
        if (ok) mbar_arrive(b == 0 ? &lread[ring] : &mread[b - 1][ring]);
      }
    }
  } else if (warp < 16) {
    // ---------------- epilogues
    const uint32_t grp = (uint32_t)(warp - 8) >> 2;
    const int m = tid & 127;
    const uint32_t d0 = tmem + ((uint32_t)((warp & 3) * 32) << 16) + 64u * grp;
    uint32_t item = 0, turn = 0;
    bool ok = true;
    for (uint32_t step = 0; step < steps && ok; ++step) {
      for (int b = 0; b < nblk && ok; ++b) {
        if (step - (uint32_t)b >= my_tiles || chain_group(step, nblk, b) != grp) continue;
        const uint32_t it = item++;   // of this pipeline
        const uint32_t t = step - (uint32_t)b, ring = t % kRing;
        ok = warp_wait(&dfull[grp], it & 1u, &s_fail);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t re[32], im[32];
        tmem_ld32_nowait(d0, re);
        tmem_ld32_nowait(d0 + 32u, im);
        tmem_wait_ld();
        reg_after_wait32(re);
        reg_after_wait32(im);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(&dempty[grp]);   // the accumulator may be overwritten
        const bool last = b + 1 == nblk;
        float delta = 0.f;
        if (last) {
          uint64_t sq[4] = {0, 0, 0, 0};
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const uint64_t v = pack2(re[2 * j], re[2 * j + 1]), w = pack2(im[2 * j], im[2 * j + 1]);
            sq[j & 1] = fma2(v, v, sq[j & 1]);
            sq[2 + (j & 1)] = fma2(w, w, sq[2 + (j & 1)]);
          }
          const float nn = warp_sum(sum8(sq));
          const uint32_t k = turn & 1u;
          ++turn;
          if (lane == 0) {
            s_out[grp][k][warp & 3] = nn;
            mbar_arrive(&nsum[grp]);
          }
          ok = warp_wait(&nsum[grp], k, &s_fail);
          if (!ok) break;
          // y <- y (1 + delta), 1 + delta = sqrt(nx / ny).  With q = (nx - ny) / ny, delta = q / 2 -
          // q^2 / 8 + ..; beyond |q| = 2^-10 (a tile of subnormal squares, say) the closed form.
          const float* si = s_in[t & 7u];
          const float* so = s_out[grp][k];
          const float ny = (so[0] + so[1]) + (so[2] + so[3]);
          const float diff = ((si[0] - so[0]) + (si[1] - so[1])) + ((si[2] - so[2]) + (si[3] - so[3]));
          // (an infinity or a NaN stays with its row: the tile is then left as the products gave it)
          if (ny > 0.f && fabsf(diff) <= 3.402823466e38f && ny <= 3.402823466e38f) {
            const float q = __fdividef(diff, ny);
            delta = fabsf(q) < 0x1p-10f ? q * fmaf(-0.125f, q, 0.5f)
                                        : diff / (ny + sqrtf(ny) * sqrtf((si[0] + si[1]) + (si[2] + si[3])));
          }
        }
        const uint32_t cb[5] = {P.wr[b].col[0], P.wr[b].col[1], P.wr[b].col[2], P.wr[b].col[3], P.wr[b].col[4]};
        // the slot's previous content has been read
        const uint32_t back = last ? nstore : 1u, old = t - back;
        if (t >= back) {
          ok = warp_wait(last ? &stored[old % kRing] : &mread[b][old % kRing], (old / kRing) & 1u, &s_fail);
          if (!ok) break;
        }
        const uint32_t slot = last ? nload + (uint32_t)nblk - 1u + t % nstore : nload + (uint32_t)b;
        uint32_t e = slots + slot * (uint32_t)kSlotBytes + s_wr[b][m];
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          if (k) e ^= cb[(k & 1) ? 0 : (k & 2) ? 1 : (k & 4) ? 2 : (k & 8) ? 3 : 4];
          const int j = k ^ (k >> 1);
          const float yr = __uint_as_float(re[j]), yi = __uint_as_float(im[j]);
          sts64(e, fmaf(yr, delta, yr), fmaf(yi, delta, yi));
        }
        if (last) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // read by the tensor store
          mbar_arrive(&done[ring]);
        } else {
          mbar_arrive(&mfull[b][ring]);
        }
      }
    }
  } else if (warp == 17 || warp == 19) {
    // ---------------- MMA issuers
    // D = F32, A and B = BF16, both K-major, N = 64, M = 128
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((64u >> 3) << 17) | ((128u >> 4) << 24);
    const uint64_t bdesc = make_desc(smem_u32(bptr), 128, 512);
    const uint32_t grp = warp == 19 ? 1u : 0u;
    const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0), d = tm + 64u * grp;
    uint32_t item = 0;
    bool ok = true;
    for (uint32_t step = 0; step < steps && ok; ++step) {
      for (int b = 0; b < nblk && ok; ++b) {
        if (step - (uint32_t)b >= my_tiles || chain_group(step, nblk, b) != grp) continue;
        const uint32_t it = item++;   // of this pipeline
        const uint32_t buf = it & 1u, apar = (it >> 1) & 1u;
        const uint64_t b0 = bdesc + (uint32_t)(b * (kChainB >> 4)), b1 = b0 + (256 >> 4);
        const uint32_t a0 = tm + kColA + 192u * grp + 96u * buf, a1 = a0 + kHalfCols;
        ok = warp_wait(&dempty[grp], (it & 1u) ^ 1u, &s_fail) && warp_wait(&afull[grp][buf][0], apar, &s_fail);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (elect_one()) mma_corrections<true>(d, a0, b0, idesc);
        __syncwarp();
        ok = warp_wait(&afull[grp][buf][1], apar, &s_fail);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (elect_one()) {
          mma_corrections<false>(d, a1, b1, idesc);
          mma_product<false>(d, a0, b0, idesc);   // A_0 B_0
          mma_commit(smem_u32(&aempty[grp][buf][0]));
          mma_product<false>(d, a1, b1, idesc);
          mma_commit(smem_u32(&aempty[grp][buf][1]));
          mma_commit(smem_u32(&dfull[grp]));
        }
        __syncwarp();
      }
    }
    // every product issued above has finished before the tensor memory is freed (commits track
    // the issuing thread's MMAs: the elected lane is the same each time)
    if (elect_one()) {
      mma_commit(smem_u32(&drain[grp]));
      if (!mbar_wait(&drain[grp], 0, nullptr)) atomicExch(&s_fail, 1);
    }
    __syncwarp();
  } else if (warp == kWarpLoad || warp == kWarpStore) {
    // ---------------- loader / storer: lane q takes copies q, q + 32, ..
    const bool load = warp == kWarpLoad;
    const int ncopy = 1 << P.n_oth;
    const uint32_t copy_bytes = 128u << (P.g1 + P.g2);
    const uint64_t m1 = (1ull << (P.a1 - kChainLow)) - 1, m3 = (1ull << (P.b - P.a1 - P.g1)) - 1;
    const uint64_t outside = spread_bits(P.nt_pos, P.n_nt, 0xffffffffu), stride = spread_bits(P.nt_pos, P.n_nt, gridDim.x);
    uint64_t base = spread_bits(P.nt_pos, P.n_nt, blockIdx.x);
    uint32_t issued = 0;
    for (uint32_t t = 0; t < my_tiles; ++t) {
      const uint32_t ring = t % kRing, old = t - nload;
      if (load ? t >= nload && !warp_wait(&lread[old % kRing], (old / kRing) & 1u, &s_fail)
               : !warp_wait(&done[ring], (t / kRing) & 1u, &s_fail))
        break;
      const uint32_t slot = load ? t % nload : nload + (uint32_t)nblk - 1u + t % nstore;
      if (load) {
        if (lane == 0) mbar_arrive_tx(&full[ring], kSlotBytes);   // before any of the copies
        __syncwarp();
      }
      for (int q = lane; q < ncopy; q += 32) {
        const uint64_t a = base | spread_bits(P.oth_pos, P.n_oth, (uint32_t)q);
        const int c1 = (int)((a >> kChainLow) & m1), c3 = (int)((a >> (P.a1 + P.g1)) & m3), c4 = (int)(a >> P.b);
        const uint32_t sm = slots + slot * (uint32_t)kSlotBytes + (uint32_t)q * copy_bytes;
        if (load) box_load5(sm, &tmap, c1, c3, c4, &full[ring]);
        else box_store5(&tmap, c1, c3, c4, sm);
      }
      issued = t + 1;
      if (!load) {
        bulk_commit();
        bulk_wait_read_all();
        __syncwarp();
        if (lane == 0) mbar_arrive(&stored[ring]);
      }
      base = ((base | ~outside) + stride) & outside;   // the tile number + gridDim.x
    }
    if (load) {
      // no copy may still be writing shared memory when the CTA exits
      if (lane == 0)
        for (uint32_t t = issued > nload ? issued - nload : 0; t < issued; ++t)
          if (!mbar_wait(&full[t % kRing], (t / kRing) & 1u, nullptr)) atomicExch(&s_fail, 1);
    } else {
      bulk_wait_all();
    }
  }
  __syncthreads();
  if (tid == 0 && s_fail) atomicExch(status, (int)QS_ETIMEOUT);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// The state as [16 | bits 4..a1-1 | run1 | bits up to b | run2 and above] amplitudes of 8
// bytes, box [16 | 1 | 2^g1 | 1 | 2^g2].
qs_status chain_tensor_map(const State* st, const ChainPass& P, CUtensorMap* map) {
  static PFN_cuTensorMapEncodeTiled_v12000 encode = [] {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      fn = nullptr;
    return (PFN_cuTensorMapEncodeTiled_v12000)fn;
  }();
  if (!encode) {
    set_error("cuTensorMapEncodeTiled is not available");
    return QS_ECUDA;
  }
  const int n = st->n, e1 = P.a1 + P.g1;
  const cuuint64_t dims[5] = {16, 1ull << (P.a1 - kChainLow), 1ull << P.g1, 1ull << (P.b - e1), 1ull << (n - P.b)};
  const cuuint64_t strides[4] = {128, 8ull << P.a1, 8ull << e1, 8ull << P.b};
  const cuuint32_t box[5] = {16, 1, 1u << P.g1, 1, 1u << P.g2};
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 5, st->data, dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE,
                            P.swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled failed for a block chain (%d)", (int)r);
    return QS_ECUDA;
  }
  return QS_OK;
}

}  // namespace

qs_status launch_chain_setup() {
  QS_CUDA(cudaFuncSetAttribute(chain_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmem));
  return QS_OK;
}

qs_status launch_chain_pass(State* st, const ChainPass& P, const void* b_dev, int* status_dev) {
  CUtensorMap map;
  const qs_status ms = chain_tensor_map(st, P, &map);
  if (ms != QS_OK) return ms;
  const uint64_t ntiles = 1ull << (st->n - 12);
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // one CTA holds all tensor memory of its SM; leave the SMs a server's persistent kernel may hold
  uint64_t grid = (uint64_t)std::max(1, sms - reserved_sms());
  if (grid > ntiles) grid = ntiles;
  chain_kernel<<<(unsigned)grid, kThreads, kDynSmem, st->stream>>>(P, map, (const unsigned char*)b_dev, (uint32_t)ntiles,
                                                               status_dev);
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

}  // namespace qs
