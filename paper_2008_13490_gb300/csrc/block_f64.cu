// Dense 5-qubit blocks of complex128 states on the tcgen05 tensor cores.
//
// FP64 runs at 1/75 of the FP32 rate on this GPU (1.06 TFLOP/s), so a complex128 circuit on
// tile passes is bound by it: 278 ms for 40 Haar + CZ layers at 25 qubits, 0.5 % of HBM.  Here
// the product y = U x of a row of 32 amplitudes is formed in integers instead, exactly but
// for one rounding of the inputs and one of the result (the error-free splitting of matrix products of
// Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59 (2012), with digits on a common exponent):
//   - the 64 real parts of a row become 54-bit integers on the exponent of the row's largest
//     (rounded to nearest; the row's own scale), in six balanced digits: a top one of |d| <= 512
//     and five of 9 bits, |d| <= 256; the block's entries likewise (55 bits, block_f64_plan.cpp);
//   - digits are FP16 integers, so a tcgen05.mma of one digit slice by another sums up to 64
//     products of at most 2^19 in FP32 exactly; slices (i, j) of the same order s = i + j share an
//     accumulator, seven orders s = 0..6 (26 slice products) reach 2^-60 of the row;
//   - the epilogue adds the orders as 64-bit integers and converts once to FP64;
//   - rows whose amplitudes do not share an exponent well, or leave its range, are multiplied in FP64
//     arithmetic instead (row_in_fp64; the bounds are in block_f64.h).
// 25 qubits, 40 layers: 33 ms (81 blocks, 0.37 ms each) against 278 ms.  Error against 112-bit
// arithmetic at 15 qubits, 80 layers: 8.9e-16, against 2.7e-15 of FP64 arithmetic gate by gate.
//
// A persistent CTA (one per SM) takes a tile of 2^12 amplitudes (128 rows) at a time:
//   16 worker warps: thread = a row's quarter (8 amplitudes); read it, agree on the row's
//     exponent, form the digits, store them as operand A in tensor memory; then, while the MMAs
//     of the next quarter of the outputs run, read a quarter's seven accumulators, combine them
//     and write two amplitudes back in place;
//   1 MMA warp: per quarter of the outputs (N = 16) 26 x 4 MMAs into one of two sets of
//     accumulators (7 x 16 columns), so that a set is read while the other is filled;
//   1 warp loads tiles (tensor boxes) into two slots and stores finished ones.
// What bounds it, per tile and SM sub-partition: about 3200 cycles of integer instructions to
// form the digits, then 3800 of MMAs beside 4100 of 64-bit conversions (FP64 pipe); HBM would
// take 6200 a tile at most, overlapped.  Every wait is bounded as in the other block kernels.
#include <cudaTypedefs.h>

#include <algorithm>

#include "block_f64.h"
#include "tc_ptx.cuh"

namespace qs {

namespace {

constexpr int kWorkers = 512;
constexpr int kWarpMma = 16, kWarpTma = 17;
constexpr int kThreads = 576;
constexpr int kSlotBytes = 4096 * 16;
// Dynamic shared memory: B, then the two slots from the next multiple of 64 KiB (addresses are
// XORs of the slot's and 16-bit offsets): 64 .. 192 KiB.  The kernel checks that they fit.
constexpr int kDynSmem = 190 * 1024;
// tensor-memory columns: accumulator set d at 112 d (order s at +16 s), operand A at 224 (digit
// slice i at +32 i: K step j, 8 real then 8 imaginary parts, at +8 j)
constexpr uint32_t kSetCols = 112, kColA = 224;

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

template <bool ACC>
__device__ __forceinline__ void mma_f16(uint32_t d, uint32_t a, uint64_t b, uint32_t idesc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}\n" ::"r"(d),
      "r"(a), "l"(b), "r"(idesc), "n"(ACC ? 1 : 0));
}
__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr), "r"(r[0]), "r"(r[1]),
               "r"(r[2]), "r"(r[3])
               : "memory");
}
__device__ __forceinline__ void tmem_ld4_nowait(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr));
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts128(uint32_t a, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ uint64_t spread_bits(const uint8_t* pos, int n, uint32_t v) {
  uint64_t a = 0;
  for (int j = 0; j < n; ++j) a |= (uint64_t)((v >> j) & 1u) << pos[j];
  return a;
}
__device__ __forceinline__ bool warp_wait(uint64_t* b, uint32_t parity, int* fail) {
  const bool ok = mbar_wait(b, parity, fail);
  if (__any_sync(0xffffffffu, !ok)) {
    atomicExch(fail, 1);
    return false;
  }
  return true;
}

// The digits of a double (words lo, hi) on exponent E (biased, that of the row's largest): the
// integer round(x 2^(1076 - E)) + bias, shifted up by one (the rounding bit): digit i from the
// bottom at bit 1 + 9 i, biased by 256 (512 at the top).
__device__ __forceinline__ uint64_t digits_of(uint32_t lo, uint32_t hi, uint32_t E) {
  const uint32_t e = (hi >> 20) & 0x7ffu;
  uint32_t s = E - e;
  uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 2;
  m = s < 64u ? m >> s : 0ull;   // (x = 0 has e = 0, and E >= kF64MinExp)
  const uint64_t sign = (uint64_t)(int64_t)((int32_t)hi >> 31);
  // bias: 256 in each of the five 9-bit digits, 512 in the top one; plus 1/2 for the rounding
  constexpr uint64_t kBias = 256ull * (1ull + (1ull << 9) + (1ull << 18) + (1ull << 27) + (1ull << 36)) + (512ull << 45);
  return (m ^ sign) - sign + (2 * kBias + 1);
}
// digit i (0 = top) of two numbers as a pair of FP16 integers
template <int I>
__device__ __forceinline__ uint32_t digit_pair(uint64_t a, uint64_t b) {
  constexpr int sh = 1 + 9 * (kF64Slices - 1 - I);
  constexpr uint32_t mask = I == 0 ? 0x7ffu : 0x1ffu;
  // FP16 1024 + u (u up to 1024 at the top: added, not merged)
  const uint32_t u = ((uint32_t)(a >> sh) & mask) + (((uint32_t)(b >> sh) & mask) << 16) + 0x64006400u;
  uint32_t r;
  // - (1024 + bias): -1536 or -1280
  asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(u), "r"(I == 0 ? 0xe600e600u : 0xe500e500u));
  return r;
}

// A row multiplied in FP64 arithmetic, where `mine`: the eight outputs from u on (rows of 32 entries) of
// the row at `row` in shared memory, to columns `first` and on.  Entries that are zero are left out, so that an
// infinity or a NaN goes only where gates take it.  All 128 threads of the row's warps call this.  (Rolled
// loops and a local array: the code around it has no registers to spare.)
__device__ __forceinline__ void row_in_fp64(bool mine, const double2* __restrict__ u, uint32_t row, uint32_t first,
                                            const F64Pass& P, int barrier) {
  double2 y[8];
  if (mine) {
#pragma unroll 1
    for (int r = 0; r < 8; ++r) {
      double re = 0.0, im = 0.0;
      uint32_t e = row;
#pragma unroll 1
      for (int k = 0, c = 0; k < 32; ++k) {   // columns in Gray-code order
        if (k) {
          const int j = __ffs(k) - 1;
          e ^= 16u * P.col[j];
          c ^= 1 << j;
        }
        const uint4 v = lds128(e);
        const double xr = __hiloint2double((int)v.y, (int)v.x), xi = __hiloint2double((int)v.w, (int)v.z);
        const double2 m = u[32 * r + c];
        if (m.x != 0.0) {
          re = fma(m.x, xr, re);
          im = fma(m.x, xi, im);
        }
        if (m.y != 0.0) {
          re = fma(-m.y, xi, re);
          im = fma(m.y, xr, im);
        }
      }
      y[r] = make_double2(re, im);
    }
  }
  __syncwarp();
  bar_sync(barrier, 128);
#pragma unroll 1
  for (int r = 0; mine && r < 8; ++r) {
    const uint32_t e = row ^ first ^ 16u * ((r & 1 ? P.col[0] : 0u) ^ (r & 2 ? P.col[1] : 0u) ^ (r & 4 ? P.col[2] : 0u));
    const double2 v = y[r];
    sts128(e, make_uint4((uint32_t)__double2loint(v.x), (uint32_t)__double2hiint(v.x), (uint32_t)__double2loint(v.y),
                         (uint32_t)__double2hiint(v.y)));
  }
  __syncwarp();
}

__global__ void __launch_bounds__(kThreads, 1)
    block_f64_kernel(const __grid_constant__ F64Pass P, const __grid_constant__ CUtensorMap tmap,
                     const unsigned char* __restrict__ bmat, uint32_t ntiles, int* __restrict__ status) {
  const double2* __restrict__ umat = reinterpret_cast<const double2*>(bmat + kF64B);   // the block in FP64
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[2], done[2], afull, dfull[2], dempty[2], drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_fail;
  __shared__ uint32_t s_exp[4][128];   // by quarter and row: exponents of the largest and smallest amplitude
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const uint32_t bsm = smem_u32(smem_raw);
  const uint32_t slots = (bsm + (uint32_t)kF64B + (kSlotBytes - 1u)) & ~(kSlotBytes - 1u);
  if (slots + 2u * kSlotBytes > bsm + (uint32_t)kDynSmem) {   // (the same for all threads)
    if (tid == 0) *reinterpret_cast<volatile int*>(status) = (int)QS_EUNSUPPORTED;   // (host memory)
    return;
  }
  if (tid == 0) {
    s_fail = 0;
    for (int k = 0; k < 2; ++k) {
      mbar_init(&full[k], 1);
      mbar_init(&done[k], kWorkers);
      mbar_init(&dfull[k], 1);
      mbar_init(&dempty[k], kWorkers);
    }
    mbar_init(&afull, kWorkers);
    mbar_init(&drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  {
    const uint4* src = reinterpret_cast<const uint4*>(bmat);
    uint4* dst = reinterpret_cast<uint4*>(smem_raw);
    for (int i = tid; i < kF64B / 16; i += kThreads) dst[i] = src[i];
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
  const uint32_t tmem = __shfl_sync(0xffffffffu, tmem_slot, 0);
  const uint32_t my_tiles = blockIdx.x < ntiles ? (ntiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;

  if (warp < kWarpMma) {
    // ---------------- workers
    const int m = (warp & 3) * 32 + lane, quarter = warp >> 2;   // row; columns 8 quarter ..
    const uint32_t lanes = tmem + ((uint32_t)((warp & 3) * 32) << 16);
    uint32_t rbase = 0, cq = 0;
    for (int j = 0; j < 7; ++j)
      if ((m >> j) & 1) rbase ^= P.row[j];
    if (quarter & 1) cq ^= P.col[3];
    if (quarter & 2) cq ^= P.col[4];
    uint32_t cb[5];
#pragma unroll
    for (int j = 0; j < 5; ++j) cb[j] = 16u * P.col[j];
    bool alive = true;   // a warp that gave up says so at the next tile's barrier, where all stop
    for (uint32_t i = 0; i < my_tiles; ++i) {
      const uint32_t slot = i & 1u, sbase = slots + slot * (uint32_t)kSlotBytes;
      bool ok = alive && warp_wait(&full[slot], (i >> 1) & 1u, &s_fail);
      uint4 x[8];
      uint32_t top = 0, low = 0xffffffffu;
      if (ok) {
        uint32_t e = sbase + 16u * (rbase ^ cq);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (k) e ^= cb[(k & 1) ? 0 : (k & 2) ? 1 : 2];
          x[k ^ (k >> 1)] = lds128(e);
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const uint32_t a = max(x[k].y & 0x7fffffffu, x[k].w & 0x7fffffffu);
          top = max(top, a);
          low = min(low, a - 1u);   // (zero, and what is below 2^-1042: the largest)
        }
        s_exp[quarter][m] = (top >> 20) << 16 | (0xfffu - (low >> 20));
      }
      ok = !bar_or(1, kWorkers, !ok);
      if (!ok) break;
      const uint32_t ex = __vmaxu2(__vmaxu2(s_exp[0][m], s_exp[1][m]), __vmaxu2(s_exp[2][m], s_exp[3][m]));
      const uint32_t least = 0xfffu - (ex & 0xffffu);   // 0xfff: a row of zeros
      uint32_t E = ex >> 16;
      // rows that the integers do not hold (kF64Spread)
      const bool apart = least != 0xfffu && (E > kF64MaxExp || E < kF64MinExp || E - least > kF64Spread);
      if (apart || least == 0xfffu) E = 2047u + 64u;   // every digit zero: the shift is 64 or more
#pragma unroll
      for (int part = 0; part < 2; ++part) {   // real parts, then imaginary
        uint32_t w[kF64Slices][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint64_t a = part ? digits_of(x[2 * k].z, x[2 * k].w, E) : digits_of(x[2 * k].x, x[2 * k].y, E);
          const uint64_t b = part ? digits_of(x[2 * k + 1].z, x[2 * k + 1].w, E)
                                  : digits_of(x[2 * k + 1].x, x[2 * k + 1].y, E);
          w[0][k] = digit_pair<0>(a, b);
          w[1][k] = digit_pair<1>(a, b);
          w[2][k] = digit_pair<2>(a, b);
          w[3][k] = digit_pair<3>(a, b);
          w[4][k] = digit_pair<4>(a, b);
          w[5][k] = digit_pair<5>(a, b);
        }
#pragma unroll
        for (int s = 0; s < kF64Slices; ++s)
          tmem_st4(lanes + kColA + 32u * s + 8u * (uint32_t)quarter + 4u * part, w[s]);
      }
      tmem_wait_st();
      // Rows apart are read whole before any of the row's four threads writes to it (their warps, w and
      // w + 4 .., agree on whether there are any), and all rows are written after this arrival.
      if (__any_sync(0xffffffffu, apart))
        row_in_fp64(apart, umat + 256 * quarter, sbase + 16u * rbase, 16u * cq, P, 2 + (warp & 3));
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      mbar_arrive(&afull);
      // the outputs, a quarter (8 amplitudes a row) at a time: this thread's are 8 q + 2 quarter
      // and the next
      const uint32_t exp_add = (uint32_t)((int32_t)E - 1024 - P.vs) << 20;
#pragma unroll 1
      for (uint32_t q = 0; q < 4 && ok; ++q) {
        const uint32_t set = q & 1u;
        ok = warp_wait(&dfull[set], (q >> 1) & 1u, &s_fail);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t r[7][4];
#pragma unroll
        for (int s = 0; s < 7; ++s) tmem_ld4_nowait(lanes + kSetCols * set + 16u * s + 4u * (uint32_t)quarter, r[s]);
        tmem_wait_ld();
#pragma unroll
        for (int s = 0; s < 7; ++s)
          asm volatile("" : "+r"(r[s][0]), "+r"(r[s][1]), "+r"(r[s][2]), "+r"(r[s][3]));
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        mbar_arrive(&dempty[set]);
        uint32_t out[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          // sum of D_s 2^(38 - 9 s); the last two orders are below its unit and rounded into it
          const float low = fmaf(__uint_as_float(r[6][k]), 0x1p-16f, __uint_as_float(r[5][k]) * 0x1p-7f);
          long long y = __float2int_rn(low);
          y += (long long)__float2int_rn(__uint_as_float(r[4][k])) * 4;
          y += (long long)__float2int_rn(__uint_as_float(r[3][k])) * 2048;
          y += (long long)__float2int_rn(__uint_as_float(r[2][k])) * (1 << 20);
          y += (long long)__float2int_rn(__uint_as_float(r[1][k])) * (1 << 29);
          y += (long long)((uint64_t)(uint32_t)(__float2int_rn(__uint_as_float(r[0][k])) << 6) << 32);
          const double d = __ll2double_rn(y);
          uint32_t hi = (uint32_t)__double2hiint(d), lo = (uint32_t)__double2loint(d);
          if (hi | lo) hi += exp_add;
          out[2 * k] = lo;
          out[2 * k + 1] = hi;
        }
        // (in place: every row has been read when the first accumulators are full)
        uint32_t c = (q & 1u ? cb[3] : 0u) ^ (q & 2u ? cb[4] : 0u) ^ (quarter & 1 ? cb[1] : 0u) ^ (quarter & 2 ? cb[2] : 0u);
        const uint32_t e = (sbase + 16u * rbase) ^ c;
        if (!apart) {
          sts128(e, make_uint4(out[0], out[1], out[2], out[3]));
          sts128(e ^ cb[0], make_uint4(out[4], out[5], out[6], out[7]));
        }
      }
      alive = ok;
      if (!ok) continue;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // read by the tensor store
      mbar_arrive(&done[slot]);
    }
  } else if (warp == kWarpMma) {
    // ---------------- MMA issuer: D = F32, A and B = F16, both K-major, N = 16, M = 128
    const uint32_t idesc = (1u << 4) | ((16u >> 3) << 17) | ((128u >> 4) << 24);
    const uint64_t bdesc = make_desc(bsm, 128, 1024);
    bool ok = true;
    for (uint32_t i = 0; i < my_tiles && ok; ++i) {
      ok = warp_wait(&afull, i & 1u, &s_fail);
      for (uint32_t q = 0; q < 4 && ok; ++q) {
        const uint32_t set = q & 1u;
        ok = warp_wait(&dempty[set], ((q >> 1) & 1u) ^ 1u, &s_fail);   // two uses a tile
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t d = tmem + kSetCols * set, a = tmem + kColA;
        const uint64_t b = bdesc + q * (2048u >> 4);
        if (elect_one()) {
#pragma unroll
          for (int s = 0; s < 7; ++s) {
#pragma unroll
            for (int ai = s < 6 ? 0 : 1; ai <= (s < 6 ? s : 5); ++ai) {
              const uint32_t aa = a + 32u * ai;
              const uint64_t bb = b + (uint32_t)((s - ai) * (8192 >> 4));
              if (ai == (s < 6 ? 0 : 1)) mma_f16<false>(d + 16u * s, aa, bb, idesc);
              else mma_f16<true>(d + 16u * s, aa, bb, idesc);
#pragma unroll
              for (int ks = 1; ks < 4; ++ks) mma_f16<true>(d + 16u * s, aa + 8u * ks, bb + ks * (256 >> 4), idesc);
            }
          }
          mma_commit(smem_u32(&dfull[set]));
        }
        __syncwarp();
      }
    }
    // every product issued above has finished before the tensor memory is freed
    if (elect_one()) {
      mma_commit(smem_u32(&drain));
      if (!mbar_wait(&drain, 0, nullptr)) atomicExch(&s_fail, 1);
    }
    __syncwarp();
  } else if (warp == kWarpTma) {
    // ---------------- loads and stores: lane q takes copies q, q + 32, ..
    const int ncopy = 1 << P.n_oth;
    const uint32_t copy_bytes = 128u << (P.g1 + P.g2);
    const uint64_t m1 = (1ull << (P.a1 - kF64Low)) - 1, m3 = (1ull << (P.b - P.a1 - P.g1)) - 1;
    uint32_t issued = 0;
    auto move = [&](uint32_t t, bool load) {
      const uint64_t base = spread_bits(P.nt_pos, P.n_nt, blockIdx.x + t * gridDim.x);
      if (load) {
        if (lane == 0) mbar_arrive_tx(&full[t & 1u], kSlotBytes);   // before any of the copies
        __syncwarp();
      }
      for (int q = lane; q < ncopy; q += 32) {
        const uint64_t a = base | spread_bits(P.oth_pos, P.n_oth, (uint32_t)q);
        const int c1 = (int)((a >> kF64Low) & m1), c3 = (int)((a >> (P.a1 + P.g1)) & m3), c4 = (int)(a >> P.b);
        const uint32_t sm = slots + (t & 1u) * (uint32_t)kSlotBytes + (uint32_t)q * copy_bytes;
        if (load) box_load5(sm, &tmap, c1, c3, c4, &full[t & 1u]);
        else box_store5(&tmap, c1, c3, c4, sm);
      }
      if (load) issued = t + 1;
    };
    for (uint32_t t = 0; t < 2 && t < my_tiles; ++t) move(t, true);
    for (uint32_t t = 0; t < my_tiles; ++t) {
      if (!warp_wait(&done[t & 1u], (t >> 1) & 1u, &s_fail)) break;
      move(t, false);
      bulk_commit();
      bulk_wait_read_all();
      __syncwarp();
      if (t + 2 < my_tiles) move(t + 2, true);
    }
    // no copy may still be writing shared memory when the CTA exits
    if (lane == 0)
      for (uint32_t t = issued > 2 ? issued - 2 : 0; t < issued; ++t)
        if (!mbar_wait(&full[t & 1u], (t >> 1) & 1u, nullptr)) atomicExch(&s_fail, 1);
    bulk_wait_all();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0 && s_fail) *reinterpret_cast<volatile int*>(status) = (int)QS_ETIMEOUT;
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// The state as [16 | bits 3..a1-1 | run1 | bits up to b | run2 and above] doubles, box
// [16 | 1 | 2^g1 | 1 | 2^g2].
qs_status f64_tensor_map(const State* st, const F64Pass& P, CUtensorMap* map) {
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
  const cuuint64_t dims[5] = {16, 1ull << (P.a1 - kF64Low), 1ull << P.g1, 1ull << (P.b - e1), 1ull << (n - P.b)};
  const cuuint64_t strides[4] = {128, 16ull << P.a1, 16ull << e1, 16ull << P.b};
  const cuuint32_t box[5] = {16, 1, 1u << P.g1, 1, 1u << P.g2};
  const cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  const CUresult r = encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 5, st->data, dims, strides, box, estr,
                            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled failed for a complex128 block (%d)", (int)r);
    return QS_ECUDA;
  }
  return QS_OK;
}

}  // namespace

qs_status launch_f64_setup() {
  QS_CUDA(cudaFuncSetAttribute(block_f64_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDynSmem));
  return QS_OK;
}

qs_status launch_f64_pass(State* st, const F64Pass& P, const void* b_dev, int* status) {
  CUtensorMap map;
  const qs_status ms = f64_tensor_map(st, P, &map);
  if (ms != QS_OK) return ms;
  const uint64_t ntiles = 1ull << (st->n - 12);
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  uint64_t grid = (uint64_t)std::max(1, sms - reserved_sms());   // (one CTA takes an SM's tensor memory)
  if (grid > ntiles) grid = ntiles;
  block_f64_kernel<<<(unsigned)grid, kThreads, kDynSmem, st->stream>>>(P, map, (const unsigned char*)b_dev,
                                                                       (uint32_t)ntiles, status);
  QS_CUDA(cudaGetLastError());
  return QS_OK;
}

}  // namespace qs
