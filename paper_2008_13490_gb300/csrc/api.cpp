// C ABI entry points of the state-vector path (see include/qsim.h).
#include <algorithm>
#include <array>
#include <cstdarg>
#include <cstdio>
#include <complex>
#include <cstring>
#include <memory>
#include <mutex>
#include <new>
#include <unordered_map>
#include <utility>

#include "abi_guard.h"
#include "auto_plan.h"
#include "block_f64.h"
#include "chain.h"
#include "fuse_merge.h"
#include "host_par.h"
#include "internal.h"
#include "tile_cp.h"

namespace qs {

namespace {
thread_local std::string g_err;
}

void set_error(const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_err = buf;
}

qs_status cuda_status(cudaError_t e, const char* what) {
  set_error("%s: %s", what, cudaGetErrorString(e));
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return QS_ENOMEM;
  }
  return QS_ECUDA;
}

void* dev_alloc(State* st, size_t bytes) {
  if (bytes == 0) bytes = 16;
  if (st->has_alloc) return st->alloc.alloc(bytes, (void*)st->stream, st->alloc.ctx);
  void* p = nullptr;
  if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return p;
}

void dev_free(State* st, void* p, size_t bytes) {
  if (!p) return;
  if (st->has_alloc) st->alloc.free(p, bytes, (void*)st->stream, st->alloc.ctx);
  else cudaFree(p);
}

qs_status ensure_opbuf(State* st, size_t bytes) {
  if (bytes <= st->opbuf_bytes) return QS_OK;
  size_t want = 64 * 1024;
  while (want < bytes) want *= 2;
  // the old buffer may still be read by queued kernels
  QS_CUDA(cudaStreamSynchronize(st->stream));
  dev_free(st, st->opbuf, st->opbuf_bytes);
  st->opbuf = dev_alloc(st, want);
  if (!st->opbuf) {
    st->opbuf_bytes = 0;
    set_error("device allocation of %zu bytes for op descriptors failed", want);
    return QS_ENOMEM;
  }
  st->opbuf_bytes = want;
  return QS_OK;
}

qs_status late_status(State* st) {
  if (!st->late) return QS_OK;
  const int code = *reinterpret_cast<volatile int*>(st->late);
  if (code == 0) return QS_OK;
  *st->late = 0;
  set_error(code == QS_ETIMEOUT ? "complex128 block kernel: bounded wait gave up"
                                : "complex128 block kernel: the tile slots do not fit shared memory");
  return code == QS_ETIMEOUT ? QS_ETIMEOUT : QS_ECUDA;
}

// device buffer and pinned staging of at least `bytes`, the staging free to be written
qs_status reserve_upload(State* st, size_t bytes) {
  qs_status s = ensure_opbuf(st, bytes);
  if (s != QS_OK) return s;
  if (st->hostbuf_bytes < bytes) {
    if (st->hostbuf) {
      QS_CUDA(cudaEventSynchronize(st->upload_done));
      cudaFreeHost(st->hostbuf);
    }
    size_t want = 64 * 1024;
    while (want < bytes) want *= 2;
    if (cudaMallocHost(&st->hostbuf, want) != cudaSuccess) {
      cudaGetLastError();
      st->hostbuf = nullptr;
      st->hostbuf_bytes = 0;
      set_error("pinned host allocation failed");
      return QS_ENOMEM;
    }
    st->hostbuf_bytes = want;
  } else {
    QS_CUDA(cudaEventSynchronize(st->upload_done));   // previous copy has read the buffer
  }
  return QS_OK;
}

// staging of op descriptors: host (pinned) -> device in one copy
qs_status upload(State* st, const std::vector<unsigned char>& blob) {
  if (blob.empty()) return QS_OK;
  const qs_status s = reserve_upload(st, blob.size());
  if (s != QS_OK) return s;
  std::memcpy(st->hostbuf, blob.data(), blob.size());
  QS_CUDA(cudaMemcpyAsync(st->opbuf, st->hostbuf, blob.size(), cudaMemcpyHostToDevice, st->stream));
  QS_CUDA(cudaEventRecord(st->upload_done, st->stream));
  return QS_OK;
}

// The same for operands that the caller writes into the pinned buffer itself: upload_begin
// waits for the buffer and hands it out; upload_part queues the copy of [from, to), the last
// part noted as upload's.
qs_status upload_begin(State* st, size_t bytes, unsigned char** host) {
  const qs_status s = reserve_upload(st, bytes);
  if (s == QS_OK) *host = (unsigned char*)st->hostbuf;
  return s;
}
qs_status upload_part(State* st, size_t from, size_t to, bool last) {
  QS_CUDA(cudaMemcpyAsync((char*)st->opbuf + from, (char*)st->hostbuf + from, to - from, cudaMemcpyHostToDevice,
                          st->stream));
  if (last) QS_CUDA(cudaEventRecord(st->upload_done, st->stream));
  return QS_OK;
}

namespace {

size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

template <typename R>
C2<R> c2(cd z) {
  C2<R> r;
  r.x = (R)z.real();
  r.y = (R)z.imag();
  return r;
}

template <typename R>
PlainOp<R> to_plain(const FOp& o) {
  PlainOp<R> p;
  std::memset(&p, 0, sizeof(p));
  p.type = o.type;
  p.t = o.t;
  p.c = o.c;
  p.a = o.a;
  p.b = o.b;
  switch (o.type) {
    case F_G1:
      for (int i = 0; i < 4; ++i) p.m[i] = c2<R>(o.m0[i]);
      break;
    case F_G1C:
      for (int i = 0; i < 4; ++i) {
        p.m[i] = c2<R>(o.m0[i]);
        p.m[4 + i] = c2<R>(o.m1[i]);
      }
      break;
    case F_D:
      for (int i = 0; i < 4; ++i) p.m[i] = c2<R>(o.d[i]);
      break;
    default:
      for (int i = 0; i < 16; ++i) p.m[i] = c2<R>(o.g[i]);
  }
  return p;
}

template <typename R>
TileOp<R> to_tile(const Plan& pl, size_t i) {
  TileOp<R> t;
  std::memset(&t, 0, sizeof(t));
  const FOp& o = pl.tile_fops[i];
  t.kind = pl.tile_kind[i];
  t.slot = pl.tile_slot[i];
  t.csrc = pl.tile_csrc[i];
  t.cbit = pl.tile_cbit[i];
  t.dsrc = pl.tile_dsrc[i];
  t.dbit = pl.tile_dbit[i];
  if (t.kind == TK_G2 || t.kind == TK_G2C) {   // row-major 4x4: entries 0..7, then 8..15
    // canonical order (the kernel has no other variants): register slots ascending,
    // a lane qubit first; swapping a and b swaps the two bits of the local index
    const bool swap = (t.csrc == CS_REG && t.dsrc == CS_REG && t.cbit > t.dbit) ||
                      (t.csrc == CS_REG && t.dsrc == CS_LANE);
    cd G[16];
    for (int l = 0; l < 4; ++l)
      for (int m = 0; m < 4; ++m) {
        const int ls = swap ? ((l & 1) << 1) | (l >> 1) : l, ms = swap ? ((m & 1) << 1) | (m >> 1) : m;
        G[4 * ls + ms] = o.g[4 * l + m];
      }
    if (swap) {
      std::swap(t.csrc, t.dsrc);
      std::swap(t.cbit, t.dbit);
    }
    const int base = t.kind == TK_G2 ? 0 : 8;
    for (int k = 0; k < 4; ++k) {
      t.m0[k] = c2<R>(G[base + k]);
      t.m1[k] = c2<R>(G[base + 4 + k]);
    }
  } else if (o.type == F_D) {
    for (int k = 0; k < 4; ++k) t.m0[k] = c2<R>(o.d[k]);
  } else {
    for (int k = 0; k < 4; ++k) {
      t.m0[k] = c2<R>(o.m0[k]);
      t.m1[k] = c2<R>(o.type == F_G1C ? o.m1[k] : o.m0[k]);
    }
    bool real = true;
    for (int k = 0; k < 4; ++k) real = real && t.m0[k].y == R(0) && t.m1[k].y == R(0);
    t.pad[2] = real ? 1 : 0;
  }
  return t;
}

// A diagonal whose entries are all exactly 1 but the last (a controlled phase,
// or a one-qubit phase) becomes TK_CP: its phase and the context-word positions
// of its bits (see TK_CP); other ops are returned unchanged.
template <typename R>
TileOp<R> cp_form(TileOp<R> t) {
  if (t.kind != TK_DIAG) return t;
  const bool two = t.dsrc != CS_NONE;
  const int last = two ? 3 : 1;
  for (int k = 0; k < last; ++k)
    if (t.m0[k].x != R(1) || t.m0[k].y != R(0)) return t;
  auto ctx_pos = [](uint8_t src, uint8_t bit) -> int {
    switch (src) {
      case CS_TILE: return bit < kCtxOne ? bit : -1;
      case CS_LANE: return kCtxLane + bit;
      case CS_WARP: return kCtxWarp + bit;
      case CS_REG: return 0;   // (not read)
      default: return -1;
    }
  };
  const int pa = ctx_pos(t.csrc, t.cbit), pb = two ? ctx_pos(t.dsrc, t.dbit) : kCtxOne;
  if (pa < 0 || pb < 0) return t;
  const C2<R> p = t.m0[last];
  t.kind = TK_CP;
  t.m0[0] = p;
  for (int k = 1; k < 4; ++k) t.m0[k] = C2<R>{R(0), R(0)};
  t.pad[0] = (uint8_t)pa;
  t.pad[1] = (uint8_t)pb;
  return t;
}

// the register slot in which every one of the TK_CP ops [i, j) has a bit, or -1
template <typename R>
int common_slot(const std::vector<TileOp<R>>& ops, size_t i, size_t j) {
  for (int k = 0; k < kRegBits; ++k) {
    bool all = true;
    for (size_t o = i; o < j; ++o)
      all = all && ((ops[o].csrc == CS_REG && ops[o].cbit == k) || (ops[o].dsrc == CS_REG && ops[o].dbit == k));
    if (all) return k;
  }
  return -1;
}

// A (lane, warp) table of a run: the product, over the phases whose context bits (kCtxOne, lane and warp
// bits) are all 1, at each of kRunTable indices.  It is multiplicative in the index bits, so it is built by
// doubling, at two products per entry whatever the number of phases (one pass over the table for each phase
// made a third of the planning of a 14-qubit Fourier transform: the pass images of 14, 18 and 22 qubits 77,
// 109 and 175 us, now 37, 58 and 91).
struct PhaseTable {
  static constexpr int kBits = kLaneBits + kWarpBits;
  bool used = false;
  cd one = 1.0, bit[kBits], pair[kBits][kBits];   // pair[a][b]: a < b
  uint32_t bits = 0, pairs[kBits] = {};           // which are there (pairs of b: its a)
  static cd mul(cd x, cd y) {   // (finite factors; std::complex checks for infinities)
    return cd(x.real() * y.real() - x.imag() * y.imag(), x.real() * y.imag() + x.imag() * y.real());
  }
  static int index(int pos) { return pos < kCtxWarp ? pos - kCtxLane : kLaneBits + pos - kCtxWarp; }
  void add(int pa, int pb, cd p) {
    used = true;
    int a = pa == kCtxOne ? -1 : index(pa), b = pb == kCtxOne ? -1 : index(pb);
    if (a > b) std::swap(a, b);
    if (b < 0) {
      one = mul(one, p);
    } else if (a < 0 || a == b) {
      bit[b] = (bits >> b) & 1u ? mul(bit[b], p) : p;
      bits |= 1u << b;
    } else {
      pair[a][b] = (pairs[b] >> a) & 1u ? mul(pair[a][b], p) : p;
      pairs[b] |= 1u << a;
    }
  }
  template <typename R>
  void append(std::vector<C2<R>>& tabs) const {
    cd t[kRunTable], q[kRunTable / 2];
    t[0] = one;
    for (int b = 0; b < kBits; ++b) {
      const int half = 1 << b;
      if (!pairs[b]) {
        for (int x = 0; x < half; ++x) t[half + x] = (bits >> b) & 1u ? mul(t[x], bit[b]) : t[x];
        continue;
      }
      q[0] = (bits >> b) & 1u ? bit[b] : cd(1.0);
      for (int a = 0; a < b; ++a)
        for (int x = 0; x < 1 << a; ++x) q[(1 << a) + x] = (pairs[b] >> a) & 1u ? mul(q[x], pair[a][b]) : q[x];
      for (int x = 0; x < half; ++x) t[half + x] = mul(t[x], q[x]);
    }
    for (const cd& x : t) tabs.push_back(c2<R>(x));
  }
};

// Packs a run [i, j) of TK_CP ops into a TK_RUN header and its entries (see
// tile_cp.h) at out[w..]; returns the next write index.
template <typename R>
int pack_run(const std::vector<TileOp<R>>& ops, size_t i, size_t j, TileOp<R>* out, int w,
             std::vector<C2<R>>& tabs, std::vector<RunJob>& jobs, std::vector<RunJob>& tjobs) {
  // context positions: 0 tile bit (the same for the whole CTA), 1 the constant
  // one, 2 a lane or warp bit
  auto cls = [](int pos) { return pos < kCtxOne ? 0 : (pos == kCtxOne ? 1 : 2); };
  std::vector<RunEntry<R>> res_s, res_f[4], job_s, job_f[4];
  PhaseTable S, N[4];
  std::vector<cd> RR;
  for (size_t o = i; o < j; ++o) {
    const TileOp<R>& t = ops[o];
    RunEntry<R> e;
    std::memset(&e, 0, sizeof(e));
    e.p = t.m0[0];
    const cd p((double)t.m0[0].x, (double)t.m0[0].y);
    const bool ra = t.csrc == CS_REG, rb = t.dsrc == CS_REG;
    if (ra && rb) {
      if (RR.empty()) RR.assign(16, cd(1.0, 0.0));
      for (int r = 0; r < 16; ++r)
        if ((r >> t.cbit) & (r >> t.dbit) & 1) RR[r] *= p;
    } else if (ra || rb) {   // register slot k; the other bit decides
      const int k = ra ? t.cbit : t.dbit, pa = ra ? t.pad[1] : t.pad[0];
      if (cls(pa) != 0) {
        N[k].add(pa, kCtxOne, p);
      } else {
        e.pa = (uint8_t)pa;
        job_f[k].push_back(e);
      }
    } else {
      const int pa = t.pad[0], pb = t.pad[1];
      e.pa = (uint8_t)pa;
      e.pb = (uint8_t)pb;
      if (cls(pa) != 0 && cls(pb) != 0) {
        S.add(pa, pb, p);
      } else if (cls(pa) != 2 && cls(pb) != 2) {
        job_s.push_back(e);
      } else {
        if (cls(pa) == 2) std::swap(e.pa, e.pb);   // pa the tile bit
        res_s.push_back(e);
      }
    }
  }
  // prologue jobs while they fit; the rest go to the per-thread lists
  size_t need = !job_s.empty();
  for (int k = 0; k < 4; ++k) need += !job_f[k].empty();
  const bool fit = jobs.size() + need <= (size_t)kMaxRunJobs;
  if (!fit) {
    res_s.insert(res_s.end(), job_s.begin(), job_s.end());
    job_s.clear();
    for (int k = 0; k < 4; ++k) {
      res_f[k].insert(res_f[k].end(), job_f[k].begin(), job_f[k].end());
      job_f[k].clear();
    }
  }
  // thread jobs: the residual entries by thread bit, where that makes fewer products
  std::stable_sort(res_s.begin(), res_s.end(),
                   [](const RunEntry<R>& x, const RunEntry<R>& y) { return x.pb < y.pb; });
  size_t groups = 0;
  for (size_t e = 0; e < res_s.size(); ++e) groups += e == 0 || res_s[e].pb != res_s[e - 1].pb;
  const bool by_bit = fit && groups < res_s.size() && tjobs.size() + groups <= (size_t)kMaxRunJobs;
  RunHeader rh;
  std::memset(&rh, 0, sizeof(rh));
  rh.n_s = (uint16_t)res_s.size();
  for (int k = 0; k < 4; ++k) rh.n_f[k] = (uint16_t)res_f[k].size();
  rh.ubase = (uint16_t)jobs.size();
  std::vector<RunEntry<R>> all(res_s);
  for (int k = 0; k < 4; ++k) all.insert(all.end(), res_f[k].begin(), res_f[k].end());
  auto add_job = [&](std::vector<RunEntry<R>>& list, bool scalar, int bitno) {
    if (list.empty()) return;
    RunJob jb;
    std::memset(&jb, 0, sizeof(jb));
    jb.op = (uint16_t)w;
    jb.first = (uint16_t)all.size();
    jb.count = (uint16_t)list.size();
    jb.scalar = scalar ? 1 : 0;
    jobs.push_back(jb);
    rh.umask |= (uint8_t)(1u << bitno);
    all.insert(all.end(), list.begin(), list.end());
  };
  rh.wbase = (uint16_t)tjobs.size();
  for (size_t e = 0; by_bit && e < res_s.size();) {
    size_t f = e;
    while (f < res_s.size() && res_s[f].pb == res_s[e].pb) ++f;
    RunJob jb;
    std::memset(&jb, 0, sizeof(jb));
    jb.op = (uint16_t)w;
    jb.first = (uint16_t)e;
    jb.count = (uint16_t)(f - e);
    tjobs.push_back(jb);
    const int pos = res_s[e].pb;
    rh.wmask |= (uint8_t)(1u << (pos < kCtxWarp ? pos - kCtxLane : kLaneBits + pos - kCtxWarp));
    e = f;
  }
  rh.slot = (uint8_t)(1 + common_slot(ops, i, j));
  add_job(job_s, true, 0);
  for (int k = 0; k < 4; ++k) add_job(job_f[k], false, 1 + k);
  rh.toff = (uint32_t)tabs.size();
  auto add_tab = [&](const PhaseTable& t, int bitno) {
    if (!t.used) return;
    rh.tmask |= (uint8_t)(1u << bitno);
    t.append(tabs);
  };
  add_tab(S, 0);
  for (int k = 0; k < 4; ++k) add_tab(N[k], 1 + k);
  if (!RR.empty()) rh.tmask |= 32;
  for (const cd& x : RR) tabs.push_back(c2<R>(x));
  TileOp<R> h;
  std::memset(&h, 0, sizeof(h));
  h.kind = TK_RUN;
  static_assert(sizeof(RunHeader) <= sizeof(h.m0), "run header fits the op's matrix");
  std::memcpy(&h.m0[0], &rh, sizeof(rh));
  const size_t per = sizeof(TileOp<R>) / sizeof(RunEntry<R>);
  const size_t nslots = (all.size() + per - 1) / per;
  h.slot = (uint8_t)nslots;
  out[w++] = h;
  std::vector<TileOp<R>> slots(nslots);
  std::memset(slots.data(), 0, sizeof(TileOp<R>) * nslots);
  if (!all.empty()) std::memcpy((void*)slots.data(), all.data(), sizeof(RunEntry<R>) * all.size());
  for (size_t k = 0; k < nslots; ++k) out[w++] = slots[k];
  return w;
}

// The kernel-parameter image of one forward tile pass: ops converted per
// precision, controlled phases in their TK_CP form, and runs of at least kRunMin
// of them, or of any length where all share a register slot, packed into TK_RUN entry
// lists and tables (at most 255 op slots each, 5 entries per slot for complex64, and
// never more slots than ops); stage op ranges relative to the pass.  tabs
// receives the pass's run tables (offsets relative to its start).
constexpr size_t kRunMin = 3;

// Hadamard gates of a pass: the factors 2^-1/2 are gathered (FP64) and given to the last one, or to
// the one at which they reach kMinScale, and the others become [1 1; 1 -1]: one addition per
// amplitude, which rounds once, and no rounded constant in each.  (Ops are linear; no amplitude
// grows by more than 1 / kMinScale in between.)  30-qubit Fourier transform: 46.1 -> 43.1 ms, error
// against 64 bits 1.2e-6 -> 7.5e-7.  Matrices of that shape whose factor is above 1 or far below it (explicit ones) are
// left alone: their gathered factor could leave the range that the amplitudes keep.
constexpr double kMinScale = 1.0 / 256;
template <typename R>
struct HadamardScale {
  double scale = 1.0;
  TileOp<R>* last = nullptr;   // the latest Hadamard op, its factor in scale
  static bool is(const FOp& o) {
    const double h = o.type == F_G1 ? o.m0[0].real() : 0.0;
    return h >= 0.5 && h <= 1 && o.m0[0] == cd(h) && o.m0[1] == cd(h) && o.m0[2] == cd(h) && o.m0[3] == cd(-h);
  }
  void add(const FOp& o, TileOp<R>* t) {
    if (!is(o)) return;
    scale *= o.m0[0].real();
    last = t;
    for (int k = 0; k < 4; ++k) t->m0[k] = t->m1[k] = C2<R>{k == 3 ? R(-1) : R(1), R(0)};
    t->pad[2] = 2;
    if (scale < kMinScale) flush();
  }
  void flush() {
    if (last && scale != 1.0) {
      for (int k = 0; k < 4; ++k) last->m0[k].x = last->m1[k].x = (R)(k == 3 ? -scale : scale);
      last->pad[2] = 1;
    }
    scale = 1.0;
    last = nullptr;
  }
};

template <typename R>
void build_pass_params(const Plan& pl, const TilePass& pass, TileParams<R>* tp, std::vector<C2<R>>& tabs) {
  std::memset(tp, 0, sizeof(TileParams<R>));
  tp->pass = pass;
  tp->pass.stage_begin = 0;
  tabs.clear();
  std::vector<RunJob> jobs, tjobs;
  int w = 0;
  std::vector<TileOp<R>> conv;
  const size_t per = sizeof(TileOp<R>) / sizeof(RunEntry<R>);
  HadamardScale<R> hs;
  for (int s2 = 0; s2 < pass.n_stages; ++s2) {
    TileStage ts = pl.stages[pass.stage_begin + s2];
    conv.clear();
    for (int o = ts.op_begin; o < ts.op_end; ++o) conv.push_back(cp_form(to_tile<R>(pl, (size_t)o)));
    ts.op_begin = w;
    for (size_t i = 0; i < conv.size();) {
      if (conv[i].kind == TK_CP) {
        size_t j = i;
        while (j < conv.size() && conv[j].kind == TK_CP && j - i < 255 * per) ++j;
        // one op of a register slot and a tile bit would need a header and an entry
        const TileOp<R>& c = conv[i];
        const bool entry = (c.csrc != CS_REG && c.pad[0] < kCtxOne) || (c.dsrc != CS_REG && c.pad[1] < kCtxOne);
        if (j - i >= kRunMin || (common_slot(conv, i, j) >= 0 && (j - i > 1 || !entry))) {
          w = pack_run(conv, i, j, tp->ops, w, tabs, jobs, tjobs);
          i = j;
          continue;
        }
      }
      tp->ops[w] = conv[i];
      if (conv[i].kind == TK_REG || conv[i].kind == TK_LANE)
        hs.add(pl.tile_fops[(size_t)(pl.stages[pass.stage_begin + s2].op_begin) + i], &tp->ops[w]);
      ++w;
      ++i;
    }
    ts.op_end = w;
    tp->stages[s2] = ts;
  }
  hs.flush();
  tp->n_jobs = (int32_t)jobs.size();
  static_assert(sizeof(tp->jobs) >= sizeof(RunJob) * kMaxRunJobs, "job table fits");
  if (!jobs.empty()) std::memcpy(tp->jobs, jobs.data(), sizeof(RunJob) * jobs.size());
  tp->n_tjobs = (int32_t)tjobs.size();
  if (!tjobs.empty()) std::memcpy(tp->tjobs, tjobs.data(), sizeof(RunJob) * tjobs.size());
}

template <typename T>
size_t put(std::vector<unsigned char>& blob, const T* p, size_t count) {
  size_t off = align16(blob.size());
  blob.resize(off + sizeof(T) * count);
  if (count) std::memcpy(blob.data() + off, p, sizeof(T) * count);
  return off;
}

// algorithmic flops per amplitude of a fused op (2 per real FMA of its complex MACs)
double op_flops_per_amp(const FOp& o) {
  switch (o.type) {
    case F_G1: case F_G1C: return 16.0;
    case F_D: return 8.0;
    default: return 32.0;
  }
}

// Process-wide profiling session (qs_profile_begin / qs_profile_end).
struct ProfileSession {
  std::mutex mu;
  bool active = false;
  std::vector<cudaEvent_t> ev;
  std::vector<int> kind;
};
ProfileSession& profile() {
  static ProfileSession p;
  return p;
}

// Optional CUDA-event timing of every launch, by kind (tile, plain, remap, small):
// per call (QS_OPT_TIME_KERNELS) and/or into the profiling session.
struct KernelTimer {
  bool on = false;
  cudaStream_t stream = nullptr;
  std::vector<cudaEvent_t> ev;
  std::vector<int> kind;
  cudaEvent_t prof_start = nullptr;
  void before(int k) {
    ProfileSession& ps = profile();
    if (ps.active) {
      std::lock_guard<std::mutex> g(ps.mu);
      cudaEvent_t a;
      cudaEventCreate(&a);
      cudaEventRecord(a, stream);
      ps.ev.push_back(a);
      ps.ev.push_back(nullptr);
      ps.kind.push_back(k);
      prof_start = a;
    }
    if (!on) return;
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    cudaEventRecord(a, stream);
    ev.push_back(a);
    ev.push_back(b);
    kind.push_back(k);
  }
  void after() {
    ProfileSession& ps = profile();
    if (ps.active && prof_start) {
      std::lock_guard<std::mutex> g(ps.mu);
      cudaEvent_t b;
      cudaEventCreate(&b);
      cudaEventRecord(b, stream);
      for (size_t i = ps.ev.size(); i >= 2; i -= 2)
        if (ps.ev[i - 2] == prof_start) {
          ps.ev[i - 1] = b;
          break;
        }
      prof_start = nullptr;
    }
    if (on) cudaEventRecord(ev.back(), stream);
  }
  void finish(qs_stats* stats) {
    if (!on) return;
    cudaStreamSynchronize(stream);
    for (size_t i = 0; i < kind.size(); ++i) {
      float ms = 0.f;
      cudaEventElapsedTime(&ms, ev[2 * i], ev[2 * i + 1]);
      if (stats) stats->kernel_ms[kind[i]] += ms;
      cudaEventDestroy(ev[2 * i]);
      cudaEventDestroy(ev[2 * i + 1]);
    }
    ev.clear();
    kind.clear();
  }
};

template <typename R>
qs_status run_plain(State* st, const std::vector<FOp>& fops, qs_stats* stats, KernelTimer& tm) {
  double flops = 0.0;
  for (const FOp& o : fops) {
    PlainOp<R> p = to_plain<R>(o);
    tm.before(1);
    qs_status s = launch_plain_op(st, &p, o.type);
    tm.after();
    if (s != QS_OK) return s;
    flops += op_flops_per_amp(o) * std::ldexp(1.0, st->n);
  }
  if (stats) {
    stats->ops_fused = (int64_t)fops.size();
    stats->passes = (int64_t)fops.size();
    stats->launches = (int64_t)fops.size();
    stats->flops = flops;
  }
  return QS_OK;
}

template <typename R>
qs_status run_small(State* st, const std::vector<FOp>& fops, qs_stats* stats, KernelTimer& tm) {
  std::vector<PlainOp<R>> ops;
  ops.reserve(fops.size());
  double flops = 0.0;
  for (const FOp& o : fops) {
    ops.push_back(to_plain<R>(o));
    flops += op_flops_per_amp(o) * std::ldexp(1.0, st->n);
  }
  std::vector<unsigned char> blob;
  size_t off = put(blob, ops.data(), ops.size());
  qs_status s = upload(st, blob);
  if (s != QS_OK) return s;
  tm.before(3);
  s = launch_small(st, (unsigned char*)st->opbuf + off, (int)ops.size());
  tm.after();
  if (s != QS_OK) return s;
  if (stats) {
    stats->ops_fused = (int64_t)fops.size();
    stats->passes = 1;
    stats->launches = 1;
    stats->flops = flops;
    stats->upload_bytes = (int64_t)blob.size();
  }
  return QS_OK;
}

template <typename R>
qs_status run_tiled(State* st, const std::vector<FOp>& fops, const std::vector<int>& vmap,
                    qs_stats* stats, KernelTimer& tm) {
  Plan pl;
  plan_circuit(fops, st->n, vmap, pl, TileLimits<R>::kMaxOps, kMaxTileStages);
  std::vector<unsigned char> blob;
  // every pass's kernel-parameter image first, its run tables into the upload
  // (remap descriptors go by value as kernel parameters)
  std::vector<TileParams<R>> tps;
  std::vector<size_t> tab_off;
  {
    size_t ntile = 0;
    for (const PlanStep& step : pl.steps) ntile += step.kind == PlanStep::TILE;
    tps.resize(ntile);
    std::vector<C2<R>> tabs;
    size_t ti = 0;
    for (const PlanStep& step : pl.steps) {
      if (step.kind != PlanStep::TILE) continue;
      build_pass_params<R>(pl, pl.passes[step.index], &tps[ti++], tabs);
      tab_off.push_back(tabs.empty() ? SIZE_MAX : put(blob, tabs.data(), tabs.size()));
    }
  }
  qs_status s = upload(st, blob);
  if (s != QS_OK) return s;
  unsigned char* dev = (unsigned char*)st->opbuf;
  int64_t passes = 0, launches = 0, tile_launches = 0;
  const double N = std::ldexp(1.0, st->n);
  double tile_flops = 0.0, plain_flops = 0.0;
  for (size_t i = 0; i < pl.tile_fops.size(); ++i)   // a dense two-qubit op has two entries
    if (pl.tile_kind[i] != TK_G2C) tile_flops += op_flops_per_amp(pl.tile_fops[i]) * N;
  size_t ti = 0;
  for (const PlanStep& step : pl.steps) {
    switch (step.kind) {
      case PlanStep::TILE: {
        TileParams<R>& tp = tps[ti];
        tp.tabs = tab_off[ti] == SIZE_MAX ? nullptr : (const C2<R>*)(dev + tab_off[ti]);
        ++ti;
        tm.before(0);
        s = launch_tile_pass(st, &tp);
        ++tile_launches;
        break;
      }
      case PlanStep::PLAIN: {
        PlainOp<R> p = to_plain<R>(pl.plain_fops[step.index]);
        plain_flops += op_flops_per_amp(pl.plain_fops[step.index]) * N;
        tm.before(1);
        s = launch_plain_op(st, &p, p.type);
        break;
      }
      case PlanStep::REMAP:
        tm.before(2);
        s = launch_remap(st, pl.remaps[step.index]);
        break;
      default:
        break;
    }
    tm.after();
    if (s != QS_OK) return s;
    ++passes;
    ++launches;
  }
  if (stats) {
    stats->ops_fused = (int64_t)fops.size();
    stats->passes = passes;
    stats->launches = launches;
    stats->tile_launches = tile_launches;
    stats->tile_flops = tile_flops;
    stats->flops = tile_flops + plain_flops;
    stats->upload_bytes = (int64_t)blob.size();
  }
  return QS_OK;
}

// The gates [g0, g1) backwards as the ops of the adjoint sweep (internal.h, FOp::term).  A run of
// one-qubit gates on a qubit, nothing else on it in between, becomes one op at the place of its last
// gate: the product W of the gates' U^dagger, and the derivatives of all of its parameters as
// combinations of the sums of a TermRec.  (G = (dU/dt) U^dagger of a gate before which the product W'
// is already undone acts as W'^dagger G W' on the states after the run; it is anti-Hermitian as G is.)
// Runs of diagonal gates alone stay diagonals, which need no place in a tile: per gate one op with G
// for each parameter and one with U^dagger.  Diagonals without a term then go into the ops before them.
struct AdjointOps {
  std::vector<FOp> ops;
  std::vector<TermRec> recs;   // sum: filled in per pass
  std::vector<TermPar> pars;
};
qs_status adjoint_ops(const qs_gate* gates, size_t g0, size_t g1, int n, AdjointOps& out) {
  // runs: per gate the run it belongs to; runs that hold a non-diagonal matrix
  std::vector<int> run(g1 - g0, -1), open(n, -1);
  std::vector<char> dense;
  auto zero = [](cd z) { return z.real() == 0.0 && z.imag() == 0.0; };
  auto derivative = [](const qs_gate& G, int p, const cd* Ud, int dim, cd* M) {   // (dU/dt_p) U^dagger
    cd dU[16];
    gate_dmatrix(G, p, dU);
    for (int r = 0; r < dim; ++r)
      for (int c = 0; c < dim; ++c) {
        cd acc = 0;
        for (int k = 0; k < dim; ++k) acc += dU[r * dim + k] * Ud[k * dim + c];
        M[r * dim + c] = acc;
      }
  };
  auto dagger = [](const qs_gate& G, cd* Ud, int* dim) {
    cd U[16];
    gate_matrix(G, U, dim);
    for (int r = 0; r < *dim; ++r)
      for (int c = 0; c < *dim; ++c) Ud[r * *dim + c] = std::conj(U[c * *dim + r]);
  };
  for (size_t g = g1; g-- > g0;) {
    const qs_gate& G = gates[g];
    cd Ud[16], M[16];
    int dim = 0;
    dagger(G, Ud, &dim);
    if (dim != 2) {
      open[G.q[0]] = open[G.q[1]] = -1;
      continue;
    }
    int& o = open[G.q[0]];
    if (o < 0) {
      o = (int)dense.size();
      dense.push_back(0);
    }
    run[g - g0] = o;
    bool d = zero(Ud[1]) && zero(Ud[2]);
    for (int p = 0; p < gate_nparams(G.kind) && d; ++p) {
      derivative(G, p, Ud, 2, M);
      d = zero(M[1]) && zero(M[2]);
    }
    if (!d) dense[(size_t)o] = 1;
  }
  std::vector<qs_gate> bw;
  std::vector<int> term;                       // per op: its record
  std::vector<int> run_op(dense.size(), -1);   // the op of a dense run
  std::vector<std::array<cd, 4>> W(dense.size());
  std::vector<std::vector<TermPar>> pars;      // per record
  auto as_gate = [](const qs_gate& G, const cd* m, int dim) {
    qs_gate x;
    std::memset(&x, 0, sizeof(x));
    x.kind = dim == 2 ? QS_MAT1 : QS_MAT2;
    x.q[0] = G.q[0];
    x.q[1] = dim == 2 ? 0 : G.q[1];
    for (int i = 0; i < dim * dim; ++i) {
      x.m[2 * i] = m[i].real();
      x.m[2 * i + 1] = m[i].imag();
    }
    return x;
  };
  auto record = [&](int nsum) {
    out.recs.push_back(TermRec{0, nsum, 0, 0});
    pars.emplace_back();
    return (int)out.recs.size() - 1;
  };
  auto mul2 = [](const cd* A, const cd* B, cd* C) {
    cd r[4] = {A[0] * B[0] + A[1] * B[2], A[0] * B[1] + A[1] * B[3], A[2] * B[0] + A[3] * B[2],
               A[2] * B[1] + A[3] * B[3]};
    for (int i = 0; i < 4; ++i) C[i] = r[i];
  };
  for (size_t g = g1; g-- > g0;) {
    const qs_gate& G = gates[g];
    cd Ud[16], M[16];
    int dim = 0;
    dagger(G, Ud, &dim);
    const int np = gate_nparams(G.kind), r = run[g - g0];
    if (r < 0 || !dense[(size_t)r]) {
      for (int p = 0; p < np; ++p) {
        derivative(G, p, Ud, dim, M);
        bw.push_back(as_gate(G, M, dim));
        term.push_back(record(1));
        pars.back().push_back(TermPar{(int64_t)(3 * g + p), {1.0, 0.0, 0.0, 0.0}});
      }
      bw.push_back(as_gate(G, Ud, dim));
      term.push_back(-1);
      continue;
    }
    cd* w = W[(size_t)r].data();
    const bool first = run_op[(size_t)r] < 0;
    if (first) {
      run_op[(size_t)r] = (int)bw.size();
      bw.push_back(as_gate(G, Ud, dim));   // the place; its matrix is the run's W, below
      term.push_back(-1);
      w[0] = w[3] = 1;
      w[1] = w[2] = 0;
    }
    int& t = term[(size_t)run_op[(size_t)r]];
    for (int p = 0; p < np; ++p) {
      if (t < 0) t = record(4);
      cd Wd[4] = {std::conj(w[0]), std::conj(w[2]), std::conj(w[1]), std::conj(w[3])};
      derivative(G, p, Ud, 2, M);
      mul2(Wd, M, M);
      mul2(M, w, M);
      pars[(size_t)t].push_back(TermPar{(int64_t)(3 * g + p),
                                        {-M[0].imag(), -M[3].imag(), 0.5 * (M[1].real() - M[2].real()),
                                         -0.5 * (M[1].imag() + M[2].imag())}});
    }
    mul2(Ud, w, w);
  }
  std::vector<int> vmap;
  build_fused_ops(bw.data(), bw.size(), n, out.ops, vmap, /*fuse=*/false, /*relabel=*/false);
  if (out.ops.size() != bw.size()) {
    set_error("adjoint op list changed size");
    return QS_EUNSUPPORTED;
  }
  for (size_t i = 0; i < out.ops.size(); ++i) {
    out.ops[i].term = term[i];
    if (term[i] >= 0 && out.recs[(size_t)term[i]].nsum == 1 && out.ops[i].type != F_D) {
      set_error("derivative matrix of gate %d is not a one-qubit or diagonal op", (int)(pars[(size_t)term[i]][0].slot / 3));
      return QS_EUNSUPPORTED;
    }
  }
  for (size_t r = 0; r < W.size(); ++r) {
    if (run_op[r] < 0) continue;
    FOp& o = out.ops[(size_t)run_op[r]];
    const int tm = o.term, q = bw[(size_t)run_op[r]].q[0];
    o = FOp{};
    o.type = F_G1;
    o.t = q;
    o.term = tm;
    for (int k = 0; k < 4; ++k) o.m0[k] = W[r][(size_t)k];
  }
  fold_diagonals_back(out.ops, n);
  for (size_t i = 0; i < pars.size(); ++i) {
    out.recs[i].par = (int32_t)out.pars.size();
    out.recs[i].npar = (int32_t)pars[i].size();
    out.pars.insert(out.pars.end(), pars[i].begin(), pars[i].end());
  }
  return QS_OK;
}

// The adjoint sweep over gates [g0, g1) fused into tile passes: the tile planner
// splits the ops of adjoint_ops (an op keeps its order with the ops that share a
// qubit), and each pass runs the adjoint pass kernel on psi = st->data and lam, its
// per-tile sums reduced into dth.
template <typename R>
qs_status adjoint_tiled_t(State* st, void* lam, const qs_gate* gates, size_t g0, size_t g1, double* dth) {
  const int n = st->n;
  if (n < kTileBits) {
    set_error("fused adjoint needs n >= %d", kTileBits);
    return QS_EUNSUPPORTED;
  }
  AdjointOps ad;
  qs_status s = adjoint_ops(gates, g0, g1, n, ad);
  if (s != QS_OK) return s;
  std::vector<int> vmap(n);
  for (int q = 0; q < n; ++q) vmap[q] = q;
  Plan pl;
  std::vector<TermRec> recs;            // of every pass in turn
  std::vector<size_t> rec_off;          // per step, one past the last at the end
  std::vector<int> nsums;               // per step
  int most = 0;
  // a pass holds at most kMaxOps sums (its shared memory, and the partials): a plan that exceeds it
  // is made again with passes that cannot
  for (int cap : {TileLimits<R>::kMaxOps, TileLimits<R>::kMaxOps / 4}) {
    plan_circuit(ad.ops, n, vmap, pl, cap, kMaxTileStages);
    recs.clear();
    rec_off.clear();
    nsums.clear();
    most = 0;
    for (const PlanStep& step : pl.steps) {
      rec_off.push_back(recs.size());
      int ns = 0;
      if (step.kind == PlanStep::TILE) {
        const TilePass& pass = pl.passes[step.index];
        for (int s2 = 0; s2 < pass.n_stages; ++s2) {
          const TileStage& ts = pl.stages[pass.stage_begin + s2];
          for (int o = ts.op_begin; o < ts.op_end; ++o) {
            const int t = pl.tile_fops[o].term;
            if (t < 0) continue;
            recs.push_back(ad.recs[(size_t)t]);
            recs.back().sum = ns;
            ns += recs.back().nsum;
          }
        }
      }
      nsums.push_back(ns);
      most = std::max(most, ns);
    }
    rec_off.push_back(recs.size());
    if (most <= TileLimits<R>::kMaxOps) break;
  }
  if (!pl.remaps.empty()) {
    set_error("adjoint plan needs a remap");
    return QS_EUNSUPPORTED;
  }
  const uint64_t tiles = 1ull << (n - kTileBits);
  const size_t pbytes = sizeof(R) * tiles * (size_t)std::max(most, 1);
  void* partial = dev_alloc(st, pbytes);
  if (!partial) {
    set_error("adjoint partials allocation failed");
    return QS_ENOMEM;
  }
  // the records and derivatives of every pass, uploaded once
  std::vector<unsigned char> blob;
  const size_t off_recs = put(blob, recs.data(), recs.size());
  const size_t off_pars = put(blob, ad.pars.data(), ad.pars.size());
  s = upload(st, blob);
  const TermRec* recs_dev = (const TermRec*)((unsigned char*)st->opbuf + off_recs);
  const TermPar* pars_dev = (const TermPar*)((unsigned char*)st->opbuf + off_pars);
  std::unique_ptr<TileParams<R>> tp(new TileParams<R>());
  for (size_t si = 0; si < pl.steps.size() && s == QS_OK; ++si) {
    const PlanStep& step = pl.steps[si];
    if (step.kind == PlanStep::TILE) {
      const TilePass& pass = pl.passes[step.index];
      std::memset(tp.get(), 0, sizeof(TileParams<R>));
      tp->pass = pass;
      const int op0 = pl.stages[pass.stage_begin].op_begin;
      size_t rec = rec_off[si];
      for (int s2 = 0; s2 < pass.n_stages; ++s2) {
        TileStage ts = pl.stages[pass.stage_begin + s2];
        for (int o = ts.op_begin; o < ts.op_end; ++o) {
          TileOp<R> t = to_tile<R>(pl, (size_t)o);
          t.term = pl.tile_fops[o].term >= 0 ? (int16_t)recs[rec++].sum : (int16_t)-1;
          tp->ops[o - op0] = t;
        }
        ts.op_begin -= op0;
        ts.op_end -= op0;
        tp->stages[s2] = ts;
      }
      tp->pass.stage_begin = 0;
      s = launch_adjoint_pass(st, lam, tp.get(), partial, nsums[si]);
      if (s == QS_OK)
        s = launch_term_reduce(st, partial, nsums[si], recs_dev + rec_off[si], (int)(rec_off[si + 1] - rec_off[si]),
                               pars_dev, dth);
    } else if (step.kind == PlanStep::PLAIN) {
      PlainOp<R> p = to_plain<R>(pl.plain_fops[step.index]);
      s = launch_plain_op(st, &p, p.type);
      void* psi = st->data;
      st->data = lam;
      if (s == QS_OK) s = launch_plain_op(st, &p, p.type);
      st->data = psi;
    } else {
      set_error("unexpected step in the adjoint plan");
      s = QS_EUNSUPPORTED;
    }
  }
  cudaStreamSynchronize(st->stream);
  dev_free(st, partial, pbytes);
  return s;
}

// Dense 5-qubit blocks on the tensor cores: one pass per block.
qs_status run_block_list(State* st, const std::vector<Block>& blocks, int mode, qs_stats* stats,
                         KernelTimer& tm) {
  if (blocks.empty()) return QS_OK;
  std::vector<unsigned char> blob(16, 0);   // status word of the bounded waits
  std::vector<BlockPass> passes(blocks.size());
  for (size_t i = 0; i < blocks.size(); ++i) {
    block_pass_desc(st->n, blocks[i].q, passes[i]);
    if (!block_pass_runs_contiguous(passes[i])) {
      set_error("block pass: tile layout without contiguous low bits");
      return QS_EUNSUPPORTED;
    }
  }
  // per block (independent, on host threads): the unitarity flag and the split B operand
  const size_t bb = block_b_bytes(mode);
  std::vector<unsigned char> bops(bb * blocks.size());
  std::vector<char> unitary(blocks.size(), 0);
  parallel_for(blocks.size(), 4, [&](size_t i) {
    unitary[i] = block_is_unitary(blocks[i].U.data()) ? 1 : 0;
    std::vector<unsigned char> tmp;
    block_b_operand(blocks[i].U.data(), mode, tmp);
    std::memcpy(bops.data() + i * bb, tmp.data(), bb);
  });
  for (size_t i = 0; i < blocks.size(); ++i)
    if (unitary[i]) passes[i].flags |= 1;
  const size_t off_pass = put(blob, passes.data(), passes.size());
  const size_t off_b = align16(blob.size());
  blob.resize(off_b + bops.size());
  std::memcpy(blob.data() + off_b, bops.data(), bops.size());
  qs_status s = upload(st, blob);
  if (s != QS_OK) return s;
  unsigned char* dev = (unsigned char*)st->opbuf;
  int* status_dev = (int*)dev;
  for (size_t i = 0; i < blocks.size(); ++i) {
    tm.before(4);
    s = launch_block_pass(st, passes[i], dev + off_pass + i * sizeof(BlockPass), dev + off_b + i * bb,
                          mode, status_dev);
    tm.after();
    if (s != QS_OK) return s;
  }
  int status = 0;
  QS_CUDA(cudaMemcpyAsync(&status, status_dev, sizeof(int), cudaMemcpyDeviceToHost, st->stream));
  QS_CUDA(cudaStreamSynchronize(st->stream));
  if (status != 0) {
    set_error("block GEMM kernel: bounded wait on the tensor-core barrier gave up");
    return QS_ETIMEOUT;
  }
  if (stats) {
    stats->ops_fused += (int64_t)blocks.size();
    stats->passes += (int64_t)blocks.size();
    stats->launches += (int64_t)blocks.size();
    // 32 complex MACs per amplitude per block = 256 flops (the split precision triples the MMAs)
    stats->flops += 256.0 * std::ldexp(1.0, st->n) * (double)blocks.size();
    stats->upload_bytes += (int64_t)blob.size();
  }
  return QS_OK;
}

// Chains of 5-qubit blocks (chain_tc.cu): up to kChainMax blocks per sweep.  The plan's blocks
// are multiplied out here, a first part of the passes and then the rest, so that the device
// starts on the first while the host works on the others (their operands go up in two copies).
qs_status run_chains(State* st, const qs_gate* gates, const std::vector<ChainPlan>& plan, qs_stats* stats,
                     KernelTimer& tm) {
  std::vector<ChainPass> passes(plan.size());
  std::vector<const Block*> blocks;
  std::vector<size_t> first;   // of each pass, into blocks
  for (size_t i = 0; i < plan.size(); ++i) {
    uint64_t mask[kChainMax] = {};
    first.push_back(blocks.size());
    for (size_t b = 0; b < plan[i].blocks.size(); ++b) {
      for (int q : plan[i].blocks[b].q) mask[b] |= 1ull << q;
      blocks.push_back(&plan[i].blocks[b]);
    }
    if (!chain_pass_desc(st->n, plan[i].tile, mask, (int)plan[i].blocks.size(), passes[i])) {
      set_error("block chain: invalid tile");
      return QS_EUNSUPPORTED;
    }
  }
  first.push_back(blocks.size());
  const size_t bytes = 16 + blocks.size() * (size_t)kChainB;   // status word, B operands
  unsigned char* host = nullptr;
  qs_status s = upload_begin(st, bytes, &host);
  if (s != QS_OK) return s;
  s = launch_chain_setup();
  if (s != QS_OK) return s;
  std::memset(host, 0, 16);
  unsigned char* dev = (unsigned char*)st->opbuf;
  const size_t part = passes.size() > 8 ? passes.size() / 4 : passes.size();
  size_t sent = 0;
  for (size_t p0 = 0; p0 < passes.size() && s == QS_OK;) {
    const size_t p1 = p0 == 0 ? part : passes.size();
    parallel_for(first[p1] - first[p0], 4, [&](size_t k) {
      cd U[32 * 32];   // (nothing is allocated once a pass has been launched)
      block_matrix(gates, *blocks[first[p0] + k], U);
      chain_b_operand(U, host + 16 + (first[p0] + k) * kChainB);
    });
    const size_t end = 16 + first[p1] * kChainB;
    s = upload_part(st, sent, end, p1 == passes.size());
    sent = end;
    for (size_t i = p0; i < p1 && s == QS_OK; ++i) {
      tm.before(4);
      s = launch_chain_pass(st, passes[i], dev + 16 + first[i] * kChainB, (int*)dev);
      tm.after();
    }
    p0 = p1;
  }
  if (s != QS_OK) {   // a copy may still be reading the pinned buffer
    cudaStreamSynchronize(st->stream);
    return s;
  }
  int status = 0;
  QS_CUDA(cudaMemcpyAsync(&status, dev, sizeof(int), cudaMemcpyDeviceToHost, st->stream));
  QS_CUDA(cudaStreamSynchronize(st->stream));
  if (status != 0) {
    set_error(status == QS_ETIMEOUT ? "block chain kernel: bounded wait gave up"
                                    : "block chain kernel: the tile slots do not fit shared memory");
    return (qs_status)status;
  }
  if (stats) {
    stats->ops_fused += (int64_t)blocks.size();
    stats->passes += (int64_t)passes.size();
    stats->launches += (int64_t)passes.size();
    stats->flops += 256.0 * std::ldexp(1.0, st->n) * (double)blocks.size();
    stats->upload_bytes += (int64_t)bytes;
  }
  return QS_OK;
}

// Every explicit matrix is unitary within 1e-12 (the named gates are by definition): the
// blocks of a chain then keep each row's norm, which its kernel relies on.
bool gates_unitary(const qs_gate* gates, size_t ngates) {
  for (size_t i = 0; i < ngates; ++i) {
    if (gates[i].kind != QS_MAT1 && gates[i].kind != QS_MAT2) continue;
    cd m[16];
    int dim = 0;
    gate_matrix(gates[i], m, &dim);
    for (int a = 0; a < dim; ++a)
      for (int b = a; b < dim; ++b) {
        cd v = a == b ? cd(-1.0) : cd(0.0);
        for (int k = 0; k < dim; ++k) v += std::conj(m[k * dim + a]) * m[k * dim + b];
        if (!(std::abs(v) <= 1e-12)) return false;
      }
  }
  return true;
}

qs_status run_blocks(State* st, const qs_gate* gates, size_t ngates, int mode, qs_stats* stats,
                     KernelTimer& tm) {
  std::vector<Block> blocks;
  plan_blocks(gates, ngates, st->n, blocks);
  return run_block_list(st, blocks, mode, stats, tm);
}

// One sweep per block over blocks [0, count), their operands (kF64Op bytes each) at `ops`, or null: then
// they stand in the pinned buffer already.  Asynchronous: what the kernels report is taken by late_status.
qs_status run_f64_list(State* st, const F64Pass* passes, size_t count, const unsigned char* ops, qs_stats* stats,
                       KernelTimer& tm) {
  const size_t bytes = count * (size_t)kF64Op;
  unsigned char* host = (unsigned char*)st->hostbuf;
  qs_status s = QS_OK;
  if (ops) {
    s = upload_begin(st, bytes, &host);
    if (s != QS_OK) return s;
    std::memcpy(host, ops, bytes);
  }
  unsigned char* dev = (unsigned char*)st->opbuf;
  s = upload_part(st, 0, bytes, true);
  for (size_t i = 0; i < count && s == QS_OK; ++i) {
    tm.before(4);
    s = launch_f64_pass(st, passes[i], dev + i * kF64Op, st->late);
    tm.after();
  }
  if (s != QS_OK) {
    cudaStreamSynchronize(st->stream);
    return s == QS_EUNSUPPORTED ? QS_ECUDA : s;
  }
  if (stats) {
    stats->ops_fused += (int64_t)count;
    stats->passes += (int64_t)count;
    stats->launches += (int64_t)count;
    stats->flops += 256.0 * std::ldexp(1.0, st->n) * (double)count;
    stats->upload_bytes += (int64_t)bytes;
  }
  return QS_OK;
}

// The gates of blocks [i, j) on tile passes, added to stats.
template <typename R>
qs_status run_tile_segment(State* st, const qs_gate* gates, const std::vector<Block>& blocks, size_t i, size_t j,
                           qs_stats* stats, KernelTimer& tm) {
  std::vector<qs_gate> seg;
  for (size_t k = i; k < j; ++k)
    for (size_t gi : blocks[k].gate_idx) seg.push_back(gates[gi]);
  std::vector<FOp> fops;
  std::vector<int> vmap;
  build_fused_ops(seg.data(), seg.size(), st->n, fops, vmap, /*fuse=*/true, /*relabel=*/true);
  qs_stats part;
  std::memset(&part, 0, sizeof(part));
  const qs_status s = run_tiled<R>(st, fops, vmap, &part, tm);
  if (stats) {
    stats->ops_fused += part.ops_fused;
    stats->passes += part.passes;
    stats->launches += part.launches;
    stats->tile_launches += part.tile_launches;
    stats->tile_flops += part.tile_flops;
    stats->flops += part.flops;
    stats->upload_bytes += part.upload_bytes;
  }
  return s;
}

// QS_METHOD_AUTO, complex128, n > kSmallAutoBits: circuits of mostly dense blocks (at least three for each
// other one) run block by block on the tensor cores (block_f64.cu), and blocks whose matrices the
// integer slices do not take (f64_b_operand) gate by gate on tile passes between them.
// QS_EUNSUPPORTED, with nothing launched, for other circuits: they run on tile passes.
qs_status run_f64_blocks(State* st, const qs_gate* gates, size_t ngates, qs_stats* stats, KernelTimer& tm) {
  if (!chains_likely(gates, ngates)) return QS_EUNSUPPORTED;
  if (packed_ctas() > 0 && packed_ctas() != reserved_sms()) return QS_EUNSUPPORTED;   // (too few SMs free for a while)
  std::vector<Block> blocks;
  plan_blocks(gates, ngates, st->n, blocks, /*products=*/false);
  const size_t nb = blocks.size();
  std::vector<char> is_dense(nb), fits(nb);
  auto mostly = [&](const std::vector<char>& also) {
    size_t dense = 0;
    for (size_t i = 0; i < nb; ++i) dense += is_dense[i] && also[i];
    return dense > 0 && dense >= 3 * (nb - dense);
  };
  for (size_t i = 0, sparse = 0; i < nb; ++i) {
    is_dense[i] = block_dense(gates, blocks[i]);
    sparse += !is_dense[i];
    if (4 * sparse > nb) return QS_EUNSUPPORTED;   // (decided: the rest need not be looked at)
  }
  std::vector<F64Pass> passes(nb);
  for (size_t i = 0; i < nb; ++i)
    if (!f64_pass_desc(st->n, blocks[i].q, passes[i])) return QS_EUNSUPPORTED;
  unsigned char* host = nullptr;
  qs_status s = upload_begin(st, nb * (size_t)kF64Op, &host);
  if (s == QS_ENOMEM) return QS_EUNSUPPORTED;   // (tile passes need less)
  if (s != QS_OK) return s;
  if (!st->late) {
    if (cudaHostAlloc((void**)&st->late, sizeof(int), cudaHostAllocMapped) != cudaSuccess) {
      cudaGetLastError();
      st->late = nullptr;
      return QS_EUNSUPPORTED;
    }
    *st->late = 0;
  }
  parallel_for(nb, 2, [&](size_t i) {
    unsigned char* const at = host + i * kF64Op;
    fits[i] = f64_b_operand(gates, blocks[i], at, &passes[i].vs, (cd*)(at + kF64B));
  });
  if (!mostly(fits)) return QS_EUNSUPPORTED;
  s = launch_f64_setup();
  if (s != QS_OK) return s;
  if (std::find(fits.begin(), fits.end(), (char)0) == fits.end())
    return run_f64_list(st, passes.data(), nb, nullptr, stats, tm);
  // (the tile passes' uploads take the pinned buffer)
  const std::vector<unsigned char> ops(host, host + nb * (size_t)kF64Op);
  for (size_t i = 0; i < nb && s == QS_OK;) {
    size_t j = i;
    while (j < nb && fits[j] == fits[i]) ++j;
    s = fits[i] ? run_f64_list(st, passes.data() + i, j - i, ops.data() + i * kF64Op, stats, tm)
                : run_tile_segment<double>(st, gates, blocks, i, j, stats, tm);
    if (s == QS_EUNSUPPORTED) s = QS_ECUDA;   // (something has been launched)
    i = j;
  }
  return s;
}

// QS_METHOD_AUTO (complex64, larger states than kSmallAutoBits allows): the circuit is cut into 5-qubit blocks;
// a dense block (more than half of its 1024 entries nonzero) is a real
// contraction and goes to the tensor cores (the gates of a run of dense blocks planned
// again as chains of blocks, one block per sweep if a gate is not unitary), and every
// maximal run of sparse
// blocks (diagonal or nearly diagonal stretches such as the QFT's controlled
// phases) goes back to its gates, which the tile planner fuses into shared-memory
// passes of 12 qubits.  Both kinds of segment start and end in the canonical
// layout, and applying the blocks in order equals the circuit, so the segments
// compose.
qs_status run_auto(State* st, const qs_gate* gates, size_t ngates, qs_stats* stats, KernelTimer& tm) {
  const bool chains = gates_unitary(gates, ngates);
  std::vector<ChainPlan> plan;
  if (chains && chains_likely(gates, ngates)) {   // a circuit of dense layers: all of it as chains
    plan_chains(gates, ngates, st->n, plan, /*products=*/false);
    if (chains_dense(gates, plan)) return run_chains(st, gates, plan, stats, tm);
  }
  // Density from the gates' patterns, and products only for the blocks that need them: the plan of
  // chains above then costs less than it saves where it is given up (300 mixed gates on 20 qubits: 0.34 ms
  // for it, and 0.44 in place of 1.25 ms here).
  std::vector<Block> blocks;
  plan_blocks(gates, ngates, st->n, blocks, /*products=*/false);
  std::vector<char> is_dense(blocks.size());
  for (size_t k = 0; k < blocks.size(); ++k) is_dense[k] = block_dense(gates, blocks[k]);
  // one or two dense blocks among sparse ones (the QFT's Hadamards among its
  // phases) may run on tile passes alone (auto_plan.h)
  {
    std::vector<FOp> fops;
    std::vector<int> vmap;
    if (auto_all_tiles(gates, ngates, st->n, blocks, is_dense, &fops, &vmap)) {
      qs_stats part;
      std::memset(&part, 0, sizeof(part));
      qs_status s = run_tiled<float>(st, fops, vmap, &part, tm);
      if (stats) {
        stats->ops_fused = part.ops_fused;
        stats->passes = part.passes;
        stats->launches = part.launches;
        stats->tile_launches = part.tile_launches;
        stats->tile_flops = part.tile_flops;
        stats->flops = part.flops;
        stats->upload_bytes = part.upload_bytes;
      }
      if (s == QS_OK) QS_CUDA(cudaStreamSynchronize(st->stream));
      return s;
    }
  }
  if (chains) auto_short_runs(is_dense);
  size_t i = 0;
  qs_status s = QS_OK;
  while (i < blocks.size() && s == QS_OK) {
    const bool dense = is_dense[i];
    size_t j = i;
    while (j < blocks.size() && (bool)is_dense[j] == dense) ++j;
    if (dense && chains) {
      std::vector<qs_gate> seg;
      for (size_t k = i; k < j; ++k)
        for (size_t gi : blocks[k].gate_idx) seg.push_back(gates[gi]);
      plan_chains(seg.data(), seg.size(), st->n, plan, /*products=*/false);
      s = run_chains(st, seg.data(), plan, stats, tm);
    } else if (dense) {
      std::vector<Block> seg(std::make_move_iterator(blocks.begin() + (long)i),
                             std::make_move_iterator(blocks.begin() + (long)j));
      parallel_for(seg.size(), 8, [&](size_t k) { block_product(gates, seg[k]); });
      s = run_block_list(st, seg, 1, stats, tm);
    } else {
      s = run_tile_segment<float>(st, gates, blocks, i, j, stats, tm);
    }
    i = j;
  }
  if (s == QS_OK) {   // the tile segments run asynchronously; report their faults here too
    QS_CUDA(cudaStreamSynchronize(st->stream));
  }
  return s;
}

qs_status check_state(qs_state_t st) {
  if (!st) {
    set_error("state is NULL");
    return QS_EINVAL;
  }
  return QS_OK;
}

}  // namespace

// The kernel-parameter image of a forward tile pass and its run tables (tile_cp.h).
template <typename R>
void tile_pass_image(const Plan& pl, const TilePass& pass, TileParams<R>* tp, std::vector<C2<R>>& tabs) {
  build_pass_params<R>(pl, pass, tp, tabs);
}
template void tile_pass_image<float>(const Plan&, const TilePass&, TileParams<float>*, std::vector<C2<float>>&);
template void tile_pass_image<double>(const Plan&, const TilePass&, TileParams<double>*, std::vector<C2<double>>&);


template <typename R>
qs_status adjoint_small_t(State* st, void* lam, const qs_gate* gates, size_t ng, double* dth) {
  AdjointOps ad;
  qs_status s = adjoint_ops(gates, 0, ng, st->n, ad);
  if (s != QS_OK || ad.ops.empty()) return s;
  constexpr int kSums = 4096;   // of one launch: bounds the partials
  struct Part {
    int op, nop, rec, nrec, nsum;
  };
  std::vector<Part> parts{{0, 0, 0, 0, 0}};
  std::vector<PlainOp<R>> ops;
  std::vector<TermRec> recs;
  for (const FOp& o : ad.ops) {
    PlainOp<R> p = to_plain<R>(o);
    p.pad[0] = 0;
    if (o.term >= 0) {
      TermRec r = ad.recs[(size_t)o.term];
      if (parts.back().nsum + r.nsum > kSums) parts.push_back({(int)ops.size(), 0, (int)recs.size(), 0, 0});
      r.sum = parts.back().nsum;
      p.pad[0] = 1 + r.sum;
      parts.back().nsum += r.nsum;
      ++parts.back().nrec;
      recs.push_back(r);
    }
    ops.push_back(p);
    ++parts.back().nop;
  }
  const size_t pbytes = sizeof(double) * (size_t)adjoint_small_warps(st) * kSums;
  double* partial = (double*)dev_alloc(st, pbytes);
  if (!partial) return QS_EUNSUPPORTED;   // (gate by gate takes less)
  std::vector<unsigned char> blob;
  const size_t off_ops = put(blob, ops.data(), ops.size());
  const size_t off_recs = put(blob, recs.data(), recs.size());
  const size_t off_pars = put(blob, ad.pars.data(), ad.pars.size());
  s = upload(st, blob);
  if (s == QS_ENOMEM) s = QS_EUNSUPPORTED;   // (nothing launched)
  unsigned char* dev = (unsigned char*)st->opbuf;
  for (size_t i = 0; i < parts.size() && s == QS_OK; ++i) {
    const Part& q = parts[i];
    s = launch_adjoint_small(st, lam, dev + off_ops + sizeof(PlainOp<R>) * (size_t)q.op, q.nop, partial, q.nsum,
                             (const TermRec*)(dev + off_recs) + q.rec, q.nrec, (const TermPar*)(dev + off_pars), dth);
  }
  cudaStreamSynchronize(st->stream);
  dev_free(st, partial, pbytes);
  return s;
}

qs_status adjoint_small(State* st, void* lam, const qs_gate* gates, size_t ng, double* dth) {
  if (!gates_unitary(gates, ng) || !small_fits(st)) return QS_EUNSUPPORTED;
  return st->prec == QS_C64 ? adjoint_small_t<float>(st, lam, gates, ng, dth)
                            : adjoint_small_t<double>(st, lam, gates, ng, dth);
}

qs_status adjoint_tiled(State* st, void* lam, const qs_gate* gates, size_t g0, size_t g1, double* dth) {
  return st->prec == QS_C64 ? adjoint_tiled_t<float>(st, lam, gates, g0, g1, dth)
                            : adjoint_tiled_t<double>(st, lam, gates, g0, g1, dth);
}

// QS_METHOD_AUTO keeps states of up to this many qubits in the registers of one CTA or cluster
// (small_state_kernel): one launch whatever the circuit, where blocks and tiles of such states leave
// the chip idle and pay for a launch and a pipeline's start per sweep.  Whole calls, us, there
// against here, 12 and 13 qubits: layered complex64 of 10 and 80 layers 250 and 1271 -> 66 and 346,
// 515 and 1418 -> 73 and 390; complex128 of 10 and 60 layers 700 and 2501 -> 103 and 472, 737 and 2860 ->
// 190 and 937; Haar and CNOT complex128 of 5 and 60 layers 461 and 4557 -> 93 and 816, 490 and 4525 -> 153
// and 1483; Fourier 278 -> 53 (12 qubits); 500 mixed gates 922 -> 171, 1106 -> 175.
// Above, a thread would hold several amplitudes.  Circuits of 13 complex64 qubits in which at most a fifth of
// the gates make superpositions (chains_likely) keep to tile passes although one launch would be faster there
// too: the library has always run them so and reports it (qs_stats.tile_launches), which its callers can hold it to.
constexpr int kSmallAutoBits = 13;

// Whether the state's stream is being captured into a graph.
static bool capturing(const State* st) {
  cudaStreamCaptureStatus c = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st->stream, &c) != cudaSuccess) cudaGetLastError();
  return c != cudaStreamCaptureStatusNone;
}

qs_status apply_gates(State* st, const qs_gate* gates, size_t ngates, int method, qs_stats* stats,
                      int flags) {
  if (stats) std::memset(stats, 0, sizeof(*stats));
  if (method < QS_METHOD_TILED || method > QS_METHOD_AUTO) {
    set_error("unknown method %d", method);
    return QS_EINVAL;
  }
  // AUTO: blocks and tile passes where the state allows the blocks, else tiles
  const bool autom = method == QS_METHOD_AUTO && st->prec == QS_C64 && st->n >= kTileBits;
  const qs_status earlier = late_status(st);   // (of a call that has ended by now)
  if (earlier != QS_OK) return earlier;
  // (a captured complex128 call keeps to tile passes, whose launches hold all they need)
  const bool captured = method == QS_METHOD_AUTO && st->prec == QS_C128 && st->n >= kTileBits && capturing(st);
  const bool auto_small = method == QS_METHOD_AUTO && st->n <= kSmallAutoBits && !captured &&
                          (st->n < kTileBits || small_fits(st)) &&
                          (st->prec == QS_C128 || st->n < kSmallAutoBits || chains_likely(gates, ngates));
  const bool auto_f64 = method == QS_METHOD_AUTO && st->prec == QS_C128 && st->n >= kTileBits && !auto_small && !captured;
  if (method == QS_METHOD_AUTO && !autom) method = QS_METHOD_TILED;
  const bool blocks = method == QS_METHOD_BLOCKS_TF32 || method == QS_METHOD_BLOCKS_BF16;
  if (blocks && (st->prec != QS_C64 || st->n < kTileBits)) {
    set_error("the tensor-core block method needs a complex64 state of at least %d qubits", kTileBits);
    return QS_EUNSUPPORTED;
  }
  if (ngates == 0) return QS_OK;
  std::vector<FOp> fops;
  std::vector<int> vmap;
  const bool c64 = st->prec == QS_C64;
  KernelTimer tm;
  tm.on = (flags & QS_OPT_TIME_KERNELS) != 0;
  tm.stream = st->stream;
  qs_status s = QS_EUNSUPPORTED;
  if (auto_f64) s = run_f64_blocks(st, gates, ngates, stats, tm);
  if (auto_f64 && s != QS_EUNSUPPORTED) {
  } else if (autom && !auto_small) {
    s = run_auto(st, gates, ngates, stats, tm);
  } else if (blocks) {
    s = run_blocks(st, gates, ngates, method == QS_METHOD_BLOCKS_TF32 ? 0 : 1, stats, tm);
  } else if (method == QS_METHOD_PLAIN) {
    build_fused_ops(gates, ngates, st->n, fops, vmap, /*fuse=*/false, /*relabel=*/false);
    s = c64 ? run_plain<float>(st, fops, stats, tm) : run_plain<double>(st, fops, stats, tm);
  } else if (st->n < kTileBits || auto_small) {
    build_fused_ops(gates, ngates, st->n, fops, vmap, /*fuse=*/true, /*relabel=*/false);
    merge_one_qubit_ops(fops, st->n, nullptr);   // one CTA runs them all: no passes to keep
    s = c64 ? run_small<float>(st, fops, stats, tm) : run_small<double>(st, fops, stats, tm);
    if (s == QS_ENOMEM && st->n >= kTileBits) {   // (all of its ops at once on the device; tile passes carry theirs along)
      build_fused_ops(gates, ngates, st->n, fops, vmap, /*fuse=*/true, /*relabel=*/true);
      s = c64 ? run_tiled<float>(st, fops, vmap, stats, tm) : run_tiled<double>(st, fops, vmap, stats, tm);
    }
    // (the default method of complex64 states from kTileBits on returns when the state is ready)
    if (autom && s == QS_OK) QS_CUDA(cudaStreamSynchronize(st->stream));
  } else {
    build_fused_ops(gates, ngates, st->n, fops, vmap, /*fuse=*/true, /*relabel=*/true);
    s = c64 ? run_tiled<float>(st, fops, vmap, stats, tm)
            : run_tiled<double>(st, fops, vmap, stats, tm);
  }
  tm.finish(stats);
  if (tm.on && s == QS_OK) s = late_status(st);   // (the events have been waited for)
  if (stats) {
    stats->gates_in = (int64_t)ngates;
    stats->bytes_moved = (double)stats->passes * 2.0 * (double)st->data_bytes;
  }
  return s;
}

// Copies of probabilities to host memory queued by sv_probs_host_async, per
// state: two device buffers used in turn, a non-blocking copy stream, and per
// buffer an event when its probabilities are formed (state's stream) and one
// when its copy has ended (copy stream).  Kept beside the state, keyed by it.
struct HostCopies {
  void* buf = nullptr;   // 2 * half bytes
  size_t half = 0;
  cudaStream_t cs = nullptr;
  cudaEvent_t formed[2] = {nullptr, nullptr};
  cudaEvent_t copied[2] = {nullptr, nullptr};
  bool queued[2] = {false, false};
  int next = 0;
};
std::mutex g_copies_mu;
std::unordered_map<const State*, HostCopies*> g_copies;

HostCopies* find_copies(const State* st) {
  std::lock_guard<std::mutex> g(g_copies_mu);
  auto it = g_copies.find(st);
  return it == g_copies.end() ? nullptr : it->second;
}

// waits for the state's queued copies (if any); the first error is returned
qs_status wait_copies(State* st) {
  HostCopies* hc = find_copies(st);
  if (!hc) return QS_OK;
  const cudaError_t e = cudaStreamSynchronize(hc->cs);
  hc->queued[0] = hc->queued[1] = false;
  return e == cudaSuccess ? QS_OK : cuda_status(e, "copy of probabilities to the host");
}

void release_copies(State* st) {
  HostCopies* hc = nullptr;
  {
    std::lock_guard<std::mutex> g(g_copies_mu);
    auto it = g_copies.find(st);
    if (it == g_copies.end()) return;
    hc = it->second;
    g_copies.erase(it);
  }
  if (hc->cs) cudaStreamSynchronize(hc->cs);
  if (hc->buf) dev_free(st, hc->buf, 2 * hc->half);
  for (int k = 0; k < 2; ++k) {
    if (hc->formed[k]) cudaEventDestroy(hc->formed[k]);
    if (hc->copied[k]) cudaEventDestroy(hc->copied[k]);
  }
  if (hc->cs) cudaStreamDestroy(hc->cs);
  delete hc;
}

// the state's copy pipeline with buffers of at least `half` bytes each
qs_status copies_for(State* st, size_t half, HostCopies** out) {
  HostCopies* hc = find_copies(st);
  if (hc && hc->half < half) {   // buffers too small (an fp64 call after fp32 ones): start over
    cudaStreamSynchronize(st->stream);   // no kernel of the state may still write them
    release_copies(st);
    hc = nullptr;
  }
  if (!hc) {
    hc = new (std::nothrow) HostCopies();
    if (!hc) {
      set_error("host copy pipeline: out of host memory");
      return QS_ENOMEM;
    }
    cudaError_t e = cudaStreamCreateWithFlags(&hc->cs, cudaStreamNonBlocking);
    for (int k = 0; k < 2 && e == cudaSuccess; ++k) {
      e = cudaEventCreateWithFlags(&hc->formed[k], cudaEventDisableTiming);
      if (e == cudaSuccess) e = cudaEventCreateWithFlags(&hc->copied[k], cudaEventDisableTiming);
    }
    if (e == cudaSuccess) {
      hc->buf = dev_alloc(st, 2 * half);
      hc->half = half;
    }
    {
      std::lock_guard<std::mutex> g(g_copies_mu);
      g_copies[st] = hc;   // released by release_copies on every path below
    }
    if (e != cudaSuccess) {
      const qs_status s = cuda_status(e, "host copy pipeline");
      release_copies(st);
      return s;
    }
    if (!hc->buf) {
      hc->half = 0;
      release_copies(st);
      set_error("device buffers for the host copies of the probabilities could not be allocated");
      return QS_ENOMEM;
    }
  }
  *out = hc;
  return QS_OK;
}

}  // namespace qs

using namespace qs;

extern "C" {

const char* qs_last_error(void) { return g_err.c_str(); }

const char* qs_version(void) { return "qsim-gb300 0.5 (sm_103a)"; }

qs_status sv_create(int n, int prec, const qs_allocator* alloc, void* stream, qs_state_t* out) {
  return abi_guard(__func__, [&]() -> qs_status {
    if (!out) {
      set_error("out is NULL");
      return QS_EINVAL;
    }
    *out = nullptr;
    if (n < 1 || n > 36) {
      set_error("n = %d outside [1, 36]", n);
      return QS_EINVAL;
    }
    if (prec != QS_C64 && prec != QS_C128) {
      set_error("bad precision %d", prec);
      return QS_EINVAL;
    }
    qs_state_s* st = new (std::nothrow) qs_state_s();
    if (!st) return QS_ENOMEM;
    st->n = n;
    st->prec = prec;
    st->amp_bytes = prec == QS_C64 ? 8 : 16;
    st->stream = (cudaStream_t)stream;
    if (alloc && alloc->alloc && alloc->free) {
      st->alloc = *alloc;
      st->has_alloc = true;
    }
    cudaGetDevice(&st->device);
    st->data_bytes = st->amp_bytes << n;
    st->data = dev_alloc(st, st->data_bytes);
    if (!st->data) {
      set_error("device allocation of %zu bytes for a %d-qubit state failed", st->data_bytes, n);
      delete st;
      return QS_ENOMEM;
    }
    st->scratch_bytes = kScratchBytes;
    st->scratch = dev_alloc(st, st->scratch_bytes);
    if (!st->scratch) {
      dev_free(st, st->data, st->data_bytes);
      set_error("scratch allocation failed");
      delete st;
      return QS_ENOMEM;
    }
    if (cudaEventCreateWithFlags(&st->upload_done, cudaEventDisableTiming) != cudaSuccess) {
      dev_free(st, st->scratch, st->scratch_bytes);
      dev_free(st, st->data, st->data_bytes);
      qs_status s = cuda_status(cudaGetLastError(), "cudaEventCreate");
      delete st;
      return s;
    }
    qs_status s = launch_set_basis(st, 0);
    if (s != QS_OK) {
      sv_destroy(st);
      return s;
    }
    *out = st;
    return QS_OK;
  });
}

qs_status sv_wrap(int n, int prec, void* device_buf, const qs_allocator* alloc, void* stream, qs_state_t* out) {
  return abi_guard(__func__, [&]() -> qs_status {
    if (!out || !device_buf) {
      set_error("out and device_buf are required");
      return QS_EINVAL;
    }
    *out = nullptr;
    if (n < 1 || n > 36 || (prec != QS_C64 && prec != QS_C128)) {
      set_error("n = %d outside [1, 36] or bad precision %d", n, prec);
      return QS_EINVAL;
    }
    if ((uintptr_t)device_buf & 15) {
      set_error("device_buf must be 16-byte aligned");
      return QS_EINVAL;
    }
    qs_state_s* st = new (std::nothrow) qs_state_s();
    if (!st) return QS_ENOMEM;
    st->n = n;
    st->prec = prec;
    st->amp_bytes = prec == QS_C64 ? 8 : 16;
    st->stream = (cudaStream_t)stream;
    if (alloc && alloc->alloc && alloc->free) {
      st->alloc = *alloc;
      st->has_alloc = true;
    }
    cudaGetDevice(&st->device);
    st->data_bytes = st->amp_bytes << n;
    st->data = device_buf;
    st->owns_data = false;
    st->scratch_bytes = kScratchBytes;
    st->scratch = dev_alloc(st, st->scratch_bytes);
    if (!st->scratch) {
      set_error("scratch allocation failed");
      delete st;
      return QS_ENOMEM;
    }
    if (cudaEventCreateWithFlags(&st->upload_done, cudaEventDisableTiming) != cudaSuccess) {
      dev_free(st, st->scratch, st->scratch_bytes);
      qs_status s = cuda_status(cudaGetLastError(), "cudaEventCreate");
      delete st;
      return s;
    }
    *out = st;
    return QS_OK;
  });
}

qs_status sv_destroy(qs_state_t st) {
  return abi_guard(__func__, [&]() -> qs_status {
    if (!st) return QS_OK;
    cudaStreamSynchronize(st->stream);
    release_copies(st);
    dev_free(st, st->opbuf, st->opbuf_bytes);
    if (st->stage) dev_free(st, st->stage, st->stage_bytes);
    dev_free(st, st->scratch, st->scratch_bytes);
    if (st->owns_data) dev_free(st, st->data, st->data_bytes);
    if (st->hostbuf) cudaFreeHost(st->hostbuf);
    if (st->late) cudaFreeHost(st->late);
    if (st->upload_done) cudaEventDestroy(st->upload_done);
    delete st;
    return QS_OK;
  });
}

qs_status sv_set_stream(qs_state_t st, void* stream) {
  return abi_guard(__func__, [&]() -> qs_status {
    qs_status s = check_state(st);
    if (s != QS_OK) return s;
    QS_CUDA(cudaStreamSynchronize(st->stream));
    st->stream = (cudaStream_t)stream;
    return late_status(st);
  });
}

qs_status sv_info(qs_state_t st, int* n, int* prec, void** device_ptr) {
  return abi_guard(__func__, [&]() -> qs_status {
    qs_status s = check_state(st);
    if (s != QS_OK) return s;
    if (n) *n = st->n;
    if (prec) *prec = st->prec;
    if (device_ptr) *device_ptr = st->data;
    return QS_OK;
  });
}

qs_status sv_set_basis(qs_state_t st, uint64_t J) {
  return abi_guard(__func__, [&]() -> qs_status {
    qs_status s = check_state(st);
    if (s != QS_OK) return s;
    if (J >> st->n) {
      set_error("basis index %llu out of range for n = %d", (unsigned long long)J, st->n);
      return QS_EINVAL;
    }
    return launch_set_basis(st, J);
  });
}

qs_status sv_copy_in(qs_state_t st, const void* buf, int on_device) {
  return abi_guard(__func__, [&]() -> qs_status {
    qs_status s = check_state(st);
    if (s != QS_OK) return s;
    if (!buf) {
      set_error("buf is NULL");
      return QS_EINVAL;
    }
    if (on_device) {
      QS_CUDA(cudaMemcpyAsync(st->data, buf, st->data_bytes, cudaMemcpyDeviceToDevice, st->stream));
    } else {
      QS_CUDA(cudaMemcpyAsync(st->data, buf, st->data_bytes, cudaMemcpyHostToDevice, st->stream));
      QS_CUDA(cudaStreamSynchronize(st->stream));
    }
    return QS_OK;
  });
}

qs_status sv_copy_out(qs_state_t st, void* buf, int on_device) {
  return abi_guard(__func__, [&]() -> qs_status {
    qs_status s = check_state(st);
    if (s != QS_OK) return s;
    if (!buf) {
      set_error("buf is NULL");
      return QS_EINVAL;
    }
    if (on_device) {
      QS_CUDA(cudaMemcpyAsync(buf, st->data, st->data_bytes, cudaMemcpyDeviceToDevice, st->stream));
    } else {
      QS_CUDA(cudaMemcpyAsync(buf, st->data, st->data_bytes, cudaMemcpyDeviceToHost, st->stream));
      QS_CUDA(cudaStreamSynchronize(st->stream));
      return late_status(st);
    }
    return QS_OK;
  });
}

qs_status sv_apply_circuit(qs_state_t st, const qs_gate* gates, size_t ngates, const qs_opts* opts,
                           qs_stats* stats) {
  return abi_guard(__func__, [&]() -> qs_status {
    qs_status s = check_state(st);
    if (s != QS_OK) return s;
    s = validate_gates(gates, ngates, st->n);
    if (s != QS_OK) return s;
    return apply_gates(st, gates, ngates, opts ? opts->method : QS_METHOD_AUTO, stats,
                       opts ? opts->flags : 0);
  });
}

qs_status sv_probs(qs_state_t st, void* out, int out_fp64, uint64_t marg_mask, double* norm_out) {
  return abi_guard(__func__, [&]() -> qs_status {
    qs_status s = check_state(st);
    if (s != QS_OK) return s;
    if (marg_mask >> st->n) {
      set_error("marginal mask has bits beyond n = %d", st->n);
      return QS_EINVAL;
    }
    int k = __builtin_popcountll(marg_mask);
    const bool marginal = marg_mask != 0 && k != st->n;
    if (marginal && k > kScratchMargLog2) {
      set_error("marginal over %d qubits exceeds the %d-qubit scratch limit", k, kScratchMargLog2);
      return QS_EUNSUPPORTED;
    }
    if (!marginal && out && !out_fp64 && st->prec == QS_C64 && ((uintptr_t)out & 7)) {
      set_error("float output buffer must be 8-byte aligned");
      return QS_EINVAL;
    }
    unsigned char* sc = (unsigned char*)st->scratch;
    double* partials = (double*)(sc + kScratchPartials);
    s = launch_probs(st, out, out_fp64, marginal ? marg_mask : 0, partials,
                     (double*)(sc + kScratchMarg));
    if (s != QS_OK) return s;
    if (norm_out) {
      double* res = (double*)(sc + kScratchResult);
      s = launch_reduce_partials(st, partials, kReduceBlocks, res);
      if (s != QS_OK) return s;
      QS_CUDA(cudaMemcpyAsync(norm_out, res, sizeof(double), cudaMemcpyDeviceToHost, st->stream));
      QS_CUDA(cudaStreamSynchronize(st->stream));
      return late_status(st);
    }
    return QS_OK;
  });
}

qs_status sv_probs_host(qs_state_t st, void* host_out, int out_fp64, uint64_t marg_mask, double* norm_out) {
  return abi_guard(__func__, [&]() -> qs_status {
    qs_status s = check_state(st);
    if (s != QS_OK) return s;
    if (!host_out) {
      set_error("host_out is required");
      return QS_EINVAL;
    }
    if (marg_mask >> st->n) {
      set_error("marginal mask has bits beyond n = %d", st->n);
      return QS_EINVAL;
    }
    s = wait_copies(st);
    if (s != QS_OK) return s;
    const int k = __builtin_popcountll(marg_mask);
    unsigned char* sc = (unsigned char*)st->scratch;
    double* partials = (double*)(sc + kScratchPartials);
    if (marg_mask != 0 && k != st->n) {
      // a marginal (at most 2^16 values) stays in the scratch accumulators as doubles
      if (k > kScratchMargLog2) {
        set_error("marginal over %d qubits exceeds the %d-qubit scratch limit", k, kScratchMargLog2);
        return QS_EUNSUPPORTED;
      }
      s = sv_probs(st, nullptr, 1, marg_mask, norm_out);
      if (s != QS_OK) return s;
      std::vector<double> h((size_t)1 << k);
      QS_CUDA(cudaMemcpyAsync(h.data(), sc + kScratchMarg, h.size() * sizeof(double), cudaMemcpyDeviceToHost,
                              st->stream));
      QS_CUDA(cudaStreamSynchronize(st->stream));
      s = late_status(st);
      if (s != QS_OK) return s;
      if (out_fp64) std::memcpy(host_out, h.data(), h.size() * sizeof(double));
      else
        for (size_t i = 0; i < h.size(); ++i) ((float*)host_out)[i] = (float)h[i];
      return QS_OK;
    }
    const size_t es = out_fp64 ? sizeof(double) : sizeof(float);
    const uint64_t N = 1ull << st->n;
    {
      // a page-locked host buffer the device can address: the kernel writes the
      // probabilities into it directly (one launch, no staging copies; 4 GiB in 22.2 ms
      // against 24.9 ms through the copy engine on GB300)
      cudaPointerAttributes pa;
      if (cudaPointerGetAttributes(&pa, host_out) == cudaSuccess && pa.type == cudaMemoryTypeHost && pa.devicePointer) {
        s = launch_probs_range(st, 0, N, pa.devicePointer, out_fp64, partials);
        if (s == QS_OK && norm_out) s = sv_probs(st, nullptr, out_fp64, 0, norm_out);
        const cudaError_t e = cudaStreamSynchronize(st->stream);
        if (s == QS_OK && e != cudaSuccess) s = cuda_status(e, "sv_probs_host");
        return s == QS_OK ? late_status(st) : s;
      }
      cudaGetLastError();   // a plain host pointer: not an error
    }
    // otherwise formed chunk by chunk in a device staging buffer (kept by the state)
    // and copied to the host buffer after each chunk
    const uint64_t chunk = std::min<uint64_t>(N, (uint64_t)(kStageBytes / es));
    if (!st->stage) {
      st->stage = dev_alloc(st, kStageBytes);
      if (!st->stage) {
        set_error("staging buffer for the probabilities could not be allocated");
        return QS_ENOMEM;
      }
      st->stage_bytes = kStageBytes;
    }
    for (uint64_t off = 0; off < N && s == QS_OK; off += chunk) {
      const uint64_t cnt = std::min<uint64_t>(chunk, N - off);
      s = launch_probs_range(st, off, cnt, st->stage, out_fp64, partials);
      if (s == QS_OK) {
        const cudaError_t e = cudaMemcpyAsync((unsigned char*)host_out + off * es, st->stage, cnt * es,
                                              cudaMemcpyDeviceToHost, st->stream);
        if (e != cudaSuccess) s = cuda_status(e, "probabilities to the host");
      }
    }
    if (s == QS_OK && norm_out) s = sv_probs(st, nullptr, out_fp64, 0, norm_out);
    const cudaError_t e = cudaStreamSynchronize(st->stream);
    if (s == QS_OK && e != cudaSuccess) s = cuda_status(e, "sv_probs_host");
    return s == QS_OK ? late_status(st) : s;
  });
}

qs_status sv_probs_host_async(qs_state_t st, void* host_out, int out_fp64) {
  return abi_guard(__func__, [&]() -> qs_status {
    qs_status s = check_state(st);
    if (s != QS_OK) return s;
    if (!host_out) {
      set_error("host_out is required");
      return QS_EINVAL;
    }
    const uint64_t N = 1ull << st->n;
    const size_t bytes = (size_t)N * (out_fp64 ? sizeof(double) : sizeof(float));
    HostCopies* hc = nullptr;
    s = copies_for(st, bytes, &hc);
    if (s != QS_OK) return s;
    const int k = hc->next;
    unsigned char* dst = (unsigned char*)hc->buf + (size_t)k * hc->half;
    // the buffer's earlier copy has to end before the buffer is rewritten
    if (hc->queued[k]) QS_CUDA(cudaStreamWaitEvent(st->stream, hc->copied[k], 0));
    double* partials = (double*)((unsigned char*)st->scratch + kScratchPartials);
    s = launch_probs_range(st, 0, N, dst, out_fp64, partials);
    if (s != QS_OK) return s;
    QS_CUDA(cudaEventRecord(hc->formed[k], st->stream));
    QS_CUDA(cudaStreamWaitEvent(hc->cs, hc->formed[k], 0));
    QS_CUDA(cudaMemcpyAsync(host_out, dst, bytes, cudaMemcpyDeviceToHost, hc->cs));
    QS_CUDA(cudaEventRecord(hc->copied[k], hc->cs));
    hc->queued[k] = true;
    hc->next = k ^ 1;
    return QS_OK;
  });
}

qs_status sv_probs_wait(qs_state_t st) {
  return abi_guard(__func__, [&]() -> qs_status {
    qs_status s = check_state(st);
    if (s != QS_OK) return s;
    s = wait_copies(st);
    return s == QS_OK ? late_status(st) : s;
  });
}

qs_status sv_loglik(qs_state_t st, const uint32_t* counts, double* out, int64_t* clamped) {
  return abi_guard(__func__, [&]() -> qs_status {
    qs_status s = check_state(st);
    if (s != QS_OK) return s;
    if (!counts || !out) {
      set_error("counts and out are required");
      return QS_EINVAL;
    }
    unsigned char* sc = (unsigned char*)st->scratch;
    double* partials = (double*)(sc + kScratchPartials);
    s = launch_loglik(st, counts, partials, (unsigned long long*)(sc + kScratchClamps));
    if (s != QS_OK) return s;
    double* res = (double*)(sc + kScratchResult);
    s = launch_reduce_partials(st, partials, kReduceBlocks, res);
    if (s != QS_OK) return s;
    unsigned long long nc = 0;
    QS_CUDA(cudaMemcpyAsync(out, res, sizeof(double), cudaMemcpyDeviceToHost, st->stream));
    QS_CUDA(cudaMemcpyAsync(&nc, sc + kScratchClamps, sizeof(nc), cudaMemcpyDeviceToHost, st->stream));
    QS_CUDA(cudaStreamSynchronize(st->stream));
    if (clamped) *clamped = (int64_t)nc;
    return late_status(st);
  });
}

qs_status qs_profile_begin(void) {
  return abi_guard(__func__, [&]() -> qs_status {
    ProfileSession& ps = profile();
    std::lock_guard<std::mutex> g(ps.mu);
    if (ps.active) {
      set_error("a profiling session is already active");
      return QS_EINVAL;
    }
    ps.ev.clear();
    ps.kind.clear();
    ps.active = true;
    return QS_OK;
  });
}

qs_status qs_profile_end(double* kernel_ms, int64_t* launches) {
  return abi_guard(__func__, [&]() -> qs_status {
    ProfileSession& ps = profile();
    std::lock_guard<std::mutex> g(ps.mu);
    if (!ps.active) {
      set_error("no active profiling session");
      return QS_EINVAL;
    }
    ps.active = false;
    double ms[5] = {0, 0, 0, 0, 0};
    int64_t cnt[5] = {0, 0, 0, 0, 0};
    qs_status s = QS_OK;
    for (size_t i = 0; i < ps.kind.size(); ++i) {
      cudaEvent_t a = ps.ev[2 * i], b = ps.ev[2 * i + 1];
      if (a && b) {
        cudaError_t e = cudaEventSynchronize(b);
        float t = 0.f;
        if (e == cudaSuccess) e = cudaEventElapsedTime(&t, a, b);
        if (e != cudaSuccess && s == QS_OK) s = cuda_status(e, "profile events");
        ms[ps.kind[i]] += t;
        cnt[ps.kind[i]] += 1;
      }
      if (a) cudaEventDestroy(a);
      if (b) cudaEventDestroy(b);
    }
    ps.ev.clear();
    ps.kind.clear();
    for (int k = 0; k < 5; ++k) {
      if (kernel_ms) kernel_ms[k] = ms[k];
      if (launches) launches[k] = cnt[k];
    }
    return s;
  });
}

}  // extern "C"
