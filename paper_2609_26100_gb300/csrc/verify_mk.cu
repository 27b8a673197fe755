// Persistent verify kernel: every active layer of a verification step plus the LM head in one
// cooperative launch, one CTA per SM.
//
// The step is a fixed sequence of GEMM phases -- for each layer of the union (ascending):
// QKV, O, gate/up, down; then the LM head -- with the attention of a layer between its QKV and
// O phases.  Each phase is split stream-K over the grid (mk_seg: with whole tiles at the end of a
// phase that has a tile per CTA).  Per CTA:
//
//   warp 0      TMA producer of weight tiles (lane 0).  It walks the whole phase sequence and
//               never waits for activations, so the weight stream does not stop at phase
//               boundaries (it is bounded only by its ring in shared memory).
//   warp 1      tcgen05.mma issuer (lane 0; accumulators in TMEM, up to 8 buffers).
//   warp 2      B-operand producer: for every k-block it waits until the activations it needs
//               are final (flags polled 32 at a time), then lane 0 copies the N x 64 bf16 blocks of
//               every stage that the flags allow, into a ring of their own --
//               bf16(h * g) for QKV / gate-up / LM head, the attention output for O, the SwiGLU
//               activations for down.  (One proxy fence per batch of polls; a fence, a poll test
//               and two 64-bit divisions per stage, with the divisions of the other roles, cost
//               the 7B chain 5 % of its step: 2886 -> 2750 us.)
//   warp 3      attention only.
//   warps 4-7   epilogues (TMEM -> registers, stream-K fix-up, fused op).
// All roles run one loop over the phases; at each O phase (when the attention runs in this
// kernel) the eight warps first run the layer's attention items together, in the ring that every
// role has stopped using by then.
//
// Phases hand data over through global memory and per-tile flags stamped with a sequence
// number that grows monotonically over the step and across steps (seq = epoch*1024 + 8*(slot+1)
// + kind), so flags are never reset.  A consumer waits only for the producer tiles it reads:
// a k-block of QKV / gate-up / LM head needs one 128-feature tile of h; an O k-block needs the
// attention output of one head for every request; a down k-block needs one gate/up tile.
// The RMSNorm is split accordingly: the B operand is bf16(h * g) -- written, for the next norm
// phase, by the epilogue that finalises each 128-feature tile of h -- and the per-row factor
// 1/sqrt(mean(h^2) + eps) is applied to the accumulator in the epilogue, from per-tile partial
// sums of squares written by the same residual epilogues.
//
// Every wait is bounded (2 s by default, TSS_WAIT_LIMIT_MS at context creation); on expiry the
// kernel records TIMEOUT, raises a grid-wide abort word and all roles leave their loops.
#include "attn_body.cuh"

namespace tss {

constexpr int kMkThreads = 256;
constexpr int kMkMaxAcc = 8;  // TMEM accumulator buffers (fewer when N is large)

// Accumulator buffers for an MMA width: a power of two, at most 8, within 512 TMEM columns.
__host__ __device__ inline int mk_acc_bufs(int n_pad) {
  int nb = kMkMaxAcc;
  while (nb > 1 && nb * n_pad > 512) nb >>= 1;
  return nb;
}
constexpr uint32_t kMkWBytes = 128 * 64 * 2;

enum MkKind : int { kMkQkv = 1, kMkAtt = 2, kMkO = 3, kMkGu = 4, kMkDown = 5, kMkLm = 6 };

__device__ __forceinline__ unsigned long long mk_seq(unsigned long long base, int slot, int kind) {
  return base + static_cast<unsigned long long>(slot + 1) * 8ull + static_cast<unsigned long long>(kind);
}

__device__ __forceinline__ unsigned long long ld_acquire_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u64(unsigned long long* p, unsigned long long v) {
  asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}
__device__ __forceinline__ void fence_proxy_async_shared() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// Barrier over `n` threads that also returns the AND of every thread's `v` (uniform result).
__device__ __forceinline__ bool bar_and(int id, int n, bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %3, 0;\n\t"
      "bar.red.and.pred p, %1, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(r)
      : "r"(id), "r"(n), "r"(static_cast<uint32_t>(v))
      : "memory");
  return r != 0;
}

struct MkShared {
  volatile int* abort_s;
  int* abort_g;
  int* status;
  uint64_t limit_ns;  // bound of every wait (create-time setting, 2 s by default)
};

__device__ __forceinline__ bool mk_aborted(const MkShared& sh) {
  if (*sh.abort_s) return true;
  if (*reinterpret_cast<volatile int*>(sh.abort_g)) {
    *sh.abort_s = 1;
    return true;
  }
  return false;
}

__device__ __forceinline__ void mk_fail(const MkShared& sh) {
  *sh.abort_s = 1;
  atomicExch(sh.abort_g, 1);
  report(sh.status, kStatusTimeout);
}

// Bounded wait for *f >= target.
__device__ bool mk_wait_flag(const unsigned long long* f, unsigned long long target, const MkShared& sh) {
  uint64_t t0 = 0;
  for (uint32_t i = 1;; ++i) {
    if (ld_acquire_u64(f) >= target) return true;
    if ((i & 63) == 0) {
      if (mk_aborted(sh)) return false;
      const uint64_t now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      if (now - t0 > sh.limit_ns) {
        mk_fail(sh);
        return false;
      }
    }
    __nanosleep(64);
  }
}

// Bounded wait for the arrival counter *f to reach `target`.
__device__ bool mk_wait_count(const int* f, int target, const MkShared& sh) {
  uint64_t t0 = 0;
  for (uint32_t i = 1;; ++i) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
    if (v >= target) return true;
    if ((i & 63) == 0) {
      if (mk_aborted(sh)) return false;
      const uint64_t now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      if (now - t0 > sh.limit_ns) {
        mk_fail(sh);
        return false;
      }
    }
  }
}

// Bounded mbarrier wait that also leaves when another CTA aborted.
__device__ bool mk_wait_bar(uint64_t* bar, uint32_t parity, const MkShared& sh) {
  // (the clock is read only after a while: its latency would delay the waiting role at every stage)
  uint64_t t0 = 0;
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 255) == 0) {
      if (mk_aborted(sh)) return false;
      const uint64_t now = globaltimer_ns();
      if (t0 == 0) t0 = now;
      if (now - t0 > sh.limit_ns) {
        mk_fail(sh);
        return false;
      }
    }
  }
}

// Every thread of the CTA arrives on `bar` and waits (bounded) for all to arrive; n counts this
// thread's syncs on it (phase parity).
__device__ __forceinline__ bool mk_team_sync(uint64_t* bar, uint32_t& n, const MkShared& sh) {
  mbar_arrive(bar);
  const bool ok = mk_wait_bar(bar, n & 1u, sh);
  ++n;
  return ok;
}

// Position in a ring of n slots: slot and the parity of its current turn, advanced without a
// division (64-bit divisions by the ring size, one per role and stage, had cost about 0.3 us a
// stage).
struct MkRing {
  int s = 0;
  uint32_t turn = 0;
  __device__ __forceinline__ void next(int n) {
    if (++s == n) {
      s = 0;
      turn ^= 1u;
    }
  }
};

struct MkPhase {
  int kind, slot, layer, n_tiles, kb;
};

// Optional timeline (TSS_TRACE): per CTA, per phase, the first and last activity of each role.
// trace[cta][pi * 8 + 2 * role + {0: first, 1: last}], roles 0 weight TMA, 1 B operand, 2 MMA,
// 3 epilogue; the attention of slot j at [kMkTracePhases * 8 + 2j + {0,1}].
constexpr int kMkTracePhases = 4 * kMaxLayers + 1;
constexpr int kMkTraceSub = kMkTracePhases * 8 + 2 * kMaxLayers;  // epilogue sub-steps of a phase's last segment
constexpr int kMkTraceAttn = kMkTraceSub + kMkTracePhases * 8;  // sub-steps of the slot-1 attention item
constexpr int kMkTraceSlots = kMkTraceAttn + 16;
__device__ __forceinline__ void mk_trace(const MkParams& p, int idx) {
  if (p.trace) p.trace[static_cast<size_t>(blockIdx.x) * kMkTraceSlots + idx] = globaltimer_ns();
}

__device__ __forceinline__ MkPhase mk_phase(const MkParams& p, const PlanDev* pl, int pi) {
  MkPhase ph;
  if (pi < 4 * p.n_act) {
    ph.slot = pi >> 2;
    ph.layer = pl->act_layer[ph.slot];
    switch (pi & 3) {
      case 0: ph.kind = kMkQkv; ph.n_tiles = 3 * p.d / 128; ph.kb = p.d / 64; break;
      case 1: ph.kind = kMkO; ph.n_tiles = p.d / 128; ph.kb = p.d / 64; break;
      case 2: ph.kind = kMkGu; ph.n_tiles = p.Ft; ph.kb = p.d / 64; break;
      default: ph.kind = kMkDown; ph.n_tiles = p.d / 128; ph.kb = p.F_pad / 64; break;
    }
  } else {
    ph.kind = kMkLm;
    ph.slot = p.n_act;
    ph.layer = 0;
    ph.n_tiles = p.V_pad / 128;
    ph.kb = p.d / 64;
  }
  return ph;
}

// Pre-tiled weights of a phase's layer (blocks [tile][k-block] of 16 KiB).
__device__ __forceinline__ const __nv_bfloat16* mk_weights(const MkParams& p, const MkPhase& ph) {
  const size_t blocks = static_cast<size_t>(ph.n_tiles) * ph.kb;
  const __nv_bfloat16* base = ph.kind == kMkQkv ? p.w_qkv
                              : ph.kind == kMkO ? p.w_o
                              : ph.kind == kMkGu ? p.w_gu
                              : ph.kind == kMkDown ? p.w_down
                                                   : p.w_lm;
  return base + static_cast<size_t>(ph.layer) * blocks * kTileElems;
}

// CTA c's share of a phase as a sequence of segments (tile t, k-blocks [k0, k1)): stream-K over
// every iteration (tile x k-block) of the phase; or, when the phase has at least one tile per CTA
// and p.dp_tail is set, stream-K over its first n_tiles - G tiles followed by one whole tile per
// CTA, so that the phase ends with whole-tile epilogues (no partial tiles, no arrival counter,
// no reload of other CTAs' partials on its critical tail).  Residual phases keep plain stream-K.
// So do phases of fewer tiles than CTAs, even where a whole tile per CTA is short: it saved the tiny
// decoder's chain 10 of 134 us and four layers of 13B 4 of 955, but one accumulator then sums more
// k-blocks than a split tile's did and loses more low bits (error of the logits against 64 bits 0.4 %
// and 2 % larger), and as many accumulators as parts took longer than splitting (145 us).
// (32-bit arithmetic: T x #SMs is at most 152 / 8192 of a matrix's elements, below 2^32 for any
// matrix that fits the device; 64-bit divisions took a role about a microsecond a phase)
struct MkSeg {
  uint32_t it, it1;  // stream-K iterations of this CTA still to take
  uint32_t T;        // stream-K iterations of the phase (the fix-up contributor arithmetic)
  uint32_t geff;     // CTAs sharing them
  int kb, whole;     // this CTA's whole tile after them, -1: none
  __device__ __forceinline__ bool next(int& t, int& k0, int& k1);
  __device__ __forceinline__ bool done() const { return it >= it1 && whole < 0; }
};

__device__ __forceinline__ MkSeg mk_seg(const MkParams& p, const MkPhase& ph, int c, int G) {
  MkSeg s;
  s.kb = ph.kb;
  s.whole = -1;
  int n_split = ph.n_tiles;
  if (p.dp_tail && ph.n_tiles >= G && ph.kind != kMkO && ph.kind != kMkDown) {
    n_split = ph.n_tiles - G;
    s.whole = n_split + c;
  }
  s.T = static_cast<uint32_t>(n_split) * ph.kb;
  s.geff = min(s.T, static_cast<uint32_t>(G));
  if (static_cast<uint32_t>(c) >= s.geff) {
    s.it = s.it1 = 0;
  } else {
    s.it = s.T * c / s.geff;
    s.it1 = s.T * (c + 1) / s.geff;
  }
  return s;
}

// The CTA whose range holds stream-K iteration i.
__device__ __forceinline__ int mk_cta_of(uint32_t i, uint32_t T, uint32_t G) {
  return static_cast<int>(((i + 1) * G - 1) / T);
}

__device__ __forceinline__ bool MkSeg::next(int& t, int& k0, int& k1) {
  if (it < it1) {
    t = static_cast<int>(it / kb);
    const uint32_t t0 = static_cast<uint32_t>(t) * kb;
    k0 = static_cast<int>(it - t0);
    it = min(it1, t0 + kb);
    k1 = static_cast<int>(it - t0);
    return true;
  }
  if (whole < 0) return false;
  t = whole;
  k0 = 0;
  k1 = kb;
  whole = -1;
  return true;
}

// Slot whose compacted rows feed a phase (the LM head runs on all rows).
__device__ __forceinline__ int mk_row_slot(const MkPhase& ph) { return ph.kind == kMkLm ? kFinalSlot : ph.slot; }

// Sequence number h must have reached before a norm phase reads it (0: the embedding, i.e. the
// previous kernel, which has completed when this kernel starts).
__device__ __forceinline__ unsigned long long mk_h_dep(const MkParams& p, const MkPhase& ph) {
  if (ph.kind == kMkQkv) return ph.slot == 0 ? 0ull : mk_seq(p.seq_base, ph.slot - 1, kMkDown);
  if (ph.kind == kMkGu) return mk_seq(p.seq_base, ph.slot, kMkO);
  return p.n_act == 0 ? 0ull : mk_seq(p.seq_base, p.n_act - 1, kMkDown);  // LM head
}

// Accumulator values of tokens [16 ch, 16 ch + 16) of this thread's output row: W.hi + W.lo
// (the two parts are separate columns of one MMA when xs.parts == 1, already summed otherwise).
__device__ __forceinline__ void mk_acc_tokens(uint32_t tb, int ch, const XsLayout& xs, float* v) {
  if (xs.parts == 2) {
    tmem_ld16(tb + ch * 16, v);
  } else if (xs.half == 8) {  // up to 8 tokens: hi in columns 0..7, lo in 8..15
    float r[16];
    tmem_ld16(tb, r);
#pragma unroll
    for (int jj = 0; jj < 8; ++jj) {
      v[jj] = r[jj] + r[8 + jj];
      v[8 + jj] = 0.f;
    }
  } else {
    float lo[16];
    tmem_ld16(tb + ch * 16, v);
    tmem_ld16(tb + xs.half + ch * 16, lo);
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) v[jj] += lo[jj];
  }
}

struct MkEpi {
  int M;
  const int* rows;  // shared-memory copy of the phase's compacted row list
  int* pos;         // [kMaxRows] RoPE position of each compacted row (QKV); LM head: its row in the caller's logits
  int* kvslot;      // [kMaxRows] KV-cache slot and row of each compacted row (QKV)
  int* kvrow;
  // residual phases: the next norm phase's B operand bf16(h * g_next) is written by the epilogue
  // that updates h.  npos[j]: compacted row j's place in the next phase, -1 if it skips it; the next
  // phase's rows that this phase does not run (h unchanged) are nrows[x] >= 0 at place x.
  int nM, n_extra;
  const int* npos;
  const int* nrows;
  const float* gnext;  // RMSNorm gain of the next norm phase
  float* xch;    // [16][128]
  float* rs;     // [kMaxRows] per-row RMSNorm factors of the current phase
  const float* rcos;  // [16][D/2] RoPE cos / sin of the first 16 rows (QKV), staged at phase start
  const float* rsin;
  // values the epilogues would otherwise load from the step descriptor in global memory
  __nv_bfloat16* kv_base;  // QKV: this layer's KV cache
  size_t kv_cap;
  float* logits;           // LM head: caller's logits or null
  bool logits_vec;         // ... and whether 16-byte stores fit its rows
  int q, lane, et;
};

// Wait until every 128-feature tile of h has reached `dep`, then compute the RMSNorm factors of
// the phase's rows from the partial sums of squares (fixed order, deterministic).
__device__ bool mk_prepare_rs(const MkParams& p, const MkEpi& e, unsigned long long dep, const MkShared& sh) {
  const int nt = p.d / 128;
  bool ok = true;
  for (int t = e.et; dep != 0ull && t < nt && ok; t += 128) ok = mk_wait_flag(&p.hflag[t], dep, sh);
  if (!bar_and(1, 128, ok)) return false;
  for (int j = e.et; j < e.M; j += 128) {
    const int m = e.rows[j];
    float ss = 0.f;
#pragma unroll 8
    for (int t = 0; t < nt; ++t) ss += __ldcg(&p.ssp[static_cast<size_t>(t) * kMaxRows + m]);
    e.rs[j] = rsqrtf(ss / static_cast<float>(p.d) + p.eps);
  }
  named_bar_sync(1, 128);
  return true;
}

// Sums of G values per lane over the warp's 32 lanes, G a power of two: the values are halved
// between lane pairs first (G - 1 shuffles), then one value each remains to be summed.  Lane l ends
// with the sum of value l & (G - 1).
template <int G>
__device__ __forceinline__ float warp_sums(const float* x, int lane) {
  float y[G];
#pragma unroll
  for (int i = 0; i < G; ++i) y[i] = x[i];
#pragma unroll
  for (int w = G / 2; w >= 1; w >>= 1) {
    const bool up = lane & w;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float give = up ? y[i] : y[i + w];
      y[i] = (up ? y[i + w] : y[i]) + __shfl_xor_sync(0xffffffffu, give, w);
    }
  }
  float r = y[0];
#pragma unroll
  for (int w = G; w < 32; w <<= 1) r += __shfl_xor_sync(0xffffffffu, r, w);
  return r;
}

__device__ __forceinline__ bool mk_resid(const MkPhase& ph) { return ph.kind == kMkO || ph.kind == kMkDown; }

// Finishes rows of output tile t: the fused epilogue of the phase on the tile's fp32 sums.  A
// unit is G rows; a warp takes units u0, u0 + du, ... below n_units and each lane 4 adjacent
// features of all 128, so that the partner elements of RoPE and SwiGLU and the reductions over
// the tile's features (sums of squares, argmax) stay within one warp and every load and store is
// a 16- or 8-byte vector.  The sums are
//   whole: the accumulator in this CTA's tensor memory, read 4 G rows at a time (thread = feature)
//          and turned around through shared memory; u0 = warp, du = 4, every warp the same number
//          of turns; the accumulator buffer is released after the last read;
//   else:  the partials of contributors cf..cl, added in that order (deterministic), CB of them per
//          round of loads.
// Bound: issue of one warp per scheduler (a row's exponentials, divisions, splits and shuffles) and,
// for partials, one L2 round trip per round.  In row form a 61-row whole tile of gate/up takes
// 5.3 us and a 6-row one 1.4 us (9.8 and 2.3 us with a division and an address computation per
// element and a barrier pair per 16 rows of one thread per feature).
template <int D, int G, int CB>
__device__ void mk_finish_rows(const MkParams& p, const MkPhase& ph, const MkEpi& e, int t, bool whole, uint32_t tb,
                               uint64_t* acce, int u0, int du, int cf, int cl, const float* partials, int n_pad) {
  const int lane = e.lane, f0 = 4 * lane;  // features f0 .. f0 + 3 of the tile
  const int n_units = (e.M + G - 1) / G;
  const int n_it = whole ? (n_units + 3) >> 2 : (n_units - u0 + du - 1) / du;
  const bool resid = mk_resid(ph);
  constexpr int half = D / 2;
  const int d = p.d;
  const int sec = ph.kind != kMkQkv || t * 128 < d ? 0 : t * 128 < 2 * d ? 1 : 2;  // QKV: q, k or v (one per tile)
  const int fs = t * 128 + f0 - sec * d;
  const int head = fs / D, dim0 = fs % D;
  float4 gn = make_float4(0.f, 0.f, 0.f, 0.f);
  if (resid) gn = *reinterpret_cast<const float4*>(e.gnext + t * 128 + f0);
  const SplitAt xat = resid ? split_at(p.xn, p.xs, t * 128 + f0) : split_at(p.act, p.xs, t * 64 + (f0 & 63));
  for (int it = 0; it < n_it; ++it) {
    const int j0 = (u0 + it * du) * G;
    // residual phases: h; QKV: the rotation factors -- requested before the sums
    float4 ha[G], hb[G];
#pragma unroll
    for (int jj = 0; jj < G; ++jj) {
      const int j = j0 + jj;
      ha[jj] = hb[jj] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j < e.M) {
        if (resid) {
          ha[jj] = __ldcg(reinterpret_cast<const float4*>(p.h + static_cast<size_t>(e.rows[j]) * d + t * 128 + f0));
        } else if (ph.kind == kMkQkv && sec < 2) {
          const int ii = dim0 & (half - 1);
          if (j < 16) {
            ha[jj] = *reinterpret_cast<const float4*>(e.rcos + j * half + ii);
            hb[jj] = *reinterpret_cast<const float4*>(e.rsin + j * half + ii);
          } else {
            const size_t pe = static_cast<size_t>(e.pos[j]) * half + ii;
            ha[jj] = __ldg(reinterpret_cast<const float4*>(p.rope_cos + pe));
            hb[jj] = __ldg(reinterpret_cast<const float4*>(p.rope_sin + pe));
          }
        }
      }
    }
    float v[G][4];
    if (whole) {
      const int r = e.q * 32 + lane;
      float a[16];
      mk_acc_tokens(tb, it, p.xs, a);
      if (it == n_it - 1) {
        tc_fence_before();
        mbar_arrive(acce);
      }
#pragma unroll
      for (int jj = 0; jj < 4 * G; ++jj) e.xch[jj * 128 + r] = a[jj];
      named_bar_sync(1, 128);
#pragma unroll
      for (int jj = 0; jj < G; ++jj) {
        const float4 x = *reinterpret_cast<const float4*>(e.xch + (e.q * G + jj) * 128 + f0);
        v[jj][0] = x.x; v[jj][1] = x.y; v[jj][2] = x.z; v[jj][3] = x.w;
      }
      if (it < n_it - 1) named_bar_sync(1, 128);  // (after the last turn the caller's barrier follows)
    } else {
#pragma unroll
      for (int jj = 0; jj < G; ++jj) v[jj][0] = v[jj][1] = v[jj][2] = v[jj][3] = 0.f;
      for (int c0 = cf; c0 <= cl; c0 += CB) {
        float4 a[CB][G];
#pragma unroll
        for (int q = 0; q < CB; ++q) {
          const bool cin = c0 + q <= cl;
          const float* pa = partials + static_cast<size_t>(c0 + q + t) * 128 * n_pad;
#pragma unroll
          for (int jj = 0; jj < G; ++jj)
            a[q][jj] = cin && j0 + jj < e.M ? __ldcg(reinterpret_cast<const float4*>(pa + (j0 + jj) * 128 + f0))
                                            : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int q = 0; q < CB; ++q)
#pragma unroll
          for (int jj = 0; jj < G; ++jj) {
            v[jj][0] += a[q][jj].x;
            v[jj][1] += a[q][jj].y;
            v[jj][2] += a[q][jj].z;
            v[jj][3] += a[q][jj].w;
          }
      }
    }
    if (ph.kind == kMkQkv) {
#pragma unroll
      for (int jj = 0; jj < G; ++jj) {
        const int j = j0 + jj;
        const bool in = j < e.M;  // uniform over the warp
        const float rsj = in ? e.rs[j] : 0.f;
        float val[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) val[i] = v[jj][i] * rsj;
        if (sec < 2) {  // rotate-half RoPE: the partner feature dim ^ half sits in lane ^ half / 4
          const float cs[4] = {ha[jj].x, ha[jj].y, ha[jj].z, ha[jj].w}, sn[4] = {hb[jj].x, hb[jj].y, hb[jj].z, hb[jj].w};
          float rot[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float pv = __shfl_xor_sync(0xffffffffu, val[i], half >> 2);
            rot[i] = dim0 < half ? val[i] * cs[i] - pv * sn[i] : val[i] * cs[i] + pv * sn[i];
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) val[i] = rot[i];
        }
        if (in) {
          if (sec == 0) {  // q in fp16 (11 significant bits), split exactly into bf16 hi + lo by the attention
            const uint32_t w0 = pack_f16(val[0], val[1]), w1 = pack_f16(val[2], val[3]);
            *reinterpret_cast<uint2*>(reinterpret_cast<__half*>(p.qbuf) + static_cast<size_t>(j) * d + fs) =
                make_uint2(w0, w1);
          } else {
            const size_t off = ((static_cast<size_t>(e.kvslot[j]) * 2 + (sec - 1)) * p.H + head) * e.kv_cap + e.kvrow[j];
            *reinterpret_cast<uint2*>(e.kv_base + off * D + dim0) =
                make_uint2(pack_bf16(val[0], val[1]), pack_bf16(val[2], val[3]));
          }
        }
      }
    } else if (resid) {  // residual add, the rows' partial sums of squares, the next phase's B operand
      float sq[G];
#pragma unroll
      for (int jj = 0; jj < G; ++jj) {
        const int j = j0 + jj;
        const float nv[4] = {ha[jj].x + v[jj][0], ha[jj].y + v[jj][1], ha[jj].z + v[jj][2], ha[jj].w + v[jj][3]};
        sq[jj] = (nv[0] * nv[0] + nv[1] * nv[1]) + (nv[2] * nv[2] + nv[3] * nv[3]);
        if (j < e.M) {
          const int m = e.rows[j], np = e.npos[j];
          *reinterpret_cast<float4*>(p.h + static_cast<size_t>(m) * d + t * 128 + f0) =
              make_float4(nv[0], nv[1], nv[2], nv[3]);
          if (np >= 0) {
            const float xg[4] = {nv[0] * gn.x, nv[1] * gn.y, nv[2] * gn.z, nv[3] * gn.w};
            store_split4(xat, np, xg);
          }
        }
      }
      const float sum = warp_sums<G>(sq, lane);
      if (lane < G && j0 + lane < e.M) p.ssp[static_cast<size_t>(t) * kMaxRows + e.rows[j0 + lane]] = sum;
    } else if (ph.kind == kMkGu) {
      // lanes 0-15 hold gate features, lanes 16-31 the matching up features: of two rows the lower
      // half-warp finishes the first and the upper the second (one exchange, one division per value)
#pragma unroll
      for (int jj = 0; jj < G; jj += 2) {
        const bool upper = lane >= 16;
        const int ja = j0 + jj, jb = ja + 1, j = upper ? jb : ja;
        const float ra = ja < e.M ? e.rs[ja] : 0.f, rb = jb < e.M ? e.rs[jb] : 0.f;
        float act[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float xa = v[jj][i] * ra, xb = v[jj + 1][i] * rb;
          const float y = __shfl_xor_sync(0xffffffffu, upper ? xa : xb, 16);
          const float g = upper ? y : xa, u = upper ? xb : y;
          act[i] = silu(g) * u;
        }
        if (j < e.M) store_split4(xat, j, act);
      }
    } else {  // LM head: logits and the tile's argmax of each row, lowest index on ties
      const int o0 = t * 128 + f0;
#pragma unroll
      for (int jj = 0; jj < G; ++jj) {
        const int j = j0 + jj;
        const bool in = j < e.M;
        const float rsj = in ? e.rs[j] : 0.f;
        float bv = -INFINITY;
        int bi = o0;
        float val[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const bool on = o0 + i < p.V && in;
          val[i] = on ? v[jj][i] * rsj : -INFINITY;
          if (on && val[i] != val[i]) report(p.status, kStatusCheck);
          if (val[i] > bv) {
            bv = val[i];
            bi = o0 + i;
          }
        }
        if (e.logits && in) {
          float* lg = e.logits + static_cast<size_t>(e.pos[j]) * p.V + o0;
          if (e.logits_vec) {  // (V is a multiple of 4: all four features exist, or none)
            if (o0 < p.V) *reinterpret_cast<float4*>(lg) = make_float4(val[0], val[1], val[2], val[3]);
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (o0 + i < p.V) lg[i] = val[i];
          }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
          const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
          if (ov > bv || (ov == bv && oi < bi)) {
            bv = ov;
            bi = oi;
          }
        }
        if (in && lane == 0) {
          p.amax_val[static_cast<size_t>(t) * kMaxRows + e.rows[j]] = bv;
          p.amax_idx[static_cast<size_t>(t) * kMaxRows + e.rows[j]] = bi;
        }
      }
    }
  }
  // residual phases: the next phase's rows that skip this layer (mixed skip sets), a warp each
  if (resid && e.n_extra > 0) {
    for (int x = u0; x < e.nM; x += du) {
      const int m = e.nrows[x];
      if (m < 0) continue;
      const float4 hv = __ldcg(reinterpret_cast<const float4*>(p.h + static_cast<size_t>(m) * d + t * 128 + f0));
      const float xg[4] = {hv.x * gn.x, hv.y * gn.y, hv.z * gn.z, hv.w * gn.w};
      store_split4(xat, x, xg);
    }
  }
}

// The plan slot whose rows the next norm phase runs (O -> gate/up of the same layer; down -> QKV
// of the next layer, or the LM head).
__device__ __forceinline__ int mk_next_slot(const MkParams& p, const MkPhase& ph) {
  if (ph.kind == kMkO) return ph.slot;
  return ph.slot + 1 < p.n_act ? ph.slot + 1 : kFinalSlot;
}

__device__ __forceinline__ unsigned long long* mk_tile_flag(const MkParams& p, int kind, int t) {
  switch (kind) {
    case kMkQkv: return p.qkvflag + t;
    case kMkGu: return p.guflag + t;
    case kMkO:
    case kMkDown: return p.hflag + t;
    default: return nullptr;
  }
}

// The attention of QKV slot `slot` in this CTA: its (request, head, split) items round-robin over
// the grid, each run by all 256 threads of the CTA (team thread ttid; the epilogue warps are
// 0..127) in the weight / activation ring, which every role has stopped using when it enters:
// the epilogue warps after the slot's QKV epilogues, the other warps before their O phase.
// Returns false after a failed wait (the kernel is aborting).
template <int D>
__device__ __forceinline__ bool mk_team_attention(const MkParams& p, const AttnParams& ap0, int slot, int ttid,
                                               uint8_t* ring, size_t ring_bytes, float (*sM)[16], float (*sL)[16],
                                               int* s_last, uint64_t* team, uint32_t& team_n, const MkShared& sh) {
  if (!mk_team_sync(team, team_n, sh)) return false;
  const PlanDev* pl = p.plan;
  AttnParams ap = ap0;
  ap.slot = slot;
  const int c = blockIdx.x, G = gridDim.x;
  const int per_req = p.H * p.attn_splits, n_items = p.B * per_req;
  const unsigned long long want = mk_seq(p.seq_base, slot, kMkQkv);
  if (ttid == 0) mk_trace(p, kMkTracePhases * 8 + 2 * slot);
  fence_proxy_async_shared();  // the ring's async-proxy (TMA / MMA) use ends before generic use
  bool ok = true;
  for (int item = c; ok && item < n_items; item += G) {
    const int b = item / per_req;
    const int head = (item - b * per_req) / p.attn_splits;
    const int split = item - b * per_req - head * p.attn_splits;
    if (pl->slot_crow[slot][b] < 0) continue;
    // the Q, K and V tiles of this head (written by the QKV epilogues of this step)
    auto wait_inputs = [&]() -> bool {
      bool good = true;
      if (ttid < 3) {
        const int tile = (ttid * p.d + head * D) / 128;
        good = mk_wait_flag(&p.qkvflag[tile], want, sh);
      }
      return bar_and(2, kMkThreads, good);
    };
    unsigned long long* atr =
        p.trace && slot == 1 ? p.trace + static_cast<size_t>(blockIdx.x) * kMkTraceSlots + kMkTraceAttn : nullptr;
    bool failed = false;
    const bool wrote = attention_item_resident<D, 2, kMkThreads>(ap, split, head, b, ttid, ring, ring_bytes, sM, sL,
                                                                  s_last, atr, wait_inputs, failed, p.attn_plo != 0);
    if (failed) {
      ok = false;
      break;
    }
    if (wrote) {
      named_bar_sync(2, kMkThreads);  // the head's output precedes the flag's release
      if (ttid == 0) st_release_u64(&p.attflag[b * p.H + head], mk_seq(p.seq_base, slot, kMkAtt));
    }
    named_bar_sync(2, kMkThreads);
  }
  if (ttid == 0) mk_trace(p, kMkTracePhases * 8 + 2 * slot + 1);
  fence_proxy_async_shared();  // generic-proxy use of the ring ends before the next TMA writes
  return mk_team_sync(team, team_n, sh) && ok;
}

template <int D>
__global__ void __launch_bounds__(kMkThreads, 1)
    verify_mk_kernel(const MkParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int S = p.stages, SX = p.x_stages, n_pad = p.n_pad, KPS = p.kps, XPS = p.xps;
  const int XP = p.xs.parts;
  const uint32_t x_bytes = static_cast<uint32_t>(n_pad) * 128u;  // one block of one k-block of the B operand
  const uint32_t sw_bytes = KPS * kMkWBytes, sx_bytes = XPS * XP * x_bytes;
  uint8_t* sW = base;
  uint8_t* sX = sW + static_cast<size_t>(S) * sw_bytes;
  uint8_t* s_attn = sX + static_cast<size_t>(SX) * sx_bytes;
  uint64_t* fullw = reinterpret_cast<uint64_t*>(s_attn + p.attn_extra);
  uint64_t* emptyw = fullw + S;
  uint64_t* fullx = emptyw + S;
  uint64_t* emptyx = fullx + SX;
  uint64_t* accf = emptyx + SX;
  uint64_t* acce = accf + kMkMaxAcc;
  uint64_t* team = acce + kMkMaxAcc;  // all 256 threads: entry to / exit from a layer's attention
  int* misc = reinterpret_cast<int*>(team + 1);  // [0] tmem addr, [1] abort, [5] s_last
  // (16-byte vectors from here on: the mbarriers before are an odd number of 8-byte words)
  float* xch = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(misc + 16) + 15) & ~uintptr_t(15));
  int* s_pend = reinterpret_cast<int*>(xch + 16 * 128);  // [2][4] split tiles of this CTA's phase: t, cf, cl, complete
  float* rs = reinterpret_cast<float*>(s_pend + 128);
  float (*sM)[16] = reinterpret_cast<float (*)[16]>(rs + kMaxRows);  // [8][16] per attention warp
  float (*sL)[16] = reinterpret_cast<float (*)[16]>(rs + kMaxRows + 128);
  // [kMaxRows] x 5: rows, pos (residual phases: places in the next phase), kv slot, kv row, next rows
  int* s_rows = reinterpret_cast<int*>(rs + kMaxRows + 256);
  int* s_pos = s_rows + kMaxRows;
  int* s_kvslot = s_pos + kMaxRows;
  int* s_kvrow = s_kvslot + kMaxRows;
  int* s_nrows = s_kvrow + kMaxRows;
  float* s_rope = reinterpret_cast<float*>(s_nrows + kMaxRows);  // [2][16][64]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int NB = mk_acc_bufs(n_pad);
  const uint32_t ncols = gemm_tmem_cols(n_pad, NB);
  const PlanDev* pl = p.plan;
  const size_t ring_attn_bytes = static_cast<size_t>(s_attn - base) + p.attn_extra;
  MkShared sh;
  sh.abort_s = reinterpret_cast<volatile int*>(misc + 1);
  sh.abort_g = p.abort_word;
  sh.status = p.status;
  sh.limit_ns = p.wait_ns;

  if (threadIdx.x == 0) {
    for (int i = 0; i < S; ++i) {
      mbar_init(&fullw[i], 1);
      mbar_init(&emptyw[i], 1);
    }
    for (int i = 0; i < SX; ++i) {
      mbar_init(&fullx[i], 1);
      mbar_init(&emptyx[i], 1);
    }
    for (int i = 0; i < kMkMaxAcc; ++i) {
      mbar_init(&accf[i], 1);
      mbar_init(&acce[i], 128);
    }
    mbar_init(team, kMkThreads);
    *sh.abort_s = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(reinterpret_cast<uint32_t*>(misc), ncols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = static_cast<uint32_t>(misc[0]);
  griddep_wait();  // the controller's plan and the embedding are complete

  const int G = gridDim.x, c = blockIdx.x;
  // A host/device disagreement on the layer union (reported by the controller) runs nothing.
  const int n_phases = pl->n_act == p.n_act ? min(4 * p.n_act + 1, p.ph_end) : 0;
  const int ph0 = p.ph_begin;

  // The attention inside this kernel (not with attn_external): every warp joins the team that runs
  // a layer's attention items -- the epilogue warps after the layer's QKV phase, the others before
  // its O phase.
  AttnParams ap{};
  ap.n_splits = p.attn_splits;
  ap.n_heads = p.H;
  ap.d_model = p.d;
  ap.head_dim = D;
  ap.scale_log2 = p.scale_log2;
  ap.plan = pl;
  ap.step = p.step;
  ap.q = p.qbuf;
  ap.o = p.obuf;
  ap.o_xs = p.xs;
  ap.part_o = p.attn_po;
  ap.part_ml = p.attn_pml;
  ap.counters = p.attn_cnt;
  ap.status = p.status;
  uint32_t team_n = 0;
  auto team_attention = [&](int slot) -> bool {
    return mk_team_attention<D>(p, ap, slot, static_cast<int>(threadIdx.x) ^ 128, base, ring_attn_bytes, sM, sL,
                                misc + 5, team, team_n, sh);
  };

  // Roles, all in one loop over the phases: warp 0 lane 0 streams the weights, warp 1 lane 0
  // issues the MMAs, warp 2 loads the B operands, warps 4-7 run the epilogues; at each O phase
  // (inside this kernel's attention) all eight warps first run the layer's attention as one team.
  const uint64_t wpol = l2_policy_evict_first();
  const uint32_t idesc = idesc_bf16_m128(n_pad);
  MkRing rw, rx;  // this role's positions in the weight and B-operand rings
  MkRing use;     // ... and in the accumulator buffers
  bool ok = true;
  MkEpi e;
  e.q = warp & 3;
  e.lane = lane;
  e.et = threadIdx.x - 128;
  e.xch = xch;
  e.rs = rs;
  e.rcos = s_rope;
  e.rsin = s_rope + 16 * 64;
  const int r = e.q * 32 + lane;
  // the weight stages of this CTA's share of a phase: warp 0 lane 0 issues their bulk copies into
  // the ring (it never waits for activations, only for free ring stages)
  auto produce = [&](const MkPhase& ph, int pi) -> bool {
    MkSeg seg = mk_seg(p, ph, c, G);
    const __nv_bfloat16* wl = mk_weights(p, ph);
    int t, k0, k1, j = 0;
    while (seg.next(t, k0, k1)) {
      const bool last_seg = seg.done();
      for (int kc = k0; kc < k1; kc += KPS, ++j) {
        const int nk = min(KPS, k1 - kc);
        const int s = rw.s;
        if (!mk_wait_bar(&emptyw[s], rw.turn ^ 1u, sh)) return false;
        if (j == 0) mk_trace(p, pi * 8 + 0);
        if (last_seg && kc + nk == k1) mk_trace(p, pi * 8 + 1);
        mbar_arrive_expect_tx(&fullw[s], nk * kMkWBytes);
        if (p.w_evict_first)
          bulk_load_hint(sW + static_cast<size_t>(s) * sw_bytes,
                         wl + (static_cast<size_t>(t) * ph.kb + kc) * kTileElems, nk * kMkWBytes, &fullw[s], wpol);
        else
          bulk_load(sW + static_cast<size_t>(s) * sw_bytes,
                    wl + (static_cast<size_t>(t) * ph.kb + kc) * kTileElems, nk * kMkWBytes, &fullw[s]);
        rw.next(S);
      }
    }
    return true;
  };
  for (int pi = ph0; ok && pi < n_phases; ++pi) {
    const MkPhase ph = mk_phase(p, pl, pi);
    if (ph.kind == kMkO && !p.attn_external) {
      // this layer's attention: the epilogue warps come after the QKV epilogues (every QKV MMA of
      // this CTA has completed), the other warps before they start the O phase
      const bool t = team_attention(ph.slot);
      ok = warp >= 4 ? bar_and(1, 128, t) : __shfl_sync(0xffffffffu, t, 0);
      if (!ok) break;
    }
    if (warp == 0) {
      // ---------------- weight TMA producer (lane 0): never waits for activations ----------------
      bool good = true;
      if (lane == 0) good = produce(ph, pi);
      ok = __shfl_sync(0xffffffffu, good, 0);
    } else if (warp == 1) {
      // ---------------- MMA issuer (lane 0) ----------------
      if (lane == 0) {
        MkSeg seg = mk_seg(p, ph, c, G);
        int t, k0, k1;
        bool first = true;
        while (ok && seg.next(t, k0, k1)) {
          const int buf = use.s;
          if (!mk_wait_bar(&acce[buf], use.turn ^ 1u, sh)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(buf * n_pad);
          for (int kc = k0; ok && kc < k1; kc += KPS, rw.next(S)) {
            const int nk = min(KPS, k1 - kc);
            const int s = rw.s;
            if (!mk_wait_bar(&fullw[s], rw.turn, sh)) {
              ok = false;
              break;
            }
            for (int jx = 0; jx < nk; jx += XPS, rx.next(SX)) {
              const int sx = rx.s;
              if (!mk_wait_bar(&fullx[sx], rx.turn, sh)) {
                ok = false;
                break;
              }
              tc_fence_after();
              if (first) mk_trace(p, pi * 8 + 4);
              first = false;
              for (int j = jx; j < min(jx + XPS, nk); ++j) {
                const uint32_t a0 = smem_u32(sW + static_cast<size_t>(s) * sw_bytes + j * kMkWBytes);
                const uint32_t b0 = smem_u32(sX + static_cast<size_t>(sx) * sx_bytes + (j - jx) * XP * x_bytes);
                // (branch outside the issue loops: a conditional MMA inside them was measured to
                // slow every stage down)
                if (XP == 1) {
#pragma unroll
                  for (int k16 = 0; k16 < 4; ++k16)
                    umma_bf16(d_tmem, sdesc_sw128(a0 + k16 * 32), sdesc_sw128(b0 + k16 * 32), idesc,
                              (kc + j > k0 || k16 > 0) ? 1u : 0u);
                } else {  // the lo block accumulates into the same columns
#pragma unroll
                  for (int k16 = 0; k16 < 4; ++k16) {
                    umma_bf16(d_tmem, sdesc_sw128(a0 + k16 * 32), sdesc_sw128(b0 + k16 * 32), idesc,
                              (kc + j > k0 || k16 > 0) ? 1u : 0u);
                    umma_bf16(d_tmem, sdesc_sw128(a0 + k16 * 32), sdesc_sw128(b0 + x_bytes + k16 * 32), idesc, 1u);
                  }
                }
              }
              umma_commit(&emptyx[sx]);
            }
            umma_commit(&emptyw[s]);
          }
          if (!ok) break;
          umma_commit(&accf[buf]);
          if (seg.done()) mk_trace(p, pi * 8 + 5);
          use.next(NB);
        }
      }
      ok = __shfl_sync(0xffffffffu, ok, 0);
    } else if (warp == 2) {
      // ---------------- B-operand producer: TMA after the producing tiles are flagged ----------------
      MkSeg seg = mk_seg(p, ph, c, G);
      if (seg.done()) continue;
      // dependency index space of this phase: h tiles, heads, or gate/up tiles
      const unsigned long long* flags;
      unsigned long long want;
      int n_dep;
      if (ph.kind == kMkO) {
        flags = p.attflag;
        want = p.attn_external ? 0ull : mk_seq(p.seq_base, ph.slot, kMkAtt);  // else: an earlier launch
        n_dep = p.H;
      } else if (ph.kind == kMkDown) {
        flags = p.guflag;
        want = mk_seq(p.seq_base, ph.slot, kMkGu);
        n_dep = p.Ft;
      } else {
        flags = p.hflag;
        want = mk_h_dep(p, ph);
        n_dep = p.d / 128;
      }
      const __nv_bfloat16* xsrc = ph.kind == kMkO ? p.obuf : ph.kind == kMkDown ? p.act : p.xn;
      uint32_t ready[17] = {};  // known-complete dependency indices below 512 (others are polled each time)
      // one flag index is complete when every request that runs the slot has it (attention) or
      // the single flag reached `want`
      auto poll = [&](int x) -> bool {
        if (ph.kind != kMkO) return ld_acquire_u64(&flags[x]) >= want;
        for (int b = 0; b < p.B; ++b)
          if (pl->slot_crow[ph.slot][b] >= 0 && ld_acquire_u64(&flags[b * p.H + x]) < want) return false;
        return true;
      };
      // dependency index of a k-block, and the first k-block after those of index x
      auto dep = [&](int kk) { return ph.kind == kMkO ? kk * 64 / D : ph.kind == kMkDown ? kk : kk >> 1; };
      auto dep_end = [&](int x) { return ph.kind == kMkO ? (x + 1) * D / 64 : ph.kind == kMkDown ? x + 1 : 2 * (x + 1); };
      int t, k0, k1;
      bool first = true;
      while (ok && seg.next(t, k0, k1)) {
        const bool last_seg = seg.done();
        int kc = k0, kr = want == 0ull ? k1 : k0;  // k-blocks below kr are known to be complete
        while (ok && kc < k1) {
          // the whole warp: extend kr over the next stage, or as far as the flags already go
          const int need = min(kc + XPS, k1);
          while (ok && kr < need) {
            const int x = dep(kr);
            if (x < 512 && ((ready[x >> 5] >> (x & 31)) & 1u)) {
              kr = dep_end(x);
              continue;
            }
            // poll x .. x+31 at once; then wait (bounded) for x itself if it is not there yet
            const int y = x + lane;
            const uint32_t bal = __ballot_sync(0xffffffffu, y < n_dep && poll(y));
            __syncwarp();  // memory ordering: lane 0's copies follow the acquire loads of the others
            if (x < 512) {
              ready[x >> 5] |= bal << (x & 31);
              if (x & 31) ready[(x >> 5) + 1] |= bal >> (32 - (x & 31));
            }
            if (bal & 1u) {
              kr = dep_end(x + __ffs(~bal | 0x80000000u) - 2);
            } else {
              bool got = true;
              if (lane == 0) {
                const uint64_t t0 = globaltimer_ns();
                while (!poll(x)) {
                  if (mk_aborted(sh)) {
                    got = false;
                    break;
                  }
                  if (globaltimer_ns() - t0 > sh.limit_ns) {
                    mk_fail(sh);
                    got = false;
                    break;
                  }
                  __nanosleep(64);
                }
              }
              ok = __shfl_sync(0xffffffffu, got, 0);
              if (!ok) break;
              kr = dep_end(x);
            }
          }
          if (!ok) break;
          // lane 0: the copies of every stage below kr.  They read what the flags' producers wrote:
          // one proxy fence after the polls.
          const int kend = min(kr, k1);
          if (lane == 0) {
            fence_proxy_async_global();
            int k = kc;
            for (; k < k1 && min(k + XPS, k1) <= kend; k += XPS) {
              const int nk = min(XPS, k1 - k), s = rx.s;
              if (!mk_wait_bar(&emptyx[s], rx.turn ^ 1u, sh)) {
                ok = false;
                break;
              }
              if (first) mk_trace(p, pi * 8 + 2);
              first = false;
              if (last_seg && k + nk == k1) mk_trace(p, pi * 8 + 3);
              mbar_arrive_expect_tx(&fullx[s], nk * XP * x_bytes);
              bulk_load(sX + static_cast<size_t>(s) * sx_bytes, xsrc + static_cast<size_t>(k) * XP * n_pad * 64,
                        nk * XP * x_bytes, &fullx[s]);
              rx.next(SX);
            }
            kc = k;
          }
          ok = __shfl_sync(0xffffffffu, ok, 0);
          kc = __shfl_sync(0xffffffffu, kc, 0);
        }
      }
    } else if (warp >= 4) {
      // ---------------- epilogues ----------------
      MkSeg seg = mk_seg(p, ph, c, G);
      // (a CTA without work in a QKV or gate/up phase still waits for h there: its residual
      // epilogues read h of the phases before)
      if (seg.done() && ph.kind != kMkQkv && ph.kind != kMkGu) continue;
      // per-phase row metadata in shared memory (loaded while the first accumulator is pending)
      const int rslot = mk_row_slot(ph);
      e.M = pl->slot_M[rslot];
      named_bar_sync(1, 128);  // previous phase's readers of the caches are done
      for (int j = e.et; j < e.M; j += 128) {
        const int m = pl->slot_rows[rslot][j];
        s_rows[j] = m;
        if (ph.kind == kMkQkv) {
          const int b = p.step->row_req[m];
          s_pos[j] = p.step->row_pos[m];
          s_kvslot[j] = p.step->req_slot[b];
          s_kvrow[j] = p.step->req_ctx[b] + (m - p.step->req_rowoff[b]);
        }
        if (ph.kind == kMkLm) s_pos[j] = caller_row(p.step, m);
      }
      e.n_extra = 0;
      if (mk_resid(ph)) {
        const int ns = mk_next_slot(p, ph);
        e.nM = pl->slot_M[ns];
        for (int j = e.et; j < e.M; j += 128) {
          const int m = pl->slot_rows[rslot][j], b = p.step->row_req[m], c0 = pl->slot_crow[ns][b];
          s_pos[j] = c0 < 0 ? -1 : c0 + (m - p.step->req_rowoff[b]);
        }
        bool all_run = true;
        for (int x = e.et; x < e.nM; x += 128) {
          const int m = pl->slot_rows[ns][x];
          const bool runs = pl->slot_crow[rslot][p.step->row_req[m]] >= 0;
          s_nrows[x] = runs ? -1 : m;
          all_run = all_run && runs;
        }
        e.n_extra = bar_and(1, 128, all_run) ? 0 : 1;
        e.gnext = ph.kind == kMkO ? p.g_mlp + static_cast<size_t>(ph.layer) * p.d
                  : ns != kFinalSlot ? p.g_attn + static_cast<size_t>(pl->act_layer[ns]) * p.d
                                     : p.g_final;
      }
      named_bar_sync(1, 128);
      e.rows = s_rows;
      e.pos = s_pos;
      e.kvslot = s_kvslot;
      e.kvrow = s_kvrow;
      e.npos = s_pos;
      e.nrows = s_nrows;
      if (ph.kind == kMkQkv) {
        e.kv_base = p.step->kv_layer[ph.layer];
        e.kv_cap = static_cast<size_t>(p.step->kv_cap);
      }
      if (ph.kind == kMkLm) {
        e.logits = p.step->logits;
        e.logits_vec = (p.V & 3) == 0 && (reinterpret_cast<uintptr_t>(e.logits) & 15) == 0;
      }
      if (ph.kind == kMkQkv) {
        // stage the RoPE factors of the first 16 rows; warm L2 with the context keys and values
        // this CTA's attention items will read (they do not depend on this step)
        const int half = D / 2, m16 = e.M < 16 ? e.M : 16;
        for (int x = e.et; x < m16 * half; x += 128) {
          const int j = x / half, i = x - j * half;
          s_rope[j * half + i] = p.rope_cos[static_cast<size_t>(s_pos[j]) * half + i];
          s_rope[16 * 64 + j * half + i] = p.rope_sin[static_cast<size_t>(s_pos[j]) * half + i];
        }
        if (e.et == 0 && !p.attn_external) {
          const int per_req = p.H * p.attn_splits;
          const StepDesc* st = p.step;
          for (int item = c; item < p.B * per_req; item += G) {
            const int b = item / per_req;
            const int head = (item - b * per_req) / p.attn_splits;
            const int split = item - b * per_req - head * p.attn_splits;
            if (pl->slot_crow[ph.slot][b] < 0) continue;
            const int ctx = st->req_ctx[b];
            int k0, k1;
            attn_split_keys(ctx + st->req_nodes[b], p.attn_splits, split, k0, k1);
            k1 = k1 < ctx ? k1 : ctx;
            if (k1 <= k0) continue;
            const size_t cap = static_cast<size_t>(st->kv_cap);
            const __nv_bfloat16* kg =
                st->kv_layer[ph.layer] + ((static_cast<size_t>(st->req_slot[b]) * 2) * p.H + head) * cap * D;
            const uint32_t bytes = static_cast<uint32_t>(k1 - k0) * D * 2;
            bulk_prefetch_l2(kg + static_cast<size_t>(k0) * D, bytes);
            bulk_prefetch_l2(kg + static_cast<size_t>(p.H) * cap * D + static_cast<size_t>(k0) * D, bytes);
          }
        }
        named_bar_sync(1, 128);
      }
      const uint32_t T = seg.T, geff = seg.geff;
      float* partials = (pi & 1) ? p.partials1 : p.partials0;
      int* counters = p.counters + static_cast<size_t>(ph.kind) * p.max_tiles;
      int* done = counters + static_cast<size_t>(7) * p.max_tiles;
      const bool needs_rs = ph.kind == kMkQkv || ph.kind == kMkGu || ph.kind == kMkLm;
      // the norm factors need only h, which is final before this phase's first accumulator
      if (needs_rs && !mk_prepare_rs(p, e, mk_h_dep(p, ph), sh)) {
        ok = false;
        break;
      }
      // Tiles whose k-blocks several CTAs share: with up to 8 rows the last CTA to arrive finishes
      // the tile (two rows a warp, one round of loads).  With more rows that CTA would be busy for
      // many rounds while the others wait -- the 32 tiles of an O phase on 32 of 152 SMs, 34 us after
      // the last MMA for 144 rows -- so every contributor waits for the tile's partial sums and
      // finishes its own share of the rows, once its last split segment is stored (18 us; and
      // QKV 47 -> 25, down 31 -> 14 us).  Waiting costs a round trip more, so up to 8 rows, which
      // one CTA finishes in a single round, stay with the last arriver.  No CTA waits before it
      // has stored every partial sum of the phase that others wait for, and all are resident.
      const bool share = e.M > 8;
      int n_pend = 0;
      int t, k0, k1;
      bool first = true;
      while (ok && seg.next(t, k0, k1)) {
        const int buf = use.s;
        const bool got = e.et == 0 ? mk_wait_bar(&accf[buf], use.turn, sh) : true;
        if (!bar_and(1, 128, got)) {
          ok = false;
          break;
        }
        if (e.et == 0 && first) mk_trace(p, pi * 8 + 6);
        first = false;
        tc_fence_after();
        const uint32_t tb = tmem_base + (static_cast<uint32_t>(e.q * 32) << 16) + static_cast<uint32_t>(buf * n_pad);
        const bool tr_last = e.et == 0 && seg.done();
        if (tr_last) mk_trace(p, kMkTraceSub + pi * 8 + 0);
        const bool whole = k0 == 0 && k1 == ph.kb;
        bool finish = whole;
        if (!whole) {
          const int n_ch = (e.M + 15) >> 4;  // 16-token chunks of the accumulator
          float* part = partials + static_cast<size_t>(c + t) * 128 * n_pad;
          for (int ch = 0; ch < n_ch; ++ch) {
            float v[16];
            mk_acc_tokens(tb, ch, p.xs, v);
#pragma unroll
            for (int jj = 0; jj < 16; ++jj)
              if (ch * 16 + jj < e.M) __stcg(&part[(ch * 16 + jj) * 128 + r], v[jj]);
          }
          tc_fence_before();
          mbar_arrive(&acce[buf]);
          named_bar_sync(1, 128);  // every thread's partial stores precede the release below
          if (tr_last) mk_trace(p, kMkTraceSub + pi * 8 + 1);
          if (e.et == 0) {
            const int f = mk_cta_of(t * ph.kb, T, geff);
            const int l = mk_cta_of((t + 1) * ph.kb - 1, T, geff);
            // (fault injection: the first CTA of the first layer's first down tile does not arrive, so the
            // waits for that tile's parts run out)
            const bool missing = share && p.withhold_flag && ph.kind == kMkDown && ph.slot == 0 && t == 0 && c == f;
            const int last = !missing && atom_add_acq_rel_gpu(&counters[t], 1) == l - f;
            if (last && !share) atomicExch(&counters[t], 0);
            int* pd = s_pend + 4 * n_pend;
            pd[0] = t;
            pd[1] = f;
            pd[2] = l;
            pd[3] = last;
          }
          if (tr_last) mk_trace(p, kMkTraceSub + pi * 8 + 2);
          ++n_pend;  // (at most two: only a CTA's first and last stream-K segments are partial tiles)
        }
        // finished now: this whole tile; the pending split tiles once the CTA has stored its last
        // partial (the last arriver's own tile at once)
        const int n_fin = (whole ? 1 : 0) + (!share || seg.it >= seg.it1 ? n_pend : 0);
        if (n_pend) named_bar_sync(1, 128);  // s_pend is written (and the counter's acquire done)
        for (int k = 0; k < n_fin; ++k) {
          const bool wh = whole && k == 0;
          const int* pd = s_pend + 4 * (k - (whole ? 1 : 0));
          int ft = t, cf = c, cl = c, u0 = e.q, du = 4;
          if (!wh) {
            ft = pd[0];
            cf = pd[1];
            cl = pd[2];
            const bool full = pd[3] != 0;
            if (!share) {
              finish = full;
            } else {
              const bool all = e.et == 0 && !full ? mk_wait_count(&counters[ft], cl - cf + 1, sh) : true;
              ok = bar_and(1, 128, all);
              if (!ok) break;
              finish = true;
              u0 = 4 * (c - cf) + e.q;
              du = 4 * (cl - cf + 1);
            }
          }
          if (!finish) continue;
          if (tr_last) mk_trace(p, kMkTraceSub + pi * 8 + 3);
          if (share)
            mk_finish_rows<D, 4, 5>(p, ph, e, ft, wh, tb, &acce[buf], u0, du, cf, cl, partials, n_pad);
          else
            mk_finish_rows<D, 2, 8>(p, ph, e, ft, wh, tb, &acce[buf], u0, du, cf, cl, partials, n_pad);
          if (tr_last) mk_trace(p, kMkTraceSub + pi * 8 + 4);
          named_bar_sync(1, 128);  // the tile's outputs precede the release below
          if (tr_last) mk_trace(p, kMkTraceSub + pi * 8 + 6);
          if (e.et == 0) {
            bool publish = true;
            if (share && !wh) {
              publish = atom_add_acq_rel_gpu(&done[ft], 1) == cl - cf;
              if (publish) {
                atomicExch(&counters[ft], 0);
                atomicExch(&done[ft], 0);
              }
            }
            unsigned long long* flag = mk_tile_flag(p, ph.kind, ft);
            // (fault injection for the timeout path: the first h tile of the first layer's down
            // phase is never flagged, so its consumers' bounded waits run out)
            const bool withheld = p.withhold_flag && ph.kind == kMkDown && ph.slot == 0 && ft == 0;
            if (publish && flag && !withheld) st_release_u64(flag, mk_seq(p.seq_base, ph.slot, ph.kind));
          }
        }
        if (n_fin > (whole ? 1 : 0)) {
          n_pend = 0;
          if (!share) named_bar_sync(1, 128);  // s_pend is rewritten by the next segment
        }
        if (e.et == 0 && seg.done()) mk_trace(p, pi * 8 + 7);
        use.next(NB);
      }
    }
  }
  if (warp == 0 && lane == 0 && (!ok || *sh.abort_s)) {  // let weight tiles in flight land before the CTA exits
    const uint64_t t0 = globaltimer_ns();
    while (globaltimer_ns() - t0 < 50000) {
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, ncols);
  }
}

size_t mk_trace_slots() { return kMkTraceSlots; }

size_t mk_smem_bytes(int n_pad, int parts, int stages, int kps, int x_stages, int xps, size_t attn_extra) {
  return 1024 + static_cast<size_t>(stages) * kps * kMkWBytes +
         static_cast<size_t>(x_stages) * xps * n_pad * parts * 128 + attn_extra +
         static_cast<size_t>(2 * stages + 2 * x_stages + 2 * kMkMaxAcc + 1) * 8 + 64 + 16 * 128 * 4 +
         64 * 4 * 2 + kMaxRows * 4 + 256 * 4 + 5 * kMaxRows * 4 + 2 * 16 * 64 * 4 + 64;
}

cudaError_t mk_prepare() {
  cudaError_t e = cudaFuncSetAttribute(verify_mk_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(verify_mk_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, 232448);
  return e;
}

cudaError_t launch_verify_mk(const MkParams& p, int grid, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(kMkThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // all CTAs co-resident: the dataflow waits need it
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (p.D == 64) return cudaLaunchKernelEx(&cfg, verify_mk_kernel<64>, p);
  if (p.D == 128) return cudaLaunchKernelEx(&cfg, verify_mk_kernel<128>, p);
  return cudaErrorInvalidValue;
}

int mk_max_blocks_per_sm(int head_dim, size_t smem) {
  int n = 0;
  if (head_dim == 64)
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, verify_mk_kernel<64>, kMkThreads, smem);
  else
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, verify_mk_kernel<128>, kMkThreads, smem);
  return n;
}

}  // namespace tss
