// Compute-bound prompt prefill under the skip mask (Sec. "Domain-Aware Skip Controller": the
// mask is fixed for the whole request, prompt included; App. "Models": the LLaMA block).
//
// The prompt chunks of requests with the same skip set (each starting at a multiple of 128 rows
// of one pass of up to 4096 rows) run through the layers the skip set keeps, all rows at once: per
// layer RMSNorm, the fused QKV projection with RoPE whose K and V rows are appended to the cache,
// causal attention over the cache, the O projection with the residual, RMSNorm, gate/up with
// SwiGLU and the down projection with the residual.  Nothing past the last layer is computed (the
// prompt's logits are not needed).
//
// GEMMs (pf_gemm_kernel): out[t][o] = sum_k X[t][k] W[o][k] with the weights on the MMA's M side
// (128-row tiles, the pre-tiled 128-byte-swizzled images the verification kernels stream) and
// 128 tokens on the N side; a CTA takes two weight tiles against one token tile at a time (two
// accumulators sharing the token operand) through its whole K loop, or through a share of it where
// whole items would leave most of the last wave idle (pf_plan); items are taken weight-pair-major by
// a persistent grid so that the CTAs working at the same time share weight tiles through L2; three groups of epilogue warps keep up with the MMAs.  X is held as two bf16
// parts (hi = bf16(x), lo = bf16(x - hi)), both multiplied by the weights into one fp32
// accumulator in tensor memory, as on the verification path.  Attention (pf_attn_kernel): one CTA
// per (head, 128-query tile of one request), queries on the MMA's M side, 64-key tiles of the
// cache by TMA, S = Q K^T and O += P V in tensor memory, one thread per query row for the online
// softmax; keys past a query's position are masked (causal).
#include "internal.h"

namespace tss {

namespace {

constexpr int kPfThreads = 192;  // attention: warp 0 TMA, warp 1 MMA (+ TMEM), warps 2-5 softmax
constexpr int kPgGroups = 3;     // GEMM epilogue groups of four warps (one per TMEM lane quarter): 14 warps
                                 // leave a thread 128 registers (four groups: 96, with spills)
constexpr int kPgThreads = 64 + 128 * kPgGroups;  // warp 0 copies, warp 1 MMA (+ TMEM), then the epilogue groups
constexpr int kPfStages = 3;
constexpr uint32_t kPfA = 128 * 64 * 2;      // weight block: 16 KiB
constexpr uint32_t kPfB = 128 * 64 * 2;      // 128 tokens x 64 columns of one part: 16 KiB
constexpr uint32_t kPfStage = 2 * kPfA + 2 * kPfB;  // two weight blocks, the token block's two parts
constexpr uint32_t kPfAccCols = 128;         // one accumulator: 128 token columns

__host__ __device__ inline size_t pf_gemm_smem() {
  return 1024 + static_cast<size_t>(kPfStages) * kPfStage + kPgGroups * 16 * 128 * 4;  // + exchange per group
}

// Four consecutive elements as bf16 hi and lo parts: one 8-byte store each.
__device__ __forceinline__ void pf_split_store4(__nv_bfloat16* hi, __nv_bfloat16* lo, size_t i, const float* x) {
  uint32_t h[2], l[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    h[k] = pack_bf16(x[2 * k], x[2 * k + 1]);
    l[k] = pack_bf16(x[2 * k] - __uint_as_float(h[k] << 16), x[2 * k + 1] - __uint_as_float(h[k] & 0xffff0000u));
  }
  *reinterpret_cast<uint2*>(hi + i) = make_uint2(h[0], h[1]);
  *reinterpret_cast<uint2*>(lo + i) = make_uint2(l[0], l[1]);
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// Embedding and RMSNorm
// ---------------------------------------------------------------------------------------------
__global__ void pf_embed_kernel(const PfParams p) {
  const int j = blockIdx.x;
  if (j == 0)  // the GEMMs' arrival counters start every pass at zero, even after one that gave up on a wait
    for (int i = threadIdx.x; i < p.n_counters; i += blockDim.x) p.counters[i] = 0;
  if (j >= p.T) return;
  int tok = p.tokens[j];
  if (tok < 0 || tok >= p.vocab) {
    report(p.status, kStatusCheck);
    tok = 0;
  }
  const __nv_bfloat16* e = p.embed + static_cast<size_t>(tok) * p.d_model;
  for (int c = threadIdx.x; c < p.d_model; c += blockDim.x) p.h[static_cast<size_t>(j) * p.d_model + c] = __bfloat162float(e[c]);
}

// x = h / sqrt(mean(h^2) + eps) * g, as bf16 hi + lo (one block per token row): each thread holds
// kPfNormV groups of 8 consecutive features in registers between the sum of squares and the scaling
// (d_model <= 256 threads x 8 x kPfNormV).
constexpr int kPfNormV = 4;
__global__ void __launch_bounds__(256) pf_norm_kernel(const PfParams p, const float* g) {
  griddep_wait();
  const int j = blockIdx.x;
  if (j >= p.T) return;
  const float* h = p.h + static_cast<size_t>(j) * p.d_model;
  float x[kPfNormV][8];
  float ss = 0.f;
#pragma unroll
  for (int v = 0; v < kPfNormV; ++v) {
    const int c = (v * blockDim.x + threadIdx.x) * 8;
    if (c < p.d_model) {
      const float4 a = *reinterpret_cast<const float4*>(h + c), b = *reinterpret_cast<const float4*>(h + c + 4);
      x[v][0] = a.x; x[v][1] = a.y; x[v][2] = a.z; x[v][3] = a.w;
      x[v][4] = b.x; x[v][5] = b.y; x[v][6] = b.z; x[v][7] = b.w;
#pragma unroll
      for (int i = 0; i < 8; ++i) ss += x[v][i] * x[v][i];
    }
  }
  __shared__ float red[32];
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  const float inv = rsqrtf(red[0] / static_cast<float>(p.d_model) + p.rms_eps);
#pragma unroll
  for (int v = 0; v < kPfNormV; ++v) {
    const int c = (v * blockDim.x + threadIdx.x) * 8;
    if (c < p.d_model) {
      const float4 ga = *reinterpret_cast<const float4*>(g + c), gb = *reinterpret_cast<const float4*>(g + c + 4);
      const float gg[8] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
      uint32_t hw[4], lw[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float y0 = x[v][2 * i] * inv * gg[2 * i], y1 = x[v][2 * i + 1] * inv * gg[2 * i + 1];
        hw[i] = pack_bf16(y0, y1);
        lw[i] = pack_bf16(y0 - __uint_as_float(hw[i] << 16), y1 - __uint_as_float(hw[i] & 0xffff0000u));
      }
      const size_t e = static_cast<size_t>(j) * p.x_ld + c;
      *reinterpret_cast<uint4*>(p.xh + e) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
      *reinterpret_cast<uint4*>(p.xl + e) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Token-tiled GEMM
// ---------------------------------------------------------------------------------------------
namespace {

// OR of v over the epilogue threads (named barrier 2), which it also synchronises.
__device__ __forceinline__ bool pf_epi_or(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.or.pred p, 2, %2, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(r)
      : "r"(v ? 1u : 0u), "n"(128 * kPgGroups)
      : "memory");
  return r != 0;
}

// The fused epilogue of 4 tokens j0 .. j0 + 3 of weight tile t in row form: a warp per 4 tokens, lane
// l holds features f0 = 4 l .. f0 + 3 of each, so that the partners of RoPE (feature ^ 64) and SwiGLU
// (gate f, up f + 64) sit in lane ^ 16 and every access is an 8- or 16-byte vector.  pre() requests what
// the tokens need from global memory; finish() takes the sums.  With a thread per feature and a
// branch, a position load and 2-byte stores per element, a 16-token chunk of QKV took 8-10 us and
// bound the GEMM at short prompts (QKV at 200 tokens 81 us, in this form 58; O at 4096 tokens, with
// the residual's 16 dependent loads and stores, 215 us, 172 with its loads first and its items split).
template <int EPI>
struct PfRows {
  int4 pos, slot;      // QKV: the tokens' positions (-1: gap row) and KV slots
  float4 c[4], s[4];   // QKV, q and k: rotation factors; residual: h in c
  __device__ __forceinline__ void pre(const PfParams& p, int t, int j0, int f0) {
    if constexpr (EPI == kPfEpiResid) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        c[i] = *reinterpret_cast<const float4*>(p.h + static_cast<size_t>(j0 + i) * p.d_model + t * 128 + f0);
    } else if constexpr (EPI == kPfEpiQkv) {
      pos = *reinterpret_cast<const int4*>(p.row_pos + j0);
      slot = *reinterpret_cast<const int4*>(p.row_slot + j0);
      if (t * 128 < 2 * p.d_model) {
        const int ps[4] = {pos.x, pos.y, pos.z, pos.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const size_t e = static_cast<size_t>(ps[i] < 0 ? 0 : ps[i]) * 64 + (f0 & 63);
          c[i] = __ldg(reinterpret_cast<const float4*>(p.rope_cos + e));
          s[i] = __ldg(reinterpret_cast<const float4*>(p.rope_sin + e));
        }
      }
    }
  }
  __device__ __forceinline__ void finish(const PfParams& p, int t, int j0, int f0, const float (*v)[4]) const {
    const int d = p.d_model;
    if constexpr (EPI == kPfEpiResid) {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        *reinterpret_cast<float4*>(p.h + static_cast<size_t>(j0 + i) * d + t * 128 + f0) =
            make_float4(c[i].x + v[i][0], c[i].y + v[i][1], c[i].z + v[i][2], c[i].w + v[i][3]);
    } else if constexpr (EPI == kPfEpiQkv) {
      const int sec = t * 128 < d ? 0 : t * 128 < 2 * d ? 1 : 2;  // q, k or v (one per tile)
      const int f = t * 128 - sec * d + f0, head = f >> 7;
      const int ps[4] = {pos.x, pos.y, pos.z, pos.w}, sl[4] = {slot.x, slot.y, slot.z, slot.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float x[4] = {v[i][0], v[i][1], v[i][2], v[i][3]};
        if (sec < 2) {
          const float cs[4] = {c[i].x, c[i].y, c[i].z, c[i].w}, sn[4] = {s[i].x, s[i].y, s[i].z, s[i].w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float y = __shfl_xor_sync(0xffffffffu, v[i][k], 16);
            x[k] = f0 < 64 ? x[k] * cs[k] - y * sn[k] : x[k] * cs[k] + y * sn[k];
          }
        }
        if (ps[i] < 0) continue;  // gap row
        if (sec == 0) {
          pf_split_store4(p.qh, p.ql, static_cast<size_t>(j0 + i) * d + f, x);
        } else {
          const size_t row = ((static_cast<size_t>(sl[i]) * 2 + (sec - 1)) * p.n_heads + head) * static_cast<size_t>(p.kv_cap) +
                             static_cast<size_t>(ps[i]);
          *reinterpret_cast<uint2*>(p.kv + row * 128 + f0) = make_uint2(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]));
        }
      }
    } else {
      // of two tokens the lower half-warp finishes the first and the upper the second
      const bool upper = f0 >= 64;
#pragma unroll
      for (int i = 0; i < 4; i += 2) {
        float a[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float y = __shfl_xor_sync(0xffffffffu, upper ? v[i][k] : v[i + 1][k], 16);
          const float gt = upper ? y : v[i][k], up = upper ? v[i + 1][k] : y;
          a[k] = silu(gt) * up;
        }
        pf_split_store4(p.uh, p.ul, static_cast<size_t>(j0 + i + (upper ? 1 : 0)) * p.u_ld + t * 64 + (f0 & 63), a);
      }
    }
  }
};

}  // namespace

// Work item = (pair of weight tiles 2w, 2w + 1; token tile u): the two weight tiles share every
// stage's token operand, so a stage of 64 KiB feeds 4 MMAs of 128 x 128 x 16 per k16 step (the
// copy bytes per MMA are half those of one weight tile per item, which L2 bandwidth binds).
//
// Split of the items over the G CTAs (pf_plan): whole items round-robin leave SMs idle in the last
// wave (512 items of an O or down projection at 4096 rows: 3.4 waves in 4) and all but a few SMs
// idle on a short prompt (64 items at 512 rows).  So the first g.n_sk items -- fewer than two
// waves -- are laid end to end and cut into equal ranges of k-blocks, one per CTA, and the rest
// follow as whole items, one per CTA and wave.  A CTA's range starts and ends inside an item, at
// most; such a part goes to the CTA's slot of partial sums, and once the CTA has stored its last
// part, each contributor waits for the item's parts and finishes its own share of the item's 16
// (weight tile, 16-token) units, adding the parts in CTA order.  Every CTA stores before it waits
// and all are resident (cooperative launch), so the waits end.  Bound: the tensor pipe at full
// passes (4096 rows of a 7B layer: QKV 541 -> 497, O 215 -> 172, gate/up 893 -> 841, down 508 -> 487 us
// against whole items); at 200 tokens (O, down: 32 items) the parts' store, wait and reload, about
// 20 us of each launch (a layer 470 -> 254 us).
struct PfCursor {  // (a pass has at most 4096 / 128 x 32768 / 256 items and 2 x SMs x 512 split k-blocks)
  uint32_t it, it1, dp, n_items;  // k-blocks of the split items still to take; next whole item
  uint32_t kb, G;
  __device__ __forceinline__ void start(const PfGemm& g, uint32_t items, uint32_t c, uint32_t grid) {
    kb = g.kb;
    G = grid;
    const uint32_t T = g.n_sk * kb, geff = g.geff;
    it = c < geff ? T * c / geff : 0;
    it1 = c < geff ? T * (c + 1) / geff : 0;
    dp = g.n_sk + c;
    n_items = items;
  }
  __device__ __forceinline__ bool next(uint32_t& item, int& k0, int& k1) {
    if (it < it1) {
      item = it / kb;
      const uint32_t i0 = item * kb;
      k0 = static_cast<int>(it - i0);
      k1 = static_cast<int>(min(kb, it1 - i0));
      it += k1 - k0;
      return true;
    }
    if (dp >= n_items) return false;
    item = dp;
    dp += G;
    k0 = 0;
    k1 = static_cast<int>(kb);
    return true;
  }
};

// Bounded wait for the arrivals of an item's parts.
__device__ bool pf_wait_count(const int* f, int target, volatile int* abort, int* status) {
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t i = 1;; ++i) {
    int v;
    asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(f) : "memory");
    if (v >= target) return true;
    if ((i & 63) == 0) {
      if (*abort) return false;
      if (globaltimer_ns() - t0 > kWaitLimitNs) {
        *abort = 1;
        report(status, kStatusTimeout);
        return false;
      }
    }
  }
}

// Position in the GEMM's ring: slot, and the parity of its current turn, advanced without the 64-bit
// remainder of a running stage number, which the copy and MMA threads had on each stage's path (us,
// 3 layers: 7B, 600 tokens 1316 -> 1288; 13B, 866 tokens 2262 -> 2235; 7B, 200 tokens 741 -> 738).
struct PfRing {
  int s = 0;
  uint32_t turn = 0;
  __device__ __forceinline__ void next() {
    if (++s == kPfStages) {
      s = 0;
      turn ^= 1u;
    }
  }
};

template <int EPI>
__global__ void __launch_bounds__(kPgThreads, 1) pf_gemm_kernel(const __grid_constant__ CUtensorMap tm_xh,
                                                                 const __grid_constant__ CUtensorMap tm_xl,
                                                                 const PfParams p, const PfGemm g) {
  extern __shared__ uint8_t pf_dyn[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(pf_dyn) + 1023) & ~uintptr_t(1023));
  float* xch0 = reinterpret_cast<float*>(base + kPfStages * kPfStage);  // [group][16][128]
  __shared__ uint64_t full[kPfStages], empty[kPfStages], acc_full[2], acc_empty[2], drain;
  __shared__ uint32_t tslot;
  __shared__ int abort_s;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t n_u = (p.T + 127) >> 7;    // token tiles
  const uint32_t n_w = (g.n_o + 1) >> 1;    // weight-tile pairs (the last may hold one tile)
  const uint32_t n_items = n_w * n_u;
  if (tid == 0) {
    for (int i = 0; i < kPfStages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], 4 * kPgGroups);
    }
    mbar_init(&drain, 1);
    abort_s = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&tslot, 4 * kPfAccCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = tslot;
  volatile int* abort = &abort_s;
  const __nv_bfloat16* wl = g.w + static_cast<size_t>(g.layer) * g.w_layer_elems;

  if (warp == 0) {
    // ---------------- producer: both weight blocks and both token parts of each k-block ----------------
    if (lane == 0) {
      prefetch_tmap(&tm_xh);
      prefetch_tmap(&tm_xl);
      PfRing ring;
      uint32_t item;
      bool ok = true;
      int k0, k1;
      PfCursor cur;
      cur.start(g, n_items, blockIdx.x, gridDim.x);
      while (ok && cur.next(item, k0, k1)) {
        const int w = static_cast<int>(item / n_u), u = static_cast<int>(item) - w * n_u;
        const int t0 = 2 * w;
        const bool two = t0 + 1 < g.n_o;
        for (int k = k0; k < k1; ++k, ring.next()) {
          const int s = ring.s;
          if (!mbar_wait(&empty[s], ring.turn ^ 1u, abort, p.status)) {  // (the first turn: free at once)
            ok = false;
            break;
          }
          uint8_t* st = base + s * kPfStage;
          mbar_arrive_expect_tx(&full[s], (two ? 2 : 1) * kPfA + 2 * kPfB);
          bulk_load(st, wl + (static_cast<size_t>(t0) * g.kb + k) * kTileElems, kPfA, &full[s]);
          if (two) bulk_load(st + kPfA, wl + (static_cast<size_t>(t0 + 1) * g.kb + k) * kTileElems, kPfA, &full[s]);
          tma_load_2d(st + 2 * kPfA, &tm_xh, &full[s], k * 64, u * 128);
          tma_load_2d(st + 2 * kPfA + kPfB, &tm_xl, &full[s], k * 64, u * 128);
        }
      }
      // every copy issued has landed before the kernel returns: the last turn of each slot
      for (int i = 0; i < kPfStages; ++i, ring.next()) {
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(&full[ring.s], ring.turn ^ 1u))  // (a slot never used: passes at once)
          if (globaltimer_ns() - t0 > kWaitLimitNs) break;
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: per k16 step, (A0, A1) x (hi, lo) into two accumulators ----------------
    if (lane == 0) {
      const uint32_t idesc = idesc_bf16_m128(128);
      PfRing ring;
      uint32_t item;
      int n = 0, k0, k1;
      // fault injection: CTA 0 issues no MMA, so its epilogue's first wait runs out
      bool ok = !(g.withhold && blockIdx.x == 0);
      PfCursor cur;
      cur.start(g, n_items, blockIdx.x, gridDim.x);
      for (; ok && cur.next(item, k0, k1); ++n) {
        const int w = static_cast<int>(item / n_u);
        const bool two = 2 * w + 1 < g.n_o;
        const int buf = n & 1;
        if (n >= 2 && !mbar_wait(&acc_empty[buf], static_cast<uint32_t>((n >> 1) - 1) & 1u, abort, p.status)) break;
        tc_fence_after();
        const uint32_t d0 = tm + buf * 2 * kPfAccCols, d1 = d0 + kPfAccCols;
        for (int k = k0; k < k1; ++k, ring.next()) {
          const int s = ring.s;
          if (!mbar_wait(&full[s], ring.turn, abort, p.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t a = smem_u32(base + s * kPfStage), b = a + 2 * kPfA;
#pragma unroll
          for (int k16 = 0; k16 < 4; ++k16) {
            const uint64_t bh = sdesc_sw128(b + k16 * 32), bl = sdesc_sw128(b + kPfB + k16 * 32);
            const uint64_t a0 = sdesc_sw128(a + k16 * 32);
            umma_bf16(d0, a0, bh, idesc, (k > k0 || k16) ? 1u : 0u);
            umma_bf16(d0, a0, bl, idesc, 1u);
            if (two) {
              const uint64_t a1 = sdesc_sw128(a + kPfA + k16 * 32);
              umma_bf16(d1, a1, bh, idesc, (k > k0 || k16) ? 1u : 0u);
              umma_bf16(d1, a1, bl, idesc, 1u);
            }
          }
          umma_commit(&empty[s]);
        }
        if (ok) umma_commit(&acc_full[buf]);
      }
      // every MMA issued has completed before the kernel returns
      umma_commit(&drain);
      const uint64_t t0 = globaltimer_ns();
      while (!mbar_try_wait(&drain, 0))
        if (globaltimer_ns() - t0 > kWaitLimitNs) break;
    }
  } else {
    // ---------------- epilogue warps: TMEM lane quarter = warp & 3, thread r = weight row; group
    // (warp - 2) / 4 takes every kPgGroups-th of the item's 16-token chunks ----------------
    const int q = warp & 3, r = q * 32 + lane, grp = (warp - 2) >> 2, f0 = 4 * lane;
    float* xch = xch0 + grp * 16 * 128;
    const int bar = grp == 0 ? 1 : 2 + grp;  // (2 is the vote barrier)
    const uint32_t T = g.n_sk * g.kb, geff = g.geff;
    auto cta_of = [&](uint32_t i) { return static_cast<int>(((i + 1) * geff - 1) / T); };
    // slot of CTA cc's part of split item x: its first part, or its last when its range begins earlier
    auto slot_of = [&](uint32_t cc, uint32_t x) { return 2 * cc + (T * cc / geff < x * g.kb ? 1 : 0); };
    constexpr size_t kSlot = static_cast<size_t>(2) * 128 * 128;  // floats: [tile of the pair][token][weight row]
    int n = 0, n_pend = 0, k0, k1;
    uint32_t item, pend[2] = {0, 0};
    PfCursor cur;
    cur.start(g, n_items, blockIdx.x, gridDim.x);
    for (; cur.next(item, k0, k1); ++n) {
      const int w = static_cast<int>(item / n_u), u = static_cast<int>(item) - w * n_u;
      const int buf = n & 1;
      const bool whole = k0 == 0 && k1 == g.kb;
      const bool ok = mbar_wait(&acc_full[buf], static_cast<uint32_t>(n >> 1) & 1u, abort, p.status);
      if (pf_epi_or(!ok)) break;
      tc_fence_after();
      float* part = p.partials + (whole ? 0 : slot_of(blockIdx.x, item)) * kSlot;
      const int units = 2 * w + 1 < g.n_o ? 16 : 8;  // 16-token chunks of both accumulators
      for (int y = grp; y < units; y += kPgGroups) {
        const int a = y >> 3, ch = y & 7, t = 2 * w + a;
        const int j0 = u * 128 + ch * 16 + 4 * q;  // this warp's tokens of the chunk
        PfRows<EPI> rows;
        if (whole) rows.pre(p, t, j0, f0);
        float v[16];
        tmem_ld16(tm + (static_cast<uint32_t>(q * 32) << 16) + (buf * 2 + a) * kPfAccCols + ch * 16, v);
        if (whole) {
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) xch[jj * 128 + r] = v[jj];
          named_bar_sync(bar, 128);
          float x[4][4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 z = *reinterpret_cast<const float4*>(xch + (4 * q + i) * 128 + f0);
            x[i][0] = z.x; x[i][1] = z.y; x[i][2] = z.z; x[i][3] = z.w;
          }
          named_bar_sync(bar, 128);
          rows.finish(p, t, j0, f0, x);
        } else {
#pragma unroll
          for (int jj = 0; jj < 16; ++jj) __stcg(&part[(a * 128 + ch * 16 + jj) * 128 + r], v[jj]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[buf]);
      if (!whole) {
        pf_epi_or(false);  // every thread's part precedes the release below
        if (tid == 64) atom_add_acq_rel_gpu(&p.counters[item], 1);
        pend[n_pend++] = item;  // (at most two: a range's first and last items)
      }
      if (n_pend == 0 || cur.it < cur.it1) continue;
      bool failed = false;
      for (int x = 0; x < n_pend && !failed; ++x) {
        const uint32_t pi = pend[x];
        const int pw = static_cast<int>(pi / n_u), pu = static_cast<int>(pi) - pw * n_u;
        const int cf = cta_of(pi * g.kb), cl = cta_of((pi + 1) * g.kb - 1), nc = cl - cf + 1;
        const bool all = tid != 64 || pf_wait_count(&p.counters[pi], nc, abort, p.status);
        failed = pf_epi_or(!all);
        if (failed) break;
        if (tid == 64 && atomicAdd(&p.counters[g.n_sk + pi], 1) == nc - 1) {  // every contributor has seen the count
          p.counters[pi] = 0;
          p.counters[g.n_sk + pi] = 0;
        }
        const int n_units = 2 * pw + 1 < g.n_o ? 16 : 8;
        for (int y = static_cast<int>(blockIdx.x) - cf + nc * grp; y < n_units; y += nc * kPgGroups) {
          const int a = y >> 3, ch = y & 7;
          const int t = 2 * pw + a, j0 = pu * 128 + ch * 16 + 4 * q;
          PfRows<EPI> rows;
          // two contributors' parts per round of loads, the first round before the epilogue's own loads
          float x[4][4];
#pragma unroll
          for (int i = 0; i < 4; ++i) x[i][0] = x[i][1] = x[i][2] = x[i][3] = 0.f;
          for (int cc = cf; cc <= cl; cc += 2) {
            float4 part2[2][4];
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              const float* pp = p.partials + slot_of(min(cc + k, cl), pi) * kSlot + (a * 128 + ch * 16 + 4 * q) * 128 + f0;
#pragma unroll
              for (int i = 0; i < 4; ++i)
                part2[k][i] = cc + k <= cl ? __ldcg(reinterpret_cast<const float4*>(pp + i * 128)) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            if (cc == cf) rows.pre(p, t, j0, f0);
#pragma unroll
            for (int k = 0; k < 2; ++k)
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                x[i][0] += part2[k][i].x;
                x[i][1] += part2[k][i].y;
                x[i][2] += part2[k][i].z;
                x[i][3] += part2[k][i].w;
              }
          }
          rows.finish(p, t, j0, f0, x);
        }
      }
      n_pend = 0;
      if (failed) break;
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, 4 * kPfAccCols);
  }
}

// ---------------------------------------------------------------------------------------------
// Causal attention of the chunk's queries (head_dim 128)
// ---------------------------------------------------------------------------------------------
namespace {

constexpr int kPaKeys = 64;                          // keys per tile
constexpr int kPaSlots = 3;                          // slots of the K and of the V ring
constexpr uint32_t kPaQPart = 2 * 128 * 128;         // 128 queries x 128 dims bf16: 32 KiB
constexpr uint32_t kPaKV = 2 * kPaKeys * 128;        // 64 keys x 128 dims: 16 KiB (two 8 KiB boxes)
constexpr uint32_t kPaPPart = 128 * kPaKeys * 2;     // 128 queries x 64 keys: 16 KiB
constexpr uint32_t kPaTmem = 256;                    // S x 2 (64 cols each), O (128 cols)

__host__ __device__ inline size_t pf_attn_smem() {
  return 1024 + 2 * kPaQPart + 2 * kPaSlots * kPaKV + 2 * 2 * kPaPPart;
}

// A split item's end, by the softmax threads: this CTA's part of O (raw sums, tensor memory at tm) and
// its rows' (max, sum) go to p.partials; the last CTA of the item to arrive adds the parts in split
// order and writes the outputs.  wgt: [split][128] floats of shared memory.
__device__ __noinline__ void pa_merge(const PfParams& p, float* wgt, int* s_last, uint32_t tm, int st, int qr, int q0,
                                      int nrow, int used, float m, float l) {
  constexpr int D = 128;
  const int h = blockIdx.x, item = blockIdx.y * p.n_heads + h;
  const bool valid = qr < nrow;
  float* po = p.partials + static_cast<size_t>(item) * p.n_splits * 128 * D;
  float2* ml = reinterpret_cast<float2*>(p.partials + static_cast<size_t>(p.n_heads) * p.n_qtiles * p.n_splits * 128 * D) +
               static_cast<size_t>(item) * p.n_splits * 128 + qr;
  tc_fence_after();
  if (valid) __stcg(ml + blockIdx.z * 128, make_float2(m, l));
#pragma unroll 2
  for (int c = 0; c < D / 16; ++c) {
    float o[16];
    tmem_ld16(tm + 128 + c * 16, o);
    if (valid) {
      float4* d = reinterpret_cast<float4*>(po + (static_cast<size_t>(blockIdx.z) * 128 + qr) * D + c * 16);
#pragma unroll
      for (int i = 0; i < 4; ++i) __stcg(d + i, make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]));
    }
  }
  tc_fence_before();
  named_bar_sync(1, 128);  // every thread's part precedes the release below
  if (st == 0) {
    *s_last = atom_add_acq_rel_gpu(&p.attn_counters[item], 1) == used - 1;
    if (*s_last) atomicExch(&p.attn_counters[item], 0);
  }
  named_bar_sync(1, 128);
  if (!*s_last) return;  // (else: the counter's acquire, then the barrier: the other parts are visible)
  if (valid) {
    float M = -INFINITY, L = 0.f;
    for (int x = 0; x < used; ++x) M = fmaxf(M, __ldcg(ml + x * 128).x);
    const float mb = M == -INFINITY ? 0.f : M;
    for (int x = 0; x < used; ++x) {
      const float2 v = __ldcg(ml + x * 128);
      const float f = exp2f(v.x - mb);
      L += f * v.y;
      wgt[x * 128 + qr] = f;
    }
    if (!(L > 0.f)) report(p.status, kStatusCheck);
    const float inv = L > 0.f ? 1.f / L : 0.f;
    for (int x = 0; x < used; ++x) wgt[x * 128 + qr] *= inv;
  }
  named_bar_sync(1, 128);
  // units (4 columns of a row): the loads of kU units and two splits in flight together
  constexpr int kU = 4;
  const int n_u = nrow * (D / 4);
  for (int u0 = st; u0 < n_u; u0 += kU * 128) {
    float4 a[kU];
#pragma unroll
    for (int k = 0; k < kU; ++k) a[k] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
    for (int x = 0; x < used; ++x) {
      float4 v[kU];
#pragma unroll
      for (int k = 0; k < kU; ++k)
        v[k] = u0 + k * 128 < n_u ? __ldcg(reinterpret_cast<const float4*>(po + static_cast<size_t>(x) * 128 * D) + u0 + k * 128)
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int k = 0; k < kU; ++k) {
        const float f = wgt[x * 128 + min((u0 + k * 128) / (D / 4), 127)];
        a[k].x += f * v[k].x;
        a[k].y += f * v[k].y;
        a[k].z += f * v[k].z;
        a[k].w += f * v[k].w;
      }
    }
#pragma unroll
    for (int k = 0; k < kU; ++k) {
      const int u = u0 + k * 128;
      if (u < n_u) {
        const float o[4] = {a[k].x, a[k].y, a[k].z, a[k].w};
        pf_split_store4(p.ah, p.al, static_cast<size_t>(q0 + u / (D / 4)) * p.d_model + h * D + (u % (D / 4)) * 4, o);
      }
    }
  }
}

}  // namespace

// Grid (heads, query tiles of p.qtiles, which the host orders heaviest first, so that the CTAs
// with the most keys start first, key splits: pf_attn_splits); the KV map has 64-row boxes; tm_q: q hi / lo maps over
// [T_max][d].
__global__ void __launch_bounds__(kPfThreads, 1) pf_attn_kernel(const __grid_constant__ CUtensorMap tm_qh,
                                                                const __grid_constant__ CUtensorMap tm_ql,
                                                                const __grid_constant__ CUtensorMap tm_kv,
                                                                const PfParams p) {
  extern __shared__ uint8_t pa_dyn[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(pa_dyn) + 1023) & ~uintptr_t(1023));
  uint8_t* sq = base;                                // Q hi (2 boxes), Q lo (2 boxes)
  uint8_t* sk = sq + 2 * kPaQPart;                   // [slot] K
  uint8_t* sv = sk + kPaSlots * kPaKV;               // [slot] V
  uint8_t* sp = sv + kPaSlots * kPaKV;               // [2] P hi, P lo
  __shared__ uint64_t qfull, kfull[kPaSlots], kempty[kPaSlots], vfull[kPaSlots], vempty[kPaSlots];
  __shared__ uint64_t s_full[2], s_free[2], p_full[2], p_free[2], o_full, drain;
  __shared__ uint32_t tslot;
  __shared__ int abort_s, s_last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  griddep_wait();
  const int h = blockIdx.x;
  const int4 qi = p.qtiles[blockIdx.y];  // (first row, slot, position of the first row, rows)
  const int H = p.n_heads, D = 128;
  const int q0 = qi.x, slot = qi.y, pos_t0 = qi.z, nrow = qi.w;
  const int key_end = pos_t0 + nrow;  // keys any query of the tile may see
  const int n_tiles = (key_end + kPaKeys - 1) / kPaKeys, per = (n_tiles + p.n_splits - 1) / p.n_splits;
  const int used = (n_tiles + per - 1) / per;  // splits that hold tiles
  const int k0 = static_cast<int>(blockIdx.z) * per * kPaKeys;  // this CTA's first key, and its key tiles
  const int n = min(n_tiles - static_cast<int>(blockIdx.z) * per, per);
  if (n <= 0) return;  // (the whole CTA)
  if (tid == 0) {
    mbar_init(&qfull, 1);
    for (int i = 0; i < kPaSlots; ++i) {
      mbar_init(&kfull[i], 1);
      mbar_init(&kempty[i], 1);
      mbar_init(&vfull[i], 1);
      mbar_init(&vempty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&s_full[i], 1);
      mbar_init(&s_free[i], 4);
      mbar_init(&p_full[i], 1);
      mbar_init(&p_free[i], 1);
    }
    mbar_init(&o_full, 1);
    mbar_init(&drain, 1);
    abort_s = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&tslot, kPaTmem);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = tslot;
  volatile int* abort = &abort_s;
  const size_t cap = static_cast<size_t>(p.kv_cap);
  const int rowK = static_cast<int>(((static_cast<size_t>(slot) * 2) * H + h) * cap) + k0;
  const int rowV = rowK + static_cast<int>(static_cast<size_t>(H) * cap);

  if (warp == 0) {
    // ---------------- TMA producer: Q once, then K and V of every key tile ----------------
    if (lane == 0) {
      prefetch_tmap(&tm_kv);
      mbar_arrive_expect_tx(&qfull, 2 * kPaQPart);
      tma_load_2d(sq, &tm_qh, &qfull, h * D, q0);
      tma_load_2d(sq + kPaQPart / 2, &tm_qh, &qfull, h * D + 64, q0);
      tma_load_2d(sq + kPaQPart, &tm_ql, &qfull, h * D, q0);
      tma_load_2d(sq + kPaQPart + kPaQPart / 2, &tm_ql, &qfull, h * D + 64, q0);
      int nk = 0, nv = 0;
      for (int t = 0; t < n; ++t) {
        const int s = t % kPaSlots;
        if (t >= kPaSlots && !mbar_wait(&kempty[s], ((t / kPaSlots) - 1) & 1, abort, p.status)) break;
        mbar_arrive_expect_tx(&kfull[s], kPaKV);
        tma_load_2d(sk + s * kPaKV, &tm_kv, &kfull[s], 0, rowK + t * kPaKeys);
        tma_load_2d(sk + s * kPaKV + kPaKV / 2, &tm_kv, &kfull[s], 64, rowK + t * kPaKeys);
        ++nk;
        if (t >= kPaSlots && !mbar_wait(&vempty[s], ((t / kPaSlots) - 1) & 1, abort, p.status)) break;
        mbar_arrive_expect_tx(&vfull[s], kPaKV);
        tma_load_2d(sv + s * kPaKV, &tm_kv, &vfull[s], 0, rowV + t * kPaKeys);
        tma_load_2d(sv + s * kPaKV + kPaKV / 2, &tm_kv, &vfull[s], 64, rowV + t * kPaKeys);
        ++nv;
      }
      auto drain_bar = [](uint64_t* bar, uint32_t parity) {
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(bar, parity))
          if (globaltimer_ns() - t0 > kWaitLimitNs) return;
      };
      drain_bar(&qfull, 0);
      for (int u = nk - 1; u >= 0 && u >= nk - kPaSlots; --u) drain_bar(&kfull[u % kPaSlots], (u / kPaSlots) & 1);
      for (int u = nv - 1; u >= 0 && u >= nv - kPaSlots; --u) drain_bar(&vfull[u % kPaSlots], (u / kPaSlots) & 1);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: S(t) = Q K^T, then O += P(t - 1) V ----------------
    if (lane == 0) {
      const uint32_t idS = idesc_bf16_m128(kPaKeys), idPV = idesc_bf16_m128(D) | (1u << 16);  // (B MN-major)
      const uint32_t q_a = smem_u32(sq), k_a = smem_u32(sk), v_a = smem_u32(sv), p_a = smem_u32(sp);
      bool ok = mbar_wait(&qfull, 0, abort, p.status);
      for (int t = 0; ok && t <= n; ++t) {
        if (t < n) {
          const int s = t % kPaSlots;
          if (!mbar_wait(&kfull[s], (t / kPaSlots) & 1, abort, p.status)) break;
          if (t >= 2 && !mbar_wait(&s_free[t & 1], ((t >> 1) - 1) & 1, abort, p.status)) break;
          tc_fence_after();
          const uint32_t dS = tm + (t & 1) * kPaKeys;
#pragma unroll
          for (int part = 0; part < 2; ++part)
#pragma unroll
            for (int kb = 0; kb < 2; ++kb)
#pragma unroll
              for (int k16 = 0; k16 < 4; ++k16)
                umma_bf16(dS, sdesc_sw128(q_a + part * kPaQPart + kb * (kPaQPart / 2) + k16 * 32),
                          sdesc_sw128(k_a + s * kPaKV + kb * (kPaKV / 2) + k16 * 32), idS, (part | kb | k16) ? 1u : 0u);
          umma_commit(&s_full[t & 1]);
          umma_commit(&kempty[s]);
        }
        if (t >= 1) {
          const int u = t - 1, s = u % kPaSlots;
          if (!mbar_wait(&vfull[s], (u / kPaSlots) & 1, abort, p.status)) break;
          if (!mbar_wait(&p_full[u & 1], (u >> 1) & 1, abort, p.status)) break;
          tc_fence_after();
          const uint32_t pb = p_a + (u & 1) * 2 * kPaPPart;
#pragma unroll
          for (int part = 0; part < 2; ++part)
#pragma unroll
            for (int kk = 0; kk < kPaKeys / 16; ++kk)
              umma_bf16(tm + 128, sdesc_sw128(pb + part * kPaPPart + kk * 32),
                        sdesc_sw128_mn(v_a + s * kPaKV + kk * 16 * 128, kPaKV / 2), idPV, (u | part | kk) ? 1u : 0u);
          umma_commit(&vempty[s]);
          umma_commit(&p_free[u & 1]);
          if (u == n - 1) umma_commit(&o_full);
        }
      }
      umma_commit(&drain);
      const uint64_t t0 = globaltimer_ns();
      while (!mbar_try_wait(&drain, 0))
        if (globaltimer_ns() - t0 > kWaitLimitNs) break;
    }
  } else {
    // ---------------- softmax: thread = query row (TMEM lane) ----------------
    const int qg = warp & 3, qr = qg * 32 + lane, st = tid - 64;
    const uint32_t lanes = static_cast<uint32_t>(qg * 32) << 16;
    const int j = q0 + qr;                  // row of this query
    const bool valid = qr < nrow;
    const int pq = pos_t0 + qr - k0;        // its position, from this CTA's first key: keys <= pq are visible
    const float scale = 1.4426950408889634f / sqrtf(static_cast<float>(D));
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int t = 0; t < n; ++t) {
      ok = mbar_wait(&s_full[t & 1], (t >> 1) & 1, abort, p.status);
      if (bar_or<1>(!ok)) break;
      tc_fence_after();
      float s[kPaKeys];
#pragma unroll
      for (int c = 0; c < kPaKeys / 16; ++c) tmem_ld16(tm + lanes + (t & 1) * kPaKeys + c * 16, s + c * 16);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&s_free[t & 1]);
      float mt = -INFINITY;
#pragma unroll
      for (int c = 0; c < kPaKeys; ++c) {
        const int key = t * kPaKeys + c;
        s[c] = (valid && key <= pq) ? s[c] * scale : -INFINITY;
        mt = fmaxf(mt, s[c]);
      }
      // the row's running max is raised only when the tile exceeds it by more than 2^8; the
      // warp rescales its rows of O together (tensor-memory access is warp-wide)
      const bool raise = mt > m + 8.f;
      float alpha = 1.f;
      if (raise) {
        alpha = m == -INFINITY ? 1.f : exp2f(m - mt);
        m = mt;
        l *= alpha;
      }
      ok = t < 2 || mbar_wait(&p_free[t & 1], ((t >> 1) - 1) & 1, abort, p.status);
      if (t >= 1 && __any_sync(0xffffffffu, raise && alpha != 1.f) && ok)
        ok = mbar_wait(&p_free[(t - 1) & 1], ((t - 1) >> 1) & 1, abort, p.status);
      // in the last tile, the V rows past the keys (stale or unwritten cache rows) are zeroed
      if (ok && t == n - 1) {
        const int s_ = t % kPaSlots, r0 = key_end - k0 - t * kPaKeys;
        ok = mbar_wait(&vfull[s_], (t / kPaSlots) & 1, abort, p.status);
        if (ok && st >= r0 && st < kPaKeys) {
          uint4* v0 = reinterpret_cast<uint4*>(sv + s_ * kPaKV + st * 128);
          uint4* v1 = reinterpret_cast<uint4*>(sv + s_ * kPaKV + kPaKV / 2 + st * 128);
#pragma unroll
          for (int i = 0; i < 8; ++i) v0[i] = v1[i] = make_uint4(0, 0, 0, 0);
        }
      }
      if (bar_or<1>(!ok)) break;
      if (t >= 1 && __any_sync(0xffffffffu, raise && alpha != 1.f)) {
        tc_fence_after();
        float o[16];
#pragma unroll
        for (int c = 0; c < D / 16; ++c) {
          tmem_ld16(tm + lanes + 128 + c * 16, o);
#pragma unroll
          for (int i = 0; i < 16; ++i) o[i] *= alpha;
          tmem_st16(tm + lanes + 128 + c * 16, o);
        }
        tc_fence_before();
      }
      // weights 2^(s - m) as bf16 hi + lo into the P operand (row qr, 64 keys = one 128-byte row)
      const float mb = m == -INFINITY ? 0.f : m;
      uint8_t* ph = sp + (t & 1) * 2 * kPaPPart + qr * 128;
      uint8_t* pl = ph + kPaPPart;
#pragma unroll
      for (int c8 = 0; c8 < kPaKeys / 8; ++c8) {
        uint32_t hw[4], lw[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float w0 = exp2f(s[c8 * 8 + 2 * i] - mb), w1 = exp2f(s[c8 * 8 + 2 * i + 1] - mb);
          l += w0 + w1;
          hw[i] = pack_bf16(w0, w1);
          const float h0 = __uint_as_float(hw[i] << 16), h1 = __uint_as_float(hw[i] & 0xffff0000u);
          lw[i] = pack_bf16(w0 - h0, w1 - h1);
        }
        const int sw = (c8 ^ (qr & 7)) << 4;
        *reinterpret_cast<uint4*>(ph + sw) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
        *reinterpret_cast<uint4*>(pl + sw) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
      }
      fence_async_smem();
      named_bar_sync(1, 128);
      if (st == 0) mbar_arrive(&p_full[t & 1]);
    }
    if (ok) {
      ok = mbar_wait(&o_full, 0, abort, p.status);
      const bool fail = bar_or<1>(!ok);
      if (!fail && used > 1) {
        pa_merge(p, reinterpret_cast<float*>(sp), &s_last, tm + lanes, st, qr, q0, nrow, used, m, l);
      } else if (!fail) {
        tc_fence_after();
        const float inv = l > 0.f ? 1.f / l : 0.f;
        if (valid && !(l > 0.f)) report(p.status, kStatusCheck);
#pragma unroll
        for (int c = 0; c < D / 16; ++c) {
          float o[16];
          tmem_ld16(tm + lanes + 128 + c * 16, o);
          if (valid) {
            // this row's 16 outputs as bf16 hi and lo parts: two 16-byte stores per part
            uint32_t hw[8], lw[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float x0 = o[2 * i] * inv, x1 = o[2 * i + 1] * inv;
              hw[i] = pack_bf16(x0, x1);
              lw[i] = pack_bf16(x0 - __uint_as_float(hw[i] << 16), x1 - __uint_as_float(hw[i] & 0xffff0000u));
            }
            const size_t e = static_cast<size_t>(j) * p.d_model + h * D + c * 16;
            uint4* ph = reinterpret_cast<uint4*>(p.ah + e);
            uint4* pl = reinterpret_cast<uint4*>(p.al + e);
            ph[0] = make_uint4(hw[0], hw[1], hw[2], hw[3]);
            ph[1] = make_uint4(hw[4], hw[5], hw[6], hw[7]);
            pl[0] = make_uint4(lw[0], lw[1], lw[2], lw[3]);
            pl[1] = make_uint4(lw[4], lw[5], lw[6], lw[7]);
          }
        }
        tc_fence_before();
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, kPaTmem);
  }
}

// ---------------------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------------------
cudaError_t pf_prepare() {
  cudaError_t e = cudaFuncSetAttribute(pf_gemm_kernel<kPfEpiQkv>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(pf_gemm_smem()));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(pf_gemm_kernel<kPfEpiResid>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(pf_gemm_smem()));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(pf_gemm_kernel<kPfEpiSwiglu>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             static_cast<int>(pf_gemm_smem()));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(pf_attn_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(pf_attn_smem()));
  return e;
}

cudaError_t launch_pf_embed(const PfParams& p, cudaStream_t s) {
  return launch_k(pf_embed_kernel, dim3(p.T), dim3(256), 0, s, false, p);
}

// (the norm and the attention start while the GEMM before them drains: a launch's set-up, about 2 us)
cudaError_t launch_pf_norm(const PfParams& p, const float* g, cudaStream_t s) {
  return launch_k(pf_norm_kernel, dim3(p.T), dim3(256), 0, s, true, p, g);
}

// The items that are split (see pf_gemm_kernel) and the CTAs sharing them.  Whole items only, where
// the CTA with the most of them has at most kPfWhole k-blocks (about 0.55 us each) more than an
// even share: about what storing, counting and adding the parts costs (three layers, us, with
// 12 / 20 / 28 / 40 k-blocks: 7B 200 tokens 762 / 762 / 803 / 803, 384 tokens 970 / 925 / 925 / 925,
// 13B 866 tokens 2556 / 2307 / 2306 / 2316).
int pf_plan(PfGemm* g, int T, int sms) {
  constexpr long long kPfWhole = 20;
  const long long items = static_cast<long long>((g->n_o + 1) / 2) * ((T + 127) / 128);
  const long long even = (items * g->kb + sms - 1) / sms, whole = (items + sms - 1) / sms * g->kb;
  g->n_sk = 0;
  g->geff = 1;
  if (whole <= even + kPfWhole) return static_cast<int>(items < sms ? items : sms);
  const long long waves = items / sms;
  g->n_sk = static_cast<int>(items - (waves >= 2 ? (waves - 1) * sms : 0));
  const long long blocks = static_cast<long long>(g->n_sk) * g->kb;
  g->geff = static_cast<int>(blocks < sms ? blocks : sms);
  return g->geff;  // (whole items follow only where every CTA has a range)
}

size_t pf_partial_floats(int sms) { return static_cast<size_t>(2) * sms * 2 * 128 * 128; }
int pf_counters(int sms) { return 5 * sms; }  // (split GEMM items: up to 4 sms, split attention items: up to sms)

// Key splits of an attention item: where the items leave SMs idle, the fewest key tiles in a row plus
// what a merge costs, in halves of a key tile (about 0.8 us each).  Three layers, us, with 1 / 2 / 3 / 4
// splits (4: or as many as fit): 7B, 100 tokens after 1400: 646 / 610 / 602 / 594; 64 after 600: 576 / 569 /
// 567 / 563; 250 after 900: 798 / 780 (two fit); 200 after 333: 738 / 748 (not split); 107 alone: 533 / 557
// (not split); 13B, 100 after 800: 726 / 713 / 708 (three fit).  (At most `sms` CTAs then, whose parts
// p.partials holds four times over.)
int pf_attn_splits(int items, int max_keys, int sms) {
  const int n = (max_keys + kPaKeys - 1) / kPaKeys;
  int best = 1, cost = 2 * n;
  for (int x = 2; x <= 8 && x * items <= sms; ++x) {
    const int y = 2 * ((n + x - 1) / x) + 6 + x;
    if (y < cost) {
      cost = y;
      best = x;
    }
  }
  return best;
}

template <int EPI>
cudaError_t launch_pf_gemm_epi(const CUtensorMap& xh, const CUtensorMap& xl, const PfParams& p, PfGemm g, int sms,
                               cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(pf_plan(&g, p.T, sms));
  cfg.blockDim = dim3(kPgThreads);
  cfg.dynamicSmemBytes = pf_gemm_smem();
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;  // all CTAs resident: contributors wait for one another
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = g.n_sk > 0 ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, pf_gemm_kernel<EPI>, xh, xl, p, g);
}

cudaError_t launch_pf_gemm(int epi, const CUtensorMap& xh, const CUtensorMap& xl, const PfParams& p, const PfGemm& g,
                           int sms, cudaStream_t s) {
  switch (epi) {
    case kPfEpiQkv: return launch_pf_gemm_epi<kPfEpiQkv>(xh, xl, p, g, sms, s);
    case kPfEpiResid: return launch_pf_gemm_epi<kPfEpiResid>(xh, xl, p, g, sms, s);
    case kPfEpiSwiglu: return launch_pf_gemm_epi<kPfEpiSwiglu>(xh, xl, p, g, sms, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_pf_attn(const CUtensorMap& qh, const CUtensorMap& ql, const CUtensorMap& kv, const PfParams& p,
                           cudaStream_t s) {
  const dim3 gr(p.n_heads, p.n_qtiles, p.n_splits), blk(kPfThreads);
  return launch_k(pf_attn_kernel, gr, blk, pf_attn_smem(), s, true, qh, ql, kv, p);
}

}  // namespace tss
