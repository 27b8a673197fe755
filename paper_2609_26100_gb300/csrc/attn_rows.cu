// Split-KV attention of draft blocks of 17 to 128 rows on the 5th-generation tensor cores (tcgen05),
// head_dim 128: the operation of attention.cu, run as a separate launch per layer on the persistent
// path.  A block of that many rows takes the MMA's 128-row (M) side:
//   S [128 rows x 64 keys] = Q K^T    (Q as bf16 hi + lo, split exactly from the fp16 q rows)
//   O [128 rows x 128]    += P V      (P as bf16 hi + lo; the V tile read MN-major)
// with S (double-buffered) and O in tensor memory, one thread per row for the online softmax, whose
// running maximum is raised only past 2^8 headroom.  A CTA takes one (split, head, request): the
// request's 64-key tiles cut evenly, K and V by TMA through three-slot rings.  Several splits leave
// partials (O, max, sum) that the last CTA of the (request, head) adds in split order.
//
// Bound: latency of the chain TMA -> S -> softmax -> P V per tile (1.4 us) and the set-up and merge
// around it (18 us).  The warp-level kernel, bound by the rate of mma.sync on this GPU, takes 74 us a
// launch for a 128-row block over 777 + 128 keys of the 7B shape, this one 29.5 (one split 39.7, two
// 34.5, five -- more CTAs than SMs -- 44); over 4128 keys 55.
//
// Roles (192 threads): warp 0 TMA producer, warp 1 MMA issuer, warps 2-5 softmax (thread = row).
// Every wait is bounded; on expiry the kernel records a timeout, drains its copies and MMAs and returns.
#include "internal.h"

namespace tss {

namespace {

constexpr int kArThreads = 192;
constexpr int kArKeys = 64;                        // keys per tile
constexpr int kArSlots = 3;                        // slots of the K and of the V ring
constexpr int kArD = 128;
constexpr uint32_t kArQPart = 2 * 128 * kArD;      // 128 rows x 128 columns bf16: two 64-column halves of 16 KiB
constexpr uint32_t kArKV = 2 * kArKeys * kArD;     // one tile's K (or V): two 8 KiB boxes
constexpr uint32_t kArPPart = 128 * kArKeys * 2;   // 128 rows x 64 keys
constexpr uint32_t kArTmem = 256;                  // S x 2 (64 columns each), O (128)

__host__ __device__ inline size_t ar_smem() { return 1024 + 2 * kArQPart + 2 * kArSlots * kArKV + 2 * 2 * kArPPart; }

}  // namespace

__global__ void __launch_bounds__(kArThreads, 1) attn_rows_kernel(const AttnRowsParams p) {
  extern __shared__ uint8_t ar_dyn[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(ar_dyn) + 1023) & ~uintptr_t(1023));
  uint8_t* sq = base;                      // Q hi (two halves), Q lo
  uint8_t* sk = sq + 2 * kArQPart;         // [slot] K
  uint8_t* sv = sk + kArSlots * kArKV;     // [slot] V
  uint8_t* sp = sv + kArSlots * kArKV;     // [2] P hi, P lo; merge weights at the end
  __shared__ uint64_t qfull, kfull[kArSlots], kempty[kArSlots], vfull[kArSlots], vempty[kArSlots];
  __shared__ uint64_t s_full[2], s_free[2], p_full[2], p_free[2], o_full, drain;
  __shared__ uint32_t tslot;
  __shared__ int abort_s, s_last;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int split = blockIdx.x, h = blockIdx.y, b = blockIdx.z, H = p.n_heads;
  griddep_wait();
  const StepDesc* st = p.step;
  const PlanDev* pl = p.plan;
  if (b >= st->B || p.slot >= pl->n_act) return;
  const int crow = pl->slot_crow[p.slot][b];
  if (crow < 0) return;  // the request skips this layer (the whole CTA)
  const int N = st->req_nodes[b], ctx = st->req_ctx[b], T = ctx + N;
  const int n_tiles = (T + kArKeys - 1) / kArKeys, per = (n_tiles + p.n_splits - 1) / p.n_splits;
  const int used = (n_tiles + per - 1) / per;  // splits that hold tiles
  const int t0 = split * per, n = min(n_tiles, t0 + per) - t0;
  if (n <= 0) return;
  if (tid == 0) {
    mbar_init(&qfull, 1);
    for (int i = 0; i < kArSlots; ++i) {
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
    tmem_alloc(&tslot, kArTmem);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tm = tslot;
  volatile int* abort = &abort_s;

  if (warp == 0) {
    // ---------------- TMA producer: K and V of every key tile ----------------
    if (lane == 0) {
      const CUtensorMap* map = p.kv_maps + pl->act_layer[p.slot];
      prefetch_tmap(map);
      const size_t cap = static_cast<size_t>(st->kv_cap);
      const int rowK = static_cast<int>(((static_cast<size_t>(st->req_slot[b]) * 2) * H + h) * cap) + t0 * kArKeys;
      const int rowV = rowK + static_cast<int>(static_cast<size_t>(H) * cap);
      int nk = 0, nv = 0;
      for (int t = 0; t < n; ++t) {
        const int s = t % kArSlots;
        if (t >= kArSlots && !mbar_wait(&kempty[s], ((t / kArSlots) - 1) & 1, abort, p.status)) break;
        mbar_arrive_expect_tx(&kfull[s], kArKV);
        tma_load_2d(sk + s * kArKV, map, &kfull[s], 0, rowK + t * kArKeys);
        tma_load_2d(sk + s * kArKV + kArKV / 2, map, &kfull[s], 64, rowK + t * kArKeys);
        ++nk;
        if (t >= kArSlots && !mbar_wait(&vempty[s], ((t / kArSlots) - 1) & 1, abort, p.status)) break;
        mbar_arrive_expect_tx(&vfull[s], kArKV);
        tma_load_2d(sv + s * kArKV, map, &vfull[s], 0, rowV + t * kArKeys);
        tma_load_2d(sv + s * kArKV + kArKV / 2, map, &vfull[s], 64, rowV + t * kArKeys);
        ++nv;
      }
      // the copies issued last into each slot have landed before the kernel returns
      for (int u = nk - 1; u >= 0 && u >= nk - kArSlots; --u) mbar_drain(&kfull[u % kArSlots], (u / kArSlots) & 1);
      for (int u = nv - 1; u >= 0 && u >= nv - kArSlots; --u) mbar_drain(&vfull[u % kArSlots], (u / kArSlots) & 1);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer: S(t) = Q K^T, then O += P(t - 1) V ----------------
    if (lane == 0) {
      const uint32_t idS = idesc_bf16_m128(kArKeys), idPV = idesc_bf16_m128(kArD) | (1u << 16);  // (B MN-major)
      const uint32_t q_a = smem_u32(sq), k_a = smem_u32(sk), v_a = smem_u32(sv), p_a = smem_u32(sp);
      // fault injection: the first CTA at work issues no MMA, so its softmax's first wait runs out
      const bool withheld = p.withhold && crow == 0 && h == 0 && split == 0;
      const bool ok = mbar_wait(&qfull, 0, abort, p.status) && !withheld;
      for (int t = 0; ok && t <= n; ++t) {
        if (t < n) {
          const int s = t % kArSlots;
          if (!mbar_wait(&kfull[s], (t / kArSlots) & 1, abort, p.status)) break;
          if (t >= 2 && !mbar_wait(&s_free[t & 1], ((t >> 1) - 1) & 1, abort, p.status)) break;
          tc_fence_after();
          const uint32_t dS = tm + (t & 1) * kArKeys;
#pragma unroll
          for (int part = 0; part < 2; ++part)
#pragma unroll
            for (int kb = 0; kb < 2; ++kb)
#pragma unroll
              for (int k16 = 0; k16 < 4; ++k16)
                umma_bf16(dS, sdesc_sw128(q_a + part * kArQPart + kb * (kArQPart / 2) + k16 * 32),
                          sdesc_sw128(k_a + s * kArKV + kb * (kArKV / 2) + k16 * 32), idS, (part | kb | k16) ? 1u : 0u);
          umma_commit(&s_full[t & 1]);
          umma_commit(&kempty[s]);
        }
        if (t >= 1) {
          const int u = t - 1, s = u % kArSlots;
          if (!mbar_wait(&vfull[s], (u / kArSlots) & 1, abort, p.status)) break;
          if (!mbar_wait(&p_full[u & 1], (u >> 1) & 1, abort, p.status)) break;
          tc_fence_after();
          const uint32_t pb = p_a + (u & 1) * 2 * kArPPart;
#pragma unroll
          for (int part = 0; part < 2; ++part)
#pragma unroll
            for (int kk = 0; kk < kArKeys / 16; ++kk)
              umma_bf16(tm + 128, sdesc_sw128(pb + part * kArPPart + kk * 32),
                        sdesc_sw128_mn(v_a + s * kArKV + kk * 16 * 128, kArKV / 2), idPV, (u | part | kk) ? 1u : 0u);
          umma_commit(&vempty[s]);
          umma_commit(&p_free[u & 1]);
          if (u == n - 1) umma_commit(&o_full);
        }
      }
      // every MMA issued has completed before the kernel returns
      umma_commit(&drain);
      mbar_drain(&drain, 0);
    }
  } else {
    // ---------------- softmax: thread = row (TMEM lane) ----------------
    const int qr = (warp & 3) * 32 + lane, sth = tid - 64;
    const uint32_t lanes = static_cast<uint32_t>((warp & 3) * 32) << 16;
    const bool valid = qr < N;
    // Q: fp16, split exactly into bf16 hi + lo, K-major 128-byte swizzle; rows past the block zero.  16
    // lanes read a row, so that a warp's loads cover whole lines; eight rows' loads in flight.
    for (int r0 = (sth >> 4); r0 < 128; r0 += 64) {
      const int c = sth & 15;
      uint4 raw[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int r = r0 + 8 * k;
        raw[k] = r < N ? *reinterpret_cast<const uint4*>(p.q + static_cast<size_t>(crow + r) * p.d_model + h * kArD + c * 8)
                       : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const int r = r0 + 8 * k;
        const uint32_t w[4] = {raw[k].x, raw[k].y, raw[k].z, raw[k].w};
        uint32_t hi[4], lo[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
          hi[i] = pack_bf16(f.x, f.y);
          lo[i] = pack_bf16(f.x - __uint_as_float(hi[i] << 16), f.y - __uint_as_float(hi[i] & 0xffff0000u));
        }
        uint8_t* d = sq + (c >> 3) * (kArQPart / 2) + r * 128 + (((c & 7) ^ (r & 7)) << 4);
        *reinterpret_cast<uint4*>(d) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
        *reinterpret_cast<uint4*>(d + kArQPart) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      }
    }
    fence_async_smem();
    named_bar_sync(1, 128);
    if (sth == 0) mbar_arrive(&qfull);
    const int row0 = st->req_rowoff[b];
    const unsigned long long anc_lo = valid ? st->row_anc[row0 + qr] : 0ull, anc_hi = valid ? st->row_anc_hi[row0 + qr] : 0ull;
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int t = 0; t < n; ++t) {
      ok = mbar_wait(&s_full[t & 1], (t >> 1) & 1, abort, p.status);
      if (bar_or<1>(!ok)) break;
      tc_fence_after();
      float s[kArKeys];
#pragma unroll
      for (int c = 0; c < kArKeys / 16; ++c) tmem_ld16(tm + lanes + (t & 1) * kArKeys + c * 16, s + c * 16);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&s_free[t & 1]);
      // keys of the tile that the row sees: context keys, then the row's ancestors and itself
      const int k0 = (t0 + t) * kArKeys;
      unsigned long long vis = ~0ull;
      if (k0 + kArKeys > ctx) {
        if (k0 < ctx) {
          const int c = ctx - k0;  // 1..63
          vis = ((1ull << c) - 1) | (anc_lo << c);
        } else {
          const int j = k0 - ctx;  // block row of the tile's first key, 0..127
          vis = j == 0 ? anc_lo : j < 64 ? (anc_lo >> j) | (anc_hi << (64 - j)) : anc_hi >> (j - 64);
        }
      }
      float mt = -INFINITY;
#pragma unroll
      for (int c = 0; c < kArKeys; ++c) {
        s[c] = ((vis >> c) & 1ull) ? s[c] * p.scale_log2 : -INFINITY;
        mt = fmaxf(mt, s[c]);
      }
      // the row's running max is raised only when the tile exceeds it by more than 2^8; the warp
      // rescales its rows of O together (tensor-memory access is warp-wide)
      const bool raise = mt > m + 8.f;
      float alpha = 1.f;
      if (raise) {
        alpha = m == -INFINITY ? 1.f : exp2f(m - mt);
        m = mt;
        l *= alpha;
      }
      const bool rescale = t >= 1 && __any_sync(0xffffffffu, raise && alpha != 1.f);
      ok = t < 2 || mbar_wait(&p_free[t & 1], ((t >> 1) - 1) & 1, abort, p.status);
      if (rescale && ok) ok = mbar_wait(&p_free[(t - 1) & 1], ((t - 1) >> 1) & 1, abort, p.status);
      // in the request's last tile, the V rows past its keys (stale or unwritten cache rows) are zeroed
      if (ok && t0 + t == n_tiles - 1) {
        const int s_ = t % kArSlots, r0 = T - k0;
        ok = mbar_wait(&vfull[s_], (t / kArSlots) & 1, abort, p.status);
        if (ok && sth >= r0 && sth < kArKeys) {
          uint4* v0 = reinterpret_cast<uint4*>(sv + s_ * kArKV + sth * 128);
          uint4* v1 = reinterpret_cast<uint4*>(sv + s_ * kArKV + kArKV / 2 + sth * 128);
#pragma unroll
          for (int i = 0; i < 8; ++i) v0[i] = v1[i] = make_uint4(0, 0, 0, 0);
        }
      }
      if (bar_or<1>(!ok)) break;
      if (rescale) {
        tc_fence_after();
        float o[16];
#pragma unroll
        for (int c = 0; c < kArD / 16; ++c) {
          tmem_ld16(tm + lanes + 128 + c * 16, o);
#pragma unroll
          for (int i = 0; i < 16; ++i) o[i] *= alpha;
          tmem_st16(tm + lanes + 128 + c * 16, o);
        }
        tc_fence_before();
      }
      // weights 2^(s - m) as bf16 hi + lo into the P operand (row qr, 64 keys = one 128-byte row)
      const float mb = m == -INFINITY ? 0.f : m;
      uint8_t* ph = sp + (t & 1) * 2 * kArPPart + qr * 128;
#pragma unroll
      for (int c8 = 0; c8 < kArKeys / 8; ++c8) {
        uint32_t hw[4], lw[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float w0 = exp2f(s[c8 * 8 + 2 * i] - mb), w1 = exp2f(s[c8 * 8 + 2 * i + 1] - mb);
          l += w0 + w1;
          hw[i] = pack_bf16(w0, w1);
          lw[i] = pack_bf16(w0 - __uint_as_float(hw[i] << 16), w1 - __uint_as_float(hw[i] & 0xffff0000u));
        }
        const int sw = (c8 ^ (qr & 7)) << 4;
        *reinterpret_cast<uint4*>(ph + sw) = make_uint4(hw[0], hw[1], hw[2], hw[3]);
        *reinterpret_cast<uint4*>(ph + kArPPart + sw) = make_uint4(lw[0], lw[1], lw[2], lw[3]);
      }
      fence_async_smem();
      named_bar_sync(1, 128);
      if (sth == 0) mbar_arrive(&p_full[t & 1]);
    }
    if (ok) ok = mbar_wait(&o_full, 0, abort, p.status);
    if (!bar_or<1>(!ok)) {
      tc_fence_after();
      const size_t item = static_cast<size_t>(b) * H + h;
      if (used == 1) {
        const float inv = l > 0.f ? 1.f / l : 0.f;
        if (valid && !(l > 0.f)) report(p.status, kStatusCheck);
#pragma unroll
        for (int c = 0; c < kArD / 16; ++c) {
          float o[16];
          tmem_ld16(tm + lanes + 128 + c * 16, o);
          if (valid) {
#pragma unroll
            for (int i = 0; i < 16; ++i) o[i] *= inv;
#pragma unroll
            for (int i = 0; i < 4; ++i) store_split4(split_at(p.o, p.o_xs, h * kArD + c * 16 + 4 * i), crow + qr, o + 4 * i);
          }
        }
        tc_fence_before();
      } else {
        const size_t pi = (item * p.n_splits + split) * p.nb + qr;
        if (valid) __stcg(reinterpret_cast<float2*>(p.part_ml) + pi, make_float2(m, l));
#pragma unroll
        for (int c = 0; c < kArD / 16; ++c) {
          float o[16];
          tmem_ld16(tm + lanes + 128 + c * 16, o);
          if (valid) {
            float4* d = reinterpret_cast<float4*>(p.part_o + pi * kArD + c * 16);
#pragma unroll
            for (int i = 0; i < 4; ++i) __stcg(d + i, make_float4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]));
          }
        }
        tc_fence_before();
        named_bar_sync(1, 128);  // every thread's partial precedes the release below
        if (sth == 0) {
          s_last = atom_add_acq_rel_gpu(&p.counters[item], 1) == used - 1;
          if (s_last) atomicExch(&p.counters[item], 0);
        }
        named_bar_sync(1, 128);
        if (s_last) {  // (the counter's acquire, then the barrier: the other partials are visible)
          float* wgt = reinterpret_cast<float*>(sp);  // [split][128] (the MMAs that read P are complete)
          const float2* ml = reinterpret_cast<const float2*>(p.part_ml) + item * p.n_splits * p.nb + qr;
          if (valid) {
            float M = -INFINITY, L = 0.f;
            for (int x = 0; x < used; ++x) M = fmaxf(M, __ldcg(ml + x * p.nb).x);
            const float mb = M == -INFINITY ? 0.f : M;
            for (int x = 0; x < used; ++x) {
              const float2 v = __ldcg(ml + x * p.nb);
              const float f = exp2f(v.x - mb);
              L += f * v.y;
              wgt[x * 128 + qr] = f;
            }
            if (!(L > 0.f)) report(p.status, kStatusCheck);
            const float inv = L > 0.f ? 1.f / L : 0.f;
            for (int x = 0; x < used; ++x) wgt[x * 128 + qr] *= inv;
          }
          named_bar_sync(1, 128);
          // units (4 columns of a row): the loads of kU units and kS splits in flight together
          constexpr int kU = 4, kS = 4;
          const float* po = p.part_o + item * p.n_splits * p.nb * kArD;
          for (int u0 = sth; u0 < N * (kArD / 4); u0 += kU * 128) {
            float4 a[kU];
#pragma unroll
            for (int k = 0; k < kU; ++k) a[k] = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int x0 = 0; x0 < used; x0 += kS) {
              float4 v[kS][kU];
#pragma unroll
              for (int y = 0; y < kS; ++y)
#pragma unroll
                for (int k = 0; k < kU; ++k) {
                  const int u = u0 + k * 128;
                  v[y][k] = x0 + y < used && u < N * (kArD / 4)
                                ? __ldcg(reinterpret_cast<const float4*>(po + static_cast<size_t>(x0 + y) * p.nb * kArD) + u)
                                : make_float4(0.f, 0.f, 0.f, 0.f);
                }
#pragma unroll
              for (int y = 0; y < kS; ++y)
                if (x0 + y < used)
#pragma unroll
                  for (int k = 0; k < kU; ++k) {
                    const float f = wgt[(x0 + y) * 128 + min((u0 + k * 128) / (kArD / 4), 127)];
                    a[k].x += f * v[y][k].x;
                    a[k].y += f * v[y][k].y;
                    a[k].z += f * v[y][k].z;
                    a[k].w += f * v[y][k].w;
                  }
            }
#pragma unroll
            for (int k = 0; k < kU; ++k) {
              const int u = u0 + k * 128;
              if (u < N * (kArD / 4)) {
                const float o[4] = {a[k].x, a[k].y, a[k].z, a[k].w};
                store_split4(split_at(p.o, p.o_xs, h * kArD + (u % (kArD / 4)) * 4), crow + u / (kArD / 4), o);
              }
            }
          }
        }
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tm, kArTmem);
  }
}

cudaError_t attn_rows_prepare() {
  return cudaFuncSetAttribute(attn_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(ar_smem()));
}

cudaError_t launch_attention_rows(const AttnRowsParams& p, int B, cudaStream_t s, bool pdl) {
  return launch_k(attn_rows_kernel, dim3(p.n_splits, p.n_heads, B), dim3(kArThreads), ar_smem(), s, pdl, p);
}

}  // namespace tss
