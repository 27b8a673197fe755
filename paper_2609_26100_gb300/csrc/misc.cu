// Row-wise and per-request kernels of the verification step: the skip controller, embedding
// gather, RMSNorm, acceptance (greedy walk or speculative sampling) and KV compaction.
#include "internal.h"

namespace tss {

// ------------------------------------------------------------------------------------------
// Skip controller (Sec. "Domain-Aware Skip Controller", first equation; Sec.
// "Domain-to-Configuration Mapping"): S(x) = Phi(d(x)) if the domain is configured, else the
// empty set -- looked up on the host when the step is enqueued and passed in the step
// descriptor.  From the requests' skip sets it builds, on the device, the ascending list of
// layers that at least one request runs (the only layers that get launches) and, per layer, the
// compacted list of rows of the requests that run it.
// ------------------------------------------------------------------------------------------
// A warp builds a slot's lists: lanes over the requests for their first compacted rows (a scan of
// the running requests' row counts), then over the rows.
__device__ void controller_body(const MiscParams& p) {
  const StepDesc* st = p.step;
  PlanDev* pl = p.plan;
  __shared__ unsigned long long smask[kMaxBatch];
  __shared__ int snodes[kMaxBatch], soff[kMaxBatch];
  __shared__ int sact[kMaxLayers];
  __shared__ unsigned long long s_all;  // layers that every request skips
  const int B = st->B, L = p.n_layers;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int b = threadIdx.x; b < B; b += blockDim.x) {
    const unsigned long long m = st->req_phi[b];
    smask[b] = m;
    snodes[b] = st->req_nodes[b];
    soff[b] = st->req_rowoff[b];
    pl->req_mask[b] = m;
  }
  __syncthreads();
  if (warp == 0) {
    unsigned long long all = ~0ull;
    for (int b = lane; b < B; b += 32) all &= smask[b];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) all &= __shfl_xor_sync(0xffffffffu, all, o);
    if (lane == 0) s_all = all;
  }
  __syncthreads();
  const unsigned long long runs = ~s_all & (L == 64 ? ~0ull : (1ull << L) - 1);
  const int n = __popcll(runs);
  if (threadIdx.x < L && ((runs >> threadIdx.x) & 1ull)) {
    const int j = __popcll(runs & ((1ull << threadIdx.x) - 1));
    sact[j] = threadIdx.x;
    pl->act_layer[j] = threadIdx.x;
  }
  if (threadIdx.x == 0) {
    pl->n_act = n;
    if (n != st->n_act_host) report(p.status, kStatusCheck);
  }
  __syncthreads();
  for (int j = warp; j <= n; j += nw) {
    const int slot = j == n ? kFinalSlot : j, l = j == n ? 0 : sact[j];
    int base = 0;
    for (int b0 = 0; b0 < B; b0 += 32) {
      const int b = b0 + lane;
      const bool run = b < B && (j == n || !((smask[b] >> l) & 1ull));
      const int c = run ? snodes[b] : 0;
      int incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const int first = base + incl - c;
      if (b < B) pl->slot_crow[slot][b] = run ? first : -1;
      // the rows of each running request, by the whole warp
      unsigned todo = __ballot_sync(0xffffffffu, run);
      while (todo) {
        const int k = __ffs(todo) - 1;
        todo &= todo - 1;
        const int f = __shfl_sync(0xffffffffu, first, k), cnt = __shfl_sync(0xffffffffu, c, k), r0 = soff[b0 + k];
        for (int i = lane; i < cnt; i += 32) pl->slot_rows[slot][f + i] = r0 + i;
      }
      base += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) pl->slot_M[slot] = base;
  }
}

__global__ void controller_kernel(const MiscParams p) {
  griddep_wait();
  griddep_launch();
  controller_body(p);
}

// h[m] = E[token[m]] (fp32 residual stream).
__global__ void embed_kernel(const MiscParams p) {
  griddep_wait();
  griddep_launch();
  const StepDesc* st = p.step;
  const int m = blockIdx.x;
  if (m >= st->M) return;
  int tok = st->tokens[caller_row(st, m)];
  if (tok < 0 || tok >= p.vocab) {
    if (threadIdx.x == 0) report(p.status, kStatusCheck);
    tok = 0;
  }
  const __nv_bfloat16* e = p.embed + static_cast<size_t>(tok) * p.d_model;
  float* h = p.h + static_cast<size_t>(m) * p.d_model;
  for (int i = threadIdx.x; i < p.d_model; i += blockDim.x) h[i] = __bfloat162float(e[i]);
}

__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (lane == 0) red[w] = v;
  __syncthreads();
  float t = 0.f;
  for (int i = 0; i < nw; ++i) t += red[i];
  __syncthreads();
  return t;
}

// xn[n] = bf16(h[row_n] / sqrt(mean(h^2) + eps) * g) for the compacted rows n of a slot.
__global__ void rmsnorm_kernel(const MiscParams p, int slot, int which) {
  griddep_wait();
  griddep_launch();
  __shared__ float red[32];
  const PlanDev* pl = p.plan;
  const int n = blockIdx.x;
  const bool final_slot = which == 2;
  const int sl = final_slot ? kFinalSlot : slot;
  if (!final_slot && slot >= pl->n_act) return;
  if (n >= pl->slot_M[sl]) return;
  const int m = pl->slot_rows[sl][n];
  const int d = p.d_model;
  const float* g = final_slot ? p.g_final : (which == 0 ? p.g_attn : p.g_mlp) + static_cast<size_t>(pl->act_layer[slot]) * d;
  const float* h = p.h + static_cast<size_t>(m) * d;
  float ss = 0.f;
  for (int i = threadIdx.x; i < d; i += blockDim.x) ss += h[i] * h[i];
  ss = block_sum(ss, red);
  const float rs = rsqrtf(ss / static_cast<float>(d) + p.rms_eps);
  __nv_bfloat16* x = p.xn + static_cast<size_t>(n) * d;
  for (int i = threadIdx.x; i < d; i += blockDim.x) x[i] = __float2bfloat16_rn(h[i] * rs * g[i]);
}

// ------------------------------------------------------------------------------------------
// Acceptance.  Greedy (temperature 0, Sec. "Evaluation Protocol"): from the root, step to the
// lowest-index child whose token equals the argmax of the current row while one exists; the
// bonus is the argmax of the last row reached.  Argmax ties go to the lowest token id.
// ------------------------------------------------------------------------------------------
// Request b's results, written by every thread of the block (a, bonus and path[0..a] are the
// same in all of them; path is in shared memory).  The descriptor's fields are read once into
// registers: read inside a loop of stores through the descriptor's pointers, each would be
// reloaded from L2 after every store.
__device__ void write_result(const MiscParams& p, int b, int a, int bonus, const int* path) {
  const StepDesc* st = p.step;
  PlanDev* pl = p.plan;
  const int stride = st->path_stride, ob = st->req_rng[b];
  int* out = st->path + static_cast<size_t>(ob) * stride;
  for (int i = threadIdx.x; i < stride; i += blockDim.x) out[i] = i <= a ? path[i] : -1;
  for (int i = threadIdx.x; i <= a; i += blockDim.x) pl->res_path[b][i] = path[i];
  if (threadIdx.x == 0) {
    const int ctx = st->req_ctx[b];
    int* accept_len = st->accept_len;
    int* bonus_out = st->bonus;
    int* new_ctx = st->new_ctx;
    accept_len[ob] = a;
    bonus_out[ob] = bonus;
    new_ctx[ob] = ctx + 1 + a;
    pl->res_accept[b] = a;
  }
}

// Greedy acceptance of request b; returns the accept length (the same in every thread) and
// leaves the accepted path in path[0..a].
__device__ int accept_greedy_body(const MiscParams& p, int b, int* path) {
  const StepDesc* st = p.step;
  __shared__ int am[kMaxNodes];
  __shared__ int s_par[kMaxNodes], s_tok[kMaxNodes];
  __shared__ int s_a, s_bonus;
  const int N = st->req_nodes[b], off = st->req_rowoff[b];
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    s_par[i] = st->row_parent[off + i];
    s_tok[i] = st->tokens[st->req_orow[b] + i];
  }
  // Argmax of every row over the vocabulary tiles' partials (laid out [tile][row]): thread
  // (g, r), g < G = blockDim / RP, scans row r's tiles g, g + G, ..., so that a warp's loads
  // cover consecutive rows of one tile; then the G results of each row are combined.  The
  // maximum with ties to the lowest token id does not depend on the order of the comparisons.
  auto better = [](float v, int ix, float& bv, int& bi) {
    if (v > bv || (v == bv && ix < bi)) {
      bv = v;
      bi = ix;
    }
  };
  const int RP = N > 32 ? (N + 31) & ~31 : 32, G = blockDim.x / RP;
  const int r = threadIdx.x % RP, g = threadIdx.x / RP, n_vt = p.n_vtiles;
  float bv = -INFINITY;
  int bi = 0x7fffffff;
  if (g < G && r < N) {
    const float* pv = p.amax_val + off + r;
    const int* pi = p.amax_idx + off + r;
    constexpr int kPer = 8;  // tiles per thread in one round of loads
    for (int t0 = g; t0 < n_vt; t0 += kPer * G) {
      float vv[kPer];
      int vi[kPer];
#pragma unroll
      for (int q = 0; q < kPer; ++q) {
        const int t = t0 + q * G;
        const bool in = t < n_vt;
        vv[q] = in ? pv[static_cast<size_t>(t) * kMaxRows] : -INFINITY;
        vi[q] = in ? pi[static_cast<size_t>(t) * kMaxRows] : 0x7fffffff;
      }
#pragma unroll
      for (int q = 0; q < kPer; ++q) better(vv[q], vi[q], bv, bi);
    }
  }
  __shared__ float s_bv[1024];
  __shared__ int s_bi[1024];
  s_bv[threadIdx.x] = bv;
  s_bi[threadIdx.x] = bi;
  __syncthreads();
  if (threadIdx.x < N) {
    float v = -INFINITY;
    int ix = 0x7fffffff;
    for (int gg = 0; gg < G; ++gg) better(s_bv[gg * RP + threadIdx.x], s_bi[gg * RP + threadIdx.x], v, ix);
    am[threadIdx.x] = ix;
  }
  __syncthreads();
  if (threadIdx.x < 32) {  // one warp walks, its lanes over the nodes of each level's search
    const int lane = threadIdx.x;
    int cur = 0, a = 0;
    if (lane == 0) path[0] = 0;
    while (true) {
      const int want = am[cur];
      int nxt = -1;
      for (int c0 = cur + 1; c0 < N && nxt < 0; c0 += 32) {
        const int c = c0 + lane;
        const unsigned hit = __ballot_sync(0xffffffffu, c < N && s_par[c] == cur && s_tok[c] == want);
        if (hit) nxt = c0 + __ffs(hit) - 1;
      }
      if (nxt < 0) break;
      cur = nxt;
      ++a;
      if (lane == 0) path[a] = cur;
    }
    if (lane == 0) {
      s_a = a;
      s_bonus = am[cur];
    }
  }
  __syncthreads();
  const int a = s_a;
  write_result(p, b, a, s_bonus, path);
  return a;
}

__global__ void accept_greedy_kernel(const MiscParams p) {
  griddep_wait();
  griddep_launch();
  if (blockIdx.x >= p.step->B) return;
  __shared__ int path[kMaxNodes];
  accept_greedy_body(p, blockIdx.x, path);
}

// Philox4x32-10 (Salmon et al., SC'11): 10 rounds of the 4x32 Philox round with key bumps.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
  }
  return c;
}

// The generator's output for uniform slot `slot` of request b: counter (slot, request, offset lo,
// offset hi), key (seed lo, seed hi); the uniform is (first word >> 8) * 2^-24, exact in fp32.
__device__ __forceinline__ uint4 philox_slot(uint32_t seed_lo, uint32_t seed_hi, uint32_t off_lo, uint32_t off_hi,
                                             int b, int slot) {
  return philox4x32_10(make_uint4(static_cast<uint32_t>(slot), static_cast<uint32_t>(b), off_lo, off_hi), seed_lo,
                       seed_hi);
}
__device__ __forceinline__ float uniform24(uint32_t x) { return static_cast<float>(x >> 8) * (1.f / 16777216.f); }

__device__ __forceinline__ double draw_uniform(const StepDesc* st, int b, int slot) {
  if (st->uniforms) return static_cast<double>(st->uniforms[static_cast<size_t>(st->req_rng[b]) * st->uniform_stride + slot]);
  return static_cast<double>(
      uniform24(philox_slot(st->seed_lo, st->seed_hi, st->off_lo, st->off_hi, st->req_rng[b], slot).x));
}

// Diagnostic: the generator's words and uniforms for requests [0, n_req) and slots [0, n_slots)
// of one (seed, offset), laid out [request][slot] (the stream the acceptance draws from).
__global__ void philox_fill_kernel(uint32_t seed_lo, uint32_t seed_hi, uint32_t off_lo, uint32_t off_hi, int n_req,
                                   int n_slots, uint4* words, float* unif) {
  const size_t n = static_cast<size_t>(n_req) * n_slots;
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int b = static_cast<int>(i / n_slots), slot = static_cast<int>(i - static_cast<size_t>(b) * n_slots);
    const uint4 x = philox_slot(seed_lo, seed_hi, off_lo, off_hi, b, slot);
    if (words) words[i] = x;
    if (unif) unif[i] = uniform24(x.x);
  }
}

cudaError_t launch_philox_fill(uint64_t seed, uint64_t offset, int n_req, int n_slots, uint32_t* words, float* unif,
                               cudaStream_t s) {
  const size_t n = static_cast<size_t>(n_req) * n_slots;
  const int blocks = static_cast<int>((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  philox_fill_kernel<<<blocks, 256, 0, s>>>(static_cast<uint32_t>(seed), static_cast<uint32_t>(seed >> 32),
                                            static_cast<uint32_t>(offset), static_cast<uint32_t>(offset >> 32), n_req,
                                            n_slots, reinterpret_cast<uint4*>(words), unif);
  return cudaGetLastError();
}

template <typename T, typename Op>
__device__ __forceinline__ T block_reduce(T v, T* red, Op op) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, off));
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  if (lane == 0) red[w] = v;
  __syncthreads();
  T t = red[0];
  for (int i = 1; i < nw; ++i) t = op(t, red[i]);
  __syncthreads();
  return t;
}

// Inverse CDF over token ids in ascending order: the smallest v whose running sum of w exceeds
// u * sum(w).  Each thread owns a contiguous chunk; chunk sums are scanned in thread order.
// fp32 throughout: the sums over a 32k vocabulary are accurate to ~1e-6 of the mass, far inside
// the 2e-4 band within which a draw counts as consistent, and fp64 is slow on this GPU.
// Loads of the vocabulary passes are issued kLoadBatch at a time (one round trip per batch
// instead of one per element); every sum keeps the element order of a plain loop.
constexpr int kLoadBatch = 16;

template <typename WFn>
__device__ int inverse_cdf_block(int V, float u, WFn w, float* scan) {
  const int nt = blockDim.x, t = threadIdx.x;
  const int C = (V + nt - 1) / nt;
  const int v0 = min(V, t * C), v1 = min(V, v0 + C);
  float local = 0.f;
  for (int b0 = v0; b0 < v1; b0 += kLoadBatch) {
    float x[kLoadBatch];
#pragma unroll
    for (int j = 0; j < kLoadBatch; ++j) x[j] = b0 + j < v1 ? w(b0 + j) : 0.f;
#pragma unroll
    for (int j = 0; j < kLoadBatch; ++j) local += x[j];  // x + 0 == x: the order of a plain loop
  }
  // exclusive scan of the chunk sums in thread order: warp scans, then the warp totals
  const int lane = t & 31, warp = t >> 5, nw = nt >> 5;
  float incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  __shared__ float wsum[32];
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    float x = lane < nw ? wsum[lane] : 0.f;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    if (lane < nw) wsum[lane] = x;  // inclusive totals of warps 0..lane
  }
  __syncthreads();
  const float before = (warp > 0 ? wsum[warp - 1] : 0.f) + (incl - local);
  scan[t] = before;
  if (t == nt - 1) scan[nt] = before + local;
  __syncthreads();
  __shared__ int sel;
  if (t == 0) sel = -1;
  __syncthreads();
  const float total = scan[nt];
  const float target = u * total;
  const float lo = scan[t], hi = (t + 1 < nt) ? scan[t + 1] : total;
  if (local > 0.f && lo <= target && (target < hi || t + 1 == nt || hi >= total)) {
    float run = lo;
    int pick = -1, last_pos = -1;
    for (int v = v0; v < v1; ++v) {
      const float x = w(v);
      if (x > 0.f) last_pos = v;
      run += x;
      if (run > target && x > 0.f) {
        pick = v;
        break;
      }
    }
    if (pick < 0) pick = last_pos;
    atomicCAS(&sel, -1, pick);
  }
  __syncthreads();
  int r = sel;
  if (r < 0) {  // target at or beyond the total: the last token with positive mass
    __shared__ int lastv;
    if (t == 0) lastv = -1;
    __syncthreads();
    for (int v = v1 - 1; v >= v0; --v)
      if (w(v) > 0.f) {
        atomicMax(&lastv, v);
        break;
      }
    __syncthreads();
    r = lastv < 0 ? 0 : lastv;
  }
  __syncthreads();
  return r;
}

// The same inverse CDF over weights staged in shared memory, when the launch gave the block
// enough dynamic shared memory (cdf_stage_bytes): w(v) is computed once per token with coalesced
// loads into a buffer indexed v + v / 32 (the skew puts the 32 consecutive tokens of each
// thread's chunk in 32 different banks), then the chunk sums, scan and walk above read it there.
// Without it each warp-wide load of the chunk pass touches 32 cache lines.
__device__ __forceinline__ unsigned dyn_smem_bytes() {
  unsigned n;
  asm volatile("mov.u32 %0, %%dynamic_smem_size;" : "=r"(n));
  return n;
}

template <typename WFn>
__device__ int inverse_cdf_staged(int V, float u, WFn w, float* scan) {
  extern __shared__ float cdf_stage[];
  const size_t need = cdf_stage_bytes(V);
  if (need == 0 || dyn_smem_bytes() < need) return inverse_cdf_block(V, u, w, scan);
  // kStage weights per thread are computed before any is stored: the stores could alias the
  // generic loads inside w, so a load after a store would wait for it
  constexpr int kStage = 8;
  const int nt = blockDim.x;
  for (int v0 = threadIdx.x; v0 < V; v0 += kStage * nt) {
    float x[kStage];
#pragma unroll
    for (int j = 0; j < kStage; ++j) x[j] = v0 + j * nt < V ? w(v0 + j * nt) : 0.f;
#pragma unroll
    for (int j = 0; j < kStage; ++j) {
      const int v = v0 + j * nt;
      if (v < V) cdf_stage[v + (v >> 5)] = x[j];
    }
  }
  __syncthreads();
  return inverse_cdf_block(V, u, [&](int v) { return cdf_stage[v + (v >> 5)]; }, scan);
}

// Softmax statistics of row m's logits / T, (max, sum of exponentials), by the whole block.  Returns
// true in every thread of the block that completes the last row of m's request.
__device__ bool sample_row_stats(const MiscParams& p, int m, int b) {
  const StepDesc* st = p.step;
  __shared__ float redf[32];
  __shared__ int s_last;
  const int V = p.vocab, nt = blockDim.x;
  const float invT = st->inv_temperature;
  const float* lg = st->logits + static_cast<size_t>(caller_row(st, m)) * V;
  auto fmx = [](float a, float c) { return a > c ? a : c; };
  auto fsum = [](float a, float c) { return a + c; };
  float mx = -INFINITY;
  for (int b0 = threadIdx.x; b0 < V; b0 += kLoadBatch * nt) {
    float x[kLoadBatch];
#pragma unroll
    for (int j = 0; j < kLoadBatch; ++j) x[j] = b0 + j * nt < V ? lg[b0 + j * nt] : -INFINITY;
#pragma unroll
    for (int j = 0; j < kLoadBatch; ++j) mx = fmx(mx, x[j]);
  }
  mx = block_reduce(mx, redf, fmx);
  float z = 0.f;
  for (int b0 = threadIdx.x; b0 < V; b0 += kLoadBatch * nt) {
    float x[kLoadBatch];
#pragma unroll
    for (int j = 0; j < kLoadBatch; ++j) x[j] = b0 + j * nt < V ? lg[b0 + j * nt] : 0.f;
#pragma unroll
    for (int j = 0; j < kLoadBatch; ++j)
      if (b0 + j * nt < V) z += expf((x[j] - mx) * invT);
  }
  z = block_reduce(z, redf, fsum);
  if (threadIdx.x == 0) {
    __stcg(&p.row_stat[2 * m], mx);
    __stcg(&p.row_stat[2 * m + 1], z);
    s_last = atom_add_acq_rel_gpu(&p.row_cnt[b], 1) == st->req_nodes[b] - 1;
    if (s_last) atomicExch(&p.row_cnt[b], 0);
  }
  __syncthreads();
  return s_last != 0;
}

// Speculative sampling on a chain draft (rule of the speculative-decoding works the paper cites
// as its base methods): p_i = softmax(logits_i / T); accept draft x_i iff r_i * q_i(x_i) <
// p_{i-1}(x_i); at the first rejection draw the bonus from normalise(max(0, p_{i-1} - q_i));
// if every draft is accepted draw it from p_k.  Uniform slots: r_i at i-1, u_i at k+i-1.
// A block per row computes the rows' statistics side by side, and the block that finishes a
// request's last row runs the tests of all its drafts at once and the one inverse CDF that the walk
// ends with.  Latency-bound: with one block per request and two passes over the vocabulary for
// every row up to the first rejection, the acceptance of 8 requests of 5 drafts took 67 us.
__device__ int accept_sample_body(const MiscParams& p, int b, int* path) {
  const StepDesc* st = p.step;
  __shared__ float scan[1025];
  __shared__ float s_mx[kMaxNodes], s_iz[kMaxNodes];
  __shared__ int s_stop[kMaxNodes];  // per draft: 0 accepted, 1 rejected, 2 token out of range; + 4: q(x) not positive
  const int N = st->req_nodes[b], off = st->req_rowoff[b], k = N - 1, V = p.vocab;
  const size_t orow = static_cast<size_t>(st->req_orow[b]);
  const float invT = st->inv_temperature;
  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    s_mx[i] = __ldcg(&p.row_stat[2 * (off + i)]);
    s_iz[i] = 1.f / __ldcg(&p.row_stat[2 * (off + i) + 1]);
    path[i] = i;
  }
  __syncthreads();
  for (int i = 1 + threadIdx.x; i <= k; i += blockDim.x) {
    const int x = st->tokens[orow + i];
    int stop = 2;
    if (x >= 0 && x < V) {
      const float qx = st->draft_probs[(orow + i) * V + x];
      const float px = expf((st->logits[(orow + i - 1) * V + x] - s_mx[i - 1]) * invT) * s_iz[i - 1];
      const float r = static_cast<float>(draw_uniform(st, b, i - 1));
      stop = (r * qx < px ? 0 : 1) + (qx > 0.f ? 0 : 4);
    }
    s_stop[i] = stop;
  }
  __syncthreads();
  int i = 1;  // first draft that is not accepted, k + 1: none
  while (i <= k && (s_stop[i] & 3) == 0) ++i;
  if (threadIdx.x == 0)
    for (int j = 1; j <= min(i, k); ++j)
      if (s_stop[j] >= 2) report(p.status, kStatusCheck);
  const int a = i - 1;
  int bonus = 0;
  const float* lg = st->logits + (orow + a) * V;
  const float mx = s_mx[a], invz = s_iz[a];
  auto pr = [&](int v) { return expf((lg[v] - mx) * invT) * invz; };
  if (i > k) {
    bonus = inverse_cdf_staged(V, static_cast<float>(draw_uniform(st, b, 2 * k)), pr, scan);
  } else if ((s_stop[i] & 3) == 1) {
    const float* q = st->draft_probs + (orow + i) * V;
    bonus = inverse_cdf_staged(V, static_cast<float>(draw_uniform(st, b, k + i - 1)), [&](int v) {
      const float d = pr(v) - q[v];
      return d > 0.f ? d : 0.f;
    }, scan);
  }
  __syncthreads();
  write_result(p, b, a, bonus, path);
  return a;
}

__global__ void __launch_bounds__(1024) accept_sample_kernel(const MiscParams p) {
  griddep_wait();
  griddep_launch();
  const int m = blockIdx.x;  // a block per row
  if (m >= p.step->M) return;
  const int b = p.step->row_req[m];
  if (!sample_row_stats(p, m, b)) return;
  __shared__ int path[kMaxNodes];
  accept_sample_body(p, b, path);
}

// ------------------------------------------------------------------------------------------
// Step prologue for the persistent verify kernel: block 0 runs the skip controller; block
// 1 + m embeds row m and writes, per 128-feature tile t, the partial sum of squares
// ssp[t][m] that the RMSNorm of the first active layer needs.
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(256) prologue_kernel(const MiscParams p, float* ssp, int* zero_ints, int n_zero) {
  griddep_wait();
  griddep_launch();
  if (blockIdx.x == 0) {
    // counters and the abort word of the persistent kernel start every step at zero, even after
    // a step that gave up on a timeout
    for (int i = threadIdx.x; i < n_zero; i += blockDim.x) zero_ints[i] = 0;
    controller_body(p);
    return;
  }
  const StepDesc* st = p.step;
  const int m = blockIdx.x - 1;
  if (m >= st->M) return;
  int tok = st->tokens[caller_row(st, m)];
  if (tok < 0 || tok >= p.vocab) {
    if (threadIdx.x == 0) report(p.status, kStatusCheck);
    tok = 0;
  }
  __shared__ unsigned long long smask[kMaxBatch];
  __shared__ int s_l0, s_crow;
  // The first norm phase is the QKV of the union's first layer (or the LM head when every layer
  // is skipped); find this row's compacted position in it, as the controller does.
  for (int b = threadIdx.x; b < st->B; b += blockDim.x) smask[b] = st->req_phi[b];
  __syncthreads();
  if (threadIdx.x == 0) {
    int l0 = -1;
    for (int l = 0; l < p.n_layers && l0 < 0; ++l)
      for (int b = 0; b < st->B; ++b)
        if (!((smask[b] >> l) & 1ull)) {
          l0 = l;
          break;
        }
    const int rb = st->row_req[m];
    int crow = -1;
    if (l0 < 0) {
      crow = m;
    } else if (!((smask[rb] >> l0) & 1ull)) {
      crow = m - st->req_rowoff[rb];
      for (int b = 0; b < rb; ++b)
        if (!((smask[b] >> l0) & 1ull)) crow += st->req_nodes[b];
    }
    s_l0 = l0;
    s_crow = crow;
  }
  __syncthreads();
  const float* gain = s_l0 >= 0 ? p.g_attn + static_cast<size_t>(s_l0) * p.d_model : p.g_final;
  const int xrow = s_crow, d = p.d_model;
  const __nv_bfloat16* e = p.embed + static_cast<size_t>(tok) * d;
  float* h = p.h + static_cast<size_t>(m) * d;
  // 8 consecutive features per thread and turn, every load of the row first (one round trip); 16 lanes
  // hold a 128-feature tile.  (One feature per thread with a barrier per tile pair took 6 us of a
  // 4096-wide row: the instructions of its address arithmetic and stores.)
  constexpr int kPer = 4;  // d_model <= 8192 = 256 threads x 8 x kPer
  uint4 xe[kPer];
  float4 xg[kPer][2];
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int c = (q * 256 + static_cast<int>(threadIdx.x)) * 8;
    xe[q] = make_uint4(0, 0, 0, 0);
    xg[q][0] = xg[q][1] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c < d) {
      xe[q] = *reinterpret_cast<const uint4*>(e + c);
      if (xrow >= 0) {
        xg[q][0] = *reinterpret_cast<const float4*>(gain + c);
        xg[q][1] = *reinterpret_cast<const float4*>(gain + c + 4);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    if (q * 2048 >= d) break;  // (uniform)
    const int c = (q * 256 + static_cast<int>(threadIdx.x)) * 8;
    const uint32_t w[4] = {xe[q].x, xe[q].y, xe[q].z, xe[q].w};
    float x[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      x[2 * i] = __uint_as_float(w[i] << 16);
      x[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
    float sq = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) sq += x[i] * x[i];
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
    if (c < d) {
      *reinterpret_cast<float4*>(h + c) = make_float4(x[0], x[1], x[2], x[3]);
      *reinterpret_cast<float4*>(h + c + 4) = make_float4(x[4], x[5], x[6], x[7]);
      if (xrow >= 0) {
        const float y[8] = {x[0] * xg[q][0].x, x[1] * xg[q][0].y, x[2] * xg[q][0].z, x[3] * xg[q][0].w,
                            x[4] * xg[q][1].x, x[5] * xg[q][1].y, x[6] * xg[q][1].z, x[7] * xg[q][1].w};
        if (p.xs.rows) {
          store_split4(split_at(p.xn, p.xs, c), xrow, y);
          store_split4(split_at(p.xn, p.xs, c + 4), xrow, y + 4);
        } else {
          *reinterpret_cast<uint4*>(p.xn + static_cast<size_t>(xrow) * d + c) =
              make_uint4(pack_bf16(y[0], y[1]), pack_bf16(y[2], y[3]), pack_bf16(y[4], y[5]), pack_bf16(y[6], y[7]));
        }
      }
      if ((threadIdx.x & 15) == 0) ssp[static_cast<size_t>(c >> 7) * kMaxRows + m] = sq;
    }
  }
}

// ------------------------------------------------------------------------------------------
// Step finish: acceptance of request b (greedy walk or speculative sampling), then the KV
// compaction of its accepted path in every layer it ran (one 1024-thread block per request; when
// sampling, one per row: see accept_sample_body).
// ------------------------------------------------------------------------------------------
__global__ void __launch_bounds__(1024) finish_kernel(const MiscParams p) {
  griddep_wait();
  griddep_launch();
  const StepDesc* st = p.step;
  const PlanDev* pl = p.plan;
  __shared__ int path[kMaxNodes];
  if (st->mode == TSS_MODE_SAMPLE) {  // a block per row; chains only, whose accepted rows are in place
    const int m = blockIdx.x;
    if (m >= st->M) return;
    const int b = st->row_req[m];
    if (sample_row_stats(p, m, b)) accept_sample_body(p, b, path);
    return;
  }
  const int b = blockIdx.x;
  if (b >= st->B) return;
  const int a = accept_greedy_body(p, b, path);
  if (a <= 0) return;
  // A chain's accepted rows are already in place (path[j] == j): nothing moves in any layer.
  bool moved = false;
  for (int jj = 1; jj <= a; ++jj) moved |= path[jj] != jj;
  if (!moved) return;
  const int D = p.head_dim, H = p.n_heads;
  const size_t cap = static_cast<size_t>(st->kv_cap);
  const size_t ctx = static_cast<size_t>(st->req_ctx[b]);
  const int n_act = pl->n_act;
  // request b's cache region in every layer it ran, looked up by one thread per layer (null
  // where it skipped the layer), so that the copies below wait on no descriptor loads
  __shared__ __nv_bfloat16* s_base[kMaxLayers];
  const size_t slot_off = static_cast<size_t>(st->req_slot[b]) * 2 * H * cap * D;
  for (int j = threadIdx.x; j < n_act; j += blockDim.x)
    s_base[j] = pl->slot_crow[j][b] < 0 ? nullptr : st->kv_layer[pl->act_layer[j]] + slot_off;
  __syncthreads();
  // 16-byte units (head_dim is 64 or 128): unit e = (kind, head, 8 dims) of a layer stays with one
  // thread.  No step of the path reads a row that an earlier one wrote (path[jj] >= jj, increasing), so
  // the loads of kMove steps go out before their stores: one round trip a layer.
  const int vec = D / 8;
  constexpr int kMove = 8;
  for (int e = threadIdx.x; e < 2 * H * vec; e += blockDim.x) {
    const int kind_head = e / vec, u = e - kind_head * vec;
    const size_t off = static_cast<size_t>(kind_head) * cap * D;
    for (int j = 0; j < n_act; ++j) {
      if (!s_base[j]) continue;
      uint4* rows = reinterpret_cast<uint4*>(s_base[j] + off) + ctx * vec + u;
      for (int j0 = 1; j0 <= a; j0 += kMove) {
        uint4 x[kMove];
#pragma unroll
        for (int k = 0; k < kMove; ++k)
          if (j0 + k <= a) x[k] = rows[path[j0 + k] * vec];
#pragma unroll
        for (int k = 0; k < kMove; ++k)
          if (j0 + k <= a) rows[(j0 + k) * vec] = x[k];
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// KV compaction: for every layer the request ran, cache rows ctx + path[j] move to ctx + j,
// j = 1..a (the root's row stays).  path[j] > j - 1 and increasing, so copying j in increasing
// order never overwrites a row that a later j still reads.  Chains leave the cache unchanged.
// ------------------------------------------------------------------------------------------
__global__ void compact_kernel(const MiscParams p) {
  griddep_wait();
  griddep_launch();
  const StepDesc* st = p.step;
  const PlanDev* pl = p.plan;
  const int head = blockIdx.x, b = blockIdx.y, j = blockIdx.z;
  if (b >= st->B || j >= pl->n_act || pl->slot_crow[j][b] < 0) return;
  const int a = pl->res_accept[b];
  if (a <= 0) return;
  const int D = p.head_dim, H = p.n_heads;
  const size_t cap = static_cast<size_t>(st->kv_cap);
  __nv_bfloat16* K = st->kv_layer[pl->act_layer[j]] + ((static_cast<size_t>(st->req_slot[b]) * 2) * H + head) * cap * D;
  __nv_bfloat16* Vv = K + static_cast<size_t>(H) * cap * D;
  const size_t ctx = static_cast<size_t>(st->req_ctx[b]);
  for (int jj = 1; jj <= a; ++jj) {
    const int src = pl->res_path[b][jj];
    if (src == jj) continue;
    for (int dd = threadIdx.x; dd < D; dd += blockDim.x) {
      K[(ctx + jj) * D + dd] = K[(ctx + src) * D + dd];
      Vv[(ctx + jj) * D + dd] = Vv[(ctx + src) * D + dd];
    }
  }
}

__global__ void bf16_to_f32_kernel(const __nv_bfloat16* src, float* dst, size_t n) {
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x)
    dst[i] = __bfloat162float(src[i]);
}

cudaError_t misc_prepare() {
  const int c = cudaSharedmemCarveoutMaxShared;
  const cudaFuncAttribute a = cudaFuncAttributePreferredSharedMemoryCarveout;
  cudaError_t e;
  if ((e = cudaFuncSetAttribute(controller_kernel, a, c)) || (e = cudaFuncSetAttribute(embed_kernel, a, c)) ||
      (e = cudaFuncSetAttribute(rmsnorm_kernel, a, c)) || (e = cudaFuncSetAttribute(accept_greedy_kernel, a, c)) ||
      (e = cudaFuncSetAttribute(accept_sample_kernel, a, c)) || (e = cudaFuncSetAttribute(compact_kernel, a, c)) ||
      (e = cudaFuncSetAttribute(prologue_kernel, a, c)) || (e = cudaFuncSetAttribute(finish_kernel, a, c)))
    return e;
  const int dyn = static_cast<int>(kCdfStageMaxBytes);
  const cudaFuncAttribute mx = cudaFuncAttributeMaxDynamicSharedMemorySize;
  if ((e = cudaFuncSetAttribute(finish_kernel, mx, dyn)) || (e = cudaFuncSetAttribute(accept_sample_kernel, mx, dyn)))
    return e;
  return cudaSuccess;
}

cudaError_t launch_prologue(const MiscParams& p, float* ssp, int* zero_ints, int n_zero, int M, cudaStream_t s,
                            bool pdl) {
  return launch_k(prologue_kernel, dim3(M + 1), dim3(256), 0, s, pdl, p, ssp, zero_ints, n_zero);
}
cudaError_t launch_finish(const MiscParams& p, int B, int M, bool sample, cudaStream_t s, bool pdl) {
  return launch_k(finish_kernel, dim3(sample ? M : B), dim3(1024), sample ? cdf_stage_bytes(p.vocab) : 0, s, pdl, p);
}

cudaError_t launch_controller(const MiscParams& p, cudaStream_t s, bool pdl) {
  return launch_k(controller_kernel, dim3(1), dim3(128), 0, s, pdl, p);
}
cudaError_t launch_embed(const MiscParams& p, int M, cudaStream_t s, bool pdl) {
  return launch_k(embed_kernel, dim3(M), dim3(256), 0, s, pdl, p);
}
cudaError_t launch_rmsnorm(const MiscParams& p, int slot, int which, int M, cudaStream_t s, bool pdl) {
  return launch_k(rmsnorm_kernel, dim3(M), dim3(256), 0, s, pdl, p, slot, which);
}
cudaError_t launch_accept_greedy(const MiscParams& p, int B, cudaStream_t s, bool pdl) {
  return launch_k(accept_greedy_kernel, dim3(B), dim3(256), 0, s, pdl, p);
}
cudaError_t launch_accept_sample(const MiscParams& p, int M, cudaStream_t s, bool pdl) {
  return launch_k(accept_sample_kernel, dim3(M), dim3(1024), cdf_stage_bytes(p.vocab), s, pdl, p);
}
cudaError_t launch_compact(const MiscParams& p, int B, int n_act, cudaStream_t s, bool pdl) {
  if (n_act <= 0) n_act = 1;
  return launch_k(compact_kernel, dim3(p.n_heads, B, n_act), dim3(128), 0, s, pdl, p);
}
// One thread per 16-byte chunk (8 columns) of the source.
__global__ void tile_weights_kernel(const __nv_bfloat16* src, __nv_bfloat16* dst, int rows, int cols) {
  const size_t n_chunks = static_cast<size_t>(rows) * (cols / 8);
  const int kbs = cols / 64;
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n_chunks;
       i += static_cast<size_t>(gridDim.x) * blockDim.x) {
    const int row = static_cast<int>(i / (cols / 8));
    const int col = static_cast<int>(i % (cols / 8)) * 8;
    const int t = row >> 7, r = row & 127, kb = col >> 6, c8 = (col & 63) >> 3;
    const size_t blk = static_cast<size_t>(t) * kbs + kb;
    uint8_t* d = reinterpret_cast<uint8_t*>(dst + blk * kTileElems) + r * 128 + ((c8 ^ (r & 7)) << 4);
    *reinterpret_cast<uint4*>(d) = *reinterpret_cast<const uint4*>(src + static_cast<size_t>(row) * cols + col);
  }
}

cudaError_t launch_tile_weights(const __nv_bfloat16* src, __nv_bfloat16* dst, int rows, int cols, cudaStream_t s) {
  const size_t n = static_cast<size_t>(rows) * (cols / 8);
  const int blocks = static_cast<int>(n / 256 + 1 < 16384 ? n / 256 + 1 : 16384);
  tile_weights_kernel<<<blocks, 256, 0, s>>>(src, dst, rows, cols);
  return cudaGetLastError();
}

cudaError_t launch_bf16_to_f32(const __nv_bfloat16* src, float* dst, size_t n, cudaStream_t s) {
  const int blocks = static_cast<int>((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096);
  bf16_to_f32_kernel<<<blocks > 0 ? blocks : 1, 256, 0, s>>>(src, dst, n);
  return cudaGetLastError();
}

}  // namespace tss
