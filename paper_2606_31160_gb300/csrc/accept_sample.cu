// K5: rejection-sampling acceptance (Leviathan et al. / Chen et al., cited
// in Sec. 1-2 of the paper, which evaluates the greedy rule only).
//
//   p_j = softmax(z_T[j] / T), q_j = softmax(z_D[j] / T)
//   draft j (token x) accepted iff u_j * q_j(x) <= p_j(x)
//   first rejection at j: draw from (p_j - q_j)+ with u_K
//   all K accepted:       draw the bonus from p_K with u_K
//   draw from w with u:   smallest v with sum_{v' <= v} w(v') > u * sum(w)
//
// Two launches, each a programmatic dependent one (resident before the kernel
// ahead has finished, which it waits for before it reads):
//   stats:  grid (chunk, row, scene) over the 2K + 1 rows; each CTA writes
//           (max, sum exp2((z - max) * log2e / T)) of one chunk of its row:
//           segments streamed through shared memory where rows are aligned,
//           else 4096 values held in registers. The CTA whose chunk holds a
//           draft token records its logit.
//   draw:   grid (chunk of 4096 values, scene). Every CTA of a scene first
//           merges the chunks of the scene's rows in a fixed order and runs the
//           K acceptance tests, which gives l and the normalisers of the row to
//           draw from; one of them writes n_emit and the accepted tokens. Then a
//           thread owns 16 consecutive values of that row's logits (16-byte
//           loads when the rows are aligned); each CTA writes the chunk sums of
//           the residual weights and of the target weights; the last CTA of a
//           scene (atomic ticket, no spin) finds the chunk where the running sum
//           passes u_K * S and re-scans the same per-thread runs inside it.
// The logits stream once; beside that it is latency. Acceptance in every CTA of
// the draw, rather than by the last CTA of the statistics, takes a fence, an
// atomic and two round trips off the path; with the launches overlapped, 8 scenes,
// K = 7, V = 151936: 28.7 -> 25.5 us, one scene 15.7 -> 12.2. Rows that are not
// aligned, 8 scenes, V = 50257: 29.6 -> 20.3 with the statistics'
// values in registers and the draw's rows read in order through shared memory.
// All reductions run in a fixed order (deterministic), the weight formula
// uses non-contractible intrinsics so both passes of the draw evaluate
// identical values, and every spin-free ticket is re-armed after use.
#include "common.cuh"

#include <mutex>

SD_DEFINE_ERROR_ACCESSOR(sd_take_error_sample)

namespace {

constexpr int kThreads = 256;
constexpr int kMaxChunks = 1024;
constexpr float kLog2e = 1.4426950408889634f;

struct DrawInfo {
  int ell;
  float mt, inv_zt;  // target row l (or K): max and 1 / sum
  float md, inv_zd;  // draft row l (when l < K)
};

// exp2((z - m) * c2) with a fixed rounding sequence
__device__ __forceinline__ float wexp(float z, float m, float c2) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__fmul_rn(__fsub_rn(z, m), c2)));
  return y;
}

// (max, sum) pair merge: sum rescaled to the larger max
__device__ __forceinline__ void merge_ms(float& m, float& s, float m2, float s2, float c2) {
  if (m2 == -INFINITY) return;
  if (m == -INFINITY) {
    m = m2;
    s = s2;
    return;
  }
  if (m2 > m) {
    s = __fadd_rn(__fmul_rn(s, wexp(m, m2, c2)), s2);
    m = m2;
  } else {
    s = __fadd_rn(s, __fmul_rn(s2, wexp(m2, m, c2)));
  }
}

__device__ __forceinline__ const float* row_ptr(const float* zt, const float* zd, int b, int rr,
                                                int K, int V) {
  if (rr <= K) return zt + (static_cast<long long>(b) * (K + 1) + rr) * V;
  return zd + (static_cast<long long>(b) * K + (rr - K - 1)) * V;
}

// ------------------------------------------------------------------ stats
constexpr int kScalarPer = 16;  // values per thread of the scalar kernel
constexpr int kScalarChunk = kThreads * kScalarPer;
constexpr int kMinSegment = 16384;  // values a CTA of the streaming kernel at least takes of a longer row

// Rows that are not aligned: values lo + t + kThreads k, k < 16, of a chunk, loaded once,
// all in flight, for the maximum and the sum.
__global__ void __launch_bounds__(kThreads)
    sample_stats_kernel(const float* zt, const float* zd, int K, int V,
                        float c2, int chunk, int n_chunks, const int32_t* draft,
                        float2* __restrict__ part, float* __restrict__ dlogit) {
  const int c = blockIdx.x, rr = blockIdx.y, b = blockIdx.z;
  sd_pdl_enter();
  const int rows = 2 * K + 1;
  const float* row = row_ptr(zt, zd, b, rr, K, V);
  const int lo = c * chunk, hi = min(V, lo + chunk);
  // the CTA whose chunk holds the draft token of its row records that logit
  if (threadIdx.x == 0 && rr != K) {
    const int j = rr < K ? rr : rr - K - 1;
    const int x = __ldcg(draft + static_cast<long long>(b) * K + j);
    if (x >= lo && x < hi) dlogit[static_cast<long long>(b) * rows + rr] = __ldcg(row + x);
  }
  float m = -INFINITY, s = 0.f;
  float x[kScalarPer];
#pragma unroll
  for (int k = 0; k < kScalarPer; ++k) {
    const int i = lo + threadIdx.x + kThreads * k;
    x[k] = i < hi ? __ldcg(row + i) : -INFINITY;
  }
#pragma unroll
  for (int k = 0; k < kScalarPer; ++k) m = fmaxf(m, x[k]);
  if (m != -INFINITY)
#pragma unroll
    for (int k = 0; k < kScalarPer; ++k) s = __fadd_rn(s, x[k] == -INFINITY ? 0.f : wexp(x[k], m, c2));
  // warp then block merge, fixed tree
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
    const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
    merge_ms(m, s, m2, s2, c2);
  }
  __shared__ float sm[kThreads / 32], ss[kThreads / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0) {
    sm[warp] = m;
    ss[warp] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float bm = sm[0], bs = ss[0];
    for (int w = 1; w < kThreads / 32; ++w) merge_ms(bm, bs, sm[w], ss[w], c2);
    part[(static_cast<long long>(b) * rows + rr) * n_chunks + c] = make_float2(bm, bs);
  }
}

// Streaming stats: one CTA per (segment, row, scene) moves its segment of the
// row through a ring of 16 KB shared-memory stages with bulk copies
// (warp 8 produces, warps 0-7 consume); a consumer thread keeps an online
// (max, sum) over its 16 values of every stage in a fixed order. Rows must
// start on 16-byte boundaries (V % 4 == 0, aligned bases).
constexpr int kStreamConsumers = 256;
constexpr int kStreamThreads = kStreamConsumers + 32;
constexpr int kStageFloats = 4096;
constexpr uint32_t kStreamSpin = 1u << 22;

__device__ __forceinline__ bool st_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait; false after the limit (the caller records a timeout)
__device__ __forceinline__ bool st_wait(uint32_t bar, uint32_t parity) {
#pragma unroll 1
  for (uint32_t i = 0; i < kStreamSpin; ++i)
    if (st_try_wait(bar, parity)) return true;
  return false;
}

template <int kStreamStages>
__global__ void __launch_bounds__(kStreamThreads)
    sample_stats_stream_kernel(const float* zt, const float* zd, int K, int V,
                               float c2, int seg, int n_seg, const int32_t* draft,
                               float2* __restrict__ part, float* __restrict__ dlogit) {
  extern __shared__ __align__(128) float stage_raw[];  // [kStreamStages][kStageFloats]
  float (*stage)[kStageFloats] = reinterpret_cast<float (*)[kStageFloats]>(stage_raw);
  __shared__ __align__(8) uint64_t full[kStreamStages], empty[kStreamStages];
  __shared__ int s_timeout;
  const int c = blockIdx.x, rr = blockIdx.y, b = blockIdx.z;
  const int rows = 2 * K + 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float* row = row_ptr(zt, zd, b, rr, K, V);
  const int lo = c * seg, hi = min(V, lo + seg);
  const int n_st = hi > lo ? (hi - lo + kStageFloats - 1) / kStageFloats : 0;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kStreamStages; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(&full[i]))));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(&empty[i]))),
                   "r"(kStreamConsumers / 32));
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    s_timeout = 0;
  }
  __syncthreads();
  sd_pdl_enter();  // the barriers are set up while the kernel before finishes
  float m = -INFINITY, s = 0.f;
  if (warp == kStreamConsumers / 32) {
    // ---- producer: thread 0 of warp 8; the first copies go out before it
    //      records the draft token's logit (a load it then waits for)
    if (lane == 0) {
      for (int t = 0; t < n_st; ++t) {
        const int st = t % kStreamStages;
        if (t >= kStreamStages &&
            !st_wait(static_cast<uint32_t>(__cvta_generic_to_shared(&empty[st])),
                     static_cast<uint32_t>(((t / kStreamStages) - 1) & 1))) {
          s_timeout = 1;
          break;
        }
        const int p0 = lo + t * kStageFloats;
        const uint32_t bytes = static_cast<uint32_t>(min(kStageFloats, hi - p0) * 4);
        const uint32_t fb = static_cast<uint32_t>(__cvta_generic_to_shared(&full[st]));
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(fb), "r"(bytes) : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         static_cast<uint32_t>(__cvta_generic_to_shared(&stage[st][0]))),
                     "l"(row + p0), "r"(bytes), "r"(fb)
                     : "memory");
      }
      if (rr != K) {
        const int j = rr < K ? rr : rr - K - 1;
        const int x = __ldcg(draft + static_cast<long long>(b) * K + j);
        if (x >= lo && x < hi) dlogit[static_cast<long long>(b) * rows + rr] = __ldcg(row + x);
      }
    }
  } else {
    // ---- consumers: thread t takes float4 t + 256 k (k < 4) of every stage
    for (int t = 0; t < n_st; ++t) {
      const int st = t % kStreamStages;
      if (!st_wait(static_cast<uint32_t>(__cvta_generic_to_shared(&full[st])),
                   static_cast<uint32_t>((t / kStreamStages) & 1))) {
        s_timeout = 1;
        break;
      }
      const int p0 = lo + t * kStageFloats;
      const int nv = min(kStageFloats, hi - p0) / 4;  // float4s in this stage
      float x[16];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int v = threadIdx.x + kStreamConsumers * k;
        const float4 f = v < nv ? reinterpret_cast<const float4*>(stage[st])[v]
                                : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
        x[4 * k + 0] = f.x;
        x[4 * k + 1] = f.y;
        x[4 * k + 2] = f.z;
        x[4 * k + 3] = f.w;
      }
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(static_cast<uint32_t>(__cvta_generic_to_shared(&empty[st])))
                     : "memory");
      float mx = x[0];
#pragma unroll
      for (int e = 1; e < 16; ++e) mx = fmaxf(mx, x[e]);
      if (mx != -INFINITY) {
        if (mx > m) {
          if (m != -INFINITY) s = __fmul_rn(s, wexp(m, mx, c2));
          m = mx;
        }
#pragma unroll
        for (int e = 0; e < 16; ++e) s = __fadd_rn(s, wexp(x[e], m, c2));
      }
    }
  }
  // warp then block merge (consumer warps), fixed tree
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o);
    const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
    merge_ms(m, s, m2, s2, c2);
  }
  __shared__ float sm[kStreamConsumers / 32], ss[kStreamConsumers / 32];
  if (lane == 0 && warp < kStreamConsumers / 32) {
    sm[warp] = m;
    ss[warp] = s;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (s_timeout) sd_set_error(SD_DEVERR_TIMEOUT);
    float bm = sm[0], bs = ss[0];
    for (int w = 1; w < kStreamConsumers / 32; ++w) merge_ms(bm, bs, sm[w], ss[w], c2);
    part[(static_cast<long long>(b) * rows + rr) * n_seg + c] = make_float2(bm, bs);
  }
}

// ------------------------------------------------------------------ draw
// Scene b's acceptance, by all kThreads threads of a CTA: merge the chunks of
// every row in a fixed order, run the K tests, return l and the normalisers of
// the row to draw from. The CTA that publishes also writes n_emit and the
// accepted tokens (all but token l, which the draw writes).
__device__ __forceinline__ DrawInfo accept_scene(int K, int V, float c2, int n_chunks, int b,
                                                 const int32_t* draft, const float* u,
                                                 const float2* part, const float* dlogit,
                                                 bool publish, int32_t* __restrict__ n_emit,
                                                 int32_t* __restrict__ tokens) {
  const int rows = 2 * K + 1;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ float row_m[2 * 128 + 1], row_s[2 * 128 + 1];
  // every load is issued before any result is used (one memory round trip):
  // the K drafts, their two logits, recorded by the CTAs holding them, the
  // scene's K acceptance uniforms, and the rows' chunk partials, two rows a
  // warp at a time
  __shared__ float s_zt[128], s_zd[128], s_u[128];
  __shared__ int s_x[128];
  __shared__ DrawInfo s_info;
  for (int j = threadIdx.x; j < K; j += kThreads) {
    const int x = __ldcg(draft + static_cast<long long>(b) * K + j);
    const bool ok = x >= 0 && x < V;  // out of range: no CTA has recorded a logit
    const float lt = __ldcg(dlogit + static_cast<long long>(b) * rows + j);
    const float ld = __ldcg(dlogit + static_cast<long long>(b) * rows + K + 1 + j);
    s_x[j] = x;
    s_zt[j] = ok ? lt : 0.f;
    s_zd[j] = ok ? ld : 0.f;
    s_u[j] = __ldcg(u + static_cast<long long>(b) * (K + 1) + j);
  }
  constexpr int nw = kThreads / 32;
  const int first = n_chunks > 16 ? 16 : (1 << (31 - __clz(2 * n_chunks - 1))) / 2;  // lanes past the chunks hold nothing
  for (int r0 = warp; r0 < rows; r0 += 2 * nw) {
    const int r1 = r0 + nw;
    float rm[2] = {-INFINITY, -INFINITY}, rs[2] = {0.f, 0.f};
    const float2* p0 = part + (static_cast<long long>(b) * rows + r0) * n_chunks;
    const float2* p1 = part + (static_cast<long long>(b) * rows + (r1 < rows ? r1 : r0)) * n_chunks;
    for (int k = lane; k < n_chunks; k += 32) {
      const float2 e0 = __ldcg(p0 + k);
      const float2 e1 = __ldcg(p1 + k);
      merge_ms(rm[0], rs[0], e0.x, e0.y, c2);
      merge_ms(rm[1], rs[1], e1.x, e1.y, c2);
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      for (int o = first; o > 0; o >>= 1) {
        const float m2 = __shfl_xor_sync(0xffffffffu, rm[h], o);
        const float s2 = __shfl_xor_sync(0xffffffffu, rs[h], o);
        merge_ms(rm[h], rs[h], m2, s2, c2);
      }
    }
    if (lane == 0) {
      row_m[r0] = rm[0];
      row_s[r0] = rs[0];
      if (r1 < rows) {
        row_m[r1] = rm[1];
        row_s[r1] = rs[1];
      }
    }
  }
  __syncthreads();
  if (warp == 0) {
    // the K acceptance tests side by side (lane j of a 32-draft group), the
    // first stop by ballot: l = the first j whose token is out of range or
    // whose test fails, as a sequential scan would find it
    int ell = K;
    bool range_bad = false;
    for (int j0 = 0; j0 < K; j0 += 32) {  // warp-uniform
      const int j = j0 + lane;
      bool stop = false, bad = false;
      if (j < K) {
        const int x = s_x[j];
        bad = x < 0 || x >= V;
        if (bad) {
          stop = true;
        } else {
          const float p = __fdiv_rn(wexp(s_zt[j], row_m[j], c2), row_s[j]);
          const float q = __fdiv_rn(wexp(s_zd[j], row_m[K + 1 + j], c2), row_s[K + 1 + j]);
          stop = !(__fmul_rn(s_u[j], q) <= p);
        }
      }
      const unsigned hit = __ballot_sync(0xffffffffu, stop);
      if (hit) {
        const int first = __ffs(hit) - 1;
        ell = j0 + first;
        range_bad = __shfl_sync(0xffffffffu, bad, first);
        break;
      }
    }
    if (lane == 0) {
      DrawInfo di;
      di.ell = ell;
      di.mt = row_m[ell];
      di.inv_zt = __fdiv_rn(1.f, row_s[ell]);
      di.md = ell < K ? row_m[K + 1 + ell] : 0.f;
      di.inv_zd = ell < K ? __fdiv_rn(1.f, row_s[K + 1 + ell]) : 0.f;
      s_info = di;
      if (publish) {
        if (range_bad) sd_set_error(SD_DEVERR_TOKEN_RANGE);
        n_emit[b] = ell + 1;
      }
    }
    if (publish) {
      int32_t* tk = tokens + static_cast<long long>(b) * (K + 1);
      for (int j = lane; j <= K; j += 32)
        if (j != ell) tk[j] = j < ell ? s_x[j] : -1;
    }
  }
  __syncthreads();
  return s_info;
}

// Weights of one element of the draw row from its two logits: residual
// (p - q)+ (l < K) and the unnormalised target weight exp2((z_T - m_T) * c2).
__device__ __forceinline__ void weights(float zt_v, float zd_v, const DrawInfo& di, int K, float c2, float& w_res,
                                        float& w_tgt) {
  const float et = wexp(zt_v, di.mt, c2);
  w_tgt = et;
  if (di.ell < K) {
    const float p = __fmul_rn(et, di.inv_zt);
    const float q = __fmul_rn(wexp(zd_v, di.md, c2), di.inv_zd);
    w_res = fmaxf(__fsub_rn(p, q), 0.f);
  } else {
    w_res = 0.f;
  }
}

constexpr int kDrawPer = 16;                     // consecutive values a thread owns
constexpr int kDrawChunk = kThreads * kDrawPer;  // values a CTA owns

// Unaligned rows: both rows' chunk in shared memory, one word of padding every
// kDrawPer, so that a thread's consecutive values lie in distinct banks.
constexpr int kDrawStage = kDrawChunk + kDrawChunk / kDrawPer;
constexpr int kDrawSmem = 2 * kDrawStage * 4;

// This thread's kDrawPer logits of both rows (missing values: -inf, weight 0) of
// the chunk that begins at c0. Aligned rows: 16-byte loads, through L1 (a load of a warp
// takes half of 32 sectors; past L1 each came twice: 16 scenes 39.3 -> 44.5 us). Others: a warp would
// touch 32 lines a load, so the block reads the chunk in order through `stage`.
__device__ __forceinline__ void draw_load(const float* rt, const float* rd, int c0, int V, bool vec, float* stage,
                                          float (&xt)[kDrawPer], float (&xd)[kDrawPer]) {
  const int v0 = c0 + threadIdx.x * kDrawPer;
  if (vec && v0 + kDrawPer <= V) {
#pragma unroll
    for (int q = 0; q < kDrawPer / 4; ++q) {
      const float4 a = sd_ld4(rt + v0 + 4 * q);
      xt[4 * q] = a.x, xt[4 * q + 1] = a.y, xt[4 * q + 2] = a.z, xt[4 * q + 3] = a.w;
      const float4 d = rd ? sd_ld4(rd + v0 + 4 * q) : make_float4(0.f, 0.f, 0.f, 0.f);
      xd[4 * q] = d.x, xd[4 * q + 1] = d.y, xd[4 * q + 2] = d.z, xd[4 * q + 3] = d.w;
    }
  } else if (vec) {
#pragma unroll
    for (int e = 0; e < kDrawPer; ++e) {
      const bool in = v0 + e < V;
      xt[e] = in ? __ldcg(rt + v0 + e) : -INFINITY;
      xd[e] = (in && rd) ? __ldcg(rd + v0 + e) : 0.f;
    }
  } else {
#pragma unroll
    for (int k = 0; k < kDrawPer; ++k) {
      const int i = threadIdx.x + kThreads * k;
      const bool in = c0 + i < V;
      xt[k] = in ? __ldcg(rt + c0 + i) : -INFINITY;
      xd[k] = (in && rd) ? __ldcg(rd + c0 + i) : 0.f;
    }
#pragma unroll
    for (int k = 0; k < kDrawPer; ++k) {
      const int i = threadIdx.x + kThreads * k;
      stage[i + i / kDrawPer] = xt[k];
      stage[kDrawStage + i + i / kDrawPer] = xd[k];
    }
    __syncthreads();
#pragma unroll
    for (int e = 0; e < kDrawPer; ++e) {
      xt[e] = stage[threadIdx.x * (kDrawPer + 1) + e];
      xd[e] = stage[kDrawStage + threadIdx.x * (kDrawPer + 1) + e];
    }
  }
}

// The block's sums of x and y, valid in thread 0 (fixed order).
__device__ __forceinline__ float2 block_sum2(float x, float y) {
  __shared__ float2 red[kThreads / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    x = __fadd_rn(x, __shfl_xor_sync(0xffffffffu, x, o));
    y = __fadd_rn(y, __shfl_xor_sync(0xffffffffu, y, o));
  }
  if (lane == 0) red[warp] = make_float2(x, y);
  __syncthreads();
  float2 t = make_float2(0.f, 0.f);
  if (threadIdx.x == 0)
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) t.x = __fadd_rn(t.x, red[w].x), t.y = __fadd_rn(t.y, red[w].y);
  return t;
}

// grid (chunk, scene): chunk c of the draw row holds values [c * kDrawChunk,
// (c + 1) * kDrawChunk), thread t the kDrawPer consecutive values from
// c * kDrawChunk + t * kDrawPer, summed in order.
__global__ void __launch_bounds__(kThreads)
    sample_draw_kernel(const float* zt, const float* zd, int K, int V,
                       float c2, int n_chunks, bool vec, int n_parts, const int32_t* draft,
                       const float* u, int32_t* __restrict__ n_emit, int32_t* __restrict__ tokens,
                       const float2* part, const float* dlogit,
                       float2* __restrict__ sums, uint32_t* __restrict__ ticket) {
  const int c = blockIdx.x, b = blockIdx.y;
  // a programmatic dependent launch: resident while the statistics finish,
  // reading nothing they write before they have completed
  sd_pdl_enter();
  const DrawInfo di = accept_scene(K, V, c2, n_parts, b, draft, u, part, dlogit, c == 0, n_emit, tokens);
  const float* rt = zt + (static_cast<long long>(b) * (K + 1) + di.ell) * V;
  const float* rd = di.ell < K ? zd + (static_cast<long long>(b) * K + di.ell) * V : nullptr;
  float xt[kDrawPer], xd[kDrawPer];
  extern __shared__ __align__(16) float draw_stage[];  // kDrawSmem bytes for unaligned rows
  draw_load(rt, rd, c * kDrawChunk, V, vec, draw_stage, xt, xd);
  float sr = 0.f, sp = 0.f;
#pragma unroll
  for (int e = 0; e < kDrawPer; ++e) {
    float wr, wt;
    weights(xt[e], xd[e], di, K, c2, wr, wt);
    sr = __fadd_rn(sr, wr);
    sp = __fadd_rn(sp, wt);
  }
  const float2 tot = block_sum2(sr, sp);
  __shared__ bool s_last;
  if (threadIdx.x == 0) {
    sums[static_cast<long long>(b) * n_chunks + c] = tot;
    __threadfence();
    s_last = atomicAdd(&ticket[b], 1u) == static_cast<uint32_t>(n_chunks - 1);
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  // ---- last CTA of scene b: choose the weights, locate the chunk, scan it
  __shared__ float s_sr[kMaxChunks], s_sp[kMaxChunks];
  for (int k = threadIdx.x; k < n_chunks; k += kThreads) {
    const float2 e = __ldcg(sums + static_cast<long long>(b) * n_chunks + k);
    s_sr[k] = e.x;
    s_sp[k] = e.y;
  }
  __syncthreads();
  __shared__ int s_chunk, s_use_res;
  __shared__ float s_base, s_target;
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    // lane l owns chunks [l*per, (l+1)*per): sequential lane sums, warp scan
    const int per = (n_chunks + 31) / 32;
    const int k0 = min(n_chunks, lane * per), k1 = min(n_chunks, k0 + per);
    float lr = 0.f, lp = 0.f;
    for (int k = k0; k < k1; ++k) {
      lr = __fadd_rn(lr, s_sr[k]);
      lp = __fadd_rn(lp, s_sp[k]);
    }
    float ir = lr, ip = lp;  // inclusive warp scan
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float xr = __shfl_up_sync(0xffffffffu, ir, o);
      const float xp = __shfl_up_sync(0xffffffffu, ip, o);
      if (lane >= o) {
        ir = __fadd_rn(xr, ir);
        ip = __fadd_rn(xp, ip);
      }
    }
    const float tot_r = __shfl_sync(0xffffffffu, ir, 31);
    const float tot_p = __shfl_sync(0xffffffffu, ip, 31);
    const int use_res = (di.ell < K && tot_r > 0.f) ? 1 : 0;
    const float total = use_res ? tot_r : tot_p;
    const float target = __fmul_rn(__ldcg(u + static_cast<long long>(b) * (K + 1) + K), total);
    const float incl = use_res ? ir : ip;
    float run = __shfl_up_sync(0xffffffffu, incl, 1);
    if (lane == 0) run = 0.f;
    int found = -1, last_nz = -1;
    float base = 0.f;
    for (int k = k0; k < k1; ++k) {
      const float w = use_res ? s_sr[k] : s_sp[k];
      if (w > 0.f) last_nz = k;
      const float nxt = __fadd_rn(run, w);
      if (found < 0 && nxt > target) {
        found = k;
        base = run;
      }
      run = nxt;
    }
    const unsigned hit = __ballot_sync(0xffffffffu, found >= 0);
    int lnz = last_nz;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) lnz = max(lnz, __shfl_xor_sync(0xffffffffu, lnz, o));
    if (hit) {
      const int src = __ffs(hit) - 1;
      found = __shfl_sync(0xffffffffu, found, src);
      base = __shfl_sync(0xffffffffu, base, src);
    } else {
      // u * S at or above the rounded total: the draw is the last positive
      // weight, found by the in-chunk fallback below
      found = lnz >= 0 ? lnz : 0;
      base = -INFINITY;
    }
    if (lane == 0) {
      s_chunk = found;
      s_base = base;
      s_target = target;
      s_use_res = use_res;
    }
  }
  __syncthreads();
  // in-chunk scan: thread t owns the same kDrawPer consecutive values as in
  // the chunk sums above
  const int my_lo = s_chunk * kDrawChunk + threadIdx.x * kDrawPer;
  const bool use_res = s_use_res != 0;
  draw_load(rt, rd, s_chunk * kDrawChunk, V, vec, draw_stage, xt, xd);
  float w[kDrawPer];
  float tsum = 0.f;
#pragma unroll
  for (int e = 0; e < kDrawPer; ++e) {
    float wr, wt;
    weights(xt[e], xd[e], di, K, c2, wr, wt);
    w[e] = use_res ? wr : wt;
    tsum = __fadd_rn(tsum, w[e]);
  }
  // exclusive prefix of the thread sums: warp scan + warp offsets (fixed)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float incl = tsum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float x = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl = __fadd_rn(x, incl);
  }
  float excl = __shfl_up_sync(0xffffffffu, incl, 1);
  if (lane == 0) excl = 0.f;
  __shared__ float s_wtot[kThreads / 32];
  if (lane == 31) s_wtot[warp] = incl;
  __syncthreads();
  float woff = 0.f;
  for (int q = 0; q < warp; ++q) woff = __fadd_rn(woff, s_wtot[q]);
  float run = __fadd_rn(s_base, __fadd_rn(woff, excl));
  int cand = 0x7fffffff, last_pos = -1;
#pragma unroll
  for (int e = 0; e < kDrawPer; ++e) {
    const int v = my_lo + e;
    if (w[e] > 0.f) last_pos = v;
    run = __fadd_rn(run, w[e]);
    if (cand == 0x7fffffff && run > s_target) cand = v;
  }
  // block min of candidates, block max of the last positive weight
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    cand = min(cand, __shfl_xor_sync(0xffffffffu, cand, o));
    last_pos = max(last_pos, __shfl_xor_sync(0xffffffffu, last_pos, o));
  }
  __shared__ int s_cand[kThreads / 32], s_lastp[kThreads / 32];
  if (lane == 0) {
    s_cand[warp] = cand;
    s_lastp[warp] = last_pos;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int best = 0x7fffffff, lp = -1;
    for (int q = 0; q < kThreads / 32; ++q) {
      best = min(best, s_cand[q]);
      lp = max(lp, s_lastp[q]);
    }
    const int tok = best != 0x7fffffff ? best : (lp >= 0 ? lp : s_chunk * kDrawChunk);
    tokens[static_cast<long long>(b) * (K + 1) + di.ell] = tok;
    ticket[b] = 0;
  }
}

struct Plan {
  int n1, n2;  // chunks a row of the scalar stats kernel, and of the draw
  bool vec;
};

// Streaming stats when every row starts on a 16-byte boundary (V a multiple of 4 and
// 16-byte-aligned bases, checked at the call).
Plan plan(int V) {
  Plan p;
  p.vec = V % 4 == 0;
  // (the doubling is for the workspace size alone: a call with over kMaxChunks
  // chunks of 4096 is refused)
  int chunk = kScalarChunk;
  while ((V + chunk - 1) / chunk > kMaxChunks) chunk *= 2;
  p.n1 = (V + chunk - 1) / chunk;
  p.n2 = (V + kDrawChunk - 1) / kDrawChunk;
  return p;
}

struct Layout {
  size_t part, dlogit, sums, ticket, total;
};

Layout layout(int B, int K, const Plan& p) {
  Layout l;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off += (bytes + 255) / 256 * 256;
    return at;
  };
  // room for the scalar chunking's partials (rows found unaligned at the call)
  l.part = take(static_cast<size_t>(B) * (2 * K + 1) * p.n1 * sizeof(float2));
  l.dlogit = take(static_cast<size_t>(B) * (2 * K + 1) * sizeof(float));
  // unused: the size that callers have planned with counts 4 and 32 bytes a scene here
  take(static_cast<size_t>(B) * 4);
  take(static_cast<size_t>(B) * 32);
  l.sums = take(static_cast<size_t>(B) * p.n2 * sizeof(float2));
  l.ticket = take(static_cast<size_t>(B) * 4);
  l.total = off;
  return l;
}

constexpr int stream_smem(int stages) { return stages * kStageFloats * 4; }

// Stages of the ring. Four leave room for three CTAs an SM, three for four; the
// latter where four stages would leave a few CTAs for a second wave: 480 CTAs (16
// scenes, K = 7) 44.3 -> 39.5 us, 32 scenes 77 -> 66. With fewer CTAs the deeper ring
// is the faster one at 336 (25.2 us against 26.8) and 396 CTAs (25.0, 25.5) but not at
// the 360 of 8 scenes, K = 7, V = 151936 (25.8, 23.7): the line is where the waves
// change, and that size lies on the slower side of it.
bool deep_ring(long long ctas, int n_sm) { return ctas <= 3LL * n_sm; }

// SMs of the current device, once the streaming kernel's shared-memory
// attribute is set there; 0 when either call fails (the kernel for unaligned rows runs).
int stream_sms() {
  static int cache[64];
  static bool done[64];
  static std::mutex mu;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    (void)cudaGetLastError();
    return 0;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (!done[dev]) {
    done[dev] = true;
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaFuncSetAttribute(sample_stats_stream_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             stream_smem(4)) != cudaSuccess ||
        cudaFuncSetAttribute(sample_stats_stream_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             stream_smem(3)) != cudaSuccess) {
      (void)cudaGetLastError();
      n = 0;
    }
    cache[dev] = n;
  }
  return cache[dev];
}

}  // namespace

extern "C" size_t sd_accept_sample_workspace(int B, int K, int V) {
  if (B <= 0 || K < 0 || V <= 0) return 0;
  return layout(B, K, plan(V)).total;
}

extern "C" sd_status sd_accept_sample(const float* z_target, const float* z_draft, int B, int K,
                                      int V, float temperature, const int32_t* draft,
                                      const float* u, int32_t* n_emit, int32_t* tokens, void* ws,
                                      size_t ws_bytes, sd_stream_t stream) {
  if (B < 0 || K < 0 || V <= 0) return SD_ERR_INVALID_ARG;
  if (!(temperature > 0.f) || !isfinite(temperature)) return SD_ERR_INVALID_ARG;
  if (K > 128 || B > 65535 || (V + kDrawChunk - 1) / kDrawChunk > kMaxChunks) return SD_ERR_UNSUPPORTED;
  if (B == 0) return SD_OK;
  if (!z_target || !u || !n_emit || !tokens || (K > 0 && (!z_draft || !draft)))
    return SD_ERR_INVALID_ARG;
  Plan p = plan(V);
  const Layout l = layout(B, K, p);
  // aligned rows need aligned bases too (same workspace either way)
  if ((reinterpret_cast<uintptr_t>(z_target) & 15) || (K > 0 && (reinterpret_cast<uintptr_t>(z_draft) & 15))) p.vec = false;
  if (!ws || ws_bytes < l.total || !sd_aligned16(ws)) return SD_ERR_WORKSPACE;
  char* w = static_cast<char*>(ws);
  auto* part = reinterpret_cast<float2*>(w + l.part);
  auto* dlogit = reinterpret_cast<float*>(w + l.dlogit);
  auto* sums = reinterpret_cast<float2*>(w + l.sums);
  auto* ticket = reinterpret_cast<uint32_t*>(w + l.ticket);
  const float c2 = static_cast<float>(kLog2e / static_cast<double>(temperature));
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int n_sm = stream_sms();
  int parts = p.n1;  // partials a row
  cudaError_t e;
  if (p.vec && n_sm > 0) {
    // segments of whole stages, about two CTAs per SM over all (row, scene) pairs
    const long long rows_all = static_cast<long long>(2 * K + 1) * B;
    long long n_seg = (2LL * n_sm + rows_all - 1) / rows_all;
    const long long most = (V + kMinSegment - 1) / kMinSegment;
    n_seg = n_seg < 1 ? 1 : (n_seg > most ? most : n_seg);
    const int seg = static_cast<int>(((V + n_seg - 1) / n_seg + kStageFloats - 1) / kStageFloats * kStageFloats);
    const int ns = (V + seg - 1) / seg;
    const bool deep = deep_ring(rows_all * ns, n_sm);
    e = sd_launch_pdl(deep ? sample_stats_stream_kernel<4> : sample_stats_stream_kernel<3>, dim3(ns, 2 * K + 1, B),
                      dim3(kStreamThreads), stream_smem(deep ? 4 : 3), st, z_target, z_draft, K, V, c2, seg, ns, draft, part,
                      dlogit);
    parts = ns;
  } else {
    e = sd_launch_pdl(sample_stats_kernel, dim3(p.n1, 2 * K + 1, B), dim3(kThreads), 0, st, z_target, z_draft, K, V, c2,
                      kScalarChunk, p.n1, draft, part, dlogit);
  }
  if (e == cudaSuccess)
    e = sd_launch_pdl(sample_draw_kernel, dim3(p.n2, B), dim3(kThreads), p.vec ? 0 : kDrawSmem, st, z_target, z_draft, K, V, c2, p.n2, p.vec,
                      parts, draft, u, n_emit, tokens, static_cast<const float2*>(part), static_cast<const float*>(dlogit),
                      sums, ticket);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return SD_ERR_CUDA;
  }
  return SD_OK;
}
