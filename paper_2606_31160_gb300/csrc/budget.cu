// Attention budget of the verify rows (Sec. 4.2 "Empirical confirmation",
// Table tab:attn-budget): for every (scene, row, query head), the share of
// the row's softmax mass on the visual keys, on the trajectory / prompt-text
// keys and on the rows generated in this step, and the entropy of the
// attention among the non-visual keys (renormalised), divided by the log of
// their number.
//
// A diagnostic beside the verify path. One thread-block cluster per (KV head,
// scene) splits the visible keys over its S CTAs; the G * R query rows of the
// KV head (packed row p = i * G + j: new row i, query head j of the group)
// take their scores from bf16 tensor-core products (mma.sync m16n8k16, fp32
// accumulation), 16 rows by 8 keys a product, both operands staged in shared
// memory. Every thread folds the scores it holds of a chunk of keys into four
// sums per row, relative to their maximum m:
//   v, t, g = sum of 2^(y - m) over the visual, trajectory / prompt-text and
//             generated keys, n = sum over the non-visual keys of
//             2^(y - m) (y - m),         y = q . k * scale * log2(e),
// which merge in a fixed order over the lanes and warps, then over the
// cluster's CTAs through distributed shared memory (each CTA finishes 32 / S
// of the rows), and
//
//   entropy = (ln l' - n ln 2 / l') / ln N'     l' = t + g, N' = number of
//                                          non-visual keys the row sees
#include "common.cuh"

#include <cuda.h>  // CUtensorMap and its enums (header only; no libcuda link)

#include <math.h>
#include <mutex>

SD_DEFINE_ERROR_ACCESSOR(sd_take_error_budget)

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr float kLn2 = 0.6931471805599453f;

__device__ __forceinline__ float ex2f(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Sums of one row (see the header), relative to a maximum kept beside them.
struct RowSums {
  float v, t, g, n;
};

// The row's sums moved from the maximum m to M >= m (no key seen: m = -inf, all zero).
__device__ __forceinline__ void row_rescale(RowSums& s, float m, float M) {
  if (m == -INFINITY || m == M) return;
  const float f = ex2f(m - M);
  s.n = f * fmaf(m - M, s.t + s.g, s.n);
  s.v *= f;
  s.t *= f;
  s.g *= f;
}

// One step of the sum over an aligned group of lanes (a fixed butterfly).
__device__ __forceinline__ void row_add(RowSums& s, int o) {
  s.v += __shfl_xor_sync(0xffffffffu, s.v, o);
  s.t += __shfl_xor_sync(0xffffffffu, s.t, o);
  s.g += __shfl_xor_sync(0xffffffffu, s.g, o);
  s.n += __shfl_xor_sync(0xffffffffu, s.n, o);
}

// Merge over aligned groups of `lanes` lanes: the common maximum first, one
// rescale a lane, then plain sums.
__device__ __forceinline__ void row_merge(RowSums& s, float& m, int lanes) {
  float M = m;
  for (int o = 1; o < lanes; o <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  row_rescale(s, m, M);
  for (int o = 1; o < lanes; o <<= 1) row_add(s, o);
  m = M;
}

__device__ __forceinline__ uint32_t cta_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// grid (S, Hkv, B), clusters of S CTAs along x: CTA `rank` of the cluster of
// (KV head kvh, scene b) takes keys [rank * n / S, (rank + 1) * n / S) of the
// n = len[b] keys the scene holds, for the M = G * R packed rows in passes of
// kTiles tiles of 16 rows (lane l of a warp holds rows l / 4 and l / 4 + 8 of
// a tile, keys 2 (l % 4) and 2 (l % 4) + 1 of every 8-key block).
//
// One launch is a chain of latencies, not of bytes, so each link is cut short:
// the query rows travel while the length and then the keys do; a warp holds the
// scores of all its blocks of a chunk (kBlocks x 2 tiles of accumulators, ten
// independent product chains), takes their maximum once and folds them without a
// running one; the sums merge over lanes, warps and CTAs by a common maximum, one
// rescale and plain additions; and every CTA finishes 32 / S rows of the cluster.
// One scene, 32 rows on each of 8 KV heads, 4096 keys: 7.9 us (14.9 with a running
// maximum per thread, query fragments read from global memory before the keys, and one
// CTA merging the cluster); of it the length takes 1.0 us, the keys 2.5, the products
// 1.4, the fold 1.0, the merges and the exchange 2.2. Eight scenes 44.0 us (64.7).
constexpr int kTiles = 2;
constexpr int kPassRows = 16 * kTiles;
constexpr int kChunkKeys = 320;  // keys a CTA stages at once (10 boxes of 32)
constexpr int kBlocks = kChunkKeys / (8 * kWarps);  // 8-key blocks a warp takes of a chunk

// two CTAs an SM (at most 128 registers a thread), so that clusters of 16
// need only 8 SMs of a GPC and every cluster of a launch fits in one wave
template <int D>
__global__ void __launch_bounds__(kThreads, 2)
    budget_kernel(const __grid_constant__ CUtensorMap tm_k, const __nv_bfloat16* q,
                  const int32_t* len, const int32_t* n_visual, int R, int Hq,
                  int Hkv, int cap, float scale_log2, bool q_vec, float* __restrict__ mass, float* __restrict__ entropy) {
  static_assert(kPassRows == 32 && kPassRows * kWarps == kThreads, "one thread a (row, warp) in the merge");
  constexpr int kRowChunks = D / 8;  // 16-byte chunks of a query row
  __shared__ __align__(16) uint4 qs[kPassRows * kRowChunks];  // the pass's query rows, chunks swizzled by row
  __shared__ __align__(16) float4 red_s[kWarps][kPassRows];
  __shared__ float red_m[kWarps][kPassRows];
  // (max, v, t, g, n) of this CTA's rows from every CTA, by the parity of the pass
  __shared__ __align__(16) float recv[2][5][32];
  const int kvh = blockIdx.y, b = blockIdx.z;
  const int S = gridDim.x;  // up to 16
  const uint32_t rank = cta_rank();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gq = lane >> 2, tq = lane & 3;
  const int G = Hq / Hkv, M = G * R;
  // the CTA's keys are staged in shared memory a chunk of up to kChunkKeys at
  // a time (one TMA round trip a chunk): 32-key boxes of 64 columns with the
  // 128-byte swizzle, one region per 64-column half
  extern __shared__ uint8_t smem_raw[];
  const uint32_t kbuf = (static_cast<uint32_t>(__cvta_generic_to_shared(smem_raw)) + 1023u) & ~1023u;
  const uint32_t qbuf = static_cast<uint32_t>(__cvta_generic_to_shared(qs));
  __shared__ __align__(8) uint64_t chunk_bar;
  const uint32_t bar = static_cast<uint32_t>(__cvta_generic_to_shared(&chunk_bar));
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_k)) : "memory");
  }
  __syncthreads();
  cluster_arrive();  // waited for before the first store into another CTA
  // a programmatic dependent launch: resident while the kernel before it
  // runs, reading nothing before it has completed
  sd_pdl_enter();
  // the query rows m0 .. m0 + 31 (zero past M) into shared memory, by every warp but the first
  auto load_q = [&](int m0) {
    for (int e = threadIdx.x - 32; e < kPassRows * kRowChunks; e += kThreads - 32) {
      const int row = e / kRowChunks, chunk = e % kRowChunks, p = m0 + row, i = p / G;
      uint4 x = make_uint4(0u, 0u, 0u, 0u);
      if (p < M) {
        const __nv_bfloat16* src = q + ((static_cast<long long>(b) * R + i) * Hq + kvh * G + (p - i * G)) * D + chunk * 8;
        if (q_vec) {
          x = __ldcg(reinterpret_cast<const uint4*>(src));
        } else {
          const uint32_t* s4 = reinterpret_cast<const uint32_t*>(src);
          x = make_uint4(__ldcg(s4), __ldcg(s4 + 1), __ldcg(s4 + 2), __ldcg(s4 + 3));
        }
      }
      qs[row * kRowChunks + (chunk ^ (row & 7))] = x;
    }
  };
  const int n_keys = __ldcg(len + b), L = n_keys - R;
  int nv = __ldcg(n_visual + b);
  // every CTA of a cluster runs the same barriers, so a bad length only
  // empties the key ranges (and writes nothing)
  const bool ok = L >= 0 && n_keys <= cap;
  const int log_s = 31 - __clz(S);  // a power of two
  const int k_lo = ok ? static_cast<int>((static_cast<long long>(rank) * n_keys) >> log_s) : 0;
  const int k_hi = ok ? static_cast<int>((static_cast<long long>(rank + 1) * n_keys) >> log_s) : 0;
  const int n_chunks = (k_hi - k_lo + kChunkKeys - 1) / kChunkKeys;
  // the first warp: lane i copies box i % nbox of half i / nbox of chunk ci
  auto load_chunk = [&](int ci) {
    const int c0 = k_lo + ci * kChunkKeys, nbox = (min(kChunkKeys, k_hi - c0) + 31) / 32;
    if (lane == 0)
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
                   "r"(static_cast<uint32_t>(nbox * 32 * 128 * (D / 64)))
                   : "memory");
    __syncwarp();
    if (lane < nbox * (D / 64)) {
      const int hf = lane / nbox, bx = lane - hf * nbox;
      asm volatile(
          "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
          " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(kbuf + hf * kChunkKeys * 128 + bx * 32 * 128),
          "l"(reinterpret_cast<uint64_t>(&tm_k)), "r"(bar), "r"(hf * 64), "r"(c0 + bx * 32),
          "r"(b * Hkv + kvh)
          : "memory");
    }
  };
  if (warp == 0) {
    if (n_chunks > 0) load_chunk(0);
  } else {
    load_q(0);
  }
  if (!ok && threadIdx.x == 0 && kvh == 0 && rank == 0) sd_set_error(SD_DEVERR_LENGTH);
  if (ok && (nv < 0 || nv > L)) {
    if (threadIdx.x == 0 && kvh == 0 && rank == 0) sd_set_error(SD_DEVERR_LENGTH);
    nv = nv < 0 ? 0 : L;
  }
  int issued = 0, ready = -1;  // the chunk whose copies were issued last, and the one waited for
  uint32_t phase = 0;
  for (int m0 = 0; m0 < M; m0 += kPassRows) {
    const int par = (m0 / kPassRows) & 1;
    if (m0 > 0 && warp > 0) load_q(m0);  // the last pass's were read before its barriers
    // the keys each row sees (causal over the new rows); sums and maximum per row
    int lim[kTiles][2];
    RowSums st[kTiles][2];
    float mx[kTiles][2];
#pragma unroll
    for (int u = 0; u < kTiles; ++u)
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2) {
        const int p = m0 + 16 * u + gq + 8 * h2;
        lim[u][h2] = p < M ? L + p / G : -1;
        st[u][h2] = RowSums{0.f, 0.f, 0.f, 0.f};
        mx[u][h2] = -INFINITY;
      }
    __syncthreads();  // the query rows are in place
#pragma unroll 1
    for (int ci = 0; ci < n_chunks; ++ci) {  // block-uniform
      const int c0 = k_lo + ci * kChunkKeys, nk = min(kChunkKeys, k_hi - c0);
      if (issued != ci) {
        __syncthreads();  // every warp is done with the chunk in place
        if (warp == 0) load_chunk(ci);
        issued = ci;
        ready = -1;
      }
      if (ready != ci) {
        // bounded wait on the chunk's copies
        uint32_t done = 0;
        for (uint32_t it = 0; it < (1u << 22) && !done; ++it)
          asm volatile(
              "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
              "selp.u32 %0, 1, 0, p;\n\t}"
              : "=r"(done)
              : "r"(bar), "r"(phase)
              : "memory");
        if (!done && threadIdx.x == 0) sd_set_error(SD_DEVERR_TIMEOUT);
        phase ^= 1u;
        ready = ci;
      }
      // block j of the warp: keys c0 + 8 (warp + kWarps j) + 0 .. 7
      const int n_blk = (nk + 7) / 8;
      float c[kTiles][kBlocks][4];
#pragma unroll
      for (int u = 0; u < kTiles; ++u)
#pragma unroll
        for (int j = 0; j < kBlocks; ++j)
#pragma unroll
          for (int e = 0; e < 4; ++e) c[u][j][e] = 0.f;
#pragma unroll
      for (int ks = 0; ks < D / 16; ks += 2) {
        uint32_t af[kTiles][2][4];
#pragma unroll
        for (int u = 0; u < kTiles; ++u)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int row = 16 * u + (lane & 15), chunk = 2 * (ks + h) + (lane >> 4);
            ldmatrix4(af[u][h], qbuf + (row * kRowChunks + (chunk ^ (row & 7))) * 16);
          }
        // the 8 keys x 8 d matrices of a block, two k16 steps a load
        const int kc = 2 * ks + (lane >> 3);
        const uint32_t kcol = kbuf + (kc >> 3) * kChunkKeys * 128 + (((kc & 7) ^ (lane & 7)) << 4);
#pragma unroll
        for (int j = 0; j < kBlocks; ++j) {
          if (warp + kWarps * j >= n_blk) break;  // warp-uniform
          uint32_t bf[4];
          ldmatrix4(bf, kcol + (8 * (warp + kWarps * j) + (lane & 7)) * 128);
#pragma unroll
          for (int u = 0; u < kTiles; ++u) {
            mma_bf16(c[u][j], af[u][0], bf[0], bf[1]);
            mma_bf16(c[u][j], af[u][1], bf[2], bf[3]);
          }
        }
      }
      // products, -inf where masked, and their maximum per row over the quad of lanes
      // that holds the row (a score is the product in log2 units: one fma with the
      // maximum, which rounds once). A block's 8 keys are mostly of one
      // segment and all visible (the packed rows past M, never written, need no
      // mask): what it costs is instructions, so such blocks skip the tests.
      const int kb0 = c0 + 8 * warp, full = min(k_hi, L);
      float bm[kTiles][2];
#pragma unroll
      for (int u = 0; u < kTiles; ++u)
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) bm[u][h2] = -INFINITY;
#pragma unroll
      for (int j = 0; j < kBlocks; ++j) {
        const int kb = kb0 + 8 * kWarps * j;
        if (kb + 8 <= full) {  // warp-uniform
#pragma unroll
          for (int u = 0; u < kTiles; ++u)
#pragma unroll
            for (int e = 0; e < 4; ++e) bm[u][e >> 1] = fmaxf(bm[u][e >> 1], c[u][j][e]);
        } else {
#pragma unroll
          for (int u = 0; u < kTiles; ++u)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int key = kb + 2 * tq + (e & 1);
              c[u][j][e] = key < k_hi && key <= lim[u][e >> 1] ? c[u][j][e] : -INFINITY;
              bm[u][e >> 1] = fmaxf(bm[u][e >> 1], c[u][j][e]);
            }
        }
      }
      float ref[kTiles][2];
#pragma unroll
      for (int u = 0; u < kTiles; ++u)
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) {
#pragma unroll
          for (int o = 1; o < 4; o <<= 1) bm[u][h2] = fmaxf(bm[u][h2], __shfl_xor_sync(0xffffffffu, bm[u][h2], o));
          const float m = fmaxf(mx[u][h2], bm[u][h2] * scale_log2);
          row_rescale(st[u][h2], mx[u][h2], m);
          mx[u][h2] = m;
          ref[u][h2] = m == -INFINITY ? 0.f : m;
        }
#pragma unroll
      for (int j = 0; j < kBlocks; ++j) {
        const int kb = kb0 + 8 * kWarps * j;
        if (kb >= k_hi) break;  // warp-uniform, as the three cases
        if (kb + 8 <= min(nv, k_hi)) {  // visual keys
#pragma unroll
          for (int u = 0; u < kTiles; ++u)
#pragma unroll
            for (int e = 0; e < 4; ++e) st[u][e >> 1].v += ex2f(fmaf(c[u][j][e], scale_log2, -ref[u][e >> 1]));
        } else if (kb >= nv && kb + 8 <= full) {  // trajectory / prompt-text keys
#pragma unroll
          for (int u = 0; u < kTiles; ++u)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              RowSums& s = st[u][e >> 1];
              const float d = fmaf(c[u][j][e], scale_log2, -ref[u][e >> 1]), w = ex2f(d);
              s.t += w;
              if (w > 0.f) s.n = fmaf(w, d, s.n);
            }
        } else {
#pragma unroll
          for (int u = 0; u < kTiles; ++u)
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              RowSums& s = st[u][e >> 1];
              const int key = kb + 2 * tq + (e & 1);
              const float d = fmaf(c[u][j][e], scale_log2, -ref[u][e >> 1]), w = ex2f(d);  // masked: ex2(-inf) = 0
              const bool vis = key < nv, txt = key < L;
              s.v += vis ? w : 0.f;
              s.t += !vis && txt ? w : 0.f;
              s.g += !vis && !txt ? w : 0.f;
              if (!vis && w > 0.f) s.n = fmaf(w, d, s.n);
            }
        }
      }
    }
    // the four lanes of a row (their maximum is common), then the warps
#pragma unroll
    for (int u = 0; u < kTiles; ++u)
#pragma unroll
      for (int h2 = 0; h2 < 2; ++h2) {
        RowSums& s = st[u][h2];
        row_add(s, 1);
        row_add(s, 2);
        if (tq == 0) {
          red_s[warp][16 * u + gq + 8 * h2] = make_float4(s.v, s.t, s.g, s.n);
          red_m[warp][16 * u + gq + 8 * h2] = mx[u][h2];
        }
      }
    __syncthreads();
    const int rows_cta = kPassRows >> log_s, log_rows = 5 - log_s;
    {
      const int row = threadIdx.x / kWarps, w = threadIdx.x % kWarps;
      const float4 x = red_s[w][row];
      RowSums s{x.x, x.y, x.z, x.w};
      float m = red_m[w][row];
      row_merge(s, m, kWarps);
      if (m0 == 0) cluster_wait();  // every CTA of the cluster has started
      // lane w < 5 of a row sends one of its five values to the CTA that finishes the row
      if (w < 5) {
        const float val = w == 0 ? m : (w == 1 ? s.v : (w == 2 ? s.t : (w == 3 ? s.g : s.n)));
        const uint32_t to = static_cast<uint32_t>(row >> log_rows);
        const uint32_t local = static_cast<uint32_t>(__cvta_generic_to_shared(&recv[par][w][((row & (rows_cta - 1)) << log_s) + rank]));
        uint32_t remote;
        asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(to));
        st_cluster(remote, val);
      }
    }
    // every CTA's values have arrived; those of this parity are overwritten two
    // passes on, after the next pass's barrier
    cluster_arrive();
    cluster_wait();
    if (warp == 0) {
      // lane: row lane / S of this CTA's, the state of CTA lane % S
      RowSums s{recv[par][1][lane], recv[par][2][lane], recv[par][3][lane], recv[par][4][lane]};
      float m = recv[par][0][lane];
      row_merge(s, m, S);
      const int p = m0 + static_cast<int>(rank) * rows_cta + (lane >> log_s);
      if ((lane & (S - 1)) == 0 && p < M && ok) {
        const int i = p / G, h = kvh * G + (p - i * G);
        const float tot = s.v + s.t + s.g;
        const long long o = (static_cast<long long>(b) * R + i) * Hq + h;
        mass[o * 3 + 0] = s.v / tot;
        mass[o * 3 + 1] = s.t / tot;
        mass[o * 3 + 2] = s.g / tot;
        const float lnv = s.t + s.g;
        const int n_rest = (L - nv) + i + 1;
        entropy[o] = (n_rest > 1 && lnv > 0.f) ? (logf(lnv) - kLn2 * s.n / lnv) / logf(static_cast<float>(n_rest)) : 0.f;
      }
    }
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

// [B*Hkv][cap][D] bf16 keys as a 3-D tensor; boxes of 64 columns x 32 rows,
// 128-byte swizzle (the layout the kernel's ldmatrix reads)
bool make_key_map(CUtensorMap* map, void* base, int D, int cap, int planes) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[3] = {static_cast<cuuint64_t>(D), static_cast<cuuint64_t>(cap), static_cast<cuuint64_t>(planes)};
  cuuint64_t strides[2] = {static_cast<cuuint64_t>(D) * 2, static_cast<cuuint64_t>(cap) * static_cast<cuuint64_t>(D) * 2};
  cuuint32_t box[3] = {64, 32, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int D>
constexpr int smem_bytes() { return kChunkKeys * 128 * (D / 64) + 1024; }

}  // namespace

extern "C" sd_status sd_attention_budget(const void* q, const sd_kv_cache* cache, int R, int Hq, float scale,
                                         const int32_t* n_visual, float* mass, float* entropy,
                                         sd_stream_t stream) {
  if (!cache) return SD_ERR_INVALID_ARG;
  const int B = cache->batch, Hkv = cache->n_kv_heads, D = cache->head_dim, cap = cache->capacity;
  if (B < 0 || R <= 0 || Hq <= 0 || Hkv <= 0 || cap <= 0 || Hq % Hkv) return SD_ERR_INVALID_ARG;
  if (D != 64 && D != 128) return SD_ERR_UNSUPPORTED;
  if (B > 65535 || Hq > 65535) return SD_ERR_UNSUPPORTED;
  if (B == 0) return SD_OK;
  if (!q || !cache->k || !cache->len || !n_visual || !mass || !entropy) return SD_ERR_INVALID_ARG;
  if (!sd_aligned16(cache->k)) return SD_ERR_INVALID_ARG;
  if (!(scale >= 0.f) || !isfinite(scale)) return SD_ERR_INVALID_ARG;
  const double sc = scale > 0.f ? scale : 1.0 / sqrt(static_cast<double>(D));
  const float scale_log2 = static_cast<float>(sc * 1.4426950408889634);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  // cluster size: the smallest power of two (up to 16) that leaves each CTA
  // at most 256 keys of the largest scene (32 keys a warp)
  int S = 1;
  while (S < 16 && static_cast<long long>(cap) > 256LL * S) S *= 2;
  const auto* qq = static_cast<const __nv_bfloat16*>(q);
  const bool q_vec = sd_aligned16(q);  // else 4-byte loads
  CUtensorMap tk;
  if (!make_key_map(&tk, cache->k, D, cap, B * Hkv)) return SD_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = S;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(S, Hkv, B);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = D == 128 ? smem_bytes<128>() : smem_bytes<64>();
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  cudaError_t e;
  // clusters of 16 are non-portable and the staging buffer passes 48 KB:
  // both allowed once per device and kernel
  static bool allowed[64][2];
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 && !allowed[dev][D == 128]) {
    if (D == 128) {
      cudaFuncSetAttribute(budget_kernel<128>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      cudaFuncSetAttribute(budget_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes<128>());
    } else {
      cudaFuncSetAttribute(budget_kernel<64>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      cudaFuncSetAttribute(budget_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes<64>());
    }
    (void)cudaGetLastError();
    allowed[dev][D == 128] = true;
  }
  if (D == 128) {
    e = cudaLaunchKernelEx(&cfg, budget_kernel<128>, tk, qq, static_cast<const int32_t*>(cache->len), n_visual, R, Hq,
                           Hkv, cap, scale_log2, q_vec, mass, entropy);
  } else {
    e = cudaLaunchKernelEx(&cfg, budget_kernel<64>, tk, qq, static_cast<const int32_t*>(cache->len), n_visual, R, Hq,
                           Hkv, cap, scale_log2, q_vec, mass, entropy);
  }
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return SD_ERR_CUDA;
  }
  SD_CHECK_LAUNCH();
  return SD_OK;
}
