// K2: KV-cache append and rollback (sm_103a).
//
// Eq. commit (Sec. 3.2): an iteration commits l + 1 tokens, t <- t + l + 1.
// The verify pass appends the keys/values of all R = K + 1 rows before the
// acceptance is known; afterwards the length moves back to keep only the
// n_emit = l + 1 committed rows. Nothing is erased: later appends overwrite.
//
// Append: one CTA per scene reads len[b] once, copies the R x Hkv rows with
// 16-byte vector stores, then advances len[b]; keeping the scene in one CTA
// makes the read-then-advance of len race-free without a grid-wide ticket.
// Rollback: one thread per length entry, no host synchronisation.
#include "common.cuh"

SD_DEFINE_ERROR_ACCESSOR(sd_take_error_kv)

namespace {

__global__ void __launch_bounds__(512) kv_append_kernel(uint4* __restrict__ kc, uint4* __restrict__ vc,
                                                        int32_t* __restrict__ len,
                                                        const uint4* kn, const uint4* vn, int R, int hkv,
                                                        int cap, int vec_per_row) {
  sd_pdl_enter();
  const int b = blockIdx.x;
  __shared__ int s_len;
  if (threadIdx.x == 0) {
    const int l = len[b];
    const bool ok = l >= 0 && (long long)l + R <= cap;
    if (!ok) sd_set_error(SD_DEVERR_KV_OVERFLOW);
    s_len = ok ? l : -1;
  }
  __syncthreads();
  const int l0 = s_len;
  if (l0 < 0) return;
  const int per_scene = R * hkv * vec_per_row;
  kn += static_cast<long long>(b) * per_scene;  // [b][r][g][vec]
  vn += static_cast<long long>(b) * per_scene;
  constexpr int kBatch = 4;  // chunks a thread has in flight
  for (int i0 = threadIdx.x; i0 < per_scene; i0 += kBatch * blockDim.x) {
    uint4 k[kBatch], v[kBatch];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int i = i0 + u * blockDim.x;
      if (i < per_scene) k[u] = __ldcg(kn + i), v[u] = __ldcg(vn + i);
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int i = i0 + u * blockDim.x;
      if (i >= per_scene) break;
      const int vec = i % vec_per_row;
      const int t = i / vec_per_row;
      const int g = t % hkv;
      const int r = t / hkv;
      const long long dst = (((long long)b * hkv + g) * cap + (l0 + r)) * vec_per_row + vec;
      kc[dst] = k[u];
      vc[dst] = v[u];
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) len[b] = l0 + R;
}

// The rotation of a layer's new query and key rows and the append in one
// launch: block 0 of a scene rotates its key rows in place and copies them and
// the value rows into the cache, then advances len[b] (read by all of its
// threads before); the other blocks rotate the query rows, a 16-byte chunk a
// thread. Bound by the latency of one launch: rows, positions and length travel
// together, the rotation's table is read before the wait.
template <int D>
__global__ void __launch_bounds__(512) rope_append_kernel(uint4* __restrict__ q, uint4* __restrict__ kn,
                                                          const uint4* vn, const int32_t* pos,
                                                          uint4* __restrict__ kc, uint4* __restrict__ vc,
                                                          int32_t* __restrict__ len, int R, int hq, int hkv, int cap,
                                                          const __grid_constant__ RopeTable tab) {
  constexpr int kVec = D / 8;
  const int b = blockIdx.y, vec = threadIdx.x % kVec;
  const RopeChunk chunk = sd_rope_chunk(vec, tab);
  sd_pdl_enter();
  pos += static_cast<long long>(b) * R * 3;
  if (blockIdx.x > 0) {
    const long long i = (blockIdx.x - 1) * 512ll + threadIdx.x, n = static_cast<long long>(R) * hq * kVec;
    if (i >= n) return;
    const int32_t* p3 = pos + i / (kVec * hq) * 3;
    uint4* x = q + b * n + i;
    *x = sd_rope_rotate8(*x, __ldcg(p3), __ldcg(p3 + 1), __ldcg(p3 + 2), chunk);
    return;
  }
  const int l0 = len[b], n = R * hkv * kVec;
  const bool ok = l0 >= 0 && static_cast<long long>(l0) + R <= cap;
  for (int i = threadIdx.x; i < n; i += 512) {
    const int t = i / kVec, g = t % hkv, r = t / hkv;
    const long long src = static_cast<long long>(b) * n + i;  // [b][r][g][vec]
    const uint4 k = kn[src], v = __ldcg(vn + src);
    const uint4 kr = sd_rope_rotate8(k, __ldcg(pos + r * 3), __ldcg(pos + r * 3 + 1), __ldcg(pos + r * 3 + 2), chunk);
    kn[src] = kr;
    if (ok) {
      const long long dst = ((static_cast<long long>(b) * hkv + g) * cap + (l0 + r)) * kVec + vec;
      kc[dst] = kr;
      vc[dst] = v;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    if (ok) len[b] = l0 + R;
    else sd_set_error(SD_DEVERR_KV_OVERFLOW);
  }
}

__global__ void kv_rollback_kernel(int32_t* __restrict__ len, int count, int B,
                                   const int32_t* committed, int n_appended) {
  sd_pdl_enter();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int c = __ldcg(committed + i % B);
  const int l = len[i];
  const int nl = l - n_appended + c;
  if (c < 0 || c > n_appended || nl < 0) {
    sd_set_error(SD_DEVERR_ROLLBACK);
    return;
  }
  len[i] = nl;
}

}  // namespace

extern "C" sd_status sd_kv_append(const sd_kv_cache* cache, const void* k_new, const void* v_new,
                                  int R, sd_stream_t stream) {
  if (!cache) return SD_ERR_INVALID_ARG;
  const int B = cache->batch, hkv = cache->n_kv_heads, cap = cache->capacity, D = cache->head_dim;
  if (B < 0 || hkv <= 0 || cap <= 0 || R < 0) return SD_ERR_INVALID_ARG;
  if (D <= 0 || (D * 2) % 16) return SD_ERR_UNSUPPORTED;
  if (B == 0 || R == 0) return SD_OK;
  if (!cache->k || !cache->v || !cache->len || !k_new || !v_new) return SD_ERR_INVALID_ARG;
  if (!sd_aligned16(cache->k) || !sd_aligned16(cache->v) || !sd_aligned16(k_new) ||
      !sd_aligned16(v_new))
    return SD_ERR_INVALID_ARG;
  if (sd_launch_pdl(kv_append_kernel, dim3(B), dim3(512), 0, reinterpret_cast<cudaStream_t>(stream),
                    static_cast<uint4*>(cache->k), static_cast<uint4*>(cache->v), cache->len,
                    static_cast<const uint4*>(k_new), static_cast<const uint4*>(v_new), R, hkv, cap,
                    D / 8) != cudaSuccess) {
    (void)cudaGetLastError();
    return SD_ERR_CUDA;
  }
  return SD_OK;
}

sd_status sd_internal_rope_append(void* q, void* k_new, const void* v_new, const int32_t* pos, const RopeTable& tab,
                                  const sd_kv_cache* cache, int R, int Hq, cudaStream_t stream) {
  const int B = cache->batch, hkv = cache->n_kv_heads, D = cache->head_dim;
  const long long nq = (static_cast<long long>(R) * Hq * (D / 8) + 511) / 512;
  if (sd_launch_pdl(D == 64 ? rope_append_kernel<64> : rope_append_kernel<128>, dim3(static_cast<unsigned>(1 + nq), B),
                    dim3(512), 0, stream, static_cast<uint4*>(q), static_cast<uint4*>(k_new),
                    static_cast<const uint4*>(v_new), pos, static_cast<uint4*>(cache->k), static_cast<uint4*>(cache->v),
                    cache->len, R, Hq, hkv, cache->capacity, tab) != cudaSuccess) {
    (void)cudaGetLastError();
    return SD_ERR_CUDA;
  }
  return SD_OK;
}

extern "C" sd_status sd_kv_rollback(int32_t* len, int count, int B, const int32_t* committed,
                                    int n_appended, sd_stream_t stream) {
  if (count < 0 || B <= 0 || n_appended < 0) return SD_ERR_INVALID_ARG;
  if (count % B) return SD_ERR_INVALID_ARG;
  if (count == 0) return SD_OK;
  if (!len || !committed) return SD_ERR_INVALID_ARG;
  const int threads = 128;
  if (sd_launch_pdl(kv_rollback_kernel, dim3((count + threads - 1) / threads), dim3(threads), 0,
                    reinterpret_cast<cudaStream_t>(stream), len, count, B, committed,
                    n_appended) != cudaSuccess) {
    (void)cudaGetLastError();
    return SD_ERR_CUDA;
  }
  return SD_OK;
}
