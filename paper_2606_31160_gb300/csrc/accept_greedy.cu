// K4: greedy acceptance (Eqs. verify, accept, commit, Sec. 3.2; Eq.
// accept-length, Sec. 4.3).
//
//   r*_j = argmax_v logits[b][j][v]   (lowest index among equal maxima)
//   l    = number of leading drafts equal to r*   (draft[j] vs r*_j, j < K)
//   emit draft[0..l-1], r*_l            n_emit = l + 1
//
// One kernel: a CTA scans a segment of one row (grid: segment, row, scene) and
// raises the row's 64-bit key (ordered value, then lowest index) by atomicMax;
// the scene's last CTA (atomic ticket, no spin) reads the K + 1 keys, compares
// with the drafts, writes the outputs and zeroes keys and ticket. The order of
// the keys is total, so the result does not depend on the order they arrive in:
// bit-exact and deterministic.
//
// Bound: the logits stream from HBM once. The scan keeps a running maximum only
// (packed bf16x2 or fp32 maxima of 64 bytes a thread and step, under 1
// instruction a value) and remembers the step that raised it; the index is
// looked up afterwards by the threads that hold the segment's maximum. Carrying
// (value, index) through every comparison took ~7 instructions a value, and one
// cluster of 16 x 512 threads a row put short-lived CTAs on the SMs one at a
// time. Rows of any alignment take the same path (the elements before the first
// and after the last 16-byte boundary are read singly).
// 32 scenes, K = 7, V = 151936, bf16 (78 MB): 16.0 us, 4.9 TB/s (49.4 before); one
// scene 5.6 us (6.7), bound by the latency of one launch. Launched as a dependent of
// the kernel before it, whose end it waits for: 18.4 us of the 32 scenes without that.
#include "common.cuh"

#include <mutex>

SD_DEFINE_ERROR_ACCESSOR(sd_take_error_greedy)

namespace {

constexpr int kThreads = 256;
constexpr int kMaxChunks = 1024;
constexpr int kStep = 4;  // 16-byte vectors a thread reads per step

// Order-preserving map of a float to uint32 (-0 as +0); every value, -inf
// included, maps above 0.
__device__ __forceinline__ uint32_t ordered(float x) {
  const uint32_t u = __float_as_uint(x + 0.f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ __nv_bfloat162 as_pair(uint32_t w) {
  __nv_bfloat162 v;
  memcpy(&v, &w, 4);
  return v;
}

// Largest value of a 16-byte vector, folded into m (NaN loses to any number).
template <typename T>
struct Fold;
template <>
struct Fold<float> {
  float m = -INFINITY;
  __device__ __forceinline__ void add(const uint4& w) {
    m = fmaxf(m, fmaxf(fmaxf(__uint_as_float(w.x), __uint_as_float(w.y)),
                       fmaxf(__uint_as_float(w.z), __uint_as_float(w.w))));
  }
  __device__ __forceinline__ float value() const { return m; }
};
template <>
struct Fold<__nv_bfloat16> {
  uint32_t m = 0xff80ff80u;  // -inf pair
  __device__ __forceinline__ void add(const uint4& w) {
    const __nv_bfloat162 x = __hmax2(__hmax2(as_pair(w.x), as_pair(w.y)), __hmax2(as_pair(w.z), as_pair(w.w)));
    const __nv_bfloat162 y = __hmax2(as_pair(m), x);
    memcpy(&m, &y, 4);
  }
  __device__ __forceinline__ float value() const { return fmaxf(sd_bf16_lo(m), sd_bf16_hi(m)); }
};

// (loads past the read-only path: the kernel is resident while its inputs are written)
__device__ __forceinline__ float load_one(const float* p) { return __ldcg(p); }
__device__ __forceinline__ float load_one(const __nv_bfloat16* p) { return sd_ldcg_bf16(p); }

// First element of a vector that equals best (a value it holds), as its offset.
__device__ __forceinline__ int first_equal(const float*, const uint4& w, float best) {
  const uint32_t x[4] = {w.x, w.y, w.z, w.w};
  int at = 0x7fffffff;
#pragma unroll
  for (int j = 3; j >= 0; --j)
    if (__uint_as_float(x[j]) == best) at = j;
  return at;
}
__device__ __forceinline__ int first_equal(const __nv_bfloat16*, const uint4& w, float best) {
  const uint32_t x[4] = {w.x, w.y, w.z, w.w};
  int at = 0x7fffffff;
#pragma unroll
  for (int j = 3; j >= 0; --j) {
    if (sd_bf16_hi(x[j]) == best) at = 2 * j + 1;
    if (sd_bf16_lo(x[j]) == best) at = 2 * j;
  }
  return at;
}

// grid (segment, row, scene). A row's whole 16-byte vectors are split into
// segments of vps; segment 0 also takes the elements before the first boundary,
// the last one those after the last.
template <typename T>
__global__ void __launch_bounds__(kThreads) greedy_kernel(const T* logits, int R, int V, int vps,
                                                          const int32_t* draft,
                                                          int32_t* __restrict__ n_emit,
                                                          int32_t* __restrict__ tokens,
                                                          int32_t* __restrict__ argmax_out,
                                                          unsigned long long* __restrict__ keys,
                                                          uint32_t* __restrict__ ticket) {
  constexpr int kPer = 16 / sizeof(T);
  __shared__ uint32_t s_best[kThreads / 32];
  __shared__ uint32_t s_index;
  __shared__ bool s_last;
  const int seg = blockIdx.x, r = blockIdx.y, b = blockIdx.z;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  sd_pdl_enter();  // its CTAs are resident by the time the kernel before it has finished
  const T* row = logits + (static_cast<long long>(b) * R + r) * V;
  const int head = min(V, static_cast<int>((16 - (reinterpret_cast<uintptr_t>(row) & 15)) & 15) / static_cast<int>(sizeof(T)));
  const int n_vec = (V - head) / kPer;
  const uint4* vec = reinterpret_cast<const uint4*>(row + head);
  const int v0 = min(n_vec, seg * vps), v1 = seg == static_cast<int>(gridDim.x) - 1 ? n_vec : min(n_vec, v0 + vps);
  if (threadIdx.x == 0) s_index = 0xffffffffu;
  // ---- running maximum and the step that raised it (a thread's steps ascend)
  float best = -INFINITY;
  int step = -1;
  for (int v = v0 + static_cast<int>(threadIdx.x); v < v1; v += kStep * kThreads) {
    Fold<T> f;
    if (v + (kStep - 1) * kThreads < v1) {
      uint4 w[kStep];
#pragma unroll
      for (int k = 0; k < kStep; ++k) w[k] = __ldcg(vec + v + k * kThreads);
#pragma unroll
      for (int k = 0; k < kStep; ++k) f.add(w[k]);
    } else {
#pragma unroll
      for (int k = 0; k < kStep; ++k)
        if (v + k * kThreads < v1) f.add(__ldcg(vec + v + k * kThreads));
    }
    const float m = f.value();
    if (m > best) {
      best = m;
      step = v;
    }
  }
  // the single elements at the row's ends, one a thread (fewer than 8 each)
  float single = -INFINITY;
  int single_at = -1;
  if (seg == 0 && static_cast<int>(threadIdx.x) < head) single_at = threadIdx.x;
  if (seg == static_cast<int>(gridDim.x) - 1 && threadIdx.x >= 32) {
    const int e = head + n_vec * kPer + static_cast<int>(threadIdx.x) - 32;
    if (e < V) single_at = e;
  }
  if (single_at >= 0) single = load_one(row + single_at);
  const float top = fmaxf(best, single);
  const uint32_t wbest = __reduce_max_sync(0xffffffffu, ordered(top == top ? top : -INFINITY));
  if (lane == 0) s_best[warp] = wbest;
  __syncthreads();
  uint32_t bmax = s_best[0];
#pragma unroll
  for (int w = 1; w < kThreads / 32; ++w) bmax = max(bmax, s_best[w]);
  // ---- the lowest index of the segment's maximum (no value above -inf: its start)
  uint32_t at = 0xffffffffu;
  const bool none = bmax == ordered(-INFINITY);
  if (single_at >= 0 && !none && ordered(single) == bmax) at = single_at;
  if (step >= 0 && ordered(best) == bmax) {
#pragma unroll
    for (int k = kStep - 1; k >= 0; --k) {
      const int v = step + k * kThreads;
      if (v >= v1) continue;
      const int e = first_equal(row, __ldcg(vec + v), best);
      if (e != 0x7fffffff) at = min(static_cast<uint32_t>(head + v * kPer + e), at);
    }
  }
  const uint32_t wat = __reduce_min_sync(0xffffffffu, at);
  if (lane == 0 && wat != 0xffffffffu) atomicMin(&s_index, wat);
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t idx = s_index != 0xffffffffu ? s_index : static_cast<uint32_t>(seg == 0 ? 0 : min(V - 1, head + v0 * kPer));
    atomicMax(&keys[static_cast<long long>(b) * R + r], (static_cast<unsigned long long>(bmax) << 32) | (0xffffffffu - idx));
    __threadfence();
    s_last = atomicAdd(&ticket[b], 1u) == static_cast<uint32_t>(R * gridDim.x - 1);
  }
  __syncthreads();
  if (!s_last || warp != 0) return;
  __threadfence();
  // ---- the scene's last CTA, warp 0: l = first j < K with draft[j] != r*_j (K
  // when none): one ballot per 32 drafts
  __shared__ int s_star[128];
  const int K = R - 1;
  int ell = K;
  bool range_ok = true;
  for (int j0 = 0; j0 < R; j0 += 32) {
    const int j = j0 + lane;
    int star = 0, d = 0;
    if (j < R) {
      unsigned long long* key = keys + static_cast<long long>(b) * R + j;
      star = static_cast<int>(0xffffffffu - static_cast<uint32_t>(__ldcg(key)));
      if (j < K) d = __ldcg(draft + static_cast<long long>(b) * K + j);
      *key = 0ull;  // re-armed for the next call
      s_star[j] = star;
      if (argmax_out) argmax_out[static_cast<long long>(b) * R + j] = star;
    }
    range_ok &= j >= K || (d >= 0 && d < V);
    const uint32_t miss = __ballot_sync(0xffffffffu, j < K && d != star);
    if (miss && ell == K) ell = j0 + __ffs(miss) - 1;
  }
  __syncwarp();
  if (!__all_sync(0xffffffffu, range_ok) && lane == 0) sd_set_error(SD_DEVERR_TOKEN_RANGE);
  int32_t* tk = tokens + static_cast<long long>(b) * R;
  // an accepted draft equals its row's argmax
  for (int j = lane; j < R; j += 32) tk[j] = j <= ell ? s_star[j] : -1;
  if (lane == 0) {
    n_emit[b] = ell + 1;
    ticket[b] = 0;
  }
}

// Vectors a segment: about six CTAs an SM over all rows, so that one wave holds
// the whole scan, and at least 16 KB (one step of every thread) a segment.
int segment_vectors(int B, int R, int V, int elem_bytes) {
  const long long row = (static_cast<long long>(V) * elem_bytes + 15) / 16;
  const long long ctas = 6LL * sd_num_sms();
  long long vps = (row * B * R + ctas - 1) / ctas;
  if (vps < kStep * kThreads) vps = kStep * kThreads;
  const long long segs = (row + vps - 1) / vps;
  return static_cast<int>((row + segs - 1) / segs);
}

// The workspace size (and the room that limits the allocation-free call) counts
// 8 bytes per chunk of 4096 elements of every row, more elements when a row would
// have over kMaxChunks chunks: a function of the shape only, the same wherever it
// is queried. The keys take the first B * R of them.
void plan(int B, int R, int V, int* chunk, int* n_chunks) {
  (void)B;
  (void)R;
  long long ch = 4096;
  while ((V + ch - 1) / ch > kMaxChunks) ch *= 2;
  *chunk = static_cast<int>(ch);
  *n_chunks = static_cast<int>((V + ch - 1) / ch);
}

size_t ws_bytes_for(int B, int R, int n_chunks) {
  return static_cast<size_t>(B) * R * n_chunks * sizeof(float2) + static_cast<size_t>(B) * 4 + 256;
}

}  // namespace

extern "C" size_t sd_accept_greedy_workspace(int B, int K, int V) {
  if (B <= 0 || K < 0 || V <= 0) return 0;
  int chunk, n_chunks;
  plan(B, K + 1, V, &chunk, &n_chunks);
  return ws_bytes_for(B, K + 1, n_chunks);
}

// Host-side argument checks shared by both entry points.
static sd_status check_args(const void* logits, sd_dtype dtype, int B, int K, int V,
                            const int32_t* draft, int32_t* n_emit, int32_t* tokens) {
  if (B < 0 || K < 0 || V <= 0) return SD_ERR_INVALID_ARG;
  if (dtype != SD_BF16 && dtype != SD_F32) return SD_ERR_INVALID_ARG;
  if (K + 1 > 128 || B > 65535) return SD_ERR_UNSUPPORTED;
  if (B == 0) return SD_OK;
  if (!logits || !n_emit || !tokens || (K > 0 && !draft)) return SD_ERR_INVALID_ARG;
  return SD_OK;
}

static sd_status launch(const void* logits, sd_dtype dtype, int B, int K, int V,
                        const int32_t* draft, int32_t* n_emit, int32_t* tokens, int32_t* argmax,
                        unsigned long long* keys, uint32_t* ticket, cudaStream_t st) {
  const int R = K + 1, eb = dtype == SD_BF16 ? 2 : 4;
  const int vps = segment_vectors(B, R, V, eb);
  // whole vectors of a row at most (an unaligned row has one fewer): one segment at least
  const long long row = (static_cast<long long>(V) * eb + 15) / 16;
  const dim3 grid(static_cast<unsigned>((row + vps - 1) / vps), R, B);
  const cudaError_t e =
      dtype == SD_BF16 ? sd_launch_pdl(greedy_kernel<__nv_bfloat16>, grid, dim3(kThreads), 0, st,
                                       static_cast<const __nv_bfloat16*>(logits), R, V, vps, draft, n_emit, tokens, argmax,
                                       keys, ticket)
                       : sd_launch_pdl(greedy_kernel<float>, grid, dim3(kThreads), 0, st, static_cast<const float*>(logits),
                                       R, V, vps, draft, n_emit, tokens, argmax, keys, ticket);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    return SD_ERR_CUDA;
  }
  return SD_OK;
}

extern "C" sd_status sd_accept_greedy(const void* logits, sd_dtype dtype, int B, int K, int V,
                                      const int32_t* draft, int32_t* n_emit, int32_t* tokens,
                                      int32_t* argmax, void* ws, size_t ws_bytes,
                                      sd_stream_t stream) {
  const sd_status chk = check_args(logits, dtype, B, K, V, draft, n_emit, tokens);
  if (chk != SD_OK || B == 0) return chk;
  const int R = K + 1;
  int chunk, n_chunks;
  plan(B, R, V, &chunk, &n_chunks);
  const size_t need = ws_bytes_for(B, R, n_chunks);
  if (!ws || ws_bytes < need || !sd_aligned16(ws)) return SD_ERR_WORKSPACE;
  auto* keys = static_cast<unsigned long long*>(ws);  // the first B * R of the partials' room
  auto* ticket = reinterpret_cast<uint32_t*>(static_cast<char*>(ws) +
                                             static_cast<size_t>(B) * R * n_chunks * sizeof(float2));
  return launch(logits, dtype, B, K, V, draft, n_emit, tokens, argmax, keys, ticket,
                reinterpret_cast<cudaStream_t>(stream));
}

// ---------------------------------------------------------------------------
// Allocation-free variant. Some callers cannot allocate device memory at the
// point where they accept drafts: a serving loop whose memory pool is owned
// and fully carved up by another runtime, a pre-planned inference graph that
// forbids allocation once it runs, or an embedded host that has no device
// allocator at all. For them the scratch this kernel needs lives in a
// file-scope device array of fixed size, loaded with the library (every GPU
// that loads it holds these bytes until the process exits).
//
// Layout: tickets of up to kNoAllocMaxB scenes at the front, so their place
// never moves with the call's shape and no key lands on them; the rows' keys
// follow. The array starts zeroed when the module loads, and every completed
// call leaves tickets and keys at zero again. All calls share the array: calls that overlap on the GPU
// (other streams, other threads) race and must not be issued.
// ---------------------------------------------------------------------------
constexpr size_t kNoAllocBytes = size_t(1) << 20;  // 1 MiB
constexpr int kNoAllocMaxB = 4096;
constexpr size_t kNoAllocTicketBytes = kNoAllocMaxB * sizeof(uint32_t);
static __device__ __align__(256) unsigned char g_greedy_scratch[kNoAllocBytes];

// Device address of the array on the current device, resolved once per device
// (host code cannot use the symbol itself: it is a host-side stand-in).
static void* noalloc_scratch() {
  static void* ptrs[64] = {nullptr};
  static std::mutex mu;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    (void)cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (!ptrs[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_greedy_scratch) != cudaSuccess || !p) {
      (void)cudaGetLastError();
      return nullptr;
    }
    ptrs[dev] = p;
  }
  return ptrs[dev];
}

extern "C" size_t sd_accept_greedy_noalloc_max_bytes(void) { return kNoAllocBytes; }

extern "C" sd_status sd_accept_greedy_noalloc(const void* logits, sd_dtype dtype, int B, int K,
                                              int V, const int32_t* draft, int32_t* n_emit,
                                              int32_t* tokens, int32_t* argmax,
                                              sd_stream_t stream) {
  const sd_status chk = check_args(logits, dtype, B, K, V, draft, n_emit, tokens);
  if (chk != SD_OK || B == 0) return chk;
  const int R = K + 1;
  int chunk, n_chunks;
  plan(B, R, V, &chunk, &n_chunks);
  const size_t part_bytes = static_cast<size_t>(B) * R * n_chunks * sizeof(float2);
  if (B > kNoAllocMaxB || kNoAllocTicketBytes + part_bytes > kNoAllocBytes) return SD_ERR_WORKSPACE;
  void* scratch = noalloc_scratch();
  if (!scratch) return SD_ERR_CUDA;
  auto* ticket = static_cast<uint32_t*>(scratch);
  auto* keys = reinterpret_cast<unsigned long long*>(static_cast<char*>(scratch) + kNoAllocTicketBytes);
  return launch(logits, dtype, B, K, V, draft, n_emit, tokens, argmax, keys, ticket,
                reinterpret_cast<cudaStream_t>(stream));
}
