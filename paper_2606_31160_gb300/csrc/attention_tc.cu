// K3 on the 5th-generation tensor cores (tcgen05 + TMEM), and the choice of
// tcgen05 kernel: verify attention of the K + 1 new rows against the
// cached prefix (Eq. verify, Sec. 3.2) and the fused verify layer (M-RoPE of
// Sec. 3.3 / Sec. 4.2 + the KV append of Eq. commit + the attention).
//
// Up to 31 new rows (32 with one query head a KV head) take the row tiles of
// attention_wide.cu, whose loop covers the prefix and whose new rows enter beside it.
// With more (32 to 128, so at most 4 query heads a KV head) the attention runs here,
// every key in the loop, in m-blocks of 64 packed rows:
//     S^T[128 keys][64 rows] = K_tile[128 keys][128 d] . Q^T      (K-major A, B)
//     O^T[128 d][64 rows]   += V_tile^T[128 d][128 keys] . P^T     (MN-major A, B)
// Both accumulators live in tensor memory, S triple-buffered.
//
// Warp roles in a CTA (352 threads). The issuing warps run converged: every
// lane waits on the barriers and one elected lane issues (issued from a
// one-lane branch instead, a batch of 8 MMAs took ~270 ns).
//   warp 0      TMA producer: 128-key tiles of K and V (128B-swizzled boxes)
//               into a K ring and a V ring of two slots each, with a barrier
//               each: a K slot refills once its S product is done, a V slot once
//               its PV product is.
//   warp 1      allocates tensor memory; issues S(t) once the softmax has read
//               the buffer's previous S, S(t - 3), and commits "S(t) ready".
//   warps 2..9  softmax: thread (t, h) owns key lane t of S^T and query rows
//               32 h .. 32 h + 31; P = exp2(S - ref) goes to shared memory as
//               P^T (MN-major, 128-byte swizzle), 16-byte stores, once PV(t - 2)
//               has read that buffer.
//   warp 10     issues PV(t) once P(t) is stored and commits "PV(t) done";
//               one batch is issued while the other executes.
//
// Softmax with a fixed reference: the exact maximum of the CTA's first tile; every
// tile uses it unchanged, so the loop has no cross-warp step and O is never
// rescaled. The result is exact as long as no score exceeds its reference by more
// than kSlack (log2 units), which keeps every weight below 2^kSlack and every sum
// far inside fp32 range; each thread tracks the largest excess it saw, and a CTA
// where some excess is larger runs the whole range a second time with the exact
// maxima as references.
//
// Work split: one thread-block cluster per (scene, KV head, m-block); its CTAs
// take contiguous 32-key-aligned ranges of the keys, and their (m, l, O) partials
// merge through distributed shared memory at the end. Every wait is bounded
// (SD_DEVERR_TIMEOUT instead of a hang).
#include "tc_common.cuh"

#include <math.h>
#include <stdlib.h>
#include <atomic>
#include <mutex>

SD_DEFINE_ERROR_ACCESSOR(sd_take_error_attention_tc)

namespace {

constexpr int kStageKeys = 128; // M of S^T
constexpr int kHalf = kStageKeys * 128;     // one 64-column half of a 128-key tile (16 KB)
constexpr int kKV = 2 * kHalf;              // one K (or V) tile of 128 keys (32 KB)
constexpr int kSoftWarps = 8;
constexpr int kSoftThreads = 32 * kSoftWarps;
constexpr int kPvWarp = 2 + kSoftWarps;        // the warp after the softmax warps issues PV
constexpr int kThreads = 96 + kSoftThreads;
constexpr float kSlack = 64.f;              // log2 units a score may exceed its reference by
// a partial row sent to its owner is [O(128) | l by TMEM lane quarter (4) | m |
// 3 pad] fp32 = 544 bytes (16-byte multiple: one bulk copy per peer)
constexpr int kRowF = kD + 8;
constexpr int kRowL = kD;       // the four l terms (float4)
constexpr int kRowM = kD + 4;   // the row's reference m
constexpr int kRowBytes = kRowF * 4;

// Everything that depends on the packed query rows per CTA (kR: the N of both
// MMAs). A softmax thread owns kR / 2 rows of one key lane.
template <int kR>
struct Cfg {
  static_assert(kR == 64, "row tile");
  static constexpr int kRpt = kR / 2;                       // rows per softmax thread
  // K and V rings of kStages tiles each: a K slot is free once its S product
  // is done, a V slot once its PV product is
  static constexpr int kStages = 2;
  static constexpr int kRingV = kStages * kKV;              // V slots follow the K slots
  static constexpr int kRing = 2 * kStages * kKV;
  static constexpr int kQHalf = kR * 128;
  static constexpr int kQ = 2 * kQHalf;
  static constexpr int kPRow = kR * 2;                      // one key of P^T in bf16
  static constexpr int kP = kStageKeys * kPRow;             // one P^T buffer
  // P^T is MN-major with the 128-byte swizzle; 8-key groups are kPRow * 8 bytes apart
  static constexpr uint64_t kPLayout = 2;
  static constexpr int kTmemCols = 256;                     // S0 | S1 | S2 | O, kR columns each
  // shared memory layout (offsets from the 1024-aligned base)
  static constexpr int kOffQ = kRing;
  static constexpr int kOffP = kOffQ + kQ;
  static constexpr int kOffBar = kOffP + 2 * kP;
  static constexpr int kSBuf = 3;                           // S buffers in tensor memory
  // barriers: full_k[S] full_v[S] p_full[2] s_ready[3] pv_done[S] q_full recv
  // decide s_free[3] tmem_done
  static constexpr int kNumBars = 3 * kStages + 12;
  // tmem slot, (unused), decision, len
  static constexpr int kOffMisc = round_up(kOffBar + kNumBars * 8, 16);
  static constexpr int kOffRowA = kOffMisc + 16;            // [kR] per-row results (reductions)
  static constexpr int kOffRef = kOffRowA + kR * 4;         // [kR] per-row references
  static constexpr int kOffLim = kOffRef + kR * 4;          // [kR] per-row causal key limits
  static constexpr int kSmemBytes = kOffLim + kR * 4 + 1024;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
  static_assert(kOffQ % 1024 == 0 && kOffP % 1024 == 0 && kP % 1024 == 0 && kOffBar % 8 == 0 && kOffRowA % 16 == 0 &&
                    kOffRef % 16 == 0,
                "alignment of the shared-memory regions (swizzle atoms, vector accesses, mbarriers)");
  static_assert(kR * 128 * 4 <= 2 * kP, "row reductions fit the P buffers");
  // cluster merge buffers (in the rings, free once this CTA's last MMA is done)
  static constexpr int kSend = 0;                           // this CTA's kR rows
  static constexpr int kRecv = round_up(kR * kRowBytes, 1024);
  static constexpr int kRecvSlots = kR + 15;                // ceil(kR / c) rows from each of c <= 16 ranks
  static_assert(kRecv + kRecvSlots * kRowBytes <= kRing, "merge buffers");
};

// Sum over the 32 lanes of a warp of each of 32 per-lane values, by a butterfly
// reduce-scatter: at the step of stride s a lane keeps the half of its values
// selected by its bit s and adds its partner's copy of that half. Lane L ends with
// the sum of value `row`.
__device__ __forceinline__ float warp_rows_sum(const float (&v0)[32], int lane, int& row) {
  constexpr int kN = 32;
  float v[kN];
#pragma unroll
  for (int i = 0; i < kN; ++i) v[i] = v0[i];
  int r = 0;
#pragma unroll
  for (int n = kN, s = 16; n > 1; n >>= 1, s >>= 1) {
    const bool hi = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const float keep = hi ? v[i + n / 2] : v[i];
      const float give = hi ? v[i] : v[i + n / 2];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, s);
    }
    if (hi) r += n / 2;
  }
  row = r;
  return v[0];
}
// Per-row reduction (max or sum) over the 128 key lanes of a CTA, for the 256
// softmax threads: thread (key lane kl, rows row0 .. row0 + kN - 1) contributes
// v[j] to row row0 + j. The values pass through buf ([2 kN rows][128] fp32,
// free while this runs); the 2 kN results land in out[]. Called by all
// softmax threads; compact on purpose (it runs once or twice a launch).
template <bool kMax, int kN>
__device__ __forceinline__ void rows_reduce(const float (&v)[kN], int kl, int row0, int st, float* buf,
                                            float* out) {
  constexpr int kRowsAll = 2 * kN;
  constexpr int kPer = kSoftThreads / kRowsAll;  // threads per row (8 or 4)
  constexpr int kVals = 128 / kPer;              // values each of them reads (16 or 32)
#pragma unroll
  for (int j = 0; j < kN; ++j) buf[(row0 + j) * 128 + kl] = v[j];
  asm volatile("bar.sync 2, 256;" ::: "memory");
  const int r = st / kPer, part = st % kPer;
  // part p reads float4 q * kPer + p of its row: per load, the kPer threads of
  // a row cover kPer * 16 contiguous bytes (no bank conflicts beyond the rows)
  const float4* src = reinterpret_cast<const float4*>(buf + r * 128) + part;
  float acc = kMax ? -INFINITY : 0.f;
#pragma unroll
  for (int q = 0; q < kVals / 4; ++q) {
    const float4 x = src[q * kPer];
    acc = kMax ? fmaxf(acc, fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w))) : acc + ((x.x + x.y) + (x.z + x.w));
  }
#pragma unroll
  for (int w = 1; w < kPer; w <<= 1) {
    const float o = __shfl_xor_sync(0xffffffffu, acc, w);
    acc = kMax ? fmaxf(acc, o) : acc + o;
  }
  if (part == 0) out[r] = acc;
  asm volatile("bar.sync 2, 256;" ::: "memory");
}

// Second pass (fixed references exceeded): row r's reference moves to
// ref + max over the range of (score - ref); buf holds every thread's 16 or 32
// per-row maxima at [row][key lane]. Out of line: it runs only when a score
// exceeded its reference by more than the slack.
template <int kN>
__device__ __noinline__ void redo_references(int kl, int row0, int st, int quarter, int lane, float* buf,
                                             float* row_a, float* row_ref) {
  constexpr int kRowsAll = 2 * kN;
  constexpr int kPer = kSoftThreads / kRowsAll;
  constexpr int kVals = 128 / kPer;
  asm volatile("bar.sync 2, 256;" ::: "memory");
  const int r = st / kPer, part = st % kPer;
  const float4* src = reinterpret_cast<const float4*>(buf + r * 128) + part;
  float acc = -INFINITY;
#pragma unroll 1
  for (int q = 0; q < kVals / 4; ++q) {
    const float4 x = src[q * kPer];
    acc = fmaxf(acc, fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)));
  }
  for (int w = 1; w < kPer; w <<= 1) acc = fmaxf(acc, __shfl_xor_sync(0xffffffffu, acc, w));
  if (part == 0) row_a[r] = acc;
  asm volatile("bar.sync 2, 256;" ::: "memory");
  if (quarter == 0 && lane < kN) {
    const float e = row_a[row0 + lane];
    const float m0 = row_ref[row0 + lane] == -INFINITY ? 0.f : row_ref[row0 + lane];
    row_ref[row0 + lane] = e == -INFINITY ? -INFINITY : m0 + e;
  }
  asm volatile("bar.sync 2, 256;" ::: "memory");
}

// ------------------------------------------------------------------ kernel
// Attention over a cache that already holds the R new rows, every key in the
// tensor-core loop, the new rows under per-row key limits (a.early nonzero: the
// block mask). Grid: (cluster size, Hkv * n_mblocks, B); m-block mb takes packed
// query rows mb * kR .. mb * kR + kR - 1.
template <int kR>
__global__ void __launch_bounds__(kThreads, 1)
    verify_attn_tc_kernel(const __grid_constant__ CUtensorMap tm_k128,
                          const __grid_constant__ CUtensorMap tm_v128, const TcArgs a) {
  using C = Cfg<kR>;
  const bool block = a.early != 0;
  constexpr int kS = C::kStages;
  constexpr int kRpt = C::kRpt;
  constexpr uint32_t kIdescS = umma_idesc(128, kR, 0, 0);
  constexpr uint32_t kIdescO = umma_idesc(128, kR, 1, 1);
  constexpr int kTmemAlloc = C::kTmemCols;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const uint32_t base = smem_addr(smem);
  const uint32_t qs = base + C::kOffQ;
  auto bar = [&](int i) { return base + C::kOffBar + 8u * i; };
  // barrier indices; T counts tiles over both passes. SREADY(T) and PVDONE(T)
  // (one slot per ring stage) are tcgen05.commit arrivals. A slot's next
  // phase cannot complete before each of its waiters has seen the current
  // one: S(T + kS) needs the K tile loaded after the producer's wait for
  // SREADY(T); PV(T + kS) needs the V tile loaded after the producer's wait
  // for PVDONE(T); the softmax's tile T + 1 follows its wait for SREADY(T),
  // and its wait for PVDONE(T) comes before P(T + 2), which PV(T + kS) needs.
  // K and V of a tile have their own barriers: a K slot refills once its S
  // product is done, a V slot once its PV product is.
  auto FULLK = [&](int s) { return bar(s); };
  auto FULLV = [&](int s) { return bar(kS + s); };
  auto PFULL = [&](int b) { return bar(2 * kS + b); };
  auto SREADY = [&](int T) { return bar(2 * kS + 2 + T % 3); };  // one per S buffer
  auto PVDONE = [&](int T) { return bar(2 * kS + 5 + T % kS); };
  auto ring_parity = [](int T) { return static_cast<uint32_t>((T / kS) & 1); };
  const uint32_t QFULL = bar(3 * kS + 5);
  const uint32_t RECV = bar(3 * kS + 6);    // the cluster merge's incoming partial rows
  const uint32_t DECIDE = bar(3 * kS + 7);  // whether the range runs a second time
  // the softmax has read S(T) (its tensor-memory buffer takes S(T + 3))
  auto SFREE = [&](int T) { return bar(3 * kS + 8 + T % 3); };
  auto s_parity = [](int T) { return static_cast<uint32_t>((T / 3) & 1); };  // SREADY, SFREE phases
  const uint32_t TMEMDONE = bar(3 * kS + 11);  // every softmax warp has read its last column
  constexpr int kSB = C::kSBuf;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::kOffMisc);
  int* s_redo = reinterpret_cast<int*>(smem + C::kOffMisc + 8);
  float* row_a = reinterpret_cast<float*>(smem + C::kOffRowA);  // [kR] reduction results
  float* row_ref = reinterpret_cast<float*>(smem + C::kOffRef); // [kR] references
  int* row_lim = reinterpret_cast<int*>(smem + C::kOffLim);      // [kR] last key a row sees

  auto gdiv = [&](int p) { return __float2int_rz((static_cast<float>(p) + 0.5f) * a.inv_g); };
  const int rank = blockIdx.x;
  const int csize = gridDim.x;
  const int kvh = blockIdx.y % a.Hkv;
  const int mblock = blockIdx.y / a.Hkv;
  const int b = blockIdx.z;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kS; ++s) {
      mbar_init(FULLK(s), 1);
      mbar_init(FULLV(s), 1);
      mbar_init(PVDONE(s), 1);
    }
    for (int i = 0; i < 3; ++i) mbar_init(SREADY(i), 1);
    for (int i = 0; i < 2; ++i) mbar_init(PFULL(i), kSoftWarps);
    mbar_init(QFULL, 1);  // one softmax thread, once the query tile is stored
    mbar_init(RECV, 1);
    mbar_init(DECIDE, 1);
    for (int i = 0; i < 3; ++i) mbar_init(SFREE(i), kSoftWarps);
    mbar_init(TMEMDONE, kSoftWarps);
    *s_redo = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(tmem_slot)),
                 "r"(kTmemAlloc)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  int* s_len = reinterpret_cast<int*>(smem + C::kOffMisc + 12);
  if (threadIdx.x == 0) {
    *s_len = a.len[b];  // the scene's length advances at the producer's end
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tmem_s = tmem;            // S buffer b at column kR * b
  const uint32_t tmem_o = tmem + kSB * kR; // O^T

  const int n_keys = *s_len;
  const bool valid = n_keys >= a.R && n_keys <= a.cap;
  const int L_prefix = n_keys - a.R;
  if (!valid && rank == 0 && threadIdx.x == 0 && blockIdx.y == 0) sd_set_error(SD_DEVERR_LENGTH);
  const int loop_keys = valid ? n_keys : 0;
  const int nblk = (loop_keys + 31) / 32;
  // rank * nblk < 2^31 (16 ranks, nblk <= cap / 32): 32-bit division
  const int blk_begin = static_cast<int>((static_cast<uint32_t>(rank) * nblk) / static_cast<uint32_t>(csize));
  const int blk_end = static_cast<int>((static_cast<uint32_t>(rank + 1) * nblk) / static_cast<uint32_t>(csize));
  const int key_begin = blk_begin * 32;
  const int key_end = min(blk_end * 32, loop_keys);
  const int n_tiles = (blk_end - blk_begin + 3) / 4;
  // rank c merges packed rows [c * rpc, c * rpc + rows_of(c)) of the m-block's
  // rows_in rows that exist (the tile's rows past M are never exchanged: a
  // single-row draft step with G = 4 moves 4 rows, not 32), rpc = ceil(rows_in / csize)
  const int rows_in = max(1, min(kR, a.M - mblock * kR));
  const int rpc = (rows_in + csize - 1) / csize;
  auto rows_of = [&](int c) { return max(0, min(rpc, rows_in - c * rpc)); };
  const int my_rows = rows_of(rank);
  const int mrow0 = rank * rpc;
  if (warp == 0) {
    // -------------------------------------------------------------- producer
    // the whole warp waits, one elected lane issues the copies
    const int z = b * a.Hkv + kvh;
    const uint64_t evict_first = l2_evict_first_policy();
    auto issue_tiles = [&](int pass) {
      for (int t = 0; t < n_tiles; ++t) {
        const int T = pass * n_tiles + t;
        const int s = T % kS;
        // a whole 128-row box even for a short last tile: keys past the
        // range are masked, rows past the capacity arrive zero-filled
        const int y0 = key_begin + t * kStageKeys;
        // slot s last held tile T - kS (all of pass 0 is done before pass 1)
        const uint32_t kst = base + s * kKV, vst = base + C::kRingV + s * kKV;
        if (t >= kS) mbar_wait(SREADY(T - kS), s_parity(T - kS));
        if (elect_one()) {
          mbar_expect_tx(FULLK(s), static_cast<uint32_t>(kKV));
#pragma unroll
          for (int h = 0; h < 2; ++h) tma_load_3d_hint(kst + h * kHalf, &tm_k128, FULLK(s), h * 64, y0, z, evict_first);
        }
        __syncwarp();
        if (t >= kS) mbar_wait(PVDONE(T - kS), ring_parity(T - kS));
        if (elect_one()) {
          mbar_expect_tx(FULLV(s), static_cast<uint32_t>(kKV));
#pragma unroll
          for (int h = 0; h < 2; ++h) tma_load_3d_hint(vst + h * kHalf, &tm_v128, FULLV(s), h * 64, y0, z, evict_first);
        }
        __syncwarp();
      }
    };
    if (n_tiles > 0) {
      if (elect_one()) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_k128)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_v128)) : "memory");
      }
      __syncwarp();
      issue_tiles(0);
    }
    __syncwarp();
    // The cluster barrier lets peers write partials into this CTA's rings: the
    // softmax threads arrive only after the last MMA of the last pass, so this
    // warp (as the issuing warps) arrives before the second-pass decision.
    cluster_arrive_relaxed();
    __syncwarp();
    if (n_tiles > 0) {
      // every MMA of pass 0 is done when the decision is out
      mbar_wait(DECIDE, 0);
      if (*reinterpret_cast<volatile int*>(s_redo)) issue_tiles(1);
    }
    __syncwarp();
    cluster_wait();
  } else if (warp == 1) {
    // -------------------------------------------------------------- S issue
    // S(T) and PV(T) come from two warps (this one and the PV warp), so that
    // one batch is issued while the other executes; the whole warp waits and
    // one elected lane issues.
    bool arrived = false;
    if (n_tiles > 0) {
      mbar_wait(QFULL, 0);
      // base descriptors; a K step only moves the start address (low field, no carry)
      const uint64_t dK0 = umma_desc(base, 16, 1024);  // K tile: K-major
      const uint64_t dQ = umma_desc(qs, 16, 1024);     // Q: K-major
      for (int pass = 0; pass < 2; ++pass) {
        if (pass == 1) {
          cluster_arrive_relaxed();  // before the decision (see the producer)
          arrived = true;
          mbar_wait(DECIDE, 0);
          if (!*reinterpret_cast<volatile int*>(s_redo)) break;
        }
        const int T0 = pass * n_tiles;
        for (int t = 0; t < n_tiles; ++t) {
          // S(T) reuses the S buffer of tile T - 3: the softmax has read it
          // once SFREE(T - 3) is out; pass 1 starts after all of pass 0
          const int T = T0 + t, st_ = T % kS;
          if (t >= 3) mbar_wait(SFREE(T), s_parity(T - 3));
          mbar_wait(FULLK(st_), ring_parity(T));
          tc_fence_after();
          const uint64_t dk = dK0 + static_cast<uint64_t>((st_ * kKV) >> 4);
          const uint32_t ts = tmem_s + kR * (T % kSB);
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              umma(ts, dk + (((kk >> 2) * kHalf + (kk & 3) * 32) >> 4),
                   dQ + (((kk >> 2) * C::kQHalf + (kk & 3) * 32) >> 4), kIdescS, kk > 0 ? 1 : 0);
            umma_commit(SREADY(T));
          }
          __syncwarp();
        }
      }
    }
    __syncwarp();
    if (!arrived) cluster_arrive_relaxed();
    // the allocating warp frees the tensor memory once every softmax warp has
    // read its last column (every MMA is done by then)
    mbar_wait(TMEMDONE, 0);
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemAlloc) : "memory");
    cluster_wait();
  } else if (warp == kPvWarp) {
    // -------------------------------------------------------------- PV issue
    bool arrived = false;
    if (n_tiles > 0) {
      const uint64_t dV0 = umma_desc(base + C::kRingV, kHalf, 1024);  // V^T: MN-major
      // P^T: MN-major, one swizzle atom wide (kR rows), 8-key groups 8 * kPRow apart
      const uint64_t dP0 = umma_desc(base + C::kOffP, 0, 8 * C::kPRow, C::kPLayout);
      for (int pass = 0; pass < 2; ++pass) {
        if (pass == 1) {
          cluster_arrive_relaxed();  // before the decision (see the producer)
          arrived = true;
          mbar_wait(DECIDE, 0);
          if (!*reinterpret_cast<volatile int*>(s_redo)) break;
        }
        const int T0 = pass * n_tiles;
        for (int t = 0; t < n_tiles; ++t) {
          const int T = T0 + t;
          mbar_wait(PFULL(T & 1), (T >> 1) & 1);
          mbar_wait(FULLV(T % kS), ring_parity(T));  // the V tile has landed
          tc_fence_after();
          const uint64_t dv = dV0 + static_cast<uint64_t>(((T % kS) * kKV) >> 4);
          const uint64_t dp = dP0 + static_cast<uint64_t>(((T & 1) * C::kP) >> 4);
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)
              umma(tmem_o, dv + (kk * 2048 >> 4), dp + (kk * 16 * C::kPRow >> 4), kIdescO,
                   (t > 0 || kk > 0) ? 1 : 0);
            umma_commit(PVDONE(T));
          }
          __syncwarp();
        }
      }
    }
    __syncwarp();
    if (!arrived) cluster_arrive_relaxed();
    cluster_wait();
  } else {
    // -------------------------------------------------------------- softmax
    const int st = threadIdx.x - 64;       // 0..255
    const int half = (warp - 2) >> 2;      // query rows kRpt*half .. kRpt*half + kRpt - 1
    const int quarter = warp & 3;          // TMEM lane quarter of this warp
    const int kl = quarter * 32 + lane;    // key lane of S^T / d lane of O^T
    const uint32_t lane_off = static_cast<uint32_t>(quarter * 32) << 16;
    const int row0 = kRpt * half;          // first query row of this thread
    {
      // the packed query tile: this thread's 16-byte chunks, rows past M zero
      constexpr int kQc = kR * 16 / kSoftThreads;
#pragma unroll
      for (int u = 0; u < kQc; ++u) {
        const int idx = st + u * kSoftThreads, row = idx >> 4, c = idx & 15, p = mblock * kR + row;
        const int i = gdiv(p);
        const uint4 v = valid && p < a.M
                            ? __ldcg(reinterpret_cast<const uint4*>(
                                  a.q + ((static_cast<long long>(b) * a.R + i) * a.Hq + kvh * a.G + (p - i * a.G)) * kD + c * 8))
                            : make_uint4(0, 0, 0, 0);
        st_shared_v4(qs + (c >> 3) * C::kQHalf + row * 128 + (((c & 7) ^ (row & 7)) << 4), v.x, v.y, v.z, v.w);
      }
      // causal limit of each packed row: row p = i * G + g is new row i and
      // sees keys 0 .. L_prefix + i (Eq. verify's mask)
      if (st < kR)
        row_lim[st] = block ? n_keys - 1 : min(n_keys - a.R + gdiv(mblock * kR + st), n_keys - 1);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      named_bar_sync(2, kSoftThreads);  // Q is complete
      if (st == 0) {
        mbar_arrive(QFULL);
      }
    }

    const float sl = a.scale_log2;
    // the reference of a row (log2 units, -inf: no key yet) lives in row_ref and is
    // reloaded every tile (broadcast loads), to stay within the registers that 11
    // warps leave a thread
    float lp[kRpt];   // per-row partial sums of this thread's key lane
    float ex[kRpt];   // largest score - reference seen
#pragma unroll
    for (int j = 0; j < kRpt; ++j) {
      lp[j] = 0.f;
      ex[j] = -INFINITY;
    }
    // per-key-lane mask of rows row0 + j0 .. row0 + j0 + 15 for a tile: the
    // key range, and the causal limit of the new rows that the standalone
    // kernel's range contains
    auto tile_mask = [&](int key0, int j0, bool (&ok)[16]) {
      const int key = key0 + kl;
      const bool key_ok = key < key_end;
      const bool tail = key0 + kStageKeys - 1 > L_prefix;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        ok[j] = key_ok;
        if (tail) ok[j] = ok[j] && key <= row_lim[row0 + j0 + j];
      }
    };
    if (n_tiles > 0) {
      // references: exact row maxima of the first tile (through the P buffers,
      // which no P has used yet)
      mbar_wait(SREADY(0), 0);
      tc_fence_after();
      float v[kRpt];
#pragma unroll
      for (int j0 = 0; j0 < kRpt; j0 += 16) {
        uint32_t r[16];
        tmem_ld16(tmem_s + row0 + j0 + lane_off, r);
        bool ok[16];
        tile_mask(key_begin, j0, ok);
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j0 + j] = ok[j] ? __uint_as_float(r[j]) * sl : -INFINITY;
      }
      rows_reduce<true>(v, kl, row0, st, reinterpret_cast<float*>(smem + C::kOffP), row_ref);
    }
    bool redo = false;
    for (int pass = 0; pass < 2; ++pass) {
      if (pass == 1 && !redo) break;
      for (int t = 0; t < n_tiles; ++t) {
        const int T = pass * n_tiles + t;
        const int bb = T & 1, s = T % kS;
        const int key0 = key_begin + t * kStageKeys;
        const int key = key0 + kl;
        mbar_wait(SREADY(T), s_parity(T));  // S(T) is ready
        tc_fence_after();
        const bool key_ok = key < key_end;
        // P^T key row kl, once PV(T - 2) has read the buffer: kRpt rows =
        // kRpt / 8 16-byte chunks of 8 query rows, swizzled
        const uint32_t prow = base + C::kOffP + bb * C::kP + kl * C::kPRow;
        const int sw = kl & 7;
#pragma unroll
        for (int j0 = 0; j0 < kRpt; j0 += 16) {
          // 16 rows past the tile's existing rows (warp-uniform): no scores to
          // read and no P to write; their P columns stay stale and reach only
          // O columns that are never read. The buffer release and the PV wait
          // stay, so every barrier phase still completes in order.
          if (row0 + j0 >= rows_in) {
            if (j0 + 16 >= kRpt) {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(SFREE(T));
            }
            if (T >= 2 && j0 == 0) mbar_wait(PVDONE(T - 2), ring_parity(T - 2));
            continue;
          }
          uint32_t r[16];
          tmem_ld16(tmem_s + kR * (T % kSB) + row0 + j0 + lane_off, r);
          if (j0 + 16 >= kRpt) {
            // S(T) is in registers (its last 16 rows): its buffer may take S(T + 3)
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(SFREE(T));
          }
          bool ok[16];
          tile_mask(key0, j0, ok);
          float rc[16];
          const float4* rr4 = reinterpret_cast<const float4*>(row_ref + row0 + j0);
#pragma unroll
          for (int j4 = 0; j4 < 4; ++j4) {
            const float4 x = rr4[j4];
            rc[4 * j4 + 0] = x.x;
            rc[4 * j4 + 1] = x.y;
            rc[4 * j4 + 2] = x.z;
            rc[4 * j4 + 3] = x.w;
          }
          // P = exp2(S * scale - ref) in bf16; l partials from the same rounded weights
          uint32_t pw[8];
#pragma unroll
          for (int j = 0; j < 16; j += 2) {
            const float m0 = rc[j] == -INFINITY ? 0.f : rc[j];
            const float m1 = rc[j + 1] == -INFINITY ? 0.f : rc[j + 1];
            const float y0 = ok[j] ? fmaf(__uint_as_float(r[j]), sl, -m0) : -INFINITY;
            const float y1 = ok[j + 1] ? fmaf(__uint_as_float(r[j + 1]), sl, -m1) : -INFINITY;
            ex[j0 + j] = fmaxf(ex[j0 + j], y0);
            ex[j0 + j + 1] = fmaxf(ex[j0 + j + 1], y1);
            const uint32_t w = cvt_bf16x2(ex2(y0), ex2(y1));
            pw[j >> 1] = w;
            lp[j0 + j] += sd_bf16_lo(w);
            lp[j0 + j + 1] += sd_bf16_hi(w);
          }
          if (T >= 2 && j0 == 0) mbar_wait(PVDONE(T - 2), ring_parity(T - 2));  // PV(T - 2) has read P buffer bb
          const int ch = (row0 + j0) >> 3;
          st_shared_v4(prow + ((ch ^ sw) << 4), pw[0], pw[1], pw[2], pw[3]);
          st_shared_v4(prow + (((ch + 1) ^ sw) << 4), pw[4], pw[5], pw[6], pw[7]);
        }
        if (!key_ok) {
          // stale or foreign key row: zero its V row (this thread's 64-column
          // half) so 0 * NaN cannot reach O, once the tile has landed
          mbar_wait(FULLV(s), ring_parity(T));
          const uint32_t vrow = base + C::kRingV + s * kKV + half * kHalf + kl * 128;
#pragma unroll
          for (int c = 0; c < 8; ++c) st_shared_v4(vrow + ((c ^ (kl & 7)) << 4), 0u, 0u, 0u, 0u);  // no two lanes on one bank
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(PFULL(bb));
      }
      if (pass == 0) {
        // did any score exceed its reference by more than kSlack? (one
        // OR-reducing barrier over the softmax threads, while the last PV
        // product runs)
        bool over = false;
#pragma unroll
        for (int j = 0; j < kRpt; ++j) over |= ex[j] > kSlack;
        redo = named_bar_or(2, kSoftThreads, over);
        // before a second pass every MMA of the first is done (the producer
        // refills the rings once the decision is out)
        if (redo && n_tiles > 0) mbar_wait(PVDONE(n_tiles - 1), ring_parity(n_tiles - 1));
        if (st == 0) {
          *s_redo = redo ? 1 : 0;
          mbar_arrive(DECIDE);
        }
        if (redo) {
          // second pass with the exact row maxima of the whole range (every
          // MMA is done: the P buffers are free)
          float* rb = reinterpret_cast<float*>(smem + C::kOffP);
#pragma unroll
          for (int j = 0; j < kRpt; ++j) {
            rb[(row0 + j) * 128 + kl] = ex[j];
            lp[j] = 0.f;
          }
          redo_references<kRpt>(kl, row0, st, quarter, lane, rb, row_a, row_ref);
        }
      }
    }

    // ---- this CTA's partial, staged row-major for the rows' owners: row r =
    //      [O(128) | l per TMEM lane quarter (4) | m | pad]
    float* send = reinterpret_cast<float*>(smem + C::kSend);
    {
      // l of each row over this warp's 32 key lanes; the owner adds the four
      // quarters
      int lrow;
      const float lw = warp_rows_sum(lp, lane, lrow);
      send[(row0 + lrow) * kRowF + kRowL + quarter] = lw;
      if (quarter == 0 && lane < kRpt)
        send[(row0 + lane) * kRowF + kRowM] = n_tiles > 0 ? row_ref[row0 + lane] : -INFINITY;
    }
    if (n_tiles > 0) {
      // every MMA is done once the last PV is (PVDONE's phases complete in order)
      const int Tl = (redo ? 2 : 1) * n_tiles - 1;
      mbar_wait(PVDONE(Tl), ring_parity(Tl));
      tc_fence_after();
    }
    cluster_arrive_relaxed();
#pragma unroll
    for (int j0 = 0; j0 < kRpt; j0 += 16) {
      uint32_t o[16];
      if (n_tiles > 0) {
        tmem_ld16(tmem_o + row0 + j0 + lane_off, o);
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j] = 0u;
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) send[(row0 + j0 + j) * kRowF + kl] = __uint_as_float(o[j]);
    }
    // this warp's last tensor-memory read is done: the allocating warp frees the
    // columns while the partials merge (the kernel's end is not held by it)
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(TMEMDONE);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    named_bar_sync(2, kSoftThreads);
    if (st == 0) mbar_expect_tx(RECV, static_cast<uint32_t>(csize * my_rows * kRowBytes));
    cluster_wait();  // every peer's ring is free to receive
    // softmax warp w sends rank c's rows to rank c (c = w, w + 8), into its
    // slots [rank * rpc, ...); one elected lane of the converged warp issues
    if (elect_one()) {
#pragma unroll 1
      for (int c = warp - 2; c < csize; c += kSoftWarps)
        if (rows_of(c) > 0)
          bulk_copy_s2s(cluster_map(base + C::kRecv + rank * rpc * kRowBytes, c),
                        base + C::kSend + c * rpc * kRowBytes, static_cast<uint32_t>(rows_of(c) * kRowBytes),
                        cluster_map(RECV, c));
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    }
    __syncwarp();
    // ---- merge of the rows this CTA owns; slot c * rpc + rr came from rank c.
    // 64 threads a row, two adjacent d a thread; every partial is weighed by its own
    // reference (each CTA's is the maximum of its own first tile).
    const int rr = st >> 6, d = 2 * (st & 63);
    mbar_wait(RECV, 0);
    const float* recv = reinterpret_cast<const float*>(smem + C::kRecv);
#pragma unroll 1
    for (int r = rr; r < my_rows; r += kSoftThreads / 64) {  // warp-uniform
      const float* part = recv + r * kRowF;  // rank c's partial at part + c * rpc * kRowF
      float ox = 0.f, oy = 0.f, l = 0.f, mx = -INFINITY;
#pragma unroll 4
      for (int c = 0; c < csize; ++c) mx = fmaxf(mx, part[c * rpc * kRowF + kRowM]);
      const float msub = mx == -INFINITY ? 0.f : mx;
#pragma unroll 4
      for (int c = 0; c < csize; ++c) {
        const float* pc = part + c * rpc * kRowF;
        const float w = ex2(pc[kRowM] - msub);
        const float2 o = *reinterpret_cast<const float2*>(pc + d);
        const float4 lq = *reinterpret_cast<const float4*>(pc + kRowL);
        ox = fmaf(w, o.x, ox);
        oy = fmaf(w, o.y, oy);
        l = fmaf(w, (lq.x + lq.y) + (lq.z + lq.w), l);
      }
      const int p = mblock * kR + mrow0 + r;
      if (valid && p < a.M && l > 0.f) {
        const float inv_l = 1.f / l;
        const int i = gdiv(p), gq = p - i * a.G;
        *reinterpret_cast<uint32_t*>(a.out + ((static_cast<long long>(b) * a.R + i) * a.Hq + kvh * a.G + gq) * kD +
                                     d) = cvt_bf16x2(ox * inv_l, oy * inv_l);
      }
    }
    if (elect_one()) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    __syncwarp();
  }
  // no CTA-wide barrier at the end: every warp leaves when its own work is
  // done (the softmax warps last: they wait for the partials coming in and for
  // their outgoing copies to have been read)
}

// ------------------------------------------------------------------ host
// cluster sizes that a call may choose (sd_set_cluster_size forces 1, 2, 4, 6, 8 or 16)
constexpr int kNumClusterSizes = 9;
constexpr int kClusterSizes[kNumClusterSizes] = {1, 2, 4, 5, 6, 8, 10, 12, 16};

// The row tiles: 32, 48, 64 and 80 packed rows of attention_wide.cu (the new rows
// beside the prefix loop) for head dims 128 and 64, 64 of this file's kernel (every
// key in the loop).
enum Tile { kWide32 = 0, kWide48, kWide64, kWide80, kWideTiles, kAll64 = 2 * kWideTiles, kNumTiles };
constexpr int kTileRows[kWideTiles] = {32, 48, 64, 80};

// per device: how many clusters of each size fit at once, for each row tile
struct DevState {
  bool ready = false;
  bool ok = false;
  int active[kNumTiles][kNumClusterSizes] = {};
};

bool set_attributes(const void* const* kerns, int n_kerns, int smem, int* active) {
  for (int i = 0; i < n_kerns; ++i)
    if (cudaFuncSetAttribute(kerns[i], cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaFuncSetAttribute(kerns[i], cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      (void)cudaGetLastError();
      return false;
    }
  for (int i = 0; i < kNumClusterSizes; ++i) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = kClusterSizes[i];
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(kClusterSizes[i], 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kerns[0], &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      n = 0;
    }
    active[i] = n;
  }
  return true;
}

DevState* state() {
  static DevState st[16];
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 16) return nullptr;
  std::lock_guard<std::mutex> lock(mu);
  DevState& s = st[dev];
  if (!s.ready) {
    s.ready = true;
    const void* all64[1] = {reinterpret_cast<const void*>(verify_attn_tc_kernel<64>)};
    s.ok = set_attributes(all64, 1, Cfg<64>::kSmemBytes, s.active[kAll64]);
    for (int i = 0; i < 2 * kWideTiles; ++i)
      s.ok = s.ok && sd_internal_wide_active(kTileRows[i % kWideTiles], i < kWideTiles ? 128 : 64, kClusterSizes,
                                             kNumClusterSizes, s.active[i]);
  }
  return &s;
}

// Cluster size: the least waves x (128-key tiles a CTA + a fixed cost a wave), in
// tiles; those past the first three, which are in shared memory before the rows are,
// count a quarter more. Sizes above 8 cost more a wave (their set-up and exchange),
// and one that leaves no room for the next layer's clusters loses the overlap of its
// stream when layers are chained (the choice is the same with and without the early
// prefix, so that both give the same bits). On the wider row tiles, whose 128 keys take
// longer, these weigh less, but for size 10's charge: it is what the measurements below
// give on 32 and on 80 rows alike, and leaves 10 the shapes between 8 and 12 (8 heads:
// 5 of the next layer's clusters still fit) and those of 9 to 12 heads.
// The weights are fitted to 70 measured shapes (1 to 256 (scene, head) pairs, L = 512 to
// 16384): the choice is within 2.5% of the best size on 62 of them. The others (pairs, L:
// chosen / best, us): 80 rows 8, 4096: 8 / 12, 10.97 / 10.53; 32 rows 4, 4096: 12 / 16,
// 7.0 / 6.4; 12, 2048: 6 / 8, 7.3 / 6.8; 24, 512: 2 / 4, 6.1 / 5.6; 32, 512: 2 / 4,
// 6.3 / 5.9; 16, 2048: 5 / 4, 6.2 / 5.75; 24, 2048: 5 / 4, 7.6 / 7.2; 64, 512: 2 / 1,
// 6.8 / 6.4. Measured, one scene, 8 KV heads, us a launch at
// sizes 8 / 10 / 12 (7, 9, 11 lie between or above; 13 and more do not fit in one wave):
//   chained, 32 rows: L = 4096 6.3 / 6.6 / 7.8, 8192 9.4 / 8.9 / 9.8, 16384 14.8 / 14.6 / 13.7
//   chained, 80 rows: L = 4096 10.7 / 11.1 / 11.5, 8192 14.6 / 14.2 / 14.2, 16384 20.9 / 19.9 / 18.6
// 4 KV heads at 8 / 10 / 12 / 16: draft step L = 4096 6.9 / 6.6 / 6.1 / 6.2, chained 5.5 /
// 5.6 / 5.2 / 5.6. 20 pairs, L = 4099, 48 rows, at 5 / 6 / 8: 11.2 / 11.0 / 16.9. 24 pairs,
// L = 8192, 32 rows, at 4 / 5: 18.0 / 17.7. (All measured before the rows had references.)
int pick_cluster(const int* active, long long units, int cap, int rows) {
  const double nblk = (cap + 31) / 32, wide = rows <= 32 ? 1.0 : (rows <= 48 ? 0.8 : 0.5);
  double best_cost = -1;
  int best = 0;
  for (int i = 0; i < kNumClusterSizes; ++i) {
    const int cs = kClusterSizes[i];
    if (active[i] <= 0) continue;
    if (cs > 1 && nblk < 2.0 * cs) continue;
    const long long waves = (units + active[i] - 1) / active[i];
    // the share of the next layer's clusters that fit beside this layer's
    const double room = waves > 1 ? 0.0 : static_cast<double>(active[i] - units) / static_cast<double>(units);
    const double fixed = (waves > 1 ? 3.0 : 1.0) + (cs == 10 ? 0.8 : wide * (cs == 12 ? 1.2 : (cs == 16 ? 1.6 : 0.0))) +
                         wide * 2.3 * (room < 1.0 ? 1.0 - room : 0.0);
    const double tiles = nblk / (4.0 * cs);
    const double cost = static_cast<double>(waves) * (tiles + 0.25 * (tiles > 3.0 ? tiles - 3.0 : 0.0) + fixed);
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best = cs;
    }
  }
  return best;
}

}  // namespace

static bool tc_enabled() {
  // SD_ATTENTION_KERNEL=mma selects the mma.sync kernel for every shape
  // (comparison and testing); anything else keeps the tcgen05 path.
  static const bool on = [] {
    const char* e = getenv("SD_ATTENTION_KERNEL");
    return !(e && e[0] == 'm');
  }();
  return on;
}

// How the tcgen05 path runs a shape: row tile, its packed rows, m-blocks (row
// tiles per KV head), cluster size and whether the weights are two bf16 terms
// where the tile has both forms; cs == 0: not served.
struct TcPlan {
  int tile = kWide32, rows = 0, mblocks = 0, cs = 0;
  bool split = false;
};

// Cluster size forced by sd_set_cluster_size (0: chosen per call).
static std::atomic<int> g_forced_cluster{0};

extern "C" sd_status sd_set_cluster_size(int cluster_size) {
  if (cluster_size == 0) {
    g_forced_cluster.store(0);
    return SD_OK;
  }
  for (int cs : {1, 2, 4, 6, 8, 16})
    if (cs == cluster_size) {
      g_forced_cluster.store(cluster_size);
      return SD_OK;
    }
  return SD_ERR_INVALID_ARG;
}

// The tile and cluster size of a shape: up to 31 new rows beside the prefix loop
// on the smallest wide tile that holds the packed rows in one m-block (every key
// read once), above 80 rows on two; more new rows with every key in the loop
// (all_keys). The 32-row tile holds 16 new rows; 17 to 32 of one query head each
// take the 48-row tile with the weights in two terms (32 of them, 32 scenes of 8 heads,
// L = 2048: 45.1 us, against 60.7 on the all-keys kernel's 64 rows; 4 scenes, L = 700:
// 7.7 against 14.2). A layer of 32 new rows stays three kernels.
static TcPlan tc_plan(int B, int R, int Hq, int Hkv, int D, int cap, bool all_keys, bool layer = false) {
  TcPlan p;
  if (!tc_enabled() || (D != kD && (D != 64 || all_keys)) || Hkv <= 0 || Hq % Hkv || R <= 0) return p;
  const int M = (Hq / Hkv) * R;
  if (M > 2 * 64) return p;
  if (all_keys) {
    p.tile = kAll64;
  } else {
    if (R > 31 && !(R == 32 && M == 32 && D == kD && !layer)) return p;
    p.split = M <= 32 && R > 16;
    p.tile = M <= 32 && R <= 16 ? kWide32 : (M <= 48 ? kWide48 : (M <= 64 ? kWide64 : (M <= 80 ? kWide80 : (M <= 96 ? kWide48 : kWide64))));
  }
  p.rows = all_keys ? 64 : kTileRows[p.tile];
  if (!all_keys && D == 64) p.tile += kWideTiles;
  DevState* s = state();
  if (!s || !s->ok) return p;
  p.mblocks = (M + p.rows - 1) / p.rows;
  const int* active = s->active[p.tile];
  const int forced = g_forced_cluster.load();
  for (int i = 0; i < kNumClusterSizes && forced > 0; ++i)
    if (kClusterSizes[i] == forced && active[i] > 0) p.cs = forced;
  if (p.cs == 0) p.cs = pick_cluster(active, static_cast<long long>(B) * Hkv * p.mblocks, cap, p.rows);
  return p;
}

bool sd_internal_tc_serves(int B, int R, int Hq, int Hkv, int D, int cap) {
  return tc_plan(B, R, Hq, Hkv, D, cap, D == kD).cs > 0;
}

bool sd_internal_tc_serves_layer(int B, int R, int Hq, int Hkv, int D, int cap) {
  return D == kD && tc_plan(B, R, Hq, Hkv, D, cap, false, true).cs > 0;
}

int sd_internal_tc_cluster(int B, int R, int Hq, int Hkv, int D, int cap, bool layer) {
  if (layer) return D == kD ? tc_plan(B, R, Hq, Hkv, D, cap, false, true).cs : 0;
  const TcPlan p = tc_plan(B, R, Hq, Hkv, D, cap, false);
  return p.cs > 0 ? p.cs : tc_plan(B, R, Hq, Hkv, D, cap, true).cs;
}

template <int kR>
static sd_status launch_tc(const sd_kv_cache* cache, const TcArgs& a, const TcPlan& plan, cudaStream_t stream) {
  const int B = cache->batch, Hkv = cache->n_kv_heads, cap = cache->capacity;
  CUtensorMap k128, v128;
  if (!make_map(&k128, cache->k, cap, B * Hkv, 128) || !make_map(&v128, cache->v, cap, B * Hkv, 128))
    return SD_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = plan.cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(plan.cs, Hkv * plan.mblocks, B);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = Cfg<kR>::kSmemBytes;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cudaLaunchKernelEx(&cfg, verify_attn_tc_kernel<kR>, k128, v128, a) != cudaSuccess) {
    (void)cudaGetLastError();
    return SD_ERR_CUDA;
  }
  return SD_OK;
}

// Routed here by sd_verify_attention for G * R <= 128. Up to 31 new rows (32 of one
// query head each) take the wide tiles, whose loop covers the prefix only, with the
// prefix optionally streamed before the dependency wait (SD_ATTN_PREFIX_EARLY);
// more take the kernel whose loop covers every key (the flag is then a promise it
// does not need).
sd_status sd_internal_verify_attention_tc(const void* q, const sd_kv_cache* cache, void* out,
                                          int R, int Hq, float scale_log2, int flags, cudaStream_t stream,
                                          bool* handled) {
  *handled = false;
  const int B = cache->batch, Hkv = cache->n_kv_heads;
  const bool block = (flags & SD_ATTN_BLOCK_MASK) != 0, early = (flags & SD_ATTN_PREFIX_EARLY) != 0;
  TcPlan plan = tc_plan(B, R, Hq, Hkv, cache->head_dim, cache->capacity, false);
  const bool all_keys = plan.cs <= 0;
  if (all_keys) plan = tc_plan(B, R, Hq, Hkv, cache->head_dim, cache->capacity, true);
  if (plan.cs <= 0) return SD_OK;
  TcArgs a = {};
  a.q = static_cast<const __nv_bfloat16*>(q);
  a.out = static_cast<__nv_bfloat16*>(out);
  a.len = cache->len;
  a.kc = static_cast<__nv_bfloat16*>(cache->k);
  a.vc = static_cast<__nv_bfloat16*>(cache->v);
  a.R = R;
  a.Hq = Hq;
  a.Hkv = Hkv;
  a.G = Hq / Hkv;
  a.M = a.G * R;
  a.inv_g = 1.0f / static_cast<float>(a.G);
  a.cap = cache->capacity;
  a.n_mblocks = plan.mblocks;
  a.scale_log2 = scale_log2;
  *handled = true;
  if (!all_keys) {
    RopeTable tab = {};
    a.early = (early && cache->head_dim == kD ? 1 : 0) | (block ? 2 : 0);  // (the flag is for head dim 128)
    // a programmatic dependent launch either way: without the flag the kernel
    // waits before its first global access, so only its launch and set-up
    // (barriers, tensor memory) overlap the kernel before it
    return sd_internal_wide_launch(cache, a, tab, plan.rows, plan.split, plan.cs, false, stream);
  }
  a.early = block ? 1 : 0;  // the all-keys kernel's block mask
  return launch_tc<64>(cache, a, plan, stream);
}

// The fused verify layer (rope + append + attention) on the tcgen05 path.
sd_status sd_internal_verify_layer_tc(void* q, void* k_new, const void* v_new, const int32_t* pos,
                                      const RopeTable& tab, const sd_kv_cache* cache, void* out,
                                      int R, int Hq, float scale_log2, uint32_t* ticket, int early,
                                      int block, cudaStream_t stream, bool* handled) {
  *handled = false;
  const int B = cache->batch, Hkv = cache->n_kv_heads;
  if (cache->head_dim != kD) return SD_OK;
  const TcPlan plan = tc_plan(B, R, Hq, Hkv, cache->head_dim, cache->capacity, false, true);
  if (plan.cs <= 0) return SD_OK;
  TcArgs a = {};
  a.q = static_cast<const __nv_bfloat16*>(q);
  a.out = static_cast<__nv_bfloat16*>(out);
  a.len = cache->len;
  a.qw = static_cast<__nv_bfloat16*>(q);
  a.k_new = static_cast<__nv_bfloat16*>(k_new);
  a.v_new = static_cast<const __nv_bfloat16*>(v_new);
  a.kc = static_cast<__nv_bfloat16*>(cache->k);
  a.vc = static_cast<__nv_bfloat16*>(cache->v);
  a.pos = pos;
  a.ticket = ticket;
  a.kv_ticket = ticket + B;
  a.early = (early ? 1 : 0) | (block ? 2 : 0);  // prefix before the wait; the block mask
  a.R = R;
  a.Hq = Hq;
  a.Hkv = Hkv;
  a.G = Hq / Hkv;
  a.M = a.G * R;
  a.inv_g = 1.0f / static_cast<float>(a.G);
  a.cap = cache->capacity;
  a.n_mblocks = plan.mblocks;
  a.scale_log2 = scale_log2;
  *handled = true;
  // without the early prefix a dependent launch as well: the wait comes before any
  // global access (the draft's single-row steps, each reading the length the step
  // before advanced)
  return sd_internal_wide_launch(cache, a, tab, plan.rows, plan.split, plan.cs, true, stream);
}
