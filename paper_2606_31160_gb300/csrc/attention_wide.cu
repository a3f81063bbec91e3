// K3 / the fused verify layer for more than 32 packed query rows per KV head
// (Eq. verify, Sec. 3.2; drafts of K = 8 and the K = 16 blocks of Sec. 5), head
// dim 128, up to 31 new rows, on the 5th-generation tensor cores.
//
// As in attention_tc.cu both products run transposed, the 128-wide dimension
// on the MMA's M side:
//     S^T[128 keys][kR rows] = K_tile . Q^T,   O^T[128 d][kR rows] += V_tile^T . P^T
// with kR = 48, 64 or 80 packed rows, the smallest that holds the rows of a KV
// head (two m-blocks of 48 or 64 above 80): a K = 16 block of the 8B target
// (68 rows) is one tile and reads every key once.
//
// The new rows are one more tile: the cluster's last rank holds the R (rotated)
// new keys and values in shared memory in the operands' own layout, so their
// scores and values are products like every other tile's (32 keys, the causal
// limit per row). Scored on the CUDA cores instead, rows x new keys on the
// rows a CTA merges, they took 26 us a launch at one CTA a head and K = 16.
//
// Fixed reference. Weights are 2^(score * scale) with no reference subtracted:
// a floating-point weight keeps its relative precision at any size, so only
// overflow and underflow would matter. A row sum above 2^kHigh or, over a
// warp's keys, below 2^kLow (log2) sends the CTA through its range again with
// each row's exact maximum as its reference: one pass for the maxima, one for
// the weights. No reduction and no reference product stands between S and P.
//
// Warps (608 threads): 0 the TMA producer, 1 issues S and owns tensor memory, 2
// issues PV, 3..18 two softmax groups of eight. Group g takes tiles T with
// T % 2 == g and P buffer g, so a group has two tiles' time for its tile's
// dependent chain (barrier wake-up, tensor-memory load, exponentials, stores)
// while the other group's tile is in the products. With one group of eight on
// every tile that chain set the pace: ~1.1 us a 128-key tile of 64 rows against
// ~0.45 us of products. Products of pairs (fma / add f32x2) and a select on the
// packed weights take 4 issue slots a weight instead of ~9.5.
#include "tc_common.cuh"

#include <math.h>

#include <type_traits>

SD_DEFINE_ERROR_ACCESSOR(sd_take_error_attention_wide)

namespace {

constexpr int kStageKeys = 128;
constexpr int kHalf = kStageKeys * 128;  // one 64-column half of a 128-key tile (16 KB)
constexpr int kKV = 2 * kHalf;           // one K (or V) tile (32 KB)
constexpr int kSoftWarps = 16;
constexpr int kSoftThreads = 32 * kSoftWarps;
constexpr int kFirstSoft = 3;            // the first softmax warp
constexpr int kSoft0 = 32 * kFirstSoft;  // the first softmax thread
constexpr int kThreads = kSoft0 + kSoftThreads;
constexpr int kMaxNew = 32;              // new rows held in shared memory
constexpr int kNewHalf = kMaxNew * 128;  // one 64-column half of the new key (value) rows
constexpr float kHigh = 18446744073709551616.f;          // 2^64: a larger row sum runs the range again
constexpr float kLow = 8.271806125530277e-25f;           // 2^-80: a smaller one too
// a partial row sent to its owner: [O(128) | l by softmax group and lane
// quarter (8) | reference | 3 pad] fp32 (560 bytes)
constexpr int kRowL = kD;
constexpr int kRowM = kD + 8;
constexpr int kRowF = kD + 12;
constexpr int kRowBytes = kRowF * 4;

template <int kR>
struct Cfg {
  static_assert(kR == 48 || kR == 64 || kR == 80, "row tile");
  static constexpr int kRpt = kR / 2;   // rows of a softmax thread in its tile
  static constexpr int kStages = 2;     // K slots, and V slots
  static constexpr int kRingV = kStages * kKV;
  static constexpr int kRing = 2 * kStages * kKV;
  static constexpr int kQHalf = kR * 128;
  // P^T is MN-major with the 32-byte swizzle: 16 rows x 8 keys an atom, the
  // 16-row groups kPGroup apart
  static constexpr int kPGroup = kStageKeys * 32;
  static constexpr int kP = (kR / 16) * kPGroup;
  static constexpr int kSStride = kR == 48 ? 64 : (kR == 64 ? 64 : 128);  // columns between S0 | S1 | S2 | O
  static constexpr int kTmemCols = 4 * kSStride;
  // shared memory (offsets from the 1024-aligned base). The new-key tile's S
  // product reads 128 rows from each half of kOffNewK: rows past kMaxNew are
  // the regions behind it, their scores are never used.
  static constexpr int kOffNewK = kRing;
  static constexpr int kOffNewV = kOffNewK + 2 * kNewHalf;
  static constexpr int kOffQ = kOffNewV + 2 * kNewHalf;
  static constexpr int kOffP = kOffQ + 2 * kQHalf;
  static constexpr int kOffBar = kOffP + 2 * kP;
  // full_k[2] full_v[2] p_full[2] s_ready[3] s_free[3] pv_done[2] q_full recv decide tmem_done
  static constexpr int kNumBars = 3 * kStages + 12;
  static constexpr int kOffMisc = round_up(kOffBar + kNumBars * 8, 16);
  static constexpr int kOffRef = kOffMisc + 32;       // [kR] negated references
  static constexpr int kOffLim = kOffRef + kR * 4;    // [kR] last new key a row sees
  static constexpr int kOffSum = kOffLim + kR * 4;    // [kR][8] row sums by group and lane quarter
  static constexpr int kSmemBytes = kOffSum + kR * 32 + 1024;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
  static_assert(kOffNewV % 1024 == 0 && kOffQ % 1024 == 0 && kOffP % 1024 == 0 && kQHalf % 1024 == 0, "swizzle atoms");
  static_assert(kOffNewK + kNewHalf + kHalf <= kOffBar, "the new-key tile's product stays inside");
  static_assert(kMaxNew * 64 * 8 <= 2 * kP, "rotation table fits the P buffers");
  static_assert(kR * 128 * 4 <= 2 * kP, "row maxima fit the P buffers");
  // cluster merge: incoming rows in the K ring (free after the last S), this
  // CTA's in the V ring (free after the last PV). ceil(n / c) * c < n + 16
  static_assert((kR + 15) * kRowBytes <= kRingV && kR * kRowBytes <= kRing - kRingV, "merge buffers");
};

// kN (16 or 8) consecutive fp32 columns of this warp's 32 TMEM lanes
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[16]) { tmem_ld16(taddr, r); }
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];\n\ttcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ uint64_t pack2(uint32_t lo, uint32_t hi) {
  uint64_t d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(lo), "r"(hi));
  return d;
}
__device__ __forceinline__ uint64_t pack2f(float lo, float hi) {
  return pack2(__float_as_uint(lo), __float_as_uint(hi));
}
__device__ __forceinline__ void unpack2(uint64_t d, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(d));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// Weights of kN rows of one key: P = 2^(S * scale - ref) in bf16, the row sums
// advanced by the same rounded weights, stored to the key's P^T chunks. keep
// masks each packed pair (0 drops a weight whatever its score, NaN included).
template <int kN, typename Keep>
__device__ __forceinline__ void weights_to_p(const uint32_t (&r)[kN], const float* nref, uint64_t sl2, Keep keep,
                                             uint64_t* lp2, uint32_t (&pw)[kN / 2]) {
#pragma unroll
  for (int j = 0; j < kN; j += 4) {
    const float4 nr = *reinterpret_cast<const float4*>(nref + j);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float y0, y1;
      unpack2(fma2(pack2(r[j + 2 * e], r[j + 2 * e + 1]), sl2, e == 0 ? pack2f(nr.x, nr.y) : pack2f(nr.z, nr.w)), y0, y1);
      const uint32_t w = keep(j + 2 * e, cvt_bf16x2(ex2(y0), ex2(y1)));
      pw[j / 2 + e] = w;
      lp2[j / 2 + e] = add2(lp2[j / 2 + e], pack2(w << 16, w & 0xffff0000u));
    }
  }
}

// Sum over the 32 lanes of a warp of each of 8 per-lane values: lane L ends
// with the sum of value (L >> 2).
__device__ __forceinline__ float warp_sum8(const float (&v0)[8], int lane) {
  float v[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = v0[i];
#pragma unroll
  for (int n = 8, s = 16; n > 1; n >>= 1, s >>= 1) {
    const bool hi = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < n / 2; ++i) {
      const float keep = hi ? v[i + n / 2] : v[i];
      const float give = hi ? v[i] : v[i + n / 2];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, s);
    }
  }
  float x = v[0];
  x += __shfl_xor_sync(0xffffffffu, x, 2);
  x += __shfl_xor_sync(0xffffffffu, x, 1);
  return x;
}

// ------------------------------------------------------------------ kernel
// kMode 1: the verify layer (M-RoPE, append, attention) whose prefix, len and
// pos are read before the dependency wait; 3: the same, everything after the
// wait; 2: the attention over a cache that already holds the R new rows
// (prefix before the wait when bit 0 of a.early is set). Bit 1 of a.early: the
// block mask. Grid: (cluster size, Hkv * n_mblocks, B); m-block mb takes packed
// rows mb * kR .. mb * kR + kR - 1.
template <int kR, int kMode>
__global__ void __launch_bounds__(kThreads, 1)
    verify_wide_kernel(const __grid_constant__ CUtensorMap tm_k128, const __grid_constant__ CUtensorMap tm_v128,
                       const TcArgs a, const RopeTable tab) {
  using C = Cfg<kR>;
  constexpr bool kFused = kMode != 2;
  constexpr bool rows_first = kMode == 3;
  constexpr int kS = C::kStages;
  constexpr int kRpt = C::kRpt;
  constexpr uint32_t kIdescS = umma_idesc(128, kR, 0, 0);
  constexpr uint32_t kIdescO = umma_idesc(128, kR, 1, 1);
  const bool early = kMode == 1 || (kMode == 2 && (a.early & 1) != 0);
  const bool block = (a.early & 2) != 0;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const uint32_t base = smem_addr(smem);
  const uint32_t qs = base + C::kOffQ;
  auto bar = [&](int i) { return base + C::kOffBar + 8u * i; };
  // T counts the tiles of all passes (the new-key tile included), TL those the
  // producer loads. A barrier's next phase never completes before its waiters
  // have seen the current one: S(T + 3) and P(T + 2) follow the softmax's waits
  // for S(T) and PV(T), and a K (V) slot's next tile the producer's wait for
  // its S (PV). A waiter that skips phases of a slot (a group sees every second
  // tile) knows the skipped ones complete: products complete in order.
  auto FULLK = [&](int s) { return bar(s); };
  auto FULLV = [&](int s) { return bar(kS + s); };
  auto PFULL = [&](int T) { return bar(2 * kS + (T & 1)); };
  auto SREADY = [&](int T) { return bar(2 * kS + 2 + T % 3); };
  auto SFREE = [&](int T) { return bar(2 * kS + 5 + T % 3); };
  auto PVDONE = [&](int T) { return bar(2 * kS + 8 + T % kS); };
  const uint32_t QFULL = bar(3 * kS + 8);
  const uint32_t RECV = bar(3 * kS + 9);
  const uint32_t DECIDE = bar(3 * kS + 10);  // phase 0: whether the range runs again; phase 1: the maxima are in
  const uint32_t TMEMDONE = bar(3 * kS + 11);
  auto par3 = [](int T) { return static_cast<uint32_t>((T / 3) & 1); };
  auto parS = [](int T) { return static_cast<uint32_t>((T / kS) & 1); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::kOffMisc);
  int* s_redo = reinterpret_cast<int*>(smem + C::kOffMisc + 4);
  int* s_len = reinterpret_cast<int*>(smem + C::kOffMisc + 8);
  int* s_kvlast = reinterpret_cast<int*>(smem + C::kOffMisc + 12);
  float* row_nref = reinterpret_cast<float*>(smem + C::kOffRef);
  int* row_lim = reinterpret_cast<int*>(smem + C::kOffLim);
  float* row_sum = reinterpret_cast<float*>(smem + C::kOffSum);

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
    for (int i = 0; i < 2; ++i) mbar_init(PFULL(i), kSoftWarps / 2);
    for (int i = 0; i < 3; ++i) {
      mbar_init(SREADY(i), 1);
      mbar_init(SFREE(i), kSoftWarps / 2);
    }
    mbar_init(QFULL, 1);
    mbar_init(RECV, 1);
    mbar_init(DECIDE, 1);
    mbar_init(TMEMDONE, kSoftWarps);
    *s_redo = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                 "r"(C::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // a launch without the early prefix waits here, before any global access
  if (!early) griddep_wait();
  if (threadIdx.x == 0) *s_len = a.len[b];  // the scene's length advances at the producer's end
  const bool last_rank = rank == csize - 1;
  // this thread's 16-byte chunks: of the packed query tile (row idx >> 4, chunk
  // idx & 15, rows past M zero) and, in the cluster's last rank, of the new key
  // and value rows
  constexpr int kQc = (kR * 16 + kSoftThreads - 1) / kSoftThreads;
  const int st = static_cast<int>(threadIdx.x) - kSoft0;  // softmax threads: 0 .. 511
  auto q_off = [&](int p) {
    const int i = gdiv(p);
    return ((static_cast<long long>(b) * a.R + i) * a.Hq + kvh * a.G + (p - i * a.G)) * kD;
  };
  const bool raw_kv = last_rank && st < a.R * 16;
  const long long kv_row = ((static_cast<long long>(b) * a.R + (st >> 4)) * a.Hkv + kvh) * kD + (st & 15) * 8;
  uint4 pre_q[kQc], pre_k = make_uint4(0, 0, 0, 0), pre_v = make_uint4(0, 0, 0, 0);
  if (kFused && warp >= kFirstSoft) {
    if (rows_first) {
      // one global round trip before the tiles: the rows with the positions
#pragma unroll
      for (int u = 0; u < kQc; ++u) {
        const int idx = st + u * kSoftThreads, p = mblock * kR + (idx >> 4);
        pre_q[u] = idx < kR * 16 && p < a.M
                       ? __ldcg(reinterpret_cast<const uint4*>(a.qw + q_off(p) + (idx & 15) * 8))
                       : make_uint4(0, 0, 0, 0);
      }
      if (raw_kv) {
        pre_k = __ldcg(reinterpret_cast<const uint4*>(a.k_new + kv_row));
        pre_v = __ldcg(reinterpret_cast<const uint4*>(a.v_new + kv_row));
      }
    }
    // rotation table of the R new positions: (cos, sin) per (row, pair)
    float2* tabw = reinterpret_cast<float2*>(smem + C::kOffP);
#pragma unroll 1
    for (int idx = st; idx < a.R * 64; idx += kSoftThreads) {
      const int i = idx >> 6, d = idx & 63;
      const int32_t pc = a.pos[(static_cast<long long>(b) * a.R + i) * 3 + tab.axis[d]];
      tabw[idx] = sd_rope_cs(static_cast<float>(pc), d, tab);
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t tmem_o = tmem + 3 * C::kSStride;

  const int len0 = *s_len;
  const int L_pre = kFused ? len0 : len0 - a.R;
  const bool valid = L_pre >= 0 && L_pre + a.R <= a.cap;
  if (!valid && rank == 0 && threadIdx.x == 0 && blockIdx.y == 0)
    sd_set_error(kFused && L_pre >= 0 ? SD_DEVERR_KV_OVERFLOW : SD_DEVERR_LENGTH);
  // the prefix in 32-key blocks, split over the cluster's ranks
  const int nblk = valid ? (L_pre + 31) / 32 : 0;
  const int blk_begin = static_cast<int>((static_cast<uint32_t>(rank) * nblk) / static_cast<uint32_t>(csize));
  const int blk_end = static_cast<int>((static_cast<uint32_t>(rank + 1) * nblk) / static_cast<uint32_t>(csize));
  const int key_begin = blk_begin * 32;
  const int key_end = min(blk_end * 32, valid ? L_pre : 0);
  const int n_pre = (blk_end - blk_begin + 3) / 4;           // prefix tiles
  const bool has_new = valid && last_rank;                   // and the new-key tile
  const int n_tiles = n_pre + (has_new ? 1 : 0);
  // rank c merges packed rows [c * rpc, ...) of the m-block's rows_in rows
  const int rows_in = max(1, min(kR, a.M - mblock * kR));
  const int rpc = (rows_in + csize - 1) / csize;
  auto rows_of = [&](int c) { return max(0, min(rpc, rows_in - c * rpc)); };
  const int my_rows = rows_of(rank);
  const int mrow0 = rank * rpc;

  if (warp == 0) {
    // -------------------------------------------------------------- producer
    const int z = b * a.Hkv + kvh;
    const uint64_t evict_first = l2_evict_first_policy();
    auto issue_tiles = [&](int pass) {
      for (int t = 0; t < n_pre; ++t) {
        const int T = pass * n_tiles + t;
        const int s = (pass * n_pre + t) % kS;
        // a whole 128-row box even for a short last tile: keys past the range
        // are masked, rows past the capacity arrive zero-filled
        const int y0 = key_begin + t * kStageKeys;
        const uint32_t kst = base + s * kKV, vst = base + C::kRingV + s * kKV;
        if (t >= kS) mbar_wait(SREADY(T - kS), par3(T - kS));
        if (elect_one()) {
          mbar_expect_tx(FULLK(s), static_cast<uint32_t>(kKV));
#pragma unroll
          for (int h = 0; h < 2; ++h) tma_load_3d_hint(kst + h * kHalf, &tm_k128, FULLK(s), h * 64, y0, z, evict_first);
        }
        __syncwarp();
        if (t >= kS) mbar_wait(PVDONE(T - kS), parS(T - kS));
        if (elect_one()) {
          mbar_expect_tx(FULLV(s), static_cast<uint32_t>(kKV));
#pragma unroll
          for (int h = 0; h < 2; ++h) tma_load_3d_hint(vst + h * kHalf, &tm_v128, FULLV(s), h * 64, y0, z, evict_first);
        }
        __syncwarp();
      }
    };
    if (n_pre > 0) {
      if (elect_one()) {
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_k128)) : "memory");
        asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tm_v128)) : "memory");
        // chained layers: the cluster launched last starts only when the
        // previous layer frees its SMs; the first head's CTAs bring its tiles
        // of their own key range, and its query and new rows, into L2
        if (early && kvh == 0 && mblock == 0 && b == static_cast<int>(gridDim.z) - 1 && a.Hkv > 1) {
          const int zl = b * a.Hkv + a.Hkv - 1;
          for (int t = 0; t < n_pre; ++t)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              tma_prefetch_3d(&tm_k128, h * 64, key_begin + t * kStageKeys, zl);
              tma_prefetch_3d(&tm_v128, h * 64, key_begin + t * kStageKeys, zl);
            }
          if (rank == 0)
            for (int i = 0; i < a.R; ++i) {
              const long long row = static_cast<long long>(b) * a.R + i;
              bulk_prefetch_l2((kFused ? a.qw : a.q) + (row * a.Hq + (a.Hkv - 1) * a.G) * kD, a.G * kD * 2);
              if (kFused) {
                bulk_prefetch_l2(a.k_new + (row * a.Hkv + a.Hkv - 1) * kD, kD * 2);
                bulk_prefetch_l2(a.v_new + (row * a.Hkv + a.Hkv - 1) * kD, kD * 2);
              }
            }
        }
      }
      __syncwarp();
      issue_tiles(0);
    }
    __syncwarp();
    // the softmax threads arrive last (after the last S of the last pass), so
    // this warp and the issuing warps arrive before the decision
    if (csize > 1) cluster_arrive_relaxed();
    if (kFused && elect_one()) {
      // advance the scene's length once every CTA of the scene has read it
      __threadfence();
      const uint32_t total = gridDim.x * gridDim.y;
      if (atomicAdd(&a.ticket[b], 1u) == total - 1) {
        if (len0 >= 0 && len0 + a.R <= a.cap) a.len[b] = len0 + a.R;
        a.ticket[b] = 0;
      }
    }
    __syncwarp();
    if (n_tiles > 0) {
      mbar_wait(DECIDE, 0);
      if (*reinterpret_cast<volatile int*>(s_redo)) {
        issue_tiles(1);
        mbar_wait(DECIDE, 1);  // every product of pass 1 is done
        issue_tiles(2);
      }
    }
    __syncwarp();
    if (csize > 1) cluster_wait();
  } else if (warp == 1) {
    // -------------------------------------------------------------- S issue
    bool arrived = false;
    if (n_tiles > 0) {
      mbar_wait(QFULL, 0);
      const uint64_t dK0 = umma_desc(base, 16, 1024);
      const uint64_t dN = umma_desc(base + C::kOffNewK, 16, 1024);
      const uint64_t dQ = umma_desc(qs, 16, 1024);
      for (int pass = 0; pass < 3; ++pass) {
        if (pass == 1) {
          if (csize > 1) cluster_arrive_relaxed();
          arrived = true;
          mbar_wait(DECIDE, 0);
          if (!*reinterpret_cast<volatile int*>(s_redo)) break;
        }
        if (pass == 2) mbar_wait(DECIDE, 1);
        for (int t = 0; t < n_tiles; ++t) {
          const int T = pass * n_tiles + t;
          // the softmax has read S(T - 3): its buffer takes S(T)
          if (t >= 3) mbar_wait(SFREE(T), par3(T - 3));
          const uint32_t ts = tmem + C::kSStride * (T % 3);
          if (t < n_pre) {
            const int TL = pass * n_pre + t, s = TL % kS;
            mbar_wait(FULLK(s), parS(TL));
            tc_fence_after();
            const uint64_t dk = dK0 + static_cast<uint64_t>((s * kKV) >> 4);
            if (elect_one()) {
#pragma unroll
              for (int kk = 0; kk < 8; ++kk)
                umma(ts, dk + (((kk >> 2) * kHalf + (kk & 3) * 32) >> 4),
                     dQ + (((kk >> 2) * C::kQHalf + (kk & 3) * 32) >> 4), kIdescS, kk > 0 ? 1 : 0);
              umma_commit(SREADY(T));
            }
          } else {
            tc_fence_after();
            if (elect_one()) {
#pragma unroll
              for (int kk = 0; kk < 8; ++kk)
                umma(ts, dN + (((kk >> 2) * kNewHalf + (kk & 3) * 32) >> 4),
                     dQ + (((kk >> 2) * C::kQHalf + (kk & 3) * 32) >> 4), kIdescS, kk > 0 ? 1 : 0);
              umma_commit(SREADY(T));
            }
          }
          __syncwarp();
        }
      }
    }
    __syncwarp();
    if (!arrived && csize > 1) cluster_arrive_relaxed();
    mbar_wait(TMEMDONE, 0);  // every softmax warp has read its last column
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::kTmemCols) : "memory");
    if (csize > 1) cluster_wait();
  } else if (warp == 2) {
    // -------------------------------------------------------------- PV issue
    bool arrived = false;
    if (n_tiles > 0) {
      const uint64_t dV0 = umma_desc(base + C::kRingV, kHalf, 1024);              // V^T: MN-major
      const uint64_t dN = umma_desc(base + C::kOffNewV, kNewHalf, 1024);
      const uint64_t dP0 = umma_desc(base + C::kOffP, C::kPGroup, 256, 6);        // P^T: MN-major, 32-byte swizzle
      const int new_steps = (a.R + 15) / 16;
      for (int pass = 0; pass < 3; ++pass) {
        if (pass == 1) {
          if (csize > 1) cluster_arrive_relaxed();
          arrived = true;
          mbar_wait(DECIDE, 0);
          if (!*reinterpret_cast<volatile int*>(s_redo)) break;
        }
        if (pass == 2) mbar_wait(DECIDE, 1);
        for (int t = 0; t < n_tiles; ++t) {
          const int T = pass * n_tiles + t;
          mbar_wait(PFULL(T), (T >> 1) & 1);
          const uint64_t dp = dP0 + static_cast<uint64_t>(((T & 1) * C::kP) >> 4);
          if (t < n_pre) {
            const int TL = pass * n_pre + t, s = TL % kS;
            mbar_wait(FULLV(s), parS(TL));
            tc_fence_after();
            const uint64_t dv = dV0 + static_cast<uint64_t>((s * kKV) >> 4);
            if (elect_one()) {
#pragma unroll
              for (int kk = 0; kk < 8; ++kk)
                umma(tmem_o, dv + (kk * 2048 >> 4), dp + (kk * 512 >> 4), kIdescO, (t > 0 || kk > 0) ? 1 : 0);
              umma_commit(PVDONE(T));
            }
          } else {
            tc_fence_after();
            if (elect_one()) {
#pragma unroll
              for (int kk = 0; kk < kMaxNew / 16; ++kk)
                if (kk < new_steps)
                  umma(tmem_o, dN + (kk * 2048 >> 4), dp + (kk * 512 >> 4), kIdescO, (t > 0 || kk > 0) ? 1 : 0);
              umma_commit(PVDONE(T));
            }
          }
          __syncwarp();
        }
      }
    }
    __syncwarp();
    if (!arrived && csize > 1) cluster_arrive_relaxed();
    if (csize > 1) cluster_wait();
  } else {
    // -------------------------------------------------------------- softmax
    const int group = (warp - kFirstSoft) >> 3;
    const int half = ((warp - kFirstSoft) >> 2) & 1;  // rows kRpt * half .. + kRpt - 1 of the group's tile
    const int quarter = warp & 3;                     // TMEM lane quarter of this warp
    const int kl = quarter * 32 + lane;               // key lane of S^T / d lane of O^T
    const uint32_t lane_off = static_cast<uint32_t>(quarter * 32) << 16;
    const int row0 = kRpt * half;
    const float2* cs_tab = reinterpret_cast<const float2*>(smem + C::kOffP);
    {
      // The rows, rotated (fused) and into the operand layouts. Iteration 0 runs
      // BEFORE the dependency wait on whatever the rows hold: it brings this
      // code into the instruction cache and the rows into L2, and iteration 1
      // overwrites everything it stored (.cg loads: no stale L1 line). The
      // cluster launched last starts when the previous kernel is nearly done:
      // no warm-up pass.
      const bool last_cluster = blockIdx.y == gridDim.y - 1 && blockIdx.z == gridDim.z - 1;
      const bool has_kv = raw_kv && valid;
      const long long cache_row =
          ((static_cast<long long>(b) * a.Hkv + kvh) * a.cap + L_pre + (st >> 4)) * kD + (st & 15) * 8;
#pragma unroll 1
      for (int it = early && !last_cluster ? 0 : 1; it < 2; ++it) {
        if (it == 1 && early) griddep_wait();
        uint4 qv[kQc], kv = make_uint4(0, 0, 0, 0), vv = make_uint4(0, 0, 0, 0);
#pragma unroll
        for (int u = 0; u < kQc; ++u) {
          const int idx = st + u * kSoftThreads, p = mblock * kR + (idx >> 4);
          if (rows_first)
            qv[u] = valid ? pre_q[u] : make_uint4(0, 0, 0, 0);
          else
            qv[u] = valid && idx < kR * 16 && p < a.M
                        ? __ldcg(reinterpret_cast<const uint4*>((kFused ? a.qw : a.q) + q_off(p) + (idx & 15) * 8))
                        : make_uint4(0, 0, 0, 0);
        }
        if (has_kv) {
          if (rows_first) {
            kv = pre_k;
            vv = pre_v;
          } else {
            kv = __ldcg(reinterpret_cast<const uint4*>(kFused ? a.k_new + kv_row : a.kc + cache_row));
            vv = __ldcg(reinterpret_cast<const uint4*>(kFused ? a.v_new + kv_row : a.vc + cache_row));
          }
        }
#pragma unroll
        for (int u = 0; u < kQc; ++u) {
          const int idx = st + u * kSoftThreads, row = idx >> 4, c = idx & 15, p = mblock * kR + row;
          if (idx >= kR * 16) break;
          uint32_t w[4] = {qv[u].x, qv[u].y, qv[u].z, qv[u].w};
          if (kFused && p < a.M) {
            const float2* cs = cs_tab + gdiv(p) * 64 + c * 4;
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = sd_rope_pair(w[j], cs[j].x, cs[j].y);
          }
          st_shared_v4(qs + (c >> 3) * C::kQHalf + row * 128 + (((c & 7) ^ (row & 7)) << 4), w[0], w[1], w[2], w[3]);
        }
        if (last_rank) {
          // new key (rotated) and value rows, zero past R
          const int i = st >> 4, c = st & 15;
          uint32_t w[4] = {kv.x, kv.y, kv.z, kv.w};
          if (kFused && has_kv) {
            const float2* cs = cs_tab + i * 64 + c * 4;
#pragma unroll
            for (int j = 0; j < 4; ++j) w[j] = sd_rope_pair(w[j], cs[j].x, cs[j].y);
          }
          const uint32_t off = (c >> 3) * kNewHalf + i * 128 + (((c & 7) ^ (i & 7)) << 4);
          st_shared_v4(base + C::kOffNewK + off, w[0], w[1], w[2], w[3]);
          st_shared_v4(base + C::kOffNewV + off, vv.x, vv.y, vv.z, vv.w);
          if (kFused && has_kv && it == 1 && mblock == 0) {
            // the append: cache rows L_pre .. L_pre + R - 1, which no CTA of
            // this launch reads; and, when this cluster alone reads the head's
            // raw key rows, their rotation in place
            *reinterpret_cast<uint4*>(a.kc + cache_row) = make_uint4(w[0], w[1], w[2], w[3]);
            *reinterpret_cast<uint4*>(a.vc + cache_row) = vv;
            if (a.n_mblocks == 1) *reinterpret_cast<uint4*>(a.k_new + kv_row) = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
      }
      // row p = i * G + g is new row i: it sees new keys 0..i (all R under the block mask)
      if (st < kR) {
        row_lim[st] = block ? a.R - 1 : min(gdiv(mblock * kR + st), a.R - 1);
        row_nref[st] = 0.f;
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      named_bar_sync(2, kSoftThreads);  // Q is complete; the rotation table is no longer read
      if (st == 0) {
        mbar_arrive(QFULL);
        griddep_launch();  // every older kernel has finished: the next layer may launch
        // with several m-blocks the head's raw key rows are read by the last
        // rank of each: the last of them writes the rotated rows back (the
        // fence orders this CTA's reads before its ticket)
        if (kFused && has_new && a.n_mblocks > 1) {
          __threadfence();
          *s_kvlast = atomicAdd(&a.kv_ticket[b * a.Hkv + kvh], 1u) == static_cast<uint32_t>(a.n_mblocks - 1);
        }
      }
    }

    const float sl = a.scale_log2;
    const uint64_t sl2 = pack2f(sl, sl);
    uint64_t lp2[kRpt / 2];  // this key lane's row sums, in pairs
    const uint32_t pbuf = base + C::kOffP + group * C::kP;
    const uint32_t pkey = pbuf + kl * 32;
    const uint32_t psw = (kl >> 2) & 1;  // 32-byte swizzle
    // this thread's rows j0 .. j0 + kN - 1 of tile T (its scores in buffer T % 3)
    // to weights and P; `last`: the tile's scores are all in registers then
    auto chunk = [&](auto kn, int T, int j0, bool last, bool wait_pv, auto keep) {
      constexpr int kN = decltype(kn)::value;
      uint32_t r[kN], pw[kN / 2];
      tmem_ld(tmem + C::kSStride * (T % 3) + row0 + j0 + lane_off, r);
      if (last) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(SFREE(T));
      }
      weights_to_p<kN>(r, row_nref + row0 + j0, sl2, keep, lp2 + j0 / 2, pw);
      if (wait_pv && T >= 2) mbar_wait(PVDONE(T - 2), parS(T - 2));  // PV(T - 2) has read the buffer
#pragma unroll
      for (int h = 0; h < kN / 8; ++h) {
        const int ch = (row0 + j0) / 8 + h;
        st_shared_v4(pkey + (ch >> 1) * C::kPGroup + (((ch & 1) ^ psw) << 4), pw[4 * h], pw[4 * h + 1], pw[4 * h + 2],
                     pw[4 * h + 3]);
      }
    };
    auto tile_p = [&](int T, auto keep) {
#pragma unroll
      for (int j0 = 0; j0 + 16 <= kRpt; j0 += 16)
        chunk(std::integral_constant<int, 16>{}, T, j0, j0 + 16 == kRpt, j0 == 0, [&](int j, uint32_t w) { return keep(j0 + j, w); });
      if constexpr (kRpt % 16 != 0)
        chunk(std::integral_constant<int, 8>{}, T, kRpt - 8, true, false, [&](int j, uint32_t w) { return keep(kRpt - 8 + j, w); });
    };
    bool seen = false;  // this warp has had a key of its own (every row sees prefix keys and new key 0)
    auto run_pass = [&](int pass) {
#pragma unroll
      for (int j = 0; j < kRpt / 2; ++j) lp2[j] = 0ull;
      for (int t = ((pass * n_tiles) ^ group) & 1; t < n_tiles; t += 2) {
        const int T = pass * n_tiles + t;
        mbar_wait(SREADY(T), par3(T));
        tc_fence_after();
        if (t < n_pre) {
          const int key0 = key_begin + t * kStageKeys;
          const bool key_ok = key0 + kl < key_end;
          seen |= key0 + quarter * 32 < key_end;
          tile_p(T, [&](int, uint32_t w) { return key_ok ? w : 0u; });
          if (!key_ok) {
            // stale or foreign key row: zero its V row (this thread's 64-column
            // half) so 0 * NaN cannot reach O, once the tile has landed
            const int TL = pass * n_pre + t, s = TL % kS;
            mbar_wait(FULLV(s), parS(TL));
            const uint32_t vrow = base + C::kRingV + s * kKV + half * kHalf + kl * 128;
#pragma unroll
            for (int c = 0; c < 8; ++c) st_shared_v4(vrow + c * 16, 0u, 0u, 0u, 0u);
          }
        } else if (quarter == 0) {
          seen = true;
          tile_p(T, [&](int j, uint32_t w) {
            const int2 lim = *reinterpret_cast<const int2*>(row_lim + row0 + j);
            return w & ((kl <= lim.x ? 0xffffu : 0u) | (kl <= lim.y ? 0xffff0000u : 0u));
          });
        } else {
          // key lanes past the new keys: nothing to read or write
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(SFREE(T));
          if (T >= 2) mbar_wait(PVDONE(T - 2), parS(T - 2));
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(PFULL(T));
      }
    };
    // row sums over this warp's keys to row_sum; whether one of them left the
    // range that a single reference-free pass is exact in
    auto sum_rows = [&]() {
      bool out_of_range = false;
#pragma unroll
      for (int j0 = 0; j0 < kRpt; j0 += 8) {
        float v[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) unpack2(lp2[j0 / 2 + j], v[2 * j], v[2 * j + 1]);
        const float x = warp_sum8(v, lane);
        out_of_range |= x > kHigh || (seen && x < kLow);
        if ((lane & 3) == 0) row_sum[(row0 + j0 + (lane >> 2)) * 8 + group * 4 + quarter] = x;
      }
      return out_of_range;
    };
    run_pass(0);
    bool bad = sum_rows();
    const bool redo = named_bar_or(2, kSoftThreads, bad) && n_tiles > 0;
    if (redo) mbar_wait(PVDONE(n_tiles - 1), parS(n_tiles - 1));
    if (st == 0) {
      *s_redo = redo ? 1 : 0;
      mbar_arrive(DECIDE);
    }
    if (redo) {
      // pass 1: every row's exact maximum over this CTA's keys (the PV products
      // run on stale weights, their sums are dropped by pass 2)
      float mx[kRpt];
#pragma unroll
      for (int j = 0; j < kRpt; ++j) mx[j] = -INFINITY;
#pragma unroll 1
      for (int t = (n_tiles ^ group) & 1; t < n_tiles; t += 2) {
        const int T = n_tiles + t;
        mbar_wait(SREADY(T), par3(T));
        tc_fence_after();
        const bool is_new = t >= n_pre;
        const bool key_ok = is_new ? quarter == 0 : key_begin + t * kStageKeys + kl < key_end;
#pragma unroll
        for (int j0 = 0; j0 < kRpt; j0 += 8) {
          uint32_t r[8];
          tmem_ld(tmem + C::kSStride * (T % 3) + row0 + j0 + lane_off, r);
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (key_ok && (!is_new || kl <= row_lim[row0 + j0 + j]))
              mx[j0 + j] = fmaxf(mx[j0 + j], __uint_as_float(r[j]) * sl);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(SFREE(T));
        mbar_wait(PVDONE(T - 2 < 0 ? 0 : T - 2), parS(T - 2 < 0 ? 0 : T - 2));
        if (lane == 0) mbar_arrive(PFULL(T));
      }
      named_bar_sync(2, kSoftThreads);
      mbar_wait(PVDONE(2 * n_tiles - 1), parS(2 * n_tiles - 1));
      float* rb = reinterpret_cast<float*>(smem + C::kOffP);
      if (group == 0)
#pragma unroll
        for (int j = 0; j < kRpt; ++j) rb[(row0 + j) * 128 + kl] = mx[j];
      named_bar_sync(2, kSoftThreads);
      if (group == 1)
#pragma unroll
        for (int j = 0; j < kRpt; ++j) rb[(row0 + j) * 128 + kl] = fmaxf(rb[(row0 + j) * 128 + kl], mx[j]);
      named_bar_sync(2, kSoftThreads);
#pragma unroll 1
      for (int row = warp - kFirstSoft; row < kR; row += kSoftWarps) {
        const float4 x = reinterpret_cast<const float4*>(rb + row * 128)[lane];
        float m = fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) row_nref[row] = m == -INFINITY ? 0.f : -m;
      }
      named_bar_sync(2, kSoftThreads);
      if (st == 0) mbar_arrive(DECIDE);
      run_pass(2);
      sum_rows();
      named_bar_sync(2, kSoftThreads);
    }
    // ---- every row sum of this CTA is in row_sum, the last S product is done
    // (both groups have seen their last tile's): the K ring may receive
    const bool merge = csize > 1;
    if (merge) cluster_arrive_relaxed();
    if (n_tiles > 0) {
      const int Tl = (redo ? 3 : 1) * n_tiles - 1;
      mbar_wait(PVDONE(Tl), parS(Tl));
      tc_fence_after();
    }
    // O: this warp reads its 32 d lanes of a quarter of the rows
    constexpr int kOr = kR / 4;
    const int orow0 = (group * 2 + half) * kOr;
    uint32_t o[kOr];
    if (n_tiles > 0) {
      uint32_t x8[8];
      tmem_ld(tmem_o + orow0 + lane_off, x8);
#pragma unroll
      for (int j = 0; j < 8; ++j) o[j] = x8[j];
      if constexpr (kOr >= 16) {
        tmem_ld(tmem_o + orow0 + 8 + lane_off, x8);
#pragma unroll
        for (int j = 0; j < 8; ++j) o[8 + j] = x8[j];
      }
      if constexpr (kOr % 8 != 0) {
        uint32_t x4[4];
        tmem_ld(tmem_o + orow0 + kOr - 4 + lane_off, x4);
#pragma unroll
        for (int j = 0; j < 4; ++j) o[kOr - 4 + j] = x4[j];
      }
    } else {
#pragma unroll
      for (int j = 0; j < kOr; ++j) o[j] = 0u;
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(TMEMDONE);
    if (!merge) {
      // one CTA holds the head's keys: normalise and store (64 bytes a row and warp)
#pragma unroll
      for (int j = 0; j < kOr; ++j) {
        const int row = orow0 + j, p = mblock * kR + row;
        const float4 l0 = reinterpret_cast<const float4*>(row_sum + row * 8)[0];
        const float4 l1 = reinterpret_cast<const float4*>(row_sum + row * 8)[1];
        const float l = ((l0.x + l0.y) + (l0.z + l0.w)) + ((l1.x + l1.y) + (l1.z + l1.w));
        if (valid && p < a.M && l > 0.f) a.out[q_off(p) + kl] = __float2bfloat16_rn(__uint_as_float(o[j]) * (1.f / l));
      }
    } else {
      float* send = reinterpret_cast<float*>(smem + C::kRingV);
#pragma unroll
      for (int j = 0; j < kOr; ++j) send[(orow0 + j) * kRowF + kl] = __uint_as_float(o[j]);
      for (int idx = st; idx < kR * 8; idx += kSoftThreads) send[(idx >> 3) * kRowF + kRowL + (idx & 7)] = row_sum[idx];
      if (st < kR) send[st * kRowF + kRowM] = -row_nref[st];
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      named_bar_sync(2, kSoftThreads);
      if (st == 0) mbar_expect_tx(RECV, static_cast<uint32_t>(csize * my_rows * kRowBytes));
      cluster_wait();  // every peer's K ring is free to receive
      // softmax warp w sends rank w's rows to it, into its slots [rank * rpc, ...)
      if (elect_one()) {
        const int c = warp - kFirstSoft;
        if (c < csize && rows_of(c) > 0)
          bulk_copy_s2s(cluster_map(base + rank * rpc * kRowBytes, c), base + C::kRingV + c * rpc * kRowBytes,
                        static_cast<uint32_t>(rows_of(c) * kRowBytes), cluster_map(RECV, c));
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
      __syncwarp();
    }
    if (kFused && valid) {
      // while the partials travel: every CTA of the cluster has read the raw
      // rows (its tiles came after), so the rotated query rows this CTA merges
      // go back to q, and with several m-blocks the head's last reader of the
      // raw key rows writes the rotated ones back to k_new
#pragma unroll 1
      for (int idx = st; idx < my_rows * 16; idx += kSoftThreads) {
        const int row = mrow0 + (idx >> 4), c = idx & 15, p = mblock * kR + row;
        if (p >= a.M) continue;
        *reinterpret_cast<uint4*>(a.qw + q_off(p) + c * 8) = *reinterpret_cast<const uint4*>(
            smem + C::kOffQ + (c >> 3) * C::kQHalf + row * 128 + (((c & 7) ^ (row & 7)) << 4));
      }
      if (last_rank && a.n_mblocks > 1 && *s_kvlast != 0) {
        if (st < a.R * 16) {
          const int i = st >> 4, c = st & 15;
          *reinterpret_cast<uint4*>(a.k_new + kv_row) = *reinterpret_cast<const uint4*>(
              smem + C::kOffNewK + (c >> 3) * kNewHalf + i * 128 + (((c & 7) ^ (i & 7)) << 4));
        }
        if (st == 0) a.kv_ticket[b * a.Hkv + kvh] = 0;  // re-armed
      }
    }
    if (merge) {
      // ---- merge of the rows this CTA owns, a warp a row, four d a lane; slot
      // c * rpc + r came from rank c. Unless some rank ran its range again all
      // references are 0 and the partials add.
      mbar_wait(RECV, 0);
      const float* recv = reinterpret_cast<const float*>(smem);
#pragma unroll 1
      for (int r = warp - kFirstSoft; r < my_rows; r += kSoftWarps) {
        const float* part = recv + r * kRowF;
        float4 ov = make_float4(0.f, 0.f, 0.f, 0.f);
        float l = 0.f;
        bool same = true;
#pragma unroll 4
        for (int c = 0; c < csize; ++c) {
          const float* pc = part + c * rpc * kRowF;
          const float4 x = reinterpret_cast<const float4*>(pc)[lane];
          const float4 l0 = *reinterpret_cast<const float4*>(pc + kRowL);
          const float4 l1 = *reinterpret_cast<const float4*>(pc + kRowL + 4);
          same = same && pc[kRowM] == 0.f;
          ov.x += x.x, ov.y += x.y, ov.z += x.z, ov.w += x.w;
          l += ((l0.x + l0.y) + (l0.z + l0.w)) + ((l1.x + l1.y) + (l1.z + l1.w));
        }
        if (!same) {
          // weigh every partial by its own reference (those without a key count for nothing)
          float m = -INFINITY;
          ov = make_float4(0.f, 0.f, 0.f, 0.f);
          l = 0.f;
#pragma unroll 1
          for (int pass = 0; pass < 2; ++pass)
#pragma unroll 1
            for (int c = 0; c < csize; ++c) {
              const float* pc = part + c * rpc * kRowF;
              float lc = 0.f;
              for (int e = 0; e < 8; ++e) lc += pc[kRowL + e];
              if (!(lc > 0.f)) {
                if (lc != lc) l = lc;  // NaN reaches the row
                continue;
              }
              if (pass == 0) {
                m = fmaxf(m, pc[kRowM]);
                continue;
              }
              const float w = ex2(pc[kRowM] - m);
              const float4 x = reinterpret_cast<const float4*>(pc)[lane];
              ov.x = fmaf(w, x.x, ov.x), ov.y = fmaf(w, x.y, ov.y), ov.z = fmaf(w, x.z, ov.z), ov.w = fmaf(w, x.w, ov.w);
              l = fmaf(w, lc, l);
            }
        }
        const int p = mblock * kR + mrow0 + r;
        if (valid && p < a.M && l > 0.f) {
          const float inv_l = 1.f / l;
          *reinterpret_cast<uint2*>(a.out + q_off(p) + lane * 4) =
              make_uint2(cvt_bf16x2(ov.x * inv_l, ov.y * inv_l), cvt_bf16x2(ov.z * inv_l, ov.w * inv_l));
        }
      }
      if (elect_one()) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      __syncwarp();
    }
  }
  // no CTA-wide barrier at the end: every warp leaves when its own work is done
}

// ------------------------------------------------------------------ host
template <int kR>
bool set_attributes(const int* sizes, int n, int* active) {
  const void* kerns[3] = {reinterpret_cast<const void*>(verify_wide_kernel<kR, 1>),
                          reinterpret_cast<const void*>(verify_wide_kernel<kR, 2>),
                          reinterpret_cast<const void*>(verify_wide_kernel<kR, 3>)};
  constexpr int smem = Cfg<kR>::kSmemBytes;
  for (const void* k : kerns)
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess ||
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      (void)cudaGetLastError();
      return false;
    }
  for (int i = 0; i < n; ++i) {
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = sizes[i];
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(sizes[i], 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int m = 0;
    if (cudaOccupancyMaxActiveClusters(&m, kerns[1], &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      m = 0;
    }
    active[i] = m;
  }
  return true;
}

template <int kR, int kMode>
sd_status launch(const sd_kv_cache* cache, const TcArgs& a, const RopeTable& tab, int cs, cudaStream_t stream) {
  const int B = cache->batch, Hkv = cache->n_kv_heads, cap = cache->capacity;
  CUtensorMap k128, v128;
  if (!make_map(&k128, cache->k, cap, B * Hkv, 128) || !make_map(&v128, cache->v, cap, B * Hkv, 128))
    return SD_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cs;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(cs, Hkv * a.n_mblocks, B);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = Cfg<kR>::kSmemBytes;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, verify_wide_kernel<kR, kMode>, k128, v128, a, tab) != cudaSuccess) {
    (void)cudaGetLastError();
    return SD_ERR_CUDA;
  }
  return SD_OK;
}

template <int kMode>
sd_status launch_rows(const sd_kv_cache* cache, const TcArgs& a, const RopeTable& tab, int rows, int cs,
                      cudaStream_t stream) {
  if (rows == 48) return launch<48, kMode>(cache, a, tab, cs, stream);
  if (rows == 64) return launch<64, kMode>(cache, a, tab, cs, stream);
  return launch<80, kMode>(cache, a, tab, cs, stream);
}

}  // namespace

bool sd_internal_wide_active(int rows, const int* sizes, int n, int* active) {
  if (rows == 48) return set_attributes<48>(sizes, n, active);
  if (rows == 64) return set_attributes<64>(sizes, n, active);
  return set_attributes<80>(sizes, n, active);
}

sd_status sd_internal_wide_launch(const sd_kv_cache* cache, const TcArgs& a, const RopeTable& tab, int rows, int cs,
                                  int mode, cudaStream_t stream) {
  if (mode == 1) return launch_rows<1>(cache, a, tab, rows, cs, stream);
  if (mode == 2) return launch_rows<2>(cache, a, tab, rows, cs, stream);
  return launch_rows<3>(cache, a, tab, rows, cs, stream);
}
