// The verify attention and the fused verify layer (Eq. verify, Sec. 3.2; the
// rotations of Sec. 3.3 / 4.2, the append of Eq. commit) for up to 31 new rows (the
// attention of one query head a KV head: 32), head dim 128 and (the attention) 64, on
// the 5th-generation tensor cores (tcgen05 + TMEM).
//
// The packed query rows of a KV head (G * R) are few, so both products run
// transposed, the 128-wide dimension on the MMA's M side:
//     S^T[128 keys][kR rows] = K_tile . Q^T,   O^T[128 d][kR rows] += V_tile^T . P^T
// with kR = 32, 48, 64 or 80, the smallest that holds the rows in one tile (two
// m-blocks of 48 or 64 above 80): a K = 16 block of the 8B target (68 rows) reads
// every key once. One cluster per (scene, KV head, m-block); its CTAs take
// contiguous ranges of the prefix and merge their partials through distributed
// shared memory.
//
// What bounds it. With many scenes the stream of K and V (32 scenes, L = 8192: K = 7
// 153 -> 142 us, K = 8 165 -> 143, 1.0 of the measured copy). With one scene the
// dependent path behind the previous kernel: rows, rotation, S(0), the tiles at
// ~0.4 us of products each, the exchange (~0.7 us), the merge (target layer
// 6.77 -> 6.42 us, K = 8 10.0 -> 7.5, K = 16 block 15.9 -> 10.6, draft step 6.8 -> 6.1
// on one cache).
//
// Head dim 64 (the attention; its layers run as the rotation, append and attention
// kernels) is the same kernel with half rows and 16-bit weights: 5 scenes, 28 query
// heads on 4, L = 4099, K = 5: 15.3 -> 8.9 us against the mma.sync kernel, the tiny
// layer's 256 keys 7.3 -> 4.3.
//
// The new rows stay out of the loop: the cluster's last rank holds the R (rotated)
// new keys and values in shared memory, scores them by mma.sync, 8 rows by 16 keys a
// warp, and adds one PV product of 16 or 32 keys, its weights to 16 bits in two bf16
// terms: with one term the error at an empty prefix was 2.1e-3 against the 1.66e-3 of
// the output's rounding. Scored on the CUDA cores by the rows a CTA merges instead,
// rows x new keys took 26 us a launch at one CTA a head and K = 16.
//
// Fixed reference. Weights are 2^(score * scale - ref) with the row's score against its
// own new key as its reference on every CTA of the cluster: the row's sum is about 1 or
// more, scores may have any common offset, and the CTAs' partials add as they are. (Both
// turn by the same angles, in registers, on the way to shared memory: nothing stands
// between S and P. Their score before the rotation would do but for its rounding to
// bf16, which underflows every weight at scores of 1e4; it saved 0.07 us a layer.) A
// floating-point weight keeps its relative precision at any size, so only overflow
// matters: a row sum above 2^64 sends the CTA through its range again with each row's
// exact maximum as its reference, one pass for the maxima and one for the weights. Without a reference scores 40 away from 0 took
// those passes (8 scenes, L = 8192, K = 7: 38 -> 102 us), and values far from 1 left
// fp32's range in the product; the references cost 0.1 to 0.2 us a layer.
//
// Warps (608 threads): 0 the TMA producer, whose first tiles go out before the CTA's
// set-up is over; 1 issues S and owns tensor memory; 2 issues PV; 3..18 two softmax
// groups of eight. Group g takes tiles T with T % 2 == g and P buffer g, so a group
// has two tiles' time for its tile's dependent chain (barrier wake-up,
// tensor-memory load, exponentials, stores: ~800 cycles on 32 rows) while the other
// group's tile is in the products. With one group of eight on every tile that chain
// set the pace: ~1.1 us a 128-key tile of 64 rows. fma on pairs (f32x2) and a select
// on the packed weights take about 5 issue slots a weight instead of ~9.5.
#include "tc_common.cuh"

#include <math.h>

#include <type_traits>

SD_DEFINE_ERROR_ACCESSOR(sd_take_error_attention_wide)

namespace {

constexpr int kStageKeys = 128;
constexpr int kHalf = kStageKeys * 128;  // one 64-column half of a 128-key tile (16 KB)
constexpr int kSoftWarps = 16;
constexpr int kSoftThreads = 32 * kSoftWarps;
constexpr int kFirstSoft = 3;            // the first softmax warp
constexpr int kSoft0 = 32 * kFirstSoft;  // the first softmax thread
constexpr int kThreads = kSoft0 + kSoftThreads;
constexpr float kHigh = 18446744073709551616.f;          // 2^64: a larger row sum runs the range again
template <int kR, int kDim, bool kSplitWeights>
struct Cfg {
  static_assert(kR == 32 || kR == 48 || kR == 64 || kR == 80, "row tile");
  static_assert(kDim == 64 || kDim == 128, "head dim");
  static constexpr int kRpt = kR / 2;                   // rows of a softmax thread in its tile
  static constexpr int kHalves = kDim / 64;             // 64-column halves of a row
  static constexpr int kChunks = kDim / 8;              // 16-byte chunks of a row
  static constexpr int kKV = kHalves * kHalf;           // one K (or V) tile of 128 keys
  // K slots, and V slots: at most 3, as the producer's wait for S(T - kStages) must see
  // its phase before S(T - kStages + 3) completes the next one of that S buffer
  static constexpr int kStages = kDim == 64 || kR == 32 ? 3 : 2;
  static constexpr int kMaxNew = kR == 32 ? 16 : 32;    // new rows held in shared memory
  static constexpr int kNewHalf = kMaxNew * 128;        // one 64-column half of the new key (value) rows
  static constexpr int kRingV = kStages * kKV;
  static constexpr int kRing = 2 * kStages * kKV;
  static constexpr int kQHalf = kR * 128;
  // P^T is MN-major with the 32-byte swizzle: 16 rows x 8 keys an atom, the
  // 16-row groups kPGroup apart
  static constexpr int kPGroup = kStageKeys * 32;
  static constexpr int kP = (kR / 16) * kPGroup;
  // whether the weights are kept to 16 bits as two bf16 terms (two PV products). Head
  // dim 64 is: the mma.sync kernel that served it rounds weights below a running maximum,
  // which is 14% closer to 64 bits than one term without a reference (2.1e-3 against
  // 2.4e-3). So are 17 to 32 packed rows of a query head each at head dim 128, which ran
  // with their first tile's maximum as reference (largest weight exact: 1.8e-3 against
  // 2.1e-3 at a prefix of one tile)
  static constexpr bool kSplit = kSplitWeights;
  static constexpr int kPBuf = kSplit ? 2 * kP : kP;  // a group's P buffer: the high terms, then the low ones
  static constexpr int kSStride = kR == 32 ? 32 : (kR <= 64 ? 64 : 128);  // columns between S0 | S1 | S2 | O
  static constexpr int kTmemCols = 4 * kSStride;
  // shared memory (offsets from the 1024-aligned base)
  static constexpr int kOffNewK = kRing;
  static constexpr int kOffNewV = kOffNewK + kHalves * kNewHalf;
  static constexpr int kOffQ = kOffNewV + kHalves * kNewHalf;
  static constexpr int kOffP = kOffQ + kHalves * kQHalf;
  // the new keys' weights: on the 32-row tile, which has no room for more, in P
  // buffer 1 ahead of its first tile; on the others beside it, in the same layout
  static constexpr bool kNewFirst = kR == 32;
  static constexpr int kOffPNew = kOffP + (kNewFirst ? kPBuf : 2 * kPBuf);
  static constexpr int kPNewGroup = kNewFirst ? kPGroup : kMaxNew * 32;
  // from the high to the low terms (two for head dim 128 too: these weights were fp32 where
  // the new keys were merged on the CUDA cores): in P buffer 1 the 16 keys after the 16 new ones
  static constexpr int kPNewLow = kNewFirst ? kMaxNew * 32 : (kR / 16) * kPNewGroup;
  static constexpr int kOffBar = kNewFirst ? kOffP + 2 * kPBuf : kOffPNew + 2 * kPNewLow;
  // full_k[S] full_v[S] p_full[2] s_ready[3] s_free[3] pv_done[S] p_new new_done recv decide maxima tmem_done
  static constexpr int kNumBars = 3 * kStages + 14;
  static constexpr int kOffMisc = round_up(kOffBar + kNumBars * 8, 16);
  static constexpr int kOffRef = kOffMisc + 16;        // [kR] negated references
  static constexpr int kOffNewSum = kOffRef + kR * 4;  // [kR] row sums of the new keys
  static constexpr int kOffSum = kOffNewSum + kR * 4;  // [kR][8] row sums by group and lane quarter
  static constexpr int kSmemBytes = kOffSum + kR * 32 + 1024;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory budget");
  static_assert(kOffNewV % 1024 == 0 && kOffQ % 1024 == 0 && kOffP % 1024 == 0 && kQHalf % 1024 == 0, "swizzle atoms");
  static_assert(kMaxNew * (kDim / 2) * 8 <= 2 * kP, "rotation table fits the P buffers");
  static_assert(kR * 128 * 4 <= 2 * kP, "row maxima fit the P buffers");
  // a partial row sent to its owner: [O(kDim) | prefix row sums by softmax group and
  // lane quarter (8) | reference | new keys' row sum | 2 pad] fp32 (560 or 304 bytes)
  static constexpr int kRowL = kDim;
  static constexpr int kRowM = kDim + 8;
  static constexpr int kRowF = kDim + 12;
  static constexpr int kRowBytes = kRowF * 4;
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

// Two weights as bf16 terms: the high ones, and with kSplit what rounding left.
// l: the weights that the terms stand for.
template <bool kSplit>
__device__ __forceinline__ void weight_terms(float e0, float e1, uint32_t& hi, uint32_t& lo, uint64_t& l) {
  hi = cvt_bf16x2(e0, e1);
  if (kSplit) {
    lo = cvt_bf16x2(e0 - sd_bf16_lo(hi), e1 - sd_bf16_hi(hi));
    l = pack2f(e0, e1);
  } else {
    l = pack2(hi << 16, hi & 0xffff0000u);
  }
}

// Weights of kN rows of one key: P = 2^(S * scale - ref) in bf16 terms (0 for a key
// out of the range, whatever its score, NaN included), the row sums advanced by the
// same weights.
template <int kN, bool kSplit>
__device__ __forceinline__ void weights_to_p(const uint32_t (&r)[kN], const float* nref, uint64_t sl2, bool key_ok,
                                             uint64_t* lp2, uint32_t (&pw)[kN / 2], uint32_t (&pl)[kN / 2]) {
#pragma unroll
  for (int j = 0; j < kN; j += 4) {
    const float4 nr = *reinterpret_cast<const float4*>(nref + j);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      float y0, y1;
      unpack2(fma2(pack2(r[j + 2 * e], r[j + 2 * e + 1]), sl2, e == 0 ? pack2f(nr.x, nr.y) : pack2f(nr.z, nr.w)), y0, y1);
      uint32_t hi, lo = 0;
      uint64_t l;
      if (kSplit) {
        weight_terms<true>(key_ok ? ex2(y0) : 0.f, key_ok ? ex2(y1) : 0.f, hi, lo, l);
      } else {
        hi = key_ok ? cvt_bf16x2(ex2(y0), ex2(y1)) : 0u;
        l = pack2(hi << 16, hi & 0xffff0000u);
      }
      pw[j / 2 + e] = hi;
      pl[j / 2 + e] = lo;
      lp2[j / 2 + e] = add2(lp2[j / 2 + e], l);
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

// C += A . B of one m16n8k16 bf16 product
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldmatrix4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
// The dot product of 8 bf16 pairs
__device__ __forceinline__ float dot8(const uint32_t (&x)[4], const uint32_t (&y)[4]) {
  auto dot2 = [](uint32_t a, uint32_t b) { return fmaf(sd_bf16_hi(a), sd_bf16_hi(b), sd_bf16_lo(a) * sd_bf16_lo(b)); };
  return (dot2(x[0], y[0]) + dot2(x[1], y[1])) + (dot2(x[2], y[2]) + dot2(x[3], y[3]));
}
// Byte offset of 16-byte chunk c of row r in a 128-byte-swizzled pair of
// 64-column halves, `half` bytes each.
__device__ __forceinline__ uint32_t swz(int r, int c, int half) {
  return (c >> 3) * half + r * 128 + (((c & 7) ^ (r & 7)) << 4);
}

// A row's largest score against the new keys it sees (the range is run again:
// out of line). One warp; qrow / krow0: the packed query row and new key row 0.
template <int kDim>
__device__ __noinline__ float new_key_max(const uint8_t* q, int row, int q_half, const uint8_t* k, int k_half, int last,
                                          float sl, int lane) {
  constexpr int kPer = kDim / 32;  // d a lane: 4 or 2
  const int c = lane * kPer / 8, e = lane * kPer % 8 * 2;
  const uint32_t* qw = reinterpret_cast<const uint32_t*>(q + swz(row, c, q_half) + e);
  float m = -INFINITY;
  for (int n = 0; n <= last; ++n) {
    const uint32_t* kw = reinterpret_cast<const uint32_t*>(k + swz(n, c, k_half) + e);
    float x = 0.f;
#pragma unroll
    for (int j = 0; j < kPer / 2; ++j) {
      x = fmaf(sd_bf16_lo(qw[j]), sd_bf16_lo(kw[j]), x);
      x = fmaf(sd_bf16_hi(qw[j]), sd_bf16_hi(kw[j]), x);
    }
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    m = fmaxf(m, x * sl);
  }
  return m;
}

// ------------------------------------------------------------------ kernel
// kFused: the verify layer (M-RoPE, append, attention); otherwise the attention
// over a cache that already holds the R new rows. Bit 0 of a.early: prefix, len
// and pos may be read before the dependency wait; bit 1: the block mask. Grid:
// (cluster size, Hkv * n_mblocks, B); m-block mb takes packed rows mb * kR ..
// mb * kR + kR - 1.
template <int kR, int kDim, bool kFused, bool kSplitWeights>
__global__ void __launch_bounds__(kThreads, 1)
    verify_wide_kernel(const __grid_constant__ CUtensorMap tm_k128, const __grid_constant__ CUtensorMap tm_v128,
                       const TcArgs a, const RopeTable tab) {
  using C = Cfg<kR, kDim, kSplitWeights>;
  constexpr int kHalves = C::kHalves, kChunks = C::kChunks, kKV = C::kKV;
  constexpr int kRowL = C::kRowL, kRowM = C::kRowM, kRowF = C::kRowF, kRowBytes = C::kRowBytes;
  constexpr int kS = C::kStages;
  constexpr int kRpt = C::kRpt;
  constexpr uint32_t kIdescS = umma_idesc(128, kR, 0, 0);
  constexpr uint32_t kIdescO = umma_idesc(128, kR, 1, 1);
  const bool early = (a.early & 1) != 0;
  const bool block = (a.early & 2) != 0;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const uint32_t base = smem_addr(smem);
  const uint32_t qs = base + C::kOffQ;
  auto bar = [&](int i) { return base + C::kOffBar + 8u * i; };
  // T counts the prefix tiles of all passes. A wait names a phase by its parity,
  // so a waiter has to know that the phase before has completed, and the next one
  // must not complete before it has looked: S(T + 3) and P(T + 2) follow the
  // softmax's waits for S(T) and PV(T), a K (V) slot's next tile the producer's
  // wait for its S (PV); a group that skips phases of a ring (it sees every second
  // tile) knows the skipped ones complete, as products complete in order; and
  // between passes everything is complete.
  auto FULLK = [&](int s) { return bar(s); };
  auto FULLV = [&](int s) { return bar(kS + s); };
  auto PFULL = [&](int T) { return bar(2 * kS + (T & 1)); };
  auto SREADY = [&](int i) { return bar(2 * kS + 2 + i); };  // i = T % 3
  auto SFREE = [&](int i) { return bar(2 * kS + 5 + i); };
  auto PVDONE = [&](int i) { return bar(2 * kS + 8 + i); };  // i = T % kS
  const uint32_t PNEW = bar(3 * kS + 8);      // the new keys' weights are stored
  const uint32_t NEWDONE = bar(3 * kS + 9);   // their product is done
  const uint32_t RECV = bar(3 * kS + 10);
  const uint32_t DECIDE = bar(3 * kS + 11);   // whether the range runs again
  const uint32_t MAXIMA = bar(3 * kS + 12);   // pass 1 is over
  const uint32_t TMEMDONE = bar(3 * kS + 13);
  auto par3 = [](int T) { return static_cast<uint32_t>((T / 3) & 1); };
  auto parS = [](int T) { return static_cast<uint32_t>((T / kS) & 1); };
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C::kOffMisc);
  int* s_redo = reinterpret_cast<int*>(smem + C::kOffMisc + 4);
  int* s_len = reinterpret_cast<int*>(smem + C::kOffMisc + 8);
  int* s_kvlast = reinterpret_cast<int*>(smem + C::kOffMisc + 12);
  float* row_nref = reinterpret_cast<float*>(smem + C::kOffRef);
  float* row_new = reinterpret_cast<float*>(smem + C::kOffNewSum);
  float* row_sum = reinterpret_cast<float*>(smem + C::kOffSum);

  auto gdiv = [&](int p) { return __float2int_rz((static_cast<float>(p) + 0.5f) * a.inv_g); };
  const int rank = blockIdx.x;
  const int csize = gridDim.x;
  const int kvh = blockIdx.y % a.Hkv;
  const int mblock = blockIdx.y / a.Hkv;
  const int b = blockIdx.z;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  // the launch's arguments come into the constant cache here, ahead of the wait
  // (a first touch behind it costs a round trip to L2 on the critical path)
  const float sl = a.scale_log2;
  asm volatile("" ::"f"(sl), "l"(a.out), "l"(a.ticket), "r"(a.cap), "r"(a.M));
  const bool last_rank = rank == csize - 1;
  // the cluster launched last starts when the previous kernel is nearly done
  const bool last_cluster = blockIdx.y == gridDim.y - 1 && blockIdx.z == gridDim.z - 1;

  // this CTA's share of a scene with len0 cached rows: the prefix in 32-key
  // blocks, split over the cluster's ranks
  int L_pre, key_begin, key_end, n_pre;
  bool valid;
  auto ranges = [&](int len0) {
    L_pre = kFused ? len0 : len0 - a.R;
    valid = L_pre >= 0 && L_pre + a.R <= a.cap;
    const int nblk = valid ? (L_pre + 31) / 32 : 0;
    const int blk_begin = static_cast<int>((static_cast<uint32_t>(rank) * nblk) / static_cast<uint32_t>(csize));
    const int blk_end = static_cast<int>((static_cast<uint32_t>(rank + 1) * nblk) / static_cast<uint32_t>(csize));
    key_begin = blk_begin * 32;
    key_end = min(blk_end * 32, valid ? L_pre : 0);
    n_pre = (blk_end - blk_begin + 3) / 4;  // prefix tiles
  };
  // keys of tile t that its PV product reads: whole 16-key steps up to the last key
  auto pv_keys = [&](int t) { return min(kStageKeys, (key_end - key_begin - t * kStageKeys + 15) & ~15); };

  // a launch without the early prefix waits before any global access: here, and the
  // softmax warps after a dry run of their set-up
  if (!early && warp < kFirstSoft) griddep_wait();

  if (warp == 0) {
    // -------------------------------------------------------------- producer
    // its first tiles are under way before the CTA-wide barrier
    const int len0 = a.len[b];  // the scene's length advances at this warp's end
    if (lane == 0) {
#pragma unroll 1
      for (int s = 0; s < kS; ++s) {
        mbar_init(FULLK(s), 1);
        mbar_init(FULLV(s), 1);
        mbar_init(PVDONE(s), 1);
      }
      for (int i = 0; i < 2; ++i) mbar_init(PFULL(i), kSoftWarps / 2);
#pragma unroll 1
      for (int i = 0; i < 3; ++i) {
        mbar_init(SREADY(i), 1);
        mbar_init(SFREE(i), kSoftWarps / 2);
      }
      mbar_init(PNEW, kR / 8);
      mbar_init(NEWDONE, 1);
      mbar_init(RECV, 1);
      mbar_init(DECIDE, 1);
      mbar_init(MAXIMA, 1);
      mbar_init(TMEMDONE, kSoftWarps);
      *s_redo = 0;
      *s_len = len0;
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    __syncwarp();
    ranges(len0);
    const int z = b * a.Hkv + kvh;
    const uint64_t evict_first = l2_evict_first_policy();
    auto issue_k = [&](int pass, int t) {
      const int T = pass * n_pre + t, s = T % kS;
      // a whole 128-row box even for a short last tile: keys past the range
      // are masked, rows past the capacity arrive zero-filled
      if (t >= kS) mbar_wait(SREADY((T - kS) % 3), par3(T - kS));
      if (elect_one()) {
        mbar_expect_tx(FULLK(s), static_cast<uint32_t>(kKV));
#pragma unroll
        for (int h = 0; h < kHalves; ++h)
          tma_load_3d_hint(base + s * kKV + h * kHalf, &tm_k128, FULLK(s), h * 64, key_begin + t * kStageKeys, z, evict_first);
      }
      __syncwarp();
    };
    auto issue_v = [&](int pass, int t) {
      const int T = pass * n_pre + t, s = T % kS;
      if (t >= kS) mbar_wait(PVDONE(s), parS(T - kS));
      if (elect_one()) {
        mbar_expect_tx(FULLV(s), static_cast<uint32_t>(kKV));
#pragma unroll
        for (int h = 0; h < kHalves; ++h)
          tma_load_3d_hint(base + C::kRingV + s * kKV + h * kHalf, &tm_v128, FULLV(s), h * 64, key_begin + t * kStageKeys, z,
                           evict_first);
      }
      __syncwarp();
    };
    // a ring of tiles waits for nothing
    auto issue_first = [&](int pass, int n) {
#pragma unroll 1
      for (int t = 0; t < n; ++t) {
        issue_k(pass, t);
        issue_v(pass, t);
      }
    };
    // past it the keys go one tile ahead of the values: a key slot is free once its S
    // is done, a value slot only after the softmax and the PV product, and waiting for
    // that before the next keys left S idle for a memory round trip. Measured: a layer
    // of 16384 keys 14.2 -> 13.7 us at K = 4, 19.9 -> 18.4 at 16; of 4096 keys at K = 8
    // 7.75 -> 7.2; the attention of 8 scenes, 8192 keys, K = 16: 45.9 -> 43.9. (Every wait
    // stays ahead of the phase after the one it waits for: K(T) and V(T) are still issued
    // after S(T - kS) and PV(T - kS), and neither of those needs a later tile.)
    auto issue_rest = [&](int pass, int n0) {
#pragma unroll 1
      for (int t = n0; t <= n_pre; ++t) {
        if (t < n_pre) issue_k(pass, t);
        if (t > n0) issue_v(pass, t - 1);
      }
    };
    const int n0 = min(n_pre, kS);
    issue_first(0, n0);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (!valid && rank == 0 && lane == 0 && blockIdx.y == 0)
      sd_set_error(kFused && L_pre >= 0 ? SD_DEVERR_KV_OVERFLOW : SD_DEVERR_LENGTH);
    // chained layers: the cluster launched last starts only when the previous
    // layer frees its SMs; the first head's CTAs bring its tiles of their own key
    // range, and its query and new rows, into L2
    if (n_pre > 0 && early && kvh == 0 && mblock == 0 && b == static_cast<int>(gridDim.z) - 1 && a.Hkv > 1 && elect_one()) {
      const int zl = b * a.Hkv + a.Hkv - 1;
#pragma unroll 1
      for (int t = 0; t < n_pre; ++t)
#pragma unroll
        for (int h = 0; h < kHalves; ++h) {
          tma_prefetch_3d(&tm_k128, h * 64, key_begin + t * kStageKeys, zl);
          tma_prefetch_3d(&tm_v128, h * 64, key_begin + t * kStageKeys, zl);
        }
      if (rank == 0)
#pragma unroll 1
        for (int i = 0; i < a.R; ++i) {
          const long long row = static_cast<long long>(b) * a.R + i;
          bulk_prefetch_l2((kFused ? a.qw : a.q) + (row * a.Hq + (a.Hkv - 1) * a.G) * kDim, a.G * kDim * 2);
          if (kFused) {
            bulk_prefetch_l2(a.k_new + (row * a.Hkv + a.Hkv - 1) * kDim, kDim * 2);
            bulk_prefetch_l2(a.v_new + (row * a.Hkv + a.Hkv - 1) * kDim, kDim * 2);
          }
        }
    }
    __syncwarp();
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      if (pass == 1) {
        mbar_wait(DECIDE, 0);
        if (!*reinterpret_cast<volatile int*>(s_redo)) break;
      }
      if (pass == 2) mbar_wait(MAXIMA, 0);  // every product of pass 1 is done
      if (pass > 0) issue_first(pass, n0);
      issue_rest(pass, n0);
      if (pass > 0) continue;
      // the softmax threads arrive last (after the last S of the last pass), so
      // this warp and the issuing warps arrive before the decision
      if (csize > 1) cluster_arrive_relaxed();
      if (kFused && elect_one()) {
        // advance the scene's length once every CTA of the scene has read it (and
        // the previous kernel, which may read it, has completed)
        if (early) griddep_wait();
        __threadfence();
        const uint32_t total = gridDim.x * gridDim.y;
        if (atomicAdd(&a.ticket[b], 1u) == total - 1) {
          if (len0 >= 0 && len0 + a.R <= a.cap) a.len[b] = len0 + a.R;
          a.ticket[b] = 0;
        }
      }
      __syncwarp();
    }
    __syncwarp();
    if (csize > 1) cluster_wait();
  } else if (warp == 1) {
    // -------------------------------------------------------------- S issue
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tmem_slot)),
                 "r"(C::kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;
    ranges(*s_len);
    const uint64_t dK0 = umma_desc(base, 16, 1024);
    const uint64_t dQ = umma_desc(qs, 16, 1024);
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      if (pass == 1) {
        if (csize > 1) cluster_arrive_relaxed();
        mbar_wait(DECIDE, 0);
        if (!*reinterpret_cast<volatile int*>(s_redo)) break;
      }
      if (pass == 2) mbar_wait(MAXIMA, 0);
      // t = -1 (early prefix only, when there is time): the batch of tile 0 is issued once before Q is complete, on whatever
      // shared memory holds, and overwritten by the real one: the instructions and
      // the tensor pipe are warm when Q is there (6.47 -> 6.29 us a target layer)
      if (n_pre == 0 && pass == 0) named_bar_sync(3, kSoftThreads + 32);
#pragma unroll 1
      for (int t = pass == 0 && early && n_pre > 0 ? -1 : 0; t < n_pre; ++t) {
        const int T = pass * n_pre + max(t, 0), s = T % kS;
        if (t >= 0) {
          if (t == 0 && pass == 0) named_bar_sync(3, kSoftThreads + 32);  // a hardware barrier: its wake-up is short
          // the softmax has read S(T - 3): its buffer takes S(T)
          if (t >= 3) mbar_wait(SFREE(T % 3), par3(T - 3));
          mbar_wait(FULLK(s), parS(T));
          tc_fence_after();
        }
        const uint32_t ts = tmem + C::kSStride * (T % 3);
        const uint64_t dk = dK0 + static_cast<uint64_t>((s * kKV) >> 4);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < kDim / 16; ++kk)
            umma(ts, dk + (((kk >> 2) * kHalf + (kk & 3) * 32) >> 4),
                 dQ + (((kk >> 2) * C::kQHalf + (kk & 3) * 32) >> 4), kIdescS, kk > 0 ? 1 : 0);
          if (t >= 0) umma_commit(SREADY(T % 3));
        }
        __syncwarp();
      }
    }
    mbar_wait(TMEMDONE, 0);  // every softmax warp has read its last column
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::kTmemCols) : "memory");
    if (csize > 1) cluster_wait();
  } else if (warp == 2) {
    // -------------------------------------------------------------- PV issue
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_o = *tmem_slot + 3 * C::kSStride;
    ranges(*s_len);
    const bool has_new = valid && last_rank;
    // V^T: MN-major. Head dim 64 keeps M = 128 with both 64-row halves of the operand
    // on the same rows (stride 0): O's lanes 64..127 repeat 0..63 and are not read
    const uint64_t dV0 = umma_desc(base + C::kRingV, kHalves == 2 ? kHalf : 0, 1024);
    const uint64_t dN = umma_desc(base + C::kOffNewV, kHalves == 2 ? C::kNewHalf : 0, 1024);
    const uint64_t dP0 = umma_desc(base + C::kOffP, C::kPGroup, 256, 6);  // P^T: MN-major, 32-byte swizzle
#pragma unroll 1
    for (int pass = 0; pass < 3; ++pass) {
      if (pass == 1) {
        if (csize > 1) cluster_arrive_relaxed();
        mbar_wait(DECIDE, 0);
        if (!*reinterpret_cast<volatile int*>(s_redo)) break;
      }
      if (pass == 2) mbar_wait(MAXIMA, 0);
      const bool take_new = has_new && pass != 1;
      auto new_product = [&](bool add) {
        mbar_wait(PNEW, pass >> 1);
        tc_fence_after();
        const uint64_t dpn = umma_desc(base + C::kOffPNew, C::kPNewGroup, 256, 6);
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < C::kMaxNew / 16; ++kk)
            if (kk * 16 < a.R) {
              umma(tmem_o, dN + (kk * 2048 >> 4), dpn + (kk * 512 >> 4), kIdescO, kk > 0 || add ? 1 : 0);
              umma(tmem_o, dN + (kk * 2048 >> 4), dpn + ((C::kPNewLow + kk * 512) >> 4), kIdescO, 1);
            }
          umma_commit(NEWDONE);
        }
        __syncwarp();
      };
      if (C::kNewFirst && take_new) new_product(false);
      for (int t = 0; t < n_pre; ++t) {
        const int T = pass * n_pre + t, s = T % kS;
        mbar_wait(PFULL(T), (T >> 1) & 1);
        mbar_wait(FULLV(s), parS(T));
        tc_fence_after();
        const uint64_t dv = dV0 + static_cast<uint64_t>((s * kKV) >> 4);
        const uint64_t dp = dP0 + static_cast<uint64_t>(((T & 1) * C::kPBuf) >> 4);
        const int n_steps = pv_keys(t) >> 4;
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            if (kk < n_steps) {
              umma(tmem_o, dv + (kk * 2048 >> 4), dp + (kk * 512 >> 4), kIdescO,
                   (t > 0 || kk > 0 || (C::kNewFirst && take_new)) ? 1 : 0);
              if (C::kSplit) umma(tmem_o, dv + (kk * 2048 >> 4), dp + ((C::kP + kk * 512) >> 4), kIdescO, 1);
            }
          umma_commit(PVDONE(s));
        }
        __syncwarp();
      }
      if (!C::kNewFirst && take_new) new_product(n_pre > 0);
    }
    if (csize > 1) cluster_wait();
  } else {
    // -------------------------------------------------------------- softmax
    const int st = static_cast<int>(threadIdx.x) - kSoft0;  // 0 .. 511
    const int sw = warp - kFirstSoft;
    const int group = sw >> 3;
    const int half = (sw >> 2) & 1;      // rows kRpt * half .. + kRpt - 1 of the group's tile
    const int quarter = warp & 3;        // TMEM lane quarter of this warp
    const int kl = quarter * 32 + lane;  // key lane of S^T / d lane of O^T
    const uint32_t lane_off = static_cast<uint32_t>(quarter * 32) << 16;
    const int row0 = kRpt * half;
    // this thread's 16-byte chunks: of the packed query tile (row idx / kChunks, chunk
    // idx % kChunks, rows past M zero) and, in the cluster's last rank, of the new key
    // and value rows
    constexpr int kQc = (kR * kChunks + kSoftThreads - 1) / kSoftThreads;
    auto q_off = [&](int p) {
      const int i = gdiv(p);
      return ((static_cast<long long>(b) * a.R + i) * a.Hq + kvh * a.G + (p - i * a.G)) * kDim;
    };
    const bool new_kv = last_rank && st < a.R * kChunks;
    const long long kv_row = ((static_cast<long long>(b) * a.R + (st / kChunks)) * a.Hkv + kvh) * kDim + (st % kChunks) * 8;
    uint4 qv[kQc] = {}, own[kQc] = {};  // the row's chunk, and its own new key's
    uint4 kv = make_uint4(0, 0, 0, 0), vv = make_uint4(0, 0, 0, 0);
    auto load_q = [&] {
#pragma unroll
      for (int u = 0; u < kQc; ++u) {
        const int idx = st + u * kSoftThreads, p = mblock * kR + (idx / kChunks);
        qv[u] = idx < kR * kChunks && p < a.M
                    ? __ldcg(reinterpret_cast<const uint4*>((kFused ? a.qw : a.q) + q_off(p) + (idx % kChunks) * 8))
                    : make_uint4(0, 0, 0, 0);
      }
    };
    auto load_own = [&] {
#pragma unroll
      for (int u = 0; u < kQc; ++u) {
        const int idx = st + u * kSoftThreads, p = mblock * kR + (idx / kChunks), i = gdiv(p);
        const __nv_bfloat16* src = kFused ? a.k_new + ((static_cast<long long>(b) * a.R + i) * a.Hkv + kvh) * kDim
                                          : a.kc + ((static_cast<long long>(b) * a.Hkv + kvh) * a.cap + L_pre + i) * kDim;
        if (idx < kR * kChunks && p < a.M) own[u] = __ldcg(reinterpret_cast<const uint4*>(src + (idx % kChunks) * 8));
      }
    };
    auto load_kv = [&](const __nv_bfloat16* k, const __nv_bfloat16* v, long long src) {
      kv = __ldcg(reinterpret_cast<const uint4*>(k + src));
      vv = __ldcg(reinterpret_cast<const uint4*>(v + src));
    };
    auto cache_row = [&] {
      return ((static_cast<long long>(b) * a.Hkv + kvh) * a.cap + L_pre + (st / kChunks)) * kDim + (st % kChunks) * 8;
    };
    const float2* cs_tab = reinterpret_cast<const float2*>(smem + C::kOffP);  // [R][64] (cos, sin)
    // rotation table of the R new positions. A warp takes 4 pairs, its lanes 8
    // rows: a constant-bank read serialises over the lanes' different addresses
    // (with 32 pairs a warp the table took ~2800 cycles, on the path of the
    // cluster launched last)
    auto make_table = [&](bool known) {
      float2* tabw = reinterpret_cast<float2*>(smem + C::kOffP);
      const int d = sw * 4 + (lane & 3);
#pragma unroll 1
      for (int i = lane >> 2; i < a.R; i += 8) {
        const int32_t pc = known ? a.pos[(static_cast<long long>(b) * a.R + i) * 3 + tab.axis[d]] : tab.axis[d];
        tabw[i * 64 + d] = sd_rope_cs(static_cast<float>(pc), d, tab);
      }
    };
    // the rows, rotated (fused), into the operand layouts; on the second of two runs
    // the append too
    auto store_rows = [&](bool has_kv, int it) {
#pragma unroll
      for (int u = 0; u < kQc; ++u) {
        const int idx = st + u * kSoftThreads, row = idx / kChunks, c = idx % kChunks, p = mblock * kR + row;
        if (idx >= kR * kChunks) break;  // warp-uniform
        uint32_t w[4] = {qv[u].x, qv[u].y, qv[u].z, qv[u].w}, o[4] = {own[u].x, own[u].y, own[u].z, own[u].w};
        if (kFused) {  // (rows past M, zero, turn by the last row's angles: a branch cost 0.1 us a layer)
          const float2* cs = cs_tab + gdiv(min(p, a.M - 1)) * 64 + c * 4;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            w[j] = sd_rope_pair(w[j], cs[j].x, cs[j].y);
            o[j] = sd_rope_pair(o[j], cs[j].x, cs[j].y);
          }
        }
        st_shared_v4(qs + swz(row, c, C::kQHalf), w[0], w[1], w[2], w[3]);
        // the row's reference; a score that is not a number or infinite: 0
        float d = dot8(w, o);
#pragma unroll
        for (int x = kChunks / 2; x > 0; x >>= 1) d += __shfl_xor_sync(0xffffffffu, d, x);
        d *= sl;
        if (c == 0) row_nref[row] = fabsf(d) < INFINITY ? -d : 0.f;
      }
      if (last_rank && st < C::kMaxNew * kChunks) {
        // new key (rotated) and value rows, zero past R
        const int i = st / kChunks, c = st % kChunks;
        uint32_t w[4] = {kv.x, kv.y, kv.z, kv.w};
        if (kFused && has_kv) {
          const float2* cs = cs_tab + i * 64 + c * 4;
#pragma unroll
          for (int j = 0; j < 4; ++j) w[j] = sd_rope_pair(w[j], cs[j].x, cs[j].y);
        }
        const uint32_t off = swz(i, c, C::kNewHalf);
        st_shared_v4(base + C::kOffNewK + off, w[0], w[1], w[2], w[3]);
        st_shared_v4(base + C::kOffNewV + off, vv.x, vv.y, vv.z, vv.w);
        if (kFused && has_kv && it == 1 && mblock == 0) {
          // the append: cache rows L_pre .. L_pre + R - 1, which no CTA of
          // this launch reads
          *reinterpret_cast<uint4*>(a.kc + cache_row()) = make_uint4(w[0], w[1], w[2], w[3]);
          *reinterpret_cast<uint4*>(a.vc + cache_row()) = vv;
        }
      }
    };
    // rank c merges packed rows [c * rpc, ...) of the m-block's rows_in rows
    const int rows_in = max(1, min(kR, a.M - mblock * kR));
    const int rpc = (rows_in + csize - 1) / csize;
    auto rows_of = [&](int c) { return max(0, min(rpc, rows_in - c * rpc)); };
    const int my_rows = rows_of(rank);
    const int mrow0 = rank * rpc;
    uint32_t tmem;
    bool has_new;
    auto cta_barrier = [&] {
      tc_fence_before();
      __syncthreads();
      tc_fence_after();
      tmem = *tmem_slot;
      ranges(*s_len);
      has_new = valid && last_rank;
    };
    // Two runs, the first BEFORE the dependency wait on whatever the rows hold: it
    // brings this code into the instruction cache (and, with the early prefix, the
    // rows into L2), and the second overwrites everything it stored (.cg loads: no
    // stale L1 line). The cluster launched last has no time for it. Without the early
    // prefix the dry run and its table took the draft step from 6.14 to 5.93 us and the
    // tiny layer from 6.9 to 6.6; as one loop for both kinds of launch the target layer
    // lost 0.15 us, so each has its own.
    const int it0 = last_cluster ? 1 : 0;
    if (early) {
      if (kFused) make_table(true);
      cta_barrier();
      const bool has_kv = new_kv && valid;
#pragma unroll 1
      for (int it = it0; it < 2; ++it) {
        if (it == 1) griddep_wait();
        load_q();
        if (kFused || valid) load_own();
        if (kFused && has_kv) load_kv(a.k_new, a.v_new, kv_row);
        if (!kFused && has_kv) load_kv(a.kc, a.vc, cache_row());
        store_rows(has_kv, it);
      }
    } else {
      // Without the early prefix the rows are read together with the length and the
      // positions: one global round trip before the tiles, not two. The attention's
      // new rows need the length: the threads read it themselves rather
      // than wait for the producer's at the CTA barrier (one scene, L = 4096, K = 7:
      // 7.8 -> 7.4 us; head dim 64, L = 4099: 9.5 -> 8.9)
      valid = false;
#pragma unroll 1
      for (int it = it0; it < 2; ++it) {
        if (it == 1) {
          griddep_wait();
          load_q();
          if (!kFused) ranges(__ldcg(a.len + b));
          if (kFused || valid) load_own();
          if (kFused && new_kv) load_kv(a.k_new, a.v_new, kv_row);
          if (!kFused && new_kv && valid) load_kv(a.kc, a.vc, cache_row());
        }
        if (kFused) make_table(it == 1);
        if (it == 1) cta_barrier();
        store_rows(new_kv && valid, it);
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    named_bar_sync(3, kSoftThreads + 32);  // Q and the references are complete; the rotation table is no longer read
    if (st == 0) griddep_launch();         // every older kernel has finished: the next layer may launch

    const uint64_t sl2 = pack2f(sl, sl);
    uint64_t lp2[kRpt / 2];  // this key lane's row sums, in pairs
    const uint32_t pbuf = base + C::kOffP + group * C::kPBuf;
    const uint32_t pkey = pbuf + kl * 32;
    const uint32_t psw = (kl >> 2) & 1;  // 32-byte swizzle
    // the last new key that packed row r of this tile sees: row p = i * G + g is
    // new row i and sees new keys 0..i (all R under the block mask)
    auto last_new = [&](int r) { return block ? a.R - 1 : min(gdiv(mblock * kR + r), a.R - 1); };
    int pass = 0;
    bool out_of_range = false;
    // a warp none of whose rows exists (a draft's 4 rows of 32) skips the weights: its
    // P stays stale and reaches only O columns that are never read. On the wider
    // tiles, chosen to fit, the test cost more than it saved (47.0 -> 48.7 us at 8
    // scenes, L = 8192, K = 16)
    constexpr bool skips = kR == 32;
    // this thread's rows j0 .. j0 + kN - 1 of tile T (its scores in buffer sb) to
    // weights and P; vb, vpar: the barrier of PV(T - 2)
    auto chunk = [&](auto kn, int T, int sb, int vb, uint32_t vpar, int j0, bool key_ok, bool first) {
      constexpr int kN = decltype(kn)::value;
      uint32_t r[kN], pw[kN / 2], pl[kN / 2];
      tmem_ld(tmem + C::kSStride * sb + row0 + j0 + lane_off, r);
      if (j0 + kN == kRpt) {
        // the tile's scores are all in registers: its buffer may take S(T + 3)
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(SFREE(sb));
      }
      weights_to_p<kN, C::kSplit>(r, row_nref + row0 + j0, sl2, key_ok, lp2 + j0 / 2, pw, pl);
      if (j0 == 0) {
        // PV(T - 2), or the new keys' product, has read the buffer
        if (T >= 2) mbar_wait(PVDONE(vb), vpar);
        if (C::kNewFirst && first && has_new && group == 1) mbar_wait(NEWDONE, pass >> 1);
      }
#pragma unroll
      for (int h = 0; h < kN / 8; ++h) {
        const int ch = (row0 + j0) / 8 + h;
        const uint32_t dst = pkey + (ch >> 1) * C::kPGroup + (((ch & 1) ^ psw) << 4);
        st_shared_v4(dst, pw[4 * h], pw[4 * h + 1], pw[4 * h + 2], pw[4 * h + 3]);
        if (C::kSplit) st_shared_v4(dst + C::kP, pl[4 * h], pl[4 * h + 1], pl[4 * h + 2], pl[4 * h + 3]);
      }
    };
    bool redo = false;
    // every product of a pass is done (behind a barrier that every softmax warp
    // reaches after its last tile)
    auto wait_products = [&](int ps) {
      const int Tl = (ps + 1) * n_pre - 1;
      const bool new_last = has_new && ps != 1 && (!C::kNewFirst || n_pre == 0);
      if (new_last) mbar_wait(NEWDONE, ps >> 1);
      else if (n_pre > 0) mbar_wait(PVDONE(Tl % kS), parS(Tl));
    };
    // the new keys: scores of 8 packed rows against 16 keys a step by mma.sync,
    // weights to kOffPNew, row sums to row_new
    auto new_keys = [&](int unit) {
      const int r8 = unit * 8;
      const int lim0 = last_new(r8 + 2 * (lane & 3)), lim1 = last_new(r8 + 2 * (lane & 3) + 1);
      const float2 nr = *reinterpret_cast<const float2*>(row_nref + r8 + 2 * (lane & 3));
      float l0 = 0.f, l1 = 0.f;
      uint32_t bq[kDim / 32][4];
#pragma unroll
      for (int k2 = 0; k2 < kDim / 32; ++k2) ldmatrix4(qs + swz(r8 + (lane & 7), 4 * k2 + (lane >> 3), C::kQHalf), bq[k2]);
#pragma unroll 1
      for (int m = 0; m * 16 < a.R; ++m) {
        float c[4] = {0.f, 0.f, 0.f, 0.f}, c1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int k2 = 0; k2 < kDim / 32; ++k2) {
          uint32_t ak[4], al[4];
          ldmatrix4(base + C::kOffNewK + swz(m * 16 + (lane & 15), 4 * k2 + (lane >> 4), C::kNewHalf), ak);
          ldmatrix4(base + C::kOffNewK + swz(m * 16 + (lane & 15), 4 * k2 + 2 + (lane >> 4), C::kNewHalf), al);
          mma_bf16(c, ak, bq[k2][0], bq[k2][1]);
          mma_bf16(c1, al, bq[k2][2], bq[k2][3]);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int key = m * 16 + (lane >> 2) + 8 * h;
          // (a masked score may be anything: selected away before it is a weight)
          const float e0 = key <= lim0 ? ex2(fmaf(c[2 * h] + c1[2 * h], sl, nr.x)) : 0.f;
          const float e1 = key <= lim1 ? ex2(fmaf(c[2 * h + 1] + c1[2 * h + 1], sl, nr.y)) : 0.f;
          uint32_t hi, lo = 0;
          uint64_t l;
          weight_terms<true>(e0, e1, hi, lo, l);
          l0 += e0;
          l1 += e1;
          const uint32_t dst = base + C::kOffPNew + (unit >> 1) * C::kPNewGroup + key * 32 +
                               (((unit & 1) ^ ((key >> 2) & 1)) << 4) + (lane & 3) * 4;
          asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst), "r"(hi) : "memory");
          asm volatile("st.shared.u32 [%0], %1;" ::"r"(dst + C::kPNewLow), "r"(lo) : "memory");
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(PNEW);
#pragma unroll
      for (int o = 4; o < 32; o <<= 1) {
        l0 += __shfl_xor_sync(0xffffffffu, l0, o);
        l1 += __shfl_xor_sync(0xffffffffu, l1, o);
      }
      out_of_range |= fmaxf(l0, l1) > kHigh;
      if (lane < 4) *reinterpret_cast<float2*>(row_new + r8 + 2 * lane) = make_float2(l0, l1);
    };
    while (true) {
      // On the 32-row tile by the last warps while S(0) runs (their group's first
      // tile comes second); on the others by the group that does not have the last
      // tile, after its own.
      if (C::kNewFirst && has_new && kSoftWarps - 1 - sw < kR / 8) new_keys(kSoftWarps - 1 - sw);
      // ---- this group's prefix tiles
#pragma unroll
      for (int j = 0; j < kRpt / 2; ++j) lp2[j] = 0ull;
      const int t_first = ((pass * n_pre) ^ group) & 1;
      const int T1 = pass * n_pre + t_first, V1 = T1 + 2 * kS - 2;  // PV(T - 2) as a phase of its ring, T >= 0
      int sb = T1 % 3, vb = V1 % kS;
      uint32_t spar = (T1 / 3) & 1, vpar = (V1 / kS) & 1;
      int key0 = key_begin + t_first * kStageKeys;
#pragma unroll 1
      for (int t = t_first; t < n_pre; t += 2) {
        const int T = pass * n_pre + t;
        const bool key_ok = key0 + kl < key_end;
        key0 += 2 * kStageKeys;
        mbar_wait(SREADY(sb), spar);
        tc_fence_after();
#pragma unroll
        for (int j0 = 0; j0 + 16 <= kRpt; j0 += 16)
          if (!skips || row0 < rows_in) chunk(std::integral_constant<int, 16>{}, T, sb, vb, vpar, j0, key_ok, t == t_first);
        if constexpr (kRpt % 16 != 0)
          chunk(std::integral_constant<int, 8>{}, T, sb, vb, vpar, kRpt - 8, key_ok, t == t_first);
        if (skips && row0 >= rows_in) {
          // none of this warp's rows exists: the barriers' phases only
          if (lane == 0) mbar_arrive(SFREE(sb));
          if (T >= 2) mbar_wait(PVDONE(vb), vpar);
        }
        if ((sb += 2) >= 3) sb -= 3, spar ^= 1;
        if ((vb += 2) >= kS) vb -= kS, vpar ^= 1;
        if (!key_ok && kl < pv_keys(t) && half < kHalves) {
          // stale or foreign key row that the product reads: zero its V row (this
          // thread's 64-column half) so 0 * NaN cannot reach O, once the tile has
          // landed. Chunks in an order that differs by lane: rows are 128 bytes apart
          // (in one order every lane met the same banks, ~2500 cycles a partial tile)
          const int s = T % kS;
          mbar_wait(FULLV(s), parS(T));
          const uint32_t vrow = base + C::kRingV + s * kKV + half * kHalf + kl * 128;
#pragma unroll
          for (int c = 0; c < 8; ++c) st_shared_v4(vrow + ((c ^ (kl & 7)) << 4), 0u, 0u, 0u, 0u);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(PFULL(T));
      }
      if (!C::kNewFirst && has_new && group == (n_pre & 1))
#pragma unroll 1
        for (int unit = sw & 7; unit < kR / 8; unit += 8) new_keys(unit);
      // ---- whether a row's scores rose too far above its reference
      {
        float hi = 0.f;
#pragma unroll
        for (int j = 0; j < kRpt / 2; ++j) {
          float x, y;
          unpack2(lp2[j], x, y);
          hi = fmaxf(hi, fmaxf(x, y));
        }
        out_of_range |= hi > kHigh;
      }
      const bool again = named_bar_or(2, kSoftThreads, out_of_range);
      if (pass == 2) break;
      redo = again;
      if (redo) {
        // every product of pass 0 is done before the rings are refilled, and no
        // warp still looks for it when pass 1 moves the barriers on
        wait_products(0);
        named_bar_sync(2, kSoftThreads);
      }
      if (st == 0) {
        *s_redo = redo ? 1 : 0;
        mbar_arrive(DECIDE);
      }
      if (__builtin_expect(!redo, 1)) break;
      // ---- pass 1: every row's exact maximum over this CTA's keys (the PV products
      // run on stale weights, their sums are dropped by pass 2)
      float mx[kRpt];
#pragma unroll
      for (int j = 0; j < kRpt; ++j) mx[j] = -INFINITY;
#pragma unroll 1
      for (int t = (n_pre ^ group) & 1; t < n_pre; t += 2) {
        const int T = n_pre + t;
        mbar_wait(SREADY(T % 3), par3(T));
        tc_fence_after();
        const bool key_ok = key_begin + t * kStageKeys + kl < key_end;
#pragma unroll
        for (int j0 = 0; j0 < kRpt; j0 += 8) {
          uint32_t r[8];
          tmem_ld(tmem + C::kSStride * (T % 3) + row0 + j0 + lane_off, r);
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (key_ok) mx[j0 + j] = fmaxf(mx[j0 + j], __uint_as_float(r[j]) * sl);
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(SFREE(T % 3));
        const int Tp = max(T - 2, 0);
        mbar_wait(PVDONE(Tp % kS), parS(Tp));
        if (lane == 0) mbar_arrive(PFULL(T));
      }
      named_bar_sync(2, kSoftThreads);
      wait_products(1);
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
      for (int row = sw; row < kR; row += kSoftWarps) {
        const float4 x = reinterpret_cast<const float4*>(rb + row * 128)[lane];
        float m = fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (has_new)
          m = fmaxf(m, new_key_max<kDim>(smem + C::kOffQ, row, C::kQHalf, smem + C::kOffNewK, C::kNewHalf, last_new(row), sl, lane));
        if (lane == 0) row_nref[row] = m == -INFINITY ? 0.f : -m;
      }
      named_bar_sync(2, kSoftThreads);
      if (st == 0) mbar_arrive(MAXIMA);
      pass = 2;
    }
    // ---- the last S product is done (both groups have seen their last tile's): the
    // K ring may receive
    const bool merge = csize > 1;
    if (merge) cluster_arrive_relaxed();
    // row sums over this warp's keys, while the last products run: lane L ends with
    // that of row row0 + 8 c + (L >> 2)
    float lsum[kRpt / 8];
#pragma unroll
    for (int c = 0; c < kRpt / 8; ++c) {
      float v[8];
#pragma unroll
      for (int j = 0; j < 4; ++j) unpack2(lp2[4 * c + j], v[2 * j], v[2 * j + 1]);
      lsum[c] = warp_sum8(v, lane);
    }
    wait_products(pass);
    tc_fence_after();
    // O: this warp reads its 32 d lanes of a quarter of the rows
    constexpr int kOr = kR / 4;
    const int orow0 = (group * 2 + half) * kOr;
    uint32_t o[kOr];
    if (n_pre > 0 || has_new) {
#pragma unroll
      for (int j0 = 0; j0 + 8 <= kOr; j0 += 8) {
        uint32_t x8[8];
        tmem_ld(tmem + 3 * C::kSStride + orow0 + j0 + lane_off, x8);
#pragma unroll
        for (int j = 0; j < 8; ++j) o[j0 + j] = x8[j];
      }
      if constexpr (kOr % 8 != 0) {
        uint32_t x4[4];
        tmem_ld(tmem + 3 * C::kSStride + orow0 + kOr - 4 + lane_off, x4);
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
      if ((lane & 3) == 0)
#pragma unroll
        for (int c = 0; c < kRpt / 8; ++c) row_sum[(row0 + 8 * c + (lane >> 2)) * 8 + group * 4 + quarter] = lsum[c];
      named_bar_sync(2, kSoftThreads);
      if (st < kR) {
        const float4 l0 = reinterpret_cast<const float4*>(row_sum + st * 8)[0];
        const float4 l1 = reinterpret_cast<const float4*>(row_sum + st * 8)[1];
        float l = ((l0.x + l0.y) + (l0.z + l0.w)) + ((l1.x + l1.y) + (l1.z + l1.w));
        if (has_new) l += row_new[st];
        row_new[st] = l > 0.f ? 1.f / l : 0.f;
      }
      named_bar_sync(2, kSoftThreads);
#pragma unroll
      for (int j = 0; j < kOr; ++j) {
        const int row = orow0 + j, p = mblock * kR + row;
        const float inv_l = row_new[row];
        if (valid && p < a.M && inv_l > 0.f && kl < kDim) a.out[q_off(p) + kl] = __float2bfloat16_rn(__uint_as_float(o[j]) * inv_l);
      }
    } else {
      float* send = reinterpret_cast<float*>(smem + C::kRingV);
      if (kl < kDim)
#pragma unroll
        for (int j = 0; j < kOr; ++j) send[(orow0 + j) * kRowF + kl] = __uint_as_float(o[j]);
      if ((lane & 3) == 0)
#pragma unroll
        for (int c = 0; c < kRpt / 8; ++c) send[(row0 + 8 * c + (lane >> 2)) * kRowF + kRowL + group * 4 + quarter] = lsum[c];
      if (st < kR)
        *reinterpret_cast<float2*>(send + st * kRowF + kRowM) = make_float2(-row_nref[st], has_new ? row_new[st] : 0.f);
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      named_bar_sync(2, kSoftThreads);
      if (st == 0) mbar_expect_tx(RECV, static_cast<uint32_t>(csize * my_rows * kRowBytes));
      cluster_wait();  // every peer's K ring is free to receive
      // softmax warp w sends rank w's rows to it, into its slots [rank * rpc, ...)
      if (elect_one()) {
        if (sw < csize && rows_of(sw) > 0)
          bulk_copy_s2s(cluster_map(base + rank * rpc * kRowBytes, sw), base + C::kRingV + sw * rpc * kRowBytes,
                        static_cast<uint32_t>(rows_of(sw) * kRowBytes), cluster_map(RECV, sw));
        asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      }
      __syncwarp();
    }
    if (kFused && valid) {
      // while the partials travel: every CTA of the cluster has read the raw
      // rows (its tiles came after), so the rotated query rows this CTA merges
      // go back to q
#pragma unroll 1
      for (int idx = st; idx < my_rows * kChunks; idx += kSoftThreads) {
        const int row = mrow0 + (idx / kChunks), c = idx % kChunks, p = mblock * kR + row;
        if (p >= a.M) continue;
        *reinterpret_cast<uint4*>(a.qw + q_off(p) + c * 8) =
            *reinterpret_cast<const uint4*>(smem + C::kOffQ + swz(row, c, C::kQHalf));
      }
    }
    if (merge) {
      // ---- merge of the rows this CTA owns, a warp a row, kDim / 32 d a lane; slot
      // c * rpc + r came from rank c. Unless some rank ran its range again all have
      // the row's one reference and the partials add.
      const float* recv = reinterpret_cast<const float*>(smem);
      const int cstep = rpc * kRowF;
      constexpr int kPer = kDim / 32;
      struct alignas(kPer * 4) Row {
        float v[kPer];
      };
#pragma unroll 1
      for (int r = sw; r < my_rows; r += kSoftWarps) {
        const float* part = recv + r * kRowF;
        const int p = mblock * kR + mrow0 + r;
        __nv_bfloat16* dst = a.out + q_off(p) + lane * kPer;
        if (r == sw) mbar_wait(RECV, 0);
        Row ov = {};
        float l = 0.f;
        const float ref0 = part[kRowM];
        // the ranks' row sums and references, one a lane: element lane & 15 of every
        // second rank (8: the reference; 0..7 and 9: sums)
        const int e = lane & 15;
        bool moved = false;
#pragma unroll 2
        for (int c = lane >> 4; c < csize; c += 2) {
          const float x = part[c * cstep + kRowL + (e < 10 ? e : 0)];
          moved |= e == 8 && x != ref0;
          l += e < 10 && e != 8 ? x : 0.f;
        }
#pragma unroll 4
        for (int c = 0; c < csize; ++c) {
          const Row x = reinterpret_cast<const Row*>(part + c * cstep)[lane];
#pragma unroll
          for (int j = 0; j < kPer; ++j) ov.v[j] += x.v[j];
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
        if (__builtin_expect(__any_sync(0xffffffffu, moved), 0)) {
          // weigh every partial by its own reference (those without a key count for nothing)
          auto sums = [&](const float* pc) {
            float x = pc[kRowM + 1];
            for (int e = 0; e < 8; ++e) x += pc[kRowL + e];
            return x;
          };
          float m = -INFINITY;
          ov = Row{};
          l = 0.f;
#pragma unroll 1
          for (int c = 0; c < csize; ++c)
            if (sums(part + c * cstep) > 0.f) m = fmaxf(m, part[c * cstep + kRowM]);
#pragma unroll 1
          for (int c = 0; c < csize; ++c) {
            const float* pc = part + c * cstep;
            const float lc = sums(pc);
            if (lc == 0.f) continue;
            const float w = ex2(pc[kRowM] - m);
            const Row x = reinterpret_cast<const Row*>(pc)[lane];
#pragma unroll
            for (int j = 0; j < kPer; ++j) ov.v[j] = fmaf(w, x.v[j], ov.v[j]);
            l = fmaf(w, lc, l);
          }
        }
        if (valid && p < a.M && l > 0.f) {
          const float inv_l = 1.f / l;
#pragma unroll
          for (int j = 0; j < kPer; j += 2)
            *reinterpret_cast<uint32_t*>(dst + j) = cvt_bf16x2(ov.v[j] * inv_l, ov.v[j + 1] * inv_l);
        }
      }
      if (elect_one()) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
      __syncwarp();
    }
    if (kFused && valid && last_rank) {
      // every CTA of the cluster has read the raw key rows: the rotated ones go back to
      // k_new, by the warps that merge least. With several m-blocks each one's cluster
      // reads them: the last to come here writes (the fence orders the reads before its
      // ticket)
      bool write = true;
      if (a.n_mblocks > 1) {
        if (st == 0) {
          __threadfence();
          *s_kvlast = atomicAdd(&a.kv_ticket[b * a.Hkv + kvh], 1u) == static_cast<uint32_t>(a.n_mblocks - 1);
          if (*s_kvlast) a.kv_ticket[b * a.Hkv + kvh] = 0;  // re-armed
        }
        named_bar_sync(2, kSoftThreads);
        write = *s_kvlast != 0;
      }
      const int idx = kSoftThreads - 1 - st, i = idx / kChunks, c = idx % kChunks;
      if (write && i < a.R)
        *reinterpret_cast<uint4*>(a.k_new + ((static_cast<long long>(b) * a.R + i) * a.Hkv + kvh) * kDim + c * 8) =
            *reinterpret_cast<const uint4*>(smem + C::kOffNewK + swz(i, c, C::kNewHalf));
    }
  }
  // no CTA-wide barrier at the end: every warp leaves when its own work is done
}

// ------------------------------------------------------------------ host
template <int kR, int kDim, bool kSplitWeights>
bool set_attributes(const int* sizes, int n, int* active) {
  // (head dim 64 layers run as the rotation, append and attention kernels)
  const void* kerns[2] = {reinterpret_cast<const void*>(verify_wide_kernel<kR, kDim, false, kSplitWeights>),
                          reinterpret_cast<const void*>(verify_wide_kernel<kR, kDim, kDim == 128, kSplitWeights>)};
  constexpr int smem = Cfg<kR, kDim, kSplitWeights>::kSmemBytes;
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
    if (cudaOccupancyMaxActiveClusters(&m, kerns[0], &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      m = 0;
    }
    active[i] = m;
  }
  return true;
}

template <int kR, int kDim, bool kFused, bool kSplitWeights>
sd_status launch(const sd_kv_cache* cache, const TcArgs& a, const RopeTable& tab, int cs, cudaStream_t stream) {
  const int B = cache->batch, Hkv = cache->n_kv_heads, cap = cache->capacity;
  CUtensorMap k128, v128;
  if (!make_map(&k128, cache->k, cap, B * Hkv, 128, kDim) || !make_map(&v128, cache->v, cap, B * Hkv, 128, kDim))
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
  cfg.dynamicSmemBytes = Cfg<kR, kDim, kSplitWeights>::kSmemBytes;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, verify_wide_kernel<kR, kDim, kFused, kSplitWeights>, k128, v128, a, tab) != cudaSuccess) {
    (void)cudaGetLastError();
    return SD_ERR_CUDA;
  }
  return SD_OK;
}

template <int kDim, bool kFused>
sd_status launch_rows(const sd_kv_cache* cache, const TcArgs& a, const RopeTable& tab, int rows, bool split, int cs,
                      cudaStream_t stream) {
  constexpr bool kAll = kDim == 64;  // two terms on every tile
  if (rows == 32) return launch<32, kDim, kFused, kAll>(cache, a, tab, cs, stream);
  if (rows == 48 && split) return launch<48, kDim, kFused, true>(cache, a, tab, cs, stream);
  if (rows == 48) return launch<48, kDim, kFused, kAll>(cache, a, tab, cs, stream);
  if (rows == 64) return launch<64, kDim, kFused, kAll>(cache, a, tab, cs, stream);
  return launch<80, kDim, kFused, kAll>(cache, a, tab, cs, stream);
}

template <int kDim>
bool active_of(int rows, const int* sizes, int n, int* active) {
  constexpr bool kAll = kDim == 64;
  if (rows == 32) return set_attributes<32, kDim, kAll>(sizes, n, active);
  if (rows == 48) return set_attributes<48, kDim, true>(sizes, n, active) && set_attributes<48, kDim, kAll>(sizes, n, active);
  if (rows == 64) return set_attributes<64, kDim, kAll>(sizes, n, active);
  return set_attributes<80, kDim, kAll>(sizes, n, active);
}

}  // namespace

bool sd_internal_wide_active(int rows, int D, const int* sizes, int n, int* active) {
  return D == 64 ? active_of<64>(rows, sizes, n, active) : active_of<128>(rows, sizes, n, active);
}

sd_status sd_internal_wide_launch(const sd_kv_cache* cache, const TcArgs& a, const RopeTable& tab, int rows, bool split,
                                  int cs, bool fused, cudaStream_t stream) {
  if (cache->head_dim == 64) return launch_rows<64, false>(cache, a, tab, rows, split, cs, stream);
  return fused ? launch_rows<128, true>(cache, a, tab, rows, split, cs, stream)
               : launch_rows<128, false>(cache, a, tab, rows, split, cs, stream);
}
