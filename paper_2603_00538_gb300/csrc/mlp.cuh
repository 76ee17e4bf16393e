// The surrogate source network: x in R^3 -> 256 -> 256 -> 256 -> 256 -> 1
// with SiLU, BF16 weights of the three 256x256 layers and BF16 hidden
// activations, FP32 accumulation in tensor memory. Device pieces shared by
// the forward kernel and the training kernels (the network pass of a surrogate
// transfer runs the forward).
//
// Parameter vector (FP32, kNParam): W1 [256][3], c1 [256], W2 [256][256],
// c2, W3, c3, W4, c4, w5 [256], c5 [1]; weights row-major [out][in].
#pragma once
#include <cuda_bf16.h>
#include "internal.hpp"
#include "tc.cuh"
#include "util.cuh"

namespace sft {

constexpr int kH = 256;
constexpr int kTileM = 128;
constexpr int kKF = 16;  // K of one MMA
constexpr int kTPR = 2;  // forward tile: threads per activation row (each owns half of the columns)
constexpr int64_t kOffW1 = 0, kOffC1 = kH * 3, kOffW2 = kOffC1 + kH, kOffC2 = kOffW2 + kH * kH,
                  kOffW3 = kOffC2 + kH, kOffC3 = kOffW3 + kH * kH, kOffW4 = kOffC3 + kH,
                  kOffC4 = kOffW4 + kH * kH, kOffW5 = kOffC4 + kH, kOffC5 = kOffW5 + kH,
                  kNParam = kOffC5 + 1;

constexpr uint32_t kSmemA = kTileM * kH * 2;        // 64 KiB: activation tile (128 x 256 BF16)
constexpr uint32_t kSmemBF = kH * kKF * 2;          // 8 KiB: weights of one MMA (256 x 16 BF16)
constexpr uint32_t kSmemW1 = kH * 16;               // 4 KiB: first layer (w1_table_entry)
constexpr uint32_t kSmemBias = 4 * kH * 4;          // 4 KiB: c2, c3, c4, w5

// byte offset of weight (n, k) of a 256x256 layer in the chunked layout the
// forward tile streams: chunk k / kKF is one contiguous [256][kKF] block in
// the no-swizzle K-major core-matrix order of its shared-memory image
__host__ __device__ constexpr uint32_t wchunk_offset(int n, int k) {
  return (uint32_t)(k / kKF) * kSmemBF + tc::kmajor_offset(n, k % kKF, kKF);
}
constexpr uint32_t kIdesc = tc::idesc_bf16_f32(kTileM, kH);

// special-function-unit approximations (PTX ex2.approx / rcp.approx):
// relative errors near 2^-22, far below the BF16 rounding of an activation
__device__ __forceinline__ float ex2_sfu(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_sfu(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
constexpr float kNegLog2e = -1.4426950408889634f;
// sigma(z) = 1 / (1 + 2^(-z log2 e)); the limits are exact: 2^(+big) = inf
// gives 1/inf = 0, 2^(-big) = 0 gives 1. (The one-operation form
// u + u tanh(u), u = z/2, loses accuracy to cancellation for z << 0: its
// absolute error |u| 2^-11 exceeds the BF16 rounding of the activation.)
__device__ __forceinline__ float sigmoid_f(float z) { return rcp_sfu(1.0f + ex2_sfu(kNegLog2e * z)); }
// d silu / dz = sigma(z) (1 + z (1 - sigma(z)))
__device__ __forceinline__ float silu_grad(float z) {
  const float sg = sigmoid_f(z);
  return sg * __fmaf_rn(z, 1.0f - sg, 1.0f);
}

// The first layer in shared memory, pair-interleaved for the packed FMAs:
// outputs 2m and 2m + 1 take entries 2m = {W1[2m][0], W1[2m+1][0], W1[2m][1],
// W1[2m+1][1]} and 2m + 1 = {W1[2m][2], W1[2m+1][2], c1[2m], c1[2m+1]}.
__device__ __forceinline__ void w1_table_entry(float4* w1, const float* __restrict__ P, int o) {
  const int m = o >> 1, odd = o & 1;
  float* e0 = reinterpret_cast<float*>(w1 + 2 * m);
  float* e1 = reinterpret_cast<float*>(w1 + 2 * m + 1);
  e0[odd] = __ldg(P + kOffW1 + o * 3);
  e0[2 + odd] = __ldg(P + kOffW1 + o * 3 + 1);
  e1[odd] = __ldg(P + kOffW1 + o * 3 + 2);
  e1[2 + odd] = __ldg(P + kOffC1 + o);
}
// ---------------------------------------------------------------------------
// The forward pass on 128-row tiles: one CTA per SM, two groups of 256
// threads (two threads a row, half of the columns each). Each group runs its
// own tiles with its own activation tile, TMEM accumulator (columns 256 g ..
// +255) and named barrier: layer 1 (3 -> 256) on the FMA pipe into the BF16
// activation tile, three 256x256 layers on the tensor cores with bias + SiLU
// epilogues from TMEM, the last layer (256 -> 1) as FMA chains over each half of
// the columns beside the last epilogue, the halves added in a fixed order. The
// two groups' layers take turns on the tensor cores in a fixed order - tile
// pair j: T0 L1, T1 L1, T0 L2, T1 L2, T0 L3, T1 L3; a group without a partner
// tile at the end runs its layers alone - so one group's epilogue overlaps the
// other's MMAs, and both read one ring of kRing weight chunks (64 wide in K:
// four MMAs each) fed in that order (chunk c = 4 s + k: K-slice k of the layer
// of slot s). Per slot 1 + kRing warps of its group work at once: warp 0
// issues the MMAs as their chunks land, and warp 1 + b refills buffer b as
// soon as the MMAs that read it complete (the chunk kRing ahead); each is a
// converged warp with one elected lane (a lone thread in a divergent branch
// took about 100 cycles an MMA). Turn counters in shared memory (bounded
// waits) keep the slots' MMA issue and each buffer's copies in slot order, so
// every mbarrier phase is waited only after the phase before it completed.
//
// What bounds it: the chain of a group's phases. A tile takes 131 k
// activations, each two special-function operations (some 12 k cycles of an
// SM) and about 8 issue slots, and 6.1 k cycles of MMA; a group's tile passes
// through layer 1 (5 k cycles), three MMA phases (3.5 k) and three epilogues
// (4.3 k), and two groups a SM overlap to 17 k cycles a tile (a third
// accumulator does not fit in TMEM). 1.536 M points: 1,157 us (two CTAs of one
// tile each, one thread issuing MMAs and copies, 16-wide chunks, broadcast
// bias loads) -> 763 (two groups taking turns, every operation over 16 columns
// at a time) -> 747 (accumulator fragments, output layer inside the epilogue)
// -> 711 (64-wide chunks) -> 707 us (elected lanes) = 0.86 PFLOP/s, 0.46 of
// the measured BF16 burst rate. Measured and dropped: 512 threads a group, 5 or
// 7 smaller ring buffers, one copier warp, every thread polling the layer's
// mbarrier (770 us: the polls slow the issuer).
// ---------------------------------------------------------------------------
constexpr int kChunkK = 64;                     // K of a ring chunk
constexpr uint32_t kChunkBytes = kH * kChunkK * 2;
constexpr int kChunks = kH / kChunkK;           // chunks per layer
constexpr int kRing = 2;                        // chunk buffers
constexpr int kGroupThreads = kTPR * kTileM;    // 256
constexpr uint32_t kSmemBars = 256;             // mbarriers, TMEM slot, failed flag, turn counters, stream state
constexpr uint32_t kSmemYH = 2 * kTileM * 4;    // partial outputs of the column halves
constexpr uint32_t kSmemFwd = 2 * kSmemA + kRing * kChunkBytes + kSmemW1 + kSmemBias + 2 * kSmemYH + kSmemBars;
static_assert(kRing <= kChunks && 32 * kRing < kGroupThreads, "ring size");
static_assert(kSmemFwd <= 227u * 1024u, "forward tile exceeds the shared memory of one CTA");

struct FwdStream {
  int32_t total;             // chunks of the CTA's stream
  int32_t tail0;             // first slot of the unpaired tile (2 x layers x the paired tiles of a group)
  int32_t next_use;          // chunks whose MMAs were issued
  int32_t next_copy[kRing];  // the next chunk copied into each buffer
};

struct FwdSmem {
  unsigned char* A;   // [2] activation tiles
  unsigned char* B;   // kRing weight chunk buffers
  float4* w1;         // first layer, pair-interleaved (w1_table_entry)
  float* bias;        // [4][256]: c2, c3, c4 and the output weights w5
  float* ypart;       // [2][2][128] partial outputs of each group's column halves
  uint64_t* full;     // [kRing] chunk landed (bulk-copy transaction bytes)
  uint64_t* mdone;    // [kRing] MMAs reading the chunk completed
  uint64_t* lbar;     // [2] all MMAs of a group's layer completed
  uint32_t* slot;     // TMEM base address
  volatile int* failed;  // a wait expired: nothing is issued or waited for any more
  volatile int* issued;  // layer slots whose MMAs were issued
  volatile int* copied;  // [kRing] layer slots whose copies into each buffer were issued
  FwdStream* st;
};
__device__ __forceinline__ FwdSmem fwd_smem(unsigned char* sm) {
  FwdSmem S;
  S.A = sm;
  S.B = sm + 2 * kSmemA;
  unsigned char* q = S.B + kRing * kChunkBytes;
  S.w1 = reinterpret_cast<float4*>(q);
  q += kSmemW1;
  S.bias = reinterpret_cast<float*>(q);
  q += kSmemBias;
  S.ypart = reinterpret_cast<float*>(q);
  q += 2 * kSmemYH;
  S.full = reinterpret_cast<uint64_t*>(q);
  S.mdone = S.full + kRing;
  S.lbar = S.mdone + kRing;
  S.slot = reinterpret_cast<uint32_t*>(S.lbar + 2);
  S.failed = reinterpret_cast<volatile int*>(S.slot + 1);
  S.issued = S.failed + 1;
  S.copied = S.issued + 1;
  S.st = reinterpret_cast<FwdStream*>(q + 192);
  return S;
}
static_assert(2 * kRing * 8 + 2 * 8 + 4 + 4 + 4 + 4 * kRing <= 192,
              "barrier block overlaps the stream state");
static_assert(192 + sizeof(FwdStream) <= kSmemBars, "stream state outside its block");

__device__ __forceinline__ void group_sync(int grp) {
  if (grp == 0) asm volatile("bar.sync 1, %0;" ::"n"(kGroupThreads) : "memory");
  else asm volatile("bar.sync 2, %0;" ::"n"(kGroupThreads) : "memory");
}

// Bounded waits of the forward kernel. One that runs out sets *err and the
// CTA's failed flag; from then on every wait returns at once and no copy or
// MMA is issued, so the threads run through their loops, meet at the same
// barriers, and leave together. The lanes of a warp each see for themselves
// whether a wait ended or ran out and may differ at the limit, so nothing that
// the whole warp has to take part in stands between the first wait of an issuing
// or copying warp and the end of its work in the slot. (A vote of the lanes after
// every wait instead: 1,812 us against 1,798 for 4.2 M points.)
__device__ __forceinline__ bool turn_wait(const FwdSmem& S, volatile int* ctr, int v, int32_t* err) {
  if (*ctr == v) return true;
  const uint64_t t0 = globaltimer_ns();
  while (*ctr != v) {
    if (*S.failed) return false;
    if (globaltimer_ns() - t0 > kDefaultWaitNs) {
      set_error(err, DEV_BARRIER_TIMEOUT);
      *S.failed = 1;
      return false;
    }
    __nanosleep(32);
  }
  return true;
}
__device__ __forceinline__ bool fwd_wait(const FwdSmem& S, uint64_t* bar, uint32_t parity, int32_t* err) {
  if (tc::mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  while (!tc::mbar_try_wait(bar, parity)) {
    if (*S.failed) return false;
    if (globaltimer_ns() - t0 > kDefaultWaitNs) {
      set_error(err, DEV_BARRIER_TIMEOUT);
      *S.failed = 1;
      return false;
    }
  }
  return true;
}

// the chunked weights of the NL tensor-core layers of a tile, in their order
template <int NL>
struct LayerWeights {
  const unsigned char* w[NL];
  // layer l (selects, not an indexed local array)
  __device__ __forceinline__ const unsigned char* of(int l) const {
    const unsigned char* r = w[0];
#pragma unroll
    for (int q = 1; q < NL; ++q) r = l == q ? w[q] : r;
    return r;
  }
  // layer of slot s in the two-group order
  __device__ __forceinline__ const unsigned char* of_slot(int s, int tail0) const {
    return of(s < tail0 ? (s % (2 * NL)) >> 1 : (s - tail0) % NL);
  }
};
__device__ __forceinline__ void copy_chunk(const FwdSmem& S, const unsigned char* layer_w, int c) {
  const int b = c % kRing;
  tc::mbar_arrive_expect_tx(S.full + b, kChunkBytes);
  tc::bulk_g2s(S.B + (size_t)b * kChunkBytes, layer_w + (size_t)(c & (kChunks - 1)) * kChunkBytes, kChunkBytes,
               S.full + b);
}

// tiles a persistent CTA visits (tile = blockIdx.x + k gridDim.x < ntiles)
__device__ __forceinline__ int64_t cta_tiles(int64_t ntiles) {
  return blockIdx.x < ntiles ? (ntiles - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
}

// Setup over the CTA's tiles, split between the groups (group 0 the even
// ones): TMEM (512 columns), mbarriers, the stream state and its first kRing
// copies, the first-layer table. Every thread calls it.
template <int NL>
__device__ __forceinline__ uint32_t fwd_setup(const FwdSmem& S, const float* __restrict__ P, const LayerWeights<NL>& Wc,
                                              int64_t tiles) {
  if ((threadIdx.x >> 5) == 0) {
    tc::tmem_alloc(S.slot, 2 * kH);
    tc::tmem_relinquish();
  }
  if (threadIdx.x == 0) {
    for (int b = 0; b < kRing; ++b) {
      tc::mbar_init(S.full + b, 1);
      tc::mbar_init(S.mdone + b, 1);
    }
    tc::mbar_init(S.lbar, 1);
    tc::mbar_init(S.lbar + 1, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    FwdStream& st = *S.st;
    st.total = (int32_t)(tiles * NL * kChunks);
    st.tail0 = (int32_t)(2 * NL * (tiles / 2));
    st.next_use = 0;
    *S.issued = 0;
    *S.failed = 0;
    const unsigned char* w0 = Wc.of_slot(0, st.tail0);
    for (int c = 0; c < kRing; ++c) {
      S.copied[c] = 0;
      st.next_copy[c] = c;
      if (c < st.total) {
        copy_chunk(S, w0, c);
        st.next_copy[c] = c + kRing;
      }
    }
  }
  for (int o = threadIdx.x; o < kH; o += blockDim.x) {
    w1_table_entry(S.w1, P, o);
    S.bias[o] = __ldg(P + kOffC2 + o);
    S.bias[kH + o] = __ldg(P + kOffC3 + o);
    S.bias[2 * kH + o] = __ldg(P + kOffC4 + o);
    S.bias[3 * kH + o] = __ldg(P + kOffW5 + o);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  return *S.slot;
}

// End of both groups' tile loops (every thread calls it): thread 0 waits
// (bounded) for copies that no MMA consumed, then TMEM is released.
__device__ __forceinline__ void fwd_teardown(const FwdSmem& S, uint32_t taddr, int32_t* err) {
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (threadIdx.x == 0) {
    const FwdStream& st = *S.st;
    int hi = 0;
    for (int q = 0; q < kRing; ++q) hi = max(hi, st.next_copy[q]);
    for (int c = st.next_use; c < hi; ++c)
      if (c < st.next_copy[c % kRing] &&
          !tc::mbar_wait(S.full + (c % kRing), ((uint32_t)c / kRing) & 1u, err, 200000000ull))
        break;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if ((threadIdx.x >> 5) == 0) tc::tmem_dealloc(taddr, 2 * kH);
}

// MMAs of layer slot `slot` (group grp's warp 0): after the previous slot's
// MMAs were issued, the MMAs of each chunk as it lands, a commit per chunk
// (mdone: its buffer may be refilled) and one for the layer (lbar[grp]).
__device__ __forceinline__ void layer_issue(const FwdSmem& S, int grp, uint32_t taddr_g, int slot, int32_t* err) {
  const uint64_t a0 = tc::smem_desc(tc::smem_addr(S.A + grp * kSmemA), 128u, (uint32_t)kH * 16u);
  const uint64_t b0 = tc::smem_desc(tc::smem_addr(S.B), 128u, (uint32_t)kKF * 16u);
  const int c0 = slot * kChunks;
  const bool leader = tc::elect_one();
  if (!turn_wait(S, S.issued, slot, err)) return;
  __threadfence_block();
  tc::fence_after_sync();
#pragma unroll 1
  for (int kc = 0; kc < kChunks; ++kc) {
    const int c = c0 + kc;
    const int b = c % kRing;
    if (!fwd_wait(S, S.full + b, ((uint32_t)c / kRing) & 1u, err)) return;
    if (leader) {
#pragma unroll
      for (int m = 0; m < kChunkK / kKF; ++m) {
        // descriptor start addresses in 16-byte units: the MMA's K-slice of A
        // is 256 bytes on, its weights kSmemBF bytes on
        const int k = kc * (kChunkK / kKF) + m;
        tc::mma_bf16(taddr_g, a0 + (uint64_t)(k * (kKF * 16 / 16)),
                     b0 + (uint64_t)(b * (kChunkBytes / 16) + m * (kSmemBF / 16)), kIdesc, k != 0);
      }
      tc::mma_commit(S.mdone + b);
      if (kc == kChunks - 1) tc::mma_commit(S.lbar + grp);
    }
  }
  if (leader) {
    S.st->next_use = c0 + kChunks;
    __threadfence_block();
    *S.issued = slot + 1;
  }
}

// Refills of buffer b during layer slot `slot` (group grp's warp 1 + b):
// after the previous slot's, chunk u + kRing into the buffer as soon as the
// MMAs of chunk u (u in this slot) completed.
template <int NL>
__device__ __forceinline__ void refill_buffer(const FwdSmem& S, const LayerWeights<NL>& Wc, int slot, int b,
                                              int32_t* err) {
  const bool leader = tc::elect_one();
  if (!turn_wait(S, S.copied + b, slot, err)) return;
  __threadfence_block();
  FwdStream& st = *S.st;
  const int c0 = slot * kChunks;
  const int total = st.total;
  // chunks c0 + kRing .. belong to this slot's layer, the last to the next slot's
  const unsigned char* w_this = Wc.of_slot(slot, st.tail0);
  const unsigned char* w_next = Wc.of_slot(slot + 1, st.tail0);
  for (int kc = (b + kRing - c0 % kRing) % kRing; kc < kChunks; kc += kRing) {
    const int u = c0 + kc;  // the chunk whose buffer the next one reuses
    const int c = u + kRing;
    if (c >= total) break;
    if (!fwd_wait(S, S.mdone + b, ((uint32_t)u / kRing) & 1u, err)) return;
    if (leader) {
      copy_chunk(S, kc + kRing < kChunks ? w_this : w_next, c);
      st.next_copy[b] = c + kRing;
    }
  }
  if (leader) {
    __threadfence_block();
    S.copied[b] = slot + 1;
  }
}

// SiLU z sigma(z) of N pairs, rounded to BF16 pairs: each operation over all
// pairs (f2_*: common.cuh) before the next, so the special-function latencies
// overlap
template <int N>
__device__ __forceinline__ void silu_pairs(const uint64_t (&z)[N], uint32_t (&h)[N]) {
  float t[2 * N];
#pragma unroll
  for (int i = 0; i < N; ++i) f2_unpack(f2_mul(z[i], f2_pack(kNegLog2e, kNegLog2e)), t[2 * i], t[2 * i + 1]);
#pragma unroll
  for (int i = 0; i < 2 * N; ++i) t[i] = ex2_sfu(t[i]);
#pragma unroll
  for (int i = 0; i < N; ++i)
    f2_unpack(f2_add(f2_pack(1.0f, 1.0f), f2_pack(t[2 * i], t[2 * i + 1])), t[2 * i], t[2 * i + 1]);
#pragma unroll
  for (int i = 0; i < 2 * N; ++i) t[i] = rcp_sfu(t[i]);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    float h0, h1;
    f2_unpack(f2_mul(z[i], f2_pack(t[2 * i], t[2 * i + 1])), h0, h1);
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h[i]) : "f"(h1), "f"(h0));
  }
}

// A thread's place in its group's tile. Accumulator fragments (16 rows x 8
// columns over a warp): a lane holds two neighbouring columns 2 (l % 4) of
// rows l / 4 and l / 4 + 8, so it needs a quarter of the warp's biases, not
// all of them, and its BF16 pairs go to the activation tile by stmatrix. (With
// one row and 16 columns a thread, every bias and first-layer weight was a
// broadcast 16-byte load: the loads took 6.1 k of the 13.4 k shared-memory
// cycles of a tile.)
struct TileLane {
  static constexpr int kCols = kH / kTPR;
  int grp, lt, lane, warp;
  int w0;              // first of the warp's 32 rows
  int c0;              // first of its 128 columns
  uint32_t tcol, tw;   // TMEM: the group's accumulator, the warp's part of it
  unsigned char* A;    // the group's activation tile
  // the lane's row of the four 8x8 matrices of a store or load: matrices (rows
  // 0-7, block i), (rows 8-15, i), (rows 0-7, i + 1), (rows 8-15, i + 1)
  uint32_t a_st;
  static constexpr uint32_t kHalfRows = 2u * kH * 16u;  // 16 rows on
};
__device__ __forceinline__ TileLane tile_lane(const FwdSmem& S, uint32_t taddr) {
  TileLane t;
  t.grp = threadIdx.x / kGroupThreads;
  t.lt = threadIdx.x - t.grp * kGroupThreads;
  t.lane = t.lt & 31;
  t.warp = __shfl_sync(0xffffffffu, t.lt >> 5, 0);
  t.w0 = t.lt & 96;
  t.c0 = (t.lt / kTileM) * TileLane::kCols;
  t.tcol = taddr + (uint32_t)(t.grp * kH);
  t.tw = t.tcol + ((uint32_t)t.w0 << 16) + (uint32_t)t.c0;
  t.A = S.A + t.grp * kSmemA;
  t.a_st = tc::smem_addr(t.A) + (uint32_t)((t.w0 >> 3) + ((t.lane >> 3) & 1)) * (kH * 16) +
           (uint32_t)((t.c0 >> 3) + (t.lane >> 4)) * 128u + (uint32_t)(t.lane & 7) * 16u;
  return t;
}

// layer 1 of rows l / 4 + 8 q of the warp (inputs x[q]) into the activation tile
__device__ __forceinline__ void tile_layer1(const FwdSmem& S, const TileLane& t, const float (&x)[4][3]) {
  const float4* w1 = S.w1 + t.c0 + 2 * (t.lane & 3);
#pragma unroll 2
  for (int i = 0; i < TileLane::kCols / 8; i += 2) {
    uint64_t z[8];
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float4 a = w1[8 * (i + u)], b = w1[8 * (i + u) + 1];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        z[4 * (q >> 1) + 2 * u + (q & 1)] =
            f2_fma(f2_pack(b.x, b.y), f2_pack(x[q][2], x[q][2]),
                   f2_fma(f2_pack(a.z, a.w), f2_pack(x[q][1], x[q][1]),
                          f2_fma(f2_pack(a.x, a.y), f2_pack(x[q][0], x[q][0]), f2_pack(b.z, b.w))));
    }
    uint32_t h[8];
    silu_pairs<8>(z, h);
    tc::stmatrix4(t.a_st + (uint32_t)i * 128u, h[0], h[1], h[2], h[3]);
    tc::stmatrix4(t.a_st + (uint32_t)i * 128u + TileLane::kHalfRows, h[4], h[5], h[6], h[7]);
  }
}

// the activation tile is written: make it visible to the tensor cores
__device__ __forceinline__ void tile_written(const TileLane& t) {
  tc::fence_async_smem();
  tc::fence_before_sync();
  group_sync(t.grp);
  tc::fence_after_sync();
}

// One tensor-core layer of the group's tile: warp 0 issues, warps 1 .. kRing
// refill the ring, other(t) runs on the last warp; all meet when the layer's
// MMAs are complete. (The others wait at the barrier: 256 threads polling lbar
// slowed the issue from 3.9 k to 5.3 k cycles a layer.)
template <int NL, class Other>
__device__ __forceinline__ void tile_mma(const FwdSmem& S, const TileLane& t, const LayerWeights<NL>& Wc, int slot,
                                         uint32_t& lphase, int32_t* err, Other&& other) {
  static_assert(kRing < kGroupThreads / 32 - 1, "a warp per role");
  if (t.warp == 0) {
    layer_issue(S, t.grp, t.tcol, slot, err);
    fwd_wait(S, S.lbar + t.grp, lphase, err);
    lphase ^= 1u;
    __syncwarp();
  } else if (t.warp <= kRing) {
    refill_buffer<NL>(S, Wc, slot, t.warp - 1, err);
    __syncwarp();
  } else if (t.warp == kGroupThreads / 32 - 1) {
    other();
  }
  group_sync(t.grp);
  tc::fence_after_sync();
}

// f(cc, hh, r): accumulator fragments of columns cc .. cc + 31 of the warp's,
// rows 16 hh .. 16 hh + 15 (r as tc::tmem_ld_16x256_x4), the next loads in
// flight meanwhile; pre(cc) before the wait for the first of them (bias loads)
template <class Pre, class F>
__device__ __forceinline__ void tile_fragments(const TileLane& t, Pre&& pre, F&& f) {
  uint32_t ra[16], rb[16];
  tc::tmem_ld_16x256_x4(t.tw, ra);
#pragma unroll
  for (int cc = 0; cc < TileLane::kCols; cc += 32) {
    pre(cc);
    tc::tmem_ld_wait();
    tc::tmem_ld_16x256_x4(t.tw + (16u << 16) + (uint32_t)cc, rb);
    f(cc, 0, ra);
    tc::tmem_ld_wait();
    if (cc + 32 < TileLane::kCols) tc::tmem_ld_16x256_x4(t.tw + (uint32_t)(cc + 32), ra);
    f(cc, 1, rb);
  }
}

// the lane's biases of 32 columns (bias: the layer's, at the first of them)
__device__ __forceinline__ void load_bias(const TileLane& t, const float* bias, uint64_t (&bb)[4]) {
  const float2* b2 = reinterpret_cast<const float2*>(bias) + (t.lane & 3);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 b = b2[4 * i];
    bb[i] = f2_pack(b.x, b.y);
  }
}
// acc + bias of eight column pairs
__device__ __forceinline__ void add_bias(const uint64_t (&bb)[4], const uint32_t (&r)[16], uint64_t (&z)[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i)
    z[i] = f2_add(f2_pack(__uint_as_float(r[2 * i]), __uint_as_float(r[2 * i + 1])), bb[i >> 1]);
}

// store of one fragment set to the activation tile
__device__ __forceinline__ void put_fragments(const TileLane& t, int cc, int hh, const uint32_t (&h)[8]) {
  const uint32_t ad = t.a_st + (uint32_t)cc * 16u + (hh ? TileLane::kHalfRows : 0u);
  tc::stmatrix4(ad, h[0], h[1], h[2], h[3]);
  tc::stmatrix4(ad + 256u, h[4], h[5], h[6], h[7]);
}

// inputs of rows l / 4 + 8 q of the warp's 32 in the tile that starts at point `first`
__device__ __forceinline__ void tile_inputs(const TileLane& t, const float* __restrict__ pts, int64_t first, int64_t n,
                                            float (&x)[4][3]) {
  const int64_t i0 = first + t.w0 + (t.lane >> 2);
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int a = 0; a < 3; ++a) x[q][a] = i0 + 8 * q < n ? __ldg(pts + (i0 + 8 * q) * 3 + a) : 0.f;
}

// The network on the group's 128-row tile: layer slots slot0, slot0 + step,
// slot0 + 2 step. Lane l of each warp passes the inputs of rows l / 4 + 8 q
// (q = 0..3) of its 32 rows; threads lt < 128 get row lt's output. next() is
// called when the inputs are no longer needed.
template <class Next>
__device__ __forceinline__ void fwd_tile(const FwdSmem& S, const TileLane& t, const float* __restrict__ P,
                                         const LayerWeights<3>& Wc, const float (&x)[4][3], uint32_t& lphase,
                                         int64_t slot0, int step, int32_t* err, float& y_out, Next&& next) {
  float* ypart = S.ypart + t.grp * 2 * kTileM;
  tile_layer1(S, t, x);
  tile_written(t);
  float y = 0.f;
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    tile_mma<3>(S, t, Wc, (int)(slot0 + (int64_t)l * step), lphase, err, [] {});
    uint64_t bb[4];
    tile_fragments(t, [&](int cc) { load_bias(t, S.bias + l * kH + t.c0 + cc, bb); },
                   [&](int cc, int hh, const uint32_t (&r)[16]) {
      uint64_t z[8];
      uint32_t h[8];
      add_bias(bb, r, z);
      silu_pairs<8>(z, h);
      put_fragments(t, cc, hh, h);
      if (l == 2 && hh == 1) {
        // 256 -> 1: the warp's rows and columns are one half of 32 rows, so
        // lane r runs row r's FMA chain over the columns as they come
        __syncwarp();
#pragma unroll
        for (int k = cc; k < cc + 32; k += 8) {
          const uint4 a = *reinterpret_cast<const uint4*>(t.A + tc::kmajor_offset(t.w0 + t.lane, t.c0 + k, kH));
          const uint32_t u[4] = {a.x, a.y, a.z, a.w};
          const float4* w4 = reinterpret_cast<const float4*>(S.bias + 3 * kH + t.c0 + k);
          const float4 wa = w4[0], wb = w4[1];
          const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            y = __fmaf_rn(__uint_as_float(u[i] << 16), w[2 * i], y);
            y = __fmaf_rn(__uint_as_float(u[i] & 0xFFFF0000u), w[2 * i + 1], y);
          }
        }
      }
    });
    if (l == 1) next();
    if (l == 2) ypart[t.lt] = y;
    tile_written(t);
  }
  // the halves added in a fixed order
  y_out = 0.f;
  if (t.lt < kTileM) y_out = ypart[t.lt] + ypart[kTileM + t.lt] + __ldg(P + kOffC5);
}

}  // namespace sft

struct sft_mlp_s {
  float* P = nullptr;                                  // FP32 parameters (master)
  unsigned char* Wc[3] = {nullptr, nullptr, nullptr};   // BF16 W2, W3, W4 in the tile's chunked layout
  unsigned char* WTc[3] = {nullptr, nullptr, nullptr};  // BF16 transposes in the same layout (the backward pass)
  float* grad = nullptr;                               // FP32 gradient of the mean loss
  float* m1 = nullptr;                                 // Adam moments
  float* m2 = nullptr;
  int64_t step = 0;
  cudaStream_t stream = nullptr;
};

namespace sft {
sft_status mlp_forward_dev(sft_mlp_s* m, int64_t n, const float* pts, float* out, cudaStream_t st, int32_t* d_err);
}  // namespace sft
