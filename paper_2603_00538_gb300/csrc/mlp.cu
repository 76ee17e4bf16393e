// The surrogate source network: a learned black-box
// field x in R^3 -> 256 -> 256 -> 256 -> 256 -> 1 with SiLU, BF16 weights of
// the three 256x256 layers and BF16 hidden activations, FP32 accumulation.
// The 256x256 layers run on the 5th-generation tensor cores (tcgen05.mma,
// accumulators in tensor memory); the 3->256 and 256->1 layers are FP32 FMA.
//
// Parameter vector (FP32, MLP_NPARAM): W1 [256][3], c1 [256], W2 [256][256],
// c2, W3, c3, W4, c4, w5 [256], c5 [1]; weights row-major [out][in].
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>
#include "mlp.cuh"

namespace sft {

// Forward of the network on n points (x,y,z) [n][3] FP32 -> out [n] FP32:
// persistent CTAs (one per SM) of two groups that alternate on the tensor
// cores (fwd_tile).
__global__ void __launch_bounds__(2 * kGroupThreads, 1) k_mlp_forward(const float* __restrict__ P,
                                                                     const unsigned char* __restrict__ W2,
                                                                     const unsigned char* __restrict__ W3,
                                                                     const unsigned char* __restrict__ W4, int64_t n,
                                                                     const float* __restrict__ pts,
                                                                     float* __restrict__ out, int32_t* err) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const FwdSmem S = fwd_smem(sm);
  const LayerWeights<3> Wc{{W2, W3, W4}};
  const int64_t tiles = cta_tiles((n + kTileM - 1) / kTileM);
  const uint32_t taddr = fwd_setup<3>(S, P, Wc, tiles);
  const TileLane t = tile_lane(S, taddr);
  const int64_t J1 = tiles / 2;  // tiles of each group that have a partner
  uint32_t lphase = 0;
  float x[4][3];
  auto first = [&](int64_t k) { return (blockIdx.x + k * gridDim.x) * kTileM; };
  tile_inputs(t, pts, first(t.grp), n, x);
  for (int64_t k = t.grp; k < tiles; k += 2) {
    const int64_t gi = first(k) + t.lt;
    const int64_t j = k / 2;
    float y;
    // the next tile's inputs load during this tile's last layer
    fwd_tile(S, t, P, Wc, x, lphase, j < J1 ? 6 * j + t.grp : 6 * J1, j < J1 ? 2 : 1, err, y,
             [&] { tile_inputs(t, pts, first(k + 2), k + 2 < tiles ? n : 0, x); });
    if (t.lt < kTileM && gi < n) out[gi] = y;
  }
  fwd_teardown(S, taddr, err);
}

// ---------------------------------------------------------------------------
// Training: the gradient of the mean squared error in two kernels.
//
// k_train_tile runs the whole forward and backward pass of a 128-row tile on
// the forward's machinery (two groups per CTA that take turns on the tensor
// cores, one ring of weight chunks; six layers a tile): layer 1, three layers
// with z = acc + bias, h = SiLU(z); the output y = w5 . h4 + c5 and
// dL/dy = 2 (y - t) / n_total; dz4 = dy w5 SiLU'(z4) from the accumulators of
// layer 4; dz3, dz2, dz1 = (dz W) SiLU'(z) against the transposed weights. z2
// and z3 are kept in BF16 in the group's global buffer, by the thread that
// reads them back; z1 is formed again. The bias and output-weight gradients
// and the first layer's are column sums of the fragments at hand (shuffles,
// then sums in shared memory over the CTA's tiles). Each activation tile
// (h1, h2, h3, dz4, dz3, dz2) is copied out as it stands when its layer's MMAs
// start, one bulk copy of 64 KB.
//
// k_train_dw forms dW = dz^T h of the three square layers: the copied tiles
// are K-major operands of the tile's MMAs, and the same bytes are MN-major
// operands with the batch rows as K, so nothing is transposed. A CTA keeps a
// 256 x 256 FP32 result in all of TMEM over its share of the tiles (rows
// streamed 32 at a time through a ring) and adds it into the gradient once.
//
// What bounds them: k_train_tile the epilogues, as the forward (eight of them a
// tile with two special-function operations an activation each; 158 us at
// 70,001 points), k_train_dw the operand copies (128 KB a tile and layer, 61
// us). Separate layer, GEMM, column-sum and head kernels over row-major and
// transposed copies of every array took 0.6 ms per 16,384 points (two-byte
// stores 512 bytes apart in the first layer, atomics 1 KB apart in the split
// weight gradient, one CTA of 128 threads per SM): loss and gradient of 70,001
// points 3.20 ms, now 0.27.
// ---------------------------------------------------------------------------
constexpr int kTrainLayers = 6;
constexpr int kTrainImages = 6;                 // h1, h2, h3, dz4, dz3, dz2
// tiles per pass over the two kernels: four a SM, 240 MB of images (half as many: 313 us against 274 at
// 70,001 points). 77,824 points are one pass: 309 us a call, 78,000 two: 415, 100,000 426, 400,000 (six) 1,331
constexpr int64_t kTrainTiles = 4 * 152;
constexpr int kTrainSums = 8;                   // column sums: c1..c4, w5, W1 by input
constexpr uint32_t kSmemTrain = kSmemFwd + kTrainSums * kH * 4 + 2 * kTileM * 4;
static_assert(kSmemTrain <= 227u * 1024u, "training tile exceeds the shared memory of one CTA");
constexpr int64_t kZSave = 2 * 8 * 2 * kGroupThreads;  // uint4 per group: z2, z3 of one tile

struct TrainArgs {
  const float* P;
  LayerWeights<kTrainLayers> W;  // W2, W3, W4, then the transposes of W4, W3, W2
  int64_t n;
  const float* pts;
  const float* target;
  double inv_ntot;
  unsigned char* img;   // [tiles][kTrainImages][kSmemA]
  uint4* zsave;         // [CTAs][2][kZSave]
  float* grad;
  double* loss;
  int32_t* err;
};

__device__ __forceinline__ uint32_t bf16_pack(float lo, float hi) {
  uint32_t h;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(hi), "f"(lo));
  return h;
}
__device__ __forceinline__ float bf16_lo(uint32_t h) { return __uint_as_float(h << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t h) { return __uint_as_float(h & 0xFFFF0000u); }

// Column sums of the warp's 32 rows: v[2 i + e] = the lane's rows' sum of
// column 8 i + 2 (l % 4) + e. The eight lanes of a column exchange halves (7
// shuffles for 8 columns); lane l ends with value l / 4 and adds it to
// dst[its column].
__device__ __forceinline__ void add_columns(float (&v)[8], int lane, float* dst) {
  int o = 16;
#pragma unroll
  for (int h = 4; h >= 1; h >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const float give = up ? v[k] : v[k + h];
      const float keep = up ? v[k + h] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
    o >>= 1;
  }
  const int c = lane >> 2;
  atomicAdd(dst + 8 * (c >> 1) + 2 * (lane & 3) + (c & 1), v[0]);
}

__global__ void __launch_bounds__(2 * kGroupThreads, 1) k_train_tile(const TrainArgs a) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const FwdSmem S = fwd_smem(sm);
  float* sums = reinterpret_cast<float*>(sm + kSmemFwd);   // [kTrainSums][kH]
  float* sdy = sums + kTrainSums * kH;                     // [2][kTileM]
  for (int i = threadIdx.x; i < kTrainSums * kH; i += blockDim.x) sums[i] = 0.f;
  const int64_t ntiles = (a.n + kTileM - 1) / kTileM;
  const int64_t tiles = cta_tiles(ntiles);
  const uint32_t taddr = fwd_setup<kTrainLayers>(S, a.P, a.W, tiles);
  const TileLane t = tile_lane(S, taddr);
  const int64_t J1 = tiles / 2;
  uint4* zs = a.zsave + ((int64_t)blockIdx.x * 2 + t.grp) * kZSave + t.lt;
  float* dyg = sdy + t.grp * kTileM;
  uint32_t lphase = 0;
  double lsum = 0.0;
  float dc5 = 0.f;
  for (int64_t k = t.grp; k < tiles; k += 2) {
    const int64_t tile = blockIdx.x + k * gridDim.x, first = tile * kTileM;
    const int64_t j = k / 2;
    const int slot0 = (int)(j < J1 ? 2 * kTrainLayers * j + t.grp : 2 * kTrainLayers * J1);
    const int step = j < J1 ? 2 : 1;
    unsigned char* img = a.img + tile * kTrainImages * (int64_t)kSmemA;
    // the tensor-core layer of slot q, with the copy of its operand tile
    auto layer = [&](int q) {
      tile_mma<kTrainLayers>(S, t, a.W, slot0 + q * step, lphase, a.err, [&] {
        if (t.lane == 0) {
          tc::bulk_s2g(img + (int64_t)q * kSmemA, tc::smem_addr(t.A), kSmemA);
          tc::bulk_s2g_wait_read();
        }
        __syncwarp();
      });
    };
    float x[4][3];
    tile_inputs(t, a.pts, first, a.n, x);
    tile_layer1(S, t, x);
    tile_written(t);
#pragma unroll 1
    for (int l = 0; l < 3; ++l) {
      layer(l);
      uint64_t bb[4];
      tile_fragments(t, [&](int cc) { load_bias(t, S.bias + l * kH + t.c0 + cc, bb); },
                     [&](int cc, int hh, const uint32_t (&r)[16]) {
        uint64_t z[8];
        uint32_t h[8];
        add_bias(bb, r, z);
        if (l < 2) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float z0, z1;
            f2_unpack(z[i], z0, z1);
            h[i] = bf16_pack(z0, z1);
          }
          uint4* zp = zs + (int64_t)((l * 8 + cc / 16 + hh) * 2) * kGroupThreads;
          zp[0] = make_uint4(h[0], h[1], h[2], h[3]);
          zp[kGroupThreads] = make_uint4(h[4], h[5], h[6], h[7]);
        }
        silu_pairs<8>(z, h);
        put_fragments(t, cc, hh, h);
      });
      tile_written(t);
    }
    // output, loss and dL/dy: one FMA chain per row
    if (t.lt < kTileM) {
      float y = __ldg(a.P + kOffC5);
#pragma unroll 4
      for (int c = 0; c < kH; c += 8) {
        const uint4 h = *reinterpret_cast<const uint4*>(t.A + tc::kmajor_offset(t.lt, c, kH));
        const uint32_t u[4] = {h.x, h.y, h.z, h.w};
        const float4* w4 = reinterpret_cast<const float4*>(S.bias + 3 * kH + c);
        const float4 wa = w4[0], wb = w4[1];
        const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          y = __fmaf_rn(bf16_lo(u[i]), w[2 * i], y);
          y = __fmaf_rn(bf16_hi(u[i]), w[2 * i + 1], y);
        }
      }
      float dy = 0.f;
      if (first + t.lt < a.n) {
        const float e = y - __ldg(a.target + first + t.lt);
        lsum += (double)e * (double)e;
        dy = (float)(2.0 * (double)e * a.inv_ntot);
      }
      dyg[t.lt] = dy;
      dc5 += dy;
    }
    group_sync(t.grp);
    // dz4 and the sums over h4 and dz4
    {
      float dyr[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) dyr[q] = dyg[t.w0 + (t.lane >> 2) + 8 * q];
      float cs[8], ws[8];
      uint64_t bb[4];
      tile_fragments(t, [&](int cc) { load_bias(t, S.bias + 2 * kH + t.c0 + cc, bb); },
                     [&](int cc, int hh, const uint32_t (&r)[16]) {
        uint64_t z[8];
        uint32_t h[8], d[8];
        add_bias(bb, r, z);
        const uint32_t ad = t.a_st + (uint32_t)cc * 16u + (hh ? TileLane::kHalfRows : 0u);
        tc::ldmatrix4(ad, h[0], h[1], h[2], h[3]);
        tc::ldmatrix4(ad + 256u, h[4], h[5], h[6], h[7]);
        if (hh == 0)
#pragma unroll
          for (int i = 0; i < 8; ++i) cs[i] = ws[i] = 0.f;
        const float2* w2 = reinterpret_cast<const float2*>(S.bias + 3 * kH + t.c0 + cc) + (t.lane & 3);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float z0, z1;
          f2_unpack(z[i], z0, z1);
          const uint32_t zb = bf16_pack(z0, z1);
          const float2 w = w2[4 * (i >> 1)];
          const float dy = dyr[2 * hh + (i & 1)];
          d[i] = bf16_pack(dy * w.x * silu_grad(bf16_lo(zb)), dy * w.y * silu_grad(bf16_hi(zb)));
          cs[2 * (i >> 1)] += bf16_lo(d[i]);
          cs[2 * (i >> 1) + 1] += bf16_hi(d[i]);
          ws[2 * (i >> 1)] = __fmaf_rn(dy, bf16_lo(h[i]), ws[2 * (i >> 1)]);
          ws[2 * (i >> 1) + 1] = __fmaf_rn(dy, bf16_hi(h[i]), ws[2 * (i >> 1) + 1]);
        }
        put_fragments(t, cc, hh, d);
        if (hh == 1) {
          add_columns(cs, t.lane, sums + 3 * kH + t.c0 + cc);
          add_columns(ws, t.lane, sums + 4 * kH + t.c0 + cc);
        }
      });
    }
    tile_written(t);
    // dz3, dz2, dz1
#pragma unroll 1
    for (int q = 0; q < 3; ++q) {
      layer(3 + q);
      float cs[8], w1s[3][8];
      tile_fragments(t, [](int) {}, [&](int cc, int hh, const uint32_t (&r)[16]) {
        uint32_t zb[8], d[8];
        if (q < 2) {
          const uint4* zp = zs + (int64_t)(((1 - q) * 8 + cc / 16 + hh) * 2) * kGroupThreads;
          const uint4 za = zp[0], zc = zp[kGroupThreads];
          zb[0] = za.x; zb[1] = za.y; zb[2] = za.z; zb[3] = za.w;
          zb[4] = zc.x; zb[5] = zc.y; zb[6] = zc.z; zb[7] = zc.w;
        } else {
          const float4* w1 = S.w1 + t.c0 + cc + 2 * (t.lane & 3);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float4 wa = w1[8 * (i >> 1)], wb = w1[8 * (i >> 1) + 1];
            const float* xr = x[2 * hh + (i & 1)];
            const uint64_t z = f2_fma(f2_pack(wb.x, wb.y), f2_pack(xr[2], xr[2]),
                                      f2_fma(f2_pack(wa.z, wa.w), f2_pack(xr[1], xr[1]),
                                             f2_fma(f2_pack(wa.x, wa.y), f2_pack(xr[0], xr[0]), f2_pack(wb.z, wb.w))));
            float z0, z1;
            f2_unpack(z, z0, z1);
            zb[i] = bf16_pack(z0, z1);
          }
        }
        if (hh == 0)
#pragma unroll
          for (int i = 0; i < 8; ++i) cs[i] = w1s[0][i] = w1s[1][i] = w1s[2][i] = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          d[i] = bf16_pack(__uint_as_float(r[2 * i]) * silu_grad(bf16_lo(zb[i])),
                           __uint_as_float(r[2 * i + 1]) * silu_grad(bf16_hi(zb[i])));
          const int c = 2 * (i >> 1);
          cs[c] += bf16_lo(d[i]);
          cs[c + 1] += bf16_hi(d[i]);
          if (q == 2) {
            const float* xr = x[2 * hh + (i & 1)];
#pragma unroll
            for (int m = 0; m < 3; ++m) {
              w1s[m][c] = __fmaf_rn(bf16_lo(d[i]), xr[m], w1s[m][c]);
              w1s[m][c + 1] = __fmaf_rn(bf16_hi(d[i]), xr[m], w1s[m][c + 1]);
            }
          }
        }
        if (q < 2) put_fragments(t, cc, hh, d);
        if (hh == 1) {
          add_columns(cs, t.lane, sums + (2 - q) * kH + t.c0 + cc);
          if (q == 2)
#pragma unroll
            for (int m = 0; m < 3; ++m) add_columns(w1s[m], t.lane, sums + (5 + m) * kH + t.c0 + cc);
        }
      });
      tile_written(t);
    }
  }
  if (t.warp == kGroupThreads / 32 - 1 && t.lane == 0) tc::bulk_s2g_wait_all();
  fwd_teardown(S, taddr, a.err);   // (both groups meet here)
  for (int i = threadIdx.x; i < kTrainSums * kH; i += blockDim.x) {
    const int q = i / kH, o = i - q * kH;
    const int64_t dst = q == 0 ? kOffC1 + o : q == 1 ? kOffC2 + o : q == 2 ? kOffC3 + o : q == 3 ? kOffC4 + o
                        : q == 4 ? kOffW5 + o : kOffW1 + o * 3 + (q - 5);
    atomicAdd(a.grad + dst, sums[i]);
  }
  if (t.lt < kTileM) {
    const double l = warp_sum<double>(lsum);
    const float d = warp_sum<float>(dc5);
    if (t.lane == 0) {
      atomicAdd(a.loss, l);
      atomicAdd(a.grad + kOffC5, d);
    }
  }
}

// whether a bounded wait ended for all lanes of the warp (at the limit they may
// differ: the warp leaves its loop as a whole or not at all)
__device__ __forceinline__ bool warp_agrees(bool ok) { return __all_sync(0xffffffffu, ok); }

// dW of square layer blockIdx.y (W2, W3, W4) over tiles blockIdx.x, + gridDim.x, ...
constexpr int kDwRows = 32;                               // batch rows a stage
constexpr uint32_t kDwHalf = kDwRows * kH * 2;            // 16 KiB: one operand's rows
constexpr int kDwStages = 6;
constexpr uint32_t kSmemDw = kDwStages * 2 * kDwHalf + 128;
constexpr uint32_t kIdescDw = tc::idesc_bf16_f32(kTileM, kH, true);

__global__ void __launch_bounds__(192, 1) k_train_dw(const unsigned char* __restrict__ img, int64_t ntiles,
                                                     float* __restrict__ grad, int32_t* err) {
  extern __shared__ __align__(1024) unsigned char sm[];
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + kDwStages * 2 * kDwHalf);
  uint64_t* empty = full + kDwStages;
  uint64_t* done = empty + kDwStages;
  uint32_t* slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* state = reinterpret_cast<volatile int*>(slot + 1);  // result complete, stages copied, stages used
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int y = blockIdx.y;   // h_{y + 1} is image y, dz_{y + 2} image 5 - y
  if (warp == 0) {
    tc::tmem_alloc(slot, 2 * kH);
    tc::tmem_relinquish();
  }
  if (threadIdx.x == 0) {
    for (int s = 0; s < kDwStages; ++s) {
      tc::mbar_init(full + s, 1);
      tc::mbar_init(empty + s, 1);
    }
    tc::mbar_init(done, 1);
    state[0] = state[1] = state[2] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t taddr = *slot;
  constexpr int kPerTile = kTileM / kDwRows;
  const int64_t stages = cta_tiles(ntiles) * kPerTile;
  if (warp == 4) {
    const bool leader = tc::elect_one();
    for (int64_t c = 0; c < stages; ++c) {
      const int s = (int)(c % kDwStages);
      const uint32_t use = (uint32_t)(c / kDwStages);
      if (use > 0 && !warp_agrees(tc::mbar_wait(empty + s, (use - 1) & 1u, err))) break;
      if (leader) {
        const int64_t tile = blockIdx.x + (c / kPerTile) * gridDim.x;
        const unsigned char* src = img + tile * kTrainImages * (int64_t)kSmemA + (c % kPerTile) * (int64_t)kDwHalf;
        unsigned char* dst = sm + (size_t)s * 2 * kDwHalf;
        tc::mbar_arrive_expect_tx(full + s, 2 * kDwHalf);
        tc::bulk_g2s(dst, src + (5 - y) * (int64_t)kSmemA, kDwHalf, full + s);
        tc::bulk_g2s(dst + kDwHalf, src + y * (int64_t)kSmemA, kDwHalf, full + s);
        state[1] = (int)c + 1;
      }
      __syncwarp();
    }
  } else if (warp == 5) {
    const bool leader = tc::elect_one();
    for (int64_t c = 0; c < stages; ++c) {
      const int s = (int)(c % kDwStages);
      if (!warp_agrees(tc::mbar_wait(full + s, (uint32_t)(c / kDwStages) & 1u, err))) break;
      tc::fence_after_sync();
      if (leader) {
        const uint32_t da = tc::smem_addr(sm + (size_t)s * 2 * kDwHalf);
#pragma unroll
        for (int kk = 0; kk < kDwRows / 16; ++kk) {
          // 16 batch rows = two row groups of 4 KB; 8 columns = 128 bytes
          const uint64_t bd = tc::smem_desc(da + kDwHalf + kk * 2u * kH * 16u, (uint32_t)kH * 16u, 128u);
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            const uint64_t ad =
                tc::smem_desc(da + kk * 2u * kH * 16u + half * (kTileM / 8) * 128u, (uint32_t)kH * 16u, 128u);
            tc::mma_bf16(taddr + half * kH, ad, bd, kIdescDw, c > 0 || kk > 0);
          }
        }
        tc::mma_commit(empty + s);
        if (c + 1 == stages) tc::mma_commit(done);
        state[2] = (int)c + 1;
      }
      __syncwarp();
    }
    // the other warps wait at the barrier for the result
    const bool ok = stages > 0 && state[2] == (int)stages && tc::mbar_wait(done, 0u, err);
    if (leader) state[0] = ok;
    __syncwarp();
    __threadfence_block();
  }
  if (warp != 4) asm volatile("bar.sync 1, 160;" ::: "memory");
  if (warp < 4 && state[0]) {
    tc::fence_after_sync();
    float* W = grad + (y == 0 ? kOffW2 : y == 1 ? kOffW3 : kOffW4);
    for (int half = 0; half < 2; ++half)
#pragma unroll 1
      for (int hh = 0; hh < 2; ++hh)
#pragma unroll 1
        for (int cc = 0; cc < kH; cc += 32) {
          uint32_t r[16];
          tc::tmem_ld_16x256_x4(taddr + ((uint32_t)(32 * warp + 16 * hh) << 16) + (uint32_t)(half * kH + cc), r);
          tc::tmem_ld_wait();
          float* dst = W + (int64_t)(half * kTileM + 32 * warp + 16 * hh + (lane >> 2)) * kH + cc + 2 * (lane & 3);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            atomicAdd(reinterpret_cast<float2*>(dst + 8 * i),
                      make_float2(__uint_as_float(r[4 * i]), __uint_as_float(r[4 * i + 1])));
            atomicAdd(reinterpret_cast<float2*>(dst + 8 * kH + 8 * i),
                      make_float2(__uint_as_float(r[4 * i + 2]), __uint_as_float(r[4 * i + 3])));
          }
        }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  // after an expired wait: copies that no MMA consumed (bounded)
  if (threadIdx.x == 0)
    for (int c = state[2]; c < state[1]; ++c)
      if (!tc::mbar_wait(full + c % kDwStages, (uint32_t)(c / kDwStages) & 1u, err, 200000000ull)) break;
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(taddr, 2 * kH);
}

// Adam (Kingma & Ba) on the FP32 parameters
__global__ void k_adam(float* __restrict__ P, const float* __restrict__ g, float* __restrict__ m1,
                       float* __restrict__ m2, int64_t np, float lr, float b1, float b2, float eps, float c1,
                       float c2) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < np; i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float a = b1 * m1[i] + (1.f - b1) * gi;
    const float b = b2 * m2[i] + (1.f - b2) * gi * gi;
    m1[i] = a;
    m2[i] = b;
    P[i] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
  }
}

// BF16 copies of a 256x256 layer in the tile's chunked layout: W (rows out, K
// in) and its transpose (rows in, K out)
__global__ void k_weights_bf16(const float* __restrict__ Wf, unsigned char* __restrict__ Wc,
                               unsigned char* __restrict__ WTc) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < kH * kH; k += gridDim.x * blockDim.x) {
    const int o = k / kH, i = k % kH;
    const __nv_bfloat16 v = __float2bfloat16_rn(Wf[k]);
    *reinterpret_cast<__nv_bfloat16*>(Wc + wchunk_offset(o, i)) = v;
    *reinterpret_cast<__nv_bfloat16*>(WTc + wchunk_offset(i, o)) = v;
  }
}

static sft_status refresh_bf16(sft_mlp_s* m, cudaStream_t st) {
  const int64_t offW[3] = {kOffW2, kOffW3, kOffW4};
  for (int l = 0; l < 3; ++l) {
    ::sft::note_launch(), k_weights_bf16<<<64, 256, 0, st>>>(m->P + offW[l], m->Wc[l], m->WTc[l]);
    SFT_CUDA(cudaGetLastError());
  }
  return SFT_OK;
}

// device error word of one call, freed on every return path
struct ErrWord {
  int32_t* p = nullptr;
  cudaStream_t st = nullptr;
  ~ErrWord() { dfree(p, st); }
  cudaError_t init(cudaStream_t s) {
    st = s;
    cudaError_t e = dalloc(&p, 1, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(p, 0, sizeof(int32_t), s);
    return e;
  }
};

// work space of a training pass: at most kTrainTiles tiles at a time
struct TrainWs {
  int64_t tiles = 0;
  int ctas = 0;
  unsigned char* img = nullptr;
  uint4* zsave = nullptr;
  double* loss = nullptr;
  cudaStream_t st = nullptr;
  ~TrainWs() {
    dfree(img, st);
    dfree(zsave, st);
    dfree(loss, st);
  }
  cudaError_t init(int64_t rows, cudaStream_t s) {
    st = s;
    tiles = std::min<int64_t>(kTrainTiles, (rows + kTileM - 1) / kTileM);
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    ctas = (int)std::min<int64_t>(tiles, sms);
    if (e == cudaSuccess) e = dalloc(&img, (size_t)(tiles * kTrainImages) * kSmemA, s);
    if (e == cudaSuccess) e = dalloc(&zsave, (size_t)(2 * ctas * kZSave), s);
    if (e == cudaSuccess) e = dalloc(&loss, 1, s);
    return e;
  }
};

static sft_status train_attrs() {
  static PerDevice attrs;
  return attrs.once([]() -> sft_status {
    SFT_CUDA(cudaFuncSetAttribute(k_train_tile, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemTrain));
    SFT_CUDA(cudaFuncSetAttribute(k_train_dw, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemDw));
    return SFT_OK;
  });
}

// forward + backward of one batch of n rows, accumulating the gradient of
// loss / n_total into m->grad and sum (y - t)^2 into *ws.loss
static sft_status batch_grad(sft_mlp_s* m, TrainWs& ws, const float* pts, const float* t, int64_t n,
                             double inv_ntot, cudaStream_t st, int32_t* err) {
  for (int64_t r0 = 0; r0 < n; r0 += ws.tiles * kTileM) {
    const int64_t nr = std::min<int64_t>(ws.tiles * kTileM, n - r0), tiles = (nr + kTileM - 1) / kTileM;
    TrainArgs a;
    a.P = m->P;
    for (int l = 0; l < 3; ++l) {
      a.W.w[l] = m->Wc[l];
      a.W.w[3 + l] = m->WTc[2 - l];
    }
    a.n = nr;
    a.pts = pts + r0 * 3;
    a.target = t + r0;
    a.inv_ntot = inv_ntot;
    a.img = ws.img;
    a.zsave = ws.zsave;
    a.grad = m->grad;
    a.loss = ws.loss;
    a.err = err;
    ::sft::note_launch(), k_train_tile<<<(unsigned)std::min<int64_t>(tiles, ws.ctas), 2 * kGroupThreads, kSmemTrain, st>>>(a);
    SFT_CUDA(cudaGetLastError());
    // about one CTA per SM over the three layers
    const dim3 grid((unsigned)std::min<int64_t>(tiles, 50), 3);
    ::sft::note_launch(), k_train_dw<<<grid, 192, kSmemDw, st>>>(ws.img, tiles, m->grad, err);
    SFT_CUDA(cudaGetLastError());
  }
  return SFT_OK;
}

sft_status mlp_forward_dev(sft_mlp_s* m, int64_t n, const float* pts, float* out, cudaStream_t st, int32_t* d_err) {
  if (n <= 0) return SFT_OK;
  static PerDevice attrs;
  if (sft_status r = attrs.once([]() -> sft_status {
        SFT_CUDA(cudaFuncSetAttribute(k_mlp_forward, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemFwd));
        return SFT_OK;
      }))
    return r;
  int dev = 0, sms = 0;
  SFT_CUDA(cudaGetDevice(&dev));
  SFT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int64_t tiles = (n + kTileM - 1) / kTileM;
  const unsigned grid = (unsigned)std::min<int64_t>(tiles, (int64_t)sms);
  ::sft::note_launch(), k_mlp_forward<<<grid, 2 * kGroupThreads, kSmemFwd, st>>>(m->P, m->Wc[0], m->Wc[1], m->Wc[2], n,
                                                                             pts, out, d_err);
  SFT_CUDA(cudaGetLastError());
  return SFT_OK;
}

}  // namespace sft

using namespace sft;

extern "C" {

int64_t sft_mlp_nparam(void) { return kNParam; }

sft_status sft_mlp_create(const float* params, int32_t device_ptrs, void* cuda_stream, sft_mlp* out) {
  (void)device_ptrs;
  if (!out || !params) return fail(SFT_ERR_ARG, "null argument");
  *out = nullptr;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  auto* m = new sft_mlp_s();
  m->stream = st;
  sft_status r = SFT_OK;
  do {
    cudaError_t e = dalloc(&m->P, (size_t)kNParam, st);
    if (e != cudaSuccess) { r = cuda_fail(e, "alloc"); break; }
    e = cudaMemcpyAsync(m->P, params, sizeof(float) * kNParam, cudaMemcpyDefault, st);
    if (e != cudaSuccess) { r = cuda_fail(e, "copy"); break; }
    for (int l = 0; l < 3 && e == cudaSuccess; ++l) {
      e = dalloc(&m->Wc[l], (size_t)kH * kH * 2, st);
      if (e == cudaSuccess) e = dalloc(&m->WTc[l], (size_t)kH * kH * 2, st);
    }
    if (e != cudaSuccess) { r = cuda_fail(e, "alloc"); break; }
    if (r) break;
    if ((r = refresh_bf16(m, st))) break;
    e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) r = cuda_fail(e, "sync");
  } while (0);
  if (r) {
    sft_mlp_destroy(m);
    return r;
  }
  *out = m;
  return SFT_OK;
}

void sft_mlp_destroy(sft_mlp m) {
  if (!m) return;
  dfree(m->P, m->stream);
  for (auto& w : m->Wc) dfree(w, m->stream);
  for (auto& w : m->WTc) dfree(w, m->stream);
  dfree(m->grad, m->stream);
  dfree(m->m1, m->stream);
  dfree(m->m2, m->stream);
  delete m;
}

sft_status sft_mlp_params(sft_mlp m, float* out, int32_t out_device, void* cuda_stream) {
  if (!m || !out) return fail(SFT_ERR_ARG, "null argument");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  SFT_CUDA(cudaMemcpyAsync(out, m->P, sizeof(float) * kNParam,
                           out_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaStreamSynchronize(st));
  return SFT_OK;
}

static sft_status ensure_train_state(sft_mlp m, cudaStream_t st) {
  if (m->grad) return SFT_OK;
  SFT_CUDA(dalloc(&m->grad, (size_t)kNParam, st));
  SFT_CUDA(dalloc(&m->m1, (size_t)kNParam, st));
  SFT_CUDA(dalloc(&m->m2, (size_t)kNParam, st));
  SFT_CUDA(cudaMemsetAsync(m->m1, 0, sizeof(float) * kNParam, st));
  SFT_CUDA(cudaMemsetAsync(m->m2, 0, sizeof(float) * kNParam, st));
  return SFT_OK;
}

sft_status sft_mlp_loss_grad(sft_mlp m, int64_t n, const float* pts, const float* targets, float* grad_out,
                             double* loss_out, int32_t device_ptrs, void* cuda_stream) {
  if (!m || n < 1 || !pts || !targets || !grad_out) return fail(SFT_ERR_ARG, "null argument or n < 1");
  if (!device_ptrs) return fail(SFT_ERR_ARG, "sft_mlp_loss_grad takes device pointers");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (sft_status r = train_attrs()) return r;
  if (sft_status r = ensure_train_state(m, st)) return r;
  TrainWs ws;
  SFT_CUDA(ws.init(n, st));
  ErrWord ew;
  SFT_CUDA(ew.init(st));
  int32_t* d_err = ew.p;
  SFT_CUDA(cudaMemsetAsync(m->grad, 0, sizeof(float) * kNParam, st));
  SFT_CUDA(cudaMemsetAsync(ws.loss, 0, sizeof(double), st));
  if (sft_status r = batch_grad(m, ws, pts, targets, n, 1.0 / (double)n, st, d_err)) return r;
  double hl = 0.0;
  int32_t herr = 0;
  SFT_CUDA(cudaMemcpyAsync(grad_out, m->grad, sizeof(float) * kNParam, cudaMemcpyDeviceToDevice, st));
  SFT_CUDA(cudaMemcpyAsync(&hl, ws.loss, sizeof(double), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaMemcpyAsync(&herr, d_err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaStreamSynchronize(st));
  if (herr) return fail(SFT_ERR_DEVICE_STATUS, "tensor-core wait expired in the network backward");
  if (loss_out) *loss_out = hl / (double)n;
  return SFT_OK;
}

sft_status sft_mlp_train(sft_mlp m, int64_t n, const float* pts, const float* targets, int32_t epochs, int32_t batch,
                         float lr, float lr_final, double* loss_history, int32_t device_ptrs, void* cuda_stream) {
  if (!m || n < 1 || !pts || !targets || epochs < 1 || batch < 1) return fail(SFT_ERR_ARG, "bad training arguments");
  if (!device_ptrs) return fail(SFT_ERR_ARG, "sft_mlp_train takes device pointers");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  if (sft_status r = train_attrs()) return r;
  if (sft_status r = ensure_train_state(m, st)) return r;
  const int64_t B = std::min<int64_t>((int64_t)(batch + kTileM - 1) / kTileM * kTileM,
                                      (n + kTileM - 1) / kTileM * kTileM);
  TrainWs ws;
  SFT_CUDA(ws.init(B, st));
  ErrWord ew;
  SFT_CUDA(ew.init(st));
  int32_t* d_err = ew.p;
  const int64_t nbatch = (n + B - 1) / B;
  const int64_t total_steps = (int64_t)epochs * nbatch;
  int64_t s_step = 0;
  for (int ep = 0; ep < epochs; ++ep) {
    SFT_CUDA(cudaMemsetAsync(ws.loss, 0, sizeof(double), st));
    for (int64_t bi = 0; bi < nbatch; ++bi) {
      const int64_t b0 = bi * B, nb = std::min<int64_t>(B, n - b0);
      SFT_CUDA(cudaMemsetAsync(m->grad, 0, sizeof(float) * kNParam, st));
      if (sft_status r = batch_grad(m, ws, pts + b0 * 3, targets + b0, nb, 1.0 / (double)nb, st, d_err)) return r;
      // learning rate: geometric decay from lr to lr_final over the run
      const double frac = total_steps > 1 ? (double)(s_step++) / (double)(total_steps - 1) : 0.0;
      const float lr_t = (float)((double)lr * std::pow((double)lr_final / (double)lr, std::min(1.0, frac)));
      m->step += 1;
      const float c1 = (float)(1.0 - std::pow(0.9, (double)m->step));
      const float c2 = (float)(1.0 - std::pow(0.999, (double)m->step));
      ::sft::note_launch(), k_adam<<<256, 256, 0, st>>>(m->P, m->grad, m->m1, m->m2, kNParam, lr_t, 0.9f, 0.999f,
                                                        1e-8f, c1, c2);
      SFT_CUDA(cudaGetLastError());
      if (sft_status r = refresh_bf16(m, st)) return r;
    }
    if (loss_history) {
      double hl = 0.0;
      SFT_CUDA(cudaMemcpyAsync(&hl, ws.loss, sizeof(double), cudaMemcpyDeviceToHost, st));
      SFT_CUDA(cudaStreamSynchronize(st));
      loss_history[ep] = hl / (double)n;
    }
  }
  int32_t herr = 0;
  SFT_CUDA(cudaMemcpyAsync(&herr, d_err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaStreamSynchronize(st));
  if (herr) return fail(SFT_ERR_DEVICE_STATUS, "tensor-core wait expired in training");
  return SFT_OK;
}

sft_status sft_mlp_forward(sft_mlp m, int64_t n, const float* pts, float* out, int32_t device_ptrs,
                           void* cuda_stream) {
  if (!m || (n > 0 && (!pts || !out))) return fail(SFT_ERR_ARG, "null argument");
  if (n <= 0) return SFT_OK;
  cudaStream_t st = (cudaStream_t)cuda_stream;
  float* dp = const_cast<float*>(pts);
  float* dout = out;
  std::vector<void*> tmp;
  if (!device_ptrs) {
    SFT_CUDA(dalloc(&dp, (size_t)n * 3, st));
    SFT_CUDA(dalloc(&dout, (size_t)n, st));
    SFT_CUDA(cudaMemcpyAsync(dp, pts, sizeof(float) * 3 * n, cudaMemcpyHostToDevice, st));
  }
  int32_t* d_err = nullptr;
  SFT_CUDA(dalloc(&d_err, 1, st));
  SFT_CUDA(cudaMemsetAsync(d_err, 0, sizeof(int32_t), st));
  sft_status r = mlp_forward_dev(m, n, dp, dout, st, d_err);
  int32_t herr = 0;
  if (!r) {
    SFT_CUDA(cudaMemcpyAsync(&herr, d_err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    if (!device_ptrs) SFT_CUDA(cudaMemcpyAsync(out, dout, sizeof(float) * n, cudaMemcpyDeviceToHost, st));
    SFT_CUDA(cudaStreamSynchronize(st));
  }
  dfree(d_err, st);
  if (!device_ptrs) {
    dfree(dp, st);
    dfree(dout, st);
  }
  if (r) return r;
  if (herr) return fail(SFT_ERR_DEVICE_STATUS, "tensor-core wait expired in the network forward");
  return SFT_OK;
}

}  // extern "C"
