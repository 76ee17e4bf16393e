// Step 7 of Sec. 4: solve the target Galerkin system M u = b (Eq.
// cv_galerkin_system) from u = 0 (or, in the mixed mode on request, from the
// u the caller holds), stopping at ||b - M u||_2 <= tol ||b||_2 (the paper
// does not name its solver). Two kernels:
//   k_pcg       Jacobi-preconditioned CG in FP64 (cg_mode FP64, and the
//               allocation-free entry point, which takes any SPD CSR matrix);
//   k_mixed     mixed-precision iterative refinement (default; see below).
//
// One cooperative (co-resident) kernel runs the whole iteration: no host round
// trip per step. Each k_pcg iteration has two grid barriers:
//   A: w = M z (SpMV), then for the own row p = z + beta p and
//      q = w + beta q (= M p by linearity, one FP64 FMA per nonzero instead of
//      two), and the partial dot p.q;
//   B: u += a p, r -= a q, z = D^-1 r, partial dots r.r and r.z.
// FP64 throughput is the scarce resource on this GPU, so the iteration is
// written to minimise FP64 operations per row.
// Dot products are reduced deterministically: per-block partials, then every
// block sums all partials in the same fixed order, so all blocks take the
// same convergence decision. The barrier wait is bounded (error flag on
// timeout; the kernel then returns).
#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>
#include "internal.hpp"
#include "util.cuh"

namespace sft {

constexpr int kSolveThreads = 256;

struct PcgCtl {
  GridBarrier bar;
  int32_t err;
  int32_t iters[kMaxFields];
  double rel[kMaxFields];
  int32_t conv[kMaxFields];
};

// sum the per-block partials [nblocks][nrhs][2] -> tot[nrhs][2], identical
// in all blocks: thread t sums blocks t, t + 256, ... in order, then warps
// reduce with a fixed shuffle tree and thread k adds the 8 warp sums in order
__device__ __forceinline__ void reduce_partials(const double* part, int nblocks, int nrhs, double* sh_tot) {
  __shared__ double shw[kSolveThreads / 32][kMaxFields * 2];
  double acc[kMaxFields * 2];
#pragma unroll
  for (int k = 0; k < kMaxFields * 2; ++k) acc[k] = 0.0;
  for (int bidx = threadIdx.x; bidx < nblocks; bidx += blockDim.x) {
    const double* pb = part + (int64_t)bidx * nrhs * 2;
#pragma unroll
    for (int k = 0; k < kMaxFields * 2; ++k)
      if (k < nrhs * 2) acc[k] += __ldcg(pb + k);
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kMaxFields * 2; ++k) {
    if (k >= nrhs * 2) break;
    const double w = warp_sum<double>(acc[k]);
    if (lane == 0) shw[warp][k] = w;
  }
  __syncthreads();
  if (threadIdx.x < nrhs * 2) {
    double t = 0.0;
    for (int w = 0; w < kSolveThreads / 32; ++w) t += shw[w][threadIdx.x];
    sh_tot[threadIdx.x] = t;
  }
  __syncthreads();
}

__device__ __forceinline__ void block_partials(double v[kMaxFields][2], int nrhs, double* part) {
  __shared__ double sh[kSolveThreads / 32][kMaxFields][2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int f = 0; f < nrhs; ++f)
    for (int c = 0; c < 2; ++c) {
      const double w = warp_sum<double>(v[f][c]);
      if (lane == 0) sh[warp][f][c] = w;
    }
  __syncthreads();
  if (threadIdx.x < nrhs * 2) {
    const int f = threadIdx.x >> 1, c = threadIdx.x & 1;
    double s = 0.0;
    for (int w = 0; w < kSolveThreads / 32; ++w) s += sh[w][f][c];
    part[((int64_t)blockIdx.x * nrhs + f) * 2 + c] = s;
  }
  __syncthreads();
}

template <int TPR>
__global__ void __launch_bounds__(kSolveThreads) k_pcg(const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
                                                       const double* __restrict__ val, const double* __restrict__ dinv,
                                                       int64_t n, int nrhs, const double* __restrict__ b,
                                                       double* __restrict__ x, double* r, double* z, double* p,
                                                       double* q, double* part, PcgCtl* ctl, double tol,
                                                       int max_iter, uint64_t wait_ns) {
  __shared__ double tot[kMaxFields * 2];
  __shared__ double bnorm[kMaxFields], rz[kMaxFields], beta[kMaxFields], alpha[kMaxFields];
  __shared__ int conv[kMaxFields];
  const unsigned nb = gridDim.x;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nthreads = (int64_t)gridDim.x * blockDim.x;
  double v[kMaxFields][2];

  // init: x = 0, r = b, z = D^-1 r, p_old = 0
  for (int f = 0; f < kMaxFields; ++f) v[f][0] = v[f][1] = 0.0;
  for (int64_t i = tid; i < n; i += nthreads) {
    const double di = dinv[i];
    for (int f = 0; f < nrhs; ++f) {
      const int64_t k = (int64_t)f * n + i;
      const double bi = b[k];
      x[k] = 0.0;
      r[k] = bi;
      z[k] = di * bi;
      p[k] = 0.0;
      q[k] = 0.0;
      v[f][0] += bi * bi;
      v[f][1] += bi * di * bi;
    }
  }
  block_partials(v, nrhs, part);
  if (!grid_sync(&ctl->bar, nb, &ctl->err, wait_ns)) return;
  reduce_partials(part, nb, nrhs, tot);
  if (threadIdx.x == 0) {
    for (int f = 0; f < nrhs; ++f) {
      bnorm[f] = sqrt(tot[f * 2]);
      rz[f] = tot[f * 2 + 1];
      beta[f] = 0.0;
      conv[f] = bnorm[f] == 0.0;
    }
  }
  __syncthreads();

  int it = 0;
  constexpr int kRowsPerWarp = 32 / TPR;
  const int lane = threadIdx.x & 31;
  const int lane_in_row = lane % TPR;
  const int64_t warp_id = tid >> 5, nwarps = nthreads >> 5;
  for (;;) {
    bool all = true;
    for (int f = 0; f < nrhs; ++f) all = all && conv[f];
    if (all || it >= max_iter) break;
    // phase A (warp-uniform loop: each warp owns 32/TPR consecutive rows)
    for (int f = 0; f < kMaxFields; ++f) v[f][0] = v[f][1] = 0.0;
    for (int64_t base = warp_id * kRowsPerWarp; base < n; base += nwarps * kRowsPerWarp) {
      const int64_t row = base + lane / TPR;
      const bool valid = row < n;
      int32_t q0 = 0, q1 = 0;
      if (valid) {
        q0 = __ldg(rp + row);
        q1 = __ldg(rp + row + 1);
      }
      for (int f = 0; f < nrhs; ++f) {
        if (conv[f]) continue;
        const double* zf = z + (int64_t)f * n;
        double s = 0.0;
        // z was written by other blocks before the grid barrier; the barrier's
        // acquire fence makes those writes visible to ordinary (L1-cached)
        // loads, so neighbouring rows share the gathered lines in L1
        for (int32_t k = q0 + lane_in_row; k < q1; k += TPR) s += __ldg(val + k) * zf[__ldg(col + k)];
        if constexpr (TPR > 1) {
#pragma unroll
          for (int o = TPR / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, TPR);
        }
        if (valid && lane_in_row == 0) {
          const double bt = beta[f];
          const int64_t k = (int64_t)f * n + row;
          const double pn = __ldcg(zf + row) + bt * __ldcg(p + k);
          const double qn = s + bt * __ldcg(q + k);
          p[k] = pn;
          q[k] = qn;
          v[f][0] += pn * qn;
        }
      }
    }
    block_partials(v, nrhs, part);
    if (!grid_sync(&ctl->bar, nb, &ctl->err, wait_ns)) return;
    reduce_partials(part, nb, nrhs, tot);
    if (threadIdx.x == 0)
      for (int f = 0; f < nrhs; ++f) alpha[f] = conv[f] ? 0.0 : rz[f] / tot[f * 2];
    __syncthreads();
    // phase B
    for (int f = 0; f < kMaxFields; ++f) v[f][0] = v[f][1] = 0.0;
    for (int64_t i = tid; i < n; i += nthreads) {
      const double di = dinv[i];
      for (int f = 0; f < nrhs; ++f) {
        if (conv[f]) continue;
        const int64_t k = (int64_t)f * n + i;
        const double a = alpha[f];
        x[k] = __ldcg(x + k) + a * __ldcg(p + k);
        const double ri = __ldcg(r + k) - a * __ldcg(q + k);
        r[k] = ri;
        const double zi = di * ri;
        z[k] = zi;
        v[f][0] += ri * ri;
        v[f][1] += ri * zi;
      }
    }
    block_partials(v, nrhs, part);
    if (!grid_sync(&ctl->bar, nb, &ctl->err, wait_ns)) return;
    reduce_partials(part, nb, nrhs, tot);
    ++it;
    if (threadIdx.x == 0) {
      for (int f = 0; f < nrhs; ++f) {
        if (conv[f]) continue;
        const double rn = sqrt(tot[f * 2]);
        ctl->iters[f] = it;  // identical in every block
        ctl->rel[f] = rn / bnorm[f];
        if (rn <= tol * bnorm[f]) conv[f] = 1;
        beta[f] = tot[f * 2 + 1] / rz[f];
        rz[f] = tot[f * 2 + 1];
      }
    }
    __syncthreads();
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    for (int f = 0; f < nrhs; ++f) {
      ctl->conv[f] = conv[f];
      if (bnorm[f] == 0.0) { ctl->iters[f] = 0; ctl->rel[f] = 0.0; }
    }
  }
}

// ---------------------------------------------------------------------------
// Mixed-precision iterative refinement (cg_mode MIXED).
//
// With S = diag(M)^-1/2 the scaled matrix A = S M S has unit diagonal. For P1
// elements the element mass matrix against its own diagonal has eigenvalues
// in [1/2, 2] (triangles) or [1/2, 5/2] (tetrahedra), and the assembled
// matrix inherits the union of the element bounds, so cond(A) <= 4 or 5 on
// any mesh: an FP32 solve on A converges like Jacobi-PCG in FP64 on M, and
// its attainable accuracy (~ eps32 cond(A)) is far below the per-cycle target.
// One refinement cycle:
//   R (FP64)  r = b - M x, t = S r, ||r||_2 (the stopping test) and ||t||_2;
//   I         c = t / ||t||_2 rounded to FP32 (unit norm), y_0 = 0, y_1 = c / theta;
//   inner (FP32) on A y = c to ||c - A y||_2 <= eta, eta about the reduction
//             the stopping test still needs (between 1e-5 and 1/4): the
//             Chebyshev iteration over the spectrum interval in its three-term
//             form  y_{k+1} = y_k + rho' rho (y_k - y_{k-1}) + (2 rho'/delta) (c - A y_k),
//             K steps (the count the interval fixes for eta; util.cuh) with
//             K - 1 products by A (y_1 needs none);
//   U (FP64)  x += ||t||_2 S y   (so the new residual is ||t|| S^-1 (c - A y)),
//             in the loop of the last step.
// A warm start takes x as given (||b|| is then reduced separately first) and
// skips nothing else: the first R phase checks whether x already converged.
// The FP64 pipe does one SpMV per cycle (2 to 3 cycles) instead of one per
// iteration. Every block takes every decision from the same fixed-order
// reductions; the stopping test uses the true FP64 residual.
// smallest inner reduction asked of one FP32 solve (measured: 1e-5 gives
// 0.71 / 0.68 ms on the 1.0 M-row 2D / 0.5 M-row 3D systems, 3e-6 and 1e-6
// 0.74 / 0.71 ms: deeper FP32 solves cost more iterations than the extra
// refinement cycle they save)
constexpr double kEtaFloor = 1e-5f;
constexpr int kMaxSteps = 16;  // steps of a cycle: at most 13 (tetrahedra)

// Off-diagonal entries of A for the FP32 steps (A's diagonal is 1): rows in
// slices of 32, each slice's rows sorted by length (longest first) over the
// lanes of a warp, entry q of the rows that have one stored side by side
// (jagged diagonals). A warp's load of entry q is one contiguous read with no
// padding, and the lanes that have it are a prefix, so its place follows from
// a ballot. Slice s starts at row_ptr[32 s]; rinfo[32 s + lane] = the lane's
// row in the slice (5 bits) | its off-diagonal count << 5.
constexpr int kSlice = 32;

// team of blocks that works on one system
enum : int { kTeamBlock = 0, kTeamCluster = 1, kTeamGrid = 2 };

struct MixCtl {
  uint32_t arrived;      // grid barrier: arrivals so far (never reset)
  int32_t err;
  int32_t late[2];       // cluster barriers that overran the wait limit, by parity
  int32_t iters[kMaxFields];
  int32_t conv[kMaxFields];
  double rel[kMaxFields];
};

// Barrier over the team with the limit wait_ns on the wait; false when a wait
// expired (the caller returns). The grid's is one counter that only grows:
// a release reduction by one thread per block, then acquire polls until
// phase x blocks have arrived (no reset and no generation word on the way).
// The cluster's is the hardware barrier, which cannot be left early: an
// overrun is noted for the next barrier's parity, after which every block
// sees the same word and leaves.
template <int TEAM>
__device__ __forceinline__ bool team_sync(MixCtl* ctl, unsigned nb, unsigned& phase, uint64_t wait_ns) {
  if constexpr (TEAM == kTeamBlock) {
    __syncthreads();
    return true;
  } else if constexpr (TEAM == kTeamCluster) {
    __shared__ int ok;
    ++phase;
    uint64_t t0 = 0;
    if (threadIdx.x == 0) t0 = globaltimer_ns();
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
    if (threadIdx.x == 0) {
      ok = *reinterpret_cast<volatile int32_t*>(&ctl->late[(phase - 1) & 1]) == 0;
      if (globaltimer_ns() - t0 > wait_ns) {
        *reinterpret_cast<volatile int32_t*>(&ctl->late[phase & 1]) = 1;
        set_error(&ctl->err, DEV_BARRIER_TIMEOUT);
      }
    }
    __syncthreads();
    return ok != 0;
  } else {
    __shared__ int ok;
    ++phase;
    __syncthreads();
    if (threadIdx.x == 0) {
      ok = 1;
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&ctl->arrived) : "memory");
      const uint32_t want = phase * nb;
      const uint64_t t0 = globaltimer_ns();
      for (;;) {
        const int32_t e = *reinterpret_cast<volatile int32_t*>(&ctl->err);
        uint32_t got;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(got) : "l"(&ctl->arrived) : "memory");
        if ((int32_t)(got - want) >= 0) break;
        if (e != 0) { ok = 0; break; }
        if (globaltimer_ns() - t0 > wait_ns) {
          set_error(&ctl->err, DEV_BARRIER_TIMEOUT);
          ok = 0;
          break;
        }
      }
    }
    __syncthreads();
    return ok != 0;
  }
}

// a row's NR interleaved FP32 values
template <int NR>
__device__ __forceinline__ void ld_row(const float* p, float (&v)[NR]) {
  if constexpr (NR == 1) {
    v[0] = *p;
  } else if constexpr (NR == 2) {
    const float2 a = *reinterpret_cast<const float2*>(p);
    v[0] = a.x; v[1] = a.y;
  } else {
#pragma unroll
    for (int q = 0; q < NR; q += 4) {
      const float4 a = *reinterpret_cast<const float4*>(p + q);
      v[q] = a.x; v[q + 1] = a.y; v[q + 2] = a.z; v[q + 3] = a.w;
    }
  }
}
template <int NR>
__device__ __forceinline__ void st_row(float* p, const float (&v)[NR]) {
  if constexpr (NR == 1) {
    *p = v[0];
  } else if constexpr (NR == 2) {
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  } else {
#pragma unroll
    for (int q = 0; q < NR; q += 4) *reinterpret_cast<float4*>(p + q) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
  }
}

// Where a block keeps the Chebyshev iterates y. kTeamBlock: all in its shared
// memory. kTeamCluster: each block's rows in its shared memory, read by the
// others through the cluster's distributed shared memory (an L2 round trip
// costs about three times as much: 4.0 k cycles per step through L2 against
// 1.3 k). kTeamGrid with OWN: the block's rows in its shared memory and a
// copy in global memory for the other blocks; without OWN (more rows than
// fit): global memory only.
template <int TEAM, bool OWN>
struct YRef {
  float* sm;           // [2][rows][NR] own rows (shared)
  const float* glob;   // the current y in global memory (grid)
  int64_t r0;
  int rows;            // rows of a block
  int NRv;

  // column -> reference kept in an entry
  __device__ __forceinline__ int translate(int col) const {
    if constexpr (TEAM == kTeamBlock) {
      return col;
    } else if constexpr (TEAM == kTeamCluster) {
      const uint32_t rank = (uint32_t)col / (uint32_t)rows, loc = (uint32_t)col - rank * (uint32_t)rows;
      uint32_t addr = (uint32_t)__cvta_generic_to_shared(sm) + loc * (uint32_t)NRv * 4u;
      asm("mapa.shared::cluster.u32 %0, %0, %1;" : "+r"(addr) : "r"(rank));
      return (int)addr;
    } else if constexpr (OWN) {
      const int64_t l = col - r0;
      return l >= 0 && l < rows ? (int)l : ~col;
    } else {
      return col;
    }
  }
};

// a row's NR interleaved values of the current y by its reference; `cur` is
// the current half of the own rows (shared memory), `half` its byte offset
template <int NR, int TEAM, bool OWN>
__device__ __forceinline__ void ld_y(const float* cur, uint32_t half, const float* glob, int ref, float (&v)[NR]) {
  if constexpr (TEAM == kTeamBlock) {
    ld_row<NR>(cur + ref * NR, v);
  } else if constexpr (TEAM == kTeamCluster) {
    const uint32_t ad = (uint32_t)ref + half;
    if constexpr (NR == 1) {
      asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v[0]) : "r"(ad));
    } else if constexpr (NR == 2) {
      asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v[0]), "=f"(v[1]) : "r"(ad));
    } else {
#pragma unroll
      for (int q = 0; q < NR; q += 4)
        asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                     : "=f"(v[q]), "=f"(v[q + 1]), "=f"(v[q + 2]), "=f"(v[q + 3])
                     : "r"(ad + 4u * q));
    }
  } else if constexpr (OWN) {
    if (ref >= 0) ld_row<NR>(cur + ref * NR, v);
    else ld_row<NR>(glob + (int64_t)(~ref) * NR, v);
  } else {
    // written by other blocks before the last barrier: plain loads (cached in
    // L1, where neighbouring rows share the lines)
    ld_row<NR>(glob + (int64_t)ref * NR, v);
  }
}

// w += (A - I) y for the lane's row of a slice: `len` entries, the slice's
// longest row has `maxlen`. U entries at a time, so U gathers are in flight.
template <int NR, int TEAM, bool OWN, bool HELD>
__device__ __forceinline__ void slice_product(const int2* ent, const YRef<TEAM, OWN>& Y, const float* cur, uint32_t half,
                                              int len, int maxlen, int lane, float (&w)[NR]) {
  constexpr int U = NR <= 2 ? 8 : 4;
  const int2* e0 = ent + lane;
  for (int q = 0; q < maxlen; q += U) {
    int2 e[U];
    float g[U][NR];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const bool has = len > q + u;
      e[u] = make_int2(0, 0);
      if (has) e[u] = *e0;
      e0 += __popc(__ballot_sync(0xffffffffu, has));
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int f = 0; f < NR; ++f) g[u][f] = 0.f;
      if (len > q + u) ld_y<NR, TEAM, OWN>(cur, half, Y.glob, HELD ? e[u].x : Y.translate(e[u].x), g[u]);
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int f = 0; f < NR; ++f) w[f] = __fmaf_rn(__int_as_float(e[u].y), g[u][f], w[f]);
  }
}

// Sum of V values (a power of two up to 32) over the lanes of a warp: at each
// of the first log2 V steps a lane hands over half of its values and keeps
// the other half, so the V sums take V - 1 + 5 - log2 V additions instead of
// 5 V (an FP64 warp instruction occupies this GPU's FP64 pipe for 16 cycles).
// Lane l returns the sum of value l / (32 / V).
template <int V>
__device__ __forceinline__ double warp_sums(double (&v)[V], int lane) {
  int o = 16;
#pragma unroll
  for (int h = V / 2; h >= 1; h >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < h; ++k) {
      const double give = up ? v[k] : v[k + h];
      const double keep = up ? v[k + h] : v[k];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
    o >>= 1;
  }
#pragma unroll
  for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  return v[0];
}

struct MixArgs {
  const int32_t* rp;      // row starts of M
  const int2* jent;       // off-diagonal entries as jagged diagonals: {column, FP32 value bits of A},
  const double* jval;     //   the same entries of M,
  const double* mdiag;    //   its diagonal,
  const uint16_t* rinfo;  //   rows and lengths of the slices' lanes
  const double* sc;       // diag(M)^-1/2
  int64_t n;
  int nrhs;
  const double* b;        // [nrhs][n]
  double* x;
  double* t;              // [nrhs][n]
  float* ya;              // [n][NR] (grid)
  float* yb;
  float* c;               // [n][NR], when it is not held in shared memory
  double* partd;          // [2][2 nrhs][blocks]: the warm start's, the cycles'
  MixCtl* ctl;
  double tol;
  int max_iter;
  int warm;
  uint64_t wait_ns;
  float lmax;
  // step counts of a cycle that asks for the reduction e = 0.1 tol ||b|| / ||r||
  // (kEtaFloor to 1/4): the smallest K >= k_min with T_K(s1) >= 1 / e, which is
  // reach[K] ||b||^2 >= ||r||^2 for K < k_max, with reach[K] = (0.1 tol T_K)^2
  int k_min, k_max;
  double reach[kMaxSteps];
  int spb;                // slices per block
  int cap;                // entries held in shared memory
  int c_smem;             // c held in shared memory
  int r_smem;             // rinfo held in shared memory
};

// a block's per-field state of the refinement cycles (shared memory)
struct Cycle {
  double tot[2 * kMaxFields];   // ||r||^2 and ||t||^2 by field
  double bn2[kMaxFields], prev2[kMaxFields], sig[kMaxFields], isig[kMaxFields];
  double reach[kMaxSteps];
  int live[kMaxFields], act[kMaxFields], conv[kMaxFields], ks[kMaxFields], itf[kMaxFields];
};

// Field f after the residual of cycle cyc, by a warp: converged, given up, or
// ||t||, 1 / ||t|| and the step count of its next inner solve (the lanes try
// the counts). Out of line: inside k_mixed it changes the registers of the
// steps (3.0 M rows 2D 1,660 us a call against 1,580, 4 fields of 636 k rows 3D
// 1,160 against 1,110).
__device__ __noinline__ void decide(Cycle& c, int f, int lane, int cyc, int warm, int it, double tol, int k_min, int k_max) {
  // tests on the squared norms (no square root or quotient on the way)
  const double rn2 = c.tot[2 * f], tn2 = c.tot[2 * f + 1];
  const double b2 = cyc == 0 && !warm ? rn2 : c.bn2[f], last2 = c.prev2[f];
  const bool more = lane >= k_min && lane < k_max && c.reach[lane & (kMaxSteps - 1)] * b2 < rn2;
  const int k = k_min + __popc(__ballot_sync(0xffffffffu, more));
  if (lane != 0) return;
  c.act[f] = 0;
  c.ks[f] = 0;
  if (!c.live[f]) return;
  c.bn2[f] = b2;
  c.prev2[f] = rn2;
  c.itf[f] = it;
  if (rn2 <= tol * (tol * b2)) {  // (in this order: b = 0 has converged for any tol)
    c.live[f] = 0;
    c.conv[f] = 1;
  } else if ((cyc > 0 && rn2 > 0.25 * last2) || !(tn2 > 0.0)) {
    // a cycle that did not halve the residual (FP64 rounding floor) or a
    // residual on rows without diagonal ends the field unconverged
    c.live[f] = 0;
  } else {
    const double is = rsqrt(tn2);
    c.isig[f] = is;
    c.sig[f] = tn2 * is;
    c.ks[f] = k;
    c.act[f] = 1;
  }
}

// blocks hold as much of their part of A as fits in shared memory for the
// whole solve: bytes of it
constexpr uint32_t kMixSmemMax = 212u * 1024u;
constexpr int kMaxStaged = 1024;   // slices a block may hold
template <int NR>
constexpr int kMixThreads = NR <= 2 ? 1024 : 512;

// One block per SM. Each block owns spb consecutive slices of rows for the
// whole solve and keeps what it can of them in shared memory: its part of A,
// its rows of y, c and rinfo. So a step reads from L2 only the neighbours'
// rows of y and the part of A that does not fit (none up to about 0.6 M rows
// in 2D, 0.25 M in 3D).
// What bounds it: small systems the chain of barrier, gather and row update
// (a step takes 1.8 k cycles on a block, 3.1 k on a cluster, 5 k on the
// grid), large ones the shared-memory loads and issue of the steps (12 us a
// step at 1.0 M rows) and the FP64 pipe of the residual (38 us a cycle there
// against 25 of pure FP64 work). Kernel time, before (grid of 4 blocks per SM
// over CSR rows, all vectors in L2) and now: 1.0 M rows 2D 648 -> 421 us,
// 0.51 M 3D 574 -> 422, 0.37 M 2D 350 -> 176, 10 k 2D 179 -> 62, 784 2D
// 140 -> 46, 227 k 3D with 8 fields 1,739 -> 615.
template <int NR, int TEAM, bool OWN>
__global__ void __launch_bounds__(kMixThreads<NR>, 1) k_mixed(const MixArgs a) {
  constexpr int T = kMixThreads<NR>, W = T / 32, V = 2 * NR;
  constexpr bool YSM = TEAM != kTeamGrid || OWN;   // own rows of y in shared memory
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ int32_t s_off[kMaxStaged + 1];     // start of each held slice in ent
  __shared__ double shw[W][V];
  __shared__ Cycle C;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned nb = gridDim.x;
  const int64_t n = a.n;
  const int nrhs = NR == 1 ? 1 : a.nrhs;
  const int64_t s0 = (int64_t)blockIdx.x * a.spb;
  const int64_t nslices = (n + kSlice - 1) / kSlice;
  const int nsl = (int)(s0 >= nslices ? 0 : (nslices - s0 < a.spb ? nslices - s0 : a.spb));
  const int64_t r0 = s0 * kSlice;
  const int64_t r1 = r0 + (int64_t)nsl * kSlice < n ? r0 + (int64_t)nsl * kSlice : n;
  const int rows = a.spb * kSlice;
  float* const ysm = reinterpret_cast<float*>(dsm);   // [2][rows][NR]
  int2* const ent = reinterpret_cast<int2*>(ysm + (YSM ? (int64_t)2 * rows * NR : 0));
  float* const csm = reinterpret_cast<float*>(ent + a.cap);
  uint16_t* const rsm = reinterpret_cast<uint16_t*>(csm + (a.c_smem ? (int64_t)rows * NR : 0));
  float* const cg = a.c + r0 * NR;
  MixCtl* ctl = a.ctl;
  unsigned phase = 0;
  const ChebCoef ch = cheb_coef(a.lmax);
  YRef<TEAM, OWN> Y;
  Y.sm = ysm;
  Y.glob = a.ya;
  Y.r0 = r0;
  Y.rows = rows;
  Y.NRv = NR;

  // hold rinfo and the leading slices of A
  if (a.r_smem)
    for (int i = tid; i < nsl * kSlice; i += T) rsm[i] = a.rinfo[r0 + i];
  const int ncand = nsl < kMaxStaged ? nsl : kMaxStaged;
  for (int sl = warp; sl < ncand; sl += W) {
    const int cnt = __reduce_add_sync(0xffffffffu, a.rinfo[r0 + sl * kSlice + lane] >> 5);
    if (lane == 0) s_off[sl + 1] = cnt;
  }
  if (tid == 0) s_off[0] = 0;
  if (tid < kMaxSteps) C.reach[tid] = a.reach[tid];
  if (tid < NR) {
    C.live[tid] = tid < nrhs;
    C.act[tid] = 0;
    C.conv[tid] = 0;
    C.itf[tid] = 0;
  }
  __syncthreads();
  if (warp == 0) {
    int base = 0;
    for (int q = 0; q < ncand; q += 32) {
      const int k = q + lane;
      const int v = k < ncand ? s_off[k + 1] : 0;
      const int inc = warp_inclusive_scan<int>(v, lane) + base;
      if (k < ncand) s_off[k + 1] = inc;
      base = __shfl_sync(0xffffffffu, inc, 31);
    }
  }
  __syncthreads();
  int nheld = 0;
  for (int k = 0; k < ncand; k += 32) {  // slices whose entries all fit (a prefix)
    const bool fits = k + lane < ncand && s_off[k + lane + 1] <= a.cap;
    nheld += __popc(__ballot_sync(0xffffffffu, fits));
  }
  for (int sl = warp; sl < nheld; sl += W) {
    const int o = s_off[sl], cnt = s_off[sl + 1] - o;
    const int2* src = a.jent + __ldg(a.rp + r0 + sl * kSlice);
#pragma unroll 4
    for (int k = lane; k < cnt; k += 32) {
      int2 e = __ldg(src + k);
      e.x = Y.translate(e.x);
      ent[o + k] = e;
    }
  }
  __syncthreads();

  // per-block partial sums -> global; after the barrier every block adds all
  // of them in the same order (totals in C.tot)
  auto put_partials = [&](double (&v)[V], double* part) {
    const double ws = warp_sums<V>(v, lane);
    if (lane % (32 / V) == 0) shw[warp][lane / (32 / V)] = ws;
    __syncthreads();
    if (warp < 2 * nrhs) {
      const double s = warp_sum<double>(lane < W ? shw[lane][warp] : 0.0);
      if (lane == 0) part[(int64_t)warp * nb + blockIdx.x] = s;
    }
  };
  auto get_totals = [&](const double* part) {
    if (warp < 2 * nrhs) {
      double s = 0.0;
      for (int k = lane; k < (int)nb; k += 32) s += __ldcg(part + (int64_t)warp * nb + k);
      s = warp_sum<double>(s);
      if (lane == 0) C.tot[warp] = s;
    }
    __syncthreads();
  };

  if (a.warm) {
    // warm start from the x given: ||b|| for the stopping test first
    double v[V];
#pragma unroll
    for (int f = 0; f < V; ++f) v[f] = 0.0;
    for (int64_t i = r0 + tid; i < r1; i += T)
#pragma unroll
      for (int f = 0; f < NR; ++f) {
        if (f >= nrhs) break;
        const double bi = a.b[(int64_t)f * n + i];
        v[2 * f] += bi * bi;
      }
    put_partials(v, a.partd);
    if (!team_sync<TEAM>(ctl, nb, phase, a.wait_ns)) return;
    get_totals(a.partd);
    if (tid < nrhs) C.bn2[tid] = C.tot[2 * tid];
    __syncthreads();
  }

  double* const part = a.partd + (int64_t)nb * 2 * nrhs;
  int it = 0, cyc = 0;
  for (;; ++cyc) {
    // R: true residual in FP64 (x = 0 in the first cycle unless warm)
    double v[V];
#pragma unroll
    for (int f = 0; f < V; ++f) v[f] = 0.0;
    auto residual = [&](int64_t i, const double (&s)[NR], bool zero_x) {
      const double si = a.sc[i];
#pragma unroll
      for (int f = 0; f < NR; ++f) {
        if (f >= nrhs) break;
        if (!C.live[f]) continue;
        const int64_t o = (int64_t)f * n + i;
        if (zero_x) a.x[o] = 0.0;
        const double ri = a.b[o] - s[f];
        const double ti = si * ri;
        a.t[o] = ti;
        v[2 * f] += ri * ri;
        v[2 * f + 1] += ti * ti;
      }
    };
    if (cyc > 0 || a.warm) {
      for (int sl = warp; sl < nsl; sl += W) {
        const int64_t rb = r0 + (int64_t)sl * kSlice;
        const int ri = a.r_smem ? rsm[sl * kSlice + lane] : a.rinfo[rb + lane];
        const int64_t i = rb + (ri & 31);
        const int len = ri >> 5;
        const int maxlen = __shfl_sync(0xffffffffu, len, 0);
        double s[NR];
#pragma unroll
        for (int f = 0; f < NR; ++f) s[f] = 0.0;
        // x was written by other blocks before the barrier (plain loads)
        if (i < n) {
          const double d = a.mdiag[i];
#pragma unroll
          for (int f = 0; f < NR; ++f)
            if (f < nrhs) s[f] = d * a.x[(int64_t)f * n + i];
        }
        const int32_t base = __ldg(a.rp + rb);
        const int2* e0 = a.jent + base + lane;
        const double* m0 = a.jval + base + lane;
        constexpr int U = NR <= 2 ? 4 : 2;
        for (int q = 0; q < maxlen; q += U) {
          int col[U];
          double m[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const bool has = len > q + u;
            col[u] = 0;
            m[u] = 0.0;
            if (has) {
              col[u] = __ldg(&e0->x);
              m[u] = __ldg(m0);
            }
            const int step = __popc(__ballot_sync(0xffffffffu, has));
            e0 += step;
            m0 += step;
          }
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (len > q + u) {
#pragma unroll
              for (int f = 0; f < NR; ++f)
                if (f < nrhs) s[f] += m[u] * a.x[(int64_t)f * n + col[u]];
            }
        }
        if (i < n) residual(i, s, false);
      }
    } else {
      double s[NR];
#pragma unroll
      for (int f = 0; f < NR; ++f) s[f] = 0.0;
      for (int64_t i = r0 + tid; i < r1; i += T) residual(i, s, true);
    }
    put_partials(v, part);
    if (!team_sync<TEAM>(ctl, nb, phase, a.wait_ns)) return;
    get_totals(part);
    if (warp < nrhs) decide(C, warp, lane, cyc, a.warm, it, a.tol, a.k_min, a.k_max);
    __syncthreads();
    // every active field takes the largest step count (more steps only
    // reduce its residual further)
    int K = 0;
#pragma unroll
    for (int f = 0; f < NR; ++f)
      if (f < nrhs && C.act[f] && C.ks[f] > K) K = C.ks[f];
    if (K == 0 || it >= a.max_iter) break;
    if (K > a.max_iter - it) K = a.max_iter - it;

    // U for one row: x += ||t|| S y
    auto update_x = [&](int64_t i, const float (&y)[NR]) {
      const double si = a.sc[i];
#pragma unroll
      for (int f = 0; f < NR; ++f) {
        if (f >= nrhs) break;
        if (C.act[f]) a.x[(int64_t)f * n + i] += (C.sig[f] * si) * f2d(y[f]);
      }
    };
    // I: c = t / ||t|| in FP32, y_1 = c / theta
    const float ith = 1.f / ch.theta;
    for (int64_t i = r0 + tid; i < r1; i += T) {
      float c[NR], y[NR];
#pragma unroll
      for (int f = 0; f < NR; ++f) {
        c[f] = 0.f;
        if (f < nrhs && C.act[f]) c[f] = (float)(a.t[(int64_t)f * n + i] * C.isig[f]);
        y[f] = c[f] * ith;
      }
      if (K == 1) {
        update_x(i, y);
      } else {
        st_row<NR>((a.c_smem ? csm : cg) + (i - r0) * NR, c);
        if constexpr (YSM) st_row<NR>(ysm + (i - r0) * NR, y);
        if constexpr (TEAM == kTeamGrid) st_row<NR>(a.ya + i * NR, y);
      }
    }
    if (!team_sync<TEAM>(ctl, nb, phase, a.wait_ns)) return;
    float rho = 1.f / ch.s1;
    const float idl = 2.f / ch.delta;
    for (int k = 1; k < K; ++k) {   // y_{k+1} from y_k and y_{k-1} (whose place it takes)
      const float rn1 = 1.f / (2.f * ch.s1 - rho);
      const float c1 = rn1 * rho, c2 = rn1 * idl;
      const int h = (k & 1) ^ 1;    // half of the buffers that holds y_k
      const float* cur = ysm + (h ? (int64_t)rows * NR : 0);
      float* nxt = ysm + (h ? 0 : (int64_t)rows * NR);
      const uint32_t half = h ? (uint32_t)rows * NR * 4u : 0u;
      Y.glob = h ? a.yb : a.ya;
      float* gn = h ? a.ya : a.yb;
      const bool last = k + 1 == K;
      for (int sl = warp; sl < nsl; sl += W) {
        const int64_t rb = r0 + (int64_t)sl * kSlice;
        const int ri = a.r_smem ? rsm[sl * kSlice + lane] : a.rinfo[rb + lane];
        const int64_t i = rb + (ri & 31);
        const int loc = sl * kSlice + (ri & 31);
        const int len = ri >> 5;
        const int maxlen = __shfl_sync(0xffffffffu, len, 0);
        const bool valid = i < n;
        float c[NR], y0[NR], y1[NR], w[NR];
#pragma unroll
        for (int f = 0; f < NR; ++f) c[f] = y0[f] = y1[f] = w[f] = 0.f;
        if (valid) {
          if constexpr (YSM) {
            ld_row<NR>(cur + loc * NR, y1);
            if (k > 1) ld_row<NR>(nxt + loc * NR, y0);
          } else {
            ld_row<NR>(Y.glob + i * NR, y1);
            if (k > 1) ld_row<NR>(gn + i * NR, y0);
          }
          ld_row<NR>((a.c_smem ? csm : cg) + (int64_t)loc * NR, c);
        }
        if (sl < nheld) slice_product<NR, TEAM, OWN, true>(ent + s_off[sl], Y, cur, half, len, maxlen, lane, w);
        else slice_product<NR, TEAM, OWN, false>(a.jent + __ldg(a.rp + rb), Y, cur, half, len, maxlen, lane, w);
#pragma unroll
        for (int f = 0; f < NR; ++f) y0[f] = y1[f] + (c1 * (y1[f] - y0[f]) + c2 * (c[f] - (y1[f] + w[f])));
        if (valid) {
          if (last) {
            update_x(i, y0);
          } else {
            if constexpr (YSM) st_row<NR>(nxt + loc * NR, y0);
            if constexpr (TEAM == kTeamGrid) st_row<NR>(gn + i * NR, y0);
          }
        }
      }
      rho = rn1;
      if (!team_sync<TEAM>(ctl, nb, phase, a.wait_ns)) return;
    }
    it += K;
  }
  if (blockIdx.x == 0 && tid < nrhs) {
    ctl->iters[tid] = C.itf[tid];
    ctl->rel[tid] = C.bn2[tid] > 0.0 ? sqrt(C.prev2[tid] / C.bn2[tid]) : 0.0;
    ctl->conv[tid] = C.conv[tid];
  }
}

// S = diag(M)^-1/2 (0 on a row without diagonal)
__global__ void k_jacobi_sqrt(const double* __restrict__ dinv, int64_t n, double* __restrict__ sc) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    sc[i] = sqrt(dinv[i]);
}

// the off-diagonal entries of S M S as jagged diagonals: one warp per slice
__global__ void k_scaled_slices(const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
                                const double* __restrict__ val, const double* __restrict__ sc, int64_t n,
                                int64_t nslices, int2* __restrict__ jent, double* __restrict__ jval,
                                double* __restrict__ mdiag, uint16_t* __restrict__ rinfo) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < nslices; s += nw) {
    const int64_t i = s * kSlice + lane;
    int32_t k0 = 0, k1 = 0;
    if (i < n) {
      k0 = __ldg(rp + i);
      k1 = __ldg(rp + i + 1);
    }
    const int mylen = k1 > k0 ? k1 - k0 - 1 : 0;   // a non-empty row has its diagonal
    // rank of the row by length (longest first, ties by row)
    int rank = 0;
#pragma unroll
    for (int l = 0; l < 32; ++l) {
      const int o = __shfl_sync(0xffffffffu, mylen, l);
      rank += o > mylen || (o == mylen && l < lane);
    }
    // the row that lane takes: the inverse of the ranks
    int row = 0;
#pragma unroll
    for (int l = 0; l < 32; ++l)
      if (__shfl_sync(0xffffffffu, rank, l) == lane) row = l;
    const int len = __shfl_sync(0xffffffffu, mylen, row);
    const int32_t q0 = __shfl_sync(0xffffffffu, k0, row), q1 = __shfl_sync(0xffffffffu, k1, row);
    const int32_t base = __shfl_sync(0xffffffffu, k0, 0);
    const int maxlen = __shfl_sync(0xffffffffu, len, 0);
    const int32_t me = (int32_t)(s * kSlice) + row;
    const double si = len > 0 ? __ldg(sc + me) : 0.0;
    rinfo[s * kSlice + lane] = (uint16_t)(row | (len << 5));
    int32_t k = q0;
    int32_t out = base + lane;
    double diag = 0.0;
    for (int q = 0; q < maxlen; ++q) {
      const bool has = len > q;
      if (has) {
        int32_t c = __ldg(col + k);
        if (c == me) {   // the diagonal is kept apart
          diag = __ldg(val + k);
          c = __ldg(col + ++k);
        }
        const double m = __ldg(val + k);
        jent[out] = make_int2(c, __float_as_int((float)(m * si * __ldg(sc + c))));
        jval[out] = m;
        ++k;
      }
      out += __popc(__ballot_sync(0xffffffffu, has));
    }
    if (me < n) {
      // a diagonal after the row's last off-diagonal entry was not passed
      if (diag == 0.0 && k < q1) diag = __ldg(val + k);
      mdiag[me] = diag;
    }
  }
}

// (the arrays become the target's together, once all are there and their
// kernels are launched: a call that fails half-way leaves none behind)
sft_status scaled_slices(sft_target_s* t, cudaStream_t st) {
  if (t->jent) return SFT_OK;
  const int64_t n = t->nv, ns = (n + kSlice - 1) / kSlice;
  DevBuf<double> sc(st), jval(st), mdiag(st);
  DevBuf<uint16_t> rinfo(st);
  DevBuf<int2> jent(st);
  SFT_CUDA(sc.alloc((size_t)n));
  SFT_CUDA(rinfo.alloc((size_t)(ns * kSlice)));
  SFT_CUDA(jval.alloc((size_t)t->nnz));
  SFT_CUDA(mdiag.alloc((size_t)n));
  SFT_CUDA(jent.alloc((size_t)t->nnz));
  const unsigned nbj = (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16));
  ::sft::note_launch(), k_jacobi_sqrt<<<nbj, 256, 0, st>>>(t->dinv, n, sc.p);
  SFT_CUDA(cudaGetLastError());
  const unsigned nb = (unsigned)std::max<int64_t>(1, std::min<int64_t>((ns + 7) / 8, 152 * 16));
  ::sft::note_launch(), k_scaled_slices<<<nb, 256, 0, st>>>(t->row_ptr, t->col, t->val, sc.p, n, ns, jent.p,
                                                           jval.p, mdiag.p, rinfo.p);
  SFT_CUDA(cudaGetLastError());
  t->sc = sc.release();
  t->rinfo = rinfo.release();
  t->jval = jval.release();
  t->mdiag = mdiag.release();
  t->jent = jent.release();
  return SFT_OK;
}

static_assert(sizeof(MixCtl) <= sizeof(CallStatus::solve), "control block larger than its place in the call's status");

static void mix_result(const MixCtl& h, int nrhs, SolveResult* res) {
  for (int f = 0; f < nrhs; ++f) {
    res->iters = std::max(res->iters, (int)h.iters[f]);
    res->rel_resid = std::max(res->rel_resid, h.rel[f]);
    if (!h.conv[f]) res->converged = 0;
  }
}

sft_status finish_solve(const SolveLate& late, const CallStatus& host, SolveResult* res) {
  if (!late.pending) return SFT_OK;
  MixCtl h;
  std::memcpy(&h, host.solve, sizeof(MixCtl));
  if (h.err != 0) return fail(SFT_ERR_DEVICE_STATUS, "solve kernel: a barrier wait expired");
  mix_result(h, late.nrhs, res);
  return SFT_OK;
}

// Work (nonzeros x fields) up to which one block, or one cluster of
// kClusterBlocks, takes the system. A step on one block needs no barrier
// beyond its own, one on a cluster the hardware's (0.3 us) and distributed
// shared memory, one on the grid a counter in L2 (1.2 us); against that stand
// the FP64 phases (two lanes a clock on an SM) and the shared-memory loads of
// few SMs. Measured, kernel time on a block / a cluster / the grid: 784 rows
// 2D 46 / 50 / 76 us, 729 rows 3D 60 / 63 / 101; 2,025 rows 2D 87 / 51 / 77;
// 10,201 rows 2D - / 62 / 81, 22,801 - / 95 / 83; 4,913 rows 3D - / 84 / 106,
// 15,625 - / 135 / 108; 8 fields of 1,681 rows 2D - / 86 / 114, of 6,561
// - / 128 / 118.
constexpr int64_t kBlockWork = 10000;
constexpr int64_t kClusterWork = 110000;
constexpr int kClusterBlocks = 16;

constexpr int64_t kThinShare = 8;      // share of A over what fits, from which little is held (launch_mixed)
constexpr int kThinEntries = 12000;

// Attributes of the solve kernels on the current device, set once per device;
// false when a cluster of kClusterBlocks cannot be resident there.
template <int NR>
static sft_status mixed_attributes(int dev, bool* cluster_ok) {
  static std::mutex mu;
  static int state[64] = {0};  // 0 unset, 1 no cluster, 2 cluster
  std::lock_guard<std::mutex> lk(mu);
  int local = 0;
  int& s = dev >= 0 && dev < 64 ? state[dev] : local;
  if (s == 0) {
    const void* k[4] = {(const void*)k_mixed<NR, kTeamBlock, true>, (const void*)k_mixed<NR, kTeamCluster, true>,
                        (const void*)k_mixed<NR, kTeamGrid, true>, (const void*)k_mixed<NR, kTeamGrid, false>};
    for (const void* f : k)
      SFT_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMixSmemMax));
    SFT_CUDA(cudaFuncSetAttribute(k[1], cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kClusterBlocks);
    cfg.blockDim = dim3(kMixThreads<NR>);
    cfg.dynamicSmemBytes = kMixSmemMax;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = kClusterBlocks;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    int fit = 0;
    const cudaError_t e = cudaOccupancyMaxActiveClusters(&fit, k[1], &cfg);
    if (e != cudaSuccess) cudaGetLastError();
    s = e == cudaSuccess && fit > 0 ? 2 : 1;
  }
  *cluster_ok = s == 2;
  return SFT_OK;
}

template <int NR>
static sft_status launch_mixed(sft_target_s* t, int nrhs, const double* b, double* x, double tol, int max_iter,
                               cudaStream_t st, SolveResult* res, SolveLate* late, int warm) {
  const int64_t n = t->nv, ns = (n + kSlice - 1) / kSlice;
  int dev = 0, sms = 0;
  SFT_CUDA(cudaGetDevice(&dev));
  SFT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  bool cluster = false;
  if (sft_status r = mixed_attributes<NR>(dev, &cluster)) return r;
  const int64_t work = std::max<int64_t>(t->nnz, n) * NR;
  const int team = work <= kBlockWork ? kTeamBlock : (cluster && work <= kClusterWork ? kTeamCluster : kTeamGrid);
  const int64_t most = team == kTeamBlock ? 1 : (team == kTeamCluster ? kClusterBlocks : sms);
  MixArgs a;
  a.spb = (int)((ns + most - 1) / most);
  // the cluster keeps its size; a grid leaves out blocks that would own no slice
  const unsigned nblocks = (unsigned)(team == kTeamGrid ? (ns + a.spb - 1) / a.spb : most);
  const int64_t rows = (int64_t)a.spb * kSlice;
  // own rows of y in shared memory, and c and rinfo beside them, where they
  // leave room for A
  const bool own = rows * NR * 8 <= 128 * 1024;
  a.c_smem = own && rows * NR * 12 <= 128 * 1024;
  a.r_smem = rows * 2 <= 32 * 1024;
  const int64_t fixed = (own ? rows * NR * 8 : 0) + (a.c_smem ? rows * NR * 4 : 0) + (a.r_smem ? rows * 2 : 0);
  // shared memory for the block's share of A (with room for uneven shares)
  const int64_t want = t->nnz * a.spb / std::max<int64_t>(ns, 1) * 5 / 4 + 1024;
  a.cap = (int)(std::min<int64_t>(want, ((int64_t)kMixSmemMax - fixed) / 8) & ~(int64_t)1);  // 16-byte multiple
  // Where hardly any of the share fits and y is gathered from global memory,
  // the gathers gain more from L1 than the held entries save: then only
  // kThinEntries (96 KB) are held. Call times of k_mixed before it had the
  // rule, with it, and of the kernel of four blocks per SM without shared
  // memory that it replaced: 3.0 M rows 3D 3,065 / 2,780 / 3,165 us, 4.5 M
  // 4,415 / 4,035 / 4,475, 8.0 M 7,776 / 7,085 / 7,700; 2 fields of 2.2 M
  // 2,667 / 2,266 / 3,707. Below the line holding all that fits is better: 3.0 M
  // rows 2D (a fifth held) 1,695 against 1,756, 4 fields of 1.4 M rows 3D 3,493
  // against 3,532, of 0.64 M 1,226 against 1,466.
  if (!own && want > kThinShare * (int64_t)a.cap) a.cap = std::min(a.cap, kThinEntries);
  const size_t smem = (size_t)a.cap * 8 + (size_t)fixed;
  const void* kern = team == kTeamBlock     ? (const void*)k_mixed<NR, kTeamBlock, true>
                     : team == kTeamCluster ? (const void*)k_mixed<NR, kTeamCluster, true>
                     : own                  ? (const void*)k_mixed<NR, kTeamGrid, true>
                                            : (const void*)k_mixed<NR, kTeamGrid, false>;
  Carve lay;  // one allocation for the work vectors
  const size_t o_ctl = lay.add(late ? 0 : sizeof(MixCtl));
  const size_t o_t = lay.add(sizeof(double) * (size_t)n * nrhs);
  const size_t o_part = lay.add(sizeof(double) * (size_t)nblocks * nrhs * 4);
  const size_t o_ya = lay.add(team == kTeamGrid ? sizeof(float) * (size_t)n * NR : 0);
  const size_t o_yb = lay.add(team == kTeamGrid ? sizeof(float) * (size_t)n * NR : 0);
  const size_t o_c = lay.add(a.c_smem ? 0 : sizeof(float) * (size_t)n * NR);
  DevBuf<char> ws(st);
  SFT_CUDA(ws.alloc(lay.total));
  if (late) {
    a.ctl = reinterpret_cast<MixCtl*>(late->dev);  // zeroed by the caller
  } else {
    a.ctl = reinterpret_cast<MixCtl*>(ws.p + o_ctl);
    SFT_CUDA(cudaMemsetAsync(a.ctl, 0, sizeof(MixCtl), st));
  }
  a.rp = t->row_ptr;
  a.jent = t->jent;
  a.jval = t->jval;
  a.mdiag = t->mdiag;
  a.rinfo = t->rinfo;
  a.sc = t->sc;
  a.n = n;
  a.nrhs = nrhs;
  a.b = b;
  a.x = x;
  a.t = reinterpret_cast<double*>(ws.p + o_t);
  a.ya = reinterpret_cast<float*>(ws.p + o_ya);
  a.yb = reinterpret_cast<float*>(ws.p + o_yb);
  a.c = reinterpret_cast<float*>(ws.p + o_c);
  a.partd = reinterpret_cast<double*>(ws.p + o_part);
  a.tol = tol;
  a.max_iter = max_iter;
  a.warm = warm;
  a.wait_ns = t->wait_ns;
  a.lmax = t->dim == 2 ? 2.f : 2.5f;  // largest eigenvalue bound of S M S
  {
    const double s1 = cheb_coef(a.lmax).s1;
    double t0 = 1.0, t1 = s1;   // T_{K-1}, T_K
    a.k_min = a.k_max = 0;
    for (int k = 1; k < kMaxSteps; ++k) {
      a.reach[k] = (0.1 * tol * t1) * (0.1 * tol * t1);
      if (!a.k_min && t1 >= 4.0) a.k_min = k;
      if (!a.k_max && t1 * kEtaFloor >= 1.0) a.k_max = k;
      const double t2 = 2.0 * s1 * t1 - t0;
      t0 = t1;
      t1 = t2;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nblocks);
  cfg.blockDim = dim3(kMixThreads<NR>);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr = {};
  if (team == kTeamCluster) {
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = kClusterBlocks;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  } else {
    attr.id = cudaLaunchAttributeCooperative;
    attr.val.cooperative = team == kTeamGrid;
  }
  cfg.attrs = &attr;
  cfg.numAttrs = team == kTeamBlock ? 0 : 1;
  void* args[] = {(void*)&a};
  const cudaError_t le = (::sft::note_launch(), cudaLaunchKernelExC(&cfg, kern, args));
  if (le != cudaSuccess) return cuda_fail(le, "launch of the mixed-precision solve");
  if (late) {
    late->nrhs = nrhs;
    late->pending = true;
    return SFT_OK;  // the work buffers are freed in stream order
  }
  Events kit;
  MixCtl& h = *reinterpret_cast<MixCtl*>(kit.host().solve);
  SFT_CUDA(cudaMemcpyAsync(&h, a.ctl, sizeof(MixCtl), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaStreamSynchronize(st));
  if (h.err != 0) return fail(SFT_ERR_DEVICE_STATUS, "solve kernel: a barrier wait expired");
  mix_result(h, nrhs, res);
  return SFT_OK;
}

sft_status mass_solve(sft_target_s* t, int nrhs, const double* b, double* x, double tol, int max_iter,
                      cudaStream_t st, SolveResult* res, int cg_mode, SolveLate* late, int warm) {
  res->iters = 0;
  res->rel_resid = 0.0;
  res->converged = 1;
  const int64_t n = t->nv;
  if (n == 0 || nrhs == 0) return SFT_OK;
  if (nrhs > kMaxFields) return fail(SFT_ERR_ARG, "at most 8 right-hand sides");
  if (max_iter <= 0) {
    SFT_CUDA(cudaMemsetAsync(x, 0, sizeof(double) * n * nrhs, st));
    res->converged = 0;
    return SFT_OK;
  }
  if (warm && cg_mode != SFT_CG_MIXED) return fail(SFT_ERR_UNSUPPORTED, "a warm start needs cg_mode MIXED");
  if (cg_mode == SFT_CG_MIXED) {
    if (sft_status r = scaled_slices(t, st)) return r;
    if (nrhs == 1) return launch_mixed<1>(t, nrhs, b, x, tol, max_iter, st, res, late, warm);
    if (nrhs == 2) return launch_mixed<2>(t, nrhs, b, x, tol, max_iter, st, res, late, warm);
    if (nrhs <= 4) return launch_mixed<4>(t, nrhs, b, x, tol, max_iter, st, res, late, warm);
    return launch_mixed<8>(t, nrhs, b, x, tol, max_iter, st, res, late, warm);
  }
  int dev = 0, sms = 0, coop = 0;
  SFT_CUDA(cudaGetDevice(&dev));
  SFT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  SFT_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  if (!coop) return fail(SFT_ERR_UNSUPPORTED, "device lacks cooperative launch");
  // one thread per row: the FP64 pipe (1 warp instruction / 16 cycles / SM
  // here) is the limiter, and a row-per-thread SpMV issues one DFMA warp
  // instruction per nonzero for 32 rows, with no shuffle reductions
  int per_sm = 0;
  SFT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pcg<1>, kSolveThreads, 0));
  if (per_sm < 1) return fail(SFT_ERR_CUDA, "solver kernel cannot be resident");
  per_sm = std::min(per_sm, 4);
  // at least ~6 rows per thread: fewer blocks make the two grid barriers and
  // the partial sums of every iteration cheaper (measured: 4 blocks per SM
  // for the 1.0 M-row 2D system, about 2 for the 0.5 M-row 3D one)
  constexpr int64_t kRowsPerThread = 6;
  const int64_t want = (n + kSolveThreads * kRowsPerThread - 1) / (kSolveThreads * kRowsPerThread);
  const unsigned nblocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)per_sm * sms, want));

  double *r = nullptr, *z = nullptr, *p = nullptr, *q = nullptr, *part = nullptr;
  PcgCtl* ctl = nullptr;
  const size_t vec = (size_t)n * nrhs;
  SFT_CUDA(dalloc(&r, vec, st));
  SFT_CUDA(dalloc(&z, vec, st));
  SFT_CUDA(dalloc(&p, vec, st));
  SFT_CUDA(dalloc(&q, vec, st));
  SFT_CUDA(dalloc(&part, (size_t)nblocks * nrhs * 2, st));
  SFT_CUDA(dalloc(&ctl, 1, st));
  SFT_CUDA(cudaMemsetAsync(ctl, 0, sizeof(PcgCtl), st));
  const int32_t* rp = t->row_ptr;
  const int32_t* col = t->col;
  const double* val = t->val;
  const double* dinv = t->dinv;
  void* args[] = {(void*)&rp, (void*)&col, (void*)&val, (void*)&dinv, (void*)&n, (void*)&nrhs, (void*)&b,
                  (void*)&x, (void*)&r, (void*)&z, (void*)&p, (void*)&q, (void*)&part,
                  (void*)&ctl, (void*)&tol, (void*)&max_iter, (void*)&t->wait_ns};
  cudaError_t le;
  le = (::sft::note_launch(), cudaLaunchCooperativeKernel((const void*)k_pcg<1>, nblocks, kSolveThreads, args, 0, st));
  if (le != cudaSuccess) return cuda_fail(le, "cudaLaunchCooperativeKernel(k_pcg)");
  PcgCtl h;
  SFT_CUDA(cudaMemcpyAsync(&h, ctl, sizeof(PcgCtl), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaStreamSynchronize(st));
  dfree(r, st); dfree(z, st); dfree(p, st); dfree(q, st); dfree(part, st); dfree(ctl, st);
  if (h.err != 0) return fail(SFT_ERR_DEVICE_STATUS, "CG kernel: grid barrier wait expired");
  for (int f = 0; f < nrhs; ++f) {
    res->iters = std::max(res->iters, (int)h.iters[f]);
    res->rel_resid = std::max(res->rel_resid, h.rel[f]);
    if (!h.conv[f]) res->converged = 0;
  }
  return SFT_OK;
}

// deterministic FP64 sum of w_i u_i (the integral of a P1 target field with lumped masses)
__global__ void k_wsum_partial(const double* __restrict__ w, const double* __restrict__ u, int64_t n,
                               double* __restrict__ part) {
  double s = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    s += w[i] * u[i];
  __shared__ double sh[8];
  s = warp_sum<double>(s);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < (int)(blockDim.x / 32); ++k) t += sh[k];
    part[blockIdx.x] = t;
  }
}

sft_status weighted_sum_launch(const double* w, const double* u, int64_t n, double* part, cudaStream_t st) {
  ::sft::note_launch(), k_wsum_partial<<<kWsumBlocks, 256, 0, st>>>(w, u, n, part);
  SFT_CUDA(cudaGetLastError());
  return SFT_OK;
}

}  // namespace sft

// ---------------------------------------------------------------------------
// Allocation-free variant of the CG solve (no counterpart in the paper).
//
// Some callers cannot allocate device memory when they need a solve: for
// example a coupled simulation that hands all device memory to its own pool
// up front, or a time-stepping loop that must not call cudaMalloc/cudaFree
// because they synchronise the device and can fail mid-run. This entry point
// takes the CSR matrix, right-hand sides and solution buffers from the caller
// and keeps its work vectors in one fixed, file-scope device array instead.
// ---------------------------------------------------------------------------
namespace sft {

// 32 MiB of work space, resident on every device that loads the library
constexpr size_t kStaticScratchBytes = 32ull << 20;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];

static std::mutex g_static_mu;
static void* g_static_ptr[64] = {nullptr};

// Device address of the scratch array for the current device: looked up once
// per device (with that device current) and cached.
static sft_status static_scratch(void** out) {
  int dev = 0;
  SFT_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return fail(SFT_ERR_UNSUPPORTED, "device ordinal >= 64");
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!g_static_ptr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(static scratch)");
    g_static_ptr[dev] = p;
  }
  *out = g_static_ptr[dev];
  return SFT_OK;
}

// Jacobi inverse of the caller's matrix; a row without a positive diagonal
// entry (the matrix cannot be SPD) sets DEV_BAD_DIAGONAL, reported as
// SFT_ERR_ARG (the CG kernel sees the error word and leaves at its first
// barrier)
__global__ void k_jacobi_inverse(const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
                                 const double* __restrict__ val, int64_t n, double* __restrict__ dinv,
                                 int32_t* err) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    double d = 0.0;
    for (int32_t k = rp[i]; k < rp[i + 1]; ++k)
      if (col[k] == i) d = val[k];
    if (!(d > 0.0)) set_error(err, DEV_BAD_DIAGONAL);
    dinv[i] = d > 0.0 ? 1.0 / d : 0.0;
  }
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace sft

extern "C" sft_status sft_mass_solve_static(int64_t n, const int32_t* row_ptr, const int32_t* col,
                                            const double* val, int32_t nrhs, const double* b, double* u,
                                            double tol, int32_t max_iter, void* cuda_stream,
                                            int32_t* iters_out, double* rel_resid_out) {
  using namespace sft;
  if (n <= 0 || !row_ptr || !col || !val || !b || !u) return fail(SFT_ERR_ARG, "null argument or n <= 0");
  if (nrhs < 1 || nrhs > kMaxFields) return fail(SFT_ERR_ARG, "nrhs must be in 1..8");
  if (max_iter < 1 || !(tol >= 0)) return fail(SFT_ERR_ARG, "bad solver options");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  int dev = 0, sms = 0, coop = 0;
  SFT_CUDA(cudaGetDevice(&dev));
  SFT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  SFT_CUDA(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
  if (!coop) return fail(SFT_ERR_UNSUPPORTED, "device lacks cooperative launch");
  int per_sm = 0;
  SFT_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pcg<1>, kSolveThreads, 0));
  if (per_sm < 1) return fail(SFT_ERR_CUDA, "solver kernel cannot be resident");
  per_sm = std::min(per_sm, 4);
  // at least ~6 rows per thread: fewer blocks make the two grid barriers and
  // the partial sums of every iteration cheaper (measured: 4 blocks per SM
  // for the 1.0 M-row 2D system, about 2 for the 0.5 M-row 3D one)
  constexpr int64_t kRowsPerThread = 6;
  const int64_t want = (n + kSolveThreads * kRowsPerThread - 1) / (kSolveThreads * kRowsPerThread);
  const unsigned nblocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((int64_t)per_sm * sms, want));
  // layout: dinv [n] | r, z, p, q [nrhs][n] | partials [nblocks][nrhs][2] | control block
  const size_t vec = sizeof(double) * (size_t)n * nrhs;
  const size_t off_dinv = 0;
  const size_t off_r = align256(off_dinv + sizeof(double) * (size_t)n);
  const size_t off_z = align256(off_r + vec);
  const size_t off_p = align256(off_z + vec);
  const size_t off_q = align256(off_p + vec);
  const size_t off_part = align256(off_q + vec);
  const size_t off_ctl = align256(off_part + sizeof(double) * (size_t)nblocks * nrhs * 2);
  const size_t need = off_ctl + sizeof(PcgCtl);
  if (need > kStaticScratchBytes)
    return fail(SFT_ERR_ARG, "problem too large for the 32 MiB static work space: needs 8 n (1 + 4 nrhs) bytes "
                             "plus partials (n * (1 + 4 nrhs) <= ~4.1e6)");
  void* base = nullptr;
  if (sft_status r = static_scratch(&base)) return r;
  unsigned char* s = static_cast<unsigned char*>(base);
  double* dinv = reinterpret_cast<double*>(s + off_dinv);
  double* r = reinterpret_cast<double*>(s + off_r);
  double* z = reinterpret_cast<double*>(s + off_z);
  double* p = reinterpret_cast<double*>(s + off_p);
  double* q = reinterpret_cast<double*>(s + off_q);
  double* part = reinterpret_cast<double*>(s + off_part);
  PcgCtl* ctl = reinterpret_cast<PcgCtl*>(s + off_ctl);
  // the barrier counters and error word must start at zero; every other
  // region is written by the kernels before it is read
  SFT_CUDA(cudaMemsetAsync(ctl, 0, sizeof(PcgCtl), st));
  ::sft::note_launch(), k_jacobi_inverse<<<(unsigned)std::min<int64_t>((n + 255) / 256, 152 * 16), 256, 0, st>>>(
      row_ptr, col, val, n, dinv, &ctl->err);
  SFT_CUDA(cudaGetLastError());
  const double* dinv_c = dinv;
  const uint64_t wait_ns = kDefaultWaitNs;
  void* args[] = {(void*)&row_ptr, (void*)&col, (void*)&val, (void*)&dinv_c, (void*)&n, (void*)&nrhs, (void*)&b,
                  (void*)&u, (void*)&r, (void*)&z, (void*)&p, (void*)&q, (void*)&part,
                  (void*)&ctl, (void*)&tol, (void*)&max_iter, (void*)&wait_ns};
  const cudaError_t le =
      (::sft::note_launch(), cudaLaunchCooperativeKernel((const void*)k_pcg<1>, nblocks, kSolveThreads, args, 0, st));
  if (le != cudaSuccess) return cuda_fail(le, "cudaLaunchCooperativeKernel(k_pcg, static scratch)");
  PcgCtl h;
  SFT_CUDA(cudaMemcpyAsync(&h, ctl, sizeof(PcgCtl), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaStreamSynchronize(st));
  if (h.err == DEV_BAD_DIAGONAL) return fail(SFT_ERR_ARG, "a row has no positive diagonal entry (matrix not SPD)");
  if (h.err != 0) return fail(SFT_ERR_DEVICE_STATUS, "CG kernel: grid barrier wait expired");
  int it = 0, conv = 1;
  double rel = 0.0;
  for (int f = 0; f < nrhs; ++f) {
    it = std::max(it, (int)h.iters[f]);
    rel = std::max(rel, h.rel[f]);
    if (!h.conv[f]) conv = 0;
  }
  if (iters_out) *iters_out = it;
  if (rel_resid_out) *rel_resid_out = rel;
  if (!conv) return fail(SFT_ERR_NOT_CONVERGED, "CG reached max_iter");
  return SFT_OK;
}
