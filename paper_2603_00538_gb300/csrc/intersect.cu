// Mesh intersection in 2D on the GPU (Sec. 3, Intersection-Based Galerkin
// Projection: the target elements are partitioned by the source elements,
// Eq. partition_ts, and each piece is integrated exactly): the exact P1
// load vector b_i = int psi_i f^s of a P1 mesh source, and the supermesh L2
// error of a target field (Eq. relative_L2_error). It is the exact judge of
// the Monte Carlo transfer at scale and the paper's comparison method.
//
// All arithmetic FP64. Per target triangle t:
//   1. locate t's centroid in the source (the location walk): the first
//      source triangle s0 overlaps t with positive area;
//   2. breadth-first over source face neighbours from s0: each visited source
//      triangle is clipped against t (Sutherland-Hodgman) and a piece of
//      positive area is split into a fan from its first vertex and integrated
//      exactly; the neighbours of s are queued. Source triangles overlapping t
//      with positive area form a face-connected set (they tile the convex t),
//      so the walk reaches all of them and touches only their face neighbours
//      besides;
//   3. b: FP64 atomics per pair; L2: per-block partial sums.
// The clipping runs in t's area coordinates A_m = 2 |t| lambda_m (cross
// products with t's edges, exactly 0 at t's own vertices and on axis-parallel
// edges) with the source field carried along as one more linear attribute of
// each polygon vertex: whether a vertex is inside is the sign of a coordinate,
// and both factors of every integrand are known at the polygon's vertices, so
// int f g over a fan triangle is its area / 12 (sum f sum g + sum f g).
// What bounds it: the FP64 pipe (one warp instruction per 16 cycles and SM).
// A warp therefore keeps 32 targets' walks and fills its lanes with (target,
// source triangle) pairs of any of them: the area coordinates of 32 queued
// pairs at a time, then, 32 at a time again, the clipping of those that are
// not outside an edge, with the at most two crossings of an edge line found
// from the signs and computed together. The walks' bookkeeping stays with the
// lane that owns the target. 1.0 M source, 0.5 M target triangles: load vector
// 17.4 ms with clipping in x, y; 5.6 ms with a thread per target in area
// coordinates (6 of 32 lanes active); now 2.1 (FP64 pipe 81 % busy). L2 error 18.8, 5.7, now 2.2.
// Up to kMiQueue source triangles are visited per target triangle; beyond
// that the kernel sets DEV_VALENCE and the call reports SFT_ERR_UNSUPPORTED.
#include <algorithm>
#include <cmath>
#include <vector>
#include "internal.hpp"
#include "util.cuh"

namespace sft {

constexpr int kMiQueue = 256;
constexpr int kMiThreads = 64;

struct P2 { double x, y; };

__device__ __forceinline__ double cross3(P2 o, P2 a, P2 b) {
  return __dsub_rn(__dmul_rn(__dsub_rn(a.x, o.x), __dsub_rn(b.y, o.y)),
                   __dmul_rn(__dsub_rn(a.y, o.y), __dsub_rn(b.x, o.x)));
}

// x >= 0 (x finite; -0 counts) and x > 0 from the bit pattern: FP64
// comparisons use the FP64 pipe
__device__ __forceinline__ bool not_neg(double x) {
  return (uint64_t)__double_as_longlong(x) <= 0x8000000000000000ull;
}
__device__ __forceinline__ bool positive(double x) { return __double_as_longlong(x) > 0; }

// x 2^k by the exponent (FP64 products use the FP64 pipe), |k| <= 1022
__device__ __forceinline__ double scaled(double x, int k) {
  const long long b = __double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7FF;
  if (e > 0 && (unsigned)(e + k - 1) < 2046u) return __longlong_as_double(b + ((long long)k << 52));
  return b << 1 == 0 ? x : x * __longlong_as_double((long long)(1023 + k) << 52);
}

// a vertex of a clipped polygon: two area coordinates of the target triangle
// and the source field
struct PV { double a1, a2, f; };

// the point of the edge a -> b at fraction t
__device__ __forceinline__ PV lerp(const PV& a, const PV& b, double t) {
  return PV{fma(t, b.a1 - a.a1, a.a1), fma(t, b.a2 - a.a2, a.a2), fma(t, b.f - a.f, a.f)};
}

constexpr int kMiVerts = 6;      // vertices of a triangle clipped by three half-planes, at most
constexpr int kMiQueueSm = 20;   // entries of a walk in shared memory, the rest in global
constexpr int kMiBlocks = 5;     // per SM, by shared memory
constexpr int kMiRefill = 8;     // idle lanes that make a warp take new targets

// source triangle holding each target's centroid (it lies strictly inside t:
// that triangle overlaps t with positive area)
__global__ void k_mi_start(const GridP<double>* __restrict__ gp, const int32_t* __restrict__ cell_start,
                           const int32_t* __restrict__ cell_items, const int32_t* __restrict__ cell_first,
                           const double* __restrict__ recs, const int32_t* __restrict__ adj, const double* __restrict__ tx,
                           const int32_t* __restrict__ tconn, int64_t net, int32_t* __restrict__ start, int32_t* err) {
  const GridP<double> g = *gp;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < net; t += (int64_t)gridDim.x * blockDim.x) {
    P2 tv[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const double2 x = __ldg(reinterpret_cast<const double2*>(tx) + __ldg(tconn + t * 3 + m));
      tv[m] = P2{x.x, x.y};
    }
    double c[2] = {__ddiv_rn(__dadd_rn(__dadd_rn(tv[0].x, tv[1].x), tv[2].x), 3.0),
                   __ddiv_rn(__dadd_rn(__dadd_rn(tv[0].y, tv[1].y), tv[2].y), 3.0)};
    double mu0[3];
    int status = 0;
    const int32_t s0 = locate_point<2, double>(g, cell_start, cell_items, cell_first, recs, adj, c, mu0, status);
    if (s0 < 0) set_error(err, DEV_BAD_INDEX);
    start[t] = s0;
  }
}

// what a warp keeps in shared memory
struct alignas(16) MiWarp {
  // targets: vertices 0..5, c (edges v0 -> v1, v1 -> v2, v2 -> v0) (A_2, A_0, A_1) 6..11; of the scaled
  // coordinates L2: 1 / (48 |t|) 12, u = u0 + A_1 g1 + A_2 g2 13..15; b: 1 / (12 |t|) 12, 1 / (96 |t|^2) 13
  double tgt[16][32];
  double poly[2 * kMiVerts - 1][3][32];  // clipped polygons: rows 0..5 and 6..10 in turn
  double surv[12][64];             // pairs to clip: A_0, A_1, A_2, f at the source triangle's vertices
  int32_t surv_s[64];
  int32_t walk[kMiQueueSm][32];    // source triangles of the targets' walks, in the order found
  int32_t len[32];                 // entries of the walk
  int32_t node[3][32];             // the targets' nodes
  int32_t inflight[32];            // pairs of the target in surv
  int32_t pair_s[32];              // pairs of a batch, then the fans of the clipped ones
  uint32_t hit;                    // pairs of the batch that overlap
  uint8_t surv_t[64], pair_t[32];
};

template <bool L2>
__global__ void __launch_bounds__(kMiThreads) k_mi_2d(
    const double* __restrict__ sx, const int32_t* __restrict__ sconn, const int32_t* __restrict__ adj,
    const double* __restrict__ svals, int snf, int field, const int32_t* __restrict__ start,
    const double* __restrict__ tx, const int32_t* __restrict__ tconn, int64_t net, const double* __restrict__ u,
    double* __restrict__ b, double* __restrict__ part, int32_t* __restrict__ far_walk, int32_t* err) {
  __shared__ MiWarp smem[kMiThreads / 32];
  constexpr uint32_t kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  MiWarp& w = smem[threadIdx.x >> 5];
  // consecutive targets per warp
  const int64_t nwarps = (int64_t)gridDim.x * (kMiThreads / 32), per = (net + nwarps - 1) / nwarps;
  const int64_t wid = (int64_t)blockIdx.x * (kMiThreads / 32) + (threadIdx.x >> 5);
  int64_t next = wid * per;
  const int64_t end = next + per < net ? next + per : net;

  double e2 = 0.0, n2 = 0.0;
  int head = 0;                    // entries of the lane's walk that were taken
  int qn = 0;                      // pairs in surv
  int32_t* const far = far_walk + wid * (32 * (kMiQueue - kMiQueueSm));
  w.inflight[lane] = 0;
  w.len[lane] = 0;
  __syncwarp();
  auto entry = [&](int tl, int i) -> int32_t& {
    return i < kMiQueueSm ? w.walk[i][tl] : far[(i - kMiQueueSm) * 32 + tl];
  };

  for (;;) {
    // new targets for the lanes that are done with theirs
    int pend = w.len[lane] - head;
    const uint32_t idle = __ballot_sync(kAll, pend == 0 && w.inflight[lane] == 0);
    int total = __reduce_add_sync(kAll, pend);
    if (next < end && (__popc(idle) >= kMiRefill || total < 32)) {
      const int64_t t = next + __popc(idle & ((1u << lane) - 1u));
      if ((idle >> lane & 1u) && t < end) {
        const int32_t s0 = __ldg(start + t);
        int32_t tn[3];
        P2 tv[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          tn[m] = __ldg(tconn + t * 3 + m);
          w.node[m][lane] = tn[m];
          const double2 x = __ldg(reinterpret_cast<const double2*>(tx) + tn[m]);
          tv[m] = P2{x.x, x.y};
        }
        // the coordinates are kept as c A_m with c the power of two that brings
        // 2 |t| to d in [1, 2): their products (fourth powers of lengths) then
        // keep clear of FP64's range at any scale of the mesh, with the same bits
        const double D = cross3(tv[0], tv[1], tv[2]);
        const int k = 1023 - min(max((int)(__double_as_longlong(D) >> 52), 1), 2045);   // c = 2^k
        const double rd = 1.0 / scaled(D, k);
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          w.tgt[2 * m][lane] = tv[m].x;
          w.tgt[2 * m + 1][lane] = tv[m].y;
          w.tgt[6 + 2 * m][lane] = scaled(tv[(m + 1) % 3].x - tv[m].x, k);
          w.tgt[7 + 2 * m][lane] = scaled(tv[(m + 1) % 3].y - tv[m].y, k);
        }
        w.tgt[12][lane] = scaled(rd * (L2 ? 1.0 / 24.0 : 1.0 / 6.0), -k);
        if (!L2) {
          w.tgt[13][lane] = scaled(rd * rd * (1.0 / 24.0), -k);
        } else {
          const double u0 = __ldg(u + tn[0]);
          w.tgt[13][lane] = u0;
          w.tgt[14][lane] = (__ldg(u + tn[1]) - u0) * rd;
          w.tgt[15][lane] = (__ldg(u + tn[2]) - u0) * rd;
        }
        w.walk[0][lane] = s0;
        head = 0;
        pend = s0 >= 0 ? 1 : 0;  // (a centroid outside is reported by k_mi_start)
        w.len[lane] = pend;
      }
      next += __popc(idle);
      total = __reduce_add_sync(kAll, pend);
      if (total == 0 && qn == 0 && next < end) continue;
    }
    if (total == 0 && qn == 0) break;

    if (qn < 32 && total > 0 && (total >= 32 || qn == 0)) {
      // area coordinates of up to 32 queued pairs
      int at = warp_inclusive_scan(pend, lane) - pend;
      for (int left = pend; left > 0 && at < 32; --left) {
        w.pair_s[at] = entry(lane, head++);
        w.pair_t[at++] = (uint8_t)lane;
      }
      __syncwarp();
      bool keep = false;
      double a0[3], a1[3], a2[3], f[3];
      int32_t s = 0;
      int tl = 0;
      if (lane < total) {
        s = w.pair_s[lane];
        tl = w.pair_t[lane];
        double2 x[3];
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          x[m] = __ldg(reinterpret_cast<const double2*>(sx) + __ldg(sconn + (int64_t)s * 3 + m));
          f[m] = __ldg(svals + ((int64_t)s * snf + field) * 4 + m);
        }
        // separately rounded products: exactly 0 where x is an end of the edge
        auto area = [&](int e, double dx, double dy) {
          return __dsub_rn(__dmul_rn(w.tgt[6 + 2 * e][tl], dy), __dmul_rn(w.tgt[7 + 2 * e][tl], dx));
        };
        int in0 = 0, in1 = 0, in2 = 0;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          // v0 ends the edges of A_1 and A_2, v1 that of A_0
          const double dx = __dsub_rn(x[m].x, w.tgt[0][tl]), dy = __dsub_rn(x[m].y, w.tgt[1][tl]);
          a2[m] = area(0, dx, dy);
          a0[m] = area(1, __dsub_rn(x[m].x, w.tgt[2][tl]), __dsub_rn(x[m].y, w.tgt[3][tl]));
          a1[m] = area(2, dx, dy);
          in0 |= not_neg(a0[m]);
          in1 |= not_neg(a1[m]);
          in2 |= not_neg(a2[m]);
        }
        keep = in0 && in1 && in2;  // else outside one edge: nothing left
      }
      const uint32_t kept = __ballot_sync(kAll, keep);
      if (keep) {
        const int q = qn + __popc(kept & ((1u << lane) - 1u));
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          w.surv[m][q] = a0[m];
          w.surv[3 + m][q] = a1[m];
          w.surv[6 + m][q] = a2[m];
          w.surv[9 + m][q] = f[m];
        }
        w.surv_s[q] = s;
        w.surv_t[q] = (uint8_t)tl;
        atomicAdd(&w.inflight[tl], 1);
      }
      qn += __popc(kept);
      __syncwarp();
      continue;
    }

    // clip and integrate the last 32 pairs of surv
    const int cnt = qn < 32 ? qn : 32;
    qn -= cnt;
    int tl = 0, k = 0, buf = 1;
    int32_t s = 0;
    if (lane < cnt) {
      const int q = qn + lane;
      tl = w.surv_t[q];
      s = w.surv_s[q];
      atomicSub(&w.inflight[tl], 1);
      // axis 0 from surv, axes 1 and 2 from the polygon
      k = 3;
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        const int from = buf * kMiVerts, to = (buf ^ 1) * kMiVerts;
        auto vert = [&](int i, int c) -> double {   // c: 0 A_1, 1 A_2, 2 f
          return ax == 0 ? w.surv[3 + 3 * c + i][q] : w.poly[from + i][c][lane];
        };
        auto coord = [&](int i) -> double { return ax == 0 ? w.surv[i][q] : w.poly[from + i][ax - 1][lane]; };
        uint32_t in = 0u;
#pragma unroll
        for (int i = 0; i < 3 + ax; ++i)
          if (i < k && not_neg(coord(i))) in |= 1u << i;
        const uint32_t full = (1u << k) - 1u;
        if (ax > 0 && in == full) continue;
        // crossings of edge i -> i + 1; a vertex more than was there at most, by one run of
        // signs (more runs than one, in a polygon thinner than the rounding: the rest is dropped)
        const uint32_t x = (in ^ (in >> 1 | in << (k - 1))) & full;
        const int kk = __popc(in) + __popc(x), most = k + 1;
#pragma unroll
        for (int i = 0; i < 3 + ax; ++i) {
          if (!(in >> i & 1u)) continue;
          const uint32_t below = (1u << i) - 1u;
          const int o = __popc(in & below) + __popc(x & below);
          if (o < most)
#pragma unroll
            for (int c = 0; c < 3; ++c) w.poly[to + o][c][lane] = vert(i, c);
        }
        for (uint32_t rest = x; rest != 0u; rest &= rest - 1u) {
          const int i = __ffs(rest) - 1, j = i + 1 < k ? i + 1 : 0;
          const int o = __popc(in & ((2u << i) - 1u)) + __popc(x & ((1u << i) - 1u));
          const double ca = coord(i), cb = coord(j), t = ca / (ca - cb);
          PV v = lerp(PV{vert(i, 0), vert(i, 1), vert(i, 2)}, PV{vert(j, 0), vert(j, 1), vert(j, 2)}, t);
          if (ax == 1) v.a1 = 0.0;
          if (ax == 2) v.a2 = 0.0;
          if (o < most) {
            w.poly[to + o][0][lane] = v.a1;
            w.poly[to + o][1][lane] = v.a2;
            w.poly[to + o][2][lane] = v.f;
          }
        }
        k = kk < most ? kk : most;
        buf ^= 1;
      }
    }
    // the triangles of the fans from the first vertices, 32 at a time: polygon's lane, its rows, triangle
    uint8_t* const fan = reinterpret_cast<uint8_t*>(w.pair_s);
    const int nf = k > 2 ? k - 2 : 0;
    const int incl = warp_inclusive_scan(nf, lane), nfan = __shfl_sync(kAll, incl, 31);
    for (int i = 0; i < nf; ++i) fan[incl - nf + i] = (uint8_t)(lane | buf << 5 | i << 6);
    if (lane == 0) w.hit = 0u;
    __syncwarp();
    for (int i = lane; i < nfan; i += 32) {
      const int v = fan[i], pl = v & 31, row = (v >> 5 & 1) * kMiVerts, j = row + 1 + (v >> 6), ft = w.surv_t[qn + pl];
      auto get = [&](int r) { return PV{w.poly[r][0][pl], w.poly[r][1][pl], w.poly[r][2][pl]}; };
      const PV o = get(row), p = get(j), r = get(j + 1);
      const double cr = fma(p.a1 - o.a1, r.a2 - o.a2, -((p.a2 - o.a2) * (r.a1 - o.a1)));
      if (!positive(cr)) continue;
      atomicOr(&w.hit, 1u << pl);
      // the triangle's area is cr / (4 |t|)
      const double sf = o.f + p.f + r.f, wt = cr * w.tgt[12][ft];
      if (L2) {
        const double u0 = w.tgt[13][ft], g1 = w.tgt[14][ft], g2 = w.tgt[15][ft];
        // (f - u) at the vertices
        const double od = o.f - fma(o.a2, g2, fma(o.a1, g1, u0)), pd = p.f - fma(p.a2, g2, fma(p.a1, g1, u0)),
                     rd = r.f - fma(r.a2, g2, fma(r.a1, g1, u0)), sd = od + pd + rd;
        e2 = fma(wt, fma(sd, sd, fma(od, od, fma(pd, pd, rd * rd))), e2);
        n2 = fma(wt, fma(sf, sf, fma(o.f, o.f, fma(p.f, p.f, r.f * r.f))), n2);
      } else {
        const double s1 = o.a1 + p.a1 + r.a1, s2 = o.a2 + p.a2 + r.a2, w2 = cr * w.tgt[13][ft];
        const double b1 = w2 * fma(s1, sf, fma(o.a1, o.f, fma(p.a1, p.f, r.a1 * r.f)));
        const double b2 = w2 * fma(s2, sf, fma(o.a2, o.f, fma(p.a2, p.f, r.a2 * r.f)));
        atomicAdd(b + w.node[0][ft], fma(wt, sf, -(b1 + b2)));   // the three basis functions sum to 1
        atomicAdd(b + w.node[1][ft], b1);
        atomicAdd(b + w.node[2][ft], b2);
      }
    }
    __syncwarp();
    const bool overlap = w.hit >> lane & 1u;
    // face neighbours of an overlapping triangle that are new go to its target's walk
    int32_t nb[3] = {-1, -1, -1};
    if (overlap) {
#pragma unroll
      for (int c = 0; c < 3; ++c) nb[c] = __ldg(adj + (int64_t)s * 3 + c);
    }
    int known = 0;   // entries of the walk compared with
    auto strike = [&] {
      if (!overlap) return;
      const int m = w.len[tl];
      for (; known < m; ++known) {
        const int32_t v = entry(tl, known);
#pragma unroll
        for (int c = 0; c < 3; ++c)
          if (nb[c] == v) nb[c] = -1;
      }
    };
    strike();
    __syncwarp();  // (the fans were read)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      // of the pairs that bring the same one the first lane's does
      const bool want = nb[c] >= 0;
      const unsigned long long id = want ? (unsigned long long)tl << 32 | (uint32_t)nb[c] : ~0ull << 8 | (unsigned)lane;
      const uint32_t same = __match_any_sync(kAll, id);
      if (want && (same & ((1u << lane) - 1u)) == 0u) {
        const int at = atomicAdd(&w.len[tl], 1);
        if (at < kMiQueue) entry(tl, at) = nb[c];
        else set_error(err, DEV_VALENCE);
      }
      __syncwarp();
      // (beyond the limit the call fails and reports it: the walk ends there)
      if (w.len[lane] > kMiQueue) w.len[lane] = kMiQueue;
      __syncwarp();
      if (c < 2) strike();
    }
  }
  if (L2) {
    __shared__ double sh[2][kMiThreads / 32];
    e2 = warp_sum<double>(e2);
    n2 = warp_sum<double>(n2);
    if (lane == 0) {
      sh[0][threadIdx.x >> 5] = e2;
      sh[1][threadIdx.x >> 5] = n2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double a = 0.0, c = 0.0;
      for (int i = 0; i < kMiThreads / 32; ++i) {
        a += sh[0][i];
        c += sh[1][i];
      }
      part[blockIdx.x * 2] = a;
      part[blockIdx.x * 2 + 1] = c;
    }
  }
}

// b (load) or the L2 error (L2 = true) of field `field`
sft_status mesh_intersection_2d(sft_source_s* s, sft_target_s* t, int field, const double* u, double* b,
                                double* err_out, double* norm_out, cudaStream_t st) {
  if (s->dim != 2 || t->dim != 2) return fail(SFT_ERR_UNSUPPORTED, "mesh intersection is 2D only");
  if (field < 0 || field >= s->nf) return fail(SFT_ERR_ARG, "field out of range");
  DevBuf<int32_t> d_err(st);
  SFT_CUDA(d_err.alloc(1));
  SFT_CUDA(cudaMemsetAsync(d_err.p, 0, sizeof(int32_t), st));
  if (sft_status r = build_locator(s, SFT_PREC_FP64, st, d_err.p)) return r;
  if (sft_status r = target_coordsP(t, SFT_PREC_FP64, st)) return r;
  const Locator& L = s->loc[SFT_PREC_FP64];
  const bool l2 = u != nullptr;
  int dev = 0, sms = 0;
  SFT_CUDA(cudaGetDevice(&dev));
  SFT_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // warps with fewer targets where that fills the chip; a warp's last pairs leave lanes idle
  const int64_t want = (t->ne + kMiThreads - 1) / kMiThreads;
  const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * kMiBlocks));
  DevBuf<int32_t> start(st), far(st);
  SFT_CUDA(start.alloc((size_t)t->ne));
  SFT_CUDA(far.alloc((size_t)blocks * kMiThreads * (kMiQueue - kMiQueueSm)));
  DevBuf<double> part(st);
  SFT_CUDA(part.alloc((size_t)blocks * 2));
  if (!l2) SFT_CUDA(cudaMemsetAsync(b, 0, sizeof(double) * t->nv, st));
  const double* const tx = (const double*)t->coordsP[SFT_PREC_FP64];
  ::sft::note_launch(), k_mi_start<<<(unsigned)std::min<int64_t>((t->ne + 127) / 128, (int64_t)sms * 64), 128, 0, st>>>(
      (const GridP<double>*)L.grid, L.cell_start, L.cell_items, L.cell_first, (const double*)L.recs, L.adj, tx, t->conn, t->ne,
      start.p, d_err.p);
  SFT_CUDA(cudaGetLastError());
  auto launch = [&](auto kern) {
    ::sft::note_launch(), kern<<<blocks, kMiThreads, 0, st>>>((const double*)L.coordsP, s->conn, L.adj, (const double*)L.vals,
                                                            s->nf, field, start.p, tx, t->conn, t->ne, u, b, part.p, far.p,
                                                            d_err.p);
  };
  if (l2) launch(k_mi_2d<true>);
  else launch(k_mi_2d<false>);
  SFT_CUDA(cudaGetLastError());
  std::vector<double> hp(l2 ? (size_t)blocks * 2 : 0);
  int32_t herr = 0;
  if (l2) SFT_CUDA(cudaMemcpyAsync(hp.data(), part.p, sizeof(double) * hp.size(), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaMemcpyAsync(&herr, d_err.p, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaStreamSynchronize(st));
  if (herr == DEV_VALENCE)
    return fail(SFT_ERR_UNSUPPORTED, "a target triangle overlaps more source triangles than the intersection "
                                     "walk holds (256)");
  if (herr != 0) return fail(SFT_ERR_OUTSIDE, "a target centroid lies outside the source mesh");
  if (l2) {
    double e2 = 0.0, n2 = 0.0;
    for (unsigned i = 0; i < blocks; ++i) {  // fixed order
      e2 += hp[2 * i];
      n2 += hp[2 * i + 1];
    }
    if (err_out) *err_out = std::sqrt(e2);
    if (norm_out) *norm_out = std::sqrt(n2);
  }
  return SFT_OK;
}

}  // namespace sft

using namespace sft;

extern "C" sft_status sft_mi_load_vector(sft_source s, sft_target t, int32_t field, double* b_out,
                                         int32_t out_device, void* cuda_stream) {
  if (!s || !t || !b_out) return fail(SFT_ERR_ARG, "null argument");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  DevBuf<double> tmp(st);
  double* bd = b_out;
  if (!out_device) {
    SFT_CUDA(tmp.alloc((size_t)t->nv));
    bd = tmp.p;
  }
  if (sft_status r = mesh_intersection_2d(s, t, field, nullptr, bd, nullptr, nullptr, st)) return r;
  if (!out_device) {
    SFT_CUDA(cudaMemcpyAsync(b_out, bd, sizeof(double) * t->nv, cudaMemcpyDeviceToHost, st));
    SFT_CUDA(cudaStreamSynchronize(st));
  }
  return SFT_OK;
}

extern "C" sft_status sft_mi_l2_error(sft_source s, sft_target t, int32_t field, const double* u,
                                      int32_t u_on_device, void* cuda_stream, double* out2) {
  if (!s || !t || !u || !out2) return fail(SFT_ERR_ARG, "null argument");
  cudaStream_t st = (cudaStream_t)cuda_stream;
  DevBuf<double> tmp(st);
  const double* ud = u;
  if (!u_on_device) {
    SFT_CUDA(tmp.alloc((size_t)t->nv));
    SFT_CUDA(cudaMemcpyAsync(tmp.p, u, sizeof(double) * t->nv, cudaMemcpyHostToDevice, st));
    ud = tmp.p;
  }
  return mesh_intersection_2d(s, t, field, ud, nullptr, out2, out2 + 1, st);
}
