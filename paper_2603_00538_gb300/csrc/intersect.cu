// Mesh intersection in 2D on the GPU (Sec. 3, Intersection-Based Galerkin
// Projection: the target elements are partitioned by the source elements,
// Eq. partition_ts, and each piece is integrated exactly): the exact P1
// load vector b_i = int psi_i f^s of a P1 mesh source, and the supermesh L2
// error of a target field (Eq. relative_L2_error). It is the exact judge of
// the Monte Carlo transfer at scale and the paper's comparison method.
//
// One thread per target triangle t, all arithmetic FP64:
//   1. locate t's centroid in the source (the location walk): the first
//      source triangle s0 overlaps t with positive area;
//   2. breadth-first over source face neighbours from s0: each visited source
//      triangle is clipped against t (Sutherland-Hodgman) and a piece of
//      positive area is split into a fan from its first vertex and integrated
//      exactly; the neighbours of s are queued. Source triangles overlapping t
//      with positive area form a face-connected set (they tile the convex t),
//      so the walk reaches all of them and touches only their face neighbours
//      besides;
//   3. b: three FP64 atomics per target triangle; L2: per-block partial sums.
// The clipping runs in t's area coordinates A_m = 2 |t| lambda_m (cross
// products with t's edges, exactly 0 at t's own vertices and on axis-parallel
// edges) with the source field carried along as one more linear attribute of
// each polygon vertex: whether a vertex is inside is the sign of a coordinate,
// and both factors of every integrand are known at the polygon's vertices, so
// int f g over a fan triangle is its area / 12 (sum f sum g + sum f g).
// What bounds it: the FP64 pipe (one warp instruction per 16 cycles and SM;
// 88 % busy), about 180 operations for an overlapping pair and 45 for a
// neighbour that does not overlap, at 6 of 32 lanes (the lanes' walks and
// polygons differ). Clipping in x, y with cross products at every stage and
// the edge-midpoint rule through two barycentric maps per midpoint took about
// 1,000 operations a pair: 1.0 M source, 0.5 M target triangles, load vector
// 17.4 ms, L2 error 18.8 ms, now 5.6 and 5.7. Polygons and the first queue
// entries are in shared memory (dynamic indices).
// Up to kMiQueue source triangles are visited per target triangle; beyond
// that the kernel sets DEV_VALENCE and the call reports SFT_ERR_UNSUPPORTED.
#include <algorithm>
#include <cmath>
#include <vector>
#include "internal.hpp"
#include "util.cuh"

namespace sft {

constexpr int kMiQueue = 256;
constexpr int kMiThreads = 128;

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

// a vertex of a clipped polygon: two area coordinates of the target triangle
// and the source field
struct PV { double a1, a2, f; };

// the point of the edge a -> b at fraction t
__device__ __forceinline__ PV lerp(const PV& a, const PV& b, double t) {
  return PV{fma(t, b.a1 - a.a1, a.a1), fma(t, b.a2 - a.a2, a.a2), fma(t, b.f - a.f, a.f)};
}

constexpr int kMiVerts = 6;      // vertices of a triangle clipped by three half-planes, at most
constexpr int kMiQueueSm = 16;   // queue entries in shared memory

template <bool L2>
__global__ void __launch_bounds__(kMiThreads) k_mi_2d(
    const double* __restrict__ sx, const int32_t* __restrict__ sconn, const int32_t* __restrict__ adj,
    const double* __restrict__ svals, int snf, int field, const GridP<double>* __restrict__ gp,
    const int32_t* __restrict__ cell_start, const int32_t* __restrict__ cell_items,
    const int32_t* __restrict__ cell_first, const double* __restrict__ recs, const double* __restrict__ tx,
    const int32_t* __restrict__ tconn, int64_t net, const double* __restrict__ u, double* __restrict__ b,
    double* __restrict__ part, int32_t* err) {
  __shared__ double spoly[2][kMiVerts][3][kMiThreads];
  __shared__ int32_t squeue[kMiQueueSm][kMiThreads];
  const int tid = threadIdx.x;
  const GridP<double> g = *gp;
  double e2 = 0.0, n2 = 0.0;
  int32_t queue[kMiQueue - kMiQueueSm];
  auto put = [&](int buf, int i, const PV& v) {
    spoly[buf][i][0][tid] = v.a1;
    spoly[buf][i][1][tid] = v.a2;
    spoly[buf][i][2][tid] = v.f;
  };
  auto get = [&](int buf, int i) { return PV{spoly[buf][i][0][tid], spoly[buf][i][1][tid], spoly[buf][i][2][tid]}; };
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < net; t += (int64_t)gridDim.x * blockDim.x) {
    P2 tv[3];
    int32_t tn[3];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      tn[m] = __ldg(tconn + t * 3 + m);
      tv[m] = P2{__ldg(tx + (int64_t)tn[m] * 2), __ldg(tx + (int64_t)tn[m] * 2 + 1)};
    }
    // the centroid lies strictly inside t: the source triangle holding it
    // overlaps t with positive area
    double c[2] = {__ddiv_rn(__dadd_rn(__dadd_rn(tv[0].x, tv[1].x), tv[2].x), 3.0),
                   __ddiv_rn(__dadd_rn(__dadd_rn(tv[0].y, tv[1].y), tv[2].y), 3.0)};
    double mu0[3];
    int status = 0;
    const int32_t s0 = locate_point<2, double>(g, cell_start, cell_items, cell_first, recs, adj, c, mu0, status);
    if (s0 < 0) {
      set_error(err, DEV_BAD_INDEX);
      continue;
    }
    const double D = cross3(tv[0], tv[1], tv[2]), rD = 1.0 / D;
    // u = u0 + A_1 g1 + A_2 g2 on t
    double u0 = 0.0, g1 = 0.0, g2 = 0.0;
    if (L2) {
      u0 = __ldg(u + tn[0]);
      g1 = (__ldg(u + tn[1]) - u0) * rD;
      g2 = (__ldg(u + tn[2]) - u0) * rD;
    }
    P2 te[3];  // edges v0 -> v1, v1 -> v2, v2 -> v0 (A_2, A_0, A_1)
#pragma unroll
    for (int m = 0; m < 3; ++m) te[m] = P2{tv[(m + 1) % 3].x - tv[m].x, tv[(m + 1) % 3].y - tv[m].y};
    double q0 = 0.0, q1 = 0.0, q2 = 0.0;  // b: sums of (2 |piece| 2 |t|) f, f A_1, f A_2; L2: (f - u)^2, f^2
    int n = 1, head = 0;
    squeue[0][tid] = s0;
    while (head < n) {
      const int32_t s = head < kMiQueueSm ? squeue[head][tid] : queue[head - kMiQueueSm];
      ++head;
      PV pv[3];
      double a0[3];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const int32_t v = __ldg(sconn + (int64_t)s * 3 + m);
        const double2 x = __ldg(reinterpret_cast<const double2*>(sx) + v);
        pv[m].f = __ldg(svals + ((int64_t)s * snf + field) * 4 + m);
        // separately rounded products: exactly 0 where x is an end of the edge
        pv[m].a2 = __dsub_rn(__dmul_rn(te[0].x, __dsub_rn(x.y, tv[0].y)), __dmul_rn(te[0].y, __dsub_rn(x.x, tv[0].x)));
        a0[m] = __dsub_rn(__dmul_rn(te[1].x, __dsub_rn(x.y, tv[1].y)), __dmul_rn(te[1].y, __dsub_rn(x.x, tv[1].x)));
        pv[m].a1 = __dsub_rn(__dmul_rn(te[2].x, __dsub_rn(x.y, tv[2].y)), __dmul_rn(te[2].y, __dsub_rn(x.x, tv[2].x)));
      }
      const int in0 = (not_neg(a0[0]) ? 1 : 0) | (not_neg(a0[1]) ? 2 : 0) | (not_neg(a0[2]) ? 4 : 0);
      const int in1 = (not_neg(pv[0].a1) ? 1 : 0) | (not_neg(pv[1].a1) ? 2 : 0) | (not_neg(pv[2].a1) ? 4 : 0);
      const int in2 = (not_neg(pv[0].a2) ? 1 : 0) | (not_neg(pv[1].a2) ? 2 : 0) | (not_neg(pv[2].a2) ? 4 : 0);
      if (in0 == 0 || in1 == 0 || in2 == 0) continue;  // outside one edge: nothing left
      // clip by A_0 (from the registers), A_1, A_2
      int k = 0, buf = 0;
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        constexpr int nx[3] = {1, 2, 0};
        const bool ia = (in0 >> m) & 1, ib = (in0 >> nx[m]) & 1;
        if (ia) put(0, k++, pv[m]);
        if (ia != ib) put(0, k++, lerp(pv[m], pv[nx[m]], a0[m] / (a0[m] - a0[nx[m]])));
      }
#pragma unroll
      for (int ax = 1; ax <= 2; ++ax) {
        if ((ax == 1 ? in1 : in2) == 7) continue;  // every vertex of s inside: so is every point of s
        int kk = 0;
        const PV first = get(buf, 0);
        PV cur = first;
        for (int i = 0; i < k; ++i) {
          const PV nxt = i + 1 < k ? get(buf, i + 1) : first;
          const double ca = ax == 1 ? cur.a1 : cur.a2, cb = ax == 1 ? nxt.a1 : nxt.a2;
          const bool ia = not_neg(ca), ib = not_neg(cb);
          if (ia) put(buf ^ 1, kk++, cur);
          if (ia != ib) {
            PV x = lerp(cur, nxt, ca / (ca - cb));
            if (ax == 1) x.a1 = 0.0;
            else x.a2 = 0.0;
            put(buf ^ 1, kk++, x);
          }
          cur = nxt;
        }
        k = kk;
        buf ^= 1;
        if (k == 0) break;
      }
      if (k < 3) continue;
      bool overlap = false;
      const PV o = get(buf, 0);
      PV p = get(buf, 1);
      // (f - u) at the vertices
      double od = 0.0, pd = 0.0;
      if (L2) {
        od = o.f - fma(o.a2, g2, fma(o.a1, g1, u0));
        pd = p.f - fma(p.a2, g2, fma(p.a1, g1, u0));
      }
      for (int i = 2; i < k; ++i) {  // fan from the first vertex
        const PV q = get(buf, i);
        double qd = 0.0;
        if (L2) qd = q.f - fma(q.a2, g2, fma(q.a1, g1, u0));
        const double cr = fma(p.a1 - o.a1, q.a2 - o.a2, -((p.a2 - o.a2) * (q.a1 - o.a1)));
        if (positive(cr)) {
          overlap = true;
          const double sf = o.f + p.f + q.f;
          if (L2) {
            const double sd = od + pd + qd;
            q0 = fma(cr, fma(sd, sd, fma(od, od, fma(pd, pd, qd * qd))), q0);
            q1 = fma(cr, fma(sf, sf, fma(o.f, o.f, fma(p.f, p.f, q.f * q.f))), q1);
          } else {
            const double s1 = o.a1 + p.a1 + q.a1, s2 = o.a2 + p.a2 + q.a2;
            q0 = fma(cr, sf, q0);
            q1 = fma(cr, fma(s1, sf, fma(o.a1, o.f, fma(p.a1, p.f, q.a1 * q.f))), q1);
            q2 = fma(cr, fma(s2, sf, fma(o.a2, o.f, fma(p.a2, p.f, q.a2 * q.f))), q2);
          }
        }
        p = q;
        pd = qd;
      }
      if (!overlap) continue;
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const int32_t nb = __ldg(adj + (int64_t)s * 3 + m);
        if (nb < 0) continue;
        bool seen = false;
        for (int i = 0; i < n; ++i) seen = seen || (i < kMiQueueSm ? squeue[i][tid] : queue[i - kMiQueueSm]) == nb;
        if (seen) continue;
        if (n == kMiQueue) {
          set_error(err, DEV_VALENCE);
          head = n;  // stop this element; the call reports the overflow
          break;
        }
        if (n < kMiQueueSm) squeue[n][tid] = nb;
        else queue[n - kMiQueueSm] = nb;
        ++n;
      }
    }
    // a piece's area is cr / (2 D)
    const double w12 = rD * (1.0 / 24.0);
    if (L2) {
      e2 = fma(q0, w12, e2);
      n2 = fma(q1, w12, n2);
    } else {
      const double bf = q0 * (rD * (1.0 / 6.0)), b1 = q1 * (w12 * rD), b2 = q2 * (w12 * rD);
      atomicAdd(b + tn[0], bf - b1 - b2);   // the three basis functions sum to 1
      atomicAdd(b + tn[1], b1);
      atomicAdd(b + tn[2], b2);
    }
  }
  if (L2) {
    __shared__ double sh[2][kMiThreads / 32];
    e2 = warp_sum<double>(e2);
    n2 = warp_sum<double>(n2);
    if ((threadIdx.x & 31) == 0) {
      sh[0][threadIdx.x >> 5] = e2;
      sh[1][threadIdx.x >> 5] = n2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double a = 0.0, c = 0.0;
      for (int w = 0; w < kMiThreads / 32; ++w) {
        a += sh[0][w];
        c += sh[1][w];
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
  const int64_t want = (t->ne + kMiThreads - 1) / kMiThreads;
  const unsigned blocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * 16));
  DevBuf<double> part(st);
  SFT_CUDA(part.alloc((size_t)blocks * 2));
  if (!l2) SFT_CUDA(cudaMemsetAsync(b, 0, sizeof(double) * t->nv, st));
  auto launch = [&](auto kern) {
    ::sft::note_launch(), kern<<<blocks, kMiThreads, 0, st>>>(
        (const double*)L.coordsP, s->conn, L.adj, (const double*)L.vals, s->nf, field, (const GridP<double>*)L.grid,
        L.cell_start, L.cell_items, L.cell_first, (const double*)L.recs, (const double*)t->coordsP[SFT_PREC_FP64], t->conn,
        t->ne, u, b, part.p, d_err.p);
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
