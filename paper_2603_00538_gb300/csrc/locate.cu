// Source side of the transfer: the uniform-grid point-location structure
// (Sec. 5.3 grid search; cells per axis int(L sqrt(#elements)) in 2D, the
// cube-root analogue in 3D), built on the GPU by a counting sort of
// (cell, element) registrations, and the standalone point-query kernel used
// for the control values g (Sec. 4 step 1) and the query entry point.
//
// Layout in HBM per precision P:
//   recs  [ne][8 | 12] P  : first vertex + inverse affine map (16-B aligned rows)
//   vals  [ne][nf][4]  P  : per-element copy of the nodal values (one 16/32-B load)
//   cell_start [ncells+1], cell_items [nitems] int32: elements of each cell
//   (in no particular order); cell_first [ncells] int32: the element deepest
//   at the cell centre (largest min barycentric coordinate there, ties to the
//   lowest id), where the location walk starts; -1 for an empty cell;
//   adj [ne][d+1] int32: face neighbours (one array per source).
#include <cmath>
#include <vector>
#include "internal.hpp"
#include "util.cuh"

namespace sft {

// cells per axis: the largest n >= 1 with n^d <= L^d * ne; 0 when there would
// be 2^31 - 1 cells or more (a cell's linear index is an int32 everywhere)
static int32_t cells_per_axis(int dim, int64_t ne, double L) {
  const double target = (dim == 2 ? L * L : L * L * L) * (double)ne;
  if (!(target < 1e12)) return 0;
  int64_t n = (int64_t)std::floor(dim == 2 ? std::sqrt(target) : std::cbrt(target));
  if (n < 1) n = 1;
  auto pw = [dim](double x) { return dim == 2 ? x * x : x * x * x; };
  while (pw((double)(n + 1)) <= target) ++n;
  while (n > 1 && pw((double)n) > target) --n;
  return pw((double)n) < (double)INT32_MAX ? (int32_t)n : 0;
}

template <typename TI, typename TO>
__global__ void k_convert(const TI* __restrict__ in, TO* __restrict__ out, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    if constexpr (sizeof(TO) == 4 && sizeof(TI) == 8) out[i] = __double2float_rn(in[i]);
    else out[i] = (TO)in[i];
  }
}

sft_status convert_coords(const void* in, int in_dtype, void* out, int out_prec, int64_t n, cudaStream_t st) {
  if (n <= 0) return SFT_OK;
  const unsigned blocks = (unsigned)std::min<int64_t>((n + 255) / 256, 65535 * 8);
  if (in_dtype == SFT_F64 && out_prec == SFT_PREC_FP32)
    ::sft::note_launch(), k_convert<double, float><<<blocks, 256, 0, st>>>((const double*)in, (float*)out, n);
  else if (in_dtype == SFT_F64)
    ::sft::note_launch(), k_convert<double, double><<<blocks, 256, 0, st>>>((const double*)in, (double*)out, n);
  else if (out_prec == SFT_PREC_FP32)
    ::sft::note_launch(), k_convert<float, float><<<blocks, 256, 0, st>>>((const float*)in, (float*)out, n);
  else
    ::sft::note_launch(), k_convert<float, double><<<blocks, 256, 0, st>>>((const float*)in, (double*)out, n);
  SFT_CUDA(cudaGetLastError());
  return SFT_OK;
}

// ---------------------------------------------------------------------------
// grid box: per-block min/max, then one block combines and forms GridP
// ---------------------------------------------------------------------------
template <int D, typename P>
__global__ void k_bbox_partial(const P* __restrict__ x, int64_t nv, P* __restrict__ part) {
  P lo[D], hi[D];
#pragma unroll
  for (int a = 0; a < D; ++a) { lo[a] = P(INFINITY); hi[a] = P(-INFINITY); }
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const P v = x[i * D + a];
      lo[a] = v < lo[a] ? v : lo[a];
      hi[a] = v > hi[a] ? v : hi[a];
    }
  }
  __shared__ P slo[D][256], shi[D][256];
#pragma unroll
  for (int a = 0; a < D; ++a) { slo[a][threadIdx.x] = lo[a]; shi[a][threadIdx.x] = hi[a]; }
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const P l2 = slo[a][threadIdx.x + s], h2 = shi[a][threadIdx.x + s];
        if (l2 < slo[a][threadIdx.x]) slo[a][threadIdx.x] = l2;
        if (h2 > shi[a][threadIdx.x]) shi[a][threadIdx.x] = h2;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
#pragma unroll
    for (int a = 0; a < D; ++a) { part[blockIdx.x * 2 * D + a] = slo[a][0]; part[blockIdx.x * 2 * D + D + a] = shi[a][0]; }
  }
}

constexpr int kBoxBlocks = 256;  // partial boxes

// one block of kBoxBlocks threads, one partial box each (a single thread over
// all of them took 19 us in FP32 and 65 in FP64, now 3)
template <int D, typename P>
__global__ void __launch_bounds__(kBoxBlocks) k_grid_params(const P* __restrict__ part, int32_t n,
                                                           GridP<P>* __restrict__ g, int32_t* err) {
  __shared__ P slo[D][kBoxBlocks / 32], shi[D][kBoxBlocks / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    P lo = part[threadIdx.x * 2 * D + a], hi = part[threadIdx.x * 2 * D + D + a];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const P l2 = __shfl_xor_sync(0xffffffffu, lo, o), h2 = __shfl_xor_sync(0xffffffffu, hi, o);
      lo = l2 < lo ? l2 : lo;
      hi = h2 > hi ? h2 : hi;
    }
    if (lane == 0) {
      slo[a][warp] = lo;
      shi[a][warp] = hi;
    }
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  GridP<P> r;
#pragma unroll
  for (int a = 0; a < 3; ++a) { r.lo[a] = P(0); r.inv[a] = P(0); r.h[a] = P(0); r.n[a] = 1; }
#pragma unroll
  for (int a = 0; a < D; ++a) {
    P lo = slo[a][0], hi = shi[a][0];
    for (int w = 1; w < kBoxBlocks / 32; ++w) {
      lo = slo[a][w] < lo ? slo[a][w] : lo;
      hi = shi[a][w] > hi ? shi[a][w] : hi;
    }
    if (!(hi > lo)) set_error(err, DEV_BAD_ELEMENT);
    r.lo[a] = lo;
    r.inv[a] = Ar<P>::from_d(__ddiv_rn((double)n, __dsub_rn((double)hi, (double)lo)));
    r.h[a] = Ar<P>::from_d(__ddiv_rn(__dsub_rn((double)hi, (double)lo), (double)n));
    r.n[a] = n;
  }
  *g = r;
}

// ---------------------------------------------------------------------------
// per-element location records + per-element value copies
// ---------------------------------------------------------------------------
template <int D, typename P>
__device__ __forceinline__ void elem_vertices(const P* __restrict__ x, const int32_t* __restrict__ conn, int64_t e,
                                              P xv[D + 1][D]) {
#pragma unroll
  for (int m = 0; m <= D; ++m) {
    const int32_t v = conn[e * (D + 1) + m];
#pragma unroll
    for (int a = 0; a < D; ++a) xv[m][a] = x[(int64_t)v * D + a];
  }
}

template <int D, typename P>
__device__ __forceinline__ int64_t elem_cell_range(const GridP<P>& g, const P xv[D + 1][D], int32_t c0[3], int32_t c1[3]) {
  int64_t cnt = 1;
#pragma unroll
  for (int a = 0; a < 3; ++a) { c0[a] = 0; c1[a] = 0; }
#pragma unroll
  for (int a = 0; a < D; ++a) {
    P lo, hi;
    if constexpr (sizeof(P) == 8) {
      // by the order of the bit patterns (FP64 comparisons use the FP64 pipe);
      // -0 comes before +0, which is the same cell
      auto key = [](double x) {
        const int64_t b = __double_as_longlong(x);
        return b ^ ((b >> 63) & 0x7FFFFFFFFFFFFFFFll);
      };
      int64_t kl = key(xv[0][a]), kh = kl;
#pragma unroll
      for (int m = 1; m <= D; ++m) {
        const int64_t k = key(xv[m][a]);
        kl = k < kl ? k : kl;
        kh = k > kh ? k : kh;
      }
      lo = __longlong_as_double(kl ^ ((kl >> 63) & 0x7FFFFFFFFFFFFFFFll));
      hi = __longlong_as_double(kh ^ ((kh >> 63) & 0x7FFFFFFFFFFFFFFFll));
    } else {
      lo = hi = xv[0][a];
#pragma unroll
      for (int m = 1; m <= D; ++m) {
        lo = xv[m][a] < lo ? xv[m][a] : lo;
        hi = xv[m][a] > hi ? xv[m][a] : hi;
      }
    }
    c0[a] = cell_axis<P>(lo, g.lo[a], g.inv[a], g.n[a]);
    c1[a] = cell_axis<P>(hi, g.lo[a], g.inv[a], g.n[a]);
    cnt *= (int64_t)(c1[a] - c0[a] + 1);
  }
  return cnt;
}

// a*d - b*c in FP32 by Kahan's algorithm (the FMA recovers the rounding error
// of b*c)
__device__ __forceinline__ float det2f(float a, float d, float b, float c) {
  const float w = __fmul_rn(b, c);
  const float e = __fmaf_rn(-b, c, w);
  const float f = __fmaf_rn(a, d, -w);
  return __fadd_rn(f, e);
}

// Inverse affine map of an element into record slots [D .. D + D*D): formed in
// P from the edge vectors, with one correctly rounded reciprocal of the
// determinant (FP32: cofactors and determinant by Kahan's 2x2 determinant).
// Returns false for a non-positive element.
template <int D, typename P>
__device__ __forceinline__ bool record_map(const P xv[D + 1][D], P* r) {
  if constexpr (sizeof(P) == 4) {
    float e[D][D];
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
      for (int a = 0; a < D; ++a) e[k][a] = __fsub_rn(xv[k + 1][a], xv[0][a]);
    if constexpr (D == 2) {
      const float det = det2f(e[0][0], e[1][1], e[1][0], e[0][1]);
      const float inv = __frcp_rn(det);
      r[2] = __fmul_rn(e[1][1], inv);
      r[3] = __fmul_rn(-e[1][0], inv);
      r[4] = __fmul_rn(-e[0][1], inv);
      r[5] = __fmul_rn(e[0][0], inv);
      return det > 0.f;
    } else {
      const float* e1 = e[0];
      const float* e2 = e[1];
      const float* e3 = e[2];
      const float c23[3] = {det2f(e2[1], e3[2], e2[2], e3[1]), det2f(e2[2], e3[0], e2[0], e3[2]),
                            det2f(e2[0], e3[1], e2[1], e3[0])};
      const float c31[3] = {det2f(e3[1], e1[2], e3[2], e1[1]), det2f(e3[2], e1[0], e3[0], e1[2]),
                            det2f(e3[0], e1[1], e3[1], e1[0])};
      const float c12[3] = {det2f(e1[1], e2[2], e1[2], e2[1]), det2f(e1[2], e2[0], e1[0], e2[2]),
                            det2f(e1[0], e2[1], e1[1], e2[0])};
      const float det = __fmaf_rn(e1[2], c23[2], __fmaf_rn(e1[1], c23[1], __fmul_rn(e1[0], c23[0])));
      const float inv = __frcp_rn(det);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        r[3 + q] = __fmul_rn(c23[q], inv);
        r[6 + q] = __fmul_rn(c31[q], inv);
        r[9 + q] = __fmul_rn(c12[q], inv);
      }
      return det > 0.f;
    }
  } else {
    double e[D][D];
#pragma unroll
    for (int k = 0; k < D; ++k)
#pragma unroll
      for (int a = 0; a < D; ++a) e[k][a] = __dsub_rn(xv[k + 1][a], xv[0][a]);
    if constexpr (D == 2) {
      const double det = __dsub_rn(__dmul_rn(e[0][0], e[1][1]), __dmul_rn(e[1][0], e[0][1]));
      const double inv = __drcp_rn(det);
      r[2] = __dmul_rn(e[1][1], inv);
      r[3] = __dmul_rn(-e[1][0], inv);
      r[4] = __dmul_rn(-e[0][1], inv);
      r[5] = __dmul_rn(e[0][0], inv);
      return det > 0.0;
    } else {
      const double* e1 = e[0];
      const double* e2 = e[1];
      const double* e3 = e[2];
      auto crs = [](const double* u, const double* w, double* o) {
        o[0] = __dsub_rn(__dmul_rn(u[1], w[2]), __dmul_rn(u[2], w[1]));
        o[1] = __dsub_rn(__dmul_rn(u[2], w[0]), __dmul_rn(u[0], w[2]));
        o[2] = __dsub_rn(__dmul_rn(u[0], w[1]), __dmul_rn(u[1], w[0]));
      };
      double c23[3], c31[3], c12[3];
      crs(e2, e3, c23);
      crs(e3, e1, c31);
      crs(e1, e2, c12);
      const double det =
          __dadd_rn(__dadd_rn(__dmul_rn(e1[0], c23[0]), __dmul_rn(e1[1], c23[1])), __dmul_rn(e1[2], c23[2]));
      const double inv = __drcp_rn(det);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        r[3 + q] = __dmul_rn(c23[q], inv);
        r[6 + q] = __dmul_rn(c31[q], inv);
        r[9 + q] = __dmul_rn(c12[q], inv);
      }
      return det > 0.0;
    }
  }
}

// L values to a 16-byte aligned row (a multiple of 16 bytes). (With 4-byte
// stores, and the element measure's differences on the FP64 pipe, k_records
// took 293 us for 5.0 M tetrahedra, now 179; that pipe still bounds it.)
template <typename P, int L>
__device__ __forceinline__ void store_row(P* dst, const P (&r)[L]) {
  if constexpr (sizeof(P) == 4) {
#pragma unroll
    for (int q = 0; q < L; q += 4) *reinterpret_cast<float4*>(dst + q) = make_float4(r[q], r[q + 1], r[q + 2], r[q + 3]);
  } else {
#pragma unroll
    for (int q = 0; q < L; q += 2) *reinterpret_cast<double2*>(dst + q) = make_double2(r[q], r[q + 1]);
  }
}

template <int D, typename P, typename TV>
__global__ void k_records(const P* __restrict__ x, const int32_t* __restrict__ conn, const TV* __restrict__ values,
                          int64_t nv, int64_t ne, int nf, P* __restrict__ recs, P* __restrict__ vals, int32_t* err,
                          double* __restrict__ evol) {
  constexpr int L = RecLen<D>::value;
  
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < ne; e += (int64_t)gridDim.x * blockDim.x) {
    int32_t v[D + 1];
    bool ok = true;
#pragma unroll
    for (int m = 0; m <= D; ++m) {
      v[m] = conn[e * (D + 1) + m];
      ok = ok && v[m] >= 0 && v[m] < nv;
    }
    if (!ok) {
      set_error(err, DEV_BAD_INDEX);
      continue;
    }
    P xv[D + 1][D];
    elem_vertices<D, P>(x, conn, e, xv);
    P r[L];
#pragma unroll
    for (int q = 0; q < L; ++q) r[q] = P(0);
#pragma unroll
    for (int a = 0; a < D; ++a) r[a] = xv[0][a];
    if (!record_map<D, P>(xv, r)) set_error(err, DEV_BAD_ELEMENT);
    store_row<P, L>(recs + e * L, r);
    if (evol) evol[e] = elem_measure<D, P>(xv);
    for (int f = 0; f < nf; ++f) {
      P fv[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) fv[m] = m <= D ? P(values[(int64_t)f * nv + v[m]]) : P(0);
      store_row<P, 4>(vals + ((int64_t)e * nf + f) * 4, fv);
    }
  }
}

// centre of cell index i along axis a: lo + (i + 1/2) h as one FMA in P
template <typename P>
__device__ __forceinline__ P cell_centre(const GridP<P>& g, int a, int32_t i) {
  return Ar<P>::fma(Ar<P>::add((P)i, P(0.5)), g.h[a], g.lo[a]);
}

// Can the cell box (centre c, half widths w) hold a point of the element with
// location record r? Each barycentric coordinate is affine; its largest value
// over the box is its value at the centre plus sum_a |gradient_a| w_a. The
// element is left out when that value is below -2^-10 for some coordinate
// (the box lies outside a face plane by a margin far above the predicate's
// rounding, so the test never drops an element a point of the cell could be
// accepted by). Fixed evaluation order in P.
template <int D, typename P>
__device__ __forceinline__ bool cell_may_hold(const P* r, const P c[D], const P w[D]) {
  using A = Ar<P>;
  const P eps = P(0.0009765625);
  P d[D], s[D], tsum = P(0);
#pragma unroll
  for (int a = 0; a < D; ++a) d[a] = A::sub(c[a], r[a]);
#pragma unroll
  for (int m = 0; m < D; ++m) {
    const P* row = r + D + m * D;
    P t = A::mul(row[0], d[0]);
    P sp = A::mul(row[0] < P(0) ? -row[0] : row[0], w[0]);
#pragma unroll
    for (int a = 1; a < D; ++a) {
      t = A::fma(row[a], d[a], t);
      sp = A::fma(row[a] < P(0) ? -row[a] : row[a], w[a], sp);
    }
    if (A::add(t, sp) < -eps) return false;
    tsum = m == 0 ? t : A::add(tsum, t);
#pragma unroll
    for (int a = 0; a < D; ++a) s[a] = m == 0 ? row[a] : A::add(s[a], row[a]);
  }
  P S = A::mul(s[0] < P(0) ? -s[0] : s[0], w[0]);
#pragma unroll
  for (int a = 1; a < D; ++a) S = A::fma(s[a] < P(0) ? -s[a] : s[a], w[a], S);
  return !(A::add(A::sub(P(1), tsum), S) < -eps);
}

// Registration of the elements in the cells of their bounding boxes that pass
// cell_may_hold, and each cell's start element (deepest at the cell centre,
// ties to the lowest id). Two passes, a thread per element:
//   count  tests the box cells; which passed goes to a bit mask (bit k: the
//          k-th box cell in x-fastest order). An element whose centre
//          coordinate is not negative competes for the cell's start element
//          with an atomic maximum of (depth, id);
//   fill   from the masks alone, four registrations of an element in flight:
//          the atomic on the cell's cursor returns the place.
// Elements with more box cells than their mask has bits go to a list that
// k_register_big takes after the others. A mask is one word (MW = 1), or on fine
// grids, where the boxes of ordinary elements are larger, up to kMaskWords.
// (8-byte (id, depth) entries filled one at a time with the full test again,
// and read back for the start elements, took 1.60 ms for the 68 M
// registrations of a 5.0 M-tetrahedron source, 0.43 ms for 4.0 M triangles;
// now 1.08 ms and 0.36; the count pass of 0.61 M FP64 triangles 242 us, now 87.
// Sorting a block's registrations by cell in shared
// memory, with one global atomic per block and cell, took 1.45 ms and 0.42:
// the shared-memory atomics collide.)
constexpr int kMaskCells = 64;   // bits of a mask word
constexpr int kMaskWords = 16;   // of an element at most
constexpr int kRegThreads = 128;

// best (depth, id) at a cell's centre so far: largest depth, lowest id
template <typename P> struct FirstKey;
template <> struct FirstKey<float> { unsigned long long k; };           // depth bits | ~id; 0: none
template <> struct alignas(16) FirstKey<double> { unsigned long long id1, depth; };  // ~id (nonzero), depth bits; 0: none

__device__ __forceinline__ void first_offer(FirstKey<float>* f, float depth, int32_t e) {
  const uint32_t d = __float_as_uint(depth + 0.0f);   // depth >= 0: ordered as its bits (-0 made +0)
  atomicMax(&f->k, ((unsigned long long)d << 32) | (uint32_t)~e);
}
__device__ __forceinline__ void first_offer(FirstKey<double>* f, double depth, int32_t e) {
  const unsigned long long d = (unsigned long long)__double_as_longlong(depth + 0.0), i = (uint32_t)~e;
  unsigned long long od = 0ull, oi = 0ull;
  for (;;) {
    unsigned long long rd, ri;
    asm volatile(
        "{\n\t.reg .b128 c, n, r;\n\tmov.b128 c, {%2, %3};\n\tmov.b128 n, {%4, %5};\n\t"
        "atom.global.cas.b128 r, [%6], c, n;\n\tmov.b128 {%0, %1}, r;\n\t}"
        : "=l"(ri), "=l"(rd)
        : "l"(oi), "l"(od), "l"(i), "l"(d), "l"(f)
        : "memory");
    if (ri == oi && rd == od) return;               // taken
    if (rd > d || (rd == d && ri >= i)) return;     // a better one is there
    oi = ri;
    od = rd;
  }
}

// depth of cell centre cc in the element: its smallest barycentric coordinate
template <int D, typename P>
__device__ __forceinline__ P centre_depth(const P* r, const P (&cc)[D]) {
  P mu[D + 1];
  bary_from_record<D, P>(r, cc, mu);
  P depth = mu[0];
#pragma unroll
  for (int q = 1; q <= D; ++q) depth = mu[q] < depth ? mu[q] : depth;
  return depth;
}

// The coordinates of the box's cell centres as linear functions of the cell's
// offset, in FP32, with a bound of their difference from the evaluation in P
// by cell_may_hold and centre_depth. What lies outside the bound is settled;
// a cell at the threshold, and the depth of a centre that may be in the
// element (one per element on average), are evaluated in P. (In FP64 because its operations are
// 64 times as dear here, in FP32 because the full test takes four times the
// instructions.)
template <int D, typename P>
struct BoxFilter {
  float t0[D], st[D][D], sp[D], S, band;
  // hf = grid steps, mag = bound of the coordinates of the grid, in FP32; nc = cells of the box per axis
  __device__ __forceinline__ void init(const GridP<P>& g, const P* rec, const int32_t c0[3], const float* hf, float mag,
                                       const int (&nc)[3]) {
    constexpr float kEps = sizeof(P) == 4 ? 4.8e-7f : 4e-15f;  // P's rounding of two cell centres (8 and more units)
    float d[D], col[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      d[a] = (float)(cell_centre<P>(g, a, c0[a]) - rec[a]);
      col[a] = 0.f;
    }
    band = 2e-6f;
#pragma unroll
    for (int m = 0; m < D; ++m) {
      float abs_t = 0.f, rsum = 0.f;
      t0[m] = 0.f;
      sp[m] = 0.f;
#pragma unroll
      for (int a = 0; a < D; ++a) {
        const float row = (float)rec[D + m * D + a];
        t0[m] = fmaf(row, d[a], t0[m]);
        abs_t = fmaf(fabsf(row), fabsf(d[a]), abs_t);
        rsum += fabsf(row);
        st[m][a] = row * hf[a];
        sp[m] += 0.5f * fabsf(st[m][a]);
        abs_t = fmaf(fabsf(st[m][a]), (float)nc[a], abs_t);
        col[a] += st[m][a];
      }
      // roundings here (at most 16 x 2^-24 per term), and of the coordinates in P
      band += 2e-6f * abs_t + kEps * mag * rsum;
    }
    S = 0.f;
#pragma unroll
    for (int a = 0; a < D; ++a) S += 0.5f * fabsf(col[a]);
  }
  // coordinates beyond FP32's range for this leave all cells undecided
  __device__ __forceinline__ bool sane(const float* gf, float mag) const {
    bool ok = band < 1e30f && mag < 1e15f;
#pragma unroll
    for (int a = 0; a < D; ++a) ok = ok && gf[a] > 1e-30f;
#pragma unroll
    for (int m = 0; m < D; ++m) ok = ok && fabsf(t0[m]) < 1e30f && sp[m] < 1e30f;
    return ok;
  }
  // the filter that lane j of the warp holds
  __device__ __forceinline__ BoxFilter from_lane(int j) const {
    BoxFilter f;
#pragma unroll
    for (int m = 0; m < D; ++m) {
      f.t0[m] = __shfl_sync(0xffffffffu, t0[m], j);
      f.sp[m] = __shfl_sync(0xffffffffu, sp[m], j);
#pragma unroll
      for (int a = 0; a < D; ++a) f.st[m][a] = __shfl_sync(0xffffffffu, st[m][a], j);
    }
    f.S = __shfl_sync(0xffffffffu, S, j);
    f.band = __shfl_sync(0xffffffffu, band, j);
    return f;
  }
  // cell at offset o[] of the box: 0 not held, 1 held and the centre outside,
  // 2 held and the centre perhaps inside, 3 undecided
  __device__ __forceinline__ int operator()(const float (&o)[3]) const {
    constexpr float eps = 0.0009765625f;
    float t[D], sum = 0.f;
#pragma unroll
    for (int m = 0; m < D; ++m) {
      t[m] = t0[m];
#pragma unroll
      for (int a = 0; a < D; ++a) t[m] = fmaf(st[m][a], o[a], t[m]);
      sum += t[m];
    }
    float mn = 1.f - sum, lo = mn + S;
#pragma unroll
    for (int m = 0; m < D; ++m) {
      lo = fminf(lo, t[m] + sp[m]);
      mn = fminf(mn, t[m]);
    }
    lo += eps;
    if (lo < -band) return 0;
    return lo > band ? (mn < -band ? 1 : 2) : 3;
  }
};

// an element's bounding-box cells: linear index of the first, nx - 1 | ny - 1 << 10 |
// words of its mask << 20
struct ElemBox { int32_t lin0, dims; };

template <int D, typename P, int MW>
__global__ void __launch_bounds__(kRegThreads)
    k_register_count(const P* __restrict__ x, const int32_t* __restrict__ conn, const P* __restrict__ recs, int64_t nv,
                     int64_t ne, const GridP<P>* __restrict__ gp, int32_t* __restrict__ cell_count,
                     FirstKey<P>* __restrict__ first, unsigned long long* __restrict__ mask, ElemBox* __restrict__ box,
                     int32_t* __restrict__ big, int32_t* __restrict__ nbig, int words) {
  constexpr int RL = RecLen<D>::value;
  constexpr int W = kRegThreads / 32;
  __shared__ unsigned long long smask[MW][kRegThreads];     // cells settled in P
  __shared__ int32_t sbox[kRegThreads][4];                  // first box cell, nx - 1 | ny - 1 << 10
  constexpr int kB = MW == 1 ? 6 : 10;                      // bits of k
  __shared__ uint16_t queue[W][64];                         // undecided << (kB + 5) | lane << kB | k
  __shared__ float gf[4];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const GridP<P> g = *gp;
  if (t == 0) {
    float mag = 0.f;
    for (int a = 0; a < D; ++a) {
      gf[a] = (float)g.h[a];
      mag = fmaxf(mag, fabsf((float)g.lo[a]) + fabsf((float)g.h[a]) * (float)g.n[a]);
    }
    gf[3] = mag;
  }
  __syncthreads();
  const int64_t e0 = (int64_t)blockIdx.x * kRegThreads, e = e0 + t;

  // box of the element
  bool ok = e < ne;
  if (ok) {
#pragma unroll
    for (int m = 0; m <= D; ++m) {
      const int32_t v = conn[e * (D + 1) + m];
      ok = ok && v >= 0 && v < nv;  // reported by k_records; never read out of range
    }
  }
  int32_t c0[3] = {0, 0, 0}, c1[3] = {-1, -1, -1};
  if (ok) {
    P xv[D + 1][D];
    elem_vertices<D, P>(x, conn, e, xv);
    const int64_t nb = elem_cell_range<D, P>(g, xv, c0, c1);
    ok = c1[0] >= c0[0] && c1[1] >= c0[1] && c1[2] >= c0[2];  // (non-finite coordinates)
    if (ok && nb > (MW == 1 ? 1 : words) * kMaskCells) {
      big[atomicAdd(nbig, 1)] = (int32_t)e;
      ok = false;
    }
  }
  const int nx = ok ? c1[0] - c0[0] + 1 : 1, ny = ok ? c1[1] - c0[1] + 1 : 1;
  const int nbox = ok ? nx * ny * (c1[2] - c0[2] + 1) : 0;
  const int32_t lin0 = (int32_t)(((int64_t)c0[2] * g.n[1] + c0[1]) * g.n[0] + c0[0]);

  BoxFilter<D, P> filter;
  if (ok) {
    P r[RL];
    load_record<D, P>(recs, (int32_t)e, r);
    const int nc[3] = {nx, ny, c1[2] - c0[2] + 1};
    filter.init(g, r, c0, gf, gf[3], nc);
  }
  const bool sane = ok && filter.sane(gf, gf[3]);
#pragma unroll
  for (int w = 0; w < MW; ++w) smask[w][t] = 0ull;
  sbox[t][0] = c0[0];
  sbox[t][1] = c0[1];
  sbox[t][2] = c0[2];
  sbox[t][3] = (nx - 1) | (ny - 1) << 10;
  __syncwarp();
  // what a warp has to evaluate in P is gathered and taken 32 at a time
  auto settle = [&](int n) {
    __syncwarp();
    if (lane < n) {
      const int q = queue[warp][lane], src = warp * 32 + (q >> kB & 31), k = q & ((1 << kB) - 1);
      const int bx = (sbox[src][3] & 1023) + 1, by = (sbox[src][3] >> 10) + 1;
      const int row = k / bx;
      const int32_t idx[3] = {sbox[src][0] + k - row * bx, sbox[src][1] + (D == 3 ? row % by : row),
                              sbox[src][2] + (D == 3 ? row / by : 0)};
      const int32_t e2 = (int32_t)(e0 + src);
      P r2[RL], cc[D];
      load_record<D, P>(recs, e2, r2);
#pragma unroll
      for (int a = 0; a < D; ++a) cc[a] = cell_centre<P>(g, a, idx[a]);
      const int64_t c = ((int64_t)idx[2] * g.n[1] + idx[1]) * g.n[0] + idx[0];
      bool held = true;
      if (q >> (kB + 5)) {
        P w[D];
#pragma unroll
        for (int a = 0; a < D; ++a) w[a] = Ar<P>::mul(g.h[a], P(0.5));
        held = cell_may_hold<D, P>(r2, cc, w);
        if (held) {
          atomicOr(&smask[MW == 1 ? 0 : k >> 6][src], 1ull << (k & 63));
          atomicAdd(cell_count + c, 1);
        }
      }
      if (held) {
        const P depth = centre_depth<D, P>(r2, cc);
        if (depth >= P(0)) first_offer(first + c, depth, e2);
      }
    }
    __syncwarp();
  };
  const int kmax = __reduce_max_sync(0xffffffffu, nbox);
  const float fx = (float)nx, fy = (float)ny;
  const int32_t ystep = g.n[0] - nx, zstep = g.n[0] * (g.n[1] - ny);
  float o[3] = {0.f, 0.f, 0.f};
  int32_t c = lin0;
  unsigned long long bits = 0ull;
  int qn = 0;
  for (int k = 0; k < kmax; ++k) {
    int res = sane ? filter(o) : 3;
    if (k >= nbox) res = 0;
    if (res == 1 || res == 2) {
      bits |= 1ull << (MW == 1 ? k : k & 63);
      atomicAdd(cell_count + c, 1);
    }
    const uint32_t und = __ballot_sync(0xffffffffu, res >= 2);
    if (und != 0u) {
      if (res >= 2)
        queue[warp][qn + __popc(und & ((1u << lane) - 1u))] = (uint16_t)((res == 3 ? 1 << (kB + 5) : 0) | lane << kB | k);
      qn += __popc(und);
      if (qn >= 32) {
        settle(32);
        qn -= 32;
        if (lane < qn) queue[warp][lane] = queue[warp][32 + lane];
        __syncwarp();
      }
    }
    if (MW > 1 && (k & 63) == 63) {   // (the word is the warp's own: its lanes meet in settle)
      smask[k >> 6][t] |= bits;
      bits = 0ull;
      __syncwarp();
    }
    o[0] += 1.f;
    ++c;
    if (o[0] == fx) {
      o[0] = 0.f;
      o[1] += 1.f;
      c += ystep;
      if (o[1] == fy) {
        o[1] = 0.f;
        o[2] += 1.f;
        c += zstep;
      }
    }
  }
  settle(qn);
  if (e >= ne) return;
  const int mine = (nbox + kMaskCells - 1) / kMaskCells;
  if constexpr (MW == 1) {
    mask[e] = bits | smask[0][t];
  } else {
    for (int w = 0; w < mine; ++w) mask[(int64_t)w * ne + e] = smask[w][t] | (w == kmax >> 6 ? bits : 0ull);
  }
  box[e].lin0 = lin0;
  box[e].dims = (nx - 1) | (ny - 1) << 10 | mine << 20;
}

// The elements beyond their masks: FILL = false counts them, true fills them
// (cell_count then holds the cells' cursors). A warp takes up to 32 of them:
// each lane prepares the box of one (in FP64 also the filter), then the warp
// goes through the boxes one after the other, 32 cells at a time. FP64 settles
// by the filter in both passes what it can, and evaluates the rest in P 32 at a
// time; FP32 evaluates every cell (its test costs less than the filter and what
// follows from it: 162 k tetrahedra at L = 6, source build 3.26 ms, with the
// filter 4.82). One element at a time with every cell in P and 64-bit indices
// took 3.80 ms there in FP32 and 44.0 in FP64 (now 6.3), a thread per element
// 5.20 and 85.8.
constexpr int kBigThreads = 256;

// Words of the masks at grid scale L: an element of a structured mesh takes about
// (1.4 L + 1)^2 cells of a 2D grid, (1.8 L + 1)^3 of a 3D one. One word up to 60
// cells of that (elements a little larger than most are then few), else twice the
// cells, so that few elements are left for k_register_big. Source builds with one
// word and the list / with the words / with 8-byte entries filled one at a time,
// in ms: 2.06 M tetrahedra at L = 2 4.65 / 2.52 / 3.33, at L = 3 9.11 / 5.95 /
// 7.86, in FP64 at L = 2 68.4 / 3.8 / 55.9; 2.0 M triangles at L = 6 4.79 / 3.52 /
// 3.92, in FP64 43.2 / 5.54 / 25.8. Up to the line (L = 1.5 in 3D, 3 in 2D) most
// elements need one word, and the two-word mask gains nothing.
static int mask_words(int dim, double L) {
  const double c = (dim == 2 ? 1.4 : 1.8) * L + 1.0, cells = dim == 2 ? c * c : c * c * c;
  return cells <= 60.0 ? 1 : (int)std::fmin(kMaskWords, std::ceil(2.0 * cells / kMaskCells));
}

template <int D, typename P, bool FILL>
__global__ void __launch_bounds__(kBigThreads, D == 2 || sizeof(P) == 4 ? 3 : 2)
    k_register_big(const P* __restrict__ x, const int32_t* __restrict__ conn, const P* __restrict__ recs,
                   const GridP<P>* __restrict__ gp, const int32_t* __restrict__ big, const int32_t* __restrict__ nbig,
                   int32_t* __restrict__ cell_count, FirstKey<P>* __restrict__ first, int32_t* __restrict__ items) {
  constexpr int RL = RecLen<D>::value;
  constexpr uint32_t kAll = 0xffffffffu;
  constexpr bool kFilter = sizeof(P) == 8;
  __shared__ uint32_t queue[kFilter ? kBigThreads / 32 : 1][64];   // undecided << 31 | cell of the box
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nb = *nbig;
  const int nwarps = (int)gridDim.x * (kBigThreads / 32), wid = (int)blockIdx.x * (kBigThreads / 32) + warp;
  const int per = min(32, (nb + nwarps - 1) / nwarps);   // elements a warp prepares together
  if (nb == 0) return;
  const GridP<P> g = *gp;
  float gf[D], mag = 0.f;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    gf[a] = (float)g.h[a];
    mag = fmaxf(mag, fabsf((float)g.lo[a]) + fabsf((float)g.h[a]) * (float)g.n[a]);
  }
  for (int64_t b0 = (int64_t)wid * per; b0 < nb; b0 += (int64_t)nwarps * per) {
    int32_t my_e = 0, my_c0[3] = {0, 0, 0}, my_nx = 1, my_ny = 1;
    int64_t my_box = 0;
    bool my_sane = false;
    BoxFilter<D, P> mine;
    if (lane < per && b0 + lane < nb) {
      my_e = big[b0 + lane];
      P xv[D + 1][D];
      elem_vertices<D, P>(x, conn, my_e, xv);
      int32_t c1[3];
      my_box = elem_cell_range<D, P>(g, xv, my_c0, c1);
      my_nx = c1[0] - my_c0[0] + 1;
      my_ny = c1[1] - my_c0[1] + 1;
      if constexpr (kFilter) {
        P r[RL];
        load_record<D, P>(recs, my_e, r);
        const int nc[3] = {my_nx, my_ny, c1[2] - my_c0[2] + 1};
        mine.init(g, r, my_c0, gf, mag, nc);
        my_sane = mine.sane(gf, mag);
      }
    }
    const int m = min((int64_t)per, nb - b0);
    for (int j = 0; j < m; ++j) {
      const int32_t e = __shfl_sync(kAll, my_e, j);
      const int nx = __shfl_sync(kAll, my_nx, j), ny = __shfl_sync(kAll, my_ny, j);
      const int64_t nbox = __shfl_sync(kAll, my_box, j);
      int32_t c0[3];
#pragma unroll
      for (int a = 0; a < 3; ++a) c0[a] = __shfl_sync(kAll, my_c0[a], j);
      bool sane = false;
      BoxFilter<D, P> filter;
      P r[RL];
      if constexpr (kFilter) {
        sane = __shfl_sync(kAll, (int)my_sane, j) != 0;
        filter = mine.from_lane(j);
      } else {
        load_record<D, P>(recs, e, r);
      }
      // a cell of the box in P: held? and its centre's depth
      auto place = [&](int ox, int oy, int oz) { return ((c0[2] + oz) * g.n[1] + c0[1] + oy) * g.n[0] + c0[0] + ox; };
      auto in_p = [&](int ox, int oy, int oz, bool test, P& depth) {
        const int32_t idx[3] = {c0[0] + ox, c0[1] + oy, c0[2] + oz};
        P cc[D], w[D];
        if constexpr (kFilter) load_record<D, P>(recs, e, r);
#pragma unroll
        for (int a = 0; a < D; ++a) {
          cc[a] = cell_centre<P>(g, a, idx[a]);
          w[a] = Ar<P>::mul(g.h[a], P(0.5));
        }
        if (test && !cell_may_hold<D, P>(r, cc, w)) return false;
        if (!FILL) depth = centre_depth<D, P>(r, cc);
        return true;
      };
      auto settle = [&](int n) {
        __syncwarp();
        if (lane < n) {
          const uint32_t q = queue[warp][lane], k = q & 0x7fffffffu, row = k / (uint32_t)nx;
          const int ox = (int)(k - row * (uint32_t)nx), oz = (int)(row / (uint32_t)ny), oy = (int)row - oz * ny;
          P depth;
          if (in_p(ox, oy, oz, q >> 31, depth)) {
            const int32_t c = place(ox, oy, oz);
            if (q >> 31) atomicAdd(cell_count + c, 1);
            if (depth >= P(0)) first_offer(first + c, depth, e);
          }
        }
        __syncwarp();
      };
      // the lane's first cell, and 32 cells on, by axis
      int ox = lane % nx, oy = lane / nx % ny, oz = lane / nx / ny;
      const int dx = 32 % nx, dy = 32 / nx % ny, dz = 32 / nx / ny;
      auto decide = [&](int64_t k) {
        const float o[3] = {(float)ox, (float)oy, (float)oz};
        return k >= nbox ? 0 : kFilter && sane ? filter(o) : 3;
      };
      auto step = [&] {
        ox += dx;
        oy += dy;
        oz += dz;
        if (ox >= nx) {
          ox -= nx;
          ++oy;
        }
        if (oy >= ny) {
          oy -= ny;
          ++oz;
        }
      };
      if constexpr (FILL) {
        constexpr int U = 4;   // cells of a lane in flight
        for (int64_t k0 = lane; k0 - lane < nbox; k0 += 32 * U) {
          int32_t* at[U];
          int32_t pos[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int res = decide(k0 + 32 * u);
            P none;
            at[u] = res == 1 || res == 2 || (res == 3 && in_p(ox, oy, oz, true, none)) ? cell_count + place(ox, oy, oz)
                                                                                       : nullptr;
            step();
          }
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (at[u]) pos[u] = atomicAdd(at[u], 1);
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (at[u]) items[pos[u]] = e;
        }
      } else if constexpr (!kFilter) {
        for (int64_t k = lane; k < nbox; k += 32) {
          P depth;
          if (in_p(ox, oy, oz, true, depth)) {
            const int32_t c = place(ox, oy, oz);
            atomicAdd(cell_count + c, 1);
            if (depth >= P(0)) first_offer(first + c, depth, e);
          }
          step();
        }
      } else {
        int qn = 0;
        for (int64_t k0 = 0; k0 < nbox; k0 += 32) {
          const int res = decide(k0 + lane);
          if (res == 1 || res == 2) atomicAdd(cell_count + place(ox, oy, oz), 1);
          const uint32_t und = __ballot_sync(kAll, res >= 2);
          if (und != 0u) {
            if (res >= 2)
              queue[warp][qn + __popc(und & ((1u << lane) - 1u))] = (res == 3 ? 0x80000000u : 0u) | (uint32_t)(k0 + lane);
            qn += __popc(und);
            if (qn >= 32) {
              settle(32);
              qn -= 32;
              if (lane < qn) queue[warp][lane] = queue[warp][32 + lane];
              __syncwarp();
            }
          }
          step();
        }
        settle(qn);
      }
    }
  }
}

// cursor: place of each cell's next registration (its start before the first)
template <int D, int MW>
__global__ void k_register_fill(int64_t ne, int32_t gnx, int32_t gny, const unsigned long long* __restrict__ mask,
                                const ElemBox* __restrict__ box, int32_t* __restrict__ cursor, int32_t* __restrict__ items) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < ne; e += (int64_t)gridDim.x * blockDim.x) {
    const int2 bx = __ldg(reinterpret_cast<const int2*>(box) + e);
    const uint32_t nx = (bx.y & 1023) + 1, ny = (bx.y >> 10 & 1023) + 1;
    const int words = bx.y >> 20;
    // division of k < 1024 by n <= 1024 as (k * ceil(2^20 / n)) >> 20: exact
    const uint32_t inx = (1048575u + nx) / nx, iny = D == 3 ? (1048575u + ny) / ny : 0u;
    for (int w = 0; w < (MW == 1 ? 1 : words); ++w) {
      unsigned long long rest = MW == 1 || words > w ? __ldg(mask + (int64_t)w * ne + e) : 0ull;
      while (rest != 0ull) {
        constexpr int U = 4;
        int32_t* at[U];
        int32_t pos[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          at[u] = nullptr;
          if (rest != 0ull) {
            const uint32_t k = (uint32_t)(w * kMaskCells) + (uint32_t)__ffsll((long long)rest) - 1u;
            rest &= rest - 1ull;
            const uint32_t row = (k * inx) >> 20, lay = D == 3 ? (row * iny) >> 20 : 0u;
            at[u] = cursor + (bx.x + (int32_t)(k - row * nx) + gnx * (int32_t)(row - lay * ny + gny * lay));
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (at[u]) pos[u] = atomicAdd(at[u], 1);
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (at[u]) items[pos[u]] = (int32_t)e;
      }
    }
  }
}

// Start element of each cell from the best offer; a cell whose centre no
// element holds (outside the mesh, or in a rounding gap) takes the deepest of
// its list.
template <int D, typename P>
__global__ void k_cell_first(const int32_t* __restrict__ cell_start, const int32_t* __restrict__ items,
                             const P* __restrict__ recs, const GridP<P>* __restrict__ gp,
                             const FirstKey<P>* __restrict__ key, int64_t ncells, int32_t* __restrict__ first) {
  constexpr int RL = RecLen<D>::value;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < ncells; c += (int64_t)gridDim.x * blockDim.x) {
    const FirstKey<P> k = key[c];
    uint32_t id1;
    if constexpr (sizeof(P) == 4) id1 = (uint32_t)k.k;
    else id1 = (uint32_t)k.id1;
    if (id1 != 0u) {
      first[c] = (int32_t)~id1;
      continue;
    }
    const GridP<P> g = *gp;
    const int32_t idx[3] = {(int32_t)(c % g.n[0]), (int32_t)(c / g.n[0] % g.n[1]), (int32_t)(c / g.n[0] / g.n[1])};
    P cc[D];
#pragma unroll
    for (int a = 0; a < D; ++a) cc[a] = cell_centre<P>(g, a, idx[a]);
    int32_t best = -1;
    P bd = P(0);
    for (int32_t p = __ldg(cell_start + c); p < __ldg(cell_start + c + 1); ++p) {
      const int32_t e = items[p];
      P r[RL];
      load_record<D, P>(recs, e, r);
      const P depth = centre_depth<D, P>(r, cc);
      if (best < 0 || depth > bd || (depth == bd && e < best)) {
        best = e;
        bd = depth;
      }
    }
    first[c] = best;
  }
}

// Face neighbours of every element for the location walk: adj[e][m] = the
// other element holding every vertex of the face opposite local vertex m
// (the smallest id if several), -1 on the boundary. Found through the grid:
// an element holding vertex v has v in its closure, and registration keeps
// every cell a point of the element can fall in, so it is listed in the cell
// of v. Faces m != 0 hold vertex 0 and are matched against the list of
// cell(x_0); face 0 holds vertex 1 and is matched against the list of
// cell(x_1). Two threads per element, one per list (they write different
// entries of the element's row).
template <int D, typename P>
__global__ void k_adjacency(const P* __restrict__ x, const int32_t* __restrict__ conn, int64_t nv, int64_t ne,
                            const GridP<P>* __restrict__ gp, const int32_t* __restrict__ cell_start,
                            const int32_t* __restrict__ cell_items, int32_t* __restrict__ adj) {
  constexpr int K = D + 1;
  const GridP<P> g = *gp;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < 2 * ne; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = i >> 1;
    const int pass = (int)(i & 1);
    int32_t v[K];
    bool ok = true;
#pragma unroll
    for (int m = 0; m < K; ++m) {
      v[m] = __ldg(conn + e * K + m);
      ok = ok && v[m] >= 0 && v[m] < nv;
    }
    int32_t best[K];
#pragma unroll
    for (int m = 0; m < K; ++m) best[m] = INT32_MAX;
    if (ok) {
      P X[D];
      const int32_t vp = pass == 0 ? v[0] : v[1];
#pragma unroll
      for (int a = 0; a < D; ++a) X[a] = __ldg(x + (int64_t)vp * D + a);
      const int32_t c = cell_of<D, P>(g, X);
      const int32_t p1 = __ldg(cell_start + c + 1);
#pragma unroll 2
      for (int32_t p = __ldg(cell_start + c); p < p1; ++p) {
        const int32_t e2 = __ldg(cell_items + p);
        if (e2 == (int32_t)e) continue;
        int32_t w[K];
        if constexpr (D == 3) {
          // (four 4-byte loads kept the L1 data pipe 85 % busy: 782 us for 5.0 M tetrahedra, now 697)
          const int4 q = __ldg(reinterpret_cast<const int4*>(conn) + e2);
          w[0] = q.x; w[1] = q.y; w[2] = q.z; w[3] = q.w;
        } else {
#pragma unroll
          for (int r = 0; r < K; ++r) w[r] = __ldg(conn + (int64_t)e2 * K + r);
        }
        int shared = 0, miss = 0;
#pragma unroll
        for (int m = 0; m < K; ++m) {
          bool in = false;
#pragma unroll
          for (int r = 0; r < K; ++r) in = in || w[r] == v[m];
          shared += in;
          miss = in ? miss : m;
        }
        if (shared != D || (pass == 0) == (miss == 0)) continue;
#pragma unroll
        for (int m = 0; m < K; ++m)
          if (m == miss && e2 < best[m]) best[m] = e2;
      }
    }
    // pass 0 owns faces 1..D, pass 1 face 0
#pragma unroll
    for (int m = 0; m < K; ++m)
      if ((m == 0) == (pass == 1)) adj[e * K + m] = best[m] == INT32_MAX ? -1 : best[m];
  }
}

static unsigned grid_for(int64_t n, int threads = 256) {
  int64_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 152 * 64) b = 152 * 64;
  return (unsigned)b;
}

template <int D, typename P>
static sft_status build_locator_t(sft_source_s* s, int prec, cudaStream_t st, int32_t* d_err) {
  Locator& L = s->loc[prec];
  constexpr int RL = RecLen<D>::value;
  const int32_t n = cells_per_axis(D, s->ne, s->L);
  if (n == 0) return fail(SFT_ERR_UNSUPPORTED, "grid too fine (2^31 - 1 cells or more)");
  // coordinates in P
  P* xP = nullptr;
  SFT_CUDA(dalloc(&xP, (size_t)s->nv * D, st));
  L.coordsP = xP;
  if (sft_status r = convert_coords(s->coords, s->dtype, xP, prec, s->nv * D, st)) return r;
  // grid box and parameters
  L.n[0] = L.n[1] = L.n[2] = 1;
  L.ncells = 1;
  for (int a = 0; a < D; ++a) { L.n[a] = n; L.ncells *= n; }
  P* part = nullptr;
  SFT_CUDA(dalloc(&part, (size_t)kBoxBlocks * 2 * D, st));
  ::sft::note_launch(), k_bbox_partial<D, P><<<kBoxBlocks, 256, 0, st>>>(xP, s->nv, part);
  GridP<P>* g = nullptr;
  SFT_CUDA(dalloc(&g, 1, st));
  L.grid = g;
  ::sft::note_launch(), k_grid_params<D, P><<<1, kBoxBlocks, 0, st>>>(part, n, g, d_err);
  SFT_CUDA(cudaGetLastError());
  dfree(part, st);
  // location records and value copies
  P* recs = nullptr;
  P* vals = nullptr;
  SFT_CUDA(dalloc(&recs, (size_t)s->ne * RL, st));
  SFT_CUDA(dalloc(&vals, (size_t)s->nf * s->ne * 4, st));
  L.recs = recs;
  L.vals = vals;
  // the first locator (the source's own precision, at create) also records
  // every element's FP64 measure for the source integrals
  double* evol = nullptr;
  if (!s->evol) {
    SFT_CUDA(dalloc(&s->evol, (size_t)s->ne, st));
    evol = s->evol;
  }
  if (s->dtype == SFT_F64)
    ::sft::note_launch(), k_records<D, P, double><<<grid_for(s->ne), 256, 0, st>>>(xP, s->conn, (const double*)s->values, s->nv, s->ne,
                                                             s->nf, recs, vals, d_err, evol);
  else
    ::sft::note_launch(), k_records<D, P, float><<<grid_for(s->ne), 256, 0, st>>>(xP, s->conn, (const float*)s->values, s->nv, s->ne,
                                                            s->nf, recs, vals, d_err, evol);
  SFT_CUDA(cudaGetLastError());
  // count registrations per cell, then total (int64) -> int32 offsets must suffice
  // (temporaries freed in stream order on every return)
  DevBuf<int64_t> start64(st);
  DevBuf<char> ws(st);
  SFT_CUDA(start64.alloc((size_t)L.ncells + 1));
  Carve lay;  // the first three start at zero
  const size_t o_count = lay.add(sizeof(int32_t) * (size_t)L.ncells);
  const size_t o_key = lay.add(sizeof(FirstKey<P>) * (size_t)L.ncells);
  const size_t o_nbig = lay.add(sizeof(int32_t)), zeroed = lay.total;
  const int mw = mask_words(D, s->L);
  const size_t o_mask = lay.add(sizeof(unsigned long long) * (size_t)s->ne * mw);
  const size_t o_box = lay.add(sizeof(ElemBox) * (size_t)s->ne);
  const size_t o_big = lay.add(sizeof(int32_t) * (size_t)s->ne);
  SFT_CUDA(ws.alloc(lay.total));
  int32_t* const count = (int32_t*)(ws.p + o_count);
  FirstKey<P>* const key = (FirstKey<P>*)(ws.p + o_key);
  int32_t* const nbig = (int32_t*)(ws.p + o_nbig);
  unsigned long long* const mask = (unsigned long long*)(ws.p + o_mask);
  ElemBox* const box = (ElemBox*)(ws.p + o_box);
  int32_t* const big = (int32_t*)(ws.p + o_big);
  const unsigned reg_blocks = (unsigned)((s->ne + kRegThreads - 1) / kRegThreads);
  constexpr unsigned kBigBlocks = 152 * 4;
  SFT_CUDA(cudaMemsetAsync(ws.p, 0, zeroed, st));
  ::sft::note_launch(), (mw == 1 ? k_register_count<D, P, 1> : k_register_count<D, P, kMaskWords>)<<<reg_blocks, kRegThreads, 0, st>>>(
      xP, s->conn, recs, s->nv, s->ne, g, count, key, mask, box, big, nbig, mw);
  SFT_CUDA(cudaGetLastError());
  ::sft::note_launch(), k_register_big<D, P, false><<<kBigBlocks, kBigThreads, 0, st>>>(xP, s->conn, recs, g, big, nbig, count, key,
                                                                              nullptr);
  SFT_CUDA(cudaGetLastError());
  SFT_CUDA(exclusive_scan_i32_to_i64(count, start64.p, L.ncells, st));
  Events kit;
  SFT_CUDA(cudaMemcpyAsync(&kit.host().err, d_err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaMemcpyAsync(&kit.host().counters[0], start64.p + L.ncells, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaStreamSynchronize(st));
  const int32_t herr = kit.host().err;
  const int64_t total = kit.host().counters[0];
  if (herr != 0)
    return fail(SFT_ERR_MESH, herr == DEV_NONFINITE  ? "non-finite source coordinate"
                              : herr == DEV_BAD_INDEX ? "source connectivity index out of range"
                                                      : "source mesh has a non-positive element or a degenerate box");
  if (total >= (int64_t)INT32_MAX) return fail(SFT_ERR_UNSUPPORTED, "grid registrations exceed 2^31");
  L.nitems = total;
  SFT_CUDA(dalloc(&L.cell_start, (size_t)L.ncells + 1, st));
  SFT_CUDA(narrow_i64_to_i32(start64.p, L.cell_start, L.ncells + 1, st));
  // fill (arbitrary order within a cell), then each cell's start element
  SFT_CUDA(dalloc(&L.cell_items, (size_t)total, st));
  SFT_CUDA(cudaMemcpyAsync(count, L.cell_start, sizeof(int32_t) * (size_t)L.ncells, cudaMemcpyDeviceToDevice, st));
  ::sft::note_launch(), (mw == 1 ? k_register_fill<D, 1> : k_register_fill<D, kMaskWords>)<<<grid_for(s->ne), 256, 0, st>>>(
      s->ne, L.n[0], L.n[1], mask, box, count, L.cell_items);
  SFT_CUDA(cudaGetLastError());
  ::sft::note_launch(), k_register_big<D, P, true><<<kBigBlocks, kBigThreads, 0, st>>>(xP, s->conn, recs, g, big, nbig, count, key,
                                                                             L.cell_items);
  SFT_CUDA(cudaGetLastError());
  SFT_CUDA(dalloc(&L.cell_first, (size_t)L.ncells, st));
  ::sft::note_launch(), k_cell_first<D, P><<<grid_for(L.ncells), 256, 0, st>>>(L.cell_start, L.cell_items, recs, g, key,
                                                                             L.ncells, L.cell_first);
  SFT_CUDA(cudaGetLastError());
  // face neighbours for the location walk (one array per source mesh)
  if (!s->adj) {
    SFT_CUDA(dalloc(&s->adj, (size_t)s->ne * (D + 1), st));
    ::sft::note_launch(), k_adjacency<D, P><<<grid_for(2 * s->ne), 256, 0, st>>>(xP, s->conn, s->nv, s->ne, g, L.cell_start,
                                                                           L.cell_items, s->adj);
    SFT_CUDA(cudaGetLastError());
  }
  L.adj = s->adj;
  L.built = true;
  return SFT_OK;
}

sft_status build_locator(sft_source_s* s, int prec, cudaStream_t st, int32_t* d_err) {
  if (s->loc[prec].built) return SFT_OK;
  if (s->dim == 2)
    return prec == SFT_PREC_FP32 ? build_locator_t<2, float>(s, prec, st, d_err) : build_locator_t<2, double>(s, prec, st, d_err);
  return prec == SFT_PREC_FP32 ? build_locator_t<3, float>(s, prec, st, d_err) : build_locator_t<3, double>(s, prec, st, d_err);
}

// per-element value copies from the nodal values (after a value update)
template <int D, typename P, typename TV>
__global__ void k_value_copies(const int32_t* __restrict__ conn, const TV* __restrict__ values, int64_t nv,
                               int64_t ne, int nf, P* __restrict__ vals) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < ne; e += (int64_t)gridDim.x * blockDim.x) {
    int32_t v[D + 1];
#pragma unroll
    for (int m = 0; m <= D; ++m) v[m] = conn[e * (D + 1) + m];
    for (int f = 0; f < nf; ++f) {
      P fv[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) fv[m] = m <= D ? P(values[(int64_t)f * nv + v[m]]) : P(0);
      store_row<P, 4>(vals + ((int64_t)e * nf + f) * 4, fv);
    }
  }
}

sft_status refresh_value_copies(sft_source_s* s, cudaStream_t st) {
  for (int prec = 0; prec < 2; ++prec) {
    Locator& L = s->loc[prec];
    if (!L.built) continue;
    const unsigned blocks = grid_for(s->ne);
#define SFT_VC(DD, PP, TT)                                                                                  \
  ::sft::note_launch(), k_value_copies<DD, PP, TT><<<blocks, 256, 0, st>>>(s->conn, (const TT*)s->values, s->nv, \
                                                                          s->ne, s->nf, (PP*)L.vals)
    if (s->dim == 2) {
      if (prec == SFT_PREC_FP32) { if (s->dtype == SFT_F64) SFT_VC(2, float, double); else SFT_VC(2, float, float); }
      else { if (s->dtype == SFT_F64) SFT_VC(2, double, double); else SFT_VC(2, double, float); }
    } else {
      if (prec == SFT_PREC_FP32) { if (s->dtype == SFT_F64) SFT_VC(3, float, double); else SFT_VC(3, float, float); }
      else { if (s->dtype == SFT_F64) SFT_VC(3, double, double); else SFT_VC(3, double, float); }
    }
#undef SFT_VC
    SFT_CUDA(cudaGetLastError());
  }
  return SFT_OK;
}

// ---------------------------------------------------------------------------
// point queries: location + P1 evaluation of all fields
// ---------------------------------------------------------------------------
template <int D, typename P, typename TIn, typename TOut>
__global__ void __launch_bounds__(256) k_locate_points(const TIn* __restrict__ pts, int64_t n,
                                                       const GridP<P>* __restrict__ gp,
                                                       const int32_t* __restrict__ cell_start,
                                                       const int32_t* __restrict__ cell_items,
                                                       const int32_t* __restrict__ cell_first,
                                                       const P* __restrict__ recs, const int32_t* __restrict__ adj,
                                                       const P* __restrict__ vals,
                                                       int snf, int nf, int32_t* __restrict__ elem_out,
                                                       TOut* __restrict__ val_out, int64_t val_stride,
                                                       int64_t* __restrict__ counters, P* __restrict__ mu_out) {
  const GridP<P> g = *gp;
  int n_fallback = 0, n_empty = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    P X[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      if constexpr (sizeof(P) == 4 && sizeof(TIn) == 8) X[a] = __double2float_rn(pts[i * D + a]);
      else X[a] = (P)pts[i * D + a];
    }
    P mu[D + 1];
    int status;
    const int32_t e = locate_point<D, P>(g, cell_start, cell_items, cell_first, recs, adj, X, mu, status);
    n_fallback += status == 1;
    n_empty += status == 2;
    if (elem_out) elem_out[i] = e;
    if (mu_out) {
#pragma unroll
      for (int a = 0; a < D; ++a) mu_out[a * n + i] = mu[a + 1];
    }
    if (val_out) {
      for (int f = 0; f < nf; ++f)
        val_out[(int64_t)f * val_stride + i] = e >= 0 ? (TOut)eval_p1<D, P>(vals, snf, f, e, mu) : TOut(0);
    }
  }
  if (counters) {
    const int fb = warp_sum<int>(n_fallback), em = warp_sum<int>(n_empty);
    if ((threadIdx.x & 31) == 0) {
      if (fb) atomicAdd(reinterpret_cast<unsigned long long*>(counters), (unsigned long long)fb);
      if (em) atomicAdd(reinterpret_cast<unsigned long long*>(counters + 1), (unsigned long long)em);
    }
  }
}

template <int D, typename P>
static void launch_locate(sft_source_s* s, const Locator& L, int64_t n, const void* pts, int pts_are_double,
                          int32_t* elem_out, void* val_out, int val_is_double, int64_t val_stride,
                          int64_t* counters, cudaStream_t st, int nf, void* mu_out) {
  const unsigned blocks = grid_for(n);
  const GridP<P>* g = (const GridP<P>*)L.grid;
  const P* recs = (const P*)L.recs;
  const P* vals = (const P*)L.vals;
#define SFT_LOC(TIN, TOUT)                                                                                      \
  ::sft::note_launch(), k_locate_points<D, P, TIN, TOUT><<<blocks, 256, 0, st>>>((const TIN*)pts, n, g, L.cell_start, L.cell_items, \
                                                           L.cell_first,                                    \
                                                           recs, L.adj, vals, s->nf, nf, elem_out,          \
                                                           (TOUT*)val_out,                                   \
                                                           val_stride, counters, (P*)mu_out)
  if (pts_are_double) {
    if (val_is_double) SFT_LOC(double, double); else SFT_LOC(double, P);
  } else {
    if (val_is_double) SFT_LOC(P, double); else SFT_LOC(P, P);
  }
#undef SFT_LOC
}

sft_status locate_points(sft_source_s* s, int prec, int64_t n, const void* pts, int pts_are_double,
                         int32_t* elem_out, void* val_out, int val_is_double, int64_t val_stride,
                         int64_t* d_counters, cudaStream_t st, int nf_out, void* mu_out) {
  const Locator& L = s->loc[prec];
  const int nf = nf_out < 0 ? s->nf : nf_out;
  if (!L.built) return fail(SFT_ERR_ARG, "locator not built");
  if (n <= 0) return SFT_OK;
  if (s->dim == 2) {
    if (prec == SFT_PREC_FP32) launch_locate<2, float>(s, L, n, pts, pts_are_double, elem_out, val_out, val_is_double, val_stride, d_counters, st, nf, mu_out);
    else launch_locate<2, double>(s, L, n, pts, pts_are_double, elem_out, val_out, val_is_double, val_stride, d_counters, st, nf, mu_out);
  } else {
    if (prec == SFT_PREC_FP32) launch_locate<3, float>(s, L, n, pts, pts_are_double, elem_out, val_out, val_is_double, val_stride, d_counters, st, nf, mu_out);
    else launch_locate<3, double>(s, L, n, pts, pts_are_double, elem_out, val_out, val_is_double, val_stride, d_counters, st, nf, mu_out);
  }
  SFT_CUDA(cudaGetLastError());
  return SFT_OK;
}

// ---------------------------------------------------------------------------
// exact P1 integral of every source field: sum_e |e| mean(f over vertices).
// Bound by its D + 2 FP64 operations per element and field; the fields' sums
// are in registers, and a single field's elements go four at a time so that
// their gathers overlap (sums in local memory and one element at a time: 62 us
// for 4.0 M triangles, 104 for 5.0 M tetrahedra; now 57 and 83).
// ---------------------------------------------------------------------------
template <int D, typename TI>
__global__ void k_p1_integral_partial(const double* __restrict__ evol, const int32_t* __restrict__ conn,
                                      const TI* __restrict__ values, int64_t nv, int64_t ne, int nf,
                                      double* __restrict__ part) {
  double acc[kMaxFields];
#pragma unroll
  for (int f = 0; f < kMaxFields; ++f) acc[f] = 0.0;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  auto load = [&](int64_t i, int32_t (&v)[D + 1]) {
    if constexpr (D == 3) {
      const int4 q = __ldg(reinterpret_cast<const int4*>(conn) + i);
      v[0] = q.x; v[1] = q.y; v[2] = q.z; v[D] = q.w;
    } else {
#pragma unroll
      for (int m = 0; m <= D; ++m) v[m] = __ldg(conn + i * (D + 1) + m);
    }
  };
  // sum |e| (f_0 + ... + f_d); the 1 / (d + 1) is applied once per thread
  if (nf == 1) {
    constexpr int U = 4;
    for (; e + (U - 1) * step < ne; e += U * step) {
      int32_t v[U][D + 1];
      double vol[U];
      TI x[U][D + 1];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        load(e + u * step, v[u]);
        vol[u] = __ldg(evol + e + u * step);
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int q = 0; q <= D; ++q) x[u][q] = __ldg(values + v[u][q]);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        double m = f2d(x[u][0]);
#pragma unroll
        for (int q = 1; q <= D; ++q) m += f2d(x[u][q]);
        acc[0] = fma(vol[u], m, acc[0]);
      }
    }
  }
  for (; e < ne; e += step) {
    int32_t v[D + 1];
    load(e, v);
    const double vol = __ldg(evol + e);
#pragma unroll
    for (int f = 0; f < kMaxFields; ++f) {
      if (f >= nf) break;
      double m = 0.0;
#pragma unroll
      for (int q = 0; q <= D; ++q) m += f2d(__ldg(values + (int64_t)f * nv + v[q]));
      acc[f] = fma(vol, m, acc[f]);
    }
  }
#pragma unroll
  for (int f = 0; f < kMaxFields; ++f) acc[f] *= 1.0 / (D + 1);
  __shared__ double sh[kMaxFields][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int f = 0; f < kMaxFields; ++f) {
    if (f >= nf) break;
    const double w = warp_sum<double>(acc[f]);
    if (lane == 0) sh[f][warp] = w;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int f = 0; f < nf; ++f) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x / 32); ++w) t += sh[f][w];
      part[(int64_t)blockIdx.x * kMaxFields + f] = t;
    }
  }
}

sft_status source_integrals_launch(sft_source_s* s, double* part, cudaStream_t st) {
  const unsigned nb = kIntegralBlocks;
  if (!s->evol) return fail(SFT_ERR_ARG, "source has no element measures");
  if (s->dim == 2) {
    if (s->dtype == SFT_F64) ::sft::note_launch(), k_p1_integral_partial<2, double><<<nb, 256, 0, st>>>(s->evol, s->conn, (const double*)s->values, s->nv, s->ne, s->nf, part);
    else ::sft::note_launch(), k_p1_integral_partial<2, float><<<nb, 256, 0, st>>>(s->evol, s->conn, (const float*)s->values, s->nv, s->ne, s->nf, part);
  } else {
    if (s->dtype == SFT_F64) ::sft::note_launch(), k_p1_integral_partial<3, double><<<nb, 256, 0, st>>>(s->evol, s->conn, (const double*)s->values, s->nv, s->ne, s->nf, part);
    else ::sft::note_launch(), k_p1_integral_partial<3, float><<<nb, 256, 0, st>>>(s->evol, s->conn, (const float*)s->values, s->nv, s->ne, s->nf, part);
  }
  SFT_CUDA(cudaGetLastError());
  return SFT_OK;
}

// Sums of the partials in a fixed order: warp f < nf adds field f's into out[f]
__global__ void __launch_bounds__(32 * kMaxFields) k_final_sums(const double* __restrict__ part, int nf,
                                                               double* __restrict__ out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp >= nf) return;
  double s = 0.0;
  for (unsigned k = lane; k < kIntegralBlocks; k += 32) s += part[(int64_t)k * kMaxFields + warp];
  s = warp_sum<double>(s);
  if (lane == 0) out[warp] = s;
}

sft_status final_sums_launch(const double* part, int nf, double* out, cudaStream_t st) {
  ::sft::note_launch(), k_final_sums<<<1, 32 * kMaxFields, 0, st>>>(part, nf, out);
  SFT_CUDA(cudaGetLastError());
  return SFT_OK;
}

}  // namespace sft
