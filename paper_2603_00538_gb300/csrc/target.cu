// Target side: element measures |T| and the FP64 P1 mass matrix
// M_ki = int psi_k psi_i (Eq. mass_matrix). P1 x P1 is degree 2, so exact
// quadrature gives the closed form |T| (1 + delta_ij) / ((d+1)(d+2)).
//
// CSR build without a global sort: node -> element incidence lists by a
// counting sort, each list put in ascending element order by ranks; then one
// thread per row sums its incident elements in that order (deterministic
// values) into a hash table in shared memory, whose columns are ordered once
// at the end (k_mass_hash); rows too long for it, and all rows where the
// staging arrays cannot be had, into an ordered list (k_mass_rows).
#include <type_traits>
#include <vector>
#include "internal.hpp"
#include "util.cuh"

namespace sft {

constexpr int kMaxRow = 64;  // distinct neighbours (incl. self) per node

template <int D, typename TI>
__global__ void k_volumes(const TI* __restrict__ x, const int32_t* __restrict__ conn, int64_t nv, int64_t ne,
                          double* __restrict__ vol, float* __restrict__ vol32, double2* __restrict__ wfac,
                          int32_t* __restrict__ inc_count, int32_t* err) {
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
      vol[e] = 0.0;
      vol32[e] = 0.f;
      continue;
    }
    TI xv[D + 1][D];
#pragma unroll
    for (int m = 0; m <= D; ++m)
#pragma unroll
      for (int a = 0; a < D; ++a) xv[m][a] = x[(int64_t)v[m] * D + a];
    const double w = elem_measure<D, TI>(xv);
    // positive and finite, from the bits
    const int64_t wb = __double_as_longlong(w);
    if (wb <= 0 || wb >= 0x7FF0000000000000ll) set_error(err, DEV_BAD_ELEMENT);
    vol[e] = w;
    vol32[e] = __double2float_rn(w);
    // mass-matrix factor |T|/((d+1)(d+2)) and lumped share |T|/(d+1), by
    // the rounded reciprocals (a division costs ~10 operations on this GPU's
    // narrow FP64 pipe; the factors are within one ulp of the quotients)
    constexpr double kMassF = 1.0 / ((D + 1) * (D + 2)), kLumpF = 1.0 / (D + 1);
    wfac[e] = make_double2(w * kMassF, w * kLumpF);
#pragma unroll
    for (int m = 0; m <= D; ++m) atomicAdd(inc_count + v[m], 1);
  }
}

// node -> element incidence, filled in arbitrary order (atomic cursor) with
// the node of every entry, then put in ascending element order by rank
template <int D>
__global__ void k_inc_fill(const int32_t* __restrict__ conn, int64_t ne, int64_t nv,
                           const int32_t* __restrict__ inc_start,
                           int32_t* __restrict__ cursor, int32_t* __restrict__ inc, int32_t* __restrict__ inc_node) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < ne; e += (int64_t)gridDim.x * blockDim.x) {
    // elements with an index out of range were not counted (k_volumes) and
    // are skipped here too: the error is reported after the counting pass
    bool ok = true;
#pragma unroll
    for (int m = 0; m <= D; ++m) {
      const int32_t v = conn[e * (D + 1) + m];
      ok = ok && v >= 0 && v < nv;
    }
    if (!ok) continue;
#pragma unroll
    for (int m = 0; m <= D; ++m) {
      const int32_t v = conn[e * (D + 1) + m];
      const int32_t pos = inc_start[v] + atomicAdd(cursor + v, 1);
      inc[pos] = (int32_t)e;
      inc_node[pos] = v;
    }
  }
}

// positions [0, inc_start[nv]) were filled (skipped elements leave the tail unused)
__global__ void k_inc_rank(const int32_t* __restrict__ inc_start, const int32_t* __restrict__ inc,
                           const int32_t* __restrict__ inc_node, int64_t nv, int32_t* __restrict__ out) {
  const int64_t n = inc_start[nv];
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n; p += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = inc_node[p];
    const int32_t p0 = inc_start[v], p1 = inc_start[v + 1];
    const int32_t e = inc[p];
    int32_t rank = 0;
    for (int32_t q = p0; q < p1; ++q) rank += inc[q] < e;
    out[p0 + rank] = e;
  }
}

// Row i of M, a thread per row, into the entry-major staging arrays
// tmp_col / tmp_val [kMaxRow][nv] (the second pass copies). The row is a small
// hash table of the thread's own in shared memory, [slot][thread], so that an
// entry is found in one or two reads whatever the valence; each entry sums its
// elements in ascending order, and the columns are put in order once at the
// end. A row of more than CAP entries is marked (row_len = -1) for
// k_mass_rows. (An ordered list per thread in local memory, searched and
// shifted for each of the 4 x 24 contributions of a tetrahedral row, took
// 650 us for 0.91 M rows of a 5.0 M-tetrahedron mesh and 187 us for 2.0 M
// rows of 4.0 M triangles; now 346 and 132.)
constexpr int kHashThreads = 128;
template <int CAP>
constexpr size_t mass_hash_smem() { return (size_t)CAP * kHashThreads * (sizeof(double) + sizeof(int32_t) + 1); }

// order entries [0, N) by column: place of each among them
template <int N>
__device__ __forceinline__ void rank_columns(const int32_t* key, int cnt, int (&rank)[N], int32_t (&c)[N]) {
#pragma unroll
  for (int a = 0; a < N; ++a) {
    c[a] = a < cnt ? key[a * kHashThreads] : INT32_MAX;
    rank[a] = 0;
  }
#pragma unroll
  for (int b = 1; b < N; ++b)
#pragma unroll
    for (int a = 0; a < b; ++a) {
      const bool lt = c[a] <= c[b];
      rank[b] += lt;
      rank[a] += !lt;
    }
}

template <int D, int CAP>
__global__ void __launch_bounds__(kHashThreads)
    k_mass_hash(const int32_t* __restrict__ conn, const double2* __restrict__ wfac, const int32_t* __restrict__ inc_start,
                const int32_t* __restrict__ inc, int64_t nv, int32_t* __restrict__ row_len, int32_t* __restrict__ tmp_col,
                double* __restrict__ tmp_val, double* __restrict__ tmp_lump) {
  extern __shared__ double sm_rows[];
  double* const vals = sm_rows + threadIdx.x;                                     // [CAP][thread]
  int32_t* const keys = (int32_t*)(sm_rows + CAP * kHashThreads) + threadIdx.x;   // [CAP][thread], -1 empty
  uint8_t* const slot = (uint8_t*)((int32_t*)(sm_rows + CAP * kHashThreads) + CAP * kHashThreads) + threadIdx.x;
  constexpr int kBits = CAP == 16 ? 4 : 5;
  const int64_t i = (int64_t)blockIdx.x * kHashThreads + threadIdx.x;
  if (i >= nv) return;
#pragma unroll
  for (int q = 0; q < CAP; ++q) keys[q * kHashThreads] = -1;
  int cnt = 0;
  bool overflow = false;
  double lump = 0.0, diag = 0.0;
  // incident elements in chunks of kPre, their loads in flight together
  constexpr int kPre = 4;
  const int32_t p_end = inc_start[i + 1];
  for (int32_t p0 = inc_start[i]; p0 < p_end && !overflow; p0 += kPre) {
    int32_t ce[kPre][D + 1];
    double2 wv[kPre];
#pragma unroll
    for (int u = 0; u < kPre; ++u) {
      if (p0 + u < p_end) {
        const int32_t e = __ldg(inc + p0 + u);
        wv[u] = __ldg(wfac + e);
        if constexpr (D == 3) {
          const int4 q = __ldg(reinterpret_cast<const int4*>(conn) + e);
          ce[u][0] = q.x; ce[u][1] = q.y; ce[u][2] = q.z; ce[u][D] = q.w;
        } else {
#pragma unroll
          for (int m = 0; m <= D; ++m) ce[u][m] = __ldg(conn + (int64_t)e * (D + 1) + m);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kPre; ++u) {
      if (p0 + u >= p_end) break;
      lump += wv[u].y;
      diag += 2.0 * wv[u].x;  // (an element repeats no node: it would have no volume)
#pragma unroll
      for (int m = 0; m <= D; ++m) {
        const int32_t j = ce[u][m];
        if (j == (int32_t)i) continue;
        uint32_t h = ((uint32_t)j * 2654435761u) >> (32 - kBits);
        for (int probe = 0;; ++probe) {
          const int32_t k = keys[h * kHashThreads];
          if (k == j) {
            vals[h * kHashThreads] += wv[u].x;
            break;
          }
          if (k == -1) {
            if (cnt == CAP - 1) {  // (the diagonal takes one)
              overflow = true;
              break;
            }
            keys[h * kHashThreads] = j;
            vals[h * kHashThreads] = wv[u].x;
            ++cnt;
            break;
          }
          h = (h + 1u) & (CAP - 1);
        }
      }
    }
  }
  if (overflow) {
    row_len[i] = -1;
    return;
  }
  // the table's entries to its front (a slot moves down or stays), the diagonal with them
  int n = 0;
#pragma unroll 4
  for (int q = 0; q < CAP; ++q) {
    const int32_t k = keys[q * kHashThreads];
    if (k < 0) continue;
    keys[n * kHashThreads] = k;
    slot[n * kHashThreads] = (uint8_t)q;
    ++n;
  }
  if (p_end > inc_start[i]) {
    // a slot no entry holds takes the diagonal's value
    int q = CAP - 1;
    for (int a = n - 1; a >= 0 && slot[a * kHashThreads] == q; --a) --q;
    vals[q * kHashThreads] = diag;
    keys[n * kHashThreads] = (int32_t)i;
    slot[n * kHashThreads] = (uint8_t)q;
    ++n;
  }
  // in ascending column order
  auto order = [&](auto& rank, auto& c, auto len) {
    constexpr int N = decltype(len)::value;
    rank_columns<N>(keys, n, rank, c);
    int s[N];
#pragma unroll
    for (int a = 0; a < N; ++a) s[a] = a < n ? slot[a * kHashThreads] : 0;
#pragma unroll
    for (int a = 0; a < N; ++a)
      if (a < n) {
        keys[rank[a] * kHashThreads] = c[a];
        slot[rank[a] * kHashThreads] = (uint8_t)s[a];
      }
  };
  if (n <= CAP / 2) {
    int rank[CAP / 2];
    int32_t c[CAP / 2];
    order(rank, c, std::integral_constant<int, CAP / 2>());
  } else {
    int rank[CAP];
    int32_t c[CAP];
    order(rank, c, std::integral_constant<int, CAP>());
  }
  for (int q = 0; q < n; ++q) {
    tmp_col[(int64_t)q * nv + i] = keys[q * kHashThreads];
    tmp_val[(int64_t)q * nv + i] = vals[slot[q * kHashThreads] * kHashThreads];
  }
  row_len[i] = n;
  tmp_lump[i] = lump;
}

// Row i of M from an ordered list in local memory: FILL=false writes the row
// length (and, when tmp_col is given, the row itself into the staging arrays),
// FILL=true writes columns, values, the Jacobi inverse diagonal and the lumped
// mass. With REDO only the rows marked -1.
template <int D, bool FILL, bool REDO = false>
__global__ void k_mass_rows(const int32_t* __restrict__ conn, const double2* __restrict__ wfac,
                            const int32_t* __restrict__ inc_start, const int32_t* __restrict__ inc, int64_t nv,
                            int32_t* __restrict__ row_len, const int32_t* __restrict__ row_ptr,
                            int32_t* __restrict__ col, double* __restrict__ val, double* __restrict__ dinv,
                            double* __restrict__ lumped, int32_t* err, int32_t* __restrict__ tmp_col,
                            double* __restrict__ tmp_val, double* __restrict__ tmp_lump) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nv; i += (int64_t)gridDim.x * blockDim.x) {
    if (REDO && row_len[i] >= 0) continue;
    constexpr int CAP = kMaxRow;
    int32_t cols[CAP];
    double vals[CAP];
    int cnt = 0;
    bool overflow = false;
    double lump = 0.0;
    // incident elements in chunks of kPre: their connectivity and factors are
    // loaded first (independent loads in flight together), then merged in
    // incidence order (the same sums as one element at a time)
    constexpr int kPre = 4;
    const int32_t p_end = inc_start[i + 1];
    for (int32_t p0 = inc_start[i]; p0 < p_end; p0 += kPre) {
      int32_t ce[kPre][D + 1];
      double2 wv[kPre];
#pragma unroll
      for (int u = 0; u < kPre; ++u) {
        if (p0 + u < p_end) {
          const int32_t e = __ldg(inc + p0 + u);
          wv[u] = __ldg(wfac + e);
#pragma unroll
          for (int m = 0; m <= D; ++m) ce[u][m] = __ldg(conn + (int64_t)e * (D + 1) + m);
        }
      }
#pragma unroll
      for (int u = 0; u < kPre; ++u) {
      if (p0 + u >= p_end) break;
      const double2 wf = wv[u];
      lump += wf.y;
      // 2 RN(w/den) == RN(2w/den): same values as dividing each entry
      const double wd = wf.x;
#pragma unroll
      for (int m = 0; m <= D; ++m) {
        const int32_t j = ce[u][m];
        const double c = j == i ? 2.0 * wd : wd;
        int q = 0;
        while (q < cnt && cols[q] < j) ++q;
        if (q < cnt && cols[q] == j) {
          vals[q] += c;
        } else if (cnt < CAP) {
          for (int r = cnt; r > q; --r) { cols[r] = cols[r - 1]; vals[r] = vals[r - 1]; }
          cols[q] = j;
          vals[q] = c;
          ++cnt;
        } else {
          overflow = true;
        }
      }
      }
    }
    if (overflow) set_error(err, DEV_VALENCE);
    if (!FILL) {
      row_len[i] = cnt;
      if (tmp_col) {
        for (int q = 0; q < cnt; ++q) {
          // entry q of every row contiguous ([q][nv]): coalesced across a warp's rows
          tmp_col[(int64_t)q * nv + i] = cols[q];
          tmp_val[(int64_t)q * nv + i] = vals[q];
        }
        tmp_lump[i] = lump;
      }
    } else {
      const int32_t base = row_ptr[i];
      double diag = 0.0;
      for (int q = 0; q < cnt; ++q) {
        col[base + q] = cols[q];
        val[base + q] = vals[q];
        if (cols[q] == i) diag = vals[q];
      }
      dinv[i] = diag > 0.0 ? 1.0 / diag : 0.0;
      lumped[i] = lump;
    }
  }
}

// second pass from the staged rows: a block's rows are consecutive in the CSR
// arrays, so they are put together in shared memory and written as one run
// (writing each row by its thread took 118 us for 0.51 M rows in 3D and 75 us
// for 1.0 M in 2D, now 43 and 56; more than kCopyEntries go directly)
constexpr int kCopyThreads = 128, kCopyEntries = 20 * kCopyThreads;

__global__ void __launch_bounds__(kCopyThreads)
    k_mass_copy(const int32_t* __restrict__ tmp_col, const double* __restrict__ tmp_val, const double* __restrict__ tmp_lump,
                const int32_t* __restrict__ row_ptr, int64_t nv, int32_t* __restrict__ col, double* __restrict__ val,
                double* __restrict__ dinv, double* __restrict__ lumped) {
  __shared__ double sval[kCopyEntries];
  __shared__ int32_t scol[kCopyEntries];
  const int64_t r0 = (int64_t)blockIdx.x * kCopyThreads, i = r0 + threadIdx.x;
  const int64_t r1 = r0 + kCopyThreads < nv ? r0 + kCopyThreads : nv;
  const int32_t base0 = __ldg(row_ptr + r0), total = __ldg(row_ptr + r1) - base0;
  const bool staged = total <= kCopyEntries;
  int32_t* const oc = staged ? scol : col + base0;
  double* const ov = staged ? sval : val + base0;
  if (i < nv) {
    const int32_t base = __ldg(row_ptr + i) - base0, cnt = __ldg(row_ptr + i + 1) - base0 - base;
    double diag = 0.0;
#pragma unroll 4
    for (int q = 0; q < cnt; ++q) {
      const int32_t c = __ldg(tmp_col + (int64_t)q * nv + i);
      const double v = __ldg(tmp_val + (int64_t)q * nv + i);
      oc[base + q] = c;
      ov[base + q] = v;
      if (c == i) diag = v;
    }
    dinv[i] = diag > 0.0 ? 1.0 / diag : 0.0;
    lumped[i] = tmp_lump[i];
  }
  if (!staged) return;
  __syncthreads();
  for (int k = threadIdx.x; k < total; k += kCopyThreads) {
    col[base0 + k] = scol[k];
    val[base0 + k] = sval[k];
  }
}

static unsigned blocks_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  if (b < 1) b = 1;
  if (b > 152 * 64) b = 152 * 64;
  return (unsigned)b;
}

template <int D>
static sft_status build_target_t(sft_target_s* t, cudaStream_t st, int32_t* d_err) {
  SFT_CUDA(dalloc(&t->vol, (size_t)t->ne, st));
  SFT_CUDA(dalloc(&t->vol32, (size_t)t->ne, st));
  double2* wfac = nullptr;
  SFT_CUDA(dalloc(&wfac, (size_t)t->ne, st));
  int32_t *inc_count = nullptr, *inc_start = nullptr, *inc = nullptr, *row_len = nullptr;
  int64_t* off64 = nullptr;
  SFT_CUDA(dalloc(&inc_count, (size_t)t->nv, st));
  SFT_CUDA(cudaMemsetAsync(inc_count, 0, sizeof(int32_t) * t->nv, st));
  if (t->dtype == SFT_F64)
    ::sft::note_launch(), k_volumes<D, double><<<blocks_for(t->ne), 256, 0, st>>>((const double*)t->coords, t->conn, t->nv, t->ne, t->vol, t->vol32, wfac, inc_count, d_err);
  else
    ::sft::note_launch(), k_volumes<D, float><<<blocks_for(t->ne), 256, 0, st>>>((const float*)t->coords, t->conn, t->nv, t->ne, t->vol, t->vol32, wfac, inc_count, d_err);
  SFT_CUDA(cudaGetLastError());
  // no host check here: every later kernel only follows connectivity of
  // elements whose indices are all in range, and the error flag is read with
  // the row count below
  SFT_CUDA(dalloc(&off64, (size_t)t->nv + 1, st));
  SFT_CUDA(dalloc(&inc_start, (size_t)t->nv + 1, st));
  SFT_CUDA(dalloc(&inc, (size_t)t->ne * (D + 1), st));
  int32_t *inc_raw = nullptr, *inc_node = nullptr;
  SFT_CUDA(dalloc(&inc_raw, (size_t)t->ne * (D + 1), st));
  SFT_CUDA(dalloc(&inc_node, (size_t)t->ne * (D + 1), st));
  SFT_CUDA(exclusive_scan_i32_to_i64(inc_count, off64, t->nv, st));
  SFT_CUDA(narrow_i64_to_i32(off64, inc_start, t->nv + 1, st));
  SFT_CUDA(cudaMemsetAsync(inc_count, 0, sizeof(int32_t) * t->nv, st));
  ::sft::note_launch(), k_inc_fill<D><<<blocks_for(t->ne), 256, 0, st>>>(t->conn, t->ne, t->nv, inc_start, inc_count,
                                                                       inc_raw, inc_node);
  SFT_CUDA(cudaGetLastError());
  ::sft::note_launch(), k_inc_rank<<<blocks_for(t->ne * (D + 1)), 256, 0, st>>>(inc_start, inc_raw, inc_node, t->nv,
                                                                               inc);
  SFT_CUDA(cudaGetLastError());
  dfree(inc_raw, st);
  dfree(inc_node, st);
  row_len = inc_count;  // reuse
  // rows are staged at a fixed stride when that fits comfortably (the
  // second pass then copies instead of merging the incidence lists again)
  DevBuf<int32_t> stage_col(st);
  DevBuf<double> stage_val(st), stage_lump(st);
  int32_t* tmp_col = nullptr;
  double *tmp_val = nullptr, *tmp_lump = nullptr;
  if (t->nv * kMaxRow <= (int64_t)1 << 31) {
    if (stage_col.alloc((size_t)t->nv * kMaxRow) == cudaSuccess &&
        stage_val.alloc((size_t)t->nv * kMaxRow) == cudaSuccess && stage_lump.alloc((size_t)t->nv) == cudaSuccess) {
      tmp_col = stage_col.p;
      tmp_val = stage_val.p;
      tmp_lump = stage_lump.p;
    } else {
      cudaGetLastError();  // no staging: the second pass merges again
    }
  }
  if (tmp_col) {
    // rows of up to 16 (2D) / 32 (3D) entries in the hash tables, the rest in lists
    constexpr int kCapHash = D == 2 ? 16 : 32;
    constexpr size_t smem = mass_hash_smem<kCapHash>();
    SFT_CUDA(cudaFuncSetAttribute(k_mass_hash<D, kCapHash>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    ::sft::note_launch(), k_mass_hash<D, kCapHash><<<(unsigned)((t->nv + kHashThreads - 1) / kHashThreads), kHashThreads, smem, st>>>(
        t->conn, wfac, inc_start, inc, t->nv, row_len, tmp_col, tmp_val, tmp_lump);
    SFT_CUDA(cudaGetLastError());
    ::sft::note_launch(), k_mass_rows<D, false, true><<<blocks_for(t->nv), 256, 0, st>>>(
        t->conn, wfac, inc_start, inc, t->nv, row_len, nullptr, nullptr, nullptr, nullptr, nullptr, d_err, tmp_col, tmp_val,
        tmp_lump);
  } else {
    ::sft::note_launch(), k_mass_rows<D, false><<<blocks_for(t->nv), 256, 0, st>>>(
        t->conn, wfac, inc_start, inc, t->nv, row_len, nullptr, nullptr, nullptr, nullptr, nullptr, d_err, nullptr, nullptr,
        nullptr);
  }
  SFT_CUDA(cudaGetLastError());
  SFT_CUDA(exclusive_scan_i32_to_i64(row_len, off64, t->nv, st));
  Events kit;
  SFT_CUDA(cudaMemcpyAsync(&kit.host().counters[0], off64 + t->nv, sizeof(int64_t), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaMemcpyAsync(&kit.host().err, d_err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  SFT_CUDA(cudaStreamSynchronize(st));
  const int64_t nnz = kit.host().counters[0];
  const int32_t herr = kit.host().err;
  if (herr || nnz >= (int64_t)INT32_MAX) {
    dfree(off64, st);
    dfree(inc_start, st);
    dfree(inc, st);
    dfree(inc_count, st);
    dfree(wfac, st);
    if (herr == DEV_NONFINITE) return fail(SFT_ERR_MESH, "non-finite target coordinate");
    if (herr == DEV_BAD_INDEX) return fail(SFT_ERR_MESH, "target connectivity index out of range");
    if (herr == DEV_BAD_ELEMENT) return fail(SFT_ERR_MESH, "target mesh has a non-positive element");
    if (herr) return fail(SFT_ERR_MESH, "target node belongs to more elements than supported");
    return fail(SFT_ERR_UNSUPPORTED, "mass matrix nnz exceeds 2^31");
  }
  t->nnz = nnz;
  SFT_CUDA(dalloc(&t->row_ptr, (size_t)t->nv + 1, st));
  SFT_CUDA(narrow_i64_to_i32(off64, t->row_ptr, t->nv + 1, st));
  SFT_CUDA(dalloc(&t->col, (size_t)nnz, st));
  SFT_CUDA(dalloc(&t->val, (size_t)nnz, st));
  SFT_CUDA(dalloc(&t->dinv, (size_t)t->nv, st));
  SFT_CUDA(dalloc(&t->lumped, (size_t)t->nv, st));
  if (tmp_col) {
    ::sft::note_launch(), k_mass_copy<<<(unsigned)((t->nv + kCopyThreads - 1) / kCopyThreads), kCopyThreads, 0, st>>>(
        tmp_col, tmp_val, tmp_lump, t->row_ptr, t->nv, t->col, t->val, t->dinv, t->lumped);
  } else {
    ::sft::note_launch(), k_mass_rows<D, true><<<blocks_for(t->nv), 256, 0, st>>>(t->conn, wfac, inc_start, inc, t->nv, nullptr, t->row_ptr,
                                                            t->col, t->val, t->dinv, t->lumped, d_err, nullptr,
                                                            nullptr, nullptr);
  }
  SFT_CUDA(cudaGetLastError());
  dfree(off64, st);
  dfree(inc_start, st);
  dfree(inc, st);
  dfree(inc_count, st);
  dfree(wfac, st);
  return SFT_OK;
}

sft_status build_target(sft_target_s* t, cudaStream_t st, int32_t* d_err) {
  return t->dim == 2 ? build_target_t<2>(t, st, d_err) : build_target_t<3>(t, st, d_err);
}

sft_status target_coordsP(sft_target_s* t, int prec, cudaStream_t st) {
  if (t->coordsP[prec]) return SFT_OK;
  const size_t esz = prec == SFT_PREC_FP32 ? 4 : 8;
  void* p = nullptr;
  SFT_CUDA(pool_alloc(&p, esz * (size_t)(t->nv * t->dim > 0 ? t->nv * t->dim : 1), st));
  t->coordsP[prec] = p;
  return convert_coords(t->coords, t->dtype, p, prec, t->nv * t->dim, st);
}

}  // namespace sft
