// LU with partial pivoting of the assembled dense trace matrix (FP64, row-major) and its triangular solves.
//
// Blocks of 32 columns in four panels of 8. A cluster of eight CTAs factors a panel, an eighth of its rows in each one's
// shared memory, with one cluster barrier per column; the rest of the 32 columns follow at once, everything else once
// per block: row interchanges and the triangle (one thread per column), then the trailing update by 64 x 64 tiles. A
// tile whose left or right factor is zero is left alone: the matrix is the assembly of a sparse trace system, and most
// tiles stay zero for a while.
// The FP64 pipe (two FMA per clock and SM) bounds every part: one CTA alone takes 91 us for a panel of 2,304 rows
// and 2.8 ms for the solves, which is why both are spread over a cluster (25 us, 2.1 ms).
// 2,304 unknowns (8 x 8 x 2 triangles, p = 2): an implicit Euler step with three factorisations takes 34 ms; with three
// launches per column, a rank-1 update of the whole remainder each and solves one row per barrier, 124 ms.
#pragma once
#include <climits>
#include <cstdint>

#include "ptx_async.cuh"

namespace hdg {

constexpr int kLuNB = 8, kLuBlock = 32, kLuTile = 64;
constexpr int kLuCluster = 8;
constexpr int kLuMaxN = 16384;  // x of the solves in shared memory

// leading dimension of a CTA's rows of a panel of m rows (odd: neighbouring columns in different banks); the first CTA
// holds at least the panel's own rows
inline __host__ __device__ int lu_panel_rows(int m) {
  const int r = (m + kLuCluster - 1) / kLuCluster;
  return r < kLuNB ? kLuNB : r;
}
inline size_t lu_panel_smem(int m) { return sizeof(double) * kLuNB * (lu_panel_rows(m) | 1); }

HDG_DEVI unsigned lu_cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// all threads of the cluster; orders shared-memory stores before it against reads after it
HDG_DEVI void lu_cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
HDG_DEVI void lu_put(double* p, unsigned rank, double v) {  // *p = v in the shared memory of CTA `rank`
  asm volatile("{\n .reg .b32 ra;\n mapa.shared::cluster.u32 ra, %0, %1;\n st.shared::cluster.f64 [ra], %2;\n}" ::"r"(
                   smem_u32(p)),
               "r"(rank), "d"(v)
               : "memory");
}

// |v| as an ordered integer, 1 for zero, 0 for NaN (never a pivot)
HDG_DEVI unsigned long long lu_key(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
  return b > 0x7ff0000000000000ull ? 0ull : b + 1;
}
// the largest key of a warp and the lowest index that has it
HDG_DEVI void lu_warp_max(unsigned long long& key, int& idx) {
  const unsigned hi = (unsigned)(key >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned lo = hi == mh ? (unsigned)key : 0u, ml = __reduce_max_sync(0xffffffffu, lo);
  idx = (int)__reduce_min_sync(0xffffffffu, (unsigned)(hi == mh && lo == ml ? idx : INT_MAX));
  key = (unsigned long long)mh << 32 | ml;
}

// Columns [k0, k0 + w) of the block [b0, b1). piv[k]: the row interchanged with row k.
__global__ void __cluster_dims__(kLuCluster, 1, 1) __launch_bounds__(256)
    k_lu_panel(double* K, int64_t n, int64_t k0, int w, int64_t b0, int64_t b1, int* piv, int* bad) {
  extern __shared__ double lu_sm[];
  double* A = lu_sm;  // this CTA's rows, [column][row]
  // per column, in turn: each CTA's candidate (row, reciprocal of the pivot, key and index), and row j
  __shared__ double s_row[2][kLuCluster][kLuNB], s_inv[2][kLuCluster], s_cand[2][kLuCluster], s_top[2][kLuNB];
  __shared__ int s_piv[kLuNB];
  __shared__ unsigned long long wk[8];
  __shared__ int wi[8];
  const int m = (int)(n - k0), tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)lu_cluster_rank(), rpc = lu_panel_rows(m), ld = rpc | 1, lo = rank * rpc;
  const int nr = m - lo < 0 ? 0 : (m - lo < rpc ? m - lo : rpc);
  double* Kp = K + (k0 + lo) * n + k0;
#pragma unroll 4
  for (int t = tid; t < nr * kLuNB; t += 256)
    if (t % kLuNB < w) A[t % kLuNB * ld + t / kLuNB] = Kp[(int64_t)(t / kLuNB) * n + t % kLuNB];
  __syncthreads();
  unsigned long long key = 0;
  int idx = INT_MAX;
  for (int r = tid; r < nr; r += 256) {
    const unsigned long long k = lu_key(A[r]);
    if (k > key) {
      key = k;
      idx = lo + r;
    }
  }
  lu_cluster_sync();  // every CTA of the cluster runs before its shared memory is written
  for (int j = 0; j < w; ++j) {
    const int b = j & 1;
    lu_warp_max(key, idx);
    if (lane == 0) {
      wk[warp] = key;
      wi[warp] = idx;
    }
    __syncthreads();
    if (warp == 0) {  // this CTA's candidate to all CTAs: four lanes per destination
      key = lane < 8 ? wk[lane] : 0;
      idx = lane < 8 ? wi[lane] : INT_MAX;
      lu_warp_max(key, idx);
      const bool any = key != 0;
      const double inv = key > 1 ? 1.0 / A[j * ld + idx - lo] : 0.0;
      const unsigned dst = lane >> 2;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int c = 2 * (lane & 3) + i;
        lu_put(&s_row[b][rank][c], dst, any && c < w ? A[c * ld + idx - lo] : 0.0);
        if (rank == 0) lu_put(&s_top[b][c], dst, c < w ? A[c * ld + j] : 0.0);
      }
      if ((lane & 3) == 0) {
        lu_put(&s_inv[b][rank], dst, inv);
        lu_put(&s_cand[b][rank], dst, any ? (double)idx : -1.0);
      }
    }
    lu_cluster_sync();
    int q = 0;  // the largest candidate, the lowest row on ties
    unsigned long long kq = 0;
#pragma unroll
    for (int t = 0; t < kLuCluster; ++t) {
      const unsigned long long kt = s_cand[b][t] >= 0.0 ? lu_key(s_row[b][t][j]) : 0ull;
      if (kt > kq) {
        kq = kt;
        q = t;
      }
    }
    const int p = kq ? (int)s_cand[b][q] : j;  // no comparable entry (NaN): no interchange
    const double* prow = kq ? s_row[b][q] : s_top[b];
    const double inv = kq ? s_inv[b][q] : 1.0 / s_top[b][j];
    if (rank == 0 && tid == 0) {
      s_piv[j] = p;
      piv[k0 + j] = (int)(k0 + p);
      if (kq <= 1) *bad = 1;
    }
    double top[kLuNB];
#pragma unroll
    for (int c = 0; c < kLuNB; ++c) top[c] = prow[c];
    key = 0;
    idx = INT_MAX;
    for (int r = tid; r < nr; r += 256) {
      const int gr = lo + r;
      if (gr == j) {
#pragma unroll
        for (int c = 0; c < kLuNB; ++c)
          if (c < w) A[c * ld + r] = top[c];
      }
      if (gr <= j) continue;
      const bool sw = gr == p;  // takes row j
      const double l = (sw ? s_top[b][j] : A[j * ld + r]) * inv;
      A[j * ld + r] = l;
#pragma unroll
      for (int c = 0; c < kLuNB; ++c) {
        if (c < j && sw) A[c * ld + r] = s_top[b][c];
        if (c > j && c < w) {
          const double v = (sw ? s_top[b][c] : A[c * ld + r]) - l * top[c];
          A[c * ld + r] = v;
          if (c == j + 1) {  // the search for the next column
            const unsigned long long k = lu_key(v);
            if (k > key) {
              key = k;
              idx = gr;
            }
          }
        }
      }
    }
  }
  __syncthreads();
#pragma unroll 4
  for (int t = tid; t < nr * kLuNB; t += 256)
    if (t % kLuNB < w) Kp[(int64_t)(t / kLuNB) * n + t % kLuNB] = A[t % kLuNB * ld + t / kLuNB];
  // the block's other columns: the interchanges, and behind the panel its unit lower triangle
  const int64_t c = b0 + tid;
  if (rank != 0 || c >= b1 || (c >= k0 && c < k0 + w)) return;
  double u[kLuNB], o[kLuNB];  // rows k0 + j, and the rows interchanged with them (under the first j that names one)
#pragma unroll
  for (int j = 0; j < kLuNB; ++j) {
    u[j] = j < w ? K[(k0 + j) * n + c] : 0.0;
    o[j] = j < w ? K[(k0 + s_piv[j]) * n + c] : 0.0;
  }
#pragma unroll
  for (int j = 0; j < kLuNB; ++j) {
    if (j >= w) break;
    const int p = s_piv[j];
    bool found = false;
    const double t = u[j];
#pragma unroll
    for (int i = j + 1; i < kLuNB; ++i)
      if (p == i && i < w) {
        u[j] = u[i];
        u[i] = t;
      }
#pragma unroll
    for (int i = 0; i <= j; ++i)
      if (p >= w && !found && s_piv[i] == p) {
        u[j] = o[i];
        o[i] = t;
        found = true;
      }
  }
#pragma unroll
  for (int j = 0; j < kLuNB; ++j) {
    if (j >= w) break;
    const int p = s_piv[j];
    bool first = p >= w;
#pragma unroll
    for (int i = 0; i < j; ++i) first = first && s_piv[i] != p;
    if (first) K[(k0 + p) * n + c] = o[j];
  }
  if (c >= k0)
#pragma unroll
    for (int t = 0; t < kLuNB; ++t)
#pragma unroll
      for (int j = t + 1; j < kLuNB; ++j)
        if (j < w) u[j] -= A[t * ld + j] * u[t];
#pragma unroll
  for (int j = 0; j < kLuNB; ++j)
    if (j < w) K[(k0 + j) * n + c] = u[j];
}

// rows below the w columns at k0, columns [k0 + w, b1): -= L U
__global__ void __launch_bounds__(256) k_lu_inner(double* K, int64_t n, int64_t k0, int w, int64_t b1) {
  const int nc = (int)(b1 - k0 - w);
  const int64_t tot = (n - k0 - w) * nc;
  for (int64_t t = blockIdx.x * (int64_t)256 + threadIdx.x; t < tot; t += (int64_t)gridDim.x * 256) {
    const int64_t r = k0 + w + t / nc, c = k0 + w + t % nc;
    double s = K[r * n + c];
    for (int j = 0; j < w; ++j) s -= K[r * n + k0 + j] * K[(k0 + j) * n + c];
    K[r * n + c] = s;
  }
}

inline unsigned lu_inner_grid(int64_t rows, int64_t cols) {
  const int64_t blocks = (rows * cols + 255) / 256;
  return (unsigned)(blocks < 152 * 8 ? blocks : 152 * 8);
}

// Columns outside the block [b0, b1), 32 per CTA, four lanes each: the block's interchanges, and behind it the 32 x 32
// unit lower triangle. The first warp follows the interchanges on row numbers, so that all of a column's entries are
// loaded together. A lane holds every fourth row of its column: a warp's FP64 instruction takes 64 clocks on its own
// quarter of the SM, so the triangle is spread over all four quarters (15 us per launch; one lane per column 30).
// flag[c / 32]: whether any of these columns' U entries is nonzero.
// Columns 32 (first + blockIdx.x) .., not those of group `skip`.
__global__ void __launch_bounds__(128) k_lu_swap(double* K, int64_t n, int64_t b0, int64_t b1, const int* piv, int* flag,
                                                 int first, int skip) {
  const int group = first + (int)blockIdx.x;
  if (group == skip) return;
  constexpr int NR = kLuBlock / 4;
  __shared__ double L[kLuBlock][kLuBlock + 1];
  __shared__ int src[kLuBlock], orow[kLuBlock], osrc[kLuBlock], s_no;
  const int w = (int)(b1 - b0), tid = threadIdx.x, lane = tid & 31;
  if (tid < 32) {
    const int p = tid < w ? piv[b0 + tid] : (int)b0 + tid;
    const int owner = __ffs(__match_any_sync(0xffffffffu, p)) - 1;  // the first interchange with this row
    int in = (int)b0 + tid, out = p;                                // what rows b0 + tid and p hold
    for (int j = 0; j < w; ++j) {
      const int pj = __shfl_sync(0xffffffffu, p, j), x = __shfl_sync(0xffffffffu, in, j);
      if (pj < (int)b1) {
        const int i = pj - (int)b0, y = __shfl_sync(0xffffffffu, in, i);
        if (tid == j) in = y;
        if (tid == i) in = x;
      } else {
        const int o = __shfl_sync(0xffffffffu, owner, j), y = __shfl_sync(0xffffffffu, out, o);
        if (tid == j) in = y;
        if (tid == o) out = x;
      }
    }
    src[tid] = in;
    const bool put = tid < w && p >= (int)b1 && owner == tid;
    const unsigned mask = __ballot_sync(0xffffffffu, put);
    if (put) {
      const int q = __popc(mask & ((1u << tid) - 1u));
      orow[q] = p;
      osrc[q] = out;
    }
    if (tid == 0) s_no = __popc(mask);
  } else if ((group + 1) * (int64_t)32 > b1) {
    for (int t = tid - 32; t < kLuBlock * kLuBlock; t += 96) {
      const int r = t / kLuBlock, c = t % kLuBlock;
      L[r][c] = r < w && c < r ? K[(b0 + r) * n + b0 + c] : 0.0;
    }
  }
  __syncthreads();
  const int col = lane & 7, rg = lane >> 3;  // rows b0 + 4 i + rg
  const int64_t c = group * (int64_t)32 + (tid >> 5) * 8 + col;
  const bool live = c < n && (c < b0 || c >= b1);
  const int no = s_no;
  double u[NR], o[NR];
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const int j = 4 * i + rg;
    u[i] = live && j < w ? K[(int64_t)src[j] * n + c] : 0.0;
    o[i] = live && j < no ? K[(int64_t)osrc[j] * n + c] : 0.0;
  }
  __syncwarp();  // a column's entries are all loaded before any is stored
  bool nz = false;
#pragma unroll
  for (int i = 0; i < NR; ++i) {
    const int j = 4 * i + rg;
    if (live && j < no) K[(int64_t)orow[j] * n + c] = o[i];
    nz = nz || u[i] != 0.0;  // true for NaN
  }
  nz = nz && c >= b1;
  if (__any_sync(0xffffffffu, nz)) {  // zero columns stay zero
#pragma unroll
    for (int t = 0; t < kLuBlock; ++t) {
      const double ut = __shfl_sync(0xffffffffu, u[t / 4], (t % 4) * 8 + col);
#pragma unroll
      for (int i = t / 4; i < NR; ++i)
        if (c >= b1 && (i > t / 4 || rg > t % 4)) u[i] -= L[4 * i + rg][t] * ut;
    }
  }
#pragma unroll
  for (int i = 0; i < NR; ++i)
    if (live && 4 * i + rg < w) K[(b0 + 4 * i + rg) * n + c] = u[i];
  const int any = __syncthreads_or(nz);
  if (tid == 0) flag[group] = any;
}

// trailing update K[r][c] -= sum_j L[r][b0 + j] U[b0 + j][c], r >= b1, c >= cl (a multiple of 32), one 64 x 64 tile per CTA
__global__ void __launch_bounds__(256) k_lu_update(double* K, int64_t n, int64_t b0, int64_t b1, int64_t cl,
                                                   const int* flag) {
  const int ct = (int)(cl / kLuTile) + blockIdx.x, rt = (int)(b1 / kLuTile) + blockIdx.y;
  const bool left = 2 * ct * 32 >= cl && flag[2 * ct], right = 2 * ct + 1 < (n + 31) / 32 && flag[2 * ct + 1];
  if (!left && !right) return;
  __shared__ double A[kLuBlock][kLuTile + 2], B[kLuBlock][kLuTile + 2];  // [j][row], [j][column]
  const int w = (int)(b1 - b0), tid = threadIdx.x;
  const int64_t r0 = (int64_t)rt * kLuTile, c0 = (int64_t)ct * kLuTile;
  bool nz = false;
  for (int t = tid; t < kLuTile * kLuBlock; t += 256) {
    const int j = t % kLuBlock, r = t / kLuBlock;
    double v = 0.0;
    if (j < w && r0 + r >= b1 && r0 + r < n) v = K[(r0 + r) * n + b0 + j];
    nz = nz || v != 0.0;
    A[j][r] = v;
  }
  if (!__syncthreads_or(nz)) return;
  for (int t = tid; t < kLuTile * kLuBlock; t += 256) {
    const int c = t % kLuTile, j = t / kLuTile;
    B[j][c] = j < w && c0 + c >= cl && c0 + c < n ? K[(b0 + j) * n + c0 + c] : 0.0;
  }
  __syncthreads();
  const int ty = tid / 16, tx = tid % 16;  // rows 4 ty .., columns 2 tx, 2 tx + 1, 32 + 2 tx, 32 + 2 tx + 1
  double acc[4][4] = {};
#pragma unroll 8
  for (int j = 0; j < kLuBlock; ++j) {
    const double2 b01 = *reinterpret_cast<const double2*>(&B[j][2 * tx]), b23 = *reinterpret_cast<const double2*>(&B[j][32 + 2 * tx]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const double a = A[j][4 * ty + i];
      acc[i][0] += a * b01.x;
      acc[i][1] += a * b01.y;
      acc[i][2] += a * b23.x;
      acc[i][3] += a * b23.y;
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int64_t r = r0 + 4 * ty + i, c = c0 + (q >> 1) * 32 + 2 * tx + (q & 1);
      if (r >= b1 && c >= cl && r < n && c < n) K[r * n + c] -= acc[i][q];
    }
}

// P x, then L y = P x, U x = y by one cluster, x in every CTA's shared memory. Per 32 rows each CTA forms four rows'
// products with the part already solved (two warps per row) and sends them to all; then each solves the 32 x 32 triangle
// for itself.
__global__ void __cluster_dims__(kLuCluster, 1, 1) __launch_bounds__(256)
    k_lu_solve(const double* K, const int* piv, int64_t n, double* x) {
  extern __shared__ double lu_sm[];
  double* xs = lu_sm;  // [n]
  __shared__ double T[32][33], part[4][2], vb[2][32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)lu_cluster_rank(), row = 4 * rank + (warp >> 1), half = warp & 1;
  for (int64_t t = tid; t < n; t += 256) xs[t] = x[t];
  lu_cluster_sync();  // all have read x and run
  if (warp == 0)
    for (int64_t k0 = 0; k0 < n; k0 += 32) {
      const int pl = k0 + lane < n ? piv[k0 + lane] : 0;
      for (int i = 0; i < 32 && k0 + i < n; ++i) {
        const int p = __shfl_sync(0xffffffffu, pl, i);
        if (lane == 0 && p != (int)k0 + i) {
          const double t = xs[k0 + i];
          xs[k0 + i] = xs[p];
          xs[p] = t;
        }
      }
    }
  __syncthreads();
  const int64_t nb = (n + 31) / 32;
  for (int64_t q2 = 0; q2 < 2 * nb; ++q2) {
    const bool up = q2 >= nb;
    const int64_t i0 = 32 * (up ? 2 * nb - 1 - q2 : q2), r = i0 + row;
    const int b = (int)(q2 & 1);
    for (int t = tid; t < 32 * 32; t += 256) {
      const int64_t tr = i0 + (t >> 5), tc = i0 + (t & 31);
      T[t >> 5][t & 31] = tr < n && tc < n ? K[tr * n + tc] : 0.0;
    }
    double s = 0.0;
    if (r < n) {
      const double* Kr = K + r * n;
      const int64_t j1 = up ? n : i0;
#pragma unroll 8
      for (int64_t j = (up ? i0 + 32 : 0) + 32 * half + lane; j < j1; j += 64) s += Kr[j] * xs[j];
    }
    for (int off = 16; off > 0; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
    if (lane == 0) part[warp >> 1][half] = s;
    __syncthreads();
    if (warp == 0) {
      const int i = lane & 3;
      const int64_t ri = i0 + 4 * rank + i;
      lu_put(&vb[b][4 * rank + i], lane >> 2, ri < n ? xs[ri] - (part[i][0] + part[i][1]) : 0.0);
    }
    lu_cluster_sync();
    if (warp == 0) {
      const int m = (int)(n - i0 < 32 ? n - i0 : 32);
      double v = vb[b][lane];
      if (!up) {
        for (int t = 0; t < m; ++t) {
          const double xt = __shfl_sync(0xffffffffu, v, t);
          if (lane > t) v -= T[lane][t] * xt;
        }
      } else {
        // v / d as v r with r = 1 / d formed ahead of the chain, and its remainder
        const double d = T[lane][lane], rd = 1.0 / (lane < m ? d : 1.0);
        for (int t = m - 1; t >= 0; --t) {
          const double qv = v * rd, qc = fma(fma(-qv, d, v), rd, qv);
          const double xt = __shfl_sync(0xffffffffu, qc, t);
          if (lane == t) v = qc;
          if (lane < t) v -= T[lane][t] * xt;
        }
        // again with divisions if that left something that is no finite number (an infinite or subnormal d)
        if (__any_sync(0xffffffffu, (__double2hiint(v) & 0x7ff00000) == 0x7ff00000)) {
          v = vb[b][lane];
          for (int t = m - 1; t >= 0; --t) {
            const double xt = __shfl_sync(0xffffffffu, v / d, t);
            if (lane == t) v = xt;
            if (lane < t) v -= T[lane][t] * xt;
          }
        }
      }
      if (lane < m) xs[i0 + lane] = v;
    }
    __syncthreads();
  }
  if (rank == 0)
    for (int64_t t = tid; t < n; t += 256) x[t] = xs[t];
}

// The factorisation's launches, captured from stream `s` with a branch on `side`; flag: [n / 32 + 1] ints of scratch. The
// next block's columns are brought up to date first, on `s`, so that its panels, which keep eight SMs busy, run beside
// the interchanges and the update of all others on `side` (the step below: 42 ms with all in a row). Every kernel touches
// its own columns only; the block's own L is read by both branches and permuted by the next interchanges on `side`,
// behind the next panels.
inline cudaError_t enqueue_lu(double* K, int64_t n, int* piv, int* bad, int* flag, cudaStream_t s, cudaStream_t side,
                              cudaEvent_t panel, cudaEvent_t rest) {
  auto fine = [e = cudaSuccess](cudaError_t r) mutable { return e = e == cudaSuccess ? r : e; };
  const int groups = (int)((n + 31) / 32), tiles = (int)((n + kLuTile - 1) / kLuTile);
  for (int64_t b0 = 0; b0 < n; b0 += kLuBlock) {
    const int64_t b1 = b0 + kLuBlock < n ? b0 + kLuBlock : n, b2 = b1 + kLuBlock < n ? b1 + kLuBlock : n;
    for (int64_t k0 = b0; k0 < b1; k0 += kLuNB) {
      const int w = (int)(b1 - k0 < kLuNB ? b1 - k0 : kLuNB);
      k_lu_panel<<<kLuCluster, 256, lu_panel_smem((int)(n - k0)), s>>>(K, n, k0, w, b0, b1, piv, bad);
      if (k0 + w < b1) k_lu_inner<<<lu_inner_grid(n - k0 - w, b1 - k0 - w), 256, 0, s>>>(K, n, k0, w, b1);
    }
    const int next = b1 < n ? (int)(b1 / 32) : -1;
    fine(cudaEventRecord(panel, s));
    fine(cudaStreamWaitEvent(side, panel, 0));
    if (b1 < n) {
      if (b0 > 0) fine(cudaStreamWaitEvent(s, rest, 0));  // the next columns' share of the last update
      k_lu_swap<<<1, 128, 0, s>>>(K, n, b0, b1, piv, flag, next, -1);
      k_lu_inner<<<lu_inner_grid(n - b1, b2 - b1), 256, 0, s>>>(K, n, b0, (int)(b1 - b0), b2);
    }
    k_lu_swap<<<groups, 128, 0, side>>>(K, n, b0, b1, piv, flag, 0, next);
    if (b2 < n)
      k_lu_update<<<dim3(tiles - (int)(b2 / kLuTile), tiles - (int)(b1 / kLuTile)), 256, 0, side>>>(K, n, b0, b1, b2, flag);
    fine(cudaEventRecord(rest, side));
  }
  return fine(cudaStreamWaitEvent(s, rest, 0));
}

}  // namespace hdg
