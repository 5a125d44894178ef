// Mixed-precision assembly as one product with a constant matrix on the fifth-generation tensor cores.
//
// In reference coordinates (element_fp64.cuh) every entry of A', B', C', D' is a sum over points of a
// pointwise tensor times a number of the reference element:
//   block[(test, i)][(trial, l)] = sum_k T_il[k] W[k][(test, trial)],
// k running over (operator, point): T0, T1_r, T2_rr' at the volume points, U0, U1, U2_r' at the face
// points; W the product of the test and the trial function's values there. All elements share W, so
// the assembly is a GEMM whose rows are (element, pair (i, l)) and whose columns are (test, trial). The
// left operand is the raw tensor data: it is cut into slices once per value, where forming
// products of test functions and tensors first (the kernels this replaces) meant 6 times the
// values to form and cut, and a right operand of 444 KB per element.
//
// Arithmetic (ozaki.cuh): S = 6 integer slices per operand, the 21 slice products s + t <= 5 exact in
// FP32 accumulators, one per diagonal, over at most 128 entries of k; the diagonals are combined in
// double-float. A chunk is up to 128 entries of k with one scale per row and one per column.
//
// An MMA of M = 128, K = 16 takes about 150 clocks here whatever its width (N = 32 and N = 192 measured alike).
// So the slices t of the right operand lie behind one another in N: slice s of the left operand
// meets slices 0 .. 5 - s in ONE instruction of N = 32 (6 - s), whose accumulator columns are the diagonals
// s .. 5: six instructions per 16 entries of k instead of 21.
//
// Bound and measurements (82,944 tetrahedra, p = 3; the replaced volume, face, operator and residual kernels: 277 ms):
// rows and residuals 23 ms, products 103 to 109 ms from one GPU to another, of which the MMAs 57; the rest is the traffic of the running sums and of
// the blocks' 8-byte entries (4 MB of DRAM traffic an element).
//
// One persistent CTA per SM takes tiles of 128 rows. The tile's slices of one chunk (up to 8 steps of 16
// entries, 24 KB each) stay in shared memory while the chunk's column groups (32 columns, "jobs")
// pass; W streams through a ring. One warp copies, one issues the MMAs, 16 read the accumulators
// (two buffers in TMEM) and add them up: a column's running sum over the chunks is kept in a
// per-CTA plane [column][row] (coalesced), its last addition goes to A' or B'; a face's product goes to
// C' or D' and into the plane of its test function's node. A thread always meets the same (column,
// row): which quarter of a group a column lies in is fixed by its plane.
//
// Two row programs: pairs (i, l) with a viscous part (i, l > 0), and those without, which need the value
// operators only (elsewhere their blocks are zero).
//
// A mesh with fewer tiles than half the SMs would leave the chip idle while one CTA walks a tile's whole job list, so
// the planes are dealt by test node to several parts, each with a job list of its own (all columns of a plane
// have the same test node), and a tile is taken by one CTA per part. A plane's additions keep their order: the blocks are
// the same bit for bit. 48 tetrahedra, p = 3 (10 tiles): 0.14 ms in ten parts, 0.69 in one; the whole call 1.02 ms, 1.63
// in one part; 128 triangles, p = 3: 0.29 ms, 0.34.
#pragma once
#include "assemble_fp64.cuh"
#include "condense_t5.cuh"

namespace hdg {

constexpr int kT5Cols = 32, kT5Steps = 8, kT5Slices = 6, kT5Ring = 5;
constexpr uint32_t kT5ATile = 128 * 16 * 2, kT5BTile = kT5Cols * 16 * 2;  // one slice of one step

// one entry of k: operator kind (T5_T0 ..), its indices, the point
enum { T5_T0, T5_T1, T5_T2, T5_U0, T5_U1, T5_U2, T5_PAD };
struct T5Entry {
  short kind, f, r, r2;  // r2 = D: the sum over r'
  int pt;
};
// a column: A' (a, j), B' (a, (f2, c2)), and a face's rows (f, c) against interior j or trace (f2, c2)
enum { T5_COL_A, T5_COL_B, T5_COL_FI, T5_COL_FT, T5_COL_NONE };
struct T5ColDesc {
  short kind, f, a, j;  // a: test node (face rows: face node c), j: interior node or face node c2 of f2 (in f)
  short f2, pad;
};
// a job: a group of up to 32 columns of one kind that use the same steps of their chunk. Steps as a bit mask | chunk
// << 8 | T5_CLOSES (the chunk's last job) | T5_HAZARD (a plane of this group is also in the job before) | T5_FIRST /
// T5_LAST (its additions are the planes' first / last) | kind << 20. W holds the jobs' steps in order.
enum { T5_CLOSES = 1 << 16, T5_HAZARD = 1 << 17, T5_FIRST = 1 << 18, T5_LAST = 1 << 19, T5_KIND = 20 };
// a column's places, in bytes: its plane; the entry of C' (face rows against interior columns) or D' (against trace
// columns) it is written to at once; the entry of A' or B' that the plane's last addition is written to, both for
// pair (0, 0), -1 for an empty column; and 2^(column exponent - 16)
struct T5Col {
  int plane, direct;
  float scale;
  int fin;
};

struct T5Prog {  // device pointers
  const int* jobs;
  T5Col* cols;           // [jobs of all parts + 2][32] (two empty groups behind the last)
  const unsigned char* W;
  const int* pairs;      // [rpe] i << 8 | l
  const T5Entry* ent;    // [nchunk][128]
  const int* cstep;      // [nchunk + 1] first step of each chunk
  const int* wstep;      // [jobs] first step of each job in W
  const int* zero;       // entries that vanish for these pairs
  const int2* part;      // [nparts + 1] first job and first zero entry of each part
  unsigned char* T;        // slices of the rows [tile][steps][6][4 KB]
  int* erow;             // [tile][nchunk][128]
  int nchunk, rpe, ept, ntile, nsteps;
};

// Integer slices of a double: F = v 2^(48 - E) rounded to an integer (|v| < 2^E), split into balanced base-256
// digits on the integer pipe (GB300 converts FP64 at 1/64 of its FP32 rate). dig[0] is the leading one.
HDG_DEVI void t5_digits(double v, int E, int (&dig)[kT5Slices]) {
  const long long bits = __double_as_longlong(v);
  const int ex = (int)((bits >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)bits & 0xfffffffffffffull;
  if (ex) m |= 1ull << 52;
  // v = m 2^(ex - 1075): shift to the unit 2^(E - 48)
  const int sh = 1075 - ex + E - 48;  // >= 5 for every value below 2^E
  const unsigned long long q = sh >= 62 ? 0 : (m + (1ull << (sh - 1))) >> sh;
  long long F = bits < 0 ? -(long long)q : (long long)q;
#pragma unroll
  for (int s = kT5Slices - 1; s > 0; --s) {
    const int d = (int)(signed char)(F & 0xff);
    dig[s] = d;
    F = (F - d) >> 8;
  }
  dig[0] = (int)F;
}
// bf16 pair of two integers |d| <= 256 (exact): the high halves of their FP32 patterns
HDG_DEVI unsigned t5_pack(int d0, int d1) {
  const float f0 = __int_as_float(0x4b400000 + d0) - 12582912.f, f1 = __int_as_float(0x4b400000 + d1) - 12582912.f;
  return __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);
}
// exponent E with |v| < 2^E (clamped so that the scales stay in the float range)
HDG_DEVI int t5_exponent(double amax) {
  const int ex = (int)((__double_as_longlong(amax) >> 52) & 0x7ff);
  return max(ex - 1022, -100);
}

// Slices of a row's 8 consecutive entries, written as one 16-byte run per slice (umma_off layout).
HDG_DEVI void t5_put8(unsigned char* blk, uint32_t stride, uint32_t off, const double (&v)[8], int E) {
  uint32_t w[kT5Slices][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    int a[kT5Slices], b[kT5Slices];
    t5_digits(v[2 * p], E, a);
    t5_digits(v[2 * p + 1], E, b);
#pragma unroll
    for (int s = 0; s < kT5Slices; ++s) w[s][p] = t5_pack(a[s], b[s]);
  }
#pragma unroll
  for (int s = 0; s < kT5Slices; ++s)
    *reinterpret_cast<uint4*>(blk + s * stride + off) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

// ------------------------------------------------------------------------------------
// k_t5_rows: the two passes over the FP64 point tensors. A block forms the row exponents and slices of one (chunk, tile),
// program 0's before program 1's (the maximum and the slices read the values twice, the second time from L1), or,
// behind those, one element's residuals R_v and R_t in FP64. One launch: each part alone waits for its own latency
// on a small mesh (128 triangles, p = 3: 57 us in three launches, 32 in one).
// ------------------------------------------------------------------------------------
template <class C>
__global__ void __launch_bounds__(256) k_t5_rows(AssembleArgs a, DevTables Tb, T5Prog P0, T5Prog P1) {
  constexpr int D = C::D, M = C::M, MV = M - 1, NG = C::NG, NQ = C::NF * C::NGF;
  const int tid = threadIdx.x, n0 = P0.ntile * P0.nchunk, n1 = P1.ntile * P1.nchunk;
  if ((int)blockIdx.x >= n0 + n1) {
    __shared__ ElemTables<D> E;
    const int64_t le = blockIdx.x - n0 - n1, e = a.e0 + le;
    if (tid == 0) uniform_tables<C>(Tb, E);
    __syncthreads();
    double* R = a.R + e * (int64_t)(C::NV + C::NT);
    element_residual<D, 256>(UniformDims<C>(), E, a.ptv + le * NG * C::PT_VOL, a.ptf + le * NQ * C::PT_FACE,
                             a.hist ? a.hist + e * C::NV : nullptr, R, R + C::NV);
    return;
  }
  __shared__ T5Entry ent[128];
  __shared__ unsigned long long mx[128];
  const bool p0 = (int)blockIdx.x < n0;
  const T5Prog& P = p0 ? P0 : P1;
  const int at = p0 ? blockIdx.x : blockIdx.x - n0, tile = at % P.ntile, ch = at / P.ntile;
  const int s0 = P.cstep[ch], nk = P.cstep[ch + 1] - s0;
  for (int t = tid; t < 128; t += 256) {
    ent[t] = P.ent[ch * 128 + t];
    mx[t] = 0;
  }
  __syncthreads();
  const int row = tid & 127, el = row / P.rpe;
  const int64_t le = (int64_t)tile * P.ept + el;
  const bool live = el < P.ept && le < a.ne;
  const int pr = live ? P.pairs[row % P.rpe] : 0, i = pr >> 8, l = pr & 255;
  const int il = i * M + l, iv = (i - 1) * MV + l - 1;
  const double* pv = a.ptv + le * NG * C::PT_VOL;
  const double* pf = a.ptf + le * NQ * C::PT_FACE;
  auto load8 = [&](int kg, double (&v)[8]) {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const T5Entry en = ent[kg * 8 + j];
      double x = 0.0;
      if (live) switch (en.kind) {
          case T5_T0: x = pv[(M + D * M + il) * NG + en.pt]; break;
          case T5_T1: x = pv[(M + D * M + (1 + en.r) * M * M + il) * NG + en.pt]; break;
          case T5_T2:
            x = pv[(M + D * M + (1 + D) * M * M + (en.r * (D + 1) + en.r2) * MV * MV + iv) * NG + en.pt];
            break;
          case T5_U0: x = pf[(M + il) * NQ + en.pt]; break;
          case T5_U1: x = pf[(M + M * M + il) * NQ + en.pt]; break;
          case T5_U2: x = pf[(M + 2 * M * M + en.r2 * MV * MV + iv) * NQ + en.pt]; break;
          default: break;
        }
      v[j] = x;
    }
  };
  unsigned long long m = 0;
  for (int kg = tid >> 7; kg < 2 * nk; kg += 2) {
    double v[8];
    load8(kg, v);
#pragma unroll
    for (int j = 0; j < 8; ++j) {  // |v| compared as integers
      const unsigned long long u = (unsigned long long)__double_as_longlong(v[j]) & 0x7fffffffffffffffull;
      m = u > m ? u : m;
    }
  }
  atomicMax(mx + row, m);
  __syncthreads();
  const int E = t5_exponent(__longlong_as_double((long long)mx[row]));
  if (tid < 128) P.erow[((int64_t)tile * P.nchunk + ch) * 128 + row] = E;
  unsigned char* dst = P.T + ((int64_t)tile * P.nsteps + s0) * kT5Slices * kT5ATile;
  for (int kg = tid >> 7; kg < 2 * nk; kg += 2) {
    double v[8];
    load8(kg, v);
    t5_put8(dst + (kg >> 1) * kT5Slices * kT5ATile, kT5ATile, umma_off(row, 8 * (kg & 1)), v, E);
  }
}

// ------------------------------------------------------------------------------------
// k_t5_weights: the constant operand, one CTA per job (once per context)
// ------------------------------------------------------------------------------------
template <class C>
__global__ void __launch_bounds__(256) k_t5_weights(DevTables T, T5Prog P, const T5ColDesc* desc, unsigned char* W) {
  constexpr int D = C::D, NP = C::NP, NG = C::NG, NGF = C::NGF, NFN = C::NFN, NF = C::NF;
  const int job = P.jobs[blockIdx.x], chunk = (job >> 8) & 255, nk = __popc(job & 255);
  const int col = threadIdx.x & 31, kg0 = threadIdx.x >> 5;  // 8 groups of threads over the 8-entry runs
  const T5ColDesc cd = desc[blockIdx.x * kT5Cols + col];
  __shared__ unsigned long long mx[32];
  if (threadIdx.x < 32) mx[threadIdx.x] = 0;
  __syncthreads();
  auto value = [&](const T5Entry& e) -> double {
    const int g = e.pt, gf = e.pt - e.f * NGF;
    switch (cd.kind) {
      case T5_COL_A:
        if (e.kind == T5_T0) return T.Phi[g * NP + cd.a] * T.Phi[g * NP + cd.j];
        if (e.kind == T5_T1) return T.dPhi[(e.r * NG + g) * NP + cd.a] * T.Phi[g * NP + cd.j];
        if (e.kind == T5_T2 && e.r2 < D) return T.dPhi[(e.r * NG + g) * NP + cd.a] * T.dR[(e.r2 * NG + g) * NP + cd.j];
        return 0.0;
      case T5_COL_B:
        if (e.kind == T5_T2 && e.r2 == (cd.f ? cd.f - 1 : D)) {
          const double w = T.dPhi[(e.r * NG + g) * NP + cd.a] * T.PL[(cd.f * NG + g) * NFN + cd.j];
          return cd.f ? -w : w;
        }
        return 0.0;
      case T5_COL_FI:
        if (e.f != cd.f) return 0.0;
        if (e.kind == T5_U0 && T.nodepos[cd.f * NP + cd.j] >= 0)
          return T.Psi[(cd.f * NGF + gf) * NFN + cd.a] * T.PhiF[(cd.f * NGF + gf) * NP + cd.j];
        if (e.kind == T5_U2 && e.r2 < D)
          return T.Psi[(cd.f * NGF + gf) * NFN + cd.a] * T.dRF[((cd.f * D + e.r2) * NGF + gf) * NP + cd.j];
        return 0.0;
      case T5_COL_FT:
        if (e.f != cd.f) return 0.0;
        if (e.kind == T5_U1 && cd.f2 == cd.f)
          return T.Psi[(cd.f * NGF + gf) * NFN + cd.a] * T.Psi[(cd.f * NGF + gf) * NFN + cd.j];
        if (e.kind == T5_U2 && e.r2 == (cd.f2 ? cd.f2 - 1 : D)) {
          const double w = T.Psi[(cd.f * NGF + gf) * NFN + cd.a] * T.PLF[((cd.f * NF + cd.f2) * NGF + gf) * NFN + cd.j];
          return cd.f2 ? -w : w;
        }
        return 0.0;
      default: return 0.0;
    }
  };
  auto load8 = [&](int kg, double (&v)[8]) {
    const int step = __fns(job & 255, 0, (kg >> 1) + 1);  // the job's step number kg / 2
#pragma unroll 1
    for (int j = 0; j < 8; ++j) v[j] = value(P.ent[chunk * 128 + step * 16 + 8 * (kg & 1) + j]);
  };
  for (int kg = kg0; kg < 2 * nk; kg += 8) {
    double v[8];
    load8(kg, v);
    unsigned long long m = 0;
    for (int j = 0; j < 8; ++j) {
      const unsigned long long u = (unsigned long long)__double_as_longlong(v[j]) & 0x7fffffffffffffffull;
      m = u > m ? u : m;
    }
    atomicMax(mx + col, m);
  }
  __syncthreads();
  const int E = t5_exponent(__longlong_as_double((long long)mx[col]));
  if (threadIdx.x < 32) P.cols[blockIdx.x * kT5Cols + col].scale = oz_pow2(E - 16);
  for (int kg = kg0; kg < 2 * nk; kg += 8) {
    double v[8];
    load8(kg, v);
    t5_put8(W + (int64_t)(P.wstep[blockIdx.x] + (kg >> 1)) * kT5Slices * kT5BTile, kT5BTile, umma_off(col, 8 * (kg & 1)), v, E);
  }
}

// 4 consecutive FP32 accumulator columns, without waiting for the load
HDG_DEVI void tmem_ld4_async(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}
HDG_DEVI void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
HDG_DEVI void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// these waits last a microsecond or less: no sleep between the first polls
HDG_DEVI bool t5_wait(uint64_t* bar, uint32_t parity) { return mbar_wait(bar, parity, 4096); }

// The sum of the diagonals, sum_d 2^(-8 d) Q_d, as a normalised double-float. Every Q_d is an integer below 2^24,
// so the two pairs (Q0, Q1), (Q2, Q3) and their sum are exact two-term sums by an FMA and its residual
// (the residual's first difference is exact whichever operand is the larger: both are multiples of the
// smaller one's unit and the difference fits 24 bits); Q4 + Q5 / 256 is rounded to 2^-48 of the largest product.
HDG_DEVI df2 t5_combine(float q0, float q1, float q2, float q3, float q4, float q5) {
  constexpr float c8 = 1.f / 256.f, c16 = 1.f / 65536.f, c32 = c16 * c16;
  const float s1 = fmaf(q1, c8, q0), e1 = fmaf(q1, c8, q0 - s1);
  const float s2 = fmaf(q3, c8, q2), e2 = fmaf(q3, c8, q2 - s2);
  const float h = fmaf(s2, c16, s1), l = fmaf(s2, c16, s1 - h);
  const float lo = l + fmaf(fmaf(q5, c8, q4), c32, fmaf(e2, c16, e1));
  const float hi = h + lo;
  return {hi, lo - (hi - h)};
}

constexpr int kT5Epi = 16;                        // epilogue warps
constexpr int kT5Threads = 32 * (kT5Epi + 2);     // one warp copies, one issues the MMAs
constexpr int kT5Q = kT5Cols / (kT5Epi / 4);      // columns of a group per epilogue warp
constexpr int kT5MaxJobs = 400;                   // job words of both programs in shared memory
constexpr size_t kT5Smem = (size_t)kT5Steps * kT5Slices * kT5ATile + (size_t)kT5Ring * kT5Slices * kT5BTile + 256 +
                           kT5Epi * kT5Q * sizeof(T5Col) + sizeof(int) * kT5MaxJobs;

// ------------------------------------------------------------------------------------
// k_asm_t5: tiles [0, P0.ntile) of program 0, then those of program 1; CTA b takes part b % nparts of every
// (gridDim.x / nparts)-th one. planes: [grid][nplane + 1][128] (the last one takes the empty columns).
// Every wait is bounded; one that gives up sets s_fail, all roles then leave, the copies and MMAs in
// flight drain, and the tile's elements get HDG_STATUS_TIMEOUT.
// ------------------------------------------------------------------------------------
template <class C>
__global__ void __launch_bounds__(kT5Threads, 1) k_asm_t5(AssembleArgs a, T5Prog P0, T5Prog P1, df2* planes,
                                                          int nplane, int nparts) {
  constexpr int NV = C::NV, NT = C::NT;
  constexpr uint32_t ASTEP = kT5Slices * kT5ATile, WSTEP = kT5Slices * kT5BTile;
  extern __shared__ __align__(128) unsigned char smem_t5[];
  unsigned char* As = smem_t5;                           // [8][6][4 KB]
  unsigned char* Ws = As + (size_t)kT5Steps * ASTEP;     // [ring][6][1 KB]
  uint64_t* bars = reinterpret_cast<uint64_t*>(Ws + (size_t)kT5Ring * WSTEP);
  uint64_t* a_full = bars;                   // [8]
  uint64_t* a_empty = a_full + kT5Steps;     // [8]
  uint64_t* w_full = a_empty + kT5Steps;     // [ring]
  uint64_t* w_empty = w_full + kT5Ring;      // [ring]
  uint64_t* acc_full = w_empty + kT5Ring;    // [2]
  uint64_t* acc_empty = acc_full + 2;        // [2]
  uint64_t* drain = acc_empty + 2;
  int4* scols = reinterpret_cast<int4*>(reinterpret_cast<unsigned char*>(bars) + 256);  // [epilogue warp][kT5Q]
  int* sjobs = reinterpret_cast<int*>(scols + kT5Epi * kT5Q);
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ int4 s_part[2];  // this part of both programs: first job, jobs, first zero entry, end of its zero entries
  const int first = blockIdx.x / nparts, stride = gridDim.x / nparts;
  if (tid < 2) {
    const T5Prog& P = tid ? P1 : P0;
    const int2* pt = P.part + blockIdx.x % nparts;
    s_part[tid] = P.ntile ? make_int4(pt[0].x, pt[1].x - pt[0].x, pt[0].y, pt[1].y) : make_int4(0, 0, 0, 0);
  }
  __syncthreads();
  if (tid == 0) {
    s_fail = 0;
    for (int i = 0; i < 2 * kT5Steps + 2 * kT5Ring; ++i) mbar_init(bars + i, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(acc_full + i, 1);
      mbar_init(acc_empty + i, kT5Epi);
    }
    mbar_init(drain, 1);
    fence_mbar_init();
  }
  for (int t = tid; t < s_part[0].y; t += kT5Threads) sjobs[t] = P0.jobs[s_part[0].x + t];
  for (int t = tid; t < s_part[1].y; t += kT5Threads) sjobs[s_part[0].y + t] = P1.jobs[s_part[1].x + t];
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  const int ntile = P0.ntile + P1.ntile;

  if (warp == kT5Epi) {  // ---------------------------------------------------------------- copies
    if (lane == 0) {
      uint32_t a_use = 0, a_seen = 0;  // per slot: parity of its next "empty" wait; whether it was used before
      int w = 0, w_par = 1, nw = 0;
      uint32_t a_out = 0;              // per slot: loads issued, modulo 2 (for the drain)
      bool ok = true, stall = (a.stall_first_copy & kStallAssembly) && blockIdx.x == 0;
      for (int t = first; t < ntile && ok; t += stride) {
        const bool p0 = t < P0.ntile;
        const T5Prog& P = p0 ? P0 : P1;
        const int* jobs = sjobs + (p0 ? 0 : s_part[0].y);
        const int njob = s_part[p0 ? 0 : 1].y;
        const unsigned char* Ts = P.T + (int64_t)(p0 ? t : t - P0.ntile) * P.nsteps * ASTEP;
        const unsigned char* W = P.W + (int64_t)P.wstep[s_part[p0 ? 0 : 1].x] * WSTEP;
        int cur = -1;
        for (int j = 0; j < njob && ok; ++j) {
          const int job = jobs[j], chunk = (job >> 8) & 255;
          if (chunk != cur) {
            cur = chunk;
            const int s0 = P.cstep[cur], nk = P.cstep[cur + 1] - s0;
            for (int k = 0; k < nk; ++k) {
              if ((a_seen >> k) & 1u) {
                ok = t5_wait(a_empty + k, (a_use >> k) & 1u) && !s_fail;
                a_use ^= 1u << k;
              }
              if (!ok) break;
              a_seen |= 1u << k;
              mbar_arrive_expect_tx(a_full + k, ASTEP);
              if (!stall) bulk_g2s(As + (size_t)k * ASTEP, Ts + (int64_t)(s0 + k) * ASTEP, ASTEP, a_full + k);
              stall = false;  // the test hook leaves the first copy's phase incomplete
              a_out ^= 1u << k;
            }
          }
          for (int m = job & 255; m && ok; m &= m - 1) {
            ok = t5_wait(w_empty + w, w_par) && !s_fail;  // the first round passes at once
            if (!ok) break;
            mbar_arrive_expect_tx(w_full + w, WSTEP);
            bulk_g2s(Ws + (size_t)w * WSTEP, W, WSTEP, w_full + w);
            W += WSTEP;
            ++nw;
            if (++w == kT5Ring) {
              w = 0;
              w_par ^= 1;
            }
          }
        }
      }
      if (!ok) {  // the copies in flight land before the CTA leaves (bounded)
        s_fail = 1;
        for (int k = 0; k < kT5Steps; ++k)
          if ((a_seen >> k) & 1u) t5_wait(a_full + k, ((a_out >> k) & 1u) ^ 1u);
        for (int q = 0; q < kT5Ring && q < nw; ++q) {
          const int n = nw - 1 - q;  // the last loads, newest first
          t5_wait(w_full + n % kT5Ring, (n / kT5Ring) & 1);
        }
      }
    }
  } else if (warp > kT5Epi) {  // ---------------------------------------------------------------- MMAs
    if (lane == 0) {
      uint32_t a_par = 0, a_have = 0;  // per slot: parity of the next load; loaded for this chunk
      int w = 0, w_par = 0, buf = 0, e_par = 1;
      bool ok = true;
      const uint64_t adesc0 = umma_desc(smem_u32(As), 128, 256), wdesc0 = umma_desc(smem_u32(Ws), 128, 256);
      for (int t = first; t < ntile && ok; t += stride) {
        const bool p0 = t < P0.ntile;
        const T5Prog& P = p0 ? P0 : P1;
        const int* jobs = sjobs + (p0 ? 0 : s_part[0].y);
        const int njob = s_part[p0 ? 0 : 1].y;
        for (int j = 0; j < njob && ok; ++j) {
          const int job = jobs[j], used = job & 255;
          ok = t5_wait(acc_empty + buf, e_par) && !s_fail;  // the first use of each buffer passes at once
          if (!ok) break;
          tc_fence_after();
          if (job & T5_CLOSES) {  // steps the chunk's last job does not use are free
            const int chunk = (job >> 8) & 255, nk = P.cstep[chunk + 1] - P.cstep[chunk];
            for (int k = 0; k < nk; ++k)
              if (!((used >> k) & 1)) {
                if (!((a_have >> k) & 1u)) {  // its load is part of the slot's sequence
                  ok = ok && t5_wait(a_full + k, (a_par >> k) & 1u);
                  a_par ^= 1u << k;
                }
                umma_commit(a_empty + k);
              }
          }
          const uint32_t d0 = tmem + buf * 256;
          uint32_t acc = 0;
          for (int m = used; m && ok; m &= m - 1) {
            const int st = __ffs(m) - 1;
            if (!((a_have >> st) & 1u)) {
              ok = t5_wait(a_full + st, (a_par >> st) & 1u);
              a_par ^= 1u << st;
              a_have |= 1u << st;
            }
            ok = ok && t5_wait(w_full + w, w_par);
            if (!ok) break;
            const uint64_t ad = adesc0 + (uint64_t)(st * (ASTEP >> 4)), wd = wdesc0 + (uint64_t)(w * (WSTEP >> 4));
#pragma unroll
            for (int s = 0; s < kT5Slices; ++s) {
              constexpr uint32_t base = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24);  // UmmaIdesc<128, N>
              const uint32_t n = kT5Cols * (kT5Slices - s);
              umma_bf16(d0 + s * kT5Cols, ad + (uint64_t)(s * (kT5ATile >> 4)), wd, base | ((n >> 3) << 17), acc);
              acc = 1;
            }
            umma_commit(w_empty + w);
            if (job & T5_CLOSES) umma_commit(a_empty + st);
            if (++w == kT5Ring) {
              w = 0;
              w_par ^= 1;
            }
          }
          if (job & T5_CLOSES) a_have = 0;
          if (!ok) break;
          umma_commit(acc_full + buf);
          if (++buf == 2) {
            buf = 0;
            e_par ^= 1;
          }
        }
      }
      if (!ok) s_fail = 1;
      umma_commit(drain);  // every MMA of this thread has completed before TMEM is freed
      t5_wait(drain, 0);
    }
  } else {  // ---------------------------------------------------------------- accumulators -> blocks
    // Columns are read two jobs ahead (lane c holds the warp's column c), the planes' running sums one job ahead,
    // so that neither latency stands between two jobs.
    const int q = warp & 3, part = warp >> 2, row = 32 * q + lane;
    unsigned char* Y = reinterpret_cast<unsigned char*>(planes + (int64_t)blockIdx.x * (nplane + 1) * 128 + row);
    int4* sc = scols + warp * kT5Q;
    int f_par = 0, turn = 0;
    bool ok = true;
    for (int t = first; t < ntile && ok; t += stride) {
      const bool p0 = t < P0.ntile;
      const T5Prog& P = p0 ? P0 : P1;
      const int* jobs = sjobs + (p0 ? 0 : s_part[0].y);
      const int4 mine = s_part[p0 ? 0 : 1];
      const int tile = p0 ? t : t - P0.ntile, njob = mine.y, el = row / P.rpe;
      const int64_t le = (int64_t)tile * P.ept + el, e = a.e0 + le;
      const bool live = el < P.ept && le < a.ne;
      const int pr = live ? P.pairs[row % P.rpe] : 0, i = pr >> 8, l = pr & 255;
      unsigned char* out[4];
      out[0] = reinterpret_cast<unsigned char*>(a.Ap + le * NV * NV + i * NV + l);
      out[1] = reinterpret_cast<unsigned char*>(a.recov + e * (int64_t)(NV * NT + NV) + i * NT + l);
      out[2] = reinterpret_cast<unsigned char*>(a.Cp + le * NT * NV + i * NV + l);
      out[3] = reinterpret_cast<unsigned char*>(a.S + e * (int64_t)NT * NT + i * NT + l);
      const int4* ct = reinterpret_cast<const int4*>(P.cols) + mine.x * kT5Cols + kT5Q * part +
                       (lane & (kT5Q - 1));
      const int* er = P.erow + (int64_t)tile * P.nchunk * 128 + row;
      auto load_y = [&](int job, const int4& cc, df2 (&dst)[kT5Q]) {
        if (job & T5_FIRST) return;
#pragma unroll
        for (int c = 0; c < kT5Q; ++c)
          dst[c] = *reinterpret_cast<const df2*>(Y + __shfl_sync(0xffffffffu, cc.x, c));
      };
      int4 c0 = ct[0], c1 = ct[kT5Cols];  // this job's columns and the next one's
      int cur = -1;
      float rs = 1.f;
      // one job with its running sums y; the next job's into yn
      auto one = [&](int j, df2 (&y)[kT5Q], df2 (&yn)[kT5Q]) {
        const int job = jobs[j], next = j + 1 < njob ? jobs[j + 1] : T5_FIRST, chunk = (job >> 8) & 255;
        if (lane < kT5Q) sc[lane] = c0;
        __syncwarp();
        const int4 c2 = ct[(j + 2) * kT5Cols];
        if (!(next & T5_HAZARD)) load_y(next, c1, yn);
        if (chunk != cur) {
          cur = chunk;
          const int E = er[cur * 128];
          rs = E > 127 ? __int_as_float(0x7fffffff) : oz_pow2(E);  // NaN: an entry beyond the float range
        }
        const int kind = (job >> T5_KIND) & 3;
        unsigned char* od = kind == T5_COL_FI ? out[2] : out[3];
        unsigned char* of = kind == T5_COL_A || kind == T5_COL_FI ? out[0] : out[1];
        const bool direct = kind >= T5_COL_FI, add = !(job & T5_FIRST), fin = (job & T5_LAST) != 0;
        ok = __all_sync(0xffffffffu, t5_wait(acc_full + turn, f_par) && !s_fail);
        if (!ok) return;
        tc_fence_after();
        const uint32_t ta = tmem + ((uint32_t)(32 * q) << 16) + turn * 256 + kT5Q * part;
#pragma unroll
        for (int g4 = 0; g4 < kT5Q / 4; ++g4) {
          uint32_t v[kT5Slices][4];
#pragma unroll
          for (int d = 0; d < kT5Slices; ++d) tmem_ld4_async(ta + d * kT5Cols + 4 * g4, v[d]);
          tmem_ld_wait();
#pragma unroll
          for (int d = 0; d < kT5Slices; ++d)
#pragma unroll
            for (int c = 0; c < 4; ++c) asm volatile("" : "+r"(v[d][c]));  // no use of them moves above the wait
          if (g4 == kT5Q / 4 - 1) {  // the buffer has been read
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(acc_empty + turn);
          }
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int4 cc = sc[4 * g4 + c];
            df2 p = t5_combine(__uint_as_float(v[0][c]), __uint_as_float(v[1][c]), __uint_as_float(v[2][c]),
                               __uint_as_float(v[3][c]), __uint_as_float(v[4][c]), __uint_as_float(v[5][c]));
            const float s = __int_as_float(cc.z) * rs;
            p.hi *= s;
            p.lo *= s;
            if (direct && live && cc.y >= 0) *reinterpret_cast<df2*>(od + cc.y) = p;
            if (add) {
              const df2 u = y[4 * g4 + c];
              const float h = u.hi + p.hi, bb = h - u.hi;
              const float lo = ((u.hi - (h - bb)) + (p.hi - bb)) + (u.lo + p.lo);
              p.hi = h + lo;
              p.lo = lo - (p.hi - h);
            }
            if (fin) {
              if (live && cc.w >= 0) *reinterpret_cast<df2*>(of + cc.w) = p;
            } else {
              *reinterpret_cast<df2*>(Y + cc.x) = p;
            }
          }
        }
        __syncwarp();  // every lane has read sc
        if (next & T5_HAZARD) load_y(next, c1, yn);
        c0 = c1;
        c1 = c2;
        if (turn) f_par ^= 1;
        turn ^= 1;
      };
      df2 ya[kT5Q], yb[kT5Q];
      load_y(jobs[0], c0, ya);
      for (int j = 0; j < njob && ok; j += 2) {
        __syncwarp();
        one(j, ya, yb);
        if (j + 1 < njob && ok) {
          __syncwarp();
          one(j + 1, yb, ya);
        }
      }
      if (!ok) {
        s_fail = 1;
        break;
      }
      for (int z = s_part[p0 ? 0 : 1].z + part; z < s_part[p0 ? 0 : 1].w; z += kT5Epi / 4) {  // zero[]: array << 28 | byte offset / 8
        const int w = P.zero[z], arr = w >> 28;
        unsigned char* p = arr == 0 ? out[0] : arr == 1 ? out[1] : arr == 2 ? out[2] : out[3];
        if (live) reinterpret_cast<df2*>(p)[w & 0xfffffff] = df2{0.f, 0.f};
      }
    }
  }
  __syncthreads();
  if (s_fail)  // every element of this CTA's tiles is recomputed (or reported)
    for (int t = first; t < ntile; t += stride) {
      const T5Prog& P = t < P0.ntile ? P0 : P1;
      const int64_t l0 = (int64_t)(t < P0.ntile ? t : t - P0.ntile) * P.ept;
      for (int x = tid; x < P.ept; x += kT5Threads)
        if (l0 + x < a.ne) atomicOr(a.status + a.e0 + l0 + x, HDG_STATUS_TIMEOUT);
    }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
}

}  // namespace hdg
