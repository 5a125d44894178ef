// FP64 building blocks of one element, shared by the uniform kernels (assemble_fp64.cuh) and the
// element-class kernel of mixed-degree meshes (pclass.cu): the quadrature contractions into A', B',
// C', D' and the residuals, and the condensation X = A'^{-1}[B' | R_v], S = D' - C' X.
//
// Bound: the FP64 pipe. A GB300 SM retires two FP64 FMA per clock, so one warp FMA keeps its
// scheduler's FP64 unit busy for 64 clocks; loads and index arithmetic hide behind it and only the
// number of FMAs counts. Three properties of the problem remove most of them (tetrahedra, p = 3:
// 11.8M -> 3.8M FMA an element for the assembly; 3,072 elements: 116.0 -> 26.4 ms, 18.7 ms at the
// pipe's rate; the condensation below 49.7 -> 38.8 ms, 31.3 ms at the pipe's rate):
//   * reference operators: n_f |F| / |K| is a constant combination of the rows of Jinv (gradients
//     of the barycentric coordinates), so with dG/dq contracted at the points with Jinv on both
//     sides (T2[r][r']) every right operator is a table of the reference element:
//       R_r'(g, j) = dPhi_r' + PL_{r'+1} phi_j - PL_0 phi_j,   R_r'(g, (f, c)) = PL_0 (f = 0),
//       -PL_f (f = r' + 1), zero otherwise;
//     a trace column then needs one operator instead of D;
//   * dG_i/dq_l vanishes for i = 0 or l = 0, so 9 of the 25 pairs (i, l) have the value operator only;
//   * on a face the trial side is contracted first (16 points x all columns), then one product
//     with the face's trace basis gives the C', D' rows; the rows of A', B' are the same numbers
//     (or, where the trace degree is the higher one, combinations of them).
#pragma once
#include "hdg_device.cuh"

namespace hdg {

// Reference operators of one element (device pointers; face arrays by local face).
template <int D>
struct ElemTables {
  const double *Phi, *dPhi, *dR;   // [NG][NP], [D][NG][NP] basis, gradients, R_r' of the interior columns
  const double *PhiF, *dRF;        // [NF][NGF][NP], [NF][D][NGF][NP] the same at the face points
  const double* Psi[D + 1];        // trace basis of face f at its points [NGF][nq]
  const double* PL[D + 1];         // lift of face f's trace functions at the volume points [NG][nq]
  const double* PLF[D + 1];        // the same at the points of face ff: PLF[f] + ff sPLF[f], [NGF][nq]
  const double* Tr[D + 1];         // null: the trace nodes are the element's face nodes; else phi_a there [nq][NP]
  const int* nodepos;              // [NF][NP] position of node a among the element's nodes of face f, or -1
  int sPLF[D + 1];
  int nq[D + 1], off[D + 2];       // trace nodes of face f and the first one's local number
  int offp[D + 2];                 // the same with every face padded to an even count
};

// Sizes of the contraction: any type with members NP, NG, NGF, NTN (trace nodes), NPs, NZs (NP and
// NP + trace nodes with every group padded to an even count) and NV, NT.
// FB faces share one pass over the trial side, ZB left factors are buffered.
template <class Dm>
__host__ __device__ constexpr int element_smem_doubles(const Dm& d, int FB, int ZB) {
  const int h = FB * d.NGF * d.NZs, z = ZB * d.NG * d.NPs;
  return d.NTN * d.NZs + (h > z ? h : z);
}

// Point tensors are stored [quantity][point]: volume MU [M], FR [D][M], T0 [M][M], T1 [D][M][M],
// T2 [D][D+1][M-1][M-1]; faces (point index f NGF + gf) HF [M], U0 [M][M], U1 [M][M], U2 [D+1][M-1][M-1]. The last
// entry of a [D+1] index is the sum over the others (the operator of face 0's trace).

// R_v [NV] (hist may be null) and R_t [NT] in shared memory or global memory
template <int D, int NTH, class Dm>
HDG_DEVI void element_residual(const Dm& d, const ElemTables<D>& T, const double* ptv, const double* ptf,
                               const double* hist, double* Rv, double* Rt) {
  constexpr int M = D + 2, NF = D + 1;
  const int NP = d.NP, NG = d.NG, NGF = d.NGF, NQ = NF * NGF, tid = threadIdx.x;
  const double *MU = ptv, *FR = ptv + M * NG;
  for (int t = tid; t < d.NTN * M; t += NTH) {
    const int tn = t / M, i = t % M;
    int f = 0;
    while (tn >= T.off[f + 1]) ++f;
    const double* psi = T.Psi[f] + (tn - T.off[f]);
    double s = 0.0;
    for (int gf = 0; gf < NGF; ++gf) s += psi[gf * T.nq[f]] * ptf[i * NQ + f * NGF + gf];
    Rt[t] = s;
  }
  for (int t = tid; t < NP * M; t += NTH) {
    const int a = t / M, i = t % M;
    double s = hist ? -hist[t] : 0.0;
    for (int g = 0; g < NG; ++g) {
      s += T.Phi[g * NP + a] * MU[i * NG + g];
#pragma unroll
      for (int r = 0; r < D; ++r) s += T.dPhi[(r * NG + g) * NP + a] * FR[(r * M + i) * NG + g];
    }
    for (int f = 0; f < NF; ++f) {
      if (T.nodepos[f * NP + a] < 0) continue;
      for (int gf = 0; gf < NGF; ++gf) s += T.PhiF[(f * NGF + gf) * NP + a] * ptf[i * NQ + f * NGF + gf];
    }
    Rv[t] = s;
  }
}

// A' [NV][NV], B' [NV][NT], C' [NT][NV], D' [NT][NT] (global memory). sm: element_smem_doubles.
//
// Per pair (i, l): the trial side of the faces H, the face rows F = Psi^T H (shared memory, C' and
// D'), then up to D + 2 volume operators, each a left factor Z (test side) built in one of two
// shared buffers while the other one is multiplied. One operator's 2 x 2 tiles, those of A' and
// then those of one face's block of B', are one list over the threads (NRD rounds), so that only
// the list's last warp is partly filled; A' tiles stay in registers over the operators, a trace
// face's block is complete after one. Large classes take one face per pass and one left factor
// (FB = ZB = 1), so that two CTAs still share an SM.
template <int D, bool VISC, int NTH, int NRD, int FB, int ZB, class Dm>
HDG_DEVI void element_blocks(const Dm& d, const ElemTables<D>& T, const double* __restrict__ ptv,
                             const double* __restrict__ ptf, double* Ap, double* Bp, double* Cp, double* Dp,
                             double* sm) {
  constexpr int M = D + 2, MV = M - 1, NF = D + 1;
  const int NP = d.NP, NG = d.NG, NGF = d.NGF, NTN = d.NTN, NPs = d.NPs, NZs = d.NZs, NV = d.NV, NT = d.NT;
  const int NQ = NF * NGF, tid = threadIdx.x;
  double* F = sm;               // [NTN][NZs]
  double* H = F + NTN * NZs;    // [FB NGF][NZs]
  double* Z = H;                // [ZB][NG][NPs], after H
  const double* T0 = ptv + (M + D * M) * NG;
  const double* T1 = T0 + M * M * NG;
  const double* T2 = T1 + D * M * M * NG;
  const double* U0 = ptf + M * NQ;
  const double* U1 = U0 + M * M * NQ;
  const double* U2 = U1 + M * M * NQ;
  const int tA = NPs / 2, nAt = tA * tA;

  for (int il = 0; il < M * M; ++il) {
    const int i = il / M, l = il % M;
    const bool visc = VISC && i > 0 && l > 0;
    const int iv = visc ? (i - 1) * MV + (l - 1) : 0;
    for (int f0 = 0; f0 < NF; f0 += FB) {
      // trial side of FB faces
      for (int t = tid; t < FB * NGF * NZs; t += NTH) {
        const int p = f0 * NGF + t / NZs, col = t % NZs, f = p / NGF, gf = p % NGF;
        double v = 0.0;
        if (col < NPs) {
          if (col < NP) {
            v = U0[il * NQ + p] * T.PhiF[p * NP + col];
            if (visc)
#pragma unroll
              for (int r = 0; r < D; ++r)
                v += U2[(r * MV * MV + iv) * NQ + p] * T.dRF[((f * D + r) * NGF + gf) * NP + col];
          }
        } else {
          const int tp = col - NPs;
          int fl = 0;
          while (tp >= T.offp[fl + 1]) ++fl;
          const int c = tp - T.offp[fl], nq = T.nq[fl];
          if (c < nq) {
            if (fl == f) v = U1[il * NQ + p] * T.Psi[f][gf * nq + c];
            if (visc) {
              const double u = fl > 0 ? -U2[((fl - 1) * MV * MV + iv) * NQ + p] : U2[(D * MV * MV + iv) * NQ + p];
              v += u * T.PLF[fl][f * T.sPLF[fl] + gf * nq + c];
            }
          }
        }
        H[t] = v;
      }
      __syncthreads();
      // face rows: 2 x 2 tiles; a pair without the viscous part reaches the face's own trace columns only
      {
        int nqm = 0;
#pragma unroll
        for (int f = 0; f < NF; ++f) nqm = max(nqm, T.offp[f + 1] - T.offp[f]);
        const int ncp = visc ? NZs / 2 : (NPs + nqm) / 2, rp0 = T.offp[f0] / 2, nrp = T.offp[f0 + FB] / 2 - rp0;
        for (int t = tid; t < nrp * ncp; t += NTH) {
          const int rp = rp0 + t / ncp, cp = t % ncp;
          int f = 0;
          while (2 * rp >= T.offp[f + 1]) ++f;
          const int c0 = 2 * rp - T.offp[f], nq = T.nq[f];
          int col = 2 * cp, fl = -1, cc = col;  // fl: face of the trace columns, cc: column within the group
          if (col >= NPs) {
            if (visc) {
              fl = 0;
              while (col - NPs >= T.offp[fl + 1]) ++fl;
              cc = col - NPs - T.offp[fl];
            } else {
              fl = f;
              cc = col - NPs;
              col = NPs + T.offp[f] + cc;
            }
            if (cc >= T.nq[fl]) continue;
          }
          const bool r1 = c0 + 1 < nq;
          const double* psi = T.Psi[f] + c0;
          const double* h = H + (f - f0) * NGF * NZs + col;
          double a00 = 0.0, a01 = 0.0, a10 = 0.0, a11 = 0.0;
#pragma unroll 4
          for (int gf = 0; gf < NGF; ++gf) {
            const double p0 = psi[gf * nq], p1 = r1 ? psi[gf * nq + 1] : 0.0;
            const double2 hv = *reinterpret_cast<const double2*>(h + gf * NZs);
            a00 += p0 * hv.x;
            a01 += p0 * hv.y;
            a10 += p1 * hv.x;
            a11 += p1 * hv.y;
          }
          const bool k1 = cc + 1 < (fl < 0 ? NP : T.nq[fl]);
#pragma unroll
          for (int rr = 0; rr < 2; ++rr) {
            if (rr && !r1) break;
            const int tn = T.off[f] + c0 + rr, row = tn * M + i;
            const double v0 = rr ? a10 : a00, v1 = rr ? a11 : a01;
            *reinterpret_cast<double2*>(F + tn * NZs + col) = make_double2(v0, v1);
            double* dst = fl < 0 ? Cp + (int64_t)row * NV + cc * M + l : Dp + (int64_t)row * NT + (T.off[fl] + cc) * M + l;
            dst[0] = v0;
            if (k1) dst[M] = v1;
          }
        }
        if (!visc && f0 == 0)  // the other faces' columns of D' are zero for this pair
          for (int t = tid; t < NTN * NTN; t += NTH) {
            const int r = t / NTN, c = t % NTN;
            int f = 0;
            while (r >= T.off[f + 1]) ++f;
            if (c < T.off[f] || c >= T.off[f + 1]) Dp[(int64_t)(r * M + i) * NT + c * M + l] = 0.0;
          }
      }
      __syncthreads();
    }
    // F's share of entry (test node a, column position col of F)
    auto face_part = [&](int a, int col, int f) {
      const int pos = T.nodepos[f * NP + a];
      if (pos < 0) return 0.0;
      if (!T.Tr[f]) return F[(T.off[f] + pos) * NZs + col];
      double s = 0.0;
      for (int c = 0; c < T.nq[f]; ++c) s += T.Tr[f][c * NP + a] * F[(T.off[f] + c) * NZs + col];
      return s;
    };
    auto build = [&](int o, double* Zb) {
      for (int t = tid; t < NG * NPs; t += NTH) {
        const int g = t / NPs, a = t % NPs;
        double v = 0.0;
        if (a < NP) {
          if (o == 0) {
            v = T.Phi[g * NP + a] * T0[il * NG + g];
#pragma unroll
            for (int r = 0; r < D; ++r) v += T.dPhi[(r * NG + g) * NP + a] * T1[(r * M * M + il) * NG + g];
          } else {
#pragma unroll
            for (int r = 0; r < D; ++r)
              v += T.dPhi[(r * NG + g) * NP + a] * T2[((r * (D + 1) + o - 1) * MV * MV + iv) * NG + g];
          }
        }
        Zb[t] = v;
      }
    };
    const int nops = visc ? D + 2 : 1;
    double acc[NRD][4];
#pragma unroll
    for (int x = 0; x < NRD; ++x) acc[x][0] = acc[x][1] = acc[x][2] = acc[x][3] = 0.0;
    build(0, Z);
    __syncthreads();
    for (int o = 0; o < nops; ++o) {
      const double* Zb = Z + (o % ZB) * NG * NPs;
      if (ZB > 1 && o + 1 < nops) build(o + 1, Z + ((o + 1) % ZB) * NG * NPs);
      const int f = o <= D ? o : 0;  // the face of this operator's trace columns (o >= 1)
      const int nA = o <= D ? nAt : 0, tq = o >= 1 ? (T.nq[f] + 1) / 2 : 0, n = nAt + tA * tq;
#pragma unroll
      for (int x = 0; x < NRD; ++x) {
        const int t = tid + x * NTH;
        if (t >= n || (t < nAt && nA == 0)) continue;
        const bool isA = t < nAt;
        const int tb = t - nAt, a0 = 2 * (isA ? t / tA : tb / tq), j0 = 2 * (isA ? t % tA : tb % tq);
        const int ldw = isA ? NP : T.nq[f], d1 = j0 + 1 < ldw ? 1 : 0;
        const double* z = Zb + a0;
        const double* w = (isA ? (o == 0 ? T.Phi : T.dR + (o - 1) * NG * NP) : T.PL[f]) + j0;
#pragma unroll 4
        for (int g = 0; g < NG; ++g) {
          const double2 zv = *reinterpret_cast<const double2*>(z + g * NPs);
          const double w0 = w[g * ldw], w1 = w[g * ldw + d1];
          acc[x][0] += zv.x * w0;
          acc[x][1] += zv.x * w1;
          acc[x][2] += zv.y * w0;
          acc[x][3] += zv.y * w1;
        }
        if (!isA) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int a = a0 + (q >> 1), c = j0 + (q & 1);
            if (a < NP && c < T.nq[f]) {
              double v = o <= D ? -acc[x][q] : acc[x][q];
#pragma unroll
              for (int ff = 0; ff < NF; ++ff) v += face_part(a, NPs + T.offp[f] + c, ff);
              Bp[(int64_t)(a * M + i) * NT + (T.off[f] + c) * M + l] = v;
            }
            acc[x][q] = 0.0;
          }
        }
      }
      __syncthreads();
      if (ZB == 1 && o + 1 < nops) {
        build(o + 1, Z);
        __syncthreads();
      }
    }
#pragma unroll
    for (int x = 0; x < NRD; ++x) {
      const int t = tid + x * NTH;
      if (t >= nAt) break;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int a = 2 * (t / tA) + (q >> 1), j = 2 * (t % tA) + (q & 1);
        if (a >= NP || j >= NP) continue;
        double v = acc[x][q];
#pragma unroll
        for (int ff = 0; ff < NF; ++ff) v += face_part(a, j, ff);
        Ap[(int64_t)(a * M + i) * NV + j * M + l] = v;
      }
    }
    if (!visc)
      for (int t = tid; t < NP * NTN; t += NTH) {
        const int a = t / NTN, tn = t % NTN;
        int f = 0;
        while (tn >= T.off[f + 1]) ++f;
        Bp[(int64_t)(a * M + i) * NT + tn * M + l] = face_part(a, NPs + T.offp[f] + tn - T.off[f], f);
      }
  }
  __syncthreads();
}

// ------------------------------------------------------------------------------------
// Condensation of one element. LU: [n][ld] (shared memory, or global for an interior block that
// does not fit), factored in place with partial pivoting; column n holds R_v on entry and the
// forward-substituted L^{-1} P R_v on return (the update carries it along). perm[r]: the row of A'
// that ends in row r; dinv[r]: the reciprocal of pivot r. Step k: warp 0 searches the pivot, the
// rows are swapped, then a warp scales and updates whole rows (no division of a flat index).
// Returns true if every pivot is nonzero.
// ------------------------------------------------------------------------------------
template <int NTH>
HDG_DEVI bool element_lu(double* LU, int ld, int n, int* perm, double* dinv, int* s_piv) {
  constexpr int NW = NTH / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int r = tid; r < n; r += NTH) perm[r] = r;
  bool ok = true;
  for (int k = 0; k < n; ++k) {
    if (warp == 0) {
      double best = -1.0;
      int bi = k;
      for (int r = k + lane; r < n; r += 32) {
        const double v = fabs(LU[r * ld + k]);
        if (v > best) {
          best = v;
          bi = r;
        }
      }
      for (int off = 16; off > 0; off >>= 1) {
        const double ob = __shfl_down_sync(0xffffffffu, best, off);
        const int oi = __shfl_down_sync(0xffffffffu, bi, off);
        if (ob > best || (ob == best && oi < bi)) {
          best = ob;
          bi = oi;
        }
      }
      if (lane == 0) {
        const double dk = LU[bi * ld + k];
        s_piv[0] = bi;
        s_piv[1] = best > 0.0 ? 1 : 0;
        dinv[k] = dk != 0.0 ? 1.0 / dk : 0.0;
      }
    }
    __syncthreads();
    const int p = s_piv[0];
    ok = ok && s_piv[1] != 0;
    const double inv = dinv[k];
    if (p != k) {
      for (int j = tid; j <= n; j += NTH) {
        const double t = LU[k * ld + j];
        LU[k * ld + j] = LU[p * ld + j];
        LU[p * ld + j] = t;
      }
      if (tid == 0) {
        const int t = perm[k];
        perm[k] = perm[p];
        perm[p] = t;
      }
      __syncthreads();
    }
    for (int r = k + 1 + warp; r < n; r += NW) {
      const double m = LU[r * ld + k] * inv;
      for (int c = k + 1 + lane; c <= n; c += 32) LU[r * ld + c] -= m * LU[k * ld + c];
      __syncwarp();
      if (lane == 0) LU[r * ld + k] = m;
    }
    __syncthreads();
  }
  return ok;
}

// y = U^{-1} (column n of LU) by warp 0, into y and ys [n] (shared memory)
template <int NTH>
HDG_DEVI void element_solve_y(const double* LU, int ld, int n, const double* dinv, double* ys, double* y) {
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {
    for (int r = lane; r < n; r += 32) ys[r] = LU[r * ld + n];
    __syncwarp();
    for (int k = n - 1; k >= 0; --k) {
      const double v = ys[k] * dinv[k];
      __syncwarp();
      for (int r = lane; r < k; r += 32) ys[r] -= LU[r * ld + k] * v;
      if (lane == 0) {
        ys[k] = v;
        y[k] = v;
      }
      __syncwarp();
    }
  }
}

// X = A'^{-1} B' and S = D' - C' X in blocks of CB right-hand sides: X and S hold B' and D' on
// entry ([n][nt], [nt][nt]). Xs: [n][CB] shared memory. The triangular solves go through the rows
// in blocks of 8: one thread per column solves the block's triangle, then every thread updates 4 x 4
// tiles of the rows left with the block's 8 rows (128 FMA for 64 shared-memory operands); the Schur
// product takes 4 x 8 tiles with C' read through L1.
template <int NTH, int CB>
HDG_DEVI void element_solve_schur(const double* LU, int ld, int n, const int* perm, const double* dinv, double* Xs,
                                  const double* Cp, double* X, double* S, int nt) {
  constexpr int NB = 8;
  static_assert(CB % 4 == 0 && CB <= NTH && NTH % 32 == 0, "tiles");
  const int tid = threadIdx.x;
  for (int c0 = 0; c0 < nt; c0 += CB) {
    const int nc = min(CB, nt - c0), nct = (nc + 3) / 4;
    for (int t = tid; t < n * CB; t += NTH) {
      const int r = t / CB, c = t % CB;
      Xs[t] = c < nc ? X[(int64_t)perm[r] * nt + c0 + c] : 0.0;
    }
    __syncthreads();
    auto update = [&](int kb, int nb, int lo, int rows) {  // rows [lo, lo + rows) -= LU[., kb..] x_kb
      const int nrt = (rows + 3) / 4;
      for (int t = tid; t < nrt * nct; t += NTH) {
        const int r0 = lo + 4 * (t / nct), cc = 4 * (t % nct);
        const int rl = lo + rows - 1;
        int rr[4];
        double acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          rr[a] = min(r0 + a, rl);
          const double2 u = *reinterpret_cast<const double2*>(Xs + rr[a] * CB + cc);
          const double2 v = *reinterpret_cast<const double2*>(Xs + rr[a] * CB + cc + 2);
          acc[a][0] = u.x;
          acc[a][1] = u.y;
          acc[a][2] = v.x;
          acc[a][3] = v.y;
        }
#pragma unroll 4
        for (int k = 0; k < nb; ++k) {
          const double2 u = *reinterpret_cast<const double2*>(Xs + (kb + k) * CB + cc);
          const double2 v = *reinterpret_cast<const double2*>(Xs + (kb + k) * CB + cc + 2);
#pragma unroll
          for (int a = 0; a < 4; ++a) {
            const double m = LU[rr[a] * ld + kb + k];
            acc[a][0] -= m * u.x;
            acc[a][1] -= m * u.y;
            acc[a][2] -= m * v.x;
            acc[a][3] -= m * v.y;
          }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          if (r0 + a > rl) break;
          *reinterpret_cast<double2*>(Xs + rr[a] * CB + cc) = make_double2(acc[a][0], acc[a][1]);
          *reinterpret_cast<double2*>(Xs + rr[a] * CB + cc + 2) = make_double2(acc[a][2], acc[a][3]);
        }
      }
    };
    for (int kb = 0; kb < n; kb += NB) {  // forward, unit lower
      const int nb = min(NB, n - kb);
      if (tid < nc) {
        double x[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) x[k] = k < nb ? Xs[(kb + k) * CB + tid] : 0.0;
#pragma unroll
        for (int k = 0; k < NB; ++k) {
#pragma unroll
          for (int r = k + 1; r < NB; ++r)
            if (r < nb) x[r] -= LU[(kb + r) * ld + kb + k] * x[k];
        }
#pragma unroll
        for (int k = 1; k < NB; ++k)
          if (k < nb) Xs[(kb + k) * CB + tid] = x[k];
      }
      __syncthreads();
      if (kb + nb < n) update(kb, nb, kb + nb, n - kb - nb);
      __syncthreads();
    }
    for (int kb = (n - 1) / NB * NB; kb >= 0; kb -= NB) {  // backward, upper
      const int nb = min(NB, n - kb);
      if (tid < nc) {
        double x[NB];
#pragma unroll
        for (int k = 0; k < NB; ++k) x[k] = k < nb ? Xs[(kb + k) * CB + tid] : 0.0;
#pragma unroll
        for (int k = NB - 1; k >= 0; --k) {
          if (k < nb) {
            x[k] *= dinv[kb + k];
#pragma unroll
            for (int r = 0; r < k; ++r) x[r] -= LU[(kb + r) * ld + kb + k] * x[k];
          }
        }
#pragma unroll
        for (int k = 0; k < NB; ++k)
          if (k < nb) Xs[(kb + k) * CB + tid] = x[k];
      }
      __syncthreads();
      if (kb > 0) update(kb, nb, 0, kb);
      __syncthreads();
    }
    for (int t = tid; t < n * CB; t += NTH) {
      const int r = t / CB, c = t % CB;
      if (c < nc) X[(int64_t)r * nt + c0 + c] = Xs[t];
    }
    // S[:, block] = D' - C' X
    const int nc8 = (nc + 7) / 8, nr4 = (nt + 3) / 4;
    for (int t = tid; t < nr4 * nc8; t += NTH) {
      const int r0 = 4 * (t / nc8), cc = 8 * (t % nc8);
      const double* Cr[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) Cr[a] = Cp + (int64_t)min(r0 + a, nt - 1) * n;
      double acc[4][8];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b)
          acc[a][b] = r0 + a < nt && cc + b < nc ? S[(int64_t)(r0 + a) * nt + c0 + cc + b] : 0.0;
      const int hi = cc + 4 < CB ? 4 : 0;  // the block's last four columns may be a tile of their own
#pragma unroll 2
      for (int k = 0; k < n; ++k) {
        double x[8];
#pragma unroll
        for (int b = 0; b < 8; b += 2) {
          const double2 u = *reinterpret_cast<const double2*>(Xs + k * CB + cc + (b < 4 ? b : b - 4 + hi));
          x[b] = u.x;
          x[b + 1] = u.y;
        }
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const double m = Cr[a][k];
#pragma unroll
          for (int b = 0; b < 8; ++b) acc[a][b] -= m * x[b];
        }
      }
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 8; ++b)
          if (r0 + a < nt && cc + b < nc) S[(int64_t)(r0 + a) * nt + c0 + cc + b] = acc[a][b];
    }
    __syncthreads();
  }
}

// The whole condensation: LU holds A' and R_v (column n) in shared or global memory; scratch ys [n].
template <int NTH, int CB>
HDG_DEVI bool element_condense(double* LU, int ld, int n, int* perm, double* dinv, double* ys, int* s_piv, double* Xs,
                               const double* Cp, const double* Rt, double* X, double* y, double* S, double* g, int nt) {
  const bool ok = element_lu<NTH>(LU, ld, n, perm, dinv, s_piv);
  element_solve_y<NTH>(LU, ld, n, dinv, ys, y);
  element_solve_schur<NTH, CB>(LU, ld, n, perm, dinv, Xs, Cp, X, S, nt);
  for (int r = threadIdx.x; r < nt; r += NTH) {  // g = R_t - C' y
    double s = Rt[r];
    const double* Cr = Cp + (int64_t)r * n;
    for (int k = 0; k < n; ++k) s -= Cr[k] * ys[k];
    g[r] = s;
  }
  return ok;
}

}  // namespace hdg
