// Plain FP64 assemble + condense (the reference GPU form of the hot path).
//
// Per element K the Newton linearisation of the local equations (Eq. hDG_NS1 / hDG1,
// with q eliminated exactly through Eq. hDG_NS0, which is linear in (q, v, vhat)) and
// of the element's share of the trace equation (Eq. hDG_NS2 / hDG2) is assembled as
//   A' = dR_v/dV, B' = dR_v/dVhat, C' = dR_t/dV, D' = dR_t/dVhat
// and condensed: X = A'^{-1} B', y = A'^{-1} R_v, S = D' - C' X, g = R_t - C' y.
// This equals the block elimination of the full [q; v] interior system in the order
// q first (the q-q block is the element mass matrix times the identity).
//
// Unknowns are grouped per state component into NZ "nodal" values z = [V (NP); Vhat
// (NF x NFN)]. At each quadrature point the value of v is Phi z and the lifted
// gradient is q_k = R_k z with
//   R_k(g, b)     = sum_r Jinv[r][k] dPhi_r(g, b) - sum_{f: b on f} n_fk s_f PL_f(g, c_f(b))
//   R_k(g, (f,c)) = n_fk s_f PL_f(g, c),  s_f = |F| / |K| (face / element Jacobians),
// PL_f = Phi Mref^{-1} E_f the lift of face f. Three kernels per chunk of elements:
//   k_pointwise  one thread per quadrature point: fluxes and exact pointwise Jacobians
//                by forward-mode dual numbers, pre-contracted with weights and Jinv;
//   k_assemble   one CTA per element: quadrature contractions into A', B', C', D', R
//                (element_fp64.cuh);
//   k_condense   one CTA per element: LU with partial pivoting of A' in shared memory,
//                triangular solves for X and y, Schur products for S and g.
#pragma once
#include "dfloat.cuh"
#include "element_fp64.cuh"
#include "hdg_device.cuh"

namespace hdg {

struct AssembleArgs {
  const double* V;      // [E][NP][M]
  const double* Vhat;   // [F][NFN][M]
  const int* tgidx;     // [E][NF][NFN] global face-node index
  const double* geo;    // [E][GEO]
  const double* hist;   // [E][NP][M] or null
  double mass_coef;
  int64_t e0, ne;       // element chunk
  // scratch (chunk-local)
  double* ptv;          // [ne][NG][PT_VOL]
  double* ptf;          // [ne][NF][NGF][PT_FACE]
  double* Ap;           // [ne][NV][NV]
  double* Cp;           // [ne][NT][NV]
  uint4* oz;            // [ne][...] exact-slice operands of the mixed condensation
  float* prep;          // [ne][...] inverse, FP32 copy and scales for the mixed condensation
  // outputs (global element index)
  double* S;            // [E][NT][NT]   (D' on entry to condense)
  double* g;            // [E][NT]
  double* recov;        // [E][NV*NT + NV]  X then y (B' on entry to condense)
  double* R;            // [E][NV + NT] raw residuals R_v, R_t (always written)
  int* status;          // [E]
  // With only_flag != 0 a CTA whose element has none of these status bits returns at once:
  // the FP64 kernels then recompute just the blocks the mixed form flagged, and k_condense
  // replaces the flag by HDG_STATUS_FP64 (the block is now the FP64 form's).
  int only_flag;
  float refine_tol;     // mixed condensation: tolerance of the refinement status bit
  int stall_first_copy; // test hooks (kStall*): the kernel never issues its first operand copy
};

enum { kStallCondense = 1, kStallAssembly = 2 };  // k_condense_t5; the first CTA of k_asm_t5
enum { HDG_STATUS_NONPHYSICAL = 1, HDG_STATUS_SINGULAR = 2, HDG_STATUS_REFINE = 4, HDG_STATUS_FP64 = 8,
       HDG_STATUS_TIMEOUT = 16 };

// true if the CTA of element e has nothing to do in a flagged-only pass
HDG_DEVI bool skip_element(const AssembleArgs& a, int64_t e) {
  return a.only_flag != 0 && (__ldg(a.status + e) & a.only_flag) == 0;
}

template <class C>
HDG_DEVI void load_element(const AssembleArgs& a, int64_t e, double (*z)[C::M], double* G) {
  constexpr int M = C::M;
  for (int t = threadIdx.x; t < C::NP * M; t += blockDim.x) z[t / M][t % M] = a.V[e * C::NV + t];
  for (int t = threadIdx.x; t < C::NF * C::NFN * M; t += blockDim.x) {
    int fc = t / M, i = t % M;
    int gi = a.tgidx[e * (C::NF * C::NFN) + fc];
    z[C::NP + fc][i] = a.Vhat[(int64_t)gi * M + i];
  }
  for (int t = threadIdx.x; t < C::GEO; t += blockDim.x) G[t] = a.geo[e * C::GEO + t];
}

// v_h and, for Navier-Stokes, the gradient q_h of Eq. hDG_NS0 solved element by element (the
// gradient of v_h plus the lifting of the face jumps vhat - v) at volume quadrature point g of the
// element staged in shared memory (z: nodal values, dz: jumps at the face nodes, G: geometry).
template <class C>
HDG_DEVI void volume_point_state(int g, const DevTables& T, const double (*z)[C::M], const double (*dz)[C::M],
                                 const double* G, double* v, double (*q)[C::D]) {
  constexpr int D = C::D, M = C::M, NP = C::NP, NFN = C::NFN, NF = C::NF, NG = C::NG;
  const double* Jinv = G;
  const double detJ = G[D * D];
  for (int i = 0; i < M; ++i) {
    double s = 0.0;
    for (int b = 0; b < NP; ++b) s += T.Phi[g * NP + b] * z[b][i];
    v[i] = s;
  }
  if (C::VISC) {
    for (int i = 0; i < M; ++i) {
      double gr[D], lift[NF];
      for (int r = 0; r < D; ++r) {
        double s = 0.0;
        for (int b = 0; b < NP; ++b) s += T.dPhi[(r * NG + g) * NP + b] * z[b][i];
        gr[r] = s;
      }
      for (int f = 0; f < NF; ++f) {  // the same for every direction k
        double l = 0.0;
        for (int c = 0; c < NFN; ++c) l += T.PL[(f * NG + g) * NFN + c] * dz[f * NFN + c][i];
        lift[f] = l;
      }
      for (int k = 0; k < D; ++k) {
        double s = 0.0;
        for (int r = 0; r < D; ++r) s += Jinv[r * D + k] * gr[r];
        for (int f = 0; f < NF; ++f) {
          const double* Gf = G + D * D + 1 + f * (D + 1);
          s += Gf[k] * (Gf[D] / detJ) * lift[f];
        }
        q[i][k] = s;
      }
    }
  }
}

// ------------------------------------------------------------------------------------
// k_pointwise
// ------------------------------------------------------------------------------------
HDG_DEVI void put(double* p, int i, double v) { p[i] = v; }
HDG_DEVI void put(df2* p, int i, double v) { p[i] = df_from(v); }

// Point tensors are stored [quantity][point] (element_fp64.cuh: the contractions read one quantity over
// the points); PtOut addresses those of one point.
template <int NPT>
struct PtOut {
  double* p;
  HDG_DEVI PtOut operator+(int i) const { return {p + i * NPT}; }
};
template <int NPT>
HDG_DEVI void put(const PtOut<NPT>& o, int i, double v) {
  o.p[i * NPT] = v;
}

// row r of Jinv, or the sum of the rows (r = D)
template <int D>
HDG_DEVI void jinv_row(const double* Jinv, int r, double* out) {
#pragma unroll
  for (int k = 0; k < D; ++k) {
    double s = 0.0;
#pragma unroll
    for (int q = 0; q < D; ++q) s += Jinv[q * D + k];
    out[k] = r < D ? Jinv[r * D + k] : s;
  }
}

// The values of sigma(vhat) = d(sigma (v - vhat))/dv at one face point, [row][column]:
// lambda_max A0 (Eq. sLxF) from the wave speed and u(vhat)'s derivatives, or |A_n| A0 (Eq. symStab)
// as a table.
template <int M, bool SYM>
struct SigmaValues {
  double lam;
  const Dual<M>* uh;
  HDG_DEVI double operator()(int i, int l) const { return lam * uh[i].d[l]; }
};
template <int M>
struct SigmaValues<M, true> {
  double s[M][M];
  HDG_DEVI double operator()(int i, int l) const { return s[i][l]; }
};

// SYM: sigma_S of Eq. symStab instead of sigma_SLF (launch through launch_pointwise).
template <class C, bool SYM = false>
__global__ void __launch_bounds__(128) k_pointwise(AssembleArgs a, DevTables T, PhysParams ph) {
  constexpr int D = C::D, M = C::M, NP = C::NP, NFN = C::NFN, NF = C::NF, NG = C::NG, NGF = C::NGF;
  __shared__ double z[C::NZ][M];
  __shared__ double G[C::GEO];
  __shared__ double dz[NF * NFN][M];  // vhat - v at the face nodes (the lifting's jumps)
  const int64_t le = blockIdx.x;
  const int64_t e = a.e0 + le;
  if (skip_element(a, e)) return;
  load_element<C>(a, e, z, G);
  __syncthreads();
  if (C::VISC)
    for (int t = threadIdx.x; t < NF * NFN * M; t += blockDim.x) {
      const int fc = t / M, i = t % M;
      dz[fc][i] = z[NP + fc][i] - z[T.fnodes[fc]][i];
    }
  __syncthreads();
  const double* Jinv = G;
  const double detJ = G[D * D];
  const int tid = threadIdx.x;
  bool bad = false;
  if (tid < NG) {
    const int g = tid;
    const double W = T.W[g] * detJ;
    double v[M];
    double q[M][D];
    volume_point_state<C>(g, T, z, dz, G, v, q);
    bad = !(v[M - 1] < 0.0);
    Dual<M> vd[M];
    for (int l = 0; l < M; ++l) {
      vd[l] = dconst<M>(v[l]);
      vd[l].d[l] = 1.0;
    }
    Dual<M> rho, vel[D], p, u[M], F[M][D];
    prim_of_v<D>(vd, ph.gamma, rho, vel, p);
    cons_and_flux<D>(rho, vel, p, ph.gamma, u, F);
    bad = bad || !(rho.v > 0.0) || !(p.v > 0.0);
    if (C::VISC) {
      Dual<M> Gv[M][D];
      visc_flux<D>(vd, q, ph, Gv);
      for (int i = 0; i < M; ++i)
        for (int j = 0; j < D; ++j) F[i][j] = F[i][j] + Gv[i][j];
    }
    using Pt = PtOut<NG>;
    const Pt MU{a.ptv + le * NG * C::PT_VOL + g};
    const Pt FR = MU + M, T0 = FR + D * M, T1 = T0 + M * M, T2 = T1 + D * M * M;
    for (int i = 0; i < M; ++i) {
      put(MU, i, W * a.mass_coef * u[i].v);
      for (int l = 0; l < M; ++l) put(T0, i * M + l, W * a.mass_coef * u[i].d[l]);
    }
    for (int r = 0; r < D; ++r)
      for (int i = 0; i < M; ++i) {
        double s = 0.0;
        for (int j = 0; j < D; ++j) s += Jinv[r * D + j] * F[i][j].v;
        put(FR, r * M + i, -W * s);
        for (int l = 0; l < M; ++l) {
          double t = 0.0;
          for (int j = 0; j < D; ++j) t += Jinv[r * D + j] * F[i][j].d[l];
          put(T1, (r * M + i) * M + l, -W * t);
        }
      }
    if (C::VISC) {
      // dG/dq contracted with the rows of Jinv on both sides (G is linear in q)
      const ViscFactors<D> vf = visc_factors<D>(v);
      const PhysParams pv = visc_params_at(ph, v[M - 1]);
#pragma unroll 1
      for (int rr = 0; rr < D * (D + 1); ++rr) {
        double c2[D];
        jinv_row<D>(Jinv, rr % (D + 1), c2);
        visc_jac_pair<D>(vf, Jinv + rr / (D + 1) * D, c2, pv, [&](int i, int l, double val) {
          put(T2, (rr * (M - 1) + i - 1) * (M - 1) + l - 1, -W * val);
        });
      }
    }
  } else if (tid < NG + NF * NGF) {
    const int f = (tid - NG) / NGF;
    const int gf = (tid - NG) % NGF;
    const double* Gf = G + D * D + 1 + f * (D + 1);
    const double* n = Gf;
    const double Wf = T.WF[gf] * Gf[D];
    const double* phif = T.PhiF + (f * NGF + gf) * NP;
    double v[M], vh[M];
    for (int i = 0; i < M; ++i) {
      double s = 0.0, sh = 0.0;
      for (int b = 0; b < NP; ++b) s += phif[b] * z[b][i];
      for (int c = 0; c < NFN; ++c) sh += phif[T.fnodes[f * NFN + c]] * z[NP + f * NFN + c][i];
      v[i] = s;
      vh[i] = sh;
    }
    double q[M][D];
    if (C::VISC) {
      for (int i = 0; i < M; ++i) {
        double gr[D], lift[NF];
        for (int r = 0; r < D; ++r) {
          double s = 0.0;
          for (int b = 0; b < NP; ++b) s += T.dPhiF[((f * D + r) * NGF + gf) * NP + b] * z[b][i];
          gr[r] = s;
        }
        for (int fl = 0; fl < NF; ++fl) {  // the same for every direction k
          double l = 0.0;
          for (int c = 0; c < NFN; ++c) l += T.PLF[((f * NF + fl) * NGF + gf) * NFN + c] * dz[fl * NFN + c][i];
          lift[fl] = l;
        }
        for (int k = 0; k < D; ++k) {
          double s = 0.0;
          for (int r = 0; r < D; ++r) s += Jinv[r * D + k] * gr[r];
          for (int fl = 0; fl < NF; ++fl) {
            const double* Gl = G + D * D + 1 + fl * (D + 1);
            s += Gl[k] * (Gl[D] / detJ) * lift[fl];
          }
          q[i][k] = s;
        }
      }
    }
    bad = !(v[M - 1] < 0.0) || !(vh[M - 1] < 0.0);
    // pass A: derivatives with respect to vhat
    Dual<M> vhd[M], dvd[M];
    for (int l = 0; l < M; ++l) {
      vhd[l] = dconst<M>(vh[l]);
      vhd[l].d[l] = 1.0;
      dvd[l] = v[l] - vhd[l];
    }
    Dual<M> rh, velh[D], prh, uh[M], Fh[M][D], duh[M];
    prim_of_v<D>(vhd, ph.gamma, rh, velh, prh);
    cons_and_flux<D>(rh, velh, prh, ph.gamma, uh, Fh);
    bad = bad || !(rh.v > 0.0) || !(prh.v > 0.0);
    du_of_v<D>(vhd, dvd, ph.gamma, duh);  // A0(vhat) (v - vhat)
    Dual<M> sdu[M];                        // sigma(vhat) (v - vhat)
    SigmaValues<M, SYM> sig;
    if constexpr (SYM) {  // sigma_S = |A_n| A0 (Eq. symStab)
      abs_flux_jac_apply<D>(rh, velh, prh, n, ph.gamma, duh, sdu);
      double vv[D];
      for (int j = 0; j < D; ++j) vv[j] = velh[j].v;
      for (int l = 0; l < M; ++l) {
        double x[M], y[M];
        for (int k = 0; k < M; ++k) x[k] = uh[k].d[l];
        abs_flux_jac_apply<D>(rh.v, vv, prh.v, n, ph.gamma, x, y);
        for (int i = 0; i < M; ++i) sig.s[i][l] = y[i];
      }
    } else {  // sigma_SLF = lambda_max A0 (Eq. sLxF)
      const Dual<M> lam = lambda_max<D>(rh, velh, prh, n, ph.gamma);
      for (int i = 0; i < M; ++i) sdu[i] = lam * duh[i];
      sig.lam = lam.v;
      sig.uh = uh;
    }
    Dual<M> hA[M];
    for (int i = 0; i < M; ++i) {
      Dual<M> s = Fh[i][0] * n[0];
      for (int j = 1; j < D; ++j) s = s + Fh[i][j] * n[j];
      hA[i] = 0.5 * s + 0.5 * sdu[i];
    }
    if (C::VISC && ph.gflux != 1) {  // ghat = G(vhat, q) . n (Eq. numericalFluxNS_2)
      Dual<M> Gh[M][D];
      visc_flux<D>(vhd, q, ph, Gh);
      for (int i = 0; i < M; ++i)
        for (int j = 0; j < D; ++j) hA[i] = hA[i] + Gh[i][j] * n[j];
    }
    // pass B: derivatives with respect to v (F(v).n; the sigma term gives sigma(vhat))
    Dual<M> vd[M];
    for (int l = 0; l < M; ++l) {
      vd[l] = dconst<M>(v[l]);
      vd[l].d[l] = 1.0;
    }
    Dual<M> rv, velv[D], pv, Fv[M][D];
    prim_of_v<D>(vd, ph.gamma, rv, velv, pv);
    cons_and_flux<D>(rv, velv, pv, ph.gamma, (Dual<M>*)nullptr, Fv);
    bad = bad || !(rv.v > 0.0) || !(pv.v > 0.0);
    using Pt = PtOut<NF * NGF>;
    const Pt HF{a.ptf + le * NF * NGF * C::PT_FACE + f * NGF + gf};
    const Pt U0 = HF + M, U1 = U0 + M * M, U2 = U1 + M * M;
    Dual<M> gn[M];  // ghat = G(v, q) . n (Eq. numericalFluxNS_1): value and d/dv
    for (int i = 0; i < M; ++i) gn[i] = vd[0] * 0.0;
    if (C::VISC && ph.gflux == 1) {
      Dual<M> Gv[M][D];
      visc_flux<D>(vd, q, ph, Gv);
      for (int i = 0; i < M; ++i)
        for (int j = 0; j < D; ++j) gn[i] = gn[i] + Gv[i][j] * n[j];
    }
    for (int i = 0; i < M; ++i) {
      Dual<M> s = Fv[i][0] * n[0];
      for (int j = 1; j < D; ++j) s = s + Fv[i][j] * n[j];
      put(HF, i, Wf * (hA[i].v + 0.5 * s.v + gn[i].v));
      for (int l = 0; l < M; ++l) {
        put(U0, i * M + l, Wf * (0.5 * s.d[l] + 0.5 * sig(i, l) + gn[i].d[l]));
        put(U1, i * M + l, Wf * hA[i].d[l]);
      }
    }
    if (C::VISC) {  // dG/dq contracted with the normal, at the state the viscous flux uses
      const double* vs = ph.gflux == 1 ? v : vh;
      const ViscFactors<D> vf = visc_factors<D>(vs);
      const PhysParams pvs = visc_params_at(ph, vs[M - 1]);
#pragma unroll 1
      for (int r = 0; r <= D; ++r) {
        double c2[D];
        jinv_row<D>(Jinv, r, c2);
        visc_jac_pair<D>(vf, n, c2, pvs, [&](int i, int l, double val) {
          put(U2, (r * (M - 1) + i - 1) * (M - 1) + l - 1, Wf * val);
        });
      }
    }
  }
  if (bad) atomicOr(a.status + e, HDG_STATUS_NONPHYSICAL);
}

// k_pointwise with the stabilization matrix the physics selects
template <class C>
void launch_pointwise(const AssembleArgs& a, const DevTables& T, const PhysParams& ph, cudaStream_t s) {
  const int threads = ((C::NG + C::NF * C::NGF + 31) / 32) * 32;
  if (ph.stab == 1)
    k_pointwise<C, true><<<(unsigned)a.ne, threads, 0, s>>>(a, T, ph);
  else
    k_pointwise<C, false><<<(unsigned)a.ne, threads, 0, s>>>(a, T, ph);
}

// ------------------------------------------------------------------------------------
// k_assemble: one CTA per element (element_blocks), several per SM
// ------------------------------------------------------------------------------------
template <class C>
struct UniformDims {
  static constexpr int pad(int n) { return (n + 1) / 2 * 2; }
  static constexpr int NP = C::NP, NG = C::NG, NGF = C::NGF, NTN = C::NF * C::NFN, NV = C::NV, NT = C::NT;
  static constexpr int NPs = pad(C::NP), NZs = NPs + C::NF * pad(C::NFN);
};

template <class C>
struct AsmSmem {
  static constexpr int NTH = C::D == 3 && C::P >= 2 ? 256 : 128;
  // tiles of one operator: A' and one face's block of B'
  static constexpr int TILES = UniformDims<C>::NPs / 2 * (UniformDims<C>::NPs / 2 + (C::VISC ? (C::NFN + 1) / 2 : 0));
  static constexpr int NRD = (TILES + NTH - 1) / NTH;
  static constexpr int MINB = NTH == 256 ? 3 : 5;  // registers: 80 a thread
  static constexpr size_t bytes = sizeof(double) * element_smem_doubles(UniformDims<C>(), C::NF, 2);
};

// the reference operators of an element of one degree, filled in by one thread
template <class C>
HDG_DEVI void uniform_tables(const DevTables& T, ElemTables<C::D>& E) {
  constexpr int NF = C::NF, NFN = C::NFN, NG = C::NG, NGF = C::NGF;
  E.Phi = T.Phi;
  E.dPhi = T.dPhi;
  E.dR = T.dR;
  E.PhiF = T.PhiF;
  E.dRF = T.dRF;
  E.nodepos = T.nodepos;
  for (int f = 0; f < NF; ++f) {
    E.Psi[f] = T.Psi + f * NGF * NFN;
    E.PL[f] = T.PL + f * NG * NFN;
    E.PLF[f] = T.PLF + f * NGF * NFN;
    E.sPLF[f] = NF * NGF * NFN;
    E.Tr[f] = nullptr;
    E.nq[f] = NFN;
  }
  for (int f = 0; f <= NF; ++f) {
    E.off[f] = f * NFN;
    E.offp[f] = f * ((NFN + 1) / 2 * 2);
  }
}

template <class C>
__global__ void __launch_bounds__(AsmSmem<C>::NTH, AsmSmem<C>::MINB) k_assemble(AssembleArgs a, DevTables T) {
  constexpr int D = C::D, NF = C::NF, NG = C::NG, NGF = C::NGF, NV = C::NV, NT = C::NT, NTH = AsmSmem<C>::NTH;
  extern __shared__ __align__(16) double smem[];
  __shared__ ElemTables<D> E;
  const int64_t le = blockIdx.x;
  const int64_t e = a.e0 + le;
  if (skip_element(a, e)) return;
  if (threadIdx.x == 0) uniform_tables<C>(T, E);
  __syncthreads();
  const double* ptv = a.ptv + le * NG * C::PT_VOL;
  const double* ptf = a.ptf + le * NF * NGF * C::PT_FACE;
  double* R = a.R + e * (int64_t)(NV + NT);
  const UniformDims<C> d;
  element_residual<D, NTH>(d, E, ptv, ptf, a.hist ? a.hist + e * NV : nullptr, R, R + NV);
  element_blocks<D, C::VISC, NTH, AsmSmem<C>::NRD, NF, 2>(d, E, ptv, ptf, a.Ap + le * NV * NV,
                                                   a.recov + e * (int64_t)(NV * NT + NV), a.Cp + le * NT * NV,
                                                   a.S + e * (int64_t)NT * NT, smem);
}

// ------------------------------------------------------------------------------------
// k_condense: one CTA per element, LU in shared memory (two CTAs per SM at 3D p = 3)
// ------------------------------------------------------------------------------------
template <class C>
struct CondSmem {
  static constexpr int NTH = C::NV <= 24 ? 64 : C::NV <= 64 ? 128 : 256;
  // right-hand-side columns per block: all of them, or 40 (a divisor of 3D's 120 and 200; the most that
  // lets two CTAs share an SM at p = 3)
  static constexpr int CB = C::NT <= 60 ? (C::NT + 3) / 4 * 4 : 40;
  static constexpr int LD = C::NV % 2 ? C::NV + 2 : C::NV + 1;  // odd (a column's entries lie in different banks), > NV
  static constexpr int LUN = (C::NV * LD + 1) / 2 * 2;
  static constexpr size_t bytes = sizeof(double) * (LUN + C::NV * CB + 2 * C::NV) + sizeof(int) * C::NV;
};

template <class C>
__global__ void __launch_bounds__(CondSmem<C>::NTH, 512 / CondSmem<C>::NTH) k_condense(AssembleArgs a) {
  constexpr int NV = C::NV, NT = C::NT;
  using SM = CondSmem<C>;
  extern __shared__ __align__(16) double smem[];
  double* LU = smem;                 // [NV][LD]: A' and R_v
  double* Xs = LU + SM::LUN;         // [NV][CB]
  double* dinv = Xs + NV * SM::CB;   // [NV]
  double* ys = dinv + NV;            // [NV]
  int* perm = reinterpret_cast<int*>(ys + NV);
  __shared__ int s_piv[2];
  const int64_t le = blockIdx.x;
  const int64_t e = a.e0 + le;
  if (skip_element(a, e)) return;
  const int tid = threadIdx.x;
  const double* Ap = a.Ap + le * NV * NV;
  const double* R = a.R + e * (int64_t)(NV + NT);
  double* X = a.recov + e * (int64_t)(NV * NT + NV);
  for (int t = tid; t < NV * NV; t += SM::NTH) LU[t / NV * SM::LD + t % NV] = Ap[t];
  for (int t = tid; t < NV; t += SM::NTH) LU[t * SM::LD + NV] = R[t];
  __syncthreads();
  const bool ok = element_condense<SM::NTH, SM::CB>(LU, SM::LD, NV, perm, dinv, ys, s_piv, Xs, a.Cp + le * NT * NV,
                                                    R + NV, X, X + NV * NT, a.S + e * (int64_t)NT * NT,
                                                    a.g + e * NT, NT);
  if (tid == 0 && !ok) atomicOr(a.status + e, HDG_STATUS_SINGULAR);
  if (a.only_flag != 0 && tid == 0) {  // flagged-only pass: the block is now the FP64 form's
    atomicAnd(a.status + e, ~a.only_flag);
    atomicOr(a.status + e, HDG_STATUS_FP64);
  }
}

// ------------------------------------------------------------------------------------
// k_entropy_terms: the two integrals of Eq. PiS (Sec. 5.6) from (v_h, q_h), one CTA per element:
//   acc[0] += int_K rho s,  s = log(p / rho^gamma) (Sec. 2.3)
//   acc[1] += (1/c_v) int_K (Phi / T + kappa |grad T|^2 / T^2),  Phi = grad V : tau
// ------------------------------------------------------------------------------------
template <class C>
__global__ void __launch_bounds__(128) k_entropy_terms(AssembleArgs a, DevTables T, PhysParams ph, double* acc) {
  constexpr int D = C::D, M = C::M, NP = C::NP, NFN = C::NFN, NF = C::NF, NG = C::NG;
  __shared__ double z[C::NZ][M];
  __shared__ double G[C::GEO];
  __shared__ double dz[NF * NFN][M];
  __shared__ double red[2][4];
  const int64_t e = a.e0 + blockIdx.x;
  load_element<C>(a, e, z, G);
  __syncthreads();
  for (int t = threadIdx.x; t < NF * NFN * M; t += blockDim.x) {
    const int fc = t / M, i = t % M;
    dz[fc][i] = z[NP + fc][i] - z[T.fnodes[fc]][i];
  }
  __syncthreads();
  double rs = 0.0, pr = 0.0;
  for (int g = threadIdx.x; g < NG; g += blockDim.x) {
    const double W = T.W[g] * G[D * D];
    double v[M], q[M][D];
    volume_point_state<C>(g, T, z, dz, G, v, q);
    double rho, vel[D], p;
    prim_of_v<D>(v, ph.gamma, rho, vel, p);
    rs += W * rho * (::log(p) - ph.gamma * ::log(rho));
    if (C::VISC) {
      const double vm = v[M - 1], ivm = 1.0 / vm, Temp = -ivm / ph.cv;
      const double fac = ph.mu_exp != 0.0 ? ::exp(-ph.mu_exp * ::log(ph.cv * (-vm))) : 1.0;
      const double mu = ph.mu * fac, kappa = ph.kappa * fac;
      double gV[D][D], gT2 = 0.0, div = 0.0;
      for (int i = 0; i < D; ++i)
        for (int j = 0; j < D; ++j) gV[i][j] = v[1 + i] * ivm * ivm * q[M - 1][j] - q[1 + i][j] * ivm;
      for (int j = 0; j < D; ++j) {
        const double gt = q[M - 1][j] * ivm * ivm / ph.cv;
        gT2 += gt * gt;
        div += gV[j][j];
      }
      double Phi = 0.0;
      for (int i = 0; i < D; ++i)
        for (int j = 0; j < D; ++j) {
          const double tau = mu * (gV[i][j] + gV[j][i] - (i == j ? (2.0 / 3.0) * div : 0.0));
          Phi += gV[i][j] * tau;
        }
      pr += W * (Phi / Temp + kappa * gT2 / (Temp * Temp)) / ph.cv;
    }
  }
  for (int off = 16; off > 0; off >>= 1) {
    rs += __shfl_xor_sync(0xffffffffu, rs, off);
    pr += __shfl_xor_sync(0xffffffffu, pr, off);
  }
  const int warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  if ((threadIdx.x & 31) == 0) {
    red[0][warp] = rs;
    red[1][warp] = pr;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double s0 = 0.0, s1 = 0.0;
    for (int w = 0; w < nw; ++w) {
      s0 += red[0][w];
      s1 += red[1][w];
    }
    atomicAdd(acc, s0);
    atomicAdd(acc + 1, s1);
  }
}

}  // namespace hdg
