// Mixed-degree assemble + condense (FP64): every element of a mesh whose elements differ in
// degree, in ONE persistent launch over a work queue ordered by element class.
//
// The paper uses one degree k everywhere; elements of different degree in one mesh are this
// library's extension (a mesh with p_per_elem). Element e has degree pk = p_e; the trace on a face
// has the larger degree of its two sides, q_F = max(p_L, p_R); the element's trace degree pt is
// the largest of its faces' degrees. An element class is the pair (pk, pt), pt >= pk; 3D
// Navier-Stokes has ten classes (pk, pt in 1..4).
//
// Per element the kernel runs the steps of the uniform FP64 form:
//   1. gather vhat at the face's own nodes (degree q_f) and prolong it to the degree-pt nodes,
//      vhat_pt = I_f vhat_q (exact: P_q is contained in P_pt);
//   2. pointwise fluxes and exact pointwise Jacobians (dual numbers) at the volume points (rule
//      with pk + 1 points per direction) and face points (pt + 1), into per-CTA scratch;
//   3. the quadrature contractions (element_fp64.cuh) with the trace functions of every face's own
//      degree q_f, so that A', B_q, C_q, D_q come out in the element's own trace space;
//   4. LU of A' (in shared memory when it fits, else in the CTA's global-memory scratch),
//      X = A'^{-1} [B_q | R_v], S = D_q - C_q X, g = R_t,q - C_q y.
// Outputs are packed per element at the offsets of the mesh layout (hdg_mesh_copy_layout):
// S [nt_e][nt_e], g [nt_e], recov [nv_e nt_e + nv_e] (X then y), R [nv_e + nt_e], with
// nt_e = sum_f Nf(q_f) m the element's own trace unknowns in [face][face node][component] order.
//
// Bound: the FP64 pipe (a p = 4 element is 27M FMA in the condensation alone). 3,072 tetrahedra with
// degrees drawn 0.1/0.3/0.4/0.2: 346.8 -> 111.3 ms with the contraction in the faces' own spaces and the
// blocked condensation of element_fp64.cuh, which leave no tile shape to tune (the first call was 3.0 s).
//
// The launch is persistent: two CTAs of 256 threads per SM (one hides the other's barriers); thread 0 takes the next queue entry with an atomic counter, the queue lists the
// elements largest class first (longest work first), and one code path serves every class, reading
// the class's sizes and tables at run time. A 3D mesh of the single degree 4, which has no uniform
// kernels, runs here as the class (4, 4).
#include <algorithm>
#include <cstring>
#include <vector>

#include "assemble_fp64.cuh"
#include "ctx.hpp"
#include "pclass.hpp"

namespace hdg {

namespace {

// Sizes of one class (pk, pt), 3D Navier-Stokes: computed on the host, read by the kernel at run
// time (one code path serves every class, so the launch compiles once).
constexpr int D3 = 3, M5 = 5, NF4 = 4, GEO3 = D3 * D3 + 1 + NF4 * (D3 + 1);
// point tensors (element_fp64.cuh)
constexpr int PT_VOL = M5 + D3 * M5 + M5 * M5 + D3 * M5 * M5 + D3 * (D3 + 1) * (M5 - 1) * (M5 - 1);
constexpr int PT_FACE = M5 + 2 * M5 * M5 + (D3 + 1) * (M5 - 1) * (M5 - 1);
constexpr int kLuSmemMax = 100;  // A' factored in shared memory up to this interior size (p = 3)
constexpr int kCB = 40;          // right-hand sides per block of the condensation

HDG_DEVI constexpr int even(int n) { return (n + 1) / 2 * 2; }

// sizes of one element's contraction: its class's and its own faces' trace nodes
struct ElemDims {
  int NP, NG, NGF, NTN, NPs, NZs, NV, NT;
};

inline PDims pclass_dims(int pk, int pt) {
  PDims d{};
  d.pk = pk;
  d.pt = pt;
  d.NP = (pk + 1) * (pk + 2) * (pk + 3) / 6;
  d.NFK = (pk + 1) * (pk + 2) / 2;
  d.NFN = (pt + 1) * (pt + 2) / 2;
  d.NG = (pk + 1) * (pk + 1) * (pk + 1);
  d.NGF = (pt + 1) * (pt + 1);
  d.NV = d.NP * M5;
  d.NT = NF4 * d.NFN * M5;
  d.NZ = d.NP + NF4 * d.NFN;
  // shared memory: the element's state while the point tensors form, then the contraction's buffers
  // (every face of the widest degree), then the factors and a block of right-hand sides
  auto ev = [](int n) { return (n + 1) / 2 * 2; };
  const ElemDims e{d.NP, d.NG, d.NGF, NF4 * d.NFN, ev(d.NP), ev(d.NP) + NF4 * ev(d.NFN), d.NV, d.NT};
  const int state = d.NZ * M5 + GEO3 + NF4 * d.NFN * M5;
  const int ld = d.NV % 2 ? d.NV + 2 : d.NV + 1;
  const int lu = ev(d.NV * ld);
  const int cond = (d.NV <= kLuSmemMax ? lu : 0) + d.NV * kCB + 2 * d.NV + (d.NV + 1) / 2;
  d.SMEM = std::max(std::max(state, element_smem_doubles(e, 1, 1)), cond);
  d.SLOT = (int64_t)d.NG * PT_VOL + (int64_t)NF4 * d.NGF * PT_FACE + (int64_t)d.NV * d.NT +
           (int64_t)ev(d.NV * d.NV) + (d.NV <= kLuSmemMax ? 0 : lu) + 8;
  return d;
}

constexpr int kThreads = 256;

struct PArgs {
  const double* V;       // element e's [NP_e][M] at V + voff[e]
  const double* Vhat;    // [trace nodes][M]
  const double* hist;    // like V, or null
  double mass_coef;
  const int64_t* voff;   // [E + 1]
  const int64_t* toff;   // [E + 1] trace unknowns nt_e (g)
  const int64_t* soff;   // [E + 1] nt_e^2 (S)
  const int64_t* roff;   // [E + 1] nv_e nt_e + nv_e (recov)
  const int64_t* Roff;   // [E + 1] nv_e + nt_e (R)
  const int* tgidx;      // [E][NF][nfn_max] trace node of each local face node (-1 beyond)
  const int8_t* fdeg;    // [E][NF] degree of each face of the element
  const int8_t* cls;     // [E] class index
  const double* geo;     // [E][GEO]
  const int* queue;      // [E] elements, largest class first
  int64_t E;
  int nfn_max;
  int64_t slot_doubles;
  int* counter;          // work counter (zeroed before the launch)
  double* scratch;       // [grid][slot_doubles]
  double* S;
  double* g;
  double* recov;
  double* R;
  int* status;
  PClassDev tab[kPClasses];
};

HDG_DEVI int nfn3(int q) { return (q + 1) * (q + 2) / 2; }

// ----------------------------------------------------------------------------------- step 2
// One thread per quadrature point: fluxes and exact pointwise Jacobians by dual numbers,
// pre-contracted with the weights and Jinv (the per-point tensors of k_pointwise, FP64).
__device__ void pc_pointwise(const PArgs& a, const PClassDev& T, const PhysParams& ph, const double (*z)[M5],
                             const double (*dz)[M5], const double* G, double* ptv, double* ptf, int64_t e) {
  constexpr int D = D3, M = M5, NF = NF4;
  const int NP = T.d.NP, NFN = T.d.NFN, NG = T.d.NG, NGF = T.d.NGF;
  const double* Jinv = G;
  const double detJ = G[D * D];
  const int tid = threadIdx.x;
  bool bad = false;
  // q at a point from its element-gradient part gr[i][r] and the lifts of the face jumps
  auto lifted_q = [&](const double (*gr)[D], const double (*lift)[NF], double (*q)[D]) {
    for (int i = 0; i < M; ++i)
      for (int k = 0; k < D; ++k) {
        double s = 0.0;
        for (int r = 0; r < D; ++r) s += Jinv[r * D + k] * gr[i][r];
        for (int f = 0; f < NF; ++f) {
          const double* Gf = G + D * D + 1 + f * (D + 1);
          s += Gf[k] * (Gf[D] / detJ) * lift[i][f];
        }
        q[i][k] = s;
      }
  };
  if (tid < NG) {
    const int g = tid;
    const double W = T.W[g] * detJ;
    double v[M], gr[M][D], lift[M][NF], q[M][D];
    for (int i = 0; i < M; ++i) {
      double s = 0.0;
      for (int b = 0; b < NP; ++b) s += T.Phi[g * NP + b] * z[b][i];
      v[i] = s;
      for (int r = 0; r < D; ++r) {
        double t = 0.0;
        for (int b = 0; b < NP; ++b) t += T.dPhi[(r * NG + g) * NP + b] * z[b][i];
        gr[i][r] = t;
      }
      for (int f = 0; f < NF; ++f) {
        double l = 0.0;
        for (int c = 0; c < NFN; ++c) l += T.PL[(f * NG + g) * NFN + c] * dz[f * NFN + c][i];
        lift[i][f] = l;
      }
    }
    lifted_q(gr, lift, q);
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
    {
      Dual<M> Gv[M][D];
      visc_flux<D>(vd, q, ph, Gv);
      for (int i = 0; i < M; ++i)
        for (int j = 0; j < D; ++j) F[i][j] = F[i][j] + Gv[i][j];
    }
    double* MU = ptv + g;
    double* FR = MU + M * NG;
    double* T0 = FR + D * M * NG;
    double* T1 = T0 + M * M * NG;
    double* T2 = T1 + D * M * M * NG;
    for (int i = 0; i < M; ++i) {
      MU[i * NG] = W * a.mass_coef * u[i].v;
      for (int l = 0; l < M; ++l) T0[(i * M + l) * NG] = W * a.mass_coef * u[i].d[l];
    }
    for (int r = 0; r < D; ++r)
      for (int i = 0; i < M; ++i) {
        double s = 0.0;
        for (int j = 0; j < D; ++j) s += Jinv[r * D + j] * F[i][j].v;
        FR[(r * M + i) * NG] = -W * s;
        for (int l = 0; l < M; ++l) {
          double t = 0.0;
          for (int j = 0; j < D; ++j) t += Jinv[r * D + j] * F[i][j].d[l];
          T1[((r * M + i) * M + l) * NG] = -W * t;
        }
      }
    const ViscFactors<D> vf = visc_factors<D>(v);
    const PhysParams pv = visc_params_at(ph, v[M - 1]);
#pragma unroll 1
    for (int rr = 0; rr < D * (D + 1); ++rr) {
      double c2[D];
      jinv_row<D>(Jinv, rr % (D + 1), c2);
      visc_jac_pair<D>(vf, Jinv + rr / (D + 1) * D, c2, pv, [&](int i, int l, double val) {
        T2[((rr * (M - 1) + i - 1) * (M - 1) + l - 1) * NG] = -W * val;
      });
    }
  } else if (tid < NG + NF * NGF) {
    const int f = (tid - NG) / NGF;
    const int gf = (tid - NG) % NGF;
    const double* Gf = G + D * D + 1 + f * (D + 1);
    const double* n = Gf;
    const double Wf = T.WF[gf] * Gf[D];
    const double* phif = T.PhiF + (f * NGF + gf) * NP;
    const double* psif = T.PsiF + (f * NGF + gf) * NFN;
    double v[M], vh[M], gr[M][D], lift[M][NF], q[M][D];
    for (int i = 0; i < M; ++i) {
      double s = 0.0, sh = 0.0;
      for (int b = 0; b < NP; ++b) s += phif[b] * z[b][i];
      for (int c = 0; c < NFN; ++c) sh += psif[c] * z[NP + f * NFN + c][i];
      v[i] = s;
      vh[i] = sh;
      for (int r = 0; r < D; ++r) {
        double t = 0.0;
        for (int b = 0; b < NP; ++b) t += T.dPhiF[((f * D + r) * NGF + gf) * NP + b] * z[b][i];
        gr[i][r] = t;
      }
      for (int fl = 0; fl < NF; ++fl) {
        double l = 0.0;
        for (int c = 0; c < NFN; ++c) l += T.PLF[((f * NF + fl) * NGF + gf) * NFN + c] * dz[fl * NFN + c][i];
        lift[i][fl] = l;
      }
    }
    lifted_q(gr, lift, q);
    bad = !(v[M - 1] < 0.0) || !(vh[M - 1] < 0.0);
    // derivatives with respect to vhat: F(vhat).n, sigma(vhat) (v - vhat), G(vhat, q).n
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
    du_of_v<D>(vhd, dvd, ph.gamma, duh);
    // sigma(vhat) (v - vhat) and the matrix sigma(vhat) = d(sigma (v - vhat))/dv: sigma_SLF =
    // lambda_max A0 (Eq. sLxF) or sigma_S = |A_n| A0 (Eq. symStab), as physics selects
    Dual<M> sdu[M];
    double sig[M][M];
    if (ph.stab == 1) {
      abs_flux_jac_apply<D>(rh, velh, prh, n, ph.gamma, duh, sdu);
      double vv[D];
      for (int j = 0; j < D; ++j) vv[j] = velh[j].v;
      for (int l = 0; l < M; ++l) {
        double x[M], y[M];
        for (int k = 0; k < M; ++k) x[k] = uh[k].d[l];
        abs_flux_jac_apply<D>(rh.v, vv, prh.v, n, ph.gamma, x, y);
        for (int i = 0; i < M; ++i) sig[i][l] = y[i];
      }
    } else {
      const Dual<M> lam = lambda_max<D>(rh, velh, prh, n, ph.gamma);
      for (int i = 0; i < M; ++i) {
        sdu[i] = lam * duh[i];
        for (int l = 0; l < M; ++l) sig[i][l] = lam.v * uh[i].d[l];
      }
    }
    Dual<M> hA[M];
    for (int i = 0; i < M; ++i) {
      Dual<M> s = Fh[i][0] * n[0];
      for (int j = 1; j < D; ++j) s = s + Fh[i][j] * n[j];
      hA[i] = 0.5 * s + 0.5 * sdu[i];
    }
    if (ph.gflux != 1) {  // ghat = G(vhat, q) . n (Eq. numericalFluxNS_2)
      Dual<M> Gh[M][D];
      visc_flux<D>(vhd, q, ph, Gh);
      for (int i = 0; i < M; ++i)
        for (int j = 0; j < D; ++j) hA[i] = hA[i] + Gh[i][j] * n[j];
    }
    // derivatives with respect to v: F(v).n; the sigma term gives sigma(vhat)
    Dual<M> vd[M];
    for (int l = 0; l < M; ++l) {
      vd[l] = dconst<M>(v[l]);
      vd[l].d[l] = 1.0;
    }
    Dual<M> rv, velv[D], pv, Fv[M][D];
    prim_of_v<D>(vd, ph.gamma, rv, velv, pv);
    cons_and_flux<D>(rv, velv, pv, ph.gamma, (Dual<M>*)nullptr, Fv);
    bad = bad || !(rv.v > 0.0) || !(pv.v > 0.0);
    Dual<M> gn[M];  // ghat = G(v, q) . n (Eq. numericalFluxNS_1)
    for (int i = 0; i < M; ++i) gn[i] = vd[0] * 0.0;
    if (ph.gflux == 1) {
      Dual<M> Gv[M][D];
      visc_flux<D>(vd, q, ph, Gv);
      for (int i = 0; i < M; ++i)
        for (int j = 0; j < D; ++j) gn[i] = gn[i] + Gv[i][j] * n[j];
    }
    const int NQ = NF * NGF;
    double* HF = ptf + f * NGF + gf;
    double* U0 = HF + M * NQ;
    double* U1 = U0 + M * M * NQ;
    double* U2 = U1 + M * M * NQ;
    for (int i = 0; i < M; ++i) {
      Dual<M> s = Fv[i][0] * n[0];
      for (int j = 1; j < D; ++j) s = s + Fv[i][j] * n[j];
      HF[i * NQ] = Wf * (hA[i].v + 0.5 * s.v + gn[i].v);
      for (int l = 0; l < M; ++l) {
        U0[(i * M + l) * NQ] = Wf * (0.5 * s.d[l] + 0.5 * sig[i][l] + gn[i].d[l]);
        U1[(i * M + l) * NQ] = Wf * hA[i].d[l];
      }
    }
    const double* vs = ph.gflux == 1 ? v : vh;
    const ViscFactors<D> vf = visc_factors<D>(vs);
    const PhysParams pvs = visc_params_at(ph, vs[M - 1]);
#pragma unroll 1
    for (int r = 0; r <= D; ++r) {
      double c2[D];
      jinv_row<D>(Jinv, r, c2);
      visc_jac_pair<D>(vf, n, c2, pvs, [&](int i, int l, double val) {
        U2[((r * (M - 1) + i - 1) * (M - 1) + l - 1) * NQ] = Wf * val;
      });
    }
  }
  if (bad) atomicOr(a.status + e, HDG_STATUS_NONPHYSICAL);
}

// ----------------------------------------------------------------------------------- one element
__device__ void pc_element(const PArgs& a, const PClassDev& T, const PhysParams& ph, int64_t e, double* sm,
                           double* slot, ElemTables<D3>& E, int* s_piv) {
  constexpr int M = M5, NF = NF4;
  const int NP = T.d.NP, NFN = T.d.NFN, NV = T.d.NV, NZ = T.d.NZ;
  const int tid = threadIdx.x, nth = kThreads;
  double(*z)[M] = reinterpret_cast<double(*)[M]>(sm);
  double* G = sm + NZ * M;
  double(*dz)[M] = reinterpret_cast<double(*)[M]>(G + GEO3);
  double* ptv = slot;
  double* ptf = ptv + (int64_t)T.d.NG * PT_VOL;
  double* Ap = ptf + (int64_t)NF * T.d.NGF * PT_FACE;
  double* Cp = Ap + even(NV * NV);
  double* LUg = Cp + (int64_t)NV * T.d.NT;
  if (tid == 0) {  // the element's reference operators: its class's, and every face's of its own degree
    E.Phi = T.Phi;
    E.dPhi = T.dPhi;
    E.dR = T.dR;
    E.PhiF = T.PhiF;
    E.dRF = T.dRF;
    E.nodepos = T.nodepos;
    E.off[0] = E.offp[0] = 0;
    for (int f = 0; f < NF; ++f) {
      const int q = a.fdeg[e * NF + f], n = nfn3(q);
      E.nq[f] = n;
      E.off[f + 1] = E.off[f] + n;
      E.offp[f + 1] = E.offp[f] + even(n);
      E.Psi[f] = T.PsiQ[q - 1] + f * T.d.NGF * n;
      E.PL[f] = T.PLQ[q - 1] + f * T.d.NG * n;
      E.PLF[f] = T.PLFQ[q - 1] + f * NF * T.d.NGF * n;
      E.sPLF[f] = T.d.NGF * n;
      E.Tr[f] = q == T.d.pk ? nullptr : T.TrQ[q - 1] + f * n * NP;
    }
  }
  // 1. element state; the trace at the degree-pt nodes
  const double* Ve = a.V + a.voff[e];
  for (int t = tid; t < NP * M; t += nth) z[t / M][t % M] = Ve[t];
  for (int t = tid; t < NF * NFN * M; t += nth) {
    const int f = t / (NFN * M), c = (t / M) % NFN, i = t % M;
    const int q = a.fdeg[e * NF + f];
    const int* tg = a.tgidx + (e * NF + f) * a.nfn_max;
    double val;
    if (q == T.d.pt) {
      val = a.Vhat[(int64_t)tg[c] * M + i];
    } else {
      const double* I = T.IPro + ((size_t)(q - 1) * NF + f) * NFN * NFN;
      val = 0.0;
      for (int cq = 0; cq < nfn3(q); ++cq) val += I[c * NFN + cq] * a.Vhat[(int64_t)tg[cq] * M + i];
    }
    z[NP + f * NFN + c][i] = val;
  }
  for (int t = tid; t < GEO3; t += nth) G[t] = a.geo[e * GEO3 + t];
  __syncthreads();
  for (int t = tid; t < NF * NFN * M; t += nth) {
    const int fc = t / M, i = t % M;
    double s = 0.0;
    for (int b = 0; b < NP; ++b) s += T.PhiN[fc * NP + b] * z[b][i];
    dz[fc][i] = z[NP + fc][i] - s;
  }
  __syncthreads();
  // 2. pointwise
  pc_pointwise(a, T, ph, z, dz, G, ptv, ptf, e);
  __syncthreads();
  // 3. contractions in the element's own trace space: B_q into X, D_q into S
  const int ntn = E.off[NF], ntq = ntn * M;
  const ElemDims d{NP, T.d.NG, T.d.NGF, ntn, even(NP), even(NP) + E.offp[NF], NV, ntq};
  double* X = a.recov + a.roff[e];
  double* S = a.S + a.soff[e];
  double* Re = a.R + a.Roff[e];
  element_residual<D3, kThreads>(d, E, ptv, ptf, a.hist ? a.hist + a.voff[e] : nullptr, Re, Re + NV);
  // 2 x 2 tiles of one operator: at most 18 x (18 + 8) (degree 4)
  element_blocks<D3, true, kThreads, 2, 1, 1>(d, E, ptv, ptf, Ap, X, Cp, S, sm);
  // 4. factorisation and condensation
  const int ld = NV % 2 ? NV + 2 : NV + 1;
  const bool in_smem = NV <= kLuSmemMax;
  double* LU = in_smem ? sm : LUg;
  double* Xs = in_smem ? sm + even(NV * ld) : sm;
  double* dinv = Xs + NV * kCB;
  double* ys = dinv + NV;
  int* perm = reinterpret_cast<int*>(ys + NV);
  for (int t = tid; t < NV * NV; t += nth) LU[t / NV * ld + t % NV] = Ap[t];
  for (int t = tid; t < NV; t += nth) LU[t * ld + NV] = Re[t];
  __syncthreads();
  const bool ok = element_condense<kThreads, kCB>(LU, ld, NV, perm, dinv, ys, s_piv, Xs, Cp, Re + NV, X,
                                                  X + (int64_t)NV * ntq, S, a.g + a.toff[e], ntq);
  if (tid == 0 && !ok) atomicOr(a.status + e, HDG_STATUS_SINGULAR);
  __syncthreads();
}

__global__ void __launch_bounds__(kThreads, 2) k_pclass_fused(PArgs a, PhysParams ph) {
  extern __shared__ __align__(16) double sm[];
  __shared__ ElemTables<D3> E;
  __shared__ int s_idx, s_piv[2];
  double* slot = a.scratch + (int64_t)blockIdx.x * a.slot_doubles;
  for (;;) {
    if (threadIdx.x == 0) s_idx = atomicAdd(a.counter, 1);
    __syncthreads();
    const int idx = s_idx;
    __syncthreads();
    if (idx >= a.E) break;
    const int64_t e = a.queue[idx];
    pc_element(a, a.tab[a.cls[e]], ph, e, sm, slot, E, s_piv);
  }
}

}  // namespace

int pclass_index(int pk, int pt) {
  if (pk < 1 || pt < pk || pt > 4) return -1;
  static const int base[5] = {0, 0, 4, 7, 9};
  return base[pk] + (pt - pk);
}


int assemble_condense_pclass(hdg_ctx* c, const double* V, const double* Vhat, const double* hist, double mass_coef,
                             double* S, double* g, double* recov, double* R, int32_t* status, cudaStream_t s) {
  PMix& pm = *c->pm;
  if (!pm.attr_set) {
    int optin = 0, per_sm = 0;
    cudaFuncAttributes fa{};
    HDG_CK(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, c->device));
    HDG_CK(cudaFuncGetAttributes(&fa, k_pclass_fused));
    if (pm.smem_bytes > (size_t)optin - fa.sharedSizeBytes) {
      set_error("assemble_condense: the element classes need more shared memory than the device has");
      return HDG_ERR_UNSUPPORTED;
    }
    // the limit belongs to the kernel and the device, not to this context: always the most there is, as another
    // context's classes may need more than this one's
    HDG_CK(cudaFuncSetAttribute(k_pclass_fused, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                optin - (int)fa.sharedSizeBytes));
    HDG_CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_pclass_fused, kThreads, pm.smem_bytes));
    pm.ctas = (int)std::min<int64_t>(c->E, (int64_t)std::max(1, per_sm) * (c->num_sms > 0 ? c->num_sms : 152));
    pm.attr_set = true;
  }
  const size_t need = sizeof(double) * (size_t)pm.ctas * pm.slot_doubles;
  if (c->scr_bytes < need) {
    if (c->d_scr) cudaFree(c->d_scr);
    c->d_scr = nullptr;
    c->scr_bytes = 0;
    HDG_CK(cudaMalloc(&c->d_scr, need));
    c->scr_bytes = need;
  }
  PArgs a{};
  a.V = V;
  a.Vhat = Vhat;
  a.hist = hist;
  a.mass_coef = mass_coef;
  a.voff = pm.d_voff;
  a.toff = pm.d_toff;
  a.soff = pm.d_soff;
  a.roff = pm.d_roff;
  a.Roff = pm.d_Roff;
  a.tgidx = pm.d_tgidx;
  a.fdeg = pm.d_fdeg;
  a.cls = pm.d_cls;
  a.geo = c->d_geo;
  a.queue = pm.d_queue;
  a.E = c->E;
  a.nfn_max = pm.nfn_max;
  a.slot_doubles = pm.slot_doubles;
  a.counter = pm.d_counter;
  a.scratch = c->d_scr;
  a.S = S;
  a.g = g;
  a.recov = recov;
  a.R = R;
  a.status = status;
  for (int k = 0; k < kPClasses; ++k) a.tab[k] = pm.tab[k];
  HDG_CK(cudaMemsetAsync(pm.d_counter, 0, sizeof(int), s));
  LaunchScope ls(c, HDG_KERNEL_PCLASS, s);
  k_pclass_fused<<<pm.ctas, kThreads, pm.smem_bytes, s>>>(a, c->ph);
  HDG_CK(cudaGetLastError());
  return HDG_OK;
}

namespace {

template <class T>
int up(T** dst, const std::vector<T>& src) {
  HDG_CK(cudaMalloc(dst, sizeof(T) * std::max<size_t>(1, src.size())));
  if (!src.empty()) HDG_CK(cudaMemcpy(*dst, src.data(), sizeof(T) * src.size(), cudaMemcpyHostToDevice));
  return HDG_OK;
}

}  // namespace

int pclass_setup(hdg_ctx* c) {
  const Mesh& m = c->mesh->m;
  if (m.dim != 3 || !c->visc) {
    set_error("hdg_ctx_create: mixed-degree meshes are built for 3D Navier-Stokes");
    return HDG_ERR_UNSUPPORTED;
  }
  auto* pm = new PMix();
  c->pm = pm;
  const int NF = c->NF;
  const int64_t E = c->E;
  pm->pmin = 99;
  for (int8_t q : m.pe) {
    pm->pmin = std::min<int>(pm->pmin, q);
    pm->pmax = std::max<int>(pm->pmax, q);
  }
  pm->nfn_max = m.ref.Nf;
  pm->n_tnodes = m.fnoff.back();
  // class tables, one buffer
  std::vector<double> tab;
  std::vector<int> itab;
  size_t off[kPClasses][13], qoff[kPClasses][4][4], ioff[kPClasses];
  bool have[kPClasses] = {};
  auto append = [&](const std::vector<double>& v) {
    if (tab.size() % 2) tab.push_back(0.0);
    tab.insert(tab.end(), v.begin(), v.end());
    return tab.size() - v.size();
  };
  std::vector<ClassTables> ct(kPClasses);
  for (int pk = pm->pmin; pk <= pm->pmax; ++pk)
    for (int pt = pk; pt <= pm->pmax; ++pt) ct[pclass_index(pk, pt)] = make_class_tables(3, pk, pt);
  for (int pk = pm->pmin; pk <= pm->pmax; ++pk)
    for (int pt = pk; pt <= pm->pmax; ++pt) {
      const int k = pclass_index(pk, pt);
      const ClassTables& T = ct[k];
      const int NP = T.Np, NG = T.NG, NGF = T.NGF, NFN = T.Nft, nF = T.nF;
      // the element functions' lifted gradients in reference coordinates
      std::vector<double> dR = T.dPhi, dRF = T.dPhiF;
      for (int r = 0; r < 3; ++r)
        for (int t = 0; t < NG * NP; ++t) dR[r * NG * NP + t] += T.PLV[(r + 1) * NG * NP + t] - T.PLV[t];
      for (int f = 0; f < nF; ++f)
        for (int r = 0; r < 3; ++r)
          for (int t = 0; t < NGF * NP; ++t)
            dRF[(f * 3 + r) * NGF * NP + t] += T.PLFV[(f * nF + r + 1) * NGF * NP + t] - T.PLFV[f * nF * NGF * NP + t];
      const std::vector<double>* parts[13] = {&T.W, &T.Phi,  &T.dPhi, &dR,   &T.WF,  &T.PhiF, &T.dPhiF,
                                              &dRF, &T.PsiF, &T.PhiN, &T.PL, &T.PLF, &T.IPro};
      for (int i = 0; i < 13; ++i) off[k][i] = append(*parts[i]);
      // trace functions of a face's own degree q: combinations of the degree-pt ones
      for (int q = 1; q <= pt; ++q) {
        const int n = (q + 1) * (q + 2) / 2;
        auto combine = [&](const std::vector<double>& src, int rows, int f_of_row_div, bool lift_major) {
          // src rows [..][NFN] -> [..][n]; the face whose functions a row holds: row / f_of_row_div (% nF)
          std::vector<double> out((size_t)rows * n, 0.0);
          for (int row = 0; row < rows; ++row) {
            const int f = row / f_of_row_div % nF;
            size_t dst = row;
            if (lift_major) {  // [points' face][lift's face] -> [lift's face][points' face]
              const int ff = row / NGF / nF, fl = row / NGF % nF, g = row % NGF;
              dst = ((size_t)fl * nF + ff) * NGF + g;
            }
            for (int cq = 0; cq < n; ++cq) {
              double s = 0.0;
              for (int c = 0; c < NFN; ++c)
                s += src[(size_t)row * NFN + c] * T.IPro[(((size_t)(q - 1) * nF + f) * NFN + c) * NFN + cq];
              out[dst * n + cq] = s;
            }
          }
          return out;
        };
        qoff[k][q - 1][0] = append(combine(T.PsiF, nF * NGF, NGF, false));
        qoff[k][q - 1][1] = append(combine(T.PL, nF * NG, NG, false));
        qoff[k][q - 1][2] = append(combine(T.PLF, nF * nF * NGF, NGF, true));
        qoff[k][q - 1][3] = q > pk ? append(ct[pclass_index(pk, q)].PhiN) : 0;
      }
      ioff[k] = itab.size();
      std::vector<int> pos(nF * NP, -1);
      for (int f = 0; f < nF; ++f)
        for (int c = 0; c < T.Nfk; ++c) pos[f * NP + T.fnodesK[f * T.Nfk + c]] = c;
      itab.insert(itab.end(), pos.begin(), pos.end());
      have[k] = true;
      pm->tab[k].d = pclass_dims(pk, pt);
    }
  // classes and trace map
  auto nfn = [](int q) { return (q + 1) * (q + 2) / 2; };
  std::vector<int8_t> fdeg(E * NF), cls(E);
  std::vector<int> tg(E * NF * pm->nfn_max, -1);
  for (int64_t e = 0; e < E; ++e) {
    for (int f = 0; f < NF; ++f) {
      const int64_t F = m.face_of[e * NF + f];
      const int q = m.fdeg[F];
      fdeg[e * NF + f] = (int8_t)q;
      for (int cc = 0; cc < nfn(q); ++cc)
        tg[(e * NF + f) * pm->nfn_max + cc] = (int)(m.fnoff[F] + m.fnode_mix[(e * NF + f) * pm->nfn_max + cc]);
    }
    cls[e] = (int8_t)pclass_index(m.pe[e], m.ptr[e]);
    pm->class_count[cls[e]]++;
  }
  // trace addressing: own face-node counts, the two local occurrences of every trace node,
  // face-block offsets
  std::vector<int> fnn(E * NF), occ_e(2 * m.fnoff.back(), -1), occ_l(2 * m.fnoff.back(), -1);
  std::vector<int64_t> pcoff(c->F + 1, 0);
  for (int64_t e = 0; e < E; ++e) {
    int qoff = 0;
    for (int f = 0; f < NF; ++f) {
      const int64_t F = m.face_of[e * NF + f];
      const int nq = nfn(m.fdeg[F]);
      fnn[e * NF + f] = nq;
      const int side = m.face_side[2 * F] == (int32_t)(e * NF + f) ? 0 : 1;
      for (int cl = 0; cl < nq; ++cl) {
        const int64_t t = m.fnoff[F] + m.fnode_mix[(e * NF + f) * pm->nfn_max + cl];
        occ_e[2 * t + side] = (int)e;
        occ_l[2 * t + side] = qoff + cl * 5;
      }
      qoff += nq * 5;
    }
    pm->nt_max = std::max(pm->nt_max, qoff);
  }
  for (int64_t F = 0; F < c->F; ++F) {
    const int64_t B = (m.fnoff[F + 1] - m.fnoff[F]) * 5;
    pcoff[F + 1] = pcoff[F] + B * B;
  }
  pm->pc_len = pcoff.back();
  // queue: largest class first (interior size, then trace degree), element order within a class
  std::vector<int> queue(E);
  for (int64_t e = 0; e < E; ++e) queue[e] = (int)e;
  std::stable_sort(queue.begin(), queue.end(), [&](int x, int y) {
    const int kx = m.pe[x] * 8 + m.ptr[x], ky = m.pe[y] * 8 + m.ptr[y];
    return kx > ky;
  });
  int rc = HDG_OK;
  if ((rc = up(&pm->d_tab, tab)) || (rc = up(&pm->d_itab, itab)) || (rc = up(&pm->d_voff, m.voff)) ||
      (rc = up(&pm->d_toff, m.toff)) || (rc = up(&pm->d_soff, m.soff)) || (rc = up(&pm->d_roff, m.roff)) ||
      (rc = up(&pm->d_Roff, m.Roff)) || (rc = up(&pm->d_tgidx, tg)) || (rc = up(&pm->d_fdeg, fdeg)) ||
      (rc = up(&pm->d_cls, cls)) || (rc = up(&pm->d_queue, queue)) || (rc = up(&pm->d_fnn, fnn)) ||
      (rc = up(&pm->d_occ_e, occ_e)) || (rc = up(&pm->d_occ_l, occ_l)) || (rc = up(&pm->d_fnoff, m.fnoff)) ||
      (rc = up(&pm->d_pcoff, pcoff)))
    return rc;
  HDG_CK(cudaMalloc(&pm->d_counter, sizeof(int)));
  for (int k = 0; k < kPClasses; ++k) {
    if (!have[k]) continue;
    const double* b = pm->d_tab;
    PClassDev& d = pm->tab[k];
    const double** dst[13] = {&d.W,   &d.Phi,  &d.dPhi, &d.dR, &d.WF,  &d.PhiF, &d.dPhiF,
                              &d.dRF, &d.PsiF, &d.PhiN, &d.PL, &d.PLF, &d.IPro};
    for (int i = 0; i < 13; ++i) *dst[i] = b + off[k][i];
    for (int q = 0; q < d.d.pt; ++q) {
      d.PsiQ[q] = b + qoff[k][q][0];
      d.PLQ[q] = b + qoff[k][q][1];
      d.PLFQ[q] = b + qoff[k][q][2];
      d.TrQ[q] = b + qoff[k][q][3];
    }
    d.nodepos = pm->d_itab + ioff[k];
  }
  for (int k = 0; k < kPClasses; ++k)
    if (pm->class_count[k] > 0) {
      pm->smem_bytes = std::max(pm->smem_bytes, sizeof(double) * (size_t)pm->tab[k].d.SMEM);
      pm->slot_doubles = std::max(pm->slot_doubles, pm->tab[k].d.SLOT);
    }
  if (!c->num_sms) HDG_CK(cudaDeviceGetAttribute(&c->num_sms, cudaDevAttrMultiProcessorCount, c->device));
  return HDG_OK;
}

void pclass_free(PMix* pm) {
  if (!pm) return;
  void* bufs[] = {pm->d_voff, pm->d_toff,  pm->d_soff,    pm->d_roff, pm->d_Roff,  pm->d_tgidx,
                  pm->d_fdeg, pm->d_cls,   pm->d_queue,   pm->d_counter, pm->d_tab, pm->d_itab,
                  pm->d_fnn,  pm->d_occ_e, pm->d_occ_l,   pm->d_fnoff, pm->d_pcoff};
  for (void* b : bufs)
    if (b) cudaFree(b);
  delete pm;
}

}  // namespace hdg
