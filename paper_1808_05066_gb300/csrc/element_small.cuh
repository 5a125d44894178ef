// FP64 kernels for small elements: contraction in physical coordinates and a condensation with one LU of the whole
// block. The kernels of element_fp64.cuh spread an element over register tiles and blocks; an element of a few
// dozen unknowns does not fill those, and a mesh of fewer elements than the chip has room for waits for one
// element's latency, which is shorter here.
// small_elements() draws the line, in elements per SM for 2D meshes; measured on 152 SMs (assemble + condense, ms, here and
// there):
//   always here: 3D p = 1, 48,000 elements 50.8, 58.6; 2D Euler p = 1 (51,200) 12.4, 12.5, p = 2 (32,768) 12.4, 13.9,
//     p = 3 (18,432) 14.6, 15.3; 2D NS p = 2 (32,768) 19.9, 21.6
//   2D NS p = 3, up to seven per SM: 128 elements 0.446, 0.556; 512 0.820, 0.792; 800 1.216, 1.311; 968 1.470, 1.481;
//     1,058 1.475, 1.513; then 1,152 1.578, 1.548; 1,352 1.831, 1.830; 1,568 2.180, 2.197; 2,048 2.804, 2.640; 18,432
//     23.1, 22.0
//   2D NS p = 4, up to one: 128 0.765, 0.852; then 162 1.044, 0.973; 512 2.106, 1.671; 8,192 24.5, 19.5
//   2D Euler p = 4, up to two: 128 0.511, 0.599; 288 0.696, 0.715; then 338 0.913, 0.905; 512 1.426, 1.297
//   3D p = 2 and 3: never (6 elements 1.78, 1.68 and 7.95, 4.37; 3,072 24.7, 16.0 and 167.6, 67.5)
// The two sides round differently: an element's blocks may differ in the last bits between meshes on either side.
#pragma once
#include "assemble_fp64.cuh"
#include "ctx.hpp"

namespace hdg {
namespace small {

template <class C>
constexpr bool kCompiled = C::NV < 40 || C::D == 2;  // configurations that can take these kernels
template <class C>
bool small_elements(int64_t E, int num_sms) {
  constexpr int per_sm = C::NV == 40 ? 7 : C::VISC ? 1 : 2;
  return C::NV < 40 || (!C::VISC && C::NV == 40) || (C::D == 2 && E <= per_sm * (int64_t)num_sms);
}

// doubles per volume and face point
template <class C>
struct Pt {
  static constexpr int D = C::D, M = C::M;
  static constexpr int VOL = M + D * M + M * M + D * M * M + (C::VISC ? D * M * M * D : 0);
  static constexpr int FACE = M + 2 * M * M + (C::VISC ? M * M * D : 0);
};

// sum_j c_j dG_ij/dq_lk for one vector c: the viscous flux (Eq. viscFlux) is linear in q, and
// differentiating it by hand gives, with V_a = -w_a/v_m, A_a = w_a/v_m^2 and the Kronecker
// delta d,
//   momentum i = 1+a, l = 1+b:    mu/v_m (d_ab c_k + d_ak c_b - 2/3 d_bk c_a)
//   momentum i = 1+a, l = m-1:   -mu (A_a c_k + d_ak c.A - 2/3 A_k c_a)
//   energy   i = m-1, l = 1+b:    mu/v_m (V_b c_k + V_k c_b - 2/3 d_bk c.V)
//   energy   i = m-1, l = m-1:   -mu (V.A c_k + V_k c.A - 2/3 A_k c.V) - kappa/(c_v v_m^2) c_k
// and zero for i = 0 or l = 0. emit(i, l, k, value) receives every entry; the deltas are
// branches on unrolled indices, so no arithmetic is spent on the vanishing terms.
template <int D, class Emit>
HDG_DEVI void visc_jac_dir(const ViscFactors<D>& f, const double* c, const PhysParams& ph, Emit emit) {
  constexpr int M = D + 2;
  constexpr double t3 = 2.0 / 3.0;
  double cA = c[0] * f.A[0], cV = c[0] * f.vel[0], VA = f.vel[0] * f.A[0];
#pragma unroll
  for (int j = 1; j < D; ++j) {
    cA += c[j] * f.A[j];
    cV += c[j] * f.vel[j];
    VA += f.vel[j] * f.A[j];
  }
  const double mi = ph.mu * f.ivm, kc = (ph.kappa / ph.cv) * f.ivm2;
#pragma unroll
  for (int k = 0; k < D; ++k) {
#pragma unroll
    for (int l = 0; l < M; ++l) emit(0, l, k, 0.0);
#pragma unroll
    for (int i = 1; i < M; ++i) emit(i, 0, k, 0.0);
#pragma unroll
    for (int a = 0; a < D; ++a) {
#pragma unroll
      for (int b = 0; b < D; ++b) {
        double s = 0.0;
        bool any = false;
        if (a == b) {
          s = c[k];
          any = true;
        }
        if (a == k) {
          s = any ? s + c[b] : c[b];
          any = true;
        }
        if (b == k) {
          s = any ? s - t3 * c[a] : -t3 * c[a];
          any = true;
        }
        emit(1 + a, 1 + b, k, any ? mi * s : 0.0);
      }
      double s = f.A[a] * c[k] - t3 * f.A[k] * c[a];
      if (a == k) s += cA;
      emit(1 + a, M - 1, k, -ph.mu * s);
    }
#pragma unroll
    for (int b = 0; b < D; ++b) {
      double s = f.vel[b] * c[k] + f.vel[k] * c[b];
      if (b == k) s -= t3 * cV;
      emit(M - 1, 1 + b, k, mi * s);
    }
    emit(M - 1, M - 1, k, -ph.mu * (VA * c[k] + f.vel[k] * cA - t3 * f.A[k] * cV) - kc * c[k]);
  }
}

template <class C, bool SYM = false>
__global__ void __launch_bounds__(128) k_pointwise_small(AssembleArgs a, DevTables T, PhysParams ph) {
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
    double* out = reinterpret_cast<double*>(a.ptv) + (le * NG + g) * Pt<C>::VOL;
    double* MU = out;
    double* FR = MU + M;
    double* T0 = FR + D * M;
    double* T1 = T0 + M * M;
    double* T2 = T1 + D * M * M;
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
      // dG/dq contracted with the rows of Jinv (G is linear in q)
      const ViscFactors<D> vf = visc_factors<D>(v);
      const PhysParams pv = visc_params_at(ph, v[M - 1]);
#pragma unroll 1
      for (int r = 0; r < D; ++r)
        visc_jac_dir<D>(vf, Jinv + r * D, pv, [&](int i, int l, int k, double val) {
          put(T2, ((r * M + i) * M + l) * D + k, -W * val);
        });
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
    double* out = reinterpret_cast<double*>(a.ptf) + ((le * NF + f) * NGF + gf) * Pt<C>::FACE;
    double* HF = out;
    double* U0 = HF + M;
    double* U1 = U0 + M * M;
    double* U2 = U1 + M * M;
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
      visc_jac_dir<D>(vf, n, visc_params_at(ph, vs[M - 1]),
                      [&](int i, int l, int k, double val) { put(U2, (i * M + l) * D + k, Wf * val); });
    }
  }
  if (bad) atomicOr(a.status + e, HDG_STATUS_NONPHYSICAL);
}

// k_pointwise_small with the stabilization matrix the physics selects
template <class C>
void launch_pointwise_small(const AssembleArgs& a, const DevTables& T, const PhysParams& ph, cudaStream_t s) {
  const int threads = ((C::NG + C::NF * C::NGF + 31) / 32) * 32;
  if (ph.stab == 1)
    k_pointwise_small<C, true><<<(unsigned)a.ne, threads, 0, s>>>(a, T, ph);
  else
    k_pointwise_small<C, false><<<(unsigned)a.ne, threads, 0, s>>>(a, T, ph);
}

// ------------------------------------------------------------------------------------
// k_assemble_small
// ------------------------------------------------------------------------------------
template <class C>
struct AsmSmem {
  static constexpr int GT = C::NG < 64 ? C::NG : 64;  // volume points per tile
  static constexpr int RB = C::NR * GT * C::NZ;
  static constexpr int RBF = C::NRF * C::NGF * C::NZ;
  static constexpr int RBMAX = RB > RBF ? RB : RBF;
  static constexpr int ZS = C::NP * GT * C::NR;
  static constexpr int ZSF = C::NFN * C::NGF * C::NRF;
  static constexpr int ZSMAX = ZS > ZSF ? ZS : ZSF;
  static constexpr size_t bytes =
      sizeof(double) * (RBMAX + ZSMAX + C::NZ * C::M + C::GEO + C::NV + C::NT);
};

template <class C>
__global__ void __launch_bounds__(256) k_assemble_small(AssembleArgs a, DevTables T) {
  constexpr int D = C::D, M = C::M, NP = C::NP, NFN = C::NFN, NF = C::NF, NG = C::NG, NGF = C::NGF;
  constexpr int NZ = C::NZ, NV = C::NV, NT = C::NT, NR = C::NR, NRF = C::NRF;
  using SM = AsmSmem<C>;
  constexpr int GT = SM::GT;
  extern __shared__ double smem[];
  double* Rb = smem;
  double* Zs = Rb + SM::RBMAX;
  double(*z)[M] = reinterpret_cast<double(*)[M]>(Zs + SM::ZSMAX);
  double* G = Zs + SM::ZSMAX + NZ * M;
  double* Rv = G + C::GEO;
  double* Rt = Rv + NV;
  const int64_t le = blockIdx.x;
  const int64_t e = a.e0 + le;
  if (skip_element(a, e)) return;
  const int tid = threadIdx.x, nth = blockDim.x;
  load_element<C>(a, e, z, G);
  __syncthreads();
  const double* Jinv = G;
  const double detJ = G[D * D];
  double* Ap = a.Ap + le * NV * NV;
  double* Cp = a.Cp + le * NT * NV;
  double* Bp = a.recov + e * (int64_t)(NV * NT + NV);
  double* Dp = a.S + e * (int64_t)NT * NT;
  const double* ptv = a.ptv + le * NG * Pt<C>::VOL;
  const double* ptf = a.ptf + le * NF * NGF * Pt<C>::FACE;

  // residual R_v, volume part
  for (int t = tid; t < NV; t += nth) {
    int an = t / M, i = t % M;
    double s = a.hist ? -a.hist[e * NV + t] : 0.0;
    for (int g = 0; g < NG; ++g) {
      const double* P = ptv + g * Pt<C>::VOL;
      s += T.Phi[g * NP + an] * P[i];
      for (int r = 0; r < D; ++r) s += T.dPhi[(r * NG + g) * NP + an] * P[M + r * M + i];
    }
    Rv[t] = s;
  }

  // ---------------- volume contractions ----------------
  for (int g0 = 0; g0 < NG; g0 += GT) {
    const int ng = (NG - g0) < GT ? (NG - g0) : GT;
    __syncthreads();
    // right operators Rb[beta][gg][j]
    for (int t = tid; t < NR * GT * NZ; t += nth) {
      int beta = t / (GT * NZ), gg = (t / NZ) % GT, j = t % NZ;
      double val = 0.0;
      if (gg < ng) {
        int g = g0 + gg;
        if (beta == 0) {
          val = j < NP ? T.Phi[g * NP + j] : 0.0;
        } else {
          int k = beta - 1;
          if (j < NP) {
            for (int r = 0; r < D; ++r) val += Jinv[r * D + k] * T.dPhi[(r * NG + g) * NP + j];
            for (int f = 0; f < NF; ++f) {
              int c = T.nodepos[f * NP + j];
              if (c >= 0) {
                const double* Gf = G + D * D + 1 + f * (D + 1);
                val -= Gf[k] * (Gf[D] / detJ) * T.PL[(f * NG + g) * NFN + c];
              }
            }
          } else {
            int f = (j - NP) / NFN, c = (j - NP) % NFN;
            const double* Gf = G + D * D + 1 + f * (D + 1);
            val = Gf[k] * (Gf[D] / detJ) * T.PL[(f * NG + g) * NFN + c];
          }
        }
      }
      Rb[t] = val;
    }
    for (int il = 0; il < M * M; ++il) {
      const int i = il / M, l = il % M;
      __syncthreads();
      // Zs[a][gg][beta] = sum_alpha L_alpha(g, a) C^{il}_{alpha beta}(g)
      for (int t = tid; t < NP * GT * NR; t += nth) {
        int an = t / (GT * NR), gg = (t / NR) % GT, beta = t % NR;
        double val = 0.0;
        if (gg < ng) {
          int g = g0 + gg;
          const double* P = ptv + g * Pt<C>::VOL;
          const double* T0 = P + M + D * M;
          const double* T1 = T0 + M * M;
          const double* T2 = T1 + D * M * M;
          if (beta == 0) {
            val = T.Phi[g * NP + an] * T0[i * M + l];
            for (int r = 0; r < D; ++r) val += T.dPhi[(r * NG + g) * NP + an] * T1[(r * M + i) * M + l];
          } else {
            int k = beta - 1;
            for (int r = 0; r < D; ++r)
              val += T.dPhi[(r * NG + g) * NP + an] * T2[((r * M + i) * M + l) * D + k];
          }
        }
        Zs[t] = val;
      }
      __syncthreads();
      for (int t = tid; t < NP * NZ; t += nth) {
        int an = t / NZ, j = t % NZ;
        const int b0 = j < NP ? 0 : 1;
        double acc = 0.0;
        for (int gg = 0; gg < ng; ++gg)
          for (int beta = b0; beta < NR; ++beta) acc += Zs[(an * GT + gg) * NR + beta] * Rb[(beta * GT + gg) * NZ + j];
        int row = an * M + i;
        if (j < NP) {
          double* dst = Ap + row * NV + j * M + l;
          *dst = (g0 == 0) ? acc : *dst + acc;
        } else {
          double* dst = Bp + row * NT + (j - NP) * M + l;
          *dst = (g0 == 0) ? acc : *dst + acc;
        }
      }
    }
  }

  // ---------------- face contractions ----------------
  for (int f = 0; f < NF; ++f) {
    __syncthreads();
    const double* Gf = G + D * D + 1 + f * (D + 1);
    for (int t = tid; t < NRF * NGF * NZ; t += nth) {
      int beta = t / (NGF * NZ), gf = (t / NZ) % NGF, j = t % NZ;
      const double* phif = T.PhiF + (f * NGF + gf) * NP;
      double val = 0.0;
      if (beta == 0) {
        val = j < NP ? phif[j] : 0.0;
      } else if (beta == 1) {
        if (j >= NP && (j - NP) / NFN == f) val = phif[T.fnodes[f * NFN + (j - NP) % NFN]];
      } else {
        int k = beta - 2;
        if (j < NP) {
          for (int r = 0; r < D; ++r) val += Jinv[r * D + k] * T.dPhiF[((f * D + r) * NGF + gf) * NP + j];
          for (int fl = 0; fl < NF; ++fl) {
            int c = T.nodepos[fl * NP + j];
            if (c >= 0) {
              const double* Gl = G + D * D + 1 + fl * (D + 1);
              val -= Gl[k] * (Gl[D] / detJ) * T.PLF[((f * NF + fl) * NGF + gf) * NFN + c];
            }
          }
        } else {
          int fl = (j - NP) / NFN, c = (j - NP) % NFN;
          const double* Gl = G + D * D + 1 + fl * (D + 1);
          val = Gl[k] * (Gl[D] / detJ) * T.PLF[((f * NF + fl) * NGF + gf) * NFN + c];
        }
      }
      Rb[t] = val;
    }
    (void)Gf;
    // residual: face contribution
    __syncthreads();
    for (int t = tid; t < NFN * M; t += nth) {
      int c = t / M, i = t % M;
      double s = 0.0;
      for (int gf = 0; gf < NGF; ++gf) {
        double psi = T.PhiF[(f * NGF + gf) * NP + T.fnodes[f * NFN + c]];
        s += psi * ptf[(f * NGF + gf) * Pt<C>::FACE + i];
      }
      Rv[T.fnodes[f * NFN + c] * M + i] += s;
      Rt[(f * NFN + c) * M + i] = s;
    }
    for (int il = 0; il < M * M; ++il) {
      const int i = il / M, l = il % M;
      __syncthreads();
      for (int t = tid; t < NFN * NGF * NRF; t += nth) {
        int c = t / (NGF * NRF), gf = (t / NRF) % NGF, beta = t % NRF;
        const double* P = ptf + (f * NGF + gf) * Pt<C>::FACE;
        const double* U0 = P + M;
        const double* U1 = U0 + M * M;
        const double* U2 = U1 + M * M;
        double psi = T.PhiF[(f * NGF + gf) * NP + T.fnodes[f * NFN + c]];
        double u;
        if (beta == 0)
          u = U0[i * M + l];
        else if (beta == 1)
          u = U1[i * M + l];
        else
          u = U2[(i * M + l) * D + (beta - 2)];
        Zs[t] = psi * u;
      }
      __syncthreads();
      for (int t = tid; t < NFN * NZ; t += nth) {
        int c = t / NZ, j = t % NZ;
        double acc = 0.0;
        for (int gf = 0; gf < NGF; ++gf)
          for (int beta = 0; beta < NRF; ++beta) acc += Zs[(c * NGF + gf) * NRF + beta] * Rb[(beta * NGF + gf) * NZ + j];
        int rowv = T.fnodes[f * NFN + c] * M + i;
        int rowt = (f * NFN + c) * M + i;
        if (j < NP) {
          Ap[rowv * NV + j * M + l] += acc;
          Cp[rowt * NV + j * M + l] = acc;
        } else {
          int tcol = (j - NP) * M + l;
          Bp[rowv * NT + tcol] += acc;
          Dp[rowt * NT + tcol] = acc;
        }
      }
    }
  }
  __syncthreads();
  double* Rout = a.R + e * (int64_t)(NV + NT);
  for (int t = tid; t < NV; t += nth) Rout[t] = Rv[t];
  for (int t = tid; t < NT; t += nth) Rout[NV + t] = Rt[t];
}

// ------------------------------------------------------------------------------------
// k_condense_small
// ------------------------------------------------------------------------------------
template <class C>
struct CondSmem {
  static constexpr int CB = 64;  // right-hand-side columns per block
  static constexpr size_t bytes = sizeof(double) * (C::NV * C::NV + C::NV * CB) + sizeof(int) * C::NV + 64;
};

template <class C>
__global__ void __launch_bounds__(256) k_condense_small(AssembleArgs a) {
  constexpr int NV = C::NV, NT = C::NT;
  using SM = CondSmem<C>;
  constexpr int CB = SM::CB;
  extern __shared__ double smem[];
  double* LU = smem;                 // [NV][NV]
  double* Xs = LU + NV * NV;         // [NV][CB]
  int* piv = reinterpret_cast<int*>(Xs + NV * CB);
  __shared__ int s_piv;
  __shared__ int s_bad;
  const int64_t le = blockIdx.x;
  const int64_t e = a.e0 + le;
  if (skip_element(a, e)) return;
  const int tid = threadIdx.x, nth = blockDim.x;
  const double* Ap = a.Ap + le * NV * NV;
  const double* Cp = a.Cp + le * NT * NV;
  double* X = a.recov + e * (int64_t)(NV * NT + NV);
  double* y = X + NV * NT;
  double* S = a.S + e * (int64_t)NT * NT;
  const double* R = a.R + e * (int64_t)(NV + NT);
  for (int t = tid; t < NV * NV; t += nth) LU[t] = Ap[t];
  if (tid == 0) s_bad = 0;
  __syncthreads();
  // LU with partial pivoting (row interchanges recorded in piv)
  for (int k = 0; k < NV; ++k) {
    if (tid < 32) {
      double best = -1.0;
      int bi = k;
      for (int r = k + tid; r < NV; r += 32) {
        double v = fabs(LU[r * NV + k]);
        if (v > best) {
          best = v;
          bi = r;
        }
      }
      for (int off = 16; off > 0; off >>= 1) {
        double ob = __shfl_down_sync(0xffffffffu, best, off);
        int oi = __shfl_down_sync(0xffffffffu, bi, off);
        if (ob > best || (ob == best && oi < bi)) {
          best = ob;
          bi = oi;
        }
      }
      if (tid == 0) {
        s_piv = bi;
        piv[k] = bi;
        if (!(best > 0.0)) s_bad = 1;
      }
    }
    __syncthreads();
    const int pr = s_piv;
    if (pr != k)
      for (int j = tid; j < NV; j += nth) {
        double t = LU[k * NV + j];
        LU[k * NV + j] = LU[pr * NV + j];
        LU[pr * NV + j] = t;
      }
    __syncthreads();
    const double d = LU[k * NV + k];
    const double inv = d != 0.0 ? 1.0 / d : 0.0;
    for (int r = k + 1 + tid; r < NV; r += nth) LU[r * NV + k] *= inv;
    __syncthreads();
    const int rem = NV - k - 1;
    for (int t = tid; t < rem * rem; t += nth) {
      int r = k + 1 + t / rem, c = k + 1 + t % rem;
      LU[r * NV + c] -= LU[r * NV + k] * LU[k * NV + c];
    }
    __syncthreads();
  }
  if (tid == 0 && s_bad) atomicOr(a.status + e, HDG_STATUS_SINGULAR);
  // X = A'^{-1} [B' | R_v] in column blocks (B' stored in X)
  for (int c0 = 0; c0 < NT + 1; c0 += CB) {
    const int nc = (NT + 1 - c0) < CB ? (NT + 1 - c0) : CB;
    __syncthreads();
    for (int t = tid; t < NV * CB; t += nth) {
      int r = t / CB, c = t % CB;
      int col = c0 + c;
      double v = 0.0;
      if (c < nc) v = col < NT ? X[r * NT + col] : R[r];
      Xs[t] = v;
    }
    __syncthreads();
    // apply the row interchanges in order
    for (int t = tid; t < CB; t += nth)
      for (int k = 0; k < NV; ++k) {
        int p = piv[k];
        if (p != k) {
          double tmp = Xs[k * CB + t];
          Xs[k * CB + t] = Xs[p * CB + t];
          Xs[p * CB + t] = tmp;
        }
      }
    __syncthreads();
    for (int k = 0; k < NV; ++k) {  // forward, unit lower
      for (int t = tid; t < (NV - k - 1) * CB; t += nth) {
        int r = k + 1 + t / CB, c = t % CB;
        Xs[r * CB + c] -= LU[r * NV + k] * Xs[k * CB + c];
      }
      __syncthreads();
    }
    for (int k = NV - 1; k >= 0; --k) {  // backward, upper
      for (int c = tid; c < CB; c += nth) Xs[k * CB + c] /= LU[k * NV + k];
      __syncthreads();
      for (int t = tid; t < k * CB; t += nth) {
        int r = t / CB, c = t % CB;
        Xs[r * CB + c] -= LU[r * NV + k] * Xs[k * CB + c];
      }
      __syncthreads();
    }
    for (int t = tid; t < NV * CB; t += nth) {
      int r = t / CB, c = t % CB;
      int col = c0 + c;
      if (c < nc) {
        if (col < NT)
          X[r * NT + col] = Xs[t];
        else
          y[r] = Xs[t];
      }
    }
  }
  __syncthreads();
  // S = D' - C' X ; g = R_t - C' y
  for (int t = tid; t < NT * NT; t += nth) {
    int r = t / NT, c = t % NT;
    double s = S[t];
    const double* Cr = Cp + r * NV;
    for (int k = 0; k < NV; ++k) s -= Cr[k] * X[k * NT + c];
    S[t] = s;
  }
  double* g = a.g + e * NT;
  for (int r = tid; r < NT; r += nth) {
    double s = R[NV + r];
    const double* Cr = Cp + r * NV;
    for (int k = 0; k < NV; ++k) s -= Cr[k] * y[k];
    g[r] = s;
  }
  if (a.only_flag != 0 && tid == 0) {  // flagged-only pass: the block is now the FP64 form's
    atomicAnd(a.status + e, ~a.only_flag);
    atomicOr(a.status + e, HDG_STATUS_FP64);
  }
}

}  // namespace small

// The FP64 form's launches, by small_elements(); the mixed form's recomputation takes them too, so that a recomputed block is
// the FP64 form's bit for bit. Static: each translation unit has kernels of its own, with their own attributes.
template <class C>
static void point_doubles(bool sm, size_t* vol, size_t* face) {  // doubles of point data per element
  *vol = (size_t)C::NG * (sm ? small::Pt<C>::VOL : C::PT_VOL);
  *face = (size_t)C::NF * C::NGF * (sm ? small::Pt<C>::FACE : C::PT_FACE);
}
template <class C>
static int fp64_attributes() {
  HDG_CK(cudaFuncSetAttribute(k_assemble<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)AsmSmem<C>::bytes));
  HDG_CK(cudaFuncSetAttribute(k_condense<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CondSmem<C>::bytes));
  if constexpr (small::kCompiled<C>) {
    HDG_CK(cudaFuncSetAttribute(small::k_assemble_small<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)small::AsmSmem<C>::bytes));
    HDG_CK(cudaFuncSetAttribute(small::k_condense_small<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)small::CondSmem<C>::bytes));
  }
  return HDG_OK;
}
template <class C>
static void fp64_pointwise(bool sm, const AssembleArgs& a, const DevTables& T, const PhysParams& ph, cudaStream_t s) {
  if constexpr (small::kCompiled<C>)
    if (sm) return small::launch_pointwise_small<C>(a, T, ph, s);
  launch_pointwise<C>(a, T, ph, s);
}
template <class C>
static void fp64_assemble(bool sm, const AssembleArgs& a, const DevTables& T, cudaStream_t s) {
  if constexpr (small::kCompiled<C>)
    if (sm) {
      small::k_assemble_small<C><<<(unsigned)a.ne, 256, small::AsmSmem<C>::bytes, s>>>(a, T);
      return;
    }
  k_assemble<C><<<(unsigned)a.ne, AsmSmem<C>::NTH, AsmSmem<C>::bytes, s>>>(a, T);
}
template <class C>
static void fp64_condense(bool sm, const AssembleArgs& a, cudaStream_t s) {
  if constexpr (small::kCompiled<C>)
    if (sm) {
      small::k_condense_small<C><<<(unsigned)a.ne, 256, small::CondSmem<C>::bytes, s>>>(a);
      return;
    }
  k_condense<C><<<(unsigned)a.ne, CondSmem<C>::NTH, CondSmem<C>::bytes, s>>>(a);
}
}  // namespace hdg
