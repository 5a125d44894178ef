// Per-face MLP that predicts the trace update of the next implicit step, used to
// warm-start Newton (no counterpart in the paper; it serves the Newton solve of the
// method, which stays the judge: the converged answer is the same either way).
//
// Network: x (NIN) -> tanh(W1 x + b1) (NH) -> tanh(W2 h1 + b2) (NH) -> W3 h2 + b3 (NOUT).
// Weights are used in BF16 with FP32 accumulation; an FP32 master copy and the Adam
// moments live in the same parameter buffer:
//   params [P] FP32 master | m [P] | v [P] | w16 [P] BF16 copy used by the kernels,
// P = NH*NIN + NH + NH*NH + NH + NOUT*NH + NOUT, laid out as W1 (row-major [NH][NIN]),
// b1, W2 [NH][NH], b2, W3 [NOUT][NH], b3.
//
// Features of face F (canonical node order), all as differences so the map is
// invariant to the state level: [V_side0 - vhat^n | V_side1 - vhat^n | dvhat^n |
// dvhat^{n-1}] at the NFN face nodes, standardised by per-feature mean and scale.
#include <cuda_bf16.h>

#include <cstdint>

#include "ctx.hpp"

namespace hdg {

namespace {

constexpr int MAXH = 64;  // hidden width supported by the register-resident kernels

__host__ __device__ inline int64_t mlp_params(int nin, int nh, int nout) {
  return (int64_t)nh * nin + nh + (int64_t)nh * nh + nh + (int64_t)nout * nh + nout;
}

// SplitMix64 counter-based generator (Steele, Lea & Flood 2014), used for the initial weights.
__device__ inline uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

__global__ void k_mlp_init(float* params, int nin, int nh, int nout, uint64_t seed) {
  const int64_t P = mlp_params(nin, nh, nout);
  float* m = params + P;
  float* v = m + P;
  __nv_bfloat16* w16 = reinterpret_cast<__nv_bfloat16*>(v + P);
  const int64_t o1 = (int64_t)nh * nin, o2 = o1 + nh, o3 = o2 + (int64_t)nh * nh, o4 = o3 + nh,
                o5 = o4 + (int64_t)nout * nh;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < P; t += (int64_t)gridDim.x * blockDim.x) {
    float val = 0.f;
    int fan_in = 0, fan_out = 0;
    if (t < o1) {
      fan_in = nin;
      fan_out = nh;
    } else if (t >= o2 && t < o3) {
      fan_in = nh;
      fan_out = nh;
    } else if (t >= o4 && t < o5) {
      fan_in = nh;
      fan_out = nout;
    }
    if (fan_in) {  // Glorot-uniform
      const double u = (double)(splitmix64(seed * 0x100000001B3ull + (uint64_t)t) >> 11) * (1.0 / 9007199254740992.0);
      const double lim = ::sqrt(6.0 / (double)(fan_in + fan_out));
      val = (float)((2.0 * u - 1.0) * lim);
      if (t >= o4) val *= 0.1f;  // small output layer: the start predicts ~0 correction
    }
    params[t] = val;
    m[t] = 0.f;
    v[t] = 0.f;
    w16[t] = __float2bfloat16_rn(val);
  }
}

// Face features [F][4][NFN][M] (float), standardised: (raw - mean) / std in FP64, the reciprocals of std once per block.
// 49,152 faces of 64 features, features to corrected trace: 79 us; with an FP64 division per feature, 127 us.
__global__ void k_mlp_features(const double* V, const double* Vhat, const double* dvh1, const double* dvh2,
                               const int* fs_elem, const int* fs_loc, const int* fnodes, int64_t F, int NFN, int M,
                               int NP, int NF, const float* mean, const float* stdv, float* feat) {
  extern __shared__ double mlp_stat[];  // mean [nin], 1 / stdv [nin]
  const int per = NFN * M;
  const int nin = 4 * per;
  const int64_t n = F * per;
  double* mu = mlp_stat;
  double* inv = mlp_stat + nin;
  for (int t = threadIdx.x; t < nin; t += blockDim.x) {
    mu[t] = mean[t];
    inv[t] = 1.0 / (double)stdv[t];
  }
  __syncthreads();
  const int64_t step = (int64_t)gridDim.x * blockDim.x, dF = step / per;
  const int dr = (int)(step % per);
  int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, Fi = t / per;
  int r = (int)(t % per);
  for (; t < n; t += step) {
    const int c = r / M, i = r % M;
    const double vh = Vhat[t];
    float* out = feat + Fi * nin;
    for (int side = 0; side < 2; ++side) {
      const int64_t e = fs_elem[2 * Fi + side];
      const int loc = fs_loc[(2 * Fi + side) * NFN + c];  // f * NFN + local face node
      const int f = loc / NFN, cl = loc % NFN;
      const int a = fnodes[f * NFN + cl];
      const double v = V[(e * NP + a) * M + i];
      const int k = side * per + r;
      out[k] = (float)((v - vh - mu[k]) * inv[k]);
    }
    out[2 * per + r] = (float)((dvh1[t] - mu[2 * per + r]) * inv[2 * per + r]);
    out[3 * per + r] = (float)((dvh2[t] - mu[3 * per + r]) * inv[3 * per + r]);
    Fi += dF;
    r += dr;
    if (r >= per) {
      r -= per;
      ++Fi;
    }
  }
}

template <int NIN, int NH, int NOUT>
__device__ inline void mlp_forward_one(const __nv_bfloat16* w, const float* x, float* h1, float* h2, float* y) {
  const __nv_bfloat16* W1 = w;
  const __nv_bfloat16* b1 = W1 + NH * NIN;
  const __nv_bfloat16* W2 = b1 + NH;
  const __nv_bfloat16* b2 = W2 + NH * NH;
  const __nv_bfloat16* W3 = b2 + NH;
  const __nv_bfloat16* b3 = W3 + NOUT * NH;
#pragma unroll 4
  for (int j = 0; j < NH; ++j) {
    float s = __bfloat162float(b1[j]);
    for (int k = 0; k < NIN; ++k) s = fmaf(__bfloat162float(W1[j * NIN + k]), x[k], s);
    h1[j] = tanhf(s);
  }
#pragma unroll 4
  for (int j = 0; j < NH; ++j) {
    float s = __bfloat162float(b2[j]);
    for (int k = 0; k < NH; ++k) s = fmaf(__bfloat162float(W2[j * NH + k]), h1[k], s);
    h2[j] = tanhf(s);
  }
  for (int j = 0; j < NOUT; ++j) {
    float s = __bfloat162float(b3[j]);
    for (int k = 0; k < NH; ++k) s = fmaf(__bfloat162float(W3[j * NH + k]), h2[k], s);
    y[j] = s;
  }
}

// Forward for a batch: one thread per sample, BF16 weights staged in shared memory.
template <int NIN, int NH, int NOUT>
__global__ void __launch_bounds__(128) k_mlp_forward(const float* params, const float* x, int64_t B, float* y) {
  constexpr int P = NH * NIN + NH + NH * NH + NH + NOUT * NH + NOUT;
  __shared__ __nv_bfloat16 w[P];
  const __nv_bfloat16* w16 = reinterpret_cast<const __nv_bfloat16*>(params + 3 * (int64_t)P);
  for (int t = threadIdx.x; t < P; t += blockDim.x) w[t] = w16[t];
  __syncthreads();
  const int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (b >= B) return;
  float xin[NIN], h1[NH], h2[NH], out[NOUT];
  for (int k = 0; k < NIN; ++k) xin[k] = x[b * NIN + k];
  mlp_forward_one<NIN, NH, NOUT>(w, xin, h1, h2, out);
  for (int j = 0; j < NOUT; ++j) y[b * NOUT + j] = out[j];
}

// Forward on the tensor cores: each warp takes 16 samples, and a layer out = act W^T + b is a
// 16 x N product over K in steps of 16 (mma.sync m16n8k16, bf16 operands, FP32 accumulation).
// The FP32 activations enter as two bf16 parts, hi = bf16(a) and lo = bf16(a - hi), which carry
// them to about 2^-16 relative; the weights are the BF16 copy, exactly as in the scalar kernel.
HDG_DEVI void mlp_mma(float (&c)[4], const uint4& a, const uint2& b) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y));
}

// the bf16 pairs (x0, x1) of hi and lo parts (x0 in the low half)
HDG_DEVI void mlp_split2(float x0, float x1, unsigned& hi, unsigned& lo) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
  const float2 hf = __bfloat1622float2(h);
  const __nv_bfloat162 l = __floats2bfloat162_rn(x0 - hf.x, x1 - hf.y);
  hi = *reinterpret_cast<const unsigned*>(&h);
  lo = *reinterpret_cast<const unsigned*>(&l);
}

// One layer of a warp's 16 samples, out[16][N] = f(in[16][K] W^T + b), in and out as A fragments of m16n8k16 split into
// hi and lo (g = lane / 4, t = lane % 4: rows g, g + 8 at columns 2t, 2t + 1 and 2t + 8, 2t + 9 of each k tile). The
// accumulators of two neighbouring 8-column tiles hold exactly the entries of the next layer's k tile in its
// fragment's places, so activations stay in registers from layer to layer and are split once. W [N][LD] row-major (bf16,
// shared; LD = K + 8 puts the eight rows a fragment reads in different banks).
template <int K, int N, bool TANH, class Put>
HDG_DEVI void mlp_layer_tc(const __nv_bfloat16* W, const __nv_bfloat16* bias, const uint4 (&hi)[K / 16],
                           const uint4 (&lo)[K / 16], int lane, Put put) {
  constexpr int LD = K + 8;
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int nt = 0; nt < N / 8; ++nt) {
    float c[4] = {0.f, 0.f, 0.f, 0.f};
    const __nv_bfloat16* Wn = W + (nt * 8 + g) * LD + 2 * t;
#pragma unroll
    for (int kt = 0; kt < K / 16; ++kt) {
      uint2 b;
      b.x = *reinterpret_cast<const unsigned*>(Wn + kt * 16);
      b.y = *reinterpret_cast<const unsigned*>(Wn + kt * 16 + 8);
      mlp_mma(c, hi[kt], b);
      mlp_mma(c, lo[kt], b);
    }
    const int col = nt * 8 + 2 * t;
    const float b0 = __bfloat162float(bias[col]), b1 = __bfloat162float(bias[col + 1]);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float v = c[q] + (q & 1 ? b1 : b0);
      c[q] = TANH ? tanhf(v) : v;
    }
    put(nt, c);
  }
}

// The 64-64-16 network. Eight warps of 16 samples share one copy of the weights and go through the batch. 49,152
// samples, features to corrected trace: 19 us less (146 to 127) than with activations in shared memory between the layers
// and a block of two warps per 32 samples.
template <int NIN, int NH, int NOUT>
__global__ void __launch_bounds__(256, 2) k_mlp_forward_tc(const float* params, const float* x, int64_t B, float* y) {
  static_assert(NIN % 16 == 0 && NH % 16 == 0 && NOUT % 8 == 0, "tile shape");
  constexpr int P = NH * NIN + NH + NH * NH + NH + NOUT * NH + NOUT;
  constexpr int L1 = NIN + 8, L2 = NH + 8;
  __shared__ __align__(16) __nv_bfloat16 W1[NH * L1], W2[NH * L2], W3[NOUT * L2], bs[2 * NH + NOUT];
  const __nv_bfloat16* w16 = reinterpret_cast<const __nv_bfloat16*>(params + 3 * (int64_t)P);
  constexpr int o1 = NH * NIN, o2 = o1 + NH, o3 = o2 + NH * NH, o4 = o3 + NH, o5 = o4 + NOUT * NH;
  for (int t = threadIdx.x; t < NH * NIN; t += 256) W1[t / NIN * L1 + t % NIN] = w16[t];
  for (int t = threadIdx.x; t < NH * NH; t += 256) W2[t / NH * L2 + t % NH] = w16[o2 + t];
  for (int t = threadIdx.x; t < NOUT * NH; t += 256) W3[t / NH * L2 + t % NH] = w16[o4 + t];
  for (int t = threadIdx.x; t < 2 * NH + NOUT; t += 256)
    bs[t] = w16[t < NH ? o1 + t : t < 2 * NH ? o3 + t - NH : o5 + t - 2 * NH];
  __syncthreads();
  const int lane = threadIdx.x & 31, g = lane >> 2, t2 = 2 * (lane & 3);
  const int64_t ntile = (B + 15) / 16;
  for (int64_t tile = blockIdx.x * 8 + (threadIdx.x >> 5); tile < ntile; tile += (int64_t)gridDim.x * 8) {
    const int64_t r0 = tile * 16 + g, r1 = r0 + 8;
    uint4 hi[NIN / 16], lo[NIN / 16];
#pragma unroll
    for (int kt = 0; kt < NIN / 16; ++kt) {
      float v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {  // scalar loads: x may have any alignment of a float
        const int64_t r = q & 2 ? r1 : r0;
        v[q] = r < B ? x[r * NIN + kt * 16 + t2 + (q & 4 ? 8 : 0) + (q & 1)] : 0.f;
      }
      mlp_split2(v[0], v[1], hi[kt].x, lo[kt].x);
      mlp_split2(v[2], v[3], hi[kt].y, lo[kt].y);
      mlp_split2(v[4], v[5], hi[kt].z, lo[kt].z);
      mlp_split2(v[6], v[7], hi[kt].w, lo[kt].w);
    }
    uint4 h1h[NH / 16], h1l[NH / 16], h2h[NH / 16], h2l[NH / 16];
    auto into = [](uint4 (&H)[NH / 16], uint4 (&L)[NH / 16]) {
      return [&H, &L](int nt, const float (&c)[4]) {
        const int kt = nt >> 1;
        if (nt & 1) {
          mlp_split2(c[0], c[1], H[kt].z, L[kt].z);
          mlp_split2(c[2], c[3], H[kt].w, L[kt].w);
        } else {
          mlp_split2(c[0], c[1], H[kt].x, L[kt].x);
          mlp_split2(c[2], c[3], H[kt].y, L[kt].y);
        }
      };
    };
    mlp_layer_tc<NIN, NH, true>(W1, bs, hi, lo, lane, into(h1h, h1l));
    mlp_layer_tc<NH, NH, true>(W2, bs + NH, h1h, h1l, lane, into(h2h, h2l));
    mlp_layer_tc<NH, NOUT, false>(W3, bs + 2 * NH, h2h, h2l, lane, [&](int nt, const float (&c)[4]) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t r = q & 2 ? r1 : r0;
        if (r < B) y[r * NOUT + nt * 8 + t2 + (q & 1)] = c[q];
      }
    });
  }
}

// Forward + backward of the mean-squared error (mean over the batch and the NOUT outputs), FP32 throughout with the
// BF16 weights. A CTA of 256 threads takes tiles of TS samples; every step is a small matrix product with the
// operands in shared memory ([sample][feature], [output][input], rows padded by 4 so that 16-byte loads of
// neighbouring rows meet different banks) and register tiles: 4 outputs x TS / 16 samples for the layers, 4 x 4 weights for
// the weight gradients, which stay in registers over all tiles of the CTA and go to grad [P] once, by 16-byte
// reductions. loss [1] accumulates.
// Bound: FP32 issue and shared-memory reads (1.2G FMA at 49,152 samples of the 64-64-16 network, 31 us at the FP32
// rate). One thread per sample with all its activations in shared memory, and one atomic per weight and 64
// samples, took about 590 us; a whole training step of that network and batch (gradient and Adam) went from 609 to 97 us.
template <int NIN, int NH, int NOUT, int TS>
struct GradSmem {
  static constexpr int L1 = NIN + 4, L2 = NH + 4, LO = (NOUT + 3) / 4 * 4 + 4;
  static constexpr size_t bytes =
      sizeof(float) * (size_t)(NH * L1 + NH * L2 + NOUT * L2 + 2 * NH + NOUT + TS * (L1 + 3 * L2 + LO) + 8);
};

// out[s][j] for j < N, s < TS: tile loops over the K inputs by four; in [TS][LDI], W [N][LDW]
template <int K, int N, int TS, int LDI, int LDW, class Epi>
HDG_DEVI void mlp_tile_forward(const float* in, const float* W, Epi epi) {
  constexpr int TJ = N / 4, TR = 256 / TJ, RS = TS / TR;  // thread (tj, tr): outputs tj + TJ i, samples tr + TR q
  static_assert(N % 4 == 0 && 256 % TJ == 0 && TS % TR == 0, "tile");
  const int tj = threadIdx.x % TJ, tr = threadIdx.x / TJ;
  float acc[RS][4] = {};
#pragma unroll 4
  for (int k = 0; k < K; k += 4) {
    float4 w[4], v[RS];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = *reinterpret_cast<const float4*>(W + (tj + TJ * i) * LDW + k);
#pragma unroll
    for (int q = 0; q < RS; ++q) v[q] = *reinterpret_cast<const float4*>(in + (tr + TR * q) * LDI + k);
#pragma unroll
    for (int q = 0; q < RS; ++q)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        acc[q][i] = fmaf(w[i].x, v[q].x, acc[q][i]);
        acc[q][i] = fmaf(w[i].y, v[q].y, acc[q][i]);
        acc[q][i] = fmaf(w[i].z, v[q].z, acc[q][i]);
        acc[q][i] = fmaf(w[i].w, v[q].w, acc[q][i]);
      }
  }
#pragma unroll
  for (int q = 0; q < RS; ++q)
#pragma unroll
    for (int i = 0; i < 4; ++i) epi(tr + TR * q, tj + TJ * i, acc[q][i]);
}

// d[s][k] = (sum_j e[s][j] W[j][k]) (1 - h[s][k]^2), k < N: the gradient before a tanh layer
template <int J, int N, int TS, int LDE, int LDW, int LDH>
HDG_DEVI void mlp_tile_backward(const float* e, const float* W, const float* h, float* d) {
  constexpr int TJ = N / 4, TR = 256 / TJ, RS = TS / TR;
  static_assert(J % 4 == 0, "tile");
  const int k0 = 4 * (threadIdx.x % TJ), tr = threadIdx.x / TJ;
  float4 acc[RS] = {};
#pragma unroll 4
  for (int j = 0; j < J; j += 4) {
    float4 w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = *reinterpret_cast<const float4*>(W + (j + i) * LDW + k0);
#pragma unroll
    for (int q = 0; q < RS; ++q) {
      const float4 v = *reinterpret_cast<const float4*>(e + (tr + TR * q) * LDE + j);
      const float ev[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        acc[q].x = fmaf(w[i].x, ev[i], acc[q].x);
        acc[q].y = fmaf(w[i].y, ev[i], acc[q].y);
        acc[q].z = fmaf(w[i].z, ev[i], acc[q].z);
        acc[q].w = fmaf(w[i].w, ev[i], acc[q].w);
      }
    }
  }
#pragma unroll
  for (int q = 0; q < RS; ++q) {
    const int r = tr + TR * q;
    const float4 u = *reinterpret_cast<const float4*>(h + r * LDH + k0);
    *reinterpret_cast<float4*>(d + r * LDH + k0) =
        make_float4(acc[q].x * (1.f - u.x * u.x), acc[q].y * (1.f - u.y * u.y), acc[q].z * (1.f - u.z * u.z),
                    acc[q].w * (1.f - u.w * u.w));
  }
}

// acc[i][q] += sum_s d[s][j0 + i] v[s][k0 + q] for this thread's 4 x 4 weights
template <int TS, int LDD, int LDV>
HDG_DEVI void mlp_tile_weights(const float* d, const float* v, int j0, int k0, float (&acc)[4][4]) {
#pragma unroll 4
  for (int s = 0; s < TS; ++s) {
    const float4 a = *reinterpret_cast<const float4*>(d + s * LDD + j0), b = *reinterpret_cast<const float4*>(v + s * LDV + k0);
    const float av[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      acc[i][0] = fmaf(av[i], b.x, acc[i][0]);
      acc[i][1] = fmaf(av[i], b.y, acc[i][1]);
      acc[i][2] = fmaf(av[i], b.z, acc[i][2]);
      acc[i][3] = fmaf(av[i], b.w, acc[i][3]);
    }
  }
}

HDG_DEVI void mlp_red4(float* p, const float (&v)[4], bool vec) {
  if (vec) {
    asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3])
                 : "memory");
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) atomicAdd(p + q, v[q]);
  }
}

template <int NIN, int NH, int NOUT, int TS>
__global__ void __launch_bounds__(256, 2) k_mlp_grad(const float* params, const float* x, const float* target, int64_t B,
                                                    float* grad, float* loss) {
  using G = GradSmem<NIN, NH, NOUT, TS>;
  constexpr int P = NH * NIN + NH + NH * NH + NH + NOUT * NH + NOUT, L1 = G::L1, L2 = G::L2, LO = G::LO;
  constexpr int o1 = NH * NIN, o2 = o1 + NH, o3 = o2 + NH * NH, o4 = o3 + NH, o5 = o4 + NOUT * NH;
  extern __shared__ __align__(16) float smf[];
  float* W1 = smf;              // [NH][L1]
  float* W2 = W1 + NH * L1;     // [NH][L2]
  float* W3 = W2 + NH * L2;     // [NOUT][L2]
  float* xs = W3 + NOUT * L2;   // [TS][L1]
  float* h1 = xs + TS * L1;     // [TS][L2]
  float* h2 = h1 + TS * L2;     // [TS][L2], later the gradient before the first tanh
  float* d2 = h2 + TS * L2;     // [TS][L2]
  float* dy = d2 + TS * L2;     // [TS][LO]
  float* bs = dy + TS * LO;     // biases
  float* lsum = bs + 2 * NH + NOUT;
  const int tid = threadIdx.x;
  const __nv_bfloat16* w16 = reinterpret_cast<const __nv_bfloat16*>(params + 3 * (int64_t)P);
  for (int t = tid; t < NH * NIN; t += 256) W1[t / NIN * L1 + t % NIN] = __bfloat162float(w16[t]);
  for (int t = tid; t < NH * NH; t += 256) W2[t / NH * L2 + t % NH] = __bfloat162float(w16[o2 + t]);
  for (int t = tid; t < NOUT * NH; t += 256) W3[t / NH * L2 + t % NH] = __bfloat162float(w16[o4 + t]);
  for (int t = tid; t < 2 * NH + NOUT; t += 256)
    bs[t] = __bfloat162float(w16[t < NH ? o1 + t : t < 2 * NH ? o3 + t - NH : o5 + t - 2 * NH]);
  if (tid == 0) *lsum = 0.f;
  // this thread's weights: 4 x 4 tiles of dW1, dW2 and dW3, and one bias
  constexpr int T1 = NH * NIN / 16, T2 = NH * NH / 16, T3 = NOUT * NH / 16;
  static_assert(T1 <= 256 && T2 <= 256 && T3 <= 256 && 2 * NH + NOUT <= 256, "one tile per thread");
  const int j1 = 4 * (tid / (NIN / 4)), k1 = 4 * (tid % (NIN / 4)), j2 = 4 * (tid / (NH / 4)), k2 = 4 * (tid % (NH / 4));
  float g1[4][4] = {}, g2[4][4] = {}, g3[4][4] = {}, gb = 0.f, l = 0.f;
  const float inv = 1.f / ((float)B * (float)NOUT);
  for (int64_t base = (int64_t)blockIdx.x * TS; base < B; base += (int64_t)gridDim.x * TS) {
    __syncthreads();
    for (int t = tid; t < TS * NIN; t += 256) {
      const int s = t / NIN;
      xs[s * L1 + t % NIN] = base + s < B ? x[base * NIN + t] : 0.f;
    }
    __syncthreads();
    mlp_tile_forward<NIN, NH, TS, L1, L1>(xs, W1, [&](int s, int j, float v) { h1[s * L2 + j] = tanhf(v + bs[j]); });
    __syncthreads();
    mlp_tile_forward<NH, NH, TS, L2, L2>(h1, W2, [&](int s, int j, float v) { h2[s * L2 + j] = tanhf(v + bs[NH + j]); });
    __syncthreads();
    for (int t = tid; t < TS * NOUT; t += 256) {  // the output layer, the error and its gradient
      const int s = t / NOUT, j = t % NOUT;
      float v = 0.f;
#pragma unroll 4
      for (int k = 0; k < NH; k += 4) {
        const float4 w = *reinterpret_cast<const float4*>(W3 + j * L2 + k), h = *reinterpret_cast<const float4*>(h2 + s * L2 + k);
        v = fmaf(w.x, h.x, fmaf(w.y, h.y, fmaf(w.z, h.z, fmaf(w.w, h.w, v))));
      }
      float d = 0.f;  // samples past the batch contribute nothing
      if (base + s < B) d = v + bs[2 * NH + j] - target[base * NOUT + t];
      l += d * d * inv;
      dy[s * LO + j] = 2.f * d * inv;
    }
    __syncthreads();
    mlp_tile_backward<NOUT, NH, TS, LO, L2, L2>(dy, W3, h2, d2);
    if (tid < T3) mlp_tile_weights<TS, LO, L2>(dy, h2, j2, k2, g3);
    __syncthreads();
    mlp_tile_backward<NH, NH, TS, L2, L2, L2>(d2, W2, h1, h2);  // h2 becomes the gradient before the first tanh
    if (tid < T2) mlp_tile_weights<TS, L2, L2>(d2, h1, j2, k2, g2);
    __syncthreads();
    if (tid < T1) mlp_tile_weights<TS, L2, L1>(h2, xs, j1, k1, g1);
    if (tid < 2 * NH + NOUT) {
      const float* src = tid < NH ? h2 + tid : tid < 2 * NH ? d2 + tid - NH : dy + tid - 2 * NH;
      const int ld = tid < 2 * NH ? L2 : LO;
      for (int s = 0; s < TS; ++s) gb += src[s * ld];
    }
  }
  const bool vec = (reinterpret_cast<uintptr_t>(grad) & 15) == 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (tid < T1) mlp_red4(grad + (j1 + i) * NIN + k1, g1[i], vec);
    if (tid < T2) mlp_red4(grad + o2 + (j2 + i) * NH + k2, g2[i], vec);
    if (tid < T3) mlp_red4(grad + o4 + (j2 + i) * NH + k2, g3[i], vec);
  }
  if (tid < 2 * NH + NOUT) atomicAdd(grad + (tid < NH ? o1 + tid : tid < 2 * NH ? o3 + tid - NH : o5 + tid - 2 * NH), gb);
  for (int off = 16; off > 0; off >>= 1) l += __shfl_down_sync(0xffffffffu, l, off);
  if ((tid & 31) == 0) atomicAdd(lsum, l);
  __syncthreads();
  if (tid == 0) atomicAdd(loss, *lsum);
}

// Adam on the FP32 master weights, then refresh the BF16 copy.
__global__ void k_mlp_adam(float* params, const float* grad, int64_t P, float lr, float beta1, float beta2, float eps,
                           int step) {
  float* m = params + P;
  float* v = m + P;
  __nv_bfloat16* w16 = reinterpret_cast<__nv_bfloat16*>(v + P);
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < P; t += (int64_t)gridDim.x * blockDim.x) {
    const float g = grad[t];
    const float mt = beta1 * m[t] + (1.f - beta1) * g;
    const float vt = beta2 * v[t] + (1.f - beta2) * g * g;
    m[t] = mt;
    v[t] = vt;
    const float p = params[t] - lr * (mt / c1) / (sqrtf(vt / c2) + eps);
    params[t] = p;
    w16[t] = __float2bfloat16_rn(p);
  }
}

// vhat_out = vhat + dvh1 + pred * tscale (per output component of a face)
__global__ void k_mlp_apply(const double* Vhat, const double* dvh1, const float* pred, const float* tscale,
                            const float* tmean, int64_t F, int per, double* out) {
  const int64_t n = F * per;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
    const int r = (int)(t % per);
    out[t] = Vhat[t] + dvh1[t] + ((double)pred[t] * (double)tscale[r] + (double)tmean[r]);
  }
}

__global__ void k_mlp_zero(float* grad, int64_t P, float* loss) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < P; t += (int64_t)gridDim.x * blockDim.x) grad[t] = 0.f;
  if (blockIdx.x == 0 && threadIdx.x == 0) *loss = 0.f;
}

// TS: samples per tile (64-64-16: 48, the most that lets two CTAs share an SM)
template <int NIN, int NH, int NOUT, int TS>
int launch_grad(const float* params, const float* x, const float* target, int64_t B, float* grad, float* loss,
                cudaStream_t s) {
  using G = GradSmem<NIN, NH, NOUT, TS>;
  constexpr int P = NH * NIN + NH + NH * NH + NH + NOUT * NH + NOUT;
  HDG_CK(cudaFuncSetAttribute(k_mlp_grad<NIN, NH, NOUT, TS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)G::bytes));
  k_mlp_zero<<<(P + 255) / 256, 256, 0, s>>>(grad, P, loss);
  const int64_t tiles = (B + TS - 1) / TS;
  k_mlp_grad<NIN, NH, NOUT, TS><<<(unsigned)(tiles < 2 * 152 ? tiles : 2 * 152), 256, G::bytes, s>>>(params, x, target,
                                                                                                   B, grad, loss);
  HDG_CK(cudaGetLastError());
  return HDG_OK;
}

// Column statistics of x [B][n]: mean and standard deviation (FP64 accumulation; a
// deviation below 1e-30 is reported as 1 so that standardising leaves the column as is).
__global__ void k_mlp_stats(const float* x, int64_t B, int n, float* mean, float* stdv) {
  const int col = blockIdx.x;
  double s = 0.0, s2 = 0.0;
  for (int64_t b = threadIdx.x; b < B; b += blockDim.x) {
    const double v = x[b * n + col];
    s += v;
    s2 += v * v;
  }
  __shared__ double ps[256], ps2[256];
  ps[threadIdx.x] = s;
  ps2[threadIdx.x] = s2;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      ps[threadIdx.x] += ps[threadIdx.x + w];
      ps2[threadIdx.x] += ps2[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double m = ps[0] / (double)B;
    const double var = ps2[0] / (double)B - m * m;
    const double sd = var > 1e-60 ? ::sqrt(var) : 1.0;
    mean[col] = (float)m;
    stdv[col] = (float)sd;
  }
}

__global__ void k_mlp_standardize(float* x, int64_t B, int n, const float* mean, const float* stdv) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < B * n; t += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(t % n);
    x[t] = (x[t] - mean[c]) / stdv[c];
  }
}

// Raw training target: the correction of the extrapolated trace update,
// (vhat^{n+1} - vhat^n) - dvhat^n.
__global__ void k_mlp_target(int64_t n, const double* vh_next, const double* vh, const double* dvh1, float* out) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
    out[t] = (float)((vh_next[t] - vh[t]) - dvh1[t]);
}

inline unsigned nb(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (unsigned)(b < 1 ? 1 : (b > 152 * 32 ? 152 * 32 : b));
}

}  // namespace

}  // namespace hdg

using namespace hdg;

#define MLP_DISPATCH(NIN, NH, NOUT, ...) \
  if (nin == NIN && nh == NH && nout == NOUT) { __VA_ARGS__; }

extern "C" {

int64_t hdg_mlp_param_count(int nin, int nh, int nout) { return mlp_params(nin, nh, nout); }

int hdg_mlp_init(float* params, int nin, int nh, int nout, uint64_t seed, void* stream) {
  if (!params || nin <= 0 || nh <= 0 || nh > MAXH || nout <= 0) {
    set_error("hdg_mlp_init: invalid argument");
    return HDG_ERR_INVALID_ARG;
  }
  k_mlp_init<<<nb(mlp_params(nin, nh, nout)), 256, 0, (cudaStream_t)stream>>>(params, nin, nh, nout, seed);
  HDG_CK(cudaGetLastError());
  return HDG_OK;
}

int hdg_mlp_features(hdg_ctx_t ctx, const double* V, const double* Vhat, const double* dvh1, const double* dvh2,
                     const float* mean, const float* stdv, float* feat, void* stream) {
  if (!ctx || !V || !Vhat || !dvh1 || !dvh2 || !mean || !stdv || !feat) {
    set_error("hdg_mlp_features: null argument");
    return HDG_ERR_INVALID_ARG;
  }
  if (ctx->pm) {
    set_error("hdg_mlp_features: not built for meshes of mixed degree");
    return HDG_ERR_UNSUPPORTED;
  }
  if (ctx->scheme || !ctx->h_bface.empty()) {
    set_error("hdg_mlp_features: the per-face network works on two-sided face traces (periodic HDG) only");
    return HDG_ERR_UNSUPPORTED;
  }
  const unsigned grid = nb(ctx->ntrace) < 152 * 8 ? nb(ctx->ntrace) : 152 * 8;
  k_mlp_features<<<grid, 256, sizeof(double) * 8 * ctx->NFN * ctx->M, (cudaStream_t)stream>>>(
      V, Vhat, dvh1, dvh2, ctx->d_fs_elem, ctx->d_fs_loc, ctx->T.fnodes, ctx->F, ctx->NFN, ctx->M, ctx->NP, ctx->NF,
      mean, stdv, feat);
  HDG_CK(cudaGetLastError());
  return HDG_OK;
}

int hdg_mlp_forward(const float* params, int nin, int nh, int nout, const float* x, int64_t B, float* y,
                    void* stream) {
  if (!params || !x || !y || B < 0) {
    set_error("hdg_mlp_forward: invalid argument");
    return HDG_ERR_INVALID_ARG;
  }
  if (B == 0) return HDG_OK;
  const unsigned g = (unsigned)((B + 127) / 128);
  cudaStream_t s = (cudaStream_t)stream;
  // 64-64-16 (2D p = 3) on the tensor cores, 128 samples per block and pass; 48-32-12 keeps the scalar kernel
  // (its output width is not a multiple of the tile's 8 columns)
  const int64_t t128 = (B + 127) / 128;
  const unsigned gt = (unsigned)(t128 < 3 * 152 ? t128 : 3 * 152);
  MLP_DISPATCH(64, 64, 16, (k_mlp_forward_tc<64, 64, 16><<<gt, 256, 0, s>>>(params, x, B, y));
               HDG_CK(cudaGetLastError()); return HDG_OK)
  MLP_DISPATCH(48, 32, 12, (k_mlp_forward<48, 32, 12><<<g, 128, 0, s>>>(params, x, B, y)); HDG_CK(cudaGetLastError());
               return HDG_OK)
  set_error("hdg_mlp_forward: network size not compiled in");
  return HDG_ERR_UNSUPPORTED;
}

int hdg_mlp_train_step(float* params, float* grad, int nin, int nh, int nout, const float* x, const float* target,
                       int64_t B, float lr, int step, float* loss, void* stream) {
  if (!params || !grad || !x || !target || !loss || B <= 0 || step < 1) {
    set_error("hdg_mlp_train_step: invalid argument");
    return HDG_ERR_INVALID_ARG;
  }
  const int64_t P = mlp_params(nin, nh, nout);
  cudaStream_t s = (cudaStream_t)stream;
  bool done = false;
  int rc = HDG_OK;
  MLP_DISPATCH(64, 64, 16, rc = launch_grad<64, 64, 16, 48>(params, x, target, B, grad, loss, s); done = true)
  MLP_DISPATCH(48, 32, 12, rc = launch_grad<48, 32, 12, 64>(params, x, target, B, grad, loss, s); done = true)
  if (rc) return rc;
  if (!done) {
    set_error("hdg_mlp_train_step: network size not compiled in");
    return HDG_ERR_UNSUPPORTED;
  }
  k_mlp_adam<<<nb(P), 256, 0, s>>>(params, grad, P, lr, 0.9f, 0.999f, 1e-8f, step);
  HDG_CK(cudaGetLastError());
  return HDG_OK;
}

int hdg_mlp_gradient(const float* params, float* grad, int nin, int nh, int nout, const float* x, const float* target,
                     int64_t B, float* loss, void* stream) {
  if (!params || !grad || !x || !target || !loss || B <= 0) {
    set_error("hdg_mlp_gradient: invalid argument");
    return HDG_ERR_INVALID_ARG;
  }
  const int64_t P = mlp_params(nin, nh, nout);
  cudaStream_t s = (cudaStream_t)stream;
  MLP_DISPATCH(64, 64, 16, return launch_grad<64, 64, 16, 48>(params, x, target, B, grad, loss, s))
  MLP_DISPATCH(48, 32, 12, return launch_grad<48, 32, 12, 64>(params, x, target, B, grad, loss, s))
  set_error("hdg_mlp_gradient: network size not compiled in");
  return HDG_ERR_UNSUPPORTED;
}

int hdg_mlp_stats(const float* x, int64_t B, int n, float* mean, float* stdv, void* stream) {
  if (!x || !mean || !stdv || B <= 0 || n <= 0) {
    set_error("hdg_mlp_stats: invalid argument");
    return HDG_ERR_INVALID_ARG;
  }
  k_mlp_stats<<<n, 256, 0, (cudaStream_t)stream>>>(x, B, n, mean, stdv);
  HDG_CK(cudaGetLastError());
  return HDG_OK;
}

int hdg_mlp_standardize(float* x, int64_t B, int n, const float* mean, const float* stdv, void* stream) {
  if (!x || !mean || !stdv || B < 0 || n <= 0) {
    set_error("hdg_mlp_standardize: invalid argument");
    return HDG_ERR_INVALID_ARG;
  }
  k_mlp_standardize<<<nb(B * n), 256, 0, (cudaStream_t)stream>>>(x, B, n, mean, stdv);
  HDG_CK(cudaGetLastError());
  return HDG_OK;
}

int hdg_mlp_target(int64_t n, const double* vhat_next, const double* vhat, const double* dvhat1, float* out,
                   void* stream) {
  if (!vhat_next || !vhat || !dvhat1 || !out || n < 0) {
    set_error("hdg_mlp_target: invalid argument");
    return HDG_ERR_INVALID_ARG;
  }
  k_mlp_target<<<nb(n), 256, 0, (cudaStream_t)stream>>>(n, vhat_next, vhat, dvhat1, out);
  HDG_CK(cudaGetLastError());
  return HDG_OK;
}

int hdg_mlp_apply_trace(hdg_ctx_t ctx, const double* Vhat, const double* dvh1, const float* pred, const float* tmean,
                        const float* tscale, double* Vhat_out, void* stream) {
  if (!ctx || !Vhat || !dvh1 || !pred || !tmean || !tscale || !Vhat_out) {
    set_error("hdg_mlp_apply_trace: null argument");
    return HDG_ERR_INVALID_ARG;
  }
  if (ctx->pm) {
    set_error("hdg_mlp_apply_trace: not built for meshes of mixed degree");
    return HDG_ERR_UNSUPPORTED;
  }
  if (ctx->scheme || !ctx->h_bface.empty()) {
    set_error("hdg_mlp_apply_trace: the per-face network works on two-sided face traces (periodic HDG) only");
    return HDG_ERR_UNSUPPORTED;
  }
  k_mlp_apply<<<nb(ctx->ntrace), 256, 0, (cudaStream_t)stream>>>(Vhat, dvh1, pred, tscale, tmean, ctx->F,
                                                                 ctx->NFN * ctx->M, Vhat_out);
  HDG_CK(cudaGetLastError());
  return HDG_OK;
}

}  // extern "C"
