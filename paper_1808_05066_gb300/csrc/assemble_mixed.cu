// Dispatch of the mixed-precision assemble + condense (asm_t5.cuh, condense_tc.cuh).
#include <algorithm>
#include <array>
#include <map>
#include <set>
#include <vector>

#include "element_small.cuh"
#include "asm_t5.cuh"
#include "condense_t5.cuh"
#include "condense_tc.cuh"
#include "ctx.hpp"

namespace hdg {

namespace {

constexpr int kSlices = 6;  // exact bf16 slices per operand in every tensor-core product
constexpr int64_t kMixedChunk = 8192;  // elements per chunk, unless their scratch is too large

}  // namespace

// The assembly's constant operand and its schedule (asm_t5.cuh), built on the first mixed call of a context.
struct T5Plan {
  T5Prog prog[2] = {};  // rows with a viscous part, rows without
  int nplane = 0, nparts = 1;
  df2* planes = nullptr;
  std::vector<void*> bufs;
  ~T5Plan() {
    for (void* b : bufs) cudaFree(b);
  }
};

void t5_plan_free(void* p) { delete static_cast<T5Plan*>(p); }

namespace {

template <class T>
int t5_upload(T5Plan& pl, const std::vector<T>& v, T** out) {
  HDG_CK(cudaMalloc(out, sizeof(T) * std::max<size_t>(1, v.size())));
  pl.bufs.push_back(*out);
  if (!v.empty()) HDG_CK(cudaMemcpy(*out, v.data(), sizeof(T) * v.size(), cudaMemcpyHostToDevice));
  return HDG_OK;
}

// One row program: its entries of k in chunks of at most 128, and per part and chunk the groups of up to 32
// columns that use the same steps of 16 entries.
template <class C>
int t5_program(hdg_ctx* ctx, T5Plan& pl, bool viscous, T5Prog& P, int* jobs_of_part, cudaStream_t s) {
  constexpr int D = C::D, M = C::M, NP = C::NP, NFN = C::NFN, NF = C::NF, NG = C::NG, NGF = C::NGF, NV = C::NV,
                NT = C::NT, NTN = NF * NFN;
  const RefElement& ref = ctx->mesh->m.ref;
  std::vector<int> pairs;
  for (int i = 0; i < M; ++i)
    for (int l = 0; l < M; ++l)
      if ((C::VISC && i > 0 && l > 0) == viscous) pairs.push_back(i << 8 | l);
  P = T5Prog{};
  if (pairs.empty()) return HDG_OK;
  P.rpe = (int)pairs.size();
  P.ept = 128 / P.rpe;
  // operators in order: faces first (the running sums of A', B' end with the volume); short ones share a step
  std::vector<std::vector<T5Entry>> chunks;
  std::vector<T5Entry> cur;
  auto block = [&](int kind, int f, int r, int r2, int n, int pt0) {
    if (n > 8)
      while (cur.size() % 16) cur.push_back({T5_PAD, 0, 0, 0, 0});
    if (cur.size() + n > 128) {
      chunks.push_back(cur);
      cur.clear();
    }
    for (int g = 0; g < n; ++g) cur.push_back({(short)kind, (short)f, (short)r, (short)r2, pt0 + g});
  };
  constexpr int face_room = (D + 3) * (NGF > 8 ? (NGF + 15) / 16 * 16 : NGF) + (NGF > 8 ? 15 : 0);
  static_assert(face_room <= 128 + 15, "a face's operators share one chunk: its C', D' entries are one product");
  for (int f = 0; f < NF; ++f) {
    if (cur.size() + face_room > 128) {
      if (!cur.empty()) chunks.push_back(cur);
      cur.clear();
    }
    block(T5_U0, f, 0, 0, NGF, f * NGF);
    if (viscous)
      for (int r2 = 0; r2 <= D; ++r2) block(T5_U2, f, 0, r2, NGF, f * NGF);
    block(T5_U1, f, 0, 0, NGF, f * NGF);
  }
  chunks.push_back(cur);
  cur.clear();
  block(T5_T0, 0, 0, 0, NG, 0);
  for (int r = 0; r < D; ++r) block(T5_T1, 0, r, 0, NG, 0);
  if (viscous)
    for (int r2 = 0; r2 <= D; ++r2)
      for (int r = 0; r < D; ++r) block(T5_T2, 0, r, r2, NG, 0);
  chunks.push_back(cur);
  P.nchunk = (int)chunks.size();
  std::vector<int> cstep(1, 0);
  std::vector<T5Entry> ent;
  for (auto& c : chunks) {
    cstep.push_back(cstep.back() + (int)(c.size() + 15) / 16);
    c.resize(128, {T5_PAD, 0, 0, 0, 0});
    ent.insert(ent.end(), c.begin(), c.end());
  }
  P.nsteps = cstep.back();
  // columns
  struct Col {
    T5ColDesc d;
    int node, plane, direct;  // node: the plane's test node
  };
  std::vector<char> on_face(NF * NP, 0);
  for (int f = 0; f < NF; ++f)
    for (int c = 0; c < NFN; ++c) on_face[f * NP + ref.face_nodes[f][c]] = 1;
  const int nplane = NP * NP + NP * NTN;
  std::vector<int> fin(nplane);  // A' then B'
  std::vector<Col> all;
  for (int a = 0; a < NP; ++a) {
    for (int j = 0; j < NP; ++j) {
      fin[a * NP + j] = a * M * NV + j * M;
      all.push_back({{T5_COL_A, 0, (short)a, (short)j, 0, 0}, a, a * NP + j, -1});
    }
    for (int f = 0; f < NF; ++f)
      for (int c = 0; c < NFN; ++c) {
        const int p = NP * NP + a * NTN + f * NFN + c;
        fin[p] = 1 << 28 | (a * M * NT + (f * NFN + c) * M);
        all.push_back({{T5_COL_B, (short)f, (short)a, (short)c, 0, 0}, a, p, -1});
      }
  }
  for (int f = 0; f < NF; ++f)
    for (int c = 0; c < NFN; ++c) {
      const int node = ref.face_nodes[f][c], row = (f * NFN + c) * M;
      for (int j = 0; j < NP; ++j)
        all.push_back({{T5_COL_FI, (short)f, (short)c, (short)j, 0, 0}, node, node * NP + j, 2 << 28 | (row * NV + j * M)});
      for (int f2 = 0; f2 < NF; ++f2)
        for (int c2 = 0; c2 < NFN; ++c2)
          all.push_back({{T5_COL_FT, (short)f, (short)c, (short)c2, (short)f2, 0}, node,
                         NP * NP + node * NTN + f2 * NFN + c2, 3 << 28 | (row * NT + (f2 * NFN + c2) * M)});
    }
  auto uses = [&](const T5ColDesc& d, const T5Entry& e) {
    switch (d.kind) {
      case T5_COL_A: return e.kind == T5_T0 || e.kind == T5_T1 || (e.kind == T5_T2 && e.r2 < D);
      case T5_COL_B: return e.kind == T5_T2 && e.r2 == (d.f ? d.f - 1 : D);
      case T5_COL_FI:
        return e.f == d.f && ((e.kind == T5_U0 && on_face[d.f * NP + d.j]) || (e.kind == T5_U2 && e.r2 < D));
      default: return e.f == d.f && ((e.kind == T5_U1 && d.f2 == d.f) || (e.kind == T5_U2 && e.r2 == (d.f2 ? d.f2 - 1 : D)));
    }
  };
  // jobs: columns of one kind and one set of steps, the planes' first additions before the others of a chunk and
  // their last ones behind; a plane fixes its quarter of a group and comes once in it at most
  auto quarter = [&](int p) { return p < NP * NP ? (p / NP + p % NP) & 3 : ((p - NP * NP) / NTN + (p - NP * NP) % NTN) & 3; };
  std::vector<std::vector<int>> masks(P.nchunk, std::vector<int>(all.size(), 0));
  std::vector<int> left(nplane, 0), seen(nplane, 0);
  std::vector<char> written(all.size(), 0);
  for (int ch = 0; ch < P.nchunk; ++ch)
    for (size_t k = 0; k < all.size(); ++k) {
      int mask = 0;
      for (int x = 0; x < 128; ++x)
        if (chunks[ch][x].kind != T5_PAD && uses(all[k].d, chunks[ch][x])) mask |= 1 << (x / 16);
      masks[ch][k] = mask;
      if (mask) {
        written[k] = 1;
        ++left[all[k].plane];
      }
    }
  // the test nodes' parts: the heaviest first, each to the lightest part (a column costs its steps and its additions)
  std::vector<int> weight(NP, 0), order(NP), load(pl.nparts, 0), part_of(NP);
  for (int ch = 0; ch < P.nchunk; ++ch)
    for (size_t k = 0; k < all.size(); ++k)
      if (masks[ch][k]) weight[all[k].node] += __builtin_popcount(masks[ch][k]) + 2;
  for (int a = 0; a < NP; ++a) order[a] = a;
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return weight[a] > weight[b]; });
  for (int a : order) {
    part_of[a] = (int)(std::min_element(load.begin(), load.end()) - load.begin());
    load[part_of[a]] += weight[a];
  }
  const T5Col none = {nplane * 128 * (int)sizeof(df2), -1, 0.f, -1};
  std::vector<int> jobs, wstep, zero;  // zero: entries that vanish for these pairs
  std::vector<int2> parts;
  std::vector<T5Col> cols;
  std::vector<T5ColDesc> desc;
  int wsteps = 0;
  for (int part = 0; part < pl.nparts; ++part) {
    parts.push_back(make_int2((int)jobs.size(), (int)zero.size()));
    std::set<int> before;  // planes of the job before
    for (int ch = 0; ch < P.nchunk; ++ch) {
      std::map<std::array<int, 4>, std::vector<int>> groups;  // (not first, last, kind, steps)
      for (size_t k = 0; k < all.size(); ++k)
        if (masks[ch][k] && part_of[all[k].node] == part) {
          const int p = all[k].plane;
          groups[{seen[p] ? 1 : 0, --left[p] ? 0 : 1, all[k].d.kind, masks[ch][k]}].push_back((int)k);
          ++seen[p];
        }
      if (groups.empty()) continue;
      for (auto& gr : groups) {
        std::vector<int> rest = gr.second;
        while (!rest.empty()) {
          int job = gr.first[3] | ch << 8 | (gr.first[0] ? 0 : T5_FIRST) | (gr.first[1] ? T5_LAST : 0) |
                    gr.first[2] << T5_KIND;
          wstep.push_back(wsteps);
          for (int m = gr.first[3]; m; m &= m - 1) ++wsteps;
          cols.resize((jobs.size() + 1) * kT5Cols, none);
          desc.resize((jobs.size() + 1) * kT5Cols, {T5_COL_NONE, 0, 0, 0, 0, 0});
          int fill[4] = {0, 0, 0, 0};
          std::set<int> taken;
          std::vector<int> later;
          for (int k : rest) {
            const Col& c = all[k];
            const int h = quarter(c.plane);
            if (fill[h] == kT5Q || taken.count(c.plane)) {
              later.push_back(k);
              continue;
            }
            taken.insert(c.plane);
            if (before.count(c.plane)) job |= T5_HAZARD;
            const size_t at = jobs.size() * kT5Cols + h * kT5Q + fill[h]++;
            cols[at] = {c.plane * 128 * (int)sizeof(df2), c.direct < 0 ? -1 : (c.direct & 0xfffffff) * 8, 0.f,
                        (fin[c.plane] & 0xfffffff) * 8};
            desc[at] = c.d;
          }
          rest.swap(later);
          before.swap(taken);
          jobs.push_back(job);
        }
      }
      jobs.back() |= T5_CLOSES;
    }
    for (int p = 0; p < nplane; ++p)
      if (!seen[p] && part_of[p < NP * NP ? p / NP : (p - NP * NP) / NTN] == part) zero.push_back(fin[p]);
    for (size_t k = 0; k < all.size(); ++k)
      if (!written[k] && all[k].direct >= 0 && part_of[all[k].node] == part) zero.push_back(all[k].direct);
    jobs_of_part[part] += (int)jobs.size() - parts[part].x;
  }
  parts.push_back(make_int2((int)jobs.size(), (int)zero.size()));
  for (int k = 0; k < 2 * kT5Cols; ++k) cols.push_back(none);
  pl.nplane = nplane;
  int *dj, *dc, *dp, *dws, *dz;
  int2* dpart;
  T5Entry* de;
  T5ColDesc* dd;
  unsigned char* dw;
  int rc;
  if ((rc = t5_upload(pl, jobs, &dj)) || (rc = t5_upload(pl, cols, &P.cols)) || (rc = t5_upload(pl, desc, &dd)) ||
      (rc = t5_upload(pl, ent, &de)) || (rc = t5_upload(pl, cstep, &dc)) || (rc = t5_upload(pl, pairs, &dp)) ||
      (rc = t5_upload(pl, wstep, &dws)) || (rc = t5_upload(pl, zero, &dz)) || (rc = t5_upload(pl, parts, &dpart)))
    return rc;
  P.wstep = dws;
  P.zero = dz;
  P.part = dpart;
  HDG_CK(cudaMalloc(&dw, (size_t)wsteps * kT5Slices * kT5BTile));
  pl.bufs.push_back(dw);
  P.jobs = dj;
  P.ent = de;
  P.cstep = dc;
  P.pairs = dp;
  P.W = dw;
  k_t5_weights<C><<<(unsigned)jobs.size(), 256, 0, s>>>(ctx->T, P, dd, dw);
  HDG_CK(cudaGetLastError());
  return HDG_OK;
}

// Parts of a tile's planes for a chunk of n elements: as many as there are idle SMs per tile, but no more than leave
// every part the same number of test nodes (20 nodes in 15 parts take as long as in 10).
template <class C>
int t5_parts(int64_t n, int num_sms) {
  constexpr int M = C::M, MV = M - 1, VP = C::VISC ? MV * MV : 0;  // pairs with a viscous part
  const auto tiles = [&](int pairs) { return pairs ? (n + 128 / pairs - 1) / (128 / pairs) : 0; };
  const int64_t room = num_sms / (tiles(VP) + tiles(M * M - VP));
  if (room < 2) return 1;
  const int64_t nodes = (C::NP + room - 1) / room;  // of a part
  return (int)((C::NP + nodes - 1) / nodes);
}

template <class C>
int t5_plan(hdg_ctx* ctx, cudaStream_t s) {
  if (ctx->t5_plan) return HDG_OK;
  auto* pl = new T5Plan();
  pl->nparts = t5_parts<C>(ctx->chunk ? ctx->chunk : std::min<int64_t>(ctx->E, kMixedChunk), ctx->num_sms);
  std::vector<int> jobs(pl->nparts, 0);
  int rc = HDG_OK;
  if ((rc = t5_program<C>(ctx, *pl, true, pl->prog[0], jobs.data(), s)) ||
      (rc = t5_program<C>(ctx, *pl, false, pl->prog[1], jobs.data(), s))) {
    delete pl;
    return rc;
  }
  if (cudaMalloc(&pl->planes, sizeof(df2) * (size_t)ctx->num_sms * (pl->nplane + 1) * 128) != cudaSuccess) {
    delete pl;
    return cuda_fail(cudaGetLastError(), "cudaMalloc (assembly planes)");
  }
  pl->bufs.push_back(pl->planes);
  if (*std::max_element(jobs.begin(), jobs.end()) > kT5MaxJobs) {
    delete pl;
    set_error("assemble_condense: the assembly's schedule is longer than its table");
    return HDG_ERR_UNSUPPORTED;
  }
  // later calls may come on other streams
  if (cudaStreamSynchronize(s) != cudaSuccess) {
    delete pl;
    return cuda_fail(cudaGetLastError(), "assembly operands");
  }
  ctx->t5_plan = pl;
  return HDG_OK;
}

// tiles and scratch bytes (slices, row exponents) of a program over n elements
int64_t t5_tiles(const T5Prog& P, int64_t n) { return P.ept ? (n + P.ept - 1) / P.ept : 0; }
size_t t5_slice_bytes(const T5Prog& P, int64_t n) {
  return (size_t)t5_tiles(P, n) * P.nsteps * kT5Slices * kT5ATile;
}
size_t t5_exp_bytes(const T5Prog& P, int64_t n) { return (size_t)t5_tiles(P, n) * P.nchunk * 128 * sizeof(int); }

template <class C>
void run_asm_t5(hdg_ctx* ctx, const T5Plan& pl, const T5Prog (&pr)[2], const AssembleArgs& a, cudaStream_t s) {
  {
    LaunchScope ls(ctx, HDG_KERNEL_MIXED_OPERATORS, s);
    const int64_t blocks = (int64_t)pr[0].ntile * pr[0].nchunk + (int64_t)pr[1].ntile * pr[1].nchunk + a.ne;
    k_t5_rows<C><<<(unsigned)blocks, 256, 0, s>>>(a, ctx->T, pr[0], pr[1]);
  }
  LaunchScope ls(ctx, HDG_KERNEL_MIXED_ASSEMBLE, s);
  const int grid = std::min(ctx->num_sms / pl.nparts, pr[0].ntile + pr[1].ntile) * pl.nparts;
  k_asm_t5<C><<<grid, kT5Threads, kT5Smem, s>>>(a, pr[0], pr[1], pl.planes, pl.nplane, pl.nparts);
}

// One compiled shape of the condensation kernel, with the prep kernel that lays out its operands.
struct CondVariant {
  int threads;
  size_t smem;
  void (*kernel)(AssembleArgs);
  int ctas_per_element;
  void (*prep)(AssembleArgs);
  unsigned grid(int64_t ne) const { return (unsigned)(ne * ctas_per_element); }
};

template <class C, int NTH>
CondVariant make_cond_variant() {
  return CondVariant{NTH, CondTC<C, NTH, kSlices>::bytes, &k_condense_tc<C, NTH, kSlices>, 1,
                     &k_condense_prep<C, kSlices, false>};
}

// 16-column blocks, two CTAs per SM
template <class C>
CondVariant make_cond_variant2() {
  using Q = CondTC2<C, 256, kSlices>;
  return CondVariant{256, Q::bytes, &k_condense_tc2<C, 256, kSlices>, Q::CTAS, &k_condense_prep<C, kSlices, false>};
}

// tcgen05 products with TMEM accumulators, 32-column blocks, one CTA per SM
template <class C>
CondVariant make_cond_variant_t5() {
  using Q = CondT5<C, kSlices>;
  return CondVariant{Q::NTH, Q::bytes, &k_condense_t5<C, kSlices>, 1, &k_condense_prep<C, kSlices, true>};
}

// Times `launch` once on the stream (the chunk's outputs are rewritten each time).
template <class F>
int time_launch(cudaStream_t s, F launch, float* ms) {
  cudaEvent_t t0, t1;
  HDG_CK(cudaEventCreate(&t0));
  HDG_CK(cudaEventCreate(&t1));
  HDG_CK(cudaEventRecord(t0, s));
  launch();
  HDG_CK(cudaEventRecord(t1, s));
  HDG_CK(cudaEventSynchronize(t1));
  HDG_CK(cudaGetLastError());
  HDG_CK(cudaEventElapsedTime(ms, t0, t1));
  cudaEventDestroy(t0);
  cudaEventDestroy(t1);
  return HDG_OK;
}

template <class C>
int run_mixed(hdg_ctx* ctx, const double* V, const double* Vhat, const double* hist, double mass_coef, double* S,
              double* g, double* recov, double* R, int32_t* status, cudaStream_t s) {
  if (!ctx->num_sms) HDG_CK(cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, ctx->device));
  if (int rc = t5_plan<C>(ctx, s)) return rc;
  const T5Plan& pl = *static_cast<T5Plan*>(ctx->t5_plan);
  T5Prog pr[2] = {pl.prog[0], pl.prog[1]};
  using TC = CondTC<C, 256, kSlices>;
  // the recomputation of flagged blocks may need more room for its point data
  const bool sm = small::small_elements<C>(ctx->E, ctx->num_sms);
  size_t vol, face, rvol, rface;
  point_doubles<C>(false, &vol, &face);
  point_doubles<C>(sm, &rvol, &rface);
  const size_t pts = std::max(vol + face, rvol + rface);
  const size_t per_pt = sizeof(double) * (pts + (size_t)C::NV * C::NV + (size_t)C::NT * C::NV);
  const size_t slice_bytes = std::max(sizeof(uint4) * TC::slice_uint4, CondT5<C, kSlices>::slice_bytes);
  const size_t per_rows = t5_slice_bytes(pr[0], 1024) / 1024 + t5_slice_bytes(pr[1], 1024) / 1024;
  const size_t per = per_pt + slice_bytes + sizeof(float) * TC::prep_floats + per_rows;
  if (ctx->chunk == 0) {
    int64_t ch = std::min<int64_t>(ctx->E, kMixedChunk);
    while (ch > 256 && per * ch > ((size_t)16 << 30)) ch /= 2;
    ctx->chunk = ch;
  }
  size_t need = (per - per_rows) * ctx->chunk + 4096;  // + room to align the parts of the scratch
  for (const T5Prog& P : pr) need += t5_slice_bytes(P, ctx->chunk) + t5_exp_bytes(P, ctx->chunk) + 1024;
  if (ctx->scr_bytes < need) {
    if (ctx->d_scr) cudaFree(ctx->d_scr);
    ctx->d_scr = nullptr;
    ctx->scr_bytes = 0;
    HDG_CK(cudaMalloc(&ctx->d_scr, need));
    ctx->scr_bytes = need;
  }
  const CondVariant cvariants[] = {make_cond_variant<C, 256>(), make_cond_variant<C, 512>(), make_cond_variant2<C>(),
                                   make_cond_variant_t5<C>()};
  constexpr int NCVAR = 4;
  if (!ctx->attr_mixed) {  // per context, hence per device
    HDG_CK(cudaFuncSetAttribute(k_asm_t5<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kT5Smem));
    for (const CondVariant& v : cvariants) {
      HDG_CK(cudaFuncSetAttribute(v.kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v.smem));
      HDG_CK(cudaFuncSetAttribute(v.kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100));
    }
    HDG_CK(cudaFuncSetAttribute(k_condense_prep<C, kSlices, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)TC::prep_bytes));
    HDG_CK(cudaFuncSetAttribute(k_condense_prep<C, kSlices, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)TC::prep_bytes));
    // the FP64 kernels of the flagged-only recomputation
    if (int rc = fp64_attributes<C>()) return rc;
    ctx->attr_mixed = true;
  }
  AssembleArgs a{};
  a.V = V;
  a.Vhat = Vhat;
  a.tgidx = ctx->d_tgidx;
  a.geo = ctx->d_geo;
  a.hist = hist;
  a.mass_coef = mass_coef;
  a.S = S;
  a.g = g;
  a.recov = recov;
  a.R = R;
  a.status = status;
  a.refine_tol = (float)ctx->refine_tol;
  a.stall_first_copy = (ctx->t5_stall ? kStallCondense : 0) | (ctx->asm_stall ? kStallAssembly : 0);
  const int64_t ch = ctx->chunk;
  a.ptv = ctx->d_scr;
  a.ptf = a.ptv + ch * vol;
  a.Ap = a.ptv + ch * pts;
  a.Cp = a.Ap + ch * C::NV * C::NV;
  {  // 256-byte aligned start of the slice scratch (chunk sizes may be odd)
    const uintptr_t p = reinterpret_cast<uintptr_t>(a.Cp + ch * C::NT * C::NV);
    a.oz = reinterpret_cast<uint4*>((p + 255) & ~(uintptr_t)255);
    const uintptr_t q = reinterpret_cast<uintptr_t>(a.oz) + ch * slice_bytes;
    a.prep = reinterpret_cast<float*>((q + 255) & ~(uintptr_t)255);
    uintptr_t r = reinterpret_cast<uintptr_t>(a.prep + ch * TC::prep_floats);
    for (T5Prog& P : pr) {
      r = (r + 255) & ~(uintptr_t)255;
      P.T = reinterpret_cast<unsigned char*>(r);
      r += t5_slice_bytes(P, ch);
      P.erow = reinterpret_cast<int*>(r);
      r += t5_exp_bytes(P, ch);
    }
  }
  for (int64_t e0 = 0; e0 < ctx->E; e0 += ch) {
    a.e0 = e0;
    a.ne = std::min<int64_t>(ch, ctx->E - e0);
    {
      int rc_s = HDG_OK;
      a.S = chunk_S(ctx, S, e0, s, &rc_s);
      if (rc_s) return rc_s;
    }
    {
      LaunchScope ls(ctx, HDG_KERNEL_POINTWISE, s);
      launch_pointwise<C>(a, ctx->T, ctx->ph, s);
    }
    for (T5Prog& P : pr) P.ntile = (int)t5_tiles(P, a.ne);
    if (ctx->cond_variant < 0 && a.ne >= 512) {
      // autotune on this chunk: time every compiled shape of the condensation
      float best = 1e30f;
      int best_i = 0;
      for (int i = 0; i < NCVAR; ++i) {
        // the condensation overwrites its inputs: assemble again before each trial
        run_asm_t5<C>(ctx, pl, pr, a, s);
        const CondVariant& cv = cvariants[i];
        cv.prep<<<(unsigned)a.ne, TC::PTH, TC::prep_bytes, s>>>(a);
        float ms = 0.f;
        int rc = time_launch(s, [&] { cv.kernel<<<cv.grid(a.ne), cv.threads, cv.smem, s>>>(a); }, &ms);
        if (rc) return rc;
        if (ms < best) {
          best = ms;
          best_i = i;
        }
      }
      ctx->cond_variant = best_i;
      ctx->cond_variant_threads = cvariants[best_i].threads;
    }
    run_asm_t5<C>(ctx, pl, pr, a, s);
    if (int rc_b = boundary_patch(ctx, a, HDG_PREC_MIXED, s)) return rc_b;
    const CondVariant& cv = cvariants[ctx->cond_variant < 0 ? 0 : ctx->cond_variant];
    {
      LaunchScope ls(ctx, HDG_KERNEL_MIXED_PREP, s);
      cv.prep<<<(unsigned)a.ne, TC::PTH, TC::prep_bytes, s>>>(a);
    }
    {
      LaunchScope ls(ctx, HDG_KERNEL_MIXED_CONDENSE, s);
      cv.kernel<<<cv.grid(a.ne), cv.threads, cv.smem, s>>>(a);
    }
    if (ctx->refine_fallback) {
      // blocks whose refinement missed its tolerance (or whose condensation gave up a wait) are
      // recomputed by the FP64 kernels, from the same point tensors or those of small elements; every other CTA returns
      // at once
      AssembleArgs f = a;
      f.only_flag = HDG_STATUS_REFINE | HDG_STATUS_TIMEOUT;
      if (sm) {
        f.ptf = f.ptv + ch * rvol;
        LaunchScope ls(ctx, HDG_KERNEL_POINTWISE, s);
        fp64_pointwise<C>(sm, f, ctx->T, ctx->ph, s);
      }
      {
        LaunchScope ls(ctx, HDG_KERNEL_ASSEMBLE, s);
        fp64_assemble<C>(sm, f, ctx->T, s);
      }
      if (int rc_b = boundary_patch(ctx, f, HDG_PREC_FP64, s)) return rc_b;
      {
        LaunchScope ls(ctx, HDG_KERNEL_CONDENSE, s);
        fp64_condense<C>(sm, f, s);
      }
    }
    if (int rc_d = chunk_done(ctx, e0, a.ne, s)) return rc_d;
  }
  HDG_CK(cudaGetLastError());
  return HDG_OK;
}

}  // namespace

#define HDG_MIX_CASE(D, P, VISC)                                                                    \
  if (ctx->dim == D && ctx->p == P && ctx->K == P + 1 && ctx->visc == VISC)                        \
    return run_mixed<Cfg<D, P, P + 1, VISC>>(ctx, V, Vhat, hist, mass_coef, S, g, recov, R, status, s);

int assemble_condense_mixed(hdg_ctx* ctx, const double* V, const double* Vhat, const double* hist,
                            double mass_coef, double* S, double* g, double* recov, double* R, int32_t* status,
                            cudaStream_t s) {
  HDG_MIX_CASE(2, 2, false)
  HDG_MIX_CASE(2, 3, true)
  HDG_MIX_CASE(2, 4, true)
  HDG_MIX_CASE(3, 1, true)
  HDG_MIX_CASE(3, 2, true)
  HDG_MIX_CASE(3, 3, true)
  set_error("assemble_condense: mixed form not compiled for this configuration");
  return HDG_ERR_UNSUPPORTED;
}

}  // namespace hdg
