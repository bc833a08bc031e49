// fp32 configuration of the SwitchHead layer: launch sequences of the forward and the backward pass.
// Projections on the tensor cores in split bf16 (sh_f32_gemm.cuh), attention on the CUDA cores
// (sh_f32_attn.cuh), selection and sort in one launch (sh_f32_select.cuh).
#include "sh_internal.cuh"
#include "sh_launch.cuh"
#include "sh_f32_gemm.cuh"
#include "sh_f32_attn.cuh"
#include "sh_f32_select.cuh"

using namespace shtc;

namespace {

int sm_count(sh_layer* L) {
  if (L->sm_count == 0) {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess) L->sm_count = n;
    else { cudaGetLastError(); return 148; }
  }
  return L->sm_count;
}

// Row tiles of one head in a side's tile table (sh_f32_select_kernel).
int head_tiles(const ShDims& d) { return (int)(((long long)d.N * d.k + 127ll * d.E) / 128); }

// 64- or 128-column tiles.  A 128-column tile costs about 1.6 times a 64-column one (the row operand is
// split once either way), so the narrow tile is taken where the wide ones would leave SMs idle.
bool wide_tile(sh_layer* L, long rows, int cols, int per_head_cols) {
  const long n128 = rows * cols * ((per_head_cols + 127) / 128), n64 = rows * cols * ((per_head_cols + 63) / 64);
  const long sms = sm_count(L);
  const long w128 = (n128 + sms - 1) / sms, w64 = (n64 + sms - 1) / sms;
  return 8 * w128 <= 5 * w64;
}

template <int MODE>
int launch_x(XGemmArgs& g, bool wide, dim3 grid, cudaStream_t st) {
  if (grid.x == 0 || grid.y == 0 || grid.z == 0) return SH_OK;
  if (wide) {
    if (int rc = set_smem(sh_f32_gemm_kernel<128, MODE>, XGemmSmem<128>::TOTAL)) return rc;
    return launch_k(true, sh_f32_gemm_kernel<128, MODE>, grid, dim3(XG_THREADS), XGemmSmem<128>::TOTAL, st, g);
  }
  if (int rc = set_smem(sh_f32_gemm_kernel<64, MODE>, XGemmSmem<64>::TOTAL)) return rc;
  return launch_k(true, sh_f32_gemm_kernel<64, MODE>, grid, dim3(XG_THREADS), XGemmSmem<64>::TOTAL, st, g);
}

// Column tiles over `cols` columns: how many, and how wide (a multiple of 16).
void col_tiles(XGemmArgs& g, int cols, bool wide) {
  const int bn = wide ? 128 : 64;
  g.nsub = (cols + bn - 1) / bn;
  g.sub_cols = ((cols + g.nsub - 1) / g.nsub + 15) / 16 * 16;
}

XGemmArgs base_args(sh_layer* L, const void* x) {
  char* ws = L->ws;
  const ShDims& d = L->d;
  XGemmArgs g{};
  g.d = d;
  g.x = (const float*)x;
  g.ahat = (const float*)(ws + L->o.ahat);
  g.wqk = (const float*)(ws + L->o.wqk); g.wgate = (const float*)(ws + L->o.wgate);
  g.wv = (const float*)(ws + L->o.wv); g.wo = (const float*)(ws + L->o.wo);
  g.ldz = sh_f32_ldz(d);
  g.ksplit = 1;
  g.q = (float*)(ws + L->o.q); g.k = (float*)(ws + L->o.k); g.v = (float*)(ws + L->o.v); g.z = (float*)(ws + L->o.f32z);
  g.qscale = 1.4426950408889634f / sqrtf((float)d.Dt);
  g.rope = L->rope ? (const float2*)(ws + L->o.rope) : nullptr;
  g.vec_dy = g.vec_out = 1;
  g.status = (int*)(ws + L->o.status);
  return g;
}

// The lists, gates and row tiles of one side (0: source, 1: destination; one side with a shared selection).
void use_side(XGemmArgs& g, sh_layer* L, int side) {
  const ShDims& d = L->d;
  char* ws = L->ws;
  if (d.sides == 1) side = 0;
  const size_t s = (size_t)side * d.H * d.N * d.k;
  g.lists = (const int*)(ws + L->o.lists) + s;
  g.lgate = (const float*)(ws + L->o.lgate) + s;
  g.offsets = (const int*)(ws + L->o.offsets) + (size_t)side * d.H * (d.E + 1);
  g.tiles = (const ShTile*)(ws + L->o.tiles) + (size_t)side * d.max_tiles;
}

// x [Wq | Wk | Wgate]: `groups` heads' column groups from `first` on, and the gate columns if asked.
int launch_qk(sh_layer* L, const void* x, int first, int groups, bool gates, float* zero0, long n0, float* zero1, long n1, cudaStream_t st) {
  const ShDims& d = L->d;
  XGemmArgs g = base_args(L, x);
  g.qk_first = first; g.qk_groups = groups;
  const bool wide = groups > 0 && wide_tile(L, d.nblk, groups, d.Dt);
  col_tiles(g, d.Dt, wide);
  g.zero0 = zero0; g.nzero0 = n0 / 4; g.zero1 = zero1; g.nzero1 = n1 / 4;
  const int gt = gates ? (d.G + (wide ? 127 : 63)) / (wide ? 128 : 64) : 0;
  L->launches += 1;
  return launch_x<X_QK>(g, wide, dim3(d.nblk, groups * g.nsub + gt), st);
}

int launch_select(sh_layer* L, cudaStream_t st) {
  const ShDims& d = L->d;
  char* ws = L->ws;
  L->launches += 1;
  return launch_k(true, sh_f32_select_kernel, dim3(d.sides * d.H), dim3(1024), 0, st, (const float*)(ws + L->o.f32z), sh_f32_ldz(d),
                  (const float*)(ws + L->o.gbias), (int*)(ws + L->o.idx), (float*)(ws + L->o.gate), (int*)(ws + L->o.offsets),
                  (int*)(ws + L->o.lists), (float*)(ws + L->o.lgate), (ShTile*)(ws + L->o.tiles), d, head_tiles(d));
}

// dst += gate x W^T over a side's expert lists: value experts, and query / key experts where a layer has them.
int launch_v(sh_layer* L, const void* x, int side, const float* w, float* dst, float scale, cudaStream_t st) {
  const ShDims& d = L->d;
  XGemmArgs g = base_args(L, x);
  use_side(g, L, side);
  g.wv = w; g.v = dst; g.vscale = scale;
  const bool wide = wide_tile(L, (long)d.H * head_tiles(d), 1, d.Dt);
  col_tiles(g, d.Dt, wide);
  L->launches += 1;
  return launch_x<X_V>(g, wide, dim3(d.H * head_tiles(d), g.nsub), st);
}

template <int D>
int launch_attn_t(sh_layer* L, cudaStream_t st) {
  const ShDims& d = L->d;
  char* ws = L->ws;
  if (int rc = set_smem(sh_f32_attn_kernel<D>, FAttnSmem<D>::TOTAL)) return rc;
  const int nq = (d.T - d.Tc + 31) / 32;
  return launch_k(true, sh_f32_attn_kernel<D>, dim3((unsigned)nq * d.B * d.H), dim3(256), FAttnSmem<D>::TOTAL, st,
                  (const float*)(ws + L->o.q), (const float*)(ws + L->o.k), (const float*)(ws + L->o.v), (float*)(ws + L->o.ahat),
                  (float*)(ws + L->o.f32stats), d);
}

int launch_attn(sh_layer* L, cudaStream_t st) {
  L->launches += 1;
  switch (L->d.D) {
    case 32: return launch_attn_t<32>(L, st);
    case 64: return launch_attn_t<64>(L, st);
    case 128: return launch_attn_t<128>(L, st);
    default: return launch_attn_t<256>(L, st);
  }
}

struct BwBuffers { float *dq, *dk, *dv, *dahat, *ds, *dz, *dsum; size_t cleared; };
BwBuffers bw_buffers(sh_layer* L) {
  const ShDims& d = L->d;
  const size_t nhd = (size_t)d.N * d.H * d.D;
  BwBuffers b;
  b.dq = (float*)(L->ws + L->o.bw); b.dk = b.dq + nhd; b.dv = b.dk + nhd; b.dahat = b.dv + nhd;
  b.dz = b.dahat + nhd;
  b.ds = b.dz + (size_t)d.N * sh_f32_ldz(d);
  b.dsum = b.ds + (size_t)2 * d.N * d.H * d.k;
  b.cleared = (size_t)(b.dsum - b.dq);
  return b;
}

template <int D>
int launch_attn_bw_t(sh_layer* L, const BwBuffers& w, cudaStream_t st) {
  const ShDims& d = L->d;
  char* ws = L->ws;
  if (int rc = set_smem(sh_f32_attn_bw_kernel<D>, FBwSmem<D>::TOTAL)) return rc;
  // A block's run of query tiles: short enough that the blocks fill the device about four times over,
  // at least one tile for each of its two thread groups.
  const int qt = (d.T + FBwSmem<D>::TQ - 1) / FBwSmem<D>::TQ, kt = (d.T + 31) / 32;
  const long units = (long)kt * d.B * d.H * qt / (d.causal ? 2 : 1);
  long run = units / (4l * sm_count(L));
  run = run < 2 ? 2 : run > qt ? qt : run;
  return launch_k(true, sh_f32_attn_bw_kernel<D>, dim3((unsigned)kt * d.B * d.H, (unsigned)((qt + run - 1) / run)), dim3(256), FBwSmem<D>::TOTAL, st,
                  (const float*)(ws + L->o.q), (const float*)(ws + L->o.k), (const float*)(ws + L->o.v), (const float*)w.dahat,
                  (const float*)(ws + L->o.f32stats), (const float*)w.dsum, w.dq, w.dk, w.dv, d, (int)run);
}

// Parts of a contraction over tokens: enough blocks for the device, at least four steps each.
int k_parts(sh_layer* L, long blocks, long steps) {
  long p = (sm_count(L) + blocks - 1) / blocks;
  const long most = steps / 4 < 1 ? 1 : steps / 4;
  p = p > most ? most : p;
  return p < 1 ? 1 : (int)p;
}

}  // namespace

int sh_f32_gate_sort(sh_layer* L, const void* x, cudaStream_t st) {
  if (int rc = launch_qk(L, x, 0, 0, true, nullptr, 0, nullptr, 0, st)) return rc;
  return launch_select(L, st);
}

int sh_f32_forward(sh_layer* L, const void* x, void* out, cudaStream_t st) {
  const ShDims& d = L->d;
  char* ws = L->ws;
  const long nhd = (long)d.N * d.H * d.D, nout = (long)sh_out_rows(d) * d.M;
  const float qscale = 1.4426950408889634f / sqrtf((float)d.Dt);
  float* v = (float*)(ws + L->o.v);
  int rc;
  // Dense queries and keys (a layer with query / key experts has none of its own), and the gate logits;
  // a stage-timed pass computes the logits in a launch of their own so that its boundaries mean something.
  const int first = L->moe_q ? d.H : 0, groups = (L->moe_q ? 0 : d.H) + (L->moe_k ? 0 : d.H);
  sh_mark(L, 0, st);
  if (L->ev) {
    if ((rc = sh_f32_gate_sort(L, x, st))) return rc;
    sh_mark(L, 1, st);
    if (groups) { if ((rc = launch_qk(L, x, first, groups, false, v, nhd, (float*)out, nout, st))) return rc; }
    else {
      SH_CUDA_CHECK(cudaMemsetAsync(v, 0, (size_t)nhd * 4, st));
      SH_CUDA_CHECK(cudaMemsetAsync(out, 0, (size_t)nout * 4, st));
    }
  } else {
    if ((rc = launch_qk(L, x, first, groups, true, v, nhd, (float*)out, nout, st))) return rc;
    if ((rc = launch_select(L, st))) return rc;
  }
  if (L->moe_k) {
    SH_CUDA_CHECK(cudaMemsetAsync(ws + L->o.k, 0, (size_t)nhd * 4, st));
    if ((rc = launch_v(L, x, 0, (const float*)(ws + L->o.wk_e), (float*)(ws + L->o.k), 0.f, st))) return rc;
  }
  if (L->moe_q) {
    SH_CUDA_CHECK(cudaMemsetAsync(ws + L->o.q, 0, (size_t)nhd * 4, st));
    if ((rc = launch_v(L, x, 1, (const float*)(ws + L->o.wq_e), (float*)(ws + L->o.q), qscale, st))) return rc;
  }
  sh_mark(L, 2, st);
  if ((rc = launch_v(L, x, 0, (const float*)(ws + L->o.wv), v, 0.f, st))) return rc;
  sh_mark(L, 3, st);
  // (the relative-position term of Transformer-XL is in the one-warp-per-query kernel only)
  if ((rc = L->xl_positions ? sh_simt_attention_f32(L, st) : launch_attn(L, st))) return rc;
  sh_mark(L, 4, st);
  XGemmArgs g = base_args(L, x);
  use_side(g, L, 1);
  g.y = (float*)out;
  const bool wide = wide_tile(L, (long)d.H * head_tiles(d), 1, d.M);
  col_tiles(g, d.M, wide);
  if ((rc = launch_x<X_O>(g, wide, dim3(d.H * head_tiles(d), g.nsub), st))) return rc;
  L->launches += 1;
  sh_mark(L, 5, st);
  SH_CUDA_CHECK(cudaGetLastError());
  return SH_OK;
}

int sh_f32_backward(sh_layer* L, const void* x, const float* dout, float* dx, float* dWq, float* dWk, float* dWv,
                    float* dWo, float* dWs, float* dWd, cudaStream_t st) {
  const ShDims& d = L->d;
  char* ws = L->ws;
  const BwBuffers w = bw_buffers(L);
  const int ht = head_tiles(d), mt = (d.M + 127) / 128, dt = (d.Dt + 127) / 128;
  int rc;
  L->launches = 0;
  SH_CUDA_CHECK(cudaMemsetAsync(w.dq, 0, w.cleared * 4, st));
  SH_CUDA_CHECK(cudaMemsetAsync(dx, 0, (size_t)d.N * d.M * 4, st));
  XGemmArgs g = base_args(L, x);
  g.dy = dout; g.dq = w.dq; g.dk = w.dk; g.dv = w.dv; g.dz = w.dz; g.dahat = w.dahat; g.dx = dx;
  g.dWq = dWq; g.dWk = dWk; g.dWv = dWv; g.dWo = dWo; g.dWs = dWs; g.dWd = dWd;
  auto aligned = [](const void* p) { return (uintptr_t)p % 16 == 0; };
  g.vec_dy = aligned(dout);
  g.vec_out = aligned(dx) && aligned(dWq) && aligned(dWk) && aligned(dWv) && aligned(dWo);
  const size_t list_side = (size_t)d.H * d.N * d.k;
  // output experts: dAhat and the destination gates' gradients
  use_side(g, L, 1);
  g.ds = w.ds + list_side;
  bool wide = wide_tile(L, (long)d.H * ht, 1, d.Dt);
  col_tiles(g, d.Dt, wide);
  if ((rc = launch_x<X_DA>(g, wide, dim3(d.H * ht, g.nsub), st))) return rc;
  // attention
  const int rows = d.N * d.H;
  if ((rc = launch_k(true, sh_f32_rowdot_kernel, dim3((unsigned)((rows + 7) / 8)), dim3(256), 0, st, (const float*)w.dahat,
                     (const float*)(ws + L->o.ahat), w.dsum, rows, d.D))) return rc;
  rc = d.D == 32 ? launch_attn_bw_t<32>(L, w, st) : d.D == 64 ? launch_attn_bw_t<64>(L, w, st)
     : d.D == 128 ? launch_attn_bw_t<128>(L, w, st) : launch_attn_bw_t<256>(L, w, st);
  if (rc) return rc;
  // value experts: their part of dx, and the source gates' gradients
  use_side(g, L, 0);
  g.ds = w.ds;
  wide = wide_tile(L, (long)d.H * ht, 1, d.M);
  col_tiles(g, d.M, wide);
  if ((rc = launch_x<X_DR>(g, wide, dim3(d.H * ht, g.nsub), st))) return rc;
  if ((rc = launch_k(true, sh_f32_dz_kernel, dim3((unsigned)(((long)d.N * d.k + 255) / 256), 2 * d.H), dim3(256), 0, st, (const float*)w.ds,
                     (const int*)(ws + L->o.lists), (const float*)(ws + L->o.lgate), (const int*)(ws + L->o.offsets), w.dz, g.ldz, d))) return rc;
  // queries, keys and gates: the rest of dx, then the weight gradients
  wide = wide_tile(L, d.nblk, 1, d.M);
  col_tiles(g, d.M, wide);
  if ((rc = launch_x<X_DX>(g, wide, dim3(d.nblk, g.nsub), st))) return rc;
  g.qk_first = 0; g.qk_groups = 2 * d.H;
  wide = wide_tile(L, mt, 2 * d.H, d.Dt);
  col_tiles(g, d.Dt, wide);
  const int ct = g.qk_groups * g.nsub + (d.G + (wide ? 127 : 63)) / (wide ? 128 : 64);
  g.ksplit = k_parts(L, (long)mt * ct, (d.N + 63) / 64);
  if (g.ksplit > 1) {
    SH_CUDA_CHECK(cudaMemsetAsync(dWq, 0, (size_t)d.H * d.M * d.Dt * 4, st));
    SH_CUDA_CHECK(cudaMemsetAsync(dWk, 0, (size_t)d.H * d.M * d.Dt * 4, st));
    SH_CUDA_CHECK(cudaMemsetAsync(dWs, 0, (size_t)d.H * d.M * d.E * 4, st));
    SH_CUDA_CHECK(cudaMemsetAsync(dWd, 0, (size_t)d.H * d.M * d.E * 4, st));
  }
  if ((rc = launch_x<X_DWQK>(g, wide, dim3(mt, ct, g.ksplit), st))) return rc;
  // expert weights: contractions over the experts' lists
  const long list_steps = ((long)d.N * d.k / d.E + 63) / 64;
  wide = wide_tile(L, (long)d.H * d.E * mt, 1, d.Dt);
  col_tiles(g, d.Dt, wide);
  g.ksplit = k_parts(L, (long)d.H * d.E * mt * g.nsub, list_steps);
  if (g.ksplit > 1) SH_CUDA_CHECK(cudaMemsetAsync(dWv, 0, (size_t)d.H * d.E * d.M * d.Dt * 4, st));
  if ((rc = launch_x<X_DWV>(g, wide, dim3(d.H * d.E * g.ksplit, g.nsub, mt), st))) return rc;
  use_side(g, L, 1);
  wide = wide_tile(L, (long)d.H * d.E * dt, 1, d.M);
  col_tiles(g, d.M, wide);
  g.ksplit = k_parts(L, (long)d.H * d.E * dt * g.nsub, list_steps);
  if (g.ksplit > 1) SH_CUDA_CHECK(cudaMemsetAsync(dWo, 0, (size_t)d.H * d.E * d.Dt * d.M * 4, st));
  if ((rc = launch_x<X_DWO>(g, wide, dim3(d.H * d.E * g.ksplit, g.nsub, dt), st))) return rc;
  SH_CUDA_CHECK(cudaGetLastError());
  L->launches = 9;
  return SH_OK;
}
