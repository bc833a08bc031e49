// fp32 configuration of the SwitchHead layer: launch sequences of the forward and the backward pass.
// Projections on the tensor cores in split bf16 (sh_f32_gemm.cuh, sh_f32_wgrad.cuh), attention on the CUDA cores
// (sh_f32_attn.cuh) or, for longer sequences forward, the tensor cores (sh_f32_attn_tc.cuh), selection and sort in
// one launch (sh_f32_select.cuh).
#include "sh_internal.cuh"
#include "sh_launch.cuh"
#include "sh_simt.cuh"
#include "sh_f32_gemm.cuh"
#include "sh_f32_wgrad.cuh"
#include "sh_f32_attn.cuh"
#include "sh_f32_attn_tc.cuh"
#include "sh_f32_select.cuh"

#include <cstdlib>
#include <new>

using namespace shtc;

namespace {

// The split weights as [3 planes, rows, inner]: boxes of k_rows rows x 32 positions where a row runs along the
// contraction (k), of 32 rows x 64 columns where the contraction runs over rows (mn).
struct PlaneMap { CUtensorMap k, mn; int k_rows; };
struct F32State {
  PlaneMap wqk, wgate, wv, wo, wq_e, wk_e;
  bool pdl = true;          // kernels chained by programmatic dependent launch (the debug library's SH_NO_PDL: ordinary launches)
};

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

// Kernels are chained, except in a stage-timed pass.
bool chained(const sh_layer* L) { return ((const F32State*)L->f32)->pdl && !L->ev; }

// One mode's tiles as a part of a launch.
template <int MODE>
XPart part(sh_layer* L, const XGemmArgs& g, int gx, int gy, int gz = 1, const PlaneMap* w = nullptr) {
  const F32State* S = (const F32State*)L->f32;
  constexpr bool K_MAJOR = MODE == X_QK || MODE == X_V || MODE == X_O;
  if (!w) w = MODE == X_O || MODE == X_DA ? &S->wo : MODE == X_V || MODE == X_DR ? &S->wv : &S->wqk;
  XPart p;
  p.w = K_MAJOR ? w->k : w->mn; p.g = g; p.g.b_rows = w->k_rows; p.gx = gx; p.gy = gy; p.n = gx * gy * gz;
  // (about half of the experts' last tiles are worth counting; the rest of a side's table is empty)
  p.busy = MODE == X_QK || MODE == X_DX ? p.n : p.n - L->d.H * L->d.E / 2 * gy * gz;
  return p;
}

template <int A, int B = -1>
int launch_x(sh_layer* L, cudaStream_t st, const XPart& a, const XPart& b = XPart()) {
  const F32State* S = (const F32State*)L->f32;
  const int n = a.n + (B >= 0 ? b.n : 0);
  if (n == 0) return SH_OK;
  L->launches += 1;
  auto go = [&](auto kern, int smem) {
    if (int rc = set_smem(kern, smem)) return rc;
    return launch_k(chained(L), kern, dim3((unsigned)n), dim3(XG_THREADS), smem, st, S->wgate.mn, a, b);
  };
  if constexpr (A != X_DX && A != X_DR)
    if (a.g.sub_cols <= 64 && a.g.b_rows <= 64 && (B < 0 || (b.g.sub_cols <= 64 && b.g.b_rows <= 64)) && a.busy + (B >= 0 ? b.busy : 0) > sm_count(L))
      return go(sh_f32_gemm_kernel<A, B, true>, XGemmSmem<XG_HALF>::TOTAL);
  return go(sh_f32_gemm_kernel<A, B, false>, XGemmSmem<XG_WIDE>::TOTAL);
}

// Column tiles over `cols` columns: how many, and how wide (a multiple of 16).
int col_width(int cols) { const int n = (cols + XG_BN - 1) / XG_BN; return ((cols + n - 1) / n + 15) / 16 * 16; }
void col_tiles(XGemmArgs& g, int cols, int width = 0) {
  g.sub_cols = width ? width : col_width(cols);
  g.nsub = (cols + g.sub_cols - 1) / g.sub_cols;
}
// Row tiles of a side's lists, about.
long list_tiles(const ShDims& d) { return (long)d.H * d.N * d.k / 128 + d.H * d.E / 2; }
// A head's columns of d_head 129 to 192 are three tiles of up to 64 (one operand for three products, two blocks to an SM) and not two,
// except where two go once round the SMs and three do not.  (Two / three, a pass in us: 1 head of 160, d_model 960, 300 tokens 69.0 / 61.9, 2400
// tokens - 116 tiles or 173 - 88.2 / 92.0; 2 heads of 168, d_model 448, 900 tokens - 128 or 192 - 60.5 / 65.2, 2400 tokens 124 / 103.)
int proj_width(sh_layer* L) {
  const ShDims& d = L->d;
  const long two = 2 * (2l * d.H * d.nblk + list_tiles(d)), sms = sm_count(L);
  const bool three = d.Dt > 128 && d.Dt <= 192 && (two > sms || 3 * two <= 2 * sms);
  return three ? ((d.Dt + 2) / 3 + 15) / 16 * 16 : col_width(d.Dt);
}
// The output's columns, d_head above 128, are tiles of 64 instead of up to 128 where those leave more than a quarter of their rounds empty
// (2 heads, 2 of 4 experts: 150, d_model 192, 2400 tokens, 158 tiles 24 / 17 us; 168, d_model 448, 316 tiles 36 / 30; but 132, d_model 1024, 300 tokens
// of 4 of 8, 214 tiles, a pass 87.5 / 89.8).
bool out_narrow(sh_layer* L) {
  const long tiles = list_tiles(L->d) * ((L->d.M + XG_BN - 1) / XG_BN), sms = sm_count(L);
  return L->d.Dt > 128 && tiles > sms && 5 * ((tiles + sms - 1) / sms * sms) >= 7 * tiles;
}

// A contraction over d_head of a side's lists: up to 128 positions on the kernel that keeps its rows in tensor memory,
// the columns split among as many blocks per row tile as the device has SMs for.  (Half of the experts' last tiles are
// worth counting, the rest of the table is empty; with k = E every list is as long as the batch.)
template <int MODE>
int launch_d(sh_layer* L, cudaStream_t st, XGemmArgs g) {
  const F32State* S = (const F32State*)L->f32;
  const ShDims& d = L->d;
  const PlaneMap& w = MODE == X_O ? S->wo : S->wv;
  if (d.Dt > 128) {
    col_tiles(g, d.M, MODE == X_O && out_narrow(L) ? 64 : 0);
    return launch_x<MODE>(L, st, part<MODE>(L, g, d.H * head_tiles(d), g.nsub));
  }
  const int ntile = (d.M + XGemmDSmem::BN - 1) / XGemmDSmem::BN;
  const long rows = d.k == d.E ? (long)d.H * d.E * ((d.N + 127) / 128) : list_tiles(d);
  long split = sm_count(L) / (rows < 1 ? 1 : rows);
  split = split < 1 ? 1 : split > ntile ? ntile : split;
  auto kern = sh_f32_gemm_d_kernel<MODE>;
  if (int rc = set_smem(kern, XGemmDSmem::TOTAL)) return rc;
  L->launches += 1;
  return launch_k(chained(L), kern, dim3((unsigned)(d.H * head_tiles(d)), (unsigned)split), dim3(XG_THREADS), XGemmDSmem::TOTAL, st, MODE == X_O ? w.k : w.mn, g);
}

XGemmArgs base_args(sh_layer* L, const void* x) {
  char* ws = L->ws;
  const ShDims& d = L->d;
  XGemmArgs g{};
  g.d = d;
  g.x = (const float*)x;
  g.ahat = (const float*)(ws + L->o.ahat);
  g.ldz = sh_f32_ldz(d);
  g.ksplit = 1;
  g.q = (float*)(ws + L->o.q); g.k = (float*)(ws + L->o.k); g.v = (float*)(ws + L->o.v);
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

// Gates, selection and sort; beside them `zero` (n values), which a later kernel adds into, is cleared.
int launch_gate_sort(sh_layer* L, const void* x, float* zero, long n, cudaStream_t st) {
  const ShDims& d = L->d;
  char* ws = L->ws;
  // eight tokens a block while sixteen would leave SMs with less than two blocks (or their logits do not fit)
  const int ch = d.M <= 512 ? 512 : 1024;
  const bool small = d.N < 32 * sm_count(L) || 16 * (ch + d.G) * 4 > 200 * 1024;
  const int tok = small ? 8 : 16;
  const size_t smem = (size_t)tok * (ch + d.G) * 4;
  auto kern = small ? (ch == 512 ? sh_f32_gate_kernel<8, 512> : sh_f32_gate_kernel<8, 1024>)
                    : (ch == 512 ? sh_f32_gate_kernel<16, 512> : sh_f32_gate_kernel<16, 1024>);
  if (int rc = set_smem(kern, (int)smem)) return rc;
  const size_t ssm = sh_sort_smem_bytes(d);
  int* blockcnt = d.N > F32_SORT_MAX && ssm <= 227 * 1024 ? (int*)(ws + L->o.blockcnt) : nullptr;
  if (blockcnt) {
    SH_CUDA_CHECK(cudaMemsetAsync(blockcnt, 0, (size_t)d.nblk * d.G * 4, st));
    SH_CUDA_CHECK(cudaMemsetAsync(ws + L->o.tiles, 0, (size_t)2 * d.max_tiles * sizeof(ShTile), st));
  }
  if (int rc = launch_k(chained(L), kern, dim3((unsigned)((d.N + tok - 1) / tok)), dim3(512), smem, st, (const float*)x, (const float*)(ws + L->o.wgate32),
                        (const float*)(ws + L->o.gbias), (int*)(ws + L->o.idx), (float*)(ws + L->o.gate), blockcnt, (float4*)zero, n / 4, d, (int)((uintptr_t)x % 16 == 0)))
    return rc;
  L->launches += 2;
  if (blockcnt) {
    if (int rc = set_smem(sh_sort_kernel, (int)ssm)) return rc;
    return launch_k(chained(L), sh_sort_kernel, dim3(d.nblk), dim3(sh_sort_threads(d)), ssm, st, (const int*)(ws + L->o.idx), (const float*)(ws + L->o.gate),
                    (const int*)blockcnt, (int*)(ws + L->o.offsets), (int*)(ws + L->o.lists), (float*)(ws + L->o.lgate),
                    (ShTile*)(ws + L->o.tiles), (int*)(ws + L->o.ntiles), d);
  }
  return launch_k(chained(L), sh_f32_sort_kernel, dim3(d.sides * d.H), dim3(1024), 0, st, (const int*)(ws + L->o.idx), (const float*)(ws + L->o.gate),
                  (int*)(ws + L->o.offsets), (int*)(ws + L->o.lists), (float*)(ws + L->o.lgate), (ShTile*)(ws + L->o.tiles), d, head_tiles(d));
}

// x [Wq | Wk]: `groups` heads' column groups from `first` on.
XPart part_qk(sh_layer* L, const void* x, int first, int groups) {
  XGemmArgs g = base_args(L, x);
  g.qk_first = first; g.qk_groups = groups;
  col_tiles(g, L->d.Dt, proj_width(L));
  return part<X_QK>(L, g, L->d.nblk, groups * g.nsub);
}

// dst += gate x W^T over a side's expert lists: value experts, and query / key experts where a layer has them.
XPart part_v(sh_layer* L, const void* x, int side, const PlaneMap& w, float* dst, float scale, int ksplit = 1) {
  const ShDims& d = L->d;
  XGemmArgs g = base_args(L, x);
  use_side(g, L, side);
  g.v = dst; g.vscale = scale;
  col_tiles(g, d.Dt, proj_width(L));
  g.ksplit = ksplit;
  return part<X_V>(L, g, d.H * head_tiles(d), g.nsub, ksplit, &w);
}

// Key tiles of a part of a query tile's keys: the fewest, two at least, that keep the units at or below the number of SMs and their
// partial results in the backward pass's scratch (which decides for few heads of few columns); all of them (no parts, no scratch)
// where there are that many query tiles.
int attn_part_tiles(sh_layer* L) {
  const ShDims& d = L->d;
  const int nqt = (d.T - d.Tc + 127) / 128, most = (d.T + 63) / 64;
  const long heads = (long)d.B * d.H, room = 4l * d.N * d.H * d.D / (128 * (d.D + 2)), cap = room < sm_count(L) ? room : sm_count(L);
  if (nqt * heads > cap) return most;
  long all = 0;
  for (int i = 0; i < nqt; ++i) all += fattn_key_tiles(d, i);
  const long least = all * heads / cap;                    // (shorter parts are more units than that)
  for (int per = least < 2 ? 2 : (int)least; per < most; ++per) {
    long units = 0;
    for (int i = 0; i < nqt; ++i) units += (fattn_key_tiles(d, i) + per - 1) / per;
    if (units * heads <= cap) return per;
  }
  return most;
}

template <int D>
int launch_attn_tc(sh_layer* L, float* zero, long n, cudaStream_t st) {
  const ShDims& d = L->d;
  char* ws = L->ws;
  if (int rc = set_smem(sh_f32_attn_tc_kernel<D>, FAttnTcSmem<D>::TOTAL)) return rc;
  FAttnTcArgs g{};
  g.q = (const float*)(ws + L->o.q); g.k = (const float*)(ws + L->o.k); g.v = (const float*)(ws + L->o.v);
  g.ahat = (float*)(ws + L->o.ahat); g.stats = (float*)(ws + L->o.f32stats);
  g.part = (float*)(ws + L->o.bw); g.arrived = (unsigned*)(ws + L->o.f32arrived);
  g.zero = (float4*)zero; g.nzero = n / 4; g.d = d; g.per = attn_part_tiles(L); g.status = (int*)(ws + L->o.status);
  long units = 0;
  for (int i = 0; i < (d.T - d.Tc + 127) / 128; ++i) units += (fattn_key_tiles(d, i) + g.per - 1) / g.per;
  return launch_k(chained(L), sh_f32_attn_tc_kernel<D>, dim3((unsigned)(units * d.B * d.H)), dim3(288), FAttnTcSmem<D>::TOTAL, st, g);
}

template <int D>
int launch_attn_t(sh_layer* L, float* zero, long n, cudaStream_t st) {
  const ShDims& d = L->d;
  char* ws = L->ws;
  if (int rc = set_smem(sh_f32_attn_kernel<D>, FAttnSmem<D>::TOTAL)) return rc;
  const int nq = (d.T - d.Tc + 31) / 32;
  return launch_k(chained(L), sh_f32_attn_kernel<D>, dim3((unsigned)nq * d.B * d.H), dim3(256), FAttnSmem<D>::TOTAL, st,
                  (const float*)(ws + L->o.q), (const float*)(ws + L->o.k), (const float*)(ws + L->o.v), (float*)(ws + L->o.ahat),
                  (float*)(ws + L->o.f32stats), (float4*)zero, n / 4, d);
}

// Attention is on the tensor cores from 320 keys on, or from 129 on where the other kernel's blocks of 32 queries go one and a half
// times round the SMs: its time is that of the longest chain of key tiles, theirs mostly that of a unit.  (Whole passes of
// a small layer, CUDA cores / tensor cores, us: d_head 112, 8 heads, 256 keys 46 / 50, 320 55 / 53, 512 68 / 56, 800 102 / 77;
// 64 heads, 128 keys 66 / 64, 256 keys 110 / 86; 32 heads, 192 keys 53 / 58, 256 keys 73 / 71; d_head 32 and 64, 4 heads, 256 keys 36.8 / 38.1
// and 40.0 / 41.7, 320 39.5 / 39.3 and 44.2 / 43.0, 512 45.6 / 39.7 and 51.0 / 43.4.)
// But not up to 32 queries behind a cache - a block of the other kernel's, and a quarter of a unit, which takes a key tile in about 1.5
// times the time of a block - where the heads go round the SMs as often either way: above one round, and below it with 128 columns
// and the keys in one part.  (Whole passes, one query, d_head 32, 64 and 112: 160 heads, 330 keys 107 / 122, 116 / 134, 168 / 188;
// 128 heads, 330 keys 95 / 93, 105 / 101, 129 / 139, 1000 keys 238 / 230, 279 / 264, 313 / 342; 64 heads, 1000 keys
// 136 / 130, 151 / 144, 211 / 198; 64 queries, 160 heads, 400 keys 159 / 165, 181 / 185, 256 / 252.)
bool attn_on_tensor_cores(sh_layer* L) {
  const ShDims& d = L->d;
  const long sms = sm_count(L), heads = (long)d.B * d.H, nq = d.T - d.Tc;
  if (nq <= 32 && (heads > sms || (d.D == 128 && 2 * heads > sms))) return false;
  return d.T >= 320 || (d.T > 128 && 2 * ((nq + 31) / 32) * heads >= 3 * sms);
}

// Attention; beside it `zero` (n values), which the output projection adds into, is cleared.
int launch_attn(sh_layer* L, float* zero, long n, cudaStream_t st) {
  L->launches += 1;
  const ShDims& d = L->d;
  const bool tc = attn_on_tensor_cores(L);
  switch (d.D) {
    case 32: return tc ? launch_attn_tc<32>(L, zero, n, st) : launch_attn_t<32>(L, zero, n, st);
    case 64: return tc ? launch_attn_tc<64>(L, zero, n, st) : launch_attn_t<64>(L, zero, n, st);
    case 128: return tc ? launch_attn_tc<128>(L, zero, n, st) : launch_attn_t<128>(L, zero, n, st);
    default: return launch_attn_t<256>(L, zero, n, st);
  }
}

struct BwBuffers { float *dq, *dk, *dv, *dahat, *dz, *dsum; size_t cleared; };
BwBuffers bw_buffers(sh_layer* L) {
  const ShDims& d = L->d;
  const size_t nhd = (size_t)d.N * d.H * d.D;
  BwBuffers b;
  b.dq = (float*)(L->ws + L->o.bw); b.dk = b.dq + nhd; b.dv = b.dk + nhd; b.dahat = b.dv + nhd;
  b.dz = b.dahat + nhd;
  b.dsum = b.dz + (size_t)d.N * sh_f32_ldz(d);
  b.cleared = (size_t)(b.dsum - b.dq) + (size_t)d.N * d.H;
  return b;
}

template <int D>
int launch_attn_bw_t(sh_layer* L, const BwBuffers& w, cudaStream_t st) {
  ShDims d = L->d;
  d.causal = L->fwd_causal;
  char* ws = L->ws;
  if (int rc = set_smem(sh_f32_attn_bw_kernel<D>, FBwSmem<D>::TOTAL)) return rc;
  // A block's run of query tiles: short enough that the blocks fill the device about four times over,
  // at least one tile for each of its two thread groups.
  const int qt = (d.T + FBwSmem<D>::TQ - 1) / FBwSmem<D>::TQ, kt = (d.T + 31) / 32;
  const long units = (long)kt * d.B * d.H * qt / (d.causal ? 2 : 1);
  long run = units / (4l * sm_count(L));
  run = run < 2 ? 2 : run > qt ? qt : run;
  return launch_k(chained(L), sh_f32_attn_bw_kernel<D>, dim3((unsigned)kt * d.B * d.H, (unsigned)((qt + run - 1) / run)), dim3(256), FBwSmem<D>::TOTAL, st,
                  (const float*)(ws + L->o.q), (const float*)(ws + L->o.k), (const float*)(ws + L->o.v), (const float*)w.dahat,
                  (const float*)(ws + L->o.f32stats), (const float*)w.dsum, w.dq, w.dk, w.dv, d, (int)run);
}

// Parts of a contraction whose result is added anyway: enough blocks for every SM, at least eight steps each.
int k_parts(sh_layer* L, long blocks, long steps) {
  long p = sm_count(L) / (blocks < 1 ? 1 : blocks);
  const long most = steps / 8;
  p = p > most ? most : p;
  return p < 1 ? 1 : p > 8 ? 8 : (int)p;
}

}  // namespace

int sh_f32_prepare(sh_layer* L) {
  sh_f32_release(L);
  F32State* S = new (std::nothrow) F32State();
  if (!S) { sh_set_error("out of host memory"); return SH_ERR_INVALID_ARG; }
  L->f32 = S;
#ifdef SH_DEBUG
  S->pdl = !getenv("SH_NO_PDL");
#endif
  const ShDims& d = L->d;
  char* ws = L->ws;
  auto enc = [&](PlaneMap& m, size_t off, uint64_t inner, uint64_t rows, int k_rows) -> int {
    m.k_rows = k_rows;
    if (int rc = sh_tc_encode_planes(&m.k, ws + off, inner, rows, XG_BK, k_rows)) return rc;
    return sh_tc_encode_planes(&m.mn, ws + off, inner, rows, 64, XG_BK);
  };
  const uint64_t HD = (uint64_t)d.H * d.D;
  const int cw = proj_width(L);
  int rc;
  if ((rc = enc(S->wqk, L->o.wqk, d.M, 2 * HD, cw))) return rc;
  if ((rc = enc(S->wgate, L->o.wgate, d.M, d.G, 64))) return rc;
  if ((rc = enc(S->wv, L->o.wv, d.M, HD * d.E, cw))) return rc;
  if ((rc = enc(S->wo, L->o.wo, d.D, (uint64_t)d.H * d.E * d.M, d.Dt > 128 && !out_narrow(L) ? XG_BN : 64))) return rc;
  if (L->moe_q && (rc = enc(S->wq_e, L->o.wq_e, d.M, HD * d.E, cw))) return rc;
  if (L->moe_k && (rc = enc(S->wk_e, L->o.wk_e, d.M, HD * d.E, cw))) return rc;
  return SH_OK;
}

void sh_f32_release(sh_layer* L) {
  if (L && L->f32) { delete (F32State*)L->f32; L->f32 = nullptr; }
}

int sh_f32_gate_sort(sh_layer* L, const void* x, cudaStream_t st) { return launch_gate_sort(L, x, nullptr, 0, st); }

static size_t bf16_gate_smem(const ShDims& d) { return (size_t)(GB_TOK * (GB_XLD + d.G) + GB_NC * GB_WLD) * 4; }
bool sh_bf16_gate_ok(const sh_layer* L) { return bf16_gate_smem(L->d) <= 227 * 1024; }

int sh_bf16_gate(sh_layer* L, const void* x, int* blockcnt, bool pdl, cudaStream_t st) {
  const ShDims& d = L->d;
  char* ws = L->ws;
  const size_t smem = bf16_gate_smem(d);
  const int passes = (d.N + GB_TOK - 1) / GB_TOK, most = 2 * sm_count(L);    // (a block keeps its weights for all of its passes)
  if (int rc = set_smem(sh_bf16_gate_kernel, (int)smem)) return rc;
  L->launches += 1;
  return launch_k(pdl, sh_bf16_gate_kernel, dim3((unsigned)(passes < most ? passes : most)), dim3(GB_THREADS), smem, st, (const __nv_bfloat16*)x,
                  (const __nv_bfloat16*)(ws + L->o.wgate), (const float*)(ws + L->o.gbias), (int*)(ws + L->o.idx), (float*)(ws + L->o.gate), blockcnt, d, (int)((uintptr_t)x % 16 == 0));
}

int sh_f32_forward(sh_layer* L, const void* x, void* out, cudaStream_t st) {
  const ShDims& d = L->d;
  const F32State* S = (const F32State*)L->f32;
  char* ws = L->ws;
  const long nhd = (long)d.N * d.H * d.D, nout = (long)sh_out_rows(d) * d.M;
  float* v = (float*)(ws + L->o.v);
  int rc;
  // Dense queries and keys (a layer with query / key experts has none of its own) and the value experts
  // need nothing of one another: one launch, in a stage-timed pass two.
  const int first = L->moe_q ? d.H : 0, groups = (L->moe_q ? 0 : d.H) + (L->moe_k ? 0 : d.H);
  const XPart qk = part_qk(L, x, first, groups), pv = part_v(L, x, 0, S->wv, v, 0.f);
  sh_mark(L, 0, st);
  if ((rc = launch_gate_sort(L, x, v, nhd, st))) return rc;
  sh_mark(L, 1, st);
  if (L->ev && (rc = launch_x<X_QK>(L, st, qk))) return rc;
  if (L->moe_k) {
    SH_CUDA_CHECK(cudaMemsetAsync(ws + L->o.k, 0, (size_t)nhd * 4, st));
    if ((rc = launch_x<X_V>(L, st, part_v(L, x, 0, S->wk_e, (float*)(ws + L->o.k), 0.f)))) return rc;
  }
  if (L->moe_q) {
    SH_CUDA_CHECK(cudaMemsetAsync(ws + L->o.q, 0, (size_t)nhd * 4, st));
    if ((rc = launch_x<X_V>(L, st, part_v(L, x, 1, S->wq_e, (float*)(ws + L->o.q), 1.4426950408889634f / sqrtf((float)d.Dt))))) return rc;
  }
  sh_mark(L, 2, st);
  if ((rc = L->ev ? launch_x<X_V>(L, st, pv) : launch_x<X_QK, X_V>(L, st, qk, pv))) return rc;
  sh_mark(L, 3, st);
  // (the relative-position term of Transformer-XL is in the one-warp-per-query kernel only; `out` is cleared
  //  behind the last read of x either way: the two may be the same buffer)
  if ((rc = L->xl_positions ? sh_simt_attention_f32(L, st) : launch_attn(L, (float*)out, nout, st))) return rc;
  if (L->xl_positions) SH_CUDA_CHECK(cudaMemsetAsync(out, 0, (size_t)nout * 4, st));
  sh_mark(L, 4, st);
  XGemmArgs g = base_args(L, x);
  use_side(g, L, 1);
  g.y = (float*)out;
  if ((rc = launch_d<X_O>(L, st, g))) return rc;
  sh_mark(L, 5, st);
  SH_CUDA_CHECK(cudaGetLastError());
  return SH_OK;
}

int sh_f32_backward(sh_layer* L, const void* x, const float* dout, float* dx, float* dWq, float* dWk, float* dWv,
                    float* dWo, float* dWs, float* dWd, cudaStream_t st) {
  const ShDims& d = L->d;
  char* ws = L->ws;
  const BwBuffers w = bw_buffers(L);
  const int ht = head_tiles(d), mt = (d.M + 127) / 128;
  int rc;
  L->launches = 0;
  XGemmArgs src = base_args(L, x);                         // source side; dst: destination side
  src.dy = dout; src.dq = w.dq; src.dk = w.dk; src.dv = w.dv; src.dz = w.dz; src.dsum = w.dsum; src.dahat = w.dahat; src.dx = dx;
  src.dWq = dWq; src.dWk = dWk; src.dWv = dWv; src.dWo = dWo; src.dWs = dWs; src.dWd = dWd;
  auto aligned = [](const void* p) { return (uintptr_t)p % 16 == 0; };
  src.vec_dy = aligned(dout);
  src.vec_out = aligned(dx) && aligned(dWq) && aligned(dWk) && aligned(dWv) && aligned(dWo);
  XGemmArgs dst = src;
  use_side(src, L, 0); use_side(dst, L, 1);
  // weight gradients: how the contractions are split
  auto wpart = [](const XGemmArgs& a, int gx, int gy, int gz) { XWPart p; p.g = a; p.gx = gx; p.gy = gy; p.n = gx * gy * gz; return p; };
  XGemmArgs gq = src, gv = src, go = dst;
  col_tiles(gq, d.Dt); col_tiles(gv, d.Dt); col_tiles(go, d.Dt);
  gq.qk_groups = 2 * d.H;
  const int ct = gq.qk_groups * gq.nsub + (d.G + XW_BN - 1) / XW_BN;
  // parts: the shortest ones (of eight steps at least) that still fit the SMs in one round; one part each where
  // whole contractions already need more rounds
  const long nq = (long)mt * ct, nl = (long)d.H * d.E * mt * (gv.nsub + go.nsub);
  // (of a list, a step at least: with fewer selections than experts most are empty, and their gradients are still stored)
  const long sel = (long)d.N * d.k / d.E, sq = (d.N + XG_BK - 1) / XG_BK, sl = sel < 1 ? 1 : (sel + XG_BK - 1) / XG_BK;
  long len = sq > sl ? sq : sl;
  for (long l = 8; l < len; ++l)
    if (nq * ((sq + l - 1) / l) + nl * ((sl + l - 1) / l) <= sm_count(L)) { len = l; break; }
  gq.ksplit = (int)((sq + len - 1) / len);
  gv.ksplit = go.ksplit = (int)((sl + len - 1) / len);
  // what is added into
  const long hmd = (long)d.H * d.M * d.Dt, hme = (long)d.H * d.M * d.E;
  FClear c{};
  int nc = 0;
  auto clear = [&](float* p, long n) { c.p[nc] = p; c.n[nc++] = n; };
  clear(w.dq, (long)w.cleared); clear(dx, (long)d.N * d.M);
  if (gq.ksplit > 1) { clear(dWq, hmd); clear(dWk, hmd); clear(dWs, hme); clear(dWd, hme); }
  if (gv.ksplit > 1) { clear(dWv, hmd * d.E); clear(dWo, hmd * d.E); }
  if ((rc = launch_k(chained(L), sh_f32_clear_kernel, dim3(4u * (unsigned)sm_count(L)), dim3(256), 0, st, c))) return rc;
  XGemmArgs g;
  // output experts: dAhat and the destination gates' gradients
  g = dst;
  col_tiles(g, d.Dt);
  // (about half of the experts' last tiles are worth counting; the rest of the table is empty)
  g.ksplit = k_parts(L, list_tiles(d) * g.nsub, d.M / XG_BK);
  if ((rc = launch_x<X_DA>(L, st, part<X_DA>(L, g, d.H * ht, g.nsub, g.ksplit)))) return rc;
  // attention
  rc = d.D == 32 ? launch_attn_bw_t<32>(L, w, st) : d.D == 64 ? launch_attn_bw_t<64>(L, w, st)
     : d.D == 128 ? launch_attn_bw_t<128>(L, w, st) : launch_attn_bw_t<256>(L, w, st);
  if (rc) return rc;
  // value experts: their part of dx, and the source gates' gradients
  if ((rc = launch_d<X_DR>(L, st, src))) return rc;
  // queries, keys and gates: the rest of dx
  g = src;
  col_tiles(g, d.M);
  g.ksplit = k_parts(L, (long)d.nblk * g.nsub, 2 * d.H * ((d.Dt + XG_BK - 1) / XG_BK));
  if ((rc = launch_x<X_DX>(L, st, part<X_DX>(L, g, d.nblk, g.nsub, g.ksplit)))) return rc;
  // weight gradients, one launch
  const XWPart pq = wpart(gq, mt, ct, gq.ksplit), pv = wpart(gv, d.H * d.E * gv.ksplit, gv.nsub, mt), po = wpart(go, d.H * d.E * go.ksplit, go.nsub, mt);
  if ((rc = set_smem(sh_f32_wgrad_kernel, XWgradSmem::TOTAL))) return rc;
  if ((rc = launch_k(chained(L), sh_f32_wgrad_kernel, dim3((unsigned)(pq.n + pv.n + po.n)), dim3(XW_THREADS), XWgradSmem::TOTAL, st, pq, pv, po))) return rc;
  SH_CUDA_CHECK(cudaGetLastError());
  L->launches += 3;
  return SH_OK;
}
