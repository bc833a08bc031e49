// Internal declarations shared by the translation units of libswitchhead.
#pragma once
#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stddef.h>
#include "../../include/switchhead.h"

#define SH_TILE_ROWS 128   // rows of one grouped-GEMM tile and tokens per gate/sort block

struct ShTile {            // one row tile of one (head, expert) group
  int h, e, row0, nrows;   // row0: position inside lists[side][h]; nrows <= SH_TILE_ROWS
};

struct ShDims {
  int M, H, D, E, k;       // D: d_head as stored (padded with zero columns to 32, 64, 128 or 256)
  int Dt;                  // d_head as given (scale 1/sqrt(Dt), rotary angles)
  int B, T;
  int N;                   // B*T tokens
  int sides;               // 2: source and destination gates; 1: shared selection (one gate serves both)
  int G;                   // gate columns = sides*H*E
  int nblk;                // ceil(N / SH_TILE_ROWS)
  int max_tiles;           // upper bound on row tiles per side
  int tile_rows_src;       // rows per tile of the source-side (value expert) tile table: 128 or 256
  int Tc;                  // Transformer-XL context: the first Tc tokens of every sequence are the cache (keys and values
                           // only); queries, destination gates and out rows exist for the last T - Tc tokens.  0: no cache.
  int causal;              // 1: key s visible to query t iff s <= t (default); 0: every key of the sequence
  int early_rows;          // first tokens of every sequence whose value rows are summed in fp32 (SH_EARLY_ROWS or 0)
  unsigned long long* stamps;   // sh_forward_stamped: the pass's ShStampBlock in the workspace; nullptr otherwise
  int* status;             // the status block at the start of the workspace (nullptr: the allocation-free gate entry point)
};

// Sets of k <= 4 experts {e0 < e1 < ...} of E, numbered: pairs row by row, (0,1), (0,2), ..., (0,E-1), (1,2), ..., larger
// sets by sum of choose(e_i, i + 1) (the value projection of such a layer is tiled by (head, set): sh_tc_vset_kernel).
__host__ __device__ __forceinline__ int sh_choose(int n, int k) {
  return k == 1 ? n : k == 2 ? n * (n - 1) / 2 : k == 3 ? n * (n - 1) * (n - 2) / 6 : k == 4 ? n * (n - 1) * (n - 2) * (n - 3) / 24 : 0;
}
#ifdef __CUDACC__
__device__ __forceinline__ int sh_set_id(unsigned mask, int k, int E) {     // k >= 2 bits
  const int lo = __ffs(mask) - 1, hi = 31 - __clz(mask);
  if (k == 2) return lo * (2 * E - lo - 1) / 2 + (hi - lo - 1);
  const unsigned rest = mask & ~(1u << lo) & ~(1u << hi);
  int id = lo + sh_choose(hi, k) + sh_choose(__ffs(rest) - 1, 2);
  if (k > 3) id += sh_choose(31 - __clz(rest), 3);
  return id;
}
#endif
__host__ __device__ __forceinline__ void sh_set_decode(int id, int k, int E, int* e) {
  if (k == 2) {
    e[0] = 0;
    while (e[0] < E - 2 && id >= E - 1 - e[0]) { id -= E - 1 - e[0]; ++e[0]; }
    e[1] = e[0] + 1 + id;
    return;
  }
  for (int i = k, n = E - 1; i >= 1; --i) {
    while (n > i - 1 && sh_choose(n, i) > id) --n;
    e[i - 1] = n;
    id -= sh_choose(n--, i);
  }
}

// With a cache in front of every sequence (ShDims::Tc): the row of `out` that belongs to context token
// `tok` (-1 for a cache token), and the context token of an out row.
__host__ __device__ __forceinline__ int sh_out_row(const ShDims& d, int tok) {
  if (d.Tc == 0) return tok;
  const int b = tok / d.T, t = tok % d.T;
  return t < d.Tc ? -1 : b * (d.T - d.Tc) + t - d.Tc;
}
__host__ __device__ __forceinline__ int sh_ctx_tok(const ShDims& d, int row) {
  if (d.Tc == 0) return row;
  const int Tq = d.T - d.Tc;
  return (row / Tq) * d.T + d.Tc + row % Tq;
}
__host__ __device__ __forceinline__ int sh_out_rows(const ShDims& d) { return d.B * (d.T - d.Tc); }

// Per-kernel time stamps of one forward pass (sh_forward_stamped), %globaltimer nanoseconds:
// resident = first CTA of the kernel running, start = first CTA past its wait for the kernel before
// it, end = last CTA done.  Slot = kernel identifier below.
enum { SH_K_GATE = 0, SH_K_SORT = 1, SH_K_QK_A = 2, SH_K_QK_B = 3, SH_K_V = 4, SH_K_ATTN = 5, SH_K_O = 6, SH_K_COUNT = 7 };
struct ShStampBlock { unsigned long long resident[SH_K_COUNT], start[SH_K_COUNT], end[SH_K_COUNT]; };
#ifdef __CUDACC__
// (one thread per CTA calls these; no-ops in an ordinary pass, where the block pointer is null)
__device__ __forceinline__ unsigned long long sh_globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void sh_stamp_resident(unsigned long long* s, int k) { if (s) atomicMin(s + k, sh_globaltimer_ns()); }
__device__ __forceinline__ void sh_stamp_start(unsigned long long* s, int k) { if (s) atomicMin(s + SH_K_COUNT + k, sh_globaltimer_ns()); }
__device__ __forceinline__ void sh_stamp_end(unsigned long long* s, int k) { if (s) atomicMax(s + 2 * SH_K_COUNT + k, sh_globaltimer_ns()); }
#endif

// Workspace sub-buffers (byte offsets from the workspace base).
// Precision policy of the 16-bit path.  Under the causal mask the first tokens of a sequence attend
// to a handful of keys: their attention read-out is hardly averaged, their output rows are 10-15
// times larger than the RMS of the whole output (which is what the tolerance is measured against),
// and every fp16 rounding on their way - 2^-11 of a LARGE value - counts.  The first SH_EARLY_ROWS
// tokens of every sequence therefore take a more exact route where it is cheap to give them one:
// their value rows are summed in fp32 (scratch of [B, H, SH_EARLY_ROWS, D] floats) and rounded to
// fp16 once by whichever of the k contributions arrives last.  Later rows, averaged over many keys,
// keep the fast form (k fp16 vector reductions into V).  The ratio between the first rows and the RMS
// grows with the sequence length (measured max-abs error / RMS of the fast form alone: 8e-3 at 512
// tokens, 1.4-1.9e-2 at 2048, 1.8-2.4e-2 at 4096, against a tolerance of 2e-2), so the exact route is
// taken from SH_EARLY_MIN_SEQ tokens per sequence on.
#define SH_EARLY_ROWS 32
#define SH_EARLY_MIN_SEQ 1024

struct ShWorkspace {
  size_t status, wqk, wgate, gbias, wv, wo, q, k, v, ahat, idx, gate, blockcnt, blockoff,
         offsets, lists, lgate, tiles, ntiles, rope, vearly, vearly_cnt, xl_emb, xl_r, xl_uv, xl_r16, xl_vr, xl_uk, xl_bias, wos, gid, wq_e, wk_e, bw, wgate32, f32stats, f32arrived, wo_overflow, stamps, total;
};

// Words of the 256-byte status block at the start of the workspace.
enum {
  SH_ST_STATUS = 0,       // 0, or the first SH_ERR_TIMEOUT / SH_ERR_BOUNDS a kernel recorded
  SH_ST_DIAG = 1,         // 1..6: where the first bounded wait gave up (block, thread, barrier address, parity, grid, block size)
  SH_ST_BOUNDS = 8,       // 8..11: the first failed index check of a debug build (site, value, limit, block)
  SH_ST_SCHED = 16,       // 16, 17: tile counter and finished-claimer counter of the dense Q/K projection
  SH_ST_GRIDBAR = 24,     // 24, 25: grid barrier of the fused gate + sort kernel
  SH_ST_SORTED = 26,      // one-grid front: 128-token blocks whose selections, list entries and tiles are in memory
  SH_ST_GUARD_BAD = 32    // damaged guard words counted by sh_check_guards
};

#define SH_GUARD_BYTES 256
#define SH_GUARD_BYTE 0xC5u
#define SH_MAX_GUARDS 40

struct sh_layer {
  ShDims d{};
  bool dense = false;
  bool moe_q = false, moe_k = false;   // query / key projections are experts too (destination / source side selection)
  bool out_f16 = false;                // sh_set_output_f16: sh_forward writes its result as fp16 (bf16 storage, tensor-core output projection)
  int dtype = -1;
  char* ws = nullptr;
  size_t ws_bytes = 0;
  ShWorkspace o{};
  bool weights_set = false;
  const void* fwd_x = nullptr;   // input of the forward pass whose intermediates the workspace holds (sh_backward wants the same one); nullptr: none
  int fwd_causal = 1;            // that pass's mask (its row maxima and normalisers belong to it)
  bool rope = false;       // rotary position embeddings on Q, K (table in the workspace)
  bool xl_positions = false;   // Transformer-XL relative-position term (fp32 configuration; tables in the workspace)
  int launches = 0;
  int sm_count = 0;
  void* tc = nullptr;      // tensor-core path state (tensor maps), owned by the layer
  void* f32 = nullptr;     // fp32 configuration: tensor maps of the split weights, owned by the layer
  cudaEvent_t* ev = nullptr;  // when set (sh_forward_timed): 6 events recorded at the stage boundaries
  size_t guard_off[SH_MAX_GUARDS] = {};   // byte offsets of the guards behind the workspace sub-buffers
  int n_guards = 0;
};

// Shapes the sparse output projection (sh_tc_oproj_sp_kernel) serves: with at most two selections out of
// every four neighbouring experts a token's gate-scaled rows are 2:4 sparse along an expert-innermost
// contraction axis.  The layer then keeps a second, expert-interleaved copy of W_O in the workspace.
inline bool sh_o_sparse_ok(const sh_layer* L) {
  const ShDims& d = L->d;
  return L->dtype == SH_BF16 && !L->dense && d.k <= 2 && (d.E == 4 || d.E == 8) && d.D == 128 && d.H <= 4;
}

// Shapes whose value projection is tiled by (head, set of selected experts) instead of (head, expert): the k experts of a
// set side by side are at most 256 columns, and there are few enough sets for their partly filled tiles - half a tile of
// 256 rows each, on two SMs, against half a tile of 128 per expert - not to cost more than the k - 1 further gathers of
// every row.  A row is the fp32 sum of its experts, rounded once, where the other kernel adds fp16 results in memory.
// Passes back to back in us, by experts / by sets: 8192 tokens, 2 heads of 64, d_model 512, 3 of 5 experts 56.9 / 49.0.  At the line, 2 heads
// and d_model 512, 4 and 1024: 1200 tokens, 3 of 6: 47.2 / 45.3, 65.6 / 67.6; 2400 tokens, 3 of 7: 49.2 / 49.2, 75.8 / 77.8; 1600 tokens, 4 of 7: 49.7 / 51.2,
// 78.6 / 79.7; 3200 tokens, 2 of 8: 46.7 / 49.2, 74.8 / 75.9; 16000 tokens, 2 of 8: 80.3 / 74.9, 194.5 / 171.8; below it: 400 tokens, 4 of 6: 47.4 / 45.2,
// 69.6 / 64.1.  With two experts and an odd number of heads, whose Q/K projection is a kernel of its own beside this one, the sets cost 2 to 15 % up
// to 7000 tokens (800 tokens, 3 heads, d_model 2048, 2 of 3: 59.4 / 70.1): they stay for their rounding.
inline bool sh_v_sets_ok(const sh_layer* L) {
  const ShDims& d = L->d;
  if (L->dtype != SH_BF16 || L->dense || d.k < 2 || d.k > 4 || d.E < d.k) return false;
  const int sets = d.E <= 16 ? sh_choose(d.E, d.k) : 1 << 20;
  if (d.k == 2 && d.D == 128) return sets <= 28;
  if (d.D != 64 || sets > 35 || L->moe_q || L->moe_k) return false;
  return 128l * sets - 64l * d.E <= (long)d.N * (d.k - 1);
}

template <typename T> __device__ __forceinline__ float sh_to_float(T v);
template <> __device__ __forceinline__ float sh_to_float<float>(float v) { return v; }
template <> __device__ __forceinline__ float sh_to_float<__half>(__half v) { return __half2float(v); }
template <> __device__ __forceinline__ float sh_to_float<__nv_bfloat16>(__nv_bfloat16 v) { return __bfloat162float(v); }
template <typename T> __device__ __forceinline__ T sh_from_float(float v);
template <> __device__ __forceinline__ float sh_from_float<float>(float v) { return v; }
template <> __device__ __forceinline__ __half sh_from_float<__half>(float v) { return __float2half_rn(v); }
template <> __device__ __forceinline__ __nv_bfloat16 sh_from_float<__nv_bfloat16>(float v) { return __float2bfloat16_rn(v); }

void sh_set_error(const char* fmt, ...);

// Index checks of the debug library (built with -DSH_DEBUG): a list entry, tile-table field or
// expert index read from memory is checked against its range before it is used as an address; a
// failed check records SH_ERR_BOUNDS with the site, the value and the limit in the status block and
// the caller skips the access.  The release library compiles them away.
enum { SH_SITE_V_LIST = 1, SH_SITE_V_TILE = 2, SH_SITE_V_TOKEN = 3, SH_SITE_SORT_EXPERT = 4, SH_SITE_SORT_SLOT = 5,
       SH_SITE_O_EXPERT = 6, SH_SITE_SELFTEST = 7 };
#ifdef __CUDACC__
__device__ __forceinline__ bool sh_index_record(long long v, long long limit, int* status, int site) {
  if (v >= 0 && v < limit) return true;
  if (status && atomicCAS(status, 0, SH_ERR_BOUNDS) == 0) {
    status[SH_ST_BOUNDS] = site; status[SH_ST_BOUNDS + 1] = (int)v; status[SH_ST_BOUNDS + 2] = (int)limit; status[SH_ST_BOUNDS + 3] = (int)blockIdx.x;
  }
  return false;
}
#ifdef SH_DEBUG
#define SH_INDEX_OK(v, limit, status, site) sh_index_record((long long)(v), (long long)(limit), (status), (site))
#else
#define SH_INDEX_OK(v, limit, status, site) true
#endif
#endif

// Stage boundary marker: boundary 0 = start, 1 = after gate+sort, 2 = after Q/K, 3 = after V,
// 4 = after attention, 5 = after the output projection.
static inline void sh_mark(sh_layer* L, int boundary, cudaStream_t st) {
  if (L->ev) cudaEventRecord(L->ev[boundary], st);
}

enum { SH_STAGE_GATE = 1, SH_STAGE_QK = 2, SH_STAGE_V = 4, SH_STAGE_ATTN = 8, SH_STAGE_O = 16, SH_STAGE_ALL = 31 };

// CUDA-core stages on bf16 storage with fp16 intermediates (same buffers and layouts as the
// tensor-core kernels): the on-device reference used while a tensor-core stage is brought up.
int sh_simt_run_bf16(sh_layer* L, int stages, const void* x, void* out, cudaStream_t st);

// fp32 configuration of the SwitchHead layer (sh_f32.cu).
inline int sh_f32_ldz(const ShDims& d) { return (d.G + 31) / 32 * 32; }       // row length of the gate-gradient matrix
int sh_f32_prepare(sh_layer* L);                // tensor maps, after the weights are split
void sh_f32_release(sh_layer* L);
int sh_f32_gate_sort(sh_layer* L, const void* x, cudaStream_t st);
int sh_f32_forward(sh_layer* L, const void* x, void* out, cudaStream_t st);
int sh_f32_backward(sh_layer* L, const void* x, const float* dout, float* dx, float* dWq, float* dWk, float* dWv,
                    float* dWo, float* dWs, float* dWd, cudaStream_t st);
// Gate logits and selections on the CUDA cores for bf16 storage (sh_gate_topk with d_head above 128), with the
// per-block counts the sort wants (cleared by the caller).
int sh_bf16_gate(sh_layer* L, const void* x, int* blockcnt, bool pdl, cudaStream_t st);
bool sh_bf16_gate_ok(const sh_layer* L);        // its logits fit shared memory (up to about 2000 gate columns)
// The CUDA-core attention kernel on fp32 storage (the relative-position term of Transformer-XL).
int sh_simt_attention_f32(sh_layer* L, cudaStream_t st);

// Tensor-core (tcgen05) path of the bf16 configuration.
int sh_tc_prepare(sh_layer* L);                 // builds tensor maps after the weights are repacked
void sh_tc_release(sh_layer* L);
int sh_tc_forward(sh_layer* L, const void* x, void* out, cudaStream_t st);
int sh_tc_gate_sort(sh_layer* L, const void* x, cudaStream_t st);
int sh_tc_selftest(sh_layer* L, int which, unsigned long long arg, cudaStream_t st);
