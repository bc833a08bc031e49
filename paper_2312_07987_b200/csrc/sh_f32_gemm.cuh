// fp32 contractions on the tensor cores: every projection of the fp32 configuration, forward and
// backward, but the weight gradients, which are in sh_f32_wgrad.cuh (their modes are numbered here: they share the
// arguments).
//
// An fp32 value is the exact sum of three bf16 values, x = h + m + l (8 + 8 + 8 mantissa bits: h is x
// rounded, m the rest rounded, l what is left), so a product of two is
//   hh' + (hm' + mh') + (hl' + mm' + lh') + terms below 2^-25 of it,
// six bf16 products.  The tensor core adds into fp32 but drops the bits below the accumulator's last one
// instead of rounding, so a long chain of additions drifts towards zero: hh', which carries the size of the
// result, has an accumulator P0 of its own that is read back and added in fp32 registers every 64
// contraction positions, 4 additions.  The five others, 2^-8 of it and less, share P1, read every 1024.
//
// Why not FFMA: the CUDA cores' 74 TFLOP/s fp32 peak against 2.25 PFLOP/s / 6 = 375.
//
// The activation is operand A in TENSOR memory.  Workers read its rows as fp32, steps ahead, by asynchronous
// copies into shared memory that only the copying warp uses (a prefetch that costs no registers and no block-wide
// barrier), split them and store the planes with tcgen05.st: thread = row.  (As planes in shared memory they were
// written and read there, next to the weights: 232 KB of shared-memory traffic per 128 x 128 tile and step of 32
// positions, 1800 cycles against 768 of tensor time; now 104 KB.)  Weights are split once, when they are set, and
// come as planes by TMA.  One thread issues the UMMAs; the workers read the accumulators and write the result.
// Operands are addressed row by row (a gathered token list, a head's slice of a row), and the weights either as rows of
// the contraction (K-major) or as rows of the other index (MN-major: weights in the backward pass), so no
// transposed or gathered copy is made.  Results go through a padded copy in shared memory and leave as one bulk
// operation per row: as vector reductions from the accumulator layout (a lane per row, 16 bytes each) they were a third
// of the short contractions' time.
//
// Two kernels:
//   sh_f32_gemm_kernel   long contractions (over d_model, or over all heads): a tile of 128 rows x up to 128 columns.
//   sh_f32_gemm_d_kernel short ones (over one head's d_head <= 128): 128 rows, whose planes stay in tensor memory
//                        for all of the block's column tiles.
#pragma once
#include "sh_tc_prims.cuh"

namespace shtc {

enum { X_QK = 0,    // q, k = x [Wq | Wk]                     rows: tokens
       X_V = 1,     // v += g x Wv                           rows: a value expert's list
       X_O = 2,     // y += g ahat Wo                        rows: an output expert's list
       X_DA = 3,    // dahat += g dy Wo^T, ds = ahat . that  rows: an output expert's list
       X_DWO = 4,   // dWo = (g ahat)^T dy                   contraction: an output expert's list
       X_DR = 5,    // dx += g dv Wv^T, ds = x . that        rows: a value expert's list
       X_DWV = 6,   // dWv = (g x)^T dv                      contraction: a value expert's list
       X_DX = 7,    // dx += [dq dk dz] [Wq Wk Wgate]^T      rows: tokens
       X_DWQK = 8 };// dWq, dWk, dWgate = x^T [dq dk dz]     contraction: tokens

struct XGemmArgs {
  ShDims d;
  const float *x, *dy;                   // [N, M]; dy [N, M]
  const float* ahat;                     // [N, H, D]
  const float *dq, *dk, *dv;             // [N, H, D]
  float *dz, *dsum;                      // gate gradients [N, ldz], columns (side*H + h)*E + e; rowsum(dahat o ahat) [N, H]
  int ldz;
  const int* lists; const float* lgate; const int* offsets; const ShTile* tiles;   // of the side the mode works on
  int nsub, sub_cols;                    // column tiles per head (or of M), and columns per tile (a multiple of 16)
  int b_rows;                            // rows of a K-major weight box
  int qk_first, qk_groups;               // X_QK: first group ((which*H + h)) and how many
  int ksplit;                            // parts of the contraction (weight gradients: with more than one the results are added)
  float *q, *k, *v;                      // X_QK: q, k [B, H, T, D]; X_V: v
  float *y;                              // X_O [rows of out, M]
  float *dahat, *dx;
  float *dWq, *dWk, *dWv, *dWo, *dWs, *dWd;
  float qscale, vscale;
  const float2* rope;
  int vec_dy, vec_out;                   // dy / the written gradients are 16-byte aligned
  int* status;
};

constexpr int XG_BK = 32;                // positions of a step
constexpr int XG_BN = 128;               // columns of a tile of the long contractions, at most
constexpr int XG_WORKERS = 256, XG_THREADS = XG_WORKERS + 64;   // + a warp that issues UMMAs, + one that loads weights
constexpr int XG_A_STEP = 48;            // tensor-memory columns of a step's A planes: per 16 positions 8 each of h, m, l
constexpr int XG_CHUNK = 2;              // steps per promotion of P0: 64 positions, four additions
constexpr int XG_P1_CHUNKS = 16;         // chunks per promotion of P1

// K-major planes: rows of 32 values (64 bytes), 64-byte swizzle, 8-row groups 512 bytes apart.
constexpr uint32_t DESC_HI_SW64 = (512u >> 4) | (1u << 14) | (4u << 29);
__device__ __forceinline__ uint64_t xg_desc(uint32_t lo, bool mn_major) {
  return ((uint64_t)(mn_major ? DESC_HI_SW128 : DESC_HI_SW64) << 32) | lo;
}
// Instruction descriptor, bf16 operands, 128 rows.
__device__ __forceinline__ uint32_t xg_idesc(int n, bool b_mn) {
  return make_idesc_f16(128, 0, 1, 1, 0) | ((uint32_t)(n >> 3) << 17) | (b_mn ? 1u << 16 : 0u);
}

// acc += 32 tensor-memory columns at a time.
template <int N>
__device__ __forceinline__ void tmem_add(uint32_t taddr, float (&acc)[N]) {
#pragma unroll
  for (int c = 0; c < N; c += 32) {
    uint32_t u[32];
    tmem_ld32(taddr + c, u);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[c + i] += __uint_as_float(u[i]);
  }
}
// acc += P0 + (P1 + P2), w tensor-memory columns apart: one rounding at the size of the sum (each on its own, three: 1 to 8 % more error).
template <int N>
__device__ __forceinline__ void tmem_add3(uint32_t taddr, uint32_t w, float (&acc)[N]) {
#pragma unroll
  for (int c = 0; c < N; c += 16) {
    uint32_t a[16], b[16];
    tmem_ld16(taddr + 2 * w + c, a);
    tmem_ld16(taddr + w + c, b);
    tmem_ld_wait();
    float s[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) s[i] = __uint_as_float(a[i]) + __uint_as_float(b[i]);
    tmem_ld16(taddr + c, a);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[c + i] += __uint_as_float(a[i]) + s[i];
  }
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]) : "memory");
}

// Two fp32 values as three packed bf16 pairs whose sum they are.  (The leading part saturates: fp32 reaches half a
// bf16 step past the largest bf16 value, and an infinity there would leave a rest of minus infinity.)
__device__ __forceinline__ float2 sub_bf16x2(float2 x, uint32_t p) {
  return __ffma2_rn(make_float2(__uint_as_float(p << 16), __uint_as_float(p & 0xFFFF0000u)), make_float2(-1.f, -1.f), x);
}
__device__ __forceinline__ void split_bf16x3(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
  asm("cvt.rn.satfinite.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(b), "f"(a));
  float2 r = sub_bf16x2(make_float2(a, b), h);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(m) : "f"(r.y), "f"(r.x));
  r = sub_bf16x2(r, m);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(l) : "f"(r.y), "f"(r.x));
}

// Four adjacent floats into shared memory (16-byte aligned there).
__device__ __forceinline__ void fetch4(uint32_t dst, const float* p, bool vec, bool live = true) {
  if (vec) cp_async_16(dst, p, live ? 16 : 0);             // (a dead piece is zeros; its address is still a valid one)
  else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + i * 4), "l"(p + i), "r"(live ? 4 : 0) : "memory");
  }
}

// A warp's fp32 pieces of a step: 32 rows of 16 values (64 bytes), chunk c of row r at c ^ (r >> 1 & 3), so that the
// eight lanes of a phase meet eight different 16-byte banks, copied (lane -> chunk lane & 3 of rows lane >> 2, + 8, ...)
// or read (lane -> row).
__device__ __forceinline__ uint32_t raw16_copy(int lane) { return (uint32_t)((lane >> 2) * 64 + (((lane & 3) ^ ((lane >> 3) & 3)) << 4)); }
// A row's 16 values as the planes of 16 contraction positions.
__device__ __forceinline__ void raw16_split(const unsigned char* kb, int lane, uint32_t (&h)[8], uint32_t (&m)[8], uint32_t (&l)[8]) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float4 v = *reinterpret_cast<const float4*>(kb + lane * 64 + ((c ^ ((lane >> 1) & 3)) << 4));
    split_bf16x3(v.x, v.y, h[2 * c], m[2 * c], l[2 * c]);
    split_bf16x3(v.z, v.w, h[2 * c + 1], m[2 * c + 1], l[2 * c + 1]);
  }
}

// Token of a list entry (0 where the debug library finds that it is none).
__device__ __forceinline__ int xg_token(const XGemmArgs& g, size_t li) {
  const int t = g.lists[li];
  return SH_INDEX_OK(t, g.d.N, g.status, SH_SITE_V_LIST) ? t : 0;
}
__device__ __forceinline__ bool xg_tile_ok(const XGemmArgs& g, const ShTile& tl) {
  const ShDims& d = g.d;
  return SH_INDEX_OK(tl.h, d.H, g.status, SH_SITE_V_TILE) && SH_INDEX_OK(tl.e, d.E, g.status, SH_SITE_V_TILE) &&
         SH_INDEX_OK(tl.nrows - 1, SH_TILE_ROWS, g.status, SH_SITE_V_TILE) && SH_INDEX_OK(tl.row0, (long long)d.N * d.k - tl.nrows + 1, g.status, SH_SITE_V_TILE);
}

// Gate gradient of a list entry from a part of its columns: the ungated result against the forward operand of the same
// row.  ds s (1 - s) is linear in ds, and rowsum(dahat o ahat) = sum over the selected experts of s ds: both are
// added up here, part by part (kernels of their own for them: 5 us of a step).
template <int MODE>
__device__ __forceinline__ void xg_gate_gradient(const XGemmArgs& g, int t, int h, int e, float gt, float dot) {
  atomicAdd(g.dz + (size_t)t * g.ldz + ((MODE == X_DA ? g.d.H : 0) + h) * g.d.E + e, dot * gt * (1.f - gt));
  if (MODE == X_DA) atomicAdd(g.dsum + (size_t)t * g.d.H + h, gt * dot);
}

struct XTile { int x, y, z; };           // which tile of its mode a block works on
// Block number i of a mode's gx x gy x gz tiles.
__device__ __forceinline__ XTile xg_unpack(int i, int gx, int gy) { return {i % gx, i / gx % gy, i / (gx * gy)}; }

// ---- long contractions ------------------------------------------------------------------------------------
// Weights in a ring of four steps, fp32 rows of the four next steps on their way, A planes of two steps in tensor
// memory, P0 twice (a chunk is read under the UMMAs of the next one).  A training step of 2 x 512 tokens, d_model 1024, 4 heads
// of 112: Q, K and V 42 -> 36 us, dahat 29 -> 25, the projections' dx 25 -> 23.  The tensor pipe is active a quarter of that: a step
// takes 0.9 us, of which 0.4 is UMMAs; the rest are its hand-overs (a second issuing thread, for P0, changed nothing).
// Tiles of up to 64 columns (NARROW): the issue of a UMMA, ~57 cycles, is longer than its execution, so three do the
// six products - the planes of B lie one behind the other, one operand of three times the columns -
//   h x [h' m' l'] -> P0 P1 P2,   m x [h' m'] -> P1 P2,   l x h' -> P2,
// all of them twice in tensor memory and read every chunk.  (336 tokens, 8 heads of 32: 63 us a pass with six, 58 with three.)
// As many narrow tiles as go more than once round the SMs run two blocks to an SM (XG_HALF), each with one accumulator, the A planes of
// one step and weights of two: its hand-overs stand one behind the other, and the other block's fill them, as they do a tile's set-up and
// drain.  (Whole passes, one block / two, us: 8 heads of 64, d_model 256, 168 tiles 52.5 / 48.6, 2024 tiles 337 / 294; 4 heads of 64, d_model 1024,
// 112 tiles 68.2 / 70.5, 160 tiles 108.8 / 98.8; 2 heads of 64, d_model 512, 130 tiles 62.1 / 62.9, 192 tiles 82.9 / 75.9.)
enum { XG_WIDE = 0, XG_NARROW = 1, XG_HALF = 2 };
template <int KIND>
struct XGemmSmem {
  static constexpr int NB = KIND == XG_HALF ? 2 : 4, NR = 4, BN = KIND == XG_HALF ? 64 : XG_BN;
  static constexpr int B_STEP = 3 * BN * XG_BK * 2, RAW = 128 * XG_BK * 4;
  static constexpr int RAW_OFF = NB * B_STEP, BAR_OFF = RAW_OFF + NR * RAW;
  static constexpr int LD = BN + 4;                        // result rows (they take the weights' place, and that of the pieces)
  static constexpr int TOTAL = BAR_OFF + 256 + 1024;
  static_assert(128 * LD * 4 <= BAR_OFF, "");
};

// One tile.  mapW: planes of the mode's weights, rows [(which*H + h)*D + dd][m] (Q, K), [(h*E + e)*D + dd][m] (V),
// [(h*E + e)*M + m][dd] (O); mapG: of the gates' weights, rows [(side*H + h)*E + e][m].
template <int MODE, int KIND>
__device__ __forceinline__ void xg_tile(const CUtensorMap& mapW, const CUtensorMap& mapG, const XGemmArgs& g, XTile blk) {
  using SM = XGemmSmem<KIND>;
  constexpr bool NARROW = KIND != XG_WIDE, HALF = KIND == XG_HALF;
  constexpr int NB = SM::NB, NB_LOG = NB == 4 ? 2 : 1;     // (powers of two: a division costs the issuing thread as much as two UMMAs)
  constexpr int NA = HALF ? 1 : 2, A_LOG = HALF ? 0 : 1;   // accumulators, and steps of A planes
  constexpr bool B_MN = MODE >= X_DA;
  constexpr bool LIST_ROWS = MODE == X_V || MODE == X_O || MODE == X_DA || MODE == X_DR;
  constexpr bool ADDED = MODE != X_QK;                     // results that are added to (as one bulk operation per row; stored by X_QK)
  constexpr int COLS = NARROW ? 32 : XG_BN / 2;            // columns of a worker thread
  constexpr uint32_t P0 = 0, P0S = NARROW ? 192 : 128, P1 = 256, TA = HALF ? 192 : 384;   // tensor-memory columns
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* sgen = smem_raw + (sbase - smem_u32(smem_raw));
  uint64_t* b_full = (uint64_t*)(sgen + SM::BAR_OFF);      // [NB] the step's weights are in shared memory
  uint64_t* done = b_full + SM::NB;                        // [NB] the step's UMMAs are done
  uint64_t* a_full = done + SM::NB;                        // [2]  the step's A planes are in tensor memory
  uint64_t* acc_full = a_full + 2;                         // [2]  P0 of a chunk is complete
  uint64_t* acc_empty = acc_full + 2;                      // [2]  ... and has been read
  uint64_t* p1_empty = acc_empty + 2;
  uint32_t* tmem_slot = (uint32_t*)(p1_empty + 1);
  const ShDims& d = g.d;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int HD = d.H * d.D;
  bool dead = false;

  if (tid == 0) {
    for (int s = 0; s < SM::NB; ++s) { mbar_init(&b_full[s], 1); mbar_init(&done[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&a_full[s], 8); mbar_init(&acc_full[s], 1); mbar_init(&acc_empty[s], 8); }
    mbar_init(p1_empty, 8);
    fence_barrier_init();
  }
  pdl_wait();
  // (behind the wait: what runs ahead of the next kernel's wait sees all kernels up to the one ahead of this.  With room on the SM for a
  //  block of the next kernel, behind the allocation too: that one may want all of the tensor memory and wait for this kernel's end)
  if (!HALF) pdl_trigger();
  // ---- which tile ------------------------------------------------------------------------------
  int h = 0, e = 0, which = 0, row0 = 0, nrows = 0, n0 = 0, ncols = 0, steps = 0;
  const int sps = (d.Dt + XG_BK - 1) / XG_BK;                        // steps over one head's d_head
  if (LIST_ROWS) {
    const ShTile tl = g.tiles[blk.x];
    if (tl.nrows == 0 || !xg_tile_ok(g, tl)) return;       // (before any allocation)
    h = tl.h; e = tl.e; row0 = tl.row0; nrows = tl.nrows;
    n0 = blk.y * g.sub_cols;
    ncols = min(g.sub_cols, ((MODE == X_O || MODE == X_DR) ? d.M : d.Dt) - n0);
    steps = (MODE == X_V || MODE == X_DA) ? d.M / XG_BK : sps;
  } else if (MODE == X_DX) {
    row0 = blk.x * 128; nrows = min(128, d.N - row0);
    n0 = blk.y * g.sub_cols; ncols = min(g.sub_cols, d.M - n0);
    steps = 2 * d.H * sps + (d.G + XG_BK - 1) / XG_BK;
  } else {
    const int grp = g.qk_first + blk.y / g.nsub;
    which = grp / d.H; h = grp % d.H;
    n0 = (blk.y % g.nsub) * g.sub_cols; ncols = min(g.sub_cols, d.Dt - n0);
    row0 = blk.x * 128; nrows = min(128, d.N - row0);
    steps = d.M / XG_BK;
  }
  // a part of the contraction (modes whose results are added): steps s0 ...
  int s0 = 0;
  if (ADDED && g.ksplit > 1) {
    const int per = (steps + g.ksplit - 1) / g.ksplit;
    s0 = blk.z * per;
    steps = min(per, steps - s0);
    if (steps <= 0) return;
  }
  const int nchunk = (steps + XG_CHUNK - 1) / XG_CHUNK;
  if (warp == 8) { tmem_alloc(tmem_slot, HALF ? 256 : 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  if (HALF) pdl_trigger();

  if (warp == 8) {
    if (lane == 0) {
      // contraction positions of step i that exist (the rest of the operand rows is zero)
      int seg = MODE == X_DX ? min(s0 / sps, 2 * d.H) : 0, off = MODE == X_DX ? (s0 - seg * sps) * XG_BK : s0 * XG_BK;
      auto kvalid = [&]() -> int {
        int n = XG_BK;
        if (MODE == X_O || MODE == X_DR) n = min(XG_BK, d.Dt - off);
        if (MODE == X_DX) n = min(XG_BK, (seg < 2 * d.H ? d.Dt : d.G) - off);
        off += XG_BK;
        if (MODE == X_DX && seg < 2 * d.H && off >= d.Dt) { off = 0; ++seg; }
        return n;
      };
      const uint32_t id = xg_idesc((ncols + 15) & ~15, B_MN);
      // MN-major: 64 columns of all planes one behind the other, the next 64 behind them
      constexpr uint32_t BK = B_MN ? 128 : 2;              // 16 positions further
      const uint32_t BP = B_MN ? (64 * XG_BK * 2) >> 4 : (uint32_t)(g.b_rows * XG_BK * 2) >> 4;   // the next plane
      const uint32_t b0 = !B_MN ? desc_lo_k(sbase) : desc_lo_mn(sbase, NARROW ? 64 * XG_BK * 2 : 3 * 64 * XG_BK * 2);
      const uint32_t w = B_MN ? 64 : g.b_rows;             // NARROW: columns of a plane
      const uint32_t id3 = xg_idesc(3 * w, B_MN), id2 = xg_idesc(2 * w, B_MN), id1 = xg_idesc(w, B_MN);
      for (int i = 0; i < steps && !dead; ++i) {
        const int c = i / XG_CHUNK;
        if (i % XG_CHUNK == 0) {
          if (!mbar_wait(&acc_empty[c & (NA - 1)], ((c >> A_LOG) & 1) ^ 1, g.status, dead)) break;
          if (!NARROW && c > 0 && c % XG_P1_CHUNKS == 0 && !mbar_wait(p1_empty, (c / XG_P1_CHUNKS - 1) & 1, g.status, dead)) break;
        }
        if (!mbar_wait(&b_full[i & (NB - 1)], (i >> NB_LOG) & 1, g.status, dead)) break;
        if (!mbar_wait(&a_full[i & (NA - 1)], (i >> A_LOG) & 1, g.status, dead)) break;
        tc_fence_after();
        const int kn = (kvalid() + 15) / 16;
        const uint32_t p0 = tmem + P0 + (c & (NA - 1)) * P0S, p1 = tmem + P1;
        const uint32_t first0 = i % XG_CHUNK == 0, first1 = first0 && c % XG_P1_CHUNKS == 0;
#pragma unroll
        for (int k = 0; k < XG_BK / 16; ++k) {
          if (k >= kn) break;
          const uint32_t a = tmem + TA + (i & (NA - 1)) * XG_A_STEP + k * 24;
          const uint32_t b = b0 + (i & (NB - 1)) * (SM::B_STEP >> 4) + BK * k;
          if (NARROW) {
            umma_f16_tmem_a(p0, a, xg_desc(b, B_MN), id3, !(first0 && k == 0));
            umma_f16_tmem_a(p0 + w, a + 8, xg_desc(b, B_MN), id2, 1);
            umma_f16_tmem_a(p0 + 2 * w, a + 16, xg_desc(b, B_MN), id1, 1);
            continue;
          }
          const uint64_t bh = xg_desc(b, B_MN), bm = xg_desc(b + BP, B_MN), bl = xg_desc(b + 2 * BP, B_MN);
          umma_f16_tmem_a(p1, a, bl, id, !(first1 && k == 0));
          umma_f16_tmem_a(p1, a + 8, bm, id, 1);
          umma_f16_tmem_a(p1, a + 16, bh, id, 1);
          umma_f16_tmem_a(p1, a, bm, id, 1);
          umma_f16_tmem_a(p1, a + 8, bh, id, 1);
          umma_f16_tmem_a(p0, a, bh, id, !(first0 && k == 0));
        }
        umma_commit(&done[i & (NB - 1)]);
        if (i % XG_CHUNK == XG_CHUNK - 1 || i == steps - 1) umma_commit(&acc_full[c & (NA - 1)]);
      }
    }
    __syncwarp();
  } else if (warp == 9) {
    if (lane == 0) {
      const int chunks64 = B_MN && !NARROW && ncols > 64 ? 2 : 1;
      const uint32_t bytes = B_MN ? chunks64 * 3 * 64 * XG_BK * 2 : 3 * g.b_rows * XG_BK * 2;
      for (int i = 0; i < steps && !dead; ++i) {
        if (i >= NB && !mbar_wait(&done[i & (NB - 1)], ((i >> NB_LOG) - 1) & 1, g.status, dead)) break;
        mbar_expect_tx(&b_full[i & (NB - 1)], bytes);
        const int ii = s0 + i;
        int x = ii * XG_BK, y = 0;
        bool gm = false;
        if (MODE == X_QK) y = (which * d.H + h) * d.D + n0;
        if (MODE == X_V) y = (h * d.E + e) * d.D + n0;
        if (MODE == X_O) y = (h * d.E + e) * d.M + n0;
        if (MODE == X_DA) { x = n0; y = (h * d.E + e) * d.M + ii * XG_BK; }
        if (MODE == X_DR) { x = n0; y = (h * d.E + e) * d.D + ii * XG_BK; }
        if (MODE == X_DX) {
          const int seg = ii / sps;
          x = n0;
          gm = seg >= 2 * d.H;
          y = gm ? (ii - 2 * d.H * sps) * XG_BK : seg * d.D + (ii - seg * sps) * XG_BK;
        }
        const uint32_t dst = sbase + (i & (NB - 1)) * SM::B_STEP;
        tma_load_3d(dst, gm ? &mapG : &mapW, &b_full[i & (NB - 1)], x, y, 0);
        if (chunks64 == 2) tma_load_3d(dst + 3 * 64 * XG_BK * 2, gm ? &mapG : &mapW, &b_full[i & (NB - 1)], x + 64, y, 0);
      }
    }
    __syncwarp();
  } else {
    // ---- workers: operand, promotions, result ------------------------------------------------------
    // warp -> rows 32 q ..., positions 16 half ... of a step, columns 64 half ... of the result
    const int q = warp & 3, half = warp >> 2;
    const size_t lbase = (size_t)h * d.N * d.k;
    const bool vdy = MODE != X_DA || g.vec_dy != 0;
    // What lies past the tile never needs masking, only an address inside the operand: rows past the last one
    // end in accumulators nobody reads, and positions past d_head (or the gate columns) are zeros in memory -
    // a step of 32 never leaves the stored d_head.
    const float* arow[4];
    int zrow[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int r = row0 + min(32 * q + (lane >> 2) + 8 * u, nrows - 1);
      const size_t t = LIST_ROWS ? xg_token(g, lbase + r) : r;
      zrow[u] = r;
      arow[u] = (MODE == X_QK || MODE == X_V ? g.x + t * d.M
               : MODE == X_O ? g.ahat + t * HD + h * d.D
               : MODE == X_DA ? g.dy + t * d.M
               : MODE == X_DR ? g.dv + t * HD + h * d.D : g.dq + t * HD) + half * 16 + (lane & 3) * 4;
    }
    int xseg = min(s0 / sps, 2 * d.H), xoff = (s0 - xseg * sps) * XG_BK;   // X_DX: the step's head (of dq, then dk), and where in it
    const uint32_t rbase = sbase + SM::RAW_OFF + warp * 2048 + raw16_copy(lane);
    auto load = [&](int i) {                               // step i on its way
      long o = (long)(s0 + i) * XG_BK;
      if (MODE == X_DX) o = (xseg >= d.H ? (long)(g.dk - g.dq) + (long)(xseg - d.H) * d.D : (long)xseg * d.D) + xoff;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float* p = arow[u] + o;
        if (MODE == X_DX && xseg == 2 * d.H) p = g.dz + (size_t)zrow[u] * g.ldz + xoff + half * 16 + (lane & 3) * 4;
        fetch4(rbase + (i & 3) * SM::RAW + u * 512, p, vdy);
      }
      if (MODE == X_DX) {
        xoff += XG_BK;
        if (xseg < 2 * d.H && xoff >= d.Dt) { xoff = 0; ++xseg; }
      }
    };
    const uint32_t tlane = (uint32_t)(q * 32) << 16;
    float acc[COLS];
#pragma unroll
    for (int i = 0; i < COLS; ++i) acc[i] = 0.f;
    const bool mine = half * COLS < ncols;                 // (whole warps)
    auto promote = [&](int c) {
      if (!mbar_wait(&acc_full[c & (NA - 1)], (c >> A_LOG) & 1, g.status, dead)) return;
      tc_fence_after();
      const bool p1 = (c + 1) % XG_P1_CHUNKS == 0 || c == nchunk - 1;
      if (mine) {
        const uint32_t a0 = tmem + tlane + P0 + (c & (NA - 1)) * P0S + half * COLS, w = B_MN ? 64 : g.b_rows;
        if (NARROW) tmem_add3(a0, w, acc);
        else tmem_add(a0, acc);
        if (!NARROW && p1) tmem_add(tmem + tlane + P1 + half * COLS, acc);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&acc_empty[c & (NA - 1)]);
        if (!NARROW && p1) mbar_arrive(p1_empty);
      }
    };
#pragma unroll
    for (int i = 0; i < SM::NR; ++i) {
      if (i < steps) load(i);
      cp_async_commit();
    }
    int promoted = 0;
    for (int i = 0; i < steps && !dead; ++i) {
      cp_async_wait<SM::NR - 1>();                         // this warp's pieces of step i are there
      __syncwarp();
      uint32_t ph[8], pm[8], pl[8];
      raw16_split(sgen + SM::RAW_OFF + (i & 3) * SM::RAW + warp * 2048, lane, ph, pm, pl);
      __syncwarp();
      if (i + SM::NR < steps) load(i + SM::NR);
      cp_async_commit();
      if (i >= NA && !mbar_wait(&done[(i - NA) & (NB - 1)], ((i - NA) >> NB_LOG) & 1, g.status, dead)) break;
      tc_fence_after();
      const uint32_t ta = tmem + tlane + TA + (i & (NA - 1)) * XG_A_STEP + half * 24;
      tmem_st8(ta, ph);
      tmem_st8(ta + 8, pm);
      tmem_st8(ta + 16, pl);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&a_full[i & (NA - 1)]);
      // a chunk is read once two steps of the next one are in tensor memory, or, with one accumulator, the first of them
      if (HALF ? i % XG_CHUNK == 0 && i > 0 : i % XG_CHUNK == 1 && i > XG_CHUNK) promote(promoted++);
    }
    cp_async_wait<0>();
    for (; promoted < nchunk && !dead; ++promoted) promote(promoted);
    // ---- result: thread = row q*32 + lane, columns half*COLS ... -----------------------------------
    const int r = q * 32 + lane, c0 = half * COLS;
    const int valid = min(COLS, ncols - c0);
    if (r < nrows && valid > 0 && !dead) {
      if (LIST_ROWS) {
        const size_t li = lbase + row0 + r;
        const int t = xg_token(g, li);
        const float gt = g.lgate[li];
        if (MODE == X_DA || MODE == X_DR) {
          const float* other = MODE == X_DA ? g.ahat + (size_t)t * HD + h * d.D + n0 + c0 : g.x + (size_t)t * d.M + n0 + c0;
          float dot = 0.f;
#pragma unroll
          for (int i = 0; i < COLS; i += 4) {
            if (i + 4 <= valid) {
              const float4 o = __ldg(reinterpret_cast<const float4*>(other + i));
              dot += (acc[i] * o.x + acc[i + 1] * o.y) + (acc[i + 2] * o.z + acc[i + 3] * o.w);
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j) if (i + j < valid) dot += acc[i + j] * __ldg(other + i + j);
            }
          }
          xg_gate_gradient<MODE>(g, t, h, e, gt, dot);
        }
        const float f = MODE == X_V && g.vscale != 0.f ? gt * g.vscale : gt;
#pragma unroll
        for (int i = 0; i < COLS; ++i) acc[i] *= f;
      } else if (MODE == X_QK) {
        const int tok = row0 + r;
        if (g.rope) {
          const float2* cs = g.rope + (size_t)((n0 + c0) >> 1) * d.T + tok % d.T;
#pragma unroll
          for (int i = 0; i < COLS; i += 2)
            if (i < valid) {
              const float2 w = cs[(size_t)(i >> 1) * d.T];
              const float a0 = acc[i], a1 = acc[i + 1];
              acc[i] = a0 * w.x - a1 * w.y;
              acc[i + 1] = a0 * w.y + a1 * w.x;
            }
        }
        if (which == 0) {
#pragma unroll
          for (int i = 0; i < COLS; ++i) acc[i] *= g.qscale;
        }
      }
    }
    {
      // rows through shared memory (the weights' ring and the pieces are free: every UMMA has been waited for), 16 bytes of
      // padding a row so that eight lanes' 16-byte stores meet different banks
      float* stg = reinterpret_cast<float*>(sgen);
      if (r < nrows && valid > 0 && !dead) {
#pragma unroll
        for (int i = 0; i < COLS; i += 4)
          *reinterpret_cast<float4*>(stg + r * SM::LD + c0 + i) = make_float4(acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
      }
      fence_proxy_async_smem();
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (tid < nrows && !dead) {
        // (whole 16-byte pieces: the columns that pad the last one of a head are zero columns of its stored width)
        const int n = (ncols + 3) & ~3;
        float* o = nullptr;
        if (LIST_ROWS) {
          const int t = xg_token(g, lbase + row0 + tid);
          if (MODE == X_V) o = g.v + (((size_t)(t / d.T) * d.H + h) * d.T + t % d.T) * d.D + n0;
          if (MODE == X_O) { const int orow = sh_out_row(d, t); if (orow >= 0) o = g.y + (size_t)orow * d.M + n0; }   // (cache tokens have no output row)
          if (MODE == X_DA) o = g.dahat + (size_t)t * HD + h * d.D + n0;
          if (MODE == X_DR) o = g.dx + (size_t)t * d.M + n0;
        } else if (MODE == X_DX) {
          o = g.dx + (size_t)(row0 + tid) * d.M + n0;
        } else {
          const int tok = row0 + tid;
          o = (which ? g.k : g.q) + (((size_t)(tok / d.T) * d.H + h) * d.T + tok % d.T) * d.D + n0;
        }
        if (o) {
          const uint32_t src = smem_u32(stg + tid * SM::LD);
          if (MODE == X_QK) bulk_store(o, src, n * 4);
          else if ((MODE != X_DR && MODE != X_DX) || g.vec_out) bulk_reduce_add_f32(o, src, n * 4);
          else
            for (int i = 0; i < n; ++i) atomicAdd(o + i, stg[tid * SM::LD + i]);
        }
        bulk_commit();
        bulk_wait_all();
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem, HALF ? 256 : 512);
  }
}

// A launch of one or two modes whose tiles do not depend on one another: the first blocks work on tiles
// of mode A, the rest on mode B.  (One launch each leaves SMs idle in its last round,
// and pays its set-up and drain by itself.)
struct XPart { CUtensorMap w; XGemmArgs g; int gx, gy, n, busy; };   // busy: tiles that hold rows, about
template <int M> struct xg_mode { static constexpr int value = M; };
template <int A, int B, bool HALF>                         // HALF: all tiles are narrow, two blocks to an SM
__global__ void __launch_bounds__(XG_THREADS, HALF ? 2 : 1)
sh_f32_gemm_kernel(const __grid_constant__ CUtensorMap mapG, const __grid_constant__ XPart pa, const __grid_constant__ XPart pb) {
  const int i = blockIdx.x;
  auto run = [&](auto mode, const XPart& p, int j) {
    constexpr int MODE = decltype(mode)::value;
    // (the columns of d_model are at least 64 a tile, and as many as 128 where there are more)
    constexpr bool D_MODEL = MODE == X_DX || MODE == X_O || MODE == X_DR;
    if (HALF) xg_tile<MODE, XG_HALF>(p.w, mapG, p.g, xg_unpack(j, p.gx, p.gy));
    else if (!D_MODEL && p.g.sub_cols <= 64) xg_tile<MODE, D_MODEL ? XG_WIDE : XG_NARROW>(p.w, mapG, p.g, xg_unpack(j, p.gx, p.gy));
    else xg_tile<MODE, XG_WIDE>(p.w, mapG, p.g, xg_unpack(j, p.gx, p.gy));
  };
  if (B < 0 || i < pa.n) run(xg_mode<A>(), pa, i);
  else run(xg_mode<(B >= 0 ? B : A)>(), pb, i - pa.n);
}

// ---- short contractions: over one head's d_head, up to 128 ---------------------------------------------------
// y += g ahat Wo and dx += g dv Wv^T: 128 rows of a list, all of d_model.  A block gathers and splits its rows once -
// the planes take up to 192 tensor-memory columns - and then works off 64 output columns at a time, weights up to three
// tiles ahead.  B's planes lie one behind the other, so that they are one operand of 192 columns; accumulators P0 P1 P2
// and a second P0 (P3) for the positions from 64 on:
//   h x [h' m' l'] -> P0 P1 P2  (from 64 on: h x h' -> P3, h x [m' l'] -> P1 P2),   m x [h' m'] -> P1 P2,   l x h' -> P2.
// (A block per 128 x 64 result paid the gather, the split, the set-up and the drain, 6 us, for every 0.8 us of UMMAs: y 37 -> 19 us,
// dx 48 -> 21 us at 1024 tokens, k = 2, d_model 1024, 4 heads of 112.)  What bounds it now: a tile's read-out and reductions,
// 1.7 us, behind its UMMAs.
struct XGemmDSmem {
  static constexpr int NB = 3, BN = 64;
  static constexpr int B_TILE = 4 * 3 * BN * XG_BK * 2;    // all steps of a column tile
  static constexpr int LD = BN + 4;                        // result rows
  static constexpr int STG_OFF = NB * B_TILE, X_OFF = STG_OFF + 128 * LD * 4, X_WARP = 32 * 32 * 4;
  static constexpr int BAR_OFF = X_OFF + 8 * X_WARP;
  static constexpr int RAW_OFF = STG_OFF, RAW = 128 * XG_BK * 4;   // (the rows' pieces, before anything else is there)
  static constexpr int TOTAL = BAR_OFF + 256 + 1024;
  static_assert(RAW_OFF + 4 * RAW <= BAR_OFF, "");
};

template <int MODE>
__global__ void __launch_bounds__(XG_THREADS, 1)
sh_f32_gemm_d_kernel(const __grid_constant__ CUtensorMap mapW, const __grid_constant__ XGemmArgs g) {
  using SM = XGemmDSmem;
  constexpr bool B_MN = MODE == X_DR;
  constexpr int COLS = SM::BN / 2;
  constexpr uint32_t P0 = 0, P1 = 64, P2 = 128, P3 = 192, TA = 256;
  constexpr uint32_t PLANE = SM::BN * XG_BK * 2, B_STEP = 3 * PLANE;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* sgen = smem_raw + (sbase - smem_u32(smem_raw));
  uint64_t* b_full = (uint64_t*)(sgen + SM::BAR_OFF);      // [NB]
  uint64_t* b_empty = b_full + SM::NB;                     // [NB]
  uint64_t* a_full = b_empty + SM::NB;
  uint64_t* acc_full = a_full + 1;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 1);
  const ShDims& d = g.d;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int HD = d.H * d.D;
  bool dead = false;

  // (the tile table and the lists are older than the kernel ahead of this one)
  const ShTile tl = g.tiles[blockIdx.x];
  if (tl.nrows == 0 || !xg_tile_ok(g, tl)) return;
  if (tid == 0) {
    for (int s = 0; s < SM::NB; ++s) { mbar_init(&b_full[s], 1); mbar_init(&b_empty[s], 1); }
    mbar_init(a_full, 8); mbar_init(acc_full, 1); mbar_init(acc_empty, 8);
    fence_barrier_init();
  }
  const int h = tl.h, e = tl.e, row0 = tl.row0, nrows = tl.nrows;
  const int sps = (d.Dt + XG_BK - 1) / XG_BK, k16s = (d.Dt + 15) / 16;
  const int ntile = (d.M + SM::BN - 1) / SM::BN;
  const int tile0 = (int)((long)blockIdx.y * ntile / gridDim.y), tiles = (int)((long)(blockIdx.y + 1) * ntile / gridDim.y) - tile0;
  const size_t lbase = (size_t)h * d.N * d.k;
  const int q = warp & 3, half = warp >> 2, r = q * 32 + lane;   // workers: row; positions 16 half ... of a step, columns 32 half ... of a tile
  int t = 0;
  float gt = 0.f;
  if (warp < 8) {
    const size_t li = lbase + row0 + min(r, nrows - 1);
    t = xg_token(g, li);
    gt = g.lgate[li];
  }
  if (warp == 8) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 8) {
    pdl_wait();                                            // (no bounded wait of this kernel runs while the one ahead does)
    if (lane == 0) {
      const uint32_t id3 = xg_idesc(192, B_MN), id2 = xg_idesc(128, B_MN), id1 = xg_idesc(64, B_MN);
      const uint32_t b0 = B_MN ? desc_lo_mn(sbase, PLANE) : desc_lo_k(sbase);
      constexpr uint32_t BK = B_MN ? 128 : 2, BP = PLANE >> 4;
      if (mbar_wait(a_full, 0, g.status, dead)) {
        int s = 0;
        uint32_t par = 0;
        for (int j = 0; j < tiles; ++j) {
          if (j > 0 && !mbar_wait(acc_empty, (j - 1) & 1, g.status, dead)) break;
          if (!mbar_wait(&b_full[s], par, g.status, dead)) break;
          tc_fence_after();
          for (int k = 0; k < k16s; ++k) {
            const uint32_t a = tmem + TA + k * 24;
            const uint32_t b = b0 + s * (SM::B_TILE >> 4) + (k >> 1) * (B_STEP >> 4) + BK * (k & 1);
            if (k < 4) umma_f16_tmem_a(tmem + P0, a, xg_desc(b, B_MN), id3, k != 0);
            else {
              umma_f16_tmem_a(tmem + P1, a, xg_desc(b + BP, B_MN), id2, 1);
              umma_f16_tmem_a(tmem + P3, a, xg_desc(b, B_MN), id1, k != 4);
            }
            umma_f16_tmem_a(tmem + P1, a + 8, xg_desc(b, B_MN), id2, 1);
            umma_f16_tmem_a(tmem + P2, a + 16, xg_desc(b, B_MN), id1, 1);
          }
          umma_commit(&b_empty[s]);
          umma_commit(acc_full);
          if (++s == SM::NB) { s = 0; par ^= 1; }
        }
      }
    }
    __syncwarp();
  } else if (warp == 9) {
    if (lane == 0) {
      int s = 0;
      uint32_t par = 1;
      for (int j = 0; j < tiles; ++j) {
        if (j == SM::NB) pdl_wait();                       // (the weights do not depend on the kernel ahead)
        if (j >= SM::NB && !mbar_wait(&b_empty[s], par, g.status, dead)) break;
        mbar_expect_tx(&b_full[s], sps * B_STEP);
        const int n0 = (tile0 + j) * SM::BN;
        for (int i = 0; i < sps; ++i) {
          const uint32_t dst = sbase + s * SM::B_TILE + i * B_STEP;
          if (MODE == X_O) tma_load_3d(dst, &mapW, &b_full[s], i * XG_BK, (h * d.E + e) * d.M + n0, 0);
          else tma_load_3d(dst, &mapW, &b_full[s], n0, (h * d.E + e) * d.D + i * XG_BK, 0);
        }
        if (++s == SM::NB) { s = 0; par ^= 1; }
      }
    }
    __syncwarp();
  } else {
    pdl_wait();
    pdl_trigger();
    {
      // rows past the last one end in accumulators nobody reads, positions past d_head are zeros in memory
      const float* base = (MODE == X_O ? g.ahat : g.dv) + h * d.D + half * 16 + (lane & 3) * 4;
      const uint32_t rbase = sbase + SM::RAW_OFF + warp * 2048 + raw16_copy(lane);
      const float* arow[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) arow[u] = base + (size_t)__shfl_sync(0xffffffffu, t, (lane >> 2) + 8 * u) * HD;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if (i < sps) {
#pragma unroll
          for (int u = 0; u < 4; ++u) cp_async_16(rbase + i * SM::RAW + u * 512, arow[u] + i * XG_BK, 16);
        }
        cp_async_commit();
      }
      const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + TA + half * 24;
      auto put = [&](int i) {
        __syncwarp();
        if (i >= sps) return;
        uint32_t ph[8], pm[8], pl[8];
        raw16_split(sgen + SM::RAW_OFF + i * SM::RAW + warp * 2048, lane, ph, pm, pl);
        tmem_st8(ta + i * XG_A_STEP, ph);
        tmem_st8(ta + i * XG_A_STEP + 8, pm);
        tmem_st8(ta + i * XG_A_STEP + 16, pl);
      };
      cp_async_wait<3>(); put(0);
      cp_async_wait<2>(); put(1);
      cp_async_wait<1>(); put(2);
      cp_async_wait<0>(); put(3);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(a_full);
      asm volatile("bar.sync 1, 256;" ::: "memory");       // (the pieces' memory is the result's from here on)
    }
    const uint32_t acc_addr = tmem + ((uint32_t)(q * 32) << 16) + half * COLS;
    float* stg = reinterpret_cast<float*>(sgen + SM::STG_OFF);
    unsigned char* xrow = sgen + SM::X_OFF + warp * SM::X_WARP;
    // (the row of the result this thread hands on)
    float* orow = nullptr;
    if (tid < nrows) {
      if (MODE == X_O) { const int o = sh_out_row(d, t); if (o >= 0) orow = g.y + (size_t)o * d.M; }   // (cache tokens have no output row)
      else orow = g.dx + (size_t)t * d.M;
    }
    float dot = 0.f;
    for (int j = 0; j < tiles; ++j) {                       // (a wait that gives up does not leave the loop: the block's barriers are in it)
      const int n0 = (tile0 + j) * SM::BN, ncols = min(SM::BN, d.M - n0);
      if (MODE == X_DR) {
        // x of the same rows and columns, for the gate gradients: chunk c of row r at c ^ (r & 7)
        const float* xs = g.x + n0 + half * COLS + (lane & 7) * 4;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int rr = (lane >> 3) + 4 * u, tok = __shfl_sync(0xffffffffu, t, rr);
          cp_async_16(smem_u32(xrow) + rr * 128 + (((lane & 7) ^ (rr & 7)) << 4), xs + (size_t)tok * d.M, 16);
        }
        cp_async_commit();
      }
      mbar_wait(acc_full, j & 1, g.status, dead);
      tc_fence_after();
      float acc[COLS];
#pragma unroll
      for (int i = 0; i < COLS; ++i) acc[i] = 0.f;
      tmem_add(acc_addr + P2, acc);                        // (smallest first)
      tmem_add(acc_addr + P1, acc);
      if (k16s > 4) tmem_add(acc_addr + P3, acc);
      tmem_add(acc_addr + P0, acc);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
      if (MODE == X_DR) {
        cp_async_wait<0>();
        __syncwarp();
#pragma unroll
        for (int c = 0; c < COLS / 4; ++c) {
          const float4 o = *reinterpret_cast<const float4*>(xrow + lane * 128 + ((c ^ (lane & 7)) << 4));
          dot += (acc[4 * c] * o.x + acc[4 * c + 1] * o.y) + (acc[4 * c + 2] * o.z + acc[4 * c + 3] * o.w);
        }
        __syncwarp();                                      // (the next tile's copies)
      }
      bulk_wait_read_all();                                // the tile before has left the result rows
      asm volatile("bar.sync 1, 256;" ::: "memory");
#pragma unroll
      for (int i = 0; i < COLS; i += 4)
        *reinterpret_cast<float4*>(stg + r * SM::LD + half * COLS + i) = make_float4(acc[i] * gt, acc[i + 1] * gt, acc[i + 2] * gt, acc[i + 3] * gt);
      fence_proxy_async_smem();
      asm volatile("bar.sync 1, 256;" ::: "memory");
      if (orow && !dead) {
        if (MODE == X_O || g.vec_out) bulk_reduce_add_f32(orow + n0, smem_u32(stg + tid * SM::LD), ncols * 4);
        else
          for (int i = 0; i < ncols; ++i) atomicAdd(orow + n0 + i, stg[tid * SM::LD + i]);
      }
      bulk_commit();
    }
    if (MODE == X_DR && r < nrows && !dead) xg_gate_gradient<X_DR>(g, t, h, e, gt, dot);
    bulk_wait_all();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace shtc
