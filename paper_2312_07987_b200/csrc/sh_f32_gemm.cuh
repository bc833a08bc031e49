// fp32 contractions on the tensor cores: every projection of the fp32 configuration, forward and
// backward, but the weight gradients, which are in sh_f32_wgrad.cuh (their modes are numbered here: they share the
// arguments).
//
// An fp32 value is the exact sum of three bf16 values, x = h + m + l (8 + 8 + 8 mantissa bits: h is x
// rounded, m the rest rounded, l what is left), so a product of two is
//   hh' + (hm' + mh') + (hl' + mm' + lh') + terms below 2^-25 of it,
// six bf16 products.  The tensor core adds into fp32 but drops the bits below the accumulator's last one
// instead of rounding, so a long chain of additions drifts towards zero: the accumulators are read back
// and added in fp32 registers every 128 (64) contraction positions: 8 additions of hh', which carries the
// size of the result.
//
// Three UMMAs per 16 positions do the six products: the planes of B lie one behind the other, so that
// they are one operand of 192 columns, and with accumulator blocks P0 P1 P2 of 64 columns
//   h x [h' m' l'] -> P0 P1 P2,   m x [h' m'] -> P1 P2,   l x h' -> P2.
// (As six UMMAs of 64 columns the loop was bound by their issue, ~57 cycles each against 32 of tensor
// time: 2800 cycles a step of 64 positions.)
//
// Why not FFMA: the CUDA cores' 74 TFLOP/s fp32 peak against 2.25 PFLOP/s / 6 = 375.  What bounds a tile
// is latency: gather list -> rows -> split -> shared memory -> UMMA -> read-back, and a tile's set-up and
// result, 6 to 8 us of which little is work.  So a block is half an SM: 128 rows x 64 columns, contraction
// steps of 32, two stages of 36 KB, 256 worker threads; two blocks share an SM and fill each other's
// waits.  (One block per SM with 512 workers and steps of 64 ran the short contractions 1.5 times as long.)
//
// Weights are split once, when they are set, and come as planes by TMA (one box of all three planes).  An
// activation is read as fp32 by the workers, two steps ahead, by asynchronous copies into shared memory
// that only the copying warp uses (a prefetch that costs no registers and no block-wide barrier), split and
// stored into the swizzled planes.  One thread issues the UMMAs; the workers read the accumulators and
// write the result.
// Operands are addressed row by row (a gathered token list, a head's slice of a row), either as rows of
// the contraction (K-major) or as rows of the other index (MN-major: weights in the backward pass), so no
// transposed or gathered copy is made.  Results that are added to, and rows handed on whole, go through a
// padded copy in shared memory and leave as one bulk operation per row: as vector reductions from the
// accumulator layout (a lane per row, 16 bytes each) they were a third of the short contractions' time.
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

constexpr int XG_BN = 64, XG_BK = 32, XG_STAGES = 2;
struct XGemmSmem {
  static constexpr int A_PLANE = 128 * XG_BK * 2, B_PLANE = XG_BN * XG_BK * 2;
  static constexpr int STAGE = 3 * (A_PLANE + B_PLANE);
  static constexpr int RAW_OFF = XG_STAGES * STAGE, RAW = 128 * XG_BK * 4;     // fp32 pieces of a step, two steps
  static constexpr int BAR_OFF = RAW_OFF + 2 * RAW;
  static constexpr int TOTAL = BAR_OFF + 128 + 1024;
};

constexpr int XG_WORKERS = 256, XG_THREADS = XG_WORKERS + 64;   // + a warp that issues UMMAs, + one that loads weights
// Steps per promotion of the accumulators: 128 positions; 64 in contractions of up to 256, where an FFMA chain
// is short too and its error is the smaller one to stay below (64 everywhere: a quarter less error, 7 % more time).
__device__ __forceinline__ int xg_chunk(int steps) { return steps <= 8 ? 2 : 4; }

// K-major planes: rows of 32 values (64 bytes), 64-byte swizzle, 8-row groups 512 bytes apart.
constexpr uint32_t DESC_HI_SW64 = (512u >> 4) | (1u << 14) | (4u << 29);
__device__ __forceinline__ uint64_t xg_desc(uint32_t lo, bool mn_major) {
  return ((uint64_t)(mn_major ? DESC_HI_SW128 : DESC_HI_SW64) << 32) | lo;
}

// acc += 16 tensor-memory columns at a time (more in flight than that costs registers the operands need).
template <int N>
__device__ __forceinline__ void tmem_add(uint32_t taddr, float (&acc)[N]) {
#pragma unroll
  for (int c = 0; c < N; c += 16) {
    uint32_t u[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
          "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
        : "r"(taddr + c)
        : "memory");
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[c + i] += __uint_as_float(u[i]);
  }
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

// Eight values into the three planes at byte offset `off` of the operand's tile.
__device__ __forceinline__ void store_planes(unsigned char* tile, uint32_t off, int plane, const float (&v)[8]) {
  uint32_t h[4], m[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) split_bf16x3(v[2 * i], v[2 * i + 1], h[i], m[i], l[i]);
  *reinterpret_cast<uint4*>(tile + off) = make_uint4(h[0], h[1], h[2], h[3]);
  *reinterpret_cast<uint4*>(tile + off + plane) = make_uint4(m[0], m[1], m[2], m[3]);
  *reinterpret_cast<uint4*>(tile + off + 2 * plane) = make_uint4(l[0], l[1], l[2], l[3]);
}

// A warp's fp32 pieces of a step pass through 1 KB (64 chunks of 16 bytes) of shared memory that only this
// warp uses: copied chunk by chunk in the order of the rows, so that an instruction covers whole 128-byte
// lines, read as two neighbouring chunks (8 values of a row) by each lane.  Chunk c sits at c ^ (c >> 3 & 1):
// the eight lanes of a read phase then meet eight different 16-byte banks.
__device__ __forceinline__ uint32_t raw_chunk(int c) { return (uint32_t)((c ^ ((c >> 3) & 1)) << 4); }
__device__ __forceinline__ void fetch4(uint32_t dst, const float* p, bool vec, bool live = true) {
  if (vec) cp_async_16(dst, p, live ? 16 : 0);             // (a dead piece is zeros; its address is still a valid one)
  else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + i * 4), "l"(p + i), "r"(live ? 4 : 0) : "memory");
  }
}
__device__ __forceinline__ void read8(float (&v)[8], const unsigned char* kb, int c) {
  const float4 a = *reinterpret_cast<const float4*>(kb + raw_chunk(c)), b = *reinterpret_cast<const float4*>(kb + raw_chunk(c + 1));
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// acc += the row's gate times a value: four adjacent floats at a time when the row is 16-byte aligned.
template <int N>
__device__ __forceinline__ void red_row(float* dst, const float (&v)[N], int valid, bool vec) {
#pragma unroll
  for (int i = 0; i < N; i += 4) {
    if (vec && i + 4 <= valid) red_add_v4_f32(dst + i, v[i], v[i + 1], v[i + 2], v[i + 3]);
    else {
#pragma unroll
      for (int j = 0; j < 4; ++j) if (i + j < valid) atomicAdd(dst + i + j, v[i + j]);
    }
  }
}
template <int N>
__device__ __forceinline__ void store_row(float* dst, const float (&v)[N], int valid, bool vec) {
#pragma unroll
  for (int i = 0; i < N; i += 4) {
    if (vec && i + 4 <= valid) *reinterpret_cast<float4*>(dst + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    else {
#pragma unroll
      for (int j = 0; j < 4; ++j) if (i + j < valid) dst[i + j] = v[i + j];
    }
  }
}

// Token of a list entry (0 where the debug library finds that it is none).
__device__ __forceinline__ int xg_token(const XGemmArgs& g, size_t li) {
  const int t = g.lists[li];
  return SH_INDEX_OK(t, g.d.N, g.status, SH_SITE_V_LIST) ? t : 0;
}

struct XTile { int x, y, z; };           // which tile of its mode a block works on

// One tile.  mapW: planes of the mode's weights, rows [(which*H + h)*D + dd][m] (Q, K), [(h*E + e)*D + dd][m] (V),
// [(h*E + e)*M + m][dd] (O); mapG: of the gates' weights, rows [(side*H + h)*E + e][m].
template <int MODE>
__device__ __forceinline__ void xg_tile(const CUtensorMap& mapW, const CUtensorMap& mapG, const XGemmArgs& g, XTile blk) {
  using SM = XGemmSmem;
  constexpr int BN = XG_BN;
  constexpr bool B_MN = MODE >= X_DA;
  constexpr bool LIST_ROWS = MODE == X_V || MODE == X_O || MODE == X_DA || MODE == X_DR;
  constexpr bool ADDED = MODE != X_QK;                     // results that are added to (as one bulk operation per row; stored by X_QK)
  constexpr int COLS = BN / 2;                             // columns of a worker thread
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* sgen = smem_raw + (sbase - smem_u32(smem_raw));
  uint64_t* full_bar = (uint64_t*)(sgen + SM::BAR_OFF);    // [XG_STAGES]
  uint64_t* empty_bar = full_bar + XG_STAGES;              // [XG_STAGES]
  uint64_t* acc_full = empty_bar + XG_STAGES;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 1);
  const ShDims& d = g.d;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int HD = d.H * d.D;
  bool dead = false;

  pdl_trigger();
  if (tid == 0) {
    for (int s = 0; s < XG_STAGES; ++s) { mbar_init(&full_bar[s], 9); mbar_init(&empty_bar[s], 1); }
    mbar_init(acc_full, 1); mbar_init(acc_empty, 8);
    fence_barrier_init();
  }
  pdl_wait();
  // ---- which tile ------------------------------------------------------------------------------
  int h = 0, e = 0, which = 0, row0 = 0, nrows = 0, n0 = 0, ncols = 0, steps = 0;
  const int sps = (d.Dt + XG_BK - 1) / XG_BK;                        // steps over one head's d_head
  if (LIST_ROWS) {
    const ShTile tl = g.tiles[blk.x];
    if (tl.nrows == 0) return;                             // (before any allocation)
    if (!SH_INDEX_OK(tl.h, d.H, g.status, SH_SITE_V_TILE) || !SH_INDEX_OK(tl.e, d.E, g.status, SH_SITE_V_TILE) ||
        !SH_INDEX_OK(tl.nrows - 1, SH_TILE_ROWS, g.status, SH_SITE_V_TILE) || !SH_INDEX_OK(tl.row0, (long long)d.N * d.k - tl.nrows + 1, g.status, SH_SITE_V_TILE)) return;
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
  const int chunk = xg_chunk(steps);
  if (warp == 8) { tmem_alloc(tmem_slot, 256); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // contraction positions of step i that exist (the rest of the operand rows is zero)
  auto kvalid = [&](int i) -> int {
    i += s0;
    if (MODE == X_O || MODE == X_DR) return min(XG_BK, d.Dt - XG_BK * i);
    if (MODE == X_DX) {
      const int seg = i / sps;
      return seg < 2 * d.H ? min(XG_BK, d.Dt - (i - seg * sps) * XG_BK) : min(XG_BK, d.G - (i - 2 * d.H * sps) * XG_BK);
    }
    return XG_BK;
  };
  const uint32_t tmem = *tmem_slot;                        // accumulator blocks P0 P1 P2

  if (warp == 8) {
    if (lane == 0) {
      constexpr uint32_t maj = B_MN ? 1u << 16 : 0u;
      constexpr uint32_t id3 = make_idesc_f16(128, 192, 1, 1, 0) | maj, id2 = make_idesc_f16(128, 128, 1, 1, 0) | maj,
                         id1 = make_idesc_f16(128, 64, 1, 1, 0) | maj;
      const uint32_t a0 = desc_lo_k(sbase);
      const uint32_t b0 = B_MN ? desc_lo_mn(sbase + 3 * SM::A_PLANE, SM::B_PLANE) : desc_lo_k(sbase + 3 * SM::A_PLANE);
      constexpr uint32_t BK = B_MN ? 128 : 2, AP = SM::A_PLANE >> 4;
      int s = 0;
      uint32_t par = 0;
      for (int i = 0; i < steps && !dead; ++i) {
        if ((i & (chunk - 1)) == 0 && i > 0 && !mbar_wait(acc_empty, ((i / chunk) & 1) ^ 1, g.status, dead)) break;
        if (!mbar_wait(&full_bar[s], par, g.status, dead)) break;
        tc_fence_after();
        const uint32_t alo = a0 + s * (SM::STAGE >> 4), blo = b0 + s * (SM::STAGE >> 4);
        const int kn = (kvalid(i) + 15) / 16;
#pragma unroll
        for (int k = 0; k < XG_BK / 16; ++k) {
          if (k >= kn) break;
          const uint32_t a = alo + 2 * k;
          const uint64_t bb = xg_desc(blo + BK * k, B_MN);
          umma_f16(tmem, xg_desc(a, false), bb, id3, ((i & (chunk - 1)) | k) != 0);
          umma_f16(tmem + 64, xg_desc(a + AP, false), bb, id2, 1);
          umma_f16(tmem + 128, xg_desc(a + 2 * AP, false), bb, id1, 1);
        }
        umma_commit(&empty_bar[s]);
        if ((i & (chunk - 1)) == chunk - 1 || i == steps - 1) umma_commit(acc_full);
        if (++s == XG_STAGES) { s = 0; par ^= 1; }
      }
    }
    __syncwarp();
  } else if (warp == 9) {
    if (lane == 0) {
      int s = 0;
      uint32_t par = 1;
      for (int i = 0; i < steps && !dead; ++i) {
        if (!mbar_wait(&empty_bar[s], par, g.status, dead)) break;
        mbar_expect_tx(&full_bar[s], 3 * SM::B_PLANE);
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
        tma_load_3d(sbase + s * SM::STAGE + 3 * SM::A_PLANE, gm ? &mapG : &mapW, &full_bar[s], x, y, 0);
        if (++s == XG_STAGES) { s = 0; par ^= 1; }
      }
    }
    __syncwarp();
  } else {
    // ---- workers: operands, promotions, result -----------------------------------------------------
    // a thread's two pieces of a step: 8 values of rows ar and ar + 64
    const int ac = tid & 3, ar = tid >> 2;
    uint32_t aoff[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = ar + 64 * j;
      aoff[j] = (uint32_t)(r * 64 + ((ac ^ ((r >> 1) & 3)) << 4));
    }
    const size_t lbase = (size_t)h * d.N * d.k;
    const bool vdy = MODE != X_DA || g.vec_dy != 0;
    // What lies past the tile never needs masking, only an address inside the operand: rows past the last one
    // end in accumulators nobody reads, and positions past d_head (or the gate columns) are zeros in memory -
    // a step of 32 never leaves the stored d_head.
    // (copies: lane -> chunk lane & 7 of rows 8 warp + (lane >> 3) + 4 u + 64 j; a row's 32 positions are 8 chunks)
    const float* arow[2][2];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int r = row0 + min(8 * warp + (lane >> 3) + 4 * u + 64 * j, nrows - 1);
        const size_t t = LIST_ROWS ? xg_token(g, lbase + r) : r;
        arow[j][u] = (MODE == X_QK || MODE == X_V ? g.x + t * d.M
                    : MODE == X_O ? g.ahat + t * HD + h * d.D
                    : MODE == X_DA ? g.dy + t * d.M
                    : MODE == X_DR ? g.dv + t * HD + h * d.D : g.dq + t * HD) + (lane & 7) * 4;
      }
    int xseg = min(s0 / sps, 2 * d.H), xoff = (s0 - xseg * sps) * XG_BK;   // X_DX: the step's head (of dq, then dk), and where in it
    const uint32_t rbase = sbase + SM::RAW_OFF + warp * 2048;
    auto load = [&](int i) {                               // step i on its way
      long o = (long)(s0 + i) * XG_BK;
      if (MODE == X_DX) o = (xseg >= d.H ? (long)(g.dk - g.dq) + (long)(xseg - d.H) * d.D : (long)xseg * d.D) + xoff;
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const float* p = arow[j][u] + o;
          if (MODE == X_DX && xseg == 2 * d.H)
            p = g.dz + (size_t)(row0 + min(8 * warp + (lane >> 3) + 4 * u + 64 * j, nrows - 1)) * g.ldz + xoff + (lane & 7) * 4;
          fetch4(rbase + (i & 1) * SM::RAW + j * 1024 + raw_chunk(lane + 32 * u), p, vdy);
        }
      if (MODE == X_DX) {
        xoff += XG_BK;
        if (xseg < 2 * d.H && xoff >= d.Dt) { xoff = 0; ++xseg; }
      }
    };
    const int q = warp & 3, cb = warp >> 2;
    const uint32_t tlane = ((uint32_t)(q * 32) << 16) + cb * COLS;
    float acc[COLS];
#pragma unroll
    for (int i = 0; i < COLS; ++i) acc[i] = 0.f;
    const bool mine = cb * COLS < ncols;                   // (whole warps)
    auto promote = [&](int c) {
      if (!mbar_wait(acc_full, c & 1, g.status, dead)) return;
      tc_fence_after();
      if (mine) {
#pragma unroll
        for (int c0 = 0; c0 < COLS; c0 += 16) {
          float t[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) t[i] = 0.f;
          tmem_add<16>(tmem + 128 + tlane + c0, t);          // (smallest first)
          tmem_add<16>(tmem + 64 + tlane + c0, t);
          tmem_add<16>(tmem + tlane + c0, t);
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[c0 + i] += t[i];
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
    };
    load(0);
    cp_async_commit();
    if (steps > 1) load(1);
    cp_async_commit();
    int s = 0, done = 0;                                   // done: chunks promoted
    uint32_t par = 1;
    for (int i = 0; i < steps && !dead; ++i) {
      cp_async_wait<1>();                                  // this warp's pieces of step i are there
      __syncwarp();
      if (!mbar_wait(&empty_bar[s], par, g.status, dead)) break;
      unsigned char* at = sgen + s * SM::STAGE;
      const unsigned char* raw = sgen + SM::RAW_OFF + (i & 1) * SM::RAW + warp * 2048;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        float v[8];
        read8(v, raw + j * 1024, 2 * lane);
        store_planes(at, aoff[j], SM::A_PLANE, v);
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full_bar[s]);
      if (++s == XG_STAGES) { s = 0; par ^= 1; }
      if (i + 2 < steps) load(i + 2);
      cp_async_commit();
      // a chunk is read once two steps of the next one are in shared memory
      if ((i & (chunk - 1)) == 1 && i > chunk) promote(done++);
    }
    cp_async_wait<0>();
    for (; done < (steps + chunk - 1) / chunk && !dead; ++done) promote(done);
    // ---- result: thread = row q*32 + lane, columns cb*COLS ... ------------------------------------
    const int r = q * 32 + lane, c0 = cb * COLS;
    const int valid = min(COLS, ncols - c0);
    if (r < nrows && valid > 0 && !dead) {
      if (LIST_ROWS) {
        const size_t li = lbase + row0 + r;
        const int t = xg_token(g, li);
        const float gt = g.lgate[li];
        if (MODE == X_DA || MODE == X_DR) {
          // gate gradient: the ungated result against the forward operand of the same row
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
          // ds s (1 - s) is linear in ds, and rowsum(dahat o ahat) = sum over the selected experts of s ds: both are
          // added up here, part by part (kernels of their own for them: 5 us of a step)
          atomicAdd(g.dz + (size_t)t * g.ldz + ((MODE == X_DA ? d.H : 0) + h) * d.E + e, dot * gt * (1.f - gt));
          if (MODE == X_DA) atomicAdd(g.dsum + (size_t)t * d.H + h, gt * dot);
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
      // rows through shared memory (the operand stages are free: every UMMA has been waited for), 16 bytes of
      // padding a row so that eight lanes' 16-byte stores meet different banks
      constexpr int LD = BN + 4;
      float* stg = reinterpret_cast<float*>(sgen);
      if (r < nrows && valid > 0 && !dead) {
#pragma unroll
        for (int i = 0; i < COLS; i += 4)
          *reinterpret_cast<float4*>(stg + r * LD + c0 + i) = make_float4(acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
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
          const uint32_t src = smem_u32(stg + tid * LD);
          if (MODE == X_QK) bulk_store(o, src, n * 4);
          else if ((MODE != X_DR && MODE != X_DX) || g.vec_out) bulk_reduce_add_f32(o, src, n * 4);
          else
            for (int i = 0; i < n; ++i) atomicAdd(o + i, stg[tid * LD + i]);
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
    tmem_dealloc(tmem, 256);
  }
}

// Block number i of a mode's gx x gy x gz tiles.
__device__ __forceinline__ XTile xg_unpack(int i, int gx, int gy) { return {i % gx, i / gx % gy, i / (gx * gy)}; }

// A launch of one or two modes whose tiles do not depend on one another: the first blocks work on tiles
// of mode A, the rest on mode B.  (One launch each leaves half of the block slots idle in its last round,
// and pays its set-up and drain by itself.)
struct XPart { CUtensorMap w; XGemmArgs g; int gx, gy, n; };
template <int A, int B>
__global__ void __launch_bounds__(XG_THREADS, 2)
sh_f32_gemm_kernel(const __grid_constant__ CUtensorMap mapG, const __grid_constant__ XPart pa, const __grid_constant__ XPart pb) {
  const int i = blockIdx.x;
  if (B < 0 || i < pa.n) xg_tile<A>(pa.w, mapG, pa.g, xg_unpack(i, pa.gx, pa.gy));
  else xg_tile<(B >= 0 ? B : A)>(pb.w, mapG, pb.g, xg_unpack(i - pa.n, pb.gx, pb.gy));
}

}  // namespace shtc
