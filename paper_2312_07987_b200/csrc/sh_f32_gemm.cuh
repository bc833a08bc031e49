// fp32 contractions on the tensor cores: every projection of the fp32 configuration, forward and
// backward.
//
// An fp32 value is the exact sum of three bf16 values, x = h + m + l (8 + 8 + 8 mantissa bits: h is x
// rounded, m the rest rounded, l what is left), so a product of two is
//   hh' + (hm' + mh' + mm' + hl' + lh') + terms below 2^-25 of it,
// six bf16 UMMAs.  The tensor core adds into fp32 but drops the bits below the accumulator's last one
// instead of rounding, so a long chain of additions drifts towards zero: the hh' products, which carry
// the size of the result, go to an accumulator of their own that is read back and added in fp32
// registers every 128 contraction positions (8 additions); the five correction products, 2^-8 of it
// and smaller, share a second accumulator over the whole contraction.
//
// Why not FFMA: the CUDA cores' 74 TFLOP/s fp32 peak against 2.25 PFLOP/s / 6 = 375; what bounds this
// kernel is shared memory (a 128 x 128 x 16 UMMA reads 8 KB in 64 cycles, all an SM's shared memory
// delivers; the operand planes are written through it too).
//
// Tile: 128 rows x BN columns (64 or 128), contraction steps of 64.  512 worker threads read the fp32
// operands of step i + 1 into registers while the UMMAs of step i run, split them and store three
// 128-byte-swizzled planes per operand (two stages); one thread issues the UMMAs; the workers read
// the accumulators and write the result.  Operands are addressed row by row (a gathered token list, a
// head's slice of a row), either as rows of the contraction (K-major) or as rows of the other index
// (MN-major: the weight gradients contract over tokens), so no transposed or gathered copy is made.
#pragma once
#include "sh_tc_prims.cuh"

namespace shtc {

enum { X_QK = 0,    // z | q, k = x [Wgate | Wq | Wk]        rows: tokens
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
  const float *ahat, *dahat_in;          // [N, H, D]
  const float *dq, *dk, *dv, *dz;        // [N, H, D]; dz [N, ldz] (columns (side*H + h)*E + e)
  const float *wqk, *wgate, *wv, *wo;    // repacked weights: [(which*H + h)*D + dd][m], [g][m], [(h*E + e)*D + dd][m], [(h*E + e)*M + m][dd]
  int ldz;
  const int* lists; const float* lgate; const int* offsets; const ShTile* tiles;   // of the side the mode works on
  int nsub, sub_cols;                    // column tiles per head (or of M), and columns per tile (a multiple of 16)
  int qk_first, qk_groups;               // X_QK: first group ((which*H + h)) and how many
  int ksplit;                            // X_DW*: parts of the contraction (more than one: the results are added)
  float *q, *k, *v, *z;                  // X_QK: q, k [B, H, T, D], logits z [N, ldz]; X_V: v
  float *y;                              // X_O [rows of out, M]
  float *dahat, *ds, *dx;                // ds: gate gradients in list order
  float *dWq, *dWk, *dWv, *dWo, *dWs, *dWd;
  float *zero0, *zero1; long nzero0, nzero1;   // X_QK: buffers that later kernels add into (16-byte pieces), cleared beside the products
  float qscale, vscale;
  const float2* rope;
  int vec_dy, vec_out;                   // dy / the written gradients are 16-byte aligned
  int* status;
};

template <int BN>
struct XGemmSmem {
  static constexpr int A_PLANE = 128 * 128, B_PLANE = BN * 128;
  static constexpr int STAGE = 3 * (A_PLANE + B_PLANE);
  static constexpr int BAR_OFF = 2 * STAGE;
  static constexpr int TOTAL = BAR_OFF + 128 + 1024;
};

constexpr int XG_WORKERS = 512, XG_THREADS = XG_WORKERS + 32;
constexpr int XG_CHUNK = 2;              // steps per promotion of the main accumulator

template <int N>
__device__ __forceinline__ void tmem_ld_n(uint32_t taddr, float (&r)[N]);
template <>
__device__ __forceinline__ void tmem_ld_n<32>(uint32_t taddr, float (&r)[32]) {
  uint32_t u[32];
  tmem_ld32(taddr, u);
  tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < 32; ++i) r[i] = __uint_as_float(u[i]);
}
template <>
__device__ __forceinline__ void tmem_ld_n<16>(uint32_t taddr, float (&r)[16]) {
  uint32_t u[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(u[0]), "=r"(u[1]), "=r"(u[2]), "=r"(u[3]), "=r"(u[4]), "=r"(u[5]), "=r"(u[6]), "=r"(u[7]),
        "=r"(u[8]), "=r"(u[9]), "=r"(u[10]), "=r"(u[11]), "=r"(u[12]), "=r"(u[13]), "=r"(u[14]), "=r"(u[15])
      : "r"(taddr)
      : "memory");
  tmem_ld_wait();
#pragma unroll
  for (int i = 0; i < 16; ++i) r[i] = __uint_as_float(u[i]);
}

// Two fp32 values as three packed bf16 pairs whose sum they are.
__device__ __forceinline__ void split_bf16x3(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(h) : "f"(b), "f"(a));
  a -= __uint_as_float(h << 16); b -= __uint_as_float(h & 0xFFFF0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(m) : "f"(b), "f"(a));
  a -= __uint_as_float(m << 16); b -= __uint_as_float(m & 0xFFFF0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(l) : "f"(b), "f"(a));
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

// Eight consecutive values of a row; those at or past `valid` (and all of a null row) are zero.
__device__ __forceinline__ void load8(float (&v)[8], const float* p, int valid, bool vec) {
  if (p == nullptr || valid <= 0) {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = 0.f;
    return;
  }
  if (vec && valid >= 8) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p)), b = __ldg(reinterpret_cast<const float4*>(p) + 1);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    return;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = i < valid ? __ldg(p + i) : 0.f;
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

template <int BN, int MODE>
__global__ void __launch_bounds__(XG_THREADS, 1)
sh_f32_gemm_kernel(const __grid_constant__ XGemmArgs g) {
  using SM = XGemmSmem<BN>;
  constexpr bool A_MN = MODE == X_DWO || MODE == X_DWV || MODE == X_DWQK;
  constexpr bool B_MN = MODE >= X_DA;
  constexpr bool LIST_ROWS = MODE == X_V || MODE == X_O || MODE == X_DA || MODE == X_DR;
  constexpr bool LIST_K = MODE == X_DWO || MODE == X_DWV;
  constexpr int COLS = BN / 4;                             // columns of a worker thread
  constexpr int NB = BN / 64;                              // operand pieces (8 values) per thread: two of A, NB of B
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* sgen = smem_raw + (sbase - smem_u32(smem_raw));
  uint64_t* full_bar = (uint64_t*)(sgen + SM::BAR_OFF);    // [2]
  uint64_t* empty_bar = full_bar + 2;                      // [2]
  uint64_t* acc_full = empty_bar + 2;                      // [2]
  uint64_t* acc_empty = acc_full + 2;                      // [2]
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 2);
  const ShDims& d = g.d;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int HD = d.H * d.D;
  bool dead = false;

  pdl_trigger();
  if (tid == 0) {
    for (int s = 0; s < 2; ++s) { mbar_init(&full_bar[s], 16); mbar_init(&empty_bar[s], 1); mbar_init(&acc_full[s], 1); mbar_init(&acc_empty[s], 16); }
    fence_barrier_init();
  }
  pdl_wait();
  // ---- which tile ------------------------------------------------------------------------------
  int h = 0, e = 0, which = 0, row0 = 0, nrows = 0, n0 = 0, ncols = 0, m0 = 0, steps = 0;
  int kbeg = 0, kend = 0;                                  // LIST_K, X_DWQK: positions of the contraction
  bool gates = false;                                      // X_QK / X_DWQK: the tile of the gate columns
  const int sps = (d.Dt + 63) / 64;                        // steps over one head's d_head
  if (LIST_ROWS) {
    const ShTile tl = g.tiles[blockIdx.x];
    if (tl.nrows == 0) return;                             // (before any allocation)
    h = tl.h; e = tl.e; row0 = tl.row0; nrows = tl.nrows;
    n0 = blockIdx.y * g.sub_cols;
    ncols = min(g.sub_cols, ((MODE == X_O || MODE == X_DR) ? d.M : d.Dt) - n0);
    steps = (MODE == X_V || MODE == X_DA) ? d.M / 64 : sps;
  } else if (LIST_K) {
    const int grp = blockIdx.x / g.ksplit, part = blockIdx.x % g.ksplit;
    h = grp / d.E; e = grp % d.E;
    const int o0 = g.offsets[h * (d.E + 1) + e], o1 = g.offsets[h * (d.E + 1) + e + 1];
    const int per = (((o1 - o0 + 63) / 64 + g.ksplit - 1) / g.ksplit) * 64;
    kbeg = min(o1, o0 + part * per); kend = min(o1, kbeg + per);
    if (g.ksplit > 1 && kbeg >= kend) return;              // (the results are added to zeros)
    steps = (kend - kbeg + 63) / 64;
    n0 = blockIdx.y * g.sub_cols; m0 = blockIdx.z * 128;
    ncols = min(g.sub_cols, (MODE == X_DWO ? d.M : d.Dt) - n0);
    nrows = min(128, (MODE == X_DWO ? d.Dt : d.M) - m0);
  } else if (MODE == X_DX) {
    row0 = blockIdx.x * 128; nrows = min(128, d.N - row0);
    n0 = blockIdx.y * g.sub_cols; ncols = min(g.sub_cols, d.M - n0);
    steps = 2 * d.H * sps + (d.G + 63) / 64;
  } else {
    // X_QK, X_DWQK: column tiles 0 .. qk_groups*nsub - 1 are the heads' columns, the rest the gate columns
    const int ct = blockIdx.y;
    if (ct < g.qk_groups * g.nsub) {
      const int grp = g.qk_first + ct / g.nsub;
      which = grp / d.H; h = grp % d.H;
      n0 = (ct % g.nsub) * g.sub_cols; ncols = min(g.sub_cols, d.Dt - n0);
    } else {
      gates = true;
      n0 = (ct - g.qk_groups * g.nsub) * BN; ncols = min(BN, d.G - n0);
    }
    if (MODE == X_QK) {
      row0 = blockIdx.x * 128; nrows = min(128, d.N - row0);
      steps = d.M / 64;
    } else {
      m0 = blockIdx.x * 128; nrows = min(128, d.M - m0);
      const int per = (((d.N + 63) / 64 + g.ksplit - 1) / g.ksplit) * 64;
      kbeg = min(d.N, (int)blockIdx.z * per); kend = min(d.N, kbeg + per);
      if (g.ksplit > 1 && kbeg >= kend) return;
      steps = (kend - kbeg + 63) / 64;
    }
  }
  if (warp == 16) { tmem_alloc(tmem_slot, BN == 128 ? 512 : 256); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // contraction positions of step i that exist (the rest of the operand rows is zero)
  auto kvalid = [&](int i) -> int {
    if (MODE == X_O || MODE == X_DR) return min(64, d.Dt - 64 * i);
    if (A_MN) return min(64, kend - kbeg - 64 * i);
    if (MODE == X_DX) {
      const int seg = i / sps;
      return seg < 2 * d.H ? min(64, d.Dt - (i - seg * sps) * 64) : min(64, d.G - (i - 2 * d.H * sps) * 64);
    }
    return 64;
  };
  const uint32_t tmem = *tmem_slot;
  const uint32_t corr = tmem + 2 * BN;                     // columns: main 0, main 1, corrections
  const int chunks = (steps + XG_CHUNK - 1) / XG_CHUNK;
  const int nmma = (ncols + 15) & ~15;

  if (warp == 16) {
    if (lane == 0) {
      const uint32_t idesc = make_idesc_f16(128, nmma, 1, 1, B_MN ? 1 : 0) | (A_MN ? 1u << 15 : 0u);
      for (int i = 0; i < steps && !dead; ++i) {
        const int s = i & 1, c = i / XG_CHUNK, b = c & 1;
        if (i % XG_CHUNK == 0 && c >= 2 && !mbar_wait(&acc_empty[b], ((c >> 1) & 1) ^ 1, g.status, dead)) break;
        if (!mbar_wait(&full_bar[s], (i >> 1) & 1, g.status, dead)) break;
        tc_fence_after();
        const uint32_t abase = sbase + s * SM::STAGE, bbase = abase + 3 * SM::A_PLANE;
        const uint32_t alo = A_MN ? desc_lo_mn(abase, 8192) : desc_lo_k(abase);
        const uint32_t blo = B_MN ? desc_lo_mn(bbase, 8192) : desc_lo_k(bbase);
        constexpr uint32_t AK = A_MN ? 128 : 2, BK = B_MN ? 128 : 2;
        constexpr uint32_t AP = SM::A_PLANE >> 4, BP = SM::B_PLANE >> 4;
        const int kn = (kvalid(i) + 15) / 16;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (k >= kn) break;
          const uint32_t a = alo + AK * k, bb = blo + BK * k;
          umma_f16(tmem + b * BN, desc_pack(a), desc_pack(bb), idesc, (i % XG_CHUNK | k) != 0);
          umma_f16(corr, desc_pack(a + 2 * AP), desc_pack(bb), idesc, (i | k) != 0);
          umma_f16(corr, desc_pack(a), desc_pack(bb + 2 * BP), idesc, 1);
          umma_f16(corr, desc_pack(a + AP), desc_pack(bb + BP), idesc, 1);
          umma_f16(corr, desc_pack(a + AP), desc_pack(bb), idesc, 1);
          umma_f16(corr, desc_pack(a), desc_pack(bb + BP), idesc, 1);
        }
        umma_commit(&empty_bar[s]);
        if (i % XG_CHUNK == XG_CHUNK - 1 || i == steps - 1) umma_commit(&acc_full[b]);
      }
    }
    __syncwarp();
  } else {
    // ---- workers: operands, promotions, result -----------------------------------------------------
    // K-major pieces: 8 values of a row's 64 contraction positions; MN-major: 8 values of the row of
    // one contraction position
    const int ac = A_MN ? tid & 15 : tid & 7, ar = A_MN ? tid >> 4 : tid >> 3;    // + 32 j / + 64 j
    const int bc = B_MN && BN == 128 ? tid & 15 : tid & 7, br = B_MN && BN == 128 ? tid >> 4 : tid >> 3;
    constexpr int AR = A_MN ? 32 : 64, BR = B_MN && BN == 128 ? 32 : 64;
    uint32_t aoff[2], boff[NB];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int r = ar + AR * j;
      aoff[j] = A_MN ? (uint32_t)((ac >> 3) * 8192 + r * 128 + (((ac & 7) ^ (r & 7)) << 4)) : (uint32_t)(r * 128 + ((ac ^ (r & 7)) << 4));
    }
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const int r = br + BR * j;
      boff[j] = B_MN ? (uint32_t)((bc >> 3) * 8192 + r * 128 + (((bc & 7) ^ (r & 7)) << 4)) : (uint32_t)(r * 128 + ((bc ^ (r & 7)) << 4));
    }
    // rows that stay the same over the contraction
    const size_t lbase = (size_t)h * d.N * d.k;
    const float* arow[2] = {nullptr, nullptr};
    const float* brow[NB];
    int atok[2] = {0, 0};
    if (!A_MN) {
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int r = ar + AR * j;
        if (r < nrows) {
          const int t = LIST_ROWS ? g.lists[lbase + row0 + r] : row0 + r;
          atok[j] = t;
          arow[j] = MODE == X_QK || MODE == X_V ? g.x + (size_t)t * d.M
                  : MODE == X_O ? g.ahat + (size_t)t * HD + h * d.D
                  : MODE == X_DA ? g.dy + (size_t)t * d.M
                  : MODE == X_DR ? g.dv + (size_t)t * HD + h * d.D : g.dq;
        }
      }
    }
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const int r = br + BR * j;
      brow[j] = nullptr;
      if (!B_MN && r < ncols)
        brow[j] = MODE == X_QK ? (gates ? g.wgate + (size_t)(n0 + r) * d.M : g.wqk + ((size_t)(which * d.H + h) * d.D + n0 + r) * d.M)
                : MODE == X_V ? g.wv + ((size_t)(h * d.E + e) * d.D + n0 + r) * d.M
                : g.wo + ((size_t)(h * d.E + e) * d.M + n0 + r) * d.D;
    }
    float ra[2][8], rb[NB][8], rg[2] = {1.f, 1.f};
    auto load = [&](int i) {
      // A
      if (!A_MN) {
        const int kv = kvalid(i);
        int seg = 0, off = i * 64;
        if (MODE == X_DX) {
          seg = i / sps;
          off = seg < 2 * d.H ? (i - seg * sps) * 64 : (i - 2 * d.H * sps) * 64;
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const float* p = arow[j];
          if (MODE == X_DX && p) {
            p = seg < d.H ? g.dq + (size_t)atok[j] * HD + seg * d.D
              : seg < 2 * d.H ? g.dk + (size_t)atok[j] * HD + (seg - d.H) * d.D : g.dz + (size_t)atok[j] * g.ldz;
          }
          load8(ra[j], p ? p + off + ac * 8 : nullptr, kv - ac * 8, MODE == X_DA ? g.vec_dy != 0 : true);
        }
      } else {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int pos = kbeg + i * 64 + ar + 32 * j;
          const float* p = nullptr;
          rg[j] = 1.f;
          if (pos < kend) {
            const int t = LIST_K ? g.lists[lbase + pos] : pos;
            if (LIST_K) rg[j] = g.lgate[lbase + pos];
            p = MODE == X_DWO ? g.ahat + (size_t)t * HD + h * d.D + m0 : g.x + (size_t)t * d.M + m0;
          }
          load8(ra[j], p ? p + ac * 8 : nullptr, nrows - ac * 8, true);
        }
      }
      // B
      if (!B_MN) {
        const int kv = kvalid(i);
#pragma unroll
        for (int j = 0; j < NB; ++j) load8(rb[j], brow[j] ? brow[j] + i * 64 + bc * 8 : nullptr, kv - bc * 8, true);
      } else {
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          const int kr = br + BR * j;
          const float* p = nullptr;
          if (MODE == X_DA) p = g.wo + ((size_t)(h * d.E + e) * d.M + i * 64 + kr) * d.D + n0;
          if (MODE == X_DR && i * 64 + kr < d.Dt) p = g.wv + ((size_t)(h * d.E + e) * d.D + i * 64 + kr) * d.M + n0;
          if (MODE == X_DX) {
            const int seg = i / sps;
            if (seg < 2 * d.H) {
              const int dd = (i - seg * sps) * 64 + kr;
              if (dd < d.Dt) p = g.wqk + ((size_t)seg * d.D + dd) * d.M + n0;
            } else {
              const int gc = (i - 2 * d.H * sps) * 64 + kr;
              if (gc < d.G) p = g.wgate + (size_t)gc * d.M + n0;
            }
          }
          if (LIST_K || MODE == X_DWQK) {
            const int pos = kbeg + i * 64 + kr;
            if (pos < kend) {
              const int t = LIST_K ? g.lists[lbase + pos] : pos;
              p = MODE == X_DWO ? g.dy + (size_t)t * d.M + n0
                : MODE == X_DWV ? g.dv + (size_t)t * HD + h * d.D + n0
                : gates ? g.dz + (size_t)t * g.ldz + n0
                : (which ? g.dk : g.dq) + (size_t)t * HD + h * d.D + n0;
            }
          }
          load8(rb[j], p ? p + bc * 8 : nullptr, ncols - bc * 8, MODE == X_DWO ? g.vec_dy != 0 : true);
        }
      }
    };
    const int q = warp & 3, cb = warp >> 2;
    const uint32_t tlane = ((uint32_t)(q * 32) << 16) + cb * COLS;
    float acc[COLS];
#pragma unroll
    for (int i = 0; i < COLS; ++i) acc[i] = 0.f;
    const bool mine = cb * COLS < nmma;                    // (whole warps: columns past the tile's are not computed)
    auto promote = [&](int c) {
      const int b = c & 1;
      if (!mbar_wait(&acc_full[b], (c >> 1) & 1, g.status, dead)) return;
      tc_fence_after();
      if (mine) {
        float t[COLS];
        tmem_ld_n<COLS>(tmem + b * BN + tlane, t);
#pragma unroll
        for (int i = 0; i < COLS; ++i) acc[i] += t[i];
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[b]);
    };
    if (steps > 0) load(0);
    if (MODE == X_QK) {
      const long n = (long)gridDim.x * gridDim.y * XG_WORKERS, i0 = ((long)blockIdx.y * gridDim.x + blockIdx.x) * XG_WORKERS + tid;
      for (long i = i0; i < g.nzero0; i += n) reinterpret_cast<float4*>(g.zero0)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      for (long i = i0; i < g.nzero1; i += n) reinterpret_cast<float4*>(g.zero1)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int i = 0; i < steps; ++i) {
      const int s = i & 1;
      if (i >= 2 && !mbar_wait(&empty_bar[s], ((i >> 1) & 1) ^ 1, g.status, dead)) break;
      unsigned char* at = sgen + s * SM::STAGE;
      unsigned char* bt = at + 3 * SM::A_PLANE;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (LIST_K) {
#pragma unroll
          for (int x = 0; x < 8; ++x) ra[j][x] *= rg[j];
        }
        store_planes(at, aoff[j], SM::A_PLANE, ra[j]);
      }
#pragma unroll
      for (int j = 0; j < NB; ++j) store_planes(bt, boff[j], SM::B_PLANE, rb[j]);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full_bar[s]);
      if (i + 1 < steps) load(i + 1);
      if (i % XG_CHUNK == XG_CHUNK - 1 && i / XG_CHUNK >= 1) promote(i / XG_CHUNK - 1);
    }
    // chunks not read yet: the last one, and the one before it when the last is a short one
    if (steps > 0) {
      const int done = steps / XG_CHUNK >= 1 ? steps / XG_CHUNK - 1 : 0;      // chunks promoted in the loop
      for (int c = done; c < chunks; ++c) promote(c);
      if (mine && !dead) {
        float t[COLS];
        tmem_ld_n<COLS>(corr + tlane, t);                  // (complete: the last chunk's commit came behind its UMMAs)
#pragma unroll
        for (int i = 0; i < COLS; ++i) acc[i] += t[i];
      }
    }
    // ---- result: thread = row q*32 + lane, columns cb*COLS ... ------------------------------------
    const int r = q * 32 + lane, c0 = cb * COLS;
    const int valid = min(COLS, ncols - c0);
    if (r < nrows && valid > 0 && !dead) {
      if (LIST_ROWS) {
        const size_t li = lbase + row0 + r;
        const int t = g.lists[li];
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
          atomicAdd(g.ds + li, dot);
        }
        const float f = MODE == X_V && g.vscale != 0.f ? gt * g.vscale : gt;
#pragma unroll
        for (int i = 0; i < COLS; ++i) acc[i] *= f;
        if (MODE == X_V) {
          const int b = t / d.T, tt = t % d.T;
          red_row(g.v + (((size_t)b * d.H + h) * d.T + tt) * d.D + n0 + c0, acc, valid, true);
        } else if (MODE == X_O) {
          const int orow = sh_out_row(d, t);               // (cache tokens have no output row)
          if (orow >= 0) red_row(g.y + (size_t)orow * d.M + n0 + c0, acc, valid, true);
        } else if (MODE == X_DA) {
          red_row(g.dahat + (size_t)t * HD + h * d.D + n0 + c0, acc, valid, true);
        } else {
          red_row(g.dx + (size_t)t * d.M + n0 + c0, acc, valid, g.vec_out != 0);
        }
      } else if (LIST_K) {
        // dWo [(h*E + e)*Dt + dd][m]; dWv [(h*E + e)*M + m][dd < Dt]
        float* o = MODE == X_DWO ? g.dWo + ((size_t)(h * d.E + e) * d.Dt + m0 + r) * d.M + n0 + c0
                                 : g.dWv + ((size_t)(h * d.E + e) * d.M + m0 + r) * d.Dt + n0 + c0;
        const bool vec = g.vec_out != 0 && (MODE == X_DWO || d.Dt % 4 == 0);
        if (g.ksplit > 1) red_row(o, acc, valid, vec);
        else store_row(o, acc, valid, vec);
      } else if (MODE == X_DX) {
        float* o = g.dx + (size_t)(row0 + r) * d.M + n0 + c0;
#pragma unroll
        for (int i = 0; i < COLS; i += 4) {
          if (i + 4 <= valid && g.vec_out) {
            float4 p = *reinterpret_cast<const float4*>(o + i);
            p.x += acc[i]; p.y += acc[i + 1]; p.z += acc[i + 2]; p.w += acc[i + 3];
            *reinterpret_cast<float4*>(o + i) = p;
          } else {
#pragma unroll
            for (int j = 0; j < 4; ++j) if (i + j < valid) o[i + j] += acc[i + j];
          }
        }
      } else if (MODE == X_DWQK) {
        const int m = m0 + r;
        if (!gates) {
          float* o = (which ? g.dWk : g.dWq) + ((size_t)h * d.M + m) * d.Dt + n0 + c0;
          const bool vec = g.vec_out != 0 && d.Dt % 4 == 0;
          if (g.ksplit > 1) red_row(o, acc, valid, vec);
          else store_row(o, acc, valid, vec);
        } else {
#pragma unroll
          for (int i = 0; i < COLS; ++i)
            if (i < valid) {
              const int gc = n0 + c0 + i, side = gc / (d.H * d.E), hh = (gc / d.E) % d.H, ee = gc % d.E;
              float* o = (side ? g.dWd : g.dWs) + ((size_t)hh * d.M + m) * d.E + ee;
              if (g.ksplit > 1) atomicAdd(o, acc[i]);
              else *o = acc[i];
            }
        }
      } else {                                             // X_QK
        const int tok = row0 + r;
        if (gates) {
          store_row(g.z + (size_t)tok * g.ldz + n0 + c0, acc, valid, true);
        } else {
          const int b = tok / d.T, t = tok % d.T;
          if (g.rope) {
            const float2* cs = g.rope + (size_t)((n0 + c0) >> 1) * d.T + t;
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
          // (columns between d_head and its stored width: zero, as the padded weight rows would give)
          float* o = (which ? g.k : g.q) + (((size_t)b * d.H + h) * d.T + t) * d.D + n0 + c0;
          store_row(o, acc, valid, true);
        }
      }
    }
    if (MODE == X_QK && !gates && n0 + ncols >= d.Dt && d.D > d.Dt && !dead && cb == 0 && r < nrows) {
      const int tok = row0 + r, b = tok / d.T, t = tok % d.T;
      float* o = (which ? g.k : g.q) + (((size_t)b * d.H + h) * d.T + t) * d.D;
      for (int i = d.Dt; i < d.D; ++i) o[i] = 0.f;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 16) {
    tc_fence_after();
    tmem_dealloc(tmem, BN == 128 ? 512 : 256);
  }
}

}  // namespace shtc
