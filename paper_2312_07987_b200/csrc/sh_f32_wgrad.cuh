// Weight gradients of the fp32 configuration: contractions over tokens, both operands activations.
//   X_DWV  dWv[h, e]  = sum over the list of value expert (h, e):  (g x[t])^T dv[t, h]
//   X_DWO  dWo[h, e]  = sum over the list of output expert (h, e): (g ahat[t, h])^T dy[t]
//   X_DWQK dWq[h], dWk[h], dWs, dWd = sum over all tokens: x[t]^T [dq dk dz][t]
//
// The split products, accumulators and promotion are those of sh_f32_gemm.cuh; both operands are
// MN-major (a row of shared memory is 64 columns of one token).  Tile 128 x 128 (B as two halves of 64
// columns, each with its three accumulator blocks), steps of 32 tokens.  Both operands pass through the
// worker threads, so what bounds a step is shared memory (208 KB of traffic, about 1600 cycles) - if the
// gathered rows are there in time: list entry -> row is two dependent trips to L2.  One block per SM with
// 512 workers, the rows of the next three steps on their way by asynchronous copies into warp-private memory
// and the list entries of one more in registers.  (262M-scale step, 2 x 512 tokens: 328 tiles in 96 us;
// 648 tiles of 64 columns took 108, of which a third was their set-up and drain; as modes of the half-SM
// kernel 150.)
#pragma once
#include "sh_f32_gemm.cuh"

namespace shtc {

// acc += 16 tensor-memory columns at a time (more in flight than that costs registers the operands need).
template <int N>
__device__ __forceinline__ void tmem_add16(uint32_t taddr, float (&acc)[N]) {
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


struct XWgradSmem {
  static constexpr int A_PLANE = 128 * XG_BK * 2, B_PLANE = 64 * XG_BK * 2, B_HALF = 3 * B_PLANE;
  static constexpr int STAGES = 2, STAGE = 3 * A_PLANE + 2 * B_HALF;
  static constexpr int NRAW = 3, RAW_A = 128 * XG_BK * 4, RAW = 2 * RAW_A;
  static constexpr int RAW_OFF = STAGES * STAGE;
  static constexpr int BAR_OFF = RAW_OFF + NRAW * RAW;
  static constexpr int TOTAL = BAR_OFF + 128 + 1024;
};
constexpr int XW_WORKERS = 512, XW_THREADS = XW_WORKERS + 32, XW_BN = 128;

template <int MODE>
__device__ __forceinline__ void xw_tile(const XGemmArgs& g, XTile blk) {
  using SM = XWgradSmem;
  constexpr bool LIST = MODE != X_DWQK;
  constexpr int COLS = XW_BN / 4;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* sgen = smem_raw + (sbase - smem_u32(smem_raw));
  uint64_t* full_bar = (uint64_t*)(sgen + SM::BAR_OFF);    // [STAGES]
  uint64_t* empty_bar = full_bar + SM::STAGES;             // [STAGES]
  uint64_t* acc_full = empty_bar + SM::STAGES;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = (uint32_t*)(acc_empty + 1);
  const ShDims& d = g.d;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int HD = d.H * d.D;
  bool dead = false;

  pdl_trigger();
  if (tid == 0) {
    for (int s = 0; s < SM::STAGES; ++s) { mbar_init(&full_bar[s], 16); mbar_init(&empty_bar[s], 1); }
    mbar_init(acc_full, 1); mbar_init(acc_empty, 16);
    fence_barrier_init();
  }
  pdl_wait();
  int h = 0, e = 0, which = 0, n0, ncols, m0, nrows, kbeg, kend;
  bool gates = false;                                      // X_DWQK: a tile of the gate columns
  if (LIST) {
    const int grp = blk.x / g.ksplit, part = blk.x % g.ksplit;
    h = grp / d.E; e = grp % d.E;
    const int o0 = g.offsets[h * (d.E + 1) + e], o1 = g.offsets[h * (d.E + 1) + e + 1];
    if (!SH_INDEX_OK(o0, (long long)d.N * d.k + 1, g.status, SH_SITE_V_TILE) || !SH_INDEX_OK(o1, (long long)d.N * d.k + 1, g.status, SH_SITE_V_TILE)) return;
    const int per = (((o1 - o0 + XG_BK - 1) / XG_BK + g.ksplit - 1) / g.ksplit) * XG_BK;
    kbeg = min(o1, o0 + part * per); kend = min(o1, kbeg + per);
    n0 = blk.y * g.sub_cols; m0 = blk.z * 128;
    ncols = min(g.sub_cols, (MODE == X_DWO ? d.M : d.Dt) - n0);
    nrows = min(128, (MODE == X_DWO ? d.Dt : d.M) - m0);
  } else {
    // column tiles 0 .. qk_groups*nsub - 1 are the heads' columns, the rest the gate columns
    if (blk.y < g.qk_groups * g.nsub) {
      const int grp = blk.y / g.nsub;
      which = grp / d.H; h = grp % d.H;
      n0 = (blk.y % g.nsub) * g.sub_cols; ncols = min(g.sub_cols, d.Dt - n0);
    } else {
      gates = true;
      n0 = (blk.y - g.qk_groups * g.nsub) * XW_BN; ncols = min(XW_BN, d.G - n0);
    }
    m0 = blk.x * 128; nrows = min(128, d.M - m0);
    const int per = (((d.N + XG_BK - 1) / XG_BK + g.ksplit - 1) / g.ksplit) * XG_BK;
    kbeg = min(d.N, blk.z * per); kend = min(d.N, kbeg + per);
  }
  if (g.ksplit > 1 && kbeg >= kend) return;                // (the results are added to zeros)
  const int steps = (kend - kbeg + XG_BK - 1) / XG_BK;
  const int chunk = steps <= 8 ? 2 : 4;
  if (warp == 16) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;                        // accumulator blocks P0 P1 P2 of the two halves, 192 columns apart

  if (warp == 16) {
    if (lane == 0) {
      constexpr uint32_t maj = 1u << 16 | 1u << 15;
      constexpr uint32_t id3 = make_idesc_f16(128, 192, 1, 1, 0) | maj, id2 = make_idesc_f16(128, 128, 1, 1, 0) | maj,
                         id1 = make_idesc_f16(128, 64, 1, 1, 0) | maj;
      const uint32_t a0 = desc_lo_mn(sbase, 64 * XG_BK * 2), b0 = desc_lo_mn(sbase + 3 * SM::A_PLANE, SM::B_PLANE);
      constexpr uint32_t AP = SM::A_PLANE >> 4;
      const int halves = ncols > 64 ? 2 : 1;
      int s = 0;
      uint32_t par = 0;
      for (int i = 0; i < steps && !dead; ++i) {
        if ((i & (chunk - 1)) == 0 && i > 0 && !mbar_wait(acc_empty, ((i / chunk) & 1) ^ 1, g.status, dead)) break;
        if (!mbar_wait(&full_bar[s], par, g.status, dead)) break;
        tc_fence_after();
        const uint32_t alo = a0 + s * (SM::STAGE >> 4), blo = b0 + s * (SM::STAGE >> 4);
        const int kn = (min(XG_BK, kend - kbeg - XG_BK * i) + 15) / 16;
#pragma unroll
        for (int k = 0; k < XG_BK / 16; ++k) {
          if (k >= kn) break;
          const uint32_t a = alo + 128 * k;
          for (int hf = 0; hf < halves; ++hf) {
            const uint32_t td = tmem + hf * 192;
            const uint64_t bb = xg_desc(blo + hf * (SM::B_HALF >> 4) + 128 * k, true);
            umma_f16(td, xg_desc(a, true), bb, id3, ((i & (chunk - 1)) | k) != 0);
            umma_f16(td + 64, xg_desc(a + AP, true), bb, id2, 1);
            umma_f16(td + 128, xg_desc(a + 2 * AP, true), bb, id1, 1);
          }
        }
        umma_commit(&empty_bar[s]);
        if ((i & (chunk - 1)) == chunk - 1 || i == steps - 1) umma_commit(acc_full);
        if (++s == SM::STAGES) { s = 0; par ^= 1; }
      }
    }
    __syncwarp();
  } else {
    // a thread's pieces of a step: 8 columns (ac) of token row ar, of A and of B
    const int ac = tid & 15, ar = tid >> 4;
    const uint32_t poff = (uint32_t)(ar * 128 + (((ac & 7) ^ (ar & 7)) << 4));
    const uint32_t aoff = (ac >> 3) * (64 * XG_BK * 2) + poff, boff = (ac >> 3) * SM::B_HALF + poff;
    const size_t lbase = (size_t)h * d.N * d.k;
    const bool vdy = MODE != X_DWO || g.vec_dy != 0;
    // (columns past the operands' widths end in accumulators nobody reads: any address inside the row will do)
    const int acol = min(m0 + lane * 4, (MODE == X_DWO ? d.D : d.M) - 4);
    const int bcol = min(n0 + lane * 4, (MODE == X_DWO ? d.M : gates ? g.ldz : d.D) - 4);
    const float* asrc = (MODE == X_DWO ? g.ahat + h * d.D : g.x) + acol;
    const size_t ald = MODE == X_DWO ? HD : d.M;
    const float* bsrc = (MODE == X_DWO ? g.dy : MODE == X_DWV ? g.dv + h * d.D : gates ? g.dz : (which ? g.dk : g.dq) + h * d.D) + bcol;
    const size_t bld = MODE == X_DWO ? d.M : gates ? g.ldz : HD;
    // copies: a warp's two token rows are two instructions, of A and of B
    int ta[2] = {0, 0};                                    // the next step's tokens
    float gnext = 0.f;
    auto entries = [&](int i) {
      const int p0 = kbeg + i * XG_BK;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int pa = p0 + 2 * warp + u;
        if (!LIST) ta[u] = min(pa, d.N - 1);
        else if (pa < kend) ta[u] = xg_token(g, lbase + pa);
      }
      if (LIST && p0 + ar < kend) gnext = __ldg(g.lgate + lbase + p0 + ar);
    };
    float gring[SM::NRAW];                                 // gates of the steps on their way
    auto load = [&](int i, int slot) {
      const uint32_t raw = sbase + SM::RAW_OFF + slot * SM::RAW + warp * 1024;
      const int p0 = kbeg + i * XG_BK;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const bool live = p0 + 2 * warp + u < kend;
        fetch4(raw + raw_chunk(lane + 32 * u), asrc + (size_t)ta[u] * ald, true, live);
        fetch4(raw + SM::RAW_A + raw_chunk(lane + 32 * u), bsrc + (size_t)ta[u] * bld, vdy, live);
      }
    };
    const int q = warp & 3, cb = warp >> 2;
    float acc[COLS];
#pragma unroll
    for (int i = 0; i < COLS; ++i) acc[i] = 0.f;
    const bool mine = cb * COLS < ncols;                   // (whole warps)
    auto promote = [&](int c) {
      if (!mbar_wait(acc_full, c & 1, g.status, dead)) return;
      tc_fence_after();
      if (mine) {
        const uint32_t tb = tmem + (cb >> 1) * 192 + ((uint32_t)(q * 32) << 16) + (cb & 1) * 32;
#pragma unroll
        for (int c0 = 0; c0 < COLS; c0 += 16) {
          float t[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) t[i] = 0.f;
          tmem_add16(tb + 128 + c0, t);                    // (smallest first)
          tmem_add16(tb + 64 + c0, t);
          tmem_add16(tb + c0, t);
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[c0 + i] += t[i];
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acc_empty);
    };
    if (steps > 0) entries(0);
#pragma unroll
    for (int u = 0; u < SM::NRAW; ++u) {
      gring[u] = gnext;
      if (u < steps) { load(u, u); if (u + 1 < steps) entries(u + 1); }
      cp_async_commit();
    }
    int s = 0, done = 0;
    uint32_t par = 1;
    for (int i0 = 0; i0 < steps && !dead; i0 += SM::NRAW) {
#pragma unroll
      for (int u = 0; u < SM::NRAW; ++u) {
        const int i = i0 + u;
        if (i >= steps) break;
        cp_async_wait<SM::NRAW - 1>();
        __syncwarp();
        if (!mbar_wait(&empty_bar[s], par, g.status, dead)) break;
        unsigned char* at = sgen + s * SM::STAGE;
        const unsigned char* raw = sgen + SM::RAW_OFF + u * SM::RAW + warp * 1024;
        float v[8];
        read8(v, raw, 2 * lane);
        if (LIST) {
#pragma unroll
          for (int x = 0; x < 8; ++x) v[x] *= gring[u];
        }
        store_planes(at, aoff, SM::A_PLANE, v);
        read8(v, raw + SM::RAW_A, 2 * lane);
        store_planes(at + 3 * SM::A_PLANE, boff, SM::B_PLANE, v);
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(&full_bar[s]);
        if (++s == SM::STAGES) { s = 0; par ^= 1; }
        if (i + SM::NRAW < steps) {
          gring[u] = gnext;
          load(i + SM::NRAW, u);
          if (i + SM::NRAW + 1 < steps) entries(i + SM::NRAW + 1);
        }
        cp_async_commit();
        if ((i & (chunk - 1)) == 1 && i > chunk) promote(done++);
      }
    }
    cp_async_wait<0>();
    for (; done < (steps + chunk - 1) / chunk && !dead; ++done) promote(done);
    const int r = q * 32 + lane, c0 = cb * COLS;
    const int valid = min(COLS, ncols - c0);
    if (r < nrows && valid > 0 && !dead) {
      const int m = m0 + r;
      if (!gates) {
        // dWo [(h*E + e)*Dt + dd][m]; dWv [(h*E + e)*M + m][dd < Dt]; dWq, dWk [h*M + m][dd < Dt]
        float* o = (MODE == X_DWO ? g.dWo + ((size_t)(h * d.E + e) * d.Dt + m) * d.M
                  : MODE == X_DWV ? g.dWv + ((size_t)(h * d.E + e) * d.M + m) * d.Dt
                  : (which ? g.dWk : g.dWq) + ((size_t)h * d.M + m) * d.Dt) + n0 + c0;
        const bool vec = g.vec_out != 0 && (MODE == X_DWO || d.Dt % 4 == 0);
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
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 16) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// All weight gradients in one launch: tiles of X_DWQK (the longest contractions) first.
struct XWPart { XGemmArgs g; int gx, gy, n; };
static __global__ void __launch_bounds__(XW_THREADS, 1)
sh_f32_wgrad_kernel(const __grid_constant__ XWPart pq, const __grid_constant__ XWPart pv, const __grid_constant__ XWPart po) {
  int i = blockIdx.x;
  if (i < pq.n) { xw_tile<X_DWQK>(pq.g, xg_unpack(i, pq.gx, pq.gy)); return; }
  i -= pq.n;
  if (i < pv.n) { xw_tile<X_DWV>(pv.g, xg_unpack(i, pv.gx, pv.gy)); return; }
  xw_tile<X_DWO>(po.g, xg_unpack(i - pv.n, po.gx, po.gy));
}

}  // namespace shtc
