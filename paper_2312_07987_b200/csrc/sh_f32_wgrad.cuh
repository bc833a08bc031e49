// Weight gradients of the fp32 configuration: contractions over tokens, both operands activations.
//   X_DWV  dWv[h, e]  = sum over the list of value expert (h, e):  (g x[t])^T dv[t, h]
//   X_DWO  dWo[h, e]^T = sum over the list of output expert (h, e): (g dy[t])^T ahat[t, h]
//   X_DWQK dWq[h], dWk[h], dWs, dWd = sum over all tokens: x[t]^T [dq dk dz][t]
//
// The split products, accumulators and promotion are those of sh_f32_gemm.cuh: tile 128 (columns of x or dy) x up to
// 128 (a head's columns), steps of 32 tokens, operand A in tensor memory, B as MN-major planes in shared memory.  A warp
// copies 8 tokens x 32 columns of each operand into memory of its own, four steps ahead (the list entries two more), and
// splits them: for A a lane takes a column (its tensor-memory lane) of the 8 tokens, for B eight columns of one.
// Shared-memory traffic per step 136 KB, 1060 cycles, against 768 of tensor time (with A's planes there as well: 208 KB,
// 1600 cycles).  One block per SM, 512 workers.  2 x 512 tokens, d_model 1024, 4 heads of 112: 328 tiles, 92 -> 84 us behind dx;
// 8 x 256 tokens, d_model 448, 2 heads of 76: 60 -> 51 us.  What bounds it: 2.2 rounds of tiles, each with its set-up and drain, and
// the hand-overs of a step, as in sh_f32_gemm.cuh.  The warp that issues UMMAs is a seventeenth, which leaves 96 registers a thread (128
// with 16 warps): 72 bytes of spills stored and 220 loaded.
#pragma once
#include "sh_f32_gemm.cuh"

namespace shtc {

struct XWgradSmem {
  static constexpr int B_PLANE = 64 * XG_BK * 2, B_HALF = 3 * B_PLANE, B_STEP = 2 * B_HALF;
  static constexpr int NR = 4, RAW_A = 128 * XG_BK * 4, RAW = 2 * RAW_A;
  static constexpr int RAW_OFF = 2 * B_STEP;
  static constexpr int GATE_OFF = RAW_OFF + NR * RAW;     // [NR][16 warps][8] gates
  static constexpr int BAR_OFF = GATE_OFF + NR * 512;
  static constexpr int TOTAL = BAR_OFF + 256 + 1024;
};
constexpr int XW_WORKERS = 512, XW_THREADS = XW_WORKERS + 32, XW_BN = 128;

__device__ __forceinline__ void tmem_st4(uint32_t taddr, const uint32_t (&r)[4]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]) : "memory");
}

template <int MODE>
__device__ __forceinline__ void xw_tile(const XGemmArgs& g, XTile blk) {
  using SM = XWgradSmem;
  constexpr bool LIST = MODE != X_DWQK;
  constexpr int COLS = XW_BN / 4;
  constexpr uint32_t P0 = 0, P1 = 256, TA = 384;           // tensor-memory columns
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* sgen = smem_raw + (sbase - smem_u32(smem_raw));
  uint64_t* full = (uint64_t*)(sgen + SM::BAR_OFF);        // [2] the step's planes are written
  uint64_t* done = full + 2;                               // [2] its UMMAs are done
  uint64_t* acc_full = done + 2;                           // [2] P0 of a chunk is complete
  uint64_t* acc_empty = acc_full + 2;                      // [2] ... and has been read
  uint64_t* p1_empty = acc_empty + 2;
  uint32_t* tmem_slot = (uint32_t*)(p1_empty + 1);
  const ShDims& d = g.d;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int HD = d.H * d.D;
  bool dead = false;

  int h = 0, e = 0, which = 0, n0, ncols, m0, nrows, kbeg, kend;
  bool gates = false;                                      // X_DWQK: a tile of the gate columns
  if (LIST) {
    const int grp = blk.x / g.ksplit, part = blk.x % g.ksplit;
    h = grp / d.E; e = grp % d.E;
    const int o0 = g.offsets[h * (d.E + 1) + e], o1 = g.offsets[h * (d.E + 1) + e + 1];
    if (!SH_INDEX_OK(o0, (long long)d.N * d.k + 1, g.status, SH_SITE_V_TILE) || !SH_INDEX_OK(o1, (long long)d.N * d.k + 1, g.status, SH_SITE_V_TILE)) return;
    const int per = (((o1 - o0 + XG_BK - 1) / XG_BK + g.ksplit - 1) / g.ksplit) * XG_BK;
    kbeg = min(o1, o0 + part * per); kend = min(o1, kbeg + per);
    n0 = blk.y * g.sub_cols; ncols = min(g.sub_cols, d.Dt - n0);
    m0 = blk.z * 128;
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
    m0 = blk.x * 128;
    const int per = (((d.N + XG_BK - 1) / XG_BK + g.ksplit - 1) / g.ksplit) * XG_BK;
    kbeg = min(d.N, blk.z * per); kend = min(d.N, kbeg + per);
  }
  nrows = min(128, d.M - m0);
  if (g.ksplit > 1 && kbeg >= kend) return;                // (the results are added to zeros)
  const int steps = (kend - kbeg + XG_BK - 1) / XG_BK;
  const int nchunk = (steps + XG_CHUNK - 1) / XG_CHUNK;
  if (tid == 0) {
    for (int s = 0; s < 2; ++s) { mbar_init(&full[s], 16); mbar_init(&done[s], 1); mbar_init(&acc_full[s], 1); mbar_init(&acc_empty[s], 16); }
    mbar_init(p1_empty, 16);
    fence_barrier_init();
  }
  if (warp == 16) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 16) {
    if (lane == 0) {
      const uint32_t id = xg_idesc((ncols + 15) & ~15, true);
      const uint32_t b0 = desc_lo_mn(sbase, SM::B_HALF);
      constexpr uint32_t BP = SM::B_PLANE >> 4;
      for (int i = 0; i < steps && !dead; ++i) {
        const int c = i / XG_CHUNK;                          // (powers of two: a division costs this thread as much as two UMMAs)
        if (i % XG_CHUNK == 0) {
          if (!mbar_wait(&acc_empty[c & 1], ((c >> 1) & 1) ^ 1, g.status, dead)) break;
          if (c > 0 && c % XG_P1_CHUNKS == 0 && !mbar_wait(p1_empty, (c / XG_P1_CHUNKS - 1) & 1, g.status, dead)) break;
        }
        if (!mbar_wait(&full[i & 1], (i >> 1) & 1, g.status, dead)) break;
        tc_fence_after();
        const int kn = (min(XG_BK, kend - kbeg - XG_BK * i) + 15) / 16;
        const uint32_t p0 = tmem + P0 + (c & 1) * 128, p1 = tmem + P1;
        const uint32_t first0 = i % XG_CHUNK == 0, first1 = first0 && c % XG_P1_CHUNKS == 0;
#pragma unroll
        for (int k = 0; k < XG_BK / 16; ++k) {
          if (k >= kn) break;
          const uint32_t a = tmem + TA + (i & 1) * XG_A_STEP + k * 24;
          const uint32_t b = b0 + (i & 1) * (SM::B_STEP >> 4) + 128 * k;
          const uint64_t bh = xg_desc(b, true), bm = xg_desc(b + BP, true), bl = xg_desc(b + 2 * BP, true);
          umma_f16_tmem_a(p1, a, bl, id, !(first1 && k == 0));
          umma_f16_tmem_a(p1, a + 8, bm, id, 1);
          umma_f16_tmem_a(p1, a + 16, bh, id, 1);
          umma_f16_tmem_a(p1, a, bm, id, 1);
          umma_f16_tmem_a(p1, a + 8, bh, id, 1);
          umma_f16_tmem_a(p0, a, bh, id, !(first0 && k == 0));
        }
        umma_commit(&done[i & 1]);
        if (i % XG_CHUNK == XG_CHUNK - 1 || i == steps - 1) umma_commit(&acc_full[c & 1]);
      }
    }
    __syncwarp();
  } else {
    // warp: tokens 8 grp ... of a step, columns 32 q ... of A and of B
    const int q = warp & 3, grp = warp >> 2;
    const size_t lbase = (size_t)h * d.N * d.k;
    const bool vdy = MODE != X_DWO || g.vec_dy != 0;
    const bool arows = m0 + q * 32 < d.M, bcols = q * 32 < ncols;   // (whole warps: what lies past the tile is left as it is)
    // copies: lane -> 16-byte chunk lane & 7 of tokens lane >> 3 and 4 + (lane >> 3)
    // (columns past the operands' widths end in accumulators nobody reads: any address inside the row will do)
    const int acol = min(m0 + q * 32 + (lane & 7) * 4, d.M - 4);
    const int bcol = min(n0 + q * 32 + (lane & 7) * 4, (gates ? g.ldz : d.D) - 4);
    const float* asrc = (MODE == X_DWO ? g.dy : g.x) + acol;
    const float* bsrc = (MODE == X_DWO ? g.ahat + h * d.D : MODE == X_DWV ? g.dv + h * d.D : gates ? g.dz : (which ? g.dk : g.dq) + h * d.D) + bcol;
    const size_t bld = gates ? g.ldz : HD;
    const uint32_t raw0 = sbase + SM::RAW_OFF + warp * 1024;
    const uint32_t ca = (lane >> 3) * 128 + (lane & 7) * 16;
    int ta[2] = {0, 0}, tn[2] = {0, 0};                    // tokens of the next step and of the one behind it: entry -> row is two trips to L2
    float ga = 0.f, gn = 0.f;                              // lane -> gate of token lane & 7
    auto entries = [&](int i) {
      const int p0 = kbeg + i * XG_BK + 8 * grp;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int pa = p0 + (lane >> 3) + 4 * u;
        if (!LIST) tn[u] = min(pa, d.N - 1);
        else if (pa < kend) tn[u] = xg_token(g, lbase + pa);
      }
      if (LIST && p0 + (lane & 7) < kend) gn = __ldg(g.lgate + lbase + p0 + (lane & 7));
    };
    float* const gring = reinterpret_cast<float*>(sgen + SM::GATE_OFF) + warp * 8;   // of the steps on their way, + 128 a slot
    auto load = [&](int i, int slot) {                     // step i on its way; the entries of step i + 2 behind it
      const uint32_t raw = raw0 + slot * SM::RAW;
      const int p0 = kbeg + i * XG_BK + 8 * grp;
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const bool live = p0 + (lane >> 3) + 4 * u < kend;
        if (arows) fetch4(raw + ca + u * 512, asrc + (size_t)ta[u] * d.M, vdy, live);
        if (bcols) cp_async_16(raw + SM::RAW_A + (ca ^ (u << 4)) + u * 512, bsrc + (size_t)ta[u] * bld, live ? 16 : 0);   // (chunk c of token t at c ^ (t >> 2))
      }
      if (LIST && lane < 8) gring[slot * 128 + lane] = ga;
      ta[0] = tn[0]; ta[1] = tn[1]; ga = gn;
      if (i + 2 < steps) entries(i + 2);
    };
    // B: lane -> token bt, columns 8 (lane & 3) ... (the two tokens of a phase differ in bit 2: different banks both ways)
    const int bt = ((lane >> 2) & 1) * 4 + (lane >> 3);
    const uint32_t braw = bt * 128, bx = (uint32_t)(bt >> 2);
    const uint32_t boff = (q >> 1) * SM::B_HALF + (8 * grp + bt) * 128 + ((((q & 1) * 4 + (lane & 3)) ^ bt) << 4);
    const uint32_t tlane = (uint32_t)(q * 32) << 16;
    float acc[COLS];
#pragma unroll
    for (int i = 0; i < COLS; ++i) acc[i] = 0.f;
    const bool mine = grp * COLS < ncols;                  // (whole warps; results: rows 32 q ..., columns 32 grp ...)
    auto promote = [&](int c) {
      if (!mbar_wait(&acc_full[c & 1], (c >> 1) & 1, g.status, dead)) return;
      tc_fence_after();
      const bool p1 = (c + 1) % XG_P1_CHUNKS == 0 || c == nchunk - 1;
      if (mine) {
        tmem_add(tmem + tlane + P0 + (c & 1) * 128 + grp * COLS, acc);
        if (p1) tmem_add(tmem + tlane + P1 + grp * COLS, acc);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&acc_empty[c & 1]);
        if (p1) mbar_arrive(p1_empty);
      }
    };
    if (steps > 0) entries(0);
    ta[0] = tn[0]; ta[1] = tn[1]; ga = gn;
    if (steps > 1) entries(1);
#pragma unroll
    for (int u = 0; u < SM::NR; ++u) {
      if (u < steps) load(u, u);
      cp_async_commit();
    }
    int promoted = 0;
    for (int i0 = 0; i0 < steps && !dead; i0 += SM::NR) {
#pragma unroll
      for (int u = 0; u < SM::NR; ++u) {
        const int i = i0 + u;
        if (i >= steps || dead) break;
        cp_async_wait<SM::NR - 1>();
        __syncwarp();
        const unsigned char* raw = sgen + SM::RAW_OFF + u * SM::RAW + warp * 1024;
        uint32_t ah[4], am[4], al[4], bh[4], bm[4], bl[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          float v0 = *reinterpret_cast<const float*>(raw + 2 * t * 128 + lane * 4), v1 = *reinterpret_cast<const float*>(raw + (2 * t + 1) * 128 + lane * 4);
          if (LIST) { const float2 g2 = *reinterpret_cast<const float2*>(gring + u * 128 + 2 * t); v0 *= g2.x; v1 *= g2.y; }
          split_bf16x3(v0, v1, ah[t], am[t], al[t]);
        }
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const float4 v = *reinterpret_cast<const float4*>(raw + SM::RAW_A + braw + (((2 * (lane & 3) + c) ^ bx) << 4));
          split_bf16x3(v.x, v.y, bh[2 * c], bm[2 * c], bl[2 * c]);
          split_bf16x3(v.z, v.w, bh[2 * c + 1], bm[2 * c + 1], bl[2 * c + 1]);
        }
        __syncwarp();
        if (i + SM::NR < steps) load(i + SM::NR, u);
        cp_async_commit();
        if (i >= 2 && !mbar_wait(&done[i & 1], ((i >> 1) - 1) & 1, g.status, dead)) break;
        tc_fence_after();
        const uint32_t tc = tmem + tlane + TA + (i & 1) * XG_A_STEP + (grp >> 1) * 24 + (grp & 1) * 4;
        tmem_st4(tc, ah);
        tmem_st4(tc + 8, am);
        tmem_st4(tc + 16, al);
        unsigned char* at = sgen + (i & 1) * SM::B_STEP + boff;
        *reinterpret_cast<uint4*>(at) = make_uint4(bh[0], bh[1], bh[2], bh[3]);
        *reinterpret_cast<uint4*>(at + SM::B_PLANE) = make_uint4(bm[0], bm[1], bm[2], bm[3]);
        *reinterpret_cast<uint4*>(at + 2 * SM::B_PLANE) = make_uint4(bl[0], bl[1], bl[2], bl[3]);
        fence_proxy_async_smem();
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&full[i & 1]);
        // a chunk is read once two steps of the next one are written
        if (i % XG_CHUNK == 1 && i > XG_CHUNK) promote(promoted++);
      }
    }
    cp_async_wait<0>();
    for (; promoted < nchunk && !dead; ++promoted) promote(promoted);
    const int r = q * 32 + lane, c0 = grp * COLS;
    const int valid = min(COLS, ncols - c0);
    if (r < nrows && valid > 0 && !dead) {
      const int m = m0 + r;
      if (MODE == X_DWO || gates) {
        // columns of the tile are rows of the result, or far apart in it: one value per lane, lanes along m
#pragma unroll
        for (int i = 0; i < COLS; ++i)
          if (i < valid) {
            const int gc = n0 + c0 + i;
            float* o;
            if (MODE == X_DWO) o = g.dWo + ((size_t)(h * d.E + e) * d.Dt + gc) * d.M + m;                 // dWo [(h*E + e)*Dt + dd][m]
            else o = (gc >= d.H * d.E ? g.dWd : g.dWs) + ((size_t)((gc / d.E) % d.H) * d.M + m) * d.E + gc % d.E;
            if (g.ksplit > 1) atomicAdd(o, acc[i]);
            else *o = acc[i];
          }
      } else {
        // dWv [(h*E + e)*M + m][dd < Dt]; dWq, dWk [h*M + m][dd < Dt]
        float* o = (MODE == X_DWV ? g.dWv + ((size_t)(h * d.E + e) * d.M + m) * d.Dt
                  : (which ? g.dWk : g.dWq) + ((size_t)h * d.M + m) * d.Dt) + n0 + c0;
        const bool vec = g.vec_out != 0 && d.Dt % 4 == 0;
#pragma unroll
        for (int i = 0; i < COLS; i += 4) {
          if (vec && i + 4 <= valid) {
            if (g.ksplit > 1) red_add_v4_f32(o + i, acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
            else *reinterpret_cast<float4*>(o + i) = make_float4(acc[i], acc[i + 1], acc[i + 2], acc[i + 3]);
          } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (i + j < valid) {
                if (g.ksplit > 1) atomicAdd(o + i + j, acc[i + j]);
                else o[i + j] = acc[i + j];
              }
          }
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

// All weight gradients in one launch: tiles of X_DWQK (the longest contractions) first.  Nothing here depends on the
// launch ahead (the rest of dx), which lets this one start once it has waited for the kernels that these contractions read
// from: the two run side by side.  The wait comes at the end, so that who waits for this kernel has waited for both.
struct XWPart { XGemmArgs g; int gx, gy, n; };
static __global__ void __launch_bounds__(XW_THREADS, 1)
sh_f32_wgrad_kernel(const __grid_constant__ XWPart pq, const __grid_constant__ XWPart pv, const __grid_constant__ XWPart po) {
  int i = blockIdx.x;
  if (i < pq.n) xw_tile<X_DWQK>(pq.g, xg_unpack(i, pq.gx, pq.gy));
  else if ((i -= pq.n) < pv.n) xw_tile<X_DWV>(pv.g, xg_unpack(i, pv.gx, pv.gy));
  else xw_tile<X_DWO>(po.g, xg_unpack(i - pv.n, po.gx, po.gy));
  pdl_wait();
  pdl_trigger();
}

}  // namespace shtc
