// Score bias of Transformer-XL's relative-position term on the tensor-core path (the positional
// encoding of the paper's main models; the decomposition is Transformer-XL's):
//   bias[b, h, i, s] = c * ( q_i . r_{p_i - s}  +  v^h . r_{p_i - s}  +  u^h . k_s ),   p_i = Tc + i, s <= p_i
// (c = log2(e)/sqrt(d_head) is already folded into the stored Q; the attention kernel adds bias to its
// S tiles, which are in the same units).  The first term is a GEMM over DISTANCES - Q[b,h] (chunk rows)
// times R16[h]^T - whose result must be shifted, row by row, from distance order to key order (the
// "relative shift" of Transformer-XL).  A warp-uniform TMEM address cannot shift per row, so the shift
// happens in shared memory: a lane holds one query row's 32 distances and puts them where its keys are, in a
// window of 64 keys of its own; 32 distances complete 32 keys of every row, with the same boundaries for all rows.
//
// The result is laid out for its reader, a thread of the attention kernel per query row that takes 8 keys (16 bytes) at
// a time: [b, h, 128-row tile, key / 8, row, 8 keys], so that a warp's 16-byte pieces are 512 contiguous bytes, here and
// there.  (In row-major order the writer stored 2 bytes per lane, 32 keys of a row at a time: 41 us at 8192 chunk tokens
// of 1024 keys, bound by issue; and the reader's lanes met 32 different lines per load.)
//
// CTA = (batch*head, 128-query tile of the chunk): Q tile loaded once, 64-distance tiles of R16[h]
// streamed through a ring of 2 (only distances up to the tile's largest query position exist), UMMA
// N = 64 into two alternating TMEM buffers, four epilogue warps (a TMEM lane quarter each).  Sized (100 KB of
// shared memory) for two CTAs per SM, which fill each other's latencies.
// Warp roles (192 threads): warp 0 = TMA producer, warp 1 = TMEM owner + UMMA issuer, warps 2..5 = epilogue.
#pragma once
#include "sh_tc_prims.cuh"

namespace shtc {

struct TcXlBiasArgs {
  ShDims d;
  const float* vr;       // [H, T]     c * v^h . r_dist
  const float* uk;       // [B, H, T]  c * u^h . k_s
  __half* bias;          // [B, H, (T - Tc) / 128, T / 8, 128, 8]
  int* status;
};

template <int D>
struct XlBiasSmem {
  static constexpr int T_BYTES = 128 * D * 2;            // the query tile
  static constexpr int R_BYTES = 64 * D * 2;             // one tile of 64 distances
  static constexpr int RST = 2;
  static constexpr int Q_OFF = 0;
  static constexpr int R_OFF = T_BYTES;
  static constexpr int STG_OFF = R_OFF + RST * R_BYTES;
  static constexpr int WIN_LD = 68;                       // a row's window of 64 keys: lanes' 4-byte stores (bank 69 row - column) and 16-byte loads are conflict-free
  static constexpr int STG_WARP = (32 * WIN_LD + 64 + 64) * 4;   // windows, v.r of 64 distances, u.k of 64 keys
  static constexpr int BAR_OFF = STG_OFF + 4 * STG_WARP;
  static constexpr int TOTAL = BAR_OFF + 256 + 1024;
};

template <int D>
__global__ void __launch_bounds__(192, 2)
sh_tc_xlbias_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapR, TcXlBiasArgs g) {
  using SM = XlBiasSmem<D>;
  constexpr int DB = D / 64, RST = SM::RST;
  constexpr uint32_t BLK = 128 * 128;                    // a 64-column block of the query tile
  constexpr uint32_t RBLK = 64 * 128;                    // a 64-column block of a distance tile
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* sgen = smem_raw + (sbase - smem_u32(smem_raw));
  uint64_t* bars = (uint64_t*)(sgen + SM::BAR_OFF);
  uint64_t* q_full = bars;
  uint64_t* r_full = bars + 1;       // [RST]
  uint64_t* r_empty = bars + 5;      // [RST]
  uint64_t* acc_full = bars + 9;     // [2]
  uint64_t* acc_empty = bars + 11;   // [2] four arrivals (epilogue warps)
  uint32_t* tmem_slot = (uint32_t*)(bars + 13);

  const ShDims& d = g.d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Tq = d.T - d.Tc, tiles_q = Tq / 128;
  const int nbh = d.B * d.H;
  const int bh = blockIdx.x % nbh, it = tiles_q - 1 - blockIdx.x / nbh, h = bh % d.H;   // longest tiles (most distances) first
  const int ncol = 2 * (d.Tc / 128 + it + 1);            // 64-distance tiles that hold a visible distance for some row of this tile
  bool dead = false;

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < RST; ++s) { mbar_init(&r_full[s], 1); mbar_init(&r_empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&acc_full[b], 1); mbar_init(&acc_empty[b], 4); }
    fence_barrier_init();
    tma_prefetch_desc(&mapQ); tma_prefetch_desc(&mapR);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, 128); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();
  pdl_wait();                                            // Q, K (hence u.k) of this pass are complete

  if (warp == 0) {
    if (lane == 0) {
      mbar_expect_tx(q_full, SM::T_BYTES);
#pragma unroll
      for (int c = 0; c < DB; ++c) tma_load_2d(sbase + SM::Q_OFF + c * BLK, &mapQ, q_full, c * 64, bh * d.T + d.Tc + it * 128);
      for (int ct = 0; ct < ncol; ++ct) {
        const int s = ct % RST;
        if (!mbar_wait(&r_empty[s], ((ct / RST) & 1) ^ 1, g.status, dead)) break;
        mbar_expect_tx(&r_full[s], SM::R_BYTES);
#pragma unroll
        for (int c = 0; c < DB; ++c) tma_load_2d(sbase + SM::R_OFF + s * SM::R_BYTES + c * RBLK, &mapR, &r_full[s], c * 64, h * d.T + ct * 64);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = make_idesc_f16(128, 64, 0, 0, 0);
      const uint32_t q_lo = desc_lo_k(sbase + SM::Q_OFF), r_lo0 = desc_lo_k(sbase + SM::R_OFF);
      if (mbar_wait(q_full, 0, g.status, dead)) {
        for (int ct = 0; ct < ncol; ++ct) {
          const int s = ct % RST, b = ct & 1;
          if (!mbar_wait(&r_full[s], (ct / RST) & 1, g.status, dead)) break;
          if (!mbar_wait(&acc_empty[b], ((ct >> 1) & 1) ^ 1, g.status, dead)) break;
          tc_fence_after();
          const uint32_t r_lo = r_lo0 + s * (SM::R_BYTES >> 4);
#pragma unroll
          for (int k = 0; k < D / 16; ++k)
            umma_f16(tmem + b * 64, desc_pack(q_lo + (k / 4) * (BLK >> 4) + 2 * (k % 4)), desc_pack(r_lo + (k / 4) * (RBLK >> 4) + 2 * (k % 4)), idesc, k != 0);
          umma_commit(&r_empty[s]);
          umma_commit(&acc_full[b]);
        }
      }
    }
  } else {
    // ---- epilogue: warp = 32 query rows (TMEM lane quarter), thread = query row ----
    const int q = warp & 3;
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    float* win = reinterpret_cast<float*>(sgen + SM::STG_OFF + (warp - 2) * SM::STG_WARP);
    float* svr = win + 32 * SM::WIN_LD;
    float* suk = svr + 64;
    float* wrow = win + lane * SM::WIN_LD;
    const int p0 = d.Tc + it * 128 + q * 32;               // position of this warp's first row
    uint4* out = reinterpret_cast<uint4*>(g.bias) + ((size_t)bh * tiles_q + it) * (d.T / 8) * 128 + q * 32 + lane;   // + 128 per 8 keys
    const float* vr = g.vr + (size_t)h * d.T;
    const float* ukr = g.uk + (size_t)bh * d.T;
    for (int ct = 0; ct < ncol; ++ct) {
      const int b = ct & 1;
      // v.r of the tile's distances and u.k of the keys it completes: p0 - 64 ct - 32 ... + 63
      const int kb = p0 - ct * 64 - 32;
      reinterpret_cast<float2*>(svr)[lane] = __ldg(reinterpret_cast<const float2*>(vr + ct * 64) + lane);
      suk[lane] = kb + lane >= 0 ? __ldg(ukr + kb + lane) : 0.f;
      suk[32 + lane] = kb + 32 + lane >= 0 ? __ldg(ukr + kb + 32 + lane) : 0.f;
      __syncwarp();
      if (!mbar_wait(&acc_full[b], (ct >> 1) & 1, g.status, dead)) break;
      tc_fence_after();
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {
        // 32 distances from dist0 on: keys base + lane - c.  Those from base on (c <= lane) complete the 32 keys from base
        // on - the distances before left the rest -, those below start the 32 before; base is a multiple of 32
        const int base = p0 - ct * 64 - hh * 32;
        float* hi = wrow + (base & 32) + lane;
        float* lo = wrow + ((base & 32) ^ 32) + 32 + lane;
        uint32_t v[32];
        tmem_ld32(tmem + lane_off + b * 64 + hh * 32, v);
        tmem_ld_wait();
        if (hh == 1) {
          tc_fence_before();                               // this warp's share of the accumulator is in registers
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_empty[b]);
        }
#pragma unroll
        for (int c = 0; c < 32; c += 4) {
          const float4 r4 = *reinterpret_cast<const float4*>(svr + hh * 32 + c);
          const float2 a = __fadd2_rn(make_float2(__uint_as_float(v[c]), __uint_as_float(v[c + 1])), make_float2(r4.x, r4.y));
          const float2 e = __fadd2_rn(make_float2(__uint_as_float(v[c + 2]), __uint_as_float(v[c + 3])), make_float2(r4.z, r4.w));
          (lane >= c ? hi : lo)[-c] = a.x;
          (lane >= c + 1 ? hi : lo)[-c - 1] = a.y;
          (lane >= c + 2 ? hi : lo)[-c - 2] = e.x;
          (lane >= c + 3 ? hi : lo)[-c - 3] = e.y;
        }
        // (a row's own window: no other lane is involved)
        if (base >= 0) {
          const float* full = wrow + (base & 32);
          const float* uk = suk + 32 - hh * 32;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 w0 = *reinterpret_cast<const float4*>(full + 8 * i), w1 = *reinterpret_cast<const float4*>(full + 8 * i + 4);
            const float4 u0 = *reinterpret_cast<const float4*>(uk + 8 * i), u1 = *reinterpret_cast<const float4*>(uk + 8 * i + 4);
            __half2 o[4];
            o[0] = __float22half2_rn(__fadd2_rn(make_float2(w0.x, w0.y), make_float2(u0.x, u0.y)));
            o[1] = __float22half2_rn(__fadd2_rn(make_float2(w0.z, w0.w), make_float2(u0.z, u0.w)));
            o[2] = __float22half2_rn(__fadd2_rn(make_float2(w1.x, w1.y), make_float2(u1.x, u1.y)));
            o[3] = __float22half2_rn(__fadd2_rn(make_float2(w1.z, w1.w), make_float2(u1.z, u1.w)));
            uint4 w;
            w.x = *reinterpret_cast<uint32_t*>(&o[0]); w.y = *reinterpret_cast<uint32_t*>(&o[1]);
            w.z = *reinterpret_cast<uint32_t*>(&o[2]); w.w = *reinterpret_cast<uint32_t*>(&o[3]);
            out[(size_t)(base / 8 + i) * 128] = w;
          }
        }
      }
      __syncwarp();                                        // (v.r and u.k of the next tile)
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 128);
  }
}

}  // namespace shtc
