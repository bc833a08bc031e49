// Causal softmax attention for d_head above 128 (stored as 256 columns), one 128-query tile per CTA.
//
// The 512 tensor-memory columns hold O (up to 256), two S buffers of 64 keys and two P buffers, so one
// query tile per CTA is all that fits; keys go in steps of 64 (K and V stages of 64 rows, two each,
// beside the query tile: up to 192 KB).  Probabilities are P_hi + P_lo, two fp16 values,
// each multiplied with V (two UMMAs per 16 keys) - such a layer's probabilities were fp32 on the CUDA
// cores before, and the second product costs nothing here: the softmax of a step, not the tensor pipe,
// bounds the loop.  They are scaled by 2^7 (the sum they are divided by is as well): with the row maximum
// behind by up to 2^8 that fills fp16's range, 22 bits for probabilities of 2^-9 of the largest and more, and
// an error of at most 2^-32 of the largest below (unscaled: 2^-25).  Measured at 16 x 512 tokens, 2 heads of 132: 18 us (one warp per query row on the CUDA
// cores: 4490); its floor is the softmax, one exponential per visible (query, key).
//
// S of step j + 1 is issued before the product of step j, so it runs under the softmax of step j.  Its
// buffer was read by the softmax of step j - 1 (whose P the issuer has waited for); a P buffer is
// rewritten at step j + 2, after S of that step, which the tensor pipe finishes behind the product of j.
//
// Warp roles (192 threads): warp 0 = TMA producer, warp 1 = TMEM owner + UMMA issuer, warps 2..5 =
// softmax (thread = query row).  Only the 64-column blocks and 16-column slices that d_head reaches
// are loaded and multiplied.
#pragma once
#include "sh_tc_attn2.cuh"

namespace shtc {

struct AttnWSmem {
  static constexpr int Q_BLK = 128 * 128, KV_BLK = 64 * 128;        // 64 columns of the query tile / of a K or V stage
  static constexpr int Q_OFF = 0, K_OFF = 4 * Q_BLK, V_OFF = K_OFF + 2 * 4 * KV_BLK;
  static constexpr int BAR_OFF = V_OFF + 2 * 4 * KV_BLK;
  static constexpr int TOTAL = BAR_OFF + 256 + 1024;
};

// One row of Ahat by plain sums over the keys it sees.  The tensor pipe multiplies the masked probabilities of a step,
// zeros, with value rows the query does not see; one of them past fp16's range makes the product NaN.  Rows
// whose result is not finite although their scores are come here.
static __device__ __noinline__ void attnw_row(const ShDims& d, const __half* q, const __half* k, const __half* v, int last, __half* dst) {
  float o[256];
  for (int c = 0; c < d.Dt; ++c) o[c] = 0.f;
  float m = -INFINITY, l = 0.f;
  for (int j = 0; j <= last; ++j) {
    const __half *kr = k + (size_t)j * d.D, *vr = v + (size_t)j * d.D;
    float s = 0.f;
    for (int c = 0; c < d.Dt; ++c) s = fmaf(__half2float(q[c]), __half2float(kr[c]), s);
    if (s > m) {
      const float alpha = exp2f(m - s);
      for (int c = 0; c < d.Dt; ++c) o[c] *= alpha;
      l *= alpha; m = s;
    }
    const float p = exp2f(s - m);
    l += p;
    for (int c = 0; c < d.Dt; ++c) o[c] = fmaf(p, __half2float(vr[c]), o[c]);
  }
  for (int c = 0; c < d.Dt; ++c) dst[c] = __float2half_rn(o[c] / l);
}

static __global__ void __launch_bounds__(192, 1)
sh_tc_attention_wide_kernel(const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
                            const __grid_constant__ CUtensorMap mapV, TcAttnArgs g) {
  using SM = AttnWSmem;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* sgen = smem_raw + (sbase - smem_u32(smem_raw));
  uint64_t* bars = (uint64_t*)(sgen + SM::BAR_OFF);
  uint64_t* q_full = bars;
  uint64_t* k_full = bars + 1;    // [2]
  uint64_t* k_empty = bars + 3;   // [2]
  uint64_t* v_full = bars + 5;    // [2]
  uint64_t* v_empty = bars + 7;   // [2]
  uint64_t* s_full = bars + 9;    // [2]
  uint64_t* p_full = bars + 11;   // [2]
  uint64_t* pv_done = bars + 13;  // [2] the product of step j has completed (barrier j & 1)
  uint64_t* o_done = bars + 15;   // the last product has completed
  uint32_t* tmem_slot = (uint32_t*)(bars + 16);

  const ShDims& d = g.d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int BH = d.B * d.H;
  const int bh = blockIdx.x % BH;
  const int ntile = (d.T + 127) / 128;
  const int qrow = (ntile - 1 - (int)(blockIdx.x / BH)) * 128;      // the longest rows first
  const int nkeys = d.causal ? min(d.T, qrow + 128) : d.T;
  const int nsteps = (nkeys + 63) / 64;
  const int db = (d.Dt + 63) / 64, kd = (d.Dt + 15) / 16;           // 64-column blocks, 16-column slices
  bool dead = false;

  if (threadIdx.x == 0) {
    mbar_init(q_full, 1); mbar_init(o_done, 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&k_full[i], 1); mbar_init(&k_empty[i], 1); mbar_init(&v_full[i], 1); mbar_init(&v_empty[i], 1);
      mbar_init(&s_full[i], 1); mbar_init(&p_full[i], 4); mbar_init(&pv_done[i], 1);
    }
    fence_barrier_init();
    tma_prefetch_desc(&mapQ); tma_prefetch_desc(&mapK); tma_prefetch_desc(&mapV);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;                        // O: columns 0..255; S: 256, 320; P (hi 32 columns, lo 32): 384, 448
  if (threadIdx.x == 0) sh_stamp_resident(d.stamps, SH_K_ATTN);
  pdl_wait();
  pdl_trigger();                                           // (behind the wait: what the next kernel does ahead of its own then sees every earlier kernel complete)
  if (threadIdx.x == 0) sh_stamp_start(d.stamps, SH_K_ATTN);

  if (warp == 0) {
    if (lane == 0) {
      mbar_expect_tx(q_full, db * SM::Q_BLK);
      for (int c = 0; c < db; ++c) tma_load_3d(sbase + SM::Q_OFF + c * SM::Q_BLK, &mapQ, q_full, c * 64, qrow, bh);
      for (int j = 0; j < nsteps; ++j) {
        const int s = j & 1;
        const uint32_t par = ((j >> 1) & 1) ^ 1;
        if (!mbar_wait(&k_empty[s], par, g.status, dead)) break;
        mbar_expect_tx(&k_full[s], db * SM::KV_BLK);
        for (int c = 0; c < db; ++c) tma_load_3d(sbase + SM::K_OFF + (4 * s + c) * SM::KV_BLK, &mapK, &k_full[s], c * 64, j * 64, bh);
        if (!mbar_wait(&v_empty[s], par, g.status, dead)) break;
        mbar_expect_tx(&v_full[s], db * SM::KV_BLK);
        for (int c = 0; c < db; ++c) tma_load_3d(sbase + SM::V_OFF + (4 * s + c) * SM::KV_BLK, &mapV, &v_full[s], c * 64, j * 64, bh);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc_s = make_idesc_f16(128, 64, 0, 0, 0);
      const uint32_t idesc_pv = make_idesc_f16(128, kd * 16, 0, 0, 1);
      const uint32_t q_lo0 = desc_lo_k(sbase + SM::Q_OFF), k_lo0 = desc_lo_k(sbase + SM::K_OFF), v_lo0 = desc_lo_mn(sbase + SM::V_OFF, SM::KV_BLK);
      auto issue_s = [&](int j) -> bool {
        const int s = j & 1;
        if (!mbar_wait(&k_full[s], (j >> 1) & 1, g.status, dead)) return false;
        tc_fence_after();
        for (int k = 0; k < kd; ++k)
          umma_f16(tmem + 256 + s * 64, desc_pack(q_lo0 + (k >> 2) * (SM::Q_BLK >> 4) + 2 * (k & 3)),
                   desc_pack(k_lo0 + (4 * s + (k >> 2)) * (SM::KV_BLK >> 4) + 2 * (k & 3)), idesc_s, k != 0);
        umma_commit(&s_full[s]);
        umma_commit(&k_empty[s]);
        return true;
      };
      bool ok = mbar_wait(q_full, 0, g.status, dead) && issue_s(0);
      for (int j = 0; ok && j < nsteps; ++j) {
        const int s = j & 1;
        if (j + 1 < nsteps && !issue_s(j + 1)) break;
        if (!mbar_wait(&v_full[s], (j >> 1) & 1, g.status, dead)) break;
        if (!mbar_wait(&p_full[s], (j >> 1) & 1, g.status, dead)) break;
        tc_fence_after();
        const uint32_t v_lo = v_lo0 + 4 * s * (SM::KV_BLK >> 4);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          umma_f16_tmem_a(tmem, tmem + 384 + s * 64 + 8 * k, desc_pack(v_lo + k * (2048 >> 4)), idesc_pv, (j | k) != 0);
          umma_f16_tmem_a(tmem, tmem + 384 + s * 64 + 32 + 8 * k, desc_pack(v_lo + k * (2048 >> 4)), idesc_pv, 1);
        }
        umma_commit(&v_empty[s]);
        umma_commit(&pv_done[s]);
        if (j == nsteps - 1) umma_commit(o_done);
      }
    }
  } else {
    const int q = warp & 3, r = q * 32 + lane;
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int j = 0; j < nsteps; ++j) {
      const int s = j & 1;
      if (!mbar_wait(&s_full[s], (j >> 1) & 1, g.status, dead)) { ok = false; break; }
      tc_fence_after();
      uint32_t sv[64];
      tmem_ld32(tmem + 256 + s * 64 + lane_off, *reinterpret_cast<uint32_t(*)[32]>(&sv[0]));
      tmem_ld32(tmem + 256 + s * 64 + lane_off + 32, *reinterpret_cast<uint32_t(*)[32]>(&sv[32]));
      tmem_ld_wait();
      const int cmax = (d.causal ? min(qrow + r, d.T - 1) : d.T - 1) - j * 64;   // last visible key of the step
      if (cmax < 63) {
#pragma unroll
        for (int c = 0; c < 64; ++c)
          if (c > cmax) sv[c] = 0xff800000u;                 // -inf
      }
      float mx4[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int c = 0; c < 64; ++c) mx4[c & 3] = fmaxf(mx4[c & 3], __uint_as_float(sv[c]));
      const float mx = fmaxf(fmaxf(mx4[0], mx4[1]), fmaxf(mx4[2], mx4[3]));
      // (the maximum is raised only when it is passed by more than 2^8: see sh_tc_attention3_kernel)
      float alpha = 1.f;
      bool raise = false;
      if (mx > m + 8.f) { alpha = fast_exp2(m - mx); m = mx; raise = j > 0; }
      const float mp = m - 7.f;                              // (the probabilities' scale of 2^7)
      float sum4[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t hi[32], lo[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        const float p0 = fast_exp2(__uint_as_float(sv[2 * c]) - mp), p1 = fast_exp2(__uint_as_float(sv[2 * c + 1]) - mp);
        sum4[c & 3] += p0 + p1;
        const __half2 h = __floats2half2_rn(p0, p1);
        const float2 hf = __half22float2(h);
        const __half2 w = __floats2half2_rn(p0 - hf.x, p1 - hf.y);
        hi[c] = *reinterpret_cast<const uint32_t*>(&h);
        lo[c] = *reinterpret_cast<const uint32_t*>(&w);
      }
      l = l * alpha + ((sum4[0] + sum4[1]) + (sum4[2] + sum4[3]));
      if (j > 0 && __any_sync(0xffffffffu, raise)) {         // rescale this warp's rows of O: every earlier product has to be in
        if (!mbar_wait(&pv_done[s ^ 1], ((j - 1) >> 1) & 1, g.status, dead)) { ok = false; break; }
        tc_fence_after();
        for (int c = 0; c < (kd + 1) / 2; ++c) {
          uint32_t ov[32];
          tmem_ld32(tmem + lane_off + c * 32, ov);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 32; ++i) ov[i] = __float_as_uint(__uint_as_float(ov[i]) * alpha);
          tmem_st32(tmem + lane_off + c * 32, ov);
        }
      }
      tmem_st32(tmem + 384 + s * 64 + lane_off, hi);
      tmem_st32(tmem + 384 + s * 64 + 32 + lane_off, lo);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_full[s]);
    }
    if (ok && mbar_wait(o_done, 0, g.status, dead)) {
      tc_fence_after();
      const int tq = qrow + r;
      const float inv = 1.f / l;
      const int bb = bh / d.H, hh = bh % d.H;
      __half* dst = g.ahat + (((size_t)bb * d.T + tq) * d.H + hh) * d.D;
      float nan4[4] = {0.f, 0.f, 0.f, 0.f};                  // (NaN once a value of the row is not finite)
      for (int c = 0; c < db * 2; ++c) {                     // (up to the 64-column block the output projection loads: zeros behind d_head)
        uint32_t ov[32];
        tmem_ld32(tmem + lane_off + c * 32, ov);
        tmem_ld_wait();
        if (tq < d.T) {
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (2 * c + (i >> 4) < kd) nan4[i & 3] = fmaf(__uint_as_float(ov[i]), 0.f, nan4[i & 3]);   // (the slices that were multiplied)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            uint32_t w[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int col = c * 32 + 8 * i + 2 * u;
              const __half2 h = __floats2half2_rn(col < d.Dt ? __uint_as_float(ov[8 * i + 2 * u]) * inv : 0.f,
                                                  col + 1 < d.Dt ? __uint_as_float(ov[8 * i + 2 * u + 1]) * inv : 0.f);
              w[u] = *reinterpret_cast<const uint32_t*>(&h);
            }
            *reinterpret_cast<uint4*>(dst + c * 32 + 8 * i) = make_uint4(w[0], w[1], w[2], w[3]);
          }
        }
      }
      const float nan = (nan4[0] + nan4[1]) + (nan4[2] + nan4[3]);
      if (tq < d.T && nan != nan && l < INFINITY) {          // (l: the scores' part, not NaN either)
        const size_t row0 = (size_t)bh * d.T;
        attnw_row(d, g.q + (row0 + tq) * d.D, g.k + row0 * d.D, g.v + row0 * d.D, d.causal ? tq : d.T - 1, dst);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) sh_stamp_end(d.stamps, SH_K_ATTN);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace shtc
