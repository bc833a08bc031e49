// Attention of the fp32 configuration, forward, on the tensor cores: d_head up to 128.
//
// The products Q K^T and P V in split bf16 (sh_f32_gemm.cuh: six products of bf16 planes are one of fp32), softmax in
// fp32 as on the CUDA cores.  A layer's share of attention is small (0.5 of the 7 GFLOP of a 262M-scale forward pass) and
// sequences are a few hundred tokens, so what counts is the longest chain of key tiles, not the work: on the CUDA cores
// a block of 32 queries worked off 512 keys in 38 us with most SMs done long before (2 x 4 heads of 112; here 25).  Here a unit is 128 queries of one
// (sequence, head) and a PART of their keys - as few 64-key tiles, two at least, as keep the number of units at or below that of
// the SMs and their partial results in the scratch -, and whoever ends last among a query tile's parts joins them (partial sums, maxima and
// normalisers; the scratch is the backward pass's, which holds nothing then).
//
// Per key tile: workers split K's rows into planes (shared memory, 128-byte swizzle; rows past the sequence are zeros),
// S = Q K^T into P0 P1 P2 (and P3 for the positions from 64 on: as in sh_f32_gemm_d_kernel), two threads per query row
// take 32 keys each, P's planes go over S in tensor memory, O_part = P V (V's rows as MN-major planes), which the workers
// read back and add to the running sum in registers.  The next K is split under P V, V under S.
//
// What is not finite: a tile with such a V is added up on the CUDA cores, key by key, leaving out what a row does not see
// (0 times infinity), so that it stays with the rows that see it.  A row that finds a NaN among a tile's scores takes them again there:
// a score of minus infinity is one (a key of weight zero), not the NaN that its split products add up to.
//
// Warp roles (288 threads): warps 0..7 workers (rows 32 (w & 3) ..., keys / columns of half w >> 2), warp 8 UMMAs.  Nine
// warps leave 168 registers a thread; with 128 columns the running sums and a piece of K or V in flight spill (212 bytes stored, 332 loaded).
#pragma once
#include "sh_f32_gemm.cuh"
#include "sh_f32_attn.cuh"

namespace shtc {

struct FAttnTcArgs {
  const float *q, *k, *v;                // [B, H, T, D]
  float* ahat;                           // [N, H, D]
  float* stats;                          // [B, H, T, 2]: the row's score maximum (base 2) and 1 / normaliser, for the backward pass
  float* part;                           // per unit: sums [128, D], maxima [128], normalisers [128]
  unsigned* arrived;                     // per query tile: parts done (zero between passes)
  float4* zero; long nzero;              // the layer's output, which the next kernel adds into: this is the first kernel behind the last read of x, which may be the same buffer
  ShDims d;
  int per;                               // 64-key tiles of a part, at most
  int* status;
};

template <int D>
struct FAttnTcSmem {
  static constexpr int NBK = D > 64 ? 2 : 1;                 // 64-column blocks of a row
  static constexpr int Q_PLANE = NBK * 128 * 128, V_PLANE = NBK * 64 * 128, K_BLK = 3 * 64 * 128;
  static constexpr int Q_OFF = 0, K_OFF = 3 * Q_PLANE, V_OFF = K_OFF + NBK * K_BLK;
  static constexpr int MAX_OFF = V_OFF + 3 * V_PLANE;        // [2][128] floats: exchange between a row's two threads
  static constexpr int BAR_OFF = MAX_OFF + 1024;
  static constexpr int TOTAL = BAR_OFF + 256 + 1024;
  static_assert(128 * (D + 4) * 4 <= 3 * Q_PLANE + NBK * K_BLK, "result rows take Q's and K's place");
};

// Query tile, its part and its number of parts behind unit u of a (sequence, head): tiles with the most keys first.
struct FAttnUnit { int qt, part, parts, first; };
__host__ __device__ __forceinline__ int fattn_key_tiles(const ShDims& d, int qt) {
  const int last = d.Tc + 128 * qt + 128;
  return ((d.causal && last < d.T ? last : d.T) + 63) / 64;
}
__device__ __forceinline__ FAttnUnit fattn_unit(const ShDims& d, int per, int u) {
  FAttnUnit r;
  r.first = 0;
  for (r.qt = (d.T - d.Tc + 127) / 128 - 1; ; --r.qt) {
    r.parts = (fattn_key_tiles(d, r.qt) + per - 1) / per;
    if (u < r.first + r.parts || r.qt == 0) break;
    r.first += r.parts;
  }
  r.part = u - r.first;
  return r;
}

// The larger one, NaN where one of them is.
__device__ __forceinline__ float fmax_nan(float a, float b) {
  float m;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
  return m;
}

// acc += 16 tensor-memory columns at a time (the running sums leave no registers for more).
template <int N>
__device__ __forceinline__ void tmem_add16(uint32_t taddr, float (&acc)[N]) {
#pragma unroll
  for (int c = 0; c < N; c += 16) {
    uint32_t u[16];
    tmem_ld16(taddr + c, u);
    tmem_ld_wait();
#pragma unroll
    for (int i = 0; i < 16; ++i) acc[c + i] += __uint_as_float(u[i]);
  }
}

// Four adjacent values as planes at byte `off` of three planes `plane` bytes apart.
__device__ __forceinline__ void fattn_put4(unsigned char* tile, uint32_t off, int plane, float4 v) {
  uint2 h, m, l;
  split_bf16x3(v.x, v.y, h.x, m.x, l.x);
  split_bf16x3(v.z, v.w, h.y, m.y, l.y);
  *reinterpret_cast<uint2*>(tile + off) = h;
  *reinterpret_cast<uint2*>(tile + off + plane) = m;
  *reinterpret_cast<uint2*>(tile + off + 2 * plane) = l;
}

template <int D>
__global__ void __launch_bounds__(288, 1)
sh_f32_attn_tc_kernel(const __grid_constant__ FAttnTcArgs g) {
  using SM = FAttnTcSmem<D>;
  constexpr int C4 = D / 4;                                // 16-byte pieces of a row
  constexpr int KV = 64 * C4 / 256;                        // pieces of a K or V tile per worker thread
  constexpr int COLS = D / 2;                              // output columns of a worker thread
  constexpr uint32_t S0 = 0, PV0 = 256, PV1 = 384;         // tensor-memory columns: S: P0 P1 P2 P3 of 64 keys; P V: hh', the others
  extern __shared__ unsigned char smem_raw[];
  const uint32_t sbase = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* sgen = smem_raw + (sbase - smem_u32(smem_raw));
  uint64_t* k_full = (uint64_t*)(sgen + SM::BAR_OFF);      // K (and Q) are in shared memory
  uint64_t* s_full = k_full + 1;                           // S is complete
  uint64_t* p_full = s_full + 1;                           // P is in tensor memory, V in shared memory
  uint64_t* o_full = p_full + 1;                           // P V is complete
  uint64_t* slow_done = o_full + 1;                        // a tile has been added up by the workers
  uint32_t* tmem_slot = (uint32_t*)(slow_done + 1);
  int* bad = (int*)(tmem_slot + 1);                        // [2] tile j's V holds a value that is not finite: bad[j & 1] == j + 1
  int* last_part = bad + 2;
  float* sx = reinterpret_cast<float*>(sgen + SM::MAX_OFF);
  const ShDims& d = g.d;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  bool dead = false;

  if (tid == 0) {
    mbar_init(k_full, 8); mbar_init(s_full, 1); mbar_init(p_full, 8); mbar_init(o_full, 1); mbar_init(slow_done, 8);
    bad[0] = bad[1] = 0;
    fence_barrier_init();
  }
  if (warp == 8) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  const int BH = d.B * d.H, bh = blockIdx.x % BH, b = bh / d.H, h = bh % d.H;
  const FAttnUnit un = fattn_unit(d, g.per, (int)(blockIdx.x / BH));
  const int q0 = d.Tc + un.qt * 128, nq = min(128, d.T - q0);
  const int kt0 = un.part * g.per, tiles = min(g.per, fattn_key_tiles(d, un.qt) - kt0);
  const int k16s = (d.Dt + 15) / 16;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();
  pdl_trigger();                                           // (behind the wait: what the next kernel reads ahead of its own is complete)

  if (warp == 8) {
    if (lane == 0) {
      const uint32_t id3 = xg_idesc(192, false), id2 = xg_idesc(128, false), id1 = xg_idesc(64, false);
      const uint32_t idv = xg_idesc(k16s * 16, true);
      const uint32_t q_lo = desc_lo_k(sbase + SM::Q_OFF), k_lo = desc_lo_k(sbase + SM::K_OFF), v_lo = desc_lo_mn(sbase + SM::V_OFF, 64 * 128);
      constexpr uint32_t QP = SM::Q_PLANE >> 4, KP = (64 * 128) >> 4, VP = SM::V_PLANE >> 4;
      int nslow = 0;
      for (int j = 0; j < tiles && !dead; ++j) {
        if (!mbar_wait(k_full, j & 1, g.status, dead)) break;
        tc_fence_after();
        for (int k = 0; k < k16s; ++k) {
          const uint32_t a = q_lo + (k >> 2) * ((128 * 128) >> 4) + 2 * (k & 3), bk = k_lo + (k >> 2) * (SM::K_BLK >> 4) + 2 * (k & 3);
          if (k < 4) umma_f16(tmem + S0, desc_pack(a), desc_pack(bk), id3, k != 0);
          else {
            umma_f16(tmem + S0 + 64, desc_pack(a), desc_pack(bk + KP), id2, 1);
            umma_f16(tmem + S0 + 192, desc_pack(a), desc_pack(bk), id1, k != 4);
          }
          umma_f16(tmem + S0 + 64, desc_pack(a + QP), desc_pack(bk), id2, 1);
          umma_f16(tmem + S0 + 128, desc_pack(a + 2 * QP), desc_pack(bk), id1, 1);
        }
        umma_commit(s_full);
        if (!mbar_wait(p_full, j & 1, g.status, dead)) break;
        tc_fence_after();
        if (*(volatile int*)&bad[j & 1] == j + 1) {        // (the workers do this tile; S of the next one comes behind them)
          mbar_arrive(o_full);
          if (!mbar_wait(slow_done, nslow++ & 1, g.status, dead)) break;
          continue;
        }
        for (int k = 0; k < 4; ++k) {
          // (P's planes lie where the two warps that wrote them had read S: 24 columns at 0, 64, 32, 96)
          const uint32_t a = tmem + S0 + (k >> 1) * 32 + (k & 1) * 64, bv = v_lo + 128 * k;
          umma_f16_tmem_a(tmem + PV1, a, desc_pack(bv + 2 * VP), idv, k != 0);
          umma_f16_tmem_a(tmem + PV1, a + 8, desc_pack(bv + VP), idv, 1);
          umma_f16_tmem_a(tmem + PV1, a + 16, desc_pack(bv), idv, 1);
          umma_f16_tmem_a(tmem + PV1, a, desc_pack(bv + VP), idv, 1);
          umma_f16_tmem_a(tmem + PV1, a + 8, desc_pack(bv), idv, 1);
          umma_f16_tmem_a(tmem + PV0, a, desc_pack(bv), idv, k != 0);
        }
        umma_commit(o_full);
      }
    }
    __syncwarp();
  } else {
    const int q = warp & 3, half = warp >> 2, r = q * 32 + lane;
    const float* Qb = g.q + ((size_t)bh * d.T + q0) * D;
    const float* Kb = g.k + (size_t)bh * d.T * D;
    const float* Vb = g.v + (size_t)bh * d.T * D;
    // piece u of this thread: row and 16-byte piece in it (a warp's are whole rows: coalesced)
    const int c4 = tid % C4, r0 = tid / C4;                // rows r0, r0 + 256 / C4, ...
    constexpr int RS = 256 / C4;
    auto fetch = [&](const float* src, int rows, float4 (&f)[KV]) {
#pragma unroll
      for (int u = 0; u < KV; ++u) {
        const int row = r0 + u * RS;
        f[u] = row < rows ? __ldg(reinterpret_cast<const float4*>(src + (size_t)row * D) + c4) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    };
    // byte offset of the piece inside a 64-column block of rows of 128 bytes (two bytes a value)
    auto piece = [&](int row) { return (uint32_t)(row * 128 + (((((c4 & 15) >> 1) ^ (row & 7)) << 4) | ((c4 & 1) << 3))); };
    float4 f[KV];
    {
      float4 fq[KV];
      fetch(Qb, nq, fq);
      fetch(Kb + (size_t)kt0 * 64 * D, d.T - kt0 * 64, f);
#pragma unroll
      for (int u = 0; u < KV; ++u) fattn_put4(sgen + SM::Q_OFF, (c4 >> 4) * (128 * 128) + piece(r0 + u * RS), SM::Q_PLANE, fq[u]);
      fetch(Qb + 64 * D, nq - 64, fq);
#pragma unroll
      for (int u = 0; u < KV; ++u) fattn_put4(sgen + SM::Q_OFF, (c4 >> 4) * (128 * 128) + piece(r0 + u * RS + 64), SM::Q_PLANE, fq[u]);
    }
    auto put_k = [&]() {
#pragma unroll
      for (int u = 0; u < KV; ++u) fattn_put4(sgen + SM::K_OFF, (c4 >> 4) * SM::K_BLK + piece(r0 + u * RS), 64 * 128, f[u]);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(k_full);
    };
    put_k();
    fetch(Vb + (size_t)kt0 * 64 * D, d.T - kt0 * 64, f);
    for (long i = (long)blockIdx.x * 256 + tid; i < g.nzero; i += (long)gridDim.x * 256) g.zero[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    const uint32_t tlane = (uint32_t)(q * 32) << 16;
    float o[COLS];
#pragma unroll
    for (int i = 0; i < COLS; ++i) o[i] = 0.f;
    const bool mine = half * COLS < d.Dt;                  // (whole warps)
    float m = -INFINITY, l = 0.f;                          // the row's maximum; the normaliser of this thread's keys
    const int seen = d.causal ? q0 + r : d.T - 1;          // the row's last visible key
    for (int j = 0; j < tiles; ++j) {                       // (a wait that gives up does not leave the loop: barriers are in it)
      const int key0 = (kt0 + j) * 64;
      bool inf = false;
#pragma unroll
      for (int u = 0; u < KV; ++u) {
        const float4 v = f[u];
        inf |= !(fabsf(v.x) <= 3.402823466e38f && fabsf(v.y) <= 3.402823466e38f && fabsf(v.z) <= 3.402823466e38f && fabsf(v.w) <= 3.402823466e38f);
        fattn_put4(sgen + SM::V_OFF, (c4 >> 4) * (64 * 128) + piece(r0 + u * RS), SM::V_PLANE, v);
      }
      if (inf) bad[j & 1] = j + 1;
      fence_proxy_async_smem();
      mbar_wait(s_full, j & 1, g.status, dead);
      tc_fence_after();
      float s[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) s[i] = 0.f;
      const uint32_t sa = tmem + tlane + S0 + half * 32;
      tmem_add16(sa + 128, s);                             // (smallest first)
      tmem_add16(sa + 64, s);
      if (k16s > 4) tmem_add16(sa + 192, s);
      tmem_add16(sa, s);
      const int left = seen - key0 - half * 32;            // this thread's keys 0 .. left are visible
      float mx = -INFINITY;                                // NaN where a score is
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        if (i > left) s[i] = -INFINITY;
        mx = fmax_nan(mx, s[i]);
      }
      if (mx != mx) {
        // (the planes of a value that is not finite are no sum, and products that overflow may do so with either sign)
        const float* qr = g.q + ((size_t)bh * d.T + q0 + min(r, nq - 1)) * D;
        mx = -INFINITY;
#pragma unroll 1
        for (int key = 0; key < min(32, min(left, d.T - 1 - key0 - half * 32) + 1); ++key) {
          const float* kr = Kb + (size_t)(key0 + half * 32 + key) * D;
          float v = 0.f;
#pragma unroll 1
          for (int c = 0; c < d.Dt; c += 4) v = dot4(__ldg(reinterpret_cast<const float4*>(qr + c)), __ldg(reinterpret_cast<const float4*>(kr + c)), v);
          mx = fmaxf(mx, v);
#pragma unroll
          for (int i = 0; i < 32; ++i) s[i] = i == key ? v : s[i];
        }
      }
      __syncwarp();
      sx[half * 128 + r] = mx;
      asm volatile("bar.sync %0, 64;" ::"r"(1 + q) : "memory");
      mx = fmaxf(m, fmaxf(mx, sx[(half ^ 1) * 128 + r]));
      // (a row that has met no visible key keeps everything at zero)
      const float ref = mx == -INFINITY ? 0.f : mx;
      const float alpha = exp2f(m - ref);
      m = mx;
      float ps = 0.f;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        s[i] = i > left ? 0.f : exp2f(s[i] - ref);
        ps += s[i];
      }
      l = l * alpha + ps;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        uint32_t ph[8], pm[8], pl[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) split_bf16x3(s[16 * k + 2 * i], s[16 * k + 2 * i + 1], ph[i], pm[i], pl[i]);
        const uint32_t ta = tmem + tlane + S0 + half * 32 + k * 64;
        tmem_st8(ta, ph);
        tmem_st8(ta + 8, pm);
        tmem_st8(ta + 16, pl);
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full);
      const bool more = j + 1 < tiles;
      if (more) fetch(Kb + (size_t)(key0 + 64) * D, d.T - key0 - 64, f);
#pragma unroll
      for (int i = 0; i < COLS; ++i) o[i] *= alpha;
      if (more) {
        put_k();                                           // (S of this tile has been waited for: K's memory is free)
        fetch(Vb + (size_t)(key0 + 64) * D, d.T - key0 - 64, f);
      }
      mbar_wait(o_full, j & 1, g.status, dead);
      tc_fence_after();
      if (*(volatile int*)&bad[j & 1] == j + 1) {
        // P is the sum of its planes; every visible key's value row on its own
        for (int k = 0; k < 4; ++k) {
          uint32_t p[32];
          tmem_ld32(tmem + tlane + S0 + (k >> 1) * 32 + (k & 1) * 64, p);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            const int key = key0 + 16 * k + i;
            auto part = [&](int pl) { const uint32_t w = p[8 * pl + i / 2]; return __uint_as_float(i & 1 ? w & 0xFFFF0000u : w << 16); };
            const float pv = part(2) + part(1) + part(0);
            if (key <= seen && key < d.T) {
#pragma unroll
              for (int c = 0; c < COLS; c += 4) {
                const float4 v = __ldg(reinterpret_cast<const float4*>(Vb + (size_t)key * D + half * COLS + c));
                o[c] = fmaf(pv, v.x, o[c]); o[c + 1] = fmaf(pv, v.y, o[c + 1]); o[c + 2] = fmaf(pv, v.z, o[c + 2]); o[c + 3] = fmaf(pv, v.w, o[c + 3]);
              }
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(slow_done);
      } else if (mine) {
        tmem_add16(tmem + tlane + PV1 + half * COLS, o);
        tmem_add16(tmem + tlane + PV0 + half * COLS, o);
      }
    }
    // ---- result: this part's sums, maximum and normaliser of every row -----------------------------
    sx[half * 128 + r] = l;
    asm volatile("bar.sync 5, 256;" ::: "memory");         // (and every UMMA has been waited for: Q's and K's memory is free)
    l += sx[(half ^ 1) * 128 + r];
    constexpr int LD = D + 4;
    float* stg = reinterpret_cast<float*>(sgen);
    const float inv = un.parts == 1 ? 1.f / l : 1.f;
#pragma unroll
    for (int i = 0; i < COLS; i += 16) {
      if (half * COLS + i >= k16s * 16) {                  // (columns past the products' width)
#pragma unroll
        for (int c = 0; c < 16; ++c) o[i + c] = 0.f;
      }
    }
#pragma unroll
    for (int i = 0; i < COLS; i += 4)
      *reinterpret_cast<float4*>(stg + r * LD + half * COLS + i) = make_float4(o[i] * inv, o[i + 1] * inv, o[i + 2] * inv, o[i + 3] * inv);
    float* const part = g.part + (size_t)blockIdx.x * 128 * (D + 2);
    if (half == 0) {
      if (un.parts == 1) {
        if (r < nq) *reinterpret_cast<float2*>(g.stats + ((size_t)bh * d.T + q0 + r) * 2) = make_float2(m, inv);
      } else {
        part[128 * D + r] = m;
        part[128 * D + 128 + r] = l;
      }
    }
    asm volatile("bar.sync 5, 256;" ::: "memory");
    float* dst = g.ahat + (((size_t)b * d.T + q0) * d.H + h) * D;
    for (int row = r0; row < (un.parts == 1 ? nq : 128); row += RS) {
      const float4 v = *reinterpret_cast<const float4*>(stg + row * LD + c4 * 4);
      if (un.parts == 1) reinterpret_cast<float4*>(dst + (size_t)row * d.H * D)[c4] = v;
      else __stcg(reinterpret_cast<float4*>(part + (size_t)row * D) + c4, v);
    }
    if (un.parts > 1) {
      __threadfence();
      asm volatile("bar.sync 5, 256;" ::: "memory");
      if (tid == 0) *last_part = atomicInc(g.arrived + un.qt * BH + bh, un.parts - 1) == (unsigned)un.parts - 1;   // (back to zero by itself)
      asm volatile("bar.sync 5, 256;" ::: "memory");
      if (*last_part) {
        __threadfence();
        const float* base = g.part + (size_t)(un.first * BH + bh) * 128 * (D + 2);
        const size_t step = (size_t)BH * 128 * (D + 2);
        // a row's weights of the parts (the result rows' memory is free), then every row's weighted sum: all loads of
        // eight rows and two parts on their way at a time (row by row, each a chain of trips to L2, this took 25 us)
        float* wt = reinterpret_cast<float*>(sgen);
        if (tid < 128) {
          const float* src = base + 128 * D + tid;
          float mm = -INFINITY, ll = 0.f;
#pragma unroll 4
          for (int p = 0; p < un.parts; ++p) mm = fmaxf(mm, __ldcg(src + p * step));
#pragma unroll 4
          for (int p = 0; p < un.parts; ++p) {
            const float lp = __ldcg(src + p * step + 128);
            const float w = lp == 0.f ? 0.f : exp2f(__ldcg(src + p * step) - mm);   // (a part none of whose keys the row sees; NaN goes on)
            wt[p * 128 + tid] = w;
            ll = fmaf(lp, w, ll);
          }
          const float iv = 1.f / ll;
          sx[tid] = iv;
          if (tid < nq) *reinterpret_cast<float2*>(g.stats + ((size_t)bh * d.T + q0 + tid) * 2) = make_float2(mm, iv);
        }
        asm volatile("bar.sync 5, 256;" ::: "memory");
        constexpr int RN = 128 / RS < 8 ? 128 / RS : 8;
        for (int rb = r0; rb < nq; rb += RN * RS) {
          float4 sum[RN];
#pragma unroll
          for (int u = 0; u < RN; ++u) sum[u] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 2
          for (int p = 0; p < un.parts; ++p) {
            float4 v[RN];
#pragma unroll
            for (int u = 0; u < RN; ++u) v[u] = __ldcg(reinterpret_cast<const float4*>(base + p * step + (size_t)(rb + u * RS) * D) + c4);
#pragma unroll
            for (int u = 0; u < RN; ++u) {
              const float w = wt[p * 128 + rb + u * RS];
              sum[u].x = fmaf(v[u].x, w, sum[u].x); sum[u].y = fmaf(v[u].y, w, sum[u].y); sum[u].z = fmaf(v[u].z, w, sum[u].z); sum[u].w = fmaf(v[u].w, w, sum[u].w);
            }
          }
#pragma unroll
          for (int u = 0; u < RN; ++u) {
            const int row = rb + u * RS;
            const float iv = sx[row];
            if (row < nq) reinterpret_cast<float4*>(dst + (size_t)row * d.H * D)[c4] = make_float4(sum[u].x * iv, sum[u].y * iv, sum[u].z * iv, sum[u].w * iv);
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

}  // namespace shtc
