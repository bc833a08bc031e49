// Attention of the fp32 configuration, forward and backward, on the CUDA cores (fp32 FMA).  The forward pass of longer
// sequences is in sh_f32_attn_tc.cuh.
//
// A layer's share of attention is small here (sequences of a few hundred tokens: 0.5 of the 7 GFLOP of
// a 262M-scale forward pass), and what bounds it is the longest chain of key tiles one SM works off,
// not the FMA peak: small tiles, two thread groups per block on alternate tiles.
#pragma once
#include "sh_tc_prims.cuh"

namespace shtc {

__device__ __forceinline__ void group_sync(int id, int threads) { asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory"); }
__device__ __forceinline__ void fa_cp16(float* dst, const float* src, bool ok) {
  const uint32_t s = (uint32_t)__cvta_generic_to_shared(dst);
  const int n = ok ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void fa_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void fa_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

template <bool B> struct fa_bool { static constexpr bool value = B; };

// `rows` rows of W floats (row stride D in memory, LD in shared memory; rows at or past `live` zero), by 128 threads.
template <int D>
__device__ __forceinline__ void fa_tile(float* dst, const float* src, int rows, int live, long src_ld, int t) {
  constexpr int LD = D + 4, C = D / 4;
  for (int i = t; i < rows * C; i += 128) {
    const int r = i / C, c = i % C;
    fa_cp16(dst + r * LD + 4 * c, src + (r < live ? (long)r * src_ld + 4 * c : 0), r < live);
  }
}

__device__ __forceinline__ float dot4(float4 a, float4 b, float s) {
  s = fmaf(a.x, b.x, s); s = fmaf(a.y, b.y, s); s = fmaf(a.z, b.z, s); return fmaf(a.w, b.w, s);
}

// ---- forward ---------------------------------------------------------------------------------------
// Block: 32 queries of one (sequence, head), 256 threads = two groups of 128; group g takes the key
// tiles (64 keys) g, g + 2, ... with its own K and V buffers and running softmax, the two are joined
// at the end.  Thread (ty of 8, tx of 16): scores of rows ty + 8 i and keys tx + 16 j, output rows
// ty + 8 i and columns 4 tx + 64 c.  K of the next tile is fetched under the P V product, V under the
// scores.  Rows are D + 4 floats apart: the eight 16-byte loads of a phase fall into different banks.
// stats [B, H, T, 2]: the row's score maximum (base 2) and 1 / normaliser, for the backward pass.
// The blocks also clear the layer's output, which the next kernel adds into: this is the first kernel behind
// the last read of x, and a caller may pass x itself as the output.
template <int D>
struct FAttnSmem {
  static constexpr int LD = D + 4, KT = D == 256 ? 32 : 64, PLD = KT + 4;
  static constexpr int GROUP = 2 * KT * LD + 32 * PLD;       // floats: K, V, P
  static constexpr int TOTAL = (32 * LD + 2 * GROUP) * 4;
};

template <int D>
__global__ void __launch_bounds__(256)
sh_f32_attn_kernel(const float* __restrict__ Q, const float* __restrict__ K, const float* __restrict__ V, float* __restrict__ Ahat,
                   float* __restrict__ stats, float4* __restrict__ zero, long nzero, ShDims d) {
  using SM = FAttnSmem<D>;
  constexpr int LD = SM::LD, KT = SM::KT, PLD = SM::PLD, KJ = KT / 16;
  constexpr int NC = D >= 64 ? D / 64 : 1;
  extern __shared__ __align__(16) float fsm[];
  pdl_wait();
  pdl_trigger();                                           // (behind the wait: what the next kernel reads ahead of its own is complete)
  const int tid = threadIdx.x, grp = tid >> 7, t = tid & 127, ty = t >> 4, tx = t & 15;
  float* sQ = fsm;
  float* sK = fsm + 32 * LD + grp * SM::GROUP;
  float* sV = sK + KT * LD;
  float* sP = sV + KT * LD;
  const int BH = d.B * d.H, bh = blockIdx.x % BH, b = bh / d.H, h = bh % d.H;
  const int q0 = d.Tc + ((int)(gridDim.x / BH) - 1 - (int)(blockIdx.x / BH)) * 32;   // the longest rows first
  const int nq = min(32, d.T - q0);
  const float* Kb = K + (size_t)bh * d.T * D;
  const float* Vb = V + (size_t)bh * d.T * D;
  const int nkeys = d.causal ? min(d.T, q0 + nq) : d.T;
  const int ntile = (nkeys + KT - 1) / KT;
  const int d4n = (d.Dt + 3) / 4;
  const bool col_ok = D >= 64 || tx < D / 4;
  if (grp == 0) fa_tile<D>(sQ, Q + ((size_t)bh * d.T + q0) * D, 32, nq, D, t);
  int kt = grp;
  if (kt < ntile) fa_tile<D>(sK, Kb + (size_t)kt * KT * D, KT, d.T - kt * KT, D, t);
  fa_commit();
  if (kt < ntile) fa_tile<D>(sV, Vb + (size_t)kt * KT * D, KT, d.T - kt * KT, D, t);
  fa_commit();
  for (long i = (long)blockIdx.x * 256 + tid; i < nzero; i += (long)gridDim.x * 256) zero[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  fa_wait<1>();
  __syncthreads();
  float o[4][4 * NC], m[4], l[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m[i] = -INFINITY; l[i] = 0.f;
#pragma unroll
    for (int c = 0; c < 4 * NC; ++c) o[i][c] = 0.f;
  }
  for (; kt < ntile; kt += 2) {
    float s[4][KJ];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < KJ; ++j) s[i][j] = 0.f;
#pragma unroll 2
    for (int c = 0; c < d4n; ++c) {
      float4 kv[KJ];
#pragma unroll
      for (int j = 0; j < KJ; ++j) kv[j] = *reinterpret_cast<const float4*>(sK + (tx + 16 * j) * LD + 4 * c);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 qv = *reinterpret_cast<const float4*>(sQ + (ty + 8 * i) * LD + 4 * c);
#pragma unroll
        for (int j = 0; j < KJ; ++j) s[i][j] = dot4(qv, kv[j], s[i][j]);
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int qi = q0 + ty + 8 * i;
      const int last = d.causal ? qi : d.T - 1;
      float mx = m[i];
#pragma unroll
      for (int j = 0; j < KJ; ++j) {
        if (kt * KT + tx + 16 * j > last) s[i][j] = -INFINITY;
        mx = fmaxf(mx, s[i][j]);
      }
#pragma unroll
      for (int x = 8; x > 0; x >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
      // (a row that has met no visible key keeps everything at zero)
      const float ref = mx == -INFINITY ? 0.f : mx;
      const float alpha = exp2f(m[i] - ref);
      float ps = 0.f;
#pragma unroll
      for (int j = 0; j < KJ; ++j) {
        const bool seen = kt * KT + tx + 16 * j <= last;
        const float p = seen ? exp2f(s[i][j] - ref) : 0.f;
        ps += p;
        sP[(ty + 8 * i) * PLD + tx + 16 * j] = p;
      }
#pragma unroll
      for (int x = 8; x > 0; x >>= 1) ps += __shfl_xor_sync(0xffffffffu, ps, x);
      l[i] = l[i] * alpha + ps;
      m[i] = mx;
#pragma unroll
      for (int c = 0; c < 4 * NC; ++c) o[i][c] *= alpha;
    }
    fa_wait<0>();                                          // V of this tile
    group_sync(1 + grp, 128);                              // K read, P written, V there for every thread
    if (kt + 2 < ntile) fa_tile<D>(sK, Kb + (size_t)(kt + 2) * KT * D, KT, d.T - (kt + 2) * KT, D, t);
    fa_commit();
    // (a tile some row sees a part of: what a row does not see is left out of its sum, not multiplied by zero -
    //  a value that is not finite stays with the rows that see it)
    auto product = [&](auto part) {
      const int kend = decltype(part)::value ? min(KT, nkeys - kt * KT) : KT;    // (past the last row's last key: nothing to add)
#pragma unroll 2
      for (int kk = 0; kk < kend; kk += 4) {
        float4 pv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) pv[i] = *reinterpret_cast<const float4*>(sP + (ty + 8 * i) * PLD + kk);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const float4 vv = *reinterpret_cast<const float4*>(sV + (kk + u) * LD + 4 * tx + 64 * c);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (decltype(part)::value && kt * KT + kk + u > q0 + ty + 8 * i) continue;
              const float p = u == 0 ? pv[i].x : u == 1 ? pv[i].y : u == 2 ? pv[i].z : pv[i].w;
              o[i][4 * c] = fmaf(p, vv.x, o[i][4 * c]);
              o[i][4 * c + 1] = fmaf(p, vv.y, o[i][4 * c + 1]);
              o[i][4 * c + 2] = fmaf(p, vv.z, o[i][4 * c + 2]);
              o[i][4 * c + 3] = fmaf(p, vv.w, o[i][4 * c + 3]);
            }
          }
        }
      }
    };
    if (col_ok) {
      if (d.causal && kt * KT + KT - 1 > q0) product(fa_bool<true>());
      else product(fa_bool<false>());
    }
    group_sync(1 + grp, 128);                              // V and P read
    if (kt + 2 < ntile) fa_tile<D>(sV, Vb + (size_t)(kt + 2) * KT * D, KT, d.T - (kt + 2) * KT, D, t);
    fa_commit();
    fa_wait<1>();                                          // K of the next tile
    group_sync(1 + grp, 128);
  }
  fa_wait<0>();
  __syncthreads();
  // group 1 hands its part over in group 1's own buffers
  float* xO = fsm + 32 * LD + SM::GROUP;                   // [32][LD]
  float* xM = xO + KT * LD;                                // [32][2]
  if (grp == 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = ty + 8 * i;
      if (tx == 0) { xM[2 * r] = m[i]; xM[2 * r + 1] = l[i]; }
      if (col_ok) {
#pragma unroll
        for (int c = 0; c < NC; ++c)
          *reinterpret_cast<float4*>(xO + r * LD + 4 * tx + 64 * c) = make_float4(o[i][4 * c], o[i][4 * c + 1], o[i][4 * c + 2], o[i][4 * c + 3]);
      }
    }
  }
  __syncthreads();
  if (grp == 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = ty + 8 * i;
      if (r >= nq) continue;
      const float m1 = xM[2 * r], l1 = xM[2 * r + 1];
      const float mm = fmaxf(m[i], m1);
      const float a0 = exp2f(m[i] - mm), a1 = l1 != 0.f ? exp2f(m1 - mm) : 0.f;   // (group 1 may have had no tile)
      const float inv = 1.f / (l[i] * a0 + l1 * a1);
      float* dst = Ahat + (((size_t)b * d.T + q0 + r) * d.H + h) * D;
      if (col_ok) {
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
          if (l1 != 0.f) x = *reinterpret_cast<const float4*>(xO + r * LD + 4 * tx + 64 * c);
          float4 w;
          w.x = (o[i][4 * c] * a0 + x.x * a1) * inv; w.y = (o[i][4 * c + 1] * a0 + x.y * a1) * inv;
          w.z = (o[i][4 * c + 2] * a0 + x.z * a1) * inv; w.w = (o[i][4 * c + 3] * a0 + x.w * a1) * inv;
          *reinterpret_cast<float4*>(dst + 4 * tx + 64 * c) = w;
        }
      }
      if (tx == 0) {
        float* st = stats + ((size_t)bh * d.T + q0 + r) * 2;
        st[0] = mm; st[1] = inv;
      }
    }
  }
}

// ---- backward --------------------------------------------------------------------------------------
// What the backward pass adds into, cleared in one launch (as memsets, up to six of them, each with a gap in the chain
// of launches in front and behind: 16 us of a step of 8 x 256 tokens with the two small kernels that went with them).  Pointers may be 4-byte aligned.
struct FClear { float* p[8]; long n[8]; };
static __global__ void __launch_bounds__(256)
sh_f32_clear_kernel(const __grid_constant__ FClear c) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const long me = (long)blockIdx.x * 256 + threadIdx.x, all = (long)gridDim.x * 256;
#pragma unroll
  for (int r = 0; r < 8; ++r) {
    float* const p = c.p[r];
    const long n = c.n[r], n4 = (uintptr_t)p % 16 == 0 ? n / 4 : 0;
    for (long i = me; i < n4; i += all) reinterpret_cast<float4*>(p)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (long i = 4 * n4 + me; i < n; i += all) p[i] = 0.f;
  }
}

// Block: 32 keys of one (sequence, head) and a run of query tiles (TQ queries each; blockIdx.y), two
// groups of 128 threads on alternate query tiles.  Per tile: S = Q K^T and dP = dAhat V^T, then
// P = exp2(S - max) / norm, dS = P o (dP - dsum); dV += P^T dAhat and dK += dS^T Q in registers,
// dQ += dS K by vector reductions (several key blocks contribute).  At the end the groups' dK and dV
// are joined in shared memory and reduced into global memory.
template <int D>
struct FBwSmem {
  static constexpr int LD = D + 4, TQ = D == 256 ? 32 : 64, PLD = 36;
  static constexpr int GROUP = 2 * TQ * LD + 2 * TQ * PLD + 4 * TQ;
  static constexpr int TOTAL = (2 * 32 * LD + 2 * GROUP) * 4;
};

template <int D>
__global__ void __launch_bounds__(256)
sh_f32_attn_bw_kernel(const float* __restrict__ Q, const float* __restrict__ K, const float* __restrict__ V, const float* __restrict__ dahat,
                      const float* __restrict__ stats, const float* __restrict__ dsum, float* __restrict__ dq, float* __restrict__ dk,
                      float* __restrict__ dv, ShDims d, int run) {
  using SM = FBwSmem<D>;
  constexpr int LD = SM::LD, TQ = SM::TQ, PLD = SM::PLD, RI = TQ / 16;
  constexpr int NC = D >= 64 ? D / 64 : 1;
  extern __shared__ __align__(16) float fsm[];
  pdl_wait();
  pdl_trigger();                                           // (behind the wait: what the next kernel reads ahead of its own is complete)
  const int tid = threadIdx.x, grp = tid >> 7, t = tid & 127;
  const int sy = t >> 3, sx = t & 7;                       // scores: rows sy + 16 i, keys sx + 8 j
  const int ty = t >> 4, tx = t & 15;                      // products: rows, columns 4 tx + 64 c
  float* sK = fsm;
  float* sV = sK + 32 * LD;
  float* sQ = sV + 32 * LD + grp * SM::GROUP;
  float* sO = sQ + TQ * LD;                                // dAhat rows
  float* sP = sO + TQ * LD;                                // [TQ][PLD]
  float* sS = sP + TQ * PLD;
  float* sR = sS + TQ * PLD;                               // [TQ][4]: maximum, 1 / normaliser, dsum
  const int BH = d.B * d.H, bh = blockIdx.x % BH, b = bh / d.H, h = bh % d.H;
  const int k0 = (int)(blockIdx.x / BH) * 32, nk = min(32, d.T - k0);
  const int qt_first = d.causal ? k0 / TQ : 0, qt_all = (d.T + TQ - 1) / TQ;
  const int qt_lo = qt_first + (int)blockIdx.y * run, qt_hi = min(qt_all, qt_lo + run);
  if (qt_lo >= qt_hi) return;
  const int HD = d.H * D;
  const int d4n = (d.Dt + 3) / 4;
  const bool col_ok = D >= 64 || tx < D / 4;
  if (grp == 0) fa_tile<D>(sK, K + ((size_t)bh * d.T + k0) * D, 32, nk, D, t);
  else fa_tile<D>(sV, V + ((size_t)bh * d.T + k0) * D, 32, nk, D, t);
  fa_commit();
  float gk[4][4 * NC], gv[4][4 * NC];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int c = 0; c < 4 * NC; ++c) gk[i][c] = gv[i][c] = 0.f;
  const float inv_sqrt_d = rsqrtf((float)d.Dt);
  fa_wait<0>();
  __syncthreads();
  for (int qt = qt_lo + grp; qt < qt_hi; qt += 2) {
    const int q0 = qt * TQ, nq = min(TQ, d.T - q0);
    const size_t tok0 = (size_t)b * d.T + q0;
    fa_tile<D>(sQ, Q + ((size_t)bh * d.T + q0) * D, TQ, nq, D, t);
    fa_tile<D>(sO, dahat + (tok0 * d.H + h) * D, TQ, nq, HD, t);
    fa_commit();
    for (int i = t; i < TQ; i += 128) {
      const bool ok = i < nq;
      const float* st = stats + ((size_t)bh * d.T + q0 + (ok ? i : 0)) * 2;
      sR[4 * i] = ok ? st[0] : 0.f; sR[4 * i + 1] = ok ? st[1] : 0.f;
      sR[4 * i + 2] = ok ? dsum[(tok0 + i) * d.H + h] : 0.f;
    }
    fa_wait<0>();
    group_sync(1 + grp, 128);
    {
      float s[RI][4], p[RI][4];
#pragma unroll
      for (int i = 0; i < RI; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) s[i][j] = p[i][j] = 0.f;
      for (int c = 0; c < d4n; ++c) {
        float4 kv[4], vv[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          kv[j] = *reinterpret_cast<const float4*>(sK + (sx + 8 * j) * LD + 4 * c);
          vv[j] = *reinterpret_cast<const float4*>(sV + (sx + 8 * j) * LD + 4 * c);
        }
#pragma unroll
        for (int i = 0; i < RI; ++i) {
          const float4 qv = *reinterpret_cast<const float4*>(sQ + (sy + 16 * i) * LD + 4 * c);
          const float4 ov = *reinterpret_cast<const float4*>(sO + (sy + 16 * i) * LD + 4 * c);
#pragma unroll
          for (int j = 0; j < 4; ++j) { s[i][j] = dot4(qv, kv[j], s[i][j]); p[i][j] = dot4(ov, vv[j], p[i][j]); }
        }
      }
#pragma unroll
      for (int i = 0; i < RI; ++i) {
        const int r = sy + 16 * i, qi = q0 + r;
        const float4 st = *reinterpret_cast<const float4*>(sR + 4 * r);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int key = k0 + sx + 8 * j;
          const bool seen = r < nq && key < d.T && (!d.causal || key <= qi);
          const float pr = seen ? exp2f(s[i][j] - st.x) * st.y : 0.f;
          sP[r * PLD + sx + 8 * j] = pr;
          sS[r * PLD + sx + 8 * j] = seen ? pr * (p[i][j] - st.z) : 0.f;
        }
      }
    }
    group_sync(1 + grp, 128);
    // (pairs of a partly visible tile that do not see one another are left out, as in the forward pass)
    auto products = [&](auto part) {
      constexpr bool PART = decltype(part)::value;
      const int rlo = PART ? max(0, k0 - q0) : 0;            // the first row that sees a key of the block
      // dV, dK: keys 4 ty ... 4 ty + 3
#pragma unroll 2
      for (int r = rlo; r < TQ; ++r) {
        const float4 p4 = *reinterpret_cast<const float4*>(sP + r * PLD + 4 * ty);
        const float4 s4 = *reinterpret_cast<const float4*>(sS + r * PLD + 4 * ty);
        const float pp[4] = {p4.x, p4.y, p4.z, p4.w}, ss[4] = {s4.x, s4.y, s4.z, s4.w};
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const float4 ov = *reinterpret_cast<const float4*>(sO + r * LD + 4 * tx + 64 * c);
          const float4 qv = *reinterpret_cast<const float4*>(sQ + r * LD + 4 * tx + 64 * c);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (PART && k0 + 4 * ty + i > q0 + r) continue;
            gv[i][4 * c] = fmaf(pp[i], ov.x, gv[i][4 * c]); gv[i][4 * c + 1] = fmaf(pp[i], ov.y, gv[i][4 * c + 1]);
            gv[i][4 * c + 2] = fmaf(pp[i], ov.z, gv[i][4 * c + 2]); gv[i][4 * c + 3] = fmaf(pp[i], ov.w, gv[i][4 * c + 3]);
            gk[i][4 * c] = fmaf(ss[i], qv.x, gk[i][4 * c]); gk[i][4 * c + 1] = fmaf(ss[i], qv.y, gk[i][4 * c + 1]);
            gk[i][4 * c + 2] = fmaf(ss[i], qv.z, gk[i][4 * c + 2]); gk[i][4 * c + 3] = fmaf(ss[i], qv.w, gk[i][4 * c + 3]);
          }
        }
      }
      // dQ: rows r0 + ty + 8 i
      for (int r0 = rlo; r0 < TQ; r0 += 32) {
        float gq[4][4 * NC];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int c = 0; c < 4 * NC; ++c) gq[i][c] = 0.f;
#pragma unroll 2
        for (int kk = 0; kk < 32; kk += 4) {
          float4 sv[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) sv[i] = *reinterpret_cast<const float4*>(sS + (r0 + ty + 8 * i) * PLD + kk);
#pragma unroll
          for (int u = 0; u < 4; ++u) {
#pragma unroll
            for (int c = 0; c < NC; ++c) {
              const float4 kv = *reinterpret_cast<const float4*>(sK + (kk + u) * LD + 4 * tx + 64 * c);
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                if (PART && k0 + kk + u > q0 + r0 + ty + 8 * i) continue;
                const float w = u == 0 ? sv[i].x : u == 1 ? sv[i].y : u == 2 ? sv[i].z : sv[i].w;
                gq[i][4 * c] = fmaf(w, kv.x, gq[i][4 * c]); gq[i][4 * c + 1] = fmaf(w, kv.y, gq[i][4 * c + 1]);
                gq[i][4 * c + 2] = fmaf(w, kv.z, gq[i][4 * c + 2]); gq[i][4 * c + 3] = fmaf(w, kv.w, gq[i][4 * c + 3]);
              }
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = r0 + ty + 8 * i;
          if (r >= nq) continue;
          float* dst = dq + ((tok0 + r) * d.H + h) * D + 4 * tx;
#pragma unroll
          for (int c = 0; c < NC; ++c)
            if (4 * tx + 64 * c < d.Dt)
              red_add_v4_f32(dst + 64 * c, gq[i][4 * c] * inv_sqrt_d, gq[i][4 * c + 1] * inv_sqrt_d, gq[i][4 * c + 2] * inv_sqrt_d, gq[i][4 * c + 3] * inv_sqrt_d);
        }
      }
    };
    if (col_ok) {
      if (d.causal && k0 + 31 > q0) products(fa_bool<true>());
      else products(fa_bool<false>());
    }
    group_sync(1 + grp, 128);                              // the tile's buffers are free
  }
  __syncthreads();
  // group 1's sums through group 1's Q and dAhat buffers
  float* xK = fsm + 2 * 32 * LD + SM::GROUP;
  float* xV = xK + 32 * LD;
  if (grp == 1 && col_ok) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        const int o = (4 * ty + i) * LD + 4 * tx + 64 * c;
        *reinterpret_cast<float4*>(xK + o) = make_float4(gk[i][4 * c], gk[i][4 * c + 1], gk[i][4 * c + 2], gk[i][4 * c + 3]);
        *reinterpret_cast<float4*>(xV + o) = make_float4(gv[i][4 * c], gv[i][4 * c + 1], gv[i][4 * c + 2], gv[i][4 * c + 3]);
      }
  }
  __syncthreads();
  if (grp == 0 && col_ok) {
    const float ks = 0.6931471805599453f;                  // dK = dS Q / sqrt(d); the stored Q carries log2(e) / sqrt(d)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int key = 4 * ty + i;
      if (key >= nk) continue;
      const size_t row = (((size_t)b * d.T + k0 + key) * d.H + h) * D;
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        if (4 * tx + 64 * c >= d.Dt) continue;
        const int o = key * LD + 4 * tx + 64 * c;
        const float4 a = *reinterpret_cast<const float4*>(xK + o), v = *reinterpret_cast<const float4*>(xV + o);
        red_add_v4_f32(dk + row + 4 * tx + 64 * c, (gk[i][4 * c] + a.x) * ks, (gk[i][4 * c + 1] + a.y) * ks, (gk[i][4 * c + 2] + a.z) * ks, (gk[i][4 * c + 3] + a.w) * ks);
        red_add_v4_f32(dv + row + 4 * tx + 64 * c, gv[i][4 * c] + v.x, gv[i][4 * c + 1] + v.y, gv[i][4 * c + 2] + v.z, gv[i][4 * c + 3] + v.w);
      }
    }
  }
}

}  // namespace shtc
