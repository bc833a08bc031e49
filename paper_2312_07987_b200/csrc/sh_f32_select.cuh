// Gates, selection and bucket sort of the fp32 configuration; sh_gate_topk's gates of bf16 storage with d_head above 128.
#pragma once
#include "sh_internal.cuh"

// Lane sums of TOK tokens (8 or 16): at each step a lane keeps half of its tokens and hands the others over; then lane
// l holds token *tok, the same as a butterfly (xor 16, 8, ... 1) over each of them.
template <int TOK>
__device__ __forceinline__ float sh_lane_sums(float (&acc)[TOK], int lane, int* tok) {
  int t = 0;
#pragma unroll
  for (int n = TOK / 2, o = 16; n >= 1; n >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int r = 0; r < n; ++r) {
      const float give = up ? acc[r] : acc[r + n], keep = up ? acc[r + n] : acc[r];
      acc[r] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
    t += up ? n : 0;
  }
#pragma unroll
  for (int o = 32 / TOK / 2; o > 0; o >>= 1) acc[0] += __shfl_xor_sync(0xffffffffu, acc[0], o);
  *tok = t;
  return acc[0];
}

// Bias, top-k and sigmoid of one (token, side, head) from its E logits in shared memory.  blockcnt, where given
// (cleared before): how often each expert is selected, per 128 tokens.
__device__ __forceinline__ void sh_select(float* z, const float* __restrict__ gbias, int* __restrict__ idx, float* __restrict__ gate,
                                          int* __restrict__ blockcnt, const ShDims& d, int t, int grp) {
  const int side = grp / d.H, h = grp % d.H;
  for (int e = 0; e < d.E; ++e) z[e] += gbias[grp * d.E + e];
  const size_t o = (((size_t)side * d.N + t) * d.H + h) * d.k;
  unsigned sel = 0;
  for (int j = 0; j < d.k; ++j) {
    float best = 0.f;
    int pick = -1;
    for (int e = 0; e < d.E; ++e) {
      const float v = z[e];
      if (!((sel >> e) & 1u) && (pick < 0 || v > best)) { best = v; pick = e; }
    }
    sel |= 1u << pick;
    idx[o + j] = pick;
    gate[o + j] = 1.f / (1.f + expf(-best));
    if (blockcnt) atomicAdd(blockcnt + (size_t)(t / SH_TILE_ROWS) * d.G + grp * d.E + pick, 1);
  }
}

// Logits, top-k (a larger logit first, the lower index on a tie) and sigmoid of the chosen ones, on the
// CUDA cores: TOK tokens per block with their rows in shared memory (CH columns at a time: 512, or 1024 where d_model is larger), a warp per
// two gate columns, lanes along d_model.  The block also clears its share of the value rows, which a later kernel
// adds into.  What bounds it is the latency of its few loads, so blocks are small: 1024 tokens of 32 gate
// columns took 490 us in blocks of 128 tokens with a warp per token.
template <int TOK, int CH>
static __global__ void __launch_bounds__(512, 1)
sh_f32_gate_kernel(const float* __restrict__ x, const float* __restrict__ wgate, const float* __restrict__ gbias, int* __restrict__ idx,
                   float* __restrict__ gate, int* __restrict__ blockcnt, float4* __restrict__ zero, long nzero, ShDims d, int vec) {
  extern __shared__ __align__(16) float gsm[];             // [TOK][CH] of x, then [TOK][G] logits
  float* s_z = gsm + TOK * CH;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  constexpr int U = CH / 32;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t0 = blockIdx.x * TOK;
  const long nthr = (long)gridDim.x * 512, me = (long)blockIdx.x * 512 + tid;
  for (int g0 = 0; g0 < d.G; g0 += 32) {                    // a warp's two columns at a time, all of their loads in flight
    const int g = g0 + warp;
    const bool one = g < d.G, two = g + 16 < d.G;
    // (lane l sums the columns l, l + 32, ... of the whole row in order and the lanes are added as a butterfly: the
    //  order of sh_gate_topk_kernel, so that the allocation-free entry point gives the same bits)
    float acc[2][TOK];
#pragma unroll
    for (int r = 0; r < TOK; ++r) acc[0][r] = acc[1][r] = 0.f;
    for (int m0 = 0; m0 < d.M; m0 += CH) {
      const int mw = min(CH, d.M - m0);         // a multiple of 64
      const bool fresh = g0 == 0 || d.M > CH;   // (a row that fits is read once)
      if (fresh) {
        __syncthreads();
        for (int i = tid; i < TOK * (CH / 4); i += 512) {
          const int r = i / (CH / 4), c = (i % (CH / 4)) * 4;
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (c < mw && t0 + r < d.N) {
            const float* p = x + (size_t)(t0 + r) * d.M + m0 + c;
            v = vec ? __ldg(reinterpret_cast<const float4*>(p)) : make_float4(__ldg(p), __ldg(p + 1), __ldg(p + 2), __ldg(p + 3));   // (x off its alignment: sh_gate_topk takes it)
          }
          *reinterpret_cast<float4*>(gsm + r * CH + c) = v;
        }
      }
      float wv[2][U];
      if (one) {
        const float* w0 = wgate + (size_t)g * d.M + m0;
        const float* w1 = w0 + (two ? (size_t)16 * d.M : 0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int c = u * 32 + lane;
          wv[0][u] = c < mw ? __ldg(w0 + c) : 0.f;
          wv[1][u] = c < mw ? __ldg(w1 + c) : 0.f;
        }
      }
      if (fresh) __syncthreads();
      if (one) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (u * 32 >= mw) break;
#pragma unroll
          for (int r = 0; r < TOK; ++r) {
            const float xv = gsm[r * CH + u * 32 + lane];
            acc[0][r] = fmaf(xv, wv[0][u], acc[0][r]);
            acc[1][r] = fmaf(xv, wv[1][u], acc[1][r]);
          }
        }
      }
    }
    if (one) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        int tokn;
        const float z = sh_lane_sums<TOK>(acc[q], lane, &tokn);
        if (lane % (32 / TOK) == 0 && (q == 0 || two)) s_z[tokn * d.G + g + 16 * q] = z;
      }
    }
  }
  for (long i = me; i < nzero; i += nthr) zero[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  const int groups = d.sides * d.H;
  for (int i = tid; i < TOK * groups; i += 512) {
    const int r = i / groups, grp = i % groups;
    if (t0 + r < d.N) sh_select(s_z + r * d.G + grp * d.E, gbias, idx, gate, blockcnt, d, t0 + r, grp);
  }
}

// The same sums for bf16 storage (sh_gate_topk with d_head above 128): 16 tokens and 32 gate columns in shared memory, a
// warp works on 8 x 8 of them.  A word holds two neighbouring columns of a row; half a warp covers 32 columns of
// one token, lane j the sums of the columns 2 j and 2 j + 1 modulo 32 as one FFMA2 per word.  8192 tokens of 32
// columns of 1024: 28 us, of which the FMA pipe's share is 7.4 (four warps a scheduler, 58 % of the issue slots).
constexpr int GB_TOK = 16, GB_NC = 32, GB_CH = 1024, GB_THREADS = 256, GB_XLD = GB_CH / 2 + 16, GB_WLD = GB_CH / 2;
static __global__ void __launch_bounds__(GB_THREADS, 2)
sh_bf16_gate_kernel(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ wgate, const float* __restrict__ gbias, int* __restrict__ idx,
                    float* __restrict__ gate, int* __restrict__ blockcnt, ShDims d, int vec) {
  extern __shared__ __align__(16) uint32_t gsw[];
  uint32_t* s_x = gsw;                                     // [GB_TOK][GB_XLD]: two tokens' words fall into different banks
  uint32_t* s_w = s_x + GB_TOK * GB_XLD;                   // [GB_NC][GB_WLD]
  float* s_z = reinterpret_cast<float*>(s_w + GB_NC * GB_WLD);   // [GB_TOK][G] logits
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int tg = (warp >> 2) * 8, cg = (warp & 3) * 8;     // this warp's tokens and columns
  const int half = lane >> 4, j = lane & 15;
  auto copy16 = [](uint32_t* dst, const __nv_bfloat16* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
  };
  const int passes = (d.N + GB_TOK - 1) / GB_TOK, groups = d.sides * d.H;
  for (int pass = blockIdx.x; pass < passes; pass += gridDim.x) {
    const int t0 = pass * GB_TOK;
    for (int g0 = 0; g0 < d.G; g0 += GB_NC) {
      float2 acc[8][4];                                    // [column][pair of tokens]
#pragma unroll
      for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[q][p] = make_float2(0.f, 0.f);
      for (int m0 = 0; m0 < d.M; m0 += GB_CH) {
        const int mw = min(GB_CH, d.M - m0), n16 = mw / 8; // a multiple of 128; its 16-byte pieces
        __syncthreads();
        if (g0 == 0 || d.M > GB_CH)                        // (a row that fits is read once)
          for (int i = tid; i < GB_TOK * n16; i += GB_THREADS) {
            const int r = i / n16, c = i % n16;
            const __nv_bfloat16* p = x + (size_t)min(t0 + r, d.N - 1) * d.M + m0 + c * 8;
            uint32_t* o = s_x + r * GB_XLD + c * 4;
            if (vec) copy16(o, p);
            else
              for (int u = 0; u < 4; ++u)                  // (x off its alignment: sh_gate_topk takes it)
                o[u] = (uint32_t)__bfloat16_as_ushort(p[2 * u]) | ((uint32_t)__bfloat16_as_ushort(p[2 * u + 1]) << 16);
          }
        if (pass == (int)blockIdx.x || d.G > GB_NC || d.M > GB_CH)
          for (int i = tid; i < GB_NC * n16; i += GB_THREADS) {
            const int r = i / n16, c = i % n16;
            copy16(s_w + r * GB_WLD + c * 4, wgate + (size_t)min(g0 + r, d.G - 1) * d.M + m0 + c * 8);
          }
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        if (g0 + cg >= d.G) continue;                      // (whole warps)
        const uint32_t* px = s_x + (tg + half) * GB_XLD + j;
        const uint32_t* pw = s_w + cg * GB_WLD + j;
        // (a sum runs over its columns of the whole row in order: the order of sh_gate_topk_kernel, bit for bit)
#pragma unroll 2
        for (int b = 0; b < mw / 2; b += 16) {
          float2 xv[4], wv[8];
#pragma unroll
          for (int p = 0; p < 4; ++p) {
            const uint32_t v = px[2 * p * GB_XLD + b];
            xv[p] = make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u));
          }
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const uint32_t v = pw[q * GB_WLD + b];
            wv[q] = make_float2(__uint_as_float(v << 16), __uint_as_float(v & 0xFFFF0000u));
          }
#pragma unroll
          for (int q = 0; q < 8; ++q)
#pragma unroll
            for (int p = 0; p < 4; ++p) acc[q][p] = __ffma2_rn(xv[p], wv[q], acc[q][p]);
        }
      }
      if (g0 + cg < d.G) {
        // sums over the 16 lanes: a lane keeps half of the 32 values at each step; value i is column i / 4, pair i % 4
        float2* v = &acc[0][0];
        int first = 0;
#pragma unroll
        for (int n = 16, o = 8; o >= 1; n >>= 1, o >>= 1) {
          const bool up = (lane & o) != 0;
#pragma unroll
          for (int i = 0; i < n; ++i) {
            const float2 give = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
            v[i] = make_float2(keep.x + __shfl_xor_sync(0xffffffffu, give.x, o), keep.y + __shfl_xor_sync(0xffffffffu, give.y, o));
          }
          first += up ? n : 0;
        }
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int col = g0 + cg + ((first + i) >> 2), r = tg + 2 * ((first + i) & 3) + half;
          if (col < d.G) s_z[r * d.G + col] = v[i].x + v[i].y;
        }
      }
    }
    __syncthreads();
    for (int i = tid; i < GB_TOK * groups; i += GB_THREADS) {
      const int r = i / groups, grp = i % groups;
      if (t0 + r < d.N) sh_select(s_z + r * d.G + grp * d.E, gbias, idx, gate, blockcnt, d, t0 + r, grp);
    }
  }
}

// Bucket sort of up to F32_SORT_MAX tokens, one block per (side, head): the stable counting sort of the tokens by chosen expert, in
// two sweeps of 1024 tokens at a time (totals, then placement).  No block needs another's counts: every
// head owns a fixed range of the row-tile table (mt = (N k + 127 E) / 128 entries, the unused ones empty).
// Above, sh_sort_kernel with a block per 128 tokens (it wants their counts and an empty tile table ahead of it): 53 us
// here for 8192 tokens, and in proportion beyond.
constexpr int F32_SORT_MAX = 4096;
static __global__ void __launch_bounds__(1024)
sh_f32_sort_kernel(const int* __restrict__ idx, const float* __restrict__ gate, int* __restrict__ offsets, int* __restrict__ lists,
                   float* __restrict__ lgate, ShTile* __restrict__ tiles, ShDims d, int mt) {
  __shared__ int s_tot[32], s_off[33], s_run[32];
  __shared__ int s_w[32][33];                              // [warp][expert]
  __shared__ int s_tile[33];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = blockIdx.x, side = grp / d.H, h = grp % d.H;
  if (tid < 32) s_tot[tid] = 0;
  __syncthreads();
  int mine = 0;                                            // lane e: selections of expert e by this warp's tokens
  for (int t0 = 0; t0 < d.N; t0 += 1024) {
    const int t = t0 + tid;
    unsigned sel = 0;
    if (t < d.N) {
      const size_t o = (((size_t)side * d.N + t) * d.H + h) * d.k;
      for (int j = 0; j < d.k; ++j)
        if (SH_INDEX_OK(idx[o + j], d.E, d.status, SH_SITE_SORT_EXPERT)) sel |= 1u << idx[o + j];
    }
    for (int e = 0; e < d.E; ++e) {
      const unsigned bal = __ballot_sync(0xffffffffu, (sel >> e) & 1u);
      if (lane == e) mine += __popc(bal);
    }
  }
  if (lane < d.E && mine) atomicAdd(&s_tot[lane], mine);
  __syncthreads();
  if (warp == 0) {                                         // lane e: exclusive sums over the experts
    const int tot = lane < d.E ? s_tot[lane] : 0, nt = (tot + SH_TILE_ROWS - 1) / SH_TILE_ROWS;
    int run = tot, tl = nt;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, run, s), w = __shfl_up_sync(0xffffffffu, tl, s);
      if (lane >= s) { run += u; tl += w; }
    }
    s_run[lane] = s_off[lane] = run - tot; s_tile[lane] = tl - nt;
    if (lane < d.E) offsets[(size_t)grp * (d.E + 1) + lane] = run - tot;
    if (lane == d.E - 1) { s_off[d.E] = run; s_tile[d.E] = tl; offsets[(size_t)grp * (d.E + 1) + d.E] = run; }
  }
  __syncthreads();
  ShTile* tp = tiles + (size_t)side * d.max_tiles + (size_t)h * mt;
  for (int i = tid; i < mt; i += 1024) {
    ShTile tl;
    tl.h = h; tl.e = 0; tl.row0 = 0; tl.nrows = 0;
    if (i < s_tile[d.E]) {
      int e = 0;
      while (s_tile[e + 1] <= i) ++e;
      const int r = (i - s_tile[e]) * SH_TILE_ROWS;
      tl.e = e; tl.row0 = s_off[e] + r; tl.nrows = min(SH_TILE_ROWS, s_off[e + 1] - s_off[e] - r);
    }
    tp[i] = tl;
  }
  int* ls = lists + (size_t)grp * d.N * d.k;
  float* lg = lgate + (size_t)grp * d.N * d.k;
  for (int t0 = 0; t0 < d.N; t0 += 1024) {
    const int t = t0 + tid;
    const bool live = t < d.N;
    const size_t o = (((size_t)side * d.N + t) * d.H + h) * d.k;
    unsigned sel = 0;
    if (live)
      for (int j = 0; j < d.k; ++j)
        if (SH_INDEX_OK(idx[o + j], d.E, d.status, SH_SITE_SORT_EXPERT)) sel |= 1u << idx[o + j];
    unsigned mybal = 0;                                    // lane e: which lanes chose expert e
    for (int e = 0; e < d.E; ++e) {
      const unsigned bal = __ballot_sync(0xffffffffu, (sel >> e) & 1u);
      if (lane == e) { s_w[warp][e] = __popc(bal); mybal = bal; }
    }
    __syncthreads();
    if (warp < d.E) {                                      // warp e: where each warp's tokens of expert e start
      const int v = s_w[lane][warp];
      int inc = v;
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, inc, s);
        if (lane >= s) inc += u;
      }
      const int base = s_run[warp];
      s_w[lane][warp] = base + inc - v;
      if (lane == 31) s_run[warp] = base + inc;
    }
    __syncthreads();
    for (int j = 0; j < d.k; ++j) {
      const int e = live ? idx[o + j] : 0;
      const unsigned bal = __shfl_sync(0xffffffffu, mybal, e);
      if (live && SH_INDEX_OK(e, d.E, d.status, SH_SITE_SORT_EXPERT)) {
        const int pos = s_w[warp][e] + __popc(bal & ((1u << lane) - 1u));
        if (SH_INDEX_OK(pos, (long long)d.N * d.k, d.status, SH_SITE_SORT_SLOT)) {
          ls[pos] = t;
          lg[pos] = gate[o + j];
        }
      }
    }
    __syncthreads();
  }
}
