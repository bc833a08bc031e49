// Selection and bucket sort of the fp32 configuration, one launch.
//
// Block = (side, head): top-k of every token's logits (a larger logit first, the lower index on a
// tie), sigmoid of the chosen ones, and the stable counting sort of the tokens by chosen expert, in two
// sweeps of 1024 tokens at a time (totals, then placement).  No block needs another's counts: every
// head owns a fixed range of the row-tile table (mt = (N k + 127 E) / 128 entries, the unused ones
// empty).  What bounds it is latency (two sweeps of a few dependent loads): a block per 128 tokens
// with a histogram exchange between two kernels took 490 + 13 us on 1024 tokens of 32 gate columns,
// this one and the gate columns of the projection GEMM a few us.
#pragma once
#include "sh_internal.cuh"

static __global__ void __launch_bounds__(1024)
sh_f32_select_kernel(const float* __restrict__ z, int ldz, const float* __restrict__ gbias, int* __restrict__ idx, float* __restrict__ gate,
                     int* __restrict__ offsets, int* __restrict__ lists, float* __restrict__ lgate, ShTile* __restrict__ tiles, ShDims d, int mt) {
  __shared__ int s_tot[32], s_off[33], s_run[32];
  __shared__ int s_w[32][33];                              // [warp][expert]
  __shared__ int s_tile[33];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int grp = blockIdx.x, side = grp / d.H, h = grp % d.H;
  const float bias = lane < d.E ? gbias[grp * d.E + lane] : 0.f;
  if (tid < 32) s_tot[tid] = 0;
  __syncthreads();
  int mine = 0;                                            // lane e: selections of expert e by this warp's tokens
  for (int t0 = 0; t0 < d.N; t0 += 1024) {
    const int t = t0 + tid;
    unsigned sel = 0;
    const bool live = t < d.N;
    const float* zr = z + (size_t)(live ? t : 0) * ldz + grp * d.E;
    const size_t o = (((size_t)side * d.N + t) * d.H + h) * d.k;
    for (int j = 0; j < d.k; ++j) {
      float best = 0.f;
      int pick = -1;
      for (int e = 0; e < d.E; ++e) {
        const float v = zr[e] + __shfl_sync(0xffffffffu, bias, e);
        if (!((sel >> e) & 1u) && (pick < 0 || v > best)) { best = v; pick = e; }
      }
      sel |= 1u << pick;
      if (live) { idx[o + j] = pick; gate[o + j] = 1.f / (1.f + expf(-best)); }
    }
    if (!live) sel = 0;
    for (int e = 0; e < d.E; ++e) {
      const unsigned bal = __ballot_sync(0xffffffffu, (sel >> e) & 1u);
      if (lane == e) mine += __popc(bal);
    }
  }
  if (lane < d.E && mine) atomicAdd(&s_tot[lane], mine);
  __syncthreads();
  if (tid == 0) {
    int run = 0, tiles_before = 0;
    for (int e = 0; e < d.E; ++e) {
      s_off[e] = run; s_run[e] = run; s_tile[e] = tiles_before;
      offsets[(size_t)grp * (d.E + 1) + e] = run;
      run += s_tot[e];
      tiles_before += (s_tot[e] + SH_TILE_ROWS - 1) / SH_TILE_ROWS;
    }
    s_off[d.E] = run; s_tile[d.E] = tiles_before;
    offsets[(size_t)grp * (d.E + 1) + d.E] = run;
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
      for (int j = 0; j < d.k; ++j) sel |= 1u << idx[o + j];           // (this thread's own entries)
    for (int e = 0; e < d.E; ++e) {
      const unsigned bal = __ballot_sync(0xffffffffu, (sel >> e) & 1u);
      if (lane == e) s_w[warp][e] = __popc(bal);
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
    for (int e = 0; e < d.E; ++e) {
      const unsigned bal = __ballot_sync(0xffffffffu, (sel >> e) & 1u);
      if ((sel >> e) & 1u) {
        const int pos = s_w[warp][e] + __popc(bal & ((1u << lane) - 1u));
        float gv = 0.f;
        for (int j = 0; j < d.k; ++j)
          if (idx[o + j] == e) gv = gate[o + j];
        ls[pos] = t;
        lg[pos] = gv;
      }
    }
    __syncthreads();
  }
}

// Gate gradients from list order into the matrix the projections' backward GEMMs contract with:
// dz[t, (side, h, e)] = ds s (1 - s) at the selected entries (the matrix is zero elsewhere).
static __global__ void __launch_bounds__(256)
sh_f32_dz_kernel(const float* __restrict__ ds, const int* __restrict__ lists, const float* __restrict__ lgate, const int* __restrict__ offsets,
                 float* __restrict__ dz, int ldz, ShDims d) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const long per = (long)d.N * d.k;
  const int grp = blockIdx.y;                              // (side, head)
  const long p = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= per) return;
  const int* off = offsets + (size_t)grp * (d.E + 1);
  int e = 0;
  while (e < d.E - 1 && off[e + 1] <= p) ++e;
  const size_t li = (size_t)grp * per + p;
  const float g = lgate[li];
  dz[(size_t)lists[li] * ldz + grp * d.E + e] = ds[li] * g * (1.f - g);
}
