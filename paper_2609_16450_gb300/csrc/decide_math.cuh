// Arithmetic shared by the decision kernels: GELU, warp sums and the merge of
// LM-head partial states.
#pragma once
#include <climits>

#include <cuda_runtime.h>

namespace ebd {
namespace {

__device__ __forceinline__ float gelu(float x) {
  return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f));
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ void merge_state(float& m, float& s, float& t, float& l2, int& idx,
                                            float bm, float bs, float bt, float bl2, int bidx) {
  if (bm > m || (bm == m && bidx < idx)) {
    float x;
    int xi;
    x = m; m = bm; bm = x;
    x = s; s = bs; bs = x;
    x = t; t = bt; bt = x;
    x = l2; l2 = bl2; bl2 = x;
    xi = idx; idx = bidx; bidx = xi;
  }
  l2 = fmaxf(l2, bm);
  if (bm == -INFINITY) return;
  const float dl = bm - m;
  const float sc = expf(dl);
  t = t + sc * (bt + dl * bs);
  s = s + sc * bs;
}

// The merge of a row's n <= 256 LM-head partial states (max, sum exp, sum
// exp (l - max), second largest; argmax) by one warp: the common maximum
// first, then every sum against it.  Empty states have max -inf.  All lanes
// return the result.
struct RowStats {
  float m, s, t, l2;
  int idx;
};
__device__ __forceinline__ RowStats merge_row(const float4* __restrict__ f, const int* __restrict__ ix, int n) {
  const int lane = threadIdx.x & 31;
  float4 v[8];
  int iv[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const int q = lane + 32 * c;
    v[c] = q < n ? f[q] : make_float4(-INFINITY, 0.f, 0.f, -INFINITY);
    iv[c] = q < n ? ix[q] : INT_MAX;
  }
  RowStats r;
  r.m = -INFINITY;
#pragma unroll
  for (int c = 0; c < 8; ++c) r.m = fmaxf(r.m, v[c].x);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) r.m = fmaxf(r.m, __shfl_xor_sync(0xffffffffu, r.m, o));
  r.idx = INT_MAX;
#pragma unroll
  for (int c = 0; c < 8; ++c)
    if (v[c].x == r.m) r.idx = min(r.idx, iv[c]);
  r.idx = __reduce_min_sync(0xffffffffu, r.idx);
  // second largest: the winner's own, or another state's maximum
  r.l2 = -INFINITY;
  r.s = r.t = 0.f;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    r.l2 = fmaxf(r.l2, v[c].x == r.m && iv[c] == r.idx ? v[c].w : v[c].x);
    if (v[c].x != -INFINITY) {
      const float d = v[c].x - r.m, e = expf(d);
      r.s = fmaf(e, v[c].y, r.s);
      r.t = fmaf(e, fmaf(d, v[c].y, v[c].z), r.t);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    r.l2 = fmaxf(r.l2, __shfl_xor_sync(0xffffffffu, r.l2, o));
    r.s += __shfl_xor_sync(0xffffffffu, r.s, o);
    r.t += __shfl_xor_sync(0xffffffffu, r.t, o);
  }
  return r;
}

}  // namespace
}  // namespace ebd
