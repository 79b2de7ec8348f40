// The EB decision of a step (App. E algorithm "Inference with LBS Block
// Selection and LPS Parallel Commit"; LBS, Sec. 5.1 and App. C.1; LPS,
// Sec. 5.2 and App. D.1; baseline rules, App. B Eq. prelim-update), one
// cluster of CTAs per sequence, the rows of a sequence split over the CTAs.
//
// Everything but attention and the selection is local to a row, so a CTA
// takes groups of 8 rows (the masked rows by rank) through whole LBS encoder
// layers on its own; the CTAs of a cluster meet only where attention needs
// every row's keys and values (once per layer) and before the selection:
// three cluster barriers.  Keys and values travel through an L2-resident
// scratch.  Windows of more than 64 rows take their LBS through three launches
// over the whole GPU instead (lbs_wide_kernel), ahead of the cluster.  The LPS
// router is small enough for a warp to take 8 rows of B n M through it in
// registers; its warps meet for the keys and values of its two attentions only.
//
// Products run on mma.sync (m16n8k16) with the weights as the M = 16 operand
// and the rows as N = 8.  The weights are bf16 values; an activation x is held
// as NP bf16 planes, x = x0 + x1 (+ x2), so that a product has the
// activation's ~16 (24) bits, and two activations multiply as the products of
// planes i, j with i + j < NP.  NP = 2 for windows of up to 64 rows, 3 (fp32
// accuracy) above.
#include <climits>

#include "decide_math.cuh"
#include "internal.h"
#include "ptx.cuh"
#include "rows_image.h"

namespace ebd {

namespace {

using namespace rowimg;

constexpr int kT = kRowsThreads;  // 256
constexpr int kNW = kT / 32;
constexpr int kVecs = V_POS;  // floats of the vectors staged in shared memory

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// byte stride of a row of K bf16: 64 mod 128, so that the 16-byte reads of
// two consecutive rows by 8 lanes fall in different banks
__device__ __host__ constexpr int row_bytes(int K) { return K == 32 ? 64 : 2 * K + 64; }

// groups of 8 rows of a window of up to kMaxSeqRows that a warp of a cluster of
// C CTAs takes through the LPS (C = 0: windows of up to 64 rows, one CTA)
__device__ __host__ constexpr int lps_groups(int C) {
  return C == 0 || C * kNW >= kMaxSeqRows / 8 ? 1 : kMaxSeqRows / 8 / (C * kNW);
}

template <int NR, int NP, int NG = 1>
struct Lay {  // shared memory, byte offsets
  static constexpr int R = 8 * NR;                  // rows of a CTA
  static constexpr int P128 = R * row_bytes(128);   // one plane of R rows x 128
  static constexpr int P256 = R * row_bytes(256);
  static constexpr int kLdF = 132;                  // fp32 row stride of F
  static constexpr int kLdO = 36;                   // partial attention output
  static constexpr int V = 0;                       // vectors of the image
  static constexpr int U = V + kVecs * 4;
  // LBS activations ...
  static constexpr int A = U;
  static constexpr int Y = A + NP * P128;
  static constexpr int Q = Y + NP * P128;
  static constexpr int H = Q + NP * P128;           // FFN hidden, or attention partials
  static constexpr int kPart = NR * kNW * 8 * kLdO * 4;
  static constexpr int kH = NP * P256 > kPart ? NP * P256 : kPart;
  static constexpr int ML = H + kH;                 // [NR][warp][8] (max, sum)
  static constexpr int F = ML + NR * kNW * 8 * 8;
  static constexpr int kLbsEnd = F + R * kLdF * 4;
  // ... and, once they are dead, the LPS weights and (windows of up to 64
  // rows) the keys and values of both blocks
  static constexpr int W = U;
  static constexpr int kLpsMat = 2 * MB_STRIDE;     // 16-byte units
  static constexpr int KV = W + kLpsMat * 16;
  static constexpr int kKvBlock = 64 * 64 * NP;     // elements of a block
  static constexpr int ST = KV + (NP == 2 ? 2 * kKvBlock * 2 : 0);   // a group's values between the parts
  static constexpr int GL = ST + NG * kNW * (16 + 4 * NP) * 32 * 4;  // LpsGlobal
  static constexpr int kLpsEnd = GL + 32;
  static constexpr int SLOT = kLbsEnd > kLpsEnd ? kLbsEnd : kLpsEnd;
  static constexpr int ROW = SLOT + 3 * 32 * 4;     // per-row arrays
};

// the rows of this CTA's groups
struct Slots {
  int mrow[32];   // window row of a masked-rank slot, -1: none
  float ent[32];
  int arg[32];
};

template <int CAP>
struct RowState {
  int pos[CAP];
  float conf[CAP];
  float prob[CAP];
  float feat[CAP][5];
  int bpos[CAP];
  int cnt[CAP / 32];
  int urow[CAP];  // unmasked rows whose statistics this CTA merges
  int cut, first, any, best, open;
};

__device__ __forceinline__ uint32_t pack2(float x, float y) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float lo_f(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float hi_f(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

__device__ __forceinline__ float rcp(float x) {  // at most 1 ulp off
  float y;
  asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// (x, y) as NP packed planes; every remainder is exact
template <int NP>
__device__ __forceinline__ void split2(float x, float y, uint32_t (&p)[NP]) {
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    p[i] = pack2(x, y);
    x -= lo_f(p[i]);
    y -= hi_f(p[i]);
  }
}

// stores columns (c, c + 1) of a row into NP planes
template <int NP>
__device__ __forceinline__ void put2(uint8_t* base, int plane, int rb, int row, int c, float x, float y) {
  uint32_t p[NP];
  split2<NP>(x, y, p);
#pragma unroll
  for (int i = 0; i < NP; ++i)
    *reinterpret_cast<uint32_t*>(base + i * plane + row * rb + 2 * c) = p[i];
}

// transpose of an 8 x 8 bf16 matrix, lane 4 g + t holding (row g, columns
// 2 t, 2 t + 1): turns a product's accumulators (output g, rows 2 t, 2 t + 1)
// into the next product's B fragment (row g, inputs 2 t, 2 t + 1)
__device__ __forceinline__ uint32_t trans8(uint32_t x) {
  uint32_t y;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
  return y;
}

__device__ __forceinline__ uint4 ld_w(const uint4* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// A fragments of the m16 tiles tile0 + 8 i of a matrix with K inputs
template <int K, int NT>
__device__ __forceinline__ void load_w(uint4 (&w)[NT * (K / 16)], const uint4* m, int tile0) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < NT; ++i)
#pragma unroll
    for (int ks = 0; ks < K / 16; ++ks)
      w[i * (K / 16) + ks] = ld_w(m + ((tile0 + 8 * i) * (K / 16) + ks) * 32 + lane);
}

__device__ __forceinline__ void mma4(float (&d)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  const uint32_t r[4] = {a.x, a.y, a.z, a.w};
  mma_bf16(d, r, b0, b1);
}

// acc[r][i]: outputs 16 tile_i + 2 g (elements 0, 1) and + 1 (2, 3) of rows
// 8 r + 2 t, 8 r + 2 t + 1 of A W^T, A in NP planes.  Each plane has its own
// accumulators, and dependent MMAs (31 cycles apart, one every 8 otherwise)
// stand as far apart as the tile allows; with NP = 3 they are added up in fp32 every 32 inputs,
// since the tensor cores truncate where they align a sum's terms.
template <int K, int NT, int NR, int NP>
__device__ __forceinline__ void gemm(const uint8_t* A, int plane, const uint4 (&w)[NT * (K / 16)], int nr,
                                     float (&acc)[NR][NT][4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  float al[NR][NT][NP - 1][4];
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int i = 0; i < NT; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        acc[r][i][e] = 0.f;
#pragma unroll
        for (int p = 0; p < NP - 1; ++p) al[r][i][p][e] = 0.f;
      }
#pragma unroll
  for (int kb = 0; kb < K / 32; ++kb)
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (NR > 1 && r >= nr) continue;
      uint4 x[NP];
#pragma unroll
      for (int p = 0; p < NP; ++p)
        x[p] = *reinterpret_cast<const uint4*>(A + p * plane + (8 * r + g) * row_bytes(K) + 64 * kb + 16 * t);
      float d[NT][4];
#pragma unroll
      for (int i = 0; i < NT; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) d[i][e] = NP == 3 ? 0.f : acc[r][i][e];
#pragma unroll
      for (int ks = 0; ks < 2; ++ks)
#pragma unroll
        for (int p = NP - 1; p >= 0; --p)
#pragma unroll
          for (int i = 0; i < NT; ++i)
            mma4(p > 0 ? al[r][i][p - 1] : d[i], w[i * (K / 16) + 2 * kb + ks], ks == 0 ? x[p].x : x[p].z,
                 ks == 0 ? x[p].y : x[p].w);
#pragma unroll
      for (int i = 0; i < NT; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[r][i][e] = NP == 3 ? acc[r][i][e] + d[i][e] : d[i][e];
    }
#pragma unroll
  for (int r = 0; r < NR; ++r)
#pragma unroll
    for (int i = 0; i < NT; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[r][i][e] += NP == 3 ? al[r][i][0][e] + al[r][i][NP - 2][e] : al[r][i][0][e];
}

// LayerNorm (eps 1e-5) of a warp's row of 32 * N values, lane holding
// columns lane * N .. + N
template <int N>
__device__ __forceinline__ void norm_row(float (&v)[N], const float* g, const float* b) {
  const int lane = threadIdx.x & 31;
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < N; ++i) s += v[i];
  const float mean = warp_sum(s) * (1.0f / (32 * N));
  float q = 0.f;
#pragma unroll
  for (int i = 0; i < N; ++i) q += (v[i] - mean) * (v[i] - mean);
  const float inv = rsqrtf(warp_sum(q) * (1.0f / (32 * N)) + 1e-5f);
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = (v[i] - mean) * inv * g[lane * N + i] + b[lane * N + i];
}

// Ranks of 0/1 flags over the rows j = 32 c + lane, chunk c = warp + 8 i:
// rank[i] = flags set before row j; returns the total.  All threads.
template <int CAP>
__device__ __forceinline__ int rank_rows(RowState<CAP>& rs, const bool* flag, int* rank) {
  constexpr int NC = CAP / 32, RPT = (NC + kNW - 1) / kNW;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t bal[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int c = warp + kNW * i;
    bal[i] = __ballot_sync(0xffffffffu, c < NC && flag[i]);
    if (lane == 0 && c < NC) rs.cnt[c] = __popc(bal[i]);
  }
  __syncthreads();
  int total = 0;
#pragma unroll
  for (int i = 0; i < RPT; ++i) rank[i] = __popc(bal[i] & ((1u << lane) - 1u));
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const int n = rs.cnt[c];
#pragma unroll
    for (int i = 0; i < RPT; ++i)
      if (c < warp + kNW * i) rank[i] += n;
    total += n;
  }
  __syncthreads();
  return total;
}

// reductions over the lanes of equal t (the 8 values of g)
__device__ __forceinline__ float gsum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 8);
  return v + __shfl_xor_sync(0xffffffffu, v, 16);
}
__device__ __forceinline__ float gmax(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 4));
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 16));
}

// One block's online softmax: s = scores (in log2 units) of TL tiles of 16
// keys (elements 0, 2: query 2 t; 1, 3: query 2 t + 1) becomes the probabilities against the
// updated running maxima m; returns the old values' factors in c.
template <int TL>
__device__ __forceinline__ void softmax_block(float (&s)[TL][4], float (&m)[2], float (&l)[2], float (&c)[2]) {
  float a0 = -INFINITY, a1 = -INFINITY;
#pragma unroll
  for (int j = 0; j < TL; ++j) {
    a0 = fmaxf(a0, fmaxf(s[j][0], s[j][2]));
    a1 = fmaxf(a1, fmaxf(s[j][1], s[j][3]));
  }
  const float n0 = fmaxf(m[0], gmax(a0)), n1 = fmaxf(m[1], gmax(a1));  // finite: a block holds a key
  c[0] = exp2f(m[0] - n0);
  c[1] = exp2f(m[1] - n1);
  m[0] = n0;
  m[1] = n1;
  float b0 = 0.f, b1 = 0.f;
#pragma unroll
  for (int j = 0; j < TL; ++j) {
    s[j][0] = exp2f(s[j][0] - n0);
    s[j][2] = exp2f(s[j][2] - n0);
    s[j][1] = exp2f(s[j][1] - n1);
    s[j][3] = exp2f(s[j][3] - n1);
    b0 += s[j][0] + s[j][2];
    b1 += s[j][1] + s[j][3];
  }
  l[0] = l[0] * c[0] + b0;
  l[1] = l[1] * c[1] + b1;
}

// LBS attention of this CTA's groups of 8 queries over n keys in blocks of
// 32, warp = (head, half of the blocks): running maximum and sum per warp,
// the unnormalised output to `part`, (max, sum) to `ml`.  Q (scaled) in
// planes in shared memory; Kp planes [key][128], Vp planes [dim][capk].
// Scores are K Q^T (keys as M), outputs V^T P^T.  Row r of key tile s of a
// block is key 8 (r / 2 % 4) + r % 2 + 2 (r / 8) + 4 s, so that lane t's keys
// of the second product are 8 consecutive ones.
template <int NR, int NP>
__device__ __forceinline__ void attend(const uint8_t* Q, const __nv_bfloat16* Kp, const __nv_bfloat16* Vp,
                                       size_t plane, int capk, int n, int nr, float* part, float* ml) {
  using L = Lay<NR, NP>;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int head = warp & 3, half = warp >> 2;
  const int n8 = (n + 7) & ~7;  // rows written
  float o[NR][2][4], m[NR][2], l[NR][2];
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    m[r][0] = m[r][1] = -INFINITY;
    l[r][0] = l[r][1] = 0.f;
#pragma unroll
    for (int d = 0; d < 2; ++d)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[r][d][e] = 0.f;
  }
  uint4 kf[2][2][NP];  // [tile][row half][plane]
  auto load_k = [&](int blk) {
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        int key = 32 * blk + 8 * (g >> 1) + (g & 1) + 2 * u + 4 * s;
        key = key < n8 ? key : 0;
#pragma unroll
        for (int p = 0; p < NP; ++p)
          kf[s][u][p] = __ldcg(reinterpret_cast<const uint4*>(Kp + p * plane + static_cast<size_t>(key) * 128 +
                                                              32 * head + 8 * t));
      }
  };
  if (32 * half < n) load_k(half);
  for (int blk = half; 32 * blk < n; blk += 2) {
    uint4 vf[2][2][NP];  // [dim tile][row half][plane]
    const bool vok = 32 * blk + 8 * t < n8;
#pragma unroll
    for (int d = 0; d < 2; ++d)
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int p = 0; p < NP; ++p)
          vf[d][u][p] = vok ? __ldcg(reinterpret_cast<const uint4*>(
                                  Vp + p * plane + static_cast<size_t>(32 * head + 16 * d + 2 * g + u) * capk +
                                  32 * blk + 8 * t))
                            : make_uint4(0u, 0u, 0u, 0u);
    uint32_t pb[NR][2][NP][2];
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (NR > 1 && r >= nr) continue;
      uint4 x[NP];
#pragma unroll
      for (int p = 0; p < NP; ++p)
        x[p] = *reinterpret_cast<const uint4*>(Q + p * L::P128 + (8 * r + g) * row_bytes(128) + 64 * head + 16 * t);
      float s[2][4], s1[2][4];
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) s[j][e] = s1[j][e] = 0.f;
#pragma unroll
      for (int sum = NP - 1; sum >= 0; --sum)
#pragma unroll
        for (int a = 0; a <= sum; ++a) {
          const uint4& q = x[sum - a];
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const uint4 &u = kf[j][0][a], &v = kf[j][1][a];
            mma4(s[j], make_uint4(u.x, v.x, u.y, v.y), q.x, q.y);
            mma4(s1[j], make_uint4(u.z, v.z, u.w, v.w), q.z, q.w);
          }
        }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
#pragma unroll
        for (int e = 0; e < 4; ++e) s[j][e] += s1[j][e];
        const int key = 32 * blk + 8 * (g >> 1) + (g & 1) + 4 * j;
        if (key >= n) s[j][0] = s[j][1] = -INFINITY;
        if (key + 2 >= n) s[j][2] = s[j][3] = -INFINITY;
      }
      float c[2];
      softmax_block<2>(s, m[r], l[r], c);
#pragma unroll
      for (int d = 0; d < 2; ++d)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[r][d][e] *= c[e & 1];
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          uint32_t q[NP];
          split2<NP>(s[j][2 * u], s[j][2 * u + 1], q);
#pragma unroll
          for (int p = 0; p < NP; ++p) pb[r][j][p][u] = trans8(q[p]);
        }
    }
    if (32 * (blk + 2) < n) load_k(blk + 2);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (NR > 1 && r >= nr) continue;
      float y[2][2][4];
#pragma unroll
      for (int d = 0; d < 2; ++d)
#pragma unroll
        for (int e = 0; e < 4; ++e) y[d][0][e] = y[d][1][e] = 0.f;
#pragma unroll
      for (int sum = NP - 1; sum >= 0; --sum)
#pragma unroll
        for (int a = 0; a <= sum; ++a)
#pragma unroll
          for (int d = 0; d < 2; ++d) {
            const uint4 &u = vf[d][0][a], &v = vf[d][1][a];
            mma4(y[d][0], make_uint4(u.x, v.x, u.y, v.y), pb[r][0][sum - a][0], pb[r][0][sum - a][1]);
            mma4(y[d][1], make_uint4(u.z, v.z, u.w, v.w), pb[r][1][sum - a][0], pb[r][1][sum - a][1]);
          }
#pragma unroll
      for (int d = 0; d < 2; ++d)
#pragma unroll
        for (int e = 0; e < 4; ++e) o[r][d][e] += y[d][0][e] + y[d][1][e];
    }
  }
#pragma unroll
  for (int r = 0; r < NR; ++r) {
    if (NR > 1 && r >= nr) continue;
    float* po = part + (r * kNW + warp) * 8 * L::kLdO;
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      *reinterpret_cast<float2*>(po + 2 * t * L::kLdO + 16 * d + 2 * g) = make_float2(o[r][d][0], o[r][d][2]);
      *reinterpret_cast<float2*>(po + (2 * t + 1) * L::kLdO + 16 * d + 2 * g) = make_float2(o[r][d][1], o[r][d][3]);
    }
    const float l0 = gsum(l[r][0]), l1 = gsum(l[r][1]);
    if (g == 0)
      *reinterpret_cast<float4*>(ml + (r * kNW + warp) * 16 + 4 * t) = make_float4(m[r][0], l0, m[r][1], l1);
  }
}

// The two halves' partial outputs merged and normalised, as NP planes of the
// concatenated heads.  All threads.
template <int NR, int NP>
__device__ __forceinline__ void attend_merge(const float* part, const float* ml, uint8_t* A, int nr) {
  using L = Lay<NR, NP>;
  for (int it = threadIdx.x; it < 8 * nr * 64; it += kT) {
    const int row = it >> 6, c = 2 * (it & 63), r = row >> 3, rr = row & 7, h = c >> 5, d = c & 31;
    const float2 u = *reinterpret_cast<const float2*>(ml + (r * kNW + h) * 16 + 2 * rr);
    const float2 v = *reinterpret_cast<const float2*>(ml + (r * kNW + 4 + h) * 16 + 2 * rr);
    const float M = fmaxf(u.x, v.x);
    const float e0 = exp2f(u.x - M), e1 = exp2f(v.x - M);  // an empty half has max -inf
    const float2 x = *reinterpret_cast<const float2*>(part + ((r * kNW + h) * 8 + rr) * L::kLdO + d);
    const float2 y = *reinterpret_cast<const float2*>(part + ((r * kNW + 4 + h) * 8 + rr) * L::kLdO + d);
    const float il = rcp(e0 * u.y + e1 * v.y);
    put2<NP>(A, L::P128, row_bytes(128), row, c, (e0 * x.x + e1 * y.x) * il, (e0 * x.y + e1 * y.y) * il);
  }
}

// ------------------------------------------------------------------ LBS
struct LbsArgs {
  const uint4* mat;
  const float* vec;
  const float* tok_table;
  __nv_bfloat16* kv;
  float* O;
  int V, gen_len, cap_rows, kbase, capk, nM;
  int nr, first, step;  // this CTA's groups of 8 masked rows: first, first + step, ..

  template <int NP>
  __device__ __forceinline__ __nv_bfloat16* keys(int l) const {
    return kv + (static_cast<size_t>(2 * l) * NP * cap_rows + kbase) * 128;
  }
  template <int NP>
  __device__ __forceinline__ __nv_bfloat16* values(int l) const {
    return kv + (static_cast<size_t>(2 * l + 1) * NP * cap_rows + kbase) * 128;
  }
};

// epi(row, column c, values of columns c, c + 1) over a product's outputs
template <class Epi>
__device__ __forceinline__ void each(const float (&a)[4], int r, int tile, Epi epi) {
  const int lane = threadIdx.x & 31, row = 8 * r + 2 * (lane & 3), c = 16 * tile + 2 * (lane >> 2);
  epi(row, c, a[0], a[2]);
  epi(row + 1, c, a[1], a[3]);
}
// F += a + bias
__device__ __forceinline__ void add_f(float* F, int ld, const float (&a)[4], int r, int tile, const float* bias) {
  each(a, r, tile, [&](int row, int c, float x, float y) {
    float2* z = reinterpret_cast<float2*>(F + row * ld + c);
    *z = make_float2(z->x + (x + bias[c]), z->y + (y + bias[c + 1]));
  });
}

// LBS input z (Eq. lbs_feat) of the CTA's rows: fp32 in F, planes in Y.  Not
// inlined, like the QKV product: run once on stand-in rows before the
// statistics are there, its instructions are on the SM when they are.
template <int NR, int NP>
__device__ __noinline__ void lbs_input(const LbsArgs a) {
  using L = Lay<NR, NP>;
  extern __shared__ __align__(16) uint8_t smem[];
  float* const F = reinterpret_cast<float*>(smem + L::F);
  const float* const sv = reinterpret_cast<const float*>(smem + L::V);
  const Slots& sl = *reinterpret_cast<const Slots*>(smem + L::SLOT);
  uint8_t* const sA = smem + L::A;
  uint8_t* const sY = smem + L::Y;
  constexpr int LDF = L::kLdF;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nr = a.nr;
  uint4 wc[8];
  // F_ent hidden, rows without a masked row as zeros
  for (int it = tid; it < 8 * nr * 32; it += kT) {
    const int row = it >> 5, c = 2 * (it & 31);
    const bool ok = sl.mrow[row] >= 0;
    const float h = ok ? sl.ent[row] : 0.f;
    // the token branch W_tok W_e[x_hat] + b (folded table): columns 64..127
    const int tok = ok ? sl.arg[row] : -1;
    float2 tv = make_float2(0.f, 0.f);
    if (tok >= 0 && tok < a.V)
      tv = __ldg(reinterpret_cast<const float2*>(a.tok_table + static_cast<size_t>(tok) * 64 + c));
    put2<NP>(sY, L::P128, row_bytes(64), row, c, gelu(fmaf(sv[V_ENT1W + c], h, sv[V_ENT1B + c])),
             gelu(fmaf(sv[V_ENT1W + c + 1], h, sv[V_ENT1B + c + 1])));
    put2<NP>(sA, L::P128, row_bytes(128), row, 64 + c, tv.x + sv[V_TOKB + c], tv.y + sv[V_TOKB + c + 1]);
  }
  {
    uint4 w[4];
    load_w<64, 1>(w, a.mat + M_ENT2, warp & 3);
    load_w<128, 1>(wc, a.mat + M_COMB, warp);
    __syncthreads();
    if (warp < 4) {
      float acc[NR][1][4];
      gemm<64, 1, NR, NP>(sY, L::P128, w, nr, acc);
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        if (r >= nr) continue;
        each(acc[r][0], r, warp, [&](int row, int c, float x, float y) {
          *reinterpret_cast<float2*>(F + row * LDF + c) = make_float2(x + sv[V_ENT2B + c], y + sv[V_ENT2B + c + 1]);
        });
      }
    }
  }
  __syncthreads();
  for (int row = warp; row < 8 * nr; row += kNW) {
    const float2 x = *reinterpret_cast<const float2*>(F + row * LDF + 2 * lane);
    float v[2] = {x.x, x.y};
    norm_row<2>(v, sv + V_ENTLNG, sv + V_ENTLNB);
    put2<NP>(sA, L::P128, row_bytes(128), row, 2 * lane, v[0], v[1]);
  }
  __syncthreads();
  {
    // fusion W_combine [e; t] + b + E_pos[rank]
    float acc[NR][1][4];
    gemm<128, 1, NR, NP>(sA, L::P128, wc, nr, acc);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (r >= nr) continue;
      each(acc[r][0], r, warp, [&](int row, int c, float x, float y) {
        const int k = 8 * (a.first + a.step * r) + (row & 7);
        float2 pe = make_float2(0.f, 0.f);
        if (k < a.gen_len)
          pe = __ldg(reinterpret_cast<const float2*>(a.vec + V_POS + static_cast<size_t>(k) * 128 + c));
        x += sv[V_COMBB + c] + pe.x;
        y += sv[V_COMBB + c + 1] + pe.y;
        *reinterpret_cast<float2*>(F + row * LDF + c) = make_float2(x, y);
        put2<NP>(sY, L::P128, row_bytes(128), row, c, x, y);
      });
    }
  }
}

// q, k and v of the CTA's rows in layer l: q (scaled) to planes in Q, k and v
// to the scratch
template <int NR, int NP>
__device__ __noinline__ void lbs_qkv(const LbsArgs a, int l) {
  using L = Lay<NR, NP>;
  extern __shared__ __align__(16) uint8_t smem[];
  const float* const sv = reinterpret_cast<const float*>(smem + L::V);
  uint8_t* const sY = smem + L::Y;
  uint8_t* const sQ = smem + L::Q;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, nr = a.nr;
  const size_t plane = static_cast<size_t>(a.cap_rows) * 128;  // elements of a K (V) plane
  const uint4* const wl = a.mat + M_LAYER + l * ML_STRIDE;
  const float* const vl = sv + V_LAYER + l * VL_STRIDE;
  __nv_bfloat16* const Kp = a.template keys<NP>(l);
  __nv_bfloat16* const Vp = a.template values<NP>(l);
  // QKV: tiles warp + 8 i, i = 0 the queries, 1 the keys, 2 the values
  constexpr int NQ = NR <= 2 ? 3 : 1;
#pragma unroll
  for (int i0 = 0; i0 < 3; i0 += NQ) {
    uint4 w[NQ * 8];
    load_w<128, NQ>(w, wl + ML_QKV, warp + 8 * i0);
    if (i0 == 0) __syncthreads();
    float acc[NR][NQ][4];
    gemm<128, NQ, NR, NP>(sY, L::P128, w, nr, acc);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (r >= nr) continue;
#pragma unroll
      for (int i = 0; i < NQ; ++i) {
        const int kind = i0 + i, c = 16 * warp + 2 * g, k = 8 * (a.first + a.step * r) + 2 * t;
        const float b0 = vl[VL_QKVB + 128 * kind + c], b1 = vl[VL_QKVB + 128 * kind + c + 1];
        const float x0 = acc[r][i][0] + b0, x1 = acc[r][i][1] + b0;  // column c of rows 2 t, 2 t + 1
        const float y0 = acc[r][i][2] + b1, y1 = acc[r][i][3] + b1;  // column c + 1
        if (kind == 0) {
          const float sc = 0.2550348616f;  // log2(e) / sqrt(32)
          put2<NP>(sQ, L::P128, row_bytes(128), 8 * r + 2 * t, c, x0 * sc, y0 * sc);
          put2<NP>(sQ, L::P128, row_bytes(128), 8 * r + 2 * t + 1, c, x1 * sc, y1 * sc);
        } else {
          uint32_t u[NP], v[NP];
          if (kind == 1) {
            split2<NP>(x0, y0, u);
            split2<NP>(x1, y1, v);
          } else {
            split2<NP>(x0, x1, u);
            split2<NP>(y0, y1, v);
          }
          __nv_bfloat16* const d0 =
              kind == 1 ? Kp + static_cast<size_t>(k) * 128 + c : Vp + static_cast<size_t>(c) * a.capk + k;
          const size_t step = kind == 1 ? 128 : a.capk;
#pragma unroll
          for (int q = 0; q < NP; ++q) {
            *reinterpret_cast<uint32_t*>(d0 + q * plane) = u[q];
            *reinterpret_cast<uint32_t*>(d0 + q * plane + step) = v[q];
          }
        }
      }
    }
  }
}

// the rest of layer l: attention, output projection, FFN; z of the next
// layer in F and Y, or the LBS logits
template <int NR, int NP>
__device__ __forceinline__ void lbs_layer(const LbsArgs& a, int l) {
  using L = Lay<NR, NP>;
  extern __shared__ __align__(16) uint8_t smem[];
  float* const F = reinterpret_cast<float*>(smem + L::F);
  const float* const sv = reinterpret_cast<const float*>(smem + L::V);
  uint8_t* const sA = smem + L::A;
  uint8_t* const sY = smem + L::Y;
  uint8_t* const sQ = smem + L::Q;
  uint8_t* const sH = smem + L::H;
  float* const part = reinterpret_cast<float*>(sH);
  float* const ml = reinterpret_cast<float*>(smem + L::ML);
  constexpr int LDF = L::kLdF;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nr = a.nr;
  const size_t plane = static_cast<size_t>(a.cap_rows) * 128;
  const uint4* const wl = a.mat + M_LAYER + l * ML_STRIDE;
  const float* const vl = sv + V_LAYER + l * VL_STRIDE;
  const __nv_bfloat16* const Kp = a.template keys<NP>(l);
  const __nv_bfloat16* const Vp = a.template values<NP>(l);
  attend<NR, NP>(sQ, Kp, Vp, plane, a.capk, a.nM, nr, part, ml);
  uint4 wo[8];
  load_w<128, 1>(wo, wl + ML_OUT, warp);
  __syncthreads();
  attend_merge<NR, NP>(part, ml, sA, nr);
  __syncthreads();
  {  // output projection + residual
    float acc[NR][1][4];
    gemm<128, 1, NR, NP>(sA, L::P128, wo, nr, acc);
#pragma unroll
    for (int r = 0; r < NR; ++r)
      if (r < nr) add_f(F, LDF, acc[r][0], r, warp, vl + VL_OUTB);
  }
  uint4 w1[16];
  load_w<128, 2>(w1, wl + ML_FF1, warp);
  __syncthreads();
  auto norm = [&](const float* gm, const float* bt) {
    for (int row = warp; row < 8 * nr; row += kNW) {
      float4* z = reinterpret_cast<float4*>(F + row * LDF) + lane;
      float v[4] = {z->x, z->y, z->z, z->w};
      norm_row<4>(v, gm, bt);
      *z = make_float4(v[0], v[1], v[2], v[3]);
      put2<NP>(sY, L::P128, row_bytes(128), row, 4 * lane, v[0], v[1]);
      put2<NP>(sY, L::P128, row_bytes(128), row, 4 * lane + 2, v[2], v[3]);
    }
  };
  norm(vl + VL_LN1G, vl + VL_LN1B);
  __syncthreads();
  {  // h = GELU(W_1 z + b_1)
    float acc[NR][2][4];
    gemm<128, 2, NR, NP>(sY, L::P128, w1, nr, acc);
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      if (r >= nr) continue;
#pragma unroll
      for (int i = 0; i < 2; ++i)
        each(acc[r][i], r, warp + 8 * i, [&](int row, int c, float x, float y) {
          put2<NP>(sH, L::P256, row_bytes(256), row, c, gelu(x + vl[VL_FF1B + c]), gelu(y + vl[VL_FF1B + c + 1]));
        });
    }
  }
  uint4 w2[16];
  load_w<256, 1>(w2, wl + ML_FF2, warp);
  __syncthreads();
  {
    float acc[NR][1][4];
    gemm<256, 1, NR, NP>(sH, L::P256, w2, nr, acc);
#pragma unroll
    for (int r = 0; r < NR; ++r)
      if (r < nr) add_f(F, LDF, acc[r][0], r, warp, vl + VL_FF2B);
  }
  __syncthreads();
  if (l == 0) {
    norm(vl + VL_LN2G, vl + VL_LN2B);
  } else {  // the last LayerNorm and the head O = w . z + b
    for (int row = warp; row < 8 * nr; row += kNW) {
      const float4 z = reinterpret_cast<const float4*>(F + row * LDF)[lane];
      float v[4] = {z.x, z.y, z.z, z.w};
      norm_row<4>(v, vl + VL_LN2G, vl + VL_LN2B);
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < 4; ++i) s = fmaf(v[i], sv[V_HEADW + 4 * lane + i], s);
      s = warp_sum(s) + sv[V_HEADB];
      const int k = 8 * (a.first + a.step * (row >> 3)) + (row & 7);
      if (lane == 0 && k < a.nM) a.O[a.kbase + k] = s;
    }
  }
}

// ------------------------------------------------------------------ LPS
// A warp's 8 rows: z[i], features 16 i + g (elements 0, 1: rows 2 t, 2 t + 1)
// and 16 i + 8 + g (2, 3).

// B fragments (rows as N) of T tiles of 16 features in NP planes
template <int T, int NP>
__device__ __forceinline__ void frags(const float (&v)[T][4], uint32_t (&f)[T][NP][2]) {
#pragma unroll
  for (int i = 0; i < T; ++i)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      uint32_t q[NP];
      split2<NP>(v[i][2 * u], v[i][2 * u + 1], q);
#pragma unroll
      for (int p = 0; p < NP; ++p) f[i][p][u] = trans8(q[p]);
    }
}

// y = W x + b for MT tiles of outputs, KT tiles of inputs; w: A fragments in
// shared memory
template <int MT, int KT, int NP>
__device__ __forceinline__ void lps_gemm(const uint4* w, const uint32_t (&f)[KT][NP][2], const float* b,
                                         float (&y)[MT][4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2;
  uint4 a[MT][KT];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int k = 0; k < KT; ++k) a[i][k] = w[(i * KT + k) * 32 + lane];
  float lo[MT][4], hi[MT][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) lo[i][e] = hi[i][e] = 0.f;
#pragma unroll
  for (int k = 0; k < KT; ++k)
#pragma unroll
    for (int p = NP - 1; p >= 0; --p)
#pragma unroll
      for (int i = 0; i < MT; ++i) mma4(p > 0 ? lo[i] : hi[i], a[i][k], f[k][p][0], f[k][p][1]);
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) y[i][e] = (hi[i][e] + lo[i][e]) + b[16 * i + g + 8 * (e >> 1)];
}

// LayerNorm over the 32 features of each row
__device__ __forceinline__ void lps_norm(const float (&z)[2][4], const float* gm, const float* bt, float (&y)[2][4]) {
  const int g = (threadIdx.x & 31) >> 2;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const float mean = gsum((z[0][c] + z[0][2 + c]) + (z[1][c] + z[1][2 + c])) * (1.0f / 32);
    float q = 0.f;
#pragma unroll
    for (int i = 0; i < 2; ++i) q += (z[i][c] - mean) * (z[i][c] - mean) + (z[i][2 + c] - mean) * (z[i][2 + c] - mean);
    const float inv = rsqrtf(gsum(q) * (1.0f / 32) + 1e-5f);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int u = 0; u < 2; ++u)
        y[i][2 * u + c] = (z[i][2 * u + c] - mean) * inv * gm[16 * i + 8 * u + g] + bt[16 * i + 8 * u + g];
  }
}

// a lane's words of a key (or of a pair of keys' values): [head][plane]
template <int NP, bool GLOBAL>
__device__ __forceinline__ void ld_kv(const __nv_bfloat16* p, uint32_t (&w)[4 * NP]) {
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    const uint4* q = reinterpret_cast<const uint4*>(p) + i;
    const uint4 v = GLOBAL ? __ldcg(q) : *q;
    w[4 * i] = v.x;
    w[4 * i + 1] = v.y;
    w[4 * i + 2] = v.z;
    w[4 * i + 3] = v.w;
  }
}

// The LPS router of one sequence's B n M, 8 rows per warp, in three parts that
// hand a warp's values over in shared memory (ST): z, the queries, the
// attention output.  They are not inlined, so that each part's instructions
// can be brought in by a warp of its own, on stand-in rows, while the
// statistics are not there yet: with the code out of L2 as well (a step on
// buffers of its own, after other work), one warp running through all of it
// took 45k cycles, 29k of them after the LM head had ended; the parts side by
// side end before it.  (One function whose parts are skipped by branches ran
// 1.5 times as long.)
// C: CTAs of the cluster that share the rows, 0 where one CTA has them all.  Keys
// and values of both blocks at kv + block * kv_stride (C = 0: in shared memory):
// K [key][dim pair][head][plane][2 dims] and, v_off further, V [key
// pair][dim][head][plane][2 keys], so that a lane reads all heads and planes of
// its key (pair) in NP 16-byte loads.
struct LpsGlobal {  // (C > 0; itself in shared memory, for all warps)
  __nv_bfloat16* kv;
  size_t kv_stride, v_off;
  float* prob;  // by rank in B n M
};
template <int NP>
constexpr int kLpsWords = 8 + 4 * NP + 8;  // z, queries, attention output
// a lane's words of them: of the warp's only group, or of group grp = rank +
// C * (warp + kNW * pass)
template <class L, int NP, int C>
__device__ __forceinline__ float* lps_values(uint8_t* smem, int grp) {
  const int slot = C > 0 ? grp / C : static_cast<int>(threadIdx.x >> 5);
  return reinterpret_cast<float*>(smem + L::ST) + slot * kLpsWords<NP> * 32 + (threadIdx.x & 31);
}

// Linear(5 -> 32), LayerNorm, GELU (block 0); LN1, QKV
template <int CAP, int NR, int NP, int C>
__device__ __noinline__ void lps_qkv(int nb, int grp, int l) {
  using L = Lay<NR, NP, lps_groups(C)>;
  extern __shared__ __align__(16) uint8_t smem[];
  const float* const sv = reinterpret_cast<const float*>(smem + L::V);
  RowState<CAP>& rs = *reinterpret_cast<RowState<CAP>*>(smem + L::ROW);
  float* const st = lps_values<L, NP, C>(smem, grp);
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const uint4* const wl = reinterpret_cast<const uint4*>(smem + L::W) + l * MB_STRIDE;
  const float* const vl = sv + V_BLOCK + l * VB_STRIDE;
  const LpsGlobal& gl = *reinterpret_cast<const LpsGlobal*>(smem + L::GL);
  __nv_bfloat16* const K =
      C > 0 ? gl.kv + l * gl.kv_stride : reinterpret_cast<__nv_bfloat16*>(smem + L::KV) + l * L::kKvBlock;
  __nv_bfloat16* const V = K + (C > 0 ? gl.v_off : L::kKvBlock / 2);
  float z[2][4];
  if (l == 0) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int row = 8 * grp + 2 * t + (e & 1), f = 16 * i + 8 * (e >> 1) + g;
        float y = sv[V_INB + f];
#pragma unroll
        for (int k = 0; k < 5; ++k) y = fmaf(row < nb ? rs.feat[row][k] : 0.f, sv[V_INT + 32 * k + f], y);
        z[i][e] = y;
      }
    lps_norm(z, sv + V_INLNG, sv + V_INLNB, z);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) z[i][e] = gelu(z[i][e]);
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) z[i >> 2][i & 3] = st[32 * i];
  }
  uint32_t qf[4][NP];  // queries of each head: dims 2 t, 2 t + 1 of row g
  float y[2][4], q[6][4];
  uint32_t f[2][NP][2];
  lps_norm(z, vl + VB_LN1G, vl + VB_LN1B, y);
  frags<2, NP>(y, f);
  lps_gemm<6, 2, NP>(wl + MB_QKV, f, vl + VB_QKVB, q);
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    const int i = h >> 1, u = 2 * (h & 1);
    const float sc = 0.5100697233f;  // log2(e) / sqrt(8)
    uint32_t qp[NP], kp[NP], vp[NP];
    split2<NP>(q[i][u] * sc, q[i][u + 1] * sc, qp);
    split2<NP>(q[2 + i][u], q[2 + i][u + 1], kp);
    split2<NP>(q[4 + i][u], q[4 + i][u + 1], vp);
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      qf[h][p] = trans8(qp[p]);
      *reinterpret_cast<uint32_t*>(K + (((8 * grp + g) * 4 + t) * (4 * NP) + h * NP + p) * 2) = trans8(kp[p]);
      *reinterpret_cast<uint32_t*>(V + (((4 * grp + t) * 8 + g) * (4 * NP) + h * NP + p) * 2) = vp[p];
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) st[32 * i] = z[i >> 2][i & 3];
#pragma unroll
  for (int h = 0; h < 4; ++h)
#pragma unroll
    for (int p = 0; p < NP; ++p) st[32 * (8 + h * NP + p)] = __uint_as_float(qf[h][p]);
}

// softmax(q k^T / sqrt(8)) v
template <int CAP, int NR, int NP, int C>
__device__ __noinline__ void lps_attend(int nb, int grp, int l) {
  using L = Lay<NR, NP, lps_groups(C)>;
  extern __shared__ __align__(16) uint8_t smem[];
  float* const st = lps_values<L, NP, C>(smem, grp);
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const LpsGlobal& gl = *reinterpret_cast<const LpsGlobal*>(smem + L::GL);
  const __nv_bfloat16* const K =
      C > 0 ? gl.kv + l * gl.kv_stride : reinterpret_cast<const __nv_bfloat16*>(smem + L::KV) + l * L::kKvBlock;
  const __nv_bfloat16* const V = K + (C > 0 ? gl.v_off : L::kKvBlock / 2);
  uint32_t qf[4][NP];
#pragma unroll
  for (int h = 0; h < 4; ++h)
#pragma unroll
    for (int p = 0; p < NP; ++p) qf[h][p] = __float_as_uint(st[32 * (8 + h * NP + p)]);
  // the four heads side by side: each block's chain of two products, a
  // maximum, exponentials and transposes is latency
  const int n8 = (nb + 7) & ~7;
  float o[4][4], m[4][2], sum[4][2];
#pragma unroll
  for (int h = 0; h < 4; ++h) {
#pragma unroll
    for (int e = 0; e < 4; ++e) o[h][e] = 0.f;
    m[h][0] = m[h][1] = -INFINITY;
    sum[h][0] = sum[h][1] = 0.f;
  }
#pragma unroll 1
  for (int k0 = 0; k0 < nb; k0 += 32) {
    float s[4][2][4], c[4][2], y[4][4];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int key = k0 + 16 * j + g;
      uint32_t k0w[4 * NP], k1w[4 * NP];  // keys key, key + 8: dims 2 t, 2 t + 1
      ld_kv<NP, (C > 0)>(K + ((key < n8 ? key : 0) * 4 + t) * (8 * NP), k0w);
      ld_kv<NP, (C > 0)>(K + ((key + 8 < n8 ? key + 8 : 0) * 4 + t) * (8 * NP), k1w);
#pragma unroll
      for (int h = 0; h < 4; ++h)
#pragma unroll
        for (int e = 0; e < 4; ++e) s[h][j][e] = 0.f;
      // 8 dims fill half a k16 step: two products of planes per MMA
#pragma unroll
      for (int part = NP == 3 ? 0 : 1; part < 3; ++part)
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const uint32_t *u = k0w + h * NP, *v = k1w + h * NP;
          if (part == 0)
            mma4(s[h][j], make_uint4(u[NP - 1], v[NP - 1], u[0], v[0]), qf[h][0], qf[h][NP - 1]);
          else if (part == 1 && NP == 3)
            mma4(s[h][j], make_uint4(u[1], v[1], u[1], v[1]), qf[h][0], qf[h][1]);
          else if (part == 1)
            mma4(s[h][j], make_uint4(u[1], v[1], 0u, 0u), qf[h][0], 0u);
          else
            mma4(s[h][j], make_uint4(u[0], v[0], u[0], v[0]), qf[h][0], qf[h][1]);
        }
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        if (key >= nb) s[h][j][0] = s[h][j][1] = -INFINITY;
        if (key + 8 >= nb) s[h][j][2] = s[h][j][3] = -INFINITY;
      }
    }
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      softmax_block<2>(s[h], m[h], sum[h], c[h]);
#pragma unroll
      for (int e = 0; e < 4; ++e) y[h][e] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      uint32_t va[2][4 * NP];  // keys 16 j + 8 u + 2 t, + 1: dim g
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int key = k0 + 16 * j + 8 * u;
        ld_kv<NP, (C > 0)>(V + (((key < n8 ? key : 0) / 2 + t) * 8 + g) * (8 * NP), va[u]);
        if (key >= n8)
#pragma unroll
          for (int i = 0; i < 4 * NP; ++i) va[u][i] = 0u;
      }
      uint32_t pb[4][NP][2];
#pragma unroll
      for (int h = 0; h < 4; ++h)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          uint32_t q[NP];
          split2<NP>(s[h][j][2 * u], s[h][j][2 * u + 1], q);
#pragma unroll
          for (int p = 0; p < NP; ++p) pb[h][p][u] = trans8(q[p]);
        }
      // 8 dims fill half of M: planes 0 and 1 of the values on top of each other
#pragma unroll
      for (int p = NP == 3 ? NP : NP - 1; p >= 0; --p)
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const uint32_t *v0 = va[0] + h * NP, *v1 = va[1] + h * NP;
          if (p == NP)
            mma4(y[h], make_uint4(v0[NP - 1], 0u, v1[NP - 1], 0u), pb[h][0][0], pb[h][0][1]);
          else
            mma4(y[h], make_uint4(v0[0], v0[1], v1[0], v1[1]), pb[h][p][0], pb[h][p][1]);
        }
    }
#pragma unroll
    for (int h = 0; h < 4; ++h)
#pragma unroll
      for (int e = 0; e < 4; ++e) o[h][e] = fmaf(o[h][e], c[h][e & 1], y[h][e]);
  }
  float x[2][4];  // heads concatenated
#pragma unroll
  for (int h = 0; h < 4; ++h) {
    x[h >> 1][2 * (h & 1)] = (o[h][0] + o[h][2]) * rcp(gsum(sum[h][0]));
    x[h >> 1][2 * (h & 1) + 1] = (o[h][1] + o[h][3]) * rcp(gsum(sum[h][1]));
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) st[32 * (8 + 4 * NP + i)] = x[i >> 2][i & 3];
}

// output projection, LN2, FFN; after block 1 the head and p_psi
template <int CAP, int NR, int NP, int C>
__device__ __noinline__ void lps_ffn(int nb, int grp, int l) {
  using L = Lay<NR, NP, lps_groups(C)>;
  extern __shared__ __align__(16) uint8_t smem[];
  const float* const sv = reinterpret_cast<const float*>(smem + L::V);
  RowState<CAP>& rs = *reinterpret_cast<RowState<CAP>*>(smem + L::ROW);
  float* const st = lps_values<L, NP, C>(smem, grp);
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const uint4* const wl = reinterpret_cast<const uint4*>(smem + L::W) + l * MB_STRIDE;
  const float* const vl = sv + V_BLOCK + l * VB_STRIDE;
  float z[2][4], x[2][4];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    z[i >> 2][i & 3] = st[32 * i];
    x[i >> 2][i & 3] = st[32 * (8 + 4 * NP + i)];
  }
  float hd[4][4];
  float y[2][4];
  uint32_t f[2][NP][2];
  frags<2, NP>(x, f);
  lps_gemm<2, 2, NP>(wl + MB_OUT, f, vl + VB_OUTB, y);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) z[i][e] += y[i][e];
  lps_norm(z, vl + VB_LN2G, vl + VB_LN2B, y);
  frags<2, NP>(y, f);
  lps_gemm<4, 2, NP>(wl + MB_FF1, f, vl + VB_FF1B, hd);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) hd[i][e] = gelu(hd[i][e]);
  uint32_t fh[4][NP][2];
  frags<4, NP>(hd, fh);
  lps_gemm<2, 4, NP>(wl + MB_FF2, fh, vl + VB_FF2B, y);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) z[i][e] += y[i][e];
#pragma unroll
  for (int i = 0; i < 8; ++i) st[32 * i] = z[i >> 2][i & 3];
  if (l == 1) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      float s = 0.f;
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int u = 0; u < 2; ++u) s = fmaf(z[i][2 * u + c], sv[V_PHEADW + 16 * i + 8 * u + g], s);
      s = gsum(s) + sv[V_PHEADB];
      const int row = 8 * grp + 2 * t + c;
      float* const prob = C > 0 ? reinterpret_cast<const LpsGlobal*>(smem + L::GL)->prob : rs.prob;
      if (g == 0 && row < nb) prob[row] = 1.0f / (1.0f + expf(-s));
    }
  }
}

// Groups of 8 rows of the nb, the warp's first and every C * kNW-th one from
// there; meet(): every warp of the sequence sees the others' keys and values
template <int CAP, int NR, int NP, int C, class Meet>
__device__ __forceinline__ void lps_router(int nb, int first, Meet meet) {
  constexpr int NG = lps_groups(C);
#pragma unroll 1
  for (int l = 0; l < 2; ++l) {
#pragma unroll 1
    for (int i = 0, grp = first; i < NG && 8 * grp < nb; ++i, grp += C * kNW) lps_qkv<CAP, NR, NP, C>(nb, grp, l);
    meet();
#pragma unroll 1
    for (int i = 0, grp = first; i < NG && 8 * grp < nb; ++i, grp += C * kNW) {
      lps_attend<CAP, NR, NP, C>(nb, grp, l);
      lps_ffn<CAP, NR, NP, C>(nb, grp, l);
    }
  }
}

// The statistics of step row r, merged by a warp from the LM head's partial
// states, to the scratch and the caller's outputs; lane 0 returns H~ and the
// argmax in `ent` and `arg`.  With `real` false no states are merged and the
// result goes to the scratch's spare row.
__device__ __forceinline__ void merge_one(const RowsParams& p, int r, bool real, float& ent, int& arg) {
  const size_t base = static_cast<size_t>(r) * p.grid_lm;
  const RowStats st = merge_row(p.part_f + base, p.part_i + base, real ? p.grid_lm : 0);
  if ((threadIdx.x & 31) != 0) return;
  const int sr = real ? r : p.spare_row;
  const float conf = 1.0f / st.s, h = logf(st.s) - st.t * conf, entn = h * p.inv_log_v;
  const float gap = (1.0f - expf(st.l2 - st.m)) * conf;
  const bool bad = !(isfinite(st.m) && isfinite(st.s) && isfinite(st.t) && st.s >= 1.0f) || st.idx < 0 ||
                   st.idx >= p.V;
  ent = entn;
  arg = bad ? -1 : st.idx;
  p.s_conf[sr] = conf;
  p.s_ent[sr] = entn;
  p.s_gap[sr] = gap;
  p.s_arg[sr] = arg;
  if (real) {
    if (p.conf) p.conf[r] = conf;
    if (p.entropy) p.entropy[r] = h;
    if (p.ent_norm) p.ent_norm[r] = entn;
    if (p.gap) p.gap[r] = gap;
    if (p.argmax) p.argmax[r] = arg;
    if (bad) atomicCAS(p.status, 0, EBD_ERR_NONFINITE);
  }
}

// The statistics of the CTA's rows: its groups' slots, then its share of the
// unmasked rows, a row per warp.  Waits for the grid before this one first.
// With `warm` each warp starts with a pass that merges no states (before the
// wait).
template <int CAP>
__device__ __forceinline__ void merge_rows(const RowsParams& p, Slots& sl, const RowState<CAP>& rs, int r0, int nr,
                                           int nu, bool warm) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  bool waited = false;
  for (int it = warm && nr + nu > 0 ? warp - kNW : warp; it < 8 * nr + nu; it += kNW) {
    const bool real = it >= 0;
    if (real && !waited) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      waited = true;
    }
    const int j = !real ? 0 : it < 8 * nr ? sl.mrow[it] : rs.urow[it - 8 * nr];
    if (j < 0 || (real && !in_bounds(r0 + j, p.R, p.status))) continue;
    float ent = 0.f;
    int arg = -1;
    merge_one(p, r0 + j, real, ent, arg);
    if (lane == 0 && real && it < 8 * nr) {
      sl.ent[it] = ent;
      sl.arg[it] = arg;
    }
  }
  if (!waited) asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace

// The statistics and the LBS of windows of more than 64 rows, ahead of the
// decision's kernel: a CTA per group of 8 masked rows (grid: groups, sequences)
// over the whole GPU, one launch per stretch between two attentions, rows and
// queries handed on through the scratch.
//   PART 0: statistics; LBS input, QKV of layer 0
//   PART 1: layer 0, QKV of layer 1      PART 2: layer 1, LBS logits
// Bound by the chain of dependent phases of a CTA.  With the LBS in the
// cluster's 16 CTAs, four groups each, an attention over 384 keys took 39k
// cycles: the unrolled loop over a CTA's groups left the instruction caches, on
// 16 SMs of 152.  ebd_decide, 384 masked rows of 512: 105 us so, 62 here; eight
// such sequences 152.
template <int PART>
__global__ void __launch_bounds__(kT, 1) lbs_wide_kernel(const RowsParams p) {
  constexpr int NP = 3, CAP = kMaxSeqRows;
  using L = Lay<1, NP>;
  constexpr int RPT = CAP / kT;
  extern __shared__ __align__(16) uint8_t smem[];
  float* const sv = reinterpret_cast<float*>(smem + L::V);
  float* const F = reinterpret_cast<float*>(smem + L::F);
  RowState<CAP>& rs = *reinterpret_cast<RowState<CAP>*>(smem + L::ROW);
  Slots& sl = *reinterpret_cast<Slots*>(smem + L::SLOT);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int b = blockIdx.y, wk = blockIdx.x, nw = gridDim.x;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  for (int i = tid; i < kVecs / 4; i += kT)
    reinterpret_cast<float4*>(sv)[i] = __ldg(reinterpret_cast<const float4*>(p.vec) + i);
  const int r0 = p.cu_rows[b];
  int n = p.cu_rows[b + 1] - r0;
  if (n < 0 || n > CAP || r0 < 0 || r0 + n > p.R || n > p.gen_len) n = 0;  // reported by the decision
  const int kbase = scratch_row(r0, b), capk = (n + 7) & ~7;
  bool m[RPT], f[RPT];
  int mrank[RPT], urank[RPT];
  if (PART == 0 && tid < 32) {
    sl.mrow[tid] = -1;
    sl.ent[tid] = 0.f;
    sl.arg[tid] = -1;
  }
  int nM = 0, nU = 0;
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int j = 32 * (warp + kNW * i) + lane;
    m[i] = j < n && p.mask[r0 + j] != 0;
    f[i] = j < n && !m[i];
    if (PART != 0) nM += __syncthreads_count(m[i]);
  }
  if (PART == 0) {
    nM = rank_rows<CAP>(rs, m, mrank);
    nU = rank_rows<CAP>(rs, f, urank);
  }
  const bool run_lbs = p.mode == EBD_DECODE_EB && p.blk_meta[2 * b + 1] == 0 && nM > p.l_min;
  const int groups = (nM + 7) >> 3;
  const int nr = wk < groups ? 1 : 0;
  const LbsArgs la{p.mat, p.vec, p.tok_table, p.kv, p.O, p.V, p.gen_len, p.cap_rows, kbase, capk, nM, nr, wk, nw};
  float* const zg = p.z + static_cast<size_t>(kbase + 8 * wk) * 128;
  uint8_t* const qg = reinterpret_cast<uint8_t*>(p.q + static_cast<size_t>(kbase + 8 * wk) * 128);
  const size_t qplane = static_cast<size_t>(p.cap_rows) * 256;  // bytes
  if (PART == 0) {
    // as in the cluster: the rows without a group go to the CTAs without one
    const int u0 = groups < nw ? groups : 0, nuw = nw - u0;
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int j = 32 * (warp + kNW * i) + lane;
      if (m[i] && (mrank[i] >> 3) == wk) sl.mrow[mrank[i] & 7] = j;
      if (f[i] && u0 + urank[i] % nuw == wk) rs.urow[urank[i] / nuw] = j;
    }
    const int nu = wk >= u0 && nU > wk - u0 ? (nU - (wk - u0) + nuw - 1) / nuw : 0;
    __syncthreads();
    if (p.features_in) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      if (tid < 8 && sl.mrow[tid] >= 0) {
        sl.ent[tid] = p.s_ent[r0 + sl.mrow[tid]];
        sl.arg[tid] = p.s_arg[r0 + sl.mrow[tid]];
      }
    } else {
      merge_rows<CAP>(p, sl, rs, r0, nr, nu, false);
      // Statistics are every row's, also of a rejected sequence and of the
      // rows before the first offset and past the last: from each offset up
      // to the next, 0 and R in place of the first and the last, the spans
      // that run forward hold every row.
      const int lo = b == 0 ? 0 : min(max(r0, 0), p.R);
      const int hi = b == p.B - 1 ? p.R : min(max(p.cu_rows[b + 1], 0), p.R);
      for (int i = wk * kNW + warp; i < hi - lo - n; i += nw * kNW) {
        const int r = lo + i < r0 ? lo + i : lo + i + n;
        float ent;
        int arg;
        merge_one(p, r, true, ent, arg);
      }
    }
    __syncthreads();
    if (!run_lbs || nr == 0) return;
    lbs_input<1, NP>(la);
  } else {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (!run_lbs || nr == 0) return;
    for (int i = tid; i < 8 * 32; i += kT)
      reinterpret_cast<float4*>(F + (i >> 5) * L::kLdF)[i & 31] = __ldcg(reinterpret_cast<const float4*>(zg) + i);
    for (int i = tid; i < NP * 8 * 16; i += kT) {
      const int pl = i >> 7, row = (i >> 4) & 7, c = i & 15;
      *reinterpret_cast<uint4*>(smem + L::Q + pl * L::P128 + row * row_bytes(128) + 16 * c) =
          __ldcg(reinterpret_cast<const uint4*>(qg + pl * qplane + row * 256) + c);
    }
    __syncthreads();
    lbs_layer<1, NP>(la, PART - 1);
    if (PART == 2) return;
  }
  lbs_qkv<1, NP>(la, PART);
  __syncthreads();
  for (int i = tid; i < 8 * 32; i += kT)
    reinterpret_cast<float4*>(zg)[i] = reinterpret_cast<const float4*>(F + (i >> 5) * L::kLdF)[i & 31];
  for (int i = tid; i < NP * 8 * 16; i += kT) {
    const int pl = i >> 7, row = (i >> 4) & 7, c = i & 15;
    reinterpret_cast<uint4*>(qg + pl * qplane + row * 256)[c] =
        *reinterpret_cast<const uint4*>(smem + L::Q + pl * L::P128 + row * row_bytes(128) + 16 * c);
  }
}

// RULE: the baselines' rules (Reading R20) on statistics that are there, which
// use no router: one CTA per sequence without the cluster's meetings, weights
// and activations.  ebd_decide under the threshold rule with a copy of its
// state, us in a graph, here / the 8-CTA cluster / the kernels before it: 1 x 64
// rows 3.4 / 5.1 / 7.0, 16 x 32 4.2 / 5.5 / 6.4, 64 x 64 3.9 / 5.6 / 28; 1 x 512
// 4.2 / - / 14.4.  Call by call the host's launches bound it, 16 to 17 us.
template <int C, int NR, int NP, int CAP, bool RULE = false>
__global__ void __launch_bounds__(kT, 1) decide_rows_kernel(const RowsParams p) {
  // windows of more than 64 rows: the LBS and the statistics come from
  // lbs_wide_kernel
  constexpr bool kWide = CAP > 64;
  using L = Lay<NR, NP, kWide ? lps_groups(C) : 1>;
  static_assert(L::ROW % 16 == 0, "vector reads of RowState");
  static_assert(kWide || RULE || CAP == 8 * NR * C, "rows of the cluster's groups");
  constexpr int NC = CAP / 32, RPT = (NC + kNW - 1) / kNW;
  extern __shared__ __align__(16) uint8_t smem[];
  float* const sv = reinterpret_cast<float*>(smem + L::V);
  RowState<CAP>& rs = *reinterpret_cast<RowState<CAP>*>(smem + (RULE ? 0 : L::ROW));
  Slots& sl = *reinterpret_cast<Slots*>(smem + L::SLOT);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int b = blockIdx.x / C;
  // the window attention, which shares no data with the decision, may start
  // on the SMs this grid leaves free once every CTA of it is resident
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // (asked anew at each use: held in a register, which the kernels of 252 lack,
  // 64 x 64 rows take 52.4 us instead of 51.4)
  auto eb = [&]() { return !RULE && p.mode == EBD_DECODE_EB; };
  if (eb())  // the baselines' rules use no router
    for (int i = tid; i < kVecs / 4; i += kT)
      reinterpret_cast<float4*>(sv)[i] = __ldg(reinterpret_cast<const float4*>(p.vec) + i);

  // ------------------------------------------------------------ decode state
  const int r0 = p.cu_rows[b];
  int n = p.cu_rows[b + 1] - r0;
  const bool bad_seq = n < 0 || n > (RULE ? p.cap : CAP) || r0 < 0 || r0 + n > p.R ||
                       (p.strict ? p.cu_rows[p.B] != p.R : n > p.gen_len);
  if (bad_seq) {
    if (rank == 0 && tid == 0) atomicCAS(p.status, 0, EBD_ERR_INVALID_ARG);
    n = 0;
  }
  const int kbase = scratch_row(r0, b), capk = (n + 7) & ~7;  // this sequence's rows of the scratch
  int meta_b = p.blk_meta[2 * b], meta_s = p.blk_meta[2 * b + 1];
  bool m[RPT], inb[RPT], f[RPT];
  int pos[RPT], mrank[RPT], urank[RPT];
  if (!RULE && tid < 32) {
    sl.mrow[tid] = -1;
    sl.ent[tid] = 0.f;
    sl.arg[tid] = -1;
  }
  if (tid == 0) {
    rs.cut = INT_MAX;
    rs.first = INT_MAX;
    rs.any = 0;
    rs.best = -1;
    rs.open = 0;
  }
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int j = 32 * (warp + kNW * i) + lane;
    const bool row = j < n;
    m[i] = row && p.mask[r0 + j] != 0;
    inb[i] = row && p.in_block[r0 + j] != 0;
    pos[i] = row ? p.row_pos[r0 + j] : 0;
    if (row) rs.pos[j] = pos[i];
    f[i] = row && !m[i];
  }
  const int nM = rank_rows<CAP>(rs, m, mrank);
  const int nU = kWide || RULE ? 0 : rank_rows<CAP>(rs, f, urank);
  const bool run_lbs = eb() && meta_s == 0 && nM > p.l_min;
  auto copy_lps = [&]() {
    for (int i = tid; i < L::kLpsMat; i += kT)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem + L::W + 16 * i)),
                   "l"(p.mat + M_BLOCK + i)
                   : "memory");
  };
  if constexpr (RULE) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
  } else if constexpr (kWide) {
    if (p.lps_enabled) copy_lps();
    // the statistics and the LBS logits of every row
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
  } else {
    // Windows of up to 64 rows: CTA 0 makes the decision.  Eight CTAs with a
    // group to spare leave all rows to the other seven, so that CTA 0 can bring
    // in the LPS and its weights meanwhile.
    const int groups = (nM + 7) >> 3;
    const bool apart = C == 8 && groups < C;
    const int nw = apart ? C - 1 : C, wk = apart ? rank - 1 : rank;
    // group k of 8 rows of M belongs to worker k % nw, its slot k / nw; the
    // statistics of the other rows are merged by the workers without a group
    const int u0 = groups < nw ? groups : 0, nuw = nw - u0;
    if (wk >= 0) {
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const int j = 32 * (warp + kNW * i) + lane, grp = mrank[i] >> 3;
        if (m[i] && grp % nw == wk) sl.mrow[8 * (grp / nw) + (mrank[i] & 7)] = j;
        if (f[i] && u0 + urank[i] % nuw == wk) rs.urow[urank[i] / nuw] = j;
      }
    }
    const int nr = wk >= 0 && groups > wk ? (groups - wk + nw - 1) / nw : 0;  // groups of this CTA
    const int nu = wk >= u0 && nU > wk - u0 ? (nU - (wk - u0) + nuw - 1) / nuw : 0;
    const LbsArgs la{p.mat, p.vec, p.tok_table, p.kv, p.O, p.V, p.gen_len, p.cap_rows, kbase, capk, nM, nr, wk, nw};
    __syncthreads();

    // The LM head has streamed its weight through L2: bring the router's back
    // while its last CTAs run.
    if (b == 0 && eb()) {
      const char* w = reinterpret_cast<const char*>(p.mat);
      for (int i = (run_lbs ? 0 : M_BLOCK / 8) + rank * kT + tid; i < M_TOTAL / 8; i += C * kT)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(w + 128 * static_cast<size_t>(i)));
    }
    // Launched behind the LM head, this grid waits some microseconds for its
    // last CTAs, with code that no SM has cached (a first pass through it costs
    // about as much again as the work itself, with the code out of L2 as well
    // several times as much): meanwhile CTA 0 runs the LPS router, one part
    // per warp, the others the LBS input layers and the first QKV product, on
    // stand-in rows.
    const bool warm = p.warm != 0 && C == 8 && eb();
    if (apart && rank == 0 && p.lps_enabled) {
      copy_lps();
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
      if (warm) {
        if (warp % 3 == 0)
          lps_qkv<CAP, NR, NP, 0>(64, warp, 0);
        else if (warp % 3 == 1)
          lps_attend<CAP, NR, NP, 0>(64, warp, 0);
        else
          lps_ffn<CAP, NR, NP, 0>(64, warp, 0);
      }
    } else if (warm && run_lbs && nr > 0) {
      lbs_input<NR, NP>(la);
      lbs_qkv<NR, NP>(la, 0);
    }

    // ------------------------------------------------------------ statistics
    // everything above overlaps the LM head's last CTAs; the partial states
    // are read only after its grid completed.  A masked row is merged by the
    // CTA that holds it in the LBS, the others are spread over the cluster.
    if (p.features_in) {
      asm volatile("griddepcontrol.wait;" ::: "memory");
      if (tid < 8 * NR && sl.mrow[tid] >= 0) {
        sl.ent[tid] = p.s_ent[r0 + sl.mrow[tid]];
        sl.arg[tid] = p.s_arg[r0 + sl.mrow[tid]];
      }
    } else {
      merge_rows<CAP>(p, sl, rs, r0, nr, nu, warm);
    }
    __syncthreads();

    // ------------------------------------------------------------ LBS
    if (run_lbs) {
      if (nr > 0) lbs_input<NR, NP>(la);
#pragma unroll 1
      for (int l = 0; l < 2; ++l) {
        if (nr > 0) lbs_qkv<NR, NP>(la, l);
        cluster_barrier();  // every row's keys and values (l = 0: and statistics) are visible
        if (nr > 0) lbs_layer<NR, NP>(la, l);
      }
    }
    cluster_barrier();  // every row's statistics and LBS logit are visible

    if (rank != 0) return;
    if (!apart && p.lps_enabled) copy_lps();  // behind the selection, over the dead LBS activations
  }

  // ------------------------------------------------------------ block selection
  // (Readings R8, R9)
  float conf[RPT], ent[RPT], gap[RPT], lbs[RPT];
  int arg[RPT], brank[RPT];
  bool bad[RPT], sel[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int j = 32 * (warp + kNW * i) + lane, r = r0 + j;
    conf[i] = ent[i] = gap[i] = 0.f;
    arg[i] = -1;
    bad[i] = false;
    lbs[i] = __int_as_float(0x7fc00000);
    if (j < n) {
      conf[i] = __ldcg(p.s_conf + r);
      ent[i] = __ldcg(p.s_ent + r);
      gap[i] = __ldcg(p.s_gap + r);
      arg[i] = __ldcg(p.s_arg + r);
      bad[i] = !(isfinite(conf[i]) && isfinite(ent[i]) && isfinite(gap[i])) || arg[i] < 0 || arg[i] >= p.V;
      if (run_lbs && m[i]) lbs[i] = __ldcg(p.O + kbase + mrank[i]);
    }
  }
  if (!eb()) {
#pragma unroll
    for (int i = 0; i < RPT; ++i) sel[i] = 32 * (warp + kNW * i) + lane < n;  // the window is the block
  } else if (meta_s != 0) {
#pragma unroll
    for (int i = 0; i < RPT; ++i) sel[i] = inb[i];
  } else {
    int nB = nM;
    if (nM <= p.l_min) {
#pragma unroll
      for (int i = 0; i < RPT; ++i) sel[i] = m[i];
    } else {
      bool cand[RPT];
      int cr[RPT];
#pragma unroll
      for (int i = 0; i < RPT; ++i) cand[i] = m[i] && lbs[i] > 0.f && arg[i] != p.eos_id && !bad[i];
      const int nC = rank_rows<CAP>(rs, cand, cr);
#pragma unroll
      for (int i = 0; i < RPT; ++i)
        if (cand[i]) rs.bpos[cr[i]] = pos[i];
      __syncthreads();
      // MaxGapFilter: cut at the first candidate farther than g_max from its predecessor
#pragma unroll
      for (int i = 0; i < RPT; ++i)
        if (cand[i] && cr[i] >= 1 && pos[i] - rs.bpos[cr[i] - 1] > p.g_max) atomicMin(&rs.cut, cr[i]);
      __syncthreads();
      nB = min(rs.cut, nC);
#pragma unroll
      for (int i = 0; i < RPT; ++i) sel[i] = cand[i] && cr[i] < nB;
      if (nB < p.l_min) {  // min-tokens fallback: the first min(L_B, |M|) masked rows
        nB = nM < p.l_b ? nM : p.l_b;
#pragma unroll
        for (int i = 0; i < RPT; ++i) sel[i] = m[i] && mrank[i] < nB;
      }
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i)
      if (sel[i]) atomicMin(&rs.first, 32 * (warp + kNW * i) + lane);
    __syncthreads();
    if (nB > 0) {
      meta_b = rs.pos[rs.first];
      meta_s = nB;
    }
  }
#pragma unroll
  for (int i = 0; i < RPT; ++i) f[i] = sel[i] && m[i] && !bad[i];
  const int nBM = rank_rows<CAP>(rs, f, brank);
  const bool run_lps = eb() && p.lps_enabled && nBM > 0;

  // ------------------------------------------------------------ LPS
  if (!RULE && run_lps) {
    const float rho = static_cast<float>(nBM) / static_cast<float>(meta_s);
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      if (!f[i]) continue;
      float* ft = rs.feat[brank[i]];
      ft[0] = conf[i];
      ft[1] = ent[i];
      ft[2] = gap[i];
      ft[3] = rho;
      ft[4] = static_cast<float>(pos[i] - meta_b) / static_cast<float>(meta_s);
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    if constexpr (RULE) {
    } else if constexpr (kWide) {
      if (tid == 0)
        *reinterpret_cast<LpsGlobal*>(smem + L::GL) =
            LpsGlobal{p.kvp + static_cast<size_t>(kbase) * 64 * NP, static_cast<size_t>(p.cap_rows) * 64 * NP,
                      static_cast<size_t>(capk) * 32 * NP, p.P + kbase};
      __syncthreads();
      lps_router<CAP, NR, NP, C>(nBM, rank + C * warp, [] { cluster_barrier(); });
      cluster_barrier();  // every row's p_psi is visible
    } else {
      lps_router<CAP, NR, NP, 0>(nBM, warp, [] { __syncthreads(); });
    }
  } else if (kWide && !RULE) {
    // Rank 0 commits in place over the decode state that every CTA has read:
    // with no LPS, whose meetings stand between the two, they meet here.
    cluster_barrier();
  }
  if (!RULE) asm volatile("cp.async.wait_all;" ::: "memory");
  if (rank != 0 || bad_seq) return;

  // ------------------------------------------------------------ accept, commit
  // union accept (Reading R14), anti-stall fallback, parallel commit, block
  // resolution; the baselines' rules (Reading R20) in their modes
  float prob[RPT];
  bool acc[RPT];
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    prob[i] = __int_as_float(0x7fc00000);
    acc[i] = false;
    if (!f[i]) continue;
    if (run_lps && kWide) prob[i] = __ldcg(p.P + kbase + brank[i]);
    rs.conf[brank[i]] = conf[i];
    rs.bpos[brank[i]] = pos[i];
  }
  if (RULE && tid < 3 && nBM + tid < CAP) rs.conf[nBM + tid] = -INFINITY;  // up to whole groups of four
  __syncthreads();
  // Top-m: rows ahead, of higher kappa, or of equal kappa and lower position.
  // Where a thread has two rows, both against four at a time: 1 x 512 rows 44
  // -> 32 us in a graph (33.5 with a thread per row in the kernels before).  The
  // routers' kernels keep the short loop: this one made them 1 to 5 % slower.
  int ahead[RPT];
  if (RULE && p.mode == EBD_DECODE_TOPM) {
#pragma unroll
    for (int i = 0; i < RPT; ++i) ahead[i] = 0;
    for (int k = 0; k < nBM; k += 4) {
      const float4 c = *reinterpret_cast<const float4*>(rs.conf + k);
      const int4 q = *reinterpret_cast<const int4*>(rs.bpos + k);
      auto before = [&](float cc, int qq, int i) { return cc > conf[i] || (cc == conf[i] && qq < pos[i]) ? 1 : 0; };
#pragma unroll
      for (int i = 0; i < RPT; ++i)
        ahead[i] += before(c.x, q.x, i) + before(c.y, q.y, i) + before(c.z, q.z, i) + before(c.w, q.w, i);
    }
  }
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    if (!f[i]) continue;
    if (run_lps && !kWide) prob[i] = rs.prob[brank[i]];
    if (p.mode == EBD_DECODE_TOPM) {
      if (!RULE) {
        ahead[i] = 0;
        for (int k = 0; k < nBM; ++k)
          ahead[i] += (rs.conf[k] > conf[i] || (rs.conf[k] == conf[i] && rs.bpos[k] < pos[i])) ? 1 : 0;
      }
      acc[i] = ahead[i] < p.top_m;
    } else {
      acc[i] = conf[i] >= p.tau || prob[i] > p.tau_psi;  // NaN where the LPS did not run
    }
    if (acc[i]) rs.any = 1;
  }
  __syncthreads();
  if (!rs.any && nBM > 0) {  // anti-stall: the highest kappa, lowest position on ties
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      if (!f[i]) continue;
      bool best = true;
      for (int k = 0; k < nBM; ++k)
        if (rs.conf[k] > conf[i] || (rs.conf[k] == conf[i] && rs.bpos[k] < pos[i])) best = false;
      if (best) rs.best = brank[i];
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < RPT; ++i) acc[i] = f[i] && brank[i] == rs.best;
  }
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    m[i] = m[i] && !acc[i];
    if (!eb()) sel[i] = inb[i];  // no block state
    if (sel[i] && m[i]) rs.open = 1;
  }
  __syncthreads();
  const bool resolve = eb() && meta_s > 0 && !rs.open;
#pragma unroll
  for (int i = 0; i < RPT; ++i) {
    const int j = 32 * (warp + kNW * i) + lane, r = r0 + j;
    if (j >= n || !in_bounds(r, p.R, p.status)) continue;
    p.tokens_out[r] = acc[i] ? arg[i] : p.tokens[r];
    p.mask_out[r] = m[i] ? 1 : 0;
    p.in_block_out[r] = (sel[i] && !resolve) ? 1 : 0;
    if (p.accepted) p.accepted[r] = acc[i] ? 1 : 0;
    if (p.lbs_logit) p.lbs_logit[r] = lbs[i];
    if (p.lps_prob) p.lps_prob[r] = prob[i];
  }
  if (tid == 0) {
    if (resolve) meta_b = meta_s = 0;
    p.blk_meta_out[2 * b] = meta_b;
    p.blk_meta_out[2 * b + 1] = meta_s;
  }
}

namespace {
template <int C, int NR, int NP>
constexpr int rows_cap() {
  return NP == 3 ? kMaxSeqRows : 8 * NR * C;
}
template <int C, int NR, int NP>
constexpr int smem_bytes() {
  return Lay<NR, NP, NP == 3 ? lps_groups(C) : 1>::ROW + static_cast<int>(sizeof(RowState<rows_cap<C, NR, NP>()>));
}
constexpr int kWideSmem = Lay<1, 3>::ROW + static_cast<int>(sizeof(RowState<kMaxSeqRows>));

template <int C, int NR, int NP>
cudaError_t configure_one() {
  const auto k = decide_rows_kernel<C, NR, NP, rows_cap<C, NR, NP>()>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_bytes<C, NR, NP>());
  if (e == cudaSuccess && C > 8) e = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}
template <int C, int NR, int NP>
cudaError_t launch_one(const RowsParams& p, cudaStream_t st, bool pdl, int* slots) {
  const auto k = decide_rows_kernel<C, NR, NP, rows_cap<C, NR, NP>()>;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(slots != nullptr ? C : p.B * C));
  cfg.blockDim = dim3(kT);
  cfg.dynamicSmemBytes = smem_bytes<C, NR, NP>();
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = C;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  if (slots != nullptr) return cudaOccupancyMaxActiveClusters(slots, k, &cfg);
  return cudaLaunchKernelEx(&cfg, k, p);
}
template <int CAP>
cudaError_t launch_rule(const RowsParams& p, cudaStream_t st, bool pdl) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(p.B));
  cfg.blockDim = dim3(kT);
  cfg.dynamicSmemBytes = sizeof(RowState<CAP>);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  static_assert(sizeof(RowState<CAP>) <= 48 * 1024, "dynamic shared memory without an attribute");
  return cudaLaunchKernelEx(&cfg, decide_rows_kernel<1, 1, 2, CAP, true>, p);
}
cudaError_t launch_wide(void (*k)(RowsParams), const RowsParams& p, int groups, cudaStream_t st, bool pdl) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(static_cast<unsigned>(groups), static_cast<unsigned>(p.B));
  cfg.blockDim = dim3(kT);
  cfg.dynamicSmemBytes = kWideSmem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, p);
}
}  // namespace

cudaError_t decide_rows_configure(DecideSlots& n) {
  cudaError_t e;
  const RowsParams none{};
  const cudaFuncAttribute smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
  if ((e = configure_one<8, 1, 2>()) != cudaSuccess || (e = configure_one<4, 2, 2>()) != cudaSuccess ||
      (e = configure_one<2, 4, 2>()) != cudaSuccess || (e = configure_one<4, 1, 2>()) != cudaSuccess ||
      (e = configure_one<2, 2, 2>()) != cudaSuccess || (e = configure_one<1, 4, 2>()) != cudaSuccess ||
      (e = configure_one<16, 1, 3>()) != cudaSuccess || (e = configure_one<8, 1, 3>()) != cudaSuccess ||
      (e = configure_one<4, 1, 3>()) != cudaSuccess || (e = configure_one<2, 1, 3>()) != cudaSuccess ||
      (e = cudaFuncSetAttribute(lbs_wide_kernel<0>, smem, kWideSmem)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(lbs_wide_kernel<1>, smem, kWideSmem)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(lbs_wide_kernel<2>, smem, kWideSmem)) != cudaSuccess ||
      (e = launch_one<8, 1, 2>(none, nullptr, false, &n.c8)) != cudaSuccess ||
      (e = launch_one<4, 2, 2>(none, nullptr, false, &n.c4)) != cudaSuccess ||
      (e = launch_one<16, 1, 3>(none, nullptr, false, &n.wide16)) != cudaSuccess ||
      (e = launch_one<8, 1, 3>(none, nullptr, false, &n.wide8)) != cudaSuccess ||
      (e = launch_one<4, 1, 3>(none, nullptr, false, &n.wide4)) != cudaSuccess)
    return e;
  return cudaSuccess;
}

// CTAs per sequence: as many as leave all sequences resident at once
// (ebd_decide, us, 8 CTAs of one group / 4 of two / 2 of four: 8 x 64 rows 35
// / 42 / 55, 16 x 64 49 / 41 / 55, 36 x 64 68 / 43 / 53, 40 x 64 68 / 66 / 53).
// Windows of up to 32 rows, 4 of one / 2 of two / 1 of four: 16 x 32 33 / 41 /
// 53, 40 x 32 48 / 40 / 52, 128 x 32 98 / 73 / 54, with the same limits, which
// are those of the larger kernels above.
// Windows of more than 64 rows, 16 CTAs / 8 / 4 (two passes over the LPS rows of
// a 512-row window) / 2 (four), LBS and LPS: 1 x 512 77 / 78 / 100 / 129, 8 x 512
// 168 / 151 / 172 / 200, 16 x 128 125 / 102 / 87 / 89, 60 x 65 319 / 227 / 188 /
// 169; inside a block 1 x 512 25.0 / 25.1 / 25.4 / 26.7, 8 x 512 54 / 39 / 39 /
// 40, 32 x 128 134 / 100 / 70 / 70, 60 x 65 234 / 155 / 122 / 106.  (16 CTAs
// whatever the batch were slower inside a block than the chain of grid-wide
// kernels before them, 32 x 128 107 us, 60 x 65 127.)
cudaError_t launch_decide_rows(const RowsParams& p, const DecideSlots& n, cudaStream_t st, bool pdl) {
  if (p.B <= 0 || p.R <= 0) return cudaSuccess;
  const bool eb = p.mode == EBD_DECODE_EB;
  if (p.cap > 64) {
    cudaError_t e = cudaSuccess;
    // a sequence may bring more rows than announced, up to all of the step's
    const int most = p.gen_len < p.R ? p.gen_len : p.R, groups = ((most < kMaxSeqRows ? most : kMaxSeqRows) + 7) / 8;
    if (eb || !p.features_in) {
      if ((e = launch_wide(lbs_wide_kernel<0>, p, groups, st, pdl)) != cudaSuccess) return e;
      pdl = true;
    }
    if (!eb) return launch_rule<kMaxSeqRows>(p, st, pdl);
    if ((e = launch_wide(lbs_wide_kernel<1>, p, groups, st, true)) != cudaSuccess ||
        (e = launch_wide(lbs_wide_kernel<2>, p, groups, st, true)) != cudaSuccess)
      return e;
    if (p.B <= n.wide16) return launch_one<16, 1, 3>(p, st, pdl, nullptr);
    if (p.B <= n.wide8) return launch_one<8, 1, 3>(p, st, pdl, nullptr);
    return p.B <= n.wide4 ? launch_one<4, 1, 3>(p, st, pdl, nullptr) : launch_one<2, 1, 3>(p, st, pdl, nullptr);
  }
  if (!eb && p.features_in) return launch_rule<64>(p, st, pdl);
  if (p.cap > 32) {
    if (p.B <= n.c8) return launch_one<8, 1, 2>(p, st, pdl, nullptr);
    return p.B <= n.c4 ? launch_one<4, 2, 2>(p, st, pdl, nullptr) : launch_one<2, 4, 2>(p, st, pdl, nullptr);
  }
  if (p.B <= n.c4) return launch_one<4, 1, 2>(p, st, pdl, nullptr);
  return p.B <= 2 * n.c4 ? launch_one<2, 2, 2>(p, st, pdl, nullptr) : launch_one<1, 4, 2>(p, st, pdl, nullptr);
}

}  // namespace ebd
