// k_attn.cu -- scattered-query causal GQA attention over the paged cache of an fp32
// model, in fp32 arithmetic.
// Row i (position pos[i]) attends keys 0..pos[i] of its document's cache at
// `layer`; keys of repaired rows were written before this launch (so every
// row of the pass sees the fresh K/V of the others), all others are stale.
#include <math.h>

#include <type_traits>

#include "kvr_internal.cuh"

namespace kvr {
namespace {

struct SimtAttn {
  const float *q;
  const int32_t *pos;
  int M, H, G, gp, layer;  // gp: query slots per row and kv head (see below)
  const KVView *views;
  const int32_t *rowdoc;
  KVView single;
  float *out;
  float scale;
};

// A CTA takes NQ queries of one kv head -- consecutive (row, query head) slots,
// gp = H / G of them per row; with several documents gp is H / G rounded up to
// NQ, so that a CTA's queries are of one row -- and its warps deal out the keys
// in blocks of 32: four lanes score a key for every query (a key's row is read
// once for all of them, 64 bytes at a time), the softmax folds a block at a
// time, then the lanes split head_dim and add the block's values.  The warps'
// partial outputs are merged in warp order.  Latency-bound: 7 us for 36 rows over
// 240 keys, 17 for 512 rows.  (A lane per key, whose loads of one instruction lay
// on 32 lines, took 11 and 25; a warp per query that walked its keys one after
// another, a shuffle reduction and two exponentials each, 207 and 441.)
constexpr int AW = 8;  // warps per CTA
template <int VPL, int NQ>
__global__ void __launch_bounds__(32 * AW, NQ * VPL <= 8 ? 3 : 2) k_attn_simt(const SimtAttn p) {
  constexpr int DH = 32 * VPL;
  __shared__ float4 sq4[NQ * DH / 4];          // queries, scaled
  __shared__ float so[AW][NQ][DH];             // warps' outputs
  __shared__ float sm[AW][NQ], sl[AW][NQ];     // and their maxima and sums
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = blockIdx.y, grp = p.H / p.G;
  float *sq = (float *)sq4;
  int row[NQ], hh[NQ], lim[NQ], kmax = 0, kmin = 0x7fffffff;
#pragma unroll
  for (int a = 0; a < NQ; ++a) {
    const int i = blockIdx.x * NQ + a;
    row[a] = i / p.gp;
    hh[a] = i % p.gp;
    const bool real = row[a] < p.M && hh[a] < grp;
    lim[a] = real ? p.pos[row[a]] : -1;
    kmax = max(kmax, lim[a]);
    if (real) kmin = min(kmin, lim[a]);
  }
  if (row[0] >= p.M) return;
  const KVView v = p.views ? p.views[p.rowdoc[row[0]]] : p.single;
  const float *c = (const float *)v.pages;
  pdl_wait();
  for (int e = threadIdx.x; e < NQ * DH; e += 32 * AW) {
    const int i = blockIdx.x * NQ + e / DH, r = i / p.gp, h = i % p.gp;
    sq[e] = r < p.M && h < grp
                ? p.q[(size_t)r * p.H * DH + (size_t)(g * grp + h) * DH + e % DH] * p.scale
                : 0.f;
  }
  __syncthreads();
  float o[NQ][VPL], m[NQ], l[NQ];
#pragma unroll
  for (int a = 0; a < NQ; ++a) {
    m[a] = -INFINITY;
    l[a] = 0.f;  // this lane's keys
#pragma unroll
    for (int e = 0; e < VPL; ++e) o[a][e] = 0.f;
  }
  for (int b = warp; b <= kmax / 32; b += AW) {
    // a block lies in one page (its slots past the last key hold finite values)
    const float *kp = c + v.offset(p.layer, 0, g, 32 * b);
    const float *vp = c + v.offset(p.layer, 1, g, 32 * b);
    // four lanes a key, each with every fourth float4 of it; of eight keys at a
    // time, a lane keeps the sum of the one in the pass of its own number
    const int part = lane & 3, kr = lane >> 2, key = 32 * b + 8 * part + kr;
    const float4 *row4 = (const float4 *)(kp + (size_t)kr * DH) + part;
    float s[NQ], t[4][NQ];
#pragma unroll
    for (int k8 = 0; k8 < 4; ++k8)
#pragma unroll
      for (int a = 0; a < NQ; ++a) t[k8][a] = 0.f;
#pragma unroll(NQ == 1 ? 4 : 1)
    for (int d = 0; d < DH / 16; ++d) {
      float4 k[4];
#pragma unroll
      for (int k8 = 0; k8 < 4; ++k8) k[k8] = row4[8 * k8 * (DH / 4) + 4 * d];
#pragma unroll
      for (int a = 0; a < NQ; ++a) {
        const float4 x = sq4[a * (DH / 4) + 4 * d + part];
#pragma unroll
        for (int k8 = 0; k8 < 4; ++k8)
          t[k8][a] = fmaf(x.x, k[k8].x,
                          fmaf(x.y, k[k8].y, fmaf(x.z, k[k8].z, fmaf(x.w, k[k8].w, t[k8][a]))));
      }
    }
#pragma unroll
    for (int a = 0; a < NQ; ++a) {
#pragma unroll
      for (int k8 = 0; k8 < 4; ++k8) {
        t[k8][a] += __shfl_xor_sync(0xffffffffu, t[k8][a], 1);
        t[k8][a] += __shfl_xor_sync(0xffffffffu, t[k8][a], 2);
      }
      s[a] = part & 2 ? (part & 1 ? t[3][a] : t[2][a]) : (part & 1 ? t[1][a] : t[0][a]);
    }
#pragma unroll
    for (int a = 0; a < NQ; ++a) {
      if (key > lim[a]) s[a] = -INFINITY;
      float mx = s[a];
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      if (mx == -INFINITY) {  // no key of the block is this query's, or its scores are NaN
        s[a] = isnan(s[a]) ? s[a] : 0.f;
        l[a] += s[a];
        continue;
      }
      const float mn = fmaxf(m[a], mx), corr = expf(m[a] - mn);
      s[a] = expf(s[a] - mn);
      l[a] = l[a] * corr + s[a];
      m[a] = mn;
#pragma unroll
      for (int e = 0; e < VPL; ++e) o[a][e] *= corr;
    }
    // values; past the last key of a query they are not touched (they may be
    // another row's, and not finite)
    const bool whole = 32 * b + 31 <= kmin;
#pragma unroll 8
    for (int j = 0; j < 32; ++j) {
      using Vec = std::conditional_t<VPL == 4, float4, float2>;
      const Vec xv = *(const Vec *)(vp + (size_t)j * DH + lane * VPL);
      const float *x = (const float *)&xv;
#pragma unroll
      for (int a = 0; a < NQ; ++a) {
        const float w = __shfl_sync(0xffffffffu, s[a], (j & 7) * 4 + (j >> 3));
        if (whole || 32 * b + j <= lim[a])
#pragma unroll
          for (int e = 0; e < VPL; ++e) o[a][e] = fmaf(w, x[e], o[a][e]);
      }
    }
  }
#pragma unroll
  for (int a = 0; a < NQ; ++a) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) l[a] += __shfl_xor_sync(0xffffffffu, l[a], off);
    if (lane == 0) {
      sm[warp][a] = m[a];
      sl[warp][a] = l[a];
    }
#pragma unroll
    for (int e = 0; e < VPL; ++e) so[warp][a][lane * VPL + e] = o[a][e];
  }
  __syncthreads();
  for (int e = threadIdx.x; e < NQ * DH; e += 32 * AW) {
    const int a = e / DH, d = e % DH, i = blockIdx.x * NQ + a, r = i / p.gp, h = i % p.gp;
    if (r >= p.M || h >= grp) continue;
    float mx = sm[0][a];
#pragma unroll
    for (int w = 1; w < AW; ++w) mx = fmaxf(mx, sm[w][a]);
    float num = 0.f, den = 0.f;
#pragma unroll
    for (int w = 0; w < AW; ++w) {
      const float f = sm[w][a] == -INFINITY ? 0.f : expf(sm[w][a] - mx);
      num += f * so[w][a][d];
      den += f * sl[w][a];
    }
    const size_t at = (size_t)r * p.H * DH + (size_t)(g * grp + h) * DH + d;
    p.out[at] = num * (1.0f / den);
  }
}

template <int VPL>
void run(SimtAttn p, int num_sms, cudaStream_t s) {
  const int grp = p.H / p.G;
  // queries per CTA: as many as share the reads of a key while the CTAs still
  // fill the SMs (about twice over)
  const int fill = 2 * num_sms;
  auto go = [&](auto nq) {
    constexpr int NQ = decltype(nq)::value;
    p.gp = p.views ? (grp + NQ - 1) / NQ * NQ : grp;
    const long long slots = (long long)p.M * p.gp;
    launch_pdl(k_attn_simt<VPL, NQ>, dim3((unsigned)((slots + NQ - 1) / NQ), p.G), 32 * AW, 0, s,
               p);
  };
  const long long q = (long long)p.M * p.H;
  if (q >= 8 * fill && !(p.views && grp < 8))
    go(std::integral_constant<int, 8>{});
  else if (q >= 4 * fill && !(p.views && grp < 4))
    go(std::integral_constant<int, 4>{});
  else
    go(std::integral_constant<int, 1>{});
}

}  // namespace

void launch_attention_simt(const float *q, const int32_t *pos, int M, const Dims &dm, int layer,
                           const KVView *views, const int32_t *rowdoc, KVView single, float *out,
                           int num_sms, cudaStream_t s) {
  if (M <= 0) return;
  SimtAttn p{q,     pos,    M,      dm.H, dm.G, dm.H / dm.G,
             layer, views,  rowdoc, single, out, (float)(1.0 / sqrt((double)dm.dh))};
  if (dm.dh == 64)
    run<2>(p, num_sms, s);
  else
    run<4>(p, num_sms, s);
}

}  // namespace kvr
