// k_gemm_simt.cu -- FFMA GEMM Y[M][N] (+)= X[M][K] W[N][K]^T (+ bias), or SwiGLU of
// interleaved gate/up rows, fp32 accumulation.  Serves the fp32 model (whose 1e-4
// parity rules out TF32 tensor cores) and shapes the tensor-core GEMM does not
// take.
#include <type_traits>

#include "kvr_internal.cuh"

namespace kvr {
namespace {

__device__ __forceinline__ float4 ld4(const float *p) { return *(const float4 *)p; }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16 *p) {
  const uint2 u = *(const uint2 *)p;
  const float2 a = __bfloat1622float2(*(const __nv_bfloat162 *)&u.x);
  const float2 b = __bfloat1622float2(*(const __nv_bfloat162 *)&u.y);
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void put(float *p, float v) { *p = v; }
__device__ __forceinline__ void put(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }

struct SimtGemm {
  const void *X, *W;
  const float *bias;
  float *Y;
  void *act;  // SwiGLU output [M][N / 2], model dtype (null: Y)
  int M, N, K, ldx, ldy, accumulate;
};

// 256 threads in KS groups: each group owns the whole BM x BN tile, 4 x 4 outputs a
// thread, and every KS-th part of each K chunk; the groups' sums meet in
// shared memory in group order.  Both operands are staged row by row, K
// contiguous (rows KC + 4 floats apart, so that eight threads' float4s fall
// on different banks), two chunks deep with the next one's loads in flight
// during the products.  A thread reads 8 float4s for 64 products.
//
// Rows and features are few where this matters (a 36-row pass of the 256-wide
// model: 4 to 22 tiles of 64 x 64, each CTA walking all of K with nothing in
// flight: 28 to 60 us a projection), so the tile shrinks until the tiles
// fill the SMs and the K groups take its place.
constexpr int NTH = 256;
template <typename T, int BM, int BN, int KS, int KC>
__global__ void __launch_bounds__(NTH) k_gemm_simt(const SimtGemm p) {
  constexpr int TX = BN / 4, TY = BM / 4;       // threads of a group along N and M
  static_assert(TX * TY * KS == NTH, "one 4 x 4 block per thread and group");
  constexpr int LD = KC + 4;
  constexpr int NX = BM * KC / 4 / NTH, NW = BN * KC / 4 / NTH;  // float4s per thread and chunk
  static_assert(NX * NTH * 4 == BM * KC && NW * NTH * 4 == BN * KC, "even staging");
  constexpr int KG = KC / KS;                   // a group's part of a chunk
  extern __shared__ float4 smem4[];
  float *const sm = (float *)smem4;             // [2][BM + BN][LD], then [KS][BM][BN]
  pdl_trigger();
  const int tid = threadIdx.x, grp = tid / (TX * TY), tx = tid % TX, ty = tid / TX % TY;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const T *X = (const T *)p.X, *W = (const T *)p.W;
  float4 rx[NX], rw[NW];
  // K is a multiple of 4 (d_model, head_dim and ffn are)
  auto load_x = [&](int k0) {
#pragma unroll
    for (int i = 0; i < NX; ++i) {
      const int e = tid + i * NTH, r = m0 + e / (KC / 4), k = k0 + e % (KC / 4) * 4;
      rx[i] = r < p.M && k < p.K ? ld4(X + (size_t)r * p.ldx + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto load_w = [&](int k0) {
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      const int e = tid + i * NTH, r = n0 + e / (KC / 4), k = k0 + e % (KC / 4) * 4;
      rw[i] = r < p.N && k < p.K ? ld4(W + (size_t)r * p.K + k) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto stage = [&](int b) {
    float *d = sm + b * (BM + BN) * LD;
#pragma unroll
    for (int i = 0; i < NX; ++i) {
      const int e = tid + i * NTH;
      *(float4 *)(d + e / (KC / 4) * LD + e % (KC / 4) * 4) = rx[i];
    }
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      const int e = tid + i * NTH;
      *(float4 *)(d + (BM + e / (KC / 4)) * LD + e % (KC / 4) * 4) = rw[i];
    }
  };
  load_w(0);  // weights do not depend on the previous kernel
  pdl_wait();
  load_x(0);
  stage(0);
  __syncthreads();
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  const int chunks = (p.K + KC - 1) / KC;
  for (int c = 0; c < chunks; ++c) {
    if (c + 1 < chunks) {
      load_w((c + 1) * KC);
      load_x((c + 1) * KC);
    }
    const float *xs = sm + (c & 1) * (BM + BN) * LD + ty * LD + grp * KG;
    const float *ws = sm + (c & 1) * (BM + BN) * LD + (BM + tx) * LD + grp * KG;
#pragma unroll 4
    for (int k = 0; k < KG; k += 4) {
      float4 a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = *(const float4 *)(xs + i * TY * LD + k);
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = *(const float4 *)(ws + j * TX * LD + k);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          acc[i][j] = fmaf(
              a[i].x, b[j].x,
              fmaf(a[i].y, b[j].y, fmaf(a[i].z, b[j].z, fmaf(a[i].w, b[j].w, acc[i][j]))));
    }
    if (c + 1 < chunks) {
      stage((c + 1) & 1);
      __syncthreads();
    }
  }
  // one output, given its complete sum; gate and up of a feature are 16 apart
  auto out = [&](int m, int n, float v) {
    if (m >= p.M || n >= p.N) return;
    v += p.bias ? p.bias[n] : 0.f;
    float *y = p.Y + (size_t)m * p.ldy + n;
    *y = p.accumulate ? *y + v : v;
  };
  auto out_act = [&](int m, int n, float gate, float up) {  // n: the gate row
    if (m >= p.M || n >= p.N) return;
    put((T *)p.act + (size_t)m * (p.N / 2) + n / 32 * 16 + n % 16,
        gate / (1.0f + expf(-gate)) * up);
  };
  if constexpr (KS == 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int m = m0 + ty + i * TY;
      if (p.act) {  // j = 0, 2: gate rows; TX = 16
#pragma unroll
        for (int j = 0; j < 4; j += 2) out_act(m, n0 + tx + j * TX, acc[i][j], acc[i][j + 1]);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) out(m, n0 + tx + j * TX, acc[i][j]);
      }
    }
  } else {
    __syncthreads();  // the chunks are consumed
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        sm[(grp * BM + ty + i * TY) * BN + tx + j * TX] = acc[i][j];
    __syncthreads();
    auto sum = [&](int m, int n) {
      float v = sm[m * BN + n];
#pragma unroll
      for (int q = 1; q < KS; ++q) v += sm[(q * BM + m) * BN + n];
      return v;
    };
    if (p.act) {
      for (int e = tid; e < BM * BN / 2; e += NTH) {
        const int m = e / (BN / 2), f = e % (BN / 2), n = f / 16 * 32 + f % 16;
        out_act(m0 + m, n0 + n, sum(m, n), sum(m, n + 16));
      }
    } else {
      for (int e = tid; e < BM * BN; e += NTH) out(m0 + e / BN, n0 + e % BN, sum(e / BN, e % BN));
    }
  }
}

template <typename T, int BM, int BN, int KS, int KC>
const char *run(const SimtGemm &p, cudaStream_t s) {
  constexpr int st = 2 * (BM + BN) * (KC + 4) * 4, red = KS > 1 ? KS * BM * BN * 4 : 0;
  constexpr int smem = st > red ? st : red;
  static PerDevice<size_t> limit;  // above 48 KB only by opt-in
  if (const char *e = smem_opt_in(limit, k_gemm_simt<T, BM, BN, KS, KC>, smem)) return e;
  launch_pdl(k_gemm_simt<T, BM, BN, KS, KC>, dim3((p.N + BN - 1) / BN, (p.M + BM - 1) / BM), NTH,
             smem, s, p);
  return nullptr;
}

template <typename T>
const char *pick(const SimtGemm &p, int num_sms, cudaStream_t s) {
  auto tiles = [&](int bm, int bn) {
    return (long long)((p.M + bm - 1) / bm) * ((p.N + bn - 1) / bn);
  };
  if (tiles(64, 64) >= 2 * num_sms) return run<T, 64, 64, 1, 32>(p, s);
  if (tiles(32, 32) >= num_sms) return run<T, 32, 32, 4, 128>(p, s);
  return run<T, 16, 32, 8, 128>(p, s);
}

}  // namespace

const char *launch_gemm_simt(const GemmArgs &g, void *act, int num_sms, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0) return nullptr;
  SimtGemm p{g.X, g.W, g.bias, g.Y, act, g.M, g.N, g.K, g.ldx, g.ldy, g.accumulate};
  return g.dtype == KVR_DTYPE_BF16 ? pick<__nv_bfloat16>(p, num_sms, s)
                                   : pick<float>(p, num_sms, s);
}

}  // namespace kvr
