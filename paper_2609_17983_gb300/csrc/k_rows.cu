// k_rows.cu -- per-row kernels of the repair pass: seeded weight init,
// embedding gather, RMSNorm, RoPE + K/V scatter into the paged cache,
// and cache row readback / save / restore.
#include <algorithm>
#include <cooperative_groups.h>
#include <utility>

#include "kvr_internal.cuh"

namespace kvr {

namespace {

constexpr uint64_t GAMMA = 0x9E3779B97F4A7C15ull;

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

template <typename T>
__device__ __forceinline__ float ld(const T *p, size_t i);
template <>
__device__ __forceinline__ float ld<float>(const float *p, size_t i) { return p[i]; }
template <>
__device__ __forceinline__ float ld<__nv_bfloat16>(const __nv_bfloat16 *p, size_t i) {
  return __bfloat162float(p[i]);
}

template <typename T>
__device__ __forceinline__ void st(T *p, size_t i, float v);
template <>
__device__ __forceinline__ void st<float>(float *p, size_t i, float v) { p[i] = v; }
template <>
__device__ __forceinline__ void st<__nv_bfloat16>(__nv_bfloat16 *p, size_t i, float v) {
  p[i] = __float2bfloat16_rn(v);
}

// Four consecutive elements, one load or store (offsets multiples of 4; every
// row here starts on the 16-byte boundary of its four fp32, or 8 of its bf16).
__device__ __forceinline__ float4 ld4(const float *p, size_t i) { return *(const float4 *)(p + i); }
__device__ __forceinline__ float4 ld4(const __nv_bfloat16 *p, size_t i) {
  const uint2 u = *(const uint2 *)(p + i);
  const float2 a = __bfloat1622float2(*(const __nv_bfloat162 *)&u.x);
  const float2 b = __bfloat1622float2(*(const __nv_bfloat162 *)&u.y);
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st4(float *p, size_t i, float4 v) { *(float4 *)(p + i) = v; }
__device__ __forceinline__ void st4(__nv_bfloat16 *p, size_t i, float4 v) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  *(uint2 *)(p + i) = make_uint2(*(const uint32_t *)&a, *(const uint32_t *)&b);
}

// One element of the seeded weight definition (SplitMix64 stream, Irwin-Hall
// sum of four 16-bit lanes, scaled in double, rounded to fp32).
__device__ __forceinline__ float init_value(uint64_t tseed, int64_t e, double scale) {
  uint64_t r = mix64(tseed + (uint64_t)(e + 1) * GAMMA);
  int s = (int)(r & 0xFFFF) + (int)((r >> 16) & 0xFFFF) + (int)((r >> 32) & 0xFFFF) +
          (int)(r >> 48);
  double x = (double)(s - 2 * 65535) * scale;
  return __double2float_rn(x);
}

__global__ void k_init_tensor(void *dst, int dtype, int out_f32, uint64_t tseed, double scale,
                              int64_t rows, int64_t cols, int64_t row_off, int inter) {
  int64_t total = rows * cols;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    float f = init_value(tseed, e, scale);
    int64_t r = e / cols, c = e % cols;
    int64_t dr = inter == 0 ? row_off + r
                            : (r / GU_BLOCK) * (2 * GU_BLOCK) + (inter == 2 ? GU_BLOCK : 0) +
                                  r % GU_BLOCK;
    size_t o = (size_t)(dr * cols + c);
    if (dtype == KVR_DTYPE_BF16) {
      __nv_bfloat16 b = __float2bfloat16_rn(f);
      if (out_f32)
        ((float *)dst)[o] = __bfloat162float(b);
      else
        ((__nv_bfloat16 *)dst)[o] = b;
    } else {
      ((float *)dst)[o] = f;
    }
  }
}

__global__ void k_fill_f32(float *dst, float v, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    dst[i] = v;
}

// A CTA per row (d % 4 == 0), four elements per access: with 2-byte loads and
// 4-byte stores 4096 rows of d = 4096 took 36.6 us (100 MB, 2.7 TB/s).
// Launched without programmatic dependence: kernels behind it read positions
// and attention blocks ahead of their own waits, so the pass begins when the
// kernel that uploads those (k_upload) is over.
constexpr int EMBED_THREADS = 256;
template <typename T>
__global__ void k_embed_rows(const T *embed, const int32_t *tokens,
                             const int32_t *const *doc_tokens, const int32_t *rowdoc,
                             const int32_t *pos, int d, float *h) {
  TraceScope ts(TK_EMBED);
  pdl_trigger();
  ts.waited();
  int i = blockIdx.x;
  const int32_t *tk = doc_tokens ? doc_tokens[rowdoc[i]] : tokens;
  size_t base = (size_t)tk[pos[i]] * d;
#pragma unroll 4
  for (int c = 4 * threadIdx.x; c < d; c += 4 * EMBED_THREADS)
    st4(h, (size_t)i * d + c, ld4(embed, base + c));
}

// A call's small arrays (edited tokens, positions, attention blocks, a batch's
// tables) from page-locked host memory, and what goes with them from device
// memory, to their places, all in one launch: blockIdx.y is the segment.
// Bound by a round trip to the host.  A copy engine takes
// 3.2 us a segment, one after another, and more to hand over to the kernels:
// the 68 segments of 64 edits in 16 documents took 230 us, k_upload 2.7.
// Tensor maps are read through the tensor-map proxy: every thread that stores part
// of one releases its stores to it, the other half of the fence that the attention
// kernels execute before they use a map.  Each call overwrites the last one's maps.
constexpr int UP_THREADS = 256, UP_WORDS = 4;
template <int N>
struct UploadList {
  Upload u[N];
};
template <int N>
__global__ void __launch_bounds__(UP_THREADS) k_upload(const __grid_constant__ UploadList<N> l) {
  const Upload u = l.u[blockIdx.y];
  const size_t i0 = (size_t)blockIdx.x * (UP_THREADS * UP_WORDS) + threadIdx.x;
  int32_t v[UP_WORDS];
#pragma unroll
  for (int k = 0; k < UP_WORDS; ++k)
    if (i0 + k * UP_THREADS < u.words) v[k] = u.src[i0 + k * UP_THREADS];
#pragma unroll
  for (int k = 0; k < UP_WORDS; ++k)
    if (i0 + k * UP_THREADS < u.words) u.dst[i0 + k * UP_THREADS] = v[k];
  if (u.tensor_maps) asm volatile("fence.proxy.tensormap::generic.release.gpu;" ::: "memory");
}

// One block per row (d <= 8192, d % 4 == 0), each load issued before its
// first use: 1024 threads with NV = 1 float4 each up to d = 4096 (else 2)
// for a pass of a few rows, 256 threads with NV = d / 1024 for many.  Block i
// normalises h row row0 + i into out row i.  With a split view, the row is
// first completed from the GEMM's split-tile partials (their tile table is
// built once per block in shared memory) and written back to h.
constexpr int NORM_THREADS = 1024;   // a few rows: one float4 per thread, one round trip
constexpr int NORM_THREADS_WIDE = 256;  // many rows: several CTAs per SM, fewer waves
// The wide variant asks for four CTAs per SM: at 86 registers only two fit
// (prefill norms 3.2 against 2.9 ms).
template <typename T, int NV, int TPB>
__global__ void __launch_bounds__(TPB, TPB == NORM_THREADS_WIDE && NV <= 4 ? 4 : 1)
    k_rmsnorm(float *h, const float *g, int row0, int d, float eps, T *out, const SplitView sv) {
  __shared__ SplitTile tiles[64];
  __shared__ float red[TPB / 32];
  TraceScope ts(TK_NORM);
  pdl_trigger();
  const int i = blockIdx.x, row = row0 + i;
  const int nq = d >> 2;
  if (sv.ws && (int)threadIdx.x < (d >> 7)) {
    const int mt = row / sv.BN;
    tiles[threadIdx.x] = split_tile(sv, (long long)threadIdx.x * sv.m_tiles + mt);
  }
  // the gains are weights: read them before waiting on the residual's producer
  float4 gw[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int q = k * TPB + threadIdx.x;
    gw[k] = q < nq ? ((const float4 *)g)[q] : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  pdl_wait();
  ts.waited();
  if (sv.ws) __syncthreads();
  float4 *x = (float4 *)(h + (size_t)row * d);
  float4 v[NV];
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int q = k * TPB + threadIdx.x;
    v[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (q < nq) {
      v[k] = x[q];
      if (sv.ws) {
        const SplitTile st = tiles[q >> 5];
        if (st.i0 != st.i1) {
          v[k] = split_value4(sv, st, v[k], row, 4 * q);
          x[q] = v[k];
        }
      }
    }
    ss += v[k].x * v[k].x + v[k].y * v[k].y + v[k].z * v[k].z + v[k].w * v[k].w;
  }
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < TPB / 32; ++w) tot += red[w];
  const float r = 1.0f / sqrtf(tot / (float)d + eps);
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const int q = k * TPB + threadIdx.x;
    if (q < nq) {
      const float4 w = gw[k];
      st4(out, (size_t)i * d + 4 * q,
          make_float4(v[k].x * r * w.x, v[k].y * r * w.y, v[k].z * r * w.z, v[k].w * r * w.w));
    }
  }
}

// Many complete rows: the CTAs that fit (four an SM, NV <= 4) stay and take rows
// in turn, the next row's loads in flight while this one is reduced and written.
// Bound by HBM: 4096 rows of d = 4096 move 100 MB.  A CTA per row waited for
// its loads, then for the sum, and left: 24 us between events, this 17.
template <typename T, int NV>
__global__ void __launch_bounds__(NORM_THREADS_WIDE, 4)
    k_rmsnorm_rows(const float *h, const float *g, int row0, int M, int d, float eps, T *out) {
  constexpr int TPB = NORM_THREADS_WIDE;
  __shared__ float red[2][TPB / 32];
  TraceScope ts(TK_NORM);
  pdl_trigger();
  const int nq = d >> 2;
  pdl_wait();
  ts.waited();
  float4 nx[NV];
  auto fetch = [&](int i) {
    const float4 *x = (const float4 *)(h + (size_t)(row0 + i) * d);
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int q = k * TPB + threadIdx.x;
      nx[k] = i < M && q < nq ? x[q] : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  fetch(blockIdx.x);
  for (int i = blockIdx.x, b = 0; i < M; i += gridDim.x, b ^= 1) {
    float4 v[NV];
    float ss = 0.f;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      v[k] = nx[k];
      ss += v[k].x * v[k].x + v[k].y * v[k].y + v[k].z * v[k].z + v[k].w * v[k].w;
    }
    fetch(i + gridDim.x);
    for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
    // two sets of sums: a warp writes a set again only when all have read it
    if ((threadIdx.x & 31) == 0) red[b][threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int w = 0; w < TPB / 32; ++w) tot += red[b][w];
    const float r = 1.0f / sqrtf(tot / (float)d + eps);
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const int q = k * TPB + threadIdx.x;
      if (q < nq) {
        const float4 w = __ldg((const float4 *)g + q);
        st4(out, (size_t)i * d + 4 * q,
            make_float4(v[k].x * r * w.x, v[k].y * r * w.y, v[k].z * r * w.z, v[k].w * r * w.w));
      }
    }
  }
}

// RoPE of the q and k heads of the projection at each row's position: q ->
// q_out fp32 (if given) and qb_out, k and v -> cache (if write_kv) and rows_out
// (if given).  With a split view the projection is completed from the GEMM's
// split-tile partials.  Positions, the RoPE table, the page table and the bias
// are written before the pass, so they are read before the wait on the
// projection.
struct RopeArgs {
  const float *qkv;
  const float2 *rope;
  const int32_t *pos;
  int M, H, G, dh, layer, L;
  int heads;  // heads to take: all, or (no K/V written) the query heads alone
  const KVView *views;
  const int32_t *rowdoc;
  KVView single;
  float *q_out;
  __nv_bfloat16 *qb_out;
  float qscale;
  int write_kv;
  SplitView sv;
  void *rows_out;
};

// The row's cache entry (o) and rows_out entry (ro), for a k or v head hh; c
// null for a query head or a pass that writes no K/V.
template <typename T>
__device__ __forceinline__ void rope_dst(const RopeArgs &a, int hh, int i, int p, T *&c, size_t &o,
                                         size_t &ro) {
  c = nullptr;
  if (hh >= a.H && a.write_kv) {
    const int kv = hh < a.H + a.G ? 0 : 1, gk = hh - a.H - kv * a.G;
    const KVView v = a.views ? a.views[a.rowdoc[i]] : a.single;
    c = (T *)v.pages;
    o = v.offset(a.layer, kv, gk, p);
    // rows_out: K then V, each [M][L][G][dh]
    ro = ((((size_t)kv * a.M + i) * a.L + a.layer) * a.G + gk) * a.dh;
  }
}

// A pair rotated, with the rounding written out (x1 cos - x2 sin fused with its first
// product, x2 cos + x1 sin with its second): left to the compiler it depended on
// the kernel, and a row's bits must not depend on how many rows share its pass
// (kvr_margin runs two answers in one).
__device__ __forceinline__ void rotate(float x1, float x2, float c, float s, float &y1, float &y2) {
  y1 = __fmaf_rn(x1, c, -__fmul_rn(x2, s));  // x1, x2: copies, y may name the same pair
  y2 = __fmaf_rn(x1, s, __fmul_rn(x2, c));
}

// A few rows: grid (M, ceil((H + 2G) / ROPE_HEADS)), block ROPE_HEADS * dh/2, a
// rotated pair per thread -- latency counts, and every load is in flight at once.
constexpr int ROPE_HEADS = 8;  // heads per CTA
template <typename T>
__global__ void __launch_bounds__(ROPE_HEADS * 64) k_rope_scatter(const RopeArgs a) {
  TraceScope ts(TK_ROPE);
  pdl_trigger();
  const int half = a.dh >> 1, i = blockIdx.x;
  const int hh = blockIdx.y * ROPE_HEADS + threadIdx.x / half, t = threadIdx.x % half;
  if (hh >= a.heads) return;
  const int n1 = hh * a.dh + t, n2 = n1 + half;
  const int p = a.pos[i];
  float2 cs = make_float2(1.f, 0.f);
  if (hh < a.H + a.G) cs = a.rope[(size_t)p * half + t];
  T *c;
  size_t o = 0, ro = 0;
  rope_dst(a, hh, i, p, c, o, ro);
  const SplitView &sv = a.sv;
  // dh divides 128: both halves of the head lie in one feature tile
  SplitTile stl{0, 0, 0};
  float b1 = 0.f, b2 = 0.f;
  if (sv.ws) {
    stl = split_tile(sv, (long long)((hh * a.dh) >> 7) * sv.m_tiles + i / sv.BN);
    if (sv.bias) {
      b1 = sv.bias[n1];
      b2 = sv.bias[n2];
    }
  }
  pdl_wait();
  ts.waited();
  float x1, x2;
  if (sv.ws && stl.i0 != stl.i1) {
    const size_t off = (size_t)(i - (i / sv.BN) * sv.BN) * 128;
    x1 = b1 + split_sum(sv, stl, off + (n1 & 127));
    x2 = b2 + split_sum(sv, stl, off + (n2 & 127));
  } else {
    const float *x = a.qkv + (size_t)i * (a.H + 2 * a.G) * a.dh;
    x1 = x[n1];
    x2 = x[n2];
  }
  if (hh < a.H + a.G) rotate(x1, x2, cs.x, cs.y, x1, x2);
  if (hh < a.H) {
    const size_t q = (size_t)i * a.H * a.dh + n1;
    if (a.q_out) {
      a.q_out[q] = x1;
      a.q_out[q + half] = x2;
    }
    if (a.qb_out) {
      a.qb_out[q] = __float2bfloat16_rn(x1 * a.qscale);
      a.qb_out[q + half] = __float2bfloat16_rn(x2 * a.qscale);
    }
    return;
  }
  if (!c) return;
  st(c, o + t, x1);
  st(c, o + t + half, x2);
  if (a.rows_out) {
    st((T *)a.rows_out, ro + t, x1);
    st((T *)a.rows_out, ro + t + half, x2);
  }
}

// Many rows: a CTA per row, four rotated pairs per thread (16-byte loads, 8- or
// 16-byte stores) of HPT heads, which share the position, its table entries and
// page; the projection's loads do not wait for any of them.  Bound by HBM: 4096
// rows of a 6144-wide projection, 100 MB read, 50 MB written, take 29 us between
// events.  One pair per thread with 2-byte stores took 75; four rows of one head
// per thread 44 (107 registers, two CTAs an SM).
constexpr int ROPE_THREADS = 256;
// rows from which it is taken (40 rows: equal; 64 rows: 9.9 -> 8.2 us)
constexpr int ROPE_MANY = 64;
template <typename T, int HPT>
__global__ void __launch_bounds__(ROPE_THREADS, HPT > 1 ? 4 : 1) k_rope_rows(const RopeArgs a) {
  TraceScope ts(TK_ROPE);
  pdl_trigger();
  const int half = a.dh >> 1, tph = half >> 2;  // threads per head
  const int slots = blockDim.x / tph, h0 = blockIdx.y * slots * HPT + threadIdx.x / tph;
  const int t = threadIdx.x % tph * 4;
  if (h0 >= a.heads) return;
  const int i = blockIdx.x, Nqkv = (a.H + 2 * a.G) * a.dh;
  const SplitView &sv = a.sv;
  const int p = a.pos[i];
  pdl_wait();
  ts.waited();
  float4 x1[HPT], x2[HPT];
#pragma unroll
  for (int k = 0; k < HPT; ++k) {
    const int hh = h0 + k * slots, n1 = hh * a.dh + t;
    if (hh >= a.heads) break;
    const float *x = a.qkv + (size_t)i * Nqkv;
    x1[k] = ld4(x, n1);
    x2[k] = ld4(x, n1 + half);
    if (HPT == 1 && sv.ws) {
      const SplitTile stl = split_tile(sv, (long long)((hh * a.dh) >> 7) * sv.m_tiles + i / sv.BN);
      x1[k] = split_value4(sv, stl, x1[k], i, n1);
      x2[k] = split_value4(sv, stl, x2[k], i, n1 + half);
    }
  }
  const float4 *cs = (const float4 *)(a.rope + (size_t)p * half + t);
  const float4 ca = cs[0], cb = cs[1];
#pragma unroll
  for (int k = 0; k < HPT; ++k) {
    const int hh = h0 + k * slots;
    if (hh >= a.heads) break;
    const float4 u = x1[k], w = x2[k];
    float4 y1 = u, y2 = w;
    if (hh < a.H + a.G) {
      rotate(u.x, w.x, ca.x, ca.y, y1.x, y2.x);
      rotate(u.y, w.y, ca.z, ca.w, y1.y, y2.y);
      rotate(u.z, w.z, cb.x, cb.y, y1.z, y2.z);
      rotate(u.w, w.w, cb.z, cb.w, y1.w, y2.w);
    }
    if (hh < a.H) {
      const size_t q = (size_t)i * a.H * a.dh + hh * a.dh + t;
      if (a.q_out) {
        st4(a.q_out, q, y1);
        st4(a.q_out, q + half, y2);
      }
      if (a.qb_out) {
        const float s = a.qscale;
        st4(a.qb_out, q, make_float4(y1.x * s, y1.y * s, y1.z * s, y1.w * s));
        st4(a.qb_out, q + half, make_float4(y2.x * s, y2.y * s, y2.z * s, y2.w * s));
      }
      continue;
    }
    T *c;
    size_t o = 0, ro = 0;
    rope_dst(a, hh, i, p, c, o, ro);
    if (!c) continue;
    st4(c, o + t, y1);
    st4(c, o + t + half, y2);
    if (a.rows_out) {
      st4((T *)a.rows_out, ro + t, y1);
      st4((T *)a.rows_out, ro + t + half, y2);
    }
  }
}

// Positions of a readback: a few come with the launch (many: in device memory).
struct HostReadPos {
  int32_t p[HOST_READ_MAX_POS];
};

template <typename T>
__global__ void k_cache_gather(KVView v, const __grid_constant__ HostReadPos pos,
                               const int32_t *many, int n_pos, int l0, int nl, int G, int dh,
                               float *k_out, float *v_out) {
  size_t total = (size_t)n_pos * nl * G * dh;
  const T *c = (const T *)v.pages;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    int i = (int)(e % dh);
    size_t r = e / dh;
    int g = (int)(r % G);
    r /= G;
    const int l = (int)(r % nl), p = many ? many[r / nl] : pos.p[r / nl];
    k_out[e] = ld(c, v.offset(l0 + l, 0, g, p) + i);
    v_out[e] = ld(c, v.offset(l0 + l, 1, g, p) + i);
  }
}

// K/V of the given positions, layers l0 .. l0+nl-1, as stored: 16-byte
// pieces of the cache rows (a row is head_dim elements, a multiple of 16
// bytes), vr pieces a row, output [n_pos][nl][G][row].
__global__ void k_cache_gather_raw(KVView v, const __grid_constant__ HostReadPos pos,
                                   const int32_t *many, int n_pos, int l0, int nl, int G, int vr,
                                   int es, uint4 *k_out, uint4 *v_out) {
  const unsigned total = (unsigned)n_pos * nl * G * vr;
  const uint4 *c = (const uint4 *)v.pages;
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += gridDim.x * blockDim.x) {
    const unsigned i = e % vr;
    unsigned r = e / vr;
    const int g = (int)(r % G);
    r /= G;
    const int l = (int)(r % nl), p = many ? many[r / nl] : pos.p[r / nl];
    k_out[e] = c[v.offset(l0 + l, 0, g, p) * es / 16 + i];
    v_out[e] = c[v.offset(l0 + l, 1, g, p) * es / 16 + i];
  }
}

// k_cache_gather_raw into page-locked host memory: the rows leave by the stores
// themselves, without a gathered copy or a copy's set-up, and the device error flag
// goes with the rows (everything queued before has run).  Bound by the link to the
// host: 82 MB at 183 GB/s.
__global__ void k_cache_read_host(KVView v, const __grid_constant__ HostReadPos pos,
                                  const int32_t *many, int n_pos, int l0, int nl, int G, int vr,
                                  int es, uint4 *k_out, uint4 *v_out, const int *flag_in,
                                  int *flag_out) {
  pdl_trigger();
  pdl_wait();
  const unsigned total = (unsigned)n_pos * nl * G * vr;
  const uint4 *c = (const uint4 *)v.pages;
  for (unsigned e = blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += gridDim.x * blockDim.x) {
    const unsigned i = e % vr;
    unsigned r = e / vr;
    const int g = (int)(r % G);
    r /= G;
    const int l = (int)(r % nl), p = many ? many[r / nl] : pos.p[r / nl];
    const uint4 k = c[v.offset(l0 + l, 0, g, p) * es / 16 + i];
    const uint4 w = c[v.offset(l0 + l, 1, g, p) * es / 16 + i];
    k_out[e] = k;
    v_out[e] = w;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) *flag_out = *flag_in;
}

// The inverse of k_cache_gather_raw for consecutive positions p0 .. p0+n_pos-1
// and every layer: rows [n_pos][L][G][dh] of k_in / v_in written into the pages.
template <typename T>
__global__ void k_cache_scatter_raw(KVView v, int p0, int n_pos, const T *k_in, const T *v_in) {
  const int L = v.L, G = v.G, dh = v.dh;
  size_t total = (size_t)n_pos * L * G * dh;
  T *c = (T *)v.pages;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    int i = (int)(e % dh);
    size_t r = e / dh;
    int g = (int)(r % G);
    r /= G;
    int l = (int)(r % L);
    int p = p0 + (int)(r / L);
    c[v.offset(l, 0, g, p) + i] = k_in[e];
    c[v.offset(l, 1, g, p) + i] = v_in[e];
  }
}

// buf layout [n_pos][nl][2][G][dh] in the cache dtype
template <typename T>
__global__ void k_rows_copy(KVView v, const int32_t *pos, int n_pos, int l0, int nl, T *buf,
                            int to_buf) {
  int G = v.G, dh = v.dh;
  size_t total = (size_t)n_pos * nl * 2 * G * dh;
  T *c = (T *)v.pages;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    int i = (int)(e % dh);
    size_t r = e / dh;
    int g = (int)(r % G);
    r /= G;
    int kv = (int)(r % 2);
    r /= 2;
    int l = (int)(r % nl);
    int p = (int)(r / nl);
    size_t o = v.offset(l0 + l, kv, g, pos[p]) + i;
    if (to_buf)
      buf[e] = c[o];
    else
      c[o] = buf[e];
  }
}

// Transplant: copy K/V of every layer at the listed positions, and their
// tokens, from one document into another (same model shape).  16-byte pieces
// of the cache rows, vr a row.
__global__ void k_transplant(KVView dst, KVView src, const int32_t *pos, int n_pos, int vr, int es,
                             int32_t *tok_dst, const int32_t *tok_src) {
  const int L = dst.L, G = dst.G;
  const size_t total = (size_t)n_pos * L * 2 * G * vr;
  const uint4 *s = (const uint4 *)src.pages;
  uint4 *d = (uint4 *)dst.pages;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % vr);
    size_t r = e / vr;
    const int g = (int)(r % G);
    r /= G;
    const int kv = (int)(r % 2);
    r /= 2;
    const int l = (int)(r % L), p = pos[r / L];
    d[dst.offset(l, kv, g, p) * es / 16 + i] = s[src.offset(l, kv, g, p) * es / 16 + i];
    if (e < n_pos) tok_dst[pos[e]] = tok_src[pos[e]];  // total >= n_pos: every position once
  }
}

// out[i] = logits[i][target[i]] - logsumexp(logits[i]) for each row; out is
// page-locked host memory, and the device error flag goes with it (copies of
// targets, results and flag took 30 us of a pass).  A cluster of LP_CTAS CTAs a
// row, each with a slice of it, in one pass: a thread keeps its maximum and the
// sum of exponentials against it, LP_VEC float4 loads in flight (V % 4 == 0
// keeps every row on a 16-byte boundary; other widths load one at a time); the
// first CTA adds the slices in order.  128256 logits: 5 us; one CTA a row 11,
// two passes of scalar loads by 256 threads 49.
constexpr int LP_THREADS = 1024, LP_VEC = 4, LP_CTAS = 8;
struct AnswerIds {
  int32_t id[KVR_QUERY_RESERVE];
};
__device__ __forceinline__ void lse_add(float &m, float &s, float m2, float s2) {
  const float mm = fmaxf(m, m2);
  if (mm == -INFINITY) {  // both empty, or NaN (which the maximum passes over)
    s += s2;
    return;
  }
  s = s * expf(m - mm) + s2 * expf(m2 - mm);
  m = mm;
}
__global__ void __cluster_dims__(LP_CTAS, 1, 1) __launch_bounds__(LP_THREADS)
    k_row_logprob(const float *logits, int V, const __grid_constant__ AnswerIds target, float *out,
                  const int *flag_in, int *flag_out) {
  if (blockIdx.x == 0 && threadIdx.x == 0) *flag_out = *flag_in;
  namespace cg = cooperative_groups;
  const cg::cluster_group cluster = cg::this_cluster();
  const int row = blockIdx.x / LP_CTAS, part = blockIdx.x % LP_CTAS;
  const float *x = logits + (size_t)row * V;
  __shared__ float2 red[LP_THREADS / 32];
  __shared__ float2 slices[LP_CTAS];  // the first CTA's: every slice's maximum and sum
  auto started = cluster.barrier_arrive();  // waited on before the first CTA's memory is written
  float m = -INFINITY, s = 0.f;
  // a batch of loaded values: its maximum first, then one rescale of the sum
  auto add = [&](const float *v, int n) {
    float mx = m;
    for (int j = 0; j < n; ++j) mx = fmaxf(mx, v[j]);
    float t = 0.f;
    if (mx == -INFINITY) {  // nothing above the lowest value, but perhaps a NaN
      for (int j = 0; j < n; ++j) t += v[j] == -INFINITY ? 0.f : v[j];
      s += t;
      return;
    }
    for (int j = 0; j < n; ++j) t += expf(v[j] - mx);
    s = s * expf(m - mx) + t;
    m = mx;
  };
  if (V % 4 == 0) {
    const float4 *x4 = (const float4 *)x;
    const int per = (V / 4 + LP_CTAS - 1) / LP_CTAS, n4 = min(V / 4, (part + 1) * per);
    for (int j0 = part * per + threadIdx.x; j0 < n4; j0 += LP_VEC * LP_THREADS) {
      float4 v[LP_VEC];
#pragma unroll
      for (int k = 0; k < LP_VEC; ++k) {
        const int j = j0 + k * LP_THREADS;
        v[k] = j < n4 ? x4[j] : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
      }
      float w[4 * LP_VEC];
#pragma unroll
      for (int k = 0; k < LP_VEC; ++k) {
        w[4 * k] = v[k].x;
        w[4 * k + 1] = v[k].y;
        w[4 * k + 2] = v[k].z;
        w[4 * k + 3] = v[k].w;
      }
      add(w, 4 * LP_VEC);
    }
  } else {
    const int per = (V + LP_CTAS - 1) / LP_CTAS, n = min(V, (part + 1) * per);
    for (int j = part * per + threadIdx.x; j < n; j += LP_THREADS) {
      const float w[1] = {x[j]};
      add(w, 1);
    }
  }
  auto fold = [&]() {
    for (int o = 16; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, m, o), s2 = __shfl_xor_sync(0xffffffffu, s, o);
      lse_add(m, s, m2, s2);
    }
  };
  fold();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = make_float2(m, s);
  cluster.barrier_wait(std::move(started));
  __syncthreads();
  if (threadIdx.x < 32) {
    m = red[threadIdx.x].x;
    s = red[threadIdx.x].y;
    fold();
    if (threadIdx.x == 0) cluster.map_shared_rank(slices, 0)[part] = make_float2(m, s);
  }
  cluster.sync();
  if (part == 0 && threadIdx.x == 0) {
    m = slices[0].x;
    s = slices[0].y;
    for (int k = 1; k < LP_CTAS; ++k) lse_add(m, s, slices[k].x, slices[k].y);
    out[row] = x[target.id[row]] - (m + logf(s));
  }
}

int grid_for(size_t n, int block) {
  size_t g = (n + block - 1) / block;
  return (int)(g > 65535 * 8 ? 65535 * 8 : (g == 0 ? 1 : g));
}

}  // namespace

void launch_init_tensor(void *dst, int dtype, bool out_f32, uint64_t tseed, double scale,
                        int64_t rows, int64_t cols, int64_t row_off, int interleave,
                        cudaStream_t s) {
  size_t n = (size_t)(rows * cols);
  k_init_tensor<<<grid_for(n, 256), 256, 0, s>>>(dst, dtype, out_f32 ? 1 : 0, tseed, scale, rows,
                                                  cols, row_off, interleave);
}

void launch_fill_f32(float *dst, float v, size_t n, cudaStream_t s) {
  k_fill_f32<<<grid_for(n, 256), 256, 0, s>>>(dst, v, n);
}

void launch_upload(const Upload *u, int n, cudaStream_t s) {
  size_t most = 1;
  for (int i = 0; i < n; ++i) most = std::max<size_t>(most, u[i].words);
  const dim3 grid((unsigned)((most + UP_THREADS * UP_WORDS - 1) / (UP_THREADS * UP_WORDS)), n);
  auto go = [&](auto list) {  // few segments: a launch without the larger list's bytes
    std::copy(u, u + n, list.u);
    k_upload<<<grid, UP_THREADS, 0, s>>>(list);
  };
  if (n <= 8)
    go(UploadList<8>{});
  else
    go(UploadList<UPLOAD_MAX>{});
}

void launch_embed_rows(const void *embed, int dtype, const int32_t *tokens,
                       const int32_t *const *doc_tokens, const int32_t *rowdoc,
                       const int32_t *pos, int M, int d, float *h, cudaStream_t s) {
  if (M <= 0) return;
  if (dtype == KVR_DTYPE_BF16)
    k_embed_rows<<<M, EMBED_THREADS, 0, s>>>((const __nv_bfloat16 *)embed, tokens, doc_tokens,
                                             rowdoc, pos, d, h);
  else
    k_embed_rows<<<M, EMBED_THREADS, 0, s>>>((const float *)embed, tokens, doc_tokens, rowdoc, pos,
                                             d, h);
}

void launch_rmsnorm(float *h, const float *g, int row0, int M, int d, double eps, void *out,
                    int out_dtype, int num_sms, cudaStream_t s, const SplitView *sv) {
  if (M <= 0) return;
  const SplitView v = sv ? *sv : SplitView{};
  // A pass of a few rows is latency-bound: 1024 threads, each with one
  // float4 in flight.  Hundreds of rows (prefill): 256 threads a row, several
  // rows per SM at once, staying on the SM unless split tiles are to be added or
  // a row does not fit 64 registers a thread twice.
  if (M > 256 && d <= 4 * 8 * NORM_THREADS_WIDE) {
    constexpr int W = NORM_THREADS_WIDE;
    const int nv = (d + 4 * W - 1) / (4 * W);
    if (!v.ws && nv <= 4) {
      const int grid = std::min(M, 4 * num_sms);
      if (out_dtype == KVR_DTYPE_BF16) {
        auto k = nv <= 1 ? k_rmsnorm_rows<__nv_bfloat16, 1>
                 : nv <= 2 ? k_rmsnorm_rows<__nv_bfloat16, 2>
                           : k_rmsnorm_rows<__nv_bfloat16, 4>;
        launch_pdl(k, grid, W, 0, s, (const float *)h, g, row0, M, d, (float)eps,
                   (__nv_bfloat16 *)out);
      } else {
        auto k = nv <= 1 ? k_rmsnorm_rows<float, 1>
                 : nv <= 2 ? k_rmsnorm_rows<float, 2>
                           : k_rmsnorm_rows<float, 4>;
        launch_pdl(k, grid, W, 0, s, (const float *)h, g, row0, M, d, (float)eps, (float *)out);
      }
      return;
    }
    if (out_dtype == KVR_DTYPE_BF16) {
      auto k = nv <= 1 ? k_rmsnorm<__nv_bfloat16, 1, W>
               : nv <= 2 ? k_rmsnorm<__nv_bfloat16, 2, W>
               : nv <= 4 ? k_rmsnorm<__nv_bfloat16, 4, W>
                         : k_rmsnorm<__nv_bfloat16, 8, W>;
      launch_pdl(k, M, W, 0, s, h, g, row0, d, (float)eps, (__nv_bfloat16 *)out, v);
    } else {
      auto k = nv <= 1 ? k_rmsnorm<float, 1, W>
               : nv <= 2 ? k_rmsnorm<float, 2, W>
               : nv <= 4 ? k_rmsnorm<float, 4, W>
                         : k_rmsnorm<float, 8, W>;
      launch_pdl(k, M, W, 0, s, h, g, row0, d, (float)eps, (float *)out, v);
    }
    return;
  }
  const bool one = d <= 4 * NORM_THREADS;
  if (out_dtype == KVR_DTYPE_BF16)
    launch_pdl(one ? k_rmsnorm<__nv_bfloat16, 1, NORM_THREADS>
                   : k_rmsnorm<__nv_bfloat16, 2, NORM_THREADS>,
               M, NORM_THREADS, 0, s, h, g, row0, d, (float)eps, (__nv_bfloat16 *)out, v);
  else
    launch_pdl(one ? k_rmsnorm<float, 1, NORM_THREADS> : k_rmsnorm<float, 2, NORM_THREADS>, M,
               NORM_THREADS, 0, s, h, g, row0, d, (float)eps, (float *)out, v);
}

void launch_rope_scatter(const float *qkv, const float2 *rope, const int32_t *pos, int M,
                         const Dims &dm, int layer, const KVView *views, const int32_t *rowdoc,
                         KVView single, float *q_out, void *qb_out, float qscale, bool write_kv,
                         cudaStream_t s, const SplitView *sv, void *rows_out) {
  if (M <= 0) return;
  const int heads = write_kv ? dm.H + 2 * dm.G : dm.H;
  RopeArgs a{qkv,   rope,   pos,    M,     dm.H,
             dm.G,  dm.dh,  layer,  dm.L,  heads,
             views, rowdoc, single, q_out, (__nv_bfloat16 *)qb_out,
             qscale, write_kv ? 1 : 0, sv ? *sv : SplitView{}, rows_out};
  auto go = [&](auto *tag) {
    using T = std::remove_pointer_t<decltype(tag)>;
    if (M < ROPE_MANY) {
      launch_pdl(k_rope_scatter<T>, dim3(M, (heads + ROPE_HEADS - 1) / ROPE_HEADS),
                 ROPE_HEADS * dm.dh / 2, 0, s, a);
    } else {
      // heads per thread: three where a CTA's thread groups are that many times
      // fewer; one to add split tiles (each has up to eight parts in flight)
      const int tph = dm.dh / 8, threads = std::min(ROPE_THREADS, (heads * tph + 31) / 32 * 32);
      const int slots = threads / tph, hpt = a.sv.ws || heads <= slots ? 1 : 3;
      launch_pdl(hpt > 1 ? k_rope_rows<T, 3> : k_rope_rows<T, 1>,
                 dim3(M, (heads + slots * hpt - 1) / (slots * hpt)), threads, 0, s, a);
    }
  };
  if (dm.dtype == KVR_DTYPE_BF16)
    go((__nv_bfloat16 *)nullptr);
  else
    go((float *)nullptr);
}

namespace {
HostReadPos launch_positions(const int32_t *pos, const int32_t *pos_d, int n_pos) {
  HostReadPos p;
  if (!pos_d) std::copy(pos, pos + n_pos, p.p);
  return p;
}
}  // namespace

void launch_cache_gather(KVView v, int dtype, const int32_t *pos, const int32_t *pos_d, int n_pos,
                         int l0, int l1, int G, int dh, float *k_out, float *v_out,
                         cudaStream_t s) {
  size_t n = (size_t)n_pos * (l1 - l0) * G * dh;
  if (n == 0) return;
  const HostReadPos p = launch_positions(pos, pos_d, n_pos);
  if (dtype == KVR_DTYPE_BF16)
    k_cache_gather<__nv_bfloat16><<<grid_for(n, 256), 256, 0, s>>>(v, p, pos_d, n_pos, l0, l1 - l0,
                                                                    G, dh, k_out, v_out);
  else
    k_cache_gather<float><<<grid_for(n, 256), 256, 0, s>>>(v, p, pos_d, n_pos, l0, l1 - l0, G, dh,
                                                            k_out, v_out);
}

void launch_cache_gather_raw(KVView v, int dtype, const int32_t *pos, const int32_t *pos_d,
                             int n_pos, int l0, int l1, int G, int dh, void *k_out, void *v_out,
                             cudaStream_t s) {
  const int es = dtype == KVR_DTYPE_BF16 ? 2 : 4, vr = dh * es / 16;
  const size_t per_pos = (size_t)(l1 - l0) * G * vr;
  if (per_pos == 0) return;
  // launches of fewer than 2^31 pieces (the kernel indexes in 32 bits)
  const int chunk = (int)std::min<size_t>((size_t)n_pos, ((size_t)1 << 31) / per_pos);
  for (int p0 = 0; p0 < n_pos; p0 += chunk) {
    const int np = std::min(chunk, n_pos - p0);
    k_cache_gather_raw<<<grid_for(np * per_pos, 256), 256, 0, s>>>(
        v, launch_positions(pos + p0, pos_d, np), pos_d ? pos_d + p0 : nullptr, np, l0, l1 - l0, G,
        vr, es, (uint4 *)k_out + p0 * per_pos, (uint4 *)v_out + p0 * per_pos);
  }
}

void launch_cache_read_host(KVView v, int dtype, const int32_t *pos, const int32_t *pos_d,
                            int n_pos, int l0, int l1, int G, int dh, void *k_out, void *v_out,
                            const int *flag_in, int *flag_out, cudaStream_t s) {
  const int es = dtype == KVR_DTYPE_BF16 ? 2 : 4, vr = dh * es / 16;
  launch_pdl(k_cache_read_host, grid_for((size_t)n_pos * (l1 - l0) * G * vr, 256), 256, 0, s, v,
             launch_positions(pos, pos_d, n_pos), pos_d, n_pos, l0, l1 - l0, G, vr, es,
             (uint4 *)k_out, (uint4 *)v_out, flag_in, flag_out);
}

void launch_cache_scatter_raw(KVView v, int dtype, int p0, int n_pos, const void *k_in,
                              const void *v_in, cudaStream_t s) {
  size_t n = (size_t)n_pos * v.L * v.G * v.dh;
  if (n == 0) return;
  if (dtype == KVR_DTYPE_BF16)
    k_cache_scatter_raw<__nv_bfloat16><<<grid_for(n, 256), 256, 0, s>>>(
        v, p0, n_pos, (const __nv_bfloat16 *)k_in, (const __nv_bfloat16 *)v_in);
  else
    k_cache_scatter_raw<float><<<grid_for(n, 256), 256, 0, s>>>(v, p0, n_pos, (const float *)k_in,
                                                                 (const float *)v_in);
}

void launch_transplant(KVView dst, KVView src, int dtype, const int32_t *pos, int n_pos,
                       int32_t *tok_dst, const int32_t *tok_src, cudaStream_t s) {
  const int es = dtype == KVR_DTYPE_BF16 ? 2 : 4, vr = dst.dh * es / 16;
  const size_t n = (size_t)n_pos * dst.L * 2 * dst.G * vr;
  if (n)
    k_transplant<<<grid_for(n, 256), 256, 0, s>>>(dst, src, pos, n_pos, vr, es, tok_dst, tok_src);
}

void launch_row_logprob(const float *logits, int rows, int V, const int32_t *target, float *out,
                        const int *flag_in, int *flag_out, cudaStream_t s) {
  AnswerIds t;
  std::copy(target, target + rows, t.id);
  k_row_logprob<<<rows * LP_CTAS, LP_THREADS, 0, s>>>(logits, V, t, out, flag_in, flag_out);
}

void launch_rows_copy(KVView v, int dtype, const int32_t *pos, int n_pos, int l0, int l1,
                      void *buf, bool to_buf, cudaStream_t s) {
  size_t n = (size_t)n_pos * (l1 - l0) * 2 * v.G * v.dh;
  if (n == 0) return;
  if (dtype == KVR_DTYPE_BF16)
    k_rows_copy<<<grid_for(n, 256), 256, 0, s>>>(v, pos, n_pos, l0, l1 - l0,
                                                  (__nv_bfloat16 *)buf, to_buf ? 1 : 0);
  else
    k_rows_copy<<<grid_for(n, 256), 256, 0, s>>>(v, pos, n_pos, l0, l1 - l0, (float *)buf,
                                                  to_buf ? 1 : 0);
}

KVR_TRACE_ATTACH(trace_attach_rows)

}  // namespace kvr
