// k_select.cu -- selector scores (Table 1) and the top-K rule.
//
// Scores become 64-bit keys, larger = better, indexed by j - s_end over the
// pool D = [s_end, n).  Key 0 marks a position the policy excludes
// (Structural: not a delimiter).  Top-K orders by key descending, then
// position ascending (ties to the lowest position), and returns the chosen
// positions ascending.
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "kvr_internal.cuh"

namespace kvr {
namespace {

constexpr uint64_t GAMMA = 0x9E3779B97F4A7C15ull;

__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Order-preserving map of a float to uint32 (NaN ranks as -inf).
__device__ __forceinline__ uint32_t ord_f32(float f) {
  if (isnan(f)) f = -INFINITY;
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Key of pool entry t (position s_end + t) under Random or Structural.
__device__ __forceinline__ unsigned long long simple_key(const SimpleKeys &g, int s_end, int t) {
  const int j = s_end + t;
  if (g.policy == KVR_POLICY_RANDOM) {
    // first SplitMix64 output of state seed ^ (j * gamma)
    return mix64((g.seed ^ ((uint64_t)j * GAMMA)) + GAMMA);
  }
  // Structural: delimiters, nearest to the span first
  return g.tokens[j] == g.delim ? 0x100000000ull - (unsigned long long)t : 0;
}

__global__ void k_float_keys(const float *scores, int n, int s_end, unsigned long long *keys) {
  int c = n - s_end;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < c; t += gridDim.x * blockDim.x)
    keys[t] = (unsigned long long)ord_f32(scores[s_end + t]) + 1ull;
}

// Top-K of c (key, index) pairs, one CTA of TOPK_THREADS: key descending, ties to
// the lowest index, the chosen indices written ascending.  Instead of a sort,
// the K-th key T is found by an MSB-first radix select (11 bits per pass, a
// shared-memory histogram of the keys that still match the prefix), starting
// at the highest bit in which the keys differ (the AND and OR of all keys give
// the bits they share, which the passes would only confirm); then
// every key above T is taken, and of the keys equal to T the lowest-indexed
// ones until K are taken.  A pass that ends with every key of the chosen bin
// taken ends the search: the digits below cannot change the set (Random's
// 64-bit keys mostly part in the first).  8-bit digits counted bin by bin of a
// warp (match.any) took 20.8 us a Random selection of 1544 keys through the
// API and 25.5 of 4894, now 19.5 and 20.8.  Thread i owns the contiguous keys
// [i*E, (i+1)*E), so a block-wide scan of per-thread counts writes the output in
// index order.
constexpr int TOPK_THREADS = 1024;
constexpr int TOPK_BITS = 11;  // two bins a thread
static_assert(1 << TOPK_BITS == 2 * TOPK_THREADS, "two bins a thread");

__device__ __forceinline__ int block_excl_scan(int x, int *tmp) {
  // tmp: TOPK_THREADS / 32 ints
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int v = x;
  for (int o = 1; o < 32; o <<= 1) {
    int y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  if (lane == 31) tmp[warp] = v;
  __syncthreads();
  if (warp == 0) {
    int w = lane < TOPK_THREADS / 32 ? tmp[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < TOPK_THREADS / 32) tmp[lane] = w;
  }
  __syncthreads();
  const int before = (warp ? tmp[warp - 1] : 0) + v - x;
  __syncthreads();
  return before;
}

__global__ void __launch_bounds__(TOPK_THREADS)
    k_topk(const unsigned long long *keys, int c, int s_end, int K, int nonzero_only,
           int32_t *out, int32_t *count, const SimpleKeys gen, const int *flag_in,
           int32_t *flag_out) {
  extern __shared__ unsigned long long sk[];  // c keys
  __shared__ int hist[1 << TOPK_BITS];
  __shared__ int scan_tmp[TOPK_THREADS / 32];
  __shared__ int s_elig, s_bin, s_above, s_in;
  __shared__ unsigned long long s_and, s_or;
  const int tid = threadIdx.x;
  if (gen.policy == KVR_POLICY_EDITLOCAL || gen.policy == KVR_POLICY_EDITLOCAL_BOUNDARY) {
    // EditLocal's keys fall strictly with t, and all are eligible (@boundary: up
    // to the first delimiter, the whole pool without one): the K largest are the
    // first K candidates, already in index order.
    int avail = c;
    if (gen.policy == KVR_POLICY_EDITLOCAL_BOUNDARY) {
      if (tid == 0) s_in = c;
      __syncthreads();
      for (int t = tid; t < c; t += TOPK_THREADS)
        if (gen.tokens[s_end + t] == gen.delim) {
          atomicMin(&s_in, t + 1);
          break;
        }
      __syncthreads();
      avail = s_in;
    }
    const int cnt = min(K, avail);
    for (int t = tid; t < cnt; t += TOPK_THREADS) out[t] = s_end + t;
    if (tid == 0) {
      *count = cnt;
      if (flag_in) *flag_out = *flag_in;
    }
    return;
  }
  const int E = (c + TOPK_THREADS - 1) / TOPK_THREADS;
  const int t0 = min(c, tid * E), t1 = min(c, t0 + E);
  if (tid == 0) {
    s_elig = 0;
    s_and = ~0ull;
    s_or = 0ull;
  }
  __syncthreads();
  auto eligible = [&](unsigned long long k) { return !nonzero_only || k != 0ull; };
  int local = 0;
  unsigned long long kand = ~0ull, kor = 0ull;
  for (int t = tid; t < c; t += TOPK_THREADS) {
    const unsigned long long k = gen.policy >= 0 ? simple_key(gen, s_end, t) : keys[t];
    sk[t] = k;
    if (eligible(k)) {
      kand &= k;
      kor |= k;
      ++local;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    local += __shfl_xor_sync(0xffffffffu, local, o);
    kand &= __shfl_xor_sync(0xffffffffu, kand, o);
    kor |= __shfl_xor_sync(0xffffffffu, kor, o);
  }
  if ((tid & 31) == 0) {
    atomicAdd(&s_elig, local);
    atomicAnd(&s_and, kand);
    atomicOr(&s_or, kor);
  }
  __syncthreads();
  const int cnt = min(K, s_elig);
  // radix select: prefix/mask of T, need = how many keys equal to the prefix
  // (so far) are still to be taken.  The bits above hi are the same in every
  // eligible key: they start the prefix.
  const unsigned long long differ = s_or ^ s_and;
  int hi = 64 - (differ ? __clzll((long long)differ) : 64);  // bits not yet in the prefix
  unsigned long long mask = hi == 64 ? 0ull : ~0ull << hi;
  unsigned long long pref = s_and & mask;
  int need = cnt;
  while (hi > 0 && need > 0) {
    const int d = max(0, hi - TOPK_BITS);  // this digit: bits d .. hi - 1
    hist[tid] = hist[tid + TOPK_THREADS] = 0;
    __syncthreads();
    // a warp whose keys all fall in one bin adds their count once (many equal keys
    // on one shared-memory address would serialise the pass); matching lanes bin
    // by bin instead took longer than their atomics
    for (int e = 0; e < E; ++e) {
      const int t = t0 + e;
      const unsigned long long k = t < t1 ? sk[t] : 0ull;
      const bool in = t < t1 && (k & mask) == pref && eligible(k);
      const int bin = in ? (int)(k >> d) & ((1 << (hi - d)) - 1) : -1;
      int same;
      __match_all_sync(0xffffffffu, bin, &same);
      if (bin >= 0 && (!same || (tid & 31) == 0)) atomicAdd(&hist[bin], same ? 32 : 1);
    }
    __syncthreads();
    // the bin that holds the need-th key from the top: thread i's two bins,
    // highest first, after the counts of the threads before it
    const int b1 = 2 * (TOPK_THREADS - 1 - tid) + 1, h1 = hist[b1], h0 = hist[b1 - 1];
    const int above = block_excl_scan(h1 + h0, scan_tmp);
    if (above < need && above + h1 + h0 >= need) {
      const bool first = above + h1 >= need;
      s_bin = first ? b1 : b1 - 1;
      s_above = first ? above : above + h1;
      s_in = first ? h1 : h0;
    }
    __syncthreads();
    pref |= (unsigned long long)s_bin << d;
    mask = d == 0 ? ~0ull : ~0ull << d;
    need -= s_above;
    hi = d;
    if (s_in == need) break;  // the bin's keys are all taken
    // the next pass writes s_bin, s_above and s_in behind three barriers
  }
  // T = pref in the digits of mask (when cnt > 0): take keys > T, and the first
  // `need` keys == T
  int gt = 0, eq = 0;
  if (cnt > 0)
    for (int t = t0; t < t1; ++t) {
      const unsigned long long k = sk[t];
      gt += eligible(k) && (k & mask) > pref ? 1 : 0;
      eq += eligible(k) && (k & mask) == pref ? 1 : 0;
    }
  const int eq_before = block_excl_scan(eq, scan_tmp);
  int take_eq = cnt > 0 ? min(eq, max(0, need - eq_before)) : 0;
  const int sel = gt + take_eq;
  int pos = block_excl_scan(sel, scan_tmp);
  if (cnt > 0)
    for (int t = t0; t < t1; ++t) {
      if (!eligible(sk[t])) continue;
      const unsigned long long k = sk[t] & mask;
      bool take = k > pref;
      if (!take && k == pref && take_eq > 0) {
        take = true;
        --take_eq;
      }
      if (take) out[pos++] = s_end + t;
    }
  if (tid == 0) {
    *count = cnt;
    if (flag_in) *flag_out = *flag_in;
  }
}

// Attention selector, a group of layers, in two kernels over a workspace.  The
// stale pool keys are written by no kernel of the pass and the span's queries
// of a group's layers are kept, so the scores of many layers run in one launch,
// where one layer's fill the chip for a few us and wait out their latencies
// for twenty.  The queries of kv group g are the span rows' heads hh with
// hh / (H/G) == g; within the group a query is ql = r * (H/G) + (hh mod H/G),
// globally qg = g * S * (H/G) + ql.  blockIdx.z is layer-major: query tile
// z % n_qtiles of layer layer0 + z / n_qtiles, whose arrays lie NQ apart.  A CTA
// of k_attn_select_logits takes SEL_QT queries of one group and some chunks of
// SEL_KC pool keys, the next chunk's keys in flight while one is computed: a
// chunk's keys are read once into shared memory and serve every query of the
// tile (so a group's key rows leave L2 once per query tile, not once per query).
// It stores the scaled logits, logit[qg * stride + (j - s_end)], and per query
// the chunk's max and sum of exp(logit - max); the last CTA of (group, query tile)
// to finish folds the chunk statistics into the pool softmax's max and 1 / sum.
// Arrival is an atomic count with no waiting: every other CTA just exits.  The contraction
// runs on mma.sync for bf16 caches and on FFMA micro-tiles for fp32 caches.
// Eight layers of 8 span rows and 2,492 keys: 69 us for both kernels with a CTA
// per chunk, run-time head sizes and scalar fragment loads, 45 now; mma.sync
// itself, twice for the split queries, takes 14 of it and the 41 MB of keys 6.
constexpr int SEL_KC = 64, SEL_QT = 32, SEL_THREADS = 128;
constexpr int SEL_KG = SEL_KC / 4;   // fp32 path: key groups of 4 (a thread: 4 queries x 4 keys)
constexpr int SEL_LTS = SEL_KC + 4;  // logits tile row stride (floats)
constexpr int SEL_FOLD = 16;         // chunk statistics in flight per thread in the fold
static_assert(SEL_KG * (SEL_QT / 4) == SEL_THREADS, "one 4x4 micro-tile per thread");

struct SelWs {
  float *logit;  // [layers][S*H][sel_stride(c)]
  float2 *ml;    // [layers][S*H][n_chunks] chunk (max, sum of exp)
  float2 *mz;    // [layers][S*H] pool (max, 1 / sum of exp)
  int *cnt;      // [layers][G][n_qtiles] arrivals
};

__host__ __device__ inline int sel_chunks(int c) { return (c + SEL_KC - 1) / SEL_KC; }
inline int sel_stride(int c) { return (c + 3) / 4 * 4; }  // logit rows on 16-byte boundaries

// (m, z) <- the (max, sum of exp) of the union of two sets, either possibly
// empty (m = -inf, z = 0).  Symmetric in its operands, bit for bit.
__device__ __forceinline__ void lse_merge(float &m, float &z, float m2, float z2) {
  if (m2 == -INFINITY) return;
  if (m == -INFINITY) {
    m = m2, z = z2;
    return;
  }
  const float mm = fmaxf(m, m2);
  z = z * expf(m - mm) + z2 * expf(m2 - mm);
  m = mm;
}

__device__ __forceinline__ uint32_t bf2_bits(__nv_bfloat162 v) { return *(const uint32_t *)&v; }

// d[0..3] += A (16 x 16, row) . B (16 x 8, col), bf16 operands, fp32 accumulate
__device__ __forceinline__ void sel_mma_bf16(float *d, uint32_t a0, uint32_t a1, uint32_t a2,
                                             uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// Four 8 x 8 matrices of 16-bit elements, lane l's address the row l % 8 of matrix l / 8.
__device__ __forceinline__ void sel_ldmatrix(uint32_t *r, const __nv_bfloat16 *row) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(row)));
}

template <typename T, int DH>
__global__ void __launch_bounds__(SEL_THREADS, sizeof(T) == 2 ? 6 : 4)
    k_attn_select_logits(const float *q, int S, int H, int G, int layer0, int n_qt, KVView v,
                         int s_end, int c, int cs, float scale, SelWs ws) {
  constexpr bool BF16 = sizeof(T) == 2;
  TraceScope ts(TK_SELECT);
  pdl_trigger();
  const int g = blockIdx.y, nch = sel_chunks(c);
  const int li = blockIdx.z / n_qt, qt = blockIdx.z - li * n_qt, layer = layer0 + li;
  const int hpg = H / G, Nq = S * hpg;
  {  // this layer's queries and arrays
    const size_t NQ = (size_t)S * H;
    q += li * NQ * DH;
    ws.logit += li * NQ * cs;
    ws.ml += li * NQ * nch;
    ws.mz += li * NQ;
    ws.cnt += (size_t)li * G * n_qt;
  }
  const int q0 = qt * SEL_QT, nq = min(SEL_QT, Nq - q0);
  const int tid = threadIdx.x;
  const size_t qg0 = (size_t)g * Nq + q0;
  extern __shared__ float4 sel_smem[];
  // bf16 keys: tensor cores (mma.sync m16n8k16, fp32 accumulate).  Each query is
  // split into two bf16 parts, q = q_hi + q_lo with q_lo the rounding
  // remainder, and logit = q_hi . k + q_lo . k: about 16 bits of q's mantissa,
  // the keys exact.  Rows are d-contiguous with a stride of dh + 8 elements (4
  // mod 32 words), so a fragment load's 8 rows x 4 lanes fall on 32 banks.
  // fp32 keys: FFMA micro-tiles.  Both operands transposed, d-major: the thread
  // of micro-tile (queries 4qg.., keys 4kg..) reads one float4 of each per d.
  constexpr int RS = DH + 8;
  __nv_bfloat16 *qh = (__nv_bfloat16 *)sel_smem;  // bf16: [SEL_QT][RS]
  __nv_bfloat16 *qo = qh + SEL_QT * RS;           // [SEL_QT][RS] the remainders
  __nv_bfloat16 *ks = qo + SEL_QT * RS;           // [SEL_KC][RS]
  float *qT = (float *)sel_smem;                  // fp32: [DH][SEL_QT]
  float *kT = qT + DH * SEL_QT;                   // [DH][SEL_KC]
  float *lt = BF16 ? (float *)ks : kT;  // [SEL_QT][SEL_LTS] logits, over the keys once consumed
  int *last = (int *)sel_smem;          // arrival flag, over the queries at the end

  // A chunk's stale keys (no kernel of the pass writes them, so the first
  // chunk's are read before the wait on the predecessor): all loads (page
  // lookups, then rows) are issued before the first is used.
  constexpr int EPV = 16 / (int)sizeof(T);  // elements per 16-byte load
  constexpr int L = DH / EPV;               // 16-byte pieces per key row
  constexpr int KLD = SEL_KC * L / SEL_THREADS;
  uint4 kx[KLD];
  // lanes: along a row (bf16), or consecutive keys (fp32, stored transposed)
  auto key = [&](int i) { return BF16 ? i / L : i % SEL_KC; };
  auto piece = [&](int i) { return BF16 ? i % L : i / SEL_KC; };
  auto load_keys = [&](int t0) {
    const T *kc = (const T *)v.pages;
#pragma unroll
    for (int u = 0; u < KLD; ++u) {
      const int i = tid + u * SEL_THREADS, kk = key(i), sub = piece(i);
      kx[u] = make_uint4(0u, 0u, 0u, 0u);
      if (kk < min(SEL_KC, c - t0))
        kx[u] = *(const uint4 *)(kc + v.offset(layer, 0, g, s_end + t0 + kk) + sub * EPV);
    }
  };
  auto store_keys = [&]() {
#pragma unroll
    for (int u = 0; u < KLD; ++u) {
      const int i = tid + u * SEL_THREADS, kk = key(i), sub = piece(i);
      if constexpr (BF16) {
        *(uint4 *)(ks + kk * RS + sub * 8) = kx[u];  // rows of 16-byte multiples
      } else {
        const float *f = (const float *)&kx[u];
#pragma unroll
        for (int e = 0; e < EPV; ++e) kT[(sub * EPV + e) * SEL_KC + kk] = f[e];
      }
    }
  };
  load_keys(blockIdx.x * SEL_KC);
  pdl_wait();  // the queries come from the RoPE kernels before
  ts.waited();
  {
    constexpr int D4 = DH / 4, QLD = SEL_QT * D4 / SEL_THREADS;
    // lanes: along a row (bf16), or consecutive queries (fp32)
    auto query = [&](int i) { return BF16 ? i / D4 : i % SEL_QT; };
    auto quad = [&](int i) { return BF16 ? i % D4 : i / SEL_QT; };
    float4 qx[QLD];
#pragma unroll
    for (int u = 0; u < QLD; ++u) {
      const int i = tid + u * SEL_THREADS, ql = query(i), d4 = quad(i);
      qx[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (ql < nq) {
        const int qq = q0 + ql, r = qq / hpg, hh = g * hpg + qq % hpg;
        qx[u] = *(const float4 *)(q + ((size_t)r * H + hh) * DH + 4 * d4);
      }
    }
#pragma unroll
    for (int u = 0; u < QLD; ++u) {
      const int i = tid + u * SEL_THREADS, ql = query(i), d4 = quad(i);
      if constexpr (BF16) {
        const float2 x01 = make_float2(qx[u].x, qx[u].y), x23 = make_float2(qx[u].z, qx[u].w);
        const __nv_bfloat162 h01 = __float22bfloat162_rn(x01), h23 = __float22bfloat162_rn(x23);
        const float2 f01 = __bfloat1622float2(h01), f23 = __bfloat1622float2(h23);
        const __nv_bfloat162 l01 = __floats2bfloat162_rn(x01.x - f01.x, x01.y - f01.y);
        const __nv_bfloat162 l23 = __floats2bfloat162_rn(x23.x - f23.x, x23.y - f23.y);
        *(uint2 *)(qh + ql * RS + 4 * d4) = make_uint2(bf2_bits(h01), bf2_bits(h23));
        *(uint2 *)(qo + ql * RS + 4 * d4) = make_uint2(bf2_bits(l01), bf2_bits(l23));
      } else {
        float *dst = qT + 4 * d4 * SEL_QT + ql;
        dst[0] = qx[u].x;
        dst[SEL_QT] = qx[u].y;
        dst[2 * SEL_QT] = qx[u].z;
        dst[3 * SEL_QT] = qx[u].w;
      }
    }
  }
  const int ql = tid >> 2, o = tid & 3;  // of the statistics: 4 threads per query
  for (int chunk = blockIdx.x; chunk < nch; chunk += gridDim.x) {
    const int t0 = chunk * SEL_KC, nk = min(SEL_KC, c - t0);
    store_keys();
    __syncthreads();
    if (tid == 0) trace_mark(0);  // keys and queries staged
    // the next chunk's keys travel while this one is computed
    if (chunk + (int)gridDim.x < nch) load_keys((chunk + gridDim.x) * SEL_KC);
    if constexpr (BF16) {
      // warp w: keys 16w .. 16w + 15 (two n-tiles of 8), all SEL_QT queries
      // (two m-tiles of 16); lane: group gr = lane / 4, pair column gc
      const int warp = tid >> 5, lane = tid & 31, gr = lane >> 2, gc = (lane & 3) * 2;
      static_assert(SEL_QT == 32 && SEL_KC == 16 * (SEL_THREADS / 32), "warp tiling");
      float acc[2][2][4];
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[mt][nt][e] = 0.f;
      const __nv_bfloat16 *ka = ks + (16 * warp + 8 * (lane >> 4) + (lane & 7)) * RS + (lane & 8);
      const __nv_bfloat16 *qa = qh + (lane & 15) * RS + (lane >> 4) * 8;
#pragma unroll
      for (int k0 = 0; k0 < DH; k0 += 16) {
        uint32_t b[4];
        sel_ldmatrix(b, ka + k0);  // both n-tiles, d k0 .. +7 and +8 .. +15
#pragma unroll
        for (int mt = 0; mt < 2; ++mt)
#pragma unroll
          for (int part = 0; part < 2; ++part) {
            uint32_t a[4];
            sel_ldmatrix(a, qa + (part * SEL_QT + 16 * mt) * RS + k0);
#pragma unroll
            for (int nt = 0; nt < 2; ++nt)
              sel_mma_bf16(acc[mt][nt], a[0], a[1], a[2], a[3], b[2 * nt], b[2 * nt + 1]);
          }
      }
      __syncthreads();  // keys consumed: lt reuses their space
      if (tid == 0) trace_mark(1);  // logits computed
#pragma unroll
      for (int mt = 0; mt < 2; ++mt)
#pragma unroll
        for (int nt = 0; nt < 2; ++nt)
#pragma unroll
          for (int e = 0; e < 4; e += 2) {  // a pair of keys; a row's last one may be padding
            const int qq = 16 * mt + gr + e * 4, kk = 16 * warp + 8 * nt + gc;
            const float2 l = make_float2(acc[mt][nt][e] * scale, acc[mt][nt][e + 1] * scale);
            *(float2 *)(lt + qq * SEL_LTS + kk) =
                make_float2(kk < nk ? l.x : -INFINITY, kk + 1 < nk ? l.y : -INFINITY);
            if (kk < nk && qq < nq) *(float2 *)(ws.logit + (qg0 + qq) * cs + t0 + kk) = l;
          }
    } else {
      const int kg = tid % SEL_KG, qg = tid / SEL_KG;
      float acc[4][4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
#pragma unroll 4
      for (int d = 0; d < DH; ++d) {
        const float4 a = *(const float4 *)(qT + d * SEL_QT + 4 * qg);
        const float4 b = *(const float4 *)(kT + d * SEL_KC + 4 * kg);
        const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
      }
      __syncthreads();  // keys consumed: lt reuses their space
      if (tid == 0) trace_mark(1);  // logits computed
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int qq = 4 * qg + i;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int kk = 4 * kg + j;
          const float l = acc[i][j] * scale;
          lt[qq * SEL_LTS + kk] = kk < nk ? l : -INFINITY;
          if (kk < nk && qq < nq) ws.logit[(qg0 + qq) * cs + t0 + kk] = l;
        }
      }
    }
    __syncthreads();
    // chunk statistics: keys o, o + 4, ... of a query (the row stride SEL_LTS = 4
    // mod 32 puts a warp's 8 queries x 4 lanes on 32 banks)
    const float *row = lt + ql * SEL_LTS;
    float mx = -INFINITY;
#pragma unroll
    for (int j = 0; j < SEL_KC / 4; ++j) mx = fmaxf(mx, row[o + 4 * j]);
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    float z = 0.f;  // key 0 is valid: mx is finite
#pragma unroll
    for (int j = 0; j < SEL_KC / 4; ++j) z += expf(row[o + 4 * j] - mx);
    z += __shfl_xor_sync(0xffffffffu, z, 2);
    z += __shfl_xor_sync(0xffffffffu, z, 1);
    if (o == 0 && ql < nq) ws.ml[(qg0 + ql) * nch + chunk] = make_float2(mx, z);
    __syncthreads();  // lt consumed: the next chunk's keys take its place
  }
  __threadfence();
  __syncthreads();
  if (tid == 0) trace_mark(2);  // chunk statistics stored
  int *cnt = ws.cnt + (size_t)g * n_qt + qt;
  if (tid == 0) *last = atomicAdd(cnt, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (tid == 0) trace_mark(3);  // arrival counted
  if (!*last) return;
  if (tid == 0) *cnt = 0;  // ready for the next launch
  __threadfence();
  // fold: 4 threads per query, each over chunks o, o + 4, ... (SEL_FOLD
  // loads in flight), then the quad
  float mx = -INFINITY, z = 0.f;
  if (ql < nq) {
    const float2 *row = ws.ml + (qg0 + ql) * nch;
    for (int base = o; base < nch; base += 4 * SEL_FOLD) {
      float2 x[SEL_FOLD];
#pragma unroll
      for (int j = 0; j < SEL_FOLD; ++j) {
        const int ch = base + 4 * j;
        x[j] = ch < nch ? __ldcg(row + ch) : make_float2(-INFINITY, 0.f);
      }
#pragma unroll
      for (int j = 0; j < SEL_FOLD; ++j) lse_merge(mx, z, x[j].x, x[j].y);
    }
  }
#pragma unroll
  for (int off = 2; off > 0; off >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, mx, off);
    const float z2 = __shfl_xor_sync(0xffffffffu, z, off);
    lse_merge(mx, z, m2, z2);
  }
  if (o == 0 && ql < nq) ws.mz[qg0 + ql] = make_float2(mx, 1.0f / z);
  if (tid == 0) trace_mark(4);  // fold done (last CTA of the group)
}

// tot[layer][t] = sum over the S*H queries of exp(logit - max) / sum, in a fixed
// order: a CTA takes 16 * VEC keys of a layer, VEC a thread; its ACC_SLICES
// thread slices sum interleaved sets of the queries, then one thread per key
// adds the slice sums in slice order (the same for every VEC).  Bound by the
// exponentials' latency, so by the warps on the chip: VEC 4 reads logits and
// statistics in a quarter of the loads where a group's launch fills the SMs
// (4 layers, 10,900 keys, 8 rows of 32 heads: a selection 464 us, 475 with VEC 1), but of
// one layer's 2,000 or 2,500 keys it has 32 or 39 CTAs (4 layers, 200 rows: 1013 and
// 1100 us, 963 and 1054 with VEC 1).
constexpr int ACC_LANES = 16, ACC_SLICES = 32;
template <int VEC>
__global__ void __launch_bounds__(ACC_LANES * ACC_SLICES)
    k_attn_select_accum(const float *logit, const float2 *mz, int NQ, int c, int cs, float *tot) {
  using V = std::conditional_t<VEC == 4, float4, std::conditional_t<VEC == 2, float2, float>>;
  constexpr int KEYS = ACC_LANES * VEC;
  TraceScope ts(TK_SELECT_ACC);
  pdl_trigger();
  __shared__ V part[ACC_SLICES][ACC_LANES];
  const int kq = threadIdx.x % ACC_LANES, sl = threadIdx.x / ACC_LANES;
  const int t = blockIdx.x * KEYS + VEC * kq;
  logit += (size_t)blockIdx.y * NQ * cs;
  mz += (size_t)blockIdx.y * NQ;
  pdl_wait();  // logits and softmax statistics of the kernel before
  alignas(16) float s[VEC] = {};
  if (t < c) {  // a row's last quad may end in its padding: sums that nobody takes
#pragma unroll 8
    for (int qg = sl; qg < NQ; qg += ACC_SLICES) {
      const float2 st = mz[qg];
      const V lv = *(const V *)(logit + (size_t)qg * cs + t);
      const float *l = (const float *)&lv;
#pragma unroll
      for (int e = 0; e < VEC; ++e) s[e] += expf(l[e] - st.x) * st.y;
    }
  }
  part[sl][kq] = *(const V *)s;
  __syncthreads();
  const int k = threadIdx.x, tk = blockIdx.x * KEYS + k;
  if (k < KEYS && tk < c) {
    float sum = 0.f;
#pragma unroll
    for (int i = 0; i < ACC_SLICES; ++i) sum += ((const float *)part[i])[k];
    tot[(size_t)blockIdx.y * c + tk] = sum;
  }
}

// Keys of the layers' sums, added in layer order.
__global__ void k_layer_sum_keys(const float *tot, int layers, int c, unsigned long long *keys) {
  pdl_trigger();
  pdl_wait();
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < c; t += gridDim.x * blockDim.x) {
    float s = 0.f;
#pragma unroll 8
    for (int l = 0; l < layers; ++l) s += tot[(size_t)l * c + t];
    keys[t] = (unsigned long long)ord_f32(s) + 1ull;
  }
}

// CacheBlend deviation: fresh layer-1 k (RoPE at the row's position) and v
// from qkv, rounded to the cache dtype, against the stale cache entries:
// score[pos] = ||dk||_2 + ||dv||_2 over all kv heads and dims.
template <typename T>
__global__ void __launch_bounds__(256)
    k_kv_deviation(const float *qkv, const float2 *rope, const int32_t *pos, int H, int G, int dh,
                   KVView v, float *score) {
  int i = blockIdx.x;
  int p = pos[i];
  int half = dh / 2, Nqkv = (H + 2 * G) * dh;
  const float *x = qkv + (size_t)i * Nqkv;
  const T *c = (const T *)v.pages;
  float dk = 0.f, dv = 0.f;
  for (int e = threadIdx.x; e < G * half; e += blockDim.x) {
    int g = e / half, t = e % half;
    float2 cs = rope[(size_t)p * half + t];
    float k1 = x[(H + g) * dh + t], k2 = x[(H + g) * dh + t + half];
    float r1 = k1 * cs.x - k2 * cs.y, r2 = k2 * cs.x + k1 * cs.y;
    float v1 = x[(H + G + g) * dh + t], v2 = x[(H + G + g) * dh + t + half];
    size_t ko = v.offset(1, 0, g, p), vo = v.offset(1, 1, g, p);
    float sk1, sk2, sv1, sv2;
    if constexpr (sizeof(T) == 2) {
      r1 = __bfloat162float(__float2bfloat16_rn(r1));
      r2 = __bfloat162float(__float2bfloat16_rn(r2));
      v1 = __bfloat162float(__float2bfloat16_rn(v1));
      v2 = __bfloat162float(__float2bfloat16_rn(v2));
      sk1 = __bfloat162float(c[ko + t]);
      sk2 = __bfloat162float(c[ko + t + half]);
      sv1 = __bfloat162float(c[vo + t]);
      sv2 = __bfloat162float(c[vo + t + half]);
    } else {
      sk1 = c[ko + t];
      sk2 = c[ko + t + half];
      sv1 = c[vo + t];
      sv2 = c[vo + t + half];
    }
    dk += (r1 - sk1) * (r1 - sk1) + (r2 - sk2) * (r2 - sk2);
    dv += (v1 - sv1) * (v1 - sv1) + (v2 - sv2) * (v2 - sv2);
  }
  __shared__ float rk[32], rv[32];
  for (int off = 16; off > 0; off >>= 1) {
    dk += __shfl_xor_sync(0xffffffffu, dk, off);
    dv += __shfl_xor_sync(0xffffffffu, dv, off);
  }
  if ((threadIdx.x & 31) == 0) {
    rk[threadIdx.x >> 5] = dk;
    rv[threadIdx.x >> 5] = dv;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    float a = 0.f, b = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      a += rk[w];
      b += rv[w];
    }
    score[p] = sqrtf(a) + sqrtf(b);
  }
}

int grid_for(int n, int block) {
  int g = (n + block - 1) / block;
  return g < 1 ? 1 : (g > 4096 ? 4096 : g);
}

}  // namespace

void launch_float_keys(const float *scores, int n, int s_end, unsigned long long *keys,
                       cudaStream_t s) {
  int c = n - s_end;
  if (c <= 0) return;
  k_float_keys<<<grid_for(c, 256), 256, 0, s>>>(scores, n, s_end, keys);
}

// Top-K over c = n - s_end candidates (c <= 16384).  nonzero_only is
// encoded in the sign of K: K < 0 means "only nonzero keys are eligible".
// Returns nullptr on success, else what failed.
const char *launch_topk(const unsigned long long *keys, int n, int s_end, int K, int32_t *out,
                        int32_t *count, cudaStream_t s, const SimpleKeys &gen,
                        const int *flag_in, int32_t *flag_out) {
  int c = n - s_end;
  int nonzero_only = K < 0 ? 1 : 0;
  if (K < 0) K = -K;
  if (c < 0) c = 0;
  size_t smem = (size_t)c * sizeof(unsigned long long);
  if (smem >= 32 * 1024) {  // the default 48 KB limit also covers static shared memory
    static PerDevice<size_t> limit;
    if (const char *e = smem_opt_in(limit, k_topk, smem)) return e;
  }
  k_topk<<<1, TOPK_THREADS, smem, s>>>(keys, c, s_end, K, nonzero_only, out, count, gen,
                                       flag_in, flag_out);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? nullptr : cudaGetErrorString(e);
}

namespace {
struct SelLayout {
  size_t q, tot, logit, ml, mz, cnt, total;  // byte offsets into the workspace
  int group;                                 // layers scored per launch
};
// The logits of a group of layers stay within SEL_GROUP_BYTES (about half of
// L2, from which the next kernel reads them), and so do its queries; at least one
// layer.
constexpr size_t SEL_GROUP_BYTES = (size_t)64 << 20;
SelLayout sel_layout(int S, const Dims &dm, int c) {
  auto al = [](size_t x) { return (x + 255) / 256 * 256; };
  const size_t NQ = (size_t)S * dm.H, nqt = ((size_t)S * (dm.H / dm.G) + SEL_QT - 1) / SEL_QT;
  const size_t cs = sel_stride(c);
  const size_t fit = SEL_GROUP_BYTES / (NQ * std::max<size_t>(cs, dm.dh) * sizeof(float));
  SelLayout o;
  o.group = fit < 1 ? 1 : fit < (size_t)dm.L ? (int)fit : dm.L;
  while (o.group > 1 && (size_t)o.group * nqt > 65535) --o.group;  // grid z
  o.q = 0;
  o.tot = o.q + al((size_t)o.group * NQ * dm.dh * sizeof(float));
  o.logit = o.tot + al((size_t)dm.L * c * sizeof(float));
  o.ml = o.logit + al(o.group * NQ * cs * sizeof(float));
  o.mz = o.ml + al(o.group * NQ * sel_chunks(c) * sizeof(float2));
  o.cnt = o.mz + al(o.group * NQ * sizeof(float2));
  o.total = o.cnt + al((size_t)o.group * dm.G * nqt * sizeof(int));
  return o;
}
}  // namespace

size_t attn_select_ws_bytes(int S, const Dims &dm, int n_pool) {
  return n_pool > 0 && S > 0 ? sel_layout(S, dm, n_pool).total : 0;
}

float *attn_select_queries(void *ws_base, int S, const Dims &dm, int n_pool, int layer) {
  const SelLayout o = sel_layout(S, dm, n_pool);
  // a group's queries take the last one's place: RoPE, which writes them, runs behind
  // that group's kernels
  return (float *)((char *)ws_base + o.q) + (size_t)(layer % o.group) * S * dm.H * dm.dh;
}

int launch_attn_select_scores(int S, const Dims &dm, int layer, KVView v, int s_end, int n,
                              void *ws_base, unsigned long long *keys, int num_sms,
                              cudaStream_t s) {
  const int c = n - s_end, cs = sel_stride(c);
  if (c <= 0 || S <= 0) return 0;
  const float scale = (float)(1.0 / sqrt((double)dm.dh));
  const SelLayout o = sel_layout(S, dm, c);
  if (layer + 1 < dm.L && (layer + 1) % o.group) return 0;  // the group's last layer scores it
  char *b = (char *)ws_base;
  SelWs ws{(float *)(b + o.logit), (float2 *)(b + o.ml), (float2 *)(b + o.mz), (int *)(b + o.cnt)};
  float *tot = (float *)(b + o.tot);
  const int nqt = (S * (dm.H / dm.G) + SEL_QT - 1) / SEL_QT;
  const int layer0 = layer / o.group * o.group, layers = layer - layer0 + 1;
  // arrival counts start at zero; each launch's last CTAs leave them at zero
  if (layer0 == 0) cudaMemsetAsync(ws.cnt, 0, (size_t)o.group * dm.G * nqt * sizeof(int), s);
  // bf16: q_hi, q_lo and keys as bf16 rows of dh + 8; fp32: q and keys as
  // fp32 columns of dh.  The logits tile reuses the keys' space.
  const bool bf16 = dm.dtype == KVR_DTYPE_BF16;
  const size_t q_b = bf16 ? (size_t)2 * SEL_QT * (dm.dh + 8) * 2 : (size_t)SEL_QT * dm.dh * 4;
  const size_t k_b = bf16 ? (size_t)SEL_KC * (dm.dh + 8) * 2 : (size_t)SEL_KC * dm.dh * 4;
  const size_t lt_b = (size_t)SEL_QT * SEL_LTS * sizeof(float);
  const size_t smem = q_b + (k_b > lt_b ? k_b : lt_b);  // 34 KB (bf16), 48 KB (fp32) at dh 128
  auto kern = dm.dh == 128 ? (bf16 ? k_attn_select_logits<__nv_bfloat16, 128>
                                   : k_attn_select_logits<float, 128>)
                           : (bf16 ? k_attn_select_logits<__nv_bfloat16, 64>
                                   : k_attn_select_logits<float, 64>);
  // fp32 at dh 128, plus the trace build's static shared memory, passes 48 KB
  static PerDevice<size_t> limit[2][2];  // (an error shows at the launch)
  smem_opt_in(limit[bf16][dm.dh == 128], kern, smem);
  // one wave: the chunks spread evenly over the CTAs that fit at once
  const int nch = sel_chunks(c), fit = (bf16 ? 6 : 4) * num_sms / (dm.G * nqt * layers);
  const int per = fit < 1 ? nch : (nch + fit - 1) / fit;
  const dim3 grid((nch + per - 1) / per, dm.G, nqt * layers);
  launch_pdl(kern, grid, SEL_THREADS, smem, s,
             (const float *)attn_select_queries(ws_base, S, dm, c, layer0), S, dm.H, dm.G,
             layer0, nqt, v, s_end, c, cs, scale, ws);
  auto accum = [&](auto kernel, int keys) {
    launch_pdl(kernel, dim3((c + keys - 1) / keys, layers), ACC_LANES * ACC_SLICES, 0, s,
               (const float *)ws.logit, (const float2 *)ws.mz, S * dm.H, c, cs,
               tot + (size_t)layer0 * c);
  };
  if ((c + 63) / 64 * layers >= num_sms)  // an SM each at least
    accum(k_attn_select_accum<4>, 64);
  else
    accum(k_attn_select_accum<1>, 16);
  if (layer + 1 < dm.L) return 2;
  launch_pdl(k_layer_sum_keys, grid_for(c, 256), 256, 0, s, (const float *)tot, dm.L, c, keys);
  return 3;
}

void launch_kv_deviation(const float *qkv, const float2 *rope, const int32_t *pos, int M,
                         const Dims &dm, KVView v, float *scores, cudaStream_t s) {
  if (M <= 0) return;
  if (dm.dtype == KVR_DTYPE_BF16)
    k_kv_deviation<__nv_bfloat16><<<M, 256, 0, s>>>(qkv, rope, pos, dm.H, dm.G, dm.dh, v, scores);
  else
    k_kv_deviation<float><<<M, 256, 0, s>>>(qkv, rope, pos, dm.H, dm.G, dm.dh, v, scores);
}

KVR_TRACE_ATTACH(trace_attach_select)

}  // namespace kvr
