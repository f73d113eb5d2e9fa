// k_attn_pair.cu -- scattered-query causal GQA attention of many rows on the
// tcgen05 tensor cores (sm_103a), bf16 cache, head_dim 64 or 128: two query
// tiles per CTA share every K and V tile.
//
// A CTA owns a pair of query tiles -- each up to 128 query vectors (rows of one
// document times the grp query heads of KV head g), the M = 128 rows of the
// MMA -- and a contiguous range of 64-key pages, taken two pages (128 keys) at
// a time.  Per step and tile:
//   S = Q K^T   M 128 x N 128 x K head_dim, Q and K from shared memory, S in
//               TMEM;
//   softmax     eight warps a tile, two threads per query vector, each with
//               half of the step's keys; causal mask key <= position;
//               exponentials against an integer reference maximum that is
//               raised (and O rescaled by a power of two) only when the
//               running maximum exceeds it by more than 8, so the two halves
//               need no common maximum but only to know whether either one
//               grew (one barrier with a reduction); P in bf16 written over
//               the first columns of the half's S;
//   O += P V    M 128 x N head_dim x K 128, P from TMEM, V MN-major straight
//               from the page layout.
// The MMA warp issues P V of tile t for step i - 1, then S of tile t for step i
// (S and P share columns, and MMAs run in issue order), and turns to the
// other tile: while one tile's softmax runs, the tensor cores work for the
// other.
//
// What bounds it: with one tile per CTA the chain S -> softmax -> P V of a
// 64-key chunk took 1.08 us, against 0.28 us of MMA, and nothing filled the
// gaps.  Two tiles fill each other's, and a step of 128 keys halves the
// hand-offs: 4096 rows over their own keys, 32 heads of 128, went from 236 to
// 125 us (0.58 to 1.10 PFLOP/s), tensor pipe 20 to 51% active.  A step takes
// about 2.0 us: its softmax 0.7 (MUFU 0.27 of it), the hand-offs and the issue
// of 32 MMAs the rest.  Also measured, for the same rows: one thread per query
// vector 155 us, a half row of scores held in registers throughout (92 bytes
// of spills) 139, one MMA warp per tile 129.
#include <math.h>

#include "kvr_internal.cuh"
#include "tc_ptx.cuh"

namespace kvr {
namespace {
using namespace ptx;

constexpr int QV = 128;             // query vectors per tile (UMMA M)
constexpr int PG = KVR_PAGE;        // keys per page
constexpr int CH = 2 * PG;          // keys per step
constexpr int KP = 2;               // threads per query vector, each with CH / KP of a step's keys
constexpr int SM_WARPS = 8 * KP;    // softmax warps: KP per tile and TMEM lane quarter
constexpr int NT = 64 + 32 * SM_WARPS;
constexpr int WS_MAXQ = 192;        // query slots per (split, block, head) of the split workspace
constexpr int NSLOT = 4;            // K and V tiles in flight (K0 V0 K1 V1 ...)
constexpr int NB = 4;               // barriers of the ring's groups: K0, (V0, K1), (V1, K2), ...
constexpr uint32_t TMEM_COLS = 512;  // S0, S1 (128 columns each; P over the first half), O0, O1
constexpr float RESCALE_LOG2 = 8.f;  // headroom of the reference maximum (P <= 2^8)

struct PairParams {
  const __nv_bfloat16 *q;  // [M][H * dh] post-RoPE
  float qk_scale;          // log2(e) / sqrt(dh): scores into the log2 domain
  const int32_t *pos;      // [M] ascending per document
  const int4 *blocks;      // tiles: (row0, nrows, kmax, doc)
  const int4 *pairs;       // (first tile, tiles: 1 or 2, kmax of the pair, doc)
  const int32_t *table;    // one document: logical page -> physical page
  const KVView *views;     // several: views and TMA views indexed by document
  const CUtensorMap *tmaps;
  int H, G, grp, layer, L;
  int n_splits, n_blocks;
  float *ws_o;    // [n_splits][n_blocks][G][WS_MAXQ][dh]
  float2 *ws_ml;  // [n_splits][n_blocks][G][WS_MAXQ]
  __nv_bfloat16 *out;  // [M][H * dh]
  int *dev_flag;
};

// A from tensor memory (row m in lane m, two bf16 of K per column), B a
// shared-memory descriptor.
__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b,
                                            uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

// 8 consecutive 32-bit TMEM columns, one lane per thread, without the wait.
__device__ __forceinline__ void tmem_st8_nowait(uint32_t taddr, const uint32_t *r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *(uint32_t *)&v;
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// (x0, x1) * s + c and a + b on pairs of fp32 (one instruction each)
__device__ __forceinline__ void fma2(float &y0, float &y1, uint32_t x0, uint32_t x1, float s,
                                     float c) {
  asm("{\n\t.reg .b64 x, s, c, y;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 s, {%4, %4};\n\t"
      "mov.b64 c, {%5, %5};\n\tfma.rn.f32x2 y, x, s, c;\n\tmov.b64 {%0, %1}, y;\n\t}"
      : "=f"(y0), "=f"(y1)
      : "r"(x0), "r"(x1), "f"(s), "f"(c));
}
__device__ __forceinline__ void add2(float &a0, float &a1, float b0, float b1) {
  asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%0, %1};\n\tmov.b64 b, {%2, %3};\n\t"
      "add.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}"
      : "+f"(a0), "+f"(a1)
      : "f"(b0), "f"(b1));
}

template <int DH>
__global__ void __launch_bounds__(NT, 1)
    k_attn_pair(const __grid_constant__ CUtensorMap tm_kv, const PairParams p) {
  constexpr int HALVES = DH / 64;                    // 128-byte column blocks of a row
  constexpr uint32_t HB = CH * 128;                  // one column block of a K (or V) tile
  constexpr uint32_t TBYTES = HB * HALVES;           // one K (or V) tile of 128 keys
  constexpr uint32_t QHB = QV * 128;                 // one column block of a Q tile
  constexpr uint32_t QBYTES = QHB * HALVES;          // one Q tile
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t full[NB], empty[NB], s_full[2], p_full[2], o_done[2],
      q_full, drain_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_f;
  // per tile: a row's maximum (a growing step), then its sum, handed over
  __shared__ float sx[2][QV];

  TraceScope ts(TK_ATTN);
  const int split = blockIdx.x, g = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // block and pair tables, positions and page table are written before the pass
  const int4 pr = p.pairs[blockIdx.z];
  const int nt = pr.y;  // tiles of this pair
  // pages [c0, c1) of this split; a tile stops at its own last page
  const int n_pages = pr.z / PG + 1;
  const int cps = (n_pages + p.n_splits - 1) / p.n_splits;
  const int c0 = split * cps, c1 = min(n_pages, c0 + cps);
  if (c0 >= c1) {  // empty split: the combine skips it
    pdl_trigger();
    return;
  }
  // steps of each tile (tile 0 holds the earlier rows: never more than tile 1)
  auto steps_of = [&](int t) {
    const int e = min(c1, p.blocks[pr.x + t].z / PG + 1);
    return e > c0 ? (e - c0 + 1) / 2 : 0;
  };
  const int n0 = steps_of(0), n1 = nt > 1 ? steps_of(1) : 0, n_steps = max(n0, n1);
  const uint32_t base = (su32(smem_raw) + 1023u) & ~1023u;
  const uint32_t sQ = base, sKV = base + 2 * QBYTES;
  volatile int *abort_v = &abort_f;

  if (tid == 0) {
    for (int b = 0; b < NB; ++b) {
      mbar_init(&full[b], 1);
      mbar_init(&empty[b], 1);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(&s_full[t], 1);
      mbar_init(&p_full[t], SM_WARPS / 2);
      mbar_init(&o_done[t], 1);
    }
    mbar_init(&q_full, SM_WARPS);
    mbar_init(&drain_bar, 1);
    abort_f = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(&tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  // Dependents may launch once this CTA holds its TMEM: no other kernel that
  // allocates TMEM fits beside it on an SM (registers), so the allocation
  // cannot wait on a CTA that waits on this grid.
  pdl_trigger();

  if (warp == 0) {
    // ------------------------------------------------------------ TMA
    const int32_t *table = p.views ? p.views[pr.w].table : p.table;
    const CUtensorMap *tmap = p.tmaps ? p.tmaps + pr.w : &tm_kv;
    if (lane == 0) {
      // a tensor map in global memory is read through the tensor-map proxy
      if (p.tmaps)
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(tmap)
                     : "memory");
      tma_prefetch_desc(tmap);
    }
    pdl_wait();
    ts.waited();
    int issued = 0, pg = 0;
    bool ok = true;
    for (int i = 0; i < n_steps && ok; ++i) {
      // 32 page-table entries at a time, one per lane; a step's second page
      // past the last one is the last again (its keys are masked)
      if ((i & 15) == 0) pg = table[min(c0 + 2 * i + lane, n_pages - 1)];
      const int pa = __shfl_sync(0xffffffffu, pg, (2 * i) & 31);
      const int pb = __shfl_sync(0xffffffffu, pg, (2 * i + 1) & 31);
      if (lane == 0) {
#pragma unroll
        for (int kv = 0; kv < 2; ++kv) {
          // tile j of the ring; group (j + 1) / 2 holds V of a step and K of the next
          const int j = 2 * i + kv, grp = (j + 1) >> 1;
          if (j >= NSLOT) {  // the tile that held this slot has been used
            const int e = (j - NSLOT + 1) >> 1;
            if (!mbar_wait(&empty[e % NB], (e / NB) & 1, abort_v, p.dev_flag, 64)) {
              ok = false;
              break;
            }
          }
          if (kv == 1 || i == 0)
            mbar_expect_tx(&full[grp % NB], kv == 1 && i + 1 < n_steps ? 2 * TBYTES : TBYTES);
          const long long ra = (((long long)pa * p.L + p.layer) * 2 + kv) * p.G + g;
          const long long rb = (((long long)pb * p.L + p.layer) * 2 + kv) * p.G + g;
#pragma unroll
          for (int h = 0; h < HALVES; ++h) {
            const uint32_t dst = sKV + (j % NSLOT) * TBYTES + h * HB;
            tma_load_2d((void *)__cvta_shared_to_generic(dst), tmap, &full[grp % NB], h * 64,
                        (int)(ra * PG));
            tma_load_2d((void *)__cvta_shared_to_generic(dst + PG * 128), tmap, &full[grp % NB],
                        h * 64, (int)(rb * PG));
          }
          ++issued;
        }
      }
      ok = __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
    }
    // copies in flight complete before the CTA may exit (a group cut short by
    // an abort, V without the next K, runs into the wait's bound)
    if (lane == 0 && issued)
      for (int e = max(0, (issued + 1) / 2 - NB + 1); e <= issued / 2; ++e)
        mbar_wait(&full[e % NB], (e / NB) & 1, abort_v, p.dev_flag, 0, false);
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA
    // The whole warp walks the loop and one elected lane issues, so the
    // operands stay in uniform registers.  A group of the ring (V of a step, K
    // of the next) is used in one go and released by one commit.
    const uint32_t id_s = idesc_bf16(QV, CH), id_o = idesc_bf16(QV, DH, 1);
    // descriptors built once; a slot, column block or K slice only moves the
    // start address (the descriptor's low field, address / 16)
    const uint64_t dq0 = sw128_desc(sQ), dk0 = sw128_desc(sKV),
                   dv0 = sw128_desc_mn(sKV, HB, 1024);
    auto wait = [&](uint64_t *bar, int parity, int code) -> bool {
      return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_v, p.dev_flag, code));
    };
    static_assert(HB == QHB, "Q and K column blocks have the same size");
    bool ok = wait(&q_full, 0, 65);
    for (int i = 0; i <= n_steps && ok; ++i) {
      ok = wait(&full[i % NB], (i / NB) & 1, 66);
      for (int t = 0; t < nt && ok; ++t) {
        const int n = t ? n1 : n0;
        const uint32_t tS = tmem + t * CH, tO = tmem + 2 * CH + t * CH;
        if (i > 0 && i <= n) ok = wait(&p_full[t], (i - 1) & 1, 68);
        if (!ok) break;
        tc_fence_after();
        if (elect_one()) {
          if (i > 0 && i <= n) {
            const uint64_t dv = dv0 + (uint64_t)((((2 * i - 1) % NSLOT) * TBYTES) >> 4);
#pragma unroll
            for (int kk = 0; kk < CH / 16; ++kk)
              mma_bf16_ts(tO, tS + (kk / (8 / KP)) * (CH / KP) + kk % (8 / KP) * 8,
                          dv + (uint64_t)((kk * 2048) >> 4), id_o, kk > 0 || i > 1 ? 1u : 0u);
            if (i == n) mma_commit(&o_done[t]);
          }
          if (i < n) {
            const uint64_t dq = dq0 + (uint64_t)((t * QBYTES) >> 4);
            const uint64_t dk = dk0 + (uint64_t)((((2 * i) % NSLOT) * TBYTES) >> 4);
#pragma unroll
            for (int kk = 0; kk < DH / 16; ++kk) {
              const uint64_t o = (uint64_t)(((kk >> 2) * HB + (kk & 3) * 32) >> 4);
              mma_bf16(tS, dq + o, dk + o, id_s, kk > 0 ? 1u : 0u);
            }
            mma_commit(&s_full[t]);
          }
          if (t == nt - 1) mma_commit(&empty[i % NB]);
        }
        __syncwarp();
      }
    }
    // every MMA issued here completes before TMEM is freed
    if (elect_one()) mma_commit(&drain_bar);
    __syncwarp();
    mbar_wait(&drain_bar, 0, abort_v, p.dev_flag, 0, false);
  } else {
    // ------------------------------------------------------------ softmax
    // Warps w and w + 4 of a tile share TMEM lane quarter w % 4: the same 32
    // query vectors, keys (and O columns) in two halves.  They meet at a named
    // barrier once a step, which both reach on every iteration -- also after
    // an abort, when they only skip their work -- so it can never wait on a
    // warp that has left.
    const int t = (warp - 2) / (4 * KP), part = ((warp - 2) >> 2) % KP;
    const int quarter = warp & 3;  // TMEM lanes 32 * quarter .. + 31
    const int v = quarter * 32 + lane;
    const bool have = t < nt;
    const int blk = pr.x + (have ? t : 0);
    const int4 bd = p.blocks[blk];
    const int mq = have ? bd.y * p.grp : 0;
    const bool real = v < mq;
    const int row = bd.x + (real ? v / p.grp : 0), hh = g * p.grp + (real ? v % p.grp : 0);
    // the last key this thread's row may see in this split; rows past the
    // tile's query vectors (Q zero, nothing stored) see key 0 like a real one
    const int lim = min(real ? p.pos[row] : 0, c1 * PG - 1);
    const int n = t ? n1 : n0;
    constexpr int HK = CH / KP;  // keys of this thread per step
    constexpr int OC = DH / KP;  // O columns of this thread
    const uint32_t tl = tmem + t * CH + ((uint32_t)(quarter * 32) << 16);
    const uint32_t tS = tl + part * HK, tO = tl + 2 * CH + part * OC;
    const int bar_id = 1 + t * 4 + quarter;
    auto pair_bar = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(bar_id) : "memory"); };
    // f(part 0's x, part 1's x) for both: part 0's through sx, the result back
    auto hand_over = [&](float x, auto f) {
      if (part == 0) sx[t][v] = x;
      pair_bar();
      if (part == 1) sx[t][v] = x = f(sx[t][v], x);
      pair_bar();
      return part == 0 ? sx[t][v] : x;
    };
    auto pair_any = [&](bool x) {
      int r;
      asm volatile(
          "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 q, %2, 0;\n\t"
          "barrier.cta.red.or.pred p, %1, 64, q;\n\tselp.s32 %0, 1, 0, p;\n\t}"
          : "=r"(r)
          : "r"(bar_id), "r"(x ? 1 : 0)
          : "memory");
      return r != 0;
    };
    pdl_wait();
    {  // half a row of Q into the swizzled tile: 128-byte rows, 16-byte pieces XORed by row
      constexpr int QP = DH / 8 / KP;  // 16-byte pieces of this thread
      const uint4 *src = (const uint4 *)(p.q + ((size_t)row * p.H + hh) * DH) + part * QP;
      uint4 x[QP];
#pragma unroll
      for (int k = 0; k < QP; ++k) x[k] = real ? src[k] : make_uint4(0u, 0u, 0u, 0u);
      const uint32_t q0 = sQ + t * QBYTES + v * 128;
#pragma unroll
      for (int k = 0; k < QP; ++k) {
        const int c = part * QP + k;
        *(uint4 *)__cvta_shared_to_generic(q0 + (c >> 3) * QHB + (((c & 7) ^ (v & 7)) << 4)) = x[k];
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&q_full);
    }
    float m = -INFINITY, l = 0.f;  // reference maximum, this half's sum of exponentials
    bool dead = false;             // warp-uniform: a wait ran out
    for (int i = 0; i < n; ++i) {
      const int key0 = (c0 + 2 * i) * PG + part * HK;
      if (!dead)
        dead = !__all_sync(0xffffffffu, mbar_wait(&s_full[t], i & 1, abort_v, p.dev_flag, 69));
      // The scores in parts of 32: the maximum of all parts first, then the
      // exponentials part by part, each read from TMEM again (the whole half
      // row in registers spilled, and a spill here costs a trip to L2).
      uint32_t s[32];
      float ms = -INFINITY;
      bool masked = false;
      auto load_scores = [&](int k) { tmem_ld32_nowait(tS + 32 * k, s); };
      auto mask_scores = [&](int k) {
        tmem_wait_ld();
        if (masked) {
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (key0 + 32 * k + j > lim) s[j] = 0xff800000u;  // -inf
        }
      };
      if (!dead) {
        tc_fence_after();
        // all but the last steps of a tile are causal for the whole warp
        masked = !__all_sync(0xffffffffu, key0 + HK - 1 <= lim);
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int k = HK / 32 - 1; k >= 0; --k) {  // part 0 last: it stays for the exponentials
          load_scores(k);
          mask_scores(k);
#pragma unroll
          for (int j = 0; j < 32; ++j) mx[j & 3] = fmaxf(mx[j & 3], __uint_as_float(s[j]));
        }
        // the scale is positive: the scaled maximum is the maximum scaled
        ms = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * p.qk_scale;
      }
      // Either half of a row of these 32 above its reference's headroom (the
      // first step, whose reference is -inf, always).
      if (pair_any(ms > m + RESCALE_LOG2)) {
        ms = hand_over(ms, [](float a, float b) { return fmaxf(a, b); });
        // (O += P V of the step before has landed: S of this one came after it)
        const bool grow = ms > m + RESCALE_LOG2;
        const float mn = ceilf(ms);
        const float alpha = grow ? ex2(m - mn) : 1.f;  // m = -inf: 0, and O is exactly zero
        if (!dead && i > 0) {
#pragma unroll
          for (int k = 0; k < OC / 16; ++k) {
            float o[16];
            tmem_ld16(tO + 16 * k, o);
#pragma unroll
            for (int j = 0; j < 16; ++j) o[j] *= alpha;
            tmem_st16(tO + 16 * k, o);
          }
        }
        l *= alpha;
        if (grow) m = mn;
      }
      if (dead) continue;
      // a row that has seen no key yet (another split's) keeps P = 0
      const float nm = m == -INFINITY ? 0.f : -m;
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int k = 0; k < HK / 32; ++k) {
        if (k) {
          load_scores(k);
          mask_scores(k);
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t w[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            float a, b;
            fma2(a, b, s[16 * h + 2 * j], s[16 * h + 2 * j + 1], p.qk_scale, nm);
            a = ex2(a);
            b = ex2(b);
            w[j] = pack2(a, b);
            add2(sum[2 * (j & 1)], sum[2 * (j & 1) + 1], a, b);
          }
          tmem_st8_nowait(tS + 16 * k + 8 * h, w);  // below the scores yet to be read
        }
      }
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_full[t]);
      l += (sum[0] + sum[1]) + (sum[2] + sum[3]);
    }
    if (n > 0 && !dead)
      dead = !__all_sync(0xffffffffu,
                         mbar_wait(&o_done[t], 0, abort_v, p.dev_flag, 71));
    // both halves' sums (same reference maximum), in key order
    const float lt = hand_over(l, [](float a, float b) { return a + b; });
    // O: TMEM -> registers -> this tile's Q space (free now; a warp stages and
    // reads back only its own half rows) -> global, 128 bytes of a row at a time
    if (have && !dead) {
      tc_fence_after();
      constexpr int RC = OC / 8;  // 16-byte pieces staged per row and warp
      uint8_t *st = (uint8_t *)__cvta_shared_to_generic(sQ + t * QBYTES) + part * OC * 2;
      auto piece = [&](int r, int c) {
        return (uint4 *)(st + r * (DH * 2) + ((c ^ (r & (RC - 1))) << 4));
      };
      const size_t bs = ((size_t)split * p.n_blocks + blk) * p.G + g;
      if (p.n_splits == 1) {
        const float inv = lt > 0.f ? 1.f / lt : 0.f;
#pragma unroll
        for (int k = 0; k < OC / 16; ++k) {
          uint32_t o[16], y[8];
          tmem_ld16_nowait(tO + 16 * k, o);
          tmem_wait_ld();
#pragma unroll
          for (int j = 0; j < 8; ++j)
            y[j] = pack2(__uint_as_float(o[2 * j]) * inv, __uint_as_float(o[2 * j + 1]) * inv);
          *piece(v, 2 * k) = make_uint4(y[0], y[1], y[2], y[3]);
          *piece(v, 2 * k + 1) = make_uint4(y[4], y[5], y[6], y[7]);
        }
        __syncwarp();
        for (int e = lane; e < 32 * RC; e += 32) {
          const int r = quarter * 32 + e / RC, c = e % RC;
          if (r < mq)
            *(uint4 *)(p.out + ((size_t)(bd.x + r / p.grp) * p.H + g * p.grp + r % p.grp) * DH +
                       part * OC + c * 8) = *piece(r, c);
        }
      } else {
        // unnormalised O and (max, sum) for the combine, DH / 4 columns at a time
        if (real && part == 0) p.ws_ml[bs * WS_MAXQ + v] = make_float2(m, lt);
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          if (half) __syncwarp();
#pragma unroll
          for (int k = 0; k < OC / 32; ++k) {
            uint32_t o[16];
            tmem_ld16_nowait(tO + half * (OC / 2) + 16 * k, o);
            tmem_wait_ld();
#pragma unroll
            for (int c = 0; c < 4; ++c)
              *piece(v, 4 * k + c) = make_uint4(o[4 * c], o[4 * c + 1], o[4 * c + 2], o[4 * c + 3]);
          }
          __syncwarp();
          for (int e = lane; e < 32 * RC; e += 32) {
            const int r = quarter * 32 + e / RC, c = e % RC;
            if (r < mq)
              *(uint4 *)(p.ws_o + (bs * WS_MAXQ + r) * DH + part * OC + half * (OC / 2) + c * 4) =
                  *piece(r, c);
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(TMEM_COLS)
                 : "memory");
  ts.finish();
}

template <int DH>
const char *run(const CUtensorMap &tm, const PairParams &p, int n_pairs, cudaStream_t s) {
  constexpr size_t smem = 1024 + (2 * QV + NSLOT * CH) * (size_t)DH * 2;
  static PerDevice<size_t> limit;
  if (const char *e = smem_opt_in(limit, k_attn_pair<DH>, smem)) return e;
  dim3 grid(p.n_splits, p.G, n_pairs);
  launch_pdl(k_attn_pair<DH>, grid, NT, smem, s, tm, p);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? nullptr : cudaGetErrorString(e);
}

}  // namespace

const char *launch_attention_pair(const void *q, const int32_t *pos, const int4 *blocks,
                                  int n_blocks, const int4 *pairs, int n_pairs, int n_splits,
                                  const Dims &dm, int layer, const int32_t *table,
                                  const CUtensorMap &tm_kv, float *ws_o, float2 *ws_ml, void *out,
                                  int *dev_flag, cudaStream_t s, const KVView *views,
                                  const CUtensorMap *tmaps) {
  if (n_pairs <= 0) return nullptr;
  if ((views == nullptr) != (tmaps == nullptr)) return "document views without tensor maps";
  PairParams p{};
  p.q = (const __nv_bfloat16 *)q;
  p.qk_scale = (float)(1.4426950408889634 / std::sqrt((double)dm.dh));
  p.pos = pos;
  p.blocks = blocks;
  p.pairs = pairs;
  p.table = table;
  p.views = views;
  p.tmaps = tmaps;
  p.H = dm.H;
  p.G = dm.G;
  p.grp = dm.H / dm.G;
  p.layer = layer;
  p.L = dm.L;
  p.n_splits = n_splits;
  p.n_blocks = n_blocks;
  p.ws_o = ws_o;
  p.ws_ml = ws_ml;
  p.out = (__nv_bfloat16 *)out;
  p.dev_flag = dev_flag;
  if (dm.dh == 128) return run<128>(tm_kv, p, n_pairs, s);
  if (dm.dh == 64) return run<64>(tm_kv, p, n_pairs, s);
  return "head_dim not supported";
}

KVR_TRACE_ATTACH(trace_attach_attn_pair)

}  // namespace kvr
