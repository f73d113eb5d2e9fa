// k_gemm_pair.cu -- bf16 tensor-core GEMM for many rows (sm_103a): two SMs on one
// tile (tcgen05.mma cta_group::2), operands staged by TMA into 128B-swizzled
// shared memory, accumulators in TMEM.
//
//   Y[M][N] (+)= X[M][K] . W[N][K]^T     (bf16 operands, fp32 accumulate)
//
// Swap-AB as in the few-row kernel: W is the MMA's A operand.  A cluster of two
// CTAs owns tiles of 256 features x BN token rows (BN <= 256): each CTA loads its
// own 128 feature rows and half of the token rows, the pair's MMA reads both
// halves, and each CTA's TMEM holds its 128 features x BN accumulators.
//
// What bounds it: one CTA alone needs 48 KB of operands per 64-wide K block for
// 128 x 256 outputs, and its tensor pipe ran at 72% at best; a pair needs 32 KB
// per CTA for twice the tile.  Measured (4096 rows): gate/up 28672 x 4096
// 595 -> 482 us (1.62 -> 1.99 PFLOP/s), down 4096 x 14336 285 us (1.69); 2608
// rows: all projections of a layer 870 -> 650 us (1.04 -> 1.75 PFLOP/s); 904
// rows: 384 -> 280 us.
//
// Work split, over the C clusters that fit at once: rounds of whole tiles, tile
// R + c + kC to cluster c in round k (neighbouring clusters share weight or
// token tiles and walk K in step, so each comes from DRAM once).  Of the R
// tiles left over each goes to s = floor(C / R) clusters, equal parts of K --
// again in step -- that the cluster of the last part sums in part order from what
// the others publish (the waits: pair_split.cuh).  The parts come first, so that
// their sum runs beside the MMAs of the whole tiles.  (Whole tiles alone: 2608 rows of a 4096-wide
// projection leave 24 of 76 clusters' slots of the last round in use.  Stream-K
// ranges over the left tiles, each cluster at K blocks of its own, re-read
// operands from DRAM: 66 us there, and 106 against a floor of 55 us for 904
// rows of a 14336-deep one.)
//
// Warp roles (320 threads): warp 0 TMA (one lane; both CTAs), warp 1 TMEM
// allocation and, in the leader (rank 0), MMA issue (one lane), warps 2-9
// epilogue.  Accumulators are double-buffered.  Every wait is bounded; a wait
// that runs out sets the device error flag, the CTA's roles stop, the peer's
// waits run out in turn, and both meet at the final cluster barrier.
#include <cstdlib>
#include <cuda.h>

#include "gemm_epilogue.cuh"
#include "kvr_internal.cuh"
#include "pair_split.cuh"
#include "tc_ptx.cuh"

namespace kvr {
namespace {
using namespace ptx;

constexpr int TM = 256;               // output features per cluster tile (UMMA M)
constexpr int BM = 128;               // of these per CTA
constexpr int BK = 64;                // K of one operand tile: a 128-byte swizzle atom of bf16
constexpr int KS = 2;                 // operand tiles (K blocks) per stage and barrier
constexpr int UK = 16;                // K per tcgen05.mma kind::f16
constexpr int A_BYTES = BM * BK * 2;  // 16 KB
constexpr int MAX_STAGES = 4;
constexpr int ACC_COLS = 256;         // TMEM columns of one accumulator buffer
constexpr int EPI_GROUPS = 2;         // epilogue warp groups, alternate column chunks
constexpr int EPI_WARPS = 4 * EPI_GROUPS;
constexpr int EPI_THREADS = 32 * EPI_WARPS;
constexpr int NT = 64 + EPI_THREADS;
constexpr int PRE_WAIT_STAGES = 2;    // weight stages requested before the wait on the predecessor
constexpr int MIN_UNITS = 4;          // units (of KS K blocks) a part of a tile has at least
constexpr int MAX_PARTS = 8;          // clusters a left-over tile is split over at most
constexpr int SUM_PARTS = 3;          // parts of a tile in flight while they are summed

struct PairGemm : PairSplit {  // its units: KS K blocks (the last may be short)
  int M, N, KB;       // K blocks
  int BN, n_tiles;
  int stages;
  float *Y;
  int ldy;
  const float *bias;
  int epi;
  void *out2;  // SwiGLU output (bf16 [M][N/2])
  int ld2;
  float *ws;      // [CTA][2][256][128] fp32 parts (the first slot of each CTA is used)
  int *ready;     // [2 * left] published parts per split tile and CTA rank (self-resetting)
  int *dev_flag;
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of the same shared-memory object in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(const void *p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(su32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar)
               : "memory");
}
// A TMA load into this CTA whose bytes count on a barrier of the pair's leader.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap *map, uint32_t bar,
                                                 int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx"
      "::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"((uint64_t)map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void mma_bf16_pair(uint32_t d_tmem, uint64_t a, uint64_t b,
                                              uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on the barrier at this offset in both CTAs once the MMAs issued so
// far are complete.
__device__ __forceinline__ void mma_commit_pair(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(su32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void epi_bar() {
  asm volatile("bar.sync 1, %0;" ::"n"(EPI_THREADS) : "memory");
}

__global__ void __launch_bounds__(NT, 1)
    k_gemm_pair(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                const PairGemm p) {
  extern __shared__ uint8_t smem_raw[];
  // full is counted in the leader alone; empty and accf are signalled in both
  // CTAs; acce in the leader by the epilogue warps of both
  __shared__ __align__(8) uint64_t full[MAX_STAGES], empty[MAX_STAGES], accf[2], acce[2], drain_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_f;

  TraceScope ts(TK_GEMM);
  pdl_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank(), cluster = (int)(blockIdx.x >> 1);
  const int S = p.stages;
  const uint32_t base = (su32(smem_raw) + 1023u) & ~1023u;
  const uint32_t b_bytes = (uint32_t)p.BN * 64u;  // BN / 2 rows of 128 bytes
  const uint32_t stage_bytes = KS * (A_BYTES + b_bytes);  // A tiles, then B tiles
  volatile int *abort_v = &abort_f;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], 2 * EPI_WARPS);
    }
    mbar_init(&drain_bar, 1);
    abort_f = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     su32(&tmem_slot)),
                 "r"(2 * ACC_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  cluster_sync();  // both CTAs' barriers are initialised, both hold their TMEM
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA
    if (lane == 0) {
      tma_prefetch_desc(&tmW);
      tma_prefetch_desc(&tmX);
      // the leader's barrier counts the bytes of both CTAs
      const uint32_t full0 = map_rank(&full[0], 0);
      auto blocks = [&](int ku) { return min(KS, p.KB - ku * KS); };
      auto load_w = [&](int s, const Segment &g, int ku) {
        for (int j = 0; j < blocks(ku); ++j)
          tma_load_2d_pair(base + (uint32_t)s * stage_bytes + j * A_BYTES, &tmW, full0 + 8u * s, 0,
                           ((2 * g.ntile + rank) * p.KB + ku * KS + j) * BM);
      };
      auto load_x = [&](int s, const Segment &g, int ku) {
        for (int j = 0; j < blocks(ku); ++j)
          tma_load_2d_pair(base + (uint32_t)s * stage_bytes + KS * A_BYTES + j * b_bytes, &tmX,
                           full0 + 8u * s, (ku * KS + j) * BK,
                           g.mtile * p.BN + rank * (p.BN / 2));
      };
      auto expect = [&](int s, int ku) {
        if (rank == 0) mbar_expect_tx(&full[s], 2 * blocks(ku) * (A_BYTES + b_bytes));
      };
      // The weights never depend on the previous kernel: the first stages'
      // tiles are requested before the wait on it, their activations after.
      const int pre = S < PRE_WAIT_STAGES ? S : PRE_WAIT_STAGES;
      int n_pre = 0;
      {
        Walk w(p, cluster);
        Segment g;
        while (n_pre < pre && w.next(p, g))
          for (int ku = g.ku0; ku < g.ku1 && n_pre < pre; ++ku, ++n_pre) {
            expect(n_pre, ku);
            load_w(n_pre, g, ku);
          }
      }
      pdl_wait();
      ts.waited();
      Walk w(p, cluster);
      Segment g;
      uint32_t it = 0;
      bool ok = true;
      while (ok && w.next(p, g))
        for (int ku = g.ku0; ku < g.ku1; ++ku, ++it) {
          const int s = (int)(it % (uint32_t)S);
          if (it >= (uint32_t)n_pre) {
            if (it >= (uint32_t)S &&
                !(ok = mbar_wait(&empty[s], (it / S - 1) & 1u, abort_v, p.dev_flag, 1)))
              break;
            expect(s, ku);
            load_w(s, g, ku);
          }
          load_x(s, g, ku);
        }
      // copies in flight complete before the CTA may exit: the leader's
      // barriers count both CTAs' (the peer waits at the cluster barrier)
      if (rank == 0)
        for (uint32_t j = it > (uint32_t)S ? it - S : 0; j < it; ++j)
          mbar_wait(&full[j % S], (j / S) & 1u, abort_v, p.dev_flag, 0, false);
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA
    // The whole warp walks the loop and one elected lane issues, so that the
    // operands stay in uniform registers, and a stage holds KS K blocks: with
    // one block a stage, the wait, four MMAs and commit of a block took longer
    // to issue than the MMAs to run (512 cycles), the tensor pipe 65% active.
    if (rank == 0) {
      const uint32_t idesc = idesc_bf16(TM, p.BN);
      Walk w(p, cluster);
      Segment g;
      uint32_t seg = 0;
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      auto wait = [&](uint64_t *bar, uint32_t parity, int code) -> bool {
        return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_v, p.dev_flag, code));
      };
      while (ok && w.next(p, g)) {
        const uint32_t buf = seg & 1u, d = tmem + buf * ACC_COLS;
        // both CTAs' epilogues have taken what the buffer held
        if (!wait(&acce[buf], ((seg >> 1) & 1u) ^ 1u, 2)) break;
        for (int ku = g.ku0; ku < g.ku1; ++ku) {
          if (!(ok = wait(&full[s], ph, 4))) break;
          tc_fence_after();
          if (elect_one()) {
            const uint32_t sa = base + (uint32_t)s * stage_bytes, sb = sa + KS * A_BYTES;
            const int nb = min(KS, p.KB - ku * KS);
#pragma unroll
            for (int j = 0; j < KS; ++j) {
              if (j >= nb) break;
              const uint64_t da = sw128_desc(sa + j * A_BYTES), db = sw128_desc(sb + j * b_bytes);
#pragma unroll
              for (int k = 0; k < BK / UK; ++k)
                mma_bf16_pair(d, da + (uint64_t)(k * UK * 2 / 16), db + (uint64_t)(k * UK * 2 / 16),
                              idesc, (ku > g.ku0 || j > 0 || k > 0) ? 1u : 0u);
            }
            mma_commit_pair(&empty[s]);
            if (ku + 1 == g.ku1) mma_commit_pair(&accf[buf]);
          }
          __syncwarp();
          if (++s == S) {
            s = 0;
            ph ^= 1u;
          }
        }
        ++seg;
      }
      if (elect_one()) mma_commit_pair(&drain_bar);
      __syncwarp();
    }
    // every MMA of the pair completes before either CTA frees its TMEM
    if (lane == 0) mbar_wait(&drain_bar, 0, abort_v, p.dev_flag, 0, false);
  } else {
    // ------------------------------------------------------------ epilogue
    pdl_wait();  // outputs, parts and counters may still be in use upstream
    const int q = warp & 3;  // TMEM lane quarter of this warp
    const int f = q * 32 + lane;
    const int et = threadIdx.x - 64;
    const int eg = (warp - 2) >> 2;  // column chunks eg, eg + EPI_GROUPS, ...
    constexpr int CC = 32;           // columns (token rows) per chunk
    const uint32_t acce0 = map_rank(&acce[0], 0);
    Walk w(p, cluster);
    Segment g;
    bool dead = false;  // warp-uniform: a wait ran out; the barriers are still met
    for (uint32_t seg = 0; w.next(p, g); ++seg) {
      const uint32_t buf = seg & 1u;
      const int t0 = g.mtile * p.BN, mv = min(p.BN, p.M - t0);
      const int n = g.ntile * TM + rank * BM + f;
      // a part of a tile: the last part's cluster sums the others' parts and its own
      const int parts = g.ku1 - g.ku0 < p.KU ? p.parts : 1;
      const bool owner = parts == 1 || sums_parts(p, cluster);
      int *ready = p.ready + 2 * g.tile + rank;
      if (owner && parts > 1) {
        // Every other cluster's part is its first segment, waits on nothing and
        // is published at its end.
        if (et == 0) {
          volatile int *r = ready;
          const uint64_t t0w = gtime_ns();
          for (uint32_t k = 0; *r < parts - 1; ++k)
            if ((k & 63) == 63 && (*abort_v || gtime_ns() - t0w > WAIT_NS)) {
              if (!*abort_v) {
                *abort_v = 1;
                atomicOr(p.dev_flag, 32);
              }
              break;
            }
        }
        epi_bar();
        asm volatile("fence.acq_rel.gpu;" ::: "memory");  // acquire the parts
      }
      if (!dead)
        dead = !__all_sync(0xffffffffu,
                           mbar_wait(&accf[buf], (seg >> 1) & 1u, abort_v, p.dev_flag, 8));
      tc_fence_after();
      const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + buf * ACC_COLS;
      for (int c = CC * eg; c < mv && !dead; c += CC * EPI_GROUPS) {
        if (owner && parts > 1) {
          // The others' parts in part order, then this cluster's own.  Sixteen rows of
          // SUM_PARTS parts are in flight at once: with 32 rows of one part, seven parts
          // took longer than the next tile's MMAs, and the tile after that waited for
          // this buffer (4096 rows of 6144 x 4096, four tiles in eight parts: 133 -> 126
          // us).  Four parts, 121 us, take 161 registers, and the next kernel no longer
          // fits beside this one: passes were no faster.
          for (int c2 = c; c2 < min(c + CC, mv); c2 += 16) {
            float v[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = -0.f;  // exact: -0 + x = x
            for (int k0 = 0; k0 < parts - 1; k0 += SUM_PARTS) {
              float x[SUM_PARTS][16];
#pragma unroll
              for (int u = 0; u < SUM_PARTS; ++u) {
                const size_t slot = 2 * part_cluster(p, g.tile, k0 + u) + rank;
                const float *src = p.ws + (slot * 2 * 256 + c2) * BM + f;
#pragma unroll
                for (int j = 0; j < 16; ++j)
                  x[u][j] = k0 + u < parts - 1 && c2 + j < mv ? __ldcg(src + (size_t)j * BM) : -0.f;
              }
#pragma unroll
              for (int u = 0; u < SUM_PARTS; ++u)
#pragma unroll
                for (int j = 0; j < 16; ++j) v[j] += x[u][j];
            }
            uint32_t r[16];
            tmem_ld16_nowait(taddr + c2, r);
            tmem_wait_ld();
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] += __uint_as_float(r[j]);
            if (n < p.N) epilogue16(p, t0 + c2, n, v, mv - c2);
          }
          continue;
        }
        uint32_t r[CC];
        tmem_ld32_nowait(taddr + c, r);
        tmem_wait_ld();
        if (!owner) {
          float *dst = p.ws + ((size_t)blockIdx.x * 2 * 256 + c) * BM + f;
#pragma unroll
          for (int j = 0; j < CC; ++j)
            if (c + j < mv) dst[(size_t)j * BM] = __uint_as_float(r[j]);
          continue;
        }
        float v[CC];
#pragma unroll
        for (int j = 0; j < CC; ++j) v[j] = __uint_as_float(r[j]);
        if (n < p.N) {
          epilogue16(p, t0 + c, n, v, mv - c);
          if (c + 16 < mv) epilogue16(p, t0 + c + 16, n, v + 16, mv - c - 16);
        }
      }
      if (!owner) {
        asm volatile("fence.acq_rel.gpu;" ::: "memory");  // release the part
        epi_bar();
        if (et == 0 && !*abort_v) atomicAdd(ready, 1);
      } else if (parts > 1 && et == 0) {
        *ready = 0;
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acce0 + 8u * buf);
    }
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync();  // no CTA leaves while its peer's MMAs, copies or arrivals need it
  tc_fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(2 * ACC_COLS)
                 : "memory");
  ts.finish();
}

// The launch's shape: token tile, split of the tiles, pipeline depth.
size_t configure(PairGemm &p, int M, int N, int K, int clusters, int smem_limit) {
  p.M = M;
  p.N = N;
  p.KB = K / BK;
  p.KU = (p.KB + KS - 1) / KS;
  p.n_tiles = (N + TM - 1) / TM;
  // The token tile whose rounds cost least: per K block the longer of its MMAs
  // (2 BN cycles) and its operands' way from L2 (256 + BN at 64 bytes a cycle).
  p.clusters = clusters;
  double best = -1;
  for (int bn = 256; bn >= 128; bn -= 16) {
    const long long mt = (M + bn - 1) / bn, tiles = mt * p.n_tiles;
    const int left = (int)(tiles % clusters);
    int parts = left ? clusters / left : 1;
    if (parts > MAX_PARTS) parts = MAX_PARTS;
    if (parts > p.KU / MIN_UNITS) parts = p.KU / MIN_UNITS > 1 ? p.KU / MIN_UNITS : 1;
    const double rounds = (double)(tiles / clusters) + (left ? 1.0 / parts : 0.0);
    const double c = rounds * (2 * bn > 256 + bn ? 2 * bn : 256 + bn);
    if (best < 0 || c < best) {
      best = c;
      p.BN = bn;
      p.m_tiles = (int)mt;
      p.left = left;
      p.parts = parts;
      p.rounds = (int)(tiles / clusters);
    }
  }
  if (!p.rounds) p.clusters = p.left * p.parts;  // no more than have work
  const int stage = KS * (A_BYTES + p.BN * 64);
  p.stages = (smem_limit - 1024) / stage;
  if (p.stages > MAX_STAGES) p.stages = MAX_STAGES;
  return 1024 + (size_t)p.stages * stage;
}

}  // namespace

// Where the pairs win (both kernels measured inside a pass, us a launch).  Above 256
// rows the few-row kernel's CTAs walk several token tiles (gate/up of 300 rows 107
// -> 67), and the sums it leaves cost the next kernel more (with its RoPE,
// 6144 x 4096: 300 rows 81 -> 73, 600 rows 116 -> 87); against that stand the pairs'
// launch and tail, about 8 us, so small products stay: 4096 x 4096 with its
// RMSNorm, 300 rows 46 against 52, 600 rows 57 against 59.
// With one token tile the few-row kernel splits K over all SMs and leaves the sums
// to the next kernel; only gate/up, which sums its own tiles, gains by pairs, where
// their rounds are full and no tile is in more than two parts (193 to 256 rows, a
// layer's GEMMs, RoPE and norms before over after: 4096 x 28672, 112 tiles for 76
// clusters, 1.00 to 1.03; 3584 x 37888, 148 tiles, 1.00 to 1.04; 8192 x 57344 1.01
// to 1.04; but 4096 x 22016, 10 of its 86 tiles in seven parts, 0.97 to 0.99, 4096 x
// 32768, 128 tiles, 0.98 to 1.02) and the product is large (2304 x 18432, 72 tiles,
// 0.97, 2560 x 19456, 76 tiles, 0.95).  192 rows and below: equal at best.
bool gemm_pair_takes(int M, int N, int K, int epi, int num_sms) {
  static const bool off = [] {
    const char *e = getenv("KVR_DISABLE_PAIR_GEMM");
    return e && e[0] == '1';
  }();
  if (off || 2.0 * M * N * K < 12e9) return false;
  if (M > 256) return true;
  if (M <= 192 || epi != GEMM_EPI_SWIGLU || 2.0 * M * N * K < 40e9) return false;
  const int clusters = num_sms / 2, tiles = (N + TM - 1) / TM, left = tiles % clusters;
  const int parts = left ? clusters / left : 1;
  const double rounds = tiles / clusters + (left ? 1.0 / parts : 0.0);
  return parts <= 2 && tiles >= 0.9 * rounds * clusters;
}

const char *launch_gemm_pair(const GemmArgs &g, const CUtensorMap &tmW, int epi, void *out2,
                             int ld2, const TcWorkspace &ws, cudaStream_t s) {
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.blockDim = dim3(NT);
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  // per device: the shared memory a CTA may use, and the pairs that fit at once
  struct Fit {
    int smem = 0, clusters = 0;
  };
  static PerDevice<size_t> limit;
  static PerDevice<Fit> fits;
  int dev = 0;
  cudaGetDevice(&dev);
  const Fit fit = fits.with(dev, [&](Fit &f) {
    if (f.clusters > 0) return f;
    Fit x;
    x.smem = smem_opt_in_all(limit, k_gemm_pair);
    cfg.gridDim = dim3(ws.num_sms / 2 * 2);
    cfg.dynamicSmemBytes = x.smem;
    if (x.smem < 0 ||
        cudaOccupancyMaxActiveClusters(&x.clusters, (void *)k_gemm_pair, &cfg) != cudaSuccess)
      x.clusters = 0;
    if (x.clusters > 0) f = x;
    return x;
  });
  if (fit.smem < 0) return "cannot raise the dynamic shared memory limit";
  if (fit.clusters < 1) return "no cluster of two CTAs fits";
  PairGemm p{};
  const int clusters = fit.clusters < ws.num_sms / 2 ? fit.clusters : ws.num_sms / 2;
  cfg.dynamicSmemBytes = configure(p, g.M, g.N, g.K, clusters, fit.smem);
  cfg.gridDim = dim3(2 * p.clusters);
  p.Y = g.Y;
  p.ldy = g.ldy;
  p.bias = g.bias;
  p.epi = epi;
  p.out2 = out2;
  p.ld2 = ld2;
  p.ws = ws.partials;
  p.ready = ws.counters;
  p.dev_flag = ws.dev_flag;
  CUtensorMap tmX;
  if (!make_tmap_bf16(&tmX, g.X, g.M, g.K, p.BN / 2)) return "activation TMA descriptor rejected";
  if (g_pdl) {
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = 2;
  }
  cudaLaunchKernelEx(&cfg, k_gemm_pair, tmW, tmX, p);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? nullptr : cudaGetErrorString(e);
}

KVR_TRACE_ATTACH(trace_attach_gemm_pair)

}  // namespace kvr
