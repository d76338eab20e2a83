// FP8 e4m3 GEMM with FP32 scales per 128 x 128 block, FP32 accumulation and
// output, and the block quantiser that produces its operands.  (The paper
// measures BF16 only; this is the precision variant of the same NN GEMM.)
//
//   A ~ qA (M x K e4m3, row-major) with sA[M/128][K/128],
//   B ~ qB (K x N e4m3, row-major) with sB[K/128][N/128],
//   C[i][j] = sum_kb sA[i/128][kb] * sB[kb][j/128] * sum_{k in kb} qA[i][k] qB[k][j].
//
// Kernel (one CTA per SM, persistent over (128 x BN output tile, K split)
// units; BN = 256 or 128; split S = 1, 2, 4 or 8):
//   warp 0     TMA producer: A block 128 x 128 bytes (K-major) and B block 128 K-rows
//              x BN bytes (N-major, 128-byte-wide column boxes), 128-byte swizzle.
//   warp 1     one lane issues tcgen05.mma kind::f8f6f4 (M = 128, K = 32) into a fresh TMEM
//              accumulator per 128-deep K block (128 x 256: one per 128-column half), and commits
//              each to its buffer's full barrier.  Warps 0 and 1 step converged with predicated
//              loads, MMAs and commits, as in the BF16 kernels, and for the same reason: with one
//              lane in the loop by itself a K block took its thread 750 cycles (128 x 128) to 1000
//              (128 x 256) for 256 and 512 cycles of MMAs.
//   warps 2-3  idle: they complete warpgroup 0, whose registers go to the promotion warps.
//   warps 4-11 promotion and epilogue (224 registers each), two warps per TMEM lane
//              quarter, each owning one half of the tile's columns: per K block, tcgen05.ld
//              the block product in 32-column chunks, the next on its way while one is added,
//              multiply by sA * sB (one scalar per warp and K block) and add into FP32 registers;
//              the buffer is released once its last chunk has arrived.  After the unit's last
//              block, 128B-swizzled staging and a TMA store (beta = 0) or reduce-add (beta = 1).
//              With S > 1 the unit's partial goes to the split-K workspace instead, and the
//              last arriving split of a (tile, warp) sums the S partials in the fixed order
//              0..S-1.  Their release of a buffer (and of the K block's operand stage) is what
//              lets the producer and the MMA warp reuse it.
// What bounds it: at 512 x 1536 x 2048 (48 CTAs of 128 x 128) about 360 cycles per K block against
// 256 of MMAs, the buffer's round trip through the promotion; on 128 x 256 about 700 against 512,
// where the MMAs alone take 620 and the promotion alone 580.  Before and after these three changes
// (converged issue, chunked promotion, halves), sweep protocol: 512 x 1536 x 2048 on 128 x 128 9.2 ->
// 7.1 us; 3072 x 2048 x 4096 38.3 -> 27.1 (128 x 128), 37.6 -> 30.4 (128 x 256); 4096^3 73.8 -> 60.8
// (128 x 256), 73.2 -> 62.2 (the pair); 8192^2 x 4096 251 -> 209 and 247 -> 210.  The half-width units of
// a partial wave (half_tiles) then take 128 x 256 to 57.5 at 4096^3.
// The 256 x 256 tile also runs as a tcgen05 cta_group::2 pair (gemm_fp8_2sm_kernel):
// each CTA of a 2-CTA cluster loads its 128 rows of A and 128 columns of B, the even
// CTA issues the M = 256 MMAs, and each CTA promotes and stores its own 128 rows.
// Padding is never materialised: tensor maps carry the logical extents, reads
// past them are zero-filled, stores clipped, and scales outside the logical
// blocks read as 0.  Every mbarrier wait is bounded; on expiry the kernel
// records an error code, lets its in-flight copies land, releases TMEM and returns.
#include <cuda.h>
#include <cuda_fp8.h>
#include <cuda_runtime.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <climits>
#include <mutex>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "ptx.cuh"
#include "rg_internal.h"

namespace rg {

namespace fp8 {

constexpr int kEpiWarps = 8;                  // two promotion warps per TMEM lane quarter
constexpr int kEpiWarp0 = 4;                  // the promotion warps are warpgroups 1 and 2
constexpr int kThreads = 32 * (kEpiWarp0 + kEpiWarps);
// Register split.  Three warps per SM sub-partition launch with 168 registers each;
// warpgroup 0 (producer, MMA issuer and two idle warps) then shrinks to 56 and the
// promotion warpgroups grow to 224 (setmaxnreg), which holds a thread's BN / 2
// accumulators plus 64 columns of a K block's product.  The shares add up to the
// launch's registers, per CTA and per sub-partition (one warp of each warpgroup).
constexpr int kLaunchRegs = 168, kRegsLow = 56, kRegsHigh = 224;
static_assert(4 * kRegsLow + kEpiWarps * kRegsHigh == (kThreads / 32) * kLaunchRegs, "register split");
static_assert(kRegsLow + 2 * kRegsHigh == 3 * kLaunchRegs, "register split per sub-partition");
constexpr int BM = 128, BK = 128;             // BK: one 128-byte swizzle row of e4m3 = one scale block
constexpr int SB = 128;                       // scale block edge
constexpr long long kDrainCycles = 1LL << 30;
constexpr uint32_t FULL = 0xffffffffu;

// PAIR: a cta_group::2 pair computes a 256 x BN tile; each CTA loads its 128 rows of A
// and BN / 2 columns of B and holds its 128 output rows x BN columns in its own TMEM.
template <int BN, bool PAIR = false>
struct Cfg {
  static constexpr int CTAS = PAIR ? 2 : 1;
  // Column halves of a K block, an MMA and a TMEM accumulator buffer each: the 1-CTA 128x256
  // tile alone has two, so that a buffer comes back after half a K block's promotion.  It then
  // takes four operand stages (TMA latency, not the MMAs, bound it with three: 4096^3 63.2 us
  // against 60.8) for one staging buffer per promotion warp instead of two.  In the pair the
  // halves' MMAs (64 of each CTA's 128 columns) were slower: 62.2 against 66.5 us.
  static constexpr int HALVES = BN == 256 && !PAIR ? 2 : 1;
  static constexpr int STAGES = PAIR ? 5 : 4;
  static constexpr int NSTG = HALVES == 2 ? 1 : 2;  // staging buffers per promotion warp
  static constexpr int A_BYTES = BM * BK;
  static constexpr int B_BYTES = BK * BN / CTAS;  // (BN / CTAS) / 128 N-major column boxes of BK rows
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int NB = BN / HALVES;      // columns of an MMA and of a TMEM accumulator buffer
  static constexpr int DEPTH = 512 / BN;      // K blocks in flight in TMEM (all 512 columns)
  static constexpr int NACC = DEPTH * HALVES; // accumulator buffers
  static constexpr int STAGING_OFF = STAGES * STAGE_BYTES;
  static constexpr int BAR_OFF = STAGING_OFF + kEpiWarps * NSTG * 4096;
  static constexpr int SMEM_BYTES = 1024 + BAR_OFF + 256;
  static constexpr int HALF = BN / 2;         // columns per promotion warp
  // E4M3 x E4M3, A K-major, B MN-major; M = 256 across a pair
  static constexpr uint32_t IDESC = instr_desc(0, 0, 0, 1, 128 * CTAS, NB);
  static_assert(SMEM_BYTES <= 232448, "shared memory budget");
  static_assert(BN == 128 || BN == 256, "tile width");
  static_assert(!PAIR || BN == 256, "pair tile");
  static_assert((2 * STAGES + 2 * NACC + 1) * 8 + 8 <= 256, "barrier block");
  static_assert(STAGES * STAGE_BYTES % 1024 == 0, "staging alignment");
};

template <uint32_t N>
__device__ __forceinline__ void setmaxnreg_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}
template <uint32_t N>
__device__ __forceinline__ void setmaxnreg_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}

// Arrive on an mbarrier given by its shared::cluster address with relaxed semantics: the pair's
// "accumulator buffer read" signal publishes no memory (the TMEM reads it covers have completed,
// tcgen05.wait::ld), so it needs none of the membar a release at cluster scope costs on every K block.
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// a0 = sc * p0 + a0, a1 = sc * p1 + a1, each rounded once: two FMAs, or one two-wide FMA (the same
// results), which saves issue slots and pays where a warp holds 128 accumulators (pair, 4096^3: 64.2
// against 62.2 us) and not where it holds 64 (128x128 at 8192^2 x 4096: 262 against 267 us).
template <bool WIDE>
__device__ __forceinline__ void add_scaled(float& a0, float& a1, uint32_t p0, uint32_t p1, float sc) {
  if constexpr (WIDE) {
    asm("{\n\t.reg .b64 x, y, z;\n\t"
        "mov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %4};\n\tmov.b64 z, {%0, %1};\n\t"
        "fma.rn.f32x2 z, x, y, z;\n\tmov.b64 {%0, %1}, z;\n\t}"
        : "+f"(a0), "+f"(a1)
        : "r"(p0), "r"(p1), "f"(sc));
  } else {
    a0 = fmaf(sc, __uint_as_float(p0), a0);
    a1 = fmaf(sc, __uint_as_float(p1), a1);
  }
}

struct Args {
  int32_t M, N;            // logical output extents
  int32_t tiles_m, tiles_n;  // tiles of the (padded) launch
  int32_t kblocks;         // K blocks of the (padded) launch
  int32_t splits;
  int32_t whole;           // tiles run whole, the rest as two half-width units each (see half_tiles)
  int32_t beta;
  int32_t mb_valid, kb_valid, nb_valid;  // logical scale blocks (reads beyond them are 0)
  int32_t sa_ld, sb_ld;    // leading dimensions of the scale arrays (blocks)
  const float* sA;
  const float* sB;
  float* ws;               // split-K partials [split][tile][BM] x BN
  int32_t* tickets;        // [tile][8], zero between launches
  int32_t* err;
  long long timeout;
};

__device__ __forceinline__ void st_shared_v4(uint32_t addr, float a, float b, float c, float d) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// One warp writes a 32 x 32 FP32 block (lane = row) through swizzled staging
// with a TMA store, or a TMA reduce-add when add is set.
template <int NSTG>
__device__ __forceinline__ void put_block(const CUtensorMap* map, const float* v, int row0, int col0, bool add,
                                          uint32_t stg0, int& sbuf, int lane) {
  if (lane == 0) bulk_wait_read<NSTG - 1>();
  __syncwarp();
  const uint32_t buf = stg0 + sbuf * 4096;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    st_shared_v4(buf + lane * 128 + ((j ^ (lane & 7)) << 4), v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
  fence_proxy_async_smem();
  __syncwarp();
  if (lane == 0) {
    if (add)
      tma_reduce_add_2d(map, buf, col0, row0);
    else
      tma_store_2d(map, buf, col0, row0);
    bulk_commit();
  }
  if constexpr (NSTG > 1) sbuf ^= 1;
}

// The kernel body.  SPLIT = false: the instance for S = 1 (no workspace path, so its
// promotion loop, which holds BN / 2 accumulators per thread, carries no split-K
// state).  PAIR: one CTA of a cta_group::2 pair (launched as 2-CTA clusters): units
// are (256-row pair tile, split); both CTAs load their operand halves, the even
// CTA's lane issues the pair MMAs, and each CTA promotes and stores its own 128
// rows; tiles, tickets and workspace rows count 128-row tiles (tiles_m is even).
template <int BN, bool SPLIT, bool PAIR>
__device__ __forceinline__ void fp8_body(const CUtensorMap& tmA, const CUtensorMap& tmB, const CUtensorMap& tmC,
                                         const CUtensorMap& tmW, const Args& args) {
  using C = Cfg<BN, PAIR>;
  // Coupled ring (as many stages as K blocks in TMEM, one CTA: the 128x128 tile): K block kb
  // uses stage and buffer kb % STAGES.  The producer refills a stage only once the promotion
  // warps have released its buffer, which they do after the block's MMAs completed, so a landed
  // stage also means a free buffer and the MMA warp waits on one barrier per K block.
  constexpr bool COUPLED = C::DEPTH == C::STAGES && !PAIR;
  // Otherwise the first promotion warp of the last half frees the K block's stage once it has
  // seen that half's products (every MMA that reads the stage has then completed).
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_s = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + ((1024u - (raw_s & 1023u)) & 1023u);
  const uint32_t sbase = smem_u32(smem);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + C::BAR_OFF);
  const uint32_t bar0 = smem_u32(bars);
  auto full_bar = [&](int i) { return bar0 + 8u * i; };
  auto empty_bar = [&](int i) { return bar0 + 8u * (C::STAGES + i); };
  auto tfull_bar = [&](int b) { return bar0 + 8u * (2 * C::STAGES + b); };
  auto tempty_bar = [&](int b) { return bar0 + 8u * (2 * C::STAGES + C::NACC + b); };
  const uint32_t drain_bar = bar0 + 8u * (2 * C::STAGES + 2 * C::NACC);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * C::STAGES + 2 * C::NACC + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int never = 0;
  volatile int* no_abort = &never;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int ntiles = args.tiles_m * args.tiles_n;  // 128-row tiles
  const int S = SPLIT ? args.splits : 1;
  const int rank = PAIR ? static_cast<int>(cluster_ctarank()) : 0;
  const int cid = PAIR ? static_cast<int>(blockIdx.x) / 2 : static_cast<int>(blockIdx.x);
  const int ncl = PAIR ? static_cast<int>(gridDim.x) / 2 : static_cast<int>(gridDim.x);
  // Units: whole ones first, then (128 x 256 tile, S = 1) halves of the tiles from args.whole on, each
  // one 128-column half of its tile's columns, promoted by the first four promotion warps; a CTA has at
  // most one of them, its last.  Its loops are their own code, behind those of the whole units.
  constexpr bool TAIL = C::HALVES == 2 && !SPLIT;
  const int total = TAIL ? args.whole : (PAIR ? ntiles / 2 : ntiles) * S;
  // the CTA's half unit (2 x its tile's place among the halved ones + the half), or -1
  int half_unit = -1;
  if constexpr (TAIL) {
    const int h = (cid - total % ncl + ncl) % ncl;
    if (h < 2 * (ntiles - args.whole)) half_unit = h;
  }
  // unit u = ((pair) tile u / S, split u % S) runs K blocks [s * kblocks / S, (s + 1) * kblocks / S)
  auto kb_lo = [&](int s) { return S == 1 ? 0 : s * args.kblocks / S; };
  // this CTA's 128-row tile of unit u: tile index (tickets, workspace) and coordinates
  auto tile_of = [&](int u, int& tm, int& tn) {
    const int t = u / S;
    if constexpr (PAIR) {
      tm = 2 * (t / args.tiles_n) + rank;
      tn = t % args.tiles_n;
    } else {
      tm = t / args.tiles_n;
      tn = t % args.tiles_n;
    }
    return tm * args.tiles_n + tn;
  };

  if (threadIdx.x == 0) {
    prefetch_tmap(&tmA);
    prefetch_tmap(&tmB);
    prefetch_tmap(&tmC);
    for (int i = 0; i < C::STAGES; ++i) {
      mbar_init(full_bar(i), 1);
      mbar_init(empty_bar(i), 1);
    }
    for (int b = 0; b < C::NACC; ++b) {
      mbar_init(tfull_bar(b), 1);
      // released by the warps that promote it (pair: both CTAs', on the even CTA)
      mbar_init(tempty_bar(b), C::CTAS * kEpiWarps / C::HALVES);
    }
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    if constexpr (PAIR) {  // collective with the partner's warp 1: the same columns in both CTAs
      tmem_alloc_pair(smem_u32(tmem_slot), 512);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(tmem_slot), 512);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  __syncthreads();
  if constexpr (PAIR) cluster_sync();  // the partner's barriers are initialised
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dependency_wait();
  grid_launch_dependents();
  // Role branches; each warpgroup first resizes its registers (setmaxnreg acts on whole
  // warpgroups, so warps 0-3 take the same instruction before they part).
  if (warp < kEpiWarp0) {
    setmaxnreg_dec<kRegsLow>();
    if (warp == 0) {
      int stage = 0, fills = 0;
      uint32_t ph = 0, issued_mask = 0, issued_ph = 0;
      bool ok = true;
      const uint32_t lead = elect_one() ? 1u : 0u;
      // loads K blocks [kb0, kb1) of tile (tm, tn): all of its columns, or (a half) one box from column bx
      auto load = [&](int tm, int bx, int kb0, int kb1, auto boxes) {
        constexpr int kBoxes = decltype(boxes)::value;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (fills >= C::STAGES &&
              !mbar_wait_warp(COUPLED ? tempty_bar(stage) : empty_bar(stage), ph ^ 1u, args.timeout, abort_flag))
            return false;
          ++fills;
          const uint32_t sa = sbase + static_cast<uint32_t>(stage) * C::STAGE_BYTES;
          // pair: both CTAs' loads complete on the even CTA's full barrier, which expects both halves
          const uint32_t fb = PAIR ? mapa_shared(full_bar(stage), 0) : full_bar(stage);
          mbar_arrive_expect_tx_lead(full_bar(stage), C::CTAS * (C::A_BYTES + kBoxes * BK * 128),
                                     PAIR && rank != 0 ? 0u : lead);
          tma_load_2d_lead<C::CTAS>(sa, &tmA, fb, kb * BK, tm * BM, lead);
#pragma unroll
          for (int j = 0; j < kBoxes; ++j)
            tma_load_2d_lead<C::CTAS>(sa + C::A_BYTES + j * (BK * 128), &tmB, fb, bx + j * 128, kb * BK, lead);
          issued_mask |= 1u << stage;
          issued_ph = (issued_ph & ~(1u << stage)) | (ph << stage);
          if (++stage == C::STAGES) {
            stage = 0;
            ph ^= 1u;
          }
        }
        return true;
      };
      for (int u = cid; ok && u < total; u += ncl) {
        const int s = u % S;
        int tm, tn;
        tile_of(u, tm, tn);
        ok = load(tm, tn * BN + (PAIR ? rank * (BN / 2) : 0), kb_lo(s), s + 1 == S ? args.kblocks : kb_lo(s + 1),
                  std::integral_constant<int, BN / C::CTAS / 128>{});
      }
      if constexpr (TAIL) {
        if (ok && half_unit >= 0) {
          int tm, tn;
          tile_of(args.whole + half_unit / 2, tm, tn);
          ok = load(tm, tn * BN + half_unit % 2 * 128, 0, args.kblocks, std::integral_constant<int, 1>{});
        }
      }
      if (lane == 0) {
        if (!ok) {
          atomicExch(args.err, 1);
          *abort_flag = 1;
        }
        // no TMA write may still be landing when the CTA exits
        if (!PAIR || rank == 0) {
          for (int i = 0; i < C::STAGES; ++i)
            if (issued_mask & (1u << i)) mbar_wait(full_bar(i), (issued_ph >> i) & 1u, kDrainCycles, no_abort);
        } else if (!ok) {
          // the odd CTA's loads complete on its partner's barriers; after an abort it gives
          // them a bounded time to land (normally every one of them was consumed)
          const long long t0 = clock64();
          while (clock64() - t0 < (kDrainCycles >> 6)) {
          }
        }
      }
      __syncwarp();
    } else if (warp == 1) {
      // A pair's odd CTA issues nothing: the even CTA's MMAs read and write both.
      if (!PAIR || rank == 0) {
        int stage = 0, acc = 0;
        uint32_t ph = 0, aph = 0;
        bool ok = true;
        const uint32_t lead = elect_one() ? 1u : 0u;
        // descriptors of stage 0: the stages and K steps differ in the start address field of the low words
        const uint64_t adesc0 = smem_desc_sw128(sbase, 16, 1024);
        const uint64_t bdesc0 = smem_desc_sw128(sbase + C::A_BYTES, BK * 128, 1024);  // column boxes BK*128 apart
        const uint32_t alo0 = static_cast<uint32_t>(adesc0), blo0 = static_cast<uint32_t>(bdesc0);
        const uint32_t desc_hi = static_cast<uint32_t>(adesc0 >> 32);  // that of both: same stride and swizzle
        // the MMAs of n K blocks, the first `halves` column halves of each
        auto multiply = [&](int n, auto halves) {
          for (int i = 0; i < n; ++i) {
            if (!mbar_wait_warp(full_bar(stage), ph, args.timeout, abort_flag)) return false;
            const uint32_t so = static_cast<uint32_t>(stage) * (C::STAGE_BYTES >> 4);
#pragma unroll
            for (int h = 0; h < decltype(halves)::value; ++h) {
              const int buf = acc * C::HALVES + h;
              if constexpr (!COUPLED) {
                if (!mbar_wait_warp(tempty_bar(buf), aph ^ 1u, args.timeout, abort_flag)) return false;
              }
              tc_fence_after();
              constexpr uint32_t hb = (BK * 128) >> 4;  // half h of the B columns is the h-th column box
#pragma unroll
              for (int k = 0; k < BK / 32; ++k)
                mma_f8_lead<C::CTAS>(tmem_base + static_cast<uint32_t>(buf * C::NB), alo0 + so + ((k * 32) >> 4), desc_hi,
                                     blo0 + so + h * hb + ((k * (32 * 128)) >> 4), desc_hi, C::IDESC, k > 0 ? 1u : 0u,
                                     lead);
              mma_commit_lead<C::CTAS>(tfull_bar(buf), lead);  // pair: both CTAs' rows of the product are ready
            }
            if (++stage == C::STAGES) {
              stage = 0;
              ph ^= 1u;
            }
            if (++acc == C::DEPTH) {
              acc = 0;
              aph ^= 1u;
            }
          }
          return true;
        };
        for (int u = cid; ok && u < total; u += ncl) {
          const int s = u % S;
          ok = multiply((s + 1 == S ? args.kblocks : kb_lo(s + 1)) - kb_lo(s), std::integral_constant<int, C::HALVES>{});
        }
        if constexpr (TAIL) {
          if (ok && half_unit >= 0) ok = multiply(args.kblocks, std::integral_constant<int, 1>{});
        }
        if (!ok) {
          if (elect_one()) {
            atomicExch(args.err, 2);
            *abort_flag = 1;
            if constexpr (PAIR)
              mma_commit_pair(drain_bar);
            else
              mma_commit(drain_bar);  // completes once every issued MMA has finished
          }
          __syncwarp();
          mbar_wait_warp(drain_bar, 0, kDrainCycles, no_abort);
        }
      }
      __syncwarp();
    }
  } else {
    setmaxnreg_inc<kRegsHigh>();
    // promotion warps 4..11: lane quarter q (the TMEM lanes this warp may read), column half hc
    const int e = warp - kEpiWarp0;
    const int q = warp & 3;
    const int hc = e / 4;
    const uint32_t stg0 = sbase + C::STAGING_OFF + e * (C::NSTG * 4096);
    int acc = 0, sbuf = 0, pstage = 0;  // pstage: the operand stage of the current K block
    uint32_t aph = 0;
    bool ok = true;
    // promotes K blocks [kb0, kb1) of the tile's row block tm and the warp's columns from `col` on into r;
    // half: of a half unit, whose one buffer per K block the first four warps read
    auto promote = [&](int tm, int col, int kb0, int kb1, float (&r)[C::HALF], auto half) {
      const int nb = col / SB;  // the scale block column
      // scale rows and the last K block with real scales (0 outside the logical blocks: padding)
      const int kbv = (tm < args.mb_valid && nb < args.nb_valid) ? args.kb_valid : 0;
#pragma unroll
      for (int i = 0; i < C::HALF; ++i) r[i] = 0.f;
      // The K blocks' scale products, 32 at a time, one per lane: lane l holds that of K block
      // kb0 + 32 j + l.  A load per K block would put its global-memory latency on the promotion's
      // critical path whenever the block's product is already waiting in TMEM.
      float sc_lane = 0.f;
      for (int kb = kb0; kb < kb1; ++kb) {
        const int rel = kb - kb0;
        if ((rel & 31) == 0) {
          // (scale pointers are recomputed from the kernel parameters: registers are scarce here)
          const int k = kb + lane;
          sc_lane = (k < kb1 && k < kbv) ? args.sA[static_cast<size_t>(tm) * args.sa_ld + k] *
                                               args.sB[static_cast<size_t>(k) * args.sb_ld + nb]
                                         : 0.f;
        }
        const float sc = __shfl_sync(FULL, sc_lane, rel & 31);
        const int buf = C::HALVES == 2 ? 2 * acc + hc : acc;
        if (!mbar_wait_warp(tfull_bar(buf), aph, args.timeout, abort_flag)) return false;
        if constexpr (!COUPLED) {
          if (e == (decltype(half)::value ? 0 : (C::HALVES - 1) * 4) && lane == 0) mbar_arrive(empty_bar(pstage));  // this CTA's copy of the stage is free
          if (++pstage == C::STAGES) pstage = 0;
        }
        tc_fence_after();
        const uint32_t t = tmem_base + (static_cast<uint32_t>(q * 32) << 16) +
                           static_cast<uint32_t>(buf * C::NB + (C::HALVES == 2 ? 0 : hc * C::HALF));
        // 32 columns at a time: the next 32 are on their way while these are added, and the
        // buffer is released as soon as the last have arrived, before they are added.
        uint32_t p[2][32];
        tmem_ld_32x32b_x32(t, p[0]);
        tmem_ld_wait_for(p[0]);
#pragma unroll
        for (int c = 0; c < C::HALF / 32; ++c) {
          if (c + 1 < C::HALF / 32) {
            tmem_ld_32x32b_x32(t + (c + 1) * 32, p[(c + 1) & 1]);
          } else {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) {
              if constexpr (PAIR)
                mbar_arrive_cluster_relaxed(mapa_shared(tempty_bar(buf), 0));  // the even CTA's MMA reuses it
              else
                mbar_arrive(tempty_bar(buf));
            }
          }
#pragma unroll
          for (int i = 0; i < 32; i += 2) add_scaled<BN == 256>(r[c * 32 + i], r[c * 32 + i + 1], p[c & 1][i], p[c & 1][i + 1], sc);
          if (c + 1 < C::HALF / 32) tmem_ld_wait_for(p[(c + 1) & 1]);
        }
        if (++acc == C::DEPTH) {
          acc = 0;
          aph ^= 1u;
        }
      }
      return true;
    };
    for (int u = cid; ok && u < total; u += ncl) {
      const int s = u % S;
      int tm, tn;
      const int tile = tile_of(u, tm, tn);
      float r[C::HALF];
      ok = promote(tm, tn * BN + hc * C::HALF, kb_lo(s), s + 1 == S ? args.kblocks : kb_lo(s + 1), r, std::false_type{});
      if (!ok) break;
      const int row0 = tm * BM + q * 32;
      if constexpr (!SPLIT) {
#pragma unroll
        for (int c = 0; c < C::HALF / 32; ++c) {
          const int col0 = tn * BN + hc * C::HALF + c * 32;
          if (row0 < args.M && col0 < args.N) put_block<C::NSTG>(&tmC, r + c * 32, row0, col0, args.beta != 0, stg0, sbuf, lane);
        }
        continue;
      }
      if constexpr (SPLIT) {
      // Split-K: store the partial to this split's slot of the workspace, wait for
      // the stores, fence them against the generic proxy and take the (tile, warp)
      // ticket.
#pragma unroll
      for (int c = 0; c < C::HALF / 32; ++c)
        put_block<C::NSTG>(&tmW, r + c * 32, (s * ntiles + tile) * BM + q * 32, hc * C::HALF + c * 32, false, stg0, sbuf, lane);
      if (lane == 0) {
        bulk_wait<0>();
        fence_proxy_async_global();
      }
      __syncwarp();
      int last = 0;
      if (lane == 0) {
        int32_t* tk = args.tickets + static_cast<size_t>(tile) * kEpiWarps + e;
        const int old = atom_add_acq_rel_gpu(tk, 1);
        last = (old == S - 1);
        if (last) *tk = 0;
      }
      last = __shfl_sync(FULL, last, 0);
      if (!last) continue;
      // The last arriver sums the S partials of its rows in the fixed order 0..S-1,
      // its own included (it was stored and fenced above), so the accumulators are
      // no longer live; lane l reads row l of the warp's 32 rows.
#pragma unroll 1
      for (int c = 0; c < C::HALF / 32; ++c) {
        float sum[32];
        for (int tb = 0; tb < S; ++tb) {  // sum = ((p_0 + p_1) + p_2) + ...
          const float4* src = reinterpret_cast<const float4*>(
              args.ws + static_cast<size_t>((tb * ntiles + tile) * BM + q * 32 + lane) * BN + hc * C::HALF + c * 32);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float4 v4 = __ldcg(src + j);
            if (tb == 0) {
              sum[4 * j] = v4.x;
              sum[4 * j + 1] = v4.y;
              sum[4 * j + 2] = v4.z;
              sum[4 * j + 3] = v4.w;
            } else {
              sum[4 * j] += v4.x;
              sum[4 * j + 1] += v4.y;
              sum[4 * j + 2] += v4.z;
              sum[4 * j + 3] += v4.w;
            }
          }
        }
        const int col0 = tn * BN + hc * C::HALF + c * 32;
        if (row0 < args.M && col0 < args.N) put_block<C::NSTG>(&tmC, sum, row0, col0, args.beta != 0, stg0, sbuf, lane);
      }
      }
    }
    if constexpr (TAIL) {
      if (ok && half_unit >= 0 && hc == 0) {
        int tm, tn;
        tile_of(args.whole + half_unit / 2, tm, tn);
        const int col = tn * BN + half_unit % 2 * C::HALF;
        float r[C::HALF];
        ok = promote(tm, col, 0, args.kblocks, r, std::true_type{});
        if (ok)
#pragma unroll
          for (int c = 0; c < C::HALF / 32; ++c)
            if (tm * BM + q * 32 < args.M && col + c * 32 < args.N)
              put_block<C::NSTG>(&tmC, r + c * 32, tm * BM + q * 32, col + c * 32, args.beta != 0, stg0, sbuf, lane);
      }
    }
    if (!ok && lane == 0) {
      atomicExch(args.err, 3);
      *abort_flag = 1;
    }
    // the staging buffers must have been read before the CTA exits; the global writes
    // themselves complete with the grid (a dependent grid's griddepcontrol.wait sees them)
    if (lane == 0) bulk_wait_read<0>();
    __syncwarp();
  }
  __syncthreads();
  // no CTA of a pair exits while its partner may still arrive on its barriers or run
  // MMAs on its shared memory and TMEM
  if constexpr (PAIR) cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    if constexpr (PAIR)
      tmem_dealloc_pair(tmem_base, 512);
    else
      tmem_dealloc(tmem_base, 512);
  }
}

template <int BN, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_fp8_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmW,
                    const Args args) {
  fp8_body<BN, SPLIT, false>(tmA, tmB, tmC, tmW, args);
}

// The 256 x 256 tile as a cta_group::2 pair (grid: 2 CTAs per cluster).
template <bool SPLIT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    gemm_fp8_2sm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                        const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmW,
                        const Args args) {
  fp8_body<256, SPLIT, true>(tmA, tmB, tmC, tmW, args);
}

__device__ __forceinline__ uint32_t e4m3x4(float a, float b, float c, float d) {
  return static_cast<uint32_t>(__nv_cvt_float2_to_fp8x2(make_float2(a, b), __NV_SATFINITE, __NV_E4M3)) |
         static_cast<uint32_t>(__nv_cvt_float2_to_fp8x2(make_float2(c, d), __NV_SATFINITE, __NV_E4M3)) << 16;
}

// One CTA per 128 x 128 block: amax, scale = amax / 448 (1 for an all-zero
// block), codes = e4m3(x / scale) rounded to nearest even with saturation.
// Bound by HBM (5 bytes per element).  X is read once, its block held in registers
// between the amax and the codes (a warp's rows in turn, four columns per lane), with
// 16-byte loads and 4-byte stores of four codes where VEC (X 16-byte aligned, ldx a
// multiple of 4, Q 4-byte aligned, ldq a multiple of 4); else, and at a ragged right
// edge, element by element.
// The codes are those of the rounded quotient x / s, found without dividing: with
// i = 1 / s rounded, x i (1 - 2^-21) and x i (1 + 2^-21) lie below and above x / s by at
// least 2^-22 of it (each of their three roundings moves them by at most 2^-24), so below
// and above its rounding to FP32; e4m3 rounding is monotonic, so where both give the same
// code it is the quotient's.  Where they differ (about one group of four in 10^4) the
// quotients are divided.  A scale outside [2^-100, 2^100] divides everywhere (there 1 / s
// may overflow or lose bits).
// 4096^2: 90 us reading X twice with 4-byte accesses; 21.2 in one pass with divisions; 15.4
// with the products, programmatic dependent launch and unguarded accesses in the interior
// blocks (512 threads); 14.4 with 256 threads, three CTAs an SM (12.4 at the measured HBM
// rate); 8192^2: 309 -> 50.4, 98 % of that rate.  512 threads are the faster where the blocks
// make less than two waves of them (1024 x 4096: 4.7 against 5.5 us) and at ragged edges,
// whose guarded blocks take longer (4000 x 4004: 18.0 against 24.2 us).
// X is no __restrict__ pointer: the kernel may start while its stream's previous kernel still writes X, so X's bytes
// are not constant over the kernel and must not be read ahead of the dependency wait.
template <bool VEC, int T>
__global__ void __launch_bounds__(T, T == 256 ? 3 : 2)
    quantize_kernel(const float* X, int64_t rows, int64_t cols, int64_t ldx, uint8_t* Q, int64_t ldq, float* scales,
                    int64_t s_ld) {
  constexpr int kWarps = T / 32, kRows = 128 / kWarps;  // warps, rows per warp
  __shared__ float red[kWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t r0 = static_cast<int64_t>(blockIdx.y) * 128 + warp;  // the warp's rows: r0 + i * kWarps
  const int64_t c = static_cast<int64_t>(blockIdx.x) * 128 + 4 * lane;
  const bool whole = VEC && c + 4 <= cols;  // the lane's four columns are a vector
  // an interior block, the same for the whole CTA: its loads and stores have no guards between them
  const bool inner = VEC && (static_cast<int64_t>(blockIdx.y) + 1) * 128 <= rows &&
                     (static_cast<int64_t>(blockIdx.x) + 1) * 128 <= cols;
  const float* src = X + r0 * ldx + c;
  uint8_t* dst = Q + r0 * ldq + c;
  grid_dependency_wait();
  grid_launch_dependents();
  float4 x[kRows];
  if (inner) {
#pragma unroll
    for (int i = 0; i < kRows; ++i) x[i] = __ldcs(reinterpret_cast<const float4*>(src + i * kWarps * ldx));
  } else {
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const float* p = src + i * kWarps * ldx;
      const bool in = r0 + i * kWarps < rows;
      if (whole && in) {
        x[i] = __ldcs(reinterpret_cast<const float4*>(p));
      } else {
        x[i].x = (in && c < cols) ? p[0] : 0.f;
        x[i].y = (in && c + 1 < cols) ? p[1] : 0.f;
        x[i].z = (in && c + 2 < cols) ? p[2] : 0.f;
        x[i].w = (in && c + 3 < cols) ? p[3] : 0.f;
      }
    }
  }
  float amax = 0.f;
#pragma unroll
  for (int i = 0; i < kRows; ++i)
    amax = fmaxf(fmaxf(fmaxf(fmaxf(amax, fabsf(x[i].x)), fabsf(x[i].y)), fabsf(x[i].z)), fabsf(x[i].w));
  for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
  if (lane == 0) red[warp] = amax;
  __syncthreads();
  float m = red[0];
#pragma unroll
  for (int w = 1; w < kWarps; ++w) m = fmaxf(m, red[w]);
  const float s = m > 0.f ? __fdiv_rn(m, 448.0f) : 1.0f;
  if (threadIdx.x == 0) scales[static_cast<int64_t>(blockIdx.y) * s_ld + blockIdx.x] = s;
  const bool divide = !(s >= 0x1p-100f && s <= 0x1p100f);
  const float inv = __fdiv_rn(1.0f, s);
  const float lo = inv * (1.0f - 0x1p-21f), hi = inv * (1.0f + 0x1p-21f);
  auto codes = [&](const float4& v) {
    uint32_t q = e4m3x4(v.x * lo, v.y * lo, v.z * lo, v.w * lo);
    if (divide || q != e4m3x4(v.x * hi, v.y * hi, v.z * hi, v.w * hi))
      q = e4m3x4(__fdiv_rn(v.x, s), __fdiv_rn(v.y, s), __fdiv_rn(v.z, s), __fdiv_rn(v.w, s));
    return q;
  };
  if (inner) {
#pragma unroll
    for (int i = 0; i < kRows; ++i) *reinterpret_cast<uint32_t*>(dst + i * kWarps * ldq) = codes(x[i]);
  } else {
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const uint32_t q = codes(x[i]);
      uint8_t* p = dst + i * kWarps * ldq;
      const bool in = r0 + i * kWarps < rows;
      if (whole && in) {
        *reinterpret_cast<uint32_t*>(p) = q;
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (in && c + j < cols) p[j] = static_cast<uint8_t>(q >> (8 * j));
      }
    }
  }
}

}  // namespace fp8

int fp8_make_map(CUtensorMap* m, CUtensorMapDataType dt, const void* base, uint64_t inner, uint64_t outer,
                 uint64_t row_bytes, uint32_t box_inner, uint32_t box_outer);
cudaError_t fp8_launch_pdl(const void* fn, dim3 grid, int threads, int smem, cudaStream_t st, void** params);

namespace fp8 {

using KernFn = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const Args);
struct TileInfo {
  KernFn fn;        // S = 1
  KernFn fn_split;  // S > 1
  int bn, smem;
  bool pair;        // cta_group::2: 256 x bn tiles on 2-CTA clusters
};
// FP8 tiles: 0 = 128 x 256, 1 = 128 x 128, 2 = 256 x 256 as a cta_group::2 pair.
static TileInfo tile_info(int tile) {
  switch (tile) {
    case 0:
      return TileInfo{gemm_fp8_kernel<256, false>, gemm_fp8_kernel<256, true>, 256, Cfg<256>::SMEM_BYTES, false};
    case 1:
      return TileInfo{gemm_fp8_kernel<128, false>, gemm_fp8_kernel<128, true>, 128, Cfg<128>::SMEM_BYTES, false};
    default:
      return TileInfo{gemm_fp8_2sm_kernel<false>, gemm_fp8_2sm_kernel<true>, 256, Cfg<256, true>::SMEM_BYTES, true};
  }
}

// The kernels' shared-memory limit, once per device.
static int kernels_ready() {
  static std::mutex mu;
  static bool done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return fail(RG_ERR_CUDA, std::string("FP8: cudaGetDevice: ") + cudaGetErrorString(e));
  std::lock_guard<std::mutex> lk(mu);
  if (dev >= 0 && dev < 64 && done[dev]) return RG_OK;
  for (int t = 0; t < RG_FP8_NUM_TILES; ++t) {
    const TileInfo ti = tile_info(t);
    for (KernFn fn : {ti.fn, ti.fn_split}) {
      e = cudaFuncSetAttribute(reinterpret_cast<const void*>(fn), cudaFuncAttributeMaxDynamicSharedMemorySize, ti.smem);
      if (e != cudaSuccess) return fail(RG_ERR_CUDA, "FP8: shared-memory attribute");
      // The register split grows the promotion warps to what warpgroup 0 gives back, so it
      // holds only if every thread launches with exactly kLaunchRegs registers: a kernel built
      // with fewer would wait forever in setmaxnreg.inc, and is never launched.
      cudaFuncAttributes fa{};
      e = cudaFuncGetAttributes(&fa, reinterpret_cast<const void*>(fn));
      if (e != cudaSuccess) return fail(RG_ERR_CUDA, "FP8: kernel attributes");
      if (fa.numRegs != kLaunchRegs)
        return fail(RG_ERR_CUDA, "FP8: kernel built with " + std::to_string(fa.numRegs) +
                                     " registers per thread; its register split needs " +
                                     std::to_string(kLaunchRegs));
    }
  }
  if (dev >= 0 && dev < 64) done[dev] = true;
  return RG_OK;
}

struct Launch {
  KernFn fn = nullptr;
  CUtensorMap a, b, c, w;
  Args args{};
  dim3 grid;
  int smem = 0;
  bool noop = false, zero_only = false;
  float* C = nullptr;
  int64_t M = 0, N = 0, ldc = 0;
};

// 128 x 256 tiles of the last (or only) wave that run as two units of half the columns each: those r = T mod P of
// T tiles on P SMs where 2 r <= P, so that the halves fill SMs the wave would leave idle.  A half takes about 0.65
// of a tile's time, and every output is summed over K in the same order.  512 x 1536 x 2048 (24 tiles) 10.6 -> 8.6 us,
// 3072 x 2048 x 4096 (40 beyond a wave) 30.3 -> 27.3, 4096^3 (56 beyond three) 60.3 -> 57.5.
static int64_t half_tiles(int64_t tiles, int64_t p) {
  const int64_t r = tiles % p;
  return 2 * r <= p ? r : 0;
}

// Checks one FP8 GEMM launch and builds its tensor maps and arguments.
static int prepare(const Fp8CtxInfo& info, int64_t M, int64_t N, int64_t K, const uint8_t* qA, int64_t lda,
                   const float* sA, int64_t lds_a, const uint8_t* qB, int64_t ldb, const float* sB, int64_t lds_b,
                   float* C, int64_t ldc, int32_t variant, int32_t beta, int64_t pm, int64_t pn, int64_t pk,
                   Launch* L) {
  if (!variant_fp8(variant)) return fail(RG_ERR_INVALID, "FP8 GEMM: not an FP8 variant id");
  if (M < 0 || N < 0 || K < 0) return fail(RG_ERR_INVALID, "FP8 GEMM: negative size");
  if (beta != 0 && beta != 1) return fail(RG_ERR_INVALID, "FP8 GEMM: beta must be 0 or 1");
  if (pm == 0) pm = M;
  if (pn == 0) pn = N;
  if (pk == 0) pk = K;
  if (pm < M || pn < N || pk < K) return fail(RG_ERR_INVALID, "FP8 GEMM: padded extents smaller than the problem");
  if (pm > (1 << 30) || pn > (1 << 30) || pk > (1 << 30)) return fail(RG_ERR_SHAPE, "FP8 GEMM: size beyond 2^30");
  *L = Launch{};
  if (M == 0 || N == 0) {
    L->noop = true;
    return RG_OK;
  }
  if (!C) return fail(RG_ERR_INVALID, "FP8 GEMM: null C");
  if (ldc < N) return fail(RG_ERR_INVALID, "FP8 GEMM: ldc < N");
  if ((reinterpret_cast<uintptr_t>(C) & 15) || (ldc % 4)) return fail(RG_ERR_ALIGN, "FP8 GEMM: C 16-byte aligned, ldc % 4");
  if (K == 0) {
    L->zero_only = beta == 0;
    L->noop = beta != 0;
    L->C = C;
    L->M = M;
    L->N = N;
    L->ldc = ldc;
    return RG_OK;
  }
  if (!qA || !qB || !sA || !sB) return fail(RG_ERR_INVALID, "FP8 GEMM: null operand");
  const int64_t kb_valid = (K + BK - 1) / BK, nb_valid = (N + SB - 1) / SB, mb_valid = (M + SB - 1) / SB;
  if (lda < K || ldb < N || lds_a < kb_valid || lds_b < nb_valid)
    return fail(RG_ERR_INVALID, "FP8 GEMM: leading dimensions");
  if ((reinterpret_cast<uintptr_t>(qA) & 15) || (reinterpret_cast<uintptr_t>(qB) & 15) || (lda % 16) || (ldb % 16))
    return fail(RG_ERR_ALIGN, "FP8 GEMM: 16-byte aligned operands, lda and ldb multiples of 16");
  const int tile = (variant - RG_FP8_VARIANT_BASE) / RG_NUM_SPLITS;
  const int splits = 1 << ((variant - RG_FP8_VARIANT_BASE) % RG_NUM_SPLITS);
  const TileInfo ti = tile_info(tile);
  int64_t tiles_m = (pm + BM - 1) / BM;
  if (ti.pair) tiles_m += tiles_m & 1;  // whole 256-row pair tiles (an odd CTA past M loads zeros, stores nothing)
  const int64_t tiles_n = (pn + ti.bn - 1) / ti.bn, kblocks = (pk + BK - 1) / BK;
  const int64_t ntiles = tiles_m * tiles_n;
  const int64_t halves = ti.pair || ti.bn != 256 || splits > 1 ? 0 : half_tiles(ntiles, info.sms);
  if (splits > 1 && (splits * ntiles * BM * ti.bn * 4 > info.ws_bytes || ntiles * kEpiWarps > info.max_tickets))
    return fail(RG_ERR_SHAPE, "FP8 GEMM: split-K workspace too small for this shape");
  if (ntiles * splits > (1LL << 30)) return fail(RG_ERR_SHAPE, "FP8 GEMM: too many work units");
  int rc = fp8_make_map(&L->a, CU_TENSOR_MAP_DATA_TYPE_UINT8, qA, K, M, lda, BK, BM);
  if (rc == RG_OK) rc = fp8_make_map(&L->b, CU_TENSOR_MAP_DATA_TYPE_UINT8, qB, N, K, ldb, 128, BK);
  if (rc == RG_OK) rc = fp8_make_map(&L->c, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, C, N, M, ldc * 4, 32, 32);
  if (rc == RG_OK) {
    if (splits > 1)
      rc = fp8_make_map(&L->w, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, info.ws, ti.bn,
                        static_cast<uint64_t>(splits * ntiles * BM), static_cast<uint64_t>(ti.bn) * 4, 32, 32);
    else
      L->w = L->c;  // unused without split-K
  }
  if (rc != RG_OK) return rc;
  Args& g = L->args;
  g.M = static_cast<int32_t>(M);
  g.N = static_cast<int32_t>(N);
  g.tiles_m = static_cast<int32_t>(tiles_m);
  g.tiles_n = static_cast<int32_t>(tiles_n);
  g.kblocks = static_cast<int32_t>(kblocks);
  g.splits = splits;
  g.whole = static_cast<int32_t>(ntiles - halves);
  g.beta = beta;
  g.mb_valid = static_cast<int32_t>(mb_valid);
  g.kb_valid = static_cast<int32_t>(kb_valid);
  g.nb_valid = static_cast<int32_t>(nb_valid);
  g.sa_ld = static_cast<int32_t>(lds_a);
  g.sb_ld = static_cast<int32_t>(lds_b);
  g.sA = sA;
  g.sB = sB;
  g.ws = info.ws;
  g.tickets = info.tickets;
  g.err = info.err;
  g.timeout = info.timeout;
  L->fn = splits > 1 ? ti.fn_split : ti.fn;
  L->smem = ti.smem;
  L->grid = ti.pair ? dim3(static_cast<unsigned>(2 * std::min<int64_t>(ntiles / 2 * splits, info.sms / 2)))
                    : dim3(static_cast<unsigned>(std::min<int64_t>(ntiles * splits + halves, info.sms)));
  return RG_OK;
}

static cudaError_t launch(const Launch& L, cudaStream_t st) {
  if (L.noop) return cudaSuccess;
  if (L.zero_only) return cudaMemset2DAsync(L.C, L.ldc * 4, 0, L.N * 4, L.M, st);
  void* params[5] = {const_cast<CUtensorMap*>(&L.a), const_cast<CUtensorMap*>(&L.b), const_cast<CUtensorMap*>(&L.c),
                     const_cast<CUtensorMap*>(&L.w), const_cast<Args*>(&L.args)};
  return fp8_launch_pdl(reinterpret_cast<const void*>(L.fn), L.grid, kThreads, L.smem, st, params);
}

// The leaves of an FP8 plan's cell covering (M, N, K), clipped to the problem, on sub-views.
static int plan_launches(const Fp8CtxInfo& info, const rg_plan* plan, int64_t M, int64_t N, int64_t K,
                         const uint8_t* qA, int64_t lda, const float* sA, int64_t lds_a, const uint8_t* qB,
                         int64_t ldb, const float* sB, int64_t lds_b, float* C, int64_t ldc, std::vector<Launch>& out) {
  out.clear();
  if (!plan) return fail(RG_ERR_INVALID, "FP8 plan: null plan");
  if (M <= 0 || N <= 0 || K <= 0) return fail(RG_ERR_INVALID, "FP8 plan: sizes must be positive");
  const Plan& P = plan->p;
  if (P.variant_ids.empty() || !variant_fp8(P.variant_ids[0]))
    return fail(RG_ERR_INVALID, "FP8 plan: a BF16 plan runs through rg_gemm_plan");
  int64_t cell = 0;
  if (plan_cell(P, M, N, K, &cell) != RG_OK) return fail(RG_ERR_SHAPE, "FP8 plan: shape beyond the plan grid");
  for (int64_t i = P.leaf_off[cell]; i < P.leaf_off[cell + 1]; ++i) {
    const rg_leaf& lf = P.leaves[i];
    if (lf.m0 >= M || lf.n0 >= N || lf.k0 >= K) continue;  // wholly in the padding
    if ((lf.m0 % SB) || (lf.n0 % SB) || (lf.k0 % SB))
      return fail(RG_ERR_SHAPE, "FP8 plan: a leaf's offsets are not multiples of the 128-element scale block");
    const int64_t m = std::min(lf.m, M - lf.m0), n = std::min(lf.n, N - lf.n0), k = std::min(lf.k, K - lf.k0);
    Launch L;
    const int rc = prepare(info, m, n, k, qA + lf.m0 * lda + lf.k0, lda, sA + (lf.m0 / SB) * lds_a + lf.k0 / SB,
                           lds_a, qB + lf.k0 * ldb + lf.n0, ldb, sB + (lf.k0 / SB) * lds_b + lf.n0 / SB, lds_b,
                           C + lf.m0 * ldc + lf.n0, ldc, lf.variant, lf.beta, lf.pm, lf.pn, lf.pk, &L);
    if (rc != RG_OK) return rc;
    out.push_back(L);
  }
  return RG_OK;
}

}  // namespace fp8

}  // namespace rg

extern "C" int rg_fp8_quantize(rg_ctx* ctx, const float* X, int64_t rows, int64_t cols, int64_t ldx, uint8_t* Q,
                               int64_t ldq, float* scales, void* stream) {
  rg::clear_error();
  if (!ctx) return rg::fail(RG_ERR_INVALID, "rg_fp8_quantize: null context");
  if (rows < 0 || cols < 0 || ldx < cols || ldq < cols) return rg::fail(RG_ERR_INVALID, "rg_fp8_quantize: sizes");
  if (rows == 0 || cols == 0) return RG_OK;
  if (!X || !Q || !scales) return rg::fail(RG_ERR_INVALID, "rg_fp8_quantize: null pointer");
  const int64_t br = (rows + 127) / 128, bc = (cols + 127) / 128;
  if (br > 65535 || bc > (1LL << 31) - 1) return rg::fail(RG_ERR_SHAPE, "rg_fp8_quantize: too many blocks");
  const bool vec = !(reinterpret_cast<uintptr_t>(X) & 15) && ldx % 4 == 0 && !(reinterpret_cast<uintptr_t>(Q) & 3) &&
                   ldq % 4 == 0;
  rg::Fp8CtxInfo info{};
  const int rc = rg::ctx_fp8_info(ctx, &info);
  if (rc != RG_OK) return rc;
  using rg::fp8::quantize_kernel;
  // the 256-thread kernel: whole blocks, more than two waves of 512-thread CTAs
  const bool many = vec && rows % 128 == 0 && cols % 128 == 0 && bc * br > 4LL * info.sms;
  const auto fn = many ? quantize_kernel<true, 256> : vec ? quantize_kernel<true, 512> : quantize_kernel<false, 512>;
  int64_t s_ld = bc;
  void* params[8] = {&X, &rows, &cols, &ldx, &Q, &ldq, &scales, &s_ld};
  const cudaError_t e = rg::fp8_launch_pdl(reinterpret_cast<const void*>(fn),
                                           dim3(static_cast<unsigned>(bc), static_cast<unsigned>(br)), many ? 256 : 512, 0,
                                           static_cast<cudaStream_t>(stream), params);
  return e == cudaSuccess ? RG_OK : rg::fail(RG_ERR_CUDA, std::string("rg_fp8_quantize: ") + cudaGetErrorString(e));
}

extern "C" int rg_gemm_fp8_ex(rg_ctx* ctx, int64_t M, int64_t N, int64_t K, const uint8_t* qA, int64_t lda,
                              const float* sA, int64_t lds_a, const uint8_t* qB, int64_t ldb, const float* sB,
                              int64_t lds_b, float* C, int64_t ldc, int32_t variant, int32_t beta, int64_t pm,
                              int64_t pn, int64_t pk, void* stream) {
  rg::clear_error();
  rg::Fp8CtxInfo info{};
  int rc = rg::ctx_fp8_info(ctx, &info);
  if (rc != RG_OK) return rc;
  rg::fp8::Launch L;
  rc = rg::fp8::prepare(info, M, N, K, qA, lda, sA, lds_a, qB, ldb, sB, lds_b, C, ldc, variant, beta, pm, pn, pk, &L);
  if (rc != RG_OK) return rc;
  if (!L.noop && !L.zero_only && (rc = rg::fp8::kernels_ready()) != RG_OK) return rc;
  const cudaError_t e = rg::fp8::launch(L, static_cast<cudaStream_t>(stream));
  if (e != cudaSuccess) return rg::fail(RG_ERR_CUDA, std::string("rg_gemm_fp8: launch: ") + cudaGetErrorString(e));
  if (!L.noop && !L.zero_only) rg::ctx_count_launches(ctx, 1);
  return RG_OK;
}

extern "C" int rg_gemm_fp8(rg_ctx* ctx, int64_t M, int64_t N, int64_t K, const uint8_t* qA, int64_t lda,
                           const float* sA, const uint8_t* qB, int64_t ldb, const float* sB, float* C, int64_t ldc,
                           void* stream) {
  return rg_gemm_fp8_ex(ctx, M, N, K, qA, lda, sA, K > 0 ? (K + 127) / 128 : 1, qB, ldb, sB,
                        N > 0 ? (N + 127) / 128 : 1, C, ldc, RG_FP8_VARIANT(0, 0), 0, 0, 0, 0, stream);
}

extern "C" int rg_gemm_fp8_plan(rg_ctx* ctx, const rg_plan* plan, int64_t M, int64_t N, int64_t K, const uint8_t* qA,
                                int64_t lda, const float* sA, int64_t lds_a, const uint8_t* qB, int64_t ldb,
                                const float* sB, int64_t lds_b, float* C, int64_t ldc, void* stream) {
  rg::clear_error();
  rg::Fp8CtxInfo info{};
  int rc = rg::ctx_fp8_info(ctx, &info);
  if (rc != RG_OK) return rc;
  std::vector<rg::fp8::Launch> ls;
  rc = rg::fp8::plan_launches(info, plan, M, N, K, qA, lda, sA, lds_a, qB, ldb, sB, lds_b, C, ldc, ls);
  if (rc != RG_OK) return rc;
  if ((rc = rg::fp8::kernels_ready()) != RG_OK) return rc;
  for (const auto& L : ls) {
    const cudaError_t e = rg::fp8::launch(L, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return rg::fail(RG_ERR_CUDA, std::string("rg_gemm_fp8_plan: launch: ") + cudaGetErrorString(e));
    if (!L.noop && !L.zero_only) rg::ctx_count_launches(ctx, 1);
  }
  return RG_OK;
}

namespace {
uint64_t splitmix_next_fp8(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
}  // namespace

extern "C" int rg_sweep_fp8(rg_ctx* ctx, const rg_grid* grid, int32_t n_variants, const int32_t* variant_ids,
                            const rg_plan* plan, const uint8_t* qA, const float* sA, const uint8_t* qB,
                            const float* sB, float* C, const rg_sweep_opts* opts, int64_t* t_ns_out,
                            double* tflops_out, double* stats_out, void* stream) {
  rg::clear_error();
  using namespace rg::fp8;
  if (!ctx || !grid || !qA || !sA || !qB || !sB || !C || !t_ns_out)
    return rg::fail(RG_ERR_INVALID, "rg_sweep_fp8: null argument");
  if (!rg::grid_valid(*grid)) return rg::fail(RG_ERR_INVALID, "rg_sweep_fp8: invalid grid");
  if (plan ? n_variants != 1 : (n_variants <= 0 || !variant_ids))
    return rg::fail(RG_ERR_INVALID, "rg_sweep_fp8: variants");
  if (!plan)
    for (int32_t i = 0; i < n_variants; ++i)
      if (!rg::variant_fp8(variant_ids[i])) return rg::fail(RG_ERR_INVALID, "rg_sweep_fp8: not an FP8 variant id");
  rg_sweep_opts o;
  rg_sweep_opts_default(&o);
  if (opts) o = *opts;
  if (o.reps <= 0 || o.warmup < 0 || o.global_warmup < 0 || o.spin_ns < 0)
    return rg::fail(RG_ERR_INVALID, "rg_sweep_fp8: options");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t cells = rg::cells_of(*grid);
  const int64_t nk = grid->k.count, nn = grid->n.count;
  rg::Fp8CtxInfo info{};
  int rc = rg::ctx_fp8_info(ctx, &info);
  if (rc != RG_OK) return rc;
  if ((rc = kernels_ready()) != RG_OK) return rc;
  std::vector<int64_t> order(static_cast<size_t>(cells) * n_variants);
  for (size_t i = 0; i < order.size(); ++i) order[i] = static_cast<int64_t>(i);
  if (o.shuffle) {
    uint64_t s = o.seed;
    for (size_t i = order.size() - 1; i > 0; --i) std::swap(order[i], order[splitmix_next_fp8(s) % (i + 1)]);
  }
  auto dims = [&](int64_t item, int64_t* M, int64_t* N, int64_t* K) {
    const int64_t cell = item % cells;
    *M = rg::axis_value(grid->m, cell / (nn * nk));
    *N = rg::axis_value(grid->n, (cell / nk) % nn);
    *K = rg::axis_value(grid->k, cell % nk);
  };
  // a split is worth timing only where the unsplit tiles leave SMs idle (counting both CTAs of
  // a pair tile), a pair tile only beyond 128 rows
  if (o.prune_splits && !plan) {
    std::vector<int64_t> keep;
    keep.reserve(order.size());
    for (int64_t it : order) {
      const int32_t v = variant_ids[it / cells];
      const int S = 1 << ((v - RG_FP8_VARIANT_BASE) % RG_NUM_SPLITS);
      const TileInfo ti = tile_info((v - RG_FP8_VARIANT_BASE) / RG_NUM_SPLITS);
      int64_t M, N, K;
      dims(it, &M, &N, &K);
      bool pruned = ti.pair && M <= 128;
      if (S > 1 && !pruned) {
        const int64_t rows = ti.pair ? 2 * ((M + 2 * BM - 1) / (2 * BM)) : (M + BM - 1) / BM;
        const int64_t ctas = rows * ((N + ti.bn - 1) / ti.bn);
        pruned = ctas >= info.sms || (K + BK - 1) / BK < 2 * S;
      }
      if (pruned)
        t_ns_out[it] = RG_T_UNMEASURED;
      else
        keep.push_back(it);
    }
    order.swap(keep);
  }
  std::vector<Launch> ls;
  auto prep = [&](int64_t item, int* launches) -> int {
    int64_t M, N, K;
    dims(item, &M, &N, &K);
    if ((K % 16) || (N % 16)) return rg::fail(RG_ERR_ALIGN, "rg_sweep_fp8: grid sizes must be multiples of 16");
    const int64_t lds_a = (K + 127) / 128, lds_b = (N + 127) / 128;
    int r;
    if (plan) {
      r = plan_launches(info, plan, M, N, K, qA, K, sA, lds_a, qB, N, sB, lds_b, C, N, ls);
    } else {
      ls.resize(1);
      r = prepare(info, M, N, K, qA, K, sA, lds_a, qB, N, sB, lds_b, C, N, variant_ids[item / cells], 0, 0, 0, 0,
                  &ls[0]);
    }
    *launches = static_cast<int>(ls.size());
    return r;
  };
  int64_t n_launch = 0;
  auto run = [&]() -> cudaError_t {
    for (const auto& L : ls) {
      const cudaError_t e = launch(L, st);
      if (e != cudaSuccess) return e;
      ++n_launch;
    }
    return cudaSuccess;
  };
  rc = rg::timed_sweep(ctx, order, o, st, t_ns_out, prep, run);
  rg::ctx_count_launches(ctx, n_launch);
  if (rc != RG_OK) return rc;
  rc = rg_check(ctx, stream);
  if (rc != RG_OK) return rc;
  return rg::sweep_surfaces(grid, plan ? 1 : n_variants, t_ns_out, tflops_out, stats_out);
}

// ------------------------------------------------------------------ FP8 requests of the serving engine
namespace rg {

int fp8_request_status(const Fp8Request& r) {
  if (r.M <= 0 || r.N <= 0 || r.K <= 0 || !r.qA || !r.qB || !r.sA || !r.sB) return RG_ERR_INVALID;
  if (r.lda < r.K || r.ldb < r.N || (r.C && r.ldc < r.N) || r.lds_a < (r.K + 127) / 128 || r.lds_b < (r.N + 127) / 128)
    return RG_ERR_INVALID;
  if ((reinterpret_cast<uintptr_t>(r.qA) & 15) || (reinterpret_cast<uintptr_t>(r.qB) & 15) || (r.lda % 16) ||
      (r.ldb % 16))
    return RG_ERR_ALIGN;
  if (r.C && ((reinterpret_cast<uintptr_t>(r.C) & 15) || (r.ldc % 4))) return RG_ERR_ALIGN;
  if (r.M > (1 << 30) || r.N > (1 << 30) || r.K > (1 << 30)) return RG_ERR_SHAPE;
  return RG_OK;
}

int fp8_enqueue_phase(rg_ctx* ctx, const rg_plan* plan, const Fp8Request& r, int32_t phase, float* ws,
                      int64_t ws_bytes, int32_t* tickets, int64_t max_tickets, void* stream, int32_t* max_phase) {
  Fp8CtxInfo info{};
  int rc = ctx_fp8_info(ctx, &info);
  if (rc != RG_OK) return rc;
  info.ws = ws;
  info.ws_bytes = ws_bytes;
  info.tickets = tickets;
  info.max_tickets = max_tickets;
  if ((rc = fp8::kernels_ready()) != RG_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  *max_phase = 0;
  if (!plan) {
    if (phase != 0) return RG_OK;
    fp8::Launch L;
    rc = fp8::prepare(info, r.M, r.N, r.K, r.qA, r.lda, r.sA, r.lds_a, r.qB, r.ldb, r.sB, r.lds_b, r.C, r.ldc,
                      RG_FP8_VARIANT(0, 0), 0, 0, 0, 0, &L);
    if (rc != RG_OK) return rc;
    const cudaError_t e = fp8::launch(L, st);
    if (e != cudaSuccess) return fail(RG_ERR_CUDA, std::string("FP8 serving: launch: ") + cudaGetErrorString(e));
    ctx_count_launches(ctx, 1);
    return RG_OK;
  }
  const Plan& P = plan->p;
  if (P.variant_ids.empty() || !variant_fp8(P.variant_ids[0]))
    return fail(RG_ERR_INVALID, "FP8 serving: the FP8 plan holds BF16 variants");
  int64_t cell = 0;
  if (plan_cell(P, r.M, r.N, r.K, &cell) != RG_OK) return fail(RG_ERR_SHAPE, "FP8 serving: shape beyond the plan grid");
  for (int64_t i = P.leaf_off[cell]; i < P.leaf_off[cell + 1]; ++i) {
    const rg_leaf& lf = P.leaves[i];
    *max_phase = std::max(*max_phase, lf.phase);
    if (lf.phase != phase || lf.m0 >= r.M || lf.n0 >= r.N || lf.k0 >= r.K) continue;
    if ((lf.m0 % fp8::SB) || (lf.n0 % fp8::SB) || (lf.k0 % fp8::SB))
      return fail(RG_ERR_SHAPE, "FP8 serving: a leaf's offsets are not multiples of the scale block");
    const int64_t m = std::min(lf.m, r.M - lf.m0), n = std::min(lf.n, r.N - lf.n0), k = std::min(lf.k, r.K - lf.k0);
    fp8::Launch L;
    rc = fp8::prepare(info, m, n, k, r.qA + lf.m0 * r.lda + lf.k0, r.lda, r.sA + (lf.m0 / fp8::SB) * r.lds_a + lf.k0 / fp8::SB,
                      r.lds_a, r.qB + lf.k0 * r.ldb + lf.n0, r.ldb, r.sB + (lf.k0 / fp8::SB) * r.lds_b + lf.n0 / fp8::SB,
                      r.lds_b, r.C + lf.m0 * r.ldc + lf.n0, r.ldc, lf.variant, lf.beta, lf.pm, lf.pn, lf.pk, &L);
    if (rc != RG_OK) return rc;
    const cudaError_t e = fp8::launch(L, st);
    if (e != cudaSuccess) return fail(RG_ERR_CUDA, std::string("FP8 serving: launch: ") + cudaGetErrorString(e));
    if (!L.noop && !L.zero_only) ctx_count_launches(ctx, 1);
  }
  return RG_OK;
}

}  // namespace rg
