// TMA-staged tensor-core grouped GEMM (tcgen05, sm_103a): BF16 operands, FP32
// accumulation in tensor memory.
//
// The operands of the sigma vector live in a few large BF16 matrices (per
// quantum-number group of the cut: the stacked two-site wavefunction Psi_g, the stacked
// right operators, the X intermediates; one matrix per width for the left-operator blocks),
// each described by one tensor map per box height.  A stage of the ring is one or more
// pieces, each a pair of TMA box copies that complete on the stage's mbarrier by transaction
// count; zero fill outside the matrix covers ragged edges.  The tiles' terms are expanded
// before the launch into per-CTA copy lists (stage word, expected bytes, box coordinates:
// fill_lists_kernel), so the producer does no term arithmetic.
//
// Persistent and warp-specialised, two CTAs per SM in the sigma modes (256 tensor-memory
// columns each), one in the exact mode:
//   warp 0     fetches its CTA's copy lists 32 stages at a time into shared memory
//              (1D bulk copies, double-buffered); per stage lane 0 waits for the ring
//              slot and posts the stage word and the expected bytes, then lane p issues
//              the two box copies of piece p
//   warp 1     one thread issues tcgen05.mma (M = 128, N = n, K = 16 per instruction)
//              and commits to the stage's empty barrier / the accumulator's full
//              barrier
//   warps 2-5  epilogue: tcgen05.ld of their 32 tensor-memory lanes; BF16 slices of the X
//              intermediates, FP32 vector reductions (sigma^T, several tiles may add into
//              one block) of per-segment partial sums, or (exact mode) two-float sums of
//              exact integer segments stored in FP64
// One or two (sigma modes) or eight (exact mode, N <= 64) accumulators.  Two CTAs of an SM
// overlap each other's epilogues, products and copies.  Every wait is bounded: on timeout the CTA raises a shared abort flag, records an error,
// waits (bounded) for the copies it issued, frees its tensor memory and returns.
//
// The sigma modes: what bounds them is the operand traffic into shared memory and the issuing
// thread, not the tensor cores: a 128 x n tile of one K=16 product needs 32 (128 + n) bytes
// through L2 for n / 2 tensor clocks.  With two or three slices the products s_i t_j, i + j < nsl,
// share their operands, so a piece brings every slice of both operands once (3 + 3 boxes' worth
// of bytes for six products instead of 6 + 6) in two copies instead of twelve, and the
// column-group layout lets each copy move 256-byte runs instead of 32-byte rows.  The products
// keep the order term, slice pair, column (they are rounded into the accumulator one by one, and
// a Davidson solve magnifies another order's rounding), so a term's pieces stay in the ring until
// its last pair.  Two CTAs per SM: with one, the copies, the products and the epilogue of a tile wait
// for each other (K=24, one CTA: 3.1 ms).  Blocks of more columns than a term may have
// (tm_term_pieces) are cut into several terms by the plan.
// Measured against one pair of swizzled boxes per slice product (16-column boxes in the
// reduce mode), one CTA per SM: three slices at K=24, M=512 3.19 -> 1.45 ms per sigma, K=40, M=1200
// 23.1 -> 12.4 ms, K=10, M=150 0.240 -> 0.137 ms; one pass at K=32, M=1024 2.71 -> 1.57 ms.  (Without
// the fixed order, four instructions of up to 2 n columns per piece and slots released piece by
// piece: 1.27 and 9.2 ms.)  The X intermediates' round trip and the stacked operators, 6.3 GB at
// K=24, take 0.93 ms of that at the measured copy rate.
#include "device_once.hpp"
#include "kernels_tma.hpp"
#include "ptx.cuh"

#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cstdint>
#include <mutex>
#include <thread>
#include <type_traits>

namespace gbdmrg {

long tc_launch_count();
void count_tc_launches(long n);

namespace {

constexpr int TM_THREADS = 192;
constexpr int TM_BOX_K = 64;                    // exact mode: columns per box (128 bytes)
constexpr int TM_A_BYTES = 128 * TM_BOX_K * 2;  // 16 KB
constexpr int TM_REC_BATCH = 32;  // stages of the copy lists fetched per bulk copy

template <int MODE, int NSL>
struct TmCfg {
  static constexpr bool STORE = MODE == TM_MODE_STORE_BF16;
  static constexpr bool EXACT = MODE == TM_MODE_EXACT_F64;
  // two or three slices: a term's 16-column pieces, one per ring slot, stay until all slice
  // products of the term have been issued
  static constexpr bool CHAIN = !EXACT && NSL > 1;
  static constexpr int CTAS = tm_ctas(MODE);
  static constexpr int NMAX = tm_max_n(MODE, NSL);
  static constexpr int TMEM = EXACT ? 512 : 256;
  static constexpr int NACC = TMEM / NMAX;
  static constexpr int SLOTS = EXACT ? 1 : tm_slots(NSL);
  // bytes of one piece of A and of the largest piece of B (all slices)
  static constexpr int A_BYTES = EXACT ? TM_A_BYTES : 128 * TM_PIECE_COLS * 2 * NSL;
  static constexpr int B_BYTES = EXACT ? NMAX * TM_BOX_K * 2 : NMAX * TM_PIECE_COLS * 2 * NSL;
  static constexpr int STAGE_BYTES = SLOTS * (A_BYTES + B_BYTES);  // (chains: a launch's own slot size)
  static constexpr int STAGES = EXACT ? 8 : (STORE ? 4 : 6);       // (chains: a launch's own count)
  static constexpr int SMEM = (CHAIN ? TM_RING_BYTES : STAGES * STAGE_BYTES) + 1024;
};
constexpr int TM_MAX_STAGES = TM_MAX_SLOTS, TM_MAX_ACC = 8;
constexpr int TM_TERMS = 32;  // term barriers of the chains (a power of two, more than twice the slots)
static_assert(TM_TERMS > 2 * TM_MAX_SLOTS, "a ring's terms need distinct barriers");

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
          dst),
      "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// box of a column-group map: all of dimension 0, row group y, every slice, column group x
__device__ __forceinline__ void tma_load_groups(uint32_t dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];\n" ::"r"(dst),
      "l"(map), "r"(0), "r"(y), "r"(0), "r"(x), "r"(smem_u32(bar))
      : "memory");
}

// 1D bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16), completing on bar
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// 16 of them
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
        "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}

template <int MODE, int NSL>
__global__ void __launch_bounds__(TM_THREADS, tm_ctas(MODE))
    gemm_tma_kernel(const TmTile* __restrict__ tiles, int ntiles, const TmTerm* __restrict__ terms,
                    const CUtensorMap* __restrict__ maps, const long* __restrict__ rowmap, void* __restrict__ out,
                    int* __restrict__ err, const int* __restrict__ expo, const int* __restrict__ cta_stage,
                    const TmStage* __restrict__ stg, const TmPiece* __restrict__ pcs, int ring_slots,
                    int slot_bytes) {
  using Cfg = TmCfg<MODE, NSL>;
  constexpr bool CHAIN = Cfg::CHAIN;
  const int S = CHAIN ? ring_slots : Cfg::STAGES;
  const int STAGE_BYTES = CHAIN ? slot_bytes : Cfg::STAGE_BYTES;
  constexpr int NACC = Cfg::NACC;
  constexpr int NMAX = Cfg::NMAX;
  constexpr bool STORE = Cfg::STORE;
  constexpr bool EXACT = Cfg::EXACT;
  extern __shared__ uint8_t dsm[];
  __shared__ __align__(8) uint64_t full_b[TM_MAX_STAGES], empty_b[TM_MAX_STAGES], tfull_b[TM_MAX_ACC],
      tempty_b[TM_MAX_ACC];
  __shared__ __align__(8) uint64_t term_b[CHAIN ? TM_TERMS : 1];
  __shared__ uint32_t tmem_base_sh;
  __shared__ int abort_sh;
  // per stage: the stage word (TmStage)
  __shared__ uint64_t meta[TM_MAX_STAGES];
  // copy lists of the producer: batches of TM_REC_BATCH stages, double-buffered, each
  // landing by bulk copy on rec_b[buffer]
  constexpr int PCS = Cfg::SLOTS;
  __shared__ __align__(16) TmStage rec_stage[2][TM_REC_BATCH];
  __shared__ __align__(16) TmPiece rec_piece[2][TM_REC_BATCH * PCS];
  __shared__ __align__(8) uint64_t rec_b[2];
  const uint32_t base = (smem_u32(dsm) + 1023u) & ~1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (warp == 2) {  // an epilogue warp (all lanes take the same path) owns the tensor memory
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&tmem_base_sh)),
                 "r"(Cfg::TMEM));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::);
  }
  if (tid == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full_b[s], 1);  // the producer's arrive (with the expected bytes)
      mbar_init(&empty_b[s], 1);
    }
    if (CHAIN)
      for (int t = 0; t < TM_TERMS; ++t) mbar_init(&term_b[t], 1);
    for (int a = 0; a < NACC; ++a) {
      mbar_init(&tfull_b[a], 1);
      mbar_init(&tempty_b[a], 128);
    }
    mbar_init(&rec_b[0], 1);
    mbar_init(&rec_b[1], 1);
    abort_sh = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::);
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
  const uint32_t tmem = tmem_base_sh;
  volatile int* abort_flag = &abort_sh;

  if (warp == 0) {
    // ---------------- TMA producer: the CTA's stages from the copy lists, fetched into
    // shared memory TM_REC_BATCH stages at a time by bulk copies one batch ahead.  Per
    // stage lane 0 waits until the ring slot is free and posts the stage word and the
    // expected bytes, then lane p < np issues the two box copies of piece p.
    constexpr int PIECES = PCS;
    constexpr unsigned FULL = 0xffffffffu;
    long j = 0;            // stages issued
    long freed = 0;        // (chains) stages released, by the terms before `th`; terms issued
    int th = 0, tq = 0, left = 0;  // pieces of the current term still to come
    __shared__ unsigned char term_size[CHAIN ? TM_TERMS : 1];
    int st = 0;            // ring slot of the next one (j % S)
    uint32_t par = 0;      // its round's parity ((j / S) & 1)
    bool wrapped = false;  // j >= S
    bool ok = true;
    const int s_beg = cta_stage[blockIdx.x], s_end = cta_stage[blockIdx.x + 1];
    const int nbatch = (s_end - s_beg + TM_REC_BATCH - 1) / TM_REC_BATCH;
    int fetched = 0;  // record batches whose copies were issued
    auto fetch = [&](int b) {  // lane 0
      const int f0 = s_beg + b * TM_REC_BATCH, n = min(TM_REC_BATCH, s_end - f0);
      const uint32_t hb = (uint32_t)n * sizeof(TmStage), pb = (uint32_t)(n * PIECES) * sizeof(TmPiece);
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      mbar_arrive_expect_tx(&rec_b[b & 1], hb + pb);
      bulk_load(smem_u32(&rec_stage[b & 1][0]), stg + f0, hb, &rec_b[b & 1]);
      bulk_load(smem_u32(&rec_piece[b & 1][0]), pcs + (long)f0 * PIECES, pb, &rec_b[b & 1]);
    };
    if (lane == 0 && nbatch > 0) fetch(0);
    fetched = nbatch > 0 ? 1 : 0;
    for (int b = 0; b < nbatch && ok; ++b) {
      __syncwarp();  // the lanes' reads of the buffer batch b + 1 reuses are done
      if (lane == 0) {
        if (b + 1 < nbatch) fetch(b + 1);
        if (!mbar_wait(&rec_b[b & 1], (uint32_t)((b >> 1) & 1), abort_flag)) ok = false;
      }
      if (b + 1 < nbatch) fetched = b + 2;
      ok = __shfl_sync(FULL, ok, 0);
      if (!ok) break;
      const int f0 = s_beg + b * TM_REC_BATCH, n = min(TM_REC_BATCH, s_end - f0);
      for (int i = 0; i < n && ok; ++i) {
        const TmStage h = rec_stage[b & 1][i];
        if (lane == 0) {
          if constexpr (CHAIN) {
            if (left == 0) {  // first piece of a term
              left = (int)((uint32_t)(h.word >> 32) & 255u);
              term_size[tq++ & (TM_TERMS - 1)] = (unsigned char)left;
            }
            --left;
            // at most S <= TM_TERMS / 2 terms are in the ring, so their barriers and sizes are distinct
            while (ok && j - freed >= S) {
              ok = mbar_wait(&term_b[th & (TM_TERMS - 1)], (uint32_t)((th / TM_TERMS) & 1), abort_flag);
              freed += term_size[th & (TM_TERMS - 1)];
              ++th;
            }
          } else {
            if (wrapped && !mbar_wait(&empty_b[st], par ^ 1u, abort_flag)) ok = false;
          }
          if (ok) {
            meta[st] = h.word;
            mbar_arrive_expect_tx(&full_b[st], h.bytes);
          }
        }
        ok = __shfl_sync(FULL, ok, 0);
        if (!ok) break;
        if (lane < h.np) {
          const TmPiece q = rec_piece[b & 1][i * PIECES + lane];
          const uint32_t sa = base + st * STAGE_BYTES;
          const uint32_t da = sa + lane * Cfg::A_BYTES, db = sa + PIECES * Cfg::A_BYTES + lane * Cfg::B_BYTES;
          if constexpr (EXACT) {
            tma_load_2d(da, maps + q.amap, q.ax, q.ay, &full_b[st]);
            tma_load_2d(db, maps + q.bmap, q.bx, q.by, &full_b[st]);
          } else {
            tma_load_groups(da, maps + q.amap, q.ax, q.ay, &full_b[st]);
            tma_load_groups(db, maps + q.bmap, q.bx, q.by, &full_b[st]);
          }
        }
        ++j;
        if (++st == S) {
          st = 0;
          par ^= 1u;
          wrapped = true;
        }
      }
    }
    if (lane == 0) {
      // every issued copy must land before the CTA may exit: the last (up to S)
      // issued stages complete their full phase when their bytes arrive, and so does
      // the last record batch fetched
      for (long qq = j - 1; qq >= 0 && qq >= j - S; --qq) {
        const int s2 = (int)(qq % S);
        for (long it = 0; it < WAIT_LIMIT && !mbar_test(&full_b[s2], (uint32_t)((qq / S) & 1)); ++it) {
        }
      }
      for (int b = max(0, fetched - 2); b < fetched; ++b)
        for (long it = 0; it < WAIT_LIMIT && !mbar_test(&rec_b[b & 1], (uint32_t)((b >> 1) & 1)); ++it) {
        }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer (one thread): one accumulator per segment
    if (lane == 0) {
      int st = 0;            // stage of the next K step
      uint32_t par = 0;      // its round's parity
      int sg = 0;  // segments issued
      bool ok = true;
      auto mma = [&](uint32_t d, uint64_t ad, uint64_t bd, uint32_t idk, uint32_t accum) {
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
            "l"(ad), "l"(bd), "r"(idk), "r"(accum));
      };
      auto commit = [&](uint64_t* bar) {
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(smem_u32(bar)));
      };
      // shared-memory descriptors of stage 0's operands; later stages, slots, slices and K
      // steps add their byte offsets / 16 to the 14-bit address field (no carry: shared
      // addresses stay below 256 KB)
      const uint64_t ad0 = sdesc(base), bd0 = sdesc(base + TM_A_BYTES);
      const uint32_t al0 = base >> 4, bl0 = (base + Cfg::SLOTS * Cfg::A_BYTES) >> 4;
      if constexpr (CHAIN) {
        // A term's products in the order of the slice pairs (i, j), by level i + j, each over all
        // 16-column pieces of the term: the order in which they are rounded into the
        // accumulator.  The pieces' slots are released during the last pair.
        // One thread issues them all and needs several clocks per instruction, so what it executes
        // per product bounds the kernel once its loops, branches and commits outnumber the products.
        // Terms (up to TM_TERM_PIECES pieces) that end inside the open segment are straight-line
        // code with one commit for all their slots (term barriers, in order), short ones that cross
        // its end too, with a check per product; the others go product by product in a loop.
        // Measured at K=24, M=512 (stage 2): all in loops 1.20-1.50 ms, whatever was moved out of
        // them, straight-line 0.80 ms.
        constexpr int SEG = STORE ? 0x7fffffff : TM_SEG_PRODUCTS;
        constexpr int NPAIR = NSL == 2 ? 3 : 6;
        constexpr uint32_t PAIR_I = 0x210100u, PAIR_J = 0x012010u;  // slices of pair q in the nibble q
        const uint32_t step = (uint32_t)(STAGE_BYTES >> 4);
        int cnt = 0;        // products in the open segment
        uint32_t dacc = 0;  // its accumulator
        int tm = 0;         // terms released
        auto open = [&]() -> bool {
          const int acc = sg % NACC;
          if (sg >= NACC && !mbar_wait(&tempty_b[acc], (uint32_t)(((sg / NACC) - 1) & 1), abort_flag)) return false;
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
          dacc = tmem + (uint32_t)(acc * NMAX);
          return true;
        };
        auto close = [&]() {
          commit(&tfull_b[sg % NACC]);
          ++sg;
          cnt = 0;
        };
        for (int ti = blockIdx.x; ti < ntiles && ok; ti += gridDim.x) {
          for (bool tile_done = false; !tile_done && ok;) {
            ok = mbar_wait(&full_b[st], par, abort_flag);
            if (!ok) break;
            const uint64_t mw = meta[st];
            const uint32_t fl = (uint32_t)(mw >> 32), id = (uint32_t)mw | ((fl >> 9 & 1u) << 13);
            const uint32_t n = ((uint32_t)mw >> 17 & 63u) << 3;  // rows of B: 8 columns of a slice are n * 16 bytes
            tile_done = (fl & 1024u) != 0;
            const int kp = (int)(fl & 255u);
            const uint32_t a0 = al0 | (uint32_t)(128 * NSL) << 16, b0 = bl0 | (n * NSL) << 16;
            // the term's pieces: their slot offsets and their arrival
            uint32_t off[TM_TERM_PIECES];
            {
              int s2 = st;
              uint32_t p2 = par;
#pragma unroll 1
              for (int c = 0; c < kp; ++c) {
                if (c > 0 && !(ok = mbar_wait(&full_b[s2], p2, abort_flag))) break;
                if (++s2 == S) {
                  s2 = 0;
                  p2 ^= 1u;
                }
              }
              if (!ok) break;
#pragma unroll
              for (int c = 0; c < TM_TERM_PIECES; ++c) off[c] = (uint32_t)(st + c < S ? st + c : st + c - S) * step;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
            if (cnt == 0 && !(ok = open())) break;
            const int after = cnt + kp * NPAIR;
            auto term = [&](auto len, auto check) {
              constexpr int K = decltype(len)::value;
              uint32_t accum = cnt > 0;
#pragma unroll
              for (int l = 0; l < NSL; ++l)
#pragma unroll
                for (int i = 0; i <= l; ++i)
#pragma unroll
                  for (int c = 0; c < K; ++c) {
                    mma(dacc, sdesc_groups(a0 + off[c] + (uint32_t)(i * 128)),
                        sdesc_groups(b0 + off[c] + (uint32_t)(l - i) * n), id, accum);
                    accum = 1u;
                    if constexpr (decltype(check)::value) {
                      const bool last = l == NSL - 1 && i == l && c == K - 1;
                      if (++cnt == SEG && !last) {
                        close();
                        ok = ok && open();
                        accum = 0u;
                      }
                    }
                  }
            };
            using std::integral_constant;
            if (after <= SEG) {
              const integral_constant<bool, false> no{};
              switch (kp) {
                case 1: term(integral_constant<int, 1>{}, no); break;
                case 2: term(integral_constant<int, 2>{}, no); break;
                case 3: term(integral_constant<int, 3>{}, no); break;
                case 4: term(integral_constant<int, 4>{}, no); break;
                case 5: term(integral_constant<int, 5>{}, no); break;
                default: term(integral_constant<int, TM_TERM_PIECES>{}, no); break;
              }
              cnt = after;
              if (cnt == SEG || tile_done) close();
            } else if (kp <= 3) {
              const integral_constant<bool, true> yes{};
              switch (kp) {
                case 1: term(integral_constant<int, 1>{}, yes); break;
                case 2: term(integral_constant<int, 2>{}, yes); break;
                default: term(integral_constant<int, 3>{}, yes); break;
              }
              if (!ok) break;
              if (cnt == SEG || tile_done) close();
            } else {
#pragma unroll 1
              for (int q = 0; q < NPAIR && ok; ++q) {
                uint32_t a = a0 + off[0] + (PAIR_I >> (4 * q) & 15u) * 128u, b = b0 + off[0] + (PAIR_J >> (4 * q) & 15u) * n;
                int s2 = st;
#pragma unroll 1
                for (int c = 0; c < kp; ++c) {
                  if (cnt == 0 && !(ok = open())) break;
                  mma(dacc, sdesc_groups(a), sdesc_groups(b), id, cnt > 0);
                  if (++cnt == SEG || (tile_done && q == NPAIR - 1 && c == kp - 1)) close();
                  a += step;
                  b += step;
                  if (++s2 == S) {
                    s2 = 0;
                    a -= (uint32_t)S * step;
                    b -= (uint32_t)S * step;
                  }
                }
              }
              if (!ok) break;
            }
            commit(&term_b[tm & (TM_TERMS - 1)]);
            ++tm;
            st += kp;
            if (st >= S) {
              st -= S;
              par ^= 1u;
            }
          }
        }
      } else {
        for (int ti = blockIdx.x; ti < ntiles && ok; ti += gridDim.x) {
          bool tile_done = false;
          while (!tile_done && ok) {
            const int acc = sg % NACC;
            if (sg >= NACC && !mbar_wait(&tempty_b[acc], (uint32_t)(((sg / NACC) - 1) & 1), abort_flag)) {
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
            const uint32_t dacc = tmem + (uint32_t)(acc * NMAX);
            for (;;) {
              if (!mbar_wait(&full_b[st], par, abort_flag)) {
                ok = false;
                break;
              }
              asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
              const uint64_t mw = meta[st];
              const uint32_t id = (uint32_t)mw, fl = (uint32_t)(mw >> 32);
              const int nk = (int)(fl & 7u);
              const uint32_t off = (uint32_t)((st * STAGE_BYTES) >> 4);
              uint32_t accum = (fl & 8u) ? 0u : 1u;
              const uint32_t n = (id >> 17 & 63u) << 3;
              for (int kk = 0; kk < nk; ++kk) {
                if constexpr (EXACT)
                  mma(dacc, ad0 + off + (uint64_t)(kk * 2), bd0 + off + (uint64_t)(kk * 2), id, accum);
                else
                  mma(dacc, sdesc_groups((al0 + off + (uint32_t)((kk * Cfg::A_BYTES) >> 4)) | 128u << 16),
                      sdesc_groups((bl0 + off + (uint32_t)((kk * Cfg::B_BYTES) >> 4)) | n << 16),
                      id | (((fl >> (8 + kk)) & 1u) << 13), accum);
                accum = 1u;
              }
              commit(&empty_b[st]);
              if (++st == S) {
                st = 0;
                par ^= 1u;
              }
              if (fl & 16u) {
                tile_done = (fl & 32u) != 0;
                break;
              }
            }
            if (!ok) break;
            commit(&tfull_b[acc]);
            ++sg;
          }
        }
      }
    }
  } else {
    // ---------------- epilogue (warps 2-5: tensor-memory lanes 32 * (warp % 4) ...)
    const int sub = warp & 3;
    const int r = sub * 32 + lane;  // row of the tile
    int sg = 0;
    bool ok = true;
    // the next tile's descriptor is loaded one tile ahead; in store mode the row map of a
    // tile is read before its accumulator is waited for
    TmTile tl_next{};
    if ((int)blockIdx.x < ntiles) tl_next = tiles[blockIdx.x];
    for (int ti = blockIdx.x; ti < ntiles && ok; ti += gridDim.x) {
      const TmTile tl = tl_next;
      if (ti + (int)gridDim.x < ntiles) tl_next = tiles[ti + gridDim.x];
      if constexpr (STORE) {
        const int acc = sg % NACC;
        const long row_own = rowmap[tl.rowmap_off + r];
        ok = mbar_wait(&tfull_b[acc], (uint32_t)((sg / NACC) & 1), abort_flag);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
        // per 8 columns one 16-byte store per slice, x = s0 + s1 + s2 from one read of each
        // value; the lanes' rows are mostly consecutive, so a warp writes contiguous runs.
        // The tensor-memory loads (32 columns, one wait) are warp-wide.
        __nv_bfloat16* g = reinterpret_cast<__nv_bfloat16*>(out) + tl.xbase + tl.out_off * NSL * tl.xrows + row_own * 8;
#pragma unroll 1
        for (int c0 = 0; c0 < tl.n; c0 += 32) {
          uint32_t v[32];
          tmem_ld32(tmem + ((uint32_t)(sub * 32) << 16) + (uint32_t)(acc * NMAX + c0), v);
#pragma unroll
          for (int u8 = 0; u8 < 32; u8 += 8) {
            if (c0 + u8 >= tl.n || row_own < 0) continue;
            uint32_t w[NSL][4];
#pragma unroll
            for (int u = 0; u < 8; u += 2) {
              float a = __uint_as_float(v[u8 + u]), b = __uint_as_float(v[u8 + u + 1]);
#pragma unroll
              for (int sl = 0; sl < NSL; ++sl) {
                const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
                w[sl][u / 2] = *reinterpret_cast<const uint32_t*>(&h);
                a -= __low2float(h);
                b -= __high2float(h);
              }
            }
            __nv_bfloat16* q = g + (long)(c0 + u8) * NSL * tl.xrows;
#pragma unroll
            for (int sl = 0; sl < NSL; ++sl)
              *reinterpret_cast<uint4*>(q + sl * tl.xrows * 8) = make_uint4(w[sl][0], w[sl][1], w[sl][2], w[sl][3]);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
        mbar_arrive(&tempty_b[acc]);
        ++sg;
      } else if constexpr (EXACT) {
        // per segment: its exact integer sums, times 2^(expo[ea] + expo[eb] - 7 (l + 2)),
        // added into two-float sums hi + lo (error-free additions)
        float hi[NMAX], lo[NMAX];
#pragma unroll
        for (int c = 0; c < NMAX; ++c) hi[c] = lo[c] = 0.0f;
        for (int sgi = 0, t = tl.t0; t < tl.t1 && ok; ++sgi) {
          const int flags = terms[t].neg;
          const int nsl = max(1, (flags >> 4) & 15);
          const int lvl = sgi;  // segment sgi of term t: level sgi
          const int e = expo[terms[t].ea] + expo[terms[t].eb] - TM_EXACT_BITS * (lvl + 2);
          if (sgi + 1 == nsl) {
            sgi = -1;
            ++t;
          }
          const int acc = sg % NACC;
          ok = mbar_wait(&tfull_b[acc], (uint32_t)((sg / NACC) & 1), abort_flag);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
#pragma unroll
          for (int cc = 0; cc < NMAX / 32; ++cc) {
            uint32_t v[32];
            tmem_ld32(tmem + ((uint32_t)(sub * 32) << 16) + (uint32_t)(acc * NMAX + cc * 32), v);
#pragma unroll
            for (int u = 0; u < 32; ++u) {
              float x = ldexpf(__uint_as_float(v[u]), e);
              if (flags & 1) x = -x;
              const float a = hi[cc * 32 + u];
              const float sum = __fadd_rn(a, x);
              const float bp = __fsub_rn(sum, a);
              const float err = __fadd_rn(__fsub_rn(a, __fsub_rn(sum, bp)), __fsub_rn(x, bp));
              hi[cc * 32 + u] = sum;
              lo[cc * 32 + u] = __fadd_rn(lo[cc * 32 + u], err);
            }
          }
          asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
          mbar_arrive(&tempty_b[acc]);
          ++sg;
        }
        if (!ok) break;
        if (r < tl.m_valid) {
          double* p = reinterpret_cast<double*>(out) + tl.out_off + (long)r * tl.ldo;
#pragma unroll
          for (int c = 0; c < NMAX; ++c)
            if (c < tl.nvalid) p[c] = (double)hi[c] + (double)lo[c];
        }
      } else {
        float run[NMAX / 16][16];  // the tile's running FP32 sum (row r)
        for (int q = 0; q < tl.nseg; ++q, ++sg) {
          const int acc = sg % NACC;
          ok = mbar_wait(&tfull_b[acc], (uint32_t)((sg / NACC) & 1), abort_flag);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
#pragma unroll
          for (int cc = 0; cc < NMAX / 16; ++cc) {
            const int c0 = cc * 16;
            if (c0 < tl.n) {
              uint32_t v[16];
              tmem_ld16(tmem + ((uint32_t)(sub * 32) << 16) + (uint32_t)(acc * NMAX + c0), v);
              if (q == 0) {
#pragma unroll
                for (int u = 0; u < 16; ++u) run[cc][u] = __uint_as_float(v[u]);
              } else {
#pragma unroll
                for (int u = 0; u < 16; ++u) run[cc][u] += __uint_as_float(v[u]);
              }
            }
          }
          asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
          mbar_arrive(&tempty_b[acc]);
        }
        if (!ok) break;
        if (r < tl.m_valid) {
          float* p = reinterpret_cast<float*>(out) + tl.out_off + (long)r * tl.ldo;
#pragma unroll
          for (int cc = 0; cc < NMAX / 16; ++cc)
            if (cc * 16 < tl.n) {
#pragma unroll
              for (int u = 0; u < 16; u += 4)
                red_add_v4(p + cc * 16 + u, __float_as_uint(run[cc][u]), __float_as_uint(run[cc][u + 1]),
                           __float_as_uint(run[cc][u + 2]), __float_as_uint(run[cc][u + 3]));
            }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::);
  __syncthreads();
  if (tid == 0 && abort_sh) atomicExch(err, 1);
  if (warp == 2) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::);
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(Cfg::TMEM));
  }
}

template <int MODE, int NSL>
cudaError_t launch_mode(const TmTile* d_tiles, int ntiles, const TmTerm* d_terms, const CUtensorMap* d_maps,
                        const long* d_rowmap, void* out, int* d_err, cudaStream_t s, const int* d_expo,
                        const TmListsDev& lists) {
  using Cfg = TmCfg<MODE, NSL>;
  static DeviceOnce once;
  if (!allow_shared_memory(once, gemm_tma_kernel<MODE, NSL>, Cfg::SMEM)) return cudaErrorInvalidValue;
  // the lists were built for this grid (every CTA's tiles and stages) and ring
  if (lists.grid != tma_grid(Cfg::CTAS, ntiles) || !lists.cta_stage || !lists.stages || !lists.pieces)
    return cudaErrorInvalidValue;
  if (Cfg::CHAIN && (lists.slots < 1 || lists.slots > TM_MAX_SLOTS || lists.slot_bytes % 1024 != 0 ||
                     lists.slots * lists.slot_bytes > TM_RING_BYTES))
    return cudaErrorInvalidValue;
  count_tc_launches(1);
  gemm_tma_kernel<MODE, NSL><<<lists.grid, TM_THREADS, Cfg::SMEM, s>>>(
      d_tiles, ntiles, d_terms, d_maps, d_rowmap, out, d_err, d_expo, lists.cta_stage, lists.stages, lists.pieces,
      lists.slots, lists.slot_bytes);
  return cudaGetLastError();
}

// exact splitting: one block of threads per job, warps over rows, lanes over columns.
// The block maximum is taken on the bit patterns (|x| orders like its bits as an
// unsigned integer), so the FP64 units see one multiply per element for the scaling by
// scale * 2^-e (exact: a power of two times the rounding of scale * x) and the split
// v = a + lo into two FP32 values; the 7-bit slices come from a by exact FP32 steps
// (w *= 2^7, q = rint(w), w -= q), and lo joins the remainder after the third slice
// (one FP32 rounding, below 2^-46 of the block's scale).  Slice magnitudes: the first
// <= 128, the fourth <= 72, the others <= 64.
__global__ void split_exact_kernel(const SplitJob* __restrict__ jobs, int nsl, int* __restrict__ expo_out) {
  const SplitJob jb = jobs[blockIdx.x];
  __shared__ unsigned long long red[32];
  __shared__ int e_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  unsigned long long m = 0;
  for (int r = warp; r < jb.rows; r += nw) {
    const double* src = jb.src + (long)r * jb.lds;
    for (int c = lane; c < jb.cols; c += 32) {
      const unsigned long long bits = (unsigned long long)__double_as_longlong(src[c]) & 0x7fffffffffffffffULL;
      m = bits > m ? bits : m;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long t = __shfl_xor_sync(0xffffffffu, m, o);
    m = t > m ? t : m;
  }
  if (lane == 0) red[warp] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long mm = 0;
    for (int w = 0; w < nw; ++w) mm = red[w] > mm ? red[w] : mm;
    // fl(|scale| * max|x|) bounds every fl(|scale * x|) (rounding is monotone)
    const double mx = fabs(jb.scale) * __longlong_as_double((long long)mm);
    int e = 0;
    if (mx > 0.0) frexp(mx, &e);  // mx = f 2^e with 0.5 <= f < 1: |scale * x| < 2^e
    e_sh = e;
    expo_out[jb.expo] = e;
  }
  __syncthreads();
  const double f = ldexp(jb.scale, -e_sh);
  constexpr float STEP = (float)(1 << TM_EXACT_BITS);
  constexpr float LO_SCALE = (float)(1 << (3 * TM_EXACT_BITS));  // lo at the scale of the remainder after three slices
  for (int r = warp; r < jb.rows; r += nw) {
    const double* src = jb.src + (long)r * jb.lds;
    for (int c = lane; c < jb.wcols; c += 32) {
      const double v = c < jb.cols ? f * src[c] : 0.0;  // |v| < 1
      float w = __double2float_rn(v);
      const float lo = __double2float_rn(v - (double)w);
      __nv_bfloat16* d = jb.trans ? jb.dst + (long)c * jb.ldd + r : jb.dst + (long)r * jb.ldd + c;
      for (int s = 0; s < nsl; ++s) {
        if (s == 3) w += lo * LO_SCALE;
        w *= STEP;
        const float q = rintf(w);  // an integer of at most 128 in magnitude: exact in BF16
        d[(long)s * jb.slice_stride] = __float2bfloat16_rn(q);
        w -= q;
      }
    }
  }
}

using EncodeTiledFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encoder() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return (EncodeTiledFn) nullptr;
    return reinterpret_cast<EncodeTiledFn>(p);
  }();
  return fn;
}

}  // namespace

cudaError_t launch_split_exact(const SplitJob* d_jobs, int njobs, int nsl, int* d_expo, cudaStream_t s) {
  if (njobs <= 0) return cudaSuccess;
  if (nsl < 1 || nsl > 6) return cudaErrorInvalidValue;  // the remainder and level-sum bounds hold up to six slices
  count_tc_launches(1);
  split_exact_kernel<<<njobs, 256, 0, s>>>(d_jobs, nsl, d_expo);
  return cudaGetLastError();
}

cudaError_t launch_gemm_slices(int mode, int nsl, const TmTile* d_tiles, int ntiles, const CUtensorMap* d_maps,
                               const long* d_rowmap, void* out, int* d_err, cudaStream_t s, const TmListsDev& lists) {
  if (ntiles <= 0) return cudaSuccess;
  auto go = [&](auto fn) { return fn(d_tiles, ntiles, nullptr, d_maps, d_rowmap, out, d_err, s, nullptr, lists); };
  if (mode == TM_MODE_STORE_BF16) {
    if (nsl == 1) return go(launch_mode<TM_MODE_STORE_BF16, 1>);
    if (nsl == 2) return go(launch_mode<TM_MODE_STORE_BF16, 2>);
    if (nsl == 3) return go(launch_mode<TM_MODE_STORE_BF16, 3>);
  }
  if (mode == TM_MODE_REDUCE_F32) {
    if (nsl == 1) return go(launch_mode<TM_MODE_REDUCE_F32, 1>);
    if (nsl == 2) return go(launch_mode<TM_MODE_REDUCE_F32, 2>);
    if (nsl == 3) return go(launch_mode<TM_MODE_REDUCE_F32, 3>);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_gemm_exact(const TmTile* d_tiles, int ntiles, const TmTerm* d_terms, const CUtensorMap* d_maps,
                              double* out, int* d_err, cudaStream_t s, const TmListsDev& lists, const int* d_expo) {
  if (ntiles <= 0) return cudaSuccess;
  if (!d_expo || !d_terms) return cudaErrorInvalidValue;
  return launch_mode<TM_MODE_EXACT_F64, 1>(d_tiles, ntiles, d_terms, d_maps, nullptr, out, d_err, s, d_expo, lists);
}

int tma_grid(int ctas, int ntiles) {
  static const int nsm = [] {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) !=
                                                   cudaSuccess)
      return 148;
    return n > 0 ? n : 148;
  }();
  return ntiles < ctas * nsm ? ntiles : ctas * nsm;
}

int tma_pieces(int mode, int nsl) { return mode == TM_MODE_EXACT_F64 ? 1 : tm_slots(nsl); }

namespace {
__host__ __device__ inline int slice_pairs(int nsl) { return nsl * (nsl + 1) / 2; }

// pieces of a term: 16 columns each, or (exact mode) 64 columns of every slice pair
__host__ __device__ inline long term_pieces(const TmTerm& m, bool exact) {
  if (!exact) return m.k / TM_PIECE_COLS;
  const int nsl = ((m.neg >> 4) & 15) > 1 ? ((m.neg >> 4) & 15) : 1;
  return (long)((m.k + TM_BOX_K - 1) / TM_BOX_K) * slice_pairs(nsl);
}

// slice pair number q in level order: its level and first index
__device__ __forceinline__ void slice_pair(int q, int& l, int& i) {
  l = 0;
  while (q > l) {
    q -= l + 1;
    ++l;
  }
  i = q;
}

// One thread per stage.  It finds its tile (stages in the launch order: sorder[i] has
// the stages from sfirst[i]) and the term of its first piece (tpiece0: a term's first
// piece within its tile), then walks the stage's pieces.  Exact mode: a term's pieces are its
// slice pairs (i, j), i + j < nsl, in level order, each its boxes along K.  Segments: store
// mode one per tile; reduce mode TM_SEG_PRODUCTS products each (they accumulate in
// tensor memory over a segment only and the epilogue adds the segments in FP32 with
// round-to-nearest, so the rounding toward zero of the tensor-core accumulation acts on
// short sums); exact mode one per level of every term.
__global__ void fill_lists_kernel(int mode, int nslices, const TmTile* __restrict__ tiles, int ntiles,
                                  const TmTerm* __restrict__ terms, const int* __restrict__ tpiece0,
                                  const int* __restrict__ sorder, const long* __restrict__ sfirst, long total,
                                  TmStage* __restrict__ stages, TmPiece* __restrict__ pieces) {
  const long g = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= total) return;
  const bool exact = mode == TM_MODE_EXACT_F64;
  const int bc = exact ? TM_BOX_K : TM_PIECE_COLS, P = exact ? 1 : tm_slots(nslices);
  int lo = 0, hi = ntiles - 1;  // the last tile (in stage order) starting at or before g
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (sfirst[mid] <= g) lo = mid; else hi = mid - 1;
  }
  const TmTile tl = tiles[sorder[lo]];
  const long sl = g - sfirst[lo];
  const long nst = (lo + 1 < ntiles ? sfirst[lo + 1] : total) - sfirst[lo];
  const long p0 = sl * P;
  int t = tl.t0, th = tl.t1 - 1;  // the last term whose first piece is at or before p0
  while (t < th) {
    const int mid = (t + th + 1) >> 1;
    if (tpiece0[mid] <= p0) t = mid; else th = mid - 1;
  }
  const long tile_pieces = tpiece0[tl.t1 - 1] + term_pieces(terms[tl.t1 - 1], exact);
  const int np = (int)min((long)P, tile_pieces - p0);
  const uint32_t piece_bytes = (uint32_t)(128 + tl.n) * bc * 2 * (exact ? 1 : nslices);
  const bool last = sl == nst - 1;
  TmTerm m = terms[t];
  long r = p0 - tpiece0[t];
  uint32_t negm = 0, fl = 0, id = 0;
  for (int slot = 0; slot < np; ++slot, ++r) {
    if (r >= term_pieces(m, exact)) {
      m = terms[++t];
      r = 0;
    }
    if (!exact) {
      const int k0 = (int)r * bc;
      pieces[g * P + slot] = TmPiece{m.amap, (m.ax + k0) / 8, m.ay / 16, m.bmap, (m.bx + k0) / 8, m.by / 16, {0, 0}};
      negm |= (uint32_t)(m.neg & 1) << slot;
      if (nslices > 1) fl = (uint32_t)(m.k / bc) | (negm & 1u) << 9 | (t == tl.t1 - 1 ? 1024u : 0u);
      continue;
    }
    const int nsl = max(1, (m.neg >> 4) & 15);
    const int kp = (m.k + bc - 1) / bc;
    const int q = (int)(r / kp), kk = (int)(r - (long)q * kp), k0 = kk * bc;
    int l, i;
    slice_pair(q, l, i);
    pieces[g * P + slot] = TmPiece{m.amap + i, m.ax + k0, m.ay, m.bmap + (l - i), m.bx + k0, m.by, {0, 0}};
    fl = (uint32_t)min(bc / 16, (m.k - k0) / 16);
    fl |= (i == 0 && kk == 0) ? 8u : 0u;
    fl |= (i == l && kk == kp - 1) ? 16u : 0u;
    id = tm_idesc_bf16(tl.n, (m.neg & 1) != 0);
  }
  for (int p = np; p < P; ++p) pieces[g * P + p] = TmPiece{0, 0, 0, 0, 0, 0, {0, 0}};
  if (!exact) id = tm_idesc_bf16(tl.n, false);
  if (!exact && nslices == 1) {
    const long seg = mode == TM_MODE_REDUCE_F32 ? TM_SEG_PRODUCTS / tm_slots(1) : nst;
    fl = (uint32_t)np | (negm << 8);
    fl |= sl % seg == 0 ? 8u : 0u;
    fl |= (last || sl % seg == seg - 1) ? 16u : 0u;
  }
  if (exact || nslices == 1) fl |= last ? 32u : 0u;
  stages[g] = TmStage{(uint64_t)id | ((uint64_t)fl << 32), (uint32_t)np * piece_bytes, np};
}
}  // namespace

// Order of the tiles for a launch whose CTA c takes the tiles c, c + grid, ...: round by round
// the longest tile goes to the CTA with the least work so far (in the order given, the
// first CTA would take the longest of every round).  Only the last rounds are dealt this way:
// they level what the earlier ones left.  Sigma, dealt in the order given and this way: K=24, M=512,
// three slices 1.54 and 1.48 ms; K=32, M=1024, one pass 1.62 and 1.56; K=40, M=1200 12.6 both.
static void level_rounds(std::vector<TmTile>& tiles, const std::vector<TmTerm>& terms, int grid) {
  constexpr size_t LAST = 24;
  const size_t G = (size_t)grid, n = tiles.size();
  if (n <= G) return;
  // cost of a tile: bytes of its operand pieces (they bound the launches), and a piece's worth for its
  // epilogue
  std::vector<long> cost(n);
  for (size_t i = 0; i < n; ++i) {
    long k = 64;
    for (int t = tiles[i].t0; t < tiles[i].t1; ++t) k += terms[(size_t)t].k;
    cost[i] = k * (128 + tiles[i].n);
  }
  const size_t rounds = (n + G - 1) / G, first = rounds > LAST ? rounds - LAST : 0;
  std::vector<long> load(G, 0);
  for (size_t i = 0; i < first * G; ++i) load[i % G] += cost[i];
  // at[c]: the tiles of CTA c in the rounds from `first` on
  std::vector<std::vector<size_t>> at(G);
  std::vector<size_t> cta(G), tile;
  for (size_t c = 0; c < G; ++c) cta[c] = c;
  for (size_t r = first; r < rounds; ++r) {
    const size_t b = r * G, m = std::min(G, n - b);
    tile.resize(m);
    for (size_t i = 0; i < m; ++i) tile[i] = b + i;
    std::stable_sort(tile.begin(), tile.end(), [&](size_t x, size_t y) { return cost[x] > cost[y]; });
    std::stable_sort(cta.begin(), cta.end(), [&](size_t x, size_t y) { return load[x] < load[y]; });
    for (size_t i = 0; i < m; ++i) {
      at[cta[i]].push_back(tile[i]);
      load[cta[i]] += cost[tile[i]];
    }
  }
  // the CTAs that got a tile of the last, partial round have to be the first ones; the earlier
  // rounds move with their CTA
  std::stable_sort(cta.begin(), cta.end(), [&](size_t x, size_t y) { return x < y; });
  std::stable_partition(cta.begin(), cta.end(), [&](size_t c) { return at[c].size() == rounds - first; });
  std::vector<TmTile> out(n);
  for (size_t c = 0; c < G; ++c) {
    for (size_t r = 0; r < first; ++r) out[r * G + c] = tiles[r * G + cta[c]];
    for (size_t r = 0; r < at[cta[c]].size(); ++r) out[(first + r) * G + c] = tiles[at[cta[c]][r]];
  }
  tiles.swap(out);
}

bool tma_plan_lists(int mode, int nsl, std::vector<TmTile>& tiles, const std::vector<TmTerm>& terms, TmListPlan& out) {
  const int ntiles = (int)tiles.size();
  const bool exact = mode == TM_MODE_EXACT_F64, chain = !exact && nsl > 1;
  const int P = tma_pieces(mode, nsl);
  int max_n = 16, max_k = 16;
  for (const TmTile& tl : tiles) max_n = std::max(max_n, tl.n);
  for (const TmTerm& m : terms) {
    if (m.k < 16 || m.k % 16) return false;
    max_k = std::max(max_k, m.k);
  }
  // ring of a launch with two or three slices: slots of one piece of all slices, enough for the
  // longest term
  out.slots = 0;
  out.slot_bytes = 0;
  if (chain) {
    out.slot_bytes = tm_slot_bytes(nsl, max_n);
    out.slots = tm_fit_slots(nsl, max_n);
    if (max_k / TM_PIECE_COLS > tm_term_pieces(nsl, max_n)) return false;
  }
  const int grid = ntiles > 0 ? tma_grid(tm_ctas(mode), ntiles) : 0;
  for (const TmTile& tl : tiles)
    if (tl.t0 < 0 || tl.t1 <= tl.t0 || tl.t1 > (int)terms.size()) return false;
  if (grid > 0) level_rounds(tiles, terms, grid);
  // every term belongs to one tile; its first piece within the tile
  out.tpiece0.assign(terms.size(), -1);
  std::vector<long> tst((size_t)ntiles), tprod((size_t)ntiles);
  for (int ti = 0; ti < ntiles; ++ti) {
    const TmTile& tl = tiles[(size_t)ti];
    long pc = 0, pr = 0;
    for (int t = tl.t0; t < tl.t1; ++t) {
      if (out.tpiece0[(size_t)t] >= 0 || pc >= (1L << 31)) return false;
      out.tpiece0[(size_t)t] = (int)pc;
      pc += term_pieces(terms[(size_t)t], exact);
      pr += (long)terms[(size_t)t].k / TM_PIECE_COLS * slice_pairs(nsl);
    }
    tst[(size_t)ti] = (pc + P - 1) / P;
    tprod[(size_t)ti] = pr;
  }
  // stages in launch order: CTA c takes the tiles c, c + grid, ...
  out.grid = grid;
  out.cta_stage.assign((size_t)grid + 1, 0);
  out.sorder.clear();
  out.sfirst.clear();
  long total = 0;
  for (int c = 0; c < grid; ++c) {
    out.cta_stage[(size_t)c] = (int)total;
    for (int ti = c; ti < ntiles; ti += grid) {
      out.sorder.push_back(ti);
      out.sfirst.push_back(total);
      total += tst[(size_t)ti];
    }
    if (total >= (1L << 31) / P) return false;
  }
  out.cta_stage[(size_t)grid] = (int)total;
  out.total = total;
  if (mode == TM_MODE_REDUCE_F32)
    for (int ti = 0; ti < ntiles; ++ti) {
      tiles[(size_t)ti].pad = (int)tst[(size_t)ti];
      tiles[(size_t)ti].nseg = (int)((tprod[(size_t)ti] + TM_SEG_PRODUCTS - 1) / TM_SEG_PRODUCTS);
    }
  return true;
}

cudaError_t launch_fill_lists(int mode, int nsl, const TmTile* d_tiles, int ntiles, const TmTerm* d_terms,
                              const int* d_tpiece0, const int* d_sorder, const long* d_sfirst, long total,
                              TmStage* d_stages, TmPiece* d_pieces, cudaStream_t s) {
  if (ntiles <= 0 || total <= 0) return cudaSuccess;
  count_tc_launches(1);
  fill_lists_kernel<<<(unsigned)((total + 255) / 256), 256, 0, s>>>(mode, nsl, d_tiles, ntiles, d_terms, d_tpiece0,
                                                                    d_sorder, d_sfirst, total, d_stages, d_pieces);
  return cudaGetLastError();
}

bool encode_bf16_map(CUtensorMap* out, const void* base, uint64_t rows, uint64_t cols, uint64_t ld,
                     uint32_t box_rows) {
  EncodeTiledFn fn = encoder();
  if (!fn || rows == 0 || cols == 0 || (ld * 2) % 16 != 0 || ((uintptr_t)base & 15) != 0 || box_rows == 0 ||
      box_rows > 256)
    return false;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {ld * 2};
  const cuuint32_t box[2] = {(cuuint32_t)TM_BOX_K, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool encode_slice_map(CUtensorMap* out, const void* base, uint64_t rows, uint64_t cols, int nsl, uint32_t box_rows) {
  EncodeTiledFn fn = encoder();
  if (!fn || rows == 0 || rows % 16 != 0 || cols == 0 || cols % 8 != 0 || nsl < 1 || nsl > 3 ||
      ((uintptr_t)base & 15) != 0 || box_rows == 0 || box_rows % 16 != 0 || box_rows > 256)
    return false;
  const cuuint64_t dims[4] = {128, rows / 16, (cuuint64_t)nsl, cols / 8};
  const cuuint64_t strides[3] = {256, rows * 16, rows * 16 * nsl};
  const cuuint32_t box[4] = {128, box_rows / 16, (cuuint32_t)nsl, TM_PIECE_COLS / 8};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(out, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace gbdmrg
