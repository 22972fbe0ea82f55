// Row softmax behind a SHORT-K GEMM:  P = softmax(alpha * A.B + mask)  over the last dimension, for K so small that
// computing a score tile twice is cheaper than moving it (the attention-score pattern of Sec. 6.1: K = head size).
//
// Stage-Stream view (Sec. 3): the row reduction (max, sum of exponentials) is the stage boundary.  The general kernel
// keeps a whole row block on-chip by spreading its columns over a cluster and aggregating the partial statistics
// through distributed shared memory (Sec. 3.2).  With K <= 256 the producer stage is so cheap that this kernel takes
// the other side of the same trade: one CTA pair owns 256 complete rows, streams the row through tensor memory in
// 256-column chunks TWICE (MainLoop re-run instead of on-chip residency), and needs no cross-CTA exchange at all:
//
//   pass 0   for every live chunk:  S = A.B_chunk (UMMA, cta_group::2)  ->  online (max, sum) per thread; the exponentials of the
//            last chunk stay in registers, those of the chunk before it in the chunk's accumulator slot (fp32 both)
//   merge    the four threads that share a row combine their partials through shared memory
//   result   the two kept chunks: exponential * 2^((m_thread - max)*log2e - log2 sum)  ->  bf16 box -> TMA store
//   pass 1   for every other live chunk:  S again  ->  P = 2^((t - max)*log2e - log2 sum), t = alpha*S + mask  ->  bf16 box -> TMA store
//
// Clusters are pairs, so all SMs are used (wider clusters leave SMs idle), any N fits, and the accumulator slots
// alternate so that the UMMAs of chunk u+1 run under the epilogue of chunk u.  Rows of up to 512 columns are computed and
// exponentiated once.  Under a causal mask, chunks above the diagonal are neither computed nor staged: a warp of its own
// writes them with TMA stores of a constant zero box, with a cursor of its own through the cluster's tiles.
//
// What bounds it: the exponentials (MUFU: 16 results per clock and SM; a pass over 64 x 32 scores of all sixteen warps takes
// 1640 clocks in a loop of its own) and, where the output outgrows the L2, the writes.  64 x 2048 x 2048 causal, K = 64 (537 MB
// written, 85 us at the best rate of any store pattern measured here): 122.5 -> 115.2 us, without its stores 99 -> 75.  A thread
// holds all its 64 columns of a chunk, so the accumulator is handed back before the arithmetic, which needs the registers that
// the control warps give up (setmaxnreg: 112 instead of 96).  96 x 504 x 504 with a mask 34.3 -> 28.3 us a call; thirty shapes drawn from
// 16 .. 2048 rows and 64 .. 2048 columns 0.995 .. 1.49 times as fast (geometric mean 1.16).  A kernel without a soft-cap carries no code for one:
// a CTA runs through a few tiles only, and the first one waits for every line of code it is the first to reach (96 x 504 x 504 29.1 / 28.2).
//
// Warp roles: warp 0 TMA producer, warp 1 TMEM allocation + UMMA issue (even CTA), warp 2 zero boxes, warp 3 idle (register
// shares are given to groups of four warps); then 16 epilogue warps (thread = row; warp e takes lane quarter e % 4 and
// 64-column group e / 4 of each chunk), which stage their boxes and issue the stores themselves.  Every wait is bounded.
#pragma once

#include <type_traits>

#include "epilogue_common.cuh"
#include "fused_params.h"
#include "sm100_primitives.cuh"

namespace comfuse {

// Maxima that are NaN if an argument is: a row with a NaN score (or one of +inf) comes out as NaN, whichever column it stands in.
__device__ __forceinline__ float max_nan(float a, float b) {
  float y;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(a), "f"(b));
  return y;
}
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float y;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}

template <int NSTAGES, int YBOXES>
struct RowSoftmaxCfg {
  static constexpr int kEpiWarps = 16;
  static constexpr int kZeroWarp = 2;                        // (a fourth warp fills up the control warps' group)
  static constexpr int kFirstEpiWarp = 4;
  static constexpr int kThreads = 32 * (kFirstEpiWarp + kEpiWarps);
  // registers a thread: the launch gives every thread 96; the control warps' group hands on what the epilogue warps take
  static constexpr int kRegsLaunch = 96, kRegsControl = 32, kRegsEpi = 112;
  static_assert(4 * kRegsControl + 16 * kRegsEpi <= 20 * kRegsLaunch, "the warps' shares have to fit what the launch holds");
  // zero boxes in flight per SM (2, 4 and 8 level in the kernel; in a kernel that writes nothing else 4 KB boxes reach 6.3 TB/s with 4 in
  // flight and 5.7 with 16 or more)
  static constexpr int ZERO_TMA_LANES = 4;
  static constexpr int CHUNK = 256;                          // columns per UMMA and per accumulator slot
  // Which of a 32-column fragment's 16 column pairs take 2^x from the FMA-pipe polynomial instead of the MUFU unit
  // (bit j = pair j).  The MUFU unit delivers 16 results per clock per SM and is this kernel's busiest pipe; the
  // polynomial costs about six issue slots per value.  Measured on the attention-score workload: none 126.2 us,
  // 4 of 16 pairs 122.7, 8: 128.8, when both passes exponentiated every score.  Now, with the writes in the way, 116.6 / 116.3 / 117.6
  // for none / 4 / 6; without them 81.9 / 76.2 / 81.8 for none / 4 / 8.
  // With a mask: a polynomial as accurate as the instruction, and in the statistics pass and the kept chunks only
  // (16 x 2048 x 2048 64.2 us, with it in the second pass too 64.4; 96 x 504 x 504 27.9, with the instruction alone 28.2).
  static constexpr uint32_t POLY_PAIRS = 0x1248u;            // pairs 3, 6, 9, 12
  static constexpr int A_BYTES = 128 * 64 * 2;
  static constexpr int STAGE_BYTES = A_BYTES + (CHUNK / 2) * 64 * 2;  // A block + this CTA's half of the B chunk
  static constexpr int WARP_BOX_BYTES = 32 * 64 * 2;
  static constexpr int OFF_YBUF = NSTAGES * STAGE_BYTES;
  static constexpr int YBUF_BYTES = kEpiWarps * YBOXES * WARP_BOX_BYTES;
  static constexpr int OFF_ZERO = OFF_YBUF + YBUF_BYTES;     // constant zero box
  static constexpr int OFF_PRE = OFF_ZERO + WARP_BOX_BYTES;  // per-row partials of the 4 column groups, two tile parities
  static constexpr int PRE_BYTES = 2 * 4 * 128 * 8;
  static constexpr int OFF_BAR = OFF_PRE + PRE_BYTES;
  static constexpr int NUM_BARS = 2 * NSTAGES + 4 + 1 + kEpiWarps * YBOXES;
  static constexpr int OFF_MISC = OFF_BAR + NUM_BARS * 8;
  static constexpr int OFF_REQ = OFF_MISC + 16;              // per epilogue warp: where its mask requests stand
  static constexpr int SMEM_BYTES = OFF_REQ + kEpiWarps * 16 + 1024;
  static_assert(SMEM_BYTES <= 232448, "shared memory budget");
  static_assert(SMEM_BYTES > 116 * 1024, "one CTA per SM is assumed (TMEM allocation never waits for a co-resident CTA)");
  static_assert(NSTAGES >= 2 && NSTAGES <= 8 && YBOXES >= 1 && YBOXES <= 4, "ring and staging depths");
};

// BKM: the B operand is stored [N, K] (one box of this CTA's 128 columns x 64 contraction elements per stage, K-major for the
// UMMA, like A) instead of [K, N] (two boxes of 64 contraction rows x 64 columns, MN-major).
// MASK: an additive mask tensor [M, N].
// kMaskThreads: a thread owns a row of the chunk and reads its mask values straight from global memory, which touches a sector per row
// and load instruction: 96 batches of 504 x 504 scores took 47.0 us that way when 36.3 with the boxes below.
// Where a batch has no more rows than one warp, that is less than a box (threads / boxes, measured with both passes over every chunk):
// 150 x 9 x 600 34.5 / 39.1, 150 x 20 x 2048 97.3 / 103.4, 40 x 32 x 6576 107.3 / 110.4; but 40 x 43 x 2048 38.1 / 37.3, 150 x 64 x
// 2048 113.4 / 103.5.
// kMaskBoxes (ADD): every epilogue warp's 32 x 64 mask box arrives by TMA in one of the warp's staging boxes, which also
// take the result: read the box, overwrite it with the probabilities, store it.
enum RowMask { kNoMask, kMaskThreads, kMaskBoxes };
template <int NSTAGES, int YBOXES, bool BKM, RowMask MASK, bool CAP>
__global__ void __launch_bounds__(32 * 20, 1)
softmax_rows_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmM, const __grid_constant__ CUtensorMap tmY, const FusedParams p) {
  using Cfg = RowSoftmaxCfg<NSTAGES, YBOXES>;
  constexpr int CHUNK = Cfg::CHUNK;
  constexpr bool ADD = MASK == kMaskBoxes;

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  const uint32_t smem_base = smem_u32(smem);

  float2* s_pre = reinterpret_cast<float2*>(smem + Cfg::OFF_PRE);
  const uint32_t bar_base = smem_base + Cfg::OFF_BAR;
  auto bar_full = [&](int s) { return bar_base + 8u * s; };                     // K-block stage landed (even CTA)
  auto bar_empty = [&](int s) { return bar_base + 8u * (NSTAGES + s); };        // stage may be overwritten
  auto bar_tfull = [&](int a) { return bar_base + 8u * (2 * NSTAGES + a); };    // accumulator slot complete
  auto bar_tempty = [&](int a) { return bar_base + 8u * (2 * NSTAGES + 2 + a); };  // slot drained by both CTAs (even CTA)
  const uint32_t bar_drain = bar_base + 8u * (2 * NSTAGES + 4);
  auto bar_mask = [&](int e, int k) { return bar_drain + 8u + 8u * (e * YBOXES + k); };
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(smem + Cfg::OFF_MISC);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + Cfg::OFF_MISC + 4);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t pm = cluster_ctarank();  // which 128-row block of the pair; rank 0 issues the UMMAs
  const int cluster_id = blockIdx.x >> 1;
  const int num_clusters = gridDim.x >> 1;
  const int KB = (p.K + 63) >> 6;
  const int nch = (p.N + CHUNK - 1) / CHUNK;
  const int rounds = (p.total_tiles + num_clusters - 1) / num_clusters;
  const WaitCtx w{s_abort, p.status, p.timeout_ns};
  griddep_launch_dependents();  // the next kernel's set-up may overlap this kernel (it waits before touching memory)

  // -------------------------------------------------------------------------------------------- set-up
  if (threadIdx.x == 0) {
    for (int s = 0; s < NSTAGES; ++s) {
      mbar_init(bar_full(s), 2);   // one arrive.expect_tx from each CTA of the pair
      mbar_init(bar_empty(s), 1);  // one commit from the issuing CTA
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(bar_tfull(a), 1);
      mbar_init(bar_tempty(a), 2 * Cfg::kEpiWarps);  // one arrival per epilogue warp of both CTAs
    }
    mbar_init(bar_drain, 1);
    for (int e = 0; e < Cfg::kEpiWarps; ++e)
      for (int k = 0; k < YBOXES; ++k) {
        mbar_init(bar_mask(e, k), 1);
      }
    *s_abort = 0;
    fence_mbar_init();
    prefetch_tensormap(&tmA);
    prefetch_tensormap(&tmB);
    prefetch_tensormap(&tmY);
    if (ADD) prefetch_tensormap(&tmM);
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(s_tmem_base), 2 * CHUNK);
    tmem_relinquish_alloc_permit_pair();
  }
  for (int i = threadIdx.x; i < Cfg::WARP_BOX_BYTES / 4; i += Cfg::kThreads) reinterpret_cast<uint32_t*>(smem + Cfg::OFF_ZERO)[i] = 0u;
  fence_proxy_async_smem();  // the zero box is read by TMA stores
  tcgen05_fence_before_sync();
  __syncthreads();
  tcgen05_fence_after_sync();
  cluster_sync_after_init();  // both CTAs' barriers exist before the peer signals them
  const uint32_t tmem_base = *s_tmem_base;
  griddep_wait();  // the set-up above may overlap the previous kernel's tail; global memory is touched only below

  // Tile of this cluster in round r.  Tiles are ordered by falling cost (under a causal mask a lower row block has
  // more live chunks) and dealt to the clusters in alternating direction, so the clusters' sums stay close.
  auto tile_at = [&](int r, int& b, int& mpair0, int& live_chunks) {
    const int pos = r * num_clusters + ((r & 1) ? num_clusters - 1 - cluster_id : cluster_id);
    if (pos >= p.total_tiles) return false;
    const int mp = p.mpairs - 1 - pos / p.batch;
    b = pos - (pos / p.batch) * p.batch;
    mpair0 = mp * 256;
    live_chunks = p.causal ? (mp + 1 < nch ? mp + 1 : nch) : nch;  // chunk c is live iff c*256 <= mpair0 + 255
    return true;
  };

  // Units (accumulators) of a tile: pass 0 takes every chunk; the exponentials of the last two stay on the chip (see the
  // epilogue), so pass 1 takes the others.  Slots alternate, except that the unit behind pass 0 takes the slot of the last
  // chunk, which is handed back as soon as it has been loaded; the one before it stays in its slot until it has been written.
  auto tile_units = [](int L) { return L < 2 ? L : 2 * L - 2; };
  auto next_slot = [](int slot, int u, int L) { return u == L - 1 && L >= 2 ? slot : slot ^ 1; };

  if (warp < Cfg::kFirstEpiWarp) {
    setmaxnreg_dec<Cfg::kRegsControl>();
    if (warp == 0) {
      // ------------------------------------------------------------------------------------------ TMA producer
      if (elect_one()) {
        int stage = 0;
        uint32_t phase = 0;
        bool ok = true;
        // every operand chunk is read twice per tile and the K matrix by every tile of its batch, while 16 times as many
        // output bytes stream through the L2: ask it to keep the operands
        const uint64_t keep = l2_policy_evict_last();
        for (int r = 0; r < rounds && ok; ++r) {
          int b, mpair0, L;
          if (!tile_at(r, b, mpair0, L)) continue;
          const int m0 = mpair0 + static_cast<int>(pm) * 128;
          for (int u = 0; u < tile_units(L) && ok; ++u) {
            const int c = u < L ? u : u - L;  // pass 0 over the live chunks, then pass 1 over those whose exponentials were not kept
            for (int kb = 0; kb < KB; ++kb) {
              if (!mbar_wait<false>(bar_empty(stage), phase ^ 1u, w)) { ok = false; break; }  // passes on a fresh barrier
              const uint32_t sa = smem_base + stage * Cfg::STAGE_BYTES;
              const uint32_t full = map_to_cta(bar_full(stage), 0);
              mbar_arrive_expect_tx_cluster(full, Cfg::STAGE_BYTES);
              tma_load_3d_pair_hint(sa, &tmA, full, kb * 64, m0, b, keep);
              // this CTA's half of the UMMA's B tile: two boxes of 64 columns, 8 KB apart
              const int col = c * CHUNK + static_cast<int>(pm) * (CHUNK / 2);
              if constexpr (BKM) {  // two boxes of 64 rows of B (columns of the product) x 64 contraction elements
                tma_load_3d_pair_hint(sa + Cfg::A_BYTES, &tmB, full, kb * 64, col, b, keep);
                tma_load_3d_pair_hint(sa + Cfg::A_BYTES + 8192, &tmB, full, kb * 64, col + 64, b, keep);
              } else {
                tma_load_3d_pair_hint(sa + Cfg::A_BYTES, &tmB, full, col, kb * 64, b, keep);
                tma_load_3d_pair_hint(sa + Cfg::A_BYTES + 8192, &tmB, full, col + 64, kb * 64, b, keep);
              }
              if (++stage == NSTAGES) { stage = 0; phase ^= 1u; }
            }
          }
        }
      }
    } else if (warp == 1) {
      // ------------------------------------------------------------------------------------------ UMMA issuer (even CTA)
      if (pm == 0 && elect_one()) {
        int stage = 0;
        uint32_t phase = 0;
        uint32_t slot_uses[2] = {0, 0};
        int slot = 0;
        constexpr uint32_t idesc = make_idesc_bf16(256, CHUNK, false, !BKM);
        bool ok = true;
        for (int r = 0; r < rounds && ok; ++r) {
          int b, mpair0, L;
          if (!tile_at(r, b, mpair0, L)) continue;
          for (int u = 0; u < tile_units(L) && ok; ++u, slot = next_slot(slot, u - 1, L)) {
            if (!mbar_wait<false>(bar_tempty(slot), (slot_uses[slot] & 1u) ^ 1u, w)) { ok = false; break; }
            ++slot_uses[slot];
            tcgen05_fence_after_sync();
            const uint32_t d_tmem = tmem_base + slot * CHUNK;
            for (int kb = 0; kb < KB; ++kb) {
              if (!mbar_wait<false>(bar_full(stage), phase, w)) { ok = false; break; }
              tcgen05_fence_after_sync();
              const uint32_t sa = smem_base + stage * Cfg::STAGE_BYTES;
              const uint64_t adesc = make_smem_desc_sw128(sa, 16, 1024);
              const uint64_t bdesc = BKM ? make_smem_desc_sw128(sa + Cfg::A_BYTES, 16, 1024)
                                         : make_smem_desc_sw128(sa + Cfg::A_BYTES, /*next 64-column block*/ 8192, /*next 8 K rows*/ 1024);
#pragma unroll
              for (int k = 0; k < 4; ++k)  // K advances by 16 elements: 32 bytes inside a K-major operand's swizzled row, 2048 bytes in an MN-major B
                umma_bf16_ss_pair(d_tmem, adesc + static_cast<uint64_t>(k * 2), bdesc + static_cast<uint64_t>(BKM ? k * 2 : k * 128), idesc,
                                  (kb | k) != 0 ? 1u : 0u);
              umma_commit_pair_both(bar_empty(stage));
              if (++stage == NSTAGES) { stage = 0; phase ^= 1u; }
            }
            if (!ok) break;
            umma_commit_pair_both(bar_tfull(slot));
          }
        }
        umma_commit_pair(bar_drain);  // nothing may still be writing either CTA's TMEM when it is freed
        mbar_drain(bar_drain, 0, w);
      }
    } else if (warp == Cfg::kZeroWarp) {
      // ------------------------------------------------------------------------------------------ zero-box warp
      // The chunks above the causal diagonal hold zeros and depend on nothing.  A few lanes, each with one TMA store of a
      // constant zero box in flight, walk them with a cursor of their own, independent of the epilogue (asynchronous
      // stores: plain stores would share the SM's memory-instruction queue with the epilogue's exponentials and
      // shared-memory traffic).  Few boxes in flight, so that a staged box never queues far behind zeros.
      if (lane < Cfg::ZERO_TMA_LANES && p.causal) {
        const uint64_t stream_out = l2_policy_evict_first();
        uint32_t k = 0;
        for (int r = 0; r < rounds; ++r) {
          int b, mpair0, L;
          if (!tile_at(r, b, mpair0, L)) continue;
          const int y0 = mpair0 + static_cast<int>(pm) * 128;
          for (int c = L; c < nch; ++c)
            for (int i = 0; i < 16; ++i, ++k) {
              if (k % Cfg::ZERO_TMA_LANES != static_cast<uint32_t>(lane)) continue;
              const int col = c * CHUNK + (i >> 2) * 64;
              if (col >= p.N) continue;
              tma_store_wait_all();
#ifdef COMFUSE_TRACE
              if (!(p.trace_flags & 4))
#endif
              if (COMFUSE_IN_BOUNDS(col >= 0 && (col & 7) == 0 && y0 >= 0 && b >= 0 && b < p.batch, p.status))
              tma_store_3d_hint(&tmY, smem_base + Cfg::OFF_ZERO, col, y0 + (i & 3) * 32, b, stream_out);
              tma_store_commit();
            }
        }
        tma_store_wait_read<0>();
      }
    }
  } else {
    setmaxnreg_inc<Cfg::kRegsEpi>();
    // ------------------------------------------------------------------------------------------ epilogue warps
    const int e = warp - Cfg::kFirstEpiWarp;
    const int q = warp & 3;  // TMEM lane quarter this warp may touch: rows 32q .. 32q+31 of the CTA's row block
    const int h = e >> 2;    // the 64-column group of every chunk this warp takes
    const int row = q * 32 + lane;
    const uint32_t lane_sel = static_cast<uint32_t>(q * 32) << 16;
    const uint32_t tempty_leader = map_to_cta(bar_tempty(0), 0);
    const uint32_t ybox0 = smem_base + Cfg::OFF_YBUF + e * YBOXES * Cfg::WARP_BOX_BYTES;
    // Exponentials are 2^(scale * (t - maximum)), t a score.  plain: t is the accumulator and the scale alpha * log2 e (a positive one);
    // with a mask: t = alpha * Acc + mask and the scale log2 e; otherwise t is transformed to the log2 domain first and the scale 1.
    // With a mask the difference comes first, which is an exact zero for the maximum whatever its size: with the scaled maximum taken
    // off in a fused multiply-add it is that product's rounding, hundreds for a column masked with -1e10.  Without one it is that
    // multiply-add, and the other order where a maximum is beyond kFar (64 x 2048 x 2048 causal 114.4 us, with the difference first 115.0).
    constexpr float kLog2e = 1.4426950408889634f;
    constexpr bool additive = MASK != kNoMask;  // additive mask tensor, applied behind the scale / soft-cap
    SoftcapLog2 cap_fn(p.alpha, CAP ? p.softcap : 1.f);
    if (additive) cap_fn.c1 = p.softcap;
    const float sc = CAP ? 1.f : additive ? p.alpha : p.alpha * kLog2e;
    const bool plain = !additive && !CAP && sc > 0.f;
    const float scale = plain ? sc : additive ? kLog2e : 1.f;
    constexpr float kFar = 1024.f;
    auto any_far = [&](float scaled) { return !additive && !CAP && __any_sync(0xFFFFFFFFu, fabsf(scaled) > kFar); };  // (with a soft-cap the scale is 1)
    auto take_off = [&](uint32_t (&va)[32], uint32_t (&vb)[32], float ref) {
#pragma unroll
      for (int j = 0; j < 32; j += 2) {
        const float2 a = add2(f2_from_bits(va[j], va[j + 1]), splat2(-ref)), b = add2(f2_from_bits(vb[j], vb[j + 1]), splat2(-ref));
        va[j] = __float_as_uint(a.x);
        va[j + 1] = __float_as_uint(a.y);
        vb[j] = __float_as_uint(b.x);
        vb[j + 1] = __float_as_uint(b.y);
      }
    };

    int slot = 0;
    // phase bits: 0, 1 of the slots, 2 .. of the mask boxes, 31 which half of s_pre
    uint32_t phases = 0;
    auto wait_slot = [&](int sl) {
      mbar_wait<false>(bar_tfull(sl), (phases >> sl) & 1u, w);
      phases ^= 1u << sl;
      __syncwarp();
      tcgen05_fence_after_sync();
    };
    auto release_slot = [&](int sl) {
      tcgen05_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster_noflush(tempty_leader + 8u * sl);
    };

    // Staging boxes: use n of this warp takes box n % YBOXES.  A use holds the chunk's mask (ADD), its result, or first one and
    // then the other.  The elected lane issues the stores itself; it hands a box on when its store has read it, and asks for the
    // mask of the box's next use then.  (The L2 policies are made where they are used: the 64 columns leave few registers.)
    const bool elected = elect_one();
    uint32_t use = 0;
    // ADD: the uses of a tile (causal off: L = nch) are nch - 1 masks, mask and result of the last chunk (if it has columns for
    // this warp), the result of the one before, masks and results of the others
    const bool has_last = (nch - 1) * CHUNK + h * 64 < p.N;
    const int tile_uses = tile_units(nch) + (nch >= 2 ? 1 : 0) - (has_last ? 0 : 1);
    // round, use and first row of the next request: in shared memory, read and written by the elected lane alone
    volatile int* req = reinterpret_cast<volatile int*>(smem + Cfg::OFF_REQ) + 4 * e;
    auto request_use = [&](uint32_t sel) {  // (the elected lane) the mask of the next use not asked for yet, if it has one, into its box
      int req_r = req[0], req_i = req[1], req_row = req[2];
      if (req_i >= tile_uses) {
        req_i = 0;
        if (req_r < rounds) {
          do {  // (tiles in which this warp's rows do not exist are passed over)
            int lb, lm = 0, lL;
            if (++req_r < rounds && !tile_at(req_r, lb, lm, lL)) req_r = rounds;
            req_row = lm + static_cast<int>(pm) * 128 + q * 32;
          } while (req_r < rounds && req_row >= p.M);
        }
        req[0] = req_r;
        req[2] = req_row;
      }
      if (tile_uses <= 0 || req_r >= rounds) return;
      const int first_out = nch - (has_last ? 0 : 1);  // the use without a mask
      const int c = req_i < first_out ? req_i : req_i - first_out - 1;
      if (c >= 0) {
        mbar_arrive_expect_tx(bar_mask(e, sel), Cfg::WARP_BOX_BYTES);
        tma_load_3d_hint(ybox0 + sel * Cfg::WARP_BOX_BYTES, &tmM, bar_mask(e, sel), c * CHUNK + h * 64, req_row, 0, l2_policy_evict_last());
      }
      req[1] = req_i + 1;
    };
    if constexpr (ADD) {
      if (elected) {
        req[0] = -1;
        req[1] = tile_uses;
        for (int i = 0; i < YBOXES; ++i) request_use(i);
      }
      __syncwarp();
    }
    bool store_pending = false;
    // in front of a use: the previous use's box, once its store has read it, takes the mask of the use after this one
    auto reclaim_box = [&]() {
      if constexpr (ADD) {
        if (!store_pending) return;
        if (elected) {
          tma_store_wait_read<0>();
          request_use((use + YBOXES - 1) % YBOXES);
        }
        __syncwarp();
        store_pending = false;
      }
    };
    auto wait_mask = [&]() {
      const uint32_t sel = use % YBOXES;
      mbar_wait<false>(bar_mask(e, sel), (phases >> (2 + sel)) & 1u, w);
      phases ^= 4u << sel;
      __syncwarp();
    };
    auto end_mask_use = [&]() {  // the use held a mask only and every lane has read its row
      __syncwarp();
      if (elected) request_use(use % YBOXES);
      __syncwarp();
      ++use;
    };
    // 64 result columns of this thread's row -> the box of this use -> global memory
    auto emit = [&](const uint32_t (&pk)[32], int colg, int row0, int b) {
      const uint32_t ybox = ybox0 + (use % YBOXES) * Cfg::WARP_BOX_BYTES;
      ++use;
      if constexpr (!ADD) {
        if (elected) tma_store_wait_read<YBOXES - 1>();
        __syncwarp();
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const uint32_t a = ybox + static_cast<uint32_t>(lane * 128 + ((i ^ (lane & 7)) << 4));  // 128-byte swizzle
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(pk[4 * i]), "r"(pk[4 * i + 1]),
                     "r"(pk[4 * i + 2]), "r"(pk[4 * i + 3])
                     : "memory");
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (elected) {
        if (COMFUSE_IN_BOUNDS(colg >= 0 && colg < p.N && (colg & 7) == 0 && row0 >= 0 && b >= 0 && b < p.batch, p.status))
        tma_store_3d_hint(&tmY, ybox, colg, row0, b, l2_policy_evict_first());  // the output is never read again
        tma_store_commit();
      }
      __syncwarp();
      store_pending = true;
    };
    // scores of 32 columns, in place (not in the plain case): soft-cap or scale, mask
    auto transform = [&](uint32_t (&v)[32], int half, int grow, int col0) {
      if constexpr (CAP) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(cap_fn(__uint_as_float(v[j])));
      }
      if constexpr (ADD) {
        const uint32_t box = ybox0 + (use % YBOXES) * Cfg::WARP_BOX_BYTES;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t w4[4];
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(w4[0]), "=r"(w4[1]), "=r"(w4[2]), "=r"(w4[3])
                       : "r"(box + static_cast<uint32_t>(lane * 128 + (((half * 4 + i) ^ (lane & 7)) << 4)))
                       : "memory");
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float2 t = fma2(f2_from_bits(v[8 * i + 2 * k], v[8 * i + 2 * k + 1]), splat2(sc), bf16x2_to_f2(w4[k]));
            v[8 * i + 2 * k] = __float_as_uint(t.x);
            v[8 * i + 2 * k + 1] = __float_as_uint(t.y);
          }
        }
      } else if constexpr (additive) {
        float2 m2[16];
        load_mask_32(p.mask + static_cast<long long>(grow) * p.N + col0, grow < p.M ? p.N - col0 : 0, m2);
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float2 t = fma2(f2_from_bits(v[2 * j], v[2 * j + 1]), splat2(sc), m2[j]);
          v[2 * j] = __float_as_uint(t.x);
          v[2 * j + 1] = __float_as_uint(t.y);
        }
      } else if constexpr (!CAP) {
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) * sc);
      }
    };
    auto scores = [&](uint32_t (&va)[32], uint32_t (&vb)[32], int c, int grow) {
      if constexpr (ADD) {
        reclaim_box();
        wait_mask();
      }
      if (!plain) {
        transform(va, 0, grow, c * CHUNK + h * 64);
        transform(vb, 1, grow, c * CHUNK + h * 64 + 32);
      }
    };
    // this thread's running maximum of the row and sum of 2^(scale * (t - max))
    float m_run, s_run;
    // takes 64 scores into (m_run, s_run) and leaves 2^(scale * (t - m_run)) in their place (kKeep), or nothing
    auto accumulate = [&](uint32_t (&va)[32], uint32_t (&vb)[32], auto keep) {
      constexpr bool kKeep = decltype(keep)::value;
      constexpr uint32_t poly = Cfg::POLY_PAIRS;
      float mx0 = -INFINITY, mx1 = -INFINITY;
#pragma unroll
      for (int j = 0; j < 32; j += 4) {
        mx0 = max3_nan(mx0, __uint_as_float(va[j]), __uint_as_float(va[j + 1]));
        mx1 = max3_nan(mx1, __uint_as_float(va[j + 2]), __uint_as_float(va[j + 3]));
      }
#pragma unroll
      for (int j = 0; j < 32; j += 4) {
        mx0 = max3_nan(mx0, __uint_as_float(vb[j]), __uint_as_float(vb[j + 1]));
        mx1 = max3_nan(mx1, __uint_as_float(vb[j + 2]), __uint_as_float(vb[j + 3]));
      }
      const float m_new = max_nan(m_run, max_nan(mx0, mx1));
      const float ref = m_new == -INFINITY ? 0.f : m_new;  // (nothing but masked columns so far)
      float r = scale * ref;  // (not with a mask)
      if (any_far(r)) {
        take_off(va, vb, ref);
        r = 0.f;
      }
      // Sums of a few pairs at a time: one chain of 32 rounds more often.  (Two are what costs nothing without a mask: 96 x 512 x 512
      // 17.9 us, four 18.5, four chains of eight 18.5.)
      constexpr int kGroup = additive ? 4 : 2;
      float2 acc = make_float2(0.f, 0.f), part = acc;
      auto exponentials = [&](uint32_t (&v)[32]) {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float2 t = f2_from_bits(v[2 * j], v[2 * j + 1]);
          float2 x;
          if constexpr (additive) {
            const float2 d = add2(t, splat2(-ref));
            if ((poly >> j) & 1u) {
              x = exp_poly2(d);
            } else {
              const float2 d2 = mul2(d, splat2(kLog2e));
              x = make_float2(ex2_approx(d2.x), ex2_approx(d2.y));
            }
          } else {
            const float2 d = fma2(t, splat2(scale), splat2(-r));
            x = ((poly >> j) & 1u) ? ex2_poly2(d) : make_float2(ex2_approx(d.x), ex2_approx(d.y));
          }
          part = j % kGroup == 0 ? x : add2(part, x);
          if (j % kGroup == kGroup - 1) acc = add2(acc, part);
          if constexpr (kKeep) {
            v[2 * j] = __float_as_uint(x.x);
            v[2 * j + 1] = __float_as_uint(x.y);
          }
        }
      };
      exponentials(va);
      exponentials(vb);
      const float sum = m_new == -INFINITY ? 0.f : acc.x + acc.y;
      s_run = fmaf(s_run, ex2_approx(scale * (m_run - ref)), sum);
      m_run = m_new;
    };
    auto load_slot = [&](uint32_t taddr, uint32_t (&va)[32], uint32_t (&vb)[32]) {
#pragma unroll
      for (int i = 0; i < 32; i += 16) {
        tmem_ld_issue_16(taddr + i, va + i);
        tmem_ld_issue_16(taddr + 32 + i, vb + i);
      }
#pragma unroll
      for (int i = 0; i < 32; i += 16) {
        tmem_ld_wait_16(va + i);
        tmem_ld_wait_16(vb + i);
      }
    };

    for (int r = 0; r < rounds; ++r) {
      int b, mpair0, L;
      if (!tile_at(r, b, mpair0, L)) continue;
      const int row0 = mpair0 + static_cast<int>(pm) * 128 + q * 32;  // the warp's first row
      const int grow = row0 + lane;
      if (additive && row0 >= p.M) {
        // none of this warp's rows exists (nor of the three it merges with): the accumulators are handed back as they come.
        // With boxes for all warps 134 x 1 x 720 took 35.0 us instead of 31.2, 64 x 16 x 1176 27.9 instead of 24.9.
        for (int u = 0; u < tile_units(L); ++u) {
          wait_slot(slot);
          release_slot(slot);
          slot = next_slot(slot, u, L);
        }
        continue;
      }
      m_run = -INFINITY;
      s_run = 0.f;
      float m_kept = -INFINITY;  // what the kept exponentials of the last chunk but one are relative to
      // ---------------- pass 0: online (max, sum of 2^(t - max)) over this thread's columns of each chunk.  All columns of all
      // chunks but the last are live.
      for (int c = 0; c < L - 2; ++c) {
        uint32_t va[32], vb[32];
        wait_slot(slot);
        load_slot(tmem_base + lane_sel + slot * CHUNK + h * 64, va, vb);
        release_slot(slot);
        slot ^= 1;
        scores(va, vb, c, grow);
        if constexpr (ADD) end_mask_use();
        accumulate(va, vb, std::false_type{});
      }
      if (L >= 2) {  // the exponentials of the last chunk but one stay in its accumulator slot
        uint32_t va[32], vb[32];
        wait_slot(slot);
        const uint32_t taddr = tmem_base + lane_sel + slot * CHUNK + h * 64;
        load_slot(taddr, va, vb);
        slot ^= 1;
        scores(va, vb, L - 2, grow);
        if constexpr (ADD) end_mask_use();
        accumulate(va, vb, std::true_type{});
        m_kept = m_run;
#pragma unroll
        for (int i = 0; i < 32; i += 16) {
          tmem_st_16(taddr + i, va + i);
          tmem_st_16(taddr + 32 + i, vb + i);
        }
        tmem_st_wait();
      }
      // The four column groups of the row (they live in the four warps of this lane quarter) meet: P = 2^(scale * (t - m_row) - off), off
      // the sum's logarithm.  A row without a live column (which cannot happen under the causal mask) is all zero: m_row 0 and off +inf.
      float m_row, off;
      auto meet = [&]() {
        float2* pre = s_pre + (phases >> 31) * 512;
        phases ^= 1u << 31;
        pre[h * 128 + row] = make_float2(m_run, s_run);
        named_barrier_sync(1 + q, 128);
        float m_all = -INFINITY, s_all = 0.f;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 o = pre[i * 128 + row];
          const float m_new = max_nan(m_all, o.x);
          if (m_new != -INFINITY) {
            s_all = s_all * ex2_approx(scale * (m_all - m_new)) + o.y * ex2_approx(scale * (o.x - m_new));
            m_all = m_new;
          }
        }
        m_row = m_all == -INFINITY ? 0.f : m_all;
        off = m_all == -INFINITY ? INFINITY : m_all < INFINITY ? __log2f(s_all) : NAN;
      };
      // what turns exponentials relative to m into probabilities
      auto factor = [&](float m) { return ex2_approx(fmaf(scale, m - m_row, -off)); };
      {
        // ---------------- the last chunk: its exponentials stay in registers
        const int colg = (L - 1) * CHUNK + h * 64;
        const bool causal = !additive && p.causal;  // (one mask or the other)
        const int lim = causal && grow < p.N - 1 ? grow : p.N - 1;  // last live column of this thread's row
        const int lim_lo = causal && row0 < p.N - 1 ? row0 : p.N - 1;
        const int lim_hi = causal && row0 + 31 < p.N - 1 ? row0 + 31 : p.N - 1;
        wait_slot(slot);
        if (colg <= lim_hi) {  // uniform over the warp
          uint32_t va[32], vb[32];
          load_slot(tmem_base + lane_sel + slot * CHUNK + h * 64, va, vb);
          release_slot(slot);
          scores(va, vb, L - 1, grow);
          if constexpr (ADD) __syncwarp();
          const bool whole = colg + 63 <= lim_lo;  // else it crosses the diagonal or the end of the row
          if (!whole) {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              if (colg + j > lim) va[j] = __float_as_uint(-INFINITY);
              if (colg + 32 + j > lim) vb[j] = __float_as_uint(-INFINITY);
            }
          }
          accumulate(va, vb, std::true_type{});
          const float m_last = m_run;
          meet();
          const float f = factor(m_last);
          uint32_t pk[32];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            pk[j] = pack_bf16x2_rn(mul2(f2_from_bits(va[2 * j], va[2 * j + 1]), splat2(f)));
            pk[16 + j] = pack_bf16x2_rn(mul2(f2_from_bits(vb[2 * j], vb[2 * j + 1]), splat2(f)));
          }
          emit(pk, colg, row0, b);
        } else {
          release_slot(slot);
          if constexpr (ADD) reclaim_box();
          meet();
          if (colg < p.N) {  // above the diagonal
            uint32_t pk[32];
#pragma unroll
            for (int j = 0; j < 32; ++j) pk[j] = 0u;
            emit(pk, colg, row0, b);
          }
        }
        slot = next_slot(slot, L - 1, L);
      }
      if (L >= 2) {
        // ---------------- the chunk before it: its exponentials are in its accumulator slot
        const int kslot = slot ^ 1;
        uint32_t va[32], vb[32];
        load_slot(tmem_base + lane_sel + kslot * CHUNK + h * 64, va, vb);
        release_slot(kslot);
        const float f = factor(m_kept);
        uint32_t pk[32];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          pk[j] = pack_bf16x2_rn(mul2(f2_from_bits(va[2 * j], va[2 * j + 1]), splat2(f)));
          pk[16 + j] = pack_bf16x2_rn(mul2(f2_from_bits(vb[2 * j], vb[2 * j + 1]), splat2(f)));
        }
        reclaim_box();
        emit(pk, (L - 2) * CHUNK + h * 64, row0, b);
      }
      // ---------------- pass 1: the other chunks' scores again, normalised, rounded once, staged and stored
      const bool far = any_far(scale * m_row);
      if (!additive && !far) off = fmaf(scale, m_row, off);
      for (int c = 0; c < L - 2; ++c) {
        wait_slot(slot);
        uint32_t va[32], vb[32];
        load_slot(tmem_base + lane_sel + slot * CHUNK + h * 64, va, vb);
        release_slot(slot);
        scores(va, vb, c, grow);
        if constexpr (ADD) __syncwarp();  // every lane has read its row of the mask
        if (additive || far) take_off(va, vb, m_row);
        constexpr uint32_t poly = additive ? 0u : Cfg::POLY_PAIRS;
        uint32_t pk[32];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float2 d0 = fma2(f2_from_bits(va[2 * j], va[2 * j + 1]), splat2(scale), splat2(-off));
          const float2 d1 = fma2(f2_from_bits(vb[2 * j], vb[2 * j + 1]), splat2(scale), splat2(-off));
          pk[j] = pack_bf16x2_rn(((poly >> j) & 1u) ? ex2_poly2(d0) : make_float2(ex2_approx(d0.x), ex2_approx(d0.y)));
          pk[16 + j] = pack_bf16x2_rn(((poly >> j) & 1u) ? ex2_poly2(d1) : make_float2(ex2_approx(d1.x), ex2_approx(d1.y)));
        }
        if (off != off) {  // a row with a NaN (the polynomial's clamp takes one for a masked score)
#pragma unroll
          for (int j = 0; j < 32; ++j) pk[j] = 0x7FFF7FFFu;
        }
        emit(pk, c * CHUNK + h * 64, row0, b);
        slot ^= 1;
      }
    }
    if (elected) tma_store_wait_read<0>();  // the boxes must outlive the last store's read
  }

  // -------------------------------------------------------------------------------------------- teardown
  tcgen05_fence_before_sync();
  __syncthreads();
  cluster_sync_all();  // the peer may no longer signal this CTA's barriers or write its TMEM
  if (warp == 1) {
    __syncwarp();
    tcgen05_fence_after_sync();
    tmem_dealloc_pair(tmem_base, 2 * CHUNK);
    if (lane == 0) linger_behind_expired_wait(w);
  }
}

}  // namespace comfuse
