// LayerNorm, RMSNorm and softmax kinds behind a GEMM of few rows.
//
// What bounds it: the weights, and below a few megabytes of them the latency of one pass through the kernel.  A decoding step
// of 40 rows through a 4096 x 4096 layer moves 33.5 MB of weights and multiplies almost nothing; the tile kernel (256-row CTA
// pairs) gives such a call as many clusters as the row has column blocks and leaves the other SMs idle, and pays a 256-row
// MainLoop and epilogue for every row block however few rows it holds.  This kernel turns the product round and cuts it finer:
//
//   * The weights are the UMMA's 128-row operand and the activations its N operand (D^T = B^T . A^T): a CTA computes
//     128 (or 2 x 128) columns of the result for `MT` = 16 .. 64 rows, so the tensor core's work follows the rows that exist.
//   * A cluster has CT x KS CTAs: CT column ranges and, for each, KS equal shares of the contraction (split K).  The shares'
//     fp32 accumulators meet in a reduce-scatter over distributed shared memory: share j receives the others' partial sums
//     of the j-th slice of the rows (one bulk copy per peer) and finishes those rows.
//   * A warp then owns a row of the CTA's columns (lane = 4 columns): the residual and the result move as coalesced 8-byte
//     accesses, the row statistic is a shuffle reduction, and the CT partials of a row are exchanged through distributed
//     shared memory as in the tile kernel.  16 epilogue warps, so that a warp has at most four rows and they advance
//     together: with 8 warps and a loop over the rows the epilogue of 64 rows took 9000 clocks, now about 2000.
//   * Softmax kind: the same, with (maximum, sum of exponentials) as the statistic.  A CTA exponentiates against the maximum
//     of its own columns, so every score takes one exponential; the exchange yields the factor that corrects for the row.
//   * Rows that the tile kernel would cut into 256-column blocks (the two-kernel form) are cut here too: x goes out as fp16
//     with the block's statistic, and the finishing kernel normalises it.
//
// A K block costs a CTA about 250 clocks (three TMA requests, 24 KB through shared memory, four UMMAs).
#include <atomic>

#include "epilogue_common.cuh"
#include "few_rows.h"

namespace comfuse {
namespace {

template <int NT, int MT>
struct FewRowsCfg {
  static constexpr int kEpiWarps = 16;
  static constexpr int kThreads = 32 * (2 + kEpiWarps);
  static constexpr int W_BYTES = NT * 128 * 64 * 2;         // weights of one K block
  static constexpr int X_BYTES = MT * 64 * 2;               // rows of one K block
  static constexpr int STAGE_BYTES = W_BYTES + X_BYTES;
  // K blocks asked of the L2 ahead of the loads: under the set-up, and at most (148 CTAs: less than half of the L2)
  static constexpr int ASK_FIRST = 128 * 1024 / W_BYTES, ASK_MOST = 384 * 1024 / W_BYTES;
  static constexpr int ROW_BYTES = NT * 128 * 4;            // one row of the CTA's columns, fp32
  static constexpr int RECV_BYTES = (MT + 7) * ROW_BYTES;   // partial sums of the CTA's row slice from up to 8 shares (8 * ceil(MT / 8) rows)
  static constexpr int STAT_BYTES = MT * 16 * 8;            // one exchange: up to 16 partials per row
  static constexpr int MISC_BYTES = 256 + 1024;
  static constexpr int STAGES_FIT = (232448 - RECV_BYTES - 2 * STAT_BYTES - MISC_BYTES) / STAGE_BYTES;
  static constexpr int NSTAGES = STAGES_FIT > 10 ? 10 : STAGES_FIT;
  static constexpr int OFF_RECV = NSTAGES * STAGE_BYTES;
  static constexpr int OFF_STAT = OFF_RECV + RECV_BYTES;
  static constexpr int OFF_BAR = OFF_STAT + 2 * STAT_BYTES;
  static constexpr int NUM_BARS = 2 * NSTAGES + 4;
  static constexpr int OFF_MISC = OFF_BAR + NUM_BARS * 8;
  static constexpr int SMEM_BYTES = OFF_MISC + 32 + 1024;
  static constexpr int TMEM_COLS = NT * MT <= 32 ? 32 : NT * MT <= 64 ? 64 : 128;
  static_assert(MT % 16 == 0 && NT * MT <= 128, "UMMA shape and tensor memory");
  static_assert(STAGE_BYTES % 1024 == 0, "swizzled tiles start on 1024-byte boundaries");
  static_assert(MT * ROW_BYTES <= NSTAGES * STAGE_BYTES, "the accumulators are staged in the idle ring");
  static_assert(NUM_BARS * 8 + 32 <= 256, "barrier room");
  static_assert(SMEM_BYTES <= 232448 && SMEM_BYTES > 116 * 1024, "one CTA per SM (tensor-memory allocation never waits)");
};

// Merge R rows' partials (a[i], b[i]) over the 32 lanes.  At step s (lane distance 16 >> s) a lane keeps one half of the rows
// it still holds and hands the other half to its partner, so R rows take R - 1 + (5 - log2 R) exchanges instead of 5 R.
// The result for row transposed_row<R>(lane) ends up in a[0], b[0].  merge(step, a0, a1, b0, b1): own partial, partner's.
template <int R>
__device__ __forceinline__ int transposed_row(int lane) {
  int row = 0;
#pragma unroll
  for (int s = 0; (1 << s) < R; ++s) row |= (lane & (16 >> s)) ? (R >> (s + 1)) : 0;
  return row;
}
template <int R, class Merge>
__device__ __forceinline__ void transposed_reduce(float (&a)[R], float (&b)[R], int lane, Merge merge) {
#pragma unroll
  for (int s = 0; s < 5; ++s) {
    const int o = 16 >> s;
    const int keep = R >> (s + 1);  // rows kept behind this step (0: down to one row already)
    if (keep > 0) {
      const bool upper = (lane & o) != 0;
#pragma unroll
      for (int i = 0; i < (keep > 0 ? keep : 1); ++i) {
        const float ga = upper ? a[i] : a[i + keep], gb = upper ? b[i] : b[i + keep];  // given away
        if (upper) { a[i] = a[i + keep]; b[i] = b[i + keep]; }
        merge(s, a[i], b[i], __shfl_xor_sync(0xFFFFFFFFu, ga, o), __shfl_xor_sync(0xFFFFFFFFu, gb, o));
      }
    } else {
      merge(s, a[0], b[0], __shfl_xor_sync(0xFFFFFFFFu, a[0], o), __shfl_xor_sync(0xFFFFFFFFu, b[0], o));
    }
  }
}

template <int EPI, int NT, int MT>
__global__ void __launch_bounds__(FewRowsCfg<NT, MT>::kThreads, 1)
few_rows_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const FewRowsParams p) {
  using Cfg = FewRowsCfg<NT, MT>;
  constexpr int NSTAGES = Cfg::NSTAGES;
  constexpr int RC = MT / Cfg::kEpiWarps;  // rows per epilogue warp
  constexpr int COLS = NT * 128;

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  const uint32_t smem_base = smem_u32(smem);
  // the ring, once idle: [row][COLS] fp32, this CTA's accumulators; OFF_RECV: [share][row of the slice][COLS], the peers'
  float2* s_stat = reinterpret_cast<float2*>(smem + Cfg::OFF_STAT);  // [exchange][row of the slice][16]
  const uint32_t bar_base = smem_base + Cfg::OFF_BAR;
  auto bar_full = [&](int s) { return bar_base + 8u * s; };
  auto bar_empty = [&](int s) { return bar_base + 8u * (NSTAGES + s); };
  const uint32_t bar_acc = bar_base + 8u * (2 * NSTAGES);  // accumulators complete
  const uint32_t bar_recv = bar_acc + 8u;                  // partial sums of the other shares have arrived
  const uint32_t bar_stat = bar_acc + 16u;                 // row statistics of the CT column ranges
  const uint32_t bar_max = bar_acc + 24u;                  // row maxima (column range 0 only)
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(smem + Cfg::OFF_MISC);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + Cfg::OFF_MISC + 4);
  volatile int* s_told = s_abort + 1;    // a wait expired in some CTA of the cluster
  volatile int* s_issued = s_abort + 2;  // K blocks whose loads are issued (fewer than all where the producer's wait expires)
  volatile int* s_begun = s_abort + 3;   // the previous kernel has ended

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int ct = rank / p.ks;       // column range
  const int ks = rank - ct * p.ks;  // share of the contraction, and slice of the rows in the epilogue
  const int work = blockIdx.x / (p.ct * p.ks);
  const int nb = work % p.nblocks;
  const int grp = (work / p.nblocks) % p.groups;
  const int b = work / (p.nblocks * p.groups);
  const int n0 = (nb * p.ct + ct) * COLS;
  const int m0 = grp * MT;
  const int rows = p.M - m0 < MT ? p.M - m0 : MT;
  const int rs = (rows + p.ks - 1) / p.ks;  // rows per slice
  auto slice_rows = [&](int j) { return rows - j * rs < 0 ? 0 : (rows - j * rs < rs ? rows - j * rs : rs); };
  const int rv = slice_rows(ks);
  const int KB = (p.K + 63) >> 6;
  const int kb0 = KB * ks / p.ks, kb1 = KB * (ks + 1) / p.ks;
  const WaitCtx w{s_abort, p.status, p.timeout_ns};
  griddep_launch_dependents();  // the next kernel's set-up may overlap this kernel (it waits before touching memory)

  // -------------------------------------------------------------------------------------------- set-up
  if (threadIdx.x == 0) {
    for (int s = 0; s < NSTAGES; ++s) {
      mbar_init(bar_full(s), 1);
      mbar_init(bar_empty(s), 1);
    }
    mbar_init(bar_acc, 1);
    mbar_init(bar_recv, 1);
    mbar_init(bar_stat, 1);
    mbar_init(bar_max, 1);
    *s_abort = 0;
    *s_told = 0;
    *s_begun = 0;
    *s_issued = kb1 - kb0;
    fence_mbar_init();
    // what each exchange will deliver is known now: arm the barriers before any peer can send
    mbar_arrive_expect_tx(bar_recv, static_cast<uint32_t>((p.ks - 1) * rv * Cfg::ROW_BYTES));
    mbar_arrive_expect_tx(bar_stat, static_cast<uint32_t>(p.ct * rv * 8));
    mbar_arrive_expect_tx(bar_max, static_cast<uint32_t>(ct == 0 ? p.ct * rv * 8 : 0));
    prefetch_tensormap(&tmW);
    prefetch_tensormap(&tmX);
  }
  // Two-kernel form: the weights are asked of the L2 while the previous kernel still runs (a prefetch returns nothing, so it may stand in
  // front of the wait whoever writes the weights: writes meet in the L2 too), by one row group.  First as many blocks as the set-up covers, which
  // a lone call gains from as well; then, while the previous kernel lasts, the others.  A request takes the time of a load: all of
  // them under the set-up held back the loads of calls that had nothing to wait for.  Us a call, without / all under the set-up / this; queued
  // with weights from memory, behind a kernel that lets no successor start early with weights from memory and from the L2:
  //   40 x 4096 x 4096  13.1 / 12.4 / 12.0, 13.4 / 13.4 / 13.3, 11.3 / 12.2 / 11.3    4 x 4096 x 1024  7.7 / 7.2 / 7.0, 8.4 / 7.2 / 7.2, 7.2 / 7.2 / 7.2
  //   16 x 2048 x 4096  9.4 / 8.6 / 8.4, 9.9 / 9.2 / 9.2, 9.2 / 9.2 / 9.2             40 x 2560 x 2048  10.1 / 9.5 / 9.6, 10.6 / 9.2 / 9.3, 9.2 / 9.2 / 9.2
  //   16 x 8192 x 4096  19.7 / 20.5 / 19.5, 19.8 / 20.0 / 19.8, 15.4 / 17.4 / 15.4    33 x 2304 x 3584  10.7 / 10.0 / 9.9, 11.3 / 11.3 / 11.3, 10.1 / 11.3 / 10.3
  // Queued with weights that are in the L2 already: level (40 x 4096 x 4096 10.7 / 10.8 / 10.7, 40 x 4096 x 1024 9.0 / 9.1 / 9.0).  Long shares: half as many blocks (16 x
  // 8192 x 4096, 64 blocks a share, 19.5 instead of 20.6, 16 x 6144 x 6144, 48 blocks, 18.4 / 18.6; 16 x 2048 x 8192, 32 blocks, 11.7 / 11.4).
  // Not where one kernel does it all: its successor's CTAs come too late for it to pay (48 x 960 x 3664 10.1 / 10.2, 69 x 3880 x 336 9.06 /
  // 9.13 with weights from memory, 10.2 / 10.4 and 9.0 / 9.1 from the L2).
  auto ask = [&](int kb) {
#pragma unroll
    for (int j = 0; j < 2 * NT; ++j)
      tma_prefetch_l2_3d(&tmW, p.b_nk ? kb * 64 : n0 + j * 64, p.b_nk ? n0 + j * 64 : kb * 64, b);
  };
  if (warp == 2 && p.wide && grp == 0 && elect_one()) {
#pragma unroll 1
    for (int kb = kb0; kb < kb1 && kb < kb0 + Cfg::ASK_FIRST; ++kb) ask(kb);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(s_tmem_base), Cfg::TMEM_COLS);
    tmem_relinquish_alloc_permit();
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  tcgen05_fence_after_sync();
  cluster_sync_after_init();  // every CTA's barriers exist and are armed before any peer signals them
  const uint32_t tmem_base = *s_tmem_base;
  // What stands above may overlap the previous kernel's tail: nothing there writes global memory or takes a value from it.  Each role waits for
  // itself (behind one wait for all 40 x 4096 x 1024 9.2 / 9.4 us, 100 x 2048 x 2048 9.3 / 9.5).

  if (warp == 0) {
    // ------------------------------------------------------------------------------------------ TMA producer
    griddep_wait();
    if (elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait<false>(bar_empty(stage), phase ^ 1u, w)) {  // passes on a fresh barrier
          *s_issued = kb - kb0;
          break;
        }
        const uint32_t sw = smem_base + stage * Cfg::STAGE_BYTES;
        mbar_arrive_expect_tx(bar_full(stage), Cfg::STAGE_BYTES);
#pragma unroll
        for (int j = 0; j < 2 * NT; ++j)
          tma_load_3d(sw + j * 8192, &tmW, bar_full(stage), p.b_nk ? kb * 64 : n0 + j * 64, p.b_nk ? n0 + j * 64 : kb * 64, b);
        tma_load_3d(sw + Cfg::W_BYTES, &tmX, bar_full(stage), kb * 64, m0, b);
        if (++stage == NSTAGES) { stage = 0; phase ^= 1u; }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------------------------------ UMMA issuer
    griddep_wait();
    if (elect_one()) {
      *s_begun = 1;
      int stage = 0;
      uint32_t phase = 0;
      // weights stored [N, K]: K-major, 16 elements = 32 bytes per step; stored [K, N]: MN-major (64-column blocks 8 KB
      // apart, 8 contraction rows 1 KB apart), 16 contraction rows = 2 KB per step
      const bool wkm = p.b_nk != 0;
      const uint64_t wlayout = wkm ? make_smem_desc_sw128(0, 16, 1024) : make_smem_desc_sw128(0, 8192, 1024);
      const uint32_t wstep = wkm ? 2u : 128u;
      const uint32_t idesc = wkm ? make_idesc_bf16(128, MT, false, false) : make_idesc_bf16(128, MT, true, false);
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait<false>(bar_full(stage), phase, w)) break;
        tcgen05_fence_after_sync();
        const uint32_t sw = smem_base + stage * Cfg::STAGE_BYTES;
        const uint64_t xdesc = make_smem_desc_sw128(sw + Cfg::W_BYTES, 16, 1024);
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          const uint64_t wdesc = wlayout + (((sw + t * 16384) & 0x3FFFFu) >> 4);
#pragma unroll
          for (int k = 0; k < 4; ++k)
            umma_bf16_ss(tmem_base + t * MT, wdesc + static_cast<uint64_t>(k * wstep), xdesc + static_cast<uint64_t>(k * 2), idesc,
                         (kb != kb0 || k != 0) ? 1u : 0u);
        }
        umma_commit(bar_empty(stage));
        if (++stage == NSTAGES) { stage = 0; phase ^= 1u; }
      }
      umma_commit(bar_acc);
      mbar_drain(bar_acc, 0, w);  // nothing may still be writing tensor memory when it is freed
    }
  } else {
    // ------------------------------------------------------------------------------------------ epilogue warps
    if (warp == 2) {
      if (p.wide && grp == 0 && elect_one()) {
        const int most = kb1 - kb0 <= 32 ? Cfg::ASK_MOST : Cfg::ASK_MOST / 2;
#pragma unroll 1
        for (int kb = kb0 + Cfg::ASK_FIRST; kb < kb1 && kb < kb0 + most && !*s_begun; ++kb) ask(kb);
      }
      __syncwarp();
    }
    griddep_wait();
    const int e = warp - 2;
    const int q = warp & 3;  // TMEM lane quarter: columns 32q .. 32q+31 of each 128-column tile
    const int h = e >> 2;    // which rows of the tile this warp moves from tensor memory to shared memory
    constexpr int MOVE = MT / 4 > 8 ? MT / 4 : 8;  // ... MOVE of them
    // row stage: lane = columns 4*lane .. 4*lane+3 of each tile, rows e, e + 16, ... of the slice
    uint2 bias[NT], gamma[NT], beta[NT];  // four bf16 each
    bool in[NT];
    int col[NT];
    const uint2 zero = make_uint2(0u, 0u), one = make_uint2(0x3F803F80u, 0x3F803F80u);
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      col[t] = n0 + t * 128 + 4 * lane;
      in[t] = col[t] < p.N;  // (N is a multiple of 8: a group of four is inside or outside)
      bias[t] = p.bias && in[t] ? __ldg(reinterpret_cast<const uint2*>(p.bias + col[t])) : zero;
      gamma[t] = p.gamma && in[t] ? __ldg(reinterpret_cast<const uint2*>(p.gamma + col[t])) : one;
      beta[t] = EPI == EPI_LN && p.beta && in[t] ? __ldg(reinterpret_cast<const uint2*>(p.beta + col[t])) : zero;
    }
    const int row0 = m0 + ks * rs;  // first row of the slice
    // asked for while the MainLoop runs: the rows' residual
    uint2 res[RC][NT];
#pragma unroll
    for (int i = 0; i < RC; ++i) {
      const int r = e + i * Cfg::kEpiWarps;
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        res[i][t] = zero;
        if (EPI == EPI_SOFTMAX && p.mask && r < rv && in[t])  // (the mask is the softmax kind's full-tensor operand)
          res[i][t] = __ldg(reinterpret_cast<const uint2*>(p.mask + static_cast<long long>(row0 + r) * p.N + col[t]));
        if (EPI != EPI_SOFTMAX && p.residual && r < rv && in[t])
          res[i][t] = __ldg(reinterpret_cast<const uint2*>(p.residual + static_cast<long long>(b) * p.batch_stride_r +
                                                           static_cast<long long>(row0 + r) * p.ldr + col[t]));
      }
    }
    // how many columns stand behind a lane's partial, and the weights of the pairwise merges (the two-kernel form counts the
    // zeros behind the end of the row: its finishing kernel expects the statistic of whole blocks)
    float mean_n = 0.f, wb[5], wm[5];
    if constexpr (EPI == EPI_LN) {
#pragma unroll
      for (int t = 0; t < NT; ++t) mean_n += (in[t] || p.wide) ? 4.f : 0.f;
      float n = mean_n;
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        const float nb2 = __shfl_xor_sync(0xFFFFFFFFu, n, 16 >> i);
        const float inv = n + nb2 > 0.f ? 1.f / (n + nb2) : 0.f;
        wb[i] = nb2 * inv;
        wm[i] = n * nb2 * inv;
        n += nb2;
      }
    }
    const float inv_mean_n = mean_n > 0.f ? 1.f / mean_n : 0.f;
    // stage 2's merge: LPR lanes per row, each with the partials of up to CPL column ranges
    constexpr int LPR = 32 / RC, CPL = 16 / LPR > 1 ? 16 / LPR : 1;
    const int mrow = lane / LPR, mlane = lane % LPR;
    float range_n[CPL];  // columns behind those partials
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
      const int c = mlane + k * LPR;
      const int left = p.N - c * COLS;
      range_n[k] = c >= p.ct ? 0.f : static_cast<float>(p.wide || left > COLS ? COLS : left);
    }
    const float n_all = p.wide ? static_cast<float>(p.ct * COLS) : static_cast<float>(p.N);
    const float inv_n_all = 1.f / n_all;
    const float alpha = p.alpha, eps = p.eps;
    const uint32_t stat_addr = smem_base + Cfg::OFF_STAT;
    const uint32_t max_addr = stat_addr + Cfg::STAT_BYTES;
    const int my_row = transposed_row<RC>(lane);  // which of the warp's RC rows a reduction leaves in this lane
    const bool gelu = EPI == EPI_RMS_MAX && !p.no_activation;

    mbar_wait<false>(bar_acc, 0, w);
    __syncwarp();
    tcgen05_fence_after_sync();
    // accumulators -> [row][column] in the ring, which nothing uses any more (every load has landed and has been multiplied)
    if (h * MOVE < MT) {
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        uint32_t v[MOVE];
        const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + t * MT + h * MOVE;
#pragma unroll
        for (int i = 0; i < MOVE; i += 8) tmem_ld_issue_8(taddr + i, v + i);
#pragma unroll
        for (int i = 0; i < MOVE; i += 8) tmem_ld_wait_8(v + i);
        const uint32_t dst = smem_base + static_cast<uint32_t>((h * MOVE * COLS + t * 128 + q * 32 + lane) * 4);
#pragma unroll
        for (int i = 0; i < MOVE; ++i)
          if (h * MOVE + i < rows) asm volatile("st.shared.b32 [%0], %1;" ::"r"(dst + i * Cfg::ROW_BYTES), "r"(v[i]) : "memory");
      }
    }
    if (p.ks > 1) {
      fence_proxy_async_smem();  // the bulk copies below read what these threads wrote
      named_barrier_sync(1, 32 * Cfg::kEpiWarps);
      if (e == 0 && lane < p.ks && lane != ks) {
        const uint32_t bytes = static_cast<uint32_t>(slice_rows(lane) * Cfg::ROW_BYTES);
        const uint32_t peer = static_cast<uint32_t>(ct * p.ks + lane);
        if (bytes)
          bulk_copy_to_peer(map_to_cta(smem_base + Cfg::OFF_RECV + ks * rs * Cfg::ROW_BYTES, peer),
                            smem_base + lane * rs * Cfg::ROW_BYTES, bytes, map_to_cta(bar_recv, peer));
      }
      __syncwarp();
      mbar_wait<true>(bar_recv, 0, w);
    } else {
      named_barrier_sync(1, 32 * Cfg::kEpiWarps);
    }

    // ---------------- stage 1: x = f(alpha*Acc + bias, R) in registers, and the rows' partial statistics.  The warp's RC rows
    // advance together (independent chains), and their reductions over the lanes are transposed: at every step a lane keeps
    // half of the rows, so that RC rows cost about as many shuffles as one.
    float x[RC][NT][4];
#pragma unroll
    for (int i = 0; i < RC; ++i)
#pragma unroll
      for (int t = 0; t < NT; ++t) x[i][t][0] = x[i][t][1] = x[i][t][2] = x[i][t][3] = 0.f;
    uint32_t row_off[RC];
#pragma unroll
    for (int i = 0; i < RC; ++i) {
      int r = e + i * Cfg::kEpiWarps;
      r = r < rv ? r : (rv > 0 ? rv - 1 : 0);  // (a row past the end repeats the last one; nothing of it is sent or stored)
      row_off[i] = static_cast<uint32_t>(r * Cfg::ROW_BYTES + lane * 16);
    }
    if (rv > 0)
      for (int s = 0; s < p.ks; ++s) {  // the shares' partial sums, in the same order whichever CTA finishes the row
        const uint32_t src = smem_base + (s == ks ? 0 : Cfg::OFF_RECV) + s * rs * Cfg::ROW_BYTES;
#pragma unroll
        for (int i = 0; i < RC; ++i)
#pragma unroll
          for (int t = 0; t < NT; ++t) {
            float o[4];
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                         : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3])
                         : "r"(src + row_off[i] + t * 512));
#pragma unroll
            for (int j = 0; j < 4; ++j) x[i][t][j] += o[j];
          }
      }
    constexpr float kLog2e = 1.4426950408889634f;
    float pa[RC], pb[RC];  // (mean, M2), (sum of squares, unused) or (maximum, sum of exponentials) of this lane's columns
    if constexpr (EPI == EPI_SOFTMAX) {
      // masked scores and the columns from N on are -inf; log2 e comes behind the difference from the maximum, so that no mask
      // value leaves the range of fp32
      const bool capped = p.softcap > 0.f;
      SoftcapLog2 cap_fn(alpha, capped ? p.softcap : 1.f);
      cap_fn.c1 = p.softcap;
#pragma unroll
      for (int i = 0; i < RC; ++i) {
        const int last = p.causal ? row0 + e + i * Cfg::kEpiWarps : p.N - 1;  // last live column of the row
        pa[i] = -INFINITY;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          float(&xx)[4] = x[i][t];
          const float2 m01 = bf16x2_to_f2(res[i][t].x), m23 = bf16x2_to_f2(res[i][t].y);
          const float mk[4] = {m01.x, m01.y, m23.x, m23.y};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            xx[j] = capped ? cap_fn(xx[j]) + mk[j] : fmaf(xx[j], alpha, mk[j]);
            if (!in[t] || col[t] + j > last) xx[j] = -INFINITY;
            pa[i] = fmaxf(pa[i], xx[j]);
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) pa[i] = fmaxf(pa[i], __shfl_xor_sync(0xFFFFFFFFu, pa[i], o));  // every lane needs it
      }
#pragma unroll
      for (int i = 0; i < RC; ++i) {
        const float m = pa[i] == -INFINITY ? 0.f : pa[i];  // (a row without a live column here: every exponential is 0)
        pb[i] = 0.f;
#pragma unroll
        for (int t = 0; t < NT; ++t)
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            x[i][t][j] = ex2_approx(kLog2e * (x[i][t][j] - m));
            pb[i] += x[i][t][j];
          }
      }
      transposed_reduce<RC>(pa, pb, lane, [&](int, float& a0, float& a1, float, float b1) { a1 += b1; });
    } else {
#pragma unroll
      for (int i = 0; i < RC; ++i) {
        pa[i] = pb[i] = 0.f;
#pragma unroll
        for (int t = 0; t < NT; ++t) {
          float(&xx)[4] = x[i][t];
          float2 z01 = fma2(splat2(alpha), make_float2(xx[0], xx[1]), bf16x2_to_f2(bias[t].x));
          float2 z23 = fma2(splat2(alpha), make_float2(xx[2], xx[3]), bf16x2_to_f2(bias[t].y));
          if (gelu) {
            z01 = gelu_tanh_f32x2(z01);
            z23 = gelu_tanh_f32x2(z23);
          }
          z01 = add2(z01, bf16x2_to_f2(res[i][t].x));
          z23 = add2(z23, bf16x2_to_f2(res[i][t].y));
          xx[0] = z01.x; xx[1] = z01.y; xx[2] = z23.x; xx[3] = z23.y;
          // (columns from N on hold exact zeros: operands outside the matrix read as zeros, bias and residual are masked)
          if constexpr (EPI == EPI_LN) {
            pa[i] += (xx[0] + xx[1]) + (xx[2] + xx[3]);
          } else {
            const float2 sq = fma2(z23, z23, mul2(z01, z01));
            pa[i] += sq.x + sq.y;
          }
        }
        if constexpr (EPI == EPI_LN) {
          pa[i] *= inv_mean_n;
#pragma unroll
          for (int t = 0; t < NT; ++t)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float d = in[t] || p.wide ? x[i][t][j] - pa[i] : 0.f;
              pb[i] = fmaf(d, d, pb[i]);
            }
        }
      }
      if constexpr (EPI == EPI_LN) {
        transposed_reduce<RC>(pa, pb, lane, [&](int step, float& a0, float& a1, float b0, float b1) {
          const float d = b0 - a0;
          a0 = fmaf(d, wb[step], a0);
          a1 = a1 + b1 + d * d * wm[step];
        });
      } else {
        transposed_reduce<RC>(pa, pb, lane, [&](int, float& a0, float&, float b0, float) { a0 += b0; });
      }
    }
    {
      // lanes that hold the same row may differ in the last bit: all of them send the first one's value
      const int first_lane = lane & (32 - 32 / RC);
      const float s0 = __shfl_sync(0xFFFFFFFFu, pa[0], first_lane);
      const float s1 = EPI != EPI_RMS_MAX ? __shfl_sync(0xFFFFFFFFu, pb[0], first_lane) : 0.f;
      const int r = e + my_row * Cfg::kEpiWarps;
#pragma unroll
      for (int k = 0; k < CPL; ++k) {
        const int c = (lane & (LPR - 1)) + k * LPR;
        const uint32_t peer = static_cast<uint32_t>(c * p.ks + ks);
        if (r < rv && c < p.ct)
          st_async_f32x2(map_to_cta(stat_addr + static_cast<uint32_t>((r * 16 + ct) * 8), peer), s0, s1, map_to_cta(bar_stat, peer));
      }
    }
    mbar_wait<true>(bar_stat, 0, w);
    __syncwarp();

    // ---------------- stage 2: merge the CT partials of the rows (the same order in every CTA), normalise, store
    float mu_l = 0.f, sq_l = 0.f;  // of row `mrow`
    {
      const int r = e + mrow * Cfg::kEpiWarps;
      float2 o[CPL];
#pragma unroll
      for (int k = 0; k < CPL; ++k) {
        o[k] = make_float2(0.f, 0.f);
        if (r < rv && mlane + k * LPR < p.ct) o[k] = s_stat[r * 16 + mlane + k * LPR];
      }
      if constexpr (EPI == EPI_LN) {
#pragma unroll
        for (int k = 0; k < CPL; ++k) mu_l = fmaf(range_n[k], o[k].x, mu_l);
#pragma unroll
        for (int d = LPR / 2; d > 0; d >>= 1) mu_l += __shfl_xor_sync(0xFFFFFFFFu, mu_l, d);
        mu_l *= inv_n_all;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
          const float d = o[k].x - mu_l;
          sq_l += fmaf(range_n[k] * d, d, o[k].y);
        }
      } else if constexpr (EPI == EPI_SOFTMAX) {
        float m = -INFINITY;
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
          if (mlane + k * LPR >= p.ct || r >= rv) o[k].x = -INFINITY;
          m = fmaxf(m, o[k].x);
        }
#pragma unroll
        for (int d = LPR / 2; d > 0; d >>= 1) m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, d));
#pragma unroll
        for (int k = 0; k < CPL; ++k) sq_l += o[k].y * (o[k].x == -INFINITY ? 0.f : ex2_approx(kLog2e * (o[k].x - m)));  // (a NaN stays one)
        const float own = r < rv ? s_stat[r * 16 + ct].x : -INFINITY;  // this CTA's exponentials are relative to its own maximum
        mu_l = own == -INFINITY ? 0.f : ex2_approx(kLog2e * (own - m));
      } else {
#pragma unroll
        for (int k = 0; k < CPL; ++k) sq_l += o[k].x;
      }
#pragma unroll
      for (int d = LPR / 2; d > 0; d >>= 1) sq_l += __shfl_xor_sync(0xFFFFFFFFu, sq_l, d);
      const int grow = row0 + r;
      if (p.wide && ct == 0 && mlane == 0 && r < rv && COMFUSE_IN_BOUNDS(grow < p.M && nb < p.nblocks && b < p.batch, p.status))
        p.wide_partials[(static_cast<long long>(b) * p.M + grow) * p.nblocks + nb] = make_float2(EPI == EPI_LN ? mu_l : sq_l, EPI == EPI_LN ? sq_l : 0.f);
    }
    // factor of the row: 1 / standard deviation, or what turns this CTA's exponentials into probabilities (a row without a live
    // column is all zero, a row with a NaN all NaN)
    const float rstd_l = EPI == EPI_SOFTMAX ? (sq_l == 0.f ? 0.f : mu_l / sq_l) : rsqrtf(sq_l * inv_n_all + eps);
    const float shift_l = -mu_l * rstd_l;
    float rstd[RC], shift[RC], best[RC], best_col[RC];
#pragma unroll
    for (int i = 0; i < RC; ++i) {
      rstd[i] = __shfl_sync(0xFFFFFFFFu, rstd_l, i * LPR);
      shift[i] = EPI == EPI_LN ? __shfl_sync(0xFFFFFFFFu, shift_l, i * LPR) : 0.f;
    }
    uint16_t* yrow = p.Y + static_cast<long long>(b) * p.batch_stride_y + static_cast<long long>(row0 + e) * p.ldy;
    const long long ystep = p.ldy * Cfg::kEpiWarps;
#pragma unroll
    for (int i = 0; i < RC; ++i) {
      const bool row_ok = e + i * Cfg::kEpiWarps < rv;
      float bv = -INFINITY;
      int bc = 0x7FFFFFFF;
#pragma unroll
      for (int t = 0; t < NT; ++t) {
        const float(&xx)[4] = x[i][t];
        uint2 out;
        if (p.wide) {  // the row is finished by the second kernel
          out = make_uint2(pack_f16x2_rn(xx[0], xx[1]), pack_f16x2_rn(xx[2], xx[3]));
        } else {
          const float2 g01 = bf16x2_to_f2(gamma[t].x), g23 = bf16x2_to_f2(gamma[t].y);
          const float2 b01 = bf16x2_to_f2(beta[t].x), b23 = bf16x2_to_f2(beta[t].y);
          const float gm[4] = {g01.x, g01.y, g23.x, g23.y}, be[4] = {b01.x, b01.y, b23.x, b23.y};
          float y[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if constexpr (EPI == EPI_LN) {
              y[j] = fmaf(fmaf(xx[j], rstd[i], shift[i]), gm[j], be[j]);
              if (p.post_relu) y[j] = fmaxf(y[j], 0.f);
            } else if constexpr (EPI == EPI_SOFTMAX) {
              y[j] = xx[j] * rstd[i];
            } else {
              y[j] = xx[j] * rstd[i] * gm[j];
              if (in[t] && y[j] > bv) { bv = y[j]; bc = col[t] + j; }
            }
          }
          out = make_uint2(pack_bf16x2_rn(y[0], y[1]), pack_bf16x2_rn(y[2], y[3]));
        }
        if (row_ok && in[t] && COMFUSE_IN_BOUNDS(row0 + e + i * Cfg::kEpiWarps < p.M && col[t] + 3 < p.N, p.status))
          *reinterpret_cast<uint2*>(yrow + col[t]) = out;
      }
      yrow += ystep;
      best[i] = bv;
      best_col[i] = __int_as_float(bc);
    }
    if (EPI == EPI_RMS_MAX && !p.wide) {
      // ---------------- stage 3: the chained reduction, row maximum and its lowest column, finished by column range 0
      transposed_reduce<RC>(best, best_col, lane, [&](int, float& a0, float& a1, float b0, float b1) {
        const float2 m = MergeArgmax()(make_float2(a0, a1), 0.f, make_float2(b0, b1), 0.f);
        a0 = m.x;
        a1 = m.y;
      });
      const int rm = e + my_row * Cfg::kEpiWarps;
      if ((lane & (LPR - 1)) == 0 && rm < rv) {
        const uint32_t peer = static_cast<uint32_t>(ks);
        st_async_f32x2(map_to_cta(max_addr + static_cast<uint32_t>((rm * 16 + ct) * 8), peer), best[0], best_col[0], map_to_cta(bar_max, peer));
      }
      if (ct == 0) {
        mbar_wait<true>(bar_max, 0, w);
        __syncwarp();
        const float2* s_max = s_stat + Cfg::STAT_BYTES / 8;
        const int r = e + mrow * Cfg::kEpiWarps;
        float2 m = make_float2(-INFINITY, __int_as_float(0x7FFFFFFF));
#pragma unroll
        for (int k = 0; k < CPL; ++k)
          if (r < rv && mlane + k * LPR < p.ct) m = MergeArgmax()(m, 0.f, s_max[r * 16 + mlane + k * LPR], 0.f);
#pragma unroll
        for (int d = LPR / 2; d > 0; d >>= 1)
          m = MergeArgmax()(m, 0.f, make_float2(__shfl_xor_sync(0xFFFFFFFFu, m.x, d), __shfl_xor_sync(0xFFFFFFFFu, m.y, d)), 0.f);
        const long long o = static_cast<long long>(b) * p.M + row0 + r;
        if (mlane == 0 && r < rv && COMFUSE_IN_BOUNDS(o < static_cast<long long>(p.batch) * p.M, p.status)) {
          p.row_max[o] = m.x;
          p.row_argmax[o] = __float_as_int(m.y);
        }
      }
    }
  }

  // -------------------------------------------------------------------------------------------- teardown
  tcgen05_fence_before_sync();
  __syncthreads();
  if (threadIdx.x == 0 && *s_abort) tell_cluster(s_told, static_cast<uint32_t>(p.ct * p.ks));
  // No CTA may leave while a peer still sends into its shared memory.  Everything that is sent here has been waited for by
  // its receiver, and a bulk copy's source has been read when its destination counts it: arriving is all that is needed, no
  // flush of this CTA's stores (the release form waited 1000 clocks for the result's stores to reach the L2).
  cluster_sync_after_init();
  if (warp == 1) {
    __syncwarp();
    tcgen05_fence_after_sync();
    tmem_dealloc(tmem_base, Cfg::TMEM_COLS);
  }
  // Unless a wait expired: then loads and the peers' sends, which are issued whatever expired, may still be under way.  (One warp
  // looks, and meets the other CTAs' once more; the others leave at once.  40 x 4096 x 4096 13.35 -> 13.39 us; with every thread
  // looking, and the outcomes of its waits carried along, 13.50.)
  if (warp == 0 && *s_told) {
    if (lane == 0) {
      const int issued = *s_issued;
      for (int u = issued > NSTAGES ? issued - NSTAGES : 0; u < issued; ++u) mbar_drain(bar_full(u % NSTAGES), (u / NSTAGES) & 1u, w);
      mbar_drain(bar_recv, 0, w);
      mbar_drain(bar_stat, 0, w);
      if (EPI == EPI_RMS_MAX && !p.wide) mbar_drain(bar_max, 0, w);
    }
    __syncwarp();
    cluster_sync_all();
  }
}

template <int EPI, int NT, int MT>
cudaError_t launch_instance(const FewRowsPlan& plan, const CUtensorMap& tmW, const CUtensorMap& tmX, const FewRowsParams& p, cudaStream_t stream) {
  using Cfg = FewRowsCfg<NT, MT>;
  auto kern = few_rows_kernel<EPI, NT, MT>;
  const DeviceInfo* dev = current_device_info();
  if (!dev) return cudaErrorInvalidDevice;
  constexpr int kMaxDev = 64;
  static std::atomic<bool> ready[kMaxDev];  // set (released) once the kernel's attributes are in place on that device
  const int di = dev->device < kMaxDev ? dev->device : kMaxDev - 1;
  if (!ready[di].load(std::memory_order_acquire)) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    ready[di].store(true, std::memory_order_release);
  }
  const int cluster = plan.ct * plan.ks;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  cfg.gridDim = dim3(static_cast<unsigned>(p.batch * p.groups * p.nblocks * cluster), 1, 1);
  cfg.blockDim = dim3(Cfg::kThreads, 1, 1);
  cfg.dynamicSmemBytes = Cfg::SMEM_BYTES;
  cfg.stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(cluster);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // set-up may overlap the previous kernel's tail
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = programmatic_launch_enabled() ? 2 : 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, kern, tmW, tmX, p);
}

// Clusters of `size` CTAs of this kernel that are resident at once; every instantiation puts one CTA on an SM, so one of them
// answers for all.
int resident_clusters(int size, const DeviceInfo& dev) {
  static ResidentClusters cache;
  using Cfg = FewRowsCfg<1, 64>;
  return cache.of(reinterpret_cast<const void*>(&few_rows_kernel<EPI_LN, 1, 64>), Cfg::kThreads, Cfg::SMEM_BYTES, size, dev);
}

}  // namespace

FewRowsPlan few_rows_plan(int epi, int batch, int M, int N, int K, int wide_block, long long ld_rows, long long ld_weights, bool b_nk, const DeviceInfo& dev) {
  FewRowsPlan none, c;
  if (epi != EPI_LN && epi != EPI_RMS_MAX && epi != EPI_SOFTMAX) return none;
  if (N > kWideRowBlock && (wide_block != 256 || epi == EPI_SOFTMAX)) return none;
  // Rows of 2048 columns and more behind a long contraction keep the two-kernel form: 256-column blocks spread the weights
  // over the machine, a row's own cluster reaches 16 SMs (40 x 4096 x 4096: 12.8 us against 37).
  c.wide = wide_block == 256 && (N > kWideRowBlock || (N >= 2048 && K >= 1024));
  c.mt = M <= 16 ? 16 : M <= 32 ? 32 : 64;
  const int KB = (K + 63) / 64;
  const long long groups = (static_cast<long long>(M) + c.mt - 1) / c.mt;
  c.nblocks = c.wide ? (N + 255) / 256 : 1;
  const long long clusters = batch * groups * c.nblocks;
  // This form is taken where all its clusters are resident at once.  Measured there (tile kernel / this one, us; LayerNorm,
  // weights [N, K]): 128 x 256 x 256 7.7 / 4.6, 128 x 1024 x 1024 19.0 / 6.1, 512 x 768 x 768 13.4 / 5.7, 512 x 1024 x 2048
  // 17.8 / 9.2, 1024 x 512 x 1024 18.8 / 6.5, 4096 x 256 x 1024 11.6 / 7.4.  With a second round of clusters the two are level
  // or the tile kernel is ahead (1024 x 1024 x 64 10.8 / 9.3, 2048 x 768 x 64 8.9 / 9.4, 2048 x 1024 x 1024 19.4 / 20.9).
  // Softmax kind, one round (row or cluster kernel / this one, K = 64): 8 x 64 x 512 11.0 / 4.4, 2 x 1024 x 1024 12.7 / 6.7,
  // 140 x 64 x 128 11.6 / 5.4; two rounds: 16 x 512 x 512 causal 10.6 / 12.8, 2 x 1171 x 1176 masked 11.4 / 12.5.
  // Two tiles per CTA halve the CTAs where one does not fit: 3000 x 512 x 768 16.3 / 10.1, 2000 x 768 x 1536 18.7 / 14.1, 2306 x 512 x
  // 4096 28.7 / 23.4 (where such calls end: l2_bound).  Not for normalised rows of up to 256 columns, which the tile kernel holds in one CTA pair (5923 x 256 x 256
  // 7.9 / 7.8, x 1536 14.1 / 15.7).
  // Every row group reads the weights anew, twice as often as the tile kernel's 256-row pairs, and with most of the machine at it the
  // L2 is what bounds the call (8.5 - 9.5 TB/s).  A box row of 128 bytes that does not start on a 128-byte line touches two of them.
  // Measured (tile kernel / this one, us; LayerNorm):
  //   two tiles per CTA, weight rows off their lines, the tile kernel's two-kernel form available: 3520 x 512 x 1032 level, x 2056
  //   21.9 / 24.0, x 3592 31.1 / 41.7, 2368 x 512 x 2056 21.4 / 22.0; rows of 513 .. 768 columns, which the tile kernel is best at, on
  //   more than three quarters of the SMs: 2880 x 768 x 520 level, x 1032 17.1 / 17.7, x 4088 40.3 / 41.4, 2880 x 520 x 1032 16.5 /
  //   17.7, but 2112 x 768 x 1032 16.8 / 15.1, x 4088 39.4 / 37.0;
  //   weight rows on their lines: 3520 x 512 x 4096 27.9 / 27.5, x 5128 32.7 / 34.7; with the activations' rows on theirs too 2306 x
  //   512 x 6144 38.1 / 33.2, 2800 x 512 x 8192 47.9 / 52.2; one kernel: 1500 x 768 x 8192 64.2 / 42.9.
  //   one tile, narrow weights [K, N] on more than half of the SMs: 7104 x 24 x 3080 27.5 / 28.6, x 8184 56.5 / 69.1; 5200 x 8 x 1024 14.9 /
  //   17.0, x 2048 19.4 / 20.0.
  auto l2_bound = [&](const FewRowsPlan& q, long long n) {
    const long long ctas = n * q.ct;
    if (q.nt == 1) return !q.wide && N < 64 && !b_nk && K > (N < 16 ? 768 : 2560) && ctas > dev.sm_count / 2;
    const bool weights_on_lines = ld_weights % 64 == 0, rows_on_lines = ld_rows % 64 == 0;
    if (!weights_on_lines && N > 512 && N <= 768 && K > 768 && ctas > 3 * dev.sm_count / 4) return true;
    return wide_block == 256 && K > (!weights_on_lines ? 1536 : rows_on_lines ? 6144 : 4096);
  };
  for (c.nt = 1; c.nt <= (N <= 256 && epi != EPI_SOFTMAX ? 1 : 2); ++c.nt) {
    c.ct = c.wide ? 2 : (N + 128 * c.nt - 1) / (128 * c.nt);
    if (c.ct > 16 || clusters > resident_clusters(c.ct, dev)) {
      if (c.wide) return none;
      continue;
    }
    if (epi != EPI_SOFTMAX && l2_bound(c, clusters)) return none;
    // Splitting the contraction pays from 12 K blocks on (one exchange costs about as much as four blocks): 128 x 512 x 1024
    // 6.3 / 5.8 / 6.2 us with 1 / 2 / 4 shares, x 2048 8.4 / 6.9 / 6.9, x 256 4.7 / 4.8 / 5.7.  A third of the SMs is left
    // to the next call's set-up (2048 x 256 x 1024: 6.5 us with 64 CTAs, 7.2 with 128).
    const long long most = 2ll * dev.sm_count / 3;
    c.ks = KB >= 64 ? 8 : KB >= 28 ? 4 : KB >= 12 ? 2 : 1;
    while (c.ks > 1 && (c.ct * c.ks > 16 || clusters * c.ct * c.ks > most || clusters > resident_clusters(c.ct * c.ks, dev))) --c.ks;
    return c;
  }
  return none;
}

cudaError_t launch_few_rows(int epi, const FewRowsPlan& plan, const CUtensorMap& tmW, const CUtensorMap& tmX, FewRowsParams p,
                            cudaStream_t stream) {
  p.ct = plan.ct;
  p.ks = plan.ks;
  p.nblocks = plan.nblocks;
  p.groups = (p.M + plan.mt - 1) / plan.mt;
#define COMFUSE_CASE(NT, MT)                                                                                     \
  if (plan.nt == NT && plan.mt == MT)                                                                            \
    return epi == EPI_LN        ? launch_instance<EPI_LN, NT, MT>(plan, tmW, tmX, p, stream)                     \
           : epi == EPI_SOFTMAX ? launch_instance<EPI_SOFTMAX, NT, MT>(plan, tmW, tmX, p, stream)                \
                                : launch_instance<EPI_RMS_MAX, NT, MT>(plan, tmW, tmX, p, stream);
  COMFUSE_CASE(1, 16)
  COMFUSE_CASE(1, 32)
  COMFUSE_CASE(1, 64)
  COMFUSE_CASE(2, 16)
  COMFUSE_CASE(2, 32)
  COMFUSE_CASE(2, 64)
#undef COMFUSE_CASE
  return cudaErrorInvalidValue;
}

}  // namespace comfuse
