// Attention form of the back-to-back GEMM for short sources and few queries (Sec. 4 with a row softmax as F):
// P = alpha X W1,  S = exp(P - rowmax),  O = (S W2) / rowsum, per batch.  Neither P nor S is written to global memory.
// (b2b_gemm.cu holds the form for longer sources, and the rule that chooses.)
//
// What bounds it: the chain scores -> row maximum -> exponentials -> S.V of one row tile, which leaves the tensor core and
// the MUFU unit (128 x 128 exponentials are 1024 clocks of it) waiting for one another.  Source positions come in blocks of 128,
// query rows in tiles of 128, and a CTA's work item is one of two things:
//
//   up to 128 positions    TWO tiles that share the one block of keys and values, in alternation: while one tile's warps
//                          exponentiate, the tensor core computes the other tile's scores and S.V  (tile B's warps idle where the
//                          second 128 rows do not exist, or where every tile has a CTA of its own)
//   up to 128 queries      ONE tile, walking the source's blocks  (tile A; tile B's warps idle)
//
//   tensor memory    scores of tile A (128 columns), of tile B (128), output of A (128), of B (128)
//   S                bf16, written over the first half of the tile's own score columns: S.V takes it from tensor memory as its
//                    A operand, so S crosses no shared memory
//   softmax warps    four per tile, a thread per row: the row maximum and the row sum need no exchange.  A block's
//                    exponentials are taken against the block's own maximum (its largest weight is then exactly 1 in bf16)
//   finish warps     rescale the output so far to each further block's maximum while that block is exponentiated; divide by
//                    the row sum and store
//   UMMA lane        S.V of block j, then the scores of block j + 1 into the columns that S just left, for A, then for B;
//                    the blocks of consecutive work items form one sequence
//
// Measured (device time, CTA-pair form of b2b_gemm.cu / this one): 109 x 1116 queries of 32 keys 28.0 / 16.8 us, 4 x 23 of 64
// 6.8 / 4.7, 83 x 35 of 320 13.9 / 9.0.  Two tiles over several blocks (longer sources of more queries) were built too and
// stay with the pair form, 32 x 4096 of 256 22.3 / 22.8 and 256 x 512 of 512 38.7 / 40.0: a block of a tile took 3200 clocks there
// (scores read 150, row maximum 320, exponentials 1550, S.V and the next scores 1000), and the score UMMAs of single CTAs
// read both operands from shared memory at its full rate, where a pair halves one of them.
#include <cuda_runtime.h>

#include <atomic>

#include "b2b_params.h"
#include "epilogue_common.cuh"
#include "host_common.h"
#include "sm100_primitives.cuh"

namespace comfuse {

namespace {

// warp 0 producer, warp 1 UMMA issuer; warps 4-7 softmax of tile A, 8-11 of tile B, 12-15 normalise and store (a warp reads the
// tensor-memory lanes 32 (warp mod 4) ..)
constexpr int kFirstSoftmaxWarp = 4, kFirstFinishWarp = 12;
constexpr int kAttnThreads = 32 * 16;
// Registers per thread of the four warpgroups: 512 threads are launched with 128 each, and the softmax threads, which hold a row's
// 128 scores, take what the others leave.
constexpr int kRegsIssue = 88, kRegsSoftmax = 160, kRegsFinish = 104;
static_assert(kRegsIssue + 2 * kRegsSoftmax + kRegsFinish == 4 * 128, "the shares add up to what the block was launched with");
constexpr int kBoxBytes = 128 * 64 * 2;  // one 128 x 64 bf16 box
constexpr int kBlockBytes = 2 * kBoxBytes;
constexpr int kKvSlots = 4;
constexpr float kKeepLog2 = 8.f;  // how far (log2) a block's maximum may lie below the reference before the reference is kept

struct AttnSmem {
  static constexpr int OFF_Q = 0;                                 // two tiles of 128 queries
  static constexpr int OFF_KV = OFF_Q + 2 * kBlockBytes;          // ring of key and value blocks
  static constexpr int OFF_OUT = OFF_KV + kKvSlots * kBlockBytes; // two 32 x 64 output boxes per finish warp
  static constexpr int OFF_BAR = OFF_OUT + 8 * 4096;
  static constexpr int NUM_BARS = 2 * kKvSlots + 9 * 2 + 1;
  static constexpr int OFF_MISC = OFF_BAR + NUM_BARS * 8;
  static constexpr int OFF_SUM = OFF_MISC + 16;                   // float [2 tiles][128]: rescaling factors, then row sums
  static constexpr int BYTES = OFF_SUM + 2 * 128 * 4 + 1024;
};
static_assert(AttnSmem::BYTES <= 232448, "shared memory budget");

// D[tmem] (+)= A[tmem] * B[smem desc]: the A operand as packed bf16 pairs, one row per lane
__device__ __forceinline__ void umma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// KM: the keys (W1) are stored [batch, N1, K], one key per row (a K-major operand), else [batch, K, N1] (MN-major).
template <bool KM>
__global__ void __launch_bounds__(kAttnThreads, 1)
b2b_attention_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW1,
                     const __grid_constant__ CUtensorMap tmW2, const __grid_constant__ CUtensorMap tmO, const B2bParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  const uint32_t smem_base = smem_u32(smem);

  const uint32_t bar_base = smem_base + AttnSmem::OFF_BAR;
  auto bar_kvfull = [&](int s) { return bar_base + 8u * s; };
  auto bar_kvempty = [&](int s) { return bar_base + 8u * (kKvSlots + s); };
  const uint32_t bar_tile = bar_base + 8u * (2 * kKvSlots);
  auto bar_qfull = [&](int t) { return bar_tile + 8u * t; };
  auto bar_qempty = [&](int t) { return bar_tile + 8u * (2 + t); };
  auto bar_sfull = [&](int t) { return bar_tile + 8u * (4 + t); };   // scores of a block complete
  auto bar_pfull = [&](int t, int half) { return bar_tile + 8u * (12 + 2 * t + half); };  // half of S written (and the scores read)
  auto bar_lfull = [&](int t) { return bar_tile + 8u * (6 + t); };   // row sums of the work item written
  auto bar_ofull = [&](int t) { return bar_tile + 8u * (8 + t); };   // output of the work item complete
  auto bar_oempty = [&](int t) { return bar_tile + 8u * (10 + t); }; // output read
  const uint32_t bar_ffull = bar_tile + 8u * 16;  // (tile A) rescaling factors of a block written
  const uint32_t bar_fdone = bar_tile + 8u * 17;  // (tile A) output rescaled
  const uint32_t bar_drain = bar_tile + 8u * 18;
  float* s_sum = reinterpret_cast<float*>(smem + AttnSmem::OFF_SUM);
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(smem + AttnSmem::OFF_MISC);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + AttnSmem::OFF_MISC + 4);
  volatile uint32_t* s_issued = reinterpret_cast<volatile uint32_t*>(smem + AttnSmem::OFF_MISC + 8);  // key / value blocks, query tiles: loads issued

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int nblk = (p.N1 + 127) >> 7;  // blocks of 128 source positions
  const int total = p.batch * p.mpairs;
  const int my_items = static_cast<int>(blockIdx.x) < total ? (total - static_cast<int>(blockIdx.x) + static_cast<int>(gridDim.x) - 1) / static_cast<int>(gridDim.x) : 0;
  const WaitCtx w{s_abort, p.status, p.timeout_ns};
  // Walks this CTA's work items (blockIdx.x, + gridDim.x, ...): batch and first row of tile A; tile B, the next 128 rows, may
  // lie past the end.  The divisions are done once.
  struct ItemWalk {
    int bz, mi, dbz, dmi, per, rows;
    __device__ __forceinline__ ItemWalk(const B2bParams& p) : per(p.mpairs), rows(p.item_rows) {
      bz = static_cast<int>(blockIdx.x) / per;
      mi = static_cast<int>(blockIdx.x) - bz * per;
      dbz = static_cast<int>(gridDim.x) / per;
      dmi = static_cast<int>(gridDim.x) - dbz * per;
    }
    __device__ __forceinline__ void next() {
      bz += dbz;
      mi += dmi;
      if (mi >= per) { mi -= per; ++bz; }
    }
    __device__ __forceinline__ int m0() const { return mi * rows; }
    __device__ __forceinline__ bool has_b(int M) const { return rows == 256 && m0() + 128 < M; }
  };
  griddep_launch_dependents();  // the next kernel's set-up may overlap this kernel (it waits before touching memory)

  if (threadIdx.x == 0) {
    for (int s = 0; s < kKvSlots; ++s) {
      mbar_init(bar_kvfull(s), 1);
      mbar_init(bar_kvempty(s), 1);
    }
    for (int t = 0; t < 2; ++t) {
      mbar_init(bar_qfull(t), 1);
      mbar_init(bar_qempty(t), 1);
      mbar_init(bar_sfull(t), 1);
      mbar_init(bar_pfull(t, 0), 4);  // one arrival per softmax warp of the tile
      mbar_init(bar_pfull(t, 1), 4);
      mbar_init(bar_lfull(t), 4);
      mbar_init(bar_ofull(t), 1);
      mbar_init(bar_oempty(t), 4);
    }
    mbar_init(bar_ffull, 4);
    mbar_init(bar_fdone, 4);
    mbar_init(bar_drain, 1);
    *s_abort = 0;
    fence_mbar_init();
    prefetch_tensormap(&tmX);
    prefetch_tensormap(&tmW1);
    prefetch_tensormap(&tmW2);
    prefetch_tensormap(&tmO);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(s_tmem_base), 512);
    tmem_relinquish_alloc_permit();
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  tcgen05_fence_after_sync();
  const uint32_t tmem_base = *s_tmem_base;
  griddep_wait();  // the set-up above may overlap the previous kernel's tail; global memory is touched only below

  if (warp < kFirstSoftmaxWarp) {
    setmaxnreg_dec<kRegsIssue>();
    if (warp == 0) {
      // ------------------------------------------------------------------------------------------ TMA producer
      if (elect_one()) {
        int slot = 0;
        uint32_t phase = 0, quse[2] = {0, 0}, blocks = 0;
        bool ok = true;
        auto next_slot = [&](uint32_t& dst, uint32_t& full) {
          if (!ok || !mbar_wait<false>(bar_kvempty(slot), phase ^ 1u, w)) { ok = false; return false; }  // passes on a fresh barrier
          dst = smem_base + AttnSmem::OFF_KV + slot * kBlockBytes;
          full = bar_kvfull(slot);
          mbar_arrive_expect_tx(full, kBlockBytes);
          if (++slot == kKvSlots) { slot = 0; phase ^= 1u; }
          ++blocks;
          return true;
        };
        ItemWalk it(p);
        for (int i = 0; i < my_items && ok; ++i, it.next()) {
          const int bz = it.bz, m0 = it.m0();
          auto load_q = [&](int t) {
            if (!ok || !mbar_wait<false>(bar_qempty(t), (quse[t] & 1u) ^ 1u, w)) { ok = false; return; }
            ++quse[t];
            const uint32_t dst = smem_base + AttnSmem::OFF_Q + t * kBlockBytes;
            mbar_arrive_expect_tx(bar_qfull(t), kBlockBytes);
            tma_load_3d(dst, &tmX, bar_qfull(t), 0, m0 + t * 128, bz);
            tma_load_3d(dst + kBoxBytes, &tmX, bar_qfull(t), 64, m0 + t * 128, bz);
          };
          load_q(0);
          for (int j = 0; j < nblk && ok; ++j) {
            uint32_t dst, full;
            if (!next_slot(dst, full)) break;
            if constexpr (KM) {  // 128 keys x 64 elements, twice
              tma_load_3d(dst, &tmW1, full, 0, j * 128, bz);
              tma_load_3d(dst + kBoxBytes, &tmW1, full, 64, j * 128, bz);
            } else {             // 64 keys x 128 contraction rows, twice
              tma_load_3d(dst, &tmW1, full, j * 128, 0, bz);
              tma_load_3d(dst + kBoxBytes, &tmW1, full, j * 128 + 64, 0, bz);
            }
            if (j == 0 && it.has_b(p.M)) load_q(1);  // behind what tile A's first scores need
            if (!next_slot(dst, full)) break;
            tma_load_3d(dst, &tmW2, full, 0, j * 128, bz);
            tma_load_3d(dst + kBoxBytes, &tmW2, full, 64, j * 128, bz);
          }
        }
        s_issued[0] = blocks;
        s_issued[1] = (quse[0] ? 2u - (quse[0] & 1u) : 0u) | (quse[1] ? 2u - (quse[1] & 1u) : 0u) << 8;  // (none, or a count of the same parity)
      }
    } else if (warp == 1) {
      // ------------------------------------------------------------------------------------------ UMMA issuer
      if (elect_one()) {
        constexpr uint32_t idesc_qk = make_idesc_bf16(128, 128, false, !KM);
        constexpr uint32_t idesc_pv = make_idesc_bf16(128, 128, false, true);
        int slot = 0;
        uint32_t phase = 0, quse[2] = {0, 0}, puse[2] = {0, 0}, ouse[2] = {0, 0}, fuse = 0;
        bool ok = true;
        // the next slot of the ring, landed; it is handed back (commit) when its last UMMAs have been issued
        auto take_slot = [&](uint32_t& addr) {
          const int s = slot;
          if (!ok || !mbar_wait<false>(bar_kvfull(s), phase, w)) { ok = false; return s; }
          tcgen05_fence_after_sync();
          addr = smem_base + AttnSmem::OFF_KV + s * kBlockBytes;
          if (++slot == kKvSlots) { slot = 0; phase ^= 1u; }
          return s;
        };
        auto scores = [&](int t, int j, uint32_t ka) {  // P = Q . K of block j
          if (j == 0) {
            if (!ok || !mbar_wait<false>(bar_qfull(t), quse[t] & 1u, w)) { ok = false; return; }
            ++quse[t];
            tcgen05_fence_after_sync();
          }
          const uint32_t qa = smem_base + AttnSmem::OFF_Q + t * kBlockBytes;
          const uint64_t q0 = make_smem_desc_sw128(qa, 16, 1024), q1 = make_smem_desc_sw128(qa + kBoxBytes, 16, 1024);
          const uint64_t k0 = KM ? make_smem_desc_sw128(ka, 16, 1024) : make_smem_desc_sw128(ka, /*next 64 keys*/ kBoxBytes, /*next 8 rows*/ 1024);
          const uint64_t k1 = make_smem_desc_sw128(ka + kBoxBytes, 16, 1024);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            umma_bf16_ss(tmem_base + t * 128, (kk < 4 ? q0 : q1) + static_cast<uint64_t>((kk & 3) * 2),
                         KM ? (kk < 4 ? k0 : k1) + static_cast<uint64_t>((kk & 3) * 2) : k0 + static_cast<uint64_t>(kk * 128), idesc_qk, kk != 0 ? 1u : 0u);
          umma_commit(bar_sfull(t));
          if (j == nblk - 1) umma_commit(bar_qempty(t));
        };
        auto weighted_sum = [&](int t, int j, uint32_t va) {  // O (+)= S . V of block j
          if (j == 0) {
            if (!ok || !mbar_wait<false>(bar_oempty(t), (ouse[t] & 1u) ^ 1u, w)) { ok = false; return; }
            ++ouse[t];
          } else {  // (tile A: items of several blocks have no tile B)
            if (!ok || !mbar_wait<false>(bar_fdone, fuse & 1u, w)) { ok = false; return; }
            ++fuse;
          }
          const uint64_t vd = make_smem_desc_sw128(va, /*next 64 columns*/ kBoxBytes, /*next 8 positions*/ 1024);
#pragma unroll
          for (int half = 0; half < 2; ++half) {  // the first half runs under the second half's exponentials
            if (!ok || !mbar_wait<false>(bar_pfull(t, half), puse[t] & 1u, w)) { ok = false; return; }
            tcgen05_fence_after_sync();
#pragma unroll
            for (int kk = 4 * half; kk < 4 * half + 4; ++kk)
              umma_bf16_ts(tmem_base + 256 + t * 128, tmem_base + t * 128 + kk * 8, vd + static_cast<uint64_t>(kk * 128), idesc_pv, (j | kk) != 0 ? 1u : 0u);
          }
          ++puse[t];
          if (j == nblk - 1) umma_commit(bar_ofull(t));
        };
        uint32_t ka = 0, va = 0;
        ItemWalk it(p);
        bool b_now = it.has_b(p.M);
        if (my_items > 0) {
          const int ks = take_slot(ka);
          if (ok) scores(0, 0, ka);
          if (ok && b_now) scores(1, 0, ka);
          if (ok) umma_commit(bar_kvempty(ks));
        }
        for (int i = 0, j = 0; i < my_items && ok;) {
          const int ni = j + 1 < nblk ? i : i + 1, nj = j + 1 < nblk ? j + 1 : 0;
          const bool more = ni < my_items;
          if (ni != i) it.next();
          const bool b_next = ni == i ? b_now : it.has_b(p.M);
          const int vs = take_slot(va);
          int ks = 0;
          if (ok) weighted_sum(0, j, va);
          if (ok && more) {
            ks = take_slot(ka);
            if (ok) scores(0, nj, ka);
          }
          if (ok && b_now) weighted_sum(1, j, va);
          if (ok && more && b_next) scores(1, nj, ka);
          if (ok) umma_commit(bar_kvempty(vs));
          if (ok && more) umma_commit(bar_kvempty(ks));
          i = ni;
          j = nj;
          b_now = b_next;
        }
        umma_commit(bar_drain);  // nothing may still be writing tensor memory when it is freed
        mbar_drain(bar_drain, 0, w);
      }
    }
  } else if (warp < kFirstFinishWarp) {
    setmaxnreg_inc<kRegsSoftmax>();
    // ------------------------------------------------------------------------------------------ softmax warps
    const int t = (warp - kFirstSoftmaxWarp) >> 2;
    const int q = warp & 3;  // tensor-memory lanes, and rows of the tile, 32q .. 32q+31
    const uint32_t lane_sel = static_cast<uint32_t>(q * 32) << 16;
    const uint32_t t_score = tmem_base + lane_sel + t * 128;
    const float sc = p.alpha * 1.4426950408889634f;  // log2 domain (sc > 0, checked by the host: scaling keeps the order)
    uint32_t suse = 0, oitem = 0, fcount = 0;
    ItemWalk it(p);
    for (int i = 0; i < my_items; ++i, it.next()) {
      if (t == 1 && !it.has_b(p.M)) continue;
      float m = -INFINITY;               // maximum the row's exponentials are taken against
      float2 sum = make_float2(0.f, 0.f), sum1 = sum;
      for (int j = 0; j < nblk; ++j) {
        mbar_wait<false>(bar_sfull(t), suse & 1u, w);
        ++suse;
        __syncwarp();
        tcgen05_fence_after_sync();
        uint32_t v[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld_issue_32cols(t_score + c * 32, v[c]);
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld_wait_32(v[c]);
        const int nv = p.N1 - j * 128;
        if (nv < 128) {  // the keys from N1 on read as zeros: their scores count as -inf
#pragma unroll
          for (int c = 0; c < 4; ++c)
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if (c * 32 + e >= nv) v[c][e] = 0xFF800000u;
        }
        float mx[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          mx[c] = __uint_as_float(v[c][0]);
#pragma unroll
          for (int e = 1; e < 31; e += 2) mx[c] = max3(mx[c], __uint_as_float(v[c][e]), __uint_as_float(v[c][e + 1]));
          mx[c] = fmaxf(mx[c], __uint_as_float(v[c][31]));
        }
        const float top = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * sc;
        if (j == 0) {
          m = top;
        } else {
          // the block's own maximum becomes the reference, so that its largest weight is exactly 1 -- unless it lies so far below
          // that the row so far would be scaled up without bound
          const float ref = top > m - kKeepLog2 ? top : m;
          const float f = ref == m ? 1.f : ex2_approx(m - ref);  // (-inf to -inf: nothing to rescale)
          m = ref;
          sum = mul2(sum, splat2(f));
          sum1 = mul2(sum1, splat2(f));
          s_sum[q * 32 + lane] = f;
          __syncwarp();
          if (lane == 0) mbar_arrive(bar_ffull);
        }
        const float2 sc2 = splat2(sc), nm = splat2(-m);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t pk[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const float2 d = fma2(f2_from_bits(v[c][2 * e], v[c][2 * e + 1]), sc2, nm);
            // (all exponentials on the MUFU unit: with an eighth / a quarter / a half of them on the FMA pipe, 256 x 512 x 512 took 37.8 /
            // 38.5 / 41.7 us against 38.1 in the version that still ran it, before every block had its own maximum)
            const float2 ex = make_float2(ex2_approx(d.x), ex2_approx(d.y));
            if (e & 1) sum1 = add2(sum1, ex);
            else sum = add2(sum, ex);
            pk[e] = pack_bf16x2_rn(ex);
          }
          tmem_st_16(t_score + c * 16, pk);
          if (c & 1) {
            tmem_st_wait();
            tcgen05_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_pfull(t, c >> 1));
          }
        }
      }
      // the row sums for the finish warps, once they have read what the array held: the last block's factors, or the previous
      // item's sums (read before the output's last columns)
      fcount += static_cast<uint32_t>(nblk - 1);
      if (nblk > 1) mbar_wait<false>(bar_fdone, (fcount - 1u) & 1u, w);
      else if (oitem > 0) mbar_wait<false>(bar_oempty(t), (oitem - 1u) & 1u, w);
      s_sum[t * 128 + q * 32 + lane] = (sum.x + sum.y) + (sum1.x + sum1.y);
      ++oitem;
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_lfull(t));
    }
  } else {
    setmaxnreg_dec<kRegsFinish>();
    // ------------------------------------------------------------------------------------------ finish warps
    const int q = warp & 3;
    const uint32_t lane_sel = static_cast<uint32_t>(q * 32) << 16;
    const uint32_t box0 = smem_base + AttnSmem::OFF_OUT + q * 2 * 4096;
    uint32_t b_uses = 0, fphase = 0;
    ItemWalk it(p);
    for (int i = 0; i < my_items; ++i, it.next()) {
      const int bz = it.bz, m0 = it.m0();
      // rescale tile A's output so far to the reference of each further block, under that block's exponentials (S.V of the previous
      // blocks is complete: the scores of this one were issued behind it, and the softmax warps have read them)
#pragma unroll 1
      for (int j = 1; j < nblk; ++j) {
        mbar_wait<false>(bar_ffull, fphase & 1u, w);
        ++fphase;
        __syncwarp();
        tcgen05_fence_after_sync();
        const float f = s_sum[q * 32 + lane];
        if (__any_sync(0xFFFFFFFFu, f != 1.f)) {
#pragma unroll 1
          for (int c = 0; c < 128; c += 64) {
            uint32_t o[2][32];
            const uint32_t addr = tmem_base + lane_sel + 256 + c;
            tmem_ld_issue_32cols(addr, o[0]);
            tmem_ld_issue_32cols(addr + 32, o[1]);
#pragma unroll
            for (int k = 0; k < 2; ++k) {
              tmem_ld_wait_32(o[k]);
#pragma unroll
              for (int e = 0; e < 32; e += 2) {
                const float2 v2 = mul2(f2_from_bits(o[k][e], o[k][e + 1]), splat2(f));
                o[k][e] = __float_as_uint(v2.x);
                o[k][e + 1] = __float_as_uint(v2.y);
              }
              tmem_st_32cols(addr + 32 * k, o[k]);
            }
          }
          tmem_st_wait();
        }
        tcgen05_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_fdone);
      }
#pragma unroll 1
      for (int t = 0; t < (it.has_b(p.M) ? 2 : 1); ++t) {
        const uint32_t n = t ? b_uses++ : static_cast<uint32_t>(i);  // items of this tile before this one
        const uint32_t t_out = tmem_base + lane_sel + 256 + t * 128;
        mbar_wait<false>(bar_lfull(t), n & 1u, w);
        __syncwarp();
        // O = (S.V) / (row sum), rounded once, 64 columns at a time through the warp's two boxes
        const float l = s_sum[t * 128 + q * 32 + lane];
        const float2 inv_l = splat2(l > 0.f ? 1.f / l : 0.f);
        mbar_wait<false>(bar_ofull(t), n & 1u, w);
        __syncwarp();
        tcgen05_fence_after_sync();
        const int row0 = m0 + t * 128 + q * 32;
#pragma unroll 1
        for (int half = 0; half < 2; ++half) {
          const uint32_t box = box0 + half * 4096;
          if (lane == 0) tma_store_wait_read<1>();  // the store before the previous one has read this box
          __syncwarp();
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t o[32];
            tmem_ld_32cols(t_out + half * 64 + c * 32, o);
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              uint32_t pk[4];
#pragma unroll
              for (int e = 0; e < 4; ++e) pk[e] = pack_bf16x2_rn(mul2(f2_from_bits(o[8 * g + 2 * e], o[8 * g + 2 * e + 1]), inv_l));
              const uint32_t a = box + static_cast<uint32_t>(lane * 128 + (((4 * c + g) ^ (lane & 7)) << 4));  // 128-byte swizzle
              asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(a), "r"(pk[0]), "r"(pk[1]), "r"(pk[2]), "r"(pk[3]) : "memory");
            }
          }
          if (half == 1) {  // the output has been read: S.V of the next item may overwrite it
            tcgen05_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_oempty(t));
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            if (row0 < p.M && COMFUSE_IN_BOUNDS(row0 >= 0 && bz >= 0 && bz < p.batch, p.status)) tma_store_3d(&tmO, box, half * 64, row0, bz);
            tma_store_commit();
          }
        }
      }
    }
    if (lane == 0) tma_store_wait_read<0>();  // the boxes must outlive the last store's read
  }

  tcgen05_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tcgen05_fence_after_sync();
    tmem_dealloc(tmem_base, 512);
  }
  if (threadIdx.x == 0 && *s_abort) {  // a wait expired: loads that nobody waited for may still be landing
    const uint32_t blocks = s_issued[0];
    for (uint32_t u = blocks > kKvSlots ? blocks - kKvSlots : 0; u < blocks; ++u) mbar_drain(bar_kvfull(u % kKvSlots), (u / kKvSlots) & 1u, w);
    for (int t = 0; t < 2; ++t) {
      const uint32_t uses = (s_issued[1] >> (8 * t)) & 255u;
      if (uses) mbar_drain(bar_qfull(t), (uses - 1u) & 1u, w);
    }
  }
}

}  // namespace

cudaError_t launch_b2b_attention(const void* X, const void* W1, const void* W2, B2bParams p, cudaStream_t st) {
  const DeviceInfo* dev = current_device_info();
  if (!dev) return cudaErrorInvalidDevice;
  if (p.N1 > 128 && p.M > 128) return cudaErrorInvalidValue;  // two tiles share one block, or one tile walks several
  CUtensorMap tmX, tmW1, tmW2, tmO;
  const uint64_t M = p.M, K = p.K, N1 = p.N1, N2 = p.N2;
  if (p.batch < 1) p.batch = 1;
  const uint64_t nb = static_cast<uint64_t>(p.batch);  // dense [batch, rows, cols] tensors
  // operand boxes are 64 elements x 128 rows, a softmax warp stores 64 elements x 32 rows
  if (!encode_tmap_bf16_3d(&tmX, X, K, M, nb, K * 2, M * K * 2, 128) ||
      !(p.keys_row_major ? encode_tmap_bf16_3d(&tmW1, W1, K, N1, nb, K * 2, N1 * K * 2, 128)    // [batch, N1, K]
                         : encode_tmap_bf16_3d(&tmW1, W1, N1, K, nb, N1 * 2, K * N1 * 2, 128)) ||
      !encode_tmap_bf16_3d(&tmW2, W2, N2, N1, nb, N2 * 2, N1 * N2 * 2, 128) ||
      !encode_tmap_bf16_3d(&tmO, p.O, N2, M, nb, N2 * 2, M * N2 * 2, 32))
    return cudaErrorInvalidValue;
  // One tile per CTA where that still leaves a CTA for each: two tiles in one CTA share its tensor core and MUFU unit.
  p.mblocks = (p.M + 127) / 128;
  p.item_rows = static_cast<long long>(p.batch) * p.mblocks <= dev->sm_count ? 128 : 256;
  p.mpairs = (p.M + p.item_rows - 1) / p.item_rows;

  constexpr int kMaxDev = 64;
  static std::atomic<bool> ready[kMaxDev];  // set (released) once the kernels' attributes are in place on that device
  const int di = dev->device < kMaxDev ? dev->device : kMaxDev - 1;
  if (!ready[di].load(std::memory_order_acquire)) {
    for (auto k : {b2b_attention_kernel<false>, b2b_attention_kernel<true>}) {
      const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, AttnSmem::BYTES);
      if (e != cudaSuccess) return e;
    }
    ready[di].store(true, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  const long long items = static_cast<long long>(p.batch) * p.mpairs;
  cfg.gridDim = dim3(static_cast<unsigned>(items < dev->sm_count ? items : dev->sm_count), 1, 1);
  cfg.blockDim = dim3(kAttnThreads, 1, 1);
  cfg.dynamicSmemBytes = AttnSmem::BYTES;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // set-up may overlap the previous kernel's tail
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = programmatic_launch_enabled() ? 1 : 0;
  count_launch();
  return p.keys_row_major ? cudaLaunchKernelEx(&cfg, b2b_attention_kernel<true>, tmX, tmW1, tmW2, tmO, p)
                          : cudaLaunchKernelEx(&cfg, b2b_attention_kernel<false>, tmX, tmW1, tmW2, tmO, p);
}

}  // namespace comfuse
