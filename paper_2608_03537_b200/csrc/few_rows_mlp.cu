// The GELU + residual + LayerNorm MLP form of the back-to-back GEMM for FEW ROWS.  (The ReLU form keeps its row-tiled kernel at every
// size: its rows are promised the same bits whatever problem they are part of, and the shares below add up in another order.)
//
// What bounds it: latency.  The row-tiled form walks the hidden layer in chunks inside one CTA pair, about a microsecond per
// chunk, however few rows there are.  Here a cluster takes the hidden layer side by side, CTA c the 128 hidden units from 128 c on:
//
//   D1^T = W1[:, units]^T . X^T     weights as the UMMA's 128-row operand, the rows as its N operand (MT = 16 .. 64 rows)
//   S    = GELU(D1 + b1)            bf16, K-major in shared memory: a thread holds one hidden unit of MT / 4 rows
//   D2^T = W2[units, :]^T . S^T     this CTA's share of the output, 128 columns
//   the shares meet in a reduce-scatter over distributed shared memory (one bulk copy per peer): CTA c finishes the c-th slice of
//   the rows, a warp per row -- the output has 128 columns, so the LayerNorm needs no exchange.
//
// Measured against the row-tiled form: see few_rows_mlp_fits.
#include <atomic>

#include "b2b_params.h"
#include "epilogue_common.cuh"
#include "host_common.h"
#include "sm100_primitives.cuh"

namespace comfuse {
namespace {

struct FewMlpParams {
  B2bParams b;
  int cluster;  // CTAs that share the hidden layer
};

template <int MT>
struct FewMlpCfg {
  static constexpr int kEpiWarps = 16;
  static constexpr int kThreads = 32 * (2 + kEpiWarps);
  static constexpr int W_BYTES = 128 * 64 * 2;          // W1 of one K block: 64 contraction rows x 128 hidden units
  static constexpr int X_BYTES = MT * 64 * 2;
  static constexpr int STAGE_BYTES = W_BYTES + X_BYTES;
  static constexpr int W2_BYTES = 2 * W_BYTES;          // 128 hidden units x 128 columns
  static constexpr int S_BYTES = 2 * X_BYTES;           // MT rows x 128 hidden units
  static constexpr int ROW_BYTES = 128 * 4;
  static constexpr int RECV_BYTES = (MT + 15) * ROW_BYTES;  // up to 16 slices of ceil(rows / 16) rows
  static constexpr int STAGES_FIT = (232448 - W2_BYTES - S_BYTES - RECV_BYTES - 2048) / STAGE_BYTES;
  static constexpr int NSTAGES = STAGES_FIT > 6 ? 6 : STAGES_FIT;
  static constexpr int OFF_W2 = NSTAGES * STAGE_BYTES;
  static constexpr int OFF_S = OFF_W2 + W2_BYTES;
  static constexpr int OFF_RECV = OFF_S + S_BYTES;
  static constexpr int OFF_BAR = OFF_RECV + RECV_BYTES;
  static constexpr int NUM_BARS = 2 * NSTAGES + 5;
  static constexpr int OFF_MISC = OFF_BAR + NUM_BARS * 8;
  static constexpr int SMEM_BYTES = OFF_MISC + 16 + 1024;
  static constexpr int TMEM_COLS = 2 * MT;              // D1 and D2
  static constexpr int MOVE = MT / 4 > 8 ? MT / 4 : 8;  // rows a warp takes out of tensor memory at a time
  static constexpr int kMoveWarps = 4 * (MT / MOVE);
  static_assert(STAGE_BYTES % 1024 == 0 && MT * ROW_BYTES <= NSTAGES * STAGE_BYTES, "the output shares are staged in the idle ring");
  static_assert(TMEM_COLS >= 32 && TMEM_COLS <= 128, "tensor memory");
  static_assert(SMEM_BYTES <= 232448 && SMEM_BYTES > 116 * 1024, "one CTA per SM (tensor-memory allocation never waits)");
};

template <int MT>
__global__ void __launch_bounds__(FewMlpCfg<MT>::kThreads, 1)
few_rows_mlp_kernel(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW1,
                    const __grid_constant__ CUtensorMap tmW2, const FewMlpParams fp) {
  using Cfg = FewMlpCfg<MT>;
  constexpr int NSTAGES = Cfg::NSTAGES;
  constexpr int RC = MT / Cfg::kEpiWarps;  // rows per epilogue warp
  constexpr int MOVE = Cfg::MOVE;
  const B2bParams& p = fp.b;

  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_addr = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + (((raw_addr + 1023u) & ~1023u) - raw_addr);
  const uint32_t smem_base = smem_u32(smem);
  const uint32_t bar_base = smem_base + Cfg::OFF_BAR;
  auto bar_full = [&](int s) { return bar_base + 8u * s; };
  auto bar_empty = [&](int s) { return bar_base + 8u * (NSTAGES + s); };
  const uint32_t bar_d1 = bar_base + 8u * (2 * NSTAGES);  // D1 complete
  const uint32_t bar_w2 = bar_d1 + 8u;                    // W2 landed
  const uint32_t bar_s = bar_d1 + 16u;                    // S written
  const uint32_t bar_d2 = bar_d1 + 24u;                   // D2 complete
  const uint32_t bar_recv = bar_d1 + 32u;                 // the peers' shares have arrived
  uint32_t* s_tmem_base = reinterpret_cast<uint32_t*>(smem + Cfg::OFF_MISC);
  volatile int* s_abort = reinterpret_cast<volatile int*>(smem + Cfg::OFF_MISC + 4);
  volatile int* s_told = s_abort + 1;    // a wait expired in some CTA of the cluster
  volatile int* s_issued = s_abort + 2;  // K blocks whose loads are issued (fewer than all where the producer's wait expires)

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int hc = fp.cluster;
  const int rank = static_cast<int>(cluster_ctarank());
  const int n0 = rank * 128;  // first hidden unit
  const int m0 = static_cast<int>(blockIdx.x) / hc * MT;
  const int rows = p.M - m0 < MT ? p.M - m0 : MT;
  const int rs = (rows + hc - 1) / hc;  // rows per slice
  auto slice_rows = [&](int j) { return rows - j * rs < 0 ? 0 : (rows - j * rs < rs ? rows - j * rs : rs); };
  const int rv = slice_rows(rank);
  const int KB = (p.K + 63) >> 6;
  const WaitCtx w{s_abort, p.status, p.timeout_ns};
  griddep_launch_dependents();  // the next kernel's set-up may overlap this kernel (it waits before touching memory)

  if (threadIdx.x == 0) {
    for (int s = 0; s < NSTAGES; ++s) {
      mbar_init(bar_full(s), 1);
      mbar_init(bar_empty(s), 1);
    }
    mbar_init(bar_d1, 1);
    mbar_init(bar_w2, 1);
    mbar_init(bar_s, Cfg::kMoveWarps);
    mbar_init(bar_d2, 1);
    mbar_init(bar_recv, 1);
    *s_abort = 0;
    *s_told = 0;
    *s_issued = KB;
    fence_mbar_init();
    mbar_arrive_expect_tx(bar_recv, static_cast<uint32_t>((hc - 1) * rv * Cfg::ROW_BYTES));  // armed before any peer can send
    prefetch_tensormap(&tmX);
    prefetch_tensormap(&tmW1);
    prefetch_tensormap(&tmW2);
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
  griddep_wait();  // the set-up above may overlap the previous kernel's tail; global memory is touched only below

  if (warp == 0) {
    // ------------------------------------------------------------------------------------------ TMA producer
    if (elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      for (int kb = 0; kb < KB; ++kb) {
        if (!mbar_wait<false>(bar_empty(stage), phase ^ 1u, w)) {  // passes on a fresh barrier
          *s_issued = kb;
          break;
        }
        const uint32_t sw = smem_base + stage * Cfg::STAGE_BYTES;
        mbar_arrive_expect_tx(bar_full(stage), Cfg::STAGE_BYTES);
        tma_load_3d(sw, &tmW1, bar_full(stage), n0, kb * 64, 0);
        tma_load_3d(sw + 8192, &tmW1, bar_full(stage), n0 + 64, kb * 64, 0);
        tma_load_3d(sw + Cfg::W_BYTES, &tmX, bar_full(stage), kb * 64, m0, 0);
        if (kb == 0) {  // W2 behind the first K block: it has the whole first product to land
          mbar_arrive_expect_tx(bar_w2, Cfg::W2_BYTES);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            tma_load_3d(smem_base + Cfg::OFF_W2 + j * 8192, &tmW2, bar_w2, (j & 1) * 64, n0 + (j >> 1) * 64, 0);
        }
        if (++stage == NSTAGES) { stage = 0; phase ^= 1u; }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------------------------------ UMMA issuer
    if (elect_one()) {
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      constexpr uint32_t idesc = make_idesc_bf16(128, MT, true, false);  // weights MN-major, rows K-major
      for (int kb = 0; kb < KB; ++kb) {
        if (!mbar_wait<false>(bar_full(stage), phase, w)) { ok = false; break; }
        tcgen05_fence_after_sync();
        const uint32_t sw = smem_base + stage * Cfg::STAGE_BYTES;
        const uint64_t wdesc = make_smem_desc_sw128(sw, 8192, 1024), xdesc = make_smem_desc_sw128(sw + Cfg::W_BYTES, 16, 1024);
#pragma unroll
        for (int k = 0; k < 4; ++k)
          umma_bf16_ss(tmem_base, wdesc + static_cast<uint64_t>(k * 128), xdesc + static_cast<uint64_t>(k * 2), idesc, (kb | k) != 0 ? 1u : 0u);
        umma_commit(bar_empty(stage));
        if (++stage == NSTAGES) { stage = 0; phase ^= 1u; }
      }
      umma_commit(bar_d1);
      ok = ok && mbar_wait<false>(bar_w2, 0, w) && mbar_wait<false>(bar_s, 0, w);
      if (ok) {
        tcgen05_fence_after_sync();
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint64_t wdesc = make_smem_desc_sw128(smem_base + Cfg::OFF_W2 + (kk >> 2) * 16384, 8192, 1024);
          const uint64_t sdesc = make_smem_desc_sw128(smem_base + Cfg::OFF_S + (kk >> 2) * Cfg::X_BYTES, 16, 1024);
          umma_bf16_ss(tmem_base + MT, wdesc + static_cast<uint64_t>((kk & 3) * 128), sdesc + static_cast<uint64_t>((kk & 3) * 2), idesc, kk != 0 ? 1u : 0u);
        }
      }
      umma_commit(bar_d2);
      mbar_drain(bar_d2, 0, w);  // nothing may still be writing tensor memory when it is freed
    }
  } else {
    // ------------------------------------------------------------------------------------------ epilogue warps
    const int e = warp - 2;
    const int q = warp & 3;  // TMEM lane quarter: hidden units / output columns 32q .. 32q+31
    const int h = e >> 2;    // rows h * MOVE .. of what this warp takes out of tensor memory
    const int unit = q * 32 + lane;
    const float b1 = p.b1 && n0 + unit < p.N1 ? bf16_lo(__ldg(p.b1 + n0 + unit)) : 0.f;  // (units from N1 on: zeros all the way)
    // row stage: lane = columns 4 lane .. 4 lane + 3, rows e, e + 16, ... of the slice
    const uint2 zero = make_uint2(0u, 0u), one = make_uint2(0x3F803F80u, 0x3F803F80u);
    const uint2 b2 = p.b2 ? __ldg(reinterpret_cast<const uint2*>(p.b2) + lane) : zero;
    const uint2 gamma = p.gamma ? __ldg(reinterpret_cast<const uint2*>(p.gamma) + lane) : one;
    const uint2 beta = p.beta ? __ldg(reinterpret_cast<const uint2*>(p.beta) + lane) : zero;
    const int row0 = m0 + rank * rs;
    uint2 res[RC];
#pragma unroll
    for (int i = 0; i < RC; ++i) {
      const int r = e + i * Cfg::kEpiWarps;
      res[i] = zero;
      if (r < rv) res[i] = __ldg(reinterpret_cast<const uint2*>(p.X + static_cast<long long>(row0 + r) * 128) + lane);
    }

    mbar_wait<false>(bar_d1, 0, w);
    __syncwarp();
    tcgen05_fence_after_sync();
    if (h * MOVE < MT) {  // S = GELU(D1 + b1)
      uint32_t v[MOVE];
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + h * MOVE;
#pragma unroll
      for (int i = 0; i < MOVE; i += 8) tmem_ld_issue_8(taddr + i, v + i);
#pragma unroll
      for (int i = 0; i < MOVE; i += 8) tmem_ld_wait_8(v + i);
      const uint32_t sbox = smem_base + Cfg::OFF_S + (unit >> 6) * Cfg::X_BYTES;
#pragma unroll
      for (int i = 0; i < MOVE; i += 2) {
        const uint32_t pk = pack_bf16x2_rn(gelu_tanh_f32x2(add2(f2_from_bits(v[i], v[i + 1]), splat2(b1))));
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int m = h * MOVE + i + k;
          const uint32_t a = sbox + static_cast<uint32_t>(m * 128 + ((((unit & 63) >> 3) ^ (m & 7)) << 4) + (unit & 7) * 2);
          asm volatile("st.shared.b16 [%0], %1;" ::"r"(a), "h"(static_cast<uint16_t>(k ? pk >> 16 : pk)) : "memory");
        }
      }
      fence_proxy_async_smem();  // the UMMAs read what these threads wrote
      tcgen05_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_s);
    }

    mbar_wait<false>(bar_d2, 0, w);
    __syncwarp();
    tcgen05_fence_after_sync();
    if (h * MOVE < MT) {  // this CTA's share of the output -> [row][column] fp32 in the ring, which nothing uses any more
      uint32_t v[MOVE];
      const uint32_t taddr = tmem_base + (static_cast<uint32_t>(q * 32) << 16) + MT + h * MOVE;
#pragma unroll
      for (int i = 0; i < MOVE; i += 8) tmem_ld_issue_8(taddr + i, v + i);
#pragma unroll
      for (int i = 0; i < MOVE; i += 8) tmem_ld_wait_8(v + i);
      const uint32_t dst = smem_base + static_cast<uint32_t>((h * MOVE * 128 + unit) * 4);
#pragma unroll
      for (int i = 0; i < MOVE; ++i)
        if (h * MOVE + i < rows) asm volatile("st.shared.b32 [%0], %1;" ::"r"(dst + i * Cfg::ROW_BYTES), "r"(v[i]) : "memory");
    }
    if (hc > 1) {
      fence_proxy_async_smem();  // the bulk copies below read what these threads wrote
      named_barrier_sync(1, 32 * Cfg::kEpiWarps);
      if (e == 0 && lane < hc && lane != rank) {
        const uint32_t bytes = static_cast<uint32_t>(slice_rows(lane) * Cfg::ROW_BYTES);
        if (bytes)
          bulk_copy_to_peer(map_to_cta(smem_base + Cfg::OFF_RECV + rank * rs * Cfg::ROW_BYTES, static_cast<uint32_t>(lane)),
                            smem_base + lane * rs * Cfg::ROW_BYTES, bytes, map_to_cta(bar_recv, static_cast<uint32_t>(lane)));
      }
      __syncwarp();
      mbar_wait<true>(bar_recv, 0, w);
    } else {
      named_barrier_sync(1, 32 * Cfg::kEpiWarps);
    }

    // ---------------- the rows of this CTA's slice, RC per warp
    float x[RC][4];
#pragma unroll
    for (int i = 0; i < RC; ++i) {
      int r = e + i * Cfg::kEpiWarps;
      r = r < rv ? r : 0;  // (a row past the end repeats the first one; it is not stored)
      x[i][0] = x[i][1] = x[i][2] = x[i][3] = 0.f;
      if (rv > 0)
        for (int s = 0; s < hc; ++s) {  // the same order whichever CTA finishes the row
          float o[4];
          asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                       : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3])
                       : "r"(smem_base + (s == rank ? 0 : Cfg::OFF_RECV) + (s * rs + r) * Cfg::ROW_BYTES + lane * 16));
#pragma unroll
          for (int j = 0; j < 4; ++j) x[i][j] += o[j];
        }
    }
    float mean[RC], m2[RC];
#pragma unroll
    for (int i = 0; i < RC; ++i) {
      const float2 x01 = add2(add2(make_float2(x[i][0], x[i][1]), bf16x2_to_f2(b2.x)), bf16x2_to_f2(res[i].x));
      const float2 x23 = add2(add2(make_float2(x[i][2], x[i][3]), bf16x2_to_f2(b2.y)), bf16x2_to_f2(res[i].y));
      x[i][0] = x01.x; x[i][1] = x01.y; x[i][2] = x23.x; x[i][3] = x23.y;
      mean[i] = (x[i][0] + x[i][1]) + (x[i][2] + x[i][3]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int i = 0; i < RC; ++i) mean[i] += __shfl_xor_sync(0xFFFFFFFFu, mean[i], o);
#pragma unroll
    for (int i = 0; i < RC; ++i) {
      mean[i] *= 1.f / 128.f;
      m2[i] = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) m2[i] = fmaf(x[i][j] - mean[i], x[i][j] - mean[i], m2[i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int i = 0; i < RC; ++i) m2[i] += __shfl_xor_sync(0xFFFFFFFFu, m2[i], o);
    const float2 g01 = bf16x2_to_f2(gamma.x), g23 = bf16x2_to_f2(gamma.y), b01 = bf16x2_to_f2(beta.x), b23 = bf16x2_to_f2(beta.y);
#pragma unroll
    for (int i = 0; i < RC; ++i) {
      const int r = e + i * Cfg::kEpiWarps;
      float2 y01 = make_float2(x[i][0], x[i][1]), y23 = make_float2(x[i][2], x[i][3]);
      const float rstd = rsqrtf(m2[i] * (1.f / 128.f) + p.eps);
      const float2 r2 = splat2(rstd), s2 = splat2(-mean[i] * rstd);
      y01 = fma2(fma2(y01, r2, s2), g01, b01);
      y23 = fma2(fma2(y23, r2, s2), g23, b23);
      if (r < rv && COMFUSE_IN_BOUNDS(row0 + r < p.M, p.status))
        *(reinterpret_cast<uint2*>(p.O + static_cast<long long>(row0 + r) * 128) + lane) = make_uint2(pack_bf16x2_rn(y01), pack_bf16x2_rn(y23));
    }
  }

  tcgen05_fence_before_sync();
  __syncthreads();
  if (threadIdx.x == 0 && *s_abort) tell_cluster(s_told, static_cast<uint32_t>(hc));
  cluster_sync_after_init();  // what is sent here has been waited for by its receiver: arriving is enough (see few_rows.cu)
  if (warp == 1) {
    __syncwarp();
    tcgen05_fence_after_sync();
    tmem_dealloc(tmem_base, Cfg::TMEM_COLS);
  }
  if (warp == 0 && *s_told) {  // ... unless a wait expired: loads and the peers' sends may still be under way
    if (lane == 0) {
      const int issued = *s_issued;
      for (int u = issued > NSTAGES ? issued - NSTAGES : 0; u < issued; ++u) mbar_drain(bar_full(u % NSTAGES), (u / NSTAGES) & 1u, w);
      if (issued > 0) mbar_drain(bar_w2, 0, w);
      mbar_drain(bar_recv, 0, w);
    }
    __syncwarp();
    cluster_sync_all();
  }
}

template <int MT>
cudaLaunchConfig_t launch_config(int cluster, unsigned grid, cudaLaunchAttribute* attr, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3(FewMlpCfg<MT>::kThreads, 1, 1);
  cfg.dynamicSmemBytes = FewMlpCfg<MT>::SMEM_BYTES;
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(cluster);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // set-up may overlap the previous kernel's tail
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = programmatic_launch_enabled() ? 2 : 1;
  return cfg;
}

template <int MT>
cudaError_t prepare() {  // the kernel's attributes, once per device
  constexpr int kMaxDev = 64;
  static std::atomic<bool> ready[kMaxDev];
  const DeviceInfo* dev = current_device_info();
  if (!dev) return cudaErrorInvalidDevice;
  const int di = dev->device < kMaxDev ? dev->device : kMaxDev - 1;
  if (ready[di].load(std::memory_order_acquire)) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(few_rows_mlp_kernel<MT>, cudaFuncAttributeMaxDynamicSharedMemorySize, FewMlpCfg<MT>::SMEM_BYTES);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(few_rows_mlp_kernel<MT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  ready[di].store(true, std::memory_order_release);
  return cudaSuccess;
}

// Clusters of `size` CTAs that are resident at once (one CTA per SM in every instantiation)
int resident_clusters(int size, const DeviceInfo& dev) {
  static ResidentClusters cache;
  return cache.of(reinterpret_cast<const void*>(&few_rows_mlp_kernel<64>), FewMlpCfg<64>::kThreads, FewMlpCfg<64>::SMEM_BYTES, size, dev);
}

int rows_per_item(int M) { return M <= 16 ? 16 : M <= 32 ? 32 : 64; }

}  // namespace

// Taken where all its clusters are resident at once.  Measured there (device time, row-tiled form / this one, us): 8 rows x 440 hidden
// units 8.2 / 3.8, 4 x 952 11.1 / 3.9, 43 x 976 11.1 / 6.2, 679 x 512 8.6 / 5.9, 1227 x 248 7.0 / 5.8, 2473 x 160 7.0 / 5.7.
// Hidden layers of fewer than 64 units: every CTA asks for the same few sectors of W1 and W2, and many CTAs at once wait for one another
// there.  8 units: 2000 rows 6.2 / 5.8, 2500 6.3 / 6.1, 3000 6.2 / 6.4, 8000 7.0 / 10.1; 24 units: 3000 6.2 / 5.8, 4000 6.3 / 6.4,
// 5000 6.5 / 7.6; 40 units: 4000 6.3 / 6.1, 5000 6.6 / 7.3; 64 units: 9000 6.3 / 5.6.
bool few_rows_mlp_fits(int M, int N1, int N2) {
  const DeviceInfo* dev = current_device_info();
  const int cluster = (N1 + 127) / 128;
  if (!dev || dev->cc_major != 10 || N2 != 128 || cluster > 16) return false;
  const int groups = (M + rows_per_item(M) - 1) / rows_per_item(M);
  if (N1 < 64 && groups > dev->sm_count / (N1 < 16 ? 4 : N1 < 32 ? 3 : 2)) return false;
  return groups <= resident_clusters(cluster, *dev);
}

cudaError_t launch_few_rows_mlp(const void* X, const void* W1, const void* W2, B2bParams p, cudaStream_t st) {
  const int mt = rows_per_item(p.form_units);
  FewMlpParams fp;
  fp.cluster = (p.N1 + 127) / 128;
  CUtensorMap tmX, tmW1, tmW2;
  const uint64_t M = p.M, K = p.K, N1 = p.N1, N2 = p.N2;
  if (!encode_tmap_bf16_3d(&tmX, X, K, M, 1, K * 2, M * K * 2, static_cast<uint32_t>(mt)) ||
      !encode_tmap_bf16_3d(&tmW1, W1, N1, K, 1, N1 * 2, K * N1 * 2, 64) || !encode_tmap_bf16_3d(&tmW2, W2, N2, N1, 1, N2 * 2, N1 * N2 * 2, 64))
    return cudaErrorInvalidValue;
  fp.b = p;
  const unsigned grid = static_cast<unsigned>((p.M + mt - 1) / mt * fp.cluster);
  cudaLaunchAttribute attr[2];
#define COMFUSE_CASE(MT)                                                                                                          \
  if (mt == MT) {                                                                                                                 \
    const cudaError_t e = prepare<MT>();                                                                                          \
    if (e != cudaSuccess) return e;                                                                                               \
    cudaLaunchConfig_t cfg = launch_config<MT>(fp.cluster, grid, attr, st);                                                       \
    count_launch();                                                                                                               \
    return cudaLaunchKernelEx(&cfg, few_rows_mlp_kernel<MT>, tmX, tmW1, tmW2, fp);                                                \
  }
  COMFUSE_CASE(16)
  COMFUSE_CASE(32)
  COMFUSE_CASE(64)
#undef COMFUSE_CASE
  return cudaErrorInvalidValue;
}

}  // namespace comfuse
