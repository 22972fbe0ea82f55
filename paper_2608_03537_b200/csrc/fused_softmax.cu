// Instantiations of the fused kernel for  P = softmax(alpha*A.B + mask)  over the last dimension
// (ReduceMode softmax of Sec. 5; the attention-score pattern of Sec. 6.1).
#include "fused_launch.cuh"

namespace comfuse {

namespace {

// Row lengths with an instantiation of their own: its clusters' CTAs, and up to how many rounds of them beat the row kernel behind a
// short contraction, without and with a soft-cap (two MUFU operations a score, which the row kernel pays twice for all but
// a row's last two chunks).  A round takes the clusters about 8 .. 10 us (5 where a CTA holds 256 columns), the row kernel a call of up
// to one round of its pairs 4 us and 2.5 for each 256 columns.  Measured, last round taken / the next one / row kernel, us, K = 64, 7 clusters of 12
// or more CTAs, 11 of 10, 15 of 8, 22 of 6 and 33 of 4 at once:
//    768  11.6 / 18.8 / 11.5, soft-cap 18.0 / 31.6 / 19.5, mask 14.2 / 24.4 / 14.9    2048  20.6 / 28.4 / 24.1, soft-cap 52.4 / 68.4 / 53.4, mask 29.6 / 41.9 / 34.2
//   1024  12.9 / 19.9 / 13.8, soft-cap 20.8 / 35.5 / 26.2, mask 17.0 / 29.0 / 18.6    2560  24.6 / 34.0 / 28.9, soft-cap 59.5 / 78.4 / 66.5, mask 32.1 / 45.5 / 41.9
//   1280  14.3 / 18.7 / 16.0, soft-cap 32.1 / 41.0 / 33.0, mask 18.7 / 25.5 / 22.4    3072  24.2 / 34.1 / 33.8, soft-cap 78.7 / 97.1 / 79.9, mask 45.8 / 59.5 / 49.6
//   1536  13.0 / 22.1 / 19.0, soft-cap 39.8 / 57.2 / 40.0, mask 16.6 / 29.4 / 26.4    3584  34.6 / 44.4 / 39.0, soft-cap 78.8 / 97.5 / 93.2, mask 45.9 / 59.7 / 57.4
//   1792  19.4 / 24.2 / 21.6, soft-cap 41.4 / 50.8 / 46.5, mask 27.3 / 34.6 / 30.2    4096  38.1 / 46.4 / 44.2, soft-cap 102.4 / 119.6 / 106.7, mask 56.8 / 69.3 / 65.1
// The causal mask spares both kernels much the same: 1024 12.8 / 18.8 / 13.6, 1792 19.3 / 24.3 / 21.2, 2048 at 3 rounds 24.2 / 23.4.
struct ClusterForm {
  int n, ctas, rounds, rounds_softcap;
};
constexpr ClusterForm kForms[] = {{256, 2, 0, 0},  {512, 2, 0, 0},  {768, 4, 1, 1},   {1024, 4, 1, 1},  {1280, 10, 2, 3}, {1536, 6, 1, 2},
                                  {1792, 14, 3, 4}, {2048, 8, 2, 3}, {2560, 10, 2, 3}, {3072, 12, 2, 4}, {3584, 14, 3, 4}, {4096, 16, 4, 6}};

// Clusters of `size` CTAs that are resident at once; every instantiation puts one CTA on an SM, so one of them answers for all.
int resident_clusters(int size) {
  static ResidentClusters cache;
  using Cfg = PairCfg<EPI_SOFTMAX, 256, 0, 1, 3, 0, 4>;
  const DeviceInfo* dev = current_device_info();
  return dev ? cache.of(reinterpret_cast<const void*>(&fused_pair_kernel<EPI_SOFTMAX, 256, 0, 1, 3, 0, 4>), Cfg::kThreads, Cfg::SMEM_BYTES, size, *dev) : 0;
}

// So few rows that the row kernel's CTA pairs do not fill the machine: clusters put 4 to 16 CTAs on every pair of row blocks.
bool clusters_are_faster(const ClusterForm& f, const FusedParams& p) {
  int rounds = p.softcap > 0.f ? f.rounds_softcap : f.rounds;
  if (rounds == 0) return false;
  if (f.n == 3072 && p.mask && p.softcap <= 0.f) ++rounds;
  const long long row_pairs = static_cast<long long>(p.batch) * ((p.M + 255) / 256);
  return row_pairs <= static_cast<long long>(rounds) * resident_clusters(f.ctas);
}

}  // namespace

cudaError_t launch_fused_softmax(const GemmMaps& maps, const FusedParams& p, cudaStream_t st, bool supported_only) {
  // Short K: recomputing a score chunk is cheaper than keeping the row block on-chip across a cluster, but for few rows.
  // COMFUSE_SOFTMAX_CLUSTER=1 forces the cluster kernel where it has an instantiation (for comparisons).
  static const bool force_cluster = std::getenv("COMFUSE_SOFTMAX_CLUSTER") != nullptr;
  // A row length between two instantiations runs on the next wider one: the columns from N on read as zeros and are
  // masked like the ones above the diagonal of a causal mask.
  int form = 0;
  bool rows = softmax_rows_supported(p) && !force_cluster;
  for (const ClusterForm& f : kForms)
    if (form == 0 && p.N <= f.n) {
      form = f.n;
      rows = rows && (supported_only || !clusters_are_faster(f, p));
    }
  if (rows) return supported_only ? cudaSuccess : launch_softmax_rows(maps, p, st);
#define COMFUSE_CASE(n, b0, b1, cn, nst, epw) \
  case n:                                     \
    return supported_only ? cudaSuccess : launch_pair_instance<EPI_SOFTMAX, b0, b1, cn, nst, 0, epw>(maps, p, st);
  // Behind a long contraction the MainLoop is what counts: three pipeline stages with both sub-tiles in lock step (the A
  // tile fetched once per K block) and eight epilogue warps, instead of two stages and sixteen warps.  Measured: 8192 x 1024,
  // K = 1024: 24.1 us against 28.7; 8192 x 4096, K = 1024: 106.6 against 126.1; but K = 320 / 512 (causal): 39.2 / 44.9
  // against 36.4 / 43.1.  COMFUSE_SOFTMAX_STAGES=2 or 3 forces either form.
  static const char* stages_env = std::getenv("COMFUSE_SOFTMAX_STAGES");
  const bool long_k = stages_env ? stages_env[0] == '3' : p.K >= 768;
  if (long_k) {
    switch (form) {
      case 256: return supported_only ? cudaSuccess : launch_pair_instance<EPI_SOFTMAX, 256, 0, 1, 5, 0, 2>(maps, p, st);
      case 512: return supported_only ? cudaSuccess : launch_pair_instance<EPI_SOFTMAX, 256, 256, 1, 3, 1, 2>(maps, p, st);
      case 1024: return supported_only ? cudaSuccess : launch_pair_instance<EPI_SOFTMAX, 256, 256, 2, 3, 1, 2>(maps, p, st);
      case 2048: return supported_only ? cudaSuccess : launch_pair_instance<EPI_SOFTMAX, 256, 256, 4, 3, 1, 2>(maps, p, st);
      case 4096: return supported_only ? cudaSuccess : launch_pair_instance<EPI_SOFTMAX, 256, 256, 8, 3, 1, 2>(maps, p, st);
      default: break;
    }
  }
  // Else the softmax passes are latency-bound on few warps and need few registers: four epilogue warps per lane quarter.
  switch (form) {
    COMFUSE_CASE(256, 256, 0, 1, 3, 4)
    COMFUSE_CASE(512, 256, 256, 1, 2, 4)
    COMFUSE_CASE(1024, 256, 256, 2, 2, 4)
    COMFUSE_CASE(2048, 256, 256, 4, 2, 4)
    COMFUSE_CASE(4096, 256, 256, 8, 2, 4)
    case 768: case 1280: case 1536: case 1792:
      return launch_fused_softmax_more_rows_a(form, maps, p, st, supported_only);  // translation units of their own
    case 2560: case 3072: case 3584:
      return launch_fused_softmax_more_rows_b(form, maps, p, st, supported_only);
    default:
      // Long K and rows wider than the largest cluster holds (N > 4096): the row kernel's statistics pass followed by a
      // second MainLoop pass takes any N.  It pays the GEMM twice, which is still less than writing and re-reading the scores.
      if (p.N >= 64) return supported_only ? cudaSuccess : launch_softmax_rows(maps, p, st);
      return cudaErrorInvalidValue;
  }
#undef COMFUSE_CASE
}

}  // namespace comfuse
