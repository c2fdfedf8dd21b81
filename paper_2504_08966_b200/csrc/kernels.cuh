// Launchers of the PACT kernels (host side); one translation unit per stage group.
#pragma once
#include "common.cuh"

namespace pact {

// Launches a kernel; pdl: with the programmatic-serialization attribute (it may start before its predecessor in
// the stream has finished and must call pdl_wait() before it reads what the predecessor wrote, or writes what the
// predecessor reads); cluster > 0: in thread-block clusters of that many CTAs along x; coop: every CTA resident at once.
struct LaunchOpt {
  bool pdl = true;
  int cluster = 0;
  bool coop = false;
};
template <typename... KArgs, typename... Args>
inline cudaError_t launch_opt(LaunchOpt opt, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[3];
  int n = 0;
  if (opt.pdl) {
    attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (opt.coop) {
    attr[n].id = cudaLaunchAttributeCooperative;
    attr[n++].val.cooperative = 1;
  }
  if (opt.cluster > 0) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = opt.cluster;
    attr[n].val.clusterDim.y = 1;
    attr[n++].val.clusterDim.z = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl,
                            Args &&...args) {
  LaunchOpt o;
  o.pdl = pdl;
  return launch_opt(o, kernel, grid, block, smem, st, args...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_coop(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool pdl,
                               Args &&...args) {
  LaunchOpt o;
  o.pdl = pdl;
  o.coop = true;
  return launch_opt(o, kernel, grid, block, smem, st, args...);
}

// The largest shared-memory carve-out for these kernels.
template <typename... K> inline cudaError_t prefer_shared(K... kernel) {
  cudaError_t e = cudaSuccess;
  ((e = e == cudaSuccess ? cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared) : e), ...);
  return e;
}

// What the launchers know about the device of a context (each context has its own: contexts may be created by several threads
// at once, on different devices, while others are in use); filled by the ..._configure functions, select_configure first.
struct DeviceCfg {
  int sm_count = 0;
  size_t smem_optin = 0;      // most shared memory of a CTA
  int centers_smem_max = 0;   // most dynamic shared memory the centre-selection kernel may ask for
  int lists_resident = 0;     // CTAs of k_lists that fit on the device at once
  int small_clusters = 0;     // clusters of the one-cluster step that do
  bool pair_gram = false, pair_assign = false, pair_spread = false;   // clusters of two CTAs of the pair kernel's forms can be launched
  void *encode_tiled = nullptr;                                       // cuTensorMapEncodeTiled
};

constexpr int kMergeMaxD = 256 * 4 * 8;   // widest hidden state the merge kernel holds in registers

// how a kernel finds its rows
enum RowMode { ROWS_ALL = 0, ROWS_KEPT_LIST = 1, ROWS_PRUNED_LIST = 2 };

// euti.cu
constexpr int kQPartRows = 8;             // most row blocks the column sums of Q are split into: the CTAs of a cluster
// First-level histogram of the threshold selection: scores are not negative, so a key's top bit is set (but of a NaN with its
// sign bit set); the bins are the thirteen top bits of the others, eight of exponent and four of mantissa.
constexpr int kHistShift = 19, kHistBins = 1 << (31 - kHistShift);
__device__ __forceinline__ int key_bin(uint32_t key) { return max(0, (int)(key >> kHistShift) - kHistBins); }
__device__ __forceinline__ uint32_t bin_first(int bin) { return (uint32_t)(bin + kHistBins) << kHistShift; }   // (bin 0 also holds what is below)
// Algorithm 1.  mode 0: scores, threshold, lists, survivor keys (four kernels; the first also clears what later
// kernels accumulate into); mode 1: scores only (three kernels); mode 2: mode 0 up to the token pass (two kernels).
// mark (optional) is called between the kernels of the group (the per-kernel timing of a profiled call)
typedef cudaError_t (*StageMark)(void *);
// The inputs of one image on their way from the host: everything but the hidden states once `keys` has been recorded,
// the rows up to end[k] (all of them for the last part) once part[k] has.
constexpr int kFeedParts = 2;
struct HostFeed {
  cudaEvent_t keys, part[kFeedParts];
  int end[kFeedParts];                     // visual tokens
};
cudaError_t launch_euti(const Batch &bt, int maxN, bool bf16, int mode, const DeviceCfg &cfg, cudaStream_t st, StageMark mark = nullptr,
                        void *mark_arg = nullptr, int *rpp = nullptr);   // rpp: receives the tokens per softmax piece
// modes 0 and 2 for one image whose hidden states arrive in parts meanwhile (one kernel more for each part with visual tokens)
cudaError_t launch_euti_fed(const Batch &bt, int maxN, bool bf16, int mode, const DeviceCfg &cfg, cudaStream_t st, const HostFeed &feed, int *rpp);
int euti_kernels(int mode);
// threshold + ordered compaction of given scores (pact_prune, one image)
cudaError_t launch_split(const Batch &bt, int N, const DeviceCfg &cfg, cudaStream_t st);
cudaError_t euti_configure(const DeviceCfg &cfg, int n_qcols, int n_qh);
cudaError_t select_configure(DeviceCfg *cfg);   // what launch_split needs, for the current device

// cluster.cu
cudaError_t cluster_configure(DeviceCfg *cfg);
// gathers survivor keys and inverse norms of the listed rows; clears what later kernels accumulate into
cudaError_t launch_keynorm_gather(const Batch &bt, int maxN, bool bf16, cudaStream_t st);
cudaError_t launch_center_key_gather(const Batch &bt, int maxN, bool bf16, bool all_rows, cudaStream_t st);
cudaError_t launch_gram(const Batch &bt, int maxN, bool bf16, const DeviceCfg &cfg, cudaStream_t st);
// centre selection, cluster ids and centre keys (two kernels); maxQ: estimate of the largest number of survivors of an
// image (sizes staging buffers only)
cudaError_t launch_centers(const Batch &bt, int maxQ, bool bf16, const DeviceCfg &cfg, int sweep_limit, cudaStream_t st);
cudaError_t launch_assign(const Batch &bt, int maxN, bool bf16, RowMode mode, const DeviceCfg &cfg, cudaStream_t st);
cudaError_t launch_label(const Batch &bt, int maxN, bool bf16, RowMode mode, cudaStream_t st);
// layer choice: inverse norms of all keys of every layer, largest pair distance (any dtype), result
cudaError_t launch_key_rnorm(const Batch &bt, int maxN, bool bf16, cudaStream_t st);
cudaError_t launch_spread(const Batch &bt, int maxN, bool bf16, const DeviceCfg &cfg, cudaStream_t st);
cudaError_t launch_spread_finish(const Batch &bt, float *max_dist, int32_t *layer_out, int layer_base, float threshold,
                          cudaStream_t st);

// gram_umma.cu: tcgen05 versions of the two tile passes for bf16 keys whose width is a multiple of 64
cudaError_t umma_configure(DeviceCfg *cfg);
bool umma_supported(int d_k);
// est_rows: an upper estimate of the survivors per image when the host has one (0: maxN)
cudaError_t launch_gram_umma(const Batch &bt, int maxN, const DeviceCfg &cfg, cudaStream_t st, int est_rows = 0);
cudaError_t launch_assign_umma(const Batch &bt, int maxN, bool kept_rows, const DeviceCfg &cfg, cudaStream_t st, bool labels = false,
                               bool pairs = false);
bool umma_pairs_for_assign(int maxN, int B, const DeviceCfg &cfg);
cudaError_t launch_members(const Batch &bt, int maxN, bool label_none, cudaStream_t st);   // label_none: where there is no centre the labels are written (-1)
cudaError_t launch_spread_umma(const Batch &bt, int maxN, const DeviceCfg &cfg, cudaStream_t st);

// small.cu: scores to member lists in one kernel, a cluster per image
cudaError_t small_configure(DeviceCfg *cfg);
bool small_fits(const Batch &bt, int maxN, bool umma, const DeviceCfg &cfg);
cudaError_t launch_small(const Batch &bt, bool in_bf16, bool umma, int rpp, int sweep_limit, cudaStream_t st);

// merge.cu
// member records in cluster order from label[] (from_best: labels are first formed from the nearest-centre
// pass, all tokens); csize, cticket and cnt_cb must be zero.  spin_limit bounds the wait of its barrier.
cudaError_t launch_lists(const Batch &bt, int maxN, bool bf16, bool from_best, int spin_limit, const DeviceCfg &cfg, cudaStream_t st);
int lists_kernels(int maxN, int B, bool from_best, const DeviceCfg &cfg);   // kernels launch_lists launches
cudaError_t launch_list_clear(const Batch &bt, cudaStream_t st);   // csize, cticket, cnt_cb and the counters
cudaError_t launch_merge(const Batch &bt, bool in_bf16, bool out_bf16, const DeviceCfg &cfg, cudaStream_t st);
cudaError_t merge_configure(DeviceCfg *cfg);
size_t merge_scratch_rows();               // rows of partial sums k_merge may need per image

}  // namespace pact
