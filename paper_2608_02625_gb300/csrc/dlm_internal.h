// Host-side interfaces between the C ABI layer (dlm_api.cu) and the kernel
// launchers. Arguments here are already validated.
#pragma once

#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>
#include <mutex>

#include "dlmrefine.h"

namespace dlm {

// Device address of the error word of the current device (set up once per device).
int* device_error_word();

// Budget of each bounded wait in the pipelined kernels (ns): 2 s, which no
// legitimate wait inside one launch approaches. Only DLM_CHECK_BOUNDS builds
// can change it (dlm_checked_set_wait_budget), to make waits run out in tests.
constexpr uint64_t kDefaultWaitBudgetNs = 2000000000ull;
uint64_t wait_budget_ns();
// Query tiles per attention work unit set on this thread (0: automatic).
int attn_tiles_per_unit();

// Records a failure message for dlm_last_error() and returns `status`.
int fail(int status, const char* fmt, ...);
// Clears the calling thread's failure message (at the start of every entry point).
void clear_error();
// The calling thread's stream (dlm_set_stream).
cudaStream_t current_stream();

// Answers kept by everything they depend on. A query that fails (ask() < 0)
// gives 0 for this time and is asked again the next.
struct ClusterSizes {
  const void* kernel;
  int dev, csize, threads;
  size_t smem;
  bool operator==(const ClusterSizes& o) const {
    return kernel == o.kernel && dev == o.dev && csize == o.csize && threads == o.threads && smem == o.smem;
  }
};

class ClusterTable {
 public:
  template <typename Ask>
  int get(const ClusterSizes& key, Ask ask) {
    std::lock_guard<std::mutex> lock(mu_);
    for (int i = 0; i < count_; ++i)
      if (keys_[i] == key) return answers_[i];
    const int n = ask();
    if (n < 0) return 0;
    if (count_ < kMax) {
      keys_[count_] = key;
      answers_[count_++] = n;
    }
    return n;
  }

 private:
  static constexpr int kMax = 256;  // past these a query is asked every time
  std::mutex mu_;
  ClusterSizes keys_[kMax];
  int answers_[kMax];
  int count_ = 0;
};

// Clusters of `csize` CTAs of `kernel` (`threads` each, `smem` bytes of dynamic
// shared memory, `csize` up to 16) that run at once on the current device, 0
// if none can; asked of the runtime once per device, kernel and sizes.
int active_clusters(const void* kernel, int csize, int threads, size_t smem);

// Launches a kernel that may start while the one before it in the stream still
// runs (every kernel launched so calls wait_for_previous), in clusters
// of `csize` CTAs; an ordinary launch where !overlap. carveout: how much of an SM's
// shared memory and L1 is to be shared memory, in percent (-1: the driver's choice).
template <typename... P, typename... A>
cudaError_t launch_carved(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream, int csize,
                          bool overlap, int carveout, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(static_cast<unsigned>(threads));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[3];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (csize > 1) {
    attr[cfg.numAttrs].id = cudaLaunchAttributeClusterDimension;
    attr[cfg.numAttrs++].val.clusterDim = {static_cast<unsigned>(csize), 1, 1};
  }
  if (carveout >= 0) {
    attr[cfg.numAttrs].id = cudaLaunchAttributePreferredSharedMemoryCarveout;
    attr[cfg.numAttrs++].val.sharedMemCarveout = static_cast<unsigned>(carveout);
  }
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

template <typename... P, typename... A>
cudaError_t launch_overlapped(void (*kernel)(P...), dim3 grid, int threads, size_t smem, cudaStream_t stream, int csize,
                              bool overlap, A... args) {
  return launch_carved(kernel, grid, threads, smem, stream, csize, overlap, -1, args...);
}

// The block size of the block masks as the kernels take it: a sequence of up to L
// positions fits in one block of L, and the sums of positions and blocks in
// key_ranges then stay below 2 L whatever size the caller gives.
inline int mask_block(int block, int64_t L) { return block < L ? block : static_cast<int>(L); }

struct AttnArgs {
  const void* q;
  const void* k;
  const void* v;
  void* out;
  const int32_t* seq_lens;  // may be null: n_b = L
  const int32_t* prompt_lens;  // may be null: p_b = 0 (block masks only)
  int mask_mode, block;        // DLM_ATTN_* and the block size (block masks)
  int B, L, Hq, Hkv, D;
  // strides in elements, (b, l, h) order; the innermost stride is 1
  int64_t sq[3], sk[3], sv[3], so[3];
};

int launch_attn_tc_bf16(const AttnArgs& a, cudaStream_t stream);  // tcgen05 path
int launch_attn_f32(const AttnArgs& a, cudaStream_t stream);      // fp32 CUDA-core path

struct VocabArgs {
  const void* logits;
  int is_bf16;
  int64_t N, V, row_stride;  // row stride in elements
  int32_t* argmax;
  float* conf;
  float* lse;
  int* err;  // device error word (input checks of DLM_CHECK_BOUNDS builds)
};

int launch_vocab_confidence(const VocabArgs& a, cudaStream_t stream);


struct UpdateArgs {
  const int32_t* tokens;
  const uint8_t* mask;
  const int32_t* argmax;
  const float* conf;
  int32_t* new_tokens;
  uint8_t* new_mask;
  int32_t* n_edits;
  int64_t s_tokens, s_mask, s_argmax, s_conf, s_new_tokens, s_new_mask;  // sequence strides
  int B, L;
  float edit_threshold;
  int32_t remask_k;
  float remask_frac;
  int32_t mask_id;
  const int32_t* prompt_lens;
  const int32_t* seq_lens;
  // Remask ranking by the resulting token's probability when non-null: the
  // probability of each position's current token, [B, L] with sequence stride s_tok_prob.
  const float* tok_prob;
  int64_t s_tok_prob;
};

int launch_refine_update(const UpdateArgs& a, cudaStream_t stream);
// The same right behind the launch_vocab_confidence that writes a.argmax and
// a.conf, on its stream: starts when that launch's CTAs have ended and waits for its end.
int launch_refine_update_after_vocab(const UpdateArgs& a, cudaStream_t stream);

// prob[r] = exp(logits[r, tokens[r]] - lse[r]) (0 for a token outside [0, V)).
int launch_token_prob(const VocabArgs& a, const int32_t* tokens, const float* lse, float* prob,
                      cudaStream_t stream);

// Vocabulary projection fused with the reduction: per row r of hidden [N, d]
// the argmax / conf / lse of hidden[r] . weight[v] over v < V.
struct LmArgs {
  const void* hidden;   // bf16 [N, d], row stride s_hidden elements
  const void* weight;   // bf16 [V, d], row stride s_weight elements
  int64_t N, V, d, s_hidden, s_weight;
  int32_t* argmax;
  float* conf;
  float* lse;
  void* workspace;      // lmhead_workspace_bytes(N)
};

constexpr int kLmMaxSplits = 64;  // parts per row in the workspace
inline size_t lmhead_workspace_bytes(int64_t N) { return static_cast<size_t>(N) * kLmMaxSplits * 12; }
int launch_lmhead(const LmArgs& a, cudaStream_t stream);

}  // namespace dlm
