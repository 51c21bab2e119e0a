// Step A3 -- the refine update (commit / edit / remask), one CTA per sequence.
//
// Sec. 4.2: the prompt stays fixed while any response position may be
// revised; the per-pass rule is token editing with confident edits
// (Appendix C.4, Table 11). For sequence b (response [p_b, n_b)):
//   1. prompt and padding are copied; masked response positions commit to the
//      argmax; filled ones whose argmax differs and whose conf >= tau are edited
//      (counted);
//   2. the k_b smallest (key(conf), index) response positions are remasked
//      (key: an order-preserving map of the fp32 bits, -0 -> +0; with tok_prob,
//      the key of the probability of the token each position holds after 1).
// Integer work and exact fp32 compares only: results are bit-exact.
//
// Bound by latency: a few KB per sequence, one chain of loads, a selection and
// stores. refine_update_kernel holds a sequence of up to 16 positions per
// thread in registers: every load of a thread is issued before any waits (by
// position, so that not even the lengths come first), the selection takes one
// barrier per 5 bits of the key and ends as soon as the remaining ties need no
// order, and each output is written once. From a CUDA graph: 8 x 2048 8.7 -> 6.4
// us, 32 x 512 5.8 -> 4.1, 4 x 64 5.6 -> 2.9, 1 x 8192 18.0 -> 13.6 against the walk in
// passes (refine_sequence, update_impl.cuh), which longer sequences still take.
#include <cmath>
#include <cstdint>

#include "dlm_common.cuh"
#include "dlm_internal.h"
#include "update_impl.cuh"

namespace dlm {
namespace {

// Lengths of sequence b, clamped into 0 <= p <= n <= L (recorded by thread 0).
__device__ __forceinline__ void lengths(const UpdateArgs& a, int b, int* err, int* n_out, int* p_out) {
  int n = a.seq_lens ? a.seq_lens[b] : a.L;
  int p = a.prompt_lens ? a.prompt_lens[b] : 0;
  bool clamped = false;
  if (n < 0 || n > a.L) { n = n < 0 ? 0 : a.L; clamped = true; }
  if (p < 0 || p > n) { p = p < 0 ? 0 : n; clamped = true; }
  if (clamped && threadIdx.x == 0) set_device_error(err, DLM_DEVERR_LENGTH);
  *n_out = n;
  *p_out = p;
}

__device__ __forceinline__ int remask_count(const UpdateArgs& a, int r) {
  const long long k = a.remask_k >= 0 ? static_cast<long long>(a.remask_k)
                                      : static_cast<long long>(floor(static_cast<double>(a.remask_frac) * static_cast<double>(r)));
  return static_cast<int>(k > r ? r : k);
}

// One sequence per CTA, position i = threadIdx.x + j * kThreads in registers of
// thread threadIdx.x (L <= kItems * kThreads). kAfterVocab: launched right behind
// the vocabulary reduction that writes argmax and conf; the tokens, masks and
// lengths, which it does not write, are loaded before the wait for its end (it
// lets this kernel start only after its own predecessor has ended).
template <int kThreads, int kItems, bool kAfterVocab>
__global__ void __launch_bounds__(kThreads) refine_update_kernel(UpdateArgs a, int* err) {
  constexpr int kWarps = kThreads / 32;
  __shared__ int count[2][kWarps][32];
  __shared__ int edits_of[kWarps];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x;
  const int items = (a.L + kThreads - 1) / kThreads;  // of the busiest thread

  if (!kAfterVocab) wait_for_previous();
  int tok[kItems], pred[kItems];
  uint8_t msk[kItems];
  float cf[kItems], tp[kItems];
  {
    const int32_t* tok_in = a.tokens + b * a.s_tokens;
    const uint8_t* msk_in = a.mask + b * a.s_mask;
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const int i = tid + j * kThreads;
      if (i < a.L) {
        tok[j] = tok_in[i];
        msk[j] = msk_in[i];
        tp[j] = a.tok_prob ? a.tok_prob[b * a.s_tok_prob + i] : 0.f;
      }
    }
  }
  int n, p;
  lengths(a, b, err, &n, &p);
  if (kAfterVocab) wait_for_previous();
  launch_dependents();
  {
    const int32_t* am = a.argmax + b * a.s_argmax;
    const float* conf = a.conf + b * a.s_conf;
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const int i = tid + j * kThreads;
      if (i < a.L) {
        pred[j] = kAfterVocab ? __ldcg(am + i) : am[i];
        cf[j] = kAfterVocab ? __ldcg(conf + i) : conf[i];
      }
    }
  }
  const int r = n - p, k = remask_count(a, r);

  // ---- commit / edit; the ranking key of each response position
  uint32_t key[kItems];
  int edits = 0;
  bool nan = false;
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    const int i = tid + j * kThreads;
    key[j] = 0;
    if (i >= p && i < n) {
      if (msk[j]) {
        tok[j] = pred[j];
      } else if (pred[j] != tok[j] && cf[j] >= a.edit_threshold) {
        tok[j] = pred[j];
        ++edits;
      }
      msk[j] = 0;
      const float v = a.tok_prob && tok[j] != pred[j] ? tp[j] : cf[j];
      nan |= v != v;
      key[j] = conf_key(v);
    }
  }
  edits = __reduce_add_sync(0xffffffffu, edits);
  if (lane == 0) edits_of[warp] = edits;

  // ---- the selection: positions whose key is below `bound`, and `ties` of those equal to it
  uint32_t prefix = 0, pmask = 0;
  int need = k;
  bool ordered = false;  // equal keys are left of which only the first `need` are taken
  if (k > 0 && k < r) {
    ordered = true;
    int buf = 0;
    for (int shift = 27; shift > -5; shift -= 5, buf ^= 1) {
      const int sh = shift < 0 ? 0 : shift;  // the last digit has two bits
      // Lane d counts this warp's keys of the current prefix whose next digit is d.
      int c = 0;
#pragma unroll
      for (int j = 0; j < kItems; ++j) {
        if (j >= items) break;
        const int i = tid + j * kThreads;
        uint32_t in = __ballot_sync(0xffffffffu, i >= p && i < n && (key[j] & pmask) == prefix);
        const uint32_t digit = (key[j] >> sh) & (shift < 0 ? 3u : 31u);
#pragma unroll
        for (int bit = 0; bit < 5; ++bit) {
          const uint32_t ones = __ballot_sync(0xffffffffu, (digit >> bit) & 1u);
          in &= (lane >> bit) & 1 ? ones : ~ones;
        }
        c += __popc(in);
      }
      count[buf][warp][lane] = c;
      __syncthreads();
      // Every warp adds up the warps' counts and finds the digit at which they reach `need`.
      int total = 0;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) total += count[buf][w][lane];
      int incl = total;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      const int d = __ffs(__ballot_sync(0xffffffffu, incl >= need)) - 1;
      const int in_digit = __shfl_sync(0xffffffffu, total, d);
      need -= __shfl_sync(0xffffffffu, incl, d) - in_digit;
      prefix |= static_cast<uint32_t>(d) << sh;
      pmask |= (shift < 0 ? 3u : 31u) << sh;
      if (need == in_digit) {  // all keys of this prefix are taken: their order does not matter
        ordered = false;
        break;
      }
    }
    if (nan) set_device_error(err, DLM_DEVERR_NAN);
  } else {
    __syncthreads();
  }
  if (tid == 0) {
    int total = 0;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) total += edits_of[w];
    a.n_edits[b] = total;
  }

  // ---- equal keys in index order: (j, warp, lane) is the order of the positions
  int before[kItems];
  if (ordered) {
    __syncthreads();  // `count` is read above
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const int i = tid + j * kThreads;
      const uint32_t eq = __ballot_sync(0xffffffffu, i >= p && i < n && key[j] == prefix);
      before[j] = __popc(eq & ((1u << lane) - 1u));
      if (lane == 0) (&count[0][0][0])[j * kWarps + warp] = __popc(eq);
    }
    __syncthreads();
    int sum = 0;
#pragma unroll
    for (int j = 0; j < kItems; ++j)
#pragma unroll 1
      for (int w = 0; w < kWarps; ++w) {
        if (w == warp) before[j] += sum;
        sum += (&count[0][0][0])[j * kWarps + w];
      }
  }

  // ---- write each position once
  int32_t* ntok = a.new_tokens + b * a.s_new_tokens;
  uint8_t* nmsk = a.new_mask + b * a.s_new_mask;
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    const int i = tid + j * kThreads;
    if (i >= a.L) continue;
    if (i >= p && i < n && k > 0) {
      const uint32_t top = key[j] & pmask;
      const bool take = k >= r || top < prefix || (top == prefix && (!ordered || before[j] < need));
      if (take) {
        tok[j] = a.mask_id;
        msk[j] = 1;
      }
    }
    ntok[i] = tok[j];
    nmsk[i] = msk[j];
  }
}

// Sequences of any length (update_impl.cuh).
constexpr int kLongThreads = 512;
__global__ void __launch_bounds__(kLongThreads) refine_update_long_kernel(UpdateArgs a, int* err) {
  __shared__ UpdateShared<kLongThreads> sh;
  wait_for_previous();
  launch_dependents();
  refine_sequence<kLongThreads>(a, blockIdx.x, err, sh);
}

template <bool kAfterVocab>
int launch(const UpdateArgs& a, cudaStream_t stream) {
  if (a.B == 0) return DLM_OK;
  const dim3 grid(static_cast<unsigned>(a.B));
  int* err = device_error_word();
  cudaError_t e;
  // The fewest threads that hold the sequence: fewer warps meet at each barrier (35
  // sequences of 2049 / 4096 / 8192 positions: 512 threads 6.9 / 8.8 / 16.0 us, 1024 threads with 8
  // positions each 10.0 / 11.4 / 17.7, the walk in passes 7.8 / 10.6 / 18.4).
  if (a.L <= 512) e = launch_overlapped(refine_update_kernel<128, 4, kAfterVocab>, grid, 128, 0, stream, 1, true, a, err);
  else if (a.L <= 2048) e = launch_overlapped(refine_update_kernel<256, 8, kAfterVocab>, grid, 256, 0, stream, 1, true, a, err);
  else if (a.L <= 4096) e = launch_overlapped(refine_update_kernel<512, 8, kAfterVocab>, grid, 512, 0, stream, 1, true, a, err);
  else if (a.L <= 8192) e = launch_overlapped(refine_update_kernel<512, 16, kAfterVocab>, grid, 512, 0, stream, 1, true, a, err);
  else e = launch_overlapped(refine_update_long_kernel, grid, kLongThreads, 0, stream, 1, true, a, err);
  if (e != cudaSuccess) return fail(DLM_ERR_CUDA, "refine_update launch: %s", cudaGetErrorString(e));
  return DLM_OK;
}

}  // namespace

int launch_refine_update(const UpdateArgs& a, cudaStream_t stream) { return launch<false>(a, stream); }

int launch_refine_update_after_vocab(const UpdateArgs& a, cudaStream_t stream) { return launch<true>(a, stream); }

}  // namespace dlm
