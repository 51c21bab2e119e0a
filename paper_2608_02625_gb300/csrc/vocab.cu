// Step A2 -- per-position reduction over the vocabulary logits.
//
// For each row x of V logits (the confidences that edits are thresholded on:
// Table 10's refine threshold, Appendix C.4's confident edits):
//   m = max x,  argmax = lowest index attaining m,
//   S = sum exp(x - m),  lse = m + ln S,  conf = 1 / S  (= exp(m - lse)).
//
// An HBM-bound stream: every logit is read exactly once, 16 bytes per load,
// coalesced across the threads of a row; what lies before a row's first
// 16-byte boundary and after its last (rows packed under an odd vocabulary
// start anywhere) is loaded one element per thread beside the stream. Each
// thread keeps an online (max, first index, scaled sum) triple; the sum is
// rescaled only when a 16-byte vector raises the running maximum, and the
// exponentials go two at a time through the packed fp32 FMA and add of the
// sm_100 family, so that the instruction stream stays below what HBM delivers
// per SM. (Rows off 16-byte boundaries took scalar loads throughout before:
// 512 rows of 151553 bf16 94.5 us, now 27.8, as long as rows of 151552.)
// Who works on a row depends on its length and on how many there are
// (launch_typed): a warp, a CTA, or a thread-block cluster whose warps' parts
// meet in one CTA through distributed shared memory (no global scratch).
#include <cooperative_groups.h>

#include <cmath>
#include <cstdint>

#include "dlm_common.cuh"
#include "dlm_internal.h"

namespace cg = cooperative_groups;

namespace dlm {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr float kLog2e = 1.4426950408889634f;

struct Partial {
  float m;    // running maximum (exact logit value)
  int idx;    // lowest index attaining m
  float s;    // sum of exp(x - m)
};

// A scan starts from a maximum of -kPlain with nothing at it, so that entries far
// below any logit (-inf, or the type's lowest value, with which tokens are often
// suppressed) add exp2(-large) = 0 and never become the maximum that the terms are
// relative to: times log2(e) such a maximum overflows or is rounded by more than
// the logits' spread. A row whose maximum is not within (-kPlain, kPlain) is read
// again (scan_any).
constexpr float kPlain = 131072.f;  // 2^17

// Order-preserving map of fp32 to int (-0 below +0).
__device__ __forceinline__ int order_key(float x) {
  const int i = __float_as_int(x);
  return i ^ ((i >> 31) & 0x7FFFFFFF);
}

// Combines two partials; the lower index wins equal maxima.
__device__ __forceinline__ Partial combine(Partial a, Partial b) {
  Partial r;
  r.m = fmaxf(a.m, b.m);
  r.idx = a.m > b.m ? a.idx : b.m > a.m ? b.idx : min(a.idx, b.idx);
  r.s = a.s * (a.m == -INFINITY ? 0.f : ex2_approx((a.m - r.m) * kLog2e)) +
        b.s * (b.m == -INFINITY ? 0.f : ex2_approx((b.m - r.m) * kLog2e));
  return r;
}

// The warp's partials as one, in every lane; the lower index wins equal maxima.
// One reduction each for the maximum and the index, then the rescaled sums.
template <int kLanes = 32>
__device__ __forceinline__ Partial warp_reduce(Partial p) {
  const int k = __reduce_max_sync(0xffffffffu, order_key(p.m));
  Partial r;
  r.m = __int_as_float(k ^ ((k >> 31) & 0x7FFFFFFF));
  r.idx = __reduce_min_sync(0xffffffffu, p.m == r.m ? p.idx : 0x7FFFFFFF);
  // A partial without a finite entry has sum 0 (or NaN, which must stay).
  r.s = p.s * (p.m == -INFINITY ? 0.f : ex2_approx((p.m - r.m) * kLog2e));
#pragma unroll
  for (int o = kLanes / 2; o > 0; o >>= 1) r.s += __shfl_xor_sync(0xffffffffu, r.s, o);
  return r;
}

// 16 bytes of a stream read once. Not ld.global.nc, which is for data that nothing
// writes while the kernel is resident: the logits' writer may still run when this
// kernel starts (wait_for_previous).
__device__ __forceinline__ uint4 ld_stream16(const void* p) {
  uint4 v;
  asm volatile("ld.global.L1::no_allocate.L2::256B.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// Elements of one 16-byte vector as fp32.
template <bool BF16>
struct Vec;

template <>
struct Vec<true> {
  static constexpr int kN = 8;
  __device__ __forceinline__ static void unpack(uint4 v, float (&x)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      x[2 * j] = __uint_as_float(w[j] << 16);
      x[2 * j + 1] = __uint_as_float(w[j] & 0xFFFF0000u);
    }
  }
  __device__ __forceinline__ static float load1(const void* base, int64_t i) {
    uint16_t h = static_cast<const uint16_t*>(base)[i];
    return __uint_as_float(static_cast<uint32_t>(h) << 16);
  }
};

template <>
struct Vec<false> {
  static constexpr int kN = 4;
  __device__ __forceinline__ static void unpack(uint4 v, float (&x)[4]) {
    x[0] = __uint_as_float(v.x);
    x[1] = __uint_as_float(v.y);
    x[2] = __uint_as_float(v.z);
    x[3] = __uint_as_float(v.w);
  }
  __device__ __forceinline__ static float load1(const void* base, int64_t i) {
    return static_cast<const float*>(base)[i];
  }
};

// Folds one value x at element index e into p, in any order of the indices
// (a row's elements outside its vectors).
__device__ __forceinline__ void fold_edge(Partial& p, float x, int e) {
  if (x > p.m) {
    p.s = p.s * (p.m == -INFINITY ? 0.f : ex2_approx((p.m - x) * kLog2e)) + 1.f;
    p.m = x;
    p.idx = e;
  } else if (x != -INFINITY) {
    p.s += ex2_approx((x - p.m) * kLog2e);  // NaN stays NaN
    if (x == p.m) p.idx = min(p.idx, e);
  }
}

// The largest of a vector's values, and the first of its elements that has it.
template <int kN>
__device__ __forceinline__ float vec_max(const float (&x)[kN]) {
  if constexpr (kN == 8) return fmaxf(fmax3(fmax3(x[0], x[1], x[2]), fmax3(x[3], x[4], x[5]), x[6]), x[7]);
  else return fmaxf(fmax3(x[0], x[1], x[2]), x[3]);
}

template <int kN>
__device__ __forceinline__ int first_of(const float (&x)[kN], float vm) {
  int first = kN - 1;
#pragma unroll
  for (int j = kN - 1; j >= 0; --j)
    if (x[j] == vm) first = j;
  return first;
}

// Folds one 16-byte vector of kN values starting at element index e0: the
// vector's maximum first (raising the running maximum rescales the sum, which
// is rare), then the kN exponentials in pairs with packed fp32 FMA and add
// into the two-lane running sum s2. mL is the running maximum times log2(e).
template <int kN>
__device__ __forceinline__ void fold_vec(Partial& p, float& mL, float2& s2, const float (&x)[kN], int e0) {
  const float vm = vec_max<kN>(x);
  if (vm > p.m) {
    const float up = vm * kLog2e, f = ex2_approx(mL - up);
    s2 = make_float2(s2.x * f, s2.y * f);
    p.m = vm;
    p.idx = e0 + first_of<kN>(x, vm);
    mL = up;
  }
  const float2 k2 = make_float2(kLog2e, kLog2e), n2 = make_float2(-mL, -mL);
#pragma unroll
  for (int j = 0; j < kN; j += 2) {
    const float2 y = ffma2(make_float2(x[j], x[j + 1]), k2, n2);
    s2 = fadd2(s2, make_float2(ex2_approx(y.x), ex2_approx(y.y)));
  }
}

// The same for maxima of any size, from none (-inf): each value is subtracted from
// the maximum before it is scaled.
template <int kN>
__device__ __forceinline__ void fold_vec_any(Partial& p, const float (&x)[kN], int e0) {
  const float vm = vec_max<kN>(x);
  if (vm > p.m) {
    p.s = p.m == -INFINITY ? 0.f : p.s * ex2_approx((p.m - vm) * kLog2e);
    p.m = vm;
    p.idx = e0 + first_of<kN>(x, vm);
  }
  if (p.m != -INFINITY) {
    float t = 0.f;  // a vector's terms first: fewer roundings of the long sum
#pragma unroll
    for (int j = 0; j < kN; ++j) t += ex2_approx((x[j] - p.m) * kLog2e);
    p.s += t;
  }
}

// Reduces the block's partials into warp 0's return value.
__device__ __forceinline__ Partial block_reduce(Partial p) {
  __shared__ Partial warp_part[kWarps];
  p = warp_reduce(p);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane == 0) warp_part[warp] = p;
  __syncthreads();
  if (warp == 0) {
    p = lane < kWarps ? warp_part[lane] : Partial{-INFINITY, 0x7FFFFFFF, 0.f};
    p = warp_reduce<kWarps>(p);
  }
  return p;
}

// A row of V elements as a run of whole 16-byte vectors with up to kN - 1
// elements before and after it.
template <bool BF16>
struct Row {
  const char* base;
  const uint4* vec;  // first vector: element `head`
  int64_t nvec;
  int head, tail;
  static constexpr int kEsz = BF16 ? 2 : 4, kN = 16 / kEsz;
  __device__ __forceinline__ Row(const VocabArgs& a, int64_t r)
      : Row(static_cast<const char*>(a.logits) + r * a.row_stride * kEsz, a.V) {}
  __device__ __forceinline__ Row(const char* first, int64_t V) : base(first) {
    const int64_t before = static_cast<int64_t>((0 - reinterpret_cast<uintptr_t>(base)) & 15u) / kEsz;
    head = static_cast<int>(before < V ? before : V);
    vec = reinterpret_cast<const uint4*>(base + head * kEsz);
    nvec = (V - head) / kN;
    tail = static_cast<int>(V - head - nvec * kN);
  }
};

// The element outside the row's vectors that thread t of a row's threads owns:
// t < 8 before them, 8 <= t < 16 after them (-inf where there is none).
template <bool BF16>
__device__ __forceinline__ float load_edge(const Row<BF16>& row, int t, bool first, bool last, int64_t V, int* e) {
  *e = t < 8 ? t : static_cast<int>(V) - row.tail + t - 8;
  const bool mine = t < 8 ? first && t < row.head : last && t < 8 + row.tail;
  return mine ? Vec<BF16>::load1(row.base, *e) : -INFINITY;
}

// The sum of exp(x - m) from that of 2^(x log2(e) - mL): mL is m log2(e) rounded,
// and what the rounding took (d, up to half an ulp of mL, the same for every term) is
// put back, as e^d - 1 = d + d^2 / 2 (|d| < 2^-7 below kPlain): the root mean square
// error of conf at 1000 values a row goes from 2.1e-7 to 7e-8, at 300 rows of 151552 bf16
// from 2.9e-7 to 2.2e-7, at the same time.
__device__ __forceinline__ float sum_of(float m, float mL, float2 s2) {
  const float s = s2.x + s2.y, d = 0.69314718f * fmaf(-m, kLog2e, mL);
  return fmaf(s, fmaf(0.5f * d, d, d), s);
}

// Scans vectors [v_begin, v_end) of a row with kWidth threads, of which this
// is number t, kUnroll loads in flight.
template <bool BF16, int kWidth, int kUnroll>
__device__ __forceinline__ Partial scan_vectors(const Row<BF16>& row, int64_t v_begin, int64_t v_end, int t) {
  using VT = Vec<BF16>;
  constexpr int kN = VT::kN;
  Partial p{-kPlain, 0x7FFFFFFF, 0.f};
  float mL = -kPlain * kLog2e;
  float2 s2 = make_float2(0.f, 0.f);
  int64_t vi = v_begin + t;
  for (; vi + (kUnroll - 1) * kWidth < v_end; vi += kUnroll * kWidth) {
    uint4 raw[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) raw[u] = ld_stream16(row.vec + vi + u * kWidth);
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      float x[kN];
      VT::unpack(raw[u], x);
      fold_vec<kN>(p, mL, s2, x, row.head + static_cast<int>((vi + u * kWidth) * kN));
    }
  }
  // The last, partial round: its loads in flight together too.
  if (vi < v_end) {
    uint4 raw[kUnroll - 1];
#pragma unroll
    for (int u = 0; u < kUnroll - 1; ++u)
      if (vi + u * kWidth < v_end) raw[u] = ld_stream16(row.vec + vi + u * kWidth);
#pragma unroll
    for (int u = 0; u < kUnroll - 1; ++u) {
      if (vi + u * kWidth < v_end) {
        float x[kN];
        VT::unpack(raw[u], x);
        fold_vec<kN>(p, mL, s2, x, row.head + static_cast<int>((vi + u * kWidth) * kN));
      }
    }
  }
  p.s = sum_of(p.m, mL, s2);
  return p;
}

// A row whose maximum is not within (-kPlain, kPlain) again, by one warp, in every
// lane: 0.1 ms for a row of 151552. Out of line, after everything else and in few
// registers, as code for such rows costs all others where it is in their way: a look
// at each vector's maximum in the scan (256 rows of 151552 bf16 15.2 us, 16.0 to 17.6
// so), each thread's vectors read again behind its scan (1 row 3.2 / 3.4), all threads
// of the CTA here (15 rows of 2492 1.9 / 2.0), more loads in flight here, with which five
// CTAs of the staged scan no longer fit on an SM (740 rows of 8054 7.0 / 7.6).
template <bool BF16>
__device__ __noinline__ Partial scan_any(const char* base, int64_t V, int lane) {
  const Row<BF16> row(base, V);
  int e;
  const float edge = load_edge(row, lane, true, true, V, &e);
  Partial p{-INFINITY, 0x7FFFFFFF, 0.f};
  uint4 next = lane < row.nvec ? ld_stream16(row.vec + lane) : make_uint4(0, 0, 0, 0);
#pragma unroll 1
  for (int64_t v = lane; v < row.nvec; v += 32) {
    float x[Vec<BF16>::kN];
    Vec<BF16>::unpack(next, x);
    if (v + 32 < row.nvec) next = ld_stream16(row.vec + v + 32);
    fold_vec_any<Vec<BF16>::kN>(p, x, row.head + static_cast<int>(v * Vec<BF16>::kN));
  }
  fold_edge(p, edge, e);
  return warp_reduce(p);
}

// 16-byte asynchronous copy global -> shared (bypassing L1), and its groups.
__device__ __forceinline__ void cp_async16(void* smem_dst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16;" ::"r"(smem_u32(smem_dst)), "l"(gsrc) : "memory");
}
// The same copy, issued only once `after` holds its value: passing a register
// loaded from the destination slot orders the slot's read before its refill.
__device__ __forceinline__ void cp_async16_after(void* smem_dst, const void* gsrc, uint32_t after) {
  asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16;" ::"r"(smem_u32(smem_dst)), "l"(gsrc), "r"(after)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// scan_vectors of a whole row by a block with the loads staged through shared
// memory: each thread keeps kStages of its vectors in flight in its own slots
// of `ring` ([kStages][kThreads]), reads back only what it copied itself (so
// no block barrier), and refills a slot as soon as its value is in registers:
// twice the bytes in flight of the register-loaded scan, with no registers
// held for them.
template <bool BF16, int kStages>
__device__ __forceinline__ Partial scan_row_staged(const Row<BF16>& row, uint4* ring) {
  using VT = Vec<BF16>;
  constexpr int kN = VT::kN;
  Partial p{-kPlain, 0x7FFFFFFF, 0.f};
  float mL = -kPlain * kLog2e;
  float2 s2 = make_float2(0.f, 0.f);
  const int64_t first = threadIdx.x;
  const int nk = first < row.nvec ? static_cast<int>((row.nvec - first + kThreads - 1) / kThreads) : 0;
  uint4* mine = ring + threadIdx.x;
#pragma unroll
  for (int k = 0; k < kStages; ++k) {
    if (k < nk) cp_async16(mine + k * kThreads, row.vec + first + static_cast<int64_t>(k) * kThreads);
    cp_async_commit();
  }
  for (int k = 0; k < nk; ++k) {
    cp_async_wait<kStages - 1>();  // the group of vector k has landed
    uint4* slot = mine + (k % kStages) * kThreads;
    const uint4 v = *slot;
    if (k + kStages < nk) cp_async16_after(slot, row.vec + first + static_cast<int64_t>(k + kStages) * kThreads, v.w);
    cp_async_commit();
    float x[kN];
    VT::unpack(v, x);
    fold_vec<kN>(p, mL, s2, x, row.head + static_cast<int>((first + static_cast<int64_t>(k) * kThreads) * kN));
  }
  cp_async_wait<0>();
  p.s = sum_of(p.m, mL, s2);
  return p;
}

__device__ __forceinline__ void write_out(const VocabArgs& a, int64_t rowi, Partial p) {
  // A NaN entry makes the sum NaN; a row of only -inf leaves the maximum -inf.
  if (kCheckBounds && (isnan(p.s) || p.m == -INFINITY)) set_device_error(a.err, DLM_DEVERR_INPUT);
  a.argmax[rowi] = p.idx;
  a.conf[rowi] = 1.0f / p.s;
  a.lse[rowi] = p.m + logf(p.s);
}

// One CTA per row (grid-stride over rows). kStaged: the loads go through the
// shared-memory staging ring of scan_row_staged.
constexpr int kStages = 8;
template <bool BF16, bool kStaged>
__global__ void __launch_bounds__(kThreads, 4) vocab_rows_kernel(VocabArgs a) {
  __shared__ uint4 ring[kStaged ? kStages * kThreads : 1];
  wait_for_previous();
  for (int64_t rowi = blockIdx.x; rowi < a.N; rowi += gridDim.x) {
    const Row<BF16> row(a, rowi);
    int e;
    const float edge = load_edge(row, threadIdx.x, true, true, a.V, &e);
    Partial p = kStaged ? scan_row_staged<BF16, kStages>(row, ring) : scan_vectors<BF16, kThreads, 4>(row, 0, row.nvec, threadIdx.x);
    fold_edge(p, edge, e);
    p = block_reduce(p);
    if (threadIdx.x < 32 && !(fabsf(p.m) < kPlain)) p = scan_any<BF16>(row.base, a.V, threadIdx.x);
    if (threadIdx.x == 0) write_out(a, rowi, p);
    __syncthreads();
  }
}

// One warp per row: many short rows.
template <bool BF16>
__global__ void __launch_bounds__(kThreads, 4) vocab_short_rows_kernel(VocabArgs a) {
  wait_for_previous();
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * kWarps;
  for (int64_t rowi = static_cast<int64_t>(blockIdx.x) * kWarps + (threadIdx.x >> 5); rowi < a.N; rowi += warps) {
    const Row<BF16> row(a, rowi);
    int e;
    const float edge = load_edge(row, lane, true, true, a.V, &e);
    Partial p = scan_vectors<BF16, 32, 4>(row, 0, row.nvec, lane);
    fold_edge(p, edge, e);
    p = warp_reduce(p);
    if (!(fabsf(p.m) < kPlain)) p = scan_any<BF16>(row.base, a.V, lane);
    if (lane == 0) write_out(a, rowi, p);
  }
}

// Rows split over a cluster of `csize` CTAs: CTA c scans chunk c of the row,
// every warp stores its part in rank 0's shared memory, and one warp of rank 0
// combines them. Persistent: cluster k takes rows k, k + clusters, ..., so a
// launch is one wave of resident CTAs, with no per-row launch and ramp-up; the
// slots alternate between rows, so one cluster barrier per row suffices (rank
// 0 reads row i's parts before it scans row i + 1, whose barrier the other
// CTAs must pass before they overwrite that slot with row i + 2's).
constexpr int kMaxCluster = 16;
template <bool BF16>
__global__ void __launch_bounds__(kThreads, 4) vocab_cluster_kernel(VocabArgs a) {
  __shared__ Partial parts[2][kMaxCluster * kWarps];
  cg::cluster_group cluster = cg::this_cluster();
  const int csize = static_cast<int>(cluster.num_blocks());
  const int crank = static_cast<int>(cluster.block_rank());
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t nclusters = gridDim.x / csize;
  wait_for_previous();
  cluster.barrier_arrive();  // rank 0's shared memory may be written once every CTA runs
  int it = 0;
  for (int64_t rowi = blockIdx.x / csize; rowi < a.N; rowi += nclusters, ++it) {
    const Row<BF16> row(a, rowi);
    const int64_t per = (row.nvec + csize - 1) / csize;
    const int64_t v0 = crank * per < row.nvec ? crank * per : row.nvec;
    const int64_t v1 = v0 + per < row.nvec ? v0 + per : row.nvec;
    int e;
    const float edge = load_edge(row, threadIdx.x, crank == 0, crank == csize - 1, a.V, &e);
    Partial p = scan_vectors<BF16, kThreads, 4>(row, v0, v1, threadIdx.x);
    fold_edge(p, edge, e);
    p = warp_reduce(p);
    if (it == 0) cluster.barrier_wait();
    if (lane == 0) *cluster.map_shared_rank(&parts[it & 1][crank * kWarps + warp], 0) = p;
    cluster.sync();
    if (crank == 0 && warp == 0) {
      const int n = csize * kWarps;
      Partial q{-INFINITY, 0x7FFFFFFF, 0.f};
#pragma unroll
      for (int j = 0; j < kMaxCluster * kWarps; j += 32)
        if (j + lane < n) q = combine(q, parts[it & 1][j + lane]);
      q = warp_reduce(q);
      if (!(fabsf(q.m) < kPlain)) q = scan_any<BF16>(row.base, a.V, lane);
      if (lane == 0) write_out(a, rowi, q);
    }
  }
  if (it == 0) cluster.barrier_wait();
}

// Probability of a given token of each row: one gathered logit per row.
template <bool BF16>
__global__ void __launch_bounds__(256) token_prob_kernel(VocabArgs a, const int32_t* tokens, const float* lse,
                                                         float* prob) {
  wait_for_previous();
  const int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r >= a.N) return;
  const int32_t t = tokens[r];
  float p = 0.f;
  if (kCheckBounds && (t < 0 || t >= a.V)) set_device_error(a.err, DLM_DEVERR_INPUT);
  if (t >= 0 && t < a.V) {
    const int64_t off = r * a.row_stride + t;
    const float x = BF16 ? __bfloat162float(static_cast<const __nv_bfloat16*>(a.logits)[off])
                         : static_cast<const float*>(a.logits)[off];
    p = expf(x - lse[r]);
  }
  prob[r] = p;
}

// Dynamic shared memory with which no more than `places` CTAs of `kernel` fit on an
// SM (4 at most, none then). A grid of fewer CTAs than the SMs have places for is launched
// with no more places than it needs: its CTAs otherwise fill the SMs that the
// kernel before it leaves first, several to an SM, while others stay empty. Behind
// attention (a loop of 4 passes, 264 rows of 151552 bf16): 122 us, 92 so; 400 rows
// 129 / 109; 160 rows, clusters of 2, 82 / 77; 100 rows, clusters of 4, 67.6 / 65.6.
// No more of it than that takes, and on SMs set to the most shared memory
// (carveout_for): what is left of an SM's 228 KB (113 KB at one place, 76 at two, 57 at
// three) stays for the kernels of other streams, which all of it taken keeps out until
// the reduction ends.
template <typename K>
size_t smem_for(K kernel, int64_t places, size_t fixed) {
  constexpr size_t kSm = 228 * 1024;
  if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSm / 2 - fixed)) != cudaSuccess) return 0;
  return places < 4 ? kSm / (static_cast<size_t>(places) + 1) - fixed : 0;
}

// Only such launches: four CTAs an SM with their loads in registers need the L1 for
// what is in flight (56 rows of 151552 fp32 in clusters of 8 7.9 us, 8.4 without it).
int carveout_for(size_t smem) { return smem > 0 ? cudaSharedmemCarveoutMaxShared : -1; }

// One wave of clusters of (at most) `csize` CTAs, each taking rows in turn.
template <bool BF16>
int launch_cluster(const VocabArgs& a, int csize, int sms, cudaStream_t stream) {
  const auto kernel = vocab_cluster_kernel<BF16>;
  const void* k = reinterpret_cast<const void*>(kernel);
  int active = 0;
  while ((active = active_clusters(k, csize, kThreads, 0)) == 0 && csize > 1) csize /= 2;
  if (active == 0) return fail(DLM_ERR_CUDA, "vocab_confidence: no cluster launch fits the device");
  const int64_t nclusters = a.N < active ? a.N : active;
  size_t smem = 0;
  for (int64_t places = (nclusters * csize + sms - 1) / sms; places < 4; ++places) {
    smem = smem_for(kernel, places, sizeof(Partial) * 2 * kMaxCluster * kWarps);
    if (active_clusters(k, csize, kThreads, smem) >= nclusters) break;
    smem = 0;
  }
  const cudaError_t e = launch_carved(kernel, dim3(static_cast<unsigned>(nclusters * csize)), kThreads, smem, stream, csize, true, carveout_for(smem), a);
  if (e != cudaSuccess) return fail(DLM_ERR_CUDA, "vocab_confidence cluster launch: %s", cudaGetErrorString(e));
  return DLM_OK;
}

template <bool BF16>
int launch_typed(const VocabArgs& a, cudaStream_t stream) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t row_bytes = a.V * (BF16 ? 2 : 4);
  const int64_t resident = 4LL * sms;  // CTAs at 4 per SM
  // Who works on a row (us measured on this GPU, 152 SMs, bf16, from a CUDA graph):
  // * long rows, at most one per SM: a cluster, the larger the fewer rows there
  //   are, up to about 2.6 CTAs per SM (V = 151552, clusters of 16 / 8 / 4: 1 row
  //   3.4 / 3.8 / 4.9, 32 rows 5.4 / 4.8 / 5.4, 64 rows 8.7 / 6.9 / 6.5, 128 rows
  //   17 / 12 / 10.3, where a CTA per row takes 11.1; rows twice as long: 64 rows
  //   11.0 / 8.8 / 11.1, so 4 CTAs per SM for those);
  // * short rows, enough of them to fill the SMs with warps: a warp (V = 1000 x
  //   16384 rows 12.2 against 34 with a CTA per row, V = 4000 x 16384 27.9 against
  //   48, V = 8000 x 8192 26.1 against 33.9, V = 16000 x 4096 23.7 against 27.3;
  //   V = 32001 x 3000 36.2 against 34.4, and V = 4000 x 1000 the same either way);
  // * else a CTA, its loads staged through shared memory (200 rows 15.4, from
  //   registers 19.9, clusters of 4 15.7; 256 rows 15.7 / 20.6 / 17.5; 400 rows 21.8 /
  //   23.8; 16384 rows 681 / 722) except where one wave of CTAs fills all places
  //   (512 rows: 30.5 staged, 27.7 from registers).
  // Clusters of 16 up to 2.25 CTAs per SM (22 rows 4.9 us, 8 to a cluster 4.4; V = 300000
  // 6.4 / 6.0; 21 rows 4.4 either way, V = 300000 5.4 / 6.0), of rows of 150 KB and less up to
  // one CTA per SM (V = 40000, 16 rows 3.5 / 2.9; V = 64000 3.6 / 3.5), and no larger clusters
  // than all fit at once (fp32, 35 rows 7.3 us in clusters of 16, 5.4 of 8; 75 rows 13.0 of 8,
  // 11.8 of 4).
  // Around one row per SM (clusters of 4, of 2, a CTA per row): where the clusters of 4 no
  // longer all fit at once (152 rows 14.1 / 12.5 / 11.0, fp32 23.3 / 19.9 / 17.9) and, rows
  // of 200 KB and less in bf16, a little before (V = 100000, 100 rows 6.2 / 7.7 / 7.3, 136
  // rows 7.9 / 8.8 / 7.3; V = 40000, 136 rows 5.2 / 4.5 / 4.2, but fp32 5.6 / 6.5 / 5.5), a
  // CTA per row; past one row per SM some SMs have two rows and most one, which halves
  // of rows even out for long bf16 rows (160 rows 14.3 / 13.4 / 14.7, 200 rows 15.5 / 14.3 /
  // 15.0, 230 rows 16.9 / 15.8 / 15.1; V = 64000, 160 rows 7.7 / 6.8 / 7.4; fp32 160 rows
  // 23.6 / 20.3 / 19.2).
  if (row_bytes >= 65536 && a.N <= sms) {
    const int64_t ctas = row_bytes > 400000 ? resident : 2 * resident / 3;
    int csize = a.N * 16 <= (row_bytes > 150000 ? 9 * sms / 4 : sms) ? 16 : a.N * 8 <= ctas ? 8 : 4;
    while (csize > 4 && a.N > active_clusters(reinterpret_cast<const void*>(vocab_cluster_kernel<BF16>), csize, kThreads, 0)) csize /= 2;
    const int most = BF16 && row_bytes <= 200000 ? 3 * sms / 4
                                                 : active_clusters(reinterpret_cast<const void*>(vocab_cluster_kernel<BF16>), 4, kThreads, 0);
    if (csize > 4 || a.N <= most) return launch_cluster<BF16>(a, csize, sms, stream);
  } else if (BF16 && row_bytes >= 100000 && a.N > sms && 3 * a.N <= 4 * sms) {
    return launch_cluster<BF16>(a, 2, sms, stream);
  }
  cudaError_t e;
  const auto grid = [&](int64_t ctas) { return dim3(static_cast<unsigned>(ctas < 64 * resident ? ctas : 64 * resident)); };
  if (a.N > resident && (row_bytes <= 8192 || (row_bytes <= 40000 && a.N >= 24LL * sms)))
    e = launch_overlapped(vocab_short_rows_kernel<BF16>, grid((a.N + kWarps - 1) / kWarps), kThreads, 0, stream, 1, true, a);
  else if (a.N > 3LL * sms && a.N <= resident)
    e = launch_overlapped(vocab_rows_kernel<BF16, false>, grid(a.N), kThreads, 0, stream, 1, true, a);
  else {
    const size_t smem = smem_for(vocab_rows_kernel<BF16, true>, (a.N + sms - 1) / sms, sizeof(uint4) * kStages * kThreads);
    e = launch_carved(vocab_rows_kernel<BF16, true>, grid(a.N), kThreads, smem, stream, 1, true, carveout_for(smem), a);
  }
  if (e != cudaSuccess) return fail(DLM_ERR_CUDA, "vocab_confidence launch: %s", cudaGetErrorString(e));
  return DLM_OK;
}

}  // namespace

int launch_vocab_confidence(const VocabArgs& a, cudaStream_t stream) {
  if (a.N == 0) return DLM_OK;
  return a.is_bf16 ? launch_typed<true>(a, stream) : launch_typed<false>(a, stream);
}

int launch_token_prob(const VocabArgs& a, const int32_t* tokens, const float* lse, float* prob,
                      cudaStream_t stream) {
  if (a.N == 0) return DLM_OK;
  const auto kernel = a.is_bf16 ? token_prob_kernel<true> : token_prob_kernel<false>;
  const cudaError_t e = launch_overlapped(kernel, dim3(static_cast<unsigned>((a.N + 255) / 256)), 256, 0, stream, 1, true, a, tokens, lse, prob);
  if (e != cudaSuccess) return fail(DLM_ERR_CUDA, "token_prob launch: %s", cudaGetErrorString(e));
  return DLM_OK;
}

}  // namespace dlm
