// The vocabulary projection fused with step A2, on the tensor cores.
//
// Every revisable position's distribution over the vocabulary comes from the
// refiner's output projection of its final hidden state (Sec. 4.2):
// logits[r, v] = hidden[r, :] . weight[v, :]. This kernel computes, per row,
// what the vocabulary reduction of those logits computes (argmax with ties to
// the lowest index, maximum softmax probability, log-sum-exp) without ever
// writing the N x V logits to memory.
//
// Persistent CTAs (one per SM) walk work items = (vocabulary split, block of
// 128 rows); items are ordered split-major, so the CTAs running at the same
// time read the same weight tiles and those stay in L2. Per 128 x 256 output
// tile (128 x 128 or 128 x 64 where the vocabulary is too small for a tile of
// 256 columns on every SM):
//   warp 0     TMA producer: hidden box 128 x 64 and weight box 256 x 64 per
//              64-wide K step, through a 4-stage ring (48 KB a stage)
//   warp 1     tensor-memory allocator and MMA issuer (all lanes run the loop,
//              one lane elected per instruction):
//              tcgen05.mma kind::f16, M = 128, N = 256, K = 16, bf16 x bf16 ->
//              fp32 accumulators; two accumulators of 256 columns, so the
//              epilogue of a tile overlaps the K loop of the next
//   warps 4-7  epilogue: thread t owns row t (TMEM lane t); 32 columns at a
//              time it takes the chunk's maximum and first index, rescales its
//              running sum of exp(x - m) when the maximum grows, and adds the
//              chunk's terms (per-tile partial sums keep the fp32 sum short)
// At the end of an item each row's (max, first index, sum) is written to the
// caller's workspace; lmhead_combine_kernel merges the parts of a row (ties
// keep the lower index). The workspace has kLmMaxSplits parts per row, fewer
// than there are SMs: with one or two row blocks (a local window, a single
// position: bound by reading the weight) the vocabulary is split over clusters
// of CTAs, which merge their rows' parts through distributed shared memory
// before one part is written, so that every SM reads a share of the weight.
// Every mbarrier wait is
// bounded; on expiry the kernel sets DLM_DEVERR_TIMEOUT, drains and exits.
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_bf16.h>

#include <cmath>
#include <cstdint>
#include <mutex>

#include "dlm_common.cuh"
#include "dlm_internal.h"

namespace cg = cooperative_groups;

namespace dlm {
namespace {

constexpr int kBM = 128;          // rows per tile = TMEM lanes
constexpr int kBK = 64;           // K per stage: one 128-byte swizzle atom of bf16
constexpr int kThreads = 256;     // warp 0 TMA, warp 1 MMA, warps 4-7 epilogue
constexpr int kEpiWarp0 = 4;
constexpr int kABytes = kBM * kBK * 2;  // 16 KB (a stage of it holds LmParams::a_rows rows)
constexpr float kLog2e = 1.4426950408889634f;

// kBN: vocabulary columns per tile, 256, or 128 or 64 where the vocabulary has
// too few columns for a tile of 256 on every SM.
template <int kBN>
struct Smem {
  static constexpr int kStages = kBN == 256 ? 4 : kBN == 128 ? 6 : 8;  // 192 KB
  static constexpr int kBBytes = kBN * kBK * 2;
  alignas(1024) uint8_t a[kStages][kABytes];
  alignas(1024) uint8_t b[kStages][kBBytes];
  uint64_t full[kStages];     // stage loaded             (TMA -> MMA)
  uint64_t empty[kStages];    // stage read by its MMAs   (MMA -> TMA)
  uint64_t acc_full[2];       // accumulator complete     (MMA -> epilogue)
  uint64_t acc_empty[2];      // accumulator read out     (epilogue -> MMA)
  uint64_t done;              // every MMA completed      (teardown)
  float part_m[kBM], part_s[kBM];  // this CTA's part of each row, read by rank 0 of its cluster
  int part_idx[kBM];
  uint32_t tmem_base;
  int abort;
};

struct LmParams {
  int N, V, d;
  int row_blocks, vtiles, items;
  int csize;    // CTAs per cluster; above 1 a cluster runs one item
  int splits;   // vocabulary splits: csize per part written
  int a_rows;   // rows of the hidden box: 128, or N rounded up to 8 when smaller
  float* part_m;
  int* part_idx;
  float* part_s;
  int* err;
  uint64_t wait_ns;  // budget of each bounded wait
};

struct Item {
  int rb, part, t0, t1;  // row block, part written, vocabulary tiles [t0, t1)
};

// Share of cluster rank `rank` of work item `item` (a part and a row block).
__device__ __forceinline__ Item item_at(const LmParams& p, int item, int rank) {
  Item it;
  it.part = item / p.row_blocks;
  it.rb = item % p.row_blocks;
  const int split = it.part * p.csize + rank;
  it.t0 = static_cast<int>(static_cast<long long>(p.vtiles) * split / p.splits);
  it.t1 = static_cast<int>(static_cast<long long>(p.vtiles) * (split + 1) / p.splits);
  return it;
}

// Merges another part (m2, idx2, s2) of a row into (m, idx, s); the lower
// vocabulary index wins equal maxima.
__device__ __forceinline__ void merge_part(float& m, int& idx, float& s, float m2, int idx2, float s2) {
  if (m2 > m) {
    s = (m == -INFINITY ? 0.f : s * expf(m - m2)) + s2;
    m = m2;
    idx = idx2;
  } else if (m2 != -INFINITY) {
    s += s2 * expf(m2 - m);
    if (m2 == m) idx = min(idx, idx2);
  }
}

__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* abort, int* err,
                                          uint64_t budget_ns) {
  bool ok = mbar_wait_for(bar, parity, abort, err, budget_ns);
  return __all_sync(0xffffffffu, ok);
}

template <int kBN>
__global__ void __launch_bounds__(kThreads, 1)
    lmhead_kernel(const __grid_constant__ CUtensorMap th, const __grid_constant__ CUtensorMap tw, const LmParams p) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int kStages = Smem<kBN>::kStages, kBBytes = Smem<kBN>::kBBytes;
  constexpr uint32_t kTmemCols = 2 * kBN;  // two accumulators
  Smem<kBN>& sm = *reinterpret_cast<Smem<kBN>*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int kblocks = p.d / kBK;
  const int rank = static_cast<int>(blockIdx.x) % p.csize;
  const int walker = static_cast<int>(blockIdx.x) / p.csize, walkers = static_cast<int>(gridDim.x) / p.csize;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&sm.full[s], 1);
      mbar_init(&sm.empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sm.acc_full[i], 1);
      mbar_init(&sm.acc_empty[i], 128);
    }
    mbar_init(&sm.done, 1);
    sm.abort = 0;
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  if (warp == 1) {
    tmem_alloc(&sm.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;
  volatile int* abort = &sm.abort;
  wait_for_previous();

  if (warp == 0) {
    // ================================================================ TMA producer
    if (lane == 0) {
      prefetch_tmap(&th);
      prefetch_tmap(&tw);
    }
    int fill = 0;
    bool ok = true;
    for (int item = walker; ok && item < p.items; item += walkers) {
      const Item it = item_at(p, item, rank);
      for (int vt = it.t0; ok && vt < it.t1; ++vt) {
        for (int kb = 0; kb < kblocks; ++kb, ++fill) {
          const int st = fill % kStages;
          if (fill >= kStages && !warp_wait(&sm.empty[st], ((fill / kStages) - 1) & 1, abort, p.err, p.wait_ns)) {
            ok = false;
            break;
          }
          if (lane == 0) {
            mbar_arrive_expect_tx(&sm.full[st], p.a_rows * (kBK * 2) + kBBytes);
            tma_load_2d(sm.a[st], &th, &sm.full[st], kb * kBK, it.rb * kBM);
            tma_load_2d(sm.b[st], &tw, &sm.full[st], kb * kBK, vt * kBN);
          }
        }
      }
    }
    // Teardown: every copy issued lands before the block exits.
    if (lane == 0) {
      for (int s = 0; s < kStages; ++s) {
        const int n_s = fill > s ? (fill - s + kStages - 1) / kStages : 0;
        if (n_s) mbar_drain(&sm.full[s], (n_s - 1) & 1);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ================================================================ MMA issuer
    // All 32 lanes run the loop (warp-uniform waits); one lane elected inside
    // each MMA / commit issues it, with no branch around the MMAs.
    {
      constexpr uint32_t idesc = idesc_bf16_f32(kBM, kBN, false, false);  // both operands K-major
      // Descriptors of the first stage; the others are these plus constants (1024 rows x
      // 151552 x 512 113 -> 108 us, d = 2048 the same either way).
      const uint64_t a_desc0 = sdesc_sw128(smem_u32(sm.a[0]), 16, 1024), b_desc0 = sdesc_sw128(smem_u32(sm.b[0]), 16, 1024);
      int fill = 0, tile = 0;
      bool ok = true;
      for (int item = walker; ok && item < p.items; item += walkers) {
        const Item it = item_at(p, item, rank);
        for (int vt = it.t0; ok && vt < it.t1; ++vt, ++tile) {
          const int acc = tile & 1;
          // The accumulator's previous tile (tile - 2) must have been read out.
          if (tile >= 2 && !warp_wait(&sm.acc_empty[acc], ((tile >> 1) - 1) & 1, abort, p.err, p.wait_ns)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d_tmem = tmem + acc * kBN;
          for (int kb = 0; kb < kblocks; ++kb, ++fill) {
            const int st = fill % kStages;
            if (!warp_wait(&sm.full[st], (fill / kStages) & 1, abort, p.err, p.wait_ns)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t a_desc = a_desc0 + static_cast<uint32_t>(st) * (kABytes >> 4);
            const uint64_t b_desc = b_desc0 + static_cast<uint32_t>(st) * (kBBytes >> 4);
#pragma unroll
            for (int kk = 0; kk < kBK / 16; ++kk)
              mma_ss_elect(d_tmem, a_desc + kk * 2, b_desc + kk * 2, idesc, (kb > 0 || kk > 0) ? 1u : 0u);
            mma_commit_elect(&sm.empty[st]);
          }
          if (!ok) break;
          mma_commit_elect(&sm.acc_full[acc]);
        }
      }
      mma_commit_elect(&sm.done);
      mbar_drain(&sm.done, 0);
    }
    __syncwarp();
  } else if (warp >= kEpiWarp0) {
    // ================================================================ epilogue
    const int qw = warp - kEpiWarp0;                 // TMEM lanes 32 qw .. 32 qw + 31
    const int t = threadIdx.x - kEpiWarp0 * 32;      // row within the tile
    const uint32_t lane_base = static_cast<uint32_t>(qw * 32) << 16;
    int tile = 0;
    bool ok = true;
    for (int item = walker; ok && item < p.items; item += walkers) {
      const Item it = item_at(p, item, rank);
      float m = -INFINITY, s = 0.f;
      int idx = 0;
      const int row = it.rb * kBM + t;
      const bool rows = row - lane < p.N;  // some row of this warp exists
      for (int vt = it.t0; vt < it.t1; ++vt, ++tile) {
        const int acc = tile & 1;
        if (!warp_wait(&sm.acc_full[acc], (tile >> 1) & 1, abort, p.err, p.wait_ns)) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (!rows) {
          tc_fence_before();
          mbar_arrive(&sm.acc_empty[acc]);
          continue;
        }
        const uint32_t base = tmem + lane_base + acc * kBN;
        float ts = 0.f;  // this tile's terms, relative to m
#pragma unroll 1
        for (int c = 0; c < kBN / 32; ++c) {
          uint32_t v[32];
          tmem_ld32(base + 32 * c, v);
          tmem_wait_ld();
          if (c == kBN / 32 - 1) {
            tc_fence_before();
            mbar_arrive(&sm.acc_empty[acc]);  // every column of the accumulator has been read
          }
          const int col0 = vt * kBN + 32 * c;
          float x[32];
#pragma unroll
          for (int e = 0; e < 32; ++e) x[e] = __uint_as_float(v[e]);
          if (col0 + 32 > p.V) {
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if (col0 + e >= p.V) x[e] = -INFINITY;
          }
          // The chunk's maximum by three-input maxima, its index only where it raises the
          // row's (rare), exponentials two at a time: at small d the epilogue is what a
          // tile waits for (a compare and two selects per element: 4096 rows x 151552 x 512
          // 456 us, 382 so; d = 1024 758 / 739, d = 2048 1502 / 1489).
          float cm0 = fmaxf(x[0], x[1]), cm1 = fmaxf(x[2], x[3]);
#pragma unroll
          for (int e = 4; e < 32; e += 4) {
            cm0 = fmax3(cm0, x[e], x[e + 1]);
            cm1 = fmax3(cm1, x[e + 2], x[e + 3]);
          }
          const float cm = fmaxf(cm0, cm1);
          if (cm > m) {
            int ci = 31;
#pragma unroll
            for (int e = 30; e >= 0; --e)
              if (x[e] == cm) ci = e;
            const float a = m == -INFINITY ? 0.f : ex2_approx((m - cm) * kLog2e);
            s *= a;
            ts *= a;
            m = cm;
            idx = col0 + ci;
          }
          if (m != -INFINITY) {
            const float ml = m * kLog2e;
            const float2 k2 = make_float2(kLog2e, kLog2e), n2 = make_float2(-ml, -ml);
            float2 sum = make_float2(0.f, 0.f);
#pragma unroll
            for (int e = 0; e < 32; e += 2) {
              const float2 y = ffma2(make_float2(x[e], x[e + 1]), k2, n2);
              sum = fadd2(sum, make_float2(ex2_approx(y.x), ex2_approx(y.y)));
            }
            ts += sum.x + sum.y;
          }
        }
        s += ts;
      }
      if (!ok) break;
      if (p.csize > 1) {
        sm.part_m[t] = m;
        sm.part_idx[t] = idx;
        sm.part_s[t] = s;
      } else if (row < p.N) {
        const int64_t o = static_cast<int64_t>(it.part) * p.N + row;
        p.part_m[o] = m;
        p.part_idx[o] = idx;
        p.part_s[o] = s;
      }
    }
  }

  if (p.csize > 1) {
    // Rank 0 merges the cluster's parts of each row; the second barrier keeps
    // the other CTAs' shared memory alive until it has read them.
    cg::cluster_group cluster = cg::this_cluster();
    cluster.sync();
    if (rank == 0 && warp >= kEpiWarp0) {
      const Item it = item_at(p, walker, 0);
      const int t = threadIdx.x - kEpiWarp0 * 32, row = it.rb * kBM + t;
      if (row < p.N) {
        float m = sm.part_m[t], s = sm.part_s[t];
        int idx = sm.part_idx[t];
        for (int r = 1; r < p.csize; ++r)
          merge_part(m, idx, s, *cluster.map_shared_rank(&sm.part_m[t], r), *cluster.map_shared_rank(&sm.part_idx[t], r),
                     *cluster.map_shared_rank(&sm.part_s[t], r));
        const int64_t o = static_cast<int64_t>(it.part) * p.N + row;
        p.part_m[o] = m;
        p.part_idx[o] = idx;
        p.part_s[o] = s;
      }
    }
    cluster.sync();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// Merges the parts of each row, one warp per row: the parts' loads are all in
// flight at once. (One thread per row walking its 64 parts took ~40 us, the
// latency of a chain of loads, where the projection of 64 rows takes ~95.)
constexpr int kCombineThreads = 256;
__global__ void __launch_bounds__(kCombineThreads)
    lmhead_combine_kernel(const float* part_m, const int* part_idx, const float* part_s, int N, int parts,
                          int32_t* argmax, float* conf, float* lse) {
  wait_for_previous();
  const int64_t r = (static_cast<int64_t>(blockIdx.x) * kCombineThreads + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (r >= N) return;
  constexpr int kPer = kLmMaxSplits / 32;
  float pm[kPer], ps[kPer];
  int pi[kPer];
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int k = lane + 32 * j;
    const int64_t o = static_cast<int64_t>(k) * N + r;
    pm[j] = k < parts ? part_m[o] : -INFINITY;
    pi[j] = k < parts ? part_idx[o] : 0x7FFFFFFF;
    ps[j] = k < parts ? part_s[o] : 0.f;
  }
  float m = pm[0], s = ps[0];
  int idx = pi[0];
#pragma unroll
  for (int j = 1; j < kPer; ++j) merge_part(m, idx, s, pm[j], pi[j], ps[j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, o), s2 = __shfl_xor_sync(0xffffffffu, s, o);
    const int idx2 = __shfl_xor_sync(0xffffffffu, idx, o);
    merge_part(m, idx, s, m2, idx2, s2);
  }
  if (lane == 0) {
    argmax[r] = idx;
    conf[r] = 1.0f / s;
    lse[r] = m + logf(s);
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  });
  return fn;
}

// 2-D map over a [rows, d] bf16 matrix (row stride in elements), box d 64 x box_rows.
int make_map_2d(CUtensorMap* map, const void* base, int64_t rows, int d, int64_t row_stride, int box_rows) {
  EncodeTiledFn enc = encode_fn();
  if (!enc) return fail(DLM_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
  cuuint64_t dims[2] = {static_cast<cuuint64_t>(d), static_cast<cuuint64_t>(rows)};
  cuuint64_t strides[1] = {static_cast<cuuint64_t>(row_stride) * 2};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(kBK), static_cast<cuuint32_t>(box_rows)};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(DLM_ERR_CUDA, "cuTensorMapEncodeTiled failed (%d)", static_cast<int>(r));
  return DLM_OK;
}

}  // namespace

namespace {

struct Split {
  int bn, csize, parts;  // columns per tile, CTAs per cluster, parts per row
};

template <int kBN>
constexpr size_t smem_bytes() {
  return sizeof(Smem<kBN>) + 1024;
}

template <int kBN>
cudaError_t allow_smem() {
  return cudaFuncSetAttribute(lmhead_kernel<kBN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(smem_bytes<kBN>()));
}

// The split that leaves the busiest CTA the fewest columns (in tiles of 256;
// narrower tiles read the hidden rows more often: a column counts 1.12 in tiles of
// 128 and 1.36 in tiles of 64), plus a small cost per item (pipeline fill, flush). Narrow tiles win where 256 columns
// leave SMs without one: 16 rows x 1000 x 4096 24.3 -> 19.4 us, x 512 9.7 -> 7.5, 100 x
// 10000 x 2048 20.6 -> 16.7, 300 x 16000 x 2048 31.6 -> 30.2. Clusters (csize > 1) run
// one item each, all at once. Measured for 64 rows x 151552 x 2048 (reading the
// weight at the HBM copy rate: 93 us): 64 single CTAs 127 us, 64 clusters of 2
// 101 us, 50 of 3 101 us, 32 of 4 101 us; 37 of 4, which are not all resident at
// once, 141 us. 200 rows: 154 us with single CTAs, 117 us. From three row
// blocks on, single CTAs fill the SMs.
template <int kBN>
void choose_split(int64_t row_blocks, int64_t V, int sms, Split* best, double* best_cost) {
  const int64_t vtiles = (V + kBN - 1) / kBN;
  for (int c = 1; c <= 4; c *= 2) {
    if (c > 1 && row_blocks * kLmMaxSplits >= sms) break;  // single CTAs already fill the SMs
    const int64_t active =
        c == 1 ? sms : active_clusters(reinterpret_cast<const void*>(lmhead_kernel<kBN>), c, kThreads, smem_bytes<kBN>());
    for (int s = 1; s <= kLmMaxSplits && s <= (vtiles + c - 1) / c; ++s) {  // a cluster's last CTAs may have no tile
      const int64_t items = row_blocks * s;
      if (c > 1 && items > active) break;
      const int64_t rounds = (items + active - 1) / active;
      const double tile = kBN / 256.0 * (0.88 + 0.12 * 256 / kBN);
      const double cost = static_cast<double>(rounds) * (static_cast<double>((vtiles + s * c - 1) / (s * c)) * tile + 0.5);
      if (cost < *best_cost - 1e-9) {
        *best_cost = cost;
        *best = {kBN, c, s};
      }
    }
  }
}

template <int kBN>
int launch_tiles(const LmArgs& a, const Split& sp, int sms, cudaStream_t stream) {
  LmParams p;
  p.N = static_cast<int>(a.N);
  p.V = static_cast<int>(a.V);
  p.d = static_cast<int>(a.d);
  p.row_blocks = static_cast<int>((a.N + kBM - 1) / kBM);
  p.vtiles = static_cast<int>((a.V + kBN - 1) / kBN);
  p.a_rows = a.N < kBM ? static_cast<int>((a.N + 7) / 8 * 8) : kBM;
  p.csize = sp.csize;
  p.splits = sp.parts * sp.csize;
  p.items = p.row_blocks * sp.parts;
  float* ws = static_cast<float*>(a.workspace);
  p.part_m = ws;
  p.part_idx = reinterpret_cast<int*>(ws + static_cast<int64_t>(sp.parts) * a.N);
  p.part_s = ws + 2 * static_cast<int64_t>(sp.parts) * a.N;
  p.err = device_error_word();
  p.wait_ns = wait_budget_ns();
  CUtensorMap mh, mw;
  int st;
  if ((st = make_map_2d(&mh, a.hidden, a.N, p.d, a.s_hidden, p.a_rows)) != DLM_OK) return st;
  if ((st = make_map_2d(&mw, a.weight, a.V, p.d, a.s_weight, kBN)) != DLM_OK) return st;
  const int grid = sp.csize > 1 ? p.items * sp.csize : (p.items < sms ? p.items : sms);
  cudaError_t e = launch_overlapped(lmhead_kernel<kBN>, dim3(static_cast<unsigned>(grid)), kThreads, smem_bytes<kBN>(), stream,
                                    sp.csize, true, mh, mw, p);
  if (e != cudaSuccess) return fail(DLM_ERR_CUDA, "lmhead launch: %s", cudaGetErrorString(e));
  e = launch_overlapped(lmhead_combine_kernel, dim3(static_cast<unsigned>((a.N * 32 + kCombineThreads - 1) / kCombineThreads)),
                        kCombineThreads, 0, stream, 1, true, p.part_m, p.part_idx, p.part_s, p.N, sp.parts, a.argmax, a.conf, a.lse);
  if (e != cudaSuccess) return fail(DLM_ERR_CUDA, "lmhead combine launch: %s", cudaGetErrorString(e));
  return DLM_OK;
}

}  // namespace

int launch_lmhead(const LmArgs& a, cudaStream_t stream) {
  if (a.N == 0) return DLM_OK;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t row_blocks = (a.N + kBM - 1) / kBM;
  cudaError_t e = allow_smem<256>();
  if (e == cudaSuccess) e = allow_smem<128>();
  if (e == cudaSuccess) e = allow_smem<64>();
  if (e != cudaSuccess) return fail(DLM_ERR_CUDA, "lmhead smem attribute: %s", cudaGetErrorString(e));
  Split sp{256, 1, 1};
  double cost = 1e300;
  choose_split<256>(row_blocks, a.V, sms, &sp, &cost);
  choose_split<128>(row_blocks, a.V, sms, &sp, &cost);
  choose_split<64>(row_blocks, a.V, sms, &sp, &cost);
  if (sp.bn == 256) return launch_tiles<256>(a, sp, sms, stream);
  if (sp.bn == 128) return launch_tiles<128>(a, sp, sms, stream);
  return launch_tiles<64>(a, sp, sms, stream);
}

}  // namespace dlm
