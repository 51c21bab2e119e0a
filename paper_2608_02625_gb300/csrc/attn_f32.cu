// Step A1, fp32 path -- non-causal GQA attention on the CUDA cores.
//
// Sec. 4.2: every valid position attends to every valid position (the block
// masks of dlm_attn_masked restrict each query to its key ranges). fp32
// inputs call for fp32 arithmetic throughout (TF32 tensor cores would not hold
// a 1e-5 error bound), so both products run as fp32 FMAs on register tiles.
//
// The query heads that share a key/value head form one list of rows, head
// after head (valid rows only), cut into tiles of 16 * kR rows, so that a tile
// may run from one head into the next and no head ends in a partial tile of its
// own (3 x 300, 32 / 4 heads: 129 us with tiles per head, 121 so). One CTA of
// 256 threads (16 x 16) computes a tile against 64-key tiles staged in shared
// memory: thread (ty, tx) owns the rows ty * kR .. + kR - 1 and, of the scores,
// the keys tx + 16 j; of the output, the columns 4 tx + 64 c .. + 3. The scores
// accumulate even and odd head-dim elements in the two halves of packed fp32
// FMAs (operands read as they lie in memory, 16 bytes a load); a row's scores
// belong to one half-warp, so its maximum is four shuffles and the numerators
// pass to the second product through a half-warp's own slice of shared memory
// without a block barrier. K and V have one buffer each: V_0 is copied beside
// K_0, V_t behind the scores of tile t, K_{t+1} behind its softmax and second
// product. Of the last key tile only the scores and products of the 16-key
// groups and 4-key groups that hold keys are computed (26 x 21 positions, 7 keys,
// block-local, D = 64: 9.1 us with whole tiles, 7.5 so; 8.3 with a warp per row).
//
// Bound by the FMA pipe: 80 % busy on the SMs that have a CTA (1 x 512, 32 / 4
// heads, D = 128: 148 tiles of 112 rows on 152 SMs, 92 us against 1022 us for a
// warp per query row; 8 x 512: 0.71 ms = 49 TFLOP/s).
#include <cmath>
#include <cstdint>
#include <type_traits>

#include "dlm_common.cuh"
#include "dlm_internal.h"

namespace dlm {
namespace {

constexpr int kThreads = 256;
constexpr int kKeys = 64;  // keys per tile

template <int D, int kR>
struct F32Tile {
  static constexpr int kM = 16 * kR;               // query rows per CTA
  static constexpr int kKStride = D + 4;           // floats; 16 lanes' rows then hit distinct banks
  static constexpr int kQGroup = kR * D + 4;       // one row group; two groups of a warp hit distinct banks
  static constexpr int kPRows = kR == 7 ? 8 : kR;  // rows of a key's numerators, padded to 16 bytes
  static constexpr int kPGroup = kKeys * kPRows + 4;  // numerators of one row group, [key][row]
  static constexpr int kQ = 16 * kQGroup, kK = kKeys * kKStride, kV = kKeys * D, kP = 16 * kPGroup;
  static constexpr size_t kBytes = sizeof(float) * (kQ + kK + kV + kP);
};

// `bytes` (16 or 4) from global to shared memory, zeros instead when !valid.
template <int kBytes>
__device__ __forceinline__ void copy_or_zero(float* dst, const float* src, bool valid) {
  const int n = valid ? kBytes : 0;
  if constexpr (kBytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(n) : "memory");
}

__device__ __forceinline__ void copy4(float* dst, const float* src, bool valid, bool vec) {
  if (vec) {
    copy_or_zero<16>(dst, src, valid);
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e) copy_or_zero<4>(dst + e, src + e, valid);
  }
}

__device__ __forceinline__ void store4(float* dst, float4 x, bool vec) {
  if (vec) *reinterpret_cast<float4*>(dst) = x;
  else dst[0] = x.x, dst[1] = x.y, dst[2] = x.z, dst[3] = x.w;
}

__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void copies_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ bool not_finite(float x) { return (__float_as_uint(x) & 0x7F800000u) == 0x7F800000u; }

// Whether the row tiles of sequences of `len` positions are cut per head.
__host__ __device__ __forceinline__ bool tiles_per_head(const AttnArgs& a, int len) {
  return a.mask_mode == DLM_ATTN_BLOCK_LOCAL && len > kKeys;
}

template <int D, int kR, bool kMasked>
__global__ void __launch_bounds__(kThreads, kR == 2 || (kR == 4 && D == 64) ? 2 : 1) attn_f32_kernel(AttnArgs a, float scale, bool vec, int* err) {
  using T = F32Tile<D, kR>;
  extern __shared__ float4 smem_f4[];
  float* const sq = reinterpret_cast<float*>(smem_f4);
  float* const sk = sq + T::kQ;
  float* const sv = sk + T::kK;
  float* const sp = sv + T::kV;
  __shared__ int2 row_of[T::kM];
  constexpr int kC4 = D / 4;    // 16-byte chunks per row
  constexpr int kCols = D / 64;  // float4 output columns per thread

  wait_for_previous();
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int g = blockIdx.y, b = blockIdx.z;
  const int G = a.Hq / a.Hkv;
  int n = a.seq_lens ? a.seq_lens[b] : a.L;
  int p = kMasked && a.prompt_lens ? a.prompt_lens[b] : 0;
  if (n < 0 || n > a.L) {
    if (tid == 0) set_device_error(err, DLM_DEVERR_LENGTH);
    n = n < 0 ? 0 : a.L;
  }
  if (kMasked && (p < 0 || p > n)) {
    if (tid == 0 && n > 0) set_device_error(err, DLM_DEVERR_LENGTH);
    p = p < 0 ? 0 : n;
  }
  const float* qb = static_cast<const float*>(a.q) + b * a.sq[0];
  const float* kb = static_cast<const float*>(a.k) + b * a.sk[0] + g * a.sk[2];
  const float* vb = static_cast<const float*>(a.v) + b * a.sv[0] + g * a.sv[2];
  float* const ob = static_cast<float*>(a.out) + b * a.so[0];

  // The group's rows: head after head, each n rows, or n rounded up to whole
  // tiles under the block-local mask (a tile that ran from one head into the
  // next would visit the blocks at both ends; where all keys are one tile that
  // does not matter).
  const int per = kMasked && tiles_per_head(a, n) ? (n + T::kM - 1) / T::kM * T::kM : n;
  const int rows = G * per, row0 = blockIdx.x * T::kM;  // below 2^31: checked by the launcher
  // Padding rows of the group's heads are zeros: written by the CTAs without a
  // tile, or where there are none by all of them when they are done.
  const int used = (rows + T::kM - 1) / T::kM, first_idle = used < static_cast<int>(gridDim.x) ? used : 0;
  auto write_padding = [&] {
    if (static_cast<int>(blockIdx.x) < first_idle) return;
    const int pad = a.L - n;
    for (int64_t e = static_cast<int64_t>(blockIdx.x - first_idle) * kThreads + tid; e < static_cast<int64_t>(G) * pad * kC4;
         e += static_cast<int64_t>(gridDim.x - first_idle) * kThreads) {
      const int z = static_cast<int>(e / kC4), head = z / pad;
      store4(ob + (g * G + head) * a.so[2] + (n + z - head * pad) * a.so[1] + e % kC4 * 4, make_float4(0.f, 0.f, 0.f, 0.f), vec);
    }
  };
  if (row0 >= rows) {
    write_padding();
    return;
  }
  // Row r of the tile: head and position (-1 past the head's last row).
  if (tid < T::kM) {
    const int rr = row0 + tid, head = rr / per, pos = rr - head * per;
    row_of[tid] = rr < rows && pos < n ? make_int2(g * G + head, pos) : make_int2(0, -1);
  }
  __syncthreads();

  // Key tiles the CTA's rows may use: tile t starts at key 64 * (t < ka ? t : t + gap).
  int tiles = (n + kKeys - 1) / kKeys, ka = tiles, gap = 0;
  KeyRanges first{n, n, n}, last{n, n, n};  // of the CTA's lowest and highest position
  if (kMasked) {
    const int end = min(row0 + T::kM, rows) - 1;
    const bool one_head = row0 / per == end / per;
    const int r_first = one_head ? row0 % per : 0, r_last = one_head ? min(end % per, n - 1) : n - 1;
    first = key_ranges(a.mask_mode, a.block, r_first, n, p);
    last = key_ranges(a.mask_mode, a.block, r_last, n, p);
    if (a.mask_mode == DLM_ATTN_BLOCK_CAUSAL || r_last < p) {
      ka = tiles = (last.hi1 + kKeys - 1) / kKeys;
    } else {
      const int prompt_end = (p + kKeys - 1) / kKeys;
      const int own = (r_first < p ? p : first.lo2) / kKeys, own_end = (last.hi2 + kKeys - 1) / kKeys;
      if (own <= prompt_end) {
        ka = tiles = max(prompt_end, own_end);
      } else {
        ka = prompt_end;
        gap = own - prompt_end;
        tiles = prompt_end + own_end - own;
      }
    }
  }
  // This thread's rows' keys: [0, hi1) and [lo2, hi2).
  int hi1[kMasked ? kR : 1], lo2[kMasked ? kR : 1], hi2[kMasked ? kR : 1];
  if (kMasked) {
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const KeyRanges kr = key_ranges(a.mask_mode, a.block, max(row_of[ty * kR + r].y, 0), n, p);
      hi1[r] = kr.hi1;
      lo2[r] = kr.lo2;
      hi2[r] = kr.hi2;
    }
  }

  float2 o[kR][2 * kCols];
  float m[kR], l[kR];  // running maximum; this thread's part of the row sum
#pragma unroll
  for (int r = 0; r < kR; ++r) {
    m[r] = -INFINITY;
    l[r] = 0.f;
#pragma unroll
    for (int c = 0; c < 2 * kCols; ++c) o[r][c] = make_float2(0.f, 0.f);
  }

  auto load_keys = [&](float* dst, int stride, const float* base, int64_t s_row, int key0) {
#pragma unroll
    for (int e = 0; e < kKeys * kC4 / kThreads; ++e) {
      const int i = tid + e * kThreads, key = i / kC4, c = i % kC4;
      const bool valid = key0 + key < n;
      copy4(dst + key * stride + 4 * c, base + (valid ? (key0 + key) * s_row + 4 * c : 0), valid, vec);
    }
  };
  auto key_of = [&](int t) { return kKeys * (t < ka ? t : t + gap); };

  for (int i = tid; i < T::kM * kC4; i += kThreads) {
    const int r = i / kC4, c = i % kC4;
    const int2 at = row_of[r];
    copy4(sq + (r / kR) * T::kQGroup + (r % kR) * D + 4 * c,
          qb + (at.y >= 0 ? at.x * a.sq[2] + at.y * a.sq[1] + 4 * c : 0), at.y >= 0, vec);
  }
  load_keys(sk, T::kKStride, kb, a.sk[1], key_of(0));
  copies_commit();
  load_keys(sv, D, vb, a.sv[1], key_of(0));
  copies_commit();
  copies_wait<1>();
  __syncthreads();
  const float* const q_mine = sq + ty * T::kQGroup;
  float* const p_mine = sp + ty * T::kPGroup;
  for (int t = 0; t < tiles; ++t) {
    const int key0 = key_of(t);
    if (t > 0) load_keys(sv, D, vb, a.sv[1], key0);
    copies_commit();
    // ---- scores of keys key0 + tx + 16 j
    float2 s2[kR][4];
#pragma unroll
    for (int r = 0; r < kR; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j) s2[r][j] = make_float2(0.f, 0.f);
    // The first kGroups * 16 keys of the tile.
    auto scores = [&](auto groups) {
      constexpr int kGroups = decltype(groups)::value;
#pragma unroll 4
      for (int c = 0; c < kC4; ++c) {
        float4 kf[kGroups];
#pragma unroll
        for (int j = 0; j < kGroups; ++j) kf[j] = *reinterpret_cast<const float4*>(sk + (tx + 16 * j) * T::kKStride + 4 * c);
#pragma unroll
        for (int r = 0; r < kR; ++r) {
          const float4 qf = *reinterpret_cast<const float4*>(q_mine + r * D + 4 * c);
#pragma unroll
          for (int j = 0; j < kGroups; ++j) {
            s2[r][j] = ffma2(make_float2(qf.x, qf.y), make_float2(kf[j].x, kf[j].y), s2[r][j]);
            s2[r][j] = ffma2(make_float2(qf.z, qf.w), make_float2(kf[j].z, kf[j].w), s2[r][j]);
          }
        }
      }
    };
    if (n - key0 > 32) scores(std::integral_constant<int, 4>());
    else if (n - key0 > 16) scores(std::integral_constant<int, 2>());
    else scores(std::integral_constant<int, 1>());
    __syncthreads();  // every warp is done with K_t
    if (t + 1 < tiles) load_keys(sk, T::kKStride, kb, a.sk[1], key_of(t + 1));
    copies_commit();
    // ---- online softmax; numerators to the half-warp's slice
    // Whether some row of the CTA may not use some key of the tile.
    const bool partial = kMasked ? !all_rows_use(first, last, key0, key0 + kKeys) : key0 + kKeys > n;
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      float s[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) s[j] = (s2[r][j].x + s2[r][j].y) * scale;
      if (partial) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int key = key0 + tx + 16 * j;
          const bool ok = kMasked ? key < hi1[r] || (key >= lo2[r] && key < hi2[r]) : key < n;
          if (!ok) s[j] = -INFINITY;
        }
      }
      float mx = fmaxf(fmaxf(s[0], s[1]), fmaxf(s[2], s[3]));
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      const float m_new = fmaxf(m[r], mx);
      // No key so far (every one masked): subtract 0, so that the numerators are exp(-inf) = 0.
      const float sub = kMasked && m_new == -INFINITY ? 0.f : m_new;
      const float corr = expf(m[r] - sub);  // 0 on the row's first keys (m = -inf)
      m[r] = m_new;
#pragma unroll
      for (int j = 0; j < 4; ++j) s[j] = expf(s[j] - sub);
      l[r] = l[r] * corr + ((s[0] + s[1]) + (s[2] + s[3]));
#pragma unroll
      for (int c = 0; c < 2 * kCols; ++c) o[r][c] = fmul2(o[r][c], make_float2(corr, corr));
#pragma unroll
      for (int j = 0; j < 4; ++j) s2[r][j].x = s[j];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float* dst = p_mine + (tx + 16 * j) * T::kPRows;
      if constexpr (kR >= 4) {
#pragma unroll
        for (int r = 0; r < kR; r += 4)
          *reinterpret_cast<float4*>(dst + r) =
              make_float4(s2[r][j].x, s2[r + 1][j].x, s2[r + 2][j].x, r + 3 < kR ? s2[r + 3 < kR ? r + 3 : 0][j].x : 0.f);
      } else {
        *reinterpret_cast<float2*>(dst) = make_float2(s2[0][j].x, s2[1][j].x);
      }
    }
    copies_wait<1>();  // V_t has landed (K_{t+1} may be in flight)
    // A key a row may not use must not reach it, whatever its V holds: a zero
    // numerator does not cancel a NaN or an infinity. (Rows past n are zeros
    // in shared memory.) Each thread looks at what it copied itself.
    bool guard = false;
    if (kMasked && partial) {
#pragma unroll
      for (int e = 0; e < kKeys * kC4 / kThreads; ++e) {
        const float4 x = reinterpret_cast<const float4*>(sv)[tid + e * kThreads];
        guard |= not_finite(x.x) | not_finite(x.y) | not_finite(x.z) | not_finite(x.w);
      }
      guard = __syncthreads_or(guard);
    } else {
      __syncthreads();
    }
    // ---- output += numerators x V
    if (!guard) {
      const int kend = min(kKeys, n - key0);  // the numerators and values past it are zeros
#pragma unroll 1
      for (int k4 = 0; k4 < kend; k4 += 4) {
#pragma unroll
        for (int key = k4; key < k4 + 4; ++key) {
          float pr[kR];
          if constexpr (kR >= 4) {
#pragma unroll
            for (int r = 0; r < kR; r += 4) {
              const float4 x = *reinterpret_cast<const float4*>(p_mine + key * T::kPRows + r);
              pr[r] = x.x, pr[r + 1] = x.y, pr[r + 2] = x.z;
              if (r + 3 < kR) pr[r + 3 < kR ? r + 3 : 0] = x.w;
            }
          } else {
            const float2 x = *reinterpret_cast<const float2*>(p_mine + key * T::kPRows);
            pr[0] = x.x, pr[1] = x.y;
          }
#pragma unroll
          for (int c = 0; c < kCols; ++c) {
            const float4 vf = *reinterpret_cast<const float4*>(sv + key * D + 64 * c + 4 * tx);
#pragma unroll
            for (int r = 0; r < kR; ++r) {
              o[r][2 * c] = ffma2(make_float2(pr[r], pr[r]), make_float2(vf.x, vf.y), o[r][2 * c]);
              o[r][2 * c + 1] = ffma2(make_float2(pr[r], pr[r]), make_float2(vf.z, vf.w), o[r][2 * c + 1]);
            }
          }
        }
      }
    } else {
#pragma unroll 1
      for (int key = 0; key < kKeys; ++key) {
        const int kpos = key0 + key;
#pragma unroll
        for (int r = 0; r < kR; ++r) {
          if (!(kpos < hi1[kMasked ? r : 0] || (kpos >= lo2[kMasked ? r : 0] && kpos < hi2[kMasked ? r : 0]))) continue;
          const float w = p_mine[key * T::kPRows + r];
#pragma unroll
          for (int c = 0; c < kCols; ++c) {
            const float4 vf = *reinterpret_cast<const float4*>(sv + key * D + 64 * c + 4 * tx);
            o[r][2 * c] = ffma2(make_float2(w, w), make_float2(vf.x, vf.y), o[r][2 * c]);
            o[r][2 * c + 1] = ffma2(make_float2(w, w), make_float2(vf.z, vf.w), o[r][2 * c + 1]);
          }
        }
      }
    }
    copies_wait<0>();
    __syncthreads();  // K_{t+1} is visible, V_t and the numerators are free
  }

#pragma unroll
  for (int r = 0; r < kR; ++r) {
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) l[r] += __shfl_xor_sync(0xffffffffu, l[r], off);
    const int2 at = row_of[ty * kR + r];
    if (at.y < 0) continue;
    float* dst = ob + at.x * a.so[2] + at.y * a.so[1] + 4 * tx;
    const float inv = 1.0f / l[r];
#pragma unroll
    for (int c = 0; c < kCols; ++c) {
      const float2 lo = o[r][2 * c], hi = o[r][2 * c + 1];
      store4(dst + 64 * c, make_float4(lo.x * inv, lo.y * inv, hi.x * inv, hi.y * inv), vec);
    }
  }
  write_padding();
}

template <int D, int kR, bool kMasked>
int launch_tile(const AttnArgs& a, bool vec, cudaStream_t stream) {
  using T = F32Tile<D, kR>;
  const float scale = 1.0f / sqrtf(static_cast<float>(D));
  cudaError_t e = cudaFuncSetAttribute(attn_f32_kernel<D, kR, kMasked>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(T::kBytes));
  if (e != cudaSuccess) return fail(DLM_ERR_CUDA, "attn_f32 smem attribute: %s", cudaGetErrorString(e));
  const int64_t G = a.Hq / a.Hkv;
  const int64_t tiles = tiles_per_head(a, a.L) ? G * ((a.L + T::kM - 1) / T::kM) : (G * a.L + T::kM - 1) / T::kM;
  const dim3 grid(static_cast<unsigned>(tiles), a.Hkv, a.B);
  e = launch_overlapped(attn_f32_kernel<D, kR, kMasked>, grid, kThreads, T::kBytes, stream, 1, true, a, scale, vec, device_error_word());
  if (e != cudaSuccess) return fail(DLM_ERR_CUDA, "attn_f32 launch: %s", cudaGetErrorString(e));
  return DLM_OK;
}

template <int D, bool kMasked>
int launch_d(const AttnArgs& a, cudaStream_t stream) {
  // 16-byte copies and stores where every base and stride allows them.
  bool vec = true;
  const void* base[4] = {a.q, a.k, a.v, a.out};
  const int64_t* strides[4] = {a.sq, a.sk, a.sv, a.so};
  for (int t = 0; t < 4; ++t) {
    vec &= reinterpret_cast<uintptr_t>(base[t]) % 16 == 0;
    for (int i = 0; i < 3; ++i) vec &= strides[t][i] % 4 == 0;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // Query rows per CTA (16 kR): the kR whose busiest SM is done first. In units
  // of one 128-row CTA, a 112-row one takes 0.94, a 64-row one 0.7 and a 32-row one
  // 0.55 alone on an SM; a further one beside it adds as much, but 0.54 for 64 rows
  // at D = 64, where two fit, and 0.44 for 32. Measured at D = 128, 32 heads, per
  // 64-key tile: 13.1 / 9.1 / 7.0 us alone for 128 / 64 / 32 rows, 11.5 us for two
  // 32-row CTAs; whole calls: L = 512 100 / 92 / 136 / 175 us with 128 / 112 / 64 / 32
  // rows, L = 256 53 / - / 33 / 46, L = 128 28 / - / 20 / 14.
  const int64_t G = a.Hq / a.Hkv;
  if (G * (a.L + 128LL) > 0x7FFFFFFFLL) return fail(DLM_ERR_SHAPE, "too many query rows per key/value head");
  auto tiles = [&](int m) {
    return tiles_per_head(a, a.L) ? G * ((a.L + m - 1) / m) : (G * a.L + m - 1) / m;
  };
  // Under the block-local mask a tile of fewer rows also visits fewer key tiles: the
  // prompt's (taken as L / 16 keys) and those its rows' blocks touch (40 x 256, 8 / 2 heads,
  // D = 64 146 us with 128 rows, 123 with 64; 1 x 512, 32 / 4, D = 64 34 / 27; 8 x 367 with 170
  // positions, 4 / 1, 39 with 112, 35 with 32).
  auto key_tiles = [&](int m) {
    if (!kMasked || a.mask_mode != DLM_ATTN_BLOCK_LOCAL) return 1.0;
    return fmin((a.L + kKeys - 1) / kKeys, a.L / (16.0 * kKeys) + 1.0 + (m + a.block - 1.0) / kKeys);
  };
  auto cost = [&](int m, double alone, double more) {
    return (alone + (ceil(static_cast<double>(tiles(m)) * a.B * a.Hkv / sms) - 1.0) * more) * key_tiles(m);
  };
  // 112 rows only where they make more tiles (7 x 150, 8 heads each its own: the same
  // 112 CTAs either way, 20.0 us with 128 rows and 23.8 with 112).
  const double c8 = cost(128, 1.0, 1.0), c7 = tiles(112) > tiles(128) ? cost(112, 0.94, 0.94) : 1e300,
               c4 = cost(64, 0.7, D == 64 ? 0.54 : 0.7), c2 = cost(32, 0.55, 0.44);
  const double best = fmin(fmin(c8, c7), fmin(c4, c2));
  if (c8 == best) return launch_tile<D, 8, kMasked>(a, vec, stream);
  if (c7 == best) return launch_tile<D, 7, kMasked>(a, vec, stream);
  if (c4 == best) return launch_tile<D, 4, kMasked>(a, vec, stream);
  return launch_tile<D, 2, kMasked>(a, vec, stream);
}

}  // namespace

int launch_attn_f32(const AttnArgs& a, cudaStream_t stream) {
  if (a.B == 0 || a.L == 0) return DLM_OK;
  if (a.mask_mode != DLM_ATTN_FULL)
    return a.D == 64 ? launch_d<64, true>(a, stream) : launch_d<128, true>(a, stream);
  return a.D == 64 ? launch_d<64, false>(a, stream) : launch_d<128, false>(a, stream);
}

}  // namespace dlm
