// Per-query top-K of influence scores (App. C ranks the stored examples of
// each query by score, descending, and reads the first 20 for NDCG@20).
// Order: score descending, equal scores by lower stored index; NaN scores
// never rank; missing places are (-inf, -1).
//
// Two kernels:
// * k_topk_select ranks one slice (at most 16,384 values) of one row of scores per
//   block. The block holds the slice as order keys in registers (32 a thread,
//   16-byte loads) and reads it once: the K-th largest of the 512 threads' own
//   maxima is a lower bound on the slice's K-th score, so the keys at or above it
//   hold the answer and are few (about K of them for scores in no particular
//   order); they are collected in shared memory and each finds its own rank among
//   them by comparison. Should they not fit (scores sorted so that few threads
//   hold all the best, or many equal ones), the exact K-th largest (score, place)
//   is built bit by bit from the top by counting. Rows of several slices are
//   ranked by the same kernel over the slices' lists, laid out as shorter rows.
//   Bound by reading the scores and the block's 22 barriers. Ranking the GPT-2
//   queries' 1024 x 16,384 scores (67 MB), top 20, takes the whole call from 583 to
//   467 us (counting 33 times over keys in shared memory alone took 147); 200
//   queries over 400,000 rows rank in 144 us, where one list per warp and a merge
//   took over 300 for 8 queries.
// * k_topk_merge merges the per-CTA lists [S][Q][K] of the fused tensor-core
//   scoring epilogue into the final [Q, K]. Every list is sorted, so the largest
//   K-th entry over the lists is a lower bound on the final K-th entry; only
//   candidates at or above it are sorted.
#include <algorithm>
#include <cmath>

#include "eogp_internal.h"
#include "topk_dev.cuh"

namespace {

constexpr int kMergeCap = 4096;  // keys sorted at once by the merge

// Order-preserving 64-bit key: larger key = larger score, then lower index
// (-0 and +0 are the same score).
__device__ __forceinline__ unsigned long long make_key(float s, int idx) {
  const uint32_t b = __float_as_uint(s == 0.f ? 0.f : s);
  const uint32_t o = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
  return (static_cast<unsigned long long>(o) << 32) | (0xFFFFFFFFu - static_cast<uint32_t>(idx));
}

__device__ __forceinline__ float key_score(unsigned long long key) {
  const uint32_t o = static_cast<uint32_t>(key >> 32);
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o);
}

__device__ __forceinline__ int key_index(unsigned long long key) {
  return static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(key));
}

constexpr int kSelThreads = 512;
constexpr int kSelWarps = kSelThreads / 32;
constexpr int kSelVecs = 8;  // 16-byte loads a thread
constexpr int kSelSlice = 4 * kSelVecs * kSelThreads;  // stored rows a block ranks
constexpr int kSelCand = 1024;  // candidates collected in shared memory
static_assert(EOGP_TOPK_MAX <= kSelThreads, "the bound is the K-th of one maximum a thread");

// 32-bit order key of a score: larger score, larger key; -0 and +0 equal; NaN
// maps to 0, below every score (no non-NaN float maps to 0).
__device__ __forceinline__ uint32_t sel_key(float s) {
  if (s != s) return 0u;
  const uint32_t b = __float_as_uint(s == 0.f ? 0.f : s);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// Sum over the block (block-uniform). red is double-buffered by `parity` so that
// consecutive calls need one barrier each.
__device__ __forceinline__ uint32_t block_sum(uint32_t c, uint32_t* red, int parity) {
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0) red[parity * kSelWarps + (threadIdx.x >> 5)] = c;
  __syncthreads();
  uint32_t tot = 0;
#pragma unroll
  for (int w = 0; w < kSelWarps; ++w) tot += red[parity * kSelWarps + w];
  return tot;
}

// Block b ranks slice b % S (values [slice s, slice (s + 1)) ) of row b / S into K
// places at K s + ld q of the outputs. A value's stored row is map[its place in
// the row] (a list of an earlier level), or without a map its place + row0.
// Missing places are (-inf, -1), in lists for a further level (`mid`) (NaN, -1).
__global__ void __launch_bounds__(kSelThreads, 2)
    k_topk_select(const float* __restrict__ sc, const int* __restrict__ map, size_t ld, int N, int row0, int K, int S,
                  int slice, int mid, float* __restrict__ out_s, size_t ld_os, int* __restrict__ out_i, size_t ld_oi) {
  __shared__ uint32_t red[2 * kSelWarps];
  __shared__ unsigned long long cand[kSelCand];
  __shared__ uint32_t s_n;
  const int q = blockIdx.x / S, s = blockIdx.x % S, tid = threadIdx.x;
  const int r0 = s * slice, len = min(slice, N - r0);
  const float* row = sc + static_cast<size_t>(q) * ld + r0;
  // Key e = 4 j + c of the thread is row 4 (512 j + tid) + c of the slice; 0 past its end.
  uint32_t key[4 * kSelVecs];
  uint32_t top = 0;
#pragma unroll
  for (int j = 0; j < kSelVecs; ++j) {
    const int i = 4 * (j * kSelThreads + tid);
    float v[4];
    if (i + 3 < len) {
      const float4 f = *reinterpret_cast<const float4*>(row + i);
      v[0] = f.x;
      v[1] = f.y;
      v[2] = f.z;
      v[3] = f.w;
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) v[c] = i + c < len ? row[i + c] : NAN;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      key[4 * j + c] = sel_key(v[c]);
      top = max(top, key[4 * j + c]);
    }
  }
  // (score, lower place first), 0 for no score. Lists come in the order of their
  // slices and equal scores within them by place, so the lower place is the lower
  // stored row at every level.
  auto composite = [&](int e) -> unsigned long long {
    const int i = 4 * ((e >> 2) * kSelThreads + tid) + (e & 3);
    return key[e] ? (static_cast<unsigned long long>(key[e]) << 32) | (0xFFFFFFFFu - static_cast<uint32_t>(i)) : 0ull;
  };
  if (tid == 0) s_n = 0;
  // Lower bound: the K-th largest thread maximum, its upper 20 bits (a few more
  // candidates for twelve barriers less). At least K keys are at or above it,
  // unless fewer than K threads hold a score: then every score is a candidate.
  uint32_t t0 = 0;
  for (int bit = 31; bit >= 12; --bit) {
    const uint32_t c = t0 | (1u << bit);
    if (__syncthreads_count(top >= c) >= K) t0 = c;
  }
  t0 = max(t0, 1u);
  if (top >= t0) {
#pragma unroll
    for (int e = 0; e < 4 * kSelVecs; ++e)
      if (key[e] >= t0) {
        const uint32_t p = atomicAdd(&s_n, 1u);
        if (p < kSelCand) cand[p] = composite(e);
      }
  }
  __syncthreads();
  int n = static_cast<int>(s_n);
  if (n > kSelCand) {
    // T = the Kv-th largest composite (all are distinct), Kv = min(K, scores): the
    // largest value with at least Kv composites at or above it.
    uint32_t c = 0;
#pragma unroll
    for (int e = 0; e < 4 * kSelVecs; ++e) c += key[e] ? 1u : 0u;
    int parity = 0;
    const uint32_t nv = block_sum(c, red, parity);
    const uint32_t Kv = min(static_cast<uint32_t>(K), nv);
    unsigned long long T = 0;
    for (int bit = 63; bit >= 0; --bit) {
      const unsigned long long t = T | (1ull << bit);
      c = 0;
#pragma unroll
      for (int e = 0; e < 4 * kSelVecs; ++e) c += composite(e) >= t ? 1u : 0u;
      parity ^= 1;
      if (block_sum(c, red, parity) >= Kv) T = t;
    }
    if (tid == 0) s_n = 0;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 4 * kSelVecs; ++e)
      if (composite(e) >= T) cand[atomicAdd(&s_n, 1u)] = composite(e);
    __syncthreads();
    n = static_cast<int>(s_n);
  }
  // Each candidate's rank among them is its place in the list.
  float* os = out_s + static_cast<size_t>(q) * ld_os + static_cast<size_t>(s) * K;
  int* oi = out_i + static_cast<size_t>(q) * ld_oi + static_cast<size_t>(s) * K;
  const int* mp = map ? map + static_cast<size_t>(q) * ld + r0 : nullptr;
  for (int i = tid; i < n; i += kSelThreads) {
    const unsigned long long mine = cand[i];
    int rank = 0;
    for (int j = 0; j < n; ++j) rank += cand[j] > mine ? 1 : 0;
    if (rank < K) {
      const int at = static_cast<int>(0xFFFFFFFFu - static_cast<uint32_t>(mine));
      os[rank] = row[at];  // the score itself (keys merge -0 into +0)
      oi[rank] = mp ? mp[at] : row0 + r0 + at;
    }
  }
  for (int p = n + tid; p < K; p += kSelThreads) {
    os[p] = mid ? NAN : -INFINITY;
    oi[p] = -1;
  }
}

__global__ void __launch_bounds__(256) k_topk_merge(const float* __restrict__ lst,
                                                    const int* __restrict__ lsi, int S, int Q, int K,
                                                    float* __restrict__ out_s, int ld_os,
                                                    int* __restrict__ out_i, int ld_oi) {
  __shared__ unsigned long long keys[kMergeCap];
  __shared__ unsigned long long red[8];
  __shared__ int fill;
  const int q = blockIdx.x, tid = threadIdx.x;
  // Lower bound: the largest K-th entry over the slots.
  unsigned long long lb = 0;
  for (int s = tid; s < S; s += blockDim.x) {
    const size_t o = (static_cast<size_t>(s) * Q + q) * K + (K - 1);
    const int ix = lsi[o];
    if (ix >= 0) lb = max(lb, make_key(lst[o], ix));
  }
  for (int off = 16; off > 0; off >>= 1) lb = max(lb, __shfl_xor_sync(0xffffffffu, lb, off));
  if ((tid & 31) == 0) red[tid >> 5] = lb;
  for (int i = tid; i < K; i += blockDim.x) keys[i] = 0;  // kept best K (0 = empty)
  __syncthreads();
  lb = red[0];
  for (int w = 1; w < (blockDim.x >> 5); ++w) lb = max(lb, red[w]);
  const long long C = static_cast<long long>(S) * K;
  const int W = kMergeCap - K;
  for (long long base = 0; base < C; base += W) {
    if (tid == 0) fill = 0;
    __syncthreads();
    const long long end = min(C, base + W);
    for (long long c = base + tid; c < end; c += blockDim.x) {
      const int s = static_cast<int>(c / K), p = static_cast<int>(c % K);
      const size_t o = (static_cast<size_t>(s) * Q + q) * K + p;
      const int ix = lsi[o];
      if (ix >= 0) {
        const unsigned long long key = make_key(lst[o], ix);
        if (key >= lb) keys[K + atomicAdd(&fill, 1)] = key;
      }
    }
    __syncthreads();
    const int n = K + fill;
    if (fill > 0) {
      int P = 2;
      while (P < n) P <<= 1;
      for (int i = n + tid; i < P; i += blockDim.x) keys[i] = 0;
      __syncthreads();
      // bitonic sort, descending
      for (int k2 = 2; k2 <= P; k2 <<= 1) {
        for (int j = k2 >> 1; j > 0; j >>= 1) {
          for (int i = tid; i < P; i += blockDim.x) {
            const int ixj = i ^ j;
            if (ixj > i) {
              const unsigned long long a = keys[i], b = keys[ixj];
              const bool desc = (i & k2) == 0;
              if (desc ? (a < b) : (a > b)) {
                keys[i] = b;
                keys[ixj] = a;
              }
            }
          }
          __syncthreads();
        }
      }
    }
    __syncthreads();
  }
  for (int p = tid; p < K; p += blockDim.x) {
    const unsigned long long key = keys[p];
    out_s[static_cast<size_t>(q) * ld_os + p] = key ? key_score(key) : -INFINITY;
    out_i[static_cast<size_t>(q) * ld_oi + p] = key ? key_index(key) : -1;
  }
}

}  // namespace

// One block ranks up to 16,384 stored rows of a query by itself; more rows take
// the fewest slices of that size, or for few queries enough of at least 4096 rows
// to give every SM two blocks.
int topk_slice(int N, int Q, int num_sms) {
  if (N <= kSelSlice) return kSelSlice;
  const int least = (N + kSelSlice - 1) / kSelSlice;
  const int S = std::max(least, std::min((N + 4095) / 4096, (2 * num_sms + Q - 1) / std::max(Q, 1)));
  return ((N + S - 1) / S + 3) & ~3;
}

cudaError_t launch_topk_select(const float* scores, const int* map, size_t ld, int Q, int N, int row0, int K, int slice,
                               bool mid, float* out_s, size_t ld_os, int* out_i, size_t ld_oi, cudaStream_t st) {
  if (Q <= 0) return cudaSuccess;
  const int S = std::max(1, (N + slice - 1) / slice);
  const long long blocks = static_cast<long long>(S) * Q;
  if (K > EOGP_TOPK_MAX || slice > kSelSlice || (slice & 3) || (ld & 3) || (reinterpret_cast<uintptr_t>(scores) & 15) ||
      blocks > 0x7FFFFFFF)
    return cudaErrorInvalidValue;
  k_topk_select<<<static_cast<unsigned>(blocks), kSelThreads, 0, st>>>(scores, map, ld, N, row0, K, S, slice, mid ? 1 : 0,
                                                                       out_s, ld_os, out_i, ld_oi);
  return cudaGetLastError();
}

cudaError_t launch_topk_merge(const float* lst, const int* lsi, int S, int Q, int K, float* out_s,
                              int ld_os, int* out_i, int ld_oi, cudaStream_t st) {
  if (Q <= 0) return cudaSuccess;
  k_topk_merge<<<Q, 256, 0, st>>>(lst, lsi, S, Q, K, out_s, ld_os, out_i, ld_oi);
  return cudaGetLastError();
}
