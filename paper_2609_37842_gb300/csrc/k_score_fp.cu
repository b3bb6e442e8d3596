// Unquantised scores <y_q, x_i> (the FP mode of eogp_score) on the tensor cores.
//
// Precision. Both sides stay 32-bit values: each fp32 number is the exact sum of
// three bf16 numbers (its 24-bit significand cut into 8 + 8 + 8 bits by
// truncation, x = x1 + x2 + x3), and eight of the nine products are formed, every
// one of them exact in fp32:
//   d0 += x1 y1,   d1 += x1 y2 + x2 y1,   d2 += x1 y3 + x2 y2 + x3 y1,   d3 += x2 y3 + x3 y2
// (with 64 queries a tile the last two go to d2). |x2| < 2^-7 |x| and |x3| < 2^-15 |x|:
// what is left out, x3 y3, is below 2^-30 of the product. Without x2 y3 and x3 y2, up
// to 2^-21 together and of the product's sign, a score of one coordinate was off by as
// much as 4.2e-7. The magnitudes have accumulators of their own, and every 256
// coordinates they are added in fp32 registers with round to nearest, so the tensor
// core's own accumulation never runs over more than 16 steps. Largest error against
// 64-bit sums, of the sum of magnitudes, in brackets that of k_simt_gemm (one fp32
// chain per score): one coordinate among 512 5.9e-8 (5.9e-8), two 1.5e-7 (1.1e-7), eight
// 1.5e-7 (2.0e-7), all 512 1.0e-7 (2.5e-7), 49,152 1.2e-8 (3.0e-7). Sums near the end of
// fp32's range are within a few units of 2^-149 a product.
// Infinities, NaN and tiny values with bits below 2^-133, where bf16 ends, have no such
// split: it leaves bits in the lower half of x3. A row or query that holds one is
// noted, and k_simt_gemm computes its scores, and no others, again afterwards.
//
// Bound: HBM (the stored coordinates, once per 64 queries), and from 48 queries on the
// power limit. One CTA takes 128 stored rows (MMA M, operand A in TMEM) against QB <=
// 64 queries; the query parts lie stacked as 3 QB rows of one operand B, so a K = 16
// step is three MMAs: x1 and x2 by all 3 QB rows, x3 by the first 2 QB, each into the
// columns one part further on. (A tile of 64 queries has no TMEM for d3 without a longer
// drain: five MMAs, 660 us against 710 for 64 queries.) 16,384 x 49,152 stored
// coordinates (3.2 GB), passes behind one another: 16 queries 539 us, 48 574 to 599 as
// the clock falls (alone 555 us at 1.79 GHz; the six larger products 565, alone 542 at
// 1.84), 0.83 of the measured copy rate, against 5,702 us on the CUDA cores.
//
// Pipeline per CTA (persistent over (row tile, K range, query tile) items):
//  * TMA producer: fp32 boxes of 128 rows x 32 coordinates (128-byte swizzle) in a
//    ring of eight or ten, and query tiles of 3 QB rows x 64 coordinates in a ring of three;
//  * eight converter warps in two groups that take the boxes in turn (one warp per
//    TMEM lane quarter): shared memory -> three bf16 parts -> TMEM, 48 columns a box;
//  * one issuing warp (converged, MMAs under elect.sync): 12 MMAs (20 with 64
//    queries) per pair of boxes (one query tile) and round of wait, fence and commit.
//    With 6 per round, one box, the rounds set the pace, 646 us for the case above
//    whatever the number of queries;
//  * four drain warps: every 256 coordinates the accumulators of a row into
//    registers; at the item's end the sums to the scores or to the K range's slab.
#include <algorithm>

#include "eogp_dev.cuh"
#include "eogp_internal.h"

using namespace eogp;

namespace {

constexpr int kConvW0 = 4, kConvW = 8;          // drain warps are 0-3
constexpr int kMmaW = kConvW0 + kConvW;         // 12: owns TMEM, issues
constexpr int kTmaW = kMmaW + 1;                // 13
constexpr int kThreads = (kTmaW + 1) * 32;
constexpr int kYRing = 3;
constexpr uint32_t kXBox = 128u * 128u;         // 128 rows x 32 fp32
constexpr int kDrainBoxes = 8;                  // boxes (of 32 coordinates) per accumulation run
constexpr int kSplitBlocks = 16;                // blocks per query of the query split, at most
constexpr int kMinD = 512;                      // fewer coordinates stay on k_simt_gemm

// TMEM: two accumulator sets of 4 QB columns, one with 48 queries, one of 3 QB with 64
// (its drain then holds up the next run's MMAs), and A slots of 96 columns, each two
// boxes.
template <int QB>
constexpr int fp_parts() {
  return QB == 64 ? 3 : 4;
}
template <int QB>
constexpr int fp_accs() {
  return QB >= 48 ? 1 : 2;
}
template <int QB>
constexpr int fp_slots() {
  return QB == 48 ? 3 : 2;
}
template <int QB>
constexpr int fp_xring() {
  return QB == 64 ? 8 : 10;
}
template <int QB>
constexpr uint32_t fp_ybox() {
  return 3u * QB * 128u;
}
template <int QB>
constexpr size_t fp_smem() {
  return 1024 + fp_xring<QB>() * kXBox + kYRing * static_cast<size_t>(fp_ybox<QB>()) +
         (2 * fp_xring<QB>() + 2 * kYRing + 2 * fp_slots<QB>() + 4) * 8 + 16;
}

struct FpArgs {
  int N, Q, nbox, bps, nrt, nqt, S, n_items;  // nbox: 32-coordinate boxes of a row, bps of them per K range
  float* out;    // scores, or with S > 1 the slabs [S][Q][ldo]
  size_t slab;
  int ldo;
  int* rbad;     // [N]: the row holds a value without a split
  unsigned* status;
};

// Three-way split: upper halves of x, x - x1 and x - x1 - x2. Exact if and only if the
// lower half of h3 is zero (an infinity or a NaN makes h3 the canonical NaN 0x7FFFFFFF).
__device__ __forceinline__ void split3(float x, uint32_t& h1, uint32_t& h2, uint32_t& h3) {
  h1 = __float_as_uint(x) & 0xFFFF0000u;
  const float r = __fsub_rn(x, __uint_as_float(h1));
  h2 = __float_as_uint(r) & 0xFFFF0000u;
  h3 = __float_as_uint(__fsub_rn(r, __uint_as_float(h2)));
}

__device__ __forceinline__ uint32_t pack_hi(uint32_t lo, uint32_t hi) { return __byte_perm(lo, hi, 0x7632); }

template <int QB>
__global__ void __launch_bounds__(kThreads, 1)
    k_score_fp(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmY, const FpArgs g) {
  constexpr int ND = fp_accs<QB>(), kXRing = fp_xring<QB>(), kSlots = fp_slots<QB>();
  constexpr uint32_t kAcc = fp_parts<QB>() * QB;             // columns of an accumulator set
  constexpr uint32_t kA0 = ND * kAcc;            // first A column
  static_assert(kXRing % 2 == 0, "each converter group owns every second box");
  static_assert(kA0 + 96u * kSlots <= 512u, "TMEM budget");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint8_t* ysm = smem + kXRing * kXBox;
  uint64_t* xfull = reinterpret_cast<uint64_t*>(ysm + kYRing * static_cast<size_t>(fp_ybox<QB>()));
  uint64_t* xempty = xfull + kXRing;
  uint64_t* yfull = xempty + kXRing;
  uint64_t* yempty = yfull + kYRing;
  uint64_t* afull = yempty + kYRing;             // A slot written
  uint64_t* aempty = afull + kSlots;             // A slot's MMAs done
  uint64_t* dfull = aempty + kSlots;
  uint64_t* dempty = dfull + 2;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(dempty + 2);
  const int warp = warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmX);
    tma_prefetch_desc(&tmY);
    for (int i = 0; i < kXRing; ++i) {
      mbar_init(&xfull[i], 1);
      mbar_init(&xempty[i], kConvW / 2);  // one group's warps
    }
    for (int i = 0; i < kYRing; ++i) {
      mbar_init(&yfull[i], 1);
      mbar_init(&yempty[i], 1);
    }
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(&afull[i], kConvW);
      mbar_init(&aempty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&dfull[i], 1);
      mbar_init(&dempty[i], 4);
    }
    fence_barrier_init();
  }
  if (warp == kMmaW) tmem_alloc(tslot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  // Item: query tiles innermost, so the CTAs of one (row tile, K range) share its
  // rows through L2. Boxes [b0, b1) of a row; b0 is even (a query tile is two boxes).
  auto item_boxes = [&](int item, int& b0, int& b1) {
    const int s = (item / g.nqt) % g.S;
    b0 = s * g.bps;
    b1 = min(g.nbox, b0 + g.bps);
  };

  if (warp < kConvW0) {
    // ---------------------------------------------------------- drain
    const uint32_t lane_base = static_cast<uint32_t>(warp * 32) << 16;
    uint32_t run = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
      int b0, b1;
      item_boxes(item, b0, b1);
      const int qt = item % g.nqt, s = (item / g.nqt) % g.S, rt = item / (g.nqt * g.S);
      float sum[QB];
#pragma unroll
      for (int c = 0; c < QB; ++c) sum[c] = 0.f;
      for (int b = b0; b < b1; b += kDrainBoxes, ++run) {
        const int buf = static_cast<int>(run % ND);
        if (!mbar_wait_warp(&dfull[buf], (run / ND) & 1u, g.status)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + lane_base + buf * kAcc;
#pragma unroll
        for (int c = 0; c < QB; c += 16) {
          uint32_t v0[16], v1[16], v2[16], v3[16];
          tmem_ld16_issue(d + c, v0);
          tmem_ld16_issue(d + QB + c, v1);
          tmem_ld16_issue(d + 2 * QB + c, v2);
          if constexpr (fp_parts<QB>() == 4) tmem_ld16_issue(d + 3 * QB + c, v3);
          tmem_wait_ld(v0);
          tmem_wait_ld(v1);
          tmem_wait_ld(v2);
          if constexpr (fp_parts<QB>() == 4) tmem_wait_ld(v3);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            float low = __uint_as_float(v2[j]);
            if constexpr (fp_parts<QB>() == 4) low += __uint_as_float(v3[j]);
            sum[c + j] += __uint_as_float(v0[j]) + (__uint_as_float(v1[j]) + low);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&dempty[buf]);
      }
      if (!ok) break;
      const int row = rt * 128 + warp * 32 + lane;
      if (row < g.N) {
        float* o = g.out + static_cast<size_t>(s) * g.slab + row;
#pragma unroll
        for (int c = 0; c < QB; ++c) {
          const int q = qt * QB + c;
          if (q < g.Q) o[static_cast<size_t>(q) * g.ldo] = sum[c];
        }
      }
    }
  } else if (warp < kMmaW) {
    // ---------------------------------------------------------- converters
    // Two groups of four warps take the boxes in turn, a whole row of 32
    // coordinates a thread, so one group's waits fall into the other's arithmetic.
    const int q4 = warp & 3, grp = (warp - kConvW0) >> 2;
    const int r = q4 * 32 + lane;  // row of the tile = TMEM lane
    const uint32_t a_lane = tmem + (static_cast<uint32_t>(q4 * 32) << 16) + kA0;
    uint32_t it = 0;  // boxes of earlier items
    bool ok = true;
    for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
      int b0, b1;
      item_boxes(item, b0, b1);
      uint32_t bad = 0;  // lower half: bits that a value's three parts leave out
      for (int b = b0; b < b1; ++b, ++it) {
        if ((it & 1u) != static_cast<uint32_t>(grp)) continue;
        const uint32_t pr = it >> 1;  // pair of boxes = A slot use
        const int xs = static_cast<int>(it % kXRing), as = static_cast<int>(pr % kSlots);
        if (!mbar_wait_warp(&xfull[xs], (it / kXRing) & 1u, g.status)) {
          ok = false;
          break;
        }
        const uint8_t* xr = smem + xs * kXBox + r * 128;
        float4 f[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) f[c] = *reinterpret_cast<const float4*>(xr + ((c ^ (r & 7)) << 4));
        uint32_t p1[16], p2[16], p3[16];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float v[4] = {f[c].x, f[c].y, f[c].z, f[c].w};
          uint32_t h1[4], h2[4], h3[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            split3(v[e], h1[e], h2[e], h3[e]);
            bad |= h3[e];
          }
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            p1[2 * c + e] = pack_hi(h1[2 * e], h1[2 * e + 1]);
            p2[2 * c + e] = pack_hi(h2[2 * e], h2[2 * e + 1]);
            p3[2 * c + e] = pack_hi(h3[2 * e], h3[2 * e + 1]);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&xempty[xs]);  // the box is in registers
        if (!mbar_wait_warp(&aempty[as], ((pr / kSlots) & 1u) ^ 1u, g.status)) {
          ok = false;
          break;
        }
        tc_fence_after();  // the MMAs that read the slot before are done
        const uint32_t a = a_lane + 96u * as + 48u * grp;
        tmem_st16_issue(a, p1);
        tmem_st16_issue(a + 16u, p2);
        tmem_st16_issue(a + 32u, p3);
        tmem_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&afull[as]);
      }
      // (rows past N are zeros)
      if (bad & 0xFFFFu) g.rbad[item / (g.nqt * g.S) * 128 + r] = 1;
    }
  } else if (warp == kMmaW) {
    // ---------------------------------------------------------- issuer
    {
      const uint32_t id3 = idesc_bf16_f32(128, 3 * QB, 0, 0), id2 = idesc_bf16_f32(128, 2 * QB, 0, 0),
                     id1 = idesc_bf16_f32(128, QB, 0, 0);
      constexpr uint64_t kPart = (QB * 128) >> 4;  // a query part on, whole swizzle atoms
      const uint64_t ydesc = sdesc_sw128(smem_u32(ysm), 16, 1024);
      uint32_t pr = 0, run = 0;  // pairs of boxes (and query tiles), accumulation runs of earlier items
      bool ok = true;
      for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
        int b0, b1;
        item_boxes(item, b0, b1);
        for (int b = b0; b < b1 && ok; b += kDrainBoxes, ++run) {
          const int buf = static_cast<int>(run % ND);
          if (!mbar_wait_warp(&dempty[buf], ((run / ND) & 1u) ^ 1u, g.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem + buf * kAcc;
          const int e = min(b1, b + kDrainBoxes);
          for (int bb = b; bb < e; bb += 2, ++pr) {
            const int as = static_cast<int>(pr % kSlots), ys = static_cast<int>(pr % kYRing);
            if (!mbar_wait_warp(&yfull[ys], (pr / kYRing) & 1u, g.status) ||
                !mbar_wait_warp(&afull[as], (pr / kSlots) & 1u, g.status)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint64_t y0 = ydesc + ((ys * fp_ybox<QB>()) >> 4);
            const uint32_t a0 = tmem + kA0 + 96u * as;
            if (elect_one()) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {
                const uint64_t y = y0 + 2 * kk;  // K = 16: 32 bytes on
                const uint32_t a = a0 + 48u * (kk >> 1) + 8u * (kk & 1);
                const bool start = kk == 0 && bb == b;  // of a run
                if constexpr (fp_parts<QB>() == 3) {
                  tc_mma_f16_ta(d, a, y, id3, start ? 0u : 1u);
                  tc_mma_f16_ta(d + QB, a + 16u, y, id2, 1u);
                  tc_mma_f16_ta(d + 2 * QB, a + 32u, y, id1, 1u);
                  tc_mma_f16_ta(d + 2 * QB, a + 16u, y + 2 * kPart, id1, 1u);
                  tc_mma_f16_ta(d + 2 * QB, a + 32u, y + kPart, id1, 1u);
                } else {
                  tc_mma_f16_ta(d, a, y, id3, start ? 0u : 1u);
                  if (start) {  // d1 and d2 hold x1's products already, d3 starts here
                    tc_mma_f16_ta(d + QB, a + 16u, y, id2, 1u);
                    tc_mma_f16_ta(d + 3 * QB, a + 16u, y + 2 * kPart, id1, 0u);
                  } else {
                    tc_mma_f16_ta(d + QB, a + 16u, y, id3, 1u);
                  }
                  tc_mma_f16_ta(d + 2 * QB, a + 32u, y, id2, 1u);
                }
              }
              tc_commit(&aempty[as]);
              tc_commit(&yempty[ys]);
            }
          }
          if (ok && elect_one()) tc_commit(&dfull[buf]);
        }
      }
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------- TMA producer
    if (lane == 0) {
      uint32_t it = 0, yt = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
        int b0, b1;
        item_boxes(item, b0, b1);
        const int qt = item % g.nqt, rt = item / (g.nqt * g.S);
        for (int b = b0; b < b1; ++b, ++it) {
          const int xs = static_cast<int>(it % kXRing);
          if (((b - b0) & 1) == 0) {
            const int ys = static_cast<int>(yt % kYRing);
            if (!mbar_wait(&yempty[ys], ((yt / kYRing) & 1u) ^ 1u, g.status)) {
              ok = false;
              break;
            }
            mbar_arrive_expect_tx(&yfull[ys], fp_ybox<QB>());
            tma_load_2d(ysm + ys * static_cast<size_t>(fp_ybox<QB>()), &tmY, b * 32, qt * 3 * QB, &yfull[ys]);
            ++yt;
          }
          if (!mbar_wait(&xempty[xs], ((it / kXRing) & 1u) ^ 1u, g.status)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&xfull[xs], kXBox);
          tma_load_2d(smem + xs * kXBox, &tmX, b * 32, rt * 128, &xfull[xs]);
        }
      }
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaW) tmem_dealloc(tmem, 512);
}

// Query q's three bf16 parts, in rows part * QB + q % QB of query tile q / QB
// (rows of Dp values, zero past D; the rows of a tile past Q are zero), and whether
// the part of it that block (q, y) splits holds a value without a split. Clears the
// rows' notes. Queries are on grid.x: whole tiles of 65,535 are 65,536 of them.
__global__ void __launch_bounds__(256) k_split3_queries(const float* __restrict__ y, int ldq, int Q, int D, int Dp,
                                                        int QB, uint16_t* __restrict__ parts, int* __restrict__ qbad,
                                                        int* __restrict__ rbad, int N) {
  const int q = blockIdx.x, c0 = 2 * (blockIdx.y * blockDim.x + threadIdx.x), nthr = gridDim.y * blockDim.x;
  uint16_t* o = parts + (static_cast<size_t>(q / QB) * 3 * QB + q % QB) * Dp;
  const size_t step = static_cast<size_t>(QB) * Dp;
  int bad = 0;
  for (int c = c0; c < Dp; c += 2 * nthr) {  // Dp is even
    uint32_t h1[2], h2[2], h3[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float v = (q < Q && c + e < D) ? y[static_cast<size_t>(q) * ldq + c + e] : 0.f;
      split3(v, h1[e], h2[e], h3[e]);
      bad |= static_cast<int>(h3[e] & 0xFFFFu);
    }
    *reinterpret_cast<uint32_t*>(o + c) = pack_hi(h1[0], h1[1]);
    *reinterpret_cast<uint32_t*>(o + step + c) = pack_hi(h2[0], h2[1]);
    *reinterpret_cast<uint32_t*>(o + 2 * step + c) = pack_hi(h3[0], h3[1]);
  }
  bad = __syncthreads_or(bad);
  if (threadIdx.x == 0) qbad[static_cast<size_t>(blockIdx.y) * gridDim.x + q] = bad;
  for (int i = (q * gridDim.y + blockIdx.y) * blockDim.x + threadIdx.x; i < N; i += gridDim.x * nthr) rbad[i] = 0;
}

// scores[q][i] = the slabs' values in order; four scores a thread (ldp is a
// multiple of four), query blockIdx.y and on.
__global__ void __launch_bounds__(256) k_sum_slabs(const float* __restrict__ part, int S, size_t slab, int ldp, int N,
                                                   int Q, float* __restrict__ out, int ldo, int vec) {
  const int i = 4 * (blockIdx.x * 256 + threadIdx.x);
  if (i >= N) return;
  for (int q = blockIdx.y; q < Q; q += gridDim.y) {
    const float* p = part + static_cast<size_t>(q) * ldp + i;
    float4 t = *reinterpret_cast<const float4*>(p);
    for (int s = 1; s < S; ++s) {
      const float4 v = *reinterpret_cast<const float4*>(p + static_cast<size_t>(s) * slab);
      t.x += v.x;
      t.y += v.y;
      t.z += v.z;
      t.w += v.w;
    }
    float* o = out + static_cast<size_t>(q) * ldo + i;
    if (vec && i + 3 < N) {
      *reinterpret_cast<float4*>(o) = t;
    } else {
      o[0] = t.x;
      if (i + 1 < N) o[1] = t.y;
      if (i + 2 < N) o[2] = t.z;
      if (i + 3 < N) o[3] = t.w;
    }
  }
}

struct FpPlan {
  int QB, nqt, nrt, Dp, nbox, S, bps, ldp;
  size_t parts, qbad, rbad, part, total;
};

int fp_tile_queries(int Q) {
  const int n = (Q + 63) / 64;
  return ((Q + n - 1) / n + 15) / 16 * 16;
}

// K ranges: the number that leaves the request's last wave of items fullest, counting 256
// coordinates of a range's time for its start, drain and sum.
FpPlan fp_plan(int N, int D, int Q, ScoreRequest all, int num_sms) {
  FpPlan p;
  p.QB = fp_tile_queries(Q);
  p.nqt = (Q + p.QB - 1) / p.QB;
  p.nrt = (N + 127) / 128;
  p.Dp = (D + 63) / 64 * 64;
  p.nbox = p.Dp / 32;  // even: boxes past D are zero
  const int qb = fp_tile_queries(all.Q);
  const long long tiles = static_cast<long long>((all.Q + qb - 1) / qb) * ((all.N + 127) / 128);
  const int nyt = p.Dp / 64;
  long long best = -1;
  p.S = 1;
  p.bps = 2 * nyt;
  for (int want = 1; want <= 32 && want * 4 <= nyt; ++want) {
    const int per = (nyt + want - 1) / want, S = (nyt + per - 1) / per;
    const long long cost = (tiles * S + num_sms - 1) / num_sms * (per + 4);
    if (best < 0 || cost < best) {
      best = cost;
      p.S = S;
      p.bps = 2 * per;
    }
  }
  p.ldp = (N + 3) & ~3;
  auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
  p.parts = 0;
  p.qbad = al(static_cast<size_t>(p.nqt) * 3 * p.QB * p.Dp * 2);
  p.rbad = p.qbad + al(static_cast<size_t>(kSplitBlocks) * p.nqt * p.QB * 4);
  p.part = p.rbad + al(static_cast<size_t>(N) * 4);
  p.total = p.part + (p.S > 1 ? al(static_cast<size_t>(p.S) * Q * p.ldp * 4) : 0);
  return p;
}

template <int QB>
cudaError_t launch_qb(const CUtensorMap& tx, const CUtensorMap& ty, const FpArgs& g, int num_sms, cudaStream_t st) {
  const cudaError_t e = cudaFuncSetAttribute(k_score_fp<QB>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(fp_smem<QB>()));
  if (e != cudaSuccess) return e;
  k_score_fp<QB><<<std::min(g.n_items, num_sms), kThreads, fp_smem<QB>(), st>>>(tx, ty, g);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_sum_slabs(const float* part, int S, size_t slab, int ldp, int N, int Q, float* out, int ldo,
                             cudaStream_t st) {
  const int vec = (ldo & 3) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0;
  k_sum_slabs<<<dim3((N + 1023) / 1024, std::min(Q, 65535)), 256, 0, st>>>(part, S, slab, ldp, N, Q, out, ldo, vec);
  return cudaGetLastError();
}

bool score_fp_supported(int N, long long D, int Q) {
  return D >= kMinD && N >= 1 && Q >= 1 && Q <= 65535 && D <= (1 << 28) &&
         static_cast<long long>((N + 127) / 128) * ((Q + 63) / 64) * 32 < (1ll << 30);
}

size_t score_fp_ws_bytes(int N, long long D, int Q, ScoreRequest all, int num_sms) {
  return fp_plan(N, static_cast<int>(D), Q, all, num_sms).total;
}

cudaError_t launch_score_fp(const float* train, int ldt, int N, int D, const float* query, int ldq, int Q,
                            ScoreRequest all, float* out, int ldo, void* ws, int num_sms, unsigned* status,
                            cudaStream_t st) {
  const FpPlan p = fp_plan(N, D, Q, all, num_sms);
  char* w = static_cast<char*>(ws);
  uint16_t* parts = reinterpret_cast<uint16_t*>(w + p.parts);
  int* qbad = reinterpret_cast<int*>(w + p.qbad);
  int* rbad = reinterpret_cast<int*>(w + p.rbad);
  float* part = reinterpret_cast<float*>(w + p.part);
  const int sb = std::min(kSplitBlocks, (p.Dp / 2 + 255) / 256);
  k_split3_queries<<<dim3(p.nqt * p.QB, sb), 256, 0, st>>>(query, ldq, Q, D, p.Dp, p.QB, parts, qbad, rbad, N);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  CUtensorMap tx, ty;
  const uint64_t xd[2] = {static_cast<uint64_t>(D), static_cast<uint64_t>(N)};
  const uint64_t xs[1] = {static_cast<uint64_t>(ldt) * 4};
  const uint32_t xb[2] = {32, 128};
  const uint64_t yd[2] = {static_cast<uint64_t>(p.Dp), static_cast<uint64_t>(p.nqt) * 3 * p.QB};
  const uint64_t ys[1] = {static_cast<uint64_t>(p.Dp) * 2};
  const uint32_t yb[2] = {64, static_cast<uint32_t>(3 * p.QB)};
  if (make_tmap(&tx, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, train, xd, xs, xb, CU_TENSOR_MAP_SWIZZLE_128B) ||
      make_tmap(&ty, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, parts, yd, ys, yb, CU_TENSOR_MAP_SWIZZLE_128B))
    return cudaErrorInvalidValue;
  FpArgs g;
  g.N = N;
  g.Q = Q;
  g.nbox = p.nbox;
  g.bps = p.bps;
  g.nrt = p.nrt;
  g.nqt = p.nqt;
  g.S = p.S;
  g.n_items = p.nrt * p.nqt * p.S;
  g.out = p.S > 1 ? part : out;
  g.ldo = p.S > 1 ? p.ldp : ldo;
  g.slab = static_cast<size_t>(Q) * p.ldp;
  g.rbad = rbad;
  g.status = status;
  e = p.QB == 64   ? launch_qb<64>(tx, ty, g, num_sms, st)
      : p.QB == 48 ? launch_qb<48>(tx, ty, g, num_sms, st)
      : p.QB == 32 ? launch_qb<32>(tx, ty, g, num_sms, st)
                   : launch_qb<16>(tx, ty, g, num_sms, st);
  if (e != cudaSuccess) return e;
  if (p.S > 1) {
    e = launch_sum_slabs(part, p.S, g.slab, p.ldp, N, Q, out, ldo, st);
    if (e != cudaSuccess) return e;
  }
  // scores of rows and queries with a value without a split, one fp32 chain each
  return launch_simt_gemm_noted(Q, N, D, query, ldq, train, ldt, out, ldo, qbad, sb, p.nqt * p.QB, rbad, st);
}
