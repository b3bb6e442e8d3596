// Unquantised queries against stored one-bit codes (the paper's asymmetric score
// sum_u s_iu <y_u, b_iu>, Sec. 3.3 Eq. onebit_influence; App. B.3) on the tensor
// cores: k_score_paper.
//
// y is split into bf16 hi + lo (y to about 2^-17 relative), the stored bits are
// bf16 +-1, every product is exact. hi and lo of a query tile lie stacked as 2 QB
// <= 256 rows of one operand B, so a K = 16 step is one MMA of M = 128 stored rows
// (operand A, in TMEM) and N = 2 QB; the drain adds the two sums of a query.
// Accumulation runs cover at most 1024 coordinates of one module; after each,
// acc = fl(acc + s_iu d) (one fused multiply-add) in fp32 registers.
//
// Bound: the bf16 tensor rate (two products a coordinate). 250 queries against
// 16,384 rows of 48 x 1024 bits: 491 us (1.68 PFLOP/s issued, 0.86 of the measured
// burst rate; the last wave of items and the drains take 0.11 of it), against 864
// us for the one-CTA kernel of k_score_tc.cu, which expands into shared memory and
// issues hi and lo separately, 8 MMAs of N = 128 a round.
//
// Pipeline per CTA (persistent over (row tile, K range, query tile) items):
//  * TMA producer: code boxes of 128 rows x 1024 bits (128-byte swizzle), ring of
//    three; per 64 coordinates the hi and lo query tiles, ring of five;
//  * four expander warps (one per TMEM lane quarter): a round of 128 coordinates of
//    a row from its four code words into 64 TMEM columns, two instructions a
//    column: column j of a word holds bits j and j + 16 (the queries are laid out in
//    the same order);
//  * one issuing warp (converged, MMAs under elect.sync: 570 -> 491 us against a
//    loop under lane == 0): 8 MMAs a round of wait, fence and commit;
//  * eight drain warps (two per lane quarter, half the queries each). One
//    accumulator: the drain of a run (~300 of 8,200 cycles) holds up the next
//    one's MMAs, and leaves TMEM for four rounds of A.
#include <algorithm>

#include "eogp_dev.cuh"
#include "eogp_internal.h"

using namespace eogp;

namespace {

constexpr int kMaxMods = 1024;
constexpr int kDrW = 8;                        // drain warps 0-7
constexpr int kExW0 = kDrW, kExW = 4;          // expander warps 8-11
constexpr int kMmaW = kExW0 + kExW;            // 12: owns TMEM, issues
constexpr int kTmaW = kMmaW + 1;               // 13
constexpr int kThreads = (kTmaW + 1) * 32;
constexpr int kQB = 128;                       // queries per tile at most
constexpr int kYRing = 5, kCRing = 3, kSlots = 4;
constexpr uint32_t kYBox = 2u * kQB * 128u;    // hi and lo rows of 64 coordinates
constexpr uint32_t kCBox = 128u * 128u;        // 128 rows x 32 words
constexpr int kRunPairs = 16;                  // 64-coordinate pairs per accumulation run, at most
constexpr uint32_t kA0 = 256u;                 // A slots of 64 TMEM columns after the accumulator
constexpr size_t kSmem =
    1024 + kYRing * static_cast<size_t>(kYBox) + kCRing * kCBox + (2 * kYRing + 2 * kCRing + 2 * kSlots + 2) * 8 + 16;
static_assert(kSmem <= 232448, "shared memory");

struct PaperArgs {
  int N, Q, QB, U, npair, pps, nrt, nqt, S, n_items;  // npair: 64-coordinate pairs of a row, pps of them per K range
  int ldts;
  const float* ts;
  float* out;  // scores, or with S > 1 the slabs [S][Q][ldo]
  size_t slab;
  int ldo;
  unsigned* status;
  int pend[kMaxMods];  // first pair after module u
};

// The accumulation runs of pairs [p0, p1): cut at module ends and every kRunPairs.
struct Runs {
  int p, end, u;  // next pair, item's end, module of p
  __device__ __forceinline__ Runs(const PaperArgs& g, int p0, int p1) : p(p0), end(p1), u(0) {
    while (u + 1 < g.U && g.pend[u] <= p0) ++u;
  }
  // The run [b, e) of module um; false when there is none left.
  __device__ __forceinline__ bool next(const PaperArgs& g, int& b, int& e, int& um) {
    if (p >= end) return false;
    if (p >= g.pend[u]) ++u;
    b = p;
    um = u;
    e = min(min(end, g.pend[u]), p + kRunPairs);
    p = e;
    return true;
  }
};

__global__ void __launch_bounds__(kThreads, 1)
    k_score_paper(const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmHi,
                  const __grid_constant__ CUtensorMap tmLo, const __grid_constant__ PaperArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint8_t* csm = smem + kYRing * static_cast<size_t>(kYBox);
  uint64_t* yfull = reinterpret_cast<uint64_t*>(csm + kCRing * kCBox);
  uint64_t* yempty = yfull + kYRing;
  uint64_t* cfull = yempty + kYRing;
  uint64_t* cempty = cfull + kCRing;
  uint64_t* afull = cempty + kCRing;
  uint64_t* aempty = afull + kSlots;
  uint64_t* dfull = aempty + kSlots;
  uint64_t* dempty = dfull + 1;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(dempty + 1);
  const int warp = warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmC);
    tma_prefetch_desc(&tmHi);
    tma_prefetch_desc(&tmLo);
    for (int i = 0; i < kYRing; ++i) {
      mbar_init(&yfull[i], 1);
      mbar_init(&yempty[i], 1);
    }
    for (int i = 0; i < kCRing; ++i) {
      mbar_init(&cfull[i], 1);
      mbar_init(&cempty[i], kExW);
    }
    for (int i = 0; i < kSlots; ++i) {
      mbar_init(&afull[i], kExW);
      mbar_init(&aempty[i], 1);
    }
    mbar_init(dfull, 1);
    mbar_init(dempty, kDrW);
    fence_barrier_init();
  }
  if (warp == kMmaW) tmem_alloc(tslot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  // Item: query tiles innermost. Pairs [p0, p1) of a row; p0 starts a code box.
  auto item_pairs = [&](int item, int& p0, int& p1) {
    p0 = ((item / g.nqt) % g.S) * g.pps;
    p1 = min(g.npair, p0 + g.pps);
  };

  if (warp < kDrW) {
    // ---------------------------------------------------------- drain
    const int q4 = warp & 3, c0 = (warp >> 2) * (kQB / 2);  // this warp's first query column
    const uint32_t d = tmem + (static_cast<uint32_t>(q4 * 32) << 16);
    uint32_t run = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
      int p0, p1, b, e, u;
      item_pairs(item, p0, p1);
      const int qt = item % g.nqt, s = (item / g.nqt) % g.S, rt = item / (g.nqt * g.S);
      const int row = rt * 128 + q4 * 32 + lane;
      float acc[kQB / 2];
#pragma unroll
      for (int c = 0; c < kQB / 2; ++c) acc[c] = 0.f;
      for (Runs r(g, p0, p1); r.next(g, b, e, u); ++run) {
        const float si = row < g.N ? g.ts[static_cast<size_t>(row) * g.ldts + u] : 0.f;
        if (!mbar_wait_warp(dfull, run & 1u, g.status)) {
          ok = false;
          break;
        }
        tc_fence_after();
#pragma unroll
        for (int c = 0; c < kQB / 2; c += 16)
          if (c0 + c < g.QB) {
            uint32_t h[16], l[16];
            tmem_ld16_issue(d + c0 + c, h);
            tmem_ld16_issue(d + g.QB + c0 + c, l);
            tmem_wait_ld(h);
            tmem_wait_ld(l);
#pragma unroll
            for (int j = 0; j < 16; ++j)
              acc[c + j] = fmaf(si, __uint_as_float(h[j]) + __uint_as_float(l[j]), acc[c + j]);
          }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(dempty);
      }
      if (!ok) break;
      if (row < g.N) {
        float* o = g.out + static_cast<size_t>(s) * g.slab + row;
#pragma unroll
        for (int c = 0; c < kQB / 2; ++c) {
          const int q = qt * g.QB + c0 + c;
          if (c0 + c < g.QB && q < g.Q) o[static_cast<size_t>(q) * g.ldo] = acc[c];
        }
      }
    }
  } else if (warp < kMmaW) {
    // ---------------------------------------------------------- expanders
    const int q4 = warp & 3;
    const int r = q4 * 32 + lane;  // row of the tile = TMEM lane
    const uint32_t a_lane = tmem + (static_cast<uint32_t>(q4 * 32) << 16) + kA0;
    uint32_t rd = 0, bx = 0;  // rounds, and code boxes of earlier items
    bool ok = true;
    for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
      int p0, p1, b, e, u, held = -1;  // held: the box (of the item) being read
      item_pairs(item, p0, p1);
      for (Runs rs(g, p0, p1); ok && rs.next(g, b, e, u);) {
        for (int p = b; p < e; p += 2, ++rd) {
          const int as = static_cast<int>(rd % kSlots);
          if (!mbar_wait_warp(&aempty[as], ((rd / kSlots) & 1u) ^ 1u, g.status)) {
            ok = false;
            break;
          }
          tc_fence_after();  // the MMAs that read the slot before are done
          const int n = min(2, e - p);
          for (int i = 0; i < n; ++i) {
            const int pb = (p + i - p0) >> 4, off = (p + i - p0) & 15;  // box, two words of it
            const int cs = static_cast<int>((bx + pb) % kCRing);
            if (pb != held) {
              if (held >= 0) {
                __syncwarp();
                if (lane == 0) mbar_arrive(&cempty[(bx + held) % kCRing]);
              }
              if (!mbar_wait_warp(&cfull[cs], ((bx + pb) / kCRing) & 1u, g.status)) {
                ok = false;
                break;
              }
              held = pb;
            }
            const uint2 w = *reinterpret_cast<const uint2*>(csm + cs * kCBox + r * 128 +
                                                            (((off >> 1) ^ (r & 7)) << 4) + (off & 1) * 8);
            uint32_t v[16], x[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              v[j] = ((w.x << (15 - j)) & 0x80008000u) ^ 0xBF80BF80u;
              x[j] = ((w.y << (15 - j)) & 0x80008000u) ^ 0xBF80BF80u;
            }
            tmem_st16_issue(a_lane + 64u * as + 32u * i, v);
            tmem_st16_issue(a_lane + 64u * as + 32u * i + 16u, x);
          }
          if (!ok) break;
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&afull[as]);
        }
      }
      if (!ok) break;
      __syncwarp();
      if (lane == 0) mbar_arrive(&cempty[(bx + held) % kCRing]);
      bx += (p1 - p0 + 15) >> 4;
    }
  } else if (warp == kMmaW) {
    // ---------------------------------------------------------- issuer
    {
      const uint32_t idesc = idesc_bf16_f32(128, 2 * g.QB, 0, 0);
      const uint64_t ydesc = sdesc_sw128(smem_u32(smem), 16, 1024);
      uint32_t rd = 0, py = 0, run = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
        int p0, p1, b, e, u;
        item_pairs(item, p0, p1);
        for (Runs rs(g, p0, p1); ok && rs.next(g, b, e, u); ++run) {
          if (!mbar_wait_warp(dempty, (run & 1u) ^ 1u, g.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          for (int p = b; p < e && ok; p += 2, ++rd) {
            const int as = static_cast<int>(rd % kSlots), n = min(2, e - p);
            if (!mbar_wait_warp(&afull[as], (rd / kSlots) & 1u, g.status)) {
              ok = false;
              break;
            }
            for (int i = 0; i < n; ++i, ++py) {
              const int ys = static_cast<int>(py % kYRing);
              if (!mbar_wait_warp(&yfull[ys], (py / kYRing) & 1u, g.status)) {
                ok = false;
                break;
              }
              tc_fence_after();
              const uint64_t y = ydesc + ((ys * kYBox) >> 4);
              const uint32_t a = tmem + kA0 + 64u * as + 32u * i;
              if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                  tc_mma_f16_ta(tmem, a + 8u * kk, y + 2 * kk, idesc, (p != b || i != 0 || kk != 0) ? 1u : 0u);
                tc_commit(&yempty[ys]);
              }
            }
            if (ok && elect_one()) tc_commit(&aempty[as]);
          }
          if (ok && elect_one()) tc_commit(dfull);
        }
      }
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------- TMA producer
    if (lane == 0) {
      const uint32_t half = static_cast<uint32_t>(g.QB) * 128u;
      uint32_t py = 0, bx = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
        int p0, p1;
        item_pairs(item, p0, p1);
        const int qt = item % g.nqt, rt = item / (g.nqt * g.S);
        for (int p = p0; p < p1; ++p, ++py) {
          if (((p - p0) & 15) == 0) {
            const int cs = static_cast<int>(bx % kCRing);
            if (!mbar_wait(&cempty[cs], ((bx / kCRing) & 1u) ^ 1u, g.status)) {
              ok = false;
              break;
            }
            mbar_arrive_expect_tx(&cfull[cs], kCBox);
            tma_load_2d(csm + cs * kCBox, &tmC, 2 * p, rt * 128, &cfull[cs]);
            ++bx;
          }
          const int ys = static_cast<int>(py % kYRing);
          if (!mbar_wait(&yempty[ys], ((py / kYRing) & 1u) ^ 1u, g.status)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&yfull[ys], 2 * half);
          tma_load_2d(smem + ys * static_cast<size_t>(kYBox), &tmHi, p * 64, qt * g.QB, &yfull[ys]);
          tma_load_2d(smem + ys * static_cast<size_t>(kYBox) + half, &tmLo, p * 64, qt * g.QB, &yfull[ys]);
        }
      }
    }
    __syncwarp();
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaW) tmem_dealloc(tmem, 512);
}

// y (fp32) -> bf16 hi = rn(y) and lo = rn(y - hi), rows of D; coordinate 32 w + j + 16 h
// at position 32 w + 2 j + h (the order of a code word's TMEM columns). Eight
// coordinates a thread: j = 4 t .. 4 t + 3 and the same + 16 of one word.
__global__ void __launch_bounds__(256) k_split_queries_perm(const float* __restrict__ y, int ldq, int D,
                                                            uint4* __restrict__ hi, uint4* __restrict__ lo) {
  const int q = blockIdx.y;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < D / 8; e += gridDim.x * blockDim.x) {
    const float* src = y + static_cast<size_t>(q) * ldq + 32 * (e >> 2) + 4 * (e & 3);
    uint32_t h[4], l[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float a = src[j], b = src[j + 16];
      const __nv_bfloat16 ha = __float2bfloat16_rn(a), hb = __float2bfloat16_rn(b);
      const __nv_bfloat16 la = __float2bfloat16_rn(a - __bfloat162float(ha)),
                          lb = __float2bfloat16_rn(b - __bfloat162float(hb));
      h[j] = __bfloat16_as_ushort(ha) | (static_cast<uint32_t>(__bfloat16_as_ushort(hb)) << 16);
      l[j] = __bfloat16_as_ushort(la) | (static_cast<uint32_t>(__bfloat16_as_ushort(lb)) << 16);
    }
    const size_t o = static_cast<size_t>(q) * (D / 8) + e;
    hi[o] = make_uint4(h[0], h[1], h[2], h[3]);
    lo[o] = make_uint4(l[0], l[1], l[2], l[3]);
  }
}

struct PaperPlan {
  int QB, nqt, nrt, npair, S, pps, ldp;
  size_t query, total;  // workspace of the queries alone, and with the slabs
};

int paper_tile_queries(int Q) {
  const int n = (Q + kQB - 1) / kQB;
  return ((Q + n - 1) / n + 15) / 16 * 16;
}

// K ranges (whole code boxes): the number that leaves the request's last wave of items
// fullest, counting four pairs of a range's time for its start, drain and sum.
PaperPlan paper_plan(int N, long long D, int Q, ScoreRequest all, int num_sms) {
  PaperPlan p;
  p.QB = paper_tile_queries(Q);
  p.nqt = (Q + p.QB - 1) / p.QB;
  p.nrt = (N + 127) / 128;
  p.npair = static_cast<int>(D / 64);
  const int nbox = (p.npair + 15) / 16;
  const int qb = paper_tile_queries(all.Q);
  const long long tiles = static_cast<long long>((all.Q + qb - 1) / qb) * ((all.N + 127) / 128);
  long long best = -1;
  p.S = 1;
  p.pps = 16 * nbox;
  for (int want = 1; want <= 16 && want <= nbox; ++want) {
    const int per = (nbox + want - 1) / want, S = (nbox + per - 1) / per;
    const long long cost = (tiles * S + num_sms - 1) / num_sms * (16 * per + 4);
    if (best < 0 || cost < best) {
      best = cost;
      p.S = S;
      p.pps = 16 * per;
    }
  }
  p.ldp = (N + 3) & ~3;
  auto al = [](size_t x) { return (x + 255) & ~size_t(255); };
  p.query = al(static_cast<size_t>(Q) * D * 4);
  p.total = p.query + (p.S > 1 ? al(static_cast<size_t>(p.S) * Q * p.ldp * 4) : 0);
  return p;
}

}  // namespace

bool score_paper_supported(int N, const int* ks, int U, int Q, const void* train, int ldt) {
  if (U < 1 || U > kMaxMods || Q < 1 || Q > 65535 || N < 1) return false;
  if ((ldt & 3) || (reinterpret_cast<uintptr_t>(train) & 15)) return false;
  if (static_cast<long long>((N + 127) / 128) * ((Q + kQB - 1) / kQB) * 16 >= (1ll << 30)) return false;
  for (int u = 0; u < U; ++u)
    if (ks[u] <= 0 || ks[u] % 64) return false;
  return true;
}

size_t score_paper_ws_bytes(int N, const int* ks, int U, int Q, ScoreRequest all, int num_sms) {
  long long D = 0;
  for (int u = 0; u < U; ++u) D += ks[u];
  return paper_plan(N, D, Q, all, num_sms).total;
}

cudaError_t launch_score_paper_tc(const uint32_t* train, int ldt, const float* ts, int ldts, int N, const int* ks,
                                  int U, const float* y, int ldy, int Q, ScoreRequest all, float* out, int ldo, void* ws,
                                  size_t ws_bytes, int num_sms, unsigned* status, cudaStream_t st) {
  PaperArgs g;  // ~4 KB parameter block, copied at launch
  int D = 0;
  for (int u = 0; u < U; ++u) {
    D += ks[u];
    g.pend[u] = D / 64;
  }
  PaperPlan p = paper_plan(N, D, Q, all, num_sms);
  if (ws_bytes < p.total) {  // room for the queries alone: one K range
    p.S = 1;
    p.pps = (p.npair + 15) / 16 * 16;
  }
  uint16_t* hi = static_cast<uint16_t*>(ws);
  uint16_t* lo = hi + static_cast<size_t>(Q) * D;
  float* part = reinterpret_cast<float*>(static_cast<char*>(ws) + p.query);
  k_split_queries_perm<<<dim3(std::max(1, std::min((D / 8 + 255) / 256, 64)), Q), 256, 0, st>>>(
      y, ldy, D, reinterpret_cast<uint4*>(hi), reinterpret_cast<uint4*>(lo));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  CUtensorMap tc, th, tl;
  const uint64_t cd[2] = {static_cast<uint64_t>(D / 32), static_cast<uint64_t>(N)};
  const uint64_t cs[1] = {static_cast<uint64_t>(ldt) * 4};
  const uint32_t cb[2] = {32, 128};
  const uint64_t yd[2] = {static_cast<uint64_t>(D), static_cast<uint64_t>(Q)};
  const uint64_t ys[1] = {static_cast<uint64_t>(D) * 2};
  const uint32_t yb[2] = {64, static_cast<uint32_t>(p.QB)};
  if (make_tmap(&tc, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, train, cd, cs, cb, CU_TENSOR_MAP_SWIZZLE_128B) ||
      make_tmap(&th, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, hi, yd, ys, yb, CU_TENSOR_MAP_SWIZZLE_128B) ||
      make_tmap(&tl, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, lo, yd, ys, yb, CU_TENSOR_MAP_SWIZZLE_128B))
    return cudaErrorInvalidValue;
  g.N = N;
  g.Q = Q;
  g.QB = p.QB;
  g.U = U;
  g.npair = p.npair;
  g.pps = p.pps;
  g.nrt = p.nrt;
  g.nqt = p.nqt;
  g.S = p.S;
  g.n_items = p.nrt * p.nqt * p.S;
  g.ldts = ldts;
  g.ts = ts;
  g.out = p.S > 1 ? part : out;
  g.ldo = p.S > 1 ? p.ldp : ldo;
  g.slab = static_cast<size_t>(Q) * p.ldp;
  g.status = status;
  e = cudaFuncSetAttribute(k_score_paper, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kSmem));
  if (e != cudaSuccess) return e;
  k_score_paper<<<std::min(g.n_items, num_sms), kThreads, kSmem, st>>>(tc, th, tl, g);
  e = cudaGetLastError();
  if (e != cudaSuccess || p.S == 1) return e;
  return launch_sum_slabs(part, p.S, g.slab, p.ldp, N, Q, out, ldo, st);
}
