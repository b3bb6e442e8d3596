// tcgen05 tensor-core kernels (bf16 in, fp32 accumulate in TMEM), fed by TMA.
//
// k_tc_gemm -- D[M x N] = sum_a X_a[M x K] W[N x K]^T, both operands K-major.
//   Used twice per module for the Kronecker rotations of Sec. 2.2
//   (A~ = A V_A[C]^T over the retained columns, S~ = S V_S[R]^T over the
//   retained rows; M = B*T tokens) and once for the second-stage projection
//   x = P^T z (Eq. second_stage; M = B examples, N = k, K = m) where z enters as
//   a bf16 hi + lo pair (two A operands into the same accumulator).
//   Epilogue 0 writes D as a bf16 hi/lo pair (hi = rn(D), lo = rn(D - hi)), so
//   the next contraction sees D to ~16 significant bits; epilogue 1 writes an
//   fp32 partial slab per K split.
//
// k_tc_contract -- for example b and one active 128 x 128 tile (R block rt,
//   C block ct) of the retained block: G~_b[tile] = sum_t S~_b[t, rows]^T
//   A~_b[t, cols] with K = tokens, both operands MN-major (chunks of eight columns).
//   hi*hi + hi*lo + lo*hi: three MMAs per K step. The epilogue stages the fp32
//   tile in shared memory and gathers the retained entries of the tile,
//   scaled by (Lambda + lambda)^{-1/2} (Eq. first_stage), into z.
//
// Warp roles (192 threads): warp 0 issues TMA, warp 1 owns TMEM and issues
// MMAs (one lane), warps 2-5 run the epilogue (warp w reads TMEM lanes
// 32*(w%4)..+31). Every mbarrier wait is bounded (eogp_dev.cuh); after a
// timeout every role falls through to the common exit, which frees TMEM.
#include <algorithm>
#include <cstdlib>
#include <mutex>

#include "eogp_dev.cuh"
#include "eogp_internal.h"
#include "rotate_order.h"

using namespace eogp;

namespace {

constexpr int kThreads = 192;
constexpr uint32_t kABytes = 128u * 64u * 2u;  // 128 rows x 64 bf16 (one 128-byte swizzle row each)

struct GemmArgs {
  int M, N, K, BN, stages, nA, nW, kbps, epi, ldo;
  float alpha;  // epilogue 1: output scale
  void* out0;
  void* out1;
  size_t slab;
  unsigned* status;
};

__device__ __forceinline__ uint32_t pack_bf16x2(__nv_bfloat16 a, __nv_bfloat16 b) {
  return static_cast<uint32_t>(__bfloat16_as_ushort(a)) |
         (static_cast<uint32_t>(__bfloat16_as_ushort(b)) << 16);
}

__device__ __forceinline__ uint32_t tmem_cols_for(int n) {
  return n <= 32 ? 32u : n <= 64 ? 64u : n <= 128 ? 128u : 256u;
}

__global__ void __launch_bounds__(kThreads, 1)
    k_tc_gemm(const __grid_constant__ CUtensorMap tmX0, const __grid_constant__ CUtensorMap tmX1,
              const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmW1,
              const GemmArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t b_bytes = static_cast<uint32_t>(g.BN) * 128u;
  const uint32_t stage_bytes = static_cast<uint32_t>(g.nA) * kABytes + static_cast<uint32_t>(g.nW) * b_bytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + static_cast<size_t>(g.stages) * stage_bytes);
  uint64_t* empty = full + g.stages;
  uint64_t* done = empty + g.stages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  const uint32_t tmem_cols = tmem_cols_for(g.BN);

  const int n0 = blockIdx.x * g.BN, m0 = blockIdx.y * 128;
  const int nkb_total = (g.K + 63) / 64;
  const int kb0 = blockIdx.z * g.kbps;
  const int nkb = max(0, min(g.kbps, nkb_total - kb0));

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmX0);
    if (g.nA > 1) tma_prefetch_desc(&tmX1);
    tma_prefetch_desc(&tmW);
    if (g.nW > 1) tma_prefetch_desc(&tmW1);
    for (int s = 0; s < g.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      int rs = 0;
      uint32_t rph = 0;
      for (int i = 0; i < nkb; ++i) {
        const int s = rs;
        const uint32_t ph = rph;
        if (++rs == g.stages) {
          rs = 0;
          rph ^= 1u;
        }
        if (!mbar_wait(&empty[s], ph ^ 1u, g.status)) break;
        uint8_t* st = smem + static_cast<size_t>(s) * stage_bytes;
        mbar_arrive_expect_tx(&full[s], stage_bytes);
        const int kx = (kb0 + i) * 64;
        tma_load_2d(st, &tmX0, kx, m0, &full[s]);
        if (g.nA > 1) tma_load_2d(st + kABytes, &tmX1, kx, m0, &full[s]);
        tma_load_2d(st + g.nA * kABytes, &tmW, kx, n0, &full[s]);
        if (g.nW > 1) tma_load_2d(st + g.nA * kABytes + b_bytes, &tmW1, kx, n0, &full[s]);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    {
      const uint32_t idesc = idesc_bf16_f32(128, g.BN, 0, 0);
      int rs = 0;
      uint32_t rph = 0;
      for (int i = 0; i < nkb; ++i) {
        const int s = rs;
        const uint32_t ph = rph;
        if (++rs == g.stages) {
          rs = 0;
          rph ^= 1u;
        }
        if (!mbar_wait_warp(&full[s], ph, g.status)) break;
        tc_fence_after();
        const uint32_t sa = smem_u32(smem + static_cast<size_t>(s) * stage_bytes);
        const uint32_t sb = sa + g.nA * kABytes;
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            for (int w = 0; w < g.nW; ++w) {
              const uint64_t bd = sdesc_sw128(sb + w * b_bytes + kk * 32, 16, 1024);
              for (int a = 0; a < g.nA; ++a) {
                if (a == 1 && w == 1) continue;  // lo x lo: below the hi/lo pair's precision
                const uint64_t ad = sdesc_sw128(sa + a * kABytes + kk * 32, 16, 1024);
                tc_mma_f16(tmem, ad, bd, idesc, (i | kk | a | w) != 0 ? 1u : 0u);
              }
            }
          }
          tc_commit(&empty[s]);
        }
      }
      if (elect_one()) tc_commit(done);
    }
    __syncwarp();
  } else {
    const int q = warp & 3;
    uint32_t ok = 1;
    if (lane == 0) ok = mbar_wait(done, 0, g.status) ? 1u : 0u;
    ok = __shfl_sync(0xffffffffu, ok, 0);
    __syncwarp();
    tc_fence_after();
    if (ok && nkb > 0) {
      const int row = m0 + q * 32 + lane;
      const uint32_t tbase = tmem + (static_cast<uint32_t>(q * 32) << 16);
      if (g.epi == 0) {
        __nv_bfloat16* hi = static_cast<__nv_bfloat16*>(g.out0);
        __nv_bfloat16* lo = static_cast<__nv_bfloat16*>(g.out1);
        for (int c = 0; c < g.BN; c += 16) {
          float v[16];
          tmem_ld16(tbase + c, v);
          const int col = n0 + c;
          if (row < g.M && col < g.ldo) {
            uint32_t h[8], l[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const __nv_bfloat16 h0 = __float2bfloat16_rn(v[2 * e]);
              const __nv_bfloat16 h1 = __float2bfloat16_rn(v[2 * e + 1]);
              const __nv_bfloat16 l0 = __float2bfloat16_rn(v[2 * e] - __bfloat162float(h0));
              const __nv_bfloat16 l1 = __float2bfloat16_rn(v[2 * e + 1] - __bfloat162float(h1));
              h[e] = pack_bf16x2(h0, h1);
              l[e] = pack_bf16x2(l0, l1);
            }
            const size_t off = static_cast<size_t>(row) * g.ldo + col;
            uint4* ph = reinterpret_cast<uint4*>(hi + off);
            uint4* pl = reinterpret_cast<uint4*>(lo + off);
            ph[0] = make_uint4(h[0], h[1], h[2], h[3]);
            ph[1] = make_uint4(h[4], h[5], h[6], h[7]);
            pl[0] = make_uint4(l[0], l[1], l[2], l[3]);
            pl[1] = make_uint4(l[4], l[5], l[6], l[7]);
          }
        }
      } else {
        float* out = static_cast<float*>(g.out0) + static_cast<size_t>(blockIdx.z) * g.slab;
        for (int c = 0; c < g.BN; c += 16) {
          float v[16];
          tmem_ld16(tbase + c, v);
          const int col = n0 + c;
          if (row < g.M && col < g.N) {
            float* o = out + static_cast<size_t>(row) * g.ldo + col;
            if (g.alpha != 1.0f) {
#pragma unroll
              for (int e = 0; e < 16; ++e) v[e] *= g.alpha;
            }
            if (col + 16 <= g.N) {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                reinterpret_cast<float4*>(o)[e] =
                    make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
            } else {
              for (int e = 0; e < 16; ++e)
                if (col + e < g.N) o[e] = v[e];
            }
          }
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, tmem_cols);
}

struct ContractArgs {
  int T, stages, n_tiles, n_items, nblkS, nblkA;
  const int32_t* tile_rc;
  const int32_t* grp_start;  // [n_tiles * 4 + 1]: entries per (tile, 32-column chunk)
  const int4* ent;           // {r, (ro << 8) | co, bits of the fp32 scale, 0}
  float* z;
  int ldz;
  __nv_bfloat16* zhi;
  __nv_bfloat16* zlo;
  int ldzb;
  unsigned* status;
};

constexpr uint32_t kOpBytes = 16384u;          // one 128-wide operand tile, 64 tokens
constexpr uint32_t kChunkBytes = 1024u;        // eight of its columns: 64 tokens of 16 bytes
constexpr uint32_t kTokGroup = 128u;           // eight tokens of a chunk
constexpr uint32_t kCStage = 4u * kOpBytes;    // S hi, S lo, A hi, A lo
constexpr uint32_t kCStageBuf = 128u * 33u * 4u;  // 128 x 32 (+1 pad) epilogue staging

// Persistent: one CTA per SM walks items (example b, active tile) with
// b = item / n_tiles, so the tiles of one example run together and share
// operands through L2. Two TMEM accumulators let the gather epilogue of one
// item overlap the loads and MMAs of the next.
__global__ void __launch_bounds__(kThreads, 1)
    k_tc_contract(const __grid_constant__ CUtensorMap tmShi, const __grid_constant__ CUtensorMap tmSlo,
                  const __grid_constant__ CUtensorMap tmAhi, const __grid_constant__ CUtensorMap tmAlo,
                  const ContractArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  const int warp = warp_index(), lane = threadIdx.x & 31;
  float* stage_buf = reinterpret_cast<float*>(smem + static_cast<size_t>(g.stages) * kCStage);
  uint64_t* full = reinterpret_cast<uint64_t*>(reinterpret_cast<uint8_t*>(stage_buf) + kCStageBuf);
  uint64_t* empty = full + g.stages;
  uint64_t* tfull = empty + g.stages;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  const int nkb = (g.T + 63) / 64;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmShi);
    tma_prefetch_desc(&tmSlo);
    tma_prefetch_desc(&tmAhi);
    tma_prefetch_desc(&tmAlo);
    for (int s = 0; s < g.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 4);
    }
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, 256);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;
      int rs = 0;         // ring slot of pipeline iteration it (it % stages)
      uint32_t rph = 0;  // and its phase parity ((it / stages) & 1)
      bool ok = true;
      for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
        const int b = item / g.n_tiles, tile = item % g.n_tiles;
        const int rc = g.tile_rc[tile];
        const int zs = b * g.nblkS + (rc >> 16), za = b * g.nblkA + (rc & 0xFFFF);
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = rs;
          const uint32_t ph = rph;
          if (++rs == g.stages) {
            rs = 0;
            rph ^= 1u;
          }
          if (!mbar_wait(&empty[s], ph ^ 1u, g.status)) {
            ok = false;
            break;
          }
          uint8_t* st = smem + static_cast<size_t>(s) * kCStage;
          mbar_arrive_expect_tx(&full[s], kCStage);
          const int x = kb * 256;  // 64 tokens of 16 bytes, in words
          tma_load_2d(st + 0 * kOpBytes, &tmShi, x, 16 * zs, &full[s]);
          tma_load_2d(st + 1 * kOpBytes, &tmSlo, x, 16 * zs, &full[s]);
          tma_load_2d(st + 2 * kOpBytes, &tmAhi, x, 16 * za, &full[s]);
          tma_load_2d(st + 3 * kOpBytes, &tmAlo, x, 16 * za, &full[s]);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    {
      const uint32_t idesc = idesc_bf16_f32(128, 128, 1, 1);
      uint32_t it = 0;
      int rs = 0;         // ring slot of pipeline iteration it (it % stages)
      uint32_t rph = 0;  // and its phase parity ((it / stages) & 1)
      int i = 0;
      bool ok = true;
      // descriptor of S hi in ring slot rs
      const uint64_t dbase = sdesc_mn_chunks(smem_u32(smem), kTokGroup, kChunkBytes);
      uint64_t dsh = dbase;
      for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x, ++i) {
        const int buf = i & 1;
        const uint32_t aph = static_cast<uint32_t>(i >> 1) & 1u;
        if (!mbar_wait_warp(&tempty[buf], aph ^ 1u, g.status)) break;
        tc_fence_after();
        const uint32_t d = tmem + buf * 128u;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = rs;
          const uint32_t ph = rph;
          const uint64_t sh0 = dsh;  // S hi of this slot; S lo, A hi, A lo follow kOpBytes apart
          if (++rs == g.stages) {
            rs = 0;
            rph ^= 1u;
            dsh = dbase;
          } else {
            dsh += kCStage >> 4;
          }
          if (!mbar_wait_warp(&full[s], ph, g.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          constexpr uint64_t kOp = kOpBytes >> 4, kRow16 = (2 * kTokGroup) >> 4;  // 16 tokens
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              const uint64_t sh = sh0 + kk * kRow16, sl = sh + kOp, ah = sh + 2 * kOp, al = sh + 3 * kOp;
              tc_mma_f16(d, sh, ah, idesc, (kb | kk) != 0 ? 1u : 0u);
              tc_mma_f16(d, sh, al, idesc, 1u);
              tc_mma_f16(d, sl, ah, idesc, 1u);
            }
            tc_commit(&empty[s]);
          }
        }
        if (elect_one()) tc_commit(&tfull[buf]);
      }
    }
    __syncwarp();
  } else {
    const int q = warp & 3;
    const int etid = threadIdx.x - 64;  // 0..127 over the four epilogue warps
    int i = 0;
    for (int item = blockIdx.x; item < g.n_items; item += gridDim.x, ++i) {
      const int buf = i & 1;
      const uint32_t aph = static_cast<uint32_t>(i >> 1) & 1u;
      uint32_t ok = 1;
      if (lane == 0) ok = mbar_wait(&tfull[buf], aph, g.status) ? 1u : 0u;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      __syncwarp();
      tc_fence_after();
      // All four warps must agree before the shared staging is used.
      ok = __syncthreads_and_named(ok);
      if (!ok) break;
      const int b = item / g.n_tiles, tile = item % g.n_tiles;
      const uint32_t tb = tmem + buf * 128u + (static_cast<uint32_t>(q * 32) << 16);
      const size_t zrow = static_cast<size_t>(b);
      for (int j = 0; j < 4; ++j) {
        float v[32];
        tmem_ld32(tb + 32 * j, v);
#pragma unroll
        for (int c = 0; c < 32; ++c) stage_buf[(q * 32 + lane) * 33 + c] = v[c];
        named_bar_sync(1, 128);
        const int e0 = g.grp_start[tile * 4 + j], e1 = g.grp_start[tile * 4 + j + 1];
        for (int e = e0 + etid; e < e1; e += 4 * 128) {
          int4 en[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int eu = e + u * 128;
            en[u] = eu < e1 ? __ldg(&g.ent[eu]) : make_int4(-1, 0, 0, 0);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (en[u].x < 0) continue;
            const int r = en[u].x, off = en[u].y;
            const float val = __int_as_float(en[u].z) * stage_buf[(off >> 8) * 33 + (off & 31)];
            if (g.z) g.z[zrow * g.ldz + r] = val;
            if (g.zhi) {
              const __nv_bfloat16 h = __float2bfloat16_rn(val);
              g.zhi[zrow * g.ldzb + r] = h;
              g.zlo[zrow * g.ldzb + r] = __float2bfloat16_rn(val - __bfloat162float(h));
            }
          }
        }
        named_bar_sync(1, 128);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_relaxed(&tempty[buf]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 256);
}

// k_tc_ekfac -- EK-FAC eigenvalue correction (Sec. 2.2 "EK-FAC approximation":
// the mean square of each coordinate of the gradients in the K-FAC eigenbasis,
// App. C.2: over examples, sequence-level gradients). For one 128 x 128 tile
// (rt, ct) of the full d_out x d_in coordinate block and a run of examples,
// G~_b[tile] is formed exactly as in k_tc_contract (3 MMAs per K step over the
// tokens) and its squares are summed over the run in TMEM (columns 256..383),
// so each item writes one fp32 partial tile. Items are chunk-major
// (item = chunk * n_tiles + tile): CTAs running together read the same
// examples' operands through L2.
struct EkfacArgs {
  int T, stages, n_rt, n_ct, n_tiles, n_items, bpc, B, nblkS, nblkA, d_out, d_in;
  float* part;  // [n_chunks][d_out][d_in]
  unsigned* status;
};

__global__ void __launch_bounds__(kThreads, 1)
    k_tc_ekfac(const __grid_constant__ CUtensorMap tmShi, const __grid_constant__ CUtensorMap tmSlo,
               const __grid_constant__ CUtensorMap tmAhi, const __grid_constant__ CUtensorMap tmAlo,
               const EkfacArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  const int warp = warp_index(), lane = threadIdx.x & 31;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + static_cast<size_t>(g.stages) * kCStage);
  uint64_t* empty = full + g.stages;
  uint64_t* tfull = empty + g.stages;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  const int nkb = (g.T + 63) / 64;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmShi);
    tma_prefetch_desc(&tmSlo);
    tma_prefetch_desc(&tmAhi);
    tma_prefetch_desc(&tmAlo);
    for (int s = 0; s < g.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 4);
    }
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;
      int rs = 0;         // ring slot of pipeline iteration it (it % stages)
      uint32_t rph = 0;  // and its phase parity ((it / stages) & 1)
      bool ok = true;
      for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
        const int chunk = item / g.n_tiles, tile = item % g.n_tiles;
        const int rt = tile / g.n_ct, ct = tile % g.n_ct;
        const int b1 = min(g.B, (chunk + 1) * g.bpc);
        for (int b = chunk * g.bpc; b < b1 && ok; ++b) {
          const int zs = b * g.nblkS + rt, za = b * g.nblkA + ct;
          for (int kb = 0; kb < nkb; ++kb, ++it) {
            const int s = rs;
            const uint32_t ph = rph;
            if (++rs == g.stages) {
              rs = 0;
              rph ^= 1u;
            }
            if (!mbar_wait(&empty[s], ph ^ 1u, g.status)) {
              ok = false;
              break;
            }
            uint8_t* st = smem + static_cast<size_t>(s) * kCStage;
            mbar_arrive_expect_tx(&full[s], kCStage);
            const int x = kb * 256;  // 64 tokens of 16 bytes, in words
            tma_load_2d(st + 0 * kOpBytes, &tmShi, x, 16 * zs, &full[s]);
            tma_load_2d(st + 1 * kOpBytes, &tmSlo, x, 16 * zs, &full[s]);
            tma_load_2d(st + 2 * kOpBytes, &tmAhi, x, 16 * za, &full[s]);
            tma_load_2d(st + 3 * kOpBytes, &tmAlo, x, 16 * za, &full[s]);
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    {
      const uint32_t idesc = idesc_bf16_f32(128, 128, 1, 1);
      uint32_t it = 0;
      int rs = 0;         // ring slot of pipeline iteration it (it % stages)
      uint32_t rph = 0;  // and its phase parity ((it / stages) & 1)
      int i = 0;  // examples issued by this CTA (selects the TMEM buffer)
      bool ok = true;
      for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
        const int chunk = item / g.n_tiles;
        const int b1 = min(g.B, (chunk + 1) * g.bpc);
        for (int b = chunk * g.bpc; b < b1 && ok; ++b, ++i) {
          const int buf = i & 1;
          const uint32_t aph = static_cast<uint32_t>(i >> 1) & 1u;
          if (!mbar_wait_warp(&tempty[buf], aph ^ 1u, g.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem + buf * 128u;
          for (int kb = 0; kb < nkb; ++kb, ++it) {
            const int s = rs;
            const uint32_t ph = rph;
            if (++rs == g.stages) {
              rs = 0;
              rph ^= 1u;
            }
            if (!mbar_wait_warp(&full[s], ph, g.status)) {
              ok = false;
              break;
            }
            tc_fence_after();
            const uint32_t sa = smem_u32(smem + static_cast<size_t>(s) * kCStage);
            if (elect_one()) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {
                const uint32_t o = kk * 2 * kTokGroup;  // 16 tokens
                const uint64_t sh = sdesc_mn_chunks(sa + 0 * kOpBytes + o, kTokGroup, kChunkBytes);
                const uint64_t sl = sdesc_mn_chunks(sa + 1 * kOpBytes + o, kTokGroup, kChunkBytes);
                const uint64_t ah = sdesc_mn_chunks(sa + 2 * kOpBytes + o, kTokGroup, kChunkBytes);
                const uint64_t al = sdesc_mn_chunks(sa + 3 * kOpBytes + o, kTokGroup, kChunkBytes);
                tc_mma_f16(d, sh, ah, idesc, (kb | kk) != 0 ? 1u : 0u);
                tc_mma_f16(d, sh, al, idesc, 1u);
                tc_mma_f16(d, sl, ah, idesc, 1u);
              }
              tc_commit(&empty[s]);
            }
          }
          if (elect_one()) tc_commit(&tfull[buf]);
        }
      }
    }
    __syncwarp();
  } else {
    const int q = warp & 3;
    const uint32_t lane_base = static_cast<uint32_t>(q * 32) << 16;
    const int row_in = q * 32 + lane;
    int i = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < g.n_items && ok; item += gridDim.x) {
      const int chunk = item / g.n_tiles, tile = item % g.n_tiles;
      const int rt = tile / g.n_ct, ct = tile % g.n_ct;
      const int b0 = chunk * g.bpc, b1 = min(g.B, (chunk + 1) * g.bpc);
      for (int b = b0; b < b1; ++b, ++i) {
        const int buf = i & 1;
        const uint32_t aph = static_cast<uint32_t>(i >> 1) & 1u;
        uint32_t w_ok = 1;
        if (lane == 0) w_ok = mbar_wait(&tfull[buf], aph, g.status) ? 1u : 0u;
        w_ok = __shfl_sync(0xffffffffu, w_ok, 0);
        __syncwarp();
        tc_fence_after();
        if (!__syncthreads_and_named(w_ok)) {
          ok = false;
          break;
        }
        for (int j = 0; j < 4; ++j) {
          float v[32], acc[32];
          tmem_ld32(tmem + lane_base + buf * 128u + 32 * j, v);
          if (b == b0) {
#pragma unroll
            for (int c = 0; c < 32; ++c) acc[c] = __fmul_rn(v[c], v[c]);
          } else {
            tmem_ld32(tmem + lane_base + 256u + 32 * j, acc);
#pragma unroll
            for (int c = 0; c < 32; ++c) acc[c] = __fadd_rn(acc[c], __fmul_rn(v[c], v[c]));
          }
          if (b + 1 < b1) {
            tmem_st32(tmem + lane_base + 256u + 32 * j, acc);
          } else {
            const int row = rt * 128 + row_in, col0 = ct * 128 + 32 * j;
            if (row < g.d_out) {
              float* dst = g.part + (static_cast<size_t>(chunk) * g.d_out + row) * g.d_in + col0;
#pragma unroll
              for (int c = 0; c < 32; ++c)
                if (col0 + c < g.d_in) dst[c] = acc[c];
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_relaxed(&tempty[buf]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// k_tc_ekfac2 -- the same sums on CTA pairs (cta_group::2): 256 x N tiles, N = 64 to
// 256 in steps of 64. Each CTA of a pair loads its own 128 columns of S~ and its half
// of the N columns of A~, hi and lo; its accumulator holds its 128 rows. Per MMA flop
// that is a third to a half of the shared-memory reads of a 128 x 128 tile, which at
// 128 bytes a cycle take as long as its MMA, and half the L2 reads. TMEM holds two
// accumulators of N columns, so the squares are summed in registers: eight epilogue
// warps, N / 2 columns of 32 rows each. Examples, runs and the order of all sums are
// those of k_tc_ekfac, the results bit for bit the same.
struct Ekfac2Args {
  int stages, nkb, N, n_ct, n_tiles, n_items, bpc, B, chS, chA, d_out, d_in;
  float* part;  // [n_chunks][d_out][d_in]
  unsigned* status;
};
constexpr int kEk2Threads = 320;

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kEk2Threads, 1)
    k_tc_ekfac2(const __grid_constant__ CUtensorMap tmShi, const __grid_constant__ CUtensorMap tmSlo,
                const __grid_constant__ CUtensorMap tmAhi, const __grid_constant__ CUtensorMap tmAlo,
                const Ekfac2Args g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const uint32_t a_bytes = static_cast<uint32_t>(g.N) * 64u;  // N / 2 columns of 64 tokens
  const uint32_t stage_bytes = 2 * kOpBytes + 2 * a_bytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + static_cast<size_t>(g.stages) * stage_bytes);
  uint64_t* empty = full + g.stages;
  uint64_t* tfull = empty + g.stages;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  const int cl = blockIdx.x >> 1, ncl = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmShi);
    tma_prefetch_desc(&tmSlo);
    tma_prefetch_desc(&tmAhi);
    tma_prefetch_desc(&tmAlo);
    for (int s = 0; s < g.stages; ++s) {
      mbar_init(&full[s], 2);   // one expect_tx arrive from each CTA (leader's copy is used)
      mbar_init(&empty[s], 1);  // MMA completion, multicast to both CTAs
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);    // multicast to both CTAs
      mbar_init(&tempty[b], 16);  // 8 epilogue warps x 2 CTAs (leader's copy is used)
    }
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // barriers of both CTAs initialised before any remote arrive
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();
  pdl_wait();

  if (warp == 0) {
    if (lane == 0) {
      int rs = 0;
      uint32_t rph = 0;
      bool ok = true;
      for (int item = cl; item < g.n_items && ok; item += ncl) {
        const int chunk = item / g.n_tiles, tile = item % g.n_tiles;
        const int rt = tile / g.n_ct, ct = tile % g.n_ct;
        const int b1 = min(g.B, (chunk + 1) * g.bpc);
        for (int b = chunk * g.bpc; b < b1 && ok; ++b) {
          const int zs = b * g.chS + rt * 32 + static_cast<int>(rank) * 16;
          const int za = b * g.chA + ct * (g.N / 8) + static_cast<int>(rank) * (g.N / 16);
          for (int kb = 0; kb < g.nkb; ++kb) {
            const int s = rs;
            const uint32_t ph = rph;
            if (++rs == g.stages) {
              rs = 0;
              rph ^= 1u;
            }
            if (!mbar_wait(&empty[s], ph ^ 1u, g.status)) {
              ok = false;
              break;
            }
            const uint32_t st = smem_u32(smem + static_cast<size_t>(s) * stage_bytes);
            const uint32_t fl = mapa_shared(smem_u32(&full[s]), 0);
            mbar_arrive_expect_tx_cluster(fl, stage_bytes);
            const int x = kb * 256;  // 64 tokens of 16 bytes, in words
            tma_load_2d_pair(st, &tmShi, x, zs, fl);
            tma_load_2d_pair(st + kOpBytes, &tmSlo, x, zs, fl);
            tma_load_2d_pair(st + 2 * kOpBytes, &tmAhi, x, za, fl);
            tma_load_2d_pair(st + 2 * kOpBytes + a_bytes, &tmAlo, x, za, fl);
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (rank == 0) {
      const uint32_t idesc = idesc_bf16_f32(256, g.N, 1, 1);
      const uint64_t dbase = sdesc_mn_chunks(smem_u32(smem), kTokGroup, kChunkBytes);
      const uint64_t dstage = stage_bytes >> 4, dsl = kOpBytes >> 4, dal = a_bytes >> 4;
      uint64_t dd = dbase;  // descriptor of S hi in ring slot rs
      int rs = 0;
      uint32_t rph = 0;
      int i = 0;  // examples issued by this pair (selects the TMEM buffer)
      bool ok = true;
      for (int item = cl; item < g.n_items && ok; item += ncl) {
        const int chunk = item / g.n_tiles;
        const int b1 = min(g.B, (chunk + 1) * g.bpc);
        for (int b = chunk * g.bpc; b < b1 && ok; ++b, ++i) {
          const int buf = i & 1;
          const uint32_t aph = static_cast<uint32_t>(i >> 1) & 1u;
          if (!mbar_wait_warp(&tempty[buf], aph ^ 1u, g.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t d = tmem + buf * 256u;
          for (int kb = 0; kb < g.nkb; ++kb) {
            const int s = rs;
            const uint32_t ph = rph;
            const uint64_t sh0 = dd;
            if (++rs == g.stages) {
              rs = 0;
              rph ^= 1u;
              dd = dbase;
            } else {
              dd += dstage;
            }
            if (!mbar_wait_warp(&full[s], ph, g.status)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (elect_one()) {
#pragma unroll
              for (int kk = 0; kk < 4; ++kk) {
                const uint64_t sh = sh0 + kk * (2 * kTokGroup >> 4);  // 16 tokens
                const uint64_t ah = sh + 2 * dsl;
                tc_mma_f16_pair(d, sh, ah, idesc, (kb | kk) != 0 ? 1u : 0u);
                tc_mma_f16_pair(d, sh, ah + dal, idesc, 1u);
                tc_mma_f16_pair(d, sh + dsl, ah, idesc, 1u);
              }
              tc_commit_pair_mc(&empty[s], 0x3);
            }
          }
          if (elect_one()) tc_commit_pair_mc(&tfull[buf], 0x3);
        }
      }
    }
    __syncwarp();
  } else {
    const int q = warp & 3, half = (warp - 2) >> 2, nj = g.N / 64;
    const uint32_t tb = tmem + (static_cast<uint32_t>(q * 32) << 16) + static_cast<uint32_t>(half * (g.N / 2));
    int i = 0;
    uint32_t ok = 1;
    for (int item = cl; item < g.n_items && ok; item += ncl) {
      const int chunk = item / g.n_tiles, tile = item % g.n_tiles;
      const int rt = tile / g.n_ct, ct = tile % g.n_ct;
      const int b0 = chunk * g.bpc, b1 = min(g.B, (chunk + 1) * g.bpc);
      float acc[4][32];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int c = 0; c < 32; ++c) acc[j][c] = 0.f;
      for (int b = b0; b < b1; ++b, ++i) {
        const int buf = i & 1;
        const uint32_t aph = static_cast<uint32_t>(i >> 1) & 1u;
        if (lane == 0) ok = mbar_wait(&tfull[buf], aph, g.status) ? 1u : 0u;
        ok = __shfl_sync(0xffffffffu, ok, 0);
        __syncwarp();
        tc_fence_after();
        if (!ok) break;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (j < nj) {
            float v[32];
            tmem_ld32(tb + buf * 256u + 32 * j, v);
#pragma unroll
            for (int c = 0; c < 32; ++c) acc[j][c] = __fadd_rn(acc[j][c], __fmul_rn(v[c], v[c]));
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_relaxed_cluster(mapa_shared(smem_u32(&tempty[buf]), 0));
      }
      const int row = rt * 256 + static_cast<int>(rank) * 128 + q * 32 + lane;
      if (ok && row < g.d_out) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int col0 = ct * g.N + half * (g.N / 2) + 32 * j;
          // d_in is a multiple of 8
          float* dst = g.part + (static_cast<size_t>(chunk) * g.d_out + row) * g.d_in + col0;
#pragma unroll
          for (int c = 0; c < 32; c += 4)
            if (j < nj && col0 + c < g.d_in)
              *reinterpret_cast<float4*>(dst + c) = make_float4(acc[j][c], acc[j][c + 1], acc[j][c + 2], acc[j][c + 3]);
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // neither CTA leaves while its peer may still signal it
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem, 512);
}

// A finite, normal float as a double, on the integer pipe (the exponent's bias and
// the significand's place differ): conversions share the few 64-bit lanes of an SM
// with the additions.
__device__ __forceinline__ double widen(float x) {
  const uint32_t u = __float_as_uint(x);
  if ((u << 1) - 0x01000000u >= 0xFE000000u) return static_cast<double>(x);  // zero, subnormal, infinite, NaN
  return __hiloint2double(static_cast<int>((u & 0x80000000u) | (((u & 0x7FFFFFFFu) >> 3) + 0x38000000u)),
                          static_cast<int>(u << 29));
}

// sumsq[j * ld + i] (+)= sum over chunks c of part[c][j][i], chunks in order (fp64).
// A thread sums four neighbouring columns of a row (16-byte loads). Bound by the
// 64-bit additions: with a conversion and an addition per partial, three partials of
// 3072 x 768 sums took 29 us whatever the loads; 8 us so.
__global__ void __launch_bounds__(64)
    k_ekfac_finalize(const float* __restrict__ part, int n_chunks, int d_out, int d_in, double* __restrict__ sumsq,
                     int ld, int accumulate) {
  pdl_wait();
  const int col = 4 * (blockIdx.x * 64 + threadIdx.x);
  if (col >= d_in) return;  // d_in is a multiple of 8
  const size_t slab = static_cast<size_t>(d_out) * d_in;
  for (int row = blockIdx.y; row < d_out; row += gridDim.y) {
    const float* p = part + static_cast<size_t>(row) * d_in + col;
    const float4 f = *reinterpret_cast<const float4*>(p);
    double t[4] = {widen(f.x), widen(f.y), widen(f.z), widen(f.w)};
#pragma unroll 4
    for (int c = 1; c < n_chunks; ++c) {
      const float4 v = *reinterpret_cast<const float4*>(p + c * slab);
      t[0] += widen(v.x);
      t[1] += widen(v.y);
      t[2] += widen(v.z);
      t[3] += widen(v.w);
    }
    double* o = sumsq + static_cast<size_t>(row) * ld + col;
#pragma unroll
    for (int c = 0; c < 4; ++c) o[c] = accumulate ? o[c] + t[c] : t[c];
  }
}

size_t gemm_smem_bytes(int BN, int stages, int nA, int nW = 1) {
  return 1024 + static_cast<size_t>(stages) * (nA * kABytes + nW * BN * 128u) + (2 * stages + 1) * 8 + 16;
}

size_t contract_smem_bytes(int stages) {
  return 1024 + static_cast<size_t>(stages) * kCStage + kCStageBuf + (2 * stages + 4) * 8 + 16;
}


// ------------------------------------------------------------------------
// k_tc_rotate -- persistent rotation GEMM: D = X W^T written as bf16 hi/lo.
// One CTA per SM walks a static tile schedule (tile t -> M block t / nN,
// N block t % nN, so the nN CTAs sharing an activation block run together and
// the block is read from HBM once). Two TMEM accumulators alternate between
// tiles: the MMA warp fills one while the epilogue warps drain the other.
// Epilogue: 32-column TMEM loads, hi/lo split, 16-byte stores. The output is laid
// out in chunks of eight columns for the contraction that reads it: element (row =
// b*T + t, col) sits at ((b * (ldo/8) + col/8) * T + t) * 8 + col % 8, so the 32
// tokens of a warp write 512 contiguous bytes an instruction (and a chunk of 64
// tokens is the no-swizzle operand tile as it stands). With token rows of 128
// columns a warp's store touched 32 lines, and those partial-line stores, not their
// DRAM traffic, set the pace of short reductions: K = 768 over 131,072 rows took 167
// us (102 without the stores, 172 with all of them aimed at 8 MB of L2), 112 now.
struct RotArgs {
  int M, K, BN, stages, nN, n_tiles, ldo, T, nbias;
  __nv_bfloat16* hi;
  __nv_bfloat16* lo;
  const float* bias;        // per output column (the constant-1 input channel), or null
  const int32_t* lengths;   // tokens kept per example (later tokens give 0), or null
  unsigned* status;
};

// One output row's place: its first element in the chunked layout (element (row,
// col) at base + (col >> 3) * 8 T + (col & 7)), and whether it is a padding token.
struct RotRow {
  size_t base;
  bool in, pad;
  __device__ __forceinline__ RotRow(const RotArgs& g, int row) {
    in = row < g.M;
    const int b = row / g.T, tok = row - b * g.T;
    base = (static_cast<size_t>(b) * (g.ldo >> 3) * g.T + tok) * 8;
    pad = in && g.lengths && tok >= __ldg(g.lengths + b);
  }
};

// One W-column chunk (W = 32 or 16) of one output row: bias channel and token
// lengths, hi/lo split, 16-byte stores (eight columns each).
template <int W>
__device__ __forceinline__ void rot_store(const RotArgs& g, const RotRow& r, int col, float (&v)[W]) {
  if (g.bias) {
    if (col + W <= g.nbias) {
      float b[W];
#pragma unroll
      for (int e = 0; e < W; ++e) b[e] = __ldg(g.bias + col + e);
#pragma unroll
      for (int e = 0; e < W; ++e) v[e] += b[e];
    } else {
#pragma unroll
      for (int e = 0; e < W; ++e) v[e] += col + e < g.nbias ? __ldg(g.bias + col + e) : 0.f;
    }
  }
  if (r.pad) {
#pragma unroll
    for (int e = 0; e < W; ++e) v[e] = 0.f;
  }
  const size_t step = static_cast<size_t>(g.T) * 8;
  size_t at = r.base + static_cast<size_t>(col >> 3) * step;
#pragma unroll
  for (int q = 0; q < W / 8; ++q, at += step) {
    uint32_t h[4], l[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float v0 = v[8 * q + 2 * e], v1 = v[8 * q + 2 * e + 1];
      const __nv_bfloat162 hi = __floats2bfloat162_rn(v0, v1);
      h[e] = *reinterpret_cast<const uint32_t*>(&hi);
      const __nv_bfloat162 lo = __floats2bfloat162_rn(v0 - __uint_as_float(h[e] << 16),
                                                      v1 - __uint_as_float(h[e] & 0xFFFF0000u));
      l[e] = *reinterpret_cast<const uint32_t*>(&lo);
    }
    if (col + 8 * q < g.ldo) {  // a tile may reach past the padded columns
      *reinterpret_cast<uint4*>(g.hi + at) = make_uint4(h[0], h[1], h[2], h[3]);
      *reinterpret_cast<uint4*>(g.lo + at) = make_uint4(l[0], l[1], l[2], l[3]);
    }
  }
}

// Drains one accumulator row of a BN-column tile (BN a multiple of 16).
__device__ __forceinline__ void rot_drain(const RotArgs& g, uint32_t tb, int row, int n0) {
  const RotRow r(g, row);
  int c = 0;
  for (; c + 32 <= g.BN; c += 32) {
    float v[32];
    tmem_ld32(tb + c, v);
    if (r.in) rot_store<32>(g, r, n0 + c, v);
  }
  if (c < g.BN) {
    float v[16];
    tmem_ld16(tb + c, v);
    if (r.in) rot_store<16>(g, r, n0 + c, v);
  }
}

// One rotation, or two in one launch (the A and S sides of a module): the tiles of
// g[0], then those of g[1], dealt to the CTAs back and forth, so that the shorter
// ones of g[1] go to the CTAs that g[0] left idle.
struct RotBoth {
  RotArgs g[2];
  int n_tiles, stages;     // of both; ring slots of `slot` bytes
  uint32_t slot, tcols;    // TMEM columns (two accumulators)
  __device__ __forceinline__ int tile(int round) const {  // this CTA's tile of a round, n_tiles or more past the end
    const int n = gridDim.x, b = blockIdx.x;
    return round * n + ((round & 1) && g[1].n_tiles ? n - 1 - b : b);
  }
};

__global__ void __launch_bounds__(kThreads, 1)
    k_tc_rotate(const __grid_constant__ CUtensorMap tmX0, const __grid_constant__ CUtensorMap tmW0,
                const __grid_constant__ CUtensorMap tmX1, const __grid_constant__ CUtensorMap tmW1,
                const __grid_constant__ RotBoth p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  const int warp = warp_index(), lane = threadIdx.x & 31;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + static_cast<size_t>(p.stages) * p.slot);
  uint64_t* empty = full + p.stages;
  uint64_t* tfull = empty + p.stages;  // accumulator ready, per TMEM buffer
  uint64_t* tempty = tfull + 2;        // accumulator drained, per TMEM buffer
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  const uint32_t bstride = p.tcols / 2;
  unsigned* status = p.g[0].status;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmX0);
    tma_prefetch_desc(&tmW0);
    if (p.g[1].n_tiles) {
      tma_prefetch_desc(&tmX1);
      tma_prefetch_desc(&tmW1);
    }
    for (int s = 0; s < p.stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);
      mbar_init(&tempty[b], 4);  // one arrive per epilogue warp
    }
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, p.tcols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();

  if (warp == 0) {
    if (lane == 0) {
      int rs = 0;         // ring slot of the next K block
      uint32_t rph = 0;   // and its phase parity
      bool ok = true;
      for (int r = 0, t; ok && (t = p.tile(r)) < p.n_tiles; ++r) {
        const int side = t >= p.g[0].n_tiles ? 1 : 0;
        const RotArgs& g = p.g[side];
        if (side) t -= p.g[0].n_tiles;
        const CUtensorMap* tx = side ? &tmX1 : &tmX0;
        const CUtensorMap* tw = side ? &tmW1 : &tmW0;
        const uint32_t bytes = kABytes + static_cast<uint32_t>(g.BN) * 128u;
        const int nkb = (g.K + 63) / 64, m0 = (t / g.nN) * 128, n0 = (t % g.nN) * g.BN;
        for (int kb = 0; kb < nkb; ++kb) {
          const int s = rs;
          const uint32_t ph = rph;
          if (++rs == p.stages) {
            rs = 0;
            rph ^= 1u;
          }
          if (!mbar_wait(&empty[s], ph ^ 1u, status)) {
            ok = false;
            break;
          }
          uint8_t* st = smem + static_cast<size_t>(s) * p.slot;
          mbar_arrive_expect_tx(&full[s], bytes);
          tma_load_2d(st, tx, kb * 64, m0, &full[s]);
          tma_load_2d(st + kABytes, tw, kb * 64, n0, &full[s]);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // Ring slot, phase and operand descriptors advance incrementally. A descriptor's
    // address field is (byte address >> 4), so +2 steps 32 bytes (K = 16 bf16).
    const uint64_t dbase = sdesc_sw128(smem_u32(smem), 16, 1024);
    const uint64_t dstage = p.slot >> 4, dab = kABytes >> 4;
    uint64_t da = dbase;  // descriptor of operand A in ring slot rs
    int rs = 0;           // ring slot of the next K block
    uint32_t rph = 0;     // and its phase parity
    bool ok = true;
    for (int r = 0, t; ok && (t = p.tile(r)) < p.n_tiles; ++r) {
      const RotArgs& g = p.g[t >= p.g[0].n_tiles ? 1 : 0];
      const uint32_t idesc = idesc_bf16_f32(128, g.BN, 0, 0);
      const int nkb = (g.K + 63) / 64;
      const int buf = r & 1;
      const uint32_t aph = static_cast<uint32_t>(r >> 1) & 1u;
      if (!mbar_wait_warp(&tempty[buf], aph ^ 1u, status)) break;
      tc_fence_after();
      const uint32_t d = tmem + buf * bstride;
      for (int kb = 0; kb < nkb; ++kb) {
        const int s = rs;
        const uint32_t ph = rph;
        const uint64_t a0 = da, b0 = da + dab;
        if (++rs == p.stages) {
          rs = 0;
          rph ^= 1u;
          da = dbase;
        } else {
          da += dstage;
        }
        if (!mbar_wait_warp(&full[s], ph, status)) {
          ok = false;
          break;
        }
        tc_fence_after();
        if (elect_one()) {
          tc_mma_f16(d, a0, b0, idesc, kb != 0 ? 1u : 0u);
          tc_mma_f16(d, a0 + 2, b0 + 2, idesc, 1u);
          tc_mma_f16(d, a0 + 4, b0 + 4, idesc, 1u);
          tc_mma_f16(d, a0 + 6, b0 + 6, idesc, 1u);
          tc_commit(&empty[s]);
        }
      }
      if (elect_one()) tc_commit(&tfull[buf]);
    }
    __syncwarp();
  } else {
    const int q = warp & 3;
    for (int r = 0, t; (t = p.tile(r)) < p.n_tiles; ++r) {
      const int side = t >= p.g[0].n_tiles ? 1 : 0;
      const RotArgs& g = p.g[side];
      if (side) t -= p.g[0].n_tiles;
      const int buf = r & 1;
      const uint32_t aph = static_cast<uint32_t>(r >> 1) & 1u;
      uint32_t ok = 1;
      if (lane == 0) ok = mbar_wait(&tfull[buf], aph, status) ? 1u : 0u;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      __syncwarp();
      tc_fence_after();
      if (!ok) break;
      const int m0 = (t / g.nN) * 128, n0 = (t % g.nN) * g.BN;
      const int row = m0 + q * 32 + lane;
      const uint32_t tb = tmem + buf * bstride + (static_cast<uint32_t>(q * 32) << 16);
      rot_drain(g, tb, row, n0);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_relaxed(&tempty[buf]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, p.tcols);
}

size_t rotate_smem_bytes(int BN, int stages) {
  return 1024 + static_cast<size_t>(stages) * (kABytes + BN * 128u) + (2 * stages + 4) * 8 + 16;
}


// ------------------------------------------------------------------------
// k_tc_rotate2 -- the rotation GEMM on CTA pairs (tcgen05 cta_group::2,
// M = 256). Each CTA of a pair loads its own 128 activation rows and its own
// half of the BN eigenvector rows (no multicast), so per-SM shared-memory
// traffic per MMA flop drops by a third against one CTA per tile; the leader
// CTA (rank 0) issues the M = 256 MMAs, whose accumulator rows are split over
// the two CTAs' TMEM. Pipeline completion (TMA bytes) and accumulator release
// are counted on the leader's barriers; MMA completion is multicast to both
// CTAs. Epilogue as in k_tc_rotate (chunked hi/lo output).
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    k_tc_rotate2(const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmW,
                 const RotArgs g) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int half = g.BN / 2;  // W rows held by this CTA
  const uint32_t stage_bytes = kABytes + static_cast<uint32_t>(half) * 128u;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + static_cast<size_t>(g.stages) * stage_bytes);
  uint64_t* empty = full + g.stages;
  uint64_t* tfull = empty + g.stages;
  uint64_t* tempty = tfull + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 2);
  const uint32_t tcols = g.BN <= 64 ? 128u : g.BN <= 128 ? 256u : 512u;
  const uint32_t bstride = tcols / 2;
  const int nkb = (g.K + 63) / 64;
  const int cl = blockIdx.x >> 1, ncl = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmX);
    tma_prefetch_desc(&tmW);
    for (int s = 0; s < g.stages; ++s) {
      mbar_init(&full[s], 2);   // one expect_tx arrive from each CTA (leader's copy is used)
      mbar_init(&empty[s], 1);  // MMA completion, multicast to both CTAs
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&tfull[b], 1);   // multicast to both CTAs
      mbar_init(&tempty[b], 8);  // 4 epilogue warps x 2 CTAs (leader's copy is used)
    }
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc_pair(tmem_slot, tcols);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // barriers of both CTAs initialised before any remote arrive
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_trigger();

  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;
      int rs = 0;         // ring slot of pipeline iteration it (it % stages)
      uint32_t rph = 0;  // and its phase parity ((it / stages) & 1)
      bool ok = true;
      for (int t = cl; t < g.n_tiles && ok; t += ncl) {
        const int m0 = (t / g.nN) * 256 + static_cast<int>(rank) * 128;
        const int n0 = (t % g.nN) * g.BN + static_cast<int>(rank) * half;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = rs;
          const uint32_t ph = rph;
          if (++rs == g.stages) {
            rs = 0;
            rph ^= 1u;
          }
          if (!mbar_wait(&empty[s], ph ^ 1u, g.status)) {
            ok = false;
            break;
          }
          const uint32_t st = smem_u32(smem + static_cast<size_t>(s) * stage_bytes);
          const uint32_t fl = mapa_shared(smem_u32(&full[s]), 0);
          mbar_arrive_expect_tx_cluster(fl, stage_bytes);
          tma_load_2d_pair(st, &tmX, kb * 64, m0, fl);
          tma_load_2d_pair(st + kABytes, &tmW, kb * 64, n0, fl);
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (rank == 0) {
      // as in k_tc_rotate: slot, phase and descriptors advance incrementally
      const uint32_t idesc = idesc_bf16_f32(256, g.BN, 0, 0);
      const uint64_t dbase = sdesc_sw128(smem_u32(smem), 16, 1024);
      const uint64_t dstage = stage_bytes >> 4, dab = kABytes >> 4;
      uint64_t da = dbase;
      int rs = 0;
      uint32_t rph = 0;
      int i = 0;
      bool ok = true;
      for (int t = cl; t < g.n_tiles && ok; t += ncl, ++i) {
        const int buf = i & 1;
        const uint32_t aph = static_cast<uint32_t>(i >> 1) & 1u;
        if (!mbar_wait_warp(&tempty[buf], aph ^ 1u, g.status)) break;
        tc_fence_after();
        const uint32_t d = tmem + buf * bstride;
        for (int kb = 0; kb < nkb; ++kb) {
          const int s = rs;
          const uint32_t ph = rph;
          const uint64_t a0 = da, b0 = da + dab;
          if (++rs == g.stages) {
            rs = 0;
            rph ^= 1u;
            da = dbase;
          } else {
            da += dstage;
          }
          if (!mbar_wait_warp(&full[s], ph, g.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          if (elect_one()) {
            tc_mma_f16_pair(d, a0, b0, idesc, kb != 0 ? 1u : 0u);
            tc_mma_f16_pair(d, a0 + 2, b0 + 2, idesc, 1u);
            tc_mma_f16_pair(d, a0 + 4, b0 + 4, idesc, 1u);
            tc_mma_f16_pair(d, a0 + 6, b0 + 6, idesc, 1u);
            tc_commit_pair_mc(&empty[s], 0x3);
          }
        }
        if (elect_one()) tc_commit_pair_mc(&tfull[buf], 0x3);
      }
    }
    __syncwarp();
  } else {
    const int q = warp & 3;
    int i = 0;
    for (int t = cl; t < g.n_tiles; t += ncl, ++i) {
      const int buf = i & 1;
      const uint32_t aph = static_cast<uint32_t>(i >> 1) & 1u;
      uint32_t ok = 1;
      if (lane == 0) ok = mbar_wait(&tfull[buf], aph, g.status) ? 1u : 0u;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      __syncwarp();
      tc_fence_after();
      if (!ok) break;
      const int m0 = (t / g.nN) * 256 + static_cast<int>(rank) * 128, n0 = (t % g.nN) * g.BN;
      const int row = m0 + q * 32 + lane;
      const uint32_t tb = tmem + buf * bstride + (static_cast<uint32_t>(q * 32) << 16);
      rot_drain(g, tb, row, n0);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_relaxed_cluster(mapa_shared(smem_u32(&tempty[buf]), 0));
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // neither CTA leaves while its peer may still signal it
  tc_fence_after();
  if (warp == 1) tmem_dealloc_pair(tmem, tcols);
}

size_t rotate2_smem_bytes(int BN, int stages) {
  return 1024 + static_cast<size_t>(stages) * (kABytes + (BN / 2) * 128u) + (2 * stages + 4) * 8 + 16;
}

}  // namespace

static int tmap_bf16_2d(CUtensorMap* tm, const void* base, uint64_t inner, uint64_t rows,
                        uint64_t row_stride_elems, uint32_t box_inner, uint32_t box_rows) {
  const uint64_t dims[2] = {inner, rows};
  const uint64_t strides[1] = {row_stride_elems * 2};
  const uint32_t box[2] = {box_inner, box_rows};
  return make_tmap(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box,
                   CU_TENSOR_MAP_SWIZZLE_128B);
}

// Chunked intermediate [nbatch * 16 chunks][T][8 columns] (bf16), as words: a box is
// 64 tokens (1 KB) of `chunks` chunks, 16 for a 128-column block.
static int tmap_chunked(CUtensorMap* tm, const void* base, uint64_t T, uint64_t nbatch, uint32_t chunks = 16) {
  const uint64_t dims[2] = {4 * T, 16 * nbatch};
  const uint64_t strides[1] = {16 * T};
  const uint32_t box[2] = {256, chunks};
  return make_tmap(tm, CU_TENSOR_MAP_DATA_TYPE_UINT32, 2, base, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_NONE);
}

static cudaError_t launch_tc_gemm_impl(int M, int N, int K, const void* X0, const void* X1, int ldx,
                                      const void* W, const void* W1, int ldw, int Wrows, int splits, int epi,
                                      void* out0, void* out1, int ldo, size_t slab, float alpha,
                                      TcGemmCfg cfg, bool behind, unsigned* status, cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  const int nA = X1 ? 2 : 1;
  const int nW = W1 ? 2 : 1;
  CUtensorMap tX0, tX1, tW, tW1;
  if (tmap_bf16_2d(&tX0, X0, static_cast<uint64_t>(K), static_cast<uint64_t>(M), ldx, 64, 128))
    return cudaErrorInvalidValue;
  if (nA > 1) {
    if (tmap_bf16_2d(&tX1, X1, K, M, ldx, 64, 128)) return cudaErrorInvalidValue;
  } else {
    tX1 = tX0;
  }
  if (tmap_bf16_2d(&tW, W, K, Wrows, ldw, 64, cfg.BN)) return cudaErrorInvalidValue;
  if (nW > 1) {
    if (tmap_bf16_2d(&tW1, W1, K, Wrows, ldw, 64, cfg.BN)) return cudaErrorInvalidValue;
  } else {
    tW1 = tW;
  }
  const int nkb = (K + 63) / 64;
  splits = max(1, min(splits, nkb));
  const int kbps = (nkb + splits - 1) / splits;
  splits = (nkb + kbps - 1) / kbps;
  GemmArgs g;
  g.M = M;
  g.N = N;
  g.K = K;
  g.BN = cfg.BN;
  g.stages = cfg.stages;
  g.nA = nA;
  g.nW = nW;
  g.kbps = kbps;
  g.epi = epi;
  g.ldo = ldo;
  g.alpha = alpha;
  g.out0 = out0;
  g.out1 = out1;
  g.slab = slab;
  g.status = status;
  const size_t smem = gemm_smem_bytes(cfg.BN, cfg.stages, nA, nW);
  cudaError_t e = allow_smem(k_tc_gemm);
  if (e != cudaSuccess) return e;
  dim3 grid((N + cfg.BN - 1) / cfg.BN, (M + 127) / 128, splits);
  if (behind) return launch_behind(k_tc_gemm, grid, kThreads, smem, st, tX0, tX1, tW, tW1, g);
  k_tc_gemm<<<grid, kThreads, smem, st>>>(tX0, tX1, tW, tW1, g);
  return cudaGetLastError();
}

cudaError_t launch_tc_gemm(int M, int N, int K, const void* X0, const void* X1, int ldx,
                                const void* W, int ldw, int Wrows, int splits, int epi,
                                void* out0, void* out1, int ldo, size_t slab, TcGemmCfg cfg,
                                unsigned* status, cudaStream_t st) {
  return launch_tc_gemm_impl(M, N, K, X0, X1, ldx, W, nullptr, ldw, Wrows, splits, epi, out0, out1, ldo,
                             slab, 1.0f, cfg, true, status, st);
}

cudaError_t launch_tc_gemm_hl(int M, int N, int K, const void* Ah, const void* Al, int lda, const void* Bh,
                              const void* Bl, int ldb, float* out, int ldo, float alpha, unsigned* status,
                              cudaStream_t st) {
  // 128-column tiles: a stage holds 2 x 16 KB of A and 2 x 16 KB of B, three stages.
  return launch_tc_gemm_impl(M, N, K, Ah, Al, lda, Bh, Bl, ldb, N, 1, 1, out, nullptr, ldo, 0, alpha,
                             TcGemmCfg{128, 3}, false, status, st);
}

// CTA pairs measured faster for short reductions (K <= 1536: the hi/lo
// epilogue dominates and halving the per-SM operand stream helps) and for few
// output columns (n <= 256: the activations stream from HBM and every 128-row
// tile re-reads the whole eigenvector operand from L2, which the pair halves;
// OLMo-2-1B stack 1,487 -> 1,557 examples/s), and slower for long reductions
// with many columns.
static bool rotate_pairs(int K, int n) { return K <= 1536 || n <= 256; }

// N tile width for `n` output columns: as few tiles of at most 256 columns as
// is cheapest, each a multiple of `gran` (16: the tcgen05 N granularity, for one
// CTA and for CTA pairs, whose halves of N / 2 rows are whole 8-row swizzle
// atoms), counting a fixed per-tile overhead of 32 columns.
int rotate_bn(int n, int gran) {
  const int n0 = (n + 255) / 256;
  int best = 0, best_cost = 1 << 30;
  for (int nN = n0; nN <= n0 + 1; ++nN) {
    const int bn = ((n + nN - 1) / nN + gran - 1) / gran * gran;
    const int cost = nN * bn + 32 * nN;
    if (cost < best_cost) {
      best_cost = cost;
      best = bn;
    }
  }
  return best;
}

static RotArgs rot_args(const RotSide& r, int M, int T, int BN, int m_tile, unsigned* status) {
  RotArgs g;
  g.M = M;
  g.K = r.K;
  g.BN = BN;
  g.stages = 0;
  g.nN = (r.rows + BN - 1) / BN;  // columns past the last tile (padding up to ldo) are not written
  g.n_tiles = ((M + m_tile - 1) / m_tile) * g.nN;
  g.ldo = r.ldo;
  g.T = T;
  g.hi = static_cast<__nv_bfloat16*>(r.hi);
  g.lo = static_cast<__nv_bfloat16*>(r.lo);
  g.bias = r.bias;
  g.nbias = r.rows;
  g.lengths = r.lengths;
  g.status = status;
  return g;
}

// One launch of k_tc_rotate over one side, or over both with tiles of BN columns.
static cudaError_t launch_rot(const RotSide* r, int n, int M, int T, const int* BN, int num_sms, unsigned* status,
                              cudaStream_t st) {
  RotBoth p;
  CUtensorMap tx[2], tw[2];
  int bn = 0;
  for (int i = 0; i < n; ++i) {
    p.g[i] = rot_args(r[i], M, T, BN[i], 128, status);
    bn = std::max(bn, BN[i]);
    if (tmap_bf16_2d(&tx[i], r[i].X, static_cast<uint64_t>(r[i].K), static_cast<uint64_t>(M), r[i].K, 64, 128) ||
        tmap_bf16_2d(&tw[i], r[i].W, r[i].K, r[i].rows, r[i].K, 64, BN[i]))
      return cudaErrorInvalidValue;
  }
  if (n == 1) {
    p.g[1] = p.g[0];
    p.g[1].n_tiles = 0;
    tx[1] = tx[0];
    tw[1] = tw[0];
  }
  p.n_tiles = p.g[0].n_tiles + p.g[1].n_tiles;
  p.slot = kABytes + static_cast<uint32_t>(bn) * 128u;
  p.tcols = bn <= 64 ? 128u : bn <= 128 ? 256u : 512u;
  // As many pipeline stages as fit in 227 KB of shared memory (at most 8).
  p.stages = 2;
  while (p.stages < 8 && rotate_smem_bytes(bn, p.stages + 1) <= 232448) ++p.stages;
  const size_t smem = rotate_smem_bytes(bn, p.stages);
  const cudaError_t e = allow_smem(k_tc_rotate);
  if (e != cudaSuccess) return e;
  k_tc_rotate<<<std::min(p.n_tiles, std::max(1, num_sms)), kThreads, smem, st>>>(tx[0], tw[0], tx[1], tw[1], p);
  return cudaGetLastError();
}

cudaError_t launch_tc_rotate(const RotSide& r, int M, int T, int num_sms, unsigned* status, cudaStream_t st) {
  if (M <= 0) return cudaSuccess;
  const int BN = rotate_bn(r.rows, 16);
  if (!rotate_pairs(r.K, r.rows)) return launch_rot(&r, 1, M, T, &BN, num_sms, status, st);
  // CTA pairs: tiles of 256 rows, W split in halves of BN / 2 rows.
  CUtensorMap tX, tWh;
  if (tmap_bf16_2d(&tX, r.X, static_cast<uint64_t>(r.K), static_cast<uint64_t>(M), r.K, 64, 128) ||
      tmap_bf16_2d(&tWh, r.W, r.K, r.rows, r.K, 64, BN / 2))
    return cudaErrorInvalidValue;
  RotArgs g = rot_args(r, M, T, BN, 256, status);
  g.stages = 2;
  while (g.stages < 8 && rotate2_smem_bytes(BN, g.stages + 1) <= 232448) ++g.stages;
  const size_t smem = rotate2_smem_bytes(BN, g.stages);
  cudaError_t e = allow_smem(k_tc_rotate2);
  if (e != cudaSuccess) return e;
  const int clusters = std::min(g.n_tiles, std::max(1, num_sms / 2));
  k_tc_rotate2<<<2 * clusters, kThreads, smem, st>>>(tX, tWh, g);
  return cudaGetLastError();
}

static long long rot_tiles(const RotSide& r, int M, int BN) {
  return static_cast<long long>((M + 127) / 128) * ((r.rows + BN - 1) / BN);
}

// Both sides of a module in one launch: when their tiles are at most two per SM,
// where a launch of its own leaves most SMs idle for a whole tile.
bool rotate_in_one(const RotSide& ra, const RotSide& rs, int M, int num_sms) {
  return rot_tiles(ra, M, rotate_bn(ra.rows, 16)) + rot_tiles(rs, M, rotate_bn(rs.rows, 16)) <= 2ll * num_sms;
}

// Five queries of 512 tokens through 768 -> 2304 take 11.6 us in one launch, 13.0 +
// 10.6 in two.
cudaError_t launch_tc_rotate_both(const RotSide& ra, const RotSide& rs, int M, int T, int num_sms, unsigned* status,
                                  cudaStream_t st) {
  if (M <= 0) return cudaSuccess;
  const bool swap = rs.K > ra.K;  // the longer reduction first
  const RotSide r[2] = {swap ? rs : ra, swap ? ra : rs};
  int bn[2];
  rotate_both_widths({r[0].rows, r[1].rows}, {r[0].K, r[1].K}, M, std::max(1, num_sms), bn);
  return launch_rot(r, 2, M, T, bn, num_sms, status, st);
}

int tc_gemm_splits_used(int K, int splits) {
  const int nkb = (K + 63) / 64;
  splits = max(1, min(splits, nkb));
  const int kbps = (nkb + splits - 1) / splits;
  return (nkb + kbps - 1) / kbps;
}

cudaError_t launch_tc_contract(const void* St_hi, const void* St_lo, int ldS, const void* At_hi,
                               const void* At_lo, int ldA, int B, int T, const eogp_plan* plan,
                               float* z, int ldz, void* zhi, void* zlo, int ldzb, int stages,
                               int num_sms, unsigned* status, cudaStream_t st) {
  if (B <= 0 || plan->n_tiles() == 0) return cudaSuccess;
  CUtensorMap tSh, tSl, tAh, tAl;
  const uint64_t nS = static_cast<uint64_t>(B) * (ldS / 128), nA = static_cast<uint64_t>(B) * (ldA / 128);
  if (tmap_chunked(&tSh, St_hi, T, nS) || tmap_chunked(&tSl, St_lo, T, nS) ||
      tmap_chunked(&tAh, At_hi, T, nA) || tmap_chunked(&tAl, At_lo, T, nA))
    return cudaErrorInvalidValue;
  ContractArgs g;
  g.T = T;
  g.nblkS = ldS / 128;
  g.nblkA = ldA / 128;
  g.stages = stages;
  g.n_tiles = plan->n_tiles();
  g.n_items = g.n_tiles * B;
  g.tile_rc = plan->d_tile_rc;
  g.grp_start = plan->d_grp_start;
  g.ent = reinterpret_cast<const int4*>(plan->d_ent);
  g.z = z;
  g.ldz = ldz;
  g.zhi = static_cast<__nv_bfloat16*>(zhi);
  g.zlo = static_cast<__nv_bfloat16*>(zlo);
  g.ldzb = ldzb;
  g.status = status;
  const size_t smem = contract_smem_bytes(stages);
  cudaError_t e = allow_smem(k_tc_contract);
  if (e != cudaSuccess) return e;
  const int grid = std::min(g.n_items, std::max(1, num_sms));
  return launch_behind(k_tc_contract, grid, kThreads, smem, st, tSh, tSl, tAh, tAl, g);
}

size_t ekfac_smem_bytes(int stages) {
  return 1024 + static_cast<size_t>(stages) * kCStage + (2 * stages + 4) * 8 + 16;
}

int ekfac_chunks(int B, int n_tiles, int num_sms) {
  // Enough items for about two per SM, each chunk as long as possible.
  const int want_items = 2 * std::max(1, num_sms);
  int nch = std::max(1, std::min(B, (want_items + n_tiles - 1) / n_tiles));
  const int bpc = (B + nch - 1) / nch;
  return (B + bpc - 1) / bpc;
}

// Columns of a pair's tile: the time of the busiest pair is that of its items, in
// columns per example; shorter than 96 columns a tile waits on its loads of S~.
static int ekfac2_width(int n_rt, int d_in, int chunks, int pairs, long long* cost) {
  int best = 0;
  for (int N = 256; N >= 64; N -= 64) {
    const long long items = static_cast<long long>(n_rt) * ((d_in + N - 1) / N) * chunks;
    const long long t = (items + pairs - 1) / pairs * (std::max(N, 96) + 16);
    if (!best || t < *cost) {
      best = N;
      *cost = t;
    }
  }
  return best;
}

static cudaError_t launch_ekfac2(const void* St_hi, const void* St_lo, int ldS, const void* At_hi, const void* At_lo,
                                 int ldA, int B, int T, int d_out, int d_in, float* part, int chunks, int N,
                                 int num_sms, unsigned* status, cudaStream_t st) {
  CUtensorMap tSh, tSl, tAh, tAl;
  const uint64_t nS = static_cast<uint64_t>(B) * (ldS / 128), nA = static_cast<uint64_t>(B) * (ldA / 128);
  if (tmap_chunked(&tSh, St_hi, T, nS) || tmap_chunked(&tSl, St_lo, T, nS) ||
      tmap_chunked(&tAh, At_hi, T, nA, N / 16) || tmap_chunked(&tAl, At_lo, T, nA, N / 16))
    return cudaErrorInvalidValue;
  Ekfac2Args g;
  g.nkb = (T + 63) / 64;
  g.N = N;
  g.n_ct = (d_in + N - 1) / N;
  g.n_tiles = (d_out + 255) / 256 * g.n_ct;
  g.n_items = g.n_tiles * chunks;
  g.bpc = (B + chunks - 1) / chunks;
  g.B = B;
  g.chS = ldS / 8;
  g.chA = ldA / 8;
  g.d_out = d_out;
  g.d_in = d_in;
  g.part = part;
  g.status = status;
  const size_t stage = 2 * kOpBytes + 128 * static_cast<size_t>(N);
  const auto bytes = [&](int stages) { return 1024 + stages * stage + (2 * stages + 4) * 8 + 16; };
  g.stages = 2;
  while (bytes(g.stages + 1) <= 232448) ++g.stages;
  const size_t smem = bytes(g.stages);
  const cudaError_t e = allow_smem(k_tc_ekfac2);
  if (e != cudaSuccess) return e;
  return launch_behind(k_tc_ekfac2, 2 * std::min(g.n_items, std::max(1, num_sms / 2)), kEk2Threads, smem, st, tSh, tSl,
                       tAh, tAl, g);
}

static cudaError_t launch_ekfac1(const void* St_hi, const void* St_lo, int ldS, const void* At_hi, const void* At_lo,
                                 int ldA, int B, int T, int d_out, int d_in, float* part, int chunks, int stages,
                                 int num_sms, unsigned* status, cudaStream_t st) {
  CUtensorMap tSh, tSl, tAh, tAl;
  const uint64_t nS = static_cast<uint64_t>(B) * (ldS / 128), nA = static_cast<uint64_t>(B) * (ldA / 128);
  if (tmap_chunked(&tSh, St_hi, T, nS) || tmap_chunked(&tSl, St_lo, T, nS) ||
      tmap_chunked(&tAh, At_hi, T, nA) || tmap_chunked(&tAl, At_lo, T, nA))
    return cudaErrorInvalidValue;
  EkfacArgs g;
  g.T = T;
  g.stages = stages;
  g.n_rt = (d_out + 127) / 128;
  g.n_ct = (d_in + 127) / 128;
  g.n_tiles = g.n_rt * g.n_ct;
  g.bpc = (B + chunks - 1) / chunks;
  g.n_items = g.n_tiles * chunks;
  g.B = B;
  g.nblkS = ldS / 128;
  g.nblkA = ldA / 128;
  g.d_out = d_out;
  g.d_in = d_in;
  g.part = part;
  g.status = status;
  const size_t smem = ekfac_smem_bytes(stages);
  cudaError_t e = allow_smem(k_tc_ekfac);
  if (e != cudaSuccess) return e;
  const int grid = std::min(g.n_items, std::max(1, num_sms));
  return launch_behind(k_tc_ekfac, grid, kThreads, smem, st, tSh, tSl, tAh, tAl, g);
}

// Pairs, unless their tiles fill the chip worse: an example of a 128 x 128 tile takes
// as long as one of 184 columns of a pair. 32 examples of 512 tokens, 3072 x 768: 187
// us in 128 x 128 tiles, 140 in 256 x 192 (two waves of pairs, as are 256 x 256: 186),
// 144 in 256 x 128 (three).
cudaError_t launch_tc_ekfac(const void* St_hi, const void* St_lo, int ldS, const void* At_hi, const void* At_lo,
                            int ldA, int B, int T, int d_out, int d_in, float* part, int n_chunks, double* sumsq,
                            int ld, int accumulate, int stages, int num_sms, unsigned* status, cudaStream_t st) {
  if (B <= 0) return cudaSuccess;
  const int bpc = (B + n_chunks - 1) / n_chunks, chunks = (B + bpc - 1) / bpc, sms = std::max(1, num_sms);
  const long long items1 = static_cast<long long>((d_out + 127) / 128) * ((d_in + 127) / 128) * chunks;
  const long long cost1 = (items1 + sms - 1) / sms * 184;
  long long cost2 = 0;
  const int N = ekfac2_width((d_out + 255) / 256, d_in, chunks, std::max(1, sms / 2), &cost2);
  cudaError_t e = cost2 <= cost1 ? launch_ekfac2(St_hi, St_lo, ldS, At_hi, At_lo, ldA, B, T, d_out, d_in, part, chunks,
                                                 N, sms, status, st)
                                 : launch_ekfac1(St_hi, St_lo, ldS, At_hi, At_lo, ldA, B, T, d_out, d_in, part, chunks,
                                                 stages, sms, status, st);
  if (e != cudaSuccess) return e;
  const dim3 grid((d_in / 4 + 63) / 64, std::min(d_out, 65535));
  return launch_behind(k_ekfac_finalize, grid, 64, 0, st, part, chunks, d_out, d_in, sumsq, ld, accumulate);
}
