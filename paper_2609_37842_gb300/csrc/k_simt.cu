// fp32 CUDA-core kernels: the EOGP_F32 path of eogp_compress_layer, the FP
// score mode, the Gram / covariance matrices of the PCA fit, and the row
// gather used to lay out retained eigenvectors.
//
//  k_simt_gemm: C[i][j] = alpha * sum_k A(i,k) B(j,k) with arbitrary element
//    strides: BM x BN tile per block, TM x TN per thread, fp32 FMAs with k
//    ascending for every element, so the tile does not show in the result. The
//    next 16 values of k travel from memory to registers while the present 16
//    are multiplied out of shared memory; a thread's TM + TN values of a k are
//    16-byte shared loads.
//  k_f32_first: the first stage of a few examples per block, when one example's
//    tokens and rotated rows fit: both rotations into shared memory, then
//    z[b][r] = scale[r] * sum_t S~[b,t][posR[r]] * A~[b,t][posC[r]]
//    (Eq. first_stage through the Kronecker identity of Sec. 2.2). 4096 examples of
//    16 tokens, 64 -> 64: 50 us, against 87 us for three kernels that pass the
//    rotated rows through memory; bound by instruction issue (14.5 us of it are
//    the FMAs themselves).
//  k_contract_f32: the same sum from rotated rows in memory, for larger modules:
//    one thread per (example, retained coordinate r).
#include <algorithm>

#include "eogp_dev.cuh"
#include "eogp_internal.h"

namespace {

constexpr int kKT = 16;  // k per shared-memory tile

// One operand of a tile: rows of X (X(r, k) = X[r sr + k sk], zero outside rows x K).
struct Operand {
  const float* x;
  long long sr, sk;
  int rows;
};

// How an operand is read: four k of a row at a time, or four rows of a k, as one
// aligned 16-byte load (a group is inside or outside as a whole), or value by
// value. Fixed at compile time: with the choice at run time the values meet in
// registers behind the branch, so a load is waited for where it is issued and
// nothing is prefetched.
enum { kAny, kAlongK, kAlongRows };

// A tile's 16 k of R rows, R * 4 groups of four values dealt to NT threads, in
// two steps: memory -> registers, registers -> shared memory t[k][row].
template <int R, int NT, int L>
struct TileLoad {
  static constexpr int kPer = (R * 4 + NT - 1) / NT;
  float4 v[kPer];
  __device__ __forceinline__ void load(const Operand& o, int r0, int k0, int K, int tid) {
#pragma unroll
    for (int p = 0; p < kPer; ++p) {
      const int e = tid + p * NT;
      const bool in = R * 4 % NT == 0 || e < R * 4;
      v[p] = make_float4(0.f, 0.f, 0.f, 0.f);
      if constexpr (L == kAlongRows) {
        const int r = r0 + 4 * (e % (R / 4)), k = k0 + e / (R / 4);
        if (in && k < K && r < o.rows) v[p] = *reinterpret_cast<const float4*>(o.x + r + k * o.sk);
      } else {
        const int r = r0 + (e >> 2), k = k0 + 4 * (e & 3);
        const float* src = o.x + r * o.sr + k * o.sk;
        if constexpr (L == kAlongK) {
          if (in && r < o.rows && k < K) v[p] = *reinterpret_cast<const float4*>(src);
        } else if (in && r < o.rows) {
          if (k < K) v[p].x = src[0];
          if (k + 1 < K) v[p].y = src[o.sk];
          if (k + 2 < K) v[p].z = src[2 * o.sk];
          if (k + 3 < K) v[p].w = src[3 * o.sk];
        }
      }
    }
  }
  __device__ __forceinline__ void store(float (*t)[R + 4], int tid) const {
#pragma unroll
    for (int p = 0; p < kPer; ++p) {
      const int e = tid + p * NT;
      if (R * 4 % NT != 0 && e >= R * 4) continue;
      if constexpr (L == kAlongRows) {
        *reinterpret_cast<float4*>(&t[e / (R / 4)][4 * (e % (R / 4))]) = v[p];
      } else {
        const int r = e >> 2, k = 4 * (e & 3);
        t[k][r] = v[p].x;
        t[k + 1][r] = v[p].y;
        t[k + 2][r] = v[p].z;
        t[k + 3][r] = v[p].w;
      }
    }
  }
};

// Row (or column) of fragment value x of thread t: groups of four (or two, for
// fragments of two) dealt round-robin, so a warp's 16-byte loads are spread.
template <int T, int NTH>
__device__ __forceinline__ int frag_pos(int t, int x) {
  constexpr int g = T < 4 ? T : 4;
  return (x / g) * (g * NTH) + t * g + x % g;
}
template <int T, int NTH>
__device__ __forceinline__ void frag_load(const float* row, int t, float (&f)[T]) {
  if constexpr (T < 4) {
    const float2 v = *reinterpret_cast<const float2*>(row + 2 * t);
    f[0] = v.x, f[1] = v.y;
  } else {
#pragma unroll
    for (int x = 0; x < T; x += 4) {
      const float4 v = *reinterpret_cast<const float4*>(row + frag_pos<T, NTH>(t, x));
      f[x] = v.x, f[x + 1] = v.y, f[x + 2] = v.z, f[x + 3] = v.w;
    }
  }
}

template <int BM, int BN>
struct alignas(16) GemmTiles {
  float a[2][kKT][BM + 4];
  float b[2][kKT][BN + 4];
};

// acc[x][y] = sum_k A(i0 + i, k) B(j0 + j, k), k ascending, of this thread's rows i
// and columns j of the tile, with PD tiles of k on their way from memory in
// registers (a tile's multiplications take a fraction of the L2 latency: the 256 x
// 128 x 512 projection takes 11.5 us with four tiles in flight, 17.3 with one). The
// block's threads all call it; the shared tiles are free for the next call after a
// barrier.
template <int BM, int BN, int TM, int TN, int PD, int L>
__device__ __forceinline__ void tile_gemm(GemmTiles<BM, BN>& sm, const Operand& A, const Operand& B, int i0, int j0,
                                          int K, float (&acc)[TM][TN]) {
  constexpr int NX = BN / TN, NY = BM / TM, NT = NX * NY;
  const int tid = threadIdx.x, tx = tid % NX, ty = tid / NX;
#pragma unroll
  for (int x = 0; x < TM; ++x)
#pragma unroll
    for (int y = 0; y < TN; ++y) acc[x][y] = 0.f;
  TileLoad<BM, NT, L> la[PD];
  TileLoad<BN, NT, L> lb[PD];
#pragma unroll
  for (int u = 0; u < PD; ++u)
    if (u * kKT < K) {
      la[u].load(A, i0, u * kKT, K, tid);
      lb[u].load(B, j0, u * kKT, K, tid);
    }
  int buf = 0;
  for (int kb = 0; kb < K; kb += PD * kKT) {
#pragma unroll
    for (int u = 0; u < PD; ++u) {
      const int k0 = kb + u * kKT;
      if (k0 >= K) break;
      la[u].store(sm.a[buf], tid);
      lb[u].store(sm.b[buf], tid);
      __syncthreads();  // also: every thread is done with the other buffer
      if (k0 + PD * kKT < K) {
        la[u].load(A, i0, k0 + PD * kKT, K, tid);
        lb[u].load(B, j0, k0 + PD * kKT, K, tid);
      }
      // the fragments of k + 1 are read while those of k are multiplied
      float a[2][TM], b[2][TN];
      frag_load<TM, NY>(sm.a[buf][0], ty, a[0]);
      frag_load<TN, NX>(sm.b[buf][0], tx, b[0]);
#pragma unroll
      for (int kk = 0; kk < kKT; ++kk) {
        if (kk + 1 < kKT) {
          frag_load<TM, NY>(sm.a[buf][kk + 1], ty, a[(kk + 1) & 1]);
          frag_load<TN, NX>(sm.b[buf][kk + 1], tx, b[(kk + 1) & 1]);
        }
#pragma unroll
        for (int x = 0; x < TM; ++x)
#pragma unroll
          for (int y = 0; y < TN; ++y) acc[x][y] = fmaf(a[kk & 1][x], b[kk & 1][y], acc[x][y]);
      }
      buf ^= 1;
    }
  }
}

// NOTED: only the entries of noted rows (one of the n_inote notes inote[b ld_inote + i])
// and noted columns (jnote[j]) are written, and only tiles with one are computed.
template <int BM, int BN, int TM, int TN, int PD, int L, bool NOTED>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
    k_simt_gemm(int M, int N, int K, float alpha, const Operand A, const Operand B, float* __restrict__ C,
                long long ldc, const int* __restrict__ inote, int n_inote, int ld_inote, const int* __restrict__ jnote) {
  constexpr int NX = BN / TN, NY = BM / TM;
  __shared__ GemmTiles<BM, BN> sm;
  __shared__ uint8_t noted[NOTED ? BM + BN : 1];  // the tile's rows, then its columns
  eogp::pdl_trigger();
  eogp::pdl_wait();
  const int i0 = blockIdx.y * BM, j0 = blockIdx.x * BN;
  if (NOTED) {
    int hit = 0;
    for (int i = threadIdx.x; i < BM && i0 + i < M; i += NX * NY) {
      int h = 0;
      for (int b = 0; b < n_inote; ++b) h |= inote[static_cast<size_t>(b) * ld_inote + i0 + i];
      noted[i] = h != 0;
      hit |= h;
    }
    for (int j = threadIdx.x; j < BN && j0 + j < N; j += NX * NY) {
      const int h = jnote[j0 + j];
      noted[BM + j] = h != 0;
      hit |= h;
    }
    if (!__syncthreads_or(hit)) return;
  }
  float acc[TM][TN];
  tile_gemm<BM, BN, TM, TN, PD, L>(sm, A, B, i0, j0, K, acc);
  const int tx = threadIdx.x % NX, ty = threadIdx.x / NX;
#pragma unroll
  for (int x = 0; x < TM; ++x) {
    const int i = i0 + frag_pos<TM, NY>(ty, x);
    if (i >= M) continue;
#pragma unroll
    for (int y = 0; y < TN; ++y) {
      const int j = j0 + frag_pos<TN, NX>(tx, y);
      if (j < N && (!NOTED || noted[i - i0] || noted[BM + j - j0])) C[i * ldc + j] = alpha * acc[x][y];
    }
  }
}

// First stage of examples [G block, G (block + 1)): tiles of BM rows (row = token
// of one of the G examples, G T <= BM) by 64 columns. The rotated rows
// lie in shared memory token-contiguous, rot[column][BM + 4], A~ then S~.
struct FirstArgs {
  int B, T, m, G, nC, nR, d_in, d_out, ldz, tvec;
  Operand VA, VS;
  const float* a;
  const float* s;
  const float* bias;
  const int32_t* lengths;
  const int32_t* posR;
  const int32_t* posC;
  const float* scale;
  float* z;
};

template <int BM>
constexpr int first_threads() {
  return BM == 64 ? 256 : 128;
}

// Place of row r of rotated column j: the four-row groups of a column are permuted
// by its index over the tile's columns, so that the 16 threads writing one group of
// 16 columns (and the lanes reading one group of columns here and there) meet
// different banks. A column of 16 rows has four groups only.
template <int BM>
__device__ __forceinline__ int rot_place(int j, int r) {
  return r ^ (((j >> 2) & (BM / 4 < 8 ? BM / 4 - 1 : 7)) << 2);
}

template <int BM, int L>
__global__ void __launch_bounds__(first_threads<BM>()) k_f32_first(const FirstArgs g) {
  constexpr int NT = first_threads<BM>(), TN = 4, NX = 16, NY = NT / NX, TM = BM / NY, P = BM + 4;
  extern __shared__ __align__(16) uint8_t smem_raw[];
  eogp::pdl_trigger();
  auto& sm = *reinterpret_cast<GemmTiles<BM, 64>*>(smem_raw);
  float* rot = reinterpret_cast<float*>(smem_raw + sizeof(GemmTiles<BM, 64>));
  const int b0 = blockIdx.x * g.G, nb = min(g.G, g.B - b0), rows = nb * g.T;
  const int tx = threadIdx.x % NX, ty = threadIdx.x / NX;
  auto rot_at = [](int j, int r) { return rot_place<BM>(j, r); };
  for (int side = 0; side < 2; ++side) {
    const int n = side ? g.nR : g.nC, d = side ? g.d_out : g.d_in;
    const Operand X{(side ? g.s : g.a) + static_cast<size_t>(b0) * g.T * d, d, 1, rows};
    float* out = rot + (side ? static_cast<size_t>(g.nC) * P : 0);
    for (int j0 = 0; j0 < n; j0 += 64) {
      float acc[TM][TN];
      __syncthreads();  // the tiles of the columns before are read
      tile_gemm<BM, 64, TM, TN, L == kAny ? 1 : BM == 64 ? 2 : 4, L>(sm, X, side ? g.VS : g.VA, 0, j0, d, acc);
#pragma unroll
      for (int y = 0; y < TN; ++y) {
        const int j = j0 + frag_pos<TN, NX>(tx, y);
        if (j >= n) continue;
        const float bias = !side && g.bias ? g.bias[j] : 0.f;
        float v[TM];
#pragma unroll
        for (int x = 0; x < TM; ++x) {
          // padding tokens contribute nothing; the bias is the component of a constant-1 channel
          const int r = frag_pos<TM, NY>(ty, x);
          const bool pad = side && g.lengths && r < rows && r % g.T >= g.lengths[b0 + r / g.T];
          v[x] = pad ? 0.f : acc[x][y];
          if (!side && g.bias) v[x] += bias;
        }
        float* col = out + static_cast<size_t>(j) * P;
        constexpr int g4 = TM < 4 ? TM : 4;
#pragma unroll
        for (int x = 0; x < TM; x += g4) {
          float* d = col + rot_at(j, frag_pos<TM, NY>(ty, x));
          if constexpr (g4 == 4)
            *reinterpret_cast<float4*>(d) = make_float4(v[x], v[x + 1], v[x + 2], v[x + 3]);
          else
            *reinterpret_cast<float2*>(d) = make_float2(v[x], v[x + 1]);
        }
      }
    }
  }
  __syncthreads();
  for (int r = threadIdx.x; r < g.m; r += NT) {
    const int pc = g.posC[r], pr = g.nC + g.posR[r];
    const float* a = rot + static_cast<size_t>(pc) * P;
    const float* s = rot + static_cast<size_t>(pr) * P;
    const int ja = pc, js = g.posR[r];
    const float sc = g.scale[r];
    for (int e = 0; e < nb; ++e) {
      const int t0 = e * g.T;
      float acc = 0.f;
      if (g.tvec) {
        for (int t = t0; t < t0 + g.T; t += 4) {
          const float4 x = *reinterpret_cast<const float4*>(s + rot_at(js, t));
          const float4 y = *reinterpret_cast<const float4*>(a + rot_at(ja, t));
          acc = fmaf(x.x, y.x, acc);
          acc = fmaf(x.y, y.y, acc);
          acc = fmaf(x.z, y.z, acc);
          acc = fmaf(x.w, y.w, acc);
        }
      } else {
        for (int t = t0; t < t0 + g.T; ++t) acc = fmaf(s[rot_at(js, t)], a[rot_at(ja, t)], acc);
      }
      g.z[static_cast<size_t>(b0 + e) * g.ldz + r] = sc * acc;
    }
  }
}

__global__ void k_contract_f32(const float* __restrict__ At, int ldA, const float* __restrict__ St,
                               int ldS, int B, int T, int m, const int32_t* __restrict__ posR,
                               const int32_t* __restrict__ posC, const float* __restrict__ scale,
                               float* __restrict__ z, int ldz) {
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (idx >= static_cast<long long>(B) * m) return;
  const int b = static_cast<int>(idx / m), r = static_cast<int>(idx % m);
  const int pr = posR[r], pc = posC[r];
  const float* s = St + static_cast<size_t>(b) * T * ldS + pr;
  const float* a = At + static_cast<size_t>(b) * T * ldA + pc;
  float acc = 0.f;
  for (int t = 0; t < T; ++t) acc = fmaf(s[static_cast<size_t>(t) * ldS], a[static_cast<size_t>(t) * ldA], acc);
  z[static_cast<size_t>(b) * ldz + r] = scale[r] * acc;
}

template <typename E>
__global__ void k_gather_rows(const E* __restrict__ src, int ld_src, const int32_t* __restrict__ idx,
                              int row_len, E* __restrict__ dst) {
  const int r = blockIdx.x;
  const E* s = src + static_cast<size_t>(idx[r]) * ld_src;
  E* d = dst + static_cast<size_t>(r) * row_len;
  for (int c = threadIdx.x; c < row_len; c += blockDim.x) d[c] = s[c];
}

}  // namespace

namespace {

bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

// How both operands of a GEMM over K can be read.
int layout_of(const Operand& a, const Operand& b, int K) {
  if (!al16(a.x) || !al16(b.x)) return kAny;
  if (a.sk == 1 && b.sk == 1 && K % 4 == 0 && a.sr % 4 == 0 && b.sr % 4 == 0) return kAlongK;
  if (a.sr == 1 && b.sr == 1 && a.rows % 4 == 0 && b.rows % 4 == 0 && a.sk % 4 == 0 && b.sk % 4 == 0) return kAlongRows;
  return kAny;
}

template <int BM, int BN, int TM, int TN, int PD, int L, bool NOTED>
cudaError_t simt_launch(int M, int N, int K, float alpha, const Operand& A, const Operand& B, float* C, long long ldc,
                        const int* inote, int n_inote, int ld_inote, const int* jnote, cudaStream_t st,
                        bool behind = false) {
  const dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM);
  if (behind)
    return launch_behind(k_simt_gemm<BM, BN, TM, TN, PD, L, NOTED>, grid, (BM / TM) * (BN / TN), 0, st, M, N, K, alpha, A,
                         B, C, ldc, inote, n_inote, ld_inote, jnote);
  k_simt_gemm<BM, BN, TM, TN, PD, L, NOTED><<<grid, (BM / TM) * (BN / TN), 0, st>>>(M, N, K, alpha, A, B, C, ldc, inote,
                                                                               n_inote, ld_inote, jnote);
  return cudaGetLastError();
}

}  // namespace

template <int BM, int BN, int TM, int TN, int PD>
static cudaError_t simt_layout(int l, int M, int N, int K, float alpha, const Operand& A, const Operand& B, float* C,
                               long long ldc, cudaStream_t st, bool behind) {
  if (l == kAlongK)
    return simt_launch<BM, BN, TM, TN, PD, kAlongK, false>(M, N, K, alpha, A, B, C, ldc, nullptr, 0, 0, nullptr, st, behind);
  if (l == kAlongRows)
    return simt_launch<BM, BN, TM, TN, PD, kAlongRows, false>(M, N, K, alpha, A, B, C, ldc, nullptr, 0, 0, nullptr, st, behind);
  return simt_launch<BM, BN, TM, TN, 1, kAny, false>(M, N, K, alpha, A, B, C, ldc, nullptr, 0, 0, nullptr, st, behind);
}

// The largest tile that still gives the SMs blocks enough; small ones shorten the
// chain of a block that has an SM to itself. Measured against one 64 x 64 tile
// without prefetch for every size: 256 x 128 x 512 (32 x 32 tiles) 40 -> 14 us a
// call, 4096 x 128 x 512 (64 x 64) 40 -> 26, 4096 x 4096 x 1024 (128 x 128) 1,192 ->
// 777 (44 TFLOP/s). 64 x 64 tiles from 100 blocks on: 4096 x 128 x 512 took 27 us
// in 32 x 32 tiles.
cudaError_t launch_simt_gemm(int M, int N, int K, float alpha, const float* A, long long sai,
                             long long sak, const float* Bm, long long sbj, long long sbk,
                             float* C, long long ldc, cudaStream_t st, bool behind) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  const Operand a{A, sai, sak, M}, b{Bm, sbj, sbk, N};
  const int l = layout_of(a, b, K);
  auto blocks = [&](int bm, int bn) { return static_cast<long long>((M + bm - 1) / bm) * ((N + bn - 1) / bn); };
  // (grid.y holds at most 65,535 tiles of rows: more rows take the largest tile)
  if (M > 65535 * 32 || (N > 64 && M > 64 && blocks(128, 128) >= 304))
    return simt_layout<128, 128, 8, 8, 2>(l, M, N, K, alpha, a, b, C, ldc, st, behind);
  if (blocks(64, 64) >= 100) return simt_layout<64, 64, 4, 4, 2>(l, M, N, K, alpha, a, b, C, ldc, st, behind);
  return simt_layout<32, 32, 4, 2, 4>(l, M, N, K, alpha, a, b, C, ldc, st, behind);
}

cudaError_t launch_simt_gemm_noted(int M, int N, int K, const float* A, long long lda, const float* Bm, long long ldb,
                                   float* C, long long ldc, const int* inote, int n_inote, int ld_inote,
                                   const int* jnote, cudaStream_t st) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  return simt_launch<64, 64, 8, 4, 1, kAny, true>(M, N, K, 1.f, Operand{A, lda, 1, M}, Operand{Bm, ldb, 1, N}, C, ldc,
                                                  inote, n_inote, ld_inote, jnote, st);
}

// Rows per block of k_f32_first (64, or 16 where that gives too few blocks), 0 when
// the module does not fit: at most 64 tokens, and the rotated rows of the block
// beside the tiles in 200 KB of shared memory.
static size_t f32_first_smem(int bm, int nC, int nR) {
  return (bm == 64 ? sizeof(GemmTiles<64, 64>) : sizeof(GemmTiles<16, 64>)) +
         static_cast<size_t>(nC + nR) * (bm + 4) * 4;
}
static int f32_first_rows(int B, int T, int nC, int nR, int num_sms) {
  if (T <= 16 && static_cast<long long>(B) * T <= 64ll * num_sms && f32_first_smem(16, nC, nR) <= 200 * 1024) return 16;
  return T <= 64 && f32_first_smem(64, nC, nR) <= 200 * 1024 ? 64 : 0;
}

template <int BM, int L>
static cudaError_t first_launch(const FirstArgs& g, size_t smem, cudaStream_t st) {
  const cudaError_t e = allow_smem(k_f32_first<BM, L>);
  if (e != cudaSuccess) return e;
  k_f32_first<BM, L><<<static_cast<unsigned>((g.B + g.G - 1) / g.G), first_threads<BM>(), smem, st>>>(g);
  return cudaGetLastError();
}

bool f32_first_supported(int B, int T, int nC, int nR, int num_sms) { return f32_first_rows(B, T, nC, nR, num_sms) > 0; }

cudaError_t launch_f32_first(const float* a, const float* s, const float* VA, const float* VS, int d_in, int d_out,
                             const float* bias, const int32_t* lengths, int B, int T, int m, int nC, int nR,
                             const int32_t* posR, const int32_t* posC, const float* scale, float* z, int ldz,
                             int num_sms, cudaStream_t st) {
  const int bm = f32_first_rows(B, T, nC, nR, num_sms);
  if (!bm) return cudaErrorInvalidValue;
  FirstArgs g;
  g.B = B;
  g.T = T;
  g.m = m;
  g.G = bm / T;
  g.nC = nC;
  g.nR = nR;
  g.d_in = d_in;
  g.d_out = d_out;
  g.ldz = ldz;
  g.tvec = T % 4 == 0;
  g.VA = Operand{VA, d_in, 1, nC};
  g.VS = Operand{VS, d_out, 1, nR};
  g.a = a;
  g.s = s;
  g.bias = bias;
  g.lengths = lengths;
  g.posR = posR;
  g.posC = posC;
  g.scale = scale;
  g.z = z;
  // every row of the four operands starts on 16 bytes when the row lengths and bases do
  const bool vec = d_in % 4 == 0 && d_out % 4 == 0 && al16(a) && al16(s) && al16(VA) && al16(VS);
  const size_t smem = f32_first_smem(bm, nC, nR);
  if (bm == 64) return vec ? first_launch<64, kAlongK>(g, smem, st) : first_launch<64, kAny>(g, smem, st);
  return vec ? first_launch<16, kAlongK>(g, smem, st) : first_launch<16, kAny>(g, smem, st);
}

cudaError_t launch_contract_f32(const float* At, int ldA, const float* St, int ldS, int B, int T,
                                int m, const int32_t* posR, const int32_t* posC,
                                const float* scale, float* z, int ldz, cudaStream_t st) {
  const long long n = static_cast<long long>(B) * m;
  if (n <= 0) return cudaSuccess;
  k_contract_f32<<<static_cast<unsigned>((n + 255) / 256), 256, 0, st>>>(At, ldA, St, ldS, B, T, m,
                                                                        posR, posC, scale, z, ldz);
  return cudaGetLastError();
}

cudaError_t launch_gather_rows(const void* src, int ld_src, int elem_bytes, const int32_t* idx,
                               int n_rows, int row_len, void* dst, cudaStream_t st) {
  if (n_rows <= 0) return cudaSuccess;
  if (elem_bytes == 4)
    k_gather_rows<uint32_t><<<n_rows, 256, 0, st>>>(static_cast<const uint32_t*>(src), ld_src, idx,
                                                    row_len, static_cast<uint32_t*>(dst));
  else
    k_gather_rows<uint16_t><<<n_rows, 256, 0, st>>>(static_cast<const uint16_t*>(src), ld_src, idx,
                                                    row_len, static_cast<uint16_t*>(dst));
  return cudaGetLastError();
}

namespace {
// sumsq[j * ld + i] = (accumulate ? sumsq : 0) + G[j][i]^2 in fp64 (G dense [rows][cols]).
__global__ void k_sq_accum(const float* __restrict__ G, int rows, int cols, double* __restrict__ sumsq,
                           int ld, int accumulate) {
  const long long n = static_cast<long long>(rows) * cols;
  for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < n;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    const double g = static_cast<double>(G[e]);
    const size_t o = static_cast<size_t>(e / cols) * ld + e % cols;
    sumsq[o] = accumulate ? sumsq[o] + g * g : g * g;
  }
}
}  // namespace

cudaError_t launch_sq_accum(const float* G, int rows, int cols, double* sumsq, int ld, int accumulate,
                            cudaStream_t st) {
  const long long n = static_cast<long long>(rows) * cols;
  if (n <= 0) return cudaSuccess;
  const unsigned blocks = static_cast<unsigned>(std::min<long long>((n + 255) / 256, 4096));
  k_sq_accum<<<blocks, 256, 0, st>>>(G, rows, cols, sumsq, ld, accumulate);
  return cudaGetLastError();
}

namespace {
// Row fix-ups of a rotated token matrix X [M x n] (row = b * T + t): add the
// bias-channel term bias[c], or zero the rows of tokens t >= lengths[b].
__global__ void k_rows_fixup(float* __restrict__ X, int M, int n, int ld, int T, const float* __restrict__ bias,
                             const int32_t* __restrict__ lengths) {
  const long long tot = static_cast<long long>(M) * n;
  for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < tot;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int row = static_cast<int>(e / n), c = static_cast<int>(e % n);
    float* p = X + static_cast<size_t>(row) * ld + c;
    if (lengths && row % T >= lengths[row / T]) {
      *p = 0.f;
    } else if (bias) {
      *p += bias[c];
    }
  }
}
}  // namespace

cudaError_t launch_rows_fixup(float* X, int M, int n, int ld, int T, const float* bias,
                              const int32_t* lengths, cudaStream_t st) {
  const long long tot = static_cast<long long>(M) * n;
  if (tot <= 0 || (!bias && !lengths)) return cudaSuccess;
  const unsigned blocks = static_cast<unsigned>(std::min<long long>((tot + 255) / 256, 8192));
  k_rows_fixup<<<blocks, 256, 0, st>>>(X, M, n, ld, T, bias, lengths);
  return cudaGetLastError();
}
