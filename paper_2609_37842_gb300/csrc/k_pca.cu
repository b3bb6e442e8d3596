// PCA fit of the second stage (App. B.2 "PCA fitting"; Alg. 1 "fit P_u by
// uncentered PCA of {z_iu}"): the top-k eigenvectors of Z^T Z / n, obtained
// from the n x n Gram matrix Z Z^T / n when n < m (the route the paper
// describes). Everything runs on the device. Two solvers, by size
// (nn = min(n, m)):
//
// Dense (nn <= 1024, or k close to nn): every eigenpair of the nn x nn matrix.
//  1. A = Z^T Z / n (or Z Z^T): CUDA-core GEMM on the fp32 Z with fp64
//     accumulation.
//  2. Cyclic two-sided Jacobi (Golub & Van Loan, Sec. 8.5) in round-robin
//     ("circle") order: each step rotates nn'/2 disjoint (p, q) pairs, J^T A J and
//     J^T V^T, in double; a sweep of steps is one kernel (k_jacobi_sweep). Sweeps
//     repeat until the off-diagonal mass stops shrinking or falls below 1e-11 of
//     ||A||_F; A and V^T are kept in fp64.
//  3. Rank the eigenvalues (descending, ties to the lower index), keep the top
//     k, map Gram-route vectors through Z^T u / ||Z^T u||, normalise, and fix
//     each vector's sign so its largest-magnitude entry is positive.
//
// Subspace iteration (larger problems): only the top k eigenpairs.
//  1. A = Z^T Z / n (or Z Z^T / n) on the tensor cores: Z as a bf16 hi/lo pair
//     (about 16 significant bits), three MMAs per step (hi hi, hi lo, lo hi),
//     fp32 accumulation; A is symmetrised and kept as a hi/lo pair.
//  2. Block power iteration on p = k + max(64, k / 4) (rounded up to 32)
//     vectors, kept as rows of X^T: Y = A X on the tensor cores, then X =
//     orthonormal basis of Y by three Cholesky-QR passes (rows normalised,
//     Gram Y^T Y on the tensor cores, Cholesky of the Gram plus a shift of
//     1e-2 / 1e-4 / 0 of its mean diagonal in fp32, X = Y L^-T): the shifts keep
//     the factorisation defined when the columns of A X are nearly dependent.
//  3. Every 5 iterations a Rayleigh-Ritz step: H = X^T A X (p x p), its
//     eigenpairs by the Jacobi solver above in fp64, X and A X rotated onto the
//     Ritz vectors (ordered by Ritz value, descending). The iteration stops
//     when every one of the top k Ritz pairs has ||A x - theta x|| <= 1e-3 theta.
//  4. The top k Ritz vectors (mapped through Z^T u on the Gram route) are
//     normalised and signed as in the dense solver; eig = the Ritz values.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "eogp_dev.cuh"
#include "eogp_internal.h"

namespace {

__device__ __forceinline__ void jac_pair(int s, int kidx, int np, int& p, int& q) {
  const int L = np - 1;
  if (kidx == 0) {
    p = s;
    q = L;
  } else {
    p = (s + kidx) % L;
    q = (s - kidx + L) % L;
  }
  if (p > q) {
    const int t = p;
    p = q;
    q = t;
  }
}

// C[i][j] = alpha * sum_k A(i,k) B(j,k) with A(i,k) = A[i*sai + k*sak] (fp32 in,
// fp64 accumulate and out). 32 x 32 tile per block, 2 x 2 per thread.
template <typename TA>
__global__ void __launch_bounds__(256) k_gemm_f64acc(int M, int N, int K, double alpha, int accumulate,
                                                     const TA* __restrict__ A, long long sai,
                                                     long long sak, const float* __restrict__ B,
                                                     long long sbj, long long sbk,
                                                     double* __restrict__ C, long long ldc) {
  __shared__ double As[16][33];
  __shared__ double Bs[16][33];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int i0 = blockIdx.y * 32, j0 = blockIdx.x * 32;
  double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
  for (int k0 = 0; k0 < K; k0 += 16) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int e = tid + 256 * r;
      int ii, kk;
      if (sak == 1) { ii = e >> 4; kk = e & 15; } else { kk = e >> 5; ii = e & 31; }
      double v = 0.0;
      if (i0 + ii < M && k0 + kk < K) v = static_cast<double>(A[(i0 + ii) * sai + (k0 + kk) * sak]);
      As[kk][ii] = v;
      int jj, kb;
      if (sbk == 1) { jj = e >> 4; kb = e & 15; } else { kb = e >> 5; jj = e & 31; }
      double w = 0.0;
      if (j0 + jj < N && k0 + kb < K) w = static_cast<double>(B[(j0 + jj) * sbj + (k0 + kb) * sbk]);
      Bs[kb][jj] = w;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      const double a0 = As[kk][ty], a1 = As[kk][ty + 16];
      const double b0 = Bs[kk][tx], b1 = Bs[kk][tx + 16];
      acc[0][0] = fma(a0, b0, acc[0][0]);
      acc[0][1] = fma(a0, b1, acc[0][1]);
      acc[1][0] = fma(a1, b0, acc[1][0]);
      acc[1][1] = fma(a1, b1, acc[1][1]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int i = i0 + ty + 16 * x;
    if (i >= M) continue;
#pragma unroll
    for (int y = 0; y < 2; ++y) {
      const int j = j0 + tx + 16 * y;
      if (j < N) C[i * ldc + j] = accumulate ? C[i * ldc + j] + alpha * acc[x][y] : alpha * acc[x][y];
    }
  }
}

template <typename TA>
cudaError_t gemm_f64acc(int M, int N, int K, double alpha, const TA* A, long long sai, long long sak,
                        const float* B, long long sbj, long long sbk, double* C, long long ldc,
                        cudaStream_t st, int accumulate = 0) {
  dim3 grid((N + 31) / 32, (M + 31) / 32);
  k_gemm_f64acc<TA><<<grid, 256, 0, st>>>(M, N, K, alpha, accumulate, A, sai, sak, B, sbj, sbk, C, ldc);
  return cudaGetLastError();
}

// A[i][j] = scale * C[i][j] (dense n x n copy of a strided fp64 matrix)
__global__ void k_scale_copy(const double* __restrict__ C, int ldc, int n, double scale, double* __restrict__ A) {
  const long long tot = static_cast<long long>(n) * n;
  for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < tot;
       e += static_cast<long long>(gridDim.x) * blockDim.x)
    A[e] = scale * C[(e / n) * ldc + e % n];
}

__global__ void k_eye(double* V, int n) {
  const long long idx = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (idx >= static_cast<long long>(n) * n) return;
  V[idx] = (idx / n == idx % n) ? 1.0 : 0.0;
}

// The pair of element x at step s (inverse of jac_pair).
__device__ __forceinline__ int jac_index(int s, int x, int np) {
  const int L = np - 1;
  if (x == L || x == s) return 0;
  const int d = x > s ? x - s : x - s + L;
  return d < np / 2 ? d : L - d;
}

// (x, y) <- (c x - s y, s x + c y). r = (c, s), or LIFT: r = (tan(angle / 2), s) and
// the rotation as three shears, three operations instead of four.
template <bool LIFT>
__device__ __forceinline__ void jac_rotate(double2 r, double& x, double& y) {
  if (LIFT) {
    x = __fma_rn(-r.x, y, x);
    y = __fma_rn(r.y, x, y);
    x = __fma_rn(-r.x, y, x);
  } else {
    const double a = x, b = y;
    x = r.x * a - r.y * b;
    y = r.y * a + r.x * b;
  }
}

// Entry (x, y) after step s, formed from A before it and the step's rotations:
// rows x and its partner rotated, then columns y and its partner. The index without a
// partner (odd n) has no rotation of its own; its row takes the column rotations and
// its column the row rotations, like any other. Loads and arithmetic apart, so that
// the loads of several entries are in flight together.
template <bool LIFT>
struct JacEntry {
  double a, b, c, d;  // rows (x's pair) by columns (y's pair)
  double2 ck, cj;
  bool low_row, low_col, row_alone, col_alone, zero;
  __device__ __forceinline__ void load(const double* __restrict__ A, int n, int np, int s,
                                       const double2* __restrict__ cs, int x, int y) {
    const int k = jac_index(s, x, np), j = jac_index(s, y, np);
    int p, q, pj, qj;
    jac_pair(s, k, np, p, q);
    jac_pair(s, j, np, pj, qj);
    row_alone = q >= n;
    col_alone = qj >= n;
    low_row = x == p;
    low_col = y == pj;
    zero = k == j && x != y;
    const double* Ap = A + static_cast<size_t>(p) * n;
    const double* Aq = A + static_cast<size_t>(row_alone ? p : q) * n;
    const int qc = col_alone ? pj : qj;
    ck = __ldcg(cs + k);
    cj = __ldcg(cs + j);
    a = __ldcg(Ap + pj);
    b = __ldcg(Ap + qc);
    c = __ldcg(Aq + pj);
    d = __ldcg(Aq + qc);
  }
  __device__ __forceinline__ double value() {
    if (LIFT) {  // no row is alone
      const double l = rotated(ck, low_row, a, c), h = rotated(ck, low_row, b, d);
      if (zero && ck.y != 0.0) return 0.0;  // the annihilated pair
      return rotated(cj, low_col, l, h);
    }
    if (row_alone) {
      if (!col_alone) jac_rotate<LIFT>(cj, a, b);
      return low_col ? a : b;
    }
    jac_rotate<LIFT>(ck, a, c);
    if (col_alone) return low_row ? a : c;
    jac_rotate<LIFT>(ck, b, d);
    jac_rotate<LIFT>(cj, a, b);
    jac_rotate<LIFT>(cj, c, d);
    if (zero && ck.y != 0.0) return 0.0;  // the annihilated pair
    return low_row ? (low_col ? a : b) : (low_col ? c : d);
  }
  static __device__ __forceinline__ double rotated(double2 r, bool low, double x, double y) {
    jac_rotate<true>(r, x, y);
    return low ? x : y;
  }
};

// The rotation that annihilates apq.
template <bool LIFT>
__device__ double2 jac_params(double app, double aqq, double apq) {
  double c = 1.0, sn = 0.0;
  if (apq != 0.0) {
    const double tau = (aqq - app) / (2.0 * apq);
    double t;
    if (fabs(tau) > 1e150) {
      t = 0.5 / tau;
    } else {
      t = (tau >= 0.0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
    }
    const double r = sqrt(1.0 + t * t);
    c = 1.0 / r;
    sn = t * c;
    if (LIFT) return make_double2(t / (1.0 + r), sn);
  }
  return make_double2(LIFT ? 0.0 : c, sn);
}

// All blocks of the grid (a cooperative launch) wait until every one has arrived;
// `count` rises by gridDim.x per barrier. Bounded: false after ~2 s, and the
// status word says so.
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned target, unsigned* status) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(count, 1u);
    const long long t0 = clock64();
    unsigned v;
    ok = 1;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
      if (static_cast<int>(v - target) < 0 && clock64() - t0 > EOGP_WAIT_CYCLES) {
        eogp::flag_status(status, EOGP_ST_TIMEOUT);
        ok = 0;
        break;
      }
    } while (static_cast<int>(v - target) < 0);
    __threadfence();
  }
  __syncthreads();
  return ok != 0;
}

// One sweep: np - 1 steps, one grid-wide barrier each. A step reads A from one
// buffer and writes the other, so everything in it is independent given its
// rotations: the 2 x 2 blocks of A (pair k's rows by pair j's columns, a thread
// each), the rows of V^T, and the rotations of the next step, whose three entries of
// the new A are formed again from the old one rather than waited for. Bound by the
// fp64 rate and the barrier (1.4 us). Even sizes rotate by three shears (LIFT), 12
// fp64 operations on a block of A instead of 16. At n = 640: 6.6 us a step; 7.3 with
// 512 threads and ten blocks for the rotations, 8.5 also with four operations a
// rotation, 16.4 with two kernels a step (rotations, then whole rows in shared
// memory). Longer tasks than 32 blocks of A or 64 columns of V^T cost 8 % (the last
// ones run alone). Odd sizes keep the plain form.
constexpr int kJacThreads = 768;

template <bool LIFT>
__global__ void __launch_bounds__(kJacThreads, 1)
    k_jacobi_sweep(double* __restrict__ A0, double* __restrict__ A1, double* __restrict__ Vt, int n, int np,
                   double2* __restrict__ cs0, double2* __restrict__ cs1, unsigned* count, unsigned* status) {
  __shared__ int s_task;
  const int h = np / 2, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int kWarps = kJacThreads / 32;
  unsigned target = gridDim.x;
  for (int k = blockIdx.x + gridDim.x * threadIdx.x; k < h; k += gridDim.x * kJacThreads) {
    int p, q;
    jac_pair(0, k, np, p, q);
    double2 r = make_double2(LIFT ? 0.0 : 1.0, 0.0);
    if (q < n)
      r = jac_params<LIFT>(__ldcg(A0 + static_cast<size_t>(p) * n + p), __ldcg(A0 + static_cast<size_t>(q) * n + q),
                           __ldcg(A0 + static_cast<size_t>(p) * n + q));
    __stcg(cs0 + k, r);
  }
  if (threadIdx.x == 0) s_task = 0;
  if (!grid_barrier(count, target, status)) return;
  const int jc = (h + 31) / 32;           // warp tasks of a pair's rows of A
  const int xc = (n + 63) / 64;           // and of V^T, two columns a lane
  const int nA = h * jc, nAll = nA + h * xc;
  const int pb = max(1, min((h + 63) / 64, static_cast<int>(gridDim.x) / 8));  // blocks for the rotations: two warps each
  for (int s = 0; s < np - 1; ++s) {
    const double* A = s & 1 ? A1 : A0;
    double* B = s & 1 ? A0 : A1;
    const double2* cs = s & 1 ? cs1 : cs0;
    double2* csn = s & 1 ? cs0 : cs1;
    // The next step's rotations, a lane each: a long chain of divisions and roots
    // that would wait for its turn at the fp64 unit behind every other warp of its
    // SM, so the first blocks do nothing else.
    if (blockIdx.x < pb) {
      if (s + 1 < np - 1)
        for (int k = 32 * (blockIdx.x + pb * warp) + lane; k < h; k += 32 * pb * kWarps) {
          int p, q;
          jac_pair(s + 1, k, np, p, q);
          double2 r = make_double2(LIFT ? 0.0 : 1.0, 0.0);
          if (q < n) {
            JacEntry<LIFT> pp, qq, pq;
            pp.load(A, n, np, s, cs, p, p);
            qq.load(A, n, np, s, cs, q, q);
            pq.load(A, n, np, s, cs, p, q);
            const double app = pp.value(), aqq = qq.value();
            r = jac_params<LIFT>(app, aqq, pq.value());
          }
          __stcg(csn + k, r);
        }
    }
    // The other blocks' tasks, taken by their warps as they come free.
    while (blockIdx.x >= pb) {
      int t = 0;
      if (lane == 0) t = atomicAdd(&s_task, 1);
      t = blockIdx.x - pb + (static_cast<int>(gridDim.x) - pb) * __shfl_sync(0xffffffffu, t, 0);
      if (t >= nAll) break;
      if (t < nA) {
        const int k = t / jc, j = (t - k * jc) * 32 + lane;
        if (j >= h) continue;
        int p, q, pj, qj;
        jac_pair(s, k, np, p, q);
        jac_pair(s, j, np, pj, qj);
        const size_t rp = static_cast<size_t>(p) * n, rq = static_cast<size_t>(q) * n;
        if (!LIFT && q >= n) {  // a row without a partner: its columns' rotations only
          double a = __ldcg(A + rp + pj);
          if (qj < n) {
            double b = __ldcg(A + rp + qj);
            jac_rotate<LIFT>(__ldcg(cs + j), a, b);
            __stcg(B + rp + qj, b);
          }
          __stcg(B + rp + pj, a);
          continue;
        }
        const double2 ck = __ldcg(cs + k);
        double a = __ldcg(A + rp + pj), c = __ldcg(A + rq + pj);
        if (LIFT || qj < n) {
          const double2 cj = __ldcg(cs + j);
          double b = __ldcg(A + rp + qj), d = __ldcg(A + rq + qj);
          jac_rotate<LIFT>(ck, a, c);
          jac_rotate<LIFT>(ck, b, d);
          jac_rotate<LIFT>(cj, a, b);
          jac_rotate<LIFT>(cj, c, d);
          if (k == j && ck.y != 0.0) b = c = 0.0;  // the annihilated pair
          __stcg(B + rp + qj, b);
          __stcg(B + rq + qj, d);
        } else {
          jac_rotate<LIFT>(ck, a, c);
        }
        __stcg(B + rp + pj, a);
        __stcg(B + rq + pj, c);
      } else {
        const int k = (t - nA) / xc, x0 = ((t - nA) - k * xc) * 64 + lane;
        int p, q;
        jac_pair(s, k, np, p, q);
        if (q >= n) continue;
        const double2 ck = __ldcg(cs + k);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int x = x0 + 32 * e;
          if (x < n) {
            double* vp = Vt + static_cast<size_t>(p) * n + x;
            double* vq = Vt + static_cast<size_t>(q) * n + x;
            double a = __ldcg(vp), b = __ldcg(vq);
            jac_rotate<LIFT>(ck, a, b);
            __stcg(vp, a);
            __stcg(vq, b);
          }
        }
      }
    }
    target += gridDim.x;
    __syncthreads();
    if (threadIdx.x == 0) s_task = 0;
    if (!grid_barrier(count, target, status)) return;
  }
}

__global__ void __launch_bounds__(256) k_offnorm(const double* __restrict__ A, int n,
                                                 double* __restrict__ red) {
  __shared__ double so[256], st[256];
  double off = 0.0, tot = 0.0;
  const long long N2 = static_cast<long long>(n) * n;
  for (long long idx = blockIdx.x * 256LL + threadIdx.x; idx < N2; idx += 256LL * gridDim.x) {
    const double v = A[idx];
    tot += v * v;
    if (idx / n != idx % n) off += v * v;
  }
  so[threadIdx.x] = off;
  st[threadIdx.x] = tot;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      so[threadIdx.x] += so[threadIdx.x + w];
      st[threadIdx.x] += st[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    atomicAdd(&red[0], so[0]);
    atomicAdd(&red[1], st[0]);
  }
}

// Order of a double as an integer: larger value, larger key; -0 and +0 equal, NaN below
// every number.
__device__ __forceinline__ long long order_key(double v) {
  const long long b = __double_as_longlong(v), mag = b & 0x7FFFFFFFFFFFFFFFll;
  if (mag > 0x7FF0000000000000ll) return -0x7FFFFFFFFFFFFFFFll - 1;
  return mag == 0 ? 0 : b < 0 ? b ^ 0x7FFFFFFFFFFFFFFFll : b;
}

// mu[i] = A[i][i]; sel[rank(i)] = i for the k largest (descending, ties to lower index:
// the ranks are a permutation whatever A holds). Integer keys: comparisons of doubles
// share the few 64-bit lanes of an SM.
__global__ void k_rank(const double* __restrict__ A, int n, int k, double* __restrict__ mu,
                       int* __restrict__ sel) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double vi = A[static_cast<size_t>(i) * n + i];
  mu[i] = vi;
  const long long ki = order_key(vi);
  int rank = 0;
  for (int j = 0; j < n; ++j) {
    const long long kj = order_key(A[static_cast<size_t>(j) * n + j]);
    rank += kj > ki || (kj == ki && j < i);
  }
  if (rank < k) sel[rank] = i;
}

// Pt row r = sign * src row (sel ? sel[r] : r) / ||row||, sign making the
// largest-magnitude entry (lowest index on ties) positive; eig[r] = mu[sel[r]] * eig_scale.
template <typename TS>
__global__ void __launch_bounds__(256) k_emit(const TS* __restrict__ src, int ld_src,
                                              const int* __restrict__ sel, int m,
                                              void* __restrict__ Pt, int ld_pt, int bf16_out,
                                              const double* __restrict__ mu, double eig_scale,
                                              float* __restrict__ eig) {
  __shared__ double s_ss[256];
  __shared__ double s_mx[256];
  __shared__ int s_ix[256];
  const int r = blockIdx.x;
  const TS* v = src + static_cast<size_t>(sel ? sel[r] : r) * ld_src;
  double ss = 0.0, mx = -1.0;
  int ix = 0;  // also the place read for a row without a number
  for (int c = threadIdx.x; c < m; c += blockDim.x) {
    const double x = static_cast<double>(v[c]);
    ss = fma(x, x, ss);
    const double a = fabs(x);
    if (a > mx) {
      mx = a;
      ix = c;
    }
  }
  s_ss[threadIdx.x] = ss;
  s_mx[threadIdx.x] = mx;
  s_ix[threadIdx.x] = ix;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) {
      s_ss[threadIdx.x] += s_ss[threadIdx.x + w];
      const double om = s_mx[threadIdx.x + w];
      const int oi = s_ix[threadIdx.x + w];
      if (om > s_mx[threadIdx.x] || (om == s_mx[threadIdx.x] && oi < s_ix[threadIdx.x])) {
        s_mx[threadIdx.x] = om;
        s_ix[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  const double nrm = sqrt(s_ss[0]);
  const double sgn = static_cast<double>(v[s_ix[0]]) < 0.0 ? -1.0 : 1.0;
  const double f = nrm > 0.0 ? sgn / nrm : 0.0;
  for (int c = threadIdx.x; c < m; c += blockDim.x) {
    const float o = static_cast<float>(static_cast<double>(v[c]) * f);
    if (bf16_out)
      static_cast<__nv_bfloat16*>(Pt)[static_cast<size_t>(r) * ld_pt + c] = __float2bfloat16_rn(o);
    else
      static_cast<float*>(Pt)[static_cast<size_t>(r) * ld_pt + c] = o;
  }
  if (threadIdx.x == 0 && eig) eig[r] = static_cast<float>(mu[sel ? sel[r] : r] * eig_scale);
}

__global__ void k_gather_f64_rows(const double* __restrict__ src, int ld, const int* __restrict__ sel,
                                  int len, double* __restrict__ dst) {
  const int r = blockIdx.x;
  for (int c = threadIdx.x; c < len; c += blockDim.x)
    dst[static_cast<size_t>(r) * len + c] = src[static_cast<size_t>(sel[r]) * ld + c];
}

__global__ void k_eig_out(const double* __restrict__ mu, const int* __restrict__ sel, int k,
                          double scale, float* __restrict__ eig) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < k) eig[r] = static_cast<float>(mu[sel[r]] * scale);
}

size_t al256(size_t x) { return (x + 255) & ~size_t(255); }
inline int rup(int x, int a) { return (x + a - 1) / a * a; }

// ------------------------------------------------ subspace-iteration kernels
using bf16 = __nv_bfloat16;

__device__ __forceinline__ void split2(float v, bf16& h, bf16& l) {
  h = __float2bfloat16_rn(v);
  l = __float2bfloat16_rn(v - __bfloat162float(h));
}

// hi/lo [rows][ldd] of rscale[r] * src[r][c] for c < cols, zero in the padding.
__global__ void k_split_rows(const float* __restrict__ src, long long lds, int rows, int cols,
                             const float* __restrict__ rscale, bf16* __restrict__ hi,
                             bf16* __restrict__ lo, int ldd) {
  const long long tot = static_cast<long long>(rows) * ldd;
  for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < tot;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int r = static_cast<int>(e / ldd), c = static_cast<int>(e % ldd);
    float v = 0.f;
    if (c < cols) {
      v = src[static_cast<long long>(r) * lds + c];
      if (rscale) v *= rscale[r];
    }
    bf16 h, l;
    split2(v, h, l);
    hi[e] = h;
    lo[e] = l;
  }
}

// Transposed hi/lo [cols][ldd]: dst[c][r] = rscale[r] * src[r][c] for r < rows,
// zero for rows <= r < ldd. Grid (ceil(cols / 32), ceil(ldd / 32)), block 32 x 8.
__global__ void k_split_T(const float* __restrict__ src, long long lds, int rows, int cols,
                          const float* __restrict__ rscale, bf16* __restrict__ hi,
                          bf16* __restrict__ lo, int ldd) {
  __shared__ float t[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int j = ty; j < 32; j += 8) {
    const int r = r0 + j, c = c0 + tx;
    float v = 0.f;
    if (r < rows && c < cols) {
      v = src[static_cast<long long>(r) * lds + c];
      if (rscale) v *= rscale[r];
    }
    t[j][tx] = v;
  }
  __syncthreads();
  for (int j = ty; j < 32; j += 8) {
    const int c = c0 + j, r = r0 + tx;
    if (c < cols && r < ldd) {
      bf16 h, l;
      split2(t[tx][j], h, l);
      hi[static_cast<long long>(c) * ldd + r] = h;
      lo[static_cast<long long>(c) * ldd + r] = l;
    }
  }
}

// hi/lo [n][ldd] of (A + A^T) / 2 for a square fp32 A, zero in the padding.
// Grid (ceil(ldd / 32), ceil(n / 32)), block 32 x 8.
__global__ void k_split_sym(const float* __restrict__ A, long long lda, int n, bf16* __restrict__ hi,
                            bf16* __restrict__ lo, int ldd) {
  __shared__ float t[32][33];
  const int c0 = blockIdx.x * 32, r0 = blockIdx.y * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;
  for (int j = ty; j < 32; j += 8) {
    const int rr = c0 + j, cc = r0 + tx;  // t[j][tx] = A[c0 + j][r0 + tx]
    t[j][tx] = (rr < n && cc < n) ? A[static_cast<long long>(rr) * lda + cc] : 0.f;
  }
  __syncthreads();
  for (int j = ty; j < 32; j += 8) {
    const int r = r0 + j, c = c0 + tx;
    if (r < n && c < ldd) {
      float v = 0.f;
      if (c < n) v = 0.5f * (A[static_cast<long long>(r) * lda + c] + t[tx][j]);
      bf16 h, l;
      split2(v, h, l);
      hi[static_cast<long long>(r) * ldd + c] = h;
      lo[static_cast<long long>(r) * ldd + c] = l;
    }
  }
}

// A32[i][j] = scale * C[i][j] (fp64 second moment -> fp32)
__global__ void k_f64_to_f32(const double* __restrict__ C, long long ldc, int n, double scale,
                             float* __restrict__ A, long long lda) {
  const long long tot = static_cast<long long>(n) * n;
  for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < tot;
       e += static_cast<long long>(gridDim.x) * blockDim.x)
    A[(e / n) * lda + e % n] = static_cast<float>(scale * C[(e / n) * ldc + e % n]);
}

// rs[r] = 1 / ||src[r][0..cols)|| (0 for a zero row); one block per row.
__global__ void __launch_bounds__(256) k_row_invnorm(const float* __restrict__ src, long long lds, int cols,
                                                     float* __restrict__ rs) {
  __shared__ double red[256];
  const float* v = src + static_cast<long long>(blockIdx.x) * lds;
  double ss = 0.0;
  for (int c = threadIdx.x; c < cols; c += 256) {
    const double x = v[c];
    ss = fma(x, x, ss);
  }
  red[threadIdx.x] = ss;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) rs[blockIdx.x] = red[0] > 0.0 ? static_cast<float>(1.0 / sqrt(red[0])) : 0.f;
}

// Start vectors: standard normal entries from a counter-based generator
// (SplitMix64 of seed + element index, then the Box-Muller transform).
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}

__global__ void k_gauss(float* __restrict__ X, long long ld, int rows, int cols, unsigned long long seed) {
  const long long tot = static_cast<long long>(rows) * cols;
  for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < tot;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    const unsigned long long h = splitmix64(seed * 0x100000001B3ull + static_cast<unsigned long long>(e));
    const float u1 = (static_cast<float>(h >> 40) + 0.5f) * (1.0f / 16777216.0f);
    const float u2 = static_cast<float>((h >> 16) & 0xFFFFFFull) * (1.0f / 16777216.0f);
    X[(e / cols) * ld + e % cols] = sqrtf(-2.0f * logf(u1)) * cospif(2.0f * u2);
  }
}

__global__ void k_add_diag(float* __restrict__ A, int lda, int n, const float* __restrict__ shift) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) A[static_cast<long long>(i) * lda + i] += *shift;
}

// shift[0] = rel * (mean diagonal of A) (the Cholesky-QR shift).
__global__ void __launch_bounds__(256) k_diag_shift(const float* __restrict__ A, int lda, int n, float rel,
                                                    float* __restrict__ shift) {
  __shared__ double red[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) s += A[static_cast<long long>(i) * lda + i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) shift[0] = static_cast<float>(rel * red[0] / n);
}

// ---- blocked Cholesky (lower, in place, fp32), panels of 32 columns: the first
// diagonal block, then per panel one kernel for the rows below it and one for the
// trailing matrix, whose first block also factors the next diagonal block.

// Factors a 32 x 32 block in one warp: lane i holds row i in registers, the column
// being eliminated is passed by shuffles. Entries above the diagonal come out as 0.
__device__ __forceinline__ void chol_block(float (&a)[32], int lane, int nb, unsigned* status) {
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    if (c < nb) {
      if (lane == c) {
        float d = a[c];
        if (!(d > 0.f) || !isfinite(d)) {  // not positive definite: flag it, keep going
          eogp::flag_status(status, EOGP_ST_DEVICE);
          d = 1e-30f;
        }
        a[c] = sqrtf(d);
      }
      const float dc = __shfl_sync(0xffffffffu, a[c], c);
      if (lane > c) a[c] /= dc;
#pragma unroll
      for (int j = c + 1; j < 32; ++j) {
        const float ajc = __shfl_sync(0xffffffffu, a[c], j);
        if (j <= lane) a[j] -= a[c] * ajc;
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 32; ++j)
    if (j > lane) a[j] = 0.f;
}

__global__ void __launch_bounds__(32) k_chol_diag(float* __restrict__ A, int lda, int n, int j0, unsigned* status) {
  eogp::pdl_trigger();
  const int lane = threadIdx.x, nb = min(32, n - j0);
  float a[32];
#pragma unroll
  for (int j = 0; j < 32; ++j)
    a[j] = (lane < nb && j < nb) ? A[static_cast<long long>(j0 + lane) * lda + j0 + j] : 0.f;
  chol_block(a, lane, nb, status);
#pragma unroll
  for (int j = 0; j < 32; ++j)
    if (lane < nb && j < nb) A[static_cast<long long>(j0 + lane) * lda + j0 + j] = a[j];
}

// Rows i >= j0 + 32: A[i][j0..j0+32) <- A[i][j0..j0+32) L_d^-T (one thread per row;
// rows are 16-byte aligned). A finished column is taken out of all later ones at
// once, in the same order for every element: one division and one product in the
// chain per column, where a column at a time its own products are one (8.7 us at
// n = 640). Panels and updates start behind one another; both changes take 5.6 us
// off a pair of them.
__global__ void __launch_bounds__(64) k_chol_panel(float* __restrict__ A, int lda, int n, int j0) {
  __shared__ __align__(16) float Lt[32][36];  // Lt[c][r] = L_d[r][c]
  eogp::pdl_trigger();
  eogp::pdl_wait();
  for (int e = threadIdx.x; e < 1024; e += 64) {
    const int r = e >> 5, c = e & 31;
    Lt[c][r] = A[static_cast<long long>(j0 + r) * lda + j0 + c];
  }
  const int i = j0 + 32 + blockIdx.x * 64 + threadIdx.x;
  float4* row = reinterpret_cast<float4*>(A + static_cast<long long>(i) * lda + j0);
  float x[32];
  if (i < n) {
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float4 v = row[c];
      x[4 * c] = v.x, x[4 * c + 1] = v.y, x[4 * c + 2] = v.z, x[4 * c + 3] = v.w;
    }
  }
  __syncthreads();
  if (i >= n) return;
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    float l[32];
#pragma unroll
    for (int t = c / 4; t < 8; ++t) {
      const float4 v = *reinterpret_cast<const float4*>(&Lt[c][4 * t]);
      l[4 * t] = v.x, l[4 * t + 1] = v.y, l[4 * t + 2] = v.z, l[4 * t + 3] = v.w;
    }
    x[c] = x[c] / l[c];
#pragma unroll
    for (int t = c + 1; t < 32; ++t) x[t] -= x[c] * l[t];
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) row[c] = make_float4(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);
}

// Trailing update of the lower triangle: A[i][j] -= sum_t A[i][j0 + t] A[j][j0 + t]
// for j0 + 32 <= j <= i < n; one block per 64 x 64 tile on or below the diagonal.
// Block 0 holds the next diagonal block and factors it.
__global__ void __launch_bounds__(256) k_chol_update(float* __restrict__ A, int lda, int n, int j0, unsigned* status) {
  __shared__ float Pi[64][33];
  __shared__ float Pj[64][33];
  eogp::pdl_trigger();
  eogp::pdl_wait();
  const int j1 = j0 + 32;
  const int b = blockIdx.x;
  int ti = static_cast<int>((sqrtf(8.0f * b + 1.0f) - 1.0f) * 0.5f);
  while ((ti + 1) * (ti + 2) / 2 <= b) ++ti;
  while (ti * (ti + 1) / 2 > b) --ti;
  const int tj = b - ti * (ti + 1) / 2;
  const int r0 = j1 + ti * 64, c0 = j1 + tj * 64;
  for (int e = threadIdx.x; e < 64 * 8; e += 256) {
    const int r = e >> 3, t = 4 * (e & 7);
    float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
    if (r0 + r < n) u = *reinterpret_cast<const float4*>(A + static_cast<long long>(r0 + r) * lda + j0 + t);
    if (c0 + r < n) v = *reinterpret_cast<const float4*>(A + static_cast<long long>(c0 + r) * lda + j0 + t);
    Pi[r][t] = u.x, Pi[r][t + 1] = u.y, Pi[r][t + 2] = u.z, Pi[r][t + 3] = u.w;
    Pj[r][t] = v.x, Pj[r][t + 1] = v.y, Pj[r][t + 2] = v.z, Pj[r][t + 3] = v.w;
  }
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float old[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int i = r0 + ty + 16 * u, j = c0 + tx + 16 * v;
      old[u][v] = (i < n && j <= i) ? A[static_cast<long long>(i) * lda + j] : 0.f;
    }
  __syncthreads();
  float acc[4][4] = {};
#pragma unroll 8
  for (int t = 0; t < 32; ++t) {
    float a[4], bb[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      a[u] = Pi[ty + 16 * u][t];
      bb[u] = Pj[tx + 16 * u][t];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc[u][v] = fmaf(a[u], bb[v], acc[u][v]);
  }
  if (b == 0) __syncthreads();  // every thread is done with Pi
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = r0 + ty + 16 * u;
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int j = c0 + tx + 16 * v;
      const float x = old[u][v] - acc[u][v];
      if (b == 0 && u < 2 && v < 2) Pi[ty + 16 * u][tx + 16 * v] = x;
      if (i < n && j <= i && !(b == 0 && u < 2 && v < 2)) A[static_cast<long long>(i) * lda + j] = x;
    }
  }
  if (b != 0) return;
  __syncthreads();
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x, nb = min(32, n - j1);
  float a[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) a[j] = (lane < nb && j <= lane) ? Pi[lane][j] : 0.f;
  chol_block(a, lane, nb, status);
#pragma unroll
  for (int j = 0; j < 32; ++j)
    if (lane < nb && j < nb) A[static_cast<long long>(j1 + lane) * lda + j1 + j] = a[j];
}

// ---- inverse of a lower-triangular matrix (fp32), 32 x 32 blocks; Li zeroed first
// Diagonal blocks: one 32-thread block per block, one column each.
__global__ void k_trinv_diag(const float* __restrict__ L, int lda, float* __restrict__ Li, int ldi, int n) {
  __shared__ float Ls[32][33];
  const int j0 = blockIdx.x * 32, nb = min(32, n - j0), c = threadIdx.x;
  for (int r = 0; r < 32; ++r)
    Ls[r][c] = (r < nb && c < nb) ? L[static_cast<long long>(j0 + r) * lda + j0 + c] : 0.f;
  __syncthreads();
  if (c >= nb) return;
  float x[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    float v = 0.f;
    if (i >= c && i < nb) {
      v = (i == c) ? 1.f : 0.f;
      for (int t = c; t < i; ++t) v -= Ls[i][t] * x[t];
      v /= Ls[i][i];
    }
    x[i] = v;
  }
  for (int i = c; i < nb; ++i) Li[static_cast<long long>(j0 + i) * ldi + j0 + c] = x[i];
}

// Blocks below the diagonal: Li[I][J] = -Li[I][I] sum_{K=J}^{I-1} L[I][K] Li[K][J].
// The columns of an inverse are independent: a block of 256 threads takes w = 8
// columns of block column J (4 where n x 8 floats exceed the shared memory) and goes
// down its rows, the columns so far in shared memory. n is a multiple of 32; two
// blocks of L are fetched ahead.
__global__ void __launch_bounds__(256) k_trinv_cols(const float* __restrict__ L, int lda, float* __restrict__ Li,
                                                    int ldi, int n, int w) {
  extern __shared__ float col[];  // [row - 32 J][w]
  __shared__ float As[2][32][33];
  __shared__ float Ts[32][8];
  const int J = blockIdx.x, c0 = J * 32 + blockIdx.y * w;
  const int r = threadIdx.x >> 3, c = threadIdx.x & 7;      // this thread's row and column of a block
  const int lr = threadIdx.x >> 3, lc = 4 * (threadIdx.x & 7);  // its 16 bytes of a 32 x 32 block
  const bool mine = c < w;
  if (mine) col[r * w + c] = Li[static_cast<long long>(J * 32 + r) * ldi + c0 + c];
  const int nblk = n / 32;
  // the blocks in the order they are used: L[I][J .. I-1], then Li[I][I]
  auto fetch = [&](int I, int K) {
    return K < I ? *reinterpret_cast<const float4*>(L + static_cast<long long>(I * 32 + lr) * lda + K * 32 + lc)
                 : *reinterpret_cast<const float4*>(Li + static_cast<long long>(I * 32 + lr) * ldi + I * 32 + lc);
  };
  auto after = [&](int& I, int& K) {
    if (++K > I) {
      ++I;
      K = J;
    }
  };
  int fI = J + 1, fK = J;
  float4 f0 = make_float4(0.f, 0.f, 0.f, 0.f), f1 = f0;
  if (fI < nblk) f0 = fetch(fI, fK);
  after(fI, fK);
  if (fI < nblk) f1 = fetch(fI, fK);
  after(fI, fK);
  int buf = 0;
  for (int I = J + 1; I < nblk; ++I) {
    float acc = 0.f;
    for (int K = J; K <= I; ++K, buf ^= 1) {
      float(*A)[33] = As[buf];
      A[lr][lc] = f0.x, A[lr][lc + 1] = f0.y, A[lr][lc + 2] = f0.z, A[lr][lc + 3] = f0.w;
      if (K == I) Ts[r][c] = acc;
      f0 = f1;
      if (fI < nblk) f1 = fetch(fI, fK);
      after(fI, fK);
      __syncthreads();
      if (!mine) continue;
      if (K < I) {
        const float* b = col + (K - J) * 32 * w + c;
#pragma unroll
        for (int t = 0; t < 32; ++t) acc = fmaf(A[r][t], b[w * t], acc);
      } else {
        float v = 0.f;
#pragma unroll
        for (int t = 0; t < 32; ++t) v = fmaf(A[r][t], Ts[t][c], v);
        col[(I - J) * 32 * w + r * w + c] = -v;
        Li[static_cast<long long>(I * 32 + r) * ldi + c0 + c] = -v;
      }
    }
  }
}

// H64[i][j] = (H[i][j] + H[j][i]) / 2
__global__ void k_sym_f64(const float* __restrict__ H, int ldh, int n, double* __restrict__ out) {
  const long long tot = static_cast<long long>(n) * n;
  for (long long e = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x; e < tot;
       e += static_cast<long long>(gridDim.x) * blockDim.x) {
    const int i = static_cast<int>(e / n), j = static_cast<int>(e % n);
    out[e] = 0.5 * (static_cast<double>(H[static_cast<long long>(i) * ldh + j]) +
                    static_cast<double>(H[static_cast<long long>(j) * ldh + i]));
  }
}

// St[j][c] = Vt[sel[j]][c] (rows of the Ritz rotation, eigenvalue descending); theta[j] = mu[sel[j]]
__global__ void k_ritz_rows(const double* __restrict__ Vt, int n, const int* __restrict__ sel,
                            const double* __restrict__ mu, float* __restrict__ St, int lds,
                            float* __restrict__ theta) {
  const int j = blockIdx.x;
  const double* v = Vt + static_cast<long long>(sel[j]) * n;
  for (int c = threadIdx.x; c < n; c += blockDim.x) St[static_cast<long long>(j) * lds + c] = static_cast<float>(v[c]);
  if (threadIdx.x == 0) theta[j] = static_cast<float>(mu[sel[j]]);
}

// out[0] = max over j < k of ||CX[j] - theta_j X[j]|| / |theta_j| (float bits, atomicMax; out zeroed first)
__global__ void __launch_bounds__(256) k_ritz_resid(const float* __restrict__ X, const float* __restrict__ CX,
                                                    long long ld, int nn, const float* __restrict__ theta,
                                                    unsigned* __restrict__ out) {
  __shared__ double red[256];
  const int j = blockIdx.x;
  const float th = theta[j];
  double ss = 0.0;
  for (int c = threadIdx.x; c < nn; c += 256) {
    const double r = static_cast<double>(CX[j * ld + c]) - static_cast<double>(th) * X[j * ld + c];
    ss = fma(r, r, ss);
  }
  red[threadIdx.x] = ss;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    float v = th != 0.f ? static_cast<float>(sqrt(red[0]) / fabs(static_cast<double>(th))) : 0.f;
    if (!(v == v)) v = 3.0e38f;  // NaN: never converged
    atomicMax(out, __float_as_uint(v));
  }
}

__global__ void k_copy_eig(const float* __restrict__ theta, int k, float* __restrict__ eig) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < k) eig[r] = theta[r];
}

// ---------------------------------------------------------------- layouts
int pca_block(int k) { return rup(k + std::max(64, k / 4), 32); }

bool use_subspace(int nn, int k) { return nn > 1024 && pca_block(k) < nn; }

struct DenseLayout {
  size_t A, A2, Vt, cs, mu, sel, red, Pr, total;
};

DenseLayout dense_layout(int n, int m, int k) {
  const size_t nn = static_cast<size_t>(std::min(n, m));
  DenseLayout L{};
  size_t o = 0;
  auto take = [&](size_t b) { const size_t at = o; o += al256(b); return at; };
  L.A = take(nn * nn * 8);
  L.A2 = take(nn * nn * 8);
  L.Vt = take(nn * nn * 8);
  L.cs = take((nn / 2 + 1) * 4 * 8);
  L.mu = take(nn * 8);
  L.sel = take(nn * 4);
  L.red = take(4 * 8);
  L.Pr = n < m ? take(static_cast<size_t>(k) * m * 8) : 0;
  L.total = o;
  return L;
}

struct SubLayout {
  int nn, p, nn4, nn8, p4, p8, n8, m8;
  size_t Zh, Zl, ZTh, ZTl;       // Z [n][m8] (Gram route); Z^T [m][n8] (both routes with Z)
  size_t A32, Ah, Al;            // A [nn][nn8] fp32 / bf16 hi, lo
  size_t X32, CX32;              // X^T, (A X)^T [p][nn4] fp32
  size_t Yh, Yl;                 // row-normalised splits [p][nn8]
  size_t YTh, YTl, CTh, CTl;     // transposed splits [nn][p8]
  size_t G32, Li32, Sh, Sl;      // [p][p4] fp32, splits [p][p8]
  size_t rs, shift, theta, resid;
  size_t H64, H64b, V64, cs, mu, sel, red;
  size_t Pr;                     // Gram route: raw directions [k][m4] fp32
  size_t total;
};

SubLayout sub_layout(int n, int m, int k, bool with_z) {
  SubLayout L{};
  L.nn = std::min(n, m);
  L.p = pca_block(k);
  L.nn4 = rup(L.nn, 4);
  L.nn8 = rup(L.nn, 8);
  L.p4 = rup(L.p, 4);
  L.p8 = rup(L.p, 8);
  L.n8 = rup(n, 8);
  L.m8 = rup(m, 8);
  const size_t nn = L.nn, p = L.p;
  size_t o = 0;
  auto take = [&](size_t b) { const size_t at = o; o += al256(b); return at; };
  const bool gram = n < m;
  if (with_z) {
    if (gram) {
      L.Zh = take(static_cast<size_t>(n) * L.m8 * 2);
      L.Zl = take(static_cast<size_t>(n) * L.m8 * 2);
    }
    L.ZTh = take(static_cast<size_t>(m) * L.n8 * 2);
    L.ZTl = take(static_cast<size_t>(m) * L.n8 * 2);
  }
  L.A32 = take(nn * L.nn8 * 4);
  L.Ah = take(nn * L.nn8 * 2);
  L.Al = take(nn * L.nn8 * 2);
  L.X32 = take(p * L.nn4 * 4);
  L.CX32 = take(p * L.nn4 * 4);
  L.Yh = take(p * L.nn8 * 2);
  L.Yl = take(p * L.nn8 * 2);
  // transposed splits [nn][p8]; also used for row splits [p][nn8]
  const size_t ybig = std::max(nn * L.p8, p * L.nn8);
  L.YTh = take(ybig * 2);
  L.YTl = take(ybig * 2);
  L.CTh = take(nn * L.p8 * 2);
  L.CTl = take(nn * L.p8 * 2);
  L.G32 = take(p * L.p4 * 4);
  L.Li32 = take(p * L.p4 * 4);
  L.Sh = take(p * L.p8 * 2);
  L.Sl = take(p * L.p8 * 2);
  L.rs = take(p * 4);
  L.shift = take(16);
  L.theta = take(p * 4);
  L.resid = take(16);
  L.H64 = take(p * p * 8);
  L.H64b = take(p * p * 8);
  L.V64 = take(p * p * 8);
  L.cs = take((p / 2 + 1) * 4 * 8);
  L.mu = take(p * 8);
  L.sel = take(p * 4);
  L.red = take(4 * 8);
  L.Pr = gram ? take(static_cast<size_t>(k) * rup(m, 4) * 4) : 0;
  L.total = o;
  return L;
}

}  // namespace

bool fit_pca_supported(int n, int m, int k) {
  const int nn = std::min(n, m);
  if (use_subspace(nn, k)) return pca_block(k) <= 12288 && nn <= 32768;
  return nn <= 12288;
}

size_t fit_pca_ws_bytes(int n, int m, int k) {
  const int nn = std::min(n, m);
  if (use_subspace(nn, k)) return sub_layout(n, m, k, true).total;
  return dense_layout(n, m, k).total;
}

#define PCA_TRY(x)                                                                         \
  do {                                                                                     \
    cudaError_t e_ = (x);                                                                  \
    if (e_ != cudaSuccess)                                                                 \
      return eogp::set_error(EOGP_ECUDA, "fit_pca: %s: %s", #x, cudaGetErrorString(e_));   \
  } while (0)

namespace {

unsigned grid_for(long long tot) {
  return static_cast<unsigned>(std::max<long long>(1, std::min<long long>((tot + 255) / 256, 152LL * 16)));
}

// Cyclic Jacobi on A (fp64, n x n, overwritten by its diagonal form; A2 of the same
// size); Vt = eigenvectors as rows. cs: 2 (n + 1) doubles; red: 4 doubles.
int jacobi_eigen(double* A, double* A2, double* Vt, int nn, double* cs, double* red, unsigned* status, cudaStream_t st,
                 int max_sweeps) {
  const int np = nn + (nn & 1);
  {
    const long long tot = static_cast<long long>(nn) * nn;
    k_eye<<<static_cast<unsigned>((tot + 255) / 256), 256, 0, st>>>(Vt, nn);
    PCA_TRY(cudaGetLastError());
  }
  int dev = 0, sms = 0;
  PCA_TRY(cudaGetDevice(&dev));
  PCA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  double* cur = A;
  double* oth = A2;
  double2* cs0 = reinterpret_cast<double2*>(cs);
  double2* cs1 = cs0 + np / 2;
  unsigned* count = reinterpret_cast<unsigned*>(red + 2);
  const void* kernel = nn == np ? reinterpret_cast<const void*>(k_jacobi_sweep<true>)
                                : reinterpret_cast<const void*>(k_jacobi_sweep<false>);
  double prev_off = -1.0;
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    PCA_TRY(cudaMemsetAsync(red, 0, 4 * sizeof(double), st));
    if (nn > 1) {
      int n = nn, npv = np;
      void* args[] = {&cur, &oth, &Vt, &n, &npv, &cs0, &cs1, &count, &status};
      PCA_TRY(cudaLaunchCooperativeKernel(kernel, dim3(sms), dim3(kJacThreads), args, 0, st));
      std::swap(cur, oth);  // np - 1 steps, an odd number
    }
    k_offnorm<<<304, 256, 0, st>>>(cur, nn, red);
    PCA_TRY(cudaGetLastError());
    double h[2];
    PCA_TRY(cudaMemcpyAsync(h, red, sizeof(h), cudaMemcpyDeviceToHost, st));
    PCA_TRY(cudaStreamSynchronize(st));
    if (!std::isfinite(h[1]))
      return eogp::set_error(EOGP_EDEVICE, "fit_pca: values that are not finite (in the input or its second moment)");
    const double off = std::sqrt(h[0]), tot = std::sqrt(h[1]);
    if (!(off > 1e-11 * tot)) break;
    if (prev_off >= 0.0 && sweep >= 4 && off > 0.5 * prev_off) break;  // rounding floor
    prev_off = off;
  }
  if (cur != A)
    PCA_TRY(cudaMemcpyAsync(A, cur, static_cast<size_t>(nn) * nn * sizeof(double), cudaMemcpyDeviceToDevice, st));
  return EOGP_OK;
}

int fit_dense(const float* Z, int n, int m, int ldz, int k, void* Pt, int ld_pt, int pt_dtype, float* eig,
              char* ws, unsigned* status, cudaStream_t st, const double* C_in, int ldc) {
  const DenseLayout L = dense_layout(C_in ? m : n, m, k);
  double* A = reinterpret_cast<double*>(ws + L.A);
  double* Vt = reinterpret_cast<double*>(ws + L.Vt);
  double* cs = reinterpret_cast<double*>(ws + L.cs);
  double* mu = reinterpret_cast<double*>(ws + L.mu);
  int* sel = reinterpret_cast<int*>(ws + L.sel);
  double* red = reinterpret_cast<double*>(ws + L.red);
  const bool gram = !C_in && n < m;
  const int nn = gram ? n : m;
  if (gram) {
    // A = Z Z^T (n x n)
    PCA_TRY(gemm_f64acc<float>(n, n, m, 1.0, Z, ldz, 1, Z, ldz, 1, A, n, st));
  } else if (C_in) {
    // A = C / n from a second moment summed elsewhere (e.g. over shards)
    k_scale_copy<<<static_cast<unsigned>((static_cast<long long>(m) * m + 255) / 256), 256, 0, st>>>(
        C_in, ldc, m, 1.0 / n, A);
    PCA_TRY(cudaGetLastError());
  } else {
    // A = Z^T Z / n (m x m): A(i,j) = sum_r Z[r][i] Z[r][j]
    PCA_TRY(gemm_f64acc<float>(m, m, n, 1.0 / n, Z, 1, ldz, Z, 1, ldz, A, m, st));
  }
  if (int rc = jacobi_eigen(A, reinterpret_cast<double*>(ws + L.A2), Vt, nn, cs, red, status, st, 40)) return rc;
  k_rank<<<(nn + 255) / 256, 256, 0, st>>>(A, nn, k, mu, sel);
  PCA_TRY(cudaGetLastError());
  const int bf = pt_dtype == EOGP_BF16 ? 1 : 0;
  if (!gram) {
    k_emit<double><<<k, 256, 0, st>>>(Vt, nn, sel, m, Pt, ld_pt, bf, mu, 1.0, eig);
    PCA_TRY(cudaGetLastError());
  } else {
    double* Pr = reinterpret_cast<double*>(ws + L.Pr);
    // U_k rows (eigenvectors of Z Z^T) -> A's storage, then Pr = U_k Z (k x m).
    k_gather_f64_rows<<<k, 256, 0, st>>>(Vt, nn, sel, nn, A);
    PCA_TRY(cudaGetLastError());
    // Pr[r][c] = sum_x U[r][x] Z[x][c]
    PCA_TRY(gemm_f64acc<double>(k, m, n, 1.0, A, n, 1, Z, 1, ldz, Pr, m, st));
    k_emit<double><<<k, 256, 0, st>>>(Pr, m, nullptr, m, Pt, ld_pt, bf, mu, 1.0 / n, nullptr);
    PCA_TRY(cudaGetLastError());
    // eigenvalues of Z^T Z / n: mu[sel[r]] / n
    k_eig_out<<<(k + 255) / 256, 256, 0, st>>>(mu, sel, k, 1.0 / n, eig);
    PCA_TRY(cudaGetLastError());
  }
  return EOGP_OK;
}

// One Cholesky-QR pass: X32 (rows of X^T, p x nn4) <- orthonormal basis of the rows of Y32
// (which may be the same buffer): rows normalised, G = Y Y^T (tensor cores),
// L = chol(G + rel * mean(diag G) I), X^T = L^-1 Y^T.
int chol_qr_pass(const SubLayout& L, char* w, const float* Y32, float* X32, float rel, unsigned* status,
                 cudaStream_t st) {
  const int p = L.p, nn = L.nn;
  float* rs = reinterpret_cast<float*>(w + L.rs);
  bf16* Yh = reinterpret_cast<bf16*>(w + L.Yh);
  bf16* Yl = reinterpret_cast<bf16*>(w + L.Yl);
  bf16* YTh = reinterpret_cast<bf16*>(w + L.YTh);
  bf16* YTl = reinterpret_cast<bf16*>(w + L.YTl);
  float* G = reinterpret_cast<float*>(w + L.G32);
  float* Li = reinterpret_cast<float*>(w + L.Li32);
  bf16* Sh = reinterpret_cast<bf16*>(w + L.Sh);
  bf16* Sl = reinterpret_cast<bf16*>(w + L.Sl);
  float* shift = reinterpret_cast<float*>(w + L.shift);
  k_row_invnorm<<<p, 256, 0, st>>>(Y32, L.nn4, nn, rs);
  k_split_rows<<<grid_for(static_cast<long long>(p) * L.nn8), 256, 0, st>>>(Y32, L.nn4, p, nn, rs, Yh, Yl, L.nn8);
  k_split_T<<<dim3((nn + 31) / 32, (L.p8 + 31) / 32), dim3(32, 8), 0, st>>>(Y32, L.nn4, p, nn, rs, YTh, YTl, L.p8);
  PCA_TRY(cudaGetLastError());
  PCA_TRY(launch_tc_gemm_hl(p, p, nn, Yh, Yl, L.nn8, Yh, Yl, L.nn8, G, L.p4, 1.0f, status, st));
  k_diag_shift<<<1, 256, 0, st>>>(G, L.p4, p, rel, shift);
  k_add_diag<<<(p + 255) / 256, 256, 0, st>>>(G, L.p4, p, shift);
  PCA_TRY(cudaGetLastError());
  k_chol_diag<<<1, 32, 0, st>>>(G, L.p4, p, 0, status);
  for (int j0 = 0; j0 + 32 < p; j0 += 32) {
    const int below = p - (j0 + 32), nt = (below + 63) / 64;
    PCA_TRY(launch_behind(k_chol_panel, (below + 63) / 64, 64, 0, st, G, L.p4, p, j0));
    PCA_TRY(launch_behind(k_chol_update, nt * (nt + 1) / 2, 256, 0, st, G, L.p4, p, j0, status));
  }
  PCA_TRY(cudaGetLastError());
  PCA_TRY(cudaMemsetAsync(Li, 0, static_cast<size_t>(p) * L.p4 * 4, st));
  const int nblk = (p + 31) / 32;
  k_trinv_diag<<<nblk, 32, 0, st>>>(G, L.p4, Li, L.p4, p);
  const int cw = static_cast<size_t>(p) * 8 * sizeof(float) <= 200 * 1024 ? 8 : 4;
  const size_t cols = static_cast<size_t>(p) * cw * sizeof(float);
  PCA_TRY(allow_smem(k_trinv_cols, 10 * 1024));
  k_trinv_cols<<<dim3(nblk, 32 / cw), 256, cols, st>>>(G, L.p4, Li, L.p4, p, cw);
  PCA_TRY(cudaGetLastError());
  k_split_rows<<<grid_for(static_cast<long long>(p) * L.p8), 256, 0, st>>>(Li, L.p4, p, p, nullptr, Sh, Sl, L.p8);
  PCA_TRY(cudaGetLastError());
  // X^T[j][l] = sum_i Li[j][i] Y^T[i][l]: A operand Li (K = p), B operand Y [nn][p8]
  PCA_TRY(launch_tc_gemm_hl(p, nn, p, Sh, Sl, L.p8, YTh, YTl, L.p8, X32, L.nn4, 1.0f, status, st));
  return EOGP_OK;
}

int orthonormalise(const SubLayout& L, char* w, const float* Y32, float* X32, unsigned* status, cudaStream_t st) {
  if (int rc = chol_qr_pass(L, w, Y32, X32, 1e-2f, status, st)) return rc;
  if (int rc = chol_qr_pass(L, w, X32, X32, 1e-4f, status, st)) return rc;
  return chol_qr_pass(L, w, X32, X32, 0.0f, status, st);
}

// CX32 = (A X)^T = X^T A: rows of X^T split, times the symmetric A (hi/lo).
int apply_A(const SubLayout& L, char* w, const float* X32, float* CX32, unsigned* status, cudaStream_t st) {
  bf16* Yh = reinterpret_cast<bf16*>(w + L.Yh);
  bf16* Yl = reinterpret_cast<bf16*>(w + L.Yl);
  k_split_rows<<<grid_for(static_cast<long long>(L.p) * L.nn8), 256, 0, st>>>(X32, L.nn4, L.p, L.nn, nullptr, Yh,
                                                                             Yl, L.nn8);
  PCA_TRY(cudaGetLastError());
  PCA_TRY(launch_tc_gemm_hl(L.p, L.nn, L.nn, Yh, Yl, L.nn8, w + L.Ah, w + L.Al, L.nn8, CX32, L.nn4, 1.0f, status,
                            st));
  return EOGP_OK;
}

// Rayleigh-Ritz: H = X^T (A X), eigenpairs, X and A X rotated onto the Ritz
// vectors (descending); returns the largest relative residual of the top k.
int rayleigh_ritz(const SubLayout& L, char* w, int k, unsigned* status, cudaStream_t st, float* max_res) {
  const int p = L.p, nn = L.nn;
  float* X32 = reinterpret_cast<float*>(w + L.X32);
  float* CX32 = reinterpret_cast<float*>(w + L.CX32);
  bf16* Yh = reinterpret_cast<bf16*>(w + L.Yh);
  bf16* Yl = reinterpret_cast<bf16*>(w + L.Yl);
  bf16* YTh = reinterpret_cast<bf16*>(w + L.YTh);
  bf16* YTl = reinterpret_cast<bf16*>(w + L.YTl);
  bf16* CTh = reinterpret_cast<bf16*>(w + L.CTh);
  bf16* CTl = reinterpret_cast<bf16*>(w + L.CTl);
  float* H = reinterpret_cast<float*>(w + L.G32);
  float* S32 = reinterpret_cast<float*>(w + L.Li32);
  bf16* Sh = reinterpret_cast<bf16*>(w + L.Sh);
  bf16* Sl = reinterpret_cast<bf16*>(w + L.Sl);
  double* H64 = reinterpret_cast<double*>(w + L.H64);
  double* V64 = reinterpret_cast<double*>(w + L.V64);
  double* mu = reinterpret_cast<double*>(w + L.mu);
  int* sel = reinterpret_cast<int*>(w + L.sel);
  float* theta = reinterpret_cast<float*>(w + L.theta);
  unsigned* resid = reinterpret_cast<unsigned*>(w + L.resid);
  // H = X^T (A X): rows of X^T and rows of (A X)^T, K = nn
  k_split_rows<<<grid_for(static_cast<long long>(p) * L.nn8), 256, 0, st>>>(X32, L.nn4, p, nn, nullptr, Yh, Yl,
                                                                          L.nn8);
  k_split_rows<<<grid_for(static_cast<long long>(p) * L.nn8), 256, 0, st>>>(CX32, L.nn4, p, nn, nullptr, YTh,
                                                                          YTl, L.nn8);
  PCA_TRY(cudaGetLastError());
  PCA_TRY(launch_tc_gemm_hl(p, p, nn, Yh, Yl, L.nn8, YTh, YTl, L.nn8, H, L.p4, 1.0f, status, st));
  k_sym_f64<<<grid_for(static_cast<long long>(p) * p), 256, 0, st>>>(H, L.p4, p, H64);
  PCA_TRY(cudaGetLastError());
  if (int rc = jacobi_eigen(H64, reinterpret_cast<double*>(w + L.H64b), V64, p, reinterpret_cast<double*>(w + L.cs),
                            reinterpret_cast<double*>(w + L.red), status, st, 40))
    return rc;
  k_rank<<<(p + 255) / 256, 256, 0, st>>>(H64, p, p, mu, sel);
  k_ritz_rows<<<p, 256, 0, st>>>(V64, p, sel, mu, S32, L.p4, theta);
  k_split_rows<<<grid_for(static_cast<long long>(p) * L.p8), 256, 0, st>>>(S32, L.p4, p, p, nullptr, Sh, Sl, L.p8);
  // X and A X as K-major operands [nn][p8] (transposed splits)
  k_split_T<<<dim3((nn + 31) / 32, (L.p8 + 31) / 32), dim3(32, 8), 0, st>>>(X32, L.nn4, p, nn, nullptr, YTh, YTl,
                                                                           L.p8);
  k_split_T<<<dim3((nn + 31) / 32, (L.p8 + 31) / 32), dim3(32, 8), 0, st>>>(CX32, L.nn4, p, nn, nullptr, CTh, CTl,
                                                                           L.p8);
  PCA_TRY(cudaGetLastError());
  PCA_TRY(launch_tc_gemm_hl(p, nn, p, Sh, Sl, L.p8, YTh, YTl, L.p8, X32, L.nn4, 1.0f, status, st));
  PCA_TRY(launch_tc_gemm_hl(p, nn, p, Sh, Sl, L.p8, CTh, CTl, L.p8, CX32, L.nn4, 1.0f, status, st));
  PCA_TRY(cudaMemsetAsync(resid, 0, 4, st));
  k_ritz_resid<<<k, 256, 0, st>>>(X32, CX32, L.nn4, nn, theta, resid);
  PCA_TRY(cudaGetLastError());
  unsigned hbits = 0;
  PCA_TRY(cudaMemcpyAsync(&hbits, resid, 4, cudaMemcpyDeviceToHost, st));
  PCA_TRY(cudaStreamSynchronize(st));
  float v;
  std::memcpy(&v, &hbits, 4);
  *max_res = v;
  return EOGP_OK;
}

int fit_subspace(const float* Z, int n, int m, int ldz, int k, void* Pt, int ld_pt, int pt_dtype, float* eig,
                 char* w, unsigned* status, cudaStream_t st, const double* C_in, int ldc) {
  const bool gram = !C_in && n < m;
  const SubLayout L = sub_layout(C_in ? m : n, m, k, !C_in);
  const int nn = L.nn, p = L.p;
  float* A32 = reinterpret_cast<float*>(w + L.A32);
  // 1. A = Z^T Z / n or Z Z^T / n (tensor cores), or C / n; symmetrised hi/lo pair
  if (C_in) {
    k_f64_to_f32<<<grid_for(static_cast<long long>(m) * m), 256, 0, st>>>(C_in, ldc, m, 1.0 / n, A32, L.nn8);
    PCA_TRY(cudaGetLastError());
  } else {
    bf16* ZTh = reinterpret_cast<bf16*>(w + L.ZTh);
    bf16* ZTl = reinterpret_cast<bf16*>(w + L.ZTl);
    k_split_T<<<dim3((m + 31) / 32, (L.n8 + 31) / 32), dim3(32, 8), 0, st>>>(Z, ldz, n, m, nullptr, ZTh, ZTl, L.n8);
    PCA_TRY(cudaGetLastError());
    if (gram) {
      bf16* Zh = reinterpret_cast<bf16*>(w + L.Zh);
      bf16* Zl = reinterpret_cast<bf16*>(w + L.Zl);
      k_split_rows<<<grid_for(static_cast<long long>(n) * L.m8), 256, 0, st>>>(Z, ldz, n, m, nullptr, Zh, Zl, L.m8);
      PCA_TRY(cudaGetLastError());
      PCA_TRY(launch_tc_gemm_hl(n, n, m, Zh, Zl, L.m8, Zh, Zl, L.m8, A32, L.nn8, 1.0f / n, status, st));
    } else {
      PCA_TRY(launch_tc_gemm_hl(m, m, n, ZTh, ZTl, L.n8, ZTh, ZTl, L.n8, A32, L.nn8, 1.0f / n, status, st));
    }
  }
  k_split_sym<<<dim3((L.nn8 + 31) / 32, (nn + 31) / 32), dim3(32, 8), 0, st>>>(
      A32, L.nn8, nn, reinterpret_cast<bf16*>(w + L.Ah), reinterpret_cast<bf16*>(w + L.Al), L.nn8);
  PCA_TRY(cudaGetLastError());
  // 2. start: orthonormal basis of p Gaussian rows
  float* X32 = reinterpret_cast<float*>(w + L.X32);
  float* CX32 = reinterpret_cast<float*>(w + L.CX32);
  PCA_TRY(cudaMemsetAsync(X32, 0, static_cast<size_t>(p) * L.nn4 * 4, st));
  PCA_TRY(cudaMemsetAsync(CX32, 0, static_cast<size_t>(p) * L.nn4 * 4, st));
  k_gauss<<<grid_for(static_cast<long long>(p) * nn), 256, 0, st>>>(X32, L.nn4, p, nn, 0x5eedull);
  PCA_TRY(cudaGetLastError());
  if (int rc = orthonormalise(L, w, X32, X32, status, st)) return rc;
  // 3. iterate: X <- orth(A X); Rayleigh-Ritz every 5 iterations
  const int kRR = 5, kMaxIt = 400;
  const float kTol = 1e-3f;
  bool converged = false;
  for (int it = 1; it <= kMaxIt; ++it) {
    if (int rc = apply_A(L, w, X32, CX32, status, st)) return rc;
    if (it % kRR == 0) {
      float res = 0.f;
      if (int rc = rayleigh_ritz(L, w, k, status, st, &res)) return rc;
      if (res <= kTol) {
        converged = true;
        break;
      }
    }
    if (int rc = orthonormalise(L, w, CX32, X32, status, st)) return rc;
  }
  if (!converged)
    return eogp::set_error(EOGP_EDEVICE, "fit_pca: subspace iteration did not reach the residual bound in %d "
                           "iterations", kMaxIt);
  // 4. outputs: the top k Ritz pairs
  const int bf = pt_dtype == EOGP_BF16 ? 1 : 0;
  const float* theta = reinterpret_cast<const float*>(w + L.theta);
  if (!gram) {
    k_emit<float><<<k, 256, 0, st>>>(X32, L.nn4, nullptr, m, Pt, ld_pt, bf, nullptr, 1.0, nullptr);
  } else {
    // P rows = U_k^T Z (normalised): A operand rows of U^T (K = n), B operand Z^T [m][n8]
    bf16* Yh = reinterpret_cast<bf16*>(w + L.Yh);
    bf16* Yl = reinterpret_cast<bf16*>(w + L.Yl);
    float* Pr = reinterpret_cast<float*>(w + L.Pr);
    k_split_rows<<<grid_for(static_cast<long long>(k) * L.nn8), 256, 0, st>>>(X32, L.nn4, k, nn, nullptr, Yh, Yl,
                                                                            L.nn8);
    PCA_TRY(cudaGetLastError());
    PCA_TRY(launch_tc_gemm_hl(k, m, n, Yh, Yl, L.nn8, w + L.ZTh, w + L.ZTl, L.n8, Pr, rup(m, 4), 1.0f, status, st));
    k_emit<float><<<k, 256, 0, st>>>(Pr, rup(m, 4), nullptr, m, Pt, ld_pt, bf, nullptr, 1.0, nullptr);
  }
  PCA_TRY(cudaGetLastError());
  k_copy_eig<<<(k + 255) / 256, 256, 0, st>>>(theta, k, eig);
  PCA_TRY(cudaGetLastError());
  return EOGP_OK;
}

}  // namespace

int fit_pca_device(const float* Z, int n, int m, int ldz, int k, void* Pt, int ld_pt, int pt_dtype,
                   float* eig, void* ws, unsigned* status, cudaStream_t st, const double* C_in, int ldc) {
  const int nn = C_in ? m : std::min(n, m);
  char* w = static_cast<char*>(ws);
  if (use_subspace(nn, k)) return fit_subspace(Z, n, m, ldz, k, Pt, ld_pt, pt_dtype, eig, w, status, st, C_in, ldc);
  return fit_dense(Z, n, m, ldz, k, Pt, ld_pt, pt_dtype, eig, w, status, st, C_in, ldc);
}

cudaError_t second_moment_device(const float* Z, int n, int m, int ldz, double* C, int ldc, int accumulate,
                                 cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  // C(i,j) (+)= sum_r Z[r][i] Z[r][j]
  return gemm_f64acc<float>(m, m, n, 1.0, Z, 1, ldz, Z, 1, ldz, C, ldc, st, accumulate);
}
