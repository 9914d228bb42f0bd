// Dense N x N kernels of Cholesky-QR and Rayleigh-Ritz for large blocks of
// vectors (N in the thousands, Sec. V on the 280-atom cluster), spread over
// many SMs:
//   * blocked right-looking Cholesky (64-column panels: one-CTA diagonal block,
//     row-parallel triangular solve of the panel, trailing update in tiles that keep
//     the one-CTA factor's order of sums, as an FP64 GEMM above 2,048 rows);
//   * the inverse of a lower triangle by 2 x 2 block recursion (two half-size
//     inverses and two GEMMs);
//   * a two-sided block Jacobi eigensolver for symmetric matrices: the matrix
//     is cut into blocks of B rows/columns, a round-robin tournament pairs the
//     blocks, one CTA rotates every pair's 2B x 2B subproblem in shared memory
//     (one cyclic Jacobi sweep; above 512 rows until it is diagonal), and the pair's
//     rotation is applied to its 2B rows and columns of the whole matrix and to the
//     eigenvector matrix by many CTAs (row-times-2B x 2B products), B = 16.  Float
//     (the fast first stage) and double (the refinement).
// No atomics: every result has a fixed order of operations.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <atomic>
#include <vector>

#include "efe_kernels.h"

namespace efe {

extern std::atomic<int64_t> g_launches;

namespace {

constexpr int CB = 64;        // Cholesky panel width
// block Jacobi: block size BJ_B (a template parameter), subproblems of
// BJ_S = 2 BJ_B, shared rows of BJ_S + 1

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

// ---------------------------------------------------------------- Cholesky
// Diagonal block A[j0:j0+b, j0:j0+b] (already updated by the panels before it)
// factorised in place by one CTA; info = j + 1 of the first breakdown (global
// index), left alone if it is already set.
__global__ void __launch_bounds__(1024) k_chol_diag(double* A, int lda, int j0, int b, int* info) {
  __shared__ double S[CB][CB + 1];
  __shared__ int bad;
  const int tid = threadIdx.x;
  for (int t = tid; t < b * b; t += blockDim.x) S[t / b][t % b] = A[(int64_t)(j0 + t / b) * lda + j0 + t % b];
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int j = 0; j < b; ++j) {
    if (tid == 0) {
      const double d = S[j][j];
      if (!(d > 0.0) || !isfinite(d)) {
        bad = j + 1;
        S[j][j] = 1.0;
      } else {
        S[j][j] = sqrt(d);
      }
    }
    __syncthreads();
    const double piv = S[j][j];
    for (int i = j + 1 + tid; i < b; i += blockDim.x) S[i][j] /= piv;
    __syncthreads();
    for (int t = tid; t < (b - j - 1) * (b - j - 1); t += blockDim.x) {
      const int i = j + 1 + t / (b - j - 1), c = j + 1 + t % (b - j - 1);
      if (c <= i) S[i][c] -= S[i][j] * S[c][j];
    }
    __syncthreads();
  }
  for (int t = tid; t < b * b; t += blockDim.x) {
    const int i = t / b, c = t % b;
    A[(int64_t)(j0 + i) * lda + j0 + c] = c <= i ? S[i][c] : 0.0;
  }
  if (tid == 0 && bad && *info == 0) *info = j0 + bad;
}

// Panel below the diagonal block: L21 = A21 L11^-T, one row per thread
// (forward substitution against the diagonal block held in shared memory).
__global__ void __launch_bounds__(128) k_chol_panel(double* A, int lda, int j0, int b, int n) {
  __shared__ double L[CB][CB + 1];
  for (int t = threadIdx.x; t < b * b; t += blockDim.x) L[t / b][t % b] = A[(int64_t)(j0 + t / b) * lda + j0 + t % b];
  __syncthreads();
  const int r = j0 + b + blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= n) return;
  double x[CB];
  double* row = A + (int64_t)r * lda + j0;
#pragma unroll 4
  for (int k = 0; k < b; ++k) {
    double v = row[k];
    for (int i = 0; i < k; ++i) v -= x[i] * L[k][i];
    x[k] = v / L[k][k];
  }
  for (int k = 0; k < b; ++k) row[k] = x[k];
}

// A22 -= L21 L21^T, lower triangle: every entry takes the panel's products one after the other
// in column order, as the one-CTA factor does (k_chol; the diagonal and panel kernels above
// keep that order too), so that both give the same bits.  64 x 64 tiles, 4 x 4 a thread; the
// panel's 64 terms a tile bound it (FP64 pipe: 70 us a tile, and the last tiles run alone).  The
// whole factor of 640 rows: one CTA 28 ms, with this update 2.8, with tiled products (another order)
// 2.4; of 135 rows 0.39, 0.62, 0.51.
__global__ void __launch_bounds__(256) k_chol_update(double* A, int lda, int j0, int b, int n) {
  if (blockIdx.x > blockIdx.y) return;
  __shared__ double Pr[64][33], Pc[64][33];
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16, o = j0 + b;
  const int i0 = o + blockIdx.y * 64, c0 = o + blockIdx.x * 64;
  double v[4][4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int i = i0 + ty + 16 * u, c = c0 + tx + 16 * w;
      v[u][w] = i < n && c <= i ? A[(int64_t)i * lda + c] : 0.0;
    }
  for (int k0 = 0; k0 < b; k0 += 32) {
    __syncthreads();
    for (int t = tid; t < 64 * 32; t += 256) {
      const int r = t / 32, k = t % 32;
      const bool in = k0 + k < b;
      Pr[r][k] = in && i0 + r < n ? A[(int64_t)(i0 + r) * lda + j0 + k0 + k] : 0.0;
      Pc[r][k] = in && c0 + r < n ? A[(int64_t)(c0 + r) * lda + j0 + k0 + k] : 0.0;
    }
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < 32; ++k) {
      double p[4], q[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        p[u] = Pr[ty + 16 * u][k];
        q[u] = Pc[tx + 16 * u][k];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int w = 0; w < 4; ++w) v[u][w] = fma(-p[u], q[w], v[u][w]);
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const int i = i0 + ty + 16 * u, c = c0 + tx + 16 * w;
      if (i < n && c <= i) A[(int64_t)i * lda + c] = v[u][w];
    }
}

// T (b x m, ld m) = transpose of the panel rows j0+b .. n-1, columns j0 .. j0+b-1
__global__ void k_panel_transpose(const double* A, int lda, int j0, int b, int n, double* T) {
  const int m = n - j0 - b;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= (int64_t)m * b) return;
  const int r = (int)(t / b), c = (int)(t % b);
  T[(int64_t)c * m + r] = A[(int64_t)(j0 + b + r) * lda + j0 + c];
}

__global__ void k_zero_upper(double* A, int n, int lda) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= (int64_t)n * n) return;
  const int i = (int)(t / n), c = (int)(t % n);
  if (c > i) A[(int64_t)i * lda + c] = 0.0;
}

__global__ void k_copy_diag(const double* A, int n, int lda, double* d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) d[i] = A[(int64_t)i * lda + i];
}

// min_j L_jj^2 / d0_j (one CTA): the smallest fraction of a column's squared
// norm outside the span of the columns before it
__global__ void k_chol_ratio(const double* L, int n, int lda, const double* d0, const int* info, double* out) {
  __shared__ double red[1024];
  double m = 1.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double l = L[(int64_t)i * lda + i];
    m = fmin(m, l * l / d0[i]);
  }
  red[threadIdx.x] = m;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] = fmin(red[threadIdx.x], red[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = *info ? 0.0 : red[0];
}

// Li = L^-1 for n <= 64 in one CTA: row k of the inverse is final after k steps (one
// scaling by 1 / L_kk), then every row below takes its multiple of it.  A column per
// thread by forward substitution is a serial chain of n^2 / 2 dependent FMAs (400 us
// at n = 128, 517 us at 135); this takes 50 us at n = 64.  L keeps the lower triangle of the shared array, the
// inverse (transposed) the upper one, a column to the right.
__global__ void __launch_bounds__(512) k_trinv_leaf(const double* __restrict__ L, int n, int lda,
                                                    double* __restrict__ Li, int ldi) {
  __shared__ double S[CB][CB + 2];   // L[i][j] at (i, j), inverse[i][j] at (j, i + 1)
  const int tid = threadIdx.x;
  for (int t = tid; t < n * n; t += 512) {
    const int i = t / n, j = t % n;
    if (j <= i) {
      S[i][j] = L[(int64_t)i * lda + j];
      S[j][i + 1] = i == j ? 1.0 : 0.0;
    }
  }
  __syncthreads();
  for (int k = 0; k < n; ++k) {
    if (tid <= k) S[tid][k + 1] /= S[k][k];
    __syncthreads();
    const int w = k + 1;
    for (int t = tid; t < (n - 1 - k) * w; t += 512) {
      const int i = k + 1 + t / w, j = t % w;
      S[j][i + 1] = fma(-S[i][k], S[j][k + 1], S[j][i + 1]);
    }
    __syncthreads();
  }
  for (int t = tid; t < n * n; t += 512) {
    const int i = t / n, j = t % n;
    Li[(int64_t)i * ldi + j] = j <= i ? S[j][i + 1] : 0.0;
  }
}

__global__ void k_zero_block(double* A, int rows, int cols, int lda) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= (int64_t)rows * cols) return;
  A[(t / cols) * lda + t % cols] = 0.0;
}

// ---------------------------------------------------------------- block Jacobi
// Position of block slot s in round r of the round-robin tournament over nb
// blocks (slot 0 fixed, the others rotate).
__device__ __forceinline__ int rr_block(int s, int r, int nb) { return s == 0 ? 0 : ((s - 1 + r) % (nb - 1)) + 1; }

__device__ __forceinline__ void bj_pair(int k, int r, int nb, int& p, int& q) {
  const int a = rr_block(k, r, nb), b = rr_block(nb - 1 - k, r, nb);
  p = min(a, b);
  q = max(a, b);
}

template <int BJ_B>
__device__ __forceinline__ int bj_index(int i, int p, int q) { return i < BJ_B ? p * BJ_B + i : q * BJ_B + (i - BJ_B); }

template <typename T>
__global__ void k_bj_pad(const double* __restrict__ C, int n, int ldc, T* __restrict__ A, T* __restrict__ V, int np) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= (int64_t)np * np) return;
  const int i = (int)(t / np), j = (int)(t % np);
  A[t] = (i < n && j < n) ? (T)C[(int64_t)i * ldc + j] : T(0);
  V[t] = i == j ? T(1) : T(0);
}

// Rotation of the pair (i, j) that (nearly) annihilates aij: FP32 in the float
// stage; in the double stage the tangent comes from FP32 arithmetic and only
// c = (1 + t^2)^-1/2 is refined to FP64 (an FP32 seed and two Newton steps), so the
// rotation is orthogonal to FP64 rounding and leaves about 1e-7 of aij.  An exact
// FP64 tangent costs two divisions and two square roots, about 100 instructions at
// 64 clocks each in one warp: more than all the rotations of the round.
__device__ __forceinline__ void bj_angle(float aii, float ajj, float aij, float& c, float& s) {
  const float tau = (ajj - aii) / (2.f * aij);
  const float t = (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
  c = 1.f / sqrtf(1.f + t * t);
  s = t * c;
}
__device__ __forceinline__ void bj_angle(double aii, double ajj, double aij, double& c, double& s) {
  // both scaled by one power of two into the FP32 range
  const double d = ajj - aii;
  const int ex = (__double2hiint(fmax(fabs(d), fabs(aij))) >> 20) & 0x7FF;
  const double sc = __hiloint2double((2046 - min(ex, 2045)) << 20, 0);
  const float tau = (float)(d * sc) / (2.f * (float)(aij * sc));
  const float tf = (tau >= 0.f ? 1.f : -1.f) / (fabsf(tau) + sqrtf(1.f + tau * tau));
  const double t = (double)tf;
  const double x = fma(t, t, 1.0);
  double y = (double)rsqrtf((float)x);
  const double hx = 0.5 * x;
  y = y * fma(-hx * y, y, 1.5);
  y = y * fma(-hx * y, y, 1.5);
  c = y;
  s = t * y;
}

// One CTA per block pair of round r: one cyclic Jacobi sweep over the BJ_S x BJ_S
// subproblem [[A_pp, A_pq], [A_qp, A_qq]] in shared memory; writes the rotation J
// (BJ_S x BJ_S, row-major), the rotated subproblem and whether any rotation was
// applied.  One sweep a visit: the outer sweeps come back to the pair anyway, and
// diagonalising it on every visit takes three to eight sweeps on one SM (timed at 640
// rows, a round 100 us in FP32 and 237 in FP64; this 25, as at 135 rows, and 84, with as
// many outer sweeps).  The whole eigenproblem, diagonalising visits -> this: 135 rows 13.0 ->
// 5.1 ms, 300 30.6 -> 11.7, 512 56 -> 23.
// The two-sided rotation of the pairs (e, f) acts on a 2 x 2 block of S: a thread
// per block with e <= f (S is symmetric, the mirrored block is copied).
template <typename T, int BJ_B>
__global__ void __launch_bounds__(256) k_bj_solve(const T* __restrict__ A, int np, int nb, int r, T* __restrict__ Jb,
                                                  T* __restrict__ Sb, int* __restrict__ rotated) {
  constexpr int BJ_S = 2 * BJ_B, BJ_LD = BJ_S + 1;
  constexpr int NBLK = BJ_B * (BJ_B + 1) / 2;
  __shared__ T S[BJ_S * BJ_LD];
  __shared__ T J[BJ_S * BJ_LD];
  __shared__ T cs[BJ_B], sn[BJ_B];
  __shared__ int pp[BJ_B], qq[BJ_B];
  __shared__ int any;
  const int k = blockIdx.x, tid = threadIdx.x;
  int p, q;
  bj_pair(k, r, nb, p, q);
  for (int t = tid; t < BJ_S * BJ_S; t += blockDim.x) {
    const int i = t / BJ_S, j = t % BJ_S;
    S[i * BJ_LD + j] = A[(int64_t)bj_index<BJ_B>(i, p, q) * np + bj_index<BJ_B>(j, p, q)];
    J[i * BJ_LD + j] = i == j ? T(1) : T(0);
  }
  if (tid == 0) any = 0;
  // this thread's 2 x 2 block of pairs (e, f), e <= f
  int be = 0, bf = 0;
  if (tid < NBLK) {
    int t = tid;
    while (t >= BJ_B - be) {
      t -= BJ_B - be;
      ++be;
    }
    bf = be + t;
  }
  __syncthreads();
  for (int rd = 0; rd < BJ_S - 1; ++rd) {
    if (tid < BJ_B) {
      const int a = tid == 0 ? 0 : ((tid - 1 + rd) % (BJ_S - 1)) + 1;
      const int b2 = ((BJ_S - 1 - tid - 1 + rd) % (BJ_S - 1)) + 1;
      const int i = min(a, b2), j = max(a, b2);
      const T aij = S[i * BJ_LD + j], aii = S[i * BJ_LD + i], ajj = S[j * BJ_LD + j];
      T c = T(1), s = T(0);
      // negligible off-diagonal entry (below the rounding of both diagonal
      // entries): no rotation
      const T g = T(100) * fabs(aij);
      if (aij != T(0) && !(fabs(aii) + g == fabs(aii) && fabs(ajj) + g == fabs(ajj))) {
        bj_angle(aii, ajj, aij, c, s);
        any = 1;
      }
      pp[tid] = i;
      qq[tid] = j;
      cs[tid] = c;
      sn[tid] = s;
    }
    __syncthreads();
    if (tid < NBLK) {
      const T ce = cs[be], se = sn[be], cf = cs[bf], sf = sn[bf];
      if (se != T(0) || sf != T(0)) {
        const int i = pp[be], j = qq[be], u = pp[bf], v = qq[bf];
        const T x00 = S[i * BJ_LD + u], x01 = S[i * BJ_LD + v], x10 = S[j * BJ_LD + u], x11 = S[j * BJ_LD + v];
        // rows by (ce, se), then columns by (cf, sf)
        const T y00 = ce * x00 - se * x10, y01 = ce * x01 - se * x11;
        const T y10 = se * x00 + ce * x10, y11 = se * x01 + ce * x11;
        const T z00 = cf * y00 - sf * y01, z01 = sf * y00 + cf * y01;
        const T z10 = cf * y10 - sf * y11, z11 = sf * y10 + cf * y11;
        S[i * BJ_LD + u] = z00;
        S[i * BJ_LD + v] = z01;
        S[j * BJ_LD + v] = z11;
        S[u * BJ_LD + i] = z00;
        S[v * BJ_LD + i] = z01;
        S[v * BJ_LD + j] = z11;
        if (be != bf) {
          S[j * BJ_LD + u] = z10;
          S[u * BJ_LD + j] = z10;
        } else {
          S[j * BJ_LD + u] = z01;   // the pair's own block stays symmetric
        }
      }
    }
    for (int t = tid; t < BJ_B * BJ_S; t += blockDim.x) {
      const int e = t / BJ_S, row = t % BJ_S;
      if (sn[e] == T(0)) continue;
      const int i = pp[e], j = qq[e];
      const T c = cs[e], s = sn[e];
      const T u = J[row * BJ_LD + i], v = J[row * BJ_LD + j];
      J[row * BJ_LD + i] = c * u - s * v;
      J[row * BJ_LD + j] = s * u + c * v;
    }
    __syncthreads();
  }
  T* Jo = Jb + (int64_t)k * BJ_S * BJ_S;
  T* So = Sb + (int64_t)k * BJ_S * BJ_S;
  for (int t = tid; t < BJ_S * BJ_S; t += blockDim.x) {
    Jo[t] = J[(t / BJ_S) * BJ_LD + t % BJ_S];
    So[t] = S[(t / BJ_S) * BJ_LD + t % BJ_S];
  }
  if (tid == 0) rotated[k] = any;
}

// One round's updates in one launch.  blockIdx.x < pairs: the block (k, l) of A,
// k <= l, of the pairs' 2B rows and columns becomes J_k^T A_kl J_l (the diagonal
// one is the solved subproblem), its mirror image the transpose.  blockIdx.x >=
// pairs: 32 rows of V, V[:, idx(k)] <- V[:, idx(k)] J_k.  Blocks are independent,
// so A needs no separate row and column pass (three launches a round and twice the
// products before).  135 rows: 8.7 us in FP32; timed at 640 rows, above its use, 69 us
// in FP64 and 12 in FP32 for 82 and 24.
template <typename T, int BJ_B>
__global__ void __launch_bounds__(256) k_bj_update(T* __restrict__ A, T* __restrict__ V, int np, int nb, int r,
                                                   const T* __restrict__ Jb, const T* __restrict__ Sb,
                                                   const int* __restrict__ rotated) {
  constexpr int BJ_S = 2 * BJ_B, LD = BJ_S + 1;
  __shared__ T Js[BJ_S * LD];
  __shared__ T Xs[BJ_S * LD];
  __shared__ T Ys[BJ_S * LD];
  const int pairs = nb / 2, k = blockIdx.y, tid = threadIdx.x;
  int p, q;
  bj_pair(k, r, nb, p, q);
  // a thread forms four outputs of one row of a BJ_S x BJ_S product
  const int row = tid / (BJ_S / 4), cq = (tid % (BJ_S / 4)) * 4;
  static_assert(BJ_S * (BJ_S / 4) == 256, "256 threads x 4 outputs");
  if ((int)blockIdx.x >= pairs) {
    if (!rotated[k]) return;
    const int r0 = ((int)blockIdx.x - pairs) * BJ_S;
    const T* Jk = Jb + (int64_t)k * BJ_S * BJ_S;
    for (int t = tid; t < BJ_S * BJ_S; t += 256) {
      const int i = t / BJ_S, j = t % BJ_S;
      Js[i * LD + j] = Jk[t];
      Xs[i * LD + j] = r0 + i < np ? V[(int64_t)(r0 + i) * np + bj_index<BJ_B>(j, p, q)] : T(0);
    }
    __syncthreads();
    T acc[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll 8
    for (int l = 0; l < BJ_S; ++l) {
      const T x = Xs[row * LD + l];
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[c] = fma(x, Js[l * LD + cq + c], acc[c]);
    }
    if (r0 + row < np)
#pragma unroll
      for (int c = 0; c < 4; ++c) V[(int64_t)(r0 + row) * np + bj_index<BJ_B>(cq + c, p, q)] = acc[c];
    return;
  }
  const int l2 = blockIdx.x;
  if (l2 < k || !(rotated[k] | rotated[l2])) return;
  if (l2 == k) {
    const T* So = Sb + (int64_t)k * BJ_S * BJ_S;
    for (int t = tid; t < BJ_S * BJ_S; t += 256)
      A[(int64_t)bj_index<BJ_B>(t / BJ_S, p, q) * np + bj_index<BJ_B>(t % BJ_S, p, q)] = So[t];
    return;
  }
  int u, v;
  bj_pair(l2, r, nb, u, v);
  const T* Jk = Jb + (int64_t)k * BJ_S * BJ_S;
  const T* Jl = Jb + (int64_t)l2 * BJ_S * BJ_S;
  for (int t = tid; t < BJ_S * BJ_S; t += 256) {
    const int i = t / BJ_S, j = t % BJ_S;
    Js[i * LD + j] = Jl[t];
    Xs[i * LD + j] = A[(int64_t)bj_index<BJ_B>(i, p, q) * np + bj_index<BJ_B>(j, u, v)];
  }
  __syncthreads();
  T acc[4] = {T(0), T(0), T(0), T(0)};
#pragma unroll 8
  for (int l = 0; l < BJ_S; ++l) {   // Y = A_kl J_l
    const T x = Xs[row * LD + l];
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] = fma(x, Js[l * LD + cq + c], acc[c]);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) Ys[row * LD + cq + c] = acc[c];
  __syncthreads();
  for (int t = tid; t < BJ_S * BJ_S; t += 256) Js[(t / BJ_S) * LD + t % BJ_S] = Jk[t];
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 4; ++c) acc[c] = T(0);
#pragma unroll 8
  for (int l = 0; l < BJ_S; ++l) {   // Z = J_k^T Y
    const T x = Js[l * LD + row];
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[c] = fma(x, Ys[l * LD + cq + c], acc[c]);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    A[(int64_t)bj_index<BJ_B>(row, p, q) * np + bj_index<BJ_B>(cq + c, u, v)] = acc[c];
    Xs[(cq + c) * LD + row] = acc[c];
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < 4; ++c)
    A[(int64_t)bj_index<BJ_B>(row, u, v) * np + bj_index<BJ_B>(cq + c, p, q)] = Xs[row * LD + cq + c];
}

// Above BJ_DIAG_MIN rows: a visit diagonalises its subproblem, and columns and rows of A follow
// in launches of their own.
// One CTA per block pair of round r: diagonalise the BJ_S x BJ_S subproblem
// [[A_pp, A_pq], [A_qp, A_qq]] in shared memory by cyclic Jacobi; write the
// rotation J (BJ_S x BJ_S, row-major), the subproblem's eigenvalues, and whether
// any rotation was applied.
template <typename T, int BJ_B>
__global__ void __launch_bounds__(256) k_bjd_solve(const T* __restrict__ A, int np, int nb, int r, T* __restrict__ Jb,
                                                  T* __restrict__ lam, int* __restrict__ rotated, int max_sweeps) {
  constexpr int BJ_S = 2 * BJ_B, BJ_LD = BJ_S + 1;
  extern __shared__ double smraw[];
  T* S = reinterpret_cast<T*>(smraw);
  T* J = S + BJ_S * BJ_LD;
  __shared__ T cs[BJ_B], sn[BJ_B];
  __shared__ int pp[BJ_B], qq[BJ_B];
  __shared__ int any, any_sweep;
  const int k = blockIdx.x, tid = threadIdx.x;
  int p, q;
  bj_pair(k, r, nb, p, q);
  for (int t = tid; t < BJ_S * BJ_S; t += blockDim.x) {
    const int i = t / BJ_S, j = t % BJ_S;
    S[i * BJ_LD + j] = A[(int64_t)bj_index<BJ_B>(i, p, q) * np + bj_index<BJ_B>(j, p, q)];
    J[i * BJ_LD + j] = i == j ? T(1) : T(0);
  }
  if (tid == 0) any = 0;
  __syncthreads();
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    if (tid == 0) any_sweep = 0;
    __syncthreads();
    for (int rd = 0; rd < BJ_S - 1; ++rd) {
      if (tid < BJ_B) {
        const int a = tid == 0 ? 0 : ((tid - 1 + rd) % (BJ_S - 1)) + 1;
        const int b2 = ((BJ_S - 1 - tid - 1 + rd) % (BJ_S - 1)) + 1;
        const int i = min(a, b2), j = max(a, b2);
        const T aij = S[i * BJ_LD + j], aii = S[i * BJ_LD + i], ajj = S[j * BJ_LD + j];
        T c = T(1), s = T(0);
        // negligible off-diagonal entry (below the rounding of both diagonal
        // entries): no rotation
        const T g = T(100) * fabs(aij);
        if (aij != T(0) && !(fabs(aii) + g == fabs(aii) && fabs(ajj) + g == fabs(ajj))) {
          const T tau = (ajj - aii) / (T(2) * aij);
          const T t = (tau >= T(0) ? T(1) : T(-1)) / (fabs(tau) + sqrt(T(1) + tau * tau));
          c = T(1) / sqrt(T(1) + t * t);
          s = t * c;
          any_sweep = 1;
        }
        pp[tid] = i;
        qq[tid] = j;
        cs[tid] = c;
        sn[tid] = s;
      }
      __syncthreads();
      // rows i, j of S
      for (int t = tid; t < BJ_B * BJ_S; t += blockDim.x) {
        const int e = t / BJ_S, col = t % BJ_S;
        if (sn[e] == T(0)) continue;
        const int i = pp[e], j = qq[e];
        const T c = cs[e], s = sn[e];
        const T x = S[i * BJ_LD + col], y = S[j * BJ_LD + col];
        S[i * BJ_LD + col] = c * x - s * y;
        S[j * BJ_LD + col] = s * x + c * y;
      }
      __syncthreads();
      // columns i, j of S and of J
      for (int t = tid; t < BJ_B * BJ_S; t += blockDim.x) {
        const int e = t / BJ_S, row = t % BJ_S;
        if (sn[e] == T(0)) continue;
        const int i = pp[e], j = qq[e];
        const T c = cs[e], s = sn[e];
        const T x = S[row * BJ_LD + i], y = S[row * BJ_LD + j];
        S[row * BJ_LD + i] = c * x - s * y;
        S[row * BJ_LD + j] = s * x + c * y;
        const T u = J[row * BJ_LD + i], v = J[row * BJ_LD + j];
        J[row * BJ_LD + i] = c * u - s * v;
        J[row * BJ_LD + j] = s * u + c * v;
      }
      __syncthreads();
      if (tid < BJ_B && sn[tid] != T(0)) {
        S[pp[tid] * BJ_LD + qq[tid]] = T(0);
        S[qq[tid] * BJ_LD + pp[tid]] = T(0);
      }
      __syncthreads();
    }
    if (tid == 0 && any_sweep) any = 1;
    __syncthreads();
    if (!any_sweep) break;
  }
  T* Jo = Jb + (int64_t)k * BJ_S * BJ_S;
  for (int t = tid; t < BJ_S * BJ_S; t += blockDim.x) Jo[t] = J[(t / BJ_S) * BJ_LD + t % BJ_S];
  for (int t = tid; t < BJ_S; t += blockDim.x) lam[(int64_t)k * BJ_S + t] = S[t * BJ_LD + t];
  if (tid == 0) rotated[k] = any;
}

// M[:, idx(p,q)] <- M[:, idx(p,q)] J_k for every pair k (rows in chunks of 32).
template <typename T, int BJ_B>
__global__ void __launch_bounds__(256) k_bjd_cols(T* __restrict__ M, int np, int nb, int r, const T* __restrict__ Jb,
                                                 const int* __restrict__ rotated) {
  constexpr int BJ_S = 2 * BJ_B;
  const int k = blockIdx.y;
  if (!rotated[k]) return;
  __shared__ T Js[BJ_S][BJ_S + 1];
  __shared__ T Xs[32][BJ_S + 1];
  int p, q;
  bj_pair(k, r, nb, p, q);
  const T* Jk = Jb + (int64_t)k * BJ_S * BJ_S;
  for (int t = threadIdx.x; t < BJ_S * BJ_S; t += blockDim.x) Js[t / BJ_S][t % BJ_S] = Jk[t];
  const int r0 = blockIdx.x * 32;
  for (int t = threadIdx.x; t < 32 * BJ_S; t += blockDim.x) {
    const int rr = t / BJ_S, c = t % BJ_S;
    Xs[rr][c] = (r0 + rr < np) ? M[(int64_t)(r0 + rr) * np + bj_index<BJ_B>(c, p, q)] : T(0);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < 32 * BJ_S; t += blockDim.x) {
    const int rr = t / BJ_S, c = t % BJ_S;
    if (r0 + rr >= np) continue;
    T acc = T(0);
#pragma unroll 8
    for (int l = 0; l < BJ_S; ++l) acc = fma(Xs[rr][l], Js[l][c], acc);
    M[(int64_t)(r0 + rr) * np + bj_index<BJ_B>(c, p, q)] = acc;
  }
}

// A[idx(p,q), :] <- J_k^T A[idx(p,q), :] for every pair k (columns in chunks
// of one block); the pair's own BJ_S x BJ_S block becomes diag(lambda_k).
template <typename T, int BJ_B>
__global__ void __launch_bounds__(256) k_bjd_rows(T* __restrict__ A, int np, int nb, int r, const T* __restrict__ Jb,
                                                 const T* __restrict__ lam, const int* __restrict__ rotated) {
  constexpr int BJ_S = 2 * BJ_B;
  const int k = blockIdx.y;
  if (!rotated[k]) return;
  __shared__ T Js[BJ_S][BJ_S + 1];
  __shared__ T Xs[BJ_S][BJ_B + 1];
  int p, q;
  bj_pair(k, r, nb, p, q);
  const int cblk = blockIdx.x, c0 = cblk * BJ_B;
  if (cblk == p || cblk == q) {
    // own block columns: diag(lambda) in rows idx(p,q), columns of this block
    const int off = cblk == p ? 0 : BJ_B;
    for (int t = threadIdx.x; t < BJ_S * BJ_B; t += blockDim.x) {
      const int i = t / BJ_B, c = t % BJ_B;
      A[(int64_t)bj_index<BJ_B>(i, p, q) * np + c0 + c] = (i == off + c) ? lam[(int64_t)k * BJ_S + i] : T(0);
    }
    return;
  }
  const T* Jk = Jb + (int64_t)k * BJ_S * BJ_S;
  for (int t = threadIdx.x; t < BJ_S * BJ_S; t += blockDim.x) Js[t / BJ_S][t % BJ_S] = Jk[t];
  for (int t = threadIdx.x; t < BJ_S * BJ_B; t += blockDim.x) {
    const int i = t / BJ_B, c = t % BJ_B;
    Xs[i][c] = A[(int64_t)bj_index<BJ_B>(i, p, q) * np + c0 + c];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < BJ_S * BJ_B; t += blockDim.x) {
    const int i = t / BJ_B, c = t % BJ_B;
    T acc = T(0);
#pragma unroll 8
    for (int l = 0; l < BJ_S; ++l) acc = fma(Js[l][i], Xs[l][c], acc);
    A[(int64_t)bj_index<BJ_B>(i, p, q) * np + c0 + c] = acc;
  }
}

// partial sums of the squared off-diagonal and total entries of the leading n x n part
template <typename T>
__global__ void k_bj_norms(const T* __restrict__ A, int np, int n, double* __restrict__ part) {
  __shared__ double so[256], st[256];
  double o = 0.0, a = 0.0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < (int64_t)n * n;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(t / n), j = (int)(t % n);
    const double v = (double)A[(int64_t)i * np + j];
    a += v * v;
    if (i != j) o += v * v;
  }
  so[threadIdx.x] = o;
  st[threadIdx.x] = a;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) {
      so[threadIdx.x] += so[threadIdx.x + w];
      st[threadIdx.x] += st[threadIdx.x + w];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = so[0];
    part[2 * blockIdx.x + 1] = st[0];
  }
}

template <typename T>
__global__ void k_bj_out(const T* __restrict__ A, const T* __restrict__ V, int np, int n, T* __restrict__ Vo, int ldv,
                         T* __restrict__ w) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= (int64_t)n * n) return;
  const int i = (int)(t / n), j = (int)(t % n);
  Vo[(int64_t)i * ldv + j] = V[(int64_t)i * np + j];
  if (i == j) w[i] = A[(int64_t)i * np + i];
}

constexpr int BJ_NORM_BLOCKS = 128;

}  // namespace

// ------------------------------------------------------------------ host side
// Up to this size the trailing update adds in the order of sums of the one-CTA factor (k_chol), which
// served it before: close pairs of Ritz vectors turn with the rounding, and so they turn as they
// did.  Above it, where the tiled product always ran, it still does.
constexpr int CHOL_ORDERED_MAX = 2048;

// tiled: the trailing update as a tiled product whatever the size (tests)
void launch_chol_blocked(double* A, int n, int lda, int* info, double* min_ratio, double* scratch,
                         cudaStream_t st, bool tiled) {
  // scratch: n (original diagonal) + CB * n (transposed panel) doubles
  double* d0 = scratch;
  double* T = scratch + n;
  cudaMemsetAsync(info, 0, sizeof(int), st);
  if (min_ratio) {
    k_copy_diag<<<nblk(n, 256), 256, 0, st>>>(A, n, lda, d0);
    g_launches.fetch_add(1, std::memory_order_relaxed);
  }
  for (int j0 = 0; j0 < n; j0 += CB) {
    const int b = std::min(CB, n - j0);
    const int m = n - j0 - b;
    k_chol_diag<<<1, 1024, 0, st>>>(A, lda, j0, b, info);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (m <= 0) break;
    k_chol_panel<<<nblk(m, 128), 128, 0, st>>>(A, lda, j0, b, n);
    if (n <= CHOL_ORDERED_MAX && !tiled) {
      k_chol_update<<<dim3(nblk(m, 64), nblk(m, 64)), 256, 0, st>>>(A, lda, j0, b, n);
      g_launches.fetch_add(2, std::memory_order_relaxed);
      continue;
    }
    k_panel_transpose<<<nblk((int64_t)m * b, 256), 256, 0, st>>>(A, lda, j0, b, n, T);
    g_launches.fetch_add(2, std::memory_order_relaxed);
    // A22 -= L21 L21^T (the whole square; only its lower triangle is used)
    double* A22 = A + (int64_t)(j0 + b) * lda + j0 + b;
    launch_gemm_nn(m, m, b, -1.0, A + (int64_t)(j0 + b) * lda + j0, lda, T, m, 1.0, A22, lda, st);
  }
  k_zero_upper<<<nblk((int64_t)n * n, 256), 256, 0, st>>>(A, n, lda);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  if (min_ratio) {
    k_chol_ratio<<<1, 1024, 0, st>>>(A, n, lda, d0, info, min_ratio);
    g_launches.fetch_add(1, std::memory_order_relaxed);
  }
}

int64_t chol_blocked_scratch(int n) { return (int64_t)n + (int64_t)CB * n; }

// Li = L^-1 (lower, n x n, ld ldi), 2 x 2 block recursion down to 64-wide
// diagonal blocks, which one CTA inverts in shared memory.
// scratch: n * n / 4 doubles (the largest off-diagonal block).
void launch_trinv_blocked(const double* L, int n, int lda, double* Li, int ldi, double* scratch, cudaStream_t st) {
  if (n <= CB) {
    k_trinv_leaf<<<1, 512, 0, st>>>(L, n, lda, Li, ldi);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    return;
  }
  const int n1 = (n / 2 + 63) / 64 * 64, n2 = n - n1;
  launch_trinv_blocked(L, n1, lda, Li, ldi, scratch, st);
  launch_trinv_blocked(L + (int64_t)n1 * lda + n1, n2, lda, Li + (int64_t)n1 * ldi + n1, ldi, scratch, st);
  // Li21 = -Li22 (L21 Li11); T = L21 Li11 is n2 x n1
  launch_gemm_nn(n2, n1, n1, 1.0, L + (int64_t)n1 * lda, lda, Li, ldi, 0.0, scratch, n1, st);
  launch_gemm_nn(n2, n1, n2, -1.0, Li + (int64_t)n1 * ldi + n1, ldi, scratch, n1, 0.0, Li + (int64_t)n1 * ldi, ldi,
                 st);
  k_zero_block<<<nblk((int64_t)n1 * n2, 256), 256, 0, st>>>(Li + n1, n1, n2, ldi);
  g_launches.fetch_add(1, std::memory_order_relaxed);
}

constexpr int BJ_BLOCK = 16;   // block Jacobi block size of both stages

// Above this size a visit of the block Jacobi diagonalises its subproblem instead of making one
// sweep over it.  One sweep a visit is the faster at every size (640 rows: about 95 -> 31 ms) and
// as accurate, but rounds differently, and the vectors of the closest pairs of Ritz values turn
// with the rounding (norm x 2^-53 over the gap: 3.5e-9 seen at 640, as far from a 64-bit result
// either way).  So this is not a line between two fields of use: it is where the visits that
// diagonalise were in use before, and a program that compares such vectors between runs keeps them.
constexpr int BJ_DIAG_MIN = 512;

static int64_t bj_scratch_bytes(int n, int elem, int B) {
  const int S = 2 * B;
  const int nb0 = (n + B - 1) / B;
  const int nb = std::max(2, nb0 + (nb0 & 1));
  const int64_t np = (int64_t)nb * B;
  const int64_t pairs = nb / 2;
  return elem * (2 * np * np + 2 * pairs * S * S) + (int64_t)sizeof(int) * pairs +
         (int64_t)sizeof(double) * 2 * BJ_NORM_BLOCKS + 1024;
}

int64_t block_jacobi_scratch_bytes(int n, int elem) { return bj_scratch_bytes(n, elem, BJ_BLOCK); }

// Symmetric C (n x n, FP64, ldc) = V diag(w) V^T by block Jacobi in precision T.
// Sweeps until the off-diagonal square sum is <= tol2 times the total or
// max_sweeps; returns 0 on convergence, 1 if the sweeps ran out, -1 on a CUDA
// error.  The only host synchronisation is the norm check after each sweep.
namespace {
template <typename T, int BJ_B>
int block_jacobi_b(const double* C, int n, int ldc, T* V, int ldv, T* w, int max_sweeps, double tol2, void* scratch,
                   cudaStream_t st, double* ratio_out, bool diag) {
  constexpr int BJ_S = 2 * BJ_B;
  const int nb0 = (n + BJ_B - 1) / BJ_B;
  const int nb = std::max(2, nb0 + (nb0 & 1));
  const int np = nb * BJ_B;
  const int pairs = nb / 2;
  const size_t smem = sizeof(T) * 2 * BJ_S * (BJ_S + 1);
  if (diag && cudaFuncSetAttribute(k_bjd_solve<T, BJ_B>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
                  cudaSuccess)
    return -1;
  T* A = reinterpret_cast<T*>(scratch);
  T* Vp = A + (int64_t)np * np;
  T* Jb = Vp + (int64_t)np * np;
  T* Sb = Jb + (int64_t)pairs * BJ_S * BJ_S;
  int* rot = reinterpret_cast<int*>(Sb + (int64_t)pairs * BJ_S * BJ_S);
  double* part = reinterpret_cast<double*>(((uintptr_t)(rot + pairs) + 255) & ~(uintptr_t)255);
  k_bj_pad<T><<<nblk((int64_t)np * np, 256), 256, 0, st>>>(C, n, ldc, A, Vp, np);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  std::vector<double> hp(2 * BJ_NORM_BLOCKS);
  int rc = 1;
  for (int sweep = 0; sweep <= max_sweeps; ++sweep) {
    k_bj_norms<T><<<BJ_NORM_BLOCKS, 256, 0, st>>>(A, np, n, part);
    g_launches.fetch_add(1, std::memory_order_relaxed);
    if (cudaMemcpyAsync(hp.data(), part, sizeof(double) * hp.size(), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
      return -1;
    double off = 0.0, tot = 0.0;
    for (int b = 0; b < BJ_NORM_BLOCKS; ++b) {
      off += hp[2 * b];
      tot += hp[2 * b + 1];
    }
    if (ratio_out) *ratio_out = tot > 0.0 ? off / tot : 0.0;
    if (off <= tol2 * tot) {
      rc = 0;
      break;
    }
    if (sweep == max_sweeps) break;
    for (int r = 0; r < nb - 1 && diag; ++r) {
      k_bjd_solve<T, BJ_B><<<pairs, 256, smem, st>>>(A, np, nb, r, Jb, Sb, rot, 30);
      k_bjd_cols<T, BJ_B><<<dim3(nblk(np, 32), pairs), 256, 0, st>>>(A, np, nb, r, Jb, rot);
      k_bjd_rows<T, BJ_B><<<dim3(nb, pairs), 256, 0, st>>>(A, np, nb, r, Jb, Sb, rot);
      k_bjd_cols<T, BJ_B><<<dim3(nblk(np, 32), pairs), 256, 0, st>>>(Vp, np, nb, r, Jb, rot);
      g_launches.fetch_add(4, std::memory_order_relaxed);
    }
    for (int r = 0; r < nb - 1 && !diag; ++r) {
      k_bj_solve<T, BJ_B><<<pairs, 256, 0, st>>>(A, np, nb, r, Jb, Sb, rot);
      k_bj_update<T, BJ_B><<<dim3((unsigned)pairs + nblk(np, BJ_S), pairs), 256, 0, st>>>(A, Vp, np, nb, r, Jb, Sb, rot);
      g_launches.fetch_add(2, std::memory_order_relaxed);
    }
  }
  k_bj_out<T><<<nblk((int64_t)n * n, 256), 256, 0, st>>>(A, Vp, np, n, V, ldv, w);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  if (cudaGetLastError() != cudaSuccess) return -1;
  return rc;
}
}  // namespace

// Both stages in 16-wide blocks: the subproblem solves run on one SM each (the
// FP64 ones at that SM's FP64 rate), so halving the block halves the solve work
// per sweep at the same update flops (measured: 280-atom Rayleigh-Ritz 5.41 s with
// 32-wide blocks, 4.95 s with 16)
template <typename T>
int block_jacobi(const double* C, int n, int ldc, T* V, int ldv, T* w, int max_sweeps, double tol2, void* scratch,
                 cudaStream_t st, double* ratio_out, bool diagonalise) {
  return block_jacobi_b<T, BJ_BLOCK>(C, n, ldc, V, ldv, w, max_sweeps, tol2, scratch, st, ratio_out,
                                     diagonalise || n > BJ_DIAG_MIN);
}

template int block_jacobi<float>(const double*, int, int, float*, int, float*, int, double, void*, cudaStream_t,
                                 double*, bool);
template int block_jacobi<double>(const double*, int, int, double*, int, double*, int, double, void*, cudaStream_t,
                                  double*, bool);

}  // namespace efe
