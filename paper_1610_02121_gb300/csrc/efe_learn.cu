// Learned initial density for the SCF (Sec. V starts from an input density):
//   * superposition of atomic densities (SAD) from normalised Slater shells,
//   * atom-centred descriptors at the quadrature points (radial Gaussians and
//     angular dipole magnitudes per species slot, smooth cosine cutoff),
//   * a fully connected network (SiLU hidden layers) with forward and backward
//     passes written as tiled GEMMs, a weighted squared-error loss and Adam,
//   * the corrected start rho = (rho_sad + floor) exp(y) - floor, rescaled.
// Every kernel is templated on the arithmetic type: float for training and
// inference, double for the gradient checks against the oracle.  All
// reductions use fixed-order partials (bitwise reproducible).
#include <math.h>

#include <type_traits>

#include <cmath>

#include "efe_kernels.h"

namespace efe {

namespace {

inline unsigned nblk(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

constexpr int RED_B = 512;  // blocks of the fixed-order reductions

template <typename T>
__device__ __forceinline__ T silu_d(T z) { return z / (T(1) + exp(-z)); }
template <typename T>
__device__ __forceinline__ T silu_grad_d(T z) {
  const T s = T(1) / (T(1) + exp(-z));
  return s * (T(1) + z * (T(1) - s));
}

// ---------------------------------------------------------------------------
// SAD: rho(x) = sum_I sum_s N_s C_s^2 r^(2 n_s - 2) exp(-2 zeta_s r) / (4 pi)
//
// The FP64 pipe bounds it (an exponential per point, atom and shell), so a point starts with
// its nearest atom and takes a further shell only if FP32 arithmetic finds it above 2^-58 of
// the sum so far (FP32 distances are off by about 1e-6 here, far less than a factor of two
// in a term).  Added to that sum in FP64 a shell below 2^-54 of it would leave it as it is, so
// however many shells fall out, the result is the one of adding them all in this order.  Most
// inner shells of most atoms do: 3.84 M points, 16 atoms of three shells 9.2 -> 5.6 ms.
constexpr int SAD_TILE = 32;     // atoms whose shells wait in shared memory

struct SadShell {
  double w, z2;    // N C^2, 2 zeta
  float lw, z2f;   // log2 of w (and one more, for the FP32 rounding), 2 zeta log2(e)
  int p;           // 2 n - 2
};

__device__ __forceinline__ SadShell sad_shell(const SadShellDev& S, int k) {
  SadShell o;
  o.w = S.occ[k] * S.c[k] * S.c[k];
  o.z2 = 2.0 * S.zeta[k];
  int e;   // w itself may lie outside FP32's range
  const double m = frexp(fabs(o.w), &e);
  o.lw = log2f((float)m) + (float)e + 1.f;
  o.z2f = (float)(o.z2 * 1.4426950408889634);
  o.p = max(0, 2 * S.n[k] - 2);
  return o;
}

__device__ __forceinline__ double sad_term(const SadShell& S, double r) {
  double rp = S.w;
  for (int i = 0; i < S.p; ++i) rp *= r;
  return rp * exp(-S.z2 * r);
}

__global__ void __launch_bounds__(256) k_sad(const double* __restrict__ qpts, int64_t nq,
                                             const double* __restrict__ axyz, int na,
                                             const SadShellDev* __restrict__ sh, double* __restrict__ rho) {
  __shared__ double ax[SAD_TILE][3];
  __shared__ SadShell ss[SAD_TILE][3];
  __shared__ int cnt[SAD_TILE];
  const int64_t q = blockIdx.x * 256LL + threadIdx.x;
  const int64_t qc = min(q, nq - 1);
  const double x = qpts[4 * qc], y = qpts[4 * qc + 1], z = qpts[4 * qc + 2];
  auto dist2 = [&](const double* c) {
    const float dx = (float)(x - c[0]), dy = (float)(y - c[1]), dz = (float)(z - c[2]);
    return dx * dx + dy * dy + dz * dz;
  };
  int near = 0;
  float best = INFINITY;
  for (int a = 0; a < na; ++a) {
    const float d = dist2(axyz + 3 * a);
    if (d < best) {
      best = d;
      near = a;
    }
  }
  auto dist = [&](const double* c) {
    const double dx = x - c[0], dy = y - c[1], dz = z - c[2];
    return sqrt(dx * dx + dy * dy + dz * dz);
  };
  double s = 0.0;
  if (na > 0) {
    const SadShellDev& S = sh[near];
    const double r = dist(axyz + 3 * near);
    for (int k = S.n_shells - 1; k >= 0; --k) s += sad_term(sad_shell(S, k), r);
  }
  for (int a0 = 0; a0 < na; a0 += SAD_TILE) {
    const int nt = min(SAD_TILE, na - a0);
    __syncthreads();
    if ((int)threadIdx.x < nt) {
      const int a = a0 + threadIdx.x;
      for (int d = 0; d < 3; ++d) ax[threadIdx.x][d] = axyz[3 * a + d];
      cnt[threadIdx.x] = sh[a].n_shells;
      for (int k = 0; k < sh[a].n_shells; ++k) ss[threadIdx.x][k] = sad_shell(sh[a], k);
    }
    __syncthreads();
    for (int i = 0; i < nt; ++i) {
      if (a0 + i == near) continue;
      const float rf = sqrtf(dist2(ax[i]));
      const float lr = log2f(rf);
      double r = -1.0;
      for (int k = cnt[i] - 1; k >= 0; --k) {
        const SadShell& S = ss[i][k];
        // s >= 2^ls (its exponent; zero and subnormal: all terms count)
        const int ls = ((__double2hiint(s) >> 20) & 0x7FF) - 1023;
        const float lt = S.lw + (S.p ? (float)S.p * lr : 0.f) - S.z2f * rf;
        if (lt < (float)(ls - 58)) continue;
        if (r < 0.0) r = dist(ax[i]);
        s += sad_term(S, r);
      }
    }
  }
  if (q < nq) rho[q] = s * 0.079577471545947667884;  // 1 / (4 pi)
}

// ---------------------------------------------------------------------------
// descriptors: per point, per species slot s: radial G[s][k], angular A[s][k]
//
// The FP64 pipe bounds it (an exponential per point, atom and Gaussian).  One thread per
// point takes the species one after the other, so that the sums of a species stay in
// registers (the order of each sum is the atoms' order), and leaves out what it can:
//   * the division by 2 sigma^2 is a product with its rounded reciprocal and one correction
//     of the quotient by the exact remainder (Markstein, IBM J. Res. Dev. 34, 1990: the
//     correctly rounded quotient, so the division's own bits), where c and 1 / c are normal;
//   * an FP32 radial term below 2^-27 of its sum (or of the smallest FP32 number) cannot
//     change the sum; FP32 arithmetic finds these before the exponential is taken.
// The rows go out through shared memory, 128 points at a time.  3.84 M points, 16 atoms, 64
// FP32 features: 20.6 -> 16.1 ms.
struct DescInv {
  double c[2], rc[2];   // 2 sigma^2 of the radial and angular Gaussians; 1 / c, or 0: divide
  float g;              // -log2(e) / (2 sigma^2), radial
};

__device__ __forceinline__ double div_by(double x, double c, double rc) {
  if (rc == 0.0) return x / c;
  const double q = x * rc;
  return fma(fma(-q, c, x), rc, q);
}

constexpr int DESC_PTS = 128;

template <typename T>
__global__ void __launch_bounds__(DESC_PTS) k_descriptors(const double* __restrict__ qpts, int64_t nq,
                                                          const double* __restrict__ axyz,
                                                          const int32_t* __restrict__ slot, int na, DescDev p,
                                                          DescInv v, T* __restrict__ D) {
  extern __shared__ __align__(16) unsigned char smd[];
  const int nr = p.n_radial, nang = p.n_ang, ns = p.n_species;
  const int nf = ns * (nr + nang);
  T* rows = reinterpret_cast<T*>(smd);        // DESC_PTS x (nf + 1)
  const int64_t q0 = blockIdx.x * (int64_t)DESC_PTS;
  const int64_t q = min(q0 + threadIdx.x, nq - 1);
  const double x = qpts[4 * q], y = qpts[4 * q + 1], z = qpts[4 * q + 2];
  constexpr double PI = 3.14159265358979323846;
  T* out = rows + threadIdx.x * (nf + 1);
  for (int s = 0; s < ns; ++s) {
    T rad[DESC_MAX_RADIAL];
    double av[DESC_MAX_ANG][3];
#pragma unroll
    for (int k = 0; k < DESC_MAX_RADIAL; ++k) rad[k] = T(0);
#pragma unroll
    for (int k = 0; k < DESC_MAX_ANG; ++k) av[k][0] = av[k][1] = av[k][2] = 0.0;
    for (int a = 0; a < na; ++a) {
      if (slot[a] != s) continue;
      const double dx = x - axyz[3 * a], dy = y - axyz[3 * a + 1], dz = z - axyz[3 * a + 2];
      const double r = sqrt(dx * dx + dy * dy + dz * dz);
      if (!(r < p.r_cut)) continue;
      const double fc = 0.5 * (1.0 + cos(PI * r / p.r_cut));
#pragma unroll
      for (int k = 0; k < DESC_MAX_RADIAL; ++k) {
        if (k >= nr) break;
        const double t = r - p.radial_mu[k];
        if (sizeof(T) == 4) {
          const float tf = (float)t;
          const int e = rad[k] > T(0) ? ((__float_as_int((float)rad[k]) >> 23) & 0xFF) - 127 : -124;
          if (tf * tf * v.g < (float)(e - 27)) continue;
        }
        rad[k] += (T)(exp(div_by(-t * t, v.c[0], v.rc[0])) * fc);
      }
      const double ir = 1.0 / fmax(r, 1e-12);
#pragma unroll
      for (int k = 0; k < DESC_MAX_ANG; ++k) {
        if (k >= nang) break;
        const double t = r - p.ang_mu[k];
        const double g = exp(div_by(-t * t, v.c[1], v.rc[1])) * fc * ir;
        av[k][0] += g * dx;
        av[k][1] += g * dy;
        av[k][2] += g * dz;
      }
    }
#pragma unroll
    for (int k = 0; k < DESC_MAX_RADIAL; ++k)
      if (k < nr) out[s * nr + k] = rad[k];
#pragma unroll
    for (int k = 0; k < DESC_MAX_ANG; ++k)
      if (k < nang) out[ns * nr + s * nang + k] = (T)(av[k][0] * av[k][0] + av[k][1] * av[k][1] + av[k][2] * av[k][2]);
  }
  if (p.standardise)
    for (int f = 0; f < nf; ++f) out[f] = (T)(((double)out[f] - p.offset[f]) * p.scale[f]);
  __syncthreads();
  const int64_t tot = min((int64_t)DESC_PTS, nq - q0) * nf;
  for (int i = threadIdx.x; i < tot; i += DESC_PTS) D[q0 * nf + i] = rows[i / nf * (nf + 1) + i % nf];
}

// ---------------------------------------------------------------------------
// Generic tiled GEMM: C[z][m][n] = sum_{k in chunk z} A(m, k) B(k, n), element
// (m, k) of A at A[m * sam + k * sak] and (k, n) of B at B[k * sbk + n * sbn];
// one 64 x 64 output tile per CTA (256 threads, 4 x 4 each), K chunk of kch
// per blockIdx.z (split-K partials for the long reductions of the backward pass).
constexpr int GM = 64, GK = 16;

template <typename T>
__global__ void __launch_bounds__(256) k_gemm_g(int64_t M, int64_t Nn, int64_t K, int64_t kch, const T* __restrict__ A,
                                                int64_t sam, int64_t sak, const T* __restrict__ B, int64_t sbk,
                                                int64_t sbn, T* __restrict__ C, int64_t ldc) {
  __shared__ T As[GK][GM + 1];
  __shared__ T Bs[GK][GM + 1];
  const int64_t m0 = (int64_t)blockIdx.x * GM, n0 = (int64_t)blockIdx.y * GM;
  const int64_t kb = (int64_t)blockIdx.z * kch, ke = min(K, kb + kch);
  C += (int64_t)blockIdx.z * M * ldc;
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
  const bool a_kfast = sak == 1;
  const bool b_nfast = sbn == 1;
  for (int64_t k0 = kb; k0 < ke; k0 += GK) {
    for (int idx = tid; idx < GK * GM; idx += 256) {
      int kk, mm;
      if (a_kfast) { kk = idx % GK; mm = idx / GK; } else { mm = idx % GM; kk = idx / GM; }
      const int64_t gm = m0 + mm, gk = k0 + kk;
      As[kk][mm] = (gm < M && gk < ke) ? A[gm * sam + gk * sak] : T(0);
      int kk2, nn;
      if (b_nfast) { nn = idx % GM; kk2 = idx / GM; } else { kk2 = idx % GK; nn = idx / GK; }
      const int64_t gn = n0 + nn, gk2 = k0 + kk2;
      Bs[kk2][nn] = (gn < Nn && gk2 < ke) ? B[gk2 * sbk + gn * sbn] : T(0);
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      T a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int64_t m = m0 + ty * 4 + i;
    if (m >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int64_t n = n0 + tx * 4 + j;
      if (n < Nn) C[m * ldc + n] = acc[i][j];
    }
  }
}

// FP32 GEMM of the network's layers: C[m][n] = sum_k A(m, k) B(k, n), FP32 FMAs in k
// order (split K: blockIdx.z takes kch of them, partial products at C + z M ldc).  A
// CTA forms a 128 x 128 tile, a thread 8 x 8 of it (two 4-wide groups per axis, so the
// shared rows are read as 16-byte vectors), K in steps of 16 through two buffers: the
// next step's global loads are in registers while this one is multiplied.  The FP32
// pipe bounds it: 64 FMAs, as 32 two-wide instructions, for four 16-byte shared loads
// a thread and k.  3.84M rows through 64 -> 256 -> 256 -> 256: 63 ms in 64 x 64 tiles
// of 4 x 4 outputs with scalar loads and separate bias/SiLU passes, 27.8 with this tile
// and one-wide FMAs, 23.0 (49 TFLOP/s) with two-wide ones; same bits.
// AK: element (m, k) of A is A[m lda + k], else A[k lda + m]; BK: (k, n) of B is
// B[n ldb + k], else B[k ldb + n].  VEC: rows and pointers allow 16-byte loads.
// EPI 0: C = product; 1: C = Z = product + bias[n], act = silu(Z) or Z; 2: C = product *
// silu'(Zp[m][n]).
constexpr int FT = 128, FK = 16;

// two FP32 FMAs (each rounded once) in one instruction: acc += (a, a) * (b0, b1)
__device__ __forceinline__ unsigned long long pack2(float a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ void fma2(unsigned long long& acc, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

template <bool AK, bool BK, bool VEC, int EPI>
__global__ void __launch_bounds__(256, 2) k_gemm_f32(int64_t M, int64_t Nn, int64_t K, int64_t kch,
                                                     const float* __restrict__ A, int64_t lda,
                                                     const float* __restrict__ B, int64_t ldb, float* __restrict__ C,
                                                     int64_t ldc, const float* __restrict__ bias,
                                                     float* __restrict__ act, const float* __restrict__ Zp, int silu) {
  __shared__ __align__(16) float As[2][FK][FT + 4];
  __shared__ __align__(16) float Bs[2][FK][FT + 4];
  const int64_t m0 = (int64_t)blockIdx.x * FT, n0 = (int64_t)blockIdx.y * FT;
  const int64_t kb = (int64_t)blockIdx.z * kch, ke = min(K, kb + kch);
  C += (int64_t)blockIdx.z * M * ldc;
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  float4 ra[2], rb[2];
  // operand tile 128 (rows of the operand's own index) x 16 k: 512 quads, two a thread.
  // KF (k fastest): quad = (row, 4 k); else quad = (k, 4 rows)
  auto load = [&](auto kf, const float* P, int64_t ld, int64_t r0, int64_t R, int64_t k0, float4 (&v)[2]) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int t = tid + 256 * u;
      v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
      float* e = reinterpret_cast<float*>(&v[u]);
      if constexpr (decltype(kf)::value) {
        const int64_t r = r0 + t / 4, k = k0 + (t % 4) * 4;
        if (r < R) {
          if (VEC && k + 4 <= ke) {
            v[u] = *reinterpret_cast<const float4*>(P + r * ld + k);
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (k + i < ke) e[i] = P[r * ld + k + i];
          }
        }
      } else {
        const int64_t k = k0 + t / 32, r = r0 + (t % 32) * 4;
        if (k < ke) {
          if (VEC && r + 4 <= R) {
            v[u] = *reinterpret_cast<const float4*>(P + k * ld + r);
          } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (r + i < R) e[i] = P[k * ld + r + i];
          }
        }
      }
    }
  };
  auto store = [&](auto kf, float (*S)[FT + 4], const float4 (&v)[2]) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int t = tid + 256 * u;
      const float* e = reinterpret_cast<const float*>(&v[u]);
      if constexpr (decltype(kf)::value) {
#pragma unroll
        for (int i = 0; i < 4; ++i) S[(t % 4) * 4 + i][t / 4] = e[i];
      } else {
        *reinterpret_cast<float4*>(&S[t / 32][(t % 32) * 4]) = v[u];
      }
    }
  };
  const std::integral_constant<bool, AK> akf{};
  const std::integral_constant<bool, BK> bkf{};
  unsigned long long acc[8][4];   // column pairs (c, c + 1) of a row
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  load(akf, A, lda, m0, M, kb, ra);
  load(bkf, B, ldb, n0, Nn, kb, rb);
  store(akf, As[0], ra);
  store(bkf, Bs[0], rb);
  __syncthreads();
  int b = 0;
  for (int64_t k0 = kb; k0 < ke; k0 += FK, b ^= 1) {
    const bool more = k0 + FK < ke;
    if (more) {
      load(akf, A, lda, m0, M, k0 + FK, ra);
      load(bkf, B, ldb, n0, Nn, k0 + FK, rb);
    }
#pragma unroll
    for (int kk = 0; kk < FK; ++kk) {
      float av[8];
      ulonglong2 b0, b1;
      *reinterpret_cast<float4*>(av) = *reinterpret_cast<const float4*>(&As[b][kk][ty * 4]);
      *reinterpret_cast<float4*>(av + 4) = *reinterpret_cast<const float4*>(&As[b][kk][64 + ty * 4]);
      b0 = *reinterpret_cast<const ulonglong2*>(&Bs[b][kk][tx * 4]);
      b1 = *reinterpret_cast<const ulonglong2*>(&Bs[b][kk][64 + tx * 4]);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const unsigned long long a2 = pack2(av[i]);
        fma2(acc[i][0], a2, b0.x);
        fma2(acc[i][1], a2, b0.y);
        fma2(acc[i][2], a2, b1.x);
        fma2(acc[i][3], a2, b1.y);
      }
    }
    if (more) {
      store(akf, As[b ^ 1], ra);
      store(bkf, Bs[b ^ 1], rb);
    }
    __syncthreads();
  }
  // 16-byte stores where the row is aligned and the four columns exist
  const bool vst = (ldc & 3) == 0 && ((uintptr_t)C & 15) == 0 && (EPI != 1 || ((uintptr_t)act & 15) == 0) &&
                   (EPI != 2 || ((uintptr_t)Zp & 15) == 0);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int64_t m = m0 + (i < 4 ? ty * 4 + i : 64 + ty * 4 + i - 4);
    if (m >= M) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t n = n0 + h * 64 + tx * 4;
      if (n >= Nn) continue;
      float z[4], a4[4];
      const bool v4 = vst && n + 4 <= Nn;
      if (EPI == 2 && v4) *reinterpret_cast<float4*>(a4) = *reinterpret_cast<const float4*>(Zp + m * ldc + n);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        z[j] = __uint_as_float((unsigned)(acc[i][h * 2 + j / 2] >> (32 * (j & 1))));
        if (n + j >= Nn) continue;
        if (EPI == 1) {
          z[j] += bias[n + j];
          a4[j] = silu ? silu_d(z[j]) : z[j];
        }
        if (EPI == 2) z[j] *= silu_grad_d(v4 ? a4[j] : Zp[m * ldc + n + j]);
      }
      if (v4) {
        *reinterpret_cast<float4*>(C + m * ldc + n) = *reinterpret_cast<float4*>(z);
        if (EPI == 1) *reinterpret_cast<float4*>(act + m * ldc + n) = *reinterpret_cast<float4*>(a4);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (n + j >= Nn) continue;
          C[m * ldc + n + j] = z[j];
          if (EPI == 1) act[m * ldc + n + j] = a4[j];
        }
      }
    }
  }
}

// the scalar output layer (one column): z = sum_k a[k] w[k] + b with the sum in k order,
// one thread a row; 256 columns of 32 rows at a time go through shared memory so that
// the loads are coalesced and many.  z goes to the pre-activation, the activation and
// y.  Read-bound (3.9 GB on 3.8M rows of 256); as a 64-column GEMM tile for the one
// column it took a quarter of the network's time.
constexpr int RD_R = 32, RD_C = 256;
__global__ void __launch_bounds__(256) k_row_dot(int64_t n, int d, const float* __restrict__ a,
                                                const float* __restrict__ w, const float* __restrict__ b,
                                                float* __restrict__ Z, float* __restrict__ A, float* __restrict__ y) {
  __shared__ float S[RD_R][RD_C + 1];
  __shared__ float ws[RD_C];
  const int tid = threadIdx.x;
  const int64_t r0 = blockIdx.x * (int64_t)RD_R;
  const int nr = (int)min((int64_t)RD_R, n - r0);
  float s = 0.f;
  for (int k0 = 0; k0 < d; k0 += RD_C) {
    const int nk = min(RD_C, d - k0);
    __syncthreads();
    if (tid < nk) {
      ws[tid] = w[k0 + tid];
      const float* ar = a + r0 * d + k0 + tid;
      if (nr == RD_R) {
#pragma unroll
        for (int r = 0; r < RD_R; ++r) S[r][tid] = ar[(int64_t)r * d];
      } else {
        for (int r = 0; r < nr; ++r) S[r][tid] = ar[(int64_t)r * d];
      }
    }
    __syncthreads();
    if (tid < nr) {
#pragma unroll 8
      for (int k = 0; k < nk; ++k) s = fmaf(S[tid][k], ws[k], s);
    }
  }
  if (tid < nr) {
    const float z = s + b[0];
    Z[r0 + tid] = z;
    A[r0 + tid] = z;
    y[r0 + tid] = z;
  }
}

// Z = C + b (bias per column), A = act(Z) (SiLU or identity); Z, A row-major n x d
template <typename T>
__global__ void k_bias_act(int64_t n, int d, const T* __restrict__ b, T* __restrict__ Z, T* __restrict__ A, int act) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n * d) return;
  const T z = Z[i] + b[i % d];
  Z[i] = z;
  A[i] = act ? silu_d(z) : z;
}

// dZ = dA * silu'(Z)
template <typename T>
__global__ void k_act_back(int64_t n, const T* __restrict__ Z, T* __restrict__ dA) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) dA[i] *= silu_grad_d(Z[i]);
}

// out[i] = sum_z part[z][i] (fixed order), i < nout: 32 outputs a block, eight thread
// rows take every eighth partial and the row sums are added in order
template <typename T>
__global__ void __launch_bounds__(256) k_sum_parts(int nz, int64_t nout, const T* __restrict__ part, T* __restrict__ out) {
  __shared__ T rs[8][33];
  const int x = threadIdx.x & 31, y = threadIdx.x >> 5;
  const int64_t i = blockIdx.x * 32LL + x;
  T s = T(0);
  if (i < nout)
    for (int z = y; z < nz; z += 8) s += part[(int64_t)z * nout + i];
  rs[y][x] = s;
  __syncthreads();
  if (y == 0 && i < nout) {
    T v = T(0);
#pragma unroll
    for (int k = 0; k < 8; ++k) v += rs[k][x];
    out[i] = v;
  }
}

// column sums of dZ (n x d) in fixed order: part[blk][j], then summed
template <typename T>
__global__ void k_colsum_part(int64_t n, int d, const T* __restrict__ dZ, int64_t rows_per_blk, T* __restrict__ part) {
  const int j = threadIdx.x + blockIdx.y * blockDim.x;
  if (j >= d) return;
  const int64_t r0 = blockIdx.x * rows_per_blk, r1 = min(n, r0 + rows_per_blk);
  T s = T(0);
  for (int64_t r = r0; r < r1; ++r) s += dZ[r * d + j];
  part[(int64_t)blockIdx.x * d + j] = s;
}

// weighted squared error: loss = sum c (yh - y)^2 / sum c; dy = 2 c (yh - y) / sum c
template <typename T>
__global__ void __launch_bounds__(256) k_wmse_part(int64_t n, const T* __restrict__ yh, const T* __restrict__ y,
                                                   const T* __restrict__ c, double* __restrict__ part) {
  __shared__ double r1[256], r2[256];
  double a = 0.0, b = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double d = (double)yh[i] - (double)y[i];
    a += (double)c[i] * d * d;
    b += (double)c[i];
  }
  r1[threadIdx.x] = a;
  r2[threadIdx.x] = b;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) {
      r1[threadIdx.x] += r1[threadIdx.x + s];
      r2[threadIdx.x] += r2[threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    part[blockIdx.x] = r1[0];
    part[gridDim.x + blockIdx.x] = r2[0];
  }
}

// fixed-order trees over the block partials (one thread adding 1024 values in turn
// took 58 us; the tree takes 6)
__global__ void __launch_bounds__(RED_B) k_wmse_finish(const double* __restrict__ part, double* __restrict__ out) {
  __shared__ double r1[RED_B], r2[RED_B];
  r1[threadIdx.x] = part[threadIdx.x];
  r2[threadIdx.x] = part[RED_B + threadIdx.x];
  __syncthreads();
  for (int s = RED_B / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) {
      r1[threadIdx.x] += r1[threadIdx.x + s];
      r2[threadIdx.x] += r2[threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = r1[0] / r2[0];
    out[1] = r2[0];
  }
}

template <typename T>
__global__ void k_wmse_grad(int64_t n, const T* __restrict__ yh, const T* __restrict__ y, const T* __restrict__ c,
                            const double* __restrict__ stats, T* __restrict__ dy) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) dy[i] = (T)(2.0 * (double)c[i] * ((double)yh[i] - (double)y[i]) / stats[1]);
}

template <typename T>
__global__ void k_adam(int64_t n, T* __restrict__ p, const T* __restrict__ g, T* __restrict__ m, T* __restrict__ v,
                       double lr, double b1, double b2, double eps, double c1, double c2) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double gi = (double)g[i];
  const double mi = b1 * (double)m[i] + (1.0 - b1) * gi;
  const double vi = b2 * (double)v[i] + (1.0 - b2) * gi * gi;
  m[i] = (T)mi;
  v[i] = (T)vi;
  p[i] = (T)((double)p[i] - lr * (mi / c1) / (sqrt(vi / c2) + eps));
}

// rho = max((rho_sad + floor) exp(y) - floor, 0)
template <typename T>
__global__ void k_apply_correction(int64_t n, const double* __restrict__ rs, const T* __restrict__ y, double floor,
                                   double* __restrict__ rho) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) rho[i] = fmax((rs[i] + floor) * exp((double)y[i]) - floor, 0.0);
}

// target y = log(rho + floor) - log(rho_sad + floor)
template <typename T>
__global__ void k_log_ratio(int64_t n, const double* __restrict__ rho, const double* __restrict__ rs, double floor,
                            T* __restrict__ y) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) y[i] = (T)(log(rho[i] + floor) - log(rs[i] + floor));
}

__global__ void __launch_bounds__(256) k_wsum_part(const double* __restrict__ qpts, int64_t nq, const double* __restrict__ x,
                                                   double* __restrict__ part) {
  __shared__ double r[256];
  double a = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nq; i += (int64_t)gridDim.x * blockDim.x)
    a += qpts[4 * i + 3] * x[i];
  r[threadIdx.x] = a;
  __syncthreads();
  for (int s = 128; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s) r[threadIdx.x] += r[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = r[0];
}

__global__ void k_scale_to_count(int nb, const double* __restrict__ part, int64_t n, double target,
                                 double* __restrict__ x) {
  __shared__ double tot;
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int i = 0; i < nb; ++i) s += part[i];
    tot = s;
  }
  __syncthreads();
  const double f = tot > 0.0 ? target / tot : 1.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] *= f;
}

// FP64 (gradient checks): kch of K per split
template <typename T>
void gemm_g(int64_t M, int64_t Nn, int64_t K, int64_t kch, const T* A, int64_t sam, int64_t sak, const T* B,
            int64_t sbk, int64_t sbn, T* C, int64_t ldc, cudaStream_t st) {
  dim3 g((unsigned)((M + GM - 1) / GM), (unsigned)((Nn + GM - 1) / GM), (unsigned)((K + kch - 1) / kch));
  k_gemm_g<T><<<g, 256, 0, st>>>(M, Nn, K, kch, A, sam, sak, B, sbk, sbn, C, ldc);
  g_launches++;
}

// FP32: AK / BK as in k_gemm_f32; 16-byte loads where both operands' rows and pointers
// are aligned for them
template <bool AK, bool BK, int EPI>
void gemm_f32(int64_t M, int64_t Nn, int64_t K, int64_t kch, const float* A, int64_t lda, const float* B, int64_t ldb,
              float* C, int64_t ldc, const float* bias, float* act, const float* Zp, int silu, cudaStream_t st) {
  const bool vec = (lda & 3) == 0 && (ldb & 3) == 0 && ((uintptr_t)A & 15) == 0 && ((uintptr_t)B & 15) == 0;
  dim3 g((unsigned)((M + FT - 1) / FT), (unsigned)((Nn + FT - 1) / FT), (unsigned)((K + kch - 1) / kch));
  if (vec) k_gemm_f32<AK, BK, true, EPI><<<g, 256, 0, st>>>(M, Nn, K, kch, A, lda, B, ldb, C, ldc, bias, act, Zp, silu);
  else k_gemm_f32<AK, BK, false, EPI><<<g, 256, 0, st>>>(M, Nn, K, kch, A, lda, B, ldb, C, ldc, bias, act, Zp, silu);
  g_launches++;
}

// rows of one K split of the weight gradients: 64 partials at most (the scratch holds
// that many), no fewer than 64 rows each
int64_t grad_chunk(int64_t n) {
  const int64_t ns = std::max<int64_t>(1, std::min<int64_t>(64, n / 64));
  return ((n + ns - 1) / ns + GK - 1) / GK * GK;
}

}  // namespace

// ---------------------------------------------------------------------------
void launch_sad(const double* qpts, int64_t nq, const double* axyz, int na, const SadShellDev* sh, double* rho,
                cudaStream_t st) {
  if (nq <= 0) return;
  k_sad<<<nblk(nq, 256), 256, 0, st>>>(qpts, nq, axyz, na, sh, rho);
  g_launches++;
}

template <typename T>
void launch_descriptors(const double* qpts, int64_t nq, const double* axyz, const int32_t* slot, int na,
                        const DescDev& p, T* D, cudaStream_t st) {
  if (nq <= 0) return;
  DescInv v{};
  const double sg[2] = {p.radial_sigma, p.ang_sigma};
  for (int i = 0; i < 2; ++i) {
    v.c[i] = 2.0 * sg[i] * sg[i];
    v.rc[i] = 1.0 / v.c[i];
    if (!std::isnormal(v.c[i]) || !std::isnormal(v.rc[i])) v.rc[i] = 0.0;
  }
  v.g = (float)(-1.4426950408889634 / v.c[0]);
  const size_t smem = sizeof(T) * DESC_PTS * (size_t)(p.n_species * (p.n_radial + p.n_ang) + 1);
  cudaFuncSetAttribute(k_descriptors<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_descriptors<T><<<nblk(nq, DESC_PTS), DESC_PTS, smem, st>>>(qpts, nq, axyz, slot, na, p, v, D);
  g_launches++;
}
template void launch_descriptors<float>(const double*, int64_t, const double*, const int32_t*, int, const DescDev&,
                                        float*, cudaStream_t);
template void launch_descriptors<double>(const double*, int64_t, const double*, const int32_t*, int, const DescDev&,
                                         double*, cudaStream_t);

int64_t mlp_param_count(const int* dims, int nl) {
  int64_t s = 0;
  for (int l = 0; l < nl; ++l) s += (int64_t)dims[l + 1] * dims[l] + dims[l + 1];
  return s;
}

int64_t mlp_work_elems(const int* dims, int nl, int64_t n) {
  int64_t s = 0;
  for (int l = 0; l < nl; ++l) s += 2 * (int64_t)dims[l + 1];
  return s * n;
}

int64_t mlp_scratch_elems(const int* dims, int nl, int64_t n) {
  int dmax = 0;
  int64_t wmax = 0;
  for (int l = 0; l < nl; ++l) {
    dmax = std::max(dmax, std::max(dims[l], dims[l + 1]));
    wmax = std::max(wmax, (int64_t)dims[l + 1] * (dims[l] + 1));
  }
  return 2 * n * dmax + 64 * wmax + (int64_t)RED_B * dmax;
}

// work layout per layer l: Z_l (n x d_{l+1}) then A_l (n x d_{l+1})
template <typename T>
void mlp_forward(const int* dims, int nl, const T* params, const T* X, int64_t n, T* y, T* work, cudaStream_t st) {
  const T* a = X;
  const T* p = params;
  T* w = work;
  for (int l = 0; l < nl; ++l) {
    const int din = dims[l], dout = dims[l + 1];
    const T* W = p;
    const T* b = p + (int64_t)dout * din;
    T* Z = w;
    T* A = w + n * dout;
    if constexpr (std::is_same<T, float>::value) {
      if (l == nl - 1 && dout == 1) {
        k_row_dot<<<nblk(n, RD_R), 256, 0, st>>>(n, din, a, W, b, Z, A, y);
        g_launches++;
        return;
      }
      gemm_f32<true, true, 1>(n, dout, din, din, a, din, W, din, Z, dout, b, A, nullptr, l < nl - 1 ? 1 : 0, st);
    } else {
      // Z = a W^T : (n x din) (din x dout), element (k, j) of W^T = W[j * din + k]
      gemm_g<T>(n, dout, din, din, a, din, 1, W, 1, din, Z, dout, st);
      k_bias_act<T><<<nblk(n * dout, 256), 256, 0, st>>>(n, dout, b, Z, A, l < nl - 1 ? 1 : 0);
      g_launches++;
    }
    a = A;
    p = b + dout;
    w = A + n * dout;
  }
  // output layer has dout = 1: y = A_last
  cudaMemcpyAsync(y, a, sizeof(T) * n, cudaMemcpyDeviceToDevice, st);
}

template <typename T>
void mlp_backward(const int* dims, int nl, const T* params, const T* X, int64_t n, const T* work, const T* dy,
                  T* grads, T* scratch, cudaStream_t st) {
  int dmax = 0;
  int64_t wmax = 0;
  for (int l = 0; l < nl; ++l) {
    dmax = std::max(dmax, std::max(dims[l], dims[l + 1]));
    wmax = std::max(wmax, (int64_t)dims[l + 1] * (dims[l] + 1));
  }
  T* dcur = scratch;                 // n x dmax
  T* dnext = scratch + n * dmax;     // n x dmax
  T* part = dnext + n * dmax;        // 64 x wmax
  T* cpart = part + 64 * wmax;       // RED_B x dmax
  // parameter and work offsets
  int64_t poff[16], woff[16];
  int64_t po = 0, wo = 0;
  for (int l = 0; l < nl; ++l) {
    poff[l] = po;
    woff[l] = wo;
    po += (int64_t)dims[l + 1] * dims[l] + dims[l + 1];
    wo += 2 * n * dims[l + 1];
  }
  cudaMemcpyAsync(dcur, dy, sizeof(T) * n, cudaMemcpyDeviceToDevice, st);  // dZ of the output layer (identity)
  for (int l = nl - 1; l >= 0; --l) {
    const int din = dims[l], dout = dims[l + 1];
    const T* a_prev = (l == 0) ? X : work + woff[l - 1] + n * dims[l];
    T* gW = grads + poff[l];
    T* gb = gW + (int64_t)dout * din;
    // dW = dZ^T a_prev : (dout x n)(n x din), split over n
    const int64_t kch = grad_chunk(n);
    const int nz = (int)((n + kch - 1) / kch);
    if constexpr (std::is_same<T, float>::value)
      gemm_f32<false, false, 0>(dout, din, n, kch, dcur, dout, a_prev, din, part, din, nullptr, nullptr, nullptr, 0, st);
    else
      gemm_g<T>(dout, din, n, kch, dcur, 1, dout, a_prev, din, 1, part, din, st);
    k_sum_parts<T><<<nblk((int64_t)dout * din, 32), 256, 0, st>>>(nz, (int64_t)dout * din, part, gW);
    // db = column sums of dZ
    const int64_t rpb = (n + RED_B - 1) / RED_B;
    dim3 gc((unsigned)((n + rpb - 1) / rpb), (unsigned)((dout + 127) / 128));
    k_colsum_part<T><<<gc, 128, 0, st>>>(n, dout, dcur, rpb, cpart);
    k_sum_parts<T><<<nblk(dout, 32), 256, 0, st>>>((int)gc.x, dout, cpart, gb);
    g_launches += 3;
    if (l > 0) {
      // dA_prev = dZ W : (n x dout)(dout x din), then dZ_prev = dA_prev * silu'(Z_prev)
      if constexpr (std::is_same<T, float>::value) {
        gemm_f32<true, false, 2>(n, din, dout, dout, dcur, dout, params + poff[l], din, dnext, din, nullptr, nullptr,
                                 work + woff[l - 1], 0, st);
      } else {
        gemm_g<T>(n, din, dout, dout, dcur, dout, 1, params + poff[l], din, 1, dnext, din, st);
        k_act_back<T><<<nblk(n * din, 256), 256, 0, st>>>(n * din, work + woff[l - 1], dnext);
        g_launches++;
      }
      T* t = dcur;
      dcur = dnext;
      dnext = t;
    }
  }
}

template void mlp_forward<float>(const int*, int, const float*, const float*, int64_t, float*, float*, cudaStream_t);
template void mlp_forward<double>(const int*, int, const double*, const double*, int64_t, double*, double*,
                                  cudaStream_t);
template void mlp_backward<float>(const int*, int, const float*, const float*, int64_t, const float*, const float*,
                                  float*, float*, cudaStream_t);
template void mlp_backward<double>(const int*, int, const double*, const double*, int64_t, const double*,
                                   const double*, double*, double*, cudaStream_t);

template <typename T>
void launch_wmse(const T* yh, const T* y, const T* c, int64_t n, T* dy, double* part, double* stats, cudaStream_t st) {
  k_wmse_part<T><<<RED_B, 256, 0, st>>>(n, yh, y, c, part);
  k_wmse_finish<<<1, RED_B, 0, st>>>(part, stats);
  k_wmse_grad<T><<<nblk(n, 256), 256, 0, st>>>(n, yh, y, c, stats, dy);
  g_launches += 3;
}
template void launch_wmse<float>(const float*, const float*, const float*, int64_t, float*, double*, double*,
                                 cudaStream_t);
template void launch_wmse<double>(const double*, const double*, const double*, int64_t, double*, double*, double*,
                                  cudaStream_t);

template <typename T>
void launch_adam(int64_t n, T* p, const T* g, T* m, T* v, double lr, double b1, double b2, double eps, int t,
                 cudaStream_t st) {
  const double c1 = 1.0 - pow(b1, (double)t), c2 = 1.0 - pow(b2, (double)t);
  k_adam<T><<<nblk(n, 256), 256, 0, st>>>(n, p, g, m, v, lr, b1, b2, eps, c1, c2);
  g_launches++;
}
template void launch_adam<float>(int64_t, float*, const float*, float*, float*, double, double, double, double, int,
                                 cudaStream_t);
template void launch_adam<double>(int64_t, double*, const double*, double*, double*, double, double, double, double,
                                  int, cudaStream_t);

template <typename T>
void launch_apply_correction(int64_t n, const double* rs, const T* y, double floor, double* rho, cudaStream_t st) {
  k_apply_correction<T><<<nblk(n, 256), 256, 0, st>>>(n, rs, y, floor, rho);
  g_launches++;
}
template void launch_apply_correction<float>(int64_t, const double*, const float*, double, double*, cudaStream_t);
template void launch_apply_correction<double>(int64_t, const double*, const double*, double, double*, cudaStream_t);

template <typename T>
void launch_log_ratio(int64_t n, const double* rho, const double* rs, double floor, T* y, cudaStream_t st) {
  k_log_ratio<T><<<nblk(n, 256), 256, 0, st>>>(n, rho, rs, floor, y);
  g_launches++;
}
template void launch_log_ratio<float>(int64_t, const double*, const double*, double, float*, cudaStream_t);
template void launch_log_ratio<double>(int64_t, const double*, const double*, double, double*, cudaStream_t);

void launch_scale_count(const double* qpts, int64_t nq, double target, double* x, double* part, cudaStream_t st) {
  k_wsum_part<<<RED_B, 256, 0, st>>>(qpts, nq, x, part);
  k_scale_to_count<<<RED_B, 256, 0, st>>>(RED_B, part, nq, target, x);
  g_launches += 2;
}

int learn_reduce_blocks() { return RED_B; }

}  // namespace efe
