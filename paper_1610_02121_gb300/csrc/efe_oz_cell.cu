// FP64-grade cell products H^cc_e Y_e of all cells on the BF16 tensor cores (the
// CELL products of the FP64 engine; the slicing and its error bound are described in
// efe_oz.cu), sm_103a tcgen05 and TMA.
//
// Three kernels per panel of columns:
//   k_ozc_slice   cuts the panel of Y into seven BF16 digit planes, one row per node
//                 (14 bytes a value, columns padded to 16);
//   k_ozc_cell    persistent, one (cell, 48-column tile) at a time: the cell's 125 node
//                 rows of every digit plane come in as 5 x 5 x 5-node TMA boxes (the
//                 nodes of a cell are a box of the node grid) in the MN-major layout
//                 the MMA reads, H^cc_e's digits as 28 KB bulk copies per 16-wide K
//                 chunk, and the products leave as FP64 rows of a scratch array;
//   k_ozc_gather  adds the products of the cells around every node in the order of
//                 their parity colours, so the sums do not depend on the launch.
//
// Why this split: with the slicing inside the product kernel every node row was
// gathered and cut once per cell that holds it (about twice) by seven warps, at
// 64 us for a 96-column tile whose MMAs take 6; and one accumulator set made the
// epilogue wait for the MMAs and the MMAs for it.  48 columns leave TMEM for two
// sets (2 x 5 x 48 of 512 columns), and shared memory for two column tiles of Y
// (2 x 84 KB) beside two chunks of H (2 x 28 KB).  Per apply, 8,424 cells x 135 columns:
// 7.2 ms before; now 0.25 (slice) + 1.94 (cells: 11.6 us a tile) + 0.63 (gather); x 640
// columns 23.6 -> 12.3 ms.  What is left: operand traffic from L2 (310 KB a tile) and
// the shared-memory reads of the MMAs (128 x 48 x 16: 44 clocks for 24 of math).
//
// Warp roles (512 threads): warp 0 issues the MMAs (one elected lane), one lane of
// warp 1 the copies, warps 4-15 share the epilogue (three per TMEM lane quarter).
// All waits are bounded; on timeout the CTA records an error, stops issuing, drains
// its copies and MMAs and frees its TMEM.
#include <cuda.h>
#include <stdint.h>

#include <algorithm>

#include "efe_kernels.h"
#include "efe_oz.cuh"

namespace efe {

namespace {

constexpr int OC_TW = 48;                                // column tile
constexpr int OC_G = OC_TW / 16;                         // 16-column groups (one TMA box each)
constexpr int OC_NCH = (NL + OZ_KC - 1) / OZ_KC;         // K chunks of a cell
constexpr uint32_t OC_BOX = 4096;                        // a box: 125 rows of 32 B, padded to 128 rows
constexpr uint32_t OC_BOX_BYTES = NL * 32;               // bytes the TMA writes of it
constexpr uint32_t OC_B = OZ_S * OC_G * OC_BOX;          // one column tile of Y, 84 KB
constexpr uint32_t OC_A = OZ_S * OZ_ASL;                 // one chunk of H, 28 KB
constexpr uint32_t OC_A0 = 2 * OC_B;
constexpr uint32_t OC_BARS = OC_A0 + 2 * OC_A;
constexpr size_t OC_SMEM = (size_t)OC_BARS + 256;
constexpr int OC_THREADS = 512;
constexpr int OC_EPI_W0 = 4, OC_EPI_WN = 12;

// A: K-major, no swizzle (core matrix 8 rows x 16 B; LBO 128 B to the next 8 K, SBO 256 B
// to the next 8 rows)
__device__ __forceinline__ uint64_t desc_a(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(256u >> 4) << 32) |
         ((uint64_t)1 << 46);
}
// B: MN-major, 32-byte swizzle (16 columns of 8 K rows a pattern; LBO to the next 16
// columns, SBO to the next 8 K)
__device__ __forceinline__ uint64_t desc_b(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(OC_BOX >> 4) << 16) | ((uint64_t)(256u >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)6 << 61);
}
// FP32 accumulate, BF16 operands, B MN-major (bit 16)
__device__ __forceinline__ uint32_t idesc_cell(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(OZ_M >> 4) << 24);
}
__device__ __forceinline__ void tma_box(void* dst, const CUtensorMap* tm, int c, int x, int y, int z, int s, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], "
      "[%7];" ::"r"(su32(dst)),
      "l"(tm), "r"(c), "r"(x), "r"(y), "r"(z), "r"(s), "r"(su32(bar))
      : "memory");
}

// digit planes of Y[:, c0 .. c0 + nc): D[s][node][ldn] (BF16 digit s times 2^-7s, columns
// nc .. ldn zero); one thread per node and eight columns.  The same truncation and digits
// as oz_pack8: 49 bits below the column's exponent.  Integer-issue bound: a digit is cut
// out, made a float by the 2^23 trick and scaled by an exact power of two (five
// operations; the leading-bit search of oz_pack8 takes about ten).
__global__ void __launch_bounds__(256) k_ozc_slice(const double* __restrict__ Y, int64_t ldy, int64_t nn, int nc, int ldn,
                                                   const int* __restrict__ fexp, uint16_t* __restrict__ D) {
  const int no = ldn / 8;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= nn * no) return;
  const int64_t g = t / no;
  const int c = (int)(t % no) * 8;
  const double* yr = Y + g * ldy + c;
  double x[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) x[q] = c + q < nc ? yr[q] : 0.0;
  uint32_t pk[OZ_S][4];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int E = c + q < nc ? fexp[c + q] : -2000;
    const long long bits = __double_as_longlong(x[q]);
    const int ex = (int)((bits >> 52) & 0x7FF);
    const float one = __uint_as_float(((uint32_t)(bits >> 32) & 0x80000000u) | 0x3F800000u);   // +-1
    unsigned long long qq = 0;
    const int rs = 1026 + E - ex;
    if (ex != 0 && rs >= 0 && rs < 64) qq = ((unsigned long long)(bits & 0xFFFFFFFFFFFFFull) | (1ull << 52)) >> rs;
    const uint32_t w1 = (uint32_t)(qq >> 21), w0 = (uint32_t)qq & 0x1FFFFFu;   // digits 1-4, 5-7
#pragma unroll
    for (int i = 0; i < OZ_S; ++i) {
      const uint32_t w = i < 4 ? w1 >> (21 - 7 * i) : w0 >> (42 - 7 * i);
      const float d = __uint_as_float((w & 127u) | 0x4B000000u) - 8388608.f;
      const uint32_t h = __float_as_uint(d * (one * __uint_as_float((uint32_t)(127 - 7 * i) << 23)));
      pk[i][q >> 1] = (q & 1) ? __byte_perm(pk[i][q >> 1], h, 0x7632) : h;
    }
  }
  uint16_t* o = D + g * ldn + c;
#pragma unroll
  for (int i = 0; i < OZ_S; ++i)
    *reinterpret_cast<uint4*>(o + (int64_t)i * nn * ldn) = make_uint4(pk[i][0], pk[i][1], pk[i][2], pk[i][3]);
}

struct OzCellArgs {
  const unsigned char* Aimg;   // digit images of H^cc_e (launch_oz_preslice)
  const int* hexp;             // n_cell x 128 row exponents
  const int* fexp;             // column exponents of the panel
  int64_t n_cell;
  int nc[3];
  double* P;                   // products, [cell][125][ldn]
  int ldn, ntiles;
  int* err;
  int stall;
};

__global__ void __launch_bounds__(OC_THREADS, 1) k_ozc_cell(const __grid_constant__ CUtensorMap tmap, OzCellArgs g) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // an earlier launch already failed: leave at once (CTA-uniform decision)
  __shared__ int s_skip;
  if (tid == 0) s_skip = *(volatile int*)g.err;
  __syncthreads();
  if (s_skip) return;
  uint64_t* afull = reinterpret_cast<uint64_t*>(sm + OC_BARS);   // [2] chunk of H landed
  uint64_t* aempty = afull + 2;                                  // [2] its MMAs are done
  uint64_t* bfull = afull + 4;                                   // [2] column tile of Y landed
  uint64_t* bempty = afull + 6;                                  // [2] its MMAs are done
  uint64_t* accf = afull + 8;                                    // [2] accumulator set complete
  uint64_t* acce = afull + 10;                                   // [2] accumulator set read
  uint64_t* never = afull + 12;                                  // no thread ever arrives here (test stall)
  uint32_t* tslot = reinterpret_cast<uint32_t*>(afull + 13);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(afull + 14);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)),
                 "r"(OZ_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    for (int i = 0; i < 2; ++i) {
      bar_init(afull + i, 1);
      bar_init(aempty + i, 1);
      bar_init(bfull + i, 1);
      bar_init(bempty + i, 1);
      bar_init(accf + i, 1);
      bar_init(acce + i, OC_EPI_WN * 32);
    }
    bar_init(never, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // K rows 125 .. 127 of every box stay zero (the TMA writes 125 rows)
  for (int t = tid; t < 2 * OZ_S * OC_G * 6; t += OC_THREADS)
    *reinterpret_cast<uint4*>(sm + (t / 6) * OC_BOX + OC_BOX_BYTES + (t % 6) * 16) = make_uint4(0, 0, 0, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const int64_t nitems = g.n_cell * g.ntiles;
  const int64_t my = nitems > blockIdx.x ? (nitems - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  // what this thread issued last (drained after an abort)
  int64_t last_mma = -1, last_a = -1, last_b = -1;

  if (warp == 0) {
    // ---------------------------------------------------------------- MMA issuer
    if (g.stall && my > 0 && !bar_wait(never, 0u)) {
      // test stall: a wait that nothing completes runs out like a real one
      if (lane == 0) { *abort_flag = 1; atomicExch(g.err, 1); }
    }
    for (int64_t t = 0; t < my && !*abort_flag; ++t) {
      const int64_t item = blockIdx.x + t * gridDim.x;
      const int c0 = (int)(item % g.ntiles) * OC_TW;
      const uint32_t id = idesc_cell(min(OC_TW, g.ldn - c0));
      const int b = (int)(t & 1);
      bool ok = true;
      if (t >= 2) ok = bar_wait(acce + b, (uint32_t)((t / 2 - 1) & 1));
      if (ok) ok = bar_wait(bfull + b, (uint32_t)((t / 2) & 1));
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int kc = 0; kc < OC_NCH && ok; ++kc) {
        const int64_t ch = t * OC_NCH + kc;
        const int s = (int)(ch & 1);
        ok = bar_wait(afull + s, (uint32_t)((ch / 2) & 1));
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!ok) break;
        if (lane == 0) {
          const uint32_t sA = su32(sm + OC_A0 + s * OC_A);
          const uint32_t sB = su32(sm + b * OC_B) + (uint32_t)kc * 512u;
          const uint32_t d = tmem + (uint32_t)(b * OZ_NACC * OC_TW);
          bool first[OZ_NACC] = {true, true, true, true, true};
#pragma unroll
          for (int tt = 2; tt <= 8; ++tt) {
            const int a = tt <= 5 ? tt - 2 : 4;
#pragma unroll
            for (int i = 1; i < tt; ++i) {
              const int j = tt - i;
              if (i > OZ_S || j > OZ_S) continue;
              const uint32_t acc = (kc > 0 || !first[a]) ? 1u : 0u;
              first[a] = false;
              mma_bf16(d + (uint32_t)(a * OC_TW), desc_a(sA + (uint32_t)(i - 1) * OZ_ASL),
                       desc_b(sB + (uint32_t)(j - 1) * (OC_G * OC_BOX)), id, acc);
            }
          }
          mma_commit(aempty + s);
          if (kc == OC_NCH - 1) {
            mma_commit(bempty + b);
            mma_commit(accf + b);
          }
        }
        last_mma = ch;
        __syncwarp();
      }
      if (!ok) {
        if (lane == 0) { *abort_flag = 1; atomicExch(g.err, 1); }
        break;
      }
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------------------------------------------------------- copies
    auto load_b = [&](int64_t t) -> bool {
      const int64_t item = blockIdx.x + t * gridDim.x;
      const int64_t e = item / g.ntiles;
      const int c0 = (int)(item % g.ntiles) * OC_TW;
      const int ng = (min(OC_TW, g.ldn - c0) + 15) / 16;
      const int b = (int)(t & 1);
      if (t >= 2 && !bar_wait(bempty + b, (uint32_t)((t / 2 - 1) & 1))) return false;
      const int x = P * (int)(e % g.nc[0]), y = P * (int)((e / g.nc[0]) % g.nc[1]),
                z = P * (int)(e / ((int64_t)g.nc[0] * g.nc[1]));
      bar_expect_tx(bfull + b, (uint32_t)(OZ_S * ng) * OC_BOX_BYTES);
      for (int s = 0; s < OZ_S; ++s)
        for (int q = 0; q < ng; ++q)
          tma_box(sm + b * OC_B + (s * OC_G + q) * OC_BOX, &tmap, c0 + 16 * q, x, y, z, s, bfull + b);
      last_b = t;
      return true;
    };
    bool ok = my > 0 ? load_b(0) : true;
    for (int64_t t = 0; t < my && ok && !*abort_flag; ++t) {
      const int64_t e = (blockIdx.x + t * gridDim.x) / g.ntiles;
      for (int kc = 0; kc < OC_NCH && ok; ++kc) {
        const int64_t ch = t * OC_NCH + kc;
        const int s = (int)(ch & 1);
        if (ch >= 2) ok = bar_wait(aempty + s, (uint32_t)((ch / 2 - 1) & 1));
        if (!ok) break;
        bar_expect_tx(afull + s, OC_A);
        bulk_g2s(sm + OC_A0 + s * OC_A, g.Aimg + (e * OC_NCH + kc) * (int64_t)OC_A, OC_A, afull + s);
        last_a = ch;
        // the next item's columns, once this item's first chunks are on their way (the
        // buffer was freed by the item before)
        if (kc == 1 && t + 1 < my) ok = load_b(t + 1);
      }
    }
    if (!ok) {
      *abort_flag = 1;
      atomicExch(g.err, 1);
    }
  } else if (warp >= OC_EPI_W0) {
    // ---------------------------------------------------------------- epilogue
    const int quarter = warp & 3;   // the TMEM lane quarter this warp may read
    const int part = (warp - OC_EPI_W0) >> 2;
    const int r = quarter * 32 + lane;
    for (int64_t t = 0; t < my && !*abort_flag; ++t) {
      const int64_t item = blockIdx.x + t * gridDim.x;
      const int64_t e = item / g.ntiles;
      const int c0 = (int)(item % g.ntiles) * OC_TW;
      const int ncol = min(OC_TW, g.ldn - c0);
      const int b = (int)(t & 1);
      const int Er = g.hexp[e * OZ_M + r];
      double* out = g.P + (e * NL + r) * (int64_t)g.ldn + c0;
      if (!bar_wait(accf + b, (uint32_t)((t / 2) & 1))) {
        *abort_flag = 1;
        atomicExch(g.err, 1);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
      for (int u = 0; u < OC_TW / 8 / 3; ++u) {
        const int cb = 8 * (part + 3 * u);
        if (cb < ncol) {
          uint32_t v[OZ_NACC][8];
#pragma unroll
          for (int a = 0; a < OZ_NACC; ++a)
            asm volatile(
                "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                : "=r"(v[a][0]), "=r"(v[a][1]), "=r"(v[a][2]), "=r"(v[a][3]), "=r"(v[a][4]), "=r"(v[a][5]),
                  "=r"(v[a][6]), "=r"(v[a][7])
                : "r"(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((b * OZ_NACC + a) * OC_TW + cb))
                : "memory");
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          int fe[8];
          *reinterpret_cast<int4*>(fe) = *reinterpret_cast<const int4*>(g.fexp + c0 + cb);
          *reinterpret_cast<int4*>(fe + 4) = *reinterpret_cast<const int4*>(g.fexp + c0 + cb + 4);
#pragma unroll
          for (int q = 0; q < 8; q += 2) {
            double val[2];
#pragma unroll
            for (int w = 0; w < 2; ++w) {
              float s1, e1, s2, e2, s3, e3;
              two_sum(__uint_as_float(v[0][q + w]), __uint_as_float(v[1][q + w]), s1, e1);
              two_sum(s1, __uint_as_float(v[2][q + w]), s2, e2);
              two_sum(s2, __uint_as_float(v[3][q + w]), s3, e3);
              const float lo = ((__uint_as_float(v[4][q + w]) + e3) + e2) + e1;
              const int k2 = Er + fe[q + w] - 14;
              val[w] = f32_scaled(s3, k2) + f32_scaled(lo, k2);
            }
            if (r < NL) *reinterpret_cast<double2*>(out + cb + q) = make_double2(val[0], val[1]);
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      bar_arrive(acce + b);
    }
  }
  // all roles done.  After an abort every copy still in flight lands and the last MMA
  // commit (it covers every MMA this CTA issued) arrives before the TMEM and the shared
  // memory are released; each drain wait is bounded like the pipeline's own.
  __syncthreads();
  if (*abort_flag) {
    for (int64_t ch = last_a - 1; ch <= last_a; ++ch)
      if (ch >= 0) bar_wait(afull + (int)(ch & 1), (uint32_t)((ch / 2) & 1));
    for (int64_t t = last_b - 1; t <= last_b; ++t)
      if (t >= 0) bar_wait(bfull + (int)(t & 1), (uint32_t)((t / 2) & 1));
    if (warp == 0 && lane == 0 && last_mma >= 0)
      bar_wait(aempty + (int)(last_mma & 1), (uint32_t)((last_mma / 2) & 1));
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM_COLS) : "memory");
  }
}

// W[node][c] = sum of the cell products around the node in the order of the parity
// colours; a block of 16 nodes x 16 column pairs
__global__ void __launch_bounds__(256) k_ozc_gather(MeshDev m, int64_t nn, const double* __restrict__ Pc, int ldn, int nc,
                                                    double* __restrict__ W, int64_t ldw) {
  const int64_t gn = blockIdx.x * 16LL + threadIdx.y;
  const int c = (blockIdx.y * 16 + threadIdx.x) * 2;
  if (gn >= nn || c >= nc) return;
  const int G[3] = {(int)(gn % m.nn[0]), (int)((gn / m.nn[0]) % m.nn[1]), (int)(gn / ((int64_t)m.nn[0] * m.nn[1]))};
  int hi[3];
  bool two[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    hi[d] = min(G[d] / P, m.nc[d] - 1);
    two[d] = G[d] % P == 0 && G[d] > 0 && G[d] / P < m.nc[d];
  }
  double2 s = make_double2(0.0, 0.0);
#pragma unroll
  for (int col = 0; col < 8; ++col) {
    int cc[3], l[3];
    bool ok = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      cc[d] = (hi[d] & 1) == ((col >> d) & 1) ? hi[d] : hi[d] - 1;
      ok = ok && (cc[d] == hi[d] || two[d]);
      l[d] = G[d] - P * cc[d];
    }
    if (!ok) continue;
    const int64_t e = cc[0] + (int64_t)m.nc[0] * (cc[1] + (int64_t)m.nc[1] * cc[2]);
    const double2 p = *reinterpret_cast<const double2*>(Pc + (e * NL + l[0] + NP1 * (l[1] + NP1 * l[2])) * (int64_t)ldn + c);
    s.x += p.x;
    s.y += p.y;
  }
  W[gn * ldw + c] = s.x;
  if (c + 1 < nc) W[gn * ldw + c + 1] = s.y;
}

typedef CUresult (*EncodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encode_tiled() {
  static const EncodeTiled fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess) {
      cudaGetLastError();
      return (EncodeTiled) nullptr;
    }
    return (EncodeTiled)p;
  }();
  return fn;
}

inline int pad16(int n) { return (n + 15) / 16 * 16; }

}  // namespace

int64_t ozc_digit_bytes(int64_t nn, int nc) { return (int64_t)OZ_S * 2 * nn * pad16(nc); }
int64_t ozc_product_bytes(int64_t n_cell, int nc) { return (int64_t)sizeof(double) * n_cell * NL * pad16(nc); }

// widest panel (at most N columns) whose digit planes and products fit the two budgets;
// whole 48-column tiles unless it is the whole block
int ozc_panel_cols(int64_t nn, int64_t n_cell, int N, int64_t digit_budget, int64_t product_budget) {
  const int64_t w = std::min(digit_budget / (OZ_S * 2 * nn), product_budget / ((int64_t)sizeof(double) * n_cell * NL));
  if (w >= pad16(N)) return N;
  return (int)std::max<int64_t>(OC_TW, w / OC_TW * OC_TW);
}

int launch_ozc_cells(const unsigned char* Aimg, const int* hexp, int64_t n_cell, const MeshDev& m, const double* Y,
                     int64_t ldy, const int* fexp, unsigned char* digits, double* products, double* W, int64_t ldw, int N,
                     int n_sm, int* err, cudaStream_t st, int stall) {
  if (n_cell <= 0 || N <= 0) return 0;
  const EncodeTiled enc = encode_tiled();
  if (!enc) return 1;
  const int64_t nn = (int64_t)m.nn[0] * m.nn[1] * m.nn[2];
  const int ldn = pad16(N);
  const int64_t ns = nn * (ldn / 8);
  k_ozc_slice<<<(unsigned)((ns + 255) / 256), 256, 0, st>>>(Y, ldy, nn, N, ldn, fexp, reinterpret_cast<uint16_t*>(digits));
  // digit planes as a 5-D tensor: column, x, y, z, digit; a box: 16 columns of the 125
  // nodes of a cell
  CUtensorMap tm;
  const cuuint64_t row = (cuuint64_t)ldn * 2;
  const cuuint64_t dims[5] = {(cuuint64_t)ldn, (cuuint64_t)m.nn[0], (cuuint64_t)m.nn[1], (cuuint64_t)m.nn[2], OZ_S};
  const cuuint64_t strides[4] = {row, row * m.nn[0], row * m.nn[0] * m.nn[1], row * (cuuint64_t)nn};
  const cuuint32_t box[5] = {16, NP1, NP1, NP1, 1};
  const cuuint32_t es[5] = {1, 1, 1, 1, 1};
  if (enc(&tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, digits, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
          CU_TENSOR_MAP_SWIZZLE_32B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return 1;
  OzCellArgs a{};
  a.Aimg = Aimg;
  a.hexp = hexp;
  a.fexp = fexp;
  a.n_cell = n_cell;
  for (int d = 0; d < 3; ++d) a.nc[d] = m.nc[d];
  a.P = products;
  a.ldn = ldn;
  a.ntiles = (ldn + OC_TW - 1) / OC_TW;
  a.err = err;
  a.stall = stall;
  const int64_t items = n_cell * a.ntiles;
  if (cudaFuncSetAttribute(k_ozc_cell, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OC_SMEM) != cudaSuccess) return 1;
  k_ozc_cell<<<(unsigned)std::min<int64_t>(items, n_sm), OC_THREADS, OC_SMEM, st>>>(tm, a);
  k_ozc_gather<<<dim3((unsigned)((nn + 15) / 16), (unsigned)((N + 31) / 32)), dim3(16, 16), 0, st>>>(m, nn, products, ldn, N, W,
                                                                                                  ldw);
  g_launches.fetch_add(3, std::memory_order_relaxed);
  return 0;
}

}  // namespace efe
