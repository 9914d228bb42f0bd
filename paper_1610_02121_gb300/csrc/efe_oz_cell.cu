// FP64-grade cell products H^cc_e Y_e of all cells on the BF16 tensor cores (the
// CELL products of the FP64 engine; the slicing and its error bound are described in
// efe_oz.cu), sm_103a tcgen05.
//
// Three kernels per panel of columns:
//   k_ozc_slice   cuts the panel of Y into seven BF16 digit planes, one row per node
//                 (14 bytes a value, columns padded to 16);
//   k_ozc_cell    persistent, one (cell, 48-column tile) at a time: per 16-wide K chunk
//                 H^cc_e's digits arrive as one 28 KB bulk copy and 16 node rows of every
//                 digit plane as 16-byte asynchronous copies in the MN-major layout the
//                 MMA reads; the products leave as FP64 rows of a scratch array;
//   k_ozc_gather  adds the products of the cells around every node in the order of
//                 their parity colours, so the sums do not depend on the launch.
//
// Why this split: with the slicing inside the product kernel every node row was
// gathered and cut once per cell that holds it (about twice) by seven warps, at
// 64 us for a 96-column tile whose MMAs take 6; and one accumulator set made the
// epilogue wait for the MMAs and the MMAs for it.  48 columns leave TMEM for two
// sets (2 x 5 x 48 of 512 columns) and shared memory for five chunks of both operands
// in flight.  Taking the rows as 5 x 5 x 5-node TMA boxes of 32-byte rows (21 boxes
// and so whole column tiles a cell) ran at 11.6 us a tile: it left room for two chunks
// of H only.  What bounds it now: the MMAs' shared-memory reads (128 x 48 x 16: 4 KB of
// H and 1.5 KB of Y, 44 clocks for 24 of math; measured 44.4 back to back).  Per apply,
// 8,424 cells x 135 columns: 7.2 ms in the old form; now 0.25 (slice) + 1.42 (cells, 8.5
// us a tile) + 0.50 (gather); x 640 columns 23.6 -> 9.3 ms.
//
// Warp roles (512 threads): warp 0 issues the MMAs (one elected lane), warps 1-3 the
// copies (a thread takes one (K row, 8 columns) of all digits), warps 4-15 share the
// epilogue (three per TMEM lane quarter).  All waits are bounded; on timeout the CTA
// records an error, stops issuing, drains its copies and MMAs and frees its TMEM.
#include <stdint.h>

#include <algorithm>

#include "efe_kernels.h"
#include "efe_oz.cuh"

namespace efe {

namespace {

constexpr int OC_TW = 48;                                // column tile
constexpr int OC_NO = OC_TW / 8;                         // 8-column octets
constexpr int OC_NCH = (NL + OZ_KC - 1) / OZ_KC;         // K chunks of a cell
// B of a chunk: per digit and octet two 8 x 16 B core matrices (K rows 0-7, 8-15); octets
// 272 B apart, so that the 16-byte copies of a row fall into different banks
constexpr uint32_t OC_OCT = 272;
constexpr uint32_t OC_BSL = OC_NO * OC_OCT;
constexpr uint32_t OC_A = OZ_S * OZ_ASL;                 // H, 28 KB
constexpr uint32_t OC_STAGE = (OC_A + OZ_S * OC_BSL + 127) / 128 * 128;
constexpr int OC_STAGES = 5;
constexpr uint32_t OC_BARS = OC_STAGES * OC_STAGE;
constexpr size_t OC_SMEM = (size_t)OC_BARS + 256;
constexpr int OC_THREADS = 512;
constexpr int OC_CPY_W0 = 1, OC_CPY_T = OZ_KC * OC_NO;   // copy threads: 16 rows x 6 octets = warps 1-3
constexpr int OC_DEPTH = 3;                              // chunks of 16-byte copies in flight per thread
constexpr int OC_EPI_W0 = 4, OC_EPI_WN = 12;
static_assert(OC_CPY_T == 96, "warps 1-3");

// A: K-major, no swizzle (core matrix 8 rows x 16 B; LBO 128 B to the next 8 K, SBO 256 B
// to the next 8 rows)
__device__ __forceinline__ uint64_t desc_a(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(256u >> 4) << 32) |
         ((uint64_t)1 << 46);
}
// B: MN-major, no swizzle (core matrix 8 K x 8 columns; LBO 128 B to the next 8 K, SBO to
// the next 8 columns)
__device__ __forceinline__ uint64_t desc_b(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(OC_OCT >> 4) << 32) |
         ((uint64_t)1 << 46);
}
// FP32 accumulate, BF16 operands, B MN-major (bit 16)
__device__ __forceinline__ uint32_t idesc_cell(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(OZ_M >> 4) << 24);
}
// 16 bytes to shared memory (zeros when valid is false)
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16u : 0u) : "memory");
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(p));
  return p != 0;
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
  const uint16_t* D;           // digit planes (k_ozc_slice)
  int64_t n_cell, nn;
  MeshDev m;
  double* P;                   // products, [cell][125][ldn]
  int ldn, ntiles;
  int* err;
  int stall;                   // tests only (EFE_OPT_TEST_STALL)
};

__global__ void __launch_bounds__(OC_THREADS, 1) k_ozc_cell(OzCellArgs g) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  // an earlier launch already failed: leave at once (CTA-uniform decision)
  __shared__ int s_skip;
  __shared__ int koff[OC_NCH * OZ_KC];   // node offset of K row k from the cell's first node; -1: padding
  if (tid == 0) s_skip = *(volatile int*)g.err;
  if (tid < OC_NCH * OZ_KC) {
    const int a = tid % NP1, b = (tid / NP1) % NP1, c = tid / (NP1 * NP1);
    koff[tid] = tid < NL ? a + g.m.nn[0] * (b + g.m.nn[1] * c) : -1;
  }
  __syncthreads();
  if (s_skip) return;
  uint64_t* full = reinterpret_cast<uint64_t*>(sm + OC_BARS);   // [stages] both operands of a chunk landed
  uint64_t* empty = full + OC_STAGES;                           // [stages] its MMAs are done
  uint64_t* accf = full + 2 * OC_STAGES;                        // [2] accumulator set complete
  uint64_t* acce = accf + 2;                                    // [2] accumulator set read
  uint32_t* tslot = reinterpret_cast<uint32_t*>(accf + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(accf + 6);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)),
                 "r"(OZ_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    for (int i = 0; i < OC_STAGES; ++i) {
      bar_init(full + i, OC_CPY_T + 1 + (g.stall == 1));
      bar_init(empty + i, 1 + (g.stall == 2));
    }
    for (int i = 0; i < 2; ++i) {
      bar_init(accf + i, 1 + (g.stall == 3));
      bar_init(acce + i, OC_EPI_WN * 32);
    }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const int64_t nitems = g.n_cell * g.ntiles;
  const int64_t my = nitems > blockIdx.x ? (nitems - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  // the last chunk whose MMAs were committed / whose bulk copy was issued (drained
  // after an abort)
  int64_t last_mma = -1, last_copy = -1;

  if (warp == 0) {
    // ---------------------------------------------------------------- MMA issuer
    int s = 0;
    uint32_t ph = 0;
    for (int64_t t = 0; t < my && !warp_aborted(abort_flag); ++t) {
      const int64_t item = blockIdx.x + t * gridDim.x;
      const int c0 = (int)(item % g.ntiles) * OC_TW;
      const uint32_t id = idesc_cell(min(OC_TW, g.ldn - c0));
      const int b = (int)(t & 1);
      bool ok = true;
      if (t >= 2) ok = warp_wait(acce + b, (uint32_t)((t / 2 - 1) & 1));
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t d = tmem + (uint32_t)(b * OZ_NACC * OC_TW);
      for (int kc = 0; kc < OC_NCH && ok; ++kc) {
        ok = warp_wait(full + s, ph);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!ok) break;
        const uint32_t sA = su32(sm) + (uint32_t)s * OC_STAGE;
        const uint64_t da = desc_a(sA), db = desc_b(sA + OC_A);
        if (elect_one()) {
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
              mma_bf16(d + (uint32_t)(a * OC_TW), da + (uint64_t)((i - 1) * (OZ_ASL >> 4)),
                       db + (uint64_t)((j - 1) * (OC_BSL >> 4)), id, acc);
            }
          }
          mma_commit(empty + s);
          if (kc == OC_NCH - 1) mma_commit(accf + b);
        }
        __syncwarp();
        last_mma = t * OC_NCH + kc;
        if (++s == OC_STAGES) { s = 0; ph ^= 1; }
      }
      if (!ok) {
        if (lane == 0) { *abort_flag = 1; atomicExch(g.err, 1); }
        break;
      }
    }
  } else if (warp < OC_EPI_W0) {
    // ---------------------------------------------------------------- copies
    const int ct = tid - OC_CPY_W0 * 32;
    const int k = ct / OC_NO, oct = ct % OC_NO;
    const uint32_t dst0 = su32(sm) + OC_A + (uint32_t)oct * OC_OCT + (uint32_t)(k >> 3) * 128u + (uint32_t)(k & 7) * 16u;
    const int64_t plane = g.nn * g.ldn;   // elements of a digit plane
    int s = 0, sd = 0;                    // stage to fill, stage whose copies are waited for next
    uint32_t ph = 0;
    int64_t ch = 0, done = 0;             // chunks issued / announced
    bool ok = true;
    auto announce = [&]() {
      // this thread's copies of the oldest chunk have landed: make them visible to the
      // MMAs' reads and arrive
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bar_arrive(full + sd);
      if (++sd == OC_STAGES) sd = 0;
      ++done;
    };
    for (int64_t t = 0; t < my && ok && !*abort_flag; ++t) {
      const int64_t item = blockIdx.x + t * gridDim.x;
      const int64_t e = item / g.ntiles;
      const int c0 = (int)(item % g.ntiles) * OC_TW;
      const int no = min(OC_TW, g.ldn - c0) / 8;
      const int ci = (int)(e % g.m.nc[0]), cj = (int)((e / g.m.nc[0]) % g.m.nc[1]),
                ck = (int)(e / ((int64_t)g.m.nc[0] * g.m.nc[1]));
      const int64_t g0 = (int64_t)(P * ci) + (int64_t)g.m.nn[0] * ((int64_t)(P * cj) + (int64_t)g.m.nn[1] * (P * ck));
      const uint16_t* src0 = g.D + g0 * g.ldn + c0 + 8 * oct;
      for (int kc = 0; kc < OC_NCH; ++kc) {
        if (ch >= OC_STAGES) {
          ok = bar_wait(empty + s, ph ^ 1u);
          if (!ok) break;
        }
        if (ct == 0) {
          bar_expect_tx(full + s, OC_A);
          bulk_g2s(sm + (uint32_t)s * OC_STAGE, g.Aimg + (e * OC_NCH + kc) * (int64_t)OC_A, OC_A, full + s);
          last_copy = ch;
        }
        if (oct < no) {
          const int ko = koff[kc * OZ_KC + k];
          const uint16_t* src = src0 + (int64_t)max(ko, 0) * g.ldn;
          const uint32_t dst = dst0 + (uint32_t)s * OC_STAGE;
#pragma unroll
          for (int i = 0; i < OZ_S; ++i) cp16(dst + (uint32_t)i * OC_BSL, src + i * plane, ko >= 0);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        ++ch;
        if (++s == OC_STAGES) { s = 0; ph ^= 1; }
        if (ch > OC_DEPTH) {
          asm volatile("cp.async.wait_group %0;" ::"n"(OC_DEPTH) : "memory");
          announce();
        }
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    while (done < ch) announce();
    if (!ok) {
      *abort_flag = 1;
      atomicExch(g.err, 1);
    }
  } else if (warp >= OC_EPI_W0) {
    // ---------------------------------------------------------------- epilogue
    const int quarter = warp & 3;   // the TMEM lane quarter this warp may read
    const int part = (warp - OC_EPI_W0) >> 2;
    const int r = quarter * 32 + lane;
    for (int64_t t = 0; t < my && !warp_aborted(abort_flag); ++t) {
      const int64_t item = blockIdx.x + t * gridDim.x;
      const int64_t e = item / g.ntiles;
      const int c0 = (int)(item % g.ntiles) * OC_TW;
      const int ncol = min(OC_TW, g.ldn - c0);
      const int b = (int)(t & 1);
      const int Er = g.hexp[e * OZ_M + r];
      double* out = g.P + (e * NL + r) * (int64_t)g.ldn + c0;
      if (!warp_wait(accf + b, (uint32_t)((t / 2) & 1))) {
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
  // all roles done.  After an abort every bulk copy still in flight lands (the copy
  // threads announced all their own copies, and at most the last OC_STAGES chunks are
  // outstanding) and the last MMA commit (it covers every MMA this CTA issued) arrives
  // before the TMEM and the shared memory are released; each drain wait is bounded like
  // the pipeline's own.
  __syncthreads();
  if (*abort_flag) {
    if (last_copy >= 0)
      for (int64_t ch = max(last_copy - OC_STAGES + 1, (int64_t)0); ch <= last_copy; ++ch)
        if (!bar_wait(full + (int)(ch % OC_STAGES), (uint32_t)((ch / OC_STAGES) & 1))) break;
    if (warp == 0 && lane == 0 && last_mma >= 0)
      bar_wait(empty + (int)(last_mma % OC_STAGES), (uint32_t)((last_mma / OC_STAGES) & 1));
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM_COLS) : "memory");
  }
}

// W[node][c] = sum of the cell products around the node in the order of the parity
// colours; a block of 16 nodes x 16 threads of CPT column pairs 32 columns apart.  (A warp per
// node with its eight row pointers found once took 2.5 times as long: seven of eight
// are absent for most nodes, and their tests sat between the loads.)
template <int CPT>
__global__ void __launch_bounds__(256) k_ozc_gather(MeshDev m, int64_t nn, const double* __restrict__ Pc, int ldn, int nc,
                                                    double* __restrict__ W, int64_t ldw) {
  const int64_t gn = blockIdx.x * 16LL + threadIdx.y;
  const int c0 = blockIdx.y * 32 * CPT + threadIdx.x * 2;
  if (gn >= nn || c0 >= nc) return;
  const int G[3] = {(int)(gn % m.nn[0]), (int)((gn / m.nn[0]) % m.nn[1]), (int)(gn / ((int64_t)m.nn[0] * m.nn[1]))};
  int hi[3];
  bool two[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    hi[d] = min(G[d] / P, m.nc[d] - 1);
    two[d] = G[d] % P == 0 && G[d] > 0 && G[d] / P < m.nc[d];
  }
  double2 s[CPT];
#pragma unroll
  for (int u = 0; u < CPT; ++u) s[u] = make_double2(0.0, 0.0);
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
    const double* row = Pc + (e * NL + l[0] + NP1 * (l[1] + NP1 * l[2])) * (int64_t)ldn + c0;
#pragma unroll
    for (int u = 0; u < CPT; ++u)
      if (c0 + 32 * u < nc) {
        const double2 p = *reinterpret_cast<const double2*>(row + 32 * u);
        s[u].x += p.x;
        s[u].y += p.y;
      }
  }
  double* w = W + gn * ldw + c0;
#pragma unroll
  for (int u = 0; u < CPT; ++u) {
    if (c0 + 32 * u < nc) w[32 * u] = s[u].x;
    if (c0 + 32 * u + 1 < nc) w[32 * u + 1] = s[u].y;
  }
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
  const int64_t nn = (int64_t)m.nn[0] * m.nn[1] * m.nn[2];
  const int ldn = pad16(N);
  const int64_t ns = nn * (ldn / 8);
  k_ozc_slice<<<(unsigned)((ns + 255) / 256), 256, 0, st>>>(Y, ldy, nn, N, ldn, fexp, reinterpret_cast<uint16_t*>(digits));
  OzCellArgs a{};
  a.Aimg = Aimg;
  a.hexp = hexp;
  a.fexp = fexp;
  a.D = reinterpret_cast<const uint16_t*>(digits);
  a.n_cell = n_cell;
  a.nn = nn;
  a.m = m;
  a.P = products;
  a.ldn = ldn;
  a.ntiles = (ldn + OC_TW - 1) / OC_TW;
  a.err = err;
  a.stall = stall;
  const int64_t items = n_cell * a.ntiles;
  if (cudaFuncSetAttribute(k_ozc_cell, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OC_SMEM) != cudaSuccess) return 1;
  k_ozc_cell<<<(unsigned)std::min<int64_t>(items, n_sm), OC_THREADS, OC_SMEM, st>>>(a);
  if (N > 32)
    k_ozc_gather<2><<<dim3((unsigned)((nn + 15) / 16), (unsigned)((N + 63) / 64)), dim3(16, 16), 0, st>>>(m, nn, products,
                                                                                                       ldn, N, W, ldw);
  else
    k_ozc_gather<1><<<(unsigned)((nn + 15) / 16), dim3(16, 16), 0, st>>>(m, nn, products, ldn, N, W, ldw);
  g_launches.fetch_add(3, std::memory_order_relaxed);
  return 0;
}

}  // namespace efe
