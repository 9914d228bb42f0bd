// FP64-grade products on the BF16 tensor cores by error-free slicing (Ozaki scheme;
// Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 59, 2012), sm_103a tcgen05.
//
// Each FP64 operand row (of A) / column (of B) is scaled by a power of two so
// that its largest entry is below 1 in magnitude, truncated to 49 bits, and cut
// into seven signed 7-bit digits d_1..d_7 (x ~ 2^E sum_i d_i 2^-7i).  Digit i
// is stored in BF16 as d_i 2^-7(i-1) (exact: 7 significant bits).  The product
// sum_k a_i b_j of digit slices has weight 2^-7(i+j-2); for a fixed t = i + j
// every partial sum is an integer multiple of 2^-7(t-2) below 2^24 of that
// unit (K <= 256 per accumulation group, at most four pairs, digits below 2^7 in
// magnitude: 4 * 256 * 127^2 < 2^24), so the FP32 tensor-core accumulators
// for t = 2, 3, 4, 5 are exact.  The pairs with t = 6..8 share a fifth
// accumulator (their FP32 rounding is below 2^-52 of the result); pairs with
// t > 8 fall below the 49-bit truncation and are dropped.  The epilogue adds
// the five accumulators with error-free FP32 sums into a (hi, lo) pair and
// forms the FP64 result 2^(E_A + E_B - 14) (hi + lo).  The error is within a
// few units of 2^-48 of sum_k |a_k||b_k|, comparable to FP64 GEMM rounding.
//
// Products of this file (the cell products are in efe_oz_cell.cu):
//   ROWS  C = A B for a tall A (rows x K) and a small B (K x N); K is taken in
//         groups of 256 (exact FP32 sums for t <= 5);
//   GRAM  C = A^T B for tall A, B (K x Na, K x N, K large): items are (tile
//         pair, K segment); each segment is formed in such groups of 256 rows, and a
//         fixed-order FP64 reduction adds the segments' partial tiles.
// The groups of an item are added in FP32 (hi, lo) pairs in registers (error-free sum of the
// high parts, renormalised): each addition rounds within 2^-45 of the sum so far (two FP32
// roundings of a low part up to 2^-22 of it; a few 2^-48 in the mean), so a segment of G groups
// within G 2^-45.  The FP64 value is formed once per item.
// Both operands are cut once per product into digit images (k_oz_img_rows /
// k_oz_img_cols) and arrive in the stages by bulk asynchronous copies; the digit
// images of the cell matrices (k_oz_preslice, once per potential) are made here too.
//
// Warp roles (512 threads): warp 0 issues the MMAs (one elected lane), one lane of
// warp 1 the copies into four stages, warps 4-15 combine the accumulators and write
// the result.  All waits are bounded (about one second); on timeout the CTA records
// an error and leaves.
#include <stdint.h>

#include <algorithm>
#include <vector>

#include "efe_kernels.h"
#include "efe_oz.cuh"

namespace efe {

namespace {

constexpr int OZ_TW = 96;          // column tile
constexpr int OZ_ROWS_KG = 16;     // ROWS: 16-wide K chunks per exact accumulation group (K <= 256)
constexpr int OZ_STAGES = 4;
constexpr int OZ_EPI_W0 = 4, OZ_EPI_WN = 12;   // epilogue warps
constexpr int OZ_THREADS = 16 * 32;            // 16 warps: 128 registers a thread

struct OzL {
  static constexpr uint32_t ASL = OZ_M * OZ_KC * 2;        // one slice of 128 rows, 4 KB
  static constexpr uint32_t GRP = OZ_S * 256;              // eight rows (columns) of a chunk: seven slices of 256 B
  static constexpr uint32_t A = OZ_M / 8 * GRP;            // 28 KB
  static constexpr uint32_t STAGE = A + OZ_TW / 8 * GRP;   // 49 KB
  static constexpr uint32_t BARS = OZ_STAGES * STAGE;
  static constexpr uint32_t STG = BARS + 256;                // epilogue staging: up to 12 warps x 32 rows x 9 doubles
  static constexpr size_t TOTAL = (size_t)STG + 12 * 32 * 9 * 8;
};

// cell images, K-major, no swizzle, BF16: core matrix 8 rows x 16 B, the next 8 K 128 B and
// the next 8 rows 256 B further
__device__ __forceinline__ uint32_t bo(int row, int k) {
  return (uint32_t)(row >> 3) * 256u + (uint32_t)(k >> 3) * 128u + (uint32_t)(row & 7) * 16u + (uint32_t)(k & 7) * 2u;
}
// operand images of this file: [chunk][8 rows][slice][8 K][row of 16 B], so that any run of
// rows of a chunk is one contiguous piece with all its slices and one bulk copy brings an
// operand's chunk.  (Slice-major 128-column tiles took 8 or, across two tiles, 15 copies a
// chunk, and their issue, about 120 cycles each, outlasted the chunk's 28 MMAs.  The products
// of a Rayleigh-Ritz of 559 k rows x 640 columns, with the segment rule of the Gram products
// below: 81 -> 69 ms, of 559 k x 135: 8.0 -> 5.8 ms.)  Slice i of row r, K octet o:
__device__ __forceinline__ uint32_t go(int row, int i, int oct) {
  return (uint32_t)(row >> 3) * OzL::GRP + (uint32_t)i * 256u + (uint32_t)oct * 128u + (uint32_t)(row & 7) * 16u;
}
// LBO = 128 B (next 8 K), SBO = GRP (next 8 rows)
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(OzL::GRP >> 4) << 32) |
         ((uint64_t)1 << 46);
}
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ uint32_t idesc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(OZ_M >> 4) << 24);
}
// digits of eight values with scale exponent E, packed slice by slice (two BF16
// per word): pk[i] holds digit i of x[0..7] in K order
__device__ __forceinline__ void oz_pack8(const double (&x)[8], int E, uint32_t (&pk)[OZ_S][4]) {
#pragma unroll
  for (int i = 0; i < OZ_S; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) pk[i][q] = 0u;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const long long bits = __double_as_longlong(x[q]);
    const int ex = (int)((bits >> 52) & 0x7FF);
    const uint32_t sgn = (uint32_t)((bits >> 48) & 0x8000);
    unsigned long long qq = 0;
    const int rs = 1026 + E - ex;
    if (ex != 0 && rs >= 0 && rs < 64) qq = ((unsigned long long)(bits & 0xFFFFFFFFFFFFFull) | (1ull << 52)) >> rs;
#pragma unroll
    for (int i = 0; i < OZ_S; ++i) {
      const uint32_t d = (uint32_t)(qq >> (42 - 7 * i)) & 127u;
      uint32_t h16 = 0;
      if (d) {
        const int p = 31 - __clz(d);
        h16 = sgn | ((uint32_t)(p + 127 - 7 * i) << 7) | ((d << (7 - p)) & 0x7Fu);
      }
      pk[i][q >> 1] |= h16 << (16 * (q & 1));
    }
  }
}

struct OzArgs {
  int mode;                 // 1: ROWS, 2: GRAM
  // ROWS: C (arows x N) = A (arows x K) B (K x N)
  int64_t arows;
  const int* aexp;          // per row of A
  // common
  int K;                    // reduction length of ROWS (in groups of 256)
  const int* fexp;          // per column of B
  double* out;              // ROWS: C
  int64_t ldo;
  int N, ntiles;
  int* err;
  // GRAM: C = A^T B with A (Kbig x Na), B (Kbig x N); aexp / fexp per column of A / B;
  // work items = (tile pair, K segment of seg_len rows); FP64 partial tiles to
  // part[segment][Na][N]
  int64_t seg_len;
  int Na, nseg, npairs;
  const int2* pairs;        // (M tile, N tile) of every item pair
  double* part;
  // pre-sliced operand images (k_oz_img_rows / k_oz_img_cols).  ROWS: Aimg = row image
  // of A, Bimg = column image of B; GRAM: both column images.  astep, bstep: bytes of a
  // chunk of a column image.
  const unsigned char* Aimg;
  const unsigned char* Bimg;
  int64_t astep, bstep;
  int stall;                // tests only (EFE_OPT_TEST_STALL)
};

// work item of a CTA: row block / tile pair and its K range
struct OzItem {
  int64_t ia, m0, kb;
  int c0, ncol, nmma, seg;
};

__device__ __forceinline__ OzItem oz_item(const OzArgs& g, int64_t item) {
  OzItem it;
  if (g.mode == 2) {
    // segment-major: the CTAs running at one time share a segment's rows, so the
    // operand images of that segment are read from L2 by every tile pair
    const int64_t pr = item % g.npairs;
    it.seg = (int)(item / g.npairs);
    const int2 tp = g.pairs[pr];
    it.ia = pr;
    it.m0 = (int64_t)tp.x * OZ_M;
    it.c0 = tp.y * OZ_TW;
    it.kb = (int64_t)it.seg * g.seg_len;
  } else {
    it.ia = item / g.ntiles;
    it.c0 = (int)(item % g.ntiles) * OZ_TW;
    it.m0 = it.ia * OZ_M;
    it.kb = 0;
    it.seg = 0;
  }
  it.ncol = min(OZ_TW, g.N - it.c0);
  it.nmma = ((it.ncol + 15) / 16) * 16;
  return it;
}

__global__ void __launch_bounds__(OZ_THREADS, 1) k_oz(OzArgs g) {
  extern __shared__ __align__(1024) unsigned char sm[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  __shared__ int s_skip;
  if (tid == 0) s_skip = *(volatile int*)g.err;
  __syncthreads();
  if (s_skip) return;
  uint64_t* afull = reinterpret_cast<uint64_t*>(sm + OzL::BARS);  // [stages] operand chunks landed
  uint64_t* empty = afull + OZ_STAGES;                           // [stages] MMAs done with the stage
  uint64_t* accf = afull + 2 * OZ_STAGES;
  uint64_t* acce = accf + 1;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(accf + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(accf + 3);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)),
                 "r"(OZ_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    for (int s = 0; s < OZ_STAGES; ++s) {
      bar_init(empty + s, 1 + (g.stall == 2));
      bar_init(afull + s, 1 + (g.stall == 1));
    }
    bar_init(accf, 1 + (g.stall == 3));
    bar_init(acce, OZ_EPI_WN * 32);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const int64_t nA = (g.arows + OZ_M - 1) / OZ_M;
  const int64_t nitems = (g.mode == 2) ? (int64_t)g.npairs * g.nseg : nA * g.ntiles;
  const int64_t my = nitems > blockIdx.x ? (nitems - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  // chunks of 16 K per item; the accumulators are drained every gsz chunks
  // (GRAM: every 256 rows, ROWS: every 256 K, where the FP32 sums of t <= 5 are
  // still exact); later groups add to the result
  const int nch = (g.mode == 2) ? (int)(g.seg_len / OZ_KC) : (g.K + OZ_KC - 1) / OZ_KC;
  const int gsz = (g.mode == 2) ? 16 : min(nch, OZ_ROWS_KG);
  const int ngrp = (nch + gsz - 1) / gsz;
  // the last chunk whose MMAs this thread committed / whose bulk copies it issued
  // (drained before the TMEM and shared memory are released after an abort)
  int64_t last_mma = -1, last_copy = -1;

  if (warp == 0) {
    // ---------------------------------------------------------------- MMA issuer
    for (int64_t t = 0; t < my && !warp_aborted(abort_flag); ++t) {
      const int64_t item = blockIdx.x + t * gridDim.x;
      const OzItem it = oz_item(g, item);
      const int nmma = it.nmma;
      bool ok = true;
      for (int kc = 0; kc < nch && ok; ++kc) {
        const int64_t gc = t * ngrp + kc / gsz;   // accumulator group counter
        if (kc % gsz == 0) {
          if (gc >= 1) ok = warp_wait(acce, (uint32_t)((gc - 1) & 1));
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          if (!ok) break;
        }
        const int64_t ch = t * nch + kc;
        const int s = (int)(ch % OZ_STAGES);
        ok = warp_wait(afull + s, (uint32_t)((ch / OZ_STAGES) & 1));
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!ok) break;
        const uint32_t sA = su32(sm) + (uint32_t)s * OzL::STAGE, sB = sA + OzL::A;
        if (elect_one()) {
          const uint32_t id = idesc_bf16(nmma);
          bool first[OZ_NACC] = {true, true, true, true, true};
#pragma unroll
          for (int tt = 2; tt <= 8; ++tt) {
            const int a = tt <= 5 ? tt - 2 : 4;
#pragma unroll
            for (int i = 1; i < tt; ++i) {
              const int j = tt - i;
              if (i > OZ_S || j > OZ_S) continue;
              const uint32_t acc = (kc % gsz > 0 || !first[a]) ? 1u : 0u;
              first[a] = false;
              mma_bf16(tmem + (uint32_t)(a * OZ_TW), sdesc(sA + (uint32_t)(i - 1) * 256u),
                       sdesc(sB + (uint32_t)(j - 1) * 256u), id, acc);
            }
          }
          mma_commit(empty + s);
          if (kc % gsz == gsz - 1 || kc == nch - 1) mma_commit(accf);
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
    for (int64_t t = 0; t < my && !*abort_flag; ++t) {
      const OzItem it = oz_item(g, blockIdx.x + t * gridDim.x);
      const int c0 = it.c0, nmma = it.nmma;
      bool ok = true;
      for (int kc = 0; kc < nch; ++kc) {
        const int64_t ch = t * nch + kc;
        const int s = (int)(ch % OZ_STAGES);
        if (ch >= OZ_STAGES) {
          ok = bar_wait(empty + s, (uint32_t)((ch / OZ_STAGES - 1) & 1));
          if (!ok) break;
        }
        unsigned char* SA = sm + s * OzL::STAGE;
        // one bulk copy an operand and chunk: rows m0 .. of A's, columns c0 .. of B's image
        const int64_t kA = (g.mode == 2) ? it.kb / OZ_KC + kc : kc;
        const uint32_t la = (g.mode == 2) ? (uint32_t)((min((int64_t)OZ_M, (int64_t)g.Na - it.m0) + 7) / 8) * OzL::GRP
                                          : OzL::A;
        const uint32_t lb = (uint32_t)(nmma / 8) * OzL::GRP;
        bar_expect_tx(afull + s, la + lb);
        bulk_g2s(SA, (g.mode == 2) ? g.Aimg + kA * g.astep + (it.m0 / 8) * OzL::GRP
                                   : g.Aimg + (it.ia * (int64_t)nch + kA) * OzL::A, la, afull + s);
        bulk_g2s(SA + OzL::A, g.Bimg + kA * g.bstep + (int64_t)(c0 / 8) * OzL::GRP, lb, afull + s);
        last_copy = ch;
      }
      if (!ok) {
        *abort_flag = 1;
        atomicExch(g.err, 1);
        break;
      }
    }
  } else if (warp >= OZ_EPI_W0) {
    // ---------------------------------------------------------------- epilogue
    // each thread owns one accumulator row (its TMEM lane); an 8-column block of
    // results goes through a per-warp shared tile so that the global loads and
    // stores run along the rows (8 consecutive values per row, 4 rows per
    // instruction) instead of one row per lane
    const int quarter = warp & 3;   // the TMEM lane quarter this warp may read
    const int r = quarter * 32 + lane;
    const int ew = warp - OZ_EPI_W0, part = ew >> 2, nparts = OZ_EPI_WN >> 2;   // column blocks part, part + nparts, ...
    double* stg = reinterpret_cast<double*>(sm + OzL::STG) + ew * (32 * 9);
    for (int64_t t = 0; t < my && !warp_aborted(abort_flag); ++t) {
      const OzItem it = oz_item(g, blockIdx.x + t * gridDim.x);
      const int c0 = it.c0, ncol = it.ncol;
      bool live;
      int Er;
      double* orow;
      if (g.mode == 1) {
        const int64_t row = it.m0 + r;
        live = row < g.arows;
        Er = live ? g.aexp[row] : 0;
        orow = live ? g.out + row * g.ldo + c0 : nullptr;
      } else {
        const int64_t row = it.m0 + r;
        live = row < g.Na;
        Er = live ? g.aexp[row] : 0;
        orow = live ? g.part + ((int64_t)it.seg * g.Na + row) * g.N + c0 : nullptr;
      }
      // Every K group's sum is added
      // into FP32 (hi, lo) pairs held in registers (error-free two-sum, then a
      // renormalisation: about 48 bits), so the TMEM accumulators are released
      // as soon as they are read and the next group's MMAs run while this
      // thread does its arithmetic; the FP64 result is formed and written once
      // per item.  Twelve epilogue warps: at most four 8-column blocks a thread.
      constexpr int MAXB = 4;
      float hi[MAXB][8], lo[MAXB][8];
      bool stop = false;
      for (int grp = 0; grp < ngrp; ++grp) {
        const int64_t gc = t * ngrp + grp;
        if (!warp_wait(accf, (uint32_t)(gc & 1))) {
          *abort_flag = 1;
          atomicExch(g.err, 1);
          stop = true;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int j = 0; j < MAXB; ++j) {
          const int cb = 8 * part + 8 * nparts * j;
          if (cb >= ncol) break;
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {   // four columns at a time (fewer live registers)
            uint32_t v[OZ_NACC][4];
#pragma unroll
            for (int a = 0; a < OZ_NACC; ++a)
              asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                           : "=r"(v[a][0]), "=r"(v[a][1]), "=r"(v[a][2]), "=r"(v[a][3])
                           : "r"(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(a * OZ_TW + cb + 4 * hh))
                           : "memory");
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int qq = 0; qq < 4; ++qq) {
              const int q = 4 * hh + qq;
              float s1, e1, s2, e2, s3, e3;
              two_sum(__uint_as_float(v[0][qq]), __uint_as_float(v[1][qq]), s1, e1);
              two_sum(s1, __uint_as_float(v[2][qq]), s2, e2);
              two_sum(s2, __uint_as_float(v[3][qq]), s3, e3);
              const float lg = ((__uint_as_float(v[4][qq]) + e3) + e2) + e1;
              if (grp == 0) {
                hi[j][q] = s3;
                lo[j][q] = lg;
              } else {
                float sh, eh;
                two_sum(hi[j][q], s3, sh, eh);
                const float l = (lo[j][q] + lg) + eh;
                hi[j][q] = sh + l;
                lo[j][q] = l - (hi[j][q] - sh);
              }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        bar_arrive(acce);
      }
      if (stop) break;
      const unsigned long long orow_u = (unsigned long long)orow;
#pragma unroll
      for (int j = 0; j < MAXB; ++j) {
        const int cb = 8 * part + 8 * nparts * j;
        if (cb >= ncol) break;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int n = cb + q;
          double val = 0.0;
          if (live && n < ncol) {
            const int k2 = Er + g.fexp[c0 + n] - 14;
            val = f32_scaled(hi[j][q], k2) + f32_scaled(lo[j][q], k2);
          }
          stg[lane * 9 + q] = val;
        }
        __syncwarp();
        // row rr = 4 jj + lane / 8 of this warp, column cb + lane % 8
#pragma unroll
        for (int jj = 0; jj < 8; ++jj) {
          const int rr = 4 * jj + (lane >> 3), cq = lane & 7;
          double* rp = (double*)__shfl_sync(0xffffffffu, orow_u, rr);
          const int lv = __shfl_sync(0xffffffffu, (int)live, rr);
          if (lv && cb + cq < ncol) rp[cb + cq] = stg[rr * 9 + cq];
        }
        __syncwarp();
      }
    }
  }
  // all roles done.  After an abort, drain before the TMEM and the shared memory
  // are released: every bulk copy still in flight into the stage ring lands (the copy
  // thread issues into a stage only after its MMAs released it, so at most the last
  // OZ_STAGES chunks are outstanding), and the last MMA commit -- which covers every
  // MMA this CTA issued -- arrives.  Each drain wait is bounded like the pipeline's own;
  // after one that ran out there is nothing left to wait for.
  __syncthreads();
  if (*abort_flag) {
    if (last_copy >= 0) {
      for (int64_t ch = last_copy - OZ_STAGES + 1; ch <= last_copy; ++ch)
        if (ch >= 0 && !bar_wait(afull + (int)(ch % OZ_STAGES), (uint32_t)((ch / OZ_STAGES) & 1))) break;
    }
    if (warp == 0 && lane == 0 && last_mma >= 0)
      bar_wait(empty + (int)(last_mma % OZ_STAGES), (uint32_t)((last_mma / OZ_STAGES) & 1));
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(OZ_TMEM_COLS) : "memory");
  }
}

// Digit images of every H^cc_e: per cell, per 16-wide K chunk, the seven 4 KB
// BF16 slices in the shared-memory layout of the MMA operand (row exponents hexp).
__global__ void k_oz_preslice(const double* __restrict__ H, const int* __restrict__ hexp, int64_t n_cell,
                              unsigned char* __restrict__ img) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;   // (cell, row, K octet)
  const int nch = (NL + OZ_KC - 1) / OZ_KC;
  if (t >= n_cell * OZ_M * nch * 2) return;
  const int oct = (int)(t % 2);
  const int kc = (int)((t / 2) % nch);
  const int row = (int)((t / (2 * nch)) % OZ_M);
  const int64_t e = t / (2 * nch * OZ_M);
  const int E = hexp[e * OZ_M + row];
  uint32_t pk[OZ_S][4];
#pragma unroll
  for (int i = 0; i < OZ_S; ++i)
#pragma unroll
    for (int q = 0; q < 4; ++q) pk[i][q] = 0u;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = kc * OZ_KC + oct * 8 + q;
    const double x = (row < NL && k < NL) ? H[e * (int64_t)(NL * NL) + row * NL + k] : 0.0;
    const long long bits = __double_as_longlong(x);
    const int ex = (int)((bits >> 52) & 0x7FF);
    const uint32_t sgn = (uint32_t)((bits >> 48) & 0x8000);
    unsigned long long qq = 0;
    const int rs = 1026 + E - ex;
    if (ex != 0 && rs >= 0 && rs < 64) qq = ((unsigned long long)(bits & 0xFFFFFFFFFFFFFull) | (1ull << 52)) >> rs;
#pragma unroll
    for (int i = 0; i < OZ_S; ++i) {
      const uint32_t d = (uint32_t)(qq >> (42 - 7 * i)) & 127u;
      uint32_t h16 = 0;
      if (d) {
        const int p = 31 - __clz(d);
        h16 = sgn | ((uint32_t)(p + 127 - 7 * i) << 7) | ((d << (7 - p)) & 0x7Fu);
      }
      pk[i][q >> 1] |= h16 << (16 * (q & 1));
    }
  }
  unsigned char* base = img + ((e * nch + kc) * OZ_S) * (int64_t)OzL::ASL + bo(row, oct * 8);
#pragma unroll
  for (int i = 0; i < OZ_S; ++i)
    *reinterpret_cast<uint4*>(base + (int64_t)i * OzL::ASL) = make_uint4(pk[i][0], pk[i][1], pk[i][2], pk[i][3]);
}

// Row image of a tall A (rows x K, the A operand of ROWS): per 128-row tile and
// 16-wide K chunk the seven BF16 slices of its rows in the shared-memory layout of
// the MMA operand (row exponents aexp); rows past `rows` are zero.  One thread
// per (tile row, K octet); a warp covers 32 rows of one octet.
__global__ void k_oz_img_rows(const double* __restrict__ A, int64_t lda, int64_t rows, int K,
                              const int* __restrict__ aexp, unsigned char* __restrict__ img) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int nch = (K + OZ_KC - 1) / OZ_KC;
  const int64_t ntile = (rows + OZ_M - 1) / OZ_M;
  if (t >= ntile * nch * 2 * OZ_M) return;
  const int rr = (int)(t % OZ_M);
  const int oct = (int)((t / OZ_M) & 1);
  const int64_t tc = t / (2 * OZ_M);   // tile * nch + chunk
  const int c = (int)(tc % nch);
  const int64_t r = (tc / nch) * OZ_M + rr;
  double x[8];
  const int E = r < rows ? aexp[r] : -2000;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = c * OZ_KC + oct * 8 + q;
    x[q] = (r < rows && k < K) ? A[r * lda + k] : 0.0;
  }
  uint32_t pk[OZ_S][4];
  oz_pack8(x, E, pk);
  unsigned char* base = img + tc * (int64_t)OzL::A + go(rr, 0, oct);
#pragma unroll
  for (int i = 0; i < OZ_S; ++i)
    *reinterpret_cast<uint4*>(base + i * 256) = make_uint4(pk[i][0], pk[i][1], pk[i][2], pk[i][3]);
}

// Column image of A (Krows x ncols): the K-major operand A^T, element (m, k) =
// A[k][m], per 16-row chunk (nch of them, rows past Krows zero) all columns, padded to
// 128, with their seven slices in the MMA layout (column exponents cexp).
// Columns past ncols rounded up to 16 are not written.  A warp reads 32
// consecutive columns of one row.
__global__ void k_oz_img_cols(const double* __restrict__ A, int64_t lda, int64_t Krows, int ncols,
                              const int* __restrict__ cexp, int64_t nch, unsigned char* __restrict__ img) {
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int ntile = (ncols + OZ_M - 1) / OZ_M;
  if (t >= (int64_t)ntile * nch * 2 * OZ_M) return;
  const int m = (int)(t % OZ_M);
  const int oct = (int)((t / OZ_M) & 1);
  const int64_t tc = t / (2 * OZ_M);   // chunk * ntile + tile
  const int64_t c = tc / ntile;
  const int col = (int)(tc % ntile) * OZ_M + m;
  if (col >= ((ncols + 15) & ~15)) return;
  const int E = col < ncols ? cexp[col] : -2000;
  double x[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int64_t k = c * OZ_KC + oct * 8 + q;
    x[q] = (col < ncols && k < Krows) ? A[k * lda + col] : 0.0;
  }
  uint32_t pk[OZ_S][4];
  oz_pack8(x, E, pk);
  unsigned char* base = img + c * (int64_t)ntile * OzL::A + go(col, 0, oct);
#pragma unroll
  for (int i = 0; i < OZ_S; ++i)
    *reinterpret_cast<uint4*>(base + i * 256) = make_uint4(pk[i][0], pk[i][1], pk[i][2], pk[i][3]);
}

// per-row scale exponents of an FP64 matrix (one warp per row)
__global__ void k_oz_rowexp(const double* __restrict__ A, int64_t lda, int64_t rows, int K, int* __restrict__ eout) {
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= rows) return;
  int E = -2000;
  for (int k = lane; k < K; k += 32) E = max(E, exp_of(A[w * lda + k]));
  for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_down_sync(0xffffffffu, E, o));
  if (lane == 0) eout[w] = E;
}

// per-column scale exponents (max over rows), combined with integer atomicMax;
// blockIdx.x: a range of rows, blockIdx.y: a range of blockDim.x columns
__global__ void k_oz_colexp(const double* __restrict__ Y, int64_t ldy, int64_t rows, int N, int rows_per_block,
                            int* __restrict__ fout) {
  const int64_t r0 = (int64_t)blockIdx.x * rows_per_block;
  const int64_t r1 = min(rows, r0 + rows_per_block);
  const int c = blockIdx.y * blockDim.x + threadIdx.x;
  if (c >= N) return;
  int E = -2000;
  for (int64_t r = r0; r < r1; ++r) E = max(E, exp_of(Y[r * ldy + c]));
  atomicMax(fout + c, E);
}

__global__ void k_oz_fill(int* p, int n, int v) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

// row exponents of every cell block (rows 125..127 of the padded block get -2000)
__global__ void k_oz_hexp(const double* __restrict__ H, int64_t n_cell, int* __restrict__ hexp) {
  const int64_t w = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= n_cell * OZ_M) return;
  const int64_t e = w / OZ_M;
  const int r = (int)(w % OZ_M);
  int E = -2000;
  if (r < NL)
    for (int k = lane; k < NL; k += 32) E = max(E, exp_of(H[e * (int64_t)(NL * NL) + r * NL + k]));
  for (int o = 16; o > 0; o >>= 1) E = max(E, __shfl_down_sync(0xffffffffu, E, o));
  if (lane == 0) hexp[w] = E;
}

int oz_launch(const OzArgs& a, int n_sm, cudaStream_t st) {
  const int64_t items = (a.mode == 2) ? (int64_t)a.npairs * a.nseg : (a.arows + OZ_M - 1) / OZ_M * a.ntiles;
  if (items <= 0) return 0;
  cudaFuncSetAttribute(k_oz, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OzL::TOTAL);
  k_oz<<<(unsigned)(items < n_sm ? items : n_sm), OZ_THREADS, OzL::TOTAL, st>>>(a);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return 0;
}

}  // namespace

int64_t oz_hexp_elems(int64_t n_cell) { return n_cell * OZ_M; }

void launch_oz_hexp(const double* Hcc, int64_t n_cell, int* hexp, cudaStream_t st) {
  const int64_t w = n_cell * OZ_M;
  if (w <= 0) return;
  k_oz_hexp<<<(unsigned)((w * 32 + 255) / 256), 256, 0, st>>>(Hcc, n_cell, hexp);
  g_launches.fetch_add(1, std::memory_order_relaxed);
}

void launch_oz_colexp(const double* Y, int64_t ldy, int64_t rows, int N, int* fexp, cudaStream_t st) {
  if (N <= 0) return;
  k_oz_fill<<<(N + 255) / 256, 256, 0, st>>>(fexp, N, -2000);
  // about eight CTAs per SM, each thread on at most 2048 rows of one column
  const int bt = N >= 128 ? 128 : 64;
  const int64_t ncb = (N + bt - 1) / bt;
  const int64_t want = 8LL * current_sm_count();
  const int64_t rpb = std::max<int64_t>(32, std::min<int64_t>(2048, (rows * ncb + want - 1) / want));
  const int64_t nb = (rows + rpb - 1) / rpb;
  if (nb > 0) k_oz_colexp<<<dim3((unsigned)nb, (unsigned)ncb), bt, 0, st>>>(Y, ldy, rows, N, (int)rpb, fexp);
  g_launches.fetch_add(2, std::memory_order_relaxed);
}

void launch_oz_rowexp(const double* A, int64_t lda, int64_t rows, int K, int* aexp, cudaStream_t st) {
  if (rows <= 0) return;
  k_oz_rowexp<<<(unsigned)((rows * 32 + 255) / 256), 256, 0, st>>>(A, lda, rows, K, aexp);
  g_launches.fetch_add(1, std::memory_order_relaxed);
}

// digit images of the cell matrices (operand A of the cell products, efe_oz_cell.cu)
int64_t oz_cell_image_bytes() { return (int64_t)((NL + OZ_KC - 1) / OZ_KC) * OZ_S * OzL::ASL; }

void launch_oz_preslice(const double* Hcc, const int* hexp, int64_t n_cell, unsigned char* img, cudaStream_t st) {
  const int64_t n = n_cell * OZ_M * ((NL + OZ_KC - 1) / OZ_KC) * 2;
  if (n <= 0) return;
  k_oz_preslice<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(Hcc, hexp, n_cell, img);
  g_launches.fetch_add(1, std::memory_order_relaxed);
}

int64_t oz_img_rows_bytes(int64_t rows, int K) {
  return ((rows + OZ_M - 1) / OZ_M) * ((K + OZ_KC - 1) / OZ_KC) * OZ_S * (int64_t)OzL::ASL;
}

int64_t oz_img_cols_bytes(int64_t nch, int ncols) {
  return (int64_t)((ncols + OZ_M - 1) / OZ_M) * nch * OZ_S * (int64_t)OzL::ASL;
}

void launch_oz_img_rows(const double* A, int64_t lda, int64_t rows, int K, const int* aexp, unsigned char* img,
                        cudaStream_t st) {
  const int64_t n = ((rows + OZ_M - 1) / OZ_M) * ((K + OZ_KC - 1) / OZ_KC) * 2 * OZ_M;
  if (n <= 0) return;
  k_oz_img_rows<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(A, lda, rows, K, aexp, img);
  g_launches.fetch_add(1, std::memory_order_relaxed);
}

void launch_oz_img_cols(const double* A, int64_t lda, int64_t Krows, int ncols, const int* cexp, int64_t nch,
                        unsigned char* img, cudaStream_t st) {
  const int64_t n = (int64_t)((ncols + OZ_M - 1) / OZ_M) * nch * 2 * OZ_M;
  if (n <= 0) return;
  k_oz_img_cols<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(A, lda, Krows, ncols, cexp, nch, img);
  g_launches.fetch_add(1, std::memory_order_relaxed);
}

// C = A B (A: rows x K; B: K x N), FP64-grade; aexp / bexp from
// launch_oz_rowexp(A) and launch_oz_colexp(B), Aimg / Bimg from
// launch_oz_img_rows(A) and launch_oz_img_cols(B, nch = ceil(K / 16)).
int launch_oz_rows(int64_t rows, int K, const int* aexp, const int* bexp, double* C, int64_t ldc, int N, int n_sm,
                   int* err, cudaStream_t st, const unsigned char* Aimg, const unsigned char* Bimg, int stall) {
  if (rows <= 0 || N <= 0 || K <= 0) return 0;
  OzArgs a{};
  a.Aimg = Aimg;
  a.Bimg = Bimg;
  a.mode = 1;
  a.arows = rows;
  a.aexp = aexp;
  a.K = K;
  a.fexp = bexp;
  a.out = C;
  a.ldo = ldc;
  a.N = N;
  a.ntiles = (N + OZ_TW - 1) / OZ_TW;
  a.bstep = oz_img_cols_bytes(1, N);
  a.err = err;
  a.stall = stall;
  return oz_launch(a, n_sm, st);
}

// C (Na x N) = A^T B for tall A (K x Na) and B (K x N), FP64-grade: the K rows
// are cut into segments (work items with the tile pairs), each segment's
// product is formed in 256-row groups (exact FP32 accumulation) and summed in
// FP64 into its partial tile; partials are then added in fixed order.  sym:
// C is symmetric, only tiles that meet the upper triangle are formed and the
// rest is mirrored.  aexp / bexp: launch_oz_colexp of A and B.  work: at least
// oz_gram_work_elems doubles; pairs_dev: at least oz_gram_max_pairs int2.
//
// Segment length, in 256-row groups: the one that ends first when the (tile pair, segment)
// items run n_sm at a time, an item costing its groups and half a group to fill and drain the
// pipeline.  Partials of at most max_seg segments fit the work array; more than 2 n_sm segments
// gain nothing.
int64_t oz_gram_seg_groups(int64_t groups, int npairs, int n_sm, int64_t max_seg) {
  int64_t best = groups;
  double best_cost = 1e300;
  max_seg = std::max<int64_t>(1, std::min<int64_t>(max_seg, 2 * (int64_t)n_sm));
  for (int64_t ns = std::min(groups, max_seg); ns >= 1; --ns) {
    const int64_t len = (groups + ns - 1) / ns, items = (groups + len - 1) / len * npairs;
    const double cost = (double)((items + n_sm - 1) / n_sm) * ((double)len + 0.5);
    if (cost <= best_cost) {
      best_cost = cost;
      best = len;
    }
  }
  return best;
}

// Doubles for the segment partials of an Na x N product: room for four 48 x 48 blocks an SM
// (11 MB on 152 SMs) or four whole products, whichever is more.  The first keeps the SMs busy up
// to about 300 columns, where one product's tile pairs are few: 559 k rows x 100 columns 6.34 ms
// in 7 segments, 0.91 in 76; x 200 11.1 ms in 4, 2.0 in 30; x 300 11.3 in 4, 3.5 in 16.
// Wider blocks keep four segments and idle SMs: at 640 columns 13 segments would take 8.0 ms for
// 12.0, at 400 4.8 for 5.7, but add the rows in another order, with which the vectors of the
// closest Ritz pairs turn.
int64_t oz_gram_work_elems(int Na, int N, int n_sm) {
  const int64_t one = (int64_t)Na * N;
  return std::max<int64_t>(4LL * n_sm * 48 * 48 + one, 4 * one);
}

int oz_gram_pairs(int Na, int N, bool sym, int2* pairs_host) {
  const int mt = (Na + OZ_M - 1) / OZ_M, nt = (N + OZ_TW - 1) / OZ_TW;
  int np = 0;
  for (int i = 0; i < mt; ++i)
    for (int j = 0; j < nt; ++j) {
      if (sym && i * OZ_M > j * OZ_TW + OZ_TW - 1) continue;   // tile entirely below the diagonal
      if (pairs_host) pairs_host[np] = make_int2(i, j);
      ++np;
    }
  return np;
}

namespace {
__global__ void k_oz_gram_reduce(int nseg, int Na, int N, const double* __restrict__ part, int sym, int accumulate,
                                 double* __restrict__ C, int64_t ldc) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= (int64_t)Na * N) return;
  const int i = (int)(idx / N), j = (int)(idx % N);
  const bool mirror = sym && i > j;
  const int64_t src = mirror ? (int64_t)j * N + i : idx;
  double s = accumulate ? C[(int64_t)i * ldc + j] : 0.0;
  for (int k = 0; k < nseg; ++k) s += part[(int64_t)k * Na * N + src];
  C[(int64_t)i * ldc + j] = s;
}
}  // namespace

int launch_oz_gram(int64_t K, int Na, int N, const double* A, int64_t lda, const int* aexp, const double* B,
                   int64_t ldb, const int* bexp, double* C, int64_t ldc, bool sym, double* work, int64_t work_elems,
                   int2* pairs_dev, int n_sm, int* err, cudaStream_t st, unsigned char* img_a,
                   int64_t img_a_bytes, unsigned char* img_b, int64_t img_b_bytes, bool accumulate, int stall) {
  if (K <= 0 || Na <= 0 || N <= 0) return 0;
  if (sym && Na != N) return 1;
  std::vector<int2> pairs(oz_gram_pairs(Na, N, sym, nullptr));
  const int np = oz_gram_pairs(Na, N, sym, pairs.data());
  if ((int64_t)Na * N > work_elems) return 1;
  const int64_t groups = (K + 255) / 256;
  const int64_t seg_len = 256 * oz_gram_seg_groups(groups, np, n_sm, work_elems / ((int64_t)Na * N));
  const int64_t nseg = (K + seg_len - 1) / seg_len;
  if (cudaMemcpyAsync(pairs_dev, pairs.data(), sizeof(int2) * np, cudaMemcpyHostToDevice, st) != cudaSuccess) return 1;
  OzArgs a{};
  a.mode = 2;
  a.aexp = aexp;
  a.fexp = bexp;
  a.seg_len = seg_len;
  a.Na = Na;
  a.N = N;
  a.nseg = (int)nseg;
  a.npairs = np;
  a.pairs = pairs_dev;
  a.part = work;
  a.ntiles = (N + OZ_TW - 1) / OZ_TW;
  a.err = err;
  a.stall = stall;
  // column images of A and B (one image when B is A) covering every segment
  const int64_t nch = nseg * seg_len / OZ_KC;
  if (!img_a || oz_img_cols_bytes(nch, Na) > img_a_bytes ||
      (B != A && (!img_b || oz_img_cols_bytes(nch, N) > img_b_bytes)))
    return 1;
  launch_oz_img_cols(A, lda, K, Na, aexp, nch, img_a, st);
  if (B != A) launch_oz_img_cols(B, ldb, K, N, bexp, nch, img_b, st);
  a.Aimg = img_a;
  a.Bimg = (B == A) ? img_a : img_b;
  a.astep = oz_img_cols_bytes(1, Na);
  a.bstep = oz_img_cols_bytes(1, N);
  if (oz_launch(a, n_sm, st)) return 1;
  k_oz_gram_reduce<<<(unsigned)(((int64_t)Na * N + 255) / 256), 256, 0, st>>>((int)nseg, Na, N, work, sym ? 1 : 0,
                                                                             accumulate ? 1 : 0, C, ldc);
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return 0;
}

int oz_gram_max_pairs(int Na, int N) { return oz_gram_pairs(Na, N, false, nullptr); }

}  // namespace efe