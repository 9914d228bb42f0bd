// Warp-specialised tensor-core cell products (tcgen05 + asynchronous copies, sm_103a).
//
// Paper, Sec. V (last paragraph): W_c(e) += H^cc_e Y_c(e) for every cell of
// one parity colour (cells of a colour share no node, so the scatter needs no
// atomics), one M = 128, K = 128 (eight 16-wide chunks), N <= 160 TF32 product
// per cell and column tile, FP32 accumulation in tensor memory.
//
// Roles of the warps of a persistent CTA (25 at a column tile of 160):
//   warp 0       MMA issuer (one elected lane): per 8 K one (one pass) or three
//                (3-term split: A1 B1 + A1 B2 + A2 B1) tcgen05.mma into one of two TMEM
//                accumulators, commits to `empty` (stage reusable) and, after
//                the last chunk, to `acc_full`;
//   then two groups of TW / 16 converter warps, one for the even and one for the odd
//                chunks: each warp copies its own 8 node rows x 32 columns of Y and its
//                share of the H^cc_e image (FP32, already in the core-matrix layout) by
//                16-byte asynchronous copies into a ring of its own, splits them into
//                A1 = TF32(A), A2 the TF32 remainder, K-major B1 = TF32(Y) and B2 (or the
//                BF16 forms) in the stage and arrives on `conv`;
//   last 4 warps epilogue: tcgen05.ld of the accumulator rows, scatter-add into
//                W as vector reductions performed in L2 (no read-back; four lanes add 64
//                contiguous bytes of a row), arrive on `acc_empty`.
// The chunks in flight come from warp-private rings because one bulk copy per node row
// bounds the whole kernel: its issue took 2,100 cycles per 16 rows, whatever the stages
// behind it (2 to 7) or the converter warps (6 to 16).  A launch over 3,670 cells x 135
// columns: 250 -> 163 us (64 KB of H, 68 KB of Y and twice 68 KB of W a cell, 6.0 TB/s: DRAM
// bounds it now); over 150 cells x 12 columns: 15 -> 11.5 us (one cell a CTA: latency).
// Every wait is bounded (about one second); on timeout the CTA records an error, stops
// issuing, drains and frees its TMEM.
#include <cuda_bf16.h>
#include <stdint.h>

#include "efe_kernels.h"

namespace efe {

namespace {

constexpr int T3_M = 128, T3_K = 128, T3_KC = 16, T3_NCH = 8;
// column tile (template parameter TW of the kernel): 64, 96 or 160, picked per
// system and N by the autotuner (efe_autotune); 160 by default
constexpr int T3_EPI_WARPS = 4;
constexpr uint32_t T3_TMEM_COLS = 512;     // accumulators at columns 0 and 256
constexpr long long T3_WAIT = 2000000000LL;
constexpr uint32_t T3_AP = T3_M * T3_KC * 4;    // a chunk of H, or one of its TF32 parts: 8 KB

template <int TW>
struct T3Layout {
  // stage: A1 | A2 (or BF16 A) | B1 | B2; ring slot: A | 1 KB of Y for each warp of the group
  static constexpr uint32_t A = 2 * T3_AP;                  // 16 KB
  static constexpr uint32_t B = TW * T3_KC * 4;             // 10 KB at TW = 160
  static constexpr uint32_t STAGE = A + 2 * B;              // 36 KB
  static constexpr int STAGES = TW == 160 ? 3 : 4;
  static constexpr int GW = TW / 16;                        // warps of a converter group
  static constexpr uint32_t SLOT = T3_AP + GW * 1024;       // 18 KB
  static constexpr int DEPTH = TW == 160 ? 3 : (TW == 96 ? 4 : 5);   // slots of a group
  static constexpr uint32_t RING = STAGES * STAGE;
  static constexpr uint32_t LUT = RING + 2 * DEPTH * SLOT;  // node offsets of the 128 rows
  static constexpr uint32_t BARS = LUT + T3_M * 4;
  static constexpr size_t TOTAL = (size_t)BARS + 256;
  static constexpr int THREADS = (1 + 2 * GW + T3_EPI_WARPS) * 32;
  static_assert(TOTAL <= 227 * 1024, "shared memory of one CTA");
};

__device__ __forceinline__ uint32_t su32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// K-major, no swizzle: core matrix 8 rows x 16 B; LBO = 128 B (next K core matrix), SBO to
// the next 8 rows, version 1
template <uint32_t SBO>
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128u >> 4) << 16) | ((uint64_t)(SBO >> 4) << 32) |
         ((uint64_t)1 << 46);
}
constexpr uint32_t T3_SBO = 512, T3_SBO_BF = 256;   // 16 K of 4 and of 2 bytes

__device__ __forceinline__ uint32_t idesc_tf32(int n) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(T3_M >> 4) << 24);
}

// BF16 operands (kind::f16): FP32 accumulate, BF16 A and B
__device__ __forceinline__ uint32_t idesc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(T3_M >> 4) << 24);
}

__device__ __forceinline__ uint32_t bmo(int row, int k) {
  return (uint32_t)(row >> 3) * T3_SBO_BF + (uint32_t)(k >> 3) * 128u + (uint32_t)(row & 7) * 16u + (uint32_t)(k & 7) * 2u;
}
__device__ __forceinline__ uint16_t bf16r(float x) {
  return __bfloat16_as_ushort(__float2bfloat16_rn(x));
}

__device__ __forceinline__ float tf32r(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

__device__ __forceinline__ void bar_init(uint64_t* b, uint32_t n) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(su32(b)), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(uint64_t* b) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(su32(b)) : "memory");
}

__device__ __forceinline__ bool bar_try(uint64_t* b, uint32_t parity) {
  uint32_t done = 0;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(su32(b)), "r"(parity)
      : "memory");
  return done != 0;
}
// one thread's bounded wait
__device__ __forceinline__ bool bar_wait(uint64_t* b, uint32_t parity) {
  const long long t0 = clock64();
  do {
    if (bar_try(b, parity)) return true;
  } while (clock64() - t0 < T3_WAIT);
  return false;
}
// the same for a warp that goes on together.  Every lane has its own clock and its own view of
// the barrier, so the lanes vote: one that left alone could not take part in the warp's next
// collective step, and the others would wait for it there without a bound.
__device__ __forceinline__ bool warp_wait(uint64_t* b, uint32_t parity) {
  const long long t0 = clock64();
  do {
    if (__all_sync(0xffffffffu, bar_try(b, parity))) return true;
  } while (__all_sync(0xffffffffu, clock64() - t0 < T3_WAIT));
  return false;
}
// the abort flag, one answer for the whole warp
__device__ __forceinline__ bool warp_aborted(const volatile int* flag) {
  return __any_sync(0xffffffffu, *flag != 0);
}

__device__ __forceinline__ void mma_tf32(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* b) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(su32(b))
               : "memory");
}

// node id of the corner of cell e (its local row 0)
__device__ __forceinline__ int64_t cell_corner(const MeshDev& m, int64_t e) {
  const int i = (int)(e % m.nc[0]), j = (int)((e / m.nc[0]) % m.nc[1]), kk = (int)(e / ((int64_t)m.nc[0] * m.nc[1]));
  return (int64_t)(P * i) + (int64_t)m.nn[0] * ((int64_t)(P * j) + (int64_t)m.nn[1] * (int64_t)(P * kk));
}

__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool real) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(real ? 16 : 0) : "memory");
}

// K-major core-matrix offset (bytes) within a 16-wide chunk of 4-byte values
__host__ __device__ __forceinline__ uint32_t cmo(int row, int k) {
  return (uint32_t)(row >> 3) * T3_SBO + (uint32_t)(k >> 2) * 128u + (uint32_t)(row & 7) * 16u;
}

__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred P;\n\telect.sync _|P, 0xffffffff;\n\tselp.u32 %0, 1, 0, P;\n\t}" : "=r"(p));
  return p != 0;
}

// MODE 0: one TF32 pass; 1: 3-term TF32 split (a1 b1 + a1 b2 + a2 b1); 2: BF16 operands
template <int MODE, int TW>
__global__ void __launch_bounds__(T3Layout<TW>::THREADS, 1)
    k_cell_tc3(const float* __restrict__ Ag, const int32_t* __restrict__ cells, int64_t ncells, MeshDev m,
               const float* __restrict__ Y, int64_t ldy, float* __restrict__ W, int64_t ldw, int N, int ntiles,
               int* __restrict__ err, int stall) {   // cells: null for all cells, their products to W's rows (e, r)
  using L = T3Layout<TW>;
  constexpr int ST = L::STAGES;
  extern __shared__ __align__(1024) unsigned char sm[];
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  uint64_t* conv = reinterpret_cast<uint64_t*>(sm + L::BARS);   // [ST]
  uint64_t* empty = conv + ST;                                  // [ST]
  uint64_t* accf = conv + 2 * ST;                               // [2]
  uint64_t* acce = accf + 2;                                    // [2]
  uint32_t* tslot = reinterpret_cast<uint32_t*>(accf + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(accf + 6);
  int32_t* lut = reinterpret_cast<int32_t*>(sm + L::LUT);
  // an earlier launch already failed: leave at once (CTA-uniform decision)
  if (tid == 0) *abort_flag = *(volatile int*)err;
  __syncthreads();
  if (*abort_flag) return;
  __syncthreads();

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tslot)),
                 "r"(T3_TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 32) {
    for (int s = 0; s < ST; ++s) {
      bar_init(conv + s, L::GW + (stall == 1));   // stall: see launch_cell_tc3
      bar_init(empty + s, 1 + (stall == 2));
    }
    for (int b = 0; b < 2; ++b) {
      bar_init(accf + b, 1 + (stall == 3));
      bar_init(acce + b, T3_EPI_WARPS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid >= 64 && tid < 64 + T3_M) {
    const int k = min(tid - 64, NL - 1);
    lut[tid - 64] = k % NP1 + m.nn[0] * (k / NP1 % NP1 + m.nn[1] * (k / (NP1 * NP1)));
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot;
  const int64_t nitems = ncells * ntiles;
  const int64_t my_items = nitems > blockIdx.x ? (nitems - blockIdx.x + gridDim.x - 1) / gridDim.x : 0;
  // the last chunk whose MMAs this thread committed (drained before the TMEM is
  // released if the CTA aborts)
  int64_t last_mma = -1;

  if (warp == 0) {
    // ------------------------------------------------------------ MMA issuer
    int s = 0;
    uint32_t ph = 0;
    for (int64_t t = 0; t < my_items && !warp_aborted(abort_flag); ++t) {
      const int64_t item = blockIdx.x + t * gridDim.x;
      const int c0 = (int)(item % ntiles) * TW;
      const int ncol = min(TW, N - c0);
      const int nmma = ((ncol + 15) / 16) * 16;
      const uint32_t id = MODE == 2 ? idesc_bf16(nmma) : idesc_tf32(nmma);
      const int b = (int)(t & 1);
      bool ok = true;
      if (t >= 2) ok = warp_wait(acce + b, (uint32_t)((t / 2 - 1) & 1));
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t d = tmem + (uint32_t)(b * 256);
      for (int kc = 0; kc < T3_NCH && ok; ++kc) {
        ok = warp_wait(conv + s, ph);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!ok) break;
        const uint32_t a1 = su32(sm) + (uint32_t)s * L::STAGE, b1 = a1 + L::A;
        if (elect_one()) {
          if (MODE == 2) {
            mma_bf16(d, sdesc<T3_SBO_BF>(a1), sdesc<T3_SBO_BF>(b1), id, kc > 0 ? 1u : 0u);
          } else {
            const uint64_t da1 = sdesc<T3_SBO>(a1), da2 = sdesc<T3_SBO>(a1 + T3_AP);
            const uint64_t db1 = sdesc<T3_SBO>(b1), db2 = sdesc<T3_SBO>(b1 + L::B);
#pragma unroll
            for (int ks = 0; ks < T3_KC / 8; ++ks) {
              const uint64_t off = (uint64_t)ks * (256u >> 4);
              mma_tf32(d, da1 + off, db1 + off, id, (kc > 0 || ks > 0) ? 1u : 0u);
              if (MODE == 1) {
                mma_tf32(d, da1 + off, db2 + off, id, 1u);
                mma_tf32(d, da2 + off, db1 + off, id, 1u);
              }
            }
          }
          mma_commit(empty + s);
          if (kc == T3_NCH - 1) mma_commit(accf + b);
        }
        __syncwarp();
        last_mma = t * T3_NCH + kc;
        if (++s == ST) {
          s = 0;
          ph ^= 1;
        }
      }
      if (!ok) {
        if (lane == 0) { *abort_flag = 1; atomicExch(err, 1); }
        break;
      }
    }
  } else if (warp <= 2 * L::GW) {
    // ------------------------------------------------------------ converters
    const int g = (warp - 1) / L::GW, w = (warp - 1) % L::GW;   // chunks of parity g
    const int cg = (w % (TW / 32)) * 32, k0 = (w / (TW / 32)) * 8;   // 32 columns, 8 rows of a chunk
    const int gt = w * 32 + lane;
    constexpr int UA = (int)(T3_AP / 16 + L::GW * 32 - 1) / (L::GW * 32);   // 16-byte units of H a thread
    unsigned char* ring = sm + L::RING + (uint32_t)(g * L::DEPTH) * L::SLOT;
    // the copies run DEPTH chunks of the group ahead, over the ends of items
    int64_t ft = 0;
    int fk = g, fs = 0, fcol = 0;
    const float* fa = nullptr;
    const float* fy = nullptr;
    auto fetch = [&]() {
      if (ft < my_items) {
        if (fk < 2) {
          const int64_t item = blockIdx.x + ft * gridDim.x;
          const int64_t e = cells ? cells[item / ntiles] : item / ntiles;
          const int c0 = (int)(item % ntiles) * TW, col = c0 + cg + (lane & 7) * 4;
          fa = Ag + e * (int64_t)(T3_M * T3_K) + gt * 4;
          fcol = col < min(N, c0 + TW);
          fy = Y + cell_corner(m, e) * ldy + (fcol ? col : c0);
        }
        const uint32_t slot = su32(ring) + (uint32_t)fs * L::SLOT;
#pragma unroll
        for (int u = 0; u < UA; ++u)
          if (gt + u * L::GW * 32 < (int)(T3_AP / 16))
            cp16(slot + (uint32_t)(gt + u * L::GW * 32) * 16u, fa + fk * (T3_M * T3_KC) + u * L::GW * 128, true);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          const int k = fk * T3_KC + k0 + u * 4 + (lane >> 3);
          cp16(slot + T3_AP + (uint32_t)w * 1024u + (uint32_t)(u * 32 + lane) * 16u, fy + (int64_t)lut[k] * ldy,
               fcol && k < NL);
        }
        fk += 2;
        if (fk >= T3_NCH) {
          fk = g;
          ++ft;
        }
        if (++fs == L::DEPTH) fs = 0;
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int i = 0; i < L::DEPTH; ++i) fetch();
    int s = g, rs = 0;
    uint32_t ph = 0;
    for (int64_t t = 0; t < my_items && !warp_aborted(abort_flag); ++t) {
      const int64_t item = blockIdx.x + t * gridDim.x;
      const int c0 = (int)(item % ntiles) * TW;
      const int ncol = min(TW, N - c0);
      const int n = cg + lane;
      const bool live = n < ((ncol + 15) / 16) * 16;
      bool ok = true;
      for (int kc = g; kc < T3_NCH; kc += 2) {
        asm volatile("cp.async.wait_group %0;" ::"n"(L::DEPTH - 1) : "memory");
        __syncwarp();
        const unsigned char* slot = ring + (uint32_t)rs * L::SLOT;
        const float* raw = reinterpret_cast<const float*>(slot + T3_AP + w * 1024) + lane;
        float4 x[UA];
        float y[2][4];
#pragma unroll
        for (int u = 0; u < UA; ++u)
          if (gt + u * L::GW * 32 < (int)(T3_AP / 16)) x[u] = reinterpret_cast<const float4*>(slot)[gt + u * L::GW * 32];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int q = 0; q < 4; ++q) y[u][q] = n < ncol ? raw[(u * 4 + q) * 32] : 0.f;
        __syncwarp();
        fetch();   // into the slot just read
        if (++rs == L::DEPTH) rs = 0;
        if (t * T3_NCH + kc >= ST) ok = warp_wait(empty + s, ph ^ 1u);
        if (!ok) break;
        unsigned char* A1 = sm + (uint32_t)s * L::STAGE;
        unsigned char* B1 = A1 + L::A;
#pragma unroll
        for (int u = 0; u < UA; ++u) {
          const int v = gt + u * L::GW * 32;
          if (v >= (int)(T3_AP / 16)) continue;
          if (MODE == 2) {
            // 16-byte unit v holds row 8 (v / 32) + v % 8, K quad (v / 8) % 4
            ushort4 h;
            h.x = bf16r(x[u].x); h.y = bf16r(x[u].y); h.z = bf16r(x[u].z); h.w = bf16r(x[u].w);
            *reinterpret_cast<ushort4*>(A1 + bmo((v >> 5) * 8 + (v & 7), ((v >> 3) & 3) * 4)) = h;
          } else {
            float4 h4;
            h4.x = tf32r(x[u].x); h4.y = tf32r(x[u].y); h4.z = tf32r(x[u].z); h4.w = tf32r(x[u].w);
            reinterpret_cast<float4*>(A1)[v] = h4;
            if (MODE == 1) {
              float4 l4;
              l4.x = tf32r(x[u].x - h4.x); l4.y = tf32r(x[u].y - h4.y);
              l4.z = tf32r(x[u].z - h4.z); l4.w = tf32r(x[u].w - h4.w);
              reinterpret_cast<float4*>(A1 + T3_AP)[v] = l4;
            }
          }
        }
        if (live) {
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            if (MODE == 2) {
              ushort4 h;
              h.x = bf16r(y[u][0]); h.y = bf16r(y[u][1]); h.z = bf16r(y[u][2]); h.w = bf16r(y[u][3]);
              *reinterpret_cast<ushort4*>(B1 + bmo(n, k0 + u * 4)) = h;
            } else {
              float4 h4;
              h4.x = tf32r(y[u][0]); h4.y = tf32r(y[u][1]); h4.z = tf32r(y[u][2]); h4.w = tf32r(y[u][3]);
              *reinterpret_cast<float4*>(B1 + cmo(n, k0 + u * 4)) = h4;
              if (MODE == 1) {
                float4 l4;
                l4.x = tf32r(y[u][0] - h4.x); l4.y = tf32r(y[u][1] - h4.y);
                l4.z = tf32r(y[u][2] - h4.z); l4.w = tf32r(y[u][3] - h4.w);
                *reinterpret_cast<float4*>(B1 + L::B + cmo(n, k0 + u * 4)) = l4;
              }
            }
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) bar_arrive(conv + s);
        s += 2;
        if (s >= ST) {
          s -= ST;
          ph ^= 1;
        }
      }
      if (!ok) {
        *abort_flag = 1;
        atomicExch(err, 1);
        break;
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  } else {
    // ------------------------------------------------------------ epilogue
    const int quarter = warp & 3;         // TMEM lane quarter accessible to this warp
    const int sub = lane & 3;
    for (int64_t t = 0; t < my_items && !warp_aborted(abort_flag); ++t) {
      const int64_t item = blockIdx.x + t * gridDim.x;
      const int64_t e = cells ? cells[item / ntiles] : item / ntiles;
      const int c0 = (int)(item % ntiles) * TW;
      const int ncol = min(TW, N - c0);
      const int b = (int)(t & 1);
      // after the exchange below this lane holds 16 bytes of each of the four rows of its lane quad
      const int r0 = quarter * 32 + (lane & ~3);
      float* wr = W + (cells ? cell_corner(m, e) : e * NL) * ldw + c0;
      int64_t ro[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) ro[i] = (int64_t)(cells ? lut[r0 + i] : r0 + i) * ldw;
      if (!warp_wait(accf + b, (uint32_t)((t / 2) & 1))) {
        *abort_flag = 1;
        atomicExch(err, 1);
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int cb = 0; cb < ncol; cb += 16) {
        uint32_t v[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * 256 + cb))
            : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        // 4 x 4 exchange of 16-byte pieces between the lanes of a quad: v[4 i ..] becomes columns
        // 4 sub .. of row r0 + i
#pragma unroll
        for (int o = 1; o < 4; o <<= 1)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (i & o) continue;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint32_t lo = v[4 * i + q], hi = v[4 * (i + o) + q];
              const uint32_t got = __shfl_xor_sync(0xffffffffu, (sub & o) ? lo : hi, o);
              v[4 * i + q] = (sub & o) ? got : lo;
              v[4 * (i + o) + q] = (sub & o) ? hi : got;
            }
          }
        // the products are added in L2 (vector reductions, no read-back): a W value
        // receives one addition per launch (cells of a colour share no node)
        const int c = cb + 4 * sub;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (r0 + i >= NL) continue;
          float* o = wr + ro[i] + c;
          if (!cells) {
            if (c + 4 <= ncol) {
              *reinterpret_cast<float4*>(o) = make_float4(__uint_as_float(v[4 * i]), __uint_as_float(v[4 * i + 1]),
                                                          __uint_as_float(v[4 * i + 2]), __uint_as_float(v[4 * i + 3]));
            } else {
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (c + q < ncol) o[q] = __uint_as_float(v[4 * i + q]);
            }
          } else if (c + 4 <= ncol) {
            asm volatile("red.relaxed.gpu.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(o),
                         "f"(__uint_as_float(v[4 * i])), "f"(__uint_as_float(v[4 * i + 1])),
                         "f"(__uint_as_float(v[4 * i + 2])), "f"(__uint_as_float(v[4 * i + 3]))
                         : "memory");
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (c + q < ncol) atomicAdd(o + q, __uint_as_float(v[4 * i + q]));
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) bar_arrive(acce + b);
    }
  }
  // all roles done (the asynchronous copies have landed).  After an abort, drain before
  // the TMEM is released: the last MMA commit (it covers every MMA this CTA issued)
  // arrives; the drain wait is bounded like the pipeline's own.
  __syncthreads();
  if (*abort_flag && warp == 0 && last_mma >= 0) bar_wait(empty + (int)(last_mma % ST), (uint32_t)((last_mma / ST) & 1));
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(T3_TMEM_COLS) : "memory");
  }
}

// W row of a node = the rows (e, r) of P that meet it, added in the order of the cells'
// parity colours (as the coloured launches add them); columns N .. 4 q4 of W are zero
__global__ void k_tc3_gather(MeshDev m, int64_t n_nodes, const float* __restrict__ Pc, int64_t ldp, int N, int q4,
                             float* __restrict__ W, int64_t ldw) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (idx >= n_nodes * q4) return;
  const int64_t g = idx / q4;
  const int c = (int)(idx % q4) * 4;
  const int G[3] = {(int)(g % m.nn[0]), (int)((g / m.nn[0]) % m.nn[1]), (int)(g / ((int64_t)m.nn[0] * m.nn[1]))};
  int hi[3], cnt[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    hi[d] = min(G[d] / P, m.nc[d] - 1);
    cnt[d] = (G[d] % P == 0 && G[d] > 0 && G[d] / P < m.nc[d]) ? 2 : 1;
  }
  float4 v[8];
  bool ok[8];
#pragma unroll
  for (int col = 0; col < 8; ++col) {
    int cc[3], l[3];
    ok[col] = c < N;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int par = (col >> d) & 1;
      cc[d] = (hi[d] & 1) == par ? hi[d] : hi[d] - 1;
      ok[col] = ok[col] && (cc[d] == hi[d] || cnt[d] == 2);
      l[d] = G[d] - P * cc[d];
    }
    const int64_t e = cc[0] + (int64_t)m.nc[0] * (cc[1] + (int64_t)m.nc[1] * cc[2]);
    if (ok[col]) v[col] = *reinterpret_cast<const float4*>(Pc + (e * NL + l[0] + NP1 * (l[1] + NP1 * l[2])) * ldp + c);
  }
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int col = 0; col < 8; ++col) {
    if (!ok[col]) continue;
    s.x += v[col].x;
    if (c + 1 < N) s.y += v[col].y;
    if (c + 2 < N) s.z += v[col].z;
    if (c + 3 < N) s.w += v[col].w;
  }
  *reinterpret_cast<float4*>(W + g * ldw + c) = s;
}

// FP32 images of H^cc_e, [cell][16-wide chunk], each in the K-major core-matrix layout
__global__ void k_build_aimg(const double* __restrict__ Hcc, int64_t n_cell, float* __restrict__ A) {
  const int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;   // (cell, row, K quad)
  if (idx >= n_cell * T3_M * (T3_K / 4)) return;
  const int64_t e = idx / (T3_M * (T3_K / 4));
  const int r = (int)(idx / (T3_K / 4)) % T3_M, k = (int)(idx % (T3_K / 4)) * 4;
  float h[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) h[q] = (r < NL && k + q < NL) ? (float)Hcc[e * (int64_t)(NL * NL) + r * NL + k + q] : 0.f;
  unsigned char* o = reinterpret_cast<unsigned char*>(A) + (e * T3_NCH + k / T3_KC) * (int64_t)T3_AP + cmo(r, k % T3_KC);
  *reinterpret_cast<float4*>(o) = make_float4(h[0], h[1], h[2], h[3]);
}

}  // namespace

int64_t tc3_image_elems(int64_t n_cell) { return n_cell * T3_M * (int64_t)T3_K; }

void launch_build_aimg(const double* Hcc, int64_t n_cell, float* A, cudaStream_t st) {
  const int64_t n = n_cell * T3_M * (T3_K / 4);
  if (n > 0) {
    k_build_aimg<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(Hcc, n_cell, A);
    g_launches.fetch_add(1, std::memory_order_relaxed);
  }
}

int64_t tc3_scratch_elems(int64_t n_cell, int64_t ld) { return n_cell * NL * ld; }

void launch_tc3_gather(const MeshDev& m, const float* Pc, int64_t ldp, int N, float* W, int64_t ldw, cudaStream_t st) {
  const int64_t nn = (int64_t)m.nn[0] * m.nn[1] * m.nn[2];
  const int q4 = (int)(ldw / 4);
  k_tc3_gather<<<(unsigned)((nn * q4 + 255) / 256), 256, 0, st>>>(m, nn, Pc, ldp, N, q4, W, ldw);
  g_launches.fetch_add(1, std::memory_order_relaxed);
}

// W += H_e Y_e over the cells of one colour; cells == nullptr: rows (e, r) of W = row r of
// H_e Y_e over all ncells cells.  Y / W: FP32 rows, ld a multiple of 4
// elements and rows 16-byte aligned (the 16-byte copies and reductions).
namespace {
template <int TW>
void tc3_launch(const float* A, const int32_t* cells, int64_t ncells, const MeshDev& m,
                const float* Y, int64_t ldy, float* W, int64_t ldw, int N, int mode, int n_sm, int* err,
                cudaStream_t st, int stall) {
  const int ntiles = (N + TW - 1) / TW;
  const int64_t items = ncells * ntiles;
  const unsigned grid = (unsigned)(items < n_sm ? items : n_sm);
  const size_t smem = T3Layout<TW>::TOTAL;
  if (mode == 1) {
    cudaFuncSetAttribute(k_cell_tc3<1, TW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_cell_tc3<1, TW><<<grid, T3Layout<TW>::THREADS, smem, st>>>(A, cells, ncells, m, Y, ldy, W, ldw, N, ntiles, err, stall);
  } else if (mode == 2) {
    cudaFuncSetAttribute(k_cell_tc3<2, TW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_cell_tc3<2, TW><<<grid, T3Layout<TW>::THREADS, smem, st>>>(A, cells, ncells, m, Y, ldy, W, ldw, N, ntiles, err, stall);
  } else {
    cudaFuncSetAttribute(k_cell_tc3<0, TW>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    k_cell_tc3<0, TW><<<grid, T3Layout<TW>::THREADS, smem, st>>>(A, cells, ncells, m, Y, ldy, W, ldw, N, ntiles, err, stall);
  }
}
}  // namespace

const int* tc3_tiles(int* count) {
  static const int tiles[3] = {64, 96, 160};
  *count = 3;
  return tiles;
}

int launch_cell_tc3(const float* A, const int32_t* cells, int64_t ncells, const MeshDev& m,
                    const float* Y, int64_t ldy, float* W, int64_t ldw, int N, int mode, int n_sm, int* err,
                    cudaStream_t st, int tile, int stall) {
  if (ncells <= 0 || N <= 0) return 0;
  if ((ldy & 3) || (ldw & 3)) return 1;
  if (tile == 64)
    tc3_launch<64>(A, cells, ncells, m, Y, ldy, W, ldw, N, mode, n_sm, err, st, stall);
  else if (tile == 96)
    tc3_launch<96>(A, cells, ncells, m, Y, ldy, W, ldw, N, mode, n_sm, err, st, stall);
  else if (tile == 160 || tile == 0)
    tc3_launch<160>(A, cells, ncells, m, Y, ldy, W, ldw, N, mode, n_sm, err, st, stall);
  else
    return 1;
  g_launches.fetch_add(1, std::memory_order_relaxed);
  return 0;
}

}  // namespace efe
