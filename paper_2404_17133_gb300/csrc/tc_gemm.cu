// tcgen05 tensor-core contraction over the auxiliary index,
//   C[m][n] (+)= sum_P sum_k A[P][m][k] B[P][n][k],
// used for the exchange terms of the response products (Eq. hessian):
//   K1[(n,i)][b] = sum_P sum_a Z[P][(n,i)][a] L^P_ab      ((ij|ab) term, k = a)
//   K2[(n,i)][a] = sum_P sum_j Q[P][(n,i)][j] L^P_ja      ((ib|ja) term, k = j)
// K1's contraction is the dominant cost of every product (about 70-90% of flops).
//
// Exact operator: every operand is scaled by a power of two s (so that
// max |s x| <= 2^14, or below 2^15 from a Cauchy-Schwarz bound for the stage-1
// results) and split into FP16 hi + lo parts, x s = hi + lo to ~2^-22 (11
// significand bits each; s keeps the lo parts of all but the negligible
// elements above FP16's normal range); each tile pair contributes
// hi*hi + hi*lo + lo*hi (lo*lo is below 2^-22), FP32 accumulation, and the
// sum is multiplied by 1 / (s_A s_B): an FP32-accurate product at the FP16
// tensor-core rate.  ris operator: BF16 factors (no scaling), the trial
// vectors as BF16 hi + lo.
//
// Layout / mapping (all K-major, so both operands stream along k):
//   A viewed as a 3-D tensor (k: Kin, P: pn, row: M), rows of ldk, M rows per P
//   B viewed as a 3-D tensor (k: Kin, n: N, P: pn), rows of ldk; for K1 the
//          rows of the symmetric L^P are its columns, for K2 B is L^P_ov
//          stored transposed ([P][a][j])
//   K loop: for each P in the CTA's split range, k-blocks of 128 bytes (one
//          128B-swizzle atom per row) or, for the hi+lo x hi+lo products, of
//          64 bytes (64B swizzle); TMA zero-fills k >= Kin, n >= N and rows >= M.
// Tiles of 256 x 256 by CTA pairs (k1_pair_kernel), of 128 x 256 by single CTAs where
// there is one M tile (k1_tc_kernel).  6 warps: warp 0 issues TMA loads, warp 1 owns
// the tensor memory and one elected lane issues tcgen05.mma, warps 2-5 drain the
// FP32 accumulator from TMEM.  A 3- or 4-stage mbarrier ring (~192 KB) connects
// producer and MMA; tcgen05.commit releases a stage when its MMAs have read it.
// Split-K: a CTA or cluster takes a contiguous range of (P, a-block) steps and writes
// its own FP32 partial tile; a fixed-order reduction sums the partials.
//
// Every wait on an mbarrier is bounded: on timeout the thread records an error
// code in `err` and leaves the loop; the host turns it into TDDFT_ERR_CUDA.
#include <algorithm>
#include <cstdlib>
#include <type_traits>
#include <cuda.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>

#include "ctx.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"
#include "vecops.cuh"

namespace tddft {

namespace {

constexpr int BM = 128;
constexpr int BN = 256;                      // 128 x 256 MMA tiles (full tcgen05 rate per CTA)
constexpr int BK = 64;                       // bf16 elements per 128-byte row
constexpr int A_BYTES = BM * 128;             // 16 KB per hi or lo tile (128-byte rows)
constexpr int B_BYTES = BN * 128;
// Operand element types of the contraction: BF16 or FP16 (kind::f16, 64
// elements per 128-byte row) or FP8 e4m3 (kind::f8f6f4, 128 elements per row).
// Either way one tcgen05.mma consumes 32 bytes of K, so the descriptors
// advance alike.
enum ElemType : int { ET_BF16 = 0, ET_F16 = 1, ET_E4M3 = 2 };
template <int ET> struct Elem {
  static constexpr int BKE = ET == ET_E4M3 ? 128 : 64;
  // instruction-descriptor A and B type fields: kind::f16 F16 = 0, BF16 = 1; kind::f8f6f4 E4M3 = 0
  static constexpr uint32_t TYPE_BITS = ET == ET_BF16 ? ((1u << 7) | (1u << 10)) : 0u;
};
constexpr int elem_of(TcElt e) { return e == TcElt::F16 ? ET_F16 : ET_BF16; }
// Operand split modes: BOTH = A and B as hi + lo (hi*hi + hi*lo + lo*hi); ASPLIT =
// A as hi + lo, B a plain operand (hi*B + lo*B: exact with respect to B, e.g.
// FP32 vectors against BF16 ris factors).
enum SplitMode : int { BOTH = 1, ASPLIT = 2 };
__host__ __device__ constexpr bool b_split(int m) { return m == BOTH; }
__host__ __device__ constexpr int n_parts_a(int) { return 2; }
__host__ __device__ constexpr int n_parts_b(int m) { return b_split(m) ? 2 : 1; }

// Ring of the contraction kernel for rows of RB bytes along K (128: one
// 128-byte swizzle atom per row; 64: half as much K per stage in a 64-byte
// swizzle, so twice as many stages fit -- the split-B products, whose hi+lo
// tiles fill 96 KB per 128-byte stage, use it for a four-deep ring).
template <int MODE, int RB = 128> struct Cfg {
  static constexpr int STAGE_BYTES = (n_parts_a(MODE) * A_BYTES + n_parts_b(MODE) * B_BYTES) * RB / 128;
  static constexpr int STAGES = (MODE == ASPLIT ? 3 : 2) * 128 / RB;   // ~192 KB ring
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 /*align*/ + 256 /*barriers*/;
};
constexpr int THREADS = 192;

struct Params {
  int M, N;          // output rows / columns
  int Kin;           // k extent per P (the last k-block of a P issues only the MMAs it needs)
  int nab;           // k-blocks per P
  int total;         // pn * nab steps
  int per_split;     // steps per split
  float* part;       // [splits][M][N]
  int* err;
};


__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar,
                                            int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}


// Instruction descriptor: D = F32, A and B of the same type (BF16 or FP16
// for kind::f16, E4M3 for kind::f8f6f4), both K-major, M = 128, N = nb.
template <int ET>
__host__ __device__ constexpr uint32_t idesc_of(int nb = BN) {
  return (1u << 4) | Elem<ET>::TYPE_BITS | ((uint32_t)(nb >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
}

template <int ET>
__device__ __forceinline__ void mma_op(uint32_t tmem, uint64_t a, uint64_t b, uint32_t accum,
                                       uint32_t idesc = idesc_of<ET>()) {
  if constexpr (ET == ET_E4M3) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accum));
  } else {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accum));
  }
}

// Shared-memory matrix descriptor for RB-byte rows: K-major, 128-byte (RB =
// 128) or 64-byte (RB = 64) swizzle, 8-row groups 8 RB bytes apart.
template <int RB>
__device__ __forceinline__ uint64_t sdesc_rb(const void* p) {
  if constexpr (RB == 128) return sdesc(p);
  const uint64_t addr = smem_u32(p);
  return ((addr & 0x3FFFFull) >> 4) | (1ull << 16) | ((uint64_t)((8 * RB) >> 4) << 32) | (1ull << 46) |
         (4ull << 61);
}

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}


// One CTA per output tile: problems with a single M tile (k1_pair_kernel takes
// the others).
template <int MODE, int ET, int RB = 128>
__global__ void __launch_bounds__(THREADS, 1)
k1_tc_kernel(const __grid_constant__ CUtensorMap mA_hi, const __grid_constant__ CUtensorMap mA_lo,
             const __grid_constant__ CUtensorMap mB_hi, const __grid_constant__ CUtensorMap mB_lo,
             Params p) {
  constexpr int STAGES = Cfg<MODE, RB>::STAGES;
  constexpr int STAGE_BYTES = Cfg<MODE, RB>::STAGE_BYTES;
  constexpr int AB = A_BYTES * RB / 128, BB = B_BYTES * RB / 128;   // one part tile
  constexpr int B_OFF = 2 * AB;                                     // first B tile in a stage
  constexpr int BKE = Elem<ET>::BKE * RB / 128;                     // K elements per k-block
  constexpr int KSTEPS = RB / 32;                                   // 32-byte K steps per k-block
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* done = empty + STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * BN, m0 = blockIdx.y * BM;
  const int k_begin = blockIdx.z * p.per_split;
  const int k_end = min(p.total, k_begin + p.per_split);
  const int nk = max(0, k_end - k_begin);

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)), "r"(BN));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // ---- TMA producer
    bool ok = true;
    for (int i = 0; i < nk && ok; ++i) {
      const int s = i % STAGES;
      const uint32_t ph = (uint32_t)(i / STAGES) & 1u;
      if (!mbar_wait(&empty[s], ph ^ 1u)) { atomicOr(p.err, 1); ok = false; break; }
      const int kb = k_begin + i;
      const int P = kb / p.nab, a0 = (kb - P * p.nab) * BKE;
      unsigned char* st = smem + s * STAGE_BYTES;
      mbar_expect_tx(&full[s], STAGE_BYTES);
      tma_load_3d(st, &mA_hi, &full[s], a0, P, m0);
      tma_load_3d(st + AB, &mA_lo, &full[s], a0, P, m0);
      tma_load_3d(st + B_OFF, &mB_hi, &full[s], a0, n0, P);
      if (b_split(MODE)) tma_load_3d(st + B_OFF + BB, &mB_lo, &full[s], a0, n0, P);
    }
    // let the copies already issued land before the CTA can exit
    for (int i = max(0, nk - STAGES); i < nk; ++i) {
      if (!mbar_wait(&full[i % STAGES], (uint32_t)(i / STAGES) & 1u)) { atomicOr(p.err, 2); break; }
    }
  } else if (warp == 1 && lane == 0) {
    // ---- MMA issuer.  The MMA spans only the tile's columns below N
    // (rounded up to 16) and, in the last k-block of each P, only the 32-byte
    // K steps below Kin: the skipped products are of TMA's zero fill.
    const int nb_cta = min(BN, (p.N - n0 + 15) & ~15);
    const uint32_t idesc = idesc_of<ET>(nb_cta);
    bool ok = true;
    for (int i = 0; i < nk; ++i) {
      const int s = i % STAGES;
      if (!mbar_wait(&full[s], (uint32_t)(i / STAGES) & 1u)) { atomicOr(p.err, 4); ok = false; break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      unsigned char* st = smem + s * STAGE_BYTES;
      const uint64_t ah = sdesc_rb<RB>(st), bh = sdesc_rb<RB>(st + B_OFF);
      const int kb = k_begin + i;
      const int rem = p.Kin - (kb % p.nab) * BKE;
      const int nks = rem >= BKE ? KSTEPS : (rem * KSTEPS + BKE - 1) / BKE;
#pragma unroll
      for (int kk = 0; kk < KSTEPS; ++kk) {
        if (kk < nks) {
          const uint64_t off = (uint64_t)(kk * 32) >> 4;   // 32 bytes along K per MMA
          mma_op<ET>(tmem, ah + off, bh + off, (i > 0 || kk > 0) ? 1u : 0u, idesc);
          if (b_split(MODE)) mma_op<ET>(tmem, ah + off, sdesc_rb<RB>(st + B_OFF + BB) + off, 1u, idesc);
          mma_op<ET>(tmem, sdesc_rb<RB>(st + AB) + off, bh + off, 1u, idesc);
        }
      }
      mma_commit(&empty[s]);
    }
    (void)ok;
    mma_commit(done);   // fires when every MMA issued above has completed
  } else if (warp >= 2) {
    // ---- epilogue: TMEM -> registers -> FP32 partial tile
    const int q = warp & 3;                 // TMEM lane quadrant of this warp
    const int row = m0 + q * 32 + lane;
    bool have = true;
    if (nk > 0) {
      if (!mbar_wait(done, 0)) { atomicOr(p.err, 8); have = false; }
      have = __all_sync(0xffffffffu, have);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    }
    float* out = p.part + (size_t)blockIdx.z * p.M * p.N;
#pragma unroll 1
    for (int c = 0; c < BN; c += 16) {
      uint32_t v[16];
      if (nk > 0 && have) {
        const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c;
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15},"
            " [%16];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
              "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
              "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = 0u;
      }
      if (row < p.M) {
        const int col0 = n0 + c;
        float* o = out + (size_t)row * p.N + col0;
        if ((p.N & 3) == 0 && col0 + 16 <= p.N) {   // 16-byte aligned: four vector stores
#pragma unroll
          for (int j = 0; j < 16; j += 4)
            *reinterpret_cast<float4*>(o + j) = make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]),
                                                            __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (col0 + j < p.N) o[j] = __uint_as_float(v[j]);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN));
  }
}

// Row pairs of CTAs on one 256-row tile (cta_group::2): the pair's tcgen05.mma
// takes 128 A rows and half of the B rows from each CTA's shared memory, so
// every SM reads and stores only half of B.  That is what bounds the single-CTA
// form: per 16-element K step of the hi + lo products it reads 36 KB of operands
// and receives 24 KB by TMA in the 384 cycles of its MMAs, against 128 bytes per
// cycle of shared memory; here 24 KB (20 KB with A_hi held in the operand
// collector for its two products) and 16 KB.
// CX = 2: clusters of two pairs along N, which also share their A rows (each CTA
// loads half of its rows and multicasts them to the CTA of the other pair that
// needs the same ones).
// Cluster rank = h + 2 y: h the row half, y the pair; the pair's leader is h = 0.
// All four (two) CTAs' loads of a pair's stage signal the leader's `full`
// barrier, the leader's commit frees the stage in every CTA that writes it.
// N is cut into tiles of whole 32-column units, as equal as they can be: tiles
// of 256 columns and a remainder would leave a cluster's lighter pair waiting.
template <int MODE, int RB> struct PCfg {
  static constexpr int AB = BM * RB, HB = (BN / 2) * RB;   // one part of A, of half of B
  static constexpr int STAGE_BYTES = n_parts_a(MODE) * AB + n_parts_b(MODE) * HB;
  static constexpr int STAGES = 196608 / STAGE_BYTES;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
};

struct PairParams {
  int M, N, Kin, nab, total, per_split;
  int nt, nt0, mp;   // N tiles (padded to whole clusters; real ones), M tile pairs
  int nq, nr;        // 32-column units per N tile; the first nr tiles have one more
  int b_rows;        // rows of half of the widest B tile (the TMA box)
  float* part;
  int* err;
};

__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

// Tensor memory of a pair (cta_group::2).  Both CTAs have to be running when either
// allocates, neither gives up the permit before both have allocated, and neither leaves before both
// have freed: a cluster barrier stands before the allocation, after it and after the
// freeing.  With only the one after it, where kernels of several streams share the
// GPU and the two CTAs start at different times, the second CTA's allocation now and then
// waited forever (once in some thousands of products, 16 streams).
__device__ __forceinline__ void pair_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
}

// Load into this CTA (or, with a mask, into the same offset of its CTAs), signalling
// the mbarrier `bar` (a shared::cluster address) of the pair's leader.
__device__ __forceinline__ void tma_load_3d_pair(void* dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                                 int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d_pair_mc(void* dst, const CUtensorMap* map, uint32_t bar, int c0, int c1,
                                                    int c2, uint16_t mask) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.multicast::cluster"
      ".cta_group::2 [%0], [%1, {%3, %4, %5}], [%2], %6;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "h"(mask)
      : "memory");
}

// Pair MMA; KEEP: 0 plain, 1 the A operand stays in the collector, 2 its last use.
template <int ET, int KEEP>
__device__ __forceinline__ void mma_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t accum, uint32_t idesc) {
#define TD_MMA2(kind, coll)                                                                       \
  asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"                                     \
               " tcgen05.mma.cta_group::2." kind coll " [%0], %1, %2, %3, p;\n}\n" ::"r"(d),      \
               "l"(a), "l"(b), "r"(idesc), "r"(accum))
  if constexpr (ET == ET_E4M3) {
    TD_MMA2("kind::f8f6f4", "");
  } else if constexpr (KEEP == 1) {
    TD_MMA2("kind::f16", ".collector::a::fill");
  } else if constexpr (KEEP == 2) {
    TD_MMA2("kind::f16", ".collector::a::lastuse");
  } else {
    TD_MMA2("kind::f16", "");
  }
#undef TD_MMA2
}

__device__ __forceinline__ void commit_pair(uint64_t* bar, uint16_t mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"(mask)
      : "memory");
}

template <int MODE, int ET, int CX, int RB>
__global__ void __launch_bounds__(THREADS, 1)
k1_pair_kernel(const __grid_constant__ CUtensorMap mA_hi, const __grid_constant__ CUtensorMap mA_lo,
               const __grid_constant__ CUtensorMap mB_hi, const __grid_constant__ CUtensorMap mB_lo,
               const PairParams p) {
  using C = PCfg<MODE, RB>;
  constexpr int STAGES = C::STAGES;
  constexpr int B_OFF = n_parts_a(MODE) * C::AB;
  constexpr int BKE = Elem<ET>::BKE * RB / 128;   // K elements per k-block
  constexpr int KSTEPS = RB / 32;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * C::STAGE_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* done = empty + STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int h = (int)(rank & 1u), y = (int)(rank >> 1);
  // N pairs fastest: the clusters that run together share their A rows through L2
  const int cid = blockIdx.x / (2 * CX), ntc = p.nt / CX;
  const int t = (cid % ntc) * CX + y;
  const int m0 = ((cid / ntc) % p.mp) * 2 * BM + h * BM;
  const int z = cid / (ntc * p.mp);
  const int n0 = 32 * (min(t, p.nt0) * p.nq + min(t, p.nr));
  const int width = t < p.nt0 ? 32 * (p.nq + (t < p.nr ? 1 : 0)) : 32;   // a padding tile is all zero fill
  const int k_begin = z * p.per_split;
  const int nk = max(0, min(p.total, k_begin + p.per_split) - k_begin);

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], CX); }
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  cluster_sync_all();   // every barrier of the cluster initialised, and both CTAs of a pair running
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)), "r"(BN));
  }
  __syncthreads();
  cluster_sync_all();   // both CTAs' tensor memory allocated
  if (warp == 1) pair_relinquish();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    // ---- TMA producer (both CTAs of the pair)
    const uint32_t lead_full = mapa(smem_u32(full), rank & ~1u);
    const uint32_t bytes = 2u * (n_parts_a(MODE) * C::AB + n_parts_b(MODE) * (uint32_t)p.b_rows * RB);
    const uint16_t mask_a = (uint16_t)((1u << h) | (1u << (h + 2)));   // CX = 2: the CTAs of this row half
    const int nh = n0 + h * (width / 2);
    for (int i = 0; i < nk; ++i) {
      const int s = i % STAGES;
      if (!mbar_wait(&empty[s], ((uint32_t)(i / STAGES) & 1u) ^ 1u)) { atomicOr(p.err, 1); break; }
      const int kb = k_begin + i;
      const int P = kb / p.nab, a0 = (kb - P * p.nab) * BKE;
      unsigned char* st = smem + s * C::STAGE_BYTES;
      const uint32_t bar = lead_full + (uint32_t)(s * 8);
      if (h == 0) mbar_expect_tx(&full[s], bytes);
      if constexpr (CX > 1) {
        constexpr int HA = C::AB / 2;
        const int mh = m0 + y * (BM / 2);
        tma_load_3d_pair_mc(st + y * HA, &mA_hi, bar, a0, P, mh, mask_a);
        tma_load_3d_pair_mc(st + C::AB + y * HA, &mA_lo, bar, a0, P, mh, mask_a);
      } else {
        tma_load_3d_pair(st, &mA_hi, bar, a0, P, m0);
        tma_load_3d_pair(st + C::AB, &mA_lo, bar, a0, P, m0);
      }
      tma_load_3d_pair(st + B_OFF, &mB_hi, bar, a0, nh, P);
      if (b_split(MODE)) tma_load_3d_pair(st + B_OFF + C::HB, &mB_lo, bar, a0, nh, P);
    }
    // let the copies already issued (they signal the leader) land, and the last
    // commits arrive on this CTA's `empty` barriers, before a CTA can exit
    if (h == 0)
      for (int i = max(0, nk - STAGES); i < nk; ++i)
        if (!mbar_wait(&full[i % STAGES], (uint32_t)(i / STAGES) & 1u)) { atomicOr(p.err, 2); break; }
    for (int i = nk; i < nk + STAGES; ++i)
      if (!mbar_wait(&empty[i % STAGES], ((uint32_t)(i / STAGES) & 1u) ^ 1u)) { atomicOr(p.err, 2); break; }
  } else if (warp == 1 && lane == 0 && h == 0) {
    // ---- MMA issuer (the leader): M = 256, N = width; the last k-block of a P
    // issues only the 32-byte K steps below Kin
    const uint32_t idesc =
        (1u << 4) | Elem<ET>::TYPE_BITS | ((uint32_t)(width >> 3) << 17) | ((uint32_t)(2 * BM >> 4) << 24);
    const uint16_t mask_all = (uint16_t)((1u << (2 * CX)) - 1);
    // the instructions between two k-blocks' MMAs leave the tensor core idle: no divisions
    int s = 0, pos = nk > 0 ? k_begin % p.nab : 0;
    uint32_t ph = 0;
    const int last_steps = (p.Kin - (p.nab - 1) * BKE) >= BKE ? KSTEPS : ((p.Kin - (p.nab - 1) * BKE) * KSTEPS + BKE - 1) / BKE;
    for (int i = 0; i < nk; ++i) {
      if (!mbar_wait(&full[s], ph)) { atomicOr(p.err, 4); break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      unsigned char* st = smem + s * C::STAGE_BYTES;
      const uint64_t ah = sdesc_rb<RB>(st), bh = sdesc_rb<RB>(st + B_OFF);
      const int nks = pos == p.nab - 1 ? last_steps : KSTEPS;
#pragma unroll
      for (int kk = 0; kk < KSTEPS; ++kk) {
        if (kk < nks) {
          const uint64_t off = (uint64_t)(kk * 32) >> 4;
          const uint32_t acc = (i > 0 || kk > 0) ? 1u : 0u;
          if (b_split(MODE)) {
            mma_pair<ET, 1>(tmem, ah + off, bh + off, acc, idesc);
            mma_pair<ET, 2>(tmem, ah + off, sdesc_rb<RB>(st + B_OFF + C::HB) + off, 1u, idesc);
          } else {
            mma_pair<ET, 0>(tmem, ah + off, bh + off, acc, idesc);
          }
          mma_pair<ET, 0>(tmem, sdesc_rb<RB>(st + C::AB) + off, bh + off, 1u, idesc);
        }
      }
      commit_pair(&empty[s], mask_all);
      if (++s == STAGES) { s = 0; ph ^= 1u; }
      if (++pos == p.nab) pos = 0;
    }
    commit_pair(done, (uint16_t)(3u << (2 * y)));   // fires when every MMA issued above has completed
  } else if (warp >= 2) {
    // ---- epilogue: this CTA's 128 rows, TMEM -> registers -> FP32 partial tile
    const int q = warp & 3;
    const int row = m0 + q * 32 + lane;
    bool have = mbar_wait(done, 0);
    if (!have) atomicOr(p.err, 8);
    have = __all_sync(0xffffffffu, have);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    float* out = p.part + (size_t)z * p.M * p.N;
#pragma unroll 1
    for (int c = 0; c < width; c += 16) {
      uint32_t v[16];
      if (nk > 0 && have) {
        const uint32_t taddr = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)c;
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15},"
            " [%16];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
              "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
              "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(taddr));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = 0u;
      }
      if (row < p.M) {
        const int col0 = n0 + c;
        float* o = out + (size_t)row * p.N + col0;
        if ((p.N & 3) == 0 && col0 + 16 <= p.N) {
#pragma unroll
          for (int j = 0; j < 16; j += 4)
            *reinterpret_cast<float4*>(o + j) = make_float4(__uint_as_float(v[j]), __uint_as_float(v[j + 1]),
                                                            __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j)
            if (col0 + j < p.N) o[j] = __uint_as_float(v[j]);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync_all();   // no CTA frees its half while the other may still use it
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(BN));
  }
  cluster_sync_all();   // nor leaves before both halves are free
}

// ---------------------------------------------------------------------------
// Stage-1 contractions of the exchange terms, for every P and trial vector n:
//   C_P[n][i][r] = sum_(k<K) L_P[i][k] X[n][r][k]
// written as hi + lo parts into the stage-2 operand layout
//   out[P][(n, i)][r], row pitch ldo (128-byte rows, tc_zpad):
//   K1: L = L_oo ([i][j]), X = X^T per trial vector ([a][j])  -> Z[P][(n,i)][a]
//   K2: L = L_ov ([i][b]), X = X ([j][b])                     -> Q[P][(n,i)][j]
// One product over all rows (P, i) and columns (n, r): the columns run along the
// contiguous index of the output, so a thread (one TMEM lane = one row) converts
// 16 consecutive results at once, and each warp passes its piece through shared
// memory and writes 64-byte runs, the two halves of a line right after one
// another.  (With the roles swapped and rows of [(n,i)][P][r] it stored single
// 2-byte elements, 27 instructions per result.)  What bounds it: the stores of Z
// and the conversions share the load/store unit (n_vir 400: 0.45 ms without the
// stores, 0.93 with them); n_vir 1350: the MMAs' share of that, 0.68 of 1.05 ms.
// Straight 32-byte stores per row (46 L1 cycles an instruction) and bulk copies of
// 128 bytes (12 cycles each) were slower.
// Measured, 20 vectors of 60 x 400, 2000 rows: Z 1002 -> 931 us, Q 627 -> 278;
// 13 vectors of 24 x 144, 840 rows: Z 84 -> 43; 40 vectors of 150 x 1350, 127
// rows: Z 1340 -> 1050; FP8 ris, 20 vectors of 150 x 1350, 150 rows: 865 -> 472.
// Tiles of 256 rows x up to 256 columns by CTA pairs (cta_group::2, as in
// k1_pair_kernel), clusters of two persistent over the tiles; the TMEM
// accumulator is double-buffered so the stores of one tile overlap the MMAs of
// the next.  A tile's columns are gn whole trial vectors of wr columns each
// (R <= 128) or a part of one in whole 64-column units, so that 16-byte stores
// never cross vectors and a part begins on a 128-byte line.
// Rows of the output are padded to 128 bytes: with rows of pad8(R) elements the
// 64- to 512-byte runs of the stores straddled lines and sectors, which the L2
// completes from DRAM (1.5 to 3.5 TB/s written in a pattern of 2704-byte rows
// against 6.2 TB/s with 2816-byte ones, 7.1 TB/s for one long run).
constexpr int S1_EPI_WARPS = 16;                     // four per TMEM lane quadrant
constexpr int S1_THREADS = 64 + 32 * S1_EPI_WARPS;   // producer, MMA and the epilogue warps
constexpr int S1_RB = 64;                            // bytes of K per shared-memory row

struct S1Params {
  int rows, no, pn;    // pn * no rows (P, i)
  int R, m, ldo;       // columns (n, r): r < R, n < m
  int K, nkb;
  int gn, wr;          // gn > 1: trial vectors per tile and their column pitch
  int nt0, nq, nr;     // gn == 1: tiles per trial vector, col_unit-column units per tile (+1 for the first nr)
  int mt, ntile;       // row tiles, column tiles
  int mseg, units;     // row tiles of one unit of work, units (column tile fastest)
  int col_unit;        // columns of a unit (64, or 32 where one tile holds the vector)
  int b_rows;          // rows of half of the widest B tile
  void* out_hi;        // BF16 / FP16 parts (2-byte elements) or e4m3 bytes
  void* out_lo;
  // FP16 output: the accumulator times *mul before its split; FP8 output:
  // times mu[P] (one scale per auxiliary row)
  const float* mul;
  const float* mu;
  int* err;
};

__device__ __forceinline__ uint32_t pack_e4m3x4(const float* x) {
  const uint32_t a = __nv_cvt_float2_to_fp8x2(make_float2(x[0], x[1]), __NV_SATFINITE, __NV_E4M3);
  const uint32_t b = __nv_cvt_float2_to_fp8x2(make_float2(x[2], x[3]), __NV_SATFINITE, __NV_E4M3);
  return a | (b << 16);
}
__device__ __forceinline__ float from_e4m3(unsigned char q) {
  return __half2float(__half(__nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)q, __NV_E4M3)));
}

// Two FP32 operations at once.
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mul.rn.f32x2 z, x, y;\n"
      " mov.b64 {%0, %1}, z;\n}\n" : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n sub.rn.f32x2 z, x, y;\n"
      " mov.b64 {%0, %1}, z;\n}\n" : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}

// hi and lo parts of the 16 accumulator values v times f (BF16: no factor), packed
// in 32-bit words
template <int OUT>
__device__ __forceinline__ void split16(const uint32_t (&v)[16], float f, uint32_t* hi, uint32_t* lo) {
  if constexpr (OUT == ET_E4M3) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      float x[4], r[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) x[t] = __uint_as_float(v[4 * j + t]) * f;
      hi[j] = pack_e4m3x4(x);
#pragma unroll
      for (int t = 0; t < 4; ++t) r[t] = x[t] - from_e4m3((unsigned char)(hi[j] >> (8 * t)));
      lo[j] = pack_e4m3x4(r);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float2 x = make_float2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
      if constexpr (OUT == ET_F16) {
        x = mul2(x, make_float2(f, f));
        const __half2 h = __float22half2_rn(x);
        const __half2 l = __float22half2_rn(sub2(x, __half22float2(h)));
        hi[j] = *reinterpret_cast<const uint32_t*>(&h);
        lo[j] = *reinterpret_cast<const uint32_t*>(&l);
      } else {
        const __nv_bfloat162 h = __float22bfloat162_rn(x);
        const __nv_bfloat162 l = __float22bfloat162_rn(sub2(x, __bfloat1622float2(h)));
        hi[j] = *reinterpret_cast<const uint32_t*>(&h);
        lo[j] = *reinterpret_cast<const uint32_t*>(&l);
      }
    }
  }
}

// LSPLIT: the L operand (A) comes as hi + lo too (three products), else plain
// (two); X (B) is always hi + lo.  RES (K <= 160): the column tile's X rows stay
// in shared memory for the row tiles of a unit and the ring streams L only, half
// the bytes per MMA.
constexpr int S1_RES_KB = 5;
template <bool LSPLIT, bool RES> struct S1Cfg {
  static constexpr int AB = BM * S1_RB, HB = (BN / 2) * S1_RB;
  static constexpr int STAGE_BYTES = (LSPLIT ? 2 : 1) * AB + (RES ? 0 : 2 * HB);
  static constexpr int RES_BYTES = RES ? S1_RES_KB * 2 * HB : 0;
  static constexpr int STAGES = (RES ? 98304 : 163840) / STAGE_BYTES;
  // epilogue staging per warp: 32 rows of 64 bytes, 16-byte segments XORed with
  // bits 1-2 of the row (no bank conflicts by rows or by segments)
  static constexpr int EPI_BYTES = 32 * 64;
  static constexpr int EPI_OFF = RES_BYTES + STAGES * STAGE_BYTES;
  static constexpr int SMEM_BYTES = EPI_OFF + S1_EPI_WARPS * EPI_BYTES + 1024 + 512;
};

template <bool LSPLIT, bool RES, int IN, int OUT>
__global__ void __launch_bounds__(S1_THREADS, 1)
k_stage1_pair(const __grid_constant__ CUtensorMap mA_hi, const __grid_constant__ CUtensorMap mA_lo,
              const __grid_constant__ CUtensorMap mB_hi, const __grid_constant__ CUtensorMap mB_lo,
              const S1Params p) {
  using C = S1Cfg<LSPLIT, RES>;
  constexpr int STAGES = C::STAGES;
  constexpr int B_OFF = (LSPLIT ? 2 : 1) * C::AB;   // !RES: first B tile in a stage
  constexpr int BKE = S1_RB / 2;                  // K elements per k-block
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* bres = smem;                       // RES: the X rows, hi and lo per k-block
  unsigned char* ring = smem + C::RES_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::EPI_OFF + S1_EPI_WARPS * C::EPI_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* tfull = empty + STAGES;      // [2] accumulator complete (both CTAs)
  uint64_t* tempty = tfull + 2;          // [2] accumulator read by this CTA's warps (the leader's: and the other's)
  uint64_t* bfull = tempty + 2;          // RES: the unit's X rows have landed (leader) ...
  uint64_t* bempty = bfull + 1;          // ... and its MMAs have read them
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bempty + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int h = (int)(rank & 1u);
  const int ncl = gridDim.x >> 1, cl = blockIdx.x >> 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], S1_EPI_WARPS / 2 + (h == 0 ? 1 : 0)); }
    mbar_init(bfull, 1);
    mbar_init(bempty, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  cluster_sync_all();   // every barrier of the cluster initialised, and both CTAs of a pair running
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)), "r"(2 * BN));
  }
  __syncthreads();
  cluster_sync_all();   // both CTAs' tensor memory allocated
  if (warp == 1) pair_relinquish();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  // column tile ct: first trial vector, first r, columns
  auto columns = [&](int ct, int& n0, int& r0, int& width) {
    if (p.gn > 1) {
      n0 = ct * p.gn;
      r0 = 0;
      width = p.gn * p.wr;
    } else {
      n0 = ct / p.nt0;
      const int t = ct - n0 * p.nt0;
      r0 = p.col_unit * (t * p.nq + min(t, p.nr));
      width = p.col_unit * (p.nq + (t < p.nr ? 1 : 0));
    }
  };

  if (warp == 0 && lane == 0) {
    // ---- TMA producer (both CTAs)
    const uint32_t lead_full = mapa(smem_u32(full), 0u), lead_bfull = mapa(smem_u32(bfull), 0u);
    const uint32_t bytes_a = 2u * (LSPLIT ? 2u : 1u) * C::AB, bytes_b = 4u * (uint32_t)p.b_rows * S1_RB;
    int i = 0, w = 0, xw = 0;   // xw: units whose X rows have been asked for
    bool ok = true;
    for (int u = cl; u < p.units && ok; u += ncl, ++w) {
      int n0, r0, width;
      columns(u % p.ntile, n0, r0, width);
      const int nb = p.gn > 1 ? n0 + h * (p.gn / 2) : n0, rb = p.gn > 1 ? 0 : r0 + h * (width / 2);
      const int mt0 = (u / p.ntile) * p.mseg, mt1 = min(p.mt, mt0 + p.mseg);
      if constexpr (RES) {
        if (!mbar_wait(bempty, ((uint32_t)w & 1u) ^ 1u)) { atomicOr(p.err, 16); ok = false; break; }
        if (h == 0) mbar_expect_tx(bfull, bytes_b * (uint32_t)p.nkb);
        for (int kb = 0; kb < p.nkb; ++kb) {
          tma_load_3d_pair(bres + kb * 2 * C::HB, &mB_hi, lead_bfull, kb * BKE, rb, nb);
          tma_load_3d_pair(bres + kb * 2 * C::HB + C::HB, &mB_lo, lead_bfull, kb * BKE, rb, nb);
        }
        ++xw;
      }
      for (int mt = mt0; mt < mt1 && ok; ++mt) {
        const int m0 = mt * 2 * BM + h * BM;
        for (int kb = 0; kb < p.nkb; ++kb, ++i) {
          const int s = i % STAGES;
          if (!mbar_wait(&empty[s], ((uint32_t)(i / STAGES) & 1u) ^ 1u)) { atomicOr(p.err, 16); ok = false; break; }
          unsigned char* st = ring + s * C::STAGE_BYTES;
          const uint32_t bar = lead_full + (uint32_t)(s * 8);
          if (h == 0) mbar_expect_tx(&full[s], bytes_a + (RES ? 0u : bytes_b));
          tma_load_3d_pair(st, &mA_hi, bar, kb * BKE, m0, 0);
          if (LSPLIT) tma_load_3d_pair(st + C::AB, &mA_lo, bar, kb * BKE, m0, 0);
          if constexpr (!RES) {
            tma_load_3d_pair(st + B_OFF, &mB_hi, bar, kb * BKE, rb, nb);
            tma_load_3d_pair(st + B_OFF + C::HB, &mB_lo, bar, kb * BKE, rb, nb);
          }
        }
      }
    }
    // the copies already issued (they signal the leader) land, and the last commits
    // arrive on this CTA's `empty` barriers, before a CTA can exit
    if (h == 0)
      for (int j = max(0, i - STAGES); j < i; ++j)
        if (!mbar_wait(&full[j % STAGES], (uint32_t)(j / STAGES) & 1u)) { atomicOr(p.err, 32); break; }
    for (int j = i; j < i + STAGES; ++j)
      if (!mbar_wait(&empty[j % STAGES], ((uint32_t)(j / STAGES) & 1u) ^ 1u)) { atomicOr(p.err, 32); break; }
    if (RES) {
      if (h == 0 && xw > 0 && !mbar_wait(bfull, (uint32_t)(xw - 1) & 1u)) atomicOr(p.err, 32);
      if (ok && !mbar_wait(bempty, ((uint32_t)w & 1u) ^ 1u)) atomicOr(p.err, 32);
    }
  } else if (warp == 1 && lane == 0 && h == 0) {
    // ---- MMA issuer (the leader)
    int i = 0, j = 0, w = 0;
    bool ok = true;
    for (int u = cl; u < p.units && ok; u += ncl, ++w) {
      int n0, r0, width;
      columns(u % p.ntile, n0, r0, width);
      const int mt0 = (u / p.ntile) * p.mseg, mt1 = min(p.mt, mt0 + p.mseg);
      const uint32_t idesc =
          (1u << 4) | Elem<IN>::TYPE_BITS | ((uint32_t)(width >> 3) << 17) | ((uint32_t)(2 * BM >> 4) << 24);
      if (RES && !mbar_wait(bfull, (uint32_t)w & 1u)) { atomicOr(p.err, 128); break; }
      for (int mt = mt0; mt < mt1 && ok; ++mt, ++j) {
        const int buf = j & 1;
        if (!mbar_wait(&tempty[buf], ((uint32_t)(j >> 1) & 1u) ^ 1u)) { atomicOr(p.err, 64); ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t acc = tmem + (uint32_t)(buf * BN);
        for (int kb = 0; kb < p.nkb; ++kb, ++i) {
          const int s = i % STAGES;
          if (!mbar_wait(&full[s], (uint32_t)(i / STAGES) & 1u)) { atomicOr(p.err, 128); ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          unsigned char* st = ring + s * C::STAGE_BYTES;
          unsigned char* bt = RES ? bres + kb * 2 * C::HB : st + B_OFF;
          const uint64_t ah = sdesc_rb<S1_RB>(st), bh = sdesc_rb<S1_RB>(bt), bl = sdesc_rb<S1_RB>(bt + C::HB);
          const int rem = p.K - kb * BKE;   // the zero-filled tail issues no MMA
#pragma unroll
          for (int kk = 0; kk < S1_RB / 32; ++kk) {
            if (kk * 16 < rem) {
              const uint64_t off = (uint64_t)(kk * 32) >> 4;
              mma_pair<IN, 1>(acc, ah + off, bh + off, (kb > 0 || kk > 0) ? 1u : 0u, idesc);
              mma_pair<IN, 2>(acc, ah + off, bl + off, 1u, idesc);
              if (LSPLIT) mma_pair<IN, 0>(acc, sdesc_rb<S1_RB>(st + C::AB) + off, bh + off, 1u, idesc);
            }
          }
          commit_pair(&empty[s], (uint16_t)3);
        }
        commit_pair(&tfull[buf], (uint16_t)3);
      }
      if (RES) commit_pair(bempty, (uint16_t)3);
    }
  } else if (warp == 1 && lane == 0) {
    // ---- the other CTA passes its "accumulator read" on to the leader: a remote
    // arrival releases at cluster scope, which in an epilogue warp would wait for
    // all of its global stores
    const uint32_t lead_tempty = mapa(smem_u32(tempty), 0u);
    int j = 0;
    bool ok = true;
    for (int u = cl; u < p.units && ok; u += ncl) {
      const int mt0 = (u / p.ntile) * p.mseg, mt1 = min(p.mt, mt0 + p.mseg);
      for (int mt = mt0; mt < mt1; ++mt, ++j) {
        const int buf = j & 1;
        if (!mbar_wait(&tempty[buf], (uint32_t)(j >> 1) & 1u)) { atomicOr(p.err, 64); ok = false; break; }
        asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(
                         lead_tempty + (uint32_t)(buf * 8))
                     : "memory");
      }
    }
  } else if (warp >= 2) {
    // ---- epilogue: two groups of eight warps take turns by tile, so that one
    // converts while the other's stores drain; a warp takes TMEM lane quadrant q and
    // every second 64-column chunk, in two halves (each as hi, then lo) through
    // the staging rows
    const int q = warp & 3, part = ((warp - 2) >> 2) & 1, group = (warp - 2) >> 3;
    const float mul = OUT == ET_F16 ? *p.mul : 1.f;
    constexpr int OB = OUT == ET_E4M3 ? 1 : 2;    // bytes per element
    constexpr int NW = 4 * OB;                    // 32-bit words of 16 elements
    constexpr int CC = 64 / OB;                   // columns of a staged piece
    constexpr int SEG = 16 / OB;                  // columns of a 16-byte segment
    unsigned char* st = smem + C::EPI_OFF + (warp - 2) * C::EPI_BYTES;
    unsigned char* srow = st + lane * 64;
    const int sx = (lane >> 1) & 3;               // segment swizzle of this lane's staging row
    // the segment that this lane stores: row (lane >> 2) + 8 it, whose swizzle is (lane >> 3) & 3
    const unsigned char* srd = st + (lane >> 2) * 64 + (((lane & 3) ^ ((lane >> 3) & 3)) * 16);
    const int prow = p.m * p.no;                  // output rows per P
    int j = 0;
    bool ok = true;
    for (int u = cl; u < p.units && ok; u += ncl) {
      int n0, r0, width;
      columns(u % p.ntile, n0, r0, width);
      const int mt0 = (u / p.ntile) * p.mseg, mt1 = min(p.mt, mt0 + p.mseg);
    for (int mt = mt0; mt < mt1; ++mt, ++j) {
      if ((j & 1) != group) continue;
      const int row = mt * 2 * BM + h * BM + q * 32 + lane;
      const int buf = group;
      ok = mbar_wait(&tfull[buf], (uint32_t)(j >> 1) & 1u);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) { if (lane == 0) atomicOr(p.err, 256); break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // output row of this lane's (P, i) for trial vector 0; -1 beyond the rows
      const int P = row / p.no;
      const int orow = row < p.rows ? P * prow + (row - P * p.no) : -1;
      const float f = OUT == ET_E4M3 ? (row < p.rows ? p.mu[P] : 0.f) : mul;
      const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * BN);
      // offsets of the rows that this lane stores (four lanes write a row's 64 bytes,
      // eight rows at a time)
      long long roff[4];
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        const int o = __shfl_sync(0xffffffffu, orow, it * 8 + (lane >> 2));
        roff[it] = o < 0 ? -1 : (long long)o * p.ldo * OB;
      }
      auto read_done = [&] {   // this warp's reads of the accumulator have completed
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0)
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty[buf])) : "memory");
      };
      // this warp's pieces: chunks part and part + 2 in halves of CC columns
      constexpr int PC = 64 / CC;               // pieces per chunk
      const int chunks = (width + 63) / 64;
      const int mine = ((chunks - part + 1) / 2) * PC;
      int left = 0;                              // pieces that hold columns
      for (int e = 0; e < mine; ++e) left += ((part + 2 * (e / PC)) * 64 + (e % PC) * CC < width) ? 1 : 0;
      if (left == 0) read_done();
#pragma unroll 1
      for (int e = 0; e < mine; ++e) {
        const int c0 = (part + 2 * (e / PC)) * 64 + (e % PC) * CC;
        if (c0 >= width) continue;
        uint32_t lo[CC / 16][NW];
        __syncwarp();
#pragma unroll
        for (int g = 0; g < CC / 16; g += 2) {
          uint32_t v[2][16];
#pragma unroll
          for (int u = 0; u < 2; ++u)
            if (c0 + 16 * (g + u) < width)
              asm volatile(
                  "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15},"
                  " [%16];"
                  : "=r"(v[u][0]), "=r"(v[u][1]), "=r"(v[u][2]), "=r"(v[u][3]), "=r"(v[u][4]), "=r"(v[u][5]),
                    "=r"(v[u][6]), "=r"(v[u][7]), "=r"(v[u][8]), "=r"(v[u][9]), "=r"(v[u][10]), "=r"(v[u][11]),
                    "=r"(v[u][12]), "=r"(v[u][13]), "=r"(v[u][14]), "=r"(v[u][15])
                  : "r"(tb + (uint32_t)(c0 + 16 * (g + u))));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            uint32_t hi[NW];
            split16<OUT>(v[u], f, hi, lo[g + u]);
#pragma unroll
            for (int k = 0; k < NW; k += 4)
              *reinterpret_cast<uint4*>(srow + ((((g + u) * OB + k / 4) ^ sx) * 16)) =
                  make_uint4(hi[k], hi[k + 1], hi[k + 2], hi[k + 3]);
          }
        }
        if (--left == 0) read_done();
        // this lane's 16-byte segment: trial vector and r (the row's padding is never read)
        const int seg = (lane & 3) * SEG, c = c0 + seg;
        const int nn = p.gn > 1 ? c / p.wr : 0;
        const int n = n0 + nn, r = r0 + c - nn * p.wr;
        const bool live = c < width && n < p.m && r < p.ldo;
        const long long coff = ((long long)n * p.no * p.ldo + r) * OB;
        auto store_rows = [&](unsigned char* out) {
          __syncwarp();
#pragma unroll
          for (int it = 0; it < 4; ++it)
            if (live && roff[it] >= 0)
              *reinterpret_cast<uint4*>(out + roff[it] + coff) = *reinterpret_cast<const uint4*>(srd + it * 512);
        };
        store_rows(static_cast<unsigned char*>(p.out_hi));
        __syncwarp();
#pragma unroll
        for (int g = 0; g < CC / 16; ++g)
#pragma unroll
          for (int k = 0; k < NW; k += 4)
            *reinterpret_cast<uint4*>(srow + (((g * OB + k / 4) ^ sx) * 16)) =
                make_uint4(lo[g][k], lo[g][k + 1], lo[g][k + 2], lo[g][k + 3]);
        store_rows(static_cast<unsigned char*>(p.out_lo));
      }
    }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync_all();   // no CTA frees its half while the other may still use it
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BN));
  }
  cluster_sync_all();   // nor leaves before both halves are free
}

__device__ __forceinline__ unsigned char to_e4m3(float x) {
  return (unsigned char)__nv_cvt_float_to_fp8(x, __NV_SATFINITE, __NV_E4M3);
}

// Sum the split partials into out (FP32), accumulating when asked.
// With `scale` (device scalar), the summed partials are multiplied by *scale
// before they are added (the FP8 operands carry a scale factor).
__global__ void k_sum_splits(const float* __restrict__ part, int S, long long MN, float* out,
                             int accumulate, const float* __restrict__ scale) {
  if (!scale) {
    for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < MN;
         t += (long long)gridDim.x * blockDim.x) {
      float acc = accumulate ? out[t] : 0.f;
      for (int s = 0; s < S; ++s) acc += part[s * MN + t];
      out[t] = acc;
    }
    return;
  }
  const float f = *scale;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < MN;
       t += (long long)gridDim.x * blockDim.x) {
    float acc = 0.f;
    for (int s = 0; s < S; ++s) acc += part[s * MN + t];
    out[t] = (accumulate ? out[t] : 0.f) + f * acc;
  }
}

// Split of x (converted to FP32, times *scale when given) into two 16-bit
// parts hi = round(x), lo = round(x - hi) of the element type E (BF16 or
// FP16); lo optional.
template <typename E> __device__ __forceinline__ E to_elem(float x);
template <> __device__ __forceinline__ __nv_bfloat16 to_elem<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }
template <> __device__ __forceinline__ __half to_elem<__half>(float x) { return __float2half_rn(x); }
__device__ __forceinline__ float from_elem(__nv_bfloat16 x) { return __bfloat162float(x); }
__device__ __forceinline__ float from_elem(__half x) { return __half2float(x); }

template <typename E>
__device__ __forceinline__ void split_store(float v, long long t, E* hi, E* lo) {
  const E h = to_elem<E>(v);
  hi[t] = h;
  if (lo) lo[t] = to_elem<E>(v - from_elem(h));
}

// Transpose + split of factor rows: src [rows][n1][n2] -> dst [rows][n2][pad8(n1)]
// (dst[r][b][a] = src[r][a][b]; pads zero).  lo may be NULL (one part).
template <typename TS, typename E>
__global__ void k_transpose_split(const TS* __restrict__ src, int rows, int n1, int n2, int ld,
                                  const float* __restrict__ scale, E* hi, E* lo) {
  const long long tot = (long long)rows * n2 * ld;
  const float sc = scale ? *scale : 1.f;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
       t += (long long)gridDim.x * blockDim.x) {
    const int a = (int)(t % ld);
    const long long rb = t / ld;
    const int b = (int)(rb % n2);
    const long long r = rb / n2;
    float v = 0.f;
    if (a < n1) v = (float)src[(r * n1 + a) * n2 + b] * sc;
    split_store<E>(v, t, hi, lo);
  }
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                              CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                              CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
  static EncodeFn fn = nullptr;
  if (!fn) {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    TD_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q));
    TD_REQUIRE(f != nullptr && q == cudaDriverEntryPointSuccess, TDDFT_ERR_CUDA,
               "cuTensorMapEncodeTiled unavailable");
    fn = reinterpret_cast<EncodeFn>(f);
  }
  return fn;
}

// 3-D tiled map with 128-byte swizzle over elements of type et (ET_BF16,
// ET_F16 or ET_E4M3, the last as bytes).
CUtensorMap make_map(const void* base, const cuuint64_t dims[3], const cuuint64_t strides[2],
                     const cuuint32_t box[3], int et = ET_BF16, int swizzle_bytes = 128) {
  TD_REQUIRE((reinterpret_cast<uintptr_t>(base) & 15) == 0, TDDFT_ERR_ARG, "TMA base not 16-byte aligned");
  TD_REQUIRE(strides[0] % 16 == 0 && strides[1] % 16 == 0, TDDFT_ERR_ARG, "TMA strides not 16-byte multiples");
  CUtensorMap m;
  const cuuint32_t es[3] = {1, 1, 1};
  const CUtensorMapDataType dt = et == ET_E4M3 ? CU_TENSOR_MAP_DATA_TYPE_UINT8
                                 : (et == ET_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16);
  CUresult r = encode_fn()(&m, dt, 3,
                           const_cast<void*>(base), dims, strides,
                           box, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           swizzle_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  TD_REQUIRE(r == CUDA_SUCCESS, TDDFT_ERR_CUDA, "cuTensorMapEncodeTiled failed");
  return m;
}

}  // namespace

CUtensorMap tc_map_f16_4d(const void* base, const uint64_t dims[4], const uint64_t strides[3], const uint32_t box[4],
                          int swizzle_bytes) {
  TD_REQUIRE((reinterpret_cast<uintptr_t>(base) & 15) == 0, TDDFT_ERR_ARG, "TMA base not 16-byte aligned");
  TD_REQUIRE(strides[0] % 16 == 0 && strides[1] % 16 == 0 && strides[2] % 16 == 0, TDDFT_ERR_ARG,
             "TMA strides not 16-byte multiples");
  CUtensorMap m;
  cuuint64_t d[4], st[3];
  cuuint32_t b[4];
  const cuuint32_t es[4] = {1, 1, 1, 1};
  for (int i = 0; i < 4; ++i) { d[i] = dims[i]; b[i] = box[i]; }
  for (int i = 0; i < 3; ++i) st[i] = strides[i];
  CUresult r = encode_fn()(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, const_cast<void*>(base), d, st, b, es,
                           CU_TENSOR_MAP_INTERLEAVE_NONE,
                           swizzle_bytes == 64 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B,
                           CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  TD_REQUIRE(r == CUDA_SUCCESS, TDDFT_ERR_CUDA, "cuTensorMapEncodeTiled failed");
  return m;
}

int tc_pad(int nv) { return (nv + 7) & ~7; }
int tc_pad16(int n) { return (n + 15) & ~15; }
int tc_zpad(int n, int es) { return (n + 128 / es - 1) & ~(128 / es - 1); }

namespace {
template <typename E>
void transpose_split_t(const void* src, DType ts, int rows, int n1, int n2, const float* scale, E* hi, E* lo,
                       cudaStream_t s) {
  const int ld = tc_pad(n1);
  const long long tot = (long long)rows * n2 * ld;
  long long g = (tot + 255) / 256;
  if (g > 152 * 16) g = 152 * 16;
  if (ts == DType::F32)
    k_transpose_split<float, E><<<(unsigned)g, 256, 0, s>>>((const float*)src, rows, n1, n2, ld, scale, hi, lo);
  else if (ts == DType::BF16)
    k_transpose_split<__nv_bfloat16, E><<<(unsigned)g, 256, 0, s>>>((const __nv_bfloat16*)src, rows, n1, n2, ld,
                                                                    scale, hi, lo);
  else
    k_transpose_split<double, E><<<(unsigned)g, 256, 0, s>>>((const double*)src, rows, n1, n2, ld, scale, hi, lo);
}
}  // namespace

void tc_transpose_split(const void* src, DType ts, int rows, int n1, int n2, void* hi, void* lo, TcElt et,
                        const float* scale, cudaStream_t s) {
  TD_REQUIRE(et == TcElt::F16 || scale == nullptr, TDDFT_ERR_ARG, "tc_transpose_split: BF16 parts take no scale");
  if (et == TcElt::F16)
    transpose_split_t<__half>(src, ts, rows, n1, n2, scale, (__half*)hi, (__half*)lo, s);
  else
    transpose_split_t<__nv_bfloat16>(src, ts, rows, n1, n2, scale, (__nv_bfloat16*)hi, (__nv_bfloat16*)lo, s);
  count_launch();
  TD_LAUNCH_CHECK();
}

// SMs of the current device (queried once).
int sm_count() {
  static int n = 0;
  if (n == 0) {
    int dev = 0, v = 0;
    if (cudaGetDevice(&dev) == cudaSuccess &&
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && v > 0)
      n = v;
    else
      n = 152;
  }
  return n;
}

// Work split for a grid of `tiles` x splits CTAs, one CTA per SM, each taking
// ceil(total / splits) consecutive units: the launch lasts (number of waves) x
// (units per CTA + a fixed per-CTA cost of `overhead` units), so a last,
// nearly empty wave costs as much as a full one.  Tries the splits that fill
// one to four waves and keeps the cheapest (the fewest splits on ties).
int wave_splits(int tiles, int total, int overhead, int sms) {
  if (sms <= 0) sms = sm_count();
  int best = 1;
  long long best_cost = -1;
  for (int w = 1; w <= 4; ++w) {
    int sp = std::max(1, (w * sms) / std::max(tiles, 1));
    sp = std::min(sp, std::max(total, 1));
    const int per = (total + sp - 1) / sp;
    sp = (total + per - 1) / per;
    const long long waves = ((long long)tiles * sp + sms - 1) / sms;
    const long long cost = waves * (per + overhead);
    if (best_cost < 0 || cost < best_cost || (cost == best_cost && sp < best)) {
      best_cost = cost;
      best = sp;
    }
  }
  return best;
}

namespace {
bool cluster_pairs_enabled() {
  const char* e = std::getenv("TDDFT_TC_CLUSTER");
  return !(e && e[0] == '0');
}

bool cluster_quads_enabled() {
  const char* e = std::getenv("TDDFT_TC_QUAD");
  return !(e && e[0] == '0');
}

// CTAs of the paired contraction that can be resident at once: two per
// co-resident cluster (an SM left over in a GPC takes no pair).
int pair_slots() {
  static int c = 0;
  if (c == 0) {
    const void* k = (const void*)k1_pair_kernel<BOTH, ET_F16, 1, 64>;
    const int smem = PCfg<BOTH, 64>::SMEM_BYTES;
    ensure_smem(k, smem);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(2, 1, 1);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, k, &cfg) != cudaSuccess || n <= 0) {
      (void)cudaGetLastError();
      n = sm_count() / 2;
    }
    c = 2 * n;
  }
  return c;
}

// Operands of one contraction; the pointers are FP16 / BF16 parts or e4m3 bytes.
struct Contraction {
  const void *Ahi, *Alo;
  int M, pn, Kin;
  const void *Bhi, *Blo;
  int N, lda, ldb, es; // row pitches (elements), element bytes
  int total, per, splits, nab;
  float* part;
  int* err;
  cudaStream_t s;
  KernelProfile* prof;
  double prof_flops, prof_bytes;
};

template <int MODE, int ET, int RB>
void launch_pair(const Contraction& c) {
  constexpr int BKE = Elem<ET>::BKE * RB / 128;
  const int mt = (c.M + BM - 1) / BM, nt0 = (c.N + BN - 1) / BN;
  const int cx = nt0 > 1 && cluster_quads_enabled() ? 2 : 1;
  const int units = (c.N + 31) / 32;
  PairParams p;
  p.M = c.M;
  p.N = c.N;
  p.Kin = c.Kin;
  p.nab = c.nab;
  p.total = c.total;
  p.per_split = c.per;
  p.nt0 = nt0;
  p.nt = (nt0 + cx - 1) / cx * cx;
  p.mp = (mt + 1) / 2;
  p.nq = units / nt0;
  p.nr = units % nt0;
  p.b_rows = 16 * (p.nq + (p.nr ? 1 : 0));
  p.part = c.part;
  p.err = c.err;
  const cuuint64_t dA[3] = {(cuuint64_t)c.Kin, (cuuint64_t)c.pn, (cuuint64_t)c.M};
  const cuuint64_t sA[2] = {(cuuint64_t)c.M * c.lda * c.es, (cuuint64_t)c.lda * c.es};
  const cuuint32_t bA[3] = {(cuuint32_t)BKE, 1, (cuuint32_t)(BM / cx)};
  const cuuint64_t dB[3] = {(cuuint64_t)c.Kin, (cuuint64_t)c.N, (cuuint64_t)c.pn};
  const cuuint64_t sB[2] = {(cuuint64_t)c.ldb * c.es, (cuuint64_t)c.N * c.ldb * c.es};
  const cuuint32_t bB[3] = {(cuuint32_t)BKE, (cuuint32_t)p.b_rows, 1};
  const CUtensorMap mAh = make_map(c.Ahi, dA, sA, bA, ET, RB), mBh = make_map(c.Bhi, dB, sB, bB, ET, RB);
  const CUtensorMap mAl = c.Alo ? make_map(c.Alo, dA, sA, bA, ET, RB) : mAh;
  const CUtensorMap mBl = c.Blo ? make_map(c.Blo, dB, sB, bB, ET, RB) : mBh;
  auto go = [&](auto kernel) {
    constexpr int smem = PCfg<MODE, RB>::SMEM_BYTES;
    ensure_smem((const void*)kernel, smem);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2 * cx;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(2 * p.mp * p.nt * c.splits), 1, 1);
    cfg.blockDim = dim3(THREADS);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = c.s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (c.prof) c.prof->begin(c.s);
    TD_CUDA(cudaLaunchKernelEx(&cfg, kernel, mAh, mAl, mBh, mBl, p));
    if (c.prof) c.prof->end(c.s, c.prof_flops, c.prof_bytes);
  };
  if (cx > 1) go(k1_pair_kernel<MODE, ET, 2, RB>);
  else go(k1_pair_kernel<MODE, ET, 1, RB>);
}

template <int MODE, int ET, int RB>
void launch_single(const Contraction& c) {
  constexpr int BKE = Elem<ET>::BKE * RB / 128;
  const cuuint64_t dA[3] = {(cuuint64_t)c.Kin, (cuuint64_t)c.pn, (cuuint64_t)c.M};
  const cuuint64_t sA[2] = {(cuuint64_t)c.M * c.lda * c.es, (cuuint64_t)c.lda * c.es};
  const cuuint32_t bA[3] = {(cuuint32_t)BKE, 1, BM};
  const cuuint64_t dB[3] = {(cuuint64_t)c.Kin, (cuuint64_t)c.N, (cuuint64_t)c.pn};
  const cuuint64_t sB[2] = {(cuuint64_t)c.ldb * c.es, (cuuint64_t)c.N * c.ldb * c.es};
  const cuuint32_t bB[3] = {(cuuint32_t)BKE, BN, 1};
  const CUtensorMap mAh = make_map(c.Ahi, dA, sA, bA, ET, RB), mBh = make_map(c.Bhi, dB, sB, bB, ET, RB);
  const CUtensorMap mAl = c.Alo ? make_map(c.Alo, dA, sA, bA, ET, RB) : mAh;
  const CUtensorMap mBl = c.Blo ? make_map(c.Blo, dB, sB, bB, ET, RB) : mBh;
  const Params p{c.M, c.N, c.Kin, c.nab, c.total, c.per, c.part, c.err};
  const dim3 grid((c.N + BN - 1) / BN, (c.M + BM - 1) / BM, c.splits);
  constexpr int smem = Cfg<MODE, RB>::SMEM_BYTES;
  ensure_smem((const void*)k1_tc_kernel<MODE, ET, RB>, smem);
  if (c.prof) c.prof->begin(c.s);
  k1_tc_kernel<MODE, ET, RB><<<grid, THREADS, smem, c.s>>>(mAh, mAl, mBh, mBl, p);
  if (c.prof) c.prof->end(c.s, c.prof_flops, c.prof_bytes);
}

// Pairs of CTAs where there are two M tiles or more, one CTA per tile below;
// both form the same sums, bit for bit (TDDFT_TC_CLUSTER=0 keeps single CTAs).
template <int MODE, int ET, int RB>
void launch_contraction(const Contraction& c) {
  if (c.M > BM && cluster_pairs_enabled()) launch_pair<MODE, ET, RB>(c);
  else launch_single<MODE, ET, RB>(c);
  count_launch();
  TD_LAUNCH_CHECK();
}

void sum_splits(const Contraction& c, float* out, bool accumulate, const float* scale) {
  const long long MN = (long long)c.M * c.N;
  long long g = (MN + 255) / 256;
  if (g > 152 * 16) g = 152 * 16;
  k_sum_splits<<<(unsigned)g, 256, 0, c.s>>>(c.part, c.splits, MN, out, accumulate ? 1 : 0, scale);
  count_launch();
  TD_LAUNCH_CHECK();
}

void finish_sums(const Contraction& c, DevBuf& part, float* out, bool accumulate, const float* scale, TcSum* keep) {
  if (!keep) {
    sum_splits(c, out, accumulate, scale);
    return;
  }
  const size_t mn = (size_t)c.M * c.N * 4;
  if (c.splits * mn <= kKeepBytes) {
    keep->part = std::move(part);
    keep->splits = c.splits;
    keep->scale = scale;
  } else {   // too much to hold on to
    keep->part = DevBuf(mn, c.s);
    sum_splits(c, keep->part.as<float>(), false, scale);
    keep->splits = 1;
    keep->scale = nullptr;
  }
}
}  // namespace

void tc_contract(const void* Ahi, const void* Alo, int lda, int M, int pn, int Kin, const void* Bhi, const void* Blo,
                 int N, float* out, bool accumulate, TcElt elt, const float* scale, int* err, cudaStream_t s,
                 KernelProfile* prof, double prof_flops, double prof_bytes, int max_kb, TcSum* keep) {
  if (M <= 0 || pn <= 0 || N <= 0) return;
  const int mode = Blo ? BOTH : ASPLIT;
  TD_REQUIRE(Alo != nullptr && mode == (elt == TcElt::F16 ? BOTH : ASPLIT), TDDFT_ERR_ARG,
             "tc_contract: FP16 operands come as hi + lo on both sides, BF16 ones with a plain B");
  // the split-B products run on 64-byte K rows (a deeper ring), the others on 128-byte rows
  const int rb = mode == BOTH ? 64 : 128;
  const int bke = BK * rb / 128;
  const int nab = (Kin + bke - 1) / bke;
  const int total = pn * nab;
  if (max_kb > 0) max_kb = max_kb * (BK / bke);   // max_kb counts 64-element k-blocks
  const int mt = (M + BM - 1) / BM, nt = (N + BN - 1) / BN;
  // a CTA's fixed cost (barriers, TMEM, pipeline fill, 128 KB epilogue) is about
  // four 64-element k-blocks of MMA work.  The split count depends on the
  // problem only (its own tiles, the pairs' residency), not on the cluster
  // shape of the launch: every shape then forms the same sums, bit for bit.
  int splits = wave_splits(mt * nt, total, 4 * (BK / bke), mode == BOTH && mt > 1 ? pair_slots() : 0);
  if (max_kb > 0) splits = std::max(splits, (total + max_kb - 1) / max_kb);   // bounded accumulation runs
  const int per = (total + splits - 1) / splits;
  splits = (total + per - 1) / per;
  DevBuf part((size_t)splits * M * N * 4, s);
  const Contraction c{Ahi, Alo, M, pn, Kin, Bhi, Blo, N, lda, tc_pad(Kin), 2, total, per, splits, nab,
                      part.as<float>(), err, s, prof, prof_flops, prof_bytes};
  if (mode == BOTH) launch_contraction<BOTH, ET_F16, 64>(c);
  else launch_contraction<ASPLIT, ET_BF16, 128>(c);
  finish_sums(c, part, out, accumulate, scale, keep);
}

void tc_contract8(const unsigned char* Ahi, const unsigned char* Alo, int M, int pn, int Kin,
                  const unsigned char* B, int N, float* out, bool accumulate, const float* scale, int* err,
                  cudaStream_t s, TcSum* keep) {
  if (M <= 0 || pn <= 0 || N <= 0) return;
  TD_REQUIRE(Ahi && Alo && B && scale, TDDFT_ERR_ARG, "tc_contract8: operands missing");
  constexpr int BKE = Elem<ET_E4M3>::BKE;
  const int nab = (Kin + BKE - 1) / BKE;
  const int total = pn * nab;
  const int mt = (M + BM - 1) / BM, nt = (N + BN - 1) / BN;
  int splits = wave_splits(mt * nt, total, 4);
  const int per = (total + splits - 1) / splits;
  splits = (total + per - 1) / per;
  DevBuf part((size_t)splits * M * N * 4, s);
  const Contraction c{Ahi, Alo, M, pn, Kin, B, nullptr, N, tc_zpad(Kin, 1), tc_pad16(Kin), 1, total, per, splits, nab,
                      part.as<float>(), err, s, nullptr, 0.0, 0.0};
  launch_contraction<ASPLIT, ET_E4M3, 128>(c);
  finish_sums(c, part, out, accumulate, scale, keep);
}

namespace {
// out_is8: e4m3 outputs with per-P multipliers mu (X as BF16 hi + lo, L plain);
// otherwise 16-bit outputs of the inputs' element type et, FP16 ones times *mul.
void stage1_impl(const void* Xhi, const void* Xlo, int m, int R, int K, const void* Lhi, const void* Llo, int no,
                 int pn, int et, bool out_is8, void* out_hi, void* out_lo, const float* mul, const float* mu, int* err,
                 cudaStream_t s) {
  if (m <= 0 || R <= 0 || pn <= 0 || no <= 0) return;
  TD_REQUIRE(no <= 256, TDDFT_ERR_ARG, "tc_stage1: n_occ above 256");
  TD_REQUIRE(Xhi && Xlo && Lhi && out_hi && out_lo && (!out_is8 || mu != nullptr) && (et == ET_F16) == (Llo != nullptr),
             TDDFT_ERR_ARG, "tc_stage1: hi/lo operands mismatch");
  TD_REQUIRE((et == ET_F16) == (mul != nullptr) && (!out_is8 || et == ET_BF16), TDDFT_ERR_ARG,
             "tc_stage1: FP16 outputs need a multiplier, FP8 outputs BF16 inputs");
  const int ldk = tc_pad(K);
  S1Params p;
  p.rows = pn * no;
  p.no = no;
  p.pn = pn;
  p.R = R;
  p.m = m;
  p.ldo = tc_zpad(R, out_is8 ? 1 : 2);
  p.K = K;
  p.nkb = (K + S1_RB / 2 - 1) / (S1_RB / 2);
  // several trial vectors per tile while they fit, else equal parts of one
  p.wr = (R + 15) & ~15;
  p.gn = 1;
  while (2 * p.gn * p.wr <= BN && p.gn < m) p.gn *= 2;
  p.nt0 = (R + BN - 1) / BN;
  p.col_unit = p.nt0 > 1 ? 64 : 32;
  const int units = (R + p.col_unit - 1) / p.col_unit;
  p.nq = units / p.nt0;
  p.nr = units % p.nt0;
  p.mt = (p.rows + 2 * BM - 1) / (2 * BM);
  p.ntile = p.gn > 1 ? (m + p.gn - 1) / p.gn : m * p.nt0;
  p.b_rows = p.gn > 1 ? p.gn / 2 * p.wr : p.col_unit / 2 * (p.nq + (p.nr ? 1 : 0));
  p.out_hi = out_hi;
  p.out_lo = out_lo;
  p.mul = mul;
  p.mu = mu;
  p.err = err;
  TD_REQUIRE((long long)p.mt * p.ntile < (1ll << 30) && (long long)m * no * pn < (1ll << 31), TDDFT_ERR_ARG, "tc_stage1: problem too large");
  const cuuint64_t dA[3] = {(cuuint64_t)K, (cuuint64_t)p.rows, 1};
  const cuuint64_t sA[2] = {(cuuint64_t)ldk * 2, (cuuint64_t)p.rows * ldk * 2};
  const cuuint32_t bA[3] = {S1_RB / 2, BM, 1};
  const cuuint64_t dB[3] = {(cuuint64_t)K, (cuuint64_t)R, (cuuint64_t)m};
  const cuuint64_t sB[2] = {(cuuint64_t)ldk * 2, (cuuint64_t)R * ldk * 2};
  const cuuint32_t bB[3] = {S1_RB / 2, (cuuint32_t)(p.gn > 1 ? p.wr : p.b_rows), (cuuint32_t)(p.gn > 1 ? p.gn / 2 : 1)};
  const CUtensorMap mAh = make_map(Lhi, dA, sA, bA, et, S1_RB), mBh = make_map(Xhi, dB, sB, bB, et, S1_RB);
  const CUtensorMap mAl = Llo ? make_map(Llo, dA, sA, bA, et, S1_RB) : mAh;
  const CUtensorMap mBl = make_map(Xlo, dB, sB, bB, et, S1_RB);
  // units of up to 16 row tiles (RES: they share the resident X rows), at least six
  // per cluster where there are that many tiles
  const int slots = std::max(1, pair_slots() / 2);
  p.mseg = std::max(1, std::min(16, (int)((long long)p.mt * p.ntile / (6 * slots))));
  p.units = p.ntile * ((p.mt + p.mseg - 1) / p.mseg);
  const int clusters = std::min(p.units, slots);
  const bool res = p.nkb <= S1_RES_KB;
  auto go = [&](auto kernel, int smem) {
    ensure_smem((const void*)kernel, smem);
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(2 * clusters), 1, 1);
    cfg.blockDim = dim3(S1_THREADS);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    TD_CUDA(cudaLaunchKernelEx(&cfg, kernel, mAh, mAl, mBh, mBl, p));
  };
  if (res) {
    if (out_is8) go(k_stage1_pair<false, true, ET_BF16, ET_E4M3>, S1Cfg<false, true>::SMEM_BYTES);
    else if (et == ET_F16) go(k_stage1_pair<true, true, ET_F16, ET_F16>, S1Cfg<true, true>::SMEM_BYTES);
    else go(k_stage1_pair<false, true, ET_BF16, ET_BF16>, S1Cfg<false, true>::SMEM_BYTES);
  } else {
    if (out_is8) go(k_stage1_pair<false, false, ET_BF16, ET_E4M3>, S1Cfg<false, false>::SMEM_BYTES);
    else if (et == ET_F16) go(k_stage1_pair<true, false, ET_F16, ET_F16>, S1Cfg<true, false>::SMEM_BYTES);
    else go(k_stage1_pair<false, false, ET_BF16, ET_BF16>, S1Cfg<false, false>::SMEM_BYTES);
  }
  count_launch();
  TD_LAUNCH_CHECK();
}
}  // namespace

void tc_stage1(const void* Xhi, const void* Xlo, int m, int R, int K, const void* Lhi, const void* Llo, int no, int pn,
               TcElt et, const float* mul, void* out_hi, void* out_lo, int* err, cudaStream_t s) {
  stage1_impl(Xhi, Xlo, m, R, K, Lhi, Llo, no, pn, elem_of(et), false, out_hi, out_lo, mul, nullptr, err, s);
}

void tc_stage1_fp8(const __nv_bfloat16* Xhi, const __nv_bfloat16* Xlo, int m, int R, int K, const __nv_bfloat16* L,
                   int no, int pn, const float* mu, unsigned char* out_hi, unsigned char* out_lo, int* err,
                   cudaStream_t s) {
  stage1_impl(Xhi, Xlo, m, R, K, L, nullptr, no, pn, ET_BF16, true, out_hi, out_lo, nullptr, mu, err, s);
}

// F64/F32/BF16 rows [rows][n] -> hi (+ lo) [rows][tc_pad(n)] (times *scale when given)
template <typename TS, typename E>
__global__ void k_pad_split(const TS* __restrict__ src, long long rows, int n, int ld,
                            const float* __restrict__ scale, E* hi, E* lo) {
  const long long tot = rows * ld;
  const float sc = scale ? *scale : 1.f;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < tot;
       t += (long long)gridDim.x * blockDim.x) {
    const int a = (int)(t % ld);
    const long long r = t / ld;
    const float v = a < n ? (float)src[r * n + a] * sc : 0.f;
    split_store<E>(v, t, hi, lo);
  }
}

template <typename E>
void pad_split_t(const void* src, DType ts, long long rows, int n, int ld, const float* scale, E* hi, E* lo,
                 cudaStream_t s) {
  const long long tot = rows * ld;
  long long g = (tot + 255) / 256;
  if (g > 152 * 16) g = 152 * 16;
  if (ts == DType::F64)
    k_pad_split<double, E><<<(unsigned)g, 256, 0, s>>>((const double*)src, rows, n, ld, scale, hi, lo);
  else if (ts == DType::F32)
    k_pad_split<float, E><<<(unsigned)g, 256, 0, s>>>((const float*)src, rows, n, ld, scale, hi, lo);
  else
    k_pad_split<__nv_bfloat16, E><<<(unsigned)g, 256, 0, s>>>((const __nv_bfloat16*)src, rows, n, ld, scale, hi, lo);
}

void tc_pad_split(const void* src, DType ts, long long rows, int n, void* hi, void* lo, TcElt et,
                  const float* scale, cudaStream_t s) {
  TD_REQUIRE(et == TcElt::F16 || scale == nullptr, TDDFT_ERR_ARG, "tc_pad_split: BF16 parts take no scale");
  if (et == TcElt::F16)
    pad_split_t<__half>(src, ts, rows, n, tc_pad(n), scale, (__half*)hi, (__half*)lo, s);
  else
    pad_split_t<__nv_bfloat16>(src, ts, rows, n, tc_pad(n), scale, (__nv_bfloat16*)hi, (__nv_bfloat16*)lo, s);
  count_launch();
  TD_LAUNCH_CHECK();
}


// ---------------------------------------------------------------------------
// FP8 (e4m3) operands of the ris exchange contractions, with a scale per
// auxiliary row P.  The ris factors L^P are stored as q^P = e4m3(L^P / s_P),
// s_P = max |L^P| / 448 (448 = the largest finite e4m3).  A product
// sum_P C_P L^P = sum_P (s_P C_P) q^P: the stage-1 result C_P is multiplied by
// mu_P = s_P * g before its own hi + lo e4m3 split, and the contraction's sum
// by 1/g, with g chosen from a bound so that |mu_P C_P| <= 224:
//   |C_P[(n,i)][k]| <= rho_P * kappa   (Cauchy-Schwarz), rho_P = max_i ||L^P_i,:||,
//   kappa = the largest norm of the trial-vector slices that C contracts with.
namespace {

__global__ void k_quant_e4m3_t(const __nv_bfloat16* __restrict__ src, int n1, int n2, int ld,
                               unsigned char* __restrict__ dst, float* __restrict__ scale) {
  const long long per = (long long)n1 * n2;
  const __nv_bfloat16* x = src + blockIdx.x * per;
  unsigned char* y = dst + (long long)blockIdx.x * n2 * ld;
  __shared__ float red[32];
  float m = 0.f;
  for (long long t = threadIdx.x; t < per; t += blockDim.x) m = fmaxf(m, fabsf(__bfloat162float(x[t])));
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x < 32) {
    m = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) red[0] = m;
  }
  __syncthreads();
  const float sc = red[0] > 0.f ? red[0] / 448.f : 1.f;
  const float inv = 1.f / sc;
  if (threadIdx.x == 0) scale[blockIdx.x] = sc;
  const long long tot = (long long)n2 * ld;
  for (long long t = threadIdx.x; t < tot; t += blockDim.x) {   // y[b][a] = x[a][b] / s
    const int a = (int)(t % ld);
    const long long b = t / ld;
    y[t] = a < n1 ? to_e4m3(__bfloat162float(x[(long long)a * n2 + b]) * inv) : (unsigned char)0;
  }
}

__global__ void k_row_norm_max(const __nv_bfloat16* __restrict__ src, int nr, int nc, float* __restrict__ rho) {
  const __nv_bfloat16* x = src + (long long)blockIdx.x * nr * nc;
  __shared__ float red[32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  float m = 0.f;
  for (int i = warp; i < nr; i += nw) {
    float acc = 0.f;
    for (int c = lane; c < nc; c += 32) {
      const float v = __bfloat162float(x[(long long)i * nc + c]);
      acc += v * v;
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    m = fmaxf(m, sqrtf(acc));
  }
  if (lane == 0) red[warp] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float r = 0.f;
    for (int w = 0; w < nw; ++w) r = fmaxf(r, red[w]);
    rho[blockIdx.x] = r;
  }
}

// 2^(top - e) for b = f 2^e, f in [0.5, 1): the largest power of two s with
// s b < 2^top (1 for b = 0).
__device__ __forceinline__ float pow2_scale(float b, int top) {
  if (!(b > 0.f)) return 1.f;
  int e = 0;
  frexpf(b, &e);
  e = max(-100, min(100, e));
  return ldexpf(1.f, top - e);
}

// st[0] = max |x| and st[1] = the largest row norm of FP32 rows [rows][n]
// (float bits); one warp per row
__global__ void k_f16_tensor_stats(const float* __restrict__ src, long long rows, int n, unsigned* __restrict__ st) {
  const int lane = threadIdx.x & 31;
  const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  float ma = 0.f, mr = 0.f;
  for (long long r = w0; r < rows; r += nw) {
    float acc = 0.f;
    for (int c = lane; c < n; c += 32) {
      const float v = src[r * n + c];
      acc += v * v;
      ma = fmaxf(ma, fabsf(v));
    }
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    mr = fmaxf(mr, sqrtf(acc));
  }
  for (int o = 16; o > 0; o >>= 1) ma = fmaxf(ma, __shfl_xor_sync(0xffffffffu, ma, o));
  if (lane == 0) {
    atomicMax(&st[0], __float_as_uint(ma));
    atomicMax(&st[1], __float_as_uint(mr));
  }
}

// sc[0] = sigma (max |sigma x| < 2^14), sc[1] = sigma * largest row norm
__global__ void k_f16_sigma(const unsigned* __restrict__ st, float* __restrict__ sc) {
  const float sg = pow2_scale(__uint_as_float(st[0]), 14);
  sc[0] = sg;
  sc[1] = sg * __uint_as_float(st[1]);
}

// Bounds of the trial vectors and the scales that follow from them, in one launch:
//   kappa[0] = max_(n,a) ||X[n][:][a]||, kappa[1] = max_(n,j) ||X[n][j][:]||,
//   kappa[2] = max |X|  (float bits: non-negative floats order like them),
// by blocks of 32 rows (which also write the FP32 copy Xw) and of 256 columns; the
// last block to finish turns them into the scales and leaves the scratch words
// ready for the next call.  Bound by launch latency up to a few MB of X, then by
// reading X twice (the second time from L2).  20 vectors of 150 x 1350: 31 us
// (171 us with one block per vector and the scales in a second launch).
struct XPrep {
  int m, no, nv, rb, cb;       // row and column blocks per vector
  unsigned* scratch;           // [0..2] kappa, [3] finished blocks, [4] max |t| (tc_t_split): zero on entry
  float* xw;                   // FP32 copy or NULL
  float* out;
  const float* fsc;            // FP16: factor-set scale block
  const float *s1, *r1, *s2, *r2;   // FP8: scales and row norms of the rows
  int nK;
};

__device__ __forceinline__ float block_max(float v, float* red) {   // 256 threads; every thread gets it
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  v = red[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) v = fmaxf(v, red[w]);
  return v;
}

template <typename T, bool FP8>
__global__ void __launch_bounds__(256) k_x_prep(const T* __restrict__ X, const XPrep p) {
  __shared__ float red[8];
  __shared__ bool last;
  const int n = blockIdx.x / (p.rb + p.cb), q = blockIdx.x - n * (p.rb + p.cb);
  const T* x = X + (long long)n * p.no * p.nv;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q < p.rb) {
    float mr = 0.f, ma = 0.f;
    for (int j = q * 32 + warp; j < min(p.no, q * 32 + 32); j += 8) {
      float acc = 0.f;
#pragma unroll 4
      for (int b = lane; b < p.nv; b += 32) {
        const float v = (float)x[(long long)j * p.nv + b];
        acc += v * v;
        ma = fmaxf(ma, fabsf(v));
        if (p.xw) p.xw[((long long)n * p.no + j) * p.nv + b] = v;
      }
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      mr = fmaxf(mr, sqrtf(acc));
    }
    mr = block_max(mr, red);
    ma = block_max(ma, red);
    if (threadIdx.x == 0) {
      atomicMax(&p.scratch[1], __float_as_uint(mr));
      atomicMax(&p.scratch[2], __float_as_uint(ma));
    }
  } else {
    const int a = (q - p.rb) * 256 + threadIdx.x;
    float acc = 0.f;
    if (a < p.nv) {
#pragma unroll 4
      for (int j = 0; j < p.no; ++j) {
        const float v = (float)x[(long long)j * p.nv + a];
        acc += v * v;
      }
    }
    const float mc = block_max(sqrtf(acc), red);
    if (threadIdx.x == 0) atomicMax(&p.scratch[0], __float_as_uint(mc));
  }
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(&p.scratch[3], 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  const float kc = __uint_as_float(__ldcg(&p.scratch[0])), kr = __uint_as_float(__ldcg(&p.scratch[1]));
  const float kx = __uint_as_float(__ldcg(&p.scratch[2]));
  if constexpr (!FP8) {
    if (threadIdx.x == 0) {   // layout in tc_gemm.cuh
      const float* fsc = p.fsc;
      const float sx = pow2_scale(kx, 14);
      // |Z'| <= rho_oo' ||X'[n][:][a]||, |Q'| <= ||X'[n][i][:]|| rho_ov' (Cauchy-Schwarz)
      const float mz = pow2_scale(fsc[1] * sx * kc, 15);
      const float mq = pow2_scale(fsc[5] * sx * kr, 15);
      p.out[0] = sx;
      p.out[1] = mz;
      p.out[2] = mq;
      p.out[3] = 1.f / (mz * fsc[0] * sx * fsc[2]);
      p.out[4] = 1.f / (mq * sx * fsc[4] * fsc[4]);
    }
  } else {
    // out[0] = 1/g1, out[1] = 1/g2, out[2 + P] = s1_P g1, out[2 + nK + P] = s2_P g2
    float b1 = 0.f, b2 = 0.f;
    for (int P = threadIdx.x; P < p.nK; P += 256) {
      b1 = fmaxf(b1, p.s1[P] * p.r1[P] * kc);
      b2 = fmaxf(b2, p.s2[P] * p.r2[P] * kr);
    }
    b1 = block_max(b1, red);
    b2 = block_max(b2, red);
    const float g1 = b1 > 0.f ? 224.f / b1 : 1.f, g2 = b2 > 0.f ? 224.f / b2 : 1.f;
    if (threadIdx.x == 0) {
      p.out[0] = 1.f / g1;
      p.out[1] = 1.f / g2;
    }
    for (int P = threadIdx.x; P < p.nK; P += 256) {
      p.out[2 + P] = p.s1[P] * g1;
      p.out[2 + p.nK + P] = p.s2[P] * g2;
    }
  }
  __syncthreads();
  if (threadIdx.x < 5) p.scratch[threadIdx.x] = 0u;
}

// Both operand forms of the trial vectors from one read: X^T per vector
// ([n][a][pad8(j)]) and, when sh is given, X ([n][j][pad8(b)]), as hi + lo parts of
// X times *scale; the FP32 copy xw when given.
template <typename T, typename E>
__global__ void __launch_bounds__(256) k_x_split(const T* __restrict__ X, int m, int no, int nv, int nop, int nvp,
                                                 const float* __restrict__ scale, E* th, E* tl, E* sh, E* sl,
                                                 float* xw) {
  __shared__ float tile[32][33];
  const int a0 = blockIdx.x * 32, j0 = blockIdx.y * 32;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const float sc = scale ? *scale : 1.f;
  for (int n = blockIdx.z; n < m; n += gridDim.z) {
#pragma unroll
    for (int r = ty; r < 32; r += 8) {
      const int j = j0 + r, a = a0 + tx;
      float v = 0.f;
      if (j < no && a < nv) {
        v = (float)X[((long long)n * no + j) * nv + a];
        if (xw) xw[((long long)n * no + j) * nv + a] = v;
      }
      v *= sc;
      tile[r][tx] = v;
      if (sh && j < no && a < nvp) split_store<E>(v, ((long long)n * no + j) * nvp + a, sh, sl);
    }
    __syncthreads();
#pragma unroll
    for (int r = ty; r < 32; r += 8) {
      const int a = a0 + r, j = j0 + tx;
      if (a < nv && j < nop) split_store<E>(tile[tx][r], ((long long)n * nv + a) * nop + j, th, tl);
    }
    __syncthreads();
  }
}

// t [K][m] -> FP16 hi + lo of s_t t^T [m][ldk], s_t the power of two with
// max |s_t t| < 2^14 (tmax: float bits of max |t|); fac = 1 / (s_t s_ov).
__global__ void __launch_bounds__(256) k_t_split(const float* __restrict__ t, int K, int m, int ldk,
                                                 const unsigned* __restrict__ tmax, const float* __restrict__ s_ov,
                                                 __half* hi, __half* lo, float* fac) {
  const float st = pow2_scale(__uint_as_float(*tmax), 14);
  if (blockIdx.x == 0 && threadIdx.x == 0) *fac = 1.f / (st * *s_ov);
  const long long tot = (long long)m * ldk;
  for (long long e = blockIdx.x * 256ll + threadIdx.x; e < tot; e += (long long)gridDim.x * 256) {
    const int n = (int)(e / ldk), k = (int)(e - (long long)n * ldk);
    split_store<__half>(k < K ? t[(long long)k * m + n] * st : 0.f, e, hi, lo);
  }
}

}  // namespace

void tc_quant_e4m3(const __nv_bfloat16* src, int rows, int n1, int n2, unsigned char* dst, float* scale,
                   cudaStream_t s) {
  if (rows <= 0) return;
  k_quant_e4m3_t<<<rows, 512, 0, s>>>(src, n1, n2, tc_pad16(n1), dst, scale);
  count_launch();
  TD_LAUNCH_CHECK();
}

void tc_row_norm_max(const __nv_bfloat16* src, int rows, int nr, int nc, float* rho, cudaStream_t s) {
  if (rows <= 0) return;
  k_row_norm_max<<<rows, 256, 0, s>>>(src, nr, nc, rho);
  count_launch();
  TD_LAUNCH_CHECK();
}

namespace {
template <bool FP8>
void x_prep(const void* X, DType xt, XPrep p, cudaStream_t s) {
  p.rb = (p.no + 31) / 32;
  p.cb = (p.nv + 255) / 256;
  TD_REQUIRE((long long)p.m * (p.rb + p.cb) < (1ll << 31), TDDFT_ERR_ARG, "trial vectors: too many");
  const unsigned grid = (unsigned)(p.m * (p.rb + p.cb));
  if (xt == DType::F32) k_x_prep<float, FP8><<<grid, 256, 0, s>>>(static_cast<const float*>(X), p);
  else k_x_prep<double, FP8><<<grid, 256, 0, s>>>(static_cast<const double*>(X), p);
  count_launch();
  TD_LAUNCH_CHECK();
}
}  // namespace

void tc_fp8_scales(const void* X, DType xt, int m, int no, int nv, const float* s_vv, const float* rho_oo,
                   const float* s_vo, const float* rho_ov, int nK, float* out, unsigned* scratch, float* xw,
                   cudaStream_t s) {
  x_prep<true>(X, xt, XPrep{m, no, nv, 0, 0, scratch, xw, out, nullptr, s_vv, rho_oo, s_vo, rho_ov, nK}, s);
}

void tc_x_split(const void* X, DType xt, int m, int no, int nv, TcElt et, const float* scale, void* th, void* tl,
                void* sh, void* sl, float* xw, cudaStream_t s) {
  const int nop = tc_pad(no), nvp = tc_pad(nv);
  TD_REQUIRE((nop + 31) / 32 <= 65535, TDDFT_ERR_ARG, "tc_x_split: n_occ");
  const dim3 grid((nvp + 31) / 32, (nop + 31) / 32, std::min(m, 65535));
  auto go = [&](auto* x, auto* e) {
    using E = std::remove_pointer_t<decltype(e)>;
    k_x_split<<<grid, 256, 0, s>>>(x, m, no, nv, nop, nvp, scale, static_cast<E*>(th), static_cast<E*>(tl),
                                   static_cast<E*>(sh), static_cast<E*>(sl), xw);
  };
  const bool f32 = xt == DType::F32;
  if (et == TcElt::F16) {
    if (f32) go(static_cast<const float*>(X), (__half*)nullptr);
    else go(static_cast<const double*>(X), (__half*)nullptr);
  } else {
    if (f32) go(static_cast<const float*>(X), (__nv_bfloat16*)nullptr);
    else go(static_cast<const double*>(X), (__nv_bfloat16*)nullptr);
  }
  count_launch();
  TD_LAUNCH_CHECK();
}

void tc_t_split(const float* t, int K, int m, const unsigned* tmax, const float* s_ov, void* hi, void* lo, float* fac,
                cudaStream_t s) {
  const int ldk = tc_pad(K);
  const long long g = std::min<long long>(((long long)m * ldk + 255) / 256, 152 * 8);
  k_t_split<<<(unsigned)g, 256, 0, s>>>(t, K, m, ldk, tmax, s_ov, static_cast<__half*>(hi), static_cast<__half*>(lo),
                                        fac);
  count_launch();
  TD_LAUNCH_CHECK();
}

void tc_f16_tensor_scale(const float* src, long long rows, int n, float* sc, unsigned* scratch, cudaStream_t s) {
  TD_CUDA(cudaMemsetAsync(scratch, 0, 2 * sizeof(unsigned), s));
  if (rows > 0 && n > 0) {
    long long g = (rows * 32 + 255) / 256;
    if (g > 152 * 16) g = 152 * 16;
    k_f16_tensor_stats<<<(unsigned)g, 256, 0, s>>>(src, rows, n, scratch);
    count_launch();
    TD_LAUNCH_CHECK();
  }
  k_f16_sigma<<<1, 1, 0, s>>>(scratch, sc);
  count_launch();
  TD_LAUNCH_CHECK();
}

void tc_f16_product_scales(const void* X, DType xt, int m, int no, int nv, const float* fsc, float* out,
                           unsigned* scratch, float* xw, cudaStream_t s) {
  x_prep<false>(X, xt, XPrep{m, no, nv, 0, 0, scratch, xw, out, fsc, nullptr, nullptr, nullptr, nullptr, 0}, s);
}

}  // namespace tddft
