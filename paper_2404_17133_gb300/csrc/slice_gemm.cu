// FP64 and FP32 contractions on the FP16 tensor cores by exact slicing (the
// splitting of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012, with
// base-256 digits as the slices).
//
// Every row of an operand is scaled by a power of two, 2^-e, so that all its
// elements lie in (-1/2, 1/2), and written as S balanced base-256 digits,
//   x 2^-e = sum_s d_s 2^(-8 (s+1)),  -128 <= d_s <= 127,
// S = 7 for FP64 (56 bits), S = 4 for FP32 (32 bits).  Digits are FP16
// integers, so a product of two is exact, and the sum of the products of one
// level l = i + j over a run of K = 256 elements is at most
// (l + 1) 256 2^14 <= 2^24 for l <= 3: exact in the FP32 accumulator of the
// tensor core.  (Deeper levels may round at 2^-24 of a sum that already weighs
// 2^-32.)  Levels l < S are kept, each in its own TMEM columns; after each run
// the epilogue warps move them to 64-bit integers (FP64) or a compensated FP32
// pair (FP32), so nothing but the digits below the last slice is ever rounded
// before the final scaling.  The error of a product is 2^-56 (2^-32) of
// max|A row| max|B row| per term, below what FP64 (FP32) accumulation leaves.
//
// Why: FP64 runs at 1.2 TFLOP/s on this GPU's vector units and FP32 at 75; S (S
// + 1) / 2 FP16 products per term (28 or 10) leave up to 69 and 190 TFLOP/s.
//
// CTA = 128 x NT output tile (NT = 64 or 128: S levels of NT FP32 columns fill
// the tensor memory), persistent over (tile, K split) items; warp 0 issues TMA
// loads of all slices of a 32-element k-block (64-byte rows, SWIZZLE_64B), warp
// 1 one tcgen05.mma per slice pair, warps 2-9 the run epilogue.  A slice of A
// stays in the tensor core's operand collector while it meets all slices of B.
//
// Every wait on an mbarrier is bounded as in tc_gemm.cu.
#include <algorithm>
#include <cstring>
#include <type_traits>
#include <cuda.h>
#include <cuda_fp16.h>

#include "slice_gemm.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace tddft {

namespace {

constexpr int SBM = 128;          // output rows per tile
constexpr int SBK = 32;           // K elements per k-block (64-byte rows)
constexpr int RUN = 8;            // k-blocks per exact accumulation run
constexpr int EPI_WARPS = 8;
constexpr int SL_THREADS = 64 + 32 * EPI_WARPS;

template <int S> struct SCfg {
  static constexpr int NT = S == 7 ? 64 : 128;
  // levels i + j kept: FP64 needs one beyond the slices (the six products of level 7
  // are 2^-58 of max max, 1e-15 of a result whose rows decay; without them the error
  // was 1.3e-15 against 1.2e-15 of FP64 arithmetic, with them 3.5e-16; 34 products
  // instead of 28)
  static constexpr int LV = S == 7 ? 8 : 4;
  static constexpr int A_SLICE = SBM * SBK * 2, B_SLICE = NT * SBK * 2;
  static constexpr int STAGE_BYTES = S * (A_SLICE + B_SLICE);
  static constexpr int STAGES = S == 7 ? 2 : 3;
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
  static constexpr int TMEM_COLS = 512;
};

struct SParams {
  int M, N;             // output rows / columns
  int Kin, nab;         // k extent per P, k-blocks per P
  int total, per;       // k-blocks in all, per split (a multiple of RUN)
  int tiles_n, tiles, items;
  const int* ea;        // exponent words of the rows of A and of B
  const int* eb;
  void* out;
  int scatter;          // 0: out[z][M][N] partials, 1: the strides below
  int R, C;
  long long rs1, cs0, cs1;
  int* err;
};

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0, int c1, int c2,
                                            int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3)
      : "memory");
}

// K-major descriptor of a tile of 64-byte rows (64-byte swizzle, 8-row groups 512 B apart).
__device__ __forceinline__ uint64_t sdesc64(const void* p) {
  const uint64_t addr = smem_u32(p);
  return ((addr & 0x3FFFFull) >> 4) | (1ull << 16) | ((uint64_t)(512 >> 4) << 32) | (1ull << 46) | (4ull << 61);
}

// Use of the A operand collector: the products of one A slice share its fetch.
enum Collect { C_FILL, C_USE, C_LAST, C_NONE };
template <int CO>
__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t accum, uint32_t idesc) {
  if constexpr (CO == C_FILL)
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16.collector::a::fill [%0], %1, %2, %3, p;\n}\n" ::"r"(d), "l"(a),
                 "l"(b), "r"(idesc), "r"(accum));
  else if constexpr (CO == C_USE)
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16.collector::a::use [%0], %1, %2, %3, p;\n}\n" ::"r"(d), "l"(a),
                 "l"(b), "r"(idesc), "r"(accum));
  else if constexpr (CO == C_LAST)
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16.collector::a::lastuse [%0], %1, %2, %3, p;\n}\n" ::"r"(d), "l"(a),
                 "l"(b), "r"(idesc), "r"(accum));
  else
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d), "l"(a), "l"(b), "r"(idesc),
                 "r"(accum));
}

__device__ __forceinline__ void tmem_ld4(float (&v)[4], uint32_t taddr) {
  uint32_t r0, r1, r2, r3;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
               : "r"(taddr));
  v[0] = __uint_as_float(r0);
  v[1] = __uint_as_float(r1);
  v[2] = __uint_as_float(r2);
  v[3] = __uint_as_float(r3);
}

// Running sum of one output over the exact runs.  v[l]: the run's level sums.
template <int S> struct Acc;
template <> struct Acc<7> {
  long long hi, lo;   // units 2^-40 (levels 0-3) and 2^-72 (levels 4-7) of the scaled product
  __device__ __forceinline__ void clear() { hi = 0; lo = 0; }
  __device__ __forceinline__ void add(const float* v) {
    hi += (long long)__float2int_rn(v[0]) * 16777216 + (long long)__float2int_rn(v[1]) * 65536 +
          (long long)__float2int_rn(v[2]) * 256 + __float2int_rn(v[3]);
    lo += (long long)__float2int_rn(v[4]) * 16777216 + (long long)__float2int_rn(v[5]) * 65536 +
          (long long)__float2int_rn(v[6]) * 256 + __float2int_rn(v[7]);
  }
  // times 2^40 (each row's scale carries 2^-20)
  __device__ __forceinline__ double value() const { return fma((double)lo, 0x1p-32, (double)hi); }
};
template <> struct Acc<4> {
  float hi, lo;       // compensated sum in units 2^-16 (level 0)
  __device__ __forceinline__ void clear() { hi = 0.f; lo = 0.f; }
  __device__ __forceinline__ void add(const float* v) {
    const float x = fmaf(fmaf(fmaf(v[3], 0x1p-8f, v[2]), 0x1p-8f, v[1]), 0x1p-8f, v[0]);
    const float s = hi + x, bb = s - hi;
    lo += (hi - (s - bb)) + (x - bb);
    hi = s;
  }
  __device__ __forceinline__ float value() const { return hi + lo; }
};

// Power-of-two scale of a row from its exponent word (the largest biased
// exponent field, or the all-ones field where the row holds a non-finite value).
template <int S> __device__ __forceinline__ auto row_scale(int w);
template <> __device__ __forceinline__ auto row_scale<7>(int w) {
  const int E = max(w, 1);
  if (E >= 2047) return __longlong_as_double(0x7ff8000000000000ll);
  return E > 18 ? __longlong_as_double((long long)(E - 18) << 52) : ldexp(1.0, E - 1041);
}
template <> __device__ __forceinline__ auto row_scale<4>(int w) {
  const int E = max(w, 1);
  if (E >= 255) return __int_as_float(0x7fc00000);
  return E > 6 ? __int_as_float((E - 6) << 23) : ldexpf(1.f, E - 133);
}

template <int S>
__global__ void __launch_bounds__(SL_THREADS, 1)
k_slice_mma(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB, const SParams p) {
  using C = SCfg<S>;
  using T = typename std::conditional<S == 7, double, float>::type;
  constexpr int NT = C::NT;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::STAGES * C::STAGE_BYTES);
  uint64_t* empty = full + C::STAGES;
  uint64_t* tfull = empty + C::STAGES;    // the run's levels are complete
  uint64_t* tempty = tfull + 1;           // ... and have been read
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(tfull, 1);
    mbar_init(tempty, EPI_WARPS);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(C::TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  // k-blocks of one item
  auto range = [&](int item, int& k0, int& nk) {
    k0 = (item / p.tiles) * p.per;
    nk = min(p.total - k0, p.per);
  };

  if (warp == 0 && lane == 0) {
    long long i = 0;   // k-blocks loaded so far
    bool ok = true;
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x) {
      int k0, nk;
      range(item, k0, nk);
      const int t = item % p.tiles;
      const int m0 = (t / p.tiles_n) * SBM, n0 = (t % p.tiles_n) * NT;
      for (int kb = k0; kb < k0 + nk; ++kb, ++i) {
        const int s = (int)(i % C::STAGES);
        if (!mbar_wait(&empty[s], ((uint32_t)(i / C::STAGES) & 1u) ^ 1u)) { atomicOr(p.err, 512); ok = false; break; }
        const int P = kb / p.nab, a0 = (kb - P * p.nab) * SBK;
        unsigned char* st = smem + s * C::STAGE_BYTES;
        mbar_expect_tx(&full[s], C::STAGE_BYTES);
        tma_load_4d(st, &mA, &full[s], a0, P, m0, 0);
        tma_load_4d(st + S * C::A_SLICE, &mB, &full[s], a0, n0, P, 0);
      }
    }
    // let the copies already issued land before the CTA can exit
    for (long long j = i > C::STAGES ? i - C::STAGES : 0; j < i; ++j)
      if (!mbar_wait(&full[j % C::STAGES], (uint32_t)(j / C::STAGES) & 1u)) { atomicOr(p.err, 512); break; }
  } else if (warp == 1 && lane == 0) {
    long long i = 0, run = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x) {
      int k0, nk;
      range(item, k0, nk);
      const int n0 = ((item % p.tiles) % p.tiles_n) * NT;
      const int nb = min(NT, (p.N - n0 + 15) & ~15);
      // kind::f16 with FP16 operands, FP32 accumulator, both K-major, M = 128, N = nb
      const uint32_t idesc = (1u << 4) | ((uint32_t)(nb >> 3) << 17) | ((uint32_t)(SBM >> 4) << 24);
      for (int kb = k0; kb < k0 + nk && ok; kb += RUN, ++run) {
        if (!mbar_wait(tempty, ((uint32_t)run & 1u) ^ 1u)) { atomicOr(p.err, 1024); ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int kn = min(RUN, k0 + nk - kb);
        for (int b = 0; b < kn; ++b, ++i) {
          const int s = (int)(i % C::STAGES);
          if (!mbar_wait(&full[s], (uint32_t)(i / C::STAGES) & 1u)) { atomicOr(p.err, 1024); ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          unsigned char* st = smem + s * C::STAGE_BYTES;
          const uint64_t da = sdesc64(st), db = sdesc64(st + S * C::A_SLICE);
          const int rem = p.Kin - ((kb + b) % p.nab) * SBK;
          const int nks = rem > 16 ? 2 : 1;   // 16-element K steps holding data
          for (int kk = 0; kk < nks; ++kk) {
            // a level of a run is opened by slice 0 of A, one past the slices by the last slice of B
            const uint32_t acc = (b > 0 || kk > 0) ? 1u : 0u;
#pragma unroll
            for (int ia = 0; ia < S; ++ia) {
              const uint64_t a = da + ((ia * C::A_SLICE + kk * 32) >> 4);
              const int nbs = S < C::LV - ia ? S : C::LV - ia;   // slices of B that ia meets
#pragma unroll
              for (int ib = 0; ib < nbs; ++ib) {
                const uint64_t bd = db + ((ib * C::B_SLICE + kk * 32) >> 4);
                const uint32_t d = tmem + (uint32_t)((ia + ib) * NT);
                const uint32_t ac = ia == 0 || ib == S - 1 ? acc : 1u;
                if (nbs == 1) mma_f16<C_NONE>(d, a, bd, ac, idesc);
                else if (ib == 0) mma_f16<C_FILL>(d, a, bd, ac, idesc);
                else if (ib == nbs - 1) mma_f16<C_LAST>(d, a, bd, ac, idesc);
                else mma_f16<C_USE>(d, a, bd, ac, idesc);
              }
            }
          }
          mma_commit(&empty[s]);
        }
        mma_commit(tfull);
      }
    }
  } else if (warp >= 2) {
    constexpr int HC = NT / 2;               // columns per warp
    constexpr int CH = 4;                    // columns per TMEM load
    const int q = warp & 3, half = (warp - 2) >> 2;
    const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * HC);
    long long run = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x) {
      int k0, nk;
      range(item, k0, nk);
      const int t = item % p.tiles;
      const int m0 = (t / p.tiles_n) * SBM + q * 32, n0 = (t % p.tiles_n) * NT + half * HC;
      const int row = m0 + lane;
      const bool live = m0 < p.M;            // this warp has rows to read
      const int ncol = min(HC, p.N - n0);    // columns of this warp (may be <= 0)
      Acc<S> acc[HC];
#pragma unroll
      for (int c = 0; c < HC; ++c) acc[c].clear();
      for (int kb = 0; kb < nk; kb += RUN, ++run) {
        bool got = mbar_wait(tfull, (uint32_t)run & 1u);
        got = __all_sync(0xffffffffu, got);
        if (!got) { if (lane == 0) atomicOr(p.err, 2048); ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (live) {
#pragma unroll
          for (int c = 0; c < HC; c += CH) {
            if (c < ncol) {
              float v[C::LV][CH];
#pragma unroll
              for (int l = 0; l < C::LV; ++l) tmem_ld4(v[l], tb + (uint32_t)(l * NT + c));
              asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
              for (int j = 0; j < CH; ++j) {
                float w[C::LV];
#pragma unroll
                for (int l = 0; l < C::LV; ++l) w[l] = v[l][j];
                acc[c + j].add(w);
              }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(tempty)) : "memory");
      }
      if (!ok || row >= p.M) continue;
      const T sa = row_scale<S>(p.ea[row]);
      T* out = static_cast<T*>(p.out);
      if (p.scatter) {
        out += (long long)(row / p.R) * p.rs1 + row % p.R;
        int cq = n0 / p.C, cr = n0 - (n0 / p.C) * p.C;
#pragma unroll
        for (int c = 0; c < HC; ++c) {
          if (c < ncol) out[cr * p.cs0 + cq * p.cs1] = acc[c].value() * sa * row_scale<S>(p.eb[n0 + c]);
          if (++cr == p.C) { cr = 0; ++cq; }
        }
      } else {
        out += ((long long)(item / p.tiles) * p.M + row) * p.N + n0;
#pragma unroll
        for (int c = 0; c < HC; ++c)
          if (c < ncol) out[c] = acc[c].value() * sa * row_scale<S>(p.eb[n0 + c]);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM_COLS));
}

// ---------------------------------------------------------------------------
// Slicing

// exponent field of the absolute value
__device__ __forceinline__ int exp_field(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }
__device__ __forceinline__ int exp_field(float x) { return (__float_as_int(x) >> 23) & 0xff; }

// The S digits of x against the row exponent E: round(x 2^-e 2^(8 S)) plus 128 in
// every base-256 place, so that byte S - 1 - s holds d_s + 128 (nine bits for
// the first digit, which reaches +128).
__device__ __forceinline__ unsigned long long digits(double x, int E) {
  const long long bits = __double_as_longlong(x);
  const int ef = (int)((bits >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)bits & 0xfffffffffffffull;
  if (ef) m |= 1ull << 52;
  const int r = max(E, 1) - max(ef, 1) - 2;   // right shift
  m = r <= 0 ? m << -r : (r > 54 ? 0ull : (m + (1ull << (r - 1))) >> r);
  const long long sm = bits < 0 ? -(long long)m : (long long)m;
  return (unsigned long long)(sm + 0x80808080808080ll);
}
__device__ __forceinline__ unsigned long long digits(float x, int E) {
  const int bits = __float_as_int(x);
  const int ef = (bits >> 23) & 0xff;
  unsigned m = (unsigned)bits & 0x7fffffu;
  if (ef) m |= 1u << 23;
  const int r = max(E, 1) - max(ef, 1) - 7;
  m = r <= 0 ? m << -r : (r > 25 ? 0u : (m + (1u << (r - 1))) >> r);
  const long long sm = bits < 0 ? -(long long)m : (long long)m;
  return (unsigned long long)(sm + 0x80808080ll);
}

// digit s of two elements as a pair of FP16 integers
template <int S>
__device__ __forceinline__ uint32_t digit_pair(unsigned long long a, unsigned long long b, int s) {
  const int byte = S - 1 - s;
  uint32_t h;   // FP16 1024 + (digit + 128)
  if (s == 0) {
    h = (uint32_t)(a >> (8 * byte)) | ((uint32_t)(b >> (8 * byte)) << 16) | 0x64006400u;
  } else {
    const uint32_t wa = byte < 4 ? (uint32_t)a : (uint32_t)(a >> 32), wb = byte < 4 ? (uint32_t)b : (uint32_t)(b >> 32);
    const uint32_t k = (uint32_t)(byte & 3);
    h = (__byte_perm(wa, wb, k | (k << 4) | ((4 + k) << 8) | ((4 + k) << 12)) & 0x00ff00ffu) | 0x64006400u;
  }
  const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&h), __half2half2(__ushort_as_half(0x6480)));   // - 1152
  return *reinterpret_cast<const uint32_t*>(&v);
}

template <typename T, int S>
__device__ __forceinline__ void store_slices(const T (&x)[8], int E, __half* dst, long long slice) {
  unsigned long long d[8];
  const bool special = E >= (S == 7 ? 2047 : 255);
#pragma unroll
  for (int j = 0; j < 8; ++j) d[j] = digits(special ? T(0) : x[j], E);
#pragma unroll
  for (int s = 0; s < S; ++s) {
    uint4 w;
    w.x = digit_pair<S>(d[0], d[1], s);
    w.y = digit_pair<S>(d[2], d[3], s);
    w.z = digit_pair<S>(d[4], d[5], s);
    w.w = digit_pair<S>(d[6], d[7], s);
    *reinterpret_cast<uint4*>(dst + s * slice) = w;
  }
}

struct CutParams {
  const void* p;
  int rows, np, K, ldk, R, p_outer, vec;
  long long rs1, rs0, ps, ks;
  __half* dst;
  int* exps;
};

__device__ __forceinline__ long long cut_dst(const CutParams& c, long long r, int P) {
  return (c.p_outer ? (long long)P * c.rows + r : r * c.np + P) * c.ldk;
}

// Eight elements along k (zero beyond n); vec: 16-byte accesses are aligned.
__device__ __forceinline__ void load8(const double* p, int n, bool vec, double (&v)[8]) {
  if (vec && n >= 8) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double2 q = reinterpret_cast<const double2*>(p)[j];
      v[2 * j] = q.x; v[2 * j + 1] = q.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = j < n ? p[j] : 0.0;
  }
}
__device__ __forceinline__ void load8(const float* p, int n, bool vec, float (&v)[8]) {
  if (vec && n >= 8) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float4 q = reinterpret_cast<const float4*>(p)[j];
      v[4 * j] = q.x; v[4 * j + 1] = q.y; v[4 * j + 2] = q.z; v[4 * j + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) v[j] = j < n ? p[j] : 0.f;
  }
}

// Rows contiguous along k: TPR threads per row find the row's exponent, then cut
// it in groups of eight elements (the second read comes from L1 or L2).  Bound by
// memory: 8 (4) bytes read and 14 (8) written per element.
template <typename T, int S, int TPR>
__global__ void __launch_bounds__(256) k_slice_rows(const CutParams c) {
  __shared__ int red[8];
  const int sub = threadIdx.x % TPR;
  const long long r = blockIdx.x * (long long)(256 / TPR) + threadIdx.x / TPR;
  const bool have = r < c.rows;
  const T* x = static_cast<const T*>(c.p) + (have ? (r / c.R) * c.rs1 + (r % c.R) * c.rs0 : 0);
  const int n8 = c.ldk >> 3;
  const int ng = have ? c.np * n8 : 0;
  int E = 0;
#pragma unroll 2
  for (int g = sub; g < ng; g += TPR) {
    const int P = g / n8, k0 = (g - P * n8) * 8;
    T v[8];
    load8(x + P * c.ps + k0, c.K - k0, c.vec, v);
#pragma unroll
    for (int j = 0; j < 8; ++j) E = max(E, exp_field(v[j]));
  }
#pragma unroll
  for (int o = (TPR < 32 ? TPR : 32) / 2; o > 0; o >>= 1) E = max(E, __shfl_xor_sync(0xffffffffu, E, o));
  if (TPR > 32) {
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = E;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; ++w) E = max(E, red[w]);
  }
  if (have && sub == 0) c.exps[r] = E;
  const long long slice = (long long)c.rows * c.np * c.ldk;
  for (int g = sub; g < ng; g += TPR) {
    const int P = g / n8, k0 = (g - P * n8) * 8;
    T v[8];
    load8(x + P * c.ps + k0, c.K - k0, c.vec, v);
    store_slices<T, S>(v, E, c.dst + cut_dst(c, r, P) + k0, slice);
  }
}

// Rows contiguous across r (transposed operands).  Exponents: one CTA per 32
// rows and group of P, warps over k; exps must be zero on entry.
template <typename T>
__global__ void __launch_bounds__(256) k_slice_exp_t(const CutParams c) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long r = blockIdx.x * 32ll + lane;
  if (r >= c.rows) return;
  const T* x = static_cast<const T*>(c.p) + (r / c.R) * c.rs1 + (r % c.R);
  int E = 0;
  for (int P = blockIdx.y; P < c.np; P += gridDim.y)
#pragma unroll 4
    for (int k = w; k < c.K; k += 8) E = max(E, exp_field(x[P * c.ps + k * c.ks]));
  atomicMax(&c.exps[r], E);
}

// 32 rows x 64 k tiles through shared memory: coalesced reads across rows, 128
// contiguous bytes written per row and slice.
template <typename T, int S>
__global__ void __launch_bounds__(256) k_slice_cut_t(const CutParams c) {
  __shared__ T tile[64][33];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long r0 = blockIdx.x * 32ll;
  const long long slice = (long long)c.rows * c.np * c.ldk;
  const long long rl = r0 + lane;
  const T* x = static_cast<const T*>(c.p) + (rl < c.rows ? (rl / c.R) * c.rs1 + (rl % c.R) : 0);
  const int rr = w * 4 + (lane >> 3), kg = (lane & 7) * 8;   // the row and 8-element group this thread cuts
  const int E = r0 + rr < c.rows ? c.exps[r0 + rr] : 0;
  for (int P = blockIdx.y; P < c.np; P += gridDim.y)
    for (int k0 = 0; k0 < c.K; k0 += 64) {
      __syncthreads();
#pragma unroll
      for (int k = w; k < 64; k += 8)
        tile[k][lane] = (rl < c.rows && k0 + k < c.K) ? x[P * c.ps + (k0 + k) * c.ks] : T(0);
      __syncthreads();
      if (r0 + rr < c.rows && k0 + kg < c.ldk) {
        T v[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = tile[kg + j][rr];
        store_slices<T, S>(v, E, c.dst + cut_dst(c, r0 + rr, P) + k0 + kg, slice);
      }
    }
}

// Sum of the K-split partials in a fixed order (FP64), C = sum + beta C.
template <typename T>
__global__ void k_slice_sum(const T* __restrict__ part, int S, long long MN, T* C, double beta) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < MN; t += (long long)gridDim.x * blockDim.x) {
    double v = 0.0;
    for (int s = 0; s < S; ++s) v += (double)part[s * MN + t];
    if (beta != 0.0) v += beta * (double)C[t];
    C[t] = (T)v;
  }
}

CUtensorMap slice_map(const SliceOperand& o, const void* parts, int box_rows) {
  const int S = slice_count(o.t);
  const long long ldk = tc_pad(o.K);
  // (k, P, row, slice) or, p_outer, (k, row, P, slice)
  const uint64_t n1 = o.p_outer ? o.rows : o.np, n2 = o.p_outer ? o.np : o.rows;
  const uint64_t dims[4] = {(uint64_t)o.K, n1, n2, (uint64_t)S};
  const uint64_t strides[3] = {(uint64_t)ldk * 2, (uint64_t)ldk * 2 * n1, (uint64_t)ldk * 2 * n1 * n2};
  const uint32_t box[4] = {SBK, o.p_outer ? (uint32_t)box_rows : 1u, o.p_outer ? 1u : (uint32_t)box_rows, (uint32_t)S};
  return tc_map_f16_4d(parts, dims, strides, box, 64);
}

template <int S>
void launch_mma(const SliceOperand& A, const void* Ap, const SliceOperand& B, const void* Bp, SParams p, int splits,
                cudaStream_t s) {
  using C = SCfg<S>;
  const CUtensorMap ma = slice_map(A, Ap, SBM), mb = slice_map(B, Bp, C::NT);
  p.items = p.tiles * splits;
  ensure_smem((const void*)k_slice_mma<S>, C::SMEM_BYTES);
  k_slice_mma<S><<<std::min(p.items, sm_count()), SL_THREADS, C::SMEM_BYTES, s>>>(ma, mb, p);
  count_launch();
  TD_LAUNCH_CHECK();
}

template <int S>
SParams make_params(const SliceOperand& A, const int* Ae, const SliceOperand& B, const int* Be, int* err) {
  SParams p;
  std::memset(&p, 0, sizeof(p));
  p.M = A.rows;
  p.N = B.rows;
  p.Kin = A.K;
  p.nab = (A.K + SBK - 1) / SBK;
  p.total = p.nab * A.np;
  p.per = p.total;
  p.tiles_n = (p.N + SCfg<S>::NT - 1) / SCfg<S>::NT;
  const long long tiles = (long long)p.tiles_n * ((p.M + SBM - 1) / SBM);
  TD_REQUIRE(tiles < (1 << 28) && (long long)p.nab * A.np < (1 << 28), TDDFT_ERR_ARG, "slice_gemm: problem too large");
  p.tiles = (int)tiles;
  p.ea = Ae;
  p.eb = Be;
  p.err = err;
  p.R = p.C = 1;
  return p;
}

void check_pair(const SliceOperand& A, const SliceOperand& B) {
  TD_REQUIRE(A.t == B.t && A.K == B.K && A.np == B.np && A.K >= 1 && A.np >= 1 && !A.p_outer && B.p_outer, TDDFT_ERR_ARG,
             "slice_gemm: operands do not match");
}

template <typename T, int S>
void cut_t(const SliceOperand& o, const CutParams& c, cudaStream_t s) {
  if (o.ks == 1) {
    // threads per row by its groups of eight elements
    const long long groups = (long long)o.np * (tc_pad(o.K) / 8);
    if (groups > 256) k_slice_rows<T, S, 256><<<o.rows, 256, 0, s>>>(c);
    else if (groups > 16) k_slice_rows<T, S, 32><<<(o.rows + 7) / 8, 256, 0, s>>>(c);
    else k_slice_rows<T, S, 8><<<(o.rows + 31) / 32, 256, 0, s>>>(c);
    count_launch();
  } else {
    TD_CUDA(cudaMemsetAsync(c.exps, 0, (size_t)o.rows * 4, s));
    const int rt = (o.rows + 31) / 32;
    const dim3 grid(rt, std::min(o.np, std::max(1, 16 * 152 / rt)));
    k_slice_exp_t<T><<<grid, 256, 0, s>>>(c);
    k_slice_cut_t<T, S><<<grid, 256, 0, s>>>(c);
    count_launch(2);
  }
  TD_LAUNCH_CHECK();
}

}  // namespace

size_t slice_bytes(const SliceOperand& o) {
  return (size_t)slice_count(o.t) * o.rows * o.np * tc_pad(o.K) * 2;
}

void slice_cut(const SliceOperand& o, void* parts, int* exps, cudaStream_t s) {
  TD_REQUIRE((o.t == DType::F64 || o.t == DType::F32) && (o.ks == 1 || o.rs0 == 1) && o.rows >= 1 && o.K >= 1,
             TDDFT_ERR_ARG, "slice_cut: unsupported operand");
  const long long es = (long long)dtype_size(o.t);
  const bool vec = o.ks == 1 && reinterpret_cast<uintptr_t>(o.p) % 16 == 0 && o.rs0 * es % 16 == 0 &&
                   o.rs1 * es % 16 == 0 && o.ps * es % 16 == 0;
  const CutParams c{o.p, o.rows, o.np, o.K, tc_pad(o.K), o.R, o.p_outer ? 1 : 0, vec ? 1 : 0, o.rs1, o.rs0, o.ps,
                    o.ks, static_cast<__half*>(parts), exps};
  TD_REQUIRE((long long)o.np * (tc_pad(o.K) / 8) < (1ll << 31), TDDFT_ERR_ARG, "slice_cut: row too long");
  if (o.t == DType::F64) cut_t<double, 7>(o, c, s);
  else cut_t<float, 4>(o, c, s);
}

void slice_gemm_scatter(const SliceOperand& A, const void* Ap, const int* Ae, const SliceOperand& B, const void* Bp,
                        const int* Be, void* out, const SliceScatter& sc, int* err, cudaStream_t s) {
  check_pair(A, B);
  const bool f64 = A.t == DType::F64;
  SParams p = f64 ? make_params<7>(A, Ae, B, Be, err) : make_params<4>(A, Ae, B, Be, err);
  p.out = out;
  p.scatter = 1;
  p.R = sc.R;
  p.C = sc.C;
  p.rs1 = sc.rs1;
  p.cs0 = sc.cs0;
  p.cs1 = sc.cs1;
  if (f64) launch_mma<7>(A, Ap, B, Bp, p, 1, s);
  else launch_mma<4>(A, Ap, B, Bp, p, 1, s);
}

void slice_gemm(const SliceOperand& A, const void* Ap, const int* Ae, const SliceOperand& B, const void* Bp,
                const int* Be, void* C, double beta, int* err, cudaStream_t s) {
  check_pair(A, B);
  const bool f64 = A.t == DType::F64;
  SParams p = f64 ? make_params<7>(A, Ae, B, Be, err) : make_params<4>(A, Ae, B, Be, err);
  // splits in whole runs; a CTA's fixed cost (pipeline fill, output) is about half a run
  const int runs = (p.total + RUN - 1) / RUN;
  int splits = wave_splits(p.tiles, runs, 1);
  const int per = (runs + splits - 1) / splits;
  splits = (runs + per - 1) / per;
  p.per = per * RUN;
  const long long MN = (long long)p.M * p.N;
  const bool direct = splits == 1 && beta == 0.0;
  DevBuf part;
  if (!direct) part = DevBuf((size_t)splits * MN * dtype_size(A.t), s);
  p.out = direct ? C : part.p;
  if (f64) launch_mma<7>(A, Ap, B, Bp, p, splits, s);
  else launch_mma<4>(A, Ap, B, Bp, p, splits, s);
  if (direct) return;
  const unsigned g = (unsigned)std::min<long long>((MN + 255) / 256, 152 * 16);
  if (f64) k_slice_sum<double><<<g, 256, 0, s>>>(part.as<double>(), splits, MN, (double*)C, beta);
  else k_slice_sum<float><<<g, 256, 0, s>>>(part.as<float>(), splits, MN, (float*)C, beta);
  count_launch();
  TD_LAUNCH_CHECK();
}

}  // namespace tddft
