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
// before the final scaling.  An element is rounded to 2^-55 (2^-31) of its row's
// largest at most, so the error of a product is 2^-55 (2^-31) of (max|A row| |b| +
// |a| max|B row|) per term, and FP32 leaves out three products of up to 2^-28.4 max max
// together.  Where an output's terms are as large as its rows' elements that is below
// what FP64 (FP32) accumulation leaves; where they are not, the output is formed
// again on the FP64 (FP32) units (the guard, below), so that every output is within
// two roundings, 2^-52 (2^-23), of the sum of its terms' absolute values.
//
// Why: FP64 runs at 1.2 TFLOP/s on this GPU's vector units and FP32 at 75; 34
// or 10 FP16 products per term leave up to 57 and 190 TFLOP/s.
//
// CTA = 128 x W output tile (W up to 64 or 128: LV levels of W FP32 columns fill the
// tensor memory), persistent over (tile, K split) items; warp 0 issues TMA loads of
// all slices of a 32-element k-block (64-byte rows, SWIZZLE_64B), warp 1 the
// products, warps 2-9 the run epilogue, in which the tensor core waits (no tensor
// memory is left for a second set of levels).  The slices of B follow one another
// in shared memory and their levels in tensor memory, so one tcgen05.mma multiplies a
// slice of A with several slices of B: N up to 256, 128 clocks, bound by the tensor
// core; one product per pair of slices (N = 64) took 48 clocks instead of 32 to
// fetch its operands.
//
// Measured, 60 x 400 orbitals, contraction of 118 rows P with 10 vectors (FP64): 787 ->
// 610 us (MMAs alone 528), its first stage 375 -> 233; 212 rows, 13 vectors (FP32): 550
// -> 458 and 290 -> 126.  The guard takes 51 and 29 us per 103 rows (FP64), 81 and 57 per
// 180 (FP32), and a sixth (fourth) more to store per element cut.  Not faster: CTA pairs (N = 64 in a pair takes twice the
// clocks), two half tiles whose runs end half a run apart (711 and 701: the shorter
// products cost more than the overlap of the epilogue gains).
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

// Tiles of NT columns (a multiple of 16): LV levels of NT FP32 columns are at most
// the tensor memory.
template <int S> constexpr int max_cols() { return S == 7 ? 64 : 128; }
// Tile width of a guard that writes its sums of a K split to out: twice the others', since it
// is bound by fetching the magnitudes of long rows (780 x 400 outputs, K 73,000: 132 -> 85 us).
constexpr int GUARD_SUMS = 256;
template <int S> constexpr int run_length() { return S == 1 ? 1 << 24 : RUN; }   // the guard accumulates in one run
template <int S, int W> struct SCfg {
  static constexpr int NT = W;
  // levels i + j kept: FP64 needs one beyond the slices (the six products of level 7
  // are 2^-58 of max max, 1e-15 of a result whose rows decay; without them the error
  // was 1.3e-15 against 1.2e-15 of FP64 arithmetic, with them 3.5e-16; 34 products
  // instead of 28)
  static constexpr int LV = S == 7 ? 8 : S;
  static constexpr int A_SLICE = SBM * SBK * 2, B_SLICE = W * SBK * 2;
  static constexpr int STAGE_BYTES = S * (A_SLICE + B_SLICE);
  static constexpr int STAGES = S == 7 ? 2 : (S == 4 ? 3 : (W == 256 ? 6 : (W == 32 ? 12 : 10)));
  static constexpr int SMEM_BYTES = STAGES * STAGE_BYTES + 1024 + 256;
  static constexpr int NBUF = S == 1 ? 2 : 1;   // sets of levels in tensor memory
  static constexpr int TMEM_COLS = S == 1 ? 2 * W : 512;
};

// What the guard knows of an operand's rows: sum of the squared magnitudes (units
// 2^-8), largest biased exponent field, nonzero elements; and where its elements are.
struct RowInfo {
  const unsigned long long* ss;
  const int* e;
  const unsigned* nnz;
};
struct View {
  const void* p;
  int R;
  long long rs1, rs0, ps, ks;
};
struct Guard {
  RowInfo ra, rb;
  View a, b;
  int np, K;
};

struct SParams {
  int M, N;             // output rows / columns
  int Kin, nab;         // k extent per P, k-blocks per P
  int total, per;       // k-blocks in all, per split (a multiple of RUN)
  int w, tiles_n, tiles, items;   // columns per tile, tiles along N and in all, items
  const int* ea;        // exponent words of the rows of A and of B
  const int* eb;
  void* out;
  int scatter;          // 0: out[z][M][N] partials, 1: the strides below
  int R, C;
  long long rs1, cs0, cs1;
  int* err;
  Guard g;              // the guard's launches
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

__device__ __forceinline__ void mma_f16(uint32_t d, uint64_t a, uint64_t b, uint32_t accum, uint32_t idesc) {
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

__device__ __forceinline__ void tmem_ld16(float (&v)[16], uint32_t taddr) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

constexpr int kNotFinite = 1 << 20;   // exponent of a row that holds a non-finite value

// Two FP32 operations at once.
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n add.rn.f32x2 z, x, y;\n"
      " mov.b64 {%0, %1}, z;\n}\n" : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 sub2(float2 a, float2 b) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n sub.rn.f32x2 z, x, y;\n"
      " mov.b64 {%0, %1}, z;\n}\n" : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float b, float2 c) {
  float2 r;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %4};\n mov.b64 z, {%5, %6};\n"
      " fma.rn.f32x2 z, x, y, z;\n mov.b64 {%0, %1}, z;\n}\n"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b), "f"(c.x), "f"(c.y));
  return r;
}
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }

// Running sum of one output over the exact runs.
template <int S> struct Acc;
template <> struct Acc<7> {
  // units 2^-40 (levels 0-3) and 2^-72 (levels 4-7) of the scaled product, less what
  // the runs still to come will add as bias
  // (unsigned: the biases pass 2^63 on the way, what is left in the end does not)
  unsigned long long hi, lo;
  static constexpr unsigned long long BIAS = 0x4b400000;   // bits of 1.5 2^23
  __device__ __forceinline__ void clear(int runs) {
    hi = 0ull - (unsigned long long)runs * ((BIAS << 24) + BIAS);
    lo = 0ull - (unsigned long long)runs * (BIAS << 8);
  }
  // The level sums v of a run for two neighbours.  Conversions to integers run at 16
  // per clock and SM (eight per output bounded this step), so only levels 1, 2 and
  // 4 are converted: x + 1.5 2^23 holds an integer |x| <= 2^22 in its low bits, and
  // level 3 passes its multiples of 256 on to level 2, levels 6 and 5 theirs to 5
  // and 4, all exactly (level 7 joins level 6 rounded at half a unit of level 6, 2^-65
  // of max max; the products not formed weigh 2^-60).
  static __device__ __forceinline__ void add(Acc& a, Acc& b, const float2 (&v)[8]) {
    const float2 M = both(0x1.8p31f), m = both(0x1.8p23f);
    const float2 h3 = sub2(add2(v[3], M), M), r3 = add2(sub2(v[3], h3), m);
    const float2 x2 = fma2(h3, 0x1p-8f, v[2]);
    const float2 x6 = fma2(v[7], 0x1p-8f, v[6]);
    const float2 h6 = sub2(add2(x6, M), M), r6 = add2(sub2(x6, h6), m);
    const float2 x5 = fma2(h6, 0x1p-8f, v[5]);
    const float2 h5 = sub2(add2(x5, M), M), r56 = fma2(sub2(x5, h5), 256.f, r6);
    const float2 x4 = fma2(h5, 0x1p-8f, v[4]), x0 = add2(v[0], m);
    a.add1(x0.x, v[1].x, x2.x, r3.x, x4.x, r56.x);
    b.add1(x0.y, v[1].y, x2.y, r3.y, x4.y, r56.y);
  }
  __device__ __forceinline__ void add1(float x0, float x1, float x2, float r3, float x4, float r56) {
    hi += (unsigned long long)((long long)__float_as_int(x0) * 16777216 + (long long)__float2int_rn(x1) * 65536 +
                               (long long)__float2int_rn(x2) * 256 + (long long)__float_as_int(r3));
    lo += (unsigned long long)((long long)__float2int_rn(x4) * 16777216 + (long long)__float_as_int(r56) * 256);
  }
  // The sum, times 2^40, times 2^e (scale exponents of the row and the column) by
  // integer arithmetic with one rounding: conversions and products on the FP64 units
  // (two per clock and SM) took 20,000 clocks per 128 x 64 tile.
  __device__ __forceinline__ double value(int e) const {
    if (e >= kNotFinite / 2) return __longlong_as_double(0x7ff8000000000000ll);
    // 96 bits in three words, sign and magnitude
    const unsigned long long h = hi + (unsigned long long)((long long)lo >> 32);
    uint32_t w0 = (uint32_t)lo, w1 = (uint32_t)h, w2 = (uint32_t)(h >> 32);
    const uint32_t neg = w2 & 0x80000000u, m = (uint32_t)((int)w2 >> 31);
    asm("add.cc.u32 %0, %3, %6;\n addc.cc.u32 %1, %4, 0;\n addc.u32 %2, %5, 0;"
        : "=r"(w0), "=r"(w1), "=r"(w2)
        : "r"(w0 ^ m), "r"(w1 ^ m), "r"(w2 ^ m), "r"(neg >> 31));
    e += 63;                                   // exponent of the highest bit of w2
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (w2 == 0) { w2 = w1; w1 = w0; w0 = 0; e -= 32; }
    if (w2 == 0) return 0.0;
    const int lz = __clz(w2);
    e -= lz;
    const unsigned long long u =
        (unsigned long long)__funnelshift_l(w1, w2, lz) << 32 | __funnelshift_l(w0, w1, lz);
    const unsigned long long f = (u >> 11) + ((u >> 10) & 1);   // 53 bits, rounded
    if (e < -1021 || e > 1022) return ldexp(neg ? -(double)f : (double)f, e - 52);
    // the leading bit of f adds one to the exponent field
    return __longlong_as_double((long long)(((unsigned long long)(e + 1022) << 52) + f | (unsigned long long)neg << 32));
  }
};
template <> struct Acc<4> {
  float hi, lo;       // compensated sum in units 2^-16 (level 0)
  __device__ __forceinline__ void clear(int) { hi = 0.f; lo = 0.f; }
  static __device__ __forceinline__ void add(Acc& a, Acc& b, const float2 (&v)[4]) {
    const float2 x = fma2(fma2(fma2(v[3], 0x1p-8f, v[2]), 0x1p-8f, v[1]), 0x1p-8f, v[0]);
    const float2 h = make_float2(a.hi, b.hi), s = add2(h, x), bb = sub2(s, h);
    const float2 l = add2(make_float2(a.lo, b.lo), add2(sub2(h, sub2(s, bb)), sub2(x, bb)));
    a.hi = s.x; b.hi = s.y;
    a.lo = l.x; b.lo = l.y;
  }
  // times the scales r of the row and c of the column
  __device__ __forceinline__ float value(float r, float c) const { return (hi + lo) * r * c; }
  // Takes in the factor 2^e, where a product with one of the scales alone could leave FP32's
  // range (of a non-finite row or column: NaN, as what it gives with a zero row; the guard
  // puts the others).
  __device__ __forceinline__ void scale_any(int e) {
    const int e1 = min(max(e, -126), 127), e2 = min(max(e - e1, -126), 127);
    hi = (hi + lo) * __int_as_float((e1 + 127) << 23) * __int_as_float((e2 + 127) << 23);
    lo = 0.f;
    if (e >= kNotFinite / 2) hi = __int_as_float(0x7fc00000);
  }
};

// Exponent of a row's power-of-two scale from its exponent word (the largest biased
// exponent field, or the all-ones field where the row holds a non-finite value).
template <int S> __device__ __forceinline__ int row_scale(int w);
template <> __device__ __forceinline__ int row_scale<7>(int w) { return w >= 2047 ? kNotFinite : max(w, 1) - 1041; }
template <> __device__ __forceinline__ int row_scale<4>(int w) { return w >= 255 ? kNotFinite : max(w, 1) - 133; }

// ---------------------------------------------------------------------------
// The guard.  Slices are fixed point against the largest element of a row, so an
// output whose terms are all small beside max|A row| max|B row| (a row that spans
// decades where the other operand has zeros) would have fewer bits than FP64 (FP32)
// arithmetic gives it.  With the magnitudes a', b' = |x| 2^(14 - e) < 2^14 of a row
// (2^e the power of two above its largest element), the error of a sliced output is
// (root mean square over the roundings)
//   FP64: 2^-42.8 (|a'| + |b'|),   FP32: 2^-18.8 (|a'| + |b'|) + 2^-4.8 sqrt(n)
// where |.| are 2-norms over the n terms with both factors nonzero (a zero is exact; the
// last term is FP32's dropped level 4, three products).  Asked for are two roundings of
// the sum of the terms' absolute values, 2^-52 N (2^-23 N) with N = sum_k a'_k b'_k, which FP64
// (FP32) arithmetic gives for sums of two terms and only bounds by n / 2 times that for
// more.  N comes from one more FP16 product of the magnitudes; |a'| is bounded by the
// norm of the whole row and by 2^14 times the square root of the other row's nonzeros.  An
// output where N is too small is formed again from the operands themselves on the FP64
// (FP32) units: so is every output of a row with a non-finite element (whose magnitudes
// are zero), which then reaches what it meets and no more.
constexpr int kThreadTerms = 256;   // terms up to which a thread forms an output alone (else its warp)
template <typename T> struct GuardWeights;
template <> struct GuardWeights<double> { static constexpr float NORM = 588.f, COUNT = 0.f; };                // 2^(52 - 42.8)
template <> struct GuardWeights<float> { static constexpr float NORM = 18.4f, COUNT = 301124.f / (18.4f * 16384.f); };   // 2^(23 - 18.8), 2^(23 - 4.8)
template <typename T> constexpr int kExpSpecial = sizeof(T) == 8 ? 2047 : 255;

// A row's part of the bound on N: from its norm and from its nonzeros (both zero: a zero row).
template <typename T>
__device__ __forceinline__ float2 row_bound(const RowInfo& r, long long i) {
  const float inf = __int_as_float(0x7f800000);
  const int e = r.e[i];
  const float n = (float)r.nnz[i], ss = (float)r.ss[i];
  if (e >= kExpSpecial<T>) return make_float2(inf, inf);
  return make_float2(GuardWeights<T>::NORM * 0.0625f * sqrtf(ss), GuardWeights<T>::NORM * 16384.f * sqrtf(n));
}
// N less the bound; the output is formed again unless it is >= 0.
template <typename T>
__device__ __forceinline__ float margin(float N, float2 a, float2 b) {
  N -= fminf(a.x, b.y) + fminf(b.x, a.y);
  return sizeof(T) == 8 ? N : N - GuardWeights<T>::COUNT * fminf(a.y, b.y);
}

template <typename T>
__device__ __forceinline__ const T* row_of(const View& v, int r) {
  const int q = r / v.R;
  return static_cast<const T*>(v.p) + q * v.rs1 + (r - q * v.R) * v.rs0;
}
// The output (r, c) on the FP64 or FP32 units, by one thread.
template <typename T>
__device__ T dot_thread(const Guard& g, int r, int c) {
  const T *a = row_of<T>(g.a, r), *b = row_of<T>(g.b, c);
  T acc = T(0);
  for (int P = 0; P < g.np; ++P) {
    const T *x = a + P * g.a.ps, *y = b + P * g.b.ps;
#pragma unroll 8
    for (int k = 0; k < g.K; ++k) acc = fma(x[k * g.a.ks], y[k * g.b.ks], acc);
  }
  return acc;
}
// The same by a warp, the terms dealt to its lanes; every lane gets it.
template <typename T>
__device__ T dot_warp(const Guard& g, int r, int c) {
  const T *a = row_of<T>(g.a, r), *b = row_of<T>(g.b, c);
  T acc = T(0);
  int k = threadIdx.x & 31, P = 0;
  while (k >= g.K && P < g.np) { k -= g.K; ++P; }
  while (P < g.np) {
    acc = fma(a[P * g.a.ps + k * g.a.ks], b[P * g.b.ps + k * g.b.ks], acc);
    k += 32;
    while (k >= g.K && P < g.np) { k -= g.K; ++P; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}

// S = 1: the guard over the magnitudes, of operands of type T.
template <int S, int W, typename T>
__global__ void __launch_bounds__(SL_THREADS, 1)
k_slice_mma(const __grid_constant__ CUtensorMap mA, const __grid_constant__ CUtensorMap mB, const SParams p) {
  using C = SCfg<S, W>;
  constexpr int NT = C::NT, RUNL = run_length<S>();
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::STAGES * C::STAGE_BYTES);
  uint64_t* empty = full + C::STAGES;
  uint64_t* tfull = empty + C::STAGES;    // the run's levels are complete
  uint64_t* tempty = tfull + C::NBUF;     // ... and have been read
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tempty + C::NBUF);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::STAGES; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < C::NBUF; ++b) { mbar_init(&tfull[b], 1); mbar_init(&tempty[b], EPI_WARPS); }
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
    // The instructions between the products of this one thread hold the tensor core
    // up (with offsets computed in loops it ran at half its rate): offsets are
    // constants, positions are counted up, nothing is divided in the loop.
    //
    // kind::f16 with FP16 operands, FP32 accumulator, both K-major, M = 128.  One
    // product of slice ia of A with g consecutive slices of B (N = g W up to 256)
    // reaches the g levels from ia + ib on: single slices (N = 64) are bound by
    // fetching A and B from shared memory, 48 clocks instead of 32.
    constexpr uint32_t IDESC = (1u << 4) | ((uint32_t)(SBM >> 4) << 24), NB = (uint32_t)(W >> 3) << 17;
    constexpr int G = 256 / W < S ? 256 / W : S;   // slices of B per product; two products meet all of them
    static_assert(2 * G >= S && C::LV <= S + 1, "slice_gemm: slices per product");
    const uint64_t da0 = sdesc64(smem);
    const int tail = p.Kin - (p.nab - 1) * SBK > 16 ? 2 : 1;   // 16-element K steps of a P's last k-block
    uint32_t s = 0, ph = 0, run = 0, buf = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x) {
      int k0, nk;
      range(item, k0, nk);
      int pos = k0 % p.nab, left = 0;   // place among the k-blocks of a P, k-blocks left of the run
      for (int b = 0; b < nk; ++b) {
        const bool start = left == 0;
        if (start) {
          left = min(RUNL, nk - b);
          buf = run % C::NBUF;
          if (!mbar_wait(&tempty[buf], ((run++ / C::NBUF) & 1u) ^ 1u)) { ok = false; break; }
        }
        if (!mbar_wait(&full[s], ph)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t da = da0 + s * (C::STAGE_BYTES >> 4);
        const int nks = pos == p.nab - 1 ? tail : 2;
        for (int kk = 0; kk < nks; ++kk) {
          // a run's levels are opened by slice 0 of A, one past the slices by the last slice of A
          const bool first = start && kk == 0;
          const uint64_t a0 = da + 2 * kk, b0 = a0 + S * C::A_SLICE / 16;
#pragma unroll
          for (int j = 0; j < S; ++j) {
            const int ia = j ? S - j : 0;                       // the longest products last
            const uint64_t a = a0 + ia * (C::A_SLICE / 16);
            const int nbs = S < C::LV - ia ? S : C::LV - ia;    // slices of B that ia meets
            const int n0 = nbs < G ? nbs : G, n1 = nbs - n0;
            const uint32_t d = tmem + buf * W + (uint32_t)(ia * W);
            if (C::LV > S && j == 1 && first) {
              mma_f16(d, a, b0, 1u, IDESC + NB);
              mma_f16(d + W, a, b0 + C::B_SLICE / 16, 0u, IDESC + NB);
            } else {
              const uint32_t ac = j == 0 && first ? 0u : 1u;
              mma_f16(d, a, b0, ac, IDESC + n0 * NB);
              if (n1 > 0) mma_f16(d + n0 * W, a, b0 + n0 * (C::B_SLICE / 16), ac, IDESC + n1 * NB);
            }
          }
        }
        mma_commit(&empty[s]);
        if (--left == 0) mma_commit(&tfull[buf]);
        if (++s == C::STAGES) { s = 0; ph ^= 1u; }
        if (++pos == p.nab) pos = 0;
      }
    }
    if (!ok) atomicOr(p.err, 1024);
  } else if (warp >= 2) {
    constexpr int HC = W / 2;                // columns per warp
    constexpr int CH = 4;                    // columns per TMEM load
    const int q = warp & 3, side = (warp - 2) >> 2;
    const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(side * HC);
    uint32_t run = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < p.items && ok; item += gridDim.x) {
      int k0, nk;
      range(item, k0, nk);
      const int t = item % p.tiles;
      const int m0 = (t / p.tiles_n) * SBM + q * 32, n0 = (t % p.tiles_n) * NT + side * HC;
      const int row = m0 + lane;
      const bool live = m0 < p.M;            // this warp has rows to read
      const int ncol = min(HC, p.N - n0);    // columns of this warp (may be <= 0)
      if constexpr (S == 1) {
        static_assert(W == GUARD_SUMS || HC <= 64, "one bit per column");
        constexpr bool SUMS = W == GUARD_SUMS;   // k_slice_sum decides
        // the bounds of this warp's rows and columns, while the tile is being formed
        __shared__ __align__(16) float2 colb[EPI_WARPS][SUMS ? 1 : HC];
        const float2 none = make_float2(0.f, 0.f);
        const bool inside = row < p.M;
        float2 ba = none;
        float2* cb = colb[warp - 2];
        if (!SUMS) {
          if (inside) ba = row_bound<T>(p.g.ra, row);
          for (int c = lane; c < HC; c += 32) cb[c] = c < ncol ? row_bound<T>(p.g.rb, n0 + c) : none;
          __syncwarp();
        }
        const uint32_t buf = run % C::NBUF;
        bool got = mbar_wait(&tfull[buf], (run / C::NBUF) & 1u);
        ++run;
        got = __all_sync(0xffffffffu, got);
        if (!got) { if (lane == 0) atomicOr(p.err, 4096); ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        unsigned long long again = 0;
        if (live) {
#pragma unroll 1
          for (int c = 0; c < ncol; c += 16) {
            float v[16];
            tmem_ld16(v, tb + buf * W + (uint32_t)c);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (SUMS) {
              float* o = static_cast<float*>(p.out) + ((long long)(item / p.tiles) * p.M + row) * p.N + n0 + c;
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (inside && c + j < ncol) o[j] = v[j];
            } else {
              float least = 0.f;
#pragma unroll
              for (int j = 0; j < 16; j += 2) {
                const float4 q = *reinterpret_cast<const float4*>(cb + c + j);
                v[j] = margin<T>(v[j], ba, make_float2(q.x, q.y));
                v[j + 1] = margin<T>(v[j + 1], ba, make_float2(q.z, q.w));
                least = fminf(least, fminf(v[j], v[j + 1]));
              }
              if (!(least >= 0.f)) {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                  if (!(v[j] >= 0.f)) again |= 1ull << (c + j);
              }
            }
          }
          if (!inside) again = 0;
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&tempty[buf])) : "memory");
        if (!SUMS && __any_sync(0xffffffffu, again != 0)) {
          T* out = static_cast<T*>(p.out);
          auto put = [&](int r, int col, T v) {
            out[p.scatter ? (long long)(r / p.R) * p.rs1 + r % p.R + (long long)(col / p.C) * p.cs1 +
                                (long long)(col % p.C) * p.cs0
                          : (long long)r * p.N + col] = v;
          };
          if (p.g.np * p.g.K <= kThreadTerms) {
            // 16 columns at a time, dealt to the lanes (one row may hold most of them)
            __shared__ unsigned short list[EPI_WARPS][512];
            unsigned short* mine = list[warp - 2];
            for (int c = 0; c < ncol; c += 16) {
              unsigned bits = (unsigned)(again >> c) & (ncol - c < 16 ? (1u << (ncol - c)) - 1u : 0xffffu);
              const int n = __popc(bits);
              int at = n;
#pragma unroll
              for (int o = 1; o < 32; o <<= 1) {
                const int q = __shfl_up_sync(0xffffffffu, at, o);
                if (lane >= o) at += q;
              }
              const int total = __shfl_sync(0xffffffffu, at, 31);
              at -= n;
              for (; bits; bits &= bits - 1) mine[at++] = (unsigned short)(lane << 8 | (__ffs(bits) - 1));
              __syncwarp();
              for (int e = lane; e < total; e += 32) {
                const int r = m0 + (mine[e] >> 8), col = n0 + c + (mine[e] & 255);
                put(r, col, dot_thread<T>(p.g, r, col));
              }
              __syncwarp();
            }
          } else {
            for (int c = 0; c < ncol; ++c) {
              const bool mine = again >> c & 1;
              for (unsigned who = __ballot_sync(0xffffffffu, mine); who; who &= who - 1) {
                const int src = __ffs(who) - 1;
                const T v = dot_warp<T>(p.g, m0 + src, n0 + c);
                if (lane == src) put(row, n0 + c, v);
              }
            }
          }
          __syncwarp();
        }
      } else {
      Acc<S> acc[HC];
#pragma unroll
      for (int c = 0; c < HC; ++c) acc[c].clear((nk + RUNL - 1) / RUNL);
      for (int kb = 0; kb < nk; kb += RUNL, ++run) {
        bool got = mbar_wait(tfull, run & 1u);
        got = __all_sync(0xffffffffu, got);
        if (!got) { if (lane == 0) atomicOr(p.err, 2048); ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (live) {
#pragma unroll
          for (int c = 0; c < HC; c += CH) {
            if (c < ncol) {
              float v[C::LV][CH];
#pragma unroll
              for (int l = 0; l < C::LV; ++l) tmem_ld4(v[l], tb + (uint32_t)(l * W + c));
              asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
              for (int j = 0; j < CH; j += 2) {
                float2 w[C::LV];
#pragma unroll
                for (int l = 0; l < C::LV; ++l) w[l] = make_float2(v[l][j], v[l][j + 1]);
                Acc<S>::add(acc[c + j], acc[c + j + 1], w);
              }
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(tempty)) : "memory");
      }
      if (!ok || !live || ncol <= 0) continue;
      // the columns' scales, one or two per lane, dealt out by shuffles
      int sb[(HC + 31) / 32];
#pragma unroll
      for (int j = 0; j < (HC + 31) / 32; ++j)
        sb[j] = row_scale<S>(32 * j + lane < ncol ? p.eb[n0 + 32 * j + lane] : 0);
      const bool inside = row < p.M;
      const int sa = row_scale<S>(inside ? p.ea[row] : 0);
      T* out = static_cast<T*>(p.out);
      long long at, step = 1;
      int cr = 0;
      if (p.scatter) {
        cr = n0 % p.C;
        at = (long long)(row / p.R) * p.rs1 + row % p.R + (long long)(n0 / p.C) * p.cs1 + cr * p.cs0;
        step = p.cs0;
      } else {
        at = ((long long)(item / p.tiles) * p.M + row) * p.N + n0;
      }
      // FP32: scales near enough to 1 are multiplied one after the other
      bool near = true;
      float fa = 1.f, fb[(HC + 31) / 32];
      if constexpr (S == 4) {
        near = !inside || (sa >= -60 && sa <= 60);
        fa = __int_as_float((max(-60, min(sa, 60)) + 127) << 23);
#pragma unroll
        for (int j = 0; j < (HC + 31) / 32; ++j) {
          near = near && (32 * j + lane >= ncol || (sb[j] >= -60 && sb[j] <= 60));
          fb[j] = __int_as_float((max(-60, min(sb[j], 60)) + 127) << 23);
        }
        if (!__all_sync(0xffffffffu, near)) {
#pragma unroll
          for (int c = 0; c < HC; ++c) acc[c].scale_any(sa + __shfl_sync(0xffffffffu, sb[c / 32], c & 31));
          fa = 1.f;
#pragma unroll
          for (int j = 0; j < (HC + 31) / 32; ++j) fb[j] = 1.f;
        }
      }
      const long long wrap = p.cs1 - (long long)(p.C - 1) * p.cs0;   // from the last of C columns to the next first
#pragma unroll
      for (int c = 0; c < HC; ++c) {
        if constexpr (S == 4) {
          const float w = __shfl_sync(0xffffffffu, fb[c / 32], c & 31);
          if (c < ncol && inside) out[at] = acc[c].value(fa, w);
        } else {
          const int w = __shfl_sync(0xffffffffu, sb[c / 32], c & 31);
          if (c < ncol && inside) out[at] = acc[c].value(sa + w);
        }
        if (p.scatter && ++cr == p.C) {
          cr = 0;
          at += wrap;
        } else {
          at += step;
        }
      }
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

// The guard's magnitude of x against the row exponent E: |x| scaled to less than 2^14
// (zero 2^-40 below the largest, where FP16 ends).
__device__ __forceinline__ float magnitude(double x, int E) {
  const long long bits = __double_as_longlong(x);
  const int ef = (int)((bits >> 52) & 0x7ff), r = E - ef;
  return ef == 0 || r > 40 ? 0.f : __uint_as_float((unsigned)(140 - r) << 23 | ((unsigned)(bits >> 29) & 0x7fffffu));
}
__device__ __forceinline__ float magnitude(float x, int E) {
  const unsigned bits = __float_as_uint(x);
  const int ef = (int)((bits >> 23) & 0xff), r = E - ef;
  return ef == 0 || r > 40 ? 0.f : __uint_as_float((unsigned)(140 - r) << 23 | (bits & 0x7fffffu));
}

// Eight elements' slices and magnitudes; their squared magnitudes and number of
// nonzeros are added to ss and nnz.
template <typename T, int S>
__device__ __forceinline__ void store_slices(const T (&x)[8], int E, __half* dst, long long slice, float& ss, int& nnz) {
  unsigned long long d[8];
  const bool special = E >= kExpSpecial<T>;
  __half2 mag[4];
#pragma unroll
  for (int j = 0; j < 8; j += 2) {
    const T x0 = special ? T(0) : x[j], x1 = special ? T(0) : x[j + 1];
    d[j] = digits(x0, E);
    d[j + 1] = digits(x1, E);
    const float m0 = magnitude(x0, E), m1 = magnitude(x1, E);
    mag[j / 2] = __floats2half2_rn(m0, m1);
    ss = fmaf(m0, m0, fmaf(m1, m1, ss));
    nnz += (x0 != T(0)) + (x1 != T(0));
  }
  *reinterpret_cast<uint4*>(dst + S * slice) = *reinterpret_cast<const uint4*>(mag);
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
  unsigned long long* ss;   // per row, see RowInfo
  int* exps;
  unsigned* nnz;
};
__device__ __forceinline__ unsigned long long fixed_ss(float ss) { return __float2ull_ru(ss * 256.f); }

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

// Sums over groups of TPR neighbouring threads (256: the CTA) in a fixed order, for the
// group's first thread.
template <int TPR>
__device__ __forceinline__ void sum_group(float& ss, int& nnz) {
  __shared__ float rs[8];
  __shared__ int rn[8];
#pragma unroll
  for (int o = (TPR < 32 ? TPR : 32) / 2; o > 0; o >>= 1) {
    ss += __shfl_xor_sync(0xffffffffu, ss, o);
    nnz += __shfl_xor_sync(0xffffffffu, nnz, o);
  }
  if (TPR > 32) {
    if ((threadIdx.x & 31) == 0) {
      rs[threadIdx.x >> 5] = ss;
      rn[threadIdx.x >> 5] = nnz;
    }
    __syncthreads();
    if (threadIdx.x == 0)
      for (int w = 1; w < 8; ++w) {
        ss += rs[w];
        nnz += rn[w];
      }
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
  const long long slice = (long long)c.rows * c.np * c.ldk;
  float ss = 0.f;
  int nnz = 0;
  for (int g = sub; g < ng; g += TPR) {
    const int P = g / n8, k0 = (g - P * n8) * 8;
    T v[8];
    load8(x + P * c.ps + k0, c.K - k0, c.vec, v);
    store_slices<T, S>(v, E, c.dst + cut_dst(c, r, P) + k0, slice, ss, nnz);
  }
  sum_group<TPR>(ss, nnz);
  if (have && sub == 0) {
    c.exps[r] = E;
    c.ss[r] = fixed_ss(ss);
    c.nnz[r] = (unsigned)nnz;
  }
}

// The same for rows of many groups, in segments: a CTA per row left the last wave
// of a few hundred long rows nearly empty.  MAX: the exponents (zero on entry),
// else the cut.  780 FP32 rows of 84,800 elements: 213 -> 179 us, 400 rows: 114 -> 101;
// 600 FP64 rows of 47,200: 139 -> 144, 400 rows: 100 -> 102 (no gain, no loss to speak of).
constexpr int SEG = 2048;   // groups of eight elements per CTA
template <typename T, int S, bool MAX>
__global__ void __launch_bounds__(256) k_slice_seg(const CutParams c) {
  __shared__ int red[8];
  const long long r = blockIdx.x;
  const T* x = static_cast<const T*>(c.p) + (r / c.R) * c.rs1 + (r % c.R) * c.rs0;
  const int n8 = c.ldk >> 3, g1 = min(c.np * n8, (int)(blockIdx.y + 1) * SEG);
  if constexpr (MAX) {
    int E = 0;
#pragma unroll 4
    for (int g = blockIdx.y * SEG + threadIdx.x; g < g1; g += 256) {
      const int P = g / n8, k0 = (g - P * n8) * 8;
      T v[8];
      load8(x + P * c.ps + k0, c.K - k0, c.vec, v);
#pragma unroll
      for (int j = 0; j < 8; ++j) E = max(E, exp_field(v[j]));
    }
    E = __reduce_max_sync(0xffffffffu, E);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = E;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll
      for (int w = 1; w < 8; ++w) E = max(E, red[w]);
      atomicMax(&c.exps[r], E);
    }
  } else {
    const int E = c.exps[r];
    const long long slice = (long long)c.rows * c.np * c.ldk;
    float ss = 0.f;
    int nnz = 0;
#pragma unroll 2
    for (int g = blockIdx.y * SEG + threadIdx.x; g < g1; g += 256) {
      const int P = g / n8, k0 = (g - P * n8) * 8;
      T v[8];
      load8(x + P * c.ps + k0, c.K - k0, c.vec, v);
      store_slices<T, S>(v, E, c.dst + cut_dst(c, r, P) + k0, slice, ss, nnz);
    }
    sum_group<256>(ss, nnz);
    if (threadIdx.x == 0) {   // whole numbers: the same sum in any order
      atomicAdd(&c.ss[r], fixed_ss(ss));
      atomicAdd(&c.nnz[r], (unsigned)nnz);
    }
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
  float ss = 0.f;
  int nnz = 0;
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
        store_slices<T, S>(v, E, c.dst + cut_dst(c, r0 + rr, P) + k0 + kg, slice, ss, nnz);
      }
    }
  sum_group<8>(ss, nnz);
  if ((lane & 7) == 0 && r0 + rr < c.rows) {
    atomicAdd(&c.ss[r0 + rr], fixed_ss(ss));
    atomicAdd(&c.nnz[r0 + rr], (unsigned)nnz);
  }
}

// Sum of the K-split partials in a fixed order (FP64), C = sum + beta C; N: the
// guard's partials, decided on here: the outputs to be formed again are
// dealt to the CTA's warps.  A CTA takes OPB outputs.
template <typename T, int OPB>
__global__ void __launch_bounds__(256) k_slice_sum(const T* __restrict__ part, int S, const float* __restrict__ N, int SN,
                                                   long long M, int ncol, T* C, double beta, const Guard g) {
  __shared__ T again[OPB];      // values formed again
  __shared__ int list[OPB];
  __shared__ int count;
  const long long MN = M * ncol;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (long long t0 = (long long)blockIdx.x * OPB; t0 < MN; t0 += (long long)gridDim.x * OPB) {
    const long long t = t0 + tid;
    const bool in = tid < OPB && t < MN;
    double v = 0.0;
    bool bad = false;
    if (tid == 0) count = 0;
    __syncthreads();
    if (in) {
      for (int s = 0; s < S; ++s) v += (double)part[s * MN + t];
      float n = 0.f;
      for (int s = 0; s < SN; ++s) n += N[s * MN + t];
      const long long r = t / ncol;
      bad = !(margin<T>(n, row_bound<T>(g.ra, r), row_bound<T>(g.rb, t - r * ncol)) >= 0.f);
      if (bad) list[atomicAdd(&count, 1)] = tid;
    }
    if (__syncthreads_or(bad)) {
      for (int q = warp; q < count; q += 8) {
        const long long u = t0 + list[q], r = u / ncol;
        const T w = dot_warp<T>(g, (int)r, (int)(u - r * ncol));
        if (lane == 0) again[list[q]] = w;
      }
      __syncthreads();
      if (bad) v = (double)again[tid];
    }
    if (in) {
      if (beta != 0.0) v += beta * (double)C[t];
      C[t] = (T)v;
    }
    __syncthreads();
  }
}

// guard: the magnitudes, which follow the slices
CUtensorMap slice_map(const SliceOperand& o, const void* parts, int box_rows, bool guard) {
  const int S = guard ? 1 : slice_count(o.t);
  const long long ldk = tc_pad(o.K);
  if (guard) parts = static_cast<const __half*>(parts) + slice_count(o.t) * (long long)o.rows * o.np * ldk;
  // (k, P, row, slice) or, p_outer, (k, row, P, slice)
  const uint64_t n1 = o.p_outer ? o.rows : o.np, n2 = o.p_outer ? o.np : o.rows;
  const uint64_t dims[4] = {(uint64_t)o.K, n1, n2, (uint64_t)S};
  const uint64_t strides[3] = {(uint64_t)ldk * 2, (uint64_t)ldk * 2 * n1, (uint64_t)ldk * 2 * n1 * n2};
  const uint32_t box[4] = {SBK, o.p_outer ? (uint32_t)box_rows : 1u, o.p_outer ? 1u : (uint32_t)box_rows, (uint32_t)S};
  return tc_map_f16_4d(parts, dims, strides, box, 64);
}

template <int S, int W, typename T>
void launch_cols(const SliceOperand& A, const void* Ap, const SliceOperand& B, const void* Bp, const SParams& p,
                 cudaStream_t s) {
  using C = SCfg<S, W>;
  const CUtensorMap ma = slice_map(A, Ap, SBM, S == 1), mb = slice_map(B, Bp, W, S == 1);
  ensure_smem((const void*)k_slice_mma<S, W, T>, C::SMEM_BYTES);
  k_slice_mma<S, W, T><<<std::min(p.items, sm_count()), SL_THREADS, C::SMEM_BYTES, s>>>(ma, mb, p);
  count_launch();
  TD_LAUNCH_CHECK();
}

void launch_mma(const SliceOperand& A, const void* Ap, const SliceOperand& B, const void* Bp, SParams p, int splits,
                cudaStream_t s) {
  p.items = p.tiles * splits;
  if (A.t == DType::F64) {
    if (p.w <= 16) launch_cols<7, 16, double>(A, Ap, B, Bp, p, s);
    else if (p.w <= 32) launch_cols<7, 32, double>(A, Ap, B, Bp, p, s);
    else if (p.w <= 48) launch_cols<7, 48, double>(A, Ap, B, Bp, p, s);
    else launch_cols<7, 64, double>(A, Ap, B, Bp, p, s);
  } else {
    if (p.w <= 32) launch_cols<4, 32, float>(A, Ap, B, Bp, p, s);
    else if (p.w <= 64) launch_cols<4, 64, float>(A, Ap, B, Bp, p, s);
    else if (p.w <= 96) launch_cols<4, 96, float>(A, Ap, B, Bp, p, s);
    else if (p.w <= 112) launch_cols<4, 112, float>(A, Ap, B, Bp, p, s);
    else launch_cols<4, 128, float>(A, Ap, B, Bp, p, s);
  }
}

// The guard's launch: p as for the product, in tiles of its own.
void launch_guard(const SliceOperand& A, const void* Ap, const SliceOperand& B, const void* Bp, SParams p, int splits,
                  cudaStream_t s) {
  p.items = p.tiles * splits;
  if (p.w == GUARD_SUMS) launch_cols<1, GUARD_SUMS, float>(A, Ap, B, Bp, p, s);   // (of either type)
  else if (A.t == DType::F64) {
    if (p.w <= 32) launch_cols<1, 32, double>(A, Ap, B, Bp, p, s);
    else launch_cols<1, 128, double>(A, Ap, B, Bp, p, s);
  } else {
    if (p.w <= 32) launch_cols<1, 32, float>(A, Ap, B, Bp, p, s);
    else launch_cols<1, 128, float>(A, Ap, B, Bp, p, s);
  }
}

// Row information of an operand behind `info` (info_bytes).
RowInfo row_info(const SliceOperand& o, const void* info) {
  RowInfo r;
  r.ss = static_cast<const unsigned long long*>(info);
  r.e = reinterpret_cast<const int*>(r.ss + o.rows);
  r.nnz = reinterpret_cast<const unsigned*>(r.e + o.rows);
  return r;
}
View view_of(const SliceOperand& o) { return View{o.p, o.R, o.rs1, o.rs0, o.ps, o.ks}; }

// Parameters of a product of S slices (1: its guard).
template <int S>
SParams make_params(const SliceOperand& A, const void* Ai, const SliceOperand& B, const void* Bi, int* err,
                    bool sums = false) {
  SParams p;
  std::memset(&p, 0, sizeof(p));
  p.M = A.rows;
  p.N = B.rows;
  p.Kin = A.K;
  p.nab = (A.K + SBK - 1) / SBK;
  p.total = p.nab * A.np;
  p.per = p.total;
  if constexpr (S == 1) {
    p.w = sums ? GUARD_SUMS : (p.N <= 32 ? 32 : 128);
    p.tiles_n = (p.N + p.w - 1) / p.w;
  } else {
    // the fewest tiles, of equal width, rounded up to an instance: FP64 every 16 columns; FP32
    // every 32 and one between the two widest, where most columns are idle otherwise
    p.tiles_n = (p.N + max_cols<S>() - 1) / max_cols<S>();
    p.w = (p.N + p.tiles_n - 1) / p.tiles_n;
    constexpr int widths[2][5] = {{16, 32, 48, 64, 64}, {32, 64, 96, 112, 128}};
    for (int w : widths[S == 7 ? 0 : 1])
      if (w >= p.w) { p.w = w; break; }
  }
  const long long tiles = (long long)p.tiles_n * ((p.M + SBM - 1) / SBM);
  TD_REQUIRE(tiles < (1 << 28) && (long long)p.nab * A.np < (1 << 28), TDDFT_ERR_ARG, "slice_gemm: problem too large");
  p.tiles = (int)tiles;
  const RowInfo ra = row_info(A, Ai), rb = row_info(B, Bi);
  p.ea = ra.e;
  p.eb = rb.e;
  p.err = err;
  p.R = p.C = 1;
  p.g = Guard{ra, rb, view_of(A), view_of(B), A.np, A.K};
  return p;
}

// K splits in whole runs; a CTA's fixed cost (pipeline fill, output) is about half a run
int choose_splits(SParams& p) {
  const int runs = (p.total + RUN - 1) / RUN;
  int splits = wave_splits(p.tiles, runs, 1);
  const int per = (runs + splits - 1) / splits;
  p.per = per * RUN;
  return (runs + per - 1) / per;
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
    const long long segs = (groups + SEG - 1) / SEG;
    if (segs > 2 && segs <= 65535) {
      TD_CUDA(cudaMemsetAsync(c.ss, 0, slice_info_bytes(o), s));
      const dim3 grid(o.rows, (unsigned)segs);
      k_slice_seg<T, S, true><<<grid, 256, 0, s>>>(c);
      k_slice_seg<T, S, false><<<grid, 256, 0, s>>>(c);
      count_launch();
    } else if (groups > 256) k_slice_rows<T, S, 256><<<o.rows, 256, 0, s>>>(c);
    else if (groups > 16) k_slice_rows<T, S, 32><<<(o.rows + 7) / 8, 256, 0, s>>>(c);
    else k_slice_rows<T, S, 8><<<(o.rows + 31) / 32, 256, 0, s>>>(c);
    count_launch();
  } else {
    TD_CUDA(cudaMemsetAsync(c.ss, 0, slice_info_bytes(o), s));
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
  return (size_t)slice_element_bytes(o.t) * o.rows * o.np * tc_pad(o.K);
}

void slice_cut(const SliceOperand& o, void* parts, void* info, cudaStream_t s) {
  TD_REQUIRE((o.t == DType::F64 || o.t == DType::F32) && (o.ks == 1 || o.rs0 == 1) && o.rows >= 1 && o.K >= 1,
             TDDFT_ERR_ARG, "slice_cut: unsupported operand");
  const long long es = (long long)dtype_size(o.t);
  const bool vec = o.ks == 1 && reinterpret_cast<uintptr_t>(o.p) % 16 == 0 && o.rs0 * es % 16 == 0 &&
                   o.rs1 * es % 16 == 0 && o.ps * es % 16 == 0;
  const RowInfo ri = row_info(o, info);
  const CutParams c{o.p, o.rows, o.np, o.K, tc_pad(o.K), o.R, o.p_outer ? 1 : 0, vec ? 1 : 0, o.rs1, o.rs0, o.ps,
                    o.ks, static_cast<__half*>(parts), const_cast<unsigned long long*>(ri.ss), const_cast<int*>(ri.e),
                    const_cast<unsigned*>(ri.nnz)};
  TD_REQUIRE((long long)o.np * (tc_pad(o.K) / 8) < (1ll << 31), TDDFT_ERR_ARG, "slice_cut: row too long");
  if (o.t == DType::F64) cut_t<double, 7>(o, c, s);
  else cut_t<float, 4>(o, c, s);
}

void slice_gemm_scatter(const SliceOperand& A, const void* Ap, const void* Ai, const SliceOperand& B, const void* Bp,
                        const void* Bi, void* out, const SliceScatter& sc, int* err, cudaStream_t s) {
  check_pair(A, B);
  const bool f64 = A.t == DType::F64;
  SParams p = f64 ? make_params<7>(A, Ai, B, Bi, err) : make_params<4>(A, Ai, B, Bi, err);
  SParams q = make_params<1>(A, Ai, B, Bi, err);
  for (SParams* x : {&p, &q}) {
    x->out = out;
    x->scatter = 1;
    x->R = sc.R;
    x->C = sc.C;
    x->rs1 = sc.rs1;
    x->cs0 = sc.cs0;
    x->cs1 = sc.cs1;
  }
  launch_mma(A, Ap, B, Bp, p, 1, s);
  launch_guard(A, Ap, B, Bp, q, 1, s);
}

void slice_gemm(const SliceOperand& A, const void* Ap, const void* Ai, const SliceOperand& B, const void* Bp,
                const void* Bi, void* C, double beta, int* err, cudaStream_t s) {
  check_pair(A, B);
  const bool f64 = A.t == DType::F64;
  SParams p = f64 ? make_params<7>(A, Ai, B, Bi, err) : make_params<4>(A, Ai, B, Bi, err);
  const int splits = choose_splits(p);
  const long long MN = (long long)p.M * p.N;
  const bool direct = splits == 1 && beta == 0.0;   // no partials: the guard forms outputs again in place
  SParams q = make_params<1>(A, Ai, B, Bi, err, !direct);
  if (direct) {
    p.out = q.out = C;
    launch_mma(A, Ap, B, Bp, p, 1, s);
    launch_guard(A, Ap, B, Bp, q, 1, s);
    return;
  }
  const int gs = choose_splits(q);
  const size_t pb = ((size_t)splits * MN * dtype_size(A.t) + 255) & ~(size_t)255;
  DevBuf part(pb + (size_t)gs * MN * 4, s);
  p.out = part.p;
  q.out = part.as<char>() + pb;
  launch_mma(A, Ap, B, Bp, p, splits, s);
  launch_guard(A, Ap, B, Bp, q, gs, s);
  const float* N = static_cast<const float*>(q.out);
  // 32 outputs per CTA where 256 leave most SMs without any
  auto sum = [&](auto* pt, auto* out, auto kernel, int opb) {
    const unsigned g = (unsigned)std::min<long long>((MN + opb - 1) / opb, 152 * 16);
    kernel<<<g, 256, 0, s>>>(pt, splits, N, gs, (long long)p.M, p.N, out, beta, q.g);
  };
  const bool few = MN < 152 * 256;
  if (f64) sum(part.as<double>(), (double*)C, few ? k_slice_sum<double, 32> : k_slice_sum<double, 256>, few ? 32 : 256);
  else sum(part.as<float>(), (float*)C, few ? k_slice_sum<float, 32> : k_slice_sum<float, 256>, few ? 32 : 256);
  count_launch();
  TD_LAUNCH_CHECK();
}

}  // namespace tddft
