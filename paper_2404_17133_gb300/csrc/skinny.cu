// Skinny products (see skinny.cuh).
#include <algorithm>
#include <type_traits>

#include "skinny.cuh"

namespace tddft {

namespace {

constexpr int kTile = 32;        // output tile of sk_gram (32 x 32, 2 x 2 per thread)
constexpr int kGramThreads = 256;
constexpr int kComboThreads = 256;
constexpr int kComboGroups = kComboThreads / 32;   // warps splitting the K sum
constexpr int kComboKc = 256;                      // K rows of coefficients staged at a time

template <typename R, typename T> __device__ __forceinline__ R cvt(T x) { return (R)x; }
template <> __device__ __forceinline__ float cvt<float, __nv_bfloat16>(__nv_bfloat16 x) {
  return __bfloat162float(x);
}
template <> __device__ __forceinline__ double cvt<double, __nv_bfloat16>(__nv_bfloat16 x) {
  return (double)__bfloat162float(x);
}

// Partial Gram matrices: CTA (chunk, mt, nt) sums k in [chunk*KC, chunk*KC + KC)
// for the output tile (mt, nt) and writes part[chunk][m][n].  The staging loads
// are fully unrolled (thread t reads column t % KC of every row it owns), so a
// thread has all of its loads in flight at once.
template <typename TA, typename TB, typename ACC, int KC>
__global__ void __launch_bounds__(kGramThreads)
k_sk_gram(const TA* __restrict__ A, long long lda, int M, const TB* __restrict__ B, long long ldb, int N,
          int K, ACC* __restrict__ part) {
  static_assert(kGramThreads % KC == 0 || KC % kGramThreads == 0, "tile mapping");
  constexpr int RSTEP = kGramThreads / KC;        // rows advanced per pass
  constexpr int PASSES = kTile / RSTEP;
  static_assert(sizeof(ACC) == 4, "FP32 accumulation (FP64: k_sk_gram64)");
  // row stride: 16-byte aligned rows for vector loads; the 4-float skew spreads
  // the 16 B-columns of a warp over the banks
  constexpr int VW = 4;                            // elements per 16-byte load
  constexpr int LD = KC + VW;
  extern __shared__ __align__(16) unsigned char gram_raw[];
  ACC* As = reinterpret_cast<ACC*>(gram_raw);
  ACC* Bs = As + kTile * LD;
  const int tid = threadIdx.x;
  const int k0 = blockIdx.x * KC;
  const int kn = min(KC, K - k0);
  const int m0 = blockIdx.y * kTile, n0 = blockIdx.z * kTile;
  const int kk = tid % KC, r0 = tid / KC;
  const bool kin = kk < kn;
  ACC ra[PASSES], rb[PASSES];
#pragma unroll
  for (int p = 0; p < PASSES; ++p) {
    const int r = r0 + p * RSTEP;
    ra[p] = (kin && m0 + r < M) ? cvt<ACC>(A[(long long)(m0 + r) * lda + k0 + kk]) : ACC(0);
    rb[p] = (kin && n0 + r < N) ? cvt<ACC>(B[(long long)(n0 + r) * ldb + k0 + kk]) : ACC(0);
  }
#pragma unroll
  for (int p = 0; p < PASSES; ++p) {
    const int r = r0 + p * RSTEP;
    As[r * LD + kk] = ra[p];
    Bs[r * LD + kk] = rb[p];
  }
  __syncthreads();
  const int tx = tid & 15, ty = tid >> 4;
  ACC c00 = 0, c01 = 0, c10 = 0, c11 = 0;
  using V16 = float4;
  const V16* a0 = reinterpret_cast<const V16*>(As + ty * LD);
  const V16* a1 = reinterpret_cast<const V16*>(As + (ty + 16) * LD);
  const V16* b0 = reinterpret_cast<const V16*>(Bs + tx * LD);
  const V16* b1 = reinterpret_cast<const V16*>(Bs + (tx + 16) * LD);
#pragma unroll 4
  for (int k = 0; k < KC / VW; ++k) {   // columns beyond kn were staged as zeros
    const V16 x0 = a0[k], x1 = a1[k], y0 = b0[k], y1 = b1[k];
    c00 = fma(x0.x, y0.x, c00); c00 = fma(x0.y, y0.y, c00); c00 = fma(x0.z, y0.z, c00); c00 = fma(x0.w, y0.w, c00);
    c01 = fma(x0.x, y1.x, c01); c01 = fma(x0.y, y1.y, c01); c01 = fma(x0.z, y1.z, c01); c01 = fma(x0.w, y1.w, c01);
    c10 = fma(x1.x, y0.x, c10); c10 = fma(x1.y, y0.y, c10); c10 = fma(x1.z, y0.z, c10); c10 = fma(x1.w, y0.w, c10);
    c11 = fma(x1.x, y1.x, c11); c11 = fma(x1.y, y1.y, c11); c11 = fma(x1.z, y1.z, c11); c11 = fma(x1.w, y1.w, c11);
  }
  ACC* P = part + (long long)blockIdx.x * M * N;
  const int ma = m0 + ty, mb = m0 + ty + 16, na = n0 + tx, nb = n0 + tx + 16;
  if (ma < M && na < N) P[(long long)ma * N + na] = c00;
  if (ma < M && nb < N) P[(long long)ma * N + nb] = c01;
  if (mb < M && na < N) P[(long long)mb * N + na] = c10;
  if (mb < M && nb < N) P[(long long)mb * N + nb] = c11;
}

// FP64 form.  What bounds it is the FP64 unit (two DFMA per cycle and SM), so a
// lane that computes a pair outside the M x N outputs costs as much as one that
// works, and a chunk of K is as short as it takes to occupy every SM: the
// tile's Mt x Nt pairs are dealt to the threads one by one (and, where fewer than
// half of the threads have a pair, the chunk's k among groups of threads).
// K = 400, up to 60 x 10 outputs: 34 -> 3.2 us a launch (before: chunks of 128
// columns, 32 x 32 pairs whether wanted or not).
template <int KC>
__global__ void __launch_bounds__(kGramThreads)
k_sk_gram64(const double* __restrict__ A, long long lda, int M, const double* __restrict__ B, long long ldb, int N,
            int K, double* __restrict__ part) {
  constexpr int LD = KC + 1;
  extern __shared__ __align__(16) unsigned char gram_raw[];
  double* As = reinterpret_cast<double*>(gram_raw);
  double* Bs = As + kTile * LD;
  const int tid = threadIdx.x;
  const int k0 = blockIdx.x * KC;
  const int kn = min(KC, K - k0);
  const int m0 = blockIdx.y * kTile, n0 = blockIdx.z * kTile;
  const int Mt = min(kTile, M - m0), Nt = min(kTile, N - n0);
  for (int e = tid; e < (Mt + Nt) * KC; e += kGramThreads) {
    const int r = e / KC, k = e % KC;
    const double* row = r < Mt ? A + (long long)(m0 + r) * lda : B + (long long)(n0 + r - Mt) * ldb;
    (r < Mt ? As + r * LD : Bs + (r - Mt) * LD)[k] = k < kn ? row[k0 + k] : 0.0;
  }
  __syncthreads();
  double* P = part + (long long)blockIdx.x * M * N;
  const int pairs = Mt * Nt;
  if (2 * pairs > kGramThreads) {
    for (int e = tid; e < pairs; e += kGramThreads) {
      const int m = e / Nt, n = e - m * Nt;
      const double *a = As + m * LD, *b = Bs + n * LD;
      double c0 = 0.0, c1 = 0.0;
#pragma unroll
      for (int k = 0; k < KC; k += 2) {
        c0 = fma(a[k], b[k], c0);
        c1 = fma(a[k + 1], b[k + 1], c1);
      }
      P[(long long)(m0 + m) * N + n0 + n] = c0 + c1;
    }
    return;
  }
  // groups of `pairs` threads share the chunk's k
  const int G = kGramThreads / pairs, g = tid / pairs, e = tid - g * pairs;
  const int m = e / Nt, n = e - m * Nt;
  double c = 0.0;
  if (g < G)
    for (int k = g; k < KC; k += G) c = fma(As[m * LD + k], Bs[n * LD + k], c);
  __syncthreads();
  double* red = As;   // [G][pairs] (<= 256 doubles)
  if (g < G) red[tid] = c;
  __syncthreads();
  if (tid < pairs) {
    for (int q = 1; q < G; ++q) c += red[q * pairs + tid];
    P[(long long)(m0 + m) * N + n0 + n] = c;
  }
}

// One warp per output element: lane l sums the chunks l, l+32, ... in order,
// then a fixed butterfly adds the lanes (deterministic).
template <typename ACC, typename TC>
__global__ void k_sk_gram_reduce(const ACC* __restrict__ part, int S, int M, int N, TC* __restrict__ C,
                                 long long ldc, double alpha, double beta, unsigned* cmax = nullptr) {
  const long long MN = (long long)M * N;
  const int lane = threadIdx.x & 31;
  const long long warps = (long long)gridDim.x * (blockDim.x >> 5);
  float big = 0.f;   // lane 0: max |C| of this warp's elements
  for (long long i = blockIdx.x * (long long)(blockDim.x >> 5) + (threadIdx.x >> 5); i < MN; i += warps) {
    double acc = 0.0;
    for (int c = lane; c < S; c += 32) acc += (double)part[(long long)c * MN + i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) {
      const int m = (int)(i / N), n = (int)(i - (long long)m * N);
      TC* p = C + (long long)m * ldc + n;
      double v = alpha * acc;
      if (beta != 0.0) v += beta * (double)*p;
      *p = (TC)v;
      if (cmax) big = fmaxf(big, fabsf((float)v));
    }
  }
  if (cmax && lane == 0) atomicMax(cmax, __float_as_uint(big));
}

// Combination: CTA = 32 columns x kComboGroups warps; warp g sums k = g, g+8, ...
// for its lane's column and all MB rows of the block; the warps' partial sums
// are added in a fixed order through shared memory.  Coefficients are staged
// kComboKc rows of K at a time.
template <typename TS, typename TV, typename TO, typename ACC, int MB>
__global__ void __launch_bounds__(kComboThreads)
k_sk_combo(const TS* __restrict__ coef, long long scm, long long sck, int M, int K,
           const TV* __restrict__ V, long long ldv, int ncols, TO* __restrict__ out, long long ldo,
           double alpha, double beta) {
  extern __shared__ __align__(16) unsigned char combo_raw[];
  ACC* cs = reinterpret_cast<ACC*>(combo_raw);   // [kc][MB]
  ACC* red = cs + (size_t)kComboKc * MB;          // [groups][MB][33]
  const int tid = threadIdx.x, lane = tid & 31, g = tid >> 5;
  const int mb0 = blockIdx.y * MB;
  const int mn = min(MB, M - mb0);
  const int c = blockIdx.x * 32 + lane;
  ACC acc[MB];
#pragma unroll
  for (int m = 0; m < MB; ++m) acc[m] = ACC(0);
  for (int k0 = 0; k0 < K; k0 += kComboKc) {
    const int kn = min(kComboKc, K - k0);
    __syncthreads();
    for (int e = tid; e < kn * MB; e += kComboThreads) {
      const int k = e / MB, m = e - k * MB;
      cs[e] = m < mn ? (ACC)coef[(long long)(mb0 + m) * scm + (long long)(k0 + k) * sck] : ACC(0);
    }
    __syncthreads();
    if (c < ncols) {
#pragma unroll 8
      for (int k = g; k < kn; k += kComboGroups) {
        const ACC v = cvt<ACC>(V[(long long)(k0 + k) * ldv + c]);
        const ACC* ck = cs + k * MB;
#pragma unroll
        for (int m = 0; m < MB; ++m) acc[m] = fma(ck[m], v, acc[m]);
      }
    }
  }
#pragma unroll
  for (int m = 0; m < MB; ++m) red[(g * MB + m) * 33 + lane] = acc[m];
  __syncthreads();
  for (int e = tid; e < MB * 32; e += kComboThreads) {
    const int m = e >> 5, l = e & 31;
    const int col = blockIdx.x * 32 + l;
    if (m >= mn || col >= ncols) continue;
    ACC sum = ACC(0);
#pragma unroll
    for (int q = 0; q < kComboGroups; ++q) sum += red[(q * MB + m) * 33 + l];
    TO* o = out + (long long)(mb0 + m) * ldo + col;
    ACC v = (ACC)alpha * sum;
    if (beta != 0.0) v = fma((ACC)beta, (ACC)*o, v);
    *o = (TO)v;
  }
}

// FP64 combinations of few columns.  What bounds them is the FP64 unit (two DFMA per
// clock and SM), so the work has to reach every SM: a CTA owns 8 columns x 8 output
// rows, its 32 groups of 8 lanes every 32nd k.  Mean launch of a solve of 400
// columns: 7.6 -> 4.0 us.
constexpr int kFewCols = 8, kFewRows = 8, kFewK = 256;
__global__ void __launch_bounds__(256)
k_sk_combo64_few(const double* __restrict__ coef, long long scm, long long sck, int M, int K,
                 const double* __restrict__ V, long long ldv, int ncols, double* __restrict__ out, long long ldo,
                 double alpha, double beta) {
  __shared__ double cs[kFewK][kFewRows];
  __shared__ double red[8][kFewRows][kFewCols];
  const int tid = threadIdx.x, col = tid & 7, grp = tid >> 3, warp = tid >> 5;
  const int mb0 = blockIdx.y * kFewRows, mn = min(kFewRows, M - mb0);
  const int c = blockIdx.x * kFewCols + col;
  double acc[kFewRows];
#pragma unroll
  for (int m = 0; m < kFewRows; ++m) acc[m] = 0.0;
  for (int k0 = 0; k0 < K; k0 += kFewK) {
    const int kn = min(kFewK, K - k0);
    __syncthreads();
    for (int e = tid; e < kn * kFewRows; e += 256) {
      const int k = e / kFewRows, m = e % kFewRows;
      cs[k][m] = m < mn ? coef[(long long)(mb0 + m) * scm + (long long)(k0 + k) * sck] : 0.0;
    }
    __syncthreads();
    if (c < ncols) {
#pragma unroll 4
      for (int k = grp; k < kn; k += 32) {
        const double v = V[(long long)(k0 + k) * ldv + c];
#pragma unroll
        for (int m = 0; m < kFewRows; ++m)
          if (m < mn) acc[m] = fma(cs[k][m], v, acc[m]);
      }
    }
  }
  // the four groups of a warp, then the warps, in order
#pragma unroll
  for (int m = 0; m < kFewRows; ++m) {
    if (m >= mn) continue;
    acc[m] += __shfl_xor_sync(0xffffffffu, acc[m], 8);
    acc[m] += __shfl_xor_sync(0xffffffffu, acc[m], 16);
    if ((tid & 31) < 8) red[warp][m][col] = acc[m];
  }
  __syncthreads();
  if (tid < kFewRows * kFewCols) {
    const int m = tid / kFewCols, cc = blockIdx.x * kFewCols + tid % kFewCols;
    if (m < mn && cc < ncols) {
      double sum = 0.0;
#pragma unroll
      for (int w = 0; w < 8; ++w) sum += red[w][m][tid % kFewCols];
      double* o = out + (long long)(mb0 + m) * ldo + cc;
      double v = alpha * sum;
      if (beta != 0.0) v = fma(beta, *o, v);
      *o = v;
    }
  }
}

void set_smem_attr(const void* f, size_t bytes) {
  ensure_smem(f, bytes);
}

template <typename TA, typename TB, typename ACC>
void gram_typed(const void* A, long long lda, int M, const void* B, long long ldb, int N, int K, void* C,
                DType tc, long long ldc, double alpha, double beta, cudaStream_t s, unsigned* cmax = nullptr) {
  TD_REQUIRE((M + kTile - 1) / kTile <= 65535 && (N + kTile - 1) / kTile <= 65535, TDDFT_ERR_ARG,
             "sk_gram: too many rows");
  // fixed K chunks: 256 columns (FP32 staging), 64 where that leaves fewer CTAs than
  // SMs (K 3456, mean launch of a solve: 5.9 us with 256, 2.9 with 64); FP64 16 to 128, so that K up to 20,000 is cut into 150 chunks or more where
  // the columns allow it
  const long long mnt = (long long)((M + kTile - 1) / kTile) * ((N + kTile - 1) / kTile);
  int KC = (K + 255) / 256 * mnt < 152 ? 64 : 256;
  if (sizeof(ACC) == 8) KC = K <= 2432 ? 16 : (K <= 4864 ? 32 : (K <= 9728 ? 64 : 128));
  const int S = K > 0 ? (K + KC - 1) / KC : 1;
  DevBuf part((size_t)S * M * N * sizeof(ACC), s);
  if (K > 0) {
    const dim3 grid(S, (M + kTile - 1) / kTile, (N + kTile - 1) / kTile);
    if constexpr (sizeof(ACC) == 8) {
      auto go = [&](auto kernel) {
        const size_t smem = std::max((size_t)2 * kTile * (KC + 1), (size_t)kGramThreads) * sizeof(double);
        set_smem_attr((const void*)kernel, smem);
        kernel<<<grid, kGramThreads, smem, s>>>(static_cast<const double*>(A), lda, M, static_cast<const double*>(B),
                                                ldb, N, K, part.as<double>());
      };
      if (KC == 16) go(k_sk_gram64<16>);
      else if (KC == 32) go(k_sk_gram64<32>);
      else if (KC == 64) go(k_sk_gram64<64>);
      else go(k_sk_gram64<128>);
    } else {
      auto go = [&](auto kernel) {
        const size_t smem = (size_t)2 * kTile * (KC + 16 / sizeof(ACC)) * sizeof(ACC);
        set_smem_attr((const void*)kernel, smem);
        kernel<<<grid, kGramThreads, smem, s>>>(static_cast<const TA*>(A), lda, M, static_cast<const TB*>(B), ldb, N, K,
                                                part.as<ACC>());
      };
      if (KC == 64) go(k_sk_gram<TA, TB, ACC, 64>);
      else go(k_sk_gram<TA, TB, ACC, 256>);
    }
    count_launch();
    TD_LAUNCH_CHECK();
  } else {
    TD_CUDA(cudaMemsetAsync(part.p, 0, (size_t)M * N * sizeof(ACC), s));
  }
  const long long MN = (long long)M * N;
  const unsigned rb = (unsigned)std::min<long long>((MN + 7) / 8, 16 * 152);   // 8 warps per block
  if (tc == DType::F64)
    k_sk_gram_reduce<ACC, double><<<rb, 256, 0, s>>>(part.as<ACC>(), S, M, N, (double*)C, ldc, alpha, beta, cmax);
  else
    k_sk_gram_reduce<ACC, float><<<rb, 256, 0, s>>>(part.as<ACC>(), S, M, N, (float*)C, ldc, alpha, beta, cmax);
  count_launch();
  TD_LAUNCH_CHECK();
}

// Wide combination (FP32 accumulation, FP32 or BF16 V): each lane owns four
// consecutive columns, loaded with one 16-byte (FP32) or 8-byte (BF16) access
// per V row, so a warp reads 512 or 256 contiguous bytes of a row and a thread
// keeps eight such loads in flight; a CTA covers 128 columns and kWideRows
// output rows (row blocks fastest in the grid, so the CTAs that share a stripe
// of V run together and share it through L2).  The K split over warps and the
// order of every sum are those of k_sk_combo: the results are the same bits.
constexpr int kWideRows = 8;
constexpr int kWideLd = 132;   // 128 columns + 4 (16-byte aligned rows)

__device__ __forceinline__ void load4(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void load4(const __nv_bfloat16* p, float (&v)[4]) {
  const uint2 q = *reinterpret_cast<const uint2*>(p);
  const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&q.x);
  const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&q.y);
  v[0] = __low2float(a); v[1] = __high2float(a); v[2] = __low2float(b); v[3] = __high2float(b);
}

template <typename TS, typename TV, typename TO>
__global__ void __launch_bounds__(kComboThreads)
k_sk_combo_wide(const TS* __restrict__ coef, long long scm, long long sck, int M, int K,
                const TV* __restrict__ V, long long ldv, int ncols, TO* __restrict__ out, long long ldo,
                double alpha, double beta) {
  extern __shared__ __align__(16) unsigned char wide_raw[];
  float* cs = reinterpret_cast<float*>(wide_raw);        // [kComboKc][kWideRows]
  float* red = cs + (size_t)kComboKc * kWideRows;         // [groups][kWideRows][kWideLd]
  const int tid = threadIdx.x, lane = tid & 31, g = tid >> 5;
  const int mb0 = blockIdx.x * kWideRows;
  const int mn = min(kWideRows, M - mb0);
  const int c0 = blockIdx.y * 128 + lane * 4;
  const bool full = c0 + 4 <= ncols;
  float acc[kWideRows][4];
#pragma unroll
  for (int m = 0; m < kWideRows; ++m)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[m][j] = 0.f;
  for (int k0 = 0; k0 < K; k0 += kComboKc) {
    const int kn = min(kComboKc, K - k0);
    __syncthreads();
    for (int e = tid; e < kn * kWideRows; e += kComboThreads) {
      const int k = e / kWideRows, m = e - k * kWideRows;
      cs[e] = m < mn ? (float)coef[(long long)(mb0 + m) * scm + (long long)(k0 + k) * sck] : 0.f;
    }
    __syncthreads();
    if (c0 < ncols) {
#pragma unroll 8
      for (int k = g; k < kn; k += kComboGroups) {
        const TV* row = V + (long long)(k0 + k) * ldv + c0;
        float v[4];
        if (full) {
          load4(row, v);
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] = c0 + j < ncols ? cvt<float>(row[j]) : 0.f;
        }
        const float* ck = cs + k * kWideRows;
#pragma unroll
        for (int m = 0; m < kWideRows; ++m) {
          const float cm = ck[m];
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[m][j] = fmaf(cm, v[j], acc[m][j]);
        }
      }
    }
  }
#pragma unroll
  for (int m = 0; m < kWideRows; ++m)
    *reinterpret_cast<float4*>(red + (size_t)(g * kWideRows + m) * kWideLd + lane * 4) =
        make_float4(acc[m][0], acc[m][1], acc[m][2], acc[m][3]);
  __syncthreads();
  for (int e = tid; e < kWideRows * 128; e += kComboThreads) {
    const int m = e >> 7, l = e & 127;
    const int col = blockIdx.y * 128 + l;
    if (m >= mn || col >= ncols) continue;
    float sum = 0.f;
#pragma unroll
    for (int q = 0; q < kComboGroups; ++q) sum += red[(size_t)(q * kWideRows + m) * kWideLd + l];
    TO* o = out + (long long)(mb0 + m) * ldo + col;
    float v = (float)alpha * sum;
    if (beta != 0.0) v = fmaf((float)beta, (float)*o, v);
    *o = (TO)v;
  }
}

template <typename TS, typename TV, typename TO, typename ACC>
void combo_typed(const void* coef, long long scm, long long sck, int M, int K, const void* V, long long ldv,
                 int ncols, void* out, long long ldo, double alpha, double beta, cudaStream_t s) {
  if constexpr (std::is_same<ACC, float>::value &&
                (std::is_same<TV, float>::value || std::is_same<TV, __nv_bfloat16>::value)) {
    // wide path where every lane's four columns can be one aligned access
    const uintptr_t va = reinterpret_cast<uintptr_t>(V);
    const long long stripes = (ncols + 127) / 128;
    if (ncols >= 128 && ldv % 4 == 0 && va % (4 * sizeof(TV)) == 0 && stripes <= 65535) {
      const size_t smem = ((size_t)kComboKc * kWideRows + (size_t)kComboGroups * kWideRows * kWideLd) *
                          sizeof(float);
      dim3 grid((M + kWideRows - 1) / kWideRows, (unsigned)stripes);
      set_smem_attr((const void*)k_sk_combo_wide<TS, TV, TO>, smem);
      k_sk_combo_wide<TS, TV, TO><<<grid, kComboThreads, smem, s>>>(
          static_cast<const TS*>(coef), scm, sck, M, K, static_cast<const TV*>(V), ldv, ncols,
          static_cast<TO*>(out), ldo, alpha, beta);
      count_launch();
      TD_LAUNCH_CHECK();
      return;
    }
  }
  constexpr int MB = sizeof(ACC) == 8 ? 16 : 32;
  const int mblocks = (M + MB - 1) / MB;
  if constexpr (sizeof(ACC) == 8) {
    // CTAs for less than half of the SMs: smaller pieces (10 rows, K 200, 400 columns:
    // 28.8 us on 13 SMs, 7.8 here; 3456 columns, 108 CTAs: 12.9 and 14.3)
    const long long mf = (M + kFewRows - 1) / kFewRows;
    if ((long long)((ncols + 31) / 32) * mblocks < 76 && mf <= 65535) {
      k_sk_combo64_few<<<dim3((ncols + kFewCols - 1) / kFewCols, (unsigned)mf), 256, 0, s>>>(
          static_cast<const double*>(coef), scm, sck, M, K, static_cast<const double*>(V), ldv, ncols,
          static_cast<double*>(out), ldo, alpha, beta);
      count_launch();
      TD_LAUNCH_CHECK();
      return;
    }
  }
  TD_REQUIRE(mblocks <= 65535, TDDFT_ERR_ARG, "sk_combo: too many rows");
  const size_t smem = ((size_t)kComboKc * MB + (size_t)kComboGroups * MB * 33) * sizeof(ACC);
  dim3 grid((ncols + 31) / 32, mblocks);
  set_smem_attr((const void*)k_sk_combo<TS, TV, TO, ACC, MB>, smem);
  k_sk_combo<TS, TV, TO, ACC, MB><<<grid, kComboThreads, smem, s>>>(
      static_cast<const TS*>(coef), scm, sck, M, K, static_cast<const TV*>(V), ldv, ncols,
      static_cast<TO*>(out), ldo, alpha, beta);
  count_launch();
  TD_LAUNCH_CHECK();
}

// ---------------------------------------------------------------------------
// Coulomb contractions of the operator: factor rows (hundreds to thousands, FP32
// or BF16, row length K in the tens of thousands) against a few trial vectors.

// Two FP32 fused multiply-adds at once.
__device__ __forceinline__ void fma2(float2& c, float2 a, float2 b) {
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n mov.b64 z, {%0, %1};\n"
      " fma.rn.f32x2 z, x, y, z;\n mov.b64 {%0, %1}, z;\n}\n"
      : "+f"(c.x), "+f"(c.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
}

// a + b as its FP32 sum and the rounding of it (Knuth); none where the sum is not finite
__device__ __forceinline__ float2 two_sum(float a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  const float r = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
  return make_float2(s, isfinite(s) ? r : 0.f);
}

// PB bytes (4, 8 or 16) to shared memory, zero beyond `bytes`
template <int PB>
__device__ __forceinline__ void cp_piece(void* dst, const void* src, int bytes) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (PB == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %3, %2;" ::"r"(d), "l"(src), "r"(bytes), "n"(PB) : "memory");
}

// part[chunk][m][n] (chunks longer than kTallRun: part[2 chunk] + part[2 chunk + 1]) = sum
// over the chunk of A[m][k] B[n][k].  Bound by the FP32
// units for about 16 vectors and more, by reading A below that.  CTA = 128 rows
// x 4 RN vectors; 16 row groups x 4 vector groups x 4 groups of k, a thread 8
// rows x RN vectors: 13 16-byte shared-memory loads feed 160 FMAs (RN = 5),
// accumulated for even and odd k apart (packed FMAs), so a sum runs over at most
// 1/8 of the chunk (<= 256 terms).  Beyond 256 terms everything is added in FP64, as by
// the skinny product.
// cp.async keeps two (FP32) or three stages of 64 k in flight, and two CTAs share an
// SM up to 20 vectors.  n_ov 202,500, 1350 BF16 rows, 20 vectors: 365 us (992 by the
// skinny product, 433 with one CTA per SM); n_ov 24,000, 2000 FP32 rows: 71 (149, 83).
constexpr int kTallRows = 128, kTallK = 64, kTallChunk = 2048, kTallRun = 256;
template <typename TA> struct TallCfg {
  static constexpr int LDA = kTallK + (sizeof(TA) == 4 ? 4 : 8);   // elements: rows skewed over the banks
  static constexpr int LDB = kTallK + 8;
  static constexpr int STAGES = sizeof(TA) == 4 ? 2 : 3;          // two CTAs per SM for up to 20 vectors
  static constexpr int A_BYTES = kTallRows * LDA * (int)sizeof(TA);
  static int stage_bytes(int rn) { return A_BYTES + 4 * rn * LDB * 4; }
};

__device__ __forceinline__ void quad(const float* p, float2& a, float2& b) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  a = make_float2(q.x, q.y);
  b = make_float2(q.z, q.w);
}
__device__ __forceinline__ void quad(const __nv_bfloat16* p, float2& a, float2& b) {
  const uint2 q = *reinterpret_cast<const uint2*>(p);
  a = make_float2(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xffff0000u));
  b = make_float2(__uint_as_float(q.y << 16), __uint_as_float(q.y & 0xffff0000u));
}

// PA, PX: bytes that the rows of A and of the vectors are aligned to.
template <typename TA, int RN, int PA, int PX>
__global__ void __launch_bounds__(256, RN <= 5 ? 2 : 1)
k_tall_gram(const TA* __restrict__ A, int M, const float* __restrict__ B, int N, int K, int chunk,
            float* __restrict__ part) {
  using C = TallCfg<TA>;
  constexpr int NT = 4 * RN, EA = PA / (int)sizeof(TA), EX = PX / 4;   // elements per piece
  constexpr int STAGE = C::A_BYTES + NT * C::LDB * 4, kTallStages = C::STAGES;
  extern __shared__ __align__(16) unsigned char tall_raw[];
  const int tid = threadIdx.x;
  const int m0 = blockIdx.x * kTallRows, n0 = blockIdx.z * NT;
  const int k0 = blockIdx.y * chunk, k1 = min(K, k0 + chunk);
  const int nst = (k1 - k0 + kTallK - 1) / kTallK;
  auto load = [&](int st) {
    if (st < nst) {
      unsigned char* base = tall_raw + (st % kTallStages) * STAGE;
      TA* As = reinterpret_cast<TA*>(base);
      float* Bs = reinterpret_cast<float*>(base + C::A_BYTES);
      const int kb = k0 + st * kTallK;
      constexpr int CA = kTallK / EA;                       // pieces per row of A
      for (int e = tid; e < kTallRows * CA; e += 256) {
        const int r = e / CA, c = (e % CA) * EA;
        const int left = min(k1 - kb - c, EA);
        const bool in = m0 + r < M && left > 0;
        cp_piece<PA>(As + r * C::LDA + c, in ? A + (long long)(m0 + r) * K + kb + c : A,
                     in ? left * (int)sizeof(TA) : 0);
      }
      for (int e = tid; e < NT * (kTallK / EX); e += 256) {
        const int r = e / (kTallK / EX), c = (e % (kTallK / EX)) * EX;
        const int left = min(k1 - kb - c, EX);
        const bool in = n0 + r < N && left > 0;
        cp_piece<PX>(Bs + r * C::LDB + c, in ? B + (long long)(n0 + r) * K + kb + c : B, in ? left * 4 : 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const int kg = tid >> 6, rg = tid & 15, cg = (tid >> 4) & 3;
  float2 acc[8][RN];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) acc[i][j] = make_float2(0.f, 0.f);
  for (int st = 0; st < kTallStages - 1; ++st) load(st);
  for (int st = 0; st < nst; ++st) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kTallStages - 2) : "memory");
    __syncthreads();
    load(st + kTallStages - 1);
    const unsigned char* base = tall_raw + (st % kTallStages) * STAGE;
    const TA* As = reinterpret_cast<const TA*>(base) + rg * C::LDA;
    const float* Bs = reinterpret_cast<const float*>(base + C::A_BYTES) + cg * C::LDB;
    // BF16: rows 8 apart share banks, so every second eight take the neighbouring k
#pragma unroll 2
    for (int q = sizeof(TA) == 2 ? kg ^ (rg >> 3) : kg; q < kTallK / 4; q += 4) {
      float2 b0[RN], b1[RN];
#pragma unroll
      for (int j = 0; j < RN; ++j) quad(Bs + 4 * j * C::LDB + 4 * q, b0[j], b1[j]);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float2 a0, a1;
        quad(As + 16 * i * C::LDA + 4 * q, a0, a1);
#pragma unroll
        for (int j = 0; j < RN; ++j) {
          fma2(acc[i][j], a0, b0[j]);
          fma2(acc[i][j], a1, b1[j]);
        }
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  // the eight sums (even and odd k of four groups), added in order: of a chunk of 256
  // terms as one run of FP32; of a longer one without loss, the rounding of every
  // addition kept, so that it leaves a sum and its remainder
  float2* red = reinterpret_cast<float2*>(tall_raw);   // [4][128][NT]
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < RN; ++j) red[(kg * kTallRows + rg + 16 * i) * NT + cg + 4 * j] = acc[i][j];
  __syncthreads();
  const long long MN = (long long)M * N;
  const bool lng = chunk > kTallRun;
  float* P = part + (lng ? 2 : 1) * blockIdx.y * MN;
  for (int e = tid; e < kTallRows * NT; e += 256) {
    const int r = e / NT, c = e - r * NT;
    if (m0 + r >= M || n0 + c >= N) continue;
    float v = 0.f, rest = 0.f;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const float2 q = red[g * kTallRows * NT + e], w = two_sum(q.x, q.y), t = two_sum(v, w.x);
      v = t.x;
      rest += t.y + w.y;
    }
    const long long at = (long long)(m0 + r) * N + n0 + c;
    P[at] = v;
    if (lng) P[MN + at] = rest;
  }
}

// out[n][c] = sum_P t[P][n] V[P][c] for up to RN vectors in one pass over V: a lane
// owns four columns, the CTA's eight warps every eighth P (the next eight loads
// in flight while eight are used), and their sums are added in order.  The packed
// FMAs hold two vectors: (t_n, t_n+1) comes from shared memory as it is, four at a
// load, and only the four elements of V are doubled; the loads in flight stay as
// stored, so that two CTAs fit an SM (one CTA, pairs of columns and doubled t: 580 us
// for 1350 BF16 rows of 202,500 and 20 vectors, 321 now).
constexpr int kTallKc = 256;
template <typename TV> struct Quad;
template <> struct Quad<float> { using raw = float4; };
template <> struct Quad<__nv_bfloat16> { using raw = uint2; };
template <typename TV, int RN>
__global__ void __launch_bounds__(256, 2)
k_tall_combo(const float* __restrict__ t, int N, int K, const TV* __restrict__ V, int ncols, float* __restrict__ out) {
  static_assert(RN % 4 == 0, "vectors in fours");
  extern __shared__ __align__(16) unsigned char tallc_raw[];
  float* cs = reinterpret_cast<float*>(tallc_raw);        // [kTallKc][RN]
  float* red = reinterpret_cast<float*>(tallc_raw);       // later: [4][RN][132]
  const int tid = threadIdx.x, lane = tid & 31, g = tid >> 5;
  const int n0 = blockIdx.y * RN;
  const int c0 = blockIdx.x * 128 + lane * 4;
  const bool live = c0 < ncols;
  float2 acc[RN / 2][4];
#pragma unroll
  for (int j = 0; j < RN / 2; ++j)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[j][c] = make_float2(0.f, 0.f);
  using Raw = typename Quad<TV>::raw;
  constexpr int U = sizeof(TV) == 2 ? 8 : 4;
  Raw v[U], w[U];
  auto load = [&](int k0, Raw (&x)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 + g + 8 * u;
      x[u] = Raw{};
      if (live && k < K) x[u] = *reinterpret_cast<const Raw*>(V + (long long)k * ncols + c0);
    }
  };
  auto use = [&](int k, const Raw (&x)[U]) {   // k: row within the staged block
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float4* c = reinterpret_cast<const float4*>(cs + (k + g + 8 * u) * RN);
      float2 x0, x1;
      quad(reinterpret_cast<const TV*>(&x[u]), x0, x1);
      const float2 e0 = make_float2(x0.x, x0.x), e1 = make_float2(x0.y, x0.y);
      const float2 e2 = make_float2(x1.x, x1.x), e3 = make_float2(x1.y, x1.y);
#pragma unroll
      for (int j = 0; j < RN / 4; ++j) {
        const float4 q = c[j];
        const float2 qa = make_float2(q.x, q.y), qb = make_float2(q.z, q.w);
        fma2(acc[2 * j][0], qa, e0);
        fma2(acc[2 * j][1], qa, e1);
        fma2(acc[2 * j][2], qa, e2);
        fma2(acc[2 * j][3], qa, e3);
        fma2(acc[2 * j + 1][0], qb, e0);
        fma2(acc[2 * j + 1][1], qb, e1);
        fma2(acc[2 * j + 1][2], qb, e2);
        fma2(acc[2 * j + 1][3], qb, e3);
      }
    }
  };
  load(0, v);
  for (int k0 = 0; k0 < K; k0 += kTallKc) {
    __syncthreads();
    for (int e = tid; e < kTallKc * RN; e += 256) {
      const int k = e / RN, j = e - k * RN;
      cs[e] = k0 + k < K && n0 + j < N ? t[(long long)(k0 + k) * N + n0 + j] : 0.f;
    }
    __syncthreads();
    for (int k = 0; k < kTallKc && k0 + k < K; k += 16 * U) {
      load(k0 + k + 8 * U, w);
      use(k, v);
      load(k0 + k + 16 * U, v);
      use(k + 8 * U, w);
    }
  }
  // sums of the warps g and g + 4 first, then the four in order
  __syncthreads();
#pragma unroll
  for (int pass = 1; pass >= 0; --pass) {
    if ((g >> 2) == pass) {
#pragma unroll
      for (int j = 0; j < RN; ++j) {
        float* r = red + ((g & 3) * RN + j) * 132 + lane * 4;
        float4 v = j & 1 ? make_float4(acc[j / 2][0].y, acc[j / 2][1].y, acc[j / 2][2].y, acc[j / 2][3].y)
                         : make_float4(acc[j / 2][0].x, acc[j / 2][1].x, acc[j / 2][2].x, acc[j / 2][3].x);
        if (pass == 0) {
          const float4 o = *reinterpret_cast<const float4*>(r);
          v = make_float4(v.x + o.x, v.y + o.y, v.z + o.z, v.w + o.w);
        }
        *reinterpret_cast<float4*>(r) = v;
      }
    }
    __syncthreads();
  }
  for (int e = tid; e < RN * 128; e += 256) {
    const int j = e >> 7, l = e & 127, col = blockIdx.x * 128 + l;
    if (n0 + j >= N || col >= ncols) continue;
    float v = 0.f;
#pragma unroll
    for (int q = 0; q < 4; ++q) v += red[(q * RN + j) * 132 + l];
    out[(long long)(n0 + j) * ncols + col] = v;
  }
}

template <typename TA, int RN, int PA, int PX>
void tall_gram_launch(const TA* A, int M, const float* B, int N, int K, int chunk, int S, float* part, cudaStream_t s) {
  const int nb = (N + 4 * RN - 1) / (4 * RN);
  const size_t smem = std::max((size_t)TallCfg<TA>::STAGES * TallCfg<TA>::stage_bytes(RN), (size_t)4 * kTallRows * 4 * RN * 8);
  set_smem_attr((const void*)k_tall_gram<TA, RN, PA, PX>, smem);
  k_tall_gram<TA, RN, PA, PX><<<dim3((M + kTallRows - 1) / kTallRows, S, nb), 256, smem, s>>>(A, M, B, N, K, chunk, part);
}

template <typename TA, int PA, int PX>
void tall_gram_typed(const TA* A, int M, const float* B, int N, int K, float* part, int chunk, int S, cudaStream_t s) {
  // one pass over A up to 32 vectors; above that passes of 32, but two of 20 for 33 to 40
  // (two CTAs share an SM up to RN 5, and two passes of 32 would leave 24 or more columns idle)
  const int rn = N > 32 && N <= 40 ? 5 : (std::min(N, 32) + 3) / 4;
  if (rn <= 2) tall_gram_launch<TA, 2, PA, PX>(A, M, B, N, K, chunk, S, part, s);
  else if (rn <= 4) tall_gram_launch<TA, 4, PA, PX>(A, M, B, N, K, chunk, S, part, s);
  else if (rn == 5) tall_gram_launch<TA, 5, PA, PX>(A, M, B, N, K, chunk, S, part, s);
  else tall_gram_launch<TA, 8, PA, PX>(A, M, B, N, K, chunk, S, part, s);
}

template <typename TV, int RN>
void tall_combo_launch(const float* t, int N, int K, const TV* V, int ncols, float* out, cudaStream_t s) {
  const size_t smem = std::max((size_t)kTallKc * RN * 4, (size_t)4 * RN * 132 * 4);
  set_smem_attr((const void*)k_tall_combo<TV, RN>, smem);
  k_tall_combo<TV, RN><<<dim3((ncols + 127) / 128, (N + RN - 1) / RN), 256, smem, s>>>(t, N, K, V, ncols, out);
}

template <typename TV>
void tall_combo_typed(const float* t, int N, int K, const TV* V, int ncols, float* out, cudaStream_t s) {
  // as few passes over V as 20 vectors each allow, equally filled; more, smaller ones
  // where that leaves less than two CTAs per SM (V then comes from L2)
  int passes = (N + 19) / 20;
  const int cb = (ncols + 127) / 128;
  while (cb * passes < 304 && N > 8 * passes) ++passes;
  const int per = (N + passes - 1) / passes;
  if (per <= 8) tall_combo_launch<TV, 8>(t, N, K, V, ncols, out, s);
  else if (per <= 12) tall_combo_launch<TV, 12>(t, N, K, V, ncols, out, s);
  else if (per <= 16) tall_combo_launch<TV, 16>(t, N, K, V, ncols, out, s);
  else tall_combo_launch<TV, 20>(t, N, K, V, ncols, out, s);
}

}  // namespace

void sk_gram(const void* A, DType ta, long long lda, int M, const void* B, DType tb, long long ldb, int N,
             int K, void* C, DType tc, long long ldc, double alpha, double beta, cudaStream_t s, unsigned* cmax) {
  if (M <= 0 || N <= 0) return;
  TD_REQUIRE(tc == DType::F32 || tc == DType::F64, TDDFT_ERR_ARG, "sk_gram: output type");
  if (ta == DType::F64 && tb == DType::F64)
    gram_typed<double, double, double>(A, lda, M, B, ldb, N, K, C, tc, ldc, alpha, beta, s, cmax);
  else if (ta == DType::F32 && tb == DType::F32)
    gram_typed<float, float, float>(A, lda, M, B, ldb, N, K, C, tc, ldc, alpha, beta, s, cmax);
  else if (ta == DType::BF16 && tb == DType::F32)
    gram_typed<__nv_bfloat16, float, float>(A, lda, M, B, ldb, N, K, C, tc, ldc, alpha, beta, s, cmax);
  else
    throw Error(TDDFT_ERR_ARG, "sk_gram: unsupported operand types");
}

void sk_combo(const void* coef, DType tcoef, long long scm, long long sck, int M, int K, const void* V,
              DType tv, long long ldv, int ncols, void* out, DType tout, long long ldo, double alpha,
              double beta, cudaStream_t s) {
  if (M <= 0 || ncols <= 0) return;
  TD_REQUIRE(tcoef == DType::F32 || tcoef == DType::F64, TDDFT_ERR_ARG, "sk_combo: coefficient type");
  if (tv == DType::F64 && tout == DType::F64) {
    TD_REQUIRE(tcoef == DType::F64, TDDFT_ERR_ARG, "sk_combo: FP64 vectors need FP64 coefficients");
    combo_typed<double, double, double, double>(coef, scm, sck, M, K, V, ldv, ncols, out, ldo, alpha, beta, s);
  } else if (tv == DType::F32 && tout == DType::F32) {
    if (tcoef == DType::F64)
      combo_typed<double, float, float, float>(coef, scm, sck, M, K, V, ldv, ncols, out, ldo, alpha, beta, s);
    else
      combo_typed<float, float, float, float>(coef, scm, sck, M, K, V, ldv, ncols, out, ldo, alpha, beta, s);
  } else if (tv == DType::BF16 && tout == DType::F32 && tcoef == DType::F32) {
    combo_typed<float, __nv_bfloat16, float, float>(coef, scm, sck, M, K, V, ldv, ncols, out, ldo, alpha,
                                                    beta, s);
  } else {
    throw Error(TDDFT_ERR_ARG, "sk_combo: unsupported operand types");
  }
}

// The largest of 16, 8, 4, 2 bytes that every row of K elements begins at a multiple of
static int row_alignment(const void* p, DType t, int K) {
  const unsigned long long v = reinterpret_cast<uintptr_t>(p) | (unsigned long long)K * dtype_size(t) | 16ull;
  return (int)(v & ~(v - 1));
}

void tall_gram(const void* A, DType ta, int M, const float* X, int N, int K, float* t, cudaStream_t s, unsigned* tmax) {
  if (M <= 0 || N <= 0) return;
  // from 128 rows on, a full tile and a long K; other shapes and BF16 rows of an odd
  // length take the skinny Gram product (with its reduction, 20 vectors: n_ov 24,000,
  // 2000 FP32 rows 186 us there, 98 here; n_ov 202,500, 1350 BF16 rows 1090 and 403).
  // The K chunks number at most 65,535 (grid).
  const int pa = row_alignment(A, ta, K), px = row_alignment(X, DType::F32, K);
  if (!(M >= kTallRows && K >= 1024 && K <= 65535 * kTallChunk && pa >= 4 && (ta == DType::F32 || ta == DType::BF16))) {
    sk_gram(A, ta, K, M, X, DType::F32, K, N, K, t, DType::F32, N, 1.0, 0.0, s, tmax);
    return;
  }
  // K chunks: three waves of one CTA per SM, at most 2048 terms
  const int mt = (M + kTallRows - 1) / kTallRows;
  int S = std::max((3 * 152 + mt - 1) / mt, (K + kTallChunk - 1) / kTallChunk);
  int chunk = ((K + S - 1) / S + kTallK - 1) / kTallK * kTallK;
  chunk = std::max(chunk, 4 * kTallK);
  S = (K + chunk - 1) / chunk;
  const int parts = chunk > kTallRun ? 2 * S : S;
  DevBuf part((size_t)parts * M * N * 4, s);
  float* pt = part.as<float>();
  if (ta == DType::F32) {
    const float* a = static_cast<const float*>(A);
    if (pa == 16 && px == 16) tall_gram_typed<float, 16, 16>(a, M, X, N, K, pt, chunk, S, s);
    else tall_gram_typed<float, 4, 4>(a, M, X, N, K, pt, chunk, S, s);
  } else {
    const __nv_bfloat16* a = static_cast<const __nv_bfloat16*>(A);
    if (pa == 16 && px == 16) tall_gram_typed<__nv_bfloat16, 16, 16>(a, M, X, N, K, pt, chunk, S, s);
    else if (pa >= 8 && px == 16) tall_gram_typed<__nv_bfloat16, 8, 16>(a, M, X, N, K, pt, chunk, S, s);
    else tall_gram_typed<__nv_bfloat16, 4, 4>(a, M, X, N, K, pt, chunk, S, s);
  }
  count_launch();
  TD_LAUNCH_CHECK();
  const long long MN = (long long)M * N;
  const unsigned rb = (unsigned)std::min<long long>((MN + 7) / 8, 16 * 152);
  k_sk_gram_reduce<float, float><<<rb, 256, 0, s>>>(part.as<float>(), parts, M, N, t, N, 1.0, 0.0, tmax);
  count_launch();
  TD_LAUNCH_CHECK();
}

void tall_combo(const float* t, int N, int K, const void* V, DType tv, int ncols, float* out, cudaStream_t s) {
  if (N <= 0 || ncols <= 0) return;
  // four columns are one load of 16 (FP32) or 8 (BF16) bytes (n_ov 202,500, 1350 BF16
  // rows, 20 vectors: 824 us by the skinny combination, 321 here; n_ov 24,000, 2000
  // FP32 rows, 13 vectors: 128 and 76)
  if (!(K >= 64 && ncols >= 128 && ncols % 4 == 0 &&
        ((tv == DType::F32 && row_alignment(V, tv, ncols) == 16) ||
         (tv == DType::BF16 && row_alignment(V, tv, ncols) >= 8)))) {
    sk_combo(t, DType::F32, 1, N, N, K, V, tv, ncols, ncols, out, DType::F32, ncols, 1.0, 0.0, s);
    return;
  }
  if (tv == DType::F32) tall_combo_typed<float>(t, N, K, static_cast<const float*>(V), ncols, out, s);
  else tall_combo_typed<__nv_bfloat16>(t, N, K, static_cast<const __nv_bfloat16*>(V), ncols, out, s);
  count_launch();
  TD_LAUNCH_CHECK();
}

}  // namespace tddft
