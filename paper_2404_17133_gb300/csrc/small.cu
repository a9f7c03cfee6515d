// Small dense subspace algebra on the GPU (the projected problems of Eq. 1-2 and
// of the inner solves of Eq. precondition).
//
// GB300 executes FP64 at about 1/64 of the FP32 SIMT rate, so the O(n^3) parts
// run in FP32 and FP64 is kept to O(n^2 k) work:
//   * eig32: parallel cyclic Jacobi (round-robin pair ordering, n/2 disjoint
//     rotations per round) in FP32: the matrix by one CTA in shared memory, the
//     eigenvectors row by row from the rotations it writes down;
//   * refine_lowest: for each wanted eigenpair, Newton-type corrections
//     q <- q - sum_{j != i} v_j (v_j^T r) / (lam_j - lam), r = Hq - lam q, with
//     the FP32 eigenvectors v_j (one CTA per pair), then Cholesky-QR of the k
//     vectors and an FP64 Rayleigh-Ritz (FP64 Jacobi on the k x k matrix);
//   * shifted_solve: (H - sigma)^-1 b from the FP32 decomposition plus FP64
//     residual-correction rounds (mixed-precision iterative refinement);
//   * cholesky / trsv_rows: FP64 factor of a projected A-B and triangular solves;
//   * chol_drop: pivot-dropping Cholesky of a candidate Gram matrix, the
//     in-block step of the Gram-Schmidt orthonormalisation.
#include "small.cuh"

namespace tddft {

namespace {

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sum over the CTA; every thread gets the result.  `red` has >= 33 doubles.
__device__ double block_sum(double v, double* red) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (w == 0) {
    double t = lane < nw ? red[lane] : 0.0;
    t = warp_sum(t);
    if (lane == 0) red[32] = t;
  }
  __syncthreads();
  return red[32];
}

// 1 / x and 1 / sqrt(x) for the pivots.  An FP64 division or square root is a
// dozen dependent FP64 instructions on a unit that issues one per 64 cycles; a
// FP32 estimate and two Newton steps (error 1e-7 -> 1e-14 -> the last bits)
// take four (six).  Values that FP32 cannot hold take the division.
__device__ __forceinline__ float fast_rcp(float x) { return 1.f / x; }
__device__ __forceinline__ double fast_rcp(double x) {
  const double ax = fabs(x);
  if (!(ax > 1e-30 && ax < 1e30)) return 1.0 / x;
  double y = (double)(1.f / (float)x);
  y = fma(y, fma(-x, y, 1.0), y);
  return fma(y, fma(-x, y, 1.0), y);
}
__device__ __forceinline__ double fast_rsqrt(double x) {
  if (!(x > 1e-30 && x < 1e30)) return 1.0 / sqrt(x);
  double y = (double)rsqrtf((float)x);
  const double hx = 0.5 * x;
  y = fma(y, fma(-hx * y, y, 0.5), y);
  return fma(y, fma(-hx * y, y, 0.5), y);
}

template <typename T> __device__ __forceinline__ T big_theta();
template <> __device__ __forceinline__ float big_theta<float>() { return 1e18f; }
template <> __device__ __forceinline__ double big_theta<double>() { return 1e150; }

// Parallel cyclic Jacobi on the symmetric matrix A (n x n, shared memory,
// leading dimension ld) accumulating Q <- Q G.  Each round applies n/2
// disjoint rotations (circle-method pairing); a sweep is n-1 rounds.  The
// two-sided update of a round is done block by block: the 2x2 block of rows
// (p_i, q_i) and columns (p_j, q_j) becomes R_i X R_j^T, so a round needs one
// pass over A (and Q) and two barriers.
template <typename T>
__device__ void jacobi_cta(T* A, T* Q, int n, int ld, double frob, int max_sweeps, double stop_rel,
                           int* pp, int* qq, T* cc, T* ss, unsigned* smax) {
  const int NP = (n + 1) & ~1;
  const int half = NP / 2;
  const int tid = threadIdx.x, nth = blockDim.x;
  const T stop = (T)(stop_rel * frob);
  const T skip = (T)(stop_rel * 1e-3 * frob);
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    if (tid == 0) *smax = 0u;
    __syncthreads();
    for (int r = 0; r < NP - 1; ++r) {
      for (int i = tid; i < half; i += nth) {
        int p, q;
        if (i == 0) { p = r; q = NP - 1; }
        else { p = (r + i) % (NP - 1); q = (r - i + NP - 1) % (NP - 1); }
        T c = 1, s = 0;
        if (p < n && q < n) {
          T apq = A[p * ld + q];
          T aa = apq < 0 ? -apq : apq;
          if (aa > skip) {
            atomicMax(smax, __float_as_uint((float)aa));
            T theta = (A[q * ld + q] - A[p * ld + p]) / (T(2) * apq);
            T at = theta < 0 ? -theta : theta;
            T t = at > big_theta<T>() ? T(0.5) / theta
                                      : (theta < 0 ? T(-1) : T(1)) / (at + sqrt(theta * theta + T(1)));
            c = T(1) / sqrt(t * t + T(1));
            s = t * c;
          }
        }
        pp[i] = p; qq[i] = q; cc[i] = c; ss[i] = s;
      }
      __syncthreads();
      // A <- G^T A G, block by block: warp w takes the row pairs w, w + nw, ...,
      // its lanes the column pairs (no index division in the loop)
      const int lane = tid & 31, warp = tid >> 5, nw = nth >> 5;
      for (int bi = warp; bi < half; bi += nw) {
        const T si = ss[bi], ci = cc[bi];
        T* rp = A + pp[bi] * ld;
        T* rq = A + qq[bi] * ld;
        for (int bj = lane; bj < half; bj += 32) {
          const T sj = ss[bj];
          if (si == T(0) && sj == T(0)) continue;
          const T cj = cc[bj];
          const int pj = pp[bj], qj = qq[bj];
          const T x00 = rp[pj], x01 = rp[qj], x10 = rq[pj], x11 = rq[qj];
          // rows: R_i = [[c, -s], [s, c]]
          const T y00 = ci * x00 - si * x10, y01 = ci * x01 - si * x11;
          const T y10 = si * x00 + ci * x10, y11 = si * x01 + ci * x11;
          // columns: times [[c, s], [-s, c]]
          T z00 = cj * y00 - sj * y01, z01 = sj * y00 + cj * y01;
          T z10 = cj * y10 - sj * y11, z11 = sj * y10 + cj * y11;
          if (bi == bj) { z01 = T(0); z10 = T(0); }   // the rotation annihilates a_pq
          rp[pj] = z00; rp[qj] = z01;
          rq[pj] = z10; rq[qj] = z11;
        }
      }
      // Q <- Q G (columns p_j, q_j of every row): warp per column pair, lanes over rows
      for (int bj = warp; bj < half; bj += nw) {
        const T sj = ss[bj];
        if (sj == T(0)) continue;
        const T cj = cc[bj];
        const int pj = pp[bj], qj = qq[bj];
        for (int row = lane; row < NP; row += 32) {
          const T qp = Q[row * ld + pj], qv = Q[row * ld + qj];
          Q[row * ld + pj] = cj * qp - sj * qv;
          Q[row * ld + qj] = sj * qp + cj * qv;
        }
      }
      __syncthreads();
    }
    float m = __uint_as_float(*smax);
    __syncthreads();
    if (m <= (float)stop) break;
  }
}

// rank of diagonal entry t among the first n (ascending, ties by index)
template <typename T>
__device__ int diag_rank(const T* A, int ld, int n, int t) {
  T v = A[t * ld + t];
  int r = 0;
  for (int j = 0; j < n; ++j) {
    T u = A[j * ld + j];
    r += (u < v) || (u == v && j < t);
  }
  return r;
}

// The rotations of one Jacobi run in order: [round][pair] (c, s), and behind
// them the number of rounds and the rank of each diagonal entry.
constexpr int kJacSweeps = 16;
constexpr int kJacHalf = kSmallMax / 2;                       // pairs per round
constexpr size_t kJacRounds = (size_t)kJacSweeps * (kSmallMax - 1);
constexpr size_t kJacBytes = kJacRounds * kJacHalf * sizeof(float2) + (1 + kSmallMax) * sizeof(int);

// eig32, part 1: the same cyclic Jacobi as jacobi_cta on the upper triangle of A
// alone, by one CTA.  A round is bound by shared memory (n = 160, both triangles
// and Q: 410 KB in 3200 cycles; here 100 KB), so Q is left to k_jacobi_q, which
// replays the rotations this kernel writes down.  Casida matrices of a 10-state
// solve (n up to 160): 1612 us before, 853 and 60 now; n up to 60: 470, 298 and 20.
__global__ void __launch_bounds__(1024) k_jacobi_a(const double* __restrict__ H, int ldh, int n,
                                                   float* __restrict__ lam32, float2* __restrict__ rot,
                                                   int* __restrict__ info) {
  extern __shared__ float sm32[];
  __shared__ float2 cs[kJacHalf];
  __shared__ unsigned smax;
  __shared__ double red[33];
  const int NP = (n + 1) & ~1, ld = NP + 1, half = NP / 2;
  float* A = sm32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  double f2 = 0.0;
  for (int idx = tid; idx < NP * NP; idx += blockDim.x) {
    int r = idx / NP, c = idx - r * NP;
    double v = 0.0;
    if (r < n && c < n) v = 0.5 * (H[(long long)r * ldh + c] + H[(long long)c * ldh + r]);
    f2 += v * v;
    A[r * ld + c] = (float)v;
  }
  const double frob = sqrt(block_sum(f2, red));
  const float stop = (float)(2e-7 * frob), skip = (float)(2e-10 * frob);
  int rounds = 0;
  for (int sweep = 0; sweep < kJacSweeps; ++sweep) {
    if (tid == 0) smax = 0u;
    __syncthreads();
    for (int r = 0; r < NP - 1; ++r, ++rounds) {
      if (tid < half) {
        int p, q;
        if (tid == 0) {
          p = r;
          q = NP - 1;
        } else {
          p = r + tid;
          if (p >= NP - 1) p -= NP - 1;
          q = r - tid;
          if (q < 0) q += NP - 1;
        }
        float c = 1.f, s = 0.f;
        if (p < n && q < n) {
          float* e = A + min(p, q) * ld + max(p, q);
          const float apq = *e, aa = fabsf(apq);
          if (aa > skip) {
            atomicMax(&smax, __float_as_uint(aa));
            const float app = A[p * ld + p], aqq = A[q * ld + q];
            const float theta = (aqq - app) / (2.f * apq), at = fabsf(theta);
            const float t = at > big_theta<float>() ? 0.5f / theta
                                                    : (theta < 0 ? -1.f : 1.f) / (at + sqrtf(theta * theta + 1.f));
            c = 1.f / sqrtf(t * t + 1.f);
            s = t * c;
            // the 2 x 2 block itself (rows [[c, -s], [s, c]], columns its transpose)
            const float y00 = c * app - s * apq, y01 = c * apq - s * aqq;
            const float y10 = s * app + c * apq, y11 = s * apq + c * aqq;
            A[p * ld + p] = c * y00 - s * y01;
            A[q * ld + q] = s * y10 + c * y11;
            *e = 0.f;
          }
        }
        cs[tid] = make_float2(c, s);
        rot[(size_t)rounds * kJacHalf + tid] = make_float2(c, s);
      }
      __syncthreads();
      // blocks (i, j), i < j: rows p_i, q_i against columns p_j, q_j.  Warps take the
      // rows back and forth (their lengths shrink), lanes the columns.
      for (int b = warp, g = 0; g * nw < half; ++g, b = (g & 1) ? g * nw + nw - 1 - warp : g * nw + warp) {
        if (b >= half) continue;
        const float ci = cs[b].x, si = cs[b].y;
        int pi = r + b, qi = r - b;
        if (b == 0) { pi = r; qi = NP - 1; }
        else { if (pi >= NP - 1) pi -= NP - 1; if (qi < 0) qi += NP - 1; }
        for (int j = b + 1 + lane; j < half; j += 32) {
          const float2 w = cs[j];
          const float cj = w.x, sj = w.y;
          if (si == 0.f && sj == 0.f) continue;
          int pj = r + j, qj = r - j;
          if (pj >= NP - 1) pj -= NP - 1;
          if (qj < 0) qj += NP - 1;
          float* e00 = A + min(pi, pj) * ld + max(pi, pj);
          float* e01 = A + min(pi, qj) * ld + max(pi, qj);
          float* e10 = A + min(qi, pj) * ld + max(qi, pj);
          float* e11 = A + min(qi, qj) * ld + max(qi, qj);
          const float x00 = *e00, x01 = *e01, x10 = *e10, x11 = *e11;
          const float y00 = ci * x00 - si * x10, y01 = ci * x01 - si * x11;
          const float y10 = si * x00 + ci * x10, y11 = si * x01 + ci * x11;
          *e00 = cj * y00 - sj * y01;
          *e01 = sj * y00 + cj * y01;
          *e10 = cj * y10 - sj * y11;
          *e11 = sj * y10 + cj * y11;
        }
      }
      __syncthreads();
    }
    const float m = __uint_as_float(smax);
    __syncthreads();
    if (m <= stop) break;
  }
  if (tid == 0) info[0] = rounds;
  for (int t = tid; t < n; t += blockDim.x) {
    const int r = diag_rank(A, ld, n, t);
    lam32[r] = A[t * ld + t];
    info[1 + t] = r;
  }
}

// eig32, part 2: rows of Q <- I G_1 G_2 ... , one warp per row.  The row stays in
// registers, pair i of a round in lane i % 32: players walk one seat per round
// (round-robin), so a round is one rotation per pair and a shift of seats.  The
// rotations come through shared memory, kJacChunk rounds at a time, the next
// ones loading meanwhile (read per round from L2 they set the pace: 400 us for
// n = 160).
constexpr int kJacChunk = 32, kJacRows = 4;
template <int G>   // pairs per lane
__global__ void __launch_bounds__(32 * kJacRows) k_jacobi_q(int n, const float2* __restrict__ rot,
                                                            const int* __restrict__ info, float* __restrict__ vec32) {
  __shared__ __align__(16) float2 buf[2][kJacChunk * G * 32];
  const int row = blockIdx.x * kJacRows + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int NP = (n + 1) & ~1, half = NP / 2;
  const int rounds = info[0];
  // seat i holds players (top) i and (bottom) NP - 1 - i, seat 0: 0 and NP - 1
  float top[G], bot[G];
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int i = g * 32 + lane;
    top[g] = i < half && i == row ? 1.f : 0.f;
    bot[g] = i < half && NP - 1 - i == row ? 1.f : 0.f;
  }
  const int last = half - 1;
  auto load = [&](int r0, int b) {   // rotations of rounds r0 .. r0 + kJacChunk - 1
    const int nr = min(kJacChunk, rounds - r0);
    for (int e = threadIdx.x; e < nr * half; e += 32 * kJacRows) {
      const int r = e / half, i = e - r * half;
      const unsigned dst = (unsigned)__cvta_generic_to_shared(&buf[b][r * (G * 32) + i]);
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(rot + (size_t)(r0 + r) * kJacHalf + i)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (rounds > 0) load(0, 0);
  for (int r0 = 0, b = 0; r0 < rounds; r0 += kJacChunk, b ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();   // the chunk is here, and the other buffer has been read
    if (r0 + kJacChunk < rounds) load(r0 + kJacChunk, b ^ 1);
    const int nr = min(kJacChunk, rounds - r0);
    for (int r = 0; r < nr; ++r) {
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float2 w = buf[b][r * (G * 32) + g * 32 + lane];   // (seats beyond half hold anything: not used)
        const float x = top[g], z = bot[g];
        if (g * 32 + lane < half) {
          top[g] = w.x * x - w.y * z;
          bot[g] = w.y * x + w.x * z;
        }
      }
      // next round: top_i <- top_(i+1), top_last <- bot_last, bot_1 <- top_0,
      // bot_i <- bot_(i-1) (i >= 2), bot_0 stays
      float nt[G], nbo[G];
      const float t0 = __shfl_sync(0xffffffffu, top[0], 0);
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const float dn = __shfl_sync(0xffffffffu, top[g], (lane + 1) & 31);
        const float first = g + 1 < G ? __shfl_sync(0xffffffffu, top[g + 1 < G ? g + 1 : g], 0) : 0.f;
        nt[g] = lane == 31 ? first : dn;
        const float up = __shfl_sync(0xffffffffu, bot[g], (lane + 31) & 31);
        const float prev = g > 0 ? __shfl_sync(0xffffffffu, bot[g > 0 ? g - 1 : 0], 31) : 0.f;
        nbo[g] = lane == 0 ? prev : up;
      }
#pragma unroll
      for (int g = 0; g < G; ++g) {
        const int i = g * 32 + lane;
        if (half > 1) {
          top[g] = i == last ? bot[g] : nt[g];
          if (i == 1) bot[g] = t0;
          else if (i > 1) bot[g] = nbo[g];
        }
      }
    }
    __syncthreads();
  }
  if (row >= n) return;
  // whole sweeps: every player is back in its seat
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const int i = g * 32 + lane;
    if (i < half) {
      if (i < n) vec32[(long long)info[1 + i] * n + row] = top[g];
      if (NP - 1 - i < n) vec32[(long long)info[1 + NP - 1 - i] * n + row] = bot[g];
    }
  }
}

// One CTA per wanted eigenpair i: Newton-type refinement in FP64.
__global__ void __launch_bounds__(256) k_refine(const double* __restrict__ H, int ldh, int n,
                                                const float* __restrict__ lam32,
                                                const float* __restrict__ vec32, int rounds,
                                                double* __restrict__ Qk, double* __restrict__ Yk) {
  __shared__ double q[kSmallMax], y[kSmallMax], r[kSmallMax], c[kSmallMax];
  __shared__ double red[33];
  const int i = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
  float lmin = lam32[0], lmax = lam32[n - 1];
  double scale = fmax(fabs((double)lmin), fabs((double)lmax));
  double gapmin = 1e-5 * scale;
  for (int t = tid; t < n; t += blockDim.x) q[t] = vec32[(long long)i * n + t];
  __syncthreads();
  for (int it = 0; it <= rounds; ++it) {
    // y = H q  (warp per row)
    for (int row = w; row < n; row += nw) {
      double acc = 0.0;
      for (int l = lane; l < n; l += 32) acc += H[(long long)row * ldh + l] * q[l];
      acc = warp_sum(acc);
      if (lane == 0) y[row] = acc;
    }
    __syncthreads();
    double qy = 0.0, qq2 = 0.0;
    for (int t = tid; t < n; t += blockDim.x) { qy += q[t] * y[t]; qq2 += q[t] * q[t]; }
    qy = block_sum(qy, red);
    qq2 = block_sum(qq2, red);
    double lam = qy / qq2;
    if (it == rounds) break;
    for (int t = tid; t < n; t += blockDim.x) r[t] = y[t] - lam * q[t];
    __syncthreads();
    for (int j = w; j < n; j += nw) {
      double acc = 0.0;
      for (int l = lane; l < n; l += 32) acc += (double)vec32[(long long)j * n + l] * r[l];
      acc = warp_sum(acc);
      if (lane == 0) {
        double den = (double)lam32[j] - lam;
        c[j] = (j == i || fabs(den) < gapmin) ? 0.0 : acc / den;
      }
    }
    __syncthreads();
    for (int t = tid; t < n; t += blockDim.x) {
      double acc = 0.0;
      for (int j = 0; j < n; ++j) acc += (double)vec32[(long long)j * n + t] * c[j];
      q[t] -= acc;
    }
    __syncthreads();
    double nn = 0.0;
    for (int t = tid; t < n; t += blockDim.x) nn += q[t] * q[t];
    nn = block_sum(nn, red);
    double inv = 1.0 / sqrt(nn);
    for (int t = tid; t < n; t += blockDim.x) q[t] *= inv;
    __syncthreads();
  }
  for (int t = tid; t < n; t += blockDim.x) {
    Qk[(long long)i * n + t] = q[t];
    Yk[(long long)i * n + t] = y[t];
  }
}

// One CTA: Cholesky-QR of the k refined vectors (rows of Qk, with Yk = H Qk
// carried along), FP64 Rayleigh-Ritz on the k x k matrix, rotate into `vecs`.
__global__ void __launch_bounds__(1024) k_orth_rr(double* __restrict__ Qk, double* __restrict__ Yk,
                                                  int k, int n, double* __restrict__ lam,
                                                  double* __restrict__ vecs) {
  extern __shared__ double sm64[];
  __shared__ int pp[kWantMax / 2 + 1], qq[kWantMax / 2 + 1];
  __shared__ double cc[kWantMax / 2 + 1], ss[kWantMax / 2 + 1];
  __shared__ unsigned smax;
  __shared__ double red[33];
  const int KP = (k + 1) & ~1, ld = KP + 1;
  double* G = sm64;             // Gram / Rayleigh matrix
  double* Z = sm64 + KP * ld;   // rotations
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
  // Gram matrix of the k vectors
  for (int pidx = w; pidx < k * k; pidx += nw) {
    int a = pidx / k, b = pidx - a * k;
    if (b < a) continue;
    double acc = 0.0;
    for (int l = lane; l < n; l += 32) acc += Qk[(long long)a * n + l] * Qk[(long long)b * n + l];
    acc = warp_sum(acc);
    if (lane == 0) { G[a * ld + b] = acc; G[b * ld + a] = acc; }
  }
  __syncthreads();
  // Cholesky G = R^T R (R upper, kept in the upper triangle of G)
  for (int j = 0; j < k; ++j) {
    if (tid == 0) G[j * ld + j] = sqrt(fmax(G[j * ld + j], 1e-300));
    __syncthreads();
    double piv = G[j * ld + j];
    for (int m = j + 1 + tid; m < k; m += blockDim.x) G[j * ld + m] /= piv;
    __syncthreads();
    for (int idx = tid; idx < (k - j - 1) * (k - j - 1); idx += blockDim.x) {
      int a = j + 1 + idx / (k - j - 1), b = j + 1 + idx % (k - j - 1);
      if (b >= a) G[a * ld + b] -= G[j * ld + a] * G[j * ld + b];
    }
    __syncthreads();
  }
  // rows j of Q' = R^-T Q (forward substitution, in place), same for Y
  for (int j = 0; j < k; ++j) {
    double inv = 1.0 / G[j * ld + j];
    for (int t = tid; t < n; t += blockDim.x) {
      double qa = Qk[(long long)j * n + t], ya = Yk[(long long)j * n + t];
      for (int l = 0; l < j; ++l) {
        double rl = G[l * ld + j];
        qa -= rl * Qk[(long long)l * n + t];
        ya -= rl * Yk[(long long)l * n + t];
      }
      Qk[(long long)j * n + t] = qa * inv;
      Yk[(long long)j * n + t] = ya * inv;
    }
    __syncthreads();
  }
  // Rayleigh matrix B = Q' Y'^T (symmetrised), Jacobi in FP64
  for (int idx = tid; idx < KP * KP; idx += blockDim.x) {
    int a = idx / KP, b = idx - a * KP;
    G[a * ld + b] = 0.0;
    Z[a * ld + b] = (a == b) ? 1.0 : 0.0;
  }
  __syncthreads();
  double f2 = 0.0;
  for (int pidx = w; pidx < k * k; pidx += nw) {
    int a = pidx / k, b = pidx - a * k;
    if (b < a) continue;
    double acc = 0.0;
    for (int l = lane; l < n; l += 32)
      acc += Qk[(long long)a * n + l] * Yk[(long long)b * n + l] +
             Qk[(long long)b * n + l] * Yk[(long long)a * n + l];
    acc = 0.5 * warp_sum(acc);
    if (lane == 0) { G[a * ld + b] = acc; G[b * ld + a] = acc; f2 += (a == b ? 1.0 : 2.0) * acc * acc; }
  }
  double frob = sqrt(block_sum(f2, red));
  jacobi_cta<double>(G, Z, k, ld, frob, 30, 1e-15, pp, qq, cc, ss, &smax);
  for (int t = tid; t < k; t += blockDim.x) lam[diag_rank(G, ld, k, t)] = G[t * ld + t];
  __syncthreads();
  // vecs[rank(t)] = sum_l Z[l][t] Q'[l]
  for (int idx = tid; idx < k * n; idx += blockDim.x) {
    int t = idx / n, e = idx - t * n;
    int r = diag_rank(G, ld, k, t);
    double acc = 0.0;
    for (int l = 0; l < k; ++l) acc += Z[l * ld + t] * Qk[(long long)l * n + e];
    vecs[(long long)r * n + e] = acc;
  }
}

__global__ void __launch_bounds__(256) k_shifted(const double* __restrict__ H, int ldh, int n,
                                                 const float* __restrict__ lam32,
                                                 const float* __restrict__ vec32,
                                                 const double* __restrict__ sigma,
                                                 const double* __restrict__ B, double* __restrict__ Y,
                                                 int nref) {
  __shared__ double b[kSmallMax], y[kSmallMax], r[kSmallMax], c[kSmallMax], best[kSmallMax];
  __shared__ double red[33];
  const int rr = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
  const double sg = sigma[rr];
  for (int t = tid; t < n; t += blockDim.x) { b[t] = B[(long long)rr * n + t]; y[t] = 0.0; r[t] = b[t]; }
  __syncthreads();
  double best_res = 1e300;
  for (int it = 0; it <= nref; ++it) {
    // y += V (Lam - sigma)^-1 V^T r
    for (int j = w; j < n; j += nw) {
      double acc = 0.0;
      for (int l = lane; l < n; l += 32) acc += (double)vec32[(long long)j * n + l] * r[l];
      acc = warp_sum(acc);
      if (lane == 0) {
        double den = (double)lam32[j] - sg;
        if (fabs(den) < 1e-8) den = den < 0 ? -1e-8 : 1e-8;
        c[j] = acc / den;
      }
    }
    __syncthreads();
    for (int t = tid; t < n; t += blockDim.x) {
      double acc = 0.0;
      for (int j = 0; j < n; ++j) acc += (double)vec32[(long long)j * n + t] * c[j];
      y[t] += acc;
    }
    __syncthreads();
    if (nref == 0) { for (int t = tid; t < n; t += blockDim.x) best[t] = y[t]; break; }
    // r = b - (H - sigma) y
    for (int row = w; row < n; row += nw) {
      double acc = 0.0;
      for (int l = lane; l < n; l += 32) acc += H[(long long)row * ldh + l] * y[l];
      acc = warp_sum(acc);
      if (lane == 0) r[row] = b[row] - (acc - sg * y[row]);
    }
    __syncthreads();
    double rn = 0.0;
    for (int t = tid; t < n; t += blockDim.x) rn += r[t] * r[t];
    rn = block_sum(rn, red);
    if (rn < best_res) {
      best_res = rn;
      for (int t = tid; t < n; t += blockDim.x) best[t] = y[t];
      __syncthreads();
    } else {
      break;
    }
  }
  __syncthreads();
  for (int t = tid; t < n; t += blockDim.x) Y[(long long)rr * n + t] = best[t];
}

template <typename S>
__global__ void __launch_bounds__(1024) k_cholesky(S* __restrict__ H, int ldh, int n,
                                                   int* __restrict__ info) {
  extern __shared__ __align__(16) unsigned char chol_raw[];
  S* A = reinterpret_cast<S*>(chol_raw);
  __shared__ int bad;
  const int ld = n + 1;
  const int tid = threadIdx.x;
  for (int idx = tid; idx < n * n; idx += blockDim.x) {
    int r = idx / n, c = idx - r * n;
    A[r * ld + c] = S(0.5) * (H[(long long)r * ldh + c] + H[(long long)c * ldh + r]);
  }
  if (tid == 0) bad = 0;
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    if (tid == 0) {
      S d = A[j * ld + j];
      if (!(d > S(0)) || !isfinite(d)) bad = j + 1;
      else A[j * ld + j] = sqrt(d);
    }
    __syncthreads();
    if (bad) break;
    S piv = A[j * ld + j];
    for (int r = j + 1 + tid; r < n; r += blockDim.x) A[r * ld + j] /= piv;
    __syncthreads();
    const int m = n - j - 1;
    for (int idx = tid; idx < m * m; idx += blockDim.x) {
      int r = j + 1 + idx / m, c = j + 1 + idx % m;
      if (c <= r) A[r * ld + c] -= A[r * ld + j] * A[c * ld + j];
    }
    __syncthreads();
  }
  if (tid == 0) info[0] = bad;
  for (int idx = tid; idx < n * n; idx += blockDim.x) {
    int r = idx / n, c = idx - r * n;
    H[(long long)r * ldh + c] = (c <= r && !bad) ? A[r * ld + c] : S(0);
  }
}

// Bordered Cholesky: rows < n0 of L already hold the factor of the leading
// block; rows n0..n-1 hold the new rows of the matrix (all n columns).  Each new
// row z solves L z = a against the old factor in its own warp (blocks of 32
// unknowns in registers, a shuffle per unknown), then the new diagonal block less
// z z^T is factored column by column.  Entries above the diagonal in the first n
// columns are zeroed.  (A shuffle reduction and a division per element before: 19.5
// -> 10.5 us in FP32 inner solves, n up to 160 with 20 new rows.)
template <typename S>
__global__ void __launch_bounds__(1024) k_chol_border(S* __restrict__ Lg, int ld, int n0, int n,
                                                      int* __restrict__ info) {
  extern __shared__ __align__(16) unsigned char cb_raw[];
  S* L = reinterpret_cast<S*>(cb_raw);   // [n][ls] working copy (odd stride)
  const int ls = n | 1;
  __shared__ S dinv[kSmallMax];          // 1 / L[j][j]
  __shared__ int bad;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
    const int r = idx / n, c = idx - r * n;
    L[r * ls + c] = Lg[(long long)r * ld + c];
  }
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  if (threadIdx.x < n0) dinv[threadIdx.x] = fast_rcp(L[threadIdx.x * ls + threadIdx.x]);
  __syncthreads();
  // phase 1: L[i][j], j < n0, for every new row i
  for (int i = n0 + warp; i < n; i += nw) {
    S* Li = L + i * ls;
    for (int j0 = 0; j0 < n0; j0 += 32) {
      const int j = j0 + lane, jn = min(32, n0 - j0);
      const S* Lj = L + min(j, n0 - 1) * ls;
      S v = S(0), v1 = S(0);
      int q = 0;
      for (; q + 1 < j0; q += 2) {
        v -= Lj[q] * Li[q];
        v1 -= Lj[q + 1] * Li[q + 1];
      }
      if (q < j0) v -= Lj[q] * Li[q];
      v = (lane < jn ? Li[j] : S(0)) + (v + v1);
      const S di = lane < jn ? dinv[j] : S(0);
      for (int t = 0; t < jn; ++t) {
        const S x = __shfl_sync(0xffffffffu, v * di, t);
        if (lane == t) v = x;
        else if (lane > t) v -= Lj[j0 + t] * x;
      }
      if (lane < jn) Li[j] = v;
      __syncwarp();
    }
  }
  __syncthreads();
  // the new diagonal block less the products of the new rows, one warp per element
  const int m = n - n0;
  for (int e = warp; e < m * (m + 1) / 2; e += nw) {
    int a = (int)((sqrtf(8.f * e + 1.f) - 1.f) * 0.5f);   // e = a (a + 1) / 2 + b, b <= a
    while (a * (a + 1) / 2 > e) --a;
    while ((a + 1) * (a + 2) / 2 <= e) ++a;
    const int b = e - a * (a + 1) / 2;
    const S *La = L + (n0 + a) * ls, *Lb = L + (n0 + b) * ls;
    S acc = S(0);
    for (int q = lane; q < n0; q += 32) acc += La[q] * Lb[q];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) L[(n0 + a) * ls + n0 + b] -= acc;
  }
  __syncthreads();
  // phase 2: its factor, column by column
  for (int j = n0; j < n; ++j) {
    if (threadIdx.x == 0) {
      const S d = L[j * ls + j];
      if (!(d > S(0)) || !isfinite(d)) {
        bad = j + 1;
      } else {
        const S r = sqrt(d);
        L[j * ls + j] = r;
        dinv[j] = fast_rcp(r);
      }
    }
    __syncthreads();
    if (bad) break;
    const int w = n - j - 1;
    for (int t = threadIdx.x; t < w; t += blockDim.x) L[(j + 1 + t) * ls + j] *= dinv[j];
    __syncthreads();
    for (int idx = threadIdx.x; idx < w * w; idx += blockDim.x) {
      const int r = j + 1 + idx / w, c = j + 1 + idx % w;
      if (c <= r) L[r * ls + c] -= L[r * ls + j] * L[c * ls + j];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) info[0] = bad;
  if (bad) return;
  // write back, zero above the diagonal
  for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
    const int r = idx / n, c = idx - r * n;
    Lg[(long long)r * ld + c] = c <= r ? L[r * ls + c] : S(0);
  }
}

template <typename S>
__global__ void __launch_bounds__(256) k_trsv(const S* __restrict__ L, int ldl, int n,
                                              S* __restrict__ B, int trans) {
  __shared__ S b[kSmallMax];
  __shared__ S xj;
  S* row = B + (long long)blockIdx.x * n;
  for (int t = threadIdx.x; t < n; t += blockDim.x) b[t] = row[t];
  __syncthreads();
  if (!trans) {
    for (int j = 0; j < n; ++j) {
      if (threadIdx.x == 0) { xj = b[j] / L[(long long)j * ldl + j]; b[j] = xj; }
      __syncthreads();
      for (int r = j + 1 + threadIdx.x; r < n; r += blockDim.x) b[r] -= L[(long long)r * ldl + j] * xj;
      __syncthreads();
    }
  } else {
    for (int j = n - 1; j >= 0; --j) {
      if (threadIdx.x == 0) { xj = b[j] / L[(long long)j * ldl + j]; b[j] = xj; }
      __syncthreads();
      for (int r = threadIdx.x; r < j; r += blockDim.x) b[r] -= L[(long long)j * ldl + r] * xj;
      __syncthreads();
    }
  }
  for (int t = threadIdx.x; t < n; t += blockDim.x) row[t] = b[t];
}

constexpr int kDropMax = 112;

// Pivot-dropping Cholesky of one candidate Gram matrix by the whole CTA
// (shared memory smd >= 2 nc (nc + 1) doubles; kj / dj shared scalars).
__device__ void chol_drop_cta(const double* __restrict__ G, int nc, const double* __restrict__ norm0sq,
                              double drop2, double* __restrict__ T, int* __restrict__ keep, double* smd,
                              int& kj, double& dj) {
  const int ld = nc + 1;
  double* R = smd;                 // working Gram -> upper factor
  double* Ti = smd + nc * ld;      // T rows
  const int tid = threadIdx.x;
  for (int idx = tid; idx < nc * nc; idx += blockDim.x) {
    int a = idx / nc, b = idx - a * nc;
    R[a * ld + b] = 0.5 * (G[a * nc + b] + G[b * nc + a]);
    Ti[a * ld + b] = 0.0;
  }
  __syncthreads();
  // right-looking: after step j the trailing block holds the Gram matrix of the
  // candidates with the kept ones among 0..j projected out
  // (the diagonal ends up holding 1 / R[j][j], zero for a dropped candidate)
  for (int j = 0; j < nc; ++j) {
    if (tid == 0) {
      double d = R[j * ld + j];
      const double n0 = norm0sq ? norm0sq[j] : 1.0;
      kj = (isfinite(d) && d > drop2 * n0 && d > 0.0) ? 1 : 0;
      dj = kj ? fast_rsqrt(d) : 0.0;
      keep[j] = kj;
    }
    __syncthreads();
    for (int m = j + tid; m < nc; m += blockDim.x) R[j * ld + m] = (m == j) ? dj : (kj ? R[j * ld + m] * dj : 0.0);
    __syncthreads();
    if (kj) {
      const int m = nc - j - 1;
      for (int idx = tid; idx < m * m; idx += blockDim.x) {
        int a = j + 1 + idx / m, b = j + 1 + idx % m;
        if (b >= a) R[a * ld + b] -= R[j * ld + a] * R[j * ld + b];
      }
    }
    __syncthreads();
  }
  // T = R^-T restricted to kept rows: T[j] = (e_j - sum_{l<j} R[l][j] T[l]) / R[j][j];
  // a column depends on itself only
  for (int c = tid; c < nc; c += blockDim.x)
    for (int j = c; j < nc; ++j) {
      const double inv = R[j * ld + j];
      if (inv == 0.0) continue;   // dropped: its row of T stays zero
      double a0 = (c == j) ? 1.0 : 0.0, a1 = 0.0;
      int l = c;
      for (; l + 1 < j; l += 2) {
        a0 = fma(-R[l * ld + j], Ti[l * ld + c], a0);
        a1 = fma(-R[(l + 1) * ld + j], Ti[(l + 1) * ld + c], a1);
      }
      if (l < j) a0 = fma(-R[l * ld + j], Ti[l * ld + c], a0);
      Ti[j * ld + c] = (a0 + a1) * inv;
    }
  __syncthreads();
  for (int idx = tid; idx < nc * nc; idx += blockDim.x) {
    int a = idx / nc, b = idx - a * nc;
    T[idx] = Ti[a * ld + b];
  }
}

__global__ void __launch_bounds__(1024) k_chol_drop(const double* __restrict__ G, int nc,
                                                    const double* __restrict__ norm0sq, double drop2,
                                                    double* __restrict__ T, int* __restrict__ keep) {
  extern __shared__ double smd[];
  __shared__ int kj;
  __shared__ double dj;
  chol_drop_cta(G, nc, norm0sq, drop2, T, keep, smd, kj, dj);
}

// |v| as an ordered integer without its low byte, row i (< 256) there instead: the
// maximum over rows is a pivot within 2^-12 of the largest element.
__device__ __forceinline__ unsigned pivot_key(float v, int i) {
  return (__float_as_uint(fabsf(v)) & ~255u) | (unsigned)(255 - i);
}
__device__ __forceinline__ unsigned pivot_key(double v, int i) {
  return ((unsigned)__double2hiint(fabs(v)) & ~255u) | (unsigned)(255 - i);
}

// Gaussian elimination with partial pivoting on the augmented matrix [M | b]
// held in shared memory (n rows, row stride ld >= n + 1, compute type T), then
// back substitution; the solution replaces column n (in the original row order).
// Rows are not moved: ord[] (shared, >= n ints) records the pivot rows.  Called by
// all threads of the CTA (two warps or more).
//
// What bounds a step is its chain: update of the next column, pivot, reciprocal,
// multipliers (700 clocks in FP64).  So warp 0 goes through it for step k + 1 while
// the other warps form the rest of step k's update, one barrier a step.  (With the
// chain between two barriers, FP64, or inside the update, FP32, the mean launch of
// the FP64 inner solves, n up to 60, took 68 us, 52 now; of the paired FP32 solves,
// n up to 120, 66 and 46.)
template <typename T>
__device__ void lu_solve_smem(T* A, int ld, int n, int* ord, T* y) {
  __shared__ T pinv[kSmallMax];             // reciprocal pivots
  __shared__ T mult[2][kSmallMax];          // multipliers of steps k, k + 1
  __shared__ int act[2][kSmallMax];         // their rows (not yet pivots)
  __shared__ unsigned recip[kSmallMax + 2]; // ceil(2^32 / w): e / w = __umulhi(e, recip[w]) for e w < 2^32
  constexpr int R = (kSmallMax + 31) / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  if constexpr (sizeof(T) == 8)
    for (int w = 2 + tid; w <= n; w += blockDim.x) recip[w] = 0xffffffffu / (unsigned)w + 1u;
  // warp 0: column k of the rows in list `from` (m of them; subtract: step k - 1's
  // update first), its pivot and multipliers, the rows left in list `to`
  auto pivot = [&](int k, int m, const int* from, int* to, const T* l, T* lnext, bool subtract) {
    T v[R];
    int row[R];
    unsigned best = 0u;
    const T pk = subtract ? A[ord[k - 1] * ld + k] : T(0);
#pragma unroll
    for (int t = 0; t < R; ++t) {
      const int e = t * 32 + lane;
      if (e < m) {
        row[t] = from ? from[e] : e;
        T* q = A + row[t] * ld + k;
        v[t] = *q;
        if (subtract) {
          v[t] -= l[e] * pk;
          *q = v[t];
        }
        best = max(best, pivot_key(v[t], row[t]));
      }
    }
    best = __reduce_max_sync(0xffffffffu, best);
    const int bi = 255 - (int)(best & 255u);
    // the pivot's place in the list and its value
    int at = -1;
    T piv = T(0);
#pragma unroll
    for (int t = 0; t < R; ++t) {
      const bool hit = t * 32 + lane < m && row[t] == bi;
      const unsigned who = __ballot_sync(0xffffffffu, hit);
      if (who) {
        const int src = __ffs(who) - 1;
        at = t * 32 + src;
        piv = __shfl_sync(0xffffffffu, v[t], src);
      }
    }
    if (piv == T(0)) piv = T(1e-30);
    const T inv = fast_rcp(piv);
    if (lane == 0) {
      ord[k] = bi;
      pinv[k] = inv;
    }
    // the last row of the list takes the pivot's place
#pragma unroll
    for (int t = 0; t < R; ++t) {
      const int e = t * 32 + lane;
      if (e < m && e != at) {
        const int o = e == m - 1 ? at : e;
        lnext[o] = v[t] * inv;
        to[o] = row[t];
      }
    }
  };
  __syncthreads();
  if (warp == 0) pivot(0, n, nullptr, act[0], nullptr, mult[0], false);
  for (int k = 0; k + 1 < n; ++k) {
    __syncthreads();
    const int m = n - k - 1;
    const int* rows = act[k & 1];
    const T* l = mult[k & 1];
    if (warp == 0) {
      pivot(k + 1, m, rows, act[(k + 1) & 1], l, mult[(k + 1) & 1], true);
    } else {
      const T* prow = A + ord[k] * ld;
      const int j0 = k + 2, w = n + 1 - j0;          // columns j0 .. n
      if constexpr (sizeof(T) == 4) {
        for (int t = warp - 1; t < m; t += nw - 1) {
          T* row = A + rows[t] * ld;
          const T lt = l[t];
          for (int j = j0 + lane; j <= n; j += 32) row[j] -= lt * prow[j];
        }
      } else {
        // the FP64 unit takes as long for one lane as for 32: the elements are dealt to
        // the lanes row after row
        const unsigned rw = recip[max(w, 2)];
        for (int e = tid - 32; e < m * w; e += blockDim.x - 32) {
          const int t = w > 1 ? (int)__umulhi((unsigned)e, rw) : e, j = j0 + e - t * w;
          T* row = A + rows[t] * ld;
          row[j] -= l[t] * prow[j];
        }
      }
    }
  }
  __syncthreads();
  // back substitution in blocks of 32 unknowns (see cta_trsv)
  for (int j0 = (n - 1) / 32 * 32; j0 >= 0; j0 -= 32) {
    const int jn = min(32, n - j0);
    if (warp == 0) {
      const T* row = A + (lane < jn ? ord[j0 + lane] : 0) * ld;
      T v = lane < jn ? row[n] : T(0);
      const T di = lane < jn ? pinv[j0 + lane] : T(0);
      for (int j = jn - 1; j >= 0; --j) {
        const T x = __shfl_sync(0xffffffffu, v * di, j);
        if (lane == j) v = x;
        else if (lane < j) v -= row[j0 + j] * x;
      }
      if (lane < jn) y[j0 + lane] = v;
    }
    __syncthreads();
    for (int r = tid; r < j0; r += blockDim.x) {
      T* row = A + ord[r] * ld;
      T acc = row[n];
#pragma unroll 4
      for (int j = 0; j < jn; ++j) acc -= row[j0 + j] * y[j0 + j];
      row[n] = acc;
    }
    __syncthreads();
  }
  for (int i = tid; i < n; i += blockDim.x) A[i * ld + n] = y[i];
  __syncthreads();
}

// One CTA per right-hand side r: Gaussian elimination with partial pivoting on
// [(H - sigma_r I) | b_r] in shared memory (compute type T), then back substitution.
template <typename T>
__global__ void __launch_bounds__(1024) k_lu_shift(const T* __restrict__ H, int ldh, int n,
                                                  const double* __restrict__ sig,
                                                  const T* __restrict__ B, T* __restrict__ Y) {
  extern __shared__ __align__(16) unsigned char lu_raw[];
  T* A = reinterpret_cast<T*>(lu_raw);
  const int ld = n + 2;
  __shared__ int perm[kSmallMax];
  __shared__ T yv[kSmallMax];
  const int r = blockIdx.x;
  const double sg = sig[r];
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int idx = tid; idx < n * (n + 1); idx += nth) {
    int i = idx / (n + 1), j = idx - i * (n + 1);
    T v;
    if (j < n) v = T(0.5) * (H[(long long)i * ldh + j] + H[(long long)j * ldh + i]) - (i == j ? T(sg) : T(0));
    else v = B[(long long)r * n + i];
    A[i * ld + j] = v;
  }
  __syncthreads();
  lu_solve_smem<T>(A, ld, n, perm, yv);
  for (int i = tid; i < n; i += nth) Y[(long long)r * n + i] = A[i * ld + n];
}

// Triangular solve by the CTA on a vector b[n] in shared memory with the lower
// factor L (row stride ldl): trans = 0: L x = b; 1: L^T x = b; dinv: 1 / L[j][j].
// Blocks of 32 unknowns: warp 0 solves one in registers (a shuffle per unknown),
// then all threads subtract its columns from the rest.
template <typename T>
__device__ void cta_trsv(const T* __restrict__ L, int ldl, int n, const T* dinv, T* b, int trans) {
  const int tid = threadIdx.x, lane = tid & 31;
  const int nb = (n + 31) / 32;
  for (int q = 0; q < nb; ++q) {
    const int j0 = (trans ? nb - 1 - q : q) * 32, jn = min(32, n - j0);
    if (tid < 32) {
      T v = lane < jn ? b[j0 + lane] : T(0);
      const T di = lane < jn ? dinv[j0 + lane] : T(0);
      for (int t = 0; t < jn; ++t) {
        const int j = trans ? jn - 1 - t : t;
        const T x = __shfl_sync(0xffffffffu, v * di, j);
        if (lane == j) v = x;
        else if (lane < jn && (trans ? lane < j : lane > j))
          v -= (trans ? L[(long long)(j0 + j) * ldl + j0 + lane] : L[(long long)(j0 + lane) * ldl + j0 + j]) * x;
      }
      if (lane < jn) b[j0 + lane] = v;
    }
    __syncthreads();
    const int r0 = trans ? 0 : j0 + jn, r1 = trans ? j0 : n;
    for (int r = r0 + tid; r < r1; r += blockDim.x) {
      T acc = b[r];
#pragma unroll 4
      for (int j = 0; j < jn; ++j)
        acc -= (trans ? L[(long long)(j0 + j) * ldl + r] : L[(long long)r * ldl + j0 + j]) * b[j0 + j];
      b[r] = acc;
    }
    __syncthreads();
  }
}

// The small part of one paired Galerkin iteration for system r (one CTA each),
// with a- = L L^T and H = L^T a+ L:
//   z = L^-1 h-,  rhs = L^T h+ + s z,  (H - s^2) u~ = rhs,  u = L u~,
//   w = L^-T (z + s u~)          (h- absent: z = 0)
template <typename T>
__global__ void __launch_bounds__(1024) k_paired_small(const T* __restrict__ Lg, const T* __restrict__ H,
                                                      int ld, int n, const T* __restrict__ hp,
                                                      const T* __restrict__ hm, const double* __restrict__ sh,
                                                      T* __restrict__ uc, T* __restrict__ wc) {
  extern __shared__ __align__(16) unsigned char ps_raw[];
  const int la = n + 2;
  T* A = reinterpret_cast<T*>(ps_raw);   // [n][n+2] augmented system
  T* z = A + (size_t)n * la;             // [n]
  T* hv = z + n;                         // [n]
  // FP32: a copy of L in shared memory (row stride n + 1, so that column walks
  // are free of bank conflicts); FP64 (too large): L read from global memory
  constexpr bool kLs = sizeof(T) == 4;
  if (kLs) {
    T* Ls = hv + n;
    for (int idx = threadIdx.x; idx < n * n; idx += blockDim.x) {
      const int r = idx / n, c = idx - r * n;
      Ls[r * (n + 1) + c] = Lg[(long long)r * ld + c];
    }
  }
  const T* L = kLs ? hv + n : Lg;
  const int ll = kLs ? n + 1 : ld;
  __shared__ int perm[kSmallMax];
  __shared__ T yv[kSmallMax], dinv[kSmallMax];
  const int r = blockIdx.x;
  const T s = (T)sh[r];
  const T s2 = (T)(sh[r] * sh[r]);
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int i = tid; i < n; i += nth) {
    z[i] = hm ? hm[(long long)r * n + i] : T(0);
    hv[i] = hp[(long long)r * n + i];
  }
  for (int idx = tid; idx < n * n; idx += nth) {
    int i = idx / n, j = idx - i * n;
    A[i * la + j] = T(0.5) * (H[(long long)i * ld + j] + H[(long long)j * ld + i]) - (i == j ? s2 : T(0));
  }
  __syncthreads();
  for (int i = tid; i < n; i += nth) dinv[i] = fast_rcp(L[(long long)i * ll + i]);
  __syncthreads();
  if (hm) cta_trsv<T>(L, ll, n, dinv, z, 0);
  for (int i = tid; i < n; i += nth) {   // rhs_i = sum_q h+_q L[q][i] + s z_i
    T acc = s * z[i];
    for (int q = i; q < n; ++q) acc += hv[q] * L[(long long)q * ll + i];
    A[i * la + n] = acc;
  }
  __syncthreads();
  lu_solve_smem<T>(A, la, n, perm, yv);
  // u = L u~ ; z <- z + s u~
  for (int i = tid; i < n; i += nth) {
    T acc = T(0);
    for (int q = 0; q <= i; ++q) acc += L[(long long)i * ll + q] * A[q * la + n];
    uc[(long long)r * n + i] = acc;
    hv[i] = z[i] + s * A[i * la + n];
  }
  __syncthreads();
  cta_trsv<T>(L, ll, n, dinv, hv, 1);
  for (int i = tid; i < n; i += nth) wc[(long long)r * n + i] = hv[i];
}

// ---- batched forms (one CTA per problem or per right-hand side), for many
// small independent solves advanced together

// Lowest k eigenpairs of the symmetric part of H (FP64 cyclic Jacobi in
// shared memory), ascending: lam[k], vec[k][n] (rows = eigenvectors).
__global__ void __launch_bounds__(512) k_beig(const BEig* __restrict__ d) {
  extern __shared__ double smb[];
  __shared__ int pp[kBatchSmall / 2 + 1], qq[kBatchSmall / 2 + 1];
  __shared__ double cc[kBatchSmall / 2 + 1], ss[kBatchSmall / 2 + 1];
  __shared__ unsigned smax;
  __shared__ double red[33];
  const BEig e = d[blockIdx.x];
  const int n = e.n;
  if (n <= 0) return;
  const int NP = (n + 1) & ~1, ld = NP + 1;
  double* A = smb;
  double* Q = smb + NP * ld;
  double f2 = 0.0;
  for (int idx = threadIdx.x; idx < NP * NP; idx += blockDim.x) {
    int r = idx / NP, c = idx - r * NP;
    double v = 0.0;
    if (r < n && c < n) v = 0.5 * (e.H[(long long)r * e.ld + c] + e.H[(long long)c * e.ld + r]);
    f2 += v * v;
    A[r * ld + c] = v;
    Q[r * ld + c] = (r == c) ? 1.0 : 0.0;
  }
  double frob = sqrt(block_sum(f2, red));
  jacobi_cta<double>(A, Q, n, ld, frob, 30, 1e-14, pp, qq, cc, ss, &smax);
  for (int t = threadIdx.x; t < n; t += blockDim.x) {
    int r = diag_rank(A, ld, n, t);
    if (r < e.k) {
      e.lam[r] = A[t * ld + t];
      for (int q = 0; q < n; ++q) e.vec[(long long)r * n + q] = Q[q * ld + t];
    }
  }
}

// y = (H - sigma I)^-1 b for one right-hand side per CTA (LU, partial pivoting).
__global__ void __launch_bounds__(512) k_blu(const BLu* __restrict__ d) {
  extern __shared__ __align__(16) unsigned char blu_raw[];
  double* A = reinterpret_cast<double*>(blu_raw);
  __shared__ int perm[kBatchSmall];
  __shared__ double yv[kBatchSmall];
  const BLu e = d[blockIdx.x];
  const int n = e.n;
  if (n <= 0) return;
  const int ld = n + 2;
  for (int idx = threadIdx.x; idx < n * (n + 1); idx += blockDim.x) {
    int i = idx / (n + 1), j = idx - i * (n + 1);
    double v;
    if (j < n) v = 0.5 * (e.H[(long long)i * e.ld + j] + e.H[(long long)j * e.ld + i]) - (i == j ? e.sigma : 0.0);
    else v = e.b[i];
    A[i * ld + j] = v;
  }
  __syncthreads();
  lu_solve_smem<double>(A, ld, n, perm, yv);
  for (int i = threadIdx.x; i < n; i += blockDim.x) e.y[i] = A[i * ld + n];
}

__global__ void __launch_bounds__(1024) k_bdrop(const BDrop* __restrict__ d, double drop2) {
  extern __shared__ double smd[];
  __shared__ int kj;
  __shared__ double dj;
  const BDrop e = d[blockIdx.x];
  if (e.nc <= 0) return;
  chol_drop_cta(e.G, e.nc, e.norm0sq, drop2, e.T, e.keep, smd, kj, dj);
}

void set_smem(const void* f, size_t bytes) {
  ensure_smem(f, bytes);
}

}  // namespace

void eig32(const double* H, int ldh, int n, float* lam32, float* vec32, cudaStream_t s) {
  TD_REQUIRE(n >= 1 && n <= kSmallMax, TDDFT_ERR_ARG, "eig32: size out of range");
  const int NP = (n + 1) & ~1, half = NP / 2;
  const size_t smem = (size_t)NP * (NP + 1) * sizeof(float);
  set_smem((const void*)k_jacobi_a, smem);
  DevBuf work(kJacBytes, s);
  float2* rot = work.as<float2>();
  int* info = reinterpret_cast<int*>(rot + kJacRounds * kJacHalf);
  k_jacobi_a<<<1, 1024, smem, s>>>(H, ldh, n, lam32, rot, info);
  const int grid = (n + kJacRows - 1) / kJacRows;
  if (half <= 32) k_jacobi_q<1><<<grid, 32 * kJacRows, 0, s>>>(n, rot, info, vec32);
  else if (half <= 64) k_jacobi_q<2><<<grid, 32 * kJacRows, 0, s>>>(n, rot, info, vec32);
  else k_jacobi_q<3><<<grid, 32 * kJacRows, 0, s>>>(n, rot, info, vec32);
  count_launch(2);
  TD_LAUNCH_CHECK();
}

void refine_lowest(const double* H, int ldh, int n, int k, const float* lam32, const float* vec32,
                   double* lam, double* vecs, double* scratch, int rounds, cudaStream_t s) {
  TD_REQUIRE(k >= 1 && k <= n && k <= kWantMax, TDDFT_ERR_ARG, "refine_lowest: bad k");
  double* Qk = scratch;
  double* Yk = scratch + (size_t)k * n;
  k_refine<<<k, 256, 0, s>>>(H, ldh, n, lam32, vec32, rounds, Qk, Yk);
  count_launch();
  TD_LAUNCH_CHECK();
  const int KP = (k + 1) & ~1;
  size_t smem = (size_t)2 * KP * (KP + 1) * sizeof(double);
  set_smem((const void*)k_orth_rr, smem);
  k_orth_rr<<<1, 1024, smem, s>>>(Qk, Yk, k, n, lam, vecs);
  count_launch();
  TD_LAUNCH_CHECK();
}

void shifted_solve(const double* H, int ldh, int n, const float* lam32, const float* vec32,
                   const double* sigma, int nr, const double* B, double* Y, int nref,
                   cudaStream_t s) {
  if (nr <= 0) return;
  k_shifted<<<nr, 256, 0, s>>>(H, ldh, n, lam32, vec32, sigma, B, Y, nref);
  count_launch();
  TD_LAUNCH_CHECK();
}

template <typename S>
void lu_shift_solve(const S* H, int ldh, int n, const double* sigma, int nr, const S* B, S* Y,
                    cudaStream_t s) {
  if (nr <= 0) return;
  TD_REQUIRE(n >= 1 && n <= kSmallMax, TDDFT_ERR_ARG, "lu_shift_solve: size out of range");
  size_t smem = (size_t)n * (n + 2) * sizeof(S);
  set_smem((const void*)k_lu_shift<S>, smem);
  k_lu_shift<S><<<nr, sizeof(S) == 4 ? 1024 : 512, smem, s>>>(H, ldh, n, sigma, B, Y);
  count_launch();
  TD_LAUNCH_CHECK();
}
template void lu_shift_solve<float>(const float*, int, int, const double*, int, const float*, float*,
                                    cudaStream_t);
template void lu_shift_solve<double>(const double*, int, int, const double*, int, const double*, double*,
                                     cudaStream_t);

template <typename S>
void paired_small_solve(const S* L, const S* H, int ld, int n, const S* hp, const S* hm, const double* sh,
                        int nr, S* uc, S* wc, cudaStream_t s) {
  if (nr <= 0) return;
  TD_REQUIRE(n >= 1 && n <= kSmallMax, TDDFT_ERR_ARG, "paired_small_solve: size out of range");
  size_t smem = ((size_t)n * (n + 2) + 2 * (size_t)n + (sizeof(S) == 4 ? (size_t)n * (n + 1) : 0)) * sizeof(S);
  set_smem((const void*)k_paired_small<S>, smem);
  k_paired_small<S><<<nr, sizeof(S) == 4 ? 1024 : 512, smem, s>>>(L, H, ld, n, hp, hm, sh, uc, wc);
  count_launch();
  TD_LAUNCH_CHECK();
}
template void paired_small_solve<float>(const float*, const float*, int, int, const float*, const float*,
                                        const double*, int, float*, float*, cudaStream_t);
template void paired_small_solve<double>(const double*, const double*, int, int, const double*,
                                         const double*, const double*, int, double*, double*, cudaStream_t);

template <typename S>
void cholesky(S* H, int ldh, int n, int* info, cudaStream_t s) {
  TD_REQUIRE(n >= 1 && n <= kSmallMax, TDDFT_ERR_ARG, "cholesky: size out of range");
  size_t smem = (size_t)n * (n + 1) * sizeof(S);
  set_smem((const void*)k_cholesky<S>, smem);
  k_cholesky<S><<<1, 1024, smem, s>>>(H, ldh, n, info);
  count_launch();
  TD_LAUNCH_CHECK();
}
template void cholesky<float>(float*, int, int, int*, cudaStream_t);

template <typename S>
void cholesky_border(S* L, int ld, int n0, int n, int* info, cudaStream_t s) {
  TD_REQUIRE(n >= 1 && n <= kSmallMax && n0 >= 0 && n0 <= n, TDDFT_ERR_ARG, "cholesky_border: bad sizes");
  const size_t smem = (size_t)n * (n | 1) * sizeof(S);
  ensure_smem((const void*)k_chol_border<S>, smem);
  k_chol_border<S><<<1, 1024, smem, s>>>(L, ld, n0, n, info);
  count_launch();
  TD_LAUNCH_CHECK();
}
template void cholesky_border<float>(float*, int, int, int, int*, cudaStream_t);
template void cholesky_border<double>(double*, int, int, int, int*, cudaStream_t);
template void cholesky<double>(double*, int, int, int*, cudaStream_t);

template <typename S>
void trsv_rows(const S* L, int ldl, int n, S* B, int nr, int trans, cudaStream_t s) {
  if (nr <= 0) return;
  TD_REQUIRE(n <= kSmallMax, TDDFT_ERR_ARG, "trsv: size out of range");
  k_trsv<S><<<nr, 256, 0, s>>>(L, ldl, n, B, trans);
  count_launch();
  TD_LAUNCH_CHECK();
}
template void trsv_rows<float>(const float*, int, int, float*, int, int, cudaStream_t);
template void trsv_rows<double>(const double*, int, int, double*, int, int, cudaStream_t);

void batch_eig(const BEig* d, int nb, int nmax, cudaStream_t s) {
  if (nb <= 0) return;
  TD_REQUIRE(nmax >= 1 && nmax <= kBatchSmall, TDDFT_ERR_ARG, "batch_eig: size out of range");
  const int NP = (nmax + 1) & ~1;
  const size_t smem = (size_t)2 * NP * (NP + 1) * sizeof(double);
  set_smem((const void*)k_beig, smem);
  k_beig<<<nb, 512, smem, s>>>(d);
  count_launch();
  TD_LAUNCH_CHECK();
}

void batch_lu(const BLu* d, int nr, int nmax, cudaStream_t s) {
  if (nr <= 0) return;
  TD_REQUIRE(nmax >= 1 && nmax <= kBatchSmall, TDDFT_ERR_ARG, "batch_lu: size out of range");
  const size_t smem = (size_t)nmax * (nmax + 2) * sizeof(double);
  set_smem((const void*)k_blu, smem);
  k_blu<<<nr, 512, smem, s>>>(d);
  count_launch();
  TD_LAUNCH_CHECK();
}

void batch_chol_drop(const BDrop* d, int nb, int ncmax, double drop2, cudaStream_t s) {
  if (nb <= 0) return;
  TD_REQUIRE(ncmax >= 1 && ncmax <= kBatchSmall, TDDFT_ERR_ARG, "batch_chol_drop: size out of range");
  const size_t smem = (size_t)2 * ncmax * (ncmax + 1) * sizeof(double);
  set_smem((const void*)k_bdrop, smem);
  k_bdrop<<<nb, 1024, smem, s>>>(d, drop2);
  count_launch();
  TD_LAUNCH_CHECK();
}

void chol_drop(const double* G, int nc, const double* norm0sq, double drop2, double* T, int* keep,
               cudaStream_t s) {
  TD_REQUIRE(nc >= 1 && nc <= kDropMax, TDDFT_ERR_ARG, "chol_drop: too many candidates");
  size_t smem = (size_t)2 * nc * (nc + 1) * sizeof(double);
  set_smem((const void*)k_chol_drop, smem);
  k_chol_drop<<<1, 256, smem, s>>>(G, nc, norm0sq, drop2, T, keep);
  count_launch();
  TD_LAUNCH_CHECK();
}

}  // namespace tddft
