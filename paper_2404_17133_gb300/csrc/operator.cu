// On-the-fly response products over density-fitted factors (Eq. hessian with
// (pq|rs) = sum_P L^P_pq L^P_rs, Eq. pqrs_approx):
//   A X     = Delta X + c_J J(X) - a_x K1(X)                      (Eq. TDA)
//   (A+B) X = Delta X + 2 c_J J(X) - a_x (K1(X) + K2(X))
//   (A-B) X = Delta X + a_x (K2(X) - K1(X))
// with J(X)_ia = sum_jb (ia|jb) X_jb, K1(X)_ib = sum_ja (ij|ab) X_ja,
// K2(X)_ia = sum_jb (ib|ja) X_jb.  The four-index integrals are never formed;
// each term is a pair of contractions over P:
//   J : t[P][n] = sum_ia L_ov[P][ia] X[n][ia];  J[n][ia] = sum_P t[P][n] L_ov[P][ia]
//   K1: Z[n][i][P][a] = sum_j L_oo[P][i][j] X[n][j][a]   (batched over P, n)
//       K1[(n,i)][b] = sum_(P,a) Z[(n,i)][(P,a)] L_vv[P][a][b]   (one tall-K GEMM)
//   K2: Q[n][i][P][j] = sum_b L_ov[P][i][b] X[n][j][b]
//       K2[(n,i)][a] = sum_(P,j) Q[(n,i)][(P,j)] L_ov[P][j][a]
// P is processed in chunks so the intermediates stay within a bounded
// workspace; the contractions of K1 and K2 (most of the flops) run on the tcgen05
// tensor cores: as FP16 hi + lo operands when asked (MIXED with tensor_cores,
// tc_gemm.cuh), else as exact slices of the FP64 or FP32 operands
// (slice_gemm.cuh).  Without tensor_cores, BF16 ris rows against FP32 vectors and
// small products run on the FP32 or FP64 units.
#include <algorithm>
#include <cmath>

#include "ctx.cuh"
#include "skinny.cuh"
#include "slice_gemm.cuh"
#include "tc_gemm.cuh"
#include "vecops.cuh"

namespace tddft {

namespace {
cudaEvent_t take_event(std::vector<cudaEvent_t>& spare) {
  cudaEvent_t e;
  if (!spare.empty()) {
    e = spare.back();
    spare.pop_back();
  } else {
    TD_CUDA(cudaEventCreate(&e));
  }
  return e;
}
}  // namespace

void KernelProfile::begin(cudaStream_t s) {
  cudaEvent_t a = take_event(spare);
  ev.push_back(a);
  TD_CUDA(cudaEventRecord(a, s));
}
void KernelProfile::end(cudaStream_t s, double launch_flops, double launch_bytes) {
  cudaEvent_t b = take_event(spare);
  ev.push_back(b);
  TD_CUDA(cudaEventRecord(b, s));
  pend_flops.push_back(launch_flops);
  pend_bytes.push_back(launch_bytes);
  launches++;
  flops += launch_flops;
}
void KernelProfile::reserve(size_t n_events) {
  while (spare.size() < n_events) {
    cudaEvent_t e;
    TD_CUDA(cudaEventCreate(&e));
    spare.push_back(e);
  }
}
void KernelProfile::collect() {
  for (size_t i = 0; i + 1 < ev.size(); i += 2) {
    TD_CUDA(cudaEventSynchronize(ev[i + 1]));
    float t = 0.f;
    TD_CUDA(cudaEventElapsedTime(&t, ev[i], ev[i + 1]));
    ms += t;
    if (rec_ms.size() < kMaxRecords) {
      rec_ms.push_back(t);
      rec_flops.push_back(pend_flops[i / 2]);
      rec_bytes.push_back(pend_bytes[i / 2]);
    }
  }
  spare.insert(spare.end(), ev.begin(), ev.end());   // recorded and waited on: reusable
  ev.clear();
  pend_flops.clear();
  pend_bytes.clear();
}
void KernelProfile::reset() {
  for (auto e : ev) cudaEventDestroy(e);   // possibly still pending: not reused
  ev.clear();
  pend_flops.clear();
  pend_bytes.clear();
  rec_ms.clear();
  rec_flops.clear();
  rec_bytes.clear();
  launches = 0;
  flops = 0.0;
  ms = 0.0;
}
KernelProfile::~KernelProfile() {
  for (auto e : spare) cudaEventDestroy(e);
  for (auto e : ev) cudaEventDestroy(e);
}

namespace {
// Exchange intermediates of one P-chunk: SIMT contractions (BF16 ris rows) keep
// them within 512 MB; the tensor-core path takes 4 GB, so that a contraction launch covers
// many auxiliary rows (longer K loops per CTA, fewer launches and pipeline fills).
constexpr size_t kChunkBytes = 512ull << 20;
constexpr size_t kChunkBytesTC = 4ull << 30;
// The sliced contractions (slice_gemm.cuh) keep Z and Q, their slices and the
// factors' slices of a chunk: 1 GB in all.
constexpr size_t kChunkBytesSliced = 1ull << 30;
// Multiply-adds per FP64 Coulomb contraction from which it is sliced, too; below, the
// launches and the cutting of L_ov cost what the FP64 units do (whole product, units
// and slices: 60 x 400 with 360 rows, 2 vectors, 2^24.0 1.61 and 1.61 ms; 24 x 144 with 840
// rows, 13 vectors, 2^25.2 1.58 and 1.59, 40 vectors, 2^26.8 3.87 and 3.54; 60 x 400 with 2000
// rows, 1 vector, 2^25.5 6.89 and 6.43, 6 vectors, 2^28.1 15.8 and 15.0).
constexpr double kCoulombSliced = 1 << 25;
// Multiply-adds of the exchange contractions from which these are sliced; below, the
// FP64 (FP32) units need fewer launches.  Products of A, units and slices, us: FP64 6 x 30
// with 180 rows, 4 vectors (2^22.1) 143 and 174, 20 vectors (2^24.5) 743 and 189; 5 x 20,
// 20 vectors (2^22.6) 206 and 187; FP32 12 x 60 with 360 rows, 8 vectors (2^27.1) 209 and
// 210, 20 vectors (2^28.5) 267 and 248; 16 x 90 with 500 rows, 4 vectors (2^28.2) 235 and 264.
constexpr double kExchangeSliced64 = 1 << 22, kExchangeSliced32 = 1 << 28;
// k-blocks one CTA accumulates in FP32 before its split-K partial is summed
// (fixed order) with the others: the rounding of an FP32 run grows with its
// length, and runs over a whole P-chunk of the exchange contraction (~1e4 MMA
// steps) left the large Casida solve's recomputed residuals 3e-6 above the
// loop's.  Exchange: 256 k-blocks (16384 terms); the Coulomb term's J = t^T
// L_ov (K = n_aux): 16.
constexpr int kExchangeKb = 256;
constexpr int kCoulombKb = 16;

int chunk_rows(int nrows, long long per_row_bytes, int m, size_t budget = kChunkBytes) {
  long long pc = (long long)(budget / (per_row_bytes > 0 ? per_row_bytes : 1));
  if (pc < 1) pc = 1;
  if (pc > nrows) pc = nrows;
  long long bmax = 65535 / (m > 0 ? m : 1);
  if (pc > bmax) pc = bmax;
  return (int)(pc < 1 ? 1 : pc);
}
}  // namespace

void raise_tc_error(int code, int* word, cudaStream_t s) {
  if (code == 0) return;
  TD_CUDA(cudaMemsetAsync(word, 0, 4, s));
  throw Error(TDDFT_ERR_CUDA, "tensor-core kernel wait timed out (code " + std::to_string(code) + ")");
}

void check_tc_error(Ctx& c) {
  int h = 0;
  TD_CUDA(cudaMemcpyAsync(&h, c.tc_err.p, 4, cudaMemcpyDeviceToHost, c.s));
  TD_CUDA(cudaStreamSynchronize(c.s));
  raise_tc_error(h, c.tc_err.as<int>(), c.s);
}

// An operand of the sliced contractions with room for its slices.
struct SliceCut {
  SliceOperand o;
  DevBuf parts, info;
  void alloc(cudaStream_t st) {
    parts = DevBuf(slice_bytes(o), st);
    info = DevBuf(slice_info_bytes(o), st);
  }
  void cut(cudaStream_t st) { slice_cut(o, parts.p, info.p, st); }
};
static SliceCut slice_operand(const void* p, DType t, int rows, int np, int K) {
  SliceCut c;
  c.o.p = p;
  c.o.t = t;
  c.o.rows = rows;
  c.o.np = np;
  c.o.K = K;
  return c;
}

// J = (t^T L_ov) with t = L_ov X^T of an FP64 factor set by exact slicing.  Both are
// chunked over the rows of the first operand (P; ia), so nothing is accumulated.
static void coulomb_sliced(const OpDims& d, const FactorSet& f, const double* X, int m, double* J, cudaStream_t s) {
  const int ov = d.ov;
  const double* L = static_cast<const double*>(f.Jov);
  const long long sb = slice_element_bytes(DType::F64);
  DevBuf t((size_t)f.nJ * m * 8, s);
  {
    SliceCut x = slice_operand(X, DType::F64, m, 1, ov);
    x.o.rs0 = ov; x.o.p_outer = true;
    x.alloc(s);
    x.cut(s);
    const int pc = chunk_rows(f.nJ, tc_pad(ov) * sb, 1, kChunkBytesSliced);
    SliceCut l = slice_operand(L, DType::F64, pc, 1, ov);
    l.o.rs0 = ov;
    l.alloc(s);
    for (int p0 = 0; p0 < f.nJ; p0 += pc) {
      l.o.p = L + (long long)p0 * ov;
      l.o.rows = std::min(pc, f.nJ - p0);
      l.cut(s);
      slice_gemm(l.o, l.parts.p, l.info.p, x.o, x.parts.p, x.info.p, t.as<double>() + (long long)p0 * m, 0.0, d.tc_err, s);
    }
  }
  SliceCut tt = slice_operand(t.p, DType::F64, m, 1, f.nJ);
  tt.o.rs0 = 1; tt.o.ks = m; tt.o.p_outer = true;
  tt.alloc(s);
  tt.cut(s);
  const int cc = chunk_rows(ov, tc_pad(f.nJ) * sb, 1, kChunkBytesSliced);
  SliceCut l = slice_operand(L, DType::F64, cc, 1, f.nJ);
  l.o.rs0 = 1; l.o.ks = ov;
  l.alloc(s);
  for (int c0 = 0; c0 < ov; c0 += cc) {
    l.o.p = L + c0;
    l.o.rows = std::min(cc, ov - c0);
    l.cut(s);
    slice_gemm_scatter(l.o, l.parts.p, l.info.p, tt.o, tt.parts.p, tt.info.p, J + c0, SliceScatter{1 << 30, 1 << 30, 0, ov, 0},
                       d.tc_err, s);
  }
}

// K1 (and K2) of an FP64 or FP32 factor set, every contraction on the tensor cores
// by exact slicing (slice_gemm.cuh): no FP64 or FP32 vector arithmetic beyond
// the cuts.  Xw: trial vectors in the factors' type.
static void exchange_sliced(const OpDims& d, const FactorSet& f, const void* Xw, int m, bool need_k2, void* K1,
                            void* K2, cudaStream_t s) {
  const int no = d.no, nv = d.nv, ov = d.ov;
  const DType t = f.dt;
  const size_t es = dtype_size(t), sb = (size_t)slice_element_bytes(t);
  const size_t nop = tc_pad(no), nvp = tc_pad(nv);
  const size_t per_row = (size_t)m * no * (nv * es + nvp * sb) + (no * nop + nv * nvp) * sb +
                         (need_k2 ? (size_t)m * no * (no * es + nop * sb) + (no * nvp + nv * nop) * sb : 0);
  const int pc = chunk_rows(f.nK, (long long)per_row, 1, kChunkBytesSliced);
  auto operand = [&](const void* p, int rows, int np, int K) { return slice_operand(p, t, rows, np, K); };
  // X^T per vector: rows (n, a), k = j; X: rows (n, j), k = b
  SliceCut xt = operand(Xw, m * nv, 1, no), xs = operand(Xw, m * no, 1, nv);
  xt.o.R = nv; xt.o.rs1 = ov; xt.o.rs0 = 1; xt.o.ks = nv;
  xt.alloc(s);
  xt.cut(s);
  if (need_k2) {
    xs.o.rs0 = nv;
    xs.alloc(s);
    xs.cut(s);
  }
  DevBuf Zb((size_t)m * no * pc * nv * es, s), Qb;
  if (need_k2) Qb = DevBuf((size_t)m * no * pc * no * es, s);
  // chunk operands, allocated for the first (largest) chunk
  SliceCut oo = operand(nullptr, pc * no, 1, no), vv = operand(nullptr, nv, pc, nv), z = operand(Zb.p, m * no, pc, nv);
  SliceCut ov_ = operand(nullptr, pc * no, 1, nv), vo = operand(nullptr, nv, pc, no), q = operand(Qb.p, m * no, pc, no);
  oo.o.rs0 = no; oo.o.p_outer = true;
  vv.o.rs0 = nv; vv.o.ps = (long long)nv * nv; vv.o.p_outer = true;
  z.o.ps = nv;
  ov_.o.rs0 = nv; ov_.o.p_outer = true;
  vo.o.rs0 = 1; vo.o.ks = nv; vo.o.ps = ov; vo.o.p_outer = true;
  q.o.ps = no;
  oo.alloc(s);
  vv.alloc(s);
  z.alloc(s);
  if (need_k2) {
    ov_.alloc(s);
    vo.alloc(s);
    q.alloc(s);
  }
  for (int p0 = 0; p0 < f.nK; p0 += pc) {
    const int pn = (f.nK - p0 < pc) ? f.nK - p0 : pc;
    const double beta = p0 > 0 ? 1.0 : 0.0;
    // Z[n][i][P][a] = sum_j Koo[P][i][j] X[n][j][a]
    oo.o.p = (const char*)f.Koo + (size_t)p0 * no * no * es;
    oo.o.rows = pn * no;
    oo.cut(s);
    slice_gemm_scatter(xt.o, xt.parts.p, xt.info.p, oo.o, oo.parts.p, oo.info.p, Zb.p,
                       SliceScatter{nv, no, (long long)no * pn * nv, (long long)pn * nv, nv}, d.tc_err, s);
    z.o.rs0 = (long long)pn * nv;
    z.o.np = pn;
    z.cut(s);
    vv.o.p = (const char*)f.Kvv + (size_t)p0 * nv * nv * es;
    vv.o.np = pn;
    vv.cut(s);
    const bool timed = d.prof_simt && d.prof_simt->on;
    if (timed) d.prof_simt->begin(s);
    slice_gemm(z.o, z.parts.p, z.info.p, vv.o, vv.parts.p, vv.info.p, K1, beta, d.tc_err, s);
    if (timed)
      d.prof_simt->end(s, 2.0 * m * no * (double)nv * (double)pn * nv,
                       (double)es * ((double)m * no * pn * nv + (double)pn * nv * nv +
                                     (double)m * no * nv * (p0 > 0 ? 2.0 : 1.0)));
    if (need_k2) {
      // Q[n][i][P][j] = sum_b Kov[P][i][b] X[n][j][b]
      ov_.o.p = (const char*)f.Kov + (size_t)p0 * ov * es;
      ov_.o.rows = pn * no;
      ov_.cut(s);
      slice_gemm_scatter(xs.o, xs.parts.p, xs.info.p, ov_.o, ov_.parts.p, ov_.info.p, Qb.p,
                         SliceScatter{no, no, (long long)no * pn * no, (long long)pn * no, no}, d.tc_err, s);
      q.o.rs0 = (long long)pn * no;
      q.o.np = pn;
      q.cut(s);
      vo.o.p = ov_.o.p;
      vo.o.np = pn;
      vo.cut(s);
      slice_gemm(q.o, q.parts.p, q.info.p, vo.o, vo.parts.p, vo.info.p, K2, beta, d.tc_err, s);
    }
  }
}

// A term of the final combination: the partial sums that its contraction left (one
// P-chunk covers the factor set), else the summed term b, if there is one.
static SumTerm term_of(const TcSum& k, const DevBuf& b) {
  SumTerm t;
  if (k.splits) {
    t.part = k.part.as<float>();
    t.splits = k.splits;
    t.scale = k.scale;
  } else if (b.p) {
    t.part = b.as<float>();
    t.splits = 1;
  }
  return t;
}

// Hi and lo parts of Z and Q for pc rows of a chunk (elements of es bytes in rows of nvz and
// noz; noz = 0: no Q), in one allocation where the stream's cache takes it: on a fresh stream
// each of megabytes costs 40 us.
struct StageParts {
  DevBuf buf[4];
  unsigned char *z[2], *q[2];
  StageParts(int m, int no, int pc, int nvz, int noz, int es, cudaStream_t s) {
    const size_t rows = (size_t)m * no * pc, zb = rows * nvz * es, qb = rows * noz * es;   // whole 128-byte lines
    if (2 * (zb + qb) <= kCacheMax) {
      buf[0] = DevBuf(2 * (zb + qb), s);
      z[0] = buf[0].as<unsigned char>();
      z[1] = z[0] + zb;
      q[0] = z[1] + zb;
      q[1] = q[0] + qb;
      return;
    }
    for (int k = 0; k < 4; ++k)
      if (k < 2 || qb) buf[k] = DevBuf(k < 2 ? zb : qb, s);
    for (int k = 0; k < 2; ++k) {
      z[k] = buf[k].as<unsigned char>();
      q[k] = buf[2 + k].as<unsigned char>();
    }
  }
};

// Operand forms of the trial vectors for the tensor-core exchange contractions,
// with their scales, in one allocation.
struct XParts {
  DevBuf buf;
  void *th = nullptr, *tl = nullptr, *sh = nullptr, *sl = nullptr;   // X^T per vector, X: hi + lo
  const float* sc = nullptr;   // tc_f16_product_scales or tc_fp8_scales block
};
static bool tc_exchange(const FactorSet& f, bool f64, bool tensor_cores) {
  return tensor_cores && !f64 && f.Kvv_hi && f.Kvo_hi && f.Koo_hi && f.Kovp_hi;
}
// scratch: five zeroed device words; xw: FP32 copy of X to write, or NULL
static XParts make_x_parts(const OpDims& d, const FactorSet& f, const void* X, DType xt, int m, bool paired,
                           unsigned* scratch, float* xw, cudaStream_t s) {
  const int no = d.no, nv = d.nv;
  const bool f16 = f.tc_elt == TcElt::F16;
  TD_REQUIRE(!f.fp8 || (f.Kvv8 && f.Kvo8 && f.s_vv), TDDFT_ERR_ARG, "FP8 ris copies missing");
  TD_REQUIRE(!f16 || (f.Kvv_lo && f.Kvo_lo && f.Koo_lo && f.Kovp_lo && f.tc_scale), TDDFT_ERR_ARG,
             "FP16 factor parts missing");
  auto pad = [](size_t b) { return (b + 255) & ~(size_t)255; };
  const size_t bt = pad((size_t)m * nv * tc_pad(no) * 2), bs = paired ? pad((size_t)m * no * tc_pad(nv) * 2) : 0;
  XParts x;
  x.buf = DevBuf(2 * bt + 2 * bs + (f.fp8 ? (size_t)(2 + 2 * f.nK) * 4 : 32), s);
  char* b = x.buf.as<char>();
  x.th = b;
  x.tl = b + bt;
  if (paired) {
    x.sh = b + 2 * bt;
    x.sl = b + 2 * bt + bs;
  }
  float* sc = reinterpret_cast<float*>(b + 2 * bt + 2 * bs);
  x.sc = sc;
  const bool scaled = f.fp8 || f16;
  if (f.fp8)
    tc_fp8_scales(X, xt, m, no, nv, f.s_vv, f.rho_oo, f.s_vo, f.rho_ov, f.nK, sc, scratch, xw, s);
  else if (f16)
    tc_f16_product_scales(X, xt, m, no, nv, f.tc_scale, sc, scratch, xw, s);
  tc_x_split(X, xt, m, no, nv, f.tc_elt, f16 ? sc : nullptr, x.th, x.tl, x.sh, x.sl, scaled ? nullptr : xw, s);
  return x;
}

template <typename TX>
static void apply_operator_t(const OpDims& d, const FactorSet& f, const TX* X, int m, OpMode mode,
                             TX* out0, TX* out1, int tc, cudaStream_t s) {
  const bool tensor_cores = tc != 0;
  if (m <= 0) return;
  const int no = d.no, nv = d.nv, ov = d.ov;
  const bool f64 = (f.dt == DType::F64);
  const DType tw = f64 ? DType::F64 : DType::F32;  // working / accumulation type
  const size_t ew = dtype_size(tw);
  const long long mov = (long long)m * ov;
  constexpr bool x32 = sizeof(TX) == 4;
  TD_REQUIRE(!(x32 && f64), TDDFT_ERR_ARG, "FP32 vectors need FP32/BF16 factors");

  const void* Xw = X;
  const DType xt = x32 ? DType::F32 : DType::F64;
  const bool need_k2 = (mode == OpMode::PAIRED);
  const bool main_x = f.nK > 0 && d.a_x != 0.0;
  const bool lr_x = f.lr && f.b_x != 0.0 && f.lr->nK > 0;
  DevBuf xbuf, words;
  XParts xp;
  if (tensor_cores && !f64) {
    words = DevBuf(5 * 4, s);   // [4]: max |t|
    TD_CUDA(cudaMemsetAsync(words.p, 0, 5 * 4, s));
  }
  const bool cast = !f64 && !x32;
  if (cast) {
    xbuf = DevBuf(mov * 4, s);
    Xw = xbuf.p;
  }
  // the pass that prepares the exchange operands writes the FP32 copy too
  if (main_x && tc_exchange(f, f64, tensor_cores))
    xp = make_x_parts(d, f, X, xt, m, need_k2, words.as<unsigned>(), cast ? xbuf.as<float>() : nullptr, s);
  else if (cast)
    cast_f64_to_f32(reinterpret_cast<const double*>(X), xbuf.as<float>(), mov, s);

  // ---- Coulomb (and the low-rank kernel term, which enters with the same prefactor)
  DevBuf Jb;
  TcSum Js;
  bool have_J = false;
  const bool kernel_rows = d.c_J != 0.0 && (f.nFpos > 0 || f.nFneg > 0);
  if (f.nJ > 0 && d.c_J != 0.0) {
    // t[P][n] = sum_ia L_ov[P][ia] X[n][ia];  J[n][ia] = sum_P t[P][n] L_ov[P][ia]
    if (tensor_cores && f.tc_elt == TcElt::F16 && f.JovT_hi && !f64) {
      // t = L_ov X^T on the SIMT path (K = ov: its FP32 reduction tree keeps t
      // at ~1e-7; one tensor-core accumulation run per 4096 terms left the
      // Coulomb products at ~2e-6), then J = t^T L_ov on the tensor cores,
      // streaming the FP16 hi+lo copy of s_ov L_ov transposed once, with t as
      // FP16 parts of s_t t
      const size_t tb = ((size_t)f.nJ * m * 4 + 255) & ~(size_t)255;
      const size_t hb = ((size_t)m * tc_pad(f.nJ) * 2 + 255) & ~(size_t)255;
      DevBuf t(tb + 2 * hb, s);
      Js.factor = DevBuf(4, s);
      char* th = t.as<char>() + tb;
      unsigned* tmax = words.as<unsigned>() + 4;
      tall_gram(f.Jov, f.dt, f.nJ, static_cast<const float*>(Xw), m, ov, t.as<float>(), s, tmax);
      tc_t_split(t.as<float>(), f.nJ, m, tmax, f.tc_scale + 4, th, th + hb, Js.factor.as<float>(), s);
      const bool keep = !kernel_rows;
      if (!keep) Jb = DevBuf(mov * ew, s);
      tc_contract(th, th + hb, tc_pad(f.nJ), m, 1, f.nJ, f.JovT_hi, f.JovT_lo, ov, Jb.as<float>(), false, TcElt::F16,
                  Js.factor.as<float>(), d.tc_err, s, nullptr, 0.0, 0.0, kCoulombKb, keep ? &Js : nullptr);
    } else {
      Jb = DevBuf(mov * ew, s);
      DevBuf t;
      const bool sliced = f64 && (double)f.nJ * ov * m >= kCoulombSliced;
      if (!sliced) t = DevBuf((size_t)f.nJ * m * ew, s);
      if (sliced) {
        coulomb_sliced(d, f, static_cast<const double*>(Xw), m, Jb.as<double>(), s);
      } else if (f64) {
        sk_gram(f.Jov, f.dt, ov, f.nJ, Xw, tw, ov, m, ov, t.p, tw, m, 1.0, 0.0, s);
        sk_combo(t.p, tw, 1, m, m, f.nJ, f.Jov, f.dt, ov, ov, Jb.p, tw, ov, 1.0, 0.0, s);
      } else {
        tall_gram(f.Jov, f.dt, f.nJ, static_cast<const float*>(Xw), m, ov, t.as<float>(), s);
        tall_combo(t.as<float>(), m, f.nJ, f.Jov, f.dt, ov, Jb.as<float>(), s);
      }
    }
    have_J = true;
  }
  if (d.c_J != 0.0) {
    // sum_g w_g F^g_ia (F^g . X): rows stored as sqrt|w_g| F^g, one pass per sign
    const void* Fr[2] = {f.Fpos, f.Fneg};
    const int nr[2] = {f.nFpos, f.nFneg};
    for (int k = 0; k < 2; ++k) {
      if (nr[k] <= 0) continue;
      if (!have_J) Jb = DevBuf(mov * ew, s);
      DevBuf t((size_t)nr[k] * m * ew, s);
      sk_gram(Fr[k], f.dt, ov, nr[k], Xw, tw, ov, m, ov, t.p, tw, m, 1.0, 0.0, s);
      sk_combo(t.p, tw, 1, m, m, nr[k], Fr[k], f.dt, ov, ov, Jb.p, tw, ov, k == 0 ? 1.0 : -1.0,
               have_J ? 1.0 : 0.0, s);
      have_J = true;
    }
  }

  // ---- exchange: K1 (and K2 for the paired products) of one factor set
  // K1s / K2s, when given, may take the partial sums instead (term_of)
  auto exchange = [&](const FactorSet& f, const XParts& xp, DevBuf& K1b, DevBuf& K2b, TcSum* K1s, TcSum* K2s) {
    const bool use_tc = tc_exchange(f, f64, tensor_cores);
    TD_REQUIRE(!tensor_cores || f64 || use_tc, TDDFT_ERR_ARG, "tensor-core factor copies missing");
    const int pc = use_tc ? chunk_rows(f.nK, (long long)m * no * tc_zpad(nv, 2) * 4, m, kChunkBytesTC)
                          : chunk_rows(f.nK, (long long)m * ov * (long long)ew, m, kChunkBytes);
    const size_t es = dtype_size(f.dt);
    if (!use_tc || pc < f.nK) K1s = K2s = nullptr;
    if (!K1s) {
      K1b = DevBuf(mov * ew, s);
      if (need_k2) K2b = DevBuf(mov * ew, s);
    }
    // 16-bit tensor-core operand pointer at element offset o
    auto at16 = [](const void* b, size_t o) { return static_cast<const void*>(static_cast<const uint16_t*>(b) + o); };
    if (use_tc && f.fp8) {
      // ris exchange rows in FP8 e4m3 (one scale per row P): the stage-1
      // products Z = L_oo X and Q = L_ov X^T run as for BF16 (trial vectors as
      // BF16 hi + lo against the BF16 rows) and leave their results as e4m3
      // hi + lo, multiplied by mu_P; the second contractions run as
      // kind::f8f6f4 (two products: hi and lo against the e4m3 rows) and the
      // sums are multiplied back by 1/g (tc_fp8_scales).
      const int nvp = tc_pad(nv), nop = tc_pad(no), nv16 = tc_pad16(nv), no16 = tc_pad16(no);
      const int nvz = tc_zpad(nv, 1), noz = tc_zpad(no, 1);
      const float* inv1 = xp.sc;
      const float* inv2 = inv1 + 1;
      const float* mu1 = inv1 + 2;
      const float* mu2 = mu1 + f.nK;
      const StageParts zq(m, no, pc, nvz, need_k2 ? noz : 0, 1, s);
      const int Mz = m * no;
      for (int p0 = 0; p0 < f.nK; p0 += pc) {
        const int pn = (f.nK - p0 < pc) ? f.nK - p0 : pc;
        tc_stage1_fp8(static_cast<const __nv_bfloat16*>(xp.th), static_cast<const __nv_bfloat16*>(xp.tl), m, nv, no,
                      static_cast<const __nv_bfloat16*>(f.Koo_hi) + (size_t)p0 * no * nop, no, pn, mu1 + p0,
                      zq.z[0], zq.z[1], d.tc_err, s);
        tc_contract8(zq.z[0], zq.z[1], Mz, pn, nv,
                     f.Kvv8 + (size_t)p0 * nv * nv16, nv, K1b.as<float>(), p0 > 0, inv1, d.tc_err, s, K1s);
        if (need_k2) {
          tc_stage1_fp8(static_cast<const __nv_bfloat16*>(xp.sh), static_cast<const __nv_bfloat16*>(xp.sl), m, no, nv,
                        static_cast<const __nv_bfloat16*>(f.Kovp_hi) + (size_t)p0 * no * nvp, no, pn, mu2 + p0,
                        zq.q[0], zq.q[1], d.tc_err, s);
          tc_contract8(zq.q[0], zq.q[1], Mz, pn, no,
                       f.Kvo8 + (size_t)p0 * nv * no16, nv, K2b.as<float>(), p0 > 0, inv2, d.tc_err, s, K2s);
        }
      }
    } else if (use_tc) {
      // Both contractions of K1 and of K2 on the tensor cores.  The trial block
      // enters twice: transposed per vector ([(n,a)][j]) for Z = L_oo X and as is
      // ([(n,j)][b]) for Q = L_ov X^T, always as hi + lo (so Z and Q are too).
      // Exact factor sets (FP16): the factors are split hi + lo as well (three
      // products); every operand carries a power of two (tc_f16_product_scales)
      // that the contractions' sums remove.  ris factor sets (BF16): the
      // factors are used as they are (two products, exact with respect to them).
      const bool f16 = f.tc_elt == TcElt::F16;
      const TcElt et = f.tc_elt;
      const int nvp = tc_pad(nv), nop = tc_pad(no);
      const float *mz = nullptr, *mq = nullptr, *f1 = nullptr, *f2 = nullptr;
      if (f16) {
        mz = xp.sc + 1; mq = xp.sc + 2; f1 = xp.sc + 3; f2 = xp.sc + 4;
      }
      const int nvz = tc_zpad(nv, 2), noz = tc_zpad(no, 2);
      const StageParts zq(m, no, pc, nvz, need_k2 ? noz : 0, 2, s);
      const int Mz = m * no;
      for (int p0 = 0; p0 < f.nK; p0 += pc) {
        const int pn = (f.nK - p0 < pc) ? f.nK - p0 : pc;
        tc_stage1(xp.th, xp.tl, m, nv, no, at16(f.Koo_hi, (size_t)p0 * no * nop),
                  f16 ? at16(f.Koo_lo, (size_t)p0 * no * nop) : nullptr, no, pn, et, mz, zq.z[0], zq.z[1], d.tc_err, s);
        const bool timed = d.prof && d.prof->on && f16;
        tc_contract(zq.z[0], zq.z[1], nvz, Mz, pn, nv, at16(f.Kvv_hi, (size_t)p0 * nv * nvp),
                    f16 ? at16(f.Kvv_lo, (size_t)p0 * nv * nvp) : nullptr, nv, K1b.as<float>(), p0 > 0, et, f1,
                    d.tc_err, s, timed ? d.prof : nullptr, 2.0 * Mz * (double)nv * (double)pn * nv,
                    // Z hi+lo [Mz][pn*nv], L_vv chunk [pn*nv][nv] (hi+lo for FP16), K1 FP32
                    // written (and read back when accumulating)
                    4.0 * Mz * (double)pn * nv + (f16 ? 4.0 : 2.0) * (double)pn * nv * nv +
                        4.0 * Mz * (double)nv * (p0 > 0 ? 2.0 : 1.0),
                    f16 ? kExchangeKb : 0, K1s);
        if (need_k2) {
          tc_stage1(xp.sh, xp.sl, m, no, nv, at16(f.Kovp_hi, (size_t)p0 * no * nvp),
                    f16 ? at16(f.Kovp_lo, (size_t)p0 * no * nvp) : nullptr, no, pn, et, mq, zq.q[0], zq.q[1], d.tc_err, s);
          tc_contract(zq.q[0], zq.q[1], noz, Mz, pn, no, at16(f.Kvo_hi, (size_t)p0 * nv * nop),
                      f16 ? at16(f.Kvo_lo, (size_t)p0 * nv * nop) : nullptr, nv, K2b.as<float>(), p0 > 0, et, f2,
                      d.tc_err, s, nullptr, 0.0, 0.0, f16 ? kExchangeKb : 0, K2s);
        }
      }
    } else if (f.dt != DType::BF16 && (double)m * f.nK * no * nv * (no + nv + (need_k2 ? 2.0 * no : 0.0)) >=
                                          (f64 ? kExchangeSliced64 : kExchangeSliced32)) {
      exchange_sliced(d, f, Xw, m, need_k2, K1b.p, K2b.p, s);
    } else {
      // ris rows (BF16) against FP32 trial vectors, and small products, on the FP32 or FP64 units
      DevBuf Zb((size_t)m * no * pc * nv * ew, s);
      DevBuf Qb;
      if (need_k2) Qb = DevBuf((size_t)m * no * pc * no * ew, s);
      for (int p0 = 0; p0 < f.nK; p0 += pc) {
        const int pn = (f.nK - p0 < pc) ? f.nK - p0 : pc;
        // Z[n][i][P][a] = sum_j Koo[P][i][j] X[n][j][a]
        GemmDesc z;
        z.acc64 = f64;
        z.M = no; z.N = nv; z.K = no;
        z.A = (const char*)f.Koo + (size_t)p0 * no * no * es; z.ta = f.dt; z.sam = no; z.sak = 1;
        z.B = Xw; z.tb = tw; z.sbk = nv; z.sbn = 1;
        z.C = Zb.p; z.tc = tw; z.scm = (long long)pn * nv; z.scn = 1;
        z.nb0 = pn; z.nb1 = m;
        z.sA0 = (long long)no * no; z.sB0 = 0; z.sC0 = nv;
        z.sA1 = 0; z.sB1 = ov; z.sC1 = (long long)no * pn * nv;
        gemm(z, s);
        const int Mz = m * no;
        const long long Kz = (long long)pn * nv;
        GemmDesc k;
        k.acc64 = f64;
        k.M = Mz; k.N = nv; k.K = (int)Kz;
        k.A = Zb.p; k.ta = tw; k.sam = Kz; k.sak = 1;
        k.B = (const char*)f.Kvv + (size_t)p0 * nv * nv * es; k.tb = f.dt; k.sbk = nv; k.sbn = 1;
        k.C = K1b.p; k.tc = tw; k.scm = nv; k.scn = 1;
        k.beta = (p0 > 0) ? 1.0 : 0.0;
        const bool timed = d.prof_simt && d.prof_simt->on && f.dt != DType::BF16;
        if (timed) d.prof_simt->begin(s);
        gemm_splitk(k, auto_splits(k.M, k.N, k.K), s);
        if (timed)
          d.prof_simt->end(s, 2.0 * Mz * (double)nv * (double)Kz,
                           (double)es * ((double)Mz * (double)Kz + (double)Kz * nv +
                                         (double)Mz * nv * (p0 > 0 ? 2.0 : 1.0)));
        if (need_k2) {
          // Q[n][i][P][j] = sum_b Kov[P][i][b] X[n][j][b]
          GemmDesc q;
          q.acc64 = f64;
          q.M = no; q.N = no; q.K = nv;
          q.A = (const char*)f.Kov + (size_t)p0 * ov * es; q.ta = f.dt; q.sam = nv; q.sak = 1;
          q.B = Xw; q.tb = tw; q.sbk = 1; q.sbn = nv;
          q.C = Qb.p; q.tc = tw; q.scm = (long long)pn * no; q.scn = 1;
          q.nb0 = pn; q.nb1 = m;
          q.sA0 = ov; q.sB0 = 0; q.sC0 = no;
          q.sA1 = 0; q.sB1 = ov; q.sC1 = (long long)no * pn * no;
          gemm(q, s);
          GemmDesc k2;
          k2.acc64 = f64;
          k2.M = m * no; k2.N = nv; k2.K = pn * no;
          k2.A = Qb.p; k2.ta = tw; k2.sam = (long long)pn * no; k2.sak = 1;
          k2.B = (const char*)f.Kov + (size_t)p0 * ov * es; k2.tb = f.dt; k2.sbk = nv; k2.sbn = 1;
          k2.C = K2b.p; k2.tc = tw; k2.scm = nv; k2.scn = 1;
          k2.beta = (p0 > 0) ? 1.0 : 0.0;
          gemm_splitk(k2, auto_splits(k2.M, k2.N, k2.K), s);
        }
      }
    }
  };
  DevBuf K1b, K2b;
  TcSum K1s, K2s;
  double kx = d.a_x;   // weight of the exchange parts in the final combination
  if (main_x) exchange(f, xp, K1b, K2b, lr_x ? nullptr : &K1s, lr_x ? nullptr : &K2s);
  if (lr_x) {
    // second exchange set: K = a_x K[L] + b_x K[M], combined with weight 1
    XParts xl;
    if (tc_exchange(*f.lr, f64, tensor_cores))
      xl = make_x_parts(d, *f.lr, X, xt, m, need_k2, words.as<unsigned>(), nullptr, s);
    DevBuf L1, L2;
    exchange(*f.lr, xl, L1, L2, nullptr, nullptr);
    if (!main_x) {
      K1b = DevBuf(mov * ew, s);
      if (need_k2) K2b = DevBuf(mov * ew, s);
    }
    axpby(K1b.p, L1.p, tw, main_x ? d.a_x : 0.0, f.b_x, mov, s);
    if (need_k2) axpby(K2b.p, L2.p, tw, main_x ? d.a_x : 0.0, f.b_x, mov, s);
    kx = 1.0;
  }

  const double cj = mode == OpMode::TDA ? d.c_J : 2.0 * d.c_J;
  if (!f64) {
    combine_sums<TX>(X, d.delta, term_of(Js, Jb), term_of(K1s, K1b), term_of(K2s, K2b), cj, -kx, -kx, m, ov, out0,
                     mode == OpMode::TDA ? nullptr : out1, s);
  } else if constexpr (!x32) {
    if (mode == OpMode::TDA) {
      combine(X, d.delta, Jb.p, K1b.p, nullptr, tw, cj, -kx, 0.0, m, ov, out0, s);
    } else {
      combine(X, d.delta, Jb.p, K1b.p, K2b.p, tw, cj, -kx, -kx, m, ov, out0, s);
      combine(X, d.delta, nullptr, K1b.p, K2b.p, tw, 0.0, -kx, kx, m, ov, out1, s);
    }
  }
}

double product_work_bytes(int no, int nv, int nJ, int nK, int m, DType t, bool tensor_cores, bool paired) {
  const double ov = (double)no * nv, mov = m * ov, es = (double)dtype_size(t);
  const bool f64 = t == DType::F64;
  const double nop = tc_pad(no), nvp = tc_pad(nv);
  auto rows = [&](double per_row, size_t budget) {   // rows of a chunk, as chunk_rows has them
    return std::max(1.0, std::min((double)nK, std::floor((double)budget / per_row)));
  };
  // K-split partials of a product of M x N outputs: whole waves of tiles, or runs of at
  // most `run` terms
  auto partials = [&](double M, double N, double K, double run, double tile_bytes) {
    return std::max(4.0 * 152 * tile_bytes, M * N * 4.0 * (std::floor(K / run) + 2.0));
  };
  // terms' sums (two exchange sets), t, and what the Coulomb Gram products of FP32 rows leave per chunk
  double b = 5.0 * mov * (f64 ? 8 : 4) + (f64 ? 0.0 : mov * 4.0) + 2.0 * nJ * m * 8.0;
  const double gram = 8.0 * m * std::max(584.0 * 128.0, (double)nJ * (ov / 2048.0 + 1.0));
  if (tensor_cores) {
    const double nvz = tc_zpad(nv, 2), noz = tc_zpad(no, 2);
    const double pc = rows(m * no * nvz * 4.0, kChunkBytesTC);
    const double tile = 128.0 * 256 * 4;
    const double k1 = partials(m * no, nv, pc * nvp, 64.0 * kExchangeKb, tile);
    const double j = partials(m, ov, nJ, 64.0 * kCoulombKb, tile), keep = (double)kKeepBytes;
    return b + gram + m * no * pc * (nvz + (paired ? noz : 0.0)) * 4.0 + 4.0 * m * (nv * nop + no * nvp) +
           std::min(j, keep) + (paired ? std::min(k1, keep) : 0.0) + std::max(j, k1);
  }
  if (t == DType::BF16) {
    const double pc = rows(mov * 4.0, kChunkBytes);
    return b + gram + pc * m * no * (nv + (paired ? no : 0.0)) * 4.0 + partials(m * no, nv, pc * nv, 1e30, 2.0 * 64 * 64 * 4);
  }
  const double sb = slice_element_bytes(t);
  const double row = m * no * (nv * es + nvp * sb) + (no * nop + nv * nvp) * sb +
                     (paired ? m * no * (no * es + nop * sb) + (no * nvp + nv * nop) * sb : 0.0);
  const double pc = rows(row, kChunkBytesSliced);
  const double sums = 4.0 * 152 * (128 * 128 * 4 + 128 * 256 * 4) + 12.0 * std::max(mov, (double)nJ * m);
  const double exchange = pc * row + 16.0 * (pc * 2 * no + 4.0 * m * (no + nv)) + m * (nv * nop + no * nvp) * sb;
  const double coulomb = f64 ? std::max((double)kChunkBytesSliced, std::max(ov, (double)nJ) * sb) + m * (ov + 8) * sb +
                                   m * (nJ + 8.0) * sb + 16.0 * (ov + nJ)
                             : gram;
  return b + sums + std::max(exchange, coulomb);
}

void apply_operator(const OpDims& d, const FactorSet& f, const double* X, int m, OpMode mode,
                    double* out0, double* out1, int tc, cudaStream_t s) {
  apply_operator_t<double>(d, f, X, m, mode, out0, out1, tc, s);
}

void apply_operator(const OpDims& d, const FactorSet& f, const float* X, int m, OpMode mode,
                    float* out0, float* out1, int tc, cudaStream_t s) {
  apply_operator_t<float>(d, f, X, m, mode, out0, out1, tc, s);
}

}  // namespace tddft
