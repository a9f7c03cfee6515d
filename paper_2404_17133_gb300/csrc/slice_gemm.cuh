// FP64 and FP32 contractions on the FP16 tensor cores by exact slicing.
#pragma once
#include "common.cuh"

namespace tddft {

// One operand of slice_gemm: `rows` rows whose K extent is (P < np, k < K),
//   element (r, P, k) = p[(r / R) * rs1 + (r % R) * rs0 + P * ps + k * ks]
// of type F64 or F32, with ks == 1 (rows contiguous along k) or rs0 == 1
// (contiguous across rows: a transposed operand).  p_outer: the slices are kept
// as [slice][P][row][k] (else [slice][row][P][k]); the second operand of a product
// has it set, the first not.
struct SliceOperand {
  const void* p = nullptr;
  DType t = DType::F64;
  int rows = 0, np = 1, K = 0;
  int R = 1 << 30;
  long long rs1 = 0, rs0 = 0, ps = 0, ks = 1;
  bool p_outer = false;
};

// Slices per element: 7 for FP64 (56 bits below the row's largest element), 4
// for FP32 (32 bits).
inline int slice_count(DType t) { return t == DType::F64 ? 7 : 4; }
// Bytes of an element's FP16 digits and of its FP16 magnitude (for the guard).
inline int slice_element_bytes(DType t) { return 2 * slice_count(t) + 2; }
// Bytes of an operand's slices and magnitudes (rows of pad8(K)), and of what is kept
// per row (exponent, squared magnitudes, nonzero elements).
size_t slice_bytes(const SliceOperand& o);
inline size_t slice_info_bytes(const SliceOperand& o) { return (size_t)o.rows * 16; }

// Cut an operand into slices: parts (slice_bytes), info (slice_info_bytes).
void slice_cut(const SliceOperand& o, void* parts, void* info, cudaStream_t s);

// Every output of the products below is within two roundings of the sum of its terms'
// absolute values (root mean square): one that the slices cannot give so (its terms
// are small beside the largest elements of its rows) is formed again from the operands
// on the FP64 (FP32) units.

// Batched products (np == 1 on both sides, no split):
//   out[(r / R) * rs1 + (r % R) + (c % C) * cs0 + (c / C) * cs1] = sum_k A(r, k) B(c, k)
struct SliceScatter {
  int R = 1, C = 1;
  long long rs1 = 0, cs0 = 0, cs1 = 0;
};
void slice_gemm_scatter(const SliceOperand& A, const void* Ap, const void* Ai, const SliceOperand& B, const void* Bp,
                        const void* Bi, void* out, const SliceScatter& sc, int* err, cudaStream_t s);

// C[r][c] = sum_(P, k) A(r, P, k) B(c, P, k) + beta C[r][c], C [A.rows][B.rows]
// of the operands' type; K is split over CTAs and the partials summed in a fixed order.
void slice_gemm(const SliceOperand& A, const void* Ap, const void* Ai, const SliceOperand& B, const void* Bp,
                const void* Bi, void* C, double beta, int* err, cudaStream_t s);

}  // namespace tddft
