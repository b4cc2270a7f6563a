// FP64-accurate complex GEMM on the tcgen05 tensor cores: every FP64 operand row is written as eight
// 8-bit integer slices with one power-of-two scale (the error-free splitting of Ozaki, Ogita, Oishi and
// Rump, Numer. Algorithms 59 (2012), on matrix engines as in Mukunoki, Ozaki, Ogita and Imamura, ISC 2020),
// the slice products are BF16 MMAs whose FP32 sums are exact integers, and the sums are combined in 64-bit
// integers.
//
//   x = 2^e sum_{s=0..7} d_s 2^-(8 s + 7),   |d_s| <= 128 (63 bits under the largest entry of the row),
//   sum_k a_k b_k = 2^(ea + eb) sum_{q=0..7} S_q 2^-(8 q + 14),   S_q = sum_k sum_{i+j=q} d_i(a_k) d_j(b_k);
// the orders q >= 8 are dropped, so the error is a few 2^-64 of (largest entry of the row) x (largest entry of the column)
// per term, however small the terms are.  FP64 sums are off by some 2^-53 of the sum of the terms' magnitudes.  The slices are
// as good as long as that sum s = sum_k |a_k||b_k| is not far below the product of the maxima; where the large entries of a
// row meet the small ones of a column they are not.  So s itself is formed, for the real and the imaginary part of
// every entry of C, as one more BF16 product, of the operands' magnitudes (a ninth plane beside the slices), and
// entries with 0 < s < sqrt(2 K) 2^-8 2^(ea + eb) are summed again in FP64 from the operands themselves.  At that
// line the slices' error is about that of an FP64 loop (root mean square over random rows, in units of 2^-53 s: 2 K = 8
// terms 0.2 against 0.45, 32: 0.15 and 0.45, 128: 0.1 and 0.35, 1000: 0.06 and 0.12), and twice to four times it one
// factor of four below; where s = 0, every term is zero.
#pragma once
#include <cstdint>

#include "kernels.cuh"
#include "tc_gemm.cuh"

namespace cclr {

constexpr int F64_SLICES = 8;
constexpr int F64_PLANES = F64_SLICES + 1;  // the slices and the magnitudes
// Scale of a row that holds a NaN or an infinity: its products are written as NaN.
constexpr int F64_NONFINITE = 1 << 20;

// Real elements per slice row of K complex entries (whole 16-byte units) and the bytes of a prepared
// operand of R rows (embed: two slice rows per complex column, as the GEMM's column operand needs).
inline int64_t f64tc_ld(int64_t K) { return (2 * K + 7) / 8 * 8; }
inline int64_t f64tc_bytes(int64_t R, int64_t K, bool embed) { return F64_PLANES * R * (embed ? 2 : 1) * f64tc_ld(K) * 2; }

// A prepared operand, or the rows [r0, r0 + rows) of one: slice s of row r is row s * stride + r0 + r of p
// (embedded operands have two slice rows per complex column; stride, r0 and rows count columns then).  The operand
// that it was prepared from has to be there, unchanged, for the products too.
struct F64Op {
  const void *p = nullptr;
  const uint32_t *tops = nullptr;  // high word of the largest magnitude of each row: its scale
  int64_t stride = 0, r0 = 0;
  const void *src = nullptr;       // complex128 entry (r, k) at v2off(rv, r) + v2off(kv, k), r from the operand's first row
  View2 rv, kv;
  F64Op rows(int64_t first) const {
    F64Op o = *this;
    o.r0 += first;
    return o;
  }
};

// Slices and magnitudes of the complex128 operand X(r, k) = src[v2off(rv, r) + v2off(kv, k)], r < R, k < K, into dst, and the
// rows' largest magnitudes into tops[R].  embed: the column operand, (re, -im) and (im, re).
F64Op f64tc_prep(const void *src, View2 rv, View2 kv, int64_t R, int64_t K, bool embed, void *dst, uint32_t *tops,
                 cudaStream_t st);

// A stream beside the caller's, made at first use.  The comparison of the magnitudes' sums depends on the slices alone and the
// slice products do not depend on it: it runs beside them (o = 10, v = 40, whose products fill a part of the SMs: sigma 1.95
// ms one after the other, 1.72 so).
class F64Side {
 public:
  F64Side() = default;
  F64Side(const F64Side &) = delete;
  ~F64Side();
  // the side stream, which goes on from the present end of st; join() makes st wait for the side stream's present end
  cudaStream_t fork(cudaStream_t st);
  void join(cudaStream_t st);

 private:
  cudaStream_t s_ = nullptr;
  cudaEvent_t fork_ = nullptr, join_ = nullptr;
};

// C(m, n) (+)= alpha sum_k A(m, k) B(k, n), complex128, from prepared operands (A: M rows, B: N embedded
// columns).  C(m, n) at C + v2off(rv, m) + v2off(cv, n) complex entries; accumulate: added to C, else C is
// overwritten.  scratch: f64tc_scratch_bytes of device memory for the integer sums (at most 256 MB), of M and N or of
// any larger numbers of rows and columns.  upper: only tiles with an entry b > a are needed, counting the rows (b, f) from
// upper_row and the columns (a, e) from upper_col.
void f64tc_gemm(const F64Op &A, int64_t M, const F64Op &B, int64_t N, int64_t K, void *C, View2 rv, View2 cv, zc alpha,
                bool accumulate, void *scratch, F64Side &side, cudaStream_t st, class UpperTiles *upper = nullptr,
                int64_t upper_row = 0, int64_t upper_col = 0);
size_t f64tc_scratch_bytes(int64_t M, int64_t N);

}  // namespace cclr
