// What the two forms of the binary64 products share (fp64.cu on the FP64 pipe, gemm_f64.cuh on the tensor
// cores): how an output ends, and which form takes a product.
#pragma once

#include <cstdint>

#include "common.cuh"

namespace spl {

// Final value of an output whose sum is acc:
//   kOut64  out64 = acc (the correction C, binary64)
//   kUnmask out32 = fl32(acc - c)
//   kSlalom out32 = ((acc - c) mod q, taken in (-q/2, q/2]) 2^-16: the Slalom comparator's unmask
//           and de-quantization (Sec. 6.2); acc and c are exact integers in binary64.
enum { kOut64 = 0, kUnmask = 1, kSlalom = 2 };
constexpr double kSlalomModulus = 10485767.0;  // 2^23 + 2^21 + 7

__device__ __forceinline__ void finish_f64(double* out64, float* out32, int64_t o, double acc, const double* c,
                                           int mode) {
  if (mode == kOut64) {
    out64[o] = acc;
  } else if (mode == kUnmask) {
    out32[o] = (float)(acc - c[o]);
  } else {
    const double t = acc - c[o];  // exact integer, |t| < 2^53
    double m = t - kSlalomModulus * floor(t / kSlalomModulus);
    if (m < 0.0) m += kSlalomModulus;
    if (m >= kSlalomModulus) m -= kSlalomModulus;
    if (m > (kSlalomModulus - 1.0) * 0.5) m -= kSlalomModulus;
    out32[o] = (float)(m * 0x1p-16);
  }
}

// Products that run as exact slices on the tensor cores (on sm_100 / sm_103; the FP64 pipe takes the rest).  The
// slices cost three launches, about 18 us at the least, and then hardly depend on M up to 16 rows, where the
// FP64 pipe takes (M + 1) K N cycles' worth.  Measured, FP64 pipe against slices: 128 x 8192 by 3072 7414 against
// 248 us (5.2 ms at the pipe's rate), 16 rows 946 against 95, 1 row 118 against 88; 16 x 512 by 512 26 against 18,
// 4 x 1024 by 1024 27 against 20, but 8 x 512 by 512 15 against 18; of one row 4096 by 2048 43 against 37 and
// 2048 by 2048 25 against 27, and with short rows 512 by 16384 41 against 54.  The bounds on K and the sizes keep
// the 96-bit sums and the grids in range.  Those are times of rows that the slices hold; what others cost stands at
// f64_again.
// Slalom's integers (below 2^24, sums below 2^53) lose nothing in the slices: in fixed point below the row's largest
// exponent E <= 23 an integer is a multiple of 2^30, so its digits 0, 1 and 2 are 0, every product of two digits that
// are not (p + s >= 6) is kept, and the exact sum, of at most 53 bits, becomes a double without rounding.
inline bool f64_on_tensor_cores(int64_t M, int64_t K, int64_t N) {
  if (K >= (int64_t(1) << 21) || M >= (int64_t(1) << 19) || N >= (int64_t(1) << 20)) return false;
  if (M < 4) return K >= 2048 && K * N >= (int64_t(1) << 23);
  return K >= 128 && M * N >= ((int64_t(1) << 22) + K - 1) / K;
}
// Workspace of that form after the counters (0: it does not take the product), and the product; the caller has
// checked the arguments and the workspace.
size_t f64_tc_bytes(int64_t M, int64_t K, int64_t N);
spl_status run_f64_tc(double* out64, float* out32, const float* A, const float* W, const double* c, int64_t M,
                      int64_t K, int64_t N, void* ws, cudaStream_t stream, int mode);
spl_status run_f64_tc(double* out64, float* out32, const double* A, const float* W, const double* c, int64_t M,
                      int64_t K, int64_t N, void* ws, cudaStream_t stream, int mode);

}  // namespace spl
