// FP64 products on the tensor cores by exact digit slices (the splitting of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix multiplication", 2012).
//
// Z(i, c) = sum_j A(i, j) B(c, j): every operand row is scaled by a power of two 2^E > max |x| and cut into OZ_S signed
// digits of OZ_BITS bits, x = 2^E sum_s d_s 2^(-8 - 9 s), |d_s| <= 256: 63 bits below the row's scale, against the 53 of
// an FP64 entry.  Digits up to 256 are exact in bf16, their products (<= 2^16) are exact, and the sums of one 64-wide
// block of j over the s + 1 digit pairs of a level i + j = s are integers that FP32 holds exactly for levels 0 to 3
// (<= 2^24); a larger sum in levels 4 to 6 would need some 300 products of one sign near their largest value.
// So a block is 28 digit pairs (those with i + j <= 6) on 7 levels; the blocks are summed in integers and an output is
// rounded to FP64 once, where a chain of FMAs rounds at every term.
//
// What is dropped (an entry's bits below 2^-63 of its row's largest, the pairs beyond level 6) adds up to about
// sqrt(n) 2^-63 2^(Ea + Eb) over n terms, whatever the entries; a chain of FMAs errs by 2e-17 to 2e-16 of sum |a||b|.  On
// rows that are small where the other operand is large the scales say little about the sum, and there the chain is the
// better one.  So the sum of |a||b| 2^-(Ea + Eb) is formed along with the digits (from magnitudes rounded down to bf16),
// and an output where it is below sqrt(n) 2^-8 is computed by FP64 FMAs after all (k_oz_fix); so is one whose level sums
// were too large, whose result is no normal number, or whose row holds an infinity or a NaN.  At that line the digits err by
// 2e-17 of sum |a||b|, the chain by 4e-17 to 7e-17 (rms; rows that peak in one entry, rows graded against each other,
// n = 256, 1158, 4614; below 2^-10 the chain is ahead).  On S^+ of 8^3 and 12^3 elastic and 64^2 heat patterns no output
// falls below it: the smallest sums are 2^-4 sqrt(n), the digits err by 1e-18 there and the chain by 3e-17.  On the factors of
// 12^3 16 % of the outputs of Lam = L_S^{-1} do (its rows peak at their diagonal) and 0.6 % of those of Lam^T.
//
// A tile of 64 rows is stored as the 7 slices of its 64 x 64 digits and their magnitudes, each in the layout the MMA reads (K-major rows of 128
// bytes, 128-byte swizzle), so that consecutive slices are contiguous rows of one operand (which of them meet in an MMA:
// oz_plan.cuh).
#pragma once
#include "common.cuh"
#include "oz_plan.cuh"

namespace fetirp {

constexpr int OZ_SLICE = 64 * 128;                           // 8 KB: 64 rows of one slice
constexpr int OZ_TILE = OZ_SLICES * OZ_SLICE;                // 64 KB: one 64 x 64 tile
constexpr int OZ_E_ZERO = -8000;                             // exponent of a row of zeros
constexpr int OZ_E_BAD = 100000;                             // of a row with an infinity or a NaN

// A sliced operand of `rows` x `cols`: its 64 x 64 tiles, a row of tiles after the other, and an exponent for every row
// (padded to 64).  Mode 1 (2): square and zero above (below) the diagonal; a row of tiles then ends (begins) with the diagonal
// tile of the second (first) of the two rows that a CTA multiplies together, which have equally many.
struct OzRow {
  long long begin;      // tiles before this row of tiles
  int first, last;      // its tile columns [first, last)
};
__host__ __device__ inline OzRow oz_row(int mode, int row, int kt) {
  const long long q = row >> 1, odd = row & 1;
  if (mode == 1) {
    const int w = kt < 2 * q + 2 ? kt : (int)(2 * q + 2);
    return {2 * q * (q + 1) + odd * w, 0, w};
  }
  if (mode == 2) return {2 * q * kt - 2 * q * (q - 1) + odd * (kt - 2 * q), (int)(2 * q), kt};
  return {(long long)row * kt, 0, kt};
}
inline long long oz_tiles(long long rows, long long cols, int mode = 0) {
  const int kt = (int)((cols + 63) / 64);
  const OzRow last = oz_row(mode, (int)((rows + 63) / 64) - 1, kt);
  return last.begin + last.last - last.first;
}
struct OzOperand {
  uint8_t* tiles = nullptr;
  int* exps = nullptr;
};

constexpr int OZ_MAXP = 16;
// Slices of row-major operands in one launch (element (r, c) at x[r ld + c]); in mode 1 (2) only c <= r (c >= r) is read.
struct OzSliceBatch {
  int n = 0;
  const double* x[OZ_MAXP];
  long long ld[OZ_MAXP];
  int rows[OZ_MAXP], cols[OZ_MAXP], mode[OZ_MAXP], row_off[OZ_MAXP];
  OzOperand out[OZ_MAXP];
  void add(const double* x_, long long ld_, int rows_, int cols_, int mode_, const OzOperand& o) {
    x[n] = x_; ld[n] = ld_; rows[n] = rows_; cols[n] = cols_; mode[n] = mode_; out[n] = o;
    ++n;
  }
};
void oz_slice(const OzSliceBatch& batch, cudaStream_t s);
void oz_slice_rows(const double* x, long long ld, int rows, int cols, int mode, const OzOperand& out, cudaStream_t s);
// The same of a column-major operand (element (r, c) at x[r + c ld]).
void oz_slice_cols(const double* x, long long ld, int rows, int cols, int mode, const OzOperand& out, cudaStream_t s);

struct OzGemm {
  int n = 0;                      // products in the launch
  OzOperand A[OZ_MAXP], B[OZ_MAXP];
  int M[OZ_MAXP], N[OZ_MAXP], K[OZ_MAXP];
  int mode[OZ_MAXP];              // A(i, j): 0 dense, 1 zero for j > i, 2 zero for j < i
  double* Z[OZ_MAXP];             // Z[c * ldz + i]
  long long ldz[OZ_MAXP];
  // the operands themselves, for the outputs that FMAs compute: A(i, j) at a[i * ai + j * aj] with ai or aj = 1, and
  // B(c, j) at b[c * ldb + j]
  const double* a[OZ_MAXP];
  long long ai[OZ_MAXP], aj[OZ_MAXP];
  const double* b[OZ_MAXP];
  long long ldb[OZ_MAXP];
  uint32_t* flags[OZ_MAXP];       // scratch: oz_flag_words(M, N) words, which outputs those are
  int* error = nullptr;
};
// A bit per output: word c ceil(M / 32) + i / 32
inline long long oz_flag_words(long long M, long long N) { return (M + 31) / 32 * N; }
void oz_gemm(const OzGemm& G, cudaStream_t s);

// One-time kernel attribute set-up (large dynamic shared memory); call before any graph capture.
void oz_init();

#ifdef __CUDACC__
// |x| as the bits that order like it, for row maxima
__device__ __forceinline__ unsigned long long oz_abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}

// The exponent E of a row from the largest of its |x| bits: 2^E > max |x|.
__device__ __forceinline__ int oz_row_exp(unsigned long long mx) {
  const int ef = (int)(mx >> 52);
  if (ef == 2047) return OZ_E_BAD;
  if (mx == 0) return OZ_E_ZERO;
  return (ef ? ef : 1) - 1022;   // x < 2^(ef - 1022); subnormals are below 2^-1022 * 2
}

// Digits of x under row exponent E, lowest first out of the 63-bit fixed-point value x 2^(62 - E).
__device__ __forceinline__ void oz_digits(double x, int E, int (&d)[OZ_S]) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ef = (int)(b >> 52) & 2047;
  unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | (ef ? 1ull << 52 : 0ull);
  const int sh = (ef ? ef : 1) - 1022 + 9 - E;   // m 2^(e - 52) 2^(62 - E), e = ef - 1023
  if (E == OZ_E_BAD || sh < -54) m = 0;
  else if (sh >= 0) m <<= sh;                     // sh <= 9: |x| < 2^E
  else m = (m + (1ull << (-sh - 1))) >> -sh;
  long long f = (long long)b < 0 ? -(long long)m : (long long)m;
#pragma unroll
  for (int s = OZ_S - 1; s > 0; --s) {
    const int q = ((int)((unsigned)f << 23)) >> 23;   // the low 9 bits, signed: -256 .. 255
    d[s] = q;
    f = (f - q) >> 9;
  }
  d[0] = (int)f;
}

// bf16 bits of |x| 2^-E, rounded down (0 below 2^-126 and in rows with an infinity or a NaN)
__device__ __forceinline__ uint32_t oz_magnitude(double x, int E) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ef = (int)(b >> 52) & 2047, f = ef - 1023 + 127 - E;
  return ef == 0 || f <= 0 || E == OZ_E_BAD ? 0u : (uint32_t)f << 7 | ((uint32_t)(b >> 45) & 127u);
}

// bf16 bits of a digit (exact: |d| <= 256)
__device__ __forceinline__ uint32_t oz_bf16(int d) { return __float_as_uint((float)d) >> 16; }

// Byte offset of digit (row, k) of slice s in a tile
__device__ __forceinline__ int oz_offset(int row, int k, int s) {
  return s * OZ_SLICE + row * 128 + ((((k >> 3) ^ row) & 7) << 4) + (k & 7) * 2;
}
#endif

}  // namespace fetirp
