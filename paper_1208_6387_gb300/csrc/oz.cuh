// FP64 products on the tensor cores by exact digit slices (the splitting of Ozaki, Ogita, Oishi and Rump, "Error-free
// transformations of matrix multiplication by using fast routines of matrix multiplication", 2012).
//
// Z(i, c) = sum_j A(i, j) B(c, j): every operand row is scaled by a power of two 2^E > max |x| and cut into OZ_S signed
// digits of OZ_BITS bits, x = 2^E sum_s d_s 2^(-8 - 9 s), |d_s| <= 256: 63 bits below the row's scale, against the 53 of
// an FP64 entry.  Digits up to 256 are exact in bf16, their products (<= 2^16) are exact, and the sums of one 64-wide
// block of j over the s + 1 digit pairs of a level i + j = s are integers that FP32 holds exactly for levels 0 to 3
// (<= 2^24); in levels 4 to 6 a sum beyond 2^24 would need some 300 products of one sign near their largest value, and
// would then round at 2^-52 of that value.  So a block is 28 bf16 MMAs (the pairs with i + j <= 6) into 7 accumulators;
// the blocks are summed in integers and an output is rounded to FP64 once, where a chain of FMAs rounds at every term.
//
// A tile of 64 rows is stored as the 7 slices of its 64 x 64 digits, each in the layout the MMA reads (K-major rows of 128
// bytes, 128-byte swizzle), so that consecutive slices are contiguous rows of one operand (which of them meet in an MMA:
// oz_plan.cuh).
#pragma once
#include "common.cuh"
#include "oz_plan.cuh"

namespace fetirp {

constexpr int OZ_SLICE = 64 * 128;                           // 8 KB: 64 rows of one slice
constexpr int OZ_TILE = OZ_S * OZ_SLICE;                     // 56 KB: one 64 x 64 tile
constexpr int OZ_E_ZERO = -8000;                             // exponent of a row of zeros
constexpr int OZ_E_BAD = 100000;                             // of a row with an infinity or a NaN: its products are NaN

// A sliced operand of `rows` x `cols`: ceil(rows / 64) x ceil(cols / 64) tiles, a row of tiles after the other, and an
// exponent for every row (padded to 64).
inline long long oz_tiles(long long rows, long long cols) { return ((rows + 63) / 64) * ((cols + 63) / 64); }
struct OzOperand {
  uint8_t* tiles = nullptr;
  int* exps = nullptr;
};

constexpr int OZ_MAXP = 16;
// Slices of row-major operands in one launch (element (r, c) at x[r ld + c]); with tri = 1 (-1) only c >= r (c <= r) is
// read and the rest is zero.
struct OzSliceBatch {
  int n = 0;
  const double* x[OZ_MAXP];
  long long ld[OZ_MAXP];
  int rows[OZ_MAXP], cols[OZ_MAXP], tri[OZ_MAXP], row_off[OZ_MAXP];
  OzOperand out[OZ_MAXP];
  void add(const double* x_, long long ld_, int rows_, int cols_, int tri_, const OzOperand& o) {
    x[n] = x_; ld[n] = ld_; rows[n] = rows_; cols[n] = cols_; tri[n] = tri_; out[n] = o;
    ++n;
  }
};
void oz_slice(const OzSliceBatch& batch, cudaStream_t s);
void oz_slice_rows(const double* x, long long ld, int rows, int cols, int tri, const OzOperand& out, cudaStream_t s);
// The same of a column-major operand (element (r, c) at x[r + c ld]).
void oz_slice_cols(const double* x, long long ld, int rows, int cols, int tri, const OzOperand& out, cudaStream_t s);

struct OzGemm {
  int n = 0;                      // products in the launch
  OzOperand A[OZ_MAXP], B[OZ_MAXP];
  int M[OZ_MAXP], N[OZ_MAXP], K[OZ_MAXP];
  int mode[OZ_MAXP];              // A(i, j): 0 dense, 1 zero for j > i, 2 zero for j < i
  double* Z[OZ_MAXP];             // Z[c * ldz + i]
  long long ldz[OZ_MAXP];
  int* error = nullptr;
};
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

// bf16 bits of a digit (exact: |d| <= 256)
__device__ __forceinline__ uint32_t oz_bf16(int d) { return __float_as_uint((float)d) >> 16; }

// Byte offset of digit (row, k) of slice s in a tile
__device__ __forceinline__ int oz_offset(int row, int k, int s) {
  return s * OZ_SLICE + row * 128 + ((((k >> 3) ^ row) & 7) << 4) + (k & 7) * 2;
}
#endif

}  // namespace fetirp
