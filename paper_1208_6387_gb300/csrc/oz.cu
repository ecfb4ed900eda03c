// FP64 products on the tensor cores by exact digit slices (see oz.cuh).
#include <algorithm>
#include <mutex>

#include "oz.cuh"
#include "tc_ptx.cuh"

namespace fetirp {

namespace {

constexpr int THREADS = 320;                         // producer warp, MMA warp, 8 epilogue warps
constexpr int EPI_WARPS = 8;
constexpr int BUF_COLS = 256;                        // TMEM columns between the two accumulator buffers (7 x 32 used)

// K-major operand, 128-byte swizzle, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t desc128(const void* p) {
  return (uint64_t)((smem_u32(p) >> 4) & 0x3FFFu) | (uint64_t)1 << 16 | (uint64_t)(1024 >> 4) << 32 |
         (uint64_t)1 << 46 | (uint64_t)2 << 61;
}
// D f32, A and B bf16, both K-major, M = 128, N = n
__device__ __forceinline__ uint32_t idesc_bf16(int n) {
  return 1u << 4 | 1u << 7 | 1u << 10 | (uint32_t)(n >> 3) << 17 | (uint32_t)(128 >> 4) << 24;
}

// v 2^q in FP64, rounded to nearest (halves away from zero), by integer operations: on this GPU an FP64 conversion or
// addition costs more than this whole routine on the integer pipe.
__device__ __forceinline__ double scaled_i64(long long v, int q) {
  const bool neg = v < 0;
  unsigned long long a = neg ? 0ull - (unsigned long long)v : (unsigned long long)v;
  if (a == 0) return 0.0;
  const int n = __clzll((long long)a);
  a <<= n;
  const int be = 1023 + 63 + q - n;
  unsigned long long r = ((unsigned long long)(uint32_t)(be - 1) << 52) + (a >> 11) + ((a >> 10) & 1ull);
  if (be <= 0) r = 0;
  else if (be >= 2047) r = 0x7FF0000000000000ull;
  return __longlong_as_double((long long)(r | (neg ? 1ull << 63 : 0ull)));
}

// (hi + lo 2^-w) 2^e in FP64, one rounding after at least 62 significant bits; |lo| < 2^(w + 17)
__device__ __forceinline__ double rounded(long long hi, long long lo, int w, int e) {
  if (e > OZ_E_BAD / 2) return __longlong_as_double(0x7FF8000000000000ll);
  const long long ah = hi < 0 ? -hi : hi;
  const int room = min(w, __clzll(ah) - 2);   // as many of lo's bits as hi leaves room for
  return scaled_i64((hi << room) + (lo >> (w - room)), e - room);
}

constexpr int G_RING = 10;                              // A slices (128 rows, 16 KB) in flight
constexpr int G_SLICE = 4 * OZ_SLICE_HALF;
constexpr int G_SMEM = G_RING * G_SLICE + OZ_TILE + 1024 + 512;

struct OzGemmKernel {
  OzGemm G;
  int tiles_n[OZ_MAXP], tile_off[OZ_MAXP + 1];
};
}  // namespace

// One CTA: 128 rows of A (two row tiles) against 64 rows of B, all of K in 64-wide blocks.  Bound by the MMAs' rate (28
// digit pairs, i + j <= 6: over a long row the dropped products stay far below the rounding of an FP64 chain).  FP64 apply of
// three 16^3 elastic patterns (n_b = 4614, 256 right-hand sides each, 32.7 GFLOP): 27.5 ms with FP64 FMAs, 1.11 ms so
// (0.87 ms of it this kernel: 28 x 32.7 GFLOP issued at 1.05 PFLOP/s), and its error against 64 bits is the same
// (2.2e-10 of the projected result, which is that of S^+).  The two 32-column halves of a block have an accumulator
// buffer each (224 TMEM columns): one is drained while the other is multiplied.  Both halves use the same A slices, so
// a slice is released after its product with the second half and the ring of ten holds the next block's first ones; the
// B halves are refilled in turn.  Drained levels are added into 91-bit integers per output (a 64-bit and a 27-bit part):
// no FP64 operation before the final rounding.  The tensor pipe is busy 44 % of the time a CTA runs, at every size; the
// apply takes 1.16 ms with sixteen epilogue warps and 1.31 ms with both halves' MMAs in turn and the levels drained in two
// parts, so neither the drain's latency nor the dependence of consecutive MMAs is what is left.
__global__ void __launch_bounds__(THREADS, 1) k_oz_gemm(const __grid_constant__ OzGemmKernel P) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + G_RING * G_SLICE;
  uint64_t* afull = reinterpret_cast<uint64_t*>(sB + OZ_TILE);   // [G_RING]
  uint64_t* aempty = afull + G_RING;                             // [G_RING]
  uint64_t* bfull = aempty + G_RING;                             // [2]
  uint64_t* bempty = bfull + 2;                                  // [2]
  uint64_t* tfull = bempty + 2;                                  // [2]
  uint64_t* tempty = tfull + 2;                                  // [2]
  uint64_t* done = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* loads = abort_flag + 1;   // [3]: A slices, B halves 0 and 1 whose copies were issued
  volatile int* seen = loads + 3;         // [3]: whose arrival the MMA thread has seen

  const OzGemm& G = P.G;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int p = 0;
  while (p + 1 < G.n && (int)blockIdx.x >= P.tile_off[p + 1]) ++p;
  const int t = (int)blockIdx.x - P.tile_off[p];
  const int tm = t / P.tiles_n[p], tn = t % P.tiles_n[p];
  const int kt = (G.K[p] + 63) / 64, mt = (G.M[p] + 63) / 64;
  const int a0 = 2 * tm, a1 = min(a0 + 1, mt - 1);
  // K blocks with nonzeros
  const int kb = G.mode[p] == 2 ? a0 : 0;
  const int ke = G.mode[p] == 1 ? min(kt, a1 + 1) : kt;
  const int nk = max(ke - kb, 0);

  if (threadIdx.x == 0) {
    for (int i = 0; i < G_RING; ++i) {
      mbar_init(&afull[i], 1);
      mbar_init(&aempty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bfull[i], 1);
      mbar_init(&bempty[i], 1);
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], EPI_WARPS);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    for (int i = 0; i < 3; ++i) loads[i] = seen[i] = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(2 * BUF_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    const uint8_t* A0 = G.A[p].tiles + (size_t)a0 * kt * OZ_TILE;
    const uint8_t* A1 = G.A[p].tiles + (size_t)a1 * kt * OZ_TILE;
    const uint8_t* B = G.B[p].tiles + (size_t)tn * kt * OZ_TILE;
    bool ok = true;
    auto load_b = [&](int c, int h) {
      if (c >= 1 && !(ok = mbar_wait(&bempty[h], (c & 1) ^ 1, abort_flag))) return;
      mbar_expect_tx(&bfull[h], OZ_HALF);
      bulk_load(sB + h * OZ_HALF, B + (size_t)(kb + c) * OZ_TILE + h * OZ_HALF, OZ_HALF, &bfull[h]);
      loads[1 + h] = c + 1;
    };
    int g = 0;   // A slices so far
    for (int c = 0; ok && c < nk; ++c) {
      load_b(c, 0);
      const size_t kofs = (size_t)(kb + c) * OZ_TILE;
      for (int i = 0; ok && i < OZ_S; ++i, ++g) {
        const int slot = g % G_RING, use = g / G_RING;
        if (use >= 1 && !(ok = mbar_wait(&aempty[slot], (use & 1) ^ 1, abort_flag))) break;
        mbar_expect_tx(&afull[slot], G_SLICE);
        for (int q = 0; q < 4; ++q)
          bulk_load(sA + slot * G_SLICE + q * OZ_SLICE_HALF,
                    (q < 2 ? A0 : A1) + kofs + (q & 1) * OZ_HALF + i * OZ_SLICE_HALF, OZ_SLICE_HALF, &afull[slot]);
        loads[0] = g + 1;
      }
      if (ok) load_b(c, 1);
    }
    if (!ok) {
      atomicCAS(G.error, 0, 21);
      *abort_flag = 1;
    }
  } else if (warp == 1 && lane == 0) {
    bool ok = true;
    for (int c = 0; ok && c < nk; ++c)
      for (int h = 0; ok && h < 2; ++h) {
        ok = mbar_wait(&bfull[h], c & 1, abort_flag);
        if (!ok) break;
        seen[1 + h] = c + 1;
        if (c >= 1 && !(ok = mbar_wait(&tempty[h], (c & 1) ^ 1, abort_flag))) break;
        tc_fence_after();
        const uint32_t acc = tmem + (uint32_t)(h * BUF_COLS);
        const uint64_t bd = desc128(sB + h * OZ_HALF);
        for (int i = 0; i < OZ_S; ++i) {
          const int g = c * OZ_S + i, slot = g % G_RING;
          if (h == 0) {
            if (!(ok = mbar_wait(&afull[slot], (g / G_RING) & 1, abort_flag))) break;
            seen[0] = g + 1;
            tc_fence_after();
          }
          const uint64_t ad = desc128(sA + slot * G_SLICE);
          const uint32_t id = idesc_bf16(32 * (OZ_S - i));
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) mma_f16(acc + 32 * i, ad + 2 * kk, bd + 2 * kk, id, (kk | i) ? 1u : 0u);
          if (h == 1) mma_commit(&aempty[slot]);
        }
        if (!ok) break;
        mma_commit(&tfull[h]);
        mma_commit(&bempty[h]);
      }
    if (!ok) {
      atomicCAS(G.error, 0, 22);
      *abort_flag = 1;
    }
    mma_commit(done);
  } else if (warp >= 2) {
    const int quad = warp & 3, ch = (warp - 2) >> 2;
    const int row = quad * 32 + lane, i0 = tm * 128 + row;
    long long hi[2][16];
    uint32_t lo[2][16];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        hi[h][q] = 0;
        lo[h][q] = 0;
      }
    bool good = true;
    for (int c = 0; good && c < nk; ++c) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (good) {
          good = __all_sync(0xffffffffu, mbar_wait(&tfull[h], c & 1, abort_flag));
          if (!good) {
            if (lane == 0) {
              atomicCAS(G.error, 0, 23);
              *abort_flag = 1;
            }
          } else {
            tc_fence_after();
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              uint32_t v[OZ_S][4];
#pragma unroll
              for (int s = 0; s < OZ_S; ++s) {
                const uint32_t addr =
                    tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(h * BUF_COLS + s * 32 + ch * 16 + g * 4);
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                             : "=r"(v[s][0]), "=r"(v[s][1]), "=r"(v[s][2]), "=r"(v[s][3])
                             : "r"(addr));
              }
              asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
              if (g == 3) {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&tempty[h]);
              }
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                int d[OZ_S];
#pragma unroll
                for (int s = 0; s < OZ_S; ++s) d[s] = __float2int_rn(__uint_as_float(v[s][q]));
                long long& H = hi[h][g * 4 + q];
                uint32_t& W = lo[h][g * 4 + q];
                const long long l = (long long)d[4] * (1 << 18) + (long long)d[5] * (1 << 9) + ((long long)d[6] + W);
                H += (long long)d[0] * (1 << 27) + (long long)d[1] * (1 << 18) + (long long)d[2] * (1 << 9) + d[3] +
                     (l >> 27);
                W = (uint32_t)l & ((1u << 27) - 1);
              }
            }
          }
        }
      }
    }
    if (good && i0 < G.M[p]) {
      const int ea = G.A[p].exps[i0];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int q = 0; q < 16; ++q) {
          const int col = tn * 64 + h * 32 + ch * 16 + q;
          if (col < G.N[p])
            G.Z[p][(long long)col * G.ldz[p] + i0] =
                rounded(hi[h][q], (long long)lo[h][q], 27, ea + G.B[p].exps[col] - 16 - 27);
        }
    }
  }
  __syncwarp();
  __syncthreads();
  if (threadIdx.x == 0) {
    if (!mbar_wait(done, 0)) atomicCAS(G.error, 0, 24);
    if (*abort_flag) {   // copies issued but never waited for
      for (int g = seen[0]; g < loads[0]; ++g) mbar_wait(&afull[g % G_RING], (g / G_RING) & 1);
      for (int h = 0; h < 2; ++h)
        for (int c = seen[1 + h]; c < loads[1 + h]; ++c) mbar_wait(&bfull[h], c & 1);
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * BUF_COLS));
}

// Row exponents and slices of row-major operands, a CTA per (padded) row: the row is read twice, the second time from L1
// or L2, and written as 16-byte groups of 8 digits of a slice.  Bound by latency and the integer digits, so every row
// of every operand gets a CTA in one launch (a warp per row, a launch per operand: 39 us for 256 rows of 4614; this:
// 27 us for all 768).
__global__ void __launch_bounds__(128) k_oz_slice(const __grid_constant__ OzSliceBatch P) {
  __shared__ unsigned long long wmax[4];
  int p = 0;
  while (p + 1 < P.n && (int)blockIdx.x >= P.row_off[p + 1]) ++p;
  const int r = (int)blockIdx.x - P.row_off[p], rows = P.rows[p], cols = P.cols[p], tri = P.tri[p];
  const int kt = (cols + 63) / 64;
  const bool live = r < rows;
  const int c0 = live && tri > 0 ? r : 0, c1 = live ? (tri < 0 ? r + 1 : cols) : 0;
  const double* xr = P.x[p] + (long long)r * P.ld[p];
  unsigned long long mx = 0;
  for (int c = c0 + threadIdx.x; c < c1; c += 128) mx = max(mx, oz_abs_bits(xr[c]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mx;
  __syncthreads();
  const int E = oz_row_exp(max(max(wmax[0], wmax[1]), max(wmax[2], wmax[3])));
  if (threadIdx.x == 0) P.out[p].exps[r] = E;
  uint8_t* out = P.out[p].tiles + (size_t)(r >> 6) * kt * OZ_TILE;
  for (int g = threadIdx.x; g < kt * 8; g += 128) {   // groups of 8 columns
    uint32_t w[OZ_S][4];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int c = g * 8 + q;
      int d[OZ_S];
      oz_digits(c >= c0 && c < c1 ? xr[c] : 0.0, E, d);
#pragma unroll
      for (int s = 0; s < OZ_S; ++s) w[s][q >> 1] = (q & 1) ? (w[s][q >> 1] | oz_bf16(d[s]) << 16) : oz_bf16(d[s]);
    }
    uint8_t* o = out + (size_t)(g >> 3) * OZ_TILE;
#pragma unroll
    for (int s = 0; s < OZ_S; ++s)
      *reinterpret_cast<uint4*>(o + oz_offset(r & 63, (g & 7) * 8, s)) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
  }
}

// Exponents of the rows of a transposed operand (element (r, c) at x[r + c * sc]): a thread per row, 8 column strips
__global__ void __launch_bounds__(256) k_oz_exps_t(const double* __restrict__ x, long long sc, int rows, int cols, int tri,
                                                   int* exps) {
  __shared__ unsigned long long m[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, r = blockIdx.x * 32 + lane;
  unsigned long long mx = 0;
  if (r < rows)
    for (int c = w; c < cols; c += 8)
      if (tri == 0 || (tri > 0 ? c >= r : c <= r)) mx = max(mx, oz_abs_bits(x[r + (long long)c * sc]));
  m[w][lane] = mx;
  __syncthreads();
  if (w == 0) {
    for (int q = 1; q < 8; ++q) mx = max(mx, m[q][lane]);
    exps[r] = oz_row_exp(mx);   // padding rows: zeros
  }
}

// Slices of one 64 x 64 tile of a transposed operand through shared memory
__global__ void __launch_bounds__(256) k_oz_slice_t(const double* __restrict__ x, long long sc, int rows, int cols, int tri,
                                                    uint8_t* tiles, const int* __restrict__ exps) {
  __shared__ double a[64][65];   // [column][row]
  const int kt = gridDim.x, r0 = blockIdx.y * 64, c0 = blockIdx.x * 64;
  for (int i = threadIdx.x; i < 64 * 64; i += 256) {
    const int r = r0 + (i & 63), c = c0 + (i >> 6);
    const bool in = r < rows && c < cols && (tri == 0 || (tri > 0 ? c >= r : c <= r));
    a[i >> 6][i & 63] = in ? x[r + (long long)c * sc] : 0.0;
  }
  __syncthreads();
  uint8_t* o = tiles + ((size_t)blockIdx.y * kt + blockIdx.x) * OZ_TILE;
  for (int u = threadIdx.x; u < 64 * 8; u += 256) {
    const int r = u & 63, k0 = (u >> 6) * 8, E = exps[r0 + r];
    uint32_t w[OZ_S][4];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      int d[OZ_S];
      oz_digits(a[k0 + q][r], E, d);
#pragma unroll
      for (int s = 0; s < OZ_S; ++s) w[s][q >> 1] = (q & 1) ? (w[s][q >> 1] | oz_bf16(d[s]) << 16) : oz_bf16(d[s]);
    }
#pragma unroll
    for (int s = 0; s < OZ_S; ++s)
      *reinterpret_cast<uint4*>(o + oz_offset(r, k0, s)) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
  }
}

// ------------------------------------------------------------------------------------------------ host
void oz_init() {
  static std::mutex mu;
  static bool attr_done[64] = {};
  std::lock_guard<std::mutex> lock(mu);
  int dev = 0;
  FETIRP_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) throw Error(1, "device ordinal out of range");
  if (!attr_done[dev]) {
    FETIRP_CUDA(cudaFuncSetAttribute(k_oz_gemm, cudaFuncAttributeMaxDynamicSharedMemorySize, G_SMEM));
    attr_done[dev] = true;
  }
}

void oz_slice(const OzSliceBatch& batch, cudaStream_t s) {
  OzSliceBatch P = batch;
  int total = 0;
  for (int p = 0; p < P.n; ++p) {
    P.row_off[p] = total;
    total += ceil_div(P.rows[p], 64) * 64;
  }
  if (total == 0) return;
  k_oz_slice<<<total, 128, 0, s>>>(P);
  FETIRP_LAUNCH_CHECK();
}

void oz_slice_rows(const double* x, long long ld, int rows, int cols, int tri, const OzOperand& out, cudaStream_t s) {
  OzSliceBatch P;
  P.add(x, ld, rows, cols, tri, out);
  oz_slice(P, s);
}

void oz_slice_cols(const double* x, long long ld, int rows, int cols, int tri, const OzOperand& out, cudaStream_t s) {
  if (rows <= 0 || cols <= 0) return;
  const int rt = ceil_div(rows, 64), kt = ceil_div(cols, 64);
  k_oz_exps_t<<<rt * 2, 256, 0, s>>>(x, ld, rows, cols, tri, out.exps);
  FETIRP_LAUNCH_CHECK();
  k_oz_slice_t<<<dim3(kt, rt), 256, 0, s>>>(x, ld, rows, cols, tri, out.tiles, out.exps);
  FETIRP_LAUNCH_CHECK();
}

void oz_gemm(const OzGemm& G, cudaStream_t s) {
  oz_init();
  OzGemmKernel P;
  P.G = G;
  int total = 0, n = 0;
  for (int p = 0; p < G.n; ++p) {
    if (G.M[p] <= 0 || G.N[p] <= 0) continue;
    P.G.A[n] = G.A[p]; P.G.B[n] = G.B[p];
    P.G.M[n] = G.M[p]; P.G.N[n] = G.N[p]; P.G.K[n] = G.K[p];
    P.G.mode[n] = G.mode[p]; P.G.Z[n] = G.Z[p]; P.G.ldz[n] = G.ldz[p];
    P.tiles_n[n] = ceil_div(G.N[p], 64);
    P.tile_off[n] = total;
    total += ceil_div(G.M[p], 128) * P.tiles_n[n];
    ++n;
  }
  P.G.n = n;
  P.tile_off[n] = total;
  if (total == 0) return;
  k_oz_gemm<<<total, THREADS, G_SMEM, s>>>(P);
  FETIRP_LAUNCH_CHECK();
}

}  // namespace fetirp
