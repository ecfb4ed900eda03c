// FP64 products on the tensor cores by exact digit slices (see oz.cuh).
#include <algorithm>
#include <mutex>

#include "oz.cuh"
#include "tc_ptx.cuh"

namespace fetirp {

namespace {

constexpr int THREADS = 320;                         // producer warp, MMA warp, 8 epilogue warps
constexpr int EPI_WARPS = 8, EPI_COLS = OZ_COLS / (EPI_WARPS / 4);   // a warp's columns of its 32 rows
constexpr int TMEM_COLS = 512;                       // 7 levels of 64 used

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

constexpr int G_A = 2 * OZ_SLICE;                       // an A slice of 128 rows: 16 KB
constexpr int G_ZEROS = OZ_PAD * OZ_SLICE;              // zero slices in front of B
constexpr int G_B = G_ZEROS + OZ_TILE;
constexpr int G_SMEM = OZ_RING * G_A + G_B + 1024 + 512;
static_assert(G_SMEM <= 227 * 1024, "shared memory of a CTA");

struct OzGemmKernel {
  OzGemm G;
  int tiles_n[OZ_MAXP], tile_off[OZ_MAXP + 1];
};
}  // namespace

// One CTA: 128 rows of A (two row tiles) against 64 rows of B, all of K in 64-wide blocks.  Bound by the MMAs (28 digit pairs,
// i + j <= 6: over a long row the dropped products stay far below the rounding of an FP64 chain, and the zero slices that
// keep one shape per accumulator, oz_plan.cuh).  FP64 apply of three 16^3 elastic patterns (n_b = 4614, 256 right-hand
// sides each, 32.7 GFLOP): 27.5 ms with FP64 FMAs, 0.97 ms so, and its error against 64 bits is the same (2.2e-10 of the
// projected result, which is that of S^+).  The two groups of levels have an accumulator each (256 and 192 TMEM columns): one
// is drained while the other is multiplied.  Drained levels are added into 91-bit integers per output (a 64-bit and a
// 27-bit part): no FP64 operation before the final rounding.
__global__ void __launch_bounds__(THREADS, 1) k_oz_gemm(const __grid_constant__ OzGemmKernel P) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + OZ_RING * G_A + G_ZEROS;
  uint64_t* afull = reinterpret_cast<uint64_t*>(sB + OZ_TILE);   // [OZ_RING], by slot
  uint64_t* aempty = afull + OZ_RING;
  uint64_t* bfull = aempty + OZ_RING;                            // [OZ_S], by slice
  uint64_t* tfull = bfull + OZ_S;                                // [2], by group of levels
  uint64_t* tempty = tfull + 2;
  uint64_t* done = tempty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* n_loads = abort_flag + 1;   // copies issued

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
    for (int i = 0; i < 2 * OZ_RING + OZ_S; ++i) mbar_init(&afull[i], 1);   // afull .. bfull
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], EPI_WARPS);
    }
    mbar_init(done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int i = threadIdx.x; i < G_ZEROS / 16; i += THREADS)   // never written again
    *reinterpret_cast<uint4*>(sB - G_ZEROS + i * 16) = make_uint4(0, 0, 0, 0);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // before the MMAs read them
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  if (warp == 0 && lane == 0) {
    const uint8_t* A0 = G.A[p].tiles + ((size_t)a0 * kt + kb) * OZ_TILE;
    const uint8_t* A1 = G.A[p].tiles + ((size_t)a1 * kt + kb) * OZ_TILE;
    const uint8_t* B = G.B[p].tiles + ((size_t)tn * kt + kb) * OZ_TILE;
    bool ok = true;
    int last = -1;   // copies issued so far
    for (int c = 0; ok && c < nk; ++c) {
      const size_t kofs = (size_t)c * OZ_TILE;
#pragma unroll
      for (int o = 0; o < OZ_LOADS; ++o) {
        const OzLoad L = oz_load(o);
        if (L.a >= 0) {
          const int slot = oz_slot(c, oz_place(L.a)), use = oz_use(c, L.a);
          if (use >= 1 && !(ok = mbar_wait(&aempty[slot], (use & 1) ^ 1, abort_flag))) break;
          mbar_expect_tx(&afull[slot], G_A);
          bulk_load(sA + slot * G_A, A0 + kofs + L.a * OZ_SLICE, OZ_SLICE, &afull[slot]);
          bulk_load(sA + slot * G_A + OZ_SLICE, A1 + kofs + L.a * OZ_SLICE, OZ_SLICE, &afull[slot]);
        } else {
          // the MMA that gave up B's last slices also gave up A slice 0; those of the slices before were waited for with A
          if (L.b == OZ_LOW && c >= 1 &&
              !(ok = mbar_wait(&aempty[oz_slot(c - 1, oz_place(0))], oz_use(c - 1, 0) & 1, abort_flag)))
            break;
          mbar_expect_tx(&bfull[L.b], OZ_SLICE);
          bulk_load(sB + L.b * OZ_SLICE, B + kofs + L.b * OZ_SLICE, OZ_SLICE, &bfull[L.b]);
        }
        last = c * OZ_LOADS + o;
      }
    }
    if (!ok) {
      atomicCAS(G.error, 0, 21);
      *abort_flag = 1;
    }
    *n_loads = last + 1;
  } else if (warp == 1 && lane == 0) {
    bool ok = true;
    for (int c = 0; ok && c < nk; ++c) {
#pragma unroll
      for (int q = 0; q < OZ_MMAS; ++q) {   // unrolled: the one thread's instructions are on the critical path
        const OzMma M = oz_mma(q);
        const int group = q < OZ_LOW ? 0 : 1;
        const int slot = oz_slot(c, oz_place(M.a));
        if (M.first && c >= 1 && !(ok = mbar_wait(&tempty[group], (c & 1) ^ 1, abort_flag))) break;
        if ((group == 0 || M.a >= OZ_LOW) &&   // the block's first use of the slice
            !(ok = mbar_wait(&afull[slot], oz_use(c, M.a) & 1, abort_flag)))
          break;
        if (M.new_b >= 0 && !(ok = mbar_wait(&bfull[M.new_b], c & 1, abort_flag))) break;
        tc_fence_after();
        const uint64_t ad = desc128(sA + slot * G_A), bd = desc128(sB + M.b * OZ_SLICE);
        const uint32_t id = idesc_bf16(M.n);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_f16(tmem + M.col, ad + 2 * kk, bd + 2 * kk, id, (kk || !M.first) ? 1u : 0u);
        if (group == 1) mma_commit(&aempty[slot]);
        if (q == OZ_LOW - 1) mma_commit(&tfull[0]);
      }
      if (!ok) break;
      mma_commit(&tfull[1]);
    }
    if (!ok) {
      atomicCAS(G.error, 0, 22);
      *abort_flag = 1;
    }
    mma_commit(done);
  } else if (warp >= 2) {
    const int quad = warp & 3, c0 = ((warp - 2) >> 2) * EPI_COLS;
    const int row = quad * 32 + lane, i0 = tm * 128 + row;
    const uint32_t tbase = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)c0;
    long long hi[EPI_COLS];
    uint32_t lo[EPI_COLS];
#pragma unroll
    for (int q = 0; q < EPI_COLS; ++q) {
      hi[q] = 0;
      lo[q] = 0;
    }
    bool good = true;
    for (int c = 0; good && c < nk; ++c) {
#pragma unroll
      for (int group = 0; group < 2; ++group) {
        if (!good) break;
        good = __all_sync(0xffffffffu, mbar_wait(&tfull[group], c & 1, abort_flag));
        if (!good) {
          if (lane == 0) {
            atomicCAS(G.error, 0, 23);
            *abort_flag = 1;
          }
          break;
        }
        tc_fence_after();
        const int l0 = group == 0 ? 0 : OZ_LOW, l1 = group == 0 ? OZ_LOW : OZ_S;
#pragma unroll
        for (int g = 0; g < EPI_COLS / 8; ++g) {
          uint32_t v[OZ_LOW][8];
#pragma unroll
          for (int l = l0; l < l1; ++l) tmem_ld8(v[l - l0], tbase + (uint32_t)(l * OZ_COLS + g * 8));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (g == EPI_COLS / 8 - 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&tempty[group]);
          }
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            int d[OZ_LOW];
#pragma unroll
            for (int l = 0; l < l1 - l0; ++l) d[l] = __float2int_rn(__uint_as_float(v[l][q]));
            long long& X = hi[g * 8 + q];
            uint32_t& W = lo[g * 8 + q];
            if (group == 0) {
              X += (long long)d[0] * (1 << 27) + (long long)d[1] * (1 << 18) + (long long)d[2] * (1 << 9) + d[3];
            } else {
              const long long l = (long long)d[0] * (1 << 18) + (long long)d[1] * (1 << 9) + ((long long)d[2] + W);
              X += l >> 27;
              W = (uint32_t)l & ((1u << 27) - 1);
            }
          }
        }
      }
    }
    if (good && i0 < G.M[p]) {
      const int ea = G.A[p].exps[i0];
#pragma unroll
      for (int q = 0; q < EPI_COLS; ++q) {
        const int col = tn * 64 + c0 + q;
        if (col < G.N[p])
          G.Z[p][(long long)col * G.ldz[p] + i0] = rounded(hi[q], (long long)lo[q], 27, ea + G.B[p].exps[col] - 16 - 27);
      }
    }
  }
  __syncwarp();
  __syncthreads();
  if (threadIdx.x == 0) {
    if (!mbar_wait(done, 0)) atomicCAS(G.error, 0, 24);
    if (*abort_flag) {   // the last copy into every slot and slice, which nobody may have waited for
      unsigned waited = 0;
      for (int n = *n_loads - 1; n >= max(0, *n_loads - 2 * OZ_LOADS); --n) {
        const int c = n / OZ_LOADS;
        const OzLoad L = oz_load(n % OZ_LOADS);
        const int bar = L.a >= 0 ? oz_slot(c, oz_place(L.a)) : 2 * OZ_RING + L.b;   // aempty lies between
        if (waited >> bar & 1u) continue;
        waited |= 1u << bar;
        mbar_wait(&afull[bar], (L.a >= 0 ? oz_use(c, L.a) : c) & 1);
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
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
