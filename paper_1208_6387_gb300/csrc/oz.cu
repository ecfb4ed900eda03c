// FP64 products on the tensor cores by exact digit slices (see oz.cuh).
#include <algorithm>
#include <mutex>

#include "oz.cuh"
#include "tc_ptx.cuh"

namespace fetirp {

namespace {

constexpr int THREADS = 320;                         // producer warp, MMA warp, 8 epilogue warps
constexpr int EPI_WARPS = 8, EPI_COLS = OZ_COLS / (EPI_WARPS / 4);   // a warp's columns of its 32 rows
constexpr int TMEM_COLS = 512;                       // 7 levels and the magnitudes, 64 each

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
// addition costs more than this whole routine on the integer pipe.  normal: the result is zero or a normal number.
__device__ __forceinline__ double scaled_i64(long long v, int q, bool* normal) {
  const bool neg = v < 0;
  unsigned long long a = neg ? 0ull - (unsigned long long)v : (unsigned long long)v;
  *normal = true;
  if (a == 0) return 0.0;
  const int n = __clzll((long long)a);
  a <<= n;
  const int be = 1023 + 63 + q - n;
  *normal = be >= 1 && be <= 2045;
  const unsigned long long r = ((unsigned long long)(uint32_t)(be - 1) << 52) + (a >> 11) + ((a >> 10) & 1ull);
  return __longlong_as_double((long long)(r | (neg ? 1ull << 63 : 0ull)));
}

// (hi + lo 2^-w) 2^e in FP64, one rounding after at least 62 significant bits; |lo| < 2^(w + 17)
__device__ __forceinline__ double rounded(long long hi, long long lo, int w, int e, bool* normal) {
  const long long ah = hi < 0 ? -hi : hi;
  const int room = min(w, __clzll(ah) - 2);   // as many of lo's bits as hi leaves room for
  return scaled_i64((hi << room) + (lo >> (w - room)), e - room, normal);
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
// the magnitudes, and the zero slices that keep one shape per accumulator, oz_plan.cuh) and the hand-over of the
// accumulators.  FP64 apply of three 16^3 elastic patterns (n_b = 4614, 256 right-hand sides each, 32.7 GFLOP): 27.5 ms with
// FP64 FMAs, 1.08 ms so (0.97 without the magnitudes; this kernel 0.86), and its error against 64 bits is the same
// (2.2e-10 of the projected result, which is that of S^+).  The two groups of levels have an accumulator each (256 and 192
// TMEM columns): one is drained while the other is multiplied.  Drained levels are added into 91-bit integers per
// output (a 64-bit and a 27-bit part): no FP64 operation before the final rounding.
__global__ void __launch_bounds__(THREADS, 1) k_oz_gemm(const __grid_constant__ OzGemmKernel P) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + OZ_RING * G_A + G_ZEROS;
  uint64_t* afull = reinterpret_cast<uint64_t*>(sB + OZ_TILE);   // [OZ_RING], by slot
  uint64_t* aempty = afull + OZ_RING;
  uint64_t* bfull = aempty + OZ_RING;                            // [OZ_SLICES], by slice
  uint64_t* tfull = bfull + OZ_SLICES;                           // [2], by group of levels
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
    for (int i = 0; i < 2 * OZ_RING + OZ_SLICES; ++i) mbar_init(&afull[i], 1);   // afull .. bfull
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
    const OzRow r0 = oz_row(G.mode[p], a0, kt), r1 = oz_row(G.mode[p], a1, kt);
    const uint8_t* A0 = G.A[p].tiles + (size_t)(r0.begin + kb - r0.first) * OZ_TILE;
    const uint8_t* A1 = G.A[p].tiles + (size_t)(r1.begin + kb - r1.first) * OZ_TILE;
    const uint8_t* B = G.B[p].tiles + ((size_t)tn * kt + kb) * OZ_TILE;
    bool ok = true;
    int last = -1;   // copies issued so far
    for (int c = 0; ok && c < nk; ++c) {
      const size_t kofs = (size_t)c * OZ_TILE;
#pragma unroll
      for (int o = 0; o < OZ_LOADS; ++o) {
        const OzLoad L = oz_load(o);
        if (L.a >= 0) {
          const int slot = oz_slot(c, oz_place(L.a));   // every slot is used once a block
          if (c >= 1 && !(ok = mbar_wait(&aempty[slot], (c & 1) ^ 1, abort_flag))) break;
          mbar_expect_tx(&afull[slot], G_A);
          bulk_load(sA + slot * G_A, A0 + kofs + L.a * OZ_SLICE, OZ_SLICE, &afull[slot]);
          bulk_load(sA + slot * G_A + OZ_SLICE, A1 + kofs + L.a * OZ_SLICE, OZ_SLICE, &afull[slot]);
        } else {
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
        const int group = q < OZ_LOW ? 0 : 1;   // (the magnitudes are committed with the second one)
        const int slot = oz_slot(c, oz_place(M.a));
        if (M.first && c >= 1 && !(ok = mbar_wait(&tempty[group], (c & 1) ^ 1, abort_flag))) break;
        if ((group == 0 || M.a >= OZ_LOW) &&   // the block's first use of the slice
            !(ok = mbar_wait(&afull[slot], c & 1, abort_flag)))
          break;
        if (M.new_b >= 0 && !(ok = mbar_wait(&bfull[M.new_b], c & 1, abort_flag))) break;
        tc_fence_after();
        const uint64_t ad = desc128(sA + slot * G_A), bd = desc128(sB + M.b * OZ_SLICE);
        const uint32_t id = idesc_bf16(M.n);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
          mma_f16(tmem + M.col, ad + 2 * kk, bd + 2 * kk, id, kk > 0 || (M.whole ? c > 0 : !M.first) ? 1u : 0u);
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
    static_assert(EPI_COLS <= 32, "a bit per column");
    uint32_t large = 0;   // columns with a level sum that FP32 may have rounded
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
              const float top = fmaxf(fmaxf(fabsf(__uint_as_float(v[0][q])), fabsf(__uint_as_float(v[1][q]))),
                                      fabsf(__uint_as_float(v[2][q])));
              if (top >= 16777216.f) large |= 1u << (g * 8 + q);
              const long long l = (long long)d[0] * (1 << 18) + (long long)d[1] * (1 << 9) + ((long long)d[2] + W);
              X += l >> 27;
              W = (uint32_t)l & ((1u << 27) - 1);
            }
          }
        }
      }
    }
    if (good) {
      const bool in = i0 < G.M[p];
      const int ea = G.A[p].exps[in ? i0 : 0];
      const float line = sqrtf(64.f * nk) * 0x1p-8f;   // see oz.cuh
      uint32_t word = 0;                               // lane q's: the rows of column q that FMAs compute
#pragma unroll
      for (int g = 0; g < EPI_COLS / 8; ++g) {
        uint32_t mag[8];
        tmem_ld8(mag, tbase + (uint32_t)(OZ_S * OZ_COLS + g * 8));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int q = g * 8 + u, col = tn * 64 + c0 + q;
          const int eb = G.B[p].exps[col];   // padded to 64 rows
          bool normal;
          const double z = rounded(hi[q], (long long)lo[q], 27, ea + eb - 16 - 27, &normal);
          const bool zero = (ea == OZ_E_ZERO && eb != OZ_E_BAD) || (eb == OZ_E_ZERO && ea != OZ_E_BAD);
          const bool fma_it = !zero && (!(__uint_as_float(mag[u]) >= line) || !normal || (large >> q & 1u));
          const uint32_t rows = __ballot_sync(0xffffffffu, in && fma_it);
          if (lane == q) word = rows;
          if (in && col < G.N[p]) G.Z[p][(long long)col * G.ldz[p] + i0] = z;
        }
      }
      const int col = tn * 64 + c0 + lane, mw = (G.M[p] + 31) / 32, wr = tm * 4 + quad;
      if (lane < EPI_COLS && col < G.N[p] && wr < mw) G.flags[p][(long long)col * mw + wr] = word;
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
        mbar_wait(&afull[bar], c & 1);
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS));
}

// The outputs that k_oz_gemm left to FMAs.  A thread per flag word looks for them (words of neighbouring threads lie a
// grid apart, so that a flagged column or row spreads over the CTAs); the CTA's warps then take its words in turn: four rows
// at a time and eight j where A's columns are contiguous (32 bytes a column), else row by row, 32 j.  Bound by the FP64 pipe
// where there are any (Lam and Lam^T on three 16^3 patterns, 64 right-hand sides each: 1.2 ms for both products; with the
// line of oz.cuh at 2^-7 2.3 ms, and 6.5 ms on 109 CTAs that took whole words), else by its launch (4 us).
constexpr int FIX_THREADS = 256;
struct OzFix {
  OzGemm G;
  long long word_off[OZ_MAXP + 1];
};
__global__ void __launch_bounds__(FIX_THREADS) k_oz_fix(const __grid_constant__ OzFix P) {
  __shared__ int n_words;
  __shared__ uint32_t todo[FIX_THREADS];      // flag words
  __shared__ long long where[FIX_THREADS];    // and their indices
  const OzGemm& G = P.G;
  const int tid = threadIdx.x, lane = tid & 31;
  const long long total = P.word_off[G.n];
  for (long long base = 0; base < total; base += (long long)gridDim.x * FIX_THREADS) {
    const long long idx = base + blockIdx.x + (long long)gridDim.x * tid;
    int p = 0;
    if (tid == 0) n_words = 0;
    __syncthreads();
    if (idx < total) {
      while (p + 1 < G.n && idx >= P.word_off[p + 1]) ++p;
      const uint32_t w = G.flags[p][idx - P.word_off[p]];
      if (w) {
        const int at = atomicAdd(&n_words, 1);
        todo[at] = w;
        where[at] = idx;
      }
    }
    __syncthreads();
    const int n = n_words;
    for (int it = tid >> 5; it < n; it += FIX_THREADS / 32) {
      uint32_t w = todo[it];
      const long long at = where[it];
      p = 0;
      while (p + 1 < G.n && at >= P.word_off[p + 1]) ++p;
      const int M = G.M[p], K = G.K[p], mode = G.mode[p], mw = (M + 31) / 32;
      const int c = (int)((at - P.word_off[p]) / mw), r0 = (int)((at - P.word_off[p]) % mw) * 32;
      if (M - r0 < 32) w &= (1u << (M - r0)) - 1;   // set for real rows only, unless the product gave up
      const double* b = G.b[p] + (long long)c * G.ldb[p];
      double* z = G.Z[p] + (long long)c * G.ldz[p];
      if (G.aj[p] != 1) {
        const int jl = lane >> 2;
        for (int g = 0; g < 32; g += 4) {
          if (!(w >> g & 15u)) continue;
          const int i = min(r0 + g + (lane & 3), M - 1);
          const double* a = G.a[p] + i;
          const int j0 = mode == 2 ? i : 0, j1 = mode == 1 ? i + 1 : K;
          double s[4] = {0.0, 0.0, 0.0, 0.0};
          for (int j = j0 + jl; j < j1; j += 32) {
            double x[4], y[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const bool in = j + 8 * u < j1;
              x[u] = in ? a[(long long)(j + 8 * u) * G.aj[p]] : 0.0;
              y[u] = in ? b[j + 8 * u] : 0.0;
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) s[u] = fma(x[u], y[u], s[u]);
          }
          double v = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
          for (int o = 16; o > 2; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          if (lane < 4 && (w >> (g + lane) & 1u)) z[i] = v;
        }
        continue;
      }
      while (w) {
        const int i = r0 + __ffs(w) - 1;
        w &= w - 1;
        const double* a = G.a[p] + (long long)i * G.ai[p];
        const int j0 = mode == 2 ? i : 0, j1 = mode == 1 ? i + 1 : K;
        double s[4] = {0.0, 0.0, 0.0, 0.0};
        for (int j = j0 + lane; j < j1; j += 128)
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (j + 32 * u < j1) s[u] = fma(a[j + 32 * u], b[j + 32 * u], s[u]);
        double v = (s[0] + s[1]) + (s[2] + s[3]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) z[i] = v;
      }
    }
    __syncthreads();   // the list is read before the next one
  }
}

// The digits and the magnitude of entry q of a group of eight, two entries a word
__device__ __forceinline__ void put_entry(double x, int E, int q, uint32_t (&w)[OZ_SLICES][4]) {
  int d[OZ_S];
  oz_digits(x, E, d);
#pragma unroll
  for (int s = 0; s < OZ_SLICES; ++s) {
    const uint32_t v = s == OZ_MAG ? oz_magnitude(x, E) : oz_bf16(d[s < OZ_S ? s : 0]);
    w[s][q >> 1] = (q & 1) ? (w[s][q >> 1] | v << 16) : v;
  }
}

// Row exponents and slices of row-major operands, a CTA per (padded) row: the row is read twice, the second time from L1
// or L2, and written as 16-byte groups of 8 digits of a slice.  Bound by latency and the integer digits, so every row
// of every operand gets a CTA in one launch (a warp per row, a launch per operand: 39 us for 256 rows of 4614; this:
// 28 us for all 768).
__global__ void __launch_bounds__(128) k_oz_slice(const __grid_constant__ OzSliceBatch P) {
  __shared__ unsigned long long wmax[4];
  int p = 0;
  while (p + 1 < P.n && (int)blockIdx.x >= P.row_off[p + 1]) ++p;
  const int r = (int)blockIdx.x - P.row_off[p], rows = P.rows[p], cols = P.cols[p], mode = P.mode[p];
  const int kt = (cols + 63) / 64;
  const bool live = r < rows;
  const int c0 = live && mode == 2 ? r : 0, c1 = live ? (mode == 1 ? r + 1 : cols) : 0;
  const double* xr = P.x[p] + (long long)r * P.ld[p];
  unsigned long long mx = 0;
  for (int c = c0 + threadIdx.x; c < c1; c += 128) mx = max(mx, oz_abs_bits(xr[c]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if ((threadIdx.x & 31) == 0) wmax[threadIdx.x >> 5] = mx;
  __syncthreads();
  const int E = oz_row_exp(max(max(wmax[0], wmax[1]), max(wmax[2], wmax[3])));
  if (threadIdx.x == 0) P.out[p].exps[r] = E;
  const OzRow tr = oz_row(mode, r >> 6, kt);
  uint8_t* out = P.out[p].tiles + (size_t)tr.begin * OZ_TILE;
  for (int g = tr.first * 8 + threadIdx.x; g < tr.last * 8; g += 128) {   // groups of 8 columns
    uint32_t w[OZ_SLICES][4];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int c = g * 8 + q;
      put_entry(c >= c0 && c < c1 ? xr[c] : 0.0, E, q, w);
    }
    uint8_t* o = out + (size_t)((g >> 3) - tr.first) * OZ_TILE;
#pragma unroll
    for (int s = 0; s < OZ_SLICES; ++s)
      *reinterpret_cast<uint4*>(o + oz_offset(r & 63, (g & 7) * 8, s)) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
  }
}

// Exponents of the rows of a transposed operand (element (r, c) at x[r + c * sc]): a thread per row, 8 column strips
__global__ void __launch_bounds__(256) k_oz_exps_t(const double* __restrict__ x, long long sc, int rows, int cols, int mode,
                                                   int* exps) {
  __shared__ unsigned long long m[8][32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, r = blockIdx.x * 32 + lane;
  unsigned long long mx = 0;
  if (r < rows)
    for (int c = w; c < cols; c += 8)
      if (mode == 0 || (mode == 2 ? c >= r : c <= r)) mx = max(mx, oz_abs_bits(x[r + (long long)c * sc]));
  m[w][lane] = mx;
  __syncthreads();
  if (w == 0) {
    for (int q = 1; q < 8; ++q) mx = max(mx, m[q][lane]);
    exps[r] = oz_row_exp(mx);   // padding rows: zeros
  }
}

// Slices of one 64 x 64 tile of a transposed operand through shared memory
__global__ void __launch_bounds__(256) k_oz_slice_t(const double* __restrict__ x, long long sc, int rows, int cols, int mode,
                                                    uint8_t* tiles, const int* __restrict__ exps) {
  __shared__ double a[64][65];   // [column][row]
  const int kt = gridDim.x, r0 = blockIdx.y * 64, c0 = blockIdx.x * 64;
  const OzRow tr = oz_row(mode, blockIdx.y, kt);
  if ((int)blockIdx.x < tr.first || (int)blockIdx.x >= tr.last) return;
  for (int i = threadIdx.x; i < 64 * 64; i += 256) {
    const int r = r0 + (i & 63), c = c0 + (i >> 6);
    const bool in = r < rows && c < cols && (mode == 0 || (mode == 2 ? c >= r : c <= r));
    a[i >> 6][i & 63] = in ? x[r + (long long)c * sc] : 0.0;
  }
  __syncthreads();
  uint8_t* o = tiles + (size_t)(tr.begin + blockIdx.x - tr.first) * OZ_TILE;
  for (int u = threadIdx.x; u < 64 * 8; u += 256) {
    const int r = u & 63, k0 = (u >> 6) * 8, E = exps[r0 + r];
    uint32_t w[OZ_SLICES][4];
#pragma unroll
    for (int q = 0; q < 8; ++q) put_entry(a[k0 + q][r], E, q, w);
#pragma unroll
    for (int s = 0; s < OZ_SLICES; ++s)
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

void oz_slice_rows(const double* x, long long ld, int rows, int cols, int mode, const OzOperand& out, cudaStream_t s) {
  OzSliceBatch P;
  P.add(x, ld, rows, cols, mode, out);
  oz_slice(P, s);
}

void oz_slice_cols(const double* x, long long ld, int rows, int cols, int mode, const OzOperand& out, cudaStream_t s) {
  if (rows <= 0 || cols <= 0) return;
  const int rt = ceil_div(rows, 64), kt = ceil_div(cols, 64);
  k_oz_exps_t<<<rt * 2, 256, 0, s>>>(x, ld, rows, cols, mode, out.exps);
  FETIRP_LAUNCH_CHECK();
  k_oz_slice_t<<<dim3(kt, rt), 256, 0, s>>>(x, ld, rows, cols, mode, out.tiles, out.exps);
  FETIRP_LAUNCH_CHECK();
}

void oz_gemm(const OzGemm& G, cudaStream_t s) {
  oz_init();
  OzGemmKernel P;
  OzFix F;
  P.G = G;
  int total = 0, n = 0;
  long long words = 0;
  for (int p = 0; p < G.n; ++p) {
    if (G.M[p] <= 0 || G.N[p] <= 0) continue;
    P.G.A[n] = G.A[p]; P.G.B[n] = G.B[p];
    P.G.M[n] = G.M[p]; P.G.N[n] = G.N[p]; P.G.K[n] = G.K[p];
    P.G.mode[n] = G.mode[p]; P.G.Z[n] = G.Z[p]; P.G.ldz[n] = G.ldz[p];
    P.G.a[n] = G.a[p]; P.G.ai[n] = G.ai[p]; P.G.aj[n] = G.aj[p];
    P.G.b[n] = G.b[p]; P.G.ldb[n] = G.ldb[p]; P.G.flags[n] = G.flags[p];
    F.word_off[n] = words;
    words += oz_flag_words(G.M[p], G.N[p]);
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
  F.G = P.G;
  F.word_off[n] = words;
  k_oz_fix<<<(unsigned)std::min<long long>((words + 7) / 8, 152 * 5), FIX_THREADS, 0, s>>>(F);
  FETIRP_LAUNCH_CHECK();
}

}  // namespace fetirp
