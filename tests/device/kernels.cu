// Single kernels of the library behind a C interface, for the tests that need their inputs and outputs (device pointers;
// linked against libfetirp.so).
#include "ops.cuh"
#include "oz.cuh"

using namespace fetirp;

template <typename F>
static int guarded(F f) {
  try {
    f();
    return cudaDeviceSynchronize() == cudaSuccess ? 0 : 1;
  } catch (const std::exception& e) {
    std::fprintf(stderr, "%s\n", e.what());
    return 2;
  }
}

extern "C" {

// out (host, k x (k + 1)) = W^T [Q | r] from the row-chunk partials, added in order
int t_eta(int n, int k, const double* W, const double* Q, const double* r, int ds, double* out) {
  return guarded([&] {
    DBuf<double> part;
    int n_read = 0;
    const int off = eta_partials(n, k, W, Q, r, part, nullptr, ds != 0, &n_read);
    const size_t nout = (size_t)k * (k + 1);
    std::vector<double> h(nout * n_read);
    FETIRP_CUDA(cudaMemcpy(h.data(), part.p + nout * off, sizeof(double) * h.size(), cudaMemcpyDeviceToHost));
    for (size_t o = 0; o < nout; ++o) {
      out[o] = 0.0;
      for (int c = 0; c < n_read; ++c) out[o] += h[nout * c + o];
    }
  });
}

// z[c * ldz + i] = sum_j A(i, j) b[c * ldb + j] as a sliced product; A(i, j) at a[i * lda + j], or (by_cols) at
// a[j * lda + i]; mode as in OzGemm.  n_fma (host): outputs that FMAs computed
int t_oz(int M, int N, int K, int mode, int by_cols, const double* a, long long lda, const double* b, long long ldb,
         double* z, long long ldz, long long* n_fma) {
  return guarded([&] {
    DBuf<uint8_t> sa(oz_tiles(M, K, mode) * OZ_TILE), sb(oz_tiles(N, K) * OZ_TILE);
    DBuf<int> ea(round_up(M, 64)), eb(round_up(N, 64)), error(1);
    DBuf<uint32_t> flags(oz_flag_words(M, N));
    error.zero(nullptr);
    OzGemm G;
    G.n = 1;
    G.A[0] = {sa.p, ea.p}; G.B[0] = {sb.p, eb.p};
    G.M[0] = M; G.N[0] = N; G.K[0] = K; G.mode[0] = mode; G.Z[0] = z; G.ldz[0] = ldz;
    G.a[0] = a; G.ai[0] = by_cols ? 1 : lda; G.aj[0] = by_cols ? lda : 1; G.b[0] = b; G.ldb[0] = ldb;
    G.flags[0] = flags.p; G.error = error.p;
    if (by_cols) oz_slice_cols(a, lda, M, K, mode, G.A[0], nullptr);
    else oz_slice_rows(a, lda, M, K, mode, G.A[0], nullptr);
    oz_slice_rows(b, ldb, N, K, 0, G.B[0], nullptr);
    oz_gemm(G, nullptr);
    int code = 0;
    std::vector<uint32_t> h(flags.n);
    FETIRP_CUDA(cudaMemcpy(&code, error.p, sizeof(int), cudaMemcpyDeviceToHost));
    FETIRP_CUDA(cudaMemcpy(h.data(), flags.p, sizeof(uint32_t) * h.size(), cudaMemcpyDeviceToHost));
    if (code) throw Error(6, "a wait expired");
    *n_fma = 0;
    for (uint32_t w : h) *n_fma += __builtin_popcount(w);
  });
}

}  // extern "C"
