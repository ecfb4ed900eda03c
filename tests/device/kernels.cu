// Single kernels of the library behind a C interface, for the tests that need their inputs and outputs (device pointers;
// linked against libfetirp.so).
#include "ops.cuh"

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

}  // extern "C"
