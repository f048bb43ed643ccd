// C entries of internal kernels for the tests (device pointers, default
// stream, synchronised): reductions and updates of csrc/kernels_blas.cu and
// the weight gradient of csrc/kernels_learned.cu.
#include "kernels.h"

using namespace mg;

namespace {
struct Scratch {
  RedScratch s{};
  explicit Scratch(size_t partials) {
    MG_CUDA(cudaMalloc(&s.partial, partials * sizeof(double2)));
    MG_CUDA(cudaMalloc(&s.ticket, kTickets * sizeof(unsigned)));
    MG_CUDA(cudaMemset(s.ticket, 0, kTickets * sizeof(unsigned)));
  }
  ~Scratch() {
    cudaFree(s.partial);
    cudaFree(s.ticket);
  }
};
template <typename F> int run(F &&f) {
  try {
    f();
    MG_CUDA(cudaDeviceSynchronize());
    return 0;
  } catch (const std::exception &) {
    return 1;
  }
}
template <typename T> const C<T> *in(const void *p) { return static_cast<const C<T> *>(p); }
}  // namespace

extern "C" {

int k_dot(int fp32, const void *x, const void *y, int64_t n, int nrhs, double2 *out) {
  return run([&] {
    Scratch t((size_t)reduce_blocks(n) * nrhs);
    if (fp32) dot<float>(in<float>(x), in<float>(y), n, nrhs, out, t.s, 0);
    else dot<double>(in<double>(x), in<double>(y), n, nrhs, out, t.s, 0);
    MG_CUDA(cudaDeviceSynchronize());
  });
}

int k_multi_dot(int fp32, const void *V, int64_t vstride, int k, const void *w, int64_t n, int nrhs, double2 *h) {
  return run([&] {
    Scratch t((size_t)reduce_blocks(n) * nrhs * k);
    if (fp32) multi_dot<float>(in<float>(V), vstride, k, in<float>(w), n, nrhs, h, k, t.s, 0);
    else multi_dot<double>(in<double>(V), vstride, k, in<double>(w), n, nrhs, h, k, t.s, 0);
    MG_CUDA(cudaDeviceSynchronize());
  });
}

int k_dot_qr(int fp32, const void *q, const void *r, int64_t n, int nrhs, double2 *qr, double2 *qq) {
  return run([&] {
    Scratch t((size_t)reduce_blocks(n) * nrhs * 2);
    if (fp32) dot_qr<float>(in<float>(q), in<float>(r), n, nrhs, qr, qq, t.s, 0);
    else dot_qr<double>(in<double>(q), in<double>(r), n, nrhs, qr, qq, t.s, 0);
    MG_CUDA(cudaDeviceSynchronize());
  });
}

// w += sign sum_j h[j] V_j; nrm (may be null): the norms of the result
int k_multi_axpy(int fp32, const void *V, int64_t vstride, int k, void *w, int64_t n, int nrhs, const double2 *h,
                 double sign, double2 *nrm) {
  return run([&] {
    Scratch t((size_t)norm_scratch(n) * nrhs);
    if (fp32) multi_axpy<float>(in<float>(V), vstride, k, static_cast<float2 *>(w), n, nrhs, h, k, sign, 0, nrm, t.s);
    else multi_axpy<double>(in<double>(V), vstride, k, static_cast<double2 *>(w), n, nrhs, h, k, sign, 0, nrm, t.s);
    MG_CUDA(cudaDeviceSynchronize());
  });
}

// the FP32 weight gradient [h][o][c][16] of a layer, links structure-of-arrays
int k_wgrad_f32(const void *gin, const void *x, const void *U, const int *dims, int cin, int cout, int B,
                double2 *out) {
  return run([&] {
    Geom g{};
    g.V = 1;
    for (int i = 0; i < 4; ++i) g.V *= g.L[i] = dims[i];
    g.dof = 12;
    Scratch t((size_t)glayer_wgrad_chunks(g) * 9 * cin * cout * 16);
    glayer_wgrad<float>(in<float>(gin), in<float>(x), in<float>(U), g, cin, cout, B, t.s.partial, out, 0);
    MG_CUDA(cudaDeviceSynchronize());
  });
}
}
