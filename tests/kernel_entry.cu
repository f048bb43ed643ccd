// C entries of internal kernels for the tests (device pointers, default
// stream, synchronised): reductions and updates of csrc/kernels_blas.cu and
// the weight gradient of csrc/kernels_learned.cu.
#include "kernels.h"

#include <algorithm>
#include <vector>

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

void k_alloc_failures(int n, int64_t bytes) { set_alloc_failures(n, (size_t)bytes); }

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

// the same for FP64 vectors V held as a Krylov basis: h = V^H w where nothing is
// to be added (sign 0), else w += sign V h
int k_basis(const void *V, int k, void *w, int64_t n, int nrhs, double2 *h, double sign, double2 *nrm) {
  return run([&] {
    Scratch t(std::max((size_t)reduce_blocks(n) * nrhs * k, (size_t)norm_scratch(n) * nrhs));
    DigitBasis b;
    double *inv;
    double2 *v;
    std::vector<double> one(nrhs, 1.0);
    MG_CUDA(cudaMalloc(&b.v, (size_t)k * nrhs * n * sizeof(int4)));
    MG_CUDA(cudaMalloc(&b.e, (size_t)k * nrhs * digit_tiles(n) * sizeof(short)));
    MG_CUDA(cudaMalloc(&v, (size_t)nrhs * n * sizeof(double2)));
    MG_CUDA(cudaMalloc(&inv, nrhs * sizeof(double)));
    MG_CUDA(cudaMemcpy(inv, one.data(), nrhs * sizeof(double), cudaMemcpyHostToDevice));
    for (int j = 0; j < k; ++j) normalise_digits(in<double>(V) + (int64_t)j * nrhs * n, v, b, j, inv, n, nrhs, 0);
    if (sign == 0.0) multi_dot_digits(b, k, in<double>(w), n, nrhs, h, k, t.s, 0);
    else multi_axpy_digits(b, k, static_cast<double2 *>(w), n, nrhs, h, k, sign, 0, nrm, t.s);
    MG_CUDA(cudaDeviceSynchronize());
    for (void *p : {(void *)b.v, (void *)b.e, (void *)v, (void *)inv}) cudaFree(p);
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

// FP32 coarse operator of 32 dofs per site whose only block is `diag` times the
// identity at every site, and its dots with the input
int k_site_dots(const void *x, void *y, float diag, int V, int nrhs, double2 *qx, double2 *qq) {
  return run([&] {
    Geom g{{V, 1, 1, 1}, V, 32};
    if (!stencil_rows_supported(g, nrhs)) throw Error(1, "not supported");
    std::vector<double2> A((size_t)V * 9 * 1024, make_double2(0.0, 0.0));
    for (int X = 0; X < V; ++X)
      for (int i = 0; i < 32; ++i) A[((size_t)X * 9 * 32 + i) * 32 + i].x = diag;
    double2 *Ad;
    float4 *AR;
    MG_CUDA(cudaMalloc(&Ad, A.size() * sizeof(double2)));
    MG_CUDA(cudaMalloc(&AR, A.size() * sizeof(float2)));
    MG_CUDA(cudaMemcpy(Ad, A.data(), A.size() * sizeof(double2), cudaMemcpyHostToDevice));
    stencil_to_rows(Ad, AR, (int64_t)A.size(), 0);
    Scratch t(stencil_dots_scratch(g, nrhs));
    stencil_apply_rows_dots(in<float>(x), static_cast<float2 *>(y), AR, g, nrhs, t.s, qx, qq, 0);
    MG_CUDA(cudaDeviceSynchronize());
    cudaFree(Ad);
    cudaFree(AR);
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
