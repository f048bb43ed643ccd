// Gauge-covariant convolution layers of the learned smoother: forward,
// adjoint (input gradient), weight gradient, and the Adam update.
//
//   phi[o](x) = sum_c sum_h W[h][o][c] (T_h psi[c])(x)
//
// h = 0 identity, 1 + 2 mu: U_mu(x) psi(x + mu), 2 + 2 mu: U_mu(x - mu)^H
// psi(x - mu), with the fermion sign on hops across the time boundary;
// W[h][o][c] is a complex 4x4 matrix on the spin index.  Activations are
// [b][c] fine-level vectors (FP32 in the structure-of-arrays order with
// structure-of-arrays links, FP64 canonical [site][12]); weights
// [h][o][c][4][4].  The adjoint uses that
// the adjoint of hop h is the reversed hop and the adjoint of W is W^H.
#include "fixed.cuh"
#include "kernels.h"

#include <type_traits>

namespace mg {

namespace {

inline int grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (int)(b < 152 * 16 ? (b < 1 ? 1 : b) : 152 * 16);
}

template <typename T> constexpr bool kSoa = sizeof(T) == 4;

// One hop: the site it reads, the site of its link, the sign of the time
// boundary; links are read as U[3 a + b] of that site.
template <typename T> struct HopAt {
  int sn, ls;
  T sign;
  bool fwd;
  __device__ __forceinline__ HopAt(const Geom &g, int s, const int (&c)[4], int h) {
    sn = ls = s;
    sign = (T)1;
    fwd = h & 1;
    if (h == 0) return;
    const int mu = (h - 1) >> 1;
    int cn[4] = {c[0], c[1], c[2], c[3]};
    if (fwd) {
      cn[mu] = (c[mu] + 1 == g.L[mu]) ? 0 : c[mu] + 1;
      if (mu == 3 && cn[3] == 0) sign = (T)-1;
    } else {
      cn[mu] = (c[mu] == 0) ? g.L[mu] - 1 : c[mu] - 1;
      if (mu == 3 && c[3] == 0) sign = (T)-1;
    }
    sn = g.index(cn);
    ls = fwd ? s : sn;
  }
};

// t = sign U v (fwd) or sign U^H v with the link of hop h > 0
template <typename T>
__device__ __forceinline__ void transport(const C<T> *__restrict__ U, int64_t V, const HopAt<T> &at, int h,
                                          const C<T> (&v)[12], C<T> (&t)[12]) {
  const int mu = (h - 1) >> 1;
  C<T> uu[9];
#pragma unroll
  for (int i = 0; i < 9; ++i)
    uu[i] = kSoa<T> ? __ldg(U + (int64_t)(mu * 9 + i) * V + at.ls) : __ldg(U + ((int64_t)at.ls * 4 + mu) * 9 + i);
#pragma unroll
  for (int sp = 0; sp < 4; ++sp) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      C<T> z = mk<T>((T)0, (T)0);
#pragma unroll
      for (int b = 0; b < 3; ++b)
        z = at.fwd ? cfma(uu[3 * a + b], v[sp * 3 + b], z) : cfmac(uu[3 * b + a], v[sp * 3 + b], z);
      t[sp * 3 + a] = cscale(z, at.sign);
    }
  }
}

// transported spinor t = T_h psi at site s (12 complex), sign folded in
template <typename T>
__device__ __forceinline__ void transported(const C<T> *__restrict__ psi, const C<T> *__restrict__ U,
                                            const Geom &g, int s, const int (&c)[4], int h,
                                            C<T> (&t)[12]) {
  const HopAt<T> at(g, s, c, h);
  if (h == 0) {
    load_fine_site<T>(psi, s, g.V, t);
    return;
  }
  C<T> v[12];
  load_fine_site<T>(psi, at.sn, g.V, v);
  transport<T>(U, g.V, at, h, v, t);
}

// acc += w t for the three colours of one spin entry.  FP32: the weight staged
// as (re, re, im, im), both halves of a complex number in one packed
// multiply-add (the same roundings as two plain ones, half the issue slots).
template <typename T> struct Spin3;
template <> struct Spin3<double> {
  using Weight = double2;
  const double2 *t;
  __device__ __forceinline__ Spin3(const double2 *v) : t(v) {}
  static __device__ __forceinline__ Weight weight(double2 w) { return w; }
  __device__ __forceinline__ void mac(const Weight &w, double2 *acc) const {
#pragma unroll
    for (int a = 0; a < 3; ++a) acc[a] = cfma(w, t[a], acc[a]);
  }
};
template <> struct Spin3<float> {
  using Weight = float4;
  P2 p[3], q[3];  // (re, im) and (-im, re)
  __device__ __forceinline__ Spin3(const float2 *v) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      p[a] = p2(v[a].x, v[a].y);
      q[a] = p2(-v[a].y, v[a].x);
    }
  }
  static __device__ __forceinline__ Weight weight(float2 w) { return make_float4(w.x, w.x, w.y, w.y); }
  __device__ __forceinline__ void mac(const Weight &w, float2 *acc) const {
    P2 d[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) d[a] = p2fma(p2(w.x, w.y), p[a], p2(acc[a].x, acc[a].y));
#pragma unroll
    for (int a = 0; a < 3; ++a) acc[a] = p2split(p2fma(p2(w.z, w.w), q[a], d[a]));
  }
};

// out_k += W_k t for a group of OG outputs; w[sq][k][sp]
template <typename T, int OG>
__device__ __forceinline__ void spin_mac(const typename Spin3<T>::Weight *__restrict__ w, const C<T> (&t)[12],
                                         C<T> (&acc)[OG][12]) {
#pragma unroll
  for (int sq = 0; sq < 4; ++sq) {
    const Spin3<T> v(t + 3 * sq);
#pragma unroll
    for (int k = 0; k < OG; ++k)
#pragma unroll
      for (int sp = 0; sp < 4; ++sp) v.mac(w[(sq * OG + k) * 4 + sp], acc[k] + 3 * sp);
  }
}

// weights of hop h, inputs c0 .. c0 + nc, outputs o0 .. o0 + OG (absent ones
// zero) as [c][sq][k][sp].  ADJ: the adjoint layer, out[c] = sum_o sum_h
// W[h][o][c]^H T_rev(h) gin[o]: the same sums with the weights
// W'[rev(h)][c][o] = W[h][o][c]^H.
template <typename T, int OG, bool ADJ>
__device__ __forceinline__ void stage_weights(const C<T> *__restrict__ W, int h, int c0, int nc, int o0, int Cin,
                                              int Cout, typename Spin3<T>::Weight *__restrict__ Ws) {
  for (int e = threadIdx.x; e < nc * OG * 16; e += blockDim.x) {
    const int c = c0 + e / (OG * 16), sq = e / (OG * 4) & 3, o = o0 + (e >> 2) % OG, sp = e & 3;
    C<T> w = mk<T>((T)0, (T)0);
    if (o < Cout && !ADJ) w = W[(((int64_t)h * Cout + o) * Cin + c) * 16 + sp * 4 + sq];
    if (o < Cout && ADJ) {
      const int hr = h == 0 ? 0 : ((h & 1) ? h + 1 : h - 1);
      w = cconj(W[(((int64_t)hr * Cin + c) * Cout + o) * 16 + sq * 4 + sp]);
    }
    Ws[e] = Spin3<T>::weight(w);
  }
}

// Layers of few inputs (Cin <= OG): one thread per site computing OG
// output channels at once, each transported input T_h psi[c] formed once for
// the group; blockIdx.x = (site range, sample) with the sample fastest, so the
// blocks of one site range run together and read its links from L2 after the
// first; blockIdx.y = output group (Cin, Cout: channels read and written).
template <typename T, int OG, bool ADJ>
__global__ void __launch_bounds__(128) glayer_early_kernel(const C<T> *__restrict__ in, C<T> *__restrict__ out,
                                                           const C<T> *__restrict__ W, const C<T> *__restrict__ U,
                                                           Geom g, int Cin, int Cout, int nb) {
  __shared__ typename Spin3<T>::Weight Ws[9 * OG * OG * 16];  // [h][c]
  const int o0 = blockIdx.y * OG, b = (int)(blockIdx.x % (unsigned)nb);
  for (int h = 0; h < 9; ++h) stage_weights<T, OG, ADJ>(W, h, 0, Cin, o0, Cin, Cout, Ws + h * Cin * OG * 16);
  __syncthreads();
  const int s = (int)(blockIdx.x / (unsigned)nb) * blockDim.x + threadIdx.x;
  if (s >= g.V) return;
  const int64_t n = g.n();
  int cc[4];
  g.coords(s, cc);
  C<T> acc[OG][12];
#pragma unroll
  for (int k = 0; k < OG; ++k)
#pragma unroll
    for (int i = 0; i < 12; ++i) acc[k][i] = mk<T>((T)0, (T)0);
  for (int c = 0; c < Cin; ++c)
    for (int h = 0; h < 9; ++h) {
      C<T> t[12];
      transported<T>(in + ((int64_t)b * Cin + c) * n, U, g, s, cc, h, t);
      spin_mac<T, OG>(Ws + (h * Cin + c) * OG * 16, t, acc);
    }
#pragma unroll
  for (int k = 0; k < OG; ++k)
    if (o0 + k < Cout) store_fine_site<T>(out + ((int64_t)b * Cout + o0 + k) * n, s, g.V, acc[k]);
}

// Layers of more inputs: the weights act before the transport, which commutes
// with them, so a hop costs one transport per output instead of one per input
// and group.  The sum over the hops waits in shared memory, a column per
// thread, while a hop's inputs are summed in registers.  Bound: FMA pipe, 62%
// of its cycles at 16 inputs and outputs with two blocks of 250 registers on an
// SM.  16^4, two samples, FP32: 2.54 ms for the layer 16 -> 16 and 3.15 ms for
// 1 -> 16 -> 16 -> 1, where transporting every input for every group of outputs
// took 4.31 ms; without the load ahead 3.35 ms, three blocks 3.55 ms (spills).
constexpr int kLateIn = 16;  // inputs whose weights are staged at a time
template <typename T, int OG> constexpr int kLateBlocks = sizeof(T) == 8 ? (OG == 1 ? 3 : 2) : OG == 4 ? 2 : OG == 2 ? 3 : 4;
template <typename T, int OG, bool ADJ>
__global__ void __launch_bounds__(128, kLateBlocks<T, OG>)
    glayer_late_kernel(const C<T> *__restrict__ in, C<T> *__restrict__ out, const C<T> *__restrict__ W,
                       const C<T> *__restrict__ U, Geom g, int Cin, int Cout, int nb) {
  using Wt = typename Spin3<T>::Weight;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Wt *Ws = reinterpret_cast<Wt *>(smem_raw);
  C<T> *sum = reinterpret_cast<C<T> *>(Ws + kLateIn * OG * 16) + threadIdx.x;
  const int o0 = blockIdx.y * OG, b = (int)(blockIdx.x % (unsigned)nb);
  const int s0 = (int)(blockIdx.x / (unsigned)nb) * 128 + threadIdx.x, s = min(s0, g.V - 1);
  const int64_t n = g.n();
  int cc[4];
  g.coords(s, cc);
#pragma unroll 1
  for (int h = 0; h < 9; ++h) {
    const HopAt<T> at(g, s, cc, h);
    C<T> acc[OG][12];
#pragma unroll
    for (int k = 0; k < OG; ++k)
#pragma unroll
      for (int i = 0; i < 12; ++i) acc[k][i] = mk<T>((T)0, (T)0);
#pragma unroll 1
    for (int c0 = 0; c0 < Cin; c0 += kLateIn) {
      const int nc = min(kLateIn, Cin - c0);
      __syncthreads();
      stage_weights<T, OG, ADJ>(W, h, c0, nc, o0, Cin, Cout, Ws);
      __syncthreads();
      const C<T> *psi = in + ((int64_t)b * Cin + c0) * n;
      // the next input is on its way while this one is multiplied
      C<T> v[12], nx[12];
      load_fine_site<T>(psi, at.sn, g.V, v);
#pragma unroll 2
      for (int c = 0; c < nc; ++c) {
        load_fine_site<T>(psi + min(c + 1, nc - 1) * n, at.sn, g.V, nx);
        spin_mac<T, OG>(Ws + c * OG * 16, v, acc);
#pragma unroll
        for (int i = 0; i < 12; ++i) v[i] = nx[i];
      }
    }
#pragma unroll
    for (int k = 0; k < OG; ++k) {
      C<T> t[12];
      if (h == 0) {
#pragma unroll
        for (int i = 0; i < 12; ++i) t[i] = acc[k][i];
      } else {
        transport<T>(U, g.V, at, h, acc[k], t);
#pragma unroll
        for (int i = 0; i < 12; ++i) t[i] = cadd(sum[(k * 12 + i) * 128], t[i]);
      }
      if (h < 8) {
#pragma unroll
        for (int i = 0; i < 12; ++i) sum[(k * 12 + i) * 128] = t[i];
      } else if (s0 < g.V && o0 + k < Cout) {
        store_fine_site<T>(out + ((int64_t)b * Cout + o0 + k) * n, s, g.V, t);
      }
    }
  }
}

// weight-gradient partials: block (chunk, c * 9 + h, output pair) sums over its
// sites and all samples g[o](x) (T_h psi[c])(x)^H (16 spin entries, colour
// summed) for OG outputs, the transported input formed once for them.  Bound:
// FP64 pipe (FP64) / FMAs; the chunks are short so that a small lattice fills
// the GPU (4096 sites in one block took 2.2 ms whatever the layer), and the
// sums over a warp are integer ones (fixed.cuh).
constexpr int kWgradThreads = 128;
// sites per block; longer on large lattices, whose partials would outgrow use (loss
// and gradient, 2 channels: 8^4 1.60 ms, with 4096 throughout 3.37; 2^18 sites
// 27.5 and 28.0; 32^4 106.7 and 106.9)
inline int wgrad_chunk(const Geom &g) { return g.V <= (1 << 18) ? 512 : 4096; }

template <typename T, int OG>
__global__ void __launch_bounds__(kWgradThreads) glayer_wgrad_kernel(const C<T> *__restrict__ gin,
                                                           const C<T> *__restrict__ in,
                                                           const C<T> *__restrict__ U, Geom g,
                                                           int Cin, int Cout, int B, int chunk,
                                                           double2 *__restrict__ partial) {
  constexpr int NW = kWgradThreads / 32;
  __shared__ double sh[OG][32][NW];
  const int ch = blockIdx.y / 9, h = blockIdx.y % 9, o0 = blockIdx.z * OG;
  const int64_t n = g.n();
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  // FP32: a thread's sums run over 16 sites of every sample, then go on in FP64
  // (16 x 128 of the 4096 sites that a block takes above 2^18)
  constexpr int kSub = 16 * kWgradThreads;
  const int beg = blockIdx.x * chunk, end = min(g.V, beg + chunk);
  double mine[OG];
#pragma unroll
  for (int q = 0; q < OG; ++q) mine[q] = 0.0;
#pragma unroll 1
  for (int sub = beg, last; sub < end; sub = last) {
    last = sizeof(T) == 4 ? min(sub + kSub, end) : end;
    C<T> acc[OG][16];
#pragma unroll
    for (int q = 0; q < OG; ++q)
#pragma unroll
      for (int k = 0; k < 16; ++k) acc[q][k] = mk<T>((T)0, (T)0);
    for (int s = sub + threadIdx.x; s < last; s += blockDim.x) {
      int cc[4];
      g.coords(s, cc);
      for (int b = 0; b < B; ++b) {
        C<T> t[12];
        transported<T>(in + ((int64_t)b * Cin + ch) * n, U, g, s, cc, h, t);
#pragma unroll
        for (int q = 0; q < OG; ++q) {
          if (o0 + q >= Cout) break;
          const C<T> *gp = gin + ((int64_t)b * Cout + o0 + q) * n;
          C<T> gv[12];
          load_fine_site<T>(gp, s, g.V, gv);
#pragma unroll
          for (int sp = 0; sp < 4; ++sp)
#pragma unroll
            for (int sq = 0; sq < 4; ++sq)
#pragma unroll
              for (int a = 0; a < 3; ++a)
                acc[q][sp * 4 + sq] = cfmac(t[sq * 3 + a], gv[sp * 3 + a], acc[q][sp * 4 + sq]);  // g conj(t)
        }
      }
    }
#pragma unroll
    for (int q = 0; q < OG; ++q) {
      std::conditional_t<sizeof(T) == 4, fx::WarpSumF, fx::WarpSumD> ws;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        ws.add(2 * k, acc[q][k].x);
        ws.add(2 * k + 1, acc[q][k].y);
      }
      if constexpr (sizeof(T) == 4) {
        if (ws.bad()) {
#pragma unroll
          for (int k = 0; k < 16; ++k) {
            ws.fix(2 * k, acc[q][k].x);
            ws.fix(2 * k + 1, acc[q][k].y);
          }
        }
      }
      mine[q] += ws.get();
    }
  }
#pragma unroll
  for (int q = 0; q < OG; ++q) sh[q][l][w] = mine[q];
  __syncthreads();
  for (int e = threadIdx.x; e < OG * 32; e += blockDim.x) {
    const int q = e >> 5, v = e & 31;
    if (o0 + q >= Cout) continue;
    double t = 0.0;
    for (int i = 0; i < NW; ++i) t += sh[q][v][i];
    // layout [chunk][h][o][c][16]
    reinterpret_cast<double *>(partial)[((((int64_t)blockIdx.x * 9 + h) * Cout + o0 + q) * Cin + ch) * 32 + v] = t;
  }
}

__global__ void wgrad_sum_kernel(const double2 *__restrict__ partial, int nchunks, int64_t count,
                                 double2 *__restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x) {
    double2 t = make_double2(0.0, 0.0);
    for (int k = 0; k < nchunks; ++k) {
      const double2 p = partial[(int64_t)k * count + e];
      t.x += p.x;
      t.y += p.y;
    }
    out[e] = t;
  }
}

// Adam on the real and imaginary parts of every complex weight; grad holds
// dL/dW* (so the real-parameter gradient is 2 grad); scale divides the
// accumulated gradient (batch mean).
__global__ void adam_kernel(double2 *__restrict__ W, const double2 *__restrict__ grad,
                            double2 *__restrict__ m, double2 *__restrict__ v, int64_t count,
                            double lr, double b1, double b2, double epsv, double bc1, double bc2,
                            double scale) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x) {
    const double gx = 2.0 * grad[e].x * scale, gy = 2.0 * grad[e].y * scale;
    double2 mm = m[e], vv = v[e];
    mm.x = b1 * mm.x + (1 - b1) * gx;
    mm.y = b1 * mm.y + (1 - b1) * gy;
    vv.x = b2 * vv.x + (1 - b2) * gx * gx;
    vv.y = b2 * vv.y + (1 - b2) * gy * gy;
    m[e] = mm;
    v[e] = vv;
    double2 w = W[e];
    w.x -= lr * (mm.x / bc1) / (sqrt(vv.x / bc2) + epsv);
    w.y -= lr * (mm.y / bc1) / (sqrt(vv.y / bc2) + epsv);
    W[e] = w;
  }
}

}  // namespace

template <typename T, int OG, bool ADJ>
static void glayer_og(const C<T> *in, C<T> *out, const C<T> *W, const C<T> *U, Geom g, int Cin, int Cout, int B,
                      cudaStream_t s) {
  const dim3 grid((unsigned)div_up(g.V, 128) * (unsigned)B, div_up(Cout, OG), 1);
  // a hop transports OG sums there, Cin inputs here
  if (Cin <= OG) {
    glayer_early_kernel<T, OG, ADJ><<<grid, 128, 0, s>>>(in, out, W, U, g, Cin, Cout, B);
  } else {
    const size_t sm = kLateIn * OG * 16 * sizeof(typename Spin3<T>::Weight) + OG * 12 * 128 * sizeof(C<T>);
    smem_optin((const void *)glayer_late_kernel<T, OG, ADJ>, (int)sm);
    glayer_late_kernel<T, OG, ADJ><<<grid, 128, sm, s>>>(in, out, W, U, g, Cin, Cout, B);
  }
  MG_LAUNCH_CHECK();
}

template <typename T, bool ADJ>
static void glayer(const C<T> *in, C<T> *out, const C<T> *W, const C<T> *U, Geom g, int Cin, int Cout, int B,
                   cudaStream_t s) {
  // four output channels share an input; two where FP64 sums and inputs of
  // four would not leave registers for two blocks
  if (Cout == 1) glayer_og<T, 1, ADJ>(in, out, W, U, g, Cin, Cout, B, s);
  else if (Cout == 2 || (sizeof(T) == 8)) glayer_og<T, 2, ADJ>(in, out, W, U, g, Cin, Cout, B, s);
  else glayer_og<T, 4, ADJ>(in, out, W, U, g, Cin, Cout, B, s);
}

template <typename T>
void glayer_forward(const C<T> *in, C<T> *out, const C<T> *W, const C<T> *U, Geom g, int Cin,
                    int Cout, int B, cudaStream_t s) {
  glayer<T, false>(in, out, W, U, g, Cin, Cout, B, s);
}

template <typename T>
void glayer_adjoint(const C<T> *gin, C<T> *out, const C<T> *W, const C<T> *U, Geom g, int Cin,
                    int Cout, int B, cudaStream_t s) {
  glayer<T, true>(gin, out, W, U, g, Cout, Cin, B, s);
}

int glayer_wgrad_chunks(const Geom &g) { return div_up(g.V, wgrad_chunk(g)); }

template <typename T>
void glayer_wgrad(const C<T> *gin, const C<T> *in, const C<T> *U, Geom g, int Cin, int Cout, int B,
                  double2 *partial, double2 *out, cudaStream_t s) {
  const int nchunks = glayer_wgrad_chunks(g);
  if (Cout == 1)
    glayer_wgrad_kernel<T, 1><<<dim3(nchunks, Cin * 9, 1), kWgradThreads, 0, s>>>(gin, in, U, g, Cin, Cout, B,
                                                                                 wgrad_chunk(g), partial);
  else
    glayer_wgrad_kernel<T, 2><<<dim3(nchunks, Cin * 9, div_up(Cout, 2)), kWgradThreads, 0, s>>>(gin, in, U, g, Cin,
                                                                                               Cout, B, wgrad_chunk(g),
                                                                                               partial);
  MG_LAUNCH_CHECK();
  const int64_t count = (int64_t)9 * Cout * Cin * 16;
  wgrad_sum_kernel<<<grid_for(count), 256, 0, s>>>(partial, nchunks, count, out);
  MG_LAUNCH_CHECK();
}

void adam_step(double2 *W, const double2 *grad, double2 *m, double2 *v, int64_t count, double lr,
               double b1, double b2, double eps, int t, double scale, cudaStream_t s) {
  const double bc1 = 1.0 - pow(b1, t), bc2 = 1.0 - pow(b2, t);
  adam_kernel<<<grid_for(count), 256, 0, s>>>(W, grad, m, v, count, lr, b1, b2, eps, bc1, bc2, scale);
  MG_LAUNCH_CHECK();
}

#define INST(T)                                                                                 \
  template void glayer_forward<T>(const C<T> *, C<T> *, const C<T> *, const C<T> *, Geom, int,  \
                                  int, int, cudaStream_t);                                      \
  template void glayer_adjoint<T>(const C<T> *, C<T> *, const C<T> *, const C<T> *, Geom, int,  \
                                  int, int, cudaStream_t);                                      \
  template void glayer_wgrad<T>(const C<T> *, const C<T> *, const C<T> *, Geom, int, int, int,  \
                                double2 *, double2 *, cudaStream_t);
INST(double)
INST(float)

}  // namespace mg
