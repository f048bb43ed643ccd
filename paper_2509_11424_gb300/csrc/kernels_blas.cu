// Level-1 vector kernels (batched over right-hand sides) and the per-rhs
// small-matrix kernels of batched FGMRES.
//
// Reductions are deterministic: a fixed number of blocks (a function of n
// only) writes partial sums that the last block to finish adds in block
// order, so a result never depends on scheduling.  FP32 products are summed
// in FP32 within a thread, FP64 ones as integers (fixed.cuh); the sums over
// the lanes of a warp are exact integer ones (51 bits of the largest lane for
// FP32), and across warps and blocks FP64.  FP64 additions are kept to those:
// a warp's shuffle reduction of one complex number in FP64 takes 640 cycles
// of the FP64 pipe, as long as 64 FP32 multiply-adds per lane.
#include "fixed.cuh"
#include "kernels.h"

#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

namespace mg {

namespace {
constexpr int RB = 256;  // reduction block size

// Single-pass reductions.  Block b of output g sums its chunk, writes the
// partial, and takes a ticket; the block that draws the last ticket adds the
// NB partials of g in block order (so the result never depends on
// scheduling) and puts the ticket back to zero.  Nothing waits on anything.
__device__ __forceinline__ bool last_block(unsigned *ticket) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    __threadfence();  // this block's partial is visible before its ticket
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  return last;
}

using fx::WarpSumF;
using fx::WarpSumI;
using fx::warp_exp;
using fx::digits;
__device__ __forceinline__ int exp2of(double2 v) { return max(fx::exp_field(v.x), fx::exp_field(v.y)); }
// conj(a) b for the digits a, b: high and middle sums
__device__ __forceinline__ void macc(int4 a, int4 b, long long &hr, long long &hi, long long &mr, long long &mi) {
  const int n1 = -a.z, n0 = -a.w;
  hr = fx::madw(a.z, b.z, fx::madw(a.x, b.x, hr));
  hi = fx::madw(n1, b.x, fx::madw(a.x, b.z, hi));
  mr = fx::madw(a.w, b.z, fx::madw(a.z, b.w, fx::madw(a.y, b.x, fx::madw(a.x, b.y, mr))));
  mi = fx::madw(n0, b.x, fx::madw(n1, b.y, fx::madw(a.y, b.z, fx::madw(a.x, b.w, mi))));
}
// a b
__device__ __forceinline__ void mac(int4 a, int4 b, long long &hr, long long &hi, long long &mr, long long &mi) {
  const int n1 = -a.z, n0 = -a.w;
  hr = fx::madw(n1, b.z, fx::madw(a.x, b.x, hr));
  hi = fx::madw(a.z, b.x, fx::madw(a.x, b.z, hi));
  mr = fx::madw(n0, b.z, fx::madw(n1, b.w, fx::madw(a.y, b.x, fx::madw(a.x, b.y, mr))));
  mi = fx::madw(a.w, b.x, fx::madw(a.z, b.y, fx::madw(a.y, b.z, fx::madw(a.x, b.w, mi))));
}

// The block's NV sums (lane v of every warp holds value v) to partial[v * NB +
// b] (doubles, pv apart); the block that finishes group g last adds the NB
// partials of every value in block order and returns true with value v in
// thread v < NV.
template <int NV>
__device__ __forceinline__ bool block_finish(double mine, double *__restrict__ partial, unsigned *__restrict__ ticket,
                                             int nv, double &out) {
  __shared__ double red[RB / 32][NV];
  __shared__ double tail[RB / NV][NV];
  static_assert((NV & (NV - 1)) == 0 && RB % NV == 0, "tree");
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, NB = gridDim.x;
  if (lane < NV) red[wp][lane] = mine;
  __syncthreads();
  if ((int)threadIdx.x < nv) {
    double t = red[0][threadIdx.x];
#pragma unroll
    for (int q = 1; q < RB / 32; ++q) t += red[q][threadIdx.x];
    if (NB == 1) out = t;
    else partial[(int64_t)threadIdx.x * NB + blockIdx.x] = t;
  }
  if (NB == 1) return true;
  __threadfence();
  __syncthreads();
  if (!last_block(ticket)) return false;
  __threadfence();
  // RB / NV threads per value, each over consecutive blocks, then a tree (one
  // thread adding all 128 took longer than the rest of a small dot: 8192
  // entries, 8 right-hand sides 9.6 us, now 5.5)
  const int v = threadIdx.x % NV, c = threadIdx.x / NV;
  double t = 0.0;
  if (v < nv) {
    const int per = (NB + RB / NV - 1) / (RB / NV), b0 = c * per, b1 = min(NB, b0 + per);
    for (int q = b0; q < b1; ++q) t += __ldcg(partial + (int64_t)v * NB + q);
  }
  tail[c][v] = t;
#pragma unroll
  for (int o = RB / NV / 2; o > 0; o >>= 1) {
    __syncthreads();
    if (c < o) tail[c][v] = t += tail[c + o][v];
  }
  if ((int)threadIdx.x < nv) out = t;
  if (threadIdx.x == 0) *ticket = 0u;
  return true;
}

// A thread's own entries of the vectors j, j + 1, ... of a basis pass through a
// ring of kRing slots of 16 TILE bytes in shared memory by asynchronous copies:
// kRing vectors' entries are in flight per thread (64 KB per block and three
// blocks per SM at TILE = 1024, 32 KB and six at 512) without a register for
// them, and without a barrier, since every thread reads only what it copied.
// FP64 digits, n = 786 k, 16 right-hand sides, 1 .. 20 vectors: updates 364 us on
// average, 6.9 TB/s, 20 dots 756 us; with the loads of one vector at a time in
// registers 707 and 1225 us, waiting for memory.  (The checks for graded entries
// have added 2.5% since.)
constexpr int kRing = 4;
template <int TILE> struct Ring {
  int4 *slot;  // [kRing][TILE]
  __device__ __forceinline__ void fetch(int s, const int4 *src, int64_t left) const {
#pragma unroll
    for (int u = 0; u < TILE / RB; ++u) {
      int4 *d = slot + s * TILE + u * RB + threadIdx.x;
      if (u * RB + (int)threadIdx.x < left)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(d)),
                     "l"(src + u * RB + threadIdx.x)
                     : "memory");
      else *d = make_int4(0, 0, 0, 0);
    }
  }
  __device__ __forceinline__ static void commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
  // the oldest of the last kRing groups has landed
  __device__ __forceinline__ static void wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(kRing - 1) : "memory"); }
  __device__ __forceinline__ int4 get(int s, int u) const { return slot[s * TILE + u * RB + threadIdx.x]; }
  __device__ __forceinline__ float4 getf(int s, int u) const {
    return *reinterpret_cast<const float4 *>(slot + s * TILE + u * RB + threadIdx.x);
  }
};

// element pairs of FP32 vectors as one 16-byte load where the operands allow
template <bool VEC>
__device__ __forceinline__ float4 ld2(const float2 *__restrict__ p, int64_t i, int64_t end) {
  if (VEC) return i < end ? __ldg(reinterpret_cast<const float4 *>(p + i)) : make_float4(0.f, 0.f, 0.f, 0.f);
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (i < end) { v.x = p[i].x; v.y = p[i].y; }
  if (i + 1 < end) { v.z = p[i + 1].x; v.w = p[i + 1].y; }
  return v;
}

// out[r * ldh + j] = sum conj(x_j,r) y_r, JG vectors x_j per block (grid z),
// y read once for them.  Block (b, r, z): elements [b chunk, (b + 1) chunk).
// Bound: memory (x once, y once per JG of them; 5.4 TB/s at n = 786 k, 8
// right-hand sides, 15 vectors), latency below n ~ 10^5: short chunks, so that
// a right-hand side of 8192 entries has 8 blocks.
template <int JG, bool VEC>
__global__ void __launch_bounds__(RB) dot_f32_kernel(const float2 *__restrict__ x, int64_t xstride, int k,
                                                     const float2 *__restrict__ y, int64_t n, int64_t chunk,
                                                     double2 *__restrict__ partial, unsigned *__restrict__ ticket,
                                                     double2 *__restrict__ out, int ldh) {
  constexpr int U = 2;  // element pairs per thread and step
  const int r = blockIdx.y, j0 = blockIdx.z * JG, kg = min(JG, k - j0);
  const float2 *xr = x + j0 * xstride + r * n, *yr = y + r * n;
  const int64_t beg = (int64_t)blockIdx.x * chunk, end = min(beg + chunk, n);
  float ar[JG], ai[JG];
#pragma unroll
  for (int j = 0; j < JG; ++j) ar[j] = ai[j] = 0.f;
  for (int64_t i0 = beg + 2 * threadIdx.x; i0 < end; i0 += 2 * RB * U) {
    float4 c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = ld2<VEC>(yr, i0 + 2 * RB * u, end);
#pragma unroll
    for (int j = 0; j < JG; ++j) {
      if (j < kg) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float4 a = ld2<VEC>(xr + j * xstride, i0 + 2 * RB * u, end);
          ar[j] = fmaf(a.x, c[u].x, fmaf(a.y, c[u].y, fmaf(a.z, c[u].z, fmaf(a.w, c[u].w, ar[j]))));
          ai[j] = fmaf(a.x, c[u].y, fmaf(-a.y, c[u].x, fmaf(a.z, c[u].w, fmaf(-a.w, c[u].z, ai[j]))));
        }
      }
    }
  }
  WarpSumF ws;
#pragma unroll
  for (int j = 0; j < JG; ++j) {
    if (j < kg) {
      ws.add(2 * j, ar[j]);
      ws.add(2 * j + 1, ai[j]);
    }
  }
  if (ws.bad()) {
#pragma unroll
    for (int j = 0; j < JG; ++j) {
      if (j < kg) {
        ws.fix(2 * j, ar[j]);
        ws.fix(2 * j + 1, ai[j]);
      }
    }
  }
  double s;
  const int64_t g = (int64_t)r * gridDim.z + blockIdx.z;
  double *part = reinterpret_cast<double *>(partial) + ((int64_t)r * k + j0) * 2 * gridDim.x;
  if (block_finish<2 * JG>(ws.get(), part, ticket + g, 2 * kg, s) && (int)threadIdx.x < 2 * kg)
    reinterpret_cast<double *>(out + r * ldh + j0)[threadIdx.x] = s;
}

// The same sums in the same order with the vectors through the ring, for 16-byte
// aligned FP32 vectors of even length.  n = 786 k, 8 right-hand sides, 9 .. 16
// vectors: 144 us on average (168 us from registers).
constexpr int kTileF = 512;  // 1024 elements
template <int JG>
__global__ void __launch_bounds__(RB) dot_f32_ring_kernel(const int4 *__restrict__ x, int64_t xstride, int k,
                                                          const float4 *__restrict__ y, int64_t n, int64_t chunk,
                                                          double2 *__restrict__ partial,
                                                          unsigned *__restrict__ ticket, double2 *__restrict__ out,
                                                          int ldh) {
  constexpr int U = kTileF / RB;
  using R = Ring<kTileF>;
  const int r = blockIdx.y, j0 = blockIdx.z * JG, kg = min(JG, k - j0);
  const int4 *xr = x + j0 * xstride + r * n;  // n, strides, chunk in pairs of elements
  const float4 *yr = y + r * n;
  const int64_t beg = (int64_t)blockIdx.x * chunk, end = min(beg + chunk, n);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const R ring{reinterpret_cast<int4 *>(smem_raw)};
  float ar[JG], ai[JG];
#pragma unroll
  for (int j = 0; j < JG; ++j) ar[j] = ai[j] = 0.f;
  for (int64_t t0 = beg; t0 < end; t0 += kTileF) {
#pragma unroll
    for (int j = 0; j < kRing; ++j) {
      if (j < kg) ring.fetch(j, xr + j * xstride + t0, end - t0);
      R::commit();
    }
    float4 c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = t0 + threadIdx.x + RB * u;
      c[u] = i < end ? __ldg(yr + i) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int j = 0; j < JG; ++j) {
      if (j < kg) {
        R::wait();
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const float4 a = ring.getf(j % kRing, u);
          ar[j] = fmaf(a.x, c[u].x, fmaf(a.y, c[u].y, fmaf(a.z, c[u].z, fmaf(a.w, c[u].w, ar[j]))));
          ai[j] = fmaf(a.x, c[u].y, fmaf(-a.y, c[u].x, fmaf(a.z, c[u].w, fmaf(-a.w, c[u].z, ai[j]))));
        }
        if (j + kRing < kg) ring.fetch(j % kRing, xr + (j + kRing) * xstride + t0, end - t0);
        R::commit();
      }
    }
  }
  WarpSumF ws;
#pragma unroll
  for (int j = 0; j < JG; ++j) {
    if (j < kg) {
      ws.add(2 * j, ar[j]);
      ws.add(2 * j + 1, ai[j]);
    }
  }
  if (ws.bad()) {
#pragma unroll
    for (int j = 0; j < JG; ++j) {
      if (j < kg) {
        ws.fix(2 * j, ar[j]);
        ws.fix(2 * j + 1, ai[j]);
      }
    }
  }
  double s;
  const int64_t g = (int64_t)r * gridDim.z + blockIdx.z;
  double *part = reinterpret_cast<double *>(partial) + ((int64_t)r * k + j0) * 2 * gridDim.x;
  if (block_finish<2 * JG>(ws.get(), part, ticket + g, 2 * kg, s) && (int)threadIdx.x < 2 * kg)
    reinterpret_cast<double *>(out + r * ldh + j0)[threadIdx.x] = s;
}

// What a group of 128 entries (one warp's of a step) adds to an FP64 dot product
// is kept in fixed point only where it is at least 2^-5 of the product S of the
// two scales, in its real or imaginary part.  Then the group's sum of |x y| is
// at least that, and what the digits lose, 256 products x (2 x 2^-58 + 2^-60) S
// at most, is within 2^-43.8 of it, near the bound of 256 FP64 additions, 2^-45.
// Any other group (large entries of one vector meet only small or no ones of
// the other; Inf or NaN) is added in FP64, out of line: 0.1% of the groups of a
// set-up's vectors (below 2^-4: 0.4%, and 3% of the dots' time, since a block
// waits for its last warp).  Groups where one vector is zero are not among them.
// t: the group's sums so far (lane v: value v); bits 2 j of redo: the vectors j.
__device__ __noinline__ double redo_groups(double t, unsigned redo, const double2 *__restrict__ x, int64_t xstride,
                                           const double2 *__restrict__ y, int64_t i0, int64_t end) {
  const int lane = threadIdx.x & 31;
  for (; redo; redo &= redo - 1) {
    const int j = (__ffs(redo) - 1) >> 1;
    double sr = 0.0, si = 0.0;
    for (int64_t i = i0; i < min(end, i0 + 4 * RB); i += RB) {
      const double2 a = x[j * xstride + i], c = y[i];
      sr = fma(a.x, c.x, fma(a.y, c.y, sr));
      si = fma(a.x, c.y, fma(-a.y, c.x, si));
    }
    fx::WarpSumD ws;
    ws.add(2 * j, sr);
    ws.add(2 * j + 1, si);
    if (lane >> 1 == j) t = ws.get();
  }
  return t;
}

// The same for FP64 vectors on the integer pipe: every warp scales its 128
// elements of y and of each x_j by their own largest entry; 12 integer
// multiply-adds per element and vector, exact sums, one conversion per warp,
// vector and 128 elements.  n = 786 k, 16 right-hand sides, 20 vectors: 1.20
// ms, 3.8 TB/s; 4 FP64 FMAs per element took 1.97 ms, y read for every vector.
template <int JG>
__global__ void __launch_bounds__(RB) dot_f64_kernel(const double2 *__restrict__ x, int64_t xstride, int k,
                                                     const double2 *__restrict__ y, int64_t n, int64_t chunk,
                                                     double2 *__restrict__ partial, unsigned *__restrict__ ticket,
                                                     double2 *__restrict__ out, int ldh) {
  constexpr int U = 4;  // elements per thread and step
  const int r = blockIdx.y, j0 = blockIdx.z * JG, kg = min(JG, k - j0);
  const double2 *xr = x + j0 * xstride + r * n, *yr = y + r * n;
  const int64_t beg = (int64_t)blockIdx.x * chunk, end = min(beg + chunk, n);
  const double2 zero = make_double2(0.0, 0.0);
  double acc = 0.0;
  for (int64_t t0 = beg; t0 < end; t0 += RB * U) {
    const int64_t i0 = t0 + threadIdx.x;
    double2 a[U];
    int4 c[U];
    int Ey = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      a[u] = i0 + RB * u < end ? __ldg(yr + i0 + RB * u) : zero;
      Ey = max(Ey, exp2of(a[u]));
    }
    Ey = __reduce_max_sync(0xffffffffu, Ey);
    const bool ny = Ey > 0;  // y is not zero here
    Ey = max(Ey, 1);
#pragma unroll
    for (int u = 0; u < U; ++u) c[u] = digits(a[u], min(Ey, fx::kBadExp - 1));
#pragma unroll
    for (int u = 0; u < U; ++u) a[u] = i0 + RB * u < end ? __ldg(xr + i0 + RB * u) : zero;
    WarpSumI ws;
    unsigned nz = 0, bad = 0;  // bits 2 j
#pragma unroll
    for (int j = 0; j < JG; ++j) {
      if (j < kg) {
        double2 b[U];
        int Ex = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          b[u] = a[u];
          Ex = max(Ex, exp2of(b[u]));
        }
        if (j + 1 < kg) {  // the next vector's elements while this one is used
#pragma unroll
          for (int u = 0; u < U; ++u)
            a[u] = i0 + RB * u < end ? __ldg(xr + (j + 1) * xstride + i0 + RB * u) : zero;
        }
        Ex = __reduce_max_sync(0xffffffffu, Ex);
        nz |= Ex > 0 ? 1u << 2 * j : 0u;
        bad |= Ex == fx::kBadExp ? 1u << 2 * j : 0u;
        Ex = max(Ex, 1);
        long long hr = 0, hi = 0, mr = 0, mi = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          macc(digits(b[u], min(Ex, fx::kBadExp - 1)), c[u], hr, hi, mr, mi);
        }
        const int e = 2 * fx::kDigit + Ex + Ey - 2 * (1022 + fx::kVecBits);
        ws.add(2 * j, fx::fold(hr, mr), e);
        ws.add(2 * j + 1, fx::fold(hi, mi), e);
      }
    }
    double t = ws.get();
    unsigned redo = bad | (ny ? nz & fx::ballot_pairs(ws.small()) : 0u);
    if (Ey == fx::kBadExp) redo = 0x55555555u & ((2u << (2 * kg - 1)) - 1u);
    if (redo) t = redo_groups(t, redo, xr, xstride, yr, i0, end);
    acc += t;
  }
  double s;
  const int64_t g = (int64_t)r * gridDim.z + blockIdx.z;
  double *part = reinterpret_cast<double *>(partial) + ((int64_t)r * k + j0) * 2 * gridDim.x;
  if (block_finish<2 * JG>(acc, part, ticket + g, 2 * kg, s) && (int)threadIdx.x < 2 * kg)
    reinterpret_cast<double *>(out + r * ldh + j0)[threadIdx.x] = s;
}

// ---- Krylov bases of FP64 solves are kept as digits (16 bytes per entry, as
// much as the FP64 entries), 57 bits of the largest entry of every tile of
// kTile entries: the vector is converted once, when it is normalised, instead
// of in each of the four passes of its every later orthogonalisation (the
// conversions took two thirds of the instructions of the kernels above).  A
// tile with a nonzero entry more than 2^-kFarTile below its largest, or with
// Inf or NaN, stays as it is in FP64 and is added in FP64; so every entry keeps
// 45 bits at least and most of them 54 or more.  Normal vectors: 0.05% of their
// tiles.
constexpr int kTile = 1024, kFarTile = 12;
constexpr int kRawTile = -1;  // in place of the exponent field of the unit

// v = w inv[r], its digits and the exponent field of each tile's unit (0 for a
// tile of zeros)
__global__ void __launch_bounds__(RB) normalise_kernel(const double2 *w, double2 *v, int4 *__restrict__ vf,
                                                       short *__restrict__ ev, const double *__restrict__ inv,
                                                       int64_t n) {
  constexpr int U = kTile / RB;
  __shared__ int top[RB / 32], low[RB / 32];
  const int r = blockIdx.y;
  const double f = inv[r];
  const int64_t i0 = (int64_t)blockIdx.x * kTile + threadIdx.x;
  double2 x[U];
  int E = 0, lo = fx::kBadExp;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t i = i0 + u * RB;
    x[u] = i < n ? cscale(w[r * n + i], f) : make_double2(0.0, 0.0);
    if (fx::nonzero(x[u].x) || fx::nonzero(x[u].y)) {
      const int e = max(exp2of(x[u]), 1);
      E = max(E, e);
      lo = min(lo, e);
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (i0 + u * RB < n) v[r * n + i0 + u * RB] = x[u];
  E = __reduce_max_sync(0xffffffffu, E);
  lo = __reduce_min_sync(0xffffffffu, lo);
  if ((threadIdx.x & 31) == 0) {
    top[threadIdx.x >> 5] = E;
    low[threadIdx.x >> 5] = lo;
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < RB / 32; ++q) {
    E = max(E, top[q]);
    lo = min(lo, low[q]);
  }
  const bool raw = E == fx::kBadExp || E - lo > kFarTile;
  if (threadIdx.x == 0) ev[(int64_t)r * gridDim.x + blockIdx.x] = (short)(raw ? kRawTile : E);
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t i = i0 + u * RB;
    if (i < n)
      vf[r * n + i] = raw ? make_int4(__double2loint(x[u].x), __double2hiint(x[u].x), __double2loint(x[u].y),
                                      __double2hiint(x[u].y))
                          : digits(x[u], max(E, 1));
  }
}

// an entry of a basis vector; ev: the exponent field of its tile's unit
__device__ __forceinline__ double2 from_digits(int4 q, int ev) {
  if (ev == kRawTile) return make_double2(__hiloint2double(q.y, q.x), __hiloint2double(q.w, q.z));
  const int e = max(ev, 1) - 1022 - fx::kVecBits;
  return make_double2(fx::scaled((double)(((long long)q.x << fx::kDigit) + q.y), e),
                      fx::scaled((double)(((long long)q.z << fx::kDigit) + q.w), e));
}

// redo_groups with the vectors as digits (ev: their tiles' exponents, es apart)
__device__ __noinline__ double redo_digits(double t, unsigned redo, const int4 *__restrict__ x,
                                           const short *__restrict__ ev, int64_t es, int64_t xstride,
                                           const double2 *__restrict__ y, int64_t i0, int64_t end) {
  const int lane = threadIdx.x & 31;
  for (; redo; redo &= redo - 1) {
    const int j = (__ffs(redo) - 1) >> 1;
    double sr = 0.0, si = 0.0;
    for (int64_t i = i0; i < min(end, i0 + kTile); i += RB) {
      const double2 a = from_digits(x[j * xstride + i], ev[j * es]), c = y[i];
      sr = fma(a.x, c.x, fma(a.y, c.y, sr));
      si = fma(a.x, c.y, fma(-a.y, c.x, si));
    }
    fx::WarpSumD ws;
    ws.add(2 * j, sr);
    ws.add(2 * j + 1, si);
    if (lane >> 1 == j) t = ws.get();
  }
  return t;
}

// dot_f64_kernel with the vectors x_j as digits (ev: their tiles' exponents,
// [j][r][tile])
template <int JG>
__global__ void __launch_bounds__(RB, 3) dot_digits_kernel(const int4 *__restrict__ x, const short *__restrict__ ev,
                                                        int64_t xstride, int k, const double2 *__restrict__ y,
                                                        int64_t n, int64_t chunk, double2 *__restrict__ partial,
                                                        unsigned *__restrict__ ticket, double2 *__restrict__ out,
                                                        int ldh) {
  constexpr int U = kTile / RB;
  const int r = blockIdx.y, nrhs = gridDim.y, j0 = blockIdx.z * JG, kg = min(JG, k - j0);
  const int64_t nt = (n + kTile - 1) / kTile;
  const int4 *xr = x + j0 * xstride + r * n;
  const double2 *yr = y + r * n;
  const int64_t beg = (int64_t)blockIdx.x * chunk, end = min(beg + chunk, n);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Ring<kTile> ring{reinterpret_cast<int4 *>(smem_raw)};
  double acc = 0.0;
  for (int64_t t0 = beg; t0 < end; t0 += kTile) {
    const int64_t i0 = t0 + threadIdx.x, tile = t0 / kTile;
#pragma unroll
    for (int j = 0; j < kRing; ++j) {
      if (j < kg) ring.fetch(j, xr + j * xstride + t0, end - t0);
      Ring<kTile>::commit();
    }
    int4 c[U];
    int Ey = 0;
    {
      double2 a[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        a[u] = i0 + RB * u < end ? __ldg(yr + i0 + RB * u) : make_double2(0.0, 0.0);
        Ey = max(Ey, exp2of(a[u]));
      }
      Ey = __reduce_max_sync(0xffffffffu, Ey);
#pragma unroll
      for (int u = 0; u < U; ++u) c[u] = digits(a[u], min(max(Ey, 1), fx::kBadExp - 1));
    }
    const bool ny = Ey > 0;  // y is not zero here
    Ey = max(Ey, 1);
    WarpSumI ws;
#pragma unroll
    for (int j = 0; j < JG; ++j) {
      if (j < kg) {
        const int Ex = ev[((int64_t)(j0 + j) * nrhs + r) * nt + tile];
        long long hr = 0, hi = 0, mr = 0, mi = 0;
        Ring<kTile>::wait();
#pragma unroll
        for (int u = 0; u < U; ++u) macc(ring.get(j % kRing, u), c[u], hr, hi, mr, mi);
        if (j + kRing < kg) ring.fetch(j % kRing, xr + (j + kRing) * xstride + t0, end - t0);
        Ring<kTile>::commit();
        const int e = 2 * fx::kDigit + Ex + Ey - 2 * (1022 + fx::kVecBits);
        ws.add(2 * j, fx::fold(hr, mr), e);
        ws.add(2 * j + 1, fx::fold(hi, mi), e);
      }
    }
    double t = ws.get();
    // the lane's Ex (0 in the lanes past the last vector, as in a tile of zeros)
    const int lane = threadIdx.x & 31;
    const int ex = lane < 2 * kg ? ws.e - (2 * fx::kDigit + Ey - 2 * (1022 + fx::kVecBits)) : 0;
    const unsigned redo =
        fx::ballot_pairs(ex == kRawTile || (ex > 0 && ny && ws.small()) || (Ey == fx::kBadExp && lane < 2 * kg));
    if (redo) t = redo_digits(t, redo, xr, ev + ((int64_t)j0 * nrhs + r) * nt + tile, nrhs * nt, xstride, yr, i0, end);
    acc += t;
  }
  double s;
  const int64_t g = (int64_t)r * gridDim.z + blockIdx.z;
  double *part = reinterpret_cast<double *>(partial) + ((int64_t)r * k + j0) * 2 * gridDim.x;
  if (block_finish<2 * JG>(acc, part, ticket + g, 2 * kg, s) && (int)threadIdx.x < 2 * kg)
    reinterpret_cast<double *>(out + r * ldh + j0)[threadIdx.x] = s;
}

// oqr[r] = <q_r, r_r>, oqq[r] = <q_r, q_r>
template <bool VEC>
__global__ void __launch_bounds__(RB) dot_qr_f32_kernel(const float2 *__restrict__ q, const float2 *__restrict__ rr,
                                                        int64_t n, int64_t chunk, double2 *__restrict__ partial,
                                                        unsigned *__restrict__ ticket, double2 *__restrict__ oqr,
                                                        double2 *__restrict__ oqq) {
  constexpr int U = 2;
  const int r = blockIdx.y;
  const float2 *qr = q + r * n, *xr = rr + r * n;
  const int64_t beg = (int64_t)blockIdx.x * chunk, end = min(beg + chunk, n);
  float sr = 0.f, si = 0.f, sq = 0.f;
  for (int64_t i0 = beg + 2 * threadIdx.x; i0 < end; i0 += 2 * RB * U) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float4 a = ld2<VEC>(qr, i0 + 2 * RB * u, end), c = ld2<VEC>(xr, i0 + 2 * RB * u, end);
      sr = fmaf(a.x, c.x, fmaf(a.y, c.y, fmaf(a.z, c.z, fmaf(a.w, c.w, sr))));
      si = fmaf(a.x, c.y, fmaf(-a.y, c.x, fmaf(a.z, c.w, fmaf(-a.w, c.z, si))));
      sq = fmaf(a.x, a.x, fmaf(a.y, a.y, fmaf(a.z, a.z, fmaf(a.w, a.w, sq))));
    }
  }
  WarpSumF ws;
  ws.add(0, sr);
  ws.add(1, si);
  ws.add(2, sq);
  if (ws.bad()) {
    ws.fix(0, sr);
    ws.fix(1, si);
    ws.fix(2, sq);
  }
  double s;
  double *part = reinterpret_cast<double *>(partial) + (int64_t)r * 4 * gridDim.x;
  if (block_finish<4>(ws.get(), part, ticket + r, 3, s) && threadIdx.x < 3) {
    if (threadIdx.x == 0) oqr[r].x = s;
    else if (threadIdx.x == 1) oqr[r].y = s;
    else oqq[r] = make_double2(s, 0.0);
  }
}

__global__ void __launch_bounds__(RB) dot_qr_f64_kernel(const double2 *__restrict__ q, const double2 *__restrict__ rr,
                                                        int64_t n, int64_t chunk, double2 *__restrict__ partial,
                                                        unsigned *__restrict__ ticket, double2 *__restrict__ oqr,
                                                        double2 *__restrict__ oqq) {
  constexpr int U = 4;
  const int r = blockIdx.y;
  const double2 *qr = q + r * n, *xr = rr + r * n;
  const int64_t beg = (int64_t)blockIdx.x * chunk, end = min(beg + chunk, n);
  const double2 zero = make_double2(0.0, 0.0);
  double acc = 0.0;
  for (int64_t t0 = beg; t0 < end; t0 += RB * U) {
    double2 a[U], c[U];
    int Ea = 0, Ec = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = t0 + threadIdx.x + RB * u;
      a[u] = i < end ? __ldg(qr + i) : zero;
      c[u] = i < end ? __ldg(xr + i) : zero;
      Ea = max(Ea, exp2of(a[u]));
      Ec = max(Ec, exp2of(c[u]));
    }
    Ea = __reduce_max_sync(0xffffffffu, Ea);
    Ec = __reduce_max_sync(0xffffffffu, Ec);
    const bool nz = Ea > 0 && Ec > 0;
    Ea = max(Ea, 1);
    Ec = max(Ec, 1);
    long long hr = 0, hi = 0, mr = 0, mi = 0, hq = 0, mq = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int4 p = digits(a[u], min(Ea, fx::kBadExp - 1)), w = digits(c[u], min(Ec, fx::kBadExp - 1));
      macc(p, w, hr, hi, mr, mi);
      hq = fx::madw(p.z, p.z, fx::madw(p.x, p.x, hq));
      mq = fx::madw(2 * p.w, p.z, fx::madw(2 * p.y, p.x, mq));
    }
    const int e = 2 * fx::kDigit + Ea + Ec - 2 * (1022 + fx::kVecBits);
    const int eq = 2 * fx::kDigit + 2 * Ea - 2 * (1022 + fx::kVecBits);
    const bool ba = Ea == fx::kBadExp, bc = ba || Ec == fx::kBadExp;
    WarpSumI ws;
    ws.add(0, fx::fold(hr, mr), e);
    ws.add(1, fx::fold(hi, mi), e);
    ws.add(2, fx::fold(hq, mq), eq);  // at least 2^-2 of its scale
    double t = ws.get();
    const int64_t i0 = t0 + threadIdx.x;
    if (bc || (nz && (fx::ballot_pairs(ws.small()) & 1u))) {
      const double p = redo_groups(t, 1u, qr, 0, xr, i0, end);
      if ((threadIdx.x & 31) < 2) t = p;
    }
    if (ba) {
      const double p = redo_groups(t, 4u, qr, 0, qr, i0, end);  // value 2: the real part
      if ((threadIdx.x & 31) == 2) t = p;
    }
    acc += t;
  }
  double s;
  double *part = reinterpret_cast<double *>(partial) + (int64_t)r * 4 * gridDim.x;
  if (block_finish<4>(acc, part, ticket + r, 3, s) && threadIdx.x < 3) {
    if (threadIdx.x == 0) oqr[r].x = s;
    else if (threadIdx.x == 1) oqr[r].y = s;
    else oqq[r] = make_double2(s, 0.0);
  }
}

// w_r += sign sum_j h[r * ldh + j] V_j,r
__global__ void __launch_bounds__(256) multi_axpy_f32_kernel(const float2 *__restrict__ V, int64_t vstride, int k,
                                                             float2 *__restrict__ w, int64_t n,
                                                             const double2 *__restrict__ h, int ldh, double sign) {
  __shared__ float2 coef[128];
  const int r = blockIdx.y;
  for (int j = threadIdx.x; j < k; j += blockDim.x) {
    const double2 c = h[r * ldh + j];
    coef[j] = make_float2((float)(sign * c.x), (float)(sign * c.y));
  }
  __syncthreads();
  float2 *wr = w + r * n;
  const float2 *Vr = V + r * n;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float2 a = wr[i];
#pragma unroll 4
    for (int j = 0; j < k; ++j) a = cfma(coef[j], Vr[j * vstride + i], a);
    wr[i] = a;
  }
}

// The same sums through the ring for 16-byte aligned vectors of even length: one
// tile of 1024 elements per block.  NORM: also nrm[r].x = <w_r, w_r> of the
// result, in the order of the dots.  n = 786 k, 8 right-hand sides, 1 .. 16
// vectors: 82 us on average with the norm (71 and 30 us as two launches).
template <bool NORM>
__global__ void __launch_bounds__(RB) multi_axpy_f32_ring_kernel(const int4 *__restrict__ V, int64_t vs, int k,
                                                                 float4 *__restrict__ w, int64_t n,
                                                                 const double2 *__restrict__ h, int ldh, double sign,
                                                                 double *__restrict__ partial,
                                                                 unsigned *__restrict__ ticket,
                                                                 double2 *__restrict__ nrm) {
  constexpr int U = kTileF / RB;
  using R = Ring<kTileF>;
  __shared__ float2 coef[128];
  const int r = blockIdx.y;
  const int64_t t0 = (int64_t)blockIdx.x * kTileF, i0 = t0 + threadIdx.x;  // pairs of elements, as n and vs
  float4 *wr = w + r * n;
  const int4 *Vr = V + r * n + t0;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const R ring{reinterpret_cast<int4 *>(smem_raw)};
#pragma unroll
  for (int j = 0; j < kRing; ++j) {
    if (j < k) ring.fetch(j, Vr + j * vs, n - t0);
    R::commit();
  }
  float4 acc[U];
#pragma unroll
  for (int u = 0; u < U; ++u) acc[u] = i0 + u * RB < n ? wr[i0 + u * RB] : make_float4(0.f, 0.f, 0.f, 0.f);
  for (int j = threadIdx.x; j < k; j += RB) {
    const double2 c = h[r * ldh + j];
    coef[j] = make_float2((float)(sign * c.x), (float)(sign * c.y));
  }
  __syncthreads();
#pragma unroll 4
  for (int j = 0; j < k; ++j) {
    const float2 c = coef[j];
    R::wait();
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float4 v = ring.getf(j % kRing, u);
      const float2 a = cfma(c, make_float2(v.x, v.y), make_float2(acc[u].x, acc[u].y));
      const float2 b = cfma(c, make_float2(v.z, v.w), make_float2(acc[u].z, acc[u].w));
      acc[u] = make_float4(a.x, a.y, b.x, b.y);
    }
    if (j + kRing < k) ring.fetch(j % kRing, Vr + (j + kRing) * vs, n - t0);
    R::commit();
  }
  float q = 0.f;
#pragma unroll
  for (int u = 0; u < U; ++u) {
    if (i0 + u * RB < n) wr[i0 + u * RB] = acc[u];
    q = fmaf(acc[u].x, acc[u].x, fmaf(acc[u].y, acc[u].y, fmaf(acc[u].z, acc[u].z, fmaf(acc[u].w, acc[u].w, q))));
  }
  if constexpr (NORM) {
    WarpSumF ws;
    ws.add(0, q);
    if (ws.bad()) ws.fix(0, q);
    double s;
    if (block_finish<4>(ws.get(), partial + (int64_t)r * gridDim.x, ticket + r, 1, s) && threadIdx.x == 0)
      nrm[r] = make_double2(s, 0.0);
  }
}

// exponent of a zero coefficient or tile: its products take no part in a scale
constexpr int kNone = -(1 << 20);

// The same for FP64 vectors on the integer pipe: JG vectors at a time are
// added as integers in the unit of the largest coefficient times entry of
// the warp's 64 elements, then once to w in FP64.  n = 786 k, 16 right-hand
// sides, 1 .. 20 vectors: 705 us on average (3.6 TB/s) against 931 us in FP64.
// The digits lose up to 2^-53 of the group's largest product (16 real products x
// 2^-57); an element whose own largest is more than 2^-kFar below that, its
// entries far smaller than its neighbours', is added in FP64 instead: 0.02% of
// the elements of normal vectors where one coefficient dominates, none else.
__global__ void __launch_bounds__(256) multi_axpy_f64_kernel(const double2 *__restrict__ V, int64_t vstride, int k,
                                                             double2 *__restrict__ w, int64_t n,
                                                             const double2 *__restrict__ h, int ldh, double sign) {
  constexpr int JG = 8, U = 2, kFar = 8;
  __shared__ int4 cd[128];
  __shared__ int ce[128];
  __shared__ double2 coef[128];
  const int r = blockIdx.y;
  for (int j = threadIdx.x; j < k; j += blockDim.x) {
    double2 c = h[r * ldh + j];
    c = make_double2(sign * c.x, sign * c.y);
    const int E = max(exp2of(c), 1);
    coef[j] = c;
    ce[j] = c.x == 0.0 && c.y == 0.0 ? kNone : E;
    cd[j] = digits(c, min(E, fx::kBadExp - 1));
  }
  __syncthreads();
  double2 *wr = w + r * n;
  const double2 *Vr = V + r * n;
  const int64_t step = (int64_t)gridDim.x * blockDim.x * U;
  for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x * U; t0 < n; t0 += step) {
    // lanes past the end work on zeros (the warp scales together)
    const int64_t i0 = t0 + threadIdx.x;
    double2 acc[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = i0 + (int64_t)u * blockDim.x;
      acc[u] = i < n ? wr[i] : make_double2(0.0, 0.0);
    }
    for (int j0 = 0; j0 < k; j0 += JG) {
      const int kg = min(JG, k - j0);
      double2 v[JG][U];
#pragma unroll
      for (int j = 0; j < JG; ++j)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int64_t i = i0 + (int64_t)u * blockDim.x;
          v[j][u] = j < kg && i < n ? __ldg(Vr + (j0 + j) * vstride + i) : make_double2(0.0, 0.0);
        }
      // largest exponent sum of a coefficient and its entries, by element
      int top[U];
      bool bad = false;
#pragma unroll
      for (int u = 0; u < U; ++u) top[u] = 0;
#pragma unroll
      for (int j = 0; j < JG; ++j) {
        if (j < kg) {
          bad |= ce[j0 + j] == fx::kBadExp;
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int e = max(exp2of(v[j][u]), 1);
            bad |= e == fx::kBadExp;
            if (fx::nonzero(v[j][u].x) || fx::nonzero(v[j][u].y)) top[u] = max(top[u], e + ce[j0 + j]);
          }
        }
      }
      int S = 0;
#pragma unroll
      for (int u = 0; u < U; ++u) S = max(S, top[u]);
      S = __reduce_max_sync(0xffffffffu, S);
      const int ex = S - 2 * (1022 + fx::kVecBits) + 2 * fx::kDigit;
      const bool any_bad = __any_sync(0xffffffffu, bad);
      if (S == 0 && !any_bad) continue;  // only products with zeros
      if (any_bad || ex < -1000 || ex > 900) {
#pragma unroll
        for (int j = 0; j < JG; ++j)
          if (j < kg)
#pragma unroll
            for (int u = 0; u < U; ++u) acc[u] = cfma(coef[j0 + j], v[j][u], acc[u]);
        continue;
      }
      long long hr[U], hi[U], mr[U], mi[U];
#pragma unroll
      for (int u = 0; u < U; ++u) hr[u] = hi[u] = mr[u] = mi[u] = 0;
#pragma unroll
      for (int j = 0; j < JG; ++j) {
        if (j < kg) {
          const int4 c = cd[j0 + j];
          // the entries in the unit that makes c v come out in units of 2^ex;
          // a far smaller product vanishes against the largest
          const int E = S - ce[j0 + j];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            mac(c, digits(v[j][u], E), hr[u], hi[u], mr[u], mi[u]);
          }
        }
      }
      const double f = __longlong_as_double((long long)(ex + 1023) << 52);
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (top[u] && S - top[u] > kFar) {
#pragma unroll
          for (int j = 0; j < JG; ++j)
            if (j < kg) acc[u] = cfma(coef[j0 + j], v[j][u], acc[u]);
          continue;
        }
        acc[u].x = fma(f, (double)fx::fold(hr[u], mr[u]), acc[u].x);
        acc[u].y = fma(f, (double)fx::fold(hi[u], mi[u]), acc[u].y);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = i0 + (int64_t)u * blockDim.x;
      if (i < n) wr[i] = acc[u];
    }
  }
}

// in place of it: a product that is added in FP64 (tile in FP64, Inf or NaN
// coefficient, near the ends of the range)
constexpr int kInFp64 = -(1 << 21);

// The same with the vectors as digits: one tile of kTile elements per block,
// whose units are the vectors' own, so a product is shifted to the largest
// unit of its group of JG before it is added.  NORM: also nrm[r].x = <w_r, w_r>
// of the result (one pass over w less, 133 us of 560 at n = 786 k and 16
// right-hand sides; partial, ticket as for the dots).
template <bool NORM>
__global__ void __launch_bounds__(RB) multi_axpy_digits_kernel(const int4 *__restrict__ V, const short *__restrict__ ev,
                                                               int64_t vs, int k, double2 *__restrict__ w, int64_t n,
                                                               const double2 *__restrict__ h, int ldh, double sign,
                                                               double *__restrict__ partial,
                                                               unsigned *__restrict__ ticket,
                                                               double2 *__restrict__ nrm) {
  constexpr int JG = 8, U = kTile / RB;
  __shared__ int4 cd[128];
  __shared__ int ce[128];  // exponent of coefficient times tile
  __shared__ double2 coef[128];
  const int r = blockIdx.y, nrhs = gridDim.y;
  const int64_t nt = gridDim.x;
  int slow = 0;  // some products are left to FP64 (ce = kInFp64)
  for (int j = threadIdx.x; j < k; j += blockDim.x) {
    double2 c = h[r * ldh + j];
    c = make_double2(sign * c.x, sign * c.y);
    const int E = max(exp2of(c), 1), Ev = ev[((int64_t)j * nrhs + r) * nt + blockIdx.x];
    coef[j] = c;
    const bool fp64 = E == fx::kBadExp || Ev == kRawTile;
    ce[j] = fp64 ? kInFp64 : Ev == 0 || (c.x == 0.0 && c.y == 0.0) ? kNone : E + Ev;
    cd[j] = fp64 ? make_int4(0, 0, 0, 0) : digits(c, E);
    slow |= fp64;
  }
  slow = __syncthreads_or(slow);
  const int64_t t0 = (int64_t)blockIdx.x * kTile, i0 = t0 + threadIdx.x;
  double2 *wr = w + r * n;
  const int4 *Vr = V + r * n;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const Ring<kTile> ring{reinterpret_cast<int4 *>(smem_raw)};
#pragma unroll
  for (int j = 0; j < kRing; ++j) {
    if (j < k) ring.fetch(j, Vr + j * vs + t0, n - t0);
    Ring<kTile>::commit();
  }
  double2 acc[U];
#pragma unroll
  for (int u = 0; u < U; ++u) acc[u] = i0 + u * RB < n ? wr[i0 + u * RB] : make_double2(0.0, 0.0);
  for (int j0 = 0; j0 < k; j0 += JG) {
    const int kg = min(JG, k - j0);
    int S = kNone;
    for (int j = 0; j < kg; ++j) S = max(S, ce[j0 + j]);  // kInFp64 is below all
    const int ex = S - 2 * (1022 + fx::kVecBits) + 2 * fx::kDigit;
    if (ex < -1000 || ex > 900) {
      // only products with zeros or left to FP64, as those near the ends of the
      // range; the ring keeps its order
      for (int j = 0; j < kg; ++j) {
        Ring<kTile>::wait();
        if (j0 + j + kRing < k) ring.fetch(j % kRing, Vr + (j0 + j + kRing) * vs + t0, n - t0);
        Ring<kTile>::commit();
      }
      __syncthreads();
      if ((int)threadIdx.x < kg && ce[j0 + threadIdx.x] != kNone) ce[j0 + threadIdx.x] = kInFp64;
      slow |= S != kNone;
      continue;
    }
    long long sr[U], si[U];
#pragma unroll
    for (int u = 0; u < U; ++u) sr[u] = si[u] = 0;
#pragma unroll
    for (int j = 0; j < JG; ++j) {
      if (j < kg) {
        const int4 c = cd[j0 + j];
        const int sh = min(S - ce[j0 + j], 63);
        Ring<kTile>::wait();
#pragma unroll
        for (int u = 0; u < U; ++u) {
          long long hr = 0, hi = 0, mr = 0, mi = 0;
          mac(c, ring.get(j % kRing, u), hr, hi, mr, mi);  // j0 is a multiple of kRing
          sr[u] += fx::fold(hr, mr) >> sh;
          si[u] += fx::fold(hi, mi) >> sh;
        }
        if (j0 + j + kRing < k) ring.fetch(j % kRing, Vr + (j0 + j + kRing) * vs + t0, n - t0);
        Ring<kTile>::commit();
      }
    }
    static_assert(JG % kRing == 0, "ring slots of a group");
    const double f = __longlong_as_double((long long)(ex + 1023) << 52);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      acc[u].x = fma(f, (double)sr[u], acc[u].x);
      acc[u].y = fma(f, (double)si[u], acc[u].y);
    }
  }
  if (slow) {
    __syncthreads();
#pragma unroll 1
    for (int j = 0; j < k; ++j) {
      if (ce[j] != kInFp64) continue;
      const int Ev = ev[((int64_t)j * nrhs + r) * nt + blockIdx.x];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (i0 + u * RB < n) acc[u] = cfma(coef[j], from_digits(Vr[j * vs + i0 + u * RB], Ev), acc[u]);
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u)
    if (i0 + u * RB < n) wr[i0 + u * RB] = acc[u];
  if constexpr (NORM) {
    int E = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (i0 + u * RB >= n) acc[u] = make_double2(0.0, 0.0);
      E = max(E, exp2of(acc[u]));
    }
    E = warp_exp(E);
    long long hq = 0, mq = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int4 q = digits(acc[u], min(E, fx::kBadExp - 1));
      hq = fx::madw(q.z, q.z, fx::madw(q.x, q.x, hq));
      mq = fx::madw(2 * q.w, q.z, fx::madw(2 * q.y, q.x, mq));
    }
    WarpSumI ws;
    ws.add(0, fx::fold(hq, mq), 2 * fx::kDigit + 2 * E - 2 * (1022 + fx::kVecBits));
    double t = ws.get();
    if (E == fx::kBadExp) {  // acc holds Inf or NaN
      double q = 0.0;
      for (int u = 0; u < U; ++u) q = fma(acc[u].x, acc[u].x, fma(acc[u].y, acc[u].y, q));
      fx::WarpSumD wd;
      wd.add(0, q);
      t = wd.get();
    }
    double s;
    if (block_finish<4>(t, partial + (int64_t)r * nt, ticket + r, 1, s) && threadIdx.x == 0)
      nrm[r] = make_double2(s, 0.0);
  }
}

// W complex entries moved by one access (16 bytes: 2 FP32 or 1 FP64 ones)
template <typename T, int W> struct alignas(W * sizeof(C<T>) < 16 ? sizeof(C<T>) : 16) Pack {
  C<T> v[W];
};
template <typename T, int W> __device__ __forceinline__ Pack<T, W> ldp(const C<T> *p) {
  return *reinterpret_cast<const Pack<T, W> *>(p);
}
template <typename T, int W> __device__ __forceinline__ void stp(C<T> *p, const Pack<T, W> &v) {
  *reinterpret_cast<Pack<T, W> *>(p) = v;
}
// first entry of the thread's pack, entries between its packs
#define MG_PACKS(i, W, n)                                                                          \
  for (int64_t i = (int64_t)(W) * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x); i < (n);       \
       i += (int64_t)(W)*gridDim.x * blockDim.x)

template <typename T, int W>
__global__ void axpby_kernel(T a, const C<T> *__restrict__ x, T b, C<T> *__restrict__ y, int64_t n) {
  MG_PACKS(i, W, n) {
    const Pack<T, W> xv = ldp<T, W>(x + i);
    Pack<T, W> yv = ldp<T, W>(y + i);
#pragma unroll
    for (int q = 0; q < W; ++q) {
      yv.v[q].x = a * xv.v[q].x + b * yv.v[q].x;
      yv.v[q].y = a * xv.v[q].y + b * yv.v[q].y;
    }
    stp<T, W>(y + i, yv);
  }
}

template <typename T, int W>
__global__ void scale_rhs_kernel(const C<T> *x, C<T> *y,  // may alias (in-place scaling)
                                 const double *__restrict__ scal, int64_t n) {
  const int64_t o = blockIdx.y * n;
  const T f = (T)scal[blockIdx.y];
  MG_PACKS(i, W, n) {
    Pack<T, W> v = ldp<T, W>(x + o + i);
#pragma unroll
    for (int q = 0; q < W; ++q) v.v[q] = cscale(v.v[q], f);
    stp<T, W>(y + o + i, v);
  }
}

template <typename T, int W>
__global__ void subtract_kernel(const C<T> *__restrict__ a, const C<T> *__restrict__ b, C<T> *__restrict__ d, int64_t n) {
  MG_PACKS(i, W, n) {
    Pack<T, W> v = ldp<T, W>(a + i);
    const Pack<T, W> w = ldp<T, W>(b + i);
#pragma unroll
    for (int q = 0; q < W; ++q) v.v[q] = csub(v.v[q], w.v[q]);
    stp<T, W>(d + i, v);
  }
}

// z += alpha e; r -= alpha q with alpha = <q, r> / <q, q> per rhs, alpha = 0
// where <q, q> is not above `tiny`.  MR_RES: along the residual itself;
// MR_DIR: along a given direction e; MR_FIRST: along the residual e of z = 0,
// neither z nor r holding anything yet.
enum MrMode { MR_RES, MR_DIR, MR_FIRST };
template <typename T, int W, MrMode MODE>
__global__ void mr_update_kernel(C<T> *__restrict__ z, C<T> *__restrict__ res, const C<T> *__restrict__ e,
                                 const C<T> *__restrict__ q, const double2 *__restrict__ dqr,
                                 const double2 *__restrict__ nq, int64_t n, double tiny) {
  const int r = blockIdx.y;
  const double qq = nq[r].x;
  const double2 d = dqr[r];
  const C<T> al = qq > tiny ? mk<T>((T)(d.x / qq), (T)(d.y / qq)) : mk<T>((T)0, (T)0);
  const int64_t o = r * n;
  MG_PACKS(i, W, n) {
    Pack<T, W> zv, rv = ldp<T, W>((MODE == MR_FIRST ? e : res) + o + i);
    const Pack<T, W> qv = ldp<T, W>(q + o + i);
    const Pack<T, W> ev = MODE == MR_DIR ? ldp<T, W>(e + o + i) : rv;
    if (MODE != MR_FIRST) zv = ldp<T, W>(z + o + i);
#pragma unroll
    for (int k = 0; k < W; ++k) {
      zv.v[k] = cfma(al, ev.v[k], MODE == MR_FIRST ? mk<T>((T)0, (T)0) : zv.v[k]);
      rv.v[k] = cfma(cneg(al), qv.v[k], rv.v[k]);
    }
    stp<T, W>(z + o + i, zv);
    stp<T, W>(res + o + i, rv);
  }
}

template <typename To, typename From>
__global__ void convert_kernel(const C<From> *__restrict__ in, C<To> *__restrict__ out, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = cvt<To>(in[i]);
}

template <typename To, typename From>
__global__ void convert_scale_kernel(const C<From> *__restrict__ in, C<To> *__restrict__ out,
                                     const double *__restrict__ scal, int64_t n) {
  const int r = blockIdx.y;
  const double f = scal[r];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    C<From> v = in[r * n + i];
    out[r * n + i] = mk<To>((To)(v.x * f), (To)(v.y * f));
  }
}

// y_r = x_r * scal[r] (scal may be null: 1) between the canonical order
// [site][12] and the fine level's structure-of-arrays order (to_soa: x
// canonical, y SoA; else the reverse), converting precision.  A block takes
// 128 sites of one right-hand side through shared memory, so that both sides
// move whole lines: 16-byte chunks in the structure-of-arrays order, and
// consecutive entries in the canonical one (8-byte accesses where a buffer is
// not aligned to 16).  Bound: memory; with scattered 8-byte accesses on one
// side and no staging it moved 1.4 TB/s.  Without scale factors nothing is
// multiplied: FP32 to FP32 through an FP64 product by one kept the FP64 pipe
// busy for most of the launch (9 us for 35 k sites; a one-sweep smoothing of
// 12^3 x 20 with two of them 56 us, now 48).
constexpr int kRelayoutSites = 128;

template <typename T, bool VEC> __device__ __forceinline__ Pack<T, 2> ld_pair(const C<T> *p) {
  if (VEC) return ldp<T, 2>(p);
  Pack<T, 2> v;
  v.v[0] = p[0];
  v.v[1] = p[1];
  return v;
}

template <typename To, typename From, bool VEC>
__global__ void __launch_bounds__(256) relayout_kernel(const C<From> *__restrict__ x, C<To> *__restrict__ y,
                                                       const double *__restrict__ scal, int64_t V, bool to_soa) {
  constexpr int S = kRelayoutSites;
  __shared__ Pack<To, 2> sh[6][S + 1];  // + 1: the six chunks of a site on different banks
  const int r = blockIdx.y;
  const double f = scal ? scal[r] : 1.0;
  const int64_t s0 = (int64_t)blockIdx.x * S;
  const int ns = (int)(V - s0 < S ? V - s0 : S);
  const C<From> *xr = x + r * V * 12;
  C<To> *yr = y + r * V * 12;
  // pairs of components: canonical position p = 6 site + chunk, SoA position
  // (chunk, site)
#pragma unroll
  for (int q = 0; q < 6 * S / 256; ++q) {
    const int p = q * 256 + threadIdx.x;
    const int site = to_soa ? p / 6 : p % S, k = to_soa ? p - site * 6 : p / S;
    if (site < ns) {
      const C<From> *src = xr + (to_soa ? (s0 * 6 + p) * 2 : ((int64_t)k * V + s0 + site) * 2);
      const Pack<From, 2> v = ld_pair<From, VEC>(src);
      Pack<To, 2> o;
#pragma unroll
      for (int j = 0; j < 2; ++j)
        o.v[j] = scal ? mk<To>((To)(v.v[j].x * f), (To)(v.v[j].y * f)) : mk<To>((To)v.v[j].x, (To)v.v[j].y);
      sh[k][site] = o;
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 6 * S / 256; ++q) {
    const int p = q * 256 + threadIdx.x;
    const int site = to_soa ? p % S : p / 6, k = to_soa ? p / S : p - site * 6;
    if (site < ns) {
      C<To> *dst = yr + (to_soa ? ((int64_t)k * V + s0 + site) * 2 : (s0 * 6 + p) * 2);
      if (VEC) {
        stp<To, 2>(dst, sh[k][site]);
      } else {
        dst[0] = sh[k][site].v[0];
        dst[1] = sh[k][site].v[1];
      }
    }
  }
}

template <typename T, typename Tlo>
__global__ void add_lo_kernel(const C<Tlo> *__restrict__ x, C<T> *__restrict__ y, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    C<T> v = y[i];
    C<Tlo> a = x[i];
    v.x += (T)a.x;
    v.y += (T)a.y;
    y[i] = v;
  }
}

template <typename T>
__global__ void finite_kernel(const C<T> *__restrict__ x, int64_t n, int *flag) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    C<T> v = x[i];
    if (!isfinite(v.x) || !isfinite(v.y)) {
      *flag = 1;
      return;
    }
  }
}

inline int grid_for(int64_t n) {
  int64_t b = (n + 255) / 256;
  return (int)(b < 152 * 16 ? (b < 1 ? 1 : b) : 152 * 16);
}

// ----------------------------------------------------------------- FGMRES
__device__ __forceinline__ double2 dcmul(double2 a, double2 b) { return cmul(a, b); }

__global__ void gmres_start_kernel(GmresState st) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= st.nrhs) return;
  const int m = st.m;
  const double beta = sqrt(fmax(st.nrm[r].x, 0.0));
  for (int i = 0; i <= m; ++i) st.g[r * (m + 1) + i] = make_double2(0.0, 0.0);
  st.g[r * (m + 1)] = make_double2(beta, 0.0);
  for (int i = 0; i < m; ++i) st.y[r * m + i] = make_double2(0.0, 0.0);
  st.res[r] = beta;
  st.nit[r] = 0;
  const int act = (beta > st.target[r]) && isfinite(beta);
  st.active[r] = act;
  st.inv[r] = (act && beta > 0.0) ? 1.0 / beta : 0.0;
}

// One warp per right-hand side: its lanes bring the coefficients and the
// previous rotations in and the column out together, lane 0 rotates (a chain
// of FP64 operations; with every operand of it loaded in turn from memory an
// iteration with 20 vectors took 20 us).
__global__ void __launch_bounds__(32) gmres_arnoldi_kernel(GmresState st, int i) {
  __shared__ double2 col[66], sn[64];
  __shared__ double cs[64];
  const int r = blockIdx.x, lane = threadIdx.x;
  if (!st.active[r]) return;
  const int m = st.m;
  double2 *out = st.H + (int64_t)r * (m + 1) * m + i * (m + 1);
  for (int j = lane; j <= i; j += 32) {
    const double2 a = st.h1[r * (m + 1) + j], b = st.h2[r * (m + 1) + j];
    col[j] = make_double2(a.x + b.x, a.y + b.y);
    if (j < i) {
      cs[j] = st.cs[r * m + j];
      sn[j] = st.sn[r * m + j];
    }
  }
  __syncwarp();
  const double hn = sqrt(fmax(st.nrm[r].x, 0.0));
  if (lane == 0) {
    col[i + 1] = make_double2(hn, 0.0);
    // previous rotations
    for (int j = 0; j < i; ++j) {
      const double c = cs[j];
      const double2 s = sn[j];
      const double2 a = col[j], b = col[j + 1];
      col[j] = cadd(cscale(a, c), dcmul(s, b));
      col[j + 1] = csub(cscale(b, c), dcmul(cconj(s), a));
    }
    // new rotation zeroing col[i+1] (real, >= 0)
    const double2 a = col[i];
    const double b = col[i + 1].x;
    const double aa = sqrt(cabs2(a));
    const double rr = sqrt(aa * aa + b * b);
    double c;
    double2 s;
    if (rr == 0.0) {
      c = 1.0;
      s = make_double2(0.0, 0.0);
    } else if (aa == 0.0) {
      c = 0.0;
      s = make_double2(1.0, 0.0);
      col[i] = make_double2(rr, 0.0);
    } else {
      c = aa / rr;
      const double2 ph = make_double2(a.x / aa, a.y / aa);
      s = cscale(ph, b / rr);
      col[i] = cscale(ph, rr);
    }
    col[i + 1] = make_double2(0.0, 0.0);
    st.cs[r * m + i] = c;
    st.sn[r * m + i] = s;
    double2 *g = st.g + r * (m + 1);
    const double2 gi = g[i];
    g[i + 1] = cneg(dcmul(cconj(s), gi));
    g[i] = cscale(gi, c);
    const double res = sqrt(cabs2(g[i + 1]));
    st.res[r] = res;
    st.nit[r] = i + 1;
    const bool done = !(res > st.target[r]) || hn == 0.0 || !isfinite(res) || rr == 0.0;
    if (done) {
      st.active[r] = 0;
      st.inv[r] = 0.0;
    } else {
      st.inv[r] = 1.0 / hn;
    }
  }
  __syncwarp();
  for (int j = lane; j <= i + 1; j += 32) out[j] = col[j];
}

// Back substitution with one warp per right-hand side: the right-hand side in
// shared memory, each solved entry taken from all others at once.
__global__ void __launch_bounds__(32) gmres_solve_kernel(GmresState st) {
  __shared__ double2 acc[64];
  const int r = blockIdx.x, lane = threadIdx.x;
  const int m = st.m;
  const int k = st.nit[r];
  const double2 *H = st.H + (int64_t)r * (m + 1) * m;
  double2 *y = st.y + r * m;
  for (int j = lane; j < k; j += 32) acc[j] = st.g[r * (m + 1) + j];
  for (int j = k + lane; j < m; j += 32) y[j] = make_double2(0.0, 0.0);
  for (int j = k - 1; j >= 0; --j) {
    const double2 *col = H + j * (m + 1);
    __syncwarp();
    const double2 a = acc[j], d = col[j];
    const double dd = cabs2(d);
    const double2 yj = dd > 0.0 ? make_double2((a.x * d.x + a.y * d.y) / dd, (a.y * d.x - a.x * d.y) / dd)
                                : make_double2(0.0, 0.0);
    if (lane == 0) y[j] = yj;
    for (int l = lane; l < j; l += 32) acc[l] = csub(acc[l], dcmul(col[l], yj));
  }
}
}  // namespace

std::atomic<int64_t> &launch_counter() {
  static std::atomic<int64_t> c{0};
  return c;
}

namespace {
std::atomic<unsigned> g_staging_extra{0};
}
void set_staging_extra_bytes(unsigned bytes) { g_staging_extra.store(bytes); }
unsigned staging_extra_bytes() { return g_staging_extra.load(); }

namespace {
std::atomic<int> g_alloc_failures{0};
std::atomic<size_t> g_alloc_failure_bytes{0};
}
void set_alloc_failures(int n, size_t bytes) {
  g_alloc_failure_bytes.store(bytes);
  g_alloc_failures.store(n);
}
cudaError_t device_malloc(void **p, size_t bytes) {
  if (g_alloc_failures.load(std::memory_order_relaxed) > 0 && bytes >= g_alloc_failure_bytes.load() &&
      g_alloc_failures.fetch_sub(1) > 0)
    return cudaErrorMemoryAllocation;
  return cudaMalloc(p, bytes);
}

void smem_optin(const void *func, int bytes) {
  static std::mutex mu;
  static std::map<std::pair<const void *, int>, int> done;  // (kernel, device) -> bytes set
  int dev = 0;
  MG_CUDA(cudaGetDevice(&dev));
  std::lock_guard<std::mutex> lock(mu);
  auto key = std::make_pair(func, dev);
  auto it = done.find(key);
  if (it != done.end() && it->second >= bytes) return;
  MG_CUDA(cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  done[key] = bytes;
}

// blocks of a reduction: chunks of 1024 elements (one step of a block), at
// most 4096 blocks, whose blocks then take several steps.  The cap bounds the
// FP32 chain of a thread, n / 2^20 elements: 16 up to n = 16.8 M (1024 blocks:
// 48 at 32^4, 488 at 48^3 x 96)
int reduce_blocks(int64_t n) {
  int64_t b = (n + 1023) / 1024;
  if (b < 1) b = 1;
  if (b > 4096) b = 4096;
  return (int)b;
}

namespace {
// elements per block, a multiple of one step's
int64_t reduce_chunk(int64_t n) {
  const int64_t c = (n + reduce_blocks(n) - 1) / reduce_blocks(n);
  return (c + 1023) / 1024 * 1024;
}
// blocks that have elements at that chunk
int blocks_of(int64_t n) { return div_up(n, reduce_chunk(n)); }
template <typename... P> bool aligned16(int64_t stride, P... p) {
  uintptr_t a = 0;
  ((a |= (uintptr_t)p), ...);
  return (a & 15) == 0 && stride % 2 == 0;
}

template <typename T, int JG>
void launch_dot(const C<T> *V, int64_t vstride, int k, const C<T> *w, int64_t n, int nrhs, double2 *h, int ldh,
                RedScratch scr, cudaStream_t s) {
  const dim3 grid(blocks_of(n), nrhs, (k + JG - 1) / JG);
  const int64_t chunk = reduce_chunk(n);
  if constexpr (sizeof(T) == 8) {
    dot_f64_kernel<JG><<<grid, RB, 0, s>>>(V, vstride, k, w, n, chunk, scr.partial, scr.ticket, h, ldh);
  } else if (!aligned16(n | vstride, V, w)) {
    dot_f32_kernel<JG, false><<<grid, RB, 0, s>>>(V, vstride, k, w, n, chunk, scr.partial, scr.ticket, h, ldh);
  } else if constexpr (JG == 1) {
    dot_f32_kernel<JG, true><<<grid, RB, 0, s>>>(V, vstride, k, w, n, chunk, scr.partial, scr.ticket, h, ldh);
  } else {
    constexpr int sm = kRing * kTileF * (int)sizeof(int4);
    smem_optin((const void *)dot_f32_ring_kernel<JG>, sm);
    dot_f32_ring_kernel<JG><<<grid, RB, sm, s>>>(reinterpret_cast<const int4 *>(V), vstride / 2, k,
                                                 reinterpret_cast<const float4 *>(w), n / 2, chunk / 2, scr.partial,
                                                 scr.ticket, h, ldh);
  }
  MG_LAUNCH_CHECK();
}
}  // namespace

void normalise_digits(const double2 *w, double2 *v, DigitBasis b, int slot, const double *inv, int64_t n, int nrhs,
                      cudaStream_t s) {
  const int nt = div_up(n, kTile);
  normalise_kernel<<<dim3(nt, nrhs), RB, 0, s>>>(w, v, b.v + (int64_t)slot * n * nrhs,
                                                 b.e + (int64_t)slot * nt * nrhs, inv, n);
  MG_LAUNCH_CHECK();
}
int64_t digit_tiles(int64_t n) { return (n + kTile - 1) / kTile; }
// a double per tile (FP32 tiles are of 2 kTileF = kTile elements, too), or the
// partials of a dot
static_assert(2 * kTileF == kTile, "tiles");
int64_t norm_scratch(int64_t n) { return std::max<int64_t>(reduce_blocks(n), (digit_tiles(n) + 1) / 2); }

void multi_dot_digits(DigitBasis V, int k, const double2 *w, int64_t n, int nrhs, double2 *h, int ldh, RedScratch scr,
                      cudaStream_t s) {
  if ((int64_t)k * nrhs > kTickets) throw Error(1, "reduction: too many outputs for the ticket array");
  const int64_t chunk = reduce_chunk(n), vs = n * nrhs;
  const int JG = k == 1 ? 1 : k <= 4 ? 4 : 8;
  const dim3 grid(blocks_of(n), nrhs, (k + JG - 1) / JG);
  constexpr int sm = kRing * kTile * (int)sizeof(int4);
  auto go = [&](auto kernel) {
    smem_optin((const void *)kernel, sm);
    kernel<<<grid, RB, sm, s>>>(V.v, V.e, vs, k, w, n, chunk, scr.partial, scr.ticket, h, ldh);
  };
  if (JG == 1) go(dot_digits_kernel<1>);
  else if (JG == 4) go(dot_digits_kernel<4>);
  else go(dot_digits_kernel<8>);
  MG_LAUNCH_CHECK();
}

void multi_axpy_digits(DigitBasis V, int k, double2 *w, int64_t n, int nrhs, const double2 *h, int ldh, double sign,
                       cudaStream_t s, double2 *nrm, RedScratch scr) {
  if (k <= 0) return;
  if (k > 128) throw Error(1, "multi_axpy: k > 128");
  constexpr int sm = kRing * kTile * (int)sizeof(int4);
  auto go = [&](auto kernel) {
    smem_optin((const void *)kernel, sm);
    kernel<<<dim3(div_up(n, kTile), nrhs), RB, sm, s>>>(V.v, V.e, n * nrhs, k, w, n, h, ldh, sign,
                                                       reinterpret_cast<double *>(scr.partial), scr.ticket, nrm);
  };
  if (nrm) go(multi_axpy_digits_kernel<true>);
  else go(multi_axpy_digits_kernel<false>);
  MG_LAUNCH_CHECK();
}

template <typename T>
void dot(const C<T> *x, const C<T> *y, int64_t n, int nrhs, double2 *out, RedScratch scr,
         cudaStream_t s) {
  if (nrhs > kTickets) throw Error(1, "reduction: too many outputs for the ticket array");
  launch_dot<T, 1>(x, 0, 1, y, n, nrhs, out, 1, scr, s);
}

template <typename T>
void dot_qr(const C<T> *q, const C<T> *r, int64_t n, int nrhs, double2 *out_qr, double2 *out_qq,
            RedScratch scr, cudaStream_t s) {
  if (nrhs > kTickets) throw Error(1, "reduction: too many outputs for the ticket array");
  const dim3 grid(blocks_of(n), nrhs);
  const int64_t chunk = reduce_chunk(n);
  if constexpr (sizeof(T) == 8) {
    dot_qr_f64_kernel<<<grid, RB, 0, s>>>(q, r, n, chunk, scr.partial, scr.ticket, out_qr, out_qq);
  } else if (aligned16(n, q, r)) {
    dot_qr_f32_kernel<true><<<grid, RB, 0, s>>>(q, r, n, chunk, scr.partial, scr.ticket, out_qr, out_qq);
  } else {
    dot_qr_f32_kernel<false><<<grid, RB, 0, s>>>(q, r, n, chunk, scr.partial, scr.ticket, out_qr, out_qq);
  }
  MG_LAUNCH_CHECK();
}

template <typename T>
void multi_dot(const C<T> *V, int64_t vstride, int k, const C<T> *w, int64_t n, int nrhs,
               double2 *h, int ldh, RedScratch scr, cudaStream_t s) {
  if ((int64_t)k * nrhs > kTickets) throw Error(1, "reduction: too many outputs for the ticket array");
  // vectors per block: w is read once for that many
  if (k == 1) launch_dot<T, 1>(V, vstride, k, w, n, nrhs, h, ldh, scr, s);
  else if (k <= 4) launch_dot<T, 4>(V, vstride, k, w, n, nrhs, h, ldh, scr, s);
  else launch_dot<T, 8>(V, vstride, k, w, n, nrhs, h, ldh, scr, s);
}

template <typename T>
void multi_axpy(const C<T> *V, int64_t vstride, int k, C<T> *w, int64_t n, int nrhs,
                const double2 *h, int ldh, double sign, cudaStream_t s, double2 *nrm, RedScratch scr) {
  if (k > 128) throw Error(1, "multi_axpy: k > 128");
  if constexpr (sizeof(T) == 4) {
    if (k > 0 && aligned16(n | vstride, V, w)) {
      constexpr int sm = kRing * kTileF * (int)sizeof(int4);
      auto go = [&](auto kernel) {
        smem_optin((const void *)kernel, sm);
        kernel<<<dim3(div_up(n, 2 * kTileF), nrhs), RB, sm, s>>>(
            reinterpret_cast<const int4 *>(V), vstride / 2, k, reinterpret_cast<float4 *>(w), n / 2, h, ldh, sign,
            reinterpret_cast<double *>(scr.partial), scr.ticket, nrm);
      };
      if (nrm) go(multi_axpy_f32_ring_kernel<true>);
      else go(multi_axpy_f32_ring_kernel<false>);
      MG_LAUNCH_CHECK();
      return;
    }
  }
  if (k > 0) {
    // at most 32 blocks per SM over all right-hand sides
    const dim3 grid((unsigned)std::min<int64_t>(div_up(n, 512), std::max(1, sm_count() * 32 / nrhs)), nrhs);
    if constexpr (sizeof(T) == 8) multi_axpy_f64_kernel<<<grid, 256, 0, s>>>(V, vstride, k, w, n, h, ldh, sign);
    else multi_axpy_f32_kernel<<<grid, 256, 0, s>>>(V, vstride, k, w, n, h, ldh, sign);
    MG_LAUNCH_CHECK();
  }
  if (nrm) dot<T>(w, w, n, nrhs, nrm, scr, s);
}

namespace {
// blocks per right-hand side of an elementwise pass over n / W packs: one
// pack per thread, at most 32 blocks per SM over all right-hand sides
dim3 pack_grid(int64_t packs, int nrhs) {
  return dim3((unsigned)std::min<int64_t>(div_up(packs, 256), std::max(1, sm_count() * 32 / nrhs)), nrhs);
}
template <typename T, typename... P> bool packs16(int64_t n, P... p) { return sizeof(T) == 4 && aligned16(n, p...); }
}  // namespace

template <typename T>
void axpby(double a, const C<T> *x, double b, C<T> *y, int64_t n, int nrhs, cudaStream_t s) {
  const int64_t tot = n * nrhs;
  if (packs16<T>(tot, x, y)) axpby_kernel<T, 2><<<pack_grid(tot / 2, 1), 256, 0, s>>>((T)a, x, (T)b, y, tot);
  else axpby_kernel<T, 1><<<pack_grid(tot, 1), 256, 0, s>>>((T)a, x, (T)b, y, tot);
  MG_LAUNCH_CHECK();
}

template <typename T>
void subtract(const C<T> *a, const C<T> *b, C<T> *d, int64_t n, cudaStream_t s) {
  if (packs16<T>(n, a, b, d)) subtract_kernel<T, 2><<<pack_grid(n / 2, 1), 256, 0, s>>>(a, b, d, n);
  else subtract_kernel<T, 1><<<pack_grid(n, 1), 256, 0, s>>>(a, b, d, n);
  MG_LAUNCH_CHECK();
}

template <typename T>
void scale_rhs(const C<T> *x, C<T> *y, const double *scal, int64_t n, int nrhs, cudaStream_t s) {
  if (packs16<T>(n, x, y)) scale_rhs_kernel<T, 2><<<pack_grid(n / 2, nrhs), 256, 0, s>>>(x, y, scal, n);
  else scale_rhs_kernel<T, 1><<<pack_grid(n, nrhs), 256, 0, s>>>(x, y, scal, n);
  MG_LAUNCH_CHECK();
}

template <typename T>
void mr_update(C<T> *z, C<T> *r, const C<T> *q, const double2 *dqr, const double2 *nq, int64_t n,
               int nrhs, cudaStream_t s, const C<T> *r0) {
  if (r0) {
    if (packs16<T>(n, z, r, q, r0))
      mr_update_kernel<T, 2, MR_FIRST><<<pack_grid(n / 2, nrhs), 256, 0, s>>>(z, r, r0, q, dqr, nq, n, 0.0);
    else mr_update_kernel<T, 1, MR_FIRST><<<pack_grid(n, nrhs), 256, 0, s>>>(z, r, r0, q, dqr, nq, n, 0.0);
  } else if (packs16<T>(n, z, r, q)) {
    mr_update_kernel<T, 2, MR_RES><<<pack_grid(n / 2, nrhs), 256, 0, s>>>(z, r, nullptr, q, dqr, nq, n, 0.0);
  } else {
    mr_update_kernel<T, 1, MR_RES><<<pack_grid(n, nrhs), 256, 0, s>>>(z, r, nullptr, q, dqr, nq, n, 0.0);
  }
  MG_LAUNCH_CHECK();
}

template <typename T>
void mr_dir_update(C<T> *z, C<T> *r, const C<T> *e, const C<T> *q, const double2 *dqr,
                   const double2 *nq, int64_t n, int nrhs, cudaStream_t s) {
  if (packs16<T>(n, z, r, e, q))
    mr_update_kernel<T, 2, MR_DIR><<<pack_grid(n / 2, nrhs), 256, 0, s>>>(z, r, e, q, dqr, nq, n, 1e-280);
  else mr_update_kernel<T, 1, MR_DIR><<<pack_grid(n, nrhs), 256, 0, s>>>(z, r, e, q, dqr, nq, n, 1e-280);
  MG_LAUNCH_CHECK();
}

template <typename To, typename From>
void convert(const C<From> *in, C<To> *out, int64_t n, cudaStream_t s) {
  convert_kernel<To, From><<<grid_for(n), 256, 0, s>>>(in, out, n);
  MG_LAUNCH_CHECK();
}

template <typename To, typename From>
void convert_scale(const C<From> *x, C<To> *y, const double *scal, int64_t n, int nrhs,
                   cudaStream_t s) {
  const int gx = (grid_for(n) + nrhs - 1) / nrhs + 1;
  convert_scale_kernel<To, From><<<dim3(gx, nrhs), 256, 0, s>>>(x, y, scal, n);
  MG_LAUNCH_CHECK();
}

template <typename To, typename From>
void relayout(const C<From> *x, C<To> *y, const double *scal, int64_t V, int nrhs, bool to_soa,
              cudaStream_t s) {
  const dim3 grid(div_up(V, kRelayoutSites), nrhs);
  if (aligned16(0, x, y)) relayout_kernel<To, From, true><<<grid, 256, 0, s>>>(x, y, scal, V, to_soa);
  else relayout_kernel<To, From, false><<<grid, 256, 0, s>>>(x, y, scal, V, to_soa);
  MG_LAUNCH_CHECK();
}

template <typename T, typename Tlo>
void add_lo(const C<Tlo> *x, C<T> *y, int64_t n, cudaStream_t s) {
  add_lo_kernel<T, Tlo><<<grid_for(n), 256, 0, s>>>(x, y, n);
  MG_LAUNCH_CHECK();
}

template <typename T>
void check_finite(const C<T> *x, int64_t n, int *flag, cudaStream_t s) {
  finite_kernel<T><<<grid_for(n), 256, 0, s>>>(x, n, flag);
  MG_LAUNCH_CHECK();
}

void gmres_start(GmresState st, cudaStream_t s) {
  gmres_start_kernel<<<(st.nrhs + 63) / 64, 64, 0, s>>>(st);
  MG_LAUNCH_CHECK();
}
void gmres_arnoldi(GmresState st, int i, cudaStream_t s) {
  gmres_arnoldi_kernel<<<st.nrhs, 32, 0, s>>>(st, i);
  MG_LAUNCH_CHECK();
}
void gmres_solve(GmresState st, cudaStream_t s) {
  gmres_solve_kernel<<<st.nrhs, 32, 0, s>>>(st);
  MG_LAUNCH_CHECK();
}

#define INST(T)                                                                                  \
  template void dot<T>(const C<T> *, const C<T> *, int64_t, int, double2 *, RedScratch,         \
                       cudaStream_t);                                                            \
  template void multi_dot<T>(const C<T> *, int64_t, int, const C<T> *, int64_t, int, double2 *,  \
                             int, RedScratch, cudaStream_t);                                     \
  template void multi_axpy<T>(const C<T> *, int64_t, int, C<T> *, int64_t, int, const double2 *, \
                              int, double, cudaStream_t, double2 *, RedScratch);                                        \
  template void axpby<T>(double, const C<T> *, double, C<T> *, int64_t, int, cudaStream_t);      \
  template void scale_rhs<T>(const C<T> *, C<T> *, const double *, int64_t, int, cudaStream_t);  \
  template void mr_update<T>(C<T> *, C<T> *, const C<T> *, const double2 *, const double2 *,     \
                             int64_t, int, cudaStream_t, const C<T> *);                          \
  template void subtract<T>(const C<T> *, const C<T> *, C<T> *, int64_t, cudaStream_t);           \
  template void check_finite<T>(const C<T> *, int64_t, int *, cudaStream_t);               \
  template void dot_qr<T>(const C<T> *, const C<T> *, int64_t, int, double2 *, double2 *,        \
                          RedScratch, cudaStream_t);                                           \
  template void mr_dir_update<T>(C<T> *, C<T> *, const C<T> *, const C<T> *, const double2 *,    \
                                 const double2 *, int64_t, int, cudaStream_t);
INST(double)
INST(float)
template void convert<float, double>(const C<double> *, C<float> *, int64_t, cudaStream_t);
template void convert<double, float>(const C<float> *, C<double> *, int64_t, cudaStream_t);
template void convert_scale<float, double>(const C<double> *, C<float> *, const double *, int64_t,
                                           int, cudaStream_t);
template void convert_scale<double, double>(const C<double> *, C<double> *, const double *,
                                            int64_t, int, cudaStream_t);
template void convert_scale<double, float>(const C<float> *, C<double> *, const double *, int64_t,
                                           int, cudaStream_t);
template void relayout<float, double>(const C<double> *, C<float> *, const double *, int64_t, int,
                                      bool, cudaStream_t);
template void relayout<double, float>(const C<float> *, C<double> *, const double *, int64_t, int,
                                      bool, cudaStream_t);
template void relayout<float, float>(const C<float> *, C<float> *, const double *, int64_t, int,
                                     bool, cudaStream_t);
template void add_lo<double, float>(const C<float> *, C<double> *, int64_t, cudaStream_t);
template void add_lo<double, double>(const C<double> *, C<double> *, int64_t, cudaStream_t);

}  // namespace mg
