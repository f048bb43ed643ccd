// FP64 operators on the integer pipe (fixed.cuh): the coarse stencil and the
// Wilson operator.
#include "fixed.cuh"
#include "kernels.h"

#include <algorithm>

namespace mg {

namespace {

// ---- the operator in digits: AF[X][d][j][i] = (re1, re0, im1, im0) of
// A[X][d][i][j] in units of 2^unit[X m + i] (one unit per row over its nine
// blocks).  One warp per row.
__global__ void stencil_digits_kernel(const double2 *__restrict__ A, int4 *__restrict__ AF,
                                      short *__restrict__ unit, int64_t rows, int m) {
  const int lane = threadIdx.x & 31;
  const int64_t row = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5);
  if (row >= rows) return;
  const int64_t X = row / m;
  const int i = (int)(row - X * m);
  const double2 *AX = A + X * 9 * m * m;
  double sum = 0.0, mx = 0.0;
  for (int e = lane; e < 9 * m; e += 32) {
    const int d = e / m, j = e - d * m;
    const double2 a = AX[((int64_t)d * m + i) * m + j];
    sum += fabs(a.x) + fabs(a.y);
    mx = fmax(mx, fmax(fabs(a.x), fabs(a.y)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  int em = 0, es = 0, u = 0;
  const bool ok = isfinite(sum);
  if (ok && mx > 0.0) {
    frexp(mx, &em);           // mx < 2^em
    frexp(sum * 1.0001, &es);  // the rounding of the sum above stays below
    u = fx::row_unit(em, es);
  }
  if (lane == 0) unit[row] = ok ? (short)u : (short)0x7fff;  // a row with Inf or NaN: in FP64
  for (int e = lane; e < 9 * m; e += 32) {
    const int d = e / m, j = e - d * m;
    const double2 a = AX[((int64_t)d * m + i) * m + j];
    int4 q = make_int4(0, 0, 0, 0);
    if (ok && mx > 0.0) {
      const long long r = llrint(scalbn(a.x, -u)), s = llrint(scalbn(a.y, -u));
      q = make_int4(fx::digit_hi(r), fx::digit_lo(r), fx::digit_hi(s), fx::digit_lo(s));
    }
    AF[((X * 9 + d) * m + j) * m + i] = q;
  }
}

// complex product of digits: high and middle sums of the real and imaginary
// parts
__device__ __forceinline__ void mac(int4 a, int4 x, long long &hr, long long &hi, long long &mr, long long &mi) {
  const int n1 = -a.z, n0 = -a.w;
  hr = fx::madw(n1, x.z, fx::madw(a.x, x.x, hr));
  hi = fx::madw(a.z, x.x, fx::madw(a.x, x.z, hi));
  mr = fx::madw(n0, x.z, fx::madw(n1, x.w, fx::madw(a.y, x.x, fx::madw(a.x, x.y, mr))));
  mi = fx::madw(a.w, x.x, fx::madw(a.z, x.y, fx::madw(a.y, x.z, fx::madw(a.x, x.w, mi))));
}

// one row in FP64 from the operator itself, A[X][d][i][j] of site X and row i, by
// a whole warp (out of line: rare; a lane by itself took 60 us of load latency)
__device__ __noinline__ double2 special_row(const double2 *x, const double2 *A, const Geom &g, int X) {
  const int m = g.dof;
  double2 v = make_double2(0.0, 0.0);
#pragma unroll 3
  for (int d = 0; d < 9; ++d) {
    const double2 *xn = x + (int64_t)g.neighbor(X, d) * m, *Ad = A + (int64_t)d * m * m;
    for (int j = threadIdx.x & 31; j < m; j += 32) v = cfma(Ad[j], xn[j], v);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    v.x += __shfl_xor_sync(0xffffffffu, v.x, o);
    v.y += __shfl_xor_sync(0xffffffffu, v.y, o);
  }
  return v;
}

// y(X) = sum_d A[X][d] x(nbr(X, d)).  One block per (site, 32-row tile, RG
// right-hand sides), one warp per direction: the warp scales its neighbour's
// vectors by their own largest entry, leaves their digits in shared memory
// for itself, and lane l forms row l of the direction; the nine partial rows
// are brought to the largest of the nine scales and added as integers.  A
// warp needs no other one before that sum.  The right-hand-side groups of a
// site are neighbouring blocks, so that its operator comes from memory once
// and from L2 after.
//
// Bound: the integer pipe (12 multiply-adds per complex product), 68% busy at
// 512 sites of 32 dofs and 8 right-hand sides: 74 us, where the FP64 form of
// this kernel took 340 us, bound by the FP64 pipe (which now converts one
// result per row).  Two columns per step with the next two in flight: four
// with predicates for ragged rows took 88 us.
//
// The digits keep 2^-59 of the row's largest entry (2^-62 of its 1-norm) and
// 2^-58 of a site vector's largest, below what FP64 additions lose where these
// entries meet.  Where they meet only small or no ones, a row's nine partial sums
// are all small: a row with none above 2^-12 of |row|_1 max|x| (blocks and
// vectors of random entries: 2^-8 to 2^-10, 18 numbers), or Inf or NaN, is formed
// in FP64 from the canonical blocks A instead.  2^-11 takes one row in 10^4 of a
// diagonally dominant operator and 7 us of the 74.
constexpr int kSmallRow = 1 << (61 + 57 - 2 * fx::kDigit - 12 - 32);  // in units of 2^32

template <int RG>
__global__ void __launch_bounds__(288, 2)
    stencil_fx_kernel(const double2 *__restrict__ in, double2 *__restrict__ out, const int4 *__restrict__ AF,
                      const short *__restrict__ unit, const double2 *__restrict__ A, Geom g, int nrhs) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int emax[9][RG];
  const int m = g.dof;
  int4 *xs = reinterpret_cast<int4 *>(smem_raw);                     // [9][RG][m]
  longlong2 *part = reinterpret_cast<longlong2 *>(xs + 9 * RG * m);  // [9][RG][32]
  const int ng = (nrhs + RG - 1) / RG;
  const int X = (int)(blockIdx.x / (unsigned)ng), r0 = (int)(blockIdx.x - (unsigned)X * ng) * RG;
  const int rg = nrhs - r0 < RG ? nrhs - r0 : RG;
  const int i0 = blockIdx.y * 32;
  const int lane = threadIdx.x & 31, d = threadIdx.x >> 5;
  const int i = i0 + lane;
  const int64_t n = g.n();
  in += (int64_t)r0 * n;
  out += (int64_t)r0 * n;
  const int4 *Ad = AF + ((int64_t)X * 9 + d) * m * m + (i < m ? i : i0);
  int4 *xq = xs + d * RG * m;
  {
    const double2 *xd = in + (int64_t)g.neighbor(X, d) * m;
#pragma unroll
    for (int r = 0; r < RG; ++r) {
      int E = 1;
      double2 v = make_double2(0.0, 0.0);
      if (r < rg) {
        for (int j = lane; j < m; j += 32) {
          v = __ldg(xd + r * n + j);
          E = max(E, max(fx::exp_field(v.x), fx::exp_field(v.y)));
        }
        __syncwarp();
      }
      E = __reduce_max_sync(0xffffffffu, E);
      if (lane == 0) emax[d][r] = E;
      for (int j = lane; j < m; j += 32) {
        if (m > 32 && r < rg) v = __ldg(xd + r * n + j);
        int4 q = make_int4(0, 0, 0, 0);
        if (E < fx::kBadExp) {
          const long long a = fx::to_nearest(v.x, E), b = fx::to_nearest(v.y, E);
          q = make_int4(fx::digit_hi(a), fx::digit_lo(a), fx::digit_hi(b), fx::digit_lo(b));
        }
        xq[r * m + j] = q;
      }
    }
    __syncwarp();
  }
  long long hr[RG], hi[RG], mr[RG], mi[RG];
#pragma unroll
  for (int r = 0; r < RG; ++r) hr[r] = hi[r] = mr[r] = mi[r] = 0;
  // two columns at a time (m is even), the next two loaded while they are used
  int4 a0 = __ldg(Ad), a1 = __ldg(Ad + m);
  for (int j0 = 0; j0 < m; j0 += 32) {
    const int jn = m - j0 < 32 ? m - j0 : 32;
#pragma unroll 2
    for (int jj = 0; jj < jn; jj += 2) {
      Ad += j0 + jj + 2 < m ? 2 * m : 0;
      const int4 b0 = __ldg(Ad), b1 = __ldg(Ad + m);
#pragma unroll
      for (int r = 0; r < RG; ++r) {
        const int4 x = xq[r * m + j0 + jj], y = xq[r * m + j0 + jj + 1];
        mac(a0, x, hr[r], hi[r], mr[r], mi[r]);
        mac(a1, y, hr[r], hi[r], mr[r], mi[r]);
      }
      a0 = b0;
      a1 = b1;
    }
    // the middle sums of 32 columns stay below 2^63 (64 products of 2^56,
    // and 2^60 from the row's digit sum)
#pragma unroll
    for (int r = 0; r < RG; ++r) {
      hr[r] = fx::fold(hr[r], mr[r]);
      hi[r] = fx::fold(hi[r], mi[r]);
      mr[r] = mi[r] = 0;
    }
  }
#pragma unroll
  for (int r = 0; r < RG; ++r) part[(d * RG + r) * 32 + lane] = make_longlong2(hr[r], hi[r]);
  __syncthreads();
  if (d >= rg) return;
  // warp d adds the partial rows of right-hand side d
  const int r = d, u = unit[(int64_t)X * m + (i < m ? i : i0)];
  int E = emax[0][r];
#pragma unroll
  for (int dd = 1; dd < 9; ++dd) E = max(E, emax[dd][r]);
  double2 v;
  long long sr = 0, si = 0;
  int top = 0;
#pragma unroll
  for (int dd = 0; dd < 9; ++dd) {
    const longlong2 t = part[(dd * RG + r) * 32 + lane];
    const int sh = min(E - emax[dd][r], 63);
    const long long a = t.x >> sh, b = t.y >> sh;
    top |= ((int)(a >> 32) ^ (int)(a >> 63)) | ((int)(b >> 32) ^ (int)(b >> 63));
    sr += a;
    si += b;
  }
  const int e = 2 * fx::kDigit + u + (E - 1022 - fx::kVecBits);
  v = make_double2(scalbn((double)sr, e), scalbn((double)si, e));
  const bool in_fp64 = u == 0x7fff || E == fx::kBadExp || (top < kSmallRow && E > 1);
  for (unsigned rows = __ballot_sync(0xffffffffu, i < m && in_fp64); rows; rows &= rows - 1) {
    const int k = __ffs(rows) - 1;
    const double2 w = special_row(in + r * n, A + ((int64_t)X * 9 * m + i0 + k) * m, g, X);
    if (lane == k) v = w;
  }
  if (i < m) out[r * n + (int64_t)X * m + i] = v;
}

template <int RG>
void launch(const double2 *in, double2 *out, const int4 *AF, const short *unit, const double2 *A, Geom g, int nrhs,
            cudaStream_t s) {
  const int m = g.dof, ng = (nrhs + RG - 1) / RG;
  const size_t sm = (size_t)9 * RG * (m + 32) * 16;
  if ((int64_t)g.V * ng > 0x7fffffff) throw Error(1, "coarse stencil: too many right-hand sides for one launch");
  smem_optin((const void *)stencil_fx_kernel<RG>, 200 * 1024);
  stencil_fx_kernel<RG>
      <<<dim3((unsigned)g.V * (unsigned)ng, (m + 31) / 32), 288, sm, s>>>(in, out, AF, unit, A, g, nrhs);
  MG_LAUNCH_CHECK();
}

// ------------------------------------------------------------------ Wilson D
// Two kernels per group of right-hand sides.  The first brings each site's 12
// components to 61-bit integers in the unit of the site's largest entry, in
// tiles of 32 sites ([tile][component][32]), so that the hops read neighbours
// with coalesced accesses at constant offsets and no conversion.
// The second forms, per site and direction, the projected half-spinor
// (integer additions), the link product (12 multiply-adds per complex product
// on 56- and 57-bit operands), and adds it in the unit of the largest of the
// nine sites; the result is one conversion per component plus the diagonal
// term in FP64.  24^4 x 3 right-hand sides: 62 + 497 us, against 1.57 ms of
// the FP64 kernel (888 instructions of the FP64 pipe per site, at its rate);
// the integer pipe is 53% busy, the rest waits for loads (16 warps per SM).
//
// An entry keeps 55 bits of the largest of its spinor and, in the sum over the
// hops, of the largest of the eight neighbours: as many as FP64 sums keep where
// that entry takes part in the sum.  Where it does not (spinors whose components
// differ much beside links that do not mix them, a site beside a far larger one)
// the row's own hop terms are all small: a site with a row whose four forward
// hops are below 2^-4 of the scale (normal entries: one site in 30 000), or below
// 2^-23 beside entries below 2^-kFarHop of it, is formed in FP64 instead.  Looking
// at all eight hops cost 5% of the kernel, at four of them 3%.
constexpr int kSiteBits = 61;   // stored components
constexpr int kHopShift = 6;    // of which the link products use 55 bits
// A link entry of 1 takes the scale to 2^55 (2^56 where no link holds a 1); in
// units of 2^32
constexpr int kSmallHop = 1 << (55 - 4 - 32);
constexpr int kFarHop = 6;

// first entry of site s in the tiled order with N entries per site
template <int N> __device__ __forceinline__ int64_t tiled(int s) { return (int64_t)(s >> 5) * (N * 32) + (s & 31); }
inline int64_t tiles(int V) { return (V + 31) / 32; }

__global__ void __launch_bounds__(128) spinor_digits_kernel(const double2 *__restrict__ in,
                                                            longlong2 *__restrict__ xs, short2 *__restrict__ ex,
                                                            int V) {
  __shared__ double2 sh[128 * 13];  // 13: a site's rows fall on different banks
  const int r = blockIdx.y, s0 = blockIdx.x * 128;
  const int ns = V - s0 < 128 ? V - s0 : 128;
  const double2 *p = in + ((int64_t)r * V + s0) * 12;
  for (int e = threadIdx.x; e < ns * 12; e += 128) sh[e / 12 * 13 + e % 12] = __ldg(p + e);
  __syncthreads();
  if ((int)threadIdx.x >= ns) return;
  int E = 1, lo = fx::kBadExp;
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const double2 v = sh[threadIdx.x * 13 + k];
    const int e = max(fx::exp_field(v.x), fx::exp_field(v.y));
    E = max(E, e);
    if (fx::nonzero(v.x) || fx::nonzero(v.y)) lo = min(lo, e);
  }
  const int64_t s = s0 + threadIdx.x;
  ex[(int64_t)r * V + s] = make_short2((short)E, (short)lo);
  longlong2 *o = xs + r * ((V + 31) / 32) * (int64_t)384 + tiled<12>((int)s);
#pragma unroll
  for (int k = 0; k < 12; ++k) {
    const double2 v = sh[threadIdx.x * 13 + k];
    o[k * 32] = E < fx::kBadExp ? make_longlong2(fx::to_nearest<kSiteBits>(v.x, E), fx::to_nearest<kSiteBits>(v.y, E))
                                        : make_longlong2(0, 0);
  }
}

// largest and smallest exponent field over the links' largest entries
__global__ void link_range_kernel(const double2 *__restrict__ U, int64_t nlinks, int *__restrict__ range) {
  int hi = 0, lo = 0x7ff;
  for (int64_t L = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; L < nlinks; L += (int64_t)gridDim.x * blockDim.x) {
    int E = 0;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      const double2 u = U[L * 9 + k];
      E = max(E, max(fx::exp_field(u.x), fx::exp_field(u.y)));
    }
    hi = max(hi, E);
    lo = min(lo, E);
  }
  atomicMax(range, hi);
  atomicMin(range + 1, lo);
}

// UF[mu][tile][k][32] = digits of U[site][mu][k] in the unit of exponent field E
__global__ void link_digits_kernel(const double2 *__restrict__ U, int4 *__restrict__ UF, int V, int E) {
  const int64_t total = (int64_t)V * 36;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = i / 36;
    const int q = (int)(i - s * 36), mu = q / 9;
    const double2 u = U[i];
    const long long a = fx::to_nearest(u.x, E), b = fx::to_nearest(u.y, E);
    UF[mu * ((V + 31) / 32) * (int64_t)288 + tiled<9>((int)s) + (q - mu * 9) * 32] = make_int4(fx::digit_hi(a), fx::digit_lo(a), fx::digit_hi(b), fx::digit_lo(b));
  }
}

// sums written out: the compiler reassociates the sums over the hops of plain
// expressions and keeps every term alive for them (246 registers, or spills);
// volatile, so that a branch over the four powers of i stays a branch (as
// selects all four forms are computed)
__device__ __forceinline__ long long ladd(long long a, long long b) {
  long long r;
  asm volatile("add.s64 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ long long lsub(long long a, long long b) {
  long long r;
  asm volatile("sub.s64 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// a + i^PH b, or a + i^PH conj(b)
template <int PH, bool CONJ> __device__ __forceinline__ longlong2 addp(longlong2 a, longlong2 b) {
  if (PH == 0) return make_longlong2(ladd(a.x, b.x), CONJ ? lsub(a.y, b.y) : ladd(a.y, b.y));
  if (PH == 1) return make_longlong2(CONJ ? ladd(a.x, b.y) : lsub(a.x, b.y), ladd(a.y, b.x));
  if (PH == 2) return make_longlong2(lsub(a.x, b.x), CONJ ? ladd(a.y, b.y) : lsub(a.y, b.y));
  return make_longlong2(CONJ ? lsub(a.x, b.y) : ladd(a.x, b.y), lsub(a.y, b.x));
}
template <int PH, bool CONJ> __device__ __forceinline__ void add3(longlong2 (&a)[3], const longlong2 (&b)[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) a[c] = addp<PH, CONJ>(a[c], b[c]);
}
template <bool CONJ> __device__ __forceinline__ void add3(longlong2 (&a)[3], const longlong2 (&b)[3], int ph) {
  switch (ph) {
    case 0: add3<0, CONJ>(a, b); break;
    case 1: add3<1, CONJ>(a, b); break;
    case 2: add3<2, CONJ>(a, b); break;
    default: add3<3, CONJ>(a, b); break;
  }
}

// x >> s for 0 <= s <= 32
__device__ __forceinline__ long long shr(long long x, int s) {
  const unsigned lo = (unsigned)x, hi = (unsigned)(x >> 32);
  return (long long)(((unsigned long long)(unsigned)((int)hi >> min(s, 31)) << 32) | __funnelshift_rc(lo, hi, s));
}

// centred digits of t >> kHopShift
__device__ __forceinline__ int2 hop_digits(long long t) {
  const int lo = (int)__funnelshift_r((unsigned)t, (unsigned)(t >> 32), kHopShift - 4) >> 4;
  return make_int2((int)(ladd(t, 1ll << (kHopShift + fx::kDigit - 1)) >> 32) >> (kHopShift + fx::kDigit - 32), lo);
}

// D at a site with Inf or NaN or very different entries among the neighbours,
// from the spinors and links themselves (out of line: rare)
__device__ __noinline__ void special_site(const double2 *in, const double2 *U, const Geom &g, int s, double diag,
                                          double2 *o) {
  for (int i = 0; i < 12; ++i) o[i] = cscale(in[(int64_t)s * 12 + i], diag);
  for (int d = 1; d < 9; ++d) {
    const int mu = (d - 1) >> 1;
    const bool fwd = d & 1;
    const int sn = g.neighbor(s, d);
    const int stride = mu == 0 ? 1 : mu == 1 ? g.L[0] : mu == 2 ? g.L[0] * g.L[1] : g.L[0] * g.L[1] * g.L[2];
    const bool wrap = mu == 3 && (fwd ? s / stride == g.L[3] - 1 : s / stride == 0);
    const double k = wrap ? 0.5 : -0.5, sg = fwd ? -1.0 : 1.0;
    const double2 *p = in + (int64_t)sn * 12, *u = U + ((int64_t)(fwd ? s : sn) * 4 + mu) * 9;
    for (int c = 0; c < 3; ++c) {
      double2 v[2];
      for (int a = 0; a < 2; ++a) {
        v[a] = make_double2(0.0, 0.0);
        for (int b = 0; b < 3; ++b) {
          const double2 l0 = p[6 + b], l1 = p[9 + b];
          double2 t;
          if (mu == 0) t = cmulmi(a == 0 ? l1 : l0);
          else if (mu == 1) t = a == 0 ? cneg(l1) : l0;
          else if (mu == 2) t = a == 0 ? cmulmi(l0) : cmuli(l1);
          else t = a == 0 ? l0 : l1;
          const double2 h = cadd(p[3 * a + b], cscale(t, sg));
          v[a] = fwd ? cfma(u[3 * c + b], h, v[a]) : cfmac(u[3 * b + c], h, v[a]);
        }
      }
      for (int a = 0; a < 2; ++a) {
        double2 w;
        if (mu == 0) w = cmuli(a == 0 ? v[1] : v[0]);
        else if (mu == 1) w = a == 0 ? v[1] : cneg(v[0]);
        else if (mu == 2) w = a == 0 ? cmuli(v[0]) : cmulmi(v[1]);
        else w = v[a];
        o[3 * a + c] = cadd(o[3 * a + c], cscale(v[a], k));
        o[6 + 3 * a + c] = cadd(o[6 + 3 * a + c], cscale(w, sg * k));
      }
    }
  }
}

// 2^e as a double, e in the normal range
__device__ __forceinline__ double pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

// loads that stay where they are written
__device__ __forceinline__ longlong2 ldv(const longlong2 *p) {
  longlong2 v;
  asm volatile("ld.global.nc.v2.s64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "l"(p));
  return v;
}
__device__ __forceinline__ int4 ldv(const int4 *p) {
  int4 v;
  asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// Row A of one hop from the neighbour whose tiled spinor is x (lower row
// `rows` entries behind the upper one) through link u: h = upper + i^pb lower,
// v = U h or, backward, conj(U^H h) = U^T conj(h), shifted right by sh.
template <bool FWD>
__device__ __forceinline__ void hop_row(const longlong2 *__restrict__ x, int rows, const int4 *__restrict__ u, int pb,
                                        int sh, longlong2 (&v)[3]) {
  int4 h[3], w[9];
  {
    // every load of the hop before its first use
    longlong2 t[3], l[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      t[k] = ldv(x + k * 32);
      l[k] = ldv(x + rows + k * 32);
    }
#pragma unroll
    for (int k = 0; k < 9; ++k) w[k] = ldv(u + k * 32);
    add3<false>(t, l, pb);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int2 re = hop_digits(t[k].x), im = hop_digits(FWD ? t[k].y : lsub(0ll, t[k].y));
      h[k] = make_int4(re.x, re.y, im.x, im.y);
    }
  }
  const int s0 = min(sh, 32);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    // the middle sums start at half a unit of the high ones: rounded by the shift
    long long hr = 0, hi = 0, mr = 1 << (fx::kDigit - 1), mi = 1 << (fx::kDigit - 1);
#pragma unroll
    for (int b = 0; b < 3; ++b) mac(w[FWD ? 3 * k + b : 3 * b + k], h[b], hr, hi, mr, mi);
    v[k] = make_longlong2(shr(ladd(hr, shr(mr, fx::kDigit)), s0), shr(ladd(hi, shr(mi, fx::kDigit)), s0));
  }
  if (__any_sync(__activemask(), sh > 32)) {
    const int s1 = min(max(sh - 32, 0), 32);
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = make_longlong2(shr(v[k].x, s1), shr(v[k].y, s1));
  }
}

// top[k] |= the magnitudes of v[k], in units of 2^32
__device__ __forceinline__ void largest(int (&top)[3], const longlong2 (&v)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int x = (int)(v[k].x >> 32), y = (int)(v[k].y >> 32);
    top[k] |= (x ^ (x >> 31)) | (y ^ (y >> 31));
  }
}

// Row A of the eight hops: up (row A of the upper half) and its parts of the
// lower rows (cross: row 1 - A, from x and y; same: row A, from z and t), in
// units of the common scale E.  Returns the sizes of the terms of up: for the
// forward hops in x and y, bit k: term k is at least kSmallHop in one of them, bit
// 4 + k: not zero (both in units of 2^32); the same from bit 8 for z and t.
//
// Chiral basis of the other Wilson kernels, B = -i sigma_k, B_4 = 1: row A of
// u + sg B_mu l takes one row of l, and row A of a product v enters one row
// of the lower half: the other one for mu = 0, 1, the same for 2, 3, each
// with a power of i.  The loop over mu stays rolled: eight unrolled hops for
// either row are more instructions than the caches hold (5 of 15 cycles per
// issue went to fetching them).
__device__ __forceinline__ unsigned hops(const longlong2 *__restrict__ xs, const int4 *__restrict__ UF,
                                     const short2 *__restrict__ er, const Geom &g, int s, int A, int E,
                                     longlong2 (&up)[3], longlong2 (&cross)[3], longlong2 (&same)[3]) {
  int top[3] = {0, 0, 0};
  unsigned sizes = 0;
  int stride = 1, rest = s;
  const int4 *u = UF;
#pragma unroll 1
  for (int mu = 0; mu < 4; ++mu) {
    const int L = mu < 2 ? (mu == 0 ? g.L[0] : g.L[1]) : (mu == 2 ? g.L[2] : g.L[3]);
    const int next = rest / L, c = rest - next * L;
    const int B = mu < 2 ? 1 - A : A, rows = (6 + 3 * B - 3 * A) * 32;
    const int sf = c + 1 == L ? s - (L - 1) * stride : s + stride;
    const int sb = c == 0 ? s + (L - 1) * stride : s - stride;
    // powers of i: B_mu in row A, times sg = -1 forward; B_mu^H in row B, likewise
    const int pb = mu == 0 ? 3 : mu == 1 ? (A == 0 ? 2 : 0) : mu == 2 ? (A == 0 ? 3 : 1) : 0;
    const int ph = mu == 0 ? 1 : mu == 1 ? (B == 0 ? 0 : 2) : mu == 2 ? (B == 0 ? 1 : 3) : 0;
    longlong2 v[3];
    hop_row<true>(xs + tiled<12>(sf) + 96 * A, rows, u + tiled<9>(s), (pb + 2) & 3, E - er[sf].x, v);
    if (mu == 3 && c + 1 == L) {
#pragma unroll
      for (int k = 0; k < 3; ++k) v[k] = make_longlong2(-v[k].x, -v[k].y);
    }
    largest(top, v);
    add3<0, false>(up, v);
    if (mu < 2) add3<false>(cross, v, (ph + 2) & 3);
    else add3<false>(same, v, (ph + 2) & 3);
    hop_row<false>(xs + tiled<12>(sb) + 96 * A, rows, u + tiled<9>(sb), pb, E - er[sb].x, v);
    if (mu == 3 && c == 0) {
#pragma unroll
      for (int k = 0; k < 3; ++k) v[k] = make_longlong2(-v[k].x, -v[k].y);
    }
    add3<0, true>(up, v);
    if (mu < 2) add3<true>(cross, v, ph);
    else add3<true>(same, v, ph);
    rest = next;
    stride *= L;
    u += ((g.V + 31) / 32) * (int64_t)288;
    if (mu & 1) {
      sizes >>= 8;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        sizes |= (top[k] >= kSmallHop ? 0x100u << k : 0u) | (top[k] ? 0x1000u << k : 0u);
        top[k] = 0;
      }
    }
  }
  return sizes;
}

// whether one of a row's three entries is small in all of these hops, or nearly
// zero in them beside entries that the scale may have lost (far)
__device__ __forceinline__ bool small_row(unsigned sizes, bool far) {
  return ((sizes >> 4) & ~sizes & 7u) || (far && (~(sizes >> 4) & 7u));
}

constexpr int kWilsonSites = 64;  // per block

// Two threads per site, in different warps: thread A forms row A of every
// half-spinor, so it holds one upper row and its part of the two lower rows
// (18 sums, against 24 and 240 registers with one thread per site, 530 us);
// the parts of a lower row meet in shared memory.  Four blocks per SM keep
// the 15 loads of a hop in flight without spills (five: 520 us).
__global__ void __launch_bounds__(2 * kWilsonSites, 4)
    wilson_fx_kernel(const double2 *__restrict__ in, double2 *__restrict__ out, const longlong2 *__restrict__ xs,
                     const short2 *__restrict__ ex, const int4 *__restrict__ UF, const double2 *__restrict__ U, Geom g,
                     double diag, int EU, int nrhs) {
  constexpr int S = kWilsonSites;
  __shared__ double2 sh[S * 13];
  __shared__ longlong2 other[2][3][S];
  __shared__ unsigned sizes[2][S];
  // the right-hand side fastest: the blocks of a site range share its links
  const int sb = (int)(blockIdx.x / (unsigned)nrhs), r = (int)(blockIdx.x - (unsigned)sb * nrhs);
  const int half = (int)threadIdx.x / S, ls = (int)threadIdx.x - half * S;
  const int s0 = sb * S, s = s0 + ls < g.V ? s0 + ls : g.V - 1;
  const int64_t V = g.V;
  const int ns = g.V - s0 < S ? g.V - s0 : S;
  {
    const double2 *pi = in + ((int64_t)r * V + s0) * 12;
    for (int q = threadIdx.x; q < ns * 12; q += 2 * S) sh[q / 12 * 13 + q % 12] = __ldg(pi + q);
  }
  const short2 *er = ex + (int64_t)r * V;
  longlong2 up[3], cross[3], same[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) up[k] = cross[k] = same[k] = make_longlong2(0, 0);
  int E = 1, lo = fx::kBadExp;
#pragma unroll 1
  for (int d = 1; d < 9; ++d) {
    const short2 e = er[g.neighbor(s, d)];
    E = max(E, (int)e.x);
    lo = min(lo, (int)e.y);
  }
  const bool far = E - lo > kFarHop;
  sizes[half][ls] = hops(xs + r * ((g.V + 31) / 32) * (int64_t)384, UF, er, g, s, half, E, up, cross, same);
#pragma unroll
  for (int k = 0; k < 3; ++k) other[half][k][ls] = cross[k];
  __syncthreads();
  double2 *o = sh + ls * 13 + 3 * half;
  // an upper row takes all eight hops of its half, a lower row z and t of its own
  // half and x and y of the other
  const unsigned z0 = sizes[0][ls], z1 = sizes[1][ls];
  const bool graded = E > 1 && (small_row(z0 | z0 >> 8, far) || small_row(z1 | z1 >> 8, far) ||
                                small_row(z0 >> 8 | z1, far) || small_row(z1 >> 8 | z0, far));
  if (E < fx::kBadExp && !graded) {
    // value = diag psi - 1/2 sum 2^(56 + (E - 1022 - 55) + (EU - 1022 - 57))
    const int ea = 2 * fx::kDigit + (E - 1022 - (kSiteBits - kHopShift)) + (EU - 1022 - fx::kVecBits);
    const bool plain = ea > -1000 && ea < 900;
    const double fa = plain ? -0.5 * pow2(ea) : 0.0;
    if (s0 + ls < g.V) {
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        const int k = q % 3;
        const longlong2 t = q < 3 ? up[k] : addp<0, false>(same[k], other[1 - half][k][ls]);
        const double2 p = o[q < 3 ? k : 6 + k];
        double2 v;
        if (plain) v = make_double2(fma(fa, (double)t.x, diag * p.x), fma(fa, (double)t.y, diag * p.y));
        else v = make_double2(diag * p.x - 0.5 * scalbn((double)t.x, ea), diag * p.y - 0.5 * scalbn((double)t.y, ea));
        o[q < 3 ? k : 6 + k] = v;
      }
    }
  } else if (half == 0) {
    special_site(in + (int64_t)r * 12 * V, U, g, s, diag, o);
  }
  __syncthreads();
  double2 *po = out + ((int64_t)r * V + s0) * 12;
  for (int q = threadIdx.x; q < ns * 12; q += 2 * S) po[q] = sh[q / 12 * 13 + q % 12];
}

}  // namespace

void stencil_digits(const double2 *A, int4 *AF, short *unit, const Geom &g, cudaStream_t s) {
  const int64_t rows = (int64_t)g.V * g.dof;
  stencil_digits_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(A, AF, unit, rows, g.dof);
  MG_LAUNCH_CHECK();
}

void stencil_apply_fx(const double2 *in, double2 *out, const int4 *AF, const short *unit, const double2 *A, Geom g,
                      int nrhs, cudaStream_t s) {
  // right-hand sides per block: 4 leave room for two blocks per SM; the
  // digits of 4 right-hand sides at 256 dofs fill 166 KB
  if (g.dof > 256) throw Error(1, "coarse stencil: too many dofs per site");
  if (nrhs == 1) launch<1>(in, out, AF, unit, A, g, nrhs, s);
  else if (nrhs == 2) launch<2>(in, out, AF, unit, A, g, nrhs, s);
  else launch<4>(in, out, AF, unit, A, g, nrhs, s);
}

size_t link_digits_elems(int V) { return (size_t)tiles(V) * 4 * 288; }
int link_digits(const double2 *U, int4 *UF, int *range, int V, cudaStream_t s) {
  const int init[2] = {0, 0x7ff};
  MG_CUDA(cudaMemcpyAsync(range, init, sizeof(init), cudaMemcpyHostToDevice, s));
  link_range_kernel<<<sm_count() * 8, 256, 0, s>>>(U, (int64_t)V * 4, range);
  MG_LAUNCH_CHECK();
  int h[2];
  MG_CUDA(cudaMemcpyAsync(h, range, sizeof(h), cudaMemcpyDeviceToHost, s));
  MG_CUDA(cudaStreamSynchronize(s));
  // one unit for all links: only where none is more than 8 times smaller than
  // the largest (SU(3) links differ by sqrt 3 at most)
  if (h[0] == 0 || h[0] - h[1] > 3) return 0;
  link_digits_kernel<<<sm_count() * 16, 256, 0, s>>>(U, UF, V, h[0]);
  MG_LAUNCH_CHECK();
  return h[0];
}

int wilson_fx_group(int V, int nrhs) {
  // right-hand sides converted together: 4 share a link read from memory; small
  // lattices take more, up to 2^18 sites (8^4 and 64 right-hand sides: 155 us, 195
  // in groups of 16; 16^4 and 16: 642, 585 in one group, for 201 MB of digits)
  const int g = std::max(4, (1 << 18) / V);
  return std::min(g, nrhs);
}
size_t wilson_fx_elems(int V, int group) {
  const size_t g = group;
  return g * tiles(V) * 384 + (g * V * sizeof(short2) + 15) / 16;
}

void wilson_apply_fx(const double2 *in, double2 *out, const int4 *UF, const double2 *U, int EU, double2 *work,
                     int group, Geom g, double m0, int nrhs, cudaStream_t s) {
  const int grp = std::min(group, nrhs);
  longlong2 *xs = reinterpret_cast<longlong2 *>(work);
  short2 *ex = reinterpret_cast<short2 *>(xs + (size_t)grp * tiles(g.V) * 384);
  for (int r0 = 0; r0 < nrhs; r0 += grp) {
    const int k = std::min(grp, nrhs - r0);
    const int64_t off = (int64_t)r0 * g.n();
    if ((int64_t)div_up(g.V, kWilsonSites) * k > 0x7fffffff) throw Error(1, "lattice too large for one launch");
    spinor_digits_kernel<<<dim3(div_up(g.V, 128), k), 128, 0, s>>>(in + off, xs, ex, g.V);
    MG_LAUNCH_CHECK();
    wilson_fx_kernel<<<(unsigned)div_up(g.V, kWilsonSites) * (unsigned)k, 2 * kWilsonSites, 0, s>>>(
        in + off, out + off, xs, ex, UF, U, g, 4.0 + m0, EU, k);
    MG_LAUNCH_CHECK();
  }
}

}  // namespace mg
