// FP64 coarse stencil on the integer pipe (fixed.cuh).
#include "fixed.cuh"
#include "kernels.h"

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
  if (lane == 0) unit[row] = ok ? (short)u : (short)0x7fff;  // an overflowed row gives NaN
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

// one entry of the operator back as a double pair
__device__ __forceinline__ double2 entry(int4 a, int u) {
  return make_double2(scalbn((double)(((long long)a.x << fx::kDigit) + a.y), u),
                      scalbn((double)(((long long)a.z << fx::kDigit) + a.w), u));
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

// one row for a right-hand side with an Inf or NaN among the neighbours, in
// FP64 from the operator's digits (out of line: rare)
__device__ __noinline__ double2 special_row(const double2 *x, const int4 *A, int u, const Geom &g, int X) {
  const int m = g.dof;
  double2 v = make_double2(0.0, 0.0);
  for (int d = 0; d < 9; ++d) {
    const double2 *xn = x + (int64_t)g.neighbor(X, d) * m;
    for (int j = 0; j < m; ++j) v = cfma(entry(A[((int64_t)d * m + j) * m], u), xn[j], v);
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
template <int RG>
__global__ void __launch_bounds__(288, 2)
    stencil_fx_kernel(const double2 *__restrict__ in, double2 *__restrict__ out, const int4 *__restrict__ AF,
                      const short *__restrict__ unit, Geom g, int nrhs) {
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
          const long long a = fx::to_fixed(v.x, E), b = fx::to_fixed(v.y, E);
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
  if (d >= rg || i >= m) return;
  // warp d adds the partial rows of right-hand side d
  const int r = d, u = unit[(int64_t)X * m + i];
  int E = emax[0][r];
#pragma unroll
  for (int dd = 1; dd < 9; ++dd) E = max(E, emax[dd][r]);
  double2 v;
  if (u == 0x7fff) {
    v = make_double2(nan(""), nan(""));
  } else if (E < fx::kBadExp) {
    long long sr = 0, si = 0;
#pragma unroll
    for (int dd = 0; dd < 9; ++dd) {
      const longlong2 t = part[(dd * RG + r) * 32 + lane];
      const int sh = min(E - emax[dd][r], 63);
      sr += t.x >> sh;
      si += t.y >> sh;
    }
    const int e = 2 * fx::kDigit + u + (E - 1022 - fx::kVecBits);
    v = make_double2(scalbn((double)sr, e), scalbn((double)si, e));
  } else {
    v = special_row(in + r * n, AF + (int64_t)X * 9 * m * m + i, u, g, X);
  }
  out[r * n + (int64_t)X * m + i] = v;
}

template <int RG>
void launch(const double2 *in, double2 *out, const int4 *AF, const short *unit, Geom g, int nrhs, cudaStream_t s) {
  const int m = g.dof, ng = (nrhs + RG - 1) / RG;
  const size_t sm = (size_t)9 * RG * (m + 32) * 16;
  if ((int64_t)g.V * ng > 0x7fffffff) throw Error(1, "coarse stencil: too many right-hand sides for one launch");
  smem_optin((const void *)stencil_fx_kernel<RG>, 200 * 1024);
  stencil_fx_kernel<RG>
      <<<dim3((unsigned)g.V * (unsigned)ng, (m + 31) / 32), 288, sm, s>>>(in, out, AF, unit, g, nrhs);
  MG_LAUNCH_CHECK();
}

}  // namespace

void stencil_digits(const double2 *A, int4 *AF, short *unit, const Geom &g, cudaStream_t s) {
  const int64_t rows = (int64_t)g.V * g.dof;
  stencil_digits_kernel<<<(unsigned)((rows + 7) / 8), 256, 0, s>>>(A, AF, unit, rows, g.dof);
  MG_LAUNCH_CHECK();
}

void stencil_apply_fx(const double2 *in, double2 *out, const int4 *AF, const short *unit, Geom g, int nrhs,
                      cudaStream_t s) {
  // right-hand sides per block: 4 leave room for two blocks per SM; the
  // digits of 4 right-hand sides at 256 dofs fill 166 KB
  if (g.dof > 256) throw Error(1, "coarse stencil: too many dofs per site");
  if (nrhs == 1) launch<1>(in, out, AF, unit, g, nrhs, s);
  else if (nrhs == 2) launch<2>(in, out, AF, unit, g, nrhs, s);
  else launch<4>(in, out, AF, unit, g, nrhs, s);
}

}  // namespace mg
