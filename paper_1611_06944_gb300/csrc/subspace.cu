// Subspace of the two-level preconditioner (Section 4):
//   noise -> a fixed number of CR steps on H x = 0 ("inverse iteration applied
//   to Gaussian noise") -> normalise -> chiral split with Gamma5 = gamma5 R5
//   -> restriction to blocks (Eq. 4.1) -> block orthonormalisation, so that
//   P_S = sum |phi_k^b><phi_k^b| (Eq. 4.3) is a projector (Cholesky QR twice,
//   Gram-Schmidt for ill-conditioned blocks).
// All of it runs in FP64; the basis is then stored in the requested dtype.
#include <algorithm>
#include <vector>

#include "host_io.cuh"
#include "chebyshev.cuh"
#include "coarse.cuh"
#include "fx_device.cuh"

namespace hdcr {

int make_block_geom(const Geom& g, const int block[4], BlockGeom* out) {
  if (!block) {
    set_error("block pointer is NULL");
    return HDCR_ERR_BAD_ARG;
  }
  out->Vc = 1;
  out->bvol = 1;
  for (int mu = 0; mu < 4; ++mu) {
    if (block[mu] < 1 || g.L[mu] % block[mu] != 0) {
      set_error("block extent %d does not divide L[%d] = %d", block[mu], mu, g.L[mu]);
      return HDCR_ERR_BAD_GEOMETRY;
    }
    if (g.L[mu] / block[mu] < 2) {
      set_error("coarse extent L[%d]/b = %d must be at least 2", mu, g.L[mu] / block[mu]);
      return HDCR_ERR_BAD_GEOMETRY;
    }
    out->b[mu] = block[mu];
    out->Lc[mu] = g.L[mu] / block[mu];
    out->Vc *= out->Lc[mu];
    out->bvol *= block[mu];
  }
  out->K5 = (long long)out->bvol * g.Ls;
  return HDCR_OK;
}

int subspace_check(const hdcr_subspace* sub) {
  if (!sub || !sub->vecs || sub->nvec < 2) {
    set_error("invalid subspace handle");
    return HDCR_ERR_BAD_ARG;
  }
  return HDCR_OK;
}

// ------------------------------------------------------------------ kernels
// v *= 1 / sqrt(*n2)
__global__ void scale_rsqrt_kernel(cpx<double>* __restrict__ v, long long n, const double* n2) {
  const double s = 1.0 / sqrt(*n2);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    cpx<double> a = v[i];
    v[i] = cpx<double>(a.re * s, a.im * s);
  }
}

// plus = (x + Gamma5 x)/2, minus = (x - Gamma5 x)/2, Gamma5 = gamma5 R5
__global__ void gamma5_split_kernel(Geom g, const cpx<double>* __restrict__ x, cpx<double>* __restrict__ plus,
                                    cpx<double>* __restrict__ minus) {
  const long long n = g.V5 * 12;
  for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (long long)gridDim.x * blockDim.x) {
    const long long row = e / g.Ls;   // x4*12 + c
    const int s = (int)(e - row * g.Ls);
    const int c = (int)(row % 12);
    const cpx<double> a = x[e];
    cpx<double> b = x[row * g.Ls + (g.Ls - 1 - s)];
    if (c >= 6) b = cpx<double>(-b.re, -b.im);
    plus[e] = cpx<double>(0.5 * (a.re + b.re), 0.5 * (a.im + b.im));
    minus[e] = cpx<double>(0.5 * (a.re - b.re), 0.5 * (a.im - b.im));
  }
}

constexpr int GS_THREADS = 256;

// sum over the block of conj(u) v (both fields in plane layout), broadcast to all threads
__device__ __forceinline__ void block_dot(const Geom& g, const BlockGeom& bg, int a, const cpx<double>* u,
                                          const cpx<double>* v, double* bcast, double out[2]) {
  double acc[2] = {0.0, 0.0};
  for (long long l = threadIdx.x; l < bg.K5; l += GS_THREADS) {
    const unsigned o = fidx(g, 0, block_site(g, bg, a, l));
#pragma unroll 4
    for (int c = 0; c < 12; ++c) {
      const cpx<double> p = u[o + c * g.Ls], q = v[o + c * g.Ls];
      acc[0] += p.re * q.re + p.im * q.im;
      acc[1] += p.re * q.im - p.im * q.re;
    }
  }
  block_reduce<2>(acc);
  if (threadIdx.x == 0) {
    bcast[0] = acc[0];
    bcast[1] = acc[1];
  }
  __syncthreads();
  out[0] = bcast[0];
  out[1] = bcast[1];
  __syncthreads();
}

// Modified Gram-Schmidt, applied twice, inside each block (one CTA per block, the
// blocks of ``list`` or all of them), in the fixed order k = 0..nvec-1.  Rank
// deficiency sets *status.  Used for the blocks the Cholesky QR below leaves.
__global__ void __launch_bounds__(GS_THREADS) block_gs_kernel(Geom g, BlockGeom bg, cpx<double>* vecs,
                                                              int nvec, double rank_tol, int* status,
                                                              const int* list) {
  __shared__ double bcast[2];
  const int a = list ? list[blockIdx.x] : blockIdx.x;
  const long long fs = g.V5 * 12;
  for (int k = 0; k < nvec; ++k) {
    cpx<double>* vk = vecs + (long long)k * fs;
    double n0[2];
    block_dot(g, bg, a, vk, vk, bcast, n0);
    for (int pass = 0; pass < 2; ++pass) {
      for (int j = 0; j < k; ++j) {
        const cpx<double>* vj = vecs + (long long)j * fs;
        double d[2];
        block_dot(g, bg, a, vj, vk, bcast, d);
        for (long long l = threadIdx.x; l < bg.K5; l += GS_THREADS) {
          const unsigned o = fidx(g, 0, block_site(g, bg, a, l));
#pragma unroll 4
          for (int c = 0; c < 12; ++c) {
            const unsigned e = o + c * g.Ls;
            const cpx<double> p = vj[e];
            cpx<double> q = vk[e];
            q.re -= d[0] * p.re - d[1] * p.im;
            q.im -= d[0] * p.im + d[1] * p.re;
            vk[e] = q;
          }
        }
        __syncthreads();
      }
    }
    double n1[2];
    block_dot(g, bg, a, vk, vk, bcast, n1);
    double scale = 0.0;
    if (n1[0] > rank_tol * rank_tol * n0[0] && n1[0] > 0.0) {
      scale = 1.0 / sqrt(n1[0]);
    } else if (threadIdx.x == 0) {
      atomicExch(status, 1 + a);
    }
    for (long long l = threadIdx.x; l < bg.K5; l += GS_THREADS) {
      const unsigned o = fidx(g, 0, block_site(g, bg, a, l));
      for (int c = 0; c < 12; ++c) {
        const unsigned e = o + c * g.Ls;
        vk[e] = cpx<double>(vk[e].re * scale, vk[e].im * scale);
      }
    }
    __syncthreads();
  }
}

// ------------------------------------------------------------------ Cholesky QR
// The same orthonormalisation by two rounds of Cholesky QR per block: the Gram
// matrix G = V^dag V of the block's nvec vectors, G = R^dag R (R upper triangular,
// positive real diagonal), V <- V R^{-1}.  The QR factor with a positive real
// diagonal is unique, so in exact arithmetic this is the Gram-Schmidt result; the
// second round removes what the first left of the rounding (about cond(V)^2 eps).
// It reads each vector twice per round instead of twice per pair of vectors, so
// it runs at the FP64 rate instead of the memory rate.  A block whose pivot
// falls below CQR_TOL of its diagonal entry (condition number above ~1e4) is
// left to the Gram-Schmidt kernel, which also decides rank deficiency.
constexpr int CQR_E = 96;         // elements (site x component) of a block per chunk
constexpr int CQR_MAXV = 64;      // largest nvec handled (else Gram-Schmidt throughout)
constexpr int CQR_TILES = 3;      // 2 x 2 Gram tiles per thread: (nvec/2)(nvec/2+1)/2 <= 3 * 256
constexpr double CQR_TOL = 1e-8;
constexpr int CQR_G = 16;         // elements that share an exponent in the fixed-point Gram kernel's chunk
constexpr int CQR_GROUPS = CQR_E / CQR_G;
constexpr int CQR_UP = 4;         // their numbers have at most 57 bits
constexpr int CQR_EX_MIN = 400, CQR_EX_MAX = 1600;
constexpr int CQR_BE_MIN = 70, CQR_BE_MAX = 2000;  // a sum's leading exponent, so that it stays a normal number
// A group's sum of 32 real products errs by 0.56 of the integers' unit (the dropped L L' and the rounded cross
// products), FP64 multiply-adds by 0.29 2^-53 of each of 32 partial sums.  So the integers are as good where the
// partial sums after 4, 8, 12 and 16 elements, squared and added up over the groups, are 0.47 2^-20 of the
// scales 2^63, squared and added up; Gaussian vectors have 6 times that, and 2.4 times where opposite
// symmetry in the fifth dimension makes a group's sum vanish.
constexpr float CQR_K2 = 0.47f * 0x1p-20f;
constexpr int CQR_SPAN = 60;      // exponents above a thread's first group's that the sums of squares may hold

// offset of element le of block a: elements ordered by the block's 4d sites, then
// component and s, so one 4d site's 12 Ls elements are contiguous in the field
__device__ __forceinline__ unsigned cqr_off(const Geom& g, const BlockGeom& bg, int a, long long le) {
  const int per = 12 * g.Ls;
  const long long r = le / per;
  const int rem = (int)(le - r * per);
  const long long i5 = block_site(g, bg, a, r * g.Ls);  // s = 0 of the block's 4d site r
  return (unsigned)((i5 / g.Ls) * per + rem);
}

__device__ __forceinline__ void cqr_tile(int t, int nt, int* j, int* k) {
  int row = 0;  // tiles (tj, tk), tj <= tk, row by row
  while (t >= nt - row) {
    t -= nt - row;
    ++row;
  }
  *j = 2 * row;
  *k = 2 * (row + t);
}

// part[a][q] = sum over share q of block a of conj(v_j) v_k (upper 2x2 tiles)
__global__ void __launch_bounds__(GS_THREADS) cqr_gram_kernel(Geom g, BlockGeom bg, const cpx<double>* __restrict__ vecs,
                                                              int nvec, int S, const int* __restrict__ skip,
                                                              cpx<double>* __restrict__ part) {
  extern __shared__ cpx<double> xs[];  // [nvec][CQR_E]
  const int a = blockIdx.x, q = blockIdx.y;
  if (skip[a]) return;
  const long long fs = g.V5 * 12;
  const long long ne = bg.K5 * 12;
  const long long e0 = ne * q / S, e1 = ne * (q + 1) / S;
  const int nt = nvec / 2, ntiles = nt * (nt + 1) / 2;
  double acc[CQR_TILES][8];
  int tj[CQR_TILES], tk[CQR_TILES];
#pragma unroll
  for (int i = 0; i < CQR_TILES; ++i) {
    const int t = threadIdx.x + i * GS_THREADS;
    tj[i] = tk[i] = -1;
    if (t < ntiles) cqr_tile(t, nt, &tj[i], &tk[i]);
#pragma unroll
    for (int m = 0; m < 8; ++m) acc[i][m] = 0.0;
  }
  for (long long c0 = e0; c0 < e1; c0 += CQR_E) {
    const int n = (int)(e1 - c0 < CQR_E ? e1 - c0 : CQR_E);
    __syncthreads();
    for (int i = threadIdx.x; i < nvec * CQR_E; i += GS_THREADS) {
      const int k = i / CQR_E, e = i - k * CQR_E;
      xs[i] = e < n ? vecs[(long long)k * fs + cqr_off(g, bg, a, c0 + e)] : cpx<double>(0.0, 0.0);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < CQR_TILES; ++i) {
      if (tj[i] < 0) continue;
      const cpx<double>* x0 = xs + tj[i] * CQR_E;
      const cpx<double>* x1 = x0 + CQR_E;
      const cpx<double>* y0 = xs + tk[i] * CQR_E;
      const cpx<double>* y1 = y0 + CQR_E;
      double* A = acc[i];
      for (int e = 0; e < n; ++e) {
        const cpx<double> u0 = x0[e], u1 = x1[e], w0 = y0[e], w1 = y1[e];
        A[0] = fma(u0.re, w0.re, fma(u0.im, w0.im, A[0]));
        A[1] = fma(u0.re, w0.im, fma(-u0.im, w0.re, A[1]));
        A[2] = fma(u0.re, w1.re, fma(u0.im, w1.im, A[2]));
        A[3] = fma(u0.re, w1.im, fma(-u0.im, w1.re, A[3]));
        A[4] = fma(u1.re, w0.re, fma(u1.im, w0.im, A[4]));
        A[5] = fma(u1.re, w0.im, fma(-u1.im, w0.re, A[5]));
        A[6] = fma(u1.re, w1.re, fma(u1.im, w1.im, A[6]));
        A[7] = fma(u1.re, w1.im, fma(-u1.im, w1.re, A[7]));
      }
    }
  }
  cpx<double>* P = part + ((long long)a * S + q) * nvec * nvec;
#pragma unroll
  for (int i = 0; i < CQR_TILES; ++i) {
    if (tj[i] < 0) continue;
    P[tj[i] * nvec + tk[i]] = cpx<double>(acc[i][0], acc[i][1]);
    P[tj[i] * nvec + tk[i] + 1] = cpx<double>(acc[i][2], acc[i][3]);
    P[(tj[i] + 1) * nvec + tk[i]] = cpx<double>(acc[i][4], acc[i][5]);
    P[(tj[i] + 1) * nvec + tk[i] + 1] = cpx<double>(acc[i][6], acc[i][7]);
  }
}

// The same in fixed point, for one tile a thread at most (nvec <= 44).  As FP64 multiply-adds it keeps
// the FP64 pipe 0.79 busy: 42.4 ms a round at 16^4 x 16 with 24 vectors, 16.7 ms so.  The chunk is encoded on
// its way to shared memory: groups of CQR_G elements of a vector share an exponent,
// x = (2^30 H + L) 2^(ex - 1079), |H| <= 2^27, -2^29 <= L < 2^29, 57 bits below the group's
// largest component.  A group's sum is exact in 64 bits up to the dropped L L' (H H' below
// 2^59, the cross products below 2^62), three wide integer multiply-adds a real product, and groups are
// added in FP64.  A pair of groups outside the format is summed in FP64 from the vectors, and so is
// the whole of a tile with a real for which the sums of squares say that FP64 is more accurate:
// vectors that are large where the others are small, bound to opposite walls for instance.  The groups of a
// chunk are dealt to P sets of threads, whose sums are added in the sets' order.
// Rows are CQR_E + 1 elements apart: the vectors of a warp's tiles then lie in different banks.
__global__ void __launch_bounds__(GS_THREADS, 2) cqr_gram_fx_kernel(Geom g, BlockGeom bg,
                                                                    const cpx<double>* __restrict__ vecs, int nvec,
                                                                    int S, const int* __restrict__ skip,
                                                                    cpx<double>* __restrict__ part) {
  extern __shared__ int4 xe[];  // [nvec][CQR_E + 1], then the groups' exponents [nvec][CQR_GROUPS]
  int* ex = reinterpret_cast<int*>(xe + nvec * (CQR_E + 1));
  const int a = blockIdx.x, q = blockIdx.y;
  if (skip[a]) return;
  const long long fs = g.V5 * 12;
  const long long ne = bg.K5 * 12;
  const long long e0 = ne * q / S, e1 = ne * (q + 1) / S;
  const int nt = nvec / 2, ntiles = nt * (nt + 1) / 2;
  const int P = min(CQR_GROUPS, GS_THREADS / ntiles);
  const int set = threadIdx.x / ntiles;  // P and above: threads without a tile
  double A[8];
  float sure[8];  // sum over the groups of (partial sums / 2^63)^2 - K2, in units of 4^ref
  int ref = 0;    // 0: no group yet
  int tj = -1, tk = -1;
  if (set < P) cqr_tile((int)threadIdx.x - set * ntiles, nt, &tj, &tk);
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    A[m] = 0.0;
    sure[m] = 0.f;
  }
  for (long long c0 = e0; c0 < e1; c0 += CQR_E) {
    const int n = (int)(e1 - c0 < CQR_E ? e1 - c0 : CQR_E);
    __syncthreads();
    // nvec is even and CQR_E a multiple of 16: a half warp holds one group, and whole half
    // warps leave the loop together
    for (int i = threadIdx.x; i < nvec * CQR_E; i += GS_THREADS) {
      const int k = i / CQR_E, e = i - k * CQR_E;
      const cpx<double> x[1] = {e < n ? vecs[(long long)k * fs + cqr_off(g, bg, a, c0 + e)] : cpx<double>(0.0, 0.0)};
      const unsigned half = 0xffffu << (threadIdx.x & 16);
      unsigned top = fx_top(x), any = top & 0x80000000u;
      top &= 0x7fffffffu;
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        top = max(top, __shfl_xor_sync(half, top, o));
        any |= __shfl_xor_sync(half, any, o);
      }
      const int m = fx_mark(top | any, CQR_EX_MIN, CQR_EX_MAX);
      xe[k * (CQR_E + 1) + e] = fx_encode(x[0], m, CQR_UP);
      if (e % CQR_G == 0) ex[k * CQR_GROUPS + e / CQR_G] = m;
    }
    __syncthreads();
    if (tj < 0) continue;
    for (int b = set; b * CQR_G < n; b += P) {
      const int ej[2] = {ex[tj * CQR_GROUPS + b], ex[(tj + 1) * CQR_GROUPS + b]};
      const int ek[2] = {ex[tk * CQR_GROUPS + b], ex[(tk + 1) * CQR_GROUPS + b]};
      const int4* x0 = xe + tj * (CQR_E + 1) + b * CQR_G;
      const int4* y0 = xe + tk * (CQR_E + 1) + b * CQR_G;
      // 4^(be - ref) of each product, infinite above CQR_SPAN (then the tile is not certain), 0 where the
      // integers are not used
      float f2[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int p = ej[m >> 1], r = ek[m & 1];
        const int be = p + r - 1012;  // both scaled by 2^-1049 (H), a leading bit 63
        f2[m] = 0.f;
        if (p == 0 || r == 0 || p == FX_RAW || r == FX_RAW || be < CQR_BE_MIN || be > CQR_BE_MAX) continue;
        if (ref == 0) ref = be;
        const int d = be - ref;
        f2[m] = __int_as_float(d > CQR_SPAN ? 0x7f800000 : (127 + 2 * max(d, -CQR_SPAN)) << 23);
      }
      i64 h[8], l[8];
#pragma unroll
      for (int m = 0; m < 8; ++m) h[m] = 0, l[m] = 1LL << 29;
#pragma unroll 1
      for (int e4 = 0; e4 < CQR_G; e4 += 4) {
#pragma unroll 2
        for (int e = e4; e < e4 + 4; ++e) {
          const int4 u[2] = {x0[e], x0[e + CQR_E + 1]}, w[2] = {y0[e], y0[e + CQR_E + 1]};
#pragma unroll
          for (int m = 0; m < 4; ++m) {
            const int4 p = u[m >> 1], r = w[m & 1];  // conj(p) r
            const int nz = -p.z, nw = -p.w;
            h[2 * m] = mw(p.z, r.z, mw(p.x, r.x, h[2 * m]));
            h[2 * m + 1] = mw(nz, r.x, mw(p.x, r.z, h[2 * m + 1]));
            l[2 * m] = mw(p.w, r.z, mw(p.z, r.w, mw(p.y, r.x, mw(p.x, r.y, l[2 * m]))));
            l[2 * m + 1] = mw(nw, r.x, mw(nz, r.y, mw(p.y, r.z, mw(p.x, r.w, l[2 * m + 1]))));
          }
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float x = (float)(int)(h[i] >> 32) * 0x1p-31f;
          sure[i] = fmaf(f2[i >> 1], x * x, sure[i]);
        }
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int p = ej[m >> 1], r = ek[m & 1];
        if (f2[m] != 0.f) {
          const int be = p + r - 1012;
#pragma unroll
          for (int i = 2 * m; i < 2 * m + 2; ++i) {
            if (h[i] == 0 && l[i] == 1LL << 29) continue;  // no products but zeros
            A[i] += fx_to_double(h[i] + (l[i] >> 30), be);
            sure[i] = fmaf(f2[m], -CQR_K2, sure[i]);
          }
          continue;
        }
        if ((p == 0 && r != FX_RAW) || (r == 0 && p != FX_RAW)) continue;
        const cpx<double>* f = vecs + (long long)(tj + (m >> 1)) * fs;
        const cpx<double>* s = vecs + (long long)(tk + (m & 1)) * fs;
        for (int e = b * CQR_G; e < min(n, (b + 1) * CQR_G); ++e) {
          const unsigned o = cqr_off(g, bg, a, c0 + e);
          const cpx<double> u = f[o], w = s[o];
          A[2 * m] = fma(u.re, w.re, fma(u.im, w.im, A[2 * m]));
          A[2 * m + 1] = fma(u.re, w.im, fma(-u.im, w.re, A[2 * m + 1]));
        }
      }
    }
  }
  // the sets' sums, one of a tile a thread
  double* sums = reinterpret_cast<double*>(xe);
  float* sures = reinterpret_cast<float*>(sums + 8 * GS_THREADS);
  int* refs = reinterpret_cast<int*>(sures + 8 * GS_THREADS);
  __syncthreads();
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    sums[m * GS_THREADS + threadIdx.x] = A[m];
    sures[m * GS_THREADS + threadIdx.x] = sure[m];
  }
  refs[threadIdx.x] = ref;
  __syncthreads();
  if (set > 0) return;
  int top = ref;
  for (int p = 1; p < P; ++p) top = max(top, refs[p * ntiles + threadIdx.x]);
  bool certain = true;
#pragma unroll
  for (int m = 0; m < 8; ++m) {
    float y = 0.f;
    for (int p = 0; p < P; ++p) {
      const int t = p * ntiles + threadIdx.x;
      const float f = __int_as_float(max(127 + refs[t] - top, 0) << 23);
      y += f * (f * sures[m * GS_THREADS + t]);
      if (p > 0) A[m] += sums[m * GS_THREADS + t];
    }
    certain = certain && y >= 0.f;
  }
  if (!certain) {
    const cpx<double>* x0 = vecs + (long long)tj * fs;
    const cpx<double>* y0 = vecs + (long long)tk * fs;
#pragma unroll
    for (int m = 0; m < 8; ++m) A[m] = 0.0;
    for (long long e = e0; e < e1; ++e) {
      const unsigned o = cqr_off(g, bg, a, e);
      const cpx<double> u[2] = {x0[o], x0[fs + o]}, w[2] = {y0[o], y0[fs + o]};
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const cpx<double> p = u[m >> 1], r = w[m & 1];
        A[2 * m] = fma(p.re, r.re, fma(p.im, r.im, A[2 * m]));
        A[2 * m + 1] = fma(p.re, r.im, fma(-p.im, r.re, A[2 * m + 1]));
      }
    }
  }
  cpx<double>* R = part + ((long long)a * S + q) * nvec * nvec;
#pragma unroll
  for (int m = 0; m < 4; ++m) R[(tj + (m >> 1)) * nvec + tk + (m & 1)] = cpx<double>(A[2 * m], A[2 * m + 1]);
}

// G = sum_q part[a][q] (fixed order), G = R^dag R, rinv[a] = R^{-1}; one warp per
// block.  A pivot below CQR_TOL of its diagonal sets skip[a] (the block goes to
// Gram-Schmidt).
__global__ void __launch_bounds__(32) cqr_chol_kernel(int nvec, int S, const cpx<double>* __restrict__ part,
                                                      cpx<double>* __restrict__ rinv, int* __restrict__ skip) {
  extern __shared__ cpx<double> G[];  // [nvec][nvec]: G, then R in the upper triangle; diag G in d0
  double* d0 = reinterpret_cast<double*>(G + nvec * nvec);
  const int a = blockIdx.x, lane = threadIdx.x;
  if (skip[a]) return;
  const cpx<double>* P = part + (long long)a * S * nvec * nvec;
  for (int i = lane; i < nvec * nvec; i += 32) {
    const int j = i / nvec, k = i - j * nvec;
    if (j > k) continue;
    cpx<double> v(0.0, 0.0);
    for (int q = 0; q < S; ++q) {
      const cpx<double> w = P[(long long)q * nvec * nvec + i];
      v.re += w.re;
      v.im += w.im;
    }
    G[i] = v;
    if (j == k) d0[j] = v.re;
  }
  __syncwarp();
  bool ok = true;
  for (int k = 0; k < nvec && ok; ++k) {
    // pivot: G_kk - sum_{i<k} |R_ik|^2
    double dk = G[k * nvec + k].re;
    for (int i = 0; i < k; ++i) dk -= G[i * nvec + k].re * G[i * nvec + k].re + G[i * nvec + k].im * G[i * nvec + k].im;
    ok = dk > CQR_TOL * d0[k] && d0[k] > 0.0;
    if (!ok) break;
    const double rkk = sqrt(dk);
    __syncwarp();
    // row k of R: R_kj = (G_kj - sum_{i<k} conj(R_ik) R_ij) / R_kk, j > k
    for (int j = k + 1 + lane; j < nvec; j += 32) {
      double re = G[k * nvec + j].re, im = G[k * nvec + j].im;
      for (int i = 0; i < k; ++i) {
        const cpx<double> r1 = G[i * nvec + k], r2 = G[i * nvec + j];
        re -= r1.re * r2.re + r1.im * r2.im;
        im -= r1.re * r2.im - r1.im * r2.re;
      }
      G[k * nvec + j] = cpx<double>(re / rkk, im / rkk);
    }
    __syncwarp();
    if (lane == 0) G[k * nvec + k] = cpx<double>(rkk, 0.0);
    __syncwarp();
  }
  if (!ok) {
    if (lane == 0) skip[a] = 1;
    return;
  }
  // R^{-1} column by column (lane j): X_jj = 1/R_jj, X_ij = -(sum_{m=i+1..j} R_im X_mj) / R_ii
  cpx<double>* X = rinv + (long long)a * nvec * nvec;
  for (int j = lane; j < nvec; j += 32) {
    for (int i = j + 1; i < nvec; ++i) X[i * nvec + j] = cpx<double>(0.0, 0.0);
    X[j * nvec + j] = cpx<double>(1.0 / G[j * nvec + j].re, 0.0);
    for (int i = j - 1; i >= 0; --i) {
      double re = 0.0, im = 0.0;
      for (int m = i + 1; m <= j; ++m) {
        const cpx<double> r = G[i * nvec + m], x = X[m * nvec + j];
        re += r.re * x.re - r.im * x.im;
        im += r.re * x.im + r.im * x.re;
      }
      const double inv = -1.0 / G[i * nvec + i].re;
      X[i * nvec + j] = cpx<double>(re * inv, im * inv);
    }
  }
}

// v_k <- sum_{j<=k} v_j rinv_jk for the elements of share q of block a
__global__ void __launch_bounds__(GS_THREADS) cqr_apply_kernel(Geom g, BlockGeom bg, cpx<double>* __restrict__ vecs,
                                                               int nvec, int S, const int* __restrict__ skip,
                                                               const cpx<double>* __restrict__ rinv) {
  extern __shared__ cpx<double> sh[];  // rinv [nvec][nvec], then xs [nvec][CQR_E]
  const int a = blockIdx.x, q = blockIdx.y;
  if (skip[a]) return;
  cpx<double>* Ri = sh;
  cpx<double>* xs = sh + nvec * nvec;
  const cpx<double>* X = rinv + (long long)a * nvec * nvec;
  for (int i = threadIdx.x; i < nvec * nvec; i += GS_THREADS) Ri[i] = X[i];
  const long long fs = g.V5 * 12;
  const long long ne = bg.K5 * 12;
  const long long e0 = ne * q / S, e1 = ne * (q + 1) / S;
  for (long long c0 = e0; c0 < e1; c0 += CQR_E) {
    const int n = (int)(e1 - c0 < CQR_E ? e1 - c0 : CQR_E);
    __syncthreads();
    for (int i = threadIdx.x; i < nvec * CQR_E; i += GS_THREADS) {
      const int k = i / CQR_E, e = i - k * CQR_E;
      if (e < n) xs[i] = vecs[(long long)k * fs + cqr_off(g, bg, a, c0 + e)];
    }
    __syncthreads();
    for (int i = threadIdx.x; i < nvec * CQR_E; i += GS_THREADS) {
      const int k = i / CQR_E, e = i - k * CQR_E;
      if (e >= n) continue;
      double re = 0.0, im = 0.0;
      for (int j = 0; j <= k; ++j) {
        const cpx<double> v = xs[j * CQR_E + e], r = Ri[j * nvec + k];
        re = fma(v.re, r.re, fma(-v.im, r.im, re));
        im = fma(v.re, r.im, fma(v.im, r.re, im));
      }
      vecs[(long long)k * fs + cqr_off(g, bg, a, c0 + e)] = cpx<double>(re, im);
    }
  }
}

// Two rounds of Cholesky QR over every block that allows it; *flagged receives the
// blocks left for Gram-Schmidt (device list, count on the host).
static int cholesky_qr2(const Geom& g, const BlockGeom& bg, cpx<double>* vecs, int nvec, cudaStream_t st,
                        int** list_out, int* nlist) {
  *list_out = nullptr;
  *nlist = 0;
  const int Vc = bg.Vc;
  int dev = 0, sms = 0;
  HDCR_CUDA_TRY(cudaGetDevice(&dev));
  HDCR_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  int S = (4 * sms + Vc - 1) / Vc;  // shares of a block, so that the grid covers the SMs about four times
  if (S < 1) S = 1;
  if (S > 8) S = 8;
  const size_t nn = (size_t)nvec * nvec;
  cpx<double>* part = nullptr;
  cpx<double>* rinv = nullptr;
  int* skip = nullptr;
  cudaError_t e = cudaMallocAsync(&part, sizeof(cpx<double>) * nn * Vc * S, st);
  if (e == cudaSuccess) e = cudaMallocAsync(&rinv, sizeof(cpx<double>) * nn * Vc, st);
  // skip flags [0, Vc), then the list of flagged blocks handed to the caller
  if (e == cudaSuccess) e = cudaMallocAsync(&skip, sizeof(int) * (2 * (size_t)Vc + 1), st);
  if (e == cudaSuccess) e = cudaMemsetAsync(skip, 0, sizeof(int) * (2 * (size_t)Vc + 1), st);
  // with more than one tile a thread the sums of squares do not fit in its registers
  const bool fixed = (nvec / 2) * (nvec / 2 + 1) / 2 <= GS_THREADS;
  auto gram = fixed ? cqr_gram_fx_kernel : cqr_gram_kernel;
  const size_t smem_gram =
      fixed ? std::max((sizeof(int4) * (CQR_E + 1) + sizeof(int) * CQR_GROUPS) * (size_t)nvec,
                       (8 * (sizeof(double) + sizeof(float)) + sizeof(int)) * (size_t)GS_THREADS)
            : sizeof(cpx<double>) * (size_t)nvec * CQR_E;
  const size_t smem_chol = sizeof(cpx<double>) * nn + sizeof(double) * nvec;
  const size_t smem_apply = sizeof(cpx<double>) * (nn + (size_t)nvec * CQR_E);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(gram, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_gram);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(cqr_chol_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_chol);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(cqr_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_apply);
  for (int round = 0; round < 2 && e == cudaSuccess; ++round) {
    gram<<<dim3(Vc, S), GS_THREADS, smem_gram, st>>>(g, bg, vecs, nvec, S, skip, part);
    cqr_chol_kernel<<<Vc, 32, smem_chol, st>>>(nvec, S, part, rinv, skip);
    cqr_apply_kernel<<<dim3(Vc, S), GS_THREADS, smem_apply, st>>>(g, bg, vecs, nvec, S, skip, rinv);
    count_launches(3);
    e = cudaGetLastError();
  }
  std::vector<int> hs(Vc);
  if (e == cudaSuccess) e = cudaMemcpyAsync(hs.data(), skip, sizeof(int) * Vc, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e == cudaSuccess) {
    std::vector<int> list;
    for (int a = 0; a < Vc; ++a)
      if (hs[a]) list.push_back(a);
    if (!list.empty()) {
      int* dl = skip + Vc;  // the second half of the flag buffer holds the list
      e = cudaMemcpyAsync(dl, list.data(), sizeof(int) * list.size(), cudaMemcpyHostToDevice, st);
      if (e == cudaSuccess) e = cudaStreamSynchronize(st);
      *list_out = dl;
      *nlist = (int)list.size();
    }
  }
  cudaFreeAsync(part, st);
  cudaFreeAsync(rinv, st);
  if (e != cudaSuccess || *nlist == 0) cudaFreeAsync(skip, st);
  if (e != cudaSuccess) {
    *list_out = nullptr;
    return cuda_status(e, "block Cholesky QR");
  }
  return HDCR_OK;
}

// ---------------------------------------------------------------- host side
// Takes ownership of ``vecs`` (freed on every failure, kept or converted on success).
static int orthonormalise_and_store(const Geom& g, const BlockGeom& bg, cpx<double>* vecs, int nvec,
                                    int store_dtype, cudaStream_t st, hdcr_subspace** out) {
  int* dstatus = nullptr;
  cudaError_t e0 = dev_malloc(&dstatus, sizeof(int));
  if (e0 != cudaSuccess) {
    cudaFree(vecs);
    return cuda_status(e0, "subspace status flag");
  }
  cudaMemsetAsync(dstatus, 0, sizeof(int), st);
  // Cholesky QR where the blocks allow it, Gram-Schmidt for the rest (all of them
  // when nvec is above the Cholesky kernels' limit)
  int* list = nullptr;
  int nlist = bg.Vc;
  if (nvec <= CQR_MAXV) {
    const int s = cholesky_qr2(g, bg, vecs, nvec, st, &list, &nlist);
    if (s != HDCR_OK) {
      cudaFree(dstatus);
      cudaFree(vecs);
      return s;
    }
  }
  if (nlist > 0) {
    block_gs_kernel<<<nlist, GS_THREADS, 0, st>>>(g, bg, vecs, nvec, 1e-12, dstatus, list);
    count_launch();
  }
  cudaError_t e = cudaGetLastError();
  if (list) cudaFreeAsync(list - bg.Vc, st);  // the list sits behind the skip flags of cholesky_qr2
  int hstatus = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hstatus, dstatus, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(dstatus);
  if (e != cudaSuccess) {
    cudaFree(vecs);
    return cuda_status(e, "block orthonormalisation");
  }
  if (hstatus != 0) {
    cudaFree(vecs);
    set_error("subspace vectors are linearly dependent in block %d", hstatus - 1);
    return HDCR_ERR_RANK_DEFICIENT;
  }
  hdcr_subspace* sub = new hdcr_subspace();
  sub->g = g;
  sub->bg = bg;
  sub->nvec = nvec;
  sub->dtype = store_dtype;
  cudaGetDevice(&sub->device);
  const long long n = (long long)nvec * g.V5 * 12;
  if (store_dtype == HDCR_C128) {
    sub->vecs = vecs;  // keep the FP64 buffer
    const int s = subspace_encode(sub, st);
    if (s != HDCR_OK) {
      hdcr_subspace_destroy(sub);
      return s;
    }
  } else {
    void* p = nullptr;
    e = dev_malloc(&p, n * sizeof(cpx<float>));
    if (e != cudaSuccess) {
      cudaFree(vecs);
      delete sub;
      return cuda_status(e, "subspace storage");
    }
    int s = launch_convert(vecs, HDCR_C128, p, HDCR_C64, n, st);
    if (s == HDCR_OK) {
      e = cudaStreamSynchronize(st);
      if (e != cudaSuccess) s = cuda_status(e, "subspace convert");
    }
    cudaFree(vecs);
    if (s != HDCR_OK) {
      cudaFree(p);
      delete sub;
      return s;
    }
    sub->vecs = p;
  }
  *out = sub;
  return HDCR_OK;
}

// step 1 for one vector: filter x (precision R, in place) towards the low modes of H
template <typename R>
static int filter_one(const FineOp<R>& H, cpx<R>* x, const cpx<R>* zero, const hdcr_subspace_params* sp,
                      CRWork<R>& w, ChebWork<R>& cw, cudaStream_t st) {
  if (sp->kind == HDCR_SUBSPACE_CR_SMOOTH) {
    CRConfig cfg;
    cfg.fixed_iters = sp->order;
    return cr_run<R>(H, zero, x, w, cfg, nullptr, st);
  }
  return cheb_filter<R>(H, x, sp->order, sp->lam_cut, sp->lam_max, cw, w.rb.rs, st);
}

// step 1 with the Chebyshev filter: all nvec/2 noise fields through one run of
// the recurrence (multi-field stencil launches), then each is normalised and split
template <typename R>
static int filter_all_cheb(const Geom& g, const hdcr_dwf_params* p, const void* U, const void* noise,
                           const hdcr_subspace_params* sp, cpx<double>* vecs, cudaStream_t st) {
  const long long fs = g.V5 * 12;
  const int half = sp->nvec / 2;
  const bool f64 = sizeof(R) == 8;
  // x (half fields), recurrence work (4 * half fields), x64 scratch, U in R
  const size_t bytes = sizeof(cpx<R>) * fs * half * 5 + sizeof(cpx<double>) * fs +
                       (f64 ? 0 : sizeof(cpx<R>) * g.V4 * 36) + 1024;
  void* mem = nullptr;
  HDCR_CUDA_TRY(dev_malloc(&mem, bytes));
  cpx<R>* x = (cpx<R>*)mem;
  cpx<R>* work = x + fs * half;
  cpx<double>* x64 = (cpx<double>*)(work + 4 * fs * half);
  const cpx<R>* Ur = (const cpx<R>*)U;
  if (!f64) {
    cpx<R>* u32 = (cpx<R>*)(x64 + fs);
    launch_convert(U, HDCR_C128, u32, HDCR_C64, (long long)g.V4 * 36, st);
    Ur = u32;
  }
  RedBuffers rb{{nullptr, nullptr}, nullptr, 0, nullptr};
  int s = red_buffers_alloc(&rb, 2);
  FineOp<R> H{g, p->M5, p->mf, Ur};
  FxCtx fx;
  if (f64) fx_ctx_alloc(&fx, g, half, 2);
  H.fx = &fx;
  if (s == HDCR_OK) s = fx_ctx_links(fx, g, (const cpx<double>*)U, st);
  if (s == HDCR_OK) s = launch_convert(noise, HDCR_C128, x, f64 ? HDCR_C128 : HDCR_C64, fs * half, st);
  if (s == HDCR_OK) s = cheb_filter_multi<R>(H, x, half, sp->order, sp->lam_cut, sp->lam_max, work, rb.scal, rb.rs, st);
  for (int i = 0; i < half && s == HDCR_OK; ++i) {
    s = launch_convert(x + (long long)i * fs, f64 ? HDCR_C128 : HDCR_C64, x64, HDCR_C128, fs, st);
    if (s == HDCR_OK) s = launch_norm2<double>(x64, fs, rb.rs, rb.scal + 1, st);
    if (s != HDCR_OK) break;
    scale_rsqrt_kernel<<<num_blocks(fs, 256, 4096), 256, 0, st>>>(x64, fs, rb.scal + 1); count_launch();
    gamma5_split_kernel<<<num_blocks(fs, 256, 4096), 256, 0, st>>>(g, x64, vecs + (long long)i * fs,
                                                                   vecs + (long long)(i + half) * fs); count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) s = cuda_status(e, "subspace filtering");
  }
  cudaStreamSynchronize(st);
  red_buffers_free(&rb);
  fx_ctx_free(&fx);
  cudaFree(mem);
  return s;
}

template <typename R>
static int filter_all(const Geom& g, const hdcr_dwf_params* p, const void* U, const void* noise,
                      const hdcr_subspace_params* sp, cpx<double>* vecs, cudaStream_t st) {
  const long long fs = g.V5 * 12;
  const int half = sp->nvec / 2;
  const bool f64 = sizeof(R) == 8;
  // x (R), zero (R), x64 scratch, U in R
  const size_t bytes = sizeof(cpx<R>) * fs * 2 + sizeof(cpx<double>) * fs + (f64 ? 0 : sizeof(cpx<R>) * g.V4 * 36) + 512;
  void* mem = nullptr;
  HDCR_CUDA_TRY(dev_malloc(&mem, bytes));
  cpx<R>* x = (cpx<R>*)mem;
  cpx<R>* zero = x + fs;
  cpx<double>* x64 = (cpx<double>*)(zero + fs);
  const cpx<R>* Ur = (const cpx<R>*)U;
  if (!f64) {
    cpx<R>* u32 = (cpx<R>*)(x64 + fs);
    launch_convert(U, HDCR_C128, u32, HDCR_C64, (long long)g.V4 * 36, st);
    Ur = u32;
  }
  CRWork<R> w;
  ChebWork<R> cw;
  int s = crwork_alloc<R>(&w, fs);
  if (s == HDCR_OK && sp->kind == HDCR_SUBSPACE_CHEBYSHEV) s = cheb_work_alloc<R>(&cw, fs);
  FineOp<R> H{g, p->M5, p->mf, Ur};
  cudaMemsetAsync(zero, 0, sizeof(cpx<R>) * fs, st);
  for (int i = 0; i < half && s == HDCR_OK; ++i) {
    const cpx<double>* src = (const cpx<double>*)noise + (long long)i * fs;
    s = launch_convert(src, HDCR_C128, x, f64 ? HDCR_C128 : HDCR_C64, fs, st);
    if (s == HDCR_OK) s = filter_one<R>(H, x, zero, sp, w, cw, st);
    if (s == HDCR_OK) s = launch_convert(x, f64 ? HDCR_C128 : HDCR_C64, x64, HDCR_C128, fs, st);
    if (s == HDCR_OK) s = launch_norm2<double>(x64, fs, w.rb.rs, &w.dev()->tr, st);
    if (s != HDCR_OK) break;
    scale_rsqrt_kernel<<<num_blocks(fs, 256, 4096), 256, 0, st>>>(x64, fs, &w.dev()->tr); count_launch();
    gamma5_split_kernel<<<num_blocks(fs, 256, 4096), 256, 0, st>>>(g, x64, vecs + (long long)i * fs,
                                                                   vecs + (long long)(i + half) * fs); count_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) s = cuda_status(e, "subspace filtering");
  }
  cudaStreamSynchronize(st);
  crwork_free<R>(&w);
  cheb_work_free<R>(&cw);
  cudaFree(mem);
  return s;
}

static int build_subspace_impl(const Geom& g, const BlockGeom& bg, const hdcr_dwf_params* p, const void* U,
                               const void* noise, const hdcr_subspace_params* sp, cudaStream_t st,
                               hdcr_subspace** out) {
  const long long fs = g.V5 * 12;
  cpx<double>* vecs = nullptr;
  HDCR_CUDA_TRY(dev_malloc(&vecs, sizeof(cpx<double>) * fs * sp->nvec));
  int s;
  if (sp->kind == HDCR_SUBSPACE_CHEBYSHEV)
    s = sp->filter_dtype == HDCR_C128 ? filter_all_cheb<double>(g, p, U, noise, sp, vecs, st)
                                      : filter_all_cheb<float>(g, p, U, noise, sp, vecs, st);
  else
    s = sp->filter_dtype == HDCR_C128 ? filter_all<double>(g, p, U, noise, sp, vecs, st)
                                      : filter_all<float>(g, p, U, noise, sp, vecs, st);
  if (s != HDCR_OK) {
    cudaFree(vecs);
    return s;
  }
  return orthonormalise_and_store(g, bg, vecs, sp->nvec, sp->store_dtype, st, out);
}

}  // namespace hdcr

using namespace hdcr;

static int subspace_args(const hdcr_geom* gp, const int block[4], int nvec, int store_dtype, Geom* g,
                         BlockGeom* bg) {
  HDCR_TRY(make_geom(gp, g));
  HDCR_TRY(make_block_geom(*g, block, bg));
  if (nvec < 2 || nvec % 2 != 0 || nvec > 256) {
    set_error("nvec = %d must be even, 2..256", nvec);
    return HDCR_ERR_BAD_ARG;
  }
  if (store_dtype != HDCR_C128 && store_dtype != HDCR_C64) {
    set_error("unknown storage dtype %d", store_dtype);
    return HDCR_ERR_BAD_ARG;
  }
  return HDCR_OK;
}

extern "C" int hdcr_build_subspace(const hdcr_geom* gp, const hdcr_dwf_params* p, const void* U,
                                   const void* noise, const hdcr_subspace_params* sp, void* stream,
                                   hdcr_subspace** out) {
  if (!sp) {
    set_error("hdcr_build_subspace: null parameters");
    return HDCR_ERR_BAD_ARG;
  }
  Geom g;
  BlockGeom bg;
  HDCR_TRY(subspace_args(gp, sp->block, sp->nvec, sp->store_dtype, &g, &bg));
  if (!p || !U || !noise || !out || sp->order < 0 ||
      (sp->kind != HDCR_SUBSPACE_CR_SMOOTH && sp->kind != HDCR_SUBSPACE_CHEBYSHEV) ||
      (sp->filter_dtype != HDCR_C128 && sp->filter_dtype != HDCR_C64)) {
    set_error("hdcr_build_subspace: null pointer or bad parameters");
    return HDCR_ERR_BAD_ARG;
  }
  if (sp->kind == HDCR_SUBSPACE_CHEBYSHEV && (sp->order < 1 || !(sp->lam_cut > 0.0) || !(sp->lam_max > sp->lam_cut))) {
    set_error("hdcr_build_subspace: Chebyshev filter needs order >= 1 and 0 < lam_cut < lam_max");
    return HDCR_ERR_BAD_ARG;
  }
  *out = nullptr;
  cudaStream_t st = as_stream(stream);
  Staged su, sn;
  HDCR_TRY(su.in(U, (size_t)g.V4 * 36 * 16, st));
  HDCR_TRY(sn.in(noise, (size_t)(sp->nvec / 2) * g.V5 * 12 * 16, st));
  return build_subspace_impl(g, bg, p, su.ptr(), sn.ptr(), sp, st, out);
}

extern "C" int hdcr_subspace_from_vectors(const hdcr_geom* gp, const int block[4], int nvec,
                                          const void* vectors, int store_dtype, void* stream,
                                          hdcr_subspace** out) {
  Geom g;
  BlockGeom bg;
  HDCR_TRY(subspace_args(gp, block, nvec, store_dtype, &g, &bg));
  if (!vectors || !out) {
    set_error("hdcr_subspace_from_vectors: null pointer");
    return HDCR_ERR_BAD_ARG;
  }
  *out = nullptr;
  cudaStream_t st = as_stream(stream);
  const long long n = (long long)nvec * g.V5 * 12;
  cpx<double>* vecs = nullptr;
  HDCR_CUDA_TRY(dev_malloc(&vecs, sizeof(cpx<double>) * n));
  cudaMemcpyAsync(vecs, vectors, sizeof(cpx<double>) * n, cudaMemcpyDeviceToDevice, st);
  return orthonormalise_and_store(g, bg, vecs, nvec, store_dtype, st, out);
}

extern "C" int hdcr_subspace_info(const hdcr_subspace* sub, int* nvec, int coarse_L[4], int* dtype) {
  HDCR_TRY(subspace_check(sub));
  if (nvec) *nvec = sub->nvec;
  if (coarse_L)
    for (int mu = 0; mu < 4; ++mu) coarse_L[mu] = sub->bg.Lc[mu];
  if (dtype) *dtype = sub->dtype;
  return HDCR_OK;
}

extern "C" int hdcr_subspace_get_vectors(const hdcr_subspace* sub, void* out, void* stream) {
  HDCR_TRY(subspace_check(sub));
  if (!out) {
    set_error("hdcr_subspace_get_vectors: null output");
    return HDCR_ERR_BAD_ARG;
  }
  const long long n = (long long)sub->nvec * sub->g.V5 * 12;
  return launch_convert(sub->vecs, sub->dtype, out, HDCR_C128, n, as_stream(stream));
}

extern "C" void hdcr_subspace_destroy(hdcr_subspace* sub) {
  if (!sub) return;
  if (sub->vecs) cudaFree(sub->vecs);
  subspace_fx_free(sub);
  if (sub->build_ws) cudaFree(sub->build_ws);
  delete sub;
}
