// FP64 restriction and prolongation on the integer pipe.
//
// Both read the whole basis once, 4.8 GB at 16^4 x 16 with 24 vectors (0.72 ms at the copy
// rate), but as four FP64 multiply-adds a complex product they took 2.42 and 1.94 ms at this
// chip's 2 FP64 operations per clock and SM.  They read a copy of the basis in fixed point
// instead, made with the subspace: as in dwf_fx.cuh with one exponent per 5d site and vector, but
// with the second limb an integer too,
//
//     x = (2^30 H + L) 2^(ex - 1081),  |H| <= 2^29, -2^29 <= L < 2^29,
//
// 60 bits below the site's largest component.  A real product is three wide integer multiply-adds
// (the dropped L L' is below 2^-60 of the scale), and a site's 12 components are summed exactly, so
// the sums are at least as accurate as in FP64 (encoding the FP64 basis in the kernels left them
// bound by the encoding, 1.55 and 1.45 ms, and FP32 cross terms left small blocks' sums
// less accurate).  Groups with a component outside the format are computed in FP64 from the
// basis itself.
#include <cooperative_groups.h>

#include "coarse.cuh"
#include "fx_device.cuh"

namespace hdcr {

namespace cg = cooperative_groups;

constexpr int FXT_THREADS = 128;
constexpr int FXT_UP = 6;  // the largest components: 2^58 <= |V| < 2^59
constexpr int FXT_KC = 8;  // basis vectors per restriction CTA
// biased exponents that a group's sum may start from, so that it stays a normal number
constexpr int FXT_LOW = 70, FXT_HIGH = 2000;

__device__ __forceinline__ int4 fxt_encode(cpx<double> x, int ex) { return fx_encode(x, ex, FXT_UP); }

__global__ void __launch_bounds__(128) fxt_encode_kernel(int ls, i64 sites, const cpx<double>* __restrict__ in, FxField f) {
  const i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= sites) return;
  const i64 x4 = i / ls;
  const i64 o = x4 * 12 * ls + (i - x4 * ls);
  cpx<double> x[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) x[c] = ld(in + o + c * ls);
  const int ex = fx_mark(fx_top(x), FX_SITE_MIN, FX_SITE_MAX);
#pragma unroll
  for (int c = 0; c < 12; ++c) f.v[o + c * ls] = fxt_encode(x[c], ex);
  f.ex[i] = ex;
}

// coarse[r][a][k] = <phi_k, fine_r> over block a: a cluster of CTAs shares a block, each
// thread sums the 12 components of a site exactly and adds sites in FP64, and the cluster's
// partial sums are added in the CTAs' order.
__global__ void __launch_bounds__(FXT_THREADS, 4) restrict_fx_kernel(Geom g, BlockGeom bg, FxField basis,
                                                                     const cpx<double>* __restrict__ phi,
                                                                     const cpx<double>* __restrict__ fine,
                                                                     cpx<double>* __restrict__ coarse, int nvec) {
  __shared__ int4 sv[12][FXT_THREADS];             // this thread's site of the field, encoded
  __shared__ double acc[2 * FXT_KC][FXT_THREADS];  // and its sums
  __shared__ double red[2 * FXT_KC];
  cg::cluster_group cluster = cg::this_cluster();
  const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int a = blockIdx.x / S, k0 = blockIdx.y * FXT_KC, r = blockIdx.z, t = threadIdx.x;
  const int nk = min(FXT_KC, nvec - k0);
  const i64 fs = g.V5 * 12;
  const cpx<double>* v = fine + r * fs;
  for (int i = 0; i < 2 * nk; ++i) acc[i][t] = 0.0;
  const int items = (int)bg.K5;
  for (int l = rank * FXT_THREADS + t; l < items; l += S * FXT_THREADS) {
    const int x4 = (int)(block_site(g, bg, a, l) / g.Ls);
    const int s = l % g.Ls;
    const unsigned o = (unsigned)(x4 * 12 * g.Ls + s);
    int ev;
    {
      cpx<double> x[12];
#pragma unroll
      for (int c = 0; c < 12; ++c) x[c] = ld(v + o + c * g.Ls);
      ev = fx_mark(fx_top(x), FX_SITE_MIN, FX_SITE_MAX);
#pragma unroll
      for (int c = 0; c < 12; ++c) sv[c][t] = fxt_encode(x[c], ev);
    }
    const int4* p = basis.v + k0 * fs + o;
    const int* pe = basis.ex + k0 * g.V5 + x4 * g.Ls + s;
#pragma unroll 2
    for (int k = 0; k < nk; ++k, p += fs, pe += g.V5) {
      const int ep = __ldg(pe);
      int4 q[12];
#pragma unroll
      for (int c = 0; c < 12; ++c) q[c] = __ldg(p + c * g.Ls);
      const int be = ev + ep - 1016;  // both scaled by 2^-1051 (H), a leading bit 63
      double sr = 0.0, si = 0.0;
      if (ev != 0 && ep != 0 && be >= FXT_LOW && be <= FXT_HIGH) {
        i64 hr = 0, hi = 0;
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          i64 lr = 1LL << 29, li = 1LL << 29;  // 24 cross products of 2^58 stay below 2^63
#pragma unroll
          for (int c = 6 * half; c < 6 * half + 6; ++c) {
            const int4 w = sv[c][t];
            const int n = -q[c].z, m = -q[c].w;  // conj(q) w
            hr = mw(q[c].z, w.z, mw(q[c].x, w.x, hr));
            hi = mw(n, w.x, mw(q[c].x, w.z, hi));
            lr = mw(q[c].w, w.z, mw(q[c].z, w.w, mw(q[c].y, w.x, mw(q[c].x, w.y, lr))));
            li = mw(m, w.x, mw(n, w.y, mw(q[c].y, w.z, mw(q[c].x, w.w, li))));
          }
          hr += lr >> 30;
          hi += li >> 30;
        }
        sr = fx_to_double(hr, be);
        si = fx_to_double(hi, be);
      } else if (ev == FX_RAW || ep == FX_RAW || (ev != 0 && ep != 0)) {
        const cpx<double>* f = phi + (k0 + k) * fs + o;
        for (int c = 0; c < 12; ++c) {
          const cpx<double> x = f[c * g.Ls], w = v[o + c * g.Ls];
          sr = fma(x.re, w.re, fma(x.im, w.im, sr));
          si = fma(x.re, w.im, fma(-x.im, w.re, si));
        }
      }
      acc[2 * k][t] += sr;
      acc[2 * k + 1][t] += si;
    }
  }
  __syncthreads();
  // warp w adds the threads' sums of every fourth value
  for (int i = t >> 5; i < 2 * nk; i += FXT_THREADS / 32) {
    double x = 0.0;
    for (int j = t & 31; j < FXT_THREADS; j += 32) x += acc[i][j];
    for (int off = 16; off > 0; off >>= 1) x += __shfl_down_sync(0xffffffffu, x, off);
    if ((t & 31) == 0) red[i] = x;
  }
  cluster.sync();
  if (rank == 0 && t < 2 * nk) {
    double x = 0.0;
    for (int q = 0; q < S; ++q) x += *cluster.map_shared_rank(red + t, q);
    reinterpret_cast<double*>(coarse + ((i64)r * bg.Vc + a) * nvec + k0)[t] = x;
  }
  cluster.sync();  // a CTA's sums stay until they are read
}

// fine = fine_in + sum_k phi_k c[a][k]; a thread has one chirality (6 components) of a 5d site and
// sums over k in 64-bit integers at the scale of the largest term so far, 2^-57 of it a step
__global__ void __launch_bounds__(FXT_THREADS, 4) prolong_fx_kernel(Geom g, BlockGeom bg, FxField basis,
                                                                    const cpx<double>* __restrict__ phi,
                                                                    const cpx<double>* __restrict__ coarse,
                                                                    const cpx<double>* fine_in, cpx<double>* fine,
                                                                    int nvec, int sh0, int parts) {
  extern __shared__ int4 cf[];  // [nvec] encoded coefficients, then [nvec] exponents
  int* ce = (int*)(cf + nvec);
  const int a = blockIdx.x / parts, r = blockIdx.z;
  const i64 fs = g.V5 * 12;
  const cpx<double>* cin = coarse + ((i64)r * bg.Vc + a) * nvec;
  for (int k = threadIdx.x; k < nvec; k += FXT_THREADS) {
    const cpx<double> x[1] = {cin[k]};
    const int e = fx_mark(fx_top(x), FX_SITE_MIN, FX_SITE_MAX);
    cf[k] = fxt_encode(x[0], e);
    ce[k] = e;
  }
  __syncthreads();
  const int items = (int)bg.K5;
  int l = (blockIdx.x - a * parts) * FXT_THREADS + threadIdx.x;
  if (l >= 2 * items) return;
  const int half = l >= items;
  l -= half * items;
  const int x4 = (int)(block_site(g, bg, a, l) / g.Ls);
  const int s = l % g.Ls;
  const unsigned o = (unsigned)((x4 * 12 + 6 * half) * g.Ls + s);
  i64 acc[6][2];
#pragma unroll
  for (int c = 0; c < 6; ++c) acc[c][0] = acc[c][1] = 0;
  int E = 0;  // the exponents' sum that acc is scaled by
  bool fp64 = false;
  const int4* p = basis.v + o;
  const int* pe = basis.ex + x4 * g.Ls + s;
#pragma unroll 2
  for (int k = 0; k < nvec; ++k, p += fs, pe += g.V5) {
    const int ep = __ldg(pe);
    int4 q[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) q[c] = __ldg(p + c * g.Ls);
    const int ek = ce[k], e = ep + ek;
    if (ep == FX_RAW || ek == FX_RAW) {
      fp64 = true;
      continue;
    }
    if (ep == 0 || ek == 0) continue;
    if (e - 1016 < FXT_LOW || e - 1016 > FXT_HIGH) {
      fp64 = true;
      continue;
    }
    if (e > E) {
      const int d = min(e - E, 62);
      if (E != 0)
#pragma unroll
        for (int c = 0; c < 6; ++c)
#pragma unroll
          for (int j = 0; j < 2; ++j) acc[c][j] = (acc[c][j] + (1LL << (d - 1))) >> d;
      E = e;
    }
    const int sh = min(E - e + sh0, 61);
    const i64 half_bit = (1LL << sh) >> 1;
    const int4 w = cf[k];
    const int n = -w.z, m = -w.w;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const i64 lr = mw(m, q[c].z, mw(n, q[c].w, mw(w.y, q[c].x, mw(w.x, q[c].y, 1LL << 29))));
      const i64 li = mw(w.w, q[c].x, mw(w.z, q[c].y, mw(w.y, q[c].z, mw(w.x, q[c].w, 1LL << 29))));
      const i64 hr = mw(n, q[c].z, mw(w.x, q[c].x, half_bit)) + (lr >> 30);
      const i64 hi = mw(w.z, q[c].x, mw(w.x, q[c].z, half_bit)) + (li >> 30);
      acc[c][0] += hr >> sh;
      acc[c][1] += hi >> sh;
    }
  }
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const i64 i = r * fs + o + c * g.Ls;
    cpx<double> y(fx_to_double(acc[c][0], E + sh0 - 1016), fx_to_double(acc[c][1], E + sh0 - 1016));
    if (fp64) {
      y = cpx<double>(0.0, 0.0);
      for (int k = 0; k < nvec; ++k) y = cmadd(y, phi[k * fs + o + c * g.Ls], cin[k]);
    }
    if (fine_in) y = fine_in[i] + y;
    fine[i] = y;
  }
}

static FxField basis_field(const hdcr_subspace* sub) {
  FxField f;
  f.v = (int4*)sub->fx;
  f.ex = (int*)(f.v + (size_t)sub->nvec * sub->g.V5 * 12);
  return f;
}

int subspace_encode(hdcr_subspace* sub, cudaStream_t st) {
  const size_t n = (size_t)sub->nvec * sub->g.V5, bytes = n * 12 * sizeof(int4) + n * sizeof(int);
  size_t free_bytes = 0, total = 0;
  if (cudaMemGetInfo(&free_bytes, &total) != cudaSuccess || free_bytes / 4 < bytes ||
      cudaMalloc(&sub->fx, bytes) != cudaSuccess) {
    cudaGetLastError();
    sub->fx = nullptr;
    return HDCR_OK;
  }
  fxt_encode_kernel<<<(unsigned)((n + 127) / 128), 128, 0, st>>>(sub->g.Ls, (i64)n, (const cpx<double>*)sub->vecs,
                                                                basis_field(sub));
  count_launch();
  HDCR_LAUNCH_CHECK();
  HDCR_CUDA_TRY(cudaStreamSynchronize(st));
  return HDCR_OK;
}

int launch_restrict_fx(const hdcr_subspace* sub, const cpx<double>* fine, cpx<double>* coarse, int nrhs,
                       cudaStream_t st) {
  const int chunks = (sub->nvec + FXT_KC - 1) / FXT_KC;
  const int S = restrict_cluster((long long)sub->bg.Vc * chunks * nrhs, sub->bg.K5 / FXT_THREADS);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(sub->bg.Vc * S, chunks, nrhs);
  cfg.blockDim = dim3(FXT_THREADS);
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = S;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  HDCR_CUDA_TRY(cudaLaunchKernelEx(&cfg, restrict_fx_kernel, sub->g, sub->bg, basis_field(sub),
                                   (const cpx<double>*)sub->vecs, fine, coarse, sub->nvec));
  count_launch();
  return HDCR_OK;
}

int launch_prolong_fx(const hdcr_subspace* sub, const cpx<double>* coarse, const cpx<double>* fine_in,
                      cpx<double>* fine, int nrhs, cudaStream_t st) {
  int sh0 = 0;  // nvec terms of 2^59 stay below 2^62
  while ((8 << sh0) < sub->nvec) ++sh0;
  const int parts = (int)((2 * sub->bg.K5 + FXT_THREADS - 1) / FXT_THREADS);
  const size_t smem = (sizeof(int4) + sizeof(int)) * (size_t)sub->nvec;  // nvec <= 256
  prolong_fx_kernel<<<dim3((unsigned)sub->bg.Vc * parts, 1, nrhs), FXT_THREADS, smem, st>>>(
      sub->g, sub->bg, basis_field(sub), (const cpx<double>*)sub->vecs, coarse, fine_in, fine, sub->nvec, sh0, parts);
  count_launch();
  HDCR_LAUNCH_CHECK();
  return HDCR_OK;
}

}  // namespace hdcr
