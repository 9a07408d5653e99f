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
// (the dropped L L' is below 2^-60 of the scale), and a site's 12 components are summed exactly
// (encoding the FP64 basis in the kernels left them bound by the encoding, 1.55 and 1.45 ms, and
// FP32 cross terms left small blocks' sums less accurate).  Groups with a component outside the format are
// computed in FP64 from the basis itself, and so is a result that FP64 sums would give more
// accurately, because the field is small where the basis is large and the other way round: the
// kernels sum how large a result's terms are beside the scale that they were held at.
#include <cooperative_groups.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "coarse.cuh"
#include "fx_device.cuh"

namespace hdcr {

namespace cg = cooperative_groups;

constexpr int FXT_THREADS = 128;
constexpr int FXT_UP = 6;  // the largest components: 2^58 <= |V| < 2^59
constexpr int FXT_KC = 8;  // basis vectors per restriction CTA
// biased exponents that a group's sum may start from, so that it stays a normal number
constexpr int FXT_LOW = 70, FXT_HIGH = 2000;
// A site's sum of 24 products errs by 0.6 of the integers' unit (the largest product is 2^58 of them),
// FP64 multiply-adds by 2^-54 of the sum or more: the integers are as good where the sites' sums, squared and
// added up, are (1.2 2^-10)^2 of the scales 2^63, squared and added up.  Gaussian fields are at 2^-13.4, 70 times
// that.
constexpr float FXT_K2 = 1.44f * 0x1p-20f;
constexpr int FXT_FULL = 1 << 25;  // 2^62 in units of 2^37
constexpr int FXT_SPAN = 60;  // exponents above the thread's first site's that the sums of squares may hold

struct RestrictShared {
  int4 sv[12][FXT_THREADS];             // a thread's site of the field, encoded
  double acc[2 * FXT_KC][FXT_THREADS];  // and its sums
  float sure[2 * FXT_KC][FXT_THREADS];  // sum of (site sum / 2^63)^2 - K2 over its sites, in units of 4^ref
  double red[2 * FXT_KC];
  float rsure[2 * FXT_KC];
  int wref[FXT_THREADS / 32];           // the warps' largest ref, then in [0] the CTA's
  unsigned again;                       // the results to be computed in FP64
};

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
  extern __shared__ int4 restrict_mem[];
  RestrictShared& sh = *reinterpret_cast<RestrictShared*>(restrict_mem);
  cg::cluster_group cluster = cg::this_cluster();
  const int S = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  const int a = blockIdx.x / S, k0 = blockIdx.y * FXT_KC, r = blockIdx.z, t = threadIdx.x;
  const int nk = min(FXT_KC, nvec - k0);
  const i64 fs = g.V5 * 12;
  const cpx<double>* v = fine + r * fs;
  for (int i = 0; i < 2 * nk; ++i) {
    sh.acc[i][t] = 0.0;
    sh.sure[i][t] = 0.f;
  }
  int ref = 0;  // 0: no site yet
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
      for (int c = 0; c < 12; ++c) sh.sv[c][t] = fxt_encode(x[c], ev);
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
            const int4 w = sh.sv[c][t];
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
        if (ref == 0) ref = be;
        const int d = be - ref;
        // 2^d, infinite above FXT_SPAN: then the result is not certain
        const float f = __int_as_float(d > FXT_SPAN ? 0x7f800000 : (127 + max(d, -FXT_SPAN)) << 23);
        const float xr = (float)(int)(hr >> 32) * 0x1p-31f, xi = (float)(int)(hi >> 32) * 0x1p-31f;
        sh.sure[2 * k][t] += f * (f * fmaf(xr, xr, -FXT_K2));
        sh.sure[2 * k + 1][t] += f * (f * fmaf(xi, xi, -FXT_K2));
      } else if (ev == FX_RAW || ep == FX_RAW || (ev != 0 && ep != 0)) {
        const cpx<double>* f = phi + (k0 + k) * fs + o;
        for (int c = 0; c < 12; ++c) {
          const cpx<double> x = f[c * g.Ls], w = v[o + c * g.Ls];
          sr = fma(x.re, w.re, fma(x.im, w.im, sr));
          si = fma(x.re, w.im, fma(-x.im, w.re, si));
        }
      }
      sh.acc[2 * k][t] += sr;
      sh.acc[2 * k + 1][t] += si;
    }
  }
  int wref = ref;
  for (int off = 16; off > 0; off >>= 1) wref = max(wref, __shfl_xor_sync(0xffffffffu, wref, off));
  if ((t & 31) == 0) sh.wref[t >> 5] = wref;
  __syncthreads();
  int cref = sh.wref[0];
#pragma unroll
  for (int w = 1; w < FXT_THREADS / 32; ++w) cref = max(cref, sh.wref[w]);
  {
    const float f = __int_as_float(max(127 + ref - cref, 0) << 23);
    for (int i = 0; i < 2 * nk; ++i) sh.sure[i][t] = f * (f * sh.sure[i][t]);
  }
  __syncthreads();
  // warp w adds the threads' sums of every fourth value
  for (int i = t >> 5; i < 2 * nk; i += FXT_THREADS / 32) {
    double x = 0.0;
    float y = 0.f;
    for (int j = t & 31; j < FXT_THREADS; j += 32) {
      x += sh.acc[i][j];
      y += sh.sure[i][j];
    }
    for (int off = 16; off > 0; off >>= 1) {
      x += __shfl_down_sync(0xffffffffu, x, off);
      y += __shfl_down_sync(0xffffffffu, y, off);
    }
    if ((t & 31) == 0) {
      sh.red[i] = x;
      sh.rsure[i] = y;
    }
  }
  if (t == 0) {
    sh.wref[0] = cref;
    sh.again = 0;
  }
  cluster.sync();
  if (rank == 0 && t < 2 * nk) {
    double x = 0.0;
    int top = 0;
    for (int q = 0; q < S; ++q) {
      x += *cluster.map_shared_rank(sh.red + t, q);
      top = max(top, *cluster.map_shared_rank(sh.wref, q));
    }
    float y = 0.f;
    for (int q = 0; q < S; ++q) {
      const float f = __int_as_float(max(127 + *cluster.map_shared_rank(sh.wref, q) - top, 0) << 23);
      y += f * (f * *cluster.map_shared_rank(sh.rsure + t, q));
    }
    if (!(y >= 0.f)) atomicOr(&sh.again, 1u << t);
    reinterpret_cast<double*>(coarse + ((i64)r * bg.Vc + a) * nvec + k0)[t] = x;
  }
  cluster.sync();  // a CTA's sums stay until they are read
  if (rank != 0 || sh.again == 0) return;
  for (int k = 0; k < nk; ++k) {
    if (!(sh.again >> (2 * k) & 3)) continue;
    const cpx<double>* f = phi + (k0 + k) * fs;
    double x[2] = {0.0, 0.0};
    for (int l = t; l < items; l += FXT_THREADS) {
      const int x4 = (int)(block_site(g, bg, a, l) / g.Ls);
      const unsigned o = (unsigned)(x4 * 12 * g.Ls + l % g.Ls);
      for (int c = 0; c < 12; ++c) {
        const cpx<double> p = ld(f + o + c * g.Ls), w = ld(v + o + c * g.Ls);
        x[0] = fma(p.re, w.re, fma(p.im, w.im, x[0]));
        x[1] = fma(p.re, w.im, fma(-p.im, w.re, x[1]));
      }
    }
    for (int j = 0; j < 2; ++j) {
      for (int off = 16; off > 0; off >>= 1) x[j] += __shfl_down_sync(0xffffffffu, x[j], off);
      if ((t & 31) == 0) sh.acc[j][t] = x[j];
    }
    __syncthreads();
    if (t < 2) {
      double y = 0.0;
      for (int w = 0; w < FXT_THREADS; w += 32) y += sh.acc[t][w];
      reinterpret_cast<double*>(coarse + ((i64)r * bg.Vc + a) * nvec + k0 + k)[t] = y;
    }
    __syncthreads();
  }
}

// fine = fine_in + sum_k phi_k c[a][k]; a thread has one chirality (6 components) of a 5d site and
// sums over k in 64-bit integers at the scale of the largest term so far.  A term of two products errs by
// 0.35 of their unit and is 2^59 at most; FP64 multiply-adds err by 0.29 2^-53 of the sum of the terms'
// magnitudes.  So that sum has to reach ``sure`` (1.5 sqrt(nvec) 2^53 in units of 2^37; Gaussian fields have
// about 9 times that), and must not reach 2^62, beyond which the terms' sum might leave its 64 bits: else the
// thread sums in FP64.
__global__ void __launch_bounds__(FXT_THREADS, 4) prolong_fx_kernel(Geom g, BlockGeom bg, FxField basis,
                                                                    const cpx<double>* __restrict__ phi,
                                                                    const cpx<double>* __restrict__ coarse,
                                                                    const cpx<double>* fine_in, cpx<double>* fine,
                                                                    int nvec, int sure, int parts) {
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
  int mag[6][2];  // the terms' magnitudes summed, in units of 2^37 (at most 2^22 each)
#pragma unroll
  for (int c = 0; c < 6; ++c) acc[c][0] = acc[c][1] = 0, mag[c][0] = mag[c][1] = 0;
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
          for (int j = 0; j < 2; ++j) {
            if (mag[c][j] >= FXT_FULL) fp64 = true;
            acc[c][j] = (acc[c][j] + (1LL << (d - 1))) >> d;
            mag[c][j] >>= min(d, 31);
          }
      E = e;
    }
    const int sh = min(E - e, 61);
    const i64 half_bit = (1LL << sh) >> 1;
    const int4 w = cf[k];
    const int n = -w.z, m = -w.w;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const i64 lr = mw(m, q[c].z, mw(n, q[c].w, mw(w.y, q[c].x, mw(w.x, q[c].y, 1LL << 29))));
      const i64 li = mw(w.w, q[c].x, mw(w.z, q[c].y, mw(w.y, q[c].z, mw(w.x, q[c].w, 1LL << 29))));
      const i64 hr = (mw(n, q[c].z, mw(w.x, q[c].x, half_bit)) + (lr >> 30)) >> sh;
      const i64 hi = (mw(w.z, q[c].x, mw(w.x, q[c].z, half_bit)) + (li >> 30)) >> sh;
      acc[c][0] += hr;
      acc[c][1] += hi;
      mag[c][0] += abs((int)(hr >> 32)) >> 5;
      mag[c][1] += abs((int)(hi >> 32)) >> 5;
    }
  }
  if (E != 0)
#pragma unroll
    for (int c = 0; c < 6; ++c)
#pragma unroll
      for (int j = 0; j < 2; ++j) fp64 |= mag[c][j] < sure || mag[c][j] >= FXT_FULL;
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    const i64 i = r * fs + o + c * g.Ls;
    cpx<double> y(fx_to_double(acc[c][0], E - 1016), fx_to_double(acc[c][1], E - 1016));
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

// the subspaces that have one
static std::mutex g_fx_mu;
static std::vector<hdcr_subspace*> g_fx_subs;

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
  std::lock_guard<std::mutex> lock(g_fx_mu);
  g_fx_subs.push_back(sub);
  return HDCR_OK;
}

void subspace_fx_free(hdcr_subspace* sub) {
  std::lock_guard<std::mutex> lock(g_fx_mu);
  g_fx_subs.erase(std::remove(g_fx_subs.begin(), g_fx_subs.end(), sub), g_fx_subs.end());
  if (sub->fx) cudaFree(sub->fx);
  sub->fx = nullptr;
}

bool subspace_fx_lock(const hdcr_subspace* sub, cudaStream_t st, std::shared_lock<std::shared_mutex>* lock) {
  *lock = std::shared_lock<std::shared_mutex>(sub->fx_mu);
  if (!sub->fx) {
    lock->unlock();
    return false;
  }
  cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &status) != cudaSuccess) {
    cudaGetLastError();
    sub->fx_captured = true;
  } else if (status != cudaStreamCaptureStatusNone) {
    sub->fx_captured = true;
  }
  return true;
}

// gives back one copy on the current device that no captured graph reads, its launches done
static bool give_back_one() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  std::lock_guard<std::mutex> lock(g_fx_mu);
  for (size_t i = 0; i < g_fx_subs.size(); ++i) {
    hdcr_subspace* sub = g_fx_subs[i];
    std::unique_lock<std::shared_mutex> own(sub->fx_mu);
    if (sub->device != dev || sub->fx_captured) continue;
    if (cudaDeviceSynchronize() != cudaSuccess || cudaFree(sub->fx) != cudaSuccess) return false;
    sub->fx = nullptr;
    g_fx_subs.erase(g_fx_subs.begin() + i);
    return true;
  }
  return false;
}

cudaError_t dev_malloc_bytes(void** p, size_t bytes) {
  for (;;) {
    const cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    if (!give_back_one()) return e;
  }
}

int launch_restrict_fx(const hdcr_subspace* sub, const cpx<double>* fine, cpx<double>* coarse, int nrhs,
                       cudaStream_t st) {
  const int chunks = (sub->nvec + FXT_KC - 1) / FXT_KC;
  const int S = restrict_cluster((long long)sub->bg.Vc * chunks * nrhs, sub->bg.K5 / FXT_THREADS);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(sub->bg.Vc * S, chunks, nrhs);
  cfg.blockDim = dim3(FXT_THREADS);
  cfg.dynamicSmemBytes = sizeof(RestrictShared);
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = S;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  HDCR_CUDA_TRY(cudaFuncSetAttribute(restrict_fx_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)sizeof(RestrictShared)));
  HDCR_CUDA_TRY(cudaLaunchKernelEx(&cfg, restrict_fx_kernel, sub->g, sub->bg, basis_field(sub),
                                   (const cpx<double>*)sub->vecs, fine, coarse, sub->nvec));
  count_launch();
  return HDCR_OK;
}

int launch_prolong_fx(const hdcr_subspace* sub, const cpx<double>* coarse, const cpx<double>* fine_in,
                      cpx<double>* fine, int nrhs, cudaStream_t st) {
  const int sure = (int)(1.5 * sqrt((double)sub->nvec) * (1 << 16));
  const int parts = (int)((2 * sub->bg.K5 + FXT_THREADS - 1) / FXT_THREADS);
  const size_t smem = (sizeof(int4) + sizeof(int)) * (size_t)sub->nvec;  // nvec <= 256
  prolong_fx_kernel<<<dim3((unsigned)sub->bg.Vc * parts, 1, nrhs), FXT_THREADS, smem, st>>>(
      sub->g, sub->bg, basis_field(sub), (const cpx<double>*)sub->vecs, coarse, fine_in, fine, sub->nvec, sure, parts);
  count_launch();
  HDCR_LAUNCH_CHECK();
  return HDCR_OK;
}

}  // namespace hdcr
