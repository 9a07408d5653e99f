// Fine operator H = Gamma5 D_dwf in FP64 accuracy on the integer pipe (the format
// and its error are described in dwf_fx.cuh).
#include "dwf_stencil.cuh"
#include "fx_device.cuh"

namespace hdcr {

// One launch: the first fblocks CTAs encode a field's 5d sites, the others links.
// Bound by the memory it streams (32 B per complex number): 16^4 x 16, 0.48 GB.
__global__ void __launch_bounds__(128) fx_encode_kernel(int ls, i64 nsites, const cpx<double>* __restrict__ in,
                                                        FxField f, int fblocks, i64 nlinks,
                                                        const cpx<double>* __restrict__ U, FxLinks u) {
  if ((int)blockIdx.x < fblocks) {
    const i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= nsites) return;
    const i64 x4 = i / ls;
    const i64 o = x4 * 12 * ls + (i - x4 * ls);
    cpx<double> x[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) x[c] = ld(in + o + c * ls);
    const int ex = fx_mark(fx_top(x), FX_SITE_MIN, FX_SITE_MAX);
#pragma unroll
    for (int c = 0; c < 12; ++c) f.v[o + c * ls] = fx_encode(x[c], ex, FX_UP);
    f.ex[i] = ex;
  } else {
    const i64 i = (i64)(blockIdx.x - fblocks) * blockDim.x + threadIdx.x;
    if (i >= nlinks) return;
    cpx<double> x[9];
#pragma unroll
    for (int c = 0; c < 9; ++c) x[c] = ld(U + i * 9 + c);
    const int ex = fx_mark(fx_top(x), FX_LINK_MIN, FX_LINK_MAX);
#pragma unroll
    for (int c = 0; c < 9; ++c) u.v[i * 9 + c] = fx_encode(x[c], ex, FX_UP + 1);
    u.ex[i] = ex;
  }
}

// ------------------------------------------------------------------- stencil
// a real coefficient of the operator, encoded on the host: (h + l / 2^30) 2^(ex - 1052)
struct FxCoef {
  int h, l, ex;
  double d;
};

struct FxParams {
  FxCoef diag, one, mmf;  // 5 - M5, 1 (the s-hops' weight) and -mf (their weight across a wall)
};

__device__ __forceinline__ int4 ldi(const int4* p) { return __ldg(p); }

// field r of a launch over several
__device__ __forceinline__ FxField fx_field_r(const Geom& g, const FxField& f, int r) {
  FxField q;
  q.v = f.v + (i64)r * 12 * g.V5;
  q.ex = f.ex + (i64)r * g.V5;
  q.f64 = f.f64 + (i64)r * 12 * g.V5;
  return q;
}

// (row, lower component) tables of i sigma_k: component a of i sigma_k w is
// sign * i^rot * w[1 - a or a]
template <int K>
struct ISigma {
  static constexpr int idx(int a) { return K < 2 ? 1 - a : a; }
  static constexpr int rot() { return K == 1 || K == 3 ? 0 : 1; }
  // K = 0: (i w1, i w0); 1: (w1, -w0); 2: (i w0, -i w1); 3 (gamma_t): (-w0, -w1)
  static constexpr int sign(int a) { return K == 0 ? 1 : K == 3 ? -1 : a == 0 ? 1 : -1; }
};

// u + S i^rot d
__device__ __forceinline__ int4 fx_add(int4 u, int4 d, int S, int rot) {
  if (rot == 0)
    return S > 0 ? make_int4(u.x + d.x, u.y + d.y, u.z + d.z, u.w + d.w)
                 : make_int4(u.x - d.x, u.y - d.y, u.z - d.z, u.w - d.w);
  return S > 0 ? make_int4(u.x - d.z, u.y - d.w, u.z + d.x, u.w + d.y)
               : make_int4(u.x + d.z, u.y + d.w, u.z - d.x, u.w - d.y);
}

// A real of a site is certain once one of its terms is at least 2^52 (high word FX_CERTAIN).  The integers
// err by about 0.9 of their unit (8 hops' rounded cross products and dropped L L', operands
// held to 1/2 of the last bit); FP64 multiply-adds round each of some 12 sums to 2^-53 of it, 0.29 of a
// unit each once it is at 2^52, so from there on they err by as much.  At 2^51 components of 0.1 of a
// site's largest came out at 1.7e-16 of themselves instead of FP64's 1.5e-16; at 2^53 the error is no
// smaller where it matters, and a solver's fields send a site or two of 8^4 x 8 to FP64 in most
// iterations: 94 instead of 68 us an iteration of CR.
// A term of 2^59 or more (high word FX_HUGE) could take the sum out of range; a term of
// numbers in the format may reach 2^60.6, with links far from unitary.
constexpr int FX_CERTAIN = 1 << 20, FX_HUGE = 1 << 27;
constexpr unsigned FX_ALL = 0xffffff;  // bit 2 (3 spin + colour) + (0 re, 1 im) for each real

// acc -= one hop without its factor 1/2, each colour component of its two spins rounded to
// nearest after a right shift by sh.  acc[spin][colour][re, im].  A complex product takes three
// real ones, a (c + d), d (a + b) and c (a - b) for (a + i b) (c + i d).
template <int MU, int SIGN>
__device__ __forceinline__ void fx_hop(const int4* __restrict__ Ul, const int4* __restrict__ nb, int ls, int sh,
                                       bool flip, i64 (&acc)[4][3][2], unsigned& ok, int& top) {
  typedef ISigma<MU> T;
  int4 h[2][3];  // the two spins of u -+ ...
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int4 u = ldi(nb + (3 * j + c) * ls), d = ldi(nb + (6 + 3 * T::idx(j) + c) * ls);
      h[j][c] = fx_add(u, d, SIGN * T::sign(j), T::rot());
    }
  const i64 half = (1LL << sh) >> 1;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    int4 m[3];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      m[b] = ldi(Ul + (SIGN > 0 ? 3 * c + b : 3 * b + c));
      if (MU == 3 && flip) m[b] = make_int4(-m[b].x, -m[b].y, -m[b].z, -m[b].w);  // the antiperiodic boundary
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      i64 k1 = half, k2 = 0, k3 = 0, x1 = 1LL << 29, x2 = 0, x3 = 0;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const int4 v = h[j][b];
        const int sH = v.x + v.z, sL = v.y + v.w;
        // a + b and a - b, b the link's imaginary part or, in its adjoint, minus that
        const int pH = SIGN > 0 ? m[b].x + m[b].z : m[b].x - m[b].z, pL = SIGN > 0 ? m[b].y + m[b].w : m[b].y - m[b].w;
        const int qH = SIGN > 0 ? m[b].x - m[b].z : m[b].x + m[b].z, qL = SIGN > 0 ? m[b].y - m[b].w : m[b].y + m[b].w;
        k1 = mw(m[b].x, sH, k1);
        k2 = mw(pH, v.z, k2);
        k3 = mw(qH, v.x, k3);
        x1 = mw(m[b].x, sL, mw(m[b].y, sH, x1));
        x2 = mw(pH, v.w, mw(pL, v.z, x2));
        x3 = mw(qH, v.y, mw(qL, v.x, x3));
      }
      const i64 pr = (k1 - k2 + ((x1 - x2) >> 30)) >> sh, pi = (k1 - k3 + ((x1 - x3) >> 30)) >> sh;
      acc[j][c][0] -= pr;
      acc[j][c][1] -= pi;
      // lower = -+ i sigma h, subtracted: component a takes S i^rot of spin j = idx(a)
      const int a = T::idx(j), S = MU == 3 ? SIGN : SIGN * T::sign(a);
      const int up = 2 * (3 * j + c), lo = 2 * (3 * (2 + a) + c);
      const int ar = abs((int)(pr >> 32)), ai = abs((int)(pi >> 32));
      if (ar >= FX_CERTAIN) ok |= 1u << up | 1u << (lo + T::rot());
      if (ai >= FX_CERTAIN) ok |= 2u << up | 1u << (lo + 1 - T::rot());
      top |= ar | ai;
      if (T::rot() == 0) {
        acc[2 + a][c][0] += S > 0 ? pr : -pr;
        acc[2 + a][c][1] += S > 0 ? pi : -pi;
      } else {
        acc[2 + a][c][0] += S > 0 ? -pi : pi;
        acc[2 + a][c][1] += S > 0 ? pr : -pr;
      }
    }
  }
}

// k v rounded to nearest after a right shift by sh >= 0, in a quarter of the unit of the integers' product
__device__ __forceinline__ i64 fx_mul(const FxCoef& k, int h, int l, int sh) {
  const i64 x = mw(k.h, l, mw(k.l, h, 1LL << 27)) >> 28;
  return ((mw(k.h, h, 0) << 2) + x + ((1LL << sh) >> 1)) >> sh;
}

// ------------------------------------------------ sites that need FP64 itself
// (D_dwf in)(x4, s), or its 4d hops alone, from the FP64 operands: the FP64 kernel's arithmetic in
// its order, with one body for the eight hops.  tab: the site's hop table.
template <bool LOCAL>
__device__ __forceinline__ void fx_fp64_site(const FxParams& p, const cpx<double>* U, const cpx<double>* in,
                                             const int4* tab, int ls, int x4, int s, cpx<double> (&acc)[12]) {
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    acc[c] = cpx<double>(0.0, 0.0);
    if (!LOCAL) continue;
    const cpx<double>* row = in + (unsigned)((x4 * 12 + c) * ls);
    const bool wall = c < 6 ? s == 0 : s + 1 == ls;
    const cpx<double> v = ld(row + s), o = ld(row + (c < 6 ? (wall ? ls - 1 : s - 1) : (wall ? 0 : s + 1)));
    const double w = wall ? p.mmf.d : 1.0;
    acc[c] = cpx<double>(fma(-w, o.re, p.diag.d * v.re), fma(-w, o.im, p.diag.d * v.im));
  }
#pragma unroll 1
  for (int d = 0; d < 8; ++d) {
    const int4 t = tab[d];
    const int mu = d >> 1;
    const bool back = d & 1, swap = mu < 2, rot = mu == 0 || mu == 2;  // (ISigma's tables)
    const double coef = t.w ? 0.5 : -0.5, S = back ? -1.0 : 1.0;
    const double s0 = mu == 3 ? -S : S, s1 = mu == 0 ? S : -S;  // the signs of i sigma's two components
    const cpx<double>* nb = in + (unsigned)(t.x * 12 + s);
    const cpx<double>* Ul = U + (unsigned)t.y;
    cpx<double> h[2][3], q[2][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const cpx<double> u0 = ld(nb + c * ls), u1 = ld(nb + (3 + c) * ls);
      cpx<double> d0 = ld(nb + (swap ? 9 + c : 6 + c) * ls), d1 = ld(nb + (swap ? 6 + c : 9 + c) * ls);
      if (rot) {
        d0 = times_i(d0);
        d1 = times_i(d1);
      }
      h[0][c] = cpx<double>(fma(s0, d0.re, u0.re), fma(s0, d0.im, u0.im));
      h[1][c] = cpx<double>(fma(s1, d1.re, u1.re), fma(s1, d1.im, u1.im));
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      q[0][c] = q[1][c] = cpx<double>(0.0, 0.0);
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        cpx<double> m = ld(Ul + (back ? 3 * b + c : 3 * c + b));
        if (back) m.im = -m.im;
        q[0][c] = cmadd(q[0][c], m, h[0][b]);
        q[1][c] = cmadd(q[1][c], m, h[1][b]);
      }
    }
    // lower = -+ i sigma of the upper
    const double c0 = mu == 3 ? -coef * S : -coef * s0, c1 = mu == 3 ? -coef * S : -coef * s1;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      cpx<double> l0 = swap ? q[1][c] : q[0][c], l1 = swap ? q[0][c] : q[1][c];
      if (rot) {
        l0 = times_i(l0);
        l1 = times_i(l1);
      }
      acc[c] = cpx<double>(fma(coef, q[0][c].re, acc[c].re), fma(coef, q[0][c].im, acc[c].im));
      acc[3 + c] = cpx<double>(fma(coef, q[1][c].re, acc[3 + c].re), fma(coef, q[1][c].im, acc[3 + c].im));
      acc[6 + c] = cpx<double>(fma(c0, l0.re, acc[6 + c].re), fma(c0, l0.im, acc[6 + c].im));
      acc[9 + c] = cpx<double>(fma(c1, l1.re, acc[9 + c].re), fma(c1, l1.im, acc[9 + c].im));
    }
  }
}

// ------------------------------------------------------------------ the kernel
// What a launch does with h = H in at each site
constexpr int FX_OUT = 0;    // out = h
constexpr int FX_BOTH = 2;   // out = h, h encoded into enc
constexpr int FX_DOT = 3;    // out = h and Re <src, h> into *result
constexpr int FX_RES = 4;    // out = src - h, also encoded into enc
constexpr int FX_CHEB = 5;   // prev <- nx = 2 (a h + b cur) - prev, acc += ck nx, nx encoded into enc
constexpr int FX_CHEB1 = 6;  // prev <- nx = a h + b cur, acc = c0 cur + ck nx, nx encoded into enc
constexpr int FX_CHEBL = 7;  // acc += ck (2 (a h + b cur) - prev), acc encoded into enc
// the red-black launches: the 4d hops alone, h = D_hop in on the sites of one parity
constexpr int FX_RB = 8;      // out = h
// w = M5 v - h, v = src: out = w, |w|^2 into *result and Gamma5 w into prev and encoded into enc; with dag
// v = Gamma5 src and out = Gamma5 w
constexpr int FX_RBS = 9;
constexpr bool fx_reduces(int mode) { return mode == FX_DOT || mode == FX_RBS; }
struct FxEpilogue {
  cpx<double>* out;
  FxField enc;
  const cpx<double>* src;
  const cpx<double>* cur;
  cpx<double>* prev;
  cpx<double>* acc;
  double a, b, ck, c0;
  int dag;
  RedScratch rs;
  double* result;
};

// one complex number of the epilogue: h in, the value to encode out.  The Chebyshev steps
// are three FP64 multiply-adds a real, 1.5 clocks of an SM beside the 1.9 of the stencil's wide integer
// multiply-adds.
template <int MODE>
__device__ __forceinline__ cpx<double> fx_epilogue(const FxEpilogue& ep, i64 o, cpx<double> h, double& dot) {
  if (MODE == FX_OUT || MODE == FX_BOTH || MODE == FX_DOT) st(ep.out + o, h);
  if (MODE == FX_DOT) {
    const cpx<double> q = ld(ep.src + o);
    dot = fma(q.re, h.re, fma(q.im, h.im, dot));
  }
  if (MODE == FX_RES) {
    h = ld(ep.src + o) - h;
    st(ep.out + o, h);
  }
  if (MODE == FX_CHEB || MODE == FX_CHEBL || MODE == FX_CHEB1) {
    const cpx<double> cv = ld(ep.cur + o);
    cpx<double> nx, av;
    if (MODE == FX_CHEB1) {
      nx.re = fma(ep.a, h.re, ep.b * cv.re);
      nx.im = fma(ep.a, h.im, ep.b * cv.im);
      av = cpx<double>(ep.c0 * cv.re, ep.c0 * cv.im);
    } else {
      const cpx<double> pv = ld(ep.prev + o);
      const double a2 = 2.0 * ep.a, b2 = 2.0 * ep.b;
      nx.re = fma(a2, h.re, fma(b2, cv.re, -pv.re));
      nx.im = fma(a2, h.im, fma(b2, cv.im, -pv.im));
      if (ep.acc) av = ld(ep.acc + o);
    }
    if (MODE != FX_CHEBL) st(ep.prev + o, nx);
    if (ep.acc) {
      av.re = fma(ep.ck, nx.re, av.re);
      av.im = fma(ep.ck, nx.im, av.im);
      st(ep.acc + o, av);
    }
    h = MODE == FX_CHEBL ? av : nx;
  }
  return h;
}

// The output of the red-black launches at one site from h = (D_hop in)(x4, s)
template <int MODE>
__device__ __forceinline__ void fx_rb_output(const Geom& g, const FxEpilogue& ep, int ls, int x4, int s,
                                             cpx<double> (&h)[12], double& dot) {
  const unsigned site = (unsigned)(x4 * 12 * ls);
  if (MODE == FX_RB) {
#pragma unroll
    for (int c = 0; c < 12; ++c) st(ep.out + site + c * ls + s, h[c]);
    return;
  }
  const int sr = ls - 1 - s;
  // M5 couples the upper spins to s - 1 and the lower to s + 1, with -mf across the wall
  const int sp = s == 0 ? ls - 1 : s - 1, sn = s + 1 == ls ? 0 : s + 1;
  const double kp = s == 0 ? ep.c0 : -1.0, kn = s + 1 == ls ? ep.c0 : -1.0;
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    const int so = c < 6 ? sp : sn;
    const double k = c < 6 ? kp : kn;
    cpx<double> v = ld(ep.src + site + c * ls + (ep.dag ? sr : s));
    cpx<double> w = ld(ep.src + site + c * ls + (ep.dag ? ls - 1 - so : so));
    const double sg = ep.dag && c >= 6 ? -1.0 : 1.0;  // Gamma5
    h[c].re = fma(sg * k, w.re, fma(sg * ep.a, v.re, -h[c].re));
    h[c].im = fma(sg * k, w.im, fma(sg * ep.a, v.im, -h[c].im));
    if (ep.dag) {
      st(ep.out + site + c * ls + sr, cpx<double>(sg * h[c].re, sg * h[c].im));
    } else {
      st(ep.out + site + c * ls + s, h[c]);
      dot = fma(h[c].re, h[c].re, fma(h[c].im, h[c].im, dot));
      if (c >= 6) h[c] = cpx<double>(-h[c].re, -h[c].im);
    }
  }
  if (!ep.dag) {
    const int ex = fx_mark(fx_top(h), FX_SITE_MIN, FX_SITE_MAX);
#pragma unroll
    for (int c = 0; c < 12; ++c) {
      ep.enc.v[site + c * ls + sr] = fx_encode(h[c], ex, FX_UP);
      st(ep.prev + site + c * ls + sr, h[c]);
    }
    ep.enc.ex[x4 * ls + sr] = ex;
  }
}

// A CTA's 4d sites: the box b[] of the lattice (n[] boxes in each direction), or ns
// consecutive ones in the field's order when b[0] is 0.  rb: of the sites of parity par,
// numbered with half the x extent.
struct FxTile {
  int rb, par;
  int b[4], n[4];
  int ns;     // 4d sites per tile
  int tiles;  // tiles per field
};

constexpr int FX_THREADS = 256;  // (4d site, s) of a tile
constexpr int FX_BLOCKS = 2;     // full tiles per SM
constexpr int FX_MAX_SITES = FX_THREADS / 2;  // Ls >= 2
constexpr int FX_SPLIT_SITES = 32;  // (4d site, s) of a tile whose sites are split over four warps
// Launches of at most this many 5d sites split them: a call (encoding and operator), whole sites
// and split, took 25 and 18 us at 4^4 x 8 (2048 sites), 34 and 28 at 18,900, 32 and 31 at
// 32,768, 43 and 51 at 65,536 and 78 and 91 at 131,072
constexpr long long FX_SPLIT_MAX = 24576;

// A site that reads an operand outside the format, or has a real that is not certain: the whole
// of its output in FP64
template <int MODE>
__device__ __forceinline__ void fx_slow_output(const Geom& g, const FxParams& p, const FxLinks& u, const FxField& in,
                                               const FxEpilogue& ep, const int4* tab, int r, int x4, int s,
                                               double& dot) {
  cpx<double> w[12];
  fx_fp64_site<MODE < FX_RB>(p, u.f64, in.f64, tab, g.Ls, x4, s, w);
  if (MODE >= FX_RB) {
    fx_rb_output<MODE>(g, ep, g.Ls, x4, s, w, dot);
    return;
  }
  const i64 site = (i64)r * g.V4 + x4, o0 = site * 12 * g.Ls + (g.Ls - 1 - s);
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    const double sg = c < 6 ? 1.0 : -1.0;
    w[c] = fx_epilogue<MODE>(ep, o0 + c * g.Ls, cpx<double>(sg * w[c].re, sg * w[c].im), dot);
  }
  if (MODE != FX_OUT && MODE != FX_DOT && ep.enc.v) {
    const int ex = fx_mark(fx_top(w), FX_SITE_MIN, FX_SITE_MAX);
#pragma unroll
    for (int c = 0; c < 12; ++c) ep.enc.v[o0 + c * g.Ls] = fx_encode(w[c], ex, FX_UP);
    ep.enc.ex[site * g.Ls + (g.Ls - 1 - s)] = ex;
  }
}

__device__ __forceinline__ int fx_tile_site(const Geom& g, const FxTile& t, int tile, int i) {
  int co[4];
  if (t.b[0] == 0) {
    const int h = tile * t.ns + i;
    if (!t.rb) return h;
    if (h >= g.V4 / 2) return g.V4;
    int r = h / (g.L[0] / 2);
    co[0] = h - r * (g.L[0] / 2);
    co[1] = r % g.L[1];
    r /= g.L[1];
    co[2] = r % g.L[2];
    co[3] = r / g.L[2];
  } else {
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const int q = i / t.b[mu], r = tile / t.n[mu];
      co[mu] = (tile - r * t.n[mu]) * t.b[mu] + (i - q * t.b[mu]);
      i = q;
      tile = r;
    }
  }
  if (t.rb) co[0] = 2 * co[0] + ((t.par + co[1] + co[2] + co[3]) & 1);
  return x4_index(g, co);
}

// entry of the tile's hop table for direction d = 2 mu + (1 for the backward hop):
// the neighbour's x4 Ls, the link's first element, the link's exponent, 1 for a
// factor -1 from the t boundary
__device__ __forceinline__ int4 fx_hop_entry(const Geom& g, const FxLinks& u, int x4, int d) {
  int co[4];
  x4_coords(g, x4, co);
  const int mu = d >> 1;
  int c = 0, L = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (k == mu) {
      c = co[k];
      L = g.L[k];
    }
  const bool wrap = d & 1 ? c == 0 : c + 1 == L;
  const int nc = d & 1 ? (wrap ? L - 1 : c - 1) : (wrap ? 0 : c + 1);
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (k == mu) co[k] = nc;
  const int y4 = x4_index(g, co);
  const int l4 = mu * g.V4 + (d & 1 ? y4 : x4);
  return make_int4(y4 * g.Ls, l4 * 9, u.ex[l4], mu == 3 && wrap && g.bc_t < 0);
}

// the encoded form of r 2^(C - 2102) in a site whose numbers have at least lz leading sign-equal bits
__device__ __forceinline__ int2 fx_renorm(i64 r, int lz) {
  return fx_limbs(lz >= 6 ? r << (lz - 6) : (r + ((1LL << (6 - lz)) >> 1)) >> (6 - lz));
}

// part < 0: the whole site; else direction part's two hops, and with parts 0 and 1 one chirality
// of the fifth-dimension part
template <int LS, int MODE>
__device__ __forceinline__ void fx_site(const Geom& g, const FxParams& p, const FxLinks& u, const FxField& in,
                                        const int4* tab, int x4, int s, int C, i64 (&acc)[4][3][2], unsigned& ok,
                                        int part = -1) {
  const int ls = ls_of<LS>(g);
#pragma unroll
  for (int c = 0; c < 12; ++c) acc[c / 3][c % 3][0] = acc[c / 3][c % 3][1] = 0;
  int top = 0;
#pragma unroll 1
  for (int d = part < 0 ? 0 : 2 * part; d < (part < 0 ? 8 : 2 * part + 2); ++d) {
    const int4 t = tab[d];
    const int sh = min(C - (t.z + __ldg(in.ex + t.x + s)), 61);
    const int4* nb = in.v + (unsigned)(t.x * 12 + s);
    const int4* Ul = u.v + (unsigned)t.y;
    switch (d) {
      case 0: fx_hop<0, 1>(Ul, nb, ls, sh, false, acc, ok, top); break;
      case 1: fx_hop<0, -1>(Ul, nb, ls, sh, false, acc, ok, top); break;
      case 2: fx_hop<1, 1>(Ul, nb, ls, sh, false, acc, ok, top); break;
      case 3: fx_hop<1, -1>(Ul, nb, ls, sh, false, acc, ok, top); break;
      case 4: fx_hop<2, 1>(Ul, nb, ls, sh, false, acc, ok, top); break;
      case 5: fx_hop<2, -1>(Ul, nb, ls, sh, false, acc, ok, top); break;
      case 6: fx_hop<3, 1>(Ul, nb, ls, sh, t.w != 0, acc, ok, top); break;
      default: fx_hop<3, -1>(Ul, nb, ls, sh, t.w != 0, acc, ok, top); break;
    }
  }
  if (top >= FX_HUGE) ok |= FX_ALL + 1;  // (never FX_ALL then)
  if (MODE >= FX_RB) return;
  // diagonal and fifth dimension: the upper spins couple to s - 1, the lower to s + 1
  const int* e = in.ex + x4 * ls;
  const int s0 = min(C - (p.diag.ex + __ldg(e + s)) + 2, 61);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    if (part >= 0 && part != h) continue;
    const bool wall = h == 0 ? s == 0 : s + 1 == ls;
    const int so = h == 0 ? (wall ? ls - 1 : s - 1) : (wall ? 0 : s + 1);
    const FxCoef k = wall ? p.mmf : p.one;
    const int s1 = min(C - (k.ex + __ldg(e + so)) + 2, 61);
    const int4* self = in.v + (unsigned)((x4 * 12 + 6 * h) * ls);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const int4 v = ldi(self + c * ls + s), w = ldi(self + c * ls + so);
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const i64 a = fx_mul(p.diag, i ? v.z : v.x, i ? v.w : v.y, s0), b = fx_mul(k, i ? w.z : w.x, i ? w.w : w.y, s1);
        if (max(abs((int)(a >> 32)), abs((int)(b >> 32))) >= FX_CERTAIN) ok |= 1u << (2 * (6 * h + c) + i);
        acc[2 * h + c / 3][c % 3][i] += a - b;
      }
    }
  }
}

// the exponent C of a site's terms: (D_dwf in)(x4, s) = sum 2^(C - 2102); FX_RAW / 2 or more
// where an operand is not in the format.  ok: every real is certain where all operands are zero
template <int LS, int MODE>
__device__ __forceinline__ int fx_scale(const Geom& g, const FxParams& p, const FxField& in, const int4* tab, int x4,
                                        int s, unsigned& ok) {
  const int ls = ls_of<LS>(g);
  const int* e = in.ex + x4 * ls;
  const int wn = s + 1 == ls, wp = s == 0;
  int C = 0, any = 0;
  if (MODE < FX_RB) {
    const int e0 = __ldg(e + s), en = __ldg(e + (wn ? 0 : s + 1)), ep = __ldg(e + (wp ? ls - 1 : s - 1));
    any = e0 | en | ep;
    C = max(p.diag.ex + e0, max((wn ? p.mmf.ex : p.one.ex) + en, (wp ? p.mmf.ex : p.one.ex) + ep)) - 2;
  }
#pragma unroll
  for (int d = 0; d < 8; ++d) {
    const int ed = __ldg(in.ex + tab[d].x + s);
    any |= ed;
    C = max(C, tab[d].z + ed);
  }
  ok = any == 0 ? FX_ALL : 0;
  return C;
}

// Persistent CTAs over the tiles of all fields; a tile's hop table is built while the
// one before is computed.  16^4 x 16 in 445 us (FP64 multiply-adds: 1.69 ms): it issues in 42 % of the slots
// with the 16 warps an SM that the accumulators allow, the wide multiply-adds (45 clocks of an SM a
// site) being a fifth of its instructions.  128-thread CTAs with 168 registers: 465 us.
template <int LS, int MODE>
__global__ void __launch_bounds__(FX_THREADS, FX_BLOCKS) g5dwf_fx_kernel(Geom g, FxParams p, FxLinks u, FxField in,
                                                                         FxEpilogue ep, FxTile t, int total) {
  __shared__ int4 tabs[2][FX_MAX_SITES * 8];
  __shared__ int sx4[2][FX_MAX_SITES];
  const int ls = ls_of<LS>(g);
  const int site = (int)threadIdx.x / ls, s = (int)threadIdx.x - site * ls;
  auto fill = [&](int tile, int b) {
    if (tile >= total) return;
    const int t4 = tile % t.tiles;
    for (int i = threadIdx.x; i < t.ns * 8; i += blockDim.x) {
      const int x4 = fx_tile_site(g, t, t4, i >> 3);
      if ((i & 7) == 0) sx4[b][i >> 3] = x4;
      if (x4 < g.V4) tabs[b][i] = fx_hop_entry(g, u, x4, i & 7);
    }
  };
  double acc_d[1] = {0.0};
  fill(blockIdx.x, 0);
  __syncthreads();
  int b = 0;
  for (int tile = blockIdx.x; tile < total; tile += gridDim.x, b ^= 1) {
    const int r = tile / t.tiles;
    const bool on = site < t.ns && sx4[b][min(site, t.ns - 1)] < g.V4;
    if (on) {
      const int x4 = sx4[b][site];
      const FxField f = fx_field_r(g, in, r);
      const int4* tab = tabs[b] + site * 8;
      unsigned ok;
      const int C = fx_scale<LS, MODE>(g, p, f, tab, x4, s, ok);
      i64 v[4][3][2];
      if (C < FX_RAW / 2) fx_site<LS, MODE>(g, p, u, f, tab, x4, s, C, v, ok);
      if (C < FX_RAW / 2 && ok == FX_ALL) {
        const i64 o0 = (i64)r * 12 * g.V5 + (unsigned)(x4 * 12 * ls + (ls - 1 - s));  // the R5 reflection
#pragma unroll
        for (int c = MODE < FX_RB ? 6 : 12; c < 12; ++c)
#pragma unroll
          for (int k = 0; k < 2; ++k) v[c / 3][c % 3][k] = -v[c / 3][c % 3][k];  // gamma5
        if (MODE == FX_BOTH) {  // encoded from the integers
          u64 any = 0;
#pragma unroll
          for (int i = 0; i < 24; ++i) {
            const i64 q = v[i / 6][i / 2 % 3][i % 2];
            any |= (u64)(q ^ (q >> 63));
          }
          const int lz = any ? __clzll((i64)any) : 64;
          int ex = lz == 64 ? 0 : C - lz - 1016;
          if (lz < 64 && (ex < FX_SITE_MIN || ex > FX_SITE_MAX)) ex = FX_RAW;
#pragma unroll
          for (int c = 0; c < 12; ++c) {
            const i64 re = v[c / 3][c % 3][0], im = v[c / 3][c % 3][1];
            int4 q = make_int4(0, 0, 0, 0);
            if (ex != 0 && ex != FX_RAW) {
              const int2 a = fx_renorm(re, lz), d = fx_renorm(im, lz);
              q = make_int4(a.x, a.y, d.x, d.y);
            }
            ep.enc.v[o0 + c * ls] = q;
          }
          ep.enc.ex[(i64)r * g.V5 + x4 * ls + (ls - 1 - s)] = ex;
        }
        if (MODE >= FX_RB) {
          cpx<double> w[12];
#pragma unroll
          for (int c = 0; c < 12; ++c)
            w[c] = cpx<double>(fx_to_double(v[c / 3][c % 3][0], C - 1016), fx_to_double(v[c / 3][c % 3][1], C - 1016));
          fx_rb_output<MODE>(g, ep, ls, x4, s, w, acc_d[0]);
        } else {
          cpx<double> w[12];
#pragma unroll
          for (int c = 0; c < 12; ++c)
            w[c] = fx_epilogue<MODE>(ep, o0 + c * ls, cpx<double>(fx_to_double(v[c / 3][c % 3][0], C - 1016),
                                                                  fx_to_double(v[c / 3][c % 3][1], C - 1016)),
                                     acc_d[0]);
          if ((MODE == FX_RES || MODE == FX_CHEB || MODE == FX_CHEB1 || MODE == FX_CHEBL) && ep.enc.v) {
            const int ex = fx_mark(fx_top(w), FX_SITE_MIN, FX_SITE_MAX);
#pragma unroll
            for (int c = 0; c < 12; ++c) ep.enc.v[o0 + c * ls] = fx_encode(w[c], ex, FX_UP);
            ep.enc.ex[(i64)r * g.V5 + x4 * ls + (ls - 1 - s)] = ex;
          }
        }
      } else {
        fx_slow_output<MODE>(g, p, u, f, ep, tab, r, x4, s, acc_d[0]);
      }
    }
    fill(tile + gridDim.x, b ^ 1);
    __syncthreads();
  }
  if (fx_reduces(MODE) && ep.result) {
    double tot[1];
    if (grid_reduce<1>(acc_d, ep.rs, tot)) *ep.result = tot[0];
  }
}

// The same for launches that would leave most of the chip idle: the four directions of a site go
// to the four warps of a CTA, whose sums (exact, so in any order) meet in shared memory, and each
// warp finishes a quarter of the components.  A thread's chain is a quarter as long.
template <int LS, int MODE>
__global__ void __launch_bounds__(4 * FX_SPLIT_SITES, 4) g5dwf_fx_split_kernel(Geom g, FxParams p, FxLinks u, FxField in,
                                                                              FxEpilogue ep, FxTile t, int total) {
  __shared__ int4 tabs[FX_SPLIT_SITES / 2 * 8];
  __shared__ int sx4[FX_SPLIT_SITES / 2];
  __shared__ i64 sum[24][4][FX_SPLIT_SITES];
  __shared__ unsigned oks[4][FX_SPLIT_SITES];
  const int ls = ls_of<LS>(g);
  const int part = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int site = lane / ls, s = lane - site * ls;
  double acc_d[1] = {0.0};
  for (int tile = blockIdx.x; tile < total; tile += gridDim.x) {
    const int r = tile / t.tiles, t4 = tile - r * t.tiles;
    for (int i = threadIdx.x; i < t.ns * 8; i += blockDim.x) {
      const int x4 = fx_tile_site(g, t, t4, i >> 3);
      if ((i & 7) == 0) sx4[i >> 3] = x4;
      if (x4 < g.V4) tabs[i] = fx_hop_entry(g, u, x4, i & 7);
    }
    __syncthreads();
    const int x4 = site < t.ns ? sx4[site] : g.V4;
    const bool on = x4 < g.V4;
    const FxField f = fx_field_r(g, in, r);
    int C = FX_RAW;
    unsigned ok = 0;
    if (on) C = fx_scale<LS, MODE>(g, p, f, tabs + site * 8, x4, s, ok);
    bool fx = C < FX_RAW / 2;
    if (fx) {
      i64 v[4][3][2];
      fx_site<LS, MODE>(g, p, u, f, tabs + site * 8, x4, s, C, v, ok, part);
#pragma unroll
      for (int i = 0; i < 24; ++i) sum[i][part][lane] = v[i / 6][i / 2 % 3][i % 2];
    }
    oks[part][lane] = ok;
    __syncthreads();
    fx = fx && (oks[0][lane] | oks[1][lane] | oks[2][lane] | oks[3][lane]) == FX_ALL;
    if (fx) {
      const i64 o0 = (i64)r * 12 * g.V5 + (unsigned)(x4 * 12 * ls + (ls - 1 - s));  // the R5 reflection
#pragma unroll
      for (int j = 0; j < 3; ++j) {
        const int c = 3 * part + j;
        i64 v[2] = {0, 0};
#pragma unroll
        for (int k = 0; k < 2; ++k) {
#pragma unroll
          for (int q = 0; q < 4; ++q) v[k] += sum[2 * c + k][q][lane];
          if (part >= 2) v[k] = -v[k];  // gamma5
        }
        fx_epilogue<MODE>(ep, o0 + c * ls, cpx<double>(fx_to_double(v[0], C - 1016), fx_to_double(v[1], C - 1016)),
                          acc_d[0]);
      }
    } else if (on && part == 0) {
      fx_slow_output<MODE>(g, p, u, f, ep, tabs + site * 8, r, x4, s, acc_d[0]);
    }
    __syncthreads();
  }
  if (fx_reduces(MODE)) {
    double tot[1];
    if (grid_reduce<1>(acc_d, ep.rs, tot)) *ep.result = tot[0];
  }
}

// ---------------------------------------------------------------------- host
static size_t up16(size_t b) { return (b + 15) & ~(size_t)15; }

size_t fx_links_bytes(const Geom& g) { return (size_t)g.V4 * 36 * 16 + up16((size_t)g.V4 * 4 * 4); }
size_t fx_field_bytes(const Geom& g, int nrhs) {
  return (size_t)g.V5 * nrhs * 12 * 16 + up16((size_t)g.V5 * nrhs * 4);
}
FxLinks fx_links_at(const Geom& g, void* mem) {
  FxLinks u;
  u.v = (int4*)mem;
  u.ex = (int*)(u.v + (size_t)g.V4 * 36);
  return u;
}
FxField fx_field_at(const Geom& g, int nrhs, void* mem) {
  FxField f;
  f.v = (int4*)mem;
  f.ex = (int*)(f.v + (size_t)g.V5 * nrhs * 12);
  return f;
}

static FxCoef fx_coef(double x) {
  FxCoef k{0, 0, 0, x};
  if (x == 0.0) return k;
  int e = 0;
  const double m = frexp(x, &e);  // 0.5 <= |m| < 1, x = m 2^e: biased exponent e + 1022
  if (!(fabs(m) < 1.0) || e + 1022 < FX_LINK_MIN || e + 1022 > FX_LINK_MAX) {
    k.ex = FX_RAW;
    return k;
  }
  const double y = ldexp(m, 30);
  k.h = (int)rint(y);
  k.l = (int)ldexp(y - k.h, 30);  // (53 bits of m below 2^30: exact)
  k.ex = e + 1022;
  return k;
}

static FxParams fx_params(double M5, double mf) { return FxParams{fx_coef(5.0 - M5), fx_coef(1.0), fx_coef(-mf)}; }

int launch_fx_encode(const Geom& g, const cpx<double>* in, int nrhs, const FxField& f, const cpx<double>* U,
                     const FxLinks& u, cudaStream_t st) {
  const i64 nsites = in ? g.V5 * nrhs : 0, nlinks = U ? (i64)g.V4 * 4 : 0;
  const i64 fb = (nsites + 127) / 128, lb = (nlinks + 127) / 128;
  if (fb + lb == 0) return HDCR_OK;
  fx_encode_kernel<<<(unsigned)(fb + lb), 128, 0, st>>>(g.Ls, nsites, in, f, (int)fb, nlinks, U, u);
  count_launch();
  HDCR_LAUNCH_CHECK();
  return HDCR_OK;
}

bool fx_ok(const Geom& g) { return g.Ls <= FX_THREADS; }

// The tile with the fewest spinors read per 4d site (itself and the neighbours outside)
// among the boxes that divide the lattice and fill the CTA's warps, or consecutive
// sites when no box does better; smaller tiles when there would be less than two per SM.
static FxTile fx_tile(const Geom& full, int nrhs, bool rb, int threads) {
  Geom g = full;
  if (rb) {
    g.L[0] /= 2;
    g.V4 /= 2;
  }
  int most = threads / g.Ls;
  while (threads == FX_THREADS && most > 1 && most * g.Ls > 32 && (i64)g.V4 * nrhs / most < 304) most = (most + 1) / 2;
  if (most > g.V4) most = g.V4;
  auto cost = [&](int ns, double reads) {
    const int lanes = (ns * g.Ls + 31) / 32 * 32;
    return (1.0 + 0.1 * reads) * lanes / (ns * g.Ls);
  };
  FxTile t{rb, 0, {0, 0, 0, 0}, {0, 0, 0, 0}, most, (g.V4 + most - 1) / most};
  const int row = most < g.L[0] ? most : g.L[0];
  double best = cost(most, 1.0 + 2.0 / row + (row < most ? 4.0 + 2.0 * row / most : 6.0));
  for (int b3 = 1; b3 <= most && b3 <= g.L[3]; ++b3) {
    if (g.L[3] % b3) continue;
    for (int b2 = 1; b3 * b2 <= most && b2 <= g.L[2]; ++b2) {
      if (g.L[2] % b2) continue;
      for (int b1 = 1; b3 * b2 * b1 <= most && b1 <= g.L[1]; ++b1) {
        if (g.L[1] % b1) continue;
        for (int b0 = 1; b3 * b2 * b1 * b0 <= most && b0 <= g.L[0]; ++b0) {
          if (g.L[0] % b0) continue;
          const int b[4] = {b0, b1, b2, b3};
          double reads = 1.0;
          for (int mu = 0; mu < 4; ++mu) reads += b[mu] == g.L[mu] ? 0.0 : 2.0 / b[mu];
          if (cost(b0 * b1 * b2 * b3, reads) >= best) continue;
          best = cost(b0 * b1 * b2 * b3, reads);
          t.ns = b0 * b1 * b2 * b3;
          t.tiles = g.V4 / t.ns;
          for (int mu = 0; mu < 4; ++mu) {
            t.b[mu] = b[mu];
            t.n[mu] = g.L[mu] / b[mu];
          }
        }
      }
    }
  }
  return t;
}

template <int MODE>
static int fx_launch(const Geom& g, double M5, double mf, const FxLinks& u, const FxField& in, const FxEpilogue& ep,
                     int nrhs, cudaStream_t st, int par = 0) {
  const FxParams p = fx_params(M5, mf);
  int sms = 0, dev = 0;
  HDCR_CUDA_TRY(cudaGetDevice(&dev));
  HDCR_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  if constexpr (MODE == FX_OUT || MODE == FX_DOT) {
    if (g.Ls <= FX_SPLIT_SITES && g.V5 * nrhs <= FX_SPLIT_MAX) {
      const FxTile t = fx_tile(g, nrhs, false, FX_SPLIT_SITES);
      const int total = t.tiles * nrhs, most = sms * 4;
      HDCR_DISPATCH_LS(g.Ls, (g5dwf_fx_split_kernel<LSC, MODE><<<total < most ? total : most, 4 * FX_SPLIT_SITES, 0, st>>>(
                                 g, p, u, in, ep, t, total)));
      HDCR_LAUNCH_CHECK();
      return HDCR_OK;
    }
  }
  FxTile t = fx_tile(g, nrhs, MODE >= FX_RB, FX_THREADS);
  t.par = par;
  const int total = t.tiles * nrhs;
  const int threads = (t.ns * g.Ls + 31) / 32 * 32;
  const int fit = sms * (FX_BLOCKS * FX_THREADS / threads);  // CTAs resident at once
  const int most = fit < RED_MAX_BLOCKS ? fit : RED_MAX_BLOCKS;
  const int grid = total < most ? total : most;
  HDCR_DISPATCH_LS(g.Ls, (g5dwf_fx_kernel<LSC, MODE><<<grid, threads, 0, st>>>(g, p, u, in, ep, t, total)));
  HDCR_LAUNCH_CHECK();
  return HDCR_OK;
}

int launch_fx_g5dwf(const Geom& g, double M5, double mf, const FxLinks& u, const FxField& in, cpx<double>* out,
                    int nrhs, cudaStream_t st, const FxField* enc) {
  FxEpilogue ep{};
  ep.out = out;
  if (enc) ep.enc = *enc;
  if (enc) return fx_launch<FX_BOTH>(g, M5, mf, u, in, ep, nrhs, st);
  return fx_launch<FX_OUT>(g, M5, mf, u, in, ep, nrhs, st);
}

int launch_fx_rb_hop(const Geom& g, const FxLinks& u, const FxField& in, cpx<double>* out, int par, cudaStream_t st) {
  FxEpilogue ep{};
  ep.out = out;
  return fx_launch<FX_RB>(g, 0.0, 0.0, u, in, ep, 1, st, par);
}

int launch_fx_rb_schur(const Geom& g, double diag, double mf, const FxLinks& u, const FxField& in,
                       const cpx<double>* src, cpx<double>* out, bool dag, const FxField& enc, cpx<double>* g5,
                       RedScratch rs, double* norm2, int par, cudaStream_t st) {
  FxEpilogue ep{};
  ep.src = src;
  ep.out = out;
  ep.enc = enc;
  ep.prev = g5;
  ep.a = diag;
  ep.c0 = mf;
  ep.dag = dag;
  ep.rs = rs;
  ep.result = dag ? nullptr : norm2;
  return fx_launch<FX_RBS>(g, 0.0, 0.0, u, in, ep, 1, st, par);
}

// M5^{-1} on the sites of one parity (rbcg.cu describes it), the result encoded: a CTA's rows
// over s are brought into shared memory in runs, each is substituted by one thread, and a site's
// 12 rows are encoded together.  FP64 substitution, 3 FP64 instructions a real.
__global__ void __launch_bounds__(128) fx_rb_m5inv_kernel(Geom g, int ns, const cpx<double>* __restrict__ in,
                                                          cpx<double>* __restrict__ out64, FxField out, int par,
                                                          double a, double mf) {
  extern __shared__ cpx<double> rows[];  // [ns * 12][Ls + 1]
  __shared__ int sx4[64];
  const int ls = g.Ls, pitch = ls + 1, half = g.V4 / 2;
  FxTile t{1, par, {0, 0, 0, 0}, {0, 0, 0, 0}, ns, 0};
  if ((int)threadIdx.x < ns) sx4[threadIdx.x] = fx_tile_site(g, t, blockIdx.x, threadIdx.x);
  __syncthreads();
  const int n = min(ns, half - (int)blockIdx.x * ns);  // sites here
  for (int i = threadIdx.x; i < n * 12 * ls; i += blockDim.x) {
    const int row = i / ls, s = i - row * ls;
    rows[row * pitch + s] = in[(unsigned)((sx4[row / 12] * 12 + row % 12) * ls + s)];
  }
  __syncthreads();
  const double ia = 1.0 / a;
  double aLs = 1.0;  // a^{-Ls}
  for (int s = 0; s < ls; ++s) aLs *= ia;
  const double f = mf / (1.0 + mf * aLs);
  for (int row = threadIdx.x; row < n * 12; row += blockDim.x) {
    cpx<double>* y = rows + row * pitch;
    const bool upper = row % 12 < 6;  // substitution from s = 0 up, else from Ls - 1 down
    const int s0 = upper ? 0 : ls - 1, d = upper ? 1 : -1;
    cpx<double> z(0.0, 0.0);
    for (int k = 0, s = s0; k < ls; ++k, s += d) {
      z = cpx<double>(ia * (y[s].re + z.re), ia * (y[s].im + z.im));
      y[s] = z;
    }
    const cpx<double> gam = f * z;
    double w = ia;
    for (int k = 0, s = s0; k < ls; ++k, s += d) {
      y[s] = cpx<double>(fma(-w, gam.re, y[s].re), fma(-w, gam.im, y[s].im));
      w *= ia;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n * ls; i += blockDim.x) {
    const int site = i / ls, s = i - site * ls;
    cpx<double> x[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) x[c] = rows[(site * 12 + c) * pitch + s];
    const int ex = fx_mark(fx_top(x), FX_SITE_MIN, FX_SITE_MAX);
#pragma unroll
    for (int c = 0; c < 12; ++c) {
      const unsigned o = (unsigned)((sx4[site] * 12 + c) * ls + s);
      out.v[o] = fx_encode(x[c], ex, FX_UP);
      st(out64 + o, x[c]);
    }
    out.ex[sx4[site] * ls + s] = ex;
  }
}

int launch_fx_rb_m5inv(const Geom& g, const cpx<double>* in, cpx<double>* out64, const FxField& out, int par,
                       double a, double mf, cudaStream_t st) {
  int ns = 128 / g.Ls;
  ns = ns < 1 ? 1 : ns > 32 ? 32 : ns;
  const size_t smem = sizeof(cpx<double>) * (size_t)ns * 12 * (g.Ls + 1);
  HDCR_CUDA_TRY(cudaFuncSetAttribute(fx_rb_m5inv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  fx_rb_m5inv_kernel<<<(g.V4 / 2 + ns - 1) / ns, 128, smem, st>>>(g, ns, in, out64, out, par, a, mf);
  count_launch();
  HDCR_LAUNCH_CHECK();
  return HDCR_OK;
}

// p <- r + beta p on the sites of one parity (beta = rr[k ^ 1] / rr[k], 0 where rr[k] is 0), encoded;
// r null: p as it is
__global__ void __launch_bounds__(128) fx_rb_p_kernel(Geom g, const cpx<double>* __restrict__ r, cpx<double>* __restrict__ p,
                                                      FxField out, int par, const double* rr, int k) {
  const int ls = g.Ls;
  const i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.V5 / 2) return;
  const int h = (int)(i / ls), s = (int)(i - (i64)h * ls);
  const FxTile t{1, par, {0, 0, 0, 0}, {0, 0, 0, 0}, 1, 0};
  const int x4 = fx_tile_site(g, t, h, 0);
  const double beta = r && rr[k] > 0.0 ? rr[k ^ 1] / rr[k] : 0.0;
  cpx<double> x[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    const unsigned o = (unsigned)((x4 * 12 + c) * ls + s);
    x[c] = p[o];
    if (r) {
      const cpx<double> v = r[o];
      x[c] = cpx<double>(fma(beta, x[c].re, v.re), fma(beta, x[c].im, v.im));
      p[o] = x[c];
    }
  }
  const int ex = fx_mark(fx_top(x), FX_SITE_MIN, FX_SITE_MAX);
#pragma unroll
  for (int c = 0; c < 12; ++c) out.v[(unsigned)((x4 * 12 + c) * ls + s)] = fx_encode(x[c], ex, FX_UP);
  out.ex[x4 * ls + s] = ex;
}

int launch_fx_rb_p(const Geom& g, const cpx<double>* r, cpx<double>* p, const FxField& out, int par, const double* rr,
                   int k, cudaStream_t st) {
  fx_rb_p_kernel<<<num_blocks(g.V5 / 2, 128), 128, 0, st>>>(g, r, p, out, par, rr, k);
  count_launch();
  HDCR_LAUNCH_CHECK();
  return HDCR_OK;
}

int launch_fx_g5dwf_res(const Geom& g, double M5, double mf, const FxLinks& u, const FxField& in,
                        const cpx<double>* src, cpx<double>* out, const FxField* enc, int nrhs, cudaStream_t st) {
  FxEpilogue ep{};
  ep.src = src;
  ep.out = out;
  if (enc) ep.enc = *enc;
  return fx_launch<FX_RES>(g, M5, mf, u, in, ep, nrhs, st);
}

int launch_fx_g5dwf_cheb(const Geom& g, double M5, double mf, const FxLinks& u, const FxField& in, const FxChebStep& c,
                         const FxField& enc, int nrhs, cudaStream_t st) {
  FxEpilogue ep{};
  ep.enc = enc;
  ep.cur = c.cur;
  ep.prev = c.prev;
  ep.acc = c.acc;
  ep.a = c.a;
  ep.b = c.b;
  ep.ck = c.ck;
  ep.c0 = c.c0;
  if (c.first) return fx_launch<FX_CHEB1>(g, M5, mf, u, in, ep, nrhs, st);
  if (c.last) return fx_launch<FX_CHEBL>(g, M5, mf, u, in, ep, nrhs, st);
  return fx_launch<FX_CHEB>(g, M5, mf, u, in, ep, nrhs, st);
}

int launch_fx_g5dwf_dot(const Geom& g, double M5, double mf, const FxLinks& u, const FxField& in, cpx<double>* out,
                        RedScratch rs, double* result, cudaStream_t st) {
  FxEpilogue ep{};
  ep.out = out;
  ep.src = in.f64;
  ep.rs = rs;
  ep.result = result;
  return fx_launch<FX_DOT>(g, M5, mf, u, in, ep, 1, st);
}

size_t fx_scratch_bytes(const Geom& g, int nrhs) { return fx_links_bytes(g) + fx_field_bytes(g, nrhs); }

bool fx_apply_fits(const Geom& g, const void* scratch, size_t bytes) {
  return fx_ok(g) && scratch && ((uintptr_t)scratch & 15) == 0 && bytes >= fx_scratch_bytes(g, 1);
}

int launch_fx_apply(const Geom& g, double M5, double mf, const cpx<double>* U, const cpx<double>* in,
                    cpx<double>* out, int nrhs, void* scratch, size_t bytes, cudaStream_t st) {
  int fit = nrhs;
  while (fit > 1 && fx_scratch_bytes(g, fit) > bytes) --fit;
  FxLinks u = fx_links_at(g, scratch);
  u.f64 = U;
  for (int r = 0; r < nrhs; r += fit) {
    const int m = nrhs - r < fit ? nrhs - r : fit;
    const i64 o = (i64)r * 12 * g.V5;
    const FxField f = fx_of(fx_field_at(g, m, (char*)scratch + fx_links_bytes(g)), in + o);
    HDCR_TRY(launch_fx_encode(g, in + o, m, f, r == 0 ? U : nullptr, u, st));
    HDCR_TRY(launch_fx_g5dwf(g, M5, mf, u, f, out + o, m, st));
  }
  return HDCR_OK;
}

void fx_ctx_alloc(FxCtx* c, const Geom& g, int nrhs, int vectors) {
  *c = FxCtx();
  if (!fx_ok(g)) return;
  const size_t lb = fx_links_bytes(g), fb = fx_field_bytes(g, nrhs);
  if (dev_malloc(&c->mem, lb + vectors * fb) != cudaSuccess) {
    cudaGetLastError();
    c->mem = nullptr;
    return;
  }
  c->u = fx_links_at(g, c->mem);
  c->e0 = fx_field_at(g, nrhs, (char*)c->mem + lb);
  if (vectors > 1) c->e1 = fx_field_at(g, nrhs, (char*)c->mem + lb + fb);
}

void fx_ctx_free(FxCtx* c) {
  if (c->mem) cudaFree(c->mem);
  *c = FxCtx();
}

int fx_ctx_links(FxCtx& c, const Geom& g, const cpx<double>* U, cudaStream_t st) {
  c.u.f64 = U;
  return c.mem ? launch_fx_encode(g, nullptr, 0, c.e0, U, c.u, st) : HDCR_OK;
}

int fx_ctx_apply(const FxCtx& c, const Geom& g, double M5, double mf, const cpx<double>* in, cpx<double>* out, int nrhs,
                 cudaStream_t st) {
  int slot;
  stencil_timer_begin(0, g.V5 * nrhs, st, &slot);
  int s = launch_fx_encode(g, in, nrhs, c.e0, nullptr, c.u, st);
  if (s == HDCR_OK) s = launch_fx_g5dwf(g, M5, mf, c.u, fx_of(c.e0, in), out, nrhs, st);
  stencil_timer_end(slot, st);
  return s;
}

int fx_ctx_apply_dot(const FxCtx& c, const Geom& g, double M5, double mf, const cpx<double>* in, cpx<double>* out,
                     RedScratch rs, double* result, cudaStream_t st) {
  int slot;
  stencil_timer_begin(0, g.V5, st, &slot);
  int s = launch_fx_encode(g, in, 1, c.e0, nullptr, c.u, st);
  if (s == HDCR_OK) s = launch_fx_g5dwf_dot(g, M5, mf, c.u, fx_of(c.e0, in), out, rs, result, st);
  stencil_timer_end(slot, st);
  return s;
}

}  // namespace hdcr
