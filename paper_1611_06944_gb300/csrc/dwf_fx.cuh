// FP64 stencil without the FP64 pipe: fields and links in fixed point, a wide integer
// limb and an FP32 rest.
//
// This chip issues 2 FP64 multiply-adds per clock and SM, 32 wide integer ones
// (32 x 32 + 64 -> 64) and 128 FP32 ones.  The operator reads its FP64 operands encoded once per
// application as
//
//     x = (H + l) 2^(ex - 1051),  H a 32-bit integer, |H| <= 2^29, l an FP32 number, |l| <= 1/2,
//
// with one exponent ex (the biased FP64 exponent of the largest component) per 5d
// site of a field, and per link (|H| <= 2^30, ex - 1052).  H and l together hold 54 bits below the
// largest component of a site, and a component near it exactly.  A product is H H' summed
// exactly in 64 bits over a hop, one wide multiply-add, and H l' + l H' in FP32, two FP32
// multiply-adds (l l' is below 2^-60 of the scale): 1/32 + 2/128 of a clock where an FP64
// multiply-add takes 1/2.  A hop is rounded to the site's common exponent, 2^-57 of the result,
// and the nine terms of a site are summed exactly.  Against 80-bit arithmetic the result is
// off by 1.1e-16 (2-norm; the largest component 0.4e-15 to 1.0e-15 of the root mean square), the FP64
// kernel, which rounds at every step, by 1.5e-16 (0.9e-15 to 2.1e-15), on Gaussian fields
// and on fields that decay into the fifth dimension.
//
// A complex number takes 16 bytes (re.H, re.l, im.H, im.l) in the field layout, as in FP64.
// A site or link that the format cannot hold (infinities, NaN, largest components below
// 2^-623 or above 2^577; links outside 2^-150 .. 2^150) is stored as its FP64 bits
// with the exponent FX_RAW; a site that reads one of them is computed in FP64.
#pragma once

#include "blas.cuh"

namespace hdcr {

constexpr int FX_RAW = 1 << 28;       // exponent mark: the words are FP64 bits
constexpr int FX_SITE_MIN = 400, FX_SITE_MAX = 1600;  // biased exponents a field's site may have
constexpr int FX_LINK_MIN = 873, FX_LINK_MAX = 1173;  // and a link (or a coefficient)

struct FxField {
  int4* v = nullptr;   // [nrhs][V4][12][Ls]
  int* ex = nullptr;   // [nrhs][V5]
};
struct FxLinks {
  int4* v = nullptr;   // [4][V4][9]
  int* ex = nullptr;   // [4][V4]
};

// bytes of the encoded links, and of nrhs encoded fields
size_t fx_links_bytes(const Geom& g);
size_t fx_field_bytes(const Geom& g, int nrhs);
// carves them out of device memory aligned to 16 bytes
FxLinks fx_links_at(const Geom& g, void* mem);
FxField fx_field_at(const Geom& g, int nrhs, void* mem);

// f <- in (nrhs FP64 fields; in may be null: nothing) and u <- U (U may be null: nothing), one launch
int launch_fx_encode(const Geom& g, const cpx<double>* in, int nrhs, const FxField& f, const cpx<double>* U,
                     const FxLinks& u, cudaStream_t st);
// bytes of scratch that nrhs fields of one application take
size_t fx_scratch_bytes(const Geom& g, int nrhs);
// whether ``bytes`` at ``scratch`` hold at least one field's application
bool fx_apply_fits(const Geom& g, const void* scratch, size_t bytes);
// out = H in for nrhs FP64 fields, as many at a time as the scratch holds
int launch_fx_apply(const Geom& g, double M5, double mf, const cpx<double>* U, const cpx<double>* in,
                    cpx<double>* out, int nrhs, void* scratch, size_t bytes, cudaStream_t st);
// whether the integer kernel takes the geometry (Ls <= 128)
bool fx_ok(const Geom& g);
// out = H in, and H in encoded into *enc when enc is set; out may be null (enc alone)
int launch_fx_g5dwf(const Geom& g, double M5, double mf, const FxLinks& u, const FxField& in, cpx<double>* out,
                    int nrhs, cudaStream_t st, const FxField* enc = nullptr);
// out = src - H in, also encoded into *enc when enc is set
int launch_fx_g5dwf_res(const Geom& g, double M5, double mf, const FxLinks& u, const FxField& in,
                        const cpx<double>* src, cpx<double>* out, const FxField* enc, int nrhs, cudaStream_t st);
// One step of the Chebyshev smoother's recurrence on t(y) = a y + b, y = H^2, with in = H cur:
// the term nx = 2 (a H in + b cur) - prev written over prev, acc += ck nx, nx encoded into enc.
// first: nx = a H in + b cur, acc = c0 cur + ck nx.  last: only acc, which is encoded into enc.
// acc may be null (a filter's step).
struct FxChebStep {
  const cpx<double>* cur;
  cpx<double>* prev;
  cpx<double>* acc;
  double a, b, ck, c0;
  bool first, last;
};
int launch_fx_g5dwf_cheb(const Geom& g, double M5, double mf, const FxLinks& u, const FxField& in, const FxChebStep& c,
                         const FxField& enc, int nrhs, cudaStream_t st);
// out = H in and Re <in, out> into *result; in64 is the field that in encodes
int launch_fx_g5dwf_dot(const Geom& g, double M5, double mf, const FxLinks& u, const FxField& in,
                        const cpx<double>* in64, cpx<double>* out, RedScratch rs, double* result, cudaStream_t st);

// Red-black pieces on the sites of parity par (every extent even; 4d sites of the other
// parity are read).  hop: out = D_hop in.  schur, with in = M5^{-1} D_hop v encoded:
// w = M5 v - D_hop in; out = w, |w|^2 into *norm2 and Gamma5 w encoded into enc, or with dag
// v = Gamma5 src and out = Gamma5 w (norm2 and enc unused).  m5inv: M5^{-1} in, encoded.
// p: p <- r + (rr[k ^ 1] / rr[k]) p (r null: p unchanged), p encoded.
int launch_fx_rb_hop(const Geom& g, const FxLinks& u, const FxField& in, cpx<double>* out, int par, cudaStream_t st);
int launch_fx_rb_schur(const Geom& g, double diag, double mf, const FxLinks& u, const FxField& in,
                       const cpx<double>* src, cpx<double>* out, bool dag, const FxField& enc, RedScratch rs,
                       double* norm2, int par, cudaStream_t st);
int launch_fx_rb_m5inv(const Geom& g, const cpx<double>* in, const FxField& out, int par, double a, double mf,
                       cudaStream_t st);
int launch_fx_rb_p(const Geom& g, const cpx<double>* r, cpx<double>* p, const FxField& out, int par, const double* rr,
                   int k, cudaStream_t st);

// What a solver keeps for FP64 applications of H on nrhs fields: the encoded links and two
// encoded field vectors.  Without memory for it mem stays null and H runs on the FP64 pipe.
struct FxCtx {
  void* mem = nullptr;
  FxLinks u;
  FxField e0, e1;
};
// allocates (leaving mem null when the device is out of memory or fx_ok is false)
void fx_ctx_alloc(FxCtx* c, const Geom& g, int nrhs);
void fx_ctx_free(FxCtx* c);
// encodes U: before the first application of a solve
int fx_ctx_links(const FxCtx& c, const Geom& g, const cpx<double>* U, cudaStream_t st);
// out = H in through e0, timed as one FP64 application
int fx_ctx_apply(const FxCtx& c, const Geom& g, double M5, double mf, const cpx<double>* in, cpx<double>* out, int nrhs,
                 cudaStream_t st);
int fx_ctx_apply_dot(const FxCtx& c, const Geom& g, double M5, double mf, const cpx<double>* in, cpx<double>* out,
                     RedScratch rs, double* result, cudaStream_t st);

}  // namespace hdcr
