// FP64 stencil without the FP64 pipe: fields and links in fixed point, two integer limbs.
//
// This chip issues 2 FP64 multiply-adds per clock and SM, 32 wide integer ones
// (32 x 32 + 64 -> 64).  The operator reads its FP64 operands encoded once per application as
//
//     x = (H + L / 2^30) 2^(ex - 1050),  |H| <= 2^28, -2^29 <= L < 2^29,
//
// with one exponent ex (the biased FP64 exponent of the largest component) per 5d
// site of a field, and per link (|H| <= 2^29, ex - 1051): 58 bits below the largest component
// of a site.  A complex product is three real ones, each H H' + (H L' + L H') / 2^30 in
// three wide multiply-adds that are summed exactly over a hop (the dropped L L' is below 2^-57 of the
// scale): 9/32 of a clock where four FP64 multiply-adds take 2 clocks.  A hop is rounded to the
// site's common exponent, and the terms of a site are summed exactly.
//
// Components of a site may differ in size, and links need not mix them.  What FP64 multiply-adds
// lose on a component is 2^-53 of that component's own terms, so the kernel notes for each real of
// a site whether one of its terms is large enough for the integers to be as good (2^52 of their
// unit, about a quarter of a typical term; dwf_fx.cu).  A site with a real that is not certain in
// this way is computed in FP64 from the numbers themselves, which every operand keeps beside its encoded
// form (f64).  So are sites that read an operand outside the format (infinities, NaN, largest
// components below 2^-623 or above 2^577; links outside 2^-150 .. 2^150), whose exponent is FX_RAW.
// Of Gaussian or wall-bound fields on links that mix the colours fewer than one site in a million
// goes that way, of plain CR's vectors one in 70,000, around a point source more; where links mix nothing
// and components differ by a factor of ten, all do: 2.4 ms at 16^4 x 16.
//
// Against 80-bit arithmetic the result is off by 5e-17 (2-norm) and the FP64 kernel's by 1.5e-16 on Gaussian
// fields and on fields that decay into the fifth dimension; where components differ in size the error
// of each, relative to itself, is at most the FP64 kernel's.
// At 16^4 x 16 an application takes 0.52 ms with the encoding, the FP64 kernel 1.69 ms (an FP32
// low limb took 0.42 ms, but its products held only 54 bits below the site's largest component).
//
// A complex number takes 16 bytes (re.H, re.L, im.H, im.L) in the field layout, as in FP64.
#pragma once

#include "blas.cuh"

namespace hdcr {

constexpr int FX_RAW = 1 << 28;       // exponent mark: outside the format, the words are zero
constexpr int FX_SITE_MIN = 400, FX_SITE_MAX = 1600;  // biased exponents a field's site may have
constexpr int FX_LINK_MIN = 873, FX_LINK_MAX = 1173;  // and a link (or a coefficient)

struct FxField {
  int4* v = nullptr;   // [nrhs][V4][12][Ls]
  int* ex = nullptr;   // [nrhs][V5]
  const cpx<double>* f64 = nullptr;  // the numbers themselves: an operand must have them
};
struct FxLinks {
  int4* v = nullptr;   // [4][V4][9]
  int* ex = nullptr;   // [4][V4]
  const cpx<double>* f64 = nullptr;
};
// the encoded form f of the numbers at v
inline FxField fx_of(FxField f, const cpx<double>* v) {
  f.f64 = v;
  return f;
}

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
// whether the integer kernel takes the geometry (Ls <= 256)
bool fx_ok(const Geom& g);
// out = H in, and H in encoded into *enc when enc is set
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
// out = H in and Re <in, out> into *result
int launch_fx_g5dwf_dot(const Geom& g, double M5, double mf, const FxLinks& u, const FxField& in, cpx<double>* out,
                        RedScratch rs, double* result, cudaStream_t st);

// Red-black pieces on the sites of parity par (every extent even; 4d sites of the other
// parity are read).  hop: out = D_hop in.  schur, with in = M5^{-1} D_hop v encoded:
// w = M5 v - D_hop in; out = w, |w|^2 into *norm2 and Gamma5 w encoded into enc and written to g5, or
// with dag v = Gamma5 src and out = Gamma5 w (norm2, enc and g5 unused).  m5inv: out64 = M5^{-1} in,
// encoded into out.
// p: p <- r + (rr[k ^ 1] / rr[k]) p (r null: p unchanged), p encoded.
int launch_fx_rb_hop(const Geom& g, const FxLinks& u, const FxField& in, cpx<double>* out, int par, cudaStream_t st);
int launch_fx_rb_schur(const Geom& g, double diag, double mf, const FxLinks& u, const FxField& in,
                       const cpx<double>* src, cpx<double>* out, bool dag, const FxField& enc, cpx<double>* g5,
                       RedScratch rs, double* norm2, int par, cudaStream_t st);
int launch_fx_rb_m5inv(const Geom& g, const cpx<double>* in, cpx<double>* out64, const FxField& out, int par, double a, double mf,
                       cudaStream_t st);
int launch_fx_rb_p(const Geom& g, const cpx<double>* r, cpx<double>* p, const FxField& out, int par, const double* rr,
                   int k, cudaStream_t st);

// What a solver keeps for FP64 applications of H on nrhs fields: the encoded links, an encoded field
// vector and, where encoded fields pass from one application to the next, a second one.  Without
// memory for it mem stays null and H runs on the FP64 pipe.
struct FxCtx {
  void* mem = nullptr;
  FxLinks u;
  FxField e0, e1;
};
// allocates ``vectors`` (1: e0, 2: e0 and e1), leaving mem null when the device is out of memory or
// fx_ok is false
void fx_ctx_alloc(FxCtx* c, const Geom& g, int nrhs, int vectors);
void fx_ctx_free(FxCtx* c);
// encodes U, which must stay: before the first application of a solve
int fx_ctx_links(FxCtx& c, const Geom& g, const cpx<double>* U, cudaStream_t st);
// out = H in through e0, timed as one FP64 application
int fx_ctx_apply(const FxCtx& c, const Geom& g, double M5, double mf, const cpx<double>* in, cpx<double>* out, int nrhs,
                 cudaStream_t st);
int fx_ctx_apply_dot(const FxCtx& c, const Geom& g, double M5, double mf, const cpx<double>* in, cpx<double>* out,
                     RedScratch rs, double* result, cudaStream_t st);

}  // namespace hdcr
