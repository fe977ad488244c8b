// wilson_fixed.cuh -- the FP64 Wilson-Dirac hop in fixed-point arithmetic.
//
// Why: this part runs FP64 at 2 operations per clock and SM, and its 32 x 32 ->
// 64 bit integer multiply-add (IMAD.WIDE) at 61 (both measured), so the 816
// FP64 instructions per site of the hopping kernel in wilson_device.cuh cost 408
// clocks while three integer multiply-adds per real product, plus the integer
// additions around them, cost about 30.
//
// Number format.  A spinor (12 complex components of one site) is a block with
// one exponent e, |component| < 2^e, each real a 57-bit integer I = x 2^(57-e)
// kept as two 32-bit limbs, I = hi 2^28 + lo.  A link matrix, with -kappa and the
// antiperiodic sign multiplied in, is a block with exponent g such that the sum
// of |Re| + |Im| over every row and column is < 2^g, I = w 2^(57-g) in the same
// two limbs.  Input components within a factor 16 of their site's largest are
// exact, the others are cut off 57 bits below it.
//
// Products keep hi*hi (unit 2^56) and hi*lo + lo*hi (unit 2^28, cut off into
// the former); lo*lo is dropped, 2^-58 of the block products.  Bounds: half
// spinors double a component (limbs below 2^30 and 2^29), a row sum is below
// 2^59 in units of 2^-58 2^(e+g), and eight hops plus the site's own term are
// below 2^62.1: nothing can overflow 64 bits.  Each hop is shifted to the largest
// exponent of the nine terms, E, before it is added, so the sum has an absolute
// error of at most 269 units of 2^-58 2^E (per hop 12 for the dropped low products, 16 for
// the link's rounding, 4 for the spinor's cut-off, 1.5 for the shifts), a few in practice, where FP64
// arithmetic has rounding errors of 2^-54 of every partial sum.  In the 2-norm the error of D^H D on
// random spinors is no larger than the FP64 kernel's (1.3e-16 against 1.6e-16;
// tests/test_gpu_fixed.py holds it to that).  The bound is by site: a component far below its
// site's largest term has less relative accuracy than in FP64 arithmetic, and none below 2^-57
// of it (seed.h says so to the caller of seed_apply; tests/test_gpu_fixed_bound.py).
//
// Sites whose components are not finite, or whose largest one lies outside
// 2^-700 .. 2^700, keep their doubles (exponent code kExpRaw), and a site with
// such a neighbour or link is computed in FP64 (fix_site_fp64).
#pragma once
#include "wilson_device.cuh"

namespace seedk {

constexpr int kExpRaw = 1 << 28;      // the block holds doubles (spinor), or cannot be represented (link)
constexpr int kExpZero = -(1 << 20);  // all components zero
constexpr int kExpSlow = 1 << 20;     // a sum of exponents from here on has a raw block in it
constexpr int kExpSite = 700;         // largest |e| of a spinor block
constexpr int kExpLink = 150;         // largest |g| of a link block
constexpr int kLimb = 28;
constexpr int kLimbMask = (1 << kLimb) - 1;

SEED_DEV long long madw(int a, int b, long long c) { return (long long)a * b + c; }

// one real of a spinor or link block: magnitude (< 2^58) and sign -> limbs
SEED_DEV int2 fix_limbs(unsigned long long mag, bool neg) {
  const int s = neg ? -1 : 0;
  const int hi = (int)(mag >> kLimb), lo = (int)(mag & kLimbMask);
  return make_int2((hi ^ s) - s, (lo ^ s) - s);
}

// biased exponent of a double
SEED_DEV int fix_bexp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// Exponent of a spinor block from the largest biased exponent of its reals
// (kExpRaw / kExpZero where it has none) ...
SEED_DEV int fix_site_exp(int bmax, bool any) {
  if (!any) return kExpZero;
  const int e = bmax - 1022;
  return (e < -kExpSite || e > kExpSite) ? kExpRaw : e;   // Inf and NaN: bmax 2047
}
// ... and the limbs of one real with respect to it (d = bmax - its biased exponent;
// subnormals only occur far below a representable block: cut off to zero)
SEED_DEV int2 fix_from_double(double x, int bmax) {
  const unsigned hw = (unsigned)__double2hiint(x);
  const unsigned long long m =
      ((unsigned long long)((hw & 0xfffffu) | 0x100000u) << 32 | (unsigned)__double2loint(x)) << 4;
  const int d = bmax - (int)((hw >> 20) & 0x7ffu);
  return fix_limbs(d > 60 ? 0ull : m >> d, (int)hw < 0);
}

// acc 2^(E-58) as a double
SEED_DEV double fix_to_double(long long acc, int E) {
  const double d = (double)acc;
  const int hi = __double2hiint(d);
  return __hiloint2double(acc != 0 ? hi + ((E - 58) << 20) : 0, __double2loint(d));
}

// a complex real pair of limbs: x = Re hi, y = Re lo, z = Im hi, w = Im lo
template <int P> SEED_DEV int4 fix_ph_add(int4 a, int4 b) {   // a + phase(P) b
  if constexpr (P == 0) return make_int4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
  else if constexpr (P == 1) return make_int4(a.x - b.z, a.y - b.w, a.z + b.x, a.w + b.y);
  else if constexpr (P == 2) return make_int4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w);
  else return make_int4(a.x + b.z, a.y + b.w, a.z - b.x, a.w - b.y);
}
// the 64-bit complex accumulator (re, im) += phase(P) (x, y)
template <int P> SEED_DEV void fix_acc(long long &re, long long &im, long long x, long long y) {
  if constexpr (P == 0) { re += x; im += y; }
  else if constexpr (P == 1) { re -= y; im += x; }
  else if constexpr (P == 2) { re -= x; im -= y; }
  else { re += y; im -= x; }
}

// One hop of (1 - S g_MU) M psi, M = U (FWD) or U^H, for one component K of the half
// spinor: M h_K into the sums up[2 colour + re/im] of spin K and low[...] of spin
// 2 + J(K).  pu, pl: the components of those two spins; lnk(k): limbs of the link's
// element k; sh: the shift to the common exponent.  The projectors' phases are
// those of K = 0; for K = 1 they have the opposite sign in directions y and z: sg =
// -1 there, applied to h here and to low by the caller.
template <int MU, int S, bool FWD, class LU>
SEED_DEV void fix_hop(const int4 (&pu)[3], const int4 (&pl)[3], LU &&lnk, int sg, int sh, long long (&up)[6],
                      long long (&low)[6]) {
  constexpr int c = S > 0 ? ph_neg(bP(MU, 0)) : bP(MU, 0);
  constexpr int l = S > 0 ? ph_neg(ph_conj(bP(MU, 0))) : ph_conj(bP(MU, 0));
  int4 h[3];
  int2 nh[3];   // minus the imaginary (FWD) or real (U^H) part, for the differences
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if constexpr (MU == 1 || MU == 2)
      h[a] = fix_ph_add<c>(pu[a], make_int4(sg * pl[a].x, sg * pl[a].y, sg * pl[a].z, sg * pl[a].w));
    else h[a] = fix_ph_add<c>(pu[a], pl[a]);
    nh[a] = FWD ? make_int2(-h[a].z, -h[a].w) : make_int2(-h[a].x, -h[a].y);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    // Re: U ur hr - ui hi, U^H ur hr + ui hi;  Im: U ur hi + ui hr, U^H ur hi - ui hr
    long long rh = 0, rm = 0, ih = 0, im = 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const int4 u = FWD ? lnk(3 * a + b) : lnk(3 * b + a);
      const int2 ri = FWD ? nh[b] : make_int2(h[b].z, h[b].w);   // times ui in the real part
      const int2 ir = FWD ? make_int2(h[b].x, h[b].y) : nh[b];   // times ui in the imaginary part
      rh = madw(u.x, h[b].x, rh);
      ih = madw(u.x, h[b].z, ih);
      rm = madw(u.x, h[b].y, rm);
      im = madw(u.x, h[b].w, im);
      rm = madw(u.y, h[b].x, rm);
      im = madw(u.y, h[b].z, im);
      rh = madw(u.z, ri.x, rh);
      ih = madw(u.z, ir.x, ih);
      rm = madw(u.z, ri.y, rm);
      im = madw(u.z, ir.y, im);
      rm = madw(u.w, ri.x, rm);
      im = madw(u.w, ir.x, im);
    }
    const long long x = (rh + (rm >> kLimb)) >> sh, y = (ih + (im >> kLimb)) >> sh;
    up[2 * a] += x;
    up[2 * a + 1] += y;
    fix_acc<l>(low[2 * a], low[2 * a + 1], x, y);
  }
}

// A fixed-point spinor vector: limbs tiled by 32 sites (component k of site s
// at ((s / 32) 12 + k) 32 + s % 32, so a warp reads 512 contiguous bytes) and one
// exponent per site.
SEED_DEV int64_t fix_at(int64_t s) { return (s >> 5) * 384 + (s & 31); }

// One component of a block as a complex double (raw blocks hold the doubles themselves).
SEED_DEV double2 fix_read(int4 q, int e) {
  if (e == kExpRaw) return c2(__hiloint2double(q.x, q.y), __hiloint2double(q.z, q.w));
  if (e == kExpZero) return c2(0.0, 0.0);
  const double s = scalbn(1.0, e - 57);
  return c2(s * (double)(((long long)q.x << kLimb) + q.y), s * (double)(((long long)q.z << kLimb) + q.w));
}

template <int MU, int S>
SEED_DEV void fix_site_fp64_dir(const WilsonFix &op, const int4 *in, const int32_t *e, int64_t s, double2 (&out)[12]) {
  const int64_t nf = op.nbr[8 * s + 2 * MU], nb = op.nbr[8 * s + 2 * MU + 1];
  unsigned long long negf = 0, negb = 0;
  if (MU == 3 && op.bc_t) {
    const int64_t t = s / ((int64_t)op.dims[0] * op.dims[1] * op.dims[2]);
    if (t == op.dims[3] - 1) negf = CxBits<double2>::sign;
    if (t == 0) negb = CxBits<double2>::sign;
  }
  double2 pf[12], pb[12], uf[9], ub[9], acc[12];
  for (int k = 0; k < 12; ++k) {
    pf[k] = fix_read(in[fix_at(nf) + 32 * k], e[nf]);
    pb[k] = fix_read(in[fix_at(nb) + 32 * k], e[nb]);
  }
  for (int k = 0; k < 9; ++k) {
    uf[k] = op.links[((int64_t)MU * op.sites + s) * 9 + k];
    ub[k] = op.links[((int64_t)MU * op.sites + nb) * 9 + k];
  }
  hop_pair_r<MU, S>(pf, uf, negf, pb, ub, negb, acc);
  for (int k = 0; k < 12; ++k) out[k] = cadd(out[k], acc[k]);
}

// The site in FP64 (blocks that have no fixed-point form): psi - kappa * hops.
template <int S>
__device__ __noinline__ void fix_site_fp64(const WilsonFix &op, const int4 *in, const int32_t *e, int64_t s,
                                           double2 (&out)[12]) {
  for (int k = 0; k < 12; ++k) out[k] = c2(0.0, 0.0);
  fix_site_fp64_dir<0, S>(op, in, e, s, out);
  fix_site_fp64_dir<1, S>(op, in, e, s, out);
  fix_site_fp64_dir<2, S>(op, in, e, s, out);
  fix_site_fp64_dir<3, S>(op, in, e, s, out);
  for (int k = 0; k < 12; ++k) {
    const double2 p = fix_read(in[fix_at(s) + 32 * k], e[s]);
    out[k] = c2(fma(-op.kappa, out[k].x, p.x), fma(-op.kappa, out[k].y, p.y));
  }
}

// Element k of the link (mu, s): tiled by 32 sites like the spinors.
SEED_DEV int64_t fix_link_at(const WilsonFix &op, int mu, int64_t s) {
  return ((int64_t)mu * ((op.sites + 31) >> 5) + (s >> 5)) * 288 + (s & 31);
}

// A neighbour's two spins for half-spinor component K, loaded ahead of their use: the
// loads are volatile so that they stay where they are written, before the products of the
// hop in front.
struct FixPsi {
  int4 u[3], l[3];
};
SEED_DEV int4 fix_load(const int4 *p) {
  int4 v;
  asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
template <int MU> SEED_DEV void fix_fetch(const int4 *in, int64_t nb, int K, FixPsi &f) {
  const int4 *pa = in + fix_at(nb) + 96 * K, *pb = in + fix_at(nb) + 96 * (MU < 2 ? 3 - K : 2 + K);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    f.u[a] = fix_load(pa + 32 * a);
    f.l[a] = fix_load(pb + 32 * a);
  }
}
template <int MU, int S, bool FWD>
SEED_DEV void fix_one(const WilsonFix &op, const FixPsi &f, int64_t s, int64_t nb, int K, int sh, long long (&up)[6],
                      long long (&low)[6]) {
  const int4 *L = op.flinks + fix_link_at(op, MU, FWD ? s : nb);
  fix_hop<MU, S, FWD>(f.u, f.l, [&](int k) { return __ldg(L + 32 * k); }, 1 - 2 * K, sh, up, low);
}

// (D psi)(s) (S = +1) or (D^H psi)(s) for half-spinor component K, in units of 2^(E-58): up =
// spin K, lb + the other component's la = spin 2 + K (la: directions x and y of spin 3
// - K).  nb: the eight neighbours; sh: their shifts to the common exponent, 8 bits
// each; shs: the site's own.  Each hop's spinors are fetched while the one
// before it is multiplied; the site's own block comes with the x neighbours,
// which are in the same lines.
template <int S>
SEED_DEV void fix_site(const WilsonFix &op, const int4 *in, int64_t s, int K, const int (&nb)[8],
                       unsigned long long sh, int shs, long long (&up)[6], long long (&la)[6], long long (&lb)[6]) {
  const long long m = -(long long)K;   // K = 1: minus the y and z parts
#pragma unroll
  for (int c = 0; c < 6; ++c) la[c] = up[c] = 0;
  FixPsi f, g;
  fix_fetch<1>(in, nb[2], K, f);
  fix_fetch<1>(in, nb[3], K, g);
  fix_one<1, S, true>(op, f, s, nb[2], K, (int)(sh >> 16 & 63), up, la);
  fix_fetch<0>(in, nb[0], K, f);
  fix_one<1, -S, false>(op, g, s, nb[3], K, (int)(sh >> 24 & 63), up, la);
  fix_fetch<0>(in, nb[1], K, g);
#pragma unroll
  for (int c = 0; c < 6; ++c) la[c] = (la[c] ^ m) - m;
  fix_one<0, S, true>(op, f, s, nb[0], K, (int)(sh & 63), up, la);
  fix_fetch<2>(in, s, K, f);   // the site itself: spins K and 2 + K
  fix_one<0, -S, false>(op, g, s, nb[1], K, (int)(sh >> 8 & 63), up, la);
  fix_fetch<2>(in, nb[4], K, g);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    up[2 * c] += ((((long long)f.u[c].x << kLimb) + f.u[c].y) << 1) >> shs;
    up[2 * c + 1] += ((((long long)f.u[c].z << kLimb) + f.u[c].w) << 1) >> shs;
    lb[2 * c] = (((((long long)f.l[c].x << kLimb) + f.l[c].y) << 1) >> shs ^ m) - m;
    lb[2 * c + 1] = (((((long long)f.l[c].z << kLimb) + f.l[c].w) << 1) >> shs ^ m) - m;
  }
  fix_fetch<2>(in, nb[5], K, f);
  fix_one<2, S, true>(op, g, s, nb[4], K, (int)(sh >> 32 & 63), up, lb);
  fix_fetch<3>(in, nb[6], K, g);
  fix_one<2, -S, false>(op, f, s, nb[5], K, (int)(sh >> 40 & 63), up, lb);
  fix_fetch<3>(in, nb[7], K, f);
#pragma unroll
  for (int c = 0; c < 6; ++c) lb[c] = (lb[c] ^ m) - m;
  fix_one<3, S, true>(op, g, s, nb[6], K, (int)(sh >> 48 & 63), up, lb);
  fix_one<3, -S, false>(op, f, s, nb[7], K, (int)(sh >> 56 & 63), up, lb);
}

// Normalisation of a block acc 2^(E-58): the OR of the reals' one's complement
// magnitudes (high and low words) gives the length of the largest, hence the
// exponent and the left shift to 63 bits.  A lone -2^j has length j, one short: it
// still fits (|I| <= 2^57).
SEED_DEV void fix_or(long long a, unsigned &mh, unsigned &ml) {
  const int hi = (int)(a >> 32), sg = hi >> 31;
  mh |= (unsigned)(hi ^ sg);
  ml |= (unsigned)((int)a ^ sg);
}
SEED_DEV int fix_bits(unsigned mh, unsigned ml) { return mh ? 64 - __clz(mh) : 32 - __clz(ml); }
SEED_DEV int2 fix_norm(long long a, int sh) {   // limbs of a 2^(sh - 6), |a 2^sh| <= 2^63
  const unsigned long long t = (unsigned long long)a << sh;
  return make_int2((int)(t >> 32) >> 2, (int)((t >> 6) & kLimbMask));
}

}  // namespace seedk
