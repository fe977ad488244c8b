// wilson_fixed.cu -- the kernels of the fixed-point Wilson-Dirac operator
// (wilson_fixed.cuh): the links' and spinors' conversion, and D / D^H.
//
// Operator: a warp handles 16 consecutive sites of one column, two threads per
// site, one for each component of the half spinor, all eight hops in registers
// (both threads use the same links, one request); consecutive warps take
// consecutive columns of the same sites, so that the columns of a block share the links in
// L1.  Bound by instruction issue and the latency between dependent integer
// instructions (0.39 instructions per clock and scheduler; long-scoreboard and fixed-latency
// waits in equal parts; L2 at 20 %, DRAM at 1.5 TB/s).  D^H D with the
// conversion of the input, GB300, FP64 kernel -> this one: 16^4 x 12 columns 2198 ->
// 597 us, x 1 column 201 -> 72 us; 8^4 x 12 columns 160 -> 54 us; with the links' conversion
// too (a seed_apply call) 16^4 x 12 columns 2198 -> 620 us.  Other splits, such calls at 16^4 x 12
// columns, beside 613 us of this one in that session: one thread per site 623 us (168
// registers, waiting for memory two thirds of the time); one per site and direction 808 us (an
// exchange of 24 KB of partial sums per tile); 16 warps an SM instead of 12 (128 registers) 629 us;
// the links fetched ahead as well (246 registers) 719 us; warps of a block kept in step
// by a barrier per hop 612 us (no gain).
#include "seed_device.cuh"
#include "wilson_fixed.cuh"

namespace seedk {

constexpr int FT = 128;                         // threads per block
constexpr int kFixPitch = 25;                   // doubles per site of a staged tile (24 + 1: no bank conflicts)

// ---------------------------------------------------------------------------
// Links: limbs of w = -kappa U (the antiperiodic sign included), tiled by 32
// sites like the spinors, and one exponent per link.  Integer arithmetic:
// the product of the two 53-bit significands is rounded once, to 57 bits below the
// block's exponent.  Run at the start of every call that applies the operator,
// so the caller's link array may change between calls.  Bound by memory
// (292 bytes per link).
// ---------------------------------------------------------------------------

// One link: limbs and exponent (kExpRaw, kExpZero: zero limbs).  minus_t: the antiperiodic sign.
SEED_DEV int fix_link(const double2 (&u)[9], double kappa, bool minus_t, int4 (&L)[9]) {
  int bmax = 0;
  bool any = false;
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    bmax = max(bmax, max(fix_bexp(u[k].x), fix_bexp(u[k].y)));
    any |= u[k].x != 0.0 || u[k].y != 0.0;
  }
  const unsigned kh = (unsigned)__double2hiint(kappa);
  const int kb = (int)((kh >> 20) & 0x7ffu);
  const int em = bmax - 1022, ek = kb - 1022;   // |entry| < 2^em, |kappa| < 2^ek
  int g = kExpZero;
  if (bmax == 2047) g = kExpRaw;
  else if (any && kappa != 0.0) g = (em < -kExpLink + 4 || em > kExpLink - 4 || ek < -kExpLink + 4 ||
                                     ek > kExpLink - 4 || em + ek < -kExpLink + 4 || em + ek > kExpLink - 4)
                                        ? kExpRaw : em + ek;
  if (g == kExpRaw || g == kExpZero) {
#pragma unroll
    for (int k = 0; k < 9; ++k) L[k] = make_int4(0, 0, 0, 0);
    return g;
  }
  // upper bound of the row and column sums of |Re| + |Im|, in units of 2^(em - 21)
  unsigned row[3] = {0, 0, 0}, col[3] = {0, 0, 0};
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    unsigned t = 0;
#pragma unroll
    for (int ri = 0; ri < 2; ++ri) {
      const unsigned hw = (unsigned)__double2hiint(ri ? u[k].y : u[k].x);
      const int d = bmax - (int)((hw >> 20) & 0x7ffu);
      t += (d > 31 ? 0u : ((hw & 0xfffffu) | 0x100000u) >> d) + 1u;
    }
    row[k / 3] += t;
    col[k % 3] += t;
  }
  unsigned l1 = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a) l1 = max(l1, max(row[a], col[a]));
  const int slack = max(0, 32 - __clz(l1) - 21);   // l1 < 2^(21 + slack)
  g += slack;
  const bool flip = !((int)kh < 0) ^ minus_t;
  const unsigned long long km = ((unsigned long long)((kh & 0xfffffu) | 0x100000u) << 32 |
                                 (unsigned)__double2loint(kappa)) << 11;   // kappa 2^(64 - ek)
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    int2 l[2];
#pragma unroll
    for (int ri = 0; ri < 2; ++ri) {
      const double v = ri ? u[k].y : u[k].x;
      const unsigned hw = (unsigned)__double2hiint(v);
      const unsigned long long m = ((unsigned long long)((hw & 0xfffffu) | 0x100000u) << 32 |
                                    (unsigned)__double2loint(v)) << 11;
      // |v kappa| = y 2^(em - d + ek - 64); to units of 2^(g - 57)
      const int sh = 7 + slack + (bmax - (int)((hw >> 20) & 0x7ffu));
      const unsigned long long y = sh > 63 ? 0ull : ((__umul64hi(m, km) >> (sh - 1)) + 1ull) >> 1;
      l[ri] = fix_limbs(y, ((int)hw < 0) ^ flip);
    }
    L[k] = make_int4(l[0].x, l[0].y, l[1].x, l[1].y);
  }
  return g;
}
// Link idx = mu * sites + s
SEED_DEV void fix_link_of(const WilsonFix &op, int4 *fl, int32_t *fe, int64_t idx) {
  if (idx >= 4 * op.sites) return;
  const int64_t mu = idx / op.sites, s = idx - mu * op.sites;
  const bool minus_t = mu == 3 && op.bc_t && s / ((int64_t)op.dims[0] * op.dims[1] * op.dims[2]) == op.dims[3] - 1;
  double2 u[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) u[k] = __ldg(op.links + idx * 9 + k);
  int4 l[9];
  fe[idx] = fix_link(u, op.kappa, minus_t, l);
  int4 *L = fl + fix_link_at(op, (int)mu, s);
#pragma unroll
  for (int k = 0; k < 9; ++k) L[32 * k] = l[k];
}

__global__ void __launch_bounds__(128) k_fix_links(WilsonFix op, int4 *__restrict__ fl, int32_t *__restrict__ fe) {
  fix_link_of(op, fl, fe, (int64_t)blockIdx.x * blockDim.x + threadIdx.x);
}

void launch_fix_links(const WilsonFix &op, cudaStream_t s) {
  const int64_t nl = 4 * op.sites;
  k_fix_links<<<(unsigned)((nl + 127) / 128), 128, 0, s>>>(op, const_cast<int4 *>(op.flinks),
                                                           const_cast<int32_t *>(op.fexp));
}

// ---------------------------------------------------------------------------
// Spinors
// ---------------------------------------------------------------------------
// One site's block from its 24 reals real(k): this thread (half = 0 or 1) stores the
// components of spins half and 2 + half as limbs, half 0 the exponent.  A block without a
// fixed-point form stores the doubles.  q: component 3 half's place, e: the site's.
template <class LD>
SEED_DEV void fix_store_block(LD &&real, int half, int4 *__restrict__ q, int32_t *__restrict__ e) {
  int bmax = 0;
  bool any = false;
#pragma unroll
  for (int k = 0; k < 24; ++k) {
    const double z = real(k);
    bmax = max(bmax, fix_bexp(z));
    any |= z != 0.0;
  }
  const int ex = fix_site_exp(bmax, any);
  if (half == 0) *e = ex;
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int k = 12 * h + 6 * half + 2 * c;
      const double x = real(k), y = real(k + 1);
      int4 v;
      if (ex == kExpRaw) {
        v = make_int4(__double2hiint(x), __double2loint(x), __double2hiint(y), __double2loint(y));
      } else {
        const int2 a = fix_from_double(x, bmax), b = fix_from_double(y, bmax);
        v = ex == kExpZero ? make_int4(0, 0, 0, 0) : make_int4(a.x, a.y, b.x, b.y);
      }
      q[32 * (6 * h + c)] = v;
    }
}

// What the last step of a kernel that works by groups of sites does with a column's
// sum: every warp leaves its partial in part[grp], and the last warp of the
// column adds them, lane l taking groups l, l + 32, ... in order, then a fixed
// shuffle tree (the same whichever warp is last).  True in the last warp.
SEED_DEV bool group_sum_last(double v, double *part, int64_t grp, int groups, unsigned *ticket, double &sum) {
  v = warp_sum(v);
  unsigned last = 0;
  if ((threadIdx.x & 31) == 0) {
    part[grp] = v;
    __threadfence();
    last = atomicAdd(ticket, 1u) == (unsigned)groups - 1u;
    if (last) *ticket = 0u;
  }
  if (!__shfl_sync(0xffffffffu, last, 0)) return false;
  __threadfence();
  sum = warp_sum_partials(part, groups, 1, 0);
  return true;
}

// A tile's 32 sites (st[site * kFixPitch + real], staged by 64 threads) -> limbs and exponents
SEED_DEV void fix_store_tile(const double *st, int4 *__restrict__ q, int32_t *__restrict__ e) {
  const int sl = threadIdx.x & 31, half = threadIdx.x >> 5;
  const double *mine = st + sl * kFixPitch;
  fix_store_block([&](int k) { return mine[k]; }, half, q + 96 * half + sl, e + sl);
}
constexpr int CT = 64;   // threads of the tile kernels

// One normalised component of a result block (raw: as doubles).
SEED_DEV int4 fix_out(long long re, long long im, int E, int sh, bool raw, bool zero) {
  if (raw) {
    const double x = fix_to_double(re, E), y = fix_to_double(im, E);
    return make_int4(__double2hiint(x), __double2loint(x), __double2hiint(y), __double2loint(y));
  }
  if (zero) return make_int4(0, 0, 0, 0);
  const int2 x = fix_norm(re, sh), y = fix_norm(im, sh);
  return make_int4(x.x, x.y, y.x, y.y);
}

// grid: tiles * ncols blocks, the column fastest
SEED_DEV void fix_spinor_tile(const double2 *X, int64_t ldx, int4 *q, int64_t ldq, int32_t *e, int64_t sites,
                              int64_t tile, int col) {
  __shared__ double st[32 * kFixPitch];
  const double2 *x = X + (int64_t)col * ldx + tile * 384;
  const int64_t left = 12 * sites - tile * 384;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int o = threadIdx.x + CT * k, sl = o / 12, c = o - 12 * sl;
    const double2 z = o < left ? __ldg(x + o) : make_double2(0.0, 0.0);
    st[sl * kFixPitch + 2 * c] = z.x;
    st[sl * kFixPitch + 2 * c + 1] = z.y;
  }
  __syncthreads();
  fix_store_tile(st, q + (int64_t)col * ldq + tile * 384, e + (int64_t)col * (ldq / 12) + tile * 32);
}

__global__ void __launch_bounds__(CT) k_fix_spinors(const double2 *__restrict__ X, int64_t ldx, int4 *__restrict__ q,
                                                    int64_t ldq, int32_t *__restrict__ e, int64_t sites, int ncols,
                                                    const int32_t *__restrict__ col_active) {
  const int64_t tile = blockIdx.x / ncols;
  const int col = (int)(blockIdx.x - tile * ncols);
  if (col_active != nullptr && col_active[col] == 0) return;
  fix_spinor_tile(X, ldx, q, ldq, e, sites, tile, col);
}

// Links and spinors in one launch, for the smallest operands: the first link_blocks blocks
// convert CT links each, the others a tile of a column each.
__global__ void __launch_bounds__(CT) k_fix_both(WilsonFix op, int4 *__restrict__ fl, int32_t *__restrict__ fe,
                                                 const double2 *__restrict__ X, int64_t ldx, int4 *__restrict__ q,
                                                 int64_t ldq, int32_t *__restrict__ e, int ncols, unsigned link_blocks) {
  if (blockIdx.x < link_blocks) {
    fix_link_of(op, fl, fe, (int64_t)blockIdx.x * CT + threadIdx.x);
    return;
  }
  const int64_t b = blockIdx.x - link_blocks, tile = b / ncols;
  fix_spinor_tile(X, ldx, q, ldq, e, op.sites, tile, (int)(b - tile * ncols));
}

void launch_fix_both(const WilsonFix &op, const double2 *X, int64_t ldx, int4 *q, int64_t ldq, int32_t *e, int ncols,
                     cudaStream_t s) {
  const unsigned links = (unsigned)((4 * op.sites + CT - 1) / CT);
  k_fix_both<<<links + (unsigned)((op.sites + 31) / 32 * ncols), CT, 0, s>>>(
      op, const_cast<int4 *>(op.flinks), const_cast<int32_t *>(op.fexp), X, ldx, q, ldq, e, ncols, links);
}

void launch_fix_spinors(const WilsonFix &op, const double2 *X, int64_t ldx, int4 *q, int64_t ldq, int32_t *e,
                        int ncols, const int32_t *col_active, cudaStream_t s) {
  if (ncols < 1) return;
  k_fix_spinors<<<(unsigned)((op.sites + 31) / 32 * ncols), CT, 0, s>>>(X, ldx, q, ldq, e, op.sites, ncols, col_active);
}

// ---------------------------------------------------------------------------
// D (S = +1) or D^H (S = -1) on ncols columns.  OUT = 0: the result as fixed-point
// blocks (the next application's input); 1: as doubles in the caller's
// site-major layout, through shared memory so that the stores are coalesced;
// 2: the same, and lockstep CG's alpha = rho / Re(p^H q) with q the result and p
// = P, formed while q is on chip: a partial per warp, added in a fixed order by the column's last.
// Consecutive warps take consecutive columns of the same sites: the columns of a
// block share the links in L1.
// ---------------------------------------------------------------------------
template <int S, int OUT>
__global__ void __launch_bounds__(FT, 3) k_dslash_fix(WilsonFix op, const int4 *__restrict__ in,
                                                      const int32_t *__restrict__ ein, int64_t ldq,
                                                      int4 *__restrict__ qout, int32_t *__restrict__ eout,
                                                      double2 *__restrict__ out, int64_t ldo, int64_t items, int ncols,
                                                      const int32_t *__restrict__ col_active, CgDot<double2> dot) {
  extern __shared__ double stage_all[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, half = lane >> 4, sl = lane & 15;
  const int64_t item = (int64_t)blockIdx.x * (FT / 32) + warp;
  if (item >= items) return;
  const int64_t grp = item / ncols;   // 16 sites
  const int col = (int)(item - grp * ncols);
  if (col_active != nullptr && col_active[col] == 0) return;
  in += (int64_t)col * ldq;
  ein += (int64_t)col * (ldq / 12);
  const int64_t s = grp * 16 + sl;
  const bool live = s < op.sites;
  // the common exponent of the nine terms
  int nb[8], E = kExpZero, es = kExpZero;
  unsigned long long shifts = 0;
  if (live) {
    const int4 *q = reinterpret_cast<const int4 *>(op.nbr + 8 * s);
    const int4 na = __ldg(q), nc = __ldg(q + 1);
    nb[0] = na.x; nb[1] = na.y; nb[2] = na.z; nb[3] = na.w;
    nb[4] = nc.x; nb[5] = nc.y; nb[6] = nc.z; nb[7] = nc.w;
    int x[8];
    E = es = __ldg(ein + s);
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      x[d] = __ldg(ein + nb[d]) + __ldg(op.fexp + (int64_t)(d >> 1) * op.sites + (d & 1 ? nb[d] : s));
      E = max(E, x[d]);
    }
#pragma unroll
    for (int d = 0; d < 8; ++d) shifts |= (unsigned long long)min(E - x[d], 63) << (8 * d);
  }
  const bool slow = E >= kExpSlow;
  long long v[2][6], la[6];   // spins half and 2 + half of the site, directions x and y of spin 3 - half
#pragma unroll
  for (int c = 0; c < 6; ++c) v[0][c] = v[1][c] = la[c] = 0;
  if (live && !slow) fix_site<S>(op, in, s, half, nb, shifts, min(E - es, 63), v[0], la, v[1]);
  // the directions x and y of spin 2 + half are the site's other thread's
#pragma unroll
  for (int c = 0; c < 6; ++c) v[1][c] += __shfl_xor_sync(0xffffffffu, la[c], 16);
  if constexpr (OUT == 0) {
    int4 *q = qout + (int64_t)col * ldq + fix_at(s) + 96 * half;
    int32_t *e = eout + (int64_t)col * (ldq / 12) + s;
    unsigned mh = 0, ml = 0;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int c = 0; c < 6; ++c) fix_or(v[h][c], mh, ml);
    mh |= __shfl_xor_sync(0xffffffffu, mh, 16);
    ml |= __shfl_xor_sync(0xffffffffu, ml, 16);
    if (!live) return;
    if (slow) {
      double2 o[12];
      fix_site_fp64<S>(op, in, ein, s, o);
      fix_store_block([&](int k) { return k & 1 ? o[k >> 1].y : o[k >> 1].x; }, half, q, e);
      return;
    }
    const int bits = fix_bits(mh, ml), ex = E - 58 + bits, sh = 63 - bits;
    const bool zero = bits == 0, raw = !zero && (ex < -kExpSite || ex > kExpSite);
    if (half == 0) *e = zero ? kExpZero : raw ? kExpRaw : ex;
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int c = 0; c < 3; ++c)
        q[32 * (6 * h + c)] = fix_out(v[h][2 * c], v[h][2 * c + 1], E, sh, raw, zero);
  } else {
    double *st = stage_all + warp * 16 * kFixPitch;
    double *mine = st + sl * kFixPitch + 6 * half;
    if (slow) {
      double2 o[12];
      fix_site_fp64<S>(op, in, ein, s, o);
      for (int c = 0; c < 3; ++c) {
        mine[2 * c] = o[3 * half + c].x;
        mine[2 * c + 1] = o[3 * half + c].y;
        mine[12 + 2 * c] = o[6 + 3 * half + c].x;
        mine[13 + 2 * c] = o[6 + 3 * half + c].y;
      }
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int c = 0; c < 6; ++c) mine[12 * h + c] = fix_to_double(v[h][c], E);
    }
    __syncwarp();
    double2 *y = out + (int64_t)col * ldo + grp * 192;
    const int64_t left = 12 * op.sites - grp * 192;
    const double2 *p = OUT == 2 ? dot.P + (int64_t)col * ldo + grp * 192 : nullptr;
    double pq = 0.0;
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int i = lane + 32 * k, is = i / 12, c = i - 12 * is;
      if (i < left) {
        const double2 z = make_double2(st[is * kFixPitch + 2 * c], st[is * kFixPitch + 2 * c + 1]);
        y[i] = z;
        if constexpr (OUT == 2) pq = Sc<double2>::redot(__ldg(p + i), z, pq);
      }
    }
    if constexpr (OUT == 2) {
      const int groups = (int)((op.sites + 15) / 16);
      double sum;
      if (group_sum_last(pq, dot.part + (int64_t)col * groups, grp, groups, dot.tickets + kColTicket + col, sum) &&
          lane == 0)
        dot.alpha[col] = dot.rho[col] / sum;
    }
  }
}

constexpr size_t kFixStage = sizeof(double) * (FT / 32) * 16 * kFixPitch;

// ---------------------------------------------------------------------------
// The same for few sites and columns: eight warps per tile, one per direction and
// half-spinor component, two hops per thread, the partial sums exchanged through
// shared memory.  A launch that leaves most schedulers with a warp or two lasts
// as long as one warp's chain of loads and products, which is a quarter as
// long here; with more work the exchange and the repeated link loads cost more than
// the chain.  D^H D of 8^4 x 2 columns (256 tiles) 26.7 -> 22.5 us, x 12 columns
// (1536) 54 -> 57 us; lockstep CG on 4^4 x 11 columns (88) 39 -> 31 us per iteration,
// on 8^4 x 11 columns 64 -> 74.
// ---------------------------------------------------------------------------
constexpr int DT = 256;

template <int MU, int S>
SEED_DEV void fix_pair_dir(const WilsonFix &op, const int4 *in, int64_t s, int nf, int nb, int K, int shf, int shb,
                           long long (*acc)[32]) {
  const int lane = threadIdx.x & 31;
  long long up[6], low[6];
#pragma unroll
  for (int c = 0; c < 6; ++c) up[c] = low[c] = 0;
  FixPsi f, g;
  fix_fetch<MU>(in, nf, K, f);
  fix_fetch<MU>(in, nb, K, g);
  fix_one<MU, S, true>(op, f, s, nf, K, shf, up, low);
  fix_one<MU, -S, false>(op, g, s, nb, K, shb, up, low);
  const long long m = (MU == 1 || MU == 2) ? -(long long)K : 0;
#pragma unroll
  for (int c = 0; c < 6; ++c) {
    acc[c][lane] = up[c];
    acc[6 + c][lane] = (low[c] ^ m) - m;
  }
}

// Component c of spin w of a site: the four directions' partial sums and its own block's value.
SEED_DEV void fix_spin_sum(const long long (*sacc)[2][12][32], int w, int c, int lane, int4 p, int shs, long long &re,
                           long long &im) {
  const int kxy = w < 2 ? w : 3 - w, kzt = w < 2 ? w : w - 2, k = (w < 2 ? 0 : 6) + 2 * c;
  const long long r = ((long long)p.x << kLimb) + p.y, i = ((long long)p.z << kLimb) + p.w;
  re = ((r << 1) >> shs) + ((sacc[0][kxy][k][lane] + sacc[1][kxy][k][lane]) + (sacc[2][kzt][k][lane] + sacc[3][kzt][k][lane]));
  im = ((i << 1) >> shs) + ((sacc[0][kxy][k + 1][lane] + sacc[1][kxy][k + 1][lane]) +
                            (sacc[2][kzt][k + 1][lane] + sacc[3][kzt][k + 1][lane]));
}

// The block's result from the sums of warps 0..3 (spin w in v), normalised over the four spins;
// sites in FP64 (slow) have their 24 reals in sacc.  Contains a CTA barrier.
SEED_DEV void fix_store_dir(const long long (*sacc)[2][12][32], unsigned (*sO)[2][32], int w, int lane, bool live,
                            bool slow, int E, const long long (&v)[6], int4 *q, int32_t *e) {
  if (w < 4) {
    unsigned mh = 0, ml = 0;
#pragma unroll
    for (int c = 0; c < 6; ++c) fix_or(v[c], mh, ml);
    sO[w][0][lane] = mh;
    sO[w][1][lane] = ml;
  }
  __syncthreads();
  if (!live || w >= 4) return;
  if (slow) {
    const double *x = reinterpret_cast<const double *>(&sacc[0][0][0][0]);
    if (w < 2) fix_store_block([&](int k) { return x[32 * k + lane]; }, w, q + 96 * w, e);
    return;
  }
  const unsigned mh = (sO[0][0][lane] | sO[1][0][lane]) | (sO[2][0][lane] | sO[3][0][lane]);
  const unsigned ml = (sO[0][1][lane] | sO[1][1][lane]) | (sO[2][1][lane] | sO[3][1][lane]);
  const int bits = fix_bits(mh, ml), ex = E - 58 + bits, sh = 63 - bits;
  const bool zero = bits == 0, raw = !zero && (ex < -kExpSite || ex > kExpSite);
  if (w == 0) *e = zero ? kExpZero : raw ? kExpRaw : ex;
#pragma unroll
  for (int c = 0; c < 3; ++c) q[32 * (3 * w + c)] = fix_out(v[2 * c], v[2 * c + 1], E, sh, raw, zero);
}

template <int S, int OUT>
__global__ void __launch_bounds__(DT, 3) k_dslash_fix_dir(WilsonFix op, const int4 *__restrict__ in,
                                                          const int32_t *__restrict__ ein, int64_t ldq,
                                                          int4 *__restrict__ qout, int32_t *__restrict__ eout,
                                                          double2 *__restrict__ out, int64_t ldo, int ncols,
                                                          const int32_t *__restrict__ col_active, CgDot<double2> dot) {
  __shared__ long long sacc[4][2][12][32];   // [direction][component][up, low reals][site]
  __shared__ int sE[4][32];
  __shared__ unsigned sO[4][2][32];
  __shared__ double sred[DT / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, mu = warp >> 1, K = warp & 1;
  const int64_t tile = blockIdx.x / ncols;
  const int col = (int)(blockIdx.x - tile * ncols);
  if (col_active != nullptr && col_active[col] == 0) return;
  in += (int64_t)col * ldq;
  ein += (int64_t)col * (ldq / 12);
  const int64_t s = tile * 32 + lane;
  const bool live = s < op.sites;
  int nf = 0, nb = 0, xf = kExpZero, xb = kExpZero, E = kExpZero;
  if (live) {
    const int2 n = __ldg(reinterpret_cast<const int2 *>(op.nbr + 8 * s) + mu);
    nf = n.x;
    nb = n.y;
    E = __ldg(ein + s);
    xf = __ldg(ein + nf) + __ldg(op.fexp + mu * op.sites + s);
    xb = __ldg(ein + nb) + __ldg(op.fexp + mu * op.sites + nb);
  }
  const int es = E;
  if (K == 0) sE[mu][lane] = max(xf, xb);
  __syncthreads();
  E = max(max(E, max(sE[0][lane], sE[1][lane])), max(sE[2][lane], sE[3][lane]));
  const bool slow = E >= kExpSlow;
  double (*sslow)[32] = reinterpret_cast<double (*)[32]>(&sacc[0][0][0][0]);   // FP64 sites: their 24 reals
  if (live && !slow) {
    const int shf = min(E - xf, 63), shb = min(E - xb, 63);
    long long (*acc)[32] = sacc[mu][K];
    switch (mu) {
      case 0: fix_pair_dir<0, S>(op, in, s, nf, nb, K, shf, shb, acc); break;
      case 1: fix_pair_dir<1, S>(op, in, s, nf, nb, K, shf, shb, acc); break;
      case 2: fix_pair_dir<2, S>(op, in, s, nf, nb, K, shf, shb, acc); break;
      default: fix_pair_dir<3, S>(op, in, s, nf, nb, K, shf, shb, acc); break;
    }
  } else if (slow && warp == 0) {
    double2 o[12];
    fix_site_fp64<S>(op, in, ein, s, o);
    for (int k = 0; k < 12; ++k) {
      sslow[2 * k][lane] = o[k].x;
      sslow[2 * k + 1][lane] = o[k].y;
    }
  }
  __syncthreads();
  // warps 0..3: spin w, its four directions and the site's own term
  const int w = warp;
  long long v[6];
  if (w < 4) {
    const int shs = min(E - es, 63);
#pragma unroll
    for (int c = 0; c < 3; ++c)
      fix_spin_sum(sacc, w, c, lane, live ? __ldg(in + fix_at(s) + 32 * (3 * w + c)) : make_int4(0, 0, 0, 0), shs,
                   v[2 * c], v[2 * c + 1]);
  }
  if constexpr (OUT == 0) {
    fix_store_dir(sacc, sO, w, lane, live, slow, E, v, qout + (int64_t)col * ldq + tile * 384 + lane,
                  eout + (int64_t)col * (ldq / 12) + s);
  } else {
    double d[6];
    if (w < 4) {
#pragma unroll
      for (int c = 0; c < 6; ++c) d[c] = slow ? sslow[6 * w + c][lane] : fix_to_double(v[c], E);
    }
    __syncthreads();
    double *st = reinterpret_cast<double *>(&sacc[0][0][0][0]);
    if (w < 4) {
#pragma unroll
      for (int c = 0; c < 6; ++c) st[lane * kFixPitch + 6 * w + c] = d[c];
    }
    __syncthreads();
    double2 *y = out + (int64_t)col * ldo + tile * 384;
    const int64_t left = 12 * op.sites - tile * 384;
    const double2 *p = OUT == 2 ? dot.P + (int64_t)col * ldo + tile * 384 : nullptr;
    double pq = 0.0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int o = threadIdx.x + DT * k, sl = o / 12, c = o - 12 * sl;
      if (o < 384 && o < left) {
        const double2 z = make_double2(st[sl * kFixPitch + 2 * c], st[sl * kFixPitch + 2 * c + 1]);
        y[o] = z;
        if constexpr (OUT == 2) pq = Sc<double2>::redot(__ldg(p + o), z, pq);
      }
    }
    if constexpr (OUT == 2) {
      const int tiles = (int)((op.sites + 31) / 32);
      double *part = dot.part + (int64_t)col * tiles;
      double t[1] = {pq};
      block_sum<1, DT>(t, sred);
      if (threadIdx.x == 0) part[tile] = t[0];
      if (!last_block_done(dot.tickets + kColTicket + col, (unsigned)tiles)) return;
      const double rho = __ldcg(dot.rho + col);
      const double sum = sum_partials<DT>(part, tiles, 1, 0, sred);
      if (threadIdx.x == 0) dot.alpha[col] = rho / sum;
    }
  }
}

// up to this many tiles x columns (two per SM) in one launch: one warp per direction and component
constexpr int64_t kFixDirItems = 304;

bool fix_few(int64_t sites, int ncols) { return (sites + 31) / 32 * ncols <= kFixDirItems; }

void launch_dslash_fix(const WilsonFix &op, int sign, const int4 *in, const int32_t *ein, int64_t ldq, int4 *qout,
                       int32_t *eout, double2 *out, int64_t ldo, int ncols, const int32_t *col_active, cudaStream_t s,
                       const CgDot<double2> *dot) {
  if (ncols < 1) return;
  const int64_t items = (op.sites + 15) / 16 * ncols;
  const unsigned grid = (unsigned)((items + FT / 32 - 1) / (FT / 32));
  const CgDot<double2> d = dot ? *dot : CgDot<double2>{};
  const int64_t tiles = (op.sites + 31) / 32;
#define FIX_GO(S, OUT)                                                                                              \
  if (fix_few(op.sites, ncols))                                                                                     \
    k_dslash_fix_dir<S, OUT><<<(unsigned)(tiles * ncols), DT, 0, s>>>(op, in, ein, ldq, qout, eout, out, ldo, ncols,  \
                                                                      col_active, d);                               \
  else                                                                                                              \
    k_dslash_fix<S, OUT><<<grid, FT, OUT == 0 ? 0 : kFixStage, s>>>(op, in, ein, ldq, qout, eout, out, ldo, items, ncols, \
                                                                  col_active, d)
  if (qout != nullptr) {
    if (sign > 0) {
      FIX_GO(+1, 0);
    } else {
      FIX_GO(-1, 0);
    }
  } else if (dot != nullptr) {   // lockstep CG: q = D^H t
    FIX_GO(-1, 2);
  } else if (sign > 0) {   // D by itself: from 16384 sites on only, never few
    k_dslash_fix<+1, 1><<<grid, FT, kFixStage, s>>>(op, in, ein, ldq, qout, eout, out, ldo, items, ncols, col_active, d);
  } else {
    FIX_GO(-1, 1);
  }
#undef FIX_GO
}

// ---------------------------------------------------------------------------
// Lockstep CG, end of an iteration: x += alpha p (deferred to here from the
// residual's update, so that p is read once), p = r + beta p, and p's blocks for
// the next D.  A column that has just stopped (stepped set, not active) takes its x
// update only.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(CT) k_cg_xp_fix(const CallArgs *call, const double2 *__restrict__ R,
                                                  double2 *__restrict__ P, int64_t ld, int4 *__restrict__ q,
                                                  int32_t *__restrict__ e, int64_t sites, CgCols c) {
  __shared__ double st[32 * kFixPitch];
  const int64_t tile = blockIdx.x / c.nc;
  const int col = (int)(blockIdx.x - tile * c.nc);
  if (!c.stepped[col]) return;
  const bool act = c.active[col] != 0;
  const double al = c.alpha[col], be = c.beta[col];
  double2 *x = reinterpret_cast<double2 *>(call->X) + (int64_t)(col + call->col0) * call->ldx + tile * 384;
  const double2 *r = R + (int64_t)col * ld + tile * 384;
  double2 *p = P + (int64_t)col * ld + tile * 384;
  const int64_t left = 12 * sites - tile * 384;
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const int o = threadIdx.x + CT * k, sl = o / 12, cc = o - 12 * sl;
    double2 z = make_double2(0.0, 0.0);
    if (o < left) {
      const double2 pv = p[o];
      x[o] = Sc<double2>::axpy(al, pv, x[o]);
      if (act) {
        z = Sc<double2>::axpy(be, pv, r[o]);
        p[o] = z;
      }
    }
    st[sl * kFixPitch + 2 * cc] = z.x;
    st[sl * kFixPitch + 2 * cc + 1] = z.y;
  }
  if (!act) return;   // uniform over the block
  __syncthreads();
  fix_store_tile(st, q + (int64_t)col * ld + tile * 384, e + (int64_t)col * (ld / 12) + tile * 32);
}

void launch_cg_xp_fix(const WilsonFix &op, const CallArgs *call, const double2 *R, double2 *P, int64_t ld, int4 *q,
                      int32_t *e, const CgCols &c, cudaStream_t s) {
  k_cg_xp_fix<<<(unsigned)((op.sites + 31) / 32 * c.nc), CT, 0, s>>>(call, R, P, ld, q, e, op.sites, c);
}

}  // namespace seedk
