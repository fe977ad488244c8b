// wilson32.cu -- the FP32 copy of the Wilson-Dirac operator used by the
// mixed-precision path (seed_params.precision = 1) on sm_103a.
//
// Same operator, spin projection and summation order as the FP64 kernel in
// wilson.cu (the hop itself is shared, wilson_device.cuh), but laid out for
// memory traffic instead of FP64 issue.
#include <stdint.h>

#include "wilson_device.cuh"

namespace seedk {

// ---------------------------------------------------------------------------
// FP32 operator of the mixed-precision path.  In FP32 the stencil is bound by
// memory traffic (1368 flop per 480 B per site and column against a balance
// point of ~11 flop/B), so this kernel is laid out for traffic instead:
//  * links are an FP32 copy in structure-of-arrays order, links[(mu*9 + k)*sites + s],
//    so a warp's 32 consecutive sites read 256 contiguous bytes per element;
//  * each thread keeps its two links (U_mu(s), U_mu(s - mu)) in registers and
//    applies them to every column of its block's column group, so the links
//    are read once per group instead of once per column;
//  * inside the solver the FP32 spinors are tiled by 32 sites (Layout32:
//    component k of site s at ((s/32)*12 + k)*32 + s%32), so the 32 lanes of a
//    warp read each component of their 32 neighbours as one or two 256-byte
//    segments; on the caller's site-major layout (seed_apply) spinors are read
//    as float4 (two complex numbers) when 16-byte aligned.
// Same thread layout and summation order as the FP64 kernel: warp mu does the
// two hops of direction mu for 32 sites; the partials meet in shared memory.
// ---------------------------------------------------------------------------
// Read-only loads; L2ONLY loads skip L1 (ld.global.cg) for data no other
// thread of the SM is likely to want soon.
template <bool L2ONLY, class V>
SEED_DEV V ldro(const V *p) {
  if constexpr (L2ONLY) return __ldcg(p);
  else return __ldg(p);
}

template <bool VEC, bool L2ONLY = false>
SEED_DEV void load_spinor(const float2 *__restrict__ p, float2 (&ps)[12]) {
  if constexpr (VEC) {
    const float4 *q = reinterpret_cast<const float4 *>(p);
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const float4 v = ldro<L2ONLY>(q + k);
      ps[2 * k] = make_float2(v.x, v.y);
      ps[2 * k + 1] = make_float2(v.z, v.w);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 12; ++k) ps[k] = ldro<L2ONLY>(p + k);
  }
}

// spinor of site q, tiled layout: 12 components 32 complex apart
template <bool L2ONLY = false>
SEED_DEV void load_spinor_tiled(const float2 *__restrict__ in, int64_t q, float2 (&ps)[12]) {
  const float2 *p = in + (q >> 5) * 384 + (q & 31);
#pragma unroll
  for (int k = 0; k < 12; ++k) ps[k] = ldro<L2ONLY>(p + 32 * k);
}

template <int MU, int S, bool VEC, bool TILED>
SEED_DEV void hops32(const float2 *__restrict__ in, int32_t nf, int32_t nb, const float2 (&uf)[9],
                     const float2 (&ub)[9], unsigned negf, unsigned negb, float2 (&acc)[12]) {
  float2 pf[12], pb[12];
  if constexpr (TILED) {
    load_spinor_tiled(in, nf, pf);
    load_spinor_tiled(in, nb, pb);
  } else {
    load_spinor<VEC>(in + 12 * (int64_t)nf, pf);
    load_spinor<VEC>(in + 12 * (int64_t)nb, pb);
  }
  hop_pair_r<MU, S>(pf, uf, negf, pb, ub, negb, acc);
}

// Lockstep CG's alpha of column c from the blocks' partial sums of p^H q (FP32 per thread, FP64
// above), in block order by the column's last of nb blocks; block: this block's place.
SEED_DEV void dot32(float pq, int c, int64_t block, int nb, const CgDot<float2> &dot, double *sm) {
  double v[1] = {(double)pq};
  block_sum<1, 128>(v, sm);
  double *part = dot.part + (int64_t)c * nb;
  if (threadIdx.x == 0) part[block] = v[0];
  if (!last_block_done(dot.tickets + kColTicket + c, (unsigned)nb)) return;
  const double rho = __ldcg(dot.rho + c);
  const double t = sum_partials<128>(part, nb, 1, 0, sm);
  if (threadIdx.x == 0) dot.alpha[c] = rho / t;
}

template <int S, bool VEC, bool TILED, bool DOT = false>
__global__ void __launch_bounds__(128) k_dslash32(WilsonOp32 op, const float2 *__restrict__ in, int64_t ldi,
                                                  float2 *__restrict__ out, int64_t ldo,
                                                  const int32_t *__restrict__ col_active, int ncols, int group,
                                                  CgDot<float2> dot) {
  __shared__ float sacc[4][24][kWilsonSites + 1];
  __shared__ double sm[4];
  const int lane = threadIdx.x & 31, mu = threadIdx.x >> 5;
  const int64_t s0 = (int64_t)blockIdx.x * kWilsonSites;
  const int64_t s = s0 + lane;
  const bool valid = s < op.sites;
  const int c_begin = blockIdx.y * group;
  const int c_end = min(ncols, c_begin + group);
  int32_t nf = 0, nb = 0;
  unsigned negf = 0u, negb = 0u;
  float2 uf[9], ub[9];
  if (valid) {
    nf = __ldg(op.nbr + 8 * s + 2 * mu);
    nb = __ldg(op.nbr + 8 * s + 2 * mu + 1);
    if (mu == 3 && op.bc_t) {
      const int64_t t = s / ((int64_t)op.dims[0] * op.dims[1] * op.dims[2]);
      if (t == op.dims[3] - 1) negf = CxBits<float2>::sign;
      if (t == 0) negb = CxBits<float2>::sign;
    }
    const float2 *L = op.links + (int64_t)mu * 9 * op.sites;
#pragma unroll
    for (int k = 0; k < 9; ++k) {
      uf[k] = __ldg(L + (int64_t)k * op.sites + s);
      ub[k] = __ldg(L + (int64_t)k * op.sites + nb);
    }
  }
  const float mk = (float)(-op.kappa);
  for (int c = c_begin; c < c_end; ++c) {
    if (col_active != nullptr && col_active[c] == 0) continue;   // uniform over the block
    const float2 *inc = in + (int64_t)c * ldi;
    float2 acc[12];
    if (valid) {
      switch (mu) {
        case 0: hops32<0, S, VEC, TILED>(inc, nf, nb, uf, ub, negf, negb, acc); break;
        case 1: hops32<1, S, VEC, TILED>(inc, nf, nb, uf, ub, negf, negb, acc); break;
        case 2: hops32<2, S, VEC, TILED>(inc, nf, nb, uf, ub, negf, negb, acc); break;
        default: hops32<3, S, VEC, TILED>(inc, nf, nb, uf, ub, negf, negb, acc); break;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[k] = make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      sacc[mu][2 * k][lane] = acc[k].x;
      sacc[mu][2 * k + 1][lane] = acc[k].y;
    }
    __syncthreads();
    const float *ind = reinterpret_cast<const float *>(inc);
    float *outd = reinterpret_cast<float *>(out + (int64_t)c * ldo);
    if constexpr (TILED) {
      // this block's tile: 768 contiguous floats, component k at [64 k, 64 k + 64)
      const int64_t base = (s0 >> 5) * 768;
      const float *pd = DOT ? reinterpret_cast<const float *>(dot.P + (int64_t)c * ldo) : nullptr;
      float pq = 0.f;
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        const int o = threadIdx.x + 128 * q;
        const int k = o >> 6, rem = o & 63, sl = rem >> 1, cc = 2 * k + (rem & 1);
        float v = 0.f;   // padding sites stay zero
        if (s0 + sl < op.sites) {
          const float sum = ((sacc[0][cc][sl] + sacc[1][cc][sl]) + sacc[2][cc][sl]) + sacc[3][cc][sl];
          v = fmaf(mk, sum, __ldg(ind + base + o));
        }
        outd[base + o] = v;
        if constexpr (DOT) pq = fmaf(__ldg(pd + base + o), v, pq);
      }
      if constexpr (DOT) dot32(pq, c, blockIdx.x, gridDim.x, dot, sm);
    } else {
      for (int o = threadIdx.x; o < kWilsonSites * 24; o += 128) {
        const int sl = o / 24, cc = o - 24 * (o / 24);
        const int64_t ss = s0 + sl;
        if (ss >= op.sites) continue;
        const float sum = ((sacc[0][cc][sl] + sacc[1][cc][sl]) + sacc[2][cc][sl]) + sacc[3][cc][sl];
        outd[24 * ss + cc] = fmaf(mk, sum, __ldg(ind + 24 * ss + cc));
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Large lattices (at least kSiteKernelSites sites): one thread per site runs
// all eight hops of its site, for two columns at a time (blockIdx.y = column
// pair), so the four direction partials never leave registers: no shared
// memory exchange and no CTA barrier.  Each link is loaded once per column
// pair and applied to both columns.  Measured on GB300 against the kernel
// above (11 columns): 16^3 x 32 125 us instead of 152, 16^4 62 us instead of
// 80; on small lattices (8^4: 4096 threads) it leaves most SMs idle, so the
// kernel above stays there.
// ---------------------------------------------------------------------------
constexpr int64_t kSiteKernelSites = 65536;

// Layout of the site kernel's input: the solver's, or the caller's (read as float4 where it is aligned)
constexpr int kInTiled = 0, kInSites = 1, kInSites4 = 2;
template <int IN, bool L2ONLY>
SEED_DEV void load_site(const float2 *__restrict__ in, int64_t q, float2 (&ps)[12]) {
  if constexpr (IN == kInTiled) load_spinor_tiled<L2ONLY>(in, q, ps);
  else load_spinor<IN == kInSites4, L2ONLY>(in + 12 * q, ps);
}

// direction MU of site s for the columns set in jm (bit j: column j of the
// pair); MU == 0 starts the sums.  Cache policy: the x and y neighbours of a
// block's sites lie in the block's own or adjacent 32-site tiles, which its
// other hops and its epilogue read again, so they go through L1; the z and t
// neighbours (another plane of the lattice) and the links are used once per
// thread and are read from L2 only, leaving L1 to the reused tiles.  Measured
// on GB300 (11 columns): 16^3 x 32 114.9 -> 103.3 us and 32^3 x 64 1985 ->
// 1879 us together with the streaming stores of the epilogue; same results
// bit for bit.
template <int MU, int S, int IN>
SEED_DEV void site_dir2(const WilsonOp32 &op, const float2 *__restrict__ in, int64_t ldi, int64_t s, int32_t nf,
                        int32_t nb, unsigned negf, unsigned negb, unsigned jm, float2 (&acc)[2][12]) {
  constexpr bool kFar = MU >= 2;
  const float2 *L = op.links + (int64_t)MU * 9 * op.sites;
  {
    float2 u[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) u[k] = __ldcg(L + (int64_t)k * op.sites + s);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (jm & (1u << j)) {
        float2 p[12];
        load_site<IN, kFar>(in + j * ldi, nf, p);
        hop_r<MU, S, true, MU == 0>(p, u, negf, acc[j]);
      }
    }
  }
  {
    float2 u[9];
#pragma unroll
    for (int k = 0; k < 9; ++k) u[k] = __ldcg(L + (int64_t)k * op.sites + nb);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (jm & (1u << j)) {
        float2 p[12];
        load_site<IN, kFar>(in + j * ldi, nb, p);
        hop_r<MU, -S, false, false>(p, u, negb, acc[j]);
      }
    }
  }
}

// Grid: one block per (128 sites, column pair), the pair fastest, so that the
// pairs of one site block run together and their link loads hit L2.
// USER: the result in the caller's site-major layout, staged through shared memory so that
// the stores are contiguous; there the input may be in that layout too (IN).
template <int S, bool DOT = false, bool USER = false, int IN = kInTiled>
__global__ void __launch_bounds__(128, 4) k_dslash32_site(WilsonOp32 op, const float2 *__restrict__ in, int64_t ldi,
                                                          float2 *__restrict__ out, int64_t ldo,
                                                          const int32_t *__restrict__ col_active, int ncols,
                                                          CgDot<float2> dot) {
  const int npairs = (ncols + 1) / 2;
  const int64_t sblock = (int64_t)blockIdx.x / npairs;
  const int c0 = 2 * (int)(blockIdx.x - sblock * npairs);
  unsigned jm = 0u;
#pragma unroll
  for (int j = 0; j < 2; ++j)
    if (c0 + j < ncols && (col_active == nullptr || col_active[c0 + j] != 0)) jm |= 1u << j;
  if (jm == 0u) return;   // uniform over the block
  const int64_t s = sblock * 128 + threadIdx.x;
  const int64_t send = (op.sites + 31) / 32 * 32;
  const bool write = s < send;
  if (!DOT && !USER && !write) return;
  const bool valid = s < op.sites;   // tiled padding sites only write zeros
  in += (int64_t)c0 * ldi;
  out += (int64_t)c0 * ldo;
  float2 acc[2][12];
  if (valid) {
    const int4 *q = reinterpret_cast<const int4 *>(op.nbr + 8 * s);
    const int4 a = __ldg(q), b = __ldg(q + 1);
    unsigned negf = 0u, negb = 0u;
    if (op.bc_t) {
      const int64_t t = s / ((int64_t)op.dims[0] * op.dims[1] * op.dims[2]);
      if (t == op.dims[3] - 1) negf = CxBits<float2>::sign;
      if (t == 0) negb = CxBits<float2>::sign;
    }
    site_dir2<0, S, IN>(op, in, ldi, s, a.x, a.y, 0u, 0u, jm, acc);
    site_dir2<1, S, IN>(op, in, ldi, s, a.z, a.w, 0u, 0u, jm, acc);
    site_dir2<2, S, IN>(op, in, ldi, s, b.x, b.y, 0u, 0u, jm, acc);
    site_dir2<3, S, IN>(op, in, ldi, s, b.z, b.w, negf, negb, jm, acc);
  }
  const float mk = (float)(-op.kappa);
  static_assert(IN == kInTiled || USER, "tiled results come from tiled columns");
  const int64_t so = IN == kInTiled ? (s >> 5) * 384 + (s & 31) : 12 * s;
  constexpr int kStride = IN == kInTiled ? 32 : 1;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    if (!(jm & (1u << j))) continue;
    const float2 *ic = in + j * ldi + so;
    if constexpr (USER) {
      __shared__ float2 stage[128 * 13];   // 12 components per site + 1: conflict-free
      if (valid) {
#pragma unroll
        for (int k = 0; k < 12; ++k) {
          const float2 x = __ldg(ic + kStride * k);
          stage[threadIdx.x * 13 + k] = make_float2(fmaf(mk, acc[j][k].x, x.x), fmaf(mk, acc[j][k].y, x.y));
        }
      }
      __syncthreads();
      float2 *y = out + j * ldo + sblock * (128 * 12);
      const int64_t left = 12 * op.sites - sblock * (128 * 12);
#pragma unroll
      for (int q = 0; q < 12; ++q) {
        const int o = threadIdx.x + 128 * q, sl = o / 12, k = o - 12 * sl;
        if (o < left) __stcs(y + o, stage[sl * 13 + k]);
      }
      __syncthreads();
      continue;
    }
    float2 *oc = out + j * ldo + so;
    float pq = 0.f;
    if (write) {
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        float2 v = make_float2(0.f, 0.f);
        if (valid) {
          const float2 x = __ldg(ic + kStride * k);
          v = make_float2(fmaf(mk, acc[j][k].x, x.x), fmaf(mk, acc[j][k].y, x.y));
          if constexpr (DOT)
            pq = Sc<float2>::redot(__ldg(dot.P + (int64_t)(c0 + j) * ldo + so + kStride * k), v, pq);
        }
        __stcs(oc + kStride * k, v);   // streaming store: this kernel does not read it again
      }
    }
    if constexpr (DOT) {
      __shared__ double sm[4];
      dot32(pq, c0 + j, sblock, gridDim.x / npairs, dot, sm);
    }
  }
}

// Caller's site-major columns -> the tiled layout (padding sites zero): one block of
// 128 threads per 32-site tile and column, through shared memory.  Bound by memory.
__global__ void __launch_bounds__(128) k_tile32(const float2 *__restrict__ in, int64_t ldi, float2 *__restrict__ out,
                                                int64_t ldo, int64_t sites) {
  __shared__ float2 stage[32 * 13];
  const int64_t tile = blockIdx.x;
  const float2 *x = in + (int64_t)blockIdx.y * ldi + tile * 384;
  float2 *y = out + (int64_t)blockIdx.y * ldo + tile * 384;
  const int64_t left = 12 * sites - tile * 384;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int o = threadIdx.x + 128 * q, sl = o / 12, k = o - 12 * sl;
    stage[sl * 13 + k] = o < left ? __ldg(x + o) : make_float2(0.f, 0.f);
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int o = threadIdx.x + 128 * q;
    y[o] = stage[(o & 31) * 13 + (o >> 5)];
  }
}

// links (caller's layout [mu][site][3][3], FP64) -> FP32 structure-of-arrays copy
__global__ void k_links_soa32(const double2 *__restrict__ links, float2 *__restrict__ out, int64_t sites) {
  const int64_t total = 36 * sites;
  for (int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; o < total; o += (int64_t)gridDim.x * blockDim.x) {
    const int64_t s = o % sites, mk = o / sites, mu = mk / 9, k = mk - 9 * mu;
    const double2 v = links[(mu * sites + s) * 9 + k];
    out[o] = make_float2((float)v.x, (float)v.y);
  }
}

void launch_links_soa32(const double2 *links, float2 *out, int64_t sites, cudaStream_t s) {
  int64_t blocks = (36 * sites + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  k_links_soa32<<<(unsigned)blocks, 256, 0, s>>>(links, out, sites);
}

// From 65536 sites on a column in the caller's layout is tiled first and the operator
// works in the tiled layout, which its neighbour loads are contiguous in: A on
// 16^3 x 32 x 12 columns 423 -> 292 us (site-major spinors throughout before).
bool dslash32_tiles(int64_t sites) { return sites >= kSiteKernelSites; }

void launch_tile32(const float2 *in, int64_t ldi, float2 *out, int64_t ldo, int64_t sites, int ncols, cudaStream_t s) {
  k_tile32<<<dim3((unsigned)((sites + 31) / 32), (unsigned)ncols), 128, 0, s>>>(in, ldi, out, ldo, sites);
}

template <int IN>
static void dslash32_user(const WilsonOp32 &op, int sign, const float2 *in, int64_t ldi, float2 *out, int64_t ldo,
                          int ncols, cudaStream_t s) {
  const unsigned g = (unsigned)(((op.sites + 127) / 128) * ((ncols + 1) / 2));
  const CgDot<float2> d{};
  if (sign > 0)
    k_dslash32_site<+1, false, true, IN><<<g, 128, 0, s>>>(op, in, ldi, out, ldo, nullptr, ncols, d);
  else
    k_dslash32_site<-1, false, true, IN><<<g, 128, 0, s>>>(op, in, ldi, out, ldo, nullptr, ncols, d);
}

void launch_wilson_dslash32_user(const WilsonOp32 &op, int sign, const float2 *in, int64_t ldi, bool tiled, float2 *out,
                                 int64_t ldo, int ncols, cudaStream_t s) {
  if (tiled) dslash32_user<kInTiled>(op, sign, in, ldi, out, ldo, ncols, s);
  else if ((uintptr_t)in % 16 == 0 && ldi % 2 == 0) dslash32_user<kInSites4>(op, sign, in, ldi, out, ldo, ncols, s);
  else dslash32_user<kInSites>(op, sign, in, ldi, out, ldo, ncols, s);
}

// Column groups: enough blocks to give every SM about four, otherwise all
// columns of a site block in one group (links read once).
void launch_wilson_dslash32(const WilsonOp32 &op, int sign, const float2 *in, int64_t ldi, float2 *out, int64_t ldo,
                            int ncols, const int32_t *col_active, bool tiled, cudaStream_t s, const CgDot<float2> *dot) {
  const int64_t nsb = (op.sites + kWilsonSites - 1) / kWilsonSites;
  int64_t group = (nsb * ncols) / (152 * 4);
  if (group < 1) group = 1;
  if (group > ncols) group = ncols;
  const int ngroups = (int)((ncols + group - 1) / group);
  const dim3 grid((unsigned)nsb, (unsigned)ngroups);
  const bool vec = ((uintptr_t)in % 16 == 0) && (ldi % 2 == 0);
  const CgDot<float2> d = dot ? *dot : CgDot<float2>{};
  if (tiled && op.sites >= kSiteKernelSites) {   // (the caller's layout: launch_tile32 first)
    const int64_t nthreads = nsb * kWilsonSites;
    const unsigned g2 = (unsigned)(((nthreads + 127) / 128) * ((ncols + 1) / 2));
    if (dot != nullptr) {   // lockstep CG: q = D^H t with alpha
      k_dslash32_site<-1, true><<<g2, 128, 0, s>>>(op, in, ldi, out, ldo, col_active, ncols, d);
    } else if (sign > 0) {
      k_dslash32_site<+1><<<g2, 128, 0, s>>>(op, in, ldi, out, ldo, col_active, ncols, d);
    } else {
      k_dslash32_site<-1><<<g2, 128, 0, s>>>(op, in, ldi, out, ldo, col_active, ncols, d);
    }
    return;
  }
  const int g = (int)group;
  if (dot != nullptr) {
    k_dslash32<-1, false, true, true><<<grid, 128, 0, s>>>(op, in, ldi, out, ldo, col_active, ncols, g, d);
  } else if (tiled) {
    if (sign > 0) k_dslash32<+1, false, true><<<grid, 128, 0, s>>>(op, in, ldi, out, ldo, col_active, ncols, g, d);
    else k_dslash32<-1, false, true><<<grid, 128, 0, s>>>(op, in, ldi, out, ldo, col_active, ncols, g, d);
  } else if (sign > 0) {
    if (vec) k_dslash32<+1, true, false><<<grid, 128, 0, s>>>(op, in, ldi, out, ldo, col_active, ncols, g, d);
    else k_dslash32<+1, false, false><<<grid, 128, 0, s>>>(op, in, ldi, out, ldo, col_active, ncols, g, d);
  } else {
    if (vec) k_dslash32<-1, true, false><<<grid, 128, 0, s>>>(op, in, ldi, out, ldo, col_active, ncols, g, d);
    else k_dslash32<-1, false, false><<<grid, 128, 0, s>>>(op, in, ldi, out, ldo, col_active, ncols, g, d);
  }
}

}  // namespace seedk
