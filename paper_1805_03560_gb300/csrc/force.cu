// Pseudo-fermion force kernel: the link derivative of 2 kappa^2 Re(W^dag H V)
// for full-lattice fields W, V (given as even and odd halves).
//
// Sec. II: delta S_PF = -X^dag delta M Y + h.c.  On even sites with
// Mhat = 1 - kappa^2 H_eo H_oe this becomes kappa^2 (W^dag delta H V + h.c.)
// with W = (Y, H_eo^dag Y), V = (X, H_oe X); the filtered action of Sec. II
// (Horner scheme) is a sum of such terms.
//
// The link U_{x,mu} enters H in the block (x, x+mu) as s (1 - gamma_mu) U and
// in (x+mu, x) as s (1 + gamma_mu) U^dag (s: fermion boundary sign).  For
// delta U = omega U the variation is s Tr(omega Q) with
//   Q = U A - B U^dag,
//   A = sum_spin V_{x+mu} ((1 - gamma_mu) W_x)^dag,
//   B = sum_spin V_x ((1 + gamma_mu) W_{x+mu})^dag.
// With the projector P = 1 - gamma_mu (or 1 + gamma_mu) of rank two, the spin
// sum equals the sum over the two independent components of the projected
// half spinors, so A and B are each two colour outer products of projected
// half spinors.  F_a = 2 kappa^2 Re Tr(T_a Q) = -kappa^2 Im Tr(lambda_a Q).
#include "dslash_ops.cuh"
#include "hmc_host.h"

namespace hmc {

// f_a = Im Tr(lambda_a Q)
template <typename R>
__device__ __forceinline__ void im_tr_lambda(const Cx<R> q[9], double f[8]) {
  const double r3 = 0.57735026918962576451;  // 1/sqrt(3)
  f[0] = (double)q[3].im + (double)q[1].im;
  f[1] = (double)q[1].re - (double)q[3].re;
  f[2] = (double)q[0].im - (double)q[4].im;
  f[3] = (double)q[6].im + (double)q[2].im;
  f[4] = (double)q[2].re - (double)q[6].re;
  f[5] = (double)q[7].im + (double)q[5].im;
  f[6] = (double)q[5].re - (double)q[7].re;
  f[7] = ((double)q[0].im + (double)q[4].im - 2.0 * (double)q[8].im) * r3;
}

// Up to HF_MAX pairs (W_q, V_q) per launch: Q is linear in the pair, so the
// kernel sums A and B over the pairs and multiplies by the link, projects and
// updates F once (the filtered force of Sec. II is a sum of n_t + 1 pairs;
// one launch reads the links and reads and writes F once for all of them).
constexpr int HF_MAX = 32;

struct HopForceArgs {
  Geo g;
  const void *gauge;      // links in the precision of the fields
  int n;                  // pairs
  const void *W[HF_MAX][2];  // W even, W odd
  const void *V[HF_MAX][2];  // V even, V odd
  double *F;              // algebra field
  double c;               // F_a += c * (-Im Tr(lambda_a Q)) ; c = coeff * kappa^2
};

// One thread per link: a block takes 32 consecutive sites of one parity and
// four warps, warp mu the links of direction mu, so that the four directions
// read the site's own spinors through L1.  Since Im Tr(lambda_a X^dag) =
// -Im Tr(lambda_a X) for Hermitian lambda_a, Q may be replaced by
//   U C,  C = A + B^dag = sum_q sum_s (hv (x) hw^*  +  hw' (x) hv'^*)
// with the projected half spinors hv = P- V_{x+mu}, hw = P- W_x, hv' = P+ V_x,
// hw' = P+ W_{x+mu}: one 3x3 accumulator and one product with the link.
constexpr int HF_SITES = 32;
constexpr int HF_NT = 4 * HF_SITES;

template <int FMT, int SP>
__device__ __forceinline__ void add_force(const HopForceArgs &a, int p, int mu, int h, double sg,
                                          const Cx<RT<SP>> C[9]) {
  using R = RT<SP>;
  const int Vh = a.g.Vh;
  Cx<R> u[9], Q[9];
  LinkIO<SP, FMT>::load(link_base<SP, FMT>(a.gauge, Vh, p, mu), Vh, h, u);
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      Cx<R> t = u[i * 3] * C[j];
      t = fmac(t, u[i * 3 + 1], C[3 + j]);
      t = fmac(t, u[i * 3 + 2], C[6 + j]);
      Q[i * 3 + j] = t;
    }
  double f[8];
  im_tr_lambda(Q, f);
  double *F = a.F + (size_t)(p * 4 + mu) * 8 * Vh + h;
  const double cf = -a.c * sg;
#pragma unroll
  for (int k = 0; k < 8; ++k) F[(size_t)k * Vh] += cf * f[k];
}

// the link of this thread; false past the end of the lattice
__device__ __forceinline__ bool force_link(const HopForceArgs &a, int &p, int &mu, int &h, int &hn,
                                           double &sg) {
  const int nbp = (a.g.Vh + HF_SITES - 1) / HF_SITES;
  p = (int)blockIdx.x >= nbp ? 1 : 0;
  mu = threadIdx.x >> 5;
  h = (blockIdx.x - p * nbp) * HF_SITES + (threadIdx.x & 31);
  if (h >= a.g.Vh) return false;
  int c[4];
  const int lex = site_coords(a.g, h, p, c);
  const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
  hn = (lex + (cm + 1 == a.g.L[mu] ? 1 - a.g.L[mu] : 1) * a.g.st[mu]) >> 1;
  sg = (mu == 0 && cm + 1 == a.g.L[0]) ? -1.0 : 1.0;
  return true;
}

template <int FMT, int SP>
__global__ void __launch_bounds__(HF_NT) k_hop_force(const HopForceArgs a) {
  using R = RT<SP>;
  using SIO = SpinorIO<SP>;
  int p, mu, h, hn;
  double sg;
  if (!force_link(a, p, mu, h, hn, sg)) return;
  const int Vh = a.g.Vh;
  Cx<R> s[12], hv[6], hw[6], C[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) C[k] = {R(0), R(0)};
  const auto outer = [&](const Cx<R> x[6], const Cx<R> y[6]) {
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
      for (int j = 0; j < 3; ++j)
        C[i * 3 + j] = fmacj(fmacj(C[i * 3 + j], y[j], x[i]), y[3 + j], x[3 + i]);
  };
#pragma unroll 1
  for (int q = 0; q < a.n; ++q) {
    SIO::load(a.V[q][1 - p], Vh, hn, s);
    project_mu<+1>(mu, s, hv);
    SIO::load(a.W[q][p], Vh, h, s);
    project_mu<+1>(mu, s, hw);
    outer(hv, hw);
    SIO::load(a.V[q][p], Vh, h, s);
    project_mu<-1>(mu, s, hv);
    SIO::load(a.W[q][1 - p], Vh, hn, s);
    project_mu<-1>(mu, s, hw);
    outer(hw, hv);
  }
  add_force<FMT, SP>(a, p, mu, h, sg, C);
}

// Emulated FP64: the spin sum of an outer product in the two lanes of the
// paired arithmetic (df64x2.cuh), the lanes added at the end; while one outer
// product is computed the two spinors of the next come into the thread's own
// slots of shared memory.
constexpr int HF_SMEM = 24 * HF_NT * 16;

// Projection (1 - s gamma_mu) of the spinor in the 12 slots, mu and s at run
// time: h = u + t, t a signed exchange of the lower spins and of real and
// imaginary parts (project_e2), made by the addresses of the loads and by sign
// masks, so that one copy of the code serves every direction and both signs
// (with a copy for each the loop outgrows the instruction cache: 3.4 of 8.3
// stall cycles per issue).
struct ProjMasks {
  f32x2 re, im;  // signs of t
  int d0, d1;    // byte offsets of the lower components of lanes 0 and 1
  int tr, ti;    // byte offsets of t's parts within a slot
};
__device__ __forceinline__ ProjMasks proj_masks(int mu, bool plus) {
  const f32x2 S = plus ? kNegBoth : 0ull;
  const bool swap = mu == 1 || mu == 2, cross = mu & 1;
  ProjMasks m;
  m.re = S ^ (mu == 0 || mu == 1 ? kNegBoth : mu == 2 ? kNeg1 : kNeg0);
  m.im = S ^ (mu == 0 ? kNegBoth : mu == 1 ? 0ull : kNeg1);
  m.d0 = (swap ? 9 : 6) * HF_NT * 16;
  m.d1 = (swap ? 6 : 9) * HF_NT * 16;
  m.tr = cross ? 8 : 0;
  m.ti = cross ? 0 : 8;
  return m;
}
__device__ __forceinline__ void project_slots(const float4 *slot, const ProjMasks &m, cdd2 h[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float4 u0 = slot[a * HF_NT], u1 = slot[(3 + a) * HF_NT];
    const char *d0 = (const char *)(slot + a * HF_NT) + m.d0;
    const char *d1 = (const char *)(slot + a * HF_NT) + m.d1;
    const float2 r0 = *(const float2 *)(d0 + m.tr), r1 = *(const float2 *)(d1 + m.tr);
    const float2 i0 = *(const float2 *)(d0 + m.ti), i1 = *(const float2 *)(d1 + m.ti);
    const dd2 tr = flip2(dd2{pk2(r0.x, r1.x), pk2(r0.y, r1.y)}, m.re);
    const dd2 ti = flip2(dd2{pk2(i0.x, i1.x), pk2(i0.y, i1.y)}, m.im);
    h[a] = {add(dd2{pk2(u0.x, u1.x), pk2(u0.y, u1.y)}, tr),
            add(dd2{pk2(u0.z, u1.z), pk2(u0.w, u1.w)}, ti)};
  }
}

template <int FMT>
__global__ void __launch_bounds__(HF_NT, 3) k_hop_force_e2(const HopForceArgs a) {
  extern __shared__ __align__(16) float4 s_buf[];
  int p, mu, h, hn;
  double sg;
  if (!force_link(a, p, mu, h, hn, sg)) return;
  const int Vh = a.g.Vh;
  float4 *slot = s_buf + threadIdx.x;
  cdd2 C[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) C[k] = {{0ull, 0ull}, {0ull, 0ull}};
  // stage t: outer product t & 1 of pair t / 2, x in slots 0..11, y in 12..23
  const auto fetch = [&](int t) {
    const int q = t >> 1;
    const float4 *x = (const float4 *)((t & 1) ? a.W[q][1 - p] : a.V[q][1 - p]) + hn;
    const float4 *y = (const float4 *)((t & 1) ? a.V[q][p] : a.W[q][p]) + h;
#pragma unroll
    for (int k = 0; k < 12; ++k) cp_async16(slot + k * HF_NT, x + (size_t)k * Vh);
#pragma unroll
    for (int k = 0; k < 12; ++k) cp_async16_l1(slot + (12 + k) * HF_NT, y + (size_t)k * Vh);
  };
  fetch(0);
#pragma unroll 1
  for (int t = 0; t < 2 * a.n; ++t) {
    cdd2 x[3], y[3];
    cp_async_wait();
    const ProjMasks m = proj_masks(mu, t & 1);
    project_slots(slot, m, x);
    project_slots(slot + 12 * HF_NT, m, y);
    if (t + 1 < 2 * a.n) fetch(t + 1);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const cneg2 n = {flip2(y[j].re, kNegBoth), y[j].im};
      const cdd2 v = {y[j].re, flip2(y[j].im, kNegBoth)};  // conj
#pragma unroll
      for (int i = 0; i < 3; ++i) C[i * 3 + j] = cmac(C[i * 3 + j], x[i], v, n);
    }
  }
  Cx<df64> Cs[9];
#pragma unroll
  for (int k = 0; k < 9; ++k)
    Cs[k] = {first(C[k].re) + second(C[k].re), first(C[k].im) + second(C[k].im)};
  add_force<FMT, HMC_F64E>(a, p, mu, h, sg, Cs);
}

template <int FMT>
static void launch_hop_force_e2(const HopForceArgs &a, int nb, cudaStream_t st) {
  k_hop_force_e2<FMT><<<nb, HF_NT, HF_SMEM, st>>>(a);
}

cudaError_t hop_force_smem() {
  const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const cudaError_t e = cudaFuncSetAttribute(k_hop_force_e2<18>, at, HF_SMEM);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(k_hop_force_e2<12>, at, HF_SMEM);
}

int hop_force(hmc_ctx *ctx, const Geo &g, const hmc_gauge &U, const void *We, const void *Wo,
              const void *Ve, const void *Vo, double *F, double c, int sprec) {
  const void *W[1][2] = {{We, Wo}}, *V[1][2] = {{Ve, Vo}};
  return hop_force_multi(ctx, g, U, 1, W, V, F, c, sprec);
}

int hop_force_multi(hmc_ctx *ctx, const Geo &g, const hmc_gauge &U, int n, const void *const W[][2],
                    const void *const V[][2], double *F, double c, int sprec) {
  if (sprec != HMC_F64 && sprec != HMC_F32 && sprec != HMC_F64E)
    return fail(ctx, HMC_EINVAL, "force: spinor precision must be F64, F32 or F64E");
  if (U.prec != sprec)
    return fail(ctx, HMC_EINVAL, "force: gauge precision must match the fields");
  if (n < 1) return HMC_OK;
  if (n > HF_MAX) {
    // in chunks of HF_MAX pairs
    for (int q0 = 0; q0 < n; q0 += HF_MAX) {
      int st = hop_force_multi(ctx, g, U, n - q0 < HF_MAX ? n - q0 : HF_MAX, W + q0, V + q0, F, c,
                               sprec);
      if (st) return st;
    }
    return HMC_OK;
  }
  HopForceArgs a{};
  a.g = g;
  a.gauge = U.data;
  a.n = n;
  for (int q = 0; q < n; ++q)
    for (int h = 0; h < 2; ++h) {
      a.W[q][h] = W[q][h];
      a.V[q][h] = V[q][h];
    }
  a.F = F;
  a.c = c;
  const int nb = 2 * blocks_for(g.Vh, HF_SITES);
  cudaStream_t st = ctx->stream;
  switch (sprec * 100 + U.fmt) {
    case HMC_F64 * 100 + 18: k_hop_force<18, HMC_F64><<<nb, HF_NT, 0, st>>>(a); break;
    case HMC_F64 * 100 + 12: k_hop_force<12, HMC_F64><<<nb, HF_NT, 0, st>>>(a); break;
    case HMC_F32 * 100 + 18: k_hop_force<18, HMC_F32><<<nb, HF_NT, 0, st>>>(a); break;
    case HMC_F32 * 100 + 12: k_hop_force<12, HMC_F32><<<nb, HF_NT, 0, st>>>(a); break;
    // emulated FP64: the outer products and U (A + B^dag) in double-float
    case HMC_F64E * 100 + 18: launch_hop_force_e2<18>(a, nb, st); break;
    case HMC_F64E * 100 + 12: launch_hop_force_e2<12>(a, nb, st); break;
    default: return fail(ctx, HMC_EINVAL, "force: bad link format %d", U.fmt);
  }
  return launched(ctx, sprec == HMC_F64 ? "hop_force_f64"
                       : sprec == HMC_F32 ? "hop_force_f32" : "hop_force_f64e");
}

}  // namespace hmc
