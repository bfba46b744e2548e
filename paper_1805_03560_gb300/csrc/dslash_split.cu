// Hemi-Dslash with one thread per site and direction, for lattices too small
// to fill the GPU with one thread per site (the operator and its algebra:
// dslash.cu).
//
// A block takes 32 consecutive sites and four warps; warp mu holds the two
// hops of direction mu of every site.  Each thread loads both neighbour
// spinors and both links at once, accumulates the two hops, and leaves the
// twelve components in shared memory; after one barrier the warps add the
// four directions of each output component and run the epilogue on one
// 16-byte chunk per thread.
//
// What bounds the small lattices is latency: one thread per site waits for
// eight hops' loads one after another, on a GPU mostly empty (8^3 x 16: 32
// blocks of 128 threads on 152 SMs).  Here a site's loads are all in flight,
// every SM has work from 4864 sites on, and inside a solve the loads of the
// links, which none of its launches writes, are issued before the wait for
// the launch before (links_ready).  Measured (one thread per site -> this
// kernel) on 8^3 x 16, 14 x 6 x 10 x 20 and 12^3 x 24: a CG iteration in FP32
// 29.7 -> 20.5, 30.0 -> 23.0 and 35.8 -> 28.0 us, in FP64 156 -> 58, 183 -> 96 and
// 286 -> 198 us; the emulated-FP64 hop 14.1 -> 9.0, 16.9 -> 10.0 and 26.5 -> 15.1 us.
// (One thread per hop, eight warps to 32 sites, was slower for FP32: 38.6 us per
// iteration on 12^3 x 24 against 36.8 with one thread per site then; the
// barrier's traffic doubles.)
#include "dslash_ops.cuh"
#include "hmc_host.h"

namespace hmc {

namespace {

constexpr int SPLIT_SITES = 32;
constexpr int SPLIT_NT = 4 * SPLIT_SITES;

// 16-byte chunk c of element s: CPC complex components per chunk
template <int P>
struct ChunkIO;
template <>
struct ChunkIO<HMC_F32> {
  using R = float;
  static constexpr int CPC = 2;
  static __device__ __forceinline__ void load(const void *b, int S, int c, int s, Cx<float> v[2]) {
    const float4 t = *((const float4 *)b + f32_chunk<6>(S, c, s));
    v[0] = {t.x, t.y};
    v[1] = {t.z, t.w};
  }
  static __device__ __forceinline__ void store(void *b, int S, int c, int s, const Cx<float> v[2]) {
    *((float4 *)b + f32_chunk<6>(S, c, s)) = make_float4(v[0].re, v[0].im, v[1].re, v[1].im);
  }
};
template <>
struct ChunkIO<HMC_F64> {
  using R = double;
  static constexpr int CPC = 1;
  static __device__ __forceinline__ void load(const void *b, int S, int c, int s, Cx<double> v[1]) {
    const double2 t = *((const double2 *)b + (size_t)c * S + s);
    v[0] = {t.x, t.y};
  }
  static __device__ __forceinline__ void store(void *b, int S, int c, int s, const Cx<double> v[1]) {
    *((double2 *)b + (size_t)c * S + s) = make_double2(v[0].re, v[0].im);
  }
};
template <>
struct ChunkIO<HMC_F64E> {
  using R = df64;
  static constexpr int CPC = 1;
  static __device__ __forceinline__ void load(const void *b, int S, int c, int s, Cx<df64> v[1]) {
    const float4 t = *((const float4 *)b + (size_t)c * S + s);
    v[0] = {df64(t.x, t.y), df64(t.z, t.w)};
  }
  static __device__ __forceinline__ void store(void *b, int S, int c, int s, const Cx<df64> v[1]) {
    *((float4 *)b + (size_t)c * S + s) = make_float4(v[0].re.hi, v[0].re.lo, v[0].im.hi,
                                                     v[0].im.lo);
  }
};

// fermion boundary sign of a hop in time that wraps around
template <typename R>
__device__ __forceinline__ void flip(bool wrap, Cx<R> h[6]) {
  if (wrap) {
#pragma unroll
    for (int k = 0; k < 6; ++k) h[k] = -h[k];
  }
}

template <int SP>
constexpr int split_min_blocks() {
  return SP == HMC_F32 ? 5 : 3;
}

template <int SP, int FMT, bool DAG>
__global__ void __launch_bounds__(SPLIT_NT, split_min_blocks<SP>()) k_dslash_split(
    const DslashArgs a) {
  using SIO = SpinorIO<SP>;
  using R = typename SIO::R;
  using LIO = LinkIO<SP, FMT>;
  using CIO = ChunkIO<SP>;
  constexpr int SF = DAG ? -1 : 1;
  constexpr int CPC = CIO::CPC, NCH = 12 / CPC;
  __shared__ __align__(16) Cx<R> s_w[4][NCH][SPLIT_SITES][CPC];
  __shared__ R s_n[4][SPLIT_SITES];
  griddep_launch_dependents();
  const int mu = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int Vh = a.g.Vh;
  if (a.red_src && blockIdx.x == gridDim.x - 1) {
    // the block after the lattice's: sum the partials of the launch before
    griddep_wait();
    if (a.gate && *a.gate == 0) return;
    const double rr = a.red_alpha ? *a.red_rr : 0.0;
    const double t = block_sum_partials<SPLIT_NT>(a.red_src, a.red_n);
    if (threadIdx.x == 0) {
      *a.red_dst = t;
      if (a.red_alpha) {
        const double al = rr / t;
        *a.red_alpha = al;
        if (!isfinite(al) || !(t > 0.0)) *a.red_flag = 2;
      }
    }
    return;
  }
  const int i = blockIdx.x * SPLIT_SITES + lane;
  const bool in = i < Vh;
  const int is = in ? i : Vh - 1;  // threads past the end work on the last site and store nothing
  int c[4];
  const int lex = site_coords(a.g, is, a.p, c);
  const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
  const int Lm = a.g.L[mu], stm = a.g.st[mu];
  const int hf = (lex + (cm + 1 == Lm ? 1 - Lm : 1) * stm) >> 1;
  const int hb = (lex + (cm == 0 ? Lm - 1 : -1) * stm) >> 1;
  const bool wf = mu == 0 && cm + 1 == Lm, wb = mu == 0 && cm == 0;
  const void *gf = link_base<SP, FMT>(a.gauge, Vh, a.p, mu);
  const void *gb = link_base<SP, FMT>(a.gauge, Vh, 1 - a.p, mu);
  // loads that depend on nothing computed here are issued before the gate is
  // looked at and before the hops: the epilogue's fields, the factor alpha
  constexpr int NE = (NCH + 3) / 4;  // chunks per thread in the epilogue
  constexpr bool EARLY = SP == HMC_F32;
  Cx<R> xe[NE][CPC], re[NE][CPC];
  const auto load_epilogue = [&] {
#pragma unroll
    for (int e = 0; e < NE; ++e)
      if (mu + 4 * e < NCH) {
        if (a.x) CIO::load(a.x, Vh, mu + 4 * e, is, xe[e]);
        if (a.cg_r) CIO::load(a.cg_r, Vh, mu + 4 * e, is, re[e]);
      }
  };
  double alpha_d = 0.0;
  Cx<R> acc[12];
  if constexpr (SP == HMC_F64E) {
    griddep_wait();
    if (a.gate && *a.gate == 0) return;
    AccE2 e2;
    if constexpr (FMT != 18) {
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[k] = {R(0), R(0)};
    }
#pragma unroll 1
    for (int d = 0; d < 2; ++d) {
      const int S = d ? -SF : SF;
      if constexpr (FMT == 18) {
        const float4 *in = (const float4 *)a.in + (d ? hb : hf);
        const float4 *lk = (const float4 *)(d ? gb : gf) + (d ? hb : is);
        float4 p[12];
#pragma unroll
        for (int k = 0; k < 12; ++k) p[k] = __ldg(in + (size_t)k * Vh);
        const size_t sr = (size_t)(d ? 1 : 3) * Vh, sc = (size_t)(d ? 3 : 1) * Vh;
        hop_e2(p, [] {}, [&](int r, int k) { return __ldg(lk + r * sr + k * sc); }, mu, d == 0,
               S, d ? wb : wf, d == 0, e2);
      } else {
        Cx<R> psi[12], u[9], hs[6], w[6];
        SIO::load(a.in, Vh, d ? hb : hf, psi);
        LIO::load(d ? gb : gf, Vh, d ? hb : is, u);
        project_rt(mu, S, psi, hs);
        flip(d ? wb : wf, hs);
        if (d)
          mul_link_dag(u, hs, w);
        else
          mul_link(u, hs, w);
        accumulate_rt(mu, S, acc, w);
      }
    }
    if constexpr (FMT == 18) unpack_e2(e2, acc);
  } else {
    Cx<R> uf[9], ub[9], pf[12], pb[12], hs[6], w[6];
    if (!a.links_ready) griddep_wait();
    LIO::load(gf, Vh, is, uf);
    LIO::load(gb, Vh, hb, ub);
    if (a.links_ready) griddep_wait();
    const int live = a.gate ? *a.gate : 1;
    SIO::load(a.in, Vh, hf, pf);
    SIO::load(a.in, Vh, hb, pb);
    if (a.cg_r) alpha_d = *a.cg_alpha;
    if constexpr (EARLY) load_epilogue();
    if (!live) return;
    project_mu<SF>(mu, pf, hs);
    flip(wf, hs);
    mul_link(uf, hs, w);
    spread_mu<SF>(mu, acc, w);
    project_mu<-SF>(mu, pb, hs);
    flip(wb, hs);
    mul_link_dag(ub, hs, w);
    accumulate_mu<-SF>(mu, acc, w);
  }
#pragma unroll
  for (int k = 0; k < NCH; ++k)
#pragma unroll
    for (int j = 0; j < CPC; ++j) s_w[mu][k][lane][j] = acc[k * CPC + j];
  if constexpr (!EARLY) load_epilogue();
  __syncthreads();
  R n2 = R(0);
  if (in) {
    const R cb = (R)a.cb, ca = (R)a.ca, alpha = (R)alpha_d;
#pragma unroll
    for (int e = 0; e < NE; ++e) {
      const int ch = mu + 4 * e;
      if (ch >= NCH) break;
      Cx<R> t[CPC];
#pragma unroll
      for (int j = 0; j < CPC; ++j)
        t[j] = ((s_w[0][ch][lane][j] + s_w[1][ch][lane][j]) + s_w[2][ch][lane][j]) +
               s_w[3][ch][lane][j];
      if (a.x) {
#pragma unroll
        for (int j = 0; j < CPC; ++j) {
          t[j].re = fma(ca, xe[e][j].re, cb * t[j].re);
          t[j].im = fma(ca, xe[e][j].im, cb * t[j].im);
        }
      } else {
#pragma unroll
        for (int j = 0; j < CPC; ++j) t[j] = cb * t[j];
      }
      if (a.cg_r) {
        // fused CG step: r -= alpha A p (A p = t is not stored)
#pragma unroll
        for (int j = 0; j < CPC; ++j) {
          t[j].re = fma(-alpha, t[j].re, re[e][j].re);
          t[j].im = fma(-alpha, t[j].im, re[e][j].im);
        }
        CIO::store(a.cg_r, Vh, ch, i, t);
      } else {
        CIO::store(a.out, Vh, ch, i, t);
      }
#pragma unroll
      for (int j = 0; j < CPC; ++j) n2 += norm2(t[j]);
    }
  }
  if (a.partials) {
    // |out|^2 of a site in the arithmetic precision, across sites in double
    // (by one warp: FP64 additions are scarce on this GPU)
    s_n[mu][lane] = n2;
    __syncthreads();
    if (mu == 0) {
      double s = (double)((s_n[0][lane] + s_n[1][lane]) + (s_n[2][lane] + s_n[3][lane]));
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
      if (lane == 0) a.partials[blockIdx.x] = s;
    }
  }
}

// Native FP64 is bound by the FP64 pipe of the SM a block runs on.  A launch
// that may start while the one before still runs gets its blocks placed on
// whichever SMs have room then, several on one SM while others stay empty; of
// a grid that would spread evenly over the SMs (half as many blocks as SMs and
// more, within one wave) that costs more than the gap between launches.  CG
// iteration with / without early launch: 64 blocks 55 / 57 us, 128 blocks 79 / 56,
// 263 blocks 121 / 92, 648 blocks 194 / 197.  (FP32 and emulated FP64 gain from
// the early launch at every size: 8^3 x 16 19.5 / 21.1 us.)
template <int SP>
bool early_launch(const DslashArgs &a, int nb, int sms) {
  if (SP == HMC_F64 && nb > sms / 2 && nb <= split_min_blocks<SP>() * sms) return false;
  return a.pdl != 0;
}

template <int SP, int FMT>
void launch_fmt(const DslashArgs &a, int dagger, int sms, cudaStream_t st) {
  const int nb = blocks_for(a.g.Vh, SPLIT_SITES) + (a.red_src ? 1 : 0);
  const bool pdl = early_launch<SP>(a, nb, sms);
  if (dagger)
    launch_pdl(k_dslash_split<SP, FMT, true>, nb, SPLIT_NT, st, pdl, a);
  else
    launch_pdl(k_dslash_split<SP, FMT, false>, nb, SPLIT_NT, st, pdl, a);
}

}  // namespace

int dslash_split_blocks(const Geo &g) { return blocks_for(g.Vh, SPLIT_SITES); }

// The sites of the fullest SM decide: 32-site blocks spread the lattice
// finer than 128-site blocks, at a cost per site (coordinates four times, the
// exchange).  Measured on 152 SMs, this kernel / one thread per site (the
// default variant), by sites per parity:
//   FP32, 12-real links, per CG iteration: 20736 28.0 / 35.8 us, 24192 28.1 /
//     35.2 (the last size in one wave of five blocks per SM), 24576 33.0 / 35.2,
//     28672 37.3 / 38.1, 31104 36.3 / 36.7, 34560 37.3 / 36.9, 38016 38.2 /
//     36.2: up to 208 sites per SM, in the second wave until the two meet.
//   FP32, 18-real links: 20736 30.3 / 35.9, 24192 30.4 / 35.1, 24576 35.5 / 35.2,
//     27648 38.2 / 36.7, 36864 41.5 / 37.3: up to 160 sites per SM, one wave.
//   emulated FP64, 18-real links, per hop: 20736 15.1 / 26.5, 40960 26.0 / 27.9,
//     42336 26.7 / 28.5, 44352 29.0 / 28.5, 49152 31.2 / 27.6: up to 288 sites per
//     SM, three waves of three blocks.
//   emulated FP64, 12-real links, per hop: 20736 18.1 / 36.0, 40960 29.6 / 38.2,
//     57344 40.5 / 42.2: up to 384 sites per SM, one wave of the other kernel.
//   FP64, per CG iteration: 20736 198 / 286, 24576 231 / 287, 34560 302 / 290,
//     40960 338 / 421, 55296 440 / 422: where the fullest SM gets a fifth fewer
//     sites (the cost per site is 4 to 6 % higher here; with fewer than a fifth
//     the gain is 4 to 8 %: 49152 407 / 424, 65536 514 / 553).
// Half storage has no form of this kernel.  Per-right-hand-side factors and totals
// (the batched CG's) are not part of it.
bool dslash_split_rule(const hmc_ctx *ctx, const DslashArgs &a, int sprec, int fmt) {
  if (a.n_rhs != 1 || a.cb_rhs || a.total) return false;
  const long long Vh = a.g.Vh, sms = ctx->sm_count;
  switch (sprec) {
    case HMC_F32: return Vh <= (fmt == 18 ? 160 : 208) * sms;
    case HMC_F64E: return Vh <= (fmt == 18 ? 288 : 384) * sms;
    case HMC_F64: {
      const long long fine = (Vh + SPLIT_SITES * sms - 1) / (SPLIT_SITES * sms) * SPLIT_SITES;
      const long long coarse = (Vh + DS_NT * sms - 1) / (DS_NT * sms) * DS_NT;
      return 5 * fine < 4 * coarse;
    }
    default: return false;
  }
}

bool launch_dslash_split(const hmc_ctx *ctx, const DslashArgs &a, int sprec, int fmt, int dagger) {
  const int sms = ctx->sm_count;
  cudaStream_t st = ctx->stream;
  switch (sprec * 100 + fmt) {
    case HMC_F64 * 100 + 18: launch_fmt<HMC_F64, 18>(a, dagger, sms, st); return true;
    case HMC_F64 * 100 + 12: launch_fmt<HMC_F64, 12>(a, dagger, sms, st); return true;
    case HMC_F32 * 100 + 18: launch_fmt<HMC_F32, 18>(a, dagger, sms, st); return true;
    case HMC_F32 * 100 + 12: launch_fmt<HMC_F32, 12>(a, dagger, sms, st); return true;
    case HMC_F64E * 100 + 18: launch_fmt<HMC_F64E, 18>(a, dagger, sms, st); return true;
    case HMC_F64E * 100 + 12: launch_fmt<HMC_F64E, 12>(a, dagger, sms, st); return true;
    default: return false;
  }
}

}  // namespace hmc
