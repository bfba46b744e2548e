// Hemi-Dslash in emulated FP64 (double-float) with 18-real links, one thread
// per output site and right-hand side: the operator of dslash.cu in the paired
// arithmetic of df64x2.cuh.
//
// What bounds it is the FP32 pipe: about 700 paired operations (two pipe
// cycles each) per hop, 103 of the 139 us of a hop on 24^3 x 48; three-register
// operands and register banks keep the pipe from more than about three quarters
// (sixteen warps per SM in 128 registers: 164 us, twelve: 160).  The eight hops
// run in a loop, and while one is computed the next hop's spinor and link come
// into the thread's own slots of shared memory (cp.async; the links in two
// buffers, the spinor's slots are free once it is projected), 165 -> 160 us.  No
// barrier: every thread reads what it asked for itself.  Measured against the
// scalar double-float form: 24^3 x 48 184 -> 160 us, 32^3 x 64 567 -> 477 us.  Without
// the reductions of dslash.cu, which nothing asks for in this precision (4 KB of
// shared memory, six registers), 158 -> 139 us and 406 us.
#include "dslash_ops.cuh"
#include "hmc_host.h"

namespace hmc {

namespace {

constexpr int E2_SLOTS = 12 + 2 * 9;  // 16-byte slots per thread
constexpr int E2_SMEM = E2_SLOTS * DS_NT * 16;

template <bool DAG>
__global__ void __launch_bounds__(DS_NT, 3) k_dslash_e2(const DslashArgs a) {
  constexpr int SF = DAG ? -1 : 1;
  using SIO = SpinorIO<HMC_F64E>;
  using R = df64;
  extern __shared__ __align__(16) float4 s_buf[];
  griddep_launch_dependents();
  griddep_wait();
  if (a.gate && *a.gate == 0) return;
  const int Vh = a.g.Vh, S_ = Vh * a.n_rhs;
  const int blk = ds_block(a, blockIdx.x), i = blk * DS_NT + threadIdx.x;
  if (i < S_) {
    const int h = a.n_rhs == 1 ? i : i / a.n_rhs;
    const int r = i - h * a.n_rhs;
    int c[4];
    const int lex = site_coords(a.g, h, a.p, c);
    float4 *slot = s_buf + threadIdx.x;  // slot k at slot[k * DS_NT]
    const auto fetch = [&](int k) {
      const int mu = k >> 1;
      const bool fwd = (k & 1) == 0;
      const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
      const int L = a.g.L[mu];
      const int d = fwd ? (cm + 1 == L ? 1 - L : 1) : (cm == 0 ? L - 1 : -1);
      const int hn = (lex + d * a.g.st[mu]) >> 1;
      const float4 *in = (const float4 *)a.in + (size_t)hn * a.n_rhs + r;
      const float4 *lk =
          (const float4 *)link_base<HMC_F64E, 18>(a.gauge, Vh, fwd ? a.p : 1 - a.p, mu) +
          (fwd ? h : hn);
      const size_t lr = (size_t)(fwd ? 3 : 1) * Vh, lc = (size_t)(fwd ? 1 : 3) * Vh;
      float4 *ls = slot + (12 + 9 * (k & 1)) * DS_NT;
#pragma unroll
      for (int q = 0; q < 12; ++q) cp_async16(slot + q * DS_NT, in + (size_t)q * S_);
#pragma unroll
      for (int q = 0; q < 9; ++q)
        cp_async16(ls + q * DS_NT, lk + (q / 3) * lr + (q % 3) * lc);
    };
    AccE2 s;
#pragma unroll
    for (int q = 0; q < 3; ++q) s.up[q] = s.dn[q] = cdd2{{0ull, 0ull}, {0ull, 0ull}};
    fetch(0);
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
      const int mu = k >> 1;
      const bool fwd = (k & 1) == 0;
      cp_async_wait();
      float4 p[12];
#pragma unroll
      for (int q = 0; q < 12; ++q) p[q] = slot[q * DS_NT];
      const float4 *ls = slot + (12 + 9 * (k & 1)) * DS_NT;
      hop_e2(
          p, [&] { if (k < 7) fetch(k + 1); },
          [&](int row, int q) { return ls[(3 * row + q) * DS_NT]; }, mu, fwd, fwd ? SF : -SF,
          mu == 0 && c[0] == (fwd ? a.g.L[0] - 1 : 0), false, s);
    }
    Cx<R> acc[12];
    unpack_e2(s, acc);
    const R cb = (R)(a.cb_rhs ? a.cb_rhs[r] : a.cb);
    if (a.x) {
      Cx<R> xv[12];
      SIO::load(a.x, S_, i, xv);
      const R ca = (R)a.ca;
#pragma unroll
      for (int k = 0; k < 12; ++k) {
        acc[k].re = fma(ca, xv[k].re, cb * acc[k].re);
        acc[k].im = fma(ca, xv[k].im, cb * acc[k].im);
      }
    } else {
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[k] = cb * acc[k];
    }
    SIO::store(a.out, S_, i, acc);
  }
}

}  // namespace

cudaError_t dslash_e2_smem() {
  const auto at = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const cudaError_t e = cudaFuncSetAttribute(k_dslash_e2<false>, at, E2_SMEM);
  return e != cudaSuccess ? e : cudaFuncSetAttribute(k_dslash_e2<true>, at, E2_SMEM);
}

void launch_dslash_e2(DslashArgs a, int dagger, cudaStream_t st) {
  const int nb = blocks_for((long long)a.g.Vh * a.n_rhs, DS_NT);
  if (a.rev) a.rev = nb;
  const auto kernel = dagger ? k_dslash_e2<true> : k_dslash_e2<false>;
  launch_pdl_smem(kernel, nb, DS_NT, E2_SMEM, st, a.pdl != 0, a);
}

}  // namespace hmc
