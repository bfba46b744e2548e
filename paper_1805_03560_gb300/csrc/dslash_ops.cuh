// Spin projection, link products and accumulation of one hop of the hopping
// matrix, shared by the hemi-Dslash kernels (the algebra is described in
// dslash.cu).
#pragma once
#include "hmc_internal.cuh"

namespace hmc {

// h = u - S B_mu d
template <int MU, int S, typename R>
__device__ __forceinline__ void project(const Cx<R> p[12], Cx<R> h[6]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Cx<R> u0 = p[a], u1 = p[3 + a], d0 = p[6 + a], d1 = p[9 + a];
    if (MU == 0) {
      h[a] = S > 0 ? u0 - d0 : u0 + d0;
      h[3 + a] = S > 0 ? u1 - d1 : u1 + d1;
    } else if (MU == 1) {
      h[a] = S > 0 ? u0 + ti(d1) : u0 - ti(d1);
      h[3 + a] = S > 0 ? u1 + ti(d0) : u1 - ti(d0);
    } else if (MU == 2) {
      h[a] = S > 0 ? u0 + d1 : u0 - d1;
      h[3 + a] = S > 0 ? u1 - d0 : u1 + d0;
    } else {
      h[a] = S > 0 ? u0 + ti(d0) : u0 - ti(d0);
      h[3 + a] = S > 0 ? u1 - ti(d1) : u1 + ti(d1);
    }
  }
}

// acc += (w, -S B_mu^dag w)
template <int MU, int S, typename R>
__device__ __forceinline__ void accumulate(Cx<R> acc[12], const Cx<R> w[6]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Cx<R> w0 = w[a], w1 = w[3 + a];
    acc[a] = acc[a] + w0;
    acc[3 + a] = acc[3 + a] + w1;
    if (MU == 0) {
      acc[6 + a] = S > 0 ? acc[6 + a] - w0 : acc[6 + a] + w0;
      acc[9 + a] = S > 0 ? acc[9 + a] - w1 : acc[9 + a] + w1;
    } else if (MU == 1) {
      acc[6 + a] = S > 0 ? acc[6 + a] - ti(w1) : acc[6 + a] + ti(w1);
      acc[9 + a] = S > 0 ? acc[9 + a] - ti(w0) : acc[9 + a] + ti(w0);
    } else if (MU == 2) {
      acc[6 + a] = S > 0 ? acc[6 + a] - w1 : acc[6 + a] + w1;
      acc[9 + a] = S > 0 ? acc[9 + a] + w0 : acc[9 + a] - w0;
    } else {
      acc[6 + a] = S > 0 ? acc[6 + a] - ti(w0) : acc[6 + a] + ti(w0);
      acc[9 + a] = S > 0 ? acc[9 + a] + ti(w1) : acc[9 + a] - ti(w1);
    }
  }
}

// w = U h (two colour vectors)
template <typename R>
__device__ __forceinline__ void mul_link(const Cx<R> u[9], const Cx<R> h[6], Cx<R> w[6]) {
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Cx<R> t = u[a * 3] * h[s * 3];
      t = fmac(t, u[a * 3 + 1], h[s * 3 + 1]);
      t = fmac(t, u[a * 3 + 2], h[s * 3 + 2]);
      w[s * 3 + a] = t;
    }
}

// w = U^dag h
template <typename R>
__device__ __forceinline__ void mul_link_dag(const Cx<R> u[9], const Cx<R> h[6], Cx<R> w[6]) {
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      Cx<R> t = cjmul(u[a], h[s * 3]);
      t = fmacj(t, u[3 + a], h[s * 3 + 1]);
      t = fmacj(t, u[6 + a], h[s * 3 + 2]);
      w[s * 3 + a] = t;
    }
}

// ---- runtime-direction forms ----------------------------------------------------
// One copy of the hop code serves all eight hops.  The fully unrolled stencil
// of the double-float kind is several times larger than the instruction
// cache (its warps stall waiting for instructions); this form keeps one
// projection, one link product of each kind and one accumulation in the
// loop body.  mu is warp-uniform, so the switches do not diverge.
// Same arithmetic as project / accumulate above, term for term.

template <typename R>
__device__ __forceinline__ Cx<R> sgn(int s, Cx<R> a) {
  return s > 0 ? a : -a;
}

// h = u - S B_mu d  with S = +-1 at run time
template <typename R>
__device__ __forceinline__ void project_rt(int mu, int S, const Cx<R> p[12], Cx<R> h[6]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const Cx<R> u0 = p[a], u1 = p[3 + a], d0 = p[6 + a], d1 = p[9 + a];
    Cx<R> t0, t1;
    int c0, c1;
    switch (mu) {
      case 0: t0 = d0; c0 = -S; t1 = d1; c1 = -S; break;
      case 1: t0 = ti(d1); c0 = S; t1 = ti(d0); c1 = S; break;
      case 2: t0 = d1; c0 = S; t1 = d0; c1 = -S; break;
      default: t0 = ti(d0); c0 = S; t1 = ti(d1); c1 = -S; break;
    }
    h[a] = u0 + sgn(c0, t0);
    h[3 + a] = u1 + sgn(c1, t1);
  }
}

// acc += (w, -S B_mu^dag w)
template <typename R>
__device__ __forceinline__ void accumulate_rt(int mu, int S, Cx<R> acc[12], const Cx<R> w[6]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const Cx<R> w0 = w[a], w1 = w[3 + a];
    acc[a] = acc[a] + w0;
    acc[3 + a] = acc[3 + a] + w1;
    Cx<R> l0, l1;
    int e0, e1;
    switch (mu) {
      case 0: l0 = w0; e0 = -S; l1 = w1; e1 = -S; break;
      case 1: l0 = ti(w1); e0 = -S; l1 = ti(w0); e1 = -S; break;
      case 2: l0 = w1; e0 = -S; l1 = w0; e1 = S; break;
      default: l0 = ti(w0); e0 = -S; l1 = ti(w1); e1 = S; break;
    }
    acc[6 + a] = acc[6 + a] + sgn(e0, l0);
    acc[9 + a] = acc[9 + a] + sgn(e1, l1);
  }
}

}  // namespace hmc
