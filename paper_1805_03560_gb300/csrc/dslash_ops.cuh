// Spin projection, link products and accumulation of one hop of the hopping
// matrix, shared by the hemi-Dslash kernels (the algebra is described in
// dslash.cu).
#pragma once
#include "df64x2.cuh"

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

// acc = (w, -S B_mu^dag w): accumulate onto zero
template <int MU, int S, typename R>
__device__ __forceinline__ void spread(Cx<R> acc[12], const Cx<R> w[6]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const Cx<R> w0 = w[a], w1 = w[3 + a];
    acc[a] = w0;
    acc[3 + a] = w1;
    if (MU == 0) {
      acc[6 + a] = S > 0 ? -w0 : w0;
      acc[9 + a] = S > 0 ? -w1 : w1;
    } else if (MU == 1) {
      acc[6 + a] = S > 0 ? -ti(w1) : ti(w1);
      acc[9 + a] = S > 0 ? -ti(w0) : ti(w0);
    } else if (MU == 2) {
      acc[6 + a] = S > 0 ? -w1 : w1;
      acc[9 + a] = S > 0 ? w0 : -w0;
    } else {
      acc[6 + a] = S > 0 ? -ti(w0) : ti(w0);
      acc[9 + a] = S > 0 ? ti(w1) : -ti(w1);
    }
  }
}

// project and accumulate of a direction known at run time (uniform over a warp)
template <int S, typename R>
__device__ __forceinline__ void project_mu(int mu, const Cx<R> p[12], Cx<R> h[6]) {
  switch (mu) {
    case 0: project<0, S>(p, h); break;
    case 1: project<1, S>(p, h); break;
    case 2: project<2, S>(p, h); break;
    default: project<3, S>(p, h); break;
  }
}
template <int S, typename R>
__device__ __forceinline__ void spread_mu(int mu, Cx<R> acc[12], const Cx<R> w[6]) {
  switch (mu) {
    case 0: spread<0, S>(acc, w); break;
    case 1: spread<1, S>(acc, w); break;
    case 2: spread<2, S>(acc, w); break;
    default: spread<3, S>(acc, w); break;
  }
}
template <int S, typename R>
__device__ __forceinline__ void accumulate_mu(int mu, Cx<R> acc[12], const Cx<R> w[6]) {
  switch (mu) {
    case 0: accumulate<0, S>(acc, w); break;
    case 1: accumulate<1, S>(acc, w); break;
    case 2: accumulate<2, S>(acc, w); break;
    default: accumulate<3, S>(acc, w); break;
  }
}

// ---- emulated FP64 with 18-real links, two spins at a time -------------------------
// One hop (direction mu, forwards or backwards, both uniform over a warp) of
// double-float fields: the two half-spinor components sit in the two lanes of
// the paired arithmetic (df64x2.cuh), a link element is duplicated into both
// lanes once for both.  U^dag is U with its indices exchanged by the loads and
// the imaginary parts negated, so one copy of the product serves both kinds
// of hop.  Same algebra as project / mul_link / accumulate.

// accumulated spinor: spins (0, 1) and (2, 3) of each colour
struct AccE2 {
  cdd2 up[3], dn[3];
};

template <int MU>
__device__ __forceinline__ void project_e2(const float4 p[12], f32x2 S, f32x2 sgn, cdd2 h[3]) {
  // S: all sign bits set for S = -1; sgn: the boundary sign's mask
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const float4 u0 = p[a], u1 = p[3 + a];
    const float4 d0 = MU == 1 || MU == 2 ? p[9 + a] : p[6 + a];
    const float4 d1 = MU == 1 || MU == 2 ? p[6 + a] : p[9 + a];
    const cdd2 u = {{pk2(u0.x, u1.x), pk2(u0.y, u1.y)}, {pk2(u0.z, u1.z), pk2(u0.w, u1.w)}};
    const cdd2 d = {{pk2(d0.x, d1.x), pk2(d0.y, d1.y)}, {pk2(d0.z, d1.z), pk2(d0.w, d1.w)}};
    // u + t with t = -S d (mu 0), S i d (1), (S, -S) d (2), (S, -S) i d (3)
    cdd2 t;
    if (MU == 0) t = {flip2(d.re, S ^ kNegBoth), flip2(d.im, S ^ kNegBoth)};
    if (MU == 1) t = {flip2(d.im, S ^ kNegBoth), flip2(d.re, S)};
    if (MU == 2) t = {flip2(d.re, S ^ kNeg1), flip2(d.im, S ^ kNeg1)};
    if (MU == 3) t = {flip2(d.im, S ^ kNeg0), flip2(d.re, S ^ kNeg1)};
    h[a] = {add(u.re, t.re), add(u.im, t.im)};
    if (MU == 0) h[a] = {flip2(h[a].re, sgn), flip2(h[a].im, sgn)};
  }
}

template <int MU>
__device__ __forceinline__ void accumulate_e2(AccE2 &acc, const cdd2 w[3], f32x2 S, bool first) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const cdd2 v = MU == 1 || MU == 2 ? cdd2{swap2(w[a].re), swap2(w[a].im)} : w[a];
    // -S v (mu 0), -S i v (1), (-S, S) v (2), (-S, S) i v (3)
    cdd2 t;
    if (MU == 0) t = {flip2(v.re, S ^ kNegBoth), flip2(v.im, S ^ kNegBoth)};
    if (MU == 1) t = {flip2(v.im, S), flip2(v.re, S ^ kNegBoth)};
    if (MU == 2) t = {flip2(v.re, S ^ kNeg0), flip2(v.im, S ^ kNeg0)};
    if (MU == 3) t = {flip2(v.im, S ^ kNeg1), flip2(v.re, S ^ kNeg0)};
    if (first) {
      acc.up[a] = w[a];
      acc.dn[a] = t;
    } else {
      acc.up[a] = {add(acc.up[a].re, w[a].re), add(acc.up[a].im, w[a].im)};
      acc.dn[a] = {add(acc.dn[a].re, t.re), add(acc.dn[a].im, t.im)};
    }
  }
}

// p: the neighbour's spinor, dead once projected() is called; link(r, k): the
// element U[r][k] of a forward hop's link, U[k][r] of a backward hop's; s: +1 or
// -1 (the sign of gamma_mu), wrap: boundary sign, first: acc is assigned
template <typename Done, typename Link>
__device__ __forceinline__ void hop_e2(const float4 p[12], Done projected, Link link, int mu,
                                       bool fwd, int s, bool wrap, bool first, AccE2 &acc) {
  const f32x2 S = s > 0 ? 0ull : kNegBoth, sgn = wrap ? kNegBoth : 0ull;
  cdd2 h[3];
  switch (mu) {
    case 0: project_e2<0>(p, S, sgn, h); break;
    case 1: project_e2<1>(p, S, sgn, h); break;
    case 2: project_e2<2>(p, S, sgn, h); break;
    default: project_e2<3>(p, S, sgn, h); break;
  }
  projected();
  cneg2 nh[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) nh[k] = negated(h[k]);
  const float si = fwd ? 1.f : -1.f;
  cdd2 w[3];
#pragma unroll
  for (int r = 0; r < 3; ++r)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float4 u = link(r, k);
      const float ih = si * u.z, il = si * u.w;
      const cdd2 ud = {{pk2(u.x, u.x), pk2(u.y, u.y)}, {pk2(ih, ih), pk2(il, il)}};
      w[r] = k == 0 ? cmul(ud, h[0], nh[0]) : cmac(w[r], ud, h[k], nh[k]);
    }
  switch (mu) {
    case 0: accumulate_e2<0>(acc, w, S, first); break;
    case 1: accumulate_e2<1>(acc, w, S, first); break;
    case 2: accumulate_e2<2>(acc, w, S, first); break;
    default: accumulate_e2<3>(acc, w, S, first); break;
  }
}

__device__ __forceinline__ void unpack_e2(const AccE2 &acc, Cx<df64> v[12]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    v[a] = {first(acc.up[a].re), first(acc.up[a].im)};
    v[3 + a] = {second(acc.up[a].re), second(acc.up[a].im)};
    v[6 + a] = {first(acc.dn[a].re), first(acc.dn[a].im)};
    v[9 + a] = {second(acc.dn[a].re), second(acc.dn[a].im)};
  }
}

}  // namespace hmc
