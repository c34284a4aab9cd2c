// dw_kernels.cuh -- the hopping-term stencil and the CG vector kernels.
//
// Hopping term (the sum in D = 1 - kappa*H):
//   (H psi)(x) = sum_mu [ (1 - gamma_mu) eta U_mu(x) psi(x+mu)
//                       + (1 + gamma_mu) eta U_mu(x-mu)^dag psi(x-mu) ]
// and for D^dag the two projectors swap.  Per output site and direction the
// kernel spin-projects the neighbour to a half spinor (2 spins x 3 colours),
// multiplies by the link or its adjoint, and reconstructs the lower two spins
// (the four stages of the paper's Fig. 1: load, linear combination, 3x3
// mat-vec, accumulate).  One thread per (output site, right-hand side) in k_hop
// (two in FP64-class storage, k_hop_rows; four on small lattices, k_hop_split);
// threads of a warp take consecutive even-odd site indices so every load is
// a coalesced 16-byte (or 8-byte) access.  The boundary sign eta (-1 on links
// crossing t = Lt-1 -> 0 when antiperiodic) is applied in the kernel, so
// links stay SU(3) and 12-real compression stays valid.
//
// Gamma basis (chiral): gamma_mu = [[0, B_mu], [B_mu^dag, 0]] with
// B_x = -i sigma_1, B_y = -i sigma_2, B_z = -i sigma_3, B_t = 1.  Then
//   (1 + s gamma_mu) psi = [ h ; s B^dag h ],  h = psi_up + s B psi_down.
#pragma once

#include <type_traits>

#include "dw_common.cuh"

namespace dw {

enum Coef { C_ONE = 0, C_MK, C_PK, C_MK2, C_PK2 };
// Stencil operator: the Wilson hopping term H, or the spin-diagonal covariant
// hopping term K = sum_mu [U_mu(x) delta_{x+mu} + U_mu(x-mu)^dag delta_{x-mu}]
// of the Laplacian 1 - kappa K (Hermitian: no dagger form).
enum Op { OP_WILSON = 0, OP_LAPLACE = 1 };
enum Gate { G_ACTIVE = 0, G_REL, G_ALL, G_XZERO, G_ZSRC };

template <int C>
__device__ __forceinline__ double coef_of(double kappa) {
  return C == C_ONE ? 1.0 : C == C_MK ? -kappa : C == C_PK ? kappa : C == C_MK2 ? -kappa * kappa : kappa * kappa;
}
// The coefficient in the arithmetic type R, from the system's pre-rounded
// kappa (FP32 and double-float) so that no thread converts from FP64.
template <int C, typename R>
__device__ __forceinline__ R coef(const SysDesc& S) {
  if constexpr (std::is_same<R, double>::value) {
    return coef_of<C>(S.kappa);
  } else if constexpr (std::is_same<R, float>::value) {
    return C == C_ONE ? 1.f : C == C_MK ? -S.kappa_f : C == C_PK ? S.kappa_f : C == C_MK2 ? -S.kappa2_f : S.kappa2_f;
  } else {
    const DF k = df_make(S.kappa_f, S.kappa_lo), k2 = df_make(S.kappa2_f, S.kappa2_lo);
    return C == C_ONE ? DF(1) : C == C_MK ? -k : C == C_PK ? k : C == C_MK2 ? -k2 : k2;
  }
}
// A CG scalar (alpha, beta) in the arithmetic type R: the finalizer's FP32
// rounding for FP32, the FP64 value split exactly for double-float.
template <typename R>
__device__ __forceinline__ R scalar_as(double v, float vf) {
  if constexpr (std::is_same<R, double>::value) return v;
  else if constexpr (std::is_same<R, float>::value) return vf;
  else return DF(v);
}

// G_ACTIVE is shut while the column's reliable update is due: what is left of an
// unrolled pass of the loop does nothing.
__device__ __forceinline__ int gate_of(int g, const RedArgs& ra, int col) {
  if (g == G_ALL) return 1;
  const ColState& C = ra.cols[col];
  if (g == G_XZERO) return C.xzero;
  if (g == G_ZSRC) return C.zsrc;
  if (g == G_REL) return C.do_rel;
  return C.active & (C.do_rel ^ 1);
}

// a + S*b,  S = +1 or -1 (compile time)
template <int S, typename R>
__device__ __forceinline__ Cx<R> pm(Cx<R> a, Cx<R> b) { return S > 0 ? a + b : a - b; }

// half spinor of (1 + S gamma_mu) psi
template <int MU, int S, typename R>
__device__ __forceinline__ void project(const Cx<R> (&p)[12], Cx<R> (&h)[6]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (MU == 0) {        // h0 = p0 - S i p3, h1 = p1 - S i p2
      h[c] = pm<-S>(p[c], mul_i(p[9 + c]));
      h[3 + c] = pm<-S>(p[3 + c], mul_i(p[6 + c]));
    } else if (MU == 1) { // h0 = p0 - S p3, h1 = p1 + S p2
      h[c] = pm<-S>(p[c], p[9 + c]);
      h[3 + c] = pm<S>(p[3 + c], p[6 + c]);
    } else if (MU == 2) { // h0 = p0 - S i p2, h1 = p1 + S i p3
      h[c] = pm<-S>(p[c], mul_i(p[6 + c]));
      h[3 + c] = pm<S>(p[3 + c], mul_i(p[9 + c]));
    } else {              // h0 = p0 + S p2, h1 = p1 + S p3
      h[c] = pm<S>(p[c], p[6 + c]);
      h[3 + c] = pm<S>(p[3 + c], p[9 + c]);
    }
  }
}

// acc += (1 + S gamma_mu) reconstructed from the multiplied half spinor g
template <int MU, int S, typename R>
__device__ __forceinline__ void accumulate(Cx<R> (&acc)[12], const Cx<R> (&g)[6]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    acc[c] = acc[c] + g[c];
    acc[3 + c] = acc[3 + c] + g[3 + c];
    if (MU == 0) {        // lower = S i (g1, g0)
      acc[6 + c] = pm<S>(acc[6 + c], mul_i(g[3 + c]));
      acc[9 + c] = pm<S>(acc[9 + c], mul_i(g[c]));
    } else if (MU == 1) { // lower = S (g1, -g0)
      acc[6 + c] = pm<S>(acc[6 + c], g[3 + c]);
      acc[9 + c] = pm<-S>(acc[9 + c], g[c]);
    } else if (MU == 2) { // lower = S i (g0, -g1)
      acc[6 + c] = pm<S>(acc[6 + c], mul_i(g[c]));
      acc[9 + c] = pm<-S>(acc[9 + c], mul_i(g[3 + c]));
    } else {              // lower = S (g0, g1)
      acc[6 + c] = pm<S>(acc[6 + c], g[c]);
      acc[9 + c] = pm<S>(acc[9 + c], g[3 + c]);
    }
  }
}

// acc + w * g  (w real), componentwise FMA
template <typename R>
__device__ __forceinline__ Cx<R> cfma(R w, Cx<R> g, Cx<R> acc) { return cx(fma(w, g.re, acc.re), fma(w, g.im, acc.im)); }

// acc += w (1 + S gamma_mu) reconstructed from g, w = dequantisation scale times
// the boundary sign (the 16-bit inputs are projected and multiplied unscaled)
template <int MU, int S, typename R>
__device__ __forceinline__ void accumulate_w(Cx<R> (&acc)[12], const Cx<R> (&g)[6], R w) {
  const R ws = S > 0 ? w : -w;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    acc[c] = cfma(w, g[c], acc[c]);
    acc[3 + c] = cfma(w, g[3 + c], acc[3 + c]);
    if (MU == 0) {        // lower = S i (g1, g0)
      acc[6 + c] = cfma(ws, mul_i(g[3 + c]), acc[6 + c]);
      acc[9 + c] = cfma(ws, mul_i(g[c]), acc[9 + c]);
    } else if (MU == 1) { // lower = S (g1, -g0)
      acc[6 + c] = cfma(ws, g[3 + c], acc[6 + c]);
      acc[9 + c] = cfma(-ws, g[c], acc[9 + c]);
    } else if (MU == 2) { // lower = S i (g0, -g1)
      acc[6 + c] = cfma(ws, mul_i(g[c]), acc[6 + c]);
      acc[9 + c] = cfma(-ws, mul_i(g[3 + c]), acc[9 + c]);
    } else {              // lower = S (g0, g1)
      acc[6 + c] = cfma(ws, g[c], acc[6 + c]);
      acc[9 + c] = cfma(ws, g[3 + c], acc[9 + c]);
    }
  }
}

// g = U h (ADJ = false) or U^dag h (ADJ = true), on both half-spinor spins
template <bool ADJ, typename R>
__device__ __forceinline__ void su3_mul(const Cx<R> (&u)[9], const Cx<R> (&h)[6], Cx<R> (&g)[6]) {
#pragma unroll
  for (int k = 0; k < 2; ++k)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      if (!ADJ) {
        Cx<R> t = cmul(u[a * 3 + 0], h[3 * k + 0]);
        t = cmadd(u[a * 3 + 1], h[3 * k + 1], t);
        g[3 * k + a] = cmadd(u[a * 3 + 2], h[3 * k + 2], t);
      } else {
        Cx<R> t = cjmul(u[0 * 3 + a], h[3 * k + 0]);
        t = cjmadd(u[1 * 3 + a], h[3 * k + 1], t);
        g[3 * k + a] = cjmadd(u[2 * 3 + a], h[3 * k + 2], t);
      }
    }
}

// 16-bit operand forms.  The projection runs on packed 16-bit lanes (one
// extra rounding to 16 bits per half-spinor component); the mat-vec takes the
// stored 16-bit link and half-spinor components directly into FP32-accumulating
// fused multiply-adds, so no component is converted to FP32 first.
template <int MU, int S, int P>
__device__ __forceinline__ void project_w(const uint32_t (&p)[12], uint32_t (&h)[6]) {
  using W = HW<P>;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (MU == 0) {        // h0 = p0 - S i p3, h1 = p1 - S i p2
      h[c] = W::template rot_add<-S>(p[c], p[9 + c]);
      h[3 + c] = W::template rot_add<-S>(p[3 + c], p[6 + c]);
    } else if (MU == 1) { // h0 = p0 - S p3, h1 = p1 + S p2
      h[c] = S > 0 ? W::sub(p[c], p[9 + c]) : W::add(p[c], p[9 + c]);
      h[3 + c] = S > 0 ? W::add(p[3 + c], p[6 + c]) : W::sub(p[3 + c], p[6 + c]);
    } else if (MU == 2) { // h0 = p0 - S i p2, h1 = p1 + S i p3
      h[c] = W::template rot_add<-S>(p[c], p[6 + c]);
      h[3 + c] = W::template rot_add<S>(p[3 + c], p[9 + c]);
    } else {              // h0 = p0 + S p2, h1 = p1 + S p3
      h[c] = S > 0 ? W::add(p[c], p[6 + c]) : W::sub(p[c], p[6 + c]);
      h[3 + c] = S > 0 ? W::add(p[3 + c], p[9 + c]) : W::sub(p[3 + c], p[9 + c]);
    }
  }
}

template <bool ADJ, int P>
__device__ __forceinline__ void su3_mul_w(const uint32_t (&u)[9], const uint32_t (&h)[6], Cx<float> (&g)[6]) {
  uint32_t hx[6];
#pragma unroll
  for (int k = 0; k < 6; ++k) hx[k] = h[k] ^ (ADJ ? kNegRe : kNegIm);
#pragma unroll
  for (int k = 0; k < 2; ++k)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float re = 0.f, im = 0.f;
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (ADJ) HW<P>::cmac_adj(re, im, u[b * 3 + a], h[3 * k + b], hx[3 * k + b]);
        else HW<P>::cmac(re, im, u[a * 3 + b], h[3 * k + b], hx[3 * k + b]);
      }
      g[3 * k + a] = cx(re, im);
    }
}

// Double-float version: each real output is one 6-term dot product.  The two
// spin rows of the half spinor are the two lanes of packed FP32x2 arithmetic,
// so each packed dot product yields one real output for both rows.
template <bool ADJ>
__device__ __forceinline__ void su3_mul(const Cx<DF> (&u)[9], const Cx<DF> (&h)[6], Cx<DF> (&g)[6]) {
  DF2 hr[3], hi[3], hrn[3], hin[3];  // rows k = 0, 1 in the lanes; n: negated
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    hr[b].hi = make_float2(h[b].re.hi, h[3 + b].re.hi);
    hr[b].lo = make_float2(h[b].re.lo, h[3 + b].re.lo);
    hi[b].hi = make_float2(h[b].im.hi, h[3 + b].im.hi);
    hi[b].lo = make_float2(h[b].im.lo, h[3 + b].im.lo);
    hrn[b].hi = make_float2(-hr[b].hi.x, -hr[b].hi.y);
    hrn[b].lo = make_float2(-hr[b].lo.x, -hr[b].lo.y);
    hin[b].hi = make_float2(-hi[b].hi.x, -hi[b].hi.y);
    hin[b].lo = make_float2(-hi[b].lo.x, -hi[b].lo.y);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    DF xr[6], xi[6];
    DF2 yr[6], yi[6];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const Cx<DF> m = ADJ ? u[b * 3 + a] : u[a * 3 + b];
      // re = m.re h.re -/+ m.im h.im ; im = m.re h.im +/- m.im h.re  (lower sign: adjoint)
      xr[2 * b] = m.re;
      yr[2 * b] = hr[b];
      xr[2 * b + 1] = m.im;
      yr[2 * b + 1] = ADJ ? hi[b] : hin[b];
      xi[2 * b] = m.re;
      yi[2 * b] = hi[b];
      xi[2 * b + 1] = m.im;
      yi[2 * b + 1] = ADJ ? hrn[b] : hr[b];
    }
    const DF2 re = df2_dot6(xr, yr), im = df2_dot6(xi, yi);
    g[a].re = df_make(re.hi.x, re.lo.x);
    g[a].im = df_make(im.hi.x, im.lo.x);
    g[3 + a].re = df_make(re.hi.y, re.lo.y);
    g[3 + a].im = df_make(im.hi.y, im.lo.y);
  }
}

// complex sums for the double-float path: lazy (no renormalisation)
__device__ __forceinline__ Cx<DF> cadd_lazy(Cx<DF> a, Cx<DF> b) { return cx(add_lazy(a.re, b.re), add_lazy(a.im, b.im)); }
// Site coordinates of even-odd index s on parity par.
struct Coord {
  int xh, x, y, z, t, row;  // row = s - xh (start of the x-row in eo indexing)
};

__device__ __forceinline__ Coord coord_of(const SysDesc& S, int s, int par) {
  Coord c;
  int q = fdiv(s, S.div_lxh);
  c.xh = s - q * S.lxh;
  c.row = s - c.xh;
  int q2 = fdiv(q, S.div_ly);
  c.y = q - q2 * S.ly;
  c.t = fdiv(q2, S.div_lz);
  c.z = q2 - c.t * S.lz;
  c.x = 2 * c.xh + ((c.y + c.z + c.t + par) & 1);
  return c;
}

// eo index of the neighbour one step in direction MU (DIR = +1/-1); *eta is
// the boundary sign of the link crossed.
template <int MU, int DIR>
__device__ __forceinline__ int neighbour(const SysDesc& S, const Coord& c, int s, float* eta) {
  *eta = 1.f;
  if (MU == 0) {
    const int lx = 2 * S.lxh;
    int xn = c.x + DIR;
    xn = xn == lx ? 0 : (xn < 0 ? lx - 1 : xn);
    return (xn >> 1) + c.row;
  } else if (MU == 1) {
    const int st = S.lxh;
    if (DIR > 0) return c.y == S.ly - 1 ? s - (S.ly - 1) * st : s + st;
    return c.y == 0 ? s + (S.ly - 1) * st : s - st;
  } else if (MU == 2) {
    const int st = S.lxh * S.ly;
    if (DIR > 0) return c.z == S.lz - 1 ? s - (S.lz - 1) * st : s + st;
    return c.z == 0 ? s + (S.lz - 1) * st : s - st;
  } else {
    const int st = S.lxh * S.ly * S.lz;
    if (DIR > 0) {
      if (c.t == S.lt - 1) {
        if (S.anti_t) *eta = -1.f;
        return s - (S.lt - 1) * st;
      }
      return s + st;
    }
    if (c.t == 0) {
      if (S.anti_t) *eta = -1.f;
      return s + (S.lt - 1) * st;
    }
    return s - st;
  }
}

__device__ __forceinline__ int neighbour_rt(const SysDesc& S, const Coord& c, int s, int mu, int dir, float* eta) {
  switch (mu) {
    case 0: return dir > 0 ? neighbour<0, +1>(S, c, s, eta) : neighbour<0, -1>(S, c, s, eta);
    case 1: return dir > 0 ? neighbour<1, +1>(S, c, s, eta) : neighbour<1, -1>(S, c, s, eta);
    case 2: return dir > 0 ? neighbour<2, +1>(S, c, s, eta) : neighbour<2, -1>(S, c, s, eta);
    default: return dir > 0 ? neighbour<3, +1>(S, c, s, eta) : neighbour<3, -1>(S, c, s, eta);
  }
}

__device__ __forceinline__ const char* slot_ptr(const SysDesc& S, int slot, int r, int par) {
  const Slot& f = S.f[slot];
  return f.p + r * f.rhs_stride + par * f.par_stride;
}
__device__ __forceinline__ char* slot_wptr(const SysDesc& S, int slot, int r, int par) {
  const Slot& f = S.f[slot];
  return f.p + r * f.rhs_stride + par * f.par_stride;
}

template <typename R, typename Q>
__device__ __forceinline__ void convert12(const Cx<Q> (&a)[12], Cx<R> (&b)[12]) {
#pragma unroll
  for (int k = 0; k < 12; ++k) b[k] = cx((R)a[k].re, (R)a[k].im);
}

// ------------------------------------------------------------------ input loaders
// Neighbour spinor from one field.
template <int SP>
struct InOne {
  int slot;
  static constexpr bool kScaled = Spin<SP>::kScaled;
  __host__ double io_bytes() const { return Spin<SP>::kBytes; }
  template <typename R>
  __device__ __forceinline__ void load(const SysDesc& S, int par, int r, int s, Cx<R> (&v)[12]) const {
    Cx<typename Spin<SP>::R> t[12];
    Spin<SP>::load(slot_ptr(S, slot, r, par), S.vh, s, t);
    convert12(t, v);
  }
  // 16-bit storage: stored words and the site scale
  __device__ __forceinline__ void load_words(const SysDesc& S, int par, int r, int s, uint32_t (&w)[12],
                                             float& sc) const {
    Spin<SP>::load_words(slot_ptr(S, slot, r, par), S.vh, s, w, sc);
  }
  // 16-bit storage: unscaled values and the site scale
  template <typename R>
  __device__ __forceinline__ void load_raw(const SysDesc& S, int par, int r, int s, Cx<R> (&v)[12], R& sc) const {
    if constexpr (Spin<SP>::kScaled) {
      Spin<SP>::load_raw(slot_ptr(S, slot, r, par), S.vh, s, v, sc);
    } else {
      load(S, par, r, s, v);
      sc = (R)1;
    }
  }
};

// ------------------------------------------------------------------ half sites
// Two threads per site (k_hop_rows): lanes j and j + 16 of a warp hold spins
// (0, 2) and (1, 3) of one site, a[c] = spin row, b[c] = spin 2 + row.
__device__ __forceinline__ uint32_t other_row(uint32_t w) { return __shfl_xor_sync(0xffffffffu, w, 16); }
__device__ __forceinline__ float other_row(float v) { return __shfl_xor_sync(0xffffffffu, v, 16); }
__device__ __forceinline__ double other_row(double v) { return __shfl_xor_sync(0xffffffffu, v, 16); }
__device__ __forceinline__ DF other_row(DF v) { return df_make(other_row(v.hi), other_row(v.lo)); }
template <typename R>
__device__ __forceinline__ Cx<R> other_row(Cx<R> v) { return cx(other_row(v.re), other_row(v.im)); }

// Store of one site in storage SP by its two threads (all lanes call it; lanes
// with ok = false take part in the exchanges only).  FP32 and 16-bit planes
// hold neighbouring complex numbers k = 3 spin + colour side by side, so the
// rows swap the ones that lie in the other's planes.
template <int SP, typename R>
__device__ __forceinline__ void store_rows(char* base, int vh, int s, int row, const Cx<R> (&a)[3],
                                           const Cx<R> (&b)[3], bool ok) {
  if constexpr (SP == P64 || SP == PDF) {
    using RS = typename Spin<SP>::R;
    Cx<RS> u[3], v[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      u[c] = cx((RS)a[c].re, (RS)a[c].im);
      v[c] = cx((RS)b[c].re, (RS)b[c].im);
    }
    if (ok) {
      Spin<SP>::store_spin(base, vh, s, row, u);
      Spin<SP>::store_spin(base, vh, s, 2 + row, v);
    }
  } else if constexpr (SP == P32) {
    Cx<float> u[3], v[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      u[c] = cx((float)a[c].re, (float)a[c].im);
      v[c] = cx((float)b[c].re, (float)b[c].im);
    }
    // row 0 holds k = 0 1 2 | 6 7 8 and stores planes 0 (0 1), 1 (2 3), 3 (6 7);
    // row 1 holds k = 3 4 5 | 9 10 11 and stores planes 2 (4 5), 4 (8 9), 5 (10 11)
    const Cx<float> got = other_row(row == 0 ? v[2] : u[0]);  // row 0: k = 3, row 1: k = 8
    float4* o = reinterpret_cast<float4*>(base) + s;
    if (ok) {
      if (row == 0) {
        o[0] = make_float4(u[0].re, u[0].im, u[1].re, u[1].im);
        o[(size_t)vh] = make_float4(u[2].re, u[2].im, got.re, got.im);
        o[(size_t)3 * vh] = make_float4(v[0].re, v[0].im, v[1].re, v[1].im);
      } else {
        o[(size_t)2 * vh] = make_float4(u[1].re, u[1].im, u[2].re, u[2].im);
        o[(size_t)4 * vh] = make_float4(got.re, got.im, v[0].re, v[0].im);
        o[(size_t)5 * vh] = make_float4(v[1].re, v[1].im, v[2].re, v[2].im);
      }
    }
  } else {
    Cx<float> u[3], v[3];
    float m = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      u[c] = cx((float)a[c].re, (float)a[c].im);
      v[c] = cx((float)b[c].re, (float)b[c].im);
      m = fmaxf(m, fmaxf(fmaxf(fabsf(u[c].re), fabsf(u[c].im)), fmaxf(fabsf(v[c].re), fabsf(v[c].im))));
    }
    m = fmaxf(m, other_row(m));
    m = m >= 1e-30f ? m : 0.f;  // as site_max
    const float inv = m > 0.f ? 1.0f / m : 0.f;
    uint32_t p[3], q[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      p[c] = H16<SP>::from2(u[c].re * inv, u[c].im * inv);
      q[c] = H16<SP>::from2(v[c].re * inv, v[c].im * inv);
    }
    // row 0 holds words 0 1 2 | 6 7 8 and stores plane 0 (0-3) and the scale;
    // row 1 holds words 3 4 5 | 9 10 11 and stores planes 1 (4-7) and 2 (8-11)
    const uint32_t x0 = other_row(row == 0 ? q[0] : p[0]);  // row 0: word 3, row 1: word 6
    const uint32_t x1 = other_row(q[1]), x2 = other_row(q[2]);
    uint4* o = reinterpret_cast<uint4*>(base) + s;
    if (ok) {
      if (row == 0) {
        o[0] = make_uint4(p[0], p[1], p[2], x0);
        reinterpret_cast<float*>(base + (size_t)48 * vh)[s] = m;
      } else {
        o[(size_t)vh] = make_uint4(p[1], p[2], x0, x1);
        o[(size_t)2 * vh] = make_uint4(x2, q[0], q[1], q[2]);
      }
    }
  }
}

// ------------------------------------------------------------------ epilogues
// write(): forms and stores the output of one site.  Reducing epilogues (kReduce)
// have prepare() (forms the stored words and the reduced value) and commit()
// (stores them) in its place, so that the kernel can publish its block's
// partial sum before the output stores.  write_rows() does both for a site
// held by two threads (k_hop_rows): a, b are the accumulated spins row and
// 2 + row; every lane calls it, lanes with ok = false store nothing.  The
// residuals, which are only taken in FP64-class arithmetic, have this form alone.
// out = coef * H in
template <int SPO, int COEF>
struct EpiOut {
  static constexpr bool kReduce = false;
  using Packed = int;
  int slot_out;
  int gate;
  __host__ double io_bytes() const { return Spin<SPO>::kBytes; }
  template <typename R, typename V>
  __device__ __forceinline__ void write(const SysDesc& S, int par, int r, int s, Cx<R> (&acc)[12], V&) const {
    using RO = typename Spin<SPO>::R;
    const R c = coef<COEF, R>(S);
    Cx<RO> o[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) o[k] = cx((RO)(c * acc[k].re), (RO)(c * acc[k].im));
    Spin<SPO>::store(slot_wptr(S, slot_out, r, par), S.vh, s, o);
  }
  template <typename R, typename V>
  __device__ __forceinline__ void write_rows(const SysDesc& S, int par, int r, int s, int row, Cx<R> (&a)[3],
                                             Cx<R> (&b)[3], V&, bool ok) const {
    if constexpr (COEF != C_ONE) {
      const R c = coef<COEF, R>(S);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        a[k] = cx(c * a[k].re, c * a[k].im);
        b[k] = cx(c * b[k].re, c * b[k].im);
      }
    }
    store_rows<SPO>(slot_wptr(S, slot_out, r, par), S.vh, s, row, a, b, ok);
  }
};

// out = X + coef * H in  (X on the output parity), optional |out|^2 reduction.
// slot_out < 0: nothing stored (norm only).
template <int SPO, int SPX, int COEF, bool RED>
struct EpiXpay {
  static constexpr bool kReduce = RED;
  using Packed = typename Spin<SPO>::Packed;
  int slot_out, slot_x;
  int gate;
  __host__ double io_bytes() const { return Spin<SPX>::kBytes + (slot_out >= 0 ? Spin<SPO>::kBytes : 0); }
  template <typename R>
  __device__ __forceinline__ Packed prepare(const SysDesc& S, int par, int r, int s, Cx<R> (&acc)[12],
                                            typename RedT<R>::type& nrm) const {
    Cx<typename Spin<SPX>::R> xv[12];
    Spin<SPX>::load(slot_ptr(S, slot_x, r, par), S.vh, s, xv);
    return form(S, acc, xv, nrm);
  }
  template <typename R>
  __device__ __forceinline__ Packed form(const SysDesc& S, Cx<R> (&acc)[12], const Cx<typename Spin<SPX>::R> (&xv)[12],
                                         typename RedT<R>::type& nrm) const {
    using RO = typename Spin<SPO>::R;
    const R c = coef<COEF, R>(S);
    Cx<RO> o[12];
    R n = (R)0;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      R re = fma(c, acc[k].re, (R)xv[k].re), im = fma(c, acc[k].im, (R)xv[k].im);
      o[k] = cx((RO)re, (RO)im);
      n = fma(re, re, fma(im, im, n));
    }
    nrm = to_red(n);
    return Spin<SPO>::pack(o);
  }
  __device__ __forceinline__ void commit(const SysDesc& S, int par, int r, int s, const Packed& o) const {
    if (slot_out >= 0) Spin<SPO>::store_packed(slot_wptr(S, slot_out, r, par), S.vh, s, o);
  }
  template <typename R>
  __device__ __forceinline__ void write(const SysDesc& S, int par, int r, int s, Cx<R> (&acc)[12],
                                        typename RedT<R>::type& nrm) const {
    const Packed o = prepare(S, par, r, s, acc, nrm);
    commit(S, par, r, s, o);
  }
  template <typename R>
  __device__ __forceinline__ void write_rows(const SysDesc& S, int par, int r, int s, int row, Cx<R> (&a)[3],
                                             Cx<R> (&b)[3], typename RedT<R>::type& nrm, bool ok) const {
    const char* xp = slot_ptr(S, slot_x, r, par);
    const R c = coef<COEF, R>(S);
    R n = (R)0;
    Cx<R> x[3];
    Spin<SPX>::load_spin(xp, S.vh, s, row, x);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a[k] = cx(fma(c, a[k].re, x[k].re), fma(c, a[k].im, x[k].im));
      if (RED) n = fma(a[k].re, a[k].re, fma(a[k].im, a[k].im, n));
    }
    Spin<SPX>::load_spin(xp, S.vh, s, 2 + row, x);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      b[k] = cx(fma(c, b[k].re, x[k].re), fma(c, b[k].im, x[k].im));
      if (RED) n = fma(b[k].re, b[k].re, fma(b[k].im, b[k].im, n));
    }
    if (RED) nrm = to_red(n);
    if (slot_out >= 0) store_rows<SPO>(slot_wptr(S, slot_out, r, par), S.vh, s, row, a, b, ok);
  }
};

// out = x + c*acc with the reduction Re <x, out> (the CG's p^dag A p for a
// Hermitian operator, x = p).
template <int SPO, int SPX, int COEF>
struct EpiXpayDot {
  static constexpr bool kReduce = true;
  using Packed = typename Spin<SPO>::Packed;
  int slot_out, slot_x;
  int gate;
  __host__ double io_bytes() const { return Spin<SPX>::kBytes + Spin<SPO>::kBytes; }
  __device__ __forceinline__ void commit(const SysDesc& S, int par, int r, int s, const Packed& o) const {
    Spin<SPO>::store_packed(slot_wptr(S, slot_out, r, par), S.vh, s, o);
  }
  template <typename R>
  __device__ __forceinline__ void write_rows(const SysDesc& S, int par, int r, int s, int row, Cx<R> (&a)[3],
                                             Cx<R> (&b)[3], typename RedT<R>::type& nrm, bool ok) const {
    const char* xp = slot_ptr(S, slot_x, r, par);
    const R c = coef<COEF, R>(S);
    R n = (R)0;
    Cx<R> x[3];
    Spin<SPX>::load_spin(xp, S.vh, s, row, x);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      a[k] = cx(fma(c, a[k].re, x[k].re), fma(c, a[k].im, x[k].im));
      n = fma(x[k].re, a[k].re, fma(x[k].im, a[k].im, n));
    }
    Spin<SPX>::load_spin(xp, S.vh, s, 2 + row, x);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      b[k] = cx(fma(c, b[k].re, x[k].re), fma(c, b[k].im, x[k].im));
      n = fma(x[k].re, b[k].re, fma(x[k].im, b[k].im, n));
    }
    nrm = to_red(n);
    store_rows<SPO>(slot_wptr(S, slot_out, r, par), S.vh, s, row, a, b, ok);
  }
  template <typename R>
  __device__ __forceinline__ Packed prepare(const SysDesc& S, int par, int r, int s, Cx<R> (&acc)[12],
                                            typename RedT<R>::type& nrm) const {
    Cx<typename Spin<SPX>::R> xv[12];
    Spin<SPX>::load(slot_ptr(S, slot_x, r, par), S.vh, s, xv);
    return form(S, acc, xv, nrm);
  }
  template <typename R>
  __device__ __forceinline__ Packed form(const SysDesc& S, Cx<R> (&acc)[12], const Cx<typename Spin<SPX>::R> (&xv)[12],
                                         typename RedT<R>::type& nrm) const {
    using RO = typename Spin<SPO>::R;
    const R c = coef<COEF, R>(S);
    Cx<RO> o[12];
    R n = (R)0;
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      const R xr = (R)xv[k].re, xi = (R)xv[k].im;
      const R re = fma(c, acc[k].re, xr), im = fma(c, acc[k].im, xi);
      o[k] = cx((RO)re, (RO)im);
      n = fma(xr, re, fma(xi, im, n));
    }
    nrm = to_red(n);
    return Spin<SPO>::pack(o);
  }
};

// One spin of a residual, v <- bh - x + c v, and its |.|^2 added to n.
template <int SPH, typename R>
__device__ __forceinline__ void resid_spin(const char* xp, const char* bp, int vh, int s, int spin, R c, Cx<R> (&v)[3],
                                           R& n) {
  Cx<R> x[3], b[3];
  Spin<SPH>::load_spin(xp, vh, s, spin, x);
  Spin<SPH>::load_spin(bp, vh, s, spin, b);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    v[k] = cx(fma(c, v[k].re, b[k].re - x[k].re), fma(c, v[k].im, b[k].im - x[k].im));
    n = fma(v[k].re, v[k].re, fma(v[k].im, v[k].im, n));
  }
}

// Residual of the even-odd system in the high precision SPH at even site s,
// once the accumulator x has absorbed the low-precision increment:
//   r_hi = bh - x + kappa^2 * acc  (acc = H_eo t, t = H_oe x);  r_low <- r_hi;
//   reduction |r_hi|^2.  r_hi itself is not stored: the iteration continues
//   from r_low, and the next correction recomputes r_hi.
template <int SPL, int SPH>
struct EpiResidEO {
  static constexpr bool kReduce = true;
  int gate;
  __host__ double io_bytes() const { return 2.0 * Spin<SPH>::kBytes + Spin<SPL>::kBytes; }
  template <typename RH>
  __device__ __forceinline__ void write_rows(const SysDesc& S, int par, int r, int s, int row, Cx<RH> (&a)[3],
                                             Cx<RH> (&b)[3], typename RedT<RH>::type& nrm, bool ok) const {
    const char *xp = slot_ptr(S, S_X, r, par), *bp = slot_ptr(S, S_BH, r, par);
    const RH k2 = coef<C_PK2, RH>(S);
    RH n = (RH)0;
    resid_spin<SPH>(xp, bp, S.vh, s, row, k2, a, n);
    resid_spin<SPH>(xp, bp, S.vh, s, 2 + row, k2, b, n);
    nrm = to_red(n);
    store_rows<SPL>(slot_wptr(S, S_R, r, par), S.vh, s, row, a, b, ok);
  }
};

// Full-lattice residual rt = b - (x - kappa*acc) on the output parity (with
// acc = H x this is b - D x; with acc = Hdag x it is b - D^dag x), in the
// precision SPH of x, b and rt, optionally also r_low <- rt.  Reduction |rt|^2.
template <int SPL, bool STORE_LOW, int SPH>
struct EpiResidFull {
  static constexpr bool kReduce = true;
  int gate;
  int slot_rt;  // < 0: norm only
  int slot_x;
  int slot_b;
  __host__ double io_bytes() const {
    return 2.0 * Spin<SPH>::kBytes + (slot_rt >= 0 ? Spin<SPH>::kBytes : 0) + (STORE_LOW ? Spin<SPL>::kBytes : 0);
  }
  template <typename RH>
  __device__ __forceinline__ void write_rows(const SysDesc& S, int par, int r, int s, int row, Cx<RH> (&a)[3],
                                             Cx<RH> (&b)[3], typename RedT<RH>::type& nrm, bool ok) const {
    const char *xp = slot_ptr(S, slot_x, r, par), *bp = slot_ptr(S, slot_b, r, par);
    const RH kap = coef<C_PK, RH>(S);
    RH n = (RH)0;
    resid_spin<SPH>(xp, bp, S.vh, s, row, kap, a, n);
    resid_spin<SPH>(xp, bp, S.vh, s, 2 + row, kap, b, n);
    nrm = to_red(n);
    if (slot_rt >= 0) store_rows<SPH>(slot_wptr(S, slot_rt, r, par), S.vh, s, row, a, b, ok);
    if (STORE_LOW) store_rows<SPL>(slot_wptr(S, S_R, r, par), S.vh, s, row, a, b, ok);
  }
};

// ------------------------------------------------------------------ block prologue
// This block's system descriptor S, this thread's site s on output parity par,
// its right-hand side r, and whether it has work (valid): in range and its
// column's gate open.  The descriptor is read where it is used, from the
// kernel parameter in the constant bank, and every thread tests its own gate:
// no copy, no barrier and one global load ahead of a thread's first operand
// load.  (A copy of the descriptor in shared memory, a barrier, the gates of
// all columns and a second barrier held every block's SM slot for about 1 us
// before its first load.)  The reduction needs no agreement between blocks on
// a gate: a closed column's partials are ignored by its finalizer.
#define DW_BLOCK_PROLOGUE(GATE)                                            \
  const int T = B.T, RB = B.RB;                                            \
  /* the right-hand-side block varies fastest: the blocks of one tile run  \
     together and share its links and neighbours in L2 */                  \
  const unsigned bx_ = B.rev ? gridDim.x - 1u - blockIdx.x : blockIdx.x;   \
  int by = 0, b = (int)bx_, par, rl = 0;                                   \
  if (B.ny > 1) {                                                          \
    b = (int)(bx_ / (unsigned)B.ny);                                       \
    by = (int)bx_ - b * B.ny;                                              \
  }                                                                        \
  if (par_mode == 2) {                                                     \
    par = b >= B.ntot ? 1 : 0;                                             \
    b -= par * B.ntot;                                                     \
  } else {                                                                 \
    par = par_mode;                                                        \
  }                                                                        \
  const SysDesc& S = B.sd[block_system(B, b)];                             \
  if (RB > 1) rl = (int)threadIdx.x / T;                                   \
  const int r = by * RB + rl;                                              \
  const int tile = b - S.tile0;                                            \
  const int s = tile * T + ((int)threadIdx.x - rl * T);                    \
  const bool valid = s < S.vh && r < S.nrhs && gate_of(GATE, ra, S.col0 + r);

#define DW_BLOCK_REDUCE(val)                                               \
  {                                                                        \
    const int ntiles = par_mode == 2 ? 2 * S.tpp : S.tpp;                  \
    const int tt = par_mode == 2 ? par * S.tpp + tile : tile;              \
    reduce_block(S, T, RB, tt, ntiles, val, ra, by);               \
  }
// As DW_BLOCK_REDUCE, with the output stores STORE (a lambda) run after the
// block's partial sums are written.
#define DW_BLOCK_REDUCE_STORE(val, STORE)                                  \
  {                                                                        \
    const int ntiles = par_mode == 2 ? 2 * S.tpp : S.tpp;                  \
    const int tt = par_mode == 2 ? par * S.tpp + tile : tile;              \
    reduce_block(S, T, RB, tt, ntiles, val, ra, by, STORE);        \
  }

// ------------------------------------------------------------------ the Laplacian's directions
// acc = K psi at output site s: the neighbour's whole spinor (no projection)
// times U_mu(x) or U_mu(x-mu)^dag, spin by spin, with the boundary sign.
template <int SPA, int LP, bool C12, class In, typename R>
__device__ __forceinline__ void laplace_dirs(const SysDesc& S, const In& in, const Coord& c, int s, int r, int pin,
                                             const char* ulink_own, const char* ulink_nb, long long mu_stride,
                                             Cx<R> (&acc)[12]) {
  // all eight directions unrolled (compile-time neighbour arithmetic)
#pragma unroll
  for (int d = 0; d < 8; ++d) {
    const int mu = d >> 1;
    const bool fwd = (d & 1) == 0;
    float eta;
    const int n = neighbour_rt(S, c, s, mu, fwd ? +1 : -1, &eta);
    const char* lb = (fwd ? ulink_own : ulink_nb) + mu * mu_stride;
    const int li = fwd ? s : n;
    if constexpr (SPA == P16 || SPA == PB16) {
      uint32_t pw[12], h0[6], h1[6], u[9];
      float sc;
      Cx<float> g0[6], g1[6];
      in.load_words(S, pin, r, n, pw, sc);
      Link<LP, C12>::load_words(lb, S.vh, li, u);
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        h0[k] = pw[k];
        h1[k] = pw[6 + k];
      }
      if (fwd) {
        su3_mul_w<false, SPA>(u, h0, g0);
        su3_mul_w<false, SPA>(u, h1, g1);
      } else {
        su3_mul_w<true, SPA>(u, h0, g0);
        su3_mul_w<true, SPA>(u, h1, g1);
      }
      const float w = eta < 0.f ? -sc : sc;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        acc[k] = cfma(w, g0[k], acc[k]);
        acc[6 + k] = cfma(w, g1[k], acc[6 + k]);
      }
    } else {
      Cx<R> p[12], h0[6], h1[6], g0[6], g1[6], u[9];
      in.load(S, pin, r, n, p);
      Link<LP, C12>::load(lb, S.vh, li, u);
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        h0[k] = p[k];
        h1[k] = p[6 + k];
      }
      if (eta < 0.f) {  // boundary sign: taken only on the t-boundary slice
#pragma unroll
        for (int k = 0; k < 6; ++k) {
          h0[k] = cx(-h0[k].re, -h0[k].im);
          h1[k] = cx(-h1[k].re, -h1[k].im);
        }
      }
      if (fwd) {
        su3_mul<false>(u, h0, g0);
        su3_mul<false>(u, h1, g1);
      } else {
        su3_mul<true>(u, h0, g0);
        su3_mul<true>(u, h1, g1);
      }
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        acc[k] = acc[k] + g0[k];
        acc[6 + k] = acc[6 + k] + g1[k];
      }
    }
  }
}

// ------------------------------------------------------------------ one direction pair
// acc += the forward and backward hop along MU at output site s (forward
// projector sign SF, backward -SF).
template <int MU, int SPA, int LP, bool C12, int SF, class In, typename R>
__device__ __forceinline__ void hop_mu(const SysDesc& S, const In& in, const Coord& c, int s, int r, int pin,
                                       const char* own, const char* nbr, long long mu_stride, Cx<R> (&acc)[12]) {
  float eta;
  const int nf = neighbour<MU, +1>(S, c, s, &eta);
  if constexpr (SPA == P16 || SPA == PB16) {
    float sc;
    uint32_t p[12], h[6], u[9];
    Cx<float> g[6];
    in.load_words(S, pin, r, nf, p, sc);
    project_w<MU, SF, SPA>(p, h);
    Link<LP, C12>::load_words(own + MU * mu_stride, S.vh, s, u);
    su3_mul_w<false, SPA>(u, h, g);
    accumulate_w<MU, SF>(acc, g, eta < 0.f ? -sc : sc);
    const int nb = neighbour<MU, -1>(S, c, s, &eta);
    in.load_words(S, pin, r, nb, p, sc);
    project_w<MU, -SF, SPA>(p, h);
    Link<LP, C12>::load_words(nbr + MU * mu_stride, S.vh, nb, u);
    su3_mul_w<true, SPA>(u, h, g);
    accumulate_w<MU, -SF>(acc, g, eta < 0.f ? -sc : sc);
  } else {
    Cx<R> p[12], h[6], g[6], u[9];
    R sc;
    in.load_raw(S, pin, r, nf, p, sc);
    project<MU, SF>(p, h);
    Link<LP, C12>::load(own + MU * mu_stride, S.vh, s, u);
    su3_mul<false>(u, h, g);
    accumulate_w<MU, SF>(acc, g, eta < 0.f ? -sc : sc);
    const int nb = neighbour<MU, -1>(S, c, s, &eta);
    in.load_raw(S, pin, r, nb, p, sc);
    project<MU, -SF>(p, h);
    Link<LP, C12>::load(nbr + MU * mu_stride, S.vh, nb, u);
    su3_mul<true>(u, h, g);
    accumulate_w<MU, -SF>(acc, g, eta < 0.f ? -sc : sc);
  }
}

// ------------------------------------------------------------------ the stencil kernel
// par_mode 0/1: output parity fixed, grid = ntot blocks.  par_mode 2: both
// parities, grid = 2*ntot (block b >= ntot works on odd output sites).
// Input is read on the opposite parity.  SPA: arithmetic-precision tag.
// Minimum resident blocks (of 256 threads) per SM requested from the compiler,
// that is a register cap (256 threads x n blocks share 65536 registers).  The
// kernels are bound by load latency at the occupancy that this leaves.
// Measured on GB300, microseconds per even-site application at 32^3x64:
//   FP16, 12 reals   2: 145.6   3: 142.5   4: 138.0 (with |out|^2 193 -> 184)
//   FP32, 18 reals   1: 284.5   2: 252.9   3: 306 (spills)
//   FP32, 12 reals   1: 224.0   2: 211.2   3: 224
//   I16, 12 reals    1: 181.8   2: 182.0   3: 179.4
// (FP64-class storage has its own kernel, k_hop_rows.)
#ifndef DW_HOP16_MINB
#define DW_HOP16_MINB 4
#endif
#ifndef DW_HOP32_MINB
#define DW_HOP32_MINB 2
#endif
#ifndef DW_HOPI16_MINB
#define DW_HOPI16_MINB 3
#endif
template <int SPA>
struct HopOccupancy {
  static constexpr int kMinBlocks = (SPA == P16 || SPA == PB16) ? DW_HOP16_MINB
                                    : SPA == P32                ? DW_HOP32_MINB
                                    : SPA == PI16               ? DW_HOPI16_MINB
                                                                : 1;
};

template <int SPA, int LP, bool C12, bool DAG, class In, class Epi, int OP = OP_WILSON>
__global__ void __launch_bounds__(256, HopOccupancy<SPA>::kMinBlocks)
    k_hop(const __grid_constant__ Batch B, int par_mode, int link_slot, In in, Epi epi, RedArgs ra) {
  using R = typename Spin<SPA>::R;
  DW_BLOCK_PROLOGUE(epi.gate)
  {
    typename RedT<R>::type nrm = red_zero(typename RedT<R>::type());
    typename Epi::Packed po;
    if (valid) {
      const Coord c = coord_of(S, s, par);
      const int pin = par ^ 1;
      const char* ulink_own = slot_ptr(S, link_slot, 0, par);  // links based at this site
      const char* ulink_nb = slot_ptr(S, link_slot, 0, pin);   // links based at the neighbour
      const long long mu_stride = (long long)Link<LP, C12>::kBytes * S.vh;
      constexpr int SF = DAG ? +1 : -1;  // forward projector sign
      Cx<R> acc[12];
#pragma unroll
      for (int k = 0; k < 12; ++k) acc[k] = cx((R)0, (R)0);

      if constexpr (OP == OP_LAPLACE) {
        laplace_dirs<SPA, LP, C12>(S, in, c, s, r, pin, ulink_own, ulink_nb, mu_stride, acc);
      } else {
        hop_mu<0, SPA, LP, C12, SF>(S, in, c, s, r, pin, ulink_own, ulink_nb, mu_stride, acc);
        hop_mu<1, SPA, LP, C12, SF>(S, in, c, s, r, pin, ulink_own, ulink_nb, mu_stride, acc);
        hop_mu<2, SPA, LP, C12, SF>(S, in, c, s, r, pin, ulink_own, ulink_nb, mu_stride, acc);
        hop_mu<3, SPA, LP, C12, SF>(S, in, c, s, r, pin, ulink_own, ulink_nb, mu_stride, acc);
      }
      if constexpr (Epi::kReduce) po = epi.prepare(S, par, r, s, acc, nrm);
      else epi.write(S, par, r, s, acc, nrm);
    }
    if constexpr (Epi::kReduce) {
      DW_BLOCK_REDUCE_STORE(nrm, [&] {
        if (valid) epi.commit(S, par, r, s, po);
      })
    }
  }
}

// ------------------------------------------------------------------ four threads per site
// The FP32 and 16-bit Wilson stencils on lattices too small to fill the GPU:
// one warp per mu for 32 consecutive sites, the four partial sums added in
// shared memory (mu = 0 1 2 3, in that order) by the warp of mu = 0, which
// runs the epilogue.  With one thread per site a 16^3x32 launch has 13 warps
// per SM, each a serial chain of eight load latencies; four times the warps
// with a quarter of the chain hide it.  On large lattices the extra pass
// through shared memory costs more than it gives (the solver's kSplitSites
// says where the line lies).
// Blocks: T sites x RB right-hand sides (T RB <= 128), 4 T RB threads, warps
// (right-hand side, site group, mu).
template <int SPA, int LP, bool C12, bool DAG, class In, class Epi>
__global__ void __launch_bounds__(512, 2)
    k_hop_split(const __grid_constant__ Batch B, int par_mode, int link_slot, In in, Epi epi, RedArgs ra) {
  using R = typename Spin<SPA>::R;
  extern __shared__ float parts[];  // [site group][3][24][32]
  const int T = B.T, RB = B.RB;
  const unsigned bx = B.rev ? gridDim.x - 1u - blockIdx.x : blockIdx.x;
  int by = 0, b = (int)bx, par, rl = 0;
  if (B.ny > 1) {
    b = (int)(bx / (unsigned)B.ny);
    by = (int)bx - b * B.ny;
  }
  if (par_mode == 2) {
    par = b >= B.ntot ? 1 : 0;
    b -= par * B.ntot;
  } else {
    par = par_mode;
  }
  const SysDesc& S = B.sd[block_system(B, b)];
  const int lane = threadIdx.x & 31, mu = (threadIdx.x >> 5) & 3, group = threadIdx.x >> 7;
  if (RB > 1) rl = group / (T >> 5);
  const int r = by * RB + rl;
  const int tile = b - S.tile0;
  const int s = tile * T + ((group - rl * (T >> 5)) << 5) + lane;
  const bool valid = s < S.vh && r < S.nrhs && gate_of(epi.gate, ra, S.col0 + r);
  Cx<R> acc[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) acc[k] = cx((R)0, (R)0);
  if (valid) {
    const Coord c = coord_of(S, s, par);
    const int pin = par ^ 1;
    const char* own = slot_ptr(S, link_slot, 0, par);
    const char* nbr = slot_ptr(S, link_slot, 0, pin);
    const long long mu_stride = (long long)Link<LP, C12>::kBytes * S.vh;
    constexpr int SF = DAG ? +1 : -1;
    if (mu == 0) hop_mu<0, SPA, LP, C12, SF>(S, in, c, s, r, pin, own, nbr, mu_stride, acc);
    else if (mu == 1) hop_mu<1, SPA, LP, C12, SF>(S, in, c, s, r, pin, own, nbr, mu_stride, acc);
    else if (mu == 2) hop_mu<2, SPA, LP, C12, SF>(S, in, c, s, r, pin, own, nbr, mu_stride, acc);
    else hop_mu<3, SPA, LP, C12, SF>(S, in, c, s, r, pin, own, nbr, mu_stride, acc);
  }
  float* mine = parts + (size_t)group * (3 * 24 * 32) + lane;
  if (mu != 0) {
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      mine[((mu - 1) * 24 + 2 * k) * 32] = acc[k].re;
      mine[((mu - 1) * 24 + 2 * k + 1) * 32] = acc[k].im;
    }
  }
  __syncthreads();
  typename RedT<R>::type nrm = red_zero(typename RedT<R>::type());
  typename Epi::Packed po;
  const bool out = valid && mu == 0;
  if (out) {
#pragma unroll
    for (int m = 0; m < 3; ++m)
#pragma unroll
      for (int k = 0; k < 12; ++k)
        acc[k] = acc[k] + cx(mine[(m * 24 + 2 * k) * 32], mine[(m * 24 + 2 * k + 1) * 32]);
    if constexpr (Epi::kReduce) po = epi.prepare(S, par, r, s, acc, nrm);
    else epi.write(S, par, r, s, acc, nrm);
  }
  if constexpr (Epi::kReduce) {
    const int ntiles = par_mode == 2 ? 2 * S.tpp : S.tpp;
    reduce_block(S, 4 * T, RB, par_mode == 2 ? par * S.tpp + tile : tile, ntiles, nrm, ra, by, [&] {
      if (out) epi.commit(S, par, r, s, po);
    });
  }
}

// ------------------------------------------------------------------ two threads per site
// g = one row of the half spinor times U (or U^dag).
template <bool ADJ>
__device__ __forceinline__ void su3_mul_row(const Cx<double> (&u)[9], const Cx<double> (&h)[3], Cx<double> (&g)[3]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    if (!ADJ) {
      Cx<double> t = cmul(u[a * 3 + 0], h[0]);
      t = cmadd(u[a * 3 + 1], h[1], t);
      g[a] = cmadd(u[a * 3 + 2], h[2], t);
    } else {
      Cx<double> t = cjmul(u[0 * 3 + a], h[0]);
      t = cjmadd(u[1 * 3 + a], h[1], t);
      g[a] = cjmadd(u[2 * 3 + a], h[2], t);
    }
  }
}
// Double-float: the real and imaginary part of an output are the two lanes of
// packed FP32x2 arithmetic.
template <bool ADJ>
__device__ __forceinline__ void su3_mul_row(const Cx<DF> (&u)[9], const Cx<DF> (&h)[3], Cx<DF> (&g)[3]) {
  DF2 yr[3], yi[3];  // what the link's real and imaginary part multiply
#pragma unroll
  for (int b = 0; b < 3; ++b) {
    yr[b].hi = make_float2(h[b].re.hi, h[b].im.hi);
    yr[b].lo = make_float2(h[b].re.lo, h[b].im.lo);
    yi[b].hi = ADJ ? make_float2(h[b].im.hi, -h[b].re.hi) : make_float2(-h[b].im.hi, h[b].re.hi);
    yi[b].lo = ADJ ? make_float2(h[b].im.lo, -h[b].re.lo) : make_float2(-h[b].im.lo, h[b].re.lo);
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    DF x[6];
    DF2 y[6];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const Cx<DF> m = ADJ ? u[b * 3 + a] : u[a * 3 + b];
      x[2 * b] = m.re;
      y[2 * b] = yr[b];
      x[2 * b + 1] = m.im;
      y[2 * b + 1] = yi[b];
    }
    const DF2 t = df2_dot6(x, y);
    g[a] = cx(df_make(t.hi.x, t.lo.x), df_make(t.hi.y, t.lo.y));
  }
}
// sign flips by mask (0 or the sign bit): bit operations, so that IEEE FP64
// negations stay off the FP64 pipe
__device__ __forceinline__ double flip(double v, uint32_t m) {
  return __hiloint2double(__double2hiint(v) ^ (int)m, __double2loint(v));
}
__device__ __forceinline__ float flip(float v, uint32_t m) { return __uint_as_float(__float_as_uint(v) ^ m); }
__device__ __forceinline__ DF flip(DF v, uint32_t m) { return df_make(flip(v.hi, m), flip(v.lo, m)); }
// +-1 (or +-i) times q, the sign by mask
template <bool IMAG, typename R>
__device__ __forceinline__ Cx<R> times_unit(Cx<R> q, uint32_t m) {
  return IMAG ? cx(flip(q.im, m ^ 0x80000000u), flip(q.re, m)) : cx(flip(q.re, m), flip(q.im, m));
}
__device__ __forceinline__ Cx<double> row_add(Cx<double> a, Cx<double> b) { return a + b; }
__device__ __forceinline__ Cx<DF> row_add(Cx<DF> a, Cx<DF> b) { return cadd_lazy(a, b); }

// One row of the half spinor projected from neighbour n: h = p_row + c p_q,
// c = +-1 or +-i with the sign by mask cm; bm flips h on the t-boundary slice.
template <int SPA, bool IMAG, typename R>
__device__ __forceinline__ void row_project(const char* in, int vh, int n, int row, int partner, uint32_t cm,
                                            uint32_t bm, Cx<R> (&h)[3]) {
  Cx<R> q[3];
  Spin<SPA>::load_spin(in, vh, n, row, h);
  Spin<SPA>::load_spin(in, vh, n, partner, q);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    h[c] = row_add(h[c], times_unit<IMAG>(q[c], cm));
    h[c] = cx(flip(h[c].re, bm), flip(h[c].im, bm));
  }
}

// IEEE FP64: both directions of one mu for one row.  With g_f = U h_f and
// g_b = U^dag h_b the upper spin takes g_f + g_b and the lower spin d (g_f - g_b),
// d the unit factor of the forward projector (the backward one is its negative).
// The FP64 pipe (64 cycles per warp instruction) is the bound, so additions are
// saved: the backward product's chain starts from g_f and yields A = g_f + g_b
// at no extra cost, and g_f - g_b = 2 g_f - A is one FMA: 18 instead of 24
// operations per mu and row, none onto empty sums.  (Where g_f + g_b is not finite,
// in the upper spin, g_f - g_b in the lower one is not either.)
template <bool C12, bool IMAG>
__device__ __forceinline__ void row_mu(const SysDesc& S, const char* in, const char* own, const char* nbr, int s, int nf,
                                       int nb, int row, int partner, uint32_t cm, uint32_t dm, uint32_t bf, uint32_t bb,
                                       Cx<double> (&up)[3], Cx<double> (&low)[3], bool first) {
  Cx<double> h[3], g[3], u[9];
  row_project<P64, IMAG>(in, S.vh, nf, row, partner, cm, bf, h);
  Link<P64, C12>::load(own, S.vh, s, u);
  su3_mul_row<false>(u, h, g);
  row_project<P64, IMAG>(in, S.vh, nb, row, partner, cm ^ 0x80000000u, bb, h);
  Link<P64, C12>::load(nbr, S.vh, nb, u);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    Cx<double> t = cjmadd(u[0 * 3 + a], h[0], g[a]);
    t = cjmadd(u[1 * 3 + a], h[1], t);
    t = cjmadd(u[2 * 3 + a], h[2], t);
    const Cx<double> d = times_unit<IMAG>(cx(fma(2.0, g[a].re, -t.re), fma(2.0, g[a].im, -t.im)), dm);
    up[a] = first ? t : up[a] + t;
    low[a] = first ? d : low[a] + d;
  }
}

// Double-float: the operands of one direction for a warp's 16 sites go through
// shared memory, copied asynchronously while the direction before is computed
// (two stages, private to the warp).  A direction is about 480 instructions per
// thread and its loads about 1 us away; in registers there is no room to hold
// the next direction's 15 words of 16 bytes at 128 registers per thread.
// Stage: 12 spinor planes, then the link's planes, 16 sites x 16 bytes each.
template <bool C12>
struct RowRing {
  static constexpr int kChunks = 12 + (C12 ? 6 : 9);
  static constexpr int kStage = kChunks * 256;  // bytes
  static constexpr int kBytes = 2 * kStage;     // per warp
  // lanes j and j + 16 copy the even and the odd planes of site j
  __device__ static __forceinline__ void issue(char* stage, const char* in, const char* lb, int vh, int n, int li) {
    const int lane = threadIdx.x & 31, half = lane >> 4;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(stage) + half * 256 + (lane & 15) * 16;
    const char* p = in + ((size_t)half * vh + n) * 16;
    const char* q = lb + ((size_t)half * vh + li) * 16;
#pragma unroll
    for (int i = 0; i < 6; ++i)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i * 512), "l"(p + (size_t)(2 * i) * vh * 16)
                   : "memory");
#pragma unroll
    for (int i = 0; i < (kChunks - 12 + 1) / 2; ++i)
      if (2 * i + half < kChunks - 12)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + (6 + i) * 512),
                     "l"(q + (size_t)(2 * i) * vh * 16)
                     : "memory");
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  __device__ static __forceinline__ Cx<DF> word(const char* stage, int chunk) {
    const float4 t = *reinterpret_cast<const float4*>(stage + chunk * 256 + (threadIdx.x & 15) * 16);
    return cx(df_make(t.x, t.y), df_make(t.z, t.w));
  }
  // one direction for one row: h projected, g = U h (or U^dag h), added up
  template <bool IMAG, bool ADJ>
  __device__ static __forceinline__ void direction(const char* stage, int row, int partner, uint32_t cm, uint32_t dm,
                                                   uint32_t bm, Cx<DF> (&up)[3], Cx<DF> (&low)[3]) {
    Cx<DF> h[3], g[3], u[9];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      h[c] = row_add(word(stage, 3 * row + c), times_unit<IMAG>(word(stage, 3 * partner + c), cm));
      h[c] = cx(flip(h[c].re, bm), flip(h[c].im, bm));
    }
#pragma unroll
    for (int k = 0; k < kChunks - 12; ++k) u[k] = word(stage, 12 + k);
    if (C12) rebuild_row2(u);
    su3_mul_row<ADJ>(u, h, g);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      up[a] = row_add(up[a], g[a]);
      low[a] = row_add(low[a], times_unit<IMAG>(g[a], dm));
    }
  }
};
// The Laplacian's directions: both spins of the thread times U (or U^dag).
template <bool C12, bool ADJ>
__device__ __forceinline__ void lap_direction(const char* stage, int row, uint32_t bm, Cx<DF> (&up)[3], Cx<DF> (&low)[3]) {
  using Ring = RowRing<C12>;
  Cx<DF> h[6], g[6], u[9];
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    const Cx<DF> w = Ring::word(stage, k < 3 ? 3 * row + k : 3 * (2 + row) + k - 3);
    h[k] = cx(flip(w.re, bm), flip(w.im, bm));
  }
#pragma unroll
  for (int k = 0; k < Ring::kChunks - 12; ++k) u[k] = Ring::word(stage, 12 + k);
  if (C12) rebuild_row2(u);
  su3_mul<ADJ>(u, h, g);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    up[a] = row_add(up[a], g[a]);
    low[a] = row_add(low[a], g[3 + a]);
  }
}
// IEEE FP64: the products chained onto the sums, no additions of their own (1152
// instead of 1344 FP64 operations per site).
template <bool C12, bool ADJ>
__device__ __forceinline__ void lap_direction(const SysDesc& S, const char* in, const char* lb, int n, int li, int row,
                                              uint32_t bm, Cx<double> (&up)[3], Cx<double> (&low)[3]) {
  Cx<double> a[3], b[3], u[9];
  Spin<P64>::load_spin(in, S.vh, n, row, a);
  Spin<P64>::load_spin(in, S.vh, n, 2 + row, b);
  Link<P64, C12>::load(lb, S.vh, li, u);
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    a[k] = cx(flip(a[k].re, bm), flip(a[k].im, bm));
    b[k] = cx(flip(b[k].re, bm), flip(b[k].im, bm));
  }
#pragma unroll
  for (int i = 0; i < 3; ++i)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      up[i] = ADJ ? cjmadd(u[k * 3 + i], a[k], up[i]) : cmadd(u[i * 3 + k], a[k], up[i]);
      low[i] = ADJ ? cjmadd(u[k * 3 + i], b[k], low[i]) : cmadd(u[i * 3 + k], b[k], low[i]);
    }
}
// The neighbour of a direction (0-7: mu = d / 2, forward for even d).
__device__ __forceinline__ int neighbour_dir(const SysDesc& S, const Coord& c, int s, int d, float* eta) {
  return neighbour_rt(S, c, s, d >> 1, (d & 1) ? -1 : +1, eta);
}

// The FP64-class stencils (IEEE FP64 and double-float): two threads per
// output site, one per row of the half spinor; lanes 0-15 of a warp take row 0
// and lanes 16-31 row 1 of 16 consecutive sites, so that one load instruction
// serves both rows' links.  Row 0 pairs with spin 3 and row 1 with spin 2 for
// mu = x, y, with 2 and 3 for z, t.  A thread holds its upper spin and one
// lower spin: through x and y it collects the other row's lower spin, then the
// rows swap what they collected and go on with their own through z and t.
// Unit factors of (1 + s gamma_mu), h = p_row + c p_partner, lower = d g:
//   x: c = -s i, d = s i (both rows)   y: c = d = -s (row 0), s (row 1)
//   t: c = s, d = s (both rows)        z: c = -s i, d = s i (row 0), the opposite (row 1)
// Blocks: T sites x RB right-hand sides, 2 T RB threads.
// The Laplacian runs the same way with spins row and 2 + row in a thread and no
// projection.
// SPLIT: small lattices, one warp per mu for 16 sites (blocks of T sites and one
// right-hand side, 8 T threads); the mu sums meet in shared memory.  A launch on
// a few hundred warps is one thread's serial chain (FP64: 432 instructions of 64
// clocks), which this cuts to a quarter; the solver's kSplitHighSites says where.
template <int SPA, bool C12, bool DAG, class Epi, int OP = OP_WILSON, bool SPLIT = false>
__global__ void __launch_bounds__(512, 1)
    k_hop_rows(const __grid_constant__ Batch B, int par_mode, int link_slot, int in_slot, Epi epi, RedArgs ra) {
  static_assert(SPA == P64 || SPA == PDF, "two threads per site: FP64-class storage");
  using R = typename Spin<SPA>::R;
  const int T = B.T, RB = B.RB;
  const unsigned bx = B.rev ? gridDim.x - 1u - blockIdx.x : blockIdx.x;
  int by = 0, b = (int)bx, par, rl = 0;
  if (B.ny > 1) {
    b = (int)(bx / (unsigned)B.ny);
    by = (int)bx - b * B.ny;
  }
  if (par_mode == 2) {
    par = b >= B.ntot ? 1 : 0;
    b -= par * B.ntot;
  } else {
    par = par_mode;
  }
  const SysDesc& S = B.sd[block_system(B, b)];
  if (!SPLIT && RB > 1) rl = (int)threadIdx.x / (2 * T);
  const int r = by * RB + rl;
  const int tile = b - S.tile0;
  const int row = (threadIdx.x >> 4) & 1;
  const int mu = SPLIT ? (threadIdx.x >> 5) & 3 : 0;
  const int at = (SPLIT ? ((int)threadIdx.x >> 7) << 4 : (((int)threadIdx.x - rl * 2 * T) >> 5) << 4) + (threadIdx.x & 15);
  const int s0 = tile * T + at;
  const bool ok = s0 < S.vh;
  // a warp works on one right-hand side: the gate is the same for all its
  // lanes, and lanes past the last site repeat site 0 without storing
  typename RedT<R>::type nrm = red_zero(typename RedT<R>::type());
  if (r < S.nrhs && gate_of(epi.gate, ra, S.col0 + r)) {
    const int s = ok ? s0 : 0;
    const Coord c = coord_of(S, s, par);
    const int pin = par ^ 1;
    const char* in = slot_ptr(S, in_slot, r, pin);
    const char* own = slot_ptr(S, link_slot, 0, par);
    const char* nbr = slot_ptr(S, link_slot, 0, pin);
    const long long mu_stride = (long long)Link<SPA, C12>::kBytes * S.vh;
    constexpr uint32_t kS = DAG ? 0u : 0x80000000u;  // sign of the forward projector's s
    const uint32_t row1 = row ? 0x80000000u : 0u;
    Cx<R> up[3], low[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) up[k] = low[k] = cx((R)0, (R)0);
    extern __shared__ __align__(16) char ring_[];
    if constexpr (SPLIT) {
      constexpr int kArea = SPA == PDF ? RowRing<C12>::kBytes : 3072;  // shared memory of a warp
      char* area = ring_ + (threadIdx.x >> 5) * kArea;
      float ef, eb;
      const int nf = neighbour_dir(S, c, s, 2 * mu, &ef), nb = neighbour_dir(S, c, s, 2 * mu + 1, &eb);
      const uint32_t bf = __float_as_uint(ef) & 0x80000000u, bb = __float_as_uint(eb) & 0x80000000u;
      const int partner = mu < 2 ? 3 - row : 2 + row;
      const uint32_t mi = kS ^ (mu == 0 ? 0u : row1), mr = kS ^ (mu == 1 ? row1 ^ 0x80000000u : 0u);
      own += mu * mu_stride;
      nbr += mu * mu_stride;
      if constexpr (SPA == PDF) {
        using Ring = RowRing<C12>;
        Ring::issue(area, in, own, S.vh, nf, s);
        Ring::issue(area + Ring::kStage, in, nbr, S.vh, nb, nb);
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
        if constexpr (OP == OP_LAPLACE) {
          lap_direction<C12, false>(area, row, bf, up, low);
          lap_direction<C12, true>(area + Ring::kStage, row, bb, up, low);
        } else if (mu == 0 || mu == 2) {
          Ring::template direction<true, false>(area, row, partner, mi ^ 0x80000000u, mi, bf, up, low);
          Ring::template direction<true, true>(area + Ring::kStage, row, partner, mi, mi ^ 0x80000000u, bb, up, low);
        } else {
          Ring::template direction<false, false>(area, row, partner, mr, mr, bf, up, low);
          Ring::template direction<false, true>(area + Ring::kStage, row, partner, mr ^ 0x80000000u, mr ^ 0x80000000u, bb, up,
                                                low);
        }
      } else if constexpr (OP == OP_LAPLACE) {
        lap_direction<C12, false>(S, in, own, nf, s, row, bf, up, low);
        lap_direction<C12, true>(S, in, nbr, nb, nb, row, bb, up, low);
      } else if (mu == 0 || mu == 2) {
        row_mu<C12, true>(S, in, own, nbr, s, nf, nb, row, partner, mi ^ 0x80000000u, mi, bf, bb, up, low, true);
      } else {
        row_mu<C12, false>(S, in, own, nbr, s, nf, nb, row, partner, mr, mr, bf, bb, up, low, true);
      }
      if (OP == OP_WILSON && mu < 2) {
#pragma unroll
        for (int k = 0; k < 3; ++k) low[k] = other_row(low[k]);
      }
      __syncwarp();  // the ring has been read
      Cx<R>* mine = reinterpret_cast<Cx<R>*>(area) + (threadIdx.x & 31);  // [6][32], then mu + 1's and so on
      if (mu != 0) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          mine[k * 32] = up[k];
          mine[(3 + k) * 32] = low[k];
        }
      }
      __syncthreads();
      if (mu == 0) {
#pragma unroll
        for (int m = 1; m < 4; ++m) {
          const Cx<R>* p = reinterpret_cast<const Cx<R>*>(area + m * kArea) + (threadIdx.x & 31);
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            up[k] = row_add(up[k], p[k * 32]);
            low[k] = row_add(low[k], p[(3 + k) * 32]);
          }
        }
      }
    } else if constexpr (SPA == PDF) {
      // x and y, then z and t: one copy of the code for both halves, which keeps
      // the kernel inside the instruction cache
      using Ring = RowRing<C12>;
      char* stage = ring_ + (threadIdx.x >> 5) * Ring::kBytes;
      float eta;
      int n = neighbour_dir(S, c, s, 0, &eta);
      Ring::issue(stage, in, own, S.vh, n, s);
      uint32_t bm = 0u;  // boundary sign of the direction in the current stage
#pragma unroll 1
      for (int ph = 0; ph < 2; ++ph) {
        const int partner = ph == 0 ? 3 - row : 2 + row;
        const uint32_t mi = kS ^ (ph == 0 ? 0u : row1), mr = kS ^ (ph == 0 ? row1 ^ 0x80000000u : 0u);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int d = 4 * ph + k;
          uint32_t next_bm = 0u;
          __syncwarp();  // the stage about to be refilled has been read
          if (k < 3 || ph == 0) {
            n = neighbour_dir(S, c, s, d + 1, &eta);
            next_bm = __float_as_uint(eta) & 0x80000000u;
            const bool back = (k + 1) & 1;
            Ring::issue(stage + ((k + 1) & 1) * Ring::kStage, in, (back ? nbr : own) + ((d + 1) >> 1) * mu_stride, S.vh, n,
                        back ? n : s);
            asm volatile("cp.async.wait_group 1;" ::: "memory");
          } else {
            asm volatile("cp.async.wait_group 0;" ::: "memory");
          }
          __syncwarp();
          const char* st = stage + (k & 1) * Ring::kStage;
          if constexpr (OP == OP_LAPLACE) {
            if (k & 1) lap_direction<C12, true>(st, row, k < 2 ? 0u : bm, up, low);
            else lap_direction<C12, false>(st, row, k < 2 ? 0u : bm, up, low);
          } else if (k == 0) Ring::template direction<true, false>(st, row, partner, mi ^ 0x80000000u, mi, 0u, up, low);
          else if (k == 1) Ring::template direction<true, true>(st, row, partner, mi, mi ^ 0x80000000u, 0u, up, low);
          else if (k == 2) Ring::template direction<false, false>(st, row, partner, mr, mr, bm, up, low);
          else Ring::template direction<false, true>(st, row, partner, mr ^ 0x80000000u, mr ^ 0x80000000u, bm, up, low);
          bm = next_bm;
        }
        if (OP == OP_WILSON && ph == 0) {
#pragma unroll
          for (int k = 0; k < 3; ++k) low[k] = other_row(low[k]);
        }
      }
    } else if constexpr (OP == OP_LAPLACE) {
#pragma unroll 1
      for (int mu = 0; mu < 4; ++mu) {
        float ef, eb;
        const int nf = neighbour_dir(S, c, s, 2 * mu, &ef), nb = neighbour_dir(S, c, s, 2 * mu + 1, &eb);
        lap_direction<C12, false>(S, in, own, nf, s, row, __float_as_uint(ef) & 0x80000000u, up, low);
        lap_direction<C12, true>(S, in, nbr, nb, nb, row, __float_as_uint(eb) & 0x80000000u, up, low);
        own += mu_stride;
        nbr += mu_stride;
      }
    } else {
#pragma unroll 1
      for (int ph = 0; ph < 2; ++ph) {
        const int partner = ph == 0 ? 3 - row : 2 + row;
        float ef, eb;
        int nf = ph == 0 ? neighbour<0, +1>(S, c, s, &ef) : neighbour<2, +1>(S, c, s, &ef);
        int nb = ph == 0 ? neighbour<0, -1>(S, c, s, &eb) : neighbour<2, -1>(S, c, s, &eb);
        const uint32_t mi = kS ^ (ph == 0 ? 0u : row1);
        row_mu<C12, true>(S, in, own, nbr, s, nf, nb, row, partner, mi ^ 0x80000000u, mi, 0u, 0u, up, low, ph == 0);
        own += mu_stride;
        nbr += mu_stride;
        nf = ph == 0 ? neighbour<1, +1>(S, c, s, &ef) : neighbour<3, +1>(S, c, s, &ef);
        nb = ph == 0 ? neighbour<1, -1>(S, c, s, &eb) : neighbour<3, -1>(S, c, s, &eb);
        const uint32_t mr = kS ^ (ph == 0 ? row1 ^ 0x80000000u : 0u);
        row_mu<C12, false>(S, in, own, nbr, s, nf, nb, row, partner, mr, mr, __float_as_uint(ef) & 0x80000000u,
                           __float_as_uint(eb) & 0x80000000u, up, low, false);
        own += mu_stride;
        nbr += mu_stride;
        if (ph == 0) {
#pragma unroll
          for (int k = 0; k < 3; ++k) low[k] = other_row(low[k]);
        }
      }
    }
    if constexpr (SPA == PDF) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        up[k] = cx(renorm(up[k].re), renorm(up[k].im));
        low[k] = cx(renorm(low[k].re), renorm(low[k].im));
      }
    }
    if (mu == 0) {
      epi.write_rows(S, par, r, s, row, up, low, nrm, ok);
      if (!ok) nrm = red_zero(typename RedT<R>::type());
    }
  }
  if constexpr (Epi::kReduce) {
    const int ntiles = par_mode == 2 ? 2 * S.tpp : S.tpp;
    reduce_block(S, SPLIT ? 8 * T : 2 * T, SPLIT ? 1 : RB, par_mode == 2 ? par * S.tpp + tile : tile, ntiles, nrm, ra, by);
  }
}

// (Since k_hop runs at 64 registers it is the faster of the two on 24^3x48 with 12
// right-hand sides, 438 against 461 us per application, although it executes a fifth
// more instructions; this one, at 128, stays for the shapes on which the tuner finds
// it ahead.)
// 16-bit stencil with two right-hand sides per thread: each link is loaded,
// and with 12-real compression its third row rebuilt, once and applied to
// both; the two neighbour loads of a direction are in flight together.  Block:
// T sites x RB thread groups, group g of right-hand-side block y taking
// right-hand sides 2(y RB + g) and 2(y RB + g) + 1, for ny = ceil(nrhs / (2 RB))
// blocks y; the grid is one-dimensional with y varying fastest.
template <int SPA, bool C12, bool DAG, class Epi>
__global__ void __launch_bounds__(256, 2)
    k_hop_pair(const __grid_constant__ Batch B, int par_mode, int link_slot, int in_slot, Epi epi, RedArgs ra) {
  static_assert(SPA == P16 || SPA == PB16, "two right-hand sides per thread: 16-bit storage");
  const int T = B.T, RB = B.RB;
  const unsigned ny = (unsigned)((B.sd[0].nrhs + 2 * RB - 1) / (2 * RB));
  const unsigned bx = B.rev ? gridDim.x - 1u - blockIdx.x : blockIdx.x;
  const int by = (int)(bx % ny);
  int b = (int)(bx / ny), par;
  if (par_mode == 2) {
    par = b >= B.ntot ? 1 : 0;
    b -= par * B.ntot;
  } else {
    par = par_mode;
  }
  const SysDesc& S = B.sd[block_system(B, b)];
  const int rl = threadIdx.x / T;
  const int r0 = (by * RB + rl) * 2, r1 = r0 + 1;
  const int tile = b - S.tile0;
  const int s = tile * T + (threadIdx.x - rl * T);
  const bool site = s < S.vh;
  const bool v0 = site && r0 < S.nrhs && gate_of(epi.gate, ra, S.col0 + r0);
  const bool v1 = site && r1 < S.nrhs && gate_of(epi.gate, ra, S.col0 + r1);
  const int r1l = r1 < S.nrhs ? r1 : r0;  // a missing second column reloads the first
  typename RedT<float>::type nrm[2] = {red_zero(typename RedT<float>::type()), red_zero(typename RedT<float>::type())};
  typename Epi::Packed po0, po1;
  if (v0 || v1) {
    const InOne<SPA> in{in_slot};
    const Coord c = coord_of(S, s, par);
    const int pin = par ^ 1;
    const char* ulink_own = slot_ptr(S, link_slot, 0, par);
    const char* ulink_nb = slot_ptr(S, link_slot, 0, pin);
    const long long mu_stride = (long long)Link<SPA, C12>::kBytes * S.vh;
    constexpr int SF = DAG ? +1 : -1;
    constexpr int SB = -SF;
    Cx<float> acc0[12], acc1[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) acc0[k] = acc1[k] = cx(0.f, 0.f);
#define DW_HOP_PAIR_DIR(MU)                                                     \
  {                                                                             \
    float eta, sc0, sc1;                                                        \
    uint32_t p0[12], p1[12], h0[6], h1[6], u[9];                                \
    Cx<float> g[6];                                                             \
    const int nf = neighbour<MU, +1>(S, c, s, &eta);                            \
    in.load_words(S, pin, r0, nf, p0, sc0);                                     \
    in.load_words(S, pin, r1l, nf, p1, sc1);                                    \
    Link<SPA, C12>::load_words(ulink_own + MU * mu_stride, S.vh, s, u);         \
    project_w<MU, SF, SPA>(p0, h0);                                             \
    project_w<MU, SF, SPA>(p1, h1);                                             \
    su3_mul_w<false, SPA>(u, h0, g);                                            \
    accumulate_w<MU, SF>(acc0, g, eta < 0.f ? -sc0 : sc0);                      \
    su3_mul_w<false, SPA>(u, h1, g);                                            \
    accumulate_w<MU, SF>(acc1, g, eta < 0.f ? -sc1 : sc1);                      \
    const int nb = neighbour<MU, -1>(S, c, s, &eta);                            \
    in.load_words(S, pin, r0, nb, p0, sc0);                                     \
    in.load_words(S, pin, r1l, nb, p1, sc1);                                    \
    Link<SPA, C12>::load_words(ulink_nb + MU * mu_stride, S.vh, nb, u);         \
    project_w<MU, SB, SPA>(p0, h0);                                             \
    project_w<MU, SB, SPA>(p1, h1);                                             \
    su3_mul_w<true, SPA>(u, h0, g);                                             \
    accumulate_w<MU, SB>(acc0, g, eta < 0.f ? -sc0 : sc0);                      \
    su3_mul_w<true, SPA>(u, h1, g);                                             \
    accumulate_w<MU, SB>(acc1, g, eta < 0.f ? -sc1 : sc1);                      \
  }
    DW_HOP_PAIR_DIR(0)
    DW_HOP_PAIR_DIR(1)
    DW_HOP_PAIR_DIR(2)
    DW_HOP_PAIR_DIR(3)
#undef DW_HOP_PAIR_DIR
    if constexpr (Epi::kReduce) {
      if (v0) po0 = epi.prepare(S, par, r0, s, acc0, nrm[0]);
      if (v1) po1 = epi.prepare(S, par, r1, s, acc1, nrm[1]);
    } else {
      if (v0) epi.write(S, par, r0, s, acc0, nrm[0]);
      if (v1) epi.write(S, par, r1, s, acc1, nrm[1]);
    }
  }
  if constexpr (Epi::kReduce) {
    const int ntiles = par_mode == 2 ? 2 * S.tpp : S.tpp;
    const int tt = par_mode == 2 ? par * S.tpp + tile : tile;
    reduce_block_n<2>(S, T, RB, tt, ntiles, nrm, ra, by, [&] {
      if (v0) epi.commit(S, par, r0, s, po0);
      if (v1) epi.commit(S, par, r1, s, po1);
    });
  }
}

// ------------------------------------------------------------------ site-local kernels
// r -= alpha w at one site: the words to store and |r|^2 as stored (the norm is
// taken of the rounded value, so the recursion sees what the next kernels read)
template <int SPL>
__device__ __forceinline__ typename Spin<SPL>::Packed update_r_site(const SysDesc& S, int par, int r, int s,
                                                                   const ColState& C,
                                                                   typename RedT<typename Spin<SPL>::R>::type& nrm) {
  using RL = typename Spin<SPL>::R;
  Cx<RL> w[12], rv[12];
  Spin<SPL>::load(slot_ptr(S, S_W, r, par), S.vh, s, w);
  Spin<SPL>::load(slot_ptr(S, S_R, r, par), S.vh, s, rv);
  const RL a = scalar_as<RL>(C.alpha, C.alpha_f);
  RL n = (RL)0;
#pragma unroll
  for (int k = 0; k < 12; ++k) rv[k] = cx(fma(-a, w[k].re, rv[k].re), fma(-a, w[k].im, rv[k].im));
  Spin<SPL>::roundtrip(rv);
#pragma unroll
  for (int k = 0; k < 12; ++k) n = fma(rv[k].re, rv[k].re, fma(rv[k].im, rv[k].im, n));
  nrm = to_red(n);
  return Spin<SPL>::pack(rv);
}

// xl += alpha_x p (the increment of the iteration that used p, unless a
// reliable update has folded it already: alpha_x = 0);  p = z + beta p
template <int SPL, int SPA>
__device__ __forceinline__ void update_p_site(const SysDesc& S, int par, int r, int s, const ColState& C) {
  using RL = typename Spin<SPL>::R;
  using RA = typename Spin<SPA>::R;
  const RL beta = scalar_as<RL>(C.beta, C.beta_f);
  Cx<RL> p[12], z[12];
  Spin<SPL>::load(slot_ptr(S, S_P, r, par), S.vh, s, p);
  Spin<SPL>::load(slot_ptr(S, S_Z, r, par), S.vh, s, z);
  if (C.alpha_x != 0.0) {
    const RA aa = scalar_as<RA>(C.alpha_x, C.alpha_xf);
    Cx<RA> xl[12];
    Spin<SPA>::load(slot_ptr(S, S_XL, r, par), S.vh, s, xl);
#pragma unroll
    for (int k = 0; k < 12; ++k) xl[k] = cx(fma(aa, (RA)p[k].re, xl[k].re), fma(aa, (RA)p[k].im, xl[k].im));
    Spin<SPA>::store(slot_wptr(S, S_XL, r, par), S.vh, s, xl);
  }
#pragma unroll
  for (int k = 0; k < 12; ++k) p[k] = cx(fma(beta, p[k].re, z[k].re), fma(beta, p[k].im, z[k].im));
  Spin<SPL>::store(slot_wptr(S, S_P, r, par), S.vh, s, p);
}

// r -= alpha w;  reduction |r|^2 -> FIN_UPDATE.  The matching x-increment
// xl += alpha p is left to k_update_p (which reads p anyway) or, when a
// reliable update comes first, to k_fold_x: ColState::alpha_x holds it.
template <int SPL>
__global__ void __launch_bounds__(256) k_update_r(const __grid_constant__ Batch B, int par_mode, RedArgs ra) {
  DW_BLOCK_PROLOGUE(G_ACTIVE)
  using RL = typename Spin<SPL>::R;
  typename RedT<RL>::type nrm = red_zero(typename RedT<RL>::type());
  typename Spin<SPL>::Packed rp;
  if (valid) rp = update_r_site<SPL>(S, par, r, s, ra.cols[S.col0 + r], nrm);
  ra.fin = FIN_UPDATE;
  DW_BLOCK_REDUCE_STORE(nrm, [&] {
    if (valid) Spin<SPL>::store_packed(slot_wptr(S, S_R, r, par), S.vh, s, rp);
  })
}

// The while-node condition set by the loop's last kernel (on = 0: no loop).
struct LoopCond {
  unsigned long long handle;
  int on;
};

// xl += alpha_x p;  p = z + beta p (update_p_site)
template <int SPL, int SPA>
__global__ void __launch_bounds__(256) k_update_p(const __grid_constant__ Batch B, int par_mode, RedArgs ra,
                                                  LoopCond lc) {
  // last kernel of an iteration: decides whether the device-driven loop goes on
  // (no kernel of its own: a one-thread node costs about 2 us per iteration)
  if (lc.on && blockIdx.x == 0 && threadIdx.x == 0) {
    const int loops = ra.flags->loops + 1;
    ra.flags->loops = loops;
    cudaGraphSetConditional(lc.handle, (ra.flags->active > 0 && loops < ra.flags->max_loops) ? 1u : 0u);
  }
  DW_BLOCK_PROLOGUE(G_ACTIVE)
  if (valid) update_p_site<SPL, SPA>(S, par, r, s, ra.cols[S.col0 + r]);
}

// First residual for a zero initial guess: r_low = src, reduction |src|^2 -> FIN_RESID0
template <int SPL, int SPH>
__global__ void __launch_bounds__(256) k_init_r(const __grid_constant__ Batch B, int par_mode, int slot_src, RedArgs ra) {
  DW_BLOCK_PROLOGUE(G_XZERO)
  using RH = typename Spin<SPH>::R;
  typename RedT<RH>::type nrm = red_zero(typename RedT<RH>::type());
  if (valid) {
    Cx<RH> v[12];
    Cx<typename Spin<SPL>::R> lo[12];
    Spin<SPH>::load(slot_ptr(S, slot_src, r, par), S.vh, s, v);
    RH n = (RH)0;
#pragma unroll
    for (int k = 0; k < 12; ++k) n = fma(v[k].re, v[k].re, fma(v[k].im, v[k].im, n));
    nrm = to_red(n);
    convert12(v, lo);
    Spin<SPL>::store(slot_wptr(S, S_R, r, par), S.vh, s, lo);
  }
  DW_BLOCK_REDUCE(nrm)
}

// x += xl + alpha_x p; xl = 0 on the launched parities (start of a reliable
// update: the pending increment of the current iteration is added first, in
// the increment's precision, as k_update_p would have)
template <int SPL, int SPA, int SPH>
__global__ void __launch_bounds__(256) k_fold_x(const __grid_constant__ Batch B, int par_mode, RedArgs ra) {
  DW_BLOCK_PROLOGUE(G_REL)
  if (valid) {
    using RL = typename Spin<SPL>::R;
    using RA = typename Spin<SPA>::R;
    using RH = typename Spin<SPH>::R;
    const ColState& C = ra.cols[S.col0 + r];
    Cx<RH> x[12];
    Cx<RA> xl[12];
    Spin<SPH>::load(slot_ptr(S, S_X, r, par), S.vh, s, x);
    Spin<SPA>::load(slot_ptr(S, S_XL, r, par), S.vh, s, xl);
    if (C.alpha_x != 0.0) {
      const RA aa = scalar_as<RA>(C.alpha_x, C.alpha_xf);
      Cx<RL> p[12];
      Spin<SPL>::load(slot_ptr(S, S_P, r, par), S.vh, s, p);
#pragma unroll
      for (int k = 0; k < 12; ++k) xl[k] = cx(fma(aa, (RA)p[k].re, xl[k].re), fma(aa, (RA)p[k].im, xl[k].im));
      Spin<SPA>::roundtrip(xl);
    }
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      x[k] = cx(x[k].re + (RH)xl[k].re, x[k].im + (RH)xl[k].im);
      xl[k] = cx((RA)0, (RA)0);
    }
    Spin<SPH>::store(slot_wptr(S, S_X, r, par), S.vh, s, x);
    Spin<SPA>::store(slot_wptr(S, S_XL, r, par), S.vh, s, xl);
  }
}

// |field|^2 of slot over the launched parities -> finalizer ra.fin (gate: all)
template <int SP>
__global__ void __launch_bounds__(256) k_norm(const __grid_constant__ Batch B, int par_mode, int slot, RedArgs ra) {
  DW_BLOCK_PROLOGUE(G_ALL)
  using RS = typename Spin<SP>::R;
  typename RedT<RS>::type nrm = red_zero(typename RedT<RS>::type());
  if (valid) {
    Cx<RS> v[12];
    Spin<SP>::load(slot_ptr(S, slot, r, par), S.vh, s, v);
    RS n = (RS)0;
#pragma unroll
    for (int k = 0; k < 12; ++k) n = fma(v[k].re, v[k].re, fma(v[k].im, v[k].im, n));
    nrm = to_red(n);
  }
  DW_BLOCK_REDUCE(nrm)
}

// dst = convert(src) and |src|^2 -> finalizer ra.fin, in one pass over src (gate: all)
template <int SPD, int SPS>
__global__ void __launch_bounds__(256) k_convert_norm(const __grid_constant__ Batch B, int par_mode, int slot_dst,
                                                      int slot_src, RedArgs ra) {
  DW_BLOCK_PROLOGUE(G_ALL)
  using RS = typename Spin<SPS>::R;
  typename RedT<RS>::type nrm = red_zero(typename RedT<RS>::type());
  if (valid) {
    Cx<RS> v[12];
    Cx<typename Spin<SPD>::R> o[12];
    Spin<SPS>::load(slot_ptr(S, slot_src, r, par), S.vh, s, v);
    RS n = (RS)0;
#pragma unroll
    for (int k = 0; k < 12; ++k) n = fma(v[k].re, v[k].re, fma(v[k].im, v[k].im, n));
    nrm = to_red(n);
    convert12(v, o);
    Spin<SPD>::store(slot_wptr(S, slot_dst, r, par), S.vh, s, o);
  }
  DW_BLOCK_REDUCE(nrm)
}

// Odd-site reconstruction x_o = b_o + kappa t_o, t_o = H_oe x_e as left in the
// odd half of S_RT by the last reliable update, in the high precision SPH.
template <int SPH, typename R>
__device__ __forceinline__ void recon_odd(const SysDesc& S, int r, int s, Cx<R> (&xv)[12]) {
  Cx<R> bv[12], tv[12];
  Spin<SPH>::load(slot_ptr(S, S_B, r, 1), S.vh, s, bv);
  Spin<SPH>::load(slot_ptr(S, S_RT, r, 1), S.vh, s, tv);
  const R k = coef<C_PK, R>(S);
#pragma unroll
  for (int j = 0; j < 12; ++j) xv[j] = cx(fma(k, tv[j].re, bv[j].re), fma(k, tv[j].im, bv[j].im));
}
template <int SPH>
__global__ void __launch_bounds__(256) k_recon_odd(const __grid_constant__ Batch B, int par_mode, RedArgs ra) {
  DW_BLOCK_PROLOGUE(G_ALL)
  if (valid) {
    Cx<typename Spin<SPH>::R> xv[12];
    recon_odd<SPH>(S, r, s, xv);
    Spin<SPH>::store(slot_wptr(S, S_X, r, par), S.vh, s, xv);
  }
}

// The caller's solution (FP64) from the accumulator in SPH: S_XU <- S_X, on odd
// sites of an even-odd system (recon) the reconstruction, 0 for a zero source.
// One pass instead of reconstruction, conversion and zeroing (32^3x64: 228 us in
// three kernels, the odd sites written and read once more in between).
template <int SPH>
__global__ void __launch_bounds__(256) k_solution(const __grid_constant__ Batch B, int par_mode, int recon, RedArgs ra) {
  DW_BLOCK_PROLOGUE(G_ALL)
  if (valid) {
    Cx<typename Spin<SPH>::R> xv[12];
    Cx<double> o[12];
    if (recon && par == 1) recon_odd<SPH>(S, r, s, xv);
    else Spin<SPH>::load(slot_ptr(S, S_X, r, par), S.vh, s, xv);
    const bool zero = ra.cols[S.col0 + r].zsrc != 0;
#pragma unroll
    for (int k = 0; k < 12; ++k) o[k] = zero ? cx(0.0, 0.0) : cx((double)xv[k].re, (double)xv[k].im);
    Spin<P64>::store(slot_wptr(S, S_XU, r, par), S.vh, s, o);
  }
}

// field <- 0 for the columns with a zero source (gate G_ZSRC)
template <int SP>
__global__ void __launch_bounds__(256) k_zero_zsrc(const __grid_constant__ Batch B, int par_mode, int slot, RedArgs ra) {
  DW_BLOCK_PROLOGUE(G_ZSRC)
  if (valid) {
    Cx<typename Spin<SP>::R> z[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) z[k] = cx((typename Spin<SP>::R)0, (typename Spin<SP>::R)0);
    Spin<SP>::store(slot_wptr(S, slot, r, par), S.vh, s, z);
  }
}

}  // namespace dw
