// Device building blocks of the Wilson-clover matrix, Eq. (2):
//   M = -1/2 sum_mu [ (1 - g_mu) (x) U_mu(x) d_{x+mu,x'} + (1 + g_mu) (x) U_mu(x-mu)^dag d_{x-mu,x'} ]
//       + (4 + m + A_x) d_{x,x'}
// in the DeGrand-Rossi chiral basis, where every gamma_mu = [[0, B],[C, 0]]
// is off-diagonal in chirality with CB = 1.  Hence
//   (1 - g) psi = [h ; -C h],  h = psi_u - B psi_l,
//   (1 + g) psi = [h ;  C h],  h = psi_u + B psi_l,
// and a hop costs one colour multiply of a 2-spinor.
// Spinor dof = spin*3 + colour; spins 0,1 (upper) are chirality 0.
#pragma once

#include "common.cuh"

namespace gbmg {

// (B_mu l) for the lower 2-spinor l = (l0, l1) of one colour.
template <int MU, typename R>
__device__ __forceinline__ void Bmul(cpx<R> l0, cpx<R> l1, cpx<R>& o0, cpx<R>& o1) {
  if constexpr (MU == 0) {         // B = i s1
    o0 = times_i(l1);
    o1 = times_i(l0);
  } else if constexpr (MU == 1) {  // B = -i s2 = [[0,-1],[1,0]]
    o0 = -l1;
    o1 = l0;
  } else if constexpr (MU == 2) {  // B = i s3
    o0 = times_i(l0);
    o1 = -times_i(l1);
  } else {                         // B = 1
    o0 = l0;
    o1 = l1;
  }
}

// (C_mu u) for the upper 2-spinor u of one colour.
template <int MU, typename R>
__device__ __forceinline__ void Cmul(cpx<R> u0, cpx<R> u1, cpx<R>& o0, cpx<R>& o1) {
  if constexpr (MU == 0) {         // C = -i s1
    o0 = -times_i(u1);
    o1 = -times_i(u0);
  } else if constexpr (MU == 1) {  // C = i s2 = [[0,1],[-1,0]]
    o0 = u1;
    o1 = -u0;
  } else if constexpr (MU == 2) {  // C = -i s3
    o0 = -times_i(u0);
    o1 = times_i(u1);
  } else {                         // C = 1
    o0 = u0;
    o1 = u1;
  }
}

// acc += -1/2 (1 - g_mu) (x) U  psi     (forward hop, U = U_mu(x))
// acc += -1/2 (1 + g_mu) (x) U^dag psi  (backward hop, U = U_mu(x - mu))
template <int MU, bool FWD, typename R>
__device__ __forceinline__ void hop_accum(const cpx<R>* __restrict__ U, const cpx<R> psi[12],
                                          cpx<R> acc[12]) {
  cpx<R> h[2][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    cpx<R> b0, b1;
    Bmul<MU>(psi[6 + k], psi[9 + k], b0, b1);
    if (FWD) {
      h[0][k] = psi[k] - b0;
      h[1][k] = psi[3 + k] - b1;
    } else {
      h[0][k] = psi[k] + b0;
      h[1][k] = psi[3 + k] + b1;
    }
  }
  cpx<R> w[2][3];
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      cpx<R> t(R(0), R(0));
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (FWD)
          cmac(t, U[a * 3 + b], h[s][b]);
        else
          cmac_conj(t, U[b * 3 + a], h[s][b]);  // (U^dag)_{ab} = conj(U_{ba})
      }
      w[s][a] = t;
    }
  const R half = R(0.5);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    cpx<R> c0, c1;
    Cmul<MU>(w[0][a], w[1][a], c0, c1);
    acc[a] -= half * w[0][a];
    acc[3 + a] -= half * w[1][a];
    if (FWD) {
      acc[6 + a] += half * c0;
      acc[9 + a] += half * c1;
    } else {
      acc[6 + a] -= half * c0;
      acc[9 + a] -= half * c1;
    }
  }
}

// hop_accum on a spinor and an accumulator kept as two halves of one
// chirality each, first the upper (sg = 1) or the lower half (sg = -1).  With
// CB = 1 the projection (1 -+ g) psi = [h; -+C h], h = psi_u -+ B psi_l, reads
// [-+B h'; h'] with h' = psi_l -+ C psi_u from the lower half, and C_mu =
// -B_mu for mu < 3, C_3 = B_3: the same steps with the sign sg on the terms
// that cross the halves, for mu < 3.
template <int MU, bool FWD, typename R>
__device__ __forceinline__ void hop_halves(const cpx<R>* __restrict__ U, const cpx<R> x[6],
                                           const cpx<R> y[6], cpx<R> ax[6], cpx<R> ay[6], R sg) {
  cpx<R> h[2][3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    cpx<R> b[2];
    Bmul<MU>(y[k], y[3 + k], b[0], b[1]);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if constexpr (MU == 3) {
        h[s][k] = FWD ? x[3 * s + k] - b[s] : x[3 * s + k] + b[s];
      } else {
        h[s][k] = cpx<R>(fma(FWD ? -sg : sg, b[s].re, x[3 * s + k].re),
                         fma(FWD ? -sg : sg, b[s].im, x[3 * s + k].im));
      }
    }
  }
  const R half = R(0.5), hs = MU == 3 ? half : half * sg;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    cpx<R> w[2], c[2];
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      cpx<R> t(R(0), R(0));
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (FWD)
          cmac(t, U[a * 3 + b], h[s][b]);
        else
          cmac_conj(t, U[b * 3 + a], h[s][b]);  // (U^dag)_{ab} = conj(U_{ba})
      }
      w[s] = t;
    }
    Cmul<MU>(w[0], w[1], c[0], c[1]);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      ax[3 * s + a] -= half * w[s];
      if (FWD)
        ay[3 * s + a] += hs * c[s];
      else
        ay[3 * s + a] -= hs * c[s];
    }
  }
}

// One complex quantity of two vectors: both real parts in one register pair,
// both imaginary parts in another.
struct cpx2 {
  f32x2 re, im;
};
__device__ __forceinline__ cpx2 pack_pair(cpx<float> a, cpx<float> b) {
  return cpx2{pack2f(a.re, b.re), pack2f(a.im, b.im)};
}
__device__ __forceinline__ void unpack_pair(cpx2 v, cpx<float>& a, cpx<float>& b) {
  unpack2f(v.re, a.re, b.re);
  unpack2f(v.im, a.im, b.im);
}

// hop_halves on two vectors a, b with one link: the projections per vector,
// the colour multiplication and the accumulation in packed arithmetic (half
// the issue slots, and none of the register-read stalls of FMAs with three
// distinct sources).
template <int MU, bool FWD>
__device__ __forceinline__ void hop_halves2(const cpx<float>* __restrict__ U,
                                            const cpx<float> xa[6], const cpx<float> ya[6],
                                            const cpx<float> xb[6], const cpx<float> yb[6],
                                            cpx2 ax[6], cpx2 ay[6], float sg) {
  // projected pairs; n: the negated part that the colour product needs
  cpx2 h[2][3];
  f32x2 n[2][3];
  auto project = [&](const cpx<float>* x, const cpx<float>* y, int k, cpx<float> r[2]) {
    cpx<float> b[2];
    Bmul<MU>(y[k], y[3 + k], b[0], b[1]);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if constexpr (MU == 3) {
        r[s] = FWD ? x[3 * s + k] - b[s] : x[3 * s + k] + b[s];
      } else {
        r[s] = cpx<float>(fmaf(FWD ? -sg : sg, b[s].re, x[3 * s + k].re),
                          fmaf(FWD ? -sg : sg, b[s].im, x[3 * s + k].im));
      }
    }
  };
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    cpx<float> pa[2], pb[2];
    project(xa, ya, k, pa);
    project(xb, yb, k, pb);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      h[s][k] = pack_pair(pa[s], pb[s]);
      // U h: re -= u.im h.im; U^dag h: im -= u.im h.re
      n[s][k] = FWD ? pack2f(-pa[s].im, -pb[s].im) : pack2f(-pa[s].re, -pb[s].re);
    }
  }
  const float hv = MU == 3 ? 0.5f : 0.5f * sg;
  const f32x2 mh = pack2f(-0.5f, -0.5f), hs = pack2f(hv, hv), nh = pack2f(-hv, -hv);
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    cpx2 w[2];
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const cpx<float> u = FWD ? U[a * 3 + b] : U[b * 3 + a];
      const f32x2 ur = pack2f(u.re, u.re), ui = pack2f(u.im, u.im);
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        if (b == 0) {
          w[s].re = mul2(ur, h[s][b].re);
          w[s].im = mul2(ur, h[s][b].im);
        } else {
          fma2(w[s].re, ur, h[s][b].re);
          fma2(w[s].im, ur, h[s][b].im);
        }
        if (FWD) {
          fma2(w[s].re, ui, n[s][b]);
          fma2(w[s].im, ui, h[s][b].re);
        } else {
          fma2(w[s].re, ui, h[s][b].im);
          fma2(w[s].im, ui, n[s][b]);
        }
      }
    }
    // first half -= w / 2; second half +- C_mu w / 2 (fwd +), the sign folded
    // into hs / nh
    const f32x2 p = FWD ? hs : nh, m = FWD ? nh : hs;
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      fma2(ax[3 * s + a].re, mh, w[s].re);
      fma2(ax[3 * s + a].im, mh, w[s].im);
    }
    if constexpr (MU == 0) {         // C w = (-i w1, -i w0)
      fma2(ay[a].re, p, w[1].im);
      fma2(ay[a].im, m, w[1].re);
      fma2(ay[3 + a].re, p, w[0].im);
      fma2(ay[3 + a].im, m, w[0].re);
    } else if constexpr (MU == 1) {  // (w1, -w0)
      fma2(ay[a].re, p, w[1].re);
      fma2(ay[a].im, p, w[1].im);
      fma2(ay[3 + a].re, m, w[0].re);
      fma2(ay[3 + a].im, m, w[0].im);
    } else if constexpr (MU == 2) {  // (-i w0, i w1)
      fma2(ay[a].re, p, w[0].im);
      fma2(ay[a].im, m, w[0].re);
      fma2(ay[3 + a].re, m, w[1].im);
      fma2(ay[3 + a].im, p, w[1].re);
    } else {                         // (w0, w1)
      fma2(ay[a].re, p, w[0].re);
      fma2(ay[a].im, p, w[0].im);
      fma2(ay[3 + a].re, p, w[1].re);
      fma2(ay[3 + a].im, p, w[1].im);
    }
  }
}

// Runtime-mu dispatch of hop_accum.
template <typename R>
__device__ __forceinline__ void hop_accum_rt(int mu, bool fwd, const cpx<R>* __restrict__ U,
                                             const cpx<R> psi[12], cpx<R> acc[12]) {
  switch (mu * 2 + (fwd ? 0 : 1)) {
    case 0: hop_accum<0, true>(U, psi, acc); break;
    case 1: hop_accum<0, false>(U, psi, acc); break;
    case 2: hop_accum<1, true>(U, psi, acc); break;
    case 3: hop_accum<1, false>(U, psi, acc); break;
    case 4: hop_accum<2, true>(U, psi, acc); break;
    case 5: hop_accum<2, false>(U, psi, acc); break;
    case 6: hop_accum<3, true>(U, psi, acc); break;
    default: hop_accum<3, false>(U, psi, acc); break;
  }
}

// acc += (diag + A_x) psi with A_x stored as two packed 6x6 Hermitian blocks
// (per chirality: 6 real diagonal entries, then the 15 complex entries
// below the diagonal in row order).
template <typename R>
__device__ __forceinline__ void clover_accum(const R* __restrict__ A, R diag, const cpx<R> psi[12],
                                             cpx<R> acc[12]) {
#pragma unroll
  for (int chi = 0; chi < 2; ++chi) {
    const R* a = A + chi * 36;
    const cpx<R>* in = psi + chi * 6;
    cpx<R>* out = acc + chi * 6;
#pragma unroll
    for (int i = 0; i < 6; ++i) out[i] += (diag + a[i]) * in[i];
#pragma unroll
    for (int i = 1; i < 6; ++i)
#pragma unroll
      for (int j = 0; j < i; ++j) {
        int k = i * (i - 1) / 2 + j;
        cpx<R> l(a[6 + 2 * k], a[7 + 2 * k]);
        cmac(out[i], l, in[j]);
        cmac_conj(out[j], l, in[i]);
      }
  }
}

// clover_accum with element k of the packed clover at A[k * stride] (a
// transposed shared-memory tile).
template <typename R>
__device__ __forceinline__ void clover_accum_strided(const R* __restrict__ A, int stride, R diag,
                                                     const cpx<R> psi[12], cpx<R> acc[12]) {
#pragma unroll
  for (int chi = 0; chi < 2; ++chi) {
    const R* a = A + chi * 36 * stride;
    const cpx<R>* in = psi + chi * 6;
    cpx<R>* out = acc + chi * 6;
#pragma unroll
    for (int i = 0; i < 6; ++i) out[i] += (diag + a[i * stride]) * in[i];
#pragma unroll
    for (int i = 1; i < 6; ++i)
#pragma unroll
      for (int j = 0; j < i; ++j) {
        int k = i * (i - 1) / 2 + j;
        cpx<R> l(a[(6 + 2 * k) * stride], a[(7 + 2 * k) * stride]);
        cmac(out[i], l, in[j]);
        cmac_conj(out[j], l, in[i]);
      }
  }
}

// acc6 += (diag + A_chi) psi6 for one packed 6x6 Hermitian chirality block.
template <typename R>
__device__ __forceinline__ void clover_block_accum(const R* __restrict__ a, R diag,
                                                   const cpx<R> in[6], cpx<R> out[6]) {
#pragma unroll
  for (int i = 0; i < 6; ++i) out[i] += (diag + a[i]) * in[i];
#pragma unroll
  for (int i = 1; i < 6; ++i)
#pragma unroll
    for (int j = 0; j < i; ++j) {
      int k = i * (i - 1) / 2 + j;
      cpx<R> l(a[6 + 2 * k], a[7 + 2 * k]);
      cmac(out[i], l, in[j]);
      cmac_conj(out[j], l, in[i]);
    }
}

}  // namespace gbmg
