// Homogenisation rules of section 2 -- Voigt (eq. 3), Reuss (eq. 4) and the 2-layer laminate
// (eqs. 5-a, 5-b) -- of isotropic phases, in closed form: Voigt and Reuss give an isotropic medium
// (averages of the moduli, or of their inverses), the laminate a medium with five constants about the
// interface normal.  The constants are templated on the scalar type, so that the filter build
// evaluates them in double and the backward pass differentiates them in forward mode with the dual
// numbers below.  FP64 arithmetic is scarce on this GPU: the laminate as a block formula on rotated
// 6 x 6 matrices held in local memory took 1.06 ms for the 344 k mixed voxels of a 135^3 cell (and its
// dual-number form 19 ms for the 111 k mixed voxels of an 81^3 gradient); the closed form takes
// 0.36 ms (and 0.95 ms for the whole gradient kernel).
#pragma once

#include <cmath>

#include "hom_common.cuh"

namespace hom {

// Forward-mode dual number v + d eps (eps^2 = 0).
struct Dual {
  double v, d;
};
HOM_HD Dual operator+(Dual a, Dual b) { return {a.v + b.v, a.d + b.d}; }
HOM_HD Dual operator-(Dual a, Dual b) { return {a.v - b.v, a.d - b.d}; }
HOM_HD Dual operator*(Dual a, Dual b) { return {a.v * b.v, a.v * b.d + a.d * b.v}; }
HOM_HD Dual operator/(Dual a, Dual b) { return {a.v / b.v, (a.d * b.v - a.v * b.d) / (b.v * b.v)}; }
HOM_HD Dual operator*(double a, Dual b) { return {a * b.v, a * b.d}; }

template <typename S> HOM_HD S scal(double x);
template <> HOM_HD double scal<double>(double x) { return x; }
template <> HOM_HD Dual scal<Dual>(double x) { return {x, 0.0}; }

// Isotropic medium: lam 1 (x) 1 + 2 mu I (plane strain in 2D).
template <typename S> struct Iso {
  S lam, mu;
};

// Eq. 3: sum_k f_k c_k over K entries (unused ones hold f = 0).
template <int K, typename S>
HOM_HD Iso<S> voigt_moduli(const S* lam, const S* mu, const S* f) {
  Iso<S> r{f[0] * lam[0], f[0] * mu[0]};
#pragma unroll
  for (int k = 1; k < K; ++k) r = {r.lam + f[k] * lam[k], r.mu + f[k] * mu[k]};
  return r;
}

// Eq. 4: (sum_k f_k c_k^-1)^-1 over the first nph of K entries; the eigenvalues dim lam + 2 mu and 2 mu
// of isotropic media are averaged harmonically.
template <int K, typename S>
HOM_HD Iso<S> reuss_moduli(const S* lam, const S* mu, const S* f, int nph, int dim) {
  S ik = scal<S>(0.0), im = scal<S>(0.0);
#pragma unroll
  for (int k = 0; k < K; ++k)
    if (k < nph) {
      ik = ik + f[k] / ((double)dim * lam[k] + 2.0 * mu[k]);
      im = im + f[k] / mu[k];
    }
  const S m = scal<S>(1.0) / im, kap = scal<S>(1.0) / ik;
  return {(1.0 / dim) * (kap - 2.0 * m), m};
}

// Eqs. 5-a, 5-b for two isotropic phases in layers: with M = lam + 2 mu and <.> the average by volume,
//   cn  = <1/M>^-1              stiffness along the normal
//   F   = <1/M>^-1 <lam/M>      coupling of the normal with the layers' plane
//   B   = 2 <lam mu/M> + <1/M>^-1 <lam/M>^2, mup = <mu>   in the plane: B tr I + 2 mup
//   mun = <1/mu>^-1             shear across the layers
// Every term is a sum of positive ones (lam > 0): no cancellation at high contrast.
template <typename S> struct Layered {
  S cn, F, B, mup, mun;
};
template <typename S>
HOM_HD Layered<S> layered_moduli(const S* lam, const S* mu, const S* f) {
  S iM = scal<S>(0.0), lM = iM, lmM = iM, mup = iM, im = iM;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const S w = f[k] / (lam[k] + 2.0 * mu[k]);
    const S wl = w * lam[k];
    iM = iM + w;
    lM = lM + wl;
    lmM = lmM + wl * mu[k];
    mup = mup + f[k] * mu[k];
    im = im + f[k] / mu[k];
  }
  const S one = scal<S>(1.0), cn = one / iM, F = cn * lM;
  return {cn, F, 2.0 * lmM + F * lM, mup, one / im};
}

// Mandel components of the tensors a layered medium about the unit normal n is made of:
//   c = cn N N^T + F (N p^T + p N^T) + B p p^T + 2 mup (I - 2 Q + N N^T) + 4 mun (Q - N N^T)
// with N = n (x) n, p = 1 - n (x) n, and Q = sum_i s_i s_i^T, s_i = sym(e_i (x) n).
template <int DIM> struct LayerBasis {
  static constexpr int NC = DIM == 2 ? 3 : 6;
  double n[DIM], N[NC], p[NC];
  HOM_HD explicit LayerBasis(const double* nrm) {
    const double s2 = 1.4142135623730950488;
    for (int d = 0; d < DIM; ++d) n[d] = nrm[d];
#pragma unroll
    for (int I = 0; I < NC; ++I) {
      int i, j;
      pair_of(I, i, j);
      N[I] = (i == j ? 1.0 : s2) * n[i] * n[j];
      p[I] = (I < DIM ? 1.0 : 0.0) - N[I];
    }
  }
  HOM_HD static constexpr void pair_of(int I, int& i, int& j) {
    if (DIM == 2) {
      i = I == 1 ? 1 : 0;
      j = I == 0 ? 0 : 1;
    } else {
      i = I < 3 ? I : I == 3 ? 1 : 0;
      j = I < 3 ? I : I == 5 ? 1 : 2;
    }
  }
  // component I of s_a = sym(e_a (x) n)
  HOM_HD double s(int a, int I) const {
    int i, j;
    pair_of(I, i, j);
    if (i == j) return a == i ? n[i] : 0.0;
    const double r = 0.70710678118654752440;
    return a == i ? r * n[j] : a == j ? r * n[i] : 0.0;
  }
  HOM_HD double Q(int I, int J) const {
    double q = 0.0;
#pragma unroll
    for (int a = 0; a < DIM; ++a) q += s(a, I) * s(a, J);
    return q;
  }
  HOM_HD double entry(const Layered<double>& c, int I, int J) const {
    const double nn = N[I] * N[J], q = Q(I, J);
    return c.cn * nn + c.F * (N[I] * p[J] + p[I] * N[J]) + c.B * p[I] * p[J] +
           2.0 * c.mup * ((I == J ? 1.0 : 0.0) - 2.0 * q + nn) + 4.0 * c.mun * (q - nn);
  }
};

}  // namespace hom
