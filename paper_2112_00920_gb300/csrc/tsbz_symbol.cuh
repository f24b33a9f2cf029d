// The kinetic symbol of the Fourier forms: T(k) + q G(k) + q^2 / 2 summed over the axes.
//
// It enters every step as the same number, so its rounding does not average out: the
// rounding of an axis' own number, or of two axes' sum, is common to a whole line or plane
// of frequencies, and so is what the transforms' rounded twiddles do to a frequency (forward
// and back it comes out times 1 + gain, a few 1e-8 in single precision: CellDev::kgain).
// Both move the energies of whole families of plane waves, and density and current feel it
// more than noise of the same size (300 steps at 16^3 in single precision: density off by 4.4e-7
// with plain sums, 1.8e-7 so).  So an axis' number is split into a multiple of a quantum, whose
// sums over the axes are exact, and a small rest, and the gains are divided out: the sum is
// rounded once, differently at each frequency.  The field kernel forms the axes' numbers, once
// per k-point, and a step's CTA their sums, once per launch.
#pragma once
#include "tsbz_internal.h"

template <typename T> struct Symbol {
  T hi, lo, gain;
};

// Axis ax at frequency k for the vector q3, transforms' normalisation folded in.
template <typename T>
__device__ __forceinline__ Symbol<T> symbol_axis(const CellDev& c, const double* q3, int ax, int k) {
  const double q = q3[ax], s0 = c.ksym[2 * ax * c.nmax + k], s1 = c.ksym[(2 * ax + 1) * c.nmax + k];
  const double t = fma(0.5 * q, q, s0), l = fma(q, s1, t);
  const double hi = rint(l * c.kquant_inv) * c.kquant;   // (powers of two, as the scale)
  double lo = l - hi;
  if (sizeof(T) == sizeof(double)) lo += fma(0.5 * q, q, s0 - t) + fma(q, s1, t - l);   // what l was rounded by
  Symbol<T> s;
  s.hi = (T)hi * (T)c.kscale;
  s.lo = (T)lo * (T)c.kscale;
  s.gain = (T)c.kgain[ax * c.nmax + k];
  return s;
}

// Sum of two axes.
template <typename T> __device__ __forceinline__ Symbol<T> symbol_add(const Symbol<T>& a, const Symbol<T>& b) {
  Symbol<T> s;
  s.hi = a.hi + b.hi;
  s.lo = a.lo + b.lo;
  s.gain = a.gain + b.gain;
  return s;
}

template <typename T> __device__ __forceinline__ T symbol_value(const Symbol<T>& s) {
  return s.hi + fma(-s.hi, s.gain, s.lo);
}

// The unit's numbers, [3][nmax].
template <typename T> __device__ __forceinline__ const Symbol<T>* symbol_unit(const LaunchSet& L, int u) {
  return (const Symbol<T>*)L.symbols + (long long)u * L.symbol_stride;
}
