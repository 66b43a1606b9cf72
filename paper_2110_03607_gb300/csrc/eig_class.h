// Classes of eigenvectors under the exchange of hat and check: +(label + 1) even, -(label + 1) odd in the
// component of that label, 0 without one.  Signs are comparable within a component only.
#pragma once

#ifdef __CUDACC__
#define HOTRG_HD __host__ __device__ __forceinline__
#else
#define HOTRG_HD inline
#endif

namespace hotrg {

// An even and an odd vector of one component: A commutes with the exchange there, so A v_p and A v_q are
// orthogonal and what is computed otherwise is rounding.  They are not turned against each other.
HOTRG_HD bool turn_forbidden(int cls_p, bool lost_p, int cls_q, bool lost_q) {
  return cls_p != 0 && cls_p == -cls_q && !lost_p && !lost_q;
}

// Whether turning two vectors by tan t leaves both without a class: they differ in it, or one of them has
// lost its own to an earlier turn and hands on what it took in.  Angles below 2^-24 mix in what the
// couplings between two components are themselves: nothing beyond rounding.
HOTRG_HD bool turn_ends_class(int cls_p, bool lost_p, int cls_q, bool lost_q, double t) {
  return (cls_p != cls_q || lost_p || lost_q) && (t > 0.0 ? t : -t) > 5.9604644775390625e-8;
}

}  // namespace hotrg
