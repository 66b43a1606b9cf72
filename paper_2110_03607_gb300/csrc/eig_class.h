// Classes of eigenvectors under the exchange of hat and check: +(label + 1) even, -(label + 1) odd in the
// component of that label, 0 without one.  Signs are comparable within a component only.
#pragma once

#ifdef __CUDACC__
#define HOTRG_HD __host__ __device__ __forceinline__
#else
#define HOTRG_HD inline
#endif

namespace hotrg {

// Whether turning two vectors against each other leaves both without a class: they differ in it, or one
// of them has lost its own to an earlier turn (and hands on what it took in).  Symmetric, and once true
// for a vector it stays so, whatever the order of the turns.
HOTRG_HD bool turn_ends_class(int cls_p, bool lost_p, int cls_q, bool lost_q) {
  return cls_p != cls_q || lost_p || lost_q;
}

}  // namespace hotrg
