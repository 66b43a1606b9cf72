// Host bookkeeping of split-K products that are summed from partial results.
#pragma once

namespace hotrg {

// The partials a product left behind: a refused product (a negative status) left none.  Offsets into a
// buffer of partials and the counts of a reduction advance by this, so they never go below zero.
inline int partials_written(int r) { return r > 0 ? r : 0; }

}  // namespace hotrg
