// Device functions that more than one stage's kernels use.
#pragma once
#include "ah_internal.h"

namespace ah {

// The amplicon with its Tm and flags from its two sites' Tm.  flags bit 0: the threshold decision (defined and
// Tm >= min_tm), bit 1: Tm within 1e-9 C of min_tm, so that the decision rests on the last digits of a double,
// bit 2: undefined.  Without the filter the list is not compacted and the bits only annotate.
__device__ __forceinline__ bool decide_amplicon(ah_amplicon* m, double ti, double tj, double min_tm) {
  const bool undefined = isnan(ti) || isnan(tj);
  const double t = undefined ? __longlong_as_double(0x7ff8000000000000ll) : fmin(ti, tj);
  const bool pass = !undefined && t >= min_tm;
  uint8_t flags = 0;
  if (pass) flags |= 1;
  if (!undefined && fabs(t - min_tm) <= 1e-9) flags |= 2;
  if (undefined) flags |= 4;
  m->tm = t;
  m->flags = flags;
  return pass;
}

}  // namespace ah
