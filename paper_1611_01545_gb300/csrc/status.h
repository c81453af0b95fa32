// Status bits that kernels set, and the error that a call returns for them.
#pragma once

#include "pm.h"

namespace pm {

enum StatusBits : int { ST_CORRUPT = 1, ST_OVERFLOW = 2, ST_RANGE = 4, ST_TIMEOUT = 8 };

// The first of several causes: a bad position or a full list can make the codes
// look corrupt, and so can a wait that ran out.
inline int status_error(int bits) {
  if (bits & ST_RANGE) return PM_ERR_RANGE;
  if (bits & ST_OVERFLOW) return PM_ERR_OVERFLOW;
  if (bits & ST_CORRUPT) return PM_ERR_CORRUPT;
  if (bits & ST_TIMEOUT) return PM_ERR_TIMEOUT;
  return PM_OK;
}

}  // namespace pm
