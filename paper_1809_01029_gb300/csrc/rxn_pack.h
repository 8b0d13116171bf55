// Host-side packing of a reaction's sides: their shapes and the short path's
// head (RxnHead).
#pragma once

#include <algorithm>

#include "pj_internal.h"

namespace pj {

// SH_* of a side of n species with coefficients nu in descending order.
inline int32_t side_shape(const int32_t* nu, int n) {
  if (n == 1 && nu[0] == 1) return SH_1;
  if (n == 1 && nu[0] == 2) return SH_2;
  if (n == 2 && nu[0] == 1 && nu[1] == 1) return SH_11;
  if (n == 2 && nu[0] == 2 && nu[1] == 1) return SH_21;
  if (n == 3 && nu[0] == 1 && nu[1] == 1 && nu[2] == 1) return SH_111;
  return SH_GEN;
}

// The factors of each side (a coefficient of 2 as two factors), the jump
// table's code and whether the reaction may take the short path; r holds the
// reaction's sides, shapes, kind and rev.  plain: none of the special types
// and constants within the fixed point.
//
// The short path's jump table (lean_shapes) has the shapes SH_1 .. SH_111
// only, and code has room for no other: a side of shape SH_GEN takes the
// general path also where it has three factors (3A).  The products of an
// irreversible reaction enter no rate, so their shape does not matter, only
// that they are three factors at most.
inline void pack_head(Rxn& r, bool plain) {
  RxnHead& hd = r.head;
  hd.kind = (uint8_t)r.kind;
  hd.rev = (uint8_t)r.rev;
  hd.lean = plain ? 1 : 0;
  hd.code = 0;
  for (int side = 0; side < 2; side++) {
    int32_t* out = side ? hd.b : hd.f;
    // in the order side_rate multiplies them: 2A + B as A B A, else last to first
    const int32_t* sp = &r.sp[side * PJ_MAX_SP];
    int cnt = 0;
    if (r.shape[side] == SH_21) {
      out[0] = out[2] = 32 * sp[0];
      out[1] = 32 * sp[1];
      cnt = 3;
    } else {
      for (int a = (side ? r.nprod : r.nreac) - 1; a >= 0; a--)
        for (int u = 0; u < r.nu[side * PJ_MAX_SP + a]; u++, cnt++)
          if (cnt < 3) out[cnt] = 32 * sp[a];
    }
    if (cnt < 1 || cnt > 3) hd.lean = 0;
    if ((side == 0 || r.rev) && r.shape[side] > SH_111) hd.lean = 0;
    for (int u = cnt; u >= 1 && u < 3; u++) out[u] = out[0];
    (side ? hd.nb : hd.nf) = (uint8_t)std::min(cnt, 3);
  }
  if (hd.lean) hd.code = (uint8_t)(6 * r.shape[0] + (r.rev ? 1 + r.shape[1] : 0));
}

}  // namespace pj
