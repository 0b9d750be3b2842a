// Work items (128 x 128 output blocks) of one tensor-core launch of the factorisation, per subdomain:
// the host counts them (prefix sums per launch), the kernel finds item t again in closed form.
//
// A launch has output columns jbeg <= j < min(Bc, jend) in pairs j, j + 1; the rows of a pair start at
// max(j, ib) (ib = 0 for an update; the first row below the diagonal block, for a panel solve) and end
// at R.  An update's pairs have one row pair less each, so item t's column pair solves a quadratic
// (a loop over the pairs cost up to 126 iterations per item at 16,384 columns, in the thread that
// requests the operand copies: 1.1 us per item, a tenth of the kernel).
#pragma once

#include "internal.h"

namespace bddc {

struct TcItems {
  int j0, n, a, step;   // n column pairs from j0; pair c has a - step c row pairs
  int ib, rend, jlim;   // rows from max(j, ib) to rend; columns below jlim
};

__host__ __device__ inline TcItems tc_items_of(const SubMeta& m, int jbeg, int jend, int ibeg, int panel) {
  TcItems t;
  t.jlim = m.Bc < jend ? m.Bc : jend;
  t.ib = ibeg < m.Bc ? ibeg : m.Bc;
  t.rend = m.R;
  t.j0 = jbeg;
  t.n = t.jlim > jbeg ? (t.jlim - jbeg + 1) / 2 : 0;
  const int first = panel ? t.ib : jbeg;
  t.a = (t.rend - first + 1) / 2;
  if (t.a < 0) t.a = 0;
  t.step = panel ? 0 : 1;
  return t;
}

__host__ __device__ inline int64_t tc_items_count(const TcItems& t) {
  return (int64_t)t.n * t.a - (t.step ? (int64_t)t.n * (t.n - 1) / 2 : 0);
}

// item q (0 <= q < tc_items_count) -> first column j and first row i0 of its block
__device__ __forceinline__ void tc_item(const TcItems& t, int q, int& j, int& i0) {
  int c;
  if (t.step) {
    const float b = (float)t.a + 0.5f;
    c = (int)(b - sqrtf(fmaxf(b * b - 2.f * (float)q, 0.f)));
    c = c < 0 ? 0 : (c >= t.n ? t.n - 1 : c);
    while (c > 0 && c * t.a - c * (c - 1) / 2 > q) --c;                      // rounding of the root
    while (c + 1 < t.n && (c + 1) * t.a - (c + 1) * c / 2 <= q) ++c;
    q -= c * t.a - c * (c - 1) / 2;
  } else {
    c = q / t.a;
    q -= c * t.a;
  }
  j = t.j0 + 2 * c;
  i0 = (j > t.ib ? j : t.ib) + 2 * q;
}

}  // namespace bddc
