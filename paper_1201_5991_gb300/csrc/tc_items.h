// Work items (128 x 128 output blocks) of one tensor-core launch of the factorisation, per subdomain:
// the host counts them (prefix sums per launch), the kernel finds item t again in closed form.
//
// A launch has output columns jbeg <= j < min(Bc, jend) in pairs j, j + 1; the rows of a pair start at
// max(j, ib) (ib = 0 for an update; the first row below the diagonal block, for a panel solve) and end at
// R, or, on a level with inverse rows (internal.h), at R + e: the first e inverse rows are those that the
// panel's columns (all below kend) have reached.  An update of every trailing column has a second
// segment there: the columns R .. R + e - 1 of the inverse block, rows from j.  The pairs of a segment have
// one row pair less each, so item t's column pair solves a quadratic (a loop over the pairs cost up to 126
// iterations per item at 16,384 columns, in the thread that requests the operand copies: 1.1 us per item,
// a tenth of the kernel).
#pragma once

#include "internal.h"

namespace bddc {

// inverse rows reached by panel columns below kend
__host__ __device__ inline int inverse_rows(const SubMeta& m, int kend) {
  const int e = kend - m.nIb;
  return e <= 0 ? 0 : (e < m.nV ? e : m.nV);
}

struct TcItems {
  int j0, n, a, step;   // n column pairs from j0; pair c has a - step c row pairs
  int R, n2;            // second segment: n2 column pairs from R; pair c has n2 - c row pairs
  int ib, rend, jlim;   // rows from max(j, ib) to rend; columns of the first segment below jlim
};

// act: first panel column of the launch; a subdomain with Bc <= act takes no part
__host__ __device__ inline TcItems tc_items_of(const SubMeta& m, int jbeg, int jend, int ibeg, int panel, int act) {
  TcItems t;
  const bool on = act < m.Bc;
  const int e = on ? inverse_rows(m, panel ? jend : jbeg) : 0;
  t.jlim = m.Bc < jend ? m.Bc : jend;
  t.ib = ibeg < m.Bc ? ibeg : m.Bc;
  t.R = m.R;
  // constraints touch interface DOFs only: their rows are zero until the first interface column
  t.rend = (panel ? jend : jbeg) <= m.nIb ? m.Bc : m.R + e;
  t.j0 = jbeg;
  t.n = on && t.jlim > jbeg ? (t.jlim - jbeg + 1) / 2 : 0;
  const int first = panel ? t.ib : jbeg;
  t.a = (t.rend - first + 1) / 2;
  if (t.a < 0) t.a = 0;
  t.step = panel ? 0 : 1;
  t.n2 = panel || jend < (1 << 30) ? 0 : (e + 1) / 2;
  return t;
}

__host__ __device__ inline int64_t tc_items_count(const TcItems& t) {
  return (int64_t)t.n * t.a - (t.step ? (int64_t)t.n * (t.n - 1) / 2 : 0) + (int64_t)t.n2 * (t.n2 + 1) / 2;
}

// largest c < n with c a - c (c - 1) / 2 <= q; q becomes the rest
__device__ __forceinline__ int tc_column_pair(int a, int n, int& q) {
  const float b = (float)a + 0.5f;
  int c = (int)(b - sqrtf(fmaxf(b * b - 2.f * (float)q, 0.f)));
  c = c < 0 ? 0 : (c >= n ? n - 1 : c);
  while (c > 0 && c * a - c * (c - 1) / 2 > q) --c;                      // rounding of the root
  while (c + 1 < n && (c + 1) * a - (c + 1) * c / 2 <= q) ++c;
  q -= c * a - c * (c - 1) / 2;
  return c;
}

// item q (0 <= q < tc_items_count) -> first column j, first row i0 of its block and its columns' end
__device__ __forceinline__ void tc_item(const TcItems& t, int q, int& j, int& i0, int& jl) {
  const int first = t.n * t.a - (t.step ? t.n * (t.n - 1) / 2 : 0);
  if (q >= first) {
    q -= first;
    j = t.R + 2 * tc_column_pair(t.n2, t.n2, q);
    i0 = j + 2 * q;
    jl = t.rend;
    return;
  }
  int c;
  if (t.step) {
    c = tc_column_pair(t.a, t.n, q);
  } else {
    c = q / t.a;
    q -= c * t.a;
  }
  j = t.j0 + 2 * c;
  i0 = (j > t.ib ? j : t.ib) + 2 * q;
  jl = t.jlim;
}

}  // namespace bddc
