// Host side of the any-size transforms (transformg.cuh): stage plans of an
// axis and the digit-reversed positions they leave the frequencies in.
#pragma once

#include "common.cuh"

// Sizes the transforms take: 2^a 3^b.
inline bool mf_smooth_size(int n) {
  if (n < 1) return false;
  while (n % 2 == 0) n /= 2;
  while (n % 3 == 0) n /= 3;
  return n == 1;
}

// Plan of a transform of length n = 2^a 3^b (1 < n <= 256) with a twiddle
// table of length ntab (a multiple of n): the fewest stages, of these the
// one with the smallest largest radix, radices in falling order.
inline bool mf_make_plan(int n, int ntab, AxisPlan* p) {
  static const int radices[] = {16, 12, 9, 8, 6, 4, 3, 2};
  int best[MF_MAX_STAGES] = {0}, nst = 0;
  auto consider = [&](const int* r, int k) {
    if (nst == 0 || k < nst || (k == nst && r[0] < best[0])) {
      nst = k;
      for (int i = 0; i < k; ++i) best[i] = r[i];
    }
  };
  for (int a : radices) {
    if (a == n) { const int r[] = {a}; consider(r, 1); }
    if (n % a) continue;
    for (int b : radices) {
      if (b > a || (n / a) % b) continue;
      if (a * b == n) { const int r[] = {a, b}; consider(r, 2); }
      for (int c : radices)
        if (c <= b && a * b * c == n) { const int r[] = {a, b, c}; consider(r, 3); }
    }
  }
  if (nst == 0) return false;
  p->n = n;
  p->nst = nst;
  p->ntab = ntab;
  int L = n;
  for (int s = 0; s < MF_MAX_STAGES; ++s) {
    const int r = s < nst ? best[s] : 1;
    p->rad[s] = r;
    p->m[s] = L / r;
    p->tstep[s] = ntab / L;
    p->dm[s] = fast_div(L / r);
    p->nb[s] = fast_div(n / r);
    if (s < nst) L /= r;
  }
  return true;
}

// Position of frequency k after the stages of plan p.
inline int mf_plan_pos(const AxisPlan& p, int k) {
  int pos = 0;
  for (int s = 0; s < p.nst; ++s) {
    pos += p.m[s] * (k % p.rad[s]);
    k /= p.rad[s];
  }
  return pos;
}
