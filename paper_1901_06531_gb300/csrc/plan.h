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

// Plan of a transform of length n = 2^a 3^b (1 < n <= 256) with a twiddle table
// of length ntab (a multiple of n): stages of radix 4, then 2, then 3, two to
// a pass; of an odd number of stages the first or the last is a pass of its
// own, whichever leaves the smaller largest pass.
inline bool mf_make_plan(int n, int ntab, bool pairs, AxisPlan* p) {
  p->n = n;
  p->ntab = ntab;
  p->nst = 0;
  int m = n;
  while (m % 4 == 0) { p->rad[p->nst++] = 4; m /= 4; }
  if (m % 2 == 0) { p->rad[p->nst++] = 2; m /= 2; }
  while (m % 3 == 0) { p->rad[p->nst++] = 3; m /= 3; }
  if (m != 1 || p->nst == 0) return false;
  auto largest = [&](int start) {   // largest pass with pairs from stage `start` on
    int big = 0;
    for (int s = start; s < p->nst; s += 2) {
      const int r = p->rad[s] * (s + 1 < p->nst ? p->rad[s + 1] : 1);
      big = r > big ? r : big;
    }
    return big;
  };
  const int start = (p->nst % 2 && largest(1) < largest(0)) ? 1 : 0;
  p->npass = 0;
  int L = n;
  for (int s = 0; s < p->nst;) {
    if (p->npass >= MF_MAX_PASSES) return false;
    AxisPass& g = p->pass[p->npass++];
    g.r1 = p->rad[s];
    g.r2 = (pairs && s >= start && s + 1 < p->nst) ? p->rad[s + 1] : 1;
    g.tstep1 = ntab / L;
    g.tstep2 = ntab / (L / g.r1);
    s += g.r2 > 1 ? 2 : 1;
    L /= g.r1 * g.r2;
    g.dm = fast_div(L);
    g.nb = fast_div(n / (g.r1 * g.r2));
  }
  return true;
}

// Position of frequency k after the stages of plan p.
inline int mf_plan_pos(const AxisPlan& p, int k) {
  int pos = 0, L = p.n;
  for (int s = 0; s < p.nst; ++s) {
    const int r = p.rad[s], m = L / r;
    pos += m * (k % r);
    k /= r;
    L = m;
  }
  return pos;
}

// Index maps of the any-size spectrum layout from the plans of nx, ny / 2 and
// nz: slot of each x-frequency (nx), x-frequency and parity of each slot (nx
// each), half y-frequency of each row (ny / 2), z-frequency of each position.
inline void mf_any_size_maps(const AxisPlan& px, const AxisPlan& py, const AxisPlan& pz, int* xpos, int* xk, int* xe,
                             int* yk, int* zk) {
  const int nx = px.n;
  for (int k = 0; k < nx; ++k) xpos[k] = mf_plan_pos(px, k);
  for (int k = 0; k < nx; ++k) {
    const int s = xpos[k];
    if (k < nx / 2) { xk[s] = k; xe[s] = 0; }
    else if (k == nx / 2) { xk[s] = 0; xe[s] = 1; }
    else { xk[s] = nx - k; xe[s] = 1; }
  }
  for (int k = 0; k < py.n; ++k) yk[mf_plan_pos(py, k)] = k;
  for (int k = 0; k < pz.n; ++k) zk[mf_plan_pos(pz, k)] = k;
}
