// Rules of the launches that need no CUDA (plain C++; not part of the ABI).
#pragma once

namespace rix {

// SMs of a GB300.  The rules that split work by it take this number and not the device's: some of
// them decide the order of a sum, and the same system gives the same bits wherever it runs.
constexpr int SMS = 152;

// Launch class of an output of cost top in a stage of cost total: a cluster of 2^c CTAs, 1 to
// 2^largest, where one CTA would take more than half of an even share of the stage on the SMs, so that
// it would run on alone at the end.  (Two waters, at most 8 -> 16 CTAs: terms 1+2 168 -> 107
// us, terms 3+4 27 -> 20 us.)
inline int cluster_class(double top, double total, int largest) {
  int c = 0;
  while (c < largest && 2.0 * top * SMS > total * (1 << c)) c++;
  return c;
}

// The largest class up to want whose clusters fit (fits(CTAs of the cluster)).
template <class Fits>
inline int fitting_class(int want, Fits fits) {
  while (want > 0 && !fits(1 << want)) want--;
  return want;
}

}  // namespace rix
