// route.h -- which solver a call takes, by its sizes, its density and its
// number of configurations.  Host code without CUDA (tests/route_check.cpp).
//
// The wavefront solver (wave.cu) pays for each reached site and for each
// level; the resident solver (resident.cu) updates every site of the causal
// window at every step, in one CTA's shared memory, at a fraction of the price
// a site.  So short, thin or dense lattices are the resident solver's, all the
// more the fewer configurations there are (then a level's latency counts).
#pragma once

#include <algorithm>
#include <cmath>

namespace pc {

// Density of metallic sites from which the resident solver is the faster one
// for n configurations with masses (A columns, L layers, nsm SMs).  The line
// is the one that separates 2,900 measured pairs best (W = 0 to 25, p = 0.15 to
// 0.95, 1 to 10,000 configurations; us per call, wavefront / resident): W = 14,
// L = 14, one configuration, p = 0.95 145 / 70, p = 0.5 97 / 81, p = 0.25 121 /
// 125; W = 8, L = 8, 10,000 of them, p = 0.95 917 / 539, p = 0.5 650 / 600, p =
// 0.25 405 / 720; W = 8, L = 48, 10,000 of them, p = 0.95 5,750 / 10,470.
// (Verdicts alone: the wavefront solver is at most a launch slower.)  A thin
// fibre far longer than it is wide is one long chain of small levels: W = 5, L =
// 100, p = 0.95, 600 configurations 388 / 1,298; W = 0, L = 64, 64 of them 139 /
// 220.
inline double resident_from(int W, int A, int L, long long n, int nsm) {
  if (L > 16 * W + 12 && (W == 0 || n > nsm)) return 1e9;  // at no density
  const double q = std::min(std::max((double)n / nsm, 1.0), 60.0);
  return 0.0053 * std::pow((double)L, 0.7) * std::pow((double)A, 0.32) * std::pow(q, 0.4);
}

// CTA size of the resident solver for n configurations of a lattice whose
// state takes smem bytes (sm_smem: of an SM's).  An SM holds 640 threads of it.
// Enough CTAs an SM for its share of the configurations in equal rounds, with
// the threads divided among them; no more threads than a configuration uses (a
// thread per column keeps the column's contacts in registers), and no fewer
// than an eighth of the sites of the first four layers.  Against
// the best of ten sizes, over 907 calls of more than 55 us: within 5 % in 808,
// 1 % faster on average than the best of the five sizes that a first call
// could time.
inline int resident_cta(int A, int L, long long n, int nsm, size_t smem, size_t sm_smem) {
  auto up = [](long long x) { return (int)std::max(64ll, (x + 63) / 64 * 64); };
  const long long sites = (long long)A * L;  // below 2^31
  const int need = std::max(std::min(384, up(std::min(sites, 4096ll) / 4)), std::min(640, up(A)));
  const int least = std::min({need, 320, std::max(up((long long)A * std::min(L, 4) / 8),
                                                  std::min(128, up(std::min(std::max(sites, 3ll * A), 4096ll) / 16)))});
  const long long share = std::max(1ll, (n + nsm - 1) / nsm);
  const long long fit = std::max<long long>(1, std::min<long long>((long long)(sm_smem / (smem + 1024)), 682 / least));
  const long long rounds = (share + fit - 1) / fit, ctas = std::max(1ll, (share + rounds - 1) / rounds);
  return std::min(need, std::max(least, (int)(640 / ctas) / 64 * 64));
}

// Roughly the density at which a W x L fibre begins to percolate (the scaling
// form of the effective threshold, Eq. (9)).
inline double fibre_threshold(int W, int L) {
  const double w = std::max(W, 1), l = std::max(L, 1), s = std::pow(l, -1.136);
  return 0.156 + 0.58 * std::pow(w / l, -1.22) * s - 0.39 * s;
}

// Density below which hardly one of n configurations is expected to
// percolate: with verdicts asked for first, their masses are then better left
// to a pass of their own than computed for all.  Long fibres only, and the
// farther below the threshold the more configurations there are and the
// softer the transition is (1,854 calls measured both ways; us in one pass and
// in two: W = 8, L = 48, 100 configurations, p = 0.18 206 / 94, p = 0.2 245 /
// 358; W = 4, L = 48, p = 0.21, 800 of them 161 / 94).
inline double few_percolate_below(int W, int L, long long n) {
  return L >= 20 ? fibre_threshold(W, L) - 0.1 * std::pow((double)n, 0.3) / std::sqrt((double)L * std::max(W, 1)) : 0.0;
}

}  // namespace pc
