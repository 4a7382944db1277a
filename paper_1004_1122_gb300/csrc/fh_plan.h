// fh_plan.h -- host-side planning: FFT radix schedules, pass tilings and
// float64 twiddle tables.  Pure host code (no CUDA calls).
#pragma once

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <map>
#include <string>
#include <tuple>
#include <vector>

#include "fh_fft.cuh"

namespace fh {

// Radices compiled into the stage dispatchers (must match FH_FOR_EACH_RADIX
// and FH_FOR_EACH_RADIX_X).  The extended radices (powers of 2 up to 16, and
// the primes 11, 13 and 17) are used only by lengths that have one of 2, 11,
// 13, 17 as a factor; those plans run the DynPlanX kernels with the register
// budget RegBudgetX.
inline const std::vector<int>& compiled_radices() {
  static const std::vector<int> r = {27, 25, 17, 16, 15, 13, 11, 9, 8, 7, 5, 4, 3, 2};
  return r;
}

inline int reg_budget(bool fp64) { return fp64 ? RegBudget<double>::value : RegBudget<float>::value; }
inline int reg_budget_x(bool fp64) { return fp64 ? RegBudgetX<double>::value : RegBudgetX<float>::value; }

// Does n factor into the supported primes 2, 3, 5, 7, 11, 13, 17?  ext is
// set when one of 2, 11, 13, 17 divides n (the extended radix set).
inline bool factorable(int n, bool& ext) {
  ext = false;
  if (n < 1) return false;
  for (int p : {2, 3, 5, 7, 11, 13, 17}) {
    while (n % p == 0) {
      n /= p;
      if (p == 2 || p > 7) ext = true;
    }
  }
  return n == 1;
}

// Radices of a plan whose sequences are worked on by tpl threads each: a stage
// of radix R is allowed iff every thread holds at most floor(budget / R)
// butterflies, i.e. ceil(n / R / tpl) * R <= budget.
inline std::vector<int> allowed_radices(int n, int tpl, int budget) {
  std::vector<int> allowed;
  for (int R : compiled_radices()) {
    if (n % R) continue;
    const int bmax = budget / R;
    if (bmax < 1) continue;
    const int need = (n / R + tpl - 1) / tpl;
    if (need > bmax) continue;
    allowed.push_back(R);
  }
  return allowed;
}

// Minimum-stage radix schedule for length n from these radices (empty if
// impossible), largest radix first.  Dynamic programme over the divisors m of
// n: best[m] is a shortest list of allowed radices whose product is m.
inline std::vector<int> plan_radices(int n, const std::vector<int>& allowed) {
  std::vector<int> divs;
  for (int m = 1; m <= n; ++m)
    if (n % m == 0) divs.push_back(m);  // ascending
  std::map<int, std::vector<int>> best;
  best[1] = {};
  for (int m : divs) {
    if (m == 1) continue;
    bool found = false;
    std::vector<int> cand;
    for (int R : allowed) {
      if (m % R) continue;
      auto it = best.find(m / R);
      if (it == best.end()) continue;
      if (!found || it->second.size() + 1 < cand.size()) {
        cand = it->second;
        cand.push_back(R);
        found = true;
      }
    }
    if (found) best[m] = cand;
  }
  auto it = best.find(n);
  if (it == best.end()) return {};
  std::vector<int> r = it->second;
  std::sort(r.begin(), r.end(), [](int u, int v) { return u > v; });
  return r;
}

// Choose (tpl, radices): fewest stages first, then the fewest threads per
// sequence (more butterflies per thread, more independent work in flight).
// Even lengths and lengths with a prime factor 11, 13 or 17 get an extended
// plan (pl.ext = 1).
// small: a plan over the small radix set (lengths that need no extended one).
inline bool make_fft_plan(int n, bool fp64, int max_tpl, FFTPlan& pl, int& tpl,
                          int force_tpl = 0, bool small = false) {
  bool ext;
  if (!factorable(n, ext)) return false;
  small = small && !ext;
  const int budget = small ? kSmallBudget : ext ? reg_budget_x(fp64) : reg_budget(fp64);
  int best_stages = 1 << 30, best_tpl = 0;
  std::vector<int> best_r, last;
  for (int t = 1; t <= max_tpl; ++t) {
    if (force_tpl && t != force_tpl) continue;
    // the same radices as for fewer threads: the same plan (trying all 1024
    // thread counts took 3 ms for n = 2187)
    std::vector<int> allowed = allowed_radices(n, t, budget);
    if (allowed == last) continue;
    last.swap(allowed);
    const std::vector<int> r = plan_radices(n, last);
    if (r.empty()) continue;
    if ((int)r.size() < best_stages) {
      best_stages = (int)r.size();
      best_tpl = t;
      best_r = r;
    }
  }
  if (best_r.empty() || (int)best_r.size() > kMaxStages) return false;
  pl.n = n;
  pl.nstages = (int)best_r.size();
  for (int s = 0; s < kMaxStages; ++s) pl.radix[s] = s < pl.nstages ? best_r[s] : 0;
  pl.ext = ext ? kRadixExt : small ? kRadixSmall : kRadixStd;
  tpl = best_tpl;
  return true;
}

// Spread plan (kRadixSpread) of length n: every stage gives each thread at most
// one butterfly of radix 2 to 7 or one output pair of a radix-11, 13 or 17
// butterfly; the split radices come first.  False where the last stage would
// be a split one.
inline bool make_spread_plan(int n, FFTPlan& pl, int& tpl) {
  std::vector<int> r;
  int m = n;
  for (int R : {17, 13, 11, 7, 5, 4, 3, 2})
    while (m % R == 0) {
      r.push_back(R);
      m /= R;
    }
  if (m != 1 || r.empty() || (int)r.size() > kMaxStages || r.back() > kMaxWholeW) return false;
  pl.n = n;
  pl.nstages = (int)r.size();
  tpl = 1;
  for (int s = 0; s < kMaxStages; ++s) {
    pl.radix[s] = s < pl.nstages ? r[s] : 0;
    if (s < pl.nstages) tpl = std::max(tpl, spread_items(n, r[s]));
  }
  pl.ext = kRadixSpread;
  return true;
}

// exp(-2 pi i m / n) for m in [0, n), float64.  The angle is reduced exactly
// on the rational m / n (octant symmetry) before calling the C library, so
// every entry is within an ulp or two of the true value.
inline void twiddles(int n, std::vector<double>& re, std::vector<double>& im) {
  re.resize(n);
  im.resize(n);
  for (int m = 0; m < n; ++m) {
    ct::cs v;
    // reuse the exact rational reduction, then evaluate with std::cos/sin
    long long num = 8LL * m, den = n;
    double sgn_s = 1.0, sgn_c = 1.0;
    bool swap = false;
    if (2 * num >= 8 * den) { num = 8 * den - num; sgn_s = -1.0; }
    if (2 * num > 4 * den) { num = 4 * den - num; sgn_c = -1.0; }
    if (num > den) { num = 2 * den - num; swap = true; }
    const double x = (ct::kPi / 4.0) * (double)num / (double)den;
    v.c = std::cos(x);
    v.s = std::sin(x);
    if (swap) std::swap(v.c, v.s);
    re[m] = sgn_c * v.c;
    im[m] = -(sgn_s * v.s);  // forward sign
  }
}

// Entries of a plan's twiddle table: its stages in order, then those of the
// reversed radix order.
inline int stage_twiddle_count(const FFTPlan& pl) {
  return 2 * pl.n - pl.radix[0] - pl.radix[pl.nstages - 1];
}
// The table (fh_fft.cuh), from the n-th roots of unity.
inline void stage_twiddles(const FFTPlan& pl, std::vector<double>& re, std::vector<double>& im) {
  std::vector<double> wr, wi;
  twiddles(pl.n, wr, wi);
  re.clear();
  im.clear();
  for (int rev = 0; rev < 2; ++rev) {
    int Ns = 1;
    for (int s = 0; s < pl.nstages; ++s) {
      const int R = pl.radix[rev ? pl.nstages - 1 - s : s];
      if (s > 0)
        for (int r = 1; r < R; ++r)
          for (int k = 0; k < Ns; ++k) {
            const int m = (int)((long long)r * k * (pl.n / (Ns * R)) % pl.n);
            re.push_back(wr[m]);
            im.push_back(wi[m]);
          }
      Ns *= R;
    }
  }
}

// Stage order of plans whose transform is followed by its mirror image: the
// smallest radix in the middle.  After a first stage of radix 3 (the mirror
// image of 27, 27, 3) the writes of the next stage collide in shared-memory
// banks; with 27, 3, 27 every stage's writes run along consecutive words.
inline void mirror_order(FFTPlan& pl) {
  if (pl.nstages < 3) return;
  for (int s = pl.nstages - 1; s > 1; --s) std::swap(pl.radix[s], pl.radix[s - 1]);
}

// Shared-memory bank cost of 8-byte accesses: lanes t of a warp access element
// addr(t) (negative: none); 16 banks of 8 bytes, one half warp at a time.
template <typename F> inline int bank_cost(int threads, F&& addr) {
  int total = 0;
  for (int h0 = 0; h0 < threads; h0 += 16) {
    long long seen[16][16];
    int cnt[16] = {};
    int worst = 0;
    for (int t = h0; t < h0 + 16 && t < threads; ++t) {
      const long long a = addr(t);
      if (a < 0) continue;
      const int b = (int)(a % 16);
      bool dup = false;
      for (int k = 0; k < cnt[b]; ++k) dup = dup || seen[b][k] == a;
      if (!dup) seen[b][cnt[b]++] = a;
      worst = std::max(worst, cnt[b]);
    }
    total += worst;
  }
  return total;
}

// Distance between sequences in shared memory (n .. n + 15 elements) with the
// fewest bank conflicts of the plan's stages over nseq sequences of thr
// threads, plus `weight` times the cost of io(stride).
template <typename F>
inline int seq_stride(const FFTPlan& pl, int thr, int nseq, int weight, F&& io) {
  const int threads = std::min(nseq * thr, 96);  // the pattern repeats
  int best = pl.n, best_cost = 1 << 30;
  for (int ss = pl.n; ss < pl.n + 16; ++ss) {
    int cost = weight * io(ss);
    int Ns = 1;
    for (int s = 0; s < pl.nstages; ++s) {
      const int R = pl.radix[s], nb = pl.n / R;
      cost += R * bank_cost(threads, [&](int t) -> long long {
        const int q = t / thr, j = t - q * thr;
        return j < nb ? (long long)q * ss + j : -1;
      });
      cost += R * bank_cost(threads, [&](int t) -> long long {
        const int q = t / thr, j = t - q * thr;
        return j < nb ? (long long)q * ss + (j / Ns) * R * Ns + j % Ns : -1;
      });
      Ns *= R;
    }
    if (cost < best_cost) {
      best_cost = cost;
      best = ss;
    }
  }
  return best;
}

}  // namespace fh
