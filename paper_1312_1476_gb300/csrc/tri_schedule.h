// tri_schedule.h -- host side of the triangular solves with an incomplete-Cholesky
// factor (sparse.cu): levels, and the schedule of merged levels that the kernels run.
// Plain C++.
#pragma once

#include <algorithm>
#include <cmath>
#include <cstddef>
#include <utility>
#include <vector>

namespace gmrf {

constexpr int kTriThreads = 256;  // of the block that runs a schedule

// Level of every row: forward (row i after the rows k < i it reads) or
// backward (row i after the rows k > i it reads); rows grouped by level.
inline void levels(int n, const std::vector<int>& ptr, const std::vector<int>& col, bool forward,
                   std::vector<int>& rows, std::vector<int>& lptr) {
  std::vector<int> lev((size_t)n, 0);
  int nlev = 0;
  for (int t = 0; t < n; ++t) {
    const int i = forward ? t : n - 1 - t;
    int l = 0;
    for (int e = ptr[(size_t)i]; e < ptr[(size_t)i + 1]; ++e) l = std::max(l, lev[(size_t)col[(size_t)e]] + 1);
    lev[(size_t)i] = l;
    nlev = std::max(nlev, l + 1);
  }
  lptr.assign((size_t)nlev + 1, 0);
  for (int i = 0; i < n; ++i) ++lptr[(size_t)lev[(size_t)i] + 1];
  for (int l = 0; l < nlev; ++l) lptr[(size_t)l + 1] += lptr[(size_t)l];
  rows.assign((size_t)n, 0);
  std::vector<int> fill(lptr.begin(), lptr.end() - 1);
  for (int i = 0; i < n; ++i) rows[(size_t)fill[(size_t)lev[(size_t)i]]++] = i;
}

// The schedule of one substitution.  Consecutive levels are merged into one:
// with the rows B of the merged levels and the rows P before them,
//   x_B = F_BB^{-1} b_B - F_BB^{-1} F_BP x_P,
// so every row of B is a dot product over right-hand sides of B and results of
// P, at the price of the fill that the small inverse brings.  A level costs a
// chain of dependent operations and a barrier whatever it holds (about
// kLevelCycles), an entry its share of the FP64 lanes and of the loads (kEntryCycles),
// so the next level is merged while the entries it adds cost less than that.
// Merged rows stay below kMergedRow entries.
// kEntryCycles and the six entries per lane are the best of a sweep on the
// Figure 3 matrix, 256 samples, drop tolerance 1e-3 / 1e-5 / 1e-2 (FP64): 4.2 /
// 6.4 / 12.5 ms a call at 3 cycles, 6.4 / 6.4 / 14.4 at 1.5, 7.9 / 7.3 / 19.4 at 14;
// 10.7 / 29.1 / 26.3 ms level by level.  The factor with 1e-3 goes from 204 to 41
// levels and from 13.4k to 28.1k entries.
//
// Accuracy.  A row's rounding error is at most (its length) u sum |c_t s_t| over its
// coefficients c and sources s.  Two rules keep that where substitution has it:
// - the coefficients are formed with twice the digits (Wide) and rounded once; formed in
//   FP64 their own errors, propagated through F_BB, are larger than those of the solve;
// - a merge ends where sum |c_t| |s_t| would exceed kGrowth times what the row's own
//   substitution adds up, for x_k of the size omega_k and b = F x: omega = 1 going forward,
//   1 / F_kk going backward, so that scaling Q to S Q S changes nothing.  Without the
//   rule a factor far from diagonally dominant loses as many digits as F_BB^{-1} grows.
// Figure 3 factors of 16^2 to 40^2, drop tolerances 1e-2 to 1e-5, error of a solve over that of
// plain substitution, both against 113 bits: random right-hand sides 0.39 to 0.96 in
// FP64 and 0.25 to 0.89 in FP32 (without the two rules FP64 0.73 to 1.29), b = F x with random
// x 0.90 to 1.32 (FP64 1.31 to 3.95); all of F^{-1} Q F^{-T} v 0.94 to 1.30, median 1.06 (0.99 to
// 1.27, median 1.12).  The growth rule costs those factors at most three levels (9 -> 12; 39 ->
// 41 at 30^2 and 1e-3) and saves up to 11 % of the entries.  256 samples, with and without the
// rules: 3.81 and 3.80 ms at 1e-3, 5.63 and 5.81 at 1e-5, 11.3 at 1e-2; creating the problem 1.53 and
// 1.52 ms, 6.0 and 5.1, 0.93 and 1.04.
struct TriHost {
  std::vector<int> rec, row, col;
  std::vector<double> val;
};
constexpr double kLevelCycles = 500.0;
constexpr double kEntryCycles = 3.0;
constexpr int kMergedRow = 128;
constexpr double kGrowth = 10.0;

// hi + lo: about 105 bits.  Every product through fma, so that no compiler contracts it
// with an addition.
struct Wide {
  double hi, lo;
};
// sum += a b (a compensated dot product: the errors of products and sums collect in lo)
inline void wide_add(Wide& sum, Wide a, double b) {
  const double p = std::fma(a.hi, b, 0.0), e = std::fma(a.lo, b, std::fma(a.hi, b, -p));
  const double s = sum.hi + p, t = s - sum.hi;  // two-sum (Knuth)
  sum.lo += ((sum.hi - (s - t)) + (p - t)) + e;
  sum.hi = s;
}
// a / d with hi the nearest double; dinv = 1 / d rounded
inline Wide wide_div(Wide a, double d, double dinv) {
  const double q = std::fma(a.hi, dinv, 0.0), r = std::fma(std::fma(-q, d, a.hi) + a.lo, dinv, 0.0);
  const double hi = q + r;
  return {hi, r - (hi - q)};
}

// rows in level order (lptr); ptr/col/val the off-diagonal entries of each row;
// b and x the positions of the right-hand side and of the result in the shared arrays
inline void tri_schedule(int n, const std::vector<int>& rows, const std::vector<int>& lptr,
                         const std::vector<int>& ptr, const std::vector<int>& col, const std::vector<double>& val,
                         const std::vector<double>& dg, bool forward, int b0, int x0, TriHost& out) {
  const int nlev = (int)lptr.size() - 1;
  typedef std::vector<std::pair<int, Wide>> Expr;  // (position, coefficient)
  std::vector<Expr> expr((size_t)n);  // of the rows of the merged level being built
  std::vector<int> in_block((size_t)n, -1);
  std::vector<Wide> acc((size_t)std::max(b0, x0) + n, Wide{0.0, 0.0});
  std::vector<int> stamp(acc.size(), -1), used;
  int block = 0, mark = 0;
  auto row_expr = [&](int i, Expr& e) {
    ++mark;
    used.clear();
    auto add = [&](int at, Wide a, double w) {
      if (stamp[(size_t)at] != mark) {
        stamp[(size_t)at] = mark;
        acc[(size_t)at] = Wide{0.0, 0.0};
        used.push_back(at);
      }
      wide_add(acc[(size_t)at], a, w);
    };
    const Wide one{1.0, 0.0};
    add(b0 + i, one, 1.0);
    for (int q = ptr[(size_t)i]; q < ptr[(size_t)i + 1]; ++q) {
      const int k = col[(size_t)q];
      if (in_block[(size_t)k] == block)
        for (const auto& t : expr[(size_t)k]) add(t.first, t.second, -val[(size_t)q]);
      else
        add(x0 + k, one, -val[(size_t)q]);
    }
    e.clear();
    e.reserve(used.size());
    const double d = dg[(size_t)i], dinv = 1.0 / d;
    for (int at : used) e.emplace_back(at, wide_div(acc[(size_t)at], d, dinv));
  };
  // sizes of x_k and of (F x)_k for the growth rule
  std::vector<double> omega((size_t)n, 1.0), size((size_t)n);
  if (!forward)
    for (int i = 0; i < n; ++i) omega[(size_t)i] = 1.0 / dg[(size_t)i];
  for (int i = 0; i < n; ++i) {
    size[(size_t)i] = dg[(size_t)i] * omega[(size_t)i];
    for (int q = ptr[(size_t)i]; q < ptr[(size_t)i + 1]; ++q)
      size[(size_t)i] += std::fabs(val[(size_t)q]) * omega[(size_t)col[(size_t)q]];
  }
  auto growth = [&](int i, const Expr& e) {
    double sum = 0.0;
    for (const auto& t : e) {
      const bool rhs = t.first >= b0 && t.first < b0 + n;
      sum += std::fabs(t.second.hi) * (rhs ? size[(size_t)(t.first - b0)] : omega[(size_t)(t.first - x0)]);
    }
    return sum * dg[(size_t)i] / size[(size_t)i];
  };
  out = TriHost();
  std::vector<Expr> cand;
  for (int l = 0; l < nlev;) {
    ++block;
    std::vector<int> members;
    int end = l;
    for (; end < nlev; ++end) {
      cand.clear();
      double extra = 0.0;
      size_t longest = 0;
      bool grows = false;
      for (int q = lptr[(size_t)end]; q < lptr[(size_t)end + 1]; ++q) {
        const int i = rows[(size_t)q];
        Expr e;
        row_expr(i, e);
        extra += (double)e.size() - (double)(ptr[(size_t)i + 1] - ptr[(size_t)i] + 1);
        longest = std::max(longest, e.size());
        if (end > l) grows |= !(growth(i, e) <= kGrowth);
        cand.push_back(std::move(e));
        if (end > l && (grows || longest > (size_t)kMergedRow)) break;
      }
      if (end > l && (grows || extra * kEntryCycles > kLevelCycles || longest > (size_t)kMergedRow)) break;
      for (int q = lptr[(size_t)end]; q < lptr[(size_t)end + 1]; ++q) {
        const int i = rows[(size_t)q];
        expr[(size_t)i] = std::move(cand[(size_t)(q - lptr[(size_t)end])]);
        in_block[(size_t)i] = block;
        members.push_back(i);
      }
    }
    l = end;
    // rounds of the merged level: rows by length, about six entries per lane
    std::stable_sort(members.begin(), members.end(),
                     [&](int p, int q) { return expr[(size_t)p].size() > expr[(size_t)q].size(); });
    double mean = 0.0;
    for (int i : members) mean += (double)expr[(size_t)i].size();
    mean /= (double)members.size();
    int lg = 0;
    while (lg < 5 && 6.0 * (1 << lg) < mean) ++lg;
    const int per = kTriThreads >> lg;
    for (size_t m0 = 0; m0 < members.size(); m0 += (size_t)per) {
      const int cnt = (int)std::min((size_t)per, members.size() - m0);
      const int lanes = ((cnt << lg) + 31) / 32 * 32;
      const int slots = (int)((expr[(size_t)members[m0]].size() + (1u << lg) - 1) >> lg);
      const size_t off = out.col.size();
      const int rec[8] = {(int)off, slots, lanes, lg, (int)out.row.size(), cnt,
                          m0 + (size_t)per >= members.size() ? 1 : 0, 0};
      out.rec.insert(out.rec.end(), rec, rec + 8);
      out.col.resize(off + (size_t)slots * lanes, -1);
      out.val.resize(out.col.size(), 0.0);
      for (int r = 0; r < cnt; ++r) {
        const int i = members[m0 + (size_t)r];
        out.row.push_back(i);
        const Expr& e = expr[(size_t)i];
        for (size_t t = 0; t < e.size(); ++t) {
          const size_t at = off + (t >> lg) * (size_t)lanes + ((size_t)r << lg) + (t & ((1u << lg) - 1));
          out.col[at] = e[t].first;
          out.val[at] = e[t].second.hi;
        }
      }
    }
    for (int i : members) Expr().swap(expr[(size_t)i]);
  }
}

}  // namespace gmrf
