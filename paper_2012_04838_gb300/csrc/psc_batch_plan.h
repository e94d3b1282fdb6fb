// The order in which the members of a graph ensemble start within a step, and what
// each is told about its company: host arithmetic on the members' sizes, no CUDA.
#pragma once

#include <algorithm>
#include <cstddef>
#include <vector>

namespace psc {

struct PlanMember {
  size_t bytes;  // its workspace
  int N;
};

struct PlanStart {
  int member;              // index into the members
  std::vector<int> after;  // members whose ends it waits for (none: it starts with the step)
  int share;               // boxes whose passes run on the chip beside it, itself included (PassArgs::share)
  bool crowd;              // other members keep the chip full whatever its tiles do
};

// Workspace let under way at once.
constexpr size_t kBatchBytes = (size_t)320 << 20;

// The largest members first, each started as soon as the members under way leave
// room for it within kBatchBytes (by a model of their run times: grid points and a
// constant), so that small boxes fill the chip together while what they stream does
// not grow far past the L2 cache.  That pays where there are many of them; with few
// it leaves the last ones alone on the chip.  So everything starts at once if it comes
// to no more than half as much again, and no member counts for more than a quarter:
// a box that does not fit the L2 cache by itself gains nothing from an empty chip.
//
// us a step, FP32, all at once / workspaces counted in full / this rule.  Many small
// boxes: 48 x 64^3 + 12 x 96^3 + 3 x 128^3 4548 / 4220 / 4180, 64 + 16 + 4 of them 5914 / 5650 /
// 5574.  Few: 3 x 128^3 940 / 1024 / 946, 8 x 96^3 956 / 1040 / 965.  Larger than the budget:
// 4 x 192^3 3591 / 4341 / 3665, 8 x 192^3 7138 / 8654 / 7323, 3 x 256^3 5655 / 5949 / 5644, 256^3 +
// 8 x 64^3 2245 / 2287 / 2260, 192^3 + 8 x 64^3 1301 / 1379 / 1322; 4 x 128^3 by phase shifts 4215 /
// 4949 / 4249.  (With fewer than four quarters to a budget, 3 x 256^3 and 4 x 192^3 lose 2 to 3%; with
// eight eighths the 63 boxes 5%.)
//
// crowd: the tile variants were measured with a box alone on the chip.  Where other
// members keep it full, the staged 8-column variant is faster in every strided pass
// than the measured mixture, whose wider and unstaged tiles pay by filling idle SMs
// (us a step, mixture -> staged: the 63 boxes 4397 -> 4240, 4 x 192^3 3684 -> 3590; 4 x 64^3, which
// leave room, 172 -> 175).  A grid of 512 or more fills the chip by itself, so its
// own measurement holds in any company (512^3 17.70 -> 17.94 ms, 1024^3 148.9 -> 151.7
// if it is overruled), as it does for a member on its own.
inline std::vector<PlanStart> batch_plan(const std::vector<PlanMember>& m) {
  const int n = (int)m.size();
  auto cost = [](const PlanMember& q) { return std::min(q.bytes, kBatchBytes / 4); };
  size_t total = 0, counted = 0;
  for (const PlanMember& q : m) {
    total += q.bytes;
    counted += cost(q);
  }
  const bool limited = counted > kBatchBytes + kBatchBytes / 2;
  std::vector<int> order(n);
  for (int i = 0; i < n; ++i) order[i] = i;
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return m[x].bytes > m[y].bytes; });
  struct Running {
    double end;
    int i;
  };
  std::vector<Running> run;
  std::vector<PlanStart> plan;
  size_t used = 0;
  double clock = 0.0;
  int last = -1;  // the member whose end made room last
  for (int i : order) {
    PlanStart s{i, {}, 1, false};
    while (limited && !run.empty() && used + cost(m[i]) > kBatchBytes) {
      auto it = std::min_element(run.begin(), run.end(), [](const Running& x, const Running& y) { return x.end < y.end; });
      clock = std::max(clock, it->end);
      last = it->i;
      used -= cost(m[last]);
      run.erase(it);
      s.after.push_back(last);
    }
    if (last >= 0 && s.after.empty()) s.after.push_back(last);
    used += cost(m[i]);
    const double N = m[i].N;
    run.push_back(Running{clock + N * N * N + 3.0e5, i});
    s.share = limited ? (int)std::max<size_t>(1, std::min<size_t>(n, kBatchBytes / std::max<size_t>(cost(m[i]), 1))) : n;
    s.crowd = n > 1 && m[i].N < 512 && total > kBatchBytes;
    plan.push_back(s);
  }
  return plan;
}

}  // namespace psc
