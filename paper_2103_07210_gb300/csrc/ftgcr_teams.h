// The schedule of a launch of several banded solves (ftgcr_band.cuh): teams of
// CTAs, each with a list of solves.  Host code without CUDA.
#pragma once
#include <algorithm>
#include <vector>

namespace ftgcr {

// The part of a launch a CTA works in.
struct TeamCta {
  int team, rank, size;
  int q0, q1;  // the team's solves: order[q0 .. q1)
};

// The launches of a batch or an epoch: 0 the solves of the other kernels, 1
// banded solves side by side in teams, 2 banded solves of kWholePoints or more
// with bands for most of the SMs, which take all CTAs one after another: on a
// few CTAs such a solve reads its vectors from L2 or memory, on all of them its
// bands stay on chip.  Smaller ones leave CTAs idle or pay for barriers among
// all.  The line lies between 512 x 256 and 1024 x 512 points: ms with none /
// 2048 x 1024 / 1024 x 512 and up / 512 x 256 and up taken whole, 32 mixed
// solves served 37.5 / 23.6 / 21.5 / 23.3, 21 FP64 ones 52.3 / 43.0 / 40.7 /
// 42.3, a batch of 128 mixed solves (to 1024 x 512) 36.4 / 36.4 / 33.6 / 40.7,
// of 28 FP64 ones 29.4 / 29.4 / 23.8 / 24.6.
// Of fewer bands, whole solves leave the other CTAs idle.  On 152 SMs, whole /
// in teams, ms: 16 FP64 1024 x 512 of 32 bands 124.0 / 34.3, of 64 68.8 / 36.6,
// of 86 57.7 / 41.1, of 103 52.6 / 45.2, of 128 42.7 / 43.0; mixed of 43 32.9 /
// 16.7, of 86 17.2 / 17.2, of 103 19.6 / 20.8, of 128 17.1 / 20.0; 16 mixed
// 4000 x 66 (66 bands) 17.7 / 11.9, 4000 x 90 18.3 / 15.2; 8 mixed 512 x 512 of
// 66 8.0 / 5.4, of 100 7.0 / 7.3.  The line at five eighths lies where mixed
// solves cross over.
constexpr long long kWholePoints = 1LL << 18;
inline int band_class(long long points, int nt, int sms) { return points >= kWholePoints && 8 * nt > 5 * sms ? 2 : 1; }

// Teams of CTAs for a launch of several banded solves.  A team runs its solves
// one after another, so a solve's rounds wait for nobody else's.  As many
// teams as keep at least kTeamMin CTAs each (a 1024 x 512 solve on one SM
// takes eight times a round's fixed cost), at most one per solve; CTAs go to
// teams by the largest solve each would take, then every solve, largest first,
// to the team that would finish it soonest.  CTAs still left then go to the
// teams whose lists hold solves of more bands than the team has CTAs: of the
// solves of a team the one with the most bands need not have the most points
// (mixed 1024 x 512 with 128 bands and 700 x 700 with 140 on one team of 128:
// the second took two bands a CTA, its vectors off chip).
constexpr int kTeamMin = 8;
struct TeamPlan {
  std::vector<TeamCta> cta;  // [grid]
  std::vector<int> order;    // solves (indices into the argument), team by team
  int teams = 0;
};
inline void plan_teams(const std::vector<long long>& points, const std::vector<int>& nt, int sms, int most_teams,
                       TeamPlan* out) {
  const int n = (int)points.size();
  std::vector<int> by(n);
  for (int i = 0; i < n; ++i) by[i] = i;
  std::stable_sort(by.begin(), by.end(), [&](int a, int b) { return points[a] > points[b]; });
  const int teams = std::max(1, std::min({n, sms / kTeamMin, most_teams}));
  // sizes: one CTA each, then one by one to the team with the most points per CTA
  std::vector<int> size(teams, 1);
  for (int left = sms - teams; left > 0; --left) {
    int best = -1;
    double load = 0;
    for (int t = 0; t < teams; ++t) {
      if (size[t] >= nt[by[t]]) continue;
      const double l = (double)points[by[t]] / size[t];
      if (best < 0 || l > load) best = t, load = l;
    }
    if (best < 0) break;
    ++size[best];
  }
  std::vector<double> busy(teams, 0.0);
  std::vector<std::vector<int>> list(teams);
  for (int i : by) {
    int best = 0;
    double end = 0;
    for (int t = 0; t < teams; ++t) {
      // a round: its points over the team's CTAs, plus a fixed cost worth about 8192 points
      const double e = busy[t] + (double)points[i] / std::min(size[t], nt[i]) + 8192.0;
      if (t == 0 || e < end) best = t, end = e;
    }
    busy[best] = end;
    list[best].push_back(i);
  }
  std::vector<int> most(teams, 0);
  std::vector<double> work(teams, 0.0);
  int left = sms;
  for (int t = 0; t < teams; ++t) {
    for (int i : list[t]) {
      most[t] = std::max(most[t], nt[i]);
      work[t] += (double)points[i];
    }
    size[t] = std::min(size[t], most[t]);
    left -= size[t];
  }
  for (; left > 0; --left) {
    int best = -1;
    for (int t = 0; t < teams; ++t)
      if (size[t] < most[t] && (best < 0 || work[t] / size[t] > work[best] / size[best])) best = t;
    if (best < 0) break;
    ++size[best];
  }
  out->cta.clear();
  out->order.clear();
  out->teams = 0;
  for (int t = 0; t < teams; ++t) {
    if (list[t].empty()) continue;
    const int q0 = (int)out->order.size();
    for (int i : list[t]) out->order.push_back(i);
    for (int r = 0; r < size[t]; ++r)
      out->cta.push_back(TeamCta{out->teams, r, size[t], q0, (int)out->order.size()});
    ++out->teams;
  }
}

}  // namespace ftgcr
