// lw_share.h — how the layer-wise select's CTAs are shared among the segments
// (host code without CUDA, so that it is tested on the CPU).
//
// A segment's selection is work for one CTA (a single) or for a team of
// co-resident CTAs; the singles are dealt onto the CTAs that the teams leave.
// The select ends with its most loaded CTA, so both get their CTAs by one
// measure: a load, in candidates a rank, that by plan no team's rank exceeds
// and no singles' CTA (but for one long single). The load starts at
// kLwRankLoad and grows until teams and singles fit the CTAs there are.
// Teams that took all but one CTA left the singles to it one after another:
// us a call, ResNet-50-shaped at 5 %, 143 singles, 1,285 -> 339; VGG-16-shaped
// at 5 % 12,500 -> 6,080; 138 M coordinates in 200 tensors at 1 % 2,304 -> 383.
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdint>
#include <vector>

namespace efs {

constexpr uint32_t kLwMaxTeam = 32;
// Candidates of a team's rank when CTAs are plenty: its passes over 8 K of
// them take about as long as a team barrier. Measured on a GB300, LSTM-shaped
// call at 1 %, an embedding with 281 K candidates, us: 24 K a rank 127, 16 K
// 117, 12 K 112, 8 K 108.
constexpr uint64_t kLwRankLoad = 8192;
// While no rank's load passes 24 K, the select keeps to 3/5 of the CTAs: the
// next call's sampling and stream begin on the others. Calls in a row, us, 3/5
// against all of them: 100 M coordinates in 60 tensors at 1 % 270 against 295,
// ResNet-50-shaped at 3 % 120 against 130, ResNet-18-shaped at 5 % 78 against
// 87. Beyond, and where the candidates outgrow their list, so that segments
// are selected from e, the select is the longest part and takes all: ResNet-50
// at 5 % 557 against 348, ResNet-18 at 10 % 250 against 180.
constexpr uint64_t kLwSharedLoad = 24 * 1024;
// A segment takes a team from this many candidates on (3/4 of what one CTA
// holds). Teams from 16 K or 24 K on: ResNet-18 at 1 % 70 -> 64, but ResNet-50
// 113 -> 120 and 117.
constexpr uint64_t kLwTeamFrom = 36 * 1024;

struct LwWork {           // a segment that selects anything
  uint64_t candidates;    // expected
  uint64_t cost;          // of its selection by one CTA, in positions handled
  uint32_t least;         // CTAs that its length alone asks for (1: none)
};

// The teams at a load; returns the CTAs that they and the singles ask for.
inline uint64_t lw_teams_at(const std::vector<LwWork>& work, uint64_t load,
                            std::vector<uint32_t>& team) {
  uint64_t ctas = 0, singles = 0, cost = 0, longest = 0;
  for (size_t s = 0; s < work.size(); ++s) {
    const LwWork& w = work[s];
    uint64_t t = w.candidates > kLwTeamFrom ? (w.candidates + load - 1) / load : 1;
    t = std::min<uint64_t>(std::max<uint64_t>(t, w.least), kLwMaxTeam);
    team[s] = static_cast<uint32_t>(t);
    if (t > 1) {
      ctas += t;
    } else {
      ++singles;
      cost += w.cost;
      longest = std::max(longest, w.cost);
    }
  }
  // (a candidate costs about 2 positions)
  const uint64_t per_cta = std::max<uint64_t>(2 * load, longest);
  return ctas + std::min(singles, (cost + per_cta - 1) / per_cta);
}

// team[s]: the CTAs of segment s's team, or 1 for a single, out of `budget`.
// from_e: the candidates are expected to outgrow their list.
inline void lw_share(const std::vector<LwWork>& work, uint32_t budget, bool from_e,
                     std::vector<uint32_t>& team) {
  team.assign(work.size(), 1);
  uint64_t most = 0;
  for (const LwWork& w : work) most = std::max(most, w.candidates);
  if (!from_e)
    for (uint64_t load = kLwRankLoad; load <= kLwSharedLoad; load += load / 8)
      if (lw_teams_at(work, load, team) <= budget * 3ull / 5) return;
  for (uint64_t load = kLwRankLoad; load <= 2 * most + kLwRankLoad; load += load / 8)
    if (lw_teams_at(work, load, team) <= budget) return;
  // lengths alone ask for more CTAs than there are (as the last load left
  // them): the largest teams give theirs up until one is left for the singles
  for (;;) {
    uint64_t asked = 0;
    bool single = false;
    for (uint32_t t : team) {
      if (t > 1)
        asked += t;
      else
        single = true;
    }
    if (asked + (single ? 1 : 0) <= budget) return;
    --*std::max_element(team.begin(), team.end());
  }
}

}  // namespace efs
