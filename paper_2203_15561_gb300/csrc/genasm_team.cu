// Launches of the team kernels, and the starts that the lanes of a team take.
#include "genasm_team.cuh"

#include <cmath>
#include <mutex>
#include <vector>

namespace ga {

namespace {

constexpr int kShort = 32;  // most bases that a start may fall short on either side, plus 1

struct Start {
  double weight;
  int ahead, p, t;
};

// The starts by weight, the known one (nothing ahead) first, packed.
void rank_starts(std::vector<Start>& v, uint16_t (&out)[kTeamLanes]) {
  std::sort(v.begin(), v.end(), [](const Start& x, const Start& y) {
    if (x.weight != y.weight) return x.weight > y.weight;
    if (x.ahead != y.ahead) return x.ahead < y.ahead;
    return x.p != y.p ? x.p < y.p : x.t < y.t;
  });
  out[0] = 0;
  for (int i = 1; i < kTeamLanes; ++i) {
    if (static_cast<size_t>(i) > v.size()) {
      out[i] = 0;
      continue;
    }
    const Start& s = v[static_cast<size_t>(i) - 1];
    out[i] = static_cast<uint16_t>(s.ahead | s.p << 4 | s.t << 10);
  }
}

// Where the windows `ahead` of a known one start if a base brings an insertion
// with probability `ins` and a deletion with `del` (lengths geometric with mean
// 1.5): after each window, the side that is used up has moved on by `commit`
// bases and the other by fewer. A start further ahead is worth less, by `later`
// each window, as it counts only if those before it were guessed.
void model_starts(int commit, double ins, double del, int most_ahead, double later,
                  uint16_t (&out)[kTeamLanes]) {
  constexpr int R = kShort - 1;
  std::vector<double> net(2 * R + 1, 0.0);
  net[R] = 1.0;
  for (int b = 0; b < commit; ++b) {
    std::vector<double> to(2 * R + 1, 0.0);
    for (int x = 0; x <= 2 * R; ++x) {
      if (net[x] < 1e-9) continue;
      to[x] += net[x] * (1.0 - ins - del);
      double q = 2.0 / 3.0;
      for (int l = 1; l <= 8; ++l, q /= 3.0) {
        if (x - l >= 0) to[x - l] += net[x] * ins * q;
        if (x + l <= 2 * R) to[x + l] += net[x] * del * q;
      }
    }
    net = to;
  }
  std::vector<double> at(kShort * kShort, 0.0);
  at[0] = 1.0;
  std::vector<Start> v;
  double worth = 1.0;
  for (int k = 1; k <= most_ahead; ++k, worth *= later) {
    std::vector<double> to(kShort * kShort, 0.0);
    for (int p = 0; p < kShort; ++p) {
      for (int t = 0; t < kShort; ++t) {
        const double x = at[p * kShort + t];
        if (x < 1e-6) continue;
        for (int d = -R; d <= R; ++d) {
          const int p1 = p + std::max(d, 0), t1 = t + std::max(-d, 0);
          if (p1 < kShort && t1 < kShort) to[p1 * kShort + t1] += x * net[d + R];
        }
      }
    }
    at = to;
    for (int p = 0; p < kShort; ++p)
      for (int t = 0; t < kShort; ++t)
        if (at[p * kShort + t] > 0.0) v.push_back({at[p * kShort + t] * worth, k, p, t});
  }
  rank_starts(v, out);
}

// Sequences that do not belong together: the text falls behind by some bases per
// window, about normally distributed round the pair's own mean (t: the distance
// from it, plus 32).
void strange_starts(int commit, uint16_t (&out)[kTeamLanes]) {
  std::vector<Start> v;
  double worth = 1.0;
  for (int k = 1; k <= 6; ++k, worth *= 0.9) {
    const double var = 0.3 * commit * k;
    for (int d = -(kShort - 1); d <= (kShort - 1); ++d)
      v.push_back({std::exp(-d * d / (2.0 * var)) / std::sqrt(var) * worth, k, 0, d + 32});
  }
  rank_starts(v, out);
}

// The starts for windows that commit `commit` bases: three orders by likelihood,
// of which a team of 8 or 16 lanes takes the first. Made once for each (0.2 ms).
const TeamStarts& team_starts(int commit) {
  static std::mutex mutex;
  static TeamStarts made[kMaxW + 1];
  static bool is_made[kMaxW + 1];
  std::lock_guard<std::mutex> lock(mutex);
  TeamStarts& s = made[commit];
  if (!is_made[commit]) {
    model_starts(commit, 0.035, 0.025, 6, 0.9, s.start[kTeamLong]);
    model_starts(commit, 0.001, 0.001, 15, 0.98, s.start[kTeamFew]);
    strange_starts(commit, s.start[kTeamStrange]);
    is_made[commit] = true;
  }
  return s;
}

int log2_of(int x) {
  int l = 0;
  while (1 << l < x) ++l;
  return l;
}

template <class Kernel>
cudaError_t opt_in(Kernel kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
}

template <int VW, int NB>
cudaError_t launch_as(const AlignParams& p, const LanePlan& plan, const uint32_t* order, cudaStream_t s) {
  using Team = TeamShape<VW, NB>;
  const cudaError_t e = opt_in(align_team_kernel<VW, NB>, Team::kBytes);
  if (e != cudaSuccess) return e;
  align_team_kernel<VW, NB>
      <<<plan.warps, Team::kThreads, Team::kBytes, s>>>(p, order, log2_of(plan.team), team_starts(p.W - p.O));
  return cudaGetLastError();
}

template <int VW, int NB>
cudaError_t launch_step_as(const AlignParams& p, int team, int blocks, const StepArgs& a, cudaStream_t s) {
  using Team = TeamShape<VW, NB>;
  const cudaError_t e = opt_in(step_team_kernel<VW, NB>, Team::kBytes);
  if (e != cudaSuccess) return e;
  step_team_kernel<VW, NB>
      <<<blocks, Team::kThreads, Team::kBytes, s>>>(p, a, log2_of(team), team_starts(p.W - p.O));
  return cudaGetLastError();
}

}  // namespace

// Lanes per pair: all that one warp per scheduler gives each of n pairs, from
// blocks of four warps for one pair down to eight lanes; 0: too many pairs, a
// lane each. Reads of 10 kb with a free start, us (one lane; 128 lanes; 32; 16;
// 8; 4), on 152 multiprocessors:
//   152 pairs: 833, 440, 487, 585, 685, 842     608: 846, 1210, 518, 592, 697, 826
//   1,216: 892, -, 855, 636, 728, 868           2,432: 904, -, 1583, 1050, 746, 913
//   4,864: 912, -, -, 1898, 1295, 917 (four lanes: one more window in two rounds)
// and 304 pairs 820 with one lane, 668 with 128, 504 with 32. (W = 64, O = 24; the
// same limits serve every W up to 64.)
int team_size(uint64_t n, int sms) {
  const uint64_t warps = 4ull * sms;
  return n <= warps / 4 ? 128 : n <= warps ? 32 : n <= 2 * warps ? 16 : n <= 4 * warps ? 8 : 0;
}

cudaError_t launch_team(const AlignParams& p, const LanePlan& plan, const uint32_t* order, cudaStream_t s) {
  cudaError_t e;
  if (plan.team == 128) e = plan.vw == 1 ? launch_as<1, 4>(p, plan, order, s) : launch_as<2, 4>(p, plan, order, s);
  else e = plan.vw == 1 ? launch_as<1, 1>(p, plan, order, s) : launch_as<2, 1>(p, plan, order, s);
  if (e == cudaSuccess) count_launches(1);
  return e;
}

cudaError_t launch_step_team(const AlignParams& p, int sms, const StepArgs& a, cudaStream_t s) {
  const int vw = (p.W + 31) / 32;
  const int team = team_size(a.n_active, sms);
  const int blocks = static_cast<int>(std::min<uint64_t>(team == 128 ? sms : 4 * sms, std::max(a.n_active, 1u)));
  cudaError_t e;
  if (team == 128) e = vw == 1 ? launch_step_as<1, 4>(p, team, blocks, a, s) : launch_step_as<2, 4>(p, team, blocks, a, s);
  else e = vw == 1 ? launch_step_as<1, 1>(p, team, blocks, a, s) : launch_step_as<2, 1>(p, team, blocks, a, s);
  if (e == cudaSuccess) count_launches(1);
  return e;
}

}  // namespace ga
