// Batch schedule: how the CTAs of one persistent launch are split into groups
// and which systems each group solves (host code only).
//
// The cost of a system is taken as N * n^2: the Arnoldi steps of
// unpreconditioned GMRES on the Poisson operator grow about like n^2 (the
// condition number) and each step moves O(N) values.  Across sides 64..512
// that spans four decades, so a list of one-CTA groups would leave the launch
// waiting for the CTA that drew a 512^2 system.  Systems whose cost exceeds
// the ideal per-CTA load get a group of several CTAs (in proportion, at most
// one per kMinPointsPerCta points); the other CTAs form one-CTA groups; then
// every system not yet placed goes, largest first, to the group on which it
// would finish earliest.
#include <math.h>

#include <algorithm>
#include <numeric>
#include <vector>

#include "../../include/mlgmres.h"
#include "schedule.h"

namespace mlg {

namespace {
constexpr long long kMinPointsPerCta = 512;  // as for single solves
}

double system_cost(int dim, int n) {
  const double N = dim == 2 ? (double)n * n : (double)n * n * n;
  return N * (double)n * (double)n;
}

int plan_batch(int dim, int count, const int* n, int ctas, std::vector<int>& group_ctas,
               std::vector<int>& group_of, std::vector<int>& order) {
  group_ctas.clear();
  group_of.assign(count, -1);
  order.resize(count);
  if (count <= 0 || ctas <= 0) return 0;
  std::vector<double> cost(count);
  double total = 0.0;
  for (int i = 0; i < count; i++) {
    cost[i] = system_cost(dim, n[i]);
    total += cost[i];
  }
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return cost[a] > cost[b]; });
  const double ideal = total / ctas;
  std::vector<double> load;
  int left = ctas;
  int placed = 0;
  // dedicated multi-CTA groups for the systems that alone exceed the ideal load
  for (int r = 0; r < count; r++) {
    const int i = order[r];
    const int unplaced_after = count - r - 1;
    int want = (int)ceil(cost[i] / ideal - 1e-9);
    const long long N = dim == 2 ? (long long)n[i] * n[i] : (long long)n[i] * n[i] * n[i];
    const int by_size = (int)std::max<long long>(1, N / kMinPointsPerCta);
    // keep one CTA for the remaining systems
    const int avail = left - (unplaced_after > 0 ? 1 : 0);
    want = std::min(want, std::min(by_size, avail));
    if (want <= 1) break;
    group_ctas.push_back(want);
    load.push_back(cost[i] / want);
    group_of[i] = (int)group_ctas.size() - 1;
    left -= want;
    placed++;
  }
  // one-CTA groups for the rest (no more groups than systems left)
  const int singles = std::min(left, count - placed);
  for (int g = 0; g < singles; g++) {
    group_ctas.push_back(1);
    load.push_back(0.0);
  }
  // LPT: the remaining systems, largest first, to the earliest finish
  for (int r = placed; r < count; r++) {
    const int i = order[r];
    int best = 0;
    double best_t = INFINITY;
    for (int g = 0; g < (int)group_ctas.size(); g++) {
      const double t = load[g] + cost[i] / group_ctas[g];
      if (t < best_t) {
        best_t = t;
        best = g;
      }
    }
    load[best] = best_t;
    group_of[i] = best;
  }
  return (int)group_ctas.size();
}

// ------------------------------------------------- V slices in shared memory --
// FP32 2D batches may keep every system's basis in the shared memory of its
// group's CTAs.  A group then needs at least tiles / max_tiles CTAs for each of its
// systems.  Whether that ends earlier than streaming the bases is estimated from a
// system's steps and from what a step takes; measured on GB300 (batches of equal
// systems, m = 5 .. 64, groups of 1 to 152 CTAs, 2 to 320 tiles per CTA): the formulas
// are within 5% rms of 1 131 and 1 590 timings, 23% at worst.  (Formulas of m = 30 alone,
// with n^2 for the steps, chose slices for batches of many small systems, or of m >= 40,
// that took up to twice as long with them.)
namespace {
// Arnoldi steps of GMRES(m) from x0 = 0: about n until the basis is full, then as n^2
// (3 200 solves of n = 5 .. 320, m = 3 .. 64, rtol 1e-4 .. 1e-12: 6-11% rms at one rtol).
double system_steps(int n, const SolveKind& k) {
  const double digits = std::max(2.0, -log10(k.rtol));
  return std::min((double)k.max_iters, (0.44 * digits - 0.35) * n * (1.0 + (double)n / k.m));
}
// us per step with slices: exchanges (few CTAs exchange directly), scalar work by m,
// the passes, and the restart's share
double slice_step_us(int m, int ctas, int tiles) {
  return 2.2 + (ctas > 1 ? 0.9 : 0.0) + (ctas > 12 ? 0.6 : 0.0) + 0.066 * m +
         (0.071 + 0.0004 * m) * tiles + 23.0 / m;
}
// ... and with a streamed basis, all SMs' CTAs sharing L2 and HBM; two_per_sm: more than
// one CTA per SM at work
double stream_step_us(int m, int ctas, int tiles, bool two_per_sm) {
  return 6.2 + (ctas > 1 ? 1.4 : 0.0) +
         (two_per_sm ? 0.16 + 0.0024 * m : 0.11 + 0.0018 * m) * tiles + 17.0 / m;
}
int tiles_per_cta(int n, int ctas) {
  const int tiles = (n * n + 31) / 32;
  return (tiles + ctas - 1) / ctas;
}
}  // namespace

double stream_makespan(int count, const int* n, const SolveKind& k, int sms,
                       const std::vector<int>& group_ctas, const std::vector<int>& group_of) {
  std::vector<double> load(group_ctas.size(), 0.0);
  const bool two = std::accumulate(group_ctas.begin(), group_ctas.end(), 0) > sms;
  for (int i = 0; i < count; i++) {
    const int c = group_ctas[group_of[i]];
    load[group_of[i]] +=
        system_steps(n[i], k) * stream_step_us(k.m, c, tiles_per_cta(n[i], c), two);
  }
  return *std::max_element(load.begin(), load.end());
}

// (Timed on 150 mixed batches of 2 to 400 systems, sides 8 to 251, m = 3 to 64: where the
// ratio of the estimates lay between 0.9 and 1.05, that of the times was within 6% of it.)
bool slices_pay(double slices, double stream) { return slices < 0.95 * stream; }

// For a target makespan every system has a least CTA count (its slices fit, and
// alone it ends in time); systems in decreasing order of size go to the group of
// at least that many CTAs where they end earliest within the target, else open a
// group of exactly that many.  The smallest target that places everything, by
// bisection; CTAs left over then go to the groups that end last.
int plan_batch_slices(int count, const int* n, const SolveKind& k, int ctas, int max_tiles,
                      std::vector<int>& group_ctas, std::vector<int>& group_of,
                      std::vector<int>& order, double* makespan) {
  order.resize(count);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return n[a] > n[b]; });
  std::vector<double> steps(count);
  for (int i = 0; i < count; i++) steps[i] = system_steps(n[i], k);
  auto time = [&](int i, int c) {
    return steps[i] * slice_step_us(k.m, c, tiles_per_cta(n[i], c));
  };
  std::vector<double> load;
  auto place = [&](double target) {
    group_ctas.clear();
    load.clear();
    group_of.assign(count, -1);
    int left = ctas;
    for (int i : order) {
      const int tiles = (n[i] * n[i] + 31) / 32;
      int need = (tiles + max_tiles - 1) / max_tiles;
      while (need <= ctas && time(i, need) > target) need++;
      if (need > ctas) return false;
      int best = -1;
      double best_t = target;
      for (int g = 0; g < (int)group_ctas.size(); g++) {
        if (group_ctas[g] < need) continue;
        const double t = load[g] + time(i, group_ctas[g]);
        if (t <= best_t) {
          best_t = t;
          best = g;
        }
      }
      if (best < 0) {
        if (need > left) return false;
        left -= need;
        group_ctas.push_back(need);
        load.push_back(0.0);
        best = (int)group_ctas.size() - 1;
        best_t = time(i, need);
      }
      load[best] = best_t;
      group_of[i] = best;
    }
    return true;
  };
  // all systems one after the other on all CTAs always fits (if any plan does)
  double hi = 0.0, lo = 0.0;
  for (int i = 0; i < count; i++) {
    if (tiles_per_cta(n[i], ctas) > max_tiles) return 0;
    hi += time(i, ctas);
    lo = std::max(lo, steps[i] * slice_step_us(k.m, 2, 1));
  }
  hi *= 1.000001;
  for (int it = 0; it < 24 && hi > 1.002 * lo; it++) {
    const double mid = 0.5 * (lo + hi);
    (place(mid) ? hi : lo) = mid;
  }
  if (!place(hi)) {  // the whole launch as one group
    group_ctas.assign(1, ctas);
    group_of.assign(count, 0);
  }
  // the CTAs left over, one at a time, to the group that ends last (as long as
  // they shorten it)
  const int G = (int)group_ctas.size();
  auto group_time = [&](int g, int c) {
    double t = 0.0;
    for (int i = 0; i < count; i++)
      if (group_of[i] == g) t += time(i, c);
    return t;
  };
  load.assign(G, 0.0);
  int left = ctas;
  for (int g = 0; g < G; g++) {
    load[g] = group_time(g, group_ctas[g]);
    left -= group_ctas[g];
  }
  while (left > 0) {
    const int g = (int)(std::max_element(load.begin(), load.end()) - load.begin());
    int add = 1;
    while (add <= left && group_time(g, group_ctas[g] + add) >= load[g]) add++;
    if (add > left) break;
    group_ctas[g] += add;
    left -= add;
    load[g] = group_time(g, group_ctas[g]);
  }
  *makespan = *std::max_element(load.begin(), load.end());
  return G;
}

}  // namespace mlg

extern "C" mlgmres_status mlgmres_batch_plan_slices(int count, const int* n, int m, double rtol,
                                                    long long max_iters, int ctas,
                                                    int stream_ctas, int max_tiles, int* groups,
                                                    int* group_ctas, int* group_of,
                                                    int* preferred) {
  if (count < 1 || m < 1 || !(rtol > 0.0 && rtol < 1.0) || max_iters < 1 || ctas < 1 ||
      stream_ctas < 1 || max_tiles < 1 || !n || !groups || !group_ctas || !group_of || !preferred)
    return MLGMRES_ERR_ARG;
  for (int i = 0; i < count; i++)
    if (n[i] < 1 || n[i] > 32768) return MLGMRES_ERR_ARG;
  const mlg::SolveKind k{m, rtol, max_iters};
  std::vector<int> gc, gof, order, sgc, sgof;
  double span = 0.0;
  mlg::plan_batch(2, count, n, stream_ctas, sgc, sgof, order);
  const int G = mlg::plan_batch_slices(count, n, k, ctas, max_tiles, gc, gof, order, &span);
  *groups = G;
  *preferred =
      G > 0 && mlg::slices_pay(span, mlg::stream_makespan(count, n, k, ctas, sgc, sgof)) ? 1 : 0;
  for (int g = 0; g < G; g++) group_ctas[g] = gc[g];
  for (int i = 0; i < count && G > 0; i++) group_of[i] = gof[i];
  return MLGMRES_OK;
}

extern "C" mlgmres_status mlgmres_batch_plan(int dim, int count, const int* n, int ctas,
                                             int* groups, int* group_ctas, int* group_of) {
  if ((dim != 2 && dim != 3) || count < 1 || ctas < 1 || !n || !groups || !group_ctas ||
      !group_of)
    return MLGMRES_ERR_ARG;
  for (int i = 0; i < count; i++)
    if (n[i] < 1) return MLGMRES_ERR_ARG;
  std::vector<int> gc, gof, order;
  const int G = mlg::plan_batch(dim, count, n, ctas, gc, gof, order);
  *groups = G;
  for (int g = 0; g < G; g++) group_ctas[g] = gc[g];
  for (int i = 0; i < count; i++) group_of[i] = gof[i];
  return MLGMRES_OK;
}
