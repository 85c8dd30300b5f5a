// Batch schedule (host code): see schedule.cu.
#pragma once
#include <vector>

namespace mlg {

// Cost estimate of one system of side n (dim 2 or 3): N * n^2.
double system_cost(int dim, int n);

// Splits `ctas` CTAs into groups and assigns each of the `count` systems to a
// group.  Returns the number of groups G; group_ctas[0..G-1] sum to at most
// `ctas`; group_of[i] is system i's group; order lists the systems by
// decreasing cost (the order in which each group takes its systems).
int plan_batch(int dim, int count, const int* n, int ctas, std::vector<int>& group_ctas,
               std::vector<int>& group_of, std::vector<int>& order);

// What the solves of a batch have in common.
struct SolveKind {
  int m;
  double rtol;
  long long max_iters;
};

// The schedule of a 2D FP32 batch whose bases stay in shared memory: group_ctas[g]
// CTAs hold slices of at most max_tiles tiles of each of their systems.  Returns
// the number of groups, 0 if some system does not fit; *makespan in the unit of
// stream_makespan, which estimates a streamed schedule on a GPU of `sms` SMs.
int plan_batch_slices(int count, const int* n, const SolveKind& k, int ctas, int max_tiles,
                      std::vector<int>& group_ctas, std::vector<int>& group_of,
                      std::vector<int>& order, double* makespan);
double stream_makespan(int count, const int* n, const SolveKind& k, int sms,
                       const std::vector<int>& group_ctas, const std::vector<int>& group_of);
// Whether the slices' estimate is enough below the streamed one's.
bool slices_pay(double slices, double stream);

}  // namespace mlg
