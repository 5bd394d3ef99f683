// Host model of the greedy's schedule over a Gram matrix (select_gram.cu): which cluster
// size ends a batch first.  Plain C++.
#pragma once

#include <algorithm>
#include <functional>
#include <vector>

namespace last {

// Requests looked at per cluster size, so that choosing one costs the same for any larger
// batch (host time of a whole call on 16384 requests: 3.3 ms when each was scheduled for
// each size, 0.47 now; 1024 requests 228 and 103 us).
constexpr int kSchedRequests = 1024;

struct SchedRequest {
  int blocks;      // of 32 tokens
  double rounds;
};

struct Schedule {
  std::vector<SchedRequest> reqs;   // most work first; a regular sample of a larger batch
  double each = 1.0;                // requests that one of them stands for
  std::vector<double> cost, busy;
};

// `request(i)`: the i-th of n requests, most work first.
template <typename F>
void schedule_begin(Schedule *s, int n, F request) {
  const int m = std::min(n, kSchedRequests);
  s->reqs.resize(m);
  for (int i = 0; i < m; ++i) s->reqs[i] = request((int)((long long)i * n / m));
  s->each = m > 0 ? (double)n / m : 1.0;
}

// When the batch ends (thousands of cycles) on `active` clusters of c CTAs of `warps` worker
// warps: requests go, most work first, to the next free cluster.  A request takes its rounds
// of 27K cycles, 4.6K more per block that a warp holds and 0.4K per CTA (measured: 32K cycles
// a round on 576 tokens in two CTAs, 66K on 4096 in one, 42K on 16384 in twelve).  Once the
// work alone, spread evenly, passes `limit`, that is returned; of a sampled batch, which
// fills many rounds of clusters, the even spread is taken.
inline double schedule_end(Schedule *s, int c, int active, int warps, double limit) {
  const int m = (int)s->reqs.size();
  s->cost.resize(m);
  double total = 0.0, longest = 0.0;
  for (int i = 0; i < m; ++i) {
    const int slots = (s->reqs[i].blocks + c * warps - 1) / (c * warps);
    s->cost[i] = s->reqs[i].rounds * (27.0 + 4.6 * slots + 0.4 * c);
    total += s->cost[i];
    longest = std::max(longest, s->cost[i]);
  }
  const double even = std::max(longest, total * s->each / active);
  if (s->each > 1.0 || even >= limit) return even;
  s->busy.assign(std::min(active, m), 0.0);   // a heap, the next free cluster on top
  double end = 0.0;
  for (int i = 0; i < m; ++i) {
    std::pop_heap(s->busy.begin(), s->busy.end(), std::greater<double>());
    s->busy.back() += s->cost[i];
    end = std::max(end, s->busy.back());
    std::push_heap(s->busy.begin(), s->busy.end(), std::greater<double>());
  }
  return end;
}

}  // namespace last
