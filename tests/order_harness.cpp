// The row order under the thread sanitizer: the OpenMP entry points that the compiler calls, on std::thread, which the
// sanitizer follows (it does not follow libgomp).  Chunks are dealt by a relaxed counter, so that only the start and the
// end of a parallel region order its threads.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <random>
#include <thread>

#include "order.h"

static std::atomic<long> g_dealt;
static thread_local int t_id, t_team = 1;
static thread_local long t_start, t_end, t_chunk;

extern "C" {
void GOMP_parallel(void (*fn)(void*), void* data, unsigned threads, unsigned) {
  const int team = (int)threads;
  g_dealt.store(0);
  auto run = [&](int id) {
    t_id = id;
    t_team = team;
    fn(data);
  };
  std::thread th[64];
  for (int i = 1; i < team; ++i) th[i] = std::thread(run, i);
  run(0);
  for (int i = 1; i < team; ++i) th[i].join();
  t_team = 1;
}
bool GOMP_loop_nonmonotonic_dynamic_next(long* lo, long* hi) {
  *lo = t_start + g_dealt.fetch_add(t_chunk, std::memory_order_relaxed);
  *hi = std::min(*lo + t_chunk, t_end);
  return *lo < t_end;
}
bool GOMP_loop_nonmonotonic_dynamic_start(long start, long end, long, long chunk, long* lo, long* hi) {
  t_start = start;
  t_end = end;
  t_chunk = chunk;
  return GOMP_loop_nonmonotonic_dynamic_next(lo, hi);
}
void GOMP_loop_end_nowait(void) {}
int omp_get_thread_num(void) { return t_id; }
int omp_get_num_threads(void) { return t_team; }
}

// random graph (symmetric pattern) of n rows in two components, `far` edges a row anywhere and one to a neighbour
static mmd::HCSR graph(int n, int far) {
  std::mt19937 rng(n);
  std::vector<std::vector<int32_t>> adj(n);
  auto edge = [&](int i, int j) {
    if ((i < n / 3) != (j < n / 3) || i == j) return;
    adj[i].push_back(j);
    adj[j].push_back(i);
  };
  for (int i = 0; i < n; ++i) {
    adj[i].push_back(i);
    edge(i, (i + 1) % n);
    for (int f = 0; f < far; ++f) edge(i, rng() % n);
  }
  mmd::HCSR A;
  A.nrows = A.ncols = n;
  A.rowptr.push_back(0);
  for (auto& r : adj) {
    std::sort(r.begin(), r.end());
    r.erase(std::unique(r.begin(), r.end()), r.end());
    A.col.insert(A.col.end(), r.begin(), r.end());
    A.rowptr.push_back((int32_t)A.col.size());
  }
  return A;
}

int main() {
  for (int n : {1, 1024, 1025, 5000, 20000})
    for (int far : {0, 3}) {
      const mmd::HCSR A = graph(n, far);
      std::vector<int32_t> own(n);
      for (int i = 0; i < n; ++i) own[i] = i;
      const bool s = mmd::scattered(A, own, 1);
      const std::vector<int32_t> serial = mmd::bisection_order(A, 1);
      if (mmd::scattered(A, own, 6) != s || s != (far > 0 && n > 1025)) return 1;
      if (mmd::bisection_order(A, 6) != serial) return 2;
      std::vector<char> seen(n, 0);
      for (int32_t r : serial) seen[r] = 1;
      for (char c : seen)
        if (!c) return 3;
    }
  std::puts("same order");
  return 0;
}
