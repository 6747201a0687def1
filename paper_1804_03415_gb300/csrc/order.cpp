// Order of a matrix's rows on the device (host code).
#include "order.h"

#include <algorithm>
#include <cstdlib>

namespace mmd {

// Device order for locality.  The persistent solver's blocks own contiguous
// shares of the rows and fetch every row their entries read once per
// iteration, so what a block reads should be few rows: consecutive ones and a
// thin rim.  True where more than a quarter of A's entries (in the order
// given by iperm) lie further than n / 32 from the diagonal: point clouds and
// geometric graphs numbered at random, not the grid operators.
bool scattered(const HCSR& A, const std::vector<int32_t>& iperm, int threads) {
  const int64_t far = std::max<int64_t>(512, A.nrows / 32);
  int64_t out = 0;
#pragma omp parallel for schedule(static) num_threads(threads) reduction(+ : out)
  for (int64_t r = 0; r < A.nrows; ++r)
    for (int32_t e = A.rowptr[r]; e < A.rowptr[r + 1]; ++e)
      out += std::abs(int64_t(iperm[r]) - iperm[A.col[e]]) > far;
  return out * 4 > A.nnz();
}

// Rows in an order whose short runs are compact pieces of A's graph:
// recursive bisection by breadth-first search.  The whole graph is searched
// from the row that a first search reaches last (an end of it) and its rows
// taken in the order they are reached; the two halves are searched again, the
// first from the row it starts with, the second from the row it ends with,
// down to kLeaf rows.  (One search over the whole graph gives fronts: on a
// 200k-row torus graph a block of 1,316 consecutive rows then reads 4,900
// rows, 3,100 with the pieces.)
std::vector<int32_t> bisection_order(const HCSR& A, int threads) {
  constexpr int64_t kLeaf = 1024;  // a window of the SELL copy
  const int64_t n = A.nrows;
  std::vector<int32_t> q(n), out(n), piece(n, 0);  // piece: the piece a row is in, fixed while pieces are searched
  std::vector<uint8_t> done(n, 0);                 // a row is placed; its own piece's thread alone reads or writes it
  for (int64_t i = 0; i < n; ++i) q[i] = (int32_t)i;
  struct Cut {
    int64_t lo, hi;
    bool from_end;
  };
  std::vector<Cut> cuts{{0, n, false}};
  int32_t pieces = 0;
  // writes the rows of piece id that start reaches to out[at ..]; returns the end
  auto search = [&](int32_t start, int32_t id, int64_t at) {
    int64_t end = at;
    out[end++] = start;
    done[start] = 1;
    for (; at < end; ++at)
      for (int32_t e = A.rowptr[out[at]]; e < A.rowptr[out[at] + 1]; ++e) {
        const int32_t j = A.col[e];
        if (piece[j] == id && !done[j]) {
          done[j] = 1;
          out[end++] = j;
        }
      }
    return end;
  };
  for (int64_t i = 0, at = 0; i < n; ++i)
    if (!done[i]) {
      const int64_t end = search((int32_t)i, 0, at);
      std::swap(out[at], out[end - 1]);  // its component's search starts at the end
      at = end;
    }
  q.swap(out);
  while (!cuts.empty()) {  // the pieces of one depth are independent
    std::vector<Cut> next(2 * cuts.size());
    const int32_t base = pieces + 1;
    pieces += (int32_t)cuts.size();
    for (size_t c = 0; c < cuts.size(); ++c)
      for (int64_t i = cuts[c].lo; i < cuts[c].hi; ++i) {
        piece[q[i]] = base + (int32_t)c;
        done[q[i]] = 0;
      }
#pragma omp parallel for schedule(dynamic, 1) num_threads(threads)
    for (int64_t c = 0; c < (int64_t)cuts.size(); ++c) {
      const int64_t lo = cuts[c].lo, hi = cuts[c].hi;
      const int32_t id = base + (int32_t)c;
      int64_t at = lo;
      for (int64_t i = lo; i < hi; ++i) {  // every component of the piece
        const int32_t start = cuts[c].from_end ? q[hi - 1 - (i - lo)] : q[i];
        if (!done[start]) at = search(start, id, at);
      }
      std::copy(out.begin() + lo, out.begin() + hi, q.begin() + lo);
      if (hi - lo > kLeaf) {
        const int64_t mid = lo + (hi - lo) / 2;
        next[2 * c] = {lo, mid, false};
        next[2 * c + 1] = {mid, hi, true};
      }
    }
    cuts.clear();
    for (const Cut& c : next)
      if (c.hi > c.lo) cuts.push_back(c);
  }
  return q;
}

}  // namespace mmd
