// Host-only program for test_segment_tables.py: prints the tables of build_segment_tables for a graph read from stdin.
#include <cstdio>
#include <vector>

#include "graph_index.hpp"

int main() {
  using namespace gcn_admm_host;
  int n, m, limit;
  long long target, rows;
  if (std::scanf("%d %d %d %lld %lld", &n, &m, &limit, &target, &rows) != 5) return 1;
  std::vector<long long> rp((size_t)n + 1);
  for (auto& v : rp)
    if (std::scanf("%lld", &v) != 1) return 1;
  std::vector<int> ci((size_t)rp[n]), comm((size_t)n);
  for (auto& v : ci)
    if (std::scanf("%d", &v) != 1) return 1;
  for (auto& v : comm)
    if (std::scanf("%d", &v) != 1) return 1;
  GraphIndex g;
  std::string err;
  if (build_graph_index(n, rp.data(), ci.data(), m, comm.data(), g, err) != IDX_OK) return 2;
  LongRowTables lt;
  build_long_row_tables(g, limit, lt);
  SegmentTables t;
  build_segment_tables(g, limit, lt, target, rows, t);
  auto row_of = [&](int entry) { return (int)(std::upper_bound(g.row_ptr.begin(), g.row_ptr.end(), entry) - g.row_ptr.begin()) - 1; };
  for (const SegChunk& c : t.chunks) {
    if (c.length == 0) std::printf("rows %d %d %d %d\n", c.first, c.count, c.comm, c.slot);
    else if (c.length < 0) {
      const Quad& it = lt.items[(size_t)c.first];
      if (it.w != c.count) return 3;
      std::printf("piece %d %d %d %d\n", it.x, c.comm, it.z - it.y, c.slot);
    } else {
      for (int k = c.first; k < c.first + c.count; ++k) {
        const int b = t.segs[(size_t)k].begin, row = row_of(b);
        if (row_of(b + c.length - 1) != row || g.dinv[(size_t)row] != t.segs[(size_t)k].dinv) return 4;
        for (int e = 0; e < c.length; ++e)
          if (g.col_comm[(size_t)(b + e)] != c.comm) return 5;
        std::printf("seg %d %d %d %d\n", row, c.comm, c.length, c.slot);
      }
    }
  }
  std::printf("slots");
  for (int s : t.slot_ptr) std::printf(" %d", s);
  std::printf("\n");
  return 0;
}
