// Checks the clustered batch kernel's tables (csrc/batch_map_plan.cpp): every
// row in one unit of its class, every vertex's flip byte in its row's place,
// every block a sender in every class of a cluster, and every index inside the
// array or the shared memory that the kernel gives it. Usage: batch_map_check K SEED
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "../paper_1807_10750_gb300/csrc/batch_map_plan.h"
#include "../paper_1807_10750_gb300/csrc/host_graph.h"

using namespace isingx;

#define CHECK(x)                                  \
  do {                                            \
    if (!(x)) {                                   \
      std::printf("line %d: %s\n", __LINE__, #x); \
      std::exit(1);                               \
    }                                             \
  } while (0)

int main(int argc, char** argv) {
  CHECK(argc == 3);
  const int K = std::atoi(argv[1]);
  std::mt19937 rng(static_cast<uint32_t>(std::atoi(argv[2])));
  std::vector<BatchMapRows> rows;
  const int sizes[] = {1, 2, 31, 32, 33, 129, 1000, 4097, 20000};
  int32_t vtx = 0;
  for (int n : sizes) {
    std::vector<int32_t> src, dst, w;
    for (int i = 0; i < 5 * n && n > 1; ++i) {
      const int a = static_cast<int>(rng() % static_cast<uint32_t>(n)), b = static_cast<int>(rng() % static_cast<uint32_t>(n));
      if (a != b) src.push_back(a), dst.push_back(b), w.push_back(static_cast<int>(rng() % 17u) - 8);
    }
    HostGraph g;
    CHECK(build_host_graph(n, static_cast<int64_t>(src.size()), src.data(), dst.data(), w.data(), &g) == 0);
    BatchMapRows r;
    r.id = static_cast<int32_t>(rows.size());
    r.vtx_base = vtx + 100;
    r.class_begin = g.class_begin;
    r.perm = g.perm;
    for (int v = 0; v < n; ++v) {
      r.degree.push_back(g.row_ptr[v + 1] - g.row_ptr[v]);
      int s = 0;
      for (int e = g.row_ptr[v]; e < g.row_ptr[v + 1]; ++e) s += g.w[e];
      r.wsum.push_back(s);
    }
    rows.push_back(r);
    vtx += n;
  }
  BatchMapPlan p;
  std::vector<const BatchMapRows*> all;
  for (const BatchMapRows& r : rows) all.push_back(&r);
  CHECK(build_batch_map(all, false, 8, K, 232448, &p));
  CHECK(p.smem <= 232448 && p.map_bytes % 32 == 0 && p.inst.size() == rows.size());
  std::vector<int> filled(static_cast<size_t>(p.groups), 0);
  for (size_t gi = 0; gi < rows.size(); ++gi) {
    const BatchMapInst& I = p.inst[gi];
    const BatchMapRows& r = rows[gi];
    CHECK(I.id == static_cast<int>(gi) && I.n == static_cast<int>(r.degree.size()) && I.vtx_base == r.vtx_base && I.flush * 4 * 8 <= 127);
    std::vector<int> seen(static_cast<size_t>(I.n), 0), at(static_cast<size_t>(p.map_bytes), 0);
    for (int c = 0; c < I.classes; ++c) {
      int bytes = 0;
      for (int k = 0; k < K; ++k) {
        const int u0 = p.block_unit[I.unit0 + k], units = p.block_unit[I.unit0 + k + 1] - u0;
        const int32_t* cu = p.class_unit.data() + I.class_unit0 + k * (I.classes + 1);
        CHECK(units <= p.units_max && cu[I.classes] == units && cu[c] <= cu[c + 1] && (K == 1 || cu[c] < cu[c + 1]));
        for (int i = cu[c]; i < cu[c + 1]; ++i) {
          const BatchMapUnit& u = p.units[u0 + i];
          const int count = u.shape & 0xffff, groups = u.shape >> 16;
          CHECK(p.unit_inst[u0 + i] == static_cast<int>(gi) && u.base >= 32 && u.base % 32 == 0 && u.base + 32 <= p.map_bytes);
          bytes += 32;
          for (int g = 0; g < groups; ++g) CHECK(!filled[u.words + g]++);
          for (int l = 0; l < 32; ++l) CHECK(!at[u.base + l]++);
          for (int l = 0; l < count; ++l) {
            const int v = u.pos + l;
            CHECK(v >= r.class_begin[c] && v < r.class_begin[c + 1] && !seen[v]++);
            CHECK(r.degree[v] <= 4 * groups && p.map_index[I.row0 + v] == u.base + l);
            CHECK(p.row_sum[I.row0 + v] == r.wsum[v]);
            const int d = p.dst[I.dst0 + r.perm[v]];
            CHECK((d >> 24) == k && (d & 0xffffff) == 32 * i + l && 32 * i + l < 32 * p.units_max);
          }
        }
      }
      CHECK(bytes == p.class_bytes[I.class_bytes0 + c]);
    }
    for (int x : seen) CHECK(x == 1);
    const int padded = (I.n + 127) / 128 * 128;
    CHECK(I.dst0 + padded <= static_cast<int>(p.dst.size()));
    for (int v = I.n; v < padded; ++v) CHECK(p.dst[I.dst0 + v] == -1);
  }
  std::printf("ok\n");
  return 0;
}
