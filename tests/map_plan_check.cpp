// Walks the spin-map engine's plan (csrc/map_plan.cpp) on the CPU the way its
// kernels do -- every block's rounds of tasks, the entries by lane, the
// stores, words or messages that carry the new spins -- with every index
// checked against its array, and compares the spins of three sweeps with a
// plain sweep over the rows. Usage: map_plan_check KIND N M WMAX MODE K WIDE SEED [SPLIT]
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <utility>
#include <vector>

#include "../paper_1807_10750_gb300/csrc/host_graph.h"

using namespace isingx;

#define CHECK(x)                                           \
  do {                                                     \
    if (!(x)) {                                            \
      std::printf("line %d: %s\n", __LINE__, #x);          \
      std::exit(1);                                        \
    }                                                      \
  } while (0)

static int decide(long f, int old, uint32_t p, int sweep) {
  const int s = f > 0 ? -1 : (f < 0 ? 1 : old);
  return (p * 2654435761u + static_cast<uint32_t>(sweep) * 97u) % 7u == 0 ? -s : s;  // some flips
}

static uint32_t spin_bytes(uint32_t bits) {
  return 0x01010101u + (((bits & 15u) * 0x00204081u) & 0x01010101u) * 0xfeu;
}

int main(int argc, char** argv) {
  CHECK(argc == 9 || argc == 10);
  const bool split = argc == 10 && std::atoi(argv[9]) != 0;
  const int kind = std::atoi(argv[1]), n = std::atoi(argv[2]), m = std::atoi(argv[3]), wmax = std::atoi(argv[4]);
  const int mode = std::atoi(argv[5]), K = std::atoi(argv[6]);
  const bool wide = std::atoi(argv[7]) != 0;
  std::mt19937 rng(static_cast<uint32_t>(std::atoi(argv[8])));
  std::vector<int32_t> src, dst, w;
  auto edge = [&](int a, int b) {
    if (a == b) return;
    const int x = 1 + static_cast<int>(rng() % static_cast<uint32_t>(wmax));
    src.push_back(a), dst.push_back(b), w.push_back((rng() & 1u) ? x : -x);
  };
  if (kind == 0)  // m random pairs
    for (int i = 0; i < m; ++i) edge(static_cast<int>(rng() % static_cast<uint32_t>(n)), static_cast<int>(rng() % static_cast<uint32_t>(n)));
  else if (kind == 1)  // complete graph
    for (int i = 0; i < n; ++i)
      for (int j = i + 1; j < n; ++j) edge(i, j);
  else  // m long rows on a cycle, with hubs (kind 3) of 256 to 1500 entries, many of them each other's
    for (int i = 0; i < n; ++i) {
      edge(i, (i + 1) % n);
      if (i < m)
        for (int j = 0; j < (kind == 2 ? 200 : 256 + 1500 * i / m); ++j)
          edge(i, kind == 2 || j % 3 != 0 ? m + static_cast<int>(rng() % static_cast<uint32_t>(n - m))
                                          : static_cast<int>(rng() % static_cast<uint32_t>(m)));
    }
  HostGraph g;
  CHECK(build_host_graph(n, static_cast<int64_t>(src.size()), src.data(), dst.data(), w.data(), &g) == 0);
  const int64_t limit = 232448;
  MapPlan mp;
  build_map_plan(g, mode, K, wide, limit, &mp, split);
  if (!mp.ok) {
    std::printf("no plan\n");
    return 2;
  }
  const int C = g.num_colours;
  const size_t stride = static_cast<size_t>(C) + 1;
  CHECK(mp.smem_bytes <= limit && mp.map_bytes % 16 == 0 && mp.warps >= 1 && mp.warps <= kMapMaxWarps);
  std::vector<int> spin(static_cast<size_t>(n)), seen(static_cast<size_t>(mp.map_bytes), 0);
  std::vector<std::vector<int8_t>> maps(static_cast<size_t>(K), std::vector<int8_t>(static_cast<size_t>(mp.map_bytes), 1));
  for (int p = 0; p < n; ++p) {
    spin[p] = (rng() & 1u) ? 1 : -1;
    CHECK(mp.map_index[p] >= 0 && mp.map_index[p] + 32 <= mp.map_bytes && !seen[mp.map_index[p]]++);
    for (auto& one : maps) one[mp.map_index[p]] = static_cast<int8_t>(spin[p]);
  }
  for (const MapBlock& b : mp.blocks) {
    CHECK(b.rounds * mp.warps <= mp.max_tasks && b.rows <= mp.max_rows && b.groups <= mp.max_groups && b.rows % 32 == 0);
    CHECK(static_cast<size_t>(b.task0 + b.rounds * mp.warps) <= mp.tasks.size());
    CHECK(b.words0 + b.groups <= mp.total_groups);
    CHECK(static_cast<size_t>(b.row0 + b.rows) <= mp.row_pos.size() && mp.row_pos.size() == mp.row_orig.size());
  }
  CHECK(mp.hubs == (split ? g.num_hubs : 0) && mp.late.size() == 2 * static_cast<size_t>(mp.hubs));
  // a part of a split row, summed in class c's step: none of its terms from that class
  std::vector<std::vector<long>> acc(static_cast<size_t>(K), std::vector<long>(static_cast<size_t>(mp.max_acc) + 32, 0));
  std::vector<std::vector<int>> summed(static_cast<size_t>(K), std::vector<int>(static_cast<size_t>(mp.max_acc) + 32, 0));
  std::vector<int> got(static_cast<size_t>(K), 0);
  auto add_part = [&](int k, const MapTask& x, int c) {
    const MapBlock& b = mp.blocks[static_cast<size_t>(k)];
    const int slot = x.base & ((1 << kMapOwnerShift) - 1), groups = x.shape >> 16;
    const int owner = (x.base & ((1 << kMapFlipShift) - 1)) >> kMapOwnerShift;
    CHECK(owner < K);
    got[static_cast<size_t>(owner)] += 4;
    const int p = mp.row_pos[static_cast<size_t>(mp.blocks[static_cast<size_t>(owner)].row0 + (x.row & ((1 << kMapSplitShift) - 1)))];
    CHECK(slot < mp.max_acc && p >= 0 && p < mp.hubs && groups <= mp.stage && x.words + groups <= b.groups);
    CHECK(p >= g.class_begin[(c + 1) % C] && p < g.class_begin[(c + 1) % C + 1]);
    const int l0 = mp.late[2 * p], l1 = mp.late[2 * p + 1];
    CHECK(l0 >= g.row_ptr[p] && l0 <= l1 && l1 <= g.row_ptr[p + 1]);
    for (int lane = 0; lane < 32; ++lane)
      for (int s = 0; s < 4 * groups; ++s) {
        int e = g.row_ptr[p] + ((x.row & 0x7fffffff) >> kMapSplitShift) * kMapPartEntries + lane + 32 * s;
        if (e >= l0) e += l1 - l0;
        if (e >= g.row_ptr[p + 1]) continue;
        CHECK(g.col[e] < g.class_begin[c] || g.col[e] >= g.class_begin[c + 1]);
        acc[static_cast<size_t>(owner)][static_cast<size_t>(slot)] += static_cast<long>(g.w[e]) * maps[k][mp.map_index[g.col[e]]];
        summed[static_cast<size_t>(owner)][static_cast<size_t>(slot)]++;
      }
  };
  for (int k = 0; k < K && split; ++k)
    for (int i = mp.blocks[k].last0; i < mp.blocks[k].rounds * mp.warps; ++i) {
      const MapTask x = mp.tasks[static_cast<size_t>(mp.blocks[k].task0 + i)];
      if (((x.shape >> 8) & 0xff) == kMapPart) add_part(k, x, C - 1);
    }
  std::vector<int> filled(static_cast<size_t>(mp.total_groups), 0);
  for (int sweep = 0; sweep < 3; ++sweep) {
    std::vector<int> round(static_cast<size_t>(K), 0);
    std::vector<std::vector<int>> drawn(static_cast<size_t>(K));
    for (int k = 0; k < K; ++k) drawn[k].assign(static_cast<size_t>(mp.blocks[k].rows / 32), 0);
    for (int c = 0; c < C; ++c) {
      std::vector<int> now;
      for (int p = g.class_begin[c]; p < g.class_begin[c + 1]; ++p) {
        long f = 0;
        for (int e = g.row_ptr[p]; e < g.row_ptr[p + 1]; ++e) f += static_cast<long>(g.w[e]) * spin[g.col[e]];
        now.push_back(decide(f, spin[p], static_cast<uint32_t>(p), sweep));
      }
      for (size_t i = 0; i < now.size(); ++i) spin[static_cast<size_t>(g.class_begin[c]) + i] = now[i];
      std::vector<std::pair<int, uint32_t>> stores, messages;  // cluster: words; grid: message and bits
      long bytes = 0;
      std::vector<std::pair<int, MapTask>> parts;
      for (int k = 0; k < K; ++k) {
        const MapBlock& b = mp.blocks[k];
        const size_t t = static_cast<size_t>(k) * stride + static_cast<size_t>(c);
        std::vector<std::pair<int, int>> own;
        int units = 0;
        for (bool more = true; more; ++round[k]) {
          CHECK(round[k] < b.rounds);
          for (int warp = 0; warp < mp.warps; ++warp) {
            const MapTask x = mp.tasks[static_cast<size_t>(b.task0 + round[k] * mp.warps + warp)];
            const int draw = static_cast<int>(static_cast<uint32_t>(x.base) >> kMapFlipShift) - 1;
            if (draw >= 0) {
              CHECK(draw < b.rows / 32);
              drawn[k][draw]++;
            }
            if (warp == 0) more = x.row >= 0;
            CHECK(more == (x.row >= 0));
            if (x.shape == 0) continue;
            if (((x.shape >> 8) & 0xff) == kMapPart) {
              parts.push_back({k, x});
              continue;
            }
            ++units;
            const int base = x.base & ((1 << kMapFlipShift) - 1), row = x.row & ((1 << kMapSplitShift) - 1);
            const int slot = (x.row & 0x7fffffff) >> kMapSplitShift;
            const int rows = x.shape & 0xff, lg = (x.shape >> 8) & 0xff, groups = x.shape >> 16;
            CHECK(lg <= 5 && rows <= (32 >> lg) && groups <= mp.stage && x.words + groups <= b.groups);
            CHECK(row >= mp.class_row[t] && row + rows <= mp.class_row[t + 1] && base + 32 <= mp.map_bytes);
            CHECK((row + (32 >> lg) - 1) / 32 < mp.max_rows / 32 || rows == 0 || row + 31 < mp.max_rows + 32);
            long f[32] = {0};
            int terms = 0, entries = 0;
            for (int lane = 0; lane < 32; ++lane) {
              const int r = lane & ((32 >> lg) - 1);
              if (r >= rows) continue;
              const int p = mp.row_pos[static_cast<size_t>(b.row0 + row + r)];
              CHECK((slot != 0) == (p < mp.hubs));
              const int begin = p < mp.hubs ? mp.late[2 * p] : g.row_ptr[p], end = p < mp.hubs ? mp.late[2 * p + 1] : g.row_ptr[p + 1];
              if (lane == r) entries += end - begin;
              for (int s = 0; s < 4 * groups; ++s) {
                const int e = begin + (lane >> (5 - lg)) + (s << lg);
                if (e >= end) continue;
                f[r] += static_cast<long>(g.w[e]) * maps[k][mp.map_index[g.col[e]]];
                ++terms;
              }
            }
            CHECK(terms == entries);
            for (int r = 0; r < rows && slot != 0; ++r) {
              const size_t i = static_cast<size_t>(slot - 1 + r);
              const int p = mp.row_pos[static_cast<size_t>(b.row0 + row + r)];
              CHECK(summed[k][i] + mp.late[2 * p + 1] - mp.late[2 * p] == g.row_ptr[p + 1] - g.row_ptr[p]);
              f[r] += acc[k][i];
              acc[k][i] = summed[k][i] = 0;
            }
            for (int gp = 0; gp < groups; ++gp) CHECK(!filled[b.words0 + x.words + gp]++ || sweep > 0);
            uint32_t bits = 0;
            for (int r = 0; r < rows; ++r) {
              const int p = mp.row_pos[static_cast<size_t>(b.row0 + row + r)];
              CHECK(p >= g.class_begin[c] && p < g.class_begin[c + 1] && mp.map_index[p] == base + r);
              CHECK(mp.row_orig[static_cast<size_t>(b.row0 + row + r)] == g.perm[p]);
              CHECK(mp.class_seg[t] + row + r - mp.class_row[t] == base + r);
              const int s = decide(f[r], maps[k][base + r], static_cast<uint32_t>(p), sweep);
              if (s < 0) bits |= 1u << r;
              own.push_back({base + r, s});
            }
            if (mode == kMapCluster) {
              const int width = lg < 3 ? 32 >> lg : 4;
              CHECK(base % width == 0);
              bytes += width;
              for (int q = 0; q < width / 4; ++q) stores.push_back({base + 4 * q, spin_bytes(bits >> (4 * q))});
            }
          }
        }
        CHECK(mode != kMapCluster || units > 0);
        if (mode != kMapCluster)
          for (const auto& o : own) maps[k][o.first] = static_cast<int8_t>(o.second);
        if (mode == kMapGrid) {
          const int rows = mp.class_row[t + 1] - mp.class_row[t];
          if (rows == 0) messages.push_back({mp.block_msg[t], 0u});
          for (int j = 0; 32 * j < rows; ++j) {
            uint32_t bits = 0;
            for (int l = 0; l < 32; ++l)
              if (mp.row_orig[static_cast<size_t>(b.row0 + mp.class_row[t] + 32 * j + l)] >= 0 &&
                  maps[k][mp.class_seg[t] + 32 * j + l] < 0)
                bits |= 1u << l;
            messages.push_back({mp.block_msg[t] + j, bits});
          }
        }
      }
      got.assign(static_cast<size_t>(K), 0);
      for (const auto& x : parts) add_part(x.first, x.second, c);
      for (int k = 0; k < K && split; ++k) CHECK(got[k] == mp.block_msg[static_cast<size_t>(k) * stride + static_cast<size_t>(c)]);
      if (mode == kMapCluster) CHECK(bytes == mp.class_bytes[c] && bytes < (1 << 20));
      if (mode == kMapGrid) {
        const int count = mp.class_msg[c + 1] - mp.class_msg[c];
        CHECK(static_cast<int>(messages.size()) == count && count <= mp.mail_stride);
        std::vector<int> came(static_cast<size_t>(count), 0);
        for (const auto& x : messages) {
          CHECK(x.first >= mp.class_msg[c] && x.first < mp.class_msg[c + 1] && !came[x.first - mp.class_msg[c]]++);
          for (int q = 0; q < (mp.msg[x.first] & 15); ++q)
            stores.push_back({(mp.msg[x.first] >> 4) * 4 + 4 * q, spin_bytes(x.second >> (4 * q))});
        }
      }
      for (const auto& x : stores)
        for (int k = 0; k < K; ++k)
          for (int i = 0; i < 4; ++i) {
            CHECK(x.first + i < mp.map_bytes);
            maps[k][x.first + i] = static_cast<int8_t>(x.second >> (8 * i));
          }
      for (int k = 0; k < K; ++k)
        for (int p = 0; p < n; ++p) CHECK(maps[k][mp.map_index[p]] == spin[p]);
    }
    for (int k = 0; k < K; ++k) {
      CHECK(round[k] == mp.blocks[k].rounds);
      for (int x : drawn[k]) CHECK(x == 1);
    }
  }
  std::printf("ok\n");
  return 0;
}
