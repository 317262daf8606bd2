// Host plan of the spin-map engine (host_graph.h, MapPlan).
#include <algorithm>
#include <cstdint>
#include <vector>

#include "host_graph.h"

namespace isingx {

namespace {

struct Unit {
  int32_t pos;  // first position
  int32_t rows, lg, groups;
  int32_t words, row, base;  // its place in the block
  int32_t acc;  // split rows: the first row's partial sum + 1
};

// A part of a split row (host_graph.h) of block `owner`.
struct Part {
  int32_t owner, acc, row, part, groups, words;
};

}  // namespace

void build_map_plan(const HostGraph& g, int32_t mode, int32_t K, bool wide, int64_t smem_limit, MapPlan* mp,
                    bool split) {
  *mp = MapPlan();
  const int32_t C = g.num_colours;
  if (g.n < 1 || g.n > kMapMaxVertices || (!split && g.max_degree > kMapMaxDegree) || C < 1 || C > 4096 || K < 1 ||
      K > kMapMaxBlocks || (mode <= kMapBlockStream && K != 1) || (mode == kMapCluster && (K > 16 || (K & (K - 1)) != 0)) ||
      (split && mode != kMapCluster))
    return;
  // At the least a block holds the map, an id and a bias byte for its share of the
  // rows, and for every class a round of eight tasks and its tables; but for the
  // grid it has a unit in every class, padded to 32 rows of 5.25 bytes.
  const int64_t rows_bytes = std::max<int64_t>(g.n / K * int64_t(5), mode != kMapGrid ? int64_t(168) * C : 0);
  if (g.n + rows_bytes + int64_t(128 + 16) * C > smem_limit) return;
  const bool cluster = mode == kMapCluster;
  const size_t stride = static_cast<size_t>(C) + 1;
  // a unit's rows in the block's row order: whole aligned words of the map
  // where they are stored as words
  // split rows (the hubs): the entries in the class before, which its step
  // must wait for
  const int32_t hubs = split ? g.num_hubs : 0;
  mp->hubs = hubs;
  mp->late.resize(2 * static_cast<size_t>(hubs));
  for (int32_t c = 0; c < C && g.class_begin[static_cast<size_t>(c)] < hubs; ++c) {
    const size_t before = static_cast<size_t>((c + C - 1) % C);
    for (int32_t v = g.class_begin[static_cast<size_t>(c)]; v < g.class_begin[static_cast<size_t>(c) + 1]; ++v) {
      const auto b = g.col.begin() + g.row_ptr[static_cast<size_t>(v)], e = g.col.begin() + g.row_ptr[static_cast<size_t>(v) + 1];
      mp->late[2 * static_cast<size_t>(v)] = static_cast<int32_t>(std::lower_bound(b, e, g.class_begin[before]) - g.col.begin());
      mp->late[2 * static_cast<size_t>(v) + 1] = static_cast<int32_t>(std::lower_bound(b, e, g.class_begin[before + 1]) - g.col.begin());
    }
  }
  // entries that a row's unit sums, and the most of rows [v, e)
  auto length = [&](int32_t v) {
    return v < hubs ? mp->late[2 * static_cast<size_t>(v) + 1] - mp->late[2 * static_cast<size_t>(v)]
                    : g.row_ptr[static_cast<size_t>(v) + 1] - g.row_ptr[static_cast<size_t>(v)];
  };
  auto longest = [&](int32_t v, int32_t e) {
    int32_t d = length(v);
    if (v < hubs)  // the others stand in order of their length
      while (++v < e) d = std::max(d, length(v));
    return d;
  };
  auto width = [&](const Unit& u) { return cluster ? std::max(4, 32 >> u.lg) : u.rows; };
  // units, dealt to the blocks in turn over all classes
  std::vector<std::vector<Unit>> of(static_cast<size_t>(K));  // per block: its units in order
  std::vector<int32_t> first(stride * static_cast<size_t>(K), 0);  // per block and class: its first unit
  std::vector<int32_t> accs(static_cast<size_t>(K), 0);
  int64_t turn = 0;
  // entries a lane, at most l: a unit costs about its slots and four entries
  // more, whatever its rows fill, so short rows are better off with 8 than with 16
  // (a cluster's sweep at 60,000 vertices of 6 neighbours 12.4 -> 9.4 us, of 8 12.4 ->
  // 10.7; 10,000 of 20: 7.0 at 16, 8.1 at 8). The grid's steps are bound by their
  // exchange (150,000 vertices of 4: 22.3 at 16, 23.0 at 8)
  auto row_lanes = [&](int32_t d, int32_t slots) {
    int32_t lg = 0;
    while (lg < 5 && ((d + (1 << lg) - 1) >> lg) > slots) ++lg;
    return int64_t(1) << lg;
  };
  int64_t cost[2] = {0, 0};
  for (int32_t v = hubs; v < g.n; ++v)
    for (int i = 0; i < 2; ++i) cost[i] += row_lanes(length(v), kMapSlots >> i) * ((kMapSlots >> i) + 4);
  const int32_t few_slots = !split && mode != kMapGrid && cost[1] < cost[0] ? kMapSlots / 2 : kMapSlots;
  for (int32_t c = 0; c < C; ++c) {
    for (int32_t k = 0; k < K; ++k)
      first[static_cast<size_t>(k) * stride + static_cast<size_t>(c)] = static_cast<int32_t>(of[static_cast<size_t>(k)].size());
    const int32_t ve = g.class_begin[static_cast<size_t>(c) + 1];
    const int64_t first_turn = turn;
    // entries a lane: the class's units at kMapSlots against one round of every warp
    int64_t lanes = 0;
    for (int32_t v = g.class_begin[static_cast<size_t>(c)]; v < ve; ++v) lanes += row_lanes(length(v), few_slots);
    const int32_t max_slots =
        few_slots == kMapSlots && lanes > int64_t(32) * kMapMaxWarps * K ? 2 * kMapSlots : few_slots;
    // a class too small to give every block a unit uses more lanes a row
    int32_t least = 0;
    while (least < 5 && ((int64_t(ve) - g.class_begin[static_cast<size_t>(c)]) << (least + 1)) <= int64_t(32) * K) ++least;
    for (int32_t v = g.class_begin[static_cast<size_t>(c)]; v < ve;) {
      int32_t lg = 0, d = longest(v, std::min(v + 32, ve));
      while (lg < 5 && ((d + (1 << lg) - 1) >> lg) > max_slots) ++lg;
      // and so do the last rows of a class, up to four entries a lane
      while (lg < 5 && ((d + (1 << lg) - 1) >> lg) > 4 && (lg < least || (32 >> (lg + 1)) >= ve - v)) ++lg;
      const int32_t rows = std::min(32 >> lg, ve - v);
      d = longest(v, v + rows);
      const int32_t slots = (d + (1 << lg) - 1) >> lg;
      const size_t k = static_cast<size_t>(turn++ % K);
      Unit u{v, rows, lg, (slots + 3) / 4, 0, 0, 0, 0};
      if (v < hubs) {
        u.acc = accs[k] + 1;
        accs[k] += rows;
        mp->max_acc = std::max(mp->max_acc, accs[k]);
      }
      of[k].push_back(u);
      v += rows;
    }
    if (cluster)
      // every block sends something in every class: a block without a unit
      // gets one without rows (and the next class's first unit is the next
      // block's all the same)
      for (int64_t k = turn; k < first_turn + K; ++k) of[static_cast<size_t>(k % K)].push_back({0, 0, 5, 0, 0, 0, 0, 0});
  }
  for (int32_t k = 0; k < K; ++k)
    first[static_cast<size_t>(k) * stride + static_cast<size_t>(C)] = static_cast<int32_t>(of[static_cast<size_t>(k)].size());
  mp->mode = mode;
  mp->K = K;
  mp->blocks.resize(static_cast<size_t>(K));
  mp->class_row.assign(stride * static_cast<size_t>(K), 0);
  mp->class_seg.assign(stride * static_cast<size_t>(K), 0);
  mp->block_msg.assign(stride * static_cast<size_t>(K), 0);
  mp->class_bytes.assign(stride, 0);
  mp->class_msg.assign(stride, 0);
  mp->map_index.assign(static_cast<size_t>(g.n), 0);
  // the blocks' rows and entries
  std::vector<std::vector<Part>> parts(hubs > 0 ? static_cast<size_t>(K) * static_cast<size_t>(C) : 0);  // by the class whose step sums them
  int32_t row0 = 0, widest = 1;
  int64_t words0 = 0;
  for (int32_t k = 0; k < K; ++k) {
    MapBlock& b = mp->blocks[static_cast<size_t>(k)];
    b.row0 = row0;
    int32_t row = 0, groups = 0;
    for (int32_t c = 0; c < C; ++c) {
      const size_t t = static_cast<size_t>(k) * stride + static_cast<size_t>(c);
      row = (row + 31) & ~31;
      mp->class_row[t] = row;
      widest = std::max(widest, first[t + 1] - first[t]);
      for (int32_t i = first[t]; i < first[t + 1]; ++i) {
        Unit& u = of[static_cast<size_t>(k)][static_cast<size_t>(i)];
        if (cluster) {
          row = (row + width(u) - 1) & ~(width(u) - 1);
          mp->class_bytes[static_cast<size_t>(c)] += width(u);
        }
        u.words = groups;
        u.row = row;
        groups += u.groups;
        mp->stage = std::max(mp->stage, u.groups);
        row += width(u);
      }
    }
    row = (row + 31) & ~31;
    mp->class_row[static_cast<size_t>(k) * stride + static_cast<size_t>(C)] = row;
    b.rows = row;
    b.groups = groups;
    row0 += row;
    mp->max_rows = std::max(mp->max_rows, b.rows);
  }
  // the parts of class c's rows, each to the block with the fewest tasks in
  // the step of the class before; the row's block waits for their bytes
  std::vector<int32_t> received(hubs > 0 ? stride * static_cast<size_t>(K) : 0, 0);
  for (int32_t c = 0; c < C && hubs > 0; ++c) {
    const size_t at = static_cast<size_t>((c + C - 1) % C);
    std::vector<int32_t> busy(static_cast<size_t>(K));
    for (int32_t k = 0; k < K; ++k) {
      const size_t t = static_cast<size_t>(k) * stride + at;
      busy[static_cast<size_t>(k)] = first[t + 1] - first[t];
    }
    for (int32_t k = 0; k < K; ++k) {
      const size_t t = static_cast<size_t>(k) * stride + static_cast<size_t>(c);
      for (int32_t i = first[t]; i < first[t + 1]; ++i) {
        const Unit& u = of[static_cast<size_t>(k)][static_cast<size_t>(i)];
        for (int32_t r = 0; u.acc != 0 && r < u.rows; ++r) {
          const size_t v = static_cast<size_t>(u.pos + r);
          const int32_t early = g.row_ptr[v + 1] - g.row_ptr[v] - length(u.pos + r);
          for (int32_t p = 0; p * kMapPartEntries < early; ++p) {
            const size_t to = static_cast<size_t>(std::min_element(busy.begin(), busy.end()) - busy.begin());
            const int32_t gr = (std::min(kMapPartEntries, early - p * kMapPartEntries) + 127) / 128;
            parts[to * static_cast<size_t>(C) + at].push_back({k, u.acc - 1 + r, u.row + r, p, gr, mp->blocks[to].groups});
            mp->blocks[to].groups += gr;
            mp->stage = std::max(mp->stage, gr);
            widest = std::max(widest, ++busy[to]);
            received[static_cast<size_t>(k) * stride + at] += 4;
          }
        }
      }
    }
  }
  for (MapBlock& b : mp->blocks) {
    b.words0 = static_cast<int32_t>(std::min<int64_t>(words0, 1 << 24));
    words0 += b.groups;
    mp->max_groups = std::max(mp->max_groups, b.groups);
  }
  if (mp->max_acc > kMapMaxSplit || g.max_degree / kMapPartEntries > kMapMaxSplit) return;
  if (words0 >= (int64_t(1) << 24) || mp->max_rows / 32 >= (1 << (32 - kMapFlipShift - 1)) - 1) return;
  // the map: class by class, block by block, a segment for a block's rows of
  // the class
  int64_t at = 0;
  for (int32_t c = 0; c < C; ++c) {
    for (int32_t k = 0; k < K; ++k) {
      const size_t t = static_cast<size_t>(k) * stride + static_cast<size_t>(c);
      std::vector<Unit>& mine = of[static_cast<size_t>(k)];
      int32_t len = 0;
      if (first[t + 1] > first[t]) {
        const Unit& last = mine[static_cast<size_t>(first[t + 1]) - 1];
        len = last.row + width(last) - mp->class_row[t];
      }
      const int32_t align = cluster ? 32 : 4;
      at = (at + align - 1) & ~int64_t(align - 1);
      mp->class_seg[t] = static_cast<int32_t>(at);
      mp->block_msg[t] = static_cast<int32_t>(mp->msg.size());
      if (mode == kMapGrid && len == 0) mp->msg.push_back(0);
      if (mode == kMapGrid)
        for (int32_t r = 0; r < len; r += 32)
          mp->msg.push_back(static_cast<int32_t>((at + r) / 4 << 4) | ((std::min(32, len - r) + 3) / 4));
      for (int32_t i = first[t]; i < first[t + 1]; ++i) {
        Unit& u = mine[static_cast<size_t>(i)];
        u.base = static_cast<int32_t>(at) + u.row - mp->class_row[t];
        for (int32_t r = 0; r < u.rows; ++r) mp->map_index[static_cast<size_t>(u.pos + r)] = u.base + r;
      }
      at += len;
      if (at > smem_limit || at >= (1 << kMapFlipShift)) return;
    }
    mp->class_msg[static_cast<size_t>(c) + 1] = static_cast<int32_t>(mp->msg.size());
    mp->mail_stride = std::max(mp->mail_stride, mp->class_msg[static_cast<size_t>(c) + 1] - mp->class_msg[static_cast<size_t>(c)]);
  }
  for (int32_t k = 0; k < K; ++k)
    mp->block_msg[static_cast<size_t>(k) * stride + static_cast<size_t>(C)] = static_cast<int32_t>(mp->msg.size());
  if (hubs > 0) mp->block_msg = received;
  mp->map_bytes = static_cast<int32_t>((at + 32 + 15) & ~int64_t(15));
  // the tasks; as many warps as the largest class has units and draws
  const int32_t class_draws = (mp->max_rows / 32 + C - 1) / C;
  const int32_t warps = std::min(kMapMaxWarps, std::max(8, (widest + class_draws + 3) / 4 * 4));
  mp->warps = warps;
  for (int32_t k = 0; k < K; ++k) {
    MapBlock& b = mp->blocks[static_cast<size_t>(k)];
    const std::vector<Unit>& mine = of[static_cast<size_t>(k)];
    b.task0 = static_cast<int32_t>(mp->tasks.size());
    for (int32_t c = 0; c < C; ++c) {
      const size_t t = static_cast<size_t>(k) * stride + static_cast<size_t>(c);
      static const std::vector<Part> none;
      const std::vector<Part>& early = hubs > 0 ? parts[static_cast<size_t>(k) * static_cast<size_t>(C) + static_cast<size_t>(c)] : none;
      const int32_t units = first[t + 1] - first[t];
      const int32_t rounds = std::max(1, (units + static_cast<int32_t>(early.size()) + warps - 1) / warps);
      if (c == C - 1) b.last0 = static_cast<int32_t>(mp->tasks.size()) - b.task0;
      for (int32_t i = 0; i < rounds * warps; ++i) {
        MapTask x{0, 0, 0, 0};
        if (i < units) {
          const Unit& u = mine[static_cast<size_t>(first[t] + i)];
          x = {u.words, u.base, u.row | (u.acc << kMapSplitShift), u.rows | (u.lg << 8) | (u.groups << 16)};
        } else if (i - units < static_cast<int32_t>(early.size())) {
          const Part& p = early[static_cast<size_t>(i - units)];
          x = {p.words, p.acc | (p.owner << kMapOwnerShift), p.row | (p.part << kMapSplitShift), (kMapPart << 8) | (p.groups << 16)};
        }
        if (i >= (rounds - 1) * warps) x.row |= static_cast<int32_t>(0x80000000u);
        mp->tasks.push_back(x);
      }
    }
    // the draws: one to every task without a unit, then one to every task,
    // then rounds of their own before the end of the last class
    const int32_t draws = b.rows / 32;
    int32_t j = 0;
    for (int pass = 0; pass < 2; ++pass)
      for (size_t i = static_cast<size_t>(b.task0); i < mp->tasks.size() && j < draws; ++i) {
        MapTask& x = mp->tasks[i];
        if ((x.base >> kMapFlipShift) != 0 || (pass == 0 && x.shape != 0)) continue;
        x.base |= (++j) << kMapFlipShift;
      }
    if (j < draws)
      for (size_t i = mp->tasks.size() - static_cast<size_t>(warps); i < mp->tasks.size(); ++i)
        mp->tasks[i].row &= 0x7fffffff;
    while (j < draws) {
      const bool last = draws - j <= warps;
      for (int32_t w = 0; w < warps; ++w) {
        MapTask x{0, 0, last ? static_cast<int32_t>(0x80000000u) : 0, 0};
        if (j < draws) x.base = (++j) << kMapFlipShift;
        mp->tasks.push_back(x);
      }
    }
    b.rounds = (static_cast<int32_t>(mp->tasks.size()) - b.task0) / warps;
    mp->max_tasks = std::max(mp->max_tasks, b.rounds * warps);
  }
  const int64_t entries = int64_t(mp->max_groups) * (wide ? 2 : 1);
  int64_t smem = map_smem_bytes(mp->map_bytes, 0, mp->max_tasks, C, mp->max_rows, mp->max_acc);
  mp->resident = mode == kMapBlock || (cluster && smem + entries * 512 <= smem_limit);
  if (mp->resident) smem += entries * 512;
  if (smem > smem_limit) return;
  mp->smem_bytes = static_cast<int32_t>(smem);
  // rows
  mp->row_pos.assign(static_cast<size_t>(row0), -1);
  mp->row_orig.assign(static_cast<size_t>(row0), -1);
  for (int32_t k = 0; k < K; ++k)
    for (const Unit& u : of[static_cast<size_t>(k)])
      for (int32_t r = 0; r < u.rows; ++r) {
        const size_t at = static_cast<size_t>(mp->blocks[static_cast<size_t>(k)].row0 + u.row + r);
        mp->row_pos[at] = u.pos + r;
        mp->row_orig[at] = g.perm[static_cast<size_t>(u.pos + r)];
      }
  mp->total_groups = words0;
  mp->ok = true;
}

}  // namespace isingx
