// Host tables of the clustered batch kernel (batch_map_plan.h).
#include "batch_map_plan.h"

#include <algorithm>

namespace isingx {

int batch_map_blocks(int64_t n, int64_t total, int num_sms) {
  const int64_t share = std::max<int64_t>(kBatchMapShare, total / (2 * std::max(num_sms, 1)));
  int K = 1;
  while (K < 16 && n > share * K * 3 / 2) K *= 2;
  return K;
}

bool build_batch_map(const std::vector<const BatchMapRows*>& rows, bool unit, int32_t wmax, int K, int64_t smem_limit,
                     BatchMapPlan* out) {
  BatchMapPlan& p = *out;
  p = BatchMapPlan();
  p.K = K;
  p.unit = unit;
  const size_t blocks = static_cast<size_t>(K);
  for (size_t gi = 0; gi < rows.size(); ++gi) {
    const BatchMapRows& r = *rows[gi];
    const int32_t n = static_cast<int32_t>(r.degree.size()), C = static_cast<int32_t>(r.class_begin.size()) - 1;
    const size_t stride = static_cast<size_t>(C) + 1;
    p.inst.push_back({r.id, n, C, r.vtx_base, static_cast<int32_t>(p.row_sum.size()), static_cast<int32_t>(p.block_unit.size()),
                      static_cast<int32_t>(p.class_unit.size()), static_cast<int32_t>(p.class_bytes.size()),
                      static_cast<int32_t>(p.dst.size()), std::max(1, 127 / (4 * std::max(wmax, 1)))});
    const std::vector<int32_t>& sum = unit ? r.degree : r.wsum;
    const size_t first_row = p.row_sum.size();
    p.row_sum.insert(p.row_sum.end(), sum.begin(), sum.end());
    p.map_index.resize(first_row + static_cast<size_t>(n));
    std::vector<std::vector<BatchMapUnit>> of(blocks);
    std::vector<int32_t> first(blocks * stride, 0);
    std::vector<int32_t> place(static_cast<size_t>(n));  // by position: block << 24 | flip slot
    int64_t at = 32, turn = 0;
    for (int32_t c = 0; c < C; ++c) {
      for (size_t k = 0; k < blocks; ++k) first[k * stride + static_cast<size_t>(c)] = static_cast<int32_t>(of[k].size());
      const int64_t first_turn = turn;
      const int32_t end = r.class_begin[static_cast<size_t>(c) + 1];
      // dealt to the blocks in turn; in a cluster every block has a unit in
      // every class (without rows if need be), so that all of them send
      for (int32_t v = r.class_begin[static_cast<size_t>(c)]; v < end || (K > 1 && turn < first_turn + K); ++turn) {
        const size_t k = static_cast<size_t>(turn % K);
        const int32_t count = std::min(32, end - v);
        const int32_t groups = count > 0 ? (r.degree[static_cast<size_t>(v)] + 3) / 4 : 0;
        for (int32_t i = 0; i < count; ++i) {
          p.map_index[first_row + static_cast<size_t>(v + i)] = static_cast<int32_t>(at) + i;
          place[static_cast<size_t>(v + i)] = static_cast<int32_t>(k << 24) | (32 * static_cast<int32_t>(of[k].size()) + i);
        }
        of[k].push_back({static_cast<int32_t>(p.groups), static_cast<int32_t>(at), v, count | (groups << 16)});
        p.groups += groups;
        at += 32;
        v += count;
      }
      p.class_bytes.push_back(static_cast<int32_t>(32 * (turn - first_turn)));
    }
    for (size_t k = 0; k < blocks; ++k) {
      first[k * stride + static_cast<size_t>(C)] = static_cast<int32_t>(of[k].size());
      p.block_unit.push_back(static_cast<int32_t>(p.units.size()));
      p.units.insert(p.units.end(), of[k].begin(), of[k].end());
      p.units_max = std::max(p.units_max, static_cast<int32_t>(of[k].size()));
    }
    p.block_unit.push_back(static_cast<int32_t>(p.units.size()));
    p.unit_inst.resize(p.units.size(), static_cast<int32_t>(gi));
    p.class_unit.insert(p.class_unit.end(), first.begin(), first.end());
    const size_t d0 = p.dst.size();
    p.dst.resize(d0 + (static_cast<size_t>(n) + 127) / 128 * 128, -1);
    for (int32_t v = 0; v < n; ++v)
      p.dst[d0 + static_cast<size_t>(r.perm[static_cast<size_t>(v)])] = place[static_cast<size_t>(v)];
    p.classes_max = std::max(p.classes_max, C);
    if (at > smem_limit || p.groups >= (int64_t(1) << 30) || p.dst.size() >= (size_t(1) << 30)) return false;
    p.map_bytes = std::max(p.map_bytes, static_cast<int32_t>(at));
    // st.async counts a class's bytes on one mbarrier phase
    for (size_t i = p.class_bytes.size() - static_cast<size_t>(C); i < p.class_bytes.size(); ++i)
      if (p.class_bytes[i] >= (1 << 20)) return false;
  }
  p.smem = batch_map_smem(p.map_bytes, p.units_max, p.classes_max);
  return p.smem <= smem_limit;
}

}  // namespace isingx
