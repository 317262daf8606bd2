// Host tables of the clustered batch kernel (batch_map.cuh).
#pragma once

#include <cstdint>
#include <vector>

namespace isingx {

constexpr int kBatchMapThreads = 512;
// Warps that run units; the other four draw. Microseconds a sweep with 8 / 10 /
// 12 / 14: 42.1 / 41.8 / 39.8 / 41.4 for 320 instances (eight replicas, +-1
// weights), 53.1 / 49.3 / 50.8 / 51.7 (weights up to 8), 14.1 / 13.0 / 12.4 / 12.2
// for 60 instances (four replicas).
constexpr int kBatchMapUnitWarps = 12;
constexpr int kBatchMapDegree = 63;  // six bit planes
constexpr int kBatchMapStage = 3;    // groups of four entries a lane loads a class ahead

// 32 rows of one colour class, one a lane; a row's entries are `groups` int4
// of its lane, (map index << 8) | (w & 0xff), padded with index 0 and weight 0
// (the map's first 32 bytes stay zero).
struct BatchMapUnit {
  int32_t words;  // first group (of 32 int4) of the unit
  int32_t base;   // map index of its first row (a multiple of 32)
  int32_t pos;    // its first row's position within the instance
  int32_t shape;  // rows | groups << 16
};

struct BatchMapInst {
  int32_t id, n, classes;
  int32_t vtx_base;      // its first byte of the batch's spins
  int32_t row0;          // its first entry of row_sum and map_index
  int32_t unit0;         // K + 1 first units of the blocks: block_unit[unit0 + k]
  int32_t class_unit0;   // K x (classes + 1): a block's first unit of every class, from its own first
  int32_t class_bytes0;  // classes: bytes a block receives
  int32_t dst0;          // 128 * ceil(n / 128) entries: the place of every vertex's flip byte
  int32_t flush;         // weighted rows: groups a byte lane can add up
};

// An instance's rows, by position (class by class, by decreasing degree).
struct BatchMapRows {
  int32_t id = 0, vtx_base = 0;
  std::vector<int32_t> class_begin, degree, wsum, perm;
};

struct BatchMapPlan {
  int K = 1;
  bool unit = false;
  int32_t map_bytes = 0, units_max = 0, classes_max = 0, smem = 0;
  int64_t groups = 0;
  std::vector<BatchMapInst> inst;
  std::vector<BatchMapUnit> units;
  std::vector<int32_t> unit_inst;    // per unit: its instance
  std::vector<int32_t> block_unit, class_unit, class_bytes;
  std::vector<int32_t> dst;          // by vertex id: block << 24 | flip slot, -1 past the last
  std::vector<int32_t> row_sum;      // by position: degree (unit) or weight sum
  std::vector<int32_t> map_index;    // by position
};

// Shared memory of a block: the map, two sweeps of flip bytes (32 per unit),
// the units, two class tables, two sweeps of replica starts (256 bytes), and
// 64 bytes of barriers and counters.
constexpr int32_t batch_map_smem(int32_t map_bytes, int32_t units, int32_t classes) {
  return map_bytes + 64 * units + 16 * units + 8 * ((classes + 4) / 4 * 4) + 256 + 64;
}

// Blocks per instance, a power of two up to 16: as many as give a block its
// share of the vertices of all instances when they run side by side, two
// blocks an SM, but not below kBatchMapShare vertices a block. Microseconds a
// sweep (eight replicas, +-1 weights) of 16 instances of 300 to 20,000 vertices
// at 500 / 1000 / 1500 / 2500 / 4000 vertices: 12.2 / 12.3 / 14.2 / 16.9 / 25.6; of
// 320 instances: 42.7 / 39.1 / 41.6 / 42.9 / 41.2, and 65 at twice the share.
constexpr int64_t kBatchMapShare = 1000;
int batch_map_blocks(int64_t n, int64_t total, int num_sms);

// Tables for K blocks an instance. unit: every weight is +-1; wmax: the largest
// |weight|, at most 31. False if an instance does not fit in smem_limit bytes.
bool build_batch_map(const std::vector<const BatchMapRows*>& rows, bool unit, int32_t wmax, int K, int64_t smem_limit,
                     BatchMapPlan* out);

}  // namespace isingx
