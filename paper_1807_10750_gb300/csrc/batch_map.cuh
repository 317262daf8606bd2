// Batched anneals, the clustered form: an instance on one block or on the
// blocks of a cluster, for batches whose rows have at most kBatchMapDegree
// entries and weights of at most 31.
//
// What bounds a batch is its largest instance: eight replicas of 20,000
// vertices are 40,000 Philox evaluations and 200,000 row entries a sweep, most
// of it instruction issue. So an instance gets as many SMs as the batch leaves
// it (batch_map_blocks picks the cluster; one launch per cluster size, side by side), every block of the cluster keeps the
// replica bytes of all of the instance's vertices in shared memory, and a class
// ends with the exchange of the map engine (map.cuh): st.async of the new
// bytes to every block, counted on the destination's mbarrier.
//   * A lane sums a row. With weights of +-1 the eight replicas are counted in
//     bit planes: a neighbour's byte, inverted under a negative weight, enters
//     a carry-save adder (about 3 logic instructions an entry for all replicas),
//     and the planes are compared with half the row's degree. Other weights
//     multiply the byte spread over eight byte lanes, which hold signed sums up
//     to 127 and are moved to integers before they could exceed it.
//   * The next sweep's flips are drawn beside the classes, by warps of their own
//     (a class would otherwise end with whoever started a draw last) that take
//     chunks of 32 quads from a counter: a lane evaluates its quad's replicas two
//     at a time (independent chains, shared round keys) and stores four flip
//     bytes in the block that owns each vertex; a cluster barrier ends every
//     sweep. (One evaluation per lane and replica, with votes to collect the
//     bits, took 180 instructions for 16 vertices; this takes 430 for 128.)
// Microseconds a sweep on GB300, eight replicas, against the one-block kernel
// with its default tuning (and its best): 320 instances of 500 to 20,000
// vertices, mean degree 10, +-1 weights 149 (116) -> 40, weights up to 8 156
// (125) -> 51; 16 instances 120 (80) -> 12; 1024 instances 130 -> 88 (autotuned).
//
// Every wait is bounded; after a failed one the warps run on without stores,
// arrivals or waits through the remaining barriers, and the host reports it.
#pragma once

#include <cstdint>

#include "batch_map_plan.h"
#include "cluster.cuh"

namespace isingx {

constexpr int kBatchMapWarps = kBatchMapThreads / 32;

struct BatchMapArgs {
  const BatchMapInst* inst;  // by decreasing size
  const int32_t* block_unit;
  const int4* units;     // BatchMapUnit
  const int32_t* class_unit;
  const int32_t* class_bytes;
  const int32_t* dst;    // by vertex id: block << 24 | flip slot, -1 past the last vertex
  const int32_t* row_sum;  // by position: the row's degree (+-1 weights) or weight sum
  const int32_t* map_index;  // by position
  const int4* words;
  uint8_t* spins;        // replica bits by position
  unsigned* work;        // the next instance
  int* error;
  int32_t num_graphs, K, replicas;
  int32_t map_bytes, units_max, classes_max;  // of the largest instance
  long long budget;
};

// All ones if the low byte of x is negative, else 0.
__device__ __forceinline__ uint32_t sign_bytes(uint32_t x) {
  uint32_t r;
  asm("prmt.b32 %0, %1, 0, 0x8888;" : "=r"(r) : "r"(x));
  return r;
}

// Six-plane counter of replica bytes, started at 32 less half the row's
// degree: plane 5 then tells whether half of the products are negative. A row
// has at most 63 entries, so the count stays below 64.
struct PlaneCount {
  uint32_t c[6];
  __device__ __forceinline__ void start(int degree) {
    const int first = 32 - ((degree + 1) >> 1);
#pragma unroll
    for (int i = 0; i < 6; ++i)
      c[i] = static_cast<uint32_t>(static_cast<int32_t>(static_cast<uint32_t>(first) << (31 - i)) >> 31);
  }
  // a + b + d -> sum, returns the carry
  static __device__ __forceinline__ uint32_t full(uint32_t& sum, uint32_t a, uint32_t b, uint32_t d) {
    const uint32_t carry = (a & b) | (d & (a ^ b));
    sum = a ^ b ^ d;
    return carry;
  }
  __device__ __forceinline__ void add4(uint32_t x0, uint32_t x1, uint32_t x2, uint32_t x3) {
    const uint32_t p = full(c[0], c[0], x0, x1), q = full(c[0], c[0], x2, x3);
    uint32_t carry = full(c[1], c[1], p, q);
#pragma unroll
    for (int i = 2; i < 6; ++i) {
      const uint32_t next = c[i] & carry;
      c[i] ^= carry;
      carry = next;
    }
  }
  // The new replica byte: with f = degree - 2 * (negative products), f > 0
  // (plane 5 clear) gives 1 (spin -1), f = 0 (the count is 32, the degree even)
  // keeps the old bit.
  __device__ __forceinline__ uint32_t decide(int degree, uint32_t old) const {
    const uint32_t past = c[0] | c[1] | c[2] | c[3] | c[4];
    const uint32_t keep = (degree & 1) ? 0u : old;
    return ~c[5] | (~past & keep);
  }
};

// Signed sums of eight replicas in byte lanes, moved to integers by `flush`.
struct LaneSums {
  int lo, hi, acc[8];
  __device__ __forceinline__ void clear() {
    lo = hi = 0;
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = 0;
  }
  __device__ __forceinline__ void add(uint32_t byte, int w) {
    lo += static_cast<int>(((byte & 15u) * 0x00204081u) & 0x01010101u) * w;
    hi += static_cast<int>(((byte >> 4) * 0x00204081u) & 0x01010101u) * w;
  }
  // the lanes are the signed base-256 digits of lo and hi
  __device__ __forceinline__ void flush() {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int a = static_cast<int8_t>(lo), b = static_cast<int8_t>(hi);
      acc[k] += a;
      acc[k + 4] += b;
      lo = (lo - a) >> 8;
      hi = (hi - b) >> 8;
    }
  }
  // f = wsum - 2 acc, acc the weights of the neighbours with spin -1
  __device__ __forceinline__ uint32_t decide(int wsum, uint32_t old) const {
    uint32_t out = 0u;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int f = wsum - 2 * acc[k];
      out |= static_cast<uint32_t>(f + static_cast<int>((old >> k) & 1u) > 0) << k;
    }
    return out;
  }
};

// Philox4x32-10 (batch.cu's batch_philox) with counter (q, t, r, 0). Its first
// two rounds multiply q and words of the second round that q alone determines,
// and r and words that (r, t) alone determine: the former serve all replicas of
// a quad, the latter all quads of a sweep.
struct QuadStart {  // by quad: x1 after two rounds, and what enters x0 and x2
  uint32_t x1, hi, x3;
};
__device__ __forceinline__ QuadStart batch_quad_start(uint32_t q, uint32_t kb) {
  const uint64_t p = static_cast<uint64_t>(0xD2511F53u) * q;
  const uint64_t s = static_cast<uint64_t>(0xCD9E8D57u) * (static_cast<uint32_t>(p >> 32) ^ kb);
  return {static_cast<uint32_t>(s), static_cast<uint32_t>(s >> 32), static_cast<uint32_t>(p)};
}
// By replica and sweep: (what enters x0, what enters x2, x3 after two rounds).
__device__ __forceinline__ uint4 batch_replica_start(uint32_t r, uint32_t t, uint32_t ka, uint32_t kb) {
  const uint64_t p = static_cast<uint64_t>(0xCD9E8D57u) * r;
  const uint64_t s = static_cast<uint64_t>(0xD2511F53u) * (static_cast<uint32_t>(p >> 32) ^ t ^ ka);
  return make_uint4(static_cast<uint32_t>(p) ^ (ka + 0x9E3779B9u), static_cast<uint32_t>(s >> 32) ^ (kb + 0xBB67AE85u),
                    static_cast<uint32_t>(s), 0u);
}

// The flips of replicas r and r + 1 (starts s[0], s[1]) of a quad: byte k holds
// bits r and r + 1 of vertex k.
__device__ __forceinline__ uint32_t batch_map_flips(const QuadStart& u, const uint4* s, uint32_t r, uint32_t ka,
                                                    uint32_t kb, uint32_t limit) {
  uint32_t x0[2], x1[2], x2[2], x3[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const uint4 v = s[j];
    x0[j] = u.hi ^ v.x;
    x1[j] = u.x1;
    x2[j] = v.y ^ u.x3;
    x3[j] = v.z;
  }
#pragma unroll
  for (int i = 2; i < 10; ++i) {
    const uint32_t a = ka + static_cast<uint32_t>(i) * 0x9E3779B9u, b = kb + static_cast<uint32_t>(i) * 0xBB67AE85u;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const uint64_t pa = static_cast<uint64_t>(0xD2511F53u) * x0[j];
      const uint64_t pb = static_cast<uint64_t>(0xCD9E8D57u) * x2[j];
      const uint32_t n0 = static_cast<uint32_t>(pb >> 32) ^ x1[j] ^ a;
      const uint32_t n2 = static_cast<uint32_t>(pa >> 32) ^ x3[j] ^ b;
      x1[j] = static_cast<uint32_t>(pb);
      x3[j] = static_cast<uint32_t>(pa);
      x0[j] = n0;
      x2[j] = n2;
    }
  }
  uint32_t out = 0u;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    if (x0[j] < limit) out |= 0x00000001u << j;
    if (x1[j] < limit) out |= 0x00000100u << j;
    if (x2[j] < limit) out |= 0x00010000u << j;
    if (x3[j] < limit) out |= 0x01000000u << j;
  }
  return out << r;
}

template <bool CLUSTER, bool UNIT>
__global__ void __launch_bounds__(kBatchMapThreads, 2)
    batch_map_kernel(BatchMapArgs a, uint64_t t_begin, uint32_t sweeps, uint64_t T, uint64_t T0, uint32_t seed_lo,
                     uint32_t seed_hi) {
  extern __shared__ __align__(128) unsigned char batch_mem[];
  constexpr int G = kBatchMapStage;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K = CLUSTER ? a.K : 1;
  constexpr int U = kBatchMapUnitWarps;  // warps 0 .. U - 1 run units, the others draw
  const int k_me = CLUSTER ? static_cast<int>(blockIdx.x) & (K - 1) : 0;
  uint8_t* map = batch_mem;
  uint8_t* flips = map + a.map_bytes;  // [sweep parity][32 units_max]
  int4* units = reinterpret_cast<int4*>(flips + 64 * a.units_max);
  int32_t* cunit = reinterpret_cast<int32_t*>(units + a.units_max);
  int32_t* cbytes = cunit + (a.classes_max + 4) / 4 * 4;  // bytes the block receives in a class
  uint4* starts = reinterpret_cast<uint4*>(cbytes + (a.classes_max + 4) / 4 * 4);  // [sweep parity][replica]
  uint64_t* bars = reinterpret_cast<uint64_t*>(starts + 16);
  unsigned* drawn = reinterpret_cast<unsigned*>(bars + 2);  // chunks taken so far
  int* slot_now = reinterpret_cast<int*>(drawn + 1);
  const uint32_t bar = smem_u32(bars);
  const uint32_t dst_lane = lane & 3;
  if (CLUSTER) {
    if (tid == 0) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(U) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar + 8), "r"(U) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    cluster_sync();
  }
  // Draws: a quad's replicas, two a pass, on one lane, or in a cluster on one
  // to four lanes, which splits the draws finely enough for the short classes of
  // its blocks.
  const int plog = !CLUSTER || a.replicas <= 2 ? 0 : (a.replicas <= 4 ? 1 : 2);
  const int pair_lanes = 1 << plog, per_chunk = 128 >> plog;
  bool ok = true;
  uint32_t step = 0;
  for (;;) {
    // the next instance, for every block of the cluster
    if (k_me == 0 && tid < K) {
      int s = 0;
      if (tid == 0) s = static_cast<int>(atomicAdd(a.work, 1u));
      s = __shfl_sync(K >= 32 ? kFullMask : ((1u << K) - 1u), s, 0);
      if (CLUSTER)
        asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(cluster_addr(smem_u32(slot_now), tid)), "r"(s) : "memory");
      else
        *slot_now = s;
    }
    if (CLUSTER)
      cluster_sync();
    else
      __syncthreads();
    const int slot = *slot_now;
    if (slot >= a.num_graphs) break;
    const BatchMapInst I = a.inst[slot];
    const int u0 = __ldg(a.block_unit + I.unit0 + k_me), nunits = __ldg(a.block_unit + I.unit0 + k_me + 1) - u0;
    const uint32_t ka = seed_lo, kb = seed_hi ^ (static_cast<uint32_t>(I.id) * 0x9E3779B9u);
    const int32_t* dst = a.dst + I.dst0;
    const int32_t* row_sum = a.row_sum + I.row0;
    // zero first: padding entries read a byte that stays zero
    for (int i = tid; i < a.map_bytes / 4; i += kBatchMapThreads) reinterpret_cast<uint32_t*>(map)[i] = 0u;
    for (int i = tid; i < nunits; i += kBatchMapThreads) units[i] = __ldg(a.units + u0 + i);
    for (int c = tid; c <= I.classes; c += kBatchMapThreads)
      cunit[c] = __ldg(a.class_unit + I.class_unit0 + k_me * (I.classes + 1) + c);
    if (tid == 0) *drawn = 0u;
    __syncthreads();
    for (int p = tid; p < I.n; p += kBatchMapThreads) map[__ldg(a.map_index + I.row0 + p)] = a.spins[I.vtx_base + p];
    // this block's chunks of 32 / pair_lanes quads: every K-th
    const int chunks = (I.n + per_chunk - 1) / per_chunk;
    const unsigned mine = static_cast<unsigned>((chunks - k_me + K - 1) / K);
    for (int c = tid; c < I.classes; c += kBatchMapThreads) cbytes[c] = __ldg(a.class_bytes + I.class_bytes0 + c);
    // the replica starts of the first two sweeps' draws
    if (tid < 16)
      starts[tid] = batch_replica_start(tid & 7, static_cast<uint32_t>(t_begin) + (tid >> 3), ka, kb);
    __syncthreads();
    uint64_t thr = 0, rem = 0;
    const uint64_t D = T > 1 ? T - 1 : 1, thr_step = T0 / D, rem_step = T0 % D;
    if (T > 1) {
      thr = T0 * (D - t_begin) / D;
      rem = T0 * (D - t_begin) % D;
    }
    auto draw = [&](unsigned j, uint32_t limit, int buffer) {
      const int q = static_cast<int>(j * K + k_me) * (32 >> plog) + (lane >> plog);
      const int pair = lane & (pair_lanes - 1);
      const int4 to = __ldg(reinterpret_cast<const int4*>(dst) + q);
      uint32_t bits = 0u;
      const QuadStart u = batch_quad_start(static_cast<uint32_t>(q), kb);
      for (int r = 2 * pair; r < a.replicas; r += 2 * pair_lanes)
        bits |= batch_map_flips(u, starts + 8 * buffer + r, static_cast<uint32_t>(r), ka, kb, limit);
      if (CLUSTER) {
        if (plog > 0) bits |= __shfl_xor_sync(kFullMask, bits, 1);
        if (plog > 1) bits |= __shfl_xor_sync(kFullMask, bits, 2);
      }
      const uint32_t at = smem_u32(flips + buffer * 32 * a.units_max);
      auto put = [&](int place, uint32_t byte) {
        if (place < 0) return;
        const uint32_t p = at + (place & 0xffffff);
        if (CLUSTER) {
          if (ok)
            asm volatile("st.shared::cluster.u8 [%0], %1;" ::"r"(cluster_addr(p, place >> 24)), "r"(byte) : "memory");
        } else {
          asm volatile("st.shared.u8 [%0], %1;" ::"r"(p), "r"(byte) : "memory");
        }
      };
      // the lanes of a quad share its four bytes
      if (pair == 0) put(to.x, bits & 0xffu);
      if (pair == (1 & (pair_lanes - 1))) put(to.y, (bits >> 8) & 0xffu);
      if (pair == (2 & (pair_lanes - 1))) put(to.z, (bits >> 16) & 0xffu);
      if (pair == (3 & (pair_lanes - 1))) put(to.w, bits >> 24);
    };
    if (thr != 0)
      for (unsigned j = warp; j < mine; j += kBatchMapWarps)
        draw(j, static_cast<uint32_t>(thr), 0);
    // the warp's next unit: its first entries and its rows' sums
    int4 nw[G];
    int4 nu = make_int4(0, 0, 0, 0);
    int nsum = 0;
    auto stage = [&](int i, int end) {
      if (i >= end) return;
      nu = units[i];
      const int4* p = a.words + static_cast<size_t>(nu.x) * 32 + lane;
      const int groups = nu.w >> 16;
      if (lane < (nu.w & 0xffff)) nsum = __ldg(row_sum + nu.z + lane);
#pragma unroll
      for (int g = 0; g < G; ++g)
        if (g < groups) nw[g] = __ldg(p + g * 32);
    };
    if (warp < U) stage(cunit[0] + warp, cunit[1]);
    const uint32_t replica_mask = (1u << a.replicas) - 1u;
    if (CLUSTER)
      cluster_sync();
    else
      __syncthreads();
    unsigned taken = 0;  // the warp's next chunk, counted over the sweeps
    if (lane == 0) taken = atomicAdd(drawn, 1u);
    taken = __shfl_sync(kFullMask, taken, 0);
    for (uint32_t k = 0; k < sweeps; ++k) {
      const bool flip_now = thr != 0;
      const uint8_t* flip = flips + (k & 1u) * 32 * a.units_max;
      if (T > 1 && k + 1 < sweeps) {
        thr -= thr_step;
        if (rem < rem_step) {
          rem += D - rem_step;
          --thr;
        } else {
          rem -= rem_step;
        }
      }
      // sweep k + 2's replica starts, in the buffer that sweep k's draws used
      if (tid >= kBatchMapThreads - 8)
        starts[8 * (k & 1u) + (tid & 7)] = batch_replica_start(tid & 7, static_cast<uint32_t>(t_begin) + k + 2, ka, kb);
      for (int c = warp < U ? 0 : I.classes; c < I.classes; ++c, ++step) {
        const int ue = cunit[c + 1], cn = c + 1 < I.classes ? c + 1 : 0;
        for (int i = cunit[c] + warp; i < ue; i += U) {
          const int4 u = nu;
          const int sum = nsum;
          int4 w[G];
#pragma unroll
          for (int g = 0; g < G; ++g) w[g] = nw[g];
          if (i + U < ue)
            stage(i + U, ue);
          else
            stage(cunit[cn] + warp, cunit[cn + 1]);
          // 1. the row of this lane
          const int rows = u.w & 0xffff, groups = u.w >> 16;
          const uint32_t old = map[u.y + lane];
          const uint32_t fl = flip_now ? flip[32 * i + lane] : 0u;
          uint32_t nb;
          if (UNIT) {
            PlaneCount n;
            n.start(sum);
            auto add = [&](const int4& e) {
              const uint32_t e0 = e.x, e1 = e.y, e2 = e.z, e3 = e.w;
              n.add4(map[e0 >> 8] ^ sign_bytes(e0), map[e1 >> 8] ^ sign_bytes(e1),
                     map[e2 >> 8] ^ sign_bytes(e2), map[e3 >> 8] ^ sign_bytes(e3));
            };
#pragma unroll
            for (int g = 0; g < G; ++g)
              if (g < groups) add(w[g]);
            for (int g = G; g < groups; ++g) add(__ldg(a.words + (static_cast<size_t>(u.x) + g) * 32 + lane));
            nb = n.decide(sum, old);
          } else {
            LaneSums n;
            n.clear();
            auto add = [&](const int4& e) {
              n.add(map[static_cast<uint32_t>(e.x) >> 8], static_cast<int8_t>(e.x));
              n.add(map[static_cast<uint32_t>(e.y) >> 8], static_cast<int8_t>(e.y));
              n.add(map[static_cast<uint32_t>(e.z) >> 8], static_cast<int8_t>(e.z));
              n.add(map[static_cast<uint32_t>(e.w) >> 8], static_cast<int8_t>(e.w));
            };
            int left = I.flush;
#pragma unroll
            for (int g = 0; g < G; ++g)
              if (g < groups) {
                add(w[g]);
                if (--left == 0) {
                  n.flush();
                  left = I.flush;
                }
              }
            for (int g = G; g < groups; ++g) {
              add(__ldg(a.words + (static_cast<size_t>(u.x) + g) * 32 + lane));
              if (--left == 0) {
                n.flush();
                left = I.flush;
              }
            }
            n.flush();
            nb = n.decide(sum, old);
          }
          nb = lane < rows ? (nb ^ fl) & replica_mask : 0u;
          // 2. the new bytes into the maps
          if (CLUSTER) {
            uint32_t word = nb << (8 * dst_lane);
            word |= __shfl_xor_sync(kFullMask, word, 1);
            word |= __shfl_xor_sync(kFullMask, word, 2);
            const uint32_t to = smem_u32(map + u.y) + (lane & 28), on = bar + 8 * (step & 1u);
            for (uint32_t b = dst_lane; b < static_cast<uint32_t>(K) && ok; b += 4)
              asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(
                               cluster_addr(to, b)),
                           "r"(word), "r"(cluster_addr(on, b))
                           : "memory");
            __syncwarp();
          } else if (lane < rows) {
            map[u.y + lane] = static_cast<uint8_t>(nb);
          }
        }
        // a warp without a unit in this class may have one in the next
        if (cunit[c] + warp >= ue) stage(cunit[cn] + warp, cunit[cn + 1]);
        // 3. the exchange, between the unit warps
        if (CLUSTER) {
          const uint32_t on = bar + 8 * (step & 1u), parity = (step >> 1) & 1u;
          __syncwarp();
          if (lane == 0 && ok) {
            if (warp == 0)
              asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(on), "r"(cbytes[c])
                           : "memory");
            else
              asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(on) : "memory");
          }
          if (__any_sync(kFullMask, ok && !map_try(on, parity)))
            ok = __all_sync(kFullMask, map_wait(on, parity, a.error, a.budget));
        } else if (c + 1 < I.classes) {
          asm volatile("bar.sync 1, %0;" ::"r"(32 * U) : "memory");
        }
      }
      // 4. the next sweep's draws: by the draw warps all along, by the unit
      // warps once they are through
      const unsigned upto = (k + 1 < sweeps ? k + 1 : k) * mine;
      while (static_cast<int>(taken - upto) < 0) {
        unsigned next = 0;
        if (lane == 0) next = atomicAdd(drawn, 1u);
        if (thr != 0) draw(taken - k * mine, static_cast<uint32_t>(thr), (k & 1u) ^ 1u);
        taken = __shfl_sync(kFullMask, next, 0);
      }
      if (CLUSTER)
        cluster_sync();
      else
        __syncthreads();
    }
    for (int i = warp; i < nunits; i += kBatchMapWarps) {
      const int4 x = units[i];
      if (lane < (x.w & 0xffff)) a.spins[I.vtx_base + x.z + lane] = map[x.y + lane];
    }
    __syncthreads();
  }
  if (CLUSTER) cluster_sync();
}

// The entries of the units from the instances' rows: block b writes every
// gridDim.x-th unit of 8, a warp each.
static __global__ void __launch_bounds__(256)
    batch_map_fill_kernel(const int4* __restrict__ units, const int32_t* __restrict__ unit_inst, int num_units,
                          const BatchMapInst* __restrict__ inst, const int32_t* __restrict__ row_base,
                          const int32_t* __restrict__ row_ptr, const int32_t* __restrict__ adj,
                          const int32_t* __restrict__ map_index, int4* words) {
  const int lane = threadIdx.x & 31;
  for (int i = blockIdx.x * 8 + (threadIdx.x >> 5); i < num_units; i += gridDim.x * 8) {
    const int4 u = __ldg(units + i);
    const int gi = __ldg(unit_inst + i), row0 = inst[gi].row0;
    int e = 0, e1 = 0;
    if (lane < (u.w & 0xffff)) {
      const int32_t* rp = row_ptr + __ldg(row_base + inst[gi].id);
      e = __ldg(rp + u.z + lane);
      e1 = __ldg(rp + u.z + lane + 1);
    }
    for (int g = 0; g < (u.w >> 16); ++g) {
      int x[4];
#pragma unroll
      for (int s = 0; s < 4; ++s, ++e) {
        x[s] = 0;
        if (e < e1) {
          const int word = __ldg(adj + e);
          x[s] = (__ldg(map_index + row0 + (static_cast<unsigned>(word) >> 8)) << 8) | (word & 0xff);
        }
      }
      words[(static_cast<size_t>(u.x) + g) * 32 + lane] = make_int4(x[0], x[1], x[2], x[3]);
    }
  }
}

}  // namespace isingx
