// Spin-map engine: deterministic anneals of graphs whose spins fit in one
// block's shared memory, a byte each (n <= 200 K), on one block, on the
// blocks of one cluster, or on one block per SM.
//
// A colour class is a short, latency-bound step: its rows' fields need the
// spins of the classes before it, and a class of the graphs this engine
// serves holds a few hundred to a few thousand rows. What a step costs
// is the exchange of the new spins, not the sums. So every block keeps the
// spins of the whole graph in shared memory; a warp's unit of 32 / L rows
// (host_graph.h, MapPlan) sums each row with L lanes, the entries loaded
// before the exchange of the class before it ends, and the new spins go
// straight into the other blocks' maps:
//   * one block: ordinary shared-memory stores and a block barrier;
//   * a cluster: one st.async per unit and destination, counted in bytes on the
//     destination's mbarrier, so a block waits for the data itself and no
//     barrier is exchanged. Two mbarriers alternate by class; every block
//     sends at least four bytes per class (a unit without rows if need be), so
//     no block runs more than one class ahead of another, and a class's
//     rows are overwritten only after every block has read the old ones;
//   * the grid: messages of 32 spins and a 32-bit sequence number in one
//     64-bit word, so a reader that polls the word gets data and arrival at
//     once (one L2 round trip instead of a barrier's and a refresh's). Two
//     buffers alternate by class step: a block writes a message of step t + 2 only
//     after it has read a message of step t + 1 from every block, each of which
//     was sent after its block had read step t.
// The flips of sweep t + 1 are drawn while sweep t runs, by the warps with no
// unit left, and Algorithm 1's picks by a kernel before this one (they do not
// depend on the spins).
//
// What bounds a step is its warps' instruction count, at 6 to 8 cycles per
// instruction of the one or two warps a scheduler has: hence few warps (8 to
// 16), a task table that one counter walks, up to 16 entries a lane before a
// row takes more lanes, rows strided over the lanes so that lane r ends up with
// row r, and no branch in the sums (missing groups have weight 0). Entries are
// read a task ahead, from shared memory where they fit beside the map: in a
// class of several rounds the L2 latency shows (20,099-vertex torus 4.07 -> 3.63
// us a sweep, 5,000-vertex power-law graph 16.6 -> 15.6; one round a class, the
// same). Two tasks ahead costs more in moves than it hides (10,000 vertices, 100k
// edges: 7.0 -> 7.6).
// Microseconds a sweep on GB300, against the engine that ran before (a block
// with its CSR in shared memory, item dataflow, or the grid barrier):
// 800 vertices, 19k edges, 17 classes, one block: 12.1 -> 6.5; 20,099-vertex
// torus, 4 classes, cluster: 12.5 -> 3.6; 10,000 vertices, 100k edges, 11
// classes, cluster: 48 -> 6.4; 30,011 vertices, 600k wide edges, 16 classes,
// cluster: 97 -> 17; 100,000 vertices, 5M edges, 30 classes, grid: 253 -> 62.
//
// Graphs with hubs (SPLIT). A power-law graph's hubs form a near-clique, so it
// has tens of classes of a few hubs each, whose rows hold thousands of entries;
// a row summed by one warp, in its own step, made that step 1 to 2 us. Only the
// terms from the class before need the step to wait: the rest of a row is
// summed one step earlier, in parts of 256 entries that go to whichever block
// has the fewest tasks then, and reach the row's partial sum with a red.async
// counted on the same mbarrier as the spins. A step is then its exchange (0.55
// to 0.8 us). Two staged groups: the units' padding is what more would cost (67
// against 63 us a sweep at four). Microseconds a sweep on power-law graphs, int8
// weights, engine before (hub.cuh, one block for the hub classes) / rows whole /
// split, parts in the row's own block / as it is: 5,000 vertices 46 / 17 / 16 /
// 16, 20,000 vertices 63 / 48 / 34 / 32, 100,000 vertices 93 / 154 / 83 / 63.
//
// Every wait is bounded (the handle's budget): then the error flag is set, the
// other blocks' waits end by it, every block leaves its loop, and the blocks of
// a cluster meet once more before they exit, so that no store reaches a block
// that has gone. A sweep with Algorithm 1's flips ends in a cluster barrier that
// a block still at work counts on: a warp whose wait ran out goes straight to it
// and says so in every block, and all of them leave together behind it.
#pragma once

#include <cstdint>

#include "cluster.cuh"
#include "host_graph.h"
#include "philox.cuh"
#include "sweep.cuh"

namespace isingx {

struct MapArgs {
  const MapBlock* blocks;
  const int4* tasks;  // MapTask
  const int4* words;
  const int4* weights;  // wide only
  const int32_t* row_pos;
  const int32_t* row_orig;
  const int32_t* class_row;
  const int32_t* class_seg;
  const int32_t* block_msg;
  const int32_t* class_bytes;
  const int32_t* class_msg;
  const int32_t* msg;
  const int32_t* map_index;
  unsigned long long* mail;  // two buffers of K mailboxes, zero at launch (grid)
  int32_t mail_stride;       // messages of a mailbox
  int32_t n, classes, map_bytes, tasks_max, rows_max, groups_max;
  int32_t par_end;           // update parity of every state byte after the launch
  long long budget;
  int* error;
  int32_t skip_block;        // failure-detection tests: this block + 1 keeps its first messages
  const uint32_t* pick_count;  // Algorithm 1: flips after each sweep of the launch (or null)
  const int32_t* picks;        // their map indices, pick_stride per sweep
  int32_t pick_stride;
  int32_t accs;                // split rows of a block, at most
};

// The bounded wait for a message of sequence number seq.
static __device__ __noinline__ bool map_poll(const unsigned long long* p, uint32_t seq, unsigned long long* x,
                                             int* error, long long budget) {
  const long long t0 = global_ns();
  for (;;) {
    for (int it = 0; it < 64; ++it) {
      asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(*x) : "l"(p) : "memory");
      if (static_cast<uint32_t>(*x >> 32) == seq) return true;
    }
    if (ld_relaxed_s32(error) != 0) return false;
    if (global_ns() - t0 > budget) {
      atomicExch(error, 1);
      return false;
    }
  }
}

// Four spins as bytes 0x01 / 0xff from the low four bits (set: spin -1).
__device__ __forceinline__ uint32_t map_spin_bytes(uint32_t bits) {
  return 0x01010101u + (((bits & 15u) * 0x00204081u) & 0x01010101u) * 0xfeu;
}

// A lane's first entries of its warp's next task; those past the unit's
// groups have weight 0.
template <bool WIDE, int G>
struct MapStaged {
  int4 w[G];
  int4 c[WIDE ? G : 1];
};

template <bool RES>
__device__ __forceinline__ int4 map_load(const int4* p) {
  return RES ? *p : __ldg(p);
}

template <bool WIDE>
__device__ __forceinline__ int map_group(const int8_t* map, const int4& w, const int4& c) {
  const int s0 = map[static_cast<unsigned>(w.x) >> 8], s1 = map[static_cast<unsigned>(w.y) >> 8];
  const int s2 = map[static_cast<unsigned>(w.z) >> 8], s3 = map[static_cast<unsigned>(w.w) >> 8];
  if (WIDE) return c.x * s0 + c.y * s1 + c.z * s2 + c.w * s3;
  return static_cast<int8_t>(w.x) * s0 + static_cast<int8_t>(w.y) * s1 + static_cast<int8_t>(w.z) * s2 +
         static_cast<int8_t>(w.w) * s3;
}

// Sums f over the lanes of a row (lanes r, r + R, r + 2 R, ... of a unit of
// R = 32 >> lg rows); the unit's stores need no other exchange, since lane r
// holds row r.
__device__ __forceinline__ int map_row_sum(int f, int lg) {
  switch (lg) {
    case 5: f += __shfl_xor_sync(kFullMask, f, 1); [[fallthrough]];
    case 4: f += __shfl_xor_sync(kFullMask, f, 2); [[fallthrough]];
    case 3: f += __shfl_xor_sync(kFullMask, f, 4); [[fallthrough]];
    case 2: f += __shfl_xor_sync(kFullMask, f, 8); [[fallthrough]];
    case 1: f += __shfl_xor_sync(kFullMask, f, 16); [[fallthrough]];
    default: return f;
  }
}

// Every vertex's spin into the map, four a load and four loads in flight a thread
// (eight: the same): a call of one sweep is mostly this and the way back. With a
// vertex a load, and the way back by the blocks' own rows, class by class: 130,000
// vertices of 8 on a cluster 66 us a call, now 50; 600 vertices in 600 classes on one
// block 504, now 323. Both are functions of their own: inlined they changed the
// registers of the sweep (800 vertices, 1000 sweeps on one block 6.58 -> 6.81 ms).
static __device__ __noinline__ void map_fill_spins(int8_t* map, const int32_t* index, const int8_t* spins, int n) {
  const int tid = threadIdx.x, threads = blockDim.x;
  const int4* index4 = reinterpret_cast<const int4*>(index);
  const uint32_t* spins4 = reinterpret_cast<const uint32_t*>(spins);
  if (tid < (n & 3)) map[__ldg(index + (n & ~3) + tid)] = static_cast<int8_t>(spin_of(spins[(n & ~3) + tid]));
  for (int i0 = tid; i0 < n >> 2; i0 += 4 * threads) {
    int4 to[4];
    uint32_t s[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * threads;
      if (i < n >> 2) {
        to[u] = __ldg(index4 + i);
        s[u] = spins4[i];
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int i = i0 + u * threads;
      if (i < n >> 2) {
        map[to[u].x] = static_cast<int8_t>(spin_of(static_cast<int>(s[u])));
        map[to[u].y] = static_cast<int8_t>(spin_of(static_cast<int>(s[u] >> 8)));
        map[to[u].z] = static_cast<int8_t>(spin_of(static_cast<int>(s[u] >> 16)));
        map[to[u].w] = static_cast<int8_t>(spin_of(static_cast<int>(s[u] >> 24)));
      }
    }
  }
}

// The k-th of K shares of the positions back to the state bytes, a word a thread.
static __device__ __noinline__ void map_write_back(const int8_t* map, const int32_t* index, int8_t* spins, int n, int k,
                                                   int K, int parity) {
  const int4* index4 = reinterpret_cast<const int4*>(index);
  uint32_t* spins4 = reinterpret_cast<uint32_t*>(spins);
  const int tid = threadIdx.x, words = n >> 2, share = (words + K - 1) / K, last = min(words, (k + 1) * share);
  const int rest = (n & ~3) + tid;
  if (k == K - 1 && rest < n) spins[rest] = static_cast<int8_t>(state_byte(map[__ldg(index + rest)], parity));
  for (int i = k * share + tid; i < last; i += static_cast<int>(blockDim.x)) {
    const int4 at = __ldg(index4 + i);
    spins4[i] = static_cast<uint32_t>(state_byte(map[at.x], parity)) |
                static_cast<uint32_t>(state_byte(map[at.y], parity)) << 8 |
                static_cast<uint32_t>(state_byte(map[at.z], parity)) << 16 |
                static_cast<uint32_t>(state_byte(map[at.w], parity)) << 24;
  }
}

// K blocks; sweeps t_begin .. t_begin + sweeps - 1.
// SPLIT: a cluster's plan with split rows (no Algorithm 1); G covers a part.
// RES: the block's entries are in shared memory.
template <int MODE, bool WIDE, int G, bool SPLIT, bool RES>
__global__ void __launch_bounds__(32 * kMapMaxWarps, 1)
    map_kernel(DevGraph d, MapArgs a, uint64_t t_begin, uint32_t sweeps, uint64_t T, uint64_t T0,
               uint32_t replica, PhiloxRounds rk) {
  extern __shared__ __align__(128) unsigned char map_mem[];
  constexpr bool CLUSTER = MODE == kMapCluster;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int threads = blockDim.x, warps = threads >> 5;
  const int k_me = blockIdx.x, K = gridDim.x;
  const int C = a.classes;
  const MapBlock B = a.blocks[k_me];
  // shared memory (map_smem_bytes)
  int8_t* map = reinterpret_cast<int8_t*>(map_mem);
  int4* res_words = reinterpret_cast<int4*>(map_mem + a.map_bytes);
  int4* res_weights = res_words + (RES ? a.groups_max * 32 : 0);
  int4* tasks = res_weights + (RES && WIDE ? a.groups_max * 32 : 0);
  const int CT = (C + 4) / 4 * 4;
  int32_t* crow = reinterpret_cast<int32_t*>(tasks + a.tasks_max);
  int32_t* cseg = crow + CT;
  int32_t* cbytes = cseg + CT;  // grid: the block's first message of every class
  int32_t* cmsg = cbytes + CT;
  int32_t* orig = cmsg + CT;
  uint32_t* flips = reinterpret_cast<uint32_t*>(orig + a.rows_max);
  uint8_t* bias = reinterpret_cast<uint8_t*>(flips + 2 * (a.rows_max / 32));
  uint64_t* bars = reinterpret_cast<uint64_t*>(bias + a.rows_max);
  volatile int* failed = reinterpret_cast<volatile int*>(bars + 2);  // cluster: a wait of some block ran out
  const int flip_words = a.rows_max / 32;

  int32_t* acc = reinterpret_cast<int32_t*>(bars + 8);
  if (SPLIT)
    for (int i = tid; i < a.accs + 32; i += threads) acc[i] = 0;
  if (MODE <= kMapBlockStream) {  // few vertices: a call would wait for its loads before the next ones start
    for (int p = tid; p < a.n; p += threads) map[__ldg(a.map_index + p)] = static_cast<int8_t>(spin_of(d.spins[p]));
  } else {
    map_fill_spins(map, a.map_index, d.spins, a.n);
  }
  for (int i = tid; i < B.rounds * warps; i += threads) tasks[i] = __ldg(a.tasks + B.task0 + i);
  for (int c = tid; c <= C; c += threads) {
    crow[c] = __ldg(a.class_row + k_me * (C + 1) + c);
    cseg[c] = __ldg(a.class_seg + k_me * (C + 1) + c);
    cbytes[c] = MODE == kMapGrid || SPLIT ? __ldg(a.block_msg + k_me * (C + 1) + c) : 0;
    if (MODE != kMapGrid) cbytes[c] += __ldg(a.class_bytes + c);
    cmsg[c] = __ldg(a.class_msg + c);
  }
  for (int r = tid; r < B.rows; r += threads) {
    orig[r] = __ldg(a.row_orig + B.row0 + r);
    const int p = __ldg(a.row_pos + B.row0 + r);
    bias[r] = d.bias != nullptr && p >= 0 ? __ldg(d.bias + p) : 128;
  }
  if (RES)
    for (int i = tid; i < B.groups * 32; i += threads) {
      res_words[i] = __ldg(a.words + static_cast<size_t>(B.words0) * 32 + i);
      if (WIDE) res_weights[i] = __ldg(a.weights + static_cast<size_t>(B.words0) * 32 + i);
    }
  const int4* words = (RES ? res_words : a.words + static_cast<size_t>(B.words0) * 32) + lane;
  const int4* weights = (RES ? res_weights : a.weights + (WIDE ? static_cast<size_t>(B.words0) * 32 : 0)) + lane;
  uint32_t bar = smem_u32(bars);
  if (CLUSTER && tid == 0) {
    // one arrival per warp and phase; the bytes on top of it
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(warps) : "memory");
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar + 8), "r"(warps) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    *failed = 0;
  }
  // this lane's share of a unit's stores: 16 bytes at most, to one block. The
  // failure-detection tests' block sends nothing.
  const bool skip = a.skip_block == k_me + 1;
  const bool sends = CLUSTER && (lane & 15) < K && !skip;
  uint32_t map_to = 0, bar_to = 0;
  if (sends) {
    map_to = cluster_addr(smem_u32(map), lane & 15) + (lane & 16);
    bar_to = cluster_addr(bar, lane & 15);
  }
  __syncthreads();

  // floor(T0 (T - 1 - t) / (T - 1)) and its remainder, stepped from sweep to
  // sweep (sweep_args without its division)
  const uint64_t D = T > 1 ? T - 1 : 1;
  uint32_t thr = 0, rem = 0;
  const uint32_t thr_step = static_cast<uint32_t>(T0 / D), rem_step = static_cast<uint32_t>(T0 % D);
  if (T > 1) {
    thr = static_cast<uint32_t>(T0 * (D - t_begin) / D);
    rem = static_cast<uint32_t>(T0 * (D - t_begin) % D);
  }
  // flip bits of rows 32 j .. 32 j + 31 in sweep t
  auto draw_flips = [&](int j, uint32_t t, uint32_t* out) {
    const uint32_t o = static_cast<uint32_t>(orig[32 * j + lane]);
    bool flip = false;
    if (thr != 0u && o != 0xffffffffu) {
      uint32_t lim = thr;
      if (d.bias != nullptr) {
        const unsigned long long x = (static_cast<unsigned long long>(lim) * bias[32 * j + lane]) >> 7;
        lim = x > 0xffffffffull ? 0xffffffffu : static_cast<uint32_t>(x);
      }
      flip = vertex_word(o, t, replica, 0u, rk) < lim;
    }
    const unsigned m = __ballot_sync(kFullMask, flip);
    if (lane == 0) out[j] = m;
  };
  for (int j = warp; j < B.rows / 32; j += warps) draw_flips(j, static_cast<uint32_t>(t_begin), flips);

  MapStaged<WIDE, G> st;
  auto stage = [&](const int4& task) {
    const int groups = task.w >> 16;
    const int at = task.x * 32;
#pragma unroll
    for (int g = 0; g < G; ++g) {
      st.w[g] = make_int4(0, 0, 0, 0);
      if (WIDE) st.c[g] = make_int4(0, 0, 0, 0);
      if (g < groups) {
        st.w[g] = map_load<RES>(words + at + g * 32);
        if (WIDE) st.c[g] = map_load<RES>(weights + at + g * 32);
      }
    }
  };
  // where a part's row has its partial sum: the address in that block of the
  // address `at` here, plus the sum's place with sum = 1
  auto owner = [&](uint32_t at, int sum, const int4& task) {
    const int to = (task.y & ((1 << kMapFlipShift) - 1)) >> kMapOwnerShift;
    return cluster_addr(at + 4 * sum * (task.y & ((1 << kMapOwnerShift) - 1)), to);
  };
  if (SPLIT) {
    // the parts of the first class, which later sweeps sum in the last class's
    // step, once every block has its map and cleared its partial sums
    cluster_sync();
    for (int i = B.last0 + warp; i < B.rounds * warps; i += warps) {
      const int4 x = tasks[i];
      if (((x.w >> 8) & 0xff) != kMapPart) continue;
      int f = 0;
      for (int g = 0; g < (x.w >> 16); ++g) {
        const int4 w = map_load<RES>(words + (x.x + g) * 32);
        f += map_group<WIDE>(map, w, WIDE ? map_load<RES>(weights + (x.x + g) * 32) : w);
      }
      f = __reduce_add_sync(kFullMask, f);
      if (lane == 0)
        asm volatile("red.relaxed.cluster.shared::cluster.add.s32 [%0], %1;" ::"r"(owner(smem_u32(acc), 1, x)), "r"(f)
                     : "memory");
    }
  }
  const int4* const tasks_end = tasks + B.rounds * warps;
  const int4* next = tasks + warp;  // the task after the staged one
  int4 t = *next;
  stage(t);
  next += warps;
  if (next >= tasks_end) next = tasks + warp;
  int4 coming = *next;
  if (CLUSTER)
    cluster_sync();
  else
    __syncthreads();

  bool ok = true;
  uint32_t step = 0;  // classes done in this launch
  for (uint32_t k = 0; k < sweeps; ++k) {
    const uint32_t* flip_now = flips + (k & 1u) * flip_words;
    uint32_t* flip_next = flips + ((k & 1u) ^ 1u) * flip_words;
    const bool more = k + 1 < sweeps;
    if (T > 1 && more) {  // sweep k + 1's threshold
      thr -= thr_step;
      if (rem < rem_step) {
        rem += static_cast<uint32_t>(D) - rem_step;
        --thr;
      } else {
        rem -= rem_step;
      }
    }
    uint32_t npick = 0;
    int pick = 0;
    if (a.pick_count != nullptr) {
      npick = __ldg(a.pick_count + k);
      if (static_cast<uint32_t>(tid) < npick) pick = __ldg(a.picks + static_cast<size_t>(k) * a.pick_stride + tid);
    }
    for (int c = 0; c < C;) {
      const int draw = static_cast<int>(static_cast<unsigned>(t.y) >> kMapFlipShift) - 1;
      if (SPLIT && ((t.w >> 8) & 0xff) == kMapPart) {
        int f = 0;
#pragma unroll
        for (int g = 0; g < G; ++g) f += map_group<WIDE>(map, st.w[g], st.c[WIDE ? g : 0]);
        f = __reduce_add_sync(kFullMask, f);
        if (lane == 0 && !skip)
          asm volatile("red.async.relaxed.cluster.shared::cluster.mbarrier::complete_tx::bytes.add.s32 [%0], %1, [%2];" ::"r"(
                           owner(smem_u32(acc), 1, t)),
                       "r"(f), "r"(owner(bar + 8 * (step & 1u), 0, t))
                       : "memory");
      } else if (t.w != 0) {
        // 1. the unit's fields
        const int lg = (t.w >> 8) & 0xff, groups = t.w >> 16;
        const int r = lane & ((32 >> lg) - 1);
        const int own = (t.y & ((1 << kMapFlipShift) - 1)) + r, row = (t.z & ((1 << kMapSplitShift) - 1)) + r;
        const int part = SPLIT ? static_cast<int>((t.z & 0x7fffffff) >> kMapSplitShift) : 0;
        int f = 0, early = 0;
        if (part != 0) early = acc[part - 1 + r];
#pragma unroll
        for (int g = 0; g < G; ++g) f += map_group<WIDE>(map, st.w[g], st.c[WIDE ? g : 0]);
        const int hold = map[own] >> 1;  // f > hold: spin -1 (f = 0 keeps the old spin)
        const bool flip = (flip_now[row >> 5] >> (row & 31)) & 1u;
        for (int g = G; g < groups; ++g) {
          const int4 w = map_load<RES>(words + (t.x + g) * 32);
          f += map_group<WIDE>(map, w, WIDE ? map_load<RES>(weights + (t.x + g) * 32) : w);
        }
        // 2. every lane of a row decides it: Eq. 2, then the flip
        f = map_row_sum(f, lg) + early;
        if (part != 0 && lane < (t.w & 0xff)) acc[part - 1 + lane] = 0;
        const bool neg = (f > hold) != flip;
        // 3. the new spins into the maps
        if (CLUSTER) {
          const unsigned bits = __ballot_sync(kFullMask, neg) >> (lane & 16);
          const uint32_t to = map_to + own - r, on = bar_to + 8 * (step & 1u);
          if (sends) {
            if (lg < 2) {
              if (lane < 16 || lg == 0)
                asm volatile(
                    "st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(to),
                    "r"(map_spin_bytes(bits)), "r"(map_spin_bytes(bits >> 4)), "r"(map_spin_bytes(bits >> 8)),
                    "r"(map_spin_bytes(bits >> 12)), "r"(on)
                    : "memory");
            } else if (lane < 16) {
              if (lg == 2)
                asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(to),
                             "r"(map_spin_bytes(bits)), "r"(map_spin_bytes(bits >> 4)), "r"(on)
                             : "memory");
              else
                asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(to),
                             "r"(map_spin_bytes(bits)), "r"(on)
                             : "memory");
            }
          }
        } else if (lane < (t.w & 0xff)) {
          map[own] = neg ? -1 : 1;
        }
      }
      // 4. the next task's entries; flips of the next sweep
      const bool last = t.z < 0;
      t = coming;
      stage(t);
      next += warps;
      if (next >= tasks_end) next = tasks + warp;
      if (draw >= 0 && more) draw_flips(draw, static_cast<uint32_t>(t_begin + k + 1), flip_next);
      coming = *next;
      if (!last) continue;  // the class has another round
      // 5. the exchange
      if (CLUSTER) {
        const uint32_t on = bar + 8 * (step & 1u);
        __syncwarp();
        if (lane == 0) {
          if (warp == 0)
            asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(on), "r"(cbytes[c])
                         : "memory");
          else
            asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(on) : "memory");
        }
        const uint32_t parity = (step >> 1) & 1u;
        if (__any_sync(kFullMask, !map_try(on, parity))) {
          ok = __all_sync(kFullMask, map_wait(on, parity, a.error, a.budget));
          if (!ok) {
            // to the next cluster barrier: the sweep's, or the last one (N_t only
            // falls, so no later sweep has one either)
            if (npick == 0u) goto done;
            break;
          }
        }
      } else if (MODE != kMapGrid) {
        __syncthreads();
      } else {
        __syncthreads();
        // the block's words of 32 spins to every block's mailbox, a warp for
        // each word and 32 blocks
        const uint32_t seq = step + 1;
        const size_t box = static_cast<size_t>(a.mail_stride);
        unsigned long long* mail = a.mail + (step & 1u) * box * K;
        const int r0 = crow[c], count = max(1, (crow[c + 1] - r0) >> 5), parts = (K + 31) >> 5;
        for (int x = warp; x < count * parts; x += warps) {
          const int j = x / parts, to = (x - j * parts) * 32 + lane;
          const bool neg = crow[c + 1] > r0 && orig[r0 + 32 * j + lane] >= 0 && map[cseg[c] + 32 * j + lane] < 0;
          const unsigned m = __ballot_sync(kFullMask, neg);
          if (to < K && !skip)
            asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(mail + to * box + (cbytes[c] - cmsg[c]) + j),
                         "l"((static_cast<unsigned long long>(seq) << 32) | m)
                         : "memory");
        }
        mail += k_me * box;
        for (int i = tid; i < cmsg[c + 1] - cmsg[c] && ok; i += threads) {
          const int meta = __ldg(a.msg + cmsg[c] + i);
          unsigned long long x;
          asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(x) : "l"(mail + i) : "memory");
          if (static_cast<uint32_t>(x >> 32) != seq) ok = map_poll(mail + i, seq, &x, a.error, a.budget);
          uint32_t* to = reinterpret_cast<uint32_t*>(map) + (meta >> 4);
          const int len = meta & 15;
          if (ok)
#pragma unroll
            for (int q = 0; q < 8; ++q)
              if (q < len) to[q] = map_spin_bytes(static_cast<uint32_t>(x) >> (4 * q));
        }
        ok = __syncthreads_and(ok);
        if (!ok) return;  // the launch has failed: the host reports it
      }
      ++c;
      ++step;
    }
    // 6. Algorithm 1's flips of the sweep, into every block's map
    if (npick != 0u) {
      for (uint32_t i = ok ? tid : npick; i < npick; i += threads) {
        const int p = i == static_cast<uint32_t>(tid) ? pick : __ldg(a.picks + static_cast<size_t>(k) * a.pick_stride + i);
        map[p] = static_cast<int8_t>(-map[p]);
      }
      if (CLUSTER) {
        if (!ok && lane < K)
          asm volatile("st.shared::cluster.s32 [%0], 1;" ::"r"(cluster_addr(bar + 16, lane)) : "memory");
        cluster_sync();  // no block's next spins may come before this block's flips
        if (*failed != 0) {
          ok = false;
          break;
        }
      } else {
        __syncthreads();
      }
    }
  }
done:
  map_write_back(map, a.map_index, d.spins, a.n, k_me, K, a.par_end);
  if (CLUSTER) {
    if (!ok) __nanosleep(20000);  // its last stores may still be on their way (a fraction of a microsecond)
    cluster_sync();
  }
}

// The entries of a plan's units (host_graph.h, MapPlan) from the graph's rows:
// block (k, y) writes every gridDim.y-th task of block k, a warp per task.
template <bool PACKED>
__global__ void __launch_bounds__(256)
    map_fill_kernel(DevGraph d, const MapBlock* __restrict__ blocks, const int4* __restrict__ tasks, int warps,
                    const int32_t* __restrict__ row_pos, const int32_t* __restrict__ map_index,
                    const int2* __restrict__ late, int hubs, int4* words, int4* weights) {
  const MapBlock B = blocks[blockIdx.x];
  const int lane = threadIdx.x & 31;
  for (int i = blockIdx.y * 8 + (threadIdx.x >> 5); i < B.rounds * warps; i += gridDim.y * 8) {
    const int4 t = __ldg(tasks + B.task0 + i);
    const int rows = t.w & 0xff, lg = (t.w >> 8) & 0xff, groups = t.w >> 16;
    const int first = t.z & ((1 << kMapSplitShift) - 1), none = lg == kMapPart ? 0 : (t.y & ((1 << kMapFlipShift) - 1)) << 8;  // weight 0, a valid index
    // entry 4 g + s of the lane: e0 + ((4 g + s) << step), past a gap of `gap`
    // entries from e_gap on
    int e0 = 0, e1 = 0, e_gap = 0x7fffffff, gap = 0, step = lg;
    if (lg == kMapPart) {
      const int p = __ldg(row_pos + blocks[(t.y & ((1 << kMapFlipShift) - 1)) >> kMapOwnerShift].row0 + first);
      const int2 l = __ldg(late + p);
      step = 5;
      e0 = __ldg(d.row_ptr + p) + static_cast<int>((t.z & 0x7fffffff) >> kMapSplitShift) * kMapPartEntries + lane;
      e1 = __ldg(d.row_ptr + p + 1);
      e_gap = l.x;
      gap = l.y - l.x;
    } else if ((lane & ((32 >> lg) - 1)) < rows && groups > 0) {
      const int p = __ldg(row_pos + B.row0 + first + (lane & ((32 >> lg) - 1)));
      e0 = (p < hubs ? __ldg(late + p).x : __ldg(d.row_ptr + p)) + (lane >> (5 - lg));
      e1 = p < hubs ? __ldg(late + p).y : __ldg(d.row_ptr + p + 1);
    }
    for (int g = 0; g < groups; ++g) {
      int w[4], c[4];
#pragma unroll
      for (int s = 0; s < 4; ++s) {
        int e = e0 + ((4 * g + s) << step);
        if (e >= e_gap) e += gap;
        Edge<PACKED> x;
        x.load(d, e, e < e1);
        c[s] = e < e1 ? x.weight() : 0;
        w[s] = e < e1 ? (__ldg(map_index + x.col()) << 8) | (PACKED ? c[s] & 0xff : 0) : none;
      }
      const size_t at = (static_cast<size_t>(B.words0) + t.x + g) * 32 + lane;
      words[at] = make_int4(w[0], w[1], w[2], w[3]);
      if (!PACKED) weights[at] = make_int4(c[0], c[1], c[2], c[3]);
    }
  }
}

// Algorithm 1's picks (ising.h): block b draws the flips of sweep t_begin + b,
// the first N distinct candidates, as map indices; one warp, the chosen
// vertices in a shared bit map. The sweeps are independent of one another, so
// they are drawn side by side before the anneal needs them.
__global__ void __launch_bounds__(32)
    map_picks_kernel(int n, uint64_t t_begin, uint64_t T, uint32_t n0, uint32_t replica, PhiloxRounds rk,
                     const int32_t* __restrict__ pos, const int32_t* __restrict__ map_index,
                     uint32_t* count, int32_t* picks, int stride) {
  extern __shared__ unsigned pick_bits[];
  const int lane = threadIdx.x;
  const uint64_t t = t_begin + blockIdx.x;
  const uint32_t N = nflip_count(n0, T, t);
  if (lane == 0) count[blockIdx.x] = N;
  for (int i = lane; i < (n + 31) / 32; i += 32) pick_bits[i] = 0u;
  __syncwarp();
  int32_t* out = picks + static_cast<size_t>(blockIdx.x) * stride;
  uint32_t have = 0;
  for (uint32_t j0 = 0; have < N; j0 += 32) {
    const uint32_t x = philox4x32_10_word0(j0 + lane, static_cast<uint32_t>(t), replica, 2u, rk);
    const uint32_t c = static_cast<uint32_t>((static_cast<uint64_t>(x) * static_cast<uint64_t>(n)) >> 32);
    const unsigned same = __match_any_sync(kFullMask, c);
    const bool fresh = (__ffs(same) - 1) == lane && !((pick_bits[c >> 5] >> (c & 31)) & 1u);
    const unsigned fmask = __ballot_sync(kFullMask, fresh);
    const uint32_t take = min(static_cast<uint32_t>(__popc(fmask)), N - have);
    const uint32_t rank = static_cast<uint32_t>(__popc(fmask & ((1u << lane) - 1u)));
    if (fresh && rank < take) {
      atomicOr(pick_bits + (c >> 5), 1u << (c & 31));
      out[have + rank] = __ldg(map_index + __ldg(pos + c));
    }
    have += take;
    __syncwarp();
  }
}

}  // namespace isingx
