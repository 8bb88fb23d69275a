// Partitioned HASH_AGGREGATE for global tables that outgrow a CTA: perfect
// arrays and linear-probing tables whose slots are updated once per row cost
// one or two random atomics a row in L2 or, past its size, in DRAM, and a
// skewed key queues every CTA on the same words.  Here the table is split into
// ranges of S = 2^shift slots that fit in shared memory:
//   k_part_hist     counts the rows of each range; its last CTA turns the
//                   counts into row offsets and into units of at most
//                   unit_rows rows, so that a hot range is shared by CTAs;
//   k_part_scatter  sorts tiles of rows by range in shared memory and appends
//                   each range's run to the range (group and value);
//   k_part_agg      takes a unit at a time into a shared-memory table and
//                   writes its groups straight to the result columns.  The
//                   units of a shared range add into the range's slots of the
//                   global table, which the last one extracts and empties.
// A record is the row's group (key or slot) and the value of its SUM: 12 bytes.
// The bytes: the key twice and the value once from the table, one write and one
// read of a record a row, each group once.  60M rows of an
// int32 key with 1e7 groups and an int64 value took 2041 us of atomics and
// 312 us of extraction; they take 57 + 373 + 233 us.  The count reads at 0.6 of
// the copy rate; the scatter is bound by the latency of its phases (a tile of
// 8192 rows fills the shared memory, so two tiles an SM are all there are to
// overlap), the last kernel by shared-memory atomics, two a row.
// A range of a linear-probing table whose keys do not fit raises a flag, and
// the general kernels behind then run the whole pipeline (GroupOut::guard).
#pragma once

#include "pv_eval.cuh"

namespace pv {

constexpr int kPartBlock = 512;
constexpr int kPartMax = kPartMaxRanges;  // two words each in the scatter's shared memory
constexpr uint32_t kPartNone = 0xFFFFFFFFu;

// The aggregate of a record's value: the one SUM of a shape whose other
// aggregates are COUNTs (-1: another shape).
template <class A>
constexpr int part_sum() {
  int at = -1;
  for (int i = 0; i < A::N; ++i) {
    if (A::func_of[i] == PV_COUNT) continue;
    if (A::func_of[i] != PV_SUM || at >= 0) return -1;
    at = i;
  }
  return at;
}

// Shapes with partitioned kernels: one SUM, no probes (they would run twice),
// keys of 32-bit parts (a perfect array's slot number is the record's group; a
// hash table's key must itself be 32 bits).
template <class SH>
constexpr bool part_perfect_ok() {
  return SH::Probes::N == 0 && part_sum<typename SH::Aggs>() >= 0 && key_narrow<SH>();
}
template <class SH>
constexpr bool part_hash_ok() { return part_perfect_ok<SH>() && SH::Key::N == 1; }

template <class SH>
using PartKeyShape =
    Shape<typename SH::Cols, typename SH::Where, typename SH::Probes, typename SH::Key, Aggs<>, Proj<>>;
template <class SH>
using PartValShape = Shape<typename SH::Cols, Where<>, Probes<>, Key<>, typename SH::Aggs, Proj<>>;

// Record key and range of row r; ok: false outside a perfect array's domain.
template <class SH, bool HASH>
__device__ __forceinline__ uint32_t part_key(const GroupDesc& gd, const GroupOut& g, int shift,
                                             Item<PartKeyShape<SH>>& it, const KParams& kp, int r, uint32_t& part,
                                             bool& ok) {
  using KS = PartKeyShape<SH>;
  if constexpr (HASH) {
    ok = true;
    const uint32_t key = static_cast<uint32_t>(pack_key<KS>(it, kp, r));
    part = static_cast<uint32_t>(ht_index(key, g.hash, g.seed[0], g.log2cap) >> shift);
    return key;
  } else {
    const uint32_t slot = static_cast<uint32_t>(row_perfect_index<KS>(gd, it, kp, r, ok));
    part = slot >> shift;
    return slot;
  }
}

// Exclusive scan of one 32-bit value per thread; every thread calls it, and a
// barrier has to come before the next call.
__device__ __forceinline__ uint32_t part_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t ws[33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) ws[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const uint32_t w = lane < nwarps ? ws[lane] : 0;
    uint32_t wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += y;
    }
    if (lane < nwarps) ws[lane] = wi - w;
    if (lane == 31) ws[32] = wi;
  }
  __syncthreads();
  *total = ws[32];
  return ws[warp] + incl - v;
}

// Bulk prefetch into L2 of rows [row, row + n) of a column of T that starts on
// a 16-byte boundary (whole 16-byte words only).
template <class T>
__device__ __forceinline__ void part_prefetch(const T* col, int64_t row, int64_t n) {
  constexpr int64_t per = 16 / sizeof(T);
  row &= ~(per - 1);
  n &= ~(per - 1);
  if (n > 0) asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(col + row), "r"(static_cast<uint32_t>(n * sizeof(T))) : "memory");
}

constexpr int kPartPer = kPartMax / kPartBlock;  // ranges a thread scans

template <class SH, bool HASH>
__global__ void __launch_bounds__(kPartBlock) k_part_hist(const __grid_constant__ KParams kp,
                                                          const __grid_constant__ GroupDesc gd,
                                                          const __grid_constant__ GroupOut g,
                                                          const __grid_constant__ PartOut po) {
  __shared__ uint32_t h[kPartMax];
  __shared__ bool last;
  using KS = PartKeyShape<SH>;
  if (blockIdx.x == 0 && threadIdx.x == 0) *g.out_count = 0;
  for (int p = threadIdx.x; p < po.n_parts; p += kPartBlock) h[p] = 0;
  __syncthreads();
  constexpr int U = 2;
  for_items<false, U>(kp.n_items, [&](const int64_t (&idx)[U]) {
    Item<KS> it[U];
    eval_items<KS, false, U>(it, kp, idx);
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if ((it[u].mask >> r) & 1u) {
          uint32_t part;
          bool ok;
          part_key<SH, HASH>(gd, g, po.shift, it[u], kp, r, part, ok);
          if (ok) atomicAdd(h + part, 1u);
          else set_error(kp.err, PV_ERR_KEY_OUT_OF_RANGE);
        }
  });
  __syncthreads();
  for (int p = threadIdx.x; p < po.n_parts; p += kPartBlock)
    if (h[p]) atomicAdd(po.hist + p, h[p]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(po.ctl + kPartCtlDone, 1u) == gridDim.x - 1;
  __syncthreads();
  if (last) {
    __threadfence();
    uint32_t rows[kPartPer], units[kPartPer], nr = 0, nu = 0;
#pragma unroll
    for (int i = 0; i < kPartPer; ++i) {
      const int p = threadIdx.x * kPartPer + i;
      rows[i] = p < po.n_parts ? __ldcg(po.hist + p) : 0;
      units[i] = rows[i] / po.unit_rows + (rows[i] % po.unit_rows != 0);
      nr += rows[i];
      nu += units[i];
    }
    uint32_t tr, tu;
    uint32_t r0 = part_scan(nr, &tr);
    __syncthreads();
    uint32_t u0 = part_scan(nu, &tu);
#pragma unroll
    for (int i = 0; i < kPartPer; ++i) {
      const int p = threadIdx.x * kPartPer + i;
      if (p < po.n_parts) {
        po.off[p] = r0;
        po.cursor[p] = r0;
        po.unit_off[p] = u0;
      }
      r0 += rows[i];
      u0 += units[i];
    }
    if (threadIdx.x == 0) {
      po.off[po.n_parts] = tr;
      po.unit_off[po.n_parts] = tu;
    }
  }
  pdl_launch_dependents();
}

// Tile of the scatter: 8192 rows, so that runs have several rows per range even
// at 2048 ranges, and two CTAs fit an SM.
constexpr int kPartItems = 4;  // per thread
inline size_t part_scatter_smem(int n_parts) {
  return static_cast<size_t>(kPartBlock) * 4 * kPartItems * 12 + 2 * sizeof(uint32_t) * n_parts;
}

template <class SH, bool HASH>
__global__ void __launch_bounds__(kPartBlock, 2) k_part_scatter(const __grid_constant__ KParams kp,
                                                                const __grid_constant__ GroupDesc gd,
                                                                const __grid_constant__ GroupOut g,
                                                                const __grid_constant__ PartOut po) {
  using KS = PartKeyShape<SH>;
  using VS = PartValShape<SH>;
  using A = typename SH::Aggs;
  using Sum = typename At<part_sum<A>(), typename A::L>::type;
  constexpr int U = kPartItems;
  constexpr int TR = kPartBlock * 4 * U;
  extern __shared__ unsigned long long smem[];
  unsigned long long* sval = smem;                           // [TR]
  uint32_t* skey = reinterpret_cast<uint32_t*>(smem + TR);   // [TR]
  uint32_t* start = skey + TR;                                    // rows of a range, then its first row in the tile
  uint32_t* delta = start + po.n_parts;                           // range's next output row - first row in the tile
  pdl_wait();
  const int64_t n_tiles = (kp.n_items + kPartBlock * U - 1) / (kPartBlock * U);
  // The CTA's next tile of the columns every item reads is fetched into L2 while this one is sorted.
  constexpr uint32_t ahead = SH::Where::N > 0 ? SH::Where::slots : (SH::Key::slots | A::slots);
  // Without filters and with one key column, its next tile's keys are loaded into registers as well.
  constexpr bool kEarly = SH::Where::N == 0 && (SH::Key::slots & (SH::Key::slots - 1)) == 0;
  Item<KS> early[kEarly ? U : 1];
  auto load_early = [&](int64_t tile) {
    int64_t idx[U];
#pragma unroll
    for (int u = 0; u < U; ++u) idx[u] = (tile * U + u) * kPartBlock + threadIdx.x;
    if constexpr (kEarly) load_items_all<KS, U>(early, kp, idx);
  };
  auto part_of = [&](uint32_t k) -> uint32_t {
    return HASH ? static_cast<uint32_t>(ht_index(k, g.hash, g.seed[0], g.log2cap) >> po.shift) : k >> po.shift;
  };
  load_early(blockIdx.x);
  for (int p = threadIdx.x; p < po.n_parts; p += kPartBlock) start[p] = 0;
  __syncthreads();
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    const int64_t next = (tile + gridDim.x) * TR;
    if (threadIdx.x == 0 && next < kp.n_rows) {
      static_for<SH::Cols::N>([&](auto c) {
        constexpr int C = decltype(c)::value;
        using T = typename At<C, typename SH::Cols::L>::type::T;
        if constexpr ((ahead >> C) & 1u)
          part_prefetch(static_cast<const T*>(kp.col[C]), next, kp.n_rows - next < TR ? kp.n_rows - next : TR);
      });
    }
    int64_t idx[U];
#pragma unroll
    for (int u = 0; u < U; ++u) idx[u] = (tile * U + u) * kPartBlock + threadIdx.x;
    uint32_t key[U][4], rank[U][2];  // rank among the tile's rows of the range, two to a word
    uint32_t live = 0;
#pragma unroll
    for (int h = 0; h < U; h += 2) {  // two items at a time: more would not fit 64 registers
      Item<KS> it[2];
      if constexpr (kEarly) {
#pragma unroll
        for (int u = 0; u < 2; ++u) it[u] = early[h + u];
      } else {
        const int64_t two[2] = {idx[h], idx[h + 1]};
        eval_items<KS, false, 2>(it, kp, two);
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        rank[h + u][0] = rank[h + u][1] = 0;
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          key[h + u][r] = 0;
          if ((it[u].mask >> r) & 1u) {
            uint32_t part;
            bool ok;
            key[h + u][r] = part_key<SH, HASH>(gd, g, po.shift, it[u], kp, r, part, ok);
            if (ok) {
              rank[h + u][r >> 1] |= atomicAdd(start + part, 1u) << (16 * (r & 1));
              live |= 1u << (4 * (h + u) + r);
            }
          }
        }
      }
    }
    // The first two items' values are on their way while the tile's runs find their places.
    auto load_values = [&](Item<VS> (&it)[2], int h) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int64_t left = kp.n_rows - idx[h + u] * 4;
        it[u].nvalid = left >= 4 ? 4 : (left > 0 ? static_cast<int>(left) : 0);
        it[u].mask = (live >> (4 * (h + u))) & 0xFu;
        if (it[u].mask) load_slots<VS, A::slots>(it[u], kp, idx[h + u]);
      }
    };
    Item<VS> vals[2];
    if constexpr (kEarly) load_values(vals, 0);
    __syncthreads();
    // Room for the tile's run in each range (neighbouring lanes ask for neighbouring words, and every lane
    // asks, so that the requests are in flight together), and the run's first row in the tile.
    uint32_t to[kPartPer], n[kPartPer], mine = 0, total;
#pragma unroll
    for (int i = 0; i < kPartPer; ++i) {
      const int p = i * kPartBlock + threadIdx.x;
      to[i] = p < po.n_parts ? start[p] : 0;
    }
#pragma unroll
    for (int i = 0; i < kPartPer; ++i) {
      const int p = i * kPartBlock + threadIdx.x;
      if (i * kPartBlock < po.n_parts) to[i] = atomicAdd(po.cursor + p, to[i]);  // padded to whole blocks of words
    }
#pragma unroll
    for (int i = 0; i < kPartPer; ++i) {
      const int p = threadIdx.x * kPartPer + i;
      n[i] = p < po.n_parts ? start[p] : 0;
      mine += n[i];
    }
    uint32_t first = part_scan(mine, &total);
#pragma unroll
    for (int i = 0; i < kPartPer; ++i) {
      const int p = threadIdx.x * kPartPer + i;
      if (p < po.n_parts) start[p] = first;
      first += n[i];
    }
    __syncthreads();
#pragma unroll
    for (int h = 0; h < U; h += 2) {
      if (h > 0 || !kEarly) load_values(vals, h);
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          if (!((vals[u].mask >> r) & 1u)) continue;
          const uint32_t pos =
              start[part_of(key[h + u][r])] + ((rank[h + u][r >> 1] >> (16 * (r & 1))) & 0xFFFFu);
          skey[pos] = key[h + u][r];
          sval[pos] = static_cast<unsigned long long>(agg_value<Sum>(vals[u], kp, r));
        }
    }
#pragma unroll
    for (int i = 0; i < kPartPer; ++i) {
      const int p = i * kPartBlock + threadIdx.x;
      if (p < po.n_parts) delta[p] = to[i] - start[p];
    }
    if constexpr (kEarly) load_early(tile + gridDim.x);  // used after the runs are written out
    __syncthreads();
    for (int p = threadIdx.x; p < po.n_parts; p += kPartBlock) start[p] = 0;
#pragma unroll 4
    for (uint32_t i = threadIdx.x; i < total; i += kPartBlock) {
      const uint32_t k = skey[i];
      const uint32_t to_row = delta[part_of(k)] + i;
      po.key[to_row] = k;
      po.val[to_row] = sval[i];
    }
    __syncthreads();
  }
  pdl_launch_dependents();
}

// Shared memory of k_part_agg: per slot (and one side slot for the hash key
// equal to the empty marker) the sum, the row count, the hash key.
inline size_t part_agg_smem(bool hash, int shift) {
  const size_t s = (size_t{1} << shift) + 2;
  return s * (8 + 4 + (hash ? 4 : 0));
}

// Result row of slot `key` of a perfect array, or of hash key `key`.
template <class SH, bool HASH>
__device__ __forceinline__ void part_write_group(const GroupDesc& gd, const GroupOut& g, int64_t pos, uint32_t key,
                                                 unsigned long long sum, uint64_t count) {
  using A = typename SH::Aggs;
  write_keys(gd, g, pos, !HASH, key);
  static_for<A::N>([&](auto a) {
    constexpr int I = decltype(a)::value;
    g.out[(SH::Key::N + I) * g.out_cap + pos] = static_cast<int64_t>(I == part_sum<A>() ? sum : count);
  });
}

template <class SH, bool HASH>
__global__ void __launch_bounds__(1024) k_part_agg(const __grid_constant__ KParams kp,
                                                            const __grid_constant__ GroupDesc gd,
                                                            const __grid_constant__ GroupOut g,
                                                            const __grid_constant__ PartOut po) {
  constexpr int kSum = part_sum<typename SH::Aggs>();  // the sum's word of a global slot
  extern __shared__ unsigned long long smem[];
  const uint32_t S = 1u << po.shift;
  const uint32_t SS = S + 2;  // slot S: the side slot
  unsigned long long* sval = smem;                           // [SS]
  uint32_t* scnt = reinterpret_cast<uint32_t*>(smem + SS);   // [SS]
  uint32_t* skey = scnt + SS;                                // [SS], hash only
  __shared__ uint32_t s_unit, s_part, s_last;
  __shared__ unsigned long long s_base;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t warps = blockDim.x >> 5;
  // One row (or a warp's rows of one key) into the table.
  auto add = [&](uint32_t k, unsigned long long v, uint32_t count) {
    uint32_t s = k & (S - 1);
    if constexpr (HASH) {
      if (k == kPartNone) {
        s = S;
      } else {
        s = static_cast<uint32_t>(ht_index(k, g.hash, g.seed[0], g.log2cap)) & (S - 1);
        uint32_t step = 0;
        for (; step < S; ++step) {
          uint32_t cur = *reinterpret_cast<volatile uint32_t*>(skey + s);
          if (cur == kPartNone) cur = atomicCAS(skey + s, kPartNone, k);
          if (cur == kPartNone || cur == k) break;
          s = (s + 1) & (S - 1);
        }
        if (step == S) {  // the range is full: the general kernels take over
          po.ctl[kPartCtlFull] = 1u;
          return;
        }
      }
    }
    atomicAdd(scnt + s, count);
    shared_add64(sval + s, v);
  };
  pdl_wait();
  for (;;) {
    if (threadIdx.x == 0) s_unit = atomicAdd(po.ctl + kPartCtlUnit, 1u);
    for (uint32_t i = threadIdx.x; i < SS; i += blockDim.x) sval[i] = 0;
    for (uint32_t i = threadIdx.x; i < SS; i += blockDim.x) {
      scnt[i] = 0;
      if constexpr (HASH) skey[i] = kPartNone;
    }
    __syncthreads();
    const uint32_t unit = s_unit;
    if (unit >= po.unit_off[po.n_parts]) break;
    for (int p = threadIdx.x; p < po.n_parts; p += blockDim.x)
      if (po.unit_off[p] <= unit && unit < po.unit_off[p + 1]) s_part = p;
    __syncthreads();
    const uint32_t part = s_part;
    const uint32_t units = po.unit_off[part + 1] - po.unit_off[part];
    const uint32_t r0 = po.off[part] + (unit - po.unit_off[part]) * po.unit_rows;
    const uint32_t r1 = min(po.off[part + 1], r0 + po.unit_rows);
    constexpr int K = 4;              // rows of a thread in flight
    const uint32_t trip = K * blockDim.x;
    const uint32_t ahead = 3 * trip;  // rows fetched into L2 ahead of their use
    for (uint32_t b = r0 + warp * 32; b < r1; b += trip) {
      if (threadIdx.x == 0) {
        const uint32_t f = b == r0 ? b : b + ahead - trip;  // the first trip fetches all of the distance
        if (f < r1) {
          const uint32_t n = min(r1 - f, b == r0 ? ahead : trip);
          part_prefetch(po.key, f, n);
          part_prefetch(po.val, f, n);
        }
      }
      uint32_t k[K];
      unsigned long long v[K];
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const uint32_t r = b + lane + j * blockDim.x;
        const bool in = r < r1;
        k[j] = in ? __ldcs(po.key + r) : 0u;
        v[j] = in ? __ldcs(po.val + r) : 0ull;
      }
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const uint32_t r = b + lane + j * blockDim.x;
        bool mine = r < r1;
        if (units > 1) {
          // A shared range has a hot key: the rows of the key of the first (else the middle) lane, when
          // they are many, are combined by shuffles into one update instead of queueing on one word.
          for (int lead = 0; lead < 32; lead += 16) {
            const uint32_t hk = __shfl_sync(0xffffffffu, k[j], lead);
            const uint32_t same = __ballot_sync(0xffffffffu, mine && k[j] == hk);
            if (__popc(same) < 8) continue;
            const bool peer = mine && k[j] == hk;
            const unsigned long long s = warp_reduce<PV_SUM>(peer ? v[j] : 0ull);
            if (lane == 0) add(hk, s, __popc(same));
            mine = mine && !peer;
          }
        }
        if (mine) add(k[j], v[j], 1u);
      }
    }
    __syncthreads();
    // Where the groups are: this table, or for a shared range the global table's
    // slots, once the last of the range's units has added its own.
    const uint64_t slot0 = static_cast<uint64_t>(part) << po.shift;
    bool emit = true;
    if (units > 1) {
      for (uint32_t i = threadIdx.x; i <= S; i += blockDim.x) {
        const uint32_t count = scnt[i];
        if (count == 0) continue;
        uint64_t slot = slot0 + i;
        if constexpr (HASH) {
          const unsigned long long key = i == S ? kPartNone : skey[i];
          uint32_t s = static_cast<uint32_t>(ht_index(key, g.hash, g.seed[0], g.log2cap)) & (S - 1);
          uint32_t step = 0;
          for (; step < S; ++step) {
            unsigned long long cur = __ldcg(g.keys + slot0 + s);
            if (cur == kEmpty64) cur = atomicCAS(g.keys + slot0 + s, kEmpty64, key);
            if (cur == kEmpty64 || cur == key) break;
            s = (s + 1) & (S - 1);
          }
          if (step == S) {
            po.ctl[kPartCtlFull] = 1u;
            continue;
          }
          slot = slot0 + s;
        }
        unsigned long long* dst = g.vals + slot * g.stride;
        atomicAdd(dst + gd.count_word, static_cast<unsigned long long>(count));
        if (sval[i]) atomicAdd(dst + kSum, sval[i]);
      }
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0) s_last = atomicAdd(po.done + part, 1u) == units - 1;
      __syncthreads();
      emit = s_last != 0;
      __threadfence();
    }
    if (emit) {
      // A warp takes a run of slots, so the groups come out in slot order.
      const uint64_t table_slots = static_cast<uint64_t>(g.cap) - slot0;  // of the global table, from the range on
      const uint32_t n_slots = table_slots < S ? static_cast<uint32_t>(table_slots) : S;
      const uint32_t side = HASH && units == 1 ? 1u : 0u;
      const uint32_t per = ((n_slots + side + warps - 1) / warps + 31) & ~31u;
      const uint32_t i0 = warp * per, i1 = min(i0 + per, n_slots + side);
      auto occupied = [&](uint32_t i) -> bool {
        if (i >= i1) return false;
        return units == 1 ? scnt[i] != 0 : __ldcg(g.vals + (slot0 + i) * g.stride + gd.count_word) != 0;
      };
      uint32_t mine = 0, total;
      for (uint32_t i = i0 + lane; i < i1; i += 32) mine += occupied(i);
      mine = __reduce_add_sync(0xffffffffu, mine);
      const uint32_t first = part_scan(lane == 0 ? mine : 0u, &total);
      if (threadIdx.x == 0) s_base = atomicAdd(g.out_count, static_cast<unsigned long long>(total));
      __syncthreads();
      int64_t pos = static_cast<int64_t>(s_base) + __shfl_sync(0xffffffffu, first, 0);
      for (uint32_t b = i0; b < i1; b += 32) {
        const uint32_t i = b + lane;
        const bool occ = occupied(i);
        const uint32_t ball = __ballot_sync(0xffffffffu, occ);
        const int64_t at = pos + __popc(ball & ((1u << lane) - 1u));
        pos += __popc(ball);
        if (occ) {
          unsigned long long sum;
          uint64_t count;
          uint32_t key = static_cast<uint32_t>(slot0) + i;
          if (units == 1) {
            count = scnt[i];
            sum = sval[i];
            if constexpr (HASH) key = i == S ? kPartNone : skey[i];
          } else {
            unsigned long long* src = g.vals + (slot0 + i) * g.stride;
            count = __ldcg(src + gd.count_word);
            sum = __ldcg(src + kSum);
            if constexpr (HASH) key = static_cast<uint32_t>(__ldcg(g.keys + slot0 + i));
            for (int a = 0; a <= gd.n_aggs; ++a) src[a] = 0;
            if constexpr (HASH) g.keys[slot0 + i] = kEmpty64;
          }
          if (at < g.out_cap) part_write_group<SH, HASH>(gd, g, at, key, sum, count);
        }
      }
    }
    __syncthreads();  // the table and the shared words are free again
  }
  pdl_launch_dependents();
}

template <class SH, bool HASH>
static pv_status run_part(const LaunchCfg& c, const KParams& kp, const GroupDesc& gd, const GroupOut& g,
                          const PartOut& po) {
  LaunchCfg cp = c;
  cp.block = kPartBlock;
  cp.grid_mult = 0;
  auto kh = k_part_hist<SH, HASH>;
  auto ks = k_part_scatter<SH, HASH>;
  auto ka = k_part_agg<SH, HASH>;
  const size_t ssmem = part_scatter_smem(po.n_parts);
  const size_t asmem = part_agg_smem(HASH, po.shift);
  if (cudaFuncSetAttribute(ks, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(ssmem)) != cudaSuccess ||
      cudaFuncSetAttribute(ka, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(asmem)) != cudaSuccess)
    return PV_ERR_CUDA;
  const int gh = grid_for(cp, reinterpret_cast<const void*>(kh), 0, kp.n_items, kPartBlock * 4);
  const int gs = grid_for(cp, reinterpret_cast<const void*>(ks), ssmem, kp.n_items, kPartBlock * kPartItems);
  LaunchCfg ca = cp;
  ca.block = asmem > (size_t{110} << 10) ? 1024 : kPartBlock;  // a table that leaves room for one CTA on an SM
  const int ga = grid_for(ca, reinterpret_cast<const void*>(ka), asmem, kp.n_rows / po.unit_rows + po.n_parts, 1);
  if (gh <= 0 || gs <= 0 || ga <= 0) return PV_ERR_CUDA;
  if (cudaMemsetAsync(po.hist, 0, po.clear_bytes, c.stream) != cudaSuccess) return PV_ERR_CUDA;
  auto launch = [&](auto k, int grid, int block, size_t smem, bool dependent) {
    kmark(c);
    cudaError_t e = cudaSuccess;
    if (c.mark || !dependent) k<<<grid, block, smem, c.stream>>>(kp, gd, g, po);
    else e = pdl_launch(k, dim3(grid), dim3(block), smem, c.stream, kp, gd, g, po);
    kmark(c);
    ++*c.launches;
    return e == cudaSuccess && cudaGetLastError() == cudaSuccess;
  };
  if (!launch(kh, gh, kPartBlock, 0, false) || !launch(ks, gs, kPartBlock, ssmem, true) ||
      !launch(ka, ga, ca.block, asmem, true))
    return PV_ERR_CUDA;
  return PV_OK;
}

}  // namespace pv
