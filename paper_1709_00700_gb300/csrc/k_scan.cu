// Scan pipelines without a hash-aggregation sink:
//   AGGREGATE (ungrouped, Table 1; Section 7.3 aggregate fragment),
//   PROJECT single pass (Section 4.1 coarse-grained strategy, here with
//     warp-aggregated atomics on one output cursor),
//   PROJECT multi pass (Section 4.1 fine-grained strategy: matches are
//     counted, a prefix sum yields unique write positions, the matches are
//     written in table order): matches are marked as bits and counted, then
//     written; the allocation-free entry point has no room for the bits and
//     filters again to write.
#include <algorithm>
#include <mutex>

#include "pv_eval.cuh"

namespace pv {

// ---------------------------------------------------------------------------
// AGGREGATE: per-thread accumulators (predicated mode folds every row with
// its flag as a 0/-1 mask, the multiplication of Section 6), warp shuffle
// reduction, one shared-memory pass per CTA, one atomic per CTA and
// aggregate; the last CTA decodes the result and re-zeroes the accumulators.
// ---------------------------------------------------------------------------
// CTA epilogue of the ungrouped aggregation: warp shuffles, one slot per warp
// in shared memory, one atomic per aggregate per CTA; the last CTA to finish
// decodes the MIN/MAX codes into the result and resets the accumulators.
template <class SH>
__device__ __forceinline__ void aggregate_epilogue(uint64_t (&acc)[SH::Aggs::N + 1], const AggOut& out) {
  using A = typename SH::Aggs;
  constexpr int NA = A::N;
  __shared__ unsigned long long red[32][NA + 1];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  static_for<NA + 1>([&](auto a) {
    constexpr int I = decltype(a)::value;
    constexpr int F = I < NA ? A::func_of[I < NA ? I : 0] : PV_COUNT;
    acc[I] = warp_reduce<F>(acc[I]);
  });
  if (lane == 0) {
#pragma unroll
    for (int a = 0; a <= NA; ++a) red[warp][a] = acc[a];
  }
  __syncthreads();
  if (warp == 0) {
    static_for<NA + 1>([&](auto a) {
      constexpr int I = decltype(a)::value;
      constexpr int F = I < NA ? A::func_of[I < NA ? I : 0] : PV_COUNT;
      uint64_t v = lane < nwarps ? red[lane][I] : 0;
      v = warp_reduce<F>(v);
      if (lane == 0 && v != 0) acc_atomic<F>(out.acc + I, v);
    });
  }
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(out.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    __threadfence();
    const uint64_t rows = atomicExch(out.acc + NA, 0ull);
    static_for<NA>([&](auto a) {
      constexpr int I = decltype(a)::value;
      constexpr int F = A::func_of[I];
      const uint64_t c = atomicExch(out.acc + I, 0ull);
      int64_t v = static_cast<int64_t>(c);
      if constexpr (F == PV_MIN) v = rows ? decode_min(c) : 0;
      if constexpr (F == PV_MAX) v = rows ? decode_max(c) : 0;
      out.result[I] = v;
    });
    *out.done = 0;
  }
}

template <class SH, bool PRED, bool CHUNK, int U>
__global__ void __maxnreg__(128) k_aggregate(const __grid_constant__ KParams kp, const __grid_constant__ AggOut out) {
  using A = typename SH::Aggs;
  constexpr int NA = A::N;
  uint64_t acc[NA + 1];
#pragma unroll
  for (int a = 0; a <= NA; ++a) acc[a] = 0;

  auto consume = [&](Item<SH> (&it)[U]) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const uint32_t live = (it[u].mask >> r) & 1u;
        if constexpr (PRED) {
          const uint64_t m = 0ull - live;
          static_for<NA>([&](auto a) {
            constexpr int I = decltype(a)::value;
            using AG = typename At<I, typename A::L>::type;
            acc[I] = acc_combine<AG::func>(acc[I], acc_code<AG::func>(agg_value<AG>(it[u], kp, r)) & m);
          });
          acc[NA] += live;
        } else if (live) {
          static_for<NA>([&](auto a) {
            constexpr int I = decltype(a)::value;
            using AG = typename At<I, typename A::L>::type;
            acc[I] = acc_combine<AG::func>(acc[I], acc_code<AG::func>(agg_value<AG>(it[u], kp, r)));
          });
          acc[NA] += 1;
        }
      }
    }
  };
  if constexpr (PRED) {
    for_items_pipelined<SH, CHUNK, U>(kp, consume);
  } else {
    for_items_pf<SH, CHUNK, U, first_stage_slots<SH>()>(kp, [&](const int64_t (&idx)[U]) {
      Item<SH> it[U];
      eval_items<SH, PRED, U>(it, kp, idx);
      consume(it);
    });
  }

  aggregate_epilogue<SH>(acc, out);
}

// ---------------------------------------------------------------------------
// PROJECT helpers
// ---------------------------------------------------------------------------
template <class SH>
__device__ __forceinline__ void write_row(const ProjOut& out, Item<SH>& it, int r, int64_t pos) {
  using PJ = typename SH::Proj;
  static_for<PJ::N>([&](auto c) {
    constexpr int C = decltype(c)::value;
    constexpr int S = PJ::slot_of[C];
    if constexpr (S >= 0) {
      using T = typename At<S, typename SH::Cols::L>::type::T;
      static_cast<T*>(out.col[C])[pos] = VGet<S>::get(it.v)[r];
    } else {
      static_cast<int32_t*>(out.col[C])[pos] = it.pay[-S - 1][r];
    }
  });
}

__device__ __forceinline__ int warp_incl_scan(int v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// Block-wide exclusive scan of a 64-bit value; returns the prefix and sets
// *total.  Every thread of the block must call it.
__device__ __forceinline__ uint64_t block_excl_scan(uint64_t v, uint64_t* total) {
  __shared__ unsigned long long ws[33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  uint64_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t y = __shfl_up_sync(0xffffffffu, static_cast<unsigned long long>(incl), o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) ws[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint64_t w = lane < nwarps ? ws[lane] : 0;
    uint64_t wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint64_t y = __shfl_up_sync(0xffffffffu, static_cast<unsigned long long>(wi), o);
      if (lane >= o) wi += y;
    }
    if (lane < nwarps) ws[lane] = wi - w;
    if (lane == 31) ws[32] = wi;  // nwarps <= 32: lane 31 holds the grand total
  }
  __syncthreads();
  const uint64_t ex = ws[warp] + incl - v;
  *total = ws[32];
  __syncthreads();
  return ex;
}

// Bytes of one projected row before projected column C (source column types;
// payloads are int32); proj_offset<SH, N> is the whole row.
template <class SH, int C>
constexpr int proj_offset() {
  if constexpr (C == 0) {
    return 0;
  } else {
    constexpr int S = SH::Proj::slot_of[C - 1];
    constexpr int sz = S >= 0 ? static_cast<int>(sizeof(typename At<(S >= 0 ? S : 0), typename SH::Cols::L>::type::T)) : 4;
    return proj_offset<SH, C - 1>() + sz;
  }
}

// A warp's output stage in shared memory, R rows: column C at R * offset(C).
template <class SH, int R>
__host__ __device__ constexpr size_t out_stage_bytes() {
  return (static_cast<size_t>(R) * proj_offset<SH, SH::Proj::N>() + 15) & ~size_t(15);
}

// Row r of an item into row `slot` of the stage.
template <class SH, int R>
__device__ __forceinline__ void stage_out_row(char* st, int slot, Item<SH>& it, int r) {
  using PJ = typename SH::Proj;
  static_for<PJ::N>([&](auto c) {
    constexpr int C = decltype(c)::value;
    constexpr int S = PJ::slot_of[C];
    char* col = st + R * proj_offset<SH, C>();
    if constexpr (S >= 0) {
      using T = typename At<S, typename SH::Cols::L>::type::T;
      reinterpret_cast<T*>(col)[slot] = VGet<S>::get(it.v)[r];
    } else {
      reinterpret_cast<int32_t*>(col)[slot] = it.pay[-S - 1][r];
    }
  });
}

// The warp's n staged rows to the output at positions reserved with one
// atomicAdd; rows past the capacity are dropped (overflow).  All lanes.
template <class SH, int R>
__device__ __forceinline__ void flush_out_rows(const char* st, int n, const ProjOut& out, bool& overflow) {
  using PJ = typename SH::Proj;
  const int lane = threadIdx.x & 31;
  __syncwarp();
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(out.cursor, static_cast<unsigned long long>(n));
  base = __shfl_sync(0xffffffffu, base, 0);
  for (int i = lane; i < n; i += 32) {
    const int64_t pos = static_cast<int64_t>(base) + i;
    if (pos >= out.capacity) {
      overflow = true;
      continue;
    }
    static_for<PJ::N>([&](auto c) {
      constexpr int C = decltype(c)::value;
      constexpr int S = PJ::slot_of[C];
      const char* col = st + R * proj_offset<SH, C>();
      if constexpr (S >= 0) {
        using T = typename At<S, typename SH::Cols::L>::type::T;
        static_cast<T*>(out.col[C])[pos] = reinterpret_cast<const T*>(col)[i];
      } else {
        static_cast<int32_t*>(out.col[C])[pos] = reinterpret_cast<const int32_t*>(col)[i];
      }
    });
  }
  __syncwarp();
}

// Single pass: a warp's matches of a trip (counts are scanned with shuffles)
// are written at positions reserved with one atomicAdd on the output cursor.
// The cursor takes about one atomic a nanosecond, so a trip of fewer than
// sp_flush rows is staged in shared memory until that many are there: 15M
// rows with 9% matching, 12 rows a trip, were bound by the cursor (118 us).
// Output order is arbitrary across warps.  Trips of several items flush more
// rows: 50M rows with 25% matching, 64 a trip of two items, took 235 us without
// stages, 274 when flushed at 64 and 168 at 96.
template <int U>
constexpr int sp_flush() { return U == 1 ? 64 : 96; }
template <int U>
constexpr int sp_stage() { return 2 * sp_flush<U>(); }  // rows staged at most: sp_flush - 1 and one trip's
// REGS: 64 for one item, where the next trip's first column is loaded ahead
// (50M rows, 1% kept by one filter: 226 us without stages and load, 74 with),
// and for blocks past 512 threads, which launch with no more.  More items hold
// their loads in flight in up to 128 instead: two at 64, with the load ahead,
// took 442 us against 367 for the join and projection of 50M rows, 72% kept.
template <class SH, bool PRED, bool CHUNK, int U, int REGS>
__global__ void __maxnreg__(REGS) k_project_sp(const __grid_constant__ KParams kp, const __grid_constant__ ProjOut out) {
  extern __shared__ float4 spmem[];
  char* st = reinterpret_cast<char*>(spmem) + (threadIdx.x >> 5) * out_stage_bytes<SH, sp_stage<U>()>();
  bool overflow = false;
  int staged = 0;  // warp-uniform
  auto write_items = [&](Item<SH> (&it)[U]) {
    int cnt = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) cnt += __popc(it[u].mask);
    const int incl = warp_incl_scan(cnt);
    const int total = __shfl_sync(0xffffffffu, incl, 31);
    if (total == 0) return;
    if (total < sp_flush<U>()) {
      int slot = staged + incl - cnt;
#pragma unroll
      for (int u = 0; u < U; ++u)
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if ((it[u].mask >> r) & 1u) stage_out_row<SH, sp_stage<U>()>(st, slot++, it[u], r);
      staged += total;
      if (staged >= sp_flush<U>()) {
        flush_out_rows<SH, sp_stage<U>()>(st, staged, out, overflow);
        staged = 0;
      }
      return;
    }
    unsigned long long base = 0;
    if ((threadIdx.x & 31) == 31) base = atomicAdd(out.cursor, static_cast<unsigned long long>(total));
    base = __shfl_sync(0xffffffffu, base, 31);
    int64_t pos = static_cast<int64_t>(base) + incl - cnt;
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        if ((it[u].mask >> r) & 1u) {
          if (pos < out.capacity) write_row<SH>(out, it[u], r, pos);
          else overflow = true;
          ++pos;
        }
      }
    }
  };
  if constexpr (!PRED && !CHUNK && U == 1 && first_slot<SH>() >= 0) {
    for_items_ahead<SH, U>(kp, [&](Item<SH> (&it)[U], const int64_t (&idx)[U]) {
      eval_items<SH, false, U, true>(it, kp, idx);
      write_items(it);
    });
  } else {
    for_items_uniform<CHUNK, U>(kp.n_items, [&](const int64_t (&idx)[U]) {
      Item<SH> it[U];
      eval_items<SH, PRED, U>(it, kp, idx);
      write_items(it);
    });
  }
  if (staged > 0) flush_out_rows<SH, sp_stage<U>()>(st, staged, out, overflow);
  if (overflow) set_error(kp.err, PV_ERR_OUTPUT_OVERFLOW);
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(out.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    __threadfence();
    const int64_t n = static_cast<int64_t>(atomicExch(out.cursor, 0ull));
    *out.count = n < out.capacity ? n : out.capacity;
    *out.done = 0;
  }
}

// Tile of the ordered projection without bits: blockDim * U items; its item of
// (thread t, unroll u) is u * blockDim + t.
template <int U>
__device__ __forceinline__ void tile_items(int64_t tile, int64_t (&idx)[U]) {
#pragma unroll
  for (int u = 0; u < U; ++u) idx[u] = (tile * U + u) * static_cast<int64_t>(blockDim.x) + threadIdx.x;
}

// Exclusive prefix sum over the tile counts (one CTA of 1024 threads), for the
// generic kernels' multi-pass projection.
__global__ void __launch_bounds__(1024) k_tile_scan(const __grid_constant__ ProjOut out, int32_t* err) {
  pdl_wait();  // launched early behind the count kernel
  const int64_t n = out.n_tiles;
  const int64_t per = (n + blockDim.x - 1) / blockDim.x;
  const int64_t b = threadIdx.x * per;
  const int64_t e = b + per < n ? b + per : n;
  uint64_t s = 0;
  for (int64_t i = b; i < e; ++i) s += out.tile_count[i];
  uint64_t total;
  uint64_t run = block_excl_scan(s, &total);
  for (int64_t i = b; i < e; ++i) {
    out.tile_offset[i] = static_cast<int64_t>(run);
    run += out.tile_count[i];
  }
  pdl_launch_dependents();
  if (threadIdx.x == 0) {
    const int64_t t = static_cast<int64_t>(total);
    *out.count = t < out.capacity ? t : out.capacity;
    if (t > out.capacity) set_error(err, PV_ERR_OUTPUT_OVERFLOW);
  }
}

// ---------------------------------------------------------------------------
// Ordered projection.  A first kernel streams the filter columns and leaves one
// bit per row (n / 8 bytes, which stay in L2) and the matches per tile of 8192
// rows and per super of 16 tiles; the second takes a tile, or a part of one, per
// CTA: its first output position is the sum of the counts before it (supers,
// tiles of the super, words of the tile, so no scan kernel), its set bits become
// a row list in shared memory, and the listed rows are read and written one per
// lane, coalesced.  The filter runs once and the projected columns are read for
// matching rows only: bound by the filter columns' bytes.  Filtering twice
// around a scan kernel took 97 + 13 + 146 us for 50M rows with 2% matching (the
// query with its result delivered 264 us, now 111 us).
// ---------------------------------------------------------------------------
// The shape's filters and probes alone (no sink).
template <class SH>
using FilterShape = Shape<typename SH::Cols, typename SH::Where, typename SH::Probes, Key<>, Aggs<>, Proj<>>;

// A warp takes units of 32 * U items (128 * U consecutive rows); nothing in the
// loop waits for another warp.
template <class SH, bool PRED, int U>
__global__ void __maxnreg__(64) k_project_mark(const __grid_constant__ KParams kp,
                                               const __grid_constant__ ProjOut out) {
  static_assert(U <= 4 && kMarkTileRows % 512 == 0, "a unit lies within one tile");
  using FS = FilterShape<SH>;
  const int lane = threadIdx.x & 31;
  const int64_t W = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  const int64_t n_units = (kp.n_items + 32 * U - 1) / (32 * U);
  for (int64_t unit = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; unit < n_units; unit += W) {
    int64_t idx[U];
#pragma unroll
    for (int u = 0; u < U; ++u) idx[u] = (unit * U + u) * 32 + lane;
    Item<FS> it[U];
    eval_items<FS, PRED, U>(it, kp, idx);
    int count = 0;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      count += __popc(it[u].mask);
      uint32_t w = it[u].mask << (4 * (lane & 7));  // 8 lanes make a word
      w |= __shfl_xor_sync(0xffffffffu, w, 1);
      w |= __shfl_xor_sync(0xffffffffu, w, 2);
      w |= __shfl_xor_sync(0xffffffffu, w, 4);
      if (out.bits != nullptr && (lane & 7) == 0) out.bits[(unit * U + u) * 4 + (lane >> 3)] = w;
    }
    count = __reduce_add_sync(0xffffffffu, count);
    if (lane == 0 && count != 0) {
      const int64_t tile = unit * (128 * U) / kMarkTileRows;
      atomicAdd(out.mark_count + tile, static_cast<unsigned int>(count));
      atomicAdd(out.mark_super + (tile >> out.mark_shift), static_cast<unsigned long long>(count));
    }
  }
  pdl_launch_dependents();
}

// A CTA's unit is a tile's 2^split-th part: few rows are spread over the SMs, as
// a whole tile is 8 trips of dependent loads per lane.
template <class SH>
__global__ void __launch_bounds__(kMarkTileRows / 32) k_project_emit(const __grid_constant__ KParams kp,
                                                                     const __grid_constant__ ProjOut out, int split) {
  __shared__ uint16_t list[kMarkTileRows];  // matching rows of the unit, in order
  pdl_wait();  // launched early behind the mark kernel
  constexpr int TW = kMarkTileRows / 32;
  const int uw = TW >> split;  // words of a unit
  const int64_t n_words = (kp.n_rows + 31) >> 5;
  const int64_t n_units = n_words > uw ? (n_words + uw - 1) / uw : 1;
  for (int64_t unit = blockIdx.x; unit < n_units; unit += gridDim.x) {
    const int64_t word0 = unit * uw, tile = unit >> split;
    const int64_t word = word0 + threadIdx.x;
    uint32_t w = threadIdx.x < uw && word < n_words ? out.bits[word] : 0u;
    uint64_t before = 0;  // matches of earlier units, this thread's share
    const int64_t super = tile >> out.mark_shift;
    for (int64_t i = threadIdx.x; i < super; i += blockDim.x) before += out.mark_super[i];
    for (int64_t i = (super << out.mark_shift) + threadIdx.x; i < tile; i += blockDim.x) before += out.mark_count[i];
    if (tile * TW + threadIdx.x < word0) before += __popc(out.bits[tile * TW + threadIdx.x]);
    // one scan for both sums: the unit's matches (at most 8192) in the low 16 bits
    uint64_t sums;
    int p = static_cast<int>(block_excl_scan((before << 16) | static_cast<uint64_t>(__popc(w)), &sums) & 0xFFFFu);
    const int total = static_cast<int>(sums & 0xFFFFu);
    const int64_t base = static_cast<int64_t>(sums >> 16);
    for (; w != 0; w &= w - 1) list[p++] = static_cast<uint16_t>(threadIdx.x * 32 + __ffs(w) - 1);
    __syncthreads();
    constexpr int K = 4;  // rows of a lane read together
    for (int i = threadIdx.x; i < total; i += K * blockDim.x) {
      Item<SH> it[K];
      bool ok[K], has[K];
      int64_t rows[K];
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int j = i + k * blockDim.x;
        has[k] = j < total;
        rows[k] = word0 * 32 + (has[k] ? list[j] : 0);
      }
      compact_load_rows<SH, K, 1>(it, ok, kp, rows, has);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int64_t at = base + i + k * blockDim.x;
        if (ok[k] && at < out.capacity) write_row<SH>(out, it[k], 0, at);
      }
    }
    if (unit == n_units - 1 && threadIdx.x == 0) {
      const int64_t n = base + total;
      *out.count = n < out.capacity ? n : out.capacity;
      if (n > out.capacity) set_error(kp.err, PV_ERR_OUTPUT_OVERFLOW);
    }
    __syncthreads();  // the list is free again
  }
  // The last CTA leaves the counters at zero for the next run: a clear ahead of the marks was a launch of its own.
  __shared__ bool last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(out.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last) {
    const int64_t n_tiles = mark_tiles(kp.n_rows);
    for (int64_t i = threadIdx.x; i < n_tiles; i += blockDim.x) out.mark_count[i] = 0;
    for (int64_t i = threadIdx.x; i <= (n_tiles - 1) >> out.mark_shift; i += blockDim.x) out.mark_super[i] = 0;
    if (threadIdx.x == 0) *out.done = 0;
  }
}

// Ordered projection without bits, for the allocation-free entry point, whose
// static scratch holds the counts only: the second kernel filters its tile again.
// One CTA per tile; the tile's matches become a row list in shared memory, and
// the listed rows are read and written one per lane.  (One kernel with a chained
// prefix sum, which filters once, is bound by its look-back: 1M rows took 18 us
// against 15 by counting, scanning and filtering again, 10M 43 against 40.)
template <class SH, int U>
__global__ void __maxnreg__(64) k_project_refilter(const __grid_constant__ KParams kp,
                                                   const __grid_constant__ ProjOut out) {
  static_assert(U <= 4, "16-bit scan fields hold at most 4 unroll slots");
  __shared__ uint16_t list[kMarkTileRows];  // rows of the tile that match, in output order
  pdl_wait();  // launched early behind the mark kernel
  const int64_t n_tiles = mark_tiles(kp.n_rows);
  for (int64_t tile = blockIdx.x; tile < n_tiles; tile += gridDim.x) {
    int64_t idx[U];
    tile_items<U>(tile, idx);
    uint32_t mask[U];
    {
      using FS = FilterShape<SH>;
      Item<FS> it[U];
      eval_items<FS, false, U>(it, kp, idx);
#pragma unroll
      for (int u = 0; u < U; ++u) mask[u] = it[u].mask;
    }
    uint64_t before = 0, base;  // matches of earlier tiles
    const int64_t super = tile >> out.mark_shift;
    for (int64_t i = threadIdx.x; i < super; i += blockDim.x) before += out.mark_super[i];
    for (int64_t i = (super << out.mark_shift) + threadIdx.x; i < tile; i += blockDim.x) before += out.mark_count[i];
    block_excl_scan(before, &base);
    int total, pos[U];  // tile matches; list position of each item's first match
    {  // row order inside the tile: (u, thread, row); one scan of U packed 16-bit counters (at most 4 * 512 each)
      uint64_t packed = 0, t;
#pragma unroll
      for (int u = 0; u < U; ++u) packed |= static_cast<uint64_t>(__popc(mask[u])) << (16 * u);
      const uint64_t ex = block_excl_scan(packed, &t);
      total = 0;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        pos[u] = total + static_cast<int>((ex >> (16 * u)) & 0xFFFF);
        total += static_cast<int>((t >> (16 * u)) & 0xFFFF);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      int p = pos[u];
      const uint16_t r0 = static_cast<uint16_t>(idx[u] * 4 - tile * kMarkTileRows);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if ((mask[u] >> r) & 1u) list[p++] = static_cast<uint16_t>(r0 + r);
    }
    __syncthreads();
    constexpr int K = 2;  // rows of a lane read together
    for (int i = threadIdx.x; i < total; i += K * blockDim.x) {
      Item<SH> it[K];
      bool ok[K], has[K];
      int64_t rows[K];
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int j = i + k * blockDim.x;
        has[k] = j < total;
        rows[k] = tile * kMarkTileRows + (has[k] ? list[j] : 0);
      }
      compact_load_rows<SH, K, 1>(it, ok, kp, rows, has);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        const int64_t at = static_cast<int64_t>(base) + i + k * blockDim.x;
        if (ok[k] && at < out.capacity) write_row<SH>(out, it[k], 0, at);
      }
    }
    if (tile == n_tiles - 1 && threadIdx.x == 0) {
      const int64_t n = static_cast<int64_t>(base) + total;
      *out.count = n < out.capacity ? n : out.capacity;
      if (n > out.capacity) set_error(kp.err, PV_ERR_OUTPUT_OVERFLOW);
    }
    __syncthreads();  // the list is free again
  }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
// Compacted execution of an ungrouped aggregation: the rows that survive the
// first operation are queued per warp and accumulated one per lane.
template <class SH, int K, int FI>
__global__ void __maxnreg__(128) k_aggregate_compact(const __grid_constant__ KParams kp,
                                                     const __grid_constant__ AggOut out) {
  using A = typename SH::Aggs;
  constexpr int NA = A::N;
  extern __shared__ uint32_t qmem[];
  uint64_t acc[NA + 1];
#pragma unroll
  for (int a = 0; a <= NA; ++a) acc[a] = 0;
  for_rows_compacted<SH, K, 1, false, FI>(kp, qmem + (threadIdx.x >> 5) * queue_cap<K>(),
                            [&](const uint32_t (&rows)[K], const bool (&has)[K]) {
    Item<SH> it[K];
    bool ok[K];
    compact_load_rows<SH, K, 1>(it, ok, kp, rows, has);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (!ok[k]) continue;
      static_for<NA>([&](auto a) {
        constexpr int I = decltype(a)::value;
        using AG = typename At<I, typename A::L>::type;
        acc[I] = acc_combine<AG::func>(acc[I], acc_code<AG::func>(agg_value<AG>(it[k], kp, 0)));
      });
      acc[NA] += 1;
    }
  });
  aggregate_epilogue<SH>(acc, out);
}

// Output rows a warp stages in shared memory before it reserves their
// positions: a flush starts at 64 rows, and one drain adds at most 32 * K.
template <int K>
__host__ __device__ constexpr int out_stage_rows() { return 32 * (2 + K); }

// Compacted single-pass PROJECT: the rows that survive the first operation
// are queued per warp; at each drain every lane takes its queued rows through
// the rest of the pipeline, and the rows that survive are appended to the
// warp's output stage in shared memory (ballot + popc).  Once 64 or more are
// staged the warp reserves their output positions with one atomicAdd and
// writes them out coalesced: one atomic per 64 to 127 output rows, where one
// per drain put the whole grid on one counter.  Output order is arbitrary, as
// for the other single-pass projection.  Held to 48 registers (none of the
// compiled projections spills there): five 256-thread or two 512-thread CTAs
// per SM, more warps to hide the gathers' latency (the best variant of the
// 100M-row filter/project measured 171.7 us against 185.9 us at 128).
template <class SH, int K, int FI>
__global__ void __maxnreg__(48) k_project_compact(const __grid_constant__ KParams kp,
                                                   const __grid_constant__ ProjOut out) {
  extern __shared__ uint32_t qmem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  char* ost = reinterpret_cast<char*>(qmem + nwarps * queue_cap<K>()) + warp * out_stage_bytes<SH, out_stage_rows<K>()>();
  bool overflow = false;
  int staged = 0;  // warp-uniform
  for_rows_compacted<SH, K, 1, true, FI>(kp, qmem + warp * queue_cap<K>(),
                                     [&](const uint32_t (&rows)[K], const bool (&has)[K]) {
    Item<SH> it[K];
    bool ok[K];
    compact_load_rows<SH, K, 1>(it, ok, kp, rows, has);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const unsigned b = __ballot_sync(0xffffffffu, ok[k]);
      if (ok[k]) stage_out_row<SH, out_stage_rows<K>()>(ost, staged + __popc(b & ((1u << lane) - 1u)), it[k], 0);
      staged += __popc(b);
    }
    if (staged >= 64) {
      flush_out_rows<SH, out_stage_rows<K>()>(ost, staged, out, overflow);
      staged = 0;
    }
  });
  if (staged > 0) flush_out_rows<SH, out_stage_rows<K>()>(ost, staged, out, overflow);
  if (overflow) set_error(kp.err, PV_ERR_OUTPUT_OVERFLOW);
  __shared__ bool last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(out.done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (last && threadIdx.x == 0) {
    __threadfence();
    const int64_t n = static_cast<int64_t>(atomicExch(out.cursor, 0ull));
    *out.count = n < out.capacity ? n : out.capacity;
    *out.done = 0;
  }
}

template <class SH, int K>
static pv_status launch_proj_compact_k(const LaunchCfg& c, const KParams& kp, const ProjOut& out) {
  auto k = c.first_items == 2 ? k_project_compact<SH, K, first_items_max<SH>()> : k_project_compact<SH, K, 1>;
  const size_t smem = static_cast<size_t>(c.block / 32) * (queue_cap<K>() * 4 + out_stage_bytes<SH, out_stage_rows<K>()>());
  if (smem > 48 * 1024 &&
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess)
    return PV_ERR_UNSUPPORTED;
  const int grid = grid_for(c, reinterpret_cast<const void*>(k), smem, kp.n_items, c.block);
  if (grid <= 0) return PV_ERR_UNSUPPORTED;
  kmark(c);
  k<<<grid, c.block, smem, c.stream>>>(kp, out);
  kmark(c);
  ++*c.launches;
  return cudaGetLastError() == cudaSuccess ? PV_OK : PV_ERR_CUDA;
}

template <class SH>
static pv_status launch_proj_compact(const LaunchCfg& c, const KParams& kp, const ProjOut& out, int exec) {
  if constexpr (SH::Where::N == 0 && SH::Probes::N == 0) {
    return PV_ERR_UNSUPPORTED;  // nothing to compact on
  } else {
    // single pass only: the queues reorder rows, and multi-pass output keeps input order
    if (exec != PV_EXEC_SINGLE_PASS || c.chunk || (c.U != 1 && c.U != 2) ||
        kp.n_rows > static_cast<int64_t>(UINT32_MAX) || c.first_items > first_items_max<SH>())
      return PV_ERR_UNSUPPORTED;
    return c.U == 2 ? launch_proj_compact_k<SH, 2>(c, kp, out) : launch_proj_compact_k<SH, 1>(c, kp, out);
  }
}

template <class SH, int K>
static pv_status launch_agg_compact_k(const LaunchCfg& c, const KParams& kp, const AggOut& out) {
  auto k = c.first_items == 2 ? k_aggregate_compact<SH, K, first_items_max<SH>()> : k_aggregate_compact<SH, K, 1>;
  const size_t smem = static_cast<size_t>(c.block / 32) * queue_cap<K>() * 4;
  const int grid = grid_for(c, reinterpret_cast<const void*>(k), smem, kp.n_items, c.block);
  if (grid <= 0) return PV_ERR_UNSUPPORTED;
  kmark(c);
  k<<<grid, c.block, smem, c.stream>>>(kp, out);
  kmark(c);
  ++*c.launches;
  return cudaGetLastError() == cudaSuccess ? PV_OK : PV_ERR_CUDA;
}

template <class SH>
static pv_status launch_agg_compact(const LaunchCfg& c, const KParams& kp, const AggOut& out) {
  if constexpr (SH::Where::N == 0 && SH::Probes::N == 0) {
    return PV_ERR_UNSUPPORTED;  // nothing to compact on
  } else {
    // items_per_thread: queued rows a lane takes through the row stage at once
    if (c.chunk || (c.U != 1 && c.U != 2) || kp.n_rows > static_cast<int64_t>(UINT32_MAX) ||
        c.first_items > first_items_max<SH>())
      return PV_ERR_UNSUPPORTED;
    return c.U == 2 ? launch_agg_compact_k<SH, 2>(c, kp, out) : launch_agg_compact_k<SH, 1>(c, kp, out);
  }
}

template <class SH, bool P, bool C, int U>
static pv_status launch_agg_t(const LaunchCfg& c, const KParams& kp, const AggOut& out) {
  auto k = k_aggregate<SH, P, C, U>;
  const int grid = grid_for(c, reinterpret_cast<const void*>(k), 0, kp.n_items, static_cast<int64_t>(c.block) * U);
  if (grid <= 0) return PV_ERR_UNSUPPORTED;
  kmark(c);
  k<<<grid, c.block, 0, c.stream>>>(kp, out);
  kmark(c);
  ++*c.launches;
  return cudaGetLastError() == cudaSuccess ? PV_OK : PV_ERR_CUDA;
}

pv_status launch_tile_scan(const LaunchCfg& c, const ProjOut& out, int32_t* err) {
  kmark(c);
  cudaError_t e = c.mark ? (k_tile_scan<<<1, 1024, 0, c.stream>>>(out, err), cudaSuccess)
                         : pdl_launch(k_tile_scan, dim3(1), dim3(1024), 0, c.stream, out, err);
  kmark(c);
  ++*c.launches;
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? PV_OK : PV_ERR_CUDA;
}

template <class SH, bool P, bool C, int U>
static pv_status launch_proj_sp(const LaunchCfg& c, const KParams& kp, const ProjOut& out) {
  auto k = k_project_sp<SH, P, C, U, U == 1 ? 64 : 128>;
  if constexpr (U == 2)
    if (c.block > 512) k = k_project_sp<SH, P, C, U, 64>;
  const size_t smem = static_cast<size_t>(c.block / 32) * out_stage_bytes<SH, sp_stage<U>()>();
  // the kernel's static shared memory counts too: 48 KB of stages (12-byte rows, 1024 threads) need the attribute
  if (smem >= 40 * 1024 &&
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem)) != cudaSuccess)
    return PV_ERR_UNSUPPORTED;
  const int grid = grid_for(c, reinterpret_cast<const void*>(k), smem, kp.n_items, static_cast<int64_t>(c.block) * U);
  if (grid <= 0) return PV_ERR_UNSUPPORTED;
  kmark(c);
  k<<<grid, c.block, smem, c.stream>>>(kp, out);
  kmark(c);
  ++*c.launches;
  return cudaGetLastError() == cudaSuccess ? PV_OK : PV_ERR_CUDA;
}

// The rows of an ordered projection and their order do not depend on access and
// items_per_thread, so its kernels choose both: the marks take 4 items a lane
// once that leaves an SM four warps with a unit each (10M rows, one filter,
// 10% matching: 72 us with one item, 37 with four; 100K rows 6.9 / 8.2).
static bool mark_wide(const LaunchCfg& c, const KParams& kp) {
  return kp.n_items >= static_cast<int64_t>(512) * c.sm_count;
}
template <class SH, bool P>
static pv_status launch_proj_ordered(const LaunchCfg& c, const KParams& kp, const ProjOut& out) {
  const bool wide = mark_wide(c, kp);
  auto km = wide ? k_project_mark<SH, P, 4> : k_project_mark<SH, P, 1>;
  auto ke = k_project_emit<SH>;
  LaunchCfg ce = c;
  ce.block = kMarkTileRows / 32;
  ce.grid_mult = 0;
  const int gm = grid_for(c, reinterpret_cast<const void*>(km), 0, kp.n_items,
                          static_cast<int64_t>(c.block) * (wide ? 4 : 1));
  const int resident = grid_for(ce, reinterpret_cast<const void*>(ke), 0, INT32_MAX, 1);
  if (gm <= 0 || resident <= 0) return PV_ERR_UNSUPPORTED;
  // until an SM has three units (100K rows, all matching: 14 us by whole tiles, 8 so)
  int split = 0;
  while (split < 3 && (mark_tiles(kp.n_rows) << split) < 3 * static_cast<int64_t>(c.sm_count)) ++split;
  const int ge = static_cast<int>(std::min<int64_t>(resident, mark_tiles(kp.n_rows) << split));
  kmark(c);
  km<<<gm, c.block, 0, c.stream>>>(kp, out);
  kmark(c);
  kmark(c);
  cudaError_t e = c.mark ? (ke<<<ge, ce.block, 0, c.stream>>>(kp, out, split), cudaSuccess)
                         : pdl_launch(ke, dim3(ge), dim3(ce.block), 0, c.stream, kp, out, split);
  kmark(c);
  *c.launches += 2;
  return e == cudaSuccess && cudaGetLastError() == cudaSuccess ? PV_OK : PV_ERR_CUDA;
}

template <class SH>
static pv_status launch_agg(const LaunchCfg& c, const KParams& kp, const AggOut& out) {
  using F = pv_status (*)(const LaunchCfg&, const KParams&, const AggOut&);
  static const F tab[2][2][3] = {
      {{launch_agg_t<SH, false, false, 1>, launch_agg_t<SH, false, false, 2>, launch_agg_t<SH, false, false, 4>},
       {launch_agg_t<SH, false, true, 1>, launch_agg_t<SH, false, true, 2>, launch_agg_t<SH, false, true, 4>}},
      {{launch_agg_t<SH, true, false, 1>, launch_agg_t<SH, true, false, 2>, launch_agg_t<SH, true, false, 4>},
       {launch_agg_t<SH, true, true, 1>, launch_agg_t<SH, true, true, 2>, launch_agg_t<SH, true, true, 4>}}};
  if (c.compact) return c.compact_probes != 1 ? PV_ERR_UNSUPPORTED : launch_agg_compact<SH>(c, kp, out);
  const int ui = c.U == 1 ? 0 : c.U == 2 ? 1 : c.U == 4 ? 2 : -1;
  if (ui < 0) return PV_ERR_UNSUPPORTED;
  return tab[c.pred][c.chunk][ui](c, kp, out);
}

template <class SH>
static pv_status launch_proj(const LaunchCfg& c, const KParams& kp, const ProjOut& out, int exec) {
  using F = pv_status (*)(const LaunchCfg&, const KParams&, const ProjOut&);
  static const F tab[2][2][3] = {
      {{launch_proj_sp<SH, false, false, 1>, launch_proj_sp<SH, false, false, 2>, launch_proj_sp<SH, false, false, 4>},
       {launch_proj_sp<SH, false, true, 1>, launch_proj_sp<SH, false, true, 2>, launch_proj_sp<SH, false, true, 4>}},
      {{launch_proj_sp<SH, true, false, 1>, launch_proj_sp<SH, true, false, 2>, launch_proj_sp<SH, true, false, 4>},
       {launch_proj_sp<SH, true, true, 1>, launch_proj_sp<SH, true, true, 2>, launch_proj_sp<SH, true, true, 4>}}};
  if (c.compact) return c.compact_probes != 1 ? PV_ERR_UNSUPPORTED : launch_proj_compact<SH>(c, kp, out, exec);
  const int ui = c.U == 1 ? 0 : c.U == 2 ? 1 : c.U == 4 ? 2 : -1;
  if (ui < 0) return PV_ERR_UNSUPPORTED;
  if (exec == PV_EXEC_SINGLE_PASS) return tab[c.pred][c.chunk][ui](c, kp, out);
  return c.pred ? launch_proj_ordered<SH, true>(c, kp, out) : launch_proj_ordered<SH, false>(c, kp, out);
}

template <class SH>
static void reg_aggregate() {
  ShapeEntry e{};
  e.sig = SH::signature();
  e.mode = MODE_AGGREGATE;
  e.aggregate = launch_agg<SH>;
  register_shape(e);
}
template <class SH>
static void reg_project() {
  ShapeEntry e{};
  e.sig = SH::signature();
  e.mode = MODE_PROJECT;
  e.project = launch_proj<SH>;
  register_shape(e);
}

// ---- compiled shapes -------------------------------------------------------
// Filter/aggregate/project table (a int32, b int32, price int64):
//   WHERE range(a) AND range(b) -> SUM(price), COUNT(*)   |   -> (a, price)
using ShFilterAgg = Shape<Cols<TI32, TI32, TI64>, Where<P<0>, P<1>>, Probes<>, Key<>,
                          Aggs<Sum<Mul<X<2>>>, Count>, Proj<>>;
using ShFilterProj = Shape<Cols<TI32, TI32, TI64>, Where<P<0>, P<1>>, Probes<>, Key<>, Aggs<>, Proj<0, 2>>;
// Same table, one predicate (projection query with a single filter).
using ShFilterProj1 = Shape<Cols<TI32, TI32, TI64>, Where<P<0>>, Probes<>, Key<>, Aggs<>, Proj<1, 2>>;
// Ungrouped fixed-point aggregation of the low-cardinality table (all 8
// aggregates, no grouping) — the totals of the grouped query.
using ShLowcardTotals =
    Shape<Cols<TI32, TI64, TI64, TI64, TI64>, Where<P<0>>, Probes<>, Key<>,
          Aggs<Sum<Mul<X<1>>>, Sum<Mul<X<2>>>, Sum<Mul<X<3>>>, Sum<Mul<X<4>>>, Sum<Mul<X<2>, CMX<3, 0>>>,
               Sum<Mul<X<2>, CMX<3, 1>, XPC<4, 2>>>, Sum<Mul<X<1>, X<2>>>, Count>,
          Proj<>>;
// key/value table: filtered SUM/COUNT/MIN/MAX of val.
using ShKeyValTotals = Shape<Cols<TI64>, Where<P<0>>, Probes<>, Key<>,
                             Aggs<Sum<Mul<X<0>>>, Count, Min<Mul<X<0>>>, Max<Mul<X<0>>>>, Proj<>>;

// One probe, COUNT(*) of the joining rows (join cardinality).
using ShJoinCount = Shape<Cols<TI32>, Where<>, Probes<0>, Key<>, Aggs<Count>, Proj<>>;
// Join then project: the probe's payload beside a fact column, without and
// with a fact filter in front (Table 2's pipeline shape ending in PROJECT).
using ShJoinProj = Shape<Cols<TI32, TI64>, Where<>, Probes<0>, Key<>, Aggs<>, Proj<-1, 1>>;
using ShFilterJoinProj = Shape<Cols<TI32, TI32, TI64>, Where<P<0>>, Probes<1>, Key<>, Aggs<>, Proj<-1, 2>>;

// The projection steps of the TPC-H Q5-shaped multi-pipeline query: rows
// that pass a probe, projected with their probe key (customers of the
// selected nations: key, nation), and rows that pass a filter and a probe,
// projected with the payload the probe binds (orders of the year: key, the
// customer's nation).
using ShProbeProjKey = Shape<Cols<TI32, TI32>, Where<>, Probes<0>, Key<>, Aggs<>, Proj<1, 0>>;
using ShFilterProbeProjPay = Shape<Cols<TI32, TI32, TI32>, Where<P<0>>, Probes<1>, Key<>, Aggs<>, Proj<2, -1>>;

void register_scan_shapes() {
  reg_project<ShProbeProjKey>();
  reg_project<ShFilterProbeProjPay>();
  reg_aggregate<ShJoinCount>();
  reg_aggregate<ShFilterAgg>();
  reg_project<ShFilterProj>();
  reg_project<ShFilterProj1>();
  reg_project<ShJoinProj>();
  reg_project<ShFilterJoinProj>();
  reg_aggregate<ShLowcardTotals>();
  reg_aggregate<ShKeyValTotals>();
}

// ---------------------------------------------------------------------------
// Allocation-free multi-pass projection (k_project_mark and k_project_refilter,
// branched).  Its scratch -- the error word and the match counts per tile and
// per super -- lives in one file-scope device array instead of memory from an
// allocator.  Every GPU that loads this library holds the array until the
// process exits.
// ---------------------------------------------------------------------------
namespace {

constexpr int kNoAllocBlock = 512;
constexpr int kNoAllocU = 4;
static_assert(kNoAllocBlock * kNoAllocU * 4 == kMarkTileRows, "a CTA filters one tile");
constexpr int64_t kNoAllocMaxTiles = (PV_NOALLOC_MAX_ROWS + kMarkTileRows - 1) / kMarkTileRows;
constexpr int64_t kNoAllocHeader = 32;  // words: [0] error word (int32), rest unused padding

// Scratch of every call: header, then the supers (one per 16 tiles), then the
// tiles' 32-bit counts.
__device__ __align__(256) int64_t g_noalloc_scratch[kNoAllocHeader + kNoAllocMaxTiles / 16 + 1 +
                                                    (kNoAllocMaxTiles + 1) / 2];
static_assert(kNoAllocMaxTiles >> 4 <= 2048, "supers of 16 tiles at every row count");

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
int64_t* g_noalloc_addr[kNoAllocMaxDevices];  // device address of the array, per device
int g_noalloc_sms[kNoAllocMaxDevices];

// Device address of the scratch array on the current device.  In host code
// the array's name is only a host-side stand-in, so the address is looked up
// once per device (with that device current) and cached.
pv_status noalloc_scratch(int64_t** addr, int* sms) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) return PV_ERR_CUDA;
  std::lock_guard<std::mutex> lk(g_noalloc_mu);
  if (!g_noalloc_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) return PV_ERR_CUDA;
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return PV_ERR_CUDA;
    g_noalloc_addr[dev] = static_cast<int64_t*>(p);
    g_noalloc_sms[dev] = n;
  }
  *addr = g_noalloc_addr[dev];
  *sms = g_noalloc_sms[dev];
  return PV_OK;
}

void clamp_i32_range(int64_t& lo, int64_t& hi) {
  if (lo > hi) { lo = 1; hi = 0; return; }
  lo = lo < INT32_MIN ? INT32_MIN : lo;
  hi = hi > INT32_MAX ? INT32_MAX : hi;
  if (lo > hi) { lo = 1; hi = 0; }
}

}  // namespace
}  // namespace pv

extern "C" pv_status pv_filter_project_noalloc(const int32_t* a, const int32_t* b, const int64_t* price,
                                                int64_t n_rows, int64_t a_lo, int64_t a_hi, int64_t b_lo,
                                                int64_t b_hi, int32_t* out_a, int64_t* out_price,
                                                int64_t out_capacity, int64_t* out_count, int32_t* out_status,
                                                void* stream) {
  using namespace pv;
  if (n_rows < 0 || n_rows > PV_NOALLOC_MAX_ROWS || out_capacity < 0) return PV_ERR_INVALID_ARG;
  if (!out_count || !out_status) return PV_ERR_INVALID_ARG;
  if (n_rows > 0 && (!a || !b || !price)) return PV_ERR_INVALID_ARG;
  if (out_capacity > 0 && (!out_a || !out_price)) return PV_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) | reinterpret_cast<uintptr_t>(price)) % 16)
    return PV_ERR_INVALID_ARG;
  int64_t* scratch = nullptr;
  int sms = 0;
  pv_status st = noalloc_scratch(&scratch, &sms);
  if (st != PV_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  KParams kp{};
  kp.n_rows = n_rows;
  kp.n_items = (n_rows + 3) / 4;
  kp.col[0] = a;
  kp.col[1] = b;
  kp.col[2] = price;
  clamp_i32_range(a_lo, a_hi);
  clamp_i32_range(b_lo, b_hi);
  kp.lo[0] = a_lo;
  kp.hi[0] = a_hi;
  kp.lo[1] = b_lo;
  kp.hi[1] = b_hi;
  kp.err = reinterpret_cast<int32_t*>(scratch);
  ProjOut out{};
  out.col[0] = out_a;
  out.col[1] = out_price;
  out.capacity = out_capacity;
  out.count = out_count;
  out.mark_shift = mark_shift(n_rows);
  out.mark_super = reinterpret_cast<unsigned long long*>(scratch + kNoAllocHeader);
  out.mark_count = reinterpret_cast<unsigned int*>(scratch + kNoAllocHeader + mark_super_bytes(n_rows) / 8);
  LaunchCfg c{};
  c.stream = s;
  c.sm_count = sms;
  c.block = 256;
  const bool wide = mark_wide(c, kp);
  auto km = wide ? k_project_mark<ShFilterProj, false, 4> : k_project_mark<ShFilterProj, false, 1>;
  auto ke = k_project_refilter<ShFilterProj, kNoAllocU>;
  const int gm = grid_for(c, reinterpret_cast<const void*>(km), 0, kp.n_items, int64_t(c.block) * (wide ? 4 : 1));
  LaunchCfg ce = c;
  ce.block = kNoAllocBlock;
  const int ge = grid_for(ce, reinterpret_cast<const void*>(ke), 0, mark_tiles(n_rows), 1);
  if (gm <= 0 || ge <= 0) return PV_ERR_UNSUPPORTED;
  // the array keeps the previous call's contents: clear the error word and the counts
  if (cudaMemsetAsync(scratch, 0, kNoAllocHeader * 8 + mark_count_bytes(n_rows), s) != cudaSuccess) return PV_ERR_CUDA;
  km<<<gm, c.block, 0, s>>>(kp, out);
  if (pdl_launch(ke, dim3(ge), dim3(kNoAllocBlock), 0, s, kp, out) != cudaSuccess) return PV_ERR_CUDA;
  if (cudaGetLastError() != cudaSuccess) return PV_ERR_CUDA;
  if (cudaMemcpyAsync(out_status, scratch, sizeof(int32_t), cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return PV_ERR_CUDA;
  return PV_OK;
}
