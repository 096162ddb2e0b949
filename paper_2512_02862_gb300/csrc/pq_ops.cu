// pq_ops.cu -- standalone operators: filter, radix partition, hash-join
// build/probe, group-by SUM, top-k.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>

#include "pq_internal.h"
#include "pq_topk.cuh"

using namespace pqk;
using pqh::S;

namespace {

// ============================================================== filter ====
// Tile of 4096 elements: 8 warps x 512; lane l of warp w reads elements
// w*512 + g*128 + 4l + {0..3} for g = 0..3 (row order = element order), so a
// warp-wide load instruction covers 512 contiguous bytes of an int32 column.
constexpr int kFilterTile = 4096;

template <typename T, bool VEC>
__device__ __forceinline__ void load4(const T* __restrict__ col, i64 e0, i64 n, i64 v[4]) {
  if (VEC && e0 + 4 <= n) {
    if constexpr (sizeof(T) == 4) {
      int4 q = ld_stream(reinterpret_cast<const int4*>(col + e0));
      v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
    } else if constexpr (sizeof(T) == 8) {
      longlong2 a = ld_stream(reinterpret_cast<const longlong2*>(col + e0));
      longlong2 b = ld_stream(reinterpret_cast<const longlong2*>(col + e0 + 2));
      v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
    } else {
      char4 q = ld_stream(reinterpret_cast<const char4*>(col + e0));
      v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
    }
  } else {
#pragma unroll
    for (int s = 0; s < 4; ++s) v[s] = e0 + s < n ? (i64)ld_stream(col + e0 + s) : 0;
  }
}

template <typename T, bool SEL, bool VEC>
__global__ void __launch_bounds__(256) k_filter(const T* __restrict__ col,
                                                const i64* __restrict__ sel_in, i64 n_cap,
                                                const i64* d_n, Pred p, i64* __restrict__ out,
                                                i64* d_count, u64* state, u32* tile_ctr,
                                                i64 spin_limit, DevStatus* st) {
  __shared__ i64 s_tile;
  __shared__ u32 s_w[8];
  __shared__ i64 s_prefix;
  const i64 n = d_n ? min(*d_n, n_cap) : n_cap;
  const i64 ntiles = (n + kFilterTile - 1) / kFilterTile;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  while (true) {
    if (threadIdx.x == 0) s_tile = atomicAdd(tile_ctr, 1u);
    __syncthreads();
    const i64 tile = s_tile;
    if (tile >= ntiles) break;
    const i64 wbase = tile * kFilterTile + warp * 512;
    u32 bits = 0;
    i64 rows[16];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const i64 e0 = wbase + g * 128 + lane * 4;
      i64 v[4];
      if (SEL) {
        i64 r[4];
        load4<i64, VEC>(sel_in, e0, n, r);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          rows[g * 4 + s] = r[s];
          v[s] = e0 + s < n ? (i64)__ldg(col + r[s]) : 0;
        }
      } else {
        load4<T, VEC>(col, e0, n, v);
#pragma unroll
        for (int s = 0; s < 4; ++s) rows[g * 4 + s] = e0 + s;
      }
#pragma unroll
      for (int s = 0; s < 4; ++s)
        if (e0 + s < n && pass(p, v[s])) bits |= 1u << (g * 4 + s);
    }
    // Per-group counts packed in 16-bit fields: one warp scan covers 4 groups.
    u64 packed = 0;
#pragma unroll
    for (int g = 0; g < 4; ++g) packed |= (u64)__popc((bits >> (4 * g)) & 0xFu) << (16 * g);
    u64 incl = packed;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      u64 y = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += y;
    }
    const u64 wt = __shfl_sync(kFull, incl, 31);
    const u64 excl = incl - packed;
    if (lane == 0)
      s_w[warp] = (u32)((wt & 0xFFFF) + ((wt >> 16) & 0xFFFF) + ((wt >> 32) & 0xFFFF) + (wt >> 48));
    __syncthreads();
    if (warp == 0) {
      const int nw = blockDim.x >> 5;
      u32 c = lane < nw ? s_w[lane] : 0, x = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        u32 y = __shfl_up_sync(kFull, x, o);
        if (lane >= o) x += y;
      }
      const u32 total = __shfl_sync(kFull, x, 31);
      const i64 prefix = lookback_prefix(state, tile, total, spin_limit, st);
      if (lane < nw) s_w[lane] = x - c;
      if (lane == 0) {
        s_prefix = prefix;
        if (tile == ntiles - 1) *d_count = prefix + total;
      }
    }
    __syncthreads();
    i64 pos = s_prefix + s_w[warp];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const u32 bg = (bits >> (4 * g)) & 0xFu;
      i64 at = pos + (i64)((excl >> (16 * g)) & 0xFFFF);
#pragma unroll
      for (int s = 0; s < 4; ++s)
        if (bg & (1u << s)) {
          if (at < n_cap) out[at] = rows[g * 4 + s];
          ++at;
        }
      pos += (i64)((wt >> (16 * g)) & 0xFFFF);
    }
    __syncthreads();
  }
}

// The operator's selection: two passes with no chain between blocks, the
// column read once.  A warp owns a contiguous run of 512-row warp tiles (16
// rows per lane).  Pass 1 tests the rows, keeps each lane's 16 predicate bits
// as one u16 (n / 8 bytes in all) and counts per warp and per block.  Pass 2
// takes the same warp tiles: a block sums the counts of the blocks before it
// (one load per block, shared by its threads), a warp adds
// those of the warps before it, and from then on a warp needs only its own
// bits: it orders the passing rows of a tile in shared memory and writes them
// as one contiguous run.  Pass 1 is bound by reading the column, pass 2 by
// writing the ids.  In a stream that is being captured, whose scratch is kept
// for the graph's replays, pass 1 keeps only the counts (36 bytes per block)
// and pass 2 tests the rows again.  60M int32 rows, 31.5M ids out (0.49 GB):
// 0.188 ms with a second read of the column, a scan launch between the passes
// and each lane writing its own ids (runs with gaps: sectors written in four
// parts); 0.042 + 0.048 ms like this, 5.4 TB/s.
constexpr int kWarpTile = 512;
// Resident blocks per SM: 6 leave 40 registers a thread, enough for the 16
// values of a narrow column; wide ones and row ids take 4.
__host__ __device__ constexpr int filter_blocks(bool wide) { return wide ? 4 : 6; }
constexpr int kFilterOne = 32;     // warp tiles one block does in a single launch

// Four elements from e0 on (rows at or beyond n read as 0).
template <typename T, bool VEC, bool FULL>
__device__ __forceinline__ void load4t(const T* __restrict__ col, i64 e0, i64 n, T v[4]) {
  if (VEC && (FULL || e0 + 4 <= n)) {
    if constexpr (sizeof(T) == 8) {
      const longlong2 a = ld_stream(reinterpret_cast<const longlong2*>(col + e0));
      const longlong2 b = ld_stream(reinterpret_cast<const longlong2*>(col + e0 + 2));
      v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
    } else if constexpr (sizeof(T) == 4) {
      const int4 q = ld_stream(reinterpret_cast<const int4*>(col + e0));
      v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
    } else {
      const char4 q = ld_stream(reinterpret_cast<const char4*>(col + e0));
      v[0] = q.x, v[1] = q.y, v[2] = q.z, v[3] = q.w;
    }
  } else {
#pragma unroll
    for (int s = 0; s < 4; ++s) v[s] = FULL || e0 + s < n ? ld_stream(col + e0 + s) : T(0);
  }
}

// The predicate in the column's own width: a 32-bit range test for the
// narrow types.
template <typename T>
struct PredT {
  Pred p;
  __device__ explicit PredT(const Pred& q) : p(q) {}
  __device__ __forceinline__ bool operator()(T v) const { return pass(p, (i64)v); }
};
template <>
struct PredT<int> {
  Pred32 p;
  __device__ explicit PredT(const Pred& q) : p(to32(q)) {}
  __device__ __forceinline__ bool operator()(int v) const { return pass32(p, v); }
};
template <>
struct PredT<signed char> : PredT<int> {
  using PredT<int>::PredT;
};

// The predicate bits of a lane's 16 rows of a warp tile: bit g * 4 + s is row
// base + g * 128 + 4 * lane + s.  All of a tile's loads are independent.
template <typename T, bool SEL, bool VEC, bool FULL>
__device__ __forceinline__ u32 filter_bits_t(const T* __restrict__ col,
                                             const i64* __restrict__ sel_in, i64 n,
                                             const PredT<T>& p, i64 base) {
  const int lane = threadIdx.x & 31;
  T v[16];
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const i64 e0 = base + g * 128 + lane * 4;
    if (SEL) {
      i64 r[4];
      load4t<i64, VEC, FULL>(sel_in, e0, n, r);
#pragma unroll
      for (int s = 0; s < 4; ++s) v[g * 4 + s] = FULL || e0 + s < n ? __ldg(col + r[s]) : T(0);
    } else {
      load4t<T, VEC, FULL>(col, e0, n, v + g * 4);
    }
  }
  u32 bits = 0;
#pragma unroll
  for (int j = 0; j < 16; ++j)
    bits |= (u32)((FULL || base + (j >> 2) * 128 + lane * 4 + (j & 3) < n) && p(v[j])) << j;
  return bits;
}
template <typename T, bool SEL, bool VEC>
__device__ __forceinline__ u32 filter_bits(const T* __restrict__ col,
                                           const i64* __restrict__ sel_in, i64 n,
                                           const PredT<T>& p, i64 base) {
  return base + kWarpTile <= n ? filter_bits_t<T, SEL, VEC, true>(col, sel_in, n, p, base)
                               : filter_bits_t<T, SEL, VEC, false>(col, sel_in, n, p, base);
}

// Orders the passing rows of a warp tile in the warp's stage (offsets within
// the tile) and writes them from `pos` on; returns their number.
template <bool SEL>
__device__ __forceinline__ u32 filter_emit_tile(u32 bits, i64 base, const i64* __restrict__ sel_in,
                                                unsigned short* stage, i64* __restrict__ out,
                                                i64 pos) {
  const int lane = threadIdx.x & 31;
  // Per-group counts packed in 16-bit fields: one warp scan covers 4 groups.
  u64 packed = 0;
#pragma unroll
  for (int g = 0; g < 4; ++g) packed |= (u64)__popc((bits >> (4 * g)) & 0xFu) << (16 * g);
  u64 incl = packed;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u64 y = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += y;
  }
  const u64 wt = __shfl_sync(kFull, incl, 31), excl = incl - packed;
  u32 first = 0;  // first place of the group
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    u32 at = first + (u32)((excl >> (16 * g)) & 0xFFFF);
#pragma unroll
    for (int s = 0; s < 4; ++s)
      if ((bits >> (4 * g + s)) & 1u) stage[at++] = (unsigned short)(g * 128 + lane * 4 + s);
    first += (u32)((wt >> (16 * g)) & 0xFFFF);
  }
  __syncwarp();
  for (u32 j = lane; j < first; j += 32) {
    const i64 e = base + stage[j];
    __stcs(out + pos + j, SEL ? __ldg(sel_in + e) : e);
  }
  __syncwarp();
  return first;
}

// Warp tiles of warp gw of nw: a contiguous, even share.
__device__ __forceinline__ i64 filter_share(i64 ntiles, i64 nw, i64 gw) {
  return ntiles / nw * gw + min(gw, ntiles % nw);
}

template <typename T, bool SEL, bool VEC>
__global__ void __launch_bounds__(256, filter_blocks(SEL || sizeof(T) == 8))
    k_filter_mark(const T* __restrict__ col, const i64* __restrict__ sel_in, i64 n_cap,
                  const i64* d_n, Pred p, unsigned short* __restrict__ bits_out,
                  u32* __restrict__ warp_cnt, u32* __restrict__ block_cnt) {
  __shared__ u32 s_w[8];
  const i64 n = d_n ? min(*d_n, n_cap) : n_cap;
  const i64 ntiles = (n + kWarpTile - 1) / kWarpTile, nw = (i64)gridDim.x * 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const i64 gw = (i64)blockIdx.x * 8 + warp;
  const i64 t1 = filter_share(ntiles, nw, gw + 1);
  const PredT<T> pt(p);
  u32 cnt = 0;
  for (i64 t = filter_share(ntiles, nw, gw); t < t1; ++t) {
    const u32 bits = filter_bits<T, SEL, VEC>(col, sel_in, n, pt, t * kWarpTile);
    if (bits_out) bits_out[t * 32 + lane] = (unsigned short)bits;
    cnt += __popc(bits);
  }
  cnt = __reduce_add_sync(kFull, cnt);
  if (lane == 0) s_w[warp] = cnt, warp_cnt[gw] = cnt;
  __syncthreads();
  if (threadIdx.x == 0) {
    u32 t = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) t += s_w[w];
    block_cnt[blockIdx.x] = t;
  }
}

// Pass 2 of a block; bits_of(t): the lane's bits of warp tile t, asked for one
// tile ahead.
template <bool SEL, typename F>
__device__ __forceinline__ void filter_emit(const i64* __restrict__ sel_in, i64 n,
                                            const u32* __restrict__ warp_cnt,
                                            const u32* __restrict__ block_cnt,
                                            i64* __restrict__ out, i64* d_count, F bits_of) {
  __shared__ unsigned short s_stage[8][kWarpTile];
  __shared__ u64 s_before;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) s_before = 0;
  __syncthreads();
  u64 before = 0;  // ids of the blocks before this one
  for (int j = threadIdx.x; j < (int)blockIdx.x; j += 256) before += __ldg(block_cnt + j);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(kFull, before, o);
  if (lane == 0 && before) atomicAdd((unsigned long long*)&s_before, (unsigned long long)before);
  __syncthreads();
  const i64 ntiles = (n + kWarpTile - 1) / kWarpTile, nw = (i64)gridDim.x * 8;
  const i64 gw = (i64)blockIdx.x * 8 + warp;
  i64 pos = (i64)s_before;
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *d_count = pos + block_cnt[blockIdx.x];
  for (int w = 0; w < warp; ++w) pos += __ldg(warp_cnt + (i64)blockIdx.x * 8 + w);
  const i64 t1 = filter_share(ntiles, nw, gw + 1);
  i64 t = filter_share(ntiles, nw, gw);
  u32 next = t < t1 ? bits_of(t) : 0;
  for (; t < t1; ++t) {
    const u32 bits = next;
    if (t + 1 < t1) next = bits_of(t + 1);
    pos += filter_emit_tile<SEL>(bits, t * kWarpTile, sel_in, s_stage[warp], out, pos);
  }
}

template <bool SEL>
__global__ void __launch_bounds__(256, filter_blocks(false))
    k_filter_emit(const i64* __restrict__ sel_in, i64 n_cap, const i64* d_n,
                  const unsigned short* __restrict__ bits_in, const u32* __restrict__ warp_cnt,
                  const u32* __restrict__ block_cnt, i64* __restrict__ out, i64* d_count) {
  const i64 n = d_n ? min(*d_n, n_cap) : n_cap;
  filter_emit<SEL>(sel_in, n, warp_cnt, block_cnt, out, d_count,
                   [&](i64 t) -> u32 { return __ldg(bits_in + t * 32 + (threadIdx.x & 31)); });
}

// Pass 2 without kept bits: the rows are tested again.
template <typename T, bool SEL, bool VEC>
__global__ void __launch_bounds__(256, filter_blocks(SEL || sizeof(T) == 8))
    k_filter_again(const T* __restrict__ col, const i64* __restrict__ sel_in, i64 n_cap,
                   const i64* d_n, Pred p, const u32* __restrict__ warp_cnt,
                   const u32* __restrict__ block_cnt, i64* __restrict__ out, i64* d_count) {
  const i64 n = d_n ? min(*d_n, n_cap) : n_cap;
  const PredT<T> pt(p);
  filter_emit<SEL>(sel_in, n, warp_cnt, block_cnt, out, d_count, [&](i64 t) -> u32 {
    return filter_bits<T, SEL, VEC>(col, sel_in, n, pt, t * kWarpTile);
  });
}

// Few rows (kFilterOne warp tiles): both passes in one block and one launch,
// no scratch.
template <typename T, bool SEL, bool VEC>
__global__ void __launch_bounds__(kFilterOne * 32)
    k_filter_one(const T* __restrict__ col, const i64* __restrict__ sel_in, i64 n_cap,
                 const i64* d_n, Pred p, i64* __restrict__ out, i64* d_count) {
  __shared__ unsigned short s_stage[kFilterOne][kWarpTile];
  const i64 n = d_n ? min(*d_n, n_cap) : n_cap;
  const int warp = threadIdx.x >> 5;
  const i64 base = (i64)warp * kWarpTile;
  const u32 bits = base < n ? filter_bits<T, SEL, VEC>(col, sel_in, n, PredT<T>(p), base) : 0u;
  const u32 cnt = __reduce_add_sync(kFull, (u32)__popc(bits));
  const u32 before = block_exclusive_sum((threadIdx.x & 31) == 0 ? cnt : 0u);
  const u32 pos = __shfl_sync(kFull, before, 0);
  if (threadIdx.x == blockDim.x - 1) *d_count = (i64)pos + cnt;
  if (cnt) filter_emit_tile<SEL>(bits, base, sel_in, s_stage[warp], out, (i64)pos);
}

// =========================================================== partition ====
// 8192 rows per tile; warp w owns rows w*1024 .. w*1024+1023 of the tile and
// walks them in 32 steps of 32 rows, so ranks assigned in step order keep the
// input order inside every bucket.
constexpr int kPartTile = 8192;

template <typename T>
__global__ void __launch_bounds__(256) k_part_hist(const T* __restrict__ key, i64 n, int log2P,
                                                   u32* __restrict__ hist, i64 ntiles) {
  extern __shared__ u32 sh[];
  const int P = 1 << log2P;
  for (int b = threadIdx.x; b < P; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const i64 tile = blockIdx.x;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const i64 base = tile * kPartTile + warp * 1024;
  for (int s = 0; s < 32; ++s) {
    const i64 r = base + s * 32 + lane;
    const bool valid = r < n;
    const u32 b = valid ? fib_bucket((i64)__ldg(key + r), log2P) : 0xFFFFFFFFu;
    const u32 peers = __match_any_sync(kFull, b);
    if (valid && lane == __ffs(peers) - 1) atomicAdd(&sh[b], (u32)__popc(peers));
  }
  __syncthreads();
  for (int b = threadIdx.x; b < P; b += blockDim.x) hist[(i64)b * ntiles + tile] = sh[b];
}

// Exclusive scan of a u32 array into i64 (single pass, decoupled look-back).
__global__ void __launch_bounds__(256) k_scan_u32(const u32* __restrict__ in, i64 n,
                                                  i64* __restrict__ out, u64* state,
                                                  u32* tile_ctr, i64 spin_limit, DevStatus* st) {
  __shared__ i64 s_tile;
  __shared__ i64 s_w[8];
  __shared__ i64 s_prefix;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const i64 ntiles = (n + 4095) / 4096;
  while (true) {
    if (threadIdx.x == 0) s_tile = atomicAdd(tile_ctr, 1u);
    __syncthreads();
    const i64 tile = s_tile;
    if (tile >= ntiles) break;
    const i64 e0 = tile * 4096 + threadIdx.x * 16;
    u32 v[16];
    i64 sum = 0;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      v[j] = e0 + j < n ? in[e0 + j] : 0u;
      sum += v[j];
    }
    i64 x = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      i64 y = __shfl_up_sync(kFull, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_w[warp] = x;
    __syncthreads();
    if (warp == 0) {
      const int nw = blockDim.x >> 5;
      i64 c = lane < nw ? s_w[lane] : 0, y = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        i64 z = __shfl_up_sync(kFull, y, o);
        if (lane >= o) y += z;
      }
      const i64 total = __shfl_sync(kFull, y, 31);
      const i64 prefix = lookback_prefix(state, tile, total, spin_limit, st);
      if (lane < nw) s_w[lane] = y - c;
      if (lane == 0) s_prefix = prefix;
    }
    __syncthreads();
    i64 run = s_prefix + s_w[warp] + (x - sum);
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      if (e0 + j < n) out[e0 + j] = run;
      run += v[j];
    }
    __syncthreads();
  }
}

struct PayArgs {
  const void* src[PQ_MAX_PAYLOAD];
  void* dst[PQ_MAX_PAYLOAD];
  int type[PQ_MAX_PAYLOAD];
  int n;
};

__device__ __forceinline__ void copy_elem(int type, const void* src, void* dst, i64 from, i64 to) {
  if (type == PQ_INT64) ((i64*)dst)[to] = __ldg((const i64*)src + from);
  else if (type == PQ_INT32) ((int*)dst)[to] = __ldg((const int*)src + from);
  else ((signed char*)dst)[to] = __ldg((const signed char*)src + from);
}

template <typename T>
__global__ void __launch_bounds__(256) k_part_scatter(const T* __restrict__ key, i64 n, int log2P,
                                                      const i64* __restrict__ gofs, i64 ntiles,
                                                      PayArgs pa, T* __restrict__ out_key,
                                                      i64* d_offsets) {
  extern __shared__ u32 wc[];  // [8][P]: per-warp counts, then per-warp bases
  const int P = 1 << log2P;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  for (int b = threadIdx.x; b < nw * P; b += blockDim.x) wc[b] = 0;
  __syncthreads();
  const i64 tile = blockIdx.x;
  const i64 base = tile * kPartTile + warp * 1024;
  for (int s = 0; s < 32; ++s) {
    const i64 r = base + s * 32 + lane;
    const bool valid = r < n;
    const u32 b = valid ? fib_bucket((i64)__ldg(key + r), log2P) : 0xFFFFFFFFu;
    const u32 peers = __match_any_sync(kFull, b);
    if (valid && lane == __ffs(peers) - 1) wc[warp * P + b] += (u32)__popc(peers);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < P; b += blockDim.x) {
    u32 run = 0;
    for (int w = 0; w < nw; ++w) {
      const u32 c = wc[w * P + b];
      wc[w * P + b] = run;
      run += c;
    }
    if (tile == 0) d_offsets[b] = gofs[(i64)b * ntiles];
  }
  if (tile == 0 && threadIdx.x == 0) d_offsets[P] = n;
  __syncthreads();
  for (int s = 0; s < 32; ++s) {
    const i64 r = base + s * 32 + lane;
    const bool valid = r < n;
    const T k = valid ? __ldg(key + r) : T(0);
    const u32 b = valid ? fib_bucket((i64)k, log2P) : 0xFFFFFFFFu;
    const u32 peers = __match_any_sync(kFull, b);
    if (valid) {
      const i64 pos = __ldg(gofs + (i64)b * ntiles + tile) + wc[warp * P + b] +
                      __popc(peers & lanemask_lt());
      if (pos >= n) continue;  // only after a timed-out scan; never in a correct run
      out_key[pos] = k;
      for (int j = 0; j < pa.n; ++j) copy_elem(pa.type[j], pa.src[j], pa.dst[j], r, pos);
    }
    __syncwarp();
    if (valid && lane == __ffs(peers) - 1) wc[warp * P + b] += (u32)__popc(peers);
    __syncwarp();
  }
}

// ------------------------------------------------- staged partition ----
// For fan-outs up to 2^kStagedMaxLog2: persistent blocks, block k taking the
// contiguous rows [k * n / G, (k + 1) * n / G).  The histogram is then one
// count per (bucket, block), so the scan and the per-bucket cursor reads are
// small.  Each block walks its rows in sub-tiles of kSub: warp w takes rows
// w * kSubWarpRows .. of the sub-tile in steps of 32, which fixes every
// row's place in the sub-tile sorted by (bucket, input order); each
// column is then staged in shared memory in that order and every bucket's
// run is written with consecutive threads on consecutive rows.  Within a
// bucket the order is input order: blocks in block order, sub-tiles in
// order, warps in order, steps in order, lanes in order.
constexpr int kStagedMaxLog2 = 10;
constexpr int kSub = 2048;
constexpr int kSubWarpRows = kSub / 8;     // rows of a warp in a sub-tile
constexpr int kSubSteps = kSubWarpRows / 32;

// What a pass orders by: the whole bucket number of log2P bits, or (PART, a
// partition in two passes) `bits` bits of it from `shift` on.  One multiply and
// shift per key, and a mask for a part: 4-byte rows are bound by instructions,
// and a mask on the whole number cost them 2 %.
template <bool PART>
struct Digit {
  int log2P, bits, rshift;
  u32 mask;
  Digit() = default;
  __host__ __device__ Digit(int log2P_, int shift, int bits_)
      : log2P(log2P_), bits(bits_), rshift(log2P_ ? 64 - log2P_ + shift : 63),
        mask((1u << bits_) - 1u) {}
  __host__ __device__ int count() const { return 1 << bits; }
  __device__ __forceinline__ u32 operator()(i64 k) const {
    if constexpr (!PART) return fib_bucket(k, log2P);
    return (u32)(((u64)k * 0x9E3779B97F4A7C15ULL) >> rshift) & mask;
  }
};

// Lanes of the warp whose bucket equals this lane's, from one ballot per
// bucket bit (all lanes taking part): cheaper than a general match for small
// bucket ids.  nbits = log2P when every lane holds a row; otherwise
// log2P + 1, an invalid lane passing a bucket of its own, 2^log2P.
__device__ __forceinline__ u32 bucket_peers(u32 b, int nbits) {
  u32 peers = kFull;
#pragma unroll
  for (int k = 0; k <= kStagedMaxLog2; ++k) {
    if (k >= nbits) break;  // warp-uniform
    const u32 m = __ballot_sync(kFull, (b >> k) & 1u);
    peers &= (b >> k) & 1u ? m : ~m;
  }
  return peers;
}

// First row of block k's chunk: a multiple of 16 rows (so that every column's
// slice starts on a 16-byte boundary for the bulk copies), n for k = g.
__host__ __device__ inline i64 chunk_begin(i64 n, i64 g, i64 k) {
  if (k >= g) return n;
  const i64 r = (i64)((__int128)n * k / g + 15) & ~(i64)15;
  return r < n ? r : n;
}

// Histogram of the scatter's chunks: hsplit blocks per chunk (chunk k =
// blockIdx.x / hsplit), each counting a share of the chunk's rows and adding
// its counts into hist[b * g + k] (zeroed before).
template <typename T, bool PART, bool TOT>
__global__ void __launch_bounds__(256, 8) k_part_hist_blk(const T* __restrict__ key, i64 n,
                                                          Digit<PART> dg, u32* __restrict__ hist,
                                                          i64 g, int hsplit,
                                                          u64* __restrict__ tot) {
  extern __shared__ u32 sh[];
  // TOT (the first of two passes): whole buckets are counted, into tot (over
  // all rows: 64 bits) and, added up by digit, into hist.
  const int P = TOT ? 1 << dg.log2P : dg.count();
  auto cd = [&](i64 k) { return TOT ? fib_bucket(k, dg.log2P) : dg(k); };
  for (int b = threadIdx.x; b < P; b += blockDim.x) sh[b] = 0;
  __syncthreads();
  const i64 k = blockIdx.x / hsplit, h = blockIdx.x % hsplit;
  const i64 c0 = chunk_begin(n, g, k), c1 = chunk_begin(n, g, k + 1);
  auto cut = [&](i64 x) { return x >= hsplit ? c1 : min(c1, c0 + (((c1 - c0) * x / hsplit + 15) & ~15LL)); };
  const i64 r0 = cut(h), r1 = cut(h + 1);  // 16-row aligned shares
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kPerVec = 16 / sizeof(T);    // keys per 16-byte load
  constexpr int kLd = 4;                     // 16-byte loads per lane per step
  constexpr int kRows = kLd * 32 * kPerVec;  // rows of a warp step
  // Whole warp steps (kRows consecutive rows: kLd loads of 16 bytes per
  // lane, issued together, then counted with no bounds tests) while the
  // share's start is 16-byte aligned; the rest row by row.
  const bool vec = ((uintptr_t)(key + r0) & 15) == 0;
  const i64 steps = vec ? (r1 - r0) / kRows : 0;
  for (i64 st = warp; st < steps; st += 8) {  // warp-uniform
    const uint4* p = reinterpret_cast<const uint4*>(key + r0 + st * kRows);
    uint4 x[kLd];
#pragma unroll
    for (int j = 0; j < kLd; ++j) x[j] = __ldcs(p + j * 32 + lane);
#pragma unroll
    for (int j = 0; j < kLd; ++j) {
      T v[kPerVec];
      memcpy(v, &x[j], 16);
#pragma unroll
      for (int e = 0; e < kPerVec; ++e) atomicAdd(&sh[cd((i64)v[e])], 1u);
    }
  }
  for (i64 i = r0 + steps * kRows + threadIdx.x; i < r1; i += blockDim.x)
    atomicAdd(&sh[cd((i64)__ldg(key + i))], 1u);
  __syncthreads();
  if (!TOT) {
    for (int b = threadIdx.x; b < P; b += blockDim.x)
      if (sh[b]) atomicAdd(&hist[(i64)b * g + k], sh[b]);
    return;
  }
  for (int b = threadIdx.x; b < P; b += blockDim.x)
    if (sh[b]) atomicAdd((unsigned long long*)&tot[b], (unsigned long long)sh[b]);
  // Lane l of a warp adds up a digit's buckets l, l + 32, ...
  for (int d = warp; d < dg.count(); d += 8) {
    u32 c = 0;
    for (int o = lane; o < P >> dg.bits; o += 32) c += sh[(o << dg.bits) | d];  // shift 0
    c = __reduce_add_sync(kFull, c);
    if (lane == 0 && c) atomicAdd(&hist[(i64)d * g + k], c);
  }
}

// The buckets' offsets from their counts (P <= 4096: four per thread), n last.
// One block.
__global__ void __launch_bounds__(1024) k_part_offsets(const u64* __restrict__ tot, int P, i64 n,
                                                       i64* __restrict__ out) {
  __shared__ i64 s_w[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b0 = threadIdx.x * 4;
  i64 v[4], sum = 0;
#pragma unroll
  for (int j = 0; j < 4; ++j) v[j] = b0 + j < P ? (i64)tot[b0 + j] : 0, sum += v[j];
  i64 x = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const i64 y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s_w[warp] = x;
  __syncthreads();
  i64 run = x - sum;
  for (int w = 0; w < warp; ++w) run += s_w[w];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (b0 + j < P) out[b0 + j] = run;
    run += v[j];
  }
  if (threadIdx.x == 0) out[P] = n;
}

// Shared memory of the staged scatter for P buckets (bytes).
__host__ __device__ inline size_t staged_smem(int P) {
  return (size_t)P * 8        // s_gb: global cursor per bucket
         + (size_t)8 * P * 4  // s_cnt: per-warp counts, then per-warp offsets
         + (size_t)P * 4      // s_run: run start of each bucket in the sub-tile
         + (size_t)P * 4      // s_tot: the sub-tile's rows per bucket
         + (size_t)kSub * 8   // s_stage: one column of the sub-tile, sorted
         + (size_t)kSub * 2   // s_lpos: sorted place of each row
         + (size_t)kSub * 2;  // s_sbk: bucket of each sorted place
}

// One column of a sub-tile: each thread issues its 16 loads before it uses
// any of them, places the values in sorted order in shared memory, then
// writes sorted places i = thread, thread + 256, ... to their runs.
template <typename V>
__device__ __forceinline__ void stage_column(const V* __restrict__ src, V* __restrict__ dst,
                                             i64 r, int cnt, const unsigned short* s_lpos,
                                             const unsigned short* s_sbk, const u32* s_run,
                                             const i64* s_gb, V* s_stage) {
  constexpr int kPer = kSub / 256;
  V v[kPer];
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int i = j * 256 + (int)threadIdx.x;
    v[j] = i < cnt ? __ldcs(src + r + i) : V(0);
  }
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int i = j * 256 + (int)threadIdx.x;
    if (i < cnt) s_stage[s_lpos[i]] = v[j];
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int i = j * 256 + (int)threadIdx.x;
    if (i < cnt) {
      const u32 b = s_sbk[i];
      __stcs(dst + s_gb[b] + (i - (i64)s_run[b]), s_stage[i]);
    }
  }
  __syncthreads();
}

template <typename T, bool PART>
__global__ void __launch_bounds__(256) k_part_scatter_blk(const T* __restrict__ key, i64 n,
                                                          Digit<PART> dg, const i64* __restrict__ gofs,
                                                          PayArgs pa, T* __restrict__ out_key,
                                                          i64* d_offsets) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int log2P = dg.bits, P = 1 << log2P;
  i64* s_gb = reinterpret_cast<i64*>(smem);
  u32* s_cnt = reinterpret_cast<u32*>(s_gb + P);
  u32* s_run = s_cnt + 8 * P;
  u32* s_tot = s_run + P;
  u64* s_stage = reinterpret_cast<u64*>(s_tot + P);
  unsigned short* s_lpos = reinterpret_cast<unsigned short*>(s_stage + kSub);
  unsigned short* s_sbk = s_lpos + kSub;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const i64 g = gridDim.x, k = blockIdx.x;
  const i64 r0 = chunk_begin(n, g, k), r1 = chunk_begin(n, g, k + 1);
  for (int b = threadIdx.x; b < P; b += blockDim.x) {
    s_gb[b] = gofs[(i64)b * g + k];
    if (k == 0 && d_offsets) d_offsets[b] = s_gb[b];
  }
  if (k == 0 && threadIdx.x == 0 && d_offsets) d_offsets[P] = n;
  for (i64 r = r0; r < r1; r += kSub) {
    const int cnt = (int)min((i64)kSub, r1 - r);
    for (int b = threadIdx.x; b < 8 * P; b += blockDim.x) s_cnt[b] = 0;
    __syncthreads();
    // Bucket and place within the warp's rows of each of the lane's rows
    // (the keys loaded first, so that their loads are in flight together).
    const int nbits = cnt == kSub ? log2P : log2P + 1;  // every lane holds a row?
    u32 bp[kSubSteps];  // bucket << 9 | place among the warp's rows of that bucket
#pragma unroll
    for (int st = 0; st < kSubSteps; ++st) {
      const int i = warp * kSubWarpRows + st * 32 + lane;
      bp[st] = i < cnt ? dg((i64)__ldg(key + r + i)) : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int st = 0; st < kSubSteps; ++st) {
      const bool valid = bp[st] != 0xFFFFFFFFu;
      const u32 b = bp[st];
      const u32 peers = bucket_peers(valid ? b : (1u << log2P), nbits);
      u32 place = 0;
      if (valid) place = s_cnt[warp * P + b] + __popc(peers & lanemask_lt());
      __syncwarp();
      if (valid && lane == __ffs(peers) - 1) s_cnt[warp * P + b] += (u32)__popc(peers);
      __syncwarp();
      bp[st] = valid ? b << 9 | place : 0xFFFFFFFFu;
    }
    __syncthreads();
    static_assert(kSubWarpRows <= 512, "place takes 9 bits");
    // Per bucket: offsets of the warps' rows, the sub-tile's total.
    for (int b = threadIdx.x; b < P; b += blockDim.x) {
      u32 run = 0;
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        const u32 c = s_cnt[w * P + b];
        s_cnt[w * P + b] = run;
        run += c;
      }
      s_tot[b] = run;
    }
    __syncthreads();
    {  // run starts: exclusive scan of the totals (P <= 4 * 256)
      static_assert((1 << kStagedMaxLog2) <= 4 * 256, "four buckets per thread");
      u32 v[4], sum = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int b = (int)threadIdx.x * 4 + j;
        v[j] = b < P ? s_tot[b] : 0u;
        sum += v[j];
      }
      u32 run = block_exclusive_sum(sum);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int b = (int)threadIdx.x * 4 + j;
        if (b < P) s_run[b] = run;
        run += v[j];
      }
    }
    __syncthreads();
#pragma unroll
    for (int st = 0; st < kSubSteps; ++st) {
      if (bp[st] == 0xFFFFFFFFu) continue;
      const u32 b = bp[st] >> 9;
      const int i = warp * kSubWarpRows + st * 32 + lane;
      const u32 at = s_run[b] + s_cnt[warp * P + b] + (bp[st] & 511u);
      s_lpos[i] = (unsigned short)at;
      s_sbk[at] = (unsigned short)b;
    }
    __syncthreads();
    stage_column<T>(key, out_key, r, cnt, s_lpos, s_sbk, s_run, s_gb,
                    reinterpret_cast<T*>(s_stage));
    for (int j = 0; j < pa.n; ++j) {
      if (pa.type[j] == PQ_INT64)
        stage_column<i64>((const i64*)pa.src[j], (i64*)pa.dst[j], r, cnt, s_lpos, s_sbk, s_run,
                          s_gb, reinterpret_cast<i64*>(s_stage));
      else if (pa.type[j] == PQ_INT32)
        stage_column<int>((const int*)pa.src[j], (int*)pa.dst[j], r, cnt, s_lpos, s_sbk, s_run,
                          s_gb, reinterpret_cast<int*>(s_stage));
      else
        stage_column<signed char>((const signed char*)pa.src[j], (signed char*)pa.dst[j], r, cnt,
                                  s_lpos, s_sbk, s_run, s_gb,
                                  reinterpret_cast<signed char*>(s_stage));
    }
    for (int b = threadIdx.x; b < P; b += blockDim.x) s_gb[b] += s_tot[b];
    __syncthreads();
  }
}

// The staged scatter with its sub-tiles brought into shared memory by bulk
// copies (TMA), double-buffered: while the block orders and writes sub-tile
// j, the copies of sub-tile j + 1 are in flight.  The columns of a sub-tile
// sit one after another in its buffer (kSub elements each, raw row order);
// after the places are fixed, s_inv[i] holds the row of sorted place i, and
// each column is written by gathering through it.  Used when every column
// is 16-byte aligned and the buffers fit in shared memory.
struct TmaCols {
  const void* src[1 + PQ_MAX_PAYLOAD];
  void* dst[1 + PQ_MAX_PAYLOAD];
  int es[1 + PQ_MAX_PAYLOAD];   // element bytes
  int off[1 + PQ_MAX_PAYLOAD];  // byte offset of the column in a buffer
  int n;                        // columns, the key first
  int buf_bytes;                // bytes of one buffer
};

// SUB: rows of a sub-tile (2048, or 4096 where many buckets would leave
// runs of about two rows per bucket and sub-tile).
__host__ __device__ inline size_t tma_smem(int P, int buf_bytes, int sub) {
  return 16                          // two mbarriers
         + 2 * (size_t)buf_bytes     // double-buffered sub-tile
         + (size_t)P * 8             // s_gb
         + (size_t)8 * P * 2         // s_cnt (u16: at most sub / 8 per warp)
         + (size_t)P * 2 * 2         // s_run, s_tot (u16)
         + (size_t)sub * 2 * 2;      // s_inv, s_sbk
}

// One column of a sub-tile of SUB rows, written in sorted order: sorted
// place i = j * 256 + thread takes the buffered row src[j] to output row
// drow[j] (both worked out once for all columns).
template <typename V, int SUB>
__device__ __forceinline__ void gather_column(const char* buf, int off, V* __restrict__ dst,
                                              int cnt, const unsigned short* src,
                                              const i64* drow) {
  const V* col = reinterpret_cast<const V*>(buf + off);
  constexpr int kPer = SUB / 256;
#pragma unroll
  for (int j = 0; j < kPer; ++j)
    if (j * 256 + (int)threadIdx.x < cnt) __stcs(dst + drow[j], col[src[j]]);
}

// BLOCKS: the launch bound.  Three blocks per SM (71 to 80 registers) where the
// buffers leave room for three at most; rows of up to 9 bytes, of which more
// blocks fit, take no bound: the compiler then holds the kernel to 40
// registers.  60M rows of 8 bytes by 64: 443 us with room for three blocks, 450
// us bounded to five (48 registers), 422 us with none; of 21 bytes by 32 587 us
// with room for three and 629 us with none.
template <typename T, bool PART, int SUB, int BLOCKS>
__global__ void __launch_bounds__(256, BLOCKS) k_part_scatter_tma(i64 n, Digit<PART> dg,
                                                          const i64* __restrict__ gofs,
                                                          TmaCols tc, i64* d_offsets,
                                                          i64 spin_limit, DevStatus* st) {
  constexpr int kWRows = SUB / 8;  // rows of a warp in a sub-tile
  constexpr int kSteps = kWRows / 32;
  static_assert(kWRows <= 512, "place takes 9 bits");
  extern __shared__ __align__(16) unsigned char smem[];
  const int log2P = dg.bits, P = 1 << log2P;
  u64* bar = reinterpret_cast<u64*>(smem);
  char* bufs = reinterpret_cast<char*>(smem + 16);
  i64* s_gb = reinterpret_cast<i64*>(bufs + 2 * (size_t)tc.buf_bytes);
  unsigned short* s_cnt = reinterpret_cast<unsigned short*>(s_gb + P);
  unsigned short* s_run = s_cnt + 8 * P;
  unsigned short* s_tot = s_run + P;
  unsigned short* s_inv = s_tot + P;
  unsigned short* s_sbk = s_inv + SUB;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const i64 g = gridDim.x, k = blockIdx.x;
  const i64 r0 = chunk_begin(n, g, k), r1 = chunk_begin(n, g, k + 1);
  const i64 nsub = (r1 - r0 + SUB - 1) / SUB;
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    fence_mbar_init();
  }
  for (int b = threadIdx.x; b < P; b += blockDim.x) {
    s_gb[b] = gofs[(i64)b * g + k];
    if (k == 0 && d_offsets) d_offsets[b] = s_gb[b];
  }
  if (k == 0 && threadIdx.x == 0 && d_offsets) d_offsets[P] = n;
  __syncthreads();
  // Thread 0 starts the copies of sub-tile j into buffer j & 1: the part of
  // each column slice that is a whole number of 16-byte units (all of it but
  // possibly the last sub-tile's tail, which the block loads itself).
  auto issue = [&](i64 j) {
    if (threadIdx.x != 0 || j >= nsub) return;
    const i64 r = r0 + j * SUB;
    const i64 cnt = min((i64)SUB, r1 - r);
    char* buf = bufs + (j & 1) * (size_t)tc.buf_bytes;
    u32 total = 0;
    for (int c = 0; c < tc.n; ++c) total += (u32)((cnt * tc.es[c]) & ~15LL);
    mbar_expect_tx(&bar[j & 1], total);
    for (int c = 0; c < tc.n; ++c) {
      const u32 bytes = (u32)((cnt * tc.es[c]) & ~15LL);
      if (bytes)
        bulk_g2s(buf + tc.off[c], static_cast<const char*>(tc.src[c]) + r * tc.es[c], bytes,
                 &bar[j & 1]);
    }
  };
  issue(0);
  issue(1);
  for (i64 j = 0; j < nsub; ++j) {
    const i64 r = r0 + j * SUB;
    const int cnt = (int)min((i64)SUB, r1 - r);
    char* buf = bufs + (j & 1) * (size_t)tc.buf_bytes;
    const bool arrived = mbar_wait(&bar[j & 1], (u32)((j >> 1) & 1), spin_limit);
    if (__syncthreads_or(!arrived)) {  // block-uniform
      // The copies did not complete: report, give them a second bounded wait
      // (they write this block's shared memory) and stop.
      if (threadIdx.x == 0) latch(st, PQ_ERR_TIMEOUT, r);
      mbar_wait(&bar[j & 1], (u32)((j >> 1) & 1), spin_limit);
      if (j + 1 < nsub) mbar_wait(&bar[(j + 1) & 1], (u32)(((j + 1) >> 1) & 1), spin_limit);
      return;
    }
    // The tail that is not a whole 16-byte unit (last sub-tile only).
    for (int c = 0; cnt < SUB && c < tc.n; ++c) {
      const int es = tc.es[c];
      const int done = (int)(((i64)cnt * es) & ~15LL) / es;
      for (int i = done + (int)threadIdx.x; i < cnt; i += blockDim.x) {
        const char* src = static_cast<const char*>(tc.src[c]) + (r + i) * es;
        char* d = buf + tc.off[c] + (size_t)i * es;
        if (es == 8) *reinterpret_cast<i64*>(d) = *reinterpret_cast<const i64*>(src);
        else if (es == 4) *reinterpret_cast<int*>(d) = *reinterpret_cast<const int*>(src);
        else *d = *src;
      }
    }
    for (int b = threadIdx.x; b < 8 * P; b += blockDim.x) s_cnt[b] = 0;
    __syncthreads();
    const T* s_key = reinterpret_cast<const T*>(buf + tc.off[0]);
    const int nbits = cnt == SUB ? log2P : log2P + 1;  // every lane holds a row?
    u32 bp[kSteps];  // bucket << 9 | place among the warp's rows of that bucket
#pragma unroll
    for (int q = 0; q < kSteps; ++q) {
      const int i = warp * kWRows + q * 32 + lane;
      bp[q] = i < cnt ? dg((i64)s_key[i]) : 0xFFFFFFFFu;
    }
#pragma unroll
    for (int q = 0; q < kSteps; ++q) {
      const bool valid = bp[q] != 0xFFFFFFFFu;
      const u32 b = bp[q];
      const u32 peers = bucket_peers(valid ? b : (1u << log2P), nbits);
      u32 place = 0;
      if (valid) place = s_cnt[warp * P + b] + __popc(peers & lanemask_lt());
      __syncwarp();
      if (valid && lane == __ffs(peers) - 1)
        s_cnt[warp * P + b] = (unsigned short)(s_cnt[warp * P + b] + __popc(peers));
      __syncwarp();
      bp[q] = valid ? b << 9 | place : 0xFFFFFFFFu;
    }
    __syncthreads();
    for (int b = threadIdx.x; b < P; b += blockDim.x) {
      u32 run = 0;
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        const u32 c = s_cnt[w * P + b];
        s_cnt[w * P + b] = (unsigned short)run;
        run += c;
      }
      s_tot[b] = (unsigned short)run;
    }
    __syncthreads();
    {
      u32 v[4], sum = 0;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int b = (int)threadIdx.x * 4 + q;
        v[q] = b < P ? s_tot[b] : 0u;
        sum += v[q];
      }
      u32 run = block_exclusive_sum(sum);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int b = (int)threadIdx.x * 4 + q;
        if (b < P) s_run[b] = (unsigned short)run;
        run += v[q];
      }
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kSteps; ++q) {
      if (bp[q] == 0xFFFFFFFFu) continue;
      const u32 b = bp[q] >> 9;
      const int i = warp * kWRows + q * 32 + lane;
      const u32 at = s_run[b] + s_cnt[warp * P + b] + (bp[q] & 511u);
      s_inv[at] = (unsigned short)i;
      s_sbk[at] = (unsigned short)b;
    }
    __syncthreads();
    // This thread's sorted places: their rows in the buffer and output rows.
    constexpr int kPer = SUB / 256;
    unsigned short src[kPer];
    i64 drow[kPer];
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      const int i = q * 256 + (int)threadIdx.x;
      src[q] = 0, drow[q] = 0;
      if (i < cnt) {
        const u32 b = s_sbk[i];
        src[q] = s_inv[i];
        drow[q] = s_gb[b] + (i - (i64)s_run[b]);
      }
    }
    for (int c = 0; c < tc.n; ++c) {
      if (tc.es[c] == 8)
        gather_column<i64, SUB>(buf, tc.off[c], static_cast<i64*>(tc.dst[c]), cnt, src, drow);
      else if (tc.es[c] == 4)
        gather_column<int, SUB>(buf, tc.off[c], static_cast<int*>(tc.dst[c]), cnt, src, drow);
      else
        gather_column<signed char, SUB>(buf, tc.off[c], static_cast<signed char*>(tc.dst[c]), cnt,
                                   src, drow);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < P; b += blockDim.x) s_gb[b] += s_tot[b];
    // Every thread's reads of this buffer are done: the next copies into it
    // may start (ordered after the reads for the copy engine).
    fence_proxy_async_smem();
    __syncthreads();
    issue(j + 2);
  }
}

// ========================================================== hash join ====
// The join's hash table: 2^log2cap slots of 16 bytes, {key, value} side by
// side, so that an insert and a match each touch one sector.  Linear probing
// from the key's hash; or, where the build keys lie evenly in their range
// (ht_spread looks at a sample), a first slot that follows the key order, as
// many slots as the range has parts, and then the rest of its line of 8 (128
// bytes): keys built or probed in order then go through a line together,
// where hashed ones go to a sector of their own each.  Keys that are hashed
// gain nothing from lines: 3 % of lines are full, and a warp whose 64 probes
// wait for the longest path met one nearly every time (4M keys in no order:
// build 154 -> 192 us, 16M probes 198 -> 261 us).
struct HtMeta {
  i64 dup;        // a build key repeats
  i64 pad;
  u64 umin, range;  // the sample's smallest key (ukey) and its last key's distance
  u64 scale;        // slots per key distance, in 2^-64 (0: hashed)
};
// A path in key order: the first slot, the other slots of that line in turn,
// and, as long as lines are full, lines from the key's hash on, an odd number
// of lines near the golden section of the table apart (so each line is met
// once, and a few steps leave any part of the table).  Keys that crowd one
// part so spread over all of it: taken slot after slot from the hash on, a path
// that met a full part had to walk through it (2M keys, a quarter of them in a
// twelfth of the range: paths of up to 346211 slots, 422 on average; like this
// the longest has 21).
__device__ __forceinline__ u64 ht_first(const HtMeta& m, i64 k, u64 mask) {
  const u64 d = ((u64)k ^ 0x8000000000000000ULL) - m.umin;
  return d <= m.range ? __umul64hi(d, m.scale) : slot_hash(k) & mask;
}
// Slot i of the path that starts at slot s.
__device__ __forceinline__ u64 ht_line_slot(u64 s, u64 i) { return (s & ~7ULL) | ((s + i) & 7); }
__device__ __forceinline__ u64 ht_slot(u64 s, i64 k, u64 i, u64 mask) {
  if (i < 8) return ht_line_slot(s, i);
  const u64 step = __umul64hi(0x9E3779B97F4A7C15ULL, (mask + 1) >> 3) | 1;
  return (((slot_hash(k) >> 20) + ((i & ~7ULL) - 8) * step) & mask & ~7ULL) | ((s + i) & 7);
}

// 512 build keys spread over the input (the first and the last among them):
// their range, and whether each 512th of it holds about one of them.  Keys in
// no order fail that (random counts reach 4 and more) and gain nothing from
// it.  Then 512 neighbouring rows at a third and at two thirds of the input:
// no line gets more of them than it has slots (keys that come in dense groups
// with gaps between them are hashed).  One block.
constexpr int kHtSample = 512;
// Fewer keys: the table lies in L2 whatever the order.  At 1M keys in order
// build and 4M probes take 103 us hashed and 87 us in key order, at 2^18 42 us
// either way.
constexpr i64 kHtSpreadMin = 3 << 18;
template <typename TK>
__device__ __forceinline__ void ht_spread(const TK* __restrict__ key, i64 n, int log2cap,
                                          HtMeta* meta) {
  __shared__ u64 s_lo, s_hi;
  __shared__ u32 s_cnt[kHtSample];
  const i64 k = (i64)__ldg(key + (i64)((double)(n - 1) / (kHtSample - 1) * threadIdx.x));
  const u64 u = (u64)k ^ 0x8000000000000000ULL;
  if (threadIdx.x == 0) s_lo = ~0ULL, s_hi = 0;
  s_cnt[threadIdx.x] = 0;
  __syncthreads();
  atomicMin((unsigned long long*)&s_lo, (unsigned long long)u);
  atomicMax((unsigned long long*)&s_hi, (unsigned long long)u);
  __syncthreads();
  const u64 lo = s_lo, range = s_hi - lo;
  const u64 lines = 1ULL << (log2cap - 3);
  // Floor of 2^64 * parts / (range + 1): parts <= range + 1 keeps it in 64 bits.
  auto per_key = [&](u64 parts) {
    return (u64)(((unsigned __int128)parts << 64) / ((unsigned __int128)range + 1));
  };
  const bool fits = range >= 8 * lines;  // a slot for one distance or more
  if (fits) atomicAdd(&s_cnt[__umul64hi(u - lo, per_key(kHtSample))], 1u);
  int crowded = __syncthreads_or(fits && s_cnt[threadIdx.x] > 3);
  const u64 scale = per_key(8 * lines);
  for (int h = 1; h <= 2; ++h) {
    const i64 r0 = n / 3 * h;  // r0 + 511 < n: kHtSpreadMin rows at least
    auto line = [&](i64 r) {
      const u64 d = ((u64)(i64)__ldg(key + r) ^ 0x8000000000000000ULL) - lo;
      return __umul64hi(min(d, range), scale) >> 3;
    };
    s_cnt[threadIdx.x] = 0;
    __syncthreads();
    // Neighbours in key order fall on neighbouring lines: counted modulo 512.
    const u64 l = fits ? line(r0 + threadIdx.x) : 0;
    if (fits) atomicAdd(&s_cnt[l % kHtSample], 1u);
    __syncthreads();
    crowded |= __syncthreads_or(fits && s_cnt[threadIdx.x] > 8);
  }
  if (threadIdx.x == 0 && fits && !crowded)
    meta->umin = lo, meta->range = range, meta->scale = scale;
}

// Clears the table; with `look` block 0 looks at the keys meanwhile (7 us of
// waiting for a few loads, beside 10 us and more of writes).
template <typename TK>
__global__ void __launch_bounds__(kHtSample) k_ht_clear(longlong2* __restrict__ slots, int log2cap,
                                                        const TK* __restrict__ key, i64 n,
                                                        HtMeta* meta, int look) {
  if (look && blockIdx.x == 0) {
    ht_spread(key, n, log2cap, meta);
    return;
  }
  const i64 stride = (i64)(gridDim.x - look) * blockDim.x;
  for (i64 i = (i64)(blockIdx.x - look) * blockDim.x + threadIdx.x; i < 1LL << log2cap; i += stride)
    slots[i] = make_longlong2(kEmpty, 0);
}

// Hashed: one key per thread, as many threads as fit (two claims in flight per
// thread and half the warps: 4M keys 154 -> 240 us).  With `only` the kernel
// leaves a table in key order to k_ht_build_spread.
template <typename TK, typename TV>
__global__ void __launch_bounds__(256) k_ht_build(const TK* __restrict__ key,
                                                  const TV* __restrict__ val, i64 n,
                                                  i64* __restrict__ slots, int log2cap,
                                                  HtMeta* meta, int only, DevStatus* st) {
  if (only && meta->scale) return;
  const u64 mask = (1ULL << log2cap) - 1;
  const i64 stride = (i64)gridDim.x * blockDim.x;
  for (i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const i64 k = (i64)__ldg(key + i);
    if (k == kEmpty) {
      latch(st, PQ_ERR_RESERVED_KEY, i);
      continue;
    }
    const i64 v = val ? (i64)__ldg(val + i) : i;
    u64 s = slot_hash(k) & mask;
    u64 probes = 0;
    for (; probes <= mask; ++probes) {
      const i64 old = (i64)atomicCAS((u64*)&slots[2 * s], (u64)kEmpty, (u64)k);
      if (old == kEmpty) {
        slots[2 * s + 1] = v;
        break;
      }
      if (old == k) meta->dup = 1;
      s = (s + 1) & mask;
    }
    if (probes > mask) latch(st, PQ_ERR_CAPACITY, i);
  }
}

// In key order: two keys per thread whose claims are in flight together.  15M
// keys 4i + U{0..3} in order: 0.97 ms hashed, 0.35 ms with its clear like this
// (0.5 GB of lines read and written back); one key at a time 0.77 ms.
constexpr int kBldKeys = 2;
template <typename TK, typename TV>
__global__ void __launch_bounds__(256) k_ht_build_spread(const TK* __restrict__ key,
                                                         const TV* __restrict__ val, i64 n,
                                                         i64* __restrict__ slots, int log2cap,
                                                         HtMeta* meta, DevStatus* st) {
  const HtMeta m = *meta;
  if (!m.scale) return;
  const u64 mask = (1ULL << log2cap) - 1;
  const i64 stride = (i64)gridDim.x * blockDim.x;
  for (i64 i0 = (i64)blockIdx.x * blockDim.x + threadIdx.x; i0 < n; i0 += kBldKeys * stride) {
    i64 k[kBldKeys], v[kBldKeys], old[kBldKeys];
    u64 s[kBldKeys];
#pragma unroll
    for (int h = 0; h < kBldKeys; ++h) {
      const i64 i = i0 + h * stride;
      k[h] = i < n ? (i64)__ldg(key + i) : kEmpty;
      v[h] = i < n && val ? (i64)__ldg(val + i) : i;
      if (i < n && k[h] == kEmpty) latch(st, PQ_ERR_RESERVED_KEY, i);
    }
#pragma unroll
    for (int h = 0; h < kBldKeys; ++h) {
      s[h] = ht_first(m, k[h], mask);
      old[h] = kEmpty;
      if (k[h] != kEmpty) old[h] = (i64)atomicCAS((u64*)&slots[2 * s[h]], (u64)kEmpty, (u64)k[h]);
    }
#pragma unroll
    for (int h = 0; h < kBldKeys; ++h) {
      if (k[h] == kEmpty) continue;
      u64 probes = 0, at = s[h];
      while (old[h] != kEmpty) {
        if (old[h] == k[h]) meta->dup = 1;
        if (++probes > mask + 8) break;
        at = ht_slot(s[h], k[h], probes, mask);
        old[h] = (i64)atomicCAS((u64*)&slots[2 * at], (u64)kEmpty, (u64)k[h]);
      }
      if (old[h] == kEmpty) slots[2 * at + 1] = v[h];
      else latch(st, PQ_ERR_CAPACITY, i0 + h * stride);
    }
  }
}

// Hash-join probe: a warp probes 64 rows at a time, two per lane, whose
// chains of loads (key, then slot after slot of its path, every
// matching build row when the build keys repeat) run side by side.  The
// warp stages its matches in shared memory and writes them out kPrbBuf at a
// time, reserving each run with one atomic on the output counter: one
// reservation per pair-producing round would make that counter the bound
// (millions of atomics on one address).  Blocks of 8 warps, one resident
// wave, five of them per SM (48 registers).  60M rows in key order against
// 15M build keys: 1.00 ms hashed, 0.46 ms with lines in key order, whose first 8
// slots are a loop without the hash of the rest of the path (with it 0.55 ms;
// four rows per lane at 64 registers 0.48 ms).  The hashed loop is a function of
// its own: inlined with the other one it was 9 % slower, and as two kernels of
// which one returns at once a probe took 6 us more.
constexpr int kPrbBuf = 256, kPrbBlocks = 5;
struct PrbStage {
  i64 row[8][kPrbBuf], val[8][kPrbBuf];
};
template <typename TK, bool SPREAD>
__device__ __forceinline__ void ht_probe(const TK* __restrict__ pkey, i64 n,
                                         const longlong2* __restrict__ slots, int log2cap,
                                         const HtMeta* meta, i64* __restrict__ out_row,
                                         i64* __restrict__ out_val, i64 cap, u64* d_count,
                                         PrbStage& stage) {
  const u64 mask = (1ULL << log2cap) - 1;
  const HtMeta m = *meta;
  const bool dup = m.dup != 0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  i64* br = stage.row[warp];
  i64* bv = stage.val[warp];
  u32 nb = 0;  // staged pairs (warp-uniform)
  auto flush = [&]() {
    __syncwarp();
    u64 base = 0;
    if (lane == 0) base = atomicAdd(d_count, (u64)nb);
    base = __shfl_sync(kFull, base, 0);
    for (u32 e = lane; e < nb; e += 32) {
      const u64 pos = base + e;
      if (pos < (u64)cap) out_row[pos] = br[e], out_val[pos] = bv[e];
    }
    __syncwarp();
    nb = 0;
  };
  const i64 gw = ((i64)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const i64 nwarps = ((i64)gridDim.x * blockDim.x) >> 5;
  for (i64 wb = gw * 64; wb < n; wb += nwarps * 64) {
    i64 i[2], k[2];
    bool active[2];
    u64 s[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      i[h] = wb + h * 32 + lane;
      active[h] = i[h] < n;
      k[h] = active[h] ? (i64)__ldg(pkey + i[h]) : 0;
      if (k[h] == kEmpty) active[h] = false;
      s[h] = SPREAD ? ht_first(m, k[h], mask) : slot_hash(k[h]) & mask;
    }
    // The two rows' slots at(h); met(h): the slot was met before on the path.
    auto step = [&](auto at, auto met) {
      longlong2 kv[2];  // {key, value} of each row's current slot
#pragma unroll
      for (int h = 0; h < 2; ++h)
        kv[h] = active[h] ? __ldg(slots + at(h)) : make_longlong2(kEmpty, 0);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        bool emit = false;
        if (active[h]) {
          if (kv[h].x == kEmpty) {
            active[h] = false;
          } else if (kv[h].x == k[h] && !met(h)) {
            emit = true;
            if (!dup) active[h] = false;
          }
        }
        const u32 em = __ballot_sync(kFull, emit);
        if (emit) {
          const u32 to = nb + __popc(em & lanemask_lt());
          br[to] = i[h], bv[to] = kv[h].y;
        }
        nb += __popc(em);
      }
      if (nb > kPrbBuf - 64) flush();  // room for a full round stays
    };
    if constexpr (SPREAD) {
      for (u32 j = 0; j < 8 && __any_sync(kFull, active[0] || active[1]); ++j)
        step([&](int h) { return ht_line_slot(s[h], j); }, [](int) { return false; });
      // Past a full line (the path may come by it again).
      for (u64 j = 8; j <= mask + 8 && __any_sync(kFull, active[0] || active[1]); ++j)
        step([&](int h) { return ht_slot(s[h], k[h], j, mask); },
             [&](int h) { return !((ht_slot(s[h], k[h], j, mask) ^ s[h]) & ~7ULL); });
    } else {
      while (__any_sync(kFull, active[0] || active[1])) {  // a slot is always free
        step([&](int h) { return s[h]; }, [](int) { return false; });
#pragma unroll
        for (int h = 0; h < 2; ++h) s[h] = (s[h] + 1) & mask;
      }
    }
  }
  if (nb) flush();
}
template <typename TK>
__device__ __noinline__ void ht_probe_hashed(const TK* __restrict__ pkey, i64 n,
                                             const longlong2* __restrict__ slots, int log2cap,
                                             const HtMeta* meta, i64* __restrict__ out_row,
                                             i64* __restrict__ out_val, i64 cap, u64* d_count,
                                             PrbStage& stage) {
  ht_probe<TK, false>(pkey, n, slots, log2cap, meta, out_row, out_val, cap, d_count, stage);
}
template <typename TK>
__global__ void __launch_bounds__(256, kPrbBlocks)
    k_ht_probe(const TK* __restrict__ pkey, i64 n, const longlong2* __restrict__ slots, int log2cap,
               const HtMeta* meta, i64* __restrict__ out_row, i64* __restrict__ out_val, i64 cap,
               u64* d_count) {
  __shared__ PrbStage stage;
  if (meta->scale)
    ht_probe<TK, true>(pkey, n, slots, log2cap, meta, out_row, out_val, cap, d_count, stage);
  else
    ht_probe_hashed<TK>(pkey, n, slots, log2cap, meta, out_row, out_val, cap, d_count, stage);
}

__global__ void k_check_cap(const i64* d_count, i64 cap, DevStatus* st) {
  if (*d_count > cap) latch(st, PQ_ERR_CAPACITY, *d_count);
}

// ============================================================= group-by ====
__device__ __forceinline__ u64 gb_ukey(i64 k) { return (u64)k ^ 0x8000000000000000ULL; }

// Four consecutive rows from r0 on, widened (rows at or beyond n: `none`);
// VEC: the column starts on a 16-byte boundary.
template <typename T, bool VEC>
__device__ __forceinline__ void gb_load4(const T* __restrict__ p, i64 r0, i64 n, i64 none,
                                         i64 (&v)[4]) {
  T t[4];
  if (r0 + 4 <= n) {
    load4t<T, VEC, true>(p, r0, n, t);
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = (i64)t[j];
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = r0 + j < n ? (i64)ld_stream(p + r0 + j) : none;
  }
}

// Input in key order (or nearly: see GbSummary) is grouped by its runs of
// equal keys, with no table: one pass over the keys counts the runs of each
// warp's contiguous share of the rows (and measures the range), a scan gives
// every run its place, and a second pass writes one group per run.
struct GbSummary {
  u64 umin, umax;   // key range (ukey)
  i64 runs;         // runs of equal keys
  i64 first;        // runs before the first descent (all of them: no descent)
  i64 descents;     // rows whose key is below the row's before
  u32 over;         // the hash table did not hold the groups
  u32 top;          // rows of the most frequent key in a sample (0: fewer than kGbTopHot)
};
struct GbWarp {
  u32 runs, before, descents;  // of the warp's rows; before its first descent
  int joined;                  // its first row continues the run before it
};

// How often the most frequent key comes among 1024 rows spread over the input:
// from kGbTopHot of them on the tables keep frequent groups per block.
constexpr int kGbSample = 1024;
constexpr u32 kGbTopHot = 4;
template <typename TK>
__device__ __forceinline__ void gb_sample(const TK* __restrict__ key, i64 n, GbSummary* sum) {
  constexpr int kN = 2 * kGbSample;
  __shared__ i64 s_key[kN];
  __shared__ u32 s_cnt[kN], s_top;
  i64 k[kGbSample / 256];
#pragma unroll
  for (int j = 0; j < kGbSample / 256; ++j)
    k[j] = (i64)__ldg(key + n / kGbSample * (j * 256 + threadIdx.x));
  for (int i = threadIdx.x; i < kN; i += 256) s_key[i] = kEmpty, s_cnt[i] = 0;
  if (threadIdx.x == 0) s_top = 0;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kGbSample / 256; ++j) {
    if (k[j] == kEmpty) continue;
    u32 at = (u32)slot_hash(k[j]) & (kN - 1);
    for (;; at = (at + 1) & (kN - 1)) {  // half of the slots stay free
      const i64 was = (i64)atomicCAS((unsigned long long*)&s_key[at], (unsigned long long)kEmpty,
                                     (unsigned long long)k[j]);
      if (was == kEmpty || was == k[j]) break;
    }
    const u32 c = atomicAdd(&s_cnt[at], 1u) + 1;
    if (c >= kGbTopHot) atomicMax(&s_top, c);
  }
  __syncthreads();
  if (threadIdx.x == 0) sum->top = s_top;
}

// The first block samples the keys meanwhile.  Four blocks per SM, of this pass
// and of the one over the runs, whose shares of the rows are the same: 61
// registers and one wave.  (Six, which the scan alone would fit, held it to 40
// registers with 72 bytes of spills and made the runs one wave and a half: 40M
// ordered rows of 400 groups 198 -> 186 us a call, 8M 78 -> 68.)
constexpr int kGbScanBlocks = 4;
template <typename TK, bool VEC>
__global__ void __launch_bounds__(256, kGbScanBlocks) k_gb_scan(const TK* __restrict__ key, i64 n,
                                                    GbWarp* __restrict__ wout, GbSummary* sum) {
  if (blockIdx.x == 0) {
    gb_sample(key, n, sum);
    return;
  }
  __shared__ u64 s_lo[8], s_hi[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const i64 steps = (n + 127) / 128, nw = (i64)(gridDim.x - 1) * 8;
  const i64 gw = (i64)(blockIdx.x - 1) * 8 + warp;
  const i64 t0 = filter_share(steps, nw, gw), t1 = filter_share(steps, nw, gw + 1);
  u32 starts = 0, desc = 0, before = 0;
  bool any_desc = false, joined = false;
  const i64 end = (i64)__ldg(key + n - 1);  // rows past the end repeat the last key
  i64 last = t0 < t1 && t0 > 0 ? (i64)__ldg(key + t0 * 128 - 1) : 0;  // before the step
  // Between descents keys only grow: the range is that of the share's first
  // and last keys and of the keys at its descents.
  i64 lo = t0 < t1 ? (i64)__ldg(key + t0 * 128) : INT64_MAX;
  i64 hi = t0 < t1 ? (i64)__ldg(key + min(n, t1 * 128) - 1) : INT64_MIN;
  i64 kn[4] = {0, 0, 0, 0};  // the next step's keys
  if (t0 < t1) gb_load4<TK, VEC>(key, t0 * 128 + 4 * lane, n, end, kn);
  for (i64 t = t0; t < t1; ++t) {
    const i64 k[4] = {kn[0], kn[1], kn[2], kn[3]};
    if (t + 1 < t1) gb_load4<TK, VEC>(key, (t + 1) * 128 + 4 * lane, n, end, kn);
    i64 prev = __shfl_up_sync(kFull, k[3], 1);
    if (lane == 0) prev = last;
    last = __shfl_sync(kFull, k[3], 31);
    u32 hd = (u32)(k[0] != prev), ds = (u32)(k[0] < prev);
#pragma unroll
    for (int j = 1; j < 4; ++j) {
      hd |= (u32)(k[j] != k[j - 1]) << j;
      ds |= (u32)(k[j] < k[j - 1]) << j;
    }
    if (t == 0 && lane == 0) hd |= 1u, ds &= ~1u;  // row 0
    if (t == t0) joined = __shfl_sync(kFull, hd & 1u, 0) == 0;
    if (__any_sync(kFull, ds)) {
      if (!any_desc) {  // the first descent: runs before it
        any_desc = true;
        const int fl = __ffs(__ballot_sync(kFull, ds)) - 1;
        const int fj = __shfl_sync(kFull, __ffs(ds) - 1, fl);
        const u32 mine = lane < fl ? __popc(hd) : lane == fl ? __popc(hd & ((1u << fj) - 1u)) : 0u;
        before = __reduce_add_sync(kFull, starts + mine);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if ((ds >> j) & 1u) lo = min(lo, k[j]), hi = max(hi, j ? k[j - 1] : prev);
      desc += __popc(ds);
    }
    starts += __popc(hd);
  }
  starts = __reduce_add_sync(kFull, starts), desc = __reduce_add_sync(kFull, desc);
  u64 ulo = gb_ukey(lo), uhi = gb_ukey(hi);
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    ulo = min(ulo, (u64)__shfl_xor_sync(kFull, ulo, o));
    uhi = max(uhi, (u64)__shfl_xor_sync(kFull, uhi, o));
  }
  if (lane == 0) {
    GbWarp w;
    w.runs = starts, w.before = before, w.descents = desc, w.joined = joined;
    wout[gw] = w;
    s_lo[warp] = ulo, s_hi[warp] = uhi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int w = 1; w < 8; ++w) ulo = min(ulo, s_lo[w]), uhi = max(uhi, s_hi[w]);
    atomicMin((unsigned long long*)&sum->umin, (unsigned long long)ulo);
    atomicMax((unsigned long long*)&sum->umax, (unsigned long long)uhi);
  }
}

// One block: each warp's first run number, and the summary.
__global__ void __launch_bounds__(1024) k_gb_bounds(const GbWarp* __restrict__ w, int nw,
                                                    i64* __restrict__ base, GbSummary* sum) {
  __shared__ i64 s_carry;
  __shared__ int s_first;
  if (threadIdx.x == 0) s_carry = 0, s_first = nw;
  __syncthreads();
  u32 desc = 0;
  GbWarp next = (int)threadIdx.x < nw ? w[threadIdx.x] : GbWarp{};
  for (int b = 0; b < nw; b += 1024) {
    const int i = b + threadIdx.x;
    const GbWarp x = next;
    next = i + 1024 < nw ? w[i + 1024] : GbWarp{};
    const u32 ex = block_exclusive_sum(x.runs);  // 1024 warps' runs: below 2^32
    const i64 carry = s_carry;
    if (i < nw) base[i] = carry + ex;
    if (x.descents) atomicMin(&s_first, i);
    desc += x.descents;
    __syncthreads();
    if (threadIdx.x == 1023) s_carry = carry + ex + x.runs;
    __syncthreads();
  }
  if (desc) atomicAdd((unsigned long long*)&sum->descents, (unsigned long long)desc);
  if (threadIdx.x == 0) {
    base[nw] = s_carry;
    sum->runs = s_carry;
    sum->first = s_first < nw ? base[s_first] + w[s_first].before : s_carry;
  }
}

// Where run p goes: the output, or (a run of the rows after the descent) the
// scratch list that is folded in afterwards.
struct GbOut {
  i64* keys;
  i64* sums;
  i64 cap, first;
  i64* tail_keys;
  i64* tail_sums;
};
__device__ __forceinline__ i64* gb_at(const GbOut& o, i64 p, bool key) {
  if (p < o.first) return p < o.cap ? (key ? o.keys : o.sums) + p : nullptr;
  return (key ? o.tail_keys : o.tail_sums) + (p - o.first);
}

// Runs that cross from one warp's share into the next are added up in place:
// their sums start at 0.
__global__ void k_gb_joins(const GbWarp* __restrict__ w, const i64* __restrict__ base, int nw,
                           GbOut o, i64* d_ngroups) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) *d_ngroups = o.first;
  if (i < nw && w[i].joined)
    if (i64* p = gb_at(o, base[i] - 1, false)) *p = 0;
}

// One group per run.  A warp walks its share 128 rows a step (lane l: rows
// 4l .. 4l+3): the s-th row of the step that starts a run closes the run
// before it, whose sum (a segmented scan over the lanes, and what the steps
// before left) goes to place s of the warp's stage; the stage is written as
// one contiguous piece.  Bound by reading the rows and writing the groups:
// 60M rows, 15M groups (1.2 GB) in 0.192 ms, 6.2 TB/s, after 0.085 ms of
// k_gb_scan; the range pass, slot array and its emit took 0.63 ms (and three
// clears), which unordered rows still take.
template <typename TK, typename TV, bool VEC>
__global__ void __launch_bounds__(256, kGbScanBlocks) k_gb_runs(const TK* __restrict__ key,
                                                    const TV* __restrict__ val, i64 n,
                                                    const GbWarp* __restrict__ winfo,
                                                    const i64* __restrict__ base, GbOut o) {
  __shared__ i64 s_k[8][128], s_s[8][128];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const i64 steps = (n + 127) / 128, nw = (i64)gridDim.x * 8, gw = (i64)blockIdx.x * 8 + warp;
  const i64 t0 = filter_share(steps, nw, gw), t1 = filter_share(steps, nw, gw + 1);
  if (t0 >= t1) return;
  i64* const sk = s_k[warp];
  i64* const ss = s_s[warp];
  const bool joined = winfo[gw].joined != 0;
  const i64 b0 = base[gw];
  i64 run = b0 - 1;  // the run that is open
  i64 carry = 0, last = t0 > 0 ? (i64)__ldg(key + t0 * 128 - 1) : 0;
  const i64 end = (i64)__ldg(key + n - 1);  // rows past the end: its key, value 0
  i64 kn[4], vn[4];                         // the next step's rows
  gb_load4<TK, VEC>(key, t0 * 128 + 4 * lane, n, end, kn);
  gb_load4<TV, VEC>(val, t0 * 128 + 4 * lane, n, 0, vn);
  for (i64 t = t0; t < t1; ++t) {
    const i64 r0 = t * 128 + 4 * lane;
    const i64 k[4] = {kn[0], kn[1], kn[2], kn[3]}, v[4] = {vn[0], vn[1], vn[2], vn[3]};
    if (t + 1 < t1) {
      gb_load4<TK, VEC>(key, r0 + 128, n, end, kn);
      gb_load4<TV, VEC>(val, r0 + 128, n, 0, vn);
    }
    i64 prev = __shfl_up_sync(kFull, k[3], 1);
    if (lane == 0) prev = last;
    last = __shfl_sync(kFull, k[3], 31);
    u32 hd = (u32)(k[0] != prev || r0 == 0);
#pragma unroll
    for (int j = 1; j < 4; ++j) hd |= (u32)(k[j] != k[j - 1]) << j;
    // Starts before this lane's, and in the step.
    u32 rank = 0, c = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const u32 m = __ballot_sync(kFull, (hd >> j) & 1u);
      rank += __popc(m & lanemask_lt()), c += __popc(m);
    }
    // The sum since the last start, up to and with each lane.
    i64 ls = 0;
    u32 fl = hd != 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) ls = ((hd >> j) & 1u) ? v[j] : ls + v[j];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      if (__all_sync(kFull, fl)) break;
      const i64 us = __shfl_up_sync(kFull, ls, d);
      const u32 uf = __shfl_up_sync(kFull, fl, d);
      if (lane >= d && !fl) ls += us, fl = uf;
    }
    if (!fl) ls += carry;  // no start up to here: the open run goes on
    i64 acc = __shfl_up_sync(kFull, ls, 1);
    if (lane == 0) acc = carry;
    carry = __shfl_sync(kFull, ls, 31);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if ((hd >> j) & 1u) sk[rank] = k[j], ss[rank] = acc, ++rank, acc = 0;
      acc += v[j];
    }
    __syncwarp();
    for (u32 s = lane; s < c; s += 32) {
      if (i64* q = gb_at(o, run + 1 + s, true)) *q = sk[s];
      const i64 p = run + s;
      if (p >= b0) {
        if (i64* q = gb_at(o, p, false)) *q = ss[s];
      } else if (joined) {  // the run the warp before started
        if (i64* q = gb_at(o, p, false)) atomicAdd((unsigned long long*)q, (unsigned long long)ss[s]);
      }
    }
    __syncwarp();
    run += c;
  }
  if (lane == 0 && (run >= b0 || joined)) {
    // The run open at the share's end: more of it may follow in the next share.
    const bool shared = run < b0 || (gw + 1 < nw && t1 < steps && winfo[gw + 1].joined);
    if (i64* q = gb_at(o, run, false)) {
      if (shared) atomicAdd((unsigned long long*)q, (unsigned long long)carry);
      else *q = carry;
    }
  }
}

// The runs after the one descent (few: at most an eighth of the rows): each
// is looked up among the groups before it, which are in key order, and is
// added there or becomes a group of its own.
__global__ void __launch_bounds__(256) k_gb_fold(GbOut o, i64 m, i64* d_ngroups) {
  const i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const i64 k = o.tail_keys[i], v = o.tail_sums[i];
  i64 lo = 0, hi = o.first;
  while (lo < hi) {
    const i64 mid = (lo + hi) >> 1;
    if (o.keys[mid] < k) lo = mid + 1;
    else hi = mid;
  }
  if (lo < o.first && o.keys[lo] == k) {
    atomicAdd((unsigned long long*)(o.sums + lo), (unsigned long long)v);
  } else {
    const i64 q = (i64)atomicAdd((unsigned long long*)d_ngroups, 1ULL);
    if (q < o.cap) o.keys[q] = k, o.sums[q] = v;
  }
}

// Other inputs: each lane takes 4 consecutive rows of a 128-row warp step;
// runs of equal keys are summed by a segmented scan over the lanes and each
// run calls on(key, sum) once.  The reserved key is reported and left out.
template <typename TK, typename TV, bool VEC, typename On>
__device__ __forceinline__ void gb_each_run(const TK* __restrict__ key, const TV* __restrict__ val,
                                            i64 n, DevStatus* st, On on) {
  const int lane = threadIdx.x & 31;
  const i64 gw = ((i64)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const i64 nw = ((i64)gridDim.x * blockDim.x) >> 5;
  for (i64 wb = gw * 128; wb < n; wb += nw * 128) {
    const i64 r0 = wb + 4 * lane;
    i64 k[4], v[4];
    gb_load4<TK, VEC>(key, r0, n, kEmpty, k);
    gb_load4<TV, VEC>(val, r0, n, 0, v);
    u32 ok = 0;  // bit j: row j exists and its key is not the reserved one
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (r0 + j < n && k[j] == kEmpty) latch(st, PQ_ERR_RESERVED_KEY, r0 + j);
      ok |= (u32)(k[j] != kEmpty) << j;
    }
    // Runs: a row starts one when its key differs from the row before it;
    // lane 0's first row always does.
    const i64 prev = __shfl_up_sync(kFull, k[3], 1);
    u32 head = lane == 0 ? 1u : (u32)(k[0] != prev);
#pragma unroll
    for (int j = 1; j < 4; ++j) head |= (u32)(k[j] != k[j - 1]) << j;
    // The lane's last run, summed back to the lane where it starts.
    i64 ls = 0;
    u32 fl = head != 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) ls = ((head >> j) & 1u) ? v[j] : ls + v[j];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      if (__all_sync(kFull, fl)) break;
      const i64 us = __shfl_up_sync(kFull, ls, d);
      const u32 uf = __shfl_up_sync(kFull, fl, d);
      if (lane >= d && !fl) ls += us, fl = uf;
    }
    const i64 in_s = __shfl_up_sync(kFull, ls, 1);
    const bool next_head = __shfl_down_sync(kFull, head & 1u, 1);
    i64 acc = (head & 1u) ? 0 : in_s;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (j > 0 && ((head >> j) & 1u)) acc = 0;
      acc += v[j];
      const bool end = j < 3 ? (head >> (j + 1)) & 1u : (lane == 31 || next_head);
      if (end && ((ok >> j) & 1u)) on(k[j], acc);
    }
  }
}

// Slots of the hash table: keys and sums in arrays of their own (STRIDE 1) while
// they fit in L2, so that the sectors of the keys are only read once they are
// filled; {key, sum} side by side (STRIDE 2), one sector per row, in tables
// beyond it (kGbPairBytes).  40M rows: of 400000 groups 0.62 and 1.2 ms, of 10M
// groups 2.7 and 2.1 ms, of 40M 4.5 and 3.6 ms.
constexpr size_t kGbPairBytes = 128 << 20;
struct GbTable {
  i64 *keys, *sums;
  int log2cap;
};

// Rows of no frequent key, or few rows: a lane takes a row (rows in flight are
// what counts: four rows per lane one after another took 40M rows of 400000
// groups 616 -> 860 us), equal keys of a warp are added first, and a key that
// a warp meets twice goes to the block's small table of frequent groups, which
// the others only look at.  With `over`, a table that fills up is given up instead of
// reported: a key that finds no slot within kGbMaxProbes sets the flag, and the
// others stop looking a line (8 slots) further on, so that the whole pass costs
// no more than a few lines a row.
constexpr u64 kGbMaxProbes = 1024;
// A key's slot, inserted if need be; ~0: none (`over` is set or was).
template <int STRIDE>
__device__ __forceinline__ u64 gb_slot(const GbTable& t, i64 k, u64 mask, u64 limit, u32* over,
                                       DevStatus* st) {
  u64 s = slot_hash(k) & mask;
  for (u64 probes = 0; probes <= limit; ++probes) {
    i64 cur = t.keys[STRIDE * s];  // a stale free slot is seen by the CAS
    if (cur == kEmpty)
      cur = (i64)atomicCAS((u64*)&t.keys[STRIDE * s], (u64)kEmpty, (u64)k);
    if (cur == kEmpty || cur == k) return s;
    if (over && (probes & 7) == 7 && *(volatile u32*)over) return ~0ULL;
    s = (s + 1) & mask;
  }
  if (over) *(volatile u32*)over = 1;
  else latch(st, PQ_ERR_CAPACITY, -1);
  return ~0ULL;
}
// Adds the block's frequent groups to the table.
template <int STRIDE, int HOT>
__device__ __forceinline__ void gb_flush(const HotSums<HOT>& hot, const GbTable& t) {
  __syncthreads();
  for (int i = threadIdx.x; i < hot.kN; i += blockDim.x)
    if (hot.key[i] != kHotFree)
      atomicAdd((u64*)&t.sums[STRIDE * (u64)hot.key[i]], (u64)hot.hi[i] << 32 | hot.lo[i]);
}
template <typename TK, typename TV, int STRIDE>
__global__ void __launch_bounds__(256) k_gb_rows(const TK* __restrict__ key,
                                                 const TV* __restrict__ val, i64 n, GbTable t,
                                                 DevStatus* st, u32* over) {
  __shared__ HotSums<8> hot;
  hot.clear();
  __syncthreads();
  const u64 mask = (1ULL << t.log2cap) - 1;
  const u64 limit = over ? min(mask, kGbMaxProbes - 1) : mask;
  const bool use_hot = t.log2cap < 32;
  const int lane = threadIdx.x & 31;
  const i64 gw = ((i64)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const i64 nwarps = ((i64)gridDim.x * blockDim.x) >> 5;
  bool gone = false;  // the table is given up
  for (i64 wb = gw * 32; wb < n; wb += nwarps * 32) {
    if (over && __any_sync(kFull, gone)) break;
    const i64 i = wb + lane;
    bool active = i < n;
    const i64 k = active ? (i64)__ldg(key + i) : kEmpty;
    i64 v = active ? (i64)__ldg(val + i) : 0;
    if (active && k == kEmpty) {
      latch(st, PQ_ERR_RESERVED_KEY, i);
      active = false;
    }
    const u32 peers = __match_any_sync(kFull, (u64)k);
    if (__any_sync(kFull, active && __popc(peers) > 1)) {
      i64 agg = 0;
      for (int src = 0; src < 32; ++src) {
        const i64 x = __shfl_sync(kFull, v, src);
        if ((peers >> src) & 1u) agg += x;
      }
      v = agg;
    }
    if (!active || lane != __ffs(peers) - 1) continue;
    const u64 s = gb_slot<STRIDE>(t, k, mask, limit, over, st);
    if (s == ~0ULL) {
      gone = true;
      continue;
    }
    if (!(use_hot && hot.add_if((u32)s, v, __popc(peers) > 1)))
      atomicAdd((u64*)&t.sums[STRIDE * s], (u64)v);
  }
  gb_flush<STRIDE>(hot, t);
}

// Many rows with frequent keys: runs as in the slot array below, and a large
// table of frequent groups per block (a reduction on one address takes 1.8 ns:
// a key that holds a sixteenth of 30M rows took the hash table to 2.7 ms and
// the slot array to 3.3 ms).
constexpr int kGbHotLog2 = 11;
template <typename TK, typename TV, bool VEC, int STRIDE>
__global__ void __launch_bounds__(256) k_gb_insert(const TK* __restrict__ key,
                                                   const TV* __restrict__ val, i64 n, GbTable t,
                                                   DevStatus* st, u32* over) {
  __shared__ HotSums<kGbHotLog2> hot;
  hot.clear();
  __syncthreads();
  const u64 mask = (1ULL << t.log2cap) - 1;
  const u64 limit = over ? min(mask, kGbMaxProbes - 1) : mask;
  const bool use_hot = t.log2cap < 32;
  gb_each_run<TK, TV, VEC>(key, val, n, st, [&](i64 k, i64 acc) {
    const u64 s = gb_slot<STRIDE>(t, k, mask, limit, over, st);
    if (s == ~0ULL || (use_hot && hot.add((u32)s, acc, hot.owner((u32)s)))) return;
    atomicAdd((u64*)&t.sums[STRIDE * s], (u64)acc);
  });
  gb_flush<STRIDE>(hot, t);
}

// kEmpty in every key, 0 in every sum (sums = keys + 1, or keys + the slots).
__global__ void k_gb_clear(longlong2* __restrict__ p, i64 n, int pairs) {
  const i64 stride = (i64)gridDim.x * blockDim.x;
  for (i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    p[i] = pairs || 2 * i < n ? make_longlong2(kEmpty, pairs ? 0 : kEmpty) : make_longlong2(0, 0);
}


// The slot array's kernels take `if_over`: with it they run only if the flag
// is set (the hash table before them did not hold the groups).
__global__ void k_gb_zero_if(longlong2* __restrict__ p, i64 n, const u32* if_over) {
  if (!*if_over) return;
  const i64 stride = (i64)gridDim.x * blockDim.x;
  for (i64 i = (i64)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    p[i] = make_longlong2(0, 0);
}

// Dense keys (a key range of at most 4 rows per key): the group of key k is
// slot k - min, its sum in a zeroed array and its existence in a bitmap, so
// a run costs one reduction and one bit, at addresses that follow the key
// order.  HOT: with the table of frequent groups, where the sample met a
// frequent key (without one it costs up to a tenth).  A small bitmap's words
// are looked at before a bit is set: 1000 groups keep theirs in 32 words, on
// which 8M rows waited for each other 1.6 ms.
constexpr u64 kGbAskSpan = 1 << 16;
template <typename TK, typename TV, bool VEC, bool HOT>
__global__ void __launch_bounds__(256) k_gb_dense(const TK* __restrict__ key,
                                                  const TV* __restrict__ val, i64 n, u64 umin,
                                                  u64 span, i64* __restrict__ sums,
                                                  u32* __restrict__ bm, DevStatus* st,
                                                  const u32* if_over) {
  if (if_over && !*if_over) return;
  const bool ask = span <= kGbAskSpan;
  auto add = [&](u64 idx, i64 acc) {
    atomicAdd(reinterpret_cast<unsigned long long*>(sums + idx), (unsigned long long)acc);
    const u32 bit = 1u << (idx & 31);
    if (!ask || !(__ldcg(bm + (idx >> 5)) & bit)) atomicOr(bm + (idx >> 5), bit);
  };
  if constexpr (HOT) {
    __shared__ HotSums<kGbHotLog2> hot;
    hot.clear();
    __syncthreads();
    const bool use_hot = span < kHotFree;
    gb_each_run<TK, TV, VEC>(key, val, n, st, [&](i64 k, i64 acc) {
      const u64 idx = gb_ukey(k) - umin;
      if (use_hot && hot.add((u32)idx, acc, hot.owner((u32)idx))) return;
      add(idx, acc);
    });
    __syncthreads();
    for (int i = threadIdx.x; i < hot.kN; i += blockDim.x)
      if (hot.key[i] != kHotFree)
        add(hot.key[i], (i64)((u64)hot.hi[i] << 32 | hot.lo[i]));
  } else {
    gb_each_run<TK, TV, VEC>(key, val, n, st,
                             [&](i64 k, i64 acc) { add(gb_ukey(k) - umin, acc); });
  }
}

// Positions for a block's outputs, cnt per thread: one atomic on the
// output counter per block step (a block-wide scan of the counts), so that
// the counter is not a point of contention.  Every thread of the block
// calls it; returns this thread's first position.
__device__ __forceinline__ u64 block_reserve(u64* counter, u32 cnt) {
  __shared__ u64 s_base;
  const u32 before = block_exclusive_sum(cnt);
  if (threadIdx.x == blockDim.x - 1) s_base = atomicAdd(counter, (u64)(before + cnt));
  __syncthreads();
  const u64 pos = s_base + before;
  __syncthreads();  // s_base is read before the next call writes it
  return pos;
}

// The groups of the dense slot array, from its existence bitmap, in key
// order within each block step: a thread reserves the positions of one
// bitmap word's groups (one atomic per block step), then the warp writes
// its 32 words one after another, lane l taking bit l, so that the sums are
// read and the groups written in contiguous runs.
__global__ void __launch_bounds__(256) k_gb_dense_emit(const u32* __restrict__ bm,
                                                       const i64* __restrict__ sums, u64 span,
                                                       u64 umin, i64* __restrict__ out_keys,
                                                       i64* __restrict__ out_sums, i64 cap,
                                                       u64* d_ngroups, const u32* if_over) {
  if (if_over && !*if_over) return;
  const i64 words = (i64)((span + 31) / 32);
  const i64 stride = (i64)gridDim.x * blockDim.x;
  for (i64 w0 = (i64)blockIdx.x * blockDim.x; w0 < words; w0 += stride) {  // block-uniform
    const i64 w = w0 + threadIdx.x;
    const u32 bits = w < words ? __ldg(bm + w) : 0u;
    const u64 pos = block_reserve(d_ngroups, (u32)__popc(bits));
    const int lane = threadIdx.x & 31;
    const i64 wfirst = w - lane;
    for (int c = 0; c < 32; ++c) {
      const u32 wc = __shfl_sync(kFull, bits, c);
      const u64 pc = __shfl_sync(kFull, pos, c);
      if (!((wc >> lane) & 1u)) continue;
      const u64 p = pc + __popc(wc & lanemask_lt());
      const u64 idx = (u64)(wfirst + c) * 32 + (u64)lane;
      if (p < (u64)cap) {
        out_keys[p] = (i64)((umin + idx) ^ 0x8000000000000000ULL);
        out_sums[p] = __ldg(sums + idx);
      }
    }
  }
}

// The groups of the hash table: a thread takes kGbEmitPer consecutive slots
// and writes their groups at consecutive positions reserved per block step.
constexpr int kGbEmitPer = 8;
template <int STRIDE>
__global__ void __launch_bounds__(256) k_gb_emit(GbTable t, i64* __restrict__ out_keys,
                                                 i64* __restrict__ out_sums, i64 cap,
                                                 u64* d_ngroups, const u32* over) {
  if (over && *over) return;
  const i64 slots = 1LL << t.log2cap, step = (i64)gridDim.x * blockDim.x * kGbEmitPer;
  for (i64 b0 = (i64)blockIdx.x * blockDim.x * kGbEmitPer; b0 < slots; b0 += step) {  // block-uniform
    const i64 b = b0 + (i64)threadIdx.x * kGbEmitPer;
    longlong2 e[kGbEmitPer];  // the slots are a power of two, 64 at least
    u32 m = 0;
#pragma unroll
    for (int j = 0; j < kGbEmitPer; ++j) {
      const i64 at = min(b + j, slots - 1);
      if (STRIDE == 2) e[j] = __ldcs(reinterpret_cast<const longlong2*>(t.keys) + at);
      else e[j].x = __ldcs(t.keys + at);
    }
#pragma unroll
    for (int j = 0; j < kGbEmitPer; ++j) m |= (u32)(b + j < slots && e[j].x != kEmpty) << j;
    if (STRIDE == 1)
#pragma unroll
      for (int j = 0; j < kGbEmitPer; ++j)
        if ((m >> j) & 1u) e[j].y = __ldcs(t.sums + b + j);
    u64 pos = block_reserve(d_ngroups, (u32)__popc(m));
#pragma unroll
    for (int j = 0; j < kGbEmitPer; ++j)
      if ((m >> j) & 1u) {
        if (pos < (u64)cap) out_keys[pos] = e[j].x, out_sums[pos] = e[j].y;
        ++pos;
      }
  }
}

// ================================================================ top-k ====
// Least pairs of a block beyond 2048 in all.  3.1M of 12.5M groups over a sum,
// found by an aggregate-first plan of 50M rows: the plan takes 353 us with 1024,
// 359 us with 256 or 2048; 250k groups, k = 64: 214, 220 and 205 us.
constexpr int kTopkPer = 1024;
__global__ void __launch_bounds__(256, 2) k_topk(const i64* __restrict__ keys,
                                              const i64* __restrict__ sums, i64 n_cap,
                                              const i64* d_n, int K, i64* part_k, i64* part_s,
                                              int* part_c, u32* ticket, i64* out_keys,
                                              i64* out_sums, i64* d_nout, const u64* rec_ctr,
                                              pq_result* rec) {
  __shared__ i64 sk[8 * kMaxK], ss[8 * kMaxK];
  __shared__ int sc[8];
  __shared__ bool s_last;
  __shared__ i64 s_scr[8][kTopScr];
  __shared__ LaneRankSmem<256> s_lr;
  chain_begin();
  const i64 n = d_n ? min(*d_n, n_cap) : n_cap;
  // Only the first nb blocks take pairs, so that a small count read on the
  // device leaves few lists to merge, or none: one block up to 2048 pairs, else
  // at least kTopkPer each.
  const int nb = n <= 2048 ? 1 : (int)min((i64)gridDim.x, (n + kTopkPer - 1) / kTopkPer);
  if ((int)blockIdx.x >= nb) return;  // no pairs: the nb blocks take the ticket
  const i64 per = (n + nb - 1) / nb;
  const i64 lo = min(n, per * blockIdx.x), hi = min(n, lo + per);
  const int lane = threadIdx.x & 31;
  // A single block writes the result itself; otherwise its list.
  i64* bk = nb == 1 ? out_keys : part_k + (i64)blockIdx.x * K;
  i64* bs = nb == 1 ? out_sums : part_s + (i64)blockIdx.x * K;
  // K <= 32: each thread keeps its best kLL pairs in registers and the
  // block ranks the few that can be in its top K (tk_lane_rank); when that
  // cannot vouch for its result, and for K > 32, the warps' register lists
  // are merged in shared memory (TopList).
  int cnt = -1;
  if (K <= 32) {
    // A first threshold: the K-th best of the threads' best pairs, each of 16
    // spread over the thread's share (a sorted input then gives a threshold
    // near its end).  At least K pairs are not after it, so a pair after it
    // cannot be among the block's K best: only the others enter the lists,
    // which keeps the lanes of a warp on the same path.  Blocks with fewer than
    // 16 pairs per thread skip it (block-uniform).
    bool filt = false;
    i64 thk = 0, ths = 0;
    if (hi - lo >= 16 * 256) {
      const i64 mine = (hi - lo - threadIdx.x + 255) / 256;  // 16 at least
      const i64 at = lo + threadIdx.x;
      i64 x[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) x[q] = __ldcs(sums + at + mine * q / 16 * 256);
      i64 hs = x[0], hk = INT64_MAX;
#pragma unroll
      for (int q = 1; q < 16; ++q) hs = max(hs, x[q]);
#pragma unroll
      for (int q = 0; q < 16; ++q)
        if (x[q] == hs) hk = min(hk, __ldcs(keys + at + mine * q / 16 * 256));
      s_lr.hk[threadIdx.x] = hk, s_lr.hs[threadIdx.x] = hs;
      __syncthreads();
      if (rank_among(s_lr.hk, s_lr.hs, 256, hk, hs, (int)threadIdx.x) == K - 1)
        s_lr.thk = hk, s_lr.ths = hs;
      __syncthreads();
      filt = true;
      thk = s_lr.thk, ths = s_lr.ths;
      __syncthreads();  // tk_lane_rank reuses s_lr
    }
    LaneTop T;
    T.clear();
    i64 i = lo + threadIdx.x;
    if (filt) {
      // Most pairs fall short by their sum alone: only the sums are read, 16
      // in flight, and the keys of those that pass or tie (so half the bytes).
      // Without the keys of ties all of 15M equal sums entered the lists: 168 us
      // instead of 66 (with them 15M sums that differ take 51 us, 47 without).
      for (; i + 15 * 256 < hi; i += 16 * 256) {
        i64 s[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) s[u] = __ldcs(sums + i + u * 256);
        u32 m = 0, tie = 0;
#pragma unroll
        for (int u = 0; u < 16; ++u) m |= (u32)(s[u] > ths) << u, tie |= (u32)(s[u] == ths) << u;
        if (tie) {
#pragma unroll
          for (int u = 0; u < 16; ++u)
            s[u] = (tie >> u) & 1u ? __ldcs(keys + i + u * 256) : INT64_MAX;
#pragma unroll
          for (int u = 0; u < 16; ++u) m |= (tie >> u & (u32)(s[u] <= thk)) << u;
        }
        for (; m; m &= m - 1) {
          const i64 e = i + (__ffs(m) - 1) * 256;
          T.insert(keys[e], sums[e]);
        }
      }
    } else {
      for (; i + 3 * 256 < hi; i += 4 * 256) {  // four pairs' loads in flight
        i64 k[4], s[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) k[u] = __ldcs(keys + i + u * 256), s[u] = __ldcs(sums + i + u * 256);
#pragma unroll
        for (int u = 0; u < 4; ++u) T.insert(k[u], s[u]);
      }
    }
    for (; i < hi; i += blockDim.x) {
      const i64 xk = keys[i], xs = sums[i];
      if (!filt || xs > ths || (xs == ths && xk <= thk)) T.insert(xk, xs);
    }
    cnt = tk_lane_rank(T, K, s_lr, bk, bs);
  }
  TopList L;
  L.bind(s_scr[threadIdx.x >> 5]);
  if (cnt < 0) {
    L.clear();
    for (i64 b = lo; b < hi; b += blockDim.x) {
      const i64 i = b + threadIdx.x;
      const bool v = i < hi;
      L.offer(K, v, v ? keys[i] : 0, v ? sums[i] : 0);
    }
    tk_block_merge(L, K, sk, ss, sc);
    if (threadIdx.x < 32) {
      L.store(bk, bs);
      cnt = L.cnt;
    }
  }
  // Thread 0 holds the count on either path.
  if (nb == 1) {
    if (threadIdx.x == 0) *d_nout = cnt;
  } else {
    if (threadIdx.x == 0) part_c[blockIdx.x] = cnt;
    __threadfence();  // every thread's list writes, before the ticket
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(ticket, 1u) == (u32)nb - 1;
    __syncthreads();
    if (!s_last) return;
    // The last block merges the blocks' lists, read from L2 (other blocks
    // wrote them): entry e of the nb * K list slots is valid when its slot
    // is below its list's count.
    __threadfence();
    const int total = nb * K;
    cnt = -1;
    if (K <= 32) {
      LaneTop T;
      T.clear();
      for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int b = e / K;
        const int c = __ldcg(part_c + b);
        const i64 k = __ldcg(part_k + e), s = __ldcg(part_s + e);
        if (e - b * K < c) T.insert(k, s);
      }
      cnt = tk_lane_rank(T, K, s_lr, out_keys, out_sums);
    }
    if (cnt < 0) {
      // Each warp offers 32 of the list slots per round.
      L.clear();
      for (int base = (threadIdx.x >> 5) * 32; base < total; base += blockDim.x) {
        const int e = base + lane;
        bool v = false;
        i64 k = 0, s = 0;
        if (e < total) {
          const int b = e / K;
          const int c = __ldcg(part_c + b);
          k = __ldcg(part_k + e);
          s = __ldcg(part_s + e);
          v = e - b * K < c;
        }
        L.offer(K, v, k, s);
      }
      tk_block_merge(L, K, sk, ss, sc);
      if (threadIdx.x < 32) {
        L.store(out_keys, out_sums);
        cnt = L.cnt;
      }
    }
    if (threadIdx.x == 0) *d_nout = cnt;
  }
  // A plan's result record (out_keys, out_sums, d_nout point into it): the
  // rest of it from the plan's counters (groups, status, F rows).
  if (threadIdx.x == 0 && rec) {
    rec->ngroups = (i64)rec_ctr[0];
    rec->status = (int)rec_ctr[3];
    rec->reserved = 0;
    rec->hits = (i64)rec_ctr[2];
  }
}

template <typename T>
int filter_grid(pq_ctx* ctx, i64 n) {
  i64 tiles = (n + kFilterTile - 1) / kFilterTile;
  return (int)std::max<i64>(1, std::min<i64>(tiles, (i64)ctx->num_sms * 4));
}

template <typename T, bool SEL, bool VEC>
void launch_filter(pq_ctx* ctx, int grid, cudaStream_t s, const void* col, const i64* sel,
                   i64 n_cap, const i64* d_n, Pred p, i64* out, i64* d_count, u64* state,
                   u32* ctr) {
  k_filter<T, SEL, VEC><<<grid, 256, 0, s>>>((const T*)col, sel, n_cap, d_n, p, out, d_count,
                                             state, ctr, ctx->opt.spin_limit, ctx->d_status);
}

template <typename T, bool SEL>
void launch_filter_v(pq_ctx* ctx, bool vec, int grid, cudaStream_t s, const void* col,
                     const i64* sel, i64 n_cap, const i64* d_n, Pred p, i64* out, i64* d_count,
                     u64* state, u32* ctr) {
  if (vec) launch_filter<T, SEL, true>(ctx, grid, s, col, sel, n_cap, d_n, p, out, d_count, state, ctr);
  else launch_filter<T, SEL, false>(ctx, grid, s, col, sel, n_cap, d_n, p, out, d_count, state, ctr);
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

bool overlaps(const void* a, size_t a_bytes, const void* b, size_t b_bytes) {
  return (uintptr_t)a < (uintptr_t)b + b_bytes && (uintptr_t)b < (uintptr_t)a + a_bytes;
}

}  // namespace

namespace pqh {
namespace {
int topk_grid(pq_ctx* ctx, i64 n) {
  return (int)std::max<i64>(1, std::min<i64>((n + 2047) / 2048, (i64)ctx->num_sms * 2));
}
}  // namespace

size_t topk_scratch_bytes(pq_ctx* ctx, int64_t n, int k) {
  const int grid = topk_grid(ctx, n);
  return (size_t)grid * k * 16 + (size_t)grid * 4;
}

cudaError_t topk_launch(pq_ctx* ctx, const int64_t* keys, const int64_t* sums, int64_t n,
                        const int64_t* d_n, int k, int64_t* out_keys, int64_t* out_sums,
                        int64_t* d_nout, unsigned* ticket, void* lists, bool chained,
                        cudaStream_t s, const uint64_t* rec_ctr, pq_result* rec) {
  const int grid = topk_grid(ctx, n);
  i64* pk = (i64*)lists;
  i64* ps = pk + (i64)grid * k;
  int* pc = (int*)(ps + (i64)grid * k);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = chained ? 1 : 0;
  ctx->launches++;
  return cudaLaunchKernelEx(&cfg, k_topk, (const i64*)keys, (const i64*)sums, (i64)n,
                            (const i64*)d_n, k, pk, ps, pc, (u32*)ticket, (i64*)out_keys,
                            (i64*)out_sums, (i64*)d_nout, (const u64*)rec_ctr, rec);
}

}  // namespace pqh

#define PQ_DISPATCH_T(type, T, ...)              \
  switch (type) {                                \
    case PQ_INT8: { typedef signed char T; __VA_ARGS__; break; } \
    case PQ_INT32: { typedef int T; __VA_ARGS__; break; }        \
    default: { typedef long long T; __VA_ARGS__; break; }        \
  }

extern "C" {

pq_status pq_filter(pq_ctx* ctx, pq_col col, int op, int64_t c, const int64_t* sel_in,
                    int64_t n_in, const int64_t* d_n_in, int64_t* sel_out, int64_t* d_count,
                    void* stream) {
  if (!ctx) return PQ_ERR_INVALID_ARG;
  bool ok;
  Pred p = pqh::make_pred(op, c, &ok);
  if (!ok || !pqh::valid_dtype(col.type) || col.n < 0 || !d_count || col.reserved != 0)
    return pqh::fail(ctx, PQ_ERR_INVALID_ARG, "pq_filter: bad arguments");
  const bool sel = sel_in != nullptr;
  const i64 n_cap = sel ? n_in : col.n;
  if (n_cap < 0 || (n_cap > 0 && (!sel_out || (!col.data && col.n > 0))))
    return pqh::fail(ctx, PQ_ERR_INVALID_ARG, "pq_filter: bad arguments");
  if (d_n_in && !sel) return pqh::fail(ctx, PQ_ERR_INVALID_ARG, "pq_filter: d_n_in needs sel_in");
  cudaStream_t s = S(stream);
  if (n_cap == 0) {
    PQ_CUDA(ctx, cudaMemsetAsync(d_count, 0, sizeof(int64_t), s));
    return PQ_OK;
  }
  const bool vec = sel ? aligned16(sel_in) : aligned16(col.data);
  const i64 wtiles = (n_cap + kWarpTile - 1) / kWarpTile;
  // A selection refined in place: only the single pass reads a tile's ids
  // before any id is written over them.
  const bool in_place = sel && overlaps(sel_in, (size_t)n_cap * 8, sel_out, (size_t)n_cap * 8);
  if (wtiles <= kFilterOne && !in_place) {
    PQ_DISPATCH_T(col.type, T, {
      auto one = [&](auto k) {
        k<<<1, kFilterOne * 32, 0, s>>>((const T*)col.data, (const i64*)sel_in, n_cap,
                                        (const i64*)d_n_in, p, (i64*)sel_out, (i64*)d_count);
      };
      if (sel) vec ? one(k_filter_one<T, true, true>) : one(k_filter_one<T, true, false>);
      else vec ? one(k_filter_one<T, false, true>) : one(k_filter_one<T, false, false>);
    });
    PQ_LAUNCHED(ctx);
    return PQ_OK;
  }
  pqh::Scratch scr(ctx, s);
  // At least two warp tiles per warp, at most one wave of blocks.
  const int g = (int)std::max<i64>(1, std::min<i64>((wtiles + 15) / 16,
                                                       (i64)ctx->num_sms * filter_blocks(sel || col.type == PQ_INT64)));
  // Scratch of a capture is kept for the graph's replays: only the counts (the
  // bits of 2^18 rows take as much; small calls do not ask, it costs 1 us).
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (n_cap > 1 << 18) cudaStreamIsCapturing(s, &cap);
  const bool keep = cap == cudaStreamCaptureStatusNone;
  const size_t bits_b = keep ? (size_t)wtiles * 64 : 0, cnt_b = (size_t)g * 9 * 4;
  if (char* w = in_place ? nullptr : (char*)scr.get(bits_b + cnt_b)) {
    unsigned short* bits = keep ? (unsigned short*)w : nullptr;
    u32* block_cnt = (u32*)(w + bits_b);
    u32* warp_cnt = block_cnt + g;
    PQ_DISPATCH_T(col.type, T, {
      auto mark = [&](auto k) {
        k<<<g, 256, 0, s>>>((const T*)col.data, (const i64*)sel_in, n_cap, (const i64*)d_n_in, p,
                            bits, warp_cnt, block_cnt);
      };
      if (sel) vec ? mark(k_filter_mark<T, true, true>) : mark(k_filter_mark<T, true, false>);
      else vec ? mark(k_filter_mark<T, false, true>) : mark(k_filter_mark<T, false, false>);
    });
    PQ_LAUNCHED(ctx);
    if (keep) {
      auto emit = [&](auto k) {
        k<<<g, 256, 0, s>>>((const i64*)sel_in, n_cap, (const i64*)d_n_in, bits, warp_cnt,
                            block_cnt, (i64*)sel_out, (i64*)d_count);
      };
      sel ? emit(k_filter_emit<true>) : emit(k_filter_emit<false>);
    } else {
      PQ_DISPATCH_T(col.type, T, {
        auto again = [&](auto k) {
          k<<<g, 256, 0, s>>>((const T*)col.data, (const i64*)sel_in, n_cap, (const i64*)d_n_in,
                              p, warp_cnt, block_cnt, (i64*)sel_out, (i64*)d_count);
        };
        if (sel) vec ? again(k_filter_again<T, true, true>) : again(k_filter_again<T, true, false>);
        else vec ? again(k_filter_again<T, false, true>) : again(k_filter_again<T, false, false>);
      });
    }
    PQ_LAUNCHED(ctx);
    return PQ_OK;
  }
  // In place, or no room for the bits (n / 8 bytes): the single pass with
  // look-back, whose scratch is 8 bytes per 4096 rows.
  PQ_CUDA(ctx, cudaMemsetAsync(d_count, 0, sizeof(int64_t), s));
  const i64 ntiles = (n_cap + kFilterTile - 1) / kFilterTile;
  char* w = (char*)scr.get(ntiles * 8 + 256);
  if (!w) return pqh::fail(ctx, PQ_ERR_BUDGET, "pq_filter: no scratch");
  u64* state = (u64*)(w + 256);
  u32* ctr = (u32*)w;
  PQ_CUDA(ctx, cudaMemsetAsync(w, 0, ntiles * 8 + 256, s));
  const int grid = filter_grid<int>(ctx, n_cap);
  PQ_DISPATCH_T(col.type, T, {
    if (sel)
      launch_filter_v<T, true>(ctx, vec, grid, s, col.data, (const i64*)sel_in, n_cap,
                               (const i64*)d_n_in, p, (i64*)sel_out, (i64*)d_count, state, ctr);
    else
      launch_filter_v<T, false>(ctx, vec, grid, s, col.data, nullptr, n_cap, nullptr, p,
                                (i64*)sel_out, (i64*)d_count, state, ctr);
  });
  PQ_LAUNCHED(ctx);
  return PQ_OK;
}

}  // extern "C"

namespace {
constexpr int kPartSmem = 200 * 1024;  // most dynamic shared memory of a scatter
// One stable pass of the partition: rows ordered by digit `dg` of their
// bucket.  d_offsets: the digits' offsets (or null); tot: null, or counts of
// whole buckets to be added to (zeroed by the caller).
template <bool PART>
pq_status part_pass(pq_ctx* ctx, pq_col key, const pq_col* payload, int npay, Digit<PART> dg,
                    void* out_key, void* const* out_payload, i64* d_offsets, u64* tot,
                    cudaStream_t s) {
  const i64 n = key.n;
  const int P = dg.count();
  PayArgs pa{};
  pa.n = npay;
  for (int j = 0; j < npay; ++j) {
    pa.src[j] = payload[j].data;
    pa.dst[j] = out_payload[j];
    pa.type[j] = payload[j].type;
  }
  // Staged scatter: G persistent blocks, one chunk of rows each; with bulk
  // copies into double-buffered sub-tiles when every column is 16-byte
  // aligned and the buffers fit.
  TmaCols tc{};
  tc.n = 1 + npay;
  tc.src[0] = key.data;
  tc.dst[0] = out_key;
  tc.es[0] = (int)pqh::dtype_size(key.type);
  bool aligned = ((uintptr_t)key.data & 15) == 0 && ((uintptr_t)out_key & 15) == 0;
  for (int j = 0; j < npay; ++j) {
    tc.src[1 + j] = payload[j].data;
    tc.dst[1 + j] = out_payload[j];
    tc.es[1 + j] = (int)pqh::dtype_size(payload[j].type);
    aligned = aligned && ((uintptr_t)payload[j].data & 15) == 0;
  }
  // Sub-tiles of 4096 rows from 512 buckets on (when they fit; of 5 to 8 bytes a
  // row from 256 on), so that a bucket's run in a sub-tile fills its sectors;
  // 2048 otherwise.  By 256, 60M rows of 8 bytes: 565 -> 445 us, of 4 bytes 460
  // -> 468; 4M of 8 bytes 70 -> 73.
  auto layout = [&](int rows) {
    int off = 0;
    for (int c = 0; c < tc.n; ++c) tc.off[c] = off, off += rows * tc.es[c];
    tc.buf_bytes = off;
    return tma_smem(P, tc.buf_bytes, rows);
  };
  int sub = 4096;
  size_t smem = layout(sub);
  const int row_bytes = tc.buf_bytes / sub;
  const bool runs = dg.bits >= 9 || (dg.bits == 8 && row_bytes > 4 && row_bytes <= 8);
  if (!runs || smem > kPartSmem) smem = layout(sub = kSub);
  const bool use_tma = aligned && smem <= kPartSmem;
  if (!use_tma) sub = kSub, smem = staged_smem(P);
  // Blocks per SM: by shared memory (228 KB, 1 KB and the static part of it
  // taken per block) and, at most, by registers.
  // 9-byte rows, of which four blocks fit, gain by them up to 64 buckets (60M by
  // 32: 447 us at four, 463 at three; by 128 607 and 560).
  i64 occ = std::max<i64>(1, std::min<i64>(use_tma ? 5 : 6, 228 * 1024 / (i64)(smem + 1024 + 256)));
  const bool bound = PART || sub == 4096 || occ <= 3 || (occ == 4 && dg.bits >= 7);
  if (use_tma && bound) occ = std::min<i64>(occ, 3);
  const i64 g = std::max<i64>(1, std::min<i64>((n + sub - 1) / sub, (i64)ctx->num_sms * occ));
  const i64 m = g * P;
  const i64 stiles = (m + 4095) / 4096;
  // One block of scratch: the scan's state and the histogram (both zeroed),
  // then the scanned offsets.
  pqh::Scratch scr(ctx, s);
  const size_t w_b = (size_t)(stiles * 8 + 256 + 255) / 256 * 256;
  const size_t hist_b = (size_t)(m * 4 + 255) / 256 * 256;
  char* w = (char*)scr.get(w_b + hist_b + m * 8);
  if (!w) return pqh::fail(ctx, PQ_ERR_BUDGET, "pq_partition: no scratch");
  u32* hist = (u32*)(w + w_b);
  i64* gofs = (i64*)(w + w_b + hist_b);
  PQ_CUDA(ctx, cudaMemsetAsync(w, 0, w_b + hist_b, s));
  // Histogram blocks: at most one wave of eight per SM (hsplit blocks per
  // chunk), each with at least 4096 rows; one per chunk where whole buckets
  // are counted, so that fewer blocks add their counts of up to 4096 buckets.
  const int hsplit = tot ? 1 : (int)std::max<i64>(
      1, std::min<i64>(((i64)ctx->num_sms * 8) / g, (n / g) / 4096));
  PQ_DISPATCH_T(key.type, T, {
    const size_t hist_smem = (size_t)(tot ? 1 << dg.log2P : P) * 4;
    auto count = [&](auto k) {
      k<<<(unsigned)(g * hsplit), 256, hist_smem, s>>>((const T*)key.data, n, dg, hist, g, hsplit,
                                                       tot);
    };
    if constexpr (PART) tot ? count(k_part_hist_blk<T, PART, true>) : count(k_part_hist_blk<T, PART, false>);
    else count(k_part_hist_blk<T, PART, false>);
    PQ_LAUNCHED(ctx);
    k_scan_u32<<<(unsigned)std::min<i64>(stiles, (i64)ctx->num_sms * 4), 256, 0, s>>>(
        hist, m, gofs, (u64*)(w + 256), (u32*)w, ctx->opt.spin_limit, ctx->d_status);
    PQ_LAUNCHED(ctx);
    auto launch = [&](int variant, auto k, auto... args) -> pq_status {
      // Once per context, and the same limit whatever this call needs: another
      // thread may be between its own setting and its launch.
      const uint32_t bit = 1u << ((key.type - 1) * 8 + variant);
      if (!(ctx->part_ready.load(std::memory_order_acquire) & bit)) {
        PQ_CUDA(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kPartSmem));
        ctx->part_ready.fetch_or(bit, std::memory_order_release);
      }
      k<<<(unsigned)g, 256, smem, s>>>(args...);
      PQ_LAUNCHED(ctx);
      return PQ_OK;
    };
    if (!use_tma)
      return launch(PART ? 1 : 0, k_part_scatter_blk<T, PART>, (const T*)key.data, n, dg, (const i64*)gofs, pa,
                    (T*)out_key, d_offsets);
    auto scatter = [&](int variant, auto k) {
      return launch(variant, k, n, dg, (const i64*)gofs, tc, d_offsets, (i64)ctx->opt.spin_limit,
                    ctx->d_status);
    };
    if constexpr (!PART) {  // a part has 64 digits at most
      if (sub == 4096) return scatter(2, k_part_scatter_tma<T, PART, 4096, 3>);
      if (!bound) return scatter(3, k_part_scatter_tma<T, PART, kSub, 0>);
    }
    return scatter(PART ? 4 : 5, k_part_scatter_tma<T, PART, kSub, 3>);
  });
  return PQ_OK;
}

// Whether a partition takes two passes: each writes runs of 64 and more rows
// per bucket and sub-tile, where one pass by 1024 buckets writes runs of two
// to four (partly written sectors, and 8 x 1024 counters a sub-tile that leave
// room for one block per SM), and above that 8192-row tiles are scattered row
// by row.  It moves the rows twice and takes six more launches and clears, so it
// pays from some size on.  Uniform keys, 20M rows of 21 bytes by 1024: 0.94 ->
// 0.46 ms (clustered keys 0.67 -> 0.44), 60M of 16 bytes 1.20 -> 0.99 ms (20M of
// them 0.40 either way; by 512 buckets one pass is faster, 0.97 against 0.99 ms);
// 20M rows of 16 bytes by 2048 0.94 -> 0.40 ms, by 4096 1.44 -> 0.41 ms; 4M of
// them by 2048 0.22 -> 0.15 ms, by 4096 0.34 -> 0.16.
bool part_two_passes(int log2P, i64 n, const pq_col& key, const pq_col* payload, int npay) {
  i64 row = (i64)pqh::dtype_size(key.type);
  for (int j = 0; j < npay; ++j) row += (i64)pqh::dtype_size(payload[j].type);
  const i64 bytes = n * row;
  return bytes >= (log2P == 10 ? 320LL << 20 : log2P == 11 ? 48LL << 20 : 16LL << 20) &&
         log2P >= 10;
}
}  // namespace

extern "C" {

pq_status pq_partition(pq_ctx* ctx, pq_col key, const pq_col* payload, int npay, int log2P,
                       void* out_key, void* const* out_payload, int64_t* d_offsets,
                       void* stream) {
  if (!ctx) return PQ_ERR_INVALID_ARG;
  if (log2P < 0 || log2P > PQ_MAX_LOG2P || npay < 0 || npay > PQ_MAX_PAYLOAD || !d_offsets ||
      (key.type != PQ_INT32 && key.type != PQ_INT64) || key.n < 0 || key.reserved != 0 ||
      (npay > 0 && (!payload || !out_payload)))
    return pqh::fail(ctx, PQ_ERR_INVALID_ARG, "pq_partition: bad arguments");
  PayArgs pa{};
  pa.n = npay;
  for (int j = 0; j < npay; ++j) {
    if (!pqh::valid_dtype(payload[j].type) || payload[j].n != key.n ||
        (key.n && (!payload[j].data || !out_payload[j])))
      return pqh::fail(ctx, PQ_ERR_INVALID_ARG, "pq_partition: payload %d", j);
    pa.src[j] = payload[j].data;
    pa.dst[j] = out_payload[j];
    pa.type[j] = payload[j].type;
  }
  cudaStream_t s = S(stream);
  const i64 n = key.n;
  const int P = 1 << log2P;
  if (n == 0) {
    PQ_CUDA(ctx, cudaMemsetAsync(d_offsets, 0, (P + 1) * sizeof(int64_t), s));
    return PQ_OK;
  }
  if (!key.data || !out_key) return pqh::fail(ctx, PQ_ERR_INVALID_ARG, "pq_partition: null key");
  // Many buckets: two stable passes, by the low half of the bucket number into
  // scratch and by the high half into the output, when the scratch fits.
  // Not while the stream is being captured: scratch is then kept for the
  // graph's replays, and a second copy of the rows is too much to keep.
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (part_two_passes(log2P, n, key, payload, npay) &&
      cudaStreamIsCapturing(s, &cap) == cudaSuccess && cap == cudaStreamCaptureStatusNone) {
    pqh::Scratch scr(ctx, s);
    size_t bytes = 0;
    auto put = [&](int type) {
      const size_t at = bytes;
      bytes += ((size_t)n * pqh::dtype_size(type) + 255) / 256 * 256;
      return at;
    };
    size_t at[1 + PQ_MAX_PAYLOAD];
    at[0] = put(key.type);
    for (int j = 0; j < npay; ++j) at[1 + j] = put(payload[j].type);
    char* w = (char*)scr.get(bytes);
    const size_t tot_b = (size_t)P * 8;
    u64* tot = w ? (u64*)scr.get(tot_b) : nullptr;
    if (tot) {
      PQ_CUDA(ctx, cudaMemsetAsync(tot, 0, tot_b, s));
      const int lo = log2P / 2;
      pq_col k1 = key, p1[PQ_MAX_PAYLOAD];
      void* o1[PQ_MAX_PAYLOAD];
      k1.data = w + at[0];
      for (int j = 0; j < npay; ++j) p1[j] = payload[j], p1[j].data = o1[j] = w + at[1 + j];
      pq_status st = part_pass(ctx, key, payload, npay, Digit<true>(log2P, 0, lo), w + at[0], o1, nullptr,
                               tot, s);
      if (st == PQ_OK)
        st = part_pass(ctx, k1, p1, npay, Digit<true>(log2P, lo, log2P - lo), out_key, out_payload,
                       nullptr, nullptr, s);
      if (st == PQ_OK) {
        k_part_offsets<<<1, 1024, 0, s>>>(tot, P, n, (i64*)d_offsets);
        PQ_LAUNCHED(ctx);
        return PQ_OK;
      }
      if (st != PQ_ERR_BUDGET) return st;
    }
  }
  if (log2P <= kStagedMaxLog2)
    return part_pass(ctx, key, payload, npay, Digit<false>(log2P, 0, log2P), out_key, out_payload,
                     (i64*)d_offsets, nullptr, s);
  const i64 ntiles = (n + kPartTile - 1) / kPartTile;
  const i64 m = ntiles * P;
  const i64 stiles = (m + 4095) / 4096;
  pqh::Scratch scr(ctx, s);
  u32* hist = (u32*)scr.get(m * 4);
  i64* gofs = (i64*)scr.get(m * 8);
  char* w = (char*)scr.get(stiles * 8 + 256);
  if (!hist || !gofs || !w) return pqh::fail(ctx, PQ_ERR_BUDGET, "pq_partition: no scratch");
  PQ_CUDA(ctx, cudaMemsetAsync(w, 0, stiles * 8 + 256, s));
  const size_t smem_hist = (size_t)P * 4, smem_scatter = (size_t)8 * P * 4;
  PQ_DISPATCH_T(key.type, T, {
    if (smem_scatter > 48 * 1024)
      cudaFuncSetAttribute(k_part_scatter<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem_scatter);
    k_part_hist<T><<<(unsigned)ntiles, 256, smem_hist, s>>>((const T*)key.data, n, log2P, hist,
                                                            ntiles);
    PQ_LAUNCHED(ctx);
    k_scan_u32<<<(unsigned)std::min<i64>(stiles, (i64)ctx->num_sms * 4), 256, 0, s>>>(
        hist, m, gofs, (u64*)(w + 256), (u32*)w, ctx->opt.spin_limit, ctx->d_status);
    PQ_LAUNCHED(ctx);
    k_part_scatter<T><<<(unsigned)ntiles, 256, smem_scatter, s>>>(
        (const T*)key.data, n, log2P, gofs, ntiles, pa, (T*)out_key, (i64*)d_offsets);
  });
  PQ_LAUNCHED(ctx);
  return PQ_OK;
}

pq_status pq_join_build(pq_ctx* ctx, pq_col key, pq_col val, float load_factor, pq_ht** out,
                        void* stream) {
  if (!ctx || !out) return PQ_ERR_INVALID_ARG;
  *out = nullptr;
  if (load_factor <= 0) load_factor = ctx->opt.load_factor;
  if (!pqh::valid_dtype(key.type) || key.n < 0 || (key.n && !key.data) || load_factor < 0.05f ||
      load_factor > 0.9f || (val.data && (!pqh::valid_dtype(val.type) || val.n != key.n)))
    return pqh::fail(ctx, PQ_ERR_INVALID_ARG, "pq_join_build: bad arguments");
  cudaStream_t s = S(stream);
  const int lf = (int)(load_factor * 1024 + 0.5f);
  const int log2cap = cap_log2(key.n, lf);
  const i64 cap = (i64)1 << log2cap;
  auto* ht = new pq_ht();
  ht->block = ctx->arena.alloc((size_t)cap * 16 + 256);
  if (!ht->block) {
    delete ht;
    return pqh::fail(ctx, PQ_ERR_BUDGET, "pq_join_build: table of %lld slots", (long long)cap);
  }
  ht->meta = (i64*)ht->block;
  ht->keys = (i64*)((char*)ht->block + 256);  // {key, value} per slot
  ht->vals = ht->keys + 1;
  ht->log2cap = log2cap;
  ht->n = key.n;
  HtMeta* const meta = (HtMeta*)ht->meta;
  // Both builds are launched where the sample decides (on the device): the one
  // that is not meant returns at once.
  const int look = key.n >= kHtSpreadMin;
  const pq_status st = [&]() -> pq_status {
    PQ_CUDA(ctx, cudaMemsetAsync(ht->meta, 0, 256, s));
    const int gc = (int)std::min<i64>((cap + 2047) / 2048, (i64)ctx->num_sms * 4) + look;
    const int grid = (int)std::min<i64>((key.n + 255) / 256, (i64)ctx->num_sms * 8);
    PQ_DISPATCH_T(key.type, TK, {
      const TK* k = (const TK*)key.data;
      k_ht_clear<TK><<<gc, kHtSample, 0, s>>>((longlong2*)ht->keys, log2cap, k, key.n, meta, look);
      PQ_LAUNCHED(ctx);
      if (key.n == 0) return PQ_OK;
      auto build = [&](auto tag) -> pq_status {
        using TV = decltype(tag);
        k_ht_build<TK, TV><<<grid, 256, 0, s>>>(k, (const TV*)val.data, key.n, ht->keys, log2cap,
                                                meta, look, ctx->d_status);
        PQ_LAUNCHED(ctx);
        if (!look) return PQ_OK;
        k_ht_build_spread<TK, TV><<<grid, 256, 0, s>>>(k, (const TV*)val.data, key.n, ht->keys,
                                                       log2cap, meta, ctx->d_status);
        PQ_LAUNCHED(ctx);
        return PQ_OK;
      };
      if (!val.data) return build((long long)0);
      PQ_DISPATCH_T(val.type, TV, { return build(TV()); });
    });
    return PQ_OK;
  }();
  if (st != PQ_OK) {
    ctx->arena.release(ht->block, s);
    delete ht;
    return st;
  }
  *out = ht;
  return PQ_OK;
}

pq_status pq_join_probe(pq_ctx* ctx, const pq_ht* ht, pq_col probe_key, int64_t* out_probe_row,
                        int64_t* out_build_val, int64_t cap, int64_t* d_count, void* stream) {
  if (!ctx || !ht || !d_count || cap < 0 || !pqh::valid_dtype(probe_key.type) ||
      probe_key.n < 0 || (probe_key.n && !probe_key.data) ||
      (cap > 0 && (!out_probe_row || !out_build_val)))
    return pqh::fail(ctx, PQ_ERR_INVALID_ARG, "pq_join_probe: bad arguments");
  cudaStream_t s = S(stream);
  PQ_CUDA(ctx, cudaMemsetAsync(d_count, 0, sizeof(int64_t), s));
  if (probe_key.n == 0) return PQ_OK;
  PQ_DISPATCH_T(probe_key.type, TK, {
    const int grid = (int)std::min<i64>((probe_key.n + 511) / 512, (i64)ctx->num_sms * kPrbBlocks);
    k_ht_probe<TK><<<grid, 256, 0, s>>>((const TK*)probe_key.data, probe_key.n,
                                        (const longlong2*)ht->keys, ht->log2cap,
                                        (const HtMeta*)ht->meta, (i64*)out_probe_row,
                                        (i64*)out_build_val, cap, (u64*)d_count);
  });
  PQ_LAUNCHED(ctx);
  k_check_cap<<<1, 1, 0, s>>>((const i64*)d_count, cap, ctx->d_status);
  PQ_LAUNCHED(ctx);
  return PQ_OK;
}

pq_status pq_groupby_sum(pq_ctx* ctx, pq_col key, pq_col val, int64_t* out_keys,
                         int64_t* out_sums, int64_t cap, int64_t* d_ngroups, void* stream) {
  if (!ctx || !d_ngroups || cap < 0 || !pqh::valid_dtype(key.type) || !pqh::valid_dtype(val.type) ||
      key.n < 0 || val.n != key.n || (key.n && (!key.data || !val.data)) ||
      (cap > 0 && (!out_keys || !out_sums)))
    return pqh::fail(ctx, PQ_ERR_INVALID_ARG, "pq_groupby_sum: bad arguments");
  cudaStream_t s = S(stream);
  PQ_CUDA(ctx, cudaMemsetAsync(d_ngroups, 0, sizeof(int64_t), s));
  if (key.n == 0) return PQ_OK;
  const bool vec = aligned16(key.data) && aligned16(val.data);
  const int lf = (int)(ctx->opt.load_factor * 1024 + 0.5f);
  const int log2cap = cap_log2(std::min<i64>(key.n, std::max<i64>(cap, 1)), lf);
  const i64 slots = (i64)1 << log2cap;
  pqh::Scratch tscr(ctx, s);
  auto table = [&]() { return (i64*)tscr.get((size_t)slots * 16); };
  const bool pairs = (size_t)slots * 16 > kGbPairBytes;
  auto layout = [&](i64* tab) {
    return GbTable{tab, tab + (pairs ? 1 : slots), log2cap};
  };
  // Clear and fill the hash table; runs: at least 128 rows per warp.
  const int grid = (int)std::min<i64>((key.n + 1023) / 1024, (i64)ctx->num_sms * 6);
  const int grid1 = (int)std::min<i64>((key.n + 255) / 256, (i64)ctx->num_sms * 8);
  auto insert = [&](i64* tab, bool hot, u32* over) -> pq_status {
    k_gb_clear<<<(int)std::min<i64>((slots + 255) / 256, (i64)ctx->num_sms * 8), 256, 0, s>>>(
        (longlong2*)tab, slots, pairs);
    PQ_LAUNCHED(ctx);
    PQ_DISPATCH_T(key.type, TK, {
      PQ_DISPATCH_T(val.type, TV, {
        auto ins = [&](auto k, int g) {
          k<<<g, 256, 0, s>>>((const TK*)key.data, (const TV*)val.data, key.n, layout(tab),
                              ctx->d_status, over);
        };
        if (!hot)
          pairs ? ins(k_gb_rows<TK, TV, 2>, grid1) : ins(k_gb_rows<TK, TV, 1>, grid1);
        else if (vec)
          pairs ? ins(k_gb_insert<TK, TV, true, 2>, grid) : ins(k_gb_insert<TK, TV, true, 1>, grid);
        else
          pairs ? ins(k_gb_insert<TK, TV, false, 2>, grid) : ins(k_gb_insert<TK, TV, false, 1>, grid);
      });
    });
    PQ_LAUNCHED(ctx);
    return PQ_OK;
  };
  auto emit = [&](i64* tab, const u32* over) -> pq_status {
    const int g = (int)std::min<i64>((slots + 2047) / 2048, (i64)ctx->num_sms * 8);
    auto em = [&](auto k) {
      k<<<g, 256, 0, s>>>(layout(tab), (i64*)out_keys, (i64*)out_sums, cap, (u64*)d_ngroups, over);
    };
    pairs ? em(k_gb_emit<2>) : em(k_gb_emit<1>);
    PQ_LAUNCHED(ctx);
    return PQ_OK;
  };
  bool hot = false;  // a sample met a frequent key
  // Large inputs outside stream capture: one read of the keys and one small
  // read-back tell whether they come in order (groups are then their runs),
  // and their range; dense keys take the slot array.
  cudaStreamCaptureStatus capst = cudaStreamCaptureStatusNone;
  cudaStreamIsCapturing(s, &capst);
  if (capst == cudaStreamCaptureStatusNone && key.n >= (1 << 20)) {
    pqh::Scratch rs(ctx, s);
    const int g = ctx->num_sms * kGbScanBlocks, nw = g * 8;
    const size_t base_b = 256 + (size_t)(nw + 1) * 8;
    char* w = (char*)rs.get(base_b + (size_t)nw * sizeof(GbWarp));
    if (w) {
      GbSummary* sum = (GbSummary*)w;
      i64* base = (i64*)(w + 256);
      GbWarp* winfo = (GbWarp*)(w + base_b);
      PQ_CUDA(ctx, cudaMemsetAsync(sum, 0, sizeof(GbSummary), s));
      PQ_CUDA(ctx, cudaMemsetAsync(&sum->umin, 0xFF, 8, s));
      PQ_DISPATCH_T(key.type, TK, {
        if (vec) k_gb_scan<TK, true><<<g + 1, 256, 0, s>>>((const TK*)key.data, key.n, winfo, sum);
        else k_gb_scan<TK, false><<<g + 1, 256, 0, s>>>((const TK*)key.data, key.n, winfo, sum);
      });
      PQ_LAUNCHED(ctx);
      k_gb_bounds<<<1, 1024, 0, s>>>(winfo, nw, base, sum);
      PQ_LAUNCHED(ctx);
      pqh::SmallPinned hp(ctx);
      PQ_CUDA(ctx, cudaMemcpyAsync(hp.p, sum, sizeof(GbSummary), cudaMemcpyDeviceToHost, s));
      PQ_CUDA(ctx, cudaStreamSynchronize(s));
      GbSummary m;
      memcpy(&m, hp.p, sizeof m);
      hot = m.top >= kGbTopHot;
      // In order, or in order but for one descent with few runs after it (a
      // late part appended to an ordered table); the reserved key (ukey 0)
      // goes to the tables, which report it.
      const i64 tail = m.runs - m.first;
      // The runs' groups are written while other rows are read: not over the
      // inputs.  The tables write after the last read.
      const size_t out_b = (size_t)std::min<i64>(key.n, cap) * 8;
      bool over_inputs = false;
      for (const pq_col& c : {key, val})
        for (const int64_t* o : {out_keys, out_sums})
          over_inputs |= overlaps(o, out_b, c.data, (size_t)c.n * pqh::dtype_size(c.type));
      if (m.umin != 0 && !over_inputs && (m.descents == 0 ||
                                          (m.descents == 1 && tail <= key.n / 8 &&
                                           m.first <= cap))) {
        pqh::Scratch ts(ctx, s);
        i64* tk = tail ? (i64*)ts.get((size_t)tail * 16) : nullptr;
        if (!tail || tk) {
          const GbOut o = {(i64*)out_keys, (i64*)out_sums, cap, m.first, tk, tk ? tk + tail : tk};
          k_gb_joins<<<(nw + 255) / 256, 256, 0, s>>>(winfo, base, nw, o, (i64*)d_ngroups);
          PQ_LAUNCHED(ctx);
          PQ_DISPATCH_T(key.type, TK, {
            PQ_DISPATCH_T(val.type, TV, {
              auto runs = [&](auto k) {
                k<<<g, 256, 0, s>>>((const TK*)key.data, (const TV*)val.data, key.n, winfo, base, o);
              };
              vec ? runs(k_gb_runs<TK, TV, true>) : runs(k_gb_runs<TK, TV, false>);
            });
          });
          PQ_LAUNCHED(ctx);
          if (tail) {
            k_gb_fold<<<(unsigned)((tail + 255) / 256), 256, 0, s>>>(o, tail, (i64*)d_ngroups);
            PQ_LAUNCHED(ctx);
          }
          k_check_cap<<<1, 1, 0, s>>>((const i64*)d_ngroups, cap, ctx->d_status);
          PQ_LAUNCHED(ctx);
          return PQ_OK;
        }
      }
      const u64 span = m.umax >= m.umin ? m.umax - m.umin + 1 : 0;
      if (span && span <= 4 * (u64)key.n && span <= (1ULL << 34)) {
        pqh::Scratch scr(ctx, s);
        const size_t sb = (size_t)((span * 8 + 255) / 256 * 256);
        const size_t bb = (size_t)(((span + 31) / 32 * 4 + 255) / 256 * 256);
        char* blk = (char*)scr.get(sb + bb);
        if (blk) {
          // Rows in no order with frequent keys: what counts is how much memory
          // the other groups take (30M Zipf rows, 7.5M groups in a range of 30M:
          // slot array of 240 MB 0.94 ms, hash table of 134 MB 0.45 ms).  Without
          // frequent keys the slot array's reductions, which nobody waits for,
          // are ahead of the look-ups whatever their memory (40M rows, 400000
          // groups in a range of 26M: 0.62 ms, hash table of 16 MB 0.96 ms), and
          // rows in runs follow its order.  The hash table holds `cap` groups; the
          // slot array takes over, decided on the device, when there are more, as
          // every group is counted.
          i64* const tab = hot && m.runs > key.n / 2 && span > (u64)slots ? table() : nullptr;
          u32* const over = tab ? &sum->over : nullptr;
          i64* sums = (i64*)blk;
          u32* bm = (u32*)(blk + sb);
          if (tab) {
            const pq_status st = insert(tab, hot, over);
            if (st != PQ_OK) return st;
            k_gb_zero_if<<<ctx->num_sms * 8, 256, 0, s>>>((longlong2*)blk, (i64)((sb + bb) / 16),
                                                          over);
            PQ_LAUNCHED(ctx);
          } else {
            PQ_CUDA(ctx, cudaMemsetAsync(blk, 0, sb + bb, s));
          }
          PQ_DISPATCH_T(key.type, TK, {
            PQ_DISPATCH_T(val.type, TV, {
              const int gd = hot ? grid : (int)std::min<i64>((key.n + 1023) / 1024,
                                                             (i64)ctx->num_sms * 8);
              auto dense = [&](auto k) {
                k<<<gd, 256, 0, s>>>((const TK*)key.data, (const TV*)val.data, key.n, m.umin,
                                       span, sums, bm, ctx->d_status, over);
              };
              if (hot) vec ? dense(k_gb_dense<TK, TV, true, true>) : dense(k_gb_dense<TK, TV, false, true>);
              else vec ? dense(k_gb_dense<TK, TV, true, false>) : dense(k_gb_dense<TK, TV, false, false>);
            });
          });
          PQ_LAUNCHED(ctx);
          const i64 words = (i64)((span + 31) / 32);
          const int ge = (int)std::max<i64>(1, std::min<i64>((words + 255) / 256, (i64)ctx->num_sms * 8));
          k_gb_dense_emit<<<ge, 256, 0, s>>>(bm, sums, span, m.umin, (i64*)out_keys,
                                             (i64*)out_sums, cap, (u64*)d_ngroups, over);
          PQ_LAUNCHED(ctx);
          if (tab) {
            const pq_status st = emit(tab, over);
            if (st != PQ_OK) return st;
          }
          k_check_cap<<<1, 1, 0, s>>>((const i64*)d_ngroups, cap, ctx->d_status);
          PQ_LAUNCHED(ctx);
          return PQ_OK;
        }
      }
    }
  }
  i64* const tab = table();
  if (!tab) return pqh::fail(ctx, PQ_ERR_BUDGET, "pq_groupby_sum: table of %lld slots",
                             (long long)slots);
  pq_status st = insert(tab, hot, nullptr);
  if (st == PQ_OK) st = emit(tab, nullptr);
  if (st != PQ_OK) return st;
  k_check_cap<<<1, 1, 0, s>>>((const i64*)d_ngroups, cap, ctx->d_status);
  PQ_LAUNCHED(ctx);
  return PQ_OK;
}

pq_status pq_topk(pq_ctx* ctx, const int64_t* keys, const int64_t* sums, int64_t n,
                  const int64_t* d_n, int k, int64_t* out_keys, int64_t* out_sums,
                  int64_t* d_nout, void* stream) {
  if (!ctx || k < 1 || k > PQ_MAX_K || n < 0 || !d_nout || !out_keys || !out_sums ||
      (n > 0 && (!keys || !sums)))
    return pqh::fail(ctx, PQ_ERR_INVALID_ARG, "pq_topk: bad arguments");
  cudaStream_t s = S(stream);
  PQ_CUDA(ctx, cudaMemsetAsync(d_nout, 0, sizeof(int64_t), s));
  if (n == 0) return PQ_OK;
  pqh::Scratch scr(ctx, s);
  char* w = (char*)scr.get(pqh::topk_scratch_bytes(ctx, n, k) + 256);
  if (!w) return pqh::fail(ctx, PQ_ERR_BUDGET, "pq_topk: no scratch");
  PQ_CUDA(ctx, cudaMemsetAsync(w, 0, 256, s));
  PQ_CUDA(ctx, pqh::topk_launch(ctx, keys, sums, n, d_n, k, out_keys, out_sums, d_nout,
                                (unsigned*)w, w + 256, false, s));
  return PQ_OK;
}

}  // extern "C"

// ===================================================== allocation-free filter ====
// pq_filter takes its scratch from the context's arena.  Some callers cannot
// allocate device memory at all (for example code that runs while a CUDA graph
// is being captured, or inside a runtime that owns every allocation and forbids
// others), and they may not have a context either.  For them the single-pass
// kernel with look-back (k_filter, pq_filter's way in place and without scratch
// for its bits) runs with its tile states in
// this file-scope device array: a fixed 1 MiB of tile states plus a small
// header, which every GPU that loads the library keeps until the process
// exits.  All calls share the array, so calls that overlap on the GPU race;
// each call clears the part it uses before its kernel runs.
namespace {

constexpr i64 kNoAllocTiles = 1 << 17;                  // 131072 tiles
constexpr i64 kNoAllocRows = kNoAllocTiles * kFilterTile;  // 536,870,912 rows
constexpr int kNoAllocHeader = 32;                      // words: ticket, status

__device__ __align__(256) u64 g_noalloc_scratch[kNoAllocHeader + kNoAllocTiles];

struct NoAllocDevice {
  std::once_flag once;
  cudaError_t err = cudaSuccess;
  u64* scratch = nullptr;  // device address of g_noalloc_scratch
  int sms = 0;
};
NoAllocDevice g_noalloc_dev[256];

// Per-device set-up, run once with that device current: the host cannot use
// the array's name as a device address, so it asks the runtime for it.
cudaError_t noalloc_setup(int dev, NoAllocDevice** out) {
  if (dev < 0 || dev >= 256) return cudaErrorInvalidDevice;
  NoAllocDevice& d = g_noalloc_dev[dev];
  std::call_once(d.once, [&d, dev] {
    d.err = cudaGetSymbolAddress((void**)&d.scratch, g_noalloc_scratch);
    if (d.err == cudaSuccess)
      d.err = cudaDeviceGetAttribute(&d.sms, cudaDevAttrMultiProcessorCount, dev);
  });
  *out = &d;
  return d.err;
}

}  // namespace

extern "C" pq_status pq_filter_noalloc(pq_col col, int op, int64_t c, const int64_t* sel_in,
                                       int64_t n_in, int64_t* sel_out, int64_t* d_count,
                                       int32_t* d_error, void* stream) {
  bool ok;
  Pred p = pqh::make_pred(op, c, &ok);
  if (!ok || !pqh::valid_dtype(col.type) || col.n < 0 || !d_count || col.reserved != 0)
    return PQ_ERR_INVALID_ARG;
  const bool sel = sel_in != nullptr;
  const i64 n_cap = sel ? n_in : col.n;
  if (n_cap < 0 || (n_cap > 0 && (!sel_out || (!col.data && col.n > 0))))
    return PQ_ERR_INVALID_ARG;
  if (n_cap > kNoAllocRows) return PQ_ERR_CAPACITY;  // beyond the static scratch
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return PQ_ERR_CUDA;
  NoAllocDevice* d = nullptr;
  if (noalloc_setup(dev, &d) != cudaSuccess) return PQ_ERR_CUDA;
  cudaStream_t s = S(stream);
  if (cudaMemsetAsync(d_count, 0, sizeof(int64_t), s) != cudaSuccess) return PQ_ERR_CUDA;
  if (d_error && cudaMemsetAsync(d_error, 0, sizeof(int32_t), s) != cudaSuccess)
    return PQ_ERR_CUDA;
  if (n_cap == 0) return PQ_OK;
  const i64 ntiles = (n_cap + kFilterTile - 1) / kFilterTile;
  u64* hdr = d->scratch;
  if (cudaMemsetAsync(hdr, 0, (kNoAllocHeader + ntiles) * sizeof(u64), s) != cudaSuccess)
    return PQ_ERR_CUDA;
  u32* ticket = (u32*)hdr;
  DevStatus* status = (DevStatus*)(hdr + 2);
  u64* state = hdr + kNoAllocHeader;
  const bool vec = sel ? aligned16(sel_in) : aligned16(col.data);
  const int grid = (int)std::max<i64>(1, std::min<i64>(ntiles, (i64)d->sms * 4));
  const i64 spin = 1ll << 22;
  PQ_DISPATCH_T(col.type, T, {
    if (sel) {
      if (vec)
        k_filter<T, true, true><<<grid, 256, 0, s>>>((const T*)col.data, (const i64*)sel_in,
                                                     n_cap, nullptr, p, (i64*)sel_out,
                                                     (i64*)d_count, state, ticket, spin, status);
      else
        k_filter<T, true, false><<<grid, 256, 0, s>>>((const T*)col.data, (const i64*)sel_in,
                                                      n_cap, nullptr, p, (i64*)sel_out,
                                                      (i64*)d_count, state, ticket, spin, status);
    } else {
      if (vec)
        k_filter<T, false, true><<<grid, 256, 0, s>>>((const T*)col.data, nullptr, n_cap,
                                                      nullptr, p, (i64*)sel_out, (i64*)d_count,
                                                      state, ticket, spin, status);
      else
        k_filter<T, false, false><<<grid, 256, 0, s>>>((const T*)col.data, nullptr, n_cap,
                                                       nullptr, p, (i64*)sel_out, (i64*)d_count,
                                                       state, ticket, spin, status);
    }
  });
  if (cudaGetLastError() != cudaSuccess) return PQ_ERR_CUDA;
  if (d_error &&
      cudaMemcpyAsync(d_error, &status->code, sizeof(int32_t), cudaMemcpyDeviceToDevice, s) !=
          cudaSuccess)
    return PQ_ERR_CUDA;
  return PQ_OK;
}
