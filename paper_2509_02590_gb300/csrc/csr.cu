// csr.cu -- the CSR builder by buckets of rows.
//
// The CSR of Section 2.1's graph store (both directions, self-loops and
// repeated edges dropped, every row ascending), built as a partition of the
// directed entries into buckets of 2^s consecutive rows and a sort of every
// bucket on chip:
//   1. the entries are counted by the leading digit of their bucket (an
//      endpoint outside [0, n) is an error; a self-loop goes to a bucket of
//      its own past the last one);
//   2. they are partitioned by that digit: a CTA ranks a tile's entries by
//      shared-memory atomics, takes a range per digit from a global cursor,
//      and writes the tile in digit order, so that runs of a digit are written
//      together.  Nothing needs the entries' order, so no pass is stable and
//      no tile waits for another;
//   3. with more than BIN_MAX buckets the same two steps again by the second
//      digit, inside each range of the first.  The last partition writes
//      32-bit entries: the row within the bucket and the column;
//   4. every bucket is sorted by one CTA: its rows are counted and gathered in
//      shared memory (long rows as parts by their columns' top bits), rows and
//      parts of up to 512 entries sorted by a warp in registers (bitonic, 1 to
//      16 values a lane), longer ones by the CTA in shared memory, repeats
//      dropped, and the result written at the bucket's place;
//      buckets too large for shared memory are taken by a second kernel that
//      gathers rows in global memory and splits rows that are themselves too
//      long by the columns' leading bits; the entries of still larger ones (and
//      of those with too many equal columns) are sorted together, by the radix
//      sort;
//   5. a scan of the rows' degrees gives the offsets; without repeats or loops
//      the columns are in place already, else one more copy packs them.
// It moves each entry 5 times (read as an edge twice, written and read as 8
// and as 4 bytes, written as a column); the full sort it replaces moves 8
// bytes in and out six times on a 10M-vertex graph.
//
// Measured (builds with L2 flushed, before: rows by global atomics up to 2^24
// edges, one radix sort of 64-bit keys above): 172M edges on 10M vertices
// 23.5 -> 9.1 ms, 53M on 3M 7.4 -> 2.5 ms, 11.7M raw on 1M 1.69 -> 0.78 ms,
// 0.9M on 100,000 0.197 -> 0.136 ms, 21,000 on 2,000 0.110 -> 0.111 ms.  On the
// 3M-vertex graph the bucket sort takes 1.09 ms (107M entries, 3.2 cycles an
// entry and SM: shuffles and shared-memory atomics), the two partitions 0.85
// (2.6 GB moved, 3 TB/s: ranking bounds it), the counts 0.30.
#include <algorithm>

#include "internal.h"

namespace wccg {

namespace {

constexpr int PT = 512;              // threads of a partition CTA
constexpr int PK = 16;               // entries a thread
constexpr int TILE = PT * PK;        // entries a tile
constexpr int BIN_MAX = 1024;        // buckets told apart by one digit
// Entries a bucket is meant to hold: 2,560 builds 11.7M raw edges on 1M vertices in
// 0.79 ms instead of 0.92 (fewer of them outgrow a CTA's shared memory) but 53M on
// 3M vertices in 2.94 instead of 2.74 (twice as many); with 8,192 both take as long
// as with 5,120.
constexpr int BUCKET_AVG = 5120;
constexpr int BUCKET_CAP = 12288;    // entries a CTA sorts in shared memory
constexpr int SB = 256;              // threads of a bucket's CTA
constexpr int ROWS_MAX = 256;        // rows of a bucket (one a thread of its CTA)
constexpr int ROW_WARP = 512;        // rows up to this long: one warp, in registers
constexpr int ROW_PART = 256;        // longer rows are split into parts by their columns' top bits
// Entries a part is meant to hold.  A warp's sorting network costs what its size
// rounded up to a power of two does: at 96 a part mostly takes the one of 128, at 192
// that of 256.  96 / 192 / 384: 53M edges on 3M vertices 2.66 / 2.74 / 3.56 ms, 11.7M
// raw on 1M 0.88 / 0.92 / 1.02.
constexpr int PART_AVG = 96;
constexpr int PARTS_MAX = 256;       // parts of one row
constexpr int SUB_MAX = ROWS_MAX + 2 * BUCKET_CAP / PART_AVG;  // rows and parts of a bucket
constexpr int BB = 512;              // threads of a large bucket's CTA
constexpr int BIG_CAP = 16384;       // entries it sorts in shared memory at once
constexpr int BIG_CTAS = 304;
// Entries of a bucket that one CTA takes; the ones of larger buckets are sorted
// together.  One row of 20,000 / 50,000 / 99,000 neighbours in 500,000 edges: 0.38 /
// 0.56 / 0.81 ms by a CTA, 0.30 / 0.31 / 0.33 by the sort; but a thousand buckets of
// 20,000 keep all CTAs busy: 0.81 ms against 1.16.
constexpr uint32_t HUGE_CAP = 32768;
constexpr int SMALL_T = 1024;        // a graph one CTA builds alone: its threads,
constexpr int SMALL_ROWS = 4096;     // rows
constexpr int SMALL_ENTRIES = 12 * 1024;  // and directed entries
constexpr size_t SMALL_SMEM = 4 * (size_t)(2 * SMALL_ROWS + 1 + SMALL_ENTRIES);
// Above SMALL_ENTRIES the steps' launches cost less than one CTA's time: 5,300
// edges 0.087 ms by one CTA against 0.122, 21,000 edges 0.149 against 0.127.

// What a build reports back in one copy.
struct Result {
  unsigned err, big, huge;  // DERR_* bits, large buckets, those left to the radix sort
  uint32_t placed;          // entries in the buckets (the loops' excluded)
  int64_t nnz;
};

// Sizes of one build.
struct Plan {
  int64_t n;
  int b, s;            // column bits, row bits within a bucket
  unsigned nb;         // buckets; bucket nb takes the self-loops
  int low;             // bits of the second digit (0: one digit)
  unsigned nhigh;      // values of the first digit
};

// Ranks of a thread's entries among equal digits, by shared-memory atomics.
// A warp whose 32 entries share the digit (sorted input) takes one atomic.
template <int K>
__device__ __forceinline__ void tile_rank(const int (&dig)[K], uint32_t *cnt, uint32_t (&rank)[K]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    const int d0 = __shfl_sync(FULL, dig[k], 0);
    if (__all_sync(FULL, dig[k] == d0)) {
      uint32_t base = 0;
      if (lane == 0 && d0 >= 0) base = atomicAdd(&cnt[d0], 32u);
      rank[k] = __shfl_sync(FULL, base, 0) + lane;
    } else {
      rank[k] = dig[k] >= 0 ? atomicAdd(&cnt[dig[k]], 1u) : 0u;
    }
  }
}

// The entries of a tile: from the edge list (edge e of the tile gives entries
// (u, v) and (v, u); a self-loop two entries of the loop bucket) or from the
// first partition.  key = row << b | column; bucket -1: none.
template <bool EDGES>
__device__ __forceinline__ void load_tile(const Plan &p, const int32_t *__restrict__ src,
                                          const int32_t *__restrict__ dst, int64_t m,
                                          const uint64_t *__restrict__ in, int64_t at, int64_t end,
                                          uint64_t (&key)[PK], int (&bucket)[PK], unsigned *err) {
  if (EDGES) {
    int32_t u[PK / 2], v[PK / 2];
#pragma unroll
    for (int k = 0; k < PK / 2; ++k) {
      const int64_t e = at + (int64_t)k * PT + threadIdx.x;
      u[k] = e < m ? __ldcs(src + e) : -1;
      v[k] = e < m ? __ldcs(dst + e) : -1;
    }
#pragma unroll
    for (int k = 0; k < PK / 2; ++k) {
      const int64_t e = at + (int64_t)k * PT + threadIdx.x;
      bool ok = e < m;
      if (ok && (u[k] < 0 || u[k] >= p.n || v[k] < 0 || v[k] >= p.n)) {
        atomicOr(err, DERR_INVALID);
        ok = false;
      }
      const bool loop = ok && u[k] == v[k];
      key[2 * k] = ((uint64_t)(uint32_t)u[k] << p.b) | (uint32_t)v[k];
      key[2 * k + 1] = ((uint64_t)(uint32_t)v[k] << p.b) | (uint32_t)u[k];
      bucket[2 * k] = !ok ? -1 : loop ? (int)p.nb : (int)((uint32_t)u[k] >> p.s);
      bucket[2 * k + 1] = !ok ? -1 : loop ? (int)p.nb : (int)((uint32_t)v[k] >> p.s);
      if (loop) key[2 * k] = key[2 * k + 1] = (uint64_t)p.nb << (p.s + p.b);
    }
  } else {
#pragma unroll
    for (int k = 0; k < PK; ++k) {
      const int64_t i = at + (int64_t)k * PT + threadIdx.x;
      key[k] = i < end ? __ldcs(in + i) : 0ull;
      bucket[k] = i < end ? (int)(key[k] >> (p.s + p.b)) : -1;
    }
  }
}

// Tile blockIdx.x of the second level: the first digit its entries share and
// its range of the first partition's output.  False past the last tile.
struct Level2 {
  const uint32_t *start1;   // [nhigh + 1] ranges of the first digit
  const uint32_t *tile0;    // [nhigh + 1] first tile of each
  const uint16_t *owner;    // tile -> first digit
};
__device__ __forceinline__ bool tile_range(const Plan &p, const Level2 &l, int &h, int64_t &at,
                                           int64_t &end) {
  if (blockIdx.x >= l.tile0[p.nhigh]) return false;
  h = l.owner[blockIdx.x];
  at = (int64_t)l.start1[h] + (int64_t)(blockIdx.x - l.tile0[h]) * TILE;
  end = l.start1[h + 1];
  return true;
}

// hist[digit] += entries (first digit: hist[h]; second: hist[h << low | l],
// which is the bucket).
template <bool EDGES>
__global__ void __launch_bounds__(PT) k_count(Plan p, const int32_t *__restrict__ src,
                                             const int32_t *__restrict__ dst, int64_t m,
                                             const uint64_t *__restrict__ in, Level2 l2,
                                             uint32_t *hist, unsigned *err) {
  __shared__ uint32_t cnt[BIN_MAX];
  const int bins = EDGES ? (int)p.nhigh : 1 << p.low;
  for (int d = threadIdx.x; d < bins; d += PT) cnt[d] = 0;
  __syncthreads();
  int h = 0;
  int64_t at = (int64_t)blockIdx.x * (TILE / 2), end = 0;
  if (!EDGES && !tile_range(p, l2, h, at, end)) return;
  const int lane = threadIdx.x & 31;
  for (;;) {
    uint64_t key[PK];
    int dig[PK];
    load_tile<EDGES>(p, src, dst, m, in, at, end, key, dig, err);
#pragma unroll
    for (int k = 0; k < PK; ++k) {
      if (dig[k] >= 0) dig[k] = EDGES ? dig[k] >> p.low : dig[k] & ((1 << p.low) - 1);
      const int d0 = __shfl_sync(FULL, dig[k], 0);
      if (__all_sync(FULL, dig[k] == d0)) {
        if (lane == 0 && d0 >= 0) atomicAdd(&cnt[d0], 32u);
      } else if (dig[k] >= 0) {
        atomicAdd(&cnt[dig[k]], 1u);
      }
    }
    if (!EDGES) break;
    at += (int64_t)gridDim.x * (TILE / 2);
    if (at >= m) break;
  }
  __syncthreads();
  uint32_t *to = EDGES ? hist : hist + ((size_t)h << p.low);
  for (int d = threadIdx.x; d < bins; d += PT)
    if (cnt[d]) atomicAdd(&to[d], cnt[d]);
}

// One block: exclusive scan of the first digit's counts (start, a copy as
// cursors), and, for a second level, the tiles of each range.
__global__ void __launch_bounds__(1024) k_starts1(Plan p, const uint32_t *__restrict__ hist,
                                                 uint32_t *start, uint32_t *cursor,
                                                 uint32_t *tile0, uint16_t *owner) {
  __shared__ uint32_t sm[1024 / 32 + 1];
  const int d = threadIdx.x;
  const uint32_t c = d < (int)p.nhigh ? hist[d] : 0u;
  uint32_t tot;
  const uint32_t ex = block_exclusive_scan<1024>(c, &tot, sm);
  if (d < (int)p.nhigh) {
    start[d] = ex;
    cursor[d] = ex;
  }
  if (d == 0) start[p.nhigh] = tot;
  if (p.low == 0) return;
  const uint32_t t = c / TILE + (c % TILE != 0u);  // (c + TILE - 1 can wrap)
  const uint32_t t0 = block_exclusive_scan<1024>(t, &tot, sm);
  if (d < (int)p.nhigh) {
    tile0[d] = t0;
    for (uint32_t q = 0; q < t; ++q) owner[t0 + q] = (uint16_t)d;
  }
  if (d == 0) tile0[p.nhigh] = tot;
}

// One partition; LAST writes the 32-bit entries of the buckets.
template <bool EDGES, bool LAST>
__global__ void __launch_bounds__(PT, 2) k_partition(Plan p, const int32_t *__restrict__ src,
                                                    const int32_t *__restrict__ dst, int64_t m,
                                                    const uint64_t *__restrict__ in, Level2 l2,
                                                    uint32_t *cursor, uint64_t *out64,
                                                    uint32_t *out32, unsigned *err) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint64_t *st64 = reinterpret_cast<uint64_t *>(smem);
  uint32_t *st32 = reinterpret_cast<uint32_t *>(smem);
  uint16_t *stdig = reinterpret_cast<uint16_t *>(smem + 4 * TILE);
  __shared__ uint32_t cnt[BIN_MAX], first[BIN_MAX], gpos[BIN_MAX];
  __shared__ uint32_t sm[PT / 32 + 1];
  const int bins = EDGES ? (int)p.nhigh : 1 << p.low;
  for (int d = threadIdx.x; d < bins; d += PT) cnt[d] = 0;
  __syncthreads();
  int h = 0;
  int64_t at = (int64_t)blockIdx.x * (TILE / 2), end = 0;
  if (!EDGES && !tile_range(p, l2, h, at, end)) return;
  uint64_t key[PK];
  int dig[PK];
  uint32_t rank[PK];
  load_tile<EDGES>(p, src, dst, m, in, at, end, key, dig, err);
#pragma unroll
  for (int k = 0; k < PK; ++k)
    if (dig[k] >= 0) dig[k] = EDGES ? dig[k] >> p.low : dig[k] & ((1 << p.low) - 1);
  tile_rank<PK>(dig, cnt, rank);
  __syncthreads();
  // thread t owns digits 2t and 2t + 1
  const int d0 = 2 * threadIdx.x;
  const uint32_t c0 = d0 < bins ? cnt[d0] : 0u, c1 = d0 + 1 < bins ? cnt[d0 + 1] : 0u;
  uint32_t total;
  const uint32_t ex = block_exclusive_scan<PT>(c0 + c1, &total, sm);
  uint32_t *cur = EDGES ? cursor : cursor + ((size_t)h << p.low);
  if (d0 < bins) {
    first[d0] = ex;
    gpos[d0] = (c0 ? atomicAdd(&cur[d0], c0) : 0u) - ex;
  }
  if (d0 + 1 < bins) {
    first[d0 + 1] = ex + c0;
    gpos[d0 + 1] = (c1 ? atomicAdd(&cur[d0 + 1], c1) : 0u) - (ex + c0);
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < PK; ++k) {
    if (dig[k] < 0) continue;
    const uint32_t pos = first[dig[k]] + rank[k];
    if (LAST) {
      st32[pos] = (uint32_t)(key[k] & ((1ull << (p.s + p.b)) - 1));
      stdig[pos] = (uint16_t)dig[k];
    } else {
      st64[pos] = key[k];
    }
  }
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < total; i += PT) {
    if (LAST) {
      out32[gpos[stdig[i]] + i] = st32[i];
    } else {
      const uint64_t k = st64[i];
      out64[gpos[(uint32_t)(k >> (p.s + p.b)) >> p.low] + i] = k;
    }
  }
}

// ---- sorting rows ------------------------------------------------------------

// Bitonic sort of 32 * R values held R to a lane: value i = r * 32 + lane
// sits in x[r] of lane `lane`; ascending in i at the end.  Partners closer
// than 32 apart are exchanged across lanes, farther ones within a lane.
template <int R>
__device__ __forceinline__ void warp_bitonic(uint32_t (&x)[R], int lane) {
#pragma unroll
  for (int k = 2; k <= 32 * R; k <<= 1) {
#pragma unroll
    for (int j = k >> 1; j > 0; j >>= 1) {
      if (j >= 32) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int p = r ^ (j >> 5);
          if (p > r) {
            const bool up = ((r * 32 + lane) & k) == 0;
            const uint32_t lo = min(x[r], x[p]), hi = max(x[r], x[p]);
            x[r] = up ? lo : hi;
            x[p] = up ? hi : lo;
          }
        }
      } else {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const uint32_t y = __shfl_xor_sync(FULL, x[r], j);
          const bool up = ((r * 32 + lane) & k) == 0, lower = (lane & j) == 0;
          x[r] = (lower == up) ? min(x[r], y) : max(x[r], y);
        }
      }
    }
  }
}

// One row of len <= 32 * R values: sorted, first copies written to the
// front of the row in order; returns their number.
template <int R>
__device__ __forceinline__ int warp_sort_row(uint32_t *row, int len, int lane) {
  uint32_t x[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = r * 32 + lane;
    x[r] = i < len ? row[i] : 0xffffffffu;
  }
  warp_bitonic<R>(x, lane);
  int base = 0;
  const unsigned lt = lanemask_lt();
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const uint32_t up = __shfl_up_sync(FULL, x[r], 1);
    const uint32_t last = __shfl_sync(FULL, r > 0 ? x[r > 0 ? r - 1 : 0] : 0u, 31);
    const uint32_t prev = lane > 0 ? up : last;
    const int i = r * 32 + lane;
    const bool keep = i < len && (i == 0 || x[r] != prev);
    const unsigned mask = __ballot_sync(FULL, keep);
    if (keep) row[base + __popc(mask & lt)] = x[r];
    base += __popc(mask);
  }
  return base;
}

__device__ __forceinline__ int warp_sort_any(uint32_t *row, int len, int lane) {
  if (len <= 32) return warp_sort_row<1>(row, len, lane);
  if (len <= 64) return warp_sort_row<2>(row, len, lane);
  if (len <= 128) return warp_sort_row<4>(row, len, lane);
  if (len <= 256) return warp_sort_row<8>(row, len, lane);
  return warp_sort_row<16>(row, len, lane);
}

// a[0..len) ascending, by the whole block: the bitonic network whose
// exchanges all put the smaller value first (each merge starts with mirrored
// partners), so that missing values past len stay there.
template <int T>
__device__ __forceinline__ void block_sort(uint32_t *a, int len) {
  int P = 2;
  while (P < len) P <<= 1;
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      const bool first = 2 * j == k;
      for (int i = threadIdx.x; i < P / 2; i += T) {
        const int o = i & (j - 1), lo = 2 * (i - o) + o;
        const int hi = first ? lo ^ (k - 1) : lo + j;
        if (hi < len) {
          const uint32_t x = a[lo], y = a[hi];
          if (x > y) {
            a[lo] = y;
            a[hi] = x;
          }
        }
      }
      __syncthreads();
    }
}

// First copies of a[0..len) (sorted) to out, which may be a; returns their
// number.  Whole block.
template <int T>
__device__ __forceinline__ int block_unique(const uint32_t *a, int len, uint32_t *out, int32_t *scan) {
  int carry = 0;
  for (int base = 0; base < len; base += T) {
    const int i = base + threadIdx.x;
    const uint32_t x = i < len ? a[i] : 0u;
    const bool keep = i < len && (i == 0 || x != a[i - 1]);
    int tot;
    const int ex = block_exclusive_scan<T>(keep ? 1 : 0, &tot, scan);  // reads before writes
    if (keep) out[carry + ex] = x;
    carry += tot;
    __syncthreads();
  }
  return carry;
}

// Exclusive scan of v[0..ROWS_MAX) into out[0..ROWS_MAX], by the first
// ROWS_MAX threads' values; whole block of T >= ROWS_MAX threads.
template <int T>
__device__ __forceinline__ int scan_rows(const uint32_t *v, uint32_t *out, int32_t *scan) {
  int tot;
  const int ex = block_exclusive_scan<T>(threadIdx.x < ROWS_MAX ? (int)v[threadIdx.x] : 0, &tot, scan);
  if (threadIdx.x < ROWS_MAX) out[threadIdx.x] = (uint32_t)ex;
  if (threadIdx.x == 0) out[ROWS_MAX] = (uint32_t)tot;
  __syncthreads();
  return tot;
}

// Bits of the part number of a row of len entries.
__device__ __forceinline__ int part_bits(int len) {
  int k = 0;
  while (k < 8 && (PART_AVG << k) < len) ++k;
  return k;
}

// The buckets, one CTA each: rows gathered in shared memory, sorted, and the
// columns written at the bucket's place in out; deg[row] = its columns.
// Rows above ROW_PART entries are gathered as parts by their columns' top bits
// (parts follow each other in column order, so a row is its parts one after
// the other), which keeps them at one warp's register sort; what is still
// above ROW_WARP is sorted by the CTA.  Buckets above BUCKET_CAP are listed.
__global__ void __launch_bounds__(SB) k_bucket_sort(Plan p, const uint32_t *__restrict__ in,
                                                   const uint32_t *__restrict__ start,
                                                   uint32_t *out, int64_t *deg, uint32_t *big,
                                                   uint32_t *huge, Result *res) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t *buf = reinterpret_cast<uint32_t *>(smem);
  __shared__ uint32_t cnt[SUB_MAX], rs[SUB_MAX + 1], us[SUB_MAX + 1];
  __shared__ uint16_t sub0[ROWS_MAX + 1], longs[SUB_MAX];
  __shared__ uint8_t shift[ROWS_MAX];
  __shared__ int32_t scan[SB / 32 + 1];
  __shared__ int nlong;
  const uint32_t q = blockIdx.x, base = start[q];
  const uint32_t entries = start[q + 1] - base;  // up to 2^32 - 2, with many copies of an edge
  const int64_t row0 = (int64_t)q << p.s;
  const int rows = (int)min((int64_t)1 << p.s, p.n - row0);
  if (threadIdx.x == 0 && q == p.nb - 1) res->placed = start[p.nb];
  if (entries > (uint32_t)BUCKET_CAP) {
    if (threadIdx.x == 0) {
      if (entries > HUGE_CAP)
        huge[atomicAdd(&res->huge, 1u)] = q;
      else
        big[atomicAdd(&res->big, 1u)] = q;
    }
    return;
  }
  const int size = (int)entries;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int r = threadIdx.x; r < SUB_MAX; r += SB) cnt[r] = 0;
  if (threadIdx.x == 0) nlong = 0;
  __syncthreads();
  const uint32_t cmask = (1u << p.b) - 1u;
  auto row_of = [&](uint32_t e) { return p.s ? e >> p.b : 0u; };
  for (int i = threadIdx.x; i < size; i += SB) atomicAdd(&cnt[row_of(in[base + i])], 1u);
  __syncthreads();
  // the rows' parts
  const int len0 = threadIdx.x < rows ? (int)cnt[threadIdx.x] : 0;
  const int bits = threadIdx.x < rows && len0 > ROW_PART ? min(part_bits(len0), p.b) : 0;
  int subs;
  const int s0 = block_exclusive_scan<SB>(threadIdx.x < rows ? 1 << bits : 0, &subs, scan);
  sub0[threadIdx.x] = (uint16_t)s0;
  shift[threadIdx.x] = (uint8_t)(p.b - bits);
  if (threadIdx.x == 0) sub0[ROWS_MAX] = (uint16_t)subs;
  __syncthreads();
  auto sub_of = [&](uint32_t e) {
    const uint32_t r = row_of(e);
    return (uint32_t)sub0[r] + ((e & cmask) >> shift[r]);
  };
  if (subs > rows) {  // some row has parts: count again by part
    for (int r = threadIdx.x; r < subs; r += SB) cnt[r] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < size; i += SB) atomicAdd(&cnt[sub_of(in[base + i])], 1u);
    __syncthreads();
  }
  auto scan_subs = [&](uint32_t *to) {
    int carry = 0;
    for (int r0 = 0; r0 < subs; r0 += SB) {
      const int r = r0 + threadIdx.x;
      int tot;
      const int ex = block_exclusive_scan<SB>(r < subs ? (int)cnt[r] : 0, &tot, scan);
      if (r < subs) to[r] = (uint32_t)(carry + ex);
      carry += tot;
    }
    if (threadIdx.x == 0) to[subs] = (uint32_t)carry;
    __syncthreads();
    return carry;
  };
  scan_subs(rs);
  for (int r = threadIdx.x; r < subs; r += SB) cnt[r] = rs[r];  // cursors
  __syncthreads();
  for (int i = threadIdx.x; i < size; i += SB) {
    const uint32_t e = in[base + i];
    buf[atomicAdd(&cnt[sub_of(e)], 1u)] = e & cmask;
  }
  __syncthreads();
  // rows and parts by the warps; cnt = unique entries
  for (int r = warp; r < subs; r += SB / 32) {
    const int len = (int)(rs[r + 1] - rs[r]);
    if (len > ROW_WARP) {
      if (lane == 0) longs[atomicAdd(&nlong, 1)] = (uint16_t)r;
      continue;
    }
    const int d = warp_sort_any(buf + rs[r], len, lane);
    if (lane == 0) cnt[r] = (uint32_t)d;
  }
  __syncthreads();
  for (int k = 0; k < nlong; ++k) {
    const int r = longs[k], len = (int)(rs[r + 1] - rs[r]);
    block_sort<SB>(buf + rs[r], len);
    const int d = block_unique<SB>(buf + rs[r], len, buf + rs[r], scan);
    if (threadIdx.x == 0) cnt[r] = (uint32_t)d;
  }
  __syncthreads();
  const int total = scan_subs(us);
  if (total == size) {
    for (int i = threadIdx.x; i < size; i += SB) out[base + i] = buf[i];
  } else {
    for (int r = warp; r < subs; r += SB / 32) {
      const int d = (int)cnt[r];
      for (int i = lane; i < d; i += 32) out[base + us[r] + i] = buf[rs[r] + i];
    }
  }
  if (threadIdx.x < rows) {
    const int s1 = threadIdx.x + 1 < rows ? sub0[threadIdx.x + 1] : subs;
    deg[row0 + threadIdx.x] = (int64_t)(us[s1] - us[s0]);
  }
}

// The values from[0..len), all in [lo, lo + span), sorted with repeats
// dropped into out (which may be from), through len words of shared memory:
// split into parts by their top bits, parts sorted by warps (by the block
// above ROW_WARP).  Returns the number written.  Whole block of T threads.
struct PartSpace {
  uint32_t cnt[PARTS_MAX], at[PARTS_MAX + 1], to[PARTS_MAX + 1];
  int32_t scan[32 + 1];
  uint16_t longs[PARTS_MAX];
  int nlong;
};
template <int T>
__device__ __forceinline__ int sort_by_parts(const uint32_t *from, int len, uint32_t lo,
                                             uint32_t span, uint32_t *buf, uint32_t *out,
                                             PartSpace &ps) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sb = 32 - __clz(max(span, 2u) - 1u);  // bits of a value within the span
  const int shift = max(0, sb - part_bits(len)), parts = 1 << (sb - shift);
  auto scan_parts = [&](uint32_t *to) {
    int tot;
    const int ex = block_exclusive_scan<T>(threadIdx.x < parts ? (int)ps.cnt[threadIdx.x] : 0, &tot,
                                           ps.scan);
    if (threadIdx.x < parts) to[threadIdx.x] = (uint32_t)ex;
    if (threadIdx.x == 0) to[parts] = (uint32_t)tot;
    __syncthreads();
    return tot;
  };
  if (threadIdx.x < PARTS_MAX) ps.cnt[threadIdx.x] = 0;
  if (threadIdx.x == 0) ps.nlong = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < len; i += T) atomicAdd(&ps.cnt[(from[i] - lo) >> shift], 1u);
  __syncthreads();
  scan_parts(ps.at);
  if (threadIdx.x < parts) ps.cnt[threadIdx.x] = ps.at[threadIdx.x];
  __syncthreads();
  for (int i = threadIdx.x; i < len; i += T) {
    const uint32_t v = from[i];
    buf[atomicAdd(&ps.cnt[(v - lo) >> shift], 1u)] = v;
  }
  __syncthreads();
  for (int r = warp; r < parts; r += T / 32) {
    const int l = (int)(ps.at[r + 1] - ps.at[r]);
    if (l > ROW_WARP) {
      if (lane == 0) ps.longs[atomicAdd(&ps.nlong, 1)] = (uint16_t)r;
      continue;
    }
    const int d = warp_sort_any(buf + ps.at[r], l, lane);
    if (lane == 0) ps.cnt[r] = (uint32_t)d;
  }
  __syncthreads();
  for (int k = 0; k < ps.nlong; ++k) {
    const int r = ps.longs[k], l = (int)(ps.at[r + 1] - ps.at[r]);
    block_sort<T>(buf + ps.at[r], l);
    const int d = block_unique<T>(buf + ps.at[r], l, buf + ps.at[r], ps.scan);
    if (threadIdx.x == 0) ps.cnt[r] = (uint32_t)d;
  }
  __syncthreads();
  const int total = scan_parts(ps.to);
  for (int r = warp; r < parts; r += T / 32) {
    const int d = (int)ps.cnt[r];
    for (int i = lane; i < d; i += 32) out[ps.to[r] + i] = buf[ps.at[r] + i];
  }
  __syncthreads();
  return total;
}

// The listed buckets, by whole CTAs in global memory: rows gathered into alt,
// then sorted there: short ones by warps, rows of up to BIG_CAP entries in
// shared memory, longer ones split by the columns' top bits into at most 256
// parts through out and sorted part by part.  A bucket with a part above
// BIG_CAP is left to the radix sort.
__global__ void __launch_bounds__(BB) k_bucket_big(Plan p, const uint32_t *in,
                                                  const uint32_t *__restrict__ start, uint32_t *alt,
                                                  uint32_t *out, int64_t *deg,
                                                  const uint32_t *__restrict__ big,
                                                  uint32_t *huge, Result *res) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t *buf = reinterpret_cast<uint32_t *>(smem);
  __shared__ uint32_t cnt[ROWS_MAX], rs[ROWS_MAX + 1], us[ROWS_MAX + 1];
  __shared__ uint32_t pc[256], ps[257];
  __shared__ int32_t scan[BB / 32 + 1];
  __shared__ PartSpace sp;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t cmask = (1u << p.b) - 1u;  // b <= 31
  const uint32_t vshift = p.b > 8 ? p.b - 8 : 0;
  const unsigned total_big = res->big;
  for (unsigned k = blockIdx.x; k < total_big; k += gridDim.x) {
    const uint32_t q = big[k], base = start[q], size = start[q + 1] - base;
    const int64_t row0 = (int64_t)q << p.s;
    const int rows = (int)min((int64_t)1 << p.s, p.n - row0);
    uint32_t *ab = alt + base, *ob = out + base;
    const uint32_t *ib = in + base;
    auto gather = [&](const uint32_t *from, uint32_t len, uint32_t *c, uint32_t *st, uint32_t *to,
                      uint32_t shift, uint32_t keep) {
      // from[0..len) grouped by value >> shift (at most 256 groups, group g at
      // st[g]) into to, masked by keep
      if (threadIdx.x < 256) c[threadIdx.x] = 0;
      __syncthreads();
      for (uint32_t i0 = 0; i0 < len; i0 += BB) {
        const uint32_t i = i0 + threadIdx.x;
        const int g = i < len ? (shift >= 32 ? 0 : (int)(from[i] >> shift)) : -1;
        const unsigned peers = __match_any_sync(FULL, g);
        if (g >= 0 && (peers & lanemask_lt()) == 0u) atomicAdd(&c[g], (uint32_t)__popc(peers));
      }
      __syncthreads();
      scan_rows<BB>(c, st, scan);
      if (threadIdx.x < 256) c[threadIdx.x] = st[threadIdx.x];
      __syncthreads();
      for (uint32_t i0 = 0; i0 < len; i0 += BB) {
        const uint32_t i = i0 + threadIdx.x;
        const uint32_t e = i < len ? from[i] : 0u;
        const int g = i < len ? (shift >= 32 ? 0 : (int)(e >> shift)) : -1;
        const unsigned peers = __match_any_sync(FULL, g);
        const int leader = __ffs(peers) - 1;
        uint32_t at = 0;
        if (g >= 0 && lane == leader) at = atomicAdd(&c[g], (uint32_t)__popc(peers));
        at = __shfl_sync(FULL, at, leader);
        if (g >= 0) to[at + __popc(peers & lanemask_lt())] = e & keep;
      }
      __syncthreads();
    };
    gather(ib, size, cnt, rs, ab, p.s ? (uint32_t)p.b : 32u, cmask);
    // short rows by warps; cnt = unique entries
    for (int r = warp; r < rows; r += BB / 32) {
      const int len = (int)(rs[r + 1] - rs[r]);
      if (len > ROW_WARP) continue;
      const int d = warp_sort_any(ab + rs[r], len, lane);
      if (lane == 0) cnt[r] = (uint32_t)d;
    }
    __syncthreads();
    bool over = false;
    for (int r = 0; r < rows && !over; ++r) {
      const uint32_t len = rs[r + 1] - rs[r];
      if (len <= (uint32_t)ROW_WARP) continue;
      uint32_t *row = ab + rs[r];
      uint32_t d = 0;
      if (len <= (uint32_t)BIG_CAP) {
        d = (uint32_t)sort_by_parts<BB>(row, (int)len, 0u, cmask + 1u, buf, row, sp);
      } else {
        // parts by the columns' top bits, through out and back
        gather(row, len, pc, ps, ob + rs[r], vshift, 0xffffffffu);
        // neighbouring parts are sorted together while they fit
        for (int g0 = 0; g0 < 256;) {
          int g1 = g0 + 1;
          while (g1 < 256 && ps[g1 + 1] - ps[g0] <= (uint32_t)BIG_CAP) ++g1;
          const uint32_t a = ps[g0], l = ps[g1] - a;
          over = l > (uint32_t)BIG_CAP;
          if (over) break;
          d += (uint32_t)sort_by_parts<BB>(ob + rs[r] + a, (int)l, (uint32_t)g0 << vshift,
                                           (uint32_t)(g1 - g0) << vshift, buf, row + d, sp);
          g0 = g1;
        }
      }
      if (threadIdx.x == 0) cnt[r] = d;
      __syncthreads();
    }
    if (over) {
      if (threadIdx.x == 0) huge[atomicAdd(&res->huge, 1u)] = q;
      continue;
    }
    if (threadIdx.x < ROWS_MAX && threadIdx.x >= rows) cnt[threadIdx.x] = 0;
    __syncthreads();
    scan_rows<BB>(cnt, us, scan);
    for (int r = 0; r < rows; ++r) {
      const uint32_t d = cnt[r];
      for (uint32_t i = threadIdx.x; i < d; i += BB) ob[us[r] + i] = ab[rs[r] + i];
    }
    if (threadIdx.x < rows) deg[row0 + threadIdx.x] = (int64_t)cnt[threadIdx.x];
    __syncthreads();
  }
}

// A small graph by one CTA: rows counted, gathered, sorted and packed in
// shared memory (columns, then the rows' ends and places).  The steps above
// take eight launches, which is most of their time here.
__global__ void __launch_bounds__(SMALL_T) k_csr_small(const int32_t *__restrict__ src,
                                                       const int32_t *__restrict__ dst, int m, int n,
                                                       int64_t *off, int32_t *adj, Result *res) {
  extern __shared__ __align__(16) unsigned char smem[];
  uint32_t *cnt = reinterpret_cast<uint32_t *>(smem), *rs = cnt + SMALL_ROWS, *buf = rs + SMALL_ROWS + 1;
  __shared__ int32_t scan[SMALL_T / 32 + 1];
  __shared__ int nlong;
  __shared__ unsigned bad;
  __shared__ uint16_t longs[SMALL_ENTRIES / ROW_WARP];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int r = threadIdx.x; r < n; r += SMALL_T) cnt[r] = 0;
  if (threadIdx.x == 0) {
    nlong = 0;
    bad = 0u;
  }
  __syncthreads();
  // four edges a thread in flight
  auto edges = [&](auto f) {
    for (int e0 = threadIdx.x; e0 < m; e0 += 4 * SMALL_T) {
      int32_t u[4], v[4];
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        const int e = e0 + z * SMALL_T;
        u[z] = e < m ? src[e] : 0;
        v[z] = e < m ? dst[e] : 0;
      }
#pragma unroll
      for (int z = 0; z < 4; ++z)
        if (e0 + z * SMALL_T < m) f(u[z], v[z]);
    }
  };
  edges([&](int32_t u, int32_t v) {
    if (u < 0 || u >= n || v < 0 || v >= n) {
      bad = 1u;
    } else if (u != v) {
      atomicAdd(&cnt[u], 1u);
      atomicAdd(&cnt[v], 1u);
    }
  });
  __syncthreads();
  if (bad) {
    if (threadIdx.x == 0) res->err = DERR_INVALID;
    return;
  }
  auto scan_all = [&](uint32_t *out) {  // out[r] = cnt[0] + .. + cnt[r - 1]; the total
    int carry = 0;
    for (int r0 = 0; r0 < n; r0 += SMALL_T) {
      const int r = r0 + threadIdx.x;
      int tot;
      const int ex = block_exclusive_scan<SMALL_T>(r < n ? (int)cnt[r] : 0, &tot, scan);
      if (r < n) out[r] = (uint32_t)(carry + ex);
      carry += tot;
    }
    return carry;
  };
  const int size = scan_all(rs);
  if (threadIdx.x == 0) rs[n] = (uint32_t)size;
  for (int r = threadIdx.x; r < n; r += SMALL_T) cnt[r] = rs[r];
  __syncthreads();
  edges([&](int32_t u, int32_t v) {
    if (u == v) return;
    buf[atomicAdd(&cnt[u], 1u)] = (uint32_t)v;
    buf[atomicAdd(&cnt[v], 1u)] = (uint32_t)u;
  });
  __syncthreads();
  for (int r = warp; r < n; r += SMALL_T / 32) {
    const int len = (int)(rs[r + 1] - rs[r]);
    if (len > ROW_WARP) {
      if (lane == 0) longs[atomicAdd(&nlong, 1)] = (uint16_t)r;
      continue;
    }
    const int d = warp_sort_any(buf + rs[r], len, lane);
    if (lane == 0) cnt[r] = (uint32_t)d;
  }
  __syncthreads();
  for (int k = 0; k < nlong; ++k) {
    const int r = longs[k], len = (int)(rs[r + 1] - rs[r]);
    block_sort<SMALL_T>(buf + rs[r], len);
    const int d = block_unique<SMALL_T>(buf + rs[r], len, buf + rs[r], scan);
    if (threadIdx.x == 0) cnt[r] = (uint32_t)d;
  }
  __syncthreads();
  // the rows' final places
  int carry = 0;
  for (int r0 = 0; r0 < n; r0 += SMALL_T) {
    const int r = r0 + threadIdx.x;
    int tot;
    const int ex = block_exclusive_scan<SMALL_T>(r < n ? (int)cnt[r] : 0, &tot, scan);
    if (r < n) off[r] = (int64_t)(carry + ex);
    carry += tot;
  }
  if (threadIdx.x == 0) {
    off[n] = carry;
    res->err = 0u;
    res->nnz = carry;
  }
  __syncthreads();
  for (int r = warp; r < n; r += SMALL_T / 32) {
    const int64_t to = off[r];
    const int d = (int)cnt[r];
    for (int i = lane; i < d; i += 32) adj[to + i] = (int32_t)buf[rs[r] + i];
  }
}

// ---- the buckets left to the radix sort ------------------------------------------
// Bucket k of the list huge[0..count): its entries are hstart[k] .. hstart[k + 1]
// of all the listed ones'.  One block.
__global__ void __launch_bounds__(1024) k_huge_starts(const uint32_t *__restrict__ start,
                                                     const uint32_t *__restrict__ huge,
                                                     uint32_t count, uint32_t *hstart) {
  __shared__ uint32_t sm[1024 / 32 + 1];
  uint32_t carry = 0;
  for (uint32_t k0 = 0; k0 < count; k0 += 1024) {
    const uint32_t k = k0 + threadIdx.x;
    uint32_t tot;
    const uint32_t ex = block_exclusive_scan<1024>(
        k < count ? start[huge[k] + 1] - start[huge[k]] : 0u, &tot, sm);
    if (k < count) hstart[k] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0) hstart[count] = carry;
}

// keys[i] = (k, entry) of the listed buckets' entry i, in bucket k.
__global__ void k_huge_keys(Plan p, const uint32_t *__restrict__ in,
                            const uint32_t *__restrict__ start, const uint32_t *__restrict__ huge,
                            uint32_t count, const uint32_t *__restrict__ hstart, int64_t total,
                            uint64_t *keys) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= total) return;
  uint32_t lo = 0, hi = count - 1;  // the last k with hstart[k] <= i
  while (lo < hi) {
    const uint32_t mid = (lo + hi + 1) >> 1;
    if (hstart[mid] <= (uint32_t)i) lo = mid; else hi = mid - 1;
  }
  keys[i] = ((uint64_t)lo << (p.b + p.s)) | in[start[huge[lo]] + ((uint32_t)i - hstart[lo])];
}

__global__ void k_huge_first(const uint64_t *__restrict__ keys, int64_t total, uint32_t *keep) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < total) keep[i] = i == 0 || keys[i - 1] != keys[i] ? 1u : 0u;
}

// deg[r] = the columns of row r by the offsets; 0 in the listed buckets (block
// = rows of one bucket).
__global__ void k_huge_degrees(const int64_t *__restrict__ off, int64_t n, int64_t *deg) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n) deg[r] = off[r + 1] - off[r];
}
__global__ void __launch_bounds__(ROWS_MAX) k_huge_clear(Plan p, const uint32_t *__restrict__ huge,
                                                        int64_t *deg) {
  const int64_t r = ((int64_t)huge[blockIdx.x] << p.s) + threadIdx.x;
  if (threadIdx.x < (1 << p.s) && r < p.n) deg[r] = 0;
}

// The first copies in order to their bucket's place in out, and their rows'
// degrees (sorted keys: one atomic per row and warp).
__global__ void k_huge_write(Plan p, const uint64_t *__restrict__ keys,
                             const uint32_t *__restrict__ keep, const uint32_t *__restrict__ pos,
                             int64_t total, const uint32_t *__restrict__ start,
                             const uint32_t *__restrict__ huge, const uint32_t *__restrict__ hstart,
                             uint32_t *out, int64_t *deg) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool kept = i < total && keep[i];
  int64_t row = -1;
  if (kept) {
    const uint32_t k = (uint32_t)(keys[i] >> (p.b + p.s)), q = huge[k];
    const uint64_t e = keys[i] & ((1ull << (p.b + p.s)) - 1);
    row = ((int64_t)q << p.s) + (int64_t)(e >> p.b);
    out[start[q] + (pos[i] - pos[hstart[k]])] = (uint32_t)(e & ((1ull << p.b) - 1));
  }
  const unsigned peers = __match_any_sync(FULL, (unsigned long long)row);
  if (kept && (peers & lanemask_lt()) == 0u)
    atomicAdd((unsigned long long *)&deg[row], (unsigned long long)__popc(peers));
}

// With repeats or loops dropped: every bucket's columns to their final place.
// Those above HUGE_CAP (list: huge) by PACK_CTAS CTAs each, the others by one.
constexpr unsigned PACK_CTAS = 64;
__global__ void __launch_bounds__(SB) k_bucket_pack(Plan p, const uint32_t *__restrict__ in,
                                                   const uint32_t *__restrict__ start,
                                                   const uint32_t *__restrict__ huge,
                                                   const int64_t *__restrict__ off, int32_t *adj) {
  const uint32_t q = huge ? huge[blockIdx.x] : blockIdx.x;
  const uint32_t from = start[q];
  if ((start[q + 1] - from > HUGE_CAP) != (huge != nullptr)) return;
  const int64_t r0 = (int64_t)q << p.s, r1 = min(r0 + ((int64_t)1 << p.s), p.n);
  const int64_t to = off[r0], len = off[r1] - to;
  for (int64_t i = (int64_t)blockIdx.y * SB + threadIdx.x; i < len; i += gridDim.y * SB)
    adj[to + i] = (int32_t)in[from + i];
}

// Sorts the entries of the huge listed buckets all at once, writes their
// columns and makes the offsets anew.  keys: 64-bit memory that may be
// overwritten (grown when it is too small); in: their entries, overwritten too.
// A row of 1,900,000 neighbours in 20M edges: 1.46 ms in all (one CTA taking the
// bucket 12.9, one CTA packing it 2.38; the full sort of all entries 3.5).
Result sort_huge(const Plan &p, uint32_t *in, const uint32_t *start, const uint32_t *huge,
                 uint32_t count, uint32_t *out, int64_t *off, DevBuf &keys, DevBuf &temp,
                 Result *res, cudaStream_t s) {
  DevBuf bstart, bkeys2, bpos, bdeg;
  uint32_t *hstart = static_cast<uint32_t *>(bstart.ensure(4 * ((size_t)count + 1)));
  k_huge_starts<<<1, 1024, 0, s>>>(start, huge, count, hstart); note_launch();
  WCC_CUDA(cudaGetLastError());
  const int64_t total = read_back(hstart + count, s);
  uint64_t *k1 = static_cast<uint64_t *>(keys.ensure(8 * (size_t)total));
  uint64_t *k2 = static_cast<uint64_t *>(bkeys2.ensure(8 * (size_t)total));
  uint32_t *pos = static_cast<uint32_t *>(bpos.ensure(4 * ((size_t)total + 1)));
  int64_t *deg = static_cast<int64_t *>(bdeg.ensure(8 * (size_t)(p.n + 1)));
  void *t = temp.ensure(std::max({radix_temp_bytes(total), scan_temp_bytes(total + 1),
                                  scan_temp_bytes(p.n + 1)}) + 64);
  const unsigned g = grid_for(total);
  k_huge_keys<<<g, SB, 0, s>>>(p, in, start, huge, count, hstart, total, k1); note_launch();
  WCC_CUDA(cudaGetLastError());
  const int bits = p.b + p.s + (int)bitlen_u64(count - 1);
  const uint64_t *sorted = radix_sort_keys_u64(k1, k2, total, bits, t, &res->err, s) ? k2 : k1;
  if (read_back(&res->err, s)) fail(WCC_ERR_TIMEOUT, "CSR build: a bounded wait of the sort ran out");
  uint32_t *keep = in;
  k_huge_first<<<g, SB, 0, s>>>(sorted, total, keep); note_launch();
  exclusive_scan_u32(keep, pos, total, pos + total, t, s);
  k_huge_degrees<<<grid_for(p.n), SB, 0, s>>>(off, p.n, deg); note_launch();
  k_huge_clear<<<count, ROWS_MAX, 0, s>>>(p, huge, deg); note_launch();
  k_huge_write<<<g, SB, 0, s>>>(p, sorted, keep, pos, total, start, huge, hstart, out, deg);
  note_launch();
  WCC_CUDA(cudaMemsetAsync(deg + p.n, 0, 8, s));
  exclusive_scan_i64(deg, off, p.n + 1, &res->nnz, t, s);
  WCC_CUDA(cudaGetLastError());
  return read_back(res, s);  // (the buffers above are given back only after it)
}

}  // namespace

bool csr_by_buckets(const int32_t *src, const int32_t *dst, int64_t m, int64_t n, int64_t *off,
                    DevBuf &adj_buf, int64_t *nnz_out, DevBuf (&w)[CSR_BUCKET_BUFS],
                    cudaStream_t s) {
  auto opt_in = [](const void *f, size_t bytes) {
    WCC_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
  };
  if (n <= SMALL_ROWS && 2 * m <= SMALL_ENTRIES) {
    Result *res = static_cast<Result *>(w[0].ensure(sizeof(Result)));
    int32_t *a = static_cast<int32_t *>(adj_buf.ensure(8 * (size_t)std::max<int64_t>(m, 1)));
    opt_in((const void *)k_csr_small, SMALL_SMEM);
    k_csr_small<<<1, SMALL_T, SMALL_SMEM, s>>>(src, dst, (int)m, (int)n, off, a, res); note_launch();
    WCC_CUDA(cudaGetLastError());
    const Result r = read_back(res, s);
    if (r.err & DERR_INVALID) fail(WCC_ERR_INVALID, "edge endpoint outside [0, n)");
    *nnz_out = r.nnz;
    return true;
  }
  Plan p{};
  p.n = n;
  p.b = (int)std::max<int64_t>(1, bitlen_u64(n > 0 ? (uint64_t)(n - 1) : 0));
  const int64_t n2 = 2 * m;
  // rows a bucket: BUCKET_AVG entries on average, row and column in 32 bits
  while (p.s < 8 && p.b + p.s + 1 <= 32 && (n2 << (p.s + 1)) <= (int64_t)BUCKET_AVG * std::max<int64_t>(n, 1))
    ++p.s;
  const int64_t nb = n > 0 ? ((n - 1) >> p.s) + 1 : 0;
  // too many buckets, or (copies of few edges) all of them huge
  if (nb + 1 > (int64_t)BIN_MAX * BIN_MAX || n2 > (int64_t)HUGE_CAP * nb) return false;
  p.nb = (unsigned)nb;
  if (nb + 1 > BIN_MAX) {
    const int bits = (int)bitlen_u64((uint64_t)nb);
    p.low = bits / 2;
  }
  p.nhigh = (unsigned)(nb >> p.low) + 1;
  const bool two = p.low > 0;
  const size_t nq = two ? (size_t)p.nhigh << p.low : p.nhigh;  // buckets that can be named
  const int64_t tiles1 = (m + TILE / 2 - 1) / (TILE / 2);
  const int64_t tiles2 = n2 / TILE + p.nhigh;
  if (tiles1 > 0x7fffffff || tiles2 > 0x7fffffff) return false;
  // counters and cursors (cleared together), starts, tiles, lists
  const size_t heads = sizeof(Result) + 4 * (nq + BIN_MAX);
  Result *res = static_cast<Result *>(w[0].ensure(heads));
  uint32_t *hist1 = reinterpret_cast<uint32_t *>(res + 1), *hist2 = hist1 + BIN_MAX;
  unsigned *err = &res->err;
  uint32_t *start2 = static_cast<uint32_t *>(w[1].ensure(4 * (nq + 1)));
  uint32_t *cur2 = static_cast<uint32_t *>(w[2].ensure(4 * (nq + 1)));
  uint32_t *start1 = static_cast<uint32_t *>(
      w[3].ensure(4 * (3 * (BIN_MAX + 1)) + 2 * (size_t)(two ? tiles2 : 1)));
  uint32_t *cur1 = start1 + BIN_MAX + 1, *tile0 = cur1 + BIN_MAX + 1;
  uint16_t *owner = reinterpret_cast<uint16_t *>(tile0 + BIN_MAX + 1);
  void *temp = w[4].ensure(std::max(scan_temp_bytes((int64_t)nq + 1), scan_temp_bytes(n + 1)) + 64);
  uint32_t *big = static_cast<uint32_t *>(w[5].ensure(8 * (size_t)std::max<int64_t>(nb, 1)));
  uint32_t *huge = big + nb;
  // the 64-bit entries of the first partition; later the large buckets' rows
  uint64_t *k64 = static_cast<uint64_t *>(w[6].ensure((two ? 8 : 4) * (size_t)n2));
  uint32_t *k32 = static_cast<uint32_t *>(w[7].ensure(4 * (size_t)n2));
  uint32_t *adj = static_cast<uint32_t *>(adj_buf.ensure(4 * (size_t)std::max<int64_t>(n2, 1)));
  const size_t sm64 = 8 * (size_t)TILE, sm32 = 6 * (size_t)TILE, smb = 4 * (size_t)BUCKET_CAP,
               smg = 4 * (size_t)BIG_CAP;
  opt_in((const void *)k_bucket_sort, smb);
  opt_in((const void *)k_bucket_big, smg);
  WCC_CUDA(cudaMemsetAsync(res, 0, heads, s));
  const Level2 l2{start1, tile0, owner};
  const unsigned gc = (unsigned)std::min<int64_t>(tiles1, 152 * 4);
  k_count<true><<<gc, PT, 0, s>>>(p, src, dst, m, nullptr, l2, hist1, err); note_launch();
  k_starts1<<<1, 1024, 0, s>>>(p, hist1, start1, cur1, tile0, owner); note_launch();
  const uint32_t *start = start1;
  if (two) {
    opt_in((const void *)k_partition<true, false>, sm64);
    opt_in((const void *)k_partition<false, true>, sm32);
    k_partition<true, false><<<(unsigned)tiles1, PT, sm64, s>>>(p, src, dst, m, nullptr, l2, cur1,
                                                              k64, nullptr, err);
    note_launch();
    k_count<false><<<(unsigned)tiles2, PT, 0, s>>>(p, nullptr, nullptr, 0, k64, l2, hist2, err);
    note_launch();
    exclusive_scan_u32(hist2, start2, (int64_t)nq, start2 + nq, temp, s);
    WCC_CUDA(cudaMemcpyAsync(cur2, start2, 4 * nq, cudaMemcpyDeviceToDevice, s));
    k_partition<false, true><<<(unsigned)tiles2, PT, sm32, s>>>(p, nullptr, nullptr, 0, k64, l2,
                                                              cur2, nullptr, k32, err);
    note_launch();
    start = start2;
  } else {
    opt_in((const void *)k_partition<true, true>, sm32);
    k_partition<true, true><<<(unsigned)tiles1, PT, sm32, s>>>(p, src, dst, m, nullptr, l2, cur1,
                                                             nullptr, k32, err);
    note_launch();
  }
  WCC_CUDA(cudaGetLastError());
  if (nb > 0) {
    k_bucket_sort<<<(unsigned)nb, SB, smb, s>>>(p, k32, start, adj, off, big, huge, res);
    note_launch();
    k_bucket_big<<<(unsigned)std::min<int64_t>(nb, BIG_CTAS), BB, smg, s>>>(
        p, k32, start, reinterpret_cast<uint32_t *>(k64), adj, off, big, huge, res);
    note_launch();
  }
  WCC_CUDA(cudaMemsetAsync(off + n, 0, 8, s));
  exclusive_scan_i64(off, off, n + 1, &res->nnz, temp, s);
  WCC_CUDA(cudaGetLastError());
  Result r = read_back(res, s);
  if (r.err & DERR_INVALID) fail(WCC_ERR_INVALID, "edge endpoint outside [0, n)");
  if (r.huge > 0) r = sort_huge(p, k32, start, huge, r.huge, adj, off, w[6], w[4], res, s);
  const int64_t nnz = r.nnz;
  if (nnz != (int64_t)r.placed) {
    // repeats were dropped: the buckets' columns close up, into k32's memory
    int32_t *to = reinterpret_cast<int32_t *>(k32);
    k_bucket_pack<<<(unsigned)nb, SB, 0, s>>>(p, adj, start, nullptr, off, to); note_launch();
    if (r.huge > 0) {
      k_bucket_pack<<<dim3(r.huge, PACK_CTAS), SB, 0, s>>>(p, adj, start, huge, off, to);
      note_launch();
    }
    WCC_CUDA(cudaGetLastError());
    std::swap(adj_buf.p, w[7].p);
    std::swap(adj_buf.bytes, w[7].bytes);
    std::swap(adj_buf.dev, w[7].dev);
    WCC_CUDA(cudaStreamSynchronize(s));
  }
  *nnz_out = nnz;
  return true;
}

}  // namespace wccg
