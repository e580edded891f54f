// pipeline.cu -- the stages around the refinement kernel, shared by wcc_run
// and the serving loop: grouping the vertices of a request by input label
// (a2), publishing its input clusters as work items (a8 seeding), and
// numbering the accepted clusters (a9).
#include "internal.h"

namespace wccg {

namespace {

constexpr int TB = 256;

// Workspace slots.
enum {
  B_KEYS, B_VALS, B_KEYS2, B_VALS2, B_TEMP, B_CL, B_CSTART, B_DSUM, B_KEEP, B_QIDX, B_OK1, B_OV1,
  B_OK2, B_OV2, B_INFO, B_FLAG, B_RANK, B_BASE, B_COUNT
};
static_assert(B_COUNT <= 24, "workspace slots");

struct SeedInfo {
  unsigned long long max_n;     // largest kept cluster
  unsigned long long max_dsum;  // largest degree sum of a kept cluster
  long long clusters;           // K: distinct labels
  long long skip;               // unclustered vertices (they sort first)
  unsigned err;                 // DERR_* bits
  unsigned maxkey;              // largest label + 1
  unsigned kept;                // clusters with >= min_size members
  unsigned ticket;              // tiles handed out (k_clusters)
};

// Graphs of at most GROUP_SMALL vertices are grouped, seeded and numbered by
// one CTA each (see k_group_small), whose sorting network grows with the vertices
// while the launches it saves do not.  Whole runs, one CTA / the general path, two
// kinds of graph: 1,000 vertices 0.132, 0.144 / 0.174, 0.188 ms; 2,000 0.147, 0.208 /
// 0.182, 0.212; 3,000 0.167, 0.307 / 0.184, 0.269; 4,096 0.187, 0.347 / 0.191, 0.284;
// 8,192 0.246, 0.488 / 0.212, 0.362.
constexpr int GROUP_SMALL = 2048;
constexpr int GT = 1024;  // its threads
static_assert(8 * GROUP_SMALL <= 32 * 1024, "its keys fit the shared memory of any launch");

// keys[v] = label + 1 (0 for unclustered), vals[v] = v; largest key; labels
// below -1 are malformed.
__global__ void k_make_keys(const int32_t *__restrict__ lab, int64_t n, uint32_t *keys,
                            uint32_t *vals, unsigned *maxkey, unsigned *err) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned k = 0;
  if (i < n) {
    int32_t c = lab[i];
    if (c < -1) atomicOr(err, DERR_INVALID);
    k = c < 0 ? 0u : (unsigned)c + 1u;
    keys[i] = k;
    vals[i] = (uint32_t)i;
  }
  k = warp_max(k);
  if ((threadIdx.x & 31) == 0 && k) atomicMax(maxkey, k);
}

// ---- single-pass running counts over tiles -----------------------------------
// A tile's status word: 2 bits of state (its own count, or the count up to its
// end), 62 of value.  Warp 0 of the tile's block calls; returns the count of all
// earlier tiles, 32 of them at a look.  Tiles are handed out in order, so every
// wait ends; one that outlasts a second sets DERR_TIMEOUT.
// (One thread walking back tile by tile takes as long as the tiles in flight are
// many: numbering 1M vertices 0.094 ms a call instead of 0.080, 100M 1.65 instead of
// 1.36; grouping 10M 1.09 instead of 1.03.)
constexpr unsigned long long TS_OWN = 1ull << 62, TS_ALL = 2ull << 62, TS_VAL = (1ull << 62) - 1;
__device__ __forceinline__ unsigned long long tiles_before(unsigned long long *status, int64_t tile,
                                                           unsigned long long own, unsigned *err) {
  const int lane = threadIdx.x & 31;
  unsigned long long before = 0;
  if (tile > 0) {
    if (lane == 0) atomicExch(&status[tile], TS_OWN | own);
    const uint64_t t0 = globaltimer_ns();
    for (int64_t p = tile - 1; p >= 0;) {
      unsigned long long w = TS_ALL;  // before the first tile: nothing
      if (p - lane >= 0) w = *(volatile unsigned long long *)&status[p - lane];
      const unsigned ready = __ballot_sync(FULL, (w >> 62) != 0);
      const unsigned all = __ballot_sync(FULL, (w >> 62) == 2ull);
      // the tiles up to the first with a count from the start, as far as they have one
      const int ends = all ? __ffs(all) : 33, gap = ready == FULL ? 32 : __ffs(~ready) - 1;
      const int use = min(ends, gap);
      before += warp_sum(lane < use ? w & TS_VAL : 0ull);
      if (use == ends) break;
      p -= use;
      if (use == 0 && globaltimer_ns() - t0 > 1000ull * 1000 * 1000) {
        if (lane == 0) atomicOr(err, DERR_TIMEOUT);
        break;
      }
    }
  }
  if (lane == 0) atomicExch(&status[tile], TS_ALL | (before + own));
  return before;
}

constexpr int CI = 8;             // sorted positions a thread
constexpr int CTILE = TB * CI;    // ... and a tile

// The clusters of the sorted labels: cl[i] = the cluster of sorted position i
// (-1: unclustered), cstart[c] = its first position (cstart[K] = n), dsum[c]
// += the degrees of its members; also K and the unclustered vertices (they
// sort first).  One pass: a tile counts its first-of-a-label positions and
// adds the earlier tiles' count by look-back.
__global__ void __launch_bounds__(TB) k_clusters(const uint32_t *__restrict__ sk,
                                                const uint32_t *__restrict__ sv,
                                                const int64_t *__restrict__ off, int64_t n,
                                                int32_t *cl, int64_t *cstart,
                                                unsigned long long *dsum,
                                                unsigned long long *status, SeedInfo *info) {
  __shared__ int sm[TB / 32 + 1];
  __shared__ unsigned tile_sh;
  __shared__ unsigned long long before_sh;
  if (threadIdx.x == 0) tile_sh = atomicAdd(&info->ticket, 1u);
  __syncthreads();
  const int64_t tile = tile_sh, base = tile * CTILE + (int64_t)threadIdx.x * CI;
  uint32_t k[CI];
  long long deg[CI];
  uint32_t prev = base > 0 && base - 1 < n ? sk[base - 1] : 0u;
  int heads = 0;
#pragma unroll
  for (int z = 0; z < CI; ++z) k[z] = base + z < n ? sk[base + z] : 0u;
#pragma unroll
  for (int z = 0; z < CI; ++z) {
    const uint32_t v = base + z < n && k[z] ? sv[base + z] : 0u;
    // (v is any value after a sort whose wait ran out; the host fails the call later)
    deg[z] = base + z < n && k[z] && (int64_t)v < n ? off[v + 1] - off[v] : 0;
  }
  unsigned first = 0u;
#pragma unroll
  for (int z = 0; z < CI; ++z) {
    if (base + z < n && k[z] != 0u && k[z] != prev) {
      first |= 1u << z;
      ++heads;
    }
    prev = k[z];
  }
  int tot;
  const int ex = block_exclusive_scan<TB>(heads, &tot, sm);
  if (threadIdx.x < 32) {
    const unsigned long long b = tiles_before(status, tile, (unsigned long long)tot, &info->err);
    if (threadIdx.x == 0) before_sh = b;
  }
  __syncthreads();
  int64_t c = (int64_t)before_sh + ex - 1;  // the cluster the thread's first position continues
  const int64_t c0 = c + ((first & 1u) ? 1 : 0);
  const bool whole = first == 0u || first == 1u;  // the thread's positions are one cluster's
  long long sum = 0;
#pragma unroll
  for (int z = 0; z < CI; ++z) {
    const int64_t i = base + z;
    if (i >= n) break;
    if ((first >> z) & 1u) {
      if (sum && c >= 0) atomicAdd(&dsum[c], (unsigned long long)sum);
      sum = 0;
      ++c;
      cstart[c] = i;
      if (c == 0) info->skip = i;
    }
    cl[i] = k[z] ? (int32_t)c : -1;
    sum += deg[z];
  }
  // the last run's sum, once per warp when the warp is inside one cluster
  const int64_t lead = __shfl_sync(FULL, c0, 0);
  const bool same = __all_sync(FULL, whole && c0 == lead);
  if (same) {
    sum = warp_sum(sum);
    if ((threadIdx.x & 31) != 0) sum = 0;
  }
  if (sum && c >= 0) atomicAdd(&dsum[c], (unsigned long long)sum);
  if (threadIdx.x == 0 && tile == (n - 1) / CTILE) {
    const int64_t K = (int64_t)before_sh + tot;
    cstart[K] = n;
    info->clusters = K;
    if (K == 0) info->skip = n;
  }
}

// Which clusters are kept, how many, and the largest size and degree sum.
__global__ void k_keep(const int64_t *__restrict__ cstart, int min_size, uint32_t *keep,
                       const unsigned long long *__restrict__ dsum, SeedInfo *info) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t K = info->clusters;
  if (c - (int64_t)(threadIdx.x & 31) >= K) return;  // the whole warp is past the last cluster
  unsigned long long sz = 0, ds = 0;
  bool k = false;
  if (c < K) {
    sz = (unsigned long long)(cstart[c + 1] - cstart[c]);
    k = (int64_t)sz >= min_size;
    keep[c] = k ? 1u : 0u;
    ds = k ? dsum[c] : 0ull;
    if (!k) sz = 0;
  }
  sz = warp_max(sz);
  ds = warp_max(ds);
  const unsigned kept = __popc(__ballot_sync(FULL, k));
  if ((threadIdx.x & 31) == 0) {
    if (sz) atomicMax(&info->max_n, sz);
    if (ds) atomicMax(&info->max_dsum, ds);
    if (kept) atomicAdd(&info->kept, kept);
  }
}

// All values a[0..P) ascending, P a power of two, by a block of T threads.
template <int T>
__device__ __forceinline__ void block_bitonic(unsigned long long *a, int P) {
  for (int k = 2; k <= P; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < P / 2; i += T) {
        const int o = i & (j - 1), lo = 2 * (i - o) + o, hi = lo + j;
        const unsigned long long x = a[lo], y = a[hi];
        if ((x > y) == ((lo & k) == 0)) {
          a[lo] = y;
          a[hi] = x;
        }
      }
      __syncthreads();
    }
}

// The whole grouping of a graph of at most GROUP_SMALL vertices by one CTA, in
// place of about fifteen launches whose gaps would be most of its time: labels
// sorted with their vertices in shared memory, clusters, degree sums and the
// queue order as the kernels above and below give them.
__global__ void __launch_bounds__(GT) k_group_small(const int32_t *__restrict__ lab, int n,
                                                   const int64_t *__restrict__ off, int min_size,
                                                   uint32_t *sv, int32_t *cl, int64_t *cstart,
                                                   uint32_t *keep, uint32_t *qidx, SeedInfo *info) {
  extern __shared__ __align__(16) unsigned long long a[];
  __shared__ int sm[GT / 32 + 1];
  __shared__ unsigned bad, kept;
  __shared__ int skip;
  __shared__ unsigned long long max_n, max_d;
  if (threadIdx.x == 0) {
    bad = kept = 0u;
    skip = n;
    max_n = max_d = 0ull;
  }
  __syncthreads();
  int P = 2;
  while (P < n) P <<= 1;
  for (int i = threadIdx.x; i < P; i += GT) {
    unsigned long long key = ~0ull;
    if (i < n) {
      const int32_t c = lab[i];
      if (c < -1) bad = 1u;
      key = ((unsigned long long)((unsigned)c + 1u) << 32) | (unsigned)i;
    }
    a[i] = key;
  }
  __syncthreads();
  if (bad) {
    if (threadIdx.x == 0) {
      SeedInfo r{};
      r.err = DERR_INVALID;
      *info = r;
    }
    return;
  }
  block_bitonic<GT>(a, P);
  int K = 0;
  for (int i0 = 0; i0 < n; i0 += GT) {
    const int i = i0 + threadIdx.x;
    const unsigned key = i < n ? (unsigned)(a[i] >> 32) : 0u;
    const bool head = key != 0u && (i == 0 || (unsigned)(a[i - 1] >> 32) != key);
    int tot;
    const int ex = block_exclusive_scan<GT>(head ? 1 : 0, &tot, sm);
    if (i < n) {
      const int c = K + ex + (head ? 1 : 0) - 1;
      sv[i] = (unsigned)a[i];
      cl[i] = key ? c : -1;
      if (head) cstart[c] = i;
      if (head && c == 0) skip = i;
    }
    K += tot;
  }
  if (threadIdx.x == 0) cstart[K] = n;
  __syncthreads();
  for (int c = threadIdx.x; c < K; c += GT) a[c] = 0ull;  // degree sums
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += GT) {
    const int c = cl[i];
    const uint32_t v = sv[i];
    if (c >= 0) atomicAdd(&a[c], (unsigned long long)(off[v + 1] - off[v]));
  }
  __syncthreads();
  for (int c = threadIdx.x; c < K; c += GT) {
    const unsigned long long sz = (unsigned long long)(cstart[c + 1] - cstart[c]);
    const bool k = (int64_t)sz >= min_size;
    keep[c] = k ? 1u : 0u;
    if (k) {
      atomicAdd(&kept, 1u);
      atomicMax(&max_n, sz);
      atomicMax(&max_d, a[c]);
    }
  }
  __syncthreads();
  // queue order: kept clusters first, larger ones earlier
  int Q = 2;
  while (Q < K) Q <<= 1;
  for (int c = threadIdx.x; c < Q; c += GT) {
    unsigned long long key = ~0ull;
    if (c < K)
      key = ((keep[c] ? max_n - (unsigned long long)(cstart[c + 1] - cstart[c]) : max_n + 1) << 32) |
            (unsigned)c;
    a[c] = key;
  }
  __syncthreads();
  block_bitonic<GT>(a, Q);
  for (int i = threadIdx.x; i < (int)kept; i += GT) qidx[(unsigned)a[i]] = (uint32_t)i;
  if (threadIdx.x == 0) {
    SeedInfo r{};
    r.max_n = max_n;
    r.max_dsum = max_d;
    r.clusters = K;
    r.skip = skip;
    r.kept = kept;
    *info = r;
  }
}

// Sort keys putting kept clusters first, larger ones earlier (longest work
// first); unkept clusters get the largest key.
__global__ void k_size_keys(const int64_t *__restrict__ cstart, const uint32_t *__restrict__ keep,
                            int64_t K, uint32_t max_n, uint32_t *keys, uint32_t *vals) {
  int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= K) return;
  uint32_t sz = (uint32_t)(cstart[c + 1] - cstart[c]);
  keys[c] = keep[c] ? max_n - sz : max_n + 1;
  vals[c] = (uint32_t)c;
}

// The same order for at most ORDER_SMALL clusters in one block: the keys of
// k_size_keys paired with the cluster index (which breaks ties as the
// stable sort does), sorted by a bitonic network in shared memory, and the
// kept clusters' ranks written as k_invert does.
constexpr int ORDER_SMALL = 4096;
__global__ void __launch_bounds__(1024) k_order_small(const int64_t *__restrict__ cstart,
                                                      const uint32_t *__restrict__ keep, int64_t K,
                                                      uint32_t max_n, int64_t nkept,
                                                      uint32_t *qidx) {
  __shared__ unsigned long long a[ORDER_SMALL];
  int P = 2;
  while (P < K) P <<= 1;
  for (int i = threadIdx.x; i < P; i += blockDim.x) {
    unsigned long long v = ~0ull;
    if (i < K) {
      const uint32_t sz = (uint32_t)(cstart[i + 1] - cstart[i]);
      const uint32_t key = keep[i] ? max_n - sz : max_n + 1;
      v = ((unsigned long long)key << 32) | (unsigned)i;
    }
    a[i] = v;
  }
  __syncthreads();
  block_bitonic<1024>(a, P);
  for (int i = threadIdx.x; i < nkept; i += blockDim.x) qidx[(uint32_t)a[i]] = (uint32_t)i;
}

__global__ void k_invert(const uint32_t *__restrict__ order, int64_t nkept, int64_t K,
                         uint32_t *qidx) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nkept && order[i] < K) qidx[order[i]] = (uint32_t)i;  // (any value after a failed sort)
}

// Reserves queue indices [base, base + nkept) for the items of one request
// and counts them as pending (globally and for the request) before any of
// them is published.  One thread.
__device__ __forceinline__ unsigned long long reserve(RunCounters *ctr, ReqCtx *ctx,
                                                      long long nkept) {
  atomicAdd(reinterpret_cast<unsigned long long *>(&ctx->pending),
            static_cast<unsigned long long>(nkept));
  atomicAdd(reinterpret_cast<unsigned long long *>(&ctr->pending),
            static_cast<unsigned long long>(nkept));
  __threadfence();
  const unsigned long long b = atomicAdd(&ctr->tail, (unsigned long long)nkept);
  ctx->seed_end = b + (unsigned long long)nkept;
  return b;
}
__global__ void k_reserve(RunCounters *ctr, ReqCtx *ctx, long long nkept,
                          unsigned long long *base) {
  if (threadIdx.x == 0 && blockIdx.x == 0) *base = reserve(ctr, ctx, nkept);
}

// What seeding reads: the grouping's arrays.
struct SeedIn {
  const uint32_t *sv;
  const int32_t *cl;
  const int64_t *cstart;
  const uint32_t *keep, *qidx;
  int64_t n, skip, K;
};

// pool[i - skip] = sorted vertex; slot[v] = (queue index << 32) | rank
__device__ __forceinline__ void seed_vertex(const SeedIn &in, int64_t i, unsigned long long base,
                                            int32_t *pool, unsigned long long *slot) {
  const uint32_t v = in.sv[i];
  pool[i - in.skip] = (int32_t)v;
  const int32_t c = in.cl[i];
  if (in.keep[c])
    slot[v] = ((unsigned long long)queue_tag(base + in.qidx[c]) << 32) |
              (unsigned)(i - in.cstart[c]);
}

// The descriptor of a kept cluster, then its publication.
__device__ __forceinline__ void seed_cluster(const SeedIn &in, int64_t c, unsigned long long base,
                                             uint16_t req, QSlot *ring, uint64_t cap) {
  const uint64_t q = base + in.qidx[c];
  QSlot *s = &ring[q % cap];
  s->item.vbeg = in.cstart[c] - in.skip;
  s->item.n = (int32_t)(in.cstart[c + 1] - in.cstart[c]);
  s->item.flags = ITEM_TOP;
  s->item.req = req;
  __threadfence();
  atomicExch((unsigned long long *)&s->seq, (unsigned long long)q);
}

__global__ void k_pool_slots(SeedIn in, const unsigned long long *__restrict__ base, int32_t *pool,
                             unsigned long long *slot) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < in.n && i >= in.skip) seed_vertex(in, i, *base, pool, slot);
}

__global__ void k_seed(SeedIn in, const unsigned long long *__restrict__ base, uint16_t req,
                       QSlot *ring, uint64_t cap) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c < in.K && in.keep[c]) seed_cluster(in, c, *base, req, ring, cap);
}

// The three steps above in one launch, for a small graph.
__global__ void __launch_bounds__(GT) k_seed_small(SeedIn in, RunCounters *ctr, ReqCtx *ctx,
                                                  long long nkept, uint16_t req, int32_t *pool,
                                                  unsigned long long *slot, QSlot *ring,
                                                  uint64_t cap) {
  __shared__ unsigned long long base;
  if (threadIdx.x == 0) base = reserve(ctr, ctx, nkept);
  __syncthreads();
  for (int64_t i = in.skip + threadIdx.x; i < in.n; i += GT) seed_vertex(in, i, base, pool, slot);
  __threadfence();
  __syncthreads();
  for (int64_t c = threadIdx.x; c < in.K; c += GT)
    if (in.keep[c]) seed_cluster(in, c, base, req, ring, cap);
}

// rank[v] = representatives (label_min[v] == v) before v, in one pass over
// tiles (see tiles_before).
__global__ void __launch_bounds__(TB) k_rank(const int32_t *__restrict__ lmin, int64_t n,
                                            uint32_t *rank, unsigned long long *status,
                                            unsigned *ticket, unsigned *err) {
  __shared__ int sm[TB / 32 + 1];
  __shared__ unsigned tile_sh;
  __shared__ unsigned long long before_sh;
  if (threadIdx.x == 0) tile_sh = atomicAdd(ticket, 1u);
  __syncthreads();
  const int64_t tile = tile_sh, base = tile * CTILE + (int64_t)threadIdx.x * CI;
  int32_t l[CI];
#pragma unroll
  for (int z = 0; z < CI; ++z) l[z] = base + z < n ? lmin[base + z] : -1;
  int mine = 0;
#pragma unroll
  for (int z = 0; z < CI; ++z) mine += base + z < n && l[z] == (int32_t)(base + z);
  int tot;
  const int ex = block_exclusive_scan<TB>(mine, &tot, sm);
  if (threadIdx.x < 32) {
    const unsigned long long b = tiles_before(status, tile, (unsigned long long)tot, err);
    if (threadIdx.x == 0) before_sh = b;
  }
  __syncthreads();
  uint32_t r = (uint32_t)before_sh + (uint32_t)ex;
#pragma unroll
  for (int z = 0; z < CI; ++z) {
    if (base + z >= n) break;
    rank[base + z] = r;
    r += l[z] == (int32_t)(base + z);
  }
}

// Both steps of the numbering for a small graph, by one CTA.
__global__ void __launch_bounds__(GT) k_number_small(const int32_t *__restrict__ lmin, int n,
                                                    int32_t *out, const unsigned *err) {
  extern __shared__ __align__(16) unsigned long long a[];
  int32_t *rank = reinterpret_cast<int32_t *>(a);
  __shared__ int sm[GT / 32 + 1];
  if (err && *err) return;
  int carry = 0;
  for (int i0 = 0; i0 < n; i0 += GT) {
    const int i = i0 + threadIdx.x;
    const int f = i < n && lmin[i] == i ? 1 : 0;
    int tot;
    const int ex = block_exclusive_scan<GT>(f, &tot, sm);
    if (i < n) rank[i] = carry + ex;
    carry += tot;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += GT) {
    const int32_t r = lmin[i];
    out[i] = r >= 0 ? rank[r] : -1;
  }
}

__global__ void k_out_final(const int32_t *__restrict__ lmin, const uint32_t *__restrict__ rank,
                            int64_t n, int32_t *out, const unsigned *err) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n || *err) return;
  int32_t r = lmin[i];
  out[i] = r >= 0 ? (int32_t)rank[r] : -1;
}

// The state a run starts from: every vertex in no item and no cluster, no ring
// slot published, the counters zero, the request's context.
__global__ void k_run_init(int64_t n, unsigned long long *slot, int32_t *lmin, QSlot *ring,
                           uint64_t cap, RunCounters *ctr, ReqCtx *req, ReqCtx value) {
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = i0; i < n; i += step) {
    slot[i] = ~0ull;
    lmin[i] = -1;
  }
  for (int64_t i = i0; i < (int64_t)cap; i += step) ring[i].seq = ~0ull;
  if (i0 == 0) {
    *ctr = RunCounters{};
    *req = value;
  }
}

template <typename T>
T *buf(Workspace &ws, int k, size_t count) {
  return static_cast<T *>(ws.b[k].ensure(sizeof(T) * (count > 0 ? count : 1)));
}

}  // namespace

int64_t bitlen_u64(uint64_t x) {
  int64_t b = 0;
  while (x) { ++b; x >>= 1; }
  return b;
}

unsigned grid_for(int64_t n, int per) {
  int64_t b = (n + per - 1) / per;
  if (b < 1) b = 1;
  if (b > 0x7fffffff) b = 0x7fffffff;
  return (unsigned)b;
}

void check_device_error(unsigned err, const char *what) {
  if (!err) return;
  if (err & DERR_INVALID) fail(WCC_ERR_INVALID, std::string(what) + ": malformed input");
  if (err & DERR_TIMEOUT)
    fail(WCC_ERR_TIMEOUT, std::string(what) + ": a device-side queue wait exceeded its limit");
  if (err & DERR_CAPACITY)
    fail(WCC_ERR_INTERNAL, std::string(what) + ": an internal capacity bound was exceeded");
  fail(WCC_ERR_INTERNAL, std::string(what) + ": internal consistency check failed");
}

GroupInfo group_by_label(const int64_t *off, int64_t n, const int32_t *labels, int min_size,
                         Workspace &ws, cudaStream_t s) {
  GroupInfo gi{};
  uint32_t *keys = buf<uint32_t>(ws, B_KEYS, n);
  uint32_t *vals = buf<uint32_t>(ws, B_VALS, n);
  int32_t *cl = buf<int32_t>(ws, B_CL, n);
  int64_t *cstart = buf<int64_t>(ws, B_CSTART, n + 1);
  uint32_t *keep = buf<uint32_t>(ws, B_KEEP, n + 1);
  uint32_t *qidx = buf<uint32_t>(ws, B_QIDX, n + 1);
  auto fill = [&](const SeedInfo &hi) {
    if (hi.err) check_device_error(hi.err, "grouping");
    gi.clusters = hi.clusters;
    gi.skip = hi.skip;
    gi.kept = (int64_t)hi.kept;
    gi.max_n = (int64_t)hi.max_n;
    gi.max_dsum = (int64_t)hi.max_dsum;
  };
  if (n <= GROUP_SMALL) {
    SeedInfo *info = buf<SeedInfo>(ws, B_INFO, 1);
    size_t P = 2;
    while ((int64_t)P < n) P <<= 1;
    k_group_small<<<1, GT, 8 * P, s>>>(labels, (int)n, off, min_size, vals, cl, cstart, keep, qidx,
                                       info);
    note_launch();
    WCC_CUDA(cudaGetLastError());
    const SeedInfo hi = read_back(info, s);
    if (hi.err) check_device_error(hi.err, "clustering_in");
    ws.sv = vals;
    fill(hi);
    return gi;
  }
  uint32_t *keys2 = buf<uint32_t>(ws, B_KEYS2, n);
  uint32_t *vals2 = buf<uint32_t>(ws, B_VALS2, n);
  void *temp = ws.b[B_TEMP].ensure(std::max(radix_temp_bytes(n), scan_temp_bytes(n + 1)));
  // the counters, the tiles' status words and the degree sums start at zero
  const int64_t tiles = (n + CTILE - 1) / CTILE;
  const size_t zero = sizeof(SeedInfo) + 8 * (size_t)tiles + 8 * (size_t)n;
  SeedInfo *info = static_cast<SeedInfo *>(ws.b[B_INFO].ensure(zero));
  unsigned long long *status = reinterpret_cast<unsigned long long *>(info + 1);
  unsigned long long *dsum = status + tiles;
  WCC_CUDA(cudaMemsetAsync(info, 0, zero, s));
  k_make_keys<<<grid_for(n), TB, 0, s>>>(labels, n, keys, vals, &info->maxkey, &info->err);
  note_launch();
  WCC_CUDA(cudaGetLastError());
  SeedInfo h0 = read_back(info, s);
  if (h0.err) check_device_error(h0.err, "clustering_in");
  uint32_t *sk = keys, *sv = vals;
  if (radix_sort_pairs_u32(keys, vals, keys2, vals2, n, (int)bitlen_u64(h0.maxkey), temp,
                           &info->err, s)) {
    sk = keys2;
    sv = vals2;
  }
  ws.sv = sv;
  k_clusters<<<(unsigned)tiles, TB, 0, s>>>(sk, sv, off, n, cl, cstart, dsum, status, info);
  note_launch();
  k_keep<<<grid_for(n), TB, 0, s>>>(cstart, min_size, keep, dsum, info); note_launch();
  WCC_CUDA(cudaGetLastError());
  fill(read_back(info, s));
  const int64_t K = gi.clusters;
  if (gi.kept > 0 && K <= ORDER_SMALL) {
    // queue order: largest input clusters first (qidx = rank by size), in one block
    k_order_small<<<1, 1024, 0, s>>>(cstart, keep, K, (uint32_t)gi.max_n, gi.kept, qidx);
    note_launch();
    WCC_CUDA(cudaGetLastError());
  } else if (gi.kept > 0) {
    // queue order: largest input clusters first (qidx = rank by size)
    uint32_t *ok1 = buf<uint32_t>(ws, B_OK1, K);
    uint32_t *ov1 = buf<uint32_t>(ws, B_OV1, K);
    uint32_t *ok2 = buf<uint32_t>(ws, B_OK2, K);
    uint32_t *ov2 = buf<uint32_t>(ws, B_OV2, K);
    k_size_keys<<<grid_for(K), TB, 0, s>>>(cstart, keep, K, (uint32_t)gi.max_n, ok1, ov1);
    note_launch();
    uint32_t *ov = ov1;
    if (radix_sort_pairs_u32(ok1, ov1, ok2, ov2, K, (int)bitlen_u64(gi.max_n + 1), temp,
                             &info->err, s))
      ov = ov2;
    k_invert<<<grid_for(gi.kept), TB, 0, s>>>(ov, gi.kept, K, qidx); note_launch();
    WCC_CUDA(cudaGetLastError());
    const unsigned e = read_back(&info->err, s);
    if (e) check_device_error(e, "grouping");
  }
  return gi;
}

void seed_items(const GroupInfo &gi, int64_t n, Workspace &ws, uint16_t req, ReqCtx *ctx_dev,
                int32_t *pool, unsigned long long *slot, QSlot *ring, uint64_t cap,
                RunCounters *ctr, cudaStream_t s) {
  if (gi.kept <= 0) return;
  const SeedIn in{ws.sv,
                  static_cast<int32_t *>(ws.b[B_CL].p),
                  static_cast<int64_t *>(ws.b[B_CSTART].p),
                  static_cast<uint32_t *>(ws.b[B_KEEP].p),
                  static_cast<uint32_t *>(ws.b[B_QIDX].p),
                  n,
                  gi.skip,
                  gi.clusters};
  if (n <= GROUP_SMALL) {
    k_seed_small<<<1, GT, 0, s>>>(in, ctr, ctx_dev, gi.kept, req, pool, slot, ring, cap);
    note_launch();
    WCC_CUDA(cudaGetLastError());
    return;
  }
  unsigned long long *base = buf<unsigned long long>(ws, B_BASE, 1);
  k_reserve<<<1, 32, 0, s>>>(ctr, ctx_dev, gi.kept, base); note_launch();
  k_pool_slots<<<grid_for(n), TB, 0, s>>>(in, base, pool, slot); note_launch();
  k_seed<<<grid_for(gi.clusters), TB, 0, s>>>(in, base, req, ring, cap); note_launch();
  WCC_CUDA(cudaGetLastError());
}

// ---- merging refinements of disjoint sets of input clusters ------------------
__global__ void k_fill_i32(int32_t *a, int64_t n, int32_t v) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] = v;
}

// Per vertex, the smallest vertex of its cluster, from labels in [-1, n):
// every vertex lowers its label's entry of mins (initially n) to its id.
__global__ void k_label_mins(const int32_t *__restrict__ lab, int64_t n, int32_t *mins,
                             unsigned *err) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t l = lab[i];
  if (l < -1 || l >= n) {
    atomicOr(err, DERR_INVALID);
    return;
  }
  if (l >= 0) atomicMin(&mins[l], (int32_t)i);
}

__global__ void k_vertex_mins(const int32_t *__restrict__ lab, const int32_t *__restrict__ mins,
                              int64_t n, int32_t *out) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t l = lab[i];
  out[i] = (l >= 0 && l < n) ? mins[l] : -1;
}

// Minima must name a vertex of the same cluster whose own minimum is
// itself (a representative), and never exceed the vertex.
__global__ void k_check_minima(const int32_t *__restrict__ mn, int64_t n, unsigned *err) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t r = mn[i];
  if (r == -1) return;
  if (r < 0 || r > i || mn[r] != r) atomicOr(err, DERR_INVALID);
}

__global__ void k_max_i32(const int32_t *__restrict__ a, int64_t n, int32_t *out) {
  int32_t m = -1;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    m = a[i] > m ? a[i] : m;
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) atomicMax(out, m);
}

void k_max_i32_launch(const int32_t *a, int64_t n, int32_t *out, cudaStream_t s) {
  const unsigned g = grid_for(n) < 1024u ? grid_for(n) : 1024u;
  k_max_i32<<<g, TB, 0, s>>>(a, n, out); note_launch();
  WCC_CUDA(cudaGetLastError());
}

void cluster_minima(const int32_t *labels, int64_t n, int32_t *minima, Workspace &ws,
                    cudaStream_t s) {
  int32_t *mins = buf<int32_t>(ws, B_RANK, n);
  unsigned *err = buf<unsigned>(ws, B_FLAG, 1);
  WCC_CUDA(cudaMemsetAsync(err, 0, 4, s));
  if (n > 0) {
    k_fill_i32<<<grid_for(n), TB, 0, s>>>(mins, n, (int32_t)n); note_launch();
    k_label_mins<<<grid_for(n), TB, 0, s>>>(labels, n, mins, err); note_launch();
    k_vertex_mins<<<grid_for(n), TB, 0, s>>>(labels, mins, n, minima); note_launch();
    WCC_CUDA(cudaGetLastError());
  }
  unsigned h = 0;
  WCC_CUDA(cudaMemcpyAsync(&h, err, 4, cudaMemcpyDeviceToHost, s));
  WCC_CUDA(cudaStreamSynchronize(s));
  if (h) fail(WCC_ERR_INVALID, "a label outside [-1, n)");
}

void check_minima(const int32_t *minima, int64_t n, Workspace &ws, cudaStream_t s) {
  unsigned *err = buf<unsigned>(ws, B_TEMP, 1);
  WCC_CUDA(cudaMemsetAsync(err, 0, 4, s));
  if (n > 0) {
    k_check_minima<<<grid_for(n), TB, 0, s>>>(minima, n, err); note_launch();
    WCC_CUDA(cudaGetLastError());
  }
  unsigned h = 0;
  WCC_CUDA(cudaMemcpyAsync(&h, err, 4, cudaMemcpyDeviceToHost, s));
  WCC_CUDA(cudaStreamSynchronize(s));
  if (h) fail(WCC_ERR_INVALID, "minima: an entry is not the smallest vertex of a cluster");
}

void run_init(int64_t n, unsigned long long *slot, int32_t *lmin, QSlot *ring, uint64_t cap,
              RunCounters *ctr, ReqCtx *req, const ReqCtx &value, cudaStream_t s) {
  const int64_t most = std::max<int64_t>(n, (int64_t)cap);
  k_run_init<<<std::min<unsigned>(grid_for(most), 152 * 16), TB, 0, s>>>(n, slot, lmin, ring, cap,
                                                                       ctr, req, value);
  note_launch();
  WCC_CUDA(cudaGetLastError());
}

unsigned *number_clusters(const int32_t *label_min, int64_t n, int32_t *out, Workspace &ws,
                          cudaStream_t s, unsigned *err) {
  if (n <= GROUP_SMALL) {
    k_number_small<<<1, GT, 4 * (size_t)n, s>>>(label_min, (int)n, out, err); note_launch();
    WCC_CUDA(cudaGetLastError());
    return nullptr;
  }
  uint32_t *rank = buf<uint32_t>(ws, B_RANK, n);
  const int64_t tiles = (n + CTILE - 1) / CTILE;
  const size_t zero = 8 * (size_t)(tiles + 1);
  unsigned long long *status = static_cast<unsigned long long *>(ws.b[B_FLAG].ensure(zero));
  unsigned *ticket = reinterpret_cast<unsigned *>(status + tiles);
  if (!err) err = ticket + 1;
  WCC_CUDA(cudaMemsetAsync(status, 0, zero, s));
  k_rank<<<(unsigned)tiles, TB, 0, s>>>(label_min, n, rank, status, ticket, err); note_launch();
  k_out_final<<<grid_for(n), TB, 0, s>>>(label_min, rank, n, out, err); note_launch();
  WCC_CUDA(cudaGetLastError());
  return err;
}

}  // namespace wccg
