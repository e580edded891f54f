// refine.cu -- the refinement kernel: one CTA processes one work item at a
// time (an input cluster, or a part produced by an earlier split), entirely
// in on-chip shared memory when the item fits, else in a per-CTA slab of
// global memory.
//
// Per item (paper: Algorithm 1 for input clusters, then Algorithm 3 with a
// peel and a connectivity check in front of the cut):
//   1. extraction of the induced subgraph G[S] (Algorithm 1 / 3: E_c = edges
//      with both ends in V_c) into local rows, local id = rank of the global
//      id in S: one pass over all adjacency entries of the members with an
//      8-byte gather of slot[u] = (item << 32 | local id) per entry; local
//      ids are 16-bit when the item has < 65535 vertices;
//   2. input clusters only: connected components (CCR); each component with
//      at least min_size vertices is queued, or refinement continues in place
//      when the cluster is one component;
//   3. round-synchronous peel of vertices with degree <= T(n);
//   4. if the peel removed anything: connected components; more than one ->
//      queue each large component (an item arrives connected, so without a
//      peel the check is skipped);
//   5. Nagamochi-Ibaraki contraction with k = T+1: maximum-adjacency passes
//      (keys capped at k, ties to the smallest id) merging every edge whose
//      key reaches k, until one super-vertex (accept: min cut > T) or a pass
//      merges nothing; a pass is grown phase by phase by the whole CTA (see
//      "contraction passes");
//   6. otherwise canonical Stoer-Wagner on the contracted graph (ties to the
//      smallest id, earliest minimum phase, side = last-added super-vertex)
//      and both sides with at least min_size vertices are queued
//      (MinCutPartition and the recursion of Algorithm 3).
// Children are written in place into the parent's range of the vertex pool
// and published to a device-side ring queue; CTAs claim queue indices with
// an atomic counter and wait (bounded by %globaltimer) for publication.
#include "internal.h"

namespace wccg {

namespace {

// Threads per CTA, one CTA per SM.  The block-wide loops are bound by latency,
// so more warps hide more of it, until 128 registers a thread are too few and
// a barrier costs more than it saves.  Graph resident, with 256 / 512 / 1024
// threads: clusters of up to 50,000 vertices (1M vertices) 8.96 / 6.78 / 6.20
// ms, small clusters (2M) 4.28 / 3.98 / 4.21, LFR-style 100k 0.567 / 0.557 /
// 0.593, planted 1k 0.246 / 0.255 / 0.283.
constexpr int RB = 512;
constexpr int RW = RB / 32;    // warps per CTA
constexpr size_t SMEM_MAX_BYTES = 227 * 1024;  // opt-in limit per CTA

// Dynamic shared memory of a refinement CTA.  Item code instantiated for
// shared memory derives every pointer from this symbol, so the compiler
// knows their address space and uses shared-memory instructions instead of
// generic ones.
extern __shared__ __align__(16) char wcc_dyn_smem[];

// Components that a contraction pass finds one after the other; beyond that
// many the union-find finds all at once.
constexpr int MAX_COMP = 32;
// A search for components alone (CCR) that has added fewer than THIN_FRONT
// vertices a round on average, after THIN_ROUNDS of them, leaves the item to the
// union-find too: a round costs about 1,000 cycles whatever it adds, the
// union-find about 30 ns a vertex whatever the diameter.  One path of 50,000
// vertices 29.7 -> 2.7 ms, 200 of 2,000 1.66 -> 0.38, 200 chains of 300 triangles
// 0.94 -> 0.30 (after 16 or 64 rounds: 0.28, 0.35); without the average a 300 x 300
// grid takes 4.8 ms instead of 2.4.
constexpr int THIN_ROUNDS = 32;
constexpr int THIN_FRONT = 32;
// Rows of more entries are extracted by all warps together.
constexpr int LONG_ROW = 1024;
// Most small input clusters a CTA claims at once (see k_refine).  With one per
// warp and a barrier after them (a block of 7, 3.3 items a batch on average)
// 2M vertices in 100,000 small clusters took 9.29 ms instead of 4.21.
constexpr int TINY_BLOCK = 64;
// Items whose first contraction pass covers at least this many vertices
// record it for the sides of a later cut.
constexpr int INH_MIN_N = 64;

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }
// Keys of the first contraction pass: 16 bits a vertex, two to a word.
__host__ __device__ inline size_t key_bytes(int64_t n) { return align16(2 * (size_t)(n + 1)); }

// Working memory of one item of n vertices and at most d local adjacency
// entries (d = sum of the members' global degrees); see carve().
template <typename IT>
__host__ __device__ inline size_t ws_bytes(int64_t n, int64_t d) {
  size_t b = 0;
  b += align16(4 * (size_t)n);              // gid
  b += align16(4 * (size_t)(n + 1));        // off
  b += 6 * align16(4 * (size_t)(n + 1));    // A, B, C, D, G, H
  b += align16(8 * (size_t)(n + 1));        // E and F (one int64 array during extraction)
  b += 3 * align16((size_t)n);              // alive, flag, side
  b += key_bytes(n);                        // first contraction pass: keys
  b += align16(4 * (size_t)((d + 31) / 32 + 1));  // contraction marks, one bit per entry
  b += align16(sizeof(IT) * (size_t)n);     // row lengths
  b += align16(sizeof(IT) * (size_t)d);     // local adjacency
  return b + 64;
}

template <typename IT>
struct Mem {
  int32_t *gid, *off, *A, *B, *C, *D, *E, *F, *G, *H;
  int64_t *wide;       // E..F viewed as int64[n+1]
  uint8_t *alive, *flag, *side;
  uint32_t *kw;        // first contraction pass: 16-bit keys, two to a word
  uint32_t *ebits;     // one bit per local adjacency entry
  IT *len;             // row i: adj[off[i] .. off[i] + len[i]), in any order
  IT *adj;
  size_t smem_used;    // bytes of dynamic shared memory the item occupies
  __device__ __forceinline__ int end(int i) const { return off[i] + (int)len[i]; }
  bool off_in_smem;    // a global-slab item keeps its row offsets in shared memory
};

template <typename IT>
__device__ __forceinline__ Mem<IT> carve(char *base, int n, int64_t d) {
  Mem<IT> m;
  char *p = base;
  auto take = [&](size_t b) { char *r = p; p += align16(b); return r; };
  m.gid = (int32_t *)take(4 * (size_t)n);
  m.off = (int32_t *)take(4 * (size_t)(n + 1));
  m.A = (int32_t *)take(4 * (size_t)(n + 1));
  m.B = (int32_t *)take(4 * (size_t)(n + 1));
  m.C = (int32_t *)take(4 * (size_t)(n + 1));
  m.D = (int32_t *)take(4 * (size_t)(n + 1));
  m.G = (int32_t *)take(4 * (size_t)(n + 1));
  m.H = (int32_t *)take(4 * (size_t)(n + 1));
  m.wide = (int64_t *)take(8 * (size_t)(n + 1));
  m.E = (int32_t *)m.wide;
  m.F = m.E + (n + 1);
  m.alive = (uint8_t *)take((size_t)n);
  m.flag = (uint8_t *)take((size_t)n);
  m.side = (uint8_t *)take((size_t)n);
  m.kw = (uint32_t *)take(key_bytes(n));
  m.ebits = (uint32_t *)take(4 * (size_t)((d + 31) / 32 + 1));
  m.len = (IT *)take(sizeof(IT) * (size_t)n);
  m.adj = (IT *)take(sizeof(IT) * (size_t)d);
  m.smem_used = 0;
  m.off_in_smem = false;
  return m;
}

// An item in the global slab keeps the first contraction pass's keys (one
// random access per adjacency entry) in shared memory when they fit, and its
// row offsets too when they fit beside them.
template <typename IT>
__device__ __forceinline__ bool carve_hot(Mem<IT> &m, int n, size_t smem_bytes) {
  const size_t hb = key_bytes(n);
  if (hb > smem_bytes) return false;
  m.kw = reinterpret_cast<uint32_t *>(wcc_dyn_smem);
  m.smem_used = hb;
  if (hb + align16(4 * (size_t)(n + 1)) <= smem_bytes) {
    m.off = reinterpret_cast<int32_t *>(wcc_dyn_smem + hb);
    m.smem_used = hb + align16(4 * (size_t)(n + 1));
    m.off_in_smem = true;
  }
  return true;
}

// The item's memory in a function that is not inlined: an item in shared
// memory is carved again, so that its pointers keep their address space.
template <typename IT, bool SM>
__device__ __forceinline__ Mem<IT> item_mem(const Mem<IT> *m0, int n, int64_t d) {
  return SM ? carve<IT>(wcc_dyn_smem, n, d) : *m0;
}

// Block-level scalars.
struct Sh {
  int32_t scan[RW + 1];
  long long lscan[RW + 1];
  int go;
  int32_t i0;
  unsigned long long u0, u1;
  int32_t ntouched;
  int32_t changed;
  int32_t sw_s, sw_t, sw_cut, sw_x, sw_key;
  // per-item profile (only when RefineParams::prof is set)
  long long ts[9];
  long long dbg[4];
  int32_t used_slab, pf_E, pf_nalive, pf_passes, pf_nsv, pf_forest, pf_nsv1;
  long long pf_forest_cycles, pf_t0;
  long long fdbg[6];
  int32_t qn[3];                  // contraction pass: super-vertices pushed in a round
  int32_t ngrp;                   // ... groups touched since the last pick
  int32_t grp_all;                // ... or all of them
  unsigned long long wbest[RW];   // contraction pass: each warp's best unadded key
  Item first;         // the claimed item
  unsigned long long first_seq;
  unsigned long long claim_h;  // first index of the block of small items claimed after it
  int32_t claim_k;             // its length
  int32_t bnext;               // small items of the batch taken by warps so far
  int32_t bdone;               // ... and refined by them
  int32_t ncta;                // items for the whole CTA
  int32_t has_own;             // the CTA keeps a part of its last item as its next one
  Item own;
  Item cta_item[TINY_BLOCK + 1];
  unsigned long long cta_seq[TINY_BLOCK + 1];
  unsigned long long tst[7];   // statistics of the batch's small items
  int32_t wgrp[128];  // dense finish: the index that holds each initial one
  uint32_t wside[4];  // dense finish: side of the minimum cut (mask of indices)
  int32_t dcut, dpasses, dphases;
};

// Outcome of one item.
enum : int { OUT_ERROR = -1, OUT_DROPPED = 0, OUT_CCR_SPLIT = 1, OUT_CC_SPLIT = 2,
             OUT_ACCEPT = 3, OUT_CUT_SPLIT = 4 };

// Cycle stamp k of the per-item profile (thread 0; no-op unless enabled).
__device__ __forceinline__ void prof_stamp(const RefineParams &P, Sh &sh, int k) {
  if (P.prof && threadIdx.x == 0) sh.ts[k] = clock64();
}

// ---- small device helpers ----------------------------------------------------

// A request's context as this CTA sees it: loaded through L2 (not L1), since
// a server reuses a table entry for a later request while the kernel runs.
__device__ __forceinline__ ReqCtx load_ctx(const ReqCtx *g) {
  ReqCtx r;
  r.off = reinterpret_cast<const int64_t *>(__ldcg(reinterpret_cast<const unsigned long long *>(&g->off)));
  r.adj = reinterpret_cast<const int32_t *>(__ldcg(reinterpret_cast<const unsigned long long *>(&g->adj)));
  r.n_vertices = __ldcg(reinterpret_cast<const long long *>(&g->n_vertices));
  r.pool = reinterpret_cast<int32_t *>(__ldcg(reinterpret_cast<const unsigned long long *>(&g->pool)));
  r.slot = reinterpret_cast<unsigned long long *>(
      __ldcg(reinterpret_cast<const unsigned long long *>(&g->slot)));
  r.label_min =
      reinterpret_cast<int32_t *>(__ldcg(reinterpret_cast<const unsigned long long *>(&g->label_min)));
  r.inh = reinterpret_cast<unsigned long long *>(
      __ldcg(reinterpret_cast<const unsigned long long *>(&g->inh)));
  r.rule_kind = __ldcg(&g->rule_kind);
  r.min_size = __ldcg(&g->min_size);
  r.rule_num = __ldcg(reinterpret_cast<const long long *>(&g->rule_num));
  r.rule_den = __ldcg(reinterpret_cast<const long long *>(&g->rule_den));
  return r;
}

// Signed 64-bit atomic add (two's complement through the unsigned overload).
__device__ __forceinline__ void add_ll(long long *p, long long v) {
  atomicAdd(reinterpret_cast<unsigned long long *>(p), static_cast<unsigned long long>(v));
}

// Criterion threshold T(n) (Section 2, criterion f(n)): the largest integer
// with cut <= T(n) <=> cut <= f(n) for integer cuts.
__device__ int64_t threshold_of(int kind, int64_t num, int64_t den, int64_t n) {
  if (n < 1) return -1;
  int64_t t = 0, p = 1;
  switch (kind) {
    case WCC_RULE_LOG10:
      while (p <= n / 10) { p *= 10; ++t; }
      return t;
    case WCC_RULE_LOG2:
      return 63 - __clzll((unsigned long long)n);
    case WCC_RULE_SQRT: {
      t = (int64_t)sqrt((double)n);
      while (t > 0 && t * t > n) --t;
      while ((t + 1) * (t + 1) <= n) ++t;
      return t;
    }
    case WCC_RULE_LINEAR:
      return den > 0 ? (num * n) / den : -1;
    default:
      return -1;
  }
}

// Lock-free union-find over ids whose links always point to a smaller id, so
// the root of a set is its smallest member.
__device__ __forceinline__ int uf_find(int32_t *p, int x) {
  volatile int32_t *vp = p;
  int y = vp[x];
  while (y != x) {
    int z = vp[y];
    if (z != y) vp[x] = z;  // path halving: z is an ancestor of x
    x = y;
    y = z;
  }
  return x;
}

// The same without writing.
__device__ __forceinline__ int uf_root(const int32_t *p, int x) {
  const volatile int32_t *vp = p;
  for (int y; (y = vp[x]) != x;) x = y;
  return x;
}

__device__ __forceinline__ void uf_union(int32_t *p, int a, int b) {
  for (;;) {
    a = uf_find(p, a);
    b = uf_find(p, b);
    if (a == b) return;
    if (a > b) { int t = a; a = b; b = t; }
    int old = atomicCAS(&p[b], b, a);
    if (old == b) return;
    b = old;
  }
}

// Like uf_union, but reports whether the call joined two different sets.
// Concurrent calls are linearisable, so the edges whose call returned true
// form a spanning forest of all the edges tried.
__device__ __forceinline__ bool uf_link(int32_t *p, int a, int b) {
  for (;;) {
    a = uf_find(p, a);
    b = uf_find(p, b);
    if (a == b) return false;
    if (a > b) { int t = a; a = b; b = t; }
    if (atomicCAS(&p[b], b, a) == b) return true;
  }
}

// In-place exclusive scan of a[0..n) by the whole block; returns the total.
__device__ int block_scan_array(int32_t *a, int n, Sh &sh) {
  int carry = 0;
  for (int base = 0; base < n; base += RB) {
    int i = base + threadIdx.x;
    int v = i < n ? a[i] : 0;
    int tot;
    int ex = block_exclusive_scan<RB>(v, &tot, sh.scan);
    if (i < n) a[i] = carry + ex;
    carry += tot;
  }
  return carry;
}

__device__ int block_sum_int(int v, Sh &sh) {
  int tot;
  block_exclusive_scan<RB>(v, &tot, sh.scan);
  return tot;
}

__device__ long long block_sum_ll(long long v, Sh &sh) {
  long long tot;
  block_exclusive_scan<RB>(v, &tot, sh.lscan);
  return tot;
}

// ---- connected components (Afforest-style) ---------------------------------
// For items of more than MAX_COMP components (fewer come out of a contraction
// pass, see first_pass).  Union-find over the alive vertices (uf, root = smallest id): every vertex
// first links along its first two alive neighbours, the sets are
// compressed, and then only vertices outside the set of the smallest alive
// vertex process the rest of their rows (an edge with one end in that set is
// seen from its other end; an edge with both ends in it is already inside
// one set).  The result is exactly the connected components, with far fewer
// unions than hooking every edge.  cur is per-vertex scratch.
template <typename IT>
__device__ __forceinline__ void afforest(const Mem<IT> &m, int n, int32_t *uf, int32_t *cur,
                                         Sh &sh) {
  for (int i = threadIdx.x; i < n; i += RB) {
    uf[i] = i;
    cur[i] = m.off[i];
  }
  if (threadIdx.x == 0) sh.i0 = n;
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += RB)
    if (m.alive[i]) { atomicMin(&sh.i0, i); break; }
  // sampling: two alive neighbours per vertex
  for (int r = 0; r < 2; ++r) {
    for (int i = threadIdx.x; i < n; i += RB) {
      if (!m.alive[i]) continue;
      const int e = m.end(i);
      int q = cur[i];
      for (; q < e; ++q) {
        const int j = m.adj[q];
        if (m.alive[j]) {
          uf_union(uf, i, j);
          ++q;
          break;
        }
      }
      cur[i] = q;
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < n; i += RB)
    if (m.alive[i]) uf[i] = uf_find(uf, i);
  __syncthreads();
  const int i0 = sh.i0;
  const int giant = i0 < n ? uf_find(uf, i0) : -1;
  // every vertex outside the giant set processes the rest of its row
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < n; i += RB) {
    if (!m.alive[i]) continue;
    const int e = m.end(i);
    if (e - cur[i] > 64 || uf_find(uf, i) == giant) continue;
    for (int q = cur[i]; q < e; ++q) {
      const int j = m.adj[q];
      if (m.alive[j]) uf_union(uf, i, j);
    }
  }
  for (int i = warp; i < n; i += RW) {
    if (!m.alive[i]) continue;
    const int e = m.end(i);
    if (e - cur[i] <= 64 || uf_find(uf, i) == giant) continue;
    for (int q = cur[i] + lane; q < e; q += 32) {
      const int j = m.adj[q];
      if (m.alive[j]) uf_union(uf, i, j);
    }
  }
  __syncthreads();
  // the roots, by walks that write nothing on their way: a walk that halves its
  // path could store an ancestor over a root that another thread has just written,
  // and leave that vertex a component of its own
  for (int i = threadIdx.x; i < n; i += RB)
    if (m.alive[i]) uf[i] = uf_root(uf, i);
  __syncthreads();
}

// Connected components of the alive vertices by afforest(): B[i] = smallest
// alive id of i's component (-1 if dead); returns the number of components.
template <typename IT, bool SM>
__device__ __noinline__ int components_af(const Mem<IT> *m0, int64_t d, int n, Sh *shp) {
  Sh &sh = *shp;
  const Mem<IT> m = item_mem<IT, SM>(m0, n, d);
  int32_t *f = m.B, *cur = m.H;
  afforest(m, n, f, cur, sh);
  int roots = 0;
  for (int i = threadIdx.x; i < n; i += RB) {
    if (!m.alive[i]) {
      f[i] = -1;
      continue;
    }
    roots += f[i] == i;
  }
  __syncthreads();
  return block_sum_int(roots, sh);
}

// ---- publishing children -------------------------------------------------
// tag[i] (B or H) in [0, n) names the child of local vertex i (-1: none).  Every tag
// with at least min_size members becomes a new queue item whose vertex list
// (ascending) is written into the parent's pool range.  Uses C, D, E, F.
// With keep_largest, the kept child with the most members (ties: smallest
// tag) is not published: the caller refines it in place, and the children
// that are published fill the front of the range.  Returns that child's tag
// (-1: none) and, in *emitted, the members published ahead of it.
//
// With keep_own, that child is written to the pool like the others but not
// published: the CTA takes it as its next item (sh.own) under the queue index
// seq of the item it came from, which no one else uses any more.  A queue
// index then always stands for an unclaimed item, so that a request's
// unclaimed indices stay at half its vertices; the price is that a member of
// the parent which is in no child must not keep the parent's tag in its slot.
//
// This and the other parts of an item that are rare, long or used at several
// places are not inlined (item_mem says how they find the item's memory): the
// kernel's code then fits the instruction cache better and its main path the
// registers of 512 threads.
enum : int { TAG_B = 0, TAG_H = 1 };
template <typename IT, bool SM>
__device__ __noinline__ int emit_children(const RefineParams &P, const ReqCtx &R, ReqCtx *Rg,
                                          uint16_t req, const Mem<IT> *m0, int64_t d, int which,
                                          int n, int64_t vbeg, Sh *shp, uint16_t cflags = 0,
                                          bool keep_largest = false, int *emitted = nullptr,
                                          bool keep_own = false, unsigned long long seq = 0ull) {
  Sh &sh = *shp;
  const Mem<IT> m = item_mem<IT, SM>(m0, n, d);
  const int32_t *tag = which == TAG_H ? m.H : m.B;
  int32_t *cnt = m.C, *cidx = m.D, *cbase = m.E, *run = m.F;
  for (int t = threadIdx.x; t < n; t += RB) cnt[t] = 0;
  if (threadIdx.x == 0) sh.u1 = 0ull;
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += RB)
    if (tag[i] >= 0) atomicAdd(&cnt[tag[i]], 1);
  __syncthreads();
  if (keep_largest || keep_own) {
    unsigned long long best = 0ull;
    for (int t = threadIdx.x; t < n; t += RB)
      if (cnt[t] >= R.min_size) {
        const unsigned long long pk = ((unsigned long long)cnt[t] << 32) | (unsigned)(0x7fffffff - t);
        best = pk > best ? pk : best;
      }
    if (best) atomicMax(&sh.u1, best);
    __syncthreads();
  }
  const int big = sh.u1 ? 0x7fffffff - (int)(unsigned)(sh.u1 & 0xffffffffull) : -1;
  const int L = keep_own ? -1 : big, own = keep_own ? big : -1;
  for (int t = threadIdx.x; t < n; t += RB) {
    bool keep = cnt[t] >= R.min_size && t != L;
    cidx[t] = keep && t != own ? 1 : 0;
    cbase[t] = keep ? cnt[t] : 0;
    run[t] = 0;
  }
  __syncthreads();
  int nchild = block_scan_array(cidx, n, sh);
  const int total = block_scan_array(cbase, n, sh);
  if (emitted) *emitted = total;
  if (nchild == 0 && own < 0) return L;
  if (threadIdx.x == 0) {
    const long long pend = (long long)nchild + (own >= 0 ? 1 : 0);
    add_ll(&Rg->pending, pend);
    add_ll(&P.ctr->pending, pend);
    __threadfence();
    sh.u0 = nchild > 0 ? atomicAdd(&P.ctr->tail, (unsigned long long)nchild) : 0ull;
    if (own >= 0) atomicMax(&P.ctr->kept_ns, (unsigned long long)globaltimer_ns());
  }
  if (own >= 0) {
    // members in no child: a side that is too small, or no longer alive (of
    // those, the ones an earlier split published have another item's tag)
    for (int i = threadIdx.x; i < n; i += RB) {
      const int t = tag[i];
      if (t >= 0 && cnt[t] >= R.min_size) continue;
      unsigned long long *sl = &R.slot[m.gid[i]];
      if (t >= 0 || (uint32_t)(__ldcg(sl) >> 32) == queue_tag(seq)) *sl = ~0ull;
    }
  }
  __syncthreads();
  const unsigned long long s0 = sh.u0;
  // members in ascending local order, one warp, 32 at a time
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    for (int b = 0; b < n; b += 32) {
      int i = b + lane;
      int t = i < n ? tag[i] : -1;
      bool kept = t >= 0 && t != L && cnt[t] >= R.min_size;
      int key = kept ? t : -1;
      unsigned peers = __match_any_sync(FULL, key);
      int rank = __popc(peers & lanemask_lt());
      int before = kept ? run[t] : 0;
      __syncwarp();
      if (kept) {
        int pos = before + rank;
        int32_t v = m.gid[i];
        R.pool[vbeg + cbase[t] + pos] = v;
        R.slot[v] = ((unsigned long long)queue_tag(t == own ? seq : s0 + cidx[t]) << 32) | (unsigned)pos;
        if (rank == 0) run[t] = before + __popc(peers);
      }
      __syncwarp();
    }
  }
  __syncthreads();
  __threadfence();
  // descriptors, then publication
  for (int t = threadIdx.x; t < n; t += RB) {
    if (cnt[t] < R.min_size || t == L) continue;
    const Item child{vbeg + cbase[t], cnt[t], cflags, req};
    if (t == own) {
      sh.own = child;
      sh.has_own = 1;
    } else {
      P.ring[(s0 + cidx[t]) % P.ring_cap].item = child;
    }
  }
  __threadfence();
  __syncthreads();
  for (int t = threadIdx.x; t < n; t += RB) {
    if (cnt[t] < R.min_size || t == L || t == own) continue;
    unsigned long long q = s0 + cidx[t];
    atomicExch((unsigned long long *)&P.ring[q % P.ring_cap].seq, q);
  }
  __syncthreads();
  return L;
}

// CM (Algorithm 5): the two sides of a cut split (tag 0 / 1, -1 = not a
// member) with at least min_size members are written to the item's pool
// range in ascending local order, side 0 first, and listed in P.cda for the
// community step, which runs after the kernel; nothing is published.
template <typename IT>
__device__ __forceinline__ void park_sides(const RefineParams &P, const ReqCtx &R, uint16_t req,
                                           const Mem<IT> &m, const int32_t *tag, int n,
                                           int64_t vbeg, Sh &sh) {
  int a0 = 0, a1 = 0;
  for (int i = threadIdx.x; i < n; i += RB) {
    a0 += tag[i] == 0;
    a1 += tag[i] == 1;
  }
  const int c0 = block_sum_int(a0, sh);
  const int c1 = block_sum_int(a1, sh);
  const bool k0 = c0 >= R.min_size, k1 = c1 >= R.min_size;
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    const unsigned lt = lanemask_lt();
    int r0 = 0, r1 = 0;
    for (int b = 0; b < n; b += 32) {
      const int i = b + lane;
      const int t = i < n ? tag[i] : -1;
      const bool w0 = k0 && t == 0, w1 = k1 && t == 1;
      const unsigned m0 = __ballot_sync(FULL, w0), m1 = __ballot_sync(FULL, w1);
      if (w0) R.pool[vbeg + r0 + __popc(m0 & lt)] = m.gid[i];
      if (w1) R.pool[vbeg + (k0 ? c0 : 0) + r1 + __popc(m1 & lt)] = m.gid[i];
      r0 += __popc(m0);
      r1 += __popc(m1);
    }
  }
  if (threadIdx.x == 0 && (k0 || k1)) {
    const unsigned long long k = (k0 ? 1ull : 0ull) + (k1 ? 1ull : 0ull);
    unsigned long long at = atomicAdd(P.cda_count, k);
    if (at + k > P.cda_cap) {
      atomicOr(&P.ctr->error, DERR_CAPACITY);
    } else {
      if (k0) P.cda[at++] = Item{vbeg, c0, (uint16_t)0, req};
      if (k1) P.cda[at] = Item{vbeg + (k0 ? c0 : 0), c1, (uint16_t)0, req};
    }
  }
  __syncthreads();
}

// Continues an item in place as its child L (the component labelled L in
// tag): every other vertex becomes dead.  Returns the child's size.
template <typename IT>
__device__ __forceinline__ int restrict_alive(const Mem<IT> &m, const int32_t *tag, int L, int n,
                                              Sh &sh) {
  int c = 0;
  for (int i = threadIdx.x; i < n; i += RB) {
    const bool a = m.alive[i] && tag[i] == L;
    m.alive[i] = a;
    c += a;
  }
  return block_sum_int(c, sh);
}

// ---- maximum-adjacency machinery -----------------------------------------
// The current super-vertices are the ids X with grp[X] == X among alive
// vertices.  group_members() counts and lists their members: members of X
// are D[C[X] .. C[X+1]) (C indexed by id), and G[0..nsv) lists the
// super-vertices in ascending order.  Uses C, D, G, H; returns nsv.
template <typename IT>
__device__ __forceinline__ int group_members(const Mem<IT> &m, const int32_t *grp, int n, Sh &sh) {
  int32_t *gof = m.C, *mem = m.D, *svl = m.G, *tmp = m.H;
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i <= n; i += RB) gof[i] = 0;
  __syncthreads();
  // counts and slots are taken once per group present in a warp (large
  // super-vertices would otherwise serialise on one counter)
  for (int base = 0; base < n; base += RB) {
    const int i = base + threadIdx.x;
    const int g = (i < n && m.alive[i]) ? grp[i] : -1;
    const unsigned peers = __match_any_sync(FULL, g);
    if (g >= 0 && lane == __ffs(peers) - 1) atomicAdd(&gof[g], __popc(peers));
  }
  __syncthreads();
  block_scan_array(gof, n + 1, sh);
  for (int i = threadIdx.x; i < n; i += RB) tmp[i] = gof[i];
  __syncthreads();
  for (int base = 0; base < n; base += RB) {
    const int i = base + threadIdx.x;
    const int g = (i < n && m.alive[i]) ? grp[i] : -1;
    const unsigned peers = __match_any_sync(FULL, g);
    const int leader = __ffs(peers) - 1;
    int at = 0;
    if (g >= 0 && lane == leader) at = atomicAdd(&tmp[g], __popc(peers));
    at = __shfl_sync(FULL, at, leader);
    if (g >= 0) mem[at + __popc(peers & lanemask_lt())] = i;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += RB) tmp[i] = (m.alive[i] && grp[i] == i) ? 1 : 0;
  __syncthreads();
  const int nsv = block_scan_array(tmp, n, sh);
  for (int i = threadIdx.x; i < n; i += RB)
    if (m.alive[i] && grp[i] == i) svl[tmp[i]] = i;
  __syncthreads();
  return nsv;
}

__device__ __forceinline__ unsigned long long pack_key(int key, int id) {
  return ((unsigned long long)(unsigned)key << 32) | (unsigned)(~(unsigned)id);
}

// Adds the weights of super-vertex X's edges to every not-yet-added
// neighbour Y: acc[Y] += w(X, Y); each Y reached is listed once in touched.
// Warp 0 only.
template <typename IT>
__device__ __forceinline__ void scan_super_vertex(const Mem<IT> &m, const int32_t *grp, int X,
                                                  Sh &sh) {
  const int lane = threadIdx.x & 31;
  int32_t *acc = m.E, *touched = m.H;
  const int mb = m.C[X], me = m.C[X + 1];
  if (me - mb == 1) {
    const int i = m.D[mb];
    for (int e = m.off[i] + lane; e < m.end(i); e += 32) {
      const int j = m.adj[e];
      if (!m.alive[j]) continue;
      const int Y = grp[j];
      if (Y == X || m.flag[Y]) continue;
      if (atomicAdd(&acc[Y], 1) == 0) touched[atomicAdd(&sh.ntouched, 1)] = Y;
    }
  } else {
    for (int q = mb + lane; q < me; q += 32) {
      const int i = m.D[q];
      for (int e = m.off[i]; e < m.end(i); ++e) {
        const int j = m.adj[e];
        if (!m.alive[j]) continue;
        const int Y = grp[j];
        if (Y == X || m.flag[Y]) continue;
        if (atomicAdd(&acc[Y], 1) == 0) touched[atomicAdd(&sh.ntouched, 1)] = Y;
      }
    }
  }
}

// One Stoer-Wagner phase: a maximum-adjacency ordering over the current
// super-vertices with exact keys (ties to the smallest id) and a linear
// argmax, run by warp 0; reports the last two super-vertices s, t and the
// cut of the phase.  Needs group_members() and zeroed E (acc), F (key), flag.
// touched (H) is reused: the grouping's temporaries are dead by then.
template <typename IT>
__device__ __forceinline__ void ma_ordering(const Mem<IT> &m, const int32_t *grp, int nsv, Sh &sh) {
  int32_t *acc = m.E, *key = m.F, *touched = m.H, *svl = m.G;
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    int s = -1, t = -1, cut = 0;
    if (lane == 0) sh.ntouched = 0;
    __syncwarp();
    for (int step = 0; step < nsv; ++step) {
      unsigned long long best = 0;
      for (int j = lane; j < nsv; j += 32) {
        const int Y = svl[j];
        if (!m.flag[Y]) {
          const unsigned long long v = pack_key(key[Y], Y);
          best = v > best ? v : best;
        }
      }
      best = warp_max(best);
      const int X = (int)(~(unsigned)(best & 0xffffffffu));
      s = t;
      t = X;
      cut = (int)(best >> 32);
      if (lane == 0) m.flag[X] = 1;
      __syncwarp();
      if (step == nsv - 1) break;  // the last super-vertex has no unadded neighbour
      scan_super_vertex(m, grp, X, sh);
      __syncwarp();
      const int nt = sh.ntouched;
      for (int q = lane; q < nt; q += 32) {
        const int Y = touched[q];
        key[Y] += acc[Y];
        acc[Y] = 0;
      }
      __syncwarp();
      if (lane == 0) sh.ntouched = 0;
      __syncwarp();
    }
    if (lane == 0) {
      sh.sw_s = s;
      sh.sw_t = t;
      sh.sw_cut = cut;
    }
  }
  __syncthreads();
}

// ---- contraction passes --------------------------------------------------------
// A pass adds the super-vertices one by one, always one of largest capped key
// r(Y) = min(kcap, edges from Y to the added ones), ties to the smallest id,
// and merges X and Y whenever Y's key has reached kcap once X is scanned.
// What it merges does not depend on the order inside a run of picks at kcap:
//   - While some unadded key is at kcap, the next pick has key kcap.  Adding
//     such super-vertices only raises keys, so when none is left the added set
//     is the closure of the set before the run (every super-vertex that gets
//     kcap edges into it joins), whatever order they were taken in; the keys
//     of the others count their edges into that set, so the next pick, of
//     largest key below kcap and smallest id, is the same too.
//   - Call such a pick s and the closure after it C.  A key that reached kcap
//     in C did so by a scan of s or of another member of C (it was below kcap
//     before s), and merged with it: by induction {s} + C is one merged set.
//     A merge of X and Y needs Y unadded at kcap when X is scanned, and all
//     unadded keys were below kcap before s: X and Y are in the same phase.
// So the sets a pass merges are exactly its phases {s} + C, and each closure
// can be grown by the whole block at once, a breadth-first search over the
// super-vertices at kcap.  A pass is then a dozen to forty short rounds (23 on
// a 50,000-vertex cluster of mean degree 36, 36 on one of 1,900 vertices)
// instead of one dependent step a vertex, which took about 490 cycles in
// shared memory and 1,800 in the global slab.  Measured on whole runs, graph
// resident: clusters of up to 50,000 vertices (1M vertices, 20M edges) 64.9 ->
// 26.7 ms, LFR-style 100k 1.19 -> 0.78 ms, its CM 2.97 -> 2.43 ms.
constexpr unsigned KEY_IN = 0x8000u;    // added, or queued to be
constexpr unsigned KEY_DEAD = 0x4000u;  // peeled: never below kcap, never added
constexpr int KEY_MAX = 0x3fff;         // largest kcap the 16-bit keys hold
// A round looks from the unadded vertices' side when the vertices added in
// the round before are at least as many: the last rounds add most of the
// vertices at once, and an unadded one stops at kcap added neighbours, most
// often within its first 32 entries.
constexpr int PULL_MIN = 64;
constexpr int PULL_STEP = 32;
// Picks of an item with 32-bit local ids (65,535 vertices or more) go by groups
// of 64 vertices, each with its best key: after the usual small round only the
// groups of the vertices it touched are looked through again (after at most
// PICK_ROUNDS rounds of at most RW rows of at most PICK_ROW entries, else all).
// With all keys looked through for every pick the passes of one random cluster
// of mean degree 12 grow with the square of its size: whole runs at 66,000 /
// 200,000 / 500,000 vertices take 81 / 1,285 / 7,149 ms, by groups 42 / 287 / 869.
// Below 65,535 vertices the keys are in shared memory and a look at all of them
// is at most 64 words a thread.
constexpr int PICK_GROUP = 64;
constexpr int PICK_ROUNDS = 8;
constexpr int PICK_ROW = 256;
static_assert(PICK_ROUNDS * RW * PICK_ROW + PICK_ROUNDS + 1 <= 65535 - 65535 / PICK_GROUP,
              "a phase's touched groups fit the array beside the groups' best keys");

// The entries of up to 32 rows, lane r holding row r = adj[b .. b + d), walked
// by one warp as one flat range.  Calls fn(j, base) for every 128 entries:
// j[z] the lane's entry base + 32 z + lane (-1: none); the lane's own row is
// the range [exc, exc + d) of them.  Every lane calls.
template <typename IT, typename Fn>
__device__ __forceinline__ void flat_rows(const IT *adj, int b, int d, int &exc, Fn fn) {
  const int lane = threadIdx.x & 31;
  const int inc = warp_inclusive_scan(d);
  exc = inc - d;
  const int total = __shfl_sync(FULL, inc, 31), g = b - exc;
  for (int f0 = 0; f0 < total; f0 += 128) {
    int j[4], lo[4] = {0, 0, 0, 0};  // lo: rows that end at or before the entry
#pragma unroll
    for (int st = 16; st > 0; st >>= 1)
#pragma unroll
      for (int z = 0; z < 4; ++z)
        if (__shfl_sync(FULL, inc, lo[z] + st - 1) <= f0 + 32 * z + lane) lo[z] += st;
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      const int f = f0 + 32 * z + lane;
      const int gr = __shfl_sync(FULL, g, lo[z]);
      j[z] = f < total ? (int)adj[gr + f] : -1;
    }
    fn(j, f0);
  }
}

// The same for a single row adj[b .. b + d).
template <typename IT, typename Fn>
__device__ __forceinline__ void one_row(const IT *adj, int b, int d, Fn fn) {
  const int lane = threadIdx.x & 31;
  for (int f0 = 0; f0 < d; f0 += 128) {
    int j[4];
#pragma unroll
    for (int z = 0; z < 4; ++z) {
      const int f = f0 + 32 * z + lane;
      j[z] = f < d ? (int)adj[b + f] : -1;
    }
    fn(j, f0);
  }
}

// Block maximum of a 32- or 64-bit value; every thread returns it.  Two
// calls need a barrier between them.
__device__ __forceinline__ unsigned block_best(unsigned v, Sh &sh) {
  v = __reduce_max_sync(FULL, v);
  if ((threadIdx.x & 31) == 0) sh.wbest[threadIdx.x >> 5] = v;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  return __reduce_max_sync(FULL, lane < RW ? (unsigned)sh.wbest[lane] : 0u);
}
__device__ __forceinline__ unsigned long long block_best(unsigned long long v, Sh &sh) {
  v = warp_max(v);
  if ((threadIdx.x & 31) == 0) sh.wbest[threadIdx.x >> 5] = v;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  return warp_max(lane < RW ? sh.wbest[lane] : 0ull);
}

// Appends the lanes' vertices with take set to queue at base + *cnt.
__device__ __forceinline__ int warp_push(bool take, int32_t v, int32_t *queue, int base,
                                         int32_t *cnt) {
  const unsigned b = __ballot_sync(FULL, take);
  if (b == 0u) return 0;
  const int lane = threadIdx.x & 31, leader = __ffs(b) - 1;
  int at = 0;
  if (lane == leader) at = atomicAdd(cnt, __popc(b));
  at = __shfl_sync(FULL, at, leader);
  if (take) queue[base + at + __popc(b & lanemask_lt())] = v;
  return __popc(b);
}

// The same for up to four vertices a lane, with one atomic.
__device__ __forceinline__ void warp_push4(const bool (&take)[4], const int (&v)[4],
                                           int32_t *queue, int base, int32_t *cnt) {
  unsigned b[4];
  int k = 0;
#pragma unroll
  for (int z = 0; z < 4; ++z) {
    b[z] = __ballot_sync(FULL, take[z]);
    k += __popc(b[z]);
  }
  if (k == 0) return;
  int at = 0;
  if ((threadIdx.x & 31) == 0) at = atomicAdd(cnt, k);
  at = base + __shfl_sync(FULL, at, 0);
#pragma unroll
  for (int z = 0; z < 4; ++z) {
    if (take[z]) queue[at + __popc(b[z] & lanemask_lt())] = v[z];
    at += __popc(b[z]);
  }
}

// The first contraction pass, on the item's own vertices (every super-vertex
// a single vertex, every edge weight 1).  Returns the number of phases (1:
// everything merged; nalive: nothing did; -1 after an error) and of
// components.  rep[i] (B or A) = the smallest member of i's phase, -1 if
// dead; the vertices in the order they were added are left in D.  A first
// vertex of key 0 starts another component (every vertex of the one before
// has been added); with more than one, H[i] = the smallest member of i's
// component, -1 if dead; past MAX_COMP the pass gives up (-2).  With kcap = 1
// the phases are the components; a pass run for them alone (ccr: rep is B)
// gives up on long thin items too.  Uses C, D, F, G, H and the keys.  Keys are
// 16 bits: several threads may raise one vertex past kcap, each by up to the four
// entries it has in flight, which stays below KEY_IN and so out of the other
// half-word.
static_assert(KEY_MAX + 4 * RB < (int)KEY_IN, "a key raised past the cap keeps to its half-word");
template <typename IT, bool SM>
__device__ __noinline__ int2 first_pass(const Mem<IT> *m0, int64_t d, bool ccr, int n, int nalive,
                                        int kcap, unsigned *err, Sh *shp) {
  Sh &sh = *shp;
  const Mem<IT> m = item_mem<IT, SM>(m0, n, d);
  int32_t *rep = ccr ? m.B : m.A;
  uint32_t *kw = m.kw;
  volatile uint16_t *kh = reinterpret_cast<volatile uint16_t *>(m.kw);
  int32_t *queue = m.D, *phmin = m.C, *lr = m.G;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nw = (n + 1) >> 1;
  for (int w = threadIdx.x; w < nw; w += RB) {
    const int i = 2 * w;
    const unsigned lo = m.alive[i] ? 0u : KEY_DEAD;
    const unsigned hi = (i + 1 < n && m.alive[i + 1]) ? 0u : KEY_DEAD;
    kw[w] = lo | (hi << 16);
  }
  for (int i = threadIdx.x; i < n; i += RB) rep[i] = -1;
  if (threadIdx.x < 3) sh.qn[threadIdx.x] = 0;
  if (threadIdx.x == 0) sh.ntouched = sh.ngrp = sh.grp_all = 0;
  int tail = 0, phases = 0, r = 0, rounds = 0, comps = 0, comp = -1;
  // 32-bit local ids: every group's best key ((key << 6 | 63 - place) + 1, 0:
  // none), then the list of groups touched since the last pick
  constexpr bool GROUPS = sizeof(IT) == 4;
  const int ng = (n + PICK_GROUP - 1) / PICK_GROUP;
  unsigned *gbest = reinterpret_cast<unsigned *>(m.H);
  int32_t *glist = m.H + ng;
  bool gall = true;  // all groups are to be looked through
  int marked = 0;    // rounds since the last pick
  __syncthreads();
  while (tail < nalive) {
    // the phase's first vertex: largest key, then smallest id
    int X;
    bool fresh;  // its key is 0
    if (sizeof(IT) == 2) {
      unsigned best = 0u;
      for (int w = threadIdx.x; w < nw; w += RB) {
        const uint32_t k2 = kw[w];
        const unsigned lo = k2 & 0xffffu, hi = k2 >> 16;
        if (lo < (unsigned)kcap) best = max(best, (lo << 16) | (0xffffu - (unsigned)(2 * w)));
        if (hi < (unsigned)kcap) best = max(best, (hi << 16) | (0xfffeu - (unsigned)(2 * w)));
      }
      best = block_best(best, sh);
      X = best ? (int)(0xffffu - (best & 0xffffu)) : -1;
      fresh = (best >> 16) == 0u;
    } else {
      gall = gall || sh.grp_all != 0;
      auto look = [&](int g, uint32_t k2) {  // group g's best key from its words, one a lane
        const unsigned lo = k2 & 0xffffu, hi = k2 >> 16;
        unsigned b = lo < (unsigned)kcap ? ((lo << 6) | (unsigned)(63 - 2 * lane)) + 1u : 0u;
        if (hi < (unsigned)kcap) b = max(b, ((hi << 6) | (unsigned)(62 - 2 * lane)) + 1u);
        b = __reduce_max_sync(FULL, b);
        if (lane == 0) gbest[g] = b;
      };
      auto words = [&](int g) {  // (no key below kcap past the end)
        const int w = g * (PICK_GROUP / 2) + lane;
        return w < nw ? kw[w] : FULL;
      };
      if (gall) {
        for (int g0 = warp; g0 < ng; g0 += 8 * RW) {  // eight groups in flight
          uint32_t k2[8];
#pragma unroll
          for (int z = 0; z < 8; ++z) k2[z] = words(g0 + z * RW);
#pragma unroll
          for (int z = 0; z < 8; ++z)
            if (g0 + z * RW < ng) look(g0 + z * RW, k2[z]);
        }
      } else {
        const int nd = sh.ngrp;
        for (int k = warp; k < nd; k += RW) look(glist[k], words(glist[k]));
      }
      __syncthreads();
      if (threadIdx.x == 0) sh.ngrp = sh.grp_all = 0;
      gall = false;
      marked = 0;
      unsigned long long best = 0ull;
      for (int g = threadIdx.x; g < ng; g += RB) {
        const unsigned b = gbest[g];
        if (b == 0u) continue;
        const unsigned id = (unsigned)(g * PICK_GROUP + 63) - ((b - 1u) & 63u);
        best = max(best, ((unsigned long long)((b - 1u) >> 6) << 32) | (unsigned)~id);
      }
      best = block_best(best, sh);
      X = best ? (int)~(unsigned)best : -1;
      fresh = (best >> 32) == 0ull;
    }
    if (X < 0 || X >= n) {  // cannot happen: an unadded vertex has a key below kcap here
      if (threadIdx.x == 0) atomicOr(err, DERR_INTERNAL);
      return make_int2(-1, 0);
    }
    if (fresh) {
      comp = X;
      if (++comps > MAX_COMP) return make_int2(-2, 0);
    }
    if (threadIdx.x == 0) {
      queue[tail] = X;
      rep[X] = phases;
      phmin[phases] = X;
      m.F[phases] = comp;
      kh[X] = (uint16_t)KEY_IN;
      if (GROUPS) glist[sh.ngrp++] = X / PICK_GROUP;
    }
    int head = tail++;
    __syncthreads();
    while (head < tail && tail < nalive) {
      if (ccr && rounds >= THIN_ROUNDS && tail < THIN_FRONT * rounds) return make_int2(-2, 0);
      const int F = tail - head, U = nalive - tail;
      int32_t *qn = &sh.qn[r];
      const int rn = r == 2 ? 0 : r + 1;
      if (threadIdx.x == 0) sh.qn[rn] = 0;
      if (GROUPS && (F > RW || ++marked > PICK_ROUNDS)) gall = true;
      if (F >= PULL_MIN && F >= U) {
        // every unadded vertex counts its added neighbours afresh; those it
        // takes are marked only after the round, so that the keys of the
        // rest are exact
        for (int i0 = 0; i0 < n; i0 += RB) {
          const int i = i0 + threadIdx.x;
          warp_push(i < n && kh[i] < kcap, i, lr, 0, &sh.ntouched);
        }
        __syncthreads();
        const int nl = sh.ntouched;
        const int per = min(32, (nl + RW - 1) / RW);
        for (int c0 = warp * per; c0 < nl; c0 += RW * per) {
          int i = -1, b = 0, left = 0, c = 0;
          if (lane < min(per, nl - c0)) {
            i = lr[c0 + lane];
            b = m.off[i];
            left = (int)m.len[i];
          }
          for (int st = PULL_STEP; __any_sync(FULL, left > 0); st *= 2) {
            const int d = min(left, st);
            int exc;
            flat_rows(m.adj, b, d, exc, [&](const int (&j)[4], int f0) {
              unsigned k[4];
#pragma unroll
              for (int z = 0; z < 4; ++z) k[z] = j[z] >= 0 ? kh[j[z]] : 0u;
#pragma unroll
              for (int z = 0; z < 4; ++z) {
                // hits within the lane's row
                const int lo = min(max(exc - f0 - 32 * z, 0), 32);
                const int hi = min(max(exc + d - f0 - 32 * z, 0), 32);
                const unsigned mine = (unsigned)((1ull << hi) - (1ull << lo));
                c += __popc(__ballot_sync(FULL, (k[z] & KEY_IN) != 0u) & mine);
              }
            });
            b += d;
            left = c >= kcap ? 0 : left - d;
          }
          const bool take = c >= kcap;
          if (i >= 0) {
            kh[i] = (uint16_t)(take ? KEY_DEAD : (unsigned)c);
            if (take) rep[i] = phases;
          }
          warp_push(take, i, queue, tail, qn);
        }
        __syncthreads();
        for (int q = threadIdx.x; q < *(volatile int32_t *)qn; q += RB)
          kh[queue[tail + q]] = (uint16_t)KEY_IN;
        if (threadIdx.x == 0) sh.ntouched = 0;
      } else {
        // the vertices added last raise their neighbours' keys; loads and
        // atomics of four entries a lane overlap
        bool mark = false;  // the groups of the vertices raised are listed
        auto raise = [&](const int (&j)[4], int) {
          unsigned k[4], old[4];
          bool take[4];
#pragma unroll
          for (int z = 0; z < 4; ++z) k[z] = j[z] >= 0 ? kh[j[z]] : KEY_DEAD;
#pragma unroll
          for (int z = 0; z < 4; ++z)
            old[z] = k[z] < (unsigned)kcap ? atomicAdd(&kw[j[z] >> 1], 1u << ((j[z] & 1) * 16)) : 0u;
#pragma unroll
          for (int z = 0; z < 4; ++z) {
            take[z] = k[z] < (unsigned)kcap &&
                      ((old[z] >> ((j[z] & 1) * 16)) & 0xffffu) + 1u == (unsigned)kcap;
            if (take[z]) {
              atomicOr(&kw[j[z] >> 1], KEY_IN << ((j[z] & 1) * 16));
              rep[j[z]] = phases;
            }
          }
          warp_push4(take, j, queue, tail, qn);
          if (GROUPS && mark) {
            bool up[4];
            int g[4];
#pragma unroll
            for (int z = 0; z < 4; ++z) {
              up[z] = k[z] < (unsigned)kcap;
              g[z] = j[z] / PICK_GROUP;
            }
            warp_push4(up, g, glist, 0, &sh.ngrp);
          }
        };
        if (F <= RW) {
          if (warp < F) {
            const int v = queue[head + warp], d = (int)m.len[v];
            if (GROUPS) {
              mark = !gall && d <= PICK_ROW;
              if (!mark && lane == 0) sh.grp_all = 1;
            }
            one_row(m.adj, m.off[v], d, raise);
          }
        } else {
          const int per = min(32, (F + RW - 1) / RW);
          for (int c0 = head + warp * per; c0 < tail; c0 += RW * per) {
            int b = 0, d = 0, exc;
            if (lane < min(per, tail - c0)) {
              const int v = queue[c0 + lane];
              b = m.off[v];
              d = (int)m.len[v];
            }
            flat_rows(m.adj, b, d, exc, raise);
          }
        }
      }
      __syncthreads();
      head = tail;
      tail += *(volatile int32_t *)qn;
      r = rn;
      ++rounds;
    }
    ++phases;
  }
  if (threadIdx.x == 0) {
    sh.dbg[1] = rounds;
    sh.dbg[2] = phases;
  }
  // the phases' smallest members, one atomic per phase and warp (ids ascend
  // with the lanes, so a phase's first lane holds its smallest)
  __syncthreads();
  if (phases > 1) {
    for (int i0 = 0; i0 < n; i0 += RB) {
      const int i = i0 + threadIdx.x;
      const int p = i < n ? rep[i] : -1;
      const unsigned peers = __match_any_sync(FULL, p);
      if (p >= 0 && (peers & lanemask_lt()) == 0u) atomicMin(&phmin[p], i);
    }
    __syncthreads();
  }
  for (int i = threadIdx.x; i < n; i += RB) {
    const int p = rep[i];
    if (comps > 1) m.H[i] = p >= 0 ? m.F[p] : -1;
    if (p >= 0) rep[i] = phmin[p];
  }
  __syncthreads();
  return make_int2(phases, comps);
}

// A later pass, on super-vertices with members (rep[i], in A, = the smallest
// member of i's set): the same phases, keys counting the edges of all
// members.  Returns the number of phases (-1 after an error) and moves rep
// to their sets.  Uses B, C, D, E, F, G, H.
template <typename IT, bool SM>
__device__ __noinline__ int class_pass(const Mem<IT> *m0, int64_t d, int n, int kcap,
                                       unsigned *err, Sh *shp) {
  Sh &sh = *shp;
  const Mem<IT> m = item_mem<IT, SM>(m0, n, d);
  int32_t *rep = m.A;
  const int nsv = group_members(m, rep, n, sh);
  constexpr unsigned IN = 0x80000000u;
  unsigned *key = reinterpret_cast<unsigned *>(m.F);
  volatile unsigned *vkey = key;
  int32_t *svl = m.G, *ph = m.E, *queue = m.H, *phmin = m.B;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int k = threadIdx.x; k < nsv; k += RB) key[svl[k]] = 0u;
  if (threadIdx.x < 3) sh.qn[threadIdx.x] = 0;
  int tail = 0, phases = 0, r = 0;
  __syncthreads();
  while (tail < nsv) {
    unsigned long long best = 0ull;
    for (int k = threadIdx.x; k < nsv; k += RB) {
      const int Y = svl[k];
      if (key[Y] < (unsigned)kcap) best = max(best, pack_key((int)key[Y], Y));
    }
    best = block_best(best, sh);
    if (best == 0ull) {  // cannot happen: an unadded super-vertex has a key below kcap here
      if (threadIdx.x == 0) atomicOr(err, DERR_INTERNAL);
      return -1;
    }
    const int X = (int)(~(unsigned)(best & 0xffffffffu));
    if (threadIdx.x == 0) {
      queue[tail] = X;
      ph[X] = phases;
      phmin[phases] = X;
      key[X] = IN;
    }
    int head = tail++;
    __syncthreads();
    while (head < tail && tail < nsv) {
      int32_t *qn = &sh.qn[r];
      const int rn = r == 2 ? 0 : r + 1;
      if (threadIdx.x == 0) sh.qn[rn] = 0;
      auto scan_row = [&](int i) {  // one member's row, by a warp
        const int b = m.off[i], e = m.end(i);
        for (int q0 = b; q0 < e; q0 += 32) {
          bool take = false;
          int Y = -1;
          if (q0 + lane < e) {
            Y = rep[(int)m.adj[q0 + lane]];
            if (Y >= 0 && vkey[Y] < (unsigned)kcap) {
              take = atomicAdd(&key[Y], 1u) + 1u == (unsigned)kcap;
              if (take) {
                atomicOr(&key[Y], IN);
                ph[Y] = phases;
              }
            }
          }
          warp_push(take, Y, queue, tail, qn);
        }
      };
      for (int f = head; f < tail; ++f) {
        const int Xf = queue[f], mb = m.C[Xf], me = m.C[Xf + 1];
        if (me - mb < RW) {  // few members: one warp, the next super-vertex on the next one
          if ((f - head) % RW == warp)
            for (int q = mb; q < me; ++q) scan_row(m.D[q]);
        } else {
          for (int q = mb + warp; q < me; q += RW) scan_row(m.D[q]);
        }
      }
      __syncthreads();
      head = tail;
      tail += *(volatile int32_t *)qn;
      r = rn;
    }
    ++phases;
  }
  for (int k = threadIdx.x; k < nsv; k += RB) atomicMin(&phmin[ph[svl[k]]], svl[k]);
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += RB)
    if (rep[i] >= 0) rep[i] = phmin[ph[rep[i]]];
  __syncthreads();
  return phases;
}

// The ordering of ma_ordering() with the whole block scanning each added
// super-vertex: for a few large super-vertices (after the contraction passes
// merged most edges), where one warp walking thousands of member rows would
// dominate.  Warp 0 picks
// (linear argmax, ties to the smallest id); same contract as ma_ordering().
constexpr int BLOCK_NSV = 64;  // at most this many super-vertices

template <typename IT>
__device__ __forceinline__ void ma_ordering_block(const Mem<IT> &m, const int32_t *grp, int nsv,
                                                  Sh &sh) {
  int32_t *acc = m.E, *key = m.F, *touched = m.H, *svl = m.G;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int s = -1, t = -1, cut = 0;
  if (threadIdx.x == 0) sh.ntouched = 0;
  for (int step = 0; step < nsv; ++step) {
    if (warp == 0) {
      unsigned long long best = 0;
      for (int j = lane; j < nsv; j += 32) {
        const int Y = svl[j];
        if (!m.flag[Y]) {
          const unsigned long long v = pack_key(key[Y], Y);
          best = v > best ? v : best;
        }
      }
      best = warp_max(best);
      if (lane == 0) {
        const int X = (int)(~(unsigned)(best & 0xffffffffu));
        m.flag[X] = 1;
        sh.sw_x = X;
        sh.sw_key = (int)(best >> 32);
      }
    }
    __syncthreads();
    const int X = sh.sw_x;
    s = t;
    t = X;
    cut = sh.sw_key;
    if (step == nsv - 1) break;  // the last super-vertex has no unadded neighbour
    const int mb = m.C[X], me = m.C[X + 1];
    auto visit = [&](int e) {
      const int j = m.adj[e];
      if (!m.alive[j]) return;
      const int Y = grp[j];
      if (Y == X || m.flag[Y]) return;
      if (atomicAdd(&acc[Y], 1) == 0) touched[atomicAdd(&sh.ntouched, 1)] = Y;
    };
    if (me - mb <= RW) {
      // few members: a warp per member, lanes along its row
      for (int q = mb + warp; q < me; q += RW) {
        const int i = m.D[q];
        for (int e = m.off[i] + lane; e < m.end(i); e += 32) visit(e);
      }
    } else {
      for (int q = mb + threadIdx.x; q < me; q += RB) {
        const int i = m.D[q];
        for (int e = m.off[i]; e < m.end(i); ++e) visit(e);
      }
    }
    __syncthreads();
    const int nt = sh.ntouched;
    for (int q = threadIdx.x; q < nt; q += RB) {
      const int Y = touched[q];
      key[Y] += acc[Y];
      acc[Y] = 0;
    }
    __syncthreads();
    if (threadIdx.x == 0) sh.ntouched = 0;  // ordered before the next scan by the pick's barrier
  }
  if (threadIdx.x == 0) {
    sh.sw_s = s;
    sh.sw_t = t;
    sh.sw_cut = cut;
  }
  __syncthreads();
}

template <typename IT>
__device__ __forceinline__ void reset_ma_state(const Mem<IT> &m, int n) {
  for (int i = threadIdx.x; i < n; i += RB) {
    m.E[i] = 0;
    m.F[i] = 0;
    m.flag[i] = 0;
  }
  __syncthreads();
}

// Canonical Stoer-Wagner over the sets grp (in A), phase by phase: the first
// smallest cut of a phase, its side in m.side; *phases counts them.
template <typename IT, bool SM>
__device__ __noinline__ int sparse_cut(const Mem<IT> *m0, int64_t d, int n, int nsv,
                                       long long *phases, Sh *shp) {
  Sh &sh = *shp;
  const Mem<IT> m = item_mem<IT, SM>(m0, n, d);
  int32_t *grp = m.A;
  int best = 0x7fffffff;
  while (nsv > 1) {
    group_members(m, grp, n, sh);
    reset_ma_state(m, n);
    if (threadIdx.x == 0) add_ll(phases, 1ll);
    if (nsv <= BLOCK_NSV)
      ma_ordering_block(m, grp, nsv, sh);
    else
      ma_ordering(m, grp, nsv, sh);
    const int s = sh.sw_s, t = sh.sw_t, cut = sh.sw_cut;
    if (cut < best) {
      best = cut;
      for (int i = threadIdx.x; i < n; i += RB) m.side[i] = m.alive[i] && grp[i] == t;
    }
    __syncthreads();
    const int lo = s < t ? s : t, hi = s < t ? t : s;
    for (int i = threadIdx.x; i < n; i += RB)
      if (m.alive[i] && grp[i] == hi) grp[i] = lo;
    __syncthreads();
    --nsv;
  }
  return best;
}

// ---- few super-vertices: a dense finish ---------------------------------------
// With at most 128 super-vertices left (indexed in ascending order of their
// smallest member, so index order is id order), their integer edge weights
// fit a small matrix w[nsv][nsv] and one warp runs the remaining capped
// contraction passes and the Stoer-Wagner phases on it, lane l holding
// super-vertices l, l + 32, ... (K of them), with exactly the rules of the
// sparse passes: largest key, ties to the smallest id; a capped pass merges
// its phases (see "contraction passes"; survivor: the smallest id); a
// Stoer-Wagner phase's cut is the key of the last super-vertex t, the earliest
// minimum is kept, its side is t's members, and t merges into the one added
// before it.  Sets of indices are bit masks, bit l of word j = index l + 32 j,
// the same in every lane.  (With a capped pass as an ordering, one pick and
// its union-find links a super-vertex, 67 of them took 1,500 cycles a pick and
// the dense finish 0.29M of an item's 0.71M cycles; as phases it takes 0.09M.)
constexpr int DENSE_NSV = 128;

template <int K>
struct Mask {
  uint32_t w[K];
  __device__ __forceinline__ bool any() const {
    uint32_t r = 0u;
#pragma unroll
    for (int j = 0; j < K; ++j) r |= w[j];
    return r != 0u;
  }
  __device__ __forceinline__ int count() const {
    int r = 0;
#pragma unroll
    for (int j = 0; j < K; ++j) r += __popc(w[j]);
    return r;
  }
  __device__ __forceinline__ int first() const {  // -1: none
    int r = -1;
#pragma unroll
    for (int j = K - 1; j >= 0; --j) r = w[j] ? 32 * j + __ffs(w[j]) - 1 : r;
    return r;
  }
  __device__ __forceinline__ void clear(int x) {
#pragma unroll
    for (int j = 0; j < K; ++j) w[j] &= (x >> 5) == j ? ~(1u << (x & 31)) : FULL;
  }
  __device__ __forceinline__ bool mine(int j) const { return (w[j] >> (threadIdx.x & 31)) & 1u; }
};

// Folds the rows and columns of the indices in C into its first one's, zeroes
// that one's diagonal and takes the others out of live.  One warp.
template <int K>
__device__ __forceinline__ void dense_fold(int32_t *w, int nsv, Mask<K> C, Mask<K> &live) {
  const int l = threadIdx.x & 31, r = C.first();
  C.clear(r);
  int32_t sum[K];
#pragma unroll
  for (int j = 0; j < K; ++j) sum[j] = 0;
  for (Mask<K> c = C; c.any();) {
    const int x = c.first();
    c.clear(x);
#pragma unroll
    for (int j = 0; j < K; ++j)
      if (l + 32 * j < nsv) sum[j] += w[x * nsv + l + 32 * j];
  }
#pragma unroll
  for (int j = 0; j < K; ++j) {
    if (l + 32 * j < nsv) w[r * nsv + l + 32 * j] += sum[j];
    sum[j] = 0;
  }
  __syncwarp();
  for (Mask<K> c = C; c.any();) {
    const int x = c.first();
    c.clear(x);
#pragma unroll
    for (int j = 0; j < K; ++j)
      if (l + 32 * j < nsv) sum[j] += w[(l + 32 * j) * nsv + x];
  }
#pragma unroll
  for (int j = 0; j < K; ++j) {
    if (l + 32 * j < nsv) w[(l + 32 * j) * nsv + r] += sum[j];
    live.w[j] &= ~C.w[j];
  }
  __syncwarp();
  if (l == 0) w[r * nsv + r] = 0;
  __syncwarp();
}

// The index in left of largest key, ties to the smallest.
template <int K>
__device__ __forceinline__ int dense_pick(const unsigned (&key)[K], const Mask<K> &left,
                                          unsigned &top) {
  unsigned best = 0u;
#pragma unroll
  for (int j = 0; j < K; ++j) best = max(best, left.mine(j) ? key[j] : 0u);
  top = __reduce_max_sync(FULL, best);
  Mask<K> m;
#pragma unroll
  for (int j = 0; j < K; ++j) m.w[j] = __ballot_sync(FULL, left.mine(j) && key[j] == top);
  return m.first();
}

struct DenseResult {
  int cut;        // minimum cut, or -1 when the contraction left one super-vertex
  uint32_t side[DENSE_NSV / 32];  // the minimum cut's side (mask of initial indices)
  int passes, phases;
};

// Runs the dense finish on w (nsv <= 32 K indices) with one warp (any warp;
// all its lanes call).  grp: nsv ints of scratch.  Every lane returns the
// result (side: K words).
template <int K>
__device__ __forceinline__ DenseResult dense_finish(int32_t *w, int nsv, int kcap, int32_t *grp) {
  const int l = threadIdx.x & 31;
  Mask<K> live;
#pragma unroll
  for (int j = 0; j < K; ++j) {
    const int b = 32 * j;
    live.w[j] = nsv >= b + 32 ? FULL : (nsv > b ? (1u << (nsv - b)) - 1u : 0u);
    // grp[initial index] = the index that holds it now
    if (l + b < nsv) grp[l + b] = l + b;
  }
  __syncwarp();
  DenseResult res;
  res.cut = -1;
  res.passes = res.phases = 0;
#pragma unroll
  for (int j = 0; j < K; ++j) res.side[j] = 0u;
  // moves the members of every index in C to its first one
  auto regroup = [&](const Mask<K> &C) {
    const int r = C.first();
#pragma unroll
    for (int j = 0; j < K; ++j)
      if (l + 32 * j < nsv) {
        const int g = grp[l + 32 * j];
        bool in = false;
#pragma unroll
        for (int i = 0; i < K; ++i) in |= (g >> 5) == i && ((C.w[i] >> (g & 31)) & 1u);
        if (in) grp[l + 32 * j] = r;
      }
  };
  while (live.count() > 1) {
    unsigned key[K];
#pragma unroll
    for (int j = 0; j < K; ++j) key[j] = 0u;
    Mask<K> left = live;
    const Mask<K> start = live;
    bool merged = false;
    ++res.passes;
    // the pass reads the matrix as it was: its phases are folded after it
    while (left.any()) {
      unsigned top;
      const int X = dense_pick<K>(key, left, top);
      Mask<K> C, todo;
#pragma unroll
      for (int j = 0; j < K; ++j) C.w[j] = todo.w[j] = (X >> 5) == j ? 1u << (X & 31) : 0u;
      left.clear(X);
      while (todo.any() && left.any()) {
        const int x = todo.first();
        todo.clear(x);
#pragma unroll
        for (int j = 0; j < K; ++j) {
          if (left.mine(j)) key[j] += (unsigned)w[x * nsv + l + 32 * j];
          const unsigned sat = __ballot_sync(FULL, left.mine(j) && key[j] >= (unsigned)kcap);
          C.w[j] |= sat;
          todo.w[j] |= sat;
          left.w[j] &= ~sat;
        }
      }
      // members point to their phase's smallest through grp, where only an
      // index's own entry (grp[x] for live x) is read back below
      if (C.count() > 1) {
        merged = true;
        regroup(C);
        __syncwarp();
      }
    }
    if (!merged) break;
    // fold every phase: the live indices by the index that holds them now
    Mask<K> rest = start;
    while (rest.any()) {
      const int r = rest.first();
      const int g = grp[r];
      Mask<K> C;
#pragma unroll
      for (int j = 0; j < K; ++j) {
        const bool in = rest.mine(j) && grp[l + 32 * j] == g;
        C.w[j] = __ballot_sync(FULL, in);
        rest.w[j] &= ~C.w[j];
      }
      if (C.count() > 1) dense_fold<K>(w, nsv, C, live);
    }
  }
  while (live.count() > 1) {
    unsigned key[K], cut = 0u;
#pragma unroll
    for (int j = 0; j < K; ++j) key[j] = 0u;
    Mask<K> left = live;
    int s = -1, t = -1;
    while (left.any()) {
      const int X = dense_pick<K>(key, left, cut);
      s = t;
      t = X;
      left.clear(X);
#pragma unroll
      for (int j = 0; j < K; ++j)
        if (left.mine(j)) key[j] += (unsigned)w[X * nsv + l + 32 * j];
    }
    ++res.phases;
    if (res.cut < 0 || (int)cut < res.cut) {
      res.cut = (int)cut;
#pragma unroll
      for (int j = 0; j < K; ++j)
        res.side[j] = __ballot_sync(FULL, l + 32 * j < nsv && grp[l + 32 * j] == t);
    }
    Mask<K> C;
#pragma unroll
    for (int j = 0; j < K; ++j)
      C.w[j] = ((s >> 5) == j ? 1u << (s & 31) : 0u) | ((t >> 5) == j ? 1u << (t & 31) : 0u);
    regroup(C);
    __syncwarp();
    dense_fold<K>(w, nsv, C, live);
  }
  __syncwarp();
  return res;
}

// The dense finish of a CTA's item, by its first warp; w: nsv x nsv weights.
// The result and the cut's side are left in sh for the other warps.
template <int K>
__device__ __forceinline__ void dense_cta_k(int32_t *w, int nsv, int kcap, Sh &sh) {
  const DenseResult dr = dense_finish<K>(w, nsv, kcap, sh.wgrp);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int j = 0; j < K; ++j) sh.wside[j] = dr.side[j];
    sh.dcut = dr.cut;
    sh.dpasses = dr.passes;
    sh.dphases = dr.phases;
  }
}
__device__ __noinline__ void dense_cta(int32_t *w, int nsv, int kcap, Sh *shp) {
  if (nsv <= 32)
    dense_cta_k<1>(w, nsv, kcap, *shp);
  else if (nsv <= 64)
    dense_cta_k<2>(w, nsv, kcap, *shp);
  else
    dense_cta_k<4>(w, nsv, kcap, *shp);
}

// Exact acceptance test for lambda >= kcap by forest certificates.  Take
// kcap-1 edge-disjoint spanning forests, each maximal in the edges the earlier
// ones left.  An edge (u, v) in none of them has u and v joined by a path in
// every forest (else that forest could have taken it) and by itself: kcap
// edge-disjoint paths, so lambda(u, v) >= kcap and contracting u, v keeps
// every cut below kcap (the sparse-certificate argument of Nagamochi and
// Ibaraki).  Rounds repeat on the contracted multigraph (a super-vertex is
// labelled by its smallest member; parallel edges stay separate copies).  One
// super-vertex left certifies lambda >= kcap; that is exactly the item's
// acceptance, whichever contraction reached it, so the result is the one the
// canonical passes give.  When few super-vertices are left, the dense
// finish's capped passes decide on their weight matrix (they keep every cut
// below kcap as well).  A super-vertex of degree below kcap (lambda < kcap),
// a round that contracts nothing, too many super-vertices after the last
// round, or a failing dense check gives up and the canonical passes decide.
//
// Each forest is one pass of union-find links over the unused edges (each
// undirected edge once, from its smaller end): the edges whose link joined
// two sets form a spanning forest of them, and it is maximal.  The
// union-find array lives in shared memory when the item leaves room.
// Returns the rounds taken (> 0: certified) or minus the rounds tried.
// Uses C, D, E, G, H, ebits (and wide for the dense check).
constexpr int FOREST_MAX_K = 16;       // at most 15 forests a round
constexpr int FOREST_ROUNDS = 4;
constexpr int FOREST_LONG_ROW = 32;    // rows longer than this go to a whole warp

// Calls f(a, q, b) for every adjacency entry q = (a -> b) of every alive
// vertex a with sel(a): rows up to FOREST_LONG_ROW entries by one thread,
// longer rows (listed in lr[0..nlr)) by a whole warp.
template <typename IT, typename Sel, typename F>
__device__ __forceinline__ void rows_pass(const Mem<IT> &m, int n, const int32_t *lr, int nlr,
                                          Sel sel, F f) {
  for (int a = threadIdx.x; a < n; a += RB) {
    if (!m.alive[a]) continue;
    const int b0 = m.off[a], e0 = m.end(a);
    if (e0 - b0 > FOREST_LONG_ROW || !sel(a)) continue;
    for (int q = b0; q < e0; ++q) f(a, q, (int)m.adj[q]);
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int k = warp; k < nlr; k += RW) {
    const int a = lr[k];
    if (!sel(a)) continue;
    for (int q = m.off[a] + lane; q < m.end(a); q += 32) f(a, q, (int)m.adj[q]);
  }
}

template <typename IT>
__device__ __noinline__ int forest_accept(const Mem<IT> *m0, int n, int kcap, int32_t *cf, Sh *shp,
                                          bool prof) {
  Sh &sh = *shp;
  const Mem<IT> m = *m0;
  long long tc = prof ? clock64() : 0;
  auto lap = [&](int k) {  // profile: cycles since the last lap into fdbg[k]
    if (prof) {
      const long long t = clock64();
      if (threadIdx.x == 0) sh.fdbg[k] += t - tc;
      tc = t;
    }
  };
  int32_t *lr = m.D, *rep = m.G, *deg = m.H;
  uint32_t *used = m.ebits;
  volatile uint32_t *vu = used;
  const int E = m.off[n];  // entries the rows have room for
  if (threadIdx.x == 0) sh.ntouched = 0;
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += RB) {
    rep[i] = m.alive[i] ? i : -1;
    if (m.alive[i] && (int)m.len[i] > FOREST_LONG_ROW) lr[atomicAdd(&sh.ntouched, 1)] = i;
  }
  __syncthreads();
  const int nlr = sh.ntouched;
  auto all = [](int) { return true; };
  auto is_used = [&](int q) { return (vu[q >> 5] >> (q & 31)) & 1u; };
  int nroots = 0;
  for (int round = 1; round <= FOREST_ROUNDS; ++round) {
    if (round > 1) {
      // a super-vertex with fewer than kcap edges to the others is a cut
      // below kcap: the item fails, the canonical passes find its cut
      for (int i = threadIdx.x; i < n; i += RB) deg[i] = 0;
      __syncthreads();
      rows_pass(m, n, lr, nlr, all, [&](int a, int q, int b) {
        const int A = rep[a], B = rep[b];
        if (B >= 0 && B != A) atomicAdd(&deg[A], 1);
      });
      __syncthreads();
      int low = 0;
      for (int i = threadIdx.x; i < n; i += RB) low |= rep[i] == i && deg[i] < kcap;
      if (__syncthreads_or(low)) return -round;
      lap(4);
    }
    for (int q = threadIdx.x; q < (E + 31) / 32; q += RB) used[q] = 0u;
    for (int f = 1; f < kcap; ++f) {
      for (int i = threadIdx.x; i < n; i += RB) cf[i] = i;
      __syncthreads();
      rows_pass(m, n, lr, nlr, all, [&](int a, int q, int b) {
        if (b < a) return;  // each undirected edge once
        const int A = rep[a], B = rep[b];
        if (B < 0 || B == A || is_used(q)) return;
        if (uf_link(cf, A, B)) atomicOr(&used[q >> 5], 1u << (q & 31));
      });
      __syncthreads();
      if (prof && threadIdx.x == 0) sh.fdbg[1] += 1;
      lap(0);
    }
    for (int i = threadIdx.x; i < n; i += RB) cf[i] = i;
    __syncthreads();
    int merged = 0;
    rows_pass(m, n, lr, nlr, all, [&](int a, int q, int b) {
      if (b < a) return;
      const int A = rep[a], B = rep[b];
      if (B < 0 || B == A || is_used(q)) return;
      merged |= uf_link(cf, A, B);
    });
    if (!__syncthreads_or(merged)) return -round;
    lap(2);
    int roots = 0;
    for (int i = threadIdx.x; i < n; i += RB) {
      const int r = rep[i];
      if (r >= 0) {
        const int nr = uf_find(cf, r);
        rep[i] = nr;
        roots += nr == i;
      }
    }
    nroots = block_sum_int(roots, sh);
    lap(5);
    if (nroots == 1) return round;
    if (nroots <= DENSE_NSV && nroots * nroots <= 2 * (n + 1)) {
      // few super-vertices: the dense finish's capped passes decide
      int32_t *idx = m.C, *rank = m.H;
      int32_t *w = reinterpret_cast<int32_t *>(m.wide);
      for (int i = threadIdx.x; i < n; i += RB) rank[i] = (rep[i] == i) ? 1 : 0;
      for (int q = threadIdx.x; q < nroots * nroots; q += RB) w[q] = 0;
      __syncthreads();
      block_scan_array(rank, n, sh);
      for (int i = threadIdx.x; i < n; i += RB)
        if (rep[i] == i) idx[i] = rank[i];
      __syncthreads();
      rows_pass(m, n, lr, nlr, all, [&](int a, int q, int b) {
        const int A = rep[a], B = rep[b];
        if (B >= 0 && B != A) atomicAdd(&w[idx[A] * nroots + idx[B]], 1);
      });
      __syncthreads();
      if (threadIdx.x < 32) dense_cta(w, nroots, kcap, &sh);
      __syncthreads();
      lap(3);
      return sh.dcut < 0 ? round : -round;
    }
  }
  return -FOREST_ROUNDS;
}

// ---- items of at most 64 vertices: one warp each ---------------------------------
// A CTA that claims such an input cluster claims a block of up to TINY_BLOCK
// more at once, and its warps take them one after the other (what a warp
// cannot take runs on the whole CTA afterwards).  With n <= 32 R (R = 1 or 2 rows per lane) the induced
// subgraph is a bit matrix: lane l holds the rows of members l and l + 32 as
// bitmasks over local ids, components grow by OR-reductions of rows, the
// peel is a popcount, the first contraction pass grows its phases by popcounts
// and ballots, and what it leaves goes to the dense finish -- the same steps
// and rules as the CTA path, in registers.  (With every pass on the whole
// matrix in the dense finish, one shuffle reduction a vertex and pass, an item
// of 45-64 vertices took 100 us instead of 21 and 2M vertices in 100,000 small
// clusters 10.5 ms instead of 9.3.)  The parts an item splits into (components, the two
// sides of its cut) are subsets of the same matrix, so the warp refines
// them itself, one after the other, instead of queueing them: each part is
// the same child item (its vertex set alone decides its outcome, and the
// local ids keep their order), only without its own claim and extraction.

template <int R>
struct TinyMask;
template <>
struct TinyMask<1> { using T = uint32_t; };
template <>
struct TinyMask<2> { using T = unsigned long long; };

// Scratch of one warp, in ints: the weights of at most 32 sets, the sets that
// hold them, the part stack (32 masks of R words), row bits (32R masks) and
// the degree prefix (32R).
template <int R>
__host__ __device__ constexpr size_t tiny_scratch_ints() {
  return 32 * 32 + 32 + 32 * R + (32 * R) * R + 32 * R;
}
constexpr size_t TINY_SCRATCH = 4 * tiny_scratch_ints<2>();     // items of up to 64 vertices
constexpr size_t TINY_SCRATCH_32 = 4 * tiny_scratch_ints<1>();  // up to 32
static_assert(TINY_SCRATCH % 8 == 0 && TINY_SCRATCH_32 % 8 == 0, "mask arrays stay aligned");

__device__ __forceinline__ uint32_t warp_or(uint32_t x) { return __reduce_or_sync(FULL, x); }
__device__ __forceinline__ unsigned long long warp_or(unsigned long long x) {
  const uint32_t lo = __reduce_or_sync(FULL, (uint32_t)x);
  const uint32_t hi = __reduce_or_sync(FULL, (uint32_t)(x >> 32));
  return ((unsigned long long)hi << 32) | lo;
}
__device__ __forceinline__ int popc_m(uint32_t x) { return __popc(x); }
__device__ __forceinline__ int popc_m(unsigned long long x) { return __popcll(x); }
__device__ __forceinline__ int ffs_m(uint32_t x) { return __ffs(x); }
__device__ __forceinline__ int ffs_m(unsigned long long x) { return __ffsll((long long)x); }

template <int R, typename M>
__device__ __forceinline__ M tiny_component(const M (&row)[R], M set, int start) {
  const int l = threadIdx.x & 31;
  M V = (M)1 << start, F = V;
  for (;;) {
    M acc = 0;
#pragma unroll
    for (int j = 0; j < R; ++j)
      if ((F >> (l + 32 * j)) & 1u) acc |= row[j];
    const M nx = warp_or(acc) & set & ~V;
    if (!nx) return V;
    V |= nx;
    F = nx;
  }
}

// Pushes every component of set (with at least min_size members) onto the
// part stack stk[0..*sp).  Returns the number of components.
template <int R, typename M>
__device__ __forceinline__ int tiny_push_components(const M (&row)[R], M set, int min_size, M *stk,
                                                    int &sp) {
  int k = 0;
  M rem = set;
  while (rem) {
    const M c = tiny_component<R, M>(row, set, ffs_m(rem) - 1);
    if ((threadIdx.x & 31) == 0 && popc_m(c) >= min_size) stk[sp] = c;
    sp += popc_m(c) >= min_size ? 1 : 0;
    ++k;
    rem &= ~c;
  }
  __syncwarp();
  return k;
}

// Returns false when the whole CTA has to take the item: its members' degree
// sum exceeds P.tiny_max_deg (a hub's row would keep one warp busy while its
// CTA waits), or a part is left with more than 32 sets after its first pass
// (parts accepted before that are accepted again, with the same result).
template <int R>
__device__ bool tiny_item_body(const RefineParams &P, unsigned long long seq, const Item &it,
                               int32_t *scratch, unsigned long long *tst) {
  using M = typename TinyMask<R>::T;
  constexpr int NV = 32 * R;  // vertices a warp holds
  const int l = threadIdx.x & 31;
  const int n = it.n;
  ReqCtx *Rg = &P.reqs[it.req];
  const ReqCtx Rc = load_ctx(Rg);
  int32_t *w = scratch, *grp = scratch + 32 * 32;
  M *stk = reinterpret_cast<M *>(grp + 32);
  M *rbits = stk + 32;
  int32_t *pre = reinterpret_cast<int32_t *>(rbits + NV);
  int32_t v[R];
  int64_t rb[R];
  int len[R];
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int i = l + 32 * j;
    v[j] = i < n ? __ldcg(&Rc.pool[it.vbeg + i]) : -1;
    rb[j] = i < n ? Rc.off[v[j]] : 0;
    len[j] = i < n ? (int)(Rc.off[v[j] + 1] - rb[j]) : 0;
  }
  int D = 0;
#pragma unroll
  for (int j = 0; j < R; ++j) {
    const int inc = warp_inclusive_scan(len[j]) + D;
    pre[l + 32 * j] = inc;
    D = __shfl_sync(FULL, inc, 31);
  }
  if (D > P.tiny_max_deg) return false;
  const uint32_t tag = queue_tag(seq);
  // 1. extraction, flat over the D adjacency entries of the members: lane l
  // takes entries l, l+32, ..., eight at a time (eight neighbour loads, then
  // eight slot gathers in flight); entry f belongs to the row whose degree
  // prefix first exceeds f, and a hit sets that row's bit in shared memory
#pragma unroll
  for (int j = 0; j < R; ++j) rbits[l + 32 * j] = 0;
  __syncwarp();
  constexpr int Q = 8;
  for (int f0 = 0; f0 < D; f0 += 32 * Q) {
    int32_t u[Q];
    int rr[Q];
#pragma unroll
    for (int z = 0; z < Q; ++z) {
      const int f = f0 + 32 * z + l;
      int lo = 0, hi = NV - 1;  // smallest r with pre[r] > f
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (pre[mid] > f) hi = mid; else lo = mid + 1;
      }
      rr[z] = f < D ? lo : -1;
    }
#pragma unroll
    for (int z = 0; z < Q; ++z) {
      const int r = rr[z] < 0 ? 0 : rr[z];
      int64_t br = __shfl_sync(FULL, rb[0], r & 31);
      int lr = __shfl_sync(FULL, len[0], r & 31);
      if (R == 2) {
        const int64_t b1 = __shfl_sync(FULL, rb[R - 1], r & 31);
        const int l1 = __shfl_sync(FULL, len[R - 1], r & 31);
        if (r >= 32) { br = b1; lr = l1; }
      }
      const int sr = pre[r] - lr;
      u[z] = rr[z] >= 0 ? Rc.adj[br + (f0 + 32 * z + l - sr)] : -1;
    }
    unsigned long long sl[Q];
#pragma unroll
    for (int z = 0; z < Q; ++z) sl[z] = u[z] >= 0 ? __ldcg(&Rc.slot[u[z]]) : 0ull;
#pragma unroll
    for (int z = 0; z < Q; ++z)
      if (u[z] >= 0 && (unsigned)(sl[z] >> 32) == tag)
        atomicOr(&rbits[rr[z]], (M)1 << (unsigned)(sl[z] & 0xffffffffu));
  }
  __syncwarp();
  M row[R];
#pragma unroll
  for (int j = 0; j < R; ++j) row[j] = l + 32 * j < n ? rbits[l + 32 * j] : (M)0;
  // statistics of the whole subtree, added once at the end (lane 0)
  long long st_items = 1, st_peeled = 0, st_passes = 0, st_phases = 0, st_acc = 0, st_splits = 0;
  bool failed = false;
  const M all = n >= NV ? ~(M)0 : (((M)1 << n) - 1);
  int sp = 0;
  bool whole = true;  // the item itself is refined as it is
  // 2. input cluster: CCR (Algorithm 1); when it splits, its components are
  // the parts
  if (it.flags & ITEM_TOP) {
    const int k = tiny_push_components<R, M>(row, all, Rc.min_size, stk, sp);
    if (k == 1) sp = 0;
    else whole = false;
  }
  M set = all;
  for (;;) {
    if (!whole) {
      if (sp == 0) break;
      set = stk[--sp];
      st_items += 1;
    }
    whole = false;
    __syncwarp();
    const int nset = popc_m(set);
    // 3. peel, round-synchronous, T from the alive count
    M cur = set;
    for (;;) {
      const int64_t T = threshold_of(Rc.rule_kind, Rc.rule_num, Rc.rule_den, popc_m(cur));
      M rm = 0;
#pragma unroll
      for (int j = 0; j < R; ++j) {
        const bool r = ((cur >> (l + 32 * j)) & 1u) && popc_m(row[j] & cur) <= T;
        rm |= (M)__ballot_sync(FULL, r) << (32 * j);
      }
      if (!rm) break;
      cur &= ~rm;
    }
    const int nal = popc_m(cur);
    st_peeled += nset - nal;
    if (nal < Rc.min_size) continue;
    // 4. connectivity of what is left (only a peel can disconnect it)
    if (nal < nset) {
      const int sp0 = sp;
      const int k = tiny_push_components<R, M>(row, cur, Rc.min_size, stk, sp);
      if (k > 1) continue;
      sp = sp0;  // one component: refine it as it is
    }
    // 5-6. contraction with k = T+1, then canonical Stoer-Wagner.  The first
    // pass phase by phase (see "contraction passes"): a key is a popcount of
    // the vertex's row with the added set, so a round of a closure is one
    // ballot per 32 vertices
    const int64_t T = threshold_of(Rc.rule_kind, Rc.rule_num, Rc.rule_den, nal);
    const int kcap = (int)(T + 1 < (1ll << 30) ? T + 1 : (1ll << 30));
    M rw[R], mine[R];  // mine: the phase each of the lane's vertices is in
#pragma unroll
    for (int j = 0; j < R; ++j) {
      rw[j] = ((cur >> (l + 32 * j)) & 1u) ? row[j] & cur : (M)0;
      mine[j] = 0;
    }
    M left = cur, roots = 0;
    int p = 0;
    while (left) {
      unsigned best = 0u;  // largest key, then smallest id
      const M in = cur & ~left;
#pragma unroll
      for (int j = 0; j < R; ++j)
        if ((left >> (l + 32 * j)) & 1u)
          best = max(best, ((unsigned)popc_m(rw[j] & in) << 8) | (unsigned)(255 - (l + 32 * j)));
      best = __reduce_max_sync(FULL, best);
      M C = (M)1 << (255u - (best & 255u));
      left &= ~C;
      while (left) {
        M add = 0;
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const bool t = ((left >> (l + 32 * j)) & 1u) && popc_m(rw[j] & ~left) >= kcap;
          add |= (M)__ballot_sync(FULL, t) << (32 * j);
        }
        if (!add) break;
        C |= add;
        left &= ~add;
      }
#pragma unroll
      for (int j = 0; j < R; ++j)
        if ((C >> (l + 32 * j)) & 1u) mine[j] = C;
      roots |= C & (~C + 1);
      ++p;
    }
    int cut = -1, passes = 1, phases = 0;
    M side = 0;
    if (p > 32) return false;  // more sets than the matrix holds: the whole CTA takes the item
    if (p > 1) {
      // the sets' weights (indexed by their smallest members in ascending
      // order), then the dense finish; a first pass that merged nothing is
      // the one it repeats
      int at[R];
#pragma unroll
      for (int j = 0; j < R; ++j) at[j] = popc_m(roots & ((mine[j] & (~mine[j] + 1)) - 1));
      for (int q = l; q < p * p; q += 32) w[q] = 0;
      __syncwarp();
      M rem = roots;
      for (int b = 0; b < p; ++b) {
        // the set of root b, from a lane that holds its smallest member
        const int r0 = ffs_m(rem) - 1;
        rem &= rem - 1;
        M Cb = __shfl_sync(FULL, mine[0], r0 & 31);
        if (R == 2) {
          const M C1 = __shfl_sync(FULL, mine[R - 1], r0 & 31);
          if (r0 >= 32) Cb = C1;
        }
#pragma unroll
        for (int j = 0; j < R; ++j) {
          const int c = (mine[j] && at[j] != b) ? popc_m(rw[j] & Cb) : 0;
          if (c) atomicAdd(&w[at[j] * p + b], c);
        }
      }
      __syncwarp();
      const DenseResult dr = dense_finish<1>(w, p, kcap, grp);
      cut = dr.cut;
      passes = dr.passes + (p < nal ? 1 : 0);
      phases = dr.phases;
#pragma unroll
      for (int j = 0; j < R; ++j)
        side |= (M)__ballot_sync(FULL, mine[j] && ((dr.side[0] >> at[j]) & 1u)) << (32 * j);
      __syncwarp();
    }
    st_passes += passes;
    st_phases += phases;
    if (cut < 0) {
      // accept (Algorithm 3: save V_c); output id resolved after the run
      const int i0 = ffs_m(cur) - 1;
      int32_t minv = __shfl_sync(FULL, v[0], i0 & 31);
      if (R == 2) {
        const int32_t m1 = __shfl_sync(FULL, v[R - 1], i0 & 31);
        if (i0 >= 32) minv = m1;
      }
#pragma unroll
      for (int j = 0; j < R; ++j)
        if ((cur >> (l + 32 * j)) & 1u) Rc.label_min[v[j]] = minv;
      st_acc += 1;
      continue;
    }
    if (cut > T) {
      failed = true;
      break;
    }
    // Algorithm 3: bisect on the minimum cut; both sides are parts
    st_splits += 1;
    const M s0 = cur & ~side, s1 = cur & side;
    if (l == 0) {
      int q = sp;
      if (popc_m(s0) >= Rc.min_size) stk[q++] = s0;
      if (popc_m(s1) >= Rc.min_size) stk[q++] = s1;
    }
    sp += (popc_m(s0) >= Rc.min_size ? 1 : 0) + (popc_m(s1) >= Rc.min_size ? 1 : 0);
    __syncwarp();
  }
  if (l == 0) {
    if (failed) atomicOr(&P.ctr->error, DERR_INTERNAL);
    // added to the request once per batch (one address for all CTAs)
    atomicAdd(&tst[0], (unsigned long long)st_items);
    atomicAdd(&tst[1], (unsigned long long)(((it.flags & ITEM_TOP) ? 8ll * n : 0ll) + 8ll * D));
    if (st_peeled) atomicAdd(&tst[2], (unsigned long long)st_peeled);
    if (st_passes) atomicAdd(&tst[3], (unsigned long long)st_passes);
    if (st_phases) atomicAdd(&tst[4], (unsigned long long)st_phases);
    if (st_acc) atomicAdd(&tst[5], (unsigned long long)st_acc);
    if (st_splits) atomicAdd(&tst[6], (unsigned long long)st_splits);
  }
  return true;
}

// tiny_item_body, recorded in the per-item profile when it is enabled
// (outcome 100, no phase split).
__device__ __forceinline__ bool tiny_item_any(const RefineParams &P, unsigned long long seq,
                                              const Item &it, int32_t *scratch,
                                              unsigned long long *tst) {
  return it.n <= 32 ? tiny_item_body<1>(P, seq, it, scratch, tst)
                    : tiny_item_body<2>(P, seq, it, scratch, tst);
}

__device__ __forceinline__ bool tiny_item(const RefineParams &P, unsigned long long seq,
                                          const Item &it, int32_t *scratch,
                                          unsigned long long *tst) {
  if (!P.prof) return tiny_item_any(P, seq, it, scratch, tst);
  const long long t0 = (long long)globaltimer_ns();
  const bool done = tiny_item_any(P, seq, it, scratch, tst);
  __syncwarp();
  if ((threadIdx.x & 31) == 0 && done) {
    const unsigned r = atomicAdd(P.prof_count, 1u);
    if (r < P.prof_cap) {
      ItemProf *q = &P.prof[r];
      q->seq = (unsigned)seq;
      q->n = it.n;
      q->E = q->nalive = q->passes = q->nsv = -1;
      q->outcome = 100;
      unsigned smid;
      asm("mov.u32 %0, %%smid;" : "=r"(smid));
      q->smid = (int)smid;
      q->slab = 0;
      q->top = (int)(it.flags & ITEM_TOP);
      for (int z = 0; z < 8; ++z) q->dt[z] = 0;
      q->t_begin = t0;
      q->t_end = (long long)globaltimer_ns();
      for (int z = 0; z < 4; ++z) q->dbg[z] = 0;
      q->forest = q->nsv1 = 0;
      q->forest_cycles = 0;
      for (int z = 0; z < 6; ++z) q->fdbg[z] = 0;
    }
  }
  return done;
}

// The end of count items of a request: its and the run's pending counts drop
// (the request's last item raises its host-mapped done flag).  One thread.
__device__ __forceinline__ void finish_items(const RefineParams &P, uint16_t req, int count) {
  __threadfence();
  ReqCtx &R = P.reqs[req];
  const unsigned long long c = (unsigned long long)count;
  const unsigned long long left =
      atomicAdd(reinterpret_cast<unsigned long long *>(&R.pending), 0ull - c);
  if (left == c && P.done_flags) {
    // the request's last item: everything it wrote is visible first
    __threadfence_system();
    ((volatile int *)P.done_flags)[req] = 1;
  }
  add_ll(&P.ctr->pending, -(long long)count);
}

// ---- one work item ---------------------------------------------------------
template <typename IT, bool SM>
__device__ __noinline__ int process_item(const RefineParams &P, unsigned long long seq,
                                         const Item &it, char *slab, int64_t dbound, Sh &sh) {
  char *base = SM ? wcc_dyn_smem : slab;
  const int n = it.n;
  const int64_t vbeg = it.vbeg;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  ReqCtx *Rg = &P.reqs[it.req];
  const ReqCtx R = load_ctx(Rg);
  ReqCtx *ctr = Rg;  // per-request statistics (atomics)
  Mem<IT> m = carve<IT>(base, n, dbound);
  if (SM) m.smem_used = ws_bytes<IT>(n, dbound);
  if (!SM) {
    carve_hot(m, n, P.smem_bytes);
  }

  // global row start and degree of every member; a local row gets room for
  // all of its vertex's entries
  int64_t *gbeg = m.wide;
  int32_t *deg0 = m.C, *cnt = m.D, *lr = m.G;
  for (int i = threadIdx.x; i < n; i += RB) {
    const int32_t v = __ldcg(&R.pool[vbeg + i]);
    m.gid[i] = v;
    const int64_t b = R.off[v];
    const int32_t d = (int32_t)(R.off[v + 1] - b);
    gbeg[i] = b;
    deg0[i] = d;
    m.off[i] = d;
    if (d > LONG_ROW) cnt[i] = 0;
    m.alive[i] = 1;
  }
  if (threadIdx.x == 0) sh.ntouched = 0;
  __syncthreads();
  const int D = block_scan_array(m.off, n, sh);
  if (threadIdx.x == 0) m.off[n] = D;
  __syncthreads();
  prof_stamp(P, sh, 1);

  // 1. extraction: entry (i, u) stays iff slot[u] names this item, as u's
  // local id; the entries of a local row are in any order.  What bounds it is
  // the latency of two dependent gathers an entry (neighbour, then its slot),
  // so every lane keeps four entries in flight whatever the row lengths: a
  // warp takes up to 32 rows, lane r holding row r's bounds, and walks their
  // entries as one flat range, 128 at a time; an entry's row is found by a
  // binary search over the lanes' degree prefix, its place by a ballot and
  // the count of hits that the row's lane holds.  Long rows are shared by
  // all warps in segments of 128 entries.  A cluster of 47,000 vertices and
  // 2.15M entries takes 9.3M cycles (two rows a warp at a time, all entries
  // kept and compacted by a second pass: 20.7M; eight rows a warp, each lane
  // waiting for the longest: 13.4M).
  {
    const uint32_t tag = queue_tag(seq);
    const unsigned lt = lanemask_lt();
    const int per = min(32, (n + RW - 1) / RW);
    for (int r0 = warp * per; r0 < n; r0 += RW * per) {
      const int rows = min(per, n - r0);
      int o = 0, d = 0;
      long long g = 0;
      bool is_long = false;
      if (lane < rows) {
        const int i = r0 + lane;
        o = m.off[i];
        d = deg0[i];
        g = gbeg[i];
        is_long = d > LONG_ROW;
        if (is_long) {
          lr[atomicAdd(&sh.ntouched, 1)] = i;
          d = 0;
        }
      }
      const int inc = warp_inclusive_scan(d), exc = inc - d;
      const int total = __shfl_sync(FULL, inc, 31);
      g -= exc;
      int c = 0;  // hits of the lane's row so far
      for (int f0 = 0; f0 < total; f0 += 128) {
        int row[4];
        int32_t u[4];
        unsigned long long sl[4];
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const int f = f0 + 32 * z + lane;
          int lo = 0;  // rows that end at or before f
#pragma unroll
          for (int st = 16; st > 0; st >>= 1)
            if (__shfl_sync(FULL, inc, lo + st - 1) <= f) lo += st;
          row[z] = lo;
          const long long gr = __shfl_sync(FULL, g, lo);
          u[z] = f < total ? R.adj[gr + f] : -1;
        }
#pragma unroll
        for (int z = 0; z < 4; ++z) sl[z] = u[z] >= 0 ? __ldcg(&R.slot[u[z]]) : ~0ull;
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const bool hit = (uint32_t)(sl[z] >> 32) == tag;
          const unsigned b = __ballot_sync(FULL, hit);
          // the lane's row within these 32 entries
          const int base = f0 + 32 * z;
          const int lo = min(max(exc - base, 0), 32), hi = min(max(inc - base, 0), 32);
          const unsigned mine = (unsigned)((1ull << hi) - (1ull << lo));
          const unsigned rm = __shfl_sync(FULL, mine, row[z]);
          const int at = __shfl_sync(FULL, o + c, row[z]);
          if (hit) m.adj[at + __popc(b & rm & lt)] = (IT)(unsigned)(sl[z] & 0xffffffffu);
          c += __popc(b & mine);
        }
      }
      if (lane < rows && !is_long) m.len[r0 + lane] = (IT)c;
    }
    __syncthreads();
    const int nl = sh.ntouched;
    for (int k = 0; k < nl; ++k) {
      const int i = lr[k], d = deg0[i], o = m.off[i];
      const int64_t g = gbeg[i];
      for (int f0 = 128 * ((warp + k) % RW); f0 < d; f0 += 128 * RW) {
        int32_t u[4];
        unsigned long long sl[4];
#pragma unroll
        for (int z = 0; z < 4; ++z) u[z] = f0 + 32 * z + lane < d ? R.adj[g + f0 + 32 * z + lane] : -1;
#pragma unroll
        for (int z = 0; z < 4; ++z) sl[z] = u[z] >= 0 ? __ldcg(&R.slot[u[z]]) : ~0ull;
#pragma unroll
        for (int z = 0; z < 4; ++z) {
          const bool hit = (uint32_t)(sl[z] >> 32) == tag;
          const unsigned b = __ballot_sync(FULL, hit);
          int at = 0;
          if (lane == 0 && b) at = atomicAdd(&cnt[i], __popc(b));
          at = __shfl_sync(FULL, at, 0);
          if (hit) m.adj[o + at + __popc(b & lanemask_lt())] = (IT)(unsigned)(sl[z] & 0xffffffffu);
        }
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < nl; k += RB) m.len[lr[k]] = (IT)cnt[lr[k]];
    if (threadIdx.x == 0) sh.ntouched = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    add_ll(&ctr->items, 1ll);
    // algorithmic bytes of the extraction: an input cluster reads its
    // members' row offsets (8 B) and, per adjacency entry, the neighbour id
    // and its label (4 + 4 B); re-inducing a part after a split reads the
    // entries again (8 B each)
    add_ll(&ctr->alg_bytes, (long long)((it.flags & ITEM_TOP) ? 8 * n : 0) + 8 * (long long)D);
    sh.pf_E = D;
  }
  prof_stamp(P, sh, 2);

  // The item's vertices are the alive ones.  When it splits into components,
  // the largest one with at least min_size vertices is not queued: this CTA
  // continues with it in place (its induced subgraph is already here; it is
  // the same child item, only without waiting behind the queue), and its
  // later children go to the pool range vb behind the published ones.
  int nalive = n;
  int64_t vb = vbeg;

  // 2. input cluster: CCR (Algorithm 1)
  if (it.flags & ITEM_TOP) {
    int nc = first_pass<IT, SM>(&m, dbound, true, n, n, 1, &P.ctr->error, &sh).x;
    if (nc == -1) return OUT_ERROR;
    if (nc == -2) nc = components_af<IT, SM>(&m, dbound, n, &sh);
    if (nc != 1) {
      int emitted = 0;
      const int L = emit_children<IT, SM>(P, R, Rg, it.req, &m, dbound, TAG_B, n, vb, &sh, 0, true,
                                              &emitted);
      if (L < 0) return OUT_CCR_SPLIT;
      nalive = restrict_alive(m, m.B, L, n, sh);
      vb += emitted;
      if (threadIdx.x == 0) add_ll(&ctr->items, 1ll);
    }
  }
  prof_stamp(P, sh, 3);

  // 3. peel (round-synchronous, T recomputed from the alive count).  T never
  // grows, so after the first round only a vertex whose degree has just
  // dropped to T can go: each drop to T lists it once, and the next round
  // takes the listed ones that its own T still covers (the others are listed
  // again when they drop to it).
  int32_t *deg = m.A;
  const int n_item = nalive;
  {
    int32_t *cand = m.G, *next = m.H;
    int64_t T = threshold_of(R.rule_kind, R.rule_num, R.rule_den, nalive);
    if (threadIdx.x < 3) sh.qn[threadIdx.x] = 0;
    __syncthreads();
    for (int i0 = 0; i0 < n; i0 += RB) {
      const int i = i0 + threadIdx.x;
      int d = 0;
      if (i < n) deg[i] = d = (int)m.len[i];
      warp_push(i < n && m.alive[i] && d <= T, i, cand, 0, &sh.qn[0]);
    }
    __syncthreads();
    int nc = *(volatile int32_t *)&sh.qn[0];
    for (int r = 1; nc > 0; r = r == 2 ? 0 : r + 1) {
      T = threshold_of(R.rule_kind, R.rule_num, R.rule_den, nalive);
      int rem = 0;
      for (int q = threadIdx.x; q < nc; q += RB) {
        const int i = cand[q];
        if (deg[i] <= T) {
          m.alive[i] = 0;
          ++rem;
        } else {
          cand[q] = -1;
        }
      }
      if (threadIdx.x == 0) sh.qn[r == 2 ? 0 : r + 1] = 0;
      rem = block_sum_int(rem, sh);
      if (rem == 0) break;
      nalive -= rem;
      const int per = min(32, (nc + RW - 1) / RW);
      for (int c0 = warp * per; c0 < nc; c0 += RW * per) {
        int b = 0, d = 0, exc;
        if (lane < min(per, nc - c0)) {
          const int i = cand[c0 + lane];
          if (i >= 0) {
            b = m.off[i];
            d = (int)m.len[i];
          }
        }
        flat_rows(m.adj, b, d, exc, [&](const int (&j)[4], int) {
          bool drop[4];
#pragma unroll
          for (int z = 0; z < 4; ++z) drop[z] = j[z] >= 0 && m.alive[j[z]];
#pragma unroll
          for (int z = 0; z < 4; ++z)
            if (drop[z]) drop[z] = (int64_t)atomicSub(&deg[j[z]], 1) - 1 == T;
          warp_push4(drop, j, next, 0, &sh.qn[r]);
        });
      }
      __syncthreads();
      nc = *(volatile int32_t *)&sh.qn[r];
      int32_t *t = cand;
      cand = next;
      next = t;
    }
  }
  if (threadIdx.x == 0) {
    if (nalive < n_item) add_ll(&ctr->peeled, (long long)(n_item - nalive));
    sh.pf_nalive = nalive;
  }
  prof_stamp(P, sh, 4);
  if (nalive < R.min_size) return OUT_DROPPED;

  // 4. connectivity of what is left (an item arrives connected: input
  // clusters passed CCR above, children are components or sides of a
  // minimum cut, which are connected; only a peel can disconnect it).  The
  // first contraction pass of step 5 finds the components on its way: it
  // runs here, and stands for the component continued in place too (no edge
  // joins the components, so that one's phases are those it has alone) unless
  // its smaller size changes T.  That component needs no peel of its own: T
  // only grows with n, so every vertex left already has degree > T of its
  // smaller size.
  int32_t *rep = m.A;
  int pre = 0;             // > 0: sets of the first pass, which has run already
  bool pre_order = false;  // ... and the order of adding is in D
  if (nalive < n_item) {
    const int64_t T0 = threshold_of(R.rule_kind, R.rule_num, R.rule_den, nalive);
    int comps = 0, ph = -2;
        if (T0 < KEY_MAX) {
      const int2 r = first_pass<IT, SM>(&m, dbound, false, n, nalive, (int)T0 + 1, &P.ctr->error, &sh);
      ph = r.x;
      comps = r.y;
    }
    if (ph == -1) return OUT_ERROR;
    if (ph == -2) {
      comps = components_af<IT, SM>(&m, dbound, n, &sh);
    }
    if (comps > 1) {
      int emitted = 0;
      const int L = emit_children<IT, SM>(P, R, Rg, it.req, &m, dbound, ph == -2 ? TAG_B : TAG_H, n, vb,
                                              &sh, 0, true, &emitted);
      if (L < 0) return OUT_CC_SPLIT;
      nalive = restrict_alive(m, ph == -2 ? m.B : m.H, L, n, sh);
      vb += emitted;
      if (threadIdx.x == 0) add_ll(&ctr->items, 1ll);
      if (ph > 0 && threshold_of(R.rule_kind, R.rule_num, R.rule_den, nalive) == T0) {
        int r1 = 0;
        for (int i = threadIdx.x; i < n; i += RB) {
          if (!m.alive[i]) rep[i] = -1;
          r1 += rep[i] == i;
        }
        pre = block_sum_int(r1, sh);
      }
    } else if (ph > 0) {
      pre = ph;
      pre_order = true;
    }
  }
  prof_stamp(P, sh, 5);

  // 5. contraction with k = T+1
  const int64_t T = threshold_of(R.rule_kind, R.rule_num, R.rule_den, nalive);
  const int kcap = (int)(T + 1 < (1ll << 30) ? T + 1 : (1ll << 30));
  int nsv = 1, passes = 0;
  int dense_cut = -1;  // >= 0: the dense finish found the cut (side in m.side)
  bool certified = false;
  bool inh_valid = false;  // R.inh holds this item's first-pass records
  if (kcap <= FOREST_MAX_K && P.forest_min_n > 0 && nalive >= P.forest_min_n) {
    const long long f0 = P.prof ? clock64() : 0;
    // the forests' union-find: in shared memory for an item in the global
    // slab when its row offsets did not move there (the first pass's state
    // there is set up only later)
    int32_t *cf = m.B;
    if (!SM && !m.off_in_smem && 4 * (size_t)n <= P.smem_bytes)
      cf = reinterpret_cast<int32_t *>(wcc_dyn_smem);
    const int fr = forest_accept(&m, n, kcap, cf, &sh, P.prof != nullptr);
    certified = fr > 0;
    pre_order = false;
    if (P.prof && threadIdx.x == 0) {
      sh.pf_forest = fr;
      sh.pf_forest_cycles = clock64() - f0;
    }
  }
  if (!certified) {
    nsv = nalive;
    bool more = true;
    if (kcap <= KEY_MAX) {
      if (threadIdx.x == 0) add_ll(&ctr->ni_passes, 1ll);
      ++passes;
      // A side S of a parent's cut (value <= T) whose members are the first
      // |S| vertices the parent's first pass added, with the same kcap and
      // nothing peeled here, would run exactly that order's prefix: until
      // the order left S no vertex outside S had been added, so S's keys,
      // its phases' first vertices and their closures are the same in the
      // induced subgraph (and the order leaves S between two phases: a
      // vertex outside S added inside one would have kcap > T neighbours in
      // S, across a cut of at most T).  The phases' smallest members are
      // taken from the records instead of repeating the pass; any record
      // that does not fit falls back to it.
      const bool recordable = kcap < 256 && n < (1 << 24);
      bool inherited = false;
      if ((it.flags & ITEM_INH) && recordable && R.inh != nullptr && nalive == n) {
        int bad = 0;
        for (int i = threadIdx.x; i < n; i += RB) {
          const unsigned long long rec = __ldcg(&R.inh[m.gid[i]]);
          const int kc = (int)(rec >> 56), p = (int)((rec >> 32) & 0xffffffu);
          const long long r = (long long)(uint32_t)rec;
          int loc = -1;
          if (kc == kcap && p < n && r < R.n_vertices) {
            const unsigned long long sr = __ldcg(&R.slot[r]);
            if ((unsigned)(sr >> 32) == queue_tag(seq)) loc = (int)(unsigned)(sr & 0xffffffffu);
          }
          if (loc < 0 || loc > i) bad = 1;  // a root is the smallest member of its set
          rep[i] = loc;
        }
        if (!__syncthreads_or(bad)) {
          for (int i = threadIdx.x; i < n; i += RB)
            if (rep[rep[i]] != rep[i]) bad = 1;
          inherited = !__syncthreads_or(bad);
        }
      }
      if (inherited) {
        int r1 = 0;
        for (int i = threadIdx.x; i < n; i += RB) r1 += rep[i] == i;
        nsv = block_sum_int(r1, sh);
        inh_valid = true;
      } else {
        const long long p0 = P.prof ? clock64() : 0;
        if (pre > 0) {
          nsv = pre;
        } else {
          // (what is left is connected)
          nsv = first_pass<IT, SM>(&m, dbound, false, n, nalive, kcap, &P.ctr->error, &sh).x;
          if (nsv < 0) {
            if (threadIdx.x == 0) atomicOr(&P.ctr->error, DERR_INTERNAL);
            return OUT_ERROR;
          }
        }
        // this pass's records, for the sides of a later cut (the order of
        // adding is in D)
        inh_valid = R.inh != nullptr && recordable && nalive >= INH_MIN_N && (pre == 0 || pre_order);
        if (inh_valid) {
          for (int q = threadIdx.x; q < nalive; q += RB) {
            const int i = m.D[q];
            R.inh[m.gid[i]] = ((unsigned long long)kcap << 56) |
                              ((unsigned long long)(unsigned)q << 32) | (unsigned)m.gid[rep[i]];
          }
          __syncthreads();
        }
        if (P.prof && threadIdx.x == 0) sh.dbg[0] = clock64() - p0;
      }
      more = nsv < nalive;  // the pass merged something
      if (P.prof && threadIdx.x == 0) sh.pf_nsv1 = nsv;
    } else {
      for (int i = threadIdx.x; i < n; i += RB) rep[i] = m.alive[i] ? i : -1;
      __syncthreads();
    }
    const long long tl0 = P.prof ? clock64() : 0;
    while (more && nsv > 1) {
      // the weight matrix of the dense finish: in E..F when it fits, else in
      // the dynamic shared memory past what the item occupies
      int32_t *wmat = nullptr;
      if (nsv <= P.dense_max && nsv <= DENSE_NSV) {
        if (nsv * nsv <= 2 * (n + 1)) {
          wmat = reinterpret_cast<int32_t *>(m.wide);
        } else {
          const size_t at = align16(m.smem_used);
          if (at + 4 * (size_t)nsv * (size_t)nsv <= P.smem_bytes)
            wmat = reinterpret_cast<int32_t *>(wcc_dyn_smem + at);
        }
      }
      if (wmat == nullptr) {  // another pass on the sets
        if (threadIdx.x == 0) add_ll(&ctr->ni_passes, 1ll);
        ++passes;
        const int k = class_pass<IT, SM>(&m, dbound, n, kcap, &P.ctr->error, &sh);
        if (k < 0) return OUT_ERROR;
        more = k < nsv;
        nsv = k;
        continue;
      }
      // few super-vertices left: their weight matrix, then the dense finish.
      // Rows of the largest one (most often it holds nearly all vertices)
      // are not looked through: its weights come from the other ends.
      int32_t *idx = m.C, *lr = m.D, *roots = m.H;
      int32_t *w = wmat;
      if (threadIdx.x < 32) {  // the set of most of 32 spread vertices
        const int v = (int)(((long long)lane * n) / 32);
        const int r = m.alive[v] ? rep[v] : -1;
        const unsigned peers = __match_any_sync(FULL, r);
        const unsigned long long best =
            warp_max(r >= 0 ? ((unsigned long long)__popc(peers) << 32) | (unsigned)r : 0ull);
        if (lane == 0) sh.i0 = best ? (int)(best & 0xffffffffu) : -1;
      }
      if (threadIdx.x == 0) sh.ntouched = sh.qn[0] = 0;
      __syncthreads();
      // the sets' smallest members, each one's index the number of smaller ones
      for (int i0 = 0; i0 < n; i0 += RB) {
        const int i = i0 + threadIdx.x;
        warp_push(i < n && rep[i] == i, i, roots, 0, &sh.qn[0]);
      }
      for (int q = threadIdx.x; q < nsv * nsv; q += RB) w[q] = 0;
      __syncthreads();
      for (int k = threadIdx.x; k < nsv; k += RB) {
        const int r = roots[k];
        int at = 0;
        for (int q = 0; q < nsv; ++q) at += roots[q] < r;
        idx[r] = at;
      }
      __syncthreads();
      const int big = sh.i0;
      auto weigh = [&](int A, int u) {  // the entry from a member of A to u
        const int r = rep[u];
        if (r < 0) return;
        const int B = idx[r];
        if (B == A) return;
        atomicAdd(&w[A * nsv + B], 1);
        if (r == big) atomicAdd(&w[B * nsv + A], 1);
      };
      for (int a = threadIdx.x; a < n; a += RB) {
        if (!m.alive[a] || rep[a] == big) continue;
        const int b0 = m.off[a], e0 = m.end(a);
        if (e0 - b0 > 32) {
          lr[atomicAdd(&sh.ntouched, 1)] = a;
          continue;
        }
        const int A = idx[rep[a]];
        for (int q = b0; q < e0; ++q) weigh(A, (int)m.adj[q]);
      }
      __syncthreads();
      {
        const int nl = sh.ntouched;
        for (int k = warp; k < nl; k += RW) {
          const int a = lr[k], A = idx[rep[a]];
          for (int q = m.off[a] + lane; q < m.end(a); q += 32) weigh(A, (int)m.adj[q]);
        }
      }
      __syncthreads();
      if (threadIdx.x < 32) dense_cta(w, nsv, kcap, &sh);
      __syncthreads();
      passes += sh.dpasses;
      if (threadIdx.x == 0) {
        add_ll(&ctr->ni_passes, (long long)sh.dpasses);
        add_ll(&ctr->sw_phases, (long long)sh.dphases);
      }
      if (sh.dcut < 0) {
        nsv = 1;
      } else {
        dense_cut = sh.dcut;
        for (int i = threadIdx.x; i < n; i += RB) {
          const int k = m.alive[i] ? idx[rep[i]] : 0;
          m.side[i] = m.alive[i] && ((sh.wside[k >> 5] >> (k & 31)) & 1u);
        }
        __syncthreads();
      }
      more = false;
    }
    if (P.prof && threadIdx.x == 0) sh.dbg[3] = clock64() - tl0;
  }
  if (threadIdx.x == 0) {
    sh.pf_passes = passes;
    sh.pf_nsv = nsv;
  }
  prof_stamp(P, sh, 6);
  if (nsv <= 1) {
    // accept (Algorithm 3: save V_c); output id resolved after the run
    if (threadIdx.x == 0) sh.i0 = n;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += RB)
      if (m.alive[i]) { atomicMin(&sh.i0, i); break; }
    __syncthreads();
    const int32_t minv = m.gid[sh.i0];
    for (int i = threadIdx.x; i < n; i += RB)
      if (m.alive[i]) R.label_min[m.gid[i]] = minv;
    if (threadIdx.x == 0) add_ll(&ctr->accepted, 1ll);
    __syncthreads();
    return OUT_ACCEPT;
  }

  // 6. canonical Stoer-Wagner on the contracted graph; grp = A (starts as rep)
  if (dense_cut >= 0) {
    if (dense_cut > T) {
      if (threadIdx.x == 0) atomicOr(&P.ctr->error, DERR_INTERNAL);
      return OUT_ERROR;
    }
  } else {
    const int best = sparse_cut<IT, SM>(&m, dbound, n, nsv, &ctr->sw_phases, &sh);
    prof_stamp(P, sh, 7);
    if (best > T) {
      if (threadIdx.x == 0) atomicOr(&P.ctr->error, DERR_INTERNAL);
      return OUT_ERROR;
    }
  }
  if (threadIdx.x == 0) add_ll(&ctr->splits, 1ll);
  for (int i = threadIdx.x; i < n; i += RB) m.B[i] = m.alive[i] ? (m.side[i] ? 1 : 0) : -1;
  __syncthreads();
  if (P.cm)
    park_sides(P, R, it.req, m, m.B, n, vb, sh);
  else
    // the larger side is refined next by this CTA: queued, it would wait behind
    // every input cluster, and a chain of parts as often as it has cuts (10M
    // vertices 38.7 -> 37.2 ms a step, small clusters 2M 3.98 -> 3.77)
    emit_children<IT, SM>(P, R, Rg, it.req, &m, dbound, TAG_B, n, vb, &sh,
                          inh_valid ? ITEM_INH : (uint16_t)0, false, nullptr,
                          P.stop_flag == nullptr && !P.single_item, seq);
  return OUT_CUT_SPLIT;
}

// Chooses the local id width and the memory (shared or the CTA's slab) for
// an item, then processes it.
__device__ int run_item(const RefineParams &P, unsigned long long seq, const Item &it, char *slab,
                        Sh &sh) {
  const int n = it.n;
  const ReqCtx R = load_ctx(&P.reqs[it.req]);
  long long dsum = 0;
  for (int i = threadIdx.x; i < n; i += RB) {
    const int32_t v = __ldcg(&R.pool[it.vbeg + i]);
    dsum += R.off[v + 1] - R.off[v];
  }
  dsum = block_sum_ll(dsum, sh);
  // at 65,535 vertices the working memory is far above what a CTA can hold
  // in shared memory: 32-bit local ids only occur in the slab
  const bool narrow = n < 65535;
  const size_t need = narrow ? ws_bytes<uint16_t>(n, dsum) : ws_bytes<int32_t>(n, dsum);
  const bool in_smem = narrow && need <= P.smem_bytes;
  if (!in_smem && (need > P.slab_bytes || dsum >= (1ll << 31))) {
    if (threadIdx.x == 0) {
      atomicOr(&P.ctr->error, DERR_CAPACITY);
      atomicExch(&P.ctr->err_info, (unsigned)n);
    }
    return OUT_ERROR;
  }
  if (threadIdx.x == 0) sh.used_slab = !in_smem;
  if (in_smem) return process_item<uint16_t, true>(P, seq, it, slab, dsum, sh);
  return narrow ? process_item<uint16_t, false>(P, seq, it, slab, dsum, sh)
                : process_item<int32_t, false>(P, seq, it, slab, dsum, sh);
}

// Whether a wait for work that began at t0 has outlasted the limit.  A CTA
// that goes on with a part of its own item may publish nothing for long: the
// time counts from the last part kept so, as it would from a published one.
__device__ __forceinline__ bool outlasted(const volatile RunCounters *c, uint64_t t0,
                                          uint64_t limit_ns) {
  return globaltimer_ns() - t0 > limit_ns &&
         (long long)(globaltimer_ns() - c->kept_ns) > (long long)limit_ns;
}

// Waits (bounded) for queue index q to be published and reads its item
// with two 8-byte loads.  False, with DERR_TIMEOUT set, when the wait runs
// out or the run has failed meanwhile.
static_assert(offsetof(Item, vbeg) == 0 && offsetof(Item, n) == 8 && offsetof(Item, flags) == 12 &&
                  offsetof(Item, req) == 14 && sizeof(Item) == 16,
              "an item is read as two 8-byte words");
__device__ __forceinline__ bool fetch_item(const RefineParams &P, unsigned long long q, Item &out) {
  QSlot *sl = &P.ring[q % P.ring_cap];
  volatile RunCounters *vctr = P.ctr;
  const uint64_t t1 = globaltimer_ns();
  unsigned ns2 = 32;
  for (;;) {
    if (*(volatile unsigned long long *)&sl->seq == q) break;
    if (vctr->error != 0 || globaltimer_ns() - t1 > P.wait_limit_ns) {
      atomicOr(&P.ctr->error, DERR_TIMEOUT);
      return false;
    }
    __nanosleep(ns2);
    ns2 = ns2 < 1024 ? ns2 * 2 : ns2;
  }
  __threadfence();
  const volatile unsigned long long *w = reinterpret_cast<const volatile unsigned long long *>(&sl->item);
  const unsigned long long a = w[0], b = w[1];
  out.vbeg = (int64_t)a;
  out.n = (int32_t)(uint32_t)b;
  out.flags = (uint16_t)(b >> 32);
  out.req = (uint16_t)(b >> 48);
  return true;
}

// ---- the persistent kernel ---------------------------------------------------
// Thread 0 claims a queue index only when one has been reserved (head <
// tail), by compare-and-swap, and then waits -- bounded by wait_limit_ns --
// for its publication.  With nothing reserved it waits for more: the kernel
// ends when nothing is pending and the queue is closed, or (open, serving)
// once one CTA has found nothing pending for idle_limit_ns and set closing
// (what is queued by then waits for the next launch);
// a wait for work that is pending but never published ends at wait_limit_ns
// with DERR_TIMEOUT.
__global__ void __launch_bounds__(RB, 1) k_refine(RefineParams P) {
  __shared__ Sh sh;
  char *slab = P.slab + (size_t)blockIdx.x * P.slab_bytes;
  RunCounters *ctr = P.ctr;
  volatile RunCounters *vctr = ctr;
  // items of up to 64 vertices on single warps when the scratch of all
  // warps fits the shared memory, else up to 32, else none
  int tiny_lim = P.tiny_max;
  if (tiny_lim > 32 && P.smem_bytes < (size_t)RW * TINY_SCRATCH) tiny_lim = 32;
  if (tiny_lim > 0 && P.smem_bytes < (size_t)RW * TINY_SCRATCH_32) tiny_lim = 0;
  const size_t tiny_scr = tiny_lim > 32 ? TINY_SCRATCH : TINY_SCRATCH_32;
  const bool tiny_ok = tiny_lim > 0;
  bool took = false;  // thread 0: this CTA has claimed an item in this launch
  CtaProf cp{0, 0, 0, 0, 0, 0, 0};  // thread 0, profile only
  if (threadIdx.x == 0) sh.has_own = 0;
  long long pc = P.prof ? clock64() : 0;
  for (;;) {
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x;
      if (lane == 0 && P.tickets) {
        // A closed run (nothing is added from outside while it runs) claims
        // its first item by ticket: a fetch-and-add on the head never fails,
        // so the CTAs do not contend on a compare-and-swap.  Ticket j is an
        // item once it is reserved (j < tail); while it is not, the CTA
        // waits for it, holding no other work, and leaves once nothing is
        // pending (no item in flight could reserve it any more: an
        // unfinished reserved index keeps pending above zero).
        int go = 0;
        const unsigned long long j = atomicAdd(&ctr->head, 1ull);
        const uint64_t t0 = globaltimer_ns();
        unsigned ns = 32;
        for (;;) {
          if (vctr->error != 0) break;
          if (j < vctr->tail) {
            go = 1;
            break;
          }
          if (vctr->pending <= 0) break;
          if (outlasted(vctr, t0, P.wait_limit_ns)) {
            atomicOr(&ctr->error, DERR_TIMEOUT);
            break;
          }
          __nanosleep(ns);
          ns = ns < 4096 ? ns * 2 : ns;
        }
        if (go && !fetch_item(P, j, sh.first)) go = 0;
        sh.first_seq = j;
        sh.go = go;
      } else if (lane == 0) {
        int go = 0;
        unsigned long long j = 0;
        const uint64_t t0 = globaltimer_ns();
        unsigned ns = 32;
        for (;;) {
          if (vctr->error != 0) break;
          if (P.single_item) {
            j = P.single_index;
            go = 1;
            break;
          }
          // a job step whose time is up: leave at this item boundary (the
          // queue keeps everything not yet claimed).  A CTA takes one item
          // before it looks, so that every step makes progress.
          if (P.stop_flag && took && *P.stop_flag) break;
          // an open (serving) kernel leaves as a whole: the first CTA that
          // idled out closes it for all, and the host relaunches it for what
          // was admitted meanwhile.  Looked at before the queue: work that
          // arrives while the CTAs are leaving would otherwise run on the few
          // that found it, and under load those never see the queue empty
          // (a stream of 1,318 requests/s then completes 184/s).
          if (vctr->closing) break;
          const unsigned long long h = vctr->head, t = vctr->tail;
          if (h < t) {
            if (atomicCAS(&ctr->head, h, h + 1) == h) {
              j = h;
              go = 1;
              took = true;
              break;
            }
            continue;
          }
          if (P.stop_flag && *P.stop_flag) break;
          const long long pend = vctr->pending;
          const uint64_t waited = globaltimer_ns() - t0;
          if (pend <= 0) {
            if (!vctr->open) break;
            if (waited > P.idle_limit_ns) {
              atomicExch(&ctr->closing, 1);
              break;
            }
          } else if (outlasted(vctr, t0, P.wait_limit_ns)) {
            atomicOr(&ctr->error, DERR_TIMEOUT);
            break;
          }
          __nanosleep(ns);
          ns = ns < 4096 ? ns * 2 : ns;
        }
        if (go && !fetch_item(P, j, sh.first)) go = 0;
        sh.first_seq = j;
        sh.go = go;
      }
      if (lane == 0) {
        // a small input cluster: claim a block of more for the CTA's warps.
        // A request's input clusters are queued largest first in one range,
        // so the ones after a small one up to the range's end are small too;
        // a block costs one compare-and-swap and never holds a larger item
        // back behind it.  Half of an even share of what is left, so that
        // blocks shrink towards the end, at least one item a warp.
        int k = 0;
        unsigned long long hb = 0;
        if (sh.go && tiny_ok && !P.single_item && sh.first.n <= tiny_lim &&
            (sh.first.flags & ITEM_TOP) && !(P.stop_flag && *P.stop_flag)) {
          const unsigned long long send = __ldcg(&P.reqs[sh.first.req].seed_end);
          for (int tries = 0; tries < 8; ++tries) {
            if (vctr->error != 0) break;
            const unsigned long long h = vctr->head, t = vctr->tail;
            const unsigned long long lim = t < send ? t : send;
            if (h >= lim) break;
            const unsigned long long share = (lim - h) / (2ull * gridDim.x);
            const unsigned long long want =
                share < RW - 1 ? RW - 1 : (share > TINY_BLOCK ? TINY_BLOCK : share);
            const int kk = (int)min(want, lim - h);
            if (atomicCAS(&ctr->head, h, h + kk) == h) {
              k = kk;
              hb = h;
              break;
            }
          }
        }
        sh.claim_h = hb;
        sh.claim_k = k;
        sh.bnext = 0;
        sh.bdone = 0;
        sh.ncta = 0;
      }
      __syncwarp();  // lane 0 has read the last batch's statistics
      if (lane < 7) sh.tst[lane] = 0ull;
    }
    __syncthreads();
    if (P.prof && threadIdx.x == 0) {
      const long long t = clock64();
      cp.claim += t - pc;
      pc = t;
    }
    if (!sh.go) break;
    if (tiny_ok && sh.first.n <= tiny_lim) {
      // every warp takes the batch's items one after the other
      const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, k = sh.claim_k;
      int32_t *scratch = reinterpret_cast<int32_t *>(wcc_dyn_smem + (size_t)warp * tiny_scr);
      for (;;) {
        int idx = 0;
        if (lane == 0) idx = atomicAdd(&sh.bnext, 1);
        idx = __shfl_sync(FULL, idx, 0);
        if (idx > k) break;
        Item ti = sh.first;
        unsigned long long q = sh.first_seq;
        if (idx > 0) {
          q = sh.claim_h + (unsigned long long)(idx - 1);
          // every lane waits for the item and reads it (one broadcast load);
          // a failed wait has set the error, and the run ends with it
          if (__any_sync(FULL, !fetch_item(P, q, ti))) break;
        }
        const bool done = ti.n <= tiny_lim && tiny_item(P, q, ti, scratch, sh.tst);
        __syncwarp();
        if (lane == 0) {
          if (done) {
            atomicAdd(&sh.bdone, 1);
          } else {
            const int at = atomicAdd(&sh.ncta, 1);
            sh.cta_item[at] = ti;
            sh.cta_seq[at] = q;
          }
        }
      }
      __threadfence();
      __syncthreads();
      if (threadIdx.x == 0 && sh.bdone > 0) {
        ReqCtx *Rg = &P.reqs[sh.first.req];
        long long *to[7] = {&Rg->items,     &Rg->alg_bytes, &Rg->peeled, &Rg->ni_passes,
                            &Rg->sw_phases, &Rg->accepted,  &Rg->splits};
#pragma unroll
        for (int z = 0; z < 7; ++z)
          if (sh.tst[z]) add_ll(to[z], (long long)sh.tst[z]);
        finish_items(P, sh.first.req, sh.bdone);
      }
      if (P.prof && threadIdx.x == 0) {
        const long long t = clock64();
        cp.tiny += t - pc;
        pc = t;
        ++cp.batches;
        cp.tiny_items += sh.bdone;
      }
    } else {
      if (threadIdx.x == 0) {
        sh.cta_item[0] = sh.first;
        sh.cta_seq[0] = sh.first_seq;
        sh.ncta = 1;
      }
      __syncthreads();
    }
    const int ncta = sh.ncta;
    for (int k = 0; k < ncta;) {
      // the part kept from the last item (under its index), else the next of
      // the batch
      const Item it = sh.has_own ? sh.own : sh.cta_item[k];
      const unsigned long long iseq = sh.cta_seq[k];
      __syncthreads();
      if (threadIdx.x == 0) sh.has_own = 0;
      if (P.prof && threadIdx.x == 0) {
        const long long t = clock64();
        for (int z = 0; z < 9; ++z) sh.ts[z] = t;
        sh.used_slab = 0;
        sh.pf_E = sh.pf_nalive = sh.pf_passes = sh.pf_nsv = -1;
        sh.pf_forest = sh.pf_nsv1 = 0;
        sh.pf_forest_cycles = 0;
        sh.pf_t0 = (long long)globaltimer_ns();
        for (int z = 0; z < 6; ++z) sh.fdbg[z] = 0;
        for (int z = 0; z < 4; ++z) sh.dbg[z] = 0;
      }
      __syncthreads();
      const int outcome = run_item(P, iseq, it, slab, sh);
      __syncthreads();
      if (P.prof && threadIdx.x == 0) {
        // fill skipped stamps forward, then record
        sh.ts[8] = clock64();
        for (int z = 1; z < 8; ++z)
          if (sh.ts[z] < sh.ts[z - 1]) sh.ts[z] = sh.ts[z - 1];
        const unsigned r = atomicAdd(P.prof_count, 1u);
        if (r < P.prof_cap) {
          ItemProf *q = &P.prof[r];
          q->seq = (unsigned)iseq;
          q->n = it.n;
          q->E = sh.pf_E;
          q->nalive = sh.pf_nalive;
          q->passes = sh.pf_passes;
          q->nsv = sh.pf_nsv;
          q->outcome = outcome;
          unsigned smid;
          asm("mov.u32 %0, %%smid;" : "=r"(smid));
          q->smid = (int)smid;
          q->slab = sh.used_slab;
          q->top = (int)(it.flags & ITEM_TOP);
          for (int z = 0; z < 8; ++z) q->dt[z] = (unsigned)(sh.ts[z + 1] - sh.ts[z]);
          q->t_begin = sh.pf_t0;
          q->t_end = (long long)globaltimer_ns();
          for (int z = 0; z < 4; ++z) q->dbg[z] = sh.dbg[z];
          q->forest = sh.pf_forest;
          q->nsv1 = sh.pf_nsv1;
          q->forest_cycles = sh.pf_forest_cycles;
          for (int z = 0; z < 6; ++z) q->fdbg[z] = sh.fdbg[z];
        }
      }
      if (threadIdx.x == 0) {
        finish_items(P, it.req, 1);
        // (only a chain needs it: the next claim looks too)
        if (sh.has_own) sh.go = vctr->error == 0;
      }
      __syncthreads();
      if (!sh.go) break;  // the run has failed: a chain of kept parts ends too
      if (P.prof && threadIdx.x == 0) {
        const long long t = clock64();
        cp.cta += t - pc;
        pc = t;
        ++cp.cta_items;
      }
      // an item is done with when none of its parts was kept
      if (!sh.has_own) ++k;
    }
    if (P.single_item) break;
  }
  if (P.prof && P.prof_cta && threadIdx.x == 0) P.prof_cta[blockIdx.x] = cp;
}

}  // namespace

size_t item_workspace_bytes(int64_t n, int64_t d) {
  return n < 65535 ? ws_bytes<uint16_t>(n, d) : ws_bytes<int32_t>(n, d);
}

int refine_block_threads() { return RB; }

// Largest dynamic shared memory a refinement CTA can opt into on this
// device: the per-block opt-in limit minus the kernel's static shared memory.
size_t refine_smem_max_bytes(int device) {
  int optin = 0;
  WCC_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device));
  cudaFuncAttributes fa;
  WCC_CUDA(cudaFuncGetAttributes(&fa, k_refine));
  size_t mx = (size_t)optin > fa.sharedSizeBytes ? (size_t)optin - fa.sharedSizeBytes : 0;
  mx &= ~(size_t)1023;
  return mx < SMEM_MAX_BYTES ? mx : SMEM_MAX_BYTES;
}

static void set_smem_attr(int device) {
  WCC_CUDA(cudaFuncSetAttribute(k_refine, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)refine_smem_max_bytes(device)));
}

int refine_max_ctas(int device, size_t smem_bytes) {
  set_smem_attr(device);
  int per_sm = 0;
  WCC_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_refine, RB, smem_bytes));
  int sms = 0;
  WCC_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device));
  int r = per_sm * sms;
  if (r < 1) fail(WCC_ERR_CUDA, "refinement kernel cannot be resident on this device");
  return r;
}

void launch_refine(const RefineParams &p, int grid, bool cooperative, cudaStream_t s) {
  int device = 0;
  WCC_CUDA(cudaGetDevice(&device));
  set_smem_attr(device);
  RefineParams pc = p;
  if (cooperative) {
    void *args[] = {&pc};
    WCC_CUDA(cudaLaunchCooperativeKernel((const void *)k_refine, dim3(grid), dim3(RB), args,
                                         p.smem_bytes, s));
    note_launch();
  } else {
    k_refine<<<grid, RB, p.smem_bytes, s>>>(pc); note_launch();
    WCC_CUDA(cudaGetLastError());
  }
}

}  // namespace wccg
