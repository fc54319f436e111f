// Device functions shared by the staged kernels (gs_kernels.cu) and the
// one-kernel matcher (gs_direct.cu).
#pragma once

#include "gs_engine.cuh"

namespace gs {

namespace {

constexpr int kThreads = 256;

__device__ __forceinline__ uint64_t gtid() { return blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; }
__device__ __forceinline__ uint64_t gthreads() { return (uint64_t)gridDim.x * blockDim.x; }

// ------------------------------------------------------------ bitmaps
// A candidate set over V is a three-level bitmap: W0 words of one bit per
// vertex, W1 summary words with one bit per non-zero level-0 word, and ipg
// words with one bit per non-zero group of 32 summary words (a "chunk" of
// 32,768 vertices).  Compaction and clearing visit only non-zero chunks.
__device__ __forceinline__ uint32_t *slot_of(const Wave &W, uint32_t gqv) { return W.bm + (uint64_t)gqv * W.slot_words; }
__device__ __forceinline__ bool bit_test(const uint32_t *slot, uint32_t v) { return (slot[v >> 5] >> (v & 31)) & 1u; }
__device__ __forceinline__ void bit_set(const Wave &W, uint32_t *slot, uint32_t v) {
  uint32_t old = atomicOr(&slot[v >> 5], 1u << (v & 31));
  if (old == 0) {
    uint32_t old1 = atomicOr(&slot[W.G.W0 + (v >> 10)], 1u << ((v >> 5) & 31));
    if (old1 == 0) atomicOr(&slot[W.G.W0 + W.G.W1 + (v >> 20)], 1u << ((v >> 15) & 31));
  }
}
__device__ __forceinline__ void bit_clear(uint32_t *slot, uint32_t v) { atomicAnd(&slot[v >> 5], ~(1u << (v & 31))); }

// Matching through a compressed graph (Section 3.5, Theorem 3.2): v can be
// a match of u only if the weighted node whose mapping list holds v is a
// candidate of u in the weighted graph.
__device__ __forceinline__ bool wmask_ok(const DQuery &Q, uint32_t u, uint32_t v) {
  if (!Q.wmask) return true;
  const uint32_t x = reinterpret_cast<const uint32_t *>(Q.wgroup)[v];
  const uint32_t *m = reinterpret_cast<const uint32_t *>(Q.wmask) + (uint64_t)u * Q.wstride;
  return (m[x >> 5] >> (x & 31)) & 1u;
}

// Candidate test of Definition 3.3 read per direction and relation: binding,
// type, and for every (direction, relation) at least as many distinct data
// neighbours as the query vertex has query neighbours.
__device__ __forceinline__ bool cand_ok(const DevGraph &G, const DQuery &Q, uint32_t u, uint32_t v) {
  uint32_t b = Q.vbind[u];
  if (b != kUnbound && b != v) return false;
  uint32_t t = Q.vtype[u];
  if (t != kAny && G.vtype[v] != t) return false;
  if (!wmask_ok(Q, u, v)) return false;
  for (uint32_t i = Q.need_begin[u]; i < Q.need_begin[u + 1]; ++i) {
    uint32_t w = G.sig[(uint64_t)Q.need_plane[i] * G.sig_words + (v >> 3)];
    if (((w >> ((v & 7) * 4)) & 15u) < Q.need_cnt[i]) return false;
  }
  return true;
}

// ------------------------------------------------------------ plan
// Section 3.5 ("Modify the query plan"): start at the bound vertex of largest
// degree; with no bound vertex, Section 3.3.2 ranks by deg(u)/freq(type(u)),
// which this plan refines into the expected size of u's filtered set (type
// frequency times, per degree need, the measured fraction of that type's
// vertices meeting it), so the exploration starts from the fewest
// candidates; then repeatedly explore the already-covered vertex with the
// most uncovered neighbours until every vertex is covered.  The explored vertices
// form the visit order; each newly covered vertex hangs below the vertex that
// covered it (the spanning tree T).
// A warp plans a query in shared memory, lane u for vertex u.  Every incident
// edge of every vertex is packed for exploration and refinement: direction,
// relation, other endpoint and, for a vertex that is explored (leaves of the
// spanning tree are not), the endpoint's role at that step (0: set not built
// yet, 1: set built, 2: child initialised now).  STAGED: with the options
// only the staged kernels run (a fixed root, the refinement variants).
template <bool STAGED>
__device__ __forceinline__ void plan_query(const DevGraph &G, DQuery &Q) {
  const uint32_t u = threadIdx.x & 31, k = Q.k;
  uint32_t nbr = 0;
  float est = 0.f;
  if (u < k) {
    for (uint32_t i = Q.inc_begin[u]; i < Q.inc_begin[u + 1]; ++i) {
      const uint32_t e = Q.inc_edge[i];
      nbr |= 1u << (Q.esrc[e] == u ? Q.edst[e] : Q.esrc[e]);
    }
  }
  const uint32_t bound = __ballot_sync(kFull, u < k && Q.vbind[u] != kUnbound);
  int root = -1;
  if (STAGED && Q.force_root != 0xFF) {
    root = Q.force_root;
  } else if (bound) {  // the bound vertex of most neighbours
    const uint32_t deg = (bound >> u) & 1u ? __popc(nbr) + 1u : 0u;
    const uint32_t most = __reduce_max_sync(kFull, deg);
    root = __ffs(__ballot_sync(kFull, deg == most)) - 1;
  } else {  // the smallest expected filtered set (ties: more neighbours)
    if (u < k) {
      const uint32_t P = 2 * G.R + 2, t = Q.vtype[u] == kAny ? G.T : Q.vtype[u];
      const float f = (float)(t == G.T ? G.V : G.toff[t + 1] - G.toff[t]);
      est = f;
      for (uint32_t i = Q.need_begin[u]; i < Q.need_begin[u + 1] && f > 0.f; ++i)
        est *= (float)G.sigge[((uint64_t)t * P + Q.need_plane[i]) * 16 + Q.need_cnt[i]] / f;
    }
    float best = 0.f;
    int most = 0;
    for (uint32_t x = 0; x < k; ++x) {
      const float e = __shfl_sync(kFull, est, x);
      const int n = __popc(__shfl_sync(kFull, nbr, x));
      if (root < 0 || e < best || (e == best && n > most)) {
        root = (int)x;
        best = e;
        most = n;
      }
    }
  }
  const uint32_t all = (1u << k) - 1;  // k is at most 16
  uint32_t covered = 1u << root, seen = 0, nv = 0, cur = (uint32_t)root;
  uint32_t parent = 0xFF, pedge = 0xFF, init = u == cur ? 0u : 0xFFu, at_step = 0xFF;
  for (;;) {
    if (u == cur) at_step = nv;
    if (u == 0) Q.visit[nv] = (uint8_t)cur;
    seen |= 1u << cur;
    const uint32_t fresh = __shfl_sync(kFull, nbr, cur) & ~covered;
    if ((fresh >> u) & 1u) {
      parent = cur;
      init = nv + 1;
      for (uint32_t i = Q.inc_begin[cur]; i < Q.inc_begin[cur + 1]; ++i) {
        const uint32_t e = Q.inc_edge[i];
        if ((Q.esrc[e] == cur ? Q.edst[e] : Q.esrc[e]) == u) {
          pedge = e;
          break;
        }
      }
    }
    covered |= fresh;
    ++nv;
    if (covered == all) break;
    const uint32_t c = ((covered & ~seen) >> u) & 1u ? __popc(nbr & ~covered) : 0u;
    const uint32_t most = __reduce_max_sync(kFull, c);
    if (most == 0) break;  // disconnected (the host rejects these)
    cur = __ffs(__ballot_sync(kFull, c == most)) - 1;
  }
  if (u < kMaxK) {
    Q.parent[u] = (uint8_t)parent;
    Q.pedge[u] = (uint8_t)pedge;
    Q.init_step[u] = (uint8_t)init;
  }
  if (u == 0) {
    Q.nvisit = nv;
    Q.status = covered == all ? QS_OK : QS_INVALID;
  }
  __syncwarp();
  if (u < k)
    for (uint32_t i = Q.inc_begin[u]; i < Q.inc_begin[u + 1]; ++i) {
      const uint32_t e = Q.inc_edge[i], dir = Q.esrc[e] == u ? 0u : 1u, w = dir == 0 ? Q.edst[e] : Q.esrc[e];
      uint32_t role = 0;
      if (at_step != 0xFF) {
        role = Q.init_step[w] <= at_step ? 1u : 0u;
        if (Q.parent[w] == u && Q.init_step[w] == at_step + 1 && Q.pedge[w] == e) role = 2u;
        // the baseline checks only spanning-tree edges it can follow forwards
        if (STAGED && (Q.refine_flags & kRefineBase) && (role != 2u || dir != 0u)) role = 3u;
      }
      Q.xinc[i] = xinc_pack(dir, Q.erel[e], w, role);
    }
  // reversed refinement order (only when asked for): vertices by the step
  // that gave them a candidate set, last first (ties: higher index first);
  // u's position is the number of vertices that come before it
  if (STAGED && (Q.refine_flags & kRefineRev) && u < k) {
    uint32_t before = 0;
    for (uint32_t w = 0; w < k; ++w) {
      const uint32_t iw = Q.init_step[w];
      before += iw > init || (iw == init && w > u);
    }
    Q.rorder[before] = (uint8_t)u;
  }
  __syncwarp();
}

// Algorithmic bytes: each thread accumulates in a register; at the end of
// the kernel one warp-reduced atomic per warp adds them up (statistics runs
// only).  Every lane of the warp must reach flush_bytes.
__device__ __forceinline__ void flush_bytes(const Wave &W, int kind, uint64_t b) {
  if (!W.stats) return;
  for (int o = 16; o; o >>= 1) b += __shfl_down_sync(kFull, b, o);
  if ((threadIdx.x & 31) == 0 && b) atomicAdd((unsigned long long *)&W.ctrl->bytes[kind], (unsigned long long)b);
}

__device__ __forceinline__ void mark(DQuery &Q, uint32_t st) { atomicCAS(&Q.status, QS_OK, st); }

// Restore every touched bitmap word to zero (only chunks flagged at level 2
// and words flagged at level 1 are visited), so the slots are clean for the
// next run.
__device__ __forceinline__ void clear_sets(const Wave &W) {
  const DevGraph &G = W.G;
  const uint32_t lane = threadIdx.x & 31;
  const uint64_t warps = gthreads() / 32;
  const uint64_t items = (uint64_t)W.nqv * G.ipg;
  for (uint64_t it = gtid() / 32; it < items; it += warps) {
    const uint32_t gqv = (uint32_t)(it / G.ipg), grp = (uint32_t)(it % G.ipg);
    uint32_t *slot = slot_of(W, gqv);
    uint32_t m2 = slot[G.W0 + G.W1 + grp];
    while (m2) {
      const uint32_t c = grp * 32 + (__ffs(m2) - 1);
      m2 &= m2 - 1;
      const uint32_t w1 = c * 32 + lane;
      const uint32_t sw = w1 < G.W1 ? slot[G.W0 + w1] : 0;
      uint32_t m = __ballot_sync(kFull, sw != 0);
      while (m) {
        const int j = __ffs(m) - 1;
        m &= m - 1;
        const uint32_t swj = __shfl_sync(kFull, sw, j);
        if ((swj >> lane) & 1u) slot[(c * 32 + j) * 32 + lane] = 0;
      }
      if (sw) slot[G.W0 + w1] = 0;
    }
    __syncwarp();
    if (lane == 0) slot[G.W0 + G.W1 + grp] = 0;
  }
}

__device__ __forceinline__ bool rows_wanted(const DQuery &Q) { return Q.mode != GS_COUNT_ONLY && Q.cap; }

// A query's outcome after the one-kernel matcher, and the place of its rows:
// those that left in one segment stay there, several get room for all.
// need_rows, need_words: the caller's sums of what outputs take of the pools.
// open: tasks of the run that no warp took (every wait is bounded); its
// queries start over.
__device__ __forceinline__ void direct_layout(const Wave &W, uint32_t qi, uint32_t open, uint64_t &need_rows,
                                              uint64_t &need_words) {
  DQuery &Q = W.dq[qi];
  QState &S = W.qs[qi];
  DState &D = W.d.ds[qi];
  const uint32_t k = Q.k;
  uint64_t inter = 0, peak = 0;
#pragma unroll
  for (uint32_t l = 0; l + 1 < kMaxK; ++l) {  // all loads together
    const uint64_t w = l + 1 < k ? D.lv[l] * (l + 1) : 0;
    inter += w;
    peak = w > peak ? w : peak;
  }
  S.inter_words = inter;
  S.peak_words = peak;
  S.out_rows = 0;
  if (open && Q.status != QS_INVALID) Q.status = QS_OVERFLOW;
  if (Q.status != QS_OK || !rows_wanted(Q)) return;
  if (S.count > over_cap_rows(Q.cap)) {
    Q.status = QS_TOPCAP;
    return;
  }
  // What this output takes of the pools, whether or not there was room: the
  // host enlarges them by it.  Outputs that end on the chunked path are not
  // in it, so a query that found no room because of them does in a second
  // pass.
  const uint64_t n = S.count, words = n * Q.k;
  need_rows += n;
  need_words += D.nseg == 1 && !D.over ? words : 2 * words;
  bool fits = !D.over;
  if (fits) {  // room that does not suffice is given back for smaller outputs
    fits = atomicAdd((unsigned long long *)&W.ctrl->out_rows_total, (unsigned long long)n) + n <= W.out_rows_cap;
    if (!fits) atomicAdd((unsigned long long *)&W.ctrl->out_rows_total, ~(unsigned long long)n + 1);
  }
  if (fits && D.nseg > 1) {
    D.word = atomicAdd((unsigned long long *)&W.ctrl->out_top, (unsigned long long)words);
    fits = D.word + words <= W.out_words;
    if (!fits) atomicAdd((unsigned long long *)&W.ctrl->out_top, ~(unsigned long long)words + 1);
  }
  if (!fits) {
    Q.status = QS_OVERFLOW;
    return;
  }
  S.out_rows = n;
  S.out_row_base = 0;
  S.out_word_base = D.word;
}

// splitmix64 finaliser (Steele, Lea & Flood 2014); row hash for fingerprints.
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

}  // namespace

}  // namespace gs
