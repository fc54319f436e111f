// The one-kernel matcher: exploration (kernel_explore) and join
// (combine_edge_candidates) of a whole batch in one persistent kernel over a
// work queue, for runs without refinement rounds.
//
// The staged pipeline (gs_kernels.cu) runs every step of every query as a
// launch of its own: 65 to 150 launches for one call, each with a handful of
// items per query and a drain behind its slowest item.  Here a warp takes a
// query and walks it through all of its steps, so steps of different queries
// overlap freely and a step costs a warp barrier instead of a launch; only a
// step with many candidates, or a join with many partial embeddings while
// other warps have nothing to do, is cut into tasks that others take from a
// queue.  Candidate sets stay the three-level bitmaps of the staged path,
// with a count of live bits per set; the join reads the adjacency rows and
// those bitmaps directly, so there are no candidate lists, candidate-edge
// tables, count passes, scans or row allocators.
//
// What bounds it: chains of dependent loads of random vertices (row offsets,
// row entries, type and signature, bitmap word), so the design is about many
// chains in flight: one candidate or row per lane for the row look-ups, the
// rows' entries dealt out evenly over the lanes with several loads per lane,
// and as many warps as the registers allow.  Measured against the staged
// pipeline as default calls ran it (32 lanes per item, up to eight refinement
// rounds), device time of one batch: one query on the 1M-vertex graph 0.39 ->
// 0.25 ms, 2,001 queries on the 4M-vertex graph 5.7 -> 2.6, 5,000 there 27.0
// -> 8.3, 200 shape queries on the 16M-vertex graph 21.9 -> 9.2; this kernel
// was 1.7, 4.6 and 6.9 ms of the last three.  With the plan and the filter
// inside (six launches and a grid-wide pass less) the four are 0.20, 2.3, 7.4
// and 7.5 ms a batch, the last 6.7 with the task sizes below.  A block of 256 threads per query
// instead of a warp took 2.8, 13.1 and 16.6: its barriers and idle lanes cost
// more than the wider steps gained.
//
// Nothing waits for another warp: one that finds no work polls a bounded
// number of times and leaves, and whatever is queued then is taken by the
// warps that are still there.
#include <algorithm>

#include "gs_device.cuh"

namespace gs {

namespace {

// Workers per block, and blocks per SM: 24 warps of 80 registers.  More warps
// are no faster (32 of 64 registers: 5,000 queries on the 4M-vertex graph 7.7
// ms a batch instead of 7.4, 40 and 48 warps 9.4 and 10.0), fewer cost large
// batches more than they give single queries (16: 9.2 ms), and blocks of two
// start a single query sooner than blocks of four (0.116 ms against 0.128).
constexpr int kWarps = 2;
constexpr int kBlocksPerSm = 12;
constexpr uint32_t kLvlCap = 256;     // partial embeddings per level of a worker's scratch
constexpr uint32_t kRootCap = 4096;   //   and candidates of the first joined vertex
constexpr uint32_t kVCap = 1024;      // next candidates of a batch of rows
constexpr uint32_t kListCap = 512;    // ids kept beside a set while one worker builds it
constexpr uint32_t kU = 4;            // neighbours per lane and pass: independent loads in flight
constexpr uint32_t kQueue = 32 + 256; // fewer than 32 left over and one pass of the filter
constexpr uint32_t kLvlWords = (kMaxK * (kMaxK + 1) / 2 - 1) * kLvlCap;  // levels 1 to 15
constexpr uint32_t kScratch = kRootCap + kLvlWords + kMaxK * kVCap + kMaxK * kListCap;  // words per worker
constexpr uint32_t kShareMin = 32;    // rows left at a level for idle workers to be given some
constexpr unsigned long long kNoSlot = ~0ull;
constexpr uint32_t kMostPolls = 1u << 23;  // every wait ends there, although none is known to come near it
constexpr uint32_t kNoPiece = 0xFFFFFFFFu;

enum : uint32_t { TK_START = 1, TK_EXPLORE, TK_ROOT, TK_ROWS, TK_EXIT };

// A worker's state in shared memory.
struct __align__(8) Worker {
  DQuery Q;
  uint32_t lc[kMaxK];  // ids listed per query vertex ...
  uint32_t listed;     //   and the vertices whose lists hold their whole sets
  // join plan: order, position of each vertex, edges of each level's vertex
  // to the joined part (column, adjacency plane and relation of each)
  uint8_t order[kMaxK], pos[kMaxK], ebeg[kMaxK + 1], ecol[kMaxM], epl[kMaxM], erel[kMaxM];
  // join levels: rows, rows done, rows in hand, next candidates written out
  // of those in hand, entries of a long run done and the rows that share it
  // (0 unless parts of it are still to come)
  uint32_t ln[kMaxK], lr[kMaxK], hb[kMaxK], lt[kMaxK], lo[kMaxK], lg[kMaxK];
  uint16_t vb[kMaxK][32], vc[kMaxK][32];  // next candidates of each row in hand: first, number
  uint32_t vn[32];
  uint16_t cmp[kMaxK];  // columns that can hold the vertex joined at a level
  unsigned long long lv[kMaxK];  // rows made per level
  uint32_t queue[kQueue];  // neighbours, or positions of the filter, that passed a first test
  unsigned long long ticket;  // position this worker serves, kept while it starts queries (kNoSlot: none)
  uint32_t part;   // part of the ring that the task in hand is still to be counted in (kRingParts: none)
  uint32_t piece;  // shared rows that the task in hand started from (kNoPiece: none)
  uint32_t full;  // rows of this task are no longer kept: the query leaves the device, or the pool is full
};

__device__ __forceinline__ uint32_t ldv(const uint32_t *p) { return *reinterpret_cast<const volatile uint32_t *>(p); }
__device__ __forceinline__ unsigned long long ldv(const unsigned long long *p) {
  return *reinterpret_cast<const volatile unsigned long long *>(p);
}
__device__ __forceinline__ void add_release(uint32_t *p, uint32_t x) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(x) : "memory");
}
__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31; }
__device__ __forceinline__ uint32_t worker_id() { return blockIdx.x * kWarps + (threadIdx.x >> 5); }
__device__ __forceinline__ uint32_t below_me() { return (1u << lane_id()) - 1; }
__device__ __forceinline__ uint32_t *scratch_of(const Wave &W) { return W.d.scratch + (uint64_t)worker_id() * kScratch; }

// Is v a live candidate?  Sets change while a query is explored and are read
// past the first-level cache then; by the time of its join they are final.
__device__ __forceinline__ bool bit_live(const uint32_t *slot, uint32_t v) { return (__ldcg(slot + (v >> 5)) >> (v & 31)) & 1u; }
__device__ __forceinline__ bool bit_final(const uint32_t *slot, uint32_t v) { return (__ldca(slot + (v >> 5)) >> (v & 31)) & 1u; }

// Exclusive prefix over the warp and its total.
__device__ __forceinline__ uint32_t warp_excl(uint32_t x, uint32_t &total) {
  uint32_t y = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t z = __shfl_up_sync(kFull, y, o);
    if (lane_id() >= o) y += z;
  }
  total = __shfl_sync(kFull, y, 31);
  return y - x;
}

// The lane that owns item t of runs laid out back to back, lane i's from ex
// on: the last with ex <= t.  Every lane calls it.
__device__ __forceinline__ uint32_t owner_of(uint32_t ex, uint32_t t) {
  uint32_t i = 0;
#pragma unroll
  for (uint32_t s = 16; s; s >>= 1)
    if (__shfl_sync(kFull, ex, i + s) <= t) i += s;
  return i;
}

// First index in [l, h) whose entry is at least `key`, by one thread: eight
// probes at a time, so that a row of up to eight entries takes one load
// latency and one of up to 80 takes two.
__device__ __forceinline__ uint32_t lower8(const uint32_t *a, uint32_t l, uint32_t h, uint32_t key) {
  while (h - l > 8) {
    const uint32_t step = (h - l + 8) / 9;
    uint32_t c = 0;
#pragma unroll
    for (uint32_t i = 1; i <= 8; ++i) {
      const uint32_t p = l + i * step - 1;
      c += (p < h ? __ldg(a + p) : 0xFFFFFFFFu) < key;
    }
    l += c * step;
    if (c < 8) h = min(h, l + step - 1);
  }
  uint32_t c = 0;
#pragma unroll
  for (uint32_t i = 0; i < 8; ++i) c += (l + i < h ? __ldg(a + l + i) : 0xFFFFFFFFu) < key;
  return l + c;
}

// Relation run of v's row in an adjacency plane, by one thread.
__device__ __forceinline__ void run_of(const DevGraph &G, uint32_t plane, uint32_t rel, uint32_t v, uint32_t &lo,
                                       uint32_t &len) {
  const uint64_t *off = G.off[plane] + v;
  const uint32_t *a = G.adj[plane];
  uint32_t l = (uint32_t)__ldg(off);
  const uint32_t e = (uint32_t)__ldg(off + 1);
  const uint32_t k0 = rel << kNbrBits, k1 = k0 + (1u << kNbrBits);
  if (e - l > 8) l = lower8(a, l, e, k0);
  uint32_t c0 = 0, c1 = 0;  // entries of the next eight before the run, and before its end
#pragma unroll
  for (uint32_t i = 0; i < 8; ++i) {
    const uint32_t x = l + i < e ? __ldg(a + l + i) : 0xFFFFFFFFu;
    c0 += x < k0;
    c1 += x < k1;
  }
  lo = l + c0;
  len = (c1 < 8 ? l + c1 : lower8(a, l + 8, e, k1)) - lo;
}

// Is (rel, x) in v's row of the plane?
__device__ __forceinline__ bool has_nbr(const DevGraph &G, uint32_t plane, uint32_t rel, uint32_t v, uint32_t x) {
  const uint64_t *off = G.off[plane] + v;
  const uint32_t *a = G.adj[plane];
  const uint32_t key = (rel << kNbrBits) | x, e = (uint32_t)__ldg(off + 1);
  const uint32_t l = lower8(a, (uint32_t)__ldg(off), e, key);
  return l < e && __ldg(a + l) == key;
}

// ------------------------------------------------------------ the queue
// Tasks are appended to a ring of slots; positions in it only grow, and a
// slot's flag says for which of its turns it is filled.  A worker that wants a
// task takes a ticket, the position it will serve, and polls that slot: no two
// workers poll or swap the same word, so thousands of waiting workers cost the
// working ones nothing (a shared head moved by compare-and-swap handed out a
// task a microsecond at best, 38.6 ms instead of 2.8 for 2,001 queries on the
// 4M-vertex graph).  Tickets past the last reserved position are the workers
// without work.  Slots come free a part of the ring at a time, in order, when
// every task of the part has been taken (not when it is finished: one long
// join task would hold up the ring); with none free a worker does its work itself.
// A ticket is kept while its holder starts queries.  Where half of the ring is
// in use the join of such a query, which can be long, goes to the queue, so
// that the ticket is served soon (always doing so cost 60,000 queries 6 %,
// handing the ticket back as below as soon as it turned out to be past the
// last reserved position 5 %).  The worker that finishes the last query ends the wait of the others
// through their slots.
//
// Workers that wait leave in the reverse order of their tickets: the holder of
// the last ticket takes it back, so the tickets from `tail` on are always
// those of workers that are there.  A slot whose ticket was taken back is
// served by whoever takes that ticket next, at the latest the worker that
// filled the slot.  More than Direct::keep workers wait for idle_polls polls
// (some milliseconds) at most, so that kernels of other streams find room
// beside a long query; the others wait for half a second.
__device__ __forceinline__ uint32_t idle_workers(const Wave &W) {
  const unsigned long long h = ldv(&W.d.ctl->head), t = ldv(&W.d.ctl->tail);
  return h > t ? (uint32_t)(h - t) : 0;
}
__device__ __forceinline__ DTask &slot_at(const Wave &W, unsigned long long pos) {
  return W.d.tasks[pos & ((1ull << W.d.task_log) - 1)];
}
__device__ __forceinline__ uint32_t turn_of(const Wave &W, unsigned long long pos) {
  return W.d.ctl->turn + (uint32_t)(pos >> W.d.task_log);
}

// The oldest parts of the ring whose tasks have all been taken come free.
__device__ __forceinline__ void free_parts(const Wave &W) {
  DCtl *c = W.d.ctl;
  const uint32_t size = 1u << (W.d.task_log - kRingPartsLog);
  for (uint32_t i = 0; i < kRingParts; ++i) {
    const uint32_t p = ldv(&c->part), at = p % kRingParts;
    if (ldv(&c->taken[at]) != size) return;
    if (atomicCAS(&c->part, p, p + 1) != p) continue;
    c->taken[at] = 0;
    __threadfence();
    atomicAdd(&c->room, size);
  }
}

// Room for n tasks: their first position, or none (the caller then does the
// work itself; before it fills them, a fence).  One lane.
__device__ unsigned long long reserve(const Wave &W, uint32_t n) {
  DCtl *c = W.d.ctl;
  for (int again = 1; (int)atomicSub(&c->room, n) < (int)n; --again) {
    atomicAdd(&c->room, n);
    if (!again) return kNoSlot;
    free_parts(W);
  }
  atomicAdd(&c->open, n);
  return atomicAdd(&c->tail, (unsigned long long)n);
}

// A task into a reserved slot.
__device__ __forceinline__ void push(const Wave &W, uint32_t kind, uint32_t q, uint32_t step, uint32_t a, uint32_t b,
                                     unsigned long long slot) {
  DTask &t = slot_at(W, slot);
  t.kind = kind; t.q = q; t.step = step; t.a = a; t.b = b;
  __threadfence();
  atomicExch(&t.flag, turn_of(W, slot));
}

// May the holder of `ticket`, after `spin` polls, leave?  Takes the ticket
// back if so.
__device__ __forceinline__ bool leave(const Wave &W, unsigned long long ticket, uint32_t spin) {
  DCtl *c = W.d.ctl;
  const unsigned long long h = ldv(&c->head);
  if (h != ticket + 1) return false;  // those with later tickets go first
  if (spin < W.d.keep_polls && h <= ldv(&c->tail) + W.d.keep) return false;
  return atomicCAS(&c->head, ticket + 1, ticket) == ticket + 1;
}

struct Task {
  uint32_t kind, q, step, a, b;
};

// The next task; one lane.
__device__ Task fetch(const Wave &W, Worker &K) {
  DCtl *c = W.d.ctl;
  unsigned long long ticket = K.ticket;
  for (uint32_t spin = 0; spin < kMostPolls; ++spin) {
    const bool queries = ldv(&c->next) < W.nq;
    if (ticket == kNoSlot && (!queries || ldv(&c->head) < ldv(&c->tail))) {
      ticket = atomicAdd(&c->head, 1ull);
      __threadfence();
      if (!queries && ldv(&c->open) == 0) return Task{TK_EXIT, 0, 0, 0, 0};
    }
    if (ticket != kNoSlot) {
      DTask &t = slot_at(W, ticket);
      const uint32_t ready = turn_of(W, ticket);
      // no query left to start: this slot alone is polled (now and then the
      // number of open tasks, in case the wait was to end before the ticket)
      if (!queries)
        for (; ldv(&t.flag) != ready; ++spin) {
          if (spin >= kMostPolls) return Task{TK_EXIT, 0, 0, 0, 0};
          if ((spin & (spin < W.d.idle_polls ? 63u : 15u)) == 0 &&
              (ldv(&c->open) == 0 || (spin >= W.d.idle_polls && leave(W, ticket, spin))))
            return Task{TK_EXIT, 0, 0, 0, 0};
          __nanosleep(100);
        }
      if (ldv(&t.flag) == ready) {
        __threadfence();
        const Task T{__ldcg(&t.kind), __ldcg(&t.q), __ldcg(&t.step), __ldcg(&t.a), __ldcg(&t.b)};
        // the slot may be filled anew once this is seen; a short task says so
        // when it is done, where a fence comes anyway
        K.part = (uint32_t)(ticket >> (W.d.task_log - kRingPartsLog)) % kRingParts;
        if (T.kind != TK_EXPLORE) {
          add_release(&c->taken[K.part], 1u);
          K.part = kRingParts;
        }
        K.ticket = kNoSlot;
        return T;
      }
    }
    if (queries) {
      const uint32_t q = atomicAdd(&c->next, 1u);
      if (q < W.nq) {
        K.ticket = ticket;
        K.part = kRingParts;
        return Task{TK_START, q, 0, 0, 0};
      }
    }
  }
  return Task{TK_EXIT, 0, 0, 0, 0};
}

// A task or query is finished; the last one ends every wait.
__device__ void task_done(const Wave &W, Worker &K) {
  DCtl *c = W.d.ctl;
  uint32_t last = 0;
  if (lane_id() == 0) {
    __threadfence();
    if (K.part < kRingParts) atomicAdd(&c->taken[K.part], 1u);
    if (K.piece != kNoPiece) atomicExch(W.d.piece_of + K.piece, 0u);
    K.piece = kNoPiece;
    last = atomicSub(&c->open, 1u) == 1;
    __threadfence();
  }
  if (!__shfl_sync(kFull, last, 0)) return;
  const unsigned long long t = ldv(&c->tail), h = ldv(&c->head);
  const uint32_t turn = c->turn;
  for (unsigned long long i = t + lane_id(); i < h; i += 32) slot_at(W, i).kind = TK_EXIT;
  __threadfence();
  for (unsigned long long i = t + lane_id(); i < h; i += 32) atomicExch(&slot_at(W, i).flag, turn + (uint32_t)(i >> W.d.task_log));
}

// ------------------------------------------------------------ sets as ids
// The next ids of a set from level-0 word `cur` on (below `end`), at most
// `cap` of them, into `list`; moves `cur`.  A sparse set goes by its summary
// words, eight per lane (262,144 vertices) and pass, a dense one by its
// words, four per lane.  Order does not matter: rows are sorted at the end.
// cap is at least the 4,096 ids of a dense pass.
__device__ uint32_t refill(const Wave &W, const uint32_t *slot, uint32_t &cur, uint32_t end, bool &dense,
                           uint32_t *list, uint32_t cap) {
  uint32_t have = 0;
  const uint32_t *l1 = slot + W.G.W0;
  while (cur < end) {
    if (!dense) {
      const uint32_t w1 = cur >> 5, e1 = (end + 31) >> 5;  // cur is a whole summary word here
      uint32_t w[8], n = 0, total;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const uint32_t i = w1 + j * 32 + lane_id();
        w[j] = i < e1 ? __ldcg(l1 + i) : 0;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j)
        for (uint32_t m = w[j]; m; m &= m - 1)
          n += __popc(__ldcg(slot + (w1 + j * 32 + lane_id()) * 32 + __ffs(m) - 1));
      uint32_t p = have + warp_excl(n, total);
      if (total > cap) {
        dense = true;
        continue;
      }
      if (have + total > cap) break;
      if (n) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          for (uint32_t m = w[j]; m; m &= m - 1) {
            const uint32_t i = (w1 + j * 32 + lane_id()) * 32 + __ffs(m) - 1;
            for (uint32_t x = __ldcg(slot + i); x; x &= x - 1) list[p++] = i * 32 + __ffs(x) - 1;
          }
      }
      have += total;
      cur += 256 * 32;
    } else {
      uint32_t x[4], n = 0, total;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint32_t i = cur + j * 32 + lane_id();
        x[j] = i < end ? __ldcg(slot + i) : 0;
        n += __popc(x[j]);
      }
      uint32_t p = have + warp_excl(n, total);
      if (have + total > cap) break;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        for (uint32_t m = x[j]; m; m &= m - 1) list[p++] = (cur + j * 32 + lane_id()) * 32 + __ffs(m) - 1;
      have += total;
      cur += 128;
    }
  }
  __syncwarp();
  return have;
}

// The ids of query vertex w's set as this worker lists them while it builds
// the set.
__device__ __forceinline__ uint32_t *list_of(const Wave &W, uint32_t w) {
  return scratch_of(W) + kRootCap + kLvlWords + kMaxK * kVCap + w * kListCap;
}
__device__ __forceinline__ bool listed(const Worker &K, uint32_t w) { return ((K.listed >> w) & 1u) && K.lc[w] <= kListCap; }

// ------------------------------------------------------------ exploration
// Set v's bit; true when it was clear.  The summary bits of a set that is
// still small are set without waiting for an answer; a large set's would meet
// in few words, so there only the first to touch a word goes on.
__device__ __forceinline__ void raise(const Wave &W, uint32_t *slot, uint32_t v, bool few) {
  uint32_t *l1 = &slot[W.G.W0 + (v >> 10)], *l2 = &slot[W.G.W0 + W.G.W1 + (v >> 20)];
  const uint32_t b1 = 1u << ((v >> 5) & 31), b2 = 1u << ((v >> 15) & 31);
  if (few) {
    atomicOr(l1, b1);
    atomicOr(l2, b2);
  } else if (atomicOr(l1, b1) == 0) {
    atomicOr(l2, b2);
  }
}

// Candidates list[0, n) of the visited vertex u: a candidate stays when every
// query edge at u has a data neighbour that passes (a live candidate of the
// other endpoint where its set is built, else the candidate test), and its
// neighbours over tree edges that pass join the children's sets.  One lane
// per candidate finds the relation runs of an edge; the runs' entries are
// then dealt out over the lanes, so that a hub's long run is no lane's own.
// At step 0 the candidates come from the filter and are in no set yet: those
// that stay join u's.
__device__ __forceinline__ void explore_list(const Wave &W, Worker &K, uint32_t u, uint32_t step, const uint32_t *list,
                                             uint32_t n, uint64_t &acc) {
  const DQuery &Q = K.Q;
  const DevGraph &G = W.G;
  uint32_t *us = slot_of(W, Q.qv_base + u);
  const uint32_t i0 = Q.inc_begin[u], i1 = Q.inc_begin[u + 1];
  const bool masked = step == 0 && Q.vbind[u] == kUnbound && Q.vtype[u] != kAny;
  for (uint32_t r0 = 0; r0 < n; r0 += 32) {
    const bool mine = r0 + lane_id() < n;
    const uint32_t v = mine ? list[r0 + lane_id()] : 0;
    bool live = mine;
    // neighbour-type masks first: one load per edge drops most candidates
    if (live && !masked)
      for (uint32_t i = i0; i < i1; ++i) {
        const uint32_t xi = Q.xinc[i], t = Q.vtype[xinc_w(xi)];
        if (t == kAny) continue;
        const uint32_t m = __ldg(G.tmask + (uint64_t)sig_plane(xinc_dir(xi), xinc_rel(xi), G.R) * G.V + v);
        live = live && ((m >> (t & 31u)) & 1u);
      }
    if (mine) acc += 4 + 4ull * (i1 - i0);
    for (uint32_t ii = 0; ii < 2 * (i1 - i0); ++ii) {  // edges to children last: dropped candidates expand nothing
      const bool child = ii >= i1 - i0;
      const uint32_t xi = Q.xinc[i0 + (child ? ii - (i1 - i0) : ii)], role = xinc_role(xi), w = xinc_w(xi);
      if ((role == 2) != child) continue;
      const uint32_t want = __ballot_sync(kFull, live);
      if (!want) break;
      const uint32_t plane = adj_plane(xinc_dir(xi), xinc_rel(xi));
      uint32_t lo = 0, len = 0, total, found = 0;
      if (live) {
        run_of(G, plane, adj_rel(xinc_rel(xi)), v, lo, len);
        acc += 16;
      }
      const uint32_t ex = warp_excl(len, total);
      uint32_t *ws = slot_of(W, Q.qv_base + w);
      const uint32_t tw = Q.vtype[w], bw = Q.vbind[w];
      const uint32_t *adj = G.adj[plane];
      if (lane_id() == 0) acc += (uint64_t)total * (role == 1 ? 8 : (tw != kAny ? 5 : 4));
      // The entries, kU per lane and pass.  Those of the right type (most are
      // not) queue up in shared memory, so that the rest of the candidate test
      // and the set's update run with full warps.
      const uint32_t had = K.lc[w];
      uint32_t have = had, t0 = 0, queued = 0;
      for (;;) {
        if (!child && (found & want) == want) break;
        if (queued < 32 && t0 < total) {
          uint32_t x[kU];
          bool ok[kU];
#pragma unroll
          for (uint32_t j = 0; j < kU; ++j) {
            const uint32_t it = t0 + j * 32 + lane_id(), own = owner_of(ex, it);
            const uint32_t at = __shfl_sync(kFull, lo - ex, own) + it;
            ok[j] = it < total;
            x[j] = (ok[j] ? __ldg(adj + at) & kNbrMask : 0) | (own << kNbrBits);
          }
#pragma unroll
          for (uint32_t j = 0; j < kU; ++j) {
            const uint32_t v2 = x[j] & kNbrMask;
            if (role == 1) ok[j] = ok[j] && bit_live(ws, v2);
            else if (tw != kAny) ok[j] = ok[j] && __ldg(G.vtype + v2) == tw;
            if (bw != kUnbound) ok[j] = ok[j] && v2 == bw;
          }
          if (role == 1) {
            uint32_t mine_found = 0;
#pragma unroll
            for (uint32_t j = 0; j < kU; ++j) mine_found |= ok[j] ? 1u << (x[j] >> kNbrBits) : 0u;
            found |= __reduce_or_sync(kFull, mine_found);
          } else {
#pragma unroll
            for (uint32_t j = 0; j < kU; ++j) {
              const uint32_t m = __ballot_sync(kFull, ok[j]);
              if (ok[j]) K.queue[queued + __popc(m & below_me())] = x[j];
              queued += __popc(m);
            }
            __syncwarp();
          }
          t0 += 32 * kU;
          continue;
        }
        if (queued == 0) break;
        const uint32_t take = min(queued, 32u);
        queued -= take;
        bool ok = lane_id() < take;
        const uint32_t y = ok ? K.queue[queued + lane_id()] : 0u, x = y & kNbrMask;
        if (Q.wmask) ok = ok && wmask_ok(Q, w, x);
        if (ok) {  // every need's load before its answer is used
          bool few = false;
#pragma unroll 2
          for (uint32_t i = Q.need_begin[w]; i < Q.need_begin[w + 1]; ++i)
            few |= ((__ldg(G.sig + (uint64_t)Q.need_plane[i] * G.sig_words + (x >> 3)) >> ((x & 7) * 4)) & 15u) < Q.need_cnt[i];
          ok = !few;
        }
        found |= __reduce_or_sync(kFull, ok ? 1u << (y >> kNbrBits) : 0u);
        if (child) {
          const uint32_t bit = 1u << (x & 31), old = ok ? atomicOr(&ws[x >> 5], bit) : bit;
          if (old == 0) raise(W, ws, x, had < kListCap);
          const uint32_t m = __ballot_sync(kFull, !(old & bit)), at = have + __popc(m & below_me());
          if (!(old & bit) && at < kListCap) list_of(W, w)[at] = x;
          have += __popc(m);
        }
        __syncwarp();
      }
      if (child && have != had) {
        if (lane_id() == 0) {
          K.lc[w] = have;
          atomicAdd(&W.d.setcnt[Q.qv_base + w], have - had);
        }
        __syncwarp();
      }
      live = live && ((found >> lane_id()) & 1u);
    }
    if (step == 0) {
      const uint32_t stay = __ballot_sync(kFull, live);
      if (live) {
        if (atomicOr(&us[v >> 5], 1u << (v & 31)) == 0) raise(W, us, v, n <= kListCap);
        const uint32_t at = K.lc[u] + __popc(stay & below_me());
        if (at < kListCap) list_of(W, u)[at] = v;
      }
      __syncwarp();
      if (lane_id() == 0 && stay) {
        K.lc[u] += __popc(stay);
        atomicAdd(&W.d.setcnt[Q.qv_base + u], __popc(stay));
      }
      __syncwarp();
      continue;
    }
    const uint32_t dead = __ballot_sync(kFull, mine && !live);
    if (mine && !live) bit_clear(us, v);
    if (lane_id() == 0 && dead) atomicSub(&W.d.setcnt[Q.qv_base + u], __popc(dead));
  }
  __syncwarp();
}

// ------------------------------------------------------------ filter
// Positions of the first visited vertex's filter: one for a bound vertex, the
// vertices of its type, or groups of 1,024 vertices.
__device__ __forceinline__ uint32_t filter_size(const DevGraph &G, const DQuery &Q) {
  const uint32_t u = Q.visit[0];
  if (Q.vbind[u] != kUnbound) return 1;
  return Q.vtype[u] != kAny ? G.toff[Q.vtype[u] + 1] - G.toff[Q.vtype[u]] : G.W1;
}

// Which of a word's eight 4-bit counts are at least c: even and odd nibbles
// compared as bytes, then interleaved back into order.
__device__ __forceinline__ uint32_t nibbles_ge(uint32_t w, uint32_t c) {
  const uint32_t cc = c * 0x01010101u;
  const uint32_t z = __vsetgeu4(w & 0x0F0F0F0Fu, cc) | (__vsetgeu4((w >> 4) & 0x0F0F0F0Fu, cc) << 1);
  return (z & 3u) | ((z >> 6) & 0xCu) | ((z >> 12) & 0x30u) | ((z >> 18) & 0xC0u);
}

// Candidates of the first visited vertex among positions [cur, end): the same
// tests as k_filter's.  As many as fit the list; moves `cur`.
__device__ __forceinline__ uint32_t filter_some(const Wave &W, Worker &K, uint32_t &cur, uint32_t end, uint32_t *list,
                                                uint32_t cap, uint64_t &acc) {
  const DQuery &Q = K.Q;
  const DevGraph &G = W.G;
  const uint32_t u = Q.visit[0], t = Q.vtype[u], n0 = Q.need_begin[u], n1 = Q.need_begin[u + 1];
  uint32_t have = 0;
  if (Q.vbind[u] != kUnbound) {
    const bool ok = cand_ok(G, Q, u, Q.vbind[u]);
    if (ok && lane_id() == 0) list[0] = Q.vbind[u];
    cur = end;
    have = ok;
    if (lane_id() == 0) acc += 4 + (n1 - n0);
  } else if (t != kAny) {
    // Signature counts of eight list entries per word and lane: most entries
    // fail here.  The others queue up for the neighbour-type masks.
    const uint32_t b0 = G.toff[t] + cur, e0 = G.toff[t] + end, e8 = (e0 + 7) / 8;
    uint32_t w8 = b0 / 8, queued = 0;
    for (;;) {
      if (queued < 32 && w8 < e8 && have + 32 + queued + 256 <= cap) {
        const uint32_t wd = w8 + lane_id();
        uint32_t ok = wd < e8 ? 0xFFu : 0u, total;
        if (wd * 8 < b0) ok &= 0xFFu << (b0 - wd * 8);
        if (ok && wd * 8 + 8 > e0) ok &= 0xFFu >> (wd * 8 + 8 - e0);
        for (uint32_t i = n0; i < n1; ++i)
          if (ok) ok &= nibbles_ge(__ldg(G.sig_t + (uint64_t)Q.need_plane[i] * G.sig_words + wd), Q.need_cnt[i]);
        uint32_t p = queued + warp_excl(__popc(ok), total);
        for (; ok; ok &= ok - 1) K.queue[p++] = wd * 8 + __ffs(ok) - 1;
        queued += total;
        w8 += 32;
        __syncwarp();
        continue;
      }
      if (queued == 0) break;
      const uint32_t take = min(queued, 32u);
      queued -= take;
      bool ok = lane_id() < take;
      const uint32_t x = ok ? K.queue[queued + lane_id()] : 0u;
      for (uint32_t i = Q.inc_begin[u]; i < Q.inc_begin[u + 1]; ++i) {
        const uint32_t xi = Q.xinc[i], tw = Q.vtype[xinc_w(xi)];
        if (ok && tw != kAny)
          ok = (__ldg(G.tmask_t + (uint64_t)sig_plane(xinc_dir(xi), xinc_rel(xi), G.R) * G.V + x) >> (tw & 31u)) & 1u;
      }
      const uint32_t v = ok ? __ldg(G.tvid + x) : 0u;
      ok = ok && wmask_ok(Q, u, v);
      const uint32_t m = __ballot_sync(kFull, ok);
      if (ok) list[have + __popc(m & below_me())] = v;
      have += __popc(m);
      __syncwarp();
    }
    const uint32_t to = min(w8 * 8, e0);
    if (lane_id() == 0) acc += (uint64_t)(to - b0) * (4 + (n1 - n0));
    cur = to - G.toff[t];
  } else {
    for (; cur < end && have + 1024 <= cap; ++cur) {  // a group: lane l's vertices are 32 l, 32 l + 1, ...
      const uint32_t w0 = cur * 32 + lane_id(), v0 = w0 * 32;
      uint32_t ok = 0, total;
      if (w0 < G.W0) {
        ok = kFull;
        for (uint32_t i = n0; i < n1 && ok; ++i) {
          const uint4 g = __ldg(reinterpret_cast<const uint4 *>(G.sig + (uint64_t)Q.need_plane[i] * G.sig_words + (uint64_t)w0 * 4));
          const uint32_t c = Q.need_cnt[i];
          const uint32_t m = nibbles_ge(g.x, c) | nibbles_ge(g.y, c) << 8 | nibbles_ge(g.z, c) << 16 | nibbles_ge(g.w, c) << 24;
          ok &= m;
        }
        if (v0 + 32 > G.V) ok &= (1u << (G.V - v0)) - 1;
        for (uint32_t m = Q.wmask ? ok : 0u; m; m &= m - 1)
          if (!wmask_ok(Q, u, v0 + __ffs(m) - 1)) ok &= ~(1u << (__ffs(m) - 1));
      }
      uint32_t p = have + warp_excl(__popc(ok), total);
      for (; ok; ok &= ok - 1) list[p++] = v0 + __ffs(ok) - 1;
      have += total;
      if (lane_id() == 0) acc += 32ull * 16 * (n1 - n0);
    }
  }
  __syncwarp();
  return have;
}

// ------------------------------------------------------------ the join
// Order and edges per level, as the staged join plans them: begin with the
// vertex of fewest candidates, then the vertex with most edges into the
// joined part (ties: fewer candidates, then lower index).  Lane u for vertex u.
__device__ __forceinline__ void plan_join(const Wave &W, Worker &K) {
  const DQuery &Q = K.Q;
  const uint32_t u = lane_id();
  const uint32_t size = u < Q.k ? __ldcg(&W.d.setcnt[Q.qv_base + u]) : 0;
  uint32_t joined = 0, ne = 0;
  for (uint32_t s = 0; s < Q.k; ++s) {
    uint32_t links = 0;
    if (u < Q.k && !((joined >> u) & 1u))
      for (uint32_t i = Q.inc_begin[u]; i < Q.inc_begin[u + 1]; ++i) links += (joined >> xinc_w(Q.xinc[i])) & 1u;
    const bool able = u < Q.k && !((joined >> u) & 1u) && (s == 0 || links);
    // most links first (at most 240), then fewest candidates, then lowest index
    const uint32_t most = __reduce_max_sync(kFull, able ? links + 1 : 0u);
    const uint32_t least = __reduce_min_sync(kFull, able && links + 1 == most ? size : 0xFFFFFFFFu);
    const uint32_t best = __ffs(__ballot_sync(kFull, able && links + 1 == most && size == least)) - 1;
    // joined vertices that `best` could coincide with: of its type, or where
    // one of the two is not held to a type
    const uint32_t tb = Q.vtype[best];
    const uint32_t alike = __ballot_sync(kFull, u < Q.k && ((joined >> u) & 1u) && (Q.vtype[u] == tb || Q.vtype[u] == kAny || tb == kAny));
    if (u == 0) {
      uint32_t cols = 0;
      for (uint32_t m = alike; m; m &= m - 1) cols |= 1u << K.pos[__ffs(m) - 1];
      K.cmp[s] = (uint16_t)cols;
      K.order[s] = (uint8_t)best;
      K.pos[best] = (uint8_t)s;
      K.ebeg[s] = (uint8_t)ne;
      for (uint32_t i = Q.inc_begin[best]; i < Q.inc_begin[best + 1]; ++i) {
        const uint32_t xi = Q.xinc[i], x = xinc_w(xi);
        if (!((joined >> x) & 1u)) continue;
        // the edge seen from the joined endpoint: the other direction
        K.ecol[ne] = K.pos[x];
        K.epl[ne] = (uint8_t)adj_plane(1 - xinc_dir(xi), xinc_rel(xi));
        K.erel[ne] = (uint8_t)adj_rel(xinc_rel(xi));
        ++ne;
      }
    }
    joined |= 1u << best;
  }
  if (u == 0) {
    K.ebeg[Q.k] = (uint8_t)ne;
    K.full = 0;
  }
  if (u < kMaxK) {
    K.ln[u] = K.lr[u] = K.hb[u] = K.lt[u] = K.lo[u] = K.lg[u] = 0;
    K.lv[u] = 0;
  }
  __syncwarp();
}

// Level d of the worker's scratch: d + 1 columns of stride_of(d) ids.
__device__ __forceinline__ uint32_t stride_of(uint32_t d) { return d ? kLvlCap : kRootCap; }
__device__ __forceinline__ uint32_t *level_of(const Wave &W, uint32_t d) {
  return scratch_of(W) + (d ? kRootCap + (d * (d + 1) / 2 - 1) * kLvlCap : 0u);
}
__device__ __forceinline__ uint32_t *vlist_of(const Wave &W, uint32_t d) {
  return scratch_of(W) + kRootCap + kLvlWords + d * kVCap;
}
// The final rows collected so far go to the output pool, in query-vertex
// column order, as one segment of the query's rows.
__device__ __noinline__ void flush_rows(const Wave &W, Worker &K, uint32_t q) {
  const DQuery &Q = K.Q;
  const uint32_t k = Q.k, n = K.ln[k - 1];
  if (n == 0) return;
  unsigned long long at = ~0ull;
  if (lane_id() == 0) {
    DState &D = W.d.ds[q];
    // past the rows a query may hold on the device its rows are dropped, and
    // from then on the task only counts: the chunked path finds the smallest
    // cap of them.  Where the pool is full a second pass over the query
    // follows, with room for its count of rows.
    const unsigned long long had = atomicAdd(&D.emit, (unsigned long long)n);
    if (had + n <= over_cap_rows(Q.cap)) {
      at = atomicAdd((unsigned long long *)&W.ctrl->out_top, (unsigned long long)n * k);
      const uint32_t sg = atomicAdd(&W.d.ctl->segs, 1u);
      if (at + (uint64_t)n * k > W.out_words || sg >= W.d.seg_cap) {
        D.over = 1;
        at = ~0ull;
      } else {
        W.d.seg[sg] = DSeg{at, q, n};
        if (atomicAdd(&D.nseg, 1u) == 0) D.word = at;
      }
    }
    if (at == ~0ull) K.full = 1;
  }
  at = __shfl_sync(kFull, at, 0);
  if (at != ~0ull) {
    uint32_t *dst = W.out + at;
    const uint32_t *src = level_of(W, k - 1);
    const uint32_t st = stride_of(k - 1);
    for (uint32_t t = lane_id(); t < n * k; t += 32) dst[t] = src[(uint32_t)K.pos[t % k] * st + t / k];
  }
  __syncwarp();
  if (lane_id() == 0) K.ln[k - 1] = 0;
  __syncwarp();
}

// The next candidates of a batch of up to 32 rows of level d: every row's
// shortest relation run over the edges between the next vertex and the joined
// part drives it, and of the run's entries the live candidates stay.  Rows
// next to each other mostly share the vertex the run hangs on (they come from
// one row above), so a run is read and tested once for all of them.  A batch
// ends where its runs pass kVCap entries; one longer run is taken in parts,
// by the same rows until its end.
__device__ __forceinline__ void take_rows(const Wave &W, Worker &K, uint32_t d, uint64_t &acc) {
  const DQuery &Q = K.Q;
  const DevGraph &G = W.G;
  const uint32_t w = K.order[d + 1], e0 = K.ebeg[d + 1], e1 = K.ebeg[d + 2];
  const uint32_t *src = level_of(W, d), st = stride_of(d);
  const uint32_t *ws = slot_of(W, Q.qv_base + w);
  uint32_t *vl = vlist_of(W, d);
  const uint32_t r0 = K.lr[d], off = K.lo[d];
  uint32_t nb = off ? K.lg[d] : min(32u, K.ln[d] - r0);
  const bool mine = lane_id() < nb;
  uint32_t lo = 0, len = 0, x = 0xFFFFFFFFu, drv = e0, total;
  if (mine) {
    x = src[K.ecol[e0] * st + r0 + lane_id()];
    acc += 4ull * (d + 1) + 16ull * (e1 - e0);
  }
  if (e1 - e0 > 1 && mine) {
    len = 0xFFFFFFFFu;
    for (uint32_t e = e0; e < e1 && len; ++e) {
      uint32_t l, n;
      const uint32_t y = src[K.ecol[e] * st + r0 + lane_id()];
      run_of(G, K.epl[e], K.erel[e], y, l, n);
      if (n < len) { lo = l; len = n; drv = e; x = y; }
    }
  }
  const uint32_t px = __shfl_up_sync(kFull, x, 1), pd = __shfl_up_sync(kFull, drv, 1);
  const bool first = lane_id() == 0 || px != x || pd != drv;
  const uint32_t firsts = __ballot_sync(kFull, first);
  if (!first || !mine) len = 0;
  else if (e1 - e0 == 1) run_of(G, K.epl[e0], K.erel[e0], x, lo, len);
  uint32_t ex = warp_excl(min(len, kVCap + 1), total);  // min: 32 runs of millions still sum in 32 bits
  const uint32_t fit = __ballot_sync(kFull, ex + min(len, kVCap + 1) <= kVCap);
  bool more = false;
  if (!(fit & 1u)) {  // one run in parts, for the rows that share it
    nb = min(nb, firsts & ~1u ? (uint32_t)__ffs(firsts & ~1u) - 1 : 32u);
    if (lane_id() == 0) {
      more = len - off > kVCap;
      lo += off;
      len = min(len - off, kVCap);
    } else {
      len = 0;
    }
  } else if (fit != kFull) {
    nb = min(nb, (uint32_t)__ffs(~fit) - 1);
    if (lane_id() >= nb) len = 0;
  }
  more = __shfl_sync(kFull, more, 0);
  ex = warp_excl(len, total);
  K.vn[lane_id()] = 0;
  __syncwarp();
  uint32_t have = 0;
  for (uint32_t t0 = 0; t0 < total; t0 += 32 * kU) {
    uint32_t own[kU], c[kU];
    bool ok[kU];
#pragma unroll
    for (uint32_t j = 0; j < kU; ++j) {
      const uint32_t it = t0 + j * 32 + lane_id();
      own[j] = owner_of(ex, it);
      const uint32_t at = __shfl_sync(kFull, lo - ex, own[j]) + it, e = __shfl_sync(kFull, drv, own[j]);
      ok[j] = it < total;
      c[j] = ok[j] ? __ldg(G.adj[K.epl[e]] + at) & kNbrMask : 0;
    }
#pragma unroll
    for (uint32_t j = 0; j < kU; ++j) ok[j] = ok[j] && bit_final(ws, c[j]);
#pragma unroll
    for (uint32_t j = 0; j < kU; ++j) {
      const uint32_t m = __ballot_sync(kFull, ok[j]);
      if (ok[j]) {
        vl[have + __popc(m & below_me())] = c[j];
        atomicAdd(&K.vn[own[j]], 1u);
      }
      have += __popc(m);
    }
  }
  if (lane_id() == 0) acc += 8ull * total;
  __syncwarp();
  const uint32_t cnt = K.vn[lane_id()], vs = warp_excl(cnt, total);
  const uint32_t head = 31 - __clz(firsts & (below_me() | (1u << lane_id())));
  const uint32_t hs = __shfl_sync(kFull, vs, head), hc = __shfl_sync(kFull, cnt, head);
  K.vb[d][lane_id()] = (uint16_t)hs;
  K.vc[d][lane_id()] = (uint16_t)(lane_id() < nb ? hc : 0);
  __syncwarp();
  if (lane_id() == 0) {
    K.hb[d] = nb;
    K.lt[d] = 0;
    K.lo[d] = more ? off + kVCap : 0;
    K.lg[d] = more ? nb : 0;
  }
  __syncwarp();
}

// One step of an embedding's hash: vertex x at query vertex u.
__device__ __forceinline__ uint64_t fold(uint64_t h, uint32_t u, uint32_t x) {
  return mix64(h ^ ((uint64_t)x + (uint64_t)(u + 1) * 0x9E3779B97F4A7C15ull));
}

// Rows of level d in hand, each with its next candidates, to rows of level
// d + 1 (or, at the last level, to the query's totals and output): a
// candidate stays when it is not in the row and every other edge joins it.
// Stops where the next level is full; K.lt[d] holds where to go on.
__device__ __forceinline__ void expand(const Wave &W, Worker &K, uint32_t q, uint32_t d, unsigned long long &tot,
                                       unsigned long long &tfp, uint64_t &acc) {
  const DQuery &Q = K.Q;
  const DevGraph &G = W.G;
  const uint32_t k = Q.k, w = K.order[d + 1], e0 = K.ebeg[d + 1], e1 = K.ebeg[d + 2];
  const bool final = d + 2 == k, keep = !final || (rows_wanted(Q) && !K.full);
  const uint32_t *src = level_of(W, d), st = stride_of(d);
  uint32_t *dst = level_of(W, d + 1);
  const uint32_t *vl = vlist_of(W, d);
  const uint32_t r0 = K.lr[d], nb = K.hb[d];
  const uint32_t n = K.vc[d][lane_id()], vb = K.vb[d][lane_id()], cols = K.cmp[d + 1];
  uint32_t total;
  const uint32_t ex = warp_excl(n, total);
  // an embedding's hash folds its vertices in query order: the part before w
  // is the row's own
  uint64_t before = k;
  if (final && lane_id() < nb)
    for (uint32_t u = 0; u < w; ++u) before = fold(before, u, src[r0 + lane_id() + K.pos[u] * st]);
  uint32_t t0 = K.lt[d], fill = keep ? K.ln[d + 1] : 0, made = 0;
  __syncwarp();
  for (; t0 < total; t0 += 32) {
    if (keep && fill + 32 > kLvlCap) {
      if (!final) break;
      if (lane_id() == 0) K.ln[d + 1] = fill;
      __syncwarp();
      flush_rows(W, K, q);
      fill = 0;
    }
    const uint32_t it = t0 + lane_id(), own = owner_of(ex, it);
    const uint32_t at = __shfl_sync(kFull, vb - ex, own) + it;
    bool ok = it < total;
    uint32_t c = 0;
    const uint32_t *row = src + r0 + own;
    if (ok) {
      c = vl[at];
      for (uint32_t m = cols; m; m &= m - 1) ok = ok && row[(__ffs(m) - 1) * st] != c;
      if (e1 - e0 > 1) {  // (which edge drove the row does not matter: its entry is found again)
        for (uint32_t e = e0; e < e1 && ok; ++e) ok = has_nbr(G, K.epl[e], K.erel[e], row[K.ecol[e] * st], c);
      }
    }
    const uint32_t m = __ballot_sync(kFull, ok);
    made += __popc(m);
    const uint64_t head = final ? __shfl_sync(kFull, before, own) : 0;
    if (ok) {
      if (keep) {
        const uint32_t to = fill + __popc(m & below_me());
        for (uint32_t i = 0; i <= d; ++i) dst[i * kLvlCap + to] = row[i * st];
        dst[(d + 1) * kLvlCap + to] = c;
      }
      if (final) {
        uint64_t h = fold(head, w, c);
        for (uint32_t u = w + 1; u < k; ++u) h = fold(h, u, row[K.pos[u] * st]);
        tfp += h;  // per lane: summed when the task is done
      }
    }
    fill += __popc(m);
  }
  __syncwarp();
  if (lane_id() == 0) {
    if (keep) K.ln[d + 1] = fill;
    K.lv[d + 1] += made;
    if (t0 >= total) {
      K.lt[d] = 0;
      K.hb[d] = 0;
      if (K.lo[d] == 0) K.lr[d] = r0 + nb;  // else the rest of the long run comes next
    } else {
      K.lt[d] = t0;
    }
  }
  if (final) tot += made;
  if (lane_id() == 0) acc += 4ull * (d + 2) * made;
  __syncwarp();
}

// Rows of level e that stay with the worker: those done, those in hand, and
// between two parts of a long run (none is in hand then) those that share it.
__device__ __forceinline__ uint32_t busy_rows(const Worker &K, uint32_t e) { return K.lr[e] + max(K.hb[e], K.lg[e]); }

// Rows not yet taken go to the queue when workers are idle: from the
// shallowest level of [b, d] that has some to spare, whose rows stand for the
// most work.
__device__ __noinline__ void share_rows(const Wave &W, Worker &K, uint32_t q, uint32_t b, uint32_t d, uint32_t idle) {
  DCtl *c = W.d.ctl;
  uint32_t e = b, rows = 0, want = 0;
  if (lane_id() == 0) {
    for (; e <= d; ++e) {
      const uint32_t busy = busy_rows(K, e);
      if (K.ln[e] < busy + kShareMin) continue;
      const uint32_t spare = K.ln[e] - busy;
      rows = min(max((spare + idle) / (idle + 1), 16u), 64u);
      want = min((spare - rows) / rows, idle);
      break;
    }
  }
  want = __shfl_sync(kFull, want, 0);
  e = __shfl_sync(kFull, e, 0);
  rows = __shfl_sync(kFull, rows, 0);
  const uint32_t per = rows * (e + 1), st = stride_of(e);  // at most 64 x 15
  while (want) {  // up to 32 tasks at a time
    // a piece for each task's rows; where one is still in use they stay here
    const uint32_t t = min(want, 32u);
    uint32_t piece = 0;
    if (lane_id() == 0) piece = atomicAdd(&c->piece, t);
    piece = (__shfl_sync(kFull, piece, 0) + lane_id()) & (W.d.pieces - 1);
    bool got = false;
    if (lane_id() < t) {
      uint32_t *of = W.d.piece_of + piece;
      const uint32_t used = atomicCAS(of, 0u, c->turn);  // a run that ended badly may have left its turn there
      got = used == 0 || (used != c->turn && atomicCAS(of, used, c->turn) == used);
    }
    const uint32_t with = __ballot_sync(kFull, got), nt = __popc(with);
    unsigned long long slot = kNoSlot;
    if (lane_id() == 0 && nt) slot = reserve(W, nt);
    slot = __shfl_sync(kFull, slot, 0);
    if (slot == kNoSlot) {
      if (got) W.d.piece_of[piece] = 0;
      return;
    }
    __threadfence();
    const uint32_t first = K.ln[e] - nt * rows;
    const uint32_t *src = level_of(W, e) + first;
    // task t's piece, in lane t; a piece holds e + 1 columns of `rows` ids
    const bool all = with == (nt < 32 ? (1u << nt) - 1 : kFull);
    const uint32_t of = __shfl_sync(kFull, piece, all ? lane_id() : __fns(with, 0, lane_id() + 1) & 31u);
    for (uint32_t i0 = 0; i0 < nt * per; i0 += 128) {  // four loads in flight: they bound the copy
      uint32_t x[4], to[4];
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) {
        const uint32_t i = min(i0 + j * 32 + lane_id(), nt * per - 1), task = i / per, r = i % per;
        to[j] = __shfl_sync(kFull, of, task) * kPieceWords + r;
        x[j] = src[(r / rows) * st + task * rows + r % rows];
      }
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j)
        if (i0 + j * 32 + lane_id() < nt * per) W.d.share[to[j]] = x[j];
    }
    __threadfence();
    __syncwarp();
    if (got) push(W, TK_ROWS, q, e, piece, rows, slot + __popc(with & below_me()));
    if (lane_id() == 0) K.ln[e] = first;
    __syncwarp();
    want = nt == t ? want - t : 0;
  }
}

// Tasks that n items are cut into (one lane), at most `most`: small ones of
// `few` items while workers wait, else fewer and only where there are many,
// since the pieces only add up to the same work.  With no query left to start
// small ones already while fewer tasks wait than there are workers: just then
// nobody waits yet, and whether a step of 1,759 candidates ran on one warp for
// 0.9 ms was a matter of luck (eight draws of 1,000 queries on the 1M-vertex
// graph 1.09 to 1.71 ms a call, now 1.09 to 1.71 and 5 % less in the mean;
// 5,000 there counted 2.4 -> 2.0).  Small ones always cost 200 shape queries
// 8 %; this rule from the start of a batch costs 20,000 and 60,000 queries on
// the 1M-vertex graph 8 and 11 % (10,000 on the 4M-vertex graph gain 4).
__device__ __forceinline__ uint32_t task_count(const Wave &W, uint32_t n, uint32_t few, uint32_t most) {
  if (n <= 2 * few) return 1;
  const long long waiting = (long long)(ldv(&W.d.ctl->tail) - ldv(&W.d.ctl->head)), workers = gridDim.x * kWarps;
  const uint32_t per = waiting < (ldv(&W.d.ctl->next) >= W.nq ? workers : 0) ? few : 4 * few;
  if (n <= 2 * per) return 1;
  return min(min((n + per - 1) / per, most), 16384u);
}

// Items per task while few tasks wait.  Candidates: 16, since one of them
// can be a hub with a thousand neighbours (1,000 queries on the 1M-vertex
// graph 0.81 ms a batch, with 32 0.98, with 8 0.81 but larger batches 3 %
// slower).  Positions of the filter: 1,024, and 2,048 for types of over half
// a million vertices (200 shape queries on the 16M-vertex graph 7.3 -> 6.7;
// smaller types lose 5 to 10 % with 2,048).  Groups of 1,024 vertices: 4.
constexpr uint32_t kFewCands = 16, kFewGroups = 4;
__device__ __forceinline__ uint32_t few_positions(uint32_t n) { return n > (1u << 19) ? 2048u : 1024u; }

// Start of range i of n of `all` items.
__device__ __forceinline__ uint32_t range_at(uint32_t all, uint32_t i, uint32_t n) {
  return (uint32_t)((uint64_t)all * i / n);
}

__global__ void __launch_bounds__(32 * kWarps, kBlocksPerSm) k_direct(Wave W) {
  gdc_wait();
  extern __shared__ __align__(16) uint8_t smem[];
  Worker &K = reinterpret_cast<Worker *>(smem)[threadIdx.x >> 5];
  const DQuery &Q = K.Q;
  uint64_t acc = 0;
  uint32_t have_q = 0xFFFFFFFFu;
  if (lane_id() == 0) {
    K.ticket = kNoSlot;
    K.piece = kNoPiece;
  }
  const bool second = W.d.ctl->second;  // a second pass over the batch: some queries are left out
  const WaveDesc wave = W.waves[W.ctrl->wave];
  for (;;) {
    Task T{};
    if (lane_id() == 0) T = fetch(W, K);
    const uint32_t kind = __shfl_sync(kFull, T.kind, 0), q = __shfl_sync(kFull, T.q, 0);
    uint32_t step = __shfl_sync(kFull, T.step, 0), a = __shfl_sync(kFull, T.a, 0), b = __shfl_sync(kFull, T.b, 0);
    if (kind == TK_EXIT) break;
    const bool fresh_q = kind == TK_START;
    if (fresh_q || q != have_q) {
      const bool none = fresh_q && (q >= wave.nq || (second && W.d.skip[wave.q0 + q]));
      if (none) {  // padding, or left out of a second pass
        DQuery &D = W.dq[q];
        if (lane_id() == 0) {
          D.k = D.m = D.kp = D.nvisit = 0;
          D.status = K.Q.status = QS_INVALID;
        }
      } else {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(fresh_q ? W.all_dq + wave.q0 + q : W.dq + q);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&K.Q);
#pragma unroll 8
        for (uint32_t i = lane_id(); i < sizeof(DQuery) / 4; i += 32) dst[i] = __ldcg(src + i);
      }
      have_q = q;
      __syncwarp();
      if (fresh_q && !none) {
        if (lane_id() == 0) {
          K.Q.qv_base -= wave.qv0;
          K.Q.qe_base -= wave.qe0;
        }
        __syncwarp();
        if (Q.status != QS_INVALID) plan_query<false>(W.G, K.Q);
        // rows leave in query-vertex order: the sort reads column u at u
        if (lane_id() < K.Q.k) K.Q.pos[lane_id()] = (uint8_t)lane_id();
        if (lane_id() < K.Q.kp) K.Q.opos[lane_id()] = K.Q.pu[lane_id()];
        __syncwarp();
        uint32_t *to = reinterpret_cast<uint32_t *>(W.dq + q);
        const uint32_t *from = reinterpret_cast<const uint32_t *>(&K.Q);
#pragma unroll 8
        for (uint32_t i = lane_id(); i < sizeof(DQuery) / 4; i += 32) to[i] = from[i];
      }
    }
    bool join = kind == TK_ROOT || kind == TK_ROWS;
    if (kind == TK_START || kind == TK_EXPLORE) {
      // Exploration steps.  Children of steps this worker runs alone are
      // listed whole; a range of a step that several share lists only its own.
      bool own_range = kind == TK_EXPLORE, go = kind == TK_EXPLORE || (Q.status == QS_OK && Q.nvisit);
      if (lane_id() < kMaxK) K.lc[lane_id()] = 0;
      if (lane_id() == 0) K.listed = kind == TK_START ? 0xFFFFFFFFu : 0u;
      __syncwarp();
      while (go) {
        if (step >= Q.nvisit) {
          // a set left empty: no embedding
          const bool none = lane_id() < Q.k && __ldcg(&W.d.setcnt[Q.qv_base + lane_id()]) == 0;
          join = !__any_sync(kFull, none);
          if (!join && lane_id() == 0) mark(W.dq[q], QS_EMPTY);
          break;
        }
        const uint32_t u = Q.visit[step];
        uint32_t n = 0, nt = 0;
        unsigned long long slot = kNoSlot;
        if (lane_id() == 0) {
          n = step == 0 ? filter_size(W.G, Q) : listed(K, u) ? K.lc[u] : __ldcg(&W.d.setcnt[Q.qv_base + u]);
          if (!own_range && n) {
            nt = step ? task_count(W, n, kFewCands, W.G.W1)
                      : task_count(W, n, Q.vtype[u] != kAny ? few_positions(n) : kFewGroups, n);
            if (nt > 1) {
              W.d.pend[q] = nt;
              slot = reserve(W, nt);
            }
          }
        }
        n = __shfl_sync(kFull, n, 0);
        slot = __shfl_sync(kFull, slot, 0);
        if (n == 0 && !own_range) {  // (a filter of no positions has no candidate either)
          if (lane_id() == 0) mark(W.dq[q], QS_EMPTY);
          break;
        }
        if (slot != kNoSlot) {
          nt = __shfl_sync(kFull, nt, 0);
          __threadfence();  // `pend` and every lane's part of the planned query, before a task names it
          __syncwarp();
          for (uint32_t i = lane_id(); i < nt; i += 32)
            push(W, TK_EXPLORE, q, step, range_at(step ? W.G.W1 : n, i, nt), range_at(step ? W.G.W1 : n, i + 1, nt),
                 slot + i);
          break;
        }
        // the candidates: from the filter, as listed, or by and by from the
        // set's words
        const uint32_t *slot_u = slot_of(W, Q.qv_base + u);
        uint32_t *list = scratch_of(W) + kRootCap;
        uint32_t cur = own_range ? a : 0, end = own_range ? b : step ? W.G.W1 : n, m = 0;
        bool dense = n > W.G.W0 / 4;
        if (step) {
          cur *= 32;
          end = min(end * 32, W.G.W0);
          if (listed(K, u)) {
            list = list_of(W, u);
            m = K.lc[u];
            cur = end;
          }
        }
        for (;;) {
          if (cur < end)
            m = step ? refill(W, slot_u, cur, end, dense, list, kLvlWords) : filter_some(W, K, cur, end, list, kLvlWords, acc);
          if (m) explore_list(W, K, u, step, list, m, acc);
          if (cur >= end) break;
        }
        __threadfence();
        __syncwarp();
        if (own_range) {
          uint32_t left = 0;
          if (lane_id() == 0) left = atomicSub(&W.d.pend[q], 1u);
          if (__shfl_sync(kFull, left, 0) != 1) break;
          __threadfence();  // the step's last range: the query goes on here
          own_range = false;
          // sets of later steps' children are this worker's alone from here on
          if (lane_id() < Q.k) K.lc[lane_id()] = 0;
          const uint32_t later = __ballot_sync(kFull, lane_id() < Q.k && Q.init_step[lane_id()] > step + 1);
          if (lane_id() == 0) K.listed = later;
          __syncwarp();
        }
        ++step;
      }
      if (join) {
        plan_join(W, K);
        uint32_t nt = 1;
        unsigned long long slot = kNoSlot;
        if (lane_id() == 0) {
          nt = task_count(W, __ldcg(&W.d.setcnt[Q.qv_base + K.order[0]]), 2 * kFewCands, W.G.W1);
          if (nt > 1 || (K.ticket != kNoSlot && (int)ldv(&W.d.ctl->room) < 1 << (W.d.task_log - 1))) slot = reserve(W, nt);
        }
        slot = __shfl_sync(kFull, slot, 0);
        nt = __shfl_sync(kFull, nt, 0);
        a = 0;
        b = W.G.W1;
        if (slot != kNoSlot) {
          __threadfence();
          __syncwarp();
          for (uint32_t i = lane_id(); i < nt; i += 32)
            push(W, TK_ROOT, q, 0, range_at(W.G.W1, i, nt), range_at(W.G.W1, i + 1, nt), slot + i);
          join = false;
        }
      }
    } else if (join) {
      plan_join(W, K);
    }
    if (join) {
      // Everything below the rows of level b0, depth first with as many rows
      // of each level at a time as its buffer holds.
      const uint32_t last = Q.k - 1;  // rows of this level are final
      const uint32_t b0 = kind == TK_ROWS ? step : 0, u0 = K.order[0];
      const uint32_t *us = slot_of(W, Q.qv_base + u0);
      uint32_t cur = 0, end = 0, ids = 0;  // what is left of the first vertex's set
      bool dense = false, from_list = false;
      if (kind == TK_ROWS) {
        uint32_t *dst = level_of(W, b0), st = stride_of(b0);
        const uint32_t *src = W.d.share + (uint64_t)a * kPieceWords;
        for (uint32_t i = lane_id(); i < b * (b0 + 1); i += 32) dst[(i / b) * st + i % b] = __ldcg(src + i);
        if (lane_id() == 0) {
          K.ln[b0] = b;
          K.piece = a;  // free again when the task is done
        }
      } else if (kind != TK_ROOT && listed(K, u0)) {
        from_list = true;
        ids = K.lc[u0];
      } else {
        cur = a * 32;
        end = min(b * 32, W.G.W0);
        dense = __ldcg(&W.d.setcnt[Q.qv_base + u0]) > W.G.W0 / 4;
      }
      __syncwarp();
      uint32_t d = b0;
      unsigned long long tot = 0, tfp = 0;
      for (;;) {
        if (K.lr[d] >= K.ln[d]) {  // level d is used up
          __syncwarp();
          if (lane_id() == 0) K.ln[d] = K.lr[d] = 0;
          __syncwarp();
          if (d > b0) {
            --d;
            continue;
          }
          if (kind == TK_ROWS) break;
          uint32_t *l0 = level_of(W, 0), n = 0;
          if (from_list) {  // the listed ids that are still live
            const uint32_t *list = list_of(W, u0);
            for (uint32_t r = 0; r < ids; r += 32) {
              const uint32_t v = r + lane_id() < ids ? list[r + lane_id()] : 0;
              const bool live = r + lane_id() < ids && bit_live(us, v);
              const uint32_t m = __ballot_sync(kFull, live);
              if (live) l0[n + __popc(m & below_me())] = v;
              n += __popc(m);
            }
            ids = 0;
          } else {
            n = refill(W, us, cur, end, dense, l0, kRootCap);
          }
          if (n == 0) break;
          __syncwarp();
          if (lane_id() == 0) {
            K.ln[0] = n;
            K.lv[0] += n;
          }
          __syncwarp();
          if (last == 0) {  // one vertex: the candidates are the embeddings
            tot += n;
            for (uint32_t i = lane_id(); i < n; i += 32) tfp += mix64(1ull ^ ((uint64_t)l0[i] + 0x9E3779B97F4A7C15ull));
            if (rows_wanted(Q)) flush_rows(W, K, q);
            __syncwarp();
            if (lane_id() == 0) K.ln[0] = 0;
            __syncwarp();
          }
          continue;
        }
        if (K.hb[d] == 0) take_rows(W, K, d, acc);
        expand(W, K, q, d, tot, tfp, acc);
        uint32_t idle = 0;
        const uint32_t deep = d + 1 == last ? d : d + 1;
        const bool spare = lane_id() >= b0 && lane_id() <= deep && K.ln[lane_id()] >= busy_rows(K, lane_id()) + kShareMin;
        if (__any_sync(kFull, spare)) {
          if (lane_id() == 0) idle = idle_workers(W);
          idle = __shfl_sync(kFull, idle, 0);
          if (idle) share_rows(W, K, q, b0, deep, idle);
        }
        // down when the next level is full or this one is used up
        if (d + 1 < last && K.ln[d + 1] && (K.lr[d] >= K.ln[d] || K.ln[d + 1] + 32 > kLvlCap)) ++d;
      }
      // what the task found, to the query's totals
      if (rows_wanted(Q) && last) flush_rows(W, K, q);
#pragma unroll
      for (int o = 16; o; o >>= 1) tfp += __shfl_xor_sync(kFull, tfp, o);
      if (lane_id() == 0 && tot) {
        atomicAdd((unsigned long long *)&W.qs[q].count, tot);
        atomicAdd((unsigned long long *)&W.qs[q].fp, tfp);
      }
      if (lane_id() < last && K.lv[lane_id()]) atomicAdd(&W.d.ds[q].lv[lane_id()], K.lv[lane_id()]);
    }
    __syncwarp();
    task_done(W, K);
  }
  flush_bytes(W, KK_EXPLORE, acc);
}

// Counters of a run.
__global__ void k_direct_reset(Wave W) {
  gdc_wait();
  for (uint64_t i = gtid(); i < W.nqv; i += gthreads()) W.d.setcnt[i] = 0;
  for (uint64_t i = gtid(); i < W.nq; i += gthreads()) {
    W.d.ds[i] = DState{};
    W.qs[i] = QState{};
  }
  if (gtid() < kRingParts) W.d.ctl->taken[gtid()] = 0;
  if (gtid() == 0) {
    DCtl &c = *W.d.ctl;
    const unsigned long long last = c.head > c.tail ? c.head : c.tail;
    c.turn += 1 + (uint32_t)(last >> W.d.task_log);  // past every turn of the run before
    c.head = c.tail = 0;
    c.next = c.segs = 0;
    c.open = W.nq;
    c.room = 1u << W.d.task_log;
    c.part = 0;
    c.piece = 0;
    W.ctrl->out_top = 0;
    W.ctrl->out_rows_total = 0;
  }
}

// Segments of queries with several to the room k_final_bases made for them,
// one block per segment; and the bitmaps back to zero.
__global__ void __launch_bounds__(256) k_direct_finish(Wave W) {
  gdc_wait();
  __shared__ unsigned long long at;
  const uint32_t n = min(W.d.ctl->segs, W.d.seg_cap);
  for (uint32_t i = blockIdx.x; i < n; i += gridDim.x) {
    const DSeg g = W.d.seg[i];
    DState &D = W.d.ds[g.q];
    if (D.nseg < 2 || W.qs[g.q].out_rows == 0) continue;  // block-uniform
    if (threadIdx.x == 0) at = atomicAdd(&D.fill, (unsigned long long)g.rows);
    __syncthreads();
    const uint32_t k = W.dq[g.q].k;
    const uint32_t *src = W.out + g.word;
    uint32_t *dst = W.out + D.word + at * k;
    for (uint32_t j = threadIdx.x; j < g.rows * k; j += 256) dst[j] = src[j];
    __syncthreads();
  }
  clear_sets(W);
}

}  // namespace

int direct_blocks(int sms) {
  int n = 0;
  const size_t smem = kWarps * sizeof(Worker);
  cudaFuncSetAttribute(k_direct, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_direct, 32 * kWarps, smem) != cudaSuccess || n < 1) {
    cudaGetLastError();
    n = 1;
  }
  return sms * n;
}
uint32_t direct_workers() { return kWarps; }
uint64_t direct_scratch_words() { return (uint64_t)kWarps * kScratch; }

void launch_direct_reset(const Wave &W, cudaStream_t s, int sms) {
  const uint64_t n = std::max<uint64_t>(W.nqv, W.nq);
  pdl(k_direct_reset, (unsigned)std::min<uint64_t>((n + 255) / 256 + 1, (uint64_t)sms * 4), 256, 0, s, W);
}
void launch_direct(const Wave &W, cudaStream_t s) {
  pdl(k_direct, W.d.blocks, 32 * kWarps, kWarps * sizeof(Worker), s, W);
}
void launch_direct_finish(const Wave &W, cudaStream_t s, int sms) {
  pdl(k_direct_finish, (unsigned)sms * 8, 256, 0, s, W);
}

}  // namespace gs
