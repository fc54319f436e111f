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
__device__ __forceinline__ void direct_layout(const Wave &W, uint32_t qi) {
  DQuery &Q = W.dq[qi];
  QState &S = W.qs[qi];
  DState &D = W.d.ds[qi];
  S.inter_words = S.peak_words = 0;
  for (uint32_t l = 0; l + 1 < Q.k; ++l) {
    const uint64_t w = D.lv[l] * (l + 1);
    S.inter_words += w;
    S.peak_words = w > S.peak_words ? w : S.peak_words;
  }
  S.out_rows = 0;
  if (Q.status != QS_OK || !rows_wanted(Q)) return;
  if (S.count > over_cap_rows(Q.cap)) {
    Q.status = QS_TOPCAP;
    return;
  }
  const uint64_t n = D.emit;
  const uint64_t r = atomicAdd((unsigned long long *)&W.ctrl->out_rows_total, (unsigned long long)n);
  if (D.nseg > 1) D.word = atomicAdd((unsigned long long *)&W.ctrl->out_top, (unsigned long long)(n * Q.k));
  if (D.over || r + n > W.out_rows_cap || (n && D.word + n * Q.k > W.out_words)) {
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
