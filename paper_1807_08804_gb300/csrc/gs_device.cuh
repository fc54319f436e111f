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

// splitmix64 finaliser (Steele, Lea & Flood 2014); row hash for fingerprints.
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

}  // namespace

}  // namespace gs
