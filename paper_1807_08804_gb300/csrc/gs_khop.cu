// Domain-graph exploration (Ch. 5, "Domain-specific knowledge graph
// generation"): the concepts within a few hops of a set of seed concepts,
// found level by level the way the filtering phase explores (warps over the
// frontier vertices' coalesced adjacency rows).
//
// State: level[V] (uint8, 255 = not reached), a visited bitmap claimed with
// atomicOr, and two frontier lists.  A level step reads the frontier size
// from device memory, so the whole exploration runs without a host sync.
// The last level needs neither the bitmap nor a frontier.
#include <algorithm>
#include <cstring>
#include <mutex>
#include <vector>

#include "gs_internal.h"

namespace gs {

namespace {

constexpr int kKT = 256;  // threads per block
constexpr uint32_t kFullMask = 0xFFFFFFFFu;

struct KhopArgs {
  const uint64_t *off[2];
  const uint32_t *adj[2];
  uint32_t dirs;           // bit 0: follow edges forwards, bit 1: backwards
  uint32_t relmask[8];     // relations followed (bit r)
  uint32_t all_rels;       // every relation: skip the mask test
  uint32_t V;
  uint8_t *level;
  uint32_t *vis;           // visited bitmap [ceil(V/32)]
  uint32_t *front[2];      // frontier lists [V]
  unsigned long long *cnt; // vertices per level [levels + 2]
  unsigned long long *grab;  // per level: frontier entries handed out to warps so far
  unsigned long long *edges;  // adjacency entries scanned
  uint32_t *err;           // bit 0: a seed out of range
};

__device__ __forceinline__ bool claim(const KhopArgs &A, uint32_t v) {
  const uint32_t bit = 1u << (v & 31);
  if (A.vis[v >> 5] & bit) return false;
  return !(atomicOr(&A.vis[v >> 5], bit) & bit);
}

// Seeds: level 0, frontier 0 (repeated seeds claimed once).
__global__ void k_khop_seeds(KhopArgs A, const uint32_t *seeds, uint32_t n) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const uint32_t s = seeds[i];
    if (s >= A.V) {
      atomicOr(A.err, 1u);
      continue;
    }
    if (claim(A, s)) {
      A.level[s] = 0;
      A.front[0][atomicAdd(&A.cnt[0], 1ull)] = s;
    }
  }
}

__device__ __forceinline__ bool follow(const KhopArgs &A, uint32_t x) {
  const uint32_t r = x >> kNbrBits;
  return A.all_rels || ((A.relmask[r >> 5] >> (r & 31)) & 1u);
}

// One level: the frontier vertices of level l (front[l & 1], cnt[l] of
// them) scan their rows in the followed directions; each neighbour over a
// followed relation that is not yet visited gets level l + 1.  Load
// balanced: a warp takes up to 32 frontier vertices at a time from a shared
// counter (fewer when the frontier is small, and when it is smaller than the
// grid several warps share one vertex's rows) and walks their concatenated
// rows kKU windows of 32 entries at a time, one entry per lane and window.
// The rows that are not empty sit side by side in shared memory, so the row
// of an entry is a count of row starts: those before the window, and a
// population count over the window's starts (a search by shuffles took five
// times the instructions).  4 hops from 16 seeds of a 16M-vertex / 200M-edge
// graph, 84 million entries: 1.21 -> 1.00 ms a call (0.91 ms on the device,
// second-level cache flushed); the last level is
// now bound by its random one-byte accesses, which keep the second-level
// cache 63 % and the first-level 67 % busy.
// Below the last level a neighbour is claimed in the visited bitmap and
// appended to the next frontier (one atomic per warp and pass).  The last
// level builds no frontier: an unreached neighbour's level is written
// without atomics (every writer writes the same value) and counted after.
constexpr uint32_t kKU = 4;

template <bool LAST>
__global__ void __launch_bounds__(kKT, 6) k_khop_level(KhopArgs A, uint32_t l) {
  __shared__ uint32_t s_start[kKT / 32][32], s_delta[kKT / 32][32];
  const uint32_t lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const uint32_t below = (1u << lane) - 1, upto = below | (1u << lane);
  const uint64_t nfront = A.cnt[l];
  const uint32_t *front = A.front[l & 1];
  uint32_t *next = A.front[(l + 1) & 1];
  const uint64_t nwarps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
  // work units: vpw frontier vertices per warp when the frontier is large;
  // when it is smaller than the grid, wpv warps share each vertex's rows
  const uint64_t per_warp = (nfront + nwarps - 1) / nwarps;
  const uint32_t vpw = per_warp >= 32 ? 32u : (per_warp ? (uint32_t)per_warp : 1u);
  const uint32_t wpv = nfront && nfront < nwarps ? (uint32_t)min((uint64_t)32, nwarps / nfront) : 1u;
  uint64_t scanned = 0;
  for (;;) {
    // the next unit, taken from a shared counter so that warps that drew
    // short rows take more
    unsigned long long g = 0;
    if (lane == 0) g = atomicAdd(&A.grab[l], (unsigned long long)(wpv > 1 ? 1u : vpw));
    g = __shfl_sync(kFullMask, g, 0);
    const uint64_t i0 = wpv > 1 ? g / wpv : g;
    const uint32_t sub = wpv > 1 ? (uint32_t)(g % wpv) : 0u;
    if (i0 >= nfront) break;
    // this lane's frontier vertex: its row ranges (fewer than 2^32 entries)
    uint32_t rb[2] = {0, 0}, rn[2] = {0, 0};
    if (lane < vpw && i0 + lane < nfront) {
      const uint32_t u = front[i0 + lane];
#pragma unroll
      for (int d = 0; d < 2; ++d)
        if ((A.dirs >> d) & 1u) {
          rb[d] = (uint32_t)A.off[d][u];
          rn[d] = (uint32_t)A.off[d][u + 1] - rb[d];
        }
    }
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      const uint32_t n = rn[d], some = __ballot_sync(kFullMask, n > 0);
      if (!some) continue;  // warp-uniform
      uint32_t incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kFullMask, incl, o);
        if (lane >= o) incl += y;
      }
      const uint32_t total = __shfl_sync(kFullMask, incl, 31);
      __syncwarp();
      if (n) {
        const uint32_t r = __popc(some & below);
        s_start[wib][r] = incl - n;
        s_delta[wib][r] = rb[d] - (incl - n);
      }
      __syncwarp();
      const uint32_t start = lane < (uint32_t)__popc(some) ? s_start[wib][lane] : 0xFFFFFFFFu;
      if (sub == 0) scanned += total;
      const uint32_t *adj = A.adj[d];
      for (uint32_t t0 = 32 * kKU * sub; t0 < total; t0 += 32 * kKU * wpv) {
        uint32_t x[kKU];
        bool ok[kKU];
#pragma unroll
        for (uint32_t j = 0; j < kKU; ++j) {
          const uint32_t tb = t0 + 32 * j, in = start - tb, t = tb + lane;
          const uint32_t m = __reduce_or_sync(kFullMask, in < 32 ? 1u << in : 0u);
          const uint32_t own = __popc(__ballot_sync(kFullMask, start < tb)) + __popc(m & upto) - 1;
          ok[j] = t < total;
          const uint32_t at = s_delta[wib][own] + t;  // modulo 2^32: a row can start before its place in the window
          x[j] = ok[j] ? __ldg(adj + at) : 0;
          ok[j] = ok[j] && follow(A, x[j]);
          x[j] &= kNbrMask;
        }
        if (LAST) {
          uint8_t v[kKU];
#pragma unroll
          for (uint32_t j = 0; j < kKU; ++j) v[j] = ok[j] ? A.level[x[j]] : 0;
#pragma unroll
          for (uint32_t j = 0; j < kKU; ++j)
            if (v[j] == 255) A.level[x[j]] = (uint8_t)(l + 1);
          continue;
        }
        uint32_t seen[kKU], made = 0;
#pragma unroll
        for (uint32_t j = 0; j < kKU; ++j) seen[j] = ok[j] ? A.vis[x[j] >> 5] : 0;
#pragma unroll
        for (uint32_t j = 0; j < kKU; ++j) {
          const uint32_t bit = 1u << (x[j] & 31);
          ok[j] = ok[j] && !(seen[j] & bit) && !(atomicOr(&A.vis[x[j] >> 5], bit) & bit);
        }
#pragma unroll
        for (uint32_t j = 0; j < kKU; ++j) {
          seen[j] = __ballot_sync(kFullMask, ok[j]);
          made += __popc(seen[j]);
        }
        if (made) {
          unsigned long long base = 0;
          if (lane == 0) base = atomicAdd(&A.cnt[l + 1], (unsigned long long)made);
          base = __shfl_sync(kFullMask, base, 0);
#pragma unroll
          for (uint32_t j = 0; j < kKU; ++j) {
            if (ok[j]) {
              A.level[x[j]] = (uint8_t)(l + 1);
              next[base + __popc(seen[j] & below)] = x[j];
            }
            base += __popc(seen[j]);
          }
        }
      }
    }
  }
  if (lane == 0 && scanned) atomicAdd(A.edges, (unsigned long long)scanned);
}

// Vertices whose level is l (the last level's count): sixteen level bytes per
// load where the array is aligned, single bytes before and after.
__global__ void k_count_level(KhopArgs A, uint32_t l) {
  const uint64_t tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, nt = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t head = min((uint64_t)A.V, (16 - (uint64_t)(uintptr_t)A.level % 16) % 16), q = (A.V - head) / 16;
  const uint4 *p = reinterpret_cast<const uint4 *>(A.level + head);
  const uint32_t want = l * 0x01010101u;
  uint32_t c = 0;
  for (uint64_t i = tid; i < q; i += nt) {
    const uint4 x = p[i];
    c += (__popc(__vcmpeq4(x.x, want)) + __popc(__vcmpeq4(x.y, want)) + __popc(__vcmpeq4(x.z, want)) +
          __popc(__vcmpeq4(x.w, want))) / 8;
  }
  if (tid < head) c += A.level[tid] == l;
  for (uint64_t i = head + 16 * q + tid; i < A.V; i += nt) c += A.level[i] == l;
  for (int o = 16; o; o >>= 1) c += __shfl_xor_sync(kFullMask, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(&A.cnt[l], (unsigned long long)c);
}

// The state of a new exploration: no vertex reached (level bytes 255, sixteen
// per store where aligned), nothing visited, counters zero.
__global__ void k_khop_reset(KhopArgs A, uint32_t levels) {
  const uint64_t tid = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x, nt = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t head = min((uint64_t)A.V, (16 - (uint64_t)(uintptr_t)A.level % 16) % 16), q = (A.V - head) / 16;
  uint4 *p = reinterpret_cast<uint4 *>(A.level + head);
  for (uint64_t i = tid; i < q; i += nt) p[i] = make_uint4(~0u, ~0u, ~0u, ~0u);
  if (tid < head) A.level[tid] = 255;
  for (uint64_t i = head + 16 * q + tid; i < A.V; i += nt) A.level[i] = 255;
  for (uint64_t i = tid; i < (A.V + 31) / 32; i += nt) A.vis[i] = 0;
  if (tid < levels + 2) A.cnt[tid] = 0;
  if (tid < levels + 1) A.grab[tid] = 0;
  if (tid == 0) A.cnt[256] = A.cnt[257] = 0;  // entries scanned, error word
}

}  // namespace

// Per-graph buffers of the exploration, made on first use.
struct Khop {
  uint8_t *level = nullptr;
  uint32_t *vis = nullptr, *front[2] = {}, *seeds = nullptr;
  unsigned long long *cnt = nullptr;
  uint32_t seeds_cap = 0;
  cudaStream_t stream = nullptr;
  std::mutex mu;
  ~Khop() {
    for (void *p : {(void *)level, (void *)vis, (void *)front[0], (void *)front[1], (void *)seeds, (void *)cnt})
      if (p) cudaFree(p);
    if (stream) cudaStreamDestroy(stream);
  }
};

void release_khop(gs_graph *g) {
  delete static_cast<Khop *>(g->khop);
  g->khop = nullptr;
}

static std::mutex g_khop_ctx_mu;  // first use on a graph from several threads

static gs_status khop_ctx(gs_graph *g, Khop **out) {
  std::lock_guard<std::mutex> lk(g_khop_ctx_mu);
  if (g->khop) {
    *out = static_cast<Khop *>(g->khop);
    return GS_OK;
  }
  Khop *k = new Khop();
  const uint64_t V = g->d.V, words = (V + 31) / 32;
  cudaError_t e = gs::dev_malloc(&k->level, V);
  if (e == cudaSuccess) e = gs::dev_malloc(&k->vis, 4 * words);
  if (e == cudaSuccess) e = gs::dev_malloc(&k->front[0], 4 * V);
  if (e == cudaSuccess) e = gs::dev_malloc(&k->front[1], 4 * V);
  // counts [0, 256), entries scanned, error word, hand-out counters [258, 514)
  if (e == cudaSuccess) e = gs::dev_malloc(&k->cnt, 8 * 514);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&k->stream, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    delete k;
    return cuda_fail(e, "gs_khop buffers");
  }
  g->khop = k;
  *out = k;
  return GS_OK;
}

}  // namespace gs

using namespace gs;

extern "C" gs_status gs_khop(gs_graph *g, const uint32_t *seeds, uint32_t nseeds, const gs_khop_opts *opts,
                             uint8_t *level_out, uint64_t *counts, uint64_t *edges_scanned) {
  if (!g || !opts || !level_out || !counts || (nseeds && !seeds)) return fail(GS_ERR_INVALID, "gs_khop: null argument");
  if (opts->levels > 254) return fail(GS_ERR_INVALID, "gs_khop: levels must be at most 254");
  if (opts->directions == 0 || opts->directions > (GS_KHOP_OUT | GS_KHOP_IN))
    return fail(GS_ERR_INVALID, "gs_khop: directions must be GS_KHOP_OUT, GS_KHOP_IN or both");
  if (opts->nrels && !opts->rels) return fail(GS_ERR_INVALID, "gs_khop: null relation list");
  KhopArgs A;
  memset(&A, 0, sizeof(A));
  A.all_rels = opts->rels ? 0u : 1u;
  for (uint32_t i = 0; opts->rels && i < opts->nrels; ++i) {
    const uint32_t r = opts->rels[i];
    if (r >= g->d.R) return fail(GS_ERR_INVALID, "gs_khop: relation out of range");
    A.relmask[r >> 5] |= 1u << (r & 31);
  }
  const bool on_dev = (opts->flags & GS_DEVICE_PTRS) != 0;
  if (!on_dev)
    for (uint32_t i = 0; i < nseeds; ++i)
      if (seeds[i] >= g->d.V) return fail(GS_ERR_INVALID, "gs_khop: seed out of range");
  GS_CUDA(cudaSetDevice(g->device));
  Khop *k = nullptr;
  gs_status st = khop_ctx(g, &k);
  if (st != GS_OK) return st;
  std::lock_guard<std::mutex> lk(k->mu);
  const cudaStream_t s = opts->cuda_stream ? static_cast<cudaStream_t>(opts->cuda_stream) : k->stream;
  const uint32_t V = g->d.V, L = opts->levels;
  const uint32_t *dseeds = seeds;
  if (!on_dev && nseeds) {
    if (nseeds > k->seeds_cap) {
      if (k->seeds) cudaFree(k->seeds);
      k->seeds = nullptr;
      k->seeds_cap = 0;
      GS_CUDA(gs::dev_malloc(&k->seeds, 4ull * nseeds));
      k->seeds_cap = nseeds;
    }
    GS_CUDA(cudaMemcpyAsync(k->seeds, seeds, 4ull * nseeds, cudaMemcpyHostToDevice, s));
    dseeds = k->seeds;
  }
  A.off[0] = g->d.off[0]; A.off[1] = g->d.off[1];
  A.adj[0] = g->d.adj[0]; A.adj[1] = g->d.adj[1];
  A.dirs = opts->directions;
  A.V = V;
  A.level = on_dev ? level_out : k->level;
  A.vis = k->vis;
  A.front[0] = k->front[0]; A.front[1] = k->front[1];
  A.cnt = k->cnt;
  A.edges = k->cnt + 256;
  A.err = reinterpret_cast<uint32_t *>(k->cnt + 257);
  A.grab = k->cnt + 258;
  const unsigned fill_grid = (unsigned)std::min<uint64_t>((V + kKT - 1) / kKT, (uint64_t)g->num_sms * 8);  // >= 1 block of 256
  k_khop_reset<<<fill_grid, kKT, 0, s>>>(A, L);
  if (nseeds) {
    const unsigned sg = (unsigned)std::min<uint64_t>((nseeds + kKT - 1) / kKT, (uint64_t)g->num_sms * 4);
    k_khop_seeds<<<sg, kKT, 0, s>>>(A, dseeds, nseeds);
  }
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_khop_level<false>, kKT, 0) != cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  const unsigned grid = (unsigned)(g->num_sms * std::min(per_sm, 8));
  for (uint32_t l = 0; l + 1 < L; ++l) k_khop_level<false><<<grid, kKT, 0, s>>>(A, l);
  if (L > 0) {
    k_khop_level<true><<<grid, kKT, 0, s>>>(A, L - 1);
    k_count_level<<<fill_grid, kKT, 0, s>>>(A, L);
  }
  GS_CUDA(cudaGetLastError());
  std::vector<unsigned long long> c(258);  // one copy: counts, entries scanned, error word
  GS_CUDA(cudaMemcpyAsync(c.data(), A.cnt, 8ull * 258, cudaMemcpyDeviceToHost, s));
  if (!on_dev) GS_CUDA(cudaMemcpyAsync(level_out, A.level, V, cudaMemcpyDeviceToHost, s));
  GS_CUDA(cudaStreamSynchronize(s));
  if (c[257] & 1u) return fail(GS_ERR_INVALID, "gs_khop: seed out of range");
  for (uint32_t l = 0; l <= L; ++l) counts[l] = c[l];
  if (edges_scanned) *edges_scanned = c[256];
  return GS_OK;
}
