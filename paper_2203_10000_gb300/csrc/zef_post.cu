// zef_post.cu -- post-processing of the labeled mesh (Sec. 2.2): Taubin
// smoothing (Sec. 2.2.1) and inflation towards a compartment surface
// (Sec. 2.2.2).
//
// Smoothing works on the mesh's unique edges, gathered once per call into rows of
// neighbours per node: blocks take runs of tets, find the unique edges of
// their run in shared memory and leave each node's neighbours in the run as a
// piece linked to the node; a node's row is its pieces merged, ascending and
// without repeats, so that every sum over a node's neighbours runs in
// ascending neighbour order (deterministic results).
//
// Smoothing: one iteration is the forward step x' = x + lambda L(x) with a
// fixed-order reduction of ||x' - x||^2, the backward step x'' = x' - mu L(x'),
// and a one-block kernel that decides whether to continue, with
// L(x)_i = sum_j (x_j - x_i) / (deg_i + 1) over the edge neighbours j of i
// (node i itself belongs to its neighbourhood and adds nothing to the sum).
//
// Smoothing of the tissue boundaries (surface variant of Sec. 2.2.1): the
// faces whose three nodes each touch more than one element label go into an
// open-addressing table keyed by their sorted node triple (128-bit
// compare-and-swap) with the smallest and largest element label of the tets
// that share them; a face whose two labels differ is a
// boundary face, and its three edges build the adjacency of the same
// iteration, so that only the boundary nodes move.
//
// Inflation: the nodes are labeled (inside bits of every compartment); the
// edges from a node inside compartment c to a node outside are gathered from
// the tets through a table of that size and listed by node, eight lanes per edge find its intersection with c's triangles nearest to the
// inside node, and the node moves by zeta t (x_j - x_i) averaged over its
// crossing edges, t the edge parameter of that intersection.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "zef_internal.h"

#define CK(call, what)                                      \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) return cuda_fail(ctx, e_, what); \
  } while (0)

namespace zef {

namespace {

constexpr unsigned long long kNoKey = ~0ull;
__constant__ int kEdgeLocal[6][2] = {{0, 1}, {0, 2}, {0, 3}, {1, 2}, {1, 3}, {2, 3}};
// words of the post-processing statistics (device)
enum PpWord { PP_CAND = 0, PP_BAD, PP_ITER, PP_STOP, PP_FACES, PP_FULL, PP_POOL, PP_ROWS, PP_WORDS };

__device__ __forceinline__ unsigned long long pp_mix(unsigned long long x) {
  x ^= x >> 33;
  x *= 0xff51afd7ed558ccdull;
  x ^= x >> 33;
  x *= 0xc4ceb9fe1a85ec53ull;
  x ^= x >> 33;
  return x;
}

struct Adj {
  unsigned long long *keys;  // open-addressing table of edge keys (lo << 32 | hi)
  unsigned long long mask;   // table size - 1
  int shift;                 // log2 of the slots per node (table size >= n << shift)
  uint32_t *deg;             // [n + 1] row starts (the table's: degrees, scanned)
  uint32_t *fill;            // [n] neighbours per row (the table's: scatter cursors before)
  int32_t *nbr;              // row i: nbr[deg[i]], fill[i] neighbours, ascending
  int64_t n;
  int64_t *words;            // PpWord
};

// First probe of edge (lo, hi), lo < hi: a slot of lo's run of 2^shift slots,
// picked by a hash of hi (linear probing from there may leave the run).
__device__ __forceinline__ unsigned long long edge_slot(const Adj &g, uint32_t lo, uint32_t hi) {
  return (((unsigned long long)lo << g.shift) | (pp_mix(hi) & ((1ull << g.shift) - 1ull))) & g.mask;
}

// every tet's six edges into the table; the first insertion counts the edge
// in both end nodes' degrees (the edge count is half the degree sum)
__global__ void __launch_bounds__(256) k_pp_edges(Adj g, const int32_t *tets, int64_t m, uint32_t *status) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x) {
    int32_t v[4];
    bool bad = false;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = tets[4 * t + k];
      bad |= v[k] < 0 || v[k] >= g.n;
    }
    if (bad) {
      atomicOr(status, ST_INVALID);
      atomicExch((unsigned long long *)(g.words + PP_BAD), 1ull);
      continue;
    }
#pragma unroll
    for (int e = 0; e < 6; ++e) {
      const uint32_t a = (uint32_t)v[kEdgeLocal[e][0]], b = (uint32_t)v[kEdgeLocal[e][1]];
      if (a == b) continue;
      const unsigned long long key = ((unsigned long long)min(a, b) << 32) | max(a, b);
      unsigned long long h = edge_slot(g, min(a, b), max(a, b));
      for (unsigned long long it = 0; it <= g.mask; ++it) {
        const unsigned long long prev = atomicCAS(g.keys + h, kNoKey, key);
        if (prev == kNoKey) {
          atomicAdd(g.deg + min(a, b), 1u);
          atomicAdd(g.deg + max(a, b), 1u);
          break;
        }
        if (prev == key) break;
        h = (h + 1) & g.mask;
      }
    }
  }
}

// ---- edges of runs of tets, each edge once per run
// A block takes kRunTets consecutive tets.  Their nodes go into a table in
// shared memory, their edges (pairs of node slots) into another, so that an
// edge shared inside the run -- most are: refinement appends the children of
// neighbouring tets together -- is kept once.  The run's neighbours, ordered by
// node, go to the pool as one contiguous write of pieces (next piece of the
// node, count, neighbours), each linked into its node's list.
// 14.7 M tets of a refined head: 71 M neighbours in 11.3 M pieces, for 44 M
// neighbours without repeats and 59 M tet corners.
// 512 tets would leave 68 M in 10.4 M, but fill the shared memory with half as
// many warps: volume smoothing 5.16 ms, with 256 tets 4.40, with two lanes per
// tet 4.20 (128 and 64 tets: 4.28, 4.29).
constexpr int kRunTets = 256;
constexpr int kRunThreads = 2 * kRunTets;
constexpr int kRunBits = 11;
constexpr int kRunNodes = 1 << kRunBits;  // node slots: at most 1024 nodes
constexpr int kRunEdges = 1 << kRunBits;  // edge slots: at most 1536 edges
constexpr int kRunPool = 2 * 6 * kRunTets + 2 * 4 * kRunTets;  // words of a run's pieces: 20 a tet
constexpr uint32_t kNoSlot = 0xffffffffu;
constexpr uint32_t kNoPiece = 0xffffffffu;
constexpr size_t kRunShared = (size_t)(2 * kRunNodes + kRunEdges + kRunPool) * sizeof(uint32_t);

__global__ void __launch_bounds__(kRunThreads) k_pp_runs(int64_t n, const int32_t *tets, int64_t m, uint32_t *pool,
                                                uint32_t *head, int64_t *words, uint32_t *status) {
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ uint32_t s_scan[kRunThreads / 32];
  __shared__ uint32_t s_base;
  uint32_t *nkey = sm, *ncnt = sm + kRunNodes, *ekey = ncnt + kRunNodes, *out = ekey + kRunEdges;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t t0 = (int64_t)blockIdx.x * kRunTets; t0 < m; t0 += (int64_t)gridDim.x * kRunTets) {
    for (int j = threadIdx.x; j < kRunNodes / 4; j += kRunThreads) {
      reinterpret_cast<uint4 *>(nkey)[j] = make_uint4(kNoSlot, kNoSlot, kNoSlot, kNoSlot);
      reinterpret_cast<uint4 *>(ncnt)[j] = make_uint4(0u, 0u, 0u, 0u);
    }
    for (int j = threadIdx.x; j < kRunEdges / 4; j += kRunThreads)
      reinterpret_cast<uint4 *>(ekey)[j] = make_uint4(kNoSlot, kNoSlot, kNoSlot, kNoSlot);
    __syncthreads();
    // two neighbouring lanes per tet, two nodes and three edges each
    const int64_t t = t0 + threadIdx.x / 2;
    const int h = threadIdx.x & 1;
    bool ok = t < m;
    int32_t v[4] = {0, 0, 0, 0};
    if (ok) {
      bool bad = false;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[k] = tets[4 * t + k];
        bad |= v[k] < 0 || v[k] >= n;
      }
      if (bad) {
        ok = false;
        atomicOr(status, ST_INVALID);
        atomicExch((unsigned long long *)(words + PP_BAD), 1ull);
      }
    }
    uint32_t own[2] = {0u, 0u};
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (!ok) continue;
      const uint32_t key = (uint32_t)(h ? v[2 * k + 1] : v[2 * k]);
      uint32_t s = (key * 2654435761u) >> (32 - kRunBits);
      for (;;) {  // ends: at most half of the slots are taken
        const uint32_t prev = atomicCAS(nkey + s, kNoSlot, key);
        if (prev == kNoSlot || prev == key) break;
        s = (s + 1) & (kRunNodes - 1);
      }
      own[k] = s;
    }
    const uint32_t o0 = __shfl_xor_sync(0xffffffffu, own[0], 1), o1 = __shfl_xor_sync(0xffffffffu, own[1], 1);
    const uint32_t s0 = h ? o0 : own[0], s1 = h ? own[0] : o0, s2 = h ? o1 : own[1], s3 = h ? own[1] : o1;
    __syncthreads();
#pragma unroll
    for (int e = 0; e < 3; ++e) {
      // edges 01, 02, 03 and 12, 13, 23
      const uint32_t x = h ? (e < 2 ? s1 : s2) : s0, y = h ? (e == 0 ? s2 : s3) : (e == 0 ? s1 : e == 1 ? s2 : s3);
      if (!ok || x == y) continue;  // a repeated node
      const uint32_t key = (min(x, y) << kRunBits) | max(x, y);
      uint32_t s = (key * 2654435761u) >> (32 - kRunBits);
      for (;;) {  // ends: at most three quarters of the slots are taken
        const uint32_t prev = atomicCAS(ekey + s, kNoSlot, key);
        if (prev == kNoSlot) {
          atomicAdd(ncnt + x, 1u);
          atomicAdd(ncnt + y, 1u);
          break;
        }
        if (prev == key) break;
        s = (s + 1) & (kRunEdges - 1);
      }
    }
    __syncthreads();
    // piece offsets inside the run: scan of the slots' piece sizes
    constexpr int kPer = kRunNodes / kRunThreads;
    const int j0 = threadIdx.x * kPer;
    uint32_t mine = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      const uint32_t c = ncnt[j0 + k];
      mine += c ? c + 2u : 0u;
    }
    uint32_t incl = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) s_scan[wid] = incl;
    __syncthreads();
    uint32_t at = incl - mine, total = 0;
#pragma unroll
    for (int w = 0; w < kRunThreads / 32; ++w) {
      at += w < wid ? s_scan[w] : 0u;
      total += s_scan[w];
    }
    if (threadIdx.x == 0) s_base = (uint32_t)atomicAdd((unsigned long long *)(words + PP_POOL), (unsigned long long)total);
    __syncthreads();
    const uint32_t base = s_base;
#pragma unroll 4
    for (int k = 0; k < kPer; ++k) {
      const uint32_t c = ncnt[j0 + k];
      if (!c) continue;
      out[at] = atomicExch(head + nkey[j0 + k], base + at);
      out[at + 1] = c;
      ncnt[j0 + k] = at + 2;  // the write position of the slot's neighbours
      at += c + 2u;
    }
    __syncthreads();
    for (int j = threadIdx.x; j < kRunEdges; j += kRunThreads) {
      const uint32_t key = ekey[j];
      if (key == kNoSlot) continue;
      const uint32_t x = key >> kRunBits, y = key & (kRunNodes - 1);
      out[atomicAdd(ncnt + x, 1u)] = nkey[y];
      out[atomicAdd(ncnt + y, 1u)] = nkey[x];
    }
    __syncthreads();
    for (uint32_t j = threadIdx.x; j < total; j += kRunThreads) pool[base + j] = out[j];
    __syncthreads();
  }
}
static_assert(kRunNodes >= 8 * kRunTets && kRunEdges * 3 >= 24 * kRunTets, "the tables never fill up");

// one undirected edge into the table (first insertion counts it at both ends)
__device__ __forceinline__ void insert_edge(const Adj &g, uint32_t a, uint32_t b) {
  if (a == b) return;
  const unsigned long long key = ((unsigned long long)min(a, b) << 32) | max(a, b);
  unsigned long long h = edge_slot(g, min(a, b), max(a, b));
  for (unsigned long long it = 0; it <= g.mask; ++it) {
    const unsigned long long prev = atomicCAS(g.keys + h, kNoKey, key);
    if (prev == kNoKey) {
      atomicAdd(g.deg + min(a, b), 1u);
      atomicAdd(g.deg + max(a, b), 1u);
      return;
    }
    if (prev == key) return;
    h = (h + 1) & g.mask;
  }
  atomicExch((unsigned long long *)(g.words + PP_FULL), 1ull);  // cannot happen at load <= 1/2
}

// First of cnt places from the cursor for every thread of a 256-thread block
// (all threads call): one addition per block.  (One per warp costs 0.8 ns
// each, all of them on one word: 0.37 ms for 0.46 M warps.)
__device__ __forceinline__ unsigned long long block_places(uint32_t cnt, int64_t *cursor) {
  __shared__ uint32_t s_warp[8];
  __shared__ unsigned long long s_base;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  uint32_t before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    before += w < wid ? s_warp[w] : 0u;
    total += s_warp[w];
  }
  if (threadIdx.x == 0 && total) s_base = atomicAdd((unsigned long long *)cursor, (unsigned long long)total);
  __syncthreads();
  const unsigned long long base = s_base;
  __syncthreads();  // before the next call's writes
  return base + before + (incl - cnt);
}

// ---- tissue-boundary faces
struct FaceTab {
  unsigned long long *keys;  // [2 * (mask + 1)]: (a | b << 32, c) of the sorted triple, all ones when empty
  int32_t *lo, *hi;          // smallest / largest element label of the tets sharing the face
  unsigned long long mask;
};

// 128-bit compare-and-swap (sm_90 and later): returns the previous value
__device__ __forceinline__ void cas128(unsigned long long *p, unsigned long long clo, unsigned long long chi,
                                       unsigned long long vlo, unsigned long long vhi, unsigned long long &olo,
                                       unsigned long long &ohi) {
  asm volatile(
      "{\n\t.reg .b128 d, c, v;\n\tmov.b128 c, {%2, %3};\n\tmov.b128 v, {%4, %5};\n\t"
      "atom.global.cas.b128 d, [%6], c, v;\n\tmov.b128 {%0, %1}, d;\n\t}"
      : "=l"(olo), "=l"(ohi)
      : "l"(clo), "l"(chi), "l"(vlo), "l"(vhi), "l"(p)
      : "memory");
}

__global__ void __launch_bounds__(256) k_sf_clear(FaceTab f) {
  for (unsigned long long s = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; s <= f.mask;
       s += (unsigned long long)gridDim.x * blockDim.x) {
    f.keys[2 * s] = kNoKey;
    f.keys[2 * s + 1] = kNoKey;
    f.lo[s] = INT32_MAX;
    f.hi[s] = INT32_MIN;
  }
}

// ---- which faces can lie on a boundary
// A face between two labels has three nodes that both labels touch, so only
// the faces of such (mixed) nodes go into the table.  Pass 1 leaves some tet's
// label at every node (whichever store comes last), pass 2 marks the nodes
// where a tet's label differs from it: exactly the nodes of more than one
// label.  Pass 3 counts the faces with three marked nodes, for the table's
// size.
__device__ __forceinline__ bool load_tet(const int32_t *tets, int64_t t, int64_t n, int32_t (&v)[4]) {
  bool ok = true;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[k] = tets[4 * t + k];
    ok &= v[k] >= 0 && v[k] < n;
  }
  return ok;
}

__global__ void __launch_bounds__(256) k_sf_first(const int32_t *tets, const int32_t *labels, int64_t m, int64_t n,
                                                 int32_t *first, int64_t *words, uint32_t *status) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x) {
    int32_t v[4];
    if (!load_tet(tets, t, n, v)) {
      atomicOr(status, ST_INVALID);
      atomicExch((unsigned long long *)(words + PP_BAD), 1ull);
      continue;
    }
    const int32_t lab = labels[t];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(first + v[k]), "r"(lab) : "memory");
  }
}

__global__ void __launch_bounds__(256) k_sf_mixed(const int32_t *tets, const int32_t *labels, int64_t m, int64_t n,
                                                 const int32_t *first, uint8_t *mixed) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x) {
    int32_t v[4];
    if (!load_tet(tets, t, n, v)) continue;
    const int32_t lab = labels[t];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (first[v[k]] != lab) mixed[v[k]] = 1;
  }
}

// bits of the tet's mixed nodes
__device__ __forceinline__ uint32_t mixed_bits(const uint8_t *mixed, const int32_t (&v)[4]) {
  uint32_t b = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) b |= mixed[v[k]] ? 1u << k : 0u;
  return b;
}

__global__ void __launch_bounds__(256) k_sf_count(const int32_t *tets, int64_t m, int64_t n, const uint8_t *mixed,
                                                 int64_t *words) {
  uint32_t c = 0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x) {
    int32_t v[4];
    if (!load_tet(tets, t, n, v)) continue;
    const int k = __popc(mixed_bits(mixed, v));
    c += k == 4 ? 4u : k == 3 ? 1u : 0u;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd((unsigned long long *)(words + PP_CAND), (unsigned long long)c);
}

// A face of three mixed nodes: sorted node triple and its tet's element label.
struct __align__(16) FaceItem {
  uint32_t a, b, c;
  int32_t label;
};

// the faces of mixed nodes into a list
__global__ void __launch_bounds__(256) k_sf_list(const int32_t *tets, const int32_t *labels, int64_t m, int64_t n,
                                                const uint8_t *mixed, FaceItem *items, int64_t *words) {
  for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x; t0 < m; t0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = t0 + threadIdx.x;
    int32_t v[4] = {0, 0, 0, 0};
    uint32_t mb = 0;
    if (t < m && load_tet(tets, t, n, v)) mb = mixed_bits(mixed, v);
    const uint32_t cnt = __popc(mb) == 4 ? 4u : __popc(mb) == 3 ? 1u : 0u;
    unsigned long long at = block_places(cnt, words + PP_POOL);
    if (!cnt) continue;
    const int32_t lab = labels[t];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      // face q leaves out vertex 3 - q
      if ((mb | 1u << (3 - q)) != 0xfu) continue;
      const uint32_t a = (uint32_t)v[q == 3 ? 1 : 0], b = (uint32_t)v[q >= 2 ? 2 : 1], c = (uint32_t)v[q >= 1 ? 3 : 2];
      FaceItem f;
      f.a = min(a, min(b, c));
      f.c = max(a, max(b, c));
      f.b = a ^ b ^ c ^ f.a ^ f.c;
      f.label = lab;
      items[at++] = f;
    }
  }
}

// the listed faces into the table, one thread each
__global__ void __launch_bounds__(256) k_sf_faces(FaceTab f, const FaceItem *items, int64_t *words) {
  const int64_t len = words[PP_POOL];
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < len; k += (int64_t)gridDim.x * blockDim.x) {
    const FaceItem it = items[k];
    const unsigned long long klo = (unsigned long long)it.a | ((unsigned long long)it.b << 32), khi = it.c;
    unsigned long long h = pp_mix(klo ^ pp_mix(khi)) & f.mask;
    bool placed = false;
    for (unsigned long long p = 0; p <= f.mask; ++p) {
      unsigned long long olo, ohi;
      cas128(f.keys + 2 * h, kNoKey, kNoKey, klo, khi, olo, ohi);
      if ((olo == kNoKey && ohi == kNoKey) || (olo == klo && ohi == khi)) {
        atomicMin(f.lo + h, it.label);
        atomicMax(f.hi + h, it.label);
        placed = true;
        break;
      }
      h = (h + 1) & f.mask;
    }
    if (!placed) atomicExch((unsigned long long *)(words + PP_FULL), 1ull);
  }
}

// the boundary faces (two tets, different labels) into a list
__global__ void __launch_bounds__(256) k_sf_boundary(FaceTab f, uint4 *faces, int64_t *words) {
  for (unsigned long long s0 = blockIdx.x * (unsigned long long)blockDim.x; s0 <= f.mask;
       s0 += (unsigned long long)gridDim.x * blockDim.x) {  // the table's size is a multiple of 256
    const unsigned long long s = s0 + threadIdx.x;
    const ulonglong2 k = reinterpret_cast<const ulonglong2 *>(f.keys)[s];
    const bool is = k.x != kNoKey && f.lo[s] != f.hi[s];
    const unsigned long long at = block_places(is ? 1u : 0u, words + PP_FACES);
    if (is) faces[at] = make_uint4((uint32_t)k.x, (uint32_t)(k.x >> 32), (uint32_t)k.y, 0u);
  }
}

// their edges into the edge table, one thread per edge
__global__ void __launch_bounds__(256) k_sf_edges(const uint4 *faces, Adj g) {
  const int64_t len = 3 * g.words[PP_FACES];
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < len; k += (int64_t)gridDim.x * blockDim.x) {
    const uint4 f = faces[k / 3];
    const int e = (int)(k % 3);
    insert_edge(g, e == 2 ? f.y : f.x, e == 0 ? f.y : f.z);
  }
}

__global__ void __launch_bounds__(256) k_pp_scatter(Adj g) {
  if (g.words[PP_BAD]) return;
  for (unsigned long long s = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; s <= g.mask;
       s += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned long long key = g.keys[s];
    if (key == kNoKey) continue;
    const uint32_t a = (uint32_t)(key >> 32), b = (uint32_t)(key & 0xffffffffu);
    g.nbr[g.deg[a] + atomicAdd(g.fill + a, 1u)] = (int32_t)b;
    g.nbr[g.deg[b] + atomicAdd(g.fill + b, 1u)] = (int32_t)a;
  }
}

// Every row ascending and without repeats; fill[i] becomes its length.  A warp
// takes 32 consecutive rows, which lie together in memory: they are staged in
// shared memory (coalesced), one thread per row inserts its entries into the
// row's sorted, repeat-free prefix there, and the rows go back.  Rows longer
// than kRowThread, and the rows of a warp that do not fit the stage, are
// sorted one after the other by the whole warp (places by counting; rows of
// more than kRowStage / 2 entries by merging).
constexpr int kRowThread = 48;
constexpr int kRowStage = 1536;         // entries per warp
constexpr int32_t kRepeat = INT32_MAX;  // above every node index (below 2^31 - 1)

// Batcher's bitonic merge sort (Knuth 3, 5.3.4) of any length by one warp: every exchange puts
// the smaller value first, so entries beyond the end (the largest there could
// be) stay where they are.  One step exchanges i with its mirror image in its
// run of k entries (flip), or with i + k / 2.
__device__ __forceinline__ void bitonic_step(int32_t *a, int cnt, int k, bool flip, int lane) {
  const int half = k / 2, pairs = (cnt + k - 1) / k * half;
  for (int p = lane; p < pairs; p += 32) {
    const int i = p / half * k + p % half, j = flip ? i + k - 1 - 2 * (p % half) : i + half;
    if (j >= cnt) continue;
    const int32_t x = a[i], y = a[j];
    if (x > y) {
      a[i] = y;
      a[j] = x;
    }
  }
  __syncwarp();
}

// A row too long for the stage (a node joined to hundreds of others, with the
// repeats of all pieces): steps inside runs of kRowRun entries in shared
// memory, the others where the row is, then the repeats are squeezed out.
// Its cost grows as n log^2 n: with one lane inserting, a node of 1,024
// neighbours in 5,120 tets in random order took 1.26 s, now 1.5 ms.
constexpr int kRowRun = 1024;
static_assert(kRowRun <= kRowStage, "a run fits the stage");

__device__ __noinline__ int sort_row_long(int32_t *r, int cnt, int32_t *buf, int lane) {
  for (int k = 2; k / 2 < cnt || k <= kRowRun; k *= 2) {
    if (k > kRowRun) {
      bitonic_step(r, cnt, k, true, lane);
      for (int h = k / 2; h > kRowRun; h /= 2) bitonic_step(r, cnt, h, false, lane);
    }
    if (k < kRowRun) continue;  // the first runs are sorted whole at k = kRowRun
    for (int b = 0; b < cnt; b += kRowRun) {
      const int len = min(kRowRun, cnt - b);
      for (int j = lane; j < len; j += 32) buf[j] = r[b + j];
      __syncwarp();
      if (k == kRowRun)
        for (int q = 2; q <= kRowRun; q *= 2) {
          bitonic_step(buf, len, q, true, lane);
          for (int h = q / 2; h >= 2; h /= 2) bitonic_step(buf, len, h, false, lane);
        }
      else
        for (int h = kRowRun; h >= 2; h /= 2) bitonic_step(buf, len, h, false, lane);
      for (int j = lane; j < len; j += 32) r[b + j] = buf[j];
      __syncwarp();
    }
  }
  int out = 0;
  int32_t before = kRepeat;  // the last value of the 32 before: no node has this index
  for (int b = 0; b < cnt; b += 32) {
    const int32_t v = b + lane < cnt ? r[b + lane] : kRepeat;
    int32_t prev = __shfl_up_sync(0xffffffffu, v, 1);
    if (lane == 0) prev = before;
    before = __shfl_sync(0xffffffffu, v, 31);
    const bool keep = v != kRepeat && v != prev;
    const uint32_t m = __ballot_sync(0xffffffffu, keep);
    if (keep) r[out + __popc(m & ((1u << lane) - 1u))] = v;  // at or before what has been read
    out += __popc(m);
    __syncwarp();
  }
  return out;
}

__device__ int sort_row_warp(int32_t *r, int cnt, int32_t *buf, int lane) {
  if (cnt > kRowStage / 2) return sort_row_long(r, cnt, buf, lane);
  int32_t *u = buf + kRowStage / 2;
  for (int j = lane; j < cnt; j += 32) buf[j] = r[j];
  __syncwarp();
  int out = 0;
  for (int j = lane; j < cnt; j += 32) {
    const int32_t v = buf[j];
    bool rep = false;
    for (int q = 0; q < j; ++q) rep |= buf[q] == v;
    u[j] = rep ? kRepeat : v;
    out += rep ? 0 : 1;
  }
  __syncwarp();
  for (int j = lane; j < cnt; j += 32) {
    const int32_t v = u[j];
    if (v == kRepeat) continue;
    int place = 0;
    for (int q = 0; q < cnt; ++q) place += u[q] < v ? 1 : 0;
    r[place] = v;
  }
  __syncwarp();
  return (int)__reduce_add_sync(0xffffffffu, (uint32_t)out);
}

__global__ void __launch_bounds__(256) k_pp_sort_rows(Adj g) {
  extern __shared__ int32_t s_rows[];
  if (g.words[PP_BAD]) return;
  const int lane = threadIdx.x & 31;
  int32_t *buf = s_rows + (threadIdx.x >> 5) * kRowStage;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); i0 < g.n; i0 += step) {
    const int64_t i = i0 + lane;
    const uint32_t b0 = g.deg[i0], e0 = g.deg[min(i0 + 32, g.n)];
    const uint32_t b = i < g.n ? g.deg[i] : e0, e = i < g.n ? g.deg[i + 1] : e0;
    const int cnt = (int)(e - b), total = (int)(e0 - b0);
    const bool staged = e0 - b0 <= (uint32_t)kRowStage;
    const bool mine = staged && cnt <= kRowThread;
    if (staged) {
      for (int j = lane; j < total; j += 32) buf[j] = g.nbr[b0 + j];
      __syncwarp();
      if (mine) {
        int32_t *a = buf + (b - b0);
        int out = 0;
        for (int k = 0; k < cnt; ++k) {
          const int32_t v = a[k];
          int j = out - 1;
          while (j >= 0 && a[j] > v) --j;
          if (j >= 0 && a[j] == v) continue;
          for (int q = out; q > j + 1; --q) a[q] = a[q - 1];
          a[j + 1] = v;
          ++out;
        }
        if (i < g.n) g.fill[i] = (uint32_t)out;
      }
      __syncwarp();
      for (int j = lane; j < total; j += 32) g.nbr[b0 + j] = buf[j];
      __syncwarp();
    }
    uint32_t rest = __ballot_sync(0xffffffffu, !mine && i < g.n);
    while (rest) {
      const int src = __ffs(rest) - 1;
      rest &= rest - 1;
      const uint32_t rb = __shfl_sync(0xffffffffu, b, src);
      const int out = sort_row_warp(g.nbr + rb, __shfl_sync(0xffffffffu, cnt, src), buf, lane);
      if (lane == src) g.fill[i] = (uint32_t)out;
    }
  }
}

// Batcher's odd-even merge sort of N values in registers (Knuth, The Art of
// Computer Programming 3, 5.3.4): N = 64 in 543 exchanges of two instructions,
// the same for every lane.
template <int N, int P, int K>
__device__ __forceinline__ void merge_net(int32_t (&v)[N]) {
#pragma unroll
  for (int x = 0; x + K < N; ++x) {
    constexpr int j0 = K % P;
    if (x >= j0 && (x - j0) % (2 * K) < K && x / (2 * P) == (x + K) / (2 * P)) {
      const int32_t a = min(v[x], v[x + K]), b = max(v[x], v[x + K]);
      v[x] = a;
      v[x + K] = b;
    }
  }
  if constexpr (K > 1) merge_net<N, P, K / 2>(v);
  else if constexpr (2 * P < N) merge_net<N, 2 * P, 2 * P>(v);
}

// Sorts the column of cnt <= N entries (stride 32) and writes it back without
// repeats; returns what is left.
template <int N>
__device__ __forceinline__ int sort_column(int32_t *col, int cnt) {
  int32_t v[N];
#pragma unroll
  for (int k = 0; k < N; ++k) v[k] = k < cnt ? col[32 * k] : kRepeat;
  merge_net<N, 1, 1>(v);
  int out = 0;
#pragma unroll
  for (int k = 0; k < N; ++k)
    if (v[k] != kRepeat && (k == 0 || v[k] != v[k - 1])) col[32 * out++] = v[k];
  return out;
}

// The nodes' rows from their pieces, ascending and without repeats.  A warp
// takes 32 nodes, one per thread: the pieces go into the thread's column in
// shared memory (entry k of all lanes side by side: no bank conflicts), are
// sorted by a network in registers -- an insertion sort in shared memory took
// three times as long, its steps being dependent and the longest row of the
// 32 setting the pace -- and the rows go out at a place taken from the row
// cursor.  Nodes of more than kColumn entries are gathered and sorted one
// after the other by the whole warp in their place in the rows array (room
// for the repeats stays unused).
constexpr int kColumn = 64;

__global__ void __launch_bounds__(256) k_pp_merge(Adj g, const uint32_t *pool, const uint32_t *head) {
  extern __shared__ int32_t s_rows[];
  if (g.words[PP_BAD]) return;
  const int lane = threadIdx.x & 31;
  int32_t *buf = s_rows + (threadIdx.x >> 5) * (kColumn * 32);
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); i0 < g.n; i0 += step) {
    const int64_t i = i0 + lane;
    const uint32_t first = i < g.n ? head[i] : kNoPiece;
    int cnt = 0;
    for (uint32_t p = first; p != kNoPiece;) {
      const uint32_t next = pool[p];
      const int c = (int)pool[p + 1];
      if (cnt + c <= kColumn)
#pragma unroll 4
        for (int k = 0; k < c; ++k) buf[32 * (cnt + k) + lane] = (int32_t)pool[p + 2 + k];
      cnt += c;
      p = next;
    }
    const bool mine = cnt <= kColumn;
    const int longest = (int)__reduce_max_sync(0xffffffffu, (uint32_t)(mine ? cnt : 0));
    int out = 0;
    if (longest <= 32) out = sort_column<32>(buf + lane, mine ? cnt : 0);
    else out = sort_column<64>(buf + lane, mine ? cnt : 0);
    // places of the rows: the warp's from the cursor, one after the other
    const int room = mine ? out : cnt;
    int at = room;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += t;
    }
    unsigned long long base = 0;
    if (lane == 31 && at) base = atomicAdd((unsigned long long *)(g.words + PP_ROWS), (unsigned long long)at);
    base = __shfl_sync(0xffffffffu, base, 31);
    const uint32_t row = (uint32_t)base + (uint32_t)(at - room);
    if (mine)
      for (int k = 0; k < out; ++k) g.nbr[row + k] = buf[32 * k + lane];
    if (i < g.n) {
      g.deg[i] = row;
      if (mine) g.fill[i] = (uint32_t)out;
    }
    uint32_t rest = __ballot_sync(0xffffffffu, !mine);
    while (rest) {
      const int src = __ffs(rest) - 1;
      rest &= rest - 1;
      const uint32_t r0 = __shfl_sync(0xffffffffu, row, src);
      uint32_t p = __shfl_sync(0xffffffffu, first, src), w = r0;
      while (p != kNoPiece) {
        const uint32_t next = pool[p], c = pool[p + 1];
        for (uint32_t k = lane; k < c; k += 32) g.nbr[w + k] = (int32_t)pool[p + 2 + k];
        w += c;
        p = next;
      }
      __syncwarp();
      const int len = sort_row_warp(g.nbr + r0, (int)(w - r0), buf, lane);
      if (lane == src) g.fill[i] = (uint32_t)len;
    }
    __syncwarp();
  }
}
static_assert(kColumn * 32 >= kRowStage, "sort_row_warp's stage");

// rows sorted (one launch)
zef_status sort_rows(zef_ctx *ctx, const Adj &g) {
  constexpr size_t smem = (size_t)8 * kRowStage * sizeof(int32_t);
  CK(cudaFuncSetAttribute(k_pp_sort_rows, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem), "shared memory");
  k_pp_sort_rows<<<grid_blocks(ctx, g.n, 256), 256, smem, ctx->stream>>>(g);
  return ZEF_OK;
}

// ---- smoothing
// The positions are held as float4 while the iterations run: a neighbour is
// one 16-byte read of one sector instead of three 4-byte reads over one or
// two.  Ten iterations on 3.8 M nodes and 20 M edges: 4.8 ms with packed
// positions and one thread summing the blocks' partial sums (140 us of each
// iteration), 2.5 ms now: 120 us a step, bound by the L1's handling of a
// warp's 32 scattered 16-byte reads (44 M a step).  Rows interleaved by warp,
// indices read four at a time, or staged in shared memory by the warp, took
// 145, 130 and 140.
struct Smooth {
  Adj g;
  float4 *x, *y;           // positions [n]: x current, y after the forward step
  const uint8_t *fixed;    // nullable
  float lambda, mu, xi;
  const double *x0;        // ||x^(0)||_2 (device)
  int max_iters;
  double *partial;         // per-block sums of squares of the forward step
  int nblocks;
};

// Sum of v over the block's 256 threads in a fixed order (thread 0 has it).
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double red[256];
  red[threadIdx.x] = v;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  return red[0];
}

// p + w sum_j (p_j - p), j the neighbours of node i in ascending order
__device__ __forceinline__ float4 lap_step(const Adj &g, const float4 *p, int64_t i, float4 c, float weight) {
  const uint32_t len = g.fill[i];
  const int32_t *r = g.nbr + g.deg[i];
  float a0 = 0.f, a1 = 0.f, a2 = 0.f;
  for (uint32_t k = 0; k < len; ++k) {
    const float4 q = p[r[k]];
    a0 += q.x - c.x;
    a1 += q.y - c.y;
    a2 += q.z - c.z;
  }
  const float w = weight / (float)(len + 1);
  return make_float4(fmaf(w, a0, c.x), fmaf(w, a1, c.y), fmaf(w, a2, c.z), 0.f);
}

// y = x + lambda L(x) (fixed nodes keep x); block sums of |y - x|^2 in a fixed
// order.  With xi = 0 only a sum of zero stops the loop, so NORM = false leaves
// 1 when some node of the block moved, else 0, and does no FP64 work.
// With BOUNDARY the norms run over the nodes that have a neighbour.
template <bool NORM, bool BOUNDARY>
__global__ void __launch_bounds__(256) k_sm_forward(Smooth s) {
  if (s.g.words[PP_STOP]) return;
  double acc = 0.0;
  bool moved = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < s.g.n; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 c = s.x[i];
    float4 o = c;
    if (!(s.fixed && s.fixed[i])) o = lap_step(s.g, s.x, i, c, s.lambda);
    s.y[i] = o;
    if (BOUNDARY && !s.g.fill[i]) continue;
    if (NORM) {
      const double d0 = (double)o.x - c.x, d1 = (double)o.y - c.y, d2 = (double)o.z - c.z;
      acc += d0 * d0 + d1 * d1 + d2 * d2;
    } else {
      moved |= o.x != c.x || o.y != c.y || o.z != c.z;  // true for NaN, whose sum is not zero either
    }
  }
  const double sum = NORM ? block_sum(acc) : (__syncthreads_or(moved) ? 1.0 : 0.0);
  if (threadIdx.x == 0) s.partial[blockIdx.x] = sum;
}

// x = y - mu L(y) (fixed nodes keep y)
__global__ void __launch_bounds__(256) k_sm_backward(Smooth s) {
  if (s.g.words[PP_STOP]) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < s.g.n; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 c = s.y[i];
    float4 o = c;
    if (!(s.fixed && s.fixed[i])) o = lap_step(s.g, s.y, i, c, -s.mu);
    s.x[i] = o;
  }
}

// one block: the forward step's relative size decides whether to continue
__global__ void __launch_bounds__(256) k_sm_next(Smooth s) {
  if (s.g.words[PP_STOP]) return;
  double acc = 0.0;
  for (int b = threadIdx.x; b < s.nblocks; b += 256) acc += s.partial[b];
  const double ss = block_sum(acc);
  if (threadIdx.x != 0) return;
  const int64_t it = ++s.g.words[PP_ITER];
  const double x0 = *s.x0;
  // an infinite coordinate: its difference, and so the ratio, is not a number,
  // which is not small (and which the NORM = false form does not see)
  const bool small = x0 > 0.0 ? !isinf(x0) && sqrt(ss) / x0 <= (double)s.xi : true;
  if (small || it >= s.max_iters || s.g.words[PP_BAD]) s.g.words[PP_STOP] = 1;
}

// positions into float4 and their sum of squares (with `len`, the rows'
// lengths, only of the nodes that have a neighbour): block sums in a fixed
// order, then one block
__global__ void __launch_bounds__(256) k_sm_pack(const float *x, int64_t n, const uint32_t *len, float4 *out,
                                                 double *partial) {
  double acc = 0.0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 p = make_float4(x[3 * i], x[3 * i + 1], x[3 * i + 2], 0.f);
    out[i] = p;
    if (!len || len[i]) acc += (double)p.x * p.x + (double)p.y * p.y + (double)p.z * p.z;
  }
  const double sum = block_sum(acc);
  if (threadIdx.x == 0) partial[blockIdx.x] = sum;
}

__global__ void __launch_bounds__(256) k_sm_norm(const double *partial, int nblocks, double *x0) {
  double acc = 0.0;
  for (int b = threadIdx.x; b < nblocks; b += 256) acc += partial[b];
  const double sum = block_sum(acc);
  if (threadIdx.x == 0) *x0 = sqrt(sum);
}

__global__ void __launch_bounds__(256) k_sm_unpack(const float4 *p, int64_t n, float *x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float4 q = p[i];
    x[3 * i] = q.x;
    x[3 * i + 1] = q.y;
    x[3 * i + 2] = q.z;
  }
}

__global__ void k_pp_words(int64_t *w) {
  if (threadIdx.x < PP_WORDS) w[threadIdx.x] = 0;
}

// ---- inflation
// ---- crossing edges: (inside node, outside node) pairs of the tets, each once
__global__ void __launch_bounds__(256) k_in_bits(const unsigned long long *mask, int row, int64_t n, uint8_t *inside) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    inside[i] = (uint8_t)(mask[i] >> row & 1ull);
}

__device__ __forceinline__ uint32_t inside_bits(const uint8_t *inside, const int32_t (&v)[4]) {
  uint32_t b = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) b |= inside[v[k]] ? 1u << k : 0u;
  return b;
}

// their number with repeats, for the table's size
__global__ void __launch_bounds__(256) k_in_count(const int32_t *tets, int64_t m, int64_t n, const uint8_t *inside,
                                                 int64_t *words, uint32_t *status) {
  uint32_t c = 0;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < m; t += (int64_t)gridDim.x * blockDim.x) {
    int32_t v[4];
    if (!load_tet(tets, t, n, v)) {
      atomicOr(status, ST_INVALID);
      atomicExch((unsigned long long *)(words + PP_BAD), 1ull);
      continue;
    }
    const uint32_t k = __popc(inside_bits(inside, v));
    c += k * (4u - k);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd((unsigned long long *)(words + PP_CAND), (unsigned long long)c);
}

// the pairs, with repeats, into a list
__global__ void __launch_bounds__(256) k_in_pairs(const int32_t *tets, int64_t m, int64_t n, const uint8_t *inside,
                                                 unsigned long long *pairs, int64_t *words) {
  for (int64_t t0 = blockIdx.x * (int64_t)blockDim.x; t0 < m; t0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = t0 + threadIdx.x;
    int32_t v[4] = {0, 0, 0, 0};
    uint32_t b = 0;
    if (t < m && load_tet(tets, t, n, v)) b = inside_bits(inside, v);
    const uint32_t c = __popc(b) * (4 - __popc(b));
    unsigned long long at = block_places(c, words + PP_POOL);
    if (c)
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y)
          if (x != y && (b >> x & 1u) && !(b >> y & 1u))
            pairs[at++] = ((unsigned long long)(uint32_t)v[x] << 32) | (uint32_t)v[y];
  }
}

// the list into the table (more slots than pairs), one thread per pair; a
// pair's first insertion counts it at the inside node.  (A thread per tet
// waited for up to four swaps in turn, in warps of few crossing tets: 0.63 ms
// for 14.7 M tets.)
__global__ void __launch_bounds__(256) k_in_insert(const unsigned long long *pairs, const int64_t *count,
                                                  unsigned long long *keys, unsigned long long mask, uint32_t *off) {
  const int64_t len = *count;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < len; k += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long key = pairs[k];
    unsigned long long h = pp_mix(key) & mask;
    for (;;) {  // ends: fewer pairs than slots
      const unsigned long long prev = atomicCAS(keys + h, kNoKey, key);
      if (prev == kNoKey) {
        atomicAdd(off + (uint32_t)(key >> 32), 1u);
        break;
      }
      if (prev == key) break;
      h = (h + 1) & mask;
    }
  }
}

// the table's pairs into the nodes' shares of the list
__global__ void __launch_bounds__(256) k_in_list(const unsigned long long *keys, unsigned long long mask,
                                                const uint32_t *off, uint32_t *fill, int2 *edges) {
  for (unsigned long long s = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; s <= mask;
       s += (unsigned long long)gridDim.x * blockDim.x) {
    const unsigned long long key = keys[s];
    if (key == kNoKey) continue;
    const uint32_t a = (uint32_t)(key >> 32);
    edges[off[a] + atomicAdd(fill + a, 1u)] = make_int2((int)a, (int)(uint32_t)key);
  }
}

// each node's crossing edges in ascending neighbour order (a few per node)
__global__ void __launch_bounds__(256) k_in_sort(int64_t n, const uint32_t *off, int2 *edges) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t b = off[i], e = off[i + 1];
    for (uint32_t k = b + 1; k < e; ++k) {
      const int2 v = edges[k];
      uint32_t j = k;
      while (j > b && edges[j - 1].y > v.y) {
        edges[j] = edges[j - 1];
        --j;
      }
      edges[j] = v;
    }
  }
}

// Edge parameter of the nearest intersection of each crossing edge with the
// compartment's triangles, infinity when there is none (Moller-Trumbore in
// FP32 on the scaled coordinates, inclusive by a relative 2^-20 so that an
// edge through a shared triangle edge still hits).  Eight lanes per edge.  The
// candidates are the triangles listed in the cells of the compartment's grid
// that the edge's box, grown by 2^-10, meets (a lane per cell): any triangle
// the edge meets has a point that close to it, whose cell lists the triangle,
// so the minimum is the one over all triangles.  A compartment without a grid,
// and an edge whose box meets more than kInCells cells (a mesh far coarser
// than the surface), take the leaves of the cap tree whose box meets the
// edge's box (one lane walks the tree); more than kInLeaves of them fall back
// to every triangle.  900,000 edges of a refined head: 0.30 ms, the chain of
// reads (word, block, vertices) of each edge; a warp per node, taking one edge
// after the other, needed 1.35 ms with the tree and 1.14 with the cells.
constexpr int kInLanes = 8;
constexpr int kInLeaves = 32;
constexpr int kInCells = 4096;

__global__ void __launch_bounds__(256) k_in_hits(const int2 *edges, const uint32_t *count, const float *x, const float4 *tris,
                                                int tri_cnt, const CapNode *nodes, int root, const int32_t *ctidx,
                                                float scale, GridComp cells, float *hit) {
  __shared__ int2 s_leaf[256 / kInLanes][kInLeaves];  // per edge: (first position in ctidx, triangles)
  const int l = threadIdx.x % kInLanes, slot = threadIdx.x / kInLanes;
  const uint32_t lanes = ((1u << kInLanes) - 1u) << (threadIdx.x & 31 & ~(kInLanes - 1));
  constexpr float kEps = 9.5367431640625e-07f;  // 2^-20
  constexpr float kBoxMargin = 9.765625e-04f;   // 2^-10
  const int64_t step = (int64_t)gridDim.x * (256 / kInLanes), n_edges = *count;
  for (int64_t w = (int64_t)blockIdx.x * (256 / kInLanes) + slot; w < n_edges; w += step) {
    const int64_t i = edges[w].x, j = edges[w].y;
    const float q[3] = {x[3 * i], x[3 * i + 1], x[3 * i + 2]};
    const float ed[3] = {x[3 * j] - q[0], x[3 * j + 1] - q[1], x[3 * j + 2] - q[2]};
    const float p0 = q[0] * scale, p1 = q[1] * scale, p2 = q[2] * scale;
    const float d0 = ed[0] * scale, d1 = ed[1] * scale, d2 = ed[2] * scale;
    float tmin = INFINITY;
    auto test = [&](int t) {
      const float4 A = tris[3 * t], B = tris[3 * t + 1], C = tris[3 * t + 2];
      const float ax = B.x - A.x, ay = B.y - A.y, az = B.z - A.z;   // edge 1
      const float bx = C.x - A.x, by = C.y - A.y, bz = C.z - A.z;   // edge 2
      const float px = d1 * bz - d2 * by, py = d2 * bx - d0 * bz, pz = d0 * by - d1 * bx;
      const float det = ax * px + ay * py + az * pz;
      if (det == 0.f) return;
      const float inv = 1.f / det;
      const float tx = p0 - A.x, ty = p1 - A.y, tz = p2 - A.z;
      const float u = (tx * px + ty * py + tz * pz) * inv;
      if (u < -kEps || u > 1.f + kEps) return;
      const float qx = ty * az - tz * ay, qy = tz * ax - tx * az, qz = tx * ay - ty * ax;
      const float v = (d0 * qx + d1 * qy + d2 * qz) * inv;
      if (v < -kEps || u + v > 1.f + kEps) return;
      const float tt = (bx * qx + by * qy + bz * qz) * inv;
      if (tt >= 0.f && tt <= 1.f + kEps) tmin = fminf(tmin, tt);
    };
    int c0[3] = {0, 0, 0}, cn[3] = {0, 0, 0};
    int64_t total = kInCells + 1;  // cells the edge's box meets
    if (cells.words) {
      const float grow = kBoxMargin / scale;  // a power of two
      bool miss = false;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float lo = fminf(q[d], q[d] + ed[d]) - grow, hi = fmaxf(q[d], q[d] + ed[d]) + grow;
        miss |= hi < cells.lo[d] || lo > cells.hi[d];
        c0[d] = min(max((int)((fmaxf(lo, cells.lo[d]) - cells.lo[d]) * cells.inv[d]), 0), cells.n[d] - 1);
        cn[d] = min(max((int)((fminf(hi, cells.hi[d]) - cells.lo[d]) * cells.inv[d]), 0), cells.n[d] - 1) - c0[d] + 1;
      }
      total = miss ? 0 : (int64_t)cn[0] * cn[1] * cn[2];
    }
    if (total <= kInCells) {
      for (int c = l; c < (int)total; c += kInLanes) {
        const int cx = c0[0] + c % cn[0], cy = c0[1] + c / cn[0] % cn[1], cz = c0[2] + c / cn[0] / cn[1];
        const uint32_t word = cells.words[((int64_t)cz * cells.n[1] + cy) * cells.n[0] + cx];
        if (!(word & kCellMixed)) continue;
        const float4 *block = cells.blocks + (word & kCellOffset);
        const int entries = (int)(__float_as_uint(block[0].w) >> 8);
        for (int e = 0; e < entries; ++e) test(__float_as_int(block[1 + e / kSub * kChunkWords + 2 * kSub + e % kSub].w));
      }
    } else {
      int nl = 0;
      if (l == 0) {
        const float lo0 = fminf(p0, p0 + d0) - kBoxMargin, hi0 = fmaxf(p0, p0 + d0) + kBoxMargin;
        const float lo1 = fminf(p1, p1 + d1) - kBoxMargin, hi1 = fmaxf(p1, p1 + d1) + kBoxMargin;
        const float lo2 = fminf(p2, p2 + d2) - kBoxMargin, hi2 = fmaxf(p2, p2 + d2) + kBoxMargin;
        // pre-order walk without a stack: descend to i + 1, or continue at skip
        const int end = nodes[root].skip;
        for (int k = root; k != end;) {
          const CapNode nd = nodes[k];
          if (nd.hi[0] < lo0 || nd.lo[0] > hi0 || nd.hi[1] < lo1 || nd.lo[1] > hi1 || nd.hi[2] < lo2 ||
              nd.lo[2] > hi2) {
            k = nd.skip;
          } else if (nd.left < 0) {
            if (nl < kInLeaves) s_leaf[slot][nl] = make_int2(nd.tri_begin, nd.leaf_tris);
            ++nl;
            k = nd.skip;
          } else {
            ++k;
          }
        }
      }
      nl = __shfl_sync(lanes, nl, 0, kInLanes);
      __syncwarp(lanes);
      const bool all = nl > kInLeaves;
      for (int s = 0; s < (all ? 1 : nl); ++s) {
        const int2 L = all ? make_int2(0, tri_cnt) : s_leaf[slot][s];
        for (int k = l; k < L.y; k += kInLanes) test(all ? k : ctidx[L.x + k]);
      }
      __syncwarp(lanes);  // the leaf list is rewritten for the next edge
    }
#pragma unroll
    for (int o = kInLanes / 2; o > 0; o >>= 1) tmin = fminf(tmin, __shfl_xor_sync(lanes, tmin, o));
    if (l == 0) hit[w] = tmin;
  }
}

// Moves of the nodes with an intersection, averaged over their crossing edges
// in ascending neighbour order.
__global__ void __launch_bounds__(256) k_in_move(int64_t n, const uint32_t *off, const int2 *edges, const float *hit,
                                                const float *x, float4 *moved, float zeta, int64_t *words) {
  uint32_t count = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = off[i], e = off[i + 1];
    float m0 = 0.f, m1 = 0.f, m2 = 0.f;
    int cnt = 0;
    for (int64_t k = b; k < e; ++k) {
      if (!(hit[k] < INFINITY)) continue;
      const int64_t j = edges[k].y;
      const float tc = fminf(hit[k], 1.f);
      m0 = fmaf(zeta * tc, x[3 * j] - x[3 * i], m0);
      m1 = fmaf(zeta * tc, x[3 * j + 1] - x[3 * i + 1], m1);
      m2 = fmaf(zeta * tc, x[3 * j + 2] - x[3 * i + 2], m2);
      ++cnt;
    }
    if (e > b) moved[b] = make_float4(x[3 * i] + m0 / (float)cnt, x[3 * i + 1] + m1 / (float)cnt,
                                      x[3 * i + 2] + m2 / (float)cnt, cnt > 0 ? 1.f : 0.f);
    count += cnt > 0 ? 1u : 0u;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) count += __shfl_xor_sync(0xffffffffu, count, o);
  if ((threadIdx.x & 31) == 0 && count) atomicAdd((unsigned long long *)(words + PP_STOP), (unsigned long long)count);
}

// the moved nodes' positions (after every move has been computed from the old ones)
__global__ void __launch_bounds__(256) k_in_store(int64_t n, const uint32_t *off, const float4 *moved, float *x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = off[i];
    if (off[i + 1] == b) continue;
    const float4 p = moved[b];
    if (p.w == 0.f) continue;
    x[3 * i] = p.x;
    x[3 * i + 1] = p.y;
    x[3 * i + 2] = p.z;
  }
}

bool on_dev(const void *p, int device) {
  cudaPointerAttributes a;
  if (!p || cudaPointerGetAttributes(&a, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return (a.type == cudaMemoryTypeDevice && a.device == device) || a.type == cudaMemoryTypeManaged;
}

// post-processing scratch: grow-only device buffers of the context
zef_status pp_grow(zef_ctx *ctx, int idx, size_t bytes) {
  if (ctx->pp_buf[idx] && ctx->pp_cap[idx] >= bytes) return ZEF_OK;
  if (ctx->pp_buf[idx]) cudaFree(ctx->pp_buf[idx]);
  ctx->pp_buf[idx] = nullptr;
  ctx->pp_cap[idx] = 0;
  CK(cudaMalloc(&ctx->pp_buf[idx], std::max<size_t>(bytes, 256)), "cudaMalloc(post-processing)");
  ctx->pp_cap[idx] = bytes;
  return ZEF_OK;
}

// log2 of the table slots per node: the largest s with n 2^s <= cap
int slot_shift(int64_t cap, int64_t n) {
  int sh = 0;
  while (sh < 40 && (std::max<int64_t>(n, 1) << (sh + 1)) <= cap) ++sh;
  return sh;
}

// Rows of the tets' unique edges (buffers 0-5 of pp_buf); synchronizes.  The
// pool's offsets have 32 bits and a run may need 20 words per tet; meshes
// beyond that take the table of unique edges (12 to 24 slots of 8 bytes per
// tet to clear, to fill with one swap per tet edge and to scan: 4.4 ms where
// the pieces take 1.8, 14.7 M tets).
zef_status build_adjacency(zef_ctx *ctx, const int32_t *tets, int64_t m, int64_t n, Adj *out) {
  const int64_t runs = (m + kRunTets - 1) / kRunTets;
  const bool pieces = runs * kRunPool < (int64_t)kNoPiece;
  int64_t cap = 1024;
  while (!pieces && cap < 12 * std::max<int64_t>(m, 1)) cap <<= 1;  // 6 m edge slots, load <= 1/2
  zef_status st;
  if ((st = pp_grow(ctx, 0, pieces ? (size_t)std::max<int64_t>(runs, 1) * kRunPool * sizeof(uint32_t)
                                   : (size_t)cap * sizeof(unsigned long long)))) return st;
  if ((st = pp_grow(ctx, 1, (size_t)(n + 1) * sizeof(uint32_t)))) return st;
  if ((st = pp_grow(ctx, 2, (size_t)std::max<int64_t>(n, 1) * sizeof(uint32_t)))) return st;
  if ((st = pp_grow(ctx, 4, (size_t)PP_WORDS * sizeof(int64_t)))) return st;
  if ((st = pp_grow(ctx, 5, (size_t)std::max<int64_t>((n + 1) / 2048 + 2, n) * sizeof(uint32_t)))) return st;
  Adj g;
  g.keys = (unsigned long long *)ctx->pp_buf[0];
  g.mask = (unsigned long long)(cap - 1);
  g.shift = slot_shift(cap, n);
  g.deg = (uint32_t *)ctx->pp_buf[1];
  g.fill = (uint32_t *)ctx->pp_buf[2];
  g.nbr = nullptr;
  g.n = n;
  g.words = (int64_t *)ctx->pp_buf[4];
  cudaStream_t s = ctx->stream;
  uint32_t *pool = (uint32_t *)ctx->pp_buf[0], *head = (uint32_t *)ctx->pp_buf[5];
  k_pp_words<<<1, 32, 0, s>>>(g.words);
  int64_t words[PP_WORDS];
  uint32_t deg_sum = 0;
  if (pieces) {
    CK(cudaMemsetAsync(head, 0xff, (size_t)std::max<int64_t>(n, 1) * sizeof(uint32_t), s), "clear piece lists");
    CK(cudaFuncSetAttribute(k_pp_runs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRunShared), "shared memory");
    if (m > 0)
      k_pp_runs<<<(unsigned)std::min<int64_t>(runs, (int64_t)ctx->num_sms * 12), kRunThreads, kRunShared, s>>>(
          n, tets, m, pool, head, g.words, ctx->d_status);
  } else {
    CK(cudaMemsetAsync(g.deg, 0, (size_t)(n + 1) * sizeof(uint32_t), s), "clear degrees");
    CK(cudaMemsetAsync(g.fill, 0, (size_t)std::max<int64_t>(n, 1) * sizeof(uint32_t), s), "clear cursors");
    CK(cudaMemsetAsync(g.keys, 0xff, (size_t)cap * sizeof(unsigned long long), s), "clear edge table");
    k_pp_edges<<<grid_blocks(ctx, m, 256), 256, 0, s>>>(g, tets, m, ctx->d_status);
    st = scan_exclusive(ctx, g.deg, nullptr, 1, n + 1, nullptr, (uint32_t *)ctx->pp_buf[5]);
    if (st) return st;
    CK(cudaMemcpyAsync(&deg_sum, g.deg + n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s), "read edge count");
  }
  CK(cudaMemcpyAsync(words, g.words, sizeof(words), cudaMemcpyDeviceToHost, s), "read adjacency status");
  CK(cudaStreamSynchronize(s), "build adjacency");
  if (words[PP_BAD]) {
    zef_synchronize(ctx);  // clears the recorded status
    return fail(ctx, ZEF_ERR_INVALID_ARG, "a tet references a node index outside [0, num_nodes)");
  }
  // the rows hold at most the pool's neighbours
  const int64_t entries = pieces ? words[PP_POOL] : (int64_t)deg_sum;
  if ((st = pp_grow(ctx, 3, (size_t)std::max<int64_t>(entries, 1) * sizeof(int32_t)))) return st;
  g.nbr = (int32_t *)ctx->pp_buf[3];
  if (pieces) {
    constexpr size_t smem = (size_t)8 * kColumn * 32 * sizeof(int32_t);
    CK(cudaFuncSetAttribute(k_pp_merge, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem), "shared memory");
    k_pp_merge<<<grid_blocks(ctx, n, 256), 256, smem, s>>>(g, pool, head);
  } else {
    k_pp_scatter<<<grid_blocks(ctx, cap, 256), 256, 0, s>>>(g);
    if ((st = sort_rows(ctx, g))) return st;
  }
  CK(cudaGetLastError(), "adjacency kernels");
  *out = g;
  return ZEF_OK;
}

}  // namespace

namespace {

// The Taubin iteration loop over the adjacency g, on device positions x; with
// `boundary_norm` the starting norm runs over the nodes that have a
// neighbour.  The iterations are enqueued in batches (one, two, four, ... up
// to 32; all at once up to 32 when the stop rule can only end on a standstill,
// xi = 0) whose kernels return at once after the one that stopped, and the
// host looks between batches: building and instantiating a conditional graph
// per call cost more than the launches.  Writes the iterations run; the
// caller copies back.
zef_status smooth_loop(zef_ctx *ctx, float *x, int64_t n, const Adj &g, const uint8_t *fx, const zef_smooth_opts &o,
                       bool boundary_norm, int64_t *words) {
  cudaStream_t s = ctx->stream;
  zef_status st;
  const int threads = 256;
  const int nblocks = grid_blocks(ctx, n, threads);
  if ((st = pp_grow(ctx, 9, (size_t)n * 2 * sizeof(float4)))) return st;
  if ((st = pp_grow(ctx, 10, (size_t)(nblocks + 1) * sizeof(double)))) return st;
  double *partial = (double *)ctx->pp_buf[10];
  Smooth sm;
  sm.g = g;
  sm.x = (float4 *)ctx->pp_buf[9];
  sm.y = sm.x + n;
  sm.fixed = fx;
  sm.lambda = o.lambda;
  sm.mu = o.mu;
  sm.xi = o.xi;
  sm.x0 = partial + nblocks;
  sm.max_iters = o.max_iters;
  sm.partial = partial;
  sm.nblocks = nblocks;
  k_sm_pack<<<nblocks, threads, 0, s>>>(x, n, boundary_norm ? g.fill : nullptr, sm.x, partial);
  k_sm_norm<<<1, threads, 0, s>>>(partial, nblocks, partial + nblocks);
  auto forward = o.xi > 0.f ? (boundary_norm ? k_sm_forward<true, true> : k_sm_forward<true, false>)
                            : (boundary_norm ? k_sm_forward<false, true> : k_sm_forward<false, false>);
  int batch = o.xi > 0.f ? 1 : 32;
  for (int left = o.max_iters; left > 0;) {
    const int k = std::min(batch, left);
    for (int q = 0; q < k; ++q) {
      forward<<<nblocks, threads, 0, s>>>(sm);
      k_sm_backward<<<nblocks, threads, 0, s>>>(sm);
      k_sm_next<<<1, threads, 0, s>>>(sm);
    }
    left -= k;
    batch = std::min(2 * batch, 32);
    if (left == 0) break;
    CK(cudaMemcpyAsync(words, g.words, PP_WORDS * sizeof(int64_t), cudaMemcpyDeviceToHost, s), "read smoothing state");
    CK(cudaStreamSynchronize(s), "smoothing");
    if (words[PP_STOP]) break;
  }
  k_sm_unpack<<<nblocks, threads, 0, s>>>(sm.x, n, x);
  CK(cudaMemcpyAsync(words, g.words, PP_WORDS * sizeof(int64_t), cudaMemcpyDeviceToHost, s), "read smoothing state");
  CK(cudaGetLastError(), "smoothing kernels");
  CK(cudaStreamSynchronize(s), "smoothing");
  return ZEF_OK;
}

// Rows of the tissue-boundary faces' edges (buffers 0-5 as build_adjacency, 11
// for the listed faces, 14 for the face table, 15 and 16 for the nodes' labels
// and marks); synchronizes.  14.7 M tets of a refined head with 1.6 M boundary
// faces: 0.6 + 6.1 ms clearing a table for, and inserting, all 59 M faces, and
// 4.0 ms scanning it with one counter for all faces, before the faces were
// chosen by their nodes; 0.50 and 0.41 ms for table and edges with a thread
// per tet and per table slot, waiting for several swaps in turn.
zef_status build_surface_adjacency(zef_ctx *ctx, const int32_t *tets, const int32_t *labels, int64_t m, int64_t n,
                                   Adj *out, int64_t *faces) {
  zef_status st;
  if ((st = pp_grow(ctx, 1, (size_t)(n + 1) * sizeof(uint32_t)))) return st;
  if ((st = pp_grow(ctx, 2, (size_t)std::max<int64_t>(n, 1) * sizeof(uint32_t)))) return st;
  if ((st = pp_grow(ctx, 4, (size_t)PP_WORDS * sizeof(int64_t)))) return st;
  if ((st = pp_grow(ctx, 5, (size_t)((n + 1) / 2048 + 2) * sizeof(uint32_t)))) return st;
  if ((st = pp_grow(ctx, 15, (size_t)std::max<int64_t>(n, 1) * sizeof(int32_t)))) return st;
  if ((st = pp_grow(ctx, 16, (size_t)std::max<int64_t>(n, 1)))) return st;
  int32_t *first = (int32_t *)ctx->pp_buf[15];
  uint8_t *mixed = (uint8_t *)ctx->pp_buf[16];
  int64_t *dwords = (int64_t *)ctx->pp_buf[4];
  cudaStream_t s = ctx->stream;
  int64_t words[PP_WORDS] = {0};
  k_pp_words<<<1, 32, 0, s>>>(dwords);
  if (m > 0) {
    const int g_t = grid_blocks(ctx, m, 256);
    CK(cudaMemsetAsync(mixed, 0, (size_t)n, s), "clear node marks");
    k_sf_first<<<g_t, 256, 0, s>>>(tets, labels, m, n, first, dwords, ctx->d_status);
    k_sf_mixed<<<g_t, 256, 0, s>>>(tets, labels, m, n, first, mixed);
    k_sf_count<<<g_t, 256, 0, s>>>(tets, m, n, mixed, dwords);
    CK(cudaMemcpyAsync(words, dwords, sizeof(words), cudaMemcpyDeviceToHost, s), "read face count");
    CK(cudaStreamSynchronize(s), "boundary nodes");
    if (words[PP_BAD]) {
      zef_synchronize(ctx);  // clears the recorded status
      return fail(ctx, ZEF_ERR_INVALID_ARG, "a tet references a node index outside [0, num_nodes)");
    }
  }
  const int64_t cand = words[PP_CAND];
  if (cand == 0) {
    *faces = 0;
    return ZEF_OK;
  }
  int64_t fcap = 1024;
  while (fcap < 2 * cand) fcap <<= 1;     // load <= 1/2
  int64_t cap = 1024;
  while (cap < 3 * cand) cap <<= 1;       // a boundary face was counted twice: at most 3/2 cand edges, load <= 1/2
  if ((st = pp_grow(ctx, 14, (size_t)fcap * (2 * sizeof(unsigned long long) + 2 * sizeof(int32_t))))) return st;
  if ((st = pp_grow(ctx, 0, (size_t)cap * sizeof(unsigned long long)))) return st;
  if ((st = pp_grow(ctx, 11, (size_t)cand * sizeof(FaceItem)))) return st;
  FaceItem *items = (FaceItem *)ctx->pp_buf[11];
  FaceTab f;
  f.keys = (unsigned long long *)ctx->pp_buf[14];
  f.lo = (int32_t *)(f.keys + 2 * fcap);
  f.hi = f.lo + fcap;
  f.mask = (unsigned long long)(fcap - 1);
  Adj g;
  g.keys = (unsigned long long *)ctx->pp_buf[0];
  g.mask = (unsigned long long)(cap - 1);
  g.shift = slot_shift(cap, n);
  g.deg = (uint32_t *)ctx->pp_buf[1];
  g.fill = (uint32_t *)ctx->pp_buf[2];
  g.nbr = nullptr;
  g.n = n;
  g.words = dwords;
  k_sf_clear<<<grid_blocks(ctx, fcap, 256), 256, 0, s>>>(f);
  CK(cudaMemsetAsync(g.keys, 0xff, (size_t)cap * sizeof(unsigned long long), s), "clear edge table");
  CK(cudaMemsetAsync(g.deg, 0, (size_t)(n + 1) * sizeof(uint32_t), s), "clear degrees");
  CK(cudaMemsetAsync(g.fill, 0, (size_t)std::max<int64_t>(n, 1) * sizeof(uint32_t), s), "clear cursors");
  k_sf_list<<<grid_blocks(ctx, m, 256), 256, 0, s>>>(tets, labels, m, n, mixed, items, dwords);
  k_sf_faces<<<grid_blocks(ctx, cand, 256), 256, 0, s>>>(f, items, dwords);
  // the list of candidates is free again: at most half as many boundary faces
  k_sf_boundary<<<grid_blocks(ctx, fcap, 256), 256, 0, s>>>(f, (uint4 *)items, dwords);
  k_sf_edges<<<grid_blocks(ctx, 3 * cand / 2, 256), 256, 0, s>>>((const uint4 *)items, g);
  st = scan_exclusive(ctx, g.deg, nullptr, 1, n + 1, nullptr, (uint32_t *)ctx->pp_buf[5]);
  if (st) return st;
  uint32_t deg_sum = 0;
  CK(cudaMemcpyAsync(words, g.words, sizeof(words), cudaMemcpyDeviceToHost, s), "read adjacency status");
  CK(cudaMemcpyAsync(&deg_sum, g.deg + n, sizeof(uint32_t), cudaMemcpyDeviceToHost, s), "read edge count");
  CK(cudaStreamSynchronize(s), "build boundary adjacency");
  if (words[PP_FULL]) return fail(ctx, ZEF_ERR_CUDA, "internal: face or edge table full");
  *faces = words[PP_FACES];
  if ((st = pp_grow(ctx, 3, (size_t)std::max<int64_t>((int64_t)deg_sum, 1) * sizeof(int32_t)))) return st;
  g.nbr = (int32_t *)ctx->pp_buf[3];
  k_pp_scatter<<<grid_blocks(ctx, cap, 256), 256, 0, s>>>(g);
  if ((st = sort_rows(ctx, g))) return st;
  CK(cudaGetLastError(), "boundary adjacency kernels");
  *out = g;
  return ZEF_OK;
}

}  // namespace

zef_status taubin_run(zef_ctx *ctx, float *nodes, int64_t n, const int32_t *tets, int64_t m, const uint8_t *fixed,
                      const zef_smooth_opts &o, int32_t *iters_out) {
  NvtxRange nvtx_("zef.taubin_smooth");
  const bool dn = on_dev(nodes, ctx->device);
  const bool dt = m == 0 ? dn : on_dev(tets, ctx->device);
  const bool df = fixed ? on_dev(fixed, ctx->device) : dn;
  if (!(dn == dt && dt == df)) return fail(ctx, ZEF_ERR_INVALID_ARG, "nodes, tets and fixed must all be host or all device");
  zef_status st;
  float *x = nodes;
  const int32_t *tt = tets;
  const uint8_t *fx = fixed;
  cudaStream_t s = ctx->stream;
  if (!dn) {  // stage host arrays (buffers 6: nodes, 7: tets, 8: fixed)
    if ((st = pp_grow(ctx, 6, (size_t)n * 3 * sizeof(float)))) return st;
    if ((st = pp_grow(ctx, 7, (size_t)std::max<int64_t>(m, 1) * 4 * sizeof(int32_t)))) return st;
    x = (float *)ctx->pp_buf[6];
    tt = (const int32_t *)ctx->pp_buf[7];
    CK(cudaMemcpyAsync(x, nodes, (size_t)n * 3 * sizeof(float), cudaMemcpyHostToDevice, s), "copy nodes");
    if (m > 0) CK(cudaMemcpyAsync((void *)tt, tets, (size_t)m * 4 * sizeof(int32_t), cudaMemcpyHostToDevice, s), "copy tets");
    if (fixed) {
      if ((st = pp_grow(ctx, 8, (size_t)n))) return st;
      fx = (const uint8_t *)ctx->pp_buf[8];
      CK(cudaMemcpyAsync((void *)fx, fixed, (size_t)n, cudaMemcpyHostToDevice, s), "copy fixed");
    }
  }
  Adj g;
  if ((st = build_adjacency(ctx, tt, m, n, &g))) return st;  // synchronizes
  int64_t words[PP_WORDS] = {0};
  if ((st = smooth_loop(ctx, x, n, g, fx, o, false, words))) return st;
  if (!dn) CK(cudaMemcpyAsync(nodes, x, (size_t)n * 3 * sizeof(float), cudaMemcpyDeviceToHost, s), "copy nodes back");
  if (iters_out) *iters_out = (int32_t)words[PP_ITER];
  return zef_synchronize(ctx);
}

zef_status taubin_surface_run(zef_ctx *ctx, float *nodes, int64_t n, const int32_t *tets, int64_t m,
                              const int32_t *elem_labels, const zef_smooth_opts &o, int32_t *iters_out,
                              int64_t *faces_out) {
  NvtxRange nvtx_("zef.taubin_smooth_surface");
  const bool dn = on_dev(nodes, ctx->device);
  const bool dt = m == 0 ? dn : on_dev(tets, ctx->device);
  const bool dl = m == 0 ? dn : on_dev(elem_labels, ctx->device);
  if (!(dn == dt && dt == dl))
    return fail(ctx, ZEF_ERR_INVALID_ARG, "nodes, tets and elem_labels must all be host or all device");
  zef_status st;
  float *x = nodes;
  const int32_t *tt = tets;
  const int32_t *lab = elem_labels;
  cudaStream_t s = ctx->stream;
  if (!dn) {  // stage host arrays (buffers 6: nodes, 7: tets, 17: labels)
    if ((st = pp_grow(ctx, 6, (size_t)n * 3 * sizeof(float)))) return st;
    if ((st = pp_grow(ctx, 7, (size_t)std::max<int64_t>(m, 1) * 4 * sizeof(int32_t)))) return st;
    if ((st = pp_grow(ctx, 17, (size_t)std::max<int64_t>(m, 1) * sizeof(int32_t)))) return st;
    x = (float *)ctx->pp_buf[6];
    tt = (const int32_t *)ctx->pp_buf[7];
    lab = (const int32_t *)ctx->pp_buf[17];
    CK(cudaMemcpyAsync(x, nodes, (size_t)n * 3 * sizeof(float), cudaMemcpyHostToDevice, s), "copy nodes");
    if (m > 0) {
      CK(cudaMemcpyAsync((void *)tt, tets, (size_t)m * 4 * sizeof(int32_t), cudaMemcpyHostToDevice, s), "copy tets");
      CK(cudaMemcpyAsync((void *)lab, elem_labels, (size_t)m * sizeof(int32_t), cudaMemcpyHostToDevice, s),
         "copy labels");
    }
  }
  Adj g;
  int64_t faces = 0;
  if ((st = build_surface_adjacency(ctx, tt, lab, m, n, &g, &faces))) return st;  // synchronizes
  int64_t words[PP_WORDS] = {0};
  if (faces > 0 && (st = smooth_loop(ctx, x, n, g, nullptr, o, true, words))) return st;
  if (!dn) CK(cudaMemcpyAsync(nodes, x, (size_t)n * 3 * sizeof(float), cudaMemcpyDeviceToHost, s), "copy nodes back");
  if (iters_out) *iters_out = (int32_t)words[PP_ITER];
  if (faces_out) *faces_out = faces;
  return zef_synchronize(ctx);
}

zef_status inflate_run(zef_ctx *ctx, float *nodes, int64_t n, const int32_t *tets, int64_t m, int32_t id,
                       float zeta, int64_t *moved_out) {
  NvtxRange nvtx_("zef.inflate");
  int row = -1, ci = -1;
  for (size_t r = 0; r < ctx->priority.size(); ++r)
    if (ctx->priority[r] == id) row = (int)r;
  for (size_t c = 0; c < ctx->comps.size(); ++c)
    if (ctx->comps[c].id == id) ci = (int)c;
  if (row < 0 || ci < 0) return fail(ctx, ZEF_ERR_INVALID_ARG, "unknown compartment id");
  const bool dn = on_dev(nodes, ctx->device);
  const bool dt = m == 0 ? dn : on_dev(tets, ctx->device);
  if (dn != dt) return fail(ctx, ZEF_ERR_INVALID_ARG, "nodes and tets must both be host or both device");
  zef_status st;
  float *x = nodes;
  const int32_t *tt = tets;
  cudaStream_t s = ctx->stream;
  if (!dn) {
    if ((st = pp_grow(ctx, 6, (size_t)n * 3 * sizeof(float)))) return st;
    if ((st = pp_grow(ctx, 7, (size_t)std::max<int64_t>(m, 1) * 4 * sizeof(int32_t)))) return st;
    x = (float *)ctx->pp_buf[6];
    tt = (const int32_t *)ctx->pp_buf[7];
    CK(cudaMemcpyAsync(x, nodes, (size_t)n * 3 * sizeof(float), cudaMemcpyHostToDevice, s), "copy nodes");
    if (m > 0) CK(cudaMemcpyAsync((void *)tt, tets, (size_t)m * 4 * sizeof(int32_t), cudaMemcpyHostToDevice, s), "copy tets");
  }
  // inside bits of every node (every compartment decided)
  if ((st = pp_grow(ctx, 11, (size_t)n * sizeof(unsigned long long)))) return st;
  if ((st = pp_grow(ctx, 12, (size_t)n * sizeof(int32_t)))) return st;
  unsigned long long *mask = (unsigned long long *)ctx->pp_buf[11];
  st = label_points_impl(ctx, x, n, (int32_t *)ctx->pp_buf[12], nullptr, nullptr, nullptr, mask, true);
  if (st) return st;
  // the crossing edges, by inside node (buffers 0 table, 1 offsets, 2 cursors,
  // 3 inside bytes): 14.7 M tets with 900,000 of them take 0.4 ms, the
  // neighbour rows of every node, from which they were read before, 1.8
  if ((st = pp_grow(ctx, 1, (size_t)(n + 1) * sizeof(uint32_t)))) return st;
  if ((st = pp_grow(ctx, 2, (size_t)n * sizeof(uint32_t)))) return st;
  if ((st = pp_grow(ctx, 3, (size_t)n))) return st;
  if ((st = pp_grow(ctx, 4, (size_t)PP_WORDS * sizeof(int64_t)))) return st;
  if ((st = pp_grow(ctx, 5, (size_t)((n + 1) / 2048 + 2) * sizeof(uint32_t)))) return st;
  uint32_t *off = (uint32_t *)ctx->pp_buf[1], *fill = (uint32_t *)ctx->pp_buf[2];
  uint8_t *inside = (uint8_t *)ctx->pp_buf[3];
  int64_t *dwords = (int64_t *)ctx->pp_buf[4];
  int64_t words[PP_WORDS];
  const int g_n = grid_blocks(ctx, n, 256), g_t = grid_blocks(ctx, std::max<int64_t>(m, 1), 256);
  k_pp_words<<<1, 32, 0, s>>>(dwords);
  k_in_bits<<<g_n, 256, 0, s>>>(mask, row, n, inside);
  if (m > 0) k_in_count<<<g_t, 256, 0, s>>>(tt, m, n, inside, dwords, ctx->d_status);
  CK(cudaMemcpyAsync(words, dwords, sizeof(words), cudaMemcpyDeviceToHost, s), "read crossing edges");
  CK(cudaStreamSynchronize(s), "crossing edges");
  if (words[PP_BAD]) {
    zef_synchronize(ctx);  // clears the recorded status
    return fail(ctx, ZEF_ERR_INVALID_ARG, "a tet references a node index outside [0, num_nodes)");
  }
  const int64_t crossing = words[PP_CAND];  // with repeats
  if (crossing == 0) {
    if (!dn) CK(cudaMemcpyAsync(nodes, x, (size_t)n * 3 * sizeof(float), cudaMemcpyDeviceToHost, s), "copy nodes back");
    return zef_synchronize(ctx);
  }
  int64_t cap = 1024;
  while (cap <= crossing) cap <<= 1;
  if ((st = pp_grow(ctx, 0, (size_t)cap * sizeof(unsigned long long)))) return st;
  unsigned long long *keys = (unsigned long long *)ctx->pp_buf[0];
  CK(cudaMemsetAsync(keys, 0xff, (size_t)cap * sizeof(unsigned long long), s), "clear edge table");
  CK(cudaMemsetAsync(off, 0, (size_t)(n + 1) * sizeof(uint32_t), s), "clear counts");
  CK(cudaMemsetAsync(fill, 0, (size_t)n * sizeof(uint32_t), s), "clear cursors");
  if ((st = pp_grow(ctx, 16, (size_t)crossing * sizeof(unsigned long long)))) return st;
  unsigned long long *pairs = (unsigned long long *)ctx->pp_buf[16];
  k_in_pairs<<<g_t, 256, 0, s>>>(tt, m, n, inside, pairs, dwords);
  k_in_insert<<<grid_blocks(ctx, crossing, 256), 256, 0, s>>>(pairs, dwords + PP_POOL, keys, (unsigned long long)(cap - 1),
                                                              off);
  st = scan_exclusive(ctx, off, nullptr, 1, n + 1, nullptr, (uint32_t *)ctx->pp_buf[5]);
  if (st) return st;
  // edges, their hits, the moved positions (at each node's first edge)
  if ((st = pp_grow(ctx, 14, (size_t)crossing * sizeof(int2)))) return st;
  if ((st = pp_grow(ctx, 15, (size_t)crossing * sizeof(float)))) return st;
  if ((st = pp_grow(ctx, 9, (size_t)crossing * sizeof(float4)))) return st;
  int2 *edges = (int2 *)ctx->pp_buf[14];
  float *hit = (float *)ctx->pp_buf[15];
  float4 *out = (float4 *)ctx->pp_buf[9];
  k_in_list<<<grid_blocks(ctx, cap, 256), 256, 0, s>>>(keys, (unsigned long long)(cap - 1), off, fill, edges);
  k_in_sort<<<g_n, 256, 0, s>>>(n, off, edges);
  const CompHost &c = ctx->comps[(size_t)ci];
  GridComp cells = {};
  if ((size_t)ci < ctx->grids.size() && ctx->grids[(size_t)ci].usable) {
    const CompGrid &cg = ctx->grids[(size_t)ci];
    for (int k = 0; k < 3; ++k) {
      cells.lo[k] = c.lo[k];
      cells.hi[k] = c.hi[k];
      cells.inv[k] = cg.inv[k];
      cells.n[k] = cg.n[k];
    }
    cells.words = cg.words;
    cells.blocks = cg.blocks;
  }
  k_in_hits<<<grid_blocks(ctx, crossing * kInLanes, 256), 256, 0, s>>>(
      edges, off + n, x, ctx->d_tris + c.tri_off * 3, (int)c.nt, ctx->d_nodes, c.cap_root, ctx->d_ctidx, ctx->scale,
      cells, hit);
  k_in_move<<<g_n, 256, 0, s>>>(n, off, edges, hit, x, out, zeta, dwords);
  k_in_store<<<g_n, 256, 0, s>>>(n, off, out, x);
  CK(cudaGetLastError(), "inflation kernels");
  if (!dn) CK(cudaMemcpyAsync(nodes, x, (size_t)n * 3 * sizeof(float), cudaMemcpyDeviceToHost, s), "copy nodes back");
  CK(cudaMemcpyAsync(words, dwords, sizeof(words), cudaMemcpyDeviceToHost, s), "read moved count");
  CK(cudaStreamSynchronize(s), "inflation");
  if (moved_out) *moved_out = words[PP_STOP];
  return zef_synchronize(ctx);
}

}  // namespace zef
