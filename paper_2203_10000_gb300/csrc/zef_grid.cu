// zef_grid.cu -- the cell grid of a compartment surface and the labeling
// kernel that reads it.
//
// The winding number of a closed surface S (Omega / 4 pi, Sec. 2.1.3) is
// constant on every region that S does not cross and changes by the signed
// count of crossings along a segment that does: k(p) = k(q) + (inward -
// outward crossings of the segment q -> p).  So the solid angle needs to be
// summed at a few fixed points only.  At registration every compartment's box
// is cut into cells one mean triangle edge wide; each cell lists the
// triangles that meet it, and one anchor point per cell gets its winding
// number from the solid-angle pipeline (FP32 certified, FP64 where it is not:
// zef_label.cu).  A point then takes
//   - 0 outside the compartment's box,
//   - the anchor's k in a cell that no triangle meets (a box the surface does
//     not cross: convex, hence connected),
//   - k(anchor) and the crossings of the segment anchor -> point with the
//     cell's triangles otherwise: the segment stays inside the cell, so no
//     other triangle can meet it.
//
// The crossing test of triangle (A, B, C) with d = p - q and a, b, c = A, B,
// C - q: v_ab = d . (a x b), v_bc, v_ca (the line through q and p passes
// inside the triangle when they have one sign), V = a . (b x c) and S = v_ab +
// v_bc + v_ca (the plane is met at V / S along the segment).  The cross
// products and V depend on (cell, triangle) alone: they are computed in FP64
// at registration and stored rounded to FP32 with a bound E on the error of
// the FP32 dot products, so a test is nine multiply-adds and a few compares.
// A decision is taken only from quantities beyond their bounds.  Anything
// else -- a point within about 1e-5 cell widths of a triangle's plane inside
// the triangle, a segment that close to an edge -- is re-evaluated in FP64
// from the vertices (again with a bound), and what FP64 cannot decide either
// (a point on the surface) by the FP64 solid angle over the cap tree, in the
// order of additions of zef_label.cu's re-evaluation of whole pairs.
//
// Why: the general kernels sum about 1,000 strip entries of a tile's walk for
// every point near a surface (FP32 ALUs, 54 of the 58 ms of 56.2 M points in
// 24 compartments); here such a point costs about a dozen crossing tests by
// four lanes, and every other point one cell of the label field (below).  No
// sort of the points: one launch, three for large calls, which list the points
// that the field leaves open and, of these, those on a surface.
// 56.2 M points in 24 compartments take 0.51 ms (58 ms with the tile kernels,
// 2.4 ms when every compartment met by a warp was looked up and its cells
// taken one after the other), 20.5 M in 20 small structures 0.10 ms (2.8),
// 36,864 with solid angles 8.2 us (258), 4,096 vertices of a surface 1.06 ms
// (2.9).  What bounds them now: the streaming kernel is near half the copy
// bandwidth (12 + 4 bytes a point), the open points' kernel waits on its two
// dependent L2 reads per point, points on a surface on the FP64 pipe.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "zef_fp64.cuh"
#include "zef_internal.h"

#define CK(call, what)                                      \
  do {                                                      \
    cudaError_t e_ = (call);                                \
    if (e_ != cudaSuccess) return cuda_fail(ctx, e_, what); \
  } while (0)

namespace zef {

namespace {

constexpr float kFourPi = 12.5663706143591729539f;
constexpr double kTwoPi64 = 6.283185307179586476925;
// Cell word of a cell that triangles meet: the top bit, the chunks of its
// block in two bits (0: more than three, see the block's header), and the
// block's offset in 16-byte words.  Otherwise the winding number (8 bits), or
// kUnknown.
constexpr uint32_t kMixed = kCellMixed;
constexpr uint32_t kUnknown = 0x40000000u;
constexpr int kChunkShift = kCellChunkShift;
constexpr uint32_t kOffsetMask = kCellOffset;
// W = v_ab + v_bc + v_ca - V, the point's side of the plane, is off by at most
// 8 E; four times that is left to FP64, so that it decides wherever the point is
// within about 1e-5 cell widths of a triangle.
constexpr float kPlane = 32.f;
constexpr int kNoK = -128;  // block header: the anchor's winding number is unknown
// A block: a header (anchor x, y, z; k in the low 8 bits of w and the number
// of triangles above), then chunks of kSub entries: kSub first words (a x b, V),
// kSub second (b x c, error bound), kSub third (c x a, triangle index), so
// that kSub lanes read 128 bytes at a time.  The last chunk is filled up with
// entries that the test calls a miss.
// Every cell is treated as grown by kGrow of its width on each side: a point
// whose cell index is off by the rounding of (x - lo) * n / extent (at most a
// few 2^-24 n of a cell, n <= 512) still lies in the grown cell.
constexpr double kGrow = 2e-3;
constexpr float kGrowF = 2e-3f;
constexpr int64_t kMaxCells = 1 << 23;
constexpr int kMaxAxis = 512;
// Cells of the label field: 32 MB (64 with more than 32 compartments), which
// the L2 holds beside the blocks in use.  56.2 M points: 657 us with 2^21
// cells, 630 with 2^22, 607 with 2^23; 20.5 M points in 20 small structures:
// 108, 109 and 111.
constexpr int64_t kMaxField = 1 << 22;
constexpr double kBoxCells = 67108864.0;  // cells of the triangles' boxes that any surface may have (a few ms)
constexpr size_t kScratchKept = (size_t)32 << 20;  // bytes of construction scratch kept between registrations
constexpr int kMaxList = 1024;  // longest triangle list of a usable grid

struct Geom {
  float lo[3], inv[3];
  double h[3];
  int n[3];
};

__device__ __forceinline__ float4 raw_vertex(float4 v, float s) { return make_float4(v.x * s, v.y * s, v.z * s, 0.f); }

// True when the projections of the triangle (vertices v relative to the cell's
// centre) and of the cell (half extents r) on axis edge x e_d separate them.
// FP32: its error, a few 2^-24 of the triangle's size (at most kMaxAxis cells),
// is far below the growth in r.
__device__ __forceinline__ bool axis_separates(const float (&v)[3][3], const float (&edge)[3], int d, const float (&r)[3]) {
  const int d1 = (d + 1) % 3, d2 = (d + 2) % 3;  // e_d x edge = (0, -edge_d2, edge_d1) on (d, d1, d2)
  const float a1 = -edge[d2], a2 = edge[d1];
  const float p0 = a1 * v[0][d1] + a2 * v[0][d2], p1 = a1 * v[1][d1] + a2 * v[1][d2], p2 = a1 * v[2][d1] + a2 * v[2][d2];
  const float reach = fabsf(a1) * r[d1] + fabsf(a2) * r[d2];
  return fminf(p0, fminf(p1, p2)) > reach || fmaxf(p0, fmaxf(p1, p2)) < -reach;
}

// Triangles of every cell: one warp per triangle, the lanes over the cells of
// its box; a cell counts unless one of the separating axes of a triangle and a
// box (the box's own by the choice of the cells, the triangle's normal, the
// products of their edges) separates the triangle from the grown cell.  The
// first pass counts (list null), the second, from the scanned counts, fills:
// one kernel, so that both take the same cells.
__global__ void __launch_bounds__(256) k_gr_refs(const float4 *tris, float to_raw, int nt, Geom g, uint32_t *cnt,
                                                 int32_t *list) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; t < nt; t += nw) {
    float4 v[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) v[k] = raw_vertex(tris[3 * t + k], to_raw);
    const float tlo[3] = {fminf(v[0].x, fminf(v[1].x, v[2].x)), fminf(v[0].y, fminf(v[1].y, v[2].y)),
                          fminf(v[0].z, fminf(v[1].z, v[2].z))};
    const float thi[3] = {fmaxf(v[0].x, fmaxf(v[1].x, v[2].x)), fmaxf(v[0].y, fmaxf(v[1].y, v[2].y)),
                          fmaxf(v[0].z, fmaxf(v[1].z, v[2].z))};
    int i0[3], m[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int b = (int)floorf((tlo[k] - g.lo[k]) * g.inv[k] - kGrowF);
      const int e = (int)floorf((thi[k] - g.lo[k]) * g.inv[k] + kGrowF);
      i0[k] = min(max(b, 0), g.n[k] - 1);
      m[k] = min(max(e, 0), g.n[k] - 1) - i0[k] + 1;
    }
    const double A[3] = {v[0].x, v[0].y, v[0].z};
    const double p[3] = {v[1].x - A[0], v[1].y - A[1], v[1].z - A[2]};
    const double q[3] = {v[2].x - A[0], v[2].y - A[1], v[2].z - A[2]};
    const double nrm[3] = {p[1] * q[2] - p[2] * q[1], p[2] * q[0] - p[0] * q[2], p[0] * q[1] - p[1] * q[0]};
    double reach = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) reach += fabs(nrm[k]) * g.h[k] * (0.5 + kGrow);
    reach *= 1.0 + 1e-9;
    const int64_t total = (int64_t)m[0] * m[1] * m[2];
    for (int64_t j = lane; j < total; j += 32) {
      const int x = i0[0] + (int)(j % m[0]), y = i0[1] + (int)(j / m[0] % m[1]), z = i0[2] + (int)(j / m[0] / m[1]);
      const double dist = nrm[0] * (g.lo[0] + (x + 0.5) * g.h[0] - A[0]) + nrm[1] * (g.lo[1] + (y + 0.5) * g.h[1] - A[1]) +
                          nrm[2] * (g.lo[2] + (z + 0.5) * g.h[2] - A[2]);
      if (fabs(dist) > reach) continue;
      const double ctr[3] = {g.lo[0] + (x + 0.5) * g.h[0], g.lo[1] + (y + 0.5) * g.h[1], g.lo[2] + (z + 0.5) * g.h[2]};
      float rel[3][3], half[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        rel[k][0] = (float)(v[k].x - ctr[0]);
        rel[k][1] = (float)(v[k].y - ctr[1]);
        rel[k][2] = (float)(v[k].z - ctr[2]);
        half[k] = (float)(g.h[k] * (0.5 + kGrow));
      }
      bool apart = false;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float edge[3] = {rel[(k + 1) % 3][0] - rel[k][0], rel[(k + 1) % 3][1] - rel[k][1],
                               rel[(k + 1) % 3][2] - rel[k][2]};
#pragma unroll
        for (int d = 0; d < 3; ++d) apart |= axis_separates(rel, edge, d, half);
      }
      if (apart) continue;
      const int64_t c = ((int64_t)z * g.n[1] + y) * g.n[0] + x;
      const uint32_t pos = atomicAdd(cnt + c, 1u);
      if (list) list[pos] = (int32_t)t;
    }
  }
}

// Words of every cell's block (to be scanned into offsets); the longest list,
// and the sums of the lists and of the blocks in 64 bits: the scans wrap where
// these do not fit 32, and such a grid must not be filled.
__global__ void __launch_bounds__(256) k_gr_sizes(const uint32_t *cnt, int64_t cells, uint32_t *size,
                                                  unsigned long long *longest) {
  uint32_t mx = 0;
  unsigned long long refs = 0, words = 0;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < cells; c += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t v = cnt[c];
    const uint32_t w = v ? 1u + kChunkWords * ((v + kSub - 1) / kSub) : 0u;
    size[c] = w;
    mx = max(mx, v);
    refs += v;
    words += w;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    refs += __shfl_xor_sync(0xffffffffu, refs, o);
    words += __shfl_xor_sync(0xffffffffu, words, o);
  }
  if ((threadIdx.x & 31) == 0 && mx) {
    atomicMax(longest, (unsigned long long)mx);
    atomicAdd(longest + 1, refs);
    atomicAdd(longest + 2, words);
  }
}

// Scatters the anchors: lowbias32 of C. Wellons' Hash Prospector.
__device__ __forceinline__ uint32_t hash32(uint32_t x) {
  x ^= x >> 16;
  x *= 0x7feb352du;
  x ^= x >> 15;
  x *= 0x846ca68bu;
  x ^= x >> 16;
  return x;
}

// Anchor of every cell: the one of four scattered points of the cell whose
// distance to the planes of the cell's triangles is largest.
// `last` holds the end of every cell's list.
__global__ void __launch_bounds__(256) k_gr_anchor(const float4 *tris, float to_raw, Geom g, int64_t cells,
                                                   const uint32_t *last, const int32_t *list, float *anchor) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c < cells; c += nw) {
    const uint32_t b = c ? last[c - 1] : 0u, e = last[c];
    const int x = (int)(c % g.n[0]), y = (int)(c / g.n[0] % g.n[1]), z = (int)(c / g.n[0] / g.n[1]);
    float best[3] = {0.f, 0.f, 0.f}, best_d = -1.f;
    for (int k = 0; k < (b == e ? 1 : 4); ++k) {
      float q[3];
      uint32_t r = hash32((uint32_t)c * 4u + (uint32_t)k);
      const int xyz[3] = {x, y, z};
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        q[d] = (float)(g.lo[d] + g.h[d] * (xyz[d] + 0.25 + 0.5 * (double)((r >> 8) + 0.5) / 16777216.0));
        r = hash32(r + 0x9e3779b9u);
      }
      float dmin = INFINITY;
      for (uint32_t j = b + lane; j < e; j += 32) {
        const int64_t t = list[j];
        const float4 A = raw_vertex(tris[3 * t], to_raw), B = raw_vertex(tris[3 * t + 1], to_raw),
                     C = raw_vertex(tris[3 * t + 2], to_raw);
        const float ux = B.x - A.x, uy = B.y - A.y, uz = B.z - A.z, wx = C.x - A.x, wy = C.y - A.y, wz = C.z - A.z;
        const float nx = uy * wz - uz * wy, ny = uz * wx - ux * wz, nz = ux * wy - uy * wx;
        const float len = sqrtf(nx * nx + ny * ny + nz * nz);
        if (len > 0.f) dmin = fminf(dmin, fabsf(nx * (q[0] - A.x) + ny * (q[1] - A.y) + nz * (q[2] - A.z)) / len);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) dmin = fminf(dmin, __shfl_xor_sync(0xffffffffu, dmin, o));
      if (dmin > best_d) {
        best_d = dmin;
#pragma unroll
        for (int d = 0; d < 3; ++d) best[d] = q[d];
      }
    }
    if (lane < 3) anchor[3 * c + lane] = lane == 0 ? best[0] : lane == 1 ? best[1] : best[2];
  }
}

// Words and blocks of the cells, from the anchors' solid angles.  Vertices
// relative to the anchor are exact in FP64 up to its rounding; s (a power of
// two) brings them to about [-64, 64]; the stored cross products carry one
// factor s more, for the unscaled d = p - q of the kernel.
__global__ void __launch_bounds__(256) k_gr_finish(const float4 *tris, float to_raw, double s, Geom g, int64_t cells,
                                                   const uint32_t *last, const uint32_t *off, const int32_t *list,
                                                   const float *anchor, const float *omega, uint32_t *words,
                                                   float4 *blocks) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; c < cells; c += nw) {
    const uint32_t b = c ? last[c - 1] : 0u, e = last[c];
    const float om = omega[c];
    const float kf = rintf(om / kFourPi);
    const bool known = fabsf(om - kFourPi * kf) < 1e-3f && fabsf(kf) <= 100.f;
    if (b == e) {
      if (lane == 0) words[c] = known ? ((uint32_t)(int)kf & 0xffu) : kUnknown;
      continue;
    }
    const float qx = anchor[3 * c], qy = anchor[3 * c + 1], qz = anchor[3 * c + 2];
    const uint32_t chunks = (e - b + kSub - 1) / kSub;
    float4 *block = blocks + off[c];
    if (lane == 0) {
      words[c] = kMixed | (chunks <= 3 ? chunks << kChunkShift : 0u) | off[c];
      block[0] = make_float4(qx, qy, qz, __uint_as_float(((e - b) << 8) | ((uint32_t)(known ? (int)kf : kNoK) & 0xffu)));
    }
    for (uint32_t j = b + lane; j < b + chunks * kSub; j += 32) {
      float4 *o = block + 1 + (j - b) / kSub * kChunkWords + (j - b) % kSub;
      if (j >= e) {  // V > E > 0 and W = -V < -kPlane E: the segment ends before the plane
        o[0] = make_float4(0.f, 0.f, 0.f, 1.f);
        o[kSub] = make_float4(0.f, 0.f, 0.f, 0.01f);
        o[2 * kSub] = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
        continue;
      }
      const int64_t t = list[j];
      double v[3][3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float4 p = raw_vertex(tris[3 * t + k], to_raw);
        v[k][0] = ((double)p.x - qx) * s;
        v[k][1] = ((double)p.y - qy) * s;
        v[k][2] = ((double)p.z - qz) * s;
      }
      double N[3][3], M = 0.0, P = 0.0;  // products, their reach over the cell, their terms without cancellation
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double *a = v[k], *w = v[(k + 1) % 3];
        double mk = 0.0, pk = 0.0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const int d1 = (d + 1) % 3, d2 = (d + 2) % 3;
          const double x = a[d1] * w[d2], y = a[d2] * w[d1], hd = g.h[d] * s * (1.0 + 2 * kGrow);
          N[k][d] = x - y;
          mk += hd * fabs(N[k][d]);
          pk += (hd + fabs(v[(k + 2) % 3][d])) * (fabs(x) + fabs(y));
        }
        M = fmax(M, mk);
        P = fmax(P, pk);
      }
      const double V = v[0][0] * N[1][0] + v[0][1] * N[1][1] + v[0][2] * N[1][2];
      // |error| of an FP32 dot product d . N: rounding of d, of N, of three
      // products and two sums (5 2^-24 of the sum of the |terms|, which is at
      // most M), plus the FP64 error of N and V
      const double E = 6.2 * 5.9604644775390625e-08 * M + 3.6e-15 * P + 1e-36;
      o[0] = make_float4((float)(N[0][0] * s), (float)(N[0][1] * s), (float)(N[0][2] * s), (float)V);
      o[kSub] = make_float4((float)(N[1][0] * s), (float)(N[1][1] * s), (float)(N[1][2] * s), __double2float_ru(E));
      o[2 * kSub] = make_float4((float)(N[2][0] * s), (float)(N[2][1] * s), (float)(N[2][2] * s), __int_as_float((int)t));
    }
  }
}

// ------------------------------------------------------------------ labeling
struct GridArgs {
  const float *pts;
  int32_t *labels;
  float *omega;               // nullable, [ncomp][omega_ld]
  int64_t omega_ld;
  unsigned long long *masks;  // nullable, caller's order
  const GridComp *grid;       // by priority row
  const int32_t *row_ids;
  int64_t *counters;
#ifdef ZEF_DEBUG_BOUNDS
  int64_t n_nodes, n_cseg;    // cap-tree nodes and segment entries
  int64_t pend_cap;           // entries of `pending`
#endif
  int64_t n_host;             // points, or -1: counters[CNT_N] from counters[CNT_OFF] on
  int ncomp;
  int early;                  // a point certainly inside needs no later compartment
  int stats;
  int iters;                  // streaming kernel: consecutive tiles of a warp
  int tile;                   // fused kernel: points of a warp's step
  int32_t *pending;           // streaming kernel: indices of the points the field leaves open
  OpenPoint *open;            // points for the FP64 solid angles
  UnionBox ub;
  LabelField field;
  uint32_t *status;
  const DevComp *comps;       // FP64 solid angles: cap trees (scaled coordinates)
  const CapNode *nodes;
  const Entry *cseg;
  float scale;
};

__device__ __forceinline__ void count_add(const GridArgs &a, int c, unsigned long long v) {
  atomicAdd((unsigned long long *)(a.counters + c), v);
}

// statistics of the labeling kernel, summed per warp and block before they
// reach the counters (thousands of warps adding to one word would queue)
enum GridStat { GS_EVAL = 0, GS_COHERENT, GS_OWN, GS_NONFINITE, GS_NIN, GS_COUNT };

// FP64 re-evaluation of one (point, compartment) pair by the whole warp: the
// crossings from the vertices in FP64, each sign taken only beyond its
// rounding bound.  Returns whether that decides the pair; *k = the point's
// winding number.
__device__ __noinline__ bool crossings64(const GridArgs &a, const GridComp &g, uint32_t word, float x, float y, float z,
                                         int lane, int *k) {
  if (word & kMixed) {
    const float4 *block = g.blocks + (word & kOffsetMask);
    const float4 r = block[0];
    const int k0 = (int)(signed char)(__float_as_uint(r.w) & 0xffu), count = (int)(__float_as_uint(r.w) >> 8);
    int net = 0, tested = 0;
    bool open = k0 == kNoK;
    if (!open) {
      const double dx = (double)x - r.x, dy = (double)y - r.y, dz = (double)z - r.z;
      for (int j = lane; j < count; j += 32) {
        const int64_t t = __float_as_int(block[1 + j / kSub * kChunkWords + 2 * kSub + j % kSub].w);
        if (!ZEF_BOUNDS_OK(t >= 0 && t < a.comps[g.comp].tri_cnt, a.status, 34)) continue;
        ++tested;
        double v[3][3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float4 p = raw_vertex(g.tris[3 * t + k], g.tri_raw);
          v[k][0] = (double)p.x - r.x;
          v[k][1] = (double)p.y - r.y;
          v[k][2] = (double)p.z - r.z;
        }
        double e[3], E = 0.0, V = 0.0, EV = 0.0;
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const double *p = v[k], *w = v[(k + 1) % 3], *u = v[(k + 2) % 3];
          const double t0 = p[1] * w[2], t1 = p[2] * w[1], t2 = p[2] * w[0], t3 = p[0] * w[2], t4 = p[0] * w[1],
                       t5 = p[1] * w[0];
          e[k] = dx * (t0 - t1) + dy * (t2 - t3) + dz * (t4 - t5);
          E = fmax(E, fabs(dx) * (fabs(t0) + fabs(t1)) + fabs(dy) * (fabs(t2) + fabs(t3)) +
                          fabs(dz) * (fabs(t4) + fabs(t5)));
          if (k == 0) {
            V = u[0] * (t0 - t1) + u[1] * (t2 - t3) + u[2] * (t4 - t5);
            EV = fabs(u[0]) * (fabs(t0) + fabs(t1)) + fabs(u[1]) * (fabs(t2) + fabs(t3)) +
                 fabs(u[2]) * (fabs(t4) + fabs(t5));
          }
        }
        // rounding of d, p, w (2^-53 each), products and sums: below 12 2^-53
        // of the terms' sum
        E *= 1.8e-15;
        EV *= 1.8e-15;
        const double S = e[0] + e[1] + e[2], W = S - V, EW = 4.0 * E + EV + 4.5e-16 * (fabs(S) + fabs(V));
        const double mn = fmin(e[0], fmin(e[1], e[2])), mx = fmax(e[0], fmax(e[1], e[2]));
        const bool out = V > EV && W > EW && mn > E, in = V < -EV && W < -EW && mx < -E;
        const bool none = (mn < -E && mx > E) || (V < -EV && W > EW) || (V > EV && W < -EW);
        net += in ? 1 : out ? -1 : 0;
        open |= !(in || out || none);
      }
    }
    if (!__any_sync(0xffffffffu, open)) {
      net = __reduce_add_sync(0xffffffffu, net);
      tested = __reduce_add_sync(0xffffffffu, tested);
      if (lane == 0 && a.stats) {
        count_add(a, CNT_UNC, 1);
        count_add(a, CNT_PAIRS_RESCUE, (unsigned long long)tested);
      }
      *k = k0 + net;
      return true;
    }
  }
  return false;
}

// FP64 solid angle of one pair by the whole warp, over the cap tree: what the
// crossings leave open (a point on the surface).
__device__ __noinline__ double solid64(const GridArgs &a, const GridComp &g, float x, float y, float z, int lane) {
  // FP64 solid angle: the caps of the nodes whose box misses the point, the
  // leaves whose box holds it
  const DevComp *cp = a.comps + g.comp;
  const float px = x * a.scale, py = y * a.scale, pz = z * a.scale;
  // The groups of four entries in the order of k_grid_open's block of 256
  // threads (thread g mod 256 takes group g; the sums of each 32 threads, then
  // of the eight in turn), so that a point on the surface, whose Omega is 2 pi
  // up to rounding, gets that kernel's rounding.  The walk's segments are a
  // few groups each: every lane holds one, and each time they hold 32 groups
  // together the lanes take one each (segment by segment a pair took 0.4 ms).
  double part[8];
#pragma unroll
  for (int w = 0; w < 8; ++w) part[w] = 0.0;
  int K = 0, tris = 0;
  int seg_b = 0, seg_n = 0;           // this lane's segment: first entry, groups left
  int segs = 0, held = 0, round = 0;  // segments and groups held, batches taken
  auto take = [&]() {                 // the first 32 groups held (fewer at the end)
    int end = seg_n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += t;
    }
    const int first = end - seg_n;
    int pos = -1;
    for (int q = 0; q < segs; ++q) {
      const int f = __shfl_sync(0xffffffffu, first, q), e = __shfl_sync(0xffffffffu, end, q),
                b = __shfl_sync(0xffffffffu, seg_b, q);
      if (lane >= f && lane < e) pos = b + 4 * (lane - f);
    }
    if (pos >= 0 && ZEF_BOUNDS_OK((int64_t)pos + 4 <= a.n_cseg, a.status, 36)) {
      const double h = group64(a.cseg, pos, px, py, pz, &K);
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q == (round & 7)) part[q] += h;
    }
    ++round;
    const int used = min(max(32 - first, 0), seg_n);
    seg_b += 4 * used;
    seg_n -= used;
    held = max(held - 32, 0);
    // the empty segments are the first ones
    const int gone = __popc(__ballot_sync(0xffffffffu, lane < segs && seg_n == 0));
    const int nb = __shfl_sync(0xffffffffu, seg_b, (lane + gone) & 31), nn = __shfl_sync(0xffffffffu, seg_n, (lane + gone) & 31);
    segs -= gone;
    seg_b = nb;
    seg_n = lane < segs ? nn : 0;
  };
  const int root = cp->cap_root, end = a.nodes[root].skip;
  for (int i = root; i != end;) {
    if (!ZEF_BOUNDS_OK(i >= 0 && i < a.n_nodes, a.status, 35)) break;
    const CapNode nd = a.nodes[i];
    const bool far = nd.hi[0] < px || nd.lo[0] > px || nd.hi[1] < py || nd.lo[1] > py || nd.hi[2] < pz || nd.lo[2] > pz;
    int b = nd.cap_begin, c = nd.cap_cnt;
    if (!far) {
      if (nd.left >= 0) {
        ++i;
        continue;
      }
      b = nd.leaf_begin;
      c = nd.leaf_cnt;
    }
    tris += far ? nd.cap_tris : nd.leaf_tris;
    i = nd.skip;
    if (c < 4) continue;
    if (lane == segs) {  // at most 31 are held here: a segment has at least one group
      seg_b = b;
      seg_n = c / 4;
    }
    ++segs;
    held += c / 4;
    while (held >= 32) take();
  }
  if (held > 0) take();
  double sum = 0.0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part[q] += __shfl_xor_sync(0xffffffffu, part[q], o);
    sum += part[q];
  }
  K = __reduce_add_sync(0xffffffffu, K);
  const double om = 2.0 * (sum + kTwoPi64 * (double)K);
  if (lane == 0 && a.stats) {
    count_add(a, CNT_UNC, 1);
    count_add(a, CNT_PAIRS_RESCUE, (unsigned long long)tris);
  }
  return om;
}

// Index of x on an axis of n cells; monotone in x, so the indices of a box's
// ends bound those of its points.
__device__ __forceinline__ int axis_cell(float x, float lo, float inv, int n) {
  return min(max((int)((x - lo) * inv), 0), n - 1);
}

// Word of the cell that holds a point of the surface's box.
__device__ __forceinline__ uint32_t cell_word(const GridArgs &a, const GridComp &g, float x, float y, float z) {
  const int cx = axis_cell(x, g.lo[0], g.inv[0], g.n[0]), cy = axis_cell(y, g.lo[1], g.inv[1], g.n[1]),
            cz = axis_cell(z, g.lo[2], g.inv[2], g.n[2]);
  const int c = (cz * g.n[1] + cy) * g.n[0] + cx;  // at most kMaxCells
  if (!ZEF_BOUNDS_OK(c >= 0 && c < g.n[0] * g.n[1] * g.n[2], a.status, 30)) return 0u;
  const uint32_t w = __ldg(g.words + c);
  // the words lie behind the blocks; a block is a header and a chunk at least
  if ((w & kMixed) && !ZEF_BOUNDS_OK((w & kOffsetMask) + 1u + kChunkWords * max(1u, (w & ~kMixed) >> kChunkShift) <=
                                         (uint64_t)(reinterpret_cast<const float4 *>(g.words) - g.blocks), a.status, 32))
    return 0u;
  return w;
}

// Both by the whole warp: whether the point is inside; *omega = Omega.
__device__ __noinline__ bool resolve64(const GridArgs &a, const GridComp &g, uint32_t word, float x, float y, float z,
                                       int lane, float *omega) {
  int k = 0;
  if (crossings64(a, g, word, x, y, z, lane, &k)) {
    *omega = kFourPi * (float)k;
    return k >= 1;
  }
  const double om = solid64(a, g, x, y, z, lane);
  *omega = (float)om;
  return om > kTwoPi64;
}

// The FP64 solid angle of one pair by a block of 256 threads.  The walk of the
// cap tree goes down one level at a time: the list holds, in the tree's order,
// the segments found so far and the nodes still to be opened, and each node is
// replaced by its segment or its two children: a level is one read of every
// thread's node and a scan, and eight warps share the FP64 pipe that bounds the
// sum.  A vertex of a 20,000-triangle surface: 50 us, 115 by one warp.  Every
// thread returns the same Omega; `lane` and `wid` are the thread's.
constexpr int kOpenThreads = 256;
constexpr int kOpenList = 1024;  // entries of a level; beyond that one warp walks as solid64 does

struct OpenShared {
  int2 seg[2][kOpenList];  // x: first entry, y: its groups of four, or x: node, y: 0
  int first[kOpenList];    // groups before the segment
  int scan[2][kOpenThreads / 32];
  double part[kOpenThreads / 32];
  int wraps[kOpenThreads / 32];
  int decided, k;
  double om;
};

// exclusive sum of v over the block in thread order; *total its sum
__device__ __forceinline__ int block_exclusive(int v, int (&s_scan)[kOpenThreads / 32], int lane, int wid, int *total) {
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  __syncthreads();  // the last sum's readers are done
  if (lane == 31) s_scan[wid] = incl;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kOpenThreads / 32; ++w) {
    before += w < wid ? s_scan[w] : 0;
    all += s_scan[w];
  }
  *total = all;
  return before + incl - v;
}

__device__ double solid64_block(const GridArgs &a, const GridComp &g, float x, float y, float z, OpenShared &sh, int lane,
                                int wid) {
  const DevComp *cp = a.comps + g.comp;
  const float px = x * a.scale, py = y * a.scale, pz = z * a.scale;
  int cur = 0, len = 1, tris = 0;
  if (threadIdx.x == 0) sh.seg[0][0] = make_int2(cp->cap_root, 0);
  __syncthreads();
  for (;;) {
    int out = 0;
    bool nodes = false;
    for (int e0 = 0; e0 < len; e0 += kOpenThreads) {
      const int e = e0 + (int)threadIdx.x;
      int n = 0;
      int2 o0 = make_int2(0, 0), o1 = make_int2(0, 0);
      if (e < len) {
        o0 = sh.seg[cur][e];
        n = 1;
        if (o0.y == 0 && !ZEF_BOUNDS_OK(o0.x >= 0 && o0.x < a.n_nodes, a.status, 37)) {
          n = 0;
        } else if (o0.y == 0) {
          const CapNode nd = a.nodes[o0.x];
          const bool far = nd.hi[0] < px || nd.lo[0] > px || nd.hi[1] < py || nd.lo[1] > py || nd.hi[2] < pz || nd.lo[2] > pz;
          if (!far && nd.left >= 0) {
            o1 = make_int2(nd.right, 0);
            o0 = make_int2(o0.x + 1, 0);
            n = 2;
            nodes = true;
          } else {
            const int c = far ? nd.cap_cnt : nd.leaf_cnt;
            tris += far ? nd.cap_tris : nd.leaf_tris;
            o0 = make_int2(far ? nd.cap_begin : nd.leaf_begin, c / 4);
            n = c >= 4 ? 1 : 0;
          }
        }
      }
      int total;
      const int at = out + block_exclusive(n, sh.scan[0], lane, wid, &total);
      if (n > 0 && at < kOpenList) sh.seg[cur ^ 1][at] = o0;
      if (n > 1 && at + 1 < kOpenList) sh.seg[cur ^ 1][at + 1] = o1;
      out += total;
    }
    len = out;
    cur ^= 1;
    const bool more = __syncthreads_or(nodes);
    if (len > kOpenList || !more) break;
  }
  if (len > kOpenList) {
    if (wid == 0) {
      const double om = solid64(a, g, x, y, z, lane);
      if (lane == 0) sh.om = om;
    }
    __syncthreads();
    const double om = sh.om;
    __syncthreads();
    return om;
  }
  int groups = 0;
  for (int e0 = 0; e0 < len; e0 += kOpenThreads) {
    const int e = e0 + (int)threadIdx.x;
    int total;
    const int at = groups + block_exclusive(e < len ? sh.seg[cur][e].y : 0, sh.scan[1], lane, wid, &total);
    if (e < len) sh.first[e] = at;
    groups += total;
  }
  __syncthreads();
  double part = 0.0;
  int K = 0;
  for (int j = (int)threadIdx.x; j < groups; j += kOpenThreads) {
    int lo = 0, hi = len - 1;  // the last segment that starts at or before group j
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (sh.first[mid] <= j) lo = mid;
      else hi = mid - 1;
    }
    const int pos = sh.seg[cur][lo].x + 4 * (j - sh.first[lo]);
    if (ZEF_BOUNDS_OK(pos >= 0 && (int64_t)pos + 4 <= a.n_cseg, a.status, 38)) part += group64(a.cseg, pos, px, py, pz, &K);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  K = __reduce_add_sync(0xffffffffu, K);
  tris = __reduce_add_sync(0xffffffffu, tris);
  if (lane == 0) {
    sh.part[wid] = part;
    sh.wraps[wid] = K;
    if (a.stats && tris) count_add(a, CNT_PAIRS_RESCUE, (unsigned long long)tris);
  }
  if (threadIdx.x == 0 && a.stats) count_add(a, CNT_UNC, 1);
  __syncthreads();
  double sum = 0.0;
  K = 0;
#pragma unroll
  for (int w = 0; w < kOpenThreads / 32; ++w) {
    sum += sh.part[w];
    K += sh.wraps[w];
  }
  __syncthreads();
  return 2.0 * (sum + kTwoPi64 * (double)K);
}

// ---- the label field: one cell grid over the union box of all surfaces.  A
// cell holds, per priority row, whether its points have winding number 1
// (`ins`) or need the compartment's own grid (`mix`: its cells there are not
// all empty of triangles with one winding number of 0 or 1); neither bit: 0.
template <bool WIDE>
struct FieldCell;
template <>
struct FieldCell<false> {
  using T = uint2;
  using M = uint32_t;
};
template <>
struct FieldCell<true> {
  using T = ulonglong2;
  using M = unsigned long long;
};

// A field cell's cells in one surface's grid that its thread looks at alone.
// One thread for all of them took 17 ms for a surface of 450,000 triangles in
// one fifty times as wide (50,000 cells in one of the field's), now 4.
constexpr int kFieldAlone = 64;

template <bool WIDE>
__global__ void __launch_bounds__(256) k_gr_field(LabelField f, const GridComp *grid, int ncomp) {
  using M = typename FieldCell<WIDE>::M;
  __shared__ GridComp s_g[ZEF_MAX_COMPARTMENTS];
  for (int j = threadIdx.x; j < ncomp * (int)(sizeof(GridComp) / 16); j += blockDim.x)
    reinterpret_cast<uint4 *>(s_g)[j] = reinterpret_cast<const uint4 *>(grid)[j];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t cells = (int64_t)f.n[0] * f.n[1] * f.n[2];
  for (int64_t c0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31); c0 < cells; c0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = min(c0 + lane, cells - 1);  // the last warp's spare lanes repeat the last cell
    const int xyz[3] = {(int)(c % f.n[0]), (int)(c / f.n[0] % f.n[1]), (int)(c / f.n[0] / f.n[1])};
    float lo[3], hi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {  // the cell grown by kGrow: it holds every point that k_grid_label puts in it
      lo[k] = __double2float_rd(f.lo[k] + (xyz[k] - kGrow) * f.h[k]);
      hi[k] = __double2float_ru(f.lo[k] + (xyz[k] + 1 + kGrow) * f.h[k]);
    }
    M ins = 0, mix = 0;
    for (int r = 0; r < ncomp; ++r) {
      const GridComp &g = s_g[r];
      bool out = false, part = false;  // the cell misses the surface's box / reaches out of it
      int i0[3], d[3], total = 1;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        out |= hi[k] < g.lo[k] || lo[k] > g.hi[k];
        part |= lo[k] < g.lo[k] || hi[k] > g.hi[k];
        i0[k] = axis_cell(fmaxf(lo[k], g.lo[k]), g.lo[k], g.inv[k], g.n[k]);
        d[k] = axis_cell(fminf(hi[k], g.hi[k]), g.lo[k], g.inv[k], g.n[k]) - i0[k] + 1;
        total *= d[k];  // at most kMaxCells
      }
      if (out) total = 0;
      auto word = [&](int j) {
        return g.words[((int64_t)(i0[2] + j / (d[0] * d[1])) * g.n[1] + i0[1] + j / d[0] % d[1]) * g.n[0] + i0[0] + j % d[0]];
      };
      uint32_t w = part ? 0u : 0xffffffffu;  // the winding number so far (none yet: all ones)
      bool same = true;
      const int alone = min(total, kFieldAlone);
      for (int j = 0; j < alone && same; ++j) {
        const uint32_t v = word(j);
        if (v > 1u) same = false;  // triangles, unknown, or a winding number other than 0 and 1
        else if (w == 0xffffffffu) w = v;
        else if (w != v) same = false;
      }
      // the rest of a cell that holds more (of a surface with cells much finer
      // than the field's), the warp together
      for (uint32_t left = __ballot_sync(0xffffffffu, same && total > kFieldAlone); left; left &= left - 1) {
        const int src = __ffs(left) - 1;
        const int x0 = __shfl_sync(0xffffffffu, i0[0], src), y0 = __shfl_sync(0xffffffffu, i0[1], src),
                  z0 = __shfl_sync(0xffffffffu, i0[2], src), dx = __shfl_sync(0xffffffffu, d[0], src),
                  dy = __shfl_sync(0xffffffffu, d[1], src), all = __shfl_sync(0xffffffffu, total, src);
        const uint32_t want = __shfl_sync(0xffffffffu, w, src);
        bool other = false;
        for (int j0 = kFieldAlone; j0 < all; j0 += 32 * 8) {
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const int j = j0 + 32 * u + lane;
            if (j < all)
              other |= g.words[((int64_t)(z0 + j / (dx * dy)) * g.n[1] + y0 + j / dx % dy) * g.n[0] + x0 + j % dx] != want;
          }
          if (__any_sync(0xffffffffu, other)) break;
        }
        other = __any_sync(0xffffffffu, other);
        if (lane == src) same = !other;
      }
      if (total == 0) continue;
      if (!same) mix |= (M)1 << r;
      else if (w == 1u) ins |= (M)1 << r;
    }
    if (c0 + lane >= cells) continue;
    typename FieldCell<WIDE>::T o;
    o.x = ins;
    o.y = mix;
    reinterpret_cast<typename FieldCell<WIDE>::T *>(f.cells)[c] = o;
  }
}

constexpr int kGlThreads = 256;
constexpr int kGlWarps = kGlThreads / 32;
constexpr int kGlP = 2;               // fused kernel: points per lane and step
constexpr int kGlTile = 32 * kGlP;
constexpr int kGlQueue = 32 + kGlTile;  // fewer than 32 left over, one tile's more
constexpr int kRun = 8;               // consecutive points of a warp (see run_point)
constexpr int kGsP = 4;               // streaming kernel
constexpr int kGsTile = 32 * kGsP;
constexpr int kGsFlush = 256;         // listed together (each addition to the one cursor costs about a nanosecond)
constexpr int kGsQueue = kGsFlush + kGsTile;
constexpr int kGlMaxIters = 32;       // consecutive tiles of a warp
constexpr int kLanes = 4;             // lanes per point of the crossing tests

__device__ __forceinline__ int first_row(uint32_t m) { return __ffs((int)m) - 1; }
__device__ __forceinline__ int first_row(unsigned long long m) { return __ffsll((long long)m) - 1; }
// rows that can still matter: with the priority early exit those before the
// first row the point is known to be inside of
template <class M>
__device__ __forceinline__ M open_rows(M ins, M mix, int early) {
  return early ? mix & ((ins & (M)(0 - ins)) - 1) : mix;
}

// A point whose label the field leaves open.
template <bool WIDE>
struct __align__(16) Pending {
  float x, y, z;
  int32_t i;
  typename FieldCell<WIDE>::M ins, mix;
};

// Shared memory of the batches of one block.
struct Batch {
  float4 p[kGlWarps][32];             // x, y, z, word of the batch's points in cells with triangles
  const float4 *blocks[kGlWarps][32];  // their compartments' blocks
};

// Decides a batch of up to 32 points (one per lane, `have`): every lane looks
// its point's cell up in the grid of the first row the point still needs;
// points in cells with triangles are then taken eight at a time, four lanes
// each over the entries of the point's own cell (two dependent reads per
// point -- word, block -- whatever cells and compartments the batch lies in).
// Pairs that the crossings leave open are taken to FP64 by the warp, one after
// the other; with LIST, a point whose label needs one is listed for k_grid_open
// instead, and one that the list does not hold is left to its second part.
template <bool WIDE, bool LIST>
__device__ __forceinline__ void decide(const GridArgs &a, const GridComp *s_g, const int32_t *s_id, Batch &sb, int wid,
                                       int lane, int64_t off, float x, float y, float z, int32_t i, bool have,
                                       typename FieldCell<WIDE>::M mask, typename FieldCell<WIDE>::M mix,
                                       uint32_t &st_eval, uint32_t &st_own) {
  using M = typename FieldCell<WIDE>::M;
  const int sub = lane / kLanes, ti = lane % kLanes;
  M pend = have ? open_rows<M>(mask, mix, a.early) : 0;
  M left = 0;  // LIST: rows left open
  while (__any_sync(0xffffffffu, pend != 0)) {
    const bool mine = pend != 0;
    const int r = mine ? first_row(pend) : 0;
    pend &= pend - 1;
    const GridComp &g = s_g[r];
    const bool in = mine && x >= g.lo[0] && x <= g.hi[0] && y >= g.lo[1] && y <= g.hi[1] && z >= g.lo[2] && z <= g.hi[2];
    const uint32_t word = in ? cell_word(a, g, x, y, z) : 0u;
    const bool mixed = (word & kMixed) != 0u;
    bool unc = (word & (kMixed | kUnknown)) == kUnknown;
    int k = (int)(signed char)(word & 0xffu);
    const uint32_t m = __ballot_sync(0xffffffffu, mixed);
    if (m) {
      const int np = __popc(m), rank = __popc(m & ((1u << lane) - 1u));
      if (mixed) {
        sb.p[wid][rank] = make_float4(x, y, z, __uint_as_float(word));
        sb.blocks[wid][rank] = g.blocks;
      }
      __syncwarp();
      for (int j0 = 0; j0 < np; j0 += 32 / kLanes) {
        const int j = min(j0 + sub, np - 1);  // a step short of points repeats the last one
        const float4 q = sb.p[wid][j];
        const uint32_t w = __float_as_uint(q.w);
        const float4 *block = sb.blocks[wid][j] + (w & kOffsetMask);
        const float4 h = __ldg(block);
        const float4 *t = block + 1 + ti;
        int chunks = (int)((w & ~kMixed) >> kChunkShift);
        if (!chunks) chunks = (int)(((__float_as_uint(h.w) >> 8) + kSub - 1) / kSub);
        if (!ZEF_BOUNDS_OK(chunks <= kMaxList / kSub, a.status, 33)) chunks = 0;
        const int k0 = (int)(signed char)(__float_as_uint(h.w) & 0xffu);
        const float dx = q.x - h.x, dy = q.y - h.y, dz = q.z - h.z;
        bool open = k0 == kNoK;
        int net = 0;
        for (int b = 0; b < chunks; ++b, t += kChunkWords) {
          float4 e[kSub / kLanes][3];
#pragma unroll
          for (int u = 0; u < kSub / kLanes; ++u)
#pragma unroll
            for (int d = 0; d < 3; ++d) e[u][d] = __ldg(t + u * kLanes + d * kSub);
#pragma unroll
          for (int u = 0; u < kSub / kLanes; ++u) {
            const float4 n0 = e[u][0], n1 = e[u][1], n2 = e[u][2];
            const float v0 = fmaf(n0.x, dx, fmaf(n0.y, dy, n0.z * dz));
            const float v1 = fmaf(n1.x, dx, fmaf(n1.y, dy, n1.z * dz));
            const float v2 = fmaf(n2.x, dx, fmaf(n2.y, dy, n2.z * dz));
            const float V = n0.w, E = n1.w, EW = kPlane * n1.w, W = (v0 + v1 + v2) - V;
            const float mn = fminf(v0, fminf(v1, v2)), mx = fmaxf(v0, fmaxf(v1, v2));
            const bool vp = V > E, vn = V < -E, wp = W > EW, wn = W < -EW;
            const bool cross_out = vp && wp && mn > E, cross_in = vn && wn && mx < -E;
            const bool none = (mn < -E && mx > E) || (vn && wp) || (vp && wn);
            net += cross_in ? 1 : cross_out ? -1 : 0;
            open |= !(none || cross_out || cross_in);
          }
        }
        // over the point's lanes, then back to the lane that owns the point
#pragma unroll
        for (int o = kLanes / 2; o > 0; o >>= 1) net += __shfl_xor_sync(0xffffffffu, net, o);
        const uint32_t bu = __ballot_sync(0xffffffffu, open);
        const int kn = __shfl_sync(0xffffffffu, k0 + net, (rank - j0) * kLanes & 31);
        if (mixed && rank >= j0 && rank < j0 + 32 / kLanes) {
          k = kn;
          unc = ((bu >> ((rank - j0) * kLanes)) & ((1u << kLanes) - 1u)) != 0u;
        }
        if (a.stats && j0 + sub < np && ti == 0) st_eval += __float_as_uint(h.w) >> 8;
      }
      __syncwarp();
      ++st_own;
    }
    float om = kFourPi * (float)k;
    bool inside = in && !unc && k >= 1;
    if (LIST) {
      if (unc) left |= (M)1 << r;
    } else {
      uint32_t um = __ballot_sync(0xffffffffu, unc);
      while (um) {
        const int src = __ffs(um) - 1;
        um &= um - 1;
        float o64;
        const bool i64 = resolve64(a, s_g[__shfl_sync(0xffffffffu, r, src)], __shfl_sync(0xffffffffu, word, src),
                                   __shfl_sync(0xffffffffu, x, src), __shfl_sync(0xffffffffu, y, src),
                                   __shfl_sync(0xffffffffu, z, src), lane, &o64);
        if (lane == src) {
          inside = i64;
          om = o64;
        }
      }
    }
    if (inside) {
      mask |= (M)1 << r;
      if (a.early) pend = 0;
    }
    if (a.omega && mine) a.omega[(int64_t)r * a.omega_ld + i] = in ? om : 0.f;
  }
  if (LIST) {
    left = open_rows<M>(mask, left, a.early);
    const uint32_t lm = __ballot_sync(0xffffffffu, left != 0);
    if (lm) {
      const int first = __ffs(lm) - 1;
      unsigned long long at = 0;
      if (lane == first) at = atomicAdd((unsigned long long *)(a.counters + CNT_OPEN), (unsigned long long)__popc(lm));
      at = __shfl_sync(0xffffffffu, at, first) + __popc(lm & ((1u << lane) - 1u));
      if (left && at < (unsigned long long)kOpenCap) {
        OpenPoint p;
        p.ins = mask;
        p.open = left;
        p.x = x;
        p.y = y;
        p.z = z;
        p.i = i;
        a.open[at] = p;
      }
      if (left) have = false;
    }
  }
  if (have) {
    a.labels[off + i] = mask ? s_id[first_row(mask)] : 0;
    if (a.masks) a.masks[off + i] = mask;
  }
}

// Index of a warp's k-th point of tile t of `tiles`: runs of kRun consecutive
// points, the runs of a tile `tiles` runs apart.  Points that the crossings
// leave open -- points on a surface: electrodes are vertices of the scalp mesh,
// mesh nodes may lie in a face -- cost an FP64 solid angle each, one after the
// other in a warp, and come one behind the other: 64 vertices in 64 consecutive
// points took 6.9 ms in one warp, 0.9 ms in eight (the general kernels: 4.1).
// A run is three whole sectors of coordinates and one of labels.  (The pending
// kernel keeps 32 neighbours together, whose cells share L1 lines -- 5.2 M
// points 92 us in runs, 85 so -- and lists what stays open.)
__device__ __forceinline__ int64_t run_point(int64_t t, int64_t tiles, int k) {
  return kRun * ((k / kRun) * tiles + t) + k % kRun;
}
__device__ __forceinline__ int64_t run_tiles(int64_t n, int tile) {
  return ((n + kRun - 1) / kRun + tile / kRun - 1) / (tile / kRun);
}

// Field cell of a point: zero outside the union box and for a non-finite
// point (whose comparisons fail).
template <bool WIDE>
__device__ __forceinline__ typename FieldCell<WIDE>::T field_cell(const GridArgs &a, float x, float y, float z,
                                                                  bool *in_box) {
  typename FieldCell<WIDE>::T c;
  c.x = 0;
  c.y = 0;
  *in_box = x >= a.ub.lo[0] && x <= a.ub.hi[0] && y >= a.ub.lo[1] && y <= a.ub.hi[1] && z >= a.ub.lo[2] && z <= a.ub.hi[2];
  if (*in_box) {
    // x >= lo: no cell below the first
    const int cx = min((int)((x - a.field.lo[0]) * a.field.inv[0]), a.field.n[0] - 1),
              cy = min((int)((y - a.field.lo[1]) * a.field.inv[1]), a.field.n[1] - 1),
              cz = min((int)((z - a.field.lo[2]) * a.field.inv[2]), a.field.n[2] - 1);
    const int at = (cz * a.field.n[1] + cy) * a.field.n[0] + cx;
    if (ZEF_BOUNDS_OK(at >= 0 && at < a.field.n[0] * a.field.n[1] * a.field.n[2], a.status, 39))
      c = __ldg(reinterpret_cast<const typename FieldCell<WIDE>::T *>(a.field.cells) + at);
  }
  return c;
}

struct LaneStats {
  uint32_t coh = 0, nonfin = 0, nin = 0, eval = 0, own = 0;
};

__device__ void flush_stats(const GridArgs &a, const LaneStats &st, unsigned long long (*s_stat)[GS_COUNT], int wid,
                            int lane) {
  uint32_t v[GS_COUNT];
  v[GS_EVAL] = st.eval;
  v[GS_COHERENT] = st.coh;
  v[GS_OWN] = lane == 0 ? st.own : 0u;  // counted by the whole warp
  v[GS_NONFINITE] = st.nonfin;
  v[GS_NIN] = st.nin;
#pragma unroll
  for (int q = 0; q < GS_COUNT; ++q) v[q] = __reduce_add_sync(0xffffffffu, v[q]);
  if (lane == 0)
#pragma unroll
    for (int q = 0; q < GS_COUNT; ++q) s_stat[wid][q] = v[q];
  __syncthreads();
  if (threadIdx.x < GS_COUNT) {
    unsigned long long t = 0ull;
    for (int w = 0; w < kGlWarps; ++w) t += s_stat[w][threadIdx.x];
    constexpr int kCnt[GS_COUNT] = {CNT_PAIRS_EVAL, CNT_COHERENT, CNT_LANE_TILES, CNT_NONFINITE, CNT_NIN};
    if (t) count_add(a, kCnt[threadIdx.x], t);
  }
}

__device__ __forceinline__ void load_grids(const GridArgs &a, GridComp *s_g, int32_t *s_id) {
  for (int j = threadIdx.x; j < a.ncomp * (int)(sizeof(GridComp) / 16); j += kGlThreads)
    reinterpret_cast<uint4 *>(s_g)[j] = reinterpret_cast<const uint4 *>(a.grid)[j];
  for (int j = threadIdx.x; j < a.ncomp; j += kGlThreads) s_id[j] = a.row_ids[j];
}

// Label, inside bits and Omega rows that the field decides of point i.
template <bool WIDE>
__device__ __forceinline__ void field_store(const GridArgs &a, const int32_t *s_id, int64_t off, int64_t i,
                                            typename FieldCell<WIDE>::M ins, typename FieldCell<WIDE>::M mix, bool fin,
                                            bool open) {
  if (!open) {
    a.labels[off + i] = !fin ? -1 : ins ? s_id[first_row(ins)] : 0;
    if (a.masks) a.masks[off + i] = ins;
  }
  if (a.omega)
    for (int r = 0; r < a.ncomp; ++r)
      if (!((mix >> r) & 1))
        a.omega[(int64_t)r * a.omega_ld + i] = !fin ? __int_as_float(0x7fc00000) : (ins >> r) & 1 ? kFourPi : 0.f;
}

// One launch (small calls): a warp reads the points of a tile, looks their
// field cells up and writes the labels of the points that the field decides;
// the others go to the warp's queue in shared memory, and whenever it holds
// 32 they are decided together.
template <bool WIDE>
__global__ void __launch_bounds__(kGlThreads, 4) k_grid_label(GridArgs a) {
  using M = typename FieldCell<WIDE>::M;
  __shared__ GridComp s_g[ZEF_MAX_COMPARTMENTS];
  __shared__ int32_t s_id[ZEF_MAX_COMPARTMENTS];
  __shared__ Pending<WIDE> s_q[kGlWarps][kGlQueue];
  __shared__ Batch sb;
  __shared__ unsigned long long s_stat[kGlWarps][GS_COUNT];
  load_grids(a, s_g, s_id);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  const int64_t n = a.n_host >= 0 ? a.n_host : a.counters[CNT_N];
  const int64_t off = a.n_host >= 0 ? 0 : a.counters[CNT_OFF];
  const float *pts = a.pts + 3 * off;
  int queued = 0;
  LaneStats st;
  const int64_t tiles = run_tiles(n, a.tile);
  for (int64_t t = (int64_t)wid * gridDim.x + blockIdx.x;; t += (int64_t)gridDim.x * kGlWarps) {
    const bool last = t >= tiles;  // warp-uniform: no points left, only the queue
#pragma unroll
    for (int u = 0; u < kGlP; ++u) {
      if (32 * u >= a.tile) break;
      const int64_t i = run_point(t, tiles, 32 * u + lane);
      const bool valid = !last && i < n && 32 * u + lane < a.tile;
      float x = __int_as_float(0x7fc00000), y = x, z = x;
      if (valid) {
        x = pts[3 * i];
        y = pts[3 * i + 1];
        z = pts[3 * i + 2];
      }
      bool in_box;
      const auto c = field_cell<WIDE>(a, x, y, z, &in_box);
      const M ins = c.x, mix = c.y;
      const bool fin = isfinite(x) && isfinite(y) && isfinite(z), open = open_rows<M>(ins, mix, a.early) != 0;
      if (a.stats) {
        st.coh += sizeof(M) == 8 ? __popcll(ins) : __popc((uint32_t)ins);
        st.nin += in_box ? 1 : 0;
        st.nonfin += valid && !fin ? 1 : 0;
      }
      if (valid) field_store<WIDE>(a, s_id, off, i, ins, mix, fin, open);
      const uint32_t ob = __ballot_sync(0xffffffffu, open);
      if (open) {
        Pending<WIDE> p;
        p.x = x;
        p.y = y;
        p.z = z;
        p.i = (int32_t)i;
        p.ins = ins;
        p.mix = mix;
        const int at = queued + __popc(ob & ((1u << lane) - 1u));
        if (ZEF_BOUNDS_OK(at < kGlQueue, a.status, 40)) s_q[wid][at] = p;
      }
      queued += __popc(ob);
    }
    __syncwarp();
    while (queued >= 32 || (last && queued > 0)) {
      const Pending<WIDE> p = s_q[wid][lane];
      const int cnt = min(queued, 32);
      decide<WIDE, false>(a, s_g, s_id, sb, wid, lane, off, p.x, p.y, p.z, p.i, lane < cnt, p.ins, p.mix, st.eval, st.own);
      for (int j = lane; j + 32 < queued; j += 32) {
        const Pending<WIDE> t = s_q[wid][j + 32];
        s_q[wid][j] = t;
      }
      queued -= cnt;
      __syncwarp();
    }
    if (last) break;
  }
  if (a.stats) flush_stats(a, st, s_stat, wid, lane);
}

// Three launches (large calls).  Streaming: labels of the points that the field
// decides (12 bytes in, 4 out per point, the field from L2; few registers, so
// many loads in flight); the indices of the others are listed, a warp's
// consecutive points in runs of at least kGsFlush.  PLAIN: labels alone, no
// solid angles, inside bits or statistics -- the issue slots bound the
// streaming (four of five busy at 116 instructions per 32 points), so that
// form leaves everything else out.
template <bool WIDE, bool PLAIN>
__global__ void __launch_bounds__(kGlThreads, 6) k_grid_stream(GridArgs a) {
  using M = typename FieldCell<WIDE>::M;
  __shared__ int32_t s_id[ZEF_MAX_COMPARTMENTS + 1];  // label by the number of the first row + 1, 0: none
  __shared__ int32_t s_q[kGlWarps][kGsQueue];
  __shared__ unsigned long long s_stat[kGlWarps][GS_COUNT];
  for (int j = threadIdx.x; j <= a.ncomp; j += kGlThreads) s_id[j] = j ? a.row_ids[j - 1] : 0;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  const int64_t n = a.n_host >= 0 ? a.n_host : a.counters[CNT_N];
  const int64_t off = a.n_host >= 0 ? 0 : a.counters[CNT_OFF];
  int queued = 0;
  LaneStats st;
  const int64_t first = ((int64_t)blockIdx.x * kGlWarps + wid) * a.iters * kGsTile;
  const int count = (int)(min(n, first + (int64_t)a.iters * kGsTile) - first);  // this warp's points, if positive
  const float *p = a.pts + 3 * (off + first + lane);
  int32_t *lab = a.labels + off + first + lane;
  for (int base = 0; base < count; base += kGsTile, p += 3 * kGsTile, lab += kGsTile) {
    float x[kGsP], y[kGsP], z[kGsP];
    bool in_box[kGsP];
    typename FieldCell<WIDE>::T c[kGsP];
    if (base + kGsTile <= count) {
#pragma unroll
      for (int u = 0; u < kGsP; ++u) {
        x[u] = __ldcs(p + 96 * u);
        y[u] = __ldcs(p + 96 * u + 1);
        z[u] = __ldcs(p + 96 * u + 2);
      }
    } else {
#pragma unroll
      for (int u = 0; u < kGsP; ++u) {
        x[u] = y[u] = z[u] = __int_as_float(0x7fc00000);
        if (base + 32 * u + lane < count) {
          x[u] = p[96 * u];
          y[u] = p[96 * u + 1];
          z[u] = p[96 * u + 2];
        }
      }
    }
#pragma unroll
    for (int u = 0; u < kGsP; ++u) c[u] = field_cell<WIDE>(a, x[u], y[u], z[u], &in_box[u]);
#pragma unroll
    for (int u = 0; u < kGsP; ++u) {
      const M ins = c[u].x, mix = c[u].y;
      const int row1 = sizeof(M) == 8 ? __ffsll((long long)ins) : __ffs((int)ins);
      if (PLAIN) {
        // a point with a non-finite coordinate is in no box
        const bool open = open_rows<M>(ins, mix, 1) != 0;
        int32_t l = s_id[row1];
        if (!in_box[u] && !(isfinite(x[u]) && isfinite(y[u]) && isfinite(z[u]))) l = -1;
        if (!open && base + 32 * u + lane < count) lab[32 * u] = l;
        const uint32_t ob = __ballot_sync(0xffffffffu, open);
        const int at = queued + __popc(ob & ((1u << lane) - 1u));
        if (open && ZEF_BOUNDS_OK(at < kGsQueue, a.status, 41)) s_q[wid][at] = (int32_t)(first + base + 32 * u + lane);
        queued += __popc(ob);
      } else {
        const int64_t i = first + base + 32 * u + lane;
        const bool valid = base + 32 * u + lane < count;
        const bool fin = isfinite(x[u]) && isfinite(y[u]) && isfinite(z[u]);
        const bool open = open_rows<M>(ins, mix, a.early) != 0;
        if (a.stats) {
          st.coh += sizeof(M) == 8 ? __popcll(ins) : __popc((uint32_t)ins);
          st.nin += in_box[u] ? 1 : 0;
          st.nonfin += valid && !fin ? 1 : 0;
        }
        if (valid) field_store<WIDE>(a, s_id + 1, off, i, ins, mix, fin, open);
        const uint32_t ob = __ballot_sync(0xffffffffu, open);
        const int at = queued + __popc(ob & ((1u << lane) - 1u));
        if (open && ZEF_BOUNDS_OK(at < kGsQueue, a.status, 42)) s_q[wid][at] = (int32_t)i;
        queued += __popc(ob);
      }
    }
    if (queued >= kGsFlush || (base + kGsTile >= count && queued > 0)) {
      __syncwarp();
      unsigned long long at = 0;
      if (lane == 0) at = atomicAdd((unsigned long long *)(a.counters + CNT_PEND), (unsigned long long)queued);
      at = __shfl_sync(0xffffffffu, at, 0);
      for (int j = lane; j < queued; j += 32)
        if (ZEF_BOUNDS_OK(at + j < (unsigned long long)a.pend_cap, a.status, 43)) a.pending[at + j] = s_q[wid][j];
      queued = 0;
      __syncwarp();
    }
  }
  if (!PLAIN && a.stats) flush_stats(a, st, s_stat, wid, lane);
}

// 32 of the points that the streaming kernel listed, one per lane (entry j).
template <bool WIDE, bool LIST>
__device__ __forceinline__ void pending_batch(const GridArgs &a, const GridComp *s_g, const int32_t *s_id, Batch &sb, int wid,
                                              int lane, int64_t off, int64_t j, int64_t m, LaneStats &st) {
  bool have = j < m;
  const int32_t i = have ? a.pending[j] : 0;
  have = have && ZEF_BOUNDS_OK(i >= 0 && i < (a.n_host >= 0 ? a.n_host : a.counters[CNT_N]), a.status, 44);
  float x = __int_as_float(0x7fc00000), y = x, z = x;
  if (have) {
    const float *p = a.pts + 3 * (off + i);
    x = p[0];
    y = p[1];
    z = p[2];
  }
  bool in_box;
  const auto c = field_cell<WIDE>(a, x, y, z, &in_box);
  decide<WIDE, LIST>(a, s_g, s_id, sb, wid, lane, off, x, y, z, i, have, c.x, c.y, st.eval, st.own);
}

// The listed points, 32 at a time.
template <bool WIDE>
__global__ void __launch_bounds__(kGlThreads, 4) k_grid_pending(GridArgs a) {
  __shared__ GridComp s_g[ZEF_MAX_COMPARTMENTS];
  __shared__ int32_t s_id[ZEF_MAX_COMPARTMENTS];
  __shared__ Batch sb;
  __shared__ unsigned long long s_stat[kGlWarps][GS_COUNT];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // k_grid_open may be launched (it waits)
  const int64_t m = a.counters[CNT_PEND];
  if ((int64_t)blockIdx.x * kGlThreads >= m) return;
  load_grids(a, s_g, s_id);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  const int64_t off = a.n_host >= 0 ? 0 : a.counters[CNT_OFF];
  LaneStats st;
  for (int64_t j0 = (int64_t)blockIdx.x * kGlThreads + 32 * wid; j0 < m; j0 += (int64_t)gridDim.x * kGlThreads)
    pending_batch<WIDE, true>(a, s_g, s_id, sb, wid, lane, off, j0 + lane, m, st);
  if (a.stats) flush_stats(a, st, s_stat, wid, lane);
}

// The points that the crossings left open, one block each: the rows left open
// in turn, the crossings in FP64 by one warp, then the solid angle by the
// block.  (By the warp that met them, one pair after the other, 4,096
// consecutive vertices took 11.7 ms.)  Where the list did not hold them all,
// the pending points are taken once more, their open pairs by the warps.  The
// last block leaves the lists empty, so that a call need not clear them first.
template <bool WIDE>
__global__ void __launch_bounds__(kOpenThreads) k_grid_open(GridArgs a) {
  using M = typename FieldCell<WIDE>::M;
  __shared__ union {
    OpenShared open;
    struct {
      GridComp g[ZEF_MAX_COMPARTMENTS];
      int32_t id[ZEF_MAX_COMPARTMENTS];
      Batch batch;
    } again;
  } sh;
  static_assert(kOpenThreads == kGlThreads, "the second part's batches");
  asm volatile("griddepcontrol.wait;" ::: "memory");  // for k_grid_pending, where launched beside it
  const int64_t listed = a.counters[CNT_OPEN];
  OpenPoint p = a.open[min((int)blockIdx.x, kOpenCap - 1)];  // the block's first, if it has one (with the count, not behind it)
  if (listed == 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) a.counters[CNT_PEND] = 0;
    return;
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t off = a.n_host >= 0 ? 0 : a.counters[CNT_OFF];
  const int64_t n = a.n_host >= 0 ? a.n_host : a.counters[CNT_N], m = a.counters[CNT_PEND];
  if (listed > kOpenCap) {
    load_grids(a, sh.again.g, sh.again.id);
    __syncthreads();
    LaneStats st;  // counted before
    const int64_t tiles = run_tiles(m, 32);
    for (int64_t t = (int64_t)wid * gridDim.x + blockIdx.x; t < tiles; t += (int64_t)gridDim.x * kGlWarps)
      pending_batch<WIDE, false>(a, sh.again.g, sh.again.id, sh.again.batch, wid, lane, off, run_point(t, tiles, lane), m, st);
  } else {
    for (int64_t e = blockIdx.x; e < listed; e += gridDim.x) {
      if (e != blockIdx.x) p = a.open[e];
      if (!ZEF_BOUNDS_OK(p.i >= 0 && p.i < n, a.status, 31)) continue;
      const float x = p.x, y = p.y, z = p.z;
      M mask = (M)p.ins, left = (M)p.open;
      while (left) {
        const int r = first_row(left);
        left &= left - 1;
        const GridComp &g = a.grid[r];
        if (wid == 0) {
          int k = 0;
          const bool decided = crossings64(a, g, cell_word(a, g, x, y, z), x, y, z, lane, &k);
          if (lane == 0) {
            sh.open.decided = decided;
            sh.open.k = k;
          }
        }
        __syncthreads();
        const bool decided = sh.open.decided;
        const int k = sh.open.k;
        __syncthreads();
        const double om = decided ? 0.0 : solid64_block(a, g, x, y, z, sh.open, lane, wid);
        const bool inside = decided ? k >= 1 : om > kTwoPi64;
        if (threadIdx.x == 0 && a.omega) a.omega[(int64_t)r * a.omega_ld + p.i] = decided ? kFourPi * (float)k : (float)om;
        if (inside) {
          mask |= (M)1 << r;
          if (a.early) left = 0;
        }
      }
      if (threadIdx.x == 0) {
        a.labels[off + p.i] = mask ? a.row_ids[first_row(mask)] : 0;
        if (a.masks) a.masks[off + p.i] = mask;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x == 0 &&
      atomicAdd((unsigned long long *)(a.counters + CNT_OPEN_DONE), 1ull) == (unsigned long long)gridDim.x - 1ull) {
    a.counters[CNT_PEND] = 0;
    a.counters[CNT_OPEN] = 0;
    a.counters[CNT_OPEN_DONE] = 0;
  }
}

__global__ void k_grid_reset(int64_t *cnt) {
  constexpr int c[] = {CNT_ITEMS, CNT_UNC,      CNT_NONFINITE, CNT_PAIRS_EVAL, CNT_PAIRS_RESCUE,
                       CNT_COHERENT, CNT_REP_PAIRS, CNT_LANE_TILES, CNT_NIN,     CNT_TILES,      CNT_PEND,
                       CNT_OPEN,     CNT_OPEN_DONE};
  if (threadIdx.x < sizeof(c) / sizeof(c[0])) cnt[c[threadIdx.x]] = 0;
}

bool grid_opts(const zef_label_opts &o) {
  // |4 pi k - 2 pi| >= 2 pi: no certified winding number is within a margin
  // below that of the threshold
  return o.precision == ZEF_FP32_RESCUE && o.kernel == 0 && o.flags == 0 && !o.block_threads && !o.points_per_thread &&
         o.margin < 6.f;
}

}  // namespace

// The cell grid serves a call when every compartment has one and the options
// ask for nothing the general kernels alone give: their launch shapes and
// forms, raw FP32 sums, FP32 or FP64 alone, every point evaluated for
// itself, or a margin that covers the certified values.
bool grid_serves(const zef_ctx *ctx, const zef_label_opts &o) {
  if (!grid_opts(o) || ctx->grids.size() != ctx->comps.size() || !ctx->field.cells) return false;
  for (const CompGrid &g : ctx->grids)
    if (!g.usable) return false;
  return true;
}

// Calls of at least kListedMin points list the points that the field leaves
// open and decide them in a second kernel: the streaming part alone needs 40
// registers instead of 64 and the lists fill every batch (56.2 M points: 958
// us in one kernel, 657 in two; 5 M: 151 and 97).  Below that the further
// launches cost more than they save (scratch: 4 bytes per point, which the
// allocation-free entry point, at most 65,536 points, never needs).
constexpr int64_t kListedMin = 1 << 18;
static_assert(kListedMin > ZEF_NOALLOC_MAX_POINTS, "the allocation-free entry point has no list");
static bool grid_listed(const zef_ctx *ctx, int64_t n_cap) {
  return n_cap >= kListedMin && ctx->lb.cap_pending >= n_cap && ctx->lb.open;
}

zef_status grid_reserve(zef_ctx *ctx, int64_t n_cap) {
  LabelBuffers &b = ctx->lb;
  if (n_cap < kListedMin) return ZEF_OK;
  if (!b.open) {
    const cudaError_t e = cudaMalloc(&b.open, kOpenCap * sizeof(OpenPoint));
    if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaMalloc(points on a surface)");
  }
  if (b.cap_pending >= n_cap) return ZEF_OK;
  if (b.pending) cudaFree(b.pending);
  b.pending = nullptr;
  b.cap_pending = 0;
  cudaError_t e = cudaMalloc(&b.pending, (size_t)n_cap * sizeof(int32_t));
  if (e != cudaSuccess) return cuda_fail(ctx, e, "cudaMalloc(open points)");
  b.cap_pending = n_cap;
  return ZEF_OK;
}

zef_status grid_enqueue(zef_ctx *ctx, const LabelPlan &plan) {
  cudaStream_t s = ctx->stream;
  GridArgs a;
  a.pts = plan.pts;
  a.labels = plan.labels;
  a.omega = plan.omega;
  a.omega_ld = plan.omega_ld;
  a.masks = plan.masks;
  a.grid = ctx->d_grid;
  a.row_ids = ctx->d_row_ids;
  a.counters = ctx->lb.counters;
  a.n_host = plan.n_host;
  a.ncomp = (int)ctx->comps.size();
  a.early = plan.omega == nullptr && !plan.full_masks;
  a.stats = plan.counted;
  a.ub = ctx->ubox;
  a.field = ctx->field;
  a.status = ctx->d_status;
  a.comps = ctx->d_comps;
  a.nodes = ctx->d_nodes;
  a.cseg = ctx->d_cseg;
#ifdef ZEF_DEBUG_BOUNDS
  a.n_nodes = (int64_t)ctx->h_nodes.size();
  a.n_cseg = (int64_t)ctx->h_cseg.size();
  a.pend_cap = ctx->lb.cap_pending;
#endif
  a.scale = ctx->scale;
  // The list serves calls that fill the GPU; below that one launch is shorter.
  const bool listed = grid_listed(ctx, plan.n_cap);
  a.pending = ctx->lb.pending;
  a.open = ctx->lb.open;
  if (plan.timed) cudaEventRecord(ctx->ev[0], s);
  const bool dirty = ctx->lb.lists_dirty;
  if (a.stats || (listed && dirty)) {
    k_grid_reset<<<1, 32, 0, s>>>(ctx->lb.counters);
    ++ctx->launches;
  }
  if (listed) ctx->lb.lists_dirty = true;  // until every kernel of this call is launched
  NvtxRange nvtx_stage("zef.label_kernel");
  if (plan.timed) cudaEventRecord(ctx->ev[1], s);
  const bool wide = a.ncomp > 32;
  a.tile = kGlTile;
  if (listed) {
    const int64_t tiles = (plan.n_cap + kGsTile - 1) / kGsTile;
    // a warp's consecutive tiles list neighbouring points together
    a.iters = (int)std::min<int64_t>(kGlMaxIters, std::max<int64_t>(1, tiles / ((int64_t)ctx->num_sms * 16 * kGlWarps)));
    const unsigned blocks = (unsigned)((tiles + (int64_t)a.iters * kGlWarps - 1) / ((int64_t)a.iters * kGlWarps));
    const unsigned pblocks = (unsigned)std::min<int64_t>((plan.n_cap + kGlThreads - 1) / kGlThreads, (int64_t)ctx->num_sms * 16);
    const bool plain = !a.omega && !a.masks && !a.stats && a.early;
    auto stream = wide ? (plain ? k_grid_stream<true, true> : k_grid_stream<true, false>)
                       : (plain ? k_grid_stream<false, true> : k_grid_stream<false, false>);
    stream<<<blocks, kGlThreads, 0, s>>>(a);
    if (wide) k_grid_pending<true><<<pblocks, kGlThreads, 0, s>>>(a);
    else k_grid_pending<false><<<pblocks, kGlThreads, 0, s>>>(a);
    ctx->launches += 2;
  } else {
    // as few points per warp as 16 warps an SM allow, kRun to kGlTile (calls
    // one behind the other, the three-layer head; with 8, 16, 32, 64: 5,000 points 8.2,
    // 8.3, 8.3, 10.3 us; 36,864 10.3, 10.3, 8.3, 10.3; 65,536 with solid
    // angles 16.5, 12.3, 10.3, 11.8; 200,000 with them 36, 25, 19, 14.5);
    // neighbouring tiles go to different blocks
    a.iters = 1;
    while (a.tile > kRun && plan.n_cap <= (int64_t)ctx->num_sms * 16 * (a.tile / 2)) a.tile /= 2;
    const int64_t tiles = std::max<int64_t>(1, (plan.n_cap + a.tile - 1) / a.tile);
    const unsigned blocks = (unsigned)std::min(tiles, std::max((int64_t)ctx->num_sms, (tiles + kGlWarps - 1) / kGlWarps));
    if (wide) k_grid_label<true><<<blocks, kGlThreads, 0, s>>>(a);
    else k_grid_label<false><<<blocks, kGlThreads, 0, s>>>(a);
    ++ctx->launches;
  }
  if (plan.timed) cudaEventRecord(ctx->ev[2], s);
  nvtx_stage.next("zef.rescue64");
  if (plan.timed) cudaEventRecord(ctx->ev[3], s);
  if (listed) {
    // most calls have few such points or none: the launch overlaps the kernel
    // before it (the library's own graphs, some with conditional nodes, and
    // timed calls, with events in between, launch it the plain way).  5.2 M
    // points: 84.8 us, 83.9 with the overlap; a million nodes with every row
    // decided: 75.6 and 73.8
    cudaLaunchAttribute overlap;
    overlap.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    overlap.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)ctx->num_sms * 2);
    cfg.blockDim = dim3(kOpenThreads);
    cfg.stream = s;
    cfg.attrs = &overlap;
    cfg.numAttrs = plan.n_host >= 0 && !plan.timed ? 1 : 0;
    cudaLaunchKernelEx(&cfg, wide ? k_grid_open<true> : k_grid_open<false>, a);
    ++ctx->launches;
  }
  if (plan.timed) {
    cudaEventRecord(ctx->ev[4], s);
    cudaEventRecord(ctx->ev[5], s);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(ctx, e, "k_grid_label launch");
  // enqueued into one of the library's graphs (n_host < 0) nothing has run yet
  if (listed) ctx->lb.lists_dirty = plan.n_host < 0 && dirty;
  return ZEF_OK;
}

void grid_free(zef_ctx *ctx) {
  for (CompGrid &g : ctx->grids)
    if (g.blob) cudaFree(g.blob);
  ctx->grids.clear();
  if (ctx->d_grid) cudaFree(ctx->d_grid);
  if (ctx->field_mem) cudaFree(ctx->field_mem);
  for (void *&p : ctx->gr_buf) {
    if (p) cudaFree(p);
    p = nullptr;
  }
  ctx->d_grid = nullptr;
  ctx->field.cells = ctx->field_mem = nullptr;
}

// Cells of the boxes of all triangles of a surface, n cells a side.
static double box_cells(const zef_ctx *ctx, const CompHost &h, const int (&n)[3]) {
  const float4 *v = ctx->h_tris.data() + 3 * h.tri_off;
  float inv[3];
  for (int k = 0; k < 3; ++k) inv[k] = h.hi[k] > h.lo[k] ? (float)n[k] / (h.hi[k] - h.lo[k]) : 0.f;
  double sum = 0.0;
  for (int64_t t = 0; t < h.nt; ++t, v += 3) {
    const float lo[3] = {std::min(v[0].x, std::min(v[1].x, v[2].x)), std::min(v[0].y, std::min(v[1].y, v[2].y)),
                         std::min(v[0].z, std::min(v[1].z, v[2].z))};
    const float hi[3] = {std::max(v[0].x, std::max(v[1].x, v[2].x)), std::max(v[0].y, std::max(v[1].y, v[2].y)),
                         std::max(v[0].z, std::max(v[1].z, v[2].z))};
    double box = 1.0;
    for (int k = 0; k < 3; ++k) box *= (double)((int)((hi[k] - h.lo[k]) * inv[k]) - (int)((lo[k] - h.lo[k]) * inv[k]) + 1);
    sum += box;
  }
  return sum;
}

// Cell grid of compartment c (uploaded, with its cap tree).  Cells are one
// mean triangle edge wide (a cell with triangles then lists about seven of
// them, one chunk; 56.2 M points in 24 compartments: 650 us at 0.8 edges, 657
// at 1.0, 729 at 1.3, and the memory grows with the inverse square), at least
// eight along the longest side, at most kMaxCells in all.
// A surface whose grid would not pay -- a list longer than kMaxList (all its
// triangles in a few cells), coordinates whose cubes leave FP32's range, no
// memory -- is left without: calls then take the general kernels.
static zef_status grid_build(zef_ctx *ctx, size_t c, CompGrid *out) {
  const CompHost &h = ctx->comps[c];
  CompGrid gr;
  float big = 0.f, ext[3], longest = 0.f;
  for (int k = 0; k < 3; ++k) {
    big = std::max(big, std::max(std::fabs(h.lo[k]), std::fabs(h.hi[k])));
    ext[k] = h.hi[k] - h.lo[k];
    longest = std::max(longest, ext[k]);
  }
  *out = gr;
  if (!(big > 1e-12f && big < 1e12f && longest > 1e-6f * big)) return ZEF_OK;
  double w = 1.0 * std::sqrt(h.area / (0.43 * (double)h.nt));
  w = std::min(w, (double)longest / 8.0);
  w = std::max(w, (double)longest / kMaxAxis);
  // a cell is many float32 steps wide on every axis it divides, so that its
  // anchor, rounded to float32, stays inside
  double finest[3];
  for (int k = 0; k < 3; ++k)
    finest[k] = std::max(1.0, std::floor((double)ext[k] * 65536.0 / std::max(std::fabs(h.lo[k]), std::fabs(h.hi[k]))));
  Geom g;
  int64_t cells = 0;
  for (double grow = 1.1;; w *= grow) {
    cells = 1;
    for (int k = 0; k < 3; ++k) {
      g.n[k] = (int)std::min<double>(std::min<double>(kMaxAxis, finest[k]), std::max(1.0, std::ceil(ext[k] / w)));
      cells *= g.n[k];
    }
    if (cells > kMaxCells) continue;
    // k_gr_refs goes through the cells of every triangle's box, a few of them
    // for triangles as wide as a cell; for long thin ones across the surface's
    // box nearly all, so their cells are as wide as kBoxCells allows (2,000
    // needles: 192 ms to register, 27 now)
    const double most = kBoxCells + 1024.0 * (double)h.nt, boxes = box_cells(ctx, h, g.n);
    if (boxes <= most) break;
    grow = std::max(1.1, std::cbrt(boxes / most));
  }
  for (int k = 0; k < 3; ++k) {
    g.lo[k] = h.lo[k];
    g.h[k] = (double)ext[k] / g.n[k];
    g.inv[k] = ext[k] > 0.f ? (float)(g.n[k] / (double)ext[k]) : 0.f;
  }
  int e2 = 0;
  std::frexp(big, &e2);
  const double s = std::ldexp(1.0, 6 - e2);
  const float to_raw = 1.f / ctx->scale;
  const float4 *tris = ctx->d_tris + h.tri_off * 3;
  const int nt = (int)h.nt;
  cudaStream_t st = ctx->stream;

  // scratch: counts / list ends, block sizes / offsets, scan sums, totals
  // (longest list, triangles of all lists, words of all blocks), anchors, their Omega
  const int64_t bs = cells / 2048 + 2;
  const size_t o_flag = (size_t)cells * 4, o_sum = o_flag + (size_t)cells * 4, o_tot = (o_sum + (size_t)bs * 4 + 15) & ~(size_t)15,
               o_anch = o_tot + 32, o_om = o_anch + (size_t)cells * 12, bytes = o_om + (size_t)cells * 4;
  auto no_memory = [&](cudaError_t e) {
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? ZEF_OK : cuda_fail(ctx, e, "cell grid");
  };
  auto scratch = [](void **p, size_t *cap, size_t need) {
    if (*cap >= need) return cudaSuccess;
    if (*p) cudaFree(*p);
    *p = nullptr;
    *cap = 0;
    const cudaError_t e = cudaMalloc(p, need);
    if (e == cudaSuccess) *cap = need;
    return e;
  };
  cudaError_t e = scratch(&ctx->gr_buf[0], &ctx->gr_cap[0], bytes);
  if (e != cudaSuccess) return no_memory(e);
  unsigned char *tmp = (unsigned char *)ctx->gr_buf[0];
  uint32_t *cnt = (uint32_t *)tmp, *flag = (uint32_t *)(tmp + o_flag), *bsum = (uint32_t *)(tmp + o_sum);
  int64_t *tot = (int64_t *)(tmp + o_tot);
  float *anchor = (float *)(tmp + o_anch), *omega = (float *)(tmp + o_om);
  cudaMemsetAsync(cnt, 0, (size_t)cells * 4, st);
  cudaMemsetAsync(tot, 0, 32, st);
  const int g_t = grid_blocks(ctx, (int64_t)nt * 32, 256), g_c = grid_blocks(ctx, cells, 256),
            g_w = grid_blocks(ctx, cells * 32, 256);
  k_gr_refs<<<g_t, 256, 0, st>>>(tris, to_raw, nt, g, cnt, nullptr);
  k_gr_sizes<<<g_c, 256, 0, st>>>(cnt, cells, flag, (unsigned long long *)tot);
  zef_status zs = scan_exclusive(ctx, cnt, nullptr, 1, cells, nullptr, bsum);
  if (!zs) zs = scan_exclusive(ctx, flag, nullptr, 1, cells, nullptr, bsum);
  int64_t totals[3] = {0, 0, 0};
  if (!zs) {
    e = cudaMemcpyAsync(totals, tot, sizeof(totals), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) zs = cuda_fail(ctx, e, "cell grid");
  }
  if (zs) return zs;
  const int64_t refs = totals[1], words16 = totals[2];
  if (totals[0] > kMaxList || refs > (int64_t)UINT32_MAX || refs > 64 * (int64_t)nt + 65536 || words16 > (int64_t)kOffsetMask)
    return ZEF_OK;
  // blocks and words; the triangle lists are scratch
  const size_t p_word = (size_t)words16 * 16, p_end = p_word + (size_t)cells * 4;
  unsigned char *blob = nullptr;
  e = scratch(&ctx->gr_buf[1], &ctx->gr_cap[1], std::max<size_t>((size_t)refs * 4, 16));
  if (e == cudaSuccess) e = cudaMalloc(&blob, p_end);
  if (e != cudaSuccess) return no_memory(e);
  int32_t *list = (int32_t *)ctx->gr_buf[1];
  k_gr_refs<<<g_t, 256, 0, st>>>(tris, to_raw, nt, g, cnt, list);  // cnt: list starts -> ends
  k_gr_anchor<<<g_w, 256, 0, st>>>(tris, to_raw, g, cells, cnt, list, anchor);
  // the anchors' solid angles of this compartment alone
  zs = label_reserve(ctx, cells);
  if (!zs) zs = label_reserve_stage(ctx, cells);
  if (!zs) {
    LabelPlan p;
    p.pts = anchor;
    p.labels = ctx->lb.labels_tmp;
    p.omega = omega;
    p.omega_ld = cells;
    p.n_cap = cells;
    p.n_host = -1;
    p.d_n = ctx->lb.counters + CNT_N;
    p.d_off = ctx->lb.counters + CNT_OFF;
    std::memset(&p.opts, 0, sizeof(p.opts));
    fill_default_opts(&p.opts);
    p.shape = LaunchShape{256, 2, kernel_variant(0)};
    p.timed = false;
    p.only_comp = (int)c;
    DevComp *rec = ctx->d_comps + ZEF_MAX_COMPARTMENTS;
    cudaMemcpyAsync(rec, ctx->d_comps + c, sizeof(DevComp), cudaMemcpyDeviceToDevice, st);
    cudaMemsetAsync(&rec->row, 0, sizeof(rec->row), st);
    zs = label_set_count(ctx, cells, 0);
    if (!zs) zs = label_enqueue(ctx, p);
  }
  if (zs) {
    cudaStreamSynchronize(st);
    cudaFree(blob);
    if (zs != ZEF_ERR_OOM) return zs;
    cudaGetLastError();
    return ZEF_OK;
  }
  k_gr_finish<<<g_w, 256, 0, st>>>(tris, to_raw, s, g, cells, cnt, flag, list, anchor, omega, (uint32_t *)(blob + p_word),
                                   (float4 *)blob);
  e = cudaGetLastError();
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(ctx->h_status, ctx->d_status, 2 * sizeof(uint32_t), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  // anchors whose sums were cut short: no grid from them.  The error is this
  // call's; what an earlier call recorded beside it stays to be reported.
  constexpr uint32_t cut = ST_TIMEOUT | ST_BOUNDS;
  const uint32_t status = ctx->h_status[0];
  if (e == cudaSuccess && (status & cut)) {
    ctx->h_status[0] = status & ~cut;
    e = cudaMemcpyAsync(ctx->d_status, ctx->h_status, sizeof(uint32_t), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e == cudaSuccess) {
      cudaFree(blob);
      return fail(ctx, status & ST_TIMEOUT ? ZEF_ERR_TIMEOUT : ZEF_ERR_BOUNDS,
                  "the solid angles of a cell grid's anchors were cut short (site " + std::to_string(ctx->h_status[1]) + ")");
    }
  }
  if (e != cudaSuccess) {
    cudaFree(blob);
    return cuda_fail(ctx, e, "cell grid");
  }
  gr.blob = blob;
  gr.usable = true;
  gr.words = (const uint32_t *)(blob + p_word);
  gr.blocks = (const float4 *)blob;
  for (int k = 0; k < 3; ++k) {
    gr.n[k] = g.n[k];
    gr.inv[k] = g.inv[k];
  }
  *out = gr;
  return ZEF_OK;
}

// Grids of the compartments that have none yet, then the device records in
// priority order (the surfaces are uploaded).
zef_status grid_update(zef_ctx *ctx) {
  const size_t C = ctx->comps.size();
  const int64_t held = ctx->lb.cap_points;
  while (ctx->grids.size() < C) {
    CompGrid g;
    zef_status st = grid_build(ctx, ctx->grids.size(), &g);
    if (st) return st;
    ctx->grids.push_back(g);
  }
  // what the construction alone needed is given back where it is large: the
  // anchors' work buffers (calls that the grids serve need none) and the
  // scratch (24 bytes a cell and the triangle lists), which small surfaces
  // registered one after the other reuse
  if (ctx->lb.cap_points > held && ctx->lb.cap_points > (int64_t)1 << 22) label_release(ctx);
  if (ctx->gr_cap[0] + ctx->gr_cap[1] > kScratchKept)
    for (int k = 0; k < 2; ++k) {
      if (ctx->gr_buf[k]) cudaFree(ctx->gr_buf[k]);
      ctx->gr_buf[k] = nullptr;
      ctx->gr_cap[k] = 0;
    }
  if (!ctx->d_grid) CK(cudaMalloc(&ctx->d_grid, ZEF_MAX_COMPARTMENTS * sizeof(GridComp)), "cudaMalloc(cell grids)");
  std::vector<GridComp> &d = ctx->h_grid;  // outlives the copy
  d.assign(C, GridComp{});
  for (size_t c = 0; c < C; ++c) {
    const CompHost &h = ctx->comps[c];
    const CompGrid &g = ctx->grids[c];
    size_t row = 0;
    while (row < C && ctx->priority[row] != h.id) ++row;
    GridComp &r = d[row];
    for (int k = 0; k < 3; ++k) {
      r.lo[k] = h.lo[k];
      r.hi[k] = h.hi[k];
      r.inv[k] = g.inv[k];
      r.n[k] = g.n[k];
    }
    r.comp = (int32_t)c;
    r.tri_raw = 1.f / ctx->scale;
    r.words = g.words;
    r.blocks = g.blocks;
    r.tris = ctx->d_tris + h.tri_off * 3;
  }
  CK(cudaMemcpyAsync(ctx->d_grid, d.data(), C * sizeof(GridComp), cudaMemcpyHostToDevice, ctx->stream),
     "upload cell grids");

  // the label field: cells as wide as the finest compartment grid's, at most
  // kMaxField of them (one or two 64-bit words each: it stays in L2)
  ctx->field.cells = nullptr;
  LabelField f = {};
  float ext[3], longest = 0.f;
  for (int k = 0; k < 3; ++k) {
    ext[k] = ctx->ubox.hi[k] - ctx->ubox.lo[k];
    longest = std::max(longest, ext[k]);
  }
  double w = longest;
  for (size_t c = 0; c < C; ++c) {
    if (!ctx->grids[c].usable) return ZEF_OK;
    for (int k = 0; k < 3; ++k)
      if (ctx->grids[c].n[k] > 1) w = std::min(w, (double)(ctx->comps[c].hi[k] - ctx->comps[c].lo[k]) / ctx->grids[c].n[k]);
  }
  int64_t cells = 0;
  for (;; w *= 1.05) {
    cells = 1;
    for (int k = 0; k < 3; ++k) {
      f.n[k] = (int)std::min<double>(kMaxAxis, std::max(1.0, std::ceil(ext[k] / w)));
      cells *= f.n[k];
    }
    if (cells <= kMaxField) break;
  }
  for (int k = 0; k < 3; ++k) {
    f.lo[k] = ctx->ubox.lo[k];
    f.h[k] = (double)ext[k] / f.n[k];
    f.inv[k] = ext[k] > 0.f ? (float)(f.n[k] / (double)ext[k]) : 0.f;
  }
  const bool wide = C > 32;
  const size_t need = (size_t)cells * (wide ? sizeof(ulonglong2) : sizeof(uint2));
  if (ctx->field_cap < need) {
    if (ctx->field_mem) cudaFree(ctx->field_mem);
    ctx->field_mem = nullptr;
    ctx->field_cap = 0;
    cudaError_t e = cudaMalloc(&ctx->field_mem, need);
    if (e == cudaErrorMemoryAllocation) {
      cudaGetLastError();
      return ZEF_OK;  // no field: the general kernels
    }
    CK(e, "cudaMalloc(label field)");
    ctx->field_cap = need;
  }
  f.cells = ctx->field_mem;
  ctx->field = f;
  const int g_f = grid_blocks(ctx, cells, 256);
  if (wide) k_gr_field<true><<<g_f, 256, 0, ctx->stream>>>(f, ctx->d_grid, (int)C);
  else k_gr_field<false><<<g_f, 256, 0, ctx->stream>>>(f, ctx->d_grid, (int)C);
  CK(cudaGetLastError(), "label field");
  return ZEF_OK;
}

}  // namespace zef
