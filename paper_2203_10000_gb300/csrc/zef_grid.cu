// zef_grid.cu -- the cell grid of a compartment surface and the labeling
// kernel that reads it.
//
// The winding number of a closed surface S (Omega / 4 pi, Sec. 2.1.3) is
// constant on every region that S does not cross and changes by the signed
// count of crossings along a segment that does: k(p) = k(q) + (inward -
// outward crossings of the segment q -> p).  So the solid angle needs to be
// summed at a few fixed points only.  At registration every compartment's box
// is cut into cells about two triangle edges wide; each cell lists the
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
// else -- a point within about 1e-6 cell widths of a triangle's plane inside
// the triangle, a segment that close to an edge -- is re-evaluated in FP64
// from the vertices (again with a bound), and what FP64 cannot decide either
// (a point on the surface) by the FP64 solid angle over the cap tree, as the
// re-evaluation of zef_label.cu does.
//
// Why: the general kernels sum about 1,000 strip entries of a tile's walk for
// every point near a surface (FP32 ALUs, 54 of the 58 ms of 56.2 M points in
// 24 compartments); here such a point costs about a dozen crossing tests held
// by the lanes of one warp, and every other point one word per compartment.
// No sort of the points, no work list and no work buffers: one launch.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <cstring>
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
constexpr uint32_t kMixed = 0x80000000u;    // cell word: index of the cell's record, else its winding number
constexpr uint32_t kUnknown = 0x40000000u;  // cell word: anchor's winding number unknown
constexpr int kNoK = INT32_MIN;             // record: anchor's winding number unknown
// Every cell is treated as grown by kGrow of its width on each side: a point
// whose cell index is off by the rounding of (x - lo) * n / extent (at most a
// few 2^-24 n of a cell, n <= 512) still lies in the grown cell.
constexpr double kGrow = 2e-3;
constexpr float kGrowF = 2e-3f;
constexpr int64_t kMaxCells = 1 << 23;
constexpr int kMaxAxis = 512;
constexpr int kMaxList = 1024;  // longest triangle list of a usable grid

struct Geom {
  float lo[3], inv[3];
  double h[3];
  int n[3];
};

__device__ __forceinline__ float4 raw_vertex(float4 v, float s) { return make_float4(v.x * s, v.y * s, v.z * s, 0.f); }

// Triangles of every cell: one warp per triangle, the lanes over the cells of
// its box; a cell counts when the triangle's plane meets the grown cell.  The
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
      const int64_t c = ((int64_t)z * g.n[1] + y) * g.n[0] + x;
      const uint32_t pos = atomicAdd(cnt + c, 1u);
      if (list) list[pos] = (int32_t)t;
    }
  }
}

// non-empty cells (to be scanned into record numbers) and the longest list
__global__ void __launch_bounds__(256) k_gr_flags(const uint32_t *cnt, int64_t cells, uint32_t *flag,
                                                  unsigned long long *longest) {
  uint32_t mx = 0;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < cells; c += (int64_t)gridDim.x * blockDim.x) {
    flag[c] = cnt[c] ? 1u : 0u;
    mx = max(mx, cnt[c]);
  }
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0 && mx) atomicMax(longest, (unsigned long long)mx);
}

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

// Words and records of the cells and the stored products of every (cell,
// triangle) pair, from the anchors' solid angles.  Vertices relative to the
// anchor are exact in FP64 up to its rounding; s (a power of two) brings them
// to about [-64, 64]; the stored cross products carry one factor s more, for
// the unscaled d = p - q of the kernel.
__global__ void __launch_bounds__(256) k_gr_finish(const float4 *tris, float to_raw, double s, Geom g, int64_t cells,
                                                   const uint32_t *last, const uint32_t *rank, const int32_t *list,
                                                   const float *anchor, const float *omega, uint32_t *words,
                                                   GridCell *recs, float4 *refs) {
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
    if (lane == 0) {
      words[c] = kMixed | rank[c];
      GridCell r;
      r.x = qx;
      r.y = qy;
      r.z = qz;
      r.k = known ? (int)kf : kNoK;
      r.begin = (int)b;
      r.count = (int)(e - b);
      r.pad0 = r.pad1 = 0;
      recs[rank[c]] = r;
    }
    for (uint32_t j = b + lane; j < e; j += 32) {
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
      float4 *o = refs + 3 * (int64_t)j;
      o[0] = make_float4((float)(N[0][0] * s), (float)(N[0][1] * s), (float)(N[0][2] * s), (float)V);
      o[1] = make_float4((float)(N[1][0] * s), (float)(N[1][1] * s), (float)(N[1][2] * s), __double2float_ru(E));
      o[2] = make_float4((float)(N[2][0] * s), (float)(N[2][1] * s), (float)(N[2][2] * s), 0.f);
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
  int64_t n_host;             // points, or -1: counters[CNT_N] from counters[CNT_OFF] on
  int ncomp;
  int early;                  // a point certainly inside needs no later compartment
  int stats;
  UnionBox ub;
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
enum GridStat { GS_EVAL = 0, GS_COHERENT, GS_OWN, GS_ITEMS, GS_NONFINITE, GS_NIN, GS_COUNT };

// FP64 re-evaluation of one (point, compartment) pair by the whole warp: the
// crossings from the vertices in FP64, each sign taken only beyond its
// rounding bound; where that leaves one open, the FP64 solid angle over the
// cap tree.  Returns whether the point is inside; *omega = Omega.
__device__ __noinline__ bool resolve64(const GridArgs &a, const GridComp &g, uint32_t word, float x, float y, float z,
                                       int lane, float *omega) {
  if (word & kMixed) {
    const GridCell r = g.cells[word & ~kMixed];
    int net = 0;
    bool open = r.k == kNoK;
    if (!open) {
      const double dx = (double)x - r.x, dy = (double)y - r.y, dz = (double)z - r.z;
      for (int j = lane; j < r.count; j += 32) {
        const int64_t t = g.tri[r.begin + j];
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
      if (lane == 0 && a.stats) {
        count_add(a, CNT_UNC, 1);
        count_add(a, CNT_PAIRS_RESCUE, (unsigned long long)r.count);
      }
      *omega = kFourPi * (float)(r.k + net);
      return r.k + net >= 1;
    }
  }
  // FP64 solid angle: the caps of the nodes whose box misses the point, the
  // leaves whose box holds it
  const DevComp *cp = a.comps + g.comp;
  const float px = x * a.scale, py = y * a.scale, pz = z * a.scale;
  // the groups of four entries in the order of the list kernel's block of 256
  // threads (thread g mod 256 takes group g; the sums of each 32 threads, then
  // of the eight in turn), so that a point on the surface, whose Omega is 2 pi
  // up to rounding, gets that kernel's rounding
  double part[8];
#pragma unroll
  for (int w = 0; w < 8; ++w) part[w] = 0.0;
  int K = 0, tris = 0, g0 = 0;
  const int root = cp->cap_root, end = a.nodes[root].skip;
  for (int i = root; i != end;) {
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
    for (int j = (lane - g0) & 31; j < c / 4; j += 32) {
      const double h = group64(a.cseg, b + 4 * j, px, py, pz, &K);
      const int w = ((g0 + j) >> 5) & 7;
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (q == w) part[q] += h;
    }
    g0 += c / 4;
  }
  double sum = 0.0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) part[q] += __shfl_xor_sync(0xffffffffu, part[q], o);
    sum += part[q];
  }
  K = __reduce_add_sync(0xffffffffu, K);
  const double om = 2.0 * (sum + 6.283185307179586476925 * (double)K);
  if (lane == 0 && a.stats) {
    count_add(a, CNT_UNC, 1);
    count_add(a, CNT_PAIRS_RESCUE, (unsigned long long)tris);
  }
  *omega = (float)om;
  return om > 6.283185307179586476925;
}

// order-preserving int of a float, and back
__device__ __forceinline__ int ord(float f) {
  const int b = __float_as_int(f);
  return b ^ ((b >> 31) & 0x7fffffff);
}
__device__ __forceinline__ float unord(int b) { return __int_as_float(b ^ ((b >> 31) & 0x7fffffff)); }

constexpr int kGlThreads = 256;
constexpr int kGlP = 2;               // points per lane
constexpr int kGlTile = 32 * kGlP;    // points of a warp's tile

// One warp per tile of 64 consecutive points.  The tile's box selects the
// compartments (one per lane); for each of them every lane looks its points'
// cells up; points in cells with triangles are taken cell by cell: the lanes
// hold 32 of the cell's triangles (stored products, 48 bytes each, read
// once per tile and cell) and the points of the cell are broadcast one after
// the other, so the work of a point does not depend on its neighbours' lists.
__global__ void __launch_bounds__(kGlThreads) k_grid_label(GridArgs a) {
  __shared__ GridComp s_g[ZEF_MAX_COMPARTMENTS];
  for (int j = threadIdx.x; j < a.ncomp * (int)(sizeof(GridComp) / 16); j += kGlThreads)
    reinterpret_cast<uint4 *>(s_g)[j] = reinterpret_cast<const uint4 *>(a.grid)[j];
  __shared__ unsigned long long s_stat[kGlThreads / 32][GS_COUNT];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane < GS_COUNT) s_stat[wid][lane] = 0ull;
  __syncthreads();
  const int64_t n = a.n_host >= 0 ? a.n_host : a.counters[CNT_N];
  const int64_t off = a.n_host >= 0 ? 0 : a.counters[CNT_OFF];
  const int64_t step = (int64_t)gridDim.x * (kGlThreads / 32) * kGlTile;
  for (int64_t base = ((int64_t)blockIdx.x * (kGlThreads / 32) + wid) * kGlTile; base < n; base += step) {
    float x[kGlP], y[kGlP], z[kGlP];
    bool fin[kGlP], done[kGlP];
    unsigned long long mask[kGlP];
    int lo[3] = {INT32_MAX, INT32_MAX, INT32_MAX}, hi[3] = {INT32_MIN, INT32_MIN, INT32_MIN};
#pragma unroll
    for (int u = 0; u < kGlP; ++u) {
      const int64_t i = base + 32 * u + lane;
      x[u] = y[u] = z[u] = 0.f;
      if (i < n) {
        const float *p = a.pts + 3 * (off + i);
        x[u] = p[0];
        y[u] = p[1];
        z[u] = p[2];
      }
      fin[u] = i < n && isfinite(x[u]) && isfinite(y[u]) && isfinite(z[u]);
      done[u] = !fin[u];
      mask[u] = 0ull;
      if (fin[u]) {
        lo[0] = min(lo[0], ord(x[u])); hi[0] = max(hi[0], ord(x[u]));
        lo[1] = min(lo[1], ord(y[u])); hi[1] = max(hi[1], ord(y[u]));
        lo[2] = min(lo[2], ord(z[u])); hi[2] = max(hi[2], ord(z[u]));
      }
    }
    float wlo[3], whi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      wlo[k] = unord(__reduce_min_sync(0xffffffffu, lo[k]));
      whi[k] = unord(__reduce_max_sync(0xffffffffu, hi[k]));
    }
    unsigned long long met = 0ull;
    for (int c0 = 0; c0 < a.ncomp; c0 += 32) {
      const int c = c0 + lane;
      bool ov = false;
      if (c < a.ncomp) {
        const GridComp &g = s_g[c];
        ov = wlo[0] <= g.hi[0] && whi[0] >= g.lo[0] && wlo[1] <= g.hi[1] && whi[1] >= g.lo[1] && wlo[2] <= g.hi[2] &&
             whi[2] >= g.lo[2];
      }
      met |= (unsigned long long)__ballot_sync(0xffffffffu, ov) << c0;
    }
    uint32_t ev = 0, coh = 0;  // crossing tests, points decided by their cell alone (whole warp)
    uint32_t own = 0;          // compartments with points decided by their own crossings
    unsigned long long todo = met;
    int r_done = 0;            // rows below r_done have their Omega written
    while (todo) {
      const int r = __ffsll((long long)todo) - 1;
      todo &= todo - 1;
      const GridComp &g = s_g[r];
      bool in[kGlP], mixed[kGlP], unc[kGlP], inside[kGlP];
      uint32_t word[kGlP], m[kGlP];
      int k[kGlP];
#pragma unroll
      for (int u = 0; u < kGlP; ++u) {
        in[u] = !done[u] && x[u] >= g.lo[0] && x[u] <= g.hi[0] && y[u] >= g.lo[1] && y[u] <= g.hi[1] &&
                z[u] >= g.lo[2] && z[u] <= g.hi[2];
        word[u] = 0u;
        if (in[u]) {
          const int cx = min((int)((x[u] - g.lo[0]) * g.inv[0]), g.n[0] - 1);
          const int cy = min((int)((y[u] - g.lo[1]) * g.inv[1]), g.n[1] - 1);
          const int cz = min((int)((z[u] - g.lo[2]) * g.inv[2]), g.n[2] - 1);
          const int64_t c = ((int64_t)cz * g.n[1] + cy) * g.n[0] + cx;
          if (ZEF_BOUNDS_OK(cx >= 0 && cy >= 0 && cz >= 0 && c < (int64_t)g.n[0] * g.n[1] * g.n[2], a.status, 30))
            word[u] = __ldg(g.words + c);
        }
      }
#pragma unroll
      for (int u = 0; u < kGlP; ++u) {
        mixed[u] = (word[u] & kMixed) != 0u;
        unc[u] = (word[u] & (kMixed | kUnknown)) == kUnknown;
        k[u] = (int)(signed char)(word[u] & 0xffu);
        m[u] = __ballot_sync(0xffffffffu, mixed[u]);
      }
      if (a.stats) {
        bool any_in = false;
#pragma unroll
        for (int u = 0; u < kGlP; ++u) {
          coh += __popc(__ballot_sync(0xffffffffu, in[u] && !mixed[u]));
          any_in |= m[u] != 0u;
        }
        own += any_in ? 1u : 0u;
      }
      for (;;) {
        // next cell: that of the first point left
        uint32_t w0;
        if (m[0]) w0 = __shfl_sync(0xffffffffu, word[0], __ffs(m[0]) - 1);
        else if (m[kGlP - 1]) w0 = __shfl_sync(0xffffffffu, word[kGlP - 1], __ffs(m[kGlP - 1]) - 1);
        else break;
        const GridCell *rec = g.cells + (w0 & ~kMixed);
        const float4 q = __ldg(reinterpret_cast<const float4 *>(rec));      // x, y, z, k
        const int4 l = __ldg(reinterpret_cast<const int4 *>(rec) + 1);      // begin, count
        const int k0 = __float_as_int(q.w);
        uint32_t peers[kGlP];
        float dx[kGlP], dy[kGlP], dz[kGlP];
        int net[kGlP];
        bool open[kGlP];
#pragma unroll
        for (int u = 0; u < kGlP; ++u) {
          peers[u] = __ballot_sync(0xffffffffu, mixed[u] && word[u] == w0);
          m[u] &= ~peers[u];
          dx[u] = x[u] - q.x;
          dy[u] = y[u] - q.y;
          dz[u] = z[u] - q.z;
          net[u] = 0;
          open[u] = k0 == kNoK;
        }
        for (int b = 0; b < l.y; b += 32) {
          const bool act = b + lane < l.y;
          float4 n0 = make_float4(0.f, 0.f, 0.f, 0.f), n1 = n0, n2 = n0;
          if (act) {
            const float4 *t = g.refs + 3 * (int64_t)(l.x + b + lane);
            n0 = __ldg(t);
            n1 = __ldg(t + 1);
            n2 = __ldg(t + 2);
          }
          const float V = n0.w, E = n1.w, EW = 8.f * n1.w;
          const bool vp = act && V > E, vn = act && V < -E;
#pragma unroll
          for (int u = 0; u < kGlP; ++u) {
            uint32_t pp = peers[u];
            while (pp) {
              const int src = __ffs(pp) - 1;
              pp &= pp - 1;
              const float ex = __shfl_sync(0xffffffffu, dx[u], src), ey = __shfl_sync(0xffffffffu, dy[u], src),
                          ez = __shfl_sync(0xffffffffu, dz[u], src);
              const float v0 = fmaf(n0.x, ex, fmaf(n0.y, ey, n0.z * ez));
              const float v1 = fmaf(n1.x, ex, fmaf(n1.y, ey, n1.z * ez));
              const float v2 = fmaf(n2.x, ex, fmaf(n2.y, ey, n2.z * ez));
              const float W = (v0 + v1 + v2) - V;
              const float mn = fminf(v0, fminf(v1, v2)), mx = fmaxf(v0, fmaxf(v1, v2));
              const bool wp = W > EW, wn = W < -EW;
              const bool cross_out = vp && wp && mn > E, cross_in = vn && wn && mx < -E;
              const bool none = (mn < -E && mx > E) || (vn && wp) || (vp && wn) || !act;
              const uint32_t bo = __ballot_sync(0xffffffffu, cross_out), bi = __ballot_sync(0xffffffffu, cross_in);
              const uint32_t bu = __ballot_sync(0xffffffffu, !(none || cross_out || cross_in));
              if (lane == src) {
                net[u] += __popc(bi) - __popc(bo);
                open[u] |= bu != 0u;
              }
            }
          }
        }
#pragma unroll
        for (int u = 0; u < kGlP; ++u) {
          if (mixed[u] && word[u] == w0) {
            k[u] = k0 + net[u];
            unc[u] = open[u];
          }
          if (a.stats) ev += (uint32_t)__popc(peers[u]) * (uint32_t)l.y;
        }
      }
#pragma unroll
      for (int u = 0; u < kGlP; ++u) {
        float om = kFourPi * (float)k[u];
        inside[u] = in[u] && !unc[u] && k[u] >= 1;
        uint32_t um = __ballot_sync(0xffffffffu, unc[u]);
        while (um) {
          const int src = __ffs(um) - 1;
          um &= um - 1;
          float o64;
          const bool i64 = resolve64(a, g, __shfl_sync(0xffffffffu, word[u], src), __shfl_sync(0xffffffffu, x[u], src),
                                     __shfl_sync(0xffffffffu, y[u], src), __shfl_sync(0xffffffffu, z[u], src), lane,
                                     &o64);
          if (lane == src) {
            inside[u] = i64;
            om = o64;
          }
        }
        if (inside[u]) mask[u] |= 1ull << r;
        if (a.omega) {
          const int64_t i = base + 32 * u + lane;
          if (i < n)
            a.omega[(int64_t)r * a.omega_ld + i] = !fin[u] ? __int_as_float(0x7fc00000) : in[u] ? om : 0.f;
        }
        done[u] = done[u] || (a.early && inside[u]);
      }
      if (a.omega) {  // rows of compartments the tile does not meet
        for (int q = r_done; q < r; ++q)
#pragma unroll
          for (int u = 0; u < kGlP; ++u) {
            const int64_t i = base + 32 * u + lane;
            if (i < n) a.omega[(int64_t)q * a.omega_ld + i] = fin[u] ? 0.f : __int_as_float(0x7fc00000);
          }
        r_done = r + 1;
      }
      if (a.early) {
        bool all = true;
#pragma unroll
        for (int u = 0; u < kGlP; ++u) all = all && done[u];
        if (__all_sync(0xffffffffu, all)) break;
      }
    }
    if (a.omega)
      for (int q = r_done; q < a.ncomp; ++q)
#pragma unroll
        for (int u = 0; u < kGlP; ++u) {
          const int64_t i = base + 32 * u + lane;
          if (i < n) a.omega[(int64_t)q * a.omega_ld + i] = fin[u] ? 0.f : __int_as_float(0x7fc00000);
        }
#pragma unroll
    for (int u = 0; u < kGlP; ++u) {
      const int64_t i = base + 32 * u + lane;
      if (i < n) {
        a.labels[off + i] = !fin[u] ? -1 : mask[u] ? __ldg(a.row_ids + (__ffsll((long long)mask[u]) - 1)) : 0;
        if (a.masks) a.masks[off + i] = mask[u];
      }
    }
    if (a.stats) {
      uint32_t nonfin = 0, nin = 0;
#pragma unroll
      for (int u = 0; u < kGlP; ++u) {
        const int64_t i = base + 32 * u + lane;
        nonfin += __popc(__ballot_sync(0xffffffffu, i < n && !fin[u]));
        nin += __popc(__ballot_sync(0xffffffffu, fin[u] && x[u] >= a.ub.lo[0] && x[u] <= a.ub.hi[0] &&
                                                     y[u] >= a.ub.lo[1] && y[u] <= a.ub.hi[1] &&
                                                     z[u] >= a.ub.lo[2] && z[u] <= a.ub.hi[2]));
      }
      if (lane == 0) {
        s_stat[wid][GS_EVAL] += ev;
        s_stat[wid][GS_COHERENT] += coh;
        s_stat[wid][GS_OWN] += own;
        s_stat[wid][GS_ITEMS] += met ? 1 : 0;
        s_stat[wid][GS_NONFINITE] += nonfin;
        s_stat[wid][GS_NIN] += nin;
      }
    }
  }
  if (a.stats) {
    __syncthreads();
    if (threadIdx.x < GS_COUNT) {
      unsigned long long v = 0ull;
      for (int w = 0; w < kGlThreads / 32; ++w) v += s_stat[w][threadIdx.x];
      constexpr int kCnt[GS_COUNT] = {CNT_PAIRS_EVAL, CNT_COHERENT, CNT_LANE_TILES, CNT_ITEMS, CNT_NONFINITE, CNT_NIN};
      if (v) count_add(a, kCnt[threadIdx.x], v);
    }
  }
}

__global__ void k_grid_reset(int64_t *cnt) {
  constexpr int c[] = {CNT_ITEMS, CNT_UNC,      CNT_NONFINITE, CNT_PAIRS_EVAL, CNT_PAIRS_RESCUE,
                       CNT_COHERENT, CNT_REP_PAIRS, CNT_LANE_TILES, CNT_NIN,     CNT_TILES};
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
  if (!grid_opts(o) || ctx->grids.size() != ctx->comps.size()) return false;
  for (const CompGrid &g : ctx->grids)
    if (!g.usable) return false;
  return true;
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
  a.status = ctx->d_status;
  a.comps = ctx->d_comps;
  a.nodes = ctx->d_nodes;
  a.cseg = ctx->d_cseg;
  a.scale = ctx->scale;
  if (plan.timed) cudaEventRecord(ctx->ev[0], s);
  if (a.stats) {
    k_grid_reset<<<1, 32, 0, s>>>(ctx->lb.counters);
    ++ctx->launches;
  }
  NvtxRange nvtx_stage("zef.label_kernel");
  if (plan.timed) cudaEventRecord(ctx->ev[1], s);
  const int per_block = kGlThreads / 32 * kGlTile;
  const int64_t blocks = std::min<int64_t>((plan.n_cap + per_block - 1) / per_block, (int64_t)ctx->num_sms * 32);
  k_grid_label<<<(unsigned)std::max<int64_t>(blocks, 1), kGlThreads, 0, s>>>(a);
  ++ctx->launches;
  if (plan.timed) {
    cudaEventRecord(ctx->ev[2], s);
    cudaEventRecord(ctx->ev[3], s);
    cudaEventRecord(ctx->ev[4], s);
    cudaEventRecord(ctx->ev[5], s);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(ctx, e, "k_grid_label launch");
  return ZEF_OK;
}

void grid_free(zef_ctx *ctx) {
  for (CompGrid &g : ctx->grids)
    if (g.blob) cudaFree(g.blob);
  ctx->grids.clear();
  if (ctx->d_grid) cudaFree(ctx->d_grid);
  ctx->d_grid = nullptr;
}

// Cell grid of compartment c (uploaded, with its cap tree).  Cells are two
// mean triangle edges wide (a cell then lists about a dozen triangles, which
// one warp holds at once, and about 1.5 cells per crossed cell face area are
// mixed), at least eight along the longest side, at most kMaxCells in all.
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
  double w = 2.0 * std::sqrt(h.area / (0.43 * (double)h.nt));
  w = std::min(w, (double)longest / 8.0);
  w = std::max(w, (double)longest / kMaxAxis);
  Geom g;
  int64_t cells = 0;
  for (;; w *= 1.1) {
    cells = 1;
    for (int k = 0; k < 3; ++k) {
      g.n[k] = (int)std::min<double>(kMaxAxis, std::max(1.0, std::ceil(ext[k] / w)));
      cells *= g.n[k];
    }
    if (cells <= kMaxCells) break;
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

  // scratch: counts / list ends, record numbers, block sums, two totals, anchors, their Omega
  const int64_t bs = cells / 2048 + 2;
  const size_t o_flag = (size_t)cells * 4, o_sum = o_flag + (size_t)cells * 4, o_tot = (o_sum + (size_t)bs * 4 + 15) & ~(size_t)15,
               o_anch = o_tot + 32, o_om = o_anch + (size_t)cells * 12, bytes = o_om + (size_t)cells * 4;
  unsigned char *tmp = nullptr;
  auto no_memory = [&](cudaError_t e) {
    cudaGetLastError();
    if (tmp) cudaFree(tmp);
    return e == cudaErrorMemoryAllocation ? ZEF_OK : cuda_fail(ctx, e, "cell grid");
  };
  cudaError_t e = cudaMalloc(&tmp, bytes);
  if (e != cudaSuccess) return no_memory(e);
  uint32_t *cnt = (uint32_t *)tmp, *flag = (uint32_t *)(tmp + o_flag), *bsum = (uint32_t *)(tmp + o_sum);
  int64_t *tot = (int64_t *)(tmp + o_tot);
  float *anchor = (float *)(tmp + o_anch), *omega = (float *)(tmp + o_om);
  cudaMemsetAsync(cnt, 0, (size_t)cells * 4, st);
  cudaMemsetAsync(tot, 0, 32, st);
  const int g_t = grid_blocks(ctx, (int64_t)nt * 32, 256), g_c = grid_blocks(ctx, cells, 256),
            g_w = grid_blocks(ctx, cells * 32, 256);
  k_gr_refs<<<g_t, 256, 0, st>>>(tris, to_raw, nt, g, cnt, nullptr);
  k_gr_flags<<<g_c, 256, 0, st>>>(cnt, cells, flag, (unsigned long long *)(tot + 2));
  zef_status zs = scan_exclusive(ctx, cnt, nullptr, 1, cells, tot, bsum);
  if (!zs) zs = scan_exclusive(ctx, flag, nullptr, 1, cells, tot + 1, bsum);
  int64_t totals[3] = {0, 0, 0};
  if (!zs) {
    e = cudaMemcpyAsync(totals, tot, sizeof(totals), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) zs = cuda_fail(ctx, e, "cell grid");
  }
  if (zs) {
    cudaFree(tmp);
    return zs;
  }
  const int64_t refs = totals[0], mixed = totals[1];
  if (totals[2] > kMaxList || refs > 64 * (int64_t)nt + 65536) {
    cudaFree(tmp);
    return ZEF_OK;
  }
  // stored products, records, words, triangle indices
  const size_t p_cell = (size_t)refs * 48, p_word = p_cell + (size_t)mixed * sizeof(GridCell),
               p_tri = p_word + (size_t)cells * 4, p_end = p_tri + (size_t)refs * 4;
  unsigned char *blob = nullptr;
  e = cudaMalloc(&blob, p_end);
  if (e != cudaSuccess) return no_memory(e);
  int32_t *list = (int32_t *)(blob + p_tri);
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
    cudaFree(tmp);
    if (zs != ZEF_ERR_OOM) return zs;
    cudaGetLastError();
    return ZEF_OK;
  }
  k_gr_finish<<<g_w, 256, 0, st>>>(tris, to_raw, s, g, cells, cnt, flag, list, anchor, omega, (uint32_t *)(blob + p_word),
                                   (GridCell *)(blob + p_cell), (float4 *)blob);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  cudaFree(tmp);
  if (e != cudaSuccess) {
    cudaFree(blob);
    return cuda_fail(ctx, e, "cell grid");
  }
  gr.blob = blob;
  gr.usable = true;
  gr.words = (const uint32_t *)(blob + p_word);
  gr.cells = (const GridCell *)(blob + p_cell);
  gr.refs = (const float4 *)blob;
  gr.tri = list;
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
  while (ctx->grids.size() < C) {
    CompGrid g;
    zef_status st = grid_build(ctx, ctx->grids.size(), &g);
    if (st) return st;
    ctx->grids.push_back(g);
  }
  if (!ctx->d_grid) CK(cudaMalloc(&ctx->d_grid, ZEF_MAX_COMPARTMENTS * sizeof(GridComp)), "cudaMalloc(cell grids)");
  std::vector<GridComp> d(C);
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
    r.cells = g.cells;
    r.refs = g.refs;
    r.tri = g.tri;
    r.tris = ctx->d_tris + h.tri_off * 3;
  }
  CK(cudaMemcpy(ctx->d_grid, d.data(), C * sizeof(GridComp), cudaMemcpyHostToDevice), "upload cell grids");
  return ZEF_OK;
}

}  // namespace zef
