// FP64 solid angle of a group of cap-tree segment entries, shared by the
// re-evaluation kernels of zef_label.cu and the cell-grid kernel of
// zef_grid.cu.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "zef_internal.h"

namespace zef {

// FP64 strip evaluation of one group of four cap-tree segment entries
// (positions pos .. pos + 3, a multiple of four: a group never straddles two
// segments) seen from p: the window enters the group as (E[pos-2], E[pos-1])
// (both in the same segment, since a segment starts at a multiple of four
// with its reset entry) or restarts at a reset entry; every window that is a
// triangle contributes the factor D + iN with N = w R_a . (R_b x R_c) (w the
// entry's orientation sign, the exact triple product of the stored
// vertices) and D = r_a r_b r_c + (R_a . R_b) r_c + (R_a . R_c) r_b +
// (R_b . R_c) r_a (Sec. 2.1.3), and the group returns the argument of the
// product with the 2 pi wraps of the partial products counted in *K exactly
// as the FP32 kernel does.
__device__ __forceinline__ bool sign64(double x) { return __double_as_longlong(x) < 0; }

static __device__ double group64(const Entry *E, int pos, double px, double py, double pz, int *K) {
  double a[3], b[3], ra, rb;
  const float4 v0 = E[pos].v;
  if (v0.w == 2.f) {
    a[0] = b[0] = (double)v0.x - px;
    a[1] = b[1] = (double)v0.y - py;
    a[2] = b[2] = (double)v0.z - pz;
    ra = rb = sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
  } else {
    const float4 u = E[pos - 2].v, w = E[pos - 1].v;
    a[0] = (double)u.x - px; a[1] = (double)u.y - py; a[2] = (double)u.z - pz;
    b[0] = (double)w.x - px; b[1] = (double)w.y - py; b[2] = (double)w.z - pz;
    ra = sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
    rb = sqrt(b[0] * b[0] + b[1] * b[1] + b[2] * b[2]);
  }
  double R = 1.0, I = 0.0;
  bool have = false;
  int k = 0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float4 v = E[pos + q].v;
    const double c[3] = {(double)v.x - px, (double)v.y - py, (double)v.z - pz};
    const double rc = sqrt(c[0] * c[0] + c[1] * c[1] + c[2] * c[2]);
    if (fabsf(v.w) == 1.f) {
      const double N = (double)v.w * (a[0] * (b[1] * c[2] - b[2] * c[1]) + a[1] * (b[2] * c[0] - b[0] * c[2]) +
                                      a[2] * (b[0] * c[1] - b[1] * c[0]));
      const double dab = a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
      const double dac = a[0] * c[0] + a[1] * c[1] + a[2] * c[2];
      const double dbc = b[0] * c[0] + b[1] * c[1] + b[2] * c[2];
      const double D = ra * rb * rc + dab * rc + dac * rb + dbc * ra;
      if (!have) {
        R = D;
        I = N;
        have = true;
      } else {
        const double cr = R * D - I * N, ci = R * N + I * D;
        k += (!sign64(I) && !sign64(N) && sign64(ci)) ? 1 : 0;
        k -= (sign64(I) && sign64(N) && !sign64(ci)) ? 1 : 0;
        R = cr;
        I = ci;
      }
    }
    a[0] = b[0]; a[1] = b[1]; a[2] = b[2];
    b[0] = c[0]; b[1] = c[1]; b[2] = c[2];
    ra = rb;
    rb = rc;
  }
  *K += k;
  return have ? atan2(I, R) : 0.0;
}

}  // namespace zef
