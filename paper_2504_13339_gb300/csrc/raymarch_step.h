// Where a ray's samples lie in the volume's grid, and how many of them lie in
// one macrocell: the arithmetic of the march over empty space, for the host as
// well as the device.
#pragma once

#include <cmath>
#include <cstdint>

#ifdef __CUDACC__
#define VEG_HD __host__ __device__ __forceinline__
#else
#define VEG_HD inline
#endif

namespace veg {

struct MarchRay {
  float eye[3], d[3];  // origin, unit direction
  float ta;            // where it enters the volume
  float step, inv_h;   // sample spacing; vertex cells per unit length
  int R;               // vertices per axis
};

// Sample k: its place g in vertex cells and the cell ic that holds it (both
// monotone in k on every axis, rounding included).  Returns its distance t.
VEG_HD float march_place(const MarchRay& r, int k, float g[3], int ic[3]) {
  const float t = fmaf((float)k + 0.5f, r.step, r.ta);
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) {
    g[c] = (fmaf(t, r.d[c], r.eye[c]) + 1.0f) * r.inv_h;
    const int i = (int)floorf(g[c]);
    ic[c] = i < 0 ? 0 : i > r.R - 2 ? r.R - 2 : i;
  }
  return t;
}

// A macrocell's place in the mask (2047^3 of them at the largest volume's
// single cells).
VEG_HD int64_t march_macrocell(const int m[3], int cells) {
  return ((int64_t)m[2] * cells + m[1]) * cells + m[0];
}

// How far, in vertex cells, a sample may lie from where its distance to the
// one at t says.  Both distances, at most |t| and the volume's diagonal, are
// rounded to 2^-24 of that, the points to 2^-24 of at most 1 and their sums
// with 1 to 2^-24 of at most 2, each times inv_h; twice that, and 1/64 cell for
// the rest (rates and products are good to 2^-22 of the 64 cells of the widest
// macrocell; a sample number beyond 2^23 is rounded by less than 2^-23 of the
// ray).
VEG_HD float march_margin(const MarchRay& r, float t) {
  return 0.015625f + r.inv_h * 2.384185791015625e-07f * (fabsf(t) + 8.0f);
}

// Samples per vertex cell along each axis.
VEG_HD void march_rates(const MarchRay& r, float rate[3]) {
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) rate[c] = 1.0f / (r.d[c] * r.inv_h * r.step);
}

// The first of n samples that may lie beyond macrocell m of 2^shift vertex
// cells per axis, sample k at distance t and place g being inside: one that surely lies inside
// (march_margin short of the far faces), and with it all before it, is passed
// over.
VEG_HD int march_next(const MarchRay& r, int k, int n, float t, const float g[3], const int m[3],
                      int shift, const float rate[3]) {
  const float margin = march_margin(r, t);
  float s = 1.0e6f;
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) {
    const float face = (float)((rate[c] > 0.0f ? m[c] + 1 : m[c]) << shift);
    const float ahead = (face - g[c]) * rate[c] - fabsf(rate[c]) * margin;
    if (r.d[c] != 0.0f) s = fminf(s, ahead);
  }
  const int next = k + 1 + (int)fmaxf(s, 0.0f);
  return next < n ? next : n;
}

}  // namespace veg
