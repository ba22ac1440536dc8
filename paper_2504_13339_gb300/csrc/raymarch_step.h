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
// monotone in k on every axis, rounding included).
VEG_HD void march_place(const MarchRay& r, int k, float g[3], int ic[3]) {
  const float t = fmaf((float)k + 0.5f, r.step, r.ta);
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) {
    g[c] = (fmaf(t, r.d[c], r.eye[c]) + 1.0f) * r.inv_h;
    const int i = (int)floorf(g[c]);
    ic[c] = i < 0 ? 0 : i > r.R - 2 ? r.R - 2 : i;
  }
}

// A macrocell's place in the mask (2047^3 of them at the largest volume's
// single cells).
VEG_HD int64_t march_macrocell(const int m[3], int cells) {
  return (int64_t)(m[2] * cells + m[1]) * cells + m[0];  // the row fits 32 bits
}

// How far, in vertex cells, one of a ray's n samples may lie from where its
// distance to another says.  t is rounded to 2^-24 |t|, the point to 2^-24 of at
// most 1 and its sum with 1 to 2^-24 of at most 2, each times inv_h, at both
// ends of a step; twice that, and 1/64 cell for the rest (rates and products are
// good to 2^-22 of the 64 cells of the widest macrocell; a sample number beyond
// 2^23 is rounded by less than 2^-23 of the ray).
VEG_HD float march_margin(const MarchRay& r, int n) {
  const float far = fabsf(r.ta) + (float)n * r.step;  // at least every |t|
  return 0.015625f + r.inv_h * 2.384185791015625e-07f * (far + 4.0f);
}

// Per axis: samples per vertex cell, and the last place that is surely in a
// macrocell of 2^shift vertex cells (the margin short of its far face), from its
// lowest vertex.
struct MarchStep {
  float rate[3], last[3];
};
VEG_HD MarchStep march_step(const MarchRay& r, int n, int shift) {
  MarchStep s;
  const float margin = march_margin(r, n);
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) {
    s.rate[c] = 1.0f / (r.d[c] * r.inv_h * r.step);
    s.last[c] = s.rate[c] > 0.0f ? (float)(1 << shift) - margin : margin;
  }
  return s;
}

// The first of n samples that may lie beyond macrocell m of 2^shift vertex
// cells per axis, sample k at g being inside: the last one that surely lies
// inside, and with it all before it, is passed over.
VEG_HD int march_next(const MarchRay& r, const MarchStep& s, int k, int n, const float g[3],
                      const int m[3], int shift) {
  float least = 1.0e6f;
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int c = 0; c < 3; ++c) {
    const float ahead = ((float)(m[c] << shift) + s.last[c] - g[c]) * s.rate[c];
    if (r.d[c] != 0.0f) least = fminf(least, ahead);
  }
  const int next = k + 1 + (int)fmaxf(least, 0.0f);
  return next < n ? next : n;
}

}  // namespace veg
