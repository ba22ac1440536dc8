// Emission-absorption raymarching of a gridded scalar volume: the renderer
// of the paper's training images (Sec. 4.2, 5.1: the volume is raymarched
// with an emission-absorption model and shaded with Blinn-Phong lighting
// from a headlight).
//
// Volume: R^3 vertices on [-1,1]^3 (x fastest), prepared once as float4
// (value, d/dx, d/dy, d/dz) with central-difference vertex gradients
// (one-sided on the boundary), so one sample is eight float4 loads and a
// trilinear blend of value and gradient together.
//
// Per ray (one thread per pixel, 16 x 16 pixels per CTA): the camera ray is
// clipped to the box and to the near plane; samples sit at t0 + (k + 1/2)
// Delta; each sample's transfer-function colour and opacity give alpha =
// 1 - (1 - A)^(Delta / h), the colour is Blinn-Phong shaded with the
// interpolated gradient (ambient only where it vanishes), and the samples are
// composited front to back until every table of the CTA's group has T < 1e-4.
#include <algorithm>
#include <cmath>

#include "raymarch_step.h"
#include "veg_internal.cuh"

namespace veg {

namespace {

// Hardware approximations of 2^x and log2 x (the opacity correction), whose
// errors stay far below the image tolerance.
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

struct RayView {
  float r[9];      // world-to-camera rotation, row-major
  float eye[3];    // camera centre
  float light[3];  // headlight direction (toward the light)
  float fx, fy, cx, cy, near_plane;
};

struct RaySet {
  RayView v[VEG_MAX_VIEWS];
};

struct MarchArgs {
  const float4* vol;
  int R;
  float inv_h, step, ratio;  // ratio = step / h
  const float4* lut;
  int lut_size, n_tf;
  int group;  // tables per group
  const int32_t* view_tf;
  int width, height, tiles_x, tiles_per_view;
  float ka, kd, ks, beta;
  bool leave_out;  // tables without opacity (every factor of them is finite)
  float bg0, bg1, bg2;
  // empty-space skipping: per-macrocell table masks (veg_raymarch_cells)
  // over macrocells of 2^cell_shift vertex cells per axis, or null
  const uint32_t* cell_mask;
  int cell_shift, cells;
};

__global__ void __launch_bounds__(256)
    volume_prepare_kernel(const float* __restrict__ vol, int R, float inv_h,
                          float4* __restrict__ out) {
  pdl_enter();
  const int64_t n = (int64_t)R * R * R;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int x = (int)(i % R), y = (int)((i / R) % R), z = (int)(i / ((int64_t)R * R));
  const int64_t sx = 1, sy = R, sz = (int64_t)R * R;
  auto diff = [&](int c, int64_t s) {
    if (c == 0) return (vol[i + s] - vol[i]) * inv_h;
    if (c == R - 1) return (vol[i] - vol[i - s]) * inv_h;
    return (vol[i + s] - vol[i - s]) * (0.5f * inv_h);
  };
  out[i] = make_float4(vol[i], diff(x, sx), diff(y, sy), diff(z, sz));
}

// Per macrocell (cell^3 vertex cells, vertices [c cell, c cell + cell] per
// axis clipped to the grid): bit t (t < 32) set when table t can give a
// sample in the cell a nonzero opacity.  A sample's value is a trilinear
// blend of the cell's vertex values, so it lies in their [min, max] up to
// rounding; the test widens the range by 1e-6 and takes the table entries
// that values in it interpolate between, with one more entry on each side,
// and sets the bit when any of them has a positive opacity (interpolating
// two non-positive entries gives a clamped opacity of 0).  A NaN vertex, or
// more than 32 tables, sets every bit.
// G lanes per macrocell, over its vertices (x fastest, so that neighbouring
// lanes read neighbouring vertices), then over the tables: a lane each where
// macrocells are small and many, a warp where they are large, eight lanes
// between.  256^3 vertices (268 MB) under two tables, 1, 8 and 32 lanes: single
// cells 234, 1394 and 4726 us, 4^3 cells 68, 117 and 158, 8^3 101, 66 and 73, 16^3
// 621, 157 and 90; 64^3 vertices in 4^3 cells (4096 macrocells) 14, 8 and 8.
template <int G>
__global__ void __launch_bounds__(256)
    cell_mask_kernel(const float4* __restrict__ vol, int R, int cell, int cells,
                     const float4* __restrict__ lut, int L, int n_tf, uint32_t* __restrict__ mask) {
  pdl_enter();
  const int lane = threadIdx.x & (G - 1);
  const int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) / G;
  const int64_t nc = (int64_t)cells * cells * cells;
  if (i >= nc) return;  // uniform over a macrocell's lanes
  const unsigned mine = G == 32 ? 0xffffffffu
                                : ((1u << (G & 31)) - 1u) << (threadIdx.x & 31 & ~(G - 1));
  const int cx = (int)(i % cells), cy = (int)((i / cells) % cells),
            cz = (int)(i / ((int64_t)cells * cells));
  const int x0 = cx * cell, y0 = cy * cell, z0 = cz * cell;
  const int x1 = min(x0 + cell, R - 1), y1 = min(y0 + cell, R - 1), z1 = min(z0 + cell, R - 1);
  float mn = 3.0e38f, mx = -3.0e38f;
  bool nan = false;
  auto see = [&](float v) {
    nan |= v != v;
    mn = fminf(mn, v);
    mx = fmaxf(mx, v);
  };
  if (G == 1) {
    for (int z = z0; z <= z1; ++z)
      for (int y = y0; y <= y1; ++y)
        for (int x = x0; x <= x1; ++x) see(__ldg(&vol[((int64_t)z * R + y) * R + x]).x);
  } else {
    const int nx = x1 - x0 + 1, ny = y1 - y0 + 1, nv = nx * ny * (z1 - z0 + 1);
#pragma unroll 8
    for (int e = lane; e < nv; e += G) {
      const int row = e / nx, x = e - row * nx, z = row / ny, y = row - z * ny;
      see(__ldg(&vol[((int64_t)(z0 + z) * R + y0 + y) * R + x0 + x].x));
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      nan |= __shfl_xor_sync(mine, (int)nan, o) != 0;
      mn = fminf(mn, __shfl_xor_sync(mine, mn, o));
      mx = fmaxf(mx, __shfl_xor_sync(mine, mx, o));
    }
  }
  uint32_t m = 0xffffffffu;
  if (!nan && n_tf <= 32) {
    const float lo = fminf(fmaxf(mn - 1e-6f, 0.0f), 1.0f) * (float)(L - 1);
    const float hi = fminf(fmaxf(mx + 1e-6f, 0.0f), 1.0f) * (float)(L - 1);
    const int k0 = max((int)floorf(lo) - 1, 0), k1 = min((int)floorf(hi) + 2, L - 1);
    m = 0u;
    for (int t = G == 1 ? 0 : lane; t < n_tf; t += G)
      for (int k = k0; k <= k1; ++k)
        if (__ldg(&lut[(int64_t)t * L + k].w) > 0.0f) {
          m |= 1u << t;
          break;
        }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) m |= __shfl_xor_sync(mine, m, o);
  }
  if (lane == 0) mask[i] = m;
}

// (a, b) -> a + f (b - a) of two components at a time, each half rounded like
// the scalar subtraction and fused multiply-add.
struct Sample {
  float2 vx, yz;  // value, d/dx; d/dy, d/dz
};
__device__ __forceinline__ Sample lerp_sample(Sample a, Sample b, float f) {
  const float2 ff = make_float2(f, f);
  return Sample{fma2(ff, sub2(b.vx, a.vx), a.vx), fma2(ff, sub2(b.yz, a.yz), a.yz)};
}
__device__ __forceinline__ Sample load_sample(const float4* p) {
  const float4 v = __ldg(p);
  return Sample{make_float2(v.x, v.y), make_float2(v.z, v.w)};
}

// What bounds the march is instruction issue and the latency of a sample's
// chain (ncu: 58% of the issue slots at three CTAs per SM), so a ray does as
// little as it can: one group marches up to 16 tables (each group takes the
// samples again); a run of samples in an empty macrocell is one step, to the
// last sample that surely lies in it (raymarch_step.h); and a sample evaluates
// only the tables that have some opacity at its place (a bit per table and
// entry), each lane its own next one.  The tables'
// transmittances and colours are kept in shared memory: as registers they
// held the kernel at two CTAs per SM, and every table was a branch of every
// sample.  Ten opacity maps over a 256^3 volume, three 800x800 views (with the
// macrocells' masks): 6300 us in groups of eight with every sample visited and
// every table evaluated, 4330 with the steps, bits and registers, 3430 so.  Without a material
// (SHADE false) only the value is read and blended: ten tables over 64^3
// vertices, one 400x300 view, 357 us (371 in the groups of eight, 409 with the
// whole blend), one table 99 (194).
//
// stats (instrumented build): samples taken (per ray and table group),
// table evaluations and, with a cell mask, samples skipped as empty.
template <bool MANY, bool STATS, bool SHADE>
__global__ void __launch_bounds__(256, 3)
    raymarch_kernel(MarchArgs A, const __grid_constant__ RaySet rs, float4* __restrict__ out,
                    unsigned long long* __restrict__ stats) {
  pdl_enter();
  unsigned long long n_samp = 0, n_tab = 0, n_skip = 0;
  // MANY: transmittance and colour of each (table, pixel) [group][256], then
  // the mask of tables per entry [L]
  extern __shared__ float4 s_acc[];
  const int wi = blockIdx.x;
  // tile rows from the middle of the image outwards: the rays through the
  // volume's middle are the longest, and a launch ends with short ones
  const int view = wi / A.tiles_per_view, at = wi - view * A.tiles_per_view;
  const int rows = A.tiles_per_view / A.tiles_x, r = at / A.tiles_x;
  const int row = r & 1 ? (rows >> 1) - ((r + 1) >> 1) : (rows >> 1) + (r >> 1);
  const int tile = row * A.tiles_x + at - r * A.tiles_x;
  const int t0g = blockIdx.z * A.group;
  const int lut0 = A.view_tf ? A.view_tf[view] : t0g;
  const int ntg = A.view_tf ? 1 : min(A.group, A.n_tf - t0g);
  const int n_out = A.view_tf ? 1 : A.n_tf;
  const int L = A.lut_size;
  unsigned* s_any = reinterpret_cast<unsigned*>(s_acc + (MANY ? A.group * 256 : 0));
  const bool known = lut0 >= 0 && lut0 < A.n_tf;  // else the transparent table
  const float4* lut = A.lut + (known ? (int64_t)lut0 * L : 0);
  // A table is left out between entries k and k + 1 where it adds exactly
  // nothing: neither opacity is positive (the interpolated one clamps to 0)
  // and the colours are far from infinite (0 times them, shaded, is 0).
  for (int k = threadIdx.x; k < L; k += blockDim.x) {
    unsigned m = 0u;
    for (int t = 0; known && t < ntg; ++t) {
      const float4 lo = __ldg(&lut[t * L + k]), hi = __ldg(&lut[t * L + min(k + 1, L - 1)]);
      const float big =
          fmaxf(fmaxf(fmaxf(fabsf(lo.x), fabsf(lo.y)), fmaxf(fabsf(lo.z), fabsf(hi.x))),
                fmaxf(fabsf(hi.y), fabsf(hi.z)));
      const float sum = lo.x + lo.y + lo.z + hi.x + hi.y + hi.z;  // NaN of any entry stays
      if (lo.w > 0.0f || hi.w > 0.0f || !(big <= 1.0e30f) || sum != sum) m |= 1u << t;
    }
    s_any[k] = m;
  }
  __syncthreads();
  // a warp holds 8x4 pixels
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int px = (tile % A.tiles_x) * VEG_TILE + (warp & 1) * 8 + (lane & 7);
  const int py = (tile / A.tiles_x) * VEG_TILE + (warp >> 1) * 4 + (lane >> 3);
  const bool inside = px < A.width && py < A.height;
  if (!STATS && !inside) return;
  if (inside) {
  const RayView& V = rs.v[view];
  // ray direction R^T ((px - cx)/fx, (py - cy)/fy, 1), normalised
  const float ux = (px - V.cx) / V.fx, uy = (py - V.cy) / V.fy;
  float d[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) d[c] = V.r[c] * ux + V.r[3 + c] * uy + V.r[6 + c];
  const float inv_len = rsqrtf(d[0] * d[0] + d[1] * d[1] + d[2] * d[2]);
#pragma unroll
  for (int c = 0; c < 3; ++c) d[c] *= inv_len;
  // slab clip against [-1,1]^3 and t >= near
  float ta = V.near_plane, tb = 3.0e38f;
  bool hit = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if (d[c] == 0.0f) {
      if (fabsf(V.eye[c]) > 1.0f) hit = false;
      continue;
    }
    const float inv = 1.0f / d[c];
    const float t1 = (-1.0f - V.eye[c]) * inv, t2 = (1.0f - V.eye[c]) * inv;
    ta = fmaxf(ta, fminf(t1, t2));
    tb = fminf(tb, fmaxf(t1, t2));
  }
  float4* acc = s_acc + threadIdx.x;            // (T, r, g, b) of table t at acc[256 t]
  float4 one = make_float4(1.f, 0.f, 0.f, 0.f);  // of a single table
  if (MANY)
    for (int t = 0; t < ntg; ++t) acc[256 * t] = one;
  unsigned live = (1u << ntg) - 1u;
  if (hit && tb > ta) {
    const int n = (int)floorf((tb - ta) / A.step);
    // half vector of the view direction e = -d and the headlight
    float hv[3];
    float hn = 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      hv[c] = V.light[c] - d[c];
      hn += hv[c] * hv[c];
    }
    hn = hn > 0.f ? rsqrtf(hn) : 0.f;
#pragma unroll
    for (int c = 0; c < 3; ++c) hv[c] *= hn;
    const int R = A.R;
    // the group's tables occupy bits lut0 .. lut0 + ntg - 1 of a cell mask
    const bool skip_empty = A.cell_mask != nullptr && lut0 >= 0 && lut0 + ntg <= 32;
    MarchRay ray;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ray.eye[c] = V.eye[c];
      ray.d[c] = d[c];
    }
    ray.ta = ta;
    ray.step = A.step;
    ray.inv_h = A.inv_h;
    ray.R = R;
    const MarchStep over = march_step(ray, n, A.cell_shift);
    for (int k = 0; live; ++k) {
      float g[3];
      int ic[3];
      // the next sample that a table still compositing can see
      for (; k < n;) {
        march_place(ray, k, g, ic);
        if (!skip_empty) break;
        const int m[3] = {ic[0] >> A.cell_shift, ic[1] >> A.cell_shift, ic[2] >> A.cell_shift};
        if (((__ldg(&A.cell_mask[march_macrocell(m, A.cells)]) >> lut0) & live) != 0u) break;
        // Every table still compositing has zero opacity in this macrocell:
        // its samples would leave colour and transmittance unchanged.
        const int next = march_next(ray, over, k, n, g, m, A.cell_shift);
        if (STATS) n_skip += (unsigned)(next - k);
        k = next;
      }
      if (k >= n) break;
#pragma unroll
      for (int c = 0; c < 3; ++c) g[c] -= (float)ic[c];
      const float4* base = A.vol + ((int64_t)ic[2] * R + ic[1]) * R + ic[0];
      const int64_t sy = R, sz = (int64_t)R * R;
      float sd = 1.0f, ss = 0.0f;
      unsigned on;
      TfPos q;
      if (SHADE) {
        const Sample c00 = lerp_sample(load_sample(base), load_sample(base + 1), g[0]);
        const Sample c01 = lerp_sample(load_sample(base + sy), load_sample(base + sy + 1), g[0]);
        const Sample c10 = lerp_sample(load_sample(base + sz), load_sample(base + sz + 1), g[0]);
        const Sample c11 =
            lerp_sample(load_sample(base + sz + sy), load_sample(base + sz + sy + 1), g[0]);
        const Sample sm =
            lerp_sample(lerp_sample(c00, c01, g[1]), lerp_sample(c10, c11, g[1]), g[2]);
        const float sx = sm.vx.y, sy_ = sm.yz.x, sz_ = sm.yz.y;
        q = tf_pos(sm.vx.x, L);
        // the largest gradient component; a gradient that is not finite makes
        // a NaN colour under any table, so no table is left out
        const float m = fmaxf(fmaxf(fabsf(sx), fabsf(sy_)), fabsf(sz_));
        const float chk = sx * 0.0f + sy_ * 0.0f + sz_ * 0.0f;
        on = A.leave_out && chk == 0.0f ? s_any[q.k] & live : live;
        // normal = -gradient / |gradient|; scaled by the largest component
        // first so that tiny gradients cannot underflow
        sd = A.ka;
        if (on != 0u && m > 0.0f) {
          const float gx = sx / m, gy = sy_ / m, gz = sz_ / m;
          const float ig = rsqrtf(gx * gx + gy * gy + gz * gz);
          const float nl = fabsf((gx * V.light[0] + gy * V.light[1] + gz * V.light[2]) * ig);
          const float nh = fabsf((gx * hv[0] + gy * hv[1] + gz * hv[2]) * ig);
          sd = A.ka + A.kd * nl;
          ss = nl > 0.f ? A.ks * __powf(nh, A.beta) : 0.f;
        }
      } else {  // the value alone
        auto along = [&](const float4* p) {
          const float a = __ldg(&p[0].x), b = __ldg(&p[1].x);
          return fmaf(g[0], b - a, a);
        };
        const float c00 = along(base), c01 = along(base + sy), c10 = along(base + sz),
                    c11 = along(base + sz + sy);
        const float c0 = fmaf(g[1], c01 - c00, c00), c1 = fmaf(g[1], c11 - c10, c10);
        q = tf_pos(fmaf(g[2], c1 - c0, c0), L);
        on = s_any[q.k] & live;
      }
      if (STATS) {
        ++n_samp;
        n_tab += (unsigned)__popc(on);
      }
      if (on == 0u) continue;
      // each lane its own next table: a step serves lanes at different ones
      for (unsigned left = on; left != 0u; left &= left - 1u) {
        const int tt = MANY ? __ffs((int)left) - 1 : 0;
        const float4 lo = known ? __ldg(&lut[tt * L + q.k]) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 hi = known ? __ldg(&lut[tt * L + q.k + 1]) : lo;
        float4 p = MANY ? acc[256 * tt] : one;
        const float a = fminf(fmaxf(lerp_rn(lo.w, hi.w, q), 0.0f), 1.0f);
        const float alpha = a > 0.0f ? 1.0f - ex2_approx(lg2_approx(1.0f - a) * A.ratio) : 0.0f;
        const float w = p.x * alpha;
        p.y = fmaf(w, fmaf(sd, lerp_rn(lo.x, hi.x, q), ss), p.y);
        p.z = fmaf(w, fmaf(sd, lerp_rn(lo.y, hi.y, q), ss), p.z);
        p.w = fmaf(w, fmaf(sd, lerp_rn(lo.z, hi.z, q), ss), p.w);
        p.x *= 1.0f - alpha;
        if (p.x < kTMin) live &= ~(1u << tt);
        if (MANY)
          acc[256 * tt] = p;
        else
          one = p;
      }
    }
  }
  for (int tt = 0; tt < ntg; ++tt) {
    const int64_t o = (((int64_t)view * n_out + t0g + tt) * A.height + py) * A.width + px;
    const float4 p = MANY ? acc[256 * tt] : one;
    out[o] = make_float4(fmaf(p.x, A.bg0, p.y), fmaf(p.x, A.bg1, p.z), fmaf(p.x, A.bg2, p.w), p.x);
  }
  }
  if (STATS) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      n_samp += __shfl_down_sync(0xffffffffu, n_samp, o);
      n_tab += __shfl_down_sync(0xffffffffu, n_tab, o);
      n_skip += __shfl_down_sync(0xffffffffu, n_skip, o);
    }
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(&stats[0], n_samp);
      atomicAdd(&stats[1], n_tab);
      if (A.cell_mask) atomicAdd(&stats[2], n_skip);
    }
  }
}

// Tables per group: their transmittances and colours take 4 KB of a CTA's
// shared memory each (three CTAs per SM hold 16).
constexpr int kMarchTables = 16;

template <bool MANY, bool STATS, bool SHADE>
veg_status launch_march(const MarchArgs& A, const RaySet& rs, int n_views, float4* out,
                        unsigned long long* stats, cudaStream_t stream) {
  const size_t smem = (MANY ? (size_t)A.group * 256 * sizeof(float4) : 0) +
                      (size_t)A.lut_size * sizeof(unsigned);
  auto kern = raymarch_kernel<MANY, STATS, SHADE>;
  static SmemRecord configured;  // default carveout: the volume samples want L1
  veg_status st = prepare_smem(kern, smem, configured, false);
  if (st != VEG_OK) return st;
  const unsigned groups = A.view_tf ? 1u : (unsigned)((A.n_tf + A.group - 1) / A.group);
  dim3 grid((unsigned)(A.tiles_per_view * n_views), 1u, groups);
  launch_k(kern, grid, 256, smem, stream, A, rs, out, stats);
  count_launch();
  return launch_status();
}

template <bool MANY, bool SHADE>
veg_status launch_march_s(const MarchArgs& A, const RaySet& rs, int n_views, float4* out,
                          unsigned long long* stats, cudaStream_t stream) {
  return stats ? launch_march<MANY, true, SHADE>(A, rs, n_views, out, stats, stream)
               : launch_march<MANY, false, SHADE>(A, rs, n_views, out, nullptr, stream);
}

}  // namespace

}  // namespace veg

using namespace veg;

extern "C" veg_status veg_volume_prepare(const float* volume, int32_t resolution, float* vol4,
                                         cudaStream_t stream) {
  if (!volume || !vol4 || resolution < 2 || resolution > 2048 || !aligned16(vol4))
    return VEG_ERR_INVALID_ARGUMENT;
  const int64_t n = (int64_t)resolution * resolution * resolution;
  const float inv_h = (float)((resolution - 1) / 2.0);
  launch_k(volume_prepare_kernel, (unsigned)((n + 255) / 256), 256, 0, stream, 
      volume, resolution, inv_h, reinterpret_cast<float4*>(vol4));
  count_launch();
  return launch_status();
}

namespace {

bool cell_size_ok(int32_t cell) { return cell >= 1 && cell <= 64 && (cell & (cell - 1)) == 0; }

int cells_per_axis(int32_t resolution, int32_t cell) {
  return (resolution - 1 + cell - 1) / cell;  // macrocells covering the R - 1 vertex cells
}

}  // namespace

extern "C" veg_status veg_raymarch_cells_count(int32_t resolution, int32_t cell, int64_t* count) {
  if (!count || resolution < 2 || resolution > 2048 || !cell_size_ok(cell))
    return VEG_ERR_INVALID_ARGUMENT;
  const int64_t c = cells_per_axis(resolution, cell);
  *count = c * c * c;
  return VEG_OK;
}

extern "C" veg_status veg_raymarch_cells(const float* vol4, int32_t resolution, veg_tf tf,
                                         int32_t cell, uint32_t* mask, cudaStream_t stream) {
  if (!vol4 || !mask || resolution < 2 || resolution > 2048 || !cell_size_ok(cell) || !tf.lut ||
      tf.lut_size < 2 || tf.n_tf < 1 || !aligned16(vol4) || !aligned16(tf.lut))
    return VEG_ERR_INVALID_ARGUMENT;
  const int c = cells_per_axis(resolution, cell);
  const int64_t nc = (int64_t)c * c * c;
  const int lanes = cell >= 8 ? 32 : nc >= 65536 ? 1 : 8;
  auto kern = lanes == 1   ? cell_mask_kernel<1>
              : lanes == 8 ? cell_mask_kernel<8>
                           : cell_mask_kernel<32>;
  launch_k(kern, (unsigned)((nc * lanes + 255) / 256), 256, 0, stream,
           reinterpret_cast<const float4*>(vol4), resolution, cell, c,
           reinterpret_cast<const float4*>(tf.lut), tf.lut_size, tf.n_tf, mask);
  count_launch();
  return launch_status();
}

extern "C" veg_status veg_raymarch_masked(const veg_camera* cams, int32_t n_views,
                                          const float* vol4, int32_t resolution, veg_tf tf,
                                          float step, const veg_material* material,
                                          const float* bg, const uint32_t* cell_mask,
                                          int32_t cell, float* out, unsigned long long* stats,
                                          cudaStream_t stream) {
  veg_status st = check_cameras_one_size(cams, n_views);
  if (st != VEG_OK) return st;
  if (!vol4 || !out || resolution < 2 || resolution > 2048 || !(step > 0.0f) || !tf.lut ||
      tf.lut_size < 2 || tf.n_tf < 1 || !aligned16(vol4) || !aligned16(out) ||
      !aligned16(tf.lut) || (cell_mask && !cell_size_ok(cell)))
    return VEG_ERR_INVALID_ARGUMENT;
  if (tf.lut_size > 4096) return VEG_ERR_UNSUPPORTED;
  MarchArgs A;
  A.cell_mask = cell_mask;
  A.cell_shift = 0;
  while (cell_mask && (1 << A.cell_shift) < cell) ++A.cell_shift;
  A.cells = cell_mask ? cells_per_axis(resolution, cell) : 0;
  A.vol = reinterpret_cast<const float4*>(vol4);
  A.R = resolution;
  const double h = 2.0 / (resolution - 1);
  A.inv_h = (float)(1.0 / h);
  A.step = step;
  A.ratio = (float)(step / h);
  A.lut = reinterpret_cast<const float4*>(tf.lut);
  A.lut_size = tf.lut_size;
  A.n_tf = tf.n_tf;
  A.view_tf = tf.view_tf;
  A.width = cams[0].width;
  A.height = cams[0].height;
  A.tiles_x = tiles_x_of(A.width);
  A.tiles_per_view = A.tiles_x * tiles_x_of(A.height);
  A.ka = material ? material->ka : 0.f;
  A.kd = material ? material->kd : 0.f;
  A.ks = material ? material->ks : 0.f;
  A.beta = material ? material->beta : 0.f;
  // what a sample's shade must be for zero opacity times it to be zero under
  // every table that leaves it out (colours up to 1e30): no huge coefficient or
  // light, and no shininess that is negative or lifts a cosine rounded up
  // from 1 beyond the floats
  A.leave_out = std::fabs(A.ka) <= 1e6f && std::fabs(A.kd) <= 1e6f && std::fabs(A.ks) <= 1e6f &&
                A.beta >= 0.0f && A.beta <= 1e6f;
  A.bg0 = bg ? bg[0] : 0.f;
  A.bg1 = bg ? bg[1] : 0.f;
  A.bg2 = bg ? bg[2] : 0.f;
  RaySet rs;
  for (int v = 0; v < n_views; ++v) {
    const float* w = cams[v].world_to_cam;
    RayView& V = rs.v[v];
    for (int r = 0; r < 3; ++r)
      for (int c = 0; c < 3; ++c) V.r[r * 3 + c] = w[r * 4 + c];
    for (int c = 0; c < 3; ++c) {
      V.eye[c] = -(w[0 * 4 + c] * w[3] + w[1 * 4 + c] * w[7] + w[2 * 4 + c] * w[11]);
      V.light[c] = -w[2 * 4 + c];
      A.leave_out = A.leave_out && std::fabs(V.light[c]) <= 2.0f;
    }
    V.fx = cams[v].fx;
    V.fy = cams[v].fy;
    V.cx = cams[v].cx;
    V.cy = cams[v].cy;
    V.near_plane = cams[v].near_plane;
  }
  float4* o = reinterpret_cast<float4*>(out);
  // tables per sample pass: the fewest equal groups
  const int all = tf.view_tf ? 1 : tf.n_tf, groups = (all + kMarchTables - 1) / kMarchTables;
  A.group = (all + groups - 1) / groups;
  if (material)
    return A.group > 1 ? launch_march_s<true, true>(A, rs, n_views, o, stats, stream)
                       : launch_march_s<false, true>(A, rs, n_views, o, stats, stream);
  return A.group > 1 ? launch_march_s<true, false>(A, rs, n_views, o, stats, stream)
                     : launch_march_s<false, false>(A, rs, n_views, o, stats, stream);
}

extern "C" veg_status veg_raymarch(const veg_camera* cams, int32_t n_views, const float* vol4,
                                   int32_t resolution, veg_tf tf, float step,
                                   const veg_material* material, const float* bg, float* out,
                                   unsigned long long* stats, cudaStream_t stream) {
  return veg_raymarch_masked(cams, n_views, vol4, resolution, tf, step, material, bg, nullptr, 1,
                             out, stats, stream);
}
