// Compositing kernels: front-to-back blending (Eq. 1) of depth-sorted splats
// per 16x16 tile under each transfer function, and its backward pass.
//
// One CTA of 128 threads owns one (view, tile, table) work item, in the
// longest-first order of the tiles; each warp owns an 8x8 pixel block and
// each lane two of its pixels, (x, y) and (x, y + 4).  The forward stages the
// tile's list in batches of B splats (the tile batch: 128, 256 or 512,
// chosen by the caller or its autotuner) through shared memory; the
// backward's warps each stage the chunks of 32 that they walk.  The stager
// evaluates a splat's colour and opacity under the table (linear
// interpolation, the table read through the L1 cache), the exponent below
// which it cannot reach alpha = 1/255, and which warp blocks its visible
// ellipse can touch; each warp walks only the splats that touch its block, so
// pairs that provably cannot blend cost nothing.  A pixel leaves once it has terminated
// (T (1 - alpha) < 1e-4); a work item ends once all its pixels have left.
//
// Launches of few work items take a second forward kernel, whose CTA holds one
// 8x8 block and divides staging and blending between warps (below).
//
// One table per work item: a splat that a table maps to no opacity never
// enters that item's lists, and each table stops at its own termination.
// Walking a group of 2 or 4 tables at once shares a splat's geometry but
// walks the union of their lists: on the 1M-Gaussian scene it took 2 to 4
// times as long forward.  The backward, which shares more, does so where the
// tables overlap (composite_bwd_group.cuh).
//
// What bounds both kernels is instruction issue: a tile's splats are read
// from DRAM once (1-2% of its rate) and then meet up to 256 pixels each.  Two
// pixels per lane halve what a splat costs per pixel beyond its own
// arithmetic (list entry, shared-memory loads, loop, warp votes and, in the
// backward, the warp reduction), and most of the pair's arithmetic runs in
// the two-wide float32 instructions.  From one pixel per lane (and groups of
// tables) to two, whole calls on the 1M-Gaussian scene (1024x1024, four tables)
// went from 820 to 655 us forward and from 1812 to 1231 backward; the kernels
// now take 518 and 1077.
//
// The per-pair arithmetic that decides skips, the 0.99 clamp and
// termination uses explicitly rounded operations shared by the forward and
// backward kernels, so the backward replays every forward decision bit for
// bit.  Culling (cutoff, warp mask) only removes pairs whose alpha is
// provably below 1/255, so it never changes a decision.
#pragma once

#include <algorithm>

#include "veg_internal.cuh"

namespace veg {

namespace {

constexpr int kWarps = 4;
constexpr int kCompThreads = 32 * kWarps;
constexpr float kLog2e = 1.44269502162933349609375f;
constexpr float kHuge = 3.0e38f;
// Every per-splat shared array of the forward is indexed by the splat's batch
// slot, which a thread loops over in steps of the block size; slot B is a
// splat that no pixel blends (it pads the warp lists to whole steps of the
// walk).  A warp list entry is 16 times the batch slot: the byte offset of the slot
// in every 16-byte shared array.
using ListEntry = unsigned short;

// 2^x with the hardware approximation (ex2.approx.ftz), x = power * log2(e).
// For x <= 0 the result is at most 1 (checked over every float32 below zero).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }

// The Gaussians of a lane's two pixels: e^power with
//   power = -1/2 (a dx^2 + c dy^2) - b dx dy,
// u = (ux, ux, uy, uy), q = (-a/2, -a/2, -b, -b), r = (-c/2, -c/2, ..).
// Both halves are rounded exactly like the scalar operations.
struct Offsets {
  float2 dx, dy, dxx, dyy, dxy;  // of the splat centre from the two pixels
};
__device__ __forceinline__ float2 power2(float4 u, float4 q, float4 r, float2 px, float2 py,
                                         Offsets& o) {
  o.dx = sub2(lo2(u), px);
  o.dy = sub2(hi2(u), py);
  o.dxx = mul2(o.dx, o.dx);
  o.dyy = mul2(o.dy, o.dy);
  o.dxy = mul2(o.dx, o.dy);
  return fma2(lo2(q), o.dxx, fma2(lo2(r), o.dyy, mul2(hi2(q), o.dxy)));
}

// Lowest exponent at which a splat can still reach alpha >= 1/255: alpha =
// A w G = A w e^power stays below 1/255 for power < ln(1/(255 A w)).  The
// bound is lowered by 1e-3 to absorb the float32 rounding of the exponent,
// the exp2 approximation and the log, so every pair above it still meets the
// exact test and the cull never changes a decision.  With A w < 1/255 no
// pair can blend (a cutoff above 0).
__device__ __forceinline__ float power_cutoff(float aw) {
  if (!(aw >= kAlphaMin)) return 1.0f;
  return fmaxf(__logf(kAlphaMin) - __logf(aw) - 1e-3f, -1e30f);
}

// Hardware approximations (relative error of a few 1e-7), used only where
// a bound carries a far wider margin.
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Where a splat's exponent can reach `cut`: the pixel centres d (relative to
// the splat centre) with d^T Q d <= R = -2 cut (Q = conic), tested per block
// of pixel rows by the ellipse's x extent over the rows' y range.  Its right
// edge x+(y) = (-b y + sqrt(a R - det y^2)) / a is concave with its maximum
// hx at y = -b hx / c, so over a range it is largest at that y clamped to the
// range; the left edge mirrors it.  Extents are widened by 0.2% of hx + 0.02
// px, the y ranges by 0.2% of hy + 0.02 px and R by 0.2% + 1e-4, far beyond
// the float32 error of the extents (the cancellation in det and under the
// root stays below 0.03% of hx while det > 1e-3 a c) and of the per-pixel
// exponent, so the test never drops a pixel that the per-pixel decision
// keeps.  An ill-conditioned conic reaches everywhere (the per-pixel test
// decides).
struct Reach {
  bool none, all;
  float a, b, det, aR, ia, ystar, wx, wy;
  __device__ __forceinline__ Reach(float a_, float b_, float c, float cut) : a(a_), b(b_) {
    det = a * c - b * b;
    none = !(cut < 0.0f);
    all = !(det > 1e-3f * a * c);
    const float R = -2.0f * cut * 1.002f + 1e-4f, rd = R * rcp_approx(det);
    const float hx = sqrt_approx(rd * c), hy = sqrt_approx(rd * a);
    aR = a * R;
    ia = rcp_approx(a);
    ystar = -b * hx * rcp_approx(c);
    wx = hx * 0.002f + 0.02f;
    wy = hy * 1.002f + 0.02f;
  }
  // The x extent [x0, x1] over the rows [y0, y1]; false if they miss it.
  __device__ __forceinline__ bool extent(float y0, float y1, float& x0, float& x1) const {
    y0 = fmaxf(y0 - 0.01f, -wy);
    y1 = fminf(y1 + 0.01f, wy);
    const float yr = fminf(fmaxf(ystar, y0), y1), yl = fminf(fmaxf(-ystar, y0), y1);
    x1 = (sqrt_approx(fmaxf(aR - det * yr * yr, 0.0f)) - b * yr) * ia + wx;
    x0 = (-sqrt_approx(fmaxf(aR - det * yl * yl, 0.0f)) - b * yl) * ia - wx;
    return y0 <= y1;
  }
};

// The warp blocks a splat can reach, its centre at (rx, ry) from the tile's
// first pixel: bit by * 2 + bx for the 8x8 block at (8 bx, 8 by).
__device__ __forceinline__ unsigned warp_block_mask(float rx, float ry, const Reach& e) {
  if (e.none) return 0u;
  if (e.all) return 0xfu;
  unsigned m = 0u;
#pragma unroll
  for (int by = 0; by < 2; ++by) {
    float x0, x1;
    if (!e.extent(8.0f * by - ry, 8.0f * by + 7.0f - ry, x0, x1)) continue;
    if (x0 + rx <= 7.0f && x1 + rx >= 0.0f) m |= 1u << (2 * by);
    if (x0 + rx <= 15.0f && x1 + rx >= 8.0f) m |= 2u << (2 * by);
  }
  return m;
}

// Whether it can reach the 8x8 block whose first pixel is (-rx, -ry) from
// its centre.
__device__ __forceinline__ bool block_hit(float rx, float ry, const Reach& e) {
  float x0, x1;
  const bool rows = e.extent(-ry, 7.0f - ry, x0, x1);
  return !e.none && (e.all || (rows && x0 + rx <= 7.0f && x1 + rx >= 0.0f));
}

__device__ __forceinline__ unsigned lanemask_lt_() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Compacts the batch positions whose mask has this warp's bit, in order.
// Lane l reads the masks of its P = B/32 consecutive positions P l .. P l +
// P - 1 as one 32-bit word (B = 128) or P/8 64-bit words (positions past the
// batch's count hold empty masks); an exclusive warp scan of the per-lane
// hit counts places each lane's hits in the list, which ends in four entries
// of the padding slot B.
template <int B>
__device__ __forceinline__ int build_warp_list(const unsigned char* s_mask, ListEntry* list) {
  static_assert(B == 128 || B == 256 || B == 512, "tile batch of 128, 256 or 512 splats");
  constexpr int P = B / 32;
  constexpr int NW = P >= 8 ? P / 8 : 1;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned long long bits[NW];
  int c = 0;
  if (P == 4) {
    const unsigned m = reinterpret_cast<const unsigned*>(s_mask)[lane];
    bits[0] = (m >> warp) & 0x01010101u;  // bit 8k: position 4l + k
    c = __popc((unsigned)bits[0]);
  } else {
#pragma unroll
    for (int w = 0; w < NW; ++w) {
      const unsigned long long m =
          reinterpret_cast<const unsigned long long*>(s_mask)[lane * NW + w];
      bits[w] = (m >> warp) & 0x0101010101010101ull;  // bit 8k: position P l + 8 w + k
      c += __popcll(bits[w]);
    }
  }
  int incl = c;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  int pos = incl - c;
#pragma unroll
  for (int w = 0; w < NW; ++w) {
    unsigned long long bw = bits[w];
    while (bw) {
      const int bb = __ffsll((long long)bw) - 1;
      list[pos++] = (ListEntry)(16 * (P * lane + 8 * w + (bb >> 3)));
      bw &= bw - 1;
    }
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  if (lane < 4) list[total + lane] = (ListEntry)(16 * B);
  __syncwarp();
  return total;
}

// The lane's first pixel in 8x8 block w of a tile; its second is four rows
// below.
__device__ __forceinline__ void pixel_of(int tile, int tiles_x, int w, int& px, int& py) {
  const int l = threadIdx.x & 31;
  px = (tile % tiles_x) * VEG_TILE + (w & 1) * 8 + (l & 7);
  py = (tile / tiles_x) * VEG_TILE + (w >> 1) * 8 + (l >> 3);
}

struct CompArgs {
  const float4* geo;
  const float4* aux;
  const uint32_t* vals;
  const int2* ranges;
  const int32_t* order;    // work-item order (global tile ids) or null
  const int32_t* view_tf;  // per-view table index (one image per view) or null
  const float4* lut;
  const float2* shade;     // per-record Blinn-Phong factors (s_d, s_s) or null
  int lut_size, n_tf;
  ViewMap vm;  // per-view tiles and output pixels (views may differ in size)
  float bg0, bg1, bg2;
  bool by_overlap;  // backward: groups of overlapping tables go to the group kernel
};

// A work item: its tile, output image and table.
struct WorkItem {
  int px, py;           // the lane's first pixel
  int width, height;
  float tx0, ty0;       // the tile's first pixel
  long long image;      // first pixel of the output image
  int2 rg;              // the tile's list
  const float4* lut;    // the table, or null
};
// (group: tables per work item, the first one's)
__device__ __forceinline__ WorkItem work_item(const CompArgs& A, int item, int block,
                                              int group = 1) {
  WorkItem w;
  const int wi = A.order ? A.order[item] : item;  // global tile id
  const int view = view_of_tile(A.vm, wi), tile = wi - A.vm.tile_off[view];
  const int tiles_x = A.vm.tiles_x[view], t = (int)blockIdx.z * group;
  w.width = A.vm.width[view];
  w.height = A.vm.height[view];
  w.rg = A.ranges[wi];
  w.image = A.vm.pix_off[view] + (long long)t * w.width * w.height;
  pixel_of(tile, tiles_x, block, w.px, w.py);
  w.tx0 = (float)((tile % tiles_x) * VEG_TILE);
  w.ty0 = (float)((tile / tiles_x) * VEG_TILE);
  // an index outside [0, n_tf) reads as fully transparent: no table, an empty list
  const int ti = A.view_tf ? A.view_tf[view] : t;
  const bool ok = ti >= 0 && ti < A.n_tf;
  if (!ok) w.rg = make_int2(0, 0);
  w.lut = ok ? A.lut + (int64_t)ti * A.lut_size : nullptr;
  return w;
}

// Asynchronous copies of a chunk's records into shared memory: each lane
// fetches its own record of the next chunk while the warp walks the current
// one, and alone reads it back, so the gather's latency (a list entry, then
// two or three reads at its record) stays off the warp's path.
template <int N>
__device__ __forceinline__ void async_copy(void* dst, const void* src) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  // past the L1 cache, which the tables want (through it the backward of two
  // tables over 177x170 with 2M Gaussians takes 3245 us, past it 3043); 8-byte
  // copies exist through it only
  if (N == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src) : "memory");
}
__device__ __forceinline__ void async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
__device__ __forceinline__ void async_wait() {
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

// One record on its way or arrived: geo and aux, and its shading factors.
struct RawSlot {
  float4* geo;  // geo[0]: geo, geo[32]: aux
  float2* sh;
};
template <bool LIT>
__device__ __forceinline__ void fetch_record(const CompArgs& A, RawSlot s, uint32_t g) {
  async_copy<16>(s.geo, A.geo + g);
  async_copy<16>(s.geo + 32, A.aux + g);
  if (LIT) async_copy<8>(s.sh, A.shade + g);
}

// A record's colour and opacity under the item's table: lo and hi are the
// table entries around its scalar, aw = A w.  The entries come through the L1
// cache: a copy of the table in shared memory costs each item its time and the
// SMs their CTAs (1M-Gaussian scene under four tables, forward and backward:
// 518 and 1077 us at 256 entries, 520 and 1095 at 4096; with the copy 563 and
// 1125, 1158 and 1958).
struct SplatTf {
  float4 lo, hi;
  TfPos q;
  float aw;
};
__device__ __forceinline__ SplatTf splat_tf(const float4* lut, int L, float v, float w) {
  SplatTf s;
  s.q = tf_pos(v, L);
  s.lo = __ldg(lut + s.q.k);
  s.hi = __ldg(lut + s.q.k + 1);
  s.aw = mul(lerp_rn(s.lo.w, s.hi.w, s.q), w);
  return s;
}

// A conic with a NaN (an overflowed covariance) gives every pixel power NaN,
// which Eq. 1 reads as G = 1: it is staged as the zero conic.
__device__ __forceinline__ float4 clean_conic(float4 au) {
  if (!(au.x == au.x && au.y == au.y && au.z == au.z)) au.x = au.y = au.z = 0.0f;
  return au;
}

// Records of a batch on their way to shared memory: each thread fetches the
// records of its own batch slots with asynchronous copies while the warps
// walk the batch before, and alone reads them back, so the gather's latency
// (a list entry, then two or three 16-byte reads at its record) stays off
// the staging between two barriers.
template <int B, bool LIT>
struct Prefetch {
  static constexpr int N = B / kCompThreads;  // slots per thread
  float4* raw;       // [2][B]: geo, aux
  float2* raw_sh;    // [B] (LIT)
  uint32_t next[N];  // record of each slot in the batch to fetch next

  static __device__ __forceinline__ int slot(int r) { return (int)threadIdx.x + kCompThreads * r; }
  // the list entries of a batch of cnt splats at list index first
  __device__ __forceinline__ void index(const CompArgs& A, int first, int cnt) {
#pragma unroll
    for (int r = 0; r < N; ++r)
      if (slot(r) < cnt) next[r] = __ldg(&A.vals[first + slot(r)]);
  }
  __device__ __forceinline__ void fetch(const CompArgs& A, int cnt) {
#pragma unroll
    for (int r = 0; r < N; ++r) {
      const int s = slot(r);
      if (s >= cnt) continue;
      async_copy<16>(raw + s, A.geo + next[r]);
      async_copy<16>(raw + B + s, A.aux + next[r]);
      if (LIT) async_copy<8>(raw_sh + s, A.shade + next[r]);
    }
    async_commit();
  }
};

// Stages a fetched record into batch slot `s`: the exponent's coefficients,
// the colour and A w under the item's table, and the mask of the warp blocks
// that it can reach.  LIT: the shaded colour s_d C(v) + s_s (Eq. 2).
template <int B, bool LIT>
__device__ __forceinline__ void stage_splat(float4 ge, float4 au, float2 sh, int s,
                                            const float4* lut, int L, float tx0, float ty0,
                                            float4* s_geo, float2* s_ca, float4* s_col,
                                            unsigned char* s_mask) {
  const SplatTf t = splat_tf(lut, L, au.w, ge.w);
  float r = lerp_rn(t.lo.x, t.hi.x, t.q), g = lerp_rn(t.lo.y, t.hi.y, t.q),
        b = lerp_rn(t.lo.z, t.hi.z, t.q);
  if (LIT) {
    r = __fmaf_rn(sh.x, r, sh.y);
    g = __fmaf_rn(sh.x, g, sh.y);
    b = __fmaf_rn(sh.x, b, sh.y);
  }
  const float cut = power_cutoff(t.aw);
  s_mask[s] = (unsigned char)warp_block_mask(ge.x - tx0, ge.y - ty0, Reach(au.x, au.y, au.z, cut));
  au = clean_conic(au);
  s_geo[s] = make_float4(ge.x, ge.y, -0.5f * au.x, -au.y);
  s_ca[s] = make_float2(-0.5f * au.z, t.aw);
  s_col[s] = make_float4(r, g, b, cut);
}

// Entry of a shared array at 16 times its slot (ListEntry).
__device__ __forceinline__ float4 at16(const float4* a, unsigned off) {
  return *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(a) + off);
}
__device__ __forceinline__ float2 at16(const float2* a, unsigned off) {
  return *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(a) + (off >> 1));
}

// ---------------------------------------------------------------------------
// forward
// ---------------------------------------------------------------------------

// Exponents and alphas of a splat at a lane's two pixels (x, y) and (x, y'):
// g = (u_x, u_y, -a/2, -b), h = (-c/2, A w).
__device__ __forceinline__ float2 pair_alpha(float4 g, float2 h, float x, float2 y, float2& p) {
  const float dx = sub(g.x, x);
  const float2 dy = make_float2(sub(g.y, y.x), sub(g.y, y.y));
  const float dxx = mul(dx, dx);
  const float2 dyy = mul2(dy, dy);
  p = make_float2(__fmaf_rn(g.z, dxx, __fmaf_rn(h.x, dyy.x, mul(g.w, mul(dx, dy.x)))),
                  __fmaf_rn(g.z, dxx, __fmaf_rn(h.x, dyy.y, mul(g.w, mul(dx, dy.y)))));
  const float2 e = mul2(p, dup(kLog2e));
  return make_float2(fminf(kAlphaMax, mul(h.y, ex2_approx(e.x))),
                     fminf(kAlphaMax, mul(h.y, ex2_approx(e.y))));
}

// stats (instrumented build): visited pairs (every pair reached before the
// pixel's termination, the method's own count), iterated pairs (walked by
// the warp lists), pairs above the cutoff, alpha evaluations, blended pairs.
//
// The transmittance of a terminated pixel is kept with its sign set:
// T (1 - alpha) is then below the stop at every later splat, so the pair
// needs no separate live flag.
template <int B, bool STATS, bool LIT>
__global__ void __launch_bounds__(kCompThreads, 7)
    composite_fwd_kernel(CompArgs A, float4* __restrict__ out,
                         int32_t* __restrict__ n_contrib, unsigned long long* __restrict__ stats) {
  pdl_enter();
  constexpr int P = B + 1;
  extern __shared__ float4 smem[];
  float4* s_geo = smem;       // [P]: u_x, u_y, -a/2, -b
  float4* s_col = s_geo + P;  // [P]: r, g, b, cutoff
  Prefetch<B, LIT> pre;
  pre.raw = s_col + P;        // [2][B]
  float2* s_ca = reinterpret_cast<float2*>(pre.raw + 2 * B);  // [P]: -c/2, A w
  pre.raw_sh = s_ca + P;                                      // [B] (LIT)
  ListEntry* s_list = reinterpret_cast<ListEntry*>(pre.raw_sh + (LIT ? B : 0));  // [kWarps][B + 4]
  unsigned char* s_mask = reinterpret_cast<unsigned char*>(s_list + kWarps * (B + 4));  // [B]
  const int warp = threadIdx.x >> 5;
  ListEntry* my_list = s_list + warp * (B + 4);
  unsigned long long n_vis = 0, n_it = 0, n_eval = 0, n_blend = 0;
  const WorkItem W = work_item(A, (int)blockIdx.x, (int)(threadIdx.x >> 5));
  if (threadIdx.x == 0) {  // the padding slot: A w = 0 never blends
    s_geo[B] = s_col[B] = make_float4(0.f, 0.f, 0.f, 0.f);
    s_ca[B] = make_float2(0.f, 0.f);
  }
  const float2 fx = dup((float)W.px), fy = make_float2((float)W.py, (float)(W.py + 4));
  const int n = W.rg.y - W.rg.x;  // the list's length
  pre.index(A, W.rg.x, n);
  pre.fetch(A, n);
  pre.index(A, W.rg.x + B, n - B);
  float T[2], Cr[2], Cg[2], Cb[2];
  int last[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    T[i] = W.px < W.width && W.py + 4 * i < W.height ? 1.0f : -1.0f;
    Cr[i] = Cg[i] = Cb[i] = 0.0f;
    last[i] = 0;
  }

  for (int start = 0; start < n; start += B) {
    if (__syncthreads_count(T[0] > 0.0f || T[1] > 0.0f) == 0) break;
    const int cnt = min(B, n - start);
    async_wait();
#pragma unroll
    for (int r = 0; r < pre.N; ++r) {
      const int sl = pre.slot(r);
      if (sl < cnt)
        stage_splat<B, LIT>(pre.raw[sl], pre.raw[B + sl],
                            LIT ? pre.raw_sh[sl] : make_float2(1.f, 0.f), sl, W.lut, A.lut_size,
                            W.tx0, W.ty0, s_geo, s_ca, s_col, s_mask);
      else
        s_mask[sl] = 0;
    }
    pre.fetch(A, n - start - B);
    pre.index(A, W.rg.x + start + 2 * B, n - start - 2 * B);
    __syncthreads();
    const int nw = build_warp_list<B>(s_mask, my_list);
    int lb[2] = {-1, -1};  // offset of the pixel's last blended splat of this batch
    const bool act0[2] = {T[0] > 0.0f, T[1] > 0.0f};
    int jstop[2] = {cnt, cnt};  // 1 + batch position where the pixel terminated
    // four splats per step: first everything that does not depend on the
    // transmittance (exponents, Gaussians, alpha: independent, so they
    // overlap), then the blends in list order; a splat that no pixel of the
    // warp blends is passed over by a vote (one vote for all four, or all
    // votes ahead of the blends, measured 3-10% slower, two splats per step
    // 4%).  The exponents
    // are formed per pixel from (u, -a/2, -b) and -c/2: staging every value
    // twice for two-wide operations saves five instructions and costs 24
    // bytes of shared-memory reads per splat, the same time.
    for (int k = 0; k < nw; k += 4) {
      const uint2 en = *reinterpret_cast<const uint2*>(my_list + k);
      const unsigned off[4] = {en.x & 0xffffu, en.x >> 16, en.y & 0xffffu, en.y >> 16};
      float2 al[4];
      bool ok[4][2];
      float4 col[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        col[m] = at16(s_col, off[m]);
        const float4 g = at16(s_geo, off[m]);
        const float2 h = at16(s_ca, off[m]);
        float2 p;
        al[m] = pair_alpha(g, h, fx.x, fy, p);
        ok[m][0] = !(p.x > 0.0f) && !(al[m].x < kAlphaMin);
        ok[m][1] = !(p.y > 0.0f) && !(al[m].y < kAlphaMin);
        if (STATS && k + m < nw) {
          const float cut = col[m].w, pp[2] = {p.x, p.y};
#pragma unroll
          for (int i = 0; i < 2; ++i)
            if (T[i] > 0.0f) {
              ++n_it;
              n_eval += (unsigned)(pp[i] <= 0.0f && pp[i] >= cut);
            }
        }
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        if (!__any_sync(0xffffffffu, ok[m][0] || ok[m][1])) continue;
        // Eq. 1 update of the two pixels
        const float4 c = col[m];
        const float2 Tt = make_float2(T[0], T[1]);
        const float2 test2 = mul2(Tt, sub2(dup(1.0f), al[m])), wgt2 = mul2(al[m], Tt);
        const float test[2] = {test2.x, test2.y}, wgt[2] = {wgt2.x, wgt2.y};
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const bool stop = test[i] < kTMin;
          if (STATS && ok[m][i] && !stop) ++n_blend;
          if (STATS && ok[m][i] && stop && T[i] > 0.0f) jstop[i] = (int)(off[m] >> 4) + 1;
          if (ok[m][i] && stop) T[i] = -fabsf(T[i]);
          if (ok[m][i] && !stop) {
            Cr[i] = __fmaf_rn(c.x, wgt[i], Cr[i]);
            Cg[i] = __fmaf_rn(c.y, wgt[i], Cg[i]);
            Cb[i] = __fmaf_rn(c.z, wgt[i], Cb[i]);
            T[i] = test[i];
            lb[i] = (int)off[m];
          }
        }
      }
      if (!__any_sync(0xffffffffu, T[0] > 0.0f || T[1] > 0.0f)) break;
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (lb[i] >= 0) last[i] = start + (lb[i] >> 4) + 1;
    if (STATS) n_vis += (act0[0] ? (unsigned)jstop[0] : 0u) + (act0[1] ? (unsigned)jstop[1] : 0u);
  }
  async_wait();  // no copy in flight past the CTA's end
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    if (W.px >= W.width || W.py + 4 * i >= W.height) continue;
    const int64_t o = W.image + (int64_t)(W.py + 4 * i) * W.width + W.px;
    const float Tf = fabsf(T[i]);
    out[o] = make_float4(add(Cr[i], mul(Tf, A.bg0)), add(Cg[i], mul(Tf, A.bg1)),
                         add(Cb[i], mul(Tf, A.bg2)), Tf);
    n_contrib[o] = last[i];
  }
  if (STATS) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      n_vis += __shfl_down_sync(0xffffffffu, n_vis, o);
      n_it += __shfl_down_sync(0xffffffffu, n_it, o);
      n_eval += __shfl_down_sync(0xffffffffu, n_eval, o);
      n_blend += __shfl_down_sync(0xffffffffu, n_blend, o);
    }
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(&stats[0], n_vis);
      atomicAdd(&stats[1], n_it);
      atomicAdd(&stats[2], n_eval);
      atomicAdd(&stats[3], n_eval);
      atomicAdd(&stats[4], n_blend);
    }
  }
}

// ---------------------------------------------------------------------------
// forward of few work items
// ---------------------------------------------------------------------------

// With a few CTAs per SM in all, a launch lasts as long as its longest list:
// a warp blends it splat after splat, and most of that chain (a list entry,
// the shared reads, the exponent) does not depend on the transmittance.  Here
// a CTA holds one 8x8 block; four producer warps take every fourth chunk of
// 32 list entries, stage it and form the alphas of its splats at the 64
// pixels; two consumer warps, a pixel per lane, only blend.  The alphas pass
// through shared memory, a slot per producer, full and empty barriers per
// slot.  Decisions and images are those of composite_fwd_kernel bit for bit
// (the alphas come from the same operations, a pair that does not blend
// passes as 0).  It issues more instructions per pair, so the large launches
// stay with the other kernel (48.6M warp instructions against 26.5M on the
// 512x512 frame of 500k Gaussians, most of the difference the staging, which
// each of a tile's blocks does by itself; there it takes 79 us against 105,
// the SMs' busy share rising from 45% to 70%).
//
// Ending early: a consumer warp whose pixels have all left notes the chunk at
// which they did.  A chunk's producer ends the list when both did by the
// chunk that was in its slot before, which both have handed back: so the
// first chunk to end is kProducers after the later of the two notes, whatever
// the warps' timing, the next kProducers - 1 end too, and the consumers take
// all their marks before they leave.  Every barrier is met by all that take
// part in it.
constexpr int kProducers = 4;
constexpr int kDeepThreads = 32 * (2 + kProducers);

template <int ID0>
__device__ __forceinline__ void slot_sync(int slot) {
  __syncwarp();
  asm volatile("bar.sync %0, 96;" ::"r"(ID0 + slot) : "memory");
}
template <int ID0>
__device__ __forceinline__ void slot_arrive(int slot) {
  __threadfence_block();
  __syncwarp();
  asm volatile("bar.arrive %0, 96;" ::"r"(ID0 + slot) : "memory");
}
constexpr int kFull = 1, kEmpty = 1 + kProducers;  // named barriers; 0 is __syncthreads

template <bool LIT>
struct DeepSmem {
  struct Producer {
    float4 raw[2][2 * 32];        // records, alternate chunks
    float2 raw_sh[LIT ? 64 : 1];  // their shading factors
    float4 geo[32];               // the chunk's splats that reach the block
    float2 ca[32];
  } prod[kProducers];
  float alpha[kProducers][32 * 64];  // [splat][pixel], 0: does not blend
  float4 col[kProducers][32];
  int pos[kProducers][32];           // list position of each splat
  volatile int cnt[kProducers];      // splats in the slot, -1: the end
  volatile int gone[2];              // chunk at which a consumer's last pixel left
};

template <bool LIT>
__global__ void __launch_bounds__(kDeepThreads, 4)
    composite_fwd_deep_kernel(CompArgs A, float4* __restrict__ out,
                              int32_t* __restrict__ n_contrib) {
  pdl_enter();
  extern __shared__ float4 smem[];
  DeepSmem<LIT>& S = *reinterpret_cast<DeepSmem<LIT>*>(smem);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int block = (int)blockIdx.x & 3;
  const WorkItem W = work_item(A, (int)blockIdx.x >> 2, block);
  const int n = W.rg.y - W.rg.x;
  const int chunks = (n + 31) / 32;

  if (warp < 2) {
    const int py = W.py + 4 * warp;
    const bool inside = W.px < W.width && py < W.height;
    float T = inside ? 1.0f : -1.0f, Cr = 0.0f, Cg = 0.0f, Cb = 0.0f;
    int last = 0;
    bool gone = !__any_sync(0xffffffffu, inside);
    if (lane == 0) S.gone[warp] = gone ? 0 : 0x7fffffff;
    __syncthreads();
    for (int c = 0; c < chunks; ++c) {
      const int slot = c % kProducers;
      slot_sync<kFull>(slot);
      const int cnt = S.cnt[slot];
      if (cnt < 0) {
        for (int k = c + 1; k < c + kProducers && k < chunks; ++k) slot_sync<kFull>(k % kProducers);
        break;
      }
      if (!gone) {
        const float* al = S.alpha[slot] + warp * 32 + lane;
        int lb = -1;
        // eight splats per step: their reads overlap, then they blend in
        // order (the products of a whole step as one chain, with the stop
        // tested once, measured the same: the producers are the bound)
        for (int j = 0; j < cnt; j += 8) {
          float a[8];
          float4 col[8];
#pragma unroll
          for (int m = 0; m < 8; ++m) {
            a[m] = al[(j + m) * 64];
            col[m] = S.col[slot][j + m];
          }
#pragma unroll
          for (int m = 0; m < 8; ++m) {
            const float test = mul(T, sub(1.0f, a[m])), wgt = mul(a[m], T);
            const bool ok = a[m] > 0.0f, stop = test < kTMin;
            if (ok && stop) T = -fabsf(T);
            if (ok && !stop) {
              Cr = __fmaf_rn(col[m].x, wgt, Cr);
              Cg = __fmaf_rn(col[m].y, wgt, Cg);
              Cb = __fmaf_rn(col[m].z, wgt, Cb);
              T = test;
              lb = j + m;
            }
          }
        }
        if (lb >= 0) last = S.pos[slot][lb] + 1;
        gone = !__any_sync(0xffffffffu, T > 0.0f);
        if (gone && lane == 0) S.gone[warp] = c;
      }
      if (c + kProducers < chunks) slot_arrive<kEmpty>(slot);
    }
    if (inside) {
      const int64_t o = W.image + (int64_t)py * W.width + W.px;
      const float Tf = fabsf(T);
      out[o] = make_float4(add(Cr, mul(Tf, A.bg0)), add(Cg, mul(Tf, A.bg1)),
                           add(Cb, mul(Tf, A.bg2)), Tf);
      n_contrib[o] = last;
    }
    return;
  }

  const int me = warp - 2;
  auto& P = S.prod[me];
  const float bx0 = W.tx0 + (float)((block & 1) * 8), by0 = W.ty0 + (float)((block >> 1) * 8);
  const float fx = (float)W.px;
  const float2 fy = make_float2((float)W.py, (float)(W.py + 4));
  const uint32_t* list = A.vals + W.rg.x;
  constexpr int kStride = 32 * kProducers;
  auto raw = [&](int side) {
    RawSlot r;
    r.geo = P.raw[side] + lane;
    r.sh = P.raw_sh + (LIT ? side * 32 + lane : 0);
    return r;
  };
  int at = me * 32 + lane;  // this lane's list position
  uint32_t next = 0;
  if (at < n) fetch_record<LIT>(A, raw(0), __ldg(&list[at]));
  async_commit();
  if (at + kStride < n) next = __ldg(&list[at + kStride]);
  __syncthreads();  // the consumers' marks
  int side = 0;
  for (int c = me; c < chunks; c += kProducers, at += kStride, side ^= 1) {
    async_wait();
    bool hit = false;
    float4 ge, au;
    SplatTf tf;
    float cut = 1.0f;
    if (at < n) {
      ge = P.raw[side][lane];
      au = P.raw[side][32 + lane];
      tf = splat_tf(W.lut, A.lut_size, au.w, ge.w);
      cut = power_cutoff(tf.aw);
      hit = block_hit(ge.x - bx0, ge.y - by0, Reach(au.x, au.y, au.z, cut));
    }
    const unsigned hits = __ballot_sync(0xffffffffu, hit);
    const int nh = __popc(hits), place = __popc(hits & lanemask_lt_());
    float4 col = make_float4(0.f, 0.f, 0.f, 0.f);
    if (hit) {
      col = make_float4(lerp_rn(tf.lo.x, tf.hi.x, tf.q), lerp_rn(tf.lo.y, tf.hi.y, tf.q),
                        lerp_rn(tf.lo.z, tf.hi.z, tf.q), 0.0f);
      if (LIT) {
        const float2 sh = P.raw_sh[side * 32 + lane];
        col.x = __fmaf_rn(sh.x, col.x, sh.y);
        col.y = __fmaf_rn(sh.x, col.y, sh.y);
        col.z = __fmaf_rn(sh.x, col.z, sh.y);
      }
      const float4 cc = clean_conic(au);
      P.geo[place] = make_float4(ge.x, ge.y, -0.5f * cc.x, -cc.y);
      P.ca[place] = make_float2(-0.5f * cc.z, tf.aw);
    }
    if (at + kStride < n) fetch_record<LIT>(A, raw(side ^ 1), next);
    async_commit();
    if (at + 2 * kStride < n) next = __ldg(&list[at + 2 * kStride]);
    if (c >= kProducers) {
      slot_sync<kEmpty>(me);
      if (max(S.gone[0], S.gone[1]) <= c - kProducers) {
        if (lane == 0) S.cnt[me] = -1;
        slot_arrive<kFull>(me);
        break;
      }
    }
    if (hit) {
      S.col[me][place] = col;
      S.pos[me][place] = at;
    }
    if (lane == 0) S.cnt[me] = nh;
    __syncwarp();
    float* al = S.alpha[me] + lane;
#pragma unroll 4
    for (int j = 0; j < nh; ++j) {
      float2 p;
      const float2 a = pair_alpha(P.geo[j], P.ca[j], fx, fy, p);
      al[j * 64] = !(p.x > 0.0f) && !(a.x < kAlphaMin) ? a.x : 0.0f;
      al[j * 64 + 32] = !(p.y > 0.0f) && !(a.y < kAlphaMin) ? a.y : 0.0f;
    }
    for (int j = nh; j < ((nh + 7) & ~7); ++j) al[j * 64] = al[j * 64 + 32] = 0.0f;
    slot_arrive<kFull>(me);
  }
  async_wait();  // no copy in flight past the CTA's end
}

// ---------------------------------------------------------------------------
// backward
// ---------------------------------------------------------------------------

// One halving exchange of a warp reduce-scatter: lanes keep the half of the
// 2 N slots named by their `bit` and add the partner's (lane ^ mask) values.
template <int N>
__device__ __forceinline__ void exchange(const float* v, float* w, bool bit, int mask) {
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float send = bit ? v[i] : v[i + N];
    const float keep = bit ? v[i + N] : v[i];
    w[i] = keep + __shfl_xor_sync(0xffffffffu, send, mask);
  }
}

__device__ __forceinline__ void red_add_v2(float2* p, float a, float b) {
  asm volatile("red.global.add.v2.f32 [%0], {%1, %2};" ::"l"(p), "f"(a), "f"(b) : "memory");
}

__device__ __forceinline__ void red_add_v4(float4* p, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(a), "f"(b), "f"(c),
               "f"(d)
               : "memory");
}

// Over the warp, two splats' sums of a lane's two pixels, into their
// accumulator slots: v = (dp, dL/dv (, dL/ds_d), dp dy, dp dy^2 (, dL/ds_s)) of
// each, dx0 and dx1 their offsets.
template <bool LIT>
__device__ __forceinline__ void reduce_pair(const float* v, float dx0, float dx1, float* acc) {
  constexpr int kSum = LIT ? 6 : 4, kAcc = LIT ? 12 : 8;
  // over the columns' lanes: bit 4 selects the splat, bit 3 the half of its
  // sums; then times the column's dx over the eight columns (slot bits 2 and
  // 1): slots (S0, S0 dx, S0 dx^2, V) and (S1, S1 dx, -, S2)
  const int lane = threadIdx.x & 31;
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4, b1 = lane & 2;
  float w[kSum], x[kSum / 2], y[4], z[2];
  exchange<kSum>(v, w, b4, 16);
  exchange<kSum / 2>(w, x, b3, 8);
  const float dx = b4 ? dx1 : dx0;
  y[0] = x[0];
  y[1] = x[0] * dx;
  y[2] = y[1] * dx;
  y[3] = x[1];
  exchange<2>(y, z, b2, 4);
  float f;
  exchange<1>(z, &f, b1, 2);
  f += __shfl_xor_sync(0xffffffffu, f, 1);
  acc += b4 ? kAcc : 0;
  if ((lane & 1) == 0) acc[(lane >> 1) & 7] = f;
  if (LIT) {
    float s = x[kSum / 2 - 1];
#pragma unroll
    for (int d = 4; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if ((lane & 7) == 0) acc[8 + (b3 ? 1 : 0)] = s;
  }
}

// Adds a splat's reduced sums to its record's gradients: moments of dp to the
// screen gradients, du = (-a S_x - b S_y, -b S_x - c S_y), dconic = (-S_xx / 2,
// -S_xy, -S_yy / 2).
template <bool LIT>
__device__ __forceinline__ void flush_splat(const float* sums, float weight, float4 aux,
                                            uint32_t rec, float4* grad2d, float2* grad_shade) {
  const float4* acc = reinterpret_cast<const float4*>(sums);
  const float4 a0 = acc[0], a1 = acc[1];  // (S, Sx, Sxx, dv), (Sy, Sxy, -, Syy)
  const bool any = a0.x != 0.f || a0.y != 0.f || a0.z != 0.f || a0.w != 0.f ||
                   a1.x != 0.f || a1.y != 0.f || a1.w != 0.f;
  if (any) {
    const float4 cc = clean_conic(aux);
    float4* dst = grad2d + 2 * (int64_t)rec;
    const float dw = weight > 0.0f ? a0.x / weight : 0.0f;
    red_add_v4(dst, -cc.x * a0.y - cc.y * a1.x, -cc.z * a1.x - cc.y * a0.y, -0.5f * a0.z, -a1.y);
    red_add_v4(dst + 1, -0.5f * a1.w, a0.w, dw, 0.0f);
  }
  if (LIT) {
    const float4 a2 = acc[2];
    if (a2.x != 0.f || a2.y != 0.f) red_add_v2(grad_shade + rec, a2.x, a2.y);
  }
}

// Whether the tables of the group from t0 on have opacity at the same scalars,
// by 32 samples: of the samples that any table has, each has kBwdOverlap on
// average.  Both backward kernels ask, and take the group or leave it to the
// other.  Tables of three bumps come to 0.64 to 0.91 and are the faster one by
// one (1M-Gaussian scene, four of them: 1079 us, in a group 1374), tables of
// eight to 0.88 to 0.98 and are about even (1142 and 981 there; 512x512 under
// eight 1398 and 2084), one opacity under several colour maps to 1 (1019, 760).
constexpr int kBwdGroup = 4;
constexpr float kBwdOverlap = 0.95f;
__device__ __forceinline__ bool tables_overlap(const CompArgs& A, int t0) {
  const int k = (int)(threadIdx.x & 31) * (A.lut_size - 1) / 31;
  const int n = min(kBwdGroup, A.n_tf - t0);
  unsigned any = 0u;
  int sum = 0;
#pragma unroll
  for (int t = 0; t < kBwdGroup; ++t) {
    const bool seen = t < n && __ldg(&A.lut[(int64_t)(t0 + t) * A.lut_size + k].w) >= kAlphaMin;
    const unsigned m = __ballot_sync(0xffffffffu, seen);
    any |= m;
    sum += __popc(m);
  }
  return n > 2 && (float)sum >= kBwdOverlap * (float)(n * __popc(any));
}

// Walks each pixel's list back to front, from its last contribution to the
// first splat.  Below n_contrib a pair blends exactly when its exponent is in
// range and alpha >= 1/255 (the stop only ends the list), so every decision
// is recomputed bit for bit from the same float32 operations as the forward,
// without the forward's transmittance.  With T_i the transmittance in front
// of blended splat i and Suf_i = sum over blended j > i of (c_j . g) alpha_j
// T_j + T_final (bg . g + g_T), the gradient of the loss w.r.t. alpha_i is
//   dL/dalpha_i = T_i (c_i . g) - Suf_i / (1 - alpha_i).
// Each pixel starts from T_final (the forward's output) and recovers
// T_i = T_{i+1} / (1 - alpha_i) with the reciprocal that dL/dalpha_i needs
// anyway; Suf grows from the back, so the small terms of deep splats are
// summed first and keep their relative accuracy (a front-to-back prefix
// K - S_i would leave them as a difference of two O(1) numbers).  Per splat,
// the seven screen-space gradients are summed over a lane's two pixels,
// reduced over the warp and added to the per-record gradient buffer, once per
// warp and table.
//
// The screen gradients are linear in the sums of dp = dL/dpower times 1, dx,
// dy, dx^2, dx dy, dy^2 (d = u - pixel; power = -a/2 dx^2 - b dx dy - c/2
// dy^2), with per-splat coefficients applied once at the flush.  The eight
// pixels of a block's column share dx, so the warp reduces in two stages:
// over a column (lanes 8 and 16 apart) the four sums of dp, dp dy, dp dy^2
// and dL/dv, then, multiplied by the column's dx, over the eight columns.
// Two splats go through one reduction: 41 instructions against 62 for a
// direct reduce-scatter of the seven products, and four products fewer per
// splat.
//
// The weight needs no sum of its own: below the clamp alpha = A w e^power,
// so dalpha/dw = alpha / w = (dalpha/dpower) / w and dL/dw is the summed
// exponent gradient dL/dpower divided by w (applied at the flush; a splat
// with w = 0 never blends and gets 0).
//
// Shaded (LIT): the blended colour is s_d C + s_s, so c.g = s_d (C.g) + s_s
// (g_r + g_g + g_b), dL/dC = s_d alpha T g, and the pair adds alpha T (C.g)
// to dL/ds_d and alpha T (g_r + g_g + g_b) to dL/ds_s, reduced beside the
// others; the two shading sums go to grad_shade.
//
// stats (instrumented build): replayed pairs (list positions below the
// pixel's last contribution), iterated pairs, pairs above the cutoff, alpha
// evaluations, blended pairs, blended pairs below the clamp, pairs with a
// nonzero screen-space gradient.
template <bool LIT>
struct BwdWarp {
  static constexpr int kAcc = LIT ? 12 : 8;  // accumulator slots per splat
  float4 u[34];   // u_x, u_x, u_y, u_y
  float4 q[34];   // -a/2, -a/2, -b, -b
  float4 r[34];   // -c/2, -c/2, list position (bits), cutoff
  float4 c0[34];  // r, r, g, g
  float4 c1[34];  // b, b, Aw, Aw
  float4 d0[34];  // dr/dv, dr/dv, dg/dv, dg/dv (times s_d)
  float4 d1[34];  // db/dv, db/dv, w dA/dv, w dA/dv
  float4 sh[LIT ? 34 : 1];  // s_d, s_d, s_s, s_s
  float4 raw[2][2 * 32];    // records, alternate chunks
  float acc[34 * kAcc];     // gradient sums of the chunk's splats
};

// Five CTAs per SM (95 registers) unshaded: 862 us against 897 at four (122) on a
// 1M-Gaussian training step's image under four tables, 692 and 734 on two views
// of 1200x900 under three (258 and 239 on one table at 800x800, which ends with
// its longest lists).  Shaded four (124): 650 us against 683 at five (96) on three
// views of 641x479, 283 and 320 on one table at 800x800 (1053 and 1036 on the
// 1M-Gaussian one).
template <bool STATS, bool LIT>
__global__ void __launch_bounds__(kCompThreads, LIT || STATS ? 4 : 5)
    composite_bwd_kernel(CompArgs A, const float4* __restrict__ out,
                         const int32_t* __restrict__ n_contrib, const float4* __restrict__ dout,
                         float4* __restrict__ grad2d, float2* __restrict__ grad_shade,
                         unsigned long long* __restrict__ stats) {
  pdl_enter();
  using Warp = BwdWarp<LIT>;
  constexpr int kAcc = Warp::kAcc;
  unsigned long long n_rep = 0, n_it = 0, n_eval = 0, n_blend = 0, n_free = 0, n_grad = 0;
  extern __shared__ float4 smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Warp& S = reinterpret_cast<Warp*>(smem)[warp];
  float2* s_sh = reinterpret_cast<float2*>(reinterpret_cast<Warp*>(smem) + kWarps) + threadIdx.x;
  const WorkItem W = work_item(A, (int)blockIdx.x, (int)(threadIdx.x >> 5));
  if (A.by_overlap && tables_overlap(A, (int)blockIdx.z / kBwdGroup * kBwdGroup)) return;
  const float bx0 = W.tx0 + (float)((warp & 1) * 8), by0 = W.ty0 + (float)((warp >> 1) * 8);
  const float2 fx = dup((float)W.px), fy = make_float2((float)W.py, (float)(W.py + 4));

  // per pixel: transmittance behind the splats walked so far, the negated
  // suffix sum, the upstream colour gradient and n_contrib
  float4 ov[2], dv4[2];
  int nc[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    ov[i] = make_float4(0.f, 0.f, 0.f, 1.f);
    dv4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    nc[i] = 0;
    if (W.lut && W.px < W.width && W.py + 4 * i < W.height) {
      const int64_t o = W.image + (int64_t)(W.py + 4 * i) * W.width + W.px;
      ov[i] = out[o];
      dv4[i] = dout[o];
      nc[i] = n_contrib[o];
    }
  }
  float2 T = make_float2(ov[0].w, ov[1].w);
  const float2 gr = make_float2(dv4[0].x, dv4[1].x), gg = make_float2(dv4[0].y, dv4[1].y),
               gb = make_float2(dv4[0].z, dv4[1].z);
  auto suf = [&](float4 o, float4 d) {
    return -(o.w * (A.bg0 * d.x + A.bg1 * d.y + A.bg2 * d.z + d.w));
  };
  float2 nSuf = make_float2(suf(ov[0], dv4[0]), suf(ov[1], dv4[1]));
  if (STATS) n_rep += (unsigned long long)nc[0] + (unsigned long long)nc[1];
  // the warp walks from its last contribution; lane l of a chunk ending at
  // list position `end` holds position end - 1 - l
  const int wmax = __reduce_max_sync(0xffffffffu, max(nc[0], nc[1]));
  const uint32_t* list = A.vals + W.rg.x;
  uint32_t cur = 0, next = 0;  // this lane's record in the chunk fetched last, and in the next
  int side = 0;
  auto raw = [&](int sd) {
    RawSlot s;
    s.geo = S.raw[sd] + lane;
    s.sh = s_sh;
    return s;
  };
  if (wmax - 1 - lane >= 0) {
    cur = __ldg(&list[wmax - 1 - lane]);
    fetch_record<LIT>(A, raw(0), cur);
  }
  async_commit();
  if (wmax - 33 - lane >= 0) next = __ldg(&list[wmax - 33 - lane]);
  for (int end = wmax; end > 0; end -= 32, side ^= 1) {
    // stage this chunk: each lane tests its record against the warp's block,
    // the hits are compacted, last one first
    async_wait();
    const int pos = end - 1 - lane;
    const uint32_t rec = cur;
    bool hit = false;
    float4 ge, au;
    SplatTf tf;
    float cut = 1.0f;
    if (pos >= 0) {
      ge = S.raw[side][lane];
      au = S.raw[side][32 + lane];
      tf = splat_tf(W.lut, A.lut_size, au.w, ge.w);
      cut = power_cutoff(tf.aw);
      hit = block_hit(ge.x - bx0, ge.y - by0, Reach(au.x, au.y, au.z, cut));
    }
    const unsigned hits = __ballot_sync(0xffffffffu, hit);
    const int nh = __popc(hits), slot = __popc(hits & lanemask_lt_());
    if (hit) {
      float2 sh = make_float2(1.0f, 0.0f);
      if (LIT) sh = *s_sh;
      const float sl = (au.w >= 0.0f && au.w <= 1.0f) ? (float)(A.lut_size - 1) : 0.0f;
      const float slc = LIT ? sl * sh.x : sl;  // colour slope scale
      const float r = lerp_rn(tf.lo.x, tf.hi.x, tf.q), g = lerp_rn(tf.lo.y, tf.hi.y, tf.q),
                  b = lerp_rn(tf.lo.z, tf.hi.z, tf.q);
      const float dr = slc * (tf.hi.x - tf.lo.x), dg = slc * (tf.hi.y - tf.lo.y),
                  db = slc * (tf.hi.z - tf.lo.z),
                  da = fminf(fmaxf(ge.w * sl * (tf.hi.w - tf.lo.w), -kHuge), kHuge);
      const float4 cc = clean_conic(au);
      S.u[slot] = make_float4(ge.x, ge.x, ge.y, ge.y);
      S.q[slot] = make_float4(-0.5f * cc.x, -0.5f * cc.x, -cc.y, -cc.y);
      S.r[slot] = make_float4(-0.5f * cc.z, -0.5f * cc.z, __int_as_float(pos), cut);
      S.c0[slot] = make_float4(r, r, g, g);
      S.c1[slot] = make_float4(b, b, tf.aw, tf.aw);
      S.d0[slot] = make_float4(dr, dr, dg, dg);
      S.d1[slot] = make_float4(db, db, da, da);
      if (LIT) S.sh[slot] = make_float4(sh.x, sh.x, sh.y, sh.y);
    }
    if (lane == 0) {  // pads an odd count: A w = 0 never blends
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      S.u[nh] = S.q[nh] = S.c0[nh] = S.c1[nh] = S.d0[nh] = S.d1[nh] = z;
      S.r[nh] = make_float4(0.f, 0.f, 0.f, 1.f);
      if (LIT) S.sh[nh] = z;
    }
#pragma unroll
    for (int e = 0; e < kAcc / 4; ++e)
      reinterpret_cast<float4*>(S.acc)[e * 32 + lane] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (pos - 32 >= 0) {
      cur = next;
      fetch_record<LIT>(A, raw(side ^ 1), cur);
    }
    async_commit();
    if (pos - 64 >= 0) next = __ldg(&list[pos - 64]);
    __syncwarp();
    // two splats per step: what does not depend on the transmittance is
    // formed for both, then each blend is undone in turn
    for (int k = 0; k < nh; k += 2) {
      Offsets o[2];
      float2 G[2], raw2[2], al[2];
      bool ok[2][2];
      float4 c1[2];
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const float4 u = S.u[k + m], q = S.q[k + m], r = S.r[k + m];
        c1[m] = S.c1[k + m];
        const float2 p = power2(u, q, r, fx, fy, o[m]);
        const int at = __float_as_int(r.z);
        const float2 x = mul2(p, dup(kLog2e));
        G[m] = make_float2(ex2_approx(x.x), ex2_approx(x.y));
        raw2[m] = mul2(hi2(c1[m]), G[m]);
        al[m] = make_float2(fminf(kAlphaMax, raw2[m].x), fminf(kAlphaMax, raw2[m].y));
        ok[m][0] = at < nc[0] && !(p.x > 0.0f) && !(al[m].x < kAlphaMin);
        ok[m][1] = at < nc[1] && !(p.y > 0.0f) && !(al[m].y < kAlphaMin);
        if (STATS && r.w < 0.0f) {
          n_it += 2;
          n_eval += (unsigned)(at < nc[0] && p.x <= 0.0f && p.x >= r.w) +
                    (unsigned)(at < nc[1] && p.y <= 0.0f && p.y >= r.w);
          n_blend += (unsigned)ok[m][0] + (unsigned)ok[m][1];
          n_free += (unsigned)(ok[m][0] && raw2[m].x <= kAlphaMax) +
                    (unsigned)(ok[m][1] && raw2[m].y <= kAlphaMax);
        }
      }
      if (!__any_sync(0xffffffffu, ok[0][0] || ok[0][1] || ok[1][0] || ok[1][1])) continue;
      // the splats' sums over the lane's two pixels: dp, dL/dv (, dL/ds_d),
      // dp dy, dp dy^2 (, dL/ds_s)
      constexpr int kSum = LIT ? 6 : 4;
      float v[2 * kSum];
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const float4 c0 = S.c0[k + m], s0 = S.d0[k + m], s1 = S.d1[k + m];
        const float2 om = sub2(dup(1.0f), al[m]);
        const float2 rr = make_float2(rcp_approx(om.x), rcp_approx(om.y));
        const float2 cgu = fma2(lo2(c1[m]), gb, fma2(hi2(c0), gg, mul2(lo2(c0), gr)));
        const float2 h = fma2(lo2(s1), gb, fma2(hi2(s0), gg, mul2(lo2(s0), gr)));
        const float2 Ti = mul2(T, rr);  // transmittance in front of the splat
        const float2 wgt = mul2(al[m], Ti);
        float2 cgd = cgu;
        if (LIT) {
          const float4 sh = S.sh[k + m];
          const float2 gs = add2(add2(gr, gg), gb);
          cgd = fma2(lo2(sh), cgu, mul2(hi2(sh), gs));
          const float2 d = mul2(wgt, cgu), s = mul2(wgt, gs);
          v[m * kSum + 2] = (ok[m][0] ? d.x : 0.0f) + (ok[m][1] ? d.y : 0.0f);
          v[m * kSum + 5] = (ok[m][0] ? s.x : 0.0f) + (ok[m][1] ? s.y : 0.0f);
        }
        const float2 da = fma2(Ti, cgd, mul2(nSuf, rr));
        // below the clamp alpha follows the exponent and the opacity slope (the
        // product is masked, not a factor: A w may be infinite)
        float2 mg = mul2(da, G[m]), cv = mul2(wgt, h);
        const bool free[2] = {ok[m][0] && raw2[m].x <= kAlphaMax,
                              ok[m][1] && raw2[m].y <= kAlphaMax};
        float2 dp = mul2(hi2(c1[m]), mg);
        dp.x = free[0] ? dp.x : 0.0f;
        dp.y = free[1] ? dp.y : 0.0f;
        mg.x = free[0] ? mg.x : 0.0f;
        mg.y = free[1] ? mg.y : 0.0f;
        cv.x = ok[m][0] ? cv.x : 0.0f;
        cv.y = ok[m][1] ? cv.y : 0.0f;
        const float2 dvv = fma2(hi2(s1), mg, cv);
        const float2 y1 = mul2(dp, o[m].dy), y2 = mul2(dp, o[m].dyy);
        v[m * kSum] = dp.x + dp.y;
        v[m * kSum + 1] = dvv.x + dvv.y;
        v[m * kSum + kSum / 2] = y1.x + y1.y;
        v[m * kSum + kSum / 2 + 1] = y2.x + y2.y;
        if (ok[m][0]) {
          nSuf.x = __fmaf_rn(-cgd.x, wgt.x, nSuf.x);
          T.x = Ti.x;
        }
        if (ok[m][1]) {
          nSuf.y = __fmaf_rn(-cgd.y, wgt.y, nSuf.y);
          T.y = Ti.y;
        }
        if (STATS) n_grad += (unsigned)(dp.x != 0.f) + (unsigned)(dp.y != 0.f);
      }
      reduce_pair<LIT>(v, o[0].dx.x, o[1].dx.x, S.acc + k * kAcc);
    }
    __syncwarp();
    // the lane that staged a splat adds its gradients to the record's
    if (hit)
      flush_splat<LIT>(S.acc + slot * kAcc, S.raw[side][lane].w, S.raw[side][32 + lane], rec,
                       grad2d, grad_shade);
    __syncwarp();
  }
  async_wait();  // no copy in flight past the CTA's end
  if (STATS) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      n_rep += __shfl_down_sync(0xffffffffu, n_rep, o);
      n_it += __shfl_down_sync(0xffffffffu, n_it, o);
      n_eval += __shfl_down_sync(0xffffffffu, n_eval, o);
      n_blend += __shfl_down_sync(0xffffffffu, n_blend, o);
      n_free += __shfl_down_sync(0xffffffffu, n_free, o);
      n_grad += __shfl_down_sync(0xffffffffu, n_grad, o);
    }
    if (lane == 0) {
      atomicAdd(&stats[0], n_rep);
      atomicAdd(&stats[1], n_it);
      atomicAdd(&stats[2], n_eval);
      atomicAdd(&stats[3], n_eval);
      atomicAdd(&stats[4], n_blend);
      atomicAdd(&stats[5], n_free);
      atomicAdd(&stats[6], n_grad);
    }
  }
}

// Dynamic shared memory of a CTA.  Forward: the padded splat arrays, the
// records on their way, warp lists and masks; backward: its warps' splats, the
// shading factors on their way.
size_t fwd_smem_bytes(bool lit, int B) {
  const size_t P = B + 1;
  return P * (16 + 16 + 8) + (size_t)2 * B * 16 + (lit ? (size_t)B * 8 : 0) +
         (size_t)kWarps * (B + 4) * sizeof(ListEntry) + (size_t)B;
}
size_t bwd_smem_bytes(bool lit) {
  return kWarps * (lit ? sizeof(BwdWarp<true>) : sizeof(BwdWarp<false>)) +
         (lit ? (size_t)kCompThreads * 8 : 0);
}

// Items (tiles times groups) from which a call lets the tables' overlap choose:
// fewer end with their longest lists, which one table at a time shortens (400x400,
// 20,000 Gaussians, four tables of one opacity: 165 us, in groups 181; 512x512,
// 100,000: 274 and 262).
constexpr int64_t kBwdGroupItems = 1024;
// Tile batch of the forward: the caller's choice (128, 256 or 512 splats), else
// 256 (1M-Gaussian scene under four tables 518 us, 526 at 128; 512 stages less
// often but holds fewer CTAs: 550 there, 333 against 432 for one faint table).
int pick_batch(int tile_batch) { return tile_batch > 0 ? tile_batch : 256; }

CompArgs make_args(const veg_camera* cams, int n_views, const float4* geo, const float4* aux,
                   const uint32_t* vals, const int2* ranges, const int32_t* order, veg_tf tf,
                   const float* bg, const float* shade) {
  CompArgs A;
  A.shade = reinterpret_cast<const float2*>(shade);
  A.geo = geo;
  A.aux = aux;
  A.vals = vals;
  A.ranges = ranges;
  A.order = order;
  A.view_tf = tf.view_tf;
  A.lut = reinterpret_cast<const float4*>(tf.lut);
  A.lut_size = tf.lut_size;
  A.n_tf = tf.n_tf;
  A.vm = make_viewmap(cams, n_views, tf.view_tf ? 1 : tf.n_tf);
  A.bg0 = bg ? bg[0] : 0.f;
  A.bg1 = bg ? bg[1] : 0.f;
  A.bg2 = bg ? bg[2] : 0.f;
  A.by_overlap = false;
  return A;
}

// One CTA per (tile, image): every table of the call, or one image per view.
inline dim3 comp_grid(const CompArgs& A, int n_views) {
  return dim3((unsigned)A.vm.tile_off[n_views], 1u, A.view_tf ? 1u : (unsigned)A.n_tf);
}

template <int B, bool STATS, bool LIT>
veg_status launch_fwd(const CompArgs& A, int n_views, float4* out, int32_t* nc,
                      unsigned long long* stats, cudaStream_t stream) {
  const size_t smem = fwd_smem_bytes(LIT, B);
  auto kern = composite_fwd_kernel<B, STATS, LIT>;
  static SmemRecord configured;
  veg_status st = prepare_smem(kern, smem, configured, false);
  if (st != VEG_OK) return st;
  launch_k(kern, comp_grid(A, n_views), kCompThreads, smem, stream, A, out, nc, stats);
  count_launch();
  return launch_status();
}

template <bool STATS, bool LIT>
veg_status launch_bwd(const CompArgs& A, int n_views, const float4* out, const int32_t* nc,
                      const float4* dout, float4* grad2d, float2* grad_shade,
                      unsigned long long* stats, cudaStream_t stream) {
  const size_t smem = bwd_smem_bytes(LIT);
  auto kern = composite_bwd_kernel<STATS, LIT>;
  static SmemRecord configured;
  veg_status st = prepare_smem(kern, smem, configured, false);
  if (st != VEG_OK) return st;
  launch_k(kern, comp_grid(A, n_views), kCompThreads, smem, stream, A, out, nc, dout, grad2d,
           grad_shade, stats);
  count_launch();
  return launch_status();
}

// The launches that take composite_fwd_deep_kernel.  Its time per (tile, table)
// item is mostly fixed (four CTAs that each stage a list), the other kernel's
// is its longest lists until the SMs are full, so the line rises with the
// lists' length, for which the records stand: forward with it against without,
// 500 records at 576 items 15 and 17 us, 784 19 and 17, 1024 24 and 17; 5,000 at
// 1024 35 and 45, 1296 43 and 46, 1600 52 and 46; 100,000 at 1296 63 and 79, 1600
// 73 and 77, 2025 88 and 72; 400,000 at 1600 97 and 107, 2025 112 and 100;
// 1,500,000 at 1764 155 and 172, 2025 166 and 170.
bool takes_deep(int64_t n, int64_t items) {
  return items < (n < 4096 ? 640 : n < 65536 ? 1280 : 1536);
}

template <bool LIT>
veg_status launch_fwd_deep(const CompArgs& A, int n_views, float4* out, int32_t* nc,
                           cudaStream_t stream) {
  const size_t smem = sizeof(DeepSmem<LIT>);
  auto kern = composite_fwd_deep_kernel<LIT>;
  static SmemRecord configured;
  veg_status st = prepare_smem(kern, smem, configured, false);
  if (st != VEG_OK) return st;
  dim3 grid = comp_grid(A, n_views);
  grid.x *= 4;
  launch_k(kern, grid, kDeepThreads, smem, stream, A, out, nc);
  count_launch();
  return launch_status();
}

// Dispatch over the tile batch (the instrumented build uses 256: the pair
// counts do not depend on the batch).
template <bool LIT>
veg_status fwd_batch(int B, const CompArgs& A, int n_views, int64_t n, float4* out, int32_t* nc,
                     cudaStream_t stream) {
  const dim3 items = comp_grid(A, n_views);
  if (takes_deep(n, (int64_t)items.x * items.z))
    return launch_fwd_deep<LIT>(A, n_views, out, nc, stream);
  if (B == 128) return launch_fwd<128, false, LIT>(A, n_views, out, nc, nullptr, stream);
  if (B == 512) return launch_fwd<512, false, LIT>(A, n_views, out, nc, nullptr, stream);
  return launch_fwd<256, false, LIT>(A, n_views, out, nc, nullptr, stream);
}

}  // namespace

}  // namespace veg
