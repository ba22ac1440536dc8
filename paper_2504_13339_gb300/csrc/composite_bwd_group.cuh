// Backward of the compositing for tables that overlap: four tables per pass.
//
// composite_bwd_kernel takes a table per work item, so that a splat that a table
// maps to no opacity costs that table nothing.  Where the tables have opacity
// at the same scalars (one opacity under several colour maps, broad ramps) their
// lists are the same, and each repeats the others' exponents, reductions and
// record updates.  Here a warp walks the union of four tables' lists and forms a
// pair's geometry, a splat's reduction and its update once.
//
// What bounds it is instruction issue, as there.  1M-Gaussian scene, 1024x1024,
// four tables, a table per pass and four: one opacity under four colour maps 1019
// and 760 us, opacity 0.05 throughout 3599 and 2437, 0.8 604 and 449; tables of
// three bumps 1079 and 1374, of eight 1142 and 981.  Choosing between them takes
// 8 us of the former's call and 20 of the latter's.
#pragma once

#include "composite_kernels.cuh"

namespace veg {

namespace {

template <bool LIT>
struct BwdGroupWarp {
  static constexpr int kAcc = LIT ? 12 : 8;  // accumulator slots per splat
  float4 u[34];  // u_x, u_x, u_y, u_y
  float4 q[34];  // -a/2, -a/2, -b, -b
  float4 r[34];  // -c/2, -c/2, list position (bits), -
  struct Table {
    float4 c0[34];  // r, r, g, g
    float4 c1[34];  // b, b, Aw, Aw
    float4 d0[34];  // dr/dv, dr/dv, dg/dv, dg/dv (times s_d)
    float4 d1[34];  // db/dv, db/dv, w dA/dv, w dA/dv
  } tab[kBwdGroup];
  float4 sh[LIT ? 34 : 1];  // s_d, s_d, s_s, s_s
  float4 raw[2][2 * 32];    // records, alternate chunks
  float acc[34 * kAcc];     // gradient sums of the chunk's splats
};

// Three CTAs per SM (166 registers; the four tables' transmittances, suffix sums
// and upstream gradients are 40 of them).
template <bool LIT>
__global__ void __launch_bounds__(kCompThreads, 3)
    composite_bwd_group_kernel(CompArgs A, const float4* __restrict__ out,
                               const int32_t* __restrict__ n_contrib,
                               const float4* __restrict__ dout, float4* __restrict__ grad2d,
                               float2* __restrict__ grad_shade) {
  // Behind the other kernel (which lets this one be scheduled once it runs, all
  // before it being done): a group that the other took is left without waiting
  // for it, but the grid as a whole ends behind it, as the next kernel expects.
  if (A.by_overlap && !tables_overlap(A, (int)blockIdx.z * kBwdGroup)) {
    if (blockIdx.x == 0) pdl_enter();
    return;
  }
  pdl_enter();
  using Warp = BwdGroupWarp<LIT>;
  constexpr int kAcc = Warp::kAcc;
  extern __shared__ float4 smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  Warp& S = reinterpret_cast<Warp*>(smem)[warp];
  float2* s_sh = reinterpret_cast<float2*>(reinterpret_cast<Warp*>(smem) + kWarps) + threadIdx.x;
  const int ntg = min(kBwdGroup, A.n_tf - (int)blockIdx.z * kBwdGroup);  // tables of the group
  const int L = A.lut_size;
  const WorkItem W = work_item(A, (int)blockIdx.x, warp, kBwdGroup);
  const float bx0 = W.tx0 + (float)((warp & 1) * 8), by0 = W.ty0 + (float)((warp >> 1) * 8);
  const float2 fx = dup((float)W.px), fy = make_float2((float)W.py, (float)(W.py + 4));
  // per pixel and table: transmittance behind the splats walked so far, the
  // negated suffix sum, the upstream colour gradient and n_contrib
  float2 T[kBwdGroup], nSuf[kBwdGroup], gr[kBwdGroup], gg[kBwdGroup], gb[kBwdGroup];
  int nc[kBwdGroup][2], most = 0;
#pragma unroll
  for (int t = 0; t < kBwdGroup; ++t) {
    float4 ov[2], dv4[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      ov[i] = make_float4(0.f, 0.f, 0.f, 1.f);
      dv4[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      nc[t][i] = 0;
      if (t < ntg && W.px < W.width && W.py + 4 * i < W.height) {
        const int64_t o = W.image + ((int64_t)t * W.height + W.py + 4 * i) * W.width + W.px;
        ov[i] = out[o];
        dv4[i] = dout[o];
        nc[t][i] = n_contrib[o];
      }
      most = max(most, nc[t][i]);
    }
    auto suf = [&](float4 o, float4 d) {
      return -(o.w * (A.bg0 * d.x + A.bg1 * d.y + A.bg2 * d.z + d.w));
    };
    T[t] = make_float2(ov[0].w, ov[1].w);
    gr[t] = make_float2(dv4[0].x, dv4[1].x);
    gg[t] = make_float2(dv4[0].y, dv4[1].y);
    gb[t] = make_float2(dv4[0].z, dv4[1].z);
    nSuf[t] = make_float2(suf(ov[0], dv4[0]), suf(ov[1], dv4[1]));
  }
  // the walk and its chunks as in composite_bwd_kernel
  const int wmax = __reduce_max_sync(0xffffffffu, most);
  const uint32_t* list = A.vals + W.rg.x;
  uint32_t cur = 0, next = 0;
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
    async_wait();
    const int pos = end - 1 - lane;
    const uint32_t rec = cur;
    bool hit = false;
    float4 ge, au;
    if (pos >= 0) {  // a hit under any table of the group
      ge = S.raw[side][lane];
      au = S.raw[side][32 + lane];
      float aw = 0.0f;
#pragma unroll
      for (int t = 0; t < kBwdGroup; ++t)
        if (t < ntg) aw = fmaxf(aw, splat_tf(W.lut + t * L, L, au.w, ge.w).aw);
      hit = block_hit(ge.x - bx0, ge.y - by0, Reach(au.x, au.y, au.z, power_cutoff(aw)));
    }
    const unsigned hits = __ballot_sync(0xffffffffu, hit);
    const int nh = __popc(hits), slot = __popc(hits & lanemask_lt_());
    if (hit) {
      float2 sh = make_float2(1.0f, 0.0f);
      if (LIT) sh = *s_sh;
      const float sl = (au.w >= 0.0f && au.w <= 1.0f) ? (float)(L - 1) : 0.0f;
      const float slc = LIT ? sl * sh.x : sl;  // colour slope scale
#pragma unroll
      for (int t = 0; t < kBwdGroup; ++t) {
        if (t >= ntg) continue;  // (its pixels have no contribution)
        const SplatTf tf = splat_tf(W.lut + t * L, L, au.w, ge.w);
        const float r = lerp_rn(tf.lo.x, tf.hi.x, tf.q), g = lerp_rn(tf.lo.y, tf.hi.y, tf.q),
                    b = lerp_rn(tf.lo.z, tf.hi.z, tf.q);
        const float dr = slc * (tf.hi.x - tf.lo.x), dg = slc * (tf.hi.y - tf.lo.y),
                    db = slc * (tf.hi.z - tf.lo.z),
                    da = fminf(fmaxf(ge.w * sl * (tf.hi.w - tf.lo.w), -kHuge), kHuge);
        S.tab[t].c0[slot] = make_float4(r, r, g, g);
        S.tab[t].c1[slot] = make_float4(b, b, tf.aw, tf.aw);
        S.tab[t].d0[slot] = make_float4(dr, dr, dg, dg);
        S.tab[t].d1[slot] = make_float4(db, db, da, da);
      }
      const float4 cc = clean_conic(au);
      S.u[slot] = make_float4(ge.x, ge.x, ge.y, ge.y);
      S.q[slot] = make_float4(-0.5f * cc.x, -0.5f * cc.x, -cc.y, -cc.y);
      S.r[slot] = make_float4(-0.5f * cc.z, -0.5f * cc.z, __int_as_float(pos), 0.0f);
      if (LIT) S.sh[slot] = make_float4(sh.x, sh.x, sh.y, sh.y);
    }
    if (lane == 0) {  // pads an odd count: at no pixel's list position
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      S.u[nh] = S.q[nh] = z;
      S.r[nh] = make_float4(0.f, 0.f, __int_as_float(0x7fffffff), 0.f);
#pragma unroll
      for (int t = 0; t < kBwdGroup; ++t)
        S.tab[t].c0[nh] = S.tab[t].c1[nh] = S.tab[t].d0[nh] = S.tab[t].d1[nh] = z;
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
    // two splats per step: their geometry, then table by table, then one
    // reduction for all
    for (int k = 0; k < nh; k += 2) {
      Offsets o[2];
      float2 G[2], p[2], dp[2], dvv[2], dsd[2], dss[2];  // the last four: sums over the tables
      int at[2];
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const float4 u = S.u[k + m], q = S.q[k + m], r = S.r[k + m];
        p[m] = power2(u, q, r, fx, fy, o[m]);
        at[m] = __float_as_int(r.z);
        const float2 x = mul2(p[m], dup(kLog2e));
        G[m] = make_float2(ex2_approx(x.x), ex2_approx(x.y));
        dp[m] = dvv[m] = dsd[m] = dss[m] = dup(0.0f);
      }
      bool some = false;
#pragma unroll
      for (int t = 0; t < kBwdGroup; ++t) {
        const auto& tab = S.tab[t];
        float2 raw2[2], al[2];
        bool ok[2][2];
        float4 c1[2];
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          c1[m] = tab.c1[k + m];
          raw2[m] = mul2(hi2(c1[m]), G[m]);
          al[m] = make_float2(fminf(kAlphaMax, raw2[m].x), fminf(kAlphaMax, raw2[m].y));
          ok[m][0] = at[m] < nc[t][0] && !(p[m].x > 0.0f) && !(al[m].x < kAlphaMin);
          ok[m][1] = at[m] < nc[t][1] && !(p[m].y > 0.0f) && !(al[m].y < kAlphaMin);
        }
        if (!__any_sync(0xffffffffu, ok[0][0] || ok[0][1] || ok[1][0] || ok[1][1])) continue;
        some = true;
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const float4 c0 = tab.c0[k + m], s0 = tab.d0[k + m], s1 = tab.d1[k + m];
          const float2 om = sub2(dup(1.0f), al[m]);
          const float2 rr = make_float2(rcp_approx(om.x), rcp_approx(om.y));
          const float2 cgu =
              fma2(lo2(c1[m]), gb[t], fma2(hi2(c0), gg[t], mul2(lo2(c0), gr[t])));
          const float2 h =
              fma2(lo2(s1), gb[t], fma2(hi2(s0), gg[t], mul2(lo2(s0), gr[t])));
          const float2 Ti = mul2(T[t], rr);  // transmittance in front of the splat
          const float2 wgt = mul2(al[m], Ti);
          float2 cgd = cgu;
          if (LIT) {
            const float4 sh = S.sh[k + m];
            const float2 gs = add2(add2(gr[t], gg[t]), gb[t]);
            cgd = fma2(lo2(sh), cgu, mul2(hi2(sh), gs));
            const float2 d = mul2(wgt, cgu), s = mul2(wgt, gs);
            dsd[m] = add2(dsd[m], make_float2(ok[m][0] ? d.x : 0.0f, ok[m][1] ? d.y : 0.0f));
            dss[m] = add2(dss[m], make_float2(ok[m][0] ? s.x : 0.0f, ok[m][1] ? s.y : 0.0f));
          }
          const float2 da = fma2(Ti, cgd, mul2(nSuf[t], rr));
          // below the clamp alpha follows the exponent and the opacity slope (the
          // product is masked, not a factor: A w may be infinite)
          float2 mg = mul2(da, G[m]), cv = mul2(wgt, h);
          const bool free[2] = {ok[m][0] && raw2[m].x <= kAlphaMax,
                                ok[m][1] && raw2[m].y <= kAlphaMax};
          const float2 e = mul2(hi2(c1[m]), mg);
          dp[m] = add2(dp[m], make_float2(free[0] ? e.x : 0.0f, free[1] ? e.y : 0.0f));
          mg.x = free[0] ? mg.x : 0.0f;
          mg.y = free[1] ? mg.y : 0.0f;
          cv.x = ok[m][0] ? cv.x : 0.0f;
          cv.y = ok[m][1] ? cv.y : 0.0f;
          dvv[m] = add2(dvv[m], fma2(hi2(s1), mg, cv));
          if (ok[m][0]) {
            nSuf[t].x = __fmaf_rn(-cgd.x, wgt.x, nSuf[t].x);
            T[t].x = Ti.x;
          }
          if (ok[m][1]) {
            nSuf[t].y = __fmaf_rn(-cgd.y, wgt.y, nSuf[t].y);
            T[t].y = Ti.y;
          }
        }
      }
      if (!some) continue;
      constexpr int kSum = LIT ? 6 : 4;
      float v[2 * kSum];
#pragma unroll
      for (int m = 0; m < 2; ++m) {
        const float2 y1 = mul2(dp[m], o[m].dy), y2 = mul2(dp[m], o[m].dyy);
        v[m * kSum] = dp[m].x + dp[m].y;
        v[m * kSum + 1] = dvv[m].x + dvv[m].y;
        if (LIT) {
          v[m * kSum + 2] = dsd[m].x + dsd[m].y;
          v[m * kSum + 5] = dss[m].x + dss[m].y;
        }
        v[m * kSum + kSum / 2] = y1.x + y1.y;
        v[m * kSum + kSum / 2 + 1] = y2.x + y2.y;
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
}

template <bool LIT>
veg_status launch_bwd_group(const CompArgs& A, int n_views, const float4* out, const int32_t* nc,
                            const float4* dout, float4* grad2d, float2* grad_shade,
                            cudaStream_t stream) {
  const size_t smem =
      kWarps * sizeof(BwdGroupWarp<LIT>) + (LIT ? (size_t)kCompThreads * sizeof(float2) : 0);
  auto kern = composite_bwd_group_kernel<LIT>;
  static SmemRecord configured;
  veg_status st = prepare_smem(kern, smem, configured, false);
  if (st != VEG_OK) return st;
  dim3 grid = comp_grid(A, n_views);
  grid.z = (grid.z + kBwdGroup - 1) / kBwdGroup;
  launch_k(kern, grid, kCompThreads, smem, stream, A, out, nc, dout, grad2d, grad_shade);
  count_launch();
  return launch_status();
}

}  // namespace

}  // namespace veg
