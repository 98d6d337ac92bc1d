// Mixed-precision near field (included by fmm.cu).
//
// Every point of the target tree carries its offset from its own leaf centre as FP32 hi + lo pairs
// (k_split_points, once per evaluation, one array per component).  A source of a near leaf whose centre lies
// delta * h away is moved into the target leaf's frame by an exact FP32 two-sum with h = hh + hl.  Sources are staged
// with cp.async, one chunk ahead of the one being summed.  Sums over 64 sources are folded into
// Kahan-compensated FP32 totals; no FP64 in the pair loop.
//
// A pair is 17 FP32 operations (10 without the field; 23 and 16 for leaves that touch) and two special-function
// operations (12 clocks of that unit per warp).  Two sources ride in one 64-bit register pair
// (add / mul / fma.f32x2: two lanes' worth of FP32 per issue slot), so that the 17 operations no longer fill the
// issue slots and the special functions, loads and loop run beside them.  Bound: latency ahead of any pipe.  N = 100,000, p = 10
// with the field: FP32 pipe busy 60 % of the active cycles (a packed operation takes two), special functions 24 %, an
// instruction issued in 49 % of the slots; warps wait for their own operations (1.8 cycles per issue), the block's barrier
// (1.4) and the FP32 pipe (1.0), because 127 registers leave 16 warps an SM.  Without the field 53 %, 33 % and 53 %.
// N = 1M, 10.3e9 pairs: 8.3 ms, 30 TFLOP/s at 24 a pair, 38 % of the measured FP32 peak.  The sources are packed, not
// the targets: target coordinates are duplicated once per chunk, a packed source is one load.
// One CTA of 4 warps per leaf: groups of 64 targets (two per lane), and the chunks of the near leaves
// split over the warps a group has; a last group of at most 32, 16, ... targets gives each pair of targets 2, 4,
// ... lanes.  Sums over the parts in a fixed order in FP64.
#pragma once

__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

// pts: 7 arrays of ld floats: x, y, z hi, charge, x, y, z lo
__global__ void k_split_points(const uint32_t *d_nb, const uint64_t *bkey, const uint32_t *bstart,
                               const uint32_t *bcount, const double *x, const double *y, const double *z,
                               const double *q, Geo geo, float *pts, int64_t ld) {
  const uint32_t box = blockIdx.x;
  if (box >= *d_nb) return;
  double cx, cy, cz;
  box_center(bkey[box], geo, cx, cy, cz);
  const uint32_t st = bstart[box], cnt = bcount[box];
  for (uint32_t j = threadIdx.x; j < cnt; j += blockDim.x) {
    const uint32_t k = st + j;
    const double ox = x[k] - cx, oy = y[k] - cy, oz = z[k] - cz;
    const float hx = (float)ox, hy = (float)oy, hz = (float)oz;
    pts[k] = hx;
    pts[ld + k] = hy;
    pts[2 * ld + k] = hz;
    pts[3 * ld + k] = (float)q[k];
    pts[4 * ld + k] = (float)(ox - (double)hx);
    pts[5 * ld + k] = (float)(oy - (double)hy);
    pts[6 * ld + k] = (float)(oz - (double)hz);
  }
}

__device__ __forceinline__ void two_sum_shift(float hi, float lo, float b, float bl, float &oh, float &ol) {
  // (hi + lo) + (b + bl) with b exact: oh + ol, the rounding error of hi + b kept in ol
  const float a = hi + b;
  const float bb = a - hi;
  const float e = (hi - (a - bb)) + (b - bb);
  oh = a;
  ol = (lo + bl) + e;
}

__device__ __forceinline__ void kahan_add(float &s, float &c, float v) {
  const float y = v - c;
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}

// 2^x on the special-function unit (max. relative error about 2^-22)
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 1/sqrt(x) on the special-function unit (max. relative error about 2^-22.9; subnormal inputs
// flushed to zero, which cannot occur for r^2 of distinct points at the FP32 offsets used here)
__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

constexpr int P2P_WARPS = 4, P2P_CH = 128, P2P_GROUP = 64;  // warps per leaf, sources per chunk, targets per group
// Sources between two folds into the compensated totals.  A lane adds P2P_FOLD / 2 of them to a running FP32 sum (fewer where
// several lanes share a target), whose rounding grows with that number: a fold per chunk of 128, which may span
// leaves, left sums of small leaves 12 % further from FP64 than a fold per leaf (four layers, N = 10,000, strong screening:
// 1.55e-7 against 1.38e-7), a fold per 64 gives 1.17e-7.  Its cost, 40 of some 1,400 instructions, is 0.3 % of the kernel (N = 1M,
// beside the far field, 11.65 -> 11.66 ms; N = 2.86M 32.29 -> 32.52).
constexpr int P2P_FOLD = 64;
constexpr float P2P_FAR = 1e18f;  // x of the records that fill a chunk up to fours (charge 0)

// e^{-lambda r} = 2^{(-lambda log2 e) r}; field factor (1 + lambda r) / r^2 = (1/r)(1/r + lambda).
// NEAR: the leaf itself and the boxes that touch it: compensated coordinates, the r = 0 self pair dropped by a
// select.  Otherwise a box at least one box away: r >= h, so the FP32 rounding of the plain
// differences, ~2^-23 of 3h, is below 1e-7 of r and the low parts are not used.  Two targets per
// lane.  Differences are source - target (the sign is put right at the output).
template <bool FIELD, bool NEAR>
__device__ __forceinline__ void p2p_f32_chunk(const float *__restrict__ s, int nquad, int sub, int nsub,
                                              const float2 (&ph)[2][3], const float2 (&pl)[2][3], float2 nl2, float2 lam,
                                              float2 (&ap)[2], float2 (&ax)[2], float2 (&ay)[2], float2 (&az)[2]) {
#pragma unroll 1
  for (int j = sub; j < nquad; j += nsub) {
    const float4 *v = (const float4 *)s + j;
    constexpr int LD = P2P_CH / 4;
    const float4 vx = v[0], vy = v[LD], vz = v[2 * LD], vq = v[3 * LD];
    float4 ux, uy, uz;
    if (NEAR) {
      ux = v[4 * LD];
      uy = v[5 * LD];
      uz = v[6 * LD];
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float2 sx = h ? make_float2(vx.z, vx.w) : make_float2(vx.x, vx.y);
      const float2 sy = h ? make_float2(vy.z, vy.w) : make_float2(vy.x, vy.y);
      const float2 sz = h ? make_float2(vz.z, vz.w) : make_float2(vz.x, vz.y);
      const float2 sq = h ? make_float2(vq.z, vq.w) : make_float2(vq.x, vq.y);
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        float2 dx = add2(sx, ph[t][0]), dy = add2(sy, ph[t][1]), dz = add2(sz, ph[t][2]);
        if (NEAR) {
          dx = add2(dx, add2(h ? make_float2(ux.z, ux.w) : make_float2(ux.x, ux.y), pl[t][0]));
          dy = add2(dy, add2(h ? make_float2(uy.z, uy.w) : make_float2(uy.x, uy.y), pl[t][1]));
          dz = add2(dz, add2(h ? make_float2(uz.z, uz.w) : make_float2(uz.x, uz.y), pl[t][2]));
        }
        const float2 r2 = fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
        float2 ri = make_float2(rsqrt_approx(r2.x), rsqrt_approx(r2.y));
        if (NEAR) {
          ri.x = r2.x > 0.f ? ri.x : 0.f;
          ri.y = r2.y > 0.f ? ri.y : 0.f;
        }
        const float2 a = mul2(nl2, mul2(r2, ri));
        const float2 e = mul2(sq, make_float2(ex2_approx(a.x), ex2_approx(a.y)));
        ap[t] = fma2(e, ri, ap[t]);  // the same with and without the field
        if (FIELD) {
          const float2 w = mul2(e, ri);
          const float2 f = mul2(mul2(w, ri), add2(ri, lam));
          ax[t] = fma2(f, dx, ax[t]);
          ay[t] = fma2(f, dy, ay[t]);
          az[t] = fma2(f, dz, az[t]);
        }
      }
    }
  }
}

// The near leaves of one leaf as two streams of sources: first those of the leaf itself and the leaves that
// touch it, then the others; chunks of P2P_CH consecutive sources of one stream.
struct P2PNear {
  uint32_t start[NNEAR], pre[NNEAR + 1];  // first point, position in the streams
  int off[NNEAR];                         // (dx + 2) | (dy + 2) << 3 | (dz + 2) << 6
  uint32_t s_near, s_all;                 // sources of the first stream, of both
};
constexpr int P2P_OFF0 = 2 | 2 << 3 | 2 << 6;

// one warp: nt targets of the leaf (from point first) against chunks part, part + nparts, ... of its near
// leaves.  Two targets per lane, tl and tl + 2^lg; 2^lg lanes hold them all and 32 / 2^lg such sets split the
// sources.  A chunk is staged raw, one ahead, and then moved into the target leaf's frame in place by the lanes that
// staged it, so that a chunk may span leaves (small leaves had a chunk and its overhead each).  Sums (FP64) of
// target j into out[value][j].  One loop body per stream and no other variants: six (one or two targets per
// lane, self / touching / apart) had the instruction cache as their bound.
template <bool FIELD>
__device__ __forceinline__ void p2p_warp_pass(const P2PJob &J, int lane, uint32_t first, int nt, int part, int nparts,
                                              float (*buf)[7 * P2P_CH], const P2PNear &nb, double (*out)[P2P_GROUP]) {
  const float *pts = J.pts;
  const int64_t ld = J.ld;
  const float hh = J.hh, hl = J.hl;
  int lg = 5;
  while (lg > 0 && (2 << (lg - 1)) >= nt) --lg;
  const int tl = lane & ((1 << lg) - 1), sub = lane >> lg, nsub = 32 >> lg;
  float2 ph[2][3];
#pragma unroll
  for (int t = 0; t < 2; ++t)
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const float h = -pts[d * ld + first + min(tl + (t << lg), nt - 1)];
      ph[t][d] = make_float2(h, h);
    }
  const int nchn = (int)((nb.s_near + P2P_CH - 1) / P2P_CH),
            nch = nchn + (int)((nb.s_all - nb.s_near + P2P_CH - 1) / P2P_CH);
  auto range = [&](int c, uint32_t &g0) {  // first source of chunk c, number of its sources
    g0 = c < nchn ? (uint32_t)c * P2P_CH : nb.s_near + (uint32_t)(c - nchn) * P2P_CH;
    return (int)min((uint32_t)P2P_CH, (c < nchn ? nb.s_near : nb.s_all) - g0);
  };
  int k = 0;  // this lane's near leaf: its sources ascend
  // stage chunk c raw; the offsets of this lane's four sources, a byte and a bit each
  auto issue = [&](int c, float *b) {
    uint32_t g0;
    const int nn = range(c, g0), na = c < nchn ? 7 : 4;
    uint64_t offs = 0;
#pragma unroll
    for (int a = 0; a < P2P_CH / 32; ++a) {
      const int j = lane + 32 * a;
      int o = P2P_OFF0;
      if (j < nn) {
        const uint32_t g = g0 + (uint32_t)j;
        while (nb.pre[k + 1] <= g) ++k;
        o = nb.off[k];
        const float *f = pts + nb.start[k] + (g - nb.pre[k]);
#pragma unroll
        for (int v = 0; v < 7; ++v)
          if (v < na) cp_async4(b + v * P2P_CH + j, f + v * ld);
      } else if (j < ((nn + 3) & ~3)) {  // records that fill the last four: charge 0, far away
#pragma unroll
        for (int v = 0; v < 7; ++v) b[v * P2P_CH + j] = v == 0 ? P2P_FAR : 0.f;
      }
      offs |= (uint64_t)o << (16 * a);
    }
    cp_commit();
    return offs;
  };
  float tot[2][4], cmp[2][4];
#pragma unroll
  for (int t = 0; t < 2; ++t)
#pragma unroll
    for (int v = 0; v < 4; ++v) tot[t][v] = cmp[t][v] = 0.f;
  const float2 lam = make_float2(J.lam, J.lam);
  const float nl = -J.lam * 1.44269504088896341f;
  const float2 nl2 = make_float2(nl, nl);
  int b = 0;
  uint64_t offs = part < nch ? issue(part, buf[0]) : 0;
#pragma unroll 1
  for (int c = part; c < nch; c += nparts, b ^= 1) {
    const uint64_t mine = offs;
    if (c + nparts < nch) {
      offs = issue(c + nparts, buf[b ^ 1]);
      cp_wait1();
    } else {
      cp_wait0();
    }
    // this lane's sources into the target leaf's frame: + (dx, dy, dz) h
    const bool near = c < nchn;
    uint32_t g0;
    const int nn = range(c, g0);
#pragma unroll
    for (int a = 0; a < P2P_CH / 32; ++a) {
      const int o = (int)(mine >> (16 * a)) & 0x1ff;
      if (o == P2P_OFF0) continue;  // the leaf itself, or no source
      float *r = buf[b] + lane + 32 * a;
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float m = (float)(((o >> (3 * d)) & 7) - 2);
        if (near) two_sum_shift(r[d * P2P_CH], r[(4 + d) * P2P_CH], m * hh, m * hl, r[d * P2P_CH], r[(4 + d) * P2P_CH]);
        else r[d * P2P_CH] = fmaf(m, hh, r[d * P2P_CH]);
      }
    }
    __syncwarp();
    float2 pl[2][3];
    if (near) {
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int d = 0; d < 3; ++d) {
          const float l = -pts[(4 + d) * ld + first + min(tl + (t << lg), nt - 1)];
          pl[t][d] = make_float2(l, l);
        }
    }
    const int nq = (nn + 3) >> 2, step = max(P2P_FOLD / 4, nsub);  // at least a quad per lane
#pragma unroll 1
    for (int j0 = 0; j0 < nq; j0 += step) {
      float2 ap[2], ax[2], ay[2], az[2];
#pragma unroll
      for (int t = 0; t < 2; ++t) ap[t] = ax[t] = ay[t] = az[t] = make_float2(0.f, 0.f);
      const int j1 = min(nq, j0 + step);
      if (near) p2p_f32_chunk<FIELD, true>(buf[b], j1, j0 + sub, nsub, ph, pl, nl2, lam, ap, ax, ay, az);
      else p2p_f32_chunk<FIELD, false>(buf[b], j1, j0 + sub, nsub, ph, pl, nl2, lam, ap, ax, ay, az);
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        kahan_add(tot[t][0], cmp[t][0], ap[t].x + ap[t].y);
        if (FIELD) {
          kahan_add(tot[t][1], cmp[t][1], ax[t].x + ax[t].y);
          kahan_add(tot[t][2], cmp[t][2], ay[t].x + ay[t].y);
          kahan_add(tot[t][3], cmp[t][3], az[t].x + az[t].y);
        }
      }
    }
    __syncwarp();  // buffer b is refilled by the next issue
  }
#pragma unroll
  for (int t = 0; t < 2; ++t)
#pragma unroll
    for (int v = 0; v < (FIELD ? 4 : 1); ++v) {
      double s = (double)tot[t][v] - (double)cmp[t][v];
      for (int o = 16; o >= (1 << lg); o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (sub == 0) out[v][tl + (t << lg)] = s;
    }
}

template <bool FIELD>
__global__ void __launch_bounds__(32 * P2P_WARPS, 4) k_p2p_free_f32(const P2PJob *jobs, int njobs) {
  __shared__ __align__(16) float buf_[P2P_WARPS][2][7 * P2P_CH];
  __shared__ double out_[P2P_WARPS][FIELD ? 4 : 1][P2P_GROUP];
  __shared__ P2PNear nb;
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].block0 <= (int64_t)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  const P2PJob &J = jobs[lo];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t box = (uint32_t)((int64_t)blockIdx.x - J.block0);
  if (box >= *J.d_nb) return;
  const uint32_t tst = J.bstart[box], tcnt = J.bcount[box];
  if (w == 0) {
    int nnb = 0;
    uint32_t at = 0;
    for (int far = 0; far < 2; ++far) {
      for (int o0 = 0; o0 < NNEAR; o0 += 32) {
        const int o = o0 + lane;
        int dx = 0, dy = 0, dz = 0, sb = -1;
        if (o < NNEAR) {
          near_decode(o, dx, dy, dz);
          if ((cheb3(dx, dy, dz) > 1) == (far != 0)) sb = J.ulist[(size_t)box * NNEAR + o];
        }
        const uint32_t cnt = sb >= 0 ? J.bcount[sb] : 0u;
        uint32_t x = cnt;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t y = __shfl_up_sync(0xffffffffu, x, d);
          if (lane >= d) x += y;
        }
        const unsigned m = __ballot_sync(0xffffffffu, cnt > 0);
        if (cnt > 0) {
          const int k = nnb + __popc(m & ((1u << lane) - 1u));
          nb.start[k] = J.bstart[sb];
          nb.pre[k] = at + x - cnt;
          nb.off[k] = (dx + 2) | (dy + 2) << 3 | (dz + 2) << 6;
        }
        nnb += __popc(m);
        at += __shfl_sync(0xffffffffu, x, 31);
      }
      if (lane == 0) (far ? nb.s_all : nb.s_near) = at;
    }
    if (lane == 0) nb.pre[nnb] = at;
  }
  __syncthreads();
  for (uint32_t t0 = 0; t0 < tcnt;) {
    // groups of this round: two of 64 targets with two warps each, or one with all four
    const uint32_t left = tcnt - t0;
    const int ng = left > P2P_GROUP ? 2 : 1, nparts = P2P_WARPS / ng;
    const int g = ng == 2 ? w & 1 : 0, part = ng == 2 ? w >> 1 : w;
    const uint32_t first = t0 + P2P_GROUP * g;
    const int nt = (int)min((uint32_t)P2P_GROUP, tcnt - first);
    p2p_warp_pass<FIELD>(J, lane, tst + first, nt, part, nparts, buf_[w], nb, out_[w]);
    __syncthreads();
    // thread -> target; the parts of its group in order
    const uint32_t mine = threadIdx.x;
    if (mine < (uint32_t)(P2P_GROUP * ng) && t0 + mine < tcnt) {
      const int mg = (int)mine / P2P_GROUP, mt = (int)mine % P2P_GROUP;
      const uint32_t i = J.src[tst + t0 + mine];
#pragma unroll
      for (int v = 0; v < (FIELD ? 4 : 1); ++v) {
        double s = 0.0;
        for (int q = 0; q < nparts; ++q) s += out_[ng == 2 ? mg + 2 * q : q][v][mt];
        if (v == 0) J.phi[i] += J.scale * s;
        else J.field[3 * (size_t)i + v - 1] -= J.scale * s;  // sums of source - target
      }
    }
    __syncthreads();
    t0 += (uint32_t)(P2P_GROUP * ng);
  }
}
