// Packed double-float pair arithmetic shared by the direct sums (operators.cu) and the treecode
// (treecode.cu).
#pragma once

#include <climits>

#include "common.cuh"
#include "dfloat.cuh"

namespace rbs {

// Double-float pair sums with two sources per instruction (__fadd2_rn, __fmul2_rn, __ffma2_rn, each two
// round-to-nearest float32 operations, so the error-free transformations stay exact per source).
struct df2 {
  float2 h, l;
};
__device__ __forceinline__ float2 ng2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 dup2(float a) { return make_float2(a, a); }
__device__ __forceinline__ df2 two_sum2(float2 a, float2 b) {
  const float2 s = __fadd2_rn(a, b);
  const float2 bb = __fadd2_rn(s, ng2(a));
  const float2 e = __fadd2_rn(__fadd2_rn(a, ng2(__fadd2_rn(s, ng2(bb)))), __fadd2_rn(b, ng2(bb)));
  return {s, e};
}
__device__ __forceinline__ df2 mul2(df2 a, df2 b) {
  const float2 p = __fmul2_rn(a.h, b.h);
  float2 e = __ffma2_rn(a.h, b.h, ng2(p));
  e = __ffma2_rn(a.h, b.l, e);
  e = __ffma2_rn(a.l, b.h, e);
  return {p, e};
}
__device__ __forceinline__ void acc2_add(df2& acc, df2 v) {
  const df2 s = two_sum2(acc.h, v.h);
  acc.h = s.h;
  acc.l = __fadd2_rn(acc.l, __fadd2_rn(s.l, v.l));
}
// the two lanes' double-float values added into one (unnormalised) pair
__device__ __forceinline__ dflt fold2(const df2& a) {
  const dflt s = df_two_sum(a.h.x, a.h.y);
  return {s.h, s.l + (a.l.x + a.l.y)};
}

// Bias of a sum of products whose terms are bounded: partial sums of d . q never exceed |d| |q|, so with
// B >= 2 |d| |q| added first every partial sum stays within [B / 2, 2 B], where the difference of
// successive partial sums is exact (Sterbenz) and one multiply-add gives what a step rounded off:
//   s' = fl(s + a b),  e = a b - (s' - s).
// A product and its addition then take three operations where a two-product and a two-sum take eight.
// kBiasFactor is 2 with a margin for the rounded norms.
constexpr float kBiasFactor = 2.002f;

// kBiasFactor |q|, without overflow or underflow of the squares: a plain root of their sum is infinite from 2e19 up (the
// bias less a partial sum then is not a number) and loses its digits from 1e-19 down (the bias no longer bounds the
// partial sums, whose rounding falls to float32's).  The double-float weighted densities carry it in hi's fourth component.
__device__ __forceinline__ float bias_bound(float x, float y, float z) { return kBiasFactor * norm3df(x, y, z); }

__device__ __forceinline__ df2 norm2(float2 h, float2 l) {  // h + l, renormalised
  const float2 s = __fadd2_rn(h, l);
  return {s, __fadd2_rn(l, ng2(__fadd2_rn(s, ng2(h))))};
}
// a0 b0 + a1 b1 + a2 b2 by biased accumulation (B as above); renormalised.
__device__ __forceinline__ df2 bdot2(df2 a0, df2 b0, df2 a1, df2 b1, df2 a2, df2 b2, float2 B) {
  const float2 s0 = __ffma2_rn(a0.h, b0.h, B), s1 = __ffma2_rn(a1.h, b1.h, s0), s2 = __ffma2_rn(a2.h, b2.h, s1);
  float2 e0 = __ffma2_rn(a0.h, b0.h, __fadd2_rn(B, ng2(s0)));
  float2 e1 = __ffma2_rn(a1.h, b1.h, __fadd2_rn(s0, ng2(s1)));
  float2 e2 = __ffma2_rn(a2.h, b2.h, __fadd2_rn(s1, ng2(s2)));
  e0 = __ffma2_rn(a0.l, b0.h, __ffma2_rn(a0.h, b0.l, e0));
  e1 = __ffma2_rn(a1.l, b1.h, __ffma2_rn(a1.h, b1.l, e1));
  e2 = __ffma2_rn(a2.l, b2.h, __ffma2_rn(a2.h, b2.l, e2));
  return norm2(__fadd2_rn(s2, ng2(B)), __fadd2_rn(__fadd2_rn(e0, e1), e2));
}

// Odd powers of 1 / r from r^2 = h + l and the hardware estimate y0 = (1 / r)(1 + O(2^-22)): with
// t = r^2 y0^2 - 1, below 2^-21, (1 / r)^k = y0^k (1 - k t / 2 + k (k + 2) t^2 / 8) but for k (k + 2) (k + 4) t^3 / 48,
// 2^-64 for k = 1, 2^-62 for k = 3 and 2^-60 for k = 5.  What limits the powers is their evaluation: those of y0 are
// float32 pairs, and the series, in float32, multiplies a product once, at its end (2^-24 of t: 44 bits and more).
struct inv_powers {
  float2 y0, q, qe, t;  // q + qe = y0^2
  __device__ __forceinline__ inv_powers(float2 r2h, float2 r2l, float2 y) : y0(y) {
    q = __fmul2_rn(y, y);
    qe = __ffma2_rn(y, y, ng2(q));
    t = __ffma2_rn(r2l, q, __ffma2_rn(r2h, qe, __ffma2_rn(r2h, q, dup2(-1.0f))));
  }
  __device__ __forceinline__ float2 series(float lin, float quad) const {
    return __fmul2_rn(t, __ffma2_rn(t, dup2(quad), dup2(lin)));
  }
  __device__ __forceinline__ float2 w3() const { return series(-1.5f, 1.875f); }
  __device__ __forceinline__ float2 w5() const { return series(-2.5f, 4.375f); }
  __device__ __forceinline__ df2 y3() const {
    const float2 h = __fmul2_rn(q, y0);
    return {h, __ffma2_rn(qe, y0, __ffma2_rn(q, y0, ng2(h)))};
  }
  __device__ __forceinline__ df2 inv() const { return {y0, __fmul2_rn(y0, series(-0.5f, 0.375f))}; }
};

// How a tile forms separations: by two-sums, the same with sources masked per target particle (DfSkip), or on a
// common grid (df_tile); kDfNone: every source of the tile is left out for every target.
enum DfMode { kDfPlain = 0, kDfMask = 1, kDfGrid = 2, kDfNone = 3 };

// One component of the separation from the target's coordinate and the source's negated one.
template <int MODE>
__device__ __forceinline__ df2 df_separation(df2 x, df2 y) {
  if (MODE == kDfGrid) return norm2(__fadd2_rn(x.h, y.h), __fadd2_rn(x.l, y.l));
  df2 d = two_sum2(x.h, y.h);
  d.l = __fadd2_rn(d.l, __fadd2_rn(x.l, y.l));
  return d;
}

// Powers of 1 / r for the separation d, and R = r^2 in float32; MODE kDfMask zeroes them for the sources whose
// mask holds the target's bit.
template <int MODE>
__device__ __forceinline__ inv_powers df_inv_powers(const df2 (&d)[3], int2 mask, int bit, float2& R) {
  // r^2 by biased accumulation over 5/4 of its own float32 value R (over R itself the sum can round to
  // just above 2 R, where the difference from R is inexact)
  R = __ffma2_rn(d[2].h, d[2].h, __ffma2_rn(d[1].h, d[1].h, __fmul2_rn(d[0].h, d[0].h)));
  float2 y0 = make_float2(rsqrt_hw(R.x), rsqrt_hw(R.y));
  if (MODE == kDfMask) {  // every power of 1 / r becomes zero
    if (mask.x & bit) y0.x = 0.0f;
    if (mask.y & bit) y0.y = 0.0f;
  }
  const float2 Rb = __fmul2_rn(dup2(1.25f), R);
  const float2 s0 = __ffma2_rn(d[0].h, d[0].h, Rb), s1 = __ffma2_rn(d[1].h, d[1].h, s0), s2 = __ffma2_rn(d[2].h, d[2].h, s1);
  float2 e0 = __ffma2_rn(d[0].h, d[0].h, __fadd2_rn(Rb, ng2(s0)));
  float2 e1 = __ffma2_rn(d[1].h, d[1].h, __fadd2_rn(s0, ng2(s1)));
  float2 e2 = __ffma2_rn(d[2].h, d[2].h, __fadd2_rn(s1, ng2(s2)));
  e0 = __ffma2_rn(__ffma2_rn(dup2(2.0f), d[0].h, d[0].l), d[0].l, e0);
  e1 = __ffma2_rn(__ffma2_rn(dup2(2.0f), d[1].h, d[1].l), d[1].l, e1);
  e2 = __ffma2_rn(__ffma2_rn(dup2(2.0f), d[2].h, d[2].l), d[2].l, e2);
  return inv_powers(__fadd2_rn(s2, ng2(Rb)), __fadd2_rn(__fadd2_rn(e0, e1), e2), y0);
}

// One target against two sources, KIND 0 traction into acc, 1 Stokeslet into acc, 2 traction into acc and
// Stokeslet into acc2; fb = bias_bound of the sources.  With two-sums 221 float32 operations
// for both kernels, 154 for the traction alone and 139 for the Stokeslet alone; 9 fewer on the grid.
template <int KIND, int MODE>
__device__ __forceinline__ void pair2_df(const df2 (&y)[3], const df2 (&den)[3], float2 fb, int2 mask,
                                         const df2 (&xt)[3], const df2 (&nt)[3], int bit, df2 (&acc)[3], df2 (&acc2)[3]) {
  df2 d[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) d[c] = df_separation<MODE>(xt[c], y[c]);
  float2 R;
  const inv_powers p = df_inv_powers<MODE>(d, mask, bit, R);
  const float2 y0 = p.y0;
  const float2 r = __fmul2_rn(R, y0);
  const df2 rr = bdot2(d[0], den[0], d[1], den[1], d[2], den[2], __fmul2_rn(r, fb));
  const df2 a = mul2(rr, p.y3());  // r . q / r^3 but for the series
  if (KIND == 0 || KIND == 2) {
    const df2 rn = bdot2(d[0], nt[0], d[1], nt[1], d[2], nt[2], __fmul2_rn(r, dup2(kBiasFactor)));
    df2 ck = mul2(a, mul2(rn, df2{p.q, p.qe}));
    ck.l = __ffma2_rn(p.w5(), ck.h, ck.l);
#pragma unroll
    for (int c = 0; c < 3; ++c) acc2_add(acc[c], mul2(ck, d[c]));
  }
  if (KIND == 1 || KIND == 2) {
    // q / r + (r . q) r / r^3, each component bounded by 2 |q| / r: biased by twice that
    const df2 cs = {a.h, __ffma2_rn(p.w3(), a.h, a.l)};
    const df2 inv = p.inv();
    const float2 B = __fmul2_rn(__fmul2_rn(dup2(2.0f), y0), fb);
    df2(&as)[3] = KIND == 2 ? acc2 : acc;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float2 u = __ffma2_rn(cs.h, d[c].h, B), v = __ffma2_rn(den[c].h, inv.h, u);
      float2 f = __ffma2_rn(cs.h, d[c].h, __fadd2_rn(B, ng2(u)));
      float2 g = __ffma2_rn(den[c].h, inv.h, __fadd2_rn(u, ng2(v)));
      f = __ffma2_rn(cs.l, d[c].h, __ffma2_rn(cs.h, d[c].l, f));
      g = __ffma2_rn(den[c].l, inv.h, __ffma2_rn(den[c].h, inv.l, g));
      acc2_add(as[c], df2{__fadd2_rn(v, ng2(B)), __fadd2_rn(f, g)});
    }
  }
}

constexpr int kTileDf = 64;
constexpr int kTileDfFloats = 14 * kTileDf;

// ------------------------------------------------------------------------------------------
// A warp's tile of up to kTileDf sources against its 32 targets (one a lane): the double-float sums of
// both the direct and the treecode kernels.  Lane l stages sources sidx[0] (tile slot l) and sidx[1]
// (slot 32 + l), filled in all, into the warp's kTileDfFloats floats of shared memory.
//
// Where every source is at least a quarter of the tile's extent away from the targets, coordinates are
// split so that every hi part of the tile, sources and targets, is a multiple of g = 2^-24 times the power of
// two above the largest separation: differences of hi parts are exact without a two-sum, and the lo parts
// (at most g / 2) keep the separation within a few times 2^-50 of itself.  Closer tiles take two-sums.
// split: each half-warp holds the same 16 targets and takes its half of the tile.  xm = the
// warp's largest target coordinate; totals go to tot (and tot2 for KIND 2).
//
// Sources on a target's own particle, and on the particles near it, are left out (the near corrections add the
// latter's upsampled contribution).  Near terms grow as the inverse square of a gap, and what a sum adds
// another one removes only to its own rounding of their separations: with a pair of spheres 0.003 apart a pass that
// did so was 1.5e-9 of the right-hand side away from its residual.
struct DfSkip {
  const int* first;   // per particle, its first near pair
  const int2* near;   // near pairs (target, source), by target
};
// The part of it that belongs to a warp's targets, in shared memory (the pair loops have no register to spare): one of
// the first 32 near sources of particles lo and lo + 1 per lane (-1: none), lo and hi, and whether there are others.
constexpr int kDfSkipInts = 68;
__device__ __forceinline__ void df_skip_targets(const DfSkip& skip, int lo, int hi, int* sk) {
  const int lane = threadIdx.x & 31;
  const int e0 = skip.first[lo], n0 = skip.first[lo + 1], n1 = hi > lo ? skip.first[lo + 2] : n0;
  __syncwarp();  // the previous unit's reads are done
  sk[lane] = e0 + lane < n0 ? skip.near[e0 + lane].y : -1;
  sk[32 + lane] = n0 + lane < n1 ? skip.near[n0 + lane].y : -1;
  if (lane == 0) {
    sk[64] = lo;
    sk[65] = hi;  // a particle has 12 nodes at least: at most lo + 3
    sk[66] = n0 - e0 > 32 || n1 - n0 > 32 || hi > lo + 1;
  }
  __syncwarp();
}
// Whether a tile of nodes of particles tlo to thi may hold a source to leave out.
__device__ __forceinline__ bool df_skip_any(const int* sk, int tlo, int thi) {
  const int a = sk[threadIdx.x & 31], b = sk[32 + (threadIdx.x & 31)];
  return __any_sync(0xffffffffu, (a >= tlo && a <= thi) || (b >= tlo && b <= thi)) || (thi >= sk[64] && tlo <= sk[65]) ||
         sk[66];
}

__device__ __forceinline__ float warp_max_abs(float v) {  // of non-negative values
  return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}

__device__ __forceinline__ float warp_min_abs(float v) {
  return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v)));
}

template <int KIND, int MODE>
__device__ __forceinline__ void df_tile_pairs(const float (*sa)[kTileDf], const int* smask, int l0, int l1, const df2 (&xt)[3],
                                              const df2 (&nt)[3], int bit, df2 (&acc)[3], df2 (&acc2)[3]) {
#pragma unroll 1
  for (int l = l0; l < l1; l += 2) {
    df2 ys[3], den[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      ys[c] = {*reinterpret_cast<const float2*>(&sa[2 * c][l]), *reinterpret_cast<const float2*>(&sa[2 * c + 1][l])};
      den[c] = {*reinterpret_cast<const float2*>(&sa[6 + 2 * c][l]), *reinterpret_cast<const float2*>(&sa[7 + 2 * c][l])};
    }
    const float2 fb = *reinterpret_cast<const float2*>(&sa[12][l]);
    int2 pp = make_int2(0, 0);
    if (MODE == kDfMask) pp = *reinterpret_cast<const int2*>(&smask[l]);
    pair2_df<KIND, MODE>(ys, den, fb, pp, xt, nt, bit, acc, acc2);
  }
}

// Stages the coordinates of a tile and the target's in the tile's form (xt); stage_q(l, s) stores what else
// slot l needs of source s (s < 0: a padding slot, to be given zero density).  With SKIP, where df_skip_any says so
// (sk: df_skip_targets' part), bit i - lo of a slot's mask in smask leaves it out for targets of particle i, and the mode
// is kDfMask or kDfNone (grid and plain tiles, nearly all of them, carry none of this);
// else kDfGrid or kDfPlain.
template <bool SKIP, typename StageQ>
__device__ __forceinline__ DfMode df_stage(float (*sa)[kTileDf], int* smask, const int (&sidx)[2], int filled, const DfSkip& skip,
                                         const int* sk, const float4* __restrict__ x3h, const float4* __restrict__ x3m,
                                         const float4* __restrict__ x3l, const float4& oh, const float4& om,
                                         const float4& ol, const dflt (&x0)[3], float xm, df2 (&xt)[3], StageQ stage_q) {
  const int lane = threadIdx.x & 31;
  dflt p[2][3];
  int pid[2];
  float m = 0.0f, mn = 3.0e38f;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    p[k][0] = p[k][1] = p[k][2] = dflt{0.0f, 0.0f};
    pid[k] = -2;
    if (lane + 32 * k < filled) {
      const float4 ph = x3h[sidx[k]], pm = x3m[sidx[k]], pl = x3l[sidx[k]];
      pid[k] = __float_as_int(ph.w);
      p[k][0] = df_diff3(oh.x, om.x, ol.x, ph.x, pm.x, pl.x);
      p[k][1] = df_diff3(oh.y, om.y, ol.y, ph.y, pm.y, pl.y);
      p[k][2] = df_diff3(oh.z, om.z, ol.z, ph.z, pm.z, pl.z);
      const float far = fmaxf(fabsf(p[k][0].h), fmaxf(fabsf(p[k][1].h), fabsf(p[k][2].h)));
      m = fmaxf(m, far);
      mn = fminf(mn, far);
    }
  }
  int mask[2] = {0, 0};
  if constexpr (SKIP) {
    const int lo = sk[64], hi = sk[65];
    const int tlo = __reduce_min_sync(0xffffffffu, pid[0] < 0 ? INT_MAX : pid[0]);
    const int thi = __reduce_max_sync(0xffffffffu, max(pid[0], pid[1]));
    auto near_bit = [&](int j, int bit) {  // j: a near source per lane
      for (unsigned hits = __ballot_sync(0xffffffffu, j >= tlo && j <= thi); hits; hits &= hits - 1) {
        const int jj = __shfl_sync(0xffffffffu, j, __ffs(hits) - 1);
        if (pid[0] == jj) mask[0] |= bit;
        if (pid[1] == jj) mask[1] |= bit;
      }
    };
#pragma unroll
    for (int k = 0; k < 2; ++k)
      if (pid[k] >= lo && pid[k] <= hi) mask[k] = 1 << (pid[k] - lo);
    near_bit(sk[lane], 1);
    near_bit(sk[32 + lane], 2);
    if (sk[66])
      for (int i = lo; i <= hi; ++i) {
        const int end = skip.first[i + 1];
        for (int e = skip.first[i] + (i < lo + 2 ? 32 : 0); e < end; e += 32)
          near_bit(e + lane < end ? skip.near[e + lane].y : -1, 1 << (i - lo));
      }
    const int all = (2 << (hi - lo)) - 1;
    if (__all_sync(0xffffffffu, (pid[0] < 0 || mask[0] == all) && (pid[1] < 0 || mask[1] == all))) return kDfNone;
  }
  m = warp_max_abs(m) + xm;
  // in the largest coordinate alone a source is at least mn - xm away
  const bool grid = !SKIP && warp_min_abs(mn) - xm >= 0.25f * m;
  // g = 2^(e - 24), 2^e > m; its exponent field is that of m less 23
  const int ge = max(1, (int)(__float_as_uint(m) >> 23) - 23);
  const float g = __uint_as_float((unsigned)ge << 23), ginv = __uint_as_float((unsigned)(254 - ge) << 23);
  auto on_grid = [&](dflt v) -> dflt {
    if (!grid) return v;
    const float h = rintf(v.h * ginv) * g;
    return {h, (v.h - h) + v.l};
  };
  const int cnt4 = (filled + 3) & ~3;
  __syncwarp();  // the warp's reads of the previous tile are done
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int l = lane + 32 * k;
    if (l < filled) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const dflt v = on_grid(p[k][c]);
        sa[2 * c][l] = v.h;
        sa[2 * c + 1][l] = v.l;
      }
      stage_q(l, sidx[k]);
      if (SKIP) smask[l] = mask[k];
    } else if (l < cnt4) {  // zero-density sources away from every target: they add exactly zero
      sa[0][l] = sa[2][l] = sa[4][l] = 8.0f * m;
      sa[1][l] = sa[3][l] = sa[5][l] = 0.0f;
      stage_q(l, -1);
      if (SKIP) smask[l] = 0;
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const dflt v = on_grid(x0[c]);
    xt[c] = {dup2(v.h), dup2(v.l)};
  }
  __syncwarp();
  return SKIP ? kDfMask : (grid ? kDfGrid : kDfPlain);
}

template <int KIND, bool SKIP>
__device__ __forceinline__ void df_tile(float* wsm, const int (&sidx)[2], int filled, const DfSkip& skip, const int* sk, bool split,
                                        int half, const float4* __restrict__ x3h, const float4* __restrict__ x3m,
                                        const float4* __restrict__ x3l, const float4* __restrict__ qh_,
                                        const float4* __restrict__ ql_, const float4& oh, const float4& om,
                                        const float4& ol, const dflt (&x0)[3], const dflt (&n0)[3], float xm, int bit,
                                        dflt (&tot)[3], dflt (&tot2)[3]) {
  float(*sa)[kTileDf] = reinterpret_cast<float(*)[kTileDf]>(wsm);
  int* const smask = reinterpret_cast<int*>(&sa[13][0]);
  df2 xt[3], nt[3];
  const DfMode mode = df_stage<SKIP>(sa, smask, sidx, filled, skip, sk, x3h, x3m, x3l, oh, om, ol, x0, xm, xt, [&](int l, int s) {
    float4 qh = make_float4(0, 0, 0, 0), ql = qh;
    if (s >= 0) {
      qh = qh_[s];
      ql = ql_[s];
    }
    sa[6][l] = qh.x;
    sa[7][l] = ql.x;
    sa[8][l] = qh.y;
    sa[9][l] = ql.y;
    sa[10][l] = qh.z;
    sa[11][l] = ql.z;
    sa[12][l] = qh.w;
  });
#pragma unroll
  for (int c = 0; c < 3; ++c) nt[c] = {dup2(n0[c].h), dup2(n0[c].l)};
  if (mode == kDfNone) return;
  const int cnt4 = (filled + 3) & ~3;
  df2 acc[3], acc2[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) acc[c] = acc2[c] = df2{dup2(0.0f), dup2(0.0f)};
  const int cnt = split ? cnt4 / 2 : cnt4, l0 = half * cnt;
  if constexpr (SKIP)
    df_tile_pairs<KIND, kDfMask>(sa, smask, l0, l0 + cnt, xt, nt, bit, acc, acc2);
  else if (mode == kDfGrid)
    df_tile_pairs<KIND, kDfGrid>(sa, smask, l0, l0 + cnt, xt, nt, bit, acc, acc2);
  else
    df_tile_pairs<KIND, kDfPlain>(sa, smask, l0, l0 + cnt, xt, nt, bit, acc, acc2);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    tot[c] = df_add_accurate(tot[c], fold2(acc[c]));
    if (KIND == 2) tot2[c] = df_add_accurate(tot2[c], fold2(acc2[c]));
  }
}

}  // namespace rbs
