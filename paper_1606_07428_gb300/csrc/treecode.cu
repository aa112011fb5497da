// Hierarchical far field for the smooth pair sums: barycentric Lagrange treecodes (Wang, Krasny and
// Tlupova, 2020) in place of the fast multipole method of Section 3.1, one for the float32 applies of
// the inner solve and, optionally, one at higher degree for the double-float passes.
//
// Per suspension, an octree over the particle centres (a cell with more than one particle splits at
// the midpoint of its centres' bounding box; children in octant order, particles ascending).  Each
// cell has the box of its particles' nodes, the box midpoint as centre, a radius
// r = max_j (|c_j - centre| + R_j) bounding its nodes, and a node count.  The targets of each particle
// form one batch (its leaf cell); a depth-first traversal accepts a cell C for approximation when
//   r_B + r_C < theta d,  d >= r_B + r_C + near_delta  and  (n + 1)^3 < nodes(C),
// else descends, and evaluates the particles of unaccepted leaves directly.  An accepted cell
// carries (n + 1)^3 proxy points on the tensor Chebyshev grid of its box and charges
//   q_abc = sum_s L_a(y_s,x) L_b(y_s,y) L_c(y_s,z) w_s mu_s     (barycentric Lagrange basis L),
// recomputed for every apply.  The pair kernels use the grid's tensor form: separations, and what depends on one axis of
// them alone, are formed per axis and row, not per proxy point.
//
// Layout: a cluster keeps the n + 1 coordinates of each axis of its grid and its charges by rows of the last axis
// (float32, or float32 pairs split from float64 charges); nodes are read from the context's own arrays.
// Each target particle has a list of (first, count) segments over N node indexes followed by (n + 1)^3 per accepted cell:
// its own particle first (masked by particle id in the inner solve's float32 sums, skipped in the others), then the
// particles near it (skipped in the others too), then the other directly evaluated ones, then its accepted cells.  Work
// items pair the targets of one particle (or a near-equal part of it, at most 512) with a run of those segments.  The
// host plan (plan_treecode) does no device work, so it also serves the host-only entry point rbs_treecode_plan.
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>

#include "common.cuh"
#include "pairs32.cuh"
#include "pairsdf.cuh"

namespace rbs {

namespace {

constexpr int kTreeMaxTargets = 512; // targets per work item at most
constexpr int kTreeTile32 = 128;     // sources per warp tile of the float32 treecode sum
constexpr int kTreeMaxQ64 = 13;      // degree <= 12 (double-float passes)


// Bounding box of each particle's nodes: lo (3) then hi (3) per particle.
__global__ void __launch_bounds__(128) k_particle_boxes(int n, const long long* __restrict__ offset,
                                                        const double4* __restrict__ x, double* __restrict__ out) {
  __shared__ double red[6][4];
  const int i = blockIdx.x;
  if (i >= n) return;
  double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
  for (long long t = offset[i] + threadIdx.x; t < offset[i + 1]; t += blockDim.x) {
    const double4 p = x[t];
    lo[0] = fmin(lo[0], p.x);
    lo[1] = fmin(lo[1], p.y);
    lo[2] = fmin(lo[2], p.z);
    hi[0] = fmax(hi[0], p.x);
    hi[1] = fmax(hi[1], p.y);
    hi[2] = fmax(hi[2], p.z);
  }
  for (int o = 16; o > 0; o >>= 1)
    for (int d = 0; d < 3; ++d) {
      lo[d] = fmin(lo[d], __shfl_down_sync(0xffffffffu, lo[d], o));
      hi[d] = fmax(hi[d], __shfl_down_sync(0xffffffffu, hi[d], o));
    }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (lane == 0)
    for (int d = 0; d < 3; ++d) {
      red[d][warp] = lo[d];
      red[3 + d][warp] = hi[d];
    }
  __syncthreads();
  if (threadIdx.x < 6) {
    const int d = threadIdx.x;
    double v = red[d][0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) v = d < 3 ? fmin(v, red[d][w]) : fmax(v, red[d][w]);
    out[6 * (size_t)i + d] = v;
  }
}

// Barycentric Lagrange basis of the nq Chebyshev points s (weights bw) at u in [-1, 1]; a point on a
// node gets that node's unit vector.
template <typename T, int MAXQ>
__device__ __forceinline__ void lagrange_row(T u, const T* s, const T* bw, int nq, T* L) {
  T t[MAXQ];
  T sum = 0;
  int hit = -1;
#pragma unroll
  for (int k = 0; k < MAXQ; ++k) {
    t[k] = 0;
    if (k < nq) {
      const T d = u - s[k];
      if (d == (T)0)
        hit = k;
      else
        t[k] = bw[k] / d;
      sum += t[k];
    }
  }
#pragma unroll
  for (int k = 0; k < MAXQ; ++k)
    if (k < nq) L[k] = hit >= 0 ? (k == hit ? (T)1 : (T)0) : t[k] / sum;
}

// Cluster charges, one block per (cluster, run of its particles), from the nodes' weighted densities.
// They are stored by rows of the proxy grid's last axis, the layout that the pair kernels read:
// q[(((cluster nq + a) nbp + b) 3 + k) ncp + c], rows padded to ncp and planes to nbp rows with zeros (all
// zeroed before; blocks add theirs atomically).  A node costs one product L_a L_b per row and 3
// multiply-adds per proxy on the products L_c(z) q_k.
constexpr int kChargeThreads = 256;

// Float32.  Warps take batches of 32 nodes of the run on their own: each lane forms the three Lagrange rows
// of one node, then owns two (a, b) rows of the proxy grid and every c over the batch's nodes (12 packed
// multiply-adds a node and row, loads shared by the two rows).  Grids of more than 64 rows take several passes.
constexpr int kChargeThreads32 = 128;

template <int MAXQ>
__global__ void __launch_bounds__(kChargeThreads32) k_tree_charges32(const int4* __restrict__ items,
                                                                   const int* __restrict__ order,
                                                                   const long long* __restrict__ offset,
                                                                   const double4* __restrict__ x,
                                                                   const float4* __restrict__ wmu,
                                                                   const double* __restrict__ box,
                                                                   const float* __restrict__ cheb, int nq, int nbp,
                                                                   int ncp, float* __restrict__ qproxy) {
  constexpr int W = kChargeThreads32 / 32, MQ = 3 * MAXQ + 4;  // row pitch of 4 mod 32 words: no bank conflicts
  __shared__ float sL[W][32][2 * MAXQ + 1];
  __shared__ __align__(16) float sq[W][32][MQ];
  __shared__ float s_pts[MAXQ], s_bw[MAXQ];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if ((int)threadIdx.x < nq) {
    s_pts[threadIdx.x] = cheb[threadIdx.x];
    s_bw[threadIdx.x] = cheb[nq + threadIdx.x];
  }
  __syncthreads();
  const int4 it = items[blockIdx.x];
  const int u = it.x;
  const double* bx = box + 6 * (size_t)u;
  const double m0 = bx[0], m1 = bx[1], m2 = bx[2], h0 = bx[3], h1 = bx[4], h2 = bx[5];
  for (int pass = 0; pass < nq * nq; pass += 64) {
    int ra[2], rb[2];
    bool own[2];
    float2 acc[2][3][MAXQ / 2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int ab = pass + lane + 32 * h;
      own[h] = ab < nq * nq;
      ra[h] = own[h] ? ab / nq : 0;
      rb[h] = own[h] ? ab - ra[h] * nq : 0;
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int c = 0; c < MAXQ / 2; ++c) acc[h][k][c] = make_float2(0.0f, 0.0f);
    }
    int batch = 0;
    bool any = false;
    for (int pi = it.y; pi < it.z; ++pi) {
      const int j = order[pi];
      const long long e = offset[j + 1];
      for (long long s0 = offset[j]; s0 < e; s0 += 32, ++batch) {
        if (batch % W != warp) continue;
        any = true;
        const int cnt = (int)min(32LL, e - s0);
        __syncwarp();  // the previous batch is read
        if (lane < cnt) {
          const double4 p = x[s0 + lane];
          const float4 q = wmu[s0 + lane];
          float L[MAXQ];
          lagrange_row<float, MAXQ>((float)((p.x - m0) * h0), s_pts, s_bw, nq, L);
#pragma unroll
          for (int k = 0; k < MAXQ; ++k)
            if (k < nq) sL[warp][lane][k] = L[k];
          lagrange_row<float, MAXQ>((float)((p.y - m1) * h1), s_pts, s_bw, nq, L);
#pragma unroll
          for (int k = 0; k < MAXQ; ++k)
            if (k < nq) sL[warp][lane][MAXQ + k] = L[k];
          lagrange_row<float, MAXQ>((float)((p.z - m2) * h2), s_pts, s_bw, nq, L);
#pragma unroll
          for (int k = 0; k < MAXQ; ++k) {
            const float l = k < nq ? L[k] : 0.0f;
            sq[warp][lane][k] = l * q.x;
            sq[warp][lane][MAXQ + k] = l * q.y;
            sq[warp][lane][2 * MAXQ + k] = l * q.z;
          }
        }
        __syncwarp();
#pragma unroll 2
        for (int l = 0; l < cnt; ++l) {
          float2 w[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float v = sL[warp][l][ra[h]] * sL[warp][l][MAXQ + rb[h]];
            w[h] = make_float2(v, v);
          }
#pragma unroll
          for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int c = 0; c < MAXQ / 4; ++c) {
              const float4 q = *reinterpret_cast<const float4*>(&sq[warp][l][k * MAXQ + 4 * c]);
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                acc[h][k][2 * c] = __ffma2_rn(w[h], make_float2(q.x, q.y), acc[h][k][2 * c]);
                acc[h][k][2 * c + 1] = __ffma2_rn(w[h], make_float2(q.z, q.w), acc[h][k][2 * c + 1]);
              }
            }
        }
      }
    }
    if (!any) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!own[h]) continue;
      float* dst = qproxy + ((size_t)(u * nq + ra[h]) * nbp + rb[h]) * 3 * ncp;
#pragma unroll
      for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int c = 0; c < MAXQ / 4; ++c)
          if (4 * c < ncp)
            atomicAdd(reinterpret_cast<float4*>(dst + k * ncp + 4 * c),
                      make_float4(acc[h][k][2 * c].x, acc[h][k][2 * c].y, acc[h][k][2 * c + 1].x, acc[h][k][2 * c + 1].y));
    }
  }
}

// Float64: nodes are staged kChargeTile at a time by the block, one thread per (node, axis); a thread owns
// one (a, b) row, and threads beyond the first plane take the staged nodes in turn.  Bound by the float64 pipe.
constexpr int kChargeTile = 64;

__global__ void __launch_bounds__(kChargeThreads) k_tree_charges64(const int4* __restrict__ items,
                                                                   const int* __restrict__ order,
                                                                   const long long* __restrict__ offset,
                                                                   const double4* __restrict__ x,
                                                                   const double* __restrict__ dens,
                                                                   const double* __restrict__ box,
                                                                   const double* __restrict__ cheb, int nq, int nbp,
                                                                   int ncp, double* __restrict__ qproxy) {
  constexpr int TS = kChargeTile, MAXQ = kTreeMaxQ64;
  __shared__ double sL[TS][2][MAXQ];
  __shared__ __align__(16) double sq[TS][3][MAXQ + 1];
  __shared__ double s_pts[MAXQ], s_bw[MAXQ];
  if ((int)threadIdx.x < nq) {
    s_pts[threadIdx.x] = cheb[threadIdx.x];
    s_bw[threadIdx.x] = cheb[nq + threadIdx.x];
  }
  const int4 it = items[blockIdx.x];
  const int u = it.x;
  const int plane = nq * nq;
  const int groups = kChargeThreads / plane;  // at least one: plane <= 169
  const int g = threadIdx.x / plane;
  const int ab = threadIdx.x - g * plane, a = ab / nq, b = ab - a * nq;
  double acc[3][MAXQ];
#pragma unroll
  for (int c = 0; c < MAXQ; ++c) acc[0][c] = acc[1][c] = acc[2][c] = 0;
  for (int pi = it.y; pi < it.z; ++pi) {
    const int j = order[pi];
    const long long o = offset[j], e = offset[j + 1];
    for (long long s0 = o; s0 < e; s0 += TS) {
      const int cnt = (int)min((long long)TS, e - s0);
      __syncthreads();
      const int ax = threadIdx.x / TS, l = threadIdx.x - TS * ax;
      if (ax < 3 && l < cnt) {
        const double4 p = x[s0 + l];
        const double v = ax == 0 ? p.x : (ax == 1 ? p.y : p.z);
        const double m = box[6 * (size_t)u + ax], h = box[6 * (size_t)u + 3 + ax];
        double L[MAXQ];
        lagrange_row<double, MAXQ>((v - m) * h, s_pts, s_bw, nq, L);
        if (ax < 2) {
#pragma unroll
          for (int k = 0; k < MAXQ; ++k)
            if (k < nq) sL[l][ax][k] = L[k];
        } else {
          const double* d = dens + 3 * (s0 + l);
          const double q0 = p.w * d[0], q1 = p.w * d[1], q2 = p.w * d[2];
#pragma unroll
          for (int k = 0; k < MAXQ; ++k)
            if (k < nq) {
              sq[l][0][k] = L[k] * q0;
              sq[l][1][k] = L[k] * q1;
              sq[l][2][k] = L[k] * q2;
            }
        }
      }
      __syncthreads();
      if (g < groups) {
        for (int l2 = g; l2 < cnt; l2 += groups) {
          const double w = sL[l2][0][a] * sL[l2][1][b];
#pragma unroll
          for (int c = 0; c < MAXQ; ++c)
            if (c < nq) {
              acc[0][c] = fma(w, sq[l2][0][c], acc[0][c]);
              acc[1][c] = fma(w, sq[l2][1][c], acc[1][c]);
              acc[2][c] = fma(w, sq[l2][2][c], acc[2][c]);
            }
        }
      }
    }
  }
  if (g < groups) {
    double* dst = qproxy + ((size_t)(u * nq + a) * nbp + b) * 3 * ncp;
#pragma unroll
    for (int c = 0; c < MAXQ; ++c)
      if (c < nq)
        for (int k = 0; k < 3; ++k) atomicAdd(dst + k * ncp + c, acc[k][c]);
  }
}

// Float64 cluster charges to the rows the double-float kernel reads, per row of the last proxy axis:
// (x, y, z hi, x, y, z lo, bound) x ncp, the bound of their biased sums.
__global__ void k_tree_q64_split(long long rows, int ncp, const double* __restrict__ q64, float* __restrict__ q) {
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (k >= rows * ncp) return;
  const long long r = k / ncp;
  const int c = (int)(k - r * ncp);
  float* dst = q + r * 7 * ncp + c;
  float h[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const dflt v = df_split(q64[(r * 3 + d) * ncp + c]);
    dst[d * ncp] = v.h;
    dst[(3 + d) * ncp] = v.l;
    h[d] = v.h;
  }
  dst[6 * ncp] = bias_bound(h[0], h[1], h[2]);
}

// Units of the pair sums: (work item, run of 32 NT of its targets) in item order, taken by warps from a
// counter that the launch starts at zero.  Warps never wait for one another, and no warp is tied to a
// fixed share: with whole-particle blocks striding over the items, the warp that held a particle's
// last few targets finished early and blocks of an odd warp count loaded the SM's four schedulers
// unevenly (10 of 15 resident warps active on average).

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}

// ---- float32 treecode pair sum
//
// A unit walks its item's segments: runs of nodes (direct particles), then clusters.
//
// Nodes: the packed tile loop of the direct kernel (pairs32.cuh) over per-warp tiles of 128 sources;
// tiles that may hold nodes of the targets' own particle (the first nmask sources) mask them by id.
//
// Clusters: the proxy points form a tensor grid, so a target's separations from all (n + 1)^3 of them
// come from n + 1 differences per axis.  Per row (a, b) the parts d_x^2 + d_y^2 and d_x n_x + d_y n_y are
// formed once; a proxy then takes one multiply-add for r^2, one for r . n, three for r . q, five for the
// kernel's factor c, and two for the sums: sum c and sum c d_z, the x and y components following
// per row as d_x sum c and d_y sum c.  That is 12 float32 operations per proxy pair (Stokeslet: 12)
// in place of the 20 (18) of a node pair.  Two proxies of the last axis share each packed instruction;
// NQ2 = ceil((n + 1) / 2).  Charges come in slabs (one a) through a per-warp ring of asynchronous
// copies.
//
// A unit with at most 16 targets gives its two half-warps alternate halves of the sources.  KIND 0 traction,
// 1 Stokeslet into y; 2 traction into y and Stokeslet into y2 (26 and 17 operations a pair, one target per lane),
// without the leading nskip segments (the own particle and its near ones).
//
// Bound by the float32 pipe, 76% busy.  With every source in one tile loop and blocks of whole particles, and
// now: 1,150 to 1,770 Gpair/s on 1,500 particles of 144 nodes, 1,350 to 1,820 on 700 of 312.
constexpr int kRing32 = 4;

template <int KIND, int NT, int NQ2>
__global__ void __launch_bounds__(128, NT == 1 ? (KIND == 2 ? 4 : (NQ2 <= 4 ? 6 : 5)) : 4)
    k_tree32x2(unit_t nunits, int per_item, unit_t* __restrict__ counter, const TreeItem* __restrict__ items,
               const int2* __restrict__ segs, long long N, int npx, int nq, int nbp, int ncp,
               const float4* __restrict__ xhi, const float4* __restrict__ xlo, const float4* __restrict__ nrm32,
               const float4* __restrict__ sq, const float4* __restrict__ axis, const float* __restrict__ pq,
               int warp_floats, double* __restrict__ y, double* __restrict__ y2) {
  static_assert(KIND != 2 || NT == 1, "both sums: one target per lane");
  constexpr int TW = kTreeTile32, SL = TW / 32;
  const int lane = threadIdx.x & 31;
  extern __shared__ __align__(16) float tree_smem32[];
  float* const wsm = tree_smem32 + (threadIdx.x >> 5) * warp_floats;
  float* const ssx = wsm;
  float* const ssy = ssx + TW;
  float* const ssz = ssx + 2 * TW;
  float* const srx = ssx + 3 * TW;
  float* const sry = ssx + 4 * TW;
  float* const srz = ssx + 5 * TW;
  int* const spid = reinterpret_cast<int*>(ssx + 6 * TW);
  const int slab = 3 * nbp * ncp;            // floats of one a-slab
  float* const ring = wsm;                   // kRing32 slabs
  float* const sax = wsm + kRing32 * slab;   // 3 nq (+ 3 pad) origin-relative proxy coordinates, negated
  const uint32_t ring_s = static_cast<uint32_t>(__cvta_generic_to_shared(ring));
  for (unit_t unit = take_unit(counter); unit < nunits; unit = take_unit(counter)) {
    const UnitPart u = unit_part(unit, per_item);
    const TreeItem w = items[u.item];
    const int tb = w.t0 + u.part * 32 * NT;
    if (tb >= w.t1) continue;
    const int nu = min(NT, (w.t1 - tb + 31) / 32);      // target slots that hold a target
    const bool split = w.t1 - tb <= 16;
    const int half = split ? lane >> 4 : 0;
    const float4 oh = xhi[w.t0], ol = xlo[w.t0];
    float2 xt[NT][3], nt[NT][3];
    int pt[NT];
    bool valid[NT];
#pragma unroll
    for (int u = 0; u < NT; ++u) {
      const int t = tb + 32 * u + (split ? lane & 15 : lane);
      valid[u] = t < w.t1;
      float a0 = 0.0f, a1 = 0.0f, a2 = 0.0f, n0 = 0.0f, n1 = 0.0f, n2 = 0.0f;
      pt[u] = -1;
      if (valid[u]) {
        const float4 ah = xhi[t], al = xlo[t], nn = nrm32[t];
        a0 = (ah.x - oh.x) + (al.x - ol.x);
        a1 = (ah.y - oh.y) + (al.y - ol.y);
        a2 = (ah.z - oh.z) + (al.z - ol.z);
        n0 = nn.x;
        n1 = nn.y;
        n2 = nn.z;
        pt[u] = __float_as_int(ah.w);
      }
      xt[u][0] = f2(a0, a0);
      xt[u][1] = f2(a1, a1);
      xt[u][2] = f2(a2, a2);
      nt[u][0] = f2(n0, n0);
      nt[u][1] = f2(n1, n1);
      nt[u][2] = f2(n2, n2);
    }
    float sa[NT][3], ea[NT][3];
    float sb[3] = {0.0f, 0.0f, 0.0f}, eb[3] = {0.0f, 0.0f, 0.0f};  // KIND 2: the Stokeslet sums
#pragma unroll
    for (int u = 0; u < NT; ++u) sa[u][0] = sa[u][1] = sa[u][2] = ea[u][0] = ea[u][1] = ea[u][2] = 0.0f;
    int seg = w.s0 + (KIND == 2 ? w.nskip : 0), off = 0, done = 0;
    int2 sg = seg < w.s1 ? segs[seg] : make_int2(0, 0);
    // nodes
    while (seg < w.s1 && sg.x < N) {
      // the source of each of this lane's slots (lane + 32 k) from a walk over consecutive segments
      // that every lane of the warp takes in step, then all of its loads at once
      int sidx[SL];
#pragma unroll
      for (int k = 0; k < SL; ++k) sidx[k] = 0;
      int filled = 0;
      while (filled < TW && seg < w.s1 && sg.x < N) {
        const int take = min(sg.y - off, TW - filled);
#pragma unroll
        for (int k = 0; k < SL; ++k) {
          const int l = lane + 32 * k;
          if (l >= filled && l < filled + take) sidx[k] = sg.x + off + (l - filled);
        }
        filled += take;
        off += take;
        if (off >= sg.y) {
          ++seg;
          off = 0;
          if (seg < w.s1) sg = segs[seg];
        }
      }
      const int cnt8 = (filled + 7) & ~7;
      __syncwarp();  // the warp's reads of the previous tile are done
#pragma unroll 2
      for (int k = 0; k < SL; ++k) {
        const int l = lane + 32 * k;
        if (l < filled) {
          const int s = sidx[k];
          const float4 ph = xhi[s], pl = xlo[s], q = sq[s];
          ssx[l] = (oh.x - ph.x) + (ol.x - pl.x);
          ssy[l] = (oh.y - ph.y) + (ol.y - pl.y);
          ssz[l] = (oh.z - ph.z) + (ol.z - pl.z);
          srx[l] = q.x;
          sry[l] = q.y;
          srz[l] = q.z;
          spid[l] = __float_as_int(ph.w);
        } else if (l < cnt8) {
          ssx[l] = ssy[l] = ssz[l] = 1.0e4f;
          srx[l] = sry[l] = srz[l] = 0.0f;
          spid[l] = -2;
        }
      }
      __syncwarp();
      float2 p[NT][3];
#pragma unroll
      for (int u = 0; u < NT; ++u) p[u][0] = p[u][1] = p[u][2] = f2(0.0f, 0.0f);
      const int cnt = split ? cnt8 / 2 : cnt8, l0 = half * cnt;
#define RBS_TILE(NUV)                                                                                        \
  do {                                                                                                       \
    if (done < w.nmask)                                                                                      \
      pair_tile32x2<KIND, true, NT, NUV>(ssx + l0, ssy + l0, ssz + l0, srx + l0, sry + l0, srz + l0, spid + l0, \
                                         cnt, xt, nt, pt, p);                                                \
    else                                                                                                     \
      pair_tile32x2<KIND, false, NT, NUV>(ssx + l0, ssy + l0, ssz + l0, srx + l0, sry + l0, srz + l0, spid + l0, \
                                          cnt, xt, nt, pt, p);                                               \
  } while (0)
      if constexpr (KIND == 2) {
        float2 p2[3] = {f2(0.0f, 0.0f), f2(0.0f, 0.0f), f2(0.0f, 0.0f)};
        pair_tile32_both<TW>(ssx, l0, cnt, xt[0], nt[0], p[0], p2);
#pragma unroll
        for (int c = 0; c < 3; ++c) two_sum_acc(sb[c], eb[c], p2[c].x + p2[c].y);
      } else if (nu == NT) {
        RBS_TILE(NT);
      } else if constexpr (NT > 1) {
        RBS_TILE(1);
      }
#undef RBS_TILE
      done += filled;
#pragma unroll
      for (int u = 0; u < NT; ++u)
#pragma unroll
        for (int c = 0; c < 3; ++c) two_sum_acc(sa[u][c], ea[u][c], p[u][c].x + p[u][c].y);
    }
    // clusters
    if (seg < w.s1) {
      __syncwarp();  // the tile's reads are done: the ring takes its place
      int iss_seg = seg, iss_a = 0, iss_slot = 0, iss_left = (w.s1 - seg) * nq;
      const float* iss_src = pq + (size_t)((sg.x - N) / npx) * nq * slab;
      auto issue = [&]() {
        if (iss_left > 0) {
          const uint32_t dst = ring_s + iss_slot * slab * 4;
          for (int k = lane; k < slab / 4; k += 32) cp_async16(dst + 16 * k, iss_src + 4 * k);
          --iss_left;
          iss_slot = iss_slot + 1 == kRing32 ? 0 : iss_slot + 1;
          iss_src += slab;
          if (++iss_a == nq) {
            iss_a = 0;
            ++iss_seg;
            if (iss_left > 0) iss_src = pq + (size_t)((segs[iss_seg].x - N) / npx) * nq * slab;
          }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
      };
#pragma unroll
      for (int k = 0; k < kRing32 - 1; ++k) issue();
      int slot = 0;
      for (; seg < w.s1; ++seg) {
        const long long cell = (segs[seg].x - N) / npx;
        __syncwarp();  // the previous cluster's coordinates are read
        for (int k = lane; k < 3 * nq; k += 32) {
          const float4 c4 = axis[cell * 3 * nq + k];  // hi, lo of coordinate k of its axis
          const int ax = k / nq;
          const float h = ax == 0 ? oh.x : (ax == 1 ? oh.y : oh.z), l = ax == 0 ? ol.x : (ax == 1 ? ol.y : ol.z);
          sax[k] = (h - c4.x) + (l - c4.y);
        }
        __syncwarp();
        float2 dz[NT][NQ2];
#pragma unroll
        for (int i = 0; i < NQ2; ++i) {
          const float2 s = f2(sax[2 * nq + 2 * i], sax[2 * nq + min(2 * i + 1, nq - 1)]);
#pragma unroll
          for (int u = 0; u < NT; ++u) dz[u][i] = __fadd2_rn(xt[u][2], s);
        }
        for (int a = 0; a < nq; ++a) {
          issue();
          asm volatile("cp.async.wait_group %0;" ::"n"(kRing32 - 1) : "memory");
          __syncwarp();
          const float* row = ring + slot * slab + half * 3 * ncp;
          float2 dx[NT], dx2[NT], rnx[NT], p[NT][3], s0x[NT], s0y[NT];
          float2 p2[3] = {f2(0.0f, 0.0f), f2(0.0f, 0.0f), f2(0.0f, 0.0f)}, t0x = p2[0], t0y = p2[0];  // KIND 2
          const float sxa = sax[a];
#pragma unroll
          for (int u = 0; u < NT; ++u) {
            dx[u] = __fadd2_rn(xt[u][0], f2(sxa, sxa));
            dx2[u] = __fmul2_rn(dx[u], dx[u]);
            rnx[u] = __fmul2_rn(dx[u], nt[u][0]);
            p[u][0] = p[u][1] = p[u][2] = s0x[u] = s0y[u] = f2(0.0f, 0.0f);
          }
          for (int b = half; b < nbp; b += split ? 2 : 1, row += (split ? 2 : 1) * 3 * ncp) {
            const float syb = sax[nq + min(b, nq - 1)];
            float4 q[3][(NQ2 + 1) / 2];
#pragma unroll
            for (int k = 0; k < 3; ++k)
#pragma unroll
              for (int i = 0; i < (NQ2 + 1) / 2; ++i) q[k][i] = *reinterpret_cast<const float4*>(row + k * ncp + 4 * i);
#pragma unroll
            for (int u = 0; u < NT; ++u) {
              if (u >= nu) continue;
              const float2 dy = __fadd2_rn(xt[u][1], f2(syb, syb));
              const float2 sab = __ffma2_rn(dy, dy, dx2[u]);
              const float2 rnab = __ffma2_rn(dy, nt[u][1], rnx[u]);
              float2 s0 = f2(0.0f, 0.0f), t0 = s0;
#pragma unroll
              for (int i = 0; i < NQ2; ++i) {
                const float2 qx = (i & 1) ? f2(q[0][i / 2].z, q[0][i / 2].w) : f2(q[0][i / 2].x, q[0][i / 2].y);
                const float2 qy = (i & 1) ? f2(q[1][i / 2].z, q[1][i / 2].w) : f2(q[1][i / 2].x, q[1][i / 2].y);
                const float2 qz = (i & 1) ? f2(q[2][i / 2].z, q[2][i / 2].w) : f2(q[2][i / 2].x, q[2][i / 2].y);
                const float2 d = dz[u][i];
                const float2 r2 = __ffma2_rn(d, d, sab);
                const float2 inv = f2(rsqrt_hw(r2.x), rsqrt_hw(r2.y));
                const float2 rr = __ffma2_rn(d, qz, __ffma2_rn(dy, qy, __fmul2_rn(dx[u], qx)));
                const float2 inv2 = __fmul2_rn(inv, inv);
                const float2 inv3 = __fmul2_rn(inv2, inv);
                float2 c;
                if (KIND == 0) {
                  const float2 rn = __ffma2_rn(d, nt[u][2], rnab);
                  c = __fmul2_rn(__fmul2_rn(__fmul2_rn(rn, rr), inv2), inv3);
                } else if (KIND == 2) {
                  const float2 cs = __fmul2_rn(rr, inv3);
                  c = __fmul2_rn(__fmul2_rn(__ffma2_rn(d, nt[u][2], rnab), inv2), cs);
                  p2[0] = __ffma2_rn(qx, inv, p2[0]);
                  p2[1] = __ffma2_rn(qy, inv, p2[1]);
                  p2[2] = __ffma2_rn(cs, d, __ffma2_rn(qz, inv, p2[2]));
                  t0 = __fadd2_rn(t0, cs);
                } else {
                  c = __fmul2_rn(rr, inv3);
                  p[u][0] = __ffma2_rn(qx, inv, p[u][0]);
                  p[u][1] = __ffma2_rn(qy, inv, p[u][1]);
                  p[u][2] = __ffma2_rn(qz, inv, p[u][2]);
                }
                s0 = __fadd2_rn(s0, c);
                p[u][2] = __ffma2_rn(c, d, p[u][2]);
              }
              s0x[u] = __fadd2_rn(s0x[u], s0);
              s0y[u] = __ffma2_rn(dy, s0, s0y[u]);
              if (KIND == 2) {
                t0x = __fadd2_rn(t0x, t0);
                t0y = __ffma2_rn(dy, t0, t0y);
              }
            }
          }
#pragma unroll
          for (int u = 0; u < NT; ++u) {
            p[u][0] = __ffma2_rn(dx[u], s0x[u], p[u][0]);
            p[u][1] = __fadd2_rn(p[u][1], s0y[u]);
#pragma unroll
            for (int c = 0; c < 3; ++c) two_sum_acc(sa[u][c], ea[u][c], p[u][c].x + p[u][c].y);
          }
          if (KIND == 2) {
            p2[0] = __ffma2_rn(dx[0], t0x, p2[0]);
            p2[1] = __fadd2_rn(p2[1], t0y);
#pragma unroll
            for (int c = 0; c < 3; ++c) two_sum_acc(sb[c], eb[c], p2[c].x + p2[c].y);
          }
          __syncwarp();  // every lane has read the slab before its slot is refilled
          slot = slot + 1 == kRing32 ? 0 : slot + 1;
        }
      }
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    const double sc = KIND == 1 ? kStokesletScale : kTractionScale;
#pragma unroll
    for (int u = 0; u < NT; ++u) {
      if (!valid[u]) continue;
      const long long t = tb + 32 * u + (split ? lane & 15 : lane);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        atomicAdd(y + 3 * t + c, sc * ((double)sa[u][c] + (double)ea[u][c]));
        if (KIND == 2) atomicAdd(y2 + 3 * t + c, kStokesletScale * ((double)sb[c] + (double)eb[c]));
      }
    }
  }
}

// ---- double-float treecode pair sum: KIND 0 traction into y, 1 Stokeslet into y, 2 traction into y and
// Stokeslet into y2.
//
// The same walk, one target per lane.  Nodes: the packed double-float pair of pairsdf.cuh over per-warp
// tiles of 64 sources.  Clusters: the tensor-grid form of the float32 kernel with every product and sum
// in double-float.  The z differences, their squares and products with n_z are kept per lane in shared
// memory for the whole cluster, the row sums d_x^2 + d_y^2 and d_x n_x + d_y n_y in registers, so a proxy
// pair takes 144 float32 operations (traction and Stokeslet) where the node pair takes pairsdf.cuh's.
// Charge rows are read through L1: a warp spends thousands of cycles on each 128-byte line.
//
// Bound by the float32 pipe, 83% busy.  Both sums with 248 operations for every pair, and now: 113 to 171 Gpair/s
// on 1,500 particles of 144 nodes, 128 to 154 on 700 of 312 (fewer of whose pairs are with proxies).
template <int KIND>
__global__ void __launch_bounds__(128, 4)
    k_tree_df2(unit_t nunits, int per_item, unit_t* __restrict__ counter, const TreeItem* __restrict__ items,
               const int2* __restrict__ segs, long long N, int npx, int nq, int nbp, int ncp,
               const float4* __restrict__ x3h, const float4* __restrict__ x3m, const float4* __restrict__ x3l,
               const float4* __restrict__ nh, const float4* __restrict__ nl, const float4* __restrict__ sqh,
               const float4* __restrict__ sql, const float4* __restrict__ axis, const float* __restrict__ pq,
               int warp_floats, double* __restrict__ y, double* __restrict__ y2) {
  const int lane = threadIdx.x & 31;
  extern __shared__ __align__(16) float tree_smem_df[];
  float* const wsm = tree_smem_df + (threadIdx.x >> 5) * warp_floats;
  const int nq2 = (nq + 1) / 2;
  // clusters: per lane and pair of the last axis, (d_z, d_z^2, d_z n_z) hi and lo; then the
  // origin-relative proxy coordinates
  float2* const sz = reinterpret_cast<float2*>(wsm) + lane;
  float2* const sax = reinterpret_cast<float2*>(wsm + nq2 * 6 * 64);
  for (unit_t unit = take_unit(counter); unit < nunits; unit = take_unit(counter)) {
    const UnitPart u = unit_part(unit, per_item);
    const TreeItem w = items[u.item];
    const int tb = w.t0 + u.part * 32;
    if (tb >= w.t1) continue;
    const bool split = w.t1 - tb <= 16;
    const int half = split ? lane >> 4 : 0;
    const int t = tb + (split ? lane & 15 : lane);
    const float4 oh = x3h[w.t0], om = x3m[w.t0], ol = x3l[w.t0];
    const bool valid = t < w.t1;
    dflt xt[3], nt[3], a[3], a2[3];
    {
      float4 ah = oh, am = om, al = ol, bh = make_float4(0, 0, 0, 0), bl = make_float4(0, 0, 0, 0);
      if (valid) {
        ah = x3h[t];
        am = x3m[t];
        al = x3l[t];
        bh = nh[t];
        bl = nl[t];
      }
      xt[0] = df_diff3(ah.x, am.x, al.x, oh.x, om.x, ol.x);
      xt[1] = df_diff3(ah.y, am.y, al.y, oh.y, om.y, ol.y);
      xt[2] = df_diff3(ah.z, am.z, al.z, oh.z, om.z, ol.z);
      nt[0] = {bh.x, bl.x};
      nt[1] = {bh.y, bl.y};
      nt[2] = {bh.z, bl.z};
    }
    const float xm = warp_max_abs(fmaxf(fabsf(xt[0].h), fmaxf(fabsf(xt[1].h), fabsf(xt[2].h))));
#pragma unroll
    for (int c = 0; c < 3; ++c) a[c] = a2[c] = dflt{0.0f, 0.0f};
    int seg = w.s0 + w.nskip, off = 0;
    int2 sg = seg < w.s1 ? segs[seg] : make_int2(0, 0);
    // nodes (the leading segments are the own particle and its near ones)
    while (seg < w.s1 && sg.x < N) {
      int sidx[2] = {0, 0};
      int filled = 0;
      while (filled < kTileDf && seg < w.s1 && sg.x < N) {
        const int take = min(sg.y - off, kTileDf - filled);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const int l = lane + 32 * k;
          if (l >= filled && l < filled + take) sidx[k] = sg.x + off + (l - filled);
        }
        filled += take;
        off += take;
        if (off >= sg.y) {
          ++seg;
          off = 0;
          if (seg < w.s1) sg = segs[seg];
        }
      }
      df_tile<KIND, false>(wsm, sidx, filled, DfSkip{}, nullptr, split, half, x3h, x3m, x3l, sqh, sql, oh, om, ol, xt, nt, xm, 0, a, a2);
    }
    // clusters
    for (; seg < w.s1; ++seg) {
      const long long cell = (segs[seg].x - N) / npx;
      __syncwarp();  // the reads of the tile or of the previous cluster are done
      for (int k = lane; k < 3 * nq; k += 32) {
        const float4 c4 = axis[cell * 3 * nq + k];
        const int ax = k / nq;
        const float h = ax == 0 ? oh.x : (ax == 1 ? oh.y : oh.z), m = ax == 0 ? om.x : (ax == 1 ? om.y : om.z),
                    l = ax == 0 ? ol.x : (ax == 1 ? ol.y : ol.z);
        const dflt v = df_diff3(c4.x, c4.y, c4.z, h, m, l);
        sax[k] = make_float2(v.h, v.l);
      }
      __syncwarp();
      for (int c = 0; c < 2 * nq2; ++c) {
        const dflt d = df_sub(xt[2], sax[2 * nq + min(c, nq - 1)]);
        const dflt z2 = df_sqr(d), zn = df_renorm(df_mul(d, nt[2]));
        float* dst = reinterpret_cast<float*>(sz + (c / 2) * 6 * 32) + (c & 1);
        dst[0] = d.h;
        dst[64] = d.l;
        dst[128] = z2.h;
        dst[192] = z2.l;
        dst[256] = zn.h;
        dst[320] = zn.l;
      }
      const float* row0 = pq + (size_t)cell * nq * nbp * 7 * ncp;
      df2 accf[3], acckz, accsz;
#pragma unroll
      for (int c = 0; c < 3; ++c) accf[c] = df2{dup2(0.0f), dup2(0.0f)};
      acckz = accsz = df2{dup2(0.0f), dup2(0.0f)};
      int since = 0;
      for (int ia = 0; ia < nq; ++ia) {
        const dflt dx = df_sub(xt[0], sax[ia]);
        const dflt x2 = df_sqr(dx), xn = df_mul(dx, nt[0]);
        for (int b = half; b < nbp; b += split ? 2 : 1) {
          const dflt dy = df_sub(xt[1], sax[nq + min(b, nq - 1)]);
          const dflt sab = df_add(x2, df_sqr(dy));
          const dflt rnab = df_add(xn, df_mul(dy, nt[1]));
          const float2 sh = dup2(sab.h), sl = dup2(sab.l), rh = dup2(rnab.h), rl = dup2(rnab.l);
          const df2 dx2 = {dup2(dx.h), dup2(dx.l)}, dy2 = {dup2(dy.h), dup2(dy.l)};
          const float* row = row0 + (size_t)(ia * nbp + b) * 7 * ncp;
          df2 s0k = {dup2(0.0f), dup2(0.0f)}, s0s = {dup2(0.0f), dup2(0.0f)};
#pragma unroll 1
          for (int i = 0; i < nq2; ++i) {
            const float2* z = sz + i * 6 * 32;
            const df2 d = {z[0], z[32]};
            df2 den[3];
#pragma unroll
            for (int c = 0; c < 3; ++c)
              den[c] = {__ldg(reinterpret_cast<const float2*>(row + c * ncp) + i),
                        __ldg(reinterpret_cast<const float2*>(row + (3 + c) * ncp) + i)};
            const float2 fb = __ldg(reinterpret_cast<const float2*>(row + 6 * ncp) + i);
            df2 r2 = two_sum2(sh, z[64]);
            r2.l = __fadd2_rn(r2.l, __fadd2_rn(sl, z[96]));
            const float2 y0 = make_float2(rsqrt_hw(r2.h.x), rsqrt_hw(r2.h.y));
            const inv_powers p(r2.h, r2.l, y0);
            const df2 rr = bdot2(dx2, den[0], dy2, den[1], d, den[2], __fmul2_rn(__fmul2_rn(r2.h, y0), fb));
            const df2 am = mul2(rr, p.y3());  // r . q / r^3 but for the series
            if (KIND != 1) {
              df2 rn = two_sum2(rh, z[128]);
              rn.l = __fadd2_rn(rn.l, __fadd2_rn(rl, z[160]));
              df2 ck = mul2(am, mul2(rn, df2{p.q, p.qe}));
              ck.l = __ffma2_rn(p.w5(), ck.h, ck.l);
              acc2_add(s0k, ck);
              acc2_add(acckz, mul2(ck, d));
            }
            if (KIND != 0) {
              const df2 cs = {am.h, __ffma2_rn(p.w3(), am.h, am.l)};
              const df2 inv = p.inv();
              acc2_add(s0s, cs);
              acc2_add(accsz, mul2(cs, d));
#pragma unroll
              for (int c = 0; c < 3; ++c) acc2_add(accf[c], mul2(den[c], inv));
            }
          }
          if (KIND != 1) {
            const dflt s = fold2(s0k);
            df_acc(a[0], df_mul(s, dx));
            df_acc(a[1], df_mul(s, dy));
          }
          if (KIND != 0) {
            dflt(&as)[3] = KIND == 2 ? a2 : a;
            const dflt s = fold2(s0s);
            df_acc(as[0], df_mul(s, dx));
            df_acc(as[1], df_mul(s, dy));
          }
          // the packed sums go to the totals every few rows, about 64 sources as for node tiles
          if (++since == 5 || (ia == nq - 1 && b + (split ? 2 : 1) >= nbp)) {
            since = 0;
            if (KIND != 1) {
              a[2] = df_add_accurate(a[2], fold2(acckz));
              a[0] = df_renorm(a[0]);
              a[1] = df_renorm(a[1]);
              acckz = df2{dup2(0.0f), dup2(0.0f)};
            }
            if (KIND != 0) {
              dflt(&as)[3] = KIND == 2 ? a2 : a;
              as[2] = df_add_accurate(as[2], fold2(accsz));
              accsz = df2{dup2(0.0f), dup2(0.0f)};
#pragma unroll
              for (int c = 0; c < 3; ++c) {
                as[c] = df_add_accurate(df_renorm(as[c]), fold2(accf[c]));
                accf[c] = df2{dup2(0.0f), dup2(0.0f)};
              }
            }
          }
        }
      }
    }
    const double sc = KIND == 1 ? kStokesletScale : kTractionScale;
    if (valid)
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        atomicAdd(y + 3 * (long long)t + c, sc * ((double)a[c].h + (double)a[c].l));
        if (KIND == 2) atomicAdd(y2 + 3 * (long long)t + c, kStokesletScale * ((double)a2[c].h + (double)a2[c].l));
      }
  }
}

template <typename T>
Status upload_vec(DevBuf<T>& buf, const std::vector<T>& host, cudaStream_t s) {
  RBS_TRY(buf.alloc(std::max<size_t>(1, host.size())));
  if (!host.empty())
    RBS_CUDA_TRY(cudaMemcpyAsync(buf.ptr, host.data(), sizeof(T) * host.size(), cudaMemcpyHostToDevice, s));
  return Status::Ok();
}

// Host octree cell.
struct HCell {
  int pb = 0, pe = 0;          // particles order[pb, pe)
  double lo[3], hi[3], cen[3];
  double r = 0.0;
  long long nodes = 0;
  int kid[8];
  int nkid = 0;
  int used = -1;               // index among the cells with proxy points
};

struct TreeBuilder {
  const PlanInput& c;
  const double* pbox;
  std::vector<int>& order;
  std::vector<HCell>& cells;
  std::vector<int>& leaf_of;

  int build(int pb, int pe, int depth) {
    HCell h;
    h.pb = pb;
    h.pe = pe;
    for (int d = 0; d < 3; ++d) {
      h.lo[d] = INFINITY;
      h.hi[d] = -INFINITY;
    }
    for (int q = pb; q < pe; ++q) {
      const int j = order[q];
      for (int d = 0; d < 3; ++d) {
        h.lo[d] = std::min(h.lo[d], pbox[6 * (size_t)j + d]);
        h.hi[d] = std::max(h.hi[d], pbox[6 * (size_t)j + 3 + d]);
      }
      h.nodes += c.offset[j + 1] - c.offset[j];
    }
    for (int d = 0; d < 3; ++d) h.cen[d] = 0.5 * (h.lo[d] + h.hi[d]);
    for (int q = pb; q < pe; ++q) {
      const int j = order[q];
      const double dx = c.centres[3 * j] - h.cen[0], dy = c.centres[3 * j + 1] - h.cen[1],
                   dz = c.centres[3 * j + 2] - h.cen[2];
      h.r = std::max(h.r, std::sqrt(dx * dx + dy * dy + dz * dz) + c.radius[j]);
    }
    const int id = (int)cells.size();
    cells.push_back(h);
    if (pe - pb > 1 && depth < 64) {
      double clo[3] = {INFINITY, INFINITY, INFINITY}, chi[3] = {-INFINITY, -INFINITY, -INFINITY};
      for (int q = pb; q < pe; ++q)
        for (int d = 0; d < 3; ++d) {
          clo[d] = std::min(clo[d], c.centres[3 * order[q] + d]);
          chi[d] = std::max(chi[d], c.centres[3 * order[q] + d]);
        }
      double mid[3];
      for (int d = 0; d < 3; ++d) mid[d] = 0.5 * (clo[d] + chi[d]);
      // stable partition by octant (x the low bit), keeping ascending particle order in each
      std::vector<int> oct(pe - pb);
      int count[8] = {0, 0, 0, 0, 0, 0, 0, 0};
      for (int q = pb; q < pe; ++q) {
        const int j = order[q];
        const int o = (c.centres[3 * j] > mid[0] ? 1 : 0) + (c.centres[3 * j + 1] > mid[1] ? 2 : 0) +
                      (c.centres[3 * j + 2] > mid[2] ? 4 : 0);
        oct[q - pb] = o;
        ++count[o];
      }
      int groups = 0;
      for (int o = 0; o < 8; ++o) groups += count[o] > 0;
      if (groups > 1) {
        int start[8];
        int acc = pb;
        for (int o = 0; o < 8; ++o) {
          start[o] = acc;
          acc += count[o];
        }
        std::vector<int> tmp(pe - pb);
        int pos[8];
        for (int o = 0; o < 8; ++o) pos[o] = start[o] - pb;
        for (int q = pb; q < pe; ++q) tmp[pos[oct[q - pb]]++] = order[q];
        std::copy(tmp.begin(), tmp.end(), order.begin() + pb);
        int kids[8], nk = 0;
        for (int o = 0; o < 8; ++o)
          if (count[o] > 0) kids[nk++] = build(start[o], start[o] + count[o], depth + 1);
        for (int k = 0; k < nk; ++k) cells[id].kid[k] = kids[k];
        cells[id].nkid = nk;
        return id;
      }
    }
    for (int q = pb; q < pe; ++q) leaf_of[order[q]] = id;
    return id;
  }
};

}  // namespace

void TreeState::release() {
  active = false;
  tmax = 0;
  n_cells = 0;
  n_src = 0;
  items.clear();
  segs.clear();
  charge_items.clear();
  d_axis.release();
  d_pq.release();
  d_items.release();
  d_segs.release();
  d_charge_items.release();
  d_order.release();
  d_box.release();
  d_cheb.release();
  d_cheb64.release();
  d_q64.release();
  df = false;
  direct_pairs = proxy_pairs = charge_work = lead_pairs = 0;
}

double tree_error(const Context& c) {
  if (!c.tree.active) return INFINITY;
  // empirical model of the treecode's relative error: C(theta) rho^-n with rho the Bernstein ellipse
  // parameter 1/theta + sqrt(1/theta^2 - 1) and C = 0.25 max(1, (theta / 0.5)^2)
  const double th = c.tree.theta, a = 1.0 / th;
  const double C = 0.25 * std::max(1.0, (th / 0.5) * (th / 0.5));
  return C * std::pow(a + std::sqrt(a * a - 1.0), -c.tree.degree);
}

Status plan_treecode(const PlanInput& c, double theta, int degree, TreePlan& T) {
  const int n = c.n;
  const int nq = degree + 1, npx = nq * nq * nq;
  const double* pbox = c.pbox;

  // 2. one octree per suspension (particles of a suspension are contiguous)
  std::vector<int> order(n), leaf_of(n, -1), root_of(n, -1);
  std::vector<HCell> cells;
  cells.reserve(2 * (size_t)n + 8);
  TreeBuilder tb{c, pbox, order, cells, leaf_of};
  for (int a = 0; a < n;) {
    int e = a + 1;
    while (e < n && c.sid[e] == c.sid[a]) ++e;
    for (int q = a; q < e; ++q) order[q] = q;
    const int root = tb.build(a, e, 0);
    for (int q = a; q < e; ++q) root_of[q] = root;
    a = e;
  }

  // 3. interaction lists and source segments per target particle
  const long long N = c.offset[n];
  std::vector<std::vector<int2>> seg_of(n);
  std::vector<long long> proxy_src(n, 0);
  std::vector<int> lead(n, 1);  // leading segments: the own particle and its near ones
  T.lead_pairs = 0;
  double reach = 0.0;  // of the coordinates, whose rounding d has
  for (size_t k = 0; k < 3 * (size_t)n; ++k) reach = std::max(reach, std::fabs(c.centres[k]));
  int n_used = 0;
  std::vector<int> used_cells;
  std::vector<int> stack;
  for (int i = 0; i < n; ++i) {
    const HCell& B = cells[leaf_of[i]];
    std::vector<int2>& L = seg_of[i];
    const int np_i = (int)(c.offset[i + 1] - c.offset[i]);
    L.push_back(make_int2((int)c.offset[i], np_i));
    std::vector<int> approx, direct;
    stack.clear();
    stack.push_back(root_of[i]);
    while (!stack.empty()) {
      const int id = stack.back();
      stack.pop_back();
      const HCell& C = cells[id];
      const double dx = B.cen[0] - C.cen[0], dy = B.cen[1] - C.cen[1], dz = B.cen[2] - C.cen[2];
      const double d = std::sqrt(dx * dx + dy * dy + dz * dz);
      const double rr = B.r + C.r;
      bool accept = rr < theta * d && d >= rr + c.near_delta && (long long)npx < C.nodes;
      // (near particles stay out of clusters whatever the rounding of d)
      if (accept && d - (rr + c.near_delta) <= 1e-9 * (d + reach))
        for (int q = C.pb; q < C.pe && accept; ++q)
          accept = !near_particles(c.centres, c.radius, i, order[q], c.near_delta);
      if (accept) {
        approx.push_back(id);
      } else if (C.nkid > 0) {
        for (int k = C.nkid - 1; k >= 0; --k) stack.push_back(C.kid[k]);
      } else {
        for (int q = C.pb; q < C.pe; ++q)
          if (order[q] != i) direct.push_back(order[q]);
      }
    }
    const auto far = std::stable_partition(direct.begin(), direct.end(), [&](int j) {
      return near_particles(c.centres, c.radius, i, j, c.near_delta);
    });
    lead[i] += (int)(far - direct.begin());
    for (int j : direct) L.push_back(make_int2((int)c.offset[j], (int)(c.offset[j + 1] - c.offset[j])));
    for (int k = 0; k < lead[i]; ++k) T.lead_pairs += (long long)np_i * L[k].y;
    for (int id : approx) {
      if (cells[id].used < 0) {
        cells[id].used = n_used++;
        used_cells.push_back(id);
      }
      const long long first = N + (long long)cells[id].used * npx;
      if (first + npx > INT_MAX) return Status::Err(RBS_ENOMEM, "treecode: more than 2^31 sources");
      L.push_back(make_int2((int)first, npx));
      proxy_src[i] += npx;
    }
  }
  T.n_cells = n_used;
  T.n_src = N + (long long)n_used * npx;
  if (T.n_src > INT_MAX) return Status::Err(RBS_ENOMEM, "treecode: more than 2^31 sources");

  // 4. work items: target parts of each particle times runs of its segments, split so that the grid
  // has about 96 items per SM.  A particle is one part where it has at most `cap` nodes, else
  // near-equal parts; cap is the candidate (multiples of 32 up to 512, and the particle sizes up to
  // 512) whose items waste the fewest thread slots when every block covers the largest part in
  // steps of 32 targets (ties: the larger cap, fewer stagings per pair).
  std::vector<int> caps;
  for (int cap = 32; cap <= kTreeMaxTargets; cap += 32) caps.push_back(cap);
  for (int i = 0; i < n; ++i) {
    const int np_i = (int)(c.offset[i + 1] - c.offset[i]);
    if (np_i <= kTreeMaxTargets) caps.push_back(np_i);
  }
  std::sort(caps.begin(), caps.end());
  caps.erase(std::unique(caps.begin(), caps.end()), caps.end());
  int cap = 128;
  double best_eff = -1.0;
  for (int cand : caps) {
    long long parts = 0;
    int tmax = 0;
    for (int i = 0; i < n; ++i) {
      const int np_i = (int)(c.offset[i + 1] - c.offset[i]);
      const int k = (np_i + cand - 1) / cand;
      parts += k;
      tmax = std::max(tmax, (np_i + k - 1) / k);
    }
    const double eff = (double)N / ((double)parts * (double)((tmax + 31) / 32 * 32));
    if (eff >= best_eff * (1.0 - 1e-12)) {
      best_eff = eff;
      cap = cand;
    }
  }
  long long tiles = 0;
  T.tmax = 0;
  for (int i = 0; i < n; ++i) {
    const int np_i = (int)(c.offset[i + 1] - c.offset[i]);
    const int k = (np_i + cap - 1) / cap;
    tiles += k;
    T.tmax = std::max(T.tmax, (np_i + k - 1) / k);
  }
  const long long want = 96LL * std::max(1, c.sm_count);
  const int splits = (int)std::max(1LL, (want + tiles - 1) / std::max(1LL, tiles));
  T.items.clear();
  T.segs.clear();
  T.direct_pairs = T.proxy_pairs = 0;
  for (int i = 0; i < n; ++i) {
    const std::vector<int2>& L = seg_of[i];
    const int base = (int)T.segs.size();
    T.segs.insert(T.segs.end(), L.begin(), L.end());
    long long total = 0;
    for (const int2& g : L) total += g.y;
    const int chunks = (int)std::min<long long>(splits, std::max(1LL, total / 2048));
    // cut points at segment boundaries, each run about total / chunks sources
    std::vector<int> cut = {0};
    long long acc = 0;
    for (int k = 0; k < (int)L.size(); ++k) {
      acc += L[k].y;
      const int runs = (int)cut.size();
      if (runs < chunks && k + 1 < (int)L.size() && acc * chunks >= total * runs) cut.push_back(k + 1);
    }
    cut.push_back((int)L.size());
    const int np_i = (int)(c.offset[i + 1] - c.offset[i]);
    const int nparts = (np_i + cap - 1) / cap, psize = (np_i + nparts - 1) / nparts;
    for (int t0 = (int)c.offset[i]; t0 < (int)c.offset[i + 1]; t0 += psize) {
      const int t1 = std::min(t0 + psize, (int)c.offset[i + 1]);
      for (size_t r = 0; r + 1 < cut.size(); ++r) {
        TreeItem it{};
        it.t0 = t0;
        it.t1 = t1;
        it.s0 = base + cut[r];
        it.s1 = base + cut[r + 1];
        it.nmask = r == 0 ? np_i : 0;
        it.nskip = std::max(0, std::min(cut[r + 1], lead[i]) - cut[r]);
        T.items.push_back(it);
      }
    }
    T.direct_pairs += (long long)np_i * (total - proxy_src[i]);
    T.proxy_pairs += (long long)np_i * proxy_src[i];
  }

  // 5. cluster boxes, proxy points (float64, index a (n+1)^2 + b (n+1) + c per cluster) and charge
  // blocks
  T.box.assign(6 * (size_t)std::max(1, n_used), 0.0);
  T.proxy.assign(3 * (size_t)n_used * npx, 0.0);
  T.corder.clear();
  T.charge_items.clear();
  T.charge_work = 0;
  // nodes per charge block: about eight blocks per SM over all clusters, between 256 nodes (below,
  // the atomic additions of a block's (n + 1)^3 partial charges outweigh its work) and 4,096
  long long cell_nodes = 0;
  for (int u = 0; u < n_used; ++u) cell_nodes += cells[used_cells[u]].nodes;
  const long long run = std::min(4096LL, std::max(256LL, cell_nodes / (8LL * std::max(1, c.sm_count))));
  for (int u = 0; u < n_used; ++u) {
    const HCell& C = cells[used_cells[u]];
    double mid[3], half[3];
    for (int d = 0; d < 3; ++d) {
      mid[d] = 0.5 * (C.lo[d] + C.hi[d]);
      half[d] = 0.5 * (C.hi[d] - C.lo[d]);
      T.box[6 * (size_t)u + d] = mid[d];
      T.box[6 * (size_t)u + 3 + d] = half[d] > 0.0 ? 1.0 / half[d] : 0.0;
    }
    for (int a = 0; a < nq; ++a)
      for (int b = 0; b < nq; ++b)
        for (int e = 0; e < nq; ++e) {
          const size_t k = (size_t)u * npx + ((size_t)a * nq + b) * nq + e;
          T.proxy[3 * k] = mid[0] + half[0] * std::cos(a * kPi / degree);
          T.proxy[3 * k + 1] = mid[1] + half[1] * std::cos(b * kPi / degree);
          T.proxy[3 * k + 2] = mid[2] + half[2] * std::cos(e * kPi / degree);
        }
    // charge blocks over the cell's particles
    int q = C.pb;
    while (q < C.pe) {
      const int first = (int)T.corder.size();
      long long nodes = 0;
      while (q < C.pe && (nodes == 0 || nodes + (c.offset[order[q] + 1] - c.offset[order[q]]) <= run)) {
        nodes += c.offset[order[q] + 1] - c.offset[order[q]];
        T.corder.push_back(order[q]);
        ++q;
      }
      T.charge_items.push_back(make_int4(u, first, (int)T.corder.size(), 0));
    }
    T.charge_work += C.nodes * (long long)npx;
  }
  return Status::Ok();
}

// Tree, lists, work items and proxy points of one treecode (theta, degree) over the particles'
// node boxes pbox, on the device; df: sources in the double-float layout (positions as exact
// three-float splits, weighted densities and charges as float32 pairs, charges accumulated in float64).
static Status build_lists(Context& c, TreeState& T, const std::vector<double>& pbox, double theta, int degree,
                          bool df) {
  cudaStream_t s = c.stream;
  const int nq = degree + 1, npx = nq * nq * nq;
  std::vector<double> radius(c.n);
  for (int i = 0; i < c.n; ++i) radius[i] = c.shapes[c.shape_of[i]].radius;
  const PlanInput in{c.n, c.offset.data(), c.centres.data(), radius.data(), c.sid.data(), pbox.data(),
                     c.opt.near_delta, c.sm_count};
  TreePlan P;
  RBS_TRY(plan_treecode(in, theta, degree, P));
  T.degree = degree;
  T.npx = npx;
  T.theta = theta;
  T.df = df;
  T.tmax = P.tmax;
  T.n_cells = P.n_cells;
  T.n_src = P.n_src;
  T.direct_pairs = P.direct_pairs;
  T.proxy_pairs = P.proxy_pairs;
  T.charge_work = P.charge_work;
  T.lead_pairs = P.lead_pairs;
  T.items.swap(P.items);
  T.segs.swap(P.segs);
  T.charge_items.swap(P.charge_items);
  const int n_used = P.n_cells;
  std::vector<double>& box = P.box;
  std::vector<int>& corder = P.corder;
  std::vector<double> cheb(2 * (size_t)nq);
  for (int k = 0; k < nq; ++k) {
    cheb[k] = std::cos(k * kPi / degree);
    cheb[nq + k] = ((k & 1) ? -1.0 : 1.0) * ((k == 0 || k == degree) ? 0.5 : 1.0);
  }
  // the proxy grid's coordinates per cluster and axis, as exact three-float splits
  std::vector<float4> axis(3 * (size_t)n_used * nq);
  for (int u = 0; u < n_used; ++u)
    for (int d = 0; d < 3; ++d) {
      const size_t stride = d == 0 ? (size_t)nq * nq : (d == 1 ? (size_t)nq : 1);
      for (int k = 0; k < nq; ++k) {
        const double v = P.proxy[3 * ((size_t)u * npx + k * stride) + d];
        const float h = (float)v;
        const double r = v - (double)h;
        const float m = (float)r;
        axis[((size_t)u * 3 + d) * nq + k] = make_float4(h, m, (float)(r - (double)m), 0.0f);
      }
    }

  // 6. device copies
  RBS_TRY(upload_vec(T.d_items, T.items, s));
  RBS_TRY(upload_vec(T.d_segs, T.segs, s));
  RBS_TRY(upload_vec(T.d_charge_items, T.charge_items, s));
  RBS_TRY(upload_vec(T.d_order, corder, s));
  RBS_TRY(upload_vec(T.d_box, box, s));
  {
    std::vector<float> cheb32(cheb.begin(), cheb.end());
    if (df)
      RBS_TRY(upload_vec(T.d_cheb64, cheb, s));
    else
      RBS_TRY(upload_vec(T.d_cheb, cheb32, s));
    RBS_TRY(upload_vec(T.d_axis, axis, s));
    // rows of the last proxy axis padded to a multiple of four charges, planes to an even row count
    T.nbp = (nq + 1) & ~1;
    T.ncp = (nq + 3) & ~3;
    const size_t rows = (size_t)n_used * nq * T.nbp;
    RBS_TRY(T.d_pq.alloc(std::max<size_t>(1, rows * (df ? 7 : 3) * T.ncp)));
    if (df) RBS_TRY(T.d_q64.alloc(std::max<size_t>(1, rows * 3 * T.ncp)));
    // the host vectors above must outlive their copies
    RBS_CUDA_TRY(cudaStreamSynchronize(s));
  }
  T.active = true;
  return Status::Ok();
}

Status build_far_field(Context& c) {
  c.stats.tree_pairs = c.stats.tree_proxy_pairs = c.stats.tree_df_pairs = c.stats.tree_df_proxy_pairs = 0;
  c.stats.tree_cells = c.stats.tree_df_cells = 0;
  if (c.opt.far_field == RBS_FAR_DIRECT || !prec_f32(c.opt.precision) || c.n == 0) {
    c.tree.release();
    c.tree_df.release();
    return Status::Ok();
  }
  cudaStream_t s = c.stream;
  const int n = c.n;
  // 1. node bounding boxes of the particles
  std::vector<double> pbox(6 * (size_t)n);
  {
    DevBuf<double> d_pbox;
    RBS_TRY(d_pbox.alloc(6 * (size_t)n));
    k_particle_boxes<<<n, 128, 0, s>>>(n, c.d_offset.ptr, c.d_x.ptr, d_pbox.ptr);
    RBS_CUDA_TRY(cudaGetLastError());
    RBS_CUDA_TRY(cudaMemcpyAsync(pbox.data(), d_pbox.ptr, sizeof(double) * pbox.size(), cudaMemcpyDeviceToHost, s));
    RBS_CUDA_TRY(cudaStreamSynchronize(s));
  }
  RBS_TRY(build_lists(c, c.tree, pbox, c.opt.tree_theta, c.opt.tree_degree, false));
  c.stats.tree_pairs = c.tree.direct_pairs + c.tree.proxy_pairs;
  c.stats.tree_proxy_pairs = c.tree.proxy_pairs;
  c.stats.tree_cells = c.tree.n_cells;
  if (c.opt.far_field == RBS_FAR_TREECODE_DF) {
    RBS_TRY(build_lists(c, c.tree_df, pbox, c.opt.tree_df_theta, c.opt.tree_df_degree, true));
    c.stats.tree_df_pairs = c.tree_df.direct_pairs + c.tree_df.proxy_pairs;
    c.stats.tree_df_proxy_pairs = c.tree_df.proxy_pairs;
    c.stats.tree_df_cells = c.tree_df.n_cells;
  } else {
    c.tree_df.release();
  }
  return Status::Ok();
}

// Blocks of the persistent grid: what the SMs hold at once.
static int tree_grid(Context& c, const void* kernel, size_t smem, long long units) {
  if (smem > 48 * 1024) cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 128, smem) != cudaSuccess || per_sm < 1) per_sm = 1;
  return (int)std::max(1LL, std::min<long long>((units + 3) / 4, (long long)per_sm * std::max(1, c.sm_count)));
}

template <int KIND, int NT, int NQ2>
static Status launch_tree(Context& c, const TreeState& T, double* y, double* y2 = nullptr) {
  const int nq = T.degree + 1;
  const int slab = 3 * T.nbp * T.ncp;
  const int warp_floats = std::max(7 * kTreeTile32, (kRing32 * slab + 3 * nq + 3) & ~3);
  const size_t smem = 4 * (size_t)warp_floats * sizeof(float);
  const int per_item = (T.tmax + 32 * NT - 1) / (32 * NT);
  const long long units = (long long)T.items.size() * per_item;
  if (!units_fit(units)) return Status::Err(RBS_ENOMEM, "treecode: more than 2^32 work units");
  const auto kernel = k_tree32x2<KIND, NT, NQ2>;
  kernel<<<tree_grid(c, (const void*)kernel, smem, units), 128, smem, c.stream>>>(
      (unit_t)units, per_item, c.d_unit.ptr, T.d_items.ptr, T.d_segs.ptr, c.N, T.npx, nq, T.nbp, T.ncp, c.d_xhi.ptr,
      c.d_xlo.ptr, c.d_nrm32.ptr, c.d_wmu32.ptr, T.d_axis.ptr, T.d_pq.ptr, warp_floats, y, y2);
  RBS_CUDA_TRY(cudaGetLastError());
  return Status::Ok();
}

template <int KIND>
static Status launch_tree(Context& c, double* y) {
  const TreeState& T = c.tree;
  const int nq2 = (T.degree + 2) / 2;  // pairs of the last proxy axis; degree 2 to 10
  if (tree_variant(c) == 2) {
    if (nq2 == 2) return launch_tree<KIND, 2, 2>(c, T, y);
    return nq2 == 3 ? launch_tree<KIND, 2, 3>(c, T, y) : launch_tree<KIND, 2, 4>(c, T, y);
  }
  switch (nq2) {
    case 2: return launch_tree<KIND, 1, 2>(c, T, y);
    case 3: return launch_tree<KIND, 1, 3>(c, T, y);
    case 4: return launch_tree<KIND, 1, 4>(c, T, y);
    case 5: return launch_tree<KIND, 1, 5>(c, T, y);
    default: return launch_tree<KIND, 1, 6>(c, T, y);
  }
}

// Targets per lane of the float32 treecode sum: two, which share the loads of each charge row and tile
// (1,740 against 1,620 Gpair/s on 1,500 particles of 144 nodes, 1,810 against 1,640 on 700 of 312), unless
// rbs_options.pair_variant asks for one; one above degree 7, where the z differences of two targets no
// longer fit in registers.
int tree_variant(const Context& c) {
  return c.tree.degree > 7 || c.opt.pair_variant == 1 || c.opt.pair_variant == kPacked + 1 ? 1 : 2;
}

// Cluster charges of the float32 lists from the weighted densities in d_wmu32.
static Status charges32(Context& c) {
  TreeState& T = c.tree;
  KernelTimer timer(c, RBS_KC_TREE);
  int launches = 0;
  if (T.n_cells > 0) {
    RBS_CUDA_TRY(cudaMemsetAsync(T.d_pq.ptr, 0, sizeof(float) * T.d_pq.n, c.stream));
    const int nq = T.degree + 1;
#define RBS_CHARGE_ARGS                                                                                            \
  T.d_charge_items.ptr, T.d_order.ptr, c.d_offset.ptr, c.d_x.ptr, c.d_wmu32.ptr, T.d_box.ptr, T.d_cheb.ptr, nq, T.nbp, \
      T.ncp, T.d_pq.ptr
    if (nq <= 8)
      k_tree_charges32<8><<<(unsigned)T.charge_items.size(), kChargeThreads32, 0, c.stream>>>(RBS_CHARGE_ARGS);
    else
      k_tree_charges32<12><<<(unsigned)T.charge_items.size(), kChargeThreads32, 0, c.stream>>>(RBS_CHARGE_ARGS);
#undef RBS_CHARGE_ARGS
    launches = 1;
  }
  RBS_CUDA_TRY(cudaGetLastError());
  timer.done((double)T.charge_work, launches);
  return Status::Ok();
}

Status apply_tree(Context& c, int kind, double* y) {
  TreeState& T = c.tree;
  RBS_TRY(charges32(c));
  if (T.items.empty()) return Status::Ok();
  KernelTimer timer(c, kind == 0 ? RBS_KC_PAIR_K32 : RBS_KC_PAIR_S32);
  RBS_TRY(kind == 0 ? launch_tree<0>(c, y) : launch_tree<1>(c, y));
  timer.done((double)(T.direct_pairs + T.proxy_pairs));
  return Status::Ok();
}

// y += traction and y2 += Stokeslet sum over the lists of T in float32, without the own and near particles.
static Status launch_both(Context& c, const TreeState& T, double* y, double* y2) {
  if (T.items.empty()) return Status::Ok();
  KernelTimer timer(c, RBS_KC_PAIR_K32);
  switch ((T.degree + 2) / 2) {  // degree 2 to 12
    case 2: RBS_TRY((launch_tree<2, 1, 2>(c, T, y, y2))); break;
    case 3: RBS_TRY((launch_tree<2, 1, 3>(c, T, y, y2))); break;
    case 4: RBS_TRY((launch_tree<2, 1, 4>(c, T, y, y2))); break;
    case 5: RBS_TRY((launch_tree<2, 1, 5>(c, T, y, y2))); break;
    case 6: RBS_TRY((launch_tree<2, 1, 6>(c, T, y, y2))); break;
    default: RBS_TRY((launch_tree<2, 1, 7>(c, T, y, y2)));
  }
  timer.done(2.0 * (double)(T.direct_pairs - T.lead_pairs + T.proxy_pairs));
  return Status::Ok();
}

Status apply_tree_both(Context& c, double* y, double* y2) {
  RBS_TRY(charges32(c));
  return launch_both(c, c.tree, y, y2);
}

// Float64 cluster charges of the double-float lists, as the float32 kernel reads them.
__global__ void k_tree_q64_round(long long count, const double* __restrict__ q64, float* __restrict__ q) {
  const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (k < count) q[k] = (float)q64[k];
}

static Status charges_df(Context& c, const double* x) {
  TreeState& T = c.tree_df;
  RBS_CUDA_TRY(cudaMemsetAsync(T.d_q64.ptr, 0, sizeof(double) * T.d_q64.n, c.stream));
  k_tree_charges64<<<(unsigned)T.charge_items.size(), kChargeThreads, 0, c.stream>>>(
      T.d_charge_items.ptr, T.d_order.ptr, c.d_offset.ptr, c.d_x.ptr, x, T.d_box.ptr, T.d_cheb64.ptr, T.degree + 1,
      T.nbp, T.ncp, T.d_q64.ptr);
  RBS_CUDA_TRY(cudaGetLastError());
  return Status::Ok();
}

Status apply_tree_df_f32(Context& c, const double* x, double* y, double* y2) {
  TreeState& T = c.tree_df;
  if (T.n_cells > 0) {
    KernelTimer timer(c, RBS_KC_TREE);
    RBS_TRY(charges_df(c, x));
    const long long count = (long long)T.n_cells * (T.degree + 1) * T.nbp * 3 * T.ncp;
    k_tree_q64_round<<<cdiv(count, 256), 256, 0, c.stream>>>(count, T.d_q64.ptr, T.d_pq.ptr);
    RBS_CUDA_TRY(cudaGetLastError());
    timer.done((double)T.charge_work, 2);
  }
  return launch_both(c, T, y, y2);
}

template <int KIND>
static Status launch_tree_df(Context& c, double* y, double* y2) {
  TreeState& T = c.tree_df;
  const int nq = T.degree + 1;
  const int warp_floats = std::max(kTileDfFloats, ((nq + 1) / 2 * 6 * 64 + 6 * nq + 3) & ~3);
  const size_t smem = 4 * (size_t)warp_floats * sizeof(float);
  const int per_item = (T.tmax + 31) / 32;
  const long long units = (long long)T.items.size() * per_item;
  if (!units_fit(units)) return Status::Err(RBS_ENOMEM, "treecode: more than 2^32 work units");
  const auto kernel = k_tree_df2<KIND>;
  kernel<<<tree_grid(c, (const void*)kernel, smem, units), 128, smem, c.stream>>>(
      (unit_t)units, per_item, c.d_unit.ptr, T.d_items.ptr, T.d_segs.ptr, c.N, T.npx, nq, T.nbp, T.ncp, c.d_x3h.ptr,
      c.d_x3m.ptr, c.d_x3l.ptr, c.d_nrmh.ptr, c.d_nrml.ptr, c.d_wmuh.ptr, c.d_wmul.ptr, T.d_axis.ptr, T.d_pq.ptr,
      warp_floats, y, y2);
  RBS_CUDA_TRY(cudaGetLastError());
  return Status::Ok();
}

Status apply_tree_df(Context& c, int kind, const double* x, double* y, double* y2) {
  TreeState& T = c.tree_df;
  {
    KernelTimer timer(c, RBS_KC_TREE);
    int launches = 0;
    if (T.n_cells > 0) {
      const int nq = T.degree + 1;
      const long long rows = (long long)T.n_cells * nq * T.nbp;
      RBS_TRY(charges_df(c, x));
      k_tree_q64_split<<<cdiv(rows * T.ncp, 256), 256, 0, c.stream>>>(rows, T.ncp, T.d_q64.ptr, T.d_pq.ptr);
      launches = 2;
    }
    RBS_CUDA_TRY(cudaGetLastError());
    timer.done((double)T.charge_work, launches);
  }
  if (T.items.empty()) return Status::Ok();
  KernelTimer timer(c, kind == 0 ? RBS_KC_PAIR_KDF : (kind == 1 ? RBS_KC_PAIR_SDF : RBS_KC_PAIR_KSDF));
  RBS_TRY(kind == 0 ? launch_tree_df<0>(c, y, y2) : (kind == 1 ? launch_tree_df<1>(c, y, y2) : launch_tree_df<2>(c, y, y2)));
  timer.done((double)(T.direct_pairs - T.lead_pairs + T.proxy_pairs));
  return Status::Ok();
}

}  // namespace rbs
