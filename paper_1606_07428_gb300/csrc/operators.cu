// The pieces of the discrete operators (Sections 2.1-2.3, 3, 3.1):
//  * particle-block kernel: each particle's own surface, y = R A0 R^T x with A0 its body-frame
//    singular-rule block (Eq. 38), fused with 1/2 x and the projection L of Eq. 26, or the
//    block-diagonal preconditioner of Section 3.2;
//  * smooth pair sums over node pairs of distinct particles (traction kernel of Eqs. 13 and 22 in
//    the GMRES matvec, Stokeslet of Eq. 10 for the velocity), float64 and float32 with compensated
//    accumulation;
//  * near correction: for near particle pairs, the base-grid contribution is replaced by the one
//    from the source's upsampled grid (Section 3: upsampling for close targets).
#include <algorithm>
#include <climits>
#include <type_traits>

#include <cuda_fp16.h>

#include "common.cuh"
#include "dfloat.cuh"
#include "near.cuh"
#include "pairs32.cuh"
#include "pairsdf.cuh"

namespace rbs {

namespace {


__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float fma_t(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fma_t(double a, double b, double c) { return fma(a, b, c); }

template <typename TB>
__device__ __forceinline__ TB warp_sum_t(TB v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// ------------------------------------------------------------------------------------------
// Particle-block kernel.  Block = (particle i, node range); 256 threads.  The body-frame input
// z = R_i^T x_i is staged in shared memory; each warp produces the three rows of one node at a
// time as dot products over the 3 N_p columns, then rotates back and adds 1/2 x and L x as the mode
// asks.  TB is the storage type of the blocks (float64 or float32), and the arithmetic of the
// products and their sums.
template <typename TB>
__global__ void __launch_bounds__(256) k_blocks(int mode, const int4* __restrict__ bwork,
                                                const long long* __restrict__ offset, const int* __restrict__ nodes,
                                                const double* __restrict__ rot, const double* __restrict__ centre,
                                                const int* __restrict__ shape_of, const long long* __restrict__ block_off,
                                                const TB* __restrict__ blocks, const double4* __restrict__ x,
                                                const double* __restrict__ in, double* __restrict__ out,
                                                double* __restrict__ aux, double scale) {
  extern __shared__ __align__(16) unsigned char zs_raw[];
  TB* zs = reinterpret_cast<TB*>(zs_raw);  // 3 N_p values of the block type
  __shared__ double red[8][6];
  __shared__ double mom[6];
  const int4 wk = bwork[blockIdx.x];
  const int i = wk.x, np = nodes[i];
  const long long o = offset[i];
  const double* R = rot + 9 * i;
  const double R0 = R[0], R1 = R[1], R2 = R[2], R3 = R[3], R4 = R[4], R5 = R[5], R6 = R[6], R7 = R[7], R8 = R[8];
  const double cx = centre[3 * i], cy = centre[3 * i + 1], cz = centre[3 * i + 2];
  const bool has_block = (mode != kModeL);
  const bool has_L = (mode == kModeSelfK || mode == kModeL);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double m[6] = {0, 0, 0, 0, 0, 0};
  for (int s = threadIdx.x; s < np; s += blockDim.x) {
    const double* xs = in + 3 * (o + s);
    double a = xs[0], b = xs[1], cc = xs[2];
    if (has_block) {
      zs[3 * s + 0] = (TB)(R0 * a + R3 * b + R6 * cc);
      zs[3 * s + 1] = (TB)(R1 * a + R4 * b + R7 * cc);
      zs[3 * s + 2] = (TB)(R2 * a + R5 * b + R8 * cc);
    }
    if (has_L) {
      double4 p = x[o + s];
      double rx = p.x - cx, ry = p.y - cy, rz = p.z - cz, w = p.w;
      m[0] += w * a;
      m[1] += w * b;
      m[2] += w * cc;
      m[3] += w * (ry * cc - rz * b);
      m[4] += w * (rz * a - rx * cc);
      m[5] += w * (rx * b - ry * a);
    }
  }
  if (has_L) {
#pragma unroll
    for (int q = 0; q < 6; ++q) m[q] = warp_sum(m[q]);
    if (lane == 0)
#pragma unroll
      for (int q = 0; q < 6; ++q) red[warp][q] = m[q];
  }
  __syncthreads();
  if (has_L && threadIdx.x < 6) {
    double acc = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) acc += red[w][threadIdx.x];
    mom[threadIdx.x] = acc;
  }
  __syncthreads();
  const int dim = 3 * np;  // even: n_phi is even, so N_p is
  const TB* A = blocks + (has_block ? block_off[shape_of[i]] : 0);
  // two nodes (six consecutive rows) per warp pass, two adjacent columns per lane
  for (int t0 = wk.y + 2 * warp; t0 < wk.z; t0 += 2 * (int)(blockDim.x >> 5)) {
    const int nn = (t0 + 1 < wk.z) ? 2 : 1;
    TB y[6] = {0, 0, 0, 0, 0, 0};
    if (has_block) {
      const TB* base = A + (long long)(3 * t0) * dim;
      for (int col = 2 * lane; col < dim; col += 64) {
        const TB z0 = zs[col], z1 = zs[col + 1];
#pragma unroll
        for (int r = 0; r < 6; ++r) {
          if (r < 3 * nn) {
            const TB v0 = __ldg(base + (long long)r * dim + col), v1 = __ldg(base + (long long)r * dim + col + 1);
            y[r] = fma_t(v0, z0, fma_t(v1, z1, y[r]));
          }
        }
      }
#pragma unroll
      for (int r = 0; r < 6; ++r) y[r] = warp_sum_t(y[r]);
    }
    if (lane < nn) {
      const int t = t0 + lane;
      const double y0 = (double)y[3 * lane], y1 = (double)y[3 * lane + 1], y2 = (double)y[3 * lane + 2];
      const long long g = o + t;
      double l0 = R0 * y0 + R1 * y1 + R2 * y2;
      double l1 = R3 * y0 + R4 * y1 + R5 * y2;
      double l2 = R6 * y0 + R7 * y1 + R8 * y2;
      const double* xt = in + 3 * g;
      if (mode == kModeSelfK || mode == kModeSelfKNoL) {
        l0 += 0.5 * xt[0];
        l1 += 0.5 * xt[1];
        l2 += 0.5 * xt[2];
      }
      if (has_L) {
        double4 p = x[g];
        double rx = p.x - cx, ry = p.y - cy, rz = p.z - cz;
        // a + b x r
        l0 += mom[0] + (mom[4] * rz - mom[5] * ry);
        l1 += mom[1] + (mom[5] * rx - mom[3] * rz);
        l2 += mom[2] + (mom[3] * ry - mom[4] * rx);
      }
      if (mode == kModePrecond) {
        aux[3 * g + 0] = xt[0];
        aux[3 * g + 1] = xt[1];
        aux[3 * g + 2] = xt[2];
      }
      out[3 * g + 0] = scale * l0;
      out[3 * g + 1] = scale * l1;
      out[3 * g + 2] = scale * l2;
    }
  }
}

// ------------------------------------------------------------------------------------------
// Particle-block kernel for shapes stored by the rows of their representative nodes (ellipsoids).
// The blocks commute with the grid's eight reflections g (node map g(.), sign matrix D_g):
// A_{g(t), g(s)} = D_g A_{t,s} D_g, so y_{g(t)} = D_g sum_s A_{t,s} (D_g z_{g(s)}) for each stored
// row t.  The eight reflected copies of z = R_i^T x_i are staged in shared memory, so each stored row
// is read once for all eight reflections (k_blocks_sym below); 1/2 x, L x and the preconditioner's
// copy of x are added as in k_blocks.
// Node (j, k) under the reflection g, without divisions (k in [0, n_phi)).
__device__ __forceinline__ int reflect_jk(int g, int j, int k, int p, int nphi) {
  if (g & 4) j = p - j;
  if (g & 2) k = k == 0 ? 0 : nphi - k;
  if (g & 1) {
    k = nphi / 2 - k;
    if (k < 0) k += nphi;
  }
  return j * nphi + k;
}

// Block entries stored as the bits of float16 / bfloat16.
struct F16Bits {
  uint16_t v;
};
struct BF16Bits {
  uint16_t v;
};

// Four consecutive entries of a staged block row, or of a staged input row, in the arithmetic type
// (one 16-, 8- or two 16-byte shared-memory loads; aligned to their size).
__device__ __forceinline__ void load_quad(const float* p, float (&v)[4]) {
  const float4 a = *reinterpret_cast<const float4*>(p);
  v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w;
}
__device__ __forceinline__ void load_quad(const double* p, double (&v)[4]) {
  const double2 a = *reinterpret_cast<const double2*>(p), b = *reinterpret_cast<const double2*>(p + 2);
  v[0] = a.x, v[1] = a.y, v[2] = b.x, v[3] = b.y;
}
__device__ __forceinline__ void load_quad(const F16Bits* p, float (&v)[4]) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 f0 = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
  const float2 f1 = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
  v[0] = f0.x, v[1] = f0.y, v[2] = f1.x, v[3] = f1.y;
}
__device__ __forceinline__ void load_quad(const BF16Bits* p, float (&v)[4]) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  v[0] = __uint_as_float(u.x << 16), v[1] = __uint_as_float(u.x & 0xffff0000u);
  v[2] = __uint_as_float(u.y << 16), v[3] = __uint_as_float(u.y & 0xffff0000u);
}

// Asynchronous global-to-shared copy of BYTES (4, 8 or 16) by one thread; src_bytes = 0 writes zeros
// and reads nothing.  Completion is tracked by commit groups.
template <int BYTES>
__device__ __forceinline__ void cp_async_zfill(uint32_t dst, const void* src, uint32_t src_bytes) {
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(BYTES), "r"(src_bytes)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// TS: storage type of the block entries; TB: the arithmetic of the products and sums (float64 for
// float64 blocks, float32 otherwise).  One CTA of kSymWarps warps per particle.  Each warp takes one
// representative r at a time and streams its three rows through a ring of asynchronous copies, one
// step of 512 bytes a row (each lane copies 16 bytes of each row; the ring runs several steps ahead).
// Lane (c, h) = (lane mod 16, lane / 16) multiplies the column quads 4c + 64 s of the step with the
// reflected inputs z_g, g = 4h .. 4h + 3, keeping twelve partial sums; at the end of r a reduce-scatter
// over the sixteen column groups leaves reflection g's three sums in lanes 4g .. 4g + 3.  In float32
// arithmetic the row sums go to shared memory and every node is finished by the whole CTA at the end;
// in float64 lane 4g finishes node g(r) at once.  gridDim.y CTAs share a particle, each taking every
// gridDim.y-th run of kSymWarps representatives: a float64 particle of 144 nodes is 65 us of one SM's float64
// pipe, so a list of few particles, or of few large ones, would leave the other SMs idle (8 particles: 77 us a
// float64 launch alone, 29 shared).
template <typename TS, typename TB>
__global__ void __launch_bounds__(kSymWarps * 32, sizeof(TB) == 4 ? 3 : 2)
    k_blocks_sym(int mode, const int* __restrict__ sym_list, const long long* __restrict__ offset,
                 const int* __restrict__ pvec, const int* __restrict__ nphivec, const double* __restrict__ rot,
                 const double* __restrict__ centre, const int* __restrict__ shape_of,
                 const long long* __restrict__ block_off, const TS* __restrict__ blocks, const double4* __restrict__ x,
                 const double* __restrict__ in, double* __restrict__ out, double* __restrict__ aux, double scale) {
  constexpr bool kF32 = sizeof(TB) == 4;
  constexpr int E = 16 / (int)sizeof(TS);  // entries of a 16-byte chunk
  constexpr int SC = 32 * E;               // columns of a step
  constexpr int S = sym_lane_bytes(sizeof(TS)) / 48;  // ring stages
  constexpr int kRingBytes = kSymWarps * 32 * sym_lane_bytes(sizeof(TS));
  extern __shared__ __align__(16) unsigned char zraw[];
  __shared__ TB red[kSymWarps][6];
  __shared__ TB mom[6];
  // float64 inputs in the block's arithmetic: float32 blocks convert on the integer pipe (the float64
  // pipe would otherwise bound this kernel: rotations, moments and the L term are float64-pipe work)
  auto cv = [](double d) -> TB {
    if constexpr (kF32)
      return f64_to_f32_trunc(d);
    else
      return d;
  };
  auto wide = [](TB v) -> double {
    if constexpr (kF32)
      return f32_to_f64_bits(v);
    else
      return v;
  };
  const int i = sym_list[blockIdx.x];
  const int p = pvec[i], nphi = nphivec[i], np = (p + 1) * nphi, dim = 3 * np;
  const int nk = nphi / 4 + 1, nrep = (p / 2 + 1) * nk;
  const int part = blockIdx.y, nparts = gridDim.y;
  if (kSymWarps * part >= nrep) return;  // (no block, mode L: one part)
  const int zs = sym_zstride(dim, sizeof(TB));
  TB* zg = reinterpret_cast<TB*>(zraw + kRingBytes);  // 8 rows of stride zs
  TB* ynode = zg + 8 * zs;                            // float32: 3 N_p row sums
  const long long o = offset[i];
  const double* R = rot + 9 * i;
  const TB R0 = cv(R[0]), R1 = cv(R[1]), R2 = cv(R[2]), R3 = cv(R[3]), R4 = cv(R[4]), R5 = cv(R[5]), R6 = cv(R[6]),
           R7 = cv(R[7]), R8 = cv(R[8]);
  const double cxd = centre[3 * i], cyd = centre[3 * i + 1], czd = centre[3 * i + 2];
  const TB sc = cv(scale);
  const bool has_block = (mode != kModeL);
  const bool has_L = (mode == kModeSelfK || mode == kModeL);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;

  // the copies: step = (representative of this warp, SC-column slice), one commit group per step;
  // 16-byte copies where the rows are 16-byte aligned, else copies of two entries
  const TS* A = blocks + block_off[shape_of[i]];
  const int nst = (dim + SC - 1) / SC;
  const bool al16 = ((reinterpret_cast<uintptr_t>(A) & 15u) == 0) && (dim % E == 0);
  const uint32_t ring_l = static_cast<uint32_t>(__cvta_generic_to_shared(zraw)) + warp * (S * 3 * 512) + lane * 16;
  const int rep0 = warp + kSymWarps * part, rep_step = kSymWarps * nparts;
  int iss_left = (has_block && rep0 < nrep) ? ((nrep - 1 - rep0) / rep_step + 1) * nst : 0;
  int iss_it = 0, iss_slot = 0;
  const TS* iss_src = A + (long long)(3 * rep0) * dim + E * lane;
  const long long rep_jump = (long long)3 * rep_step * dim - (long long)SC * nst;
  auto issue = [&]() {
    if (iss_left > 0) {
      // entries past the row end are zero-filled (nothing is read there)
      const int col = E * lane + SC * iss_it;
      const uint32_t dst = ring_l + iss_slot * (3 * 512);
      if (al16) {
        const bool inb = col < dim;
        const TS* s0 = inb ? iss_src : A;
        const long long d1 = inb ? dim : 0;
        const uint32_t nb = inb ? 16u : 0u;
        cp_async_zfill<16>(dst, s0, nb);
        cp_async_zfill<16>(dst + 512, s0 + d1, nb);
        cp_async_zfill<16>(dst + 1024, s0 + 2 * d1, nb);
      } else {
#pragma unroll
        for (int j = 0; j < E / 2; ++j) {
          constexpr int B2 = 2 * (int)sizeof(TS);
          const bool inb = col + 2 * j < dim;
          const TS* s0 = inb ? iss_src + 2 * j : A;
          const long long d1 = inb ? dim : 0;
          const uint32_t nb = inb ? (uint32_t)B2 : 0u;
          cp_async_zfill<B2>(dst + j * B2, s0, nb);
          cp_async_zfill<B2>(dst + 512 + j * B2, s0 + d1, nb);
          cp_async_zfill<B2>(dst + 1024 + j * B2, s0 + 2 * d1, nb);
        }
      }
      --iss_left;
      iss_src += SC;
      if (++iss_it == nst) {  // on to this warp's next representative
        iss_it = 0;
        iss_src += rep_jump;
      }
      iss_slot = (iss_slot + 1 == S) ? 0 : iss_slot + 1;
    }
    cp_async_commit();  // empty past the end
  };
  // the first stages load while the inputs are staged
  for (int q = 0; q < S - 1; ++q) issue();

  TB m[6] = {0, 0, 0, 0, 0, 0};
  for (int sp = threadIdx.x; sp < np; sp += blockDim.x) {
    const double* xs = in + 3 * (o + sp);
    const TB a = cv(xs[0]), b = cv(xs[1]), cc = cv(xs[2]);
    if (has_block) {
      const TB z0 = R0 * a + R3 * b + R6 * cc;
      const TB z1 = R1 * a + R4 * b + R7 * cc;
      const TB z2 = R2 * a + R5 * b + R8 * cc;
      const int js = sp / nphi, ks = sp - js * nphi;
#pragma unroll
      for (int g = 0; g < 8; ++g) {
        const int sn = reflect_jk(g, js, ks, p, nphi);  // g is an involution: z_{g(sn)} = z_{sp}
        TB* zz = zg + g * zs + 3 * sn;
        zz[0] = (g & 1) ? -z0 : z0;
        zz[1] = (g & 2) ? -z1 : z1;
        zz[2] = (g & 4) ? -z2 : z2;
      }
    }
    if (has_L) {
      const double4 q = x[o + sp];
      const TB rx = cv(q.x - cxd), ry = cv(q.y - cyd), rz = cv(q.z - czd), w = cv(q.w);
      m[0] += w * a;
      m[1] += w * b;
      m[2] += w * cc;
      m[3] += w * (ry * cc - rz * b);
      m[4] += w * (rz * a - rx * cc);
      m[5] += w * (rx * b - ry * a);
    }
  }
  if (has_block) {  // the padding columns [3 N_p, zs) of each z_g (their block entries are zero)
    const int pad = zs - dim;
    for (int e = threadIdx.x; e < 8 * pad; e += blockDim.x) {
      const int g = e / pad;
      zg[g * zs + dim + (e - g * pad)] = (TB)0;
    }
  }
  if (has_L) {
#pragma unroll
    for (int q = 0; q < 6; ++q) m[q] = warp_sum_t(m[q]);
    if (lane == 0)
#pragma unroll
      for (int q = 0; q < 6; ++q) red[warp][q] = m[q];
  }
  __syncthreads();
  if (has_L && threadIdx.x < 6) {
    TB acc = 0;
    for (int w = 0; w < kSymWarps; ++w) acc += red[w][threadIdx.x];
    mom[threadIdx.x] = acc;
  }
  __syncthreads();
  // finish one node t of the particle from its body-frame block product (l0, l1, l2)
  auto finish = [&](int t, TB l0b, TB l1b, TB l2b) {
    const long long gi = o + t;
    TB l0 = R0 * l0b + R1 * l1b + R2 * l2b;
    TB l1 = R3 * l0b + R4 * l1b + R5 * l2b;
    TB l2 = R6 * l0b + R7 * l1b + R8 * l2b;
    const double* xt = in + 3 * gi;
    if (mode == kModeSelfK || mode == kModeSelfKNoL) {
      l0 += (TB)0.5 * cv(xt[0]);
      l1 += (TB)0.5 * cv(xt[1]);
      l2 += (TB)0.5 * cv(xt[2]);
    }
    if (has_L) {
      const double4 q = x[gi];
      const TB rx = cv(q.x - cxd), ry = cv(q.y - cyd), rz = cv(q.z - czd);
      l0 += mom[0] + (mom[4] * rz - mom[5] * ry);
      l1 += mom[1] + (mom[5] * rx - mom[3] * rz);
      l2 += mom[2] + (mom[3] * ry - mom[4] * rx);
    }
    if (mode == kModePrecond) {
      aux[3 * gi + 0] = xt[0];
      aux[3 * gi + 1] = xt[1];
      aux[3 * gi + 2] = xt[2];
    }
    out[3 * gi + 0] = wide(sc * l0);
    out[3 * gi + 1] = wide(sc * l1);
    out[3 * gi + 2] = wide(sc * l2);
  };
  if (!has_block) {
    for (int t = threadIdx.x; t < np; t += blockDim.x) finish(t, (TB)0, (TB)0, (TB)0);
    return;
  }

  const int kc = lane & 15, hg = lane >> 4;
  const TS* ring_k = reinterpret_cast<const TS*>(zraw) + warp * (S * 3 * SC) + 4 * kc;
  const TB* zl = zg + (4 * hg) * zs + 4 * kc;
  int slot = 0;
  for (int r = rep0; r < nrep; r += rep_step) {
    float2 y2[4][3];
    TB yd[4][3];
#pragma unroll
    for (int gl = 0; gl < 4; ++gl)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        y2[gl][q] = make_float2(0.f, 0.f);
        yd[gl][q] = (TB)0;
      }
    for (int c0 = 0; c0 < SC * nst; c0 += SC) {
      issue();
      cp_async_wait<S - 1>();  // this lane's copies of the step have landed ...
      __syncwarp();            // ... and so have the other lanes'
      const TS* st = ring_k + slot * (3 * SC);
#pragma unroll
      for (int sq = 0; sq < SC / 64; ++sq) {
        if (c0 + 64 * sq + 4 * kc >= dim) continue;
        TB a[3][4];
#pragma unroll
        for (int q = 0; q < 3; ++q) load_quad(st + q * SC + 64 * sq, a[q]);
#pragma unroll
        for (int gl = 0; gl < 4; ++gl) {
          TB z[4];
          load_quad(zl + gl * zs + c0 + 64 * sq, z);
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            if constexpr (kF32) {
              y2[gl][q] = __ffma2_rn(make_float2(a[q][0], a[q][1]), make_float2(z[0], z[1]), y2[gl][q]);
              y2[gl][q] = __ffma2_rn(make_float2(a[q][2], a[q][3]), make_float2(z[2], z[3]), y2[gl][q]);
            } else {
              yd[gl][q] = fma(a[q][0], z[0], fma(a[q][1], z[1], fma(a[q][2], z[2], fma(a[q][3], z[3], yd[gl][q]))));
            }
          }
        }
      }
      __syncwarp();  // every lane has read the stage before it is refilled
      slot = (slot + 1 == S) ? 0 : slot + 1;
    }
    // reduce-scatter over the sixteen column groups: halve the set at lane bits 3 and 2, then sum
    TB v12[12], v6[6], v3[3];
#pragma unroll
    for (int k = 0; k < 12; ++k) {
      if constexpr (kF32)
        v12[k] = y2[k / 3][k % 3].x + y2[k / 3][k % 3].y;
      else
        v12[k] = yd[k / 3][k % 3];
    }
    {
      const bool hi = lane & 8;
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const TB lo_v = v12[k], hi_v = v12[6 + k];
        v6[k] = (hi ? hi_v : lo_v) + __shfl_xor_sync(0xffffffffu, hi ? lo_v : hi_v, 8);
      }
    }
    {
      const bool hi = lane & 4;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const TB lo_v = v6[k], hi_v = v6[3 + k];
        v3[k] = (hi ? hi_v : lo_v) + __shfl_xor_sync(0xffffffffu, hi ? lo_v : hi_v, 4);
      }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      v3[k] += __shfl_xor_sync(0xffffffffu, v3[k], 2);
      v3[k] += __shfl_xor_sync(0xffffffffu, v3[k], 1);
    }
    // lane 4g holds reflection g's sums: node g(r) unless a smaller reflection reaches it
    const int g = lane >> 2;
    const int j0 = r / nk, k0 = r - j0 * nk;
    const int t = reflect_jk(g, j0, k0, p, nphi);
    bool first = true;
#pragma unroll
    for (int h = 0; h < 7; ++h) {
      const int th = __shfl_sync(0xffffffffu, t, 4 * h);
      if (h < g && th == t) first = false;
    }
    if ((lane & 3) == 0 && first) {
      const TB b0 = (g & 1) ? -v3[0] : v3[0], b1 = (g & 2) ? -v3[1] : v3[1], b2 = (g & 4) ? -v3[2] : v3[2];
      if constexpr (kF32) {
        ynode[3 * t] = b0;
        ynode[3 * t + 1] = b1;
        ynode[3 * t + 2] = b2;
      } else {
        finish(t, b0, b1, b2);
      }
    }
  }
  cp_async_wait<0>();
  if constexpr (kF32) {
    __syncthreads();
    for (int t = threadIdx.x; t < np; t += blockDim.x) {
      if (nparts > 1) {  // the nodes of this part's representatives
        const int j = t / nphi, k = t - j * nphi;
        const int kh = min(k, nphi - k), kr = min(kh, nphi / 2 - kh);
        if ((min(j, p - j) * nk + kr) / kSymWarps % nparts != part) continue;
      }
      finish(t, ynode[3 * t], ynode[3 * t + 1], ynode[3 * t + 2]);
    }
  }
}

// ------------------------------------------------------------------------------------------
// Smooth pair sums in float64.  One block per work item (128 targets x a source range); each
// thread owns one target; sources are staged 128 at a time in shared memory with their weighted
// density w_s mu_s.  Pairs on the same particle are excluded (their contribution is the singular
// rule's); the select also removes the r = 0 self pair before it is used.
template <int KIND>
__global__ void __launch_bounds__(128) k_pairs64(int nitems, const longlong4* __restrict__ work, const double4* __restrict__ x,
                                                 const double4* __restrict__ nrm, const int* __restrict__ pid,
                                                 const double* __restrict__ dens, double* __restrict__ y) {
  constexpr int TS = 128;
  __shared__ double4 sp[TS];
  __shared__ double4 sd[TS];
  __shared__ int spid[TS];
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
  const longlong4 w = work[it];
  const long long t = w.x + threadIdx.x;
  const bool valid = t < w.y;
  double4 xt = make_double4(0, 0, 0, 0), nt = make_double4(0, 0, 0, 0);
  int pt = -1;
  if (valid) {
    xt = x[t];
    nt = nrm[t];
    pt = pid[t];
  }
  double a0 = 0.0, a1 = 0.0, a2 = 0.0;
  for (long long s0 = w.z; s0 < w.w; s0 += TS) {
    const int cnt = (int)min((long long)TS, w.w - s0);
    __syncthreads();
    if ((int)threadIdx.x < cnt) {
      const long long s = s0 + threadIdx.x;
      double4 ps = x[s];
      const double* d = dens + 3 * s;
      sp[threadIdx.x] = ps;
      spid[threadIdx.x] = pid[s];
      sd[threadIdx.x] = make_double4(ps.w * d[0], ps.w * d[1], ps.w * d[2], 0.0);
    }
    __syncthreads();
#pragma unroll 4
    for (int l = 0; l < cnt; ++l) {
      const double4 ps = sp[l];
      const double4 ds = sd[l];
      const double dx = xt.x - ps.x, dy = xt.y - ps.y, dz = xt.z - ps.z;
      const double r2 = dx * dx + dy * dy + dz * dz;
      double inv = rsqrt(r2);
      if (spid[l] == pt) inv = 0.0;
      const double rr = dx * ds.x + dy * ds.y + dz * ds.z;
      if (KIND == 0) {
        const double inv2 = inv * inv;
        const double rn = dx * nt.x + dy * nt.y + dz * nt.z;
        const double c = rn * rr * (inv2 * inv2 * inv);
        a0 = fma(c, dx, a0);
        a1 = fma(c, dy, a1);
        a2 = fma(c, dz, a2);
      } else {
        const double c = rr * (inv * inv * inv);
        a0 = fma(c, dx, fma(ds.x, inv, a0));
        a1 = fma(c, dy, fma(ds.y, inv, a1));
        a2 = fma(c, dz, fma(ds.z, inv, a2));
      }
    }
  }
  if (valid) {
    const double sc = KIND == 0 ? kTractionScale : kStokesletScale;
    atomicAdd(y + 3 * t + 0, sc * a0);
    atomicAdd(y + 3 * t + 1, sc * a1);
    atomicAdd(y + 3 * t + 2, sc * a2);
  }
  }
}

// ------------------------------------------------------------------------------------------
// Weighted density in float32 for the packed kernels: wmu[t] = (w_t mu_t, 0).
__global__ void k_weight_f32(long long N, const double4* __restrict__ x, const double* __restrict__ dens,
                             float4* __restrict__ wmu, unit_t* __restrict__ units) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t < 2) units[t] = 0;  // the unit counters of the smooth sum and the near correction that follow
  if (t >= N) return;
  const double w = x[t].w;
  wmu[t] = make_float4((float)(w * dens[3 * t]), (float)(w * dens[3 * t + 1]), (float)(w * dens[3 * t + 2]), 0.0f);
}

// Direct float32 pair sums.  Sources and targets are read as float32 hi + lo position pairs and float32
// weighted densities, so the kernel runs no float64 arithmetic but its final accumulation: a coordinate
// relative to the unit's origin o (its first target) is (y_hi - o_hi) + (y_lo - o_lo), within one rounding
// of the exact difference.  A unit is 32 NT targets of a work item against its sources; warps take units
// from a counter and stage their own tiles of 128 sources, summed in float32 and added into a compensated
// accumulator.  Tiles whose particles cannot meet the unit's targets skip the same-particle test.
// Bound by the float32 pipe (20 operations a traction pair, 18 a Stokeslet pair), 76% busy: 1,460 Gpair/s on 101
// particles of 220 nodes, 1,400 with blocks that took whole items; on 8 particles of 144 nodes an apply went from 34 to
// 12 us by the smaller units.
template <int KIND, int NT>
__global__ void __launch_bounds__(128, NT == 1 ? 7 : 5)
    k_pairs32x2(unit_t nunits, unit_t* __restrict__ counter, const longlong4* __restrict__ work,
                const float4* __restrict__ xhi, const float4* __restrict__ xlo, const float4* __restrict__ nrm32,
                const float4* __restrict__ wmu, double* __restrict__ y) {
  constexpr int TW = 128, kPerItem = 4 / NT;
  __shared__ __align__(16) float tiles[4][7 * TW];
  const int lane = threadIdx.x & 31;
  float* const ssx = tiles[threadIdx.x >> 5];
  int* const spid = reinterpret_cast<int*>(ssx + 6 * TW);
  while (true) {
    const unit_t unit = take_unit(counter);
    if (unit >= nunits) return;
    const UnitPart u = unit_part(unit, kPerItem);
    const longlong4 w = work[u.item];
    const int t0 = (int)w.x + 32 * NT * u.part, t1 = (int)w.y;
    if (t0 >= t1) continue;
    const bool split = t1 - t0 <= 16;  // the two half-warps take alternate halves of the sources
    const int half = split ? lane >> 4 : 0;
    const int nu = min(NT, (t1 - t0 + 31) / 32);
    const float4 oh = xhi[t0], ol = xlo[t0];
    float2 xt[NT][3], nt[NT][3];
    int pt[NT];
    bool valid[NT];
#pragma unroll
    for (int u = 0; u < NT; ++u) {
      const int t = t0 + 32 * u + (split ? lane & 15 : lane);
      valid[u] = t < t1;
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
    const int pid_lo = __float_as_int(oh.w), pid_hi = __float_as_int(xhi[min(t0 + 32 * NT, t1) - 1].w);
    float sa[NT][3], ea[NT][3];
#pragma unroll
    for (int u = 0; u < NT; ++u) sa[u][0] = sa[u][1] = sa[u][2] = ea[u][0] = ea[u][1] = ea[u][2] = 0.0f;
    for (int s0 = (int)w.z; s0 < (int)w.w; s0 += TW) {
      const int cnt = min(TW, (int)w.w - s0), cnt8 = (cnt + 7) & ~7;
      __syncwarp();  // the warp's reads of the previous tile are done
#pragma unroll
      for (int l = lane; l < TW; l += 32) {
        if (l < cnt) {
          const int s = s0 + l;
          const float4 ph = xhi[s], pl = xlo[s], q = wmu[s];
          ssx[l] = (oh.x - ph.x) + (ol.x - pl.x);
          ssx[TW + l] = (oh.y - ph.y) + (ol.y - pl.y);
          ssx[2 * TW + l] = (oh.z - ph.z) + (ol.z - pl.z);
          ssx[3 * TW + l] = q.x;
          ssx[4 * TW + l] = q.y;
          ssx[5 * TW + l] = q.z;
          spid[l] = __float_as_int(ph.w);
        } else if (l < cnt8) {
          ssx[l] = ssx[TW + l] = ssx[2 * TW + l] = 1.0e4f;
          ssx[3 * TW + l] = ssx[4 * TW + l] = ssx[5 * TW + l] = 0.0f;
          spid[l] = -2;
        }
      }
      __syncwarp();
      const int tlo = spid[0], thi = spid[cnt - 1];
      float2 p[NT][3];
#pragma unroll
      for (int u = 0; u < NT; ++u) p[u][0] = p[u][1] = p[u][2] = f2(0.0f, 0.0f);
      const int m = split ? cnt8 / 2 : cnt8, l0 = half * m;
      const float* b = ssx + l0;
#define RBS_TILE(NUV)                                                                                               \
  do {                                                                                                              \
    if (thi < pid_lo || tlo > pid_hi)                                                                               \
      pair_tile32x2<KIND, false, NT, NUV>(b, b + TW, b + 2 * TW, b + 3 * TW, b + 4 * TW, b + 5 * TW, spid + l0, m, \
                                          xt, nt, pt, p);                                                          \
    else                                                                                                            \
      pair_tile32x2<KIND, true, NT, NUV>(b, b + TW, b + 2 * TW, b + 3 * TW, b + 4 * TW, b + 5 * TW, spid + l0, m,  \
                                         xt, nt, pt, p);                                                           \
  } while (0)
      if (nu == NT) {
        RBS_TILE(NT);
      } else if constexpr (NT > 1) {
        RBS_TILE(1);
      }
#undef RBS_TILE
#pragma unroll
      for (int u = 0; u < NT; ++u)
#pragma unroll
        for (int c = 0; c < 3; ++c) two_sum_acc(sa[u][c], ea[u][c], p[u][c].x + p[u][c].y);
    }
    const double sc = KIND == 1 ? kStokesletScale : kTractionScale;
#pragma unroll
    for (int u = 0; u < NT; ++u) {
      if (!valid[u]) continue;
      const long long t = t0 + 32 * u + (split ? lane & 15 : lane);
#pragma unroll
      for (int c = 0; c < 3; ++c) atomicAdd(y + 3 * t + c, sc * ((double)sa[u][c] + (double)ea[u][c]));
    }
  }
}

// Direct float32 sums of a refinement correction: traction into y and Stokeslet into y2 in one pass (26 operations a
// pair), over the sources that lie neither on the target's own particle nor on one near it.  Near terms grow as the
// inverse square of a gap and their float32 rounding as its inverse cube, so a sum that adds them for the near correction to
// remove keeps an error without bound (with one pair of spheres 0.01 apart, a solve to 1e-10 ended at 2e-9); without
// them every separation is at least near_delta.  A unit is 32 targets of a work item, taken one target particle at a
// time: sources are relative to the run's first target, a particle's diameter away at most.  Excluded sources become
// zero-density ones far away.  The near pairs of a particle are ordered by source, so a pointer walks them beside
// the tiles.
__global__ void __launch_bounds__(128, 5)
    k_far32_both(unit_t nunits, unit_t* __restrict__ counter, const longlong4* __restrict__ work,
                 const long long* __restrict__ offset, const int* __restrict__ near_first, const int2* __restrict__ near,
                 const float4* __restrict__ xhi, const float4* __restrict__ xlo, const float4* __restrict__ nrm32,
                 const float4* __restrict__ wmu, double* __restrict__ y, double* __restrict__ y2) {
  constexpr int TW = 128, SL = 4;
  __shared__ __align__(16) float tiles[4][6 * TW];
  const int lane = threadIdx.x & 31;
  float* const ssx = tiles[threadIdx.x >> 5];
  while (true) {
    const unit_t unit = take_unit(counter);
    if (unit >= nunits) return;
    const UnitPart u = unit_part(unit, 4);
    const longlong4 w = work[u.item];
    const int ub = (int)w.x + 32 * u.part, ue = min(ub + 32, (int)w.y);
    for (int t0 = ub; t0 < ue;) {
      const float4 oh = xhi[t0], ol = xlo[t0];
      const int i = __float_as_int(oh.w);
      const int t1 = (int)min((long long)ue, offset[i + 1]);
      const bool split = t1 - t0 <= 16;  // the two half-warps take alternate halves of the sources
      const int half = split ? lane >> 4 : 0;
      const int t = t0 + (split ? lane & 15 : lane);
      const bool valid = t < t1;
      float2 xt[3], nt[3];
      {
        const float4 ah = valid ? xhi[t] : oh, al = valid ? xlo[t] : ol;
        const float4 nn = valid ? nrm32[t] : make_float4(0, 0, 0, 0);
        const float a0 = (ah.x - oh.x) + (al.x - ol.x), a1 = (ah.y - oh.y) + (al.y - ol.y),
                    a2 = (ah.z - oh.z) + (al.z - ol.z);
        xt[0] = f2(a0, a0);
        xt[1] = f2(a1, a1);
        xt[2] = f2(a2, a2);
        nt[0] = f2(nn.x, nn.x);
        nt[1] = f2(nn.y, nn.y);
        nt[2] = f2(nn.z, nn.z);
      }
      float sa[3] = {0, 0, 0}, ea[3] = {0, 0, 0}, sb[3] = {0, 0, 0}, eb[3] = {0, 0, 0};
      int k = near_first[i];
      const int ke = near_first[i + 1];
      for (int s0 = (int)w.z; s0 < (int)w.w; s0 += TW) {
        const int cnt = min(TW, (int)w.w - s0), cnt8 = (cnt + 7) & ~7;
        float4 ph[SL];
        bool out[SL];
#pragma unroll
        for (int q = 0; q < SL; ++q) {
          const int l = lane + 32 * q;
          out[q] = l >= cnt;
          ph[q] = l < cnt ? xhi[s0 + l] : make_float4(0, 0, 0, 0);
          if (__float_as_int(ph[q].w) == i) out[q] = true;
        }
        const int tlo = __float_as_int(xhi[s0].w), thi = __float_as_int(xhi[s0 + cnt - 1].w);
        while (k < ke && near[k].y < tlo) ++k;
        for (int e = k; e < ke && near[e].y <= thi; ++e) {
          const int j = near[e].y;
#pragma unroll
          for (int q = 0; q < SL; ++q)
            if (__float_as_int(ph[q].w) == j) out[q] = true;
        }
        if (__all_sync(0xffffffffu, out[0] && out[1] && out[2] && out[3])) continue;
        __syncwarp();  // the warp's reads of the previous tile are done
#pragma unroll
        for (int q = 0; q < SL; ++q) {
          const int l = lane + 32 * q;
          if (!out[q]) {
            const float4 pl = xlo[s0 + l], d = wmu[s0 + l];
            ssx[l] = (oh.x - ph[q].x) + (ol.x - pl.x);
            ssx[TW + l] = (oh.y - ph[q].y) + (ol.y - pl.y);
            ssx[2 * TW + l] = (oh.z - ph[q].z) + (ol.z - pl.z);
            ssx[3 * TW + l] = d.x;
            ssx[4 * TW + l] = d.y;
            ssx[5 * TW + l] = d.z;
          } else {
            ssx[l] = ssx[TW + l] = ssx[2 * TW + l] = 1.0e4f;
            ssx[3 * TW + l] = ssx[4 * TW + l] = ssx[5 * TW + l] = 0.0f;
          }
        }
        __syncwarp();
        const int m = split ? cnt8 / 2 : cnt8;
        float2 p[3] = {f2(0.0f, 0.0f), f2(0.0f, 0.0f), f2(0.0f, 0.0f)}, p2[3] = {p[0], p[0], p[0]};
        pair_tile32_both<TW>(ssx, half * m, m, xt, nt, p, p2);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          two_sum_acc(sa[c], ea[c], p[c].x + p[c].y);
          two_sum_acc(sb[c], eb[c], p2[c].x + p2[c].y);
        }
      }
      if (valid) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          atomicAdd(y + 3 * (long long)t + c, kTractionScale * ((double)sa[c] + (double)ea[c]));
          atomicAdd(y2 + 3 * (long long)t + c, kStokesletScale * ((double)sb[c] + (double)eb[c]));
        }
      }
      t0 = t1;
    }
  }
}

// ------------------------------------------------------------------------------------------
// Weighted density as double-float pairs for the double-float kernels: (w mu) rounded to float32 and
// the rounded remainder, with the bound of their biased sums.
__global__ void k_weight_df(long long N, const double4* __restrict__ x, const double* __restrict__ dens,
                            float4* __restrict__ wh, float4* __restrict__ wl, unit_t* __restrict__ units) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (t < 2) units[t] = 0;
  if (t >= N) return;
  const double w = x[t].w;
  const dflt a = df_split(w * dens[3 * t]), b = df_split(w * dens[3 * t + 1]), c = df_split(w * dens[3 * t + 2]);
  wh[t] = make_float4(a.h, b.h, c.h, bias_bound(a.h, b.h, c.h));
  wl[t] = make_float4(a.l, b.l, c.l, 0.0f);
}


// Direct double-float pair sums: y += traction sum (KIND 0, 2) or Stokeslet sum (KIND 1); KIND 2 also
// y2 += Stokeslet sum.  A unit is 32 targets of a work item against its sources; warps take units from
// a counter, stage their own source tiles and never wait for one another (df_tile, shared with the
// treecode).  No float64 arithmetic runs but the final accumulation per target.  Bound by the float32 pipe, 84%
// busy: both sums 126 to 153 Gpair/s (101 particles of 220 nodes; 150 since near sources are left out, on as many
// instructions), the traction alone 195 to 219 (500 of 220), against two-sum arithmetic throughout in blocks of whole
// items.
template <int KIND>
__global__ void __launch_bounds__(128, 4) k_pairs_df2(unit_t nunits, unit_t* __restrict__ counter,
                                                      const longlong4* __restrict__ work, DfSkip skip,
                                                      const float4* __restrict__ x3h, const float4* __restrict__ x3m,
                                                      const float4* __restrict__ x3l, const float4* __restrict__ nh,
                                                      const float4* __restrict__ nl, const float4* __restrict__ wh,
                                                      const float4* __restrict__ wl, double* __restrict__ y,
                                                      double* __restrict__ y2) {
  __shared__ __align__(16) float tiles[4 * kTileDfFloats];
  __shared__ int skips[4][kDfSkipInts];
  int* const sk = skips[threadIdx.x >> 5];
  float* const wsm = tiles + (threadIdx.x >> 5) * kTileDfFloats;
  const int lane = threadIdx.x & 31;
  while (true) {
    const unit_t unit = take_unit(counter);
    if (unit >= nunits) return;
    const UnitPart u = unit_part(unit, 4);
    const longlong4 w = work[u.item];
    const int t0 = (int)w.x + 32 * u.part, t1 = (int)w.y;
    if (t0 >= t1) continue;
    const bool split = t1 - t0 <= 16;
    const int half = split ? lane >> 4 : 0;
    const int t = t0 + (split ? lane & 15 : lane);
    const bool valid = t < t1;
    const float4 oh = x3h[t0], om = x3m[t0], ol = x3l[t0];
    dflt xt[3], nt[3], a[3], a2[3];
    const int pid0 = __float_as_int(oh.w);
    int bit = 0;
    df_skip_targets(skip, pid0, __float_as_int(x3h[min(t0 + 32, t1) - 1].w), sk);
    {
      float4 ah = oh, am = om, al = ol, bh = make_float4(0, 0, 0, 0), bl = make_float4(0, 0, 0, 0);
      if (valid) {
        ah = x3h[t];
        am = x3m[t];
        al = x3l[t];
        bh = nh[t];
        bl = nl[t];
        bit = 1 << (__float_as_int(ah.w) - pid0);
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
    for (int s0 = (int)w.z; s0 < (int)w.w; s0 += kTileDf) {
      const int cnt = min(kTileDf, (int)w.w - s0);
      const int sidx[2] = {s0 + lane, s0 + lane + 32};
      const int tlo = __float_as_int(x3h[s0].w), thi = __float_as_int(x3h[s0 + cnt - 1].w);
      if (df_skip_any(sk, tlo, thi))
        df_tile<KIND, true>(wsm, sidx, cnt, skip, sk, split, half, x3h, x3m, x3l, wh, wl, oh, om, ol, xt, nt, xm, bit, a,
                            a2);
      else
        df_tile<KIND, false>(wsm, sidx, cnt, skip, sk, split, half, x3h, x3m, x3l, wh, wl, oh, om, ol, xt, nt, xm, bit, a,
                             a2);
    }
    const double sc = KIND == 1 ? kStokesletScale : kTractionScale;
    if (valid) {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        atomicAdd(y + 3 * (long long)t + c, sc * ((double)a[c].h + (double)a[c].l));
        if (KIND == 2) atomicAdd(y2 + 3 * (long long)t + c, kStokesletScale * ((double)a2[c].h + (double)a2[c].l));
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// Upsampled densities of the near-source particles: mu_up = U mu_j with U stored transposed (N_p x N_up),
// in the arithmetic of U's storage type (float32 for the inner solve, float64 otherwise).  One block takes
// 64 upsampled nodes of up to four particles of one grid: its threads read U coalesced, each entry once for
// the four, in four groups that share the sum over the grid's nodes (kUpTile of them staged at a time), so that
// a few particles still fill a block and many read U from L2 a quarter as often.  The near sums take the
// results weighted: FORM 0 w mu as float64 (qd), 1 as float32 (qh), 2 as float32 pairs (qh, ql).
constexpr int kUpRows = 64, kUpTile = 64;

template <typename TU, int FORM>
__global__ void __launch_bounds__(256) k_upsample(const int4* __restrict__ groups, const int* __restrict__ up_particle,
                                                  const long long* __restrict__ up_off,
                                                  const long long* __restrict__ offset, const int* __restrict__ nodes,
                                                  const TU* const* __restrict__ Umats, const double* __restrict__ dens,
                                                  const double4* __restrict__ upx, double4* __restrict__ qd,
                                                  float4* __restrict__ qh, float4* __restrict__ ql) {
  __shared__ __align__(16) TU mus[kUpTile][12];
  __shared__ TU part[3][12][kUpRows];
  const int4 gr = groups[blockIdx.y];
  const int us[4] = {gr.x, gr.y, gr.z, gr.w};
  const int np = nodes[up_particle[gr.x]];
  const int nup = (int)(up_off[gr.x + 1] - up_off[gr.x]);
  const int r0 = blockIdx.x * kUpRows;
  if (r0 >= nup) return;
  const int row = threadIdx.x % kUpRows, sg = threadIdx.x / kUpRows;
  const int r = min(r0 + row, nup - 1);
  const TU* Ut = Umats[gr.x] + r;
  TU acc[12];
#pragma unroll
  for (int q = 0; q < 12; ++q) acc[q] = 0;
  for (int s0 = 0; s0 < np; s0 += kUpTile) {
    const int cnt = min(kUpTile, np - s0);
    __syncthreads();
    for (int e = threadIdx.x; e < 12 * kUpTile; e += 256) {
      const int s = (e / 3) % kUpTile, p = e / (3 * kUpTile), k = e % 3;
      TU v = 0;
      if (us[p] >= 0 && s < cnt) v = (TU)dens[3 * (offset[up_particle[us[p]]] + s0 + s) + k];
      mus[s][3 * p + k] = v;
    }
    __syncthreads();
    // the tile's rows of this group: sg, sg + 4, ... (zero densities beyond cnt; U stays in bounds)
#pragma unroll 8
    for (int s = sg; s < kUpTile; s += 4) {
      const TU u = __ldg(Ut + (long long)min(s0 + s, np - 1) * nup);
#pragma unroll
      for (int q = 0; q < 12; ++q) acc[q] = fma_t(u, mus[s][q], acc[q]);
    }
  }
  __syncthreads();
  if (sg > 0)
#pragma unroll
    for (int q = 0; q < 12; ++q) part[sg - 1][q][row] = acc[q];
  __syncthreads();
  // group sg finishes particle sg
  if (sg == 0)
#pragma unroll
    for (int q = 0; q < 12; ++q) {
      const TU v = acc[q] + part[0][q][row] + part[1][q][row] + part[2][q][row];
      part[0][q][row] = v;
    }
  __syncthreads();
  const int u = us[sg];
  if (u < 0 || r0 + row >= nup) return;
  const long long o = up_off[u] + r0 + row;
  const double w = upx[o].w;
  const double q0 = w * (double)part[0][3 * sg][row], q1 = w * (double)part[0][3 * sg + 1][row],
               q2 = w * (double)part[0][3 * sg + 2][row];
  if (FORM == 0) qd[o] = make_double4(q0, q1, q2, 0.0);
  if (FORM == 1) qh[o] = make_float4((float)q0, (float)q1, (float)q2, 0.0f);
  if (FORM == 2) {
    const dflt d0 = df_split(q0), d1 = df_split(q1), d2 = df_split(q2);
    qh[o] = make_float4(d0.h, d1.h, d2.h, bias_bound(d0.h, d1.h, d2.h));
    ql[o] = make_float4(d0.l, d1.l, d2.l, 0.0f);
  }
}

// Near correction by the units of near.cuh.

// Float32: the packed tile loop of the smooth sum over per-warp tiles of 128 sources.  Bound by the float32 pipe;
// against one block per pair, a solve's 17 corrections (one double-float) with 398 pairs in 24 suspensions of mixed
// orders went from 28 to 5.8 ms with their upsampling, and with 6,582 pairs of 144-node particles from 31 to 22.5 ms.
template <int KIND>
__global__ void __launch_bounds__(128, 6) k_near32(NearArgs A, const float4* __restrict__ xhi,
                                                   const float4* __restrict__ xlo, const float4* __restrict__ nrm32,
                                                   const float4* __restrict__ wmu, const float4* __restrict__ uphi,
                                                   const float4* __restrict__ uplo, const float4* __restrict__ upq,
                                                   double* __restrict__ y) {
  constexpr int TW = 128;
  __shared__ __align__(16) float tiles[4][6 * TW];
  const int lane = threadIdx.x & 31;
  float* const ssx = tiles[threadIdx.x >> 5];
  NearUnit n;
  while (next_near_unit(A, n)) {
    if (n.s0 >= n.s1) continue;
    const bool split = n.t1 - n.t0 <= 16;
    const int half = split ? lane >> 4 : 0;
    const int t = n.t0 + (split ? lane & 15 : lane);
    const bool valid = t < n.t1;
    const float4 oh = xhi[n.t0], ol = xlo[n.t0];
    float2 xt[1][3], nt[1][3];
    const int none[1] = {-1};
    {
      const float4 ah = valid ? xhi[t] : oh, al = valid ? xlo[t] : ol;
      const float4 nn = valid ? nrm32[t] : make_float4(0, 0, 0, 0);
      const float a0 = (ah.x - oh.x) + (al.x - ol.x), a1 = (ah.y - oh.y) + (al.y - ol.y),
                  a2 = (ah.z - oh.z) + (al.z - ol.z);
      xt[0][0] = f2(a0, a0);
      xt[0][1] = f2(a1, a1);
      xt[0][2] = f2(a2, a2);
      nt[0][0] = f2(nn.x, nn.x);
      nt[0][1] = f2(nn.y, nn.y);
      nt[0][2] = f2(nn.z, nn.z);
    }
    float sa[3] = {0, 0, 0}, ea[3] = {0, 0, 0};
    for (int sb = n.s0; sb < n.s1; sb += TW) {
      const int cnt = min(TW, n.s1 - sb), cnt8 = (cnt + 7) & ~7;
      __syncwarp();  // the warp's reads of the previous tile are done
#pragma unroll
      for (int l = lane; l < TW; l += 32) {
        if (l < cnt) {
          const int s = sb + l;
          float4 ph, pl, q;
          if (s < n.nup) {
            ph = uphi[n.ub + s];
            pl = uplo[n.ub + s];
            q = upq[n.ub + s];
          } else {
            const long long g = n.oj + (s - n.nup);
            ph = xhi[g];
            pl = xlo[g];
            q = wmu[g];
            q = make_float4(-q.x, -q.y, -q.z, 0.0f);
          }
          ssx[l] = (oh.x - ph.x) + (ol.x - pl.x);
          ssx[TW + l] = (oh.y - ph.y) + (ol.y - pl.y);
          ssx[2 * TW + l] = (oh.z - ph.z) + (ol.z - pl.z);
          ssx[3 * TW + l] = q.x;
          ssx[4 * TW + l] = q.y;
          ssx[5 * TW + l] = q.z;
        } else if (l < cnt8) {
          ssx[l] = ssx[TW + l] = ssx[2 * TW + l] = 1.0e4f;
          ssx[3 * TW + l] = ssx[4 * TW + l] = ssx[5 * TW + l] = 0.0f;
        }
      }
      __syncwarp();
      float2 p[1][3];
      p[0][0] = p[0][1] = p[0][2] = f2(0.0f, 0.0f);
      const int m = split ? cnt8 / 2 : cnt8, l0 = half * m;
      pair_tile32x2<KIND, false, 1>(ssx + l0, ssx + TW + l0, ssx + 2 * TW + l0, ssx + 3 * TW + l0, ssx + 4 * TW + l0,
                                    ssx + 5 * TW + l0, nullptr, m, xt, nt, none, p);
#pragma unroll
      for (int c = 0; c < 3; ++c) two_sum_acc(sa[c], ea[c], p[0][c].x + p[0][c].y);
    }
    if (valid) {
      const double sc = KIND == 0 ? kTractionScale : kStokesletScale;
#pragma unroll
      for (int c = 0; c < 3; ++c) atomicAdd(y + 3 * (long long)t + c, sc * ((double)sa[c] + (double)ea[c]));
    }
  }
}

// Double-float, upsampled nodes alone (df_tile: the smooth sums leave near sources out); KIND 2 both kernels in one
// pass.
template <int KIND>
__global__ void __launch_bounds__(128, 4) k_near_df(NearArgs A, const float4* __restrict__ x3h,
                                                    const float4* __restrict__ x3m, const float4* __restrict__ x3l,
                                                    const float4* __restrict__ nh, const float4* __restrict__ nl,
                                                    const float4* __restrict__ up3h, const float4* __restrict__ up3m,
                                                    const float4* __restrict__ up3l, const float4* __restrict__ upqh,
                                                    const float4* __restrict__ upql, double* __restrict__ y,
                                                    double* __restrict__ y2) {
  __shared__ __align__(16) float tiles[4 * kTileDfFloats];
  float* const wsm = tiles + (threadIdx.x >> 5) * kTileDfFloats;
  const int lane = threadIdx.x & 31;
  NearUnit n;
  while (next_near_unit(A, n)) {
    if (n.s0 >= n.s1) continue;
    const bool split = n.t1 - n.t0 <= 16;
    const int half = split ? lane >> 4 : 0;
    const int t = n.t0 + (split ? lane & 15 : lane);
    const bool valid = t < n.t1;
    const float4 oh = x3h[n.t0], om = x3m[n.t0], ol = x3l[n.t0];
    dflt xt[3], nt[3], a[3], a2[3];
    {
      const float4 zero = make_float4(0, 0, 0, 0);
      const float4 ah = valid ? x3h[t] : oh, am = valid ? x3m[t] : om, al = valid ? x3l[t] : ol;
      const float4 bh = valid ? nh[t] : zero, bl = valid ? nl[t] : zero;
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
    for (int sb = n.s0; sb < n.s1; sb += kTileDf) {
      const int sidx[2] = {(int)(n.ub + sb) + lane, (int)(n.ub + sb) + lane + 32};
      df_tile<KIND, false>(wsm, sidx, min(kTileDf, n.s1 - sb), DfSkip{}, nullptr, split, half, up3h, up3m, up3l, upqh, upql, oh, om, ol, xt, nt,
                    xm, 0, a, a2);
    }
    if (valid) {
      const double sc = KIND == 1 ? kStokesletScale : kTractionScale;
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        atomicAdd(y + 3 * (long long)t + c, sc * ((double)a[c].h + (double)a[c].l));
        if (KIND == 2) atomicAdd(y2 + 3 * (long long)t + c, kStokesletScale * ((double)a2[c].h + (double)a2[c].l));
      }
    }
  }
}

// Float64: per-warp tiles of 32 sources; coordinates relative to the target particle's centre cancel in the
// differences, so lab coordinates are used as they are.
template <int KIND>
__global__ void __launch_bounds__(128) k_near64(NearArgs A, const double4* __restrict__ x,
                                                const double4* __restrict__ nrm, const double* __restrict__ dens,
                                                const double4* __restrict__ upx, const double4* __restrict__ upq,
                                                double* __restrict__ y) {
  __shared__ double4 sp[4][32], sq[4][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  NearUnit n;
  while (next_near_unit(A, n)) {
    if (n.s0 >= n.s1) continue;
    const bool split = n.t1 - n.t0 <= 16;  // the half-warps take alternate halves of the sources
    const int half = split ? lane >> 4 : 0;
    const int t = n.t0 + (split ? lane & 15 : lane);
    const bool valid = t < n.t1;
    const double4 xt = x[valid ? t : n.t0], nt = nrm[valid ? t : n.t0];
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    for (int sb = n.s0; sb < n.s1; sb += 32) {
      const int cnt = min(32, n.s1 - sb);
      __syncwarp();
      if (lane < cnt) {
        const int s = sb + lane;
        if (s < n.nup) {
          sp[warp][lane] = upx[n.ub + s];
          sq[warp][lane] = upq[n.ub + s];
        } else {
          const long long g = n.oj + (s - n.nup);
          const double4 p = x[g];
          sp[warp][lane] = p;
          sq[warp][lane] = make_double4(-p.w * dens[3 * g], -p.w * dens[3 * g + 1], -p.w * dens[3 * g + 2], 0.0);
        }
      }
      __syncwarp();
#pragma unroll 4
      for (int l = half; l < cnt; l += split ? 2 : 1) {
        const double4 ps = sp[warp][l], q = sq[warp][l];
        const double dx = xt.x - ps.x, dy = xt.y - ps.y, dz = xt.z - ps.z;
        const double inv = rsqrt(dx * dx + dy * dy + dz * dz);
        const double rr = dx * q.x + dy * q.y + dz * q.z;
        if (KIND == 0) {
          const double inv2 = inv * inv;
          const double rn = dx * nt.x + dy * nt.y + dz * nt.z;
          const double c = rn * rr * (inv2 * inv2 * inv);
          a0 = fma(c, dx, a0);
          a1 = fma(c, dy, a1);
          a2 = fma(c, dz, a2);
        } else {
          const double c = rr * (inv * inv * inv);
          a0 = fma(c, dx, fma(q.x, inv, a0));
          a1 = fma(c, dy, fma(q.y, inv, a1));
          a2 = fma(c, dz, fma(q.z, inv, a2));
        }
      }
    }
    if (split) {  // one addition per target
      a0 += __shfl_xor_sync(0xffffffffu, a0, 16);
      a1 += __shfl_xor_sync(0xffffffffu, a1, 16);
      a2 += __shfl_xor_sync(0xffffffffu, a2, 16);
    }
    if (valid && half == 0) {
      const double sc = KIND == 0 ? kTractionScale : kStokesletScale;
      atomicAdd(y + 3 * (long long)t + 0, sc * a0);
      atomicAdd(y + 3 * (long long)t + 1, sc * a1);
      atomicAdd(y + 3 * (long long)t + 2, sc * a2);
    }
  }
}

}  // namespace

// Weighted densities of the float32 and double-float pair sums; they also zero the unit counters (d_unit: smooth
// sum, near correction), so each is followed by at most one of either sum.
static Status weight_f32(Context& c, const double* x) {
  k_weight_f32<<<cdiv(c.N, 256), 256, 0, c.stream>>>(c.N, c.d_x.ptr, x, c.d_wmu32.ptr, c.d_unit.ptr);
  RBS_CUDA_TRY(cudaGetLastError());
  return Status::Ok();
}
static Status weight_df(Context& c, const double* x) {
  k_weight_df<<<cdiv(c.N, 256), 256, 0, c.stream>>>(c.N, c.d_x.ptr, x, c.d_wmuh.ptr, c.d_wmul.ptr,
                                                           c.d_unit.ptr);
  RBS_CUDA_TRY(cudaGetLastError());
  return Status::Ok();
}

// Blocks of `kernel` that fit on the GPU at once (occupancy x SMs), capped at the item count: the
// pair kernels loop over their work items with this persistent grid, so the last wave is not a
// mostly idle second pass over the SMs.
static int resident_grid(Context& c, const void* kernel, int threads, int items) {
  auto it = c.resident.find(kernel);
  int per_sm = 0;
  if (it == c.resident.end()) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) != cudaSuccess || per_sm < 1)
      per_sm = 1;
    c.resident[kernel] = per_sm;
  } else {
    per_sm = it->second;
  }
  return std::max(1, std::min(items, per_sm * std::max(1, c.sm_count)));
}

// Targets per lane of the direct float32 sums: two, which share each source's loads, once that still makes 24
// units per SM (a round of its warps); one below, and where rbs_options.pair_variant asks for it.  Traction, us an
// apply with one and two on p = 8 (p = 10): at 1 unit of two targets per SM 9.8 and 12.8, at 7 (16.0 and 22.0), at 10
// 18.0 and 24.8, at 17 24.2 and 26.1, at 19 (26.1 and 26.2), at 27 33.4 and 32.3, at 38 44.1 and 41.5, at 43 (46.7
// and 44.6), at 68 69.2 and 65.7; above, two is 2 to 8% faster.  The Stokeslet sums cross at the same place.
static int pairs32_targets(const Context& c) {
  const int v = c.opt.pair_variant;
  if (v > 0) return v == 1 || v == kPacked + 1 ? 1 : 2;
  return 2 * (long long)c.work.size() >= 24LL * c.sm_count ? 2 : 1;
}

int direct_variant(const Context& c) { return kPacked + pairs32_targets(c); }

template <int KIND, int NT>
static void launch_pairs32(Context& c, double* y) {
  const int items = (int)c.work.size();
  const auto kernel = k_pairs32x2<KIND, NT>;
  kernel<<<resident_grid(c, (const void*)kernel, 128, items), 128, 0, c.stream>>>(
      (unit_t)(4 / NT) * items, c.d_unit.ptr, c.d_work.ptr, c.d_xhi.ptr, c.d_xlo.ptr, c.d_nrm32.ptr, c.d_wmu32.ptr, y);
}

template <int KIND>
static void launch_pairs_df(Context& c, double* y, double* y2) {
  const int items = (int)c.work.size();
  k_pairs_df2<KIND><<<resident_grid(c, (const void*)k_pairs_df2<KIND>, 128, items), 128, 0, c.stream>>>(
      (unit_t)4 * items, c.d_unit.ptr, c.d_work.ptr, DfSkip{c.d_near_first.ptr, c.d_near.ptr}, c.d_x3h.ptr, c.d_x3m.ptr,
      c.d_x3l.ptr, c.d_nrmh.ptr, c.d_nrml.ptr,
      c.d_wmuh.ptr, c.d_wmul.ptr, y, y2);
}

// Launch of the direct smooth pair sum; kind 2 (traction into y and Stokeslet into y2 in one pass) is for
// double-float (k_far32_both is float32's, without near sources).  The float32 and double-float sums read the weighted
// densities of this x.
static Status launch_pairs(Context& c, int kind, int prec, const double* x, double* y, double* y2 = nullptr) {
  const int items = (int)c.work.size();
  if (prec == RBS_PREC_DF) {
    if (kind == 0)
      launch_pairs_df<0>(c, y, y2);
    else if (kind == 1)
      launch_pairs_df<1>(c, y, y2);
    else
      launch_pairs_df<2>(c, y, y2);
  } else if (prec == RBS_PREC_FP64) {
#define RBS_PAIR_ARGS items, c.d_work.ptr, c.d_x.ptr, c.d_nrm.ptr, c.d_pid.ptr, x, y
    if (kind == 0)
      k_pairs64<0><<<resident_grid(c, (const void*)k_pairs64<0>, 128, items), 128, 0, c.stream>>>(RBS_PAIR_ARGS);
    else
      k_pairs64<1><<<resident_grid(c, (const void*)k_pairs64<1>, 128, items), 128, 0, c.stream>>>(RBS_PAIR_ARGS);
#undef RBS_PAIR_ARGS
  } else if (pairs32_targets(c) == 1) {
    kind == 0 ? launch_pairs32<0, 1>(c, y) : launch_pairs32<1, 1>(c, y);
  } else {
    kind == 0 ? launch_pairs32<0, 2>(c, y) : launch_pairs32<1, 2>(c, y);
  }
  RBS_CUDA_TRY(cudaGetLastError());
  return Status::Ok();
}

// ------------------------------------------------------------------------------------------

Status apply_blocks(Context& c, int mode, int prec, const double* x, double* y, double* aux, double scale) {
  if (mode == kModeZero) {
    c.stats.launches += 1;
    RBS_CUDA_TRY(cudaMemsetAsync(y, 0, sizeof(double) * 3 * c.N, c.stream));
    return Status::Ok();
  }
  const int nb = (int)c.bwork.size();
  const int ns = (int)c.sym_list.size();
  const bool kblock = mode == kModeSelfK || mode == kModeSelfKNoL || mode == kModeKOnlySelf || mode == kModePrecond;
  const bool use32 = prec_f32(prec) && kblock;
  // 16-bit entries for the ellipsoid blocks of the inner solve's arithmetic (coefficient surfaces,
  // which store every row, keep float32 blocks)
  const bool use16 = prec_16(prec) && kblock && c.d_blockK16.ptr;
  const double bytes = (mode == kModeL) ? 0.0 : (double)c.particle_block_entries * (use16 ? 2.0 : use32 ? 4.0 : 8.0);
  KernelTimer timer(c, use32 ? RBS_KC_BLOCKS : RBS_KC_BLOCKS_F64);
  // 16-bit modes: ellipsoids of shapes shared by many particles go through the tensor-core GEMM, the
  // others through the CUDA-core kernel below
  const bool gemm = use16 && !c.gemm.empty();
  const int* sym_ids = gemm ? c.d_sym_rest.ptr : c.d_sym_list.ptr;
  const int nsym = gemm ? (int)c.sym_rest.size() : ns;
  if (gemm) RBS_TRY(apply_self_gemm(c, mode, x, y, aux, scale));
  if (nsym > 0) {
    const size_t zs = (size_t)sym_smem_bytes(c.max_np_sym, use16 ? 2 : use32 ? 4 : 8, use32 ? 4 : 8);
    // parts of a particle: about six CTAs per SM, and no more than its runs of kSymWarps representatives
    int runs = 1;
    for (Grid* g : c.grids) runs = std::max(runs, (g->nrep + kSymWarps - 1) / kSymWarps);
    const int parts = mode == kModeL ? 1 : std::max(1, std::min(runs, (6 * c.sm_count + nsym - 1) / nsym));
    const dim3 grid(nsym, parts);
#define RBS_SYM_ARGS                                                                                              \
  mode, sym_ids, c.d_offset.ptr, c.d_p.ptr, c.d_nphi.ptr, c.d_rot.ptr, c.d_centre.ptr, c.d_shape.ptr, \
      c.d_block_off.ptr, B, c.d_x.ptr, x, y, aux, scale
    if (use16) {
      const uint16_t* B16 = (mode == kModePrecond) ? c.d_precond16.ptr : c.d_blockK16.ptr;
      if (prec == RBS_PREC_MIXED_FP16) {
        const F16Bits* B = reinterpret_cast<const F16Bits*>(B16);
        if (zs > 48 * 1024)
          RBS_CUDA_TRY(cudaFuncSetAttribute(k_blocks_sym<F16Bits, float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)zs));
        k_blocks_sym<F16Bits, float><<<grid, kSymWarps * 32, zs, c.stream>>>(RBS_SYM_ARGS);
      } else {
        const BF16Bits* B = reinterpret_cast<const BF16Bits*>(B16);
        if (zs > 48 * 1024)
          RBS_CUDA_TRY(cudaFuncSetAttribute(k_blocks_sym<BF16Bits, float>,
                                            cudaFuncAttributeMaxDynamicSharedMemorySize, (int)zs));
        k_blocks_sym<BF16Bits, float><<<grid, kSymWarps * 32, zs, c.stream>>>(RBS_SYM_ARGS);
      }
    } else if (use32) {
      const float* B = (mode == kModePrecond) ? c.d_precond32.ptr : c.d_blockK32.ptr;
      if (zs > 48 * 1024)
        RBS_CUDA_TRY(cudaFuncSetAttribute(k_blocks_sym<float, float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)zs));
      k_blocks_sym<float, float><<<grid, kSymWarps * 32, zs, c.stream>>>(RBS_SYM_ARGS);
    } else {
      const double* B = (mode == kModePrecond) ? c.d_precond.ptr : (mode == kModeSelfS ? c.d_blockS.ptr : c.d_blockK.ptr);
      if (zs > 48 * 1024)
        RBS_CUDA_TRY(cudaFuncSetAttribute(k_blocks_sym<double, double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)zs));
      k_blocks_sym<double, double><<<grid, kSymWarps * 32, zs, c.stream>>>(RBS_SYM_ARGS);
    }
#undef RBS_SYM_ARGS
    RBS_CUDA_TRY(cudaGetLastError());
  }
  if (nb == 0) {
    timer.done(bytes);
    return Status::Ok();
  }
  const size_t smem = (use32 ? sizeof(float) : sizeof(double)) * 3 * (size_t)c.max_np;
  if (use32) {
    const float* B = (mode == kModePrecond) ? c.d_precond32.ptr : c.d_blockK32.ptr;
    if (smem > 48 * 1024)
      RBS_CUDA_TRY(cudaFuncSetAttribute(k_blocks<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_blocks<float><<<nb, 256, smem, c.stream>>>(mode, c.d_bwork.ptr, c.d_offset.ptr, c.d_nodes.ptr, c.d_rot.ptr,
                                                 c.d_centre.ptr, c.d_shape.ptr, c.d_block_off.ptr, B, c.d_x.ptr, x, y,
                                                 aux, scale);
  } else {
    const double* B = (mode == kModePrecond) ? c.d_precond.ptr : (mode == kModeSelfS ? c.d_blockS.ptr : c.d_blockK.ptr);
    if (smem > 48 * 1024)
      RBS_CUDA_TRY(cudaFuncSetAttribute(k_blocks<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    k_blocks<double><<<nb, 256, smem, c.stream>>>(mode, c.d_bwork.ptr, c.d_offset.ptr, c.d_nodes.ptr, c.d_rot.ptr,
                                                  c.d_centre.ptr, c.d_shape.ptr, c.d_block_off.ptr, B, c.d_x.ptr, x, y,
                                                  aux, scale);
  }
  RBS_CUDA_TRY(cudaGetLastError());
  timer.done(bytes);
  return Status::Ok();
}

// Near correction, step 1: upsampled weighted densities of the near-source particles (float32
// interpolation for the inner solve, float64 otherwise), in the form the sums of arithmetic prec read.
static Status near_upsample(Context& c, int prec, const double* x) {
  int maxup = 0;
  for (Grid* g : c.grids) maxup = std::max(maxup, g->nup);
  const int ng = (int)c.up_groups.size();
#define RBS_UPSAMPLE(TU, FORM, U)                                                                                     \
  k_upsample<TU, FORM><<<dim3(cdiv(maxup, kUpRows), cnt), 256, 0, c.stream>>>(                                        \
      c.d_up_groups.ptr + g0, c.d_up_particle.ptr, c.d_up_off.ptr, c.d_offset.ptr, c.d_nodes.ptr, U, x, c.d_up_x.ptr, \
      c.d_up_q.ptr, c.d_up_qh.ptr, c.d_up_ql.ptr)
  for (int g0 = 0; g0 < ng; g0 += 65535) {
    const int cnt = std::min(65535, ng - g0);
    if (prec_f32(prec))
      RBS_UPSAMPLE(float, 1, c.d_upU32.ptr);
    else if (prec == RBS_PREC_DF)
      RBS_UPSAMPLE(double, 2, c.d_upU.ptr);
    else
      RBS_UPSAMPLE(double, 0, c.d_upU.ptr);
  }
#undef RBS_UPSAMPLE
  RBS_CUDA_TRY(cudaGetLastError());
  return Status::Ok();
}

// Node pairs of one near correction.
static double near_units(const Context& c, int prec) {
  return prec == RBS_PREC_DF ? c.near_pair_nodes - c.near_base_nodes : c.near_pair_nodes;
}

// Near correction, step 2: for every near pair, the base-grid term is replaced by the upsampled one (double-float: the
// upsampled one is added); kind 0 traction into y, 1 Stokeslet into y, 2 (double-float only) traction into y and
// Stokeslet into y2.
static Status near_sums(Context& c, int kind, int prec, const double* x, double* y, double* y2) {
  NearArgs A;
  int blocks = 0;
  RBS_TRY(near_args(c, prec != RBS_PREC_DF, A, blocks));
  if (prec == RBS_PREC_FP64) RBS_CUDA_TRY(cudaMemsetAsync(A.counter, 0, sizeof(unit_t), c.stream));
#define RBS_NEAR_LAUNCH(KERNEL, ...) \
  KERNEL<<<resident_grid(c, (const void*)KERNEL, 128, blocks), 128, 0, c.stream>>>(A, __VA_ARGS__)
  if (prec == RBS_PREC_DF) {
#define RBS_NEAR_DF c.d_x3h.ptr, c.d_x3m.ptr, c.d_x3l.ptr, c.d_nrmh.ptr, c.d_nrml.ptr, \
                    c.d_up3h.ptr, c.d_up3m.ptr, c.d_up3l.ptr, c.d_up_qh.ptr, c.d_up_ql.ptr, y, y2
    if (kind == 0)
      RBS_NEAR_LAUNCH(k_near_df<0>, RBS_NEAR_DF);
    else if (kind == 1)
      RBS_NEAR_LAUNCH(k_near_df<1>, RBS_NEAR_DF);
    else
      RBS_NEAR_LAUNCH(k_near_df<2>, RBS_NEAR_DF);
#undef RBS_NEAR_DF
  } else if (prec_f32(prec)) {
#define RBS_NEAR_32 c.d_xhi.ptr, c.d_xlo.ptr, c.d_nrm32.ptr, c.d_wmu32.ptr, c.d_up3h.ptr, c.d_up3m.ptr, c.d_up_qh.ptr, y
    if (kind == 0)
      RBS_NEAR_LAUNCH(k_near32<0>, RBS_NEAR_32);
    else
      RBS_NEAR_LAUNCH(k_near32<1>, RBS_NEAR_32);
#undef RBS_NEAR_32
  } else {
#define RBS_NEAR_64 c.d_x.ptr, c.d_nrm.ptr, x, c.d_up_x.ptr, c.d_up_q.ptr, y
    if (kind == 0)
      RBS_NEAR_LAUNCH(k_near64<0>, RBS_NEAR_64);
    else
      RBS_NEAR_LAUNCH(k_near64<1>, RBS_NEAR_64);
#undef RBS_NEAR_64
  }
#undef RBS_NEAR_LAUNCH
  RBS_CUDA_TRY(cudaGetLastError());
  return Status::Ok();
}

Status apply_pairs(Context& c, int kind, int prec, const double* x, double* y) {
  const int nw = (int)c.work.size();
  const bool f32 = prec_f32(prec);
  // the weighted densities that the smooth sums and the near correction read
  if (f32) {
    c.stats.launches++;
    RBS_TRY(weight_f32(c, x));
  } else if (prec == RBS_PREC_DF) {
    c.stats.launches++;
    RBS_TRY(weight_df(c, x));
  }
  // The float32 near correction of a small system runs beside the smooth sum (both add into y atomically): each
  // alone leaves SMs idle at its end.  Solves to 1e-6 after one another and beside, ms: 1.51 and 1.44 at 3,456 nodes,
  // 2.95 and 2.83 at 8,640, 5.73 and 5.50 at 14,544, 16.95 and 16.63 at 28,800, 49.2 and 48.7 at 57,600, 86.2 and 85.8
  // at 79,200, 165.8 and 165.4 at 115,200, 210.3 and 209.7 at 129,600: a saving of 0.1 to 0.5 ms at every size, 0.3%
  // where the line is drawn.  Not while kernel classes are timed.
  const bool beside = f32 && c.side && !c.near_pairs.empty() && c.N <= kBesideNodes && c.opt.timing == 0;
  if (beside) {
    RBS_CUDA_TRY(cudaEventRecord(c.fork_ev, c.stream));
    RBS_CUDA_TRY(cudaStreamWaitEvent(c.side, c.fork_ev, 0));
    const cudaStream_t main = c.stream;
    c.stream = c.side;
    Status st = near_upsample(c, prec, x);
    if (st.ok()) st = near_sums(c, kind, prec, x, y, nullptr);
    c.stream = main;
    c.stats.launches += 2;
    c.stats.kernel_count[RBS_KC_NEAR] += 2;
    c.stats.kernel_units[RBS_KC_NEAR] += near_units(c, prec);
    RBS_CUDA_TRY(cudaEventRecord(c.join_ev, c.side));
    if (!st.ok()) {
      cudaStreamWaitEvent(c.stream, c.join_ev, 0);
      return st;
    }
  }
  Status st;
  if (f32 && c.tree.active) {
    st = apply_tree(c, kind, y);  // treecode in place of the direct float32 sum
  } else if (prec == RBS_PREC_DF && c.tree_df.active) {
    st = apply_tree_df(c, kind, x, y, nullptr);  // and of the direct double-float sum
  } else if (nw > 0) {
    int cls = f32 ? (kind == 0 ? RBS_KC_PAIR_K32 : RBS_KC_PAIR_S32) : (kind == 0 ? RBS_KC_PAIR_K64 : RBS_KC_PAIR_S64);
    if (prec == RBS_PREC_DF) cls = kind == 0 ? RBS_KC_PAIR_KDF : RBS_KC_PAIR_SDF;
    KernelTimer timer(c, cls);
    st = launch_pairs(c, kind, prec, x, y);
    timer.done((double)c.stats.far_pairs - (prec == RBS_PREC_DF ? c.near_base_nodes : 0.0));
  }
  if (beside) RBS_CUDA_TRY(cudaStreamWaitEvent(c.stream, c.join_ev, 0));  // (also when the smooth sum failed)
  RBS_TRY(st);
  if (!beside && !c.near_pairs.empty()) {
    KernelTimer timer(c, RBS_KC_NEAR);
    RBS_TRY(near_upsample(c, prec, x));
    RBS_TRY(near_sums(c, kind, prec, x, y, nullptr));
    timer.done(near_units(c, prec), 2);
  }
  return Status::Ok();
}

Status apply_pairs_both(Context& c, int prec, const double* x, double* yK, double* yS) {
  if (prec_f32(prec)) {
    RBS_TRY(apply_pairs(c, 0, prec, x, yK));
    return apply_pairs(c, 1, prec, x, yS);
  }
  const int nw = (int)c.work.size();
  if (prec == RBS_PREC_DF) {
    c.stats.launches++;
    RBS_TRY(weight_df(c, x));
  }
  if (prec == RBS_PREC_DF && c.tree_df.active) {
    RBS_TRY(apply_tree_df(c, 2, x, yK, yS));
  } else if (nw > 0) {
    if (prec == RBS_PREC_DF) {
      KernelTimer timer(c, RBS_KC_PAIR_KSDF);
      RBS_TRY(launch_pairs(c, 2, prec, x, yK, yS));
      timer.done((double)c.stats.far_pairs - c.near_base_nodes);
    } else {
      {
        KernelTimer timer(c, RBS_KC_PAIR_K64);
        RBS_TRY(launch_pairs(c, 0, prec, x, yK));
        timer.done((double)c.stats.far_pairs);
      }
      KernelTimer timer(c, RBS_KC_PAIR_S64);
      RBS_TRY(launch_pairs(c, 1, prec, x, yS));
      timer.done((double)c.stats.far_pairs);
    }
  }
  if (!c.near_pairs.empty()) {
    KernelTimer timer(c, RBS_KC_NEAR);
    RBS_TRY(near_upsample(c, prec, x));
    if (prec == RBS_PREC_DF) {
      RBS_TRY(near_sums(c, 2, prec, x, yK, yS));
      timer.done(2.0 * near_units(c, prec), 2);
    } else {
      RBS_TRY(near_sums(c, 0, prec, x, yK, nullptr));
      RBS_TRY(near_sums(c, 1, prec, x, yS, nullptr));
      timer.done(2.0 * near_units(c, prec), 3);
    }
  }
  return Status::Ok();
}

Status apply_correction(Context& c, const double* d, double* w, double* v, bool cheap) {
  RBS_TRY(apply_blocks(c, kModeSelfK, RBS_PREC_DF, d, w, nullptr, 1.0));
  RBS_TRY(apply_blocks(c, kModeSelfS, RBS_PREC_DF, d, v, nullptr, 1.0));
  c.stats.launches += 2;
  RBS_TRY(weight_f32(c, d));
  RBS_TRY(weight_df(c, d));
  if (cheap) {
    RBS_TRY(apply_tree_both(c, w, v));
  } else if (c.tree_df.active) {
    RBS_TRY(apply_tree_df_f32(c, d, w, v));
  } else if (!c.work.empty()) {
    KernelTimer timer(c, RBS_KC_PAIR_K32);
    const int items = (int)c.work.size();
    k_far32_both<<<resident_grid(c, (const void*)k_far32_both, 128, items), 128, 0, c.stream>>>(
        (unit_t)4 * items, c.d_unit.ptr, c.d_work.ptr, c.d_offset.ptr, c.d_near_first.ptr, c.d_near.ptr, c.d_xhi.ptr, c.d_xlo.ptr,
        c.d_nrm32.ptr, c.d_wmu32.ptr, w, v);
    RBS_CUDA_TRY(cudaGetLastError());
    timer.done(2.0 * ((double)c.stats.far_pairs - c.near_base_nodes));
  }
  if (!c.near_pairs.empty()) {
    KernelTimer timer(c, RBS_KC_NEAR);
    RBS_TRY(near_upsample(c, RBS_PREC_DF, d));
    RBS_TRY(near_sums(c, 2, RBS_PREC_DF, d, w, v));
    timer.done(2.0 * near_units(c, RBS_PREC_DF), 2);
  }
  return Status::Ok();
}

Status apply_operator(Context& c, int op, int prec, const double* x, double* y) {
  switch (op) {
    case RBS_OP_A:
      RBS_TRY(apply_blocks(c, kModeSelfK, prec, x, y, nullptr, 1.0));
      return apply_pairs(c, 0, prec, x, y);
    case RBS_OP_HALF_K:
      RBS_TRY(apply_blocks(c, kModeSelfKNoL, prec, x, y, nullptr, 1.0));
      return apply_pairs(c, 0, prec, x, y);
    case RBS_OP_S:
      RBS_TRY(apply_blocks(c, kModeSelfS, prec, x, y, nullptr, 1.0));
      return apply_pairs(c, 1, prec, x, y);
    case RBS_OP_K_OFF:
      RBS_TRY(apply_blocks(c, kModeZero, prec, x, y, nullptr, 1.0));
      return apply_pairs(c, 0, prec, x, y);
    case RBS_OP_K_SELF:
      return apply_blocks(c, kModeKOnlySelf, prec, x, y, nullptr, 1.0);
    case RBS_OP_S_OFF:
      RBS_TRY(apply_blocks(c, kModeZero, prec, x, y, nullptr, 1.0));
      return apply_pairs(c, 1, prec, x, y);
    case RBS_OP_S_SELF:
      return apply_blocks(c, kModeSelfS, prec, x, y, nullptr, 1.0);
    case RBS_OP_L:
      return apply_blocks(c, kModeL, prec, x, y, nullptr, 1.0);
    default:
      return Status::Err(RBS_EINVAL, "unknown operator id " + std::to_string(op));
  }
}

}  // namespace rbs
