// Spin-1/2 H.v (Eq. 3 of arxiv 2607.25585 with every s_i = 1/2) in rotated
// product bases: the Lanczos steps of runs that start from random vectors, and
// ftlm_apply_h on dense blocks.
//
// Method.  Every pair tensor A_ij (symmetric, 3 x 3) is a sum over a few fixed
// directions u_k of scalars a^k_ij u_k u_k^T, so
//   sum_ij s_i.A_ij.s_j + sum_i h_i.s_i = sum_k [ sum_ij a^k_ij (s_i.u_k)(s_j.u_k) + sum_i h^k_i s_i.u_k ],
// and each bracket is diagonal in the product basis of the eigenstates of
// s.u_k.  With U_k the rotation of every site to that basis,
//   H v = D_0 v + sum_k U_k^+ (D_k (U_k v)),
// where direction 0 is z (no rotation).  A rotation is one 2 x 2 gate a site,
// so the product costs O(n) operations a row instead of the O(n^2) gathered
// pair flips, and every diagonal D_k is a table built once per system.
// Directions besides z: x and y when every tensor is diagonal; three in the xy
// plane 60 degrees apart when z is a principal axis of every tensor (planar
// geometries); else the five axes of an icosahedron around z (with z, their
// projectors span the symmetric tensors).  The sets are tight frames (the six
// lines within 3e-8), so the |D_k| stay on the scale of |H| and nothing cancels.
// Complex64 runs of five steps against complex128, 14 to 27 sites in and out of
// the plane, five to eight seeds each, root mean square of the relative error:
// alpha 4e-8 to 9e-8 (16e-8 at 14 sites) where the gather's is 4e-8 to 11e-8 (63e-8),
// beta and p 3e-8 to 6e-8 in both.
//
// The gate.  All u_k have the same polar angle theta; with t = tan(theta / 2)
// and the azimuth's phase e^{-i phi_k} taken out per down spin,
//   (down, up) -> (down - t up, up + t down),
// one packed FP32 FMA a value; its transpose (t -> -t) inverts it up to
// (1 + t^2), and the product of these factors is folded into D_k.
//
// Passes.  The index is split into its low T bits and the nH = n - T bits above.
//   forward:  w (the step's update, see below) -> W_k = the low bits' gates on
//             e^{-i phi_k downs} w, for every direction k;
//   middle:   W_k <- the high bits' gates, times D_k, the inverse gates
//             (tiles of 2^nH rows x 2^c columns);
//   backward: H v = D_0 v + sum_k e^{+i phi_k downs} (inverse low gates of W_k),
//             then the step's epilogue.
// A tile of 2^T values is exchanged through shared memory between groups of
// four bits; a thread holds the 16 values of a group in registers.  W's order
// serves both sides: with l the low T bits rotated by four, as the forward
// pass's last group leaves them, and h the high bits, value (l, h) is at
// (l >> b, h, low b bits of l): the outer passes move runs of 2^b values, the
// middle pass reads rows of 2^c values 2^b apart.  b = T (whole tiles contiguous)
// while the middle's rows are long; b = 4 (128 bytes) where they are 32 bytes,
// which otherwise lie 2^T values apart: 6.5 -> 5.3 ms for the middle pass over
// 2^26 x 4 values, against 0.2 ms more for the outer ones.
//
// Lanczos step j (x = q_j, y = q_{j-1}, u): the forward pass first finishes the
// previous step, q_j = w' - alpha_{j-1} sigma_{j-1} q_{j-1} with |q_j|^2 (so no
// separate update pass reads and writes the vectors), sets beta_{j-1}, sigma_j;
// the backward pass writes w' = sigma_j H q_j - beta_{j-1} sigma_{j-1} q_{j-1}
// over q_{j-1} and sums alpha_j, p_j.  Partial sums go to one slot a tile and
// are added in a fixed order by the last CTA of the vector.
//
// Its error is relative to the whole vector, where a gathered row's is relative
// to that row's terms, and a value that is not finite reaches every row.  So
// ftlm_apply_h takes these passes only for vectors whose values are spread like a
// Gaussian's (vector_density): no row is then much smaller than the vector but
// those few that a Gaussian vector has too.  The forward pass takes each vector's
// statistics as it reads it; for one that fails, the passes return and the gather
// after them runs.
//
// Bound: memory.  A step moves 8 (7 + 4 K) bytes a value in complex64 (152 for
// K = 3), against 56 for the gather, but the gather's C(n, 2) flips take 3.5 ms
// at n = 20 with 64 vectors, where these passes take 1.67 ms with the update
// (3.8 ms with it before): 6.1 TB/s.  2 x 13 sites, 4 vectors: 33 -> 11.0 ms a
// step, 3.7 TB/s: one CTA an SM loads, exchanges and stores in turn, and the middle
// pass (2.8 TB/s) reads rows of 32 bytes.  In complex128 the FP64 pipe binds both:
// 4 x 4 sites, 50 vectors: 4.0 -> 1.57 ms.  Taking one to eight vectors at a time through the three
// passes, so that W stays in L2, was slower (2.1 to 3.0 ms): each launch then
// has too few tiles.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>

#include "device_common.cuh"
#include "ftlm_internal.h"

namespace ftlm {

namespace {

template <int T>
struct Groups {
  static constexpr int N = (T + 3) / 4;
  __host__ __device__ static constexpr int lo(int g) { return T - 4 - 4 * g > 0 ? T - 4 - 4 * g : 0; }
  // bits of group g's four register bits that belong to it (the last group overlaps the one before)
  __host__ __device__ static constexpr int mask(int g) { return g == 0 || lo(g - 1) - lo(g) >= 4 ? 15 : (1 << (lo(g - 1) - lo(g))) - 1; }
};

__device__ __forceinline__ float2 axpy2(float t, float2 x, float2 y) { return __ffma2_rn(make_float2(t, t), x, y); }
__device__ __forceinline__ double2 axpy2(double t, double2 x, double2 y) {
  return make_double2(fma(t, x.x, y.x), fma(t, x.y, y.y));
}

template <typename v2>
__device__ __forceinline__ v2 cmul(v2 a, v2 b) {
  v2 o;
  o.x = a.x * b.x - a.y * b.y;
  o.y = a.x * b.y + a.y * b.x;
  return o;
}

// the gates of the register bits in `mask` (t -> -t: the inverse gates)
template <typename real, typename v2>
__device__ __forceinline__ void gates(v2 (&v)[16], real t, int mask) {
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    if (!((mask >> b) & 1)) continue;
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      if ((r >> b) & 1) continue;
      const v2 dn = v[r], up = v[r | (1 << b)];
      v[r] = axpy2(-t, up, dn);
      v[r | (1 << b)] = axpy2(t, dn, up);
    }
  }
}

// first element of thread `tid`'s 16 of the group at bits [LO, LO + 4)
template <int LO>
__device__ __forceinline__ int group_base(int tid) {
  return ((tid >> LO) << (LO + 4)) | (tid & ((1 << LO) - 1));
}

// place in W of low part l (rotated) and high part 0; linear in disjoint sets of bits
__host__ __device__ __forceinline__ unsigned w_place(unsigned l, int b, int nH) {
  return ((l >> b) << (b + nH)) | (l & ((1u << b) - 1u));
}

// shared-memory place of element i: one padding value after every 16
// (conflict-free for every group position and both element sizes)
__host__ __device__ constexpr int pad(int i) { return i + (i >> 4); }

template <int LO, typename v2>
__device__ __forceinline__ void smem_st(v2* buf, int base, const v2 (&v)[16]) {
  v2* p = buf + pad(base);
#pragma unroll
  for (int r = 0; r < 16; ++r) p[pad(r << LO)] = v[r];
}
template <int LO, typename v2>
__device__ __forceinline__ void smem_ld(const v2* buf, int base, v2 (&v)[16]) {
  const v2* p = buf + pad(base);
#pragma unroll
  for (int r = 0; r < 16; ++r) v[r] = p[pad(r << LO)];
}

// one middle group of a tile, in place in shared memory
template <typename real, int T, int NT, int SETS, int G, typename v2>
__device__ __forceinline__ void mid_group(v2* buf, real t, int mask) {
  constexpr int LO = Groups<T>::lo(G);
#pragma unroll
  for (int s = 0; s < SETS; ++s) {
    const int base = group_base<LO>(threadIdx.x + s * NT);
    v2 w[16];
    smem_ld<LO>(buf, base, w);
    gates(w, t, mask);
    smem_st<LO>(buf, base, w);
  }
  __syncthreads();
}

// e^{-i phi_k downs} by the number of up spins, [K][kRotMaxN + 1], to shared memory
template <typename real>
__device__ __forceinline__ void stage_phases(typename Cx<real>::v2* ph, const RotArgs& a) {
  const typename Cx<real>::v2* src = reinterpret_cast<const typename Cx<real>::v2*>(a.phases);
  for (int q = threadIdx.x; q < a.K * (kRotMaxN + 1); q += blockDim.x) ph[q] = __ldg(src + q);
}

// binary exponent (biased) of a sum of squares; 0 for zero and denormals
__device__ __forceinline__ int exponent_of(float s) { return (__float_as_int(s) >> 23) & 0xff; }
__device__ __forceinline__ int exponent_of(double s) { return (__double2hiint(s) >> 20) & 0x7ff; }

// Values a dense vector may have below its largest |x|^2: of n values 8 + n / 2^5
// at 2^-12, 8 + n / 2^11 at 2^-18 and 8 + n / 2^17 at 2^-24.  A complex Gaussian
// vector has an eighth to half of the fractions there (its largest of 2^11 to 2^28
// values is 2^3 to 2^5 times the mean, and the fraction below s times the mean is
// s); 8 is its Poisson tail where less than one value is expected.
struct FewBelow {
  int c12, c18, c24;
  __device__ bool in(long long n) const { return c12 <= 8 + (n >> 5) && c18 <= 8 + (n >> 11) && c24 <= 8 + (n >> 17); }
};

// Whether the CTA's values let the vector be dense: spread like those of a complex
// Gaussian -- no zero, few far below the largest (FewBelow, over each CTA's values
// and over the vector's), the CTAs' largest within 2^4 of each other -- and far
// from the ends of the range.  A CTA that says no raises a.sparse[v] and the
// vector's other CTAs return as they start; the sums over all CTAs are the last
// one's to judge.  Integers throughout: the outcome does not depend on the order of
// the CTAs, nor on the other vectors of the block.  A vector that is not dense costs
// the gather and a little: 64 basis states of 20 sites 3.73 -> 3.85 ms, one vector of
// them 0.139 -> 0.155 ms (the passes' launches), at most the forward pass (4.06 ms)
// where only the sums tell; with one flag for the block, raised by its last CTA, one
// such vector among 64 cost 4.12 ms, and 1.92 now.
template <typename real, int NT, int SETS, typename v2>
__device__ __forceinline__ bool vector_density(const RotArgs& a, int v, int tiles, const v2 (&q)[SETS][16]) {
  constexpr int W = NT / 32, N = SETS * 16 * NT;
  constexpr int bias = sizeof(real) == 4 ? 127 : 1023, range = sizeof(real) == 4 ? 60 : 400;
  __shared__ int red[W][2];
  __shared__ int raised;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) raised = __ldcg(a.sparse + v);
  auto each = [&](auto&& fn) {
#pragma unroll
    for (int s = 0; s < SETS; ++s)
#pragma unroll
      for (int r = 0; r < 16; ++r) fn(exponent_of(q[s][r].x * q[s][r].x + q[s][r].y * q[s][r].y));
  };
  int top = 0, low = 0x7fffffff;
  each([&](int e) {
    top = max(top, e);
    low = min(low, e);
  });
  top = __reduce_max_sync(0xffffffffu, top);
  low = __reduce_min_sync(0xffffffffu, low);
  if (lane == 0) {
    red[warp][0] = top;
    red[warp][1] = low;
  }
  __syncthreads();
  if (raised) return false;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    top = max(top, red[w][0]);
    low = min(low, red[w][1]);
  }
  __syncthreads();
  FewBelow f = {0, 0, 0};
  each([&](int e) {
    f.c12 += e <= top - 12;
    f.c18 += e <= top - 18;
    f.c24 += e <= top - 24;
  });
  const int lo = __reduce_add_sync(0xffffffffu, f.c12 | f.c18 << 16), hi = __reduce_add_sync(0xffffffffu, f.c24);
  if (lane == 0) {
    red[warp][0] = lo;
    red[warp][1] = hi;
  }
  __syncthreads();
  f = {0, 0, 0};
#pragma unroll
  for (int w = 0; w < W; ++w) {
    f.c12 += red[w][0] & 0xffff;
    f.c18 += red[w][0] >> 16;
    f.c24 += red[w][1];
  }
  const bool dense = low > 0 && top >= bias - range && top <= bias + range && f.in(N);
  if (threadIdx.x == 0) {
    if (!dense) {
      atomicExch(a.sparse + v, 1);
    } else {
      RotDensity* d = a.density + v;
      const int spread = max(atomicMax(&d->top, top), top) + max(atomicMax(&d->bottom, kRotBottom - top), kRotBottom - top);
      if (spread > kRotBottom + 4) atomicExch(a.sparse + v, 1);
      atomicAdd(&d->c12, f.c12);
      atomicAdd(&d->c18, f.c18);
      atomicAdd(&d->c24, f.c24);
      __threadfence();
      if (atomicAdd(&d->arrived, 1u) == (unsigned)(tiles - 1)) {
        __threadfence();
        const FewBelow all = {atomicAdd(&d->c12, 0), atomicAdd(&d->c18, 0), atomicAdd(&d->c24, 0)};
        if (!all.in(a.dim)) atomicExch(a.sparse + v, 1);
      }
    }
  }
  return dense;
}

// every vector of the launch has been found not to be dense
__device__ __forceinline__ bool all_sparse(const RotArgs& a) {
  if (!a.sparse) return false;
  bool dense = false;
  for (int v = threadIdx.x; v < a.nvec; v += blockDim.x) dense = dense || !a.sparse[a.vec0 + v];
  return !__syncthreads_or(dense);
}

template <typename real, int T, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) rot_forward_kernel(const __grid_constant__ RotArgs a) {
  using v2 = typename Cx<real>::v2;
  using Gr = Groups<T>;
  constexpr int SETS = (1 << T) / (16 * NT), LO0 = T - 4, GL = Gr::N - 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  v2* buf = reinterpret_cast<v2*>(smem_raw);
  __shared__ v2 ph[kRotMaxK * (kRotMaxN + 1)];
  const int nH = a.n - T, tiles = 1 << nH;
  const int tile = blockIdx.x & (tiles - 1), v = a.vec0 + (int)(blockIdx.x >> nH);
  const size_t off = (size_t)v * a.dim + ((size_t)tile << T);
  stage_phases<real>(ph, a);
  v2* x = reinterpret_cast<v2*>(a.x) + off;
  v2 q[SETS][16];
  double nrm[1] = {0.0};
  if (a.update) {  // q_j = w' - alpha_{j-1} sigma_{j-1} q_{j-1}, |q_j|^2
    const v2* y = reinterpret_cast<const v2*>(a.y) + off;
    const size_t e = (size_t)(a.j - 1) * a.sc.ss + v;
    const real coef = (real)(a.sc.alpha[e] * a.sc.sigma[e]);
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      const int i0 = threadIdx.x + s * NT;
      v2 yv[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) q[s][r] = x[i0 + (r << LO0)];
#pragma unroll
      for (int r = 0; r < 16; ++r) yv[r] = __ldg(y + i0 + (r << LO0));
      real sum = 0;
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        q[s][r] = axpy2(-coef, yv[r], q[s][r]);
        sum += q[s][r].x * q[s][r].x + q[s][r].y * q[s][r].y;
        x[i0 + (r << LO0)] = q[s][r];
      }
      nrm[0] += (double)sum;
    }
  } else {
#pragma unroll
    for (int s = 0; s < SETS; ++s)
#pragma unroll
      for (int r = 0; r < 16; ++r) q[s][r] = x[threadIdx.x + s * NT + (r << LO0)];
    if (a.density && !vector_density<real, NT, SETS>(a, v, tiles, q)) return;
  }
  __syncthreads();
  const real t = (real)a.t;
  for (int k = 0; k < a.K; ++k) {
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      const int i0 = threadIdx.x + s * NT;
      v2 w[16];
      if (k > 0) {  // (direction 0 has azimuth 0)
        const int pc = __popc(i0) + __popc(tile);
        v2 f[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) f[m] = ph[k * (kRotMaxN + 1) + pc + m];
#pragma unroll
        for (int r = 0; r < 16; ++r) w[r] = cmul(f[__builtin_popcount(r)], q[s][r]);
      } else {
#pragma unroll
        for (int r = 0; r < 16; ++r) w[r] = q[s][r];
      }
      gates(w, t, 15);
      smem_st<LO0>(buf, group_base<LO0>(i0), w);
    }
    __syncthreads();
    if constexpr (Gr::N >= 3) mid_group<real, T, NT, SETS, 1>(buf, t, 15);
    if constexpr (Gr::N >= 4) mid_group<real, T, NT, SETS, 2>(buf, t, 15);
    v2* W = reinterpret_cast<v2*>(a.W) + ((size_t)(v - a.vecW) * a.K + k) * a.dim + ((size_t)tile << a.b);
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      const int i0 = threadIdx.x + s * NT;
      v2 w[16];
      smem_ld<0>(buf, group_base<0>(i0), w);
      gates(w, t, Gr::mask(GL));
      v2* p = W + w_place(i0, a.b, nH);
#pragma unroll
      for (int r = 0; r < 16; ++r) p[w_place(r << LO0, a.b, nH)] = w[r];
    }
    if (k + 1 < a.K) __syncthreads();
  }
  if (a.update) {
    if (vector_total<NT, 1>(nrm, a.partials + (size_t)v * tiles * 3, tile, tiles, a.counters + v))
      finalize_beta(a.sc, a.j - 1, v, a.M, a.tol, nrm[0]);
  }
}

// Tiles of 2^TB values: 2^nH rows (the high bits) of 2^c columns, c = TB - nH <= b;
// tile element (h, col) has tile index h << c | col.
// NG: groups that hold transformed bits (the last one is transformed, multiplied
// by D and transformed back in registers).
template <typename real, int TB, int NT, int MINB, int NG>
__global__ void __launch_bounds__(NT, MINB) rot_middle_kernel(const __grid_constant__ RotArgs a) {
  using v2 = typename Cx<real>::v2;
  using Gr = Groups<TB>;
  constexpr int SETS = (1 << TB) / (16 * NT), LOC = Gr::lo(NG - 1), LO0 = TB - 4;
  if (all_sparse(a)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  v2* buf = reinterpret_cast<v2*>(smem_raw);
  const int T = a.T, nH = a.n - T, c = TB - nH;
  const int cmask = (1 << c) - 1;
  const int ncb = 1 << (T - c);  // 2^T columns in blocks of 2^c
  const int cb = blockIdx.x & (ncb - 1);
  const int rest = (int)(blockIdx.x >> (T - c));
  const int k = rest % a.K, vg = rest / a.K;
  auto at = [&](int i) { return ((unsigned)(i >> c) << a.b) + (unsigned)(i & cmask); };  // offset of tile index i
  // offset of value r of group 0: with two or more groups all its bits are high ones
  const unsigned stride0 = 1u << (LO0 - (NG > 1 ? c : 0) + a.b);
  auto at0 = [&](int r) { return NG > 1 ? r * stride0 : at(r << LO0); };
  const size_t first = (size_t)k * a.dim + w_place((unsigned)cb << c, a.b, nH);
  auto mask_of = [&](int g) {  // the transformed bits (>= c) of group g
    const int l = Gr::lo(g);
    return (c > l ? (15 << (c - l)) : 15) & Gr::mask(g);
  };
  const real t = (real)a.t;
  const real* D = reinterpret_cast<const real*>(a.D) + first;
  const int v1 = min(a.nvec, (vg + 1) * a.vpb);
  for (int v = vg * a.vpb; v < v1; ++v) {
    if (a.sparse && a.sparse[a.vec0 + v]) continue;
    v2* W = reinterpret_cast<v2*>(a.W) + (size_t)(a.vec0 - a.vecW + v) * a.K * a.dim + first;
    // gates of the last group, D (after the first vector from L1) and the inverse gates
    auto centre = [&](v2(&w)[16], int b) {
      const real* d = D + at(b);
      const int m = mask_of(NG - 1);
      gates(w, t, m);
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const real dv = __ldg(d + at(r << LOC));
        w[r].x *= dv;
        w[r].y *= dv;
      }
      gates(w, -t, m);
    };
    if constexpr (NG > 1) {
#pragma unroll
      for (int s = 0; s < SETS; ++s) {
        const int i0 = threadIdx.x + s * NT;
        const v2* p = W + at(i0);
        v2 w[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) w[r] = p[at0(r)];
        gates(w, t, 15);
        smem_st<LO0>(buf, i0, w);
      }
      __syncthreads();
      if constexpr (NG > 2) mid_group<real, TB, NT, SETS, 1>(buf, t, 15);
      if constexpr (NG > 3) mid_group<real, TB, NT, SETS, 2>(buf, t, 15);
#pragma unroll
      for (int s = 0; s < SETS; ++s) {
        const int b = group_base<LOC>(threadIdx.x + s * NT);
        v2 w[16];
        smem_ld<LOC>(buf, b, w);
        centre(w, b);
        smem_st<LOC>(buf, b, w);
      }
      __syncthreads();
      if constexpr (NG > 3) mid_group<real, TB, NT, SETS, 2>(buf, -t, 15);
      if constexpr (NG > 2) mid_group<real, TB, NT, SETS, 1>(buf, -t, 15);
#pragma unroll
      for (int s = 0; s < SETS; ++s) {
        const int i0 = threadIdx.x + s * NT;
        v2* p = W + at(i0);
        v2 w[16];
        smem_ld<LO0>(buf, i0, w);
        gates(w, -t, 15);
#pragma unroll
        for (int r = 0; r < 16; ++r) p[at0(r)] = w[r];
      }
      // (the next vector's first group writes the places this thread has just read)
    } else {
#pragma unroll
      for (int s = 0; s < SETS; ++s) {
        const int i0 = threadIdx.x + s * NT;
        v2* p = W + at(i0);
        v2 w[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) w[r] = p[at0(r)];
        centre(w, i0);
#pragma unroll
        for (int r = 0; r < 16; ++r) p[at0(r)] = w[r];
      }
    }
  }
}

// The same for the large tile (NG >= 3): one CTA an SM takes tiles one after another and loads the next into
// registers while this one is exchanged: the large tile alone fills an SM's shared
// memory, and without it loads, exchanges and stores took turns (5.3 -> 4.6 ms for
// 2^26 x 4 complex64 values).
template <typename real, int TB, int NT, int NG>
__global__ void __launch_bounds__(NT, 1) rot_middle_ahead_kernel(const __grid_constant__ RotArgs a) {
  using v2 = typename Cx<real>::v2;
  using Gr = Groups<TB>;
  constexpr int SETS = (1 << TB) / (16 * NT), LOC = Gr::lo(NG - 1), LO0 = TB - 4;
  if (all_sparse(a)) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  v2* buf = reinterpret_cast<v2*>(smem_raw);
  const int T = a.T, nH = a.n - T, c = TB - nH;
  const int cmask = (1 << c) - 1;
  const int ncb = 1 << (T - c);  // 2^T columns in blocks of 2^c
  auto at = [&](int i) { return ((unsigned)(i >> c) << a.b) + (unsigned)(i & cmask); };  // offset of tile index i
  // offset of value r of group 0 (all its bits are high ones)
  const unsigned stride0 = 1u << (LO0 - c + a.b);
  auto at0 = [&](int r) { return r * stride0; };
  auto mask_of = [&](int g) {  // the transformed bits (>= c) of group g
    const int l = Gr::lo(g);
    return (c > l ? (15 << (c - l)) : 15) & Gr::mask(g);
  };
  const real t = (real)a.t;
  // column block q of all directions and vector groups; its first value and its vectors
  const int blocks = ncb * a.K * ((a.nvec + a.vpb - 1) / a.vpb);
  auto first_of = [&](int q) { return (size_t)((q >> (T - c)) % a.K) * a.dim + w_place((unsigned)(q & (ncb - 1)) << c, a.b, nH); };
  auto vec_of = [&](int q) { return ((q >> (T - c)) / a.K) * a.vpb; };
  auto tile_of = [&](int q, int v) { return reinterpret_cast<v2*>(a.W) + (size_t)(a.vec0 - a.vecW + v) * a.K * a.dim + first_of(q); };
  v2 nx[SETS][16];
  {
    const v2* W = tile_of(blockIdx.x, vec_of(blockIdx.x));
#pragma unroll
    for (int s = 0; s < SETS; ++s)
#pragma unroll
      for (int r = 0; r < 16; ++r) nx[s][r] = W[at(threadIdx.x + s * NT) + at0(r)];
  }
  for (int q = blockIdx.x; q < blocks; q += (int)gridDim.x) {
    const real* D = reinterpret_cast<const real*>(a.D) + first_of(q);
    const int v0 = vec_of(q), v1 = min(a.nvec, v0 + a.vpb);
    for (int v = v0; v < v1; ++v) {
      v2* W = tile_of(q, v);
      // gates of the last group, D (after the first vector from L1) and the inverse gates
      auto centre = [&](v2(&w)[16], int b) {
        const real* d = D + at(b);
        const int m = mask_of(NG - 1);
        gates(w, t, m);
#pragma unroll
        for (int r = 0; r < 16; ++r) {
          const real dv = __ldg(d + at(r << LOC));
          w[r].x *= dv;
          w[r].y *= dv;
        }
        gates(w, -t, m);
      };
#pragma unroll
      for (int s = 0; s < SETS; ++s) {
        const int i0 = threadIdx.x + s * NT;
        v2 w[16];
#pragma unroll
        for (int r = 0; r < 16; ++r) w[r] = nx[s][r];
        gates(w, t, 15);
        smem_st<LO0>(buf, i0, w);
      }
      {
        const int qn = v + 1 < v1 ? q : q + (int)gridDim.x;
        if (qn < blocks) {
          const v2* N = tile_of(qn, v + 1 < v1 ? v + 1 : vec_of(qn));
#pragma unroll
          for (int s = 0; s < SETS; ++s)
#pragma unroll
            for (int r = 0; r < 16; ++r) nx[s][r] = N[at(threadIdx.x + s * NT) + at0(r)];
        }
      }
      __syncthreads();
      if constexpr (NG > 2) mid_group<real, TB, NT, SETS, 1>(buf, t, 15);
      if constexpr (NG > 3) mid_group<real, TB, NT, SETS, 2>(buf, t, 15);
#pragma unroll
      for (int s = 0; s < SETS; ++s) {
        const int b = group_base<LOC>(threadIdx.x + s * NT);
        v2 w[16];
        smem_ld<LOC>(buf, b, w);
        centre(w, b);
        smem_st<LOC>(buf, b, w);
      }
      __syncthreads();
      if constexpr (NG > 3) mid_group<real, TB, NT, SETS, 2>(buf, -t, 15);
      if constexpr (NG > 2) mid_group<real, TB, NT, SETS, 1>(buf, -t, 15);
#pragma unroll
      for (int s = 0; s < SETS; ++s) {
        const int i0 = threadIdx.x + s * NT;
        v2* p = W + at(i0);
        v2 w[16];
        smem_ld<LO0>(buf, i0, w);
        gates(w, -t, 15);
#pragma unroll
        for (int r = 0; r < 16; ++r) p[at0(r)] = w[r];
      }
      // (the next tile's first group writes the places this thread has just read)
    }
  }
}

template <typename real, int T, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) rot_backward_kernel(const __grid_constant__ RotArgs a) {
  using v2 = typename Cx<real>::v2;
  using Gr = Groups<T>;
  constexpr int SETS = (1 << T) / (16 * NT), LO0 = T - 4, GL = Gr::N - 1;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  v2* buf = reinterpret_cast<v2*>(smem_raw);
  __shared__ v2 ph[kRotMaxK * (kRotMaxN + 1)];
  const int nH = a.n - T, tiles = 1 << nH;
  const int tile = blockIdx.x & (tiles - 1), v = a.vec0 + (int)(blockIdx.x >> nH);
  if (a.sparse && a.sparse[v]) return;
  const size_t off = (size_t)v * a.dim + ((size_t)tile << T);
  stage_phases<real>(ph, a);
  const real t = (real)a.t;
  v2 acc[SETS][16];
  for (int k = 0; k < a.K; ++k) {
    const v2* W = reinterpret_cast<const v2*>(a.W) + ((size_t)(v - a.vecW) * a.K + k) * a.dim + ((size_t)tile << a.b);
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      const int i0 = threadIdx.x + s * NT;
      const v2* p = W + w_place(i0, a.b, nH);
      v2 w[16];
#pragma unroll
      for (int r = 0; r < 16; ++r) w[r] = p[w_place(r << LO0, a.b, nH)];
      gates(w, -t, Gr::mask(GL));
      if (s == 0) __syncthreads();  // the previous direction's last group has been read
      smem_st<0>(buf, group_base<0>(i0), w);
    }
    __syncthreads();
    if constexpr (Gr::N >= 4) mid_group<real, T, NT, SETS, 2>(buf, -t, 15);
    if constexpr (Gr::N >= 3) mid_group<real, T, NT, SETS, 1>(buf, -t, 15);
#pragma unroll
    for (int s = 0; s < SETS; ++s) {
      const int i0 = threadIdx.x + s * NT;
      v2 w[16];
      smem_ld<LO0>(buf, i0, w);
      gates(w, -t, 15);
      if (k == 0) {
#pragma unroll
        for (int r = 0; r < 16; ++r) acc[s][r] = w[r];
      } else {
        const int pc = __popc(i0) + __popc(tile);
        v2 f[5];
#pragma unroll
        for (int m = 0; m < 5; ++m) f[m] = ph[k * (kRotMaxN + 1) + pc + m];
#pragma unroll
        for (int r = 0; r < 16; ++r) {  // acc += conj(f) w
          const v2 g = f[__builtin_popcount(r)];
          acc[s][r].x = fma(g.x, w[r].x, fma(g.y, w[r].y, acc[s][r].x));
          acc[s][r].y = fma(g.x, w[r].y, fma(-g.y, w[r].x, acc[s][r].y));
        }
      }
    }
  }
  const v2* x = reinterpret_cast<const v2*>(a.x) + off;
  v2* y = reinterpret_cast<v2*>(a.y) + off;
  const real* D0 = reinterpret_cast<const real*>(a.D0) + ((size_t)tile << T);
  if (!a.lanczos) {  // y = H x
#pragma unroll
    for (int s = 0; s < SETS; ++s)
#pragma unroll
      for (int r = 0; r < 16; ++r) {
        const int i = threadIdx.x + s * NT + (r << LO0);
        y[i] = axpy2(__ldg(D0 + i), __ldg(x + i), acc[s][r]);
      }
    return;
  }
  const v2* u = reinterpret_cast<const v2*>(a.u) + off;
  const size_t e = (size_t)a.j * a.sc.ss + v;
  const double sgd = a.sc.sigma[e];
  const real sg = (real)sgd;
  const real bsp = a.j == 0 ? (real)0 : (real)(a.sc.beta[e - a.sc.ss] * a.sc.sigma[e - a.sc.ss]);
  double p[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int s = 0; s < SETS; ++s) {
    real pw = 0, pr = 0, pi = 0;
#pragma unroll
    for (int r = 0; r < 16; ++r) {
      const int i = threadIdx.x + s * NT + (r << LO0);
      const v2 xv = __ldg(x + i), uv = __ldg(u + i);
      const v2 hv = axpy2(__ldg(D0 + i), xv, acc[s][r]);
      v2 w;
      if (a.j == 0) {
        w.x = sg * hv.x;
        w.y = sg * hv.y;
      } else {
        const v2 qp = y[i];
        w.x = sg * hv.x - bsp * qp.x;
        w.y = sg * hv.y - bsp * qp.y;
      }
      y[i] = w;
      pw += xv.x * w.x + xv.y * w.y;
      pr += xv.x * uv.x + xv.y * uv.y;
      pi += xv.x * uv.y - xv.y * uv.x;
    }
    p[0] += (double)pw;
    p[1] += (double)pr;
    p[2] += (double)pi;
  }
  if (vector_total<NT, 3>(p, a.partials + (size_t)v * tiles * 3, tile, tiles, a.counters + v)) {
    a.sc.alpha[e] = sgd * p[0];
    a.sc.p[2 * e] = sgd * p[1];
    a.sc.p[2 * e + 1] = sgd * p[2];
  }
}

// Diagonal table of one direction, in the natural order or (f.T > 0) in W's:
//   scale (c0 + sum_i m_i (h_i + sum_{j > i} a_ij m_j)),  m_i = +-1/2 by bit i,
// in FP64, one CTA per 4096 entries: the terms of the bits above 12 once per
// CTA, a thread's 16 entries along bits 0..3.
template <typename real>
__global__ void __launch_bounds__(256) rot_table_kernel(const __grid_constant__ RotForm f, real* out) {
  __shared__ double F[12], E;
  const unsigned long long top = blockIdx.x;
  auto m = [](unsigned long long b, int i) { return ((b >> i) & 1ull) ? 0.5 : -0.5; };
  if (threadIdx.x < 12) {
    double s = f.h[threadIdx.x];
    for (int j = 12; j < f.n; ++j) s += f.a[tri(threadIdx.x, j)] * m(top, j - 12);
    F[threadIdx.x] = s;
  } else if (threadIdx.x == 32) {
    double e = f.c0;
    for (int i = 12; i < f.n; ++i) {
      double s = f.h[i];
      for (int j = i + 1; j < f.n; ++j) s += f.a[tri(i, j)] * m(top, j - 12);
      e += m(top, i - 12) * s;
    }
    E = e;
  }
  __syncthreads();
  const int mid = threadIdx.x << 4;
  double e = E, g[4];
  for (int i = 4; i < 12; ++i) {
    double s = F[i];
    for (int j = i + 1; j < 12; ++j) s += f.a[tri(i, j)] * m(mid, j);
    e += m(mid, i) * s;
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    g[i] = F[i];
    for (int j = 4; j < 12; ++j) g[i] += f.a[tri(i, j)] * m(mid, j);
  }
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    double d = e;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      double s = g[i];
#pragma unroll
      for (int j = i + 1; j < 4; ++j) s += f.a[tri(i, j)] * ((r >> j) & 1 ? 0.5 : -0.5);
      d += ((r >> i) & 1 ? 0.5 : -0.5) * s;
    }
    unsigned long long at = (top << 12) | (unsigned)mid | (unsigned)r;
    if (f.T > 0) {
      const unsigned low = (unsigned)at & ((1u << f.T) - 1u);
      at = w_place(((low & 15u) << (f.T - 4)) | (low >> 4), f.b, f.n - f.T) + ((at >> f.T) << f.b);
    }
    out[at] = (real)(f.scale * d);
  }
}

// e^{-i phi_k (n - m)} for m = 0..n up spins
template <typename real>
__global__ void rot_phase_kernel(int n, int K, RotAzimuths d, real* out) {
  const int k = threadIdx.x / (kRotMaxN + 1), m = threadIdx.x % (kRotMaxN + 1);
  if (k >= K || m > n) return;
  double sn, cs;
  sincospi((double)((n - m) * d.num[k] % (2 * d.den)) / (double)d.den, &sn, &cs);
  out[2 * threadIdx.x] = (real)cs;
  out[2 * threadIdx.x + 1] = (real)-sn;
}

template <typename real, int T>
constexpr size_t tile_smem() {
  return sizeof(typename Cx<real>::v2) * (size_t)pad(1 << T);
}

// the forward and backward passes over tiles of 2^T values
template <typename real, int T, int NT, int MINB>
int launch_outer(const RotArgs& a, int pass, cudaStream_t st) {
  const unsigned grid = (unsigned)a.nvec << (a.n - T);
  if (pass == 0) rot_forward_kernel<real, T, NT, MINB><<<grid, NT, tile_smem<real, T>(), st>>>(a);
  else rot_backward_kernel<real, T, NT, MINB><<<grid, NT, tile_smem<real, T>(), st>>>(a);
  return (int)cudaGetLastError();
}

// groups that hold high bits of the middle pass's tile
template <int TB>
int middle_groups(const RotArgs& a) {
  const int c = TB - (a.n - a.T);
  int ng = 1;
  while (ng < Groups<TB>::N && Groups<TB>::lo(ng - 1) > c) ++ng;
  return ng;
}

// the middle pass over tiles of 2^TB values
template <typename real, int TB, int NT, int MINB>
int launch_middle(const RotArgs& a, cudaStream_t st) {
  const int ng = middle_groups<TB>(a);
  const size_t smem = tile_smem<real, TB>();
  const unsigned grid = (unsigned)(((a.nvec + a.vpb - 1) / a.vpb) * a.K) << (a.n - TB);
  if (ng == 1) rot_middle_kernel<real, TB, NT, MINB, 1><<<grid, NT, 0, st>>>(a);
  else if (ng == 2) rot_middle_kernel<real, TB, NT, MINB, 2><<<grid, NT, smem, st>>>(a);
  else if (ng == 3) rot_middle_kernel<real, TB, NT, MINB, 3><<<grid, NT, smem, st>>>(a);
  else if constexpr (Groups<TB>::N >= 4) rot_middle_kernel<real, TB, NT, MINB, 4><<<grid, NT, smem, st>>>(a);
  else return (int)cudaErrorInvalidValue;
  return (int)cudaGetLastError();
}

// the same, one CTA an SM and the next tile loaded ahead
template <typename real, int TB, int NT>
int launch_middle_ahead(const RotArgs& a, cudaStream_t st) {
  const int ng = middle_groups<TB>(a);
  const size_t smem = tile_smem<real, TB>();
  const unsigned grid = std::min((unsigned)(((a.nvec + a.vpb - 1) / a.vpb) * a.K) << (a.n - TB),
                                 (unsigned)std::max(1, device_sm_count()));
  if (ng == 3) rot_middle_ahead_kernel<real, TB, NT, 3><<<grid, NT, smem, st>>>(a);
  else if (ng == 4) rot_middle_ahead_kernel<real, TB, NT, 4><<<grid, NT, smem, st>>>(a);
  else return (int)cudaErrorInvalidValue;
  return (int)cudaGetLastError();
}

int allow(const void* k, size_t smem) {
  return (int)cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}
template <typename real, int T, int NT, int MINB>
int prepare_outer() {
  const int e = allow((const void*)rot_forward_kernel<real, T, NT, MINB>, tile_smem<real, T>());
  return e ? e : allow((const void*)rot_backward_kernel<real, T, NT, MINB>, tile_smem<real, T>());
}
template <typename real, int TB, int NT, int MINB>
int prepare_middle() {
  int e = allow((const void*)rot_middle_kernel<real, TB, NT, MINB, 2>, tile_smem<real, TB>());
  if (!e) e = allow((const void*)rot_middle_kernel<real, TB, NT, MINB, 3>, tile_smem<real, TB>());
  if constexpr (Groups<TB>::N >= 4)
    if (!e) e = allow((const void*)rot_middle_kernel<real, TB, NT, MINB, 4>, tile_smem<real, TB>());
  return e;
}
template <typename real, int TB, int NT>
int prepare_middle_ahead() {
  const int e = allow((const void*)rot_middle_ahead_kernel<real, TB, NT, 3>, tile_smem<real, TB>());
  return e ? e : allow((const void*)rot_middle_ahead_kernel<real, TB, NT, 4>, tile_smem<real, TB>());
}

// The middle pass's tile for nH high bits: the small one, of which an SM runs
// four (three in complex128), while its rows are at least 32 bytes; else the
// large one.  (2^13-value tiles with 16-byte rows, three an SM: 9.8 ms instead of
// 6.5 for 2^26 x 4 values; L2 moves whole 32-byte sectors.)
int middle_bits(int nH, int c64) {
  if (c64) return nH <= 10 ? 12 : 14;
  return nH <= 10 ? 11 : (nH <= 12 ? 12 : 13);
}

}  // namespace

// b of W's order for n sites (see the top of the file)
int rot_run_bits(int n, int c64) {
  const int T = rot_tile_bits(n, c64), nH = n - T;
  return nH <= 10 ? T : std::max(middle_bits(nH, c64) - nH, c64 ? 4 : 3);
}

int launch_rot(const RotArgs& a, int pass, int c64, void* stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (a.T != rot_tile_bits(a.n, c64) || a.T == 0 || a.K < 1 || a.K > kRotMaxK || a.vpb < 1) return (int)cudaErrorInvalidValue;
  if (pass != 1) {
    if (c64) return a.T == 12 ? launch_outer<float, 12, 256, 3>(a, pass, st) : launch_outer<float, 14, 512, 1>(a, pass, st);
    return a.T == 11 ? launch_outer<double, 11, 128, 3>(a, pass, st) : launch_outer<double, 13, 256, 1>(a, pass, st);
  }
  switch (middle_bits(a.n - a.T, c64)) {
    case 11: return launch_middle<double, 11, 128, 3>(a, st);
    case 12: return c64 ? launch_middle<float, 12, 256, 4>(a, st) : launch_middle<double, 12, 128, 3>(a, st);
    case 13: return launch_middle<double, 13, 256, 1>(a, st);
    default: return launch_middle_ahead<float, 14, 512>(a, st);
  }
}

int prepare_rot(int n, int c64) {
  int e;
  const int T = rot_tile_bits(n, c64);
  if (c64) e = T == 12 ? prepare_outer<float, 12, 256, 3>() : prepare_outer<float, 14, 512, 1>();
  else e = T == 11 ? prepare_outer<double, 11, 128, 3>() : prepare_outer<double, 13, 256, 1>();
  if (e) return e;
  switch (middle_bits(n - T, c64)) {
    case 11: return prepare_middle<double, 11, 128, 3>();
    case 12: return c64 ? prepare_middle<float, 12, 256, 4>() : prepare_middle<double, 12, 128, 3>();
    case 13: return prepare_middle<double, 13, 256, 1>();
    default: return prepare_middle_ahead<float, 14, 512>();
  }
}

int launch_rot_table(const RotForm& f, void* out, int c64, void* stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (f.n < 12 || f.n > kRotMaxN) return (int)cudaErrorInvalidValue;
  const unsigned grid = 1u << (f.n - 12);
  if (c64) rot_table_kernel<float><<<grid, 256, 0, st>>>(f, reinterpret_cast<float*>(out));
  else rot_table_kernel<double><<<grid, 256, 0, st>>>(f, reinterpret_cast<double*>(out));
  return (int)cudaGetLastError();
}

int launch_rot_phases(int n, const RotDirs& d, void* out, int c64, void* stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int threads = kRotMaxK * (kRotMaxN + 1);
  if (c64) rot_phase_kernel<float><<<1, threads, 0, st>>>(n, d.K, d.az, reinterpret_cast<float*>(out));
  else rot_phase_kernel<double><<<1, threads, 0, st>>>(n, d.K, d.az, reinterpret_cast<double*>(out));
  return (int)cudaGetLastError();
}

// Low tile bits for n sites (0: none, the gather runs): the small tile, of which
// an SM runs three, while a middle tile has room for the other bits; then the
// large one, one CTA an SM.
int rot_tile_bits(int n, int c64) {
  if (n < 13) return 0;
  if (c64) return n <= 24 ? 12 : (n <= 28 ? 14 : 0);
  return n <= 23 ? 11 : (n <= 26 ? 13 : 0);
}

// Row k: the a_k of A = a_0 z z^T + sum_k a_k u_k u_k^T as combinations of A's
// elements xx, yy, zz, xy, xz, yz: the inverse of the 6 x 6 matrix whose columns
// are those of the projectors (Gauss-Jordan; its condition number is 2.2).
static void six_lines(const double (*u)[3], double (&inv)[6][6]) {
  double m[6][12] = {};
  for (int c = 0; c < 6; ++c) {
    const double z[3] = {0.0, 0.0, 1.0}, *w = c == 0 ? z : u[c - 1];
    const double e[6] = {w[0] * w[0], w[1] * w[1], w[2] * w[2], w[0] * w[1], w[0] * w[2], w[1] * w[2]};
    for (int r = 0; r < 6; ++r) m[r][c] = e[r];
    m[c][6 + c] = 1.0;
  }
  for (int c = 0; c < 6; ++c) {
    int p = c;
    for (int r = c + 1; r < 6; ++r)
      if (std::fabs(m[r][c]) > std::fabs(m[p][c])) p = r;
    for (int k = 0; k < 12; ++k) std::swap(m[c][k], m[p][k]);
    const double d = 1.0 / m[c][c];
    for (int k = 0; k < 12; ++k) m[c][k] *= d;
    for (int r = 0; r < 6; ++r) {
      const double f = r == c ? 0.0 : m[r][c];
      for (int k = 0; k < 12; ++k) m[r][k] -= f * m[c][k];
    }
  }
  for (int r = 0; r < 6; ++r)
    for (int k = 0; k < 6; ++k) inv[r][k] = m[r][6 + k];
}

// The directions and diagonal forms of a spin-1/2 system (see the top of the
// file); false when it has none (a pair tensor that is not symmetric) or no
// pair couplings at all.
bool rot_directions(const HostSystem& hs, RotDirs& d) {
  const int n = hs.n;
  if (!hs.all_half || !hs.real_pm || n > kRotMaxN) return false;
  const TabLayout& L = hs.lay;
  const double* t = hs.tab.data();
  bool planar = true, diagonal = true, coupled = false;
  for (int i = 0; i < n; ++i)
    for (int j = i + 1; j < n; ++j) {
      const int ij = i * n + j, ji = j * n + i;
      for (int c = 0; c < 2; ++c) {
        if (t[L.off_rho + 2 * ij + c] != t[L.off_rho + 2 * ji + c]) return false;
        planar = planar && t[L.off_rho + 2 * ij + c] == 0.0;
      }
      diagonal = diagonal && t[L.off_pp + 2 * ij + 1] == 0.0;
      coupled = coupled || t[L.off_pm + 2 * ij] != 0.0 || t[L.off_pp + 2 * ij] != 0.0 || t[L.off_pp + 2 * ij + 1] != 0.0 ||
                t[L.off_rho + 2 * ij] != 0.0 || t[L.off_rho + 2 * ij + 1] != 0.0;
    }
  if (!coupled) return false;
  const double pi = 3.14159265358979323846;
  // azimuths phi_k = pi num / den; the polar angle's cosine
  double ct = 0.0;
  if (planar && diagonal) {
    d.K = 2;
    d.az.num[0] = 0;
    d.az.num[1] = 1;
    d.az.den = 2;
  } else if (planar) {
    d.K = 3;
    for (int k = 0; k < 3; ++k) d.az.num[k] = k;
    d.az.den = 3;
  } else {
    d.K = 5;
    for (int k = 0; k < 5; ++k) d.az.num[k] = 2 * k;
    d.az.den = 5;
    ct = 1.0 / std::sqrt(5.0);
  }
  // The gates multiply by t in the product's precision and the tables undo
  // (1 + t^2)^n: t has to be one number in both.  So the polar angle is the one
  // whose t is an FP32 value (1 already is; 0.618... moves by 2.7e-8, and the six
  // lines are then no longer exactly an icosahedron's).  With t rounded in the gates
  // alone every product in complex64 was off by n x 1.5e-8 of itself (3e-7 at 20 sites).
  d.t = (double)(float)(std::sqrt(1.0 - ct * ct) / (1.0 + ct));
  ct = (1.0 - d.t * d.t) / (1.0 + d.t * d.t);
  const double st = 2.0 * d.t / (1.0 + d.t * d.t);
  const int K = d.K;
  double u[kRotMaxK][3];
  for (int k = 0; k < K; ++k) {
    u[k][0] = st * std::cos(pi * d.az.num[k] / d.az.den);
    u[k][1] = st * std::sin(pi * d.az.num[k] / d.az.den);
    u[k][2] = ct;
  }
  if (K == 2) u[1][0] = 0.0;  // (cos(pi / 2))
  const double inv_plane = 1.0 / (2.5 * st * st), inv_z = 1.0 / (1.0 + 5.0 * ct * ct);  // (K = 5) of sum u u^T over the six lines
  double six[6][6] = {};  // (K = 5) a_k of each element of A
  if (K == 5) six_lines(u, six);
  for (int k = 0; k <= K; ++k) {
    RotForm& f = d.form[k];
    f.n = n;
    f.c0 = 0.0;
    f.scale = k == 0 ? 1.0 : std::pow(1.0 + d.t * d.t, -n);
  }
  for (int i = 0; i < n; ++i) {
    const double h[3] = {2.0 * t[L.off_hp + 2 * i], -2.0 * t[L.off_hp + 2 * i + 1], t[L.off_hz + i]};
    d.form[0].c0 += t[L.off_iondiag + i * L.qmax];  // (s.e)^2 = 1/4: the same for both digits
    // h = sum_k (u_k . S^-1 h) u_k, S = sum_k u_k u_k^T over the set (with z for K = 5): diagonal
    for (int k = 0; k < K; ++k) {
      const double hp = h[0] * u[k][0] + h[1] * u[k][1];
      d.form[k + 1].h[i] = K == 2 ? hp : (K == 3 ? 2.0 / 3.0 * hp : inv_plane * hp + inv_z * h[2] * u[k][2]);
    }
    d.form[0].h[i] = K == 5 ? inv_z * h[2] : h[2];
  }
  for (int i = 0; i < n; ++i)
    for (int j = i + 1; j < n; ++j) {
      const int ij = i * n + j, q = (j * (j - 1)) / 2 + i;
      const double pm = t[L.off_pm + 2 * ij], pp = t[L.off_pp + 2 * ij];
      const double xx = 2.0 * (pm + pp), yy = 2.0 * (pm - pp), zz = t[L.off_zz + ij];
      const double xy = -2.0 * t[L.off_pp + 2 * ij + 1];
      const double xz = 2.0 * t[L.off_rho + 2 * ij], yz = -2.0 * t[L.off_rho + 2 * ij + 1];
      // A = sum_k a_k u_k u_k^T.  In the plane, projectors of a tight frame:
      // a_k = alpha (u_k.A.u_k) + gamma tr A solves it.
      if (K == 2) {
        d.form[0].a[q] = zz;
        d.form[1].a[q] = xx;
        d.form[2].a[q] = yy;
      } else if (K == 3) {
        d.form[0].a[q] = zz;
        // in the plane: sum_k (u_k.A.u_k) u_k u_k^T = 3/8 (2 A + tr A 1), sum_k u_k u_k^T = 3/2 1
        for (int k = 0; k < 3; ++k) {
          const double quad = xx * u[k][0] * u[k][0] + 2.0 * xy * u[k][0] * u[k][1] + yy * u[k][1] * u[k][1];
          d.form[k + 1].a[q] = 4.0 / 3.0 * quad - (xx + yy) / 3.0;
        }
      } else {
        const double A[6] = {xx, yy, zz, xy, xz, yz};
        for (int k = 0; k < 6; ++k) {
          double a = 0.0;
          for (int r = 0; r < 6; ++r) a += six[k][r] * A[r];
          d.form[k].a[q] = a;
        }
      }
    }
  return true;
}

}  // namespace ftlm
