// y = c (u.S) x, the one-body observable of Eq. (4) of arxiv 2607.25585, for any
// spins, on vector-major ([R][dim]) and row-major ([dim][R]) blocks:
//   (u.S x)[mu] = u_z (sum_i m_i) x[mu] + a sum_i <a_i|s+|a_i-1> x[mu - s_i]
//                 + conj(a) sum_i <a_i|s-|a_i+1> x[mu + s_i],   a = (u_x - i u_y)/2.
//
// A CTA owns a tile of T = q_0 q_1 ... consecutive rows (the low sites' whole
// range) of V vectors, staged in shared memory: the low sites' neighbours are
// in the tile, and the high sites' digits are the same for all of it, so their
// neighbours are whole tiles, read in order.  A row's digits and ladder
// coefficients are formed once for V vectors, and the two real-weighted sums are
// multiplied by a and conj(a) at the end.
//
// Bound: L2 (one load per high site and direction).  Tiles of at most 48 KB keep
// four CTAs an SM (64 KB: 19.7 -> 23 ms for a start and this on 2^26 x 4 values).
// Before, one thread formed a row's digits by division for
// every vector and gathered all neighbours through L1: 18.4 ms for 2^26 x 4
// complex64 values of a spin-1/2 ladder, 9.6 ms for ten molecules of 9 sites
// (2.3e6 x 8 each).
#include <cuda_runtime.h>

#include <algorithm>

#include "device_common.cuh"
#include "ftlm_internal.h"

namespace ftlm {

namespace {

constexpr int kThreads = 256;
constexpr int kTileBytes = 48 * 1024;
constexpr int kMaxSmem = kTileBytes + 4 * kMaxSites * kMaxQ * 8;  // the tile and every site's coefficients

template <typename real, int V>
__global__ void __launch_bounds__(kThreads) sdir_vectors_kernel(const __grid_constant__ SdirArgs a) {
  using v2 = typename Cx<real>::v2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  real* site = reinterpret_cast<real*>(smem_raw);                   // [n][qmax][4]: up, down, m, -
  v2* tile = reinterpret_cast<v2*>(site + 4 * a.n * a.lay.qmax);    // [V][T]
  const real* t = reinterpret_cast<const real*>(a.tab);
  const int qm = a.lay.qmax, T = a.T;
  for (int k = threadIdx.x; k < a.n * qm; k += kThreads) {
    site[4 * k] = t[a.lay.off_up1 + k];
    site[4 * k + 1] = t[a.lay.off_dn1 + k];
    site[4 * k + 2] = t[a.lay.off_m + k];
  }
  const int v0 = blockIdx.y * V, nv = min(V, a.R - v0);
  const long long row0 = (long long)blockIdx.x * T;
  const v2* x = reinterpret_cast<const v2*>(a.x);
  v2* y = reinterpret_cast<v2*>(a.y);
  auto at = [&](long long mu, int v) { return (long long)(v0 + v) * a.dim + mu; };  // vector v of row mu
#pragma unroll
  for (int v = 0; v < V; ++v)
    if (v < nv)
      for (int e = threadIdx.x; e < T; e += kThreads) tile[v * T + e] = __ldg(x + at(row0 + e, v));
  __syncthreads();
  const real uz = (real)a.obs[0], aur = (real)a.obs[1], aui = (real)a.obs[2];
  // u along z (a field along z, or none): the neighbours have the factor 0 and are not read
  // (3.4 ms less for 2^26 x 4 complex64 values)
  const bool flips = aur != 0 || aui != 0;
  real c[V];
#pragma unroll
  for (int v = 0; v < V; ++v) c[v] = a.sigma && v < nv ? (real)a.sigma[v0 + v] : (real)1;
  for (int e = threadIdx.x; e < T; e += kThreads) {
    v2 up[V], dn[V];
    real msum = 0;
#pragma unroll
    for (int v = 0; v < V; ++v) up[v].x = up[v].y = dn[v].x = dn[v].y = 0;
    auto mac = [&](v2(&s)[V], real w, const v2* p, long long vstride) {
#pragma unroll
      for (int v = 0; v < V; ++v)
        if (v < nv) {
          const v2 z = p[v * vstride];
          s[v].x = fma(w, z.x, s[v].x);
          s[v].y = fma(w, z.y, s[v].y);
        }
    };
    unsigned rem = (unsigned)e;
    int stride = 1;
    for (int i = 0; i < a.n_low; ++i) {  // neighbours within the tile
      const unsigned q = (unsigned)__ldg(a.q + i), nx = rem / q;
      const int d = (int)(rem - nx * q);
      rem = nx;
      const real* s = site + 4 * (i * qm + d);
      msum += s[2];
      if (flips && d > 0) mac(up, s[0], tile + e - stride, T);
      if (flips && d + 1 < (int)q) mac(dn, s[1], tile + e + stride, T);
      stride *= (int)q;
    }
    unsigned long long high = blockIdx.x;
    long long far = T;
    const v2* own = x + at(row0 + e, 0);
    for (int i = a.n_low; i < a.n; ++i) {  // the high sites: the same digits for the whole CTA
      const unsigned q = (unsigned)__ldg(a.q + i);
      const unsigned long long nx = (high >> 32) ? high / q : (unsigned)high / q;
      const int d = (int)(high - nx * q);
      high = nx;
      const real* s = site + 4 * (i * qm + d);
      msum += s[2];
      if (flips && d > 0) mac(up, s[0], own - far, a.dim);
      if (flips && d + 1 < (int)q) mac(dn, s[1], own + far, a.dim);
      far *= q;
    }
    const real dz = uz * msum;
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (v < nv) {
        const v2 z = tile[v * T + e];
        v2 o;  // u_z M x + a up + conj(a) down
        o.x = c[v] * fma(dz, z.x, fma(aur, up[v].x + dn[v].x, -aui * (up[v].y - dn[v].y)));
        o.y = c[v] * fma(dz, z.y, fma(aur, up[v].y + dn[v].y, aui * (up[v].x - dn[v].x)));
        y[at(row0 + e, v)] = o;
      }
  }
}

// The same where every spin is 1/2: a row's digits are its index's bits, every ladder
// coefficient is 1, and site i's one neighbour enters with a or conj(a): 0.99 -> 0.62 ms
// for 2^20 x 64 complex64 values, 5.7 -> 5.0 ms for 2^26 x 4 (there memory binds: 15 of 26
// neighbours are in other tiles, and the highest bits' are no longer in L2), of which
// 0.8 ms remain where u lies along z.
template <typename real, int V>
__global__ void __launch_bounds__(kThreads) sdir_half_kernel(const __grid_constant__ SdirArgs a) {
  using v2 = typename Cx<real>::v2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  v2* tile = reinterpret_cast<v2*>(smem_raw);  // [V][T]
  const int T = a.T, nh = a.n - a.n_low;
  const int v0 = blockIdx.y * V, nv = min(V, a.R - v0);
  const long long row0 = (long long)blockIdx.x * T;
  const v2* x = reinterpret_cast<const v2*>(a.x) + (long long)v0 * a.dim + row0;
  v2* y = reinterpret_cast<v2*>(a.y) + (long long)v0 * a.dim + row0;
  long long off[V];  // (a smaller group reads its last vector in the others' place)
#pragma unroll
  for (int v = 0; v < V; ++v) off[v] = (long long)min(v, nv - 1) * a.dim;
#pragma unroll
  for (int v = 0; v < V; ++v)
    for (int e = threadIdx.x; e < T; e += kThreads) tile[v * T + e] = __ldg(x + off[v] + e);
  __syncthreads();
  const real uz = (real)a.obs[0], aur = (real)a.obs[1], aui = (real)a.obs[2];
  const bool flips = aur != 0 || aui != 0;
  const int high_bits = __popc((unsigned)blockIdx.x);
  real c[V];
#pragma unroll
  for (int v = 0; v < V; ++v) c[v] = a.sigma && v < nv ? (real)a.sigma[v0 + v] : (real)1;
  for (int e = threadIdx.x; e < T; e += kThreads) {
    v2 sum[V], dif[V];  // the neighbours' sum, and set bits' minus clear bits'
#pragma unroll
    for (int v = 0; v < V; ++v) sum[v].x = sum[v].y = dif[v].x = dif[v].y = 0;
    auto add = [&](real sign, int v, v2 z) {
      sum[v].x += z.x;
      sum[v].y += z.y;
      dif[v].x = fma(sign, z.x, dif[v].x);
      dif[v].y = fma(sign, z.y, dif[v].y);
    };
    if (flips) {
#pragma unroll 4
      for (int i = 0; i < nh; ++i) {
        const bool set = (blockIdx.x >> i) & 1;
        const long long far = (long long)T << i;
        const v2* p = x + e + (set ? -far : far);
#pragma unroll
        for (int v = 0; v < V; ++v) add(set ? (real)1 : (real)-1, v, __ldg(p + off[v]));
      }
#pragma unroll 4
      for (int i = 0; i < a.n_low; ++i) {
        const int at = e ^ (1 << i);
#pragma unroll
        for (int v = 0; v < V; ++v) add((e >> i) & 1 ? (real)1 : (real)-1, v, tile[v * T + at]);
      }
    }
    const real dz = uz * ((real)(high_bits + __popc((unsigned)e)) - (real)0.5 * (real)a.n);
#pragma unroll
    for (int v = 0; v < V; ++v)
      if (v < nv) {
        const v2 z = tile[v * T + e];
        v2 o;  // u_z M x + Re(a) sum + i Im(a) dif
        o.x = c[v] * fma(dz, z.x, fma(aur, sum[v].x, -aui * dif[v].y));
        o.y = c[v] * fma(dz, z.y, fma(aur, sum[v].y, aui * dif[v].x));
        y[(long long)v * a.dim + e] = o;
      }
  }
}

// The row-major form: neighbouring lanes take neighbouring vectors of one row (W a
// lane, 16 bytes where that is aligned), so every access is a run of the row's
// vectors; with lanes along rows, 32 bytes a lane, the loads of the high sites
// touched a sector each (1.53 ms for 2^20 x 32 complex64 values, 0.65 ms so).
template <typename real, int W>
__global__ void __launch_bounds__(kThreads) sdir_rows_kernel(const __grid_constant__ SdirArgs a) {
  using v2 = typename Cx<real>::v2;
  struct __align__(sizeof(v2) * W) Pack {
    v2 z[W];
  };
  extern __shared__ __align__(16) unsigned char smem_raw[];
  real* site = reinterpret_cast<real*>(smem_raw);                   // [n][qmax][4]: up, down, m, -
  Pack* tile = reinterpret_cast<Pack*>(site + 4 * a.n * a.lay.qmax);  // [T][C]
  const real* t = reinterpret_cast<const real*>(a.tab);
  const int qm = a.lay.qmax, T = a.T, C = a.cols;
  for (int k = threadIdx.x; k < a.n * qm; k += kThreads) {
    site[4 * k] = t[a.lay.off_up1 + k];
    site[4 * k + 1] = t[a.lay.off_dn1 + k];
    site[4 * k + 2] = t[a.lay.off_m + k];
  }
  auto ld = [](const Pack* p) {
    if constexpr (W == 2) {
      const float4 f = __ldg(reinterpret_cast<const float4*>(p));
      Pack o;
      o.z[0].x = f.x;
      o.z[0].y = f.y;
      o.z[1].x = f.z;
      o.z[1].y = f.w;
      return o;
    } else {
      Pack o;
      o.z[0] = __ldg(reinterpret_cast<const v2*>(p));
      return o;
    }
  };
  const int RW = a.R / W;                                  // packs of a row
  const int c0 = blockIdx.y * C, nc = min(C, RW - c0);
  const long long row0 = (long long)blockIdx.x * T;
  const Pack* x = reinterpret_cast<const Pack*>(a.x);
  Pack* y = reinterpret_cast<Pack*>(a.y);
  for (int k = threadIdx.x; k < T * nc; k += kThreads) tile[k] = ld(x + (row0 + k / nc) * RW + c0 + k % nc);
  __syncthreads();
  const real uz = (real)a.obs[0], aur = (real)a.obs[1], aui = (real)a.obs[2];
  for (int k = threadIdx.x; k < T * nc; k += kThreads) {
    const int e = k / nc, c = k - e * nc;
    Pack up, dn;
#pragma unroll
    for (int w = 0; w < W; ++w) up.z[w].x = up.z[w].y = dn.z[w].x = dn.z[w].y = 0;
    real msum = 0;
    auto mac = [&](Pack& s, real f, const Pack& p) {
#pragma unroll
      for (int w = 0; w < W; ++w) {
        s.z[w].x = fma(f, p.z[w].x, s.z[w].x);
        s.z[w].y = fma(f, p.z[w].y, s.z[w].y);
      }
    };
    unsigned rem = (unsigned)e;
    int stride = nc;
    for (int i = 0; i < a.n_low; ++i) {
      const unsigned q = (unsigned)__ldg(a.q + i), nx = rem / q;
      const int d = (int)(rem - nx * q);
      rem = nx;
      const real* s = site + 4 * (i * qm + d);
      msum += s[2];
      if (d > 0) mac(up, s[0], tile[k - stride]);
      if (d + 1 < (int)q) mac(dn, s[1], tile[k + stride]);
      stride *= (int)q;
    }
    unsigned long long high = blockIdx.x;
    const Pack* own = x + (row0 + e) * RW + c0 + c;
    long long far = (long long)T * RW;
    for (int i = a.n_low; i < a.n; ++i) {
      const unsigned q = (unsigned)__ldg(a.q + i);
      const unsigned long long nx = (high >> 32) ? high / q : (unsigned)high / q;
      const int d = (int)(high - nx * q);
      high = nx;
      const real* s = site + 4 * (i * qm + d);
      msum += s[2];
      if (d > 0) mac(up, s[0], ld(own - far));
      if (d + 1 < (int)q) mac(dn, s[1], ld(own + far));
      far *= q;
    }
    const real dz = uz * msum;
    Pack o;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const v2 z = tile[k].z[w], p = up.z[w], m = dn.z[w];
      const real f = a.sigma ? (real)a.sigma[(c0 + c) * W + w] : (real)1;
      o.z[w].x = f * fma(dz, z.x, fma(aur, p.x + m.x, -aui * (p.y - m.y)));
      o.z[w].y = f * fma(dz, z.y, fma(aur, p.y + m.y, aui * (p.x - m.x)));
    }
    y[(row0 + e) * RW + c0 + c] = o;
  }
}

}  // namespace

// y = c (u.S) x for a.R vectors (c = a.sigma[vector], or 1 when a.sigma is null).
// q: the host copy of a.q.
int launch_sdir(SdirArgs a, const int* q, int c64, bool vmaj, void* stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  const int esz = c64 ? 8 : 16;
  // vector-major: four complex64 (two of spins 1/2: four share no arithmetic and cost a
  // low site) or two complex128 vectors a CTA; row-major: up to 128 bytes of a row
  const bool half = vmaj && std::all_of(q, q + a.n, [](int k) { return k == 2; });
  const int most = c64 && !half ? 4 : 2, V = std::min(a.R, most) == 3 ? 4 : std::min(a.R, most);
  const int W = c64 && a.R % 2 == 0 ? 2 : 1;
  a.cols = std::min(a.R / W, 128 / (W * esz));
  const int width = vmaj ? V : a.cols * W;
  a.T = 1;
  a.n_low = 0;
  while (a.n_low < a.n && (a.n_low == 0 || (long long)a.T * q[a.n_low] * width * esz <= kTileBytes)) a.T *= q[a.n_low++];
  const size_t smem = (half ? 0 : (size_t)4 * a.n * a.lay.qmax * (esz / 2)) + (size_t)a.T * width * esz;
  const dim3 grid((unsigned)(a.dim / a.T), (unsigned)((a.R + width - 1) / width));
  if (a.R < 1 || a.dim / a.T > 0x7fffffffll || grid.y > 65535) return (int)cudaErrorInvalidValue;
  const void* k;
  if (!vmaj) {
    k = W == 2 ? (const void*)sdir_rows_kernel<float, 2>
               : (c64 ? (const void*)sdir_rows_kernel<float, 1> : (const void*)sdir_rows_kernel<double, 1>);
  } else if (half && c64) {
    k = V == 2 ? (const void*)sdir_half_kernel<float, 2> : (const void*)sdir_half_kernel<float, 1>;
  } else if (half) {
    k = V == 2 ? (const void*)sdir_half_kernel<double, 2> : (const void*)sdir_half_kernel<double, 1>;
  } else if (c64) {
    k = V == 4 ? (const void*)sdir_vectors_kernel<float, 4>
               : (V == 2 ? (const void*)sdir_vectors_kernel<float, 2> : (const void*)sdir_vectors_kernel<float, 1>);
  } else {
    k = V == 2 ? (const void*)sdir_vectors_kernel<double, 2> : (const void*)sdir_vectors_kernel<double, 1>;
  }
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxSmem);
  if (e != cudaSuccess) return (int)e;
  void* args[] = {&a};
  return (int)cudaLaunchKernel(k, grid, dim3(kThreads), args, smem, st);
}

}  // namespace ftlm
