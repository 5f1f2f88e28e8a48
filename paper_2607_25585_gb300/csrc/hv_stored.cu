// H.v of small systems from stored rows (Eq. 3 of arxiv 2607.25585, any spins),
// and the streaming passes of vector-major runs.
//
// Why stored rows.  The matrix-free gathers give one thread a row (or a base of
// the top site's rows) and form every matrix element on the way: a serial chain
// of some hundred dependent loads.  With few rows the chip idles behind it: 174
// us for one H.v of ten vectors of a 729-state ring in complex128, of which the
// FP64 arithmetic would be 2 us.  A system whose rows fit a part of L2 has them
// written out once, on its first product (a warp a row, lanes over the terms),
// and each product is then short sums: eight lanes a row, a group of V vectors,
// added in a fixed order.  Zero elements are not stored, so rows that H does not
// connect stay exactly zero, as in the gathers.  Against extended precision the rows'
// products in complex128 have errors of 1.8 to 2.5e-16, the gathers' 3.8 to 5.0e-16.  For
// many complex64 vectors the rows are read again for every four and the gathers win
// (api.cu, stored_pays).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "device_common.cuh"
#include "ftlm_internal.h"

namespace ftlm {

namespace {

constexpr int kLanes = 8;                        // lanes of a row
constexpr int kBuildWarps = 8;
constexpr int kMaxPairs = kStoredMaxSites * (kStoredMaxSites - 1) / 2;

// One warp a row: entry 0 is the diagonal, then every nonzero element of the
// row's single-site steps and pair flips, packed in term order; coefficients in
// the product's precision from its tables, as the gathers form them.
template <typename real>
__global__ void __launch_bounds__(32 * kBuildWarps) stored_build_kernel(const real* __restrict__ t, const TabLayout L,
                                                                        const long long* __restrict__ stride,
                                                                        const int* __restrict__ q, int n, int dim, int S,
                                                                        int* __restrict__ col, real* __restrict__ val,
                                                                        int* __restrict__ cnt) {
  __shared__ unsigned short pair[kMaxPairs];
  __shared__ real sm[kBuildWarps][kStoredMaxSites];
  __shared__ int sd[kBuildWarps][kStoredMaxSites];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, qm = L.qmax;
  const int npairs = n * (n - 1) / 2;
  for (int k = threadIdx.x; k < n * n; k += blockDim.x) {
    const int i = k / n, j = k % n;
    if (i < j) pair[tri(i, j)] = (unsigned short)(i << 8 | j);
  }
  __syncthreads();
  real* m = sm[warp];
  int* dig = sd[warp];
  const int si = lane < n ? (int)stride[lane] : 1, qi = lane < n ? q[lane] : 1;
  for (int row = blockIdx.x * kBuildWarps + warp; row < dim; row += gridDim.x * kBuildWarps) {
    __syncwarp();
    const int a = (row / si) % qi;
    if (lane < n) {
      dig[lane] = a;
      m[lane] = t[L.off_m + lane * qm + a];
    }
    __syncwarp();
    int pos = 1;
    auto put = [&](bool valid, int c, real re, real im) {
      valid = valid && (re != (real)0 || im != (real)0);
      const unsigned mask = __ballot_sync(0xffffffffu, valid);
      if (valid) {
        const size_t e = (size_t)row * S + pos + __popc(mask & ((1u << lane) - 1u));
        col[e] = c;
        val[2 * e] = re;
        val[2 * e + 1] = im;
      }
      pos += __popc(mask);
    };
    real d = 0, fr = 0, fi = 0, mi = 0;
    if (lane < n) {
      mi = m[lane];
      real zs = t[L.off_hz + lane];
      for (int j = lane + 1; j < n; ++j) zs += t[L.off_zz + lane * n + j] * m[j];
      d = mi * zs + t[L.off_iondiag + lane * qm + a];
      fr = t[L.off_hp + 2 * lane];
      fi = t[L.off_hp + 2 * lane + 1];
      for (int j = 0; j < n; ++j) {
        fr += t[L.off_rho + 2 * (lane * n + j)] * m[j];
        fi += t[L.off_rho + 2 * (lane * n + j) + 1] * m[j];
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    if (lane == 0) {
      col[(size_t)row * S] = row;
      val[2 * (size_t)row * S] = d;
      val[2 * (size_t)row * S + 1] = (real)0;
    }
    {  // single-site steps of site `lane`
      const bool on = lane < n;
      const int b = on ? lane * qm + a : 0;
      const real bzr = on ? t[L.off_bz + 2 * lane] : (real)0, bzi = on ? t[L.off_bz + 2 * lane + 1] : (real)0;
      const real bbr = on ? t[L.off_bb + 2 * lane] : (real)0, bbi = on ? t[L.off_bb + 2 * lane + 1] : (real)0;
      const real u1 = t[L.off_up1 + b], d1 = t[L.off_dn1 + b], u2 = t[L.off_up2 + b], d2 = t[L.off_dn2 + b];
      const real wu = (real)2 * mi - (real)1, wd = (real)2 * mi + (real)1;
      put(on && a >= 1, row - si, (fr + bzr * wu) * u1, (fi + bzi * wu) * u1);
      put(on && a + 1 < qi, row + si, (fr + bzr * wd) * d1, -(fi + bzi * wd) * d1);
      put(on && a >= 2, row - 2 * si, bbr * u2, bbi * u2);
      put(on && a + 2 < qi, row + 2 * si, bbr * d2, -bbi * d2);
    }
    for (int p0 = 0; p0 < npairs; p0 += 32) {  // (uniform over the warp)
      const bool on = p0 + lane < npairs;
      const int ij = pair[on ? p0 + lane : 0], i = ij >> 8, j = ij & 255;
      const int ai = dig[i], aj = dig[j], s1 = (int)stride[i], s2 = (int)stride[j], e = 2 * (i * n + j);
      const real ui = t[L.off_up1 + i * qm + ai], di = t[L.off_dn1 + i * qm + ai];
      const real uj = t[L.off_up1 + j * qm + aj], dj = t[L.off_dn1 + j * qm + aj];
      const real pmr = t[L.off_pm + e], pmi = t[L.off_pm + e + 1], ppr = t[L.off_pp + e], ppi = t[L.off_pp + e + 1];
      const bool iu = on && ai >= 1, id = on && ai + 1 < q[i], ju = aj >= 1, jd = aj + 1 < q[j];
      put(iu && jd, row - s1 + s2, pmr * (ui * dj), pmi * (ui * dj));
      put(id && ju, row + s1 - s2, pmr * (di * uj), -pmi * (di * uj));
      put(iu && ju, row - s1 - s2, ppr * (ui * uj), ppi * (ui * uj));
      put(id && jd, row + s1 + s2, ppr * (di * dj), -ppi * (di * dj));
    }
    if (lane == 0) cnt[row] = pos;
  }
}

// A CTA takes 32 rows (eight lanes each) of V vectors.  STEP: a Lanczos step of a
// vector-major run, tiles from the groups' list: w' = sigma_j H q_j - beta_{j-1}
// sigma_{j-1} q_{j-1} over q_{j-1}, alpha_j and p_j by the group's last CTA.
// Else y = H x with element (row, v) at row * rs + v * vs.
template <typename real, int V, bool STEP>
__global__ void __launch_bounds__(256) stored_rows_kernel(const __grid_constant__ StoredArgs a) {
  using v2 = typename Cx<real>::v2;
  __shared__ double red[8][V * 3];
  __shared__ int last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, l = lane & (kLanes - 1);
  int g = 0, tile = blockIdx.x, tiles = 0, nv = V, vec0 = 0;
  const InstDesc* in = nullptr;
  StoredRows H;
  const v2* x;
  long long dim, rs, vs;
  if (STEP) {
    g = find_instance(a.tile_start, a.groups, tile);
    const int t0 = __ldg(a.tile_start + g);
    tiles = __ldg(a.tile_start + g + 1) - t0;
    tile -= t0;
    const int per_system = (a.R + V - 1) / V, first = g % per_system * V;  // (a system's last group may be smaller)
    vec0 = g / per_system * a.R + first;
    nv = min(V, a.R - first);
    in = a.inst + vec0;
    H = in->stored;
    dim = in->dim;
    x = reinterpret_cast<const v2*>(in->x);
    rs = 1;
    vs = dim;
  } else {
    H = a.rows;
    dim = a.dim;
    rs = a.rs;
    vs = a.vs;
    x = reinterpret_cast<const v2*>(a.x) + blockIdx.y * V * vs;
    nv = min(V, a.R - (int)blockIdx.y * V);
  }
  const long long row = (long long)tile * 32 + (threadIdx.x >> 3);
  const bool on = row < dim;
  real ar[V], ai[V];
#pragma unroll
  for (int v = 0; v < V; ++v) ar[v] = ai[v] = 0;
  if (on) {
    const int n = __ldg(H.cnt + row);
    const int* col = H.col + row * H.S;
    const v2* val = reinterpret_cast<const v2*>(H.val) + row * H.S;
    for (int e = l; e < n; e += kLanes) {
      const v2 h = __ldg(val + e);
      const v2* p = x + (long long)__ldg(col + e) * rs;
#pragma unroll
      for (int v = 0; v < V; ++v) {
        if (v >= nv) break;
        const v2 z = __ldg(p + v * vs);
        ar[v] = fma(h.x, z.x, fma(-h.y, z.y, ar[v]));
        ai[v] = fma(h.x, z.y, fma(h.y, z.x, ai[v]));
      }
    }
  }
  real hr = 0, hi = 0;  // lane l of the row keeps vector l
#pragma unroll
  for (int v = 0; v < V; ++v) {
#pragma unroll
    for (int o = kLanes / 2; o > 0; o >>= 1) {
      ar[v] += __shfl_xor_sync(0xffffffffu, ar[v], o);
      ai[v] += __shfl_xor_sync(0xffffffffu, ai[v], o);
    }
    if (v == l) {
      hr = ar[v];
      hi = ai[v];
    }
  }
  const bool mine = on && l < nv;
  if (!STEP) {
    if (mine) {
      v2 o;
      o.x = hr;
      o.y = hi;
      reinterpret_cast<v2*>(a.y)[(blockIdx.y * V + l) * vs + row * rs] = o;
    }
    return;
  }
  double p[3] = {0.0, 0.0, 0.0};
  if (mine) {
    const DevScalars& sc = in[l].sc;
    const size_t e = (size_t)a.j * sc.ss;
    const real sg = (real)sc.sigma[e];
    const long long at = l * vs + row;
    v2* y = reinterpret_cast<v2*>(in->y) + at;
    v2 w;
    w.x = sg * hr;
    w.y = sg * hi;
    if (a.j > 0) {
      const real bsp = (real)(sc.beta[e - sc.ss] * sc.sigma[e - sc.ss]);
      const v2 qp = *y;
      w.x -= bsp * qp.x;
      w.y -= bsp * qp.y;
    }
    *y = w;
    const v2 xv = __ldg(x + at), uv = __ldg(reinterpret_cast<const v2*>(in->u) + at);
    p[0] = (double)(xv.x * w.x + xv.y * w.y);
    p[1] = (double)(xv.x * uv.x + xv.y * uv.y);
    p[2] = (double)(xv.x * uv.y - xv.y * uv.x);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c)
#pragma unroll
    for (int o = 16; o >= kLanes; o >>= 1) p[c] += __shfl_xor_sync(0xffffffffu, p[c], o);
  if (lane < V)
#pragma unroll
    for (int c = 0; c < 3; ++c) red[warp][lane * 3 + c] = p[c];
  __syncthreads();
  double* slots = a.slots + (size_t)vec0 * a.max_tiles * 3;  // [vector][tile][3]
  if ((int)threadIdx.x < nv * 3) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += red[w][threadIdx.x];
    slots[((size_t)(threadIdx.x / 3) * a.max_tiles + tile) * 3 + threadIdx.x % 3] = s;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(a.counters + g, 1u) == (unsigned)(tiles - 1);
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int k = warp; k < nv * 3; k += 8) {
    const int v = k / 3, c = k % 3;
    double s = 0.0;
    for (int i = lane; i < tiles; i += 32) s += __ldcg(slots + ((size_t)v * a.max_tiles + i) * 3 + c);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      const DevScalars& sc = in[v].sc;
      const size_t e = (size_t)a.j * sc.ss;
      const double r = sc.sigma[e] * s;
      if (c == 0) sc.alpha[e] = r;
      else sc.p[2 * e + c - 1] = r;
    }
  }
  if (threadIdx.x == 0) a.counters[g] = 0u;
}

// Streaming passes over one-vector instances, a CTA a chunk of one vector:
// MODE kModeUpdate: w = w' - alpha_j sigma_j q_j with |w|^2, then beta_j, sigma_{j+1};
// kModeStartNorm: |q_0|^2, then sigma_0.  Bound: HBM.  A thread's loads (eight of 16
// bytes for each array) all precede its stores; the last CTA of each vector adds
// that vector's partial sums, so no tail over all vectors follows (with one last
// CTA for all of them the update took 0.98 ms for 1.9e8 complex64 values).
template <typename real, int W, int MODE>
__global__ void __launch_bounds__(256) stream_vectors_kernel(const __grid_constant__ StreamArgs a) {
  using v2 = typename Cx<real>::v2;
  constexpr int U = kStreamChunk / (256 * W);
  struct __align__(sizeof(v2) * W) Pack {
    v2 z[W];
  };
  const int g = find_instance(a.tile_start, a.vectors, blockIdx.x);
  const int t0 = __ldg(a.tile_start + g), tiles = __ldg(a.tile_start + g + 1) - t0, tile = (int)blockIdx.x - t0;
  const InstDesc& d = a.inst[g];
  const DevScalars& sc = d.sc;
  const long long dim = d.dim, e0 = (long long)tile * kStreamChunk;
  const Pack* x = reinterpret_cast<const Pack*>(reinterpret_cast<const v2*>(d.x) + e0) + threadIdx.x;
  Pack* y = reinterpret_cast<Pack*>(reinterpret_cast<v2*>(d.y) + e0) + threadIdx.x;
  const int left = (int)min((long long)kStreamChunk, dim - e0) / W;  // (W divides every vector's length)
  real coef = 0;
  if (MODE == kModeUpdate) {
    const size_t e = (size_t)a.j * sc.ss;
    coef = (real)(sc.alpha[e] * sc.sigma[e]);
  }
  Pack q[U], w[U];
  double p[1] = {0.0};
  real sum = 0;
#pragma unroll
  for (int u = 0; u < U; ++u)
    if ((int)threadIdx.x + u * 256 < left) {
      q[u] = x[u * 256];
      if (MODE == kModeUpdate) w[u] = y[u * 256];
    }
#pragma unroll
  for (int u = 0; u < U; ++u)
    if ((int)threadIdx.x + u * 256 < left) {
#pragma unroll
      for (int k = 0; k < W; ++k) {
        v2 z = q[u].z[k];
        if (MODE == kModeUpdate) {
          z.x = fma(-coef, z.x, w[u].z[k].x);
          z.y = fma(-coef, z.y, w[u].z[k].y);
          w[u].z[k] = z;
        }
        sum += z.x * z.x + z.y * z.y;
      }
      if (MODE == kModeUpdate) y[u * 256] = w[u];
    }
  p[0] = (double)sum;
  if (vector_total<256, 1>(p, a.slots + (size_t)g * a.max_tiles * 3, tile, tiles, a.counters + g)) {
    if (MODE == kModeUpdate) finalize_beta(sc, a.j, 0, d.M, d.tol, p[0]);
    else finalize_start(sc, 0, d.M, p[0]);
  }
}

template <typename real, int V>
int launch_step_v(const StoredArgs& a, int grid, cudaStream_t st) {
  stored_rows_kernel<real, V, true><<<grid, 256, 0, st>>>(a);
  return (int)cudaGetLastError();
}

template <typename real, int V>
int launch_product_v(const StoredArgs& a, cudaStream_t st) {
  const dim3 grid((unsigned)((a.dim + 31) / 32), (unsigned)((a.R + V - 1) / V));
  stored_rows_kernel<real, V, false><<<grid, 256, 0, st>>>(a);
  return (int)cudaGetLastError();
}

}  // namespace

// Entries a row can have at most (0: too many sites for the builder).
int stored_row_bound(const HostSystem& hs) {
  if (hs.n > kStoredMaxSites) return 0;
  const TabLayout& L = hs.lay;
  const double* t = hs.tab.data();
  int S = 1;
  for (int i = 0; i < hs.n; ++i) {
    S += hs.q[i] == 2 ? 1 : (hs.q[i] == 3 ? 3 : 4);  // +-1 and +-2 steps
    for (int j = i + 1; j < hs.n; ++j) {
      const int e = 2 * (i * hs.n + j);
      const int pm = t[L.off_pm + e] != 0.0 || t[L.off_pm + e + 1] != 0.0, pp = t[L.off_pp + e] != 0.0 || t[L.off_pp + e + 1] != 0.0;
      if (!pm && !pp) continue;
      const int halves = (hs.q[i] == 2) + (hs.q[j] == 2);
      S += halves == 2 ? 1 : (halves == 1 ? 2 : 2 * (pm + pp));
    }
  }
  return (S + 3) & ~3;
}

// Average entries of a row, from its digits' distribution, and the coupled pairs.
void stored_row_work(const HostSystem& hs, double& entries, int& pairs) {
  const TabLayout& L = hs.lay;
  const double* t = hs.tab.data();
  auto on = [&](int at) { return t[at] != 0.0 || t[at + 1] != 0.0; };
  entries = 1.0;
  pairs = 0;
  for (int i = 0; i < hs.n; ++i) {
    const double step = 2.0 - 2.0 / hs.q[i];
    bool field = on(L.off_hp + 2 * i) || on(L.off_bz + 2 * i);
    for (int j = 0; j < hs.n; ++j) field = field || on(L.off_rho + 2 * (i * hs.n + j));
    if (field) entries += step;
    if (on(L.off_bb + 2 * i)) entries += 2.0 * std::max(0, hs.q[i] - 2) / hs.q[i];
    for (int j = i + 1; j < hs.n; ++j) {
      const int e = 2 * (i * hs.n + j), kinds = on(L.off_pm + e) + on(L.off_pp + e);
      entries += kinds * 0.5 * step * (2.0 - 2.0 / hs.q[j]);
      pairs += kinds > 0;
    }
  }
}

int launch_stored_build(const void* tab, const TabLayout& L, const long long* stride, const int* q, int n, int dim,
                        int S, int* col, void* val, int* cnt, int c64, void* stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (n > kStoredMaxSites) return (int)cudaErrorInvalidValue;
  const int grid = std::min((dim + kBuildWarps - 1) / kBuildWarps, 8 * std::max(1, device_sm_count()));
  if (c64)
    stored_build_kernel<float><<<grid, 32 * kBuildWarps, 0, st>>>((const float*)tab, L, stride, q, n, dim, S, col, (float*)val, cnt);
  else
    stored_build_kernel<double><<<grid, 32 * kBuildWarps, 0, st>>>((const double*)tab, L, stride, q, n, dim, S, col, (double*)val, cnt);
  return (int)cudaGetLastError();
}

int launch_stored_step(const StoredArgs& a, int V, int c64, int grid, void* stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (V == 4) return c64 ? launch_step_v<float, 4>(a, grid, st) : launch_step_v<double, 4>(a, grid, st);
  if (V == 2) return c64 ? launch_step_v<float, 2>(a, grid, st) : launch_step_v<double, 2>(a, grid, st);
  if (V == 1) return c64 ? launch_step_v<float, 1>(a, grid, st) : launch_step_v<double, 1>(a, grid, st);
  return (int)cudaErrorInvalidValue;
}

int launch_stored_product(const StoredArgs& a, int V, int c64, void* stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (V == 4) return c64 ? launch_product_v<float, 4>(a, st) : launch_product_v<double, 4>(a, st);
  if (V == 2) return c64 ? launch_product_v<float, 2>(a, st) : launch_product_v<double, 2>(a, st);
  if (V == 1) return c64 ? launch_product_v<float, 1>(a, st) : launch_product_v<double, 1>(a, st);
  return (int)cudaErrorInvalidValue;
}

// even: every vector's length is even (complex64 then moves 16 bytes a load)
int launch_stream_vectors(const StreamArgs& a, int mode, int c64, bool even, int grid, void* stream) {
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (mode != kModeUpdate && mode != kModeStartNorm) return (int)cudaErrorInvalidValue;
  const bool up = mode == kModeUpdate;
  if (!c64) {
    if (up) stream_vectors_kernel<double, 1, kModeUpdate><<<grid, 256, 0, st>>>(a);
    else stream_vectors_kernel<double, 1, kModeStartNorm><<<grid, 256, 0, st>>>(a);
  } else if (even) {
    if (up) stream_vectors_kernel<float, 2, kModeUpdate><<<grid, 256, 0, st>>>(a);
    else stream_vectors_kernel<float, 2, kModeStartNorm><<<grid, 256, 0, st>>>(a);
  } else {
    if (up) stream_vectors_kernel<float, 1, kModeUpdate><<<grid, 256, 0, st>>>(a);
    else stream_vectors_kernel<float, 1, kModeStartNorm><<<grid, 256, 0, st>>>(a);
  }
  return (int)cudaGetLastError();
}

}  // namespace ftlm
