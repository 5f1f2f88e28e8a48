// All M Lanczos steps of small systems (stored rows, hv_stored.cu) in one launch:
// a thread-block cluster per vector.
//
// Why.  With a launch for the product and one for the update a step of a
// 729-state ring takes 25 us, of which the arithmetic is 2 us: the rest is launch
// gaps, descriptors, and sums that travel through L2 and an arrival counter.  A
// vector's chain depends on no other vector, so one cluster keeps it: every CTA
// holds q_j and q_{j-1} in shared memory (gathers read it there), owns a range of
// rows, and pushes its new rows and partial sums to the other CTAs' shared memory.
// Two hardware cluster barriers a step: after alpha_j and p_j, after |q_{j+1}|^2.
// 24 steps of ten vectors of that ring in complex128: 0.64 -> 0.35 ms (12 us a step, 4
// of them the gather's FP64 operations).
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "device_common.cuh"
#include "ftlm_internal.h"

namespace cg = cooperative_groups;

namespace ftlm {

namespace {

constexpr int kThreads = 256, kLanes = 8, kRowsPass = kThreads / kLanes, kMaxCtas = 8;

// Adds p over the CTA (its first `busy` warps hold something) and leaves the sums in
// slot [rank] of every CTA; the callers then pass a cluster barrier.
template <int NP>
__device__ __forceinline__ void share_sums(cg::cluster_group& cl, int C, int busy, double (&p)[NP], double (*red)[3],
                                           double (*slots)[3]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < busy) {
#pragma unroll
    for (int c = 0; c < NP; ++c)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) p[c] += __shfl_xor_sync(0xffffffffu, p[c], o);
    if (lane == 0)
#pragma unroll
      for (int c = 0; c < NP; ++c) red[warp][c] = p[c];
  }
  __syncthreads();
  if ((int)threadIdx.x < C * NP) {
    const int to = threadIdx.x / NP, c = threadIdx.x % NP;
    double s = 0.0;
    for (int w = 0; w < busy; ++w) s += red[w][c];
    double* remote = cl.map_shared_rank(&slots[0][0], to);
    remote[cl.block_rank() * 3 + c] = s;
  }
}

// The scalars of a step are formed by one thread a CTA: an FP64 operation of a
// whole warp takes 16 clocks of the SM's pipe, so having every thread form them
// (and the row epilogue run in the gather's lanes, one in eight busy) cost 10 of
// the 17 us a step took in the first form.
template <typename real>
__global__ void __launch_bounds__(kThreads, 2) small_run_kernel(const __grid_constant__ SmallRunArgs a) {
  using v2 = typename Cx<real>::v2;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[kThreads / 32][3];
  __shared__ double s_step[kMaxCtas][3], s_norm[kMaxCtas][3];  // by CTA of the cluster
  __shared__ double s_sigma, s_bsp, s_coef;
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int k = (int)blockIdx.x / C;  // the vector
  const InstDesc& d = a.inst[k];
  const int dim = (int)d.dim, M = d.M, l = threadIdx.x & (kLanes - 1);
  const int chunk = (dim + C - 1) / C, r0 = min(rank * chunk, dim), r1 = min(r0 + chunk, dim);
  v2* cur = reinterpret_cast<v2*>(smem_raw);   // q_j, all rows
  v2* prev = cur + dim;                         // q_{j-1}; the own rows become w', then q_{j+1}
  v2* hq = prev + dim;                          // H q_j, the own rows
  const int busy = min(kThreads / 32, (r1 - r0 + 31) / 32);
  const v2* q0 = reinterpret_cast<const v2*>(d.x);
  const v2* u = reinterpret_cast<const v2*>(d.u);
  for (int i = threadIdx.x; i < dim; i += kThreads) cur[i] = q0[i];
  const DevScalars sc = d.sc;
  const StoredRows H = d.stored;
  const v2* val = reinterpret_cast<const v2*>(H.val);
  double sigma = sc.sigma[0], scale = sc.scale[0], beta = 0.0, al = 0.0;  // (thread 0's)
  bool active = sc.active[0] != 0;
  if (threadIdx.x == 0) {
    s_sigma = sigma;
    s_bsp = 0.0;
  }
  cl.sync();
  for (int j = 0; j < M; ++j) {
    const size_t e = (size_t)j * sc.ss;
    if (a.keep) {  // q_j of the stored Lanczos vectors
      v2* out = reinterpret_cast<v2*>(a.keep) + ((size_t)j * a.R + k) * dim;
      for (int i = r0 + (int)threadIdx.x; i < r1; i += kThreads) out[i] = cur[i];
    }
    for (int base = r0; base < r1; base += kRowsPass) {
      const int row = base + (int)threadIdx.x / kLanes;
      real hr = 0, hi = 0;
      if (row < r1) {
        const int n = __ldg(H.cnt + row);
        const int* col = H.col + (size_t)row * H.S;
        const v2* h = val + (size_t)row * H.S;
#pragma unroll 4
        for (int i = l; i < n; i += kLanes) {
          const v2 c = __ldg(h + i), z = cur[__ldg(col + i)];
          hr = fma(c.x, z.x, fma(-c.y, z.y, hr));
          hi = fma(c.x, z.y, fma(c.y, z.x, hi));
        }
      }
#pragma unroll
      for (int o = kLanes / 2; o > 0; o >>= 1) {
        hr += __shfl_xor_sync(0xffffffffu, hr, o);
        hi += __shfl_xor_sync(0xffffffffu, hi, o);
      }
      if (row < r1 && l == 0) {
        hq[row - r0].x = hr;
        hq[row - r0].y = hi;
      }
    }
    __syncthreads();
    const real sg = (real)s_sigma, bs = (real)s_bsp;
    double p[3] = {0.0, 0.0, 0.0};
    for (int i = r0 + (int)threadIdx.x; i < r1; i += kThreads) {
      v2 w = hq[i - r0];
      w.x *= sg;
      w.y *= sg;
      if (j > 0) {
        const v2 qp = prev[i];
        w.x -= bs * qp.x;
        w.y -= bs * qp.y;
      }
      prev[i] = w;
      const v2 x = cur[i], o = __ldg(u + i);
      p[0] += (double)(x.x * w.x + x.y * w.y);
      p[1] += (double)(x.x * o.x + x.y * o.y);
      p[2] += (double)(x.x * o.y - x.y * o.x);
    }
    share_sums<3>(cl, C, busy, p, red, s_step);
    cl.sync();
    if (threadIdx.x == 0) {
      al = 0.0;
      for (int c = 0; c < C; ++c) al += s_step[c][0];
      al *= sigma;
      s_coef = al * sigma;
      if (rank == 0) sc.alpha[e] = al;
    } else if (rank == 0 && (threadIdx.x == 32 || threadIdx.x == 64)) {
      const int c = threadIdx.x / 32;
      double s = 0.0;
      for (int b = 0; b < C; ++b) s += s_step[b][c];
      sc.p[2 * e + c - 1] = s_sigma * s;
    }
    __syncthreads();
    const real coef = (real)s_coef;
    double nrm[1] = {0.0};
    for (int i = r0 + (int)threadIdx.x; i < r1; i += kThreads) {
      v2 w = prev[i];
      const v2 x = cur[i];
      w.x = fma(-coef, x.x, w.x);
      w.y = fma(-coef, x.y, w.y);
      nrm[0] += (double)(w.x * w.x + w.y * w.y);
      for (int c = 0; c < C; ++c) cl.map_shared_rank(prev, c)[i] = w;
    }
    share_sums<1>(cl, C, busy, nrm, red, s_norm);
    cl.sync();
    if (threadIdx.x == 0) {  // as finalize_beta
      double n2 = 0.0;
      for (int c = 0; c < C; ++c) n2 += s_norm[c][0];
      const double bnew = sqrt(fmax(n2, 0.0));
      scale = fmax(scale, fmax(fabs(al), beta));
      const bool stop = active && j < M - 1 && (!(bnew > d.tol * scale) || !isfinite(bnew) || !isfinite(al));
      const double next = active && !stop && bnew > 0.0 ? 1.0 / bnew : 0.0;
      if (rank == 0) {
        sc.beta[e] = bnew;
        sc.sigma[e + sc.ss] = next;
        if (stop) sc.meff[0] = j + 1;
      }
      active = active && !stop;
      s_bsp = bnew * sigma;
      beta = bnew;
      sigma = s_sigma = next;
    }
    v2* t = cur;
    cur = prev;
    prev = t;
    // (s_sigma and s_bsp are read after the gather's barrier)
  }
  if (rank == 0 && threadIdx.x == 0) {
    sc.scale[0] = scale;
    sc.active[0] = active;
  }
}

}  // namespace

// two vectors and the own rows of H q
size_t small_run_smem(long long dim, int ctas, int c64) {
  return (size_t)(2 * dim + (dim + ctas - 1) / ctas) * (c64 ? 8 : 16);
}

// vectors clusters of `ctas` CTAs (1, 2, 4 or 8); max_dim: the largest system's rows.
int launch_small_run(const SmallRunArgs& a, int vectors, int ctas, long long max_dim, int c64, void* stream) {
  const void* k = c64 ? (const void*)small_run_kernel<float> : (const void*)small_run_kernel<double>;
  if (ctas < 1 || ctas > kMaxCtas || max_dim < 1) return (int)cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmallRunBytes);
  if (e != cudaSuccess) return (int)e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(vectors * ctas));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = small_run_smem(max_dim, ctas, c64);
  cfg.stream = reinterpret_cast<cudaStream_t>(stream);
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)ctas;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  void* args[] = {const_cast<SmallRunArgs*>(&a)};
  return (int)cudaLaunchKernelExC(&cfg, k, args);
}

}  // namespace ftlm
