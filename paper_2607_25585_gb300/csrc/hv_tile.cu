// General H.v (Eq. 3 of arxiv 2607.25585, any spins) on vector-major blocks in
// complex64, over tiles of low sites in shared memory.
//
// Rows.  As in hv_cube.cu a thread owns one base b (the digits of all sites but
// the top one, T) and the Q = 2s+1 rows b + a s_T of the top site, for V vectors.
// A CTA's bases are one whole tile: L = q_0 q_1 ... q_{nl-1} consecutive bases, all
// digits of the nl low sites, with the high sites' digits fixed.
//
// Terms.  A pair's partner row is in the CTA's own tile when both sites are low,
// and in the tile shifted by +-s_j when one of them, j, is high.  The CTA keeps
// its own tile in shared memory and, for one high site and direction after the
// other, the shifted tile, which serves the single flip of j, its pairs with the
// top site (registers) and its pairs with every low site.  Only pairs of two high
// sites are gathered from L2, and their digits, like every high site's, are the
// same for the whole CTA, so those branches do not diverge.
//
// Bound: issue slots (44 % busy with 12 to 16 warps an SM; a third of the
// instructions are shared-memory loads and packed FMAs, the rest forms places and
// coefficients).  The register-cube gather loads every pair's rows through L1 and
// waits for L2 between them.  A step of the 24 chains of 10 to 12 spins 1 with 16
// vectors: 8.6 -> 7.0 ms; of ten 9-site molecules of spins 5/2 and 2 with 8
// vectors: 16.1 -> 14.2 ms.  Coefficients with no imaginary part (all s+ s- ones, and s+
// s+ ones of chains along an axis) take one packed FMA a value instead of two.
// Tiles of 81 bases (9.3 ms) or 729 (8.4 ms, one CTA an SM) were slower.
// Copying all the high sites' rows ahead through shared memory (8.1 ms on the chains,
// 13.0 to 13.7 on the molecules) or the shifted tiles alone (7.2 and 13.3) did not pay:
// the copies take the issue slots that the waits left.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "device_common.cuh"
#include "ftlm_internal.h"
#include "rows_common.cuh"

namespace ftlm {

namespace {

using Acc = Cx<float>;
constexpr size_t kTileSmem = 220 * 1024;

template <int Q, int V, int NTMAX, int MINB>
__global__ void __launch_bounds__(NTMAX, MINB) tile_gather_kernel(const __grid_constant__ LaunchArgs a, int L, int nl, int R) {
  constexpr int P = NTMAX;  // pitch of a tile's values: compile-time offsets between a base's Q V values
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int NT = blockDim.x, tid = threadIdx.x;
  float* t = reinterpret_cast<float*>(smem_raw);                                     // the system's tables
  float2* own = reinterpret_cast<float2*>(smem_raw + (((size_t)a.tab_reals * 4 + 15) & ~size_t(15)));  // [Q V][P]
  float2* nbr = own + (size_t)Q * V * P;                                              // [Q V][P]
  float* sacc = reinterpret_cast<float*>(nbr + (size_t)Q * V * P);                    // [V 3][P]
  float* lup = sacc + V * 3 * P + tid;                                                // [nl][P] <a|s+|a-1> of the thread's low digits
  float* ldn = lup + (size_t)nl * P;                                                  // [nl][P] <a|s-|a+1>
  float* lm = ldn + (size_t)nl * P;                                                   // [nl][P] m
  __shared__ InstDesc d;
  __shared__ int sq[kMaxSites], sst[kMaxSites], hd[kMaxSites];  // radices, strides, the tile's high digits
  __shared__ float hm[kMaxSites];                               // and their m values
  __shared__ float2 hF[kMaxSites];                              // h+_j + sum over high i of rho_ji m_i
  __shared__ float hG[kMaxSites];                               // sum over high j of zz_ij m_j
  __shared__ float hE;                                          // diagonal of the high sites alone
  __shared__ unsigned s_rho;                                    // bit j: some rho_ji is not zero
  __shared__ double s_sg[V], s_bsp[V];
  __shared__ int is_last;
  const int lane = tid & 31, warp = tid >> 5, nwarps = NT >> 5;
  const bool fused = a.fused_step != 0;
  const InstDesc* insts = a.inst;  // one a vector, R a system; groups of V, the last of a system may be smaller
  const int per_system = (R + V - 1) / V, nvec = a.n_inst / per_system * R;
  auto first_of = [&](int g) { return g / per_system * R + g % per_system * V; };
  auto count_of = [&](int g) { return min(V, R - g % per_system * V); };
  if (fused) {
    for (int k = tid; k < nvec * kNumPartials; k += NT)
      a.partials[((size_t)(k / kNumPartials) * gridDim.x + blockIdx.x) * kNumPartials + k % kNumPartials] = 0.0;
    for (int k = tid; k < V * 3 * P; k += NT) sacc[k] = 0;
  }
  auto flush = [&](int g) {  // the CTA's sums of group g's vectors, in a fixed order
    __syncthreads();
    for (int item = warp; item < count_of(g) * 3; item += nwarps) {
      double s = 0.0;
      for (int k = lane; k < NT; k += 32) {
        s += (double)sacc[item * P + k];
        sacc[item * P + k] = 0;
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0)
        a.partials[((size_t)(first_of(g) + item / 3) * gridDim.x + blockIdx.x) * kNumPartials + item % 3] = s;
    }
    __syncthreads();
  };
  const bool on = tid < L;
  const int e = on ? tid : 0;
  float diag_low = 0;  // diagonal of the thread's low sites alone
  int cur = -1;
  const void* staged = nullptr;
  for (int tile = blockIdx.x; tile < a.ntiles; tile += gridDim.x) {
    // (inline_one: one regular block, a.tiles_per_vg tiles a group)
    const int g = a.inline_one ? tile / a.tiles_per_vg : find_instance(a.tile_start, a.n_inst, tile);
    if (g != cur) {
      if (fused && cur >= 0) flush(cur);
      __syncthreads();
      if (tid == 0) {
        d = a.inline_one ? a.one : insts[first_of(g)];
        if (a.inline_one) {
          d.x = static_cast<const char*>(d.x) + first_of(g) * a.vm_stride;
          d.y = static_cast<char*>(d.y) + first_of(g) * a.vm_stride;
        }
      }
      if (fused && tid < count_of(g)) {
        const DevScalars& sc = insts[first_of(g) + tid].sc;
        const int j = a.step;
        s_sg[tid] = sc.sigma[(size_t)j * sc.ss];
        s_bsp[tid] = a.first ? 0.0 : sc.beta[(size_t)(j - 1) * sc.ss] * sc.sigma[(size_t)(j - 1) * sc.ss];
      }
      __syncthreads();
      if (d.tab != staged) {  // a new system: its tables, and what depends on the thread's low digits alone
        const float* src = reinterpret_cast<const float*>(d.tab);
        for (int i = tid; i < d.lay.total; i += NT) t[i] = src[i];
        for (int i = tid; i < d.n; i += NT) {
          sq[i] = d.q[i];
          sst[i] = (int)d.stride[i];
        }
        if (tid == 0) s_rho = 0;
        __syncthreads();
        const TabLayout& Ly = d.lay;
        if (tid < d.n) {
          bool any = false;
          for (int i = 0; i < d.n; ++i)
            any = any || t[Ly.off_rho + 2 * (tid * d.n + i)] != 0.f || t[Ly.off_rho + 2 * (tid * d.n + i) + 1] != 0.f;
          if (any) atomicOr(&s_rho, 1u << tid);
        }
        int rem = e;
        diag_low = 0;
        for (int i = 0; i < nl; ++i) {
          const int ai = rem % sq[i];
          rem /= sq[i];
          const Quad<float> ti = ld4(t + Ly.off_site4 + 4 * (i * Ly.qmax + ai));
          lup[i * P] = ti.a;
          ldn[i * P] = ti.b;
          lm[i * P] = ti.c;
          float zs = t[Ly.off_hz + i];
          for (int k = 0; k < i; ++k) zs = fmaf(t[Ly.off_zz + k * d.n + i], lm[k * P], zs);
          diag_low += fmaf(ti.c, zs, ti.d);
        }
        staged = d.tab;
      }
      cur = g;
    }
    __syncthreads();  // the previous tile's reads are done
    const int n = d.n, T = n - 1, qm = d.lay.qmax;
    const TabLayout& Ly = d.lay;
    const int h = a.inline_one ? tile % a.tiles_per_vg : tile - __ldg(a.tile_start + g);
    const int dim = (int)d.dim, sT = sst[T], b = h * L + e;  // (32-bit rows)
    const int nv = count_of(g);  // (a smaller group reads its last vector in the others' place)
    const float2* x = reinterpret_cast<const float2*>(d.x);
    auto load = [&](int row, float2(&z)[Q][V]) {
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const float2* p = x + (size_t)min(v, nv - 1) * dim + row;
#pragma unroll
        for (int q = 0; q < Q; ++q) z[q][v] = __ldg(p + q * sT);
      }
    };
    auto keep = [&](float2* buf, const float2(&z)[Q][V]) {
#pragma unroll
      for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int v = 0; v < V; ++v) buf[(q * V + v) * P + tid] = z[q][v];
    };
    Acc acc[Q][V];
    float2 z[Q][V];
    load(b, z);
    if (tid < T && tid >= nl) {  // the high digits
      int rem = h;
      for (int i = nl; i < tid; ++i) rem /= sq[i];
      hd[tid] = rem % sq[tid];
      hm[tid] = t[Ly.off_m + tid * qm + hd[tid]];
    }
    __syncthreads();
    if (tid < n) {  // their sums for every site
      float2 f = *reinterpret_cast<const float2*>(t + Ly.off_hp + 2 * tid);
      float zs = 0;
      for (int i = nl; i < T; ++i) {
        const float2 rho = *reinterpret_cast<const float2*>(t + Ly.off_rho + 2 * (tid * n + i));
        f.x = fmaf(rho.x, hm[i], f.x);
        f.y = fmaf(rho.y, hm[i], f.y);
        if (i != tid) zs = fmaf(i < tid ? t[Ly.off_zz + i * n + tid] : t[Ly.off_zz + tid * n + i], hm[i], zs);
      }
      hF[tid] = f;
      hG[tid] = zs;
    } else if (tid == NT - 1) {
      float s = 0;
      for (int i = nl; i < T; ++i) {
        float zs = t[Ly.off_hz + i];
        for (int j = i + 1; j < T; ++j) zs = fmaf(t[Ly.off_zz + i * n + j], hm[j], zs);
        s += fmaf(hm[i], zs, t[Ly.off_iondiag + i * qm + hd[i]]);
      }
      hE = s;
    }
    keep(own, z);
    __syncthreads();
    // acc += (cr + i ci) times the cube at place `at` of a tile; one packed FMA a value where re
    auto mac_tile = [&](const float2* buf, int at, float cr, float ci, bool re) {
      const float2* p = buf + at;
      if (re) {
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
          for (int v = 0; v < V; ++v) acc[q][v].mac_re(cr, p[(q * V + v) * P]);
      } else {
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
          for (int v = 0; v < V; ++v) acc[q][v].mac(cr, ci, p[(q * V + v) * P]);
      }
    };
    auto mac_regs = [&](const float2(&z)[Q][V], float cr, float ci, bool re) {
      if (re) {
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
          for (int v = 0; v < V; ++v) acc[q][v].mac_re(cr, z[q][v]);
      } else {
#pragma unroll
        for (int q = 0; q < Q; ++q)
#pragma unroll
          for (int v = 0; v < V; ++v) acc[q][v].mac(cr, ci, z[q][v]);
      }
    };
    // site j's single-flip coefficient without its own digit: the high sites' part and the low ones'
    auto field = [&](int j) {
      float2 f = hF[j];
      if ((s_rho >> j) & 1u)
        for (int i = 0; i < nl; ++i) {
          const float2 rho = *reinterpret_cast<const float2*>(t + Ly.off_rho + 2 * (j * n + i));
          const float mi = lm[i * P];
          f.x = fmaf(rho.x, mi, f.x);
          f.y = fmaf(rho.y, mi, f.y);
        }
      return f;
    };
    // diagonal and the top site's own flips
    {
      float diag = diag_low + hE, zT = hG[T];
      for (int i = 0; i < nl; ++i) {
        const float mi = lm[i * P];
        diag = fmaf(mi, hG[i], diag);
        zT = fmaf(t[Ly.off_zz + i * n + T], mi, zT);
      }
      const float2 fT = field(T);
      const float hzT = t[Ly.off_hz + T];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const Quad<float> tq = ld4(t + Ly.off_site4 + 4 * (T * qm + q));
        const float ed = diag + tq.c * (hzT + zT) + tq.d;
#pragma unroll
        for (int v = 0; v < V; ++v) acc[q][v].set(ed, z[q][v]);
      }
      const float bzr = t[Ly.off_bz + 2 * T], bzi = t[Ly.off_bz + 2 * T + 1];
      const float bbr = t[Ly.off_bb + 2 * T], bbi = t[Ly.off_bb + 2 * T + 1];
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const Quad<float> tq = ld4(t + Ly.off_site4 + 4 * (T * qm + q));
        auto row = [&](float cr, float ci, int from) {
#pragma unroll
          for (int v = 0; v < V; ++v) acc[q][v].mac(cr, ci, z[from][v]);
        };
        if (q >= 1) {  // s+_T: (F_T + bz (2m - 1)) <q|s+|q-1>
          const float w = 2.f * tq.c - 1.f;
          row((fT.x + bzr * w) * tq.a, (fT.y + bzi * w) * tq.a, q - 1);
        }
        if (q + 1 < Q) {  // s-_T
          const float w = 2.f * tq.c + 1.f;
          row((fT.x + bzr * w) * tq.b, -(fT.y + bzi * w) * tq.b, q + 1);
        }
        if (q >= 2) {
          const float u2 = t[Ly.off_up2 + T * qm + q];
          row(bbr * u2, bbi * u2, q - 2);
        }
        if (q + 2 < Q) {
          const float d2 = t[Ly.off_dn2 + T * qm + q];
          row(bbr * d2, -bbi * d2, q + 2);
        }
      }
    }
    // site j's step to the cube now in z, w its ladder coefficient: its single flip
    // (f: field(j)) and its pairs with the top site
    auto step = [&](int j, float2 f, float mj, float w, bool up) {
      const float mm = up ? 2.f * mj - 1.f : 2.f * mj + 1.f, im = up ? 1.f : -1.f;
      const float fr = (f.x + t[Ly.off_bz + 2 * j] * mm) * w, fi = im * (f.y + t[Ly.off_bz + 2 * j + 1] * mm) * w;
      const float2 rhoT = *reinterpret_cast<const float2*>(t + Ly.off_rho + 2 * (j * n + T));
      const Quad<float> c = ld4(t + Ly.off_pair4 + 4 * (j * n + T));  // s+_j s-_T and s+_j s+_T
      // with the top digit coming from q + 1 (s-_T) and from q - 1 (s+_T)
      const float ar = w * (up ? c.a : c.c), ai = im * w * (up ? c.b : c.d);
      const float br = w * (up ? c.c : c.a), bi = im * w * (up ? c.d : c.b);
      const float rr = rhoT.x * w, ri = im * rhoT.y * w;
      const bool are = ai == 0.f, bre = bi == 0.f;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const Quad<float> tq = ld4(t + Ly.off_site4 + 4 * (T * qm + q));
        const float cr = fmaf(rr, tq.c, fr), ci = fmaf(ri, tq.c, fi);
#pragma unroll
        for (int v = 0; v < V; ++v) acc[q][v].mac(cr, ci, z[q][v]);
        if (q + 1 < Q) {
#pragma unroll
          for (int v = 0; v < V; ++v)
            if (are) acc[q][v].mac_re(ar * tq.b, z[q + 1][v]);
            else acc[q][v].mac(ar * tq.b, ai * tq.b, z[q + 1][v]);
        }
        if (q >= 1) {
#pragma unroll
          for (int v = 0; v < V; ++v)
            if (bre) acc[q][v].mac_re(br * tq.a, z[q - 1][v]);
            else acc[q][v].mac(br * tq.a, bi * tq.a, z[q - 1][v]);
        }
      }
    };
    // site j's step (ladder coefficient w) with the low sites i < end, from a tile whose entry for this base is `at`
    auto with_low = [&](const float2* buf, int at, int j, int end, float w, bool up) {
      for (int i = 0; i < end; ++i) {
        const Quad<float> c = ld4(t + Ly.off_pair4 + 4 * (i * n + j));  // s+_i s-_j and s+_i s+_j
        const float ui = lup[i * P] * w, di = ldn[i * P] * w;
        const int si = sst[i];
        // s+_i: with s+_j pp, with s-_j pm;  s-_i: with s+_j conj pm, with s-_j conj pp
        const float ur = up ? c.c : c.a, uim = up ? c.d : c.b, dr = up ? c.a : c.c, dim_ = up ? c.b : c.d;
        if (ui != 0.f) mac_tile(buf, at - si, ur * ui, uim * ui, uim == 0.f);
        if (di != 0.f) mac_tile(buf, at + si, dr * di, -dim_ * di, dim_ == 0.f);
      }
    };
    // low sites j: everything from the own tile
    if (on) {
      int rem = e;
      for (int j = 0; j < nl; ++j) {
        const int sj = sst[j], qj = sq[j], aj = rem % qj;
        rem /= qj;
        const float2 f = field(j);
        const float bbr = t[Ly.off_bb + 2 * j], bbi = t[Ly.off_bb + 2 * j + 1], mj = lm[j * P];
        if (bbr != 0.f || bbi != 0.f) {
          const float u2 = t[Ly.off_up2 + j * qm + aj], d2 = t[Ly.off_dn2 + j * qm + aj];
          if (aj >= 2) mac_tile(own, e - 2 * sj, bbr * u2, bbi * u2, false);
          if (aj + 2 < qj) mac_tile(own, e + 2 * sj, bbr * d2, -bbi * d2, false);
        }
#pragma unroll 1
        for (int dir = 0; dir < 2; ++dir) {
          const bool up = dir == 0;
          const float w = up ? lup[j * P] : ldn[j * P];
          if (w == 0.f) continue;
          const int at = up ? e - sj : e + sj;
#pragma unroll
          for (int q = 0; q < Q; ++q)
#pragma unroll
            for (int v = 0; v < V; ++v) z[q][v] = own[(q * V + v) * P + at];
          step(j, f, mj, w, up);
          with_low(own, at, j, j, w, up);
        }
      }
    }
    // high sites j (their digits are the CTA's)
    for (int j = nl; j < T; ++j) {
      const int aj = hd[j], sj = sst[j], qj = sq[j];
      const Quad<float> tj = ld4(t + Ly.off_site4 + 4 * (j * qm + aj));
      const float bbr = t[Ly.off_bb + 2 * j], bbi = t[Ly.off_bb + 2 * j + 1];
      const float2 f = field(j);
      if (bbr != 0.f || bbi != 0.f) {
        const float u2 = t[Ly.off_up2 + j * qm + aj], d2 = t[Ly.off_dn2 + j * qm + aj];
        if (aj >= 2) {
          load(b - 2 * sj, z);
          mac_regs(z, bbr * u2, bbi * u2, false);
        }
        if (aj + 2 < qj) {
          load(b + 2 * sj, z);
          mac_regs(z, bbr * d2, -bbi * d2, false);
        }
      }
#pragma unroll 1
      for (int dir = 0; dir < 2; ++dir) {
        const bool up = dir == 0;
        if (up ? aj < 1 : aj + 1 >= qj) continue;
        const int bj = up ? b - sj : b + sj;
        const float w = up ? tj.a : tj.b;
        load(bj, z);
        __syncthreads();  // the previous shifted tile has been read
        keep(nbr, z);
        __syncthreads();
        if (!on) continue;
        step(j, f, tj.c, w, up);
        with_low(nbr, e, j, nl, w, up);
#pragma unroll 1
        for (int i = nl; i < j; ++i) {  // two high sites
          const int ai = hd[i], si = sst[i];
          const Quad<float> ti = ld4(t + Ly.off_site4 + 4 * (i * qm + ai));
          const Quad<float> c = ld4(t + Ly.off_pair4 + 4 * (i * n + j));
          const float ur = up ? c.c : c.a, uim = up ? c.d : c.b, dr = up ? c.a : c.c, dim_ = up ? c.b : c.d;
          if (ai >= 1) {
            const float k = w * ti.a;
            load(bj - si, z);
            mac_regs(z, ur * k, uim * k, uim == 0.f);
          }
          if (ai + 1 < sq[i]) {
            const float k = w * ti.b;
            load(bj + si, z);
            mac_regs(z, dr * k, -dim_ * k, dim_ == 0.f);
          }
        }
      }
    }
    if (!on) continue;
    float2* y = reinterpret_cast<float2*>(d.y);
    const float2* u = reinterpret_cast<const float2*>(d.u);
#pragma unroll
    for (int v = 0; v < V; ++v) {
      if (v >= nv) break;
      const float sg = fused ? (float)s_sg[v] : 1.f, bsp = fused ? (float)s_bsp[v] : 0.f;
      float pw = 0, pr = 0, pi = 0;
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const size_t at = (size_t)v * dim + (b + q * sT);
        float2 o = acc[q][v].value();
        if (fused) {  // w' = sigma_j H q_j - beta_j sigma_{j-1} q_{j-1} over q_{j-1}; <q_j|w'>, <q_j|u>
          o.x *= sg;
          o.y *= sg;
          if (!a.first) {
            const float2 qp = __ldcs(y + at);
            o.x -= bsp * qp.x;
            o.y -= bsp * qp.y;
          }
          const float2 xv = own[(q * V + v) * P + tid], uv = __ldcs(u + at);
          pw += xv.x * o.x + xv.y * o.y;
          pr += xv.x * uv.x + xv.y * uv.y;
          pi += xv.x * uv.y - xv.y * uv.x;
        }
        __stcs(y + at, o);
      }
      if (fused) {
        sacc[(v * 3 + 0) * P + tid] += pw;
        sacc[(v * 3 + 1) * P + tid] += pr;
        sacc[(v * 3 + 2) * P + tid] += pi;
      }
    }
  }
  if (!fused) return;
  if (cur >= 0) flush(cur);
  __threadfence();
  __syncthreads();
  if (tid == 0) is_last = (atomicAdd(a.counter, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  LaunchArgs f = a;
  f.n_inst = nvec;
  f.R = 1;
  f.mode = kModeApply;
  finalize(f, insts);
  if (tid == 0) *a.counter = 0u;
}

template <int Q, int V, int NTMAX, int MINB>
const void* tile_fn() {
  return (const void*)tile_gather_kernel<Q, V, NTMAX, MINB>;
}

// tiles of up to 160 and 256 bases, two or three CTAs an SM
template <int P, int MINB>
const void* tile_pick_p(int Q, int V) {
  if (Q == 2 && V == 4) return tile_fn<2, 4, P, MINB>();
  if (Q == 3 && V == 4) return tile_fn<3, 4, P, MINB>();
  if (Q == 4 && V == 4) return tile_fn<4, 4, P, 2>();
  if (Q == 2 && V == 2) return tile_fn<2, 2, P, MINB>();
  if (Q == 3 && V == 2) return tile_fn<3, 2, P, MINB>();
  if (Q == 4 && V == 2) return tile_fn<4, 2, P, MINB>();
  if (Q == 5 && V == 2) return tile_fn<5, 2, P, MINB>();
  if (Q == 6 && V == 2) return tile_fn<6, 2, P, MINB>();
  return nullptr;
}
const void* tile_pick(int Q, int V, int L) {
  if (L > 256) return nullptr;
  return L <= 160 ? tile_pick_p<160, 3>(Q, V) : tile_pick_p<256, 2>(Q, V);
}

size_t tile_smem(const TilePlan& p, int tab_reals) {
  const int P = p.L <= 160 ? 160 : 256;
  return (((size_t)tab_reals * 4 + 15) & ~size_t(15)) + (size_t)P * ((size_t)2 * p.Q * p.V * 8 + p.V * 3 * 4 + p.nl * 12);
}

}  // namespace

int make_tile(TilePlan& p, int tab_reals) {
  const void* k = tile_pick(p.Q, p.V, p.L);
  if (!k) return 0;
  p.threads = (p.L + 31) & ~31;
  p.smem = tile_smem(p, tab_reals);
  if (p.smem > kTileSmem) return 0;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTileSmem) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p.per_sm, k, p.threads, p.smem) != cudaSuccess || p.per_sm < 1) return 0;
  return 1;
}

// a: groups as instances (a.n_inst, a.tile_start over the tiles of L bases), a.inst one a vector
int launch_tile(const LaunchArgs& a, const TilePlan& p, int R, int grid, void* stream) {
  const void* k = tile_pick(p.Q, p.V, p.L);
  if (!k || a.mode != kModeApply || (a.inline_one && (a.fused_step || a.tiles_per_vg < 1))) return (int)cudaErrorInvalidValue;
  int L = p.L, nl = p.nl;
  void* args[] = {const_cast<LaunchArgs*>(&a), &L, &nl, &R};
  return (int)cudaLaunchKernel(k, dim3(grid), dim3(p.threads), args, p.smem, reinterpret_cast<cudaStream_t>(stream));
}

}  // namespace ftlm
