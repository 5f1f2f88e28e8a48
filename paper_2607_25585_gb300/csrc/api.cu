// C ABI of the FTLM library (include/ftlm.h): system objects, the H.v, u.S
// and start-block entry points, and the FTLM driver (arxiv 2607.25585,
// Eqs. 4-5 and Sec. II.C): start block, M Lanczos steps captured in one CUDA
// graph, then the host eigensolve and Boltzmann sums.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <map>
#include <memory>
#include <mutex>
#include <new>
#include <shared_mutex>
#include <string>
#include <tuple>
#include <vector>

#include "ftlm_internal.h"

using namespace ftlm;

namespace {

thread_local std::string g_err;

ftlm_status fail(ftlm_status s, const std::string& m) {
  g_err = m;
  return s;
}

#define CK(call)                                                                                  \
  do {                                                                                            \
    cudaError_t e__ = (call);                                                                     \
    if (e__ != cudaSuccess) {                                                                     \
      cudaGetLastError();                                                                         \
      return fail(e__ == cudaErrorMemoryAllocation ? FTLM_ERR_OUT_OF_MEMORY : FTLM_ERR_CUDA,      \
                  std::string(#call) + ": " + cudaGetErrorString(e__));                           \
    }                                                                                             \
  } while (0)

#define CKI(expr)                                                                                  \
  do {                                                                                             \
    int e__ = (expr);                                                                              \
    if (e__ != 0) {                                                                                \
      cudaGetLastError();                                                                          \
      return fail(FTLM_ERR_CUDA, std::string(#expr) + ": " + cudaGetErrorString((cudaError_t)e__)); \
    }                                                                                              \
  } while (0)

struct DevBuf {
  void* p = nullptr;
  size_t bytes = 0;
  void release() {
    if (p) cudaFree(p);
    p = nullptr;
    bytes = 0;
  }
  cudaError_t ensure(size_t b) {
    if (bytes >= b && p) return cudaSuccess;
    release();
    cudaError_t e = cudaMalloc(&p, b);
    if (e == cudaSuccess) bytes = b;
    else p = nullptr, cudaGetLastError();  // (reported here: the caller's next CUDA call must not find it)
    return e;
  }
};

}  // namespace

// ---------------------------------------------------------------------------
// system object
// ---------------------------------------------------------------------------
struct ftlm_system {
  HostSystem hs;
  int device = 0;
  DevBuf tab_f, tab_d;   // coupling tables, float and double
  DevBuf stride, q;
  cudaStream_t own_stream = nullptr;  // runs capture and launch their graphs here
  cudaEvent_t ev_in = nullptr, ev_out = nullptr;  // order own_stream after / before the caller's stream
  uint64_t id = 0;       // unique per system
  uint64_t gen = 0;      // bumped whenever the workspace is reallocated
  DevBuf A, B, U, scal;  // Lanczos workspace: two vector blocks, the observable block, scalars
  DevBuf Hq;             // H q_j when the gather and the step epilogue are separate launches
  DevBuf ep, ecnt, esc;  // start-block scratch: partials, arrival counter, scalars
  DevBuf Vs, Wc, Od;     // symmetric runs: stored Lanczos vectors, partial sums of O, O matrices
  DevBuf Ws;             // symmetric runs: u.S of the stored vectors (when it fits)
  DevBuf Gre;            // re-orthogonalised runs: <q_k|w_r> coefficients [R][M] complex
  DevBuf Ta, Tb;         // ftlm_apply_h on spin-1/2 blocks: x and H x in the vector-major layout
  DevBuf Tw, Ts;         // its rotated-basis blocks for one vector (more: rW) and the vectors' statistics
  DevBuf ut[2];          // per-unit coefficient tables of the one-pass vector-major gather, [c64]
  int ut_K[2] = {0, 0};  // the cube size each was built for
  cudaEvent_t ev_apply = nullptr;  // recorded after the last use of Ta, Tb
  std::unique_ptr<RotDirs> rot;  // the rotated-basis H.v's directions, if the system has any
  DevBuf rD[2];          // its diagonal tables [K + 1][dim] and phases, [c64]
  cudaEvent_t ev_rot[2] = {nullptr, nullptr};  // recorded after they were written, on whichever stream did
  DevBuf rW, rpart;      // its intermediate blocks (also of products of several vectors); partial sums and counters
  DevBuf rows[2];        // stored rows of a small system, [c64]: values, columns, counts
  cudaEvent_t ev_rows[2] = {nullptr, nullptr};  // recorded after they were written, on whichever stream did
  bool rows_done[2] = {false, false};           // that event has been seen complete
  bool rows_never[2] = {false, false};          // there was no room for them: the gathers run from then on
  size_t row_bound = 0;                         // entries of a row at most
  double row_entries = 0;                       // on average
  int row_pairs = 0;                            // coupled pairs
  std::mutex rows_mu;
  bool apply_used = false;
  std::mutex apply_mu;   // the blocks, event and tables that products use; a run holds it only to look at them
  std::mutex mu;
  std::shared_mutex use;  // shared: a call that uses the system's blocks; exclusive: giving optional ones back
};

namespace {

std::mutex g_live_mu;
std::vector<ftlm_system*> g_live;  // every system that has not been destroyed

// Shared: a run's capture in progress; exclusive: a wait for the whole device, which
// CUDA refuses while any stream is being captured.
std::shared_mutex g_capture;
cudaError_t wait_for_device() {
  std::unique_lock<std::shared_mutex> lk(g_capture);
  return cudaDeviceSynchronize();
}

std::mutex g_mu;
uint64_t g_next_id = 1;
size_t g_prepared_smem = 0;

// Asynchronous entry points run on the caller's stream; NULL is the CUDA
// default (legacy) stream.
cudaStream_t pick_stream(const ftlm_system*, void* st) { return reinterpret_cast<cudaStream_t>(st); }

int vchunk(int c64, int R) { return (c64 && R % 2 == 0) ? 2 : 1; }
int max_vectors(int c64) { return c64 ? 512 : 256; }

ftlm_status prepare_smem(size_t smem) {
  std::lock_guard<std::mutex> lk(g_mu);
  if (smem <= g_prepared_smem) return FTLM_OK;
  CKI(prepare_rows_kernels(smem));
  g_prepared_smem = smem;
  return FTLM_OK;
}

// ---- launch shapes and the autotuner ----------------------------------------

struct ShapeKey {
  int n, qmax, R, c64;
  long long dim;
  bool operator<(const ShapeKey& o) const {
    return std::tie(n, qmax, R, c64, dim) < std::tie(o.n, o.qmax, o.R, o.c64, o.dim);
  }
};
std::map<ShapeKey, Shape> g_shapes;

// a launch shape set by ftlm_tune_shape or the autotuner for this system shape
bool has_shape_override(const ftlm_system* s, int R, int c64) {
  ShapeKey key{s->hs.n, s->hs.qmax, R, c64, (long long)s->hs.dim};
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_shapes.find(key);
  return it != g_shapes.end() && !it->second.plain;
}

// the rotated-basis H.v may run: no shape was set, or the autotuner found it the fastest
bool rot_allowed(const ftlm_system* s, int R, int c64) {
  ShapeKey key{s->hs.n, s->hs.qmax, R, c64, (long long)s->hs.dim};
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_shapes.find(key);
  return it == g_shapes.end() || it->second.rot;
}

Shape shape_for(int R, int c64, int threads_target, int tile_factor) {
  const int V = vchunk(c64, R);
  const int C = R / V;
  Shape sh;
  sh.threads = C * std::max(1, threads_target / C);
  const int rows_pass = sh.threads / C;
  int rows = std::max(rows_pass, (16384 / std::max(1, R)) * tile_factor);
  sh.rows_per_tile = ((rows + rows_pass - 1) / rows_pass) * rows_pass;
  sh.ctas_per_sm = 0;  // from the occupancy calculator
  return sh;
}

Shape default_shape(int R, int c64) { return shape_for(R, c64, 256, 1); }

InstDesc base_desc(const ftlm_system* s, int c64) {
  InstDesc d;
  const HostSystem& hs = s->hs;
  d.tab = c64 ? s->tab_f.p : s->tab_d.p;
  d.stride = reinterpret_cast<const long long*>(s->stride.p);
  d.q = reinterpret_cast<const int*>(s->q.p);
  d.dim = (long long)hs.dim;
  d.n = hs.n;
  d.all_half = hs.all_half ? 1 : 0;
  d.lay = hs.lay;
  return d;
}

SdirArgs sdir_args(const ftlm_system* s, int c64, int R, const void* x, void* y) {
  SdirArgs a;
  const InstDesc d = base_desc(s, c64);
  a.tab = d.tab;
  a.lay = d.lay;
  a.q = d.q;
  a.n = d.n;
  a.dim = d.dim;
  a.R = R;
  a.x = x;
  a.y = y;
  return a;
}

struct HalfPlan {
  bool on = false;
  bool vm = false;  // vector-major kernel: R instances of one vector each (nvg = R, Rg = 1)
  bool hybrid = false;  // vector-major two-pass form
  int real_pm = 0;
  int min_blocks = 2;
  int passes = 1;  // > 1: one launch per pass, cubes covering all bits
  int K = 3, Rg = 1, threads = 256, rows_per_tile = 0, grid = 0, nvg = 0, tiles_per_vg = 0;
  size_t smem = 0;
  int stream_rows = 0, stream_tiles_per_vg = 0, stream_grid = 0;  // vector-major streaming launches
  long long dim = 0;
};

// Rotated-basis H.v of a run (hv_rot.cu): tiles of 2^T values, K directions, W
// blocks for `group` vectors at a time.
struct RotPlan {
  bool on = false;
  int T = 0, K = 0, group = 1;
};

struct Plan {
  int c64 = 0, R = 0, V = 1, C = 1;
  RotPlan rot;
  Shape sh;
  int grid = 0;
  size_t smem = 0;
  LaunchArgs base;
  std::vector<int> tile_start;
  HalfPlan half;  // spin-1/2 kernel for the H.v modes, when applicable
  int storedV = 0;  // > 0: H.v of vector-major runs from stored rows, that many vectors a group
  int small = 0;    // > 0: the whole run in one launch, clusters of that many CTAs
  int wideV = 0;  // general kernel: H.v with 4 or 8 complex64 vectors per thread (0 = off)
  // vector-major general plan (any spins, several systems): every vector of a
  // run contiguous; the streaming modes see one instance per (system, vector),
  // H.v runs rows_vm_kernel over groups of gvm_V vectors of one system
  bool gen_vm = false;
  int gvm_V = 1, gvm_groups = 0, gvm_ntiles = 0, gvm_rows = 0, gvm_grid = 0;
  int gvm_cube = 0;  // > 0: cube_gather_kernel with the top site's 2s+1 rows per thread
  size_t gvm_smem = 0;
  TilePlan tile;  // V > 0: that H.v over tiles of low sites (hv_tile.cu; gvm_cube is its Q)
  std::vector<int> tile_start_g;  // prefix sum of H.v tiles over the groups
};

// the run keeps each Lanczos vector contiguous
bool plan_vmaj(const Plan& pl) { return pl.half.vm || pl.gen_vm; }

int largest_divisor_at_most(int R, int cap) {
  for (int g = std::min(R, cap); g >= 1; --g)
    if (R % g == 0) return g;
  return 1;
}

// Spin-1/2 register-cube launch: K cube bits, Rg vectors per group, tile of
// rows_factor cubes per slot.
bool make_half(const ftlm_system* s, int R, int c64, int K, int Rg, int rows_factor, bool multipass, HalfPlan& h,
               int min_blocks = 2) {
  const HostSystem& hs = s->hs;
  if (!hs.all_half || hs.n < K + 2 || K < 2 || K > 4 || Rg < 1 || Rg > R) return false;
  h = HalfPlan();
  h.K = K;
  h.Rg = Rg;
  h.passes = multipass ? (hs.n + K - 1) / K : 1;
  h.min_blocks = multipass ? 1 : (min_blocks > 2 ? 3 : 2);
  h.real_pm = hs.real_pm ? 1 : 0;
  const int slots = std::max(1, 256 / Rg);
  h.threads = slots * Rg;
  long long rows = (long long)slots * (1ll << K) * rows_factor;
  rows = std::min<long long>(rows, (long long)hs.dim);
  rows = std::max<long long>(rows, 1ll << K);
  h.rows_per_tile = (int)rows;
  h.nvg = (R + Rg - 1) / Rg;
  h.tiles_per_vg = (int)(((long long)hs.dim + rows - 1) / rows);  // the last tile may be ragged
  const long long ntiles = (long long)h.tiles_per_vg * h.nvg;
  if (ntiles > (1ll << 30)) return false;
  h.smem = half_smem_bytes(hs.n, K, h.rows_per_tile, h.threads);
  if (h.smem > 200 * 1024) return false;
  if (prepare_half_kernels(std::max<size_t>(h.smem, 48 * 1024)) != 0) return false;
  const int per_sm = half_max_ctas_per_sm(K, c64, h.threads, h.smem, h.min_blocks, h.passes > 1, R);
  h.grid = (int)std::max<long long>(1, std::min<long long>(ntiles, (long long)std::max(1, device_sm_count()) * per_sm));
  h.on = true;
  return true;
}

// Vector-major spin-1/2 launch: K cube bits above the 5 lane bits, tiles of
// 8 warps x rows_factor slabs of 2^(5+K) rows, R tiles ranges (one per vector).
bool make_vm(const ftlm_system* s, int R, int c64, int K, int rows_factor, int min_blocks, bool multipass,
             HalfPlan& h, bool hybrid = false) {
  const HostSystem& hs = s->hs;
  if (!hs.all_half || K < 3 || K > 4 || hs.n < kVmLaneBits + K || rows_factor < 1) return false;
  if (hybrid && hs.n < kVmLaneBits + 2 * K) return false;  // the two cubes must not overlap
  if (hs.dim >= (1ull << 31)) return false;  // 32-bit element indices
  h = HalfPlan();
  h.vm = true;
  h.K = K;
  h.Rg = 1;
  h.passes = hybrid ? 2 : (multipass ? (hs.n - kVmLaneBits + K - 1) / K : 1);  // cubes cover bits [5, n)
  h.hybrid = hybrid;
  // 1: one 512-thread CTA per SM; 2 or 3: 256-thread CTAs (3 only in one pass)
  h.min_blocks = min_blocks == 1 ? 1 : (h.passes > 1 ? 2 : (min_blocks > 2 ? 3 : 2));
  h.real_pm = hs.real_pm ? 1 : 0;
  h.threads = h.min_blocks == 1 ? 512 : 256;
  const long long slab = 1ll << (kVmLaneBits + K);
  long long rows = (long long)(h.threads / 32) * slab * rows_factor;
  rows = std::min<long long>(rows, (long long)hs.dim);  // dim and rows are powers of two >= slab
  h.rows_per_tile = (int)rows;
  h.nvg = R;
  h.dim = (long long)hs.dim;
  h.tiles_per_vg = (int)((long long)hs.dim / rows);  // per vector and pass
  const long long ntiles = (long long)h.tiles_per_vg * R * h.passes;
  if (ntiles > (1ll << 30)) return false;
  h.smem = vm_smem_bytes(hs.n, K, h.threads, h.passes, c64);
  if (h.smem > 200 * 1024) return false;
  if (prepare_vm_kernels(std::max<size_t>(h.smem, 48 * 1024)) != 0) return false;
  // the register budget allows min_blocks CTAs per SM: keep only their shared memory, the rest is L1
  if (set_vm_carveout(K, c64, h.passes > 1, h.min_blocks, h.smem, h.min_blocks) != 0) return false;
  const int per_sm = vm_max_ctas_per_sm(K, h.min_blocks, c64, h.threads, h.smem, h.passes > 1);
  const long long sms = std::max(1, device_sm_count());
  h.grid = (int)std::max<long long>(1, std::min<long long>(ntiles, sms * per_sm));
  h.stream_rows = (int)std::min<long long>(16384, (long long)hs.dim);
  h.stream_tiles_per_vg = (int)((long long)hs.dim / h.stream_rows);
  // two 256-thread CTAs per SM keep enough loads in flight for HBM and give
  // the last CTA half the partials of four (measured: 2.7 ms less per
  // 200-step run at d = 2^20, R = 64; one CTA per SM was 15 ms more)
  h.stream_grid = (int)std::max<long long>(1, std::min<long long>((long long)h.stream_tiles_per_vg * R, sms * 2));
  h.on = true;
  return true;
}

// General row-kernel launch over the instances `sys` (R vectors each).
ftlm_status make_general(const std::vector<ftlm_system*>& sys, int R, int c64, Plan& pl) {
  pl.V = vchunk(c64, R);
  pl.C = R / pl.V;
  LaunchArgs a;
  a.R = R;
  a.C = pl.C;
  a.rows_per_tile = pl.sh.rows_per_tile;
  int tab = 0, maxn = 0;
  pl.tile_start.assign(1, 0);
  for (auto* s : sys) {
    tab = std::max(tab, s->hs.lay.total);
    maxn = std::max(maxn, s->hs.n);
    const long long tiles = ((long long)s->hs.dim + a.rows_per_tile - 1) / a.rows_per_tile;
    if (pl.tile_start.back() + tiles > (1ll << 30)) return fail(FTLM_ERR_UNSUPPORTED, "too many tiles");
    pl.tile_start.push_back(pl.tile_start.back() + (int)tiles);
  }
  a.tab_reals = tab;
  a.max_n = maxn;
  a.n_inst = (int)sys.size();
  a.ntiles = pl.tile_start.back();
  pl.smem = rows_smem_bytes(a, c64, pl.sh.threads);
  if (pl.smem > 227 * 1024) return fail(FTLM_ERR_UNSUPPORTED, "coupling tables do not fit in shared memory");
  ftlm_status ps = prepare_smem(std::max<size_t>(pl.smem, 48 * 1024));
  if (ps != FTLM_OK) return ps;
  // H.v with more vectors per thread: the matrix elements of a row are computed
  // once for 4 or 8 vectors instead of 2 (complex64; the same tiles)
  pl.wideV = 0;
  if (c64 && R >= 4 && R % 4 == 0) {
    const int Vw = R % 8 == 0 ? 8 : 4, Cw = R / Vw;
    // (H.v keeps no reduction space in shared memory, so pl.smem covers it)
    if (pl.sh.threads % Cw == 0 && pl.sh.rows_per_tile % (pl.sh.threads / Cw) == 0) pl.wideV = Vw;
  }
  // the grid fills the SMs with the kernel that carries H.v.  The wide H.v
  // kernel runs two CTAs per SM while a system's block fits in the L2
  // (its gathers are served on chip and more L1 per tile pays), and as many as
  // fit once the block spills to HBM (the gathers' latency wants the warps).
  int per_sm = pl.sh.ctas_per_sm > 0 ? pl.sh.ctas_per_sm : rows_max_ctas_per_sm(c64, pl.sh.threads, pl.smem, pl.wideV);
  if (pl.sh.ctas_per_sm <= 0 && pl.wideV) {
    long long maxdim = 0;
    for (auto* s : sys) maxdim = std::max(maxdim, (long long)s->hs.dim);
    const long long block_bytes = maxdim * R * 8;
    if (block_bytes <= device_l2_bytes()) per_sm = std::min(per_sm, 2);
  }
  const int sms = std::max(1, device_sm_count());
  pl.grid = std::max(1, std::min(a.ntiles, sms * per_sm));
  pl.base = a;
  return FTLM_OK;
}

// The tile plan of the systems (all with top radix Q), complex64: the tile's
// low sites have to have the same radices in every system.
bool plan_tile(const std::vector<ftlm_system*>& sys, int R, int Q, TilePlan& p) {
  if (R < 2) return false;
  int common = sys[0]->hs.n - 1, tab = 0;
  for (auto* s : sys) {
    if (s->hs.dim < (1u << 15) || s->hs.dim >= (1ull << 31)) return false;
    common = std::min(common, s->hs.n - 1);
    tab = std::max(tab, s->hs.lay.total);
    for (int i = 0; i < common; ++i)
      if (s->hs.q[i] != sys[0]->hs.q[i]) common = i;
  }
  p = TilePlan();
  p.Q = Q;
  p.V = Q >= 5 || R < 4 ? 2 : 4;  // 2 x 5 or 4 x 3 values a thread fill its registers
  p.L = 1;
  while (p.nl < common && p.L * sys[0]->hs.q[p.nl] <= 256) p.L *= sys[0]->hs.q[p.nl++];
  return p.L >= 32 && make_tile(p, tab);
}

// allow_vm: the caller keeps its Lanczos block vector-major (ftlm_run); for
// row-major blocks a vector-major shape falls back to the row-major cube kernel.
ftlm_status make_plan(const std::vector<ftlm_system*>& sys, int R, int c64, Plan& pl, const Shape* force = nullptr,
                      bool allow_vm = false) {
  pl.c64 = c64;
  pl.R = R;
  const ftlm_system* big = sys[0];
  for (auto* s : sys)
    if (s->hs.dim > big->hs.dim) big = s;
  if (force) {
    pl.sh = *force;
  } else {
    ShapeKey key{big->hs.n, big->hs.qmax, R, c64, (long long)big->hs.dim};
    std::lock_guard<std::mutex> lk(g_mu);
    auto it = g_shapes.find(key);
    pl.sh = it != g_shapes.end() ? it->second : default_shape(R, c64);
  }
  pl.half.on = false;
  if (sys.size() == 1 && pl.sh.half_K > 0 && pl.sh.half_vm && allow_vm &&
      make_vm(sys[0], R, c64, pl.sh.half_K, pl.sh.half_rows, pl.sh.half_min_blocks, pl.sh.half_multipass != 0,
              pl.half, pl.sh.half_hybrid != 0)) {
    // the streaming modes see R one-vector instances of the same system
    const Shape keep = pl.sh;
    pl.sh = default_shape(1, c64);
    ftlm_status gs = make_general(std::vector<ftlm_system*>(R, sys[0]), 1, c64, pl);
    pl.sh.half_K = keep.half_K;
    pl.sh.half_vm = 1;
    return gs;
  }
  if (sys.size() == 1 && allow_vm && !force && pl.sh.half_K == 0 && !pl.sh.explicit_general) {
    // default for runs on spin-1/2 systems: the vector-major single-pass gather
    const int K = c64 ? 4 : 3;  // complex128 cubes of 16 rows spill at 128 registers
    // one 512-thread CTA per SM (one copy of the tables, more L1), tiles of 2 units per warp
    if (make_vm(sys[0], R, c64, K, 2, 1, false, pl.half)) {
      pl.sh = default_shape(1, c64);
      ftlm_status gs = make_general(std::vector<ftlm_system*>(R, sys[0]), 1, c64, pl);
      pl.sh.half_K = K;
      pl.sh.half_vm = 1;
      return gs;
    }
  }
  // runs on other systems and batches: the vector-major general gather by
  // default when it can hold the top site's rows as a register cube (every
  // system with the same top spin, a group size dividing R), or when the
  // largest system's block of R vectors fits in L2; else the row-major one.
  // Measured on GB300: with one row a thread the vector-major gather is 24 %
  // faster than the row-major one on s = 1 chains whose largest block is
  // 68 MB but 5 % slower on a 150 MB mixed-spin block, where the cube form is
  // 17 % faster than both.  An autotuned or forced shape decides for itself.
  int Qtop = sys[0]->hs.n >= 2 ? sys[0]->hs.q.back() : 0;
  for (auto* s : sys)
    if (s->hs.n < 2 || s->hs.q.back() != Qtop) Qtop = 0;
  // the cube's group size: the default for the top spin, else 4, whichever
  // has a kernel and divides R (0: none)
  auto cube_group = [&](int want) {
    if (!Qtop) return 0;
    if (want > 0) return (cube_vectors(Qtop, c64, want) && R % want == 0) ? want : 0;
    for (int v : {cube_vectors(Qtop, c64), 4})
      if (v > 0 && cube_vectors(Qtop, c64, v) && R % v == 0) return v;
    return 0;
  };
  const int Vdef = cube_group(0);
  TilePlan tile;
  const bool tiled = c64 && allow_vm && !force && pl.sh.general_vm < 0 && pl.sh.half_K == 0 && !pl.sh.explicit_general &&
                     Qtop && plan_tile(sys, R, Qtop, tile);
  const bool gvm_fits = (long long)big->hs.dim * R * (c64 ? 8 : 16) <= device_l2_bytes();
  const bool gvm_default = gvm_fits || Vdef > 0 || tiled;
  const bool want_gvm = pl.sh.general_vm == 1 || (pl.sh.general_vm < 0 && !force && gvm_default);
  if (allow_vm && want_gvm && pl.sh.half_K == 0 && !pl.sh.explicit_general) {
    int V = 1;
    for (int v : {8, 4, 2, 1})
      if (R % v == 0 && rows_vm_supported(v, c64)) {
        V = v;
        break;
      }
    // the register cube along the top site when every system has the same top
    // spin and a kernel exists for it and for a group size dividing R
    const int Q = Qtop;
    const int Vc = (Q && pl.sh.gvm_cube != 0) ? cube_group(std::max(0, pl.sh.gvm_cube)) : 0;
    const bool cube = Vc > 0 || tiled;
    if (tiled) V = tile.V;
    else if (cube) V = Vc;
    std::vector<ftlm_system*> vecs;  // one instance per (system, vector), system-major
    for (auto* s : sys)
      for (int k = 0; k < R; ++k) vecs.push_back(s);
    const Shape keep = pl.sh;
    pl.sh = default_shape(1, c64);
    ftlm_status gs = make_general(vecs, 1, c64, pl);
    if (gs != FTLM_OK) return gs;
    pl.sh.half_K = keep.half_K;
    pl.gen_vm = true;
    pl.gvm_V = V;
    pl.gvm_cube = cube ? Q : 0;
    // 1024 rows: four a thread of a 256-thread CTA; with the cube, 256 bases
    // (one a thread: the CTAs then share the neighbourhoods they gather in L2)
    pl.gvm_rows = keep.gvm_rows > 0 && keep.general_vm == 1 ? keep.gvm_rows : (cube ? 256 : 1024);
    if (tiled) {
      pl.tile = tile;
      pl.gvm_rows = tile.L;
    }
    pl.tile_start_g.assign(1, 0);
    for (auto* s : sys)
      for (int g = 0; g < (R + V - 1) / V; ++g) {
        const long long rows = cube ? (long long)s->hs.dim / Q : (long long)s->hs.dim;  // bases, or rows
        const long long tiles = (rows + pl.gvm_rows - 1) / pl.gvm_rows;
        if (pl.tile_start_g.back() + tiles > (1ll << 30)) return fail(FTLM_ERR_UNSUPPORTED, "too many tiles");
        pl.tile_start_g.push_back(pl.tile_start_g.back() + (int)tiles);
      }
    pl.gvm_groups = (int)pl.tile_start_g.size() - 1;
    pl.gvm_ntiles = pl.tile_start_g.back();
    int per_sm = 1;
    if (tiled) {
      per_sm = tile.per_sm;
    } else if (cube) {
      pl.gvm_smem = gather_smem_bytes(pl.base, c64, 256);  // tables and per-thread columns, no reduction space
      CKI(prepare_cube(Q, V, c64, std::max<size_t>(pl.gvm_smem, 48 * 1024)));
      per_sm = cube_ctas_per_sm(Q, V, c64, 256, pl.gvm_smem);
    } else {
      pl.gvm_smem = pl.smem;  // the same tables and per-thread columns as the streaming plan
      CKI(prepare_rows_vm(V, c64, std::max<size_t>(pl.gvm_smem, 48 * 1024)));
      per_sm = rows_vm_ctas_per_sm(V, c64, 256, pl.gvm_smem);
    }
    pl.gvm_grid = std::max(1, std::min(pl.gvm_ntiles, std::max(1, device_sm_count()) * per_sm));
    return FTLM_OK;
  }
  ftlm_status gs = make_general(sys, R, c64, pl);
  if (gs != FTLM_OK) return gs;
  if (sys.size() == 1 && pl.sh.half_K > 0 && !pl.sh.half_vm)
    make_half(sys[0], R, c64, pl.sh.half_K, pl.sh.Rg, pl.sh.half_rows, pl.sh.half_multipass != 0, pl.half,
              pl.sh.half_min_blocks);
  else if (sys.size() == 1 && (!force || pl.sh.half_vm) && !pl.sh.explicit_general && sys[0]->hs.all_half)
    make_half(sys[0], R, c64, 3, largest_divisor_at_most(R, 16), 4, false, pl.half);
  return FTLM_OK;
}

// Launches one mode of the plan: the spin-1/2 kernel for H.v modes when the
// plan has it, the general row kernel otherwise.
int launch_plan(const Plan& pl, LaunchArgs a, void* st) {
  if (pl.gen_vm && a.mode == kModeApply) {  // the groups' tile list follows the instances' in the same buffer
    a.n_inst = pl.gvm_groups;
    a.ntiles = pl.gvm_ntiles;
    a.rows_per_tile = pl.gvm_rows;
    if (!a.inline_one) a.tile_start += pl.base.n_inst + 1;
    if (pl.tile.V) return launch_tile(a, pl.tile, pl.R, pl.gvm_grid, st);
    if (pl.gvm_cube) return launch_cube(a, pl.gvm_cube, pl.gvm_V, pl.c64, pl.gvm_grid, 256, pl.gvm_smem, st);
    return launch_rows_vm(a, pl.gvm_V, pl.c64, pl.gvm_grid, 256, pl.gvm_smem, st);
  }
  if (pl.half.on && pl.half.vm && a.mode == kModeStep) {
    a.rows_per_tile = pl.half.stream_rows;
    a.tiles_per_vg = pl.half.stream_tiles_per_vg;
    a.n_inst = pl.half.nvg;
    a.ntiles = pl.half.stream_tiles_per_vg * pl.half.nvg;
    a.inline_one = 0;
    return launch_vm_stream(a, pl.c64, pl.half.stream_grid, st);
  }
  if (pl.half.on && pl.half.vm && a.mode == kModeApply) {  // a.inst: R one-vector instances
    a.rows_per_tile = pl.half.rows_per_tile;
    a.tiles_per_vg = pl.half.tiles_per_vg;
    a.nvg = pl.half.nvg;
    a.n_inst = pl.half.nvg;
    a.ntiles = pl.half.tiles_per_vg * pl.half.nvg;
    a.real_pm = pl.half.real_pm;
    a.min_blocks = pl.half.min_blocks;
    // one vector, or a regular block (vm_stride): the descriptor by value
    a.inline_one = (a.inline_one && (pl.half.nvg == 1 || a.vm_stride)) ? 1 : 0;
    a.pass_stride = (long long)pl.half.nvg * pl.half.dim;
    if (pl.half.hybrid) {  // two launches: the bottom cube (one-pass kernel), then the top cube adds its terms
      LaunchArgs b = a;
      b.single_pass = 1;
      b.hybrid = 1;
      b.npass = 1;
      b.gather_alpha = 0;
      b.ntiles = pl.half.tiles_per_vg * pl.half.nvg;
      const int e = launch_vm(b, pl.half.K, pl.half.min_blocks, pl.c64, pl.half.grid, pl.half.threads, pl.half.smem, st);
      if (e) return e;
      a.single_pass = 0;
      a.hybrid = 2;
      a.npass = 1;
      a.ntiles = pl.half.tiles_per_vg * pl.half.nvg;
      return launch_vm(a, pl.half.K, pl.half.min_blocks, pl.c64, pl.half.grid, pl.half.threads, pl.half.smem, st);
    }
    a.single_pass = pl.half.passes == 1 ? 1 : 0;
    a.npass = pl.half.passes;  // pass p writes y + p * R * d (vector-major blocks)
    a.hybrid = 0;
    a.ntiles = pl.half.tiles_per_vg * pl.half.nvg * pl.half.passes;
    return launch_vm(a, pl.half.K, pl.half.min_blocks, pl.c64, pl.half.grid, pl.half.threads, pl.half.smem, st);
  }
  const bool half = pl.half.on && !pl.half.vm &&
                    (a.mode == kModeApply || (a.mode == kModeLanczos && pl.half.passes == 1));
  if (half) {
    a.rows_per_tile = pl.half.rows_per_tile;
    a.Rg = pl.half.Rg;
    a.nvg = pl.half.nvg;
    a.tiles_per_vg = pl.half.tiles_per_vg;
    a.ntiles = pl.half.tiles_per_vg * pl.half.nvg;
    a.real_pm = pl.half.real_pm;
    a.min_blocks = pl.half.min_blocks;
    const int K = pl.half.K;
    const int n = pl.base.max_n;
    if (pl.half.passes == 1) {
      a.single_pass = 1;
      return launch_half(a, K, pl.c64, pl.half.grid, pl.half.threads, pl.half.smem, st);
    }
    for (int p = 0; p < pl.half.passes; ++p) {  // cubes [min(pK, n-K), +K) cover every bit
      a.cube_lo = std::min(p * K, n - K);
      a.new_lo = p * K;
      a.later_lo = a.cube_lo + K;
      a.first_pass = p == 0;
      a.single_pass = 0;
      const int e = launch_half(a, K, pl.c64, pl.half.grid, pl.half.threads, pl.half.smem, st);
      if (e) return e;
    }
    return 0;
  }
  if (pl.wideV && a.mode == kModeApply) {
    a.C = a.R / pl.wideV;
    return launch_rows_wide(a, pl.wideV, pl.grid, pl.sh.threads, pl.smem, st);
  }
  // the streaming modes need far fewer CTAs than the gathers to saturate HBM,
  // and fewer CTAs means fewer partial sums for the last CTA to add up
  const bool streaming = a.mode == kModeEpilogue || a.mode == kModeUpdate || a.mode == kModeStartNorm ||
                         a.mode == kModeScale || a.mode == kModeStep;
  const int grid = streaming ? std::min(pl.grid, 2 * std::max(1, device_sm_count())) : pl.grid;
  return launch_rows(a, pl.c64, grid, pl.sh.threads, pl.smem, st);
}

// The Lanczos step of the plan runs as the vector-major one-pass gather with
// the step's w' in its epilogue, then the update pass (see enqueue_run).
bool vm_fused_step(const Plan& pl) { return pl.half.on && pl.half.vm && pl.half.passes == 1 && !pl.half.hybrid; }

// The per-unit coefficient tables of the one-pass vector-major gather with K
// cube bits, built once per system (and rebuilt for another K or precision)
// on stream st; their pointer is baked into captured graphs, so a rebuild
// bumps the system's generation.
ftlm_status ensure_unit_tables(ftlm_system* s, int K, int c64, cudaStream_t st) {
  DevBuf& b = s->ut[c64 ? 1 : 0];
  if (b.p && s->ut_K[c64 ? 1 : 0] == K) return FTLM_OK;
  const int n = s->hs.n;
  const long long nunits = (long long)(s->hs.dim >> (kVmLaneBits + K));
  const size_t bytes = (size_t)nunits * vm_unit_table_stride(n, K) * (c64 ? 4 : 8);
  if (b.p) CK(wait_for_device());  // a rebuild: no launch may still read the old tables
  b.release();
  CK(b.ensure(bytes));
  CKI(launch_vm_unit_tables(reinterpret_cast<const double*>(s->tab_d.p), s->hs.lay, n, K, nunits, b.p, c64, st));
  s->ut_K[c64 ? 1 : 0] = K;
  s->gen++;
  return FTLM_OK;
}

// ---- the rotated-basis H.v of spin-1/2 runs ------------------------------------

size_t rot_phase_bytes(int c64) { return (size_t)kRotMaxK * (kRotMaxN + 1) * (c64 ? 8 : 16); }

// Its tables, written once per system and precision (the caller holds apply_mu).
// The stream that wrote them may be another call's -- a run's own stream, which a
// product of one vector does not wait for, nor one after a run that failed before
// its end -- so st waits for the event recorded behind the launches that write.
// ok = false when they do not fit in memory (the gather then runs).
ftlm_status ensure_rot_tables(ftlm_system* s, const RotPlan& rp, int c64, cudaStream_t st, bool& ok) {
  ok = false;
  const size_t d = (size_t)s->hs.dim, real = c64 ? 4 : 8;
  DevBuf& D = s->rD[c64 ? 1 : 0];
  cudaEvent_t& ev = s->ev_rot[c64 ? 1 : 0];
  if (prepare_rot(s->hs.n, c64) != 0) return FTLM_OK;
  if (!ev) CK(cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
  if (!D.p) {
    const size_t bytes = (size_t)(rp.K + 1) * d * real + rot_phase_bytes(c64);
    if (D.ensure(bytes) != cudaSuccess) return cudaGetLastError(), FTLM_OK;
    int e = 0;
    for (int k = 0; k <= rp.K && !e; ++k) {
      RotForm f = s->rot->form[k];
      f.T = k > 0 ? rp.T : 0;
      f.b = rot_run_bits(s->hs.n, c64);
      e = launch_rot_table(f, static_cast<char*>(D.p) + (size_t)k * d * real, c64, st);
    }
    if (!e) e = launch_rot_phases(s->hs.n, *s->rot, static_cast<char*>(D.p) + bytes - rot_phase_bytes(c64), c64, st);
    if (!e) e = (int)cudaEventRecord(ev, st);
    if (e) D.release();
    CKI(e);
  }
  CK(cudaStreamWaitEvent(st, ev, 0));
  ok = true;
  return FTLM_OK;
}

// The intermediate blocks' buffer rW, for holders of the system's mu and apply_mu.
// Products still in flight may read the old one; captured graphs hold its address.
bool grow_rot_blocks(ftlm_system* s, size_t bytes) {
  if (s->rW.bytes >= bytes) return true;
  if (s->apply_used) cudaEventSynchronize(s->ev_apply);
  s->gen++;
  return s->rW.ensure(bytes) == cudaSuccess;
}

size_t rot_block_bytes(const ftlm_system* s, const RotPlan& rp, int c64) {
  return (size_t)rp.group * rp.K * (size_t)s->hs.dim * (c64 ? 8 : 16);
}

// The tables, W blocks and partial sums of a run over R vectors.
ftlm_status ensure_rot(ftlm_system* s, const RotPlan& rp, int R, int c64, cudaStream_t st, bool& ok) {
  ok = false;
  const size_t pbytes = sizeof(double) * 3 * ((size_t)s->hs.dim >> rp.T) * R + sizeof(unsigned) * R;
  std::lock_guard<std::mutex> lk(s->apply_mu);
  bool fits = grow_rot_blocks(s, rot_block_bytes(s, rp, c64));
  if (fits && s->rpart.bytes < pbytes) {
    s->gen++;
    fits = s->rpart.ensure(pbytes) == cudaSuccess;
  }
  return fits ? ensure_rot_tables(s, rp, c64, st, ok) : FTLM_OK;
}

// The rotated-basis plan of a block of R vectors (false: the system has none).
// The W blocks hold K times the group's vectors; a system keeps at most kRotBlocks
// of them, or one vector's: four vectors of 26 sites in one group take 11.0 ms a
// step, in groups of two (4 GB) 11.1, one at a time (2 GB) 11.5.
constexpr size_t kRotBlocks = (size_t)8 << 30;
bool rot_shape(ftlm_system* s, int R, int c64, RotPlan& rp) {
  rp = RotPlan();
  rp.T = rot_tile_bits(s->hs.n, c64);
  if (!s->rot || !rp.T) return false;
  rp.K = s->rot->K;
  const uint64_t per = s->hs.dim * (uint64_t)rp.K * (c64 ? 8 : 16);
  rp.group = (int)std::min<uint64_t>((uint64_t)R, std::max<uint64_t>(1, kRotBlocks / per));
  return true;
}

ftlm_status make_rot(ftlm_system* s, int R, int c64, RotPlan& rp, cudaStream_t st) {
  return rot_shape(s, R, c64, rp) ? ensure_rot(s, rp, R, c64, st, rp.on) : FTLM_OK;
}

RotArgs rot_args(const ftlm_system* s, const RotPlan& rp, int c64) {
  RotArgs a;
  const size_t d = (size_t)s->hs.dim, real = c64 ? 4 : 8;
  const char* D = static_cast<const char*>(s->rD[c64 ? 1 : 0].p);
  a.n = s->hs.n;
  a.T = rp.T;
  a.b = rot_run_bits(s->hs.n, c64);
  a.K = rp.K;
  a.t = s->rot->t;
  a.dim = (long long)d;
  a.D0 = D;
  a.D = D + d * real;
  a.phases = D + (size_t)(rp.K + 1) * d * real;
  return a;
}

// Work enqueued on the stream is being captured (or may not be asked now).
bool stream_captures(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  const bool yes = cudaStreamIsCapturing(st, &cs) != cudaSuccess || cs != cudaStreamCaptureStatusNone;
  cudaGetLastError();
  return yes;
}

// ---- stored rows of small systems -----------------------------------------------

// Rows are stored up to a quarter of L2, where every product reads them from
// there; larger systems have rows enough to fill the chip with the gathers.  But
// where these form coefficients for one or two vectors at a time in FP64, that
// costs more than reading them from HBM: complex128, up to 2 GB for the
// call's n systems then (a product of nine spins 3/2 and 2, 327,680 states, in
// complex128: 1.22 -> 0.29 ms for one vector, 12.6 -> 2.1 ms for eight).  Spin-1/2
// systems have the rotated-basis passes.
constexpr size_t kStoredL2 = 32u << 20;
size_t stored_limit(const ftlm_system* s, int c64, int n = 1) {
  return !s->hs.all_half && !c64 ? std::max(kStoredL2, ((size_t)2 << 30) / n) : kStoredL2;
}

// bytes of the system's stored rows; 0: too many sites for their builder
size_t stored_bytes(const ftlm_system* s, int c64) {
  const size_t S = s->row_bound;
  return S == 0 || s->hs.dim > ((size_t)2 << 30) ? 0 : (size_t)s->hs.dim * (S * (c64 ? 12 : 20) + 4);
}

// Whether a call with `products` products of a vector wants them.
bool stored_fits(const ftlm_system* s, int c64, size_t limit, long long products) {
  const size_t b = stored_bytes(s, c64);
  return b != 0 && b <= (products < 4 ? kStoredL2 : limit);
}

// Whether stored rows are the faster form for so many vectors.  They cost 4.1 ps an
// entry and vector in complex64, the gathers hardly more for many vectors than for
// one: up to 8 vectors the rows are always ahead, then while entries x vectors take
// less than the gathers' latency -- 31 us on spins 1/2 (the transposing route), on
// other spins 45 us and 7.5 us a coupled pair.  Measured at 64 to 16,384 states and 1
// to 256 vectors: 14 spins 1/2, 128 vectors 88 us (gather; 75 now, in rotated bases) against
// 788 us from rows; 8 spins 1, 64 vectors 251 against 114, 256 vectors 257 against 404.
// A run's gathers have no transposes but its steps' rows are cheaper too: up to 2e7
// entries x vectors (12 spins 1/2, eight steps: 32 vectors 515 us against 477, 64: 647 against
// 772; 7 spins 3/2: 8 vectors 576 against 502, 64: 1156 against 1827), in a batch for
// each system by itself (24 chains of 10 spins 1/2, 48 vectors: 7.0 ms against 3.0).  In
// complex128 the gathers form coefficients in FP64 and the rows win throughout.
bool stored_pays(const ftlm_system* s, int c64, int nvec) {
  if (!c64 || nvec <= 8) return true;
  const double latency = s->hs.all_half ? 31.0 : 45.0 + 7.5 * s->row_pairs;
  return 4.1e-6 * s->row_entries * (double)s->hs.dim * nvec <= latency;
}

// Rows of all live systems together, at most: a program may hold hundreds of systems
// (fields, orientations), and the gathers need no memory.  A system that finds no room
// stays with the gathers, so that its repeated calls give the same bits.
constexpr size_t kStoredTotal = (size_t)16 << 30;
std::atomic<size_t> g_stored_total{0};

bool reserve_stored(size_t bytes) {
  size_t t = g_stored_total.load();
  while (t + bytes <= kStoredTotal)
    if (g_stored_total.compare_exchange_weak(t, t + bytes)) return true;
  return false;
}

void release_stored(DevBuf& b) {
  g_stored_total -= b.bytes;
  b.release();
}

// Gives back what the current device's systems keep for speed alone (the
// rotated-basis blocks and tables, stored rows, transposed blocks) where no call is
// using them; true if there was any.
bool give_back() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaGetLastError(), false;
  std::lock_guard<std::mutex> live(g_live_mu);
  bool any = false;
  for (ftlm_system* s : g_live) {
    if (s->device != dev) continue;
    std::unique_lock<std::shared_mutex> lk(s->use, std::try_to_lock);
    if (!lk) continue;
    for (DevBuf* b : {&s->rW, &s->Tw, &s->rD[0], &s->rD[1], &s->Ta, &s->Tb, &s->rows[0], &s->rows[1]}) {
      if (!b->p) continue;
      if (!any && wait_for_device() != cudaSuccess) return cudaGetLastError(), false;  // products may be in flight
      any = true;
      if (b == &s->rows[0] || b == &s->rows[1]) release_stored(*b);
      else b->release();
    }
    s->rows_done[0] = s->rows_done[1] = false;
    s->gen++;  // captured graphs hold their addresses
  }
  return any;
}

// Allocations, event waits and copies of this thread take no part in a capture that
// another thread has open (CUDA's default mode refuses them then, and the capture is
// lost); in this thread's own capture they stay refused.
struct ApartFromCaptures {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeThreadLocal;
  ApartFromCaptures() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~ApartFromCaptures() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// Runs an entry point's body for the systems; where device memory does not suffice,
// gives back what systems keep for speed alone and runs it once more, `lean`: without
// taking such blocks again.  Nothing thrown crosses the C interface.
template <typename Body>
ftlm_status with_memory(ftlm_system* const* sys, int n, Body&& body) {
  ApartFromCaptures apart;
  try {
    for (const bool lean : {false, true}) {
      ftlm_status st;
      {
        std::shared_lock<std::shared_mutex> first;  // (one system: nothing allocated here)
        std::vector<std::shared_lock<std::shared_mutex>> others;
        if (n > 0) first = std::shared_lock<std::shared_mutex>(sys[0]->use);
        for (int k = 1; k < n; ++k) others.emplace_back(sys[k]->use);
        st = body(lean);
      }
      if (st != FTLM_ERR_OUT_OF_MEMORY || lean) return st;
      const std::string what = g_err;
      if (!give_back()) return fail(st, what);
    }
  } catch (const std::bad_alloc&) {
    return fail(FTLM_ERR_OUT_OF_MEMORY, "out of host memory");
  } catch (const std::exception& e) {
    return fail(FTLM_ERR_CUDA, e.what());
  }
  return FTLM_ERR_OUT_OF_MEMORY;
}

// Whether a run over the systems takes stored rows: all of them or none.
bool run_stores(const std::vector<ftlm_system*>& sys, int R, int M, int c64) {
  bool all = true;
  for (const ftlm_system* s : sys) {
    all = all && stored_fits(s, c64, stored_limit(s, c64, (int)sys.size()), (long long)R * M);
    if (c64 && R > 8) all = all && s->row_entries * (double)s->hs.dim * R <= 2e7;  // (see stored_pays)
  }
  return all;
}

// The system's stored rows for work on stream st: written by the first call, on
// its st (not on the system's own stream, which another thread's run may be
// capturing); other streams wait for them.  ok = false: the gathers run -- the
// rows are too large, or beyond L2 for a call of fewer than four products of a
// vector (writing them costs about two), or there was no room for them.  A repeated
// call gives the same bits.  st must not be capturing.
ftlm_status ensure_stored(ftlm_system* s, int c64, size_t limit, long long products, cudaStream_t st, StoredRows& r,
                          bool& ok) {
  ok = false;
  const int k = c64 ? 1 : 0;
  const size_t d = (size_t)s->hs.dim, esz = c64 ? 8 : 16;
  if (!stored_fits(s, c64, limit, products)) return FTLM_OK;
  const size_t S = s->row_bound;
  std::lock_guard<std::mutex> lk(s->rows_mu);
  DevBuf& b = s->rows[k];
  if (s->rows_never[k]) return FTLM_OK;
  if (!s->rows_done[k]) {
    if (!b.p) {
      if (!s->ev_rows[k]) CK(cudaEventCreateWithFlags(&s->ev_rows[k], cudaEventDisableTiming));
      const size_t bytes = stored_bytes(s, c64);
      s->rows_never[k] = !reserve_stored(bytes);
      if (!s->rows_never[k] && b.ensure(bytes) != cudaSuccess) {
        g_stored_total -= bytes;
        s->rows_never[k] = true;
      }
      if (s->rows_never[k]) return FTLM_OK;
      char* p = static_cast<char*>(b.p);
      int e = launch_stored_build(c64 ? s->tab_f.p : s->tab_d.p, s->hs.lay,
                                  reinterpret_cast<const long long*>(s->stride.p), reinterpret_cast<const int*>(s->q.p),
                                  s->hs.n, (int)d, (int)S, reinterpret_cast<int*>(p + d * S * esz), p,
                                  reinterpret_cast<int*>(p + d * S * (esz + 4)), c64, st);
      if (!e) e = (int)cudaEventRecord(s->ev_rows[k], st);
      if (e) release_stored(b);
      CKI(e);
    }
    if (cudaEventQuery(s->ev_rows[k]) == cudaSuccess) s->rows_done[k] = true;
    else CK(cudaStreamWaitEvent(st, s->ev_rows[k], 0));
    cudaGetLastError();  // (not ready is no error)
  }
  const char* p = static_cast<const char*>(b.p);
  r.val = p;
  r.col = reinterpret_cast<const int*>(p + d * S * esz);
  r.cnt = reinterpret_cast<const int*>(p + d * S * (esz + 4));
  r.S = (long long)S;
  ok = true;
  return FTLM_OK;
}

// Vectors a CTA of the stored-row kernels takes: as many as leave the chip enough
// threads (eight a row and group) to hide L2 latency.
int stored_group(uint64_t rows, int R) {
  int V = 4;
  while (V > 1 && (V / 2 >= R || rows * 8 * (uint64_t)((R + V - 1) / V) < 200000)) V /= 2;
  return V;
}

int plan_max_grid(const Plan& pl) {
  return std::max(std::max(pl.grid, pl.gen_vm ? pl.gvm_grid : 0),
                  pl.half.on ? std::max(pl.half.grid, pl.half.stream_grid) : 0);
}

// ---- workspace ----------------------------------------------------------------

size_t scalar_bytes(int R, int M) {
  return sizeof(double) * ((size_t)M * R * 4 + (size_t)(M + 1) * R + R) + sizeof(int) * 2 * (size_t)R + 64;
}

ftlm_status ensure_workspace(ftlm_system* s, int R, int M, int c64) {
  const size_t block = (size_t)s->hs.dim * R * (c64 ? 8 : 16);
  if (s->A.bytes < block || s->scal.bytes < scalar_bytes(R, M)) {
    s->A.release();
    s->B.release();
    s->U.release();
    s->scal.release();
    CK(s->A.ensure(block));
    CK(s->B.ensure(block));
    CK(s->U.ensure(block));
    CK(s->scal.ensure(scalar_bytes(R, M)));
    s->gen++;
  }
  return FTLM_OK;
}

// parts: H q_j blocks (one per pass of the vector-major multi-pass gather)
ftlm_status ensure_hq(ftlm_system* s, int R, int c64, int parts = 1) {
  const size_t block = (size_t)s->hs.dim * R * (c64 ? 8 : 16) * parts;
  if (s->Hq.bytes < block) {
    s->Hq.release();
    CK(s->Hq.ensure(block));
    s->gen++;
  }
  return FTLM_OK;
}

DevScalars scalars_at(void* base, int R, int M) {
  DevScalars sc;
  sc.ss = R;
  double* b = reinterpret_cast<double*>(base);
  sc.alpha = b;
  b += (size_t)M * R;
  sc.beta = b;
  b += (size_t)M * R;
  sc.p = b;
  b += (size_t)M * R * 2;
  sc.sigma = b;
  b += (size_t)(M + 1) * R;
  sc.scale = b;
  b += R;
  int* ib = reinterpret_cast<int*>(b);
  sc.active = ib;
  sc.meff = ib + R;
  return sc;
}

// The scalars of vector k alone, as a one-vector instance sees them (row
// stride R in the shared arrays).
DevScalars scalars_of_vector(void* base, int R, int M, int k) {
  DevScalars sc = scalars_at(base, R, M);
  sc.alpha += k;
  sc.beta += k;
  sc.p += 2 * k;
  sc.sigma += k;
  sc.scale += k;
  sc.active += k;
  sc.meff += k;
  return sc;
}

// ---- captured runs ------------------------------------------------------------

struct RunCtx {
  std::string key;
  std::vector<uint64_t> deps;  // system ids
  cudaGraph_t g = nullptr;
  cudaGraphExec_t ex = nullptr;
  DevBuf desc, tiles, partials, counter;
  DevBuf vslots;  // vector-major runs: arrival counters, then partial sums by (vector, tile)
  int stream_grid = 0, stream_tiles = 0, stored_grid = 0, stored_tiles = 0, stream_at = 0, stored_at = 0;
  bool even = false;  // every vector's length is even
  std::vector<cudaEvent_t> ev;  // [2M + 2] when kernel timing is on
  int launches = 0, hv_launches = 0;
  char* pinned = nullptr;
  size_t h2d = 0;
  ~RunCtx() {
    if (ex) cudaGraphExecDestroy(ex);
    if (g) cudaGraphDestroy(g);
    desc.release();
    tiles.release();
    partials.release();
    counter.release();
    vslots.release();
    for (auto e : ev) cudaEventDestroy(e);
    if (pinned) cudaFreeHost(pinned);
  }
};

std::vector<std::shared_ptr<RunCtx>> g_ctx;  // small cache of captured runs, newest last; a run in progress keeps its own

void purge_ctx_of(uint64_t id) {
  std::lock_guard<std::mutex> lk(g_mu);
  for (auto it = g_ctx.begin(); it != g_ctx.end();) {
    bool hit = false;
    for (auto d : (*it)->deps) hit = hit || d == id;
    if (hit) it = g_ctx.erase(it);
    else ++it;
  }
}

std::string run_key(const std::vector<ftlm_system*>& sys, const ftlm_run_params* p, const Plan& pl) {
  char buf[640];
  std::string k;
  for (auto* s : sys) {
    snprintf(buf, sizeof buf, "%llu:%llu,", (unsigned long long)s->id, (unsigned long long)s->gen);
    k += buf;
  }
  double u[3];
  observable_coefs(sys[0]->hs, p->obs_dir, u);
  snprintf(buf, sizeof buf,
           "|R%d M%d dt%d seed%llu off%llu st%d bo%llu us%p tk%d th%d rpt%d g%d tol%.17g obs%.17g,%.17g,%.17g,%d s%p",
           p->R, p->M, (int)p->dtype, (unsigned long long)p->seed, (unsigned long long)p->vec_offset, p->start,
           (unsigned long long)p->basis_offset, p->user_start, p->time_kernels, pl.sh.threads, pl.sh.rows_per_tile,
           pl.grid, p->breakdown_tol, u[0], u[1], u[2], p->obs_dir ? 1 : 0, p->stream);
  k += buf;
  k += p->symmetric ? "|sym" : "";
  k += p->reorth ? "|reorth" : "";
  k += pl.storedV ? "|rows" + std::to_string(pl.storedV) + "s" + std::to_string(pl.small) : "";
  k += pl.rot.on ? "|rot" + std::to_string(pl.rot.group) : "";
  k += pl.gen_vm ? "|gvm" + std::to_string(pl.gvm_V) + "x" + std::to_string(pl.gvm_rows) + "c" +
                       std::to_string(pl.gvm_cube) + "L" + std::to_string(pl.tile.L)
                 : "";
  snprintf(buf, sizeof buf, "|half%d vm%d hy%d K%d Rg%d rpt%d g%d P%d mb%d", pl.half.on ? 1 : 0, pl.half.vm ? 1 : 0,
           pl.half.hybrid ? 1 : 0,
           pl.half.K, pl.half.Rg, pl.half.rows_per_tile, pl.half.grid, pl.half.passes, pl.half.min_blocks);
  return k + buf;
}

ftlm_status validate_params(const ftlm_run_params* p, const std::vector<ftlm_system*>& sys) {
  if (!p) return fail(FTLM_ERR_INVALID_ARG, "params is NULL");
  if (p->dtype != FTLM_C64 && p->dtype != FTLM_C128) return fail(FTLM_ERR_INVALID_ARG, "unknown dtype");
  const int c64 = p->dtype == FTLM_C64;
  if (p->R < 1 || p->R > max_vectors(c64))
    return fail(FTLM_ERR_INVALID_ARG, "R must be in 1.." + std::to_string(max_vectors(c64)));
  if (p->M < 1 || p->M > 100000) return fail(FTLM_ERR_INVALID_ARG, "M must be in 1..100000");
  if (!p->T || p->nT < 1) return fail(FTLM_ERR_INVALID_ARG, "temperature grid missing");
  for (int t = 0; t < p->nT; ++t)
    if (!(p->T[t] > 0.0) || !std::isfinite(p->T[t])) return fail(FTLM_ERR_INVALID_ARG, "temperatures must be > 0");
  if (p->start < 0 || p->start > 3) return fail(FTLM_ERR_INVALID_ARG, "unknown start mode");
  if (p->start == FTLM_START_USER && !p->user_start) return fail(FTLM_ERR_INVALID_ARG, "user_start is NULL");
  if (p->start == FTLM_START_USER && (reinterpret_cast<uintptr_t>(p->user_start) & 15))
    return fail(FTLM_ERR_INVALID_ARG, "user_start must be 16-byte aligned");
  if (p->start == FTLM_START_USER && sys.size() != 1)
    return fail(FTLM_ERR_INVALID_ARG, "user start vectors need a single system");
  if (p->symmetric && sys.size() != 1) return fail(FTLM_ERR_INVALID_ARG, "symmetric runs take one system");
  if (p->symmetric != 0 && p->symmetric != 1) return fail(FTLM_ERR_INVALID_ARG, "symmetric must be 0 or 1");
  if (p->reorth != 0 && p->reorth != 1) return fail(FTLM_ERR_INVALID_ARG, "reorth must be 0 or 1");
  if (p->reorth && sys.size() != 1)
    return fail(FTLM_ERR_UNSUPPORTED, "re-orthogonalised runs take one system (ftlm_run)");
  if (!(p->breakdown_tol >= 0) || !std::isfinite(p->breakdown_tol))
    return fail(FTLM_ERR_INVALID_ARG, "breakdown_tol must be finite and >= 0");
  if (p->obs_dir && !(std::isfinite(p->obs_dir[0]) && std::isfinite(p->obs_dir[1]) && std::isfinite(p->obs_dir[2])))
    return fail(FTLM_ERR_INVALID_ARG, "obs_dir must be finite");
  for (auto* s : sys) {
    if (!s) return fail(FTLM_ERR_INVALID_ARG, "system is NULL");
    if (p->start == FTLM_START_BASIS && p->basis_offset + (uint64_t)p->R > s->hs.dim)
      return fail(FTLM_ERR_INVALID_ARG, "basis_offset + R exceeds the dimension");
  }
  return FTLM_OK;
}

// Staged per system: alpha, beta, p ([M][R], [M][R], [M][R][2]) and sigma ([M][R],
// the scale of the unnormalised Lanczos vectors), contiguous in the scalars;
// then M_eff [R].
size_t staged_doubles(int R, int M) { return (size_t)M * R * 5; }
size_t staged_bytes(int R, int M) { return sizeof(double) * staged_doubles(R, M) + sizeof(int) * (size_t)R; }

// The rotated-basis passes of one product or step over the whole block, group by
// group (the groups share the W blocks).
ftlm_status enqueue_rot_passes(RunCtx* ctx, ftlm_system* s, const RotPlan& rp, RotArgs a, int R, int c64, void* keep,
                               cudaStream_t st) {
  const size_t vb = (size_t)s->hs.dim * (c64 ? 8 : 16);
  for (int v0 = 0; v0 < R; v0 += rp.group) {
    a.vec0 = a.vecW = v0;
    a.nvec = std::min(rp.group, R - v0);
    a.vpb = std::min(a.nvec, 4);
    for (int pass = 0; pass < 3; ++pass) {
      CKI(launch_rot(a, pass, c64, st));
      if (pass == 0 && keep) {  // q_j is final after the forward pass
        CK(cudaMemcpyAsync(static_cast<char*>(keep) + vb * v0, static_cast<const char*>(a.x) + vb * v0, vb * a.nvec,
                           cudaMemcpyDeviceToDevice, st));
        if (ctx) ctx->launches++;
      }
    }
    if (ctx) ctx->launches += 3;
  }
  return FTLM_OK;
}

// The M Lanczos steps of a rotated-basis run; `upd` is the update launch that
// ends the last one.
ftlm_status enqueue_rot_steps(RunCtx& ctx, ftlm_system* s, const ftlm_run_params* p, const Plan& pl, StreamArgs upd,
                              const InstDesc* d_even, const InstDesc* d_odd, cudaStream_t st) {
  const int M = p->M, R = p->R, c64 = pl.c64;
  const size_t esz = c64 ? 8 : 16, d = (size_t)s->hs.dim;
  RotArgs a = rot_args(s, pl.rot, c64);
  a.M = M;
  a.tol = p->breakdown_tol > 0 ? p->breakdown_tol : (c64 ? 1e-6 : 1e-12);
  a.sc = scalars_at(s->scal.p, R, M);
  a.u = s->U.p;
  a.W = s->rW.p;
  a.partials = reinterpret_cast<double*>(s->rpart.p);
  a.counters = reinterpret_cast<unsigned*>(a.partials + 3 * (d >> pl.rot.T) * R);
  a.lanczos = 1;
  CK(cudaMemsetAsync(a.counters, 0, sizeof(unsigned) * R, st));
  auto mark = [&](int e) {
    return p->time_kernels ? cudaEventRecordWithFlags(ctx.ev[e], st, cudaEventRecordExternal) : cudaSuccess;
  };
  for (int j = 0; j < M; ++j) {
    a.x = j % 2 == 0 ? s->A.p : s->B.p;
    a.y = j % 2 == 0 ? s->B.p : s->A.p;
    a.j = j;
    a.update = j > 0;
    CK(mark(1 + 4 * j));
    CK(mark(2 + 4 * j));
    ftlm_status rs = enqueue_rot_passes(&ctx, s, pl.rot, a, R, c64,
                                        p->symmetric ? static_cast<char*>(s->Vs.p) + esz * d * R * j : nullptr, st);
    if (rs != FTLM_OK) return rs;
    ctx.hv_launches++;
    CK(mark(3 + 4 * j));
    CK(mark(4 + 4 * j));
  }
  upd.inst = (M - 1) % 2 == 0 ? d_even : d_odd;
  upd.j = M - 1;
  CKI(launch_stream_vectors(upd, kModeUpdate, c64, ctx.even, ctx.stream_grid, st));
  ctx.launches++;
  return FTLM_OK;
}

// Enqueues one whole run on `st` (which the caller is capturing).
ftlm_status enqueue_run(RunCtx& ctx, const std::vector<ftlm_system*>& sys, const ftlm_run_params* p, const Plan& pl,
                        cudaStream_t st) {
  const int M = p->M, R = p->R, c64 = pl.c64;
  const int n = (int)sys.size();
  const int nd = plan_vmaj(pl) ? n * R : n;  // descriptors per kind: one per (system, vector) in the vector-major layout
  const InstDesc* d_even = reinterpret_cast<const InstDesc*>(ctx.desc.p);
  const InstDesc* d_odd = d_even + nd;
  const InstDesc* d_start = d_even + 2 * nd;
  const InstDesc* d_gather_even = d_even + 3 * nd;  // split steps: x = q_j, y = Hq
  const InstDesc* d_gather_odd = d_even + 4 * nd;
  // the spin-1/2 gathers and the wide general gather run alone; the step epilogue streams afterwards
  const bool split = pl.half.on || pl.wideV || pl.gen_vm;
  // single-pass gathers also sum Re<q_j|H q_j>, so alpha_j is known before the
  // epilogue, which then finishes the step in one pass (no separate update)
  const bool fused = pl.half.on && (pl.half.passes == 1 || pl.half.vm);
  // the vector-major one-pass gather goes further: it writes w' over q_{j-1}
  // and sums alpha_j and p_j itself; the update pass finishes the step
  const bool fused_step = vm_fused_step(pl);
  LaunchArgs a = pl.base;
  a.tile_start = reinterpret_cast<const int*>(ctx.tiles.p);
  a.partials = reinterpret_cast<double*>(ctx.partials.p);
  a.counter = reinterpret_cast<unsigned*>(ctx.counter.p);
  if (fused_step) a.unit_tab = sys[0]->ut[c64 ? 1 : 0].p;  // built by run_impl before the capture
  ctx.launches = 0;
  ctx.hv_launches = 0;
  const bool tk = p->time_kernels != 0;
  int evi = 0;
  if (tk) CK(cudaEventRecordWithFlags(ctx.ev[evi++], st, cudaEventRecordExternal));
  const int vmaj = plan_vmaj(pl) ? 1 : 0;
  for (int k = 0; k < n; ++k) {  // start block -> A
    InstDesc h = base_desc(sys[k], c64);
    const long long dim = (long long)sys[k]->hs.dim;
    if (p->start == FTLM_START_RANDOM)
      CKI(launch_start_random(&h, nullptr, R, p->seed, p->vec_offset, sys[k]->A.p, c64, st, vmaj));
    else if (p->start == FTLM_START_PAIRS)
      CKI(launch_start_pairs(&h, R, p->seed, p->vec_offset, sys[k]->A.p, c64, st, vmaj));
    else if (p->start == FTLM_START_BASIS)
      CKI(launch_start_basis(dim, R, p->basis_offset, sys[k]->A.p, c64, st, vmaj));
    else if (vmaj)
      CKI(launch_to_vector_major(p->user_start, sys[k]->A.p, dim, R, c64, st));
    else
      CKI(launch_copy_block(p->user_start, sys[k]->A.p, (size_t)dim * R * (c64 ? 8 : 16), st));
    ctx.launches++;
  }
  // vector-major runs: streaming passes by vector
  StreamArgs sa;
  if (vmaj) {
    sa.tile_start = reinterpret_cast<const int*>(ctx.tiles.p) + ctx.stream_at;
    sa.vectors = nd;
    sa.max_tiles = ctx.stream_tiles;
    sa.counters = reinterpret_cast<unsigned*>(ctx.vslots.p);
    sa.slots = reinterpret_cast<double*>(static_cast<char*>(ctx.vslots.p) + (((size_t)nd * 4 + 255) & ~size_t(255)));
  }
  auto stream = [&](int mode, const InstDesc* inst, int j) {
    sa.inst = inst;
    sa.j = j;
    return launch_stream_vectors(sa, mode, c64, ctx.even, ctx.stream_grid, st);
  };
  a.inst = d_start;  // sigma_0 = 1/|q_0|, then U = sigma_0 (u.S) q_0
  a.mode = kModeStartNorm;
  if (vmaj) CKI(stream(kModeStartNorm, d_start, 0));
  else CKI(launch_plan(pl, a, st));
  ctx.launches++;
  for (auto* s : sys) {
    SdirArgs u = sdir_args(s, c64, R, s->A.p, s->U.p);
    observable_coefs(s->hs, p->obs_dir, u.obs);
    u.sigma = scalars_at(s->scal.p, R, M).sigma;
    CKI(launch_sdir(u, s->hs.q.data(), c64, vmaj != 0, st));
    ctx.launches++;
  }
  if (pl.rot.on) {
    ftlm_status rs = enqueue_rot_steps(ctx, sys[0], p, pl, sa, d_even, d_odd, st);
    if (rs != FTLM_OK) return rs;
  }
  if (pl.small) {
    SmallRunArgs g;
    g.inst = d_even;
    g.keep = p->symmetric ? sys[0]->Vs.p : nullptr;
    g.R = R;
    long long most = 0;
    for (auto* s : sys) most = std::max(most, (long long)s->hs.dim);
    CKI(launch_small_run(g, nd, pl.small, most, c64, st));
    ctx.launches++;
    ctx.hv_launches = M;
  }
  for (int j = 0; j < M && !pl.rot.on && !pl.small; ++j) {
    a.inst = (j % 2 == 0) ? d_even : d_odd;
    a.step = j;
    a.first = j == 0;
    // time_kernels: events at the step's start and end and around its H.v launch
    // ([1 + 4j] .. [4 + 4j]); a step's start event follows the previous step's
    // end event with no work between them, so their difference is the gap
    // between two launches of the graph
    if (tk) {
      evi = 1 + 4 * j;
      CK(cudaEventRecordWithFlags(ctx.ev[evi++], st, cudaEventRecordExternal));
    }
    if (p->symmetric || p->reorth) {  // keep q_j (vector-major): the matrix of u.S in the Lanczos basis, or
                                       // the vectors the next ones are re-orthogonalised against
      ftlm_system* s0 = sys[0];
      const size_t vb = (size_t)s0->hs.dim * R * (c64 ? 8 : 16);
      const void* q = (j % 2 == 0) ? s0->A.p : s0->B.p;
      void* dst = static_cast<char*>(s0->Vs.p) + vb * j;
      if (plan_vmaj(pl)) CK(cudaMemcpyAsync(dst, q, vb, cudaMemcpyDeviceToDevice, st));
      else CKI(launch_to_vector_major(q, dst, (long long)s0->hs.dim, R, c64, st));
      ctx.launches++;
    }
    if (pl.storedV) {  // stored rows: w' over q_{j-1}, alpha_j, p_j
      StoredArgs g;
      g.inst = a.inst;
      g.tile_start = reinterpret_cast<const int*>(ctx.tiles.p) + ctx.stored_at;
      g.groups = n * ((R + pl.storedV - 1) / pl.storedV);
      g.R = R;
      g.max_tiles = ctx.stored_tiles;
      g.j = j;
      g.slots = sa.slots;
      g.counters = sa.counters;
      if (tk) CK(cudaEventRecordWithFlags(ctx.ev[evi++], st, cudaEventRecordExternal));
      CKI(launch_stored_step(g, pl.storedV, c64, ctx.stored_grid, st));
    } else if (fused_step || (pl.gen_vm && pl.gvm_cube)) {  // these gathers write w' over q_{j-1} and set alpha_j, p_j
      LaunchArgs g = a;                                     // x = q_j, y = q_{j-1}, u
      g.mode = kModeApply;
      g.fused_step = 1;
      if (tk) CK(cudaEventRecordWithFlags(ctx.ev[evi++], st, cudaEventRecordExternal));
      CKI(launch_plan(pl, g, st));
    }
    if (pl.storedV || fused_step || (pl.gen_vm && pl.gvm_cube)) {
      if (tk) CK(cudaEventRecordWithFlags(ctx.ev[evi++], st, cudaEventRecordExternal));
      CKI(stream(kModeUpdate, a.inst, j));
      ctx.launches += 2;
      ctx.hv_launches++;
      if (tk) CK(cudaEventRecordWithFlags(ctx.ev[4 + 4 * j], st, cudaEventRecordExternal));
      continue;
    }
    if (split) {
      LaunchArgs g = a;
      g.inst = (j % 2 == 0) ? d_gather_even : d_gather_odd;
      g.mode = kModeApply;
      g.gather_alpha = fused ? 1 : 0;
      if (tk) CK(cudaEventRecordWithFlags(ctx.ev[evi++], st, cudaEventRecordExternal));
      CKI(launch_plan(pl, g, st));
      if (tk) CK(cudaEventRecordWithFlags(ctx.ev[evi++], st, cudaEventRecordExternal));
      if (fused) {
        a.mode = kModeStep;
        a.hq_parts = (pl.half.vm && !pl.half.hybrid) ? pl.half.passes : 1;  // the passes' partial H q_j blocks
        a.hq_stride = (long long)R * (long long)sys[0]->hs.dim;
        CKI(launch_plan(pl, a, st));
        a.hq_parts = 1;
        ctx.launches += 2;
        ctx.hv_launches++;
        if (tk) CK(cudaEventRecordWithFlags(ctx.ev[4 + 4 * j], st, cudaEventRecordExternal));
        continue;
      }
      a.mode = kModeEpilogue;
      CKI(launch_plan(pl, a, st));
      ctx.launches++;
    } else {
      a.mode = kModeLanczos;
      if (tk) CK(cudaEventRecordWithFlags(ctx.ev[evi++], st, cudaEventRecordExternal));
      CKI(launch_plan(pl, a, st));
      if (tk) CK(cudaEventRecordWithFlags(ctx.ev[evi++], st, cudaEventRecordExternal));
    }
    a.mode = kModeUpdate;
    if (vmaj) CKI(stream(kModeUpdate, a.inst, j));
    else CKI(launch_plan(pl, a, st));
    ctx.launches += 2;
    ctx.hv_launches++;
    if (p->reorth) {  // two Gram-Schmidt passes against q_0..q_j, then the norm of what is left
      ftlm_system* s0 = sys[0];
      const DevScalars sc = scalars_at(s0->scal.p, R, M);
      void* w = (j % 2 == 0) ? s0->B.p : s0->A.p;
      for (int pass = 0; pass < 2; ++pass)
        CKI(launch_reorth_pass(s0->Vs.p, w, (long long)s0->hs.dim, R, j, M, reinterpret_cast<double*>(s0->Gre.p),
                               sc.sigma, c64, st));
      a.mode = kModeUpdate;
      a.update_no_alpha = 1;
      CKI(launch_plan(pl, a, st));
      a.update_no_alpha = 0;
      ctx.launches += 5;
    }
    if (tk) CK(cudaEventRecordWithFlags(ctx.ev[4 + 4 * j], st, cudaEventRecordExternal));
  }
  if (tk) CK(cudaEventRecordWithFlags(ctx.ev[4 * M + 1], st, cudaEventRecordExternal));
  const size_t per = staged_bytes(R, M);
  for (int k = 0; k < n; ++k) {  // alpha, beta, p, M_eff -> pinned host staging
    DevScalars sc = scalars_at(sys[k]->scal.p, R, M);
    char* dst = ctx.pinned + per * k;
    CK(cudaMemcpyAsync(dst, sc.alpha, sizeof(double) * staged_doubles(R, M), cudaMemcpyDeviceToHost, st));
    CK(cudaMemcpyAsync(dst + sizeof(double) * staged_doubles(R, M), sc.meff, sizeof(int) * R, cudaMemcpyDeviceToHost,
                       st));
  }
  return FTLM_OK;
}

ftlm_status build_ctx(RunCtx& c, const std::vector<ftlm_system*>& sys, const ftlm_run_params* p, const Plan& pl,
                      cudaStream_t st) {
  const int c64 = pl.c64, R = p->R, M = p->M, n = (int)sys.size();
  for (auto* s : sys) c.deps.push_back(s->id);
  // descriptors: even steps (x = A, y = B), odd steps (x = B, y = A), start (x = A, y = U),
  // and for split steps the gathers (x = A or B, y = Hq); one per system, or in the
  // vector-major layout one per vector (pointers at vector k, scalars of vector k)
  const bool vmaj = plan_vmaj(pl);
  const int nd = vmaj ? n * R : n;
  std::vector<InstDesc> h(5 * nd);
  for (int k = 0; k < nd; ++k) {
    ftlm_system* s = sys[vmaj ? k / R : k];  // vector-major: instance k is vector k % R of system k / R
    const int vec = vmaj ? k % R : 0;
    InstDesc d = base_desc(s, c64);
    d.sc = vmaj ? scalars_of_vector(s->scal.p, R, M, vec) : scalars_at(s->scal.p, R, M);
    const size_t off = vmaj ? (size_t)vec * s->hs.dim * (c64 ? 8 : 16) : 0;  // bytes to vector vec
    char* A = static_cast<char*>(s->A.p) + off;
    char* B = static_cast<char*>(s->B.p) + off;
    char* U = static_cast<char*>(s->U.p) + off;
    char* Hq = s->Hq.p ? static_cast<char*>(s->Hq.p) + off : nullptr;
    d.u = U;
    d.M = M;
    d.tol = p->breakdown_tol > 0 ? p->breakdown_tol : (c64 ? 1e-6 : 1e-12);
    InstDesc e = d, o = d, t = d;
    e.x = A;
    e.y = B;
    o.x = B;
    o.y = A;
    t.x = A;
    t.y = U;
    e.hq = o.hq = Hq;
    if (pl.storedV) {
      bool ok = false;  // (built by run_impl before the capture)
      ftlm_status rs = ensure_stored(s, c64, stored_limit(s, c64, n), (long long)R * M, st, e.stored, ok);
      if (rs != FTLM_OK) return rs;
      if (!ok) return fail(FTLM_ERR_CUDA, "stored rows are missing");
      o.stored = e.stored;
    }
    InstDesc ge = d, go = d;
    ge.x = A;
    ge.y = Hq;
    go.x = B;
    go.y = Hq;
    h[k] = e;
    h[nd + k] = o;
    h[2 * nd + k] = t;
    h[3 * nd + k] = ge;
    h[4 * nd + k] = go;
  }
  CK(c.desc.ensure(sizeof(InstDesc) * h.size()));
  CK(cudaMemcpy(c.desc.p, h.data(), sizeof(InstDesc) * h.size(), cudaMemcpyHostToDevice));
  std::vector<int> tiles = pl.tile_start;  // the instances' tile list, then the H.v groups' (vector-major general)
  tiles.insert(tiles.end(), pl.tile_start_g.begin(), pl.tile_start_g.end());
  if (vmaj) {  // then the streaming passes' list by vector and the stored-row groups' list
    c.even = true;
    auto list = [&](int step, long long rows, int& at, int& most, int& grid) -> bool {
      at = (int)tiles.size();
      tiles.push_back(0);
      for (int k = 0; k < n; ++k)
        for (int v = 0; v < R; v += step) {
          const long long t = ((long long)sys[k]->hs.dim + rows - 1) / rows;
          if (tiles.back() + t > (1ll << 30)) return false;
          tiles.push_back(tiles.back() + (int)t);
          most = std::max(most, (int)t);
          c.even = c.even && sys[k]->hs.dim % 2 == 0;
        }
      grid = tiles.back();
      return true;
    };
    if (!list(1, kStreamChunk, c.stream_at, c.stream_tiles, c.stream_grid) ||
        (pl.storedV && !list(pl.storedV, 32, c.stored_at, c.stored_tiles, c.stored_grid)))
      return fail(FTLM_ERR_UNSUPPORTED, "too many tiles");
    const size_t cnt = ((size_t)nd * 4 + 255) & ~size_t(255);
    CK(c.vslots.ensure(cnt + sizeof(double) * 3 * (size_t)nd * std::max(c.stream_tiles, c.stored_tiles)));
    CK(cudaMemset(c.vslots.p, 0, cnt));
  }
  CK(c.tiles.ensure(sizeof(int) * tiles.size()));
  CK(cudaMemcpy(c.tiles.p, tiles.data(), sizeof(int) * tiles.size(), cudaMemcpyHostToDevice));
  CK(c.partials.ensure(sizeof(double) * (size_t)n * plan_max_grid(pl) * R * kNumPartials));  // n_inst x R = R x 1 when vector-major
  CK(c.counter.ensure(64));
  CK(cudaMemset(c.counter.p, 0, 64));
  c.h2d = sizeof(InstDesc) * h.size() + sizeof(int) * tiles.size();
  CK(cudaMallocHost(reinterpret_cast<void**>(&c.pinned), staged_bytes(R, M) * n));
  if (p->time_kernels) {
    c.ev.resize(4 * M + 2);
    for (auto& e : c.ev) CK(cudaEventCreate(&e));
  }
  std::shared_lock<std::shared_mutex> capturing(g_capture);
  CK(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
  ftlm_status es = enqueue_run(c, sys, p, pl, st);
  cudaGraph_t g = nullptr;
  cudaError_t ce = cudaStreamEndCapture(st, &g);
  capturing.unlock();
  if (es != FTLM_OK) {
    if (g) cudaGraphDestroy(g);
    return es;
  }
  CK(ce);
  c.g = g;
  CK(cudaGraphInstantiate(&c.ex, g, 0));
  return FTLM_OK;
}

// ---- symmetric estimator: O_ij = <v_i|u.S|v_j> per vector ---------------------

// A symmetric run's blocks besides its Lanczos vectors: partial sums of O, the O
// matrices, and u.S q_k of all stored vectors (as large as these).
ftlm_status ensure_symmetric(ftlm_system* s, int R, int M, int c64) {
  const long long d = (long long)s->hs.dim;
  if ((long long)R * M > 65535) return fail(FTLM_ERR_UNSUPPORTED, "symmetric run: R * M must not exceed 65535");
  const size_t pbytes = sizeof(double) * sym_partial_doubles(R, M, sym_ranges(d, R, M));
  const size_t obytes = sizeof(double) * 2 * (size_t)R * M * M, wbytes = (size_t)d * R * (c64 ? 8 : 16) * M;
  if (s->Wc.ensure(pbytes) != cudaSuccess) return fail(FTLM_ERR_OUT_OF_MEMORY, "O matrix partial sums");
  if (s->Od.ensure(obytes) != cudaSuccess) return fail(FTLM_ERR_OUT_OF_MEMORY, "O matrices");
  if (s->Ws.ensure(wbytes) != cudaSuccess)
    return fail(FTLM_ERR_OUT_OF_MEMORY, "symmetric run: " + std::to_string(wbytes) + " bytes for u.S of the Lanczos vectors");
  return FTLM_OK;
}

// After a symmetric run: G_r[i][j] = <q_i|u.S q_j> for the stored unnormalised
// vectors q_0 .. q_{M-1} of every vector r: u.S of all of them, the contraction
// and a fixed-order reduction of its per-range partials; then O_ij = sigma_i sigma_j G_ij on
// the host.  Omat [R][M][M] complex row-major; sigma [M][R].
ftlm_status symmetric_matrices(ftlm_system* s, const ftlm_run_params* p, cudaStream_t st, const double* sigma,
                               std::vector<double>& Omat, double& ms) {
  const int R = p->R, M = p->M, c64 = p->dtype == FTLM_C64;
  const long long d = (long long)s->hs.dim;
  const int nranges = sym_ranges(d, R, M);
  const size_t obytes = sizeof(double) * 2 * (size_t)R * M * M;
  void* W = s->Ws.p;
  SdirArgs u = sdir_args(s, c64, R * M, s->Vs.p, W);
  observable_coefs(s->hs, p->obs_dir, u.obs);
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  CK(cudaEventRecord(e0, st));
  CKI(launch_sdir(u, s->hs.q.data(), c64, true, st));
  CKI(launch_sym_omat(d, s->Vs.p, W, R, M, nranges, reinterpret_cast<double*>(s->Wc.p),
                      reinterpret_cast<double*>(s->Od.p), c64, st));
  CK(cudaEventRecord(e1, st));
  std::vector<double> host((size_t)R * M * M * 2);
  CK(cudaMemcpyAsync(host.data(), s->Od.p, obytes, cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  float fms = 0.f;
  CK(cudaEventElapsedTime(&fms, e0, e1));
  ms = fms;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  Omat.assign((size_t)R * M * M * 2, 0.0);
  for (int r = 0; r < R; ++r)
    for (int i = 0; i < M; ++i)
      for (int j = 0; j < M; ++j) {
        const size_t e = ((size_t)r * M + i) * M + j;
        const double sc = sigma[(size_t)i * R + r] * sigma[(size_t)j * R + r];
        Omat[2 * e] = sc * host[2 * e];
        Omat[2 * e + 1] = sc * host[2 * e + 1];
      }
  return FTLM_OK;
}

// lean: without the blocks that a run keeps for speed alone
ftlm_status run_impl(const std::vector<ftlm_system*>& sys, const ftlm_run_params* p, ftlm_result* res, bool lean) {
  ftlm_status vs = validate_params(p, sys);
  if (vs != FTLM_OK) return vs;
  if (!res) return fail(FTLM_ERR_INVALID_ARG, "result is NULL");
  const int c64 = p->dtype == FTLM_C64;
  const int R = p->R, M = p->M, n = (int)sys.size();
  int dev = 0;
  CK(cudaGetDevice(&dev));
  for (auto* s : sys)
    if (s->device != dev) return fail(FTLM_ERR_INVALID_ARG, "system lives on another device");
  const cudaStream_t caller = pick_stream(sys[0], p->stream);
  const cudaStream_t st = sys[0]->own_stream;  // graphs are captured and launched on the first system's stream
  for (auto* s : sys) {
    ftlm_status w = ensure_workspace(s, R, M, c64);
    if (w != FTLM_OK) return w;
  }
  Plan pl;
  ftlm_status ps;
  if (p->reorth) {  // the general row kernel on the row-major block, gather and update in two launches
    Shape gen = default_shape(R, c64);
    gen.explicit_general = true;
    ps = make_plan(sys, R, c64, pl, &gen, false);
    pl.wideV = 0;
  } else {
    ps = make_plan(sys, R, c64, pl, nullptr, true);
  }
  if (ps != FTLM_OK) return ps;
  // (what a run cannot do without comes before what it takes for speed)
  if (p->symmetric || p->reorth) {  // the M Lanczos vectors of every vector
    ftlm_system* s0 = sys[0];
    const size_t vb = (size_t)s0->hs.dim * R * (c64 ? 8 : 16) * M;
    if (s0->Vs.bytes < vb) {
      s0->Vs.release();
      if (s0->Vs.ensure(vb) != cudaSuccess)
        return fail(FTLM_ERR_OUT_OF_MEMORY, std::string(p->symmetric ? "symmetric" : "re-orthogonalised") +
                                                " run: " + std::to_string(vb) + " bytes of Lanczos vectors");
      s0->gen++;
    }
  }
  if (p->symmetric) {
    ftlm_status ss = ensure_symmetric(sys[0], R, M, c64);
    if (ss != FTLM_OK) return ss;
  }
  if (p->reorth) {
    ftlm_system* s0 = sys[0];
    const size_t gb = sizeof(double) * 2 * (size_t)R * M;
    if (s0->Gre.bytes < gb) {
      s0->Gre.release();
      CK(s0->Gre.ensure(gb));
      s0->gen++;
    }
  }
  // Runs from random vectors on the default spin-1/2 plan take the rotated-basis
  // H.v.  Its error is relative to the whole vector, so starts that may be
  // sparse (basis states, a caller's block) keep the gather, which leaves the
  // rows that H does not reach exactly zero.
  if (!lean && vm_fused_step(pl) && (p->start == FTLM_START_RANDOM || p->start == FTLM_START_PAIRS) &&
      rot_allowed(sys[0], R, c64)) {
    ftlm_status rs = make_rot(sys[0], R, c64, pl.rot, st);
    if (rs != FTLM_OK) return rs;
  }
  bool forced = lean;
  for (auto* s : sys) forced = forced || has_shape_override(s, R, c64);
  if (plan_vmaj(pl) && !pl.rot.on && !forced) {  // small systems: stored rows in the gathers' place
    bool all = run_stores(sys, R, M, c64);  // (nothing is written for a batch that one system keeps on the gathers)
    uint64_t rows = 0;
    for (auto* s : sys) {
      StoredRows r;
      if (all) {
        ftlm_status rs = ensure_stored(s, c64, stored_limit(s, c64, n), (long long)R * M, st, r, all);
        if (rs != FTLM_OK) return rs;
      }
      rows += s->hs.dim;
    }
    if (all) pl.storedV = stored_group(rows, R);
    // one launch for all steps while every cluster is resident at once (two CTAs an
    // SM at most): more vectors or rows have work enough to fill the chip step by step
    long long most = 0;
    for (auto* s : sys) most = std::max(most, (long long)s->hs.dim);
    for (int c = 8; c >= 1 && all && !p->time_kernels && !pl.small; c /= 2) {
      const size_t smem = small_run_smem(most, c, c64);
      const int fit = smem <= kSmallRunBytes ? std::min<int>(2, (int)(200 * 1024 / (smem + 4096))) * std::max(1, device_sm_count()) : 0;
      if ((long long)n * R * c <= fit) pl.small = c;
    }
  }
  if (vm_fused_step(pl) && !pl.rot.on && !pl.storedV) {
    ftlm_status ut = ensure_unit_tables(sys[0], pl.half.K, c64, st);
    if (ut != FTLM_OK) return ut;
  }
  if (pl.storedV) {
    // (no H q block)
  } else if (pl.half.on && !vm_fused_step(pl)) {  // (the fused vector-major step keeps no H q block)
    ftlm_status hs_ = ensure_hq(sys[0], R, c64, (pl.half.vm && !pl.half.hybrid) ? pl.half.passes : 1);
    if (hs_ != FTLM_OK) return hs_;
  } else if (pl.wideV || (pl.gen_vm && !pl.gvm_cube)) {  // (the cube gather keeps no H q block)
    for (auto* s : sys) {
      ftlm_status hs_ = ensure_hq(s, R, c64, 1);
      if (hs_ != FTLM_OK) return hs_;
    }
  }
  const std::string key = run_key(sys, p, pl);
  std::shared_ptr<RunCtx> ctx;  // (other threads' runs may drop it from the cache meanwhile)
  size_t h2d = 0;
  {
    std::lock_guard<std::mutex> lk(g_mu);
    for (auto& c : g_ctx)
      if (c->key == key) ctx = c;
  }
  if (!ctx) {
    auto nc = std::make_shared<RunCtx>();
    nc->key = key;
    ftlm_status bs = build_ctx(*nc, sys, p, pl, st);
    if (bs != FTLM_OK) return bs;
    h2d = nc->h2d;
    ctx = nc;
    std::lock_guard<std::mutex> lk(g_mu);
    g_ctx.push_back(std::move(nc));
    if (g_ctx.size() > 8) g_ctx.erase(g_ctx.begin());
  }
  const auto t0 = std::chrono::steady_clock::now();
  for (auto* s : sys) {  // after products of the systems still in flight (they may be writing the tables)
    std::lock_guard<std::mutex> lk(s->apply_mu);
    if (s->apply_used) CK(cudaStreamWaitEvent(st, s->ev_apply, 0));
  }
  CK(cudaEventRecord(sys[0]->ev_in, caller));  // after the caller's prior work (e.g. a user start block)
  CK(cudaStreamWaitEvent(st, sys[0]->ev_in, 0));
  CK(cudaGraphLaunch(ctx->ex, st));
  CK(cudaEventRecord(sys[0]->ev_out, st));
  CK(cudaStreamWaitEvent(caller, sys[0]->ev_out, 0));  // the caller's later work sees the run complete
  CK(cudaStreamSynchronize(st));
  const auto t1 = std::chrono::steady_clock::now();
  double hv_ms = 0.0, gap_ms = 0.0, dev_ms = std::chrono::duration<double, std::milli>(t1 - t0).count();
  if (p->time_kernels && !ctx->ev.empty()) {
    for (int j = 0; j < M; ++j) {
      float ms = 0.f;
      CK(cudaEventElapsedTime(&ms, ctx->ev[2 + 4 * j], ctx->ev[3 + 4 * j]));
      hv_ms += ms;
      if (j + 1 < M) {
        CK(cudaEventElapsedTime(&ms, ctx->ev[4 + 4 * j], ctx->ev[1 + 4 * (j + 1)]));
        gap_ms += ms;
      }
    }
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, ctx->ev[0], ctx->ev[4 * M + 1]));
    dev_ms = ms;
  }
  const size_t per = staged_bytes(R, M);
  std::vector<HostSums> sums(n);
  for (int k = 0; k < n; ++k) {  // (read where the copies left them, [M][R])
    const char* src = ctx->pinned + per * k;
    const double* alpha_d = reinterpret_cast<const double*>(src);
    const double* beta_d = alpha_d + (size_t)M * R;
    const double* p_d = beta_d + (size_t)M * R;
    const int* meff = reinterpret_cast<const int*>(src + sizeof(double) * staged_doubles(R, M));
    for (int r = 0; r < R; ++r)
      if (meff[r] < 1 || meff[r] > M) return fail(FTLM_ERR_NUMERICAL, "start vector of zero norm");
    sums[k] = {R, M, meff, alpha_d, beta_d, p_d, 1, (size_t)R, true, (double)sys[k]->hs.dim, sys[k]->hs.g,
               p->T, p->nT, &res[k]};
  }
  host_sums_many(sums);  // eigensolves and sums of all systems
  for (int k = 0; k < n; ++k) {
    ftlm_result& out = res[k];
    if (sums[k].status != FTLM_OK) return fail(sums[k].status, sums[k].msg);
    out.device_ms = dev_ms;
    out.hv_ms = hv_ms;
    out.gap_ms = gap_ms;
    out.hv_launches = ctx->hv_launches;
    out.kernel_launches = ctx->launches;
    out.h2d_bytes = k == 0 ? h2d : 0;
    out.d2h_bytes = per;
    out.cube_bits = pl.half.on && !pl.rot.on ? pl.half.K : 0;  // (0 also for the vector-major general gather)
    out.passes = pl.rot.on ? 3 : (pl.half.on ? pl.half.passes : 1);
    out.group_vectors = pl.half.on ? pl.half.Rg : (pl.gen_vm ? pl.gvm_V : R);
    out.tile_rows = pl.half.on ? pl.half.rows_per_tile : (pl.gen_vm ? pl.gvm_rows : pl.sh.rows_per_tile);
    out.grid = pl.half.on ? pl.half.grid : (pl.gen_vm ? pl.gvm_grid : pl.grid);
    out.threads = pl.half.on ? pl.half.threads : (pl.tile.V ? pl.tile.threads : (pl.gen_vm ? 256 : pl.sh.threads));
    out.vector_major = plan_vmaj(pl) ? 1 : 0;
    out.site_cube = pl.gen_vm ? pl.gvm_cube : 0;
    out.sym_ms = 0.0;
    if (p->symmetric) {  // Eqs. (E-2-G), (E-2-H)
      const double* sigma_d = reinterpret_cast<const double*>(ctx->pinned + per * k) + (size_t)M * R * 4;  // [M][R]
      std::vector<double> Omat;
      double sms = 0.0;
      ftlm_status os = symmetric_matrices(sys[k], p, st, sigma_d, Omat, sms);
      if (os != FTLM_OK) return os;
      out.sym_ms = sms;
      if (out.M_B_sym) {
        std::string m2;
        std::vector<double> al((size_t)R * M), be((size_t)R * M);  // [R][M]
        for (int r = 0; r < R; ++r)
          for (int j = 0; j < M; ++j) {
            al[(size_t)r * M + j] = sums[k].alpha[(size_t)j * R + r];
            be[(size_t)r * M + j] = sums[k].beta[(size_t)j * R + r];
          }
        ftlm_status hs2 = host_sums_sym(R, M, sums[k].M_eff, al.data(), be.data(), Omat.data(), sys[k]->hs.g, p->T,
                                        p->nT, out.M_B_sym, out.M_B_sym_imag, m2);
        if (hs2 != FTLM_OK) return fail(hs2, m2);
      }
      if (out.O_lanczos) std::memcpy(out.O_lanczos, Omat.data(), sizeof(double) * Omat.size());
    }
  }
  return FTLM_OK;
}

// Times candidate launch shapes of the H.v kernel on the system's workspace
// and keeps the fastest for (n, 2s+1, R, dtype, d).
ftlm_status autotune(ftlm_system* s, int R, int c64, cudaStream_t st, bool lean) {
  ShapeKey key{s->hs.n, s->hs.qmax, R, c64, (long long)s->hs.dim};
  {
    std::lock_guard<std::mutex> lk(g_mu);
    if (g_shapes.count(key)) return FTLM_OK;
  }
  std::vector<Shape> cands;
  if (s->hs.all_half && s->hs.n >= 4) {
    std::vector<int> rgs;
    for (int cap : {64, 32, 16}) {
      const int g = largest_divisor_at_most(R, cap);
      if (std::find(rgs.begin(), rgs.end(), g) == rgs.end()) rgs.push_back(g);
    }
    for (int mp : {0, 1})
      for (int K : {3, 4})
        for (int rg : rgs)
          for (int f : {1, 4})  // cubes per thread slot in a row tile
            for (int mb : {2, 3}) {
              if (mp && mb > 1) continue;
              Shape sh = default_shape(R, c64);
              sh.half_K = K;
              sh.Rg = rg;
              sh.half_rows = f;
              sh.half_multipass = mp;
              sh.half_min_blocks = mb;
              if (s->hs.n >= K + 2) cands.push_back(sh);
            }
    for (int mp : {0, 1, 2})  // the vector-major gather (runs only): one pass, ceil((n-5)/K) passes, two passes
      for (int K : {3, 4})
        for (int f : {1, 2, 4, 8})
          for (int mb : {1, 2}) {  // one 512-thread or two 256-thread CTAs per SM
            Shape sh = default_shape(R, c64);
            sh.half_K = K;
            sh.Rg = largest_divisor_at_most(R, 16);
            sh.half_rows = f;
            sh.half_multipass = mp == 1 ? 1 : 0;
            sh.half_hybrid = mp == 2 ? 1 : 0;
            sh.half_min_blocks = mb;
            sh.half_vm = 1;
            if (s->hs.n >= kVmLaneBits + (mp == 2 ? 2 * K : K)) cands.push_back(sh);
          }
  } else {
    for (int thr : {128, 256})
      for (int f : {1, 4}) {
        Shape sh = shape_for(R, c64, thr, f);
        sh.general_vm = 0;
        cands.push_back(sh);
      }
    for (int cube : {8, 4, 0})  // the vector-major general gather (runs only): cube over 8 or 4 vectors, none
      for (int rows : {256, 512, 1024, 2048}) {
        Shape sh = default_shape(R, c64);
        sh.general_vm = 1;
        sh.gvm_rows = rows;
        sh.gvm_cube = cube;
        cands.push_back(sh);
      }
    Shape sh = default_shape(R, c64);  // and the default plan where it is the tile gather
    sh.plain = true;
    cands.push_back(sh);
  }
  ftlm_status w = ensure_workspace(s, R, 1, c64);
  if (w != FTLM_OK) return w;
  const size_t vbytes = (size_t)s->hs.dim * (c64 ? 8 : 16);
  CK(cudaMemsetAsync(s->A.p, 0, vbytes * R, st));
  DevBuf vdesc;  // the vector-major candidates: one descriptor per vector, output in Hq (one block per pass)
  DevBuf vtiles; // the vector-major general candidates' tile lists
  if (!s->hs.all_half || s->hs.n >= kVmLaneBits + 3) {
    const int passes = s->hs.all_half ? (s->hs.n - kVmLaneBits + 2) / 3 : 1;  // the most passes a candidate uses
    ftlm_status hq = ensure_hq(s, R, c64, passes);
    if (hq != FTLM_OK) return hq;
    std::vector<InstDesc> h(R, base_desc(s, c64));
    for (int k = 0; k < R; ++k) {
      h[k].x = static_cast<char*>(s->A.p) + vbytes * k;
      h[k].y = static_cast<char*>(s->Hq.p) + vbytes * k;
    }
    CK(vdesc.ensure(sizeof(InstDesc) * R));
    CK(cudaMemcpy(vdesc.p, h.data(), sizeof(InstDesc) * R, cudaMemcpyHostToDevice));
  }
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  float best = 1e30f;
  Shape pick = default_shape(R, c64);
  std::vector<ftlm_system*> one{s};
  for (const Shape& sh : cands) {
    Plan pl;
    if (make_plan(one, R, c64, pl, sh.plain ? nullptr : &sh, sh.half_vm != 0 || sh.general_vm == 1 || sh.plain) != FTLM_OK)
      continue;
    if (sh.plain && !pl.tile.V) continue;
    if (sh.half_K > 0 && (!pl.half.on || pl.half.vm != (sh.half_vm != 0))) continue;
    if (sh.general_vm == 1 && (!pl.gen_vm || (sh.gvm_cube > 0 && (!pl.gvm_cube || pl.gvm_V != sh.gvm_cube)))) continue;
    LaunchArgs a = pl.base;
    if (pl.half.vm) {
      a.inst = reinterpret_cast<const InstDesc*>(vdesc.p);
    } else if (pl.gen_vm) {  // R one-vector instances, then the groups' tile list
      std::vector<int> tiles = pl.tile_start;
      tiles.insert(tiles.end(), pl.tile_start_g.begin(), pl.tile_start_g.end());
      CK(cudaStreamSynchronize(st));  // (the previous candidate's launches may read the old list)
      CK(vtiles.ensure(sizeof(int) * tiles.size()));
      CK(cudaMemcpy(vtiles.p, tiles.data(), sizeof(int) * tiles.size(), cudaMemcpyHostToDevice));
      a.inst = reinterpret_cast<const InstDesc*>(vdesc.p);
      a.tile_start = reinterpret_cast<const int*>(vtiles.p);
    } else {
      a.inline_one = 1;
      a.one = base_desc(s, c64);
      a.one.x = s->A.p;
      a.one.y = s->B.p;
    }
    a.mode = kModeApply;
    for (int it = 0; it < 2; ++it) CKI(launch_plan(pl, a, st));  // warm-up
    CK(cudaEventRecord(e0, st));
    for (int it = 0; it < 5; ++it) CKI(launch_plan(pl, a, st));
    CK(cudaEventRecord(e1, st));
    CK(cudaEventSynchronize(e1));
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, e0, e1));
    if (pl.half.vm && pl.half.passes > 1 && !pl.half.hybrid)  // the step then reads passes - 1 more H q blocks (~6 TB/s)
      ms += 5.0f * (float)((double)(pl.half.passes - 1) * (double)vbytes * R / 6.0e9);
    if (ms < best) {
      best = ms;
      pick = sh;
    }
  }
  RotPlan rp;  // runs from random vectors: the rotated-basis H.v
  if (s->hs.all_half && !lean) {
    ftlm_status rs = make_rot(s, R, c64, rp, st);
    if (rs != FTLM_OK) return rs;
  }
  if (rp.on) {
    RotArgs a = rot_args(s, rp, c64);
    a.x = s->A.p;
    a.y = s->B.p;
    a.W = s->rW.p;
    {  // after products still in flight, which use these blocks too
      std::lock_guard<std::mutex> lk(s->apply_mu);
      if (s->apply_used) CK(cudaStreamWaitEvent(st, s->ev_apply, 0));
    }
    for (int it = 0; it < 7; ++it) {  // two warm-up products, five timed
      if (it == 2) CK(cudaEventRecord(e0, st));
      ftlm_status rs = enqueue_rot_passes(nullptr, s, rp, a, R, c64, nullptr, st);
      if (rs != FTLM_OK) return rs;
    }
    CK(cudaEventRecord(e1, st));
    CK(cudaEventSynchronize(e1));
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, e0, e1));
    pick.rot = ms < best;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  vdesc.release();  // (every candidate's launches have completed: each ends with an event wait)
  vtiles.release();
  std::lock_guard<std::mutex> lk(g_mu);
  g_shapes[key] = pick;
  return FTLM_OK;
}

ftlm_status check_block_args(const ftlm_system* s, const void* x, const void* y, int nvec, ftlm_dtype dtype) {
  if (!s) return fail(FTLM_ERR_INVALID_ARG, "system is NULL");
  if (dtype != FTLM_C64 && dtype != FTLM_C128) return fail(FTLM_ERR_INVALID_ARG, "unknown dtype");
  const int c64 = dtype == FTLM_C64;
  if (nvec < 1 || nvec > max_vectors(c64))
    return fail(FTLM_ERR_INVALID_ARG, "nvec must be in 1.." + std::to_string(max_vectors(c64)));
  if (!x || !y) return fail(FTLM_ERR_INVALID_ARG, "vector blocks must not be NULL");
  if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15)
    return fail(FTLM_ERR_INVALID_ARG, "vector blocks must be 16-byte aligned");
  return FTLM_OK;
}

// The coupling tables and the workspace of a system live on the device that
// was current when it was created; work for it must be enqueued with that
// device current (pointers of one device are not valid on another).
ftlm_status check_device(const ftlm_system* s) {
  int dev = 0;
  CK(cudaGetDevice(&dev));
  if (dev != s->device)
    return fail(FTLM_ERR_INVALID_ARG, "system lives on device " + std::to_string(s->device) + ", current device is " +
                                          std::to_string(dev));
  return FTLM_OK;
}

// The checks that ftlm_apply_h and ftlm_apply_sdir share.
ftlm_status check_product(const ftlm_system* s, const void* x, const void* y, int nvec, ftlm_dtype dtype) {
  ftlm_status v = check_block_args(s, x, y, nvec, dtype);
  if (v != FTLM_OK) return v;
  v = check_device(s);
  if (v != FTLM_OK) return v;
  const size_t bytes = (size_t)s->hs.dim * nvec * (dtype == FTLM_C64 ? 8 : 16);
  const uintptr_t xa = reinterpret_cast<uintptr_t>(x), ya = reinterpret_cast<uintptr_t>(y);
  if (xa < ya + bytes && ya < xa + bytes) return fail(FTLM_ERR_INVALID_ARG, "x and y overlap");
  return FTLM_OK;
}

ftlm_status apply_h_entry(const ftlm_system* cs, const void* x, void* y, int nvec, ftlm_dtype dtype, void* stream,
                          bool lean) {
  const int c64 = dtype == FTLM_C64;
  ftlm_system* s = const_cast<ftlm_system*>(cs);
  const cudaStream_t st = pick_stream(s, stream);
  // Everything but the gathers on the caller's layout keeps blocks, tables or events
  // of the system, which a captured call may neither allocate nor write (a table's
  // writing would only happen when the graph runs) nor wait for: such a call takes
  // those gathers.  So does one whose shape was set.
  const bool plain = stream_captures(st) || has_shape_override(s, nvec, c64);
  if (!plain && !lean && stored_pays(s, c64, nvec)) {  // small systems: stored rows
    StoredArgs a;
    bool ok = false;
    ftlm_status rs = ensure_stored(s, c64, stored_limit(s, c64), nvec, st, a.rows, ok);
    if (rs != FTLM_OK) return rs;
    if (ok) {
      a.x = x;
      a.y = y;
      a.dim = (long long)s->hs.dim;
      a.rs = a.R = nvec;
      a.vs = 1;
      CKI(launch_stored_product(a, stored_group(s->hs.dim, nvec), c64, st));
      return FTLM_OK;
    }
  }
  Plan pl;
  std::vector<ftlm_system*> one{s};
  if (!plain) {
    // spin-1/2 blocks on the default plan: transpose to vector-major (one vector
    // is), the rotated-basis passes, the runs' gather for the vectors that these
    // found not to be dense; transpose back
    Plan vp;
    ftlm_status ps = make_plan(one, nvec, c64, vp, nullptr, true);
    RotPlan rp;
    const bool vm = ps == FTLM_OK && vp.half.on && vp.half.vm && vp.half.passes == 1 && !vp.half.hybrid;
    bool rot = vm && !lean && rot_shape(s, nvec, c64, rp);
    if (vm && (nvec > 1 || rot)) {
      // the system's blocks are shared by its calls: a call waits for the
      // previous one's kernels (on whatever stream it ran) before reusing them
      std::unique_lock<std::mutex> run_lk(s->mu, std::defer_lock);
      if (nvec > 1) run_lk.lock();  // (the unit tables and W blocks belong to runs too)
      std::lock_guard<std::mutex> lk(s->apply_mu);
      const size_t block = (size_t)s->hs.dim * nvec * (c64 ? 8 : 16);
      auto grow = [&](DevBuf& b, size_t bytes) {
        if (b.bytes >= bytes) return cudaSuccess;
        if (s->apply_used) cudaEventSynchronize(s->ev_apply);
        return b.ensure(bytes);
      };
      if (nvec > 1) {
        CK(grow(s->Ta, block));
        CK(grow(s->Tb, block));
      }
      const size_t sbytes = (sizeof(RotDensity) + sizeof(int)) * nvec;
      if (rot && nvec > 1) rot = grow_rot_blocks(s, rot_block_bytes(s, rp, c64));  // (a run waits for ev_apply)
      else if (rot) rot = grow(s->Tw, rot_block_bytes(s, rp, c64)) == cudaSuccess;
      if (rot) rot = grow(s->Ts, sbytes) == cudaSuccess;
      cudaGetLastError();
      if (nvec > 1 || rot) {
        if (s->apply_used) CK(cudaStreamWaitEvent(st, s->ev_apply, 0));
        ftlm_status ut = nvec > 1 ? ensure_unit_tables(s, vp.half.K, c64, st) : FTLM_OK;
        if (ut != FTLM_OK) return ut;
        if (rot) {
          ut = ensure_rot_tables(s, rp, c64, st, rot);
          if (ut != FTLM_OK) return ut;
        }
        const void* xv = nvec > 1 ? s->Ta.p : x;
        void* yv = nvec > 1 ? s->Tb.p : y;
        if (nvec > 1) CKI(launch_to_vector_major(x, s->Ta.p, (long long)s->hs.dim, nvec, c64, st));
        LaunchArgs a = vp.base;
        if (rot) {
          CK(cudaMemsetAsync(s->Ts.p, 0, sbytes, st));
          RotArgs r = rot_args(s, rp, c64);
          r.x = const_cast<void*>(xv);
          r.y = yv;
          r.W = nvec > 1 ? s->rW.p : s->Tw.p;
          r.density = reinterpret_cast<RotDensity*>(s->Ts.p);
          r.sparse = reinterpret_cast<int*>(r.density + nvec);
          ut = enqueue_rot_passes(nullptr, s, rp, r, nvec, c64, nullptr, st);
          if (ut != FTLM_OK) return ut;
          a.only_if = r.sparse;
        }
        a.unit_tab = nvec > 1 ? s->ut[c64 ? 1 : 0].p : nullptr;
        a.inline_one = 1;
        a.one = base_desc(s, c64);
        a.one.x = xv;
        a.one.y = yv;
        a.vm_stride = (long long)s->hs.dim * (c64 ? 8 : 16);
        a.mode = kModeApply;
        a.gather_alpha = 0;
        CKI(launch_plan(vp, a, st));
        if (nvec > 1) CKI(launch_from_vector_major(s->Tb.p, y, (long long)s->hs.dim, nvec, c64, st));
        CK(cudaEventRecord(s->ev_apply, st));
        s->apply_used = true;
        return FTLM_OK;
      }
    }
  }
  if (c64 && nvec > 1 && !plain) {
    // other spins, complex64 blocks: transposed to the tile gather's layout and back
    Plan tp;
    ftlm_status ps = make_plan(one, nvec, c64, tp, nullptr, true);
    if (ps == FTLM_OK && tp.gen_vm && tp.tile.V) {
      std::lock_guard<std::mutex> lk(s->apply_mu);
      const size_t block = (size_t)s->hs.dim * nvec * 8;
      bool fits = true;
      for (DevBuf* b : {&s->Ta, &s->Tb}) {
        if (b->bytes < block && s->apply_used) CK(cudaEventSynchronize(s->ev_apply));
        fits = fits && b->ensure(block) == cudaSuccess;
      }
      cudaGetLastError();
      if (fits) {
        if (s->apply_used) CK(cudaStreamWaitEvent(st, s->ev_apply, 0));
        CKI(launch_to_vector_major(x, s->Ta.p, (long long)s->hs.dim, nvec, c64, st));
        LaunchArgs a = tp.base;
        a.inline_one = 1;
        a.one = base_desc(s, c64);
        a.one.x = s->Ta.p;
        a.one.y = s->Tb.p;
        a.vm_stride = (long long)s->hs.dim * 8;
        a.tiles_per_vg = tp.gvm_ntiles / tp.gvm_groups;
        a.mode = kModeApply;
        CKI(launch_plan(tp, a, st));
        CKI(launch_from_vector_major(s->Tb.p, y, (long long)s->hs.dim, nvec, c64, st));
        CK(cudaEventRecord(s->ev_apply, st));
        s->apply_used = true;
        return FTLM_OK;
      }
    }
  }
  // one vector: the row-major and the vector-major layouts coincide, so H.v may
  // use the vector-major gather
  ftlm_status ps = make_plan(one, nvec, c64, pl, nullptr, nvec == 1);
  if (ps != FTLM_OK) return ps;
  if (pl.half.vm && pl.half.passes > 1) {  // the multi-pass form writes one block per pass: not for a caller's y
    ps = make_plan(one, nvec, c64, pl);
    if (ps != FTLM_OK) return ps;
  }
  LaunchArgs a = pl.base;
  a.inline_one = 1;
  a.one = base_desc(s, c64);
  a.one.x = x;
  a.one.y = y;
  a.mode = kModeApply;
  CKI(launch_plan(pl, a, st));
  return FTLM_OK;
}

// ---- the allocation-free start block ------------------------------------------
//
// Scratch of ftlm_start_block_noalloc: a file-scope device array instead of
// cudaMalloc.  Layout (doubles): [0, 8) arrival counter; then the per-vector
// scalars of a one-step run (alpha, beta, p, sigma, scale, active, M_eff);
// then the per-CTA partial sums [kNoAllocMaxCtas][kNoAllocMaxVectors][kNumPartials].
constexpr int kNoAllocMaxVectors = 64;
constexpr int kNoAllocMaxCtas = 256;
constexpr size_t kNoAllocScalars = 16 * (size_t)kNoAllocMaxVectors;
constexpr size_t kNoAllocDoubles = 8 + kNoAllocScalars + (size_t)kNoAllocMaxCtas * kNoAllocMaxVectors * kNumPartials;
__device__ __align__(256) double g_noalloc_scratch[kNoAllocDoubles];

constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
void* g_noalloc_addr[kNoAllocMaxDevices] = {};  // device address of the array, per device

// (arguments as ftlm_system_create)
ftlm_status create_system(int n_sites, const int* two_s, const double* J, const double* d_ion, const double* e_axes,
                          double g, const double* B, const double* pos, const ftlm_constants* k, ftlm_system** out) {
  std::string msg;
  auto s = std::make_unique<ftlm_system>();
  ftlm_status st = build_host_system(n_sites, two_s, J, d_ion, e_axes, g, B, pos, k, s->hs, msg);
  if (st != FTLM_OK) return fail(st, msg);
  CK(cudaGetDevice(&s->device));
  CK(cudaStreamCreateWithFlags(&s->own_stream, cudaStreamNonBlocking));
  CK(cudaEventCreateWithFlags(&s->ev_in, cudaEventDisableTiming));
  CK(cudaEventCreateWithFlags(&s->ev_out, cudaEventDisableTiming));
  CK(cudaEventCreateWithFlags(&s->ev_apply, cudaEventDisableTiming));
  {
    std::lock_guard<std::mutex> lk(g_mu);
    s->id = g_next_id++;
  }
  const HostSystem& hs = s->hs;
  s->row_bound = (size_t)stored_row_bound(hs);
  stored_row_work(hs, s->row_entries, s->row_pairs);
  s->rot = std::make_unique<RotDirs>();
  if (!rot_directions(hs, *s->rot)) s->rot.reset();
  std::vector<float> tf(hs.tab.begin(), hs.tab.end());
  std::vector<long long> stv(hs.stride.begin(), hs.stride.end());
  cudaError_t e = s->tab_d.ensure(hs.tab.size() * sizeof(double));
  if (e == cudaSuccess) e = s->tab_f.ensure(tf.size() * sizeof(float));
  if (e == cudaSuccess) e = s->stride.ensure(stv.size() * sizeof(long long));
  if (e == cudaSuccess) e = s->q.ensure(hs.q.size() * sizeof(int));
  if (e == cudaSuccess) e = cudaMemcpy(s->tab_d.p, hs.tab.data(), hs.tab.size() * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(s->tab_f.p, tf.data(), tf.size() * sizeof(float), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(s->stride.p, stv.data(), stv.size() * sizeof(long long), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(s->q.p, hs.q.data(), hs.q.size() * sizeof(int), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    cudaGetLastError();
    s->tab_d.release();
    s->tab_f.release();
    s->stride.release();
    s->q.release();
    cudaEventDestroy(s->ev_in);
    cudaEventDestroy(s->ev_out);
    cudaEventDestroy(s->ev_apply);
    cudaStreamDestroy(s->own_stream);
    return fail(e == cudaErrorMemoryAllocation ? FTLM_ERR_OUT_OF_MEMORY : FTLM_ERR_CUDA,
                std::string("uploading the coupling tables: ") + cudaGetErrorString(e));
  }
  {
    std::lock_guard<std::mutex> lk(g_live_mu);
    g_live.push_back(s.get());
  }
  *out = s.release();
  return FTLM_OK;
}

}  // namespace

// ---------------------------------------------------------------------------
// exported entry points
// ---------------------------------------------------------------------------
extern "C" {

ftlm_status ftlm_start_block_noalloc(const ftlm_system* cs, uint64_t seed, uint64_t vec_offset, void* out, int nvec,
                                     ftlm_dtype dtype, void* stream) {
  ftlm_status v = check_block_args(cs, out, out, nvec, dtype);
  if (v != FTLM_OK) return v;
  if (nvec > kNoAllocMaxVectors)
    return fail(FTLM_ERR_INVALID_ARG, "ftlm_start_block_noalloc: nvec " + std::to_string(nvec) +
                                          " exceeds the static scratch (at most " +
                                          std::to_string(kNoAllocMaxVectors) + " vectors)");
  const int c64 = dtype == FTLM_C64;
  ftlm_system* s = const_cast<ftlm_system*>(cs);
  std::lock_guard<std::mutex> lk(s->mu);
  v = check_device(s);
  if (v != FTLM_OK) return v;
  const int dev = s->device;
  if (dev < 0 || dev >= kNoAllocMaxDevices) return fail(FTLM_ERR_UNSUPPORTED, "device ordinal too large");
  void* base = nullptr;
  {
    // once per device, with that device current: the host-side name of the
    // array is not a device address, so ask the runtime for it
    std::lock_guard<std::mutex> l2(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
      void* p = nullptr;
      CK(cudaGetSymbolAddress(&p, g_noalloc_scratch));
      g_noalloc_addr[dev] = p;
    }
    base = g_noalloc_addr[dev];
  }
  double* scratch = reinterpret_cast<double*>(base);
  unsigned* counter = reinterpret_cast<unsigned*>(scratch);
  double* scal = scratch + 8;
  double* partials = scal + kNoAllocScalars;
  cudaStream_t st = pick_stream(s, stream);
  Plan pl;
  std::vector<ftlm_system*> one{s};
  ftlm_status ps = make_plan(one, nvec, c64, pl);
  if (ps != FTLM_OK) return ps;
  const int grid = std::min(pl.grid, kNoAllocMaxCtas);
  // the arrival counter must start at zero; everything else is overwritten
  CK(cudaMemsetAsync(counter, 0, sizeof(unsigned), st));
  InstDesc h = base_desc(s, c64);
  CKI(launch_start_random(&h, nullptr, nvec, seed, vec_offset, out, c64, st));
  LaunchArgs a = pl.base;
  a.inline_one = 1;
  a.one = h;
  a.one.x = out;
  a.one.y = out;
  a.one.M = 1;
  a.one.sc = scalars_at(scal, nvec, 1);
  a.partials = partials;
  a.counter = counter;
  a.mode = kModeStartNorm;
  CKI(launch_rows(a, c64, grid, pl.sh.threads, pl.smem, st));
  a.mode = kModeScale;
  CKI(launch_rows(a, c64, grid, pl.sh.threads, pl.smem, st));
  return FTLM_OK;
}

ftlm_status ftlm_system_create(int n_sites, const int* two_s, const double* J, const double* d_ion,
                               const double* e_axes, double g, const double B[3], const double* pos,
                               const ftlm_constants* k, ftlm_system** out) {
  if (!out) return fail(FTLM_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  return with_memory(nullptr, 0, [&](bool) { return create_system(n_sites, two_s, J, d_ion, e_axes, g, B, pos, k, out); });
}

void ftlm_system_destroy(ftlm_system* s) {
  if (!s) return;
  {
    std::lock_guard<std::mutex> lk(g_live_mu);
    g_live.erase(std::remove(g_live.begin(), g_live.end(), s), g_live.end());
  }
  wait_for_device();  // the system's buffers may be in use on any stream
  purge_ctx_of(s->id);
  for (DevBuf* b : {&s->tab_f, &s->tab_d, &s->stride, &s->q, &s->A, &s->B, &s->U, &s->scal, &s->ep, &s->ecnt,
                    &s->esc, &s->Hq, &s->Vs, &s->Wc, &s->Od, &s->Gre, &s->Ta, &s->Tb, &s->ut[0], &s->ut[1], &s->Ws, &s->rD[0], &s->rD[1], &s->rW, &s->rpart, &s->Tw, &s->Ts})
    b->release();
  for (DevBuf& b : s->rows) release_stored(b);
  cudaEventDestroy(s->ev_in);
  cudaEventDestroy(s->ev_out);
  cudaEventDestroy(s->ev_apply);
  for (cudaEvent_t e : {s->ev_rows[0], s->ev_rows[1], s->ev_rot[0], s->ev_rot[1]})
    if (e) cudaEventDestroy(e);
  cudaStreamDestroy(s->own_stream);
  delete s;
}

uint64_t ftlm_system_dim(const ftlm_system* s) { return s ? s->hs.dim : 0; }

uint64_t ftlm_system_table_bytes(const ftlm_system* s) {
  if (!s) return 0;
  return (uint64_t)s->hs.tab.size() * (sizeof(double) + sizeof(float)) +
         (uint64_t)s->hs.n * (sizeof(long long) + sizeof(int));
}

ftlm_status ftlm_apply_h(const ftlm_system* s, const void* x, void* y, int nvec, ftlm_dtype dtype, void* stream) {
  ftlm_status v = check_product(s, x, y, nvec, dtype);
  if (v != FTLM_OK) return v;
  ftlm_system* ms = const_cast<ftlm_system*>(s);
  return with_memory(&ms, 1, [&](bool lean) { return apply_h_entry(s, x, y, nvec, dtype, stream, lean); });
}

ftlm_status ftlm_apply_sdir(const ftlm_system* s, const double* u, const void* x, void* y, int nvec,
                            ftlm_dtype dtype, void* stream) {
  if (u && !(std::isfinite(u[0]) && std::isfinite(u[1]) && std::isfinite(u[2])))
    return fail(FTLM_ERR_INVALID_ARG, "u must be finite");
  ftlm_status v = check_product(s, x, y, nvec, dtype);
  if (v != FTLM_OK) return v;
  const int c64 = dtype == FTLM_C64;
  SdirArgs a = sdir_args(s, c64, nvec, x, y);
  observable_coefs(s->hs, u, a.obs);
  CKI(launch_sdir(a, s->hs.q.data(), c64, false, pick_stream(s, stream)));
  return FTLM_OK;
}

}  // extern "C"

namespace {

// Normalised start block: plain random vectors, or pairs of time-reversed ones.
ftlm_status start_block_impl(const ftlm_system* cs, uint64_t seed, uint64_t vec_offset, void* out, int nvec,
                             ftlm_dtype dtype, void* stream, bool pairs) {
  ftlm_status v = check_block_args(cs, out, out, nvec, dtype);
  if (v != FTLM_OK) return v;
  const int c64 = dtype == FTLM_C64;
  ftlm_system* s = const_cast<ftlm_system*>(cs);
  std::lock_guard<std::mutex> lk(s->mu);
  v = check_device(s);
  if (v != FTLM_OK) return v;
  cudaStream_t st = pick_stream(s, stream);
  Plan pl;
  std::vector<ftlm_system*> one{s};
  ftlm_status ps = make_plan(one, nvec, c64, pl);
  if (ps != FTLM_OK) return ps;
  // scratch owned by the system: per-CTA partials, the arrival counter and sigma_0
  const size_t pbytes = sizeof(double) * (size_t)pl.grid * nvec * kNumPartials;
  if (s->ep.bytes < pbytes) CK(s->ep.ensure(pbytes));
  if (!s->ecnt.p) {
    CK(s->ecnt.ensure(64));
    CK(cudaMemsetAsync(s->ecnt.p, 0, 64, st));
  }
  if (s->esc.bytes < scalar_bytes(nvec, 1)) CK(s->esc.ensure(scalar_bytes(nvec, 1)));
  InstDesc h = base_desc(s, c64);
  if (pairs) CKI(launch_start_pairs(&h, nvec, seed, vec_offset, out, c64, st, 0));
  else CKI(launch_start_random(&h, nullptr, nvec, seed, vec_offset, out, c64, st));
  LaunchArgs a = pl.base;
  a.inline_one = 1;
  a.one = h;
  a.one.x = out;
  a.one.y = out;
  a.one.M = 1;
  a.one.sc = scalars_at(s->esc.p, nvec, 1);
  a.partials = reinterpret_cast<double*>(s->ep.p);
  a.counter = reinterpret_cast<unsigned*>(s->ecnt.p);
  a.mode = kModeStartNorm;
  CKI(launch_rows(a, c64, pl.grid, pl.sh.threads, pl.smem, st));
  a.mode = kModeScale;
  CKI(launch_rows(a, c64, pl.grid, pl.sh.threads, pl.smem, st));
  return FTLM_OK;
}

ftlm_status start_block_entry(const ftlm_system* cs, uint64_t seed, uint64_t vec_offset, void* out, int nvec,
                              ftlm_dtype dtype, void* stream, bool pairs) {
  ftlm_status v = check_block_args(cs, out, out, nvec, dtype);
  if (v != FTLM_OK) return v;
  ftlm_system* s = const_cast<ftlm_system*>(cs);
  return with_memory(&s, 1, [&](bool) { return start_block_impl(cs, seed, vec_offset, out, nvec, dtype, stream, pairs); });
}

}  // namespace

extern "C" {

ftlm_status ftlm_start_block(const ftlm_system* cs, uint64_t seed, uint64_t vec_offset, void* out, int nvec,
                             ftlm_dtype dtype, void* stream) {
  return start_block_entry(cs, seed, vec_offset, out, nvec, dtype, stream, false);
}

ftlm_status ftlm_start_pairs(const ftlm_system* cs, uint64_t seed, uint64_t vec_offset, void* out, int nvec,
                             ftlm_dtype dtype, void* stream) {
  return start_block_entry(cs, seed, vec_offset, out, nvec, dtype, stream, true);
}

ftlm_status ftlm_time_reverse(const ftlm_system* cs, const void* x, void* y, int nvec, ftlm_dtype dtype,
                              void* stream) {
  ftlm_status v = check_block_args(cs, x, y, nvec, dtype);
  if (v != FTLM_OK) return v;
  const int c64 = dtype == FTLM_C64;
  const size_t bytes = (size_t)cs->hs.dim * nvec * (c64 ? 8 : 16);
  const uintptr_t xa = reinterpret_cast<uintptr_t>(x), ya = reinterpret_cast<uintptr_t>(y);
  if (xa < ya + bytes && ya < xa + bytes) return fail(FTLM_ERR_INVALID_ARG, "x and y overlap");
  v = check_device(cs);
  if (v != FTLM_OK) return v;
  InstDesc h = base_desc(cs, c64);
  CKI(launch_time_reverse(&h, x, y, nvec, c64, pick_stream(cs, stream)));
  return FTLM_OK;
}

ftlm_status ftlm_run(const ftlm_system* s, const ftlm_run_params* p, ftlm_result* res) {
  ftlm_system* ms = const_cast<ftlm_system*>(s);
  ftlm_status pv = validate_params(p, {ms});  // host-only: before any lock or CUDA call
  if (pv != FTLM_OK) return pv;
  return with_memory(&ms, 1, [&](bool lean) -> ftlm_status {
    std::lock_guard<std::mutex> lk(ms->mu);
    // stored rows have no shape to choose, and every gather is slower on systems that small
    if (p->autotune && (lean || !run_stores({ms}, p->R, p->M, p->dtype == FTLM_C64))) {
      ftlm_status vs = check_device(ms);
      if (vs != FTLM_OK) return vs;
      ftlm_status a = autotune(ms, p->R, p->dtype == FTLM_C64, pick_stream(ms, p->stream), lean);
      if (a != FTLM_OK) return a;
    }
    return run_impl({ms}, p, res, lean);
  });
}

ftlm_status ftlm_run_batch(int n, const ftlm_system* const* systems, const ftlm_run_params* p,
                           ftlm_result* results) {
  if (n < 1 || !systems || !results) return fail(FTLM_ERR_INVALID_ARG, "empty batch");
  std::vector<ftlm_system*> v;
  for (int k = 0; k < n; ++k) {
    if (!systems[k]) return fail(FTLM_ERR_INVALID_ARG, "system is NULL");
    for (auto* o : v)
      if (o == systems[k]) return fail(FTLM_ERR_INVALID_ARG, "a system appears twice in the batch");
    v.push_back(const_cast<ftlm_system*>(systems[k]));
  }
  return with_memory(v.data(), (int)v.size(), [&](bool lean) -> ftlm_status {
    std::vector<ftlm_system*> order = v;  // lock in address order
    std::sort(order.begin(), order.end());
    std::vector<std::unique_lock<std::mutex>> locks;
    for (auto* s : order) locks.emplace_back(s->mu);
    ftlm_status vs = validate_params(p, v);
    if (vs != FTLM_OK) return vs;
    if (p->autotune && (lean || !run_stores(v, p->R, p->M, p->dtype == FTLM_C64))) {
      for (auto* s : v) {
        vs = check_device(s);
        if (vs != FTLM_OK) return vs;
      }
      ftlm_system* big = v[0];
      for (auto* s : v)
        if (s->hs.dim > big->hs.dim) big = s;
      ftlm_status a = autotune(big, p->R, p->dtype == FTLM_C64, pick_stream(v[0], p->stream), lean);
      if (a != FTLM_OK) return a;
    }
    return run_impl(v, p, results, lean);
  });
}

ftlm_status ftlm_tune_shape(const ftlm_system* s, int nvec, ftlm_dtype dtype, int cube_bits, int group_vectors,
                            int tile_cubes, int multipass) {
  if (!s) return fail(FTLM_ERR_INVALID_ARG, "system is NULL");
  if (dtype != FTLM_C64 && dtype != FTLM_C128) return fail(FTLM_ERR_INVALID_ARG, "unknown dtype");
  const int c64 = dtype == FTLM_C64;
  if (nvec < 1 || nvec > max_vectors(c64)) return fail(FTLM_ERR_INVALID_ARG, "nvec out of range");
  ShapeKey key{s->hs.n, s->hs.qmax, nvec, c64, (long long)s->hs.dim};
  if (cube_bits < 0) {  // forget the override (and any autotuned shape)
    std::lock_guard<std::mutex> lk(g_mu);
    g_shapes.erase(key);
    return FTLM_OK;
  }
  Shape sh = default_shape(nvec, c64);
  sh.explicit_general = cube_bits == 0 && multipass == 0;
  if (cube_bits == 0 && multipass != 0) {  // the vector-major general gather
    if (multipass != 1) return fail(FTLM_ERR_INVALID_ARG, "multipass must be 0 or 1 with cube_bits 0");
    if (group_vectors < 0 || group_vectors > 8 || nvec % std::max(1, group_vectors) != 0)
      return fail(FTLM_ERR_INVALID_ARG, "group_vectors must be 0 or a group size (4, 8) dividing nvec");
    if (tile_cubes < 1 || tile_cubes > 64) return fail(FTLM_ERR_INVALID_ARG, "tile_cubes must be in 1..64");
    sh.general_vm = 1;
    sh.gvm_cube = group_vectors;
    sh.gvm_rows = 256 * tile_cubes;
  }
  if (cube_bits != 0) {
    if (!s->hs.all_half) return fail(FTLM_ERR_UNSUPPORTED, "register cubes need every site s = 1/2");
    if (cube_bits < 2 || cube_bits > 4 || s->hs.n < cube_bits + 2)
      return fail(FTLM_ERR_INVALID_ARG, "cube_bits must be 2..4 and at most n_sites - 2");
    if (multipass < 0 || multipass > 9) return fail(FTLM_ERR_INVALID_ARG, "multipass must be in 0..9");
    if (multipass >= 8 && (cube_bits < 3 || s->hs.n < kVmLaneBits + 2 * cube_bits))
      return fail(FTLM_ERR_INVALID_ARG, "the two-pass form needs cube_bits 3..4 and n_sites >= 5 + 2 cube_bits");
    if (multipass >= 3 && (cube_bits < 3 || s->hs.n < kVmLaneBits + cube_bits))
      return fail(FTLM_ERR_INVALID_ARG, "the vector-major kernel needs cube_bits 3..4 and n_sites >= 5 + cube_bits");
    if (multipass < 3 && (group_vectors < 1 || group_vectors > nvec || group_vectors > 256))
      return fail(FTLM_ERR_INVALID_ARG, "group_vectors must be in 1..min(nvec, 256)");
    if (tile_cubes < 1 || tile_cubes > 64) return fail(FTLM_ERR_INVALID_ARG, "tile_cubes must be in 1..64");
    sh.half_K = cube_bits;
    sh.Rg = multipass >= 3 ? largest_divisor_at_most(nvec, 16) : group_vectors;  // row-major fallback for apply_h
    sh.half_rows = tile_cubes;
    sh.half_multipass = (multipass == 1 || multipass == 5 || multipass == 7) ? 1 : 0;
    sh.half_hybrid = multipass >= 8 ? 1 : 0;
    // 2 and 4: 3-CTA register budget; 6, 7 and 8: one 512-thread CTA per SM
    sh.half_min_blocks = (multipass == 2 || multipass == 4) ? 3 : ((multipass >= 6 && multipass <= 8) ? 1 : 2);
    sh.half_vm = multipass >= 3 ? 1 : 0;
  }
  std::lock_guard<std::mutex> lk(g_mu);
  g_shapes[key] = sh;
  return FTLM_OK;
}

ftlm_status ftlm_sums(int R, int M, const int* M_eff, const double* alpha, const double* beta, const double* p,
                      double dim, double g, const double* T, int nT, ftlm_result* res) {
  std::string msg;
  ftlm_status s = host_sums(R, M, M_eff, alpha, beta, p, dim, g, T, nT, res, msg);
  if (s != FTLM_OK) return fail(s, msg);
  return FTLM_OK;
}

}  // extern "C"

struct ftlm_csr {
  int device = 0;
  int c64 = 1;
  long long dim = 0;
  uint64_t nnz = 0;
  DevBuf rp, col, val;
  DevBuf counts;  // of the rows, while it is assembled
  ~ftlm_csr() {
    for (DevBuf* b : {&rp, &col, &val, &counts}) b->release();
  }
};

namespace {
ftlm_status create_csr(const ftlm_system* s, int c64, ftlm_csr** out) {
  const long long dim = (long long)s->hs.dim;
  auto m = std::make_unique<ftlm_csr>();
  m->device = s->device;
  m->c64 = c64;
  m->dim = dim;
  LaunchArgs a;
  a.inline_one = 1;
  a.one = base_desc(s, c64);
  a.n_inst = 1;
  a.tab_reals = s->hs.lay.total;
  a.max_n = s->hs.n;
  const size_t smem = csr_smem_bytes(a, c64);
  if (smem > 227 * 1024) return fail(FTLM_ERR_UNSUPPORTED, "coupling tables do not fit in shared memory");
  CKI(csr_prepare(std::max<size_t>(smem, 48 * 1024)));
  cudaStream_t st = s->own_stream;
  if (m->counts.ensure(sizeof(int) * (size_t)dim) != cudaSuccess || m->rp.ensure(sizeof(long long) * (size_t)(dim + 1)) != cudaSuccess)
    return fail(FTLM_ERR_OUT_OF_MEMORY, "row pointers");
  CKI(launch_csr_count(a, c64, smem, reinterpret_cast<int*>(m->counts.p), st));
  CKI(csr_scan(reinterpret_cast<const int*>(m->counts.p), reinterpret_cast<long long*>(m->rp.p), dim, st));
  long long nnz = 0;
  CK(cudaMemcpyAsync(&nnz, reinterpret_cast<long long*>(m->rp.p) + dim, sizeof(long long), cudaMemcpyDeviceToHost, st));
  CK(cudaStreamSynchronize(st));
  m->counts.release();
  m->nnz = (uint64_t)nnz;
  if (m->col.ensure(sizeof(int) * (size_t)nnz) != cudaSuccess || m->val.ensure((size_t)nnz * (c64 ? 8 : 16)) != cudaSuccess)
    return fail(FTLM_ERR_OUT_OF_MEMORY, "stored matrix of " + std::to_string(nnz) + " elements");
  CKI(launch_csr_fill(a, c64, smem, reinterpret_cast<const long long*>(m->rp.p), reinterpret_cast<int*>(m->col.p),
                      m->val.p, st));
  CK(cudaStreamSynchronize(st));
  *out = m.release();
  return FTLM_OK;
}
}  // namespace

extern "C" {

ftlm_status ftlm_csr_create(const ftlm_system* s, ftlm_dtype dtype, ftlm_csr** out) {
  if (!s || !out) return fail(FTLM_ERR_INVALID_ARG, "system or out is NULL");
  if (dtype != FTLM_C64 && dtype != FTLM_C128) return fail(FTLM_ERR_INVALID_ARG, "unknown dtype");
  *out = nullptr;
  const int c64 = dtype == FTLM_C64;
  const long long dim = (long long)s->hs.dim;
  if (dim >= (1ll << 31)) return fail(FTLM_ERR_UNSUPPORTED, "the stored matrix needs dim < 2^31 (32-bit columns)");
  int dev = 0;
  CK(cudaGetDevice(&dev));
  if (dev != s->device) return fail(FTLM_ERR_INVALID_ARG, "system lives on another device");
  ftlm_system* ms = const_cast<ftlm_system*>(s);
  return with_memory(&ms, 1, [&](bool) { return create_csr(s, c64, out); });
}

uint64_t ftlm_csr_nnz(const ftlm_csr* m) { return m ? m->nnz : 0; }

uint64_t ftlm_csr_bytes(const ftlm_csr* m) {
  return m ? m->rp.bytes + m->col.bytes + m->val.bytes : 0;
}

ftlm_status ftlm_csr_apply(const ftlm_csr* m, const void* x, void* y, int nvec, void* stream) {
  if (!m) return fail(FTLM_ERR_INVALID_ARG, "matrix is NULL");
  if (nvec < 1 || nvec > max_vectors(m->c64))
    return fail(FTLM_ERR_INVALID_ARG, "nvec must be in 1.." + std::to_string(max_vectors(m->c64)));
  if (!x || !y) return fail(FTLM_ERR_INVALID_ARG, "vector blocks must not be NULL");
  if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15)
    return fail(FTLM_ERR_INVALID_ARG, "vector blocks must be 16-byte aligned");
  const size_t bytes = (size_t)m->dim * nvec * (m->c64 ? 8 : 16);
  const uintptr_t xa = reinterpret_cast<uintptr_t>(x), ya = reinterpret_cast<uintptr_t>(y);
  if (xa < ya + bytes && ya < xa + bytes) return fail(FTLM_ERR_INVALID_ARG, "x and y overlap");
  int dev = 0;
  CK(cudaGetDevice(&dev));
  if (dev != m->device) return fail(FTLM_ERR_INVALID_ARG, "matrix lives on another device");
  CKI(launch_csr_spmm(m->dim, nvec, reinterpret_cast<const long long*>(m->rp.p), reinterpret_cast<const int*>(m->col.p),
                      m->val.p, x, y, m->c64, reinterpret_cast<cudaStream_t>(stream)));
  return FTLM_OK;
}

void ftlm_csr_destroy(ftlm_csr* m) { delete m; }

ftlm_status ftlm_sums_sym(int R, int M, const int* M_eff, const double* alpha, const double* beta,
                          const double* Omat, double g, const double* T, int nT, double* M_B_sym,
                          double* M_B_sym_imag) {
  if (!M_B_sym) return fail(FTLM_ERR_INVALID_ARG, "M_B_sym is NULL");
  for (int t = 0; T && t < nT; ++t)
    if (!(T[t] > 0.0) || !std::isfinite(T[t])) return fail(FTLM_ERR_INVALID_ARG, "temperatures must be > 0");
  std::string msg;
  ftlm_status s = host_sums_sym(R, M, M_eff, alpha, beta, Omat, g, T, nT, M_B_sym, M_B_sym_imag, msg);
  return s == FTLM_OK ? FTLM_OK : fail(s, msg);
}

const char* ftlm_last_error(void) { return g_err.c_str(); }

const char* ftlm_version(void) { return "ftlm-gb300 0.1 (sm_103a)"; }

}  // extern "C"
