// Launches of the plane-factorized z-march (linmarch.cuh) for the linear ops:
// Jacobian apply, PCG apply with the fused search-direction update, and the
// Chebyshev preconditioner step, in FP32 and FP64.
#include <cuda_runtime.h>

#include <type_traits>

#include "linmarch.cuh"
#include "mg.h"
#include "pcg_ops.cuh"

namespace qcad {

// The kernels take more than the default 48 KB of dynamic shared memory; the opt-in is
// set once per kernel and device.
template <class T, int BY, int R, class Op>
static void lin_launch(const Grid<T>& g, const Op& op, int kchunk, cudaStream_t s) {
  using S = LinShape<T, BY, R>;
  static bool attr_set[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 && !attr_set[dev]) {
    // the whole shared-memory carveout: blocks per SM are limited by shared memory otherwise
    if (cudaFuncSetAttribute(lin_march_kernel<T, BY, R, Op>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)S::dyn_bytes) == cudaSuccess &&
        cudaFuncSetAttribute(lin_march_kernel<T, BY, R, Op>, cudaFuncAttributePreferredSharedMemoryCarveout,
                             100) == cudaSuccess)
      attr_set[dev] = true;
  }
  const dim3 grid = lin_grid(g.nxn, g.nyn, g.nzn, BY, R, kchunk);
  note_launch(), lin_march_kernel<T, BY, R, Op><<<grid, dim3(32, BY), S::dyn_bytes, s>>>(g, op, kchunk);
}

// Default launch shapes fitted to the grid. A march block runs one node plane after the other, so
// its time is its planes; a fixed chunk of 16 planes left most SMs idle on small grids (6 blocks of
// 16 planes on 17 x 17 x 33 nodes: 223 us per FP64 apply) and half of the last wave on others.
// FP32 is bound by the latency of a plane: slots are resident blocks, 2 per SM at 8 warps and two
// rows. FP64 is bound by the SM's FP64 pipe, which all resident blocks share: one slot per SM, the
// cost of a plane is its rows, and smaller tiles (more halo, but more SMs at work) compete.
template <class T>
static LaunchCfg fit_lin(int nxn, int nyn, int nzn, LaunchCfg cfg) {
  if (!cfg.fit || cfg.variant < 2) return cfg;
  constexpr bool F32 = std::is_same<T, float>::value;
  const long long tx = (nxn + 29) / 30;
  const long long slots = (F32 ? 2LL : 1LL) * sm_count();
  const double over = F32 ? 3.0 : 2.0;
  auto tiles = [&](int tr) { return tx * ((nyn + tr - 3) / (tr - 2)); };
  static const int shape[3][2] = {{8, 2}, {4, 2}, {4, 1}};  // warps, rows per thread; FP32: the first
  double best = FIT_GAIN * 16 * march_planes(tiles(16), nzn, slots, over, cfg.kchunk);
  LaunchCfg out = cfg;
  for (int h = 0; h < (F32 ? 1 : 3); ++h) {
    const int tr = shape[h][0] * shape[h][1];
    double cost;
    const int kc = fit_chunk(tiles(tr), nzn, slots, over, 32, &cost);
    if (cost * tr < best) {
      best = cost * tr;
      out.by = shape[h][0];
      out.variant = shape[h][1] == 2 ? 3 : 2;
      out.kchunk = kc;
    }
  }
  return out;
}

// The shape that a launch with configuration cfg takes, with an activity map or without.
template <class T>
static LaunchCfg lin_shape(int nxn, int nyn, int nzn, LaunchCfg cfg, bool act) {
  const bool fit = cfg.fit;
  cfg = fit_lin<T>(nxn, nyn, nzn, cfg);
  // With an activity map a tile with response takes about six times as long as one without in FP64, so
  // the longest tile sets the time: half the chunk (FP64 solve of the 128 x 128 x 96 device 75 -> 67 ms;
  // FP32, bound by latency, was 5 % slower with it).
  if (sizeof(T) == 8 && fit && cfg.variant >= 2 && act && cfg.kchunk > 8) cfg.kchunk = 8;
  cfg.fit = false;
  return cfg;
}
LaunchCfg default_lin_shape(int precision, int nxn, int nyn, int nzn, bool act) {
  return precision == 0 ? lin_shape<double>(nxn, nyn, nzn, LaunchCfg(), act)
                        : lin_shape<float>(nxn, nyn, nzn, LaunchCfg(), act);
}

template <class T>
static bool has_act(const ApplyOp<T>& op) { return op.a.act != nullptr; }
template <class Op>
static bool has_act(const Op& op) { return op.v.act != nullptr; }

// Supported (warps, rows per thread): FP32 4/8/16/32 x 1 and 4/8/16 x 2; FP64 4/8 x 1 and
// 4/8 x 2 (shared memory). Other requests are clamped to the nearest supported shape.
template <class T, class Op>
static void run_lin(const Grid<T>& g, const Op& op, LaunchCfg cfg, cudaStream_t s) {
  cfg = lin_shape<T>(g.nxn, g.nyn, g.nzn, cfg, has_act(op));
  const int kc = cfg.kchunk > 0 ? (cfg.kchunk < 128 ? cfg.kchunk : 128) : 16;  // LinShape::ZMAX
  const bool two = cfg.variant == 3;
  if constexpr (std::is_same<T, float>::value) {
    if (two) {
      if (cfg.by == 4) lin_launch<T, 4, 2>(g, op, kc, s);
      else if (cfg.by >= 16) lin_launch<T, 16, 2>(g, op, kc, s);
      else lin_launch<T, 8, 2>(g, op, kc, s);
    } else {
      if (cfg.by == 4) lin_launch<T, 4, 1>(g, op, kc, s);
      else if (cfg.by == 16) lin_launch<T, 16, 1>(g, op, kc, s);
      else if (cfg.by >= 32) lin_launch<T, 32, 1>(g, op, kc, s);
      else lin_launch<T, 8, 1>(g, op, kc, s);
    }
  } else {
    if (two) {
      if (cfg.by == 4) lin_launch<T, 4, 2>(g, op, kc, s);
      else lin_launch<T, 8, 2>(g, op, kc, s);
    } else {
      if (cfg.by == 4) lin_launch<T, 4, 1>(g, op, kc, s);
      else lin_launch<T, 8, 1>(g, op, kc, s);
    }
  }
}

template <class T>
void launch_apply_lin(const Grid<T>& g, const ApplyArgs<T>& args, LaunchCfg cfg, cudaStream_t s) {
  ApplyOp<T> op = {};
  op.a = args;
  run_lin<T>(g, op, cfg, s);
}
template void launch_apply_lin<float>(const Grid<float>&, const ApplyArgs<float>&, LaunchCfg, cudaStream_t);
template void launch_apply_lin<double>(const Grid<double>&, const ApplyArgs<double>&, LaunchCfg, cudaStream_t);

template <class T>
void launch_pcg_apply_lin(const Grid<T>& g, PcgVecs<T> vecs, PcgScalars* sc, LaunchCfg cfg, cudaStream_t s) {
  PcgApplyOp<T> op = {};
  op.v = vecs;
  op.sc = sc;
  run_lin<T>(g, op, cfg, s);
}
template void launch_pcg_apply_lin<float>(const Grid<float>&, PcgVecs<float>, PcgScalars*, LaunchCfg, cudaStream_t);
template void launch_pcg_apply_lin<double>(const Grid<double>&, PcgVecs<double>, PcgScalars*, LaunchCfg,
                                           cudaStream_t);

template <class T>
void launch_cheb_step_lin(const Grid<T>& g, PcgVecs<T> vecs, PcgScalars* sc, int step, int last, LaunchCfg cfg,
                          cudaStream_t s) {
  ChebStepOp<T> op = {};
  op.v = vecs;
  op.sc = sc;
  op.step = step;
  op.last = last;
  run_lin<T>(g, op, cfg, s);
}
template void launch_cheb_step_lin<float>(const Grid<float>&, PcgVecs<float>, PcgScalars*, int, int, LaunchCfg,
                                          cudaStream_t);
template void launch_cheb_step_lin<double>(const Grid<double>&, PcgVecs<double>, PcgScalars*, int, int, LaunchCfg,
                                           cudaStream_t);

// ---------------------------------------------------------------------------
// Multigrid V-cycle on level 0 (the mesh itself): the residual after pre-smoothing,
// w = r - J zp with zp = d[0] = omega D^-1 r, and the post-smoothing step that also closes the
// PCG iteration, z = zq + omega D^-1 (r - J zq) with zq = d[1] = zp + P e (coarse correction),
// accumulating r.z and running the last block's bookkeeping as the Chebyshev step does.
template <class T>
struct MgResid0Op {
  static constexpr int NIN = 1;
  struct Pre {
    T r;
  };
  PcgVecs<T> v;
  PcgScalars* sc;
  __device__ bool skip() const { return sc->done != 0; }
  __device__ void set_vec(int) {}
  __device__ const T* coeffs() const { return v.c; }
  __device__ const unsigned char* act() const { return v.act; }
  __device__ const T* lin_src(int) const { return v.d[0]; }
  __device__ T lin_mix(T x0, T) const { return x0; }
  __device__ T lin_in(int n) const { return v.d[0][n]; }
  __device__ Pre lin_pre(int n) const { return Pre{v.r[n]}; }
  __device__ bool lin_dir() const { return true; }
  __device__ void lin_out(int n, const Pre& p, T, T y) { v.w[n] = p.r - y; }
  __device__ void finish() {}
};

template <class T>
struct MgPost0Op {
  static constexpr int NIN = 1;
  struct Pre {
    T r, dinv;
  };
  PcgVecs<T> v;
  PcgScalars* sc;
  const T* par;
  T om;
  int t, slot;
  T acc;
  __device__ bool skip() const { return sc->done != 0; }
  __device__ void set_vec(int) {
    t = sc->t;
    slot = sc->phase == 0 ? 0 : ((t + 1) & 3);
    om = mg_omega<T>(par, 0);
  }
  __device__ const T* coeffs() const { return v.c; }
  __device__ const unsigned char* act() const { return v.act; }
  __device__ const T* lin_src(int) const { return v.d[1]; }
  __device__ T lin_mix(T x0, T) const { return x0; }
  __device__ T lin_in(int n) const { return v.d[1][n]; }
  __device__ Pre lin_pre(int n) const { return Pre{v.r[n], v.dinv[n]}; }
  __device__ bool lin_dir() const { return true; }
  __device__ void lin_out(int n, const Pre& p, T zq, T y) {
    const T z = zq + om * p.dinv * (p.r - y);
    v.z[n] = z;
    acc += p.r * z;
  }
  __device__ void finish() {
    double s1[1] = {(double)acc};
    block_sum_atomic<1>(s1, &sc->rz[slot]);
    if (last_block(&sc->counter) && threadIdx.x == 0 && threadIdx.y == 0) pcg_finish(sc, t, 1.0);
  }
};

template <class T>
void launch_mg_resid0(const Grid<T>& g, PcgVecs<T> v, PcgScalars* sc, LaunchCfg cfg, cudaStream_t s) {
  MgResid0Op<T> op = {};
  op.v = v;
  op.sc = sc;
  run_lin<T>(g, op, cfg, s);
}
template void launch_mg_resid0<float>(const Grid<float>&, PcgVecs<float>, PcgScalars*, LaunchCfg, cudaStream_t);
template void launch_mg_resid0<double>(const Grid<double>&, PcgVecs<double>, PcgScalars*, LaunchCfg, cudaStream_t);

template <class T>
void launch_mg_post0(const Grid<T>& g, PcgVecs<T> v, PcgScalars* sc, const T* par, LaunchCfg cfg, cudaStream_t s) {
  MgPost0Op<T> op = {};
  op.v = v;
  op.sc = sc;
  op.par = par;
  run_lin<T>(g, op, cfg, s);
}
template void launch_mg_post0<float>(const Grid<float>&, PcgVecs<float>, PcgScalars*, const float*, LaunchCfg,
                                     cudaStream_t);
template void launch_mg_post0<double>(const Grid<double>&, PcgVecs<double>, PcgScalars*, const double*, LaunchCfg,
                                      cudaStream_t);

// Batched PCG apply: a work table maps each block to (instance, tile) of instances of different
// sizes; plane-factorized march with 8 warps and two rows per thread.
__device__ __forceinline__ int lin_batch_find(const BatchApplyEntry* tab, int n, int b) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].begin <= b)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

__global__ void __launch_bounds__(256, (lin_min_blocks<float, 8, 2>()))
    batch_lin_apply_kernel(const BatchApplyEntry* tab, int n_inst) {
  extern __shared__ __align__(16) unsigned char lin_dyn[];
  const int b = blockIdx.x;
  const BatchApplyEntry& e = tab[lin_batch_find(tab, n_inst, b)];
  const int local = b - e.begin;
  const int bx = local % e.tiles_x;
  const int by = (local / e.tiles_x) % e.tiles_y;
  const int bz = local / (e.tiles_x * e.tiles_y);
  PcgApplyOp<float> op = {};
  op.v = e.v;
  op.sc = e.sc;
  lin_body<float, 8, 2, PcgApplyOp<float>>(e.g, op, e.kchunk, bx, by, bz, lin_dyn);
}

void launch_batch_lin_apply(const BatchApplyEntry* tab, int n_inst, int total_blocks, cudaStream_t s) {
  using S = LinShape<float, 8, 2>;
  static bool attr_set[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64 && !attr_set[dev]) {
    if (cudaFuncSetAttribute(batch_lin_apply_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)S::dyn_bytes) == cudaSuccess &&
        cudaFuncSetAttribute(batch_lin_apply_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100) ==
            cudaSuccess)
      attr_set[dev] = true;
  }
  note_launch(), batch_lin_apply_kernel<<<total_blocks, dim3(32, 8), S::dyn_bytes, s>>>(tab, n_inst);
}

// Resident blocks per SM of the plane-factorized apply (0 if the query fails).
template <class T, int BY, int R>
static int lin_occupancy() {
  using S = LinShape<T, BY, R>;
  int n = 0;
  cudaFuncSetAttribute(lin_march_kernel<T, BY, R, ApplyOp<T>>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)S::dyn_bytes);
  cudaFuncSetAttribute(lin_march_kernel<T, BY, R, ApplyOp<T>>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, lin_march_kernel<T, BY, R, ApplyOp<T>>, 32 * BY,
                                                    S::dyn_bytes) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

int lin_blocks_per_sm(int precision, int by, int rows) {
  if (precision == 1) {
    if (rows == 2) return by == 4 ? lin_occupancy<float, 4, 2>() : by >= 16 ? lin_occupancy<float, 16, 2>()
                                                                             : lin_occupancy<float, 8, 2>();
    return by == 4 ? lin_occupancy<float, 4, 1>() : by == 16 ? lin_occupancy<float, 16, 1>()
                                                  : by >= 32 ? lin_occupancy<float, 32, 1>()
                                                             : lin_occupancy<float, 8, 1>();
  }
  if (rows == 2) return by == 4 ? lin_occupancy<double, 4, 2>() : lin_occupancy<double, 8, 2>();
  return by == 4 ? lin_occupancy<double, 4, 1>() : lin_occupancy<double, 8, 1>();
}

}  // namespace qcad
