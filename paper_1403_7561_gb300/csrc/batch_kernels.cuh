// Batched kernels: one launch covers the PCG apply (or update) of every
// instance of a batch of meshes of different sizes. A work table maps each
// block to (instance, tile); each instance keeps its own device-resident PCG
// scalars, so instances converge and drop out independently (their blocks
// return at once). Included at the end of kernels_poisson.cu, whose operator
// ops and PCG bookkeeping it reuses.
#pragma once

namespace qcad {

// Index of the last table entry whose begin <= b (entries sorted by begin).
template <class E>
__device__ __forceinline__ int batch_find(const E* tab, int n, int b) {
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

template <int BY>
__global__ void __launch_bounds__(QCAD_BX * BY) batch_pcg_apply_kernel(const BatchApplyEntry* tab, int n_inst) {
  const int b = blockIdx.x;
  const BatchApplyEntry& e = tab[batch_find(tab, n_inst, b)];
  const int local = b - e.begin;
  const int bx = local % e.tiles_x;
  const int by = (local / e.tiles_x) % e.tiles_y;
  const int bz = local / (e.tiles_x * e.tiles_y);
  PcgApplyOp<float> op = {};
  op.v = e.v;
  op.sc = e.sc;
  march_body<float, BY, PcgApplyOp<float>>(e.g, op, e.kchunk, bx, by, bz);
}

__global__ void __launch_bounds__(VEC_THREADS) batch_pcg_update_kernel(const BatchVecEntry* tab, int n_inst) {
  const int b = blockIdx.x;
  const BatchVecEntry& e = tab[batch_find(tab, n_inst, b)];
  pcg_update_body<float>(e.n, e.v, e.sc, b - e.begin, e.blocks);
}

// status[i] = {done, t, nonfinite, iters} of instance i (one read for the whole batch).
__global__ void batch_status_kernel(const BatchVecEntry* tab, int n_inst, int* status) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_inst; i += gridDim.x * blockDim.x) {
    const PcgScalars* sc = tab[i].sc;
    status[4 * i + 0] = sc->done;
    status[4 * i + 1] = sc->t;
    status[4 * i + 2] = sc->nonfinite;
    status[4 * i + 3] = sc->iters;
  }
}

// Entry of block b for the classification pass (entries sorted by qbegin).
__device__ __forceinline__ int batch_find_q(const BatchResEntry* tab, int n, int b) {
  int lo = 0, hi = n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (tab[mid].qbegin <= b)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

constexpr int BATCH_RES_CHUNK = 4;  // element layers per block of the classification pass

// The residual's passes over the instances (resnode.cuh).
__global__ void __launch_bounds__(256) batch_residual_classify_kernel(const BatchResEntry* tab, int n_inst) {
  const int b = blockIdx.x;
  const BatchResEntry& e = tab[batch_find_q(tab, n_inst, b)];
  const long long ne = (long long)e.g.nx * e.g.ny * e.g.nz;
  const int local = b - e.qbegin, k0 = (local / e.qtiles) * BATCH_RES_CHUNK;
  residual_classify_body(e.g, e.a, e.el, e.el + 8 * ne, (local % e.qtiles) * 256 + threadIdx.x, k0,
                         min(k0 + BATCH_RES_CHUNK, e.g.nz));
}

__global__ void __launch_bounds__(256) batch_residual_density_kernel(const BatchResEntry* tab) {
  const BatchResEntry& e = tab[blockIdx.y];
  const long long ne = (long long)e.g.nx * e.g.ny * e.g.nz;
  residual_density_body(e.g, e.a, e.el, e.el + 8 * ne, blockIdx.x, gridDim.x);
}

__global__ void __launch_bounds__(32 * NODE_WARPS) batch_residual_node_kernel(const BatchResEntry* tab, int n_inst) {
  const int b = blockIdx.x;
  const BatchResEntry& e = tab[batch_find(tab, n_inst, b)];
  const int local = b - e.begin;
  const int bx = local % e.tiles_x;
  const int by = (local / e.tiles_x) % e.tiles_y;
  const int k0 = (local / (e.tiles_x * e.tiles_y)) * e.kchunk;
  const int jb = 2 * (by * NODE_WARPS + (threadIdx.x >> 5));
  const long long ne = (long long)e.g.nx * e.g.ny * e.g.nz;
  double r2 = 0.0;
  unsigned long long rmax = 0;
  if (jb < e.g.nyn)
    residual_node_body(e.g, e.a, e.el, e.el + 8 * ne, bx, jb, k0, min(k0 + e.kchunk, e.g.nzn), r2, rmax);
  residual_node_finish(e.a, r2, rmax);
}

__global__ void batch_stats_kernel(const BatchResEntry* tab, int n_inst, int mode, double* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n_inst; i += gridDim.x * blockDim.x) {
    double* st = tab[i].a.stats;
    if (mode == 0) {
      st[0] = 0.0;
      st[1] = 0.0;
      *tab[i].a.list_n = 0;
    } else if (mode == 1) {
      st[8] = 0.0;
    } else {
      out[3 * i + 0] = st[0];
      out[3 * i + 1] = st[1];
      out[3 * i + 2] = st[8];
    }
  }
}

// Clears the activity maps before the residual (one row of blocks per instance).
__global__ void __launch_bounds__(256) batch_clear_act_kernel(const BatchResEntry* tab) {
  const BatchResEntry& e = tab[blockIdx.y];
  const int n = act_cells(e.g.nx, ACT_X) * act_cells(e.g.ny, ACT_Y) * act_cells(e.g.nz, ACT_Z);
  if (e.a.act32 == nullptr) return;
  for (int q = blockIdx.x * 256 + threadIdx.x; q < n; q += gridDim.x * 256) e.a.act32[q] = 0;
}

void launch_batch_residual_2pass(const BatchResEntry* tab, int n_inst, int qp_blocks, int node_blocks,
                                 cudaStream_t s) {
  note_launch(), batch_clear_act_kernel<<<dim3(4, n_inst), 256, 0, s>>>(tab);
  note_launch(3);
  batch_residual_classify_kernel<<<qp_blocks, 256, 0, s>>>(tab, n_inst);
  // density blocks per instance: 16 per SM in all, as many as the density pass of one mesh (8 per SM) at
  // most; the blocks stride over the lists, whose lengths only the device knows
  const int all = 16 * sm_count() / n_inst, db = all < 16 ? 16 : all < 8 * sm_count() ? all : 8 * sm_count();
  batch_residual_density_kernel<<<dim3(db, n_inst), 256, 0, s>>>(tab);
  batch_residual_node_kernel<<<node_blocks, 32 * NODE_WARPS, 0, s>>>(tab, n_inst);
}

// Tiles of an instance's residual passes; total and total_q are the table's block counts so far.
void batch_residual_shape(BatchResEntry& e, const LaunchCfg& cfg, int& total, int& total_q) {
  e.kchunk = cfg.kchunk < 2 ? 2 : cfg.kchunk;
  e.tiles_x = (e.g.nxn + 29) / 30;
  e.tiles_y = (e.g.nyn + 2 * NODE_WARPS - 1) / (2 * NODE_WARPS);
  e.begin = total;
  total += e.tiles_x * e.tiles_y * ((e.g.nzn + e.kchunk - 1) / e.kchunk);
  e.qbegin = total_q;
  e.qtiles = (e.g.nx * e.g.ny + 255) / 256;
  total_q += e.qtiles * ((e.g.nz + BATCH_RES_CHUNK - 1) / BATCH_RES_CHUNK);
}

void launch_batch_stats(const BatchResEntry* tab, int n_inst, int mode, double* out, cudaStream_t s) {
  note_launch(), batch_stats_kernel<<<(n_inst + 127) / 128, 128, 0, s>>>(tab, n_inst, mode, out);
}

void launch_batch_pcg_apply(const BatchApplyEntry* tab, int n_inst, int total_blocks, int by, cudaStream_t s) {
  if (by == 16)
    note_launch(), batch_pcg_apply_kernel<16><<<total_blocks, dim3(QCAD_BX, 16), 0, s>>>(tab, n_inst);
  else
    note_launch(), batch_pcg_apply_kernel<8><<<total_blocks, dim3(QCAD_BX, 8), 0, s>>>(tab, n_inst);
}

void launch_batch_pcg_update(const BatchVecEntry* tab, int n_inst, int total_blocks, cudaStream_t s) {
  note_launch(), batch_pcg_update_kernel<<<total_blocks, VEC_THREADS, 0, s>>>(tab, n_inst);
}

void launch_batch_status(const BatchVecEntry* tab, int n_inst, int* status, cudaStream_t s) {
  note_launch(), batch_status_kernel<<<(n_inst + 127) / 128, 128, 0, s>>>(tab, n_inst, status);
}

}  // namespace qcad
