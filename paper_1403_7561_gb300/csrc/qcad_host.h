// Host-side interfaces between the kernel translation units and the solver
// driver of libqcad (not part of the public C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "qcad_internal.cuh"

namespace qcad {

// Device-resident scalars of one preconditioned CG solve. Slots are indexed
// by iteration modulo 4 so that a kernel can accumulate the next dot product
// while the current one is still being read; t is advanced by the last block
// of the update kernel, so a captured sequence of kernels needs no host input.
struct PcgScalars {
  double rz[4];
  double pAp[4];
  double rr[4];
  double rr0;
  double tol2;
  int t;
  int done;
  int iters;
  int maxit;
  unsigned int counter;
  int nonfinite;
  // Chebyshev-Jacobi preconditioner: degree (1 = Jacobi), spectral interval [theta - delta,
  // theta + delta] of D^-1 J, and the phase of the solve (0 during the initial residual, 1 after)
  int degree;
  int phase;
  double theta;
  double delta;
};

template <class T>
struct PcgVecs {
  T* x;
  T* r;
  T* z;
  T* p[2];     // search direction, ping-ponged by iteration parity
  T* Ap;
  const T* b;
  const T* dinv;
  const T* c;   // element quadrature coefficients of the operator (8 per element)
  const unsigned char* act;  // activity map of c (qcad_internal.cuh) or null (all cells active)
  T* w;         // Chebyshev inner residual
  T* d[2];      // Chebyshev correction, ping-ponged by step parity
};

struct ResidualArgs {
  const double* phi;
  const double* theta;       // fixed charge per element or null
  double* R;
  double* diag;              // or null
  double* c64;               // or null
  float* c32;                // or null
  unsigned char* act64;      // activity map of c64, cleared by the caller, or null
  unsigned char* act32;      // of c32
  double* dinv64;            // or null
  float* dinv32;             // or null
  double* b64;               // -R or null
  float* b32;                // -R or null
  const unsigned char* layer_semi;
  const double* xn;          // node coordinates (for dot membership)
  const double* yn;
  const double* zn;
  Phys P;
  DotBoxes dots;
  double* counts;            // [n_dots] accumulated electron counts or null
  double* stats;             // [2] {max|R| (as ordered bits), sum R^2} or null
  int linear;
  QuantumDensity qd;         // quantum density in the quantum region (inactive: qd.w null)
  const double* bsurf;       // [n_nodes] constant surface load b (R -= b; two-pass residual) or null
  const double* wq;          // [nz][8] per-layer load table of constant-charge elements (physics.cuh) or null
  unsigned char* ecode;      // [n_elems] per-element load code between the two residual passes, or null
  int* list;                 // [n_elems] elements whose density is evaluated, and their number (zeroed by
  int* list_n;               // the caller), or null: without counts and quantum density (resnode.cuh)
};

template <class T>
struct ApplyArgs {
  const T* v;
  T* y;
  const T* c;
  const unsigned char* act;  // activity map of c or null
  double* dot;   // accumulate v.y (writer nodes) or null
  int raw;       // 1: no identity override on Dirichlet rows (adjoint column sums)
};

// Launch shape of the z-marching kernels: by warps (tile rows) per block, kchunk node planes
// per block, and for the linear operators the kernel variant: 0 element-gather, 1 element-gather
// with two nodes per thread and packed f32x2 arithmetic (FP32 only), 2 plane-factorized with one
// node row per thread, 3 plane-factorized with two node rows per thread.
struct LaunchCfg {
  int by = 8;
  int kchunk = 16;
  int variant = 3;
  bool fit = true;  // the shape is a default: the launch fits it to the grid (fit_lin, fit_march64); a shape
                    // set or autotuned for the mesh runs as given
};

// Planes that a march's SMs (or resident slots) run one after the other with z chunk c: a block takes
// its planes + `over` (what it does before its first output plane), `tiles` blocks per chunk. The
// blocks of full chunks come first, in waves of `slots`; those of the last, shorter chunk fill the
// slots that the last wave leaves free.
inline double march_planes(long long tiles, int nzn, long long slots, double over, int c) {
  const long long full = tiles * (nzn / c);
  const int r = nzn % c;
  const double tf = c + over, tr = r + over;
  const long long rest = full % slots;
  double t = (double)(full / slots) * tf;
  long long part = r ? tiles : 0;
  if (rest > 0) {
    t += tf;
    if (part > 0) part = part > (slots - rest) * (long long)(tf / tr) ? part - (slots - rest) * (long long)(tf / tr) : 0;
  }
  return t + (double)((part + slots - 1) / slots) * tr;
}
// The z chunk (up to kmax) with the fewest; *cost receives the count.
inline int fit_chunk(long long tiles, int nzn, long long slots, double over, int kmax, double* cost) {
  int best = 1;
  *cost = 1e300;
  for (int c = 1; c <= kmax && c <= nzn; ++c) {
    const double t = march_planes(tiles, nzn, slots, over, c);
    if (t < *cost) {
      *cost = t;
      best = c;
    }
  }
  return best;
}
// A fitted shape replaces the default only where the model promises this much: on grids of several
// waves the model's differences are below what it resolves (fitted shapes without this margin were
// 1 to 3 % slower there).
constexpr double FIT_GAIN = 0.8;
int sm_count();  // of the current device (cached)

void launch_residual(const Grid<double>& g, const ResidualArgs& a, LaunchCfg cfg, cudaStream_t s);
// Adds the electron count of the elements [box0, box1) x [box2, box3) x [box4, box5) to *out.
void launch_dot_count(const Grid<double>& g, const double* phi, const unsigned char* layer_semi, const Phys& P,
                      const int box[6], double* out, cudaStream_t s);
// Same outputs in two passes (carrier density once per quadrature point); el: 16 doubles per element.
// face: the charged gates' [nx*ny] face coefficients (Robin condition) or null; with a.bsurf set,
// the surface load is subtracted and the face mass enters the stiffness and the diagonal.
void launch_residual_2pass(const Grid<double>& g, const ResidualArgs& a, double* el, LaunchCfg cfg, cudaStream_t s,
                           const double* face = nullptr);

template <class T>
void launch_apply(const Grid<T>& g, const ApplyArgs<T>& a, LaunchCfg cfg, cudaStream_t s, const T* face = nullptr);

template <class T>
void launch_pcg_init(long long n, PcgVecs<T> v, PcgScalars* sc, cudaStream_t s);
template <class T>
void launch_pcg_apply(const Grid<T>& g, PcgVecs<T> v, PcgScalars* sc, LaunchCfg cfg, cudaStream_t s,
                      const T* face = nullptr);
template <class T>
void launch_pcg_update(long long n, PcgVecs<T> v, PcgScalars* sc, cudaStream_t s);
// Chebyshev-Jacobi form: the update kernel starts the recurrence (w = r, d = D^-1 r / theta,
// z = d) and step j = 1..degree-1 applies J to d_{j-1}; the last step forms r.z and finishes
// the iteration (or the initial residual when phase = 0).
template <class T>
void launch_pcg_update_cheb(long long n, PcgVecs<T> v, PcgScalars* sc, cudaStream_t s);
template <class T>
void launch_pcg_init_cheb(long long n, PcgVecs<T> v, PcgScalars* sc, cudaStream_t s);
template <class T>
void launch_cheb_step(const Grid<T>& g, PcgVecs<T> v, PcgScalars* sc, int step, int last, LaunchCfg cfg,
                      cudaStream_t s, const T* face = nullptr);
// One power step for the largest eigenvalue of D^-1 J: v_next = D^-1 (J v) / |.|; acc[0] += v.Jv,
// acc[1] += v.D v, acc[2] += |D^-1 J v|^2 (the caller normalizes with acc[2]).
template <class T>
void launch_power_step(long long n, const T* v, const T* Jv, const T* dinv, T* vnext, double* acc, cudaStream_t s);
template <class T>
void launch_scale(long long n, T* v, double a, cudaStream_t s);
template <class T>
void launch_random_free(const Grid<T>& g, unsigned long long seed, T* v, cudaStream_t s);

// phi_out = phi + alpha * delta on every node; stats[0] accumulates max |alpha delta| (ordered bits).
template <class T>
void launch_newton_trial(long long n, const double* phi, const T* delta, double alpha, double* phi_out,
                         double* stats, cudaStream_t s);

// Dirichlet values: bottom plane (if set) gets v_bottom, top-plane nodes with gate id >= 0 get v_gate[id].
void launch_set_dirichlet(long long nxn, long long nyn, long long nzn, int bottom, double v_bottom,
                          const signed char* gate_top, const double* v_gate, double* phi, cudaStream_t s);

// Elementwise conversions.
void launch_d2f(long long n, const double* a, float* b, cudaStream_t s);
void launch_f2d(long long n, const float* a, double* b, cudaStream_t s);

// dN_d/dphi as a nodal vector for dot d: sum over dot elements of w|J| n'(phi_q) N_a(q), written
// at the nodes of the dot's element box (the caller zeroes out beforehand). box: the
// dot's element box {i0, i1, j0, j1, k0, k1} (elements i0 <= i < i1, ...) or null when it is empty;
// el: scratch of 8 doubles per box element.
void launch_count_gradient(const Grid<double>& g, const double* phi, const unsigned char* layer_semi,
                           const double* xn, const double* yn, const double* zn, const Phys& P,
                           const DotBoxes& dots, int d, const int* box, double* out, double* el, cudaStream_t s);

// theta-gradient of N_d: out[e] = qe * (|e|/8) * sum of lam over the 8 corners of e (lam is
// zero on Dirichlet nodes); |e|/8 = int_e N_a exactly on a box.
void launch_theta_gradient(int nx, int ny, int nz, const double* hx, const double* hy, const double* hz,
                           const double* lam, double qe, double* out, cudaStream_t s);

// Schrodinger operators on the subdomain grid (field 0: H, field 1: M).
template <class T>
struct HmArgs {
  const T* x;      // nvec full-subdomain vectors, stride ldx
  T* hx;           // or null
  T* mx;           // or null
  long long ld;    // vector stride (n_sub_nodes)
  int nvec;
};
// H and M with the V term assembled into a 27-point row per node (kernels_hm.cu): S [27][nodes], zt
// [planes][12] the kinetic coefficients of an output plane along x, y, z and its mass, each for the
// input planes below, at and above it. C: float, double, or float2 for double-float arithmetic on
// FP64 vectors.
template <class C>
struct HmStencil {
  const C* S;
  const C* zt;
  int nxn, nyn, nzn;
};
void launch_hm_stencil(const HmStencil<float>& st, const HmArgs<float>& a, cudaStream_t s);
void launch_hm_stencil(const HmStencil<double>& st, const HmArgs<double>& a, cudaStream_t s);
void launch_hm_stencil(const HmStencil<float2>& st, const HmArgs<double>& a, cudaStream_t s);
// The rows of the subdomain grid from its coefficients cV (8 per element), in the precisions whose
// output is not null; mom: scratch of 27 doubles per element of `slab` element layers, which are
// assembled at a time (hm_slab_layers).
void launch_hm_rows(const double* cV, int nxn, int nyn, int nzn, int slab, double* mom, float* S32, float2* Sdf,
                    double* S64, cudaStream_t s);
// Jacobi scale 1 / dk[k] of the interior nodes (0 on the boundary) and the interior mask.
void launch_hm_jacobi(int nxn, int nyn, int nzn, const double* dk, double* dinv, unsigned char* interior, cudaStream_t s);
// One fused step of the LOBPCG Chebyshev-Jacobi block preconditioner (kernels_hm.cu): the H apply
// of D_in (nvec columns at stride ld) with the recurrence W -= H D_in,
// D_out = c1 D_in + c2 D^-1 W, Z += D_out in its epilogue.
struct ChebHmArgs {
  const float* din;
  float* dout;
  float* w;
  float* z;
  const float* dinv;
  long long ld;
  int nvec;
  float c1, c2;
};
void launch_cheb_hm_step(const HmStencil<float>& st, const ChebHmArgs& args, cudaStream_t s);

}  // namespace qcad

namespace qcad {
template <class T>
void launch_dot(long long n, const T* a, const T* b, double* out, cudaStream_t s);
template <class T>
void launch_axpy(long long n, double a, const T* x, double* y, cudaStream_t s);
void launch_sub(long long n, const double* g, const double* y, double* r, float* r32, cudaStream_t s);
}  // namespace qcad

namespace qcad {
// Kernel launches issued by the library (graph replays count their kernels).
void note_launch(int n = 1);
long long launch_count();
}  // namespace qcad

namespace qcad {
// Plane-factorized launches of the linear ops (variants 2 and 3).
template <class T>
void launch_apply_lin(const Grid<T>& g, const ApplyArgs<T>& args, LaunchCfg cfg, cudaStream_t s);
template <class T>
void launch_pcg_apply_lin(const Grid<T>& g, PcgVecs<T> vecs, PcgScalars* sc, LaunchCfg cfg, cudaStream_t s);
template <class T>
void launch_cheb_step_lin(const Grid<T>& g, PcgVecs<T> vecs, PcgScalars* sc, int step, int last, LaunchCfg cfg,
                          cudaStream_t s);
int lin_blocks_per_sm(int precision, int by, int rows);
// The default shape of the plane-factorized kernels on a grid, as an explicit configuration.
LaunchCfg default_lin_shape(int precision, int nxn, int nyn, int nzn, bool act);

// Resident blocks per SM of the Jacobian apply of a precision (0 FP64, 1 FP32) and variant.
int apply_blocks_per_sm(int precision, int by, int variant);

// Work-table entries of the batched kernels (sorted by begin = first block of the entry).
struct BatchApplyEntry {
  Grid<float> g;
  PcgVecs<float> v;
  PcgScalars* sc;
  int kchunk;
  int tiles_x, tiles_y;
  int begin;
};
struct BatchVecEntry {
  PcgVecs<float> v;
  PcgScalars* sc;
  int n;
  int blocks;
  int begin;
};
// Work-table entry of the batched FP64 residual (element-gather march, 8 warps).
struct BatchResEntry {
  Grid<double> g;
  ResidualArgs a;
  int kchunk;
  int tiles_x, tiles_y;
  int begin;       // first block of the node pass (z-march tiles of 30 columns and 2 NODE_WARPS rows)
  int qbegin;      // first block of the classification pass
  int qtiles;      // its blocks per z chunk
  double* el;      // the instance's corner-contribution scratch, 16 doubles per element
};
void launch_batch_pcg_apply(const BatchApplyEntry* tab, int n_inst, int total_blocks, int by, cudaStream_t s);
// Plane-factorized batched PCG apply (8 warps, two rows per thread: tiles of 30 x 14 interior nodes).
void launch_batch_lin_apply(const BatchApplyEntry* tab, int n_inst, int total_blocks, cudaStream_t s);
// Two-pass batched residual (resnode.cuh): classification over qp_blocks blocks, density, node pass.
void batch_residual_shape(BatchResEntry& e, const LaunchCfg& cfg, int& total, int& total_q);
void launch_batch_residual_2pass(const BatchResEntry* tab, int n_inst, int qp_blocks, int node_blocks,
                                 cudaStream_t s);
// Per-instance stats slots: mode 0 zeroes the residual slots (stats[0] max |R| as ordered bits,
// stats[1] sum R^2), mode 1 zeroes the trial-step slot stats[8], mode 2 gathers the three into
// out[3i .. 3i+2].
void launch_batch_stats(const BatchResEntry* tab, int n_inst, int mode, double* out, cudaStream_t s);
void launch_batch_pcg_update(const BatchVecEntry* tab, int n_inst, int total_blocks, cudaStream_t s);
void launch_batch_status(const BatchVecEntry* tab, int n_inst, int* status, cudaStream_t s);
}  // namespace qcad
