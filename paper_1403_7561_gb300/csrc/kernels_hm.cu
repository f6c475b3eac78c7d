// Schrodinger operators H and M (Sec. II.B, Eq. SchrodEqnWeakForm) for blocks of vectors, with the
// potential's mass term assembled into one 27-point row per node.
//
// H = kinetic stencil + V term. The kinetic part is a sum of Kronecker products of 1D operators on
// uniform x and y spacings, applied per node plane from nine values as
//   a_r = 4 v + (v- + v+), b_r = 2 v - (v- + v+)       along x, for the rows r = j-1, j, j+1,
//   P2 = 4 a_0 + (a_- + a_+), P1x = 4 b_0 + (b_- + b_+), P1y = 2 a_0 - (a_- + a_+),
// then along z with the step sizes folded into the plane's coefficients (zt), the z stiffness as fluxes
// w (P2 of one plane less that of the one below): the differences of neighbouring values stay
// differences, so a smooth field loses no digits to the assembly. M uses P2 alone. The V term sum_q w|J| V_q N_a(q) N_b(q) has no such structure; its row costs 27 products
// per node and vector, where evaluating it at the Gauss points took the plane-factorized march of
// linmarch.cuh about 100 operations, 20 shuffles and shared-memory exchanges and a barrier per plane.
//
// A thread marches one (x, y) column over a chunk of planes for NV vectors at once: a plane's nine
// values per vector feed the three output planes around it, and a coefficient is loaded once for NV
// vectors. Nothing is exchanged between threads (neighbours come from L1), so there is no barrier and
// latency is hidden by independent warps. Columns are numbered linearly through the plane, so warps
// are full whatever nx is.
#include <cuda_runtime.h>

#include "dfloat.cuh"
#include "launch_rules.h"
#include "qcad_host.h"
#include "qcad_internal.cuh"

namespace qcad {

// Arithmetic type T, storage of vectors (X) and of coefficients (C), vectors per thread.
template <class T> struct HmT;
template <> struct HmT<float> {
  using X = float;
  using C = float;
  static constexpr int NV = 4, MINB = 2;
  static __device__ __forceinline__ float ld(float x) { return x; }
  static __device__ __forceinline__ float co(float c) { return c; }
  static __device__ __forceinline__ float st(float x) { return x; }
};
template <> struct HmT<double> {
  using X = double;
  using C = double;
  static constexpr int NV = 2, MINB = 2;
  static __device__ __forceinline__ double ld(double x) { return x; }
  static __device__ __forceinline__ double co(double c) { return c; }
  static __device__ __forceinline__ double st(double x) { return x; }
};
// FP64 vectors in double-float arithmetic.
template <> struct HmT<dfl> {
  using X = double;
  using C = float2;
  static constexpr int NV = 2, MINB = 2;
  static __device__ __forceinline__ dfl ld(double x) { return dfl_from_bits(x); }
  static __device__ __forceinline__ dfl co(float2 c) { return dfl(c.x, c.y); }
  static __device__ __forceinline__ double st(dfl x) { return dfl_to_double(x); }
};

__device__ __forceinline__ void hm_fma(float& s, float a, float b) { s = fmaf(a, b, s); }
__device__ __forceinline__ void hm_fma(double& s, double a, double b) { s = fma(a, b, s); }
__device__ __forceinline__ void hm_fma(dfl& s, dfl a, dfl b) { s += dfl_prod(a, b); }
// s += c0 x0 + c1 x1 + c2 x2. Double-float renormalizes once per three products: with the low word
// collecting the errors of a node's 36 products unrenormalized, H of smooth vectors on 24 x 22 x 20
// elements was off by up to 7.2e-14 of its largest entry against 64-bit extended arithmetic; now 1.4e-14
// (the march evaluating Gauss points, renormalized at each step, 1.6e-14).
template <class T>
__device__ __forceinline__ void hm_mac3(T& s, T c0, T x0, T c1, T x1, T c2, T x2) {
  hm_fma(s, c0, x0);
  hm_fma(s, c1, x1);
  hm_fma(s, c2, x2);
}
__device__ __forceinline__ void hm_mac3(dfl& s, dfl c0, dfl x0, dfl c1, dfl x1, dfl c2, dfl x2) {
  dfl_mac3(s, c0, x0, c1, x1, c2, x2);
}
// s += a x + b y
template <class T>
__device__ __forceinline__ void hm_mac2(T& s, T a, T x, T b, T y) {
  hm_fma(s, a, x);
  hm_fma(s, b, y);
}
__device__ __forceinline__ void hm_mac2(dfl& s, dfl a, dfl x, dfl b, dfl y) {
  dfl t = dfl_prod(a, x);
  dfl_mac(t, b, y);
  s += t;
}
__device__ __forceinline__ float hm_4p(float v, float s) { return fmaf(4.0f, v, s); }
__device__ __forceinline__ double hm_4p(double v, double s) { return fma(4.0, v, s); }
__device__ __forceinline__ dfl hm_4p(dfl v, dfl s) { return dfl(4.0f * v.h, 4.0f * v.l) + s; }
__device__ __forceinline__ float hm_2m(float v, float s) { return fmaf(2.0f, v, -s); }
__device__ __forceinline__ double hm_2m(double v, double s) { return fma(2.0, v, -s); }
__device__ __forceinline__ dfl hm_2m(dfl v, dfl s) { return dfl(2.0f * v.h, 2.0f * v.l) - s; }

// H and M of each vector.
template <class T, bool MASS>
struct HmOutOp {
  static constexpr bool mass = MASS;
  using X = typename HmT<T>::X;
  X *hx, *mx;
  long long ld;
  struct Pre {};
  struct Node {};
  __device__ __forceinline__ Pre pre(int, int) const { return Pre{}; }
  __device__ __forceinline__ Node node(int) const { return Node{}; }
  __device__ __forceinline__ void out(int vec, int n, const Node&, const Pre&, T, T h, T m) const {
    const long long o = vec * ld + n;
    if (hx) hx[o] = HmT<T>::st(h);
    if (MASS) mx[o] = HmT<T>::st(m);
  }
  __device__ __forceinline__ void zero(int vec, int n) const {
    const long long o = vec * ld + n;
    if (hx) hx[o] = X(0);
    if (MASS) mx[o] = X(0);
  }
};

// One step of the eigensolver's Chebyshev-Jacobi block preconditioner in the epilogue of the H apply
// of its direction block: with h = (H D_in)_n,
//   W <- W - h,  D_out <- c1 D_in + c2 D^-1 W,  Z <- Z + D_out
// D is double-buffered, since neighbours still read D_in; boundary rows hold zeros throughout.
struct HmChebOp {
  static constexpr bool mass = false;
  ChebHmArgs a;
  // the epilogue's inputs, loaded before the plane's sums: behind another vector's stores they could not
  // be (each plane then waited for memory NV more times: 150 us per step on 129 x 129 x 44 nodes)
  struct Pre {
    float w, z;
  };
  struct Node {
    float dinv;
  };
  __device__ __forceinline__ Pre pre(int vec, int n) const {
    const long long o = vec * a.ld + n;
    return Pre{a.w[o], a.z[o]};
  }
  __device__ __forceinline__ Node node(int n) const { return Node{__ldg(a.dinv + n)}; }
  __device__ __forceinline__ void out(int vec, int n, const Node& q, const Pre& p, float din, float h, float) const {
    const long long o = vec * a.ld + n;
    const float w = p.w - h;
    const float d = a.c1 * din + a.c2 * q.dinv * w;
    a.w[o] = w;
    a.dout[o] = d;
    a.z[o] = p.z + d;
  }
  __device__ __forceinline__ void zero(int vec, int n) const { a.dout[vec * a.ld + n] = 0.0f; }
};

constexpr int HM_THREADS = 256;

template <class T, class Op>
__global__ void __launch_bounds__(HM_THREADS, HmT<T>::MINB)
    hm_stencil_kernel(const HmStencil<typename HmT<T>::C> a, const typename HmT<T>::X* __restrict__ xs, long long ld, int nvec, int kchunk,
                      const Op op) {
  using Tr = HmT<T>;
  using X = typename Tr::X;
  using C = typename Tr::C;
  constexpr int NV = Tr::NV;
  const int ng = (nvec + NV - 1) / NV;
  // the vector groups of a column block run side by side: its coefficients are read from L2 after the first
  const int v0 = (blockIdx.x % ng) * NV;
  const int plane = a.nxn * a.nyn;
  const int p = (blockIdx.x / ng) * HM_THREADS + threadIdx.x;
  if (p >= plane) return;
  const int nv = min(NV, nvec - v0);
  const int k0 = blockIdx.y * kchunk, k1 = min(k0 + kchunk, a.nzn);
  const int j = p / a.nxn, i = p - j * a.nxn;
  if (i == 0 || j == 0 || i == a.nxn - 1 || j == a.nyn - 1) {
    for (int k = k0; k < k1; ++k)
      for (int v = 0; v < nv; ++v) op.zero(v0 + v, p + k * plane);
    return;
  }
  const C* __restrict__ S = a.S;
  const C* __restrict__ zt = a.zt;
  const long long ns = (long long)plane * a.nzn;
  const X* x[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) x[v] = xs + (long long)(v0 + (v < nv ? v : 0)) * ld + p;
  T h[3][NV], m[3][NV], xprev[NV], p2prev[NV];
#pragma unroll
  for (int v = 0; v < NV; ++v) {
#pragma unroll
    for (int o = 0; o < 3; ++o) h[o][v] = m[o][v] = T(0);
    xprev[v] = p2prev[v] = T(0);
  }
  const int ke = min(k1, a.nzn - 1);
  for (int kp = max(k0 - 1, 0); kp <= ke; ++kp) {
    // input plane kp feeds the output planes kp - 1, kp, kp + 1 of the chunk
    const bool on[3] = {kp - 1 >= k0, kp >= k0 && kp < k1, kp + 1 < k1};
    const int n = p + kp * plane;
    typename Op::Pre pre[NV];
    typename Op::Node nd;
    if (on[0]) {
      nd = op.node(n - plane);
#pragma unroll
      for (int v = 0; v < NV; ++v)
        if (v < nv) pre[v] = op.pre(v0 + v, n - plane);
    }
    T a0[NV], b0[NV], sa[NV], sb[NV];
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      T c[3][3];
#pragma unroll
      for (int o = 0; o < 3; ++o)
#pragma unroll
        for (int d = 0; d < 3; ++d)
          c[o][d] = on[o] ? Tr::co(__ldg(S + (9 * (2 - o) + 3 * r + d) * ns + (n + (o - 1) * plane))) : T(0);
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        const X* q = x[v] + kp * plane + (r - 1) * a.nxn;
        const T xm = Tr::ld(__ldg(q - 1)), xc = Tr::ld(__ldg(q)), xp = Tr::ld(__ldg(q + 1));
        const T s = xm + xp;
        const T av = hm_4p(xc, s), bv = hm_2m(xc, s);
        if (r == 0) {
          sa[v] = av;
          sb[v] = bv;
        } else if (r == 1) {
          a0[v] = av;
          b0[v] = bv;
        } else {
          sa[v] += av;
          sb[v] += bv;
        }
#pragma unroll
        for (int o = 0; o < 3; ++o) hm_mac3(h[o][v], c[o][0], xm, c[o][1], xc, c[o][2], xp);
      }
    }
    // per output plane: x and y kinetic coefficients and the mass, for input planes o-1, o, o+1
    T z[3][3];
#pragma unroll
    for (int o = 0; o < 3; ++o)
#pragma unroll
      for (int q = 0; q < 3; ++q)
        z[o][q] = on[o] ? Tr::co(__ldg(zt + 12 * (kp + o - 1) + 3 * (q == 2 ? 3 : q) + (2 - o))) : T(0);
    // z stiffness of the layer below plane kp, -w: plane kp gains w d, plane kp - 1 loses it. The first
    // plane's sums towards planes that are not the chunk's are dropped, and plane 0 has no layer below
    const T wz = Tr::co(__ldg(zt + 12 * kp + 6));
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const T p2 = hm_4p(a0[v], sa[v]), p1x = hm_4p(b0[v], sb[v]), p1y = hm_2m(a0[v], sa[v]);
      const T d = p2 - p2prev[v];
      p2prev[v] = p2;
      hm_mac3(h[0][v], z[0][0], p1x, z[0][1], p1y, wz, d);
      hm_mac3(h[1][v], z[1][0], p1x, z[1][1], p1y, wz, -d);
      hm_mac2(h[2][v], z[2][0], p1x, z[2][1], p1y);
      if (Op::mass) {
#pragma unroll
        for (int o = 0; o < 3; ++o) hm_fma(m[o][v], z[o][2], p2);
      }
    }
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      if (on[0] && v < nv) {
        if (kp == 1)
          op.zero(v0 + v, n - plane);  // the bottom plane
        else
          op.out(v0 + v, n - plane, nd, pre[v], xprev[v], h[0][v], m[0][v]);
      }
      xprev[v] = Tr::ld(__ldg(x[v] + kp * plane));
      h[0][v] = h[1][v];
      h[1][v] = h[2][v];
      h[2][v] = T(0);
      if (Op::mass) {
        m[0][v] = m[1][v];
        m[1][v] = m[2][v];
        m[2][v] = T(0);
      }
    }
  }
  if (k1 == a.nzn)  // the top plane
    for (int v = 0; v < nv; ++v) op.zero(v0 + v, p + (k1 - 1) * plane);
}

template <class T, class Op>
static void hm_run(const HmStencil<typename HmT<T>::C>& a, const typename HmT<T>::X* x, long long ld, int nvec, const Op& op,
                   cudaStream_t s) {
  const int plane = a.nxn * a.nyn;
  const int ng = (nvec + HmT<T>::NV - 1) / HmT<T>::NV;
  const long long tiles = (long long)ng * ((plane + HM_THREADS - 1) / HM_THREADS);
  double cost;
  const int kc = fit_chunk(tiles, a.nzn, (long long)HmT<T>::MINB * sm_count(), 2.0, 64, &cost);
  const dim3 grid((unsigned)tiles, (a.nzn + kc - 1) / kc);
  note_launch(), hm_stencil_kernel<T, Op><<<grid, HM_THREADS, 0, s>>>(a, x, ld, nvec, kc, op);
}

template <class T>
static void hm_apply(const HmStencil<typename HmT<T>::C>& a, const HmArgs<typename HmT<T>::X>& v, cudaStream_t s) {
  if (v.mx) {
    HmOutOp<T, true> op{v.hx, v.mx, v.ld};
    hm_run<T>(a, v.x, v.ld, v.nvec, op, s);
  } else {
    HmOutOp<T, false> op{v.hx, nullptr, v.ld};
    hm_run<T>(a, v.x, v.ld, v.nvec, op, s);
  }
}
void launch_hm_stencil(const HmStencil<float>& a, const HmArgs<float>& v, cudaStream_t s) { hm_apply<float>(a, v, s); }
void launch_hm_stencil(const HmStencil<double>& a, const HmArgs<double>& v, cudaStream_t s) { hm_apply<double>(a, v, s); }
void launch_hm_stencil(const HmStencil<float2>& a, const HmArgs<double>& v, cudaStream_t s) { hm_apply<dfl>(a, v, s); }
void launch_cheb_hm_step(const HmStencil<float>& a, const ChebHmArgs& v, cudaStream_t s) {
  HmChebOp op;
  op.a = v;
  hm_run<float>(a, v.din, v.ld, v.nvec, op, s);
}

// ---------------------------------------------------------------------------
// Assembly of the V rows, in FP64. An entry N_a N_b of an element matrix is one of 27 moments of the
// coefficients: per axis the corner pair is (0, 0), (0, 1) or (1, 1). Pass 1 forms the moments by
// sum factorization (114 operations per element; the direct product of the 2 x 2 x 2 rows takes
// about 600 per node), pass 2 adds the up to 8 elements' entries of every row.
__global__ void __launch_bounds__(256) hm_moments_kernel(const double* __restrict__ cV, int ne, double* mom) {
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e >= ne) return;
  double c[8];
  load_c8<double>(cV, e, c);
  const double A = GaussConst<double>::a(), B = GaussConst<double>::b();
  const double w[3][2] = {{A * A, B * B}, {A * B, A * B}, {B * B, A * A}};  // pair class, Gauss point
  double tx[4][3];
#pragma unroll
  for (int yz = 0; yz < 4; ++yz)
#pragma unroll
    for (int q = 0; q < 3; ++q) tx[yz][q] = w[q][0] * c[2 * yz] + w[q][1] * c[2 * yz + 1];
  double ty[2][9];
#pragma unroll
  for (int zq = 0; zq < 2; ++zq)
#pragma unroll
    for (int q = 0; q < 9; ++q) ty[zq][q] = w[q / 3][0] * tx[2 * zq][q % 3] + w[q / 3][1] * tx[2 * zq + 1][q % 3];
#pragma unroll
  for (int q = 0; q < 27; ++q)
    mom[(size_t)q * ne + e] = w[q / 9][0] * ty[0][q % 9] + w[q / 9][1] * ty[1][q % 9];
}

// Row of node (i, j, k): along each axis the offset -1 comes from the left element's pair (0, 1), the
// offset +1 from the right one's, the offset 0 from the left's (1, 1) and the right's (0, 0). Rows of
// boundary nodes are zero.
// (p0, p1): the node planes of the launch; mom holds the layers from e0 on, ne elements.
__global__ void __launch_bounds__(128) hm_rows_kernel(const double* __restrict__ mom, int nxn, int nyn, int nzn, int p0,
                                                      int p1, int e0, int ne, float* S32, float2* Sdf, double* S64) {
  const int n = blockIdx.x * 128 + threadIdx.x + nxn * nyn * p0;
  const int ns = nxn * nyn * nzn;
  if (n >= nxn * nyn * p1) return;
  const int i = n % nxn, j = (n / nxn) % nyn, k = n / (nxn * nyn);
  const int nx = nxn - 1, ny = nyn - 1, nz = nzn - 1;
  const bool in = i > 0 && j > 0 && k > 0 && i < nx && j < ny && k < nz;
  const int e = in ? (i - 1) + nx * ((j - 1) + ny * (k - 1 - e0)) : 0;  // the lower left element
#pragma unroll
  for (int q = 0; q < 27; ++q) {
    const int d[3] = {q % 3, (q / 3) % 3, q / 9};  // offset + 1
    double s = 0.0;
    if (in) {
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        // side of the element along each axis; off-diagonal offsets have one side only
        const int sx = t & 1, sy = (t >> 1) & 1, sz = t >> 2;
        if ((d[0] == 0 && sx) || (d[0] == 2 && !sx) || (d[1] == 0 && sy) || (d[1] == 2 && !sy) || (d[2] == 0 && sz) ||
            (d[2] == 2 && !sz))
          continue;
        const int cx = d[0] != 1 ? 1 : (sx ? 0 : 2), cy = d[1] != 1 ? 1 : (sy ? 0 : 2), cz = d[2] != 1 ? 1 : (sz ? 0 : 2);
        s += __ldg(mom + (size_t)(cx + 3 * cy + 9 * cz) * ne + (e + sx + nx * (sy + ny * sz)));
      }
    }
    const size_t o = (size_t)q * ns + n;
    if (S32) S32[o] = (float)s;
    if (Sdf) {
      // rounded to 49 bits (a truncated row entry biases a node's 27 products one way)
      const float f = d2f_bits(s);
      Sdf[o] = make_float2(f, d2f_bits(s - dfl_f2d(f)));
    }
    if (S64) S64[o] = s;
  }
}

__global__ void __launch_bounds__(256) hm_jacobi_kernel(int nxn, int nyn, int nzn, const double* __restrict__ dk,
                                                        double* dinv, unsigned char* interior) {
  const int n = blockIdx.x * 256 + threadIdx.x;
  if (n >= nxn * nyn * nzn) return;
  const int k = n / (nxn * nyn), p = n - k * (nxn * nyn), j = p / nxn, i = p - j * nxn;
  const bool in = i > 0 && j > 0 && k > 0 && i < nxn - 1 && j < nyn - 1 && k < nzn - 1;
  dinv[n] = in ? 1.0 / dk[k] : 0.0;
  interior[n] = in ? 1 : 0;
}
// One row of blocks over all nodes: a subdomain may have more planes than a grid's second axis (65535).
void launch_hm_jacobi(int nxn, int nyn, int nzn, const double* dk, double* dinv, unsigned char* interior,
                      cudaStream_t s) {
  note_launch();
  hm_jacobi_kernel<<<(nxn * nyn * nzn + 255) / 256, 256, 0, s>>>(nxn, nyn, nzn, dk, dinv, interior);
}

void launch_hm_rows(const double* cV, int nxn, int nyn, int nzn, int slab, double* mom, float* S32, float2* Sdf,
                    double* S64, cudaStream_t s) {
  const int layer = (nxn - 1) * (nyn - 1), plane = nxn * nyn;
  for (int p0 = 0; p0 < nzn;) {
    const HmSlab b = hm_next_slab(p0, nzn - 1, slab);
    const int ne = layer * (b.e1 - b.e0);
    note_launch(2);
    hm_moments_kernel<<<(ne + 255) / 256, 256, 0, s>>>(cV + 8LL * layer * b.e0, ne, mom);
    hm_rows_kernel<<<(plane * (b.p1 - b.p0) + 127) / 128, 128, 0, s>>>(mom, nxn, nyn, nzn, b.p0, b.p1, b.e0, ne, S32,
                                                                       Sdf, S64);
    p0 = b.p1;
  }
}

}  // namespace qcad
