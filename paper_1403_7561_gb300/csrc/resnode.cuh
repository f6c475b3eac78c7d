// The residual without dot counts, quantum density or surface terms (the path of every
// Newton step and line-search trial, single and batched): a classification pass over the elements, the
// density at the Gauss points of the listed elements, and a node pass. Included by kernels_poisson.cu.
//
// FP64 runs at 2 lanes per SM and clock, so each pass is held to the FP64 work that its outputs need:
//  - Classification (one thread per element column, marching z): charge zones of the node potentials by
//    integer keys, once per node and column. An element whose corners share a constant-charge zone gets
//    its load code and zero coefficients; the others are appended to a list. No FP64 arithmetic: signs,
//    keys and zero tests are taken on the halves of the pattern (written on the whole pattern they came
//    out as five FP64 additions an element: 87 us at 256 x 256 x 128 elements, 60 us now; the coefficient
//    stores take 40).
//  - Density (8 lanes per listed element): full warps whatever the shape of the charged region. In one
//    pass over all elements the charged ones left lanes idle in mixed warps and every element paid the
//    index arithmetic eight times over (256 x 256 x 128 elements at 0.5 K: 0.74 ms for the former pass).
//    The comparisons that find a point's zone are of integer keys (200 -> 186 us, fourth evaluation there).
//  - Node pass: K phi in the difference form of stiff_body (17 operations per node, where the three-stage
//    stencil took 25 and two gathered fields 14 more on tiles with 1.3 times the nodes), the corner loads
//    of four equal codes as one table entry, the diagonal from a per-plane table where no element adds to
//    it. 1.12 ms before at that size, 0.56 with the signs, magnitudes and zero tests on the FP64 pipe, 0.48
//    without them (24 operations per node with the halos; the pipe is 86 % busy).
#pragma once

namespace qcad {

constexpr int NODE_WARPS = 4;  // warps of the node pass, two node rows each

// Pass 1a for one element column (lanes hold consecutive columns) and layers [k0, k1).
__device__ __forceinline__ void residual_classify_body(const Grid<double>& g, const ResidualArgs& a, double* elR,
                                                       double* elD, int col, int k0, int k1) {
  const int lane = threadIdx.x & 31;
  const int ncol = g.nx * g.ny;
  const bool valid = col < ncol;
  const int j = valid ? col / g.nx : 0, i = valid ? col - j * g.nx : 0;
  const long long plane = g.plane;
  const double* phi = a.phi + i + (long long)g.nxn * j;
  // zone range of the column's four nodes on a plane: -1 (evaluate) or a zone, packed as (min, max)
  auto zones = [&](int k, int& lo, int& hi) {
    const double* q = phi + k * plane;
    const double v[4] = {__ldg(q), __ldg(q + 1), __ldg(q + g.nxn), __ldg(q + g.nxn + 1)};
    lo = 99;
    hi = -99;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int z = charge_zone_key(a.P, double_key(v[c]));
      lo = min(lo, z);
      hi = max(hi, z);
    }
  };
  int lo0 = 0, hi0 = 0;
  bool have = false;  // lo0, hi0 hold plane k
  for (int k = k0; k < k1; ++k) {
    const bool semi = a.layer_semi[k] && !a.linear;  // uniform
    const int e = valid ? col + ncol * k : 0;
    int zone = -2;  // no charge term at all (oxide)
    bool flat = true;
    if (semi) {
      int lo1, hi1;
      if (!have) zones(k, lo0, hi0);
      zones(k + 1, lo1, hi1);
      zone = min(lo0, lo1);
      flat = zone == max(hi0, hi1) && zone != -1;
      lo0 = lo1;
      hi0 = hi1;
    }
    have = semi;
    const bool app = valid && !flat;
    const unsigned m = __ballot_sync(FULL_MASK, app);
    if (m != 0) {
      int base = 0;
      if (lane == 0) base = atomicAdd(a.list_n, __popc(m));
      base = __shfl_sync(FULL_MASK, base, 0);
      if (app) {
        a.list[base + __popc(m & ((1u << lane) - 1))] = e;
        a.ecode[e] = 0;
      }
    }
    if (valid && flat) {
      const double th = a.theta ? a.theta[e] : 0.0;
      if (!nonzero_bits(th)) {
        // the element's corner loads are one table entry and its diagonal contributions zero
        a.ecode[e] = (unsigned char)(1 + (zone >= 0 ? (a.P.incomplete ? zone : WQ_ZONE_COMPLETE) : WQ_ZERO));
      } else {
        const double f = a.wq[8 * k + WQ_WEIGHT] * ((zone >= 0 ? zone_charge(a.P, zone) : 0.0) + th);
        double2* r = reinterpret_cast<double2*>(elR + 8LL * e);
        double2* d = reinterpret_cast<double2*>(elD + 8LL * e);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          r[q] = make_double2(f, f);
          d[q] = make_double2(0.0, 0.0);
        }
        a.ecode[e] = 0;
      }
    }
    // the flat elements' zero coefficients, a warp's 32 elements as one contiguous run
    const unsigned fl = __ballot_sync(FULL_MASK, valid && flat);
    const long long e0 = (long long)(col - lane) + (long long)ncol * k;
    if (a.c32) {
      float4* c = reinterpret_cast<float4*>(a.c32 + 8 * e0);
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if ((fl >> ((lane + 32 * h) >> 1)) & 1) c[lane + 32 * h] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    if (a.c64) {
      double2* c = reinterpret_cast<double2*>(a.c64 + 8 * e0);
#pragma unroll
      for (int h = 0; h < 4; ++h)
        if ((fl >> ((lane + 32 * h) >> 2)) & 1) c[lane + 32 * h] = make_double2(0.0, 0.0);
    }
  }
}

// Pass 1b: the listed elements, 8 lanes each (lane l: corner and Gauss point ix + 2 iy + 4 iz), block
// `blk` of `nblk`. A warp holds four elements; lanes beyond the list idle but stay in the shuffles.
__device__ __forceinline__ void residual_density_body(const Grid<double>& g, const ResidualArgs& a, double* elR,
                                                      double* elD, int blk, int nblk) {
  const int n = *a.list_n;
  const int l = threadIdx.x & 7;
  const double A = GaussConst<double>::a(), B = GaussConst<double>::b();
  const double A2 = A * A, B2 = B * B;
  const int per = blockDim.x >> 3;
  for (int first = blk * per; first < n; first += nblk * per) {
    const int q = first + (threadIdx.x >> 3);
    const bool valid = q < n;
    const int e = a.list[valid ? q : first];
    const int i = e % g.nx, r = e / g.nx;
    const int j = r % g.ny, k = r / g.ny;
    double v = __ldg(a.phi + (i + (l & 1)) + (long long)g.nxn * ((j + ((l >> 1) & 1)) + (long long)g.nyn * (k + (l >> 2))));
    v = A * v + B * __shfl_xor_sync(FULL_MASK, v, 1);
    v = A * v + B * __shfl_xor_sync(FULL_MASK, v, 2);
    v = A * v + B * __shfl_xor_sync(FULL_MASK, v, 4);
    const double w = a.wq[8 * k + WQ_WEIGHT];  // -(q/eps0) w|J|
    const Charge ch = charge_resid(a.P, v);
    double f = ch.rho;
    if (a.theta) f += a.theta[e];
    f *= w;
    double c = w * ch.drho;
    if (valid) {
      if (a.c64) a.c64[8LL * e + l] = c;
      if (a.c32) a.c32[8LL * e + l] = d2f_bits(c);
    }
    // an element with a nonzero coefficient marks its cell of the activity map
    const unsigned nz = __ballot_sync(FULL_MASK, nonzero_bits(c));
    if (valid && l == 0 && ((nz >> (threadIdx.x & 24)) & 0xffu) != 0) {
      const size_t cell = i / ACT_X + (size_t)act_cells(g.nx, ACT_X) * (j / ACT_Y + act_cells(g.ny, ACT_Y) * (k / ACT_Z));
      if (a.act64) a.act64[cell] = 1;
      if (a.act32) a.act32[cell] = 1;
    }
    f = A * f + B * __shfl_xor_sync(FULL_MASK, f, 1);
    f = A * f + B * __shfl_xor_sync(FULL_MASK, f, 2);
    f = A * f + B * __shfl_xor_sync(FULL_MASK, f, 4);
    if (nz != 0) {
      c = A2 * c + B2 * __shfl_xor_sync(FULL_MASK, c, 1);
      c = A2 * c + B2 * __shfl_xor_sync(FULL_MASK, c, 2);
      c = A2 * c + B2 * __shfl_xor_sync(FULL_MASK, c, 4);
    }
    if (valid) {
      elR[8LL * e + l] = f;
      elD[8LL * e + l] = c;
    }
  }
}

// Pass 2 for the warp whose first node row is jb and x tile bx (30 output columns), planes [k0, k1).
__device__ __forceinline__ void residual_node_body(const Grid<double>& g, const ResidualArgs& a, const double* elR,
                                                   const double* elD, int bx, int jb, int k0, int k1, double& acc_r2,
                                                   unsigned long long& acc_max) {
  const int lane = threadIdx.x & 31;
  const int i = bx * 30 - 1 + lane;
  const int plane = (int)g.plane;
  auto mirror = [](int q, int n) { return min(max(q < 0 ? -q : (q >= n ? 2 * (n - 1) - q : q), 0), n - 1); };
  const int im = mirror(i, g.nxn);
  int nrow[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) nrow[r] = im + g.nxn * mirror(jb - 1 + r, g.nyn);
  bool wr[2], top[2];
  int half[2];  // halvings of a boundary node's row
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int j = jb + r;
    wr[r] = i >= 0 && i < g.nxn && j < g.nyn && lane >= 1 && lane <= 30;
    top[r] = wr[r] && g.dir_top != nullptr && g.dir_top[nrow[r + 1]] != 0;
    half[r] = (i == 0 || i == g.nx) + (j == 0 || j == g.ny);
  }
  const bool edge = __any_sync(FULL_MASK, (half[0] | half[1]) != 0);  // a boundary tile
  // load codes of the elements (i, jb-1 .. jb+1) of a layer, a byte each; 255: no element
  const int eplane = g.nx * g.ny;
  auto codes = [&](int layer) {
    int p = 0;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const int je = jb - 1 + q;
      const bool in = i >= 0 && i < g.nx && je >= 0 && je < g.ny;
      p |= (in ? (int)a.ecode[i + g.nx * je + eplane * layer] : 255) << (8 * q);
    }
    return p;
  };
  const int kb = max(k0 - 1, 0), ke = min(k1, g.nzn - 1);
  double vn[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) vn[r] = __ldg(a.phi + nrow[r] + kb * plane);
  int cn = kb < ke ? codes(kb) : 0;  // of the layer above plane k, read one plane ahead
  double c1[3][2], c2[3][2], cold[2], up[2] = {0.0, 0.0}, dup[2] = {0.0, 0.0};
  bool dresp[2] = {false, false};
#pragma unroll
  for (int r = 0; r < 2; ++r) {
#pragma unroll
    for (int o = 0; o < 3; ++o) c1[o][r] = c2[o][r] = 0.0;
    cold[r] = 0.0;
  }
  // output plane k from the oldest sums, the loads of layer k - 1 (up, dup) and of layer k (lo, dlo);
  // resp: some adjacent element adds to the diagonal
  auto put = [&](int k, const double* lo, const double* dlo, const bool* resp) {
    const bool pdir = (g.dir_bottom && k == 0) || (g.dir_boundary && (k == 0 || k == g.nz));
    // interior stiffness diagonal of the plane; a boundary node has half or a quarter of it
    const double kd = __ldg(g.zs + 12 * k + 10);
    const float kf = d2f_bits(kd);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const double xs = __shfl_up_sync(FULL_MASK, c2[0][r], 1) + __shfl_down_sync(FULL_MASK, c2[0][r], 1);
      if (!wr[r]) continue;
      const int n = nrow[r + 1] + k * plane;
      double R = c1[0][r] + fma(-2.0, c2[0][r], xs);
      if (edge) {
        asm volatile("");  // keeps the product inside the branch
        R *= half[r] == 0 ? 1.0 : half[r] == 1 ? 0.5 : 0.25;
      }
      R += up[r] + lo[r];
      const bool dir = pdir || (k == g.nz && top[r]);
      if (dir) R = 0.0;
      a.R[n] = R;
      if (a.b64) a.b64[n] = neg_bits(R);
      if (a.b32) a.b32[n] = -d2f_bits(R);
      const float ff = half[r] == 0 ? 1.0f : half[r] == 1 ? 0.5f : 0.25f;
      const bool rs = resp[r] || dresp[r];
      if (a.dinv32 && !rs)  // the FP32 Jacobi scale as an FP32 reciprocal (within an ulp of the rounded inverse)
        a.dinv32[n] = dir ? 1.0f : __frcp_rn(ff * kf);
      if (rs || a.diag || a.dinv64) {
        double dg = kd * (half[r] == 0 ? 1.0 : half[r] == 1 ? 0.5 : 0.25);
        if (rs) dg += dup[r] + dlo[r];
        if (dir) dg = 1.0;
        if (a.diag) a.diag[n] = dg;
        if (a.dinv64) a.dinv64[n] = dir ? 1.0 : rs ? 1.0 / dg : __ldg(g.zs + 12 * k + 11) * (half[r] == 0 ? 1.0 : half[r] == 1 ? 2.0 : 4.0);
        if (a.dinv32 && rs) a.dinv32[n] = __frcp_rn(__double2float_rn(dg));
      }
      acc_r2 = fma(R, R, acc_r2);
      // max |R| by bit pattern (NaN left out, as fmax does)
      const unsigned long long b = abs_bits(R);
      if (b <= 0x7ff0000000000000ull && b > acc_max) acc_max = b;
    }
  };
  for (int k = kb; k <= ke; ++k) {
    double v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) v[r] = vn[r];
    const int code = cn;  // from the second plane on: of layer k - 1
    if (k < ke) {
#pragma unroll
      for (int r = 0; r < 4; ++r) vn[r] = __ldg(a.phi + nrow[r] + (k + 1) * plane);
    }
    double z[10];
#pragma unroll
    for (int q = 0; q < 10; ++q) z[q] = __ldg(g.zs + 12 * k + q);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const double c = v[r + 1];
      const double dy = fma(-2.0, c, v[r] + v[r + 2]);
#pragma unroll
      for (int o = 0; o < 3; ++o) {
        c1[o][r] = fma(z[3 * o], dy, c1[o][r]);
        c2[o][r] = fma(z[3 * o + 1], c, c2[o][r]);
        c2[o][r] = fma(z[3 * o + 2], dy, c2[o][r]);
      }
      const double d = k > kb ? c - cold[r] : 0.0;
      c1[0][r] = fma(-z[9], d, c1[0][r]);
      c1[1][r] = fma(z[9], d, c1[1][r]);
    }
    if (k > kb) {
      if (k < ke) cn = codes(k);
      // loads of layer k - 1: to its lower plane k - 1 (lo) and its upper plane k (hi)
      double lo[2], hi[2], dlo[2] = {0.0, 0.0}, dhi[2] = {0.0, 0.0};
      bool resp[2] = {false, false};
      const int left = __shfl_up_sync(FULL_MASK, code, 1);
      const double* wq = a.wq + 8 * (k - 1);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int pr = (code >> (8 * r)) & 0xffff, pl = (left >> (8 * r)) & 0xffff, c = pr & 255;
        if (pr == pl && c == (pr >> 8) && c != 0) {
          lo[r] = hi[r] = c == 255 ? 0.0 : times4(__ldg(wq + c - 1));
        } else {
          lo[r] = hi[r] = 0.0;
          if (!wr[r]) continue;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int ex = q & 1, ey = q >> 1;  // element (i - 1 + ex, j - 1 + ey)
            const int cc = ((ex ? pr : pl) >> (8 * ey)) & 255;
            if (cc == 255) continue;
            if (cc != 0) {
              const double t = __ldg(wq + cc - 1);
              lo[r] += t;
              hi[r] += t;
            } else {
              resp[r] = true;
              const long long at = 8LL * (i - 1 + ex + g.nx * (jb + r - 1 + ey) + (long long)eplane * (k - 1)) +
                                   (1 - ex) + 2 * (1 - ey);
              lo[r] += elR[at];
              hi[r] += elR[at + 4];
              dlo[r] += elD[at];
              dhi[r] += elD[at + 4];
            }
          }
        }
      }
      if (k - 1 >= k0) put(k - 1, lo, dlo, resp);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        up[r] = hi[r];
        dup[r] = dhi[r];
        dresp[r] = resp[r];
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      cold[r] = v[r + 1];
#pragma unroll
      for (int o = 0; o < 2; ++o) {
        c1[o][r] = c1[o + 1][r];
        c2[o][r] = c2[o + 1][r];
      }
      c1[2][r] = c2[2][r] = 0.0;
    }
  }
  if (k1 == g.nzn) {
    const double zero[2] = {0.0, 0.0};
    const bool none[2] = {false, false};
    put(k1 - 1, zero, zero, none);
  }
}

__device__ __forceinline__ void residual_node_finish(const ResidualArgs& a, double r2, unsigned long long rmax) {
  if (a.stats == nullptr) return;
  double s[1] = {r2};
  block_sum_atomic<1>(s, a.stats + 1);
  block_max_atomic(__longlong_as_double((long long)rmax), a.stats);
}

__global__ void __launch_bounds__(256) residual_classify_kernel(const __grid_constant__ Grid<double> g,
                                                                const __grid_constant__ ResidualArgs a, double* elR,
                                                                double* elD, int chunk) {
  const int k0 = blockIdx.y * chunk;
  residual_classify_body(g, a, elR, elD, blockIdx.x * 256 + threadIdx.x, k0, min(k0 + chunk, g.nz));
}
__global__ void __launch_bounds__(256) residual_density_kernel(const __grid_constant__ Grid<double> g,
                                                               const __grid_constant__ ResidualArgs a, double* elR,
                                                               double* elD) {
  residual_density_body(g, a, elR, elD, blockIdx.x, gridDim.x);
}
__global__ void __launch_bounds__(32 * NODE_WARPS) residual_node_kernel(const __grid_constant__ Grid<double> g,
                                                                        const __grid_constant__ ResidualArgs a,
                                                                        const double* elR, const double* elD,
                                                                        int kchunk) {
  const int k0 = blockIdx.z * kchunk;
  const int jb = 2 * (blockIdx.y * NODE_WARPS + (threadIdx.x >> 5));
  double r2 = 0.0;
  unsigned long long rmax = 0;
  if (jb < g.nyn) residual_node_body(g, a, elR, elD, blockIdx.x, jb, k0, min(k0 + kchunk, g.nzn), r2, rmax);
  residual_node_finish(a, r2, rmax);
}

// Blocks of the density pass: it strides over the list, whose length only the device knows.
inline int density_blocks(long long ne) {
  const long long b = (ne + 31) / 32, cap = 8LL * sm_count();
  return (int)(b < cap ? b : cap);
}
// Layers per block of the classification pass: a block rereads one plane's zones; four where that fills
// the SMs (8 blocks each), fewer on small grids.
inline int classify_chunk(int tiles, int nz) {
  int c = 4;
  while (c > 1 && (long long)tiles * ((nz + c - 1) / c) < 8LL * sm_count()) c /= 2;
  return c;
}
// z chunk of the node pass: bound by the SM's FP64 pipe, so an SM's time is its warps' planes.
inline int node_chunk(int nxn, int nyn, int nzn, const LaunchCfg& cfg) {
  if (!cfg.fit) return cfg.kchunk < nzn ? cfg.kchunk : nzn;
  const long long tiles = (long long)((nxn + 29) / 30) * ((nyn + 2 * NODE_WARPS - 1) / (2 * NODE_WARPS));
  double cost;
  return fit_chunk(tiles, nzn, sm_count(), 1.5, 32, &cost);
}

}  // namespace qcad
