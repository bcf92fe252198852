// Kernels of the entry points that read and write the caller's dense nodal
// arrays directly, without a copy into the padded level layout and back.
#pragma once
#include "mg_device.cuh"
#include "mg_zsoft.cuh"

namespace mgdev {

constexpr int DN_THREADS = 128;
constexpr int DN_TX = 32, DN_TY = 4;

// S of one point in float64 arithmetic, in stencil()'s order.  Not inlined: the
// compiler would otherwise run it at every point beside the fixed-point sum and
// select.
__device__ __noinline__ double dense_exact(double uw, double ue, double us, double un, double um, double up,
                                           const double* kx, const double* ky, const double* kz, int sy, int sz) {
  double S = __ldg(kx - 1) * uw;
  S = fma(__ldg(kx), ue, S);
  S = fma(__ldg(ky - sy), us, S);
  S = fma(__ldg(ky), un, S);
  S = fma(__ldg(kz - sz), um, S);
  return fma(__ldg(kz), up, S);
}

// y = A x for the float64 finest operator, x and y dense nodal arrays (nz + 2,
// ny + 2, nx + 2): y is written everywhere, 0 on the boundary, and boundary
// entries of x count as 0.  With SOFT a point's value is k_zsoft's bit for bit,
// otherwise OpApplyTo64's; dg is the stored float64 diagonal.
//
// What bounds it: issue slots; its rows are not aligned, so a load takes a line
// more than k_zsoft's.  Measured at 257^3: 183 us a call (48 bytes per point: 118 us of
// traffic; 202 us in float64 arithmetic alone).
// One thread owns a column of interior points and walks planes; the z
// neighbours stay in registers, the others come through L1, and the streamed
// arrays are prefetched into L2.  Warps with a point on the grid's x or y faces
// mask the neighbours outside and also write the boundary entries of y next to
// their points; the others do neither.
template <bool SOFT, bool EDGE>
__device__ __forceinline__ void dense_column(const double* __restrict__ x, double* __restrict__ y,
                                             const double* __restrict__ kx, const double* __restrict__ ky,
                                             const double* __restrict__ kz, const double* __restrict__ dg,
                                             const Geom& g, int i, int j, int k0, int k1) {
  const int sy = g.nx + 2, pz = (int)g.sz;
  const unsigned sz = (unsigned)sy * (g.ny + 2);
  unsigned q = (k0 + 1) * sz + (unsigned)((j + 1) * sy + i + 1);
  int p = (int)g.at(i, j, k0);
  const bool w = !EDGE || i > 0, e = !EDGE || i + 1 < g.nx, s = !EDGE || j > 0, n = !EDGE || j + 1 < g.ny;
  double um = k0 > 0 ? __ldg(x + (q - sz)) : 0.0, uc = __ldg(x + q);
  S64 sm = soft_unpack(um), sc = soft_unpack(uc), cm = soft_coef(__ldg(kz + p - pz));
  for (int k = k0; k < k1; ++k, q += sz, p += pz) {
    const bool top = k + 1 == g.nz;
    const double* xq = x + q;
    const double up = top ? 0.0 : __ldg(xq + sz), czp = __ldg(kz + p), d = __ldg(dg + p);
    const double cxm = __ldg(kx + p - 1), cxp = __ldg(kx + p), cym = __ldg(ky + p - g.Px), cyp = __ldg(ky + p);
    const double uw = w ? __ldg(xq - 1) : 0.0, ue = e ? __ldg(xq + 1) : 0.0;
    const double us = s ? __ldg(xq - sy) : 0.0, un = n ? __ldg(xq + sy) : 0.0;
    if (k + ZV_PF < k1) {
      const int o = p + ZV_PF * pz;
      pf_l2(kx + o);
      pf_l2(ky + o);
      pf_l2(kz + o);
      pf_l2(dg + o);
      pf_l2(xq + (ZV_PF + 1) * sz);
    }
    const S64 sp = soft_unpack(up), cp = soft_coef(czp);
    double S;
    if constexpr (SOFT) {
      if (!soft_stencil(sm, sp, us, un, uw, ue, cm, cp, cym, cyp, cxm, cxp, S))
        S = dense_exact(uw, ue, us, un, um, up, kx + p, ky + p, kz + p, g.Px, pz);
    } else {
      S = cxm * uw;
      S = fma(cxp, ue, S);
      S = fma(cym, us, S);
      S = fma(cyp, un, S);
      S = fma(__ldg(kz + p - pz), um, S);
      S = fma(czp, up, S);
    }
    double* yq = y + q;
    *yq = fma(d, uc, -S);
    if (k == 0) yq[-(i64)sz] = 0.0;
    if (top) yq[sz] = 0.0;
    if (EDGE && !(w && e && s && n)) {
      for (int c = k == 0 ? -1 : 0; c <= (top ? 1 : 0); ++c)
        for (int b = s ? 0 : -1; b <= (n ? 0 : 1); ++b)
          for (int a = w ? 0 : -1; a <= (e ? 0 : 1); ++a)
            if (a | b) yq[c * (i64)sz + (i64)b * sy + a] = 0.0;
    }
    sm = sc;
    sc = sp;
    cm = cp;
    um = uc;
    uc = up;
  }
}
template <bool SOFT>
__global__ void __launch_bounds__(DN_THREADS, 8)
    k_apply_dense(const double* __restrict__ x, double* __restrict__ y, const double* __restrict__ kx,
                  const double* __restrict__ ky, const double* __restrict__ kz, const double* __restrict__ dg, Geom g,
                  int kchunk) {
  const int i = blockIdx.x * DN_TX + (threadIdx.x & 31), j = blockIdx.y * DN_TY + (threadIdx.x >> 5);
  const int k0 = blockIdx.z * kchunk, k1 = min(k0 + kchunk, g.nz);
  if (j >= g.ny) return;  // whole warps
  const int i1 = (blockIdx.x + 1) * DN_TX;
  if (blockIdx.x > 0 && i1 < g.nx && j > 0 && j + 1 < g.ny) {
    dense_column<SOFT, false>(x, y, kx, ky, kz, dg, g, i, j, k0, k1);
  } else if (i < g.nx) {
    dense_column<SOFT, true>(x, y, kx, ky, kz, dg, g, i, j, k0, k1);
  }
}

// dL/dln k_c for every finest cell from the dense nodal arrays phi and lambda
// (boundary entries count as 0):
//   sum over the 12 edges e=(p,q) of the cell with an interior end point of
//   -h_a^-2 (lambda_p - lambda_q)(phi_p - phi_q) * dk_e/dln k_c,
//   dk_e/dln k_c = k_e^2/(4 k_c) (harmonic edge mean) or k_c/4 (arithmetic).
// With the stored float64 coefficient K_e = h_a^-2 k_e the harmonic term is
// -(dlam dphi K_e^2) h_a^2 / (4 k_c): the 12 means (5 float64 divisions each)
// need not be formed again, and an edge's value does not depend on the cell.
// wx, wy, wz are h_a^2 (harmonic) or h_a^-2 (arithmetic).
// K_e^2 may leave the range where k^2 / k does not, so a warp takes a power of
// two out of its K_e, near the reciprocal of its first cell's k 2^lg (2^lg about
// the largest h_a^-2), and puts it back at the end: neither changes a bit.
//
// What bounds it: the float64 pipe, about 43 operations per cell (one
// division among them); the 60 divisions per cell of the twelve means took
// 2.28 ms at 129^3, this kernel takes 0.25 ms with its call.  A thread owns the nodes (I, J) and (I, J + 1) of a
// column and walks node planes; the edges of column I + 1 come from the next
// lane (31 cells per warp), those of the plane below stay in registers.
constexpr int GR_TX = 31;
__global__ void __launch_bounds__(DN_THREADS)
    k_gradient(const double* __restrict__ kc, const double* __restrict__ phi, const double* __restrict__ lam,
               const double* __restrict__ kx, const double* __restrict__ ky, const double* __restrict__ kz, Geom g,
               double wx, double wy, double wz, int lg, int face_rule, int kchunk, double* __restrict__ grad) {
  const int lane = threadIdx.x & 31;
  const int cx = g.nx + 1, cy = g.ny + 1, cz = g.nz + 1;  // cells
  const int I = min(blockIdx.x * GR_TX + lane, cx), J = blockIdx.y * DN_TY + (threadIdx.x >> 5);
  if (J >= cy) return;  // whole warps
  const bool out = lane < GR_TX && blockIdx.x * GR_TX + lane < cx;
  const int K0 = blockIdx.z * kchunk, K1 = min(K0 + kchunk, cz);  // cell planes; node planes K0 .. K1
  const i64 sy = g.nx + 2, sz = sy * (g.ny + 2);
  const bool inx = I >= 1 && I <= g.nx;
  const bool in0 = inx && J >= 1, in1 = inx && J + 1 <= g.ny;  // rows J and J + 1
  i64 q = (i64)K0 * sz + (i64)J * sy + I;
  int p = (int)g.at(I - 1, J - 1, K0 - 1);
  double lm0 = 0.0, lm1 = 0.0, pm0 = 0.0, pm1 = 0.0, Pm = 0.0;
  // x: the exponent of the warp's first cell's k 2^lg; 2^x and 4 2^-x
  const unsigned long long first = dbits(__ldg(kc + ((i64)K0 * cy + J) * cx + blockIdx.x * GR_TX));
  const int x = min(max((int)(first >> 52) - 1023 + lg, -1000), 1000), dx = x * (1 << 20);
  const double up = bitsd((unsigned long long)(1023 + x) << 52), down4 = bitsd((unsigned long long)(1025 - x) << 52);
  auto edge = [&](double dl, double dp, const double* k, int at) {
    const double t = dl * dp;
    if (face_rule) return t;
    // 2^-x K by its exponent bits (five float64 products per cell more took 277 us instead of 247 at
    // 129^3).  A zero (t is 0 there) or a value out of range becomes some finite number.
    const double K = __ldg(k + at);
    const int hi = min(max(__double2hiint(K) - dx, 0), 0x7fe00000);
    const double c = __hiloint2double(hi, __double2loint(K));
    return t * (c * c);
  };
  auto east = [](double v) { return __shfl_down_sync(0xffffffffu, v, 1); };
  for (int K = K0; K <= K1; ++K, q += sz, p += (int)g.sz) {
    const bool ink = K >= 1 && K <= g.nz;
    const double l0 = in0 && ink ? __ldg(lam + q) : 0.0, l1 = in1 && ink ? __ldg(lam + q + sy) : 0.0;
    const double p0 = in0 && ink ? __ldg(phi + q) : 0.0, p1 = in1 && ink ? __ldg(phi + q + sy) : 0.0;
    const double tx = edge(east(l0) - l0, east(p0) - p0, kx, p) + edge(east(l1) - l1, east(p1) - p1, kx, p + g.Px);
    const double ty = edge(l1 - l0, p1 - p0, ky, p);
    const double P = fma(wx, tx, wy * (ty + east(ty)));
    if (K > K0) {  // the z edges between planes K - 1 and K complete the cells of plane K - 1
      const int pb = p - (int)g.sz;
      const double tz = edge(l0 - lm0, p0 - pm0, kz, pb) + edge(l1 - lm1, p1 - pm1, kz, pb + g.Px);
      const double acc = fma(wz, tz + east(tz), Pm + P);
      if (out) {
        const i64 c = ((i64)(K - 1) * cy + J) * cx + I;
        const double k = __ldg(kc + c);
        grad[c] = face_rule ? -0.25 * k * acc : up * (-acc / (down4 * k));
      }
    }
    lm0 = l0, lm1 = l1, pm0 = p0, pm1 = p1, Pm = P;
  }
}

}  // namespace mgdev
