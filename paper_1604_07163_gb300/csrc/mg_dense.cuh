// Kernels of the entry points that read and write the caller's dense nodal
// arrays directly, without a copy into the padded level layout and back.
#pragma once
#include "mg_device.cuh"

namespace mgdev {

constexpr int DN_THREADS = 128;
constexpr int DN_TX = 32, DN_TY = 4;

// y = A x for the float64 finest operator, x and y dense nodal arrays (Nz, Ny,
// Nx): y is written everywhere, 0 on the boundary, and boundary entries of x
// count as 0.  The arithmetic is OpApply's, term for term, with the stored
// float64 diagonal dg (the sum OpApply forms again at every point).
//
// What bounds it: seven float64 operations per point on GB300's float64 pipe
// (2 per clock and SM: 185 us at 257^3) against 48 bytes per point (118 us).
// Measured at 257^3: 202 us a call; a copy into the padded layout, the product
// with the diagonal summed at every point (12 operations) and a copy back took
// 510 us (65^3, where launches count: 21 -> 14 us).
// One thread owns a column of nodes and walks planes; the z neighbours stay in
// registers, the others come through L1.
__global__ void __launch_bounds__(DN_THREADS, 8)
    k_apply_dense(const double* __restrict__ x, double* __restrict__ y, const double* __restrict__ kx,
                  const double* __restrict__ ky, const double* __restrict__ kz, const double* __restrict__ dg, Geom g,
                  int kchunk) {
  const int I = blockIdx.x * DN_TX + (threadIdx.x & 31), J = blockIdx.y * DN_TY + (threadIdx.x >> 5);
  const int Nx = g.nx + 2, Ny = g.ny + 2, Nz = g.nz + 2;
  if (I >= Nx || J >= Ny) return;
  const int K0 = blockIdx.z * kchunk, K1 = min(K0 + kchunk, Nz);
  const i64 sy = Nx, sz = (i64)Nx * Ny;
  i64 q = (i64)K0 * sz + (i64)J * sy + I;
  const bool in = I >= 1 && I <= g.nx && J >= 1 && J <= g.ny;
  const bool w = I >= 2, e = I <= g.nx - 1, s = J >= 2, n = J <= g.ny - 1;  // neighbours inside the boundary
  int p = (int)g.at(I - 1, J - 1, K0 - 1);
  auto at = [&](i64 o, int K) { return in && K >= 1 && K <= g.nz ? __ldg(x + o) : 0.0; };
  double um = at(q - sz, K0 - 1), uc = at(q, K0);
  for (int K = K0; K < K1; ++K, q += sz, p += (int)g.sz) {
    const double up = at(q + sz, K + 1);
    double v = 0.0;
    if (in && K >= 1 && K <= g.nz) {
      const double uw = w ? __ldg(x + q - 1) : 0.0, ue = e ? __ldg(x + q + 1) : 0.0;
      const double us = s ? __ldg(x + q - sy) : 0.0, un = n ? __ldg(x + q + sy) : 0.0;
      double S = __ldg(kx + p - 1) * uw;
      S = fma(__ldg(kx + p), ue, S);
      S = fma(__ldg(ky + p - g.Px), us, S);
      S = fma(__ldg(ky + p), un, S);
      S = fma(__ldg(kz + p - (int)g.sz), um, S);
      S = fma(__ldg(kz + p), up, S);
      v = fma(__ldg(dg + p), uc, -S);
    }
    y[q] = v;
    um = uc;
    uc = up;
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
//
// What bounds it: the float64 pipe, about 43 operations per cell (one
// division among them); the 60 divisions per cell of the twelve means took
// 2.28 ms at 129^3, this kernel takes 0.29 ms with its call.  A thread owns the nodes (I, J) and (I, J + 1) of a
// column and walks node planes; the edges of column I + 1 come from the next
// lane (31 cells per warp), those of the plane below stay in registers.
constexpr int GR_TX = 31;
__global__ void __launch_bounds__(DN_THREADS)
    k_gradient(const double* __restrict__ kc, const double* __restrict__ phi, const double* __restrict__ lam,
               const double* __restrict__ kx, const double* __restrict__ ky, const double* __restrict__ kz, Geom g,
               double wx, double wy, double wz, int face_rule, int kchunk, double* __restrict__ grad) {
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
  auto edge = [&](double dl, double dp, const double* k, int at) {
    const double t = dl * dp;
    if (face_rule) return t;
    const double c = __ldg(k + at);
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
        grad[c] = face_rule ? -0.25 * k * acc : -acc / (4.0 * k);
      }
    }
    lm0 = l0, lm1 = l1, pm0 = p0, pm1 = p1, Pm = P;
  }
}

}  // namespace mgdev
