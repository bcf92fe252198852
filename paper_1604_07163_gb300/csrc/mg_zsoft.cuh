// Driver of the float64 stencil passes with most of a point's products on the
// integer pipe (mg_soft64.cuh): the CG operator, the operator on a V-cycle
// vector, the float64 residual and the float64 form's smoothing steps, on every
// level above the bottom kernel.
#pragma once
#include "mg_krylov.cuh"
#include "mg_soft64.cuh"
#include "mg_zvec.cuh"

namespace mgdev {

// S of stencil() at one point: the z and y products in fixed point, the two x
// products as float64 multiply-adds.  The x neighbours stay on the float64 pipe
// because an unpacked operand serves the z products of three planes but would
// serve an x product once.  False where soft_sum4 declines.
__device__ __forceinline__ bool soft_stencil(const S64& um, const S64& up, double us, double un, double uw, double ue,
                                             const S64& czm, const S64& czp, double cym, double cyp, double cxm,
                                             double cxp, double& S) {
  const S64 a[4] = {um, up, soft_unpack(us), soft_unpack(un)};
  const S64 c[4] = {czm, czp, soft_coef(cym), soft_coef(cyp)};
  const bool ok = soft_sum4(a, c, S);
  S = fma(cxm, uw, S);
  S = fma(cxp, ue, S);
  return ok;
}

// Per-operation hooks:
//   center   the pass has the stored float64 diagonal: v = A u = dg u - S; otherwise v = S
//   u, dg, kx, ky, kz   operand, diagonal and edge coefficients
//   load_p   the values read pointwise; prefetch: their L2 prefetch
//   emit     the point operation for v and the operand's value uc
template <class Op> struct Zs {
  static constexpr bool ok = false;
};

template <class Op_, bool CEN> struct ZsBase {
  using Op = Op_;
  static constexpr bool ok = true, center = CEN;
  struct P {};
  static __device__ __forceinline__ const double* kx(const Op& o) { return o.kx; }
  static __device__ __forceinline__ const double* ky(const Op& o) { return o.ky; }
  static __device__ __forceinline__ const double* kz(const Op& o) { return o.kz; }
  static __device__ __forceinline__ void prefetch(const Op&, int) {}
};

template <> struct Zs<OpApplyPQ> : ZsBase<OpApplyPQ, true> {
  static __device__ __forceinline__ const double* u(const Op& o) { return o.p; }
  static __device__ __forceinline__ const double* dg(const Op& o) { return o.dg; }
  static __device__ __forceinline__ void load_p(const Op&, int, P&) {}
  static __device__ __forceinline__ void emit(const Op& o, int p, double v, double uc, const P&, double& a0) {
    o.q[p] = v;
    a0 = fma(uc, v, a0);
  }
};

template <class TZ> struct Zs<OpApplyTo64<TZ>> : ZsBase<OpApplyTo64<TZ>, true> {
  using Op = OpApplyTo64<TZ>;
  using P = typename ZsBase<Op, true>::P;
  static __device__ __forceinline__ const TZ* u(const Op& o) { return o.u; }
  static __device__ __forceinline__ const double* dg(const Op& o) { return o.dg; }
  static __device__ __forceinline__ void load_p(const Op&, int, P&) {}
  static __device__ __forceinline__ void emit(const Op& o, int p, double v, double, const P&, double&) { o.y[p] = v; }
};

template <> struct Zs<OpResidualD<double>> : ZsBase<OpResidualD<double>, true> {
  struct P {
    double b;
  };
  static __device__ __forceinline__ const double* u(const Op& o) { return o.x; }
  static __device__ __forceinline__ const double* dg(const Op& o) { return o.dg; }
  static __device__ __forceinline__ void load_p(const Op& o, int p, P& q) { q.b = __ldg(o.b + p); }
  static __device__ __forceinline__ void prefetch(const Op& o, int p) { pf_l2(o.b + p); }
  static __device__ __forceinline__ void emit(const Op& o, int p, double v, double, const P& q, double& a0) {
    const double r = q.b - v;
    o.r[p] = r;
    a0 = fma(r, r, a0);
  }
};

using OpStep64 = OpChebStep<double, double, double>;
struct ZsStepP {
  double b, d, di;
};
__device__ __forceinline__ void zs_step_load(const OpStep64& o, int p, ZsStepP& q) {
  q.b = __ldg(o.b + p);
  q.di = __ldg(o.dinv + p);
  if (o.dprev && o.dprev != o.x) q.d = __ldg(o.dprev + p);
}
// d_{j-1} at the point: after step 0 from a zero guess it is the iterate itself
__device__ __forceinline__ double zs_d(const OpStep64& o, double xp, const ZsStepP& q) {
  return o.dprev == o.x ? xp : q.d;
}
__device__ __forceinline__ void zs_step_prefetch(const OpStep64& o, int p) {
  pf_l2(o.b + p);
  pf_l2(o.dinv + p);
  if (o.dprev && o.dprev != o.x) pf_l2(o.dprev + p);
}
// A sweep's last step needs no direction: x + c1 d + c2 s as two multiply-adds
// instead of a product, a multiply-add and an addition (with the direction that
// is the iterate itself not read again, a step went from 274 to 231 us at 257^3).
__device__ __forceinline__ double zs_step_emit(const OpStep64& o, int p, double S, double xp, const ZsStepP& q) {
  const double s = fma(q.di, q.b + S, -xp);
  double xn;
  if (o.dout) {
    const double dn = o.dprev ? fma(o.c1, zs_d(o, xp, q), o.c2 * s) : s * o.inv_theta;
    xn = xp + dn;
    o.dout[p] = dn;
  } else {
    xn = o.dprev ? fma(o.c2, s, fma(o.c1, zs_d(o, xp, q), xp)) : fma(s, o.inv_theta, xp);
  }
  o.xout[p] = xn;
  return xn;
}
template <> struct Zs<OpStep64> : ZsBase<OpStep64, false> {
  using P = ZsStepP;
  static __device__ __forceinline__ const double* u(const Op& o) { return o.x; }
  static __device__ __forceinline__ const double* dg(const Op&) { return nullptr; }
  static __device__ __forceinline__ void load_p(const Op& o, int p, P& q) { zs_step_load(o, p, q); }
  static __device__ __forceinline__ void prefetch(const Op& o, int p) { zs_step_prefetch(o, p); }
  static __device__ __forceinline__ void emit(const Op& o, int p, double v, double uc, const P& q, double&) {
    zs_step_emit(o, p, v, uc, q);
  }
};
using OpStepDot64 = OpChebStepDot<double, double, double>;
template <> struct Zs<OpStepDot64> : ZsBase<OpStepDot64, false> {
  using P = ZsStepP;
  static __device__ __forceinline__ const double* u(const Op& o) { return o.step.x; }
  static __device__ __forceinline__ const double* dg(const Op&) { return nullptr; }
  static __device__ __forceinline__ const double* kx(const Op& o) { return o.step.kx; }
  static __device__ __forceinline__ const double* ky(const Op& o) { return o.step.ky; }
  static __device__ __forceinline__ const double* kz(const Op& o) { return o.step.kz; }
  static __device__ __forceinline__ void load_p(const Op& o, int p, P& q) { zs_step_load(o.step, p, q); }
  static __device__ __forceinline__ void prefetch(const Op& o, int p) { zs_step_prefetch(o.step, p); }
  static __device__ __forceinline__ void emit(const Op& o, int p, double v, double uc, const P& q, double& a0) {
    a0 = fma(q.b, zs_step_emit(o.step, p, v, uc, q), a0);
  }
};

// S of point p in float64 arithmetic.  Where a field vanishes, as off the support
// of a source, every point comes here: with two products instead of six a float64
// V-cycle on zeros takes 1.75 ms at 257^3 (2.20; on other fields 1.48, and 2.13 with
// float64 arithmetic throughout).  The dense product was slower with the test (352 against 276 us).
template <class TU>
__device__ __noinline__ double zs_exact(const TU* u, const double* kx, const double* ky, const double* kz,
                                        const Geom& g, int p) {
  const int sz = (int)g.sz, sy = g.Px;
  double D, z;
  if (all_zero(to_double(__ldg(u + p - sz)), to_double(__ldg(u + p + sz)), to_double(__ldg(u + p - sy)),
               to_double(__ldg(u + p + sy)), z))
    return fma(__ldg(kx + p), to_double(__ldg(u + p + 1)), fma(__ldg(kx + p - 1), to_double(__ldg(u + p - 1)), z));
  typename OpApplyTo64<TU>::Ld lu{u};
  return stencil<true, double>(g, p, lu, kx, ky, kz, D);
}

// One thread owns a column of the level and walks planes; the operand's z
// neighbours and the z coefficients stay unpacked in registers.
//
// What bounds it: issue slots and the float64 pipe, about evenly, over 48 bytes
// per point of traffic.  With four float64 operations per point left on that
// pipe the CG operator takes 166 us at 257^3 (eight: 248 us; 118 us of traffic)
// and 1.21 ms at 513^3 (1.85 ms).  The float64 form's smoothing step keeps six
// (231 us a step, in float64 arithmetic 346 us), its residual four (168 us, before 244 us).  Measured on the
// operator at 257^3: two points per thread, at 120 registers, 14 us slower; a
// plane's loads kept in registers one plane ahead 10 to 25 us slower; 9 to 12
// resident blocks 4 to 50 us slower.
constexpr int ZS_TX = 32, ZS_TY = 4;
constexpr int ZS_BLOCKS = 8;  // resident blocks per SM: 64 registers per thread
constexpr int ZS_CHUNK = 8;   // least planes per block on large levels
template <class Op, bool RED>
__global__ void __launch_bounds__(ZV_THREADS, ZS_BLOCKS)
    k_zsoft(Op op, Geom g, int kchunk, double* partials, int stride) {
  using Z = Zs<Op>;
  constexpr bool CEN = Z::center;
  pdl_wait();
  const int i = blockIdx.x * ZS_TX + (threadIdx.x & 31);
  const int j = blockIdx.y * ZS_TY + (threadIdx.x >> 5);
  const int k0 = blockIdx.z * kchunk;
  const int k1 = min(k0 + kchunk, g.nz);
  double a0 = 0.0, a1 = 0.0;
  if (i < g.nx && j < g.ny) {
    const int sz = (int)g.sz, sy = g.Px;
    int p = (int)g.at(i, j, k0);
    const auto* u = Z::u(op);
    const double *kx = Z::kx(op), *ky = Z::ky(op), *kz = Z::kz(op), *dg = Z::dg(op);
    double uc = to_double(__ldg(u + p));
    S64 sm = soft_unpack(to_double(__ldg(u + p - sz))), sc = soft_unpack(uc), cm = soft_coef(__ldg(kz + p - sz));
    for (int k = k0; k < k1; ++k, p += sz) {
      const double up = to_double(__ldg(u + p + sz)), czp = __ldg(kz + p);
      const double cxm = __ldg(kx + p - 1), cxp = __ldg(kx + p), cym = __ldg(ky + p - sy), cyp = __ldg(ky + p);
      double d = 0.0;
      if constexpr (CEN) d = __ldg(dg + p);
      typename Z::P pw;
      Z::load_p(op, p, pw);
      const double uw = to_double(__ldg(u + p - 1)), ue = to_double(__ldg(u + p + 1));
      const double us = to_double(__ldg(u + p - sy)), un = to_double(__ldg(u + p + sy));
      if (k + ZV_PF < k1) {
        const int q = p + ZV_PF * sz;
        pf_l2(kx + q);
        pf_l2(ky + q);
        pf_l2(kz + q);
        pf_l2(u + q + sz);
        if constexpr (CEN) pf_l2(dg + q);
        Z::prefetch(op, q);
      }
      const S64 sp = soft_unpack(up), cp = soft_coef(czp);
      double v;
      if (!soft_stencil(sm, sp, us, un, uw, ue, cm, cp, cym, cyp, cxm, cxp, v)) v = zs_exact(u, kx, ky, kz, g, p);
      if constexpr (CEN) v = fma(d, uc, -v);
      Z::emit(op, p, v, uc, pw, a0);
      sm = sc;
      sc = sp;
      cm = cp;
      uc = up;
    }
  }
  pdl_trigger();
  if constexpr (RED) {
    block_sum2<ZV_THREADS>(a0, a1);
    if (threadIdx.x == 0) {
      const int b = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
      partials[b] = a0;
      partials[stride + b] = a1;
    }
  }
}

}  // namespace mgdev
