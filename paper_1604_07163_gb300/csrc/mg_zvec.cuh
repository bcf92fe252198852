// Vectorised z-marching driver for the stencil passes (default kernel).
//
// Each thread owns four (float64: two) consecutive x points of a row and walks a
// chunk of planes:
//   - every array row is read with 16-byte loads, and the x neighbours come from
//     the adjacent lanes by warp shuffles (from memory at the ends of a row's
//     lanes);
//   - the operand's z neighbours live in a register queue (planes k-1, k, k+1),
//     and everything read pointwise is loaded one plane ahead of its use;
//   - every streamed array is prefetched into L2 two planes ahead.
// The arithmetic is that of stencil() and the per-point operations in
// mg_device.cuh, term for term and in the same order, so results are
// bitwise identical to the one-point-per-thread kernel (only the block sums
// of the reducing passes group terms differently).
//
// What bounds it (float32): memory traffic and its latency; a warp issues on
// about 36% of the cycles.  257^3, two points per thread (115 instructions a
// point, issuing on 60 to 68%) and four: zero-guess step 92 -> 77 us (59 us of
// traffic), step 83 -> 82 (69), residual 68 -> 66 (59); 127^3 step 14.4 -> 12.2.
#pragma once
#include <type_traits>

#include "mg_device.cuh"

namespace mgdev {

constexpr int ZV_THREADS = 128;
constexpr int ZV_TX = 64, ZV_TY = 4;  // tile: 32 lanes x 2 points, 4 rows
constexpr int ZV_PF = 2;              // L2 prefetch distance in planes

// Two consecutive elements at a (a's index is even, so the vector access is
// aligned), converted to R.
template <class R> __device__ __forceinline__ void ld2(const float* a, R (&v)[2]) {
  const float2 t = __ldg(reinterpret_cast<const float2*>(a));
  v[0] = cvt<R>(t.x);
  v[1] = cvt<R>(t.y);
}
template <class R> __device__ __forceinline__ void ld2(const double* a, R (&v)[2]) {
  const double2 t = __ldg(reinterpret_cast<const double2*>(a));
  v[0] = cvt<R>(t.x);
  v[1] = cvt<R>(t.y);
}
template <class R> __device__ __forceinline__ void ld2(const __nv_bfloat16* a, R (&v)[2]) {
  const __nv_bfloat162 t = __ldg(reinterpret_cast<const __nv_bfloat162*>(a));
  v[0] = cvt<R>(t.x);
  v[1] = cvt<R>(t.y);
}
// Stores the first n (0, 1 or 2) of two consecutive results.
template <class R> __device__ __forceinline__ void st2(float* a, const R (&v)[2], int n) {
  if (n == 2) *reinterpret_cast<float2*>(a) = make_float2(store_as<float>(v[0]), store_as<float>(v[1]));
  else if (n == 1) a[0] = store_as<float>(v[0]);
}
template <class R> __device__ __forceinline__ void st2(double* a, const R (&v)[2], int n) {
  if (n == 2) *reinterpret_cast<double2*>(a) = make_double2(store_as<double>(v[0]), store_as<double>(v[1]));
  else if (n == 1) a[0] = store_as<double>(v[0]);
}
// NP (2 or 4) consecutive elements
template <class R> __device__ __forceinline__ void ldn(const float* a, R (&v)[4]) {
  const float4 t = __ldg(reinterpret_cast<const float4*>(a));
  v[0] = cvt<R>(t.x), v[1] = cvt<R>(t.y), v[2] = cvt<R>(t.z), v[3] = cvt<R>(t.w);
}
template <class R> __device__ __forceinline__ void ldn(const __nv_bfloat16* a, R (&v)[4]) {
  const uint2 t = __ldg(reinterpret_cast<const uint2*>(a));
  const __nv_bfloat162 lo = *reinterpret_cast<const __nv_bfloat162*>(&t.x);
  const __nv_bfloat162 hi = *reinterpret_cast<const __nv_bfloat162*>(&t.y);
  v[0] = cvt<R>(lo.x), v[1] = cvt<R>(lo.y), v[2] = cvt<R>(hi.x), v[3] = cvt<R>(hi.y);
}
template <class R, class T> __device__ __forceinline__ void ldn(const T* a, R (&v)[2]) { ld2(a, v); }
// Stores the first n of NP results.
template <class R> __device__ __forceinline__ void stn(float* a, const R (&v)[4], int n) {
  if (n >= 4) {
    *reinterpret_cast<float4*>(a) = make_float4(v[0], v[1], v[2], v[3]);
    return;
  }
#pragma unroll
  for (int e = 0; e < 3; ++e)
    if (e < n) a[e] = v[e];
}
template <class R, class T> __device__ __forceinline__ void stn(T* a, const R (&v)[2], int n) { st2(a, v, min(n, 2)); }
__device__ __forceinline__ void pf_l2(const void* a) { asm volatile("prefetch.global.L2 [%0];" ::"l"(a)); }

// Stencil neighbourhood of a thread's NP points p, p+1, ..: operand values u and edge
// coefficients (c_x of the edge entering point 0 comes from the left lane).
template <class R, int NP> struct ZvNb {
  R uw, ue, cxw;
  R uc[NP], um[NP], up[NP], us[NP], un[NP];
  R cx[NP], cys[NP], cy[NP], czm[NP], cz[NP];
  // S and D of stencil() for element e
  __device__ __forceinline__ R eval(int e, R& D) const {
    const R cxm = e == 0 ? cxw : cx[e > 0 ? e - 1 : 0];
    const R xw = e == 0 ? uw : uc[e > 0 ? e - 1 : 0];
    const R xe = e == NP - 1 ? ue : uc[e < NP - 1 ? e + 1 : e];
    D = ((cxm + cx[e]) + (cys[e] + cy[e])) + (czm[e] + cz[e]);
    R S = cxm * xw;
    S = fma(cx[e], xe, S);
    S = fma(cys[e], us[e], S);
    S = fma(cy[e], un[e], S);
    S = fma(czm[e], um[e], S);
    S = fma(cz[e], up[e], S);
    return S;
  }
};

// Per-operation hooks.  ok = false keeps an operation on the scalar driver.
//   U      operand storage of NP points (what the stencil is applied to)
//   P      values read pointwise at the NP points of the current plane
//   load_u / vals / u_one   operand of NP points / as values / of one point
//   load_p                  pointwise values of a plane
//   prefetch(qp, qu)        L2 prefetch of the pointwise arrays at qp and of
//                           the operand arrays at qu
//   emit                    the point operation for the first nv points
// points per thread: 16-byte vectors
template <class R> constexpr int ZV_NP = sizeof(R) == 8 ? 2 : 4;

template <class Op> struct Zv {
  static constexpr bool ok = false;
};

template <class R, class TV> struct ZvVecU {
  static constexpr int NP = ZV_NP<R>;
  struct U {
    R v[NP];
  };
  static __device__ __forceinline__ void load(const TV* a, int p, U& u) { ldn(a + p, u.v); }
  static __device__ __forceinline__ void vals(const U& u, R (&v)[NP]) {
#pragma unroll
    for (int e = 0; e < NP; ++e) v[e] = u.v[e];
  }
  static __device__ __forceinline__ R one(const TV* a, int q) { return cvt<R>(__ldg(a + q)); }
};

// y = A u
template <class R_, class TV, class TC_> struct Zv<OpApply<R_, TV, TC_>> {
  using Op = OpApply<R_, TV, TC_>;
  using R = R_;
  static constexpr int NP = ZV_NP<R>;
  using TC = TC_;
  using UU = ZvVecU<R, TV>;
  using U = typename UU::U;
  struct P {};
  static constexpr bool ok = true;
  static __device__ __forceinline__ const TC* kx(const Op& o) { return o.kx; }
  static __device__ __forceinline__ const TC* ky(const Op& o) { return o.ky; }
  static __device__ __forceinline__ const TC* kz(const Op& o) { return o.kz; }
  static __device__ __forceinline__ void load_u(const Op& o, int p, U& u) { UU::load(o.u, p, u); }
  static __device__ __forceinline__ void vals(const Op&, const U& u, R (&v)[NP]) { UU::vals(u, v); }
  static __device__ __forceinline__ R u_one(const Op& o, int q) { return UU::one(o.u, q); }
  static __device__ __forceinline__ void load_p(const Op&, int, P&) {}
  static __device__ __forceinline__ void prefetch(const Op& o, int, int qu) { pf_l2(o.u + qu); }
  static __device__ __forceinline__ void emit(const Op& o, int p, int nv, const ZvNb<R, NP>& nb, const U&, const P&,
                                              double&, double&) {
    R y[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      R D;
      const R S = nb.eval(e, D);
      y[e] = D * nb.uc[e] - S;
    }
    stn(o.y + p, y, nv);
  }
};

// Chebyshev step (OpChebStep): the pointwise part shared with the fused dot.
template <class R, class TV, class TC> struct ZvStepP {
  static constexpr int NP = ZV_NP<R>;
  R b[NP], d[NP], di[NP];
};
template <class R, class TV, class TC>
__device__ __forceinline__ void zv_step_load_p(const OpChebStep<R, TV, TC>& o, int p, ZvStepP<R, TV, TC>& P) {
  ldn(o.b + p, P.b);
  if (o.dprev) ldn(o.dprev + p, P.d);
  if constexpr (sizeof(R) == 8) ldn(o.dinv + p, P.di);
}
template <class R, class TV, class TC>
__device__ __forceinline__ void zv_step_prefetch(const OpChebStep<R, TV, TC>& o, int qp, int qu) {
  pf_l2(o.x + qu);
  pf_l2(o.b + qp);
  if (o.dprev) pf_l2(o.dprev + qp);
  if constexpr (sizeof(R) == 8) pf_l2(o.dinv + qp);
}
// x_{j+1} of the two points, stored; returns them in xn
template <class R, class TV, class TC, int NP>
__device__ __forceinline__ void zv_step_emit(const OpChebStep<R, TV, TC>& o, int p, int nv, const ZvNb<R, NP>& nb,
                                             const ZvStepP<R, TV, TC>& P, R (&xn)[NP]) {
  R dn[NP];
  if constexpr (sizeof(R) == 4) {
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      R D;
      const R S = nb.eval(e, D);
      const R xp = nb.uc[e];
      const R s = fma((R)1 / D, P.b[e] + S, -xp);
      dn[e] = o.dprev ? fma(o.c1, P.d[e], o.c2 * s) : s * o.inv_theta;
      xn[e] = xp + dn[e];
    }
  } else {
    // one branch for all points: a selection formed both directions, on the float64 pipe (step at 257^3 390 us,
    // this 344)
    R s[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      R D;
      const R S = nb.eval(e, D);
      s[e] = fma(P.di[e], P.b[e] + S, -nb.uc[e]);
    }
    if (o.dprev) {
#pragma unroll
      for (int e = 0; e < NP; ++e) dn[e] = fma(o.c1, P.d[e], o.c2 * s[e]);
    } else {
#pragma unroll
      for (int e = 0; e < NP; ++e) dn[e] = s[e] * o.inv_theta;
    }
#pragma unroll
    for (int e = 0; e < NP; ++e) xn[e] = __dadd_rn(nb.uc[e], dn[e]);
  }
  stn(o.xout + p, xn, nv);
  if (o.dout) stn(o.dout + p, dn, nv);
}

template <class R_, class TV, class TC_> struct Zv<OpChebStep<R_, TV, TC_>> {
  using Op = OpChebStep<R_, TV, TC_>;
  using R = R_;
  static constexpr int NP = ZV_NP<R>;
  using TC = TC_;
  using UU = ZvVecU<R, TV>;
  using U = typename UU::U;
  using P = ZvStepP<R, TV, TC>;
  static constexpr bool ok = true;
  static __device__ __forceinline__ const TC* kx(const Op& o) { return o.kx; }
  static __device__ __forceinline__ const TC* ky(const Op& o) { return o.ky; }
  static __device__ __forceinline__ const TC* kz(const Op& o) { return o.kz; }
  static __device__ __forceinline__ void load_u(const Op& o, int p, U& u) { UU::load(o.x, p, u); }
  static __device__ __forceinline__ void vals(const Op&, const U& u, R (&v)[NP]) { UU::vals(u, v); }
  static __device__ __forceinline__ R u_one(const Op& o, int q) { return UU::one(o.x, q); }
  static __device__ __forceinline__ void load_p(const Op& o, int p, P& q) { zv_step_load_p(o, p, q); }
  static __device__ __forceinline__ void prefetch(const Op& o, int qp, int qu) { zv_step_prefetch(o, qp, qu); }
  static __device__ __forceinline__ void emit(const Op& o, int p, int nv, const ZvNb<R, NP>& nb, const U&, const P& q,
                                              double&, double&) {
    R xn[NP];
    zv_step_emit(o, p, nv, nb, q, xn);
  }
};

// Compensated dot-product step (Ogita, Rump and Oishi, "Accurate sum and dot
// product", SIAM J. Sci. Comput. 2005, algorithm Dot2): adds x*y to the
// float-float accumulator (s, c).  x*y = h + r exactly (TwoProduct via FMA),
// s + h = t + q exactly (Knuth's TwoSum), and c collects q + r.  After n terms
// s + c is the dot product with error at most about (n u)^2 sum |x y|, u =
// 2^-24, i.e. as if summed in twice the float32 precision.  The __f*_rn
// intrinsics keep the compiler from contracting the product into the sums.
__device__ __forceinline__ void dot2_add(float x, float y, float& s, float& c) {
  const float h = __fmul_rn(x, y);
  const float r = fmaf(x, y, -h);
  const float t = __fadd_rn(s, h);
  const float bp = __fsub_rn(t, s);
  const float q = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(h, bp));
  s = t;
  c = __fadd_rn(c, __fadd_rn(q, r));
}

// Ops whose Zv hooks define float_acc = true sum their per-point terms in a
// float-float pair per thread (emit_f), which the driver adds into the
// float64 block sum after its plane loop.
template <class Z, class = void> struct ZvFloatAcc : std::false_type {};
template <class Z>
struct ZvFloatAcc<Z, std::void_t<decltype(Z::float_acc)>> : std::integral_constant<bool, Z::float_acc> {};

// last post-smoothing step with rho = b.z accumulated (OpChebStepDot: b is
// the right-hand side the step already reads, held exactly in R).  float64
// form: one float64 FMA per point.  Float32 V-cycle forms: the products of
// the float32 b and z are summed per thread with dot2_add on the float32
// pipe, so the pass needs no widening and no float64 operation per point.
template <class R_, class TV, class TC_> struct Zv<OpChebStepDot<R_, TV, TC_>> {
  using Op = OpChebStepDot<R_, TV, TC_>;
  using R = R_;
  static constexpr int NP = ZV_NP<R>;
  using TC = TC_;
  using UU = ZvVecU<R, TV>;
  using U = typename UU::U;
  using P = ZvStepP<R, TV, TC>;
  static constexpr bool ok = true;
  static __device__ __forceinline__ const TC* kx(const Op& o) { return o.step.kx; }
  static __device__ __forceinline__ const TC* ky(const Op& o) { return o.step.ky; }
  static __device__ __forceinline__ const TC* kz(const Op& o) { return o.step.kz; }
  static __device__ __forceinline__ void load_u(const Op& o, int p, U& u) { UU::load(o.step.x, p, u); }
  static __device__ __forceinline__ void vals(const Op&, const U& u, R (&v)[NP]) { UU::vals(u, v); }
  static __device__ __forceinline__ R u_one(const Op& o, int q) { return UU::one(o.step.x, q); }
  static __device__ __forceinline__ void load_p(const Op& o, int p, P& q) { zv_step_load_p(o.step, p, q); }
  static __device__ __forceinline__ void prefetch(const Op& o, int qp, int qu) { zv_step_prefetch(o.step, qp, qu); }
  static constexpr bool float_acc = sizeof(R) == 4 && sizeof(TV) == 4;
  static __device__ __forceinline__ void emit(const Op& o, int p, int nv, const ZvNb<R, NP>& nb, const U&, const P& q,
                                              double& a0, double&) {
    R xn[NP];
    zv_step_emit(o.step, p, nv, nb, q, xn);
#pragma unroll
    for (int e = 0; e < NP; ++e)
      if (e < nv) a0 = fma(to_double(store_as<TV>(q.b[e])), to_double(store_as<TV>(xn[e])), a0);
  }
  static __device__ __forceinline__ void emit_f(const Op& o, int p, int nv, const ZvNb<R, NP>& nb, const U&,
                                                const P& q, float& s, float& c) {
    R xn[NP];
    zv_step_emit(o.step, p, nv, nb, q, xn);
#pragma unroll
    for (int e = 0; e < NP; ++e)
      if (e < nv) dot2_add((float)q.b[e], (float)store_as<TV>(xn[e]), s, c);
  }
};

// pre-smoothing from a zero guess: the operand x_1 = D^-1 b / theta is formed
// from b and D^-1 at every stencil point
template <class R_, class TV, class TC_> struct Zv<OpChebZero<R_, TV, TC_>> {
  using Op = OpChebZero<R_, TV, TC_>;
  using R = R_;
  static constexpr int NP = ZV_NP<R>;
  using TC = TC_;
  struct U {
    R b[NP], di[NP];
  };
  struct P {};
  static constexpr bool ok = true;
  static __device__ __forceinline__ const TC* kx(const Op& o) { return o.kx; }
  static __device__ __forceinline__ const TC* ky(const Op& o) { return o.ky; }
  static __device__ __forceinline__ const TC* kz(const Op& o) { return o.kz; }
  static __device__ __forceinline__ void load_u(const Op& o, int p, U& u) {
    ldn(o.b + p, u.b);
    ldn(o.dinv + p, u.di);
  }
  static __device__ __forceinline__ void vals(const Op& o, const U& u, R (&v)[NP]) {
#pragma unroll
    for (int e = 0; e < NP; ++e) v[e] = o.inv_theta * (u.di[e] * u.b[e]);
  }
  static __device__ __forceinline__ R u_one(const Op& o, int q) {
    return o.inv_theta * (cvt<R>(__ldg(o.dinv + q)) * cvt<R>(__ldg(o.b + q)));
  }
  static __device__ __forceinline__ void load_p(const Op&, int, P&) {}
  static __device__ __forceinline__ void prefetch(const Op& o, int, int qu) {
    pf_l2(o.b + qu);
    pf_l2(o.dinv + qu);
  }
  static __device__ __forceinline__ void emit(const Op& o, int p, int nv, const ZvNb<R, NP>& nb, const U& uc, const P&,
                                              double&, double&) {
    R xo[NP], d1[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      R D;
      const R S = nb.eval(e, D);
      const R x1 = nb.uc[e];
      const R s = fma(uc.di[e], uc.b[e] + S, -x1);
      d1[e] = fma(o.c1, x1, o.c2 * s);
      xo[e] = x1 + d1[e];
    }
    stn(o.xout + p, xo, nv);
    if (o.dout) stn(o.dout + p, d1, nv);
  }
};

// r = b - A x (acc0 += r.r)
template <class R_, class TV, class TB, class TC_> struct Zv<OpResidual<R_, TV, TB, TC_>> {
  using Op = OpResidual<R_, TV, TB, TC_>;
  using R = R_;
  static constexpr int NP = ZV_NP<R>;
  using TC = TC_;
  using UU = ZvVecU<R, TV>;
  using U = typename UU::U;
  struct P {
    R b[NP];
  };
  static constexpr bool ok = true;
  static __device__ __forceinline__ const TC* kx(const Op& o) { return o.kx; }
  static __device__ __forceinline__ const TC* ky(const Op& o) { return o.ky; }
  static __device__ __forceinline__ const TC* kz(const Op& o) { return o.kz; }
  static __device__ __forceinline__ void load_u(const Op& o, int p, U& u) { UU::load(o.x, p, u); }
  static __device__ __forceinline__ void vals(const Op&, const U& u, R (&v)[NP]) { UU::vals(u, v); }
  static __device__ __forceinline__ R u_one(const Op& o, int q) { return UU::one(o.x, q); }
  static __device__ __forceinline__ void load_p(const Op& o, int p, P& q) { ldn(o.b + p, q.b); }
  static __device__ __forceinline__ void prefetch(const Op& o, int qp, int qu) {
    pf_l2(o.x + qu);
    pf_l2(o.b + qp);
  }
  static __device__ __forceinline__ void emit(const Op& o, int p, int nv, const ZvNb<R, NP>& nb, const U&, const P& q,
                                              double& acc, double&) {
    R rv[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      R D;
      const R S = nb.eval(e, D);
      rv[e] = (q.b[e] + S) - D * nb.uc[e];
    }
    stn(o.r + p, rv, nv);
#pragma unroll
    for (int e = 0; e < NP; ++e)
      if (e < nv) acc = fma((double)rv[e], (double)rv[e], acc);
  }
};

// float64 r = b - A x with the stored diagonal
template <class TB> struct Zv<OpResidualD<TB>> {
  using Op = OpResidualD<TB>;
  using R = double;
  static constexpr int NP = ZV_NP<R>;
  using TC = double;
  using UU = ZvVecU<double, double>;
  using U = typename UU::U;
  struct P {
    double b[NP], dg[NP];
  };
  static constexpr bool ok = true;
  static __device__ __forceinline__ const TC* kx(const Op& o) { return o.kx; }
  static __device__ __forceinline__ const TC* ky(const Op& o) { return o.ky; }
  static __device__ __forceinline__ const TC* kz(const Op& o) { return o.kz; }
  static __device__ __forceinline__ void load_u(const Op& o, int p, U& u) { UU::load(o.x, p, u); }
  static __device__ __forceinline__ void vals(const Op&, const U& u, double (&v)[NP]) { UU::vals(u, v); }
  static __device__ __forceinline__ double u_one(const Op& o, int q) { return UU::one(o.x, q); }
  static __device__ __forceinline__ void load_p(const Op& o, int p, P& q) {
    ldn(o.b + p, q.b);
    ldn(o.dg + p, q.dg);
  }
  static __device__ __forceinline__ void prefetch(const Op& o, int qp, int qu) {
    pf_l2(o.x + qu);
    pf_l2(o.b + qp);
    pf_l2(o.dg + qp);
  }
  static __device__ __forceinline__ void emit(const Op& o, int p, int nv, const ZvNb<double, NP>& nb, const U&, const P& q,
                                              double& acc, double&) {
    double rv[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      double D;
      const double S = nb.eval(e, D);
      rv[e] = (q.b[e] + S) - q.dg[e] * nb.uc[e];
    }
    stn(o.r + p, rv, nv);
#pragma unroll
    for (int e = 0; e < NP; ++e)
      if (e < nv) acc = fma(rv[e], rv[e], acc);
  }
};

// (The float64 passes run here only where the integer-pipe driver, k_zsoft, does not apply.)

// Resident blocks per SM requested from the compiler (96 registers per thread):
// zero-guess step, step and residual at 257^3 with 4, 5 and 6 blocks 81 / 84 / 68,
// 77 / 82 / 65 and 104 / 94 / 72 us.
constexpr int ZV_BLOCKS = 5;
// Blocks per SM that the plane chunks are cut for, and least planes per chunk on
// large levels, by points per thread.  Two (float64) is bound by the float64 pipe
// and wants even shares more than few planes read twice: 2 x 5 and 4 instead of 5
// and 8 take 159 instead of 168 us a step at 193^3, 52.6 instead of 55.9 at 129^3, the
// same at 257^3 and 321^3.
constexpr int zv_share(int np) { return np == 2 ? 2 * ZV_BLOCKS : ZV_BLOCKS; }
constexpr int zv_chunk(int np) { return np == 2 ? 4 : 8; }

// The driver: 2^lw lanes per row (whole rows in a warp, so that every shuffle
// stays inside a row), ZV_THREADS / 2^lw rows per block.  Lanes past the row
// read its last vector and store nothing.
template <class Op, bool RED>
__global__ void __launch_bounds__(ZV_THREADS, ZV_BLOCKS)
    k_zvec(Op op, Geom g, int lw, int kchunk, double* partials, int stride) {
  using Z = Zv<Op>;
  using R = typename Z::R;
  using TC = typename Z::TC;
  using U = typename Z::U;
  using P = typename Z::P;
  constexpr int NP = Z::NP;
  pdl_wait();
  op.prepare();
  const int W = 1 << lw, l = threadIdx.x & (W - 1);
  const int i0 = ((blockIdx.x << lw) + l) * NP, j0 = blockIdx.y * (ZV_THREADS >> lw) + (threadIdx.x >> lw);
  const int nv = j0 < g.ny ? min(max(g.nx - i0, 0), NP) : 0;
  const bool first = l == 0, last = l == W - 1;
  const int k0 = blockIdx.z * kchunk;
  const int k1 = min(k0 + kchunk, g.nz);
  double a0 = 0.0, a1 = 0.0;
  float f0 = 0.0f, f1 = 0.0f;  // float-float accumulator (ZvFloatAcc ops)
  {
    const int sz = (int)g.sz, sy = g.Px;
    int p = (int)g.at(min(i0, g.Px - NP), min(j0, g.ny - 1), k0);
    const TC* kx = Z::kx(op);
    const TC* ky = Z::ky(op);
    const TC* kz = Z::kz(op);
    U qm, qc, qp;
    Z::load_u(op, p - sz, qm);
    Z::load_u(op, p, qc);
    Z::load_u(op, p + sz, qp);
    R czm[NP], nkx[NP], nky[NP], nkz[NP];
    ldn(kz + p - sz, czm);
    ldn(kx + p, nkx);
    ldn(ky + p, nky);
    ldn(kz + p, nkz);
    P pn;
    Z::load_p(op, p, pn);
    for (int k = k0; k < k1; ++k, p += sz) {
      ZvNb<R, NP> nb;
      const P pc = pn;
#pragma unroll
      for (int e = 0; e < NP; ++e) {
        nb.cx[e] = nkx[e];
        nb.cy[e] = nky[e];
        nb.cz[e] = nkz[e];
        nb.czm[e] = czm[e];
      }
      U qn = qp;
      if (k + 1 < k1) {  // next plane: operand two planes up, pointwise values one plane up
        Z::load_u(op, p + 2 * sz, qn);
        Z::load_p(op, p + sz, pn);
        ldn(kx + p + sz, nkx);
        ldn(ky + p + sz, nky);
        ldn(kz + p + sz, nkz);
      }
      if (k + ZV_PF < k1) {
        const int q = p + ZV_PF * sz;
        pf_l2(kx + q);
        pf_l2(ky + q);
        pf_l2(kz + q);
        Z::prefetch(op, q, q + sz);
      }
      U ys, yn;
      Z::load_u(op, p - sy, ys);
      Z::load_u(op, p + sy, yn);
      ldn(ky + p - sy, nb.cys);
      Z::vals(op, qc, nb.uc);
      Z::vals(op, qm, nb.um);
      Z::vals(op, qp, nb.up);
      Z::vals(op, ys, nb.us);
      Z::vals(op, yn, nb.un);
      nb.uw = __shfl_up_sync(0xffffffffu, nb.uc[NP - 1], 1);
      nb.ue = __shfl_down_sync(0xffffffffu, nb.uc[0], 1);
      nb.cxw = __shfl_up_sync(0xffffffffu, nb.cx[NP - 1], 1);
      if (first) {
        nb.uw = Z::u_one(op, p - 1);
        nb.cxw = cvt<R>(__ldg(kx + p - 1));
      }
      if (last) nb.ue = Z::u_one(op, p + NP);
      if (nv > 0) {
        if constexpr (ZvFloatAcc<Z>::value) Z::emit_f(op, p, nv, nb, qc, pc, f0, f1);
        else Z::emit(op, p, nv, nb, qc, pc, a0, a1);
      }
      qm = qc;
      qc = qp;
      qp = qn;
#pragma unroll
      for (int e = 0; e < NP; ++e) czm[e] = nb.cz[e];
    }
  }
  pdl_trigger();
  if constexpr (RED) {
    if constexpr (ZvFloatAcc<Z>::value) a0 = (double)f0 + (double)f1;  // exact widening, once per thread
    block_sum2<ZV_THREADS>(a0, a1);
    if (threadIdx.x == 0) {
      const int b = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
      partials[b] = a0;
      partials[stride + b] = a1;
    }
  }
}

// ------------------------------------------------------------ transfers
// x += P e on the fine grid (OpProlong) without z-marching: each thread
// updates a block of four consecutive x points, two rows and two planes, fine
// (4m .. 4m+3, 2r, 2r+1, 2s, 2s+1), which draw on coarse columns 2m-1 .. 2m+1,
// rows r-1, r and planes s-1, s: twelve coarse values for sixteen points.
// Along an odd fine index both of OpProlong's two terms are the same coarse
// value, so its sum doubles exactly: the sums are formed once per coarse
// column without the doublings and the power of two goes into the factor
// 1/8, which gives OpProlong's result bit for bit.
//
// What bounds it: x read and written and e/8 of memory traffic; in float64,
// 2.25 operations per point (4.25 when each fine row formed its own sums) on
// the float64 pipe.
constexpr int PV_THREADS = 256;
// cw = 2^lw chunks of four points in x per block, 256 / cw row pairs
template <class R, class TV>
__global__ void __launch_bounds__(PV_THREADS) k_prolong_v(OpProlong<R, TV> op, Geom g, int lw) {
  pdl_wait();
  const int m = (blockIdx.x << lw) + (threadIdx.x & ((1 << lw) - 1));
  const int r = blockIdx.y * (PV_THREADS >> lw) + (threadIdx.x >> lw);
  const int s = blockIdx.z;
  const int i = 4 * m;
  if (2 * r < g.ny && i < g.nx) {
    const Geom& gc = op.gc;
    R E[2][2][3];  // [plane s-1 / s][row r-1 / r][column 2m-1 .. 2m+1]
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const i64 q = gc.at(2 * m - 1, r - 1 + c, s - 1 + a);
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) E[a][c][cc] = cvt<R>(__ldg(op.e + q + cc));
      }
    const int nv = min(g.nx - i, 4);
    R xv[2][2][4];
#pragma unroll
    for (int kk = 0; kk < 2; ++kk)
#pragma unroll
      for (int jj = 0; jj < 2; ++jj) {
        if (2 * s + kk >= g.nz || 2 * r + jj >= g.ny) continue;
        const TV* x = op.x + g.at(i, 2 * r + jj, 2 * s + kk);
        R(&v)[4] = xv[kk][jj];
        if constexpr (sizeof(TV) == 4) {
          const float4 t = *reinterpret_cast<const float4*>(x);
          v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
        } else {
          const double2 t0 = *reinterpret_cast<const double2*>(x);
          const double2 t1 = *reinterpret_cast<const double2*>(x + 2);
          v[0] = t0.x, v[1] = t0.y, v[2] = t1.x, v[3] = t1.y;
        }
      }
    R F[2][3], Y[2][2][3];  // F: the two planes' sum of a row; Y[kk][jj]: column sums without doublings
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) {
      F[0][cc] = E[0][0][cc] + E[1][0][cc];
      F[1][cc] = E[0][1][cc] + E[1][1][cc];
      Y[0][0][cc] = F[0][cc] + F[1][cc];
      Y[0][1][cc] = F[1][cc];
      Y[1][0][cc] = E[1][0][cc] + E[1][1][cc];
      Y[1][1][cc] = E[1][1][cc];
    }
#pragma unroll
    for (int kk = 0; kk < 2; ++kk)
#pragma unroll
      for (int jj = 0; jj < 2; ++jj) {
        if (2 * s + kk >= g.nz || 2 * r + jj >= g.ny) continue;
        const R w = (R)(0.125 * (1 << (kk + jj)));
        TV* x = op.x + g.at(i, 2 * r + jj, 2 * s + kk);
        const R(&y)[3] = Y[kk][jj];
        R(&v)[4] = xv[kk][jj];
        v[0] = fma(w, y[0] + y[1], v[0]);
        v[1] = fma((R)2 * w, y[1], v[1]);
        v[2] = fma(w, y[1] + y[2], v[2]);
        v[3] = fma((R)2 * w, y[2], v[3]);
        if (nv == 4) {
          if constexpr (sizeof(TV) == 4) {
            *reinterpret_cast<float4*>(x) = make_float4(v[0], v[1], v[2], v[3]);
          } else {
            reinterpret_cast<double2*>(x)[0] = make_double2(v[0], v[1]);
            reinterpret_cast<double2*>(x)[1] = make_double2(v[2], v[3]);
          }
        } else {
#pragma unroll
          for (int e = 0; e < 3; ++e)
            if (e < nv) x[e] = store_as<TV>(v[e]);
        }
      }
  }
  pdl_trigger();
}

// bc = R r on the coarse grid (OpRestrict), two coarse points (c, c+1) per
// thread: the five fine values 2c .. 2c+4 of a fine row come from one
// 16-byte load and the right lane's first value.  Per fine plane the three
// fine rows give the plane sum; consecutive coarse planes share a fine plane,
// whose sum is kept.  Same terms in the same order as OpRestrict; a row is
// summed with weights (1/2, 1, 1/2), one operation less than with (1/4, 1/2,
// 1/4), and the factor 1/2 that is left goes into the planes' weights.  Powers
// of two: the result is the same wherever nothing is subnormal, and like
// OpRestrict's the sums are finite for operands up to half the largest number.
// A coarse point takes 21 operations instead of 27, which is what bounds the
// float64 form (257^3: 127 -> 101 us; float32 21 us).  Weights (1, 2, 1) on every
// axis take 19 operations and 91 us, but their sums reach 64 times the operands.
template <class R, class TV>
__global__ void __launch_bounds__(ZV_THREADS, 8) k_restrict_v(OpRestrict<R, TV> op, Geom gc, int kchunk) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int c = blockIdx.x * ZV_TX + 2 * lane;
  const int cj = blockIdx.y * ZV_TY + (threadIdx.x >> 5);
  const int k0 = blockIdx.z * kchunk;
  const int k1 = min(k0 + kchunk, gc.nz);
  if (cj < gc.ny) {
    const Geom& gf = op.gf;
    const int nv = min(max(gc.nx - c, 0), 2);
    const int fb = min(2 * c, gf.Px - 4);  // fine x of the first of the five values (a multiple of 4)
    // plane sum of fine plane kf for the two coarse points
    auto plane = [&](int kf, R (&P)[2]) {
      R row[3][2];
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const int q = (int)gf.at(fb, 2 * cj + b, kf);
        R v[5];
        if constexpr (sizeof(TV) == 4) {
          const float4 t = __ldg(reinterpret_cast<const float4*>(op.r + q));
          v[0] = cvt<R>(t.x), v[1] = cvt<R>(t.y), v[2] = cvt<R>(t.z), v[3] = cvt<R>(t.w);
        } else {
          const double2 t0 = __ldg(reinterpret_cast<const double2*>(op.r + q));
          const double2 t1 = __ldg(reinterpret_cast<const double2*>(op.r + q + 2));
          v[0] = cvt<R>(t0.x), v[1] = cvt<R>(t0.y), v[2] = cvt<R>(t1.x), v[3] = cvt<R>(t1.y);
        }
        v[4] = __shfl_down_sync(0xffffffffu, v[0], 1);
        if (lane == 31) v[4] = cvt<R>(__ldg(op.r + q + 4));
#pragma unroll
        for (int e = 0; e < 2; ++e)
          row[b][e] = fma((R)0.5, v[2 * e] + v[2 * e + 2], v[2 * e + 1]);  // twice the weighted row
      }
#pragma unroll
      for (int e = 0; e < 2; ++e)
        P[e] = fma((R)0.25, row[2][e], fma((R)0.5, row[1][e], (R)0.25 * row[0][e]));
    };
    R Plo[2], Pmid[2], Phi[2];
    plane(2 * k0, Plo);
    for (int k = k0; k < k1; ++k) {
      if (k + 1 < k1) {  // the fine rows of the next coarse plane into L2
#pragma unroll
        for (int b = 0; b < 3; ++b) {
          pf_l2(op.r + gf.at(fb, 2 * cj + b, 2 * k + 3));
          pf_l2(op.r + gf.at(fb, 2 * cj + b, 2 * k + 4));
        }
      }
      plane(2 * k + 1, Pmid);
      plane(2 * k + 2, Phi);
      R acc[2];
#pragma unroll
      for (int e = 0; e < 2; ++e)
        acc[e] = fma((R)0.125, Phi[e], fma((R)0.25, Pmid[e], (R)0.125 * Plo[e]));
      if (nv > 0) st2(op.bc + gc.at(min(c, gc.Px - 2), cj, k), acc, nv);
#pragma unroll
      for (int e = 0; e < 2; ++e) Plo[e] = Phi[e];
    }
  }
  pdl_trigger();
}

template <class Op> struct ZvXfer {
  static constexpr bool ok = false;
};
template <class R, class TV> struct ZvXfer<OpProlong<R, TV>> {
  static constexpr bool ok = true;
};
template <class R, class TV> struct ZvXfer<OpRestrict<R, TV>> {
  static constexpr bool ok = true;
};

}  // namespace mgdev
