// Vector driver of the 27-point (Galerkin) passes: NP consecutive x points per
// thread.
//
// A point needs 26 couplings and 26 operand values.  One at a time through L1
// that is 57 four-byte loads per point and pass, and the scalar driver was
// bound by their latency at about half of the memory rate.  Here each array row
// is read with one vector load for the thread's NP points; the values one point
// to the left or right of them come from the neighbouring lane by a shuffle
// (from memory at the ends of a row's lanes).  The terms of a point are added
// in stencil27's order, so the results are the scalar driver's bit for bit.
//
// What bounds it: memory latency, with 68 to 72 bytes per point.  255^3 points
// in float32, scalar driver and this one: smoothing step 250 -> 209 us (176 us of
// traffic), zero-guess step 275 -> 187 us, residual 235 -> 200 us; 127^3: 38.8 ->
// 36.7, 43.5 -> 35.7, 36.8 -> 37.4 us.
#pragma once
#include "mg_g27.cuh"
#include "mg_zvec.cuh"

namespace mgdev {


// Per-operation hooks: w and its stride, the operand u, the point operation.
template <class Op> struct G27 {
  static constexpr bool ok = false;
};

template <class R_, class TV, class TC_> struct G27<OpChebStep27<R_, TV, TC_>> {
  using Op = OpChebStep27<R_, TV, TC_>;
  using R = R_;
  using TC = TC_;
  static constexpr bool ok = true;
  template <int NP> static __device__ __forceinline__ void load_u(const Op& o, int p, R (&v)[NP]) { ldn(o.x + p, v); }
  static __device__ __forceinline__ R u_one(const Op& o, int q) { return cvt<R>(__ldg(o.x + q)); }
  static __device__ __forceinline__ void prefetch(const Op& o, int qp, int qu) {
    pf_l2(o.x + qu);
    pf_l2(o.b + qp);
    pf_l2(o.dinv + qp);
    if (o.dprev) pf_l2(o.dprev + qp);
  }
  template <int NP>
  static __device__ __forceinline__ void emit(const Op& o, int p, int nv, const R (&S)[NP], const R (&uc)[NP]) {
    R b[NP], di[NP], d[NP], dn[NP], xn[NP];
    ldn(o.b + p, b);
    ldn(o.dinv + p, di);
    if (o.dprev) ldn(o.dprev + p, d);
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      const R s = fma(di[e], b[e] + S[e], -uc[e]);
      dn[e] = o.dprev ? fma(o.c1, d[e], o.c2 * s) : s * o.inv_theta;
      xn[e] = uc[e] + dn[e];
    }
    stn(o.xout + p, xn, nv);
    if (o.dout) stn(o.dout + p, dn, nv);
  }
};

template <class R_, class TV, class TC_> struct G27<OpChebZero27<R_, TV, TC_>> {
  using Op = OpChebZero27<R_, TV, TC_>;
  using R = R_;
  using TC = TC_;
  static constexpr bool ok = true;
  template <int NP> static __device__ __forceinline__ void load_u(const Op& o, int p, R (&v)[NP]) {
    R b[NP], di[NP];
    ldn(o.b + p, b);
    ldn(o.dinv + p, di);
#pragma unroll
    for (int e = 0; e < NP; ++e) v[e] = o.inv_theta * (di[e] * b[e]);
  }
  static __device__ __forceinline__ R u_one(const Op& o, int q) {
    return o.inv_theta * (cvt<R>(__ldg(o.dinv + q)) * cvt<R>(__ldg(o.b + q)));
  }
  static __device__ __forceinline__ void prefetch(const Op& o, int, int qu) {
    pf_l2(o.b + qu);
    pf_l2(o.dinv + qu);
  }
  template <int NP>
  static __device__ __forceinline__ void emit(const Op& o, int p, int nv, const R (&S)[NP], const R (&uc)[NP]) {
    R b[NP], di[NP], d1[NP], xn[NP];
    ldn(o.b + p, b);
    ldn(o.dinv + p, di);
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      const R s = fma(di[e], b[e] + S[e], -uc[e]);
      d1[e] = fma(o.c1, uc[e], o.c2 * s);
      xn[e] = uc[e] + d1[e];
    }
    stn(o.xout + p, xn, nv);
    if (o.dout) stn(o.dout + p, d1, nv);
  }
};

template <class R_, class TV, class TB, class TC_> struct G27<OpResidual27<R_, TV, TB, TC_>> {
  using Op = OpResidual27<R_, TV, TB, TC_>;
  using R = R_;
  using TC = TC_;
  static constexpr bool ok = true;
  template <int NP> static __device__ __forceinline__ void load_u(const Op& o, int p, R (&v)[NP]) { ldn(o.x + p, v); }
  static __device__ __forceinline__ R u_one(const Op& o, int q) { return cvt<R>(__ldg(o.x + q)); }
  static __device__ __forceinline__ void prefetch(const Op& o, int qp, int qu) {
    pf_l2(o.x + qu);
    pf_l2(o.b + qp);
    pf_l2(o.dg + qp);
  }
  template <int NP>
  static __device__ __forceinline__ void emit(const Op& o, int p, int nv, const R (&S)[NP], const R (&uc)[NP]) {
    R b[NP], dg[NP], r[NP];
    ldn(o.b + p, b);
    ldn(o.dg + p, dg);
#pragma unroll
    for (int e = 0; e < NP; ++e) r[e] = (b[e] + S[e]) - dg[e] * uc[e];
    stn(o.r + p, r, nv);
  }
};

// 2^lw lanes per row of the level (whole rows in a warp, so that every shuffle
// stays inside a row), ZV_THREADS / 2^lw rows per block.  Lanes past the row
// read its last vector and store nothing; a point's right neighbour beyond its
// own vector is never in such a lane.
// points per thread: 16-byte vectors
template <class R> constexpr int GV_NP = sizeof(R) == 8 ? 2 : 4;
// Resident blocks per SM, and whether the next plane's rows are prefetched into
// L2 (BIG, levels larger than L2).  Step, residual and zero-guess step at 255^3:
// 4 blocks without and with prefetch 237 / 249 / 216 and 240 / 217 / 213 us, 3
// blocks 257 / 238 / 216 and 209 / 200 / 187 us; at 127^3 4 blocks without are
// the fastest (36.7 / 37.6 / 35.6 against 39.7 / 39.3 / 36.5 us).
template <bool BIG> constexpr int GV_BLOCKS = BIG ? 3 : 4;

template <class Op, int NP, bool BIG>
__global__ void __launch_bounds__(ZV_THREADS, GV_BLOCKS<BIG>)
    k_g27v(Op op, Geom g, int lw, int kchunk) {
  using Z = G27<Op>;
  using R = typename Z::R;
  using TC = typename Z::TC;
  pdl_wait();
  const int W = 1 << lw, l = threadIdx.x & (W - 1);
  const int i0 = ((blockIdx.x << lw) + l) * NP, j0 = blockIdx.y * (ZV_THREADS >> lw) + (threadIdx.x >> lw);
  const int i = min(i0, g.Px - NP), j = min(j0, g.ny - 1);
  const int nv = j0 < g.ny ? g.nx - i0 : 0;
  const int k0 = blockIdx.z * kchunk, k1 = min(k0 + kchunk, g.nz);
  const int sy = g.Px, sz = (int)g.sz;
  const bool first = l == 0, last = l == W - 1;
  int p = (int)g.at(i, j, k0);
  auto left = [&](R v, auto&& at) {
    R t = __shfl_up_sync(0xffffffffu, v, 1);
    if (first) t = at();
    return t;
  };
  auto right = [&](R v, auto&& at) {
    R t = __shfl_down_sync(0xffffffffu, v, 1);
    if (last) t = at();
    return t;
  };
  for (int k = k0; k < k1; ++k, p += sz) {
    if (BIG && k + 1 < k1) {
      const int q = p + sz;
#pragma unroll
      for (int o = 0; o < 13; ++o) pf_l2(op.w + (i64)o * op.wst + q);
      Z::prefetch(op, q, q + sz);
    }
    R S[NP], uc[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) S[e] = 0;
    // operand row at q with the points on either side
    auto row = [&](int q, R (&x)[NP + 2]) {
      R v[NP];
      Z::load_u(op, q, v);
#pragma unroll
      for (int e = 0; e < NP; ++e) x[e + 1] = v[e];
      x[0] = left(v[NP - 1], [&] { return Z::u_one(op, q - 1); });
      x[NP + 1] = right(v[0], [&] { return Z::u_one(op, q + NP); });
    };
    // the two terms of coupling o for operand rows f (at p + row offset ro) and b (at p - ro), x shift dx
    auto terms = [&](int o, int dx, int ro, const R (&f)[NP + 2], const R (&b)[NP + 2]) {
      const TC* w = op.w + (i64)o * op.wst;
      R wf[NP], wv[NP], wb[NP];
      ldn(w + p, wf);
      ldn(w + (p - ro), wv);  // the backward couplings sit dx to the left of these
      if (dx == 0) {
#pragma unroll
        for (int e = 0; e < NP; ++e) wb[e] = wv[e];
      } else if (dx > 0) {
#pragma unroll
        for (int e = 1; e < NP; ++e) wb[e] = wv[e - 1];
        wb[0] = left(wv[NP - 1], [&] { return cvt<R>(__ldg(w + (p - ro) - 1)); });
      } else {
#pragma unroll
        for (int e = 0; e < NP - 1; ++e) wb[e] = wv[e + 1];
        wb[NP - 1] = right(wv[0], [&] { return cvt<R>(__ldg(w + (p - ro) + NP)); });
      }
#pragma unroll
      for (int e = 0; e < NP; ++e) {
        S[e] = fma(wf[e], f[e + 1 + dx], S[e]);
        S[e] = fma(wb[e], b[e + 1 - dx], S[e]);
      }
    };
    {
      R c[NP + 2];
      row(p, c);
#pragma unroll
      for (int e = 0; e < NP; ++e) uc[e] = c[e + 1];
      terms(0, 1, 0, c, c);
    }
#pragma unroll
    for (int t = 0; t < 4; ++t) {  // row pairs (dy, dz) = (1, 0), (-1, 1), (0, 1), (1, 1)
      const int ro = t == 0 ? sy : sz + (t - 2) * sy;
      R f[NP + 2], b[NP + 2];
      row(p + ro, f);
      row(p - ro, b);
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) terms(1 + 3 * t + dx + 1, dx, ro, f, b);
    }
    if (nv > 0) Z::emit(op, p, nv, S, uc);
  }
  pdl_trigger();
}

}  // namespace mgdev
