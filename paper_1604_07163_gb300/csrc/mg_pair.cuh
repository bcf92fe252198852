// Two successive float32 stencil passes over a re-discretised level in one
// sweep.
//
// A smoothing step, or the step from a zero guess, followed by another step or
// by the residual reads the level's coefficients and right-hand side twice and
// moves the iterate between them through memory.  Here a block sweeps a chunk
// of planes of a (4 * 2^lx) x (PR_THREADS / 2^lx) tile: the first pass is formed
// on the whole tile, its plane goes to the neighbours through shared memory,
// and the second pass follows one plane behind on the tile's interior.  The
// coefficients, the right-hand side and 1 / D are read once, the direction never
// leaves the SM and the iterate between the passes only where the residual form
// stores it: 28 bytes per point (a step and the residual 32) instead of 48 to
// 56.  The price is the first pass on the tile's rim
// (one row on either side, one plane on either side of a chunk, and four points
// on either side where a row is wider than the tile).
//
// Every point's arithmetic is that of the single passes (mg_zvec.cuh), term for
// term and in the same order: results are theirs bit for bit.  (The __f*_rn
// intrinsics keep the compiler from contracting what it leaves apart there.)
//
// What bounds it: latency at 16 warps per SM (issuing on 43 to 58% of the cycles,
// DRAM at 52 to 65%).  257^3, the two single passes and the sweep: zero-guess step
// + residual 142 -> 100 us, two steps 164 -> 119 us with b.z and 138 -> 104 us
// (Richardson) without; 513^3: 914 -> 710 us, 1066 -> 1005 us.  Reading the stored
// 1 / D for the steps instead of dividing: 124 -> 119 us (the same value).  640 and 768 threads
// per block, at 96 and 80 registers: 161 and 205 us.
#pragma once
#include "mg_zvec.cuh"

namespace mgdev {

constexpr int PR_THREADS = 512;
constexpr int PR_NP = 4;

enum { PR_ZERO = 0, PR_STEP = 1, PR_RESID = 2 };

// First pass A: PR_STEP, x' = x + d, d = D^-1 (b - A x) / theta; PR_ZERO, the two
// steps from a zero guess (OpChebZero).  Second pass B: PR_STEP, x'' = x' + d',
// d' = c1 d + c2 s (dprev) or s / theta; PR_RESID, r = b - A x', x' stored too.
template <class TC> struct PairArgs {
  const float *x, *b, *dinv;
  float *xout, *r;
  const TC *kx, *ky, *kz;
  float c1, c2, inv_theta;
  int dprev;
};

template <class TC, int A, int B, bool DOT>
__global__ void __launch_bounds__(PR_THREADS, 1)
    k_pair(PairArgs<TC> o, Geom g, int lx, int halo, int kchunk, double* partials, int stride) {
  constexpr int NP = PR_NP;
  extern __shared__ float pr_sm[];
  pdl_wait();
  const int LX = 1 << lx, LY = PR_THREADS >> lx, row = NP * LX + 8;
  const int l = threadIdx.x & (LX - 1), t = threadIdx.x >> lx;
  const int i0 = NP * (blockIdx.x * (LX - 2 * halo) + l - halo), j = blockIdx.y * (LY - 2) + t - 1;
  const int k0 = blockIdx.z * kchunk, k1 = min(k0 + kchunk, g.nz);
  const bool in_row = j >= 0 && j < g.ny;
  const int na = in_row && i0 >= 0 ? min(max(g.nx - i0, 0), NP) : 0;  // points of the first pass
  const bool inner = t > 0 && t < LY - 1 && (!halo || (l > 0 && l < LX - 1));
  const int nb = inner ? na : 0;  // points of the second
  const int w = min(LX, 32) - 1;
  // lanes whose left (right) neighbour is not the previous (next) lane
  const bool first = (threadIdx.x & w) == 0 || i0 == 0, last = (threadIdx.x & w) == w;
  const int sz = (int)g.sz, sy = g.Px;
  const int ks = max(k0 - 1, 0), ke = min(k1, g.nz - 1);  // planes of the first pass
  int p = (int)g.at(min(max(i0, 0), g.Px - NP), min(max(j, 0), g.ny - 1), ks);
  float* s0 = pr_sm + t * row + 4 + NP * l;
  const int plane = LY * row;
  for (int q = threadIdx.x; q < 2 * LY; q += PR_THREADS) {  // columns beyond the tile: the boundary
    pr_sm[q * row + 3] = 0.0f;
    pr_sm[q * row + 4 + NP * LX] = 0.0f;
  }
  const TC *kx = o.kx, *ky = o.ky, *kz = o.kz;

  // operand planes: b and D^-1 (PR_ZERO) or x
  struct U {
    float v[A == PR_ZERO ? 2 : 1][NP];
  };
  auto load_u = [&](int q, U& u) {
    if constexpr (A == PR_ZERO) {
      ldn(o.b + q, u.v[0]);
      ldn(o.dinv + q, u.v[1]);
    } else {
      ldn(o.x + q, u.v[0]);
    }
  };
  auto vals = [&](const U& u, float (&v)[NP]) {
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      if constexpr (A == PR_ZERO) v[e] = o.inv_theta * (u.v[1][e] * u.v[0][e]);
      else v[e] = u.v[0][e];
    }
  };
  auto one = [&](int q) {
    if constexpr (A == PR_ZERO) return o.inv_theta * (__ldg(o.dinv + q) * __ldg(o.b + q));
    else return __ldg(o.x + q);
  };

  float um[NP], czm[NP], nkx[NP], nky[NP], nkz[NP], nbv[NP], ndi[NP];
  U uc, up;
  {
    U t0;
    load_u(p - sz, t0);
    vals(t0, um);
  }
  load_u(p, uc);
  load_u(p + sz, up);
  ldn(kz + p - sz, czm);
  ldn(kx + p, nkx);
  ldn(ky + p, nky);
  ldn(kz + p, nkz);
  if constexpr (A != PR_ZERO) {
    ldn(o.b + p, nbv);
    ldn(o.dinv + p, ndi);
  }
  // the second pass's plane k - 1: iterate, sum without the upper neighbour, b, D^-1 or D, direction
  float y[NP], S5[NP], bp[NP], fp[NP], dp[NP];
#pragma unroll
  for (int e = 0; e < NP; ++e) y[e] = S5[e] = bp[e] = fp[e] = dp[e] = 0.0f;
  float f0 = 0.0f, f1 = 0.0f;

  // second pass on plane k - 1 at q, with the upper neighbours yn and their coefficients c
  auto emit = [&](int q, const float (&c)[NP], const float (&yn)[NP]) {
    float out[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      const float S = fmaf(c[e], yn[e], S5[e]);
      if constexpr (B == PR_RESID) {
        out[e] = (bp[e] + S) - fp[e] * y[e];
      } else {
        const float s = fmaf(fp[e], bp[e] + S, -y[e]);
        out[e] = __fadd_rn(y[e], o.dprev ? fmaf(o.c1, dp[e], o.c2 * s) : __fmul_rn(s, o.inv_theta));
        if constexpr (DOT) {
          if (e < nb) dot2_add(bp[e], out[e], f0, f1);
        }
      }
    }
    if constexpr (B == PR_RESID) {
      stn(o.r + q, out, nb);
      stn(o.xout + q, y, nb);
    } else {
      stn(o.xout + q, out, nb);
    }
  };

  for (int k = ks; k <= ke; ++k, p += sz) {
    // ---- first pass, plane k
    float cx[NP], cy[NP], cz[NP], cys[NP], b[NP], inv[NP], v[NP], us[NP], un[NP], vp[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      cx[e] = nkx[e];
      cy[e] = nky[e];
      cz[e] = nkz[e];
      b[e] = A == PR_ZERO ? uc.v[0][e] : nbv[e];
      if constexpr (A == PR_ZERO) inv[e] = uc.v[1][e];
      else inv[e] = ndi[e];
    }
    U un2 = up;
    if (k < ke) {
      load_u(p + 2 * sz, un2);
      ldn(kx + p + sz, nkx);
      ldn(ky + p + sz, nky);
      ldn(kz + p + sz, nkz);
      if constexpr (A != PR_ZERO) {
        ldn(o.b + p + sz, nbv);
        ldn(o.dinv + p + sz, ndi);
      }
    }
    if (k + ZV_PF <= ke) {
      const int q = p + ZV_PF * sz;
      pf_l2(kx + q);
      pf_l2(ky + q);
      pf_l2(kz + q);
      if constexpr (A == PR_ZERO) {
        pf_l2(o.b + q + sz);
        pf_l2(o.dinv + q + sz);
      } else {
        pf_l2(o.b + q);
        pf_l2(o.dinv + q);
        pf_l2(o.x + q + sz);
      }
    }
    {
      U ys, yn;
      load_u(p - sy, ys);
      load_u(p + sy, yn);
      vals(ys, us);
      vals(yn, un);
    }
    ldn(ky + p - sy, cys);
    vals(uc, v);
    vals(up, vp);
    float uw = __shfl_up_sync(0xffffffffu, v[NP - 1], 1), ue = __shfl_down_sync(0xffffffffu, v[0], 1);
    float cxw = __shfl_up_sync(0xffffffffu, cx[NP - 1], 1);
    if (first) {
      uw = one(p - 1);
      cxw = cvt<float>(__ldg(kx + p - 1));
    }
    if (last) ue = one(p + NP);
    float yn[NP], f[NP], d[NP];
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      const float cxm = e == 0 ? cxw : cx[e > 0 ? e - 1 : 0];
      float S = cxm * (e == 0 ? uw : v[e > 0 ? e - 1 : 0]);
      S = fmaf(cx[e], e == NP - 1 ? ue : v[e < NP - 1 ? e + 1 : e], S);
      S = fmaf(cys[e], us[e], S);
      S = fmaf(cy[e], un[e], S);
      S = fmaf(czm[e], um[e], S);
      S = fmaf(cz[e], vp[e], S);
      const float s = fmaf(inv[e], b[e] + S, -v[e]);
      float x1;
      if constexpr (A == PR_ZERO) {
        x1 = __fadd_rn(v[e], fmaf(o.c1, v[e], o.c2 * s));
      } else {
        d[e] = __fmul_rn(s, o.inv_theta);
        x1 = __fadd_rn(v[e], d[e]);
      }
      yn[e] = e < na ? x1 : 0.0f;
      f[e] = B == PR_RESID ? ((cxm + cx[e]) + (cys[e] + cy[e])) + (czm[e] + cz[e]) : inv[e];
    }
    // ---- second pass, plane k - 1
    if (k > k0 && nb > 0) emit(p - sz, czm, yn);
    // ---- this plane to the neighbours, and its sum but for the upper one
    float* s = s0 + (k & 1) * plane;
    *reinterpret_cast<float4*>(s) = make_float4(yn[0], yn[1], yn[2], yn[3]);
    __syncthreads();
    float yw = __shfl_up_sync(0xffffffffu, yn[NP - 1], 1), ye = __shfl_down_sync(0xffffffffu, yn[0], 1);
    if (first) yw = s[-1];
    if (last) ye = s[NP];
    if (nb > 0) {
      const float4 a4 = *reinterpret_cast<const float4*>(s - row), c4 = *reinterpret_cast<const float4*>(s + row);
      const float ys[NP] = {a4.x, a4.y, a4.z, a4.w}, yu[NP] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
      for (int e = 0; e < NP; ++e) {
        float S = (e == 0 ? cxw : cx[e > 0 ? e - 1 : 0]) * (e == 0 ? yw : yn[e > 0 ? e - 1 : 0]);
        S = fmaf(cx[e], e == NP - 1 ? ye : yn[e < NP - 1 ? e + 1 : e], S);
        S = fmaf(cys[e], ys[e], S);
        S = fmaf(cy[e], yu[e], S);
        S5[e] = fmaf(czm[e], y[e], S);
      }
    }
#pragma unroll
    for (int e = 0; e < NP; ++e) {
      y[e] = yn[e];
      bp[e] = b[e];
      fp[e] = f[e];
      if constexpr (A != PR_ZERO) dp[e] = d[e];
      um[e] = v[e];
      czm[e] = cz[e];
    }
    uc = up;
    up = un2;
  }
  if (k1 == g.nz && nb > 0) {  // the last plane: its upper neighbours are the boundary
    const float z[NP] = {0.0f, 0.0f, 0.0f, 0.0f};
    emit(p - sz, czm, z);
  }
  pdl_trigger();
  if constexpr (DOT) {
    double a0 = (double)f0 + (double)f1, a1 = 0.0;
    block_sum2<PR_THREADS>(a0, a1);
    if (threadIdx.x == 0) {
      const int q = (blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
      partials[q] = a0;
      partials[stride + q] = a1;
    }
  }
}

}  // namespace mgdev
