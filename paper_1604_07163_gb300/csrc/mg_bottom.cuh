// The bottom of the hierarchy in shared memory: levels lb..L-1 of the V-cycle
// as one thread-block cluster (or one block), every level's vectors and
// operator resident in the blocks' shared memory for the whole kernel.
//
// What bounds the coarse end is latency: a pass over a 15^3 level moves 60 KB,
// but k_bottom (mg_kernels.cuh), whose passes go through global memory with a
// barrier between them, needs about 2 us for it in float32 on one block and
// 3.5 us in float64 on a cluster of 4, whose acquire at every barrier sends
// its loads to L2.  Here
//   - each block owns a run of planes of every level (plane K of a coarse
//     level belongs to the block of fine plane 2K + 1, so that restriction and
//     prolongation reach at most one plane beyond it);
//   - a block holds, per level, the two iterate buffers of its planes with one
//     halo plane on each side, and the coefficients, D, D^-1, b and d of its
//     points in the order its threads visit them (conflict-free);
//   - a value that a neighbour will read is stored into the neighbour's halo
//     as well (distributed shared memory), so that every load is local and
//     only a cluster barrier separates the passes;
//   - the operators do not change after setup, so they are loaded before
//     griddepcontrol.wait, while the previous kernel still runs.
// The arithmetic of every point is that of k_bottom's operations in
// mg_device.cuh and mg_g27.cuh, term for term, whatever the number of blocks.
//
// Measured for the levels 15^3, 7^3, 3^3 (one launch timed alone, launch
// included): float32 28 -> 21 us, float64 56 -> 33 us, 27-point bfloat16
// couplings 39 -> 23 us; the whole 33^3 float64 solve 1.5 -> 1.1 ms.  Eight
// blocks are the fastest throughout (float64 89 / 70 / 42 / 33 us for 1 (in
// k_bottom) / 2 / 4 / 8; float32 28 / 27 / 23 / 21).  A cluster barrier
// with remote stores before it takes 830 to 900 cycles, a pass of a 7^3 level
// 1200; holding the levels of a few hundred points whole in every block, with
// a block barrier instead, was no faster (float32) or slower (float64).
#pragma once
#include "mg_kernels.cuh"

namespace mgdev {

constexpr int BS_THREADS = 512;
constexpr int BS_MAXB = 8;      // largest cluster
constexpr int BS_PLANES = 512;  // planes of all levels together

template <class TV, class TC> struct BsLevel {
  Geom g;
  const TV *dinv, *dg;  // dg: 27-point levels
  const TC *kx, *ky, *kz;
  const TC* w;  // 27-point level: 13 coupling arrays of length g.len (else null)
  TV inv_theta, c1[BOT_MAXDEG], c2[BOT_MAXDEG];
  int z0[BS_MAXB + 1];  // first plane of each block
  // shared memory, in elements of TV: the iterate buffers' windows, and the
  // own-point arrays [coefficients (6 or 26), D^-1, D, b, d][cap]
  int ox[2], own, cap;
  int lx, ly;  // own points are numbered (k - z0) << (lx + ly) | j << lx | i
  int np0;     // the level's first entry in the table of halo readers
};

template <class TV, class TC> struct BsArgs {
  BsLevel<TV, TC> lv[BOT_MAX];
  int nlev, nu_pre, nu_post, degree;
  int xelems;           // elements of all iterate windows (zeroed at the start)
  const TV* b;          // right-hand side of the first level
  TV* out;              // its result
  const double* Ai;     // inverse of the coarsest operator
  const double* Ac;     // the operator itself (inexact solve), else null
  double coarse_rtol;
  int coarse_maxit, nc;
};

// Index of the first element of block s's window of level V: one plane below
// its first, less a row (the coarsest level is held whole by every block).
template <class V> __host__ __device__ __forceinline__ int bs_base(const V& v, int s, bool last) {
  return (int)v.g.off + ((last ? 0 : v.z0[s]) - 1) * (int)v.g.sz - v.g.Px - 8;
}

__device__ __forceinline__ unsigned bs_remote(unsigned addr, int rank) {
  unsigned r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void bs_store(unsigned addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void bs_store(unsigned addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

template <class TV, class TC, bool CL>
__global__ void __launch_bounds__(BS_THREADS, 1) k_bottom_s(const __grid_constant__ BsArgs<TV, TC> a) {
  using R = TV;
  using BS = BotSync<CL>;
  extern __shared__ __align__(16) unsigned char bs_dyn[];
  R* const sm = reinterpret_cast<R*>(bs_dyn);
  __shared__ unsigned char need[BS_PLANES];  // per plane of every level: the other blocks that read it
  __shared__ double y[MG_COARSE_MAX], Ais[32 * 32];
  const int tid = threadIdx.x, rank = (int)BS::rank(), nb = (int)BS::blocks(), L = a.nlev;
  const unsigned smb = (unsigned)__cvta_generic_to_shared(sm);
  auto sync = [] {
    __syncwarp();
    BS::sync();
  };
  // f(t, i, j, k, p) for every own point of level V (t: own number, p: padded index)
  auto own_for = [&](const BsLevel<TV, TC>& V, auto f) {
    const int z0 = V.z0[rank], n = (V.z0[rank + 1] - z0) << (V.lx + V.ly);
    const int nx = V.g.nx, ny = V.g.ny, Px = V.g.Px, Py = V.g.Py, off = (int)V.g.off, lx = V.lx, ly = V.ly;
    for (int t = tid; t < n; t += BS_THREADS) {
      const int i = t & ((1 << lx) - 1), j = (t >> lx) & ((1 << ly) - 1), k = z0 + (t >> (lx + ly));
      if (i < nx && j < ny) f(t, i, j, k, off + (k * Py + j) * Px + i);
    }
  };
  // stores v at point p (plane k) of buffer c of level l, here and in every block that reads that plane
  auto put = [&](int l, int c, int k, int p, R v) {
    const BsLevel<TV, TC>& V = a.lv[l];
    const bool last = l == L - 1;
    sm[V.ox[c] + p - bs_base(V, rank, last)] = v;
    if constexpr (CL) {
      for (unsigned m = need[V.np0 + k]; m; m &= m - 1) {
        const int s = __ffs(m) - 1;
        bs_store(bs_remote(smb + (unsigned)((V.ox[c] + p - bs_base(V, s, last)) * (int)sizeof(R)), s), v);
      }
    }
  };
  // start of a level's pre-smoothing at an own point whose b is known: x = d = D^-1 b / theta, or a zero guess
  auto start = [&](int l, int t, int k, int p, R b) {
    const BsLevel<TV, TC>& V = a.lv[l];
    const int nc = V.w ? 26 : 6;
    R* O = sm + V.own + t;
    O[(nc + 2) * V.cap] = b;
    R x1 = 0;
    if (a.nu_pre > 0) {
      x1 = V.inv_theta * (O[nc * V.cap] * b);
      O[(nc + 3) * V.cap] = x1;
    }
    put(l, 0, k, p, x1);
  };
  auto S_at = [&](const BsLevel<TV, TC>& V, const R* x, const R* O) {
    const int sy = V.g.Px, sz = (int)V.g.sz, cap = V.cap;
    R S;
    if (V.w) {
      S = 0;
#pragma unroll
      for (int o = 0; o < 13; ++o) {
        const int off = g27_off(V.g, o);
        S = fma(O[2 * o * cap], x[off], S);
        S = fma(O[(2 * o + 1) * cap], x[-off], S);
      }
    } else {
      S = O[0] * x[-1];
      S = fma(O[cap], x[1], S);
      S = fma(O[2 * cap], x[-sy], S);
      S = fma(O[3 * cap], x[sy], S);
      S = fma(O[4 * cap], x[-sz], S);
      S = fma(O[5 * cap], x[sz], S);
    }
    return S;
  };
  // Chebyshev steps j0 .. degree-1 from buffer cur; returns the buffer of the result
  auto steps = [&](int l, int cur, int j0) {
    const BsLevel<TV, TC>& V = a.lv[l];
    const int nc = V.w ? 26 : 6, base = bs_base(V, rank, false);
    for (int j = j0; j < a.degree; ++j, cur ^= 1) {
      const R* X = sm + V.ox[cur] - base;
      const R c1 = V.c1[j], c2 = V.c2[j], it = V.inv_theta;
      own_for(V, [&](int t, int, int, int k, int p) {
        R* O = sm + V.own + t;
        const R S = S_at(V, X + p, O);
        const R xp = X[p];
        const R s = fma(O[nc * V.cap], O[(nc + 2) * V.cap] + S, -xp);
        const R dn = j > 0 ? fma(c1, O[(nc + 3) * V.cap], c2 * s) : s * it;
        const R xn = xp + dn;
        put(l, cur ^ 1, k, p, xn);
        if (j + 1 < a.degree) O[(nc + 3) * V.cap] = dn;
      });
      sync();
    }
    return cur;
  };

  // ---- constants: zero windows, halo readers, operators of the own points
  for (int e = tid; e < a.xelems; e += BS_THREADS) sm[e] = 0;
  for (int l = 0; l < L; ++l) {
    const BsLevel<TV, TC>& V = a.lv[l];
    for (int k = tid; k < V.g.nz; k += BS_THREADS) {
      unsigned m = 0;
      for (int s = 0; s < nb; ++s)
        if (l == L - 1 || (k >= V.z0[s] - 1 && k <= V.z0[s + 1])) m |= 1u << s;
      need[V.np0 + k] = (unsigned char)(m & ~(1u << rank));
    }
    if (l == L - 1) break;
    const int nc = V.w ? 26 : 6, cap = V.cap;
    own_for(V, [&](int t, int, int, int, int p) {
      R* O = sm + V.own + t;
      const int sy = V.g.Px, sz = (int)V.g.sz;
      R D;
      if (V.w) {
#pragma unroll
        for (int o = 0; o < 13; ++o) {
          const int off = g27_off(V.g, o);
          const TC* wo = V.w + (i64)o * V.g.len + p;
          O[2 * o * cap] = cvt<R>(__ldg(wo));
          O[(2 * o + 1) * cap] = cvt<R>(__ldg(wo - off));
        }
        D = __ldg(V.dg + p);
      } else {
        const R cxm = cvt<R>(__ldg(V.kx + p - 1)), cxp = cvt<R>(__ldg(V.kx + p));
        const R cym = cvt<R>(__ldg(V.ky + p - sy)), cyp = cvt<R>(__ldg(V.ky + p));
        const R czm = cvt<R>(__ldg(V.kz + p - sz)), czp = cvt<R>(__ldg(V.kz + p));
        D = ((cxm + cxp) + (cym + cyp)) + (czm + czp);
        O[0] = cxm, O[cap] = cxp, O[2 * cap] = cym, O[3 * cap] = cyp, O[4 * cap] = czm, O[5 * cap] = czp;
      }
      O[nc * cap] = __ldg(V.dinv + p);
      O[(nc + 1) * cap] = D;
    });
  }
  if (!a.Ac && a.nc <= 32)
    for (int e = tid; e < a.nc * a.nc; e += BS_THREADS) Ais[e] = __ldg(a.Ai + e);
  sync();  // every block's windows are zeroed before another block stores into them
  pdl_wait();
  own_for(a.lv[0], [&](int t, int, int, int k, int p) {
    const R b = a.b[p];
    if (L == 1) put(0, 1, k, p, b);
    else start(0, t, k, p, b);
  });
  sync();

  // ---- down: pre-smoothing, residual, restriction
  unsigned curs = 0;  // bit l: the buffer that holds level l's iterate
  for (int l = 0; l + 1 < L; ++l) {
    const BsLevel<TV, TC>&V = a.lv[l], &W = a.lv[l + 1];
    const int base = bs_base(V, rank, false);
    int cur = 0;
    for (int s = 0; s < a.nu_pre; ++s) cur = steps(l, cur, s == 0 ? 1 : 0);
    curs |= (unsigned)cur << l;
    {
      const int nc = V.w ? 26 : 6;
      const R* X = sm + V.ox[cur] - base;
      own_for(V, [&](int t, int, int, int k, int p) {
        const R* O = sm + V.own + t;
        const R S = S_at(V, X + p, O);
        const R rv = (O[(nc + 2) * V.cap] + S) - O[(nc + 1) * V.cap] * X[p];
        put(l, cur ^ 1, k, p, rv);
      });
      sync();
    }
    const R* r = sm + V.ox[cur ^ 1] - base;
    own_for(W, [&](int t, int i, int j, int k, int pc) {
      const R* rc = r + (int)V.g.at(2 * i + 1, 2 * j + 1, 2 * k + 1);
      R acc = 0;
#pragma unroll
      for (int c = -1; c <= 1; ++c) {
        R plane = 0;
#pragma unroll
        for (int b = -1; b <= 1; ++b) {
          const R* q = rc + c * (int)V.g.sz + b * V.g.Px;
          const R row = fma((R)0.5, q[0], (R)0.25 * (q[-1] + q[1]));
          plane = fma(b == 0 ? (R)0.5 : (R)0.25, row, plane);
        }
        acc = fma(c == 0 ? (R)0.5 : (R)0.25, plane, acc);
      }
      if (l + 2 == L) put(l + 1, 1, k, pc, acc);  // the coarsest right-hand side, to every block
      else start(l + 1, t, k, pc, acc);
    });
    sync();
  }

  // ---- coarsest solve: every block holds the whole right-hand side
  {
    const BsLevel<TV, TC>& V = a.lv[L - 1];
    const int n = a.nc, base = bs_base(V, rank, true);
    const R* B = sm + V.ox[1] - base;
    R* X = sm + V.ox[0] - base;
    // f(u, p) for every unknown u at padded index p
    auto all = [&](auto f) {
      for (int t = tid; t < V.g.nz << (V.lx + V.ly); t += BS_THREADS) {
        const int i = t & ((1 << V.lx) - 1), j = (t >> V.lx) & ((1 << V.ly) - 1), k = t >> (V.lx + V.ly);
        if (i < V.g.nx && j < V.g.ny) f((k * V.g.ny + j) * V.g.nx + i, (int)V.g.at(i, j, k));
      }
    };
    all([&](int u, int p) { y[u] = cvt<double>(B[p]); });
    __syncthreads();
    if (a.Ac || n <= 32) {  // small: every block forms all of it
      if (a.Ac) block_gmres(a.Ac, n, a.coarse_rtol, a.coarse_maxit, y);
      else coarse_product_small(Ais, n, y);
      __syncthreads();
      all([&](int u, int p) { X[p] = store_as<R>(y[u]); });
      __syncthreads();
    } else {  // rows over the warps of all blocks
      const int nw = BS_THREADS / 32;
      for (int r = rank * nw + (tid >> 5); r < n; r += nb * nw) {
        const double v = coarse_row(a.Ai, n, y, r);
        if ((tid & 31) == 0) {
          const int k = r / (V.g.nx * V.g.ny), j = r / V.g.nx - k * V.g.ny;
          put(L - 1, 0, k, (int)V.g.at(r % V.g.nx, j, k), store_as<R>(v));
        }
      }
      sync();
    }
  }

  // ---- up: prolongation, post-smoothing
  for (int l = L - 2; l >= 0; --l) {
    const BsLevel<TV, TC>&V = a.lv[l], &W = a.lv[l + 1];
    int cur = (curs >> l) & 1;
    const int ccur = (curs >> (l + 1)) & 1;
    const R* X = sm + V.ox[cur] - bs_base(V, rank, false);
    const R* e = sm + W.ox[ccur] - bs_base(W, rank, l + 2 == L);
    own_for(V, [&](int, int i, int j, int k, int p) {
      const int i0 = (i - 1) >> 1, i1 = i >> 1, j0 = (j - 1) >> 1, j1 = j >> 1, k0 = (k - 1) >> 1, k1 = k >> 1;
      const int a00 = (int)W.g.at(i0, j0, k0), a10 = (int)W.g.at(i0, j1, k0), a01 = (int)W.g.at(i0, j0, k1),
                a11 = (int)W.g.at(i0, j1, k1);
      auto col = [&](int o) { return (e[a00 + o] + e[a01 + o]) + (e[a10 + o] + e[a11 + o]); };
      const R s = col(0) + col(i1 - i0);
      put(l, cur, k, p, fma((R)0.125, s, X[p]));
    });
    sync();
    for (int s = 0; s < a.nu_post; ++s) cur = steps(l, cur, 0);
    curs = (curs & ~(1u << l)) | ((unsigned)cur << l);
  }
  const R* X = sm + a.lv[0].ox[curs & 1] - bs_base(a.lv[0], rank, L == 1);
  own_for(a.lv[0], [&](int, int, int, int, int p) { a.out[p] = X[p]; });
}

}  // namespace mgdev
