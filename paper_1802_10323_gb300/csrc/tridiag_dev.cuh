// tridiag_dev.cuh — device code of the z tridiagonal solves of Eq. 5 (see tridiag.cu).
#pragma once
#include "internal.h"

namespace ps {

// 1/x. FP64: the hardware's approximation (rcp.approx.ftz.f64, measured relative error
// 2^−19.9) and one cubic step r(1 + e + e²), e = 1 − x·r, with three FP64 instructions. Over
// 16.8 M values of exponents −1000 to 1000 the error is at most 1.003·2^−53, against 1·2^−53 of
// the correctly rounded division, from which 0.03 % of the results differ; the division costs
// about nine instructions, and on this part an FP64 warp instruction holds its pipe for 64 cycles.
__device__ __forceinline__ float rcp_(float x) { return 1.f / x; }
__device__ __forceinline__ double rcp_(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

constexpr int ZCH = 4;  // rows whose loads are in flight together

// Rows are taken as (a + c + g) Φ̂_k = a Φ̂_{k−1} + c Φ̂_{k+1} − f̂_k with the couplings a, c ≥ 0
// and the excess g ≥ 0 of the diagonal (|λ|, the Helmholtz shift, a Dirichlet end) kept
// apart. The elimination Φ̂_k = C Φ̂_{k+1} + V has C + G = 1 with G the excess's share,
//   t = a G_{k−1} + g,  C = c/(c + t),  G = t/(c + t),  V = (a V_{k−1} − f̂)/(c + t),
// so every diagonal is a sum of non-negative terms (as in the Grassmann–Taksar–Heyman
// elimination) and a small |λ| next to large couplings loses no digits, while b + λ rounded
// to the working precision does: on 1024 FP64 rows with g = 10^−9 of the couplings the
// error is 2e-11 against 3e-8 (two instructions a row more).
//
// One column of Eq. 5 by one thread, in place, with C in the scratch array. Periodic z: the
// last unknown y = Φ̂_{n−1} is kept aside; every other row is eliminated to
// Φ̂_k = C Φ̂_{k+1} + F y + V (C + F + G = 1; F, in a second scratch array, carries the wrap
// coupling of row 0 along), and Φ̂_0 = T Φ̂_{k+1} + U y + S (T + U + X = 1; U is not needed) is
// composed on the way, so the last row gives y at the end of the forward sweep and one backward sweep
// finishes: the cyclic Gauss elimination, with one sweep less than solving two tridiagonal
// systems and combining them.
template <class T>
__device__ void zsolve_column(const ZArgs<T>& a, int col) {
  const int ncol = a.nx * a.ny;
  if (col >= ncol) return;
  if (a.singular && col == 0) return;
  const int i = col % a.nx, j = col / a.nx;
  const T lam = -(a.lamx[i] + a.lamy[j]);
  const size_t st = (size_t)ncol;
  const int nz = a.nz;
  T* __restrict__ d = a.data + col;
  T* __restrict__ sc = a.scr_c + col;
  T* __restrict__ su = a.periodic ? a.scr_u + col : nullptr;
  const T* __restrict__ za = a.za;
  const T* __restrict__ zc = a.zc;
  const T* __restrict__ zg = a.zg;
  const bool per = a.periodic;
  const int nr = per ? nz - 1 : nz;
  T V = (T)0, G = (T)0, F = (T)1, S = (T)0, Tc = (T)1, X = (T)0, C = (T)0;
  for (int k0 = 0; k0 < nr; k0 += ZCH) {
    T r[ZCH];
#pragma unroll
    for (int u = 0; u < ZCH; ++u) r[u] = d[min(k0 + u, nz - 1) * st];
#pragma unroll
    for (int u = 0; u < ZCH; ++u) {
      const int k = k0 + u;
      if (k < nr) {
        const T ak = (k > 0 || per) ? za[k] : (T)0, ck = zc[k], g = zg[k] + lam;
        const T t = ak * G + g;
        const T m = rcp_(per ? ck + (t + ak * F) : ck + t);
        V = ((k > 0 ? ak * V : (T)0) - r[u]) * m;
        G = t * m;
        C = ck * m;  // (non-periodic: never read in the last row)
        d[k * st] = V;
        sc[k * st] = C;
        if (per) {
          F = (ak * F) * m;
          S = S + Tc * V;
          X = X + Tc * G;
          Tc = Tc * C;
          su[k * st] = F;
        }
      }
    }
  }
  T x = V, y = (T)0;
  if (per) {
    const T al = za[nz - 1], cl = zc[nz - 1];
    y = (al * V + (cl * S - d[(nz - 1) * st])) * rcp_(cl * X + (al * G + (zg[nz - 1] + lam)));
    d[(nz - 1) * st] = y;
    x = y;
  }
  for (int k = nz - 2; k >= 0; k -= ZCH) {
    T rd[ZCH], rc[ZCH], ru[ZCH];
#pragma unroll
    for (int u = 0; u < ZCH; ++u) {
      const size_t o = max(k - u, 0) * st;
      rd[u] = d[o];
      rc[u] = sc[o];
      ru[u] = per ? su[o] : (T)0;
    }
#pragma unroll
    for (int u = 0; u < ZCH; ++u)
      if (k - u >= 0) {
        x = rd[u] + rc[u] * x;
        if (per) x = x + ru[u] * y;
        d[(k - u) * st] = x;
      }
  }
}

// ---- a column by a whole warp ------------------------------------------------------
//
// A column's elimination is a serial chain (FP64: ~9 dependent instructions of 33 ns a
// row; double-float: ~140 cycles a row), so where few columns are solved that way it is
// the chain that takes the time, not the arithmetic. Here the 32 lanes take a block of
// about n_z/32 consecutive rows each (a partition method): the last row e of a block is
// its separator; the rows above it are eliminated from both ends at once,
//   Φ̂_{e−1} = C Φ̂_e + F Φ̂_{s−1} + …,   Φ̂_s = Q Φ̂_e + R Φ̂_{s−1} + …
// (two independent chains); the 32 separator equations that result are solved by cyclic
// reduction across the lanes (five steps of shuffles; the lanes form a ring, which is
// the wrap coupling of a periodic z, and a non-periodic column has a_0 = c_{n−1} = 0);
// then each lane solves its block with both neighbours known.
//
// Couplings and excess as above, r = −f̂. A periodic column needs n_z ≥ 32 (a row for every
// lane of the ring).
__device__ __forceinline__ df n_add(df a, df b) { return df_add(a, b); }
__device__ __forceinline__ df n_mul(df a, df b) { return df_mul(a, b); }
__device__ __forceinline__ df n_fma(df a, df b, df c) { return df_add(c, df_mul(a, b)); }  // a·b + c
__device__ __forceinline__ df n_shfl(df a, int l) {
  return {__shfl_sync(0xffffffffu, a.h, l), __shfl_sync(0xffffffffu, a.l, l)};
}
__device__ __forceinline__ double n_add(double a, double b) { return a + b; }
__device__ __forceinline__ double n_mul(double a, double b) { return a * b; }
__device__ __forceinline__ double n_fma(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double n_shfl(double a, int l) { return __shfl_sync(0xffffffffu, a, l); }
template <class N>
__device__ __forceinline__ N n_num(float x);
template <>
__device__ __forceinline__ df n_num<df>(float x) { return {x, 0.f}; }
template <>
__device__ __forceinline__ double n_num<double>(float x) { return (double)x; }

// 1/x of a double-float pivot: the FP32 approximation r refined by one Newton step
// carried in double-float, r + r·e with e = 1 − x·r (x.h·r is formed exactly with an
// FMA; 1 − p is exact for p near 1), about 2^−46 relative.
__device__ __forceinline__ df n_rcp(df x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x.h));
  const float p = __fmul_rn(x.h, r);
  const float pe = __fmaf_rn(x.h, r, -p);
  const float e = __fsub_rn(__fsub_rn(__fsub_rn(1.f, p), pe), __fmul_rn(x.l, r));
  return quick_two_sum(r, __fmul_rn(r, e));
}
__device__ __forceinline__ double n_rcp(double x) { return rcp_(x); }

// row(k, a, c, g): the row's couplings and excess; rhs(k): r; save/load(k, c', d'): a place
// for two values of row k, used by this lane alone; put(k, x): the solution. Called by all
// 32 lanes of a warp.
template <class N, class Row, class Rhs, class Save, class Load, class Put>
__device__ __forceinline__ void zpart_column(int nz, Row&& row, Rhs&& rhs, Save&& save, Load&& load, Put&& put) {
  const int lane = threadIdx.x & 31;
  const int base = nz >> 5, rem = nz & 31;
  const int s = lane * base + min(lane, rem), cnt = base + (lane < rem ? 1 : 0);
  const int e = s + cnt - 1, ni = max(cnt - 1, 0);
  const N zero = n_num<N>(0.f), one = n_num<N>(1.f);
  // ---- the interior rows s … e−1 from both ends ----
  // downwards: Φ̂_k = C Φ̂_{k+1} + F Φ̂_{s−1} + V with C + F + G = 1 (G the excess's share);
  // upwards:   Φ̂_k = R Φ̂_{k−1} + Q Φ̂_e + W with R + Q + H = 1
  N F = one, G = zero, V = zero, Q = one, H = zero, W = zero, R = zero;
  N rd = zero, ru = zero;  // the next right-hand sides, loaded ahead
  if (ni > 0) {
    rd = rhs(s);
    ru = rhs(e - 1);
  }
  for (int u = 0; u < ni; ++u) {
    const N r0 = rd, r1 = ru;
    if (u + 1 < ni) {
      rd = rhs(s + u + 1);
      ru = rhs(e - 2 - u);
    }
    N a, c, g;
    row(s + u, a, c, g);
    const N m = n_rcp(n_add(c, n_fma(a, n_add(F, G), g)));
    V = n_mul(n_fma(a, V, r0), m);
    G = n_mul(n_fma(a, G, g), m);
    F = n_mul(n_mul(a, F), m);
    row(e - 1 - u, a, c, g);
    const N w = n_rcp(n_add(a, n_fma(c, n_add(Q, H), g)));
    W = n_mul(n_fma(c, W, r1), w);
    H = n_mul(n_fma(c, H, g), w);
    Q = n_mul(n_mul(c, Q), w);
    R = n_mul(a, w);
  }
  // ---- the separator equations (A + C + E) Φ̂(lane) = A Φ̂(lane−1) + C Φ̂(lane+1) + D ----
  N A = zero, C = zero, E = one, D = zero;
  {
    const int up = (lane + 1) & 31;
    const N Wn = n_shfl(W, up), Qn = n_shfl(Q, up), Hn = n_shfl(H, up);
    if (cnt > 0) {
      N a, c, g;
      row(e, a, c, g);
      A = n_mul(a, F);
      C = n_mul(c, Qn);
      E = n_fma(c, Hn, n_fma(a, G, g));
      D = n_fma(c, Wn, n_fma(a, V, rhs(e)));
    }
  }
#pragma unroll 1
  for (int h = 1; h < 16; h <<= 1) {
    const int lo = (lane - h) & 31, hi = (lane + h) & 31;
    const N rB = n_rcp(n_add(n_add(A, C), E));
    const N al = n_mul(A, n_shfl(rB, lo)), ga = n_mul(C, n_shfl(rB, hi));
    const N El = n_shfl(E, lo), Eh = n_shfl(E, hi), Dl = n_shfl(D, lo), Dh = n_shfl(D, hi);
    const N Al = n_shfl(A, lo), Ch = n_shfl(C, hi);
    E = n_fma(ga, Eh, n_fma(al, El, E));
    D = n_fma(ga, Dh, n_fma(al, Dl, D));
    A = n_mul(al, Al);
    C = n_mul(ga, Ch);
  }
  N x;
  {  // both neighbours are lane ± 16
    const int o = lane ^ 16;
    const N AC = n_add(A, C);
    const N al = n_mul(AC, n_shfl(n_rcp(n_add(AC, E)), o));
    const N Eo = n_shfl(E, o), Do = n_shfl(D, o);
    x = n_mul(n_fma(al, Do, D), n_rcp(n_fma(al, Eo, E)));
  }
  // ---- the blocks, both neighbours known ----
  const N xs = n_shfl(x, (lane - 1) & 31);
  if (cnt > 0) put(e, x);
  V = xs;
  G = one;  // (Φ̂_{s−1} is known: its coupling is all excess)
  if (ni > 0) rd = rhs(s);
  for (int u = 0; u < ni; ++u) {
    const N r0 = rd;
    if (u + 1 < ni) rd = rhs(s + u + 1);
    N a, c, g;
    row(s + u, a, c, g);
    const N t = n_fma(a, G, g);
    const N m = n_rcp(n_add(c, t));
    V = n_mul(n_fma(a, V, r0), m);
    G = n_mul(t, m);
    save(s + u, n_mul(c, m), V);
  }
  for (int k = s + ni - 1; k >= s; --k) {
    N c, v;
    load(k, c, v);
    x = n_fma(c, x, v);
    put(k, x);
  }
}

// A column in FP64 by one warp, in place; `sing`: the singular column (0,0) of a problem
// whose every axis is periodic or Neumann–Neumann: its right-hand side loses its
// Δz^f-weighted mean, Φ̂_0 = 0 is pinned (row 0 dropped), and the solution's mean is removed.
__device__ __forceinline__ void zpart64(const ZArgs<double>& a, int col, bool sing) {
  const int nz = a.nz, lane = threadIdx.x & 31;
  const size_t st = (size_t)a.nx * a.ny;
  const double lam = -(a.lamx[col % a.nx] + a.lamy[col / a.nx]);
  double* d = a.data + col;
  double* sc = a.scr_c + col;
  auto wmean = [&]() {  // Δz^f-weighted mean of the column
    double num = 0.0, den = 0.0;
    for (int k = lane; k < nz; k += 32) {
      num += a.dzf[k] * d[k * st];
      den += a.dzf[k];
    }
    for (int o = 16; o > 0; o >>= 1) {
      num += __shfl_xor_sync(0xffffffffu, num, o);
      den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    return num / den;
  };
  const double mean = sing ? wmean() : 0.0;
  const bool wrap = a.periodic;
  auto row = [&](int k, double& p, double& q, double& g) {  // (a.zg: the excess without λ)
    p = (k > 0 || wrap) ? a.za[k] : 0.0;
    q = (k < nz - 1 || wrap) ? a.zc[k] : 0.0;
    g = a.zg[k] + lam;
    if (sing) {  // Φ̂_0 = 0: row 0 alone, the couplings to it are excess
      if (k == 0) p = q = 0.0, g = 1.0;
      if (k == 1) g += p, p = 0.0;
      if (k == nz - 1 && wrap) g += q, q = 0.0;
    }
  };
  auto rhs = [&](int k) { return (sing && k == 0) ? 0.0 : mean - d[k * st]; };
  auto save = [&](int k, double c, double v) {
    sc[k * st] = c;
    d[k * st] = v;
  };
  auto load = [&](int k, double& c, double& v) {
    c = sc[k * st];
    v = d[k * st];
  };
  zpart_column<double>(nz, row, rhs, save, load, [&](int k, double x) { d[k * st] = x; });
  if (sing) {
    __syncwarp();
    const double mx = wmean();
    __syncwarp();
    for (int k = lane; k < nz; k += 32) d[k * st] -= mx;
  }
}

// A column of FP32 data in double-float by one warp, in place (rounded to FP32 at the end);
// the singular column (0,0) as in zpart64. cs, ds: n_z float pairs of scratch each.
__device__ __forceinline__ void zcolumn_df(const ZArgs<float>& a, int col, float2* cs, float2* ds) {
  const int nz = a.nz, lane = threadIdx.x & 31;
  const size_t st = (size_t)a.nx * a.ny;
  const int i = col % a.nx, j = col / a.nx;
  float* d = a.data + col;
  const bool sing = a.singular && col == 0, wrap = a.periodic;
  auto total = [&](df v) {
    for (int o = 16; o > 0; o >>= 1)
      v = df_add(v, df{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)});
    return v;
  };
  df mn = {0.f, 0.f}, rws = {0.f, 0.f};
  if (sing) {  // remove the Δz^f-weighted mean of the right-hand side; Φ̂_0 = 0 pinned
    df num = {0.f, 0.f}, den = {0.f, 0.f};
    for (int k = lane; k < nz; k += 32) {
      const df w = df_from_f64(a.dzf64[k]);
      num = df_add(num, df_mul(w, df{d[k * st], 0.f}));
      den = df_add(den, w);
    }
    rws = n_rcp(total(den));
    mn = df_mul(total(num), rws);
  }
  const df lam = sing ? df{0.f, 0.f} : df_from_f64(-(a.lamx64[i] + a.lamy64[j]));  // |λ|
  auto row = [&](int k, df& p, df& q, df& g) {
    const float2 za = __ldg(a.zdf + 3 * k), zc = __ldg(a.zdf + 3 * k + 1), zg = __ldg(a.zdf + 3 * k + 2);
    p = (k > 0 || wrap) ? df{za.x, za.y} : df{0.f, 0.f};
    q = (k < nz - 1 || wrap) ? df{zc.x, zc.y} : df{0.f, 0.f};
    g = df_add(df{zg.x, zg.y}, lam);
    if (sing) {  // Φ̂_0 = 0: row 0 alone, the couplings to it are excess
      if (k == 0) p = q = df{0.f, 0.f}, g = df{1.f, 0.f};
      if (k == 1) g = df_add(g, p), p = df{0.f, 0.f};
      if (k == nz - 1 && wrap) g = df_add(g, q), q = df{0.f, 0.f};
    }
  };
  auto rhs = [&](int k) {
    const float v = -d[k * st];
    if (!sing) return df{v, 0.f};
    return k == 0 ? df{0.f, 0.f} : df_add(df{v, 0.f}, mn);
  };
  auto save = [&](int k, df c, df v) {
    cs[k] = make_float2(c.h, c.l);
    ds[k] = make_float2(v.h, v.l);
  };
  auto load = [&](int k, df& c, df& v) {
    const float2 x = cs[k], y = ds[k];
    c = df{x.x, x.y};
    v = df{y.x, y.y};
  };
  if (!sing) {
    zpart_column<df>(nz, row, rhs, save, load, [&](int k, df x) { d[k * st] = __fadd_rn(x.h, x.l); });
    return;
  }
  df xs = {0.f, 0.f};
  zpart_column<df>(nz, row, rhs, save, load, [&](int k, df x) {
    xs = df_add(xs, df_mul(df_from_f64(a.dzf64[k]), x));
    ds[k] = make_float2(x.h, x.l);
  });
  const df mx = df_mul(total(xs), rws);
  __syncwarp();  // the solution in ds is visible to the lanes below
  for (int k = lane; k < nz; k += 32) {  // the singular column keeps zero weighted mean
    const float2 v = ds[k];
    const df y = df_sub(df{v.x, v.y}, mx);
    d[k * st] = __fadd_rn(y.h, y.l);
  }
}

}  // namespace ps
