// xform_units.cuh — the units of work of the register-resident line transforms:
// one x line per warp (row_line) and one tile of CW y columns per CTA (col_tile),
// called by the per-axis kernels (xform_row.cu, xform_col.cu). The mathematics is
// the same in every unit: an M-point complex FFT per line of n = 2M reals with the
// Table 2 pre/post processing per BC; the layouts are described in the two kernel
// files.
#pragma once
#include <type_traits>

#include "xform_fast.cuh"

namespace ps {

// Twiddle tables of one axis into shared memory at stw: ω_M^t (t < M), the
// real-FFT split factors (M + 1) and the BC factors (NN/DD: n; ND: 2·M).
// The halves of the split, the 2 of the cosine outputs and the 1/M and 1/n of the
// backward transform are powers of two and sit in the factors that multiply every value
// anyway (or in a fused multiply-add with the split's sum, split_scale): the results
// keep their bits, and the FP64 passes, which the FP64 pipe bounds, lose a quarter of
// their arithmetic outside the FFT stages (NN pair of wavenumbers, forward 32 → 20
// instructions, backward 36 → 20). FP64 256³ (DD, ND, NN) 2945 → 2647 µs; FP32
// passes are bound by memory and keep their time.
template <class T, int M, bool FWD>
__device__ __forceinline__ void load_line_tables(const cplx<T>* tw, int bc, cplx<T>* stw) {
  constexpr int N = 2 * M;
  constexpr T half = (T)0.5, inv_m = (T)1 / (T)M;  // exact
  cplx<T>* ptw = stw + M;
  cplx<T>* xtw = ptw + (M + 1);
  for (int i = threadIdx.x; i < M; i += blockDim.x) stw[i] = tw[16 * i];
  const T fs = bc == BC_P ? (FWD ? half : half * inv_m) : (T)1;
  for (int i = threadIdx.x; i <= M; i += blockDim.x) ptw[i] = cscale(tw[8 * i], fs);
  if (bc == BC_NN || bc == BC_DD) {
    for (int i = threadIdx.x; i < N; i += blockDim.x)
      xtw[i] = FWD ? tw[2 * i] : cscale(tw[2 * i], half * half * inv_m);
  } else if (bc_iv(bc)) {
    for (int i = threadIdx.x; i < M; i += blockDim.x) {
      xtw[i] = tw[4 * i];
      xtw[M + i] = cscale(tw[4 * i + 1], FWD ? (T)2 : half * inv_m);
    }
  }
}

// The two wavenumbers of a pair from (or to) its even and odd parts e, o (o already
// multiplied by its table factor): h·e ± o with the factor h of periodic lines, which
// have no other table to hold it (h = 1 and a plain sum otherwise).
template <class T>
__device__ __forceinline__ cplx<T> split_add(cplx<T> e, cplx<T> o, T h) {
  return {fma(h, e.x, o.x), fma(h, e.y, o.y)};
}
template <class T>
__device__ __forceinline__ cplx<T> split_sub(cplx<T> e, cplx<T> o, T h) {
  return {fma(h, e.x, -o.x), fma(h, e.y, -o.y)};
}
// h of a line's split (see above).
template <class T, int M, bool FWD>
__device__ __forceinline__ T split_scale(int bc) {
  return bc == BC_P ? (FWD ? (T)0.5 : (T)0.5 / (T)M) : (T)1;
}

namespace row {

using fast::Shape;
using fast::cpad;

template <class T, int N>
struct alignas(sizeof(T) * N) vec {
  T v[N];
};

// Warps per CTA and wide stages (fast::Shape) for FP64: few warps with many registers, the
// pipe needs no more
template <class T>
constexpr int kWarps = sizeof(T) == 8 ? 4 : 8;
template <class T>
constexpr bool kWide = sizeof(T) == 8;
// FP64 passes of at most this many lines (two per SM sub-partition) take the narrow stages:
// there a pass is one warp's chain of FP64 instructions, which a wide warp's four lines
// (M = 128) make four times longer. Forward passes, periodic, µs, wide and narrow: n = 256,
// 512 lines 25.5 and 14.6, 1024 lines 26.1 and 17.7, 2048 lines 26.2 and 27.0; n = 512,
// 512 lines 27.4 and 18.8, 1024 lines 28.5 and 27.3, 2048 lines 44.5 and 45.6.
constexpr int kFewLines = 1216;

template <class TC, class TI>
__device__ __forceinline__ TC in_cvt(TI x) { return ld_cvt<TC, TI>::f(x); }

// Output modes of the backward transform (compile-time, so that no mode pays for
// another's registers): store; accumulate (out += v); base (out = widen(base32) + v);
// none (no FP64 output: only the FP32 copy and the max).
enum { OM_STORE = 0, OM_ACC = 1, OM_BASE = 2, OM_NONE = 3 };

// Slots of a 32-lane line (M ≥ 128): lane t holds wavenumbers k = t + 32·j, j < E.
// After the last FFT stage slot si holds j = jout(si); the first stage takes slot si
// at j = jin(si). The partner M − k of k is held by lane (32 − t) mod 32 at
// j' = E − 1 − j (lane 0: j' = E − j, and k = 0 pairs with itself).
template <int M>
struct LaneSlots {
  static constexpr int E = Shape<M>::E, R0 = Shape<M>::radix(0), RL = Shape<M>::radix(Shape<M>::NST - 1);
  __host__ __device__ static constexpr int jin(int si) { return si / R0 + (si % R0) * (M / R0 / 32); }
  __host__ __device__ static constexpr int jout(int si) { return si / RL + (si % RL) * (M / RL / 32); }
  __host__ __device__ static constexpr int sin_(int j) {
    int r = 0;
    for (int s = 0; s < E; ++s)
      if (jin(s) == j) r = s;
    return r;
  }
  __host__ __device__ static constexpr int sout(int j) {
    int r = 0;
    for (int s = 0; s < E; ++s)
      if (jout(s) == j) r = s;
    return r;
  }
};

// One line (two for M = 64, half a warp each) of the x transform: the warp's
// exchange buffers at bufs, tables in shared memory, the first line index l0.
// tmax accumulates max |FP64 output| for the caller's reduction (before widening; FP64
// transforms only when asked: the comparison costs their pipe).
template <class T, class TI, class TO, int M, bool FWD, int OM, bool W>
__device__ __forceinline__ void row_line(const FastArgs<T>& a, const cplx<T>* stw, const cplx<T>* ptw,
                                         const cplx<T>* xtw, cplx<T>* bufs, int l0, T& tmax) {
  using S = Shape<M, W>;
  constexpr int N = 2 * M, E = S::E, TPL = S::TPL;
  constexpr int R0 = S::radix(0), RL = S::radix(S::NST - 1);
  constexpr int LB = M + M / 8;  // complex slots of a line's exchange buffer (skewed)
  const int bc = a.bc;
  const int lane = threadIdx.x & 31;
  const int t = lane % TPL, half = lane / TPL;
  const int mate = lane ^ (TPL - 1);  // lane of the mirrored points M−1−p
  cplx<T>* lc = bufs + half * LB;
  const TI* in = static_cast<const TI*>(a.in);  // may equal out (in-place passes)
  TO* out = static_cast<TO*>(a.out);
  const int ny = a.ny, nlines = a.nlines;
  const unsigned full = 0xffffffffu;
  const int line = l0 + half;
  const bool live = line < nlines;  // the other half-warp line may be past the end
  const size_t base = (size_t)(live ? line : l0) * N;
  const TI* src = in + base;
  TO* dst = out + base;
  const bool scaled = a.plane_scale != nullptr;
  const T s = scaled ? a.plane_scale[(live ? line : l0) / ny] : (T)1;
  const T h = split_scale<T, M, FWD>(bc);
  cplx<T> v[E];
  if (FWD) {
    // ---- gather the first-stage operands from the line ----
    // slot si = q·R0 + r holds point p = t + q·TPL + r·(M/R0); p < M/2 iff r < R0/2
    if (bc == BC_P) {
#pragma unroll
      for (int si = 0; si < E; ++si) {
        const int p = t + (si / R0) * TPL + (si % R0) * (M / R0);
        const vec<TI, 2> x = *reinterpret_cast<const vec<TI, 2>*>(src + 2 * p);
        v[si] = {in_cvt<T>(x.v[0]), in_cvt<T>(x.v[1])};
      }
    } else if (bc_iv(bc)) {
      // z_p = (x_{2p}, x_{n−1−2p})·e^{−iπp/n}; x_{n−1−2p} = x_{2p'+1} of p' = M−1−p
      // (DN, the reversed line: z_p = (x_{n−1−2p}, x_{2p}), the two parts trade places)
#pragma unroll
      for (int si = 0; si < E; ++si) {
        const int p = t + (si / R0) * TPL + (si % R0) * (M / R0);
        const vec<TI, 2> x = *reinterpret_cast<const vec<TI, 2>*>(src + 2 * p);
        v[si].x = in_cvt<T>(x.v[0]);
        const T odd = in_cvt<T>(x.v[1]);
        v[E - 1 - si].y = __shfl_sync(full, odd, mate);
      }
      if (bc == BC_DN) {
#pragma unroll
        for (int si = 0; si < E; ++si) v[si] = {v[si].y, v[si].x};
      }
#pragma unroll
      for (int si = 0; si < E; ++si) {
        const int p = t + (si / R0) * TPL + (si % R0) * (M / R0);
        v[si] = cmul(v[si], xtw[p]);
      }
    } else {
      // z_p = (v_{2p}, v_{2p+1}) with v_j = x_{2j} (j < M), ±x_{2n−1−2j} (j ≥ M, − for DD);
      // the 4-vector at 4p (p < M/2) is (z_p.x, z_{p'}.y, z_p.y, z_{p'}.x), p' = M−1−p
      const bool neg = (bc == BC_DD);
#pragma unroll
      for (int si = 0; si < E; ++si) {
        if ((si % R0) >= R0 / 2) continue;
        const int p = t + (si / R0) * TPL + (si % R0) * (M / R0);
        T x[4];
        if constexpr (sizeof(TI) == 4) {
          const vec<TI, 4> q = *reinterpret_cast<const vec<TI, 4>*>(src + 4 * p);
#pragma unroll
          for (int u = 0; u < 4; ++u) x[u] = in_cvt<T>(q.v[u]);
        } else {
          const vec<TI, 2> q0 = *reinterpret_cast<const vec<TI, 2>*>(src + 4 * p);
          const vec<TI, 2> q1 = *reinterpret_cast<const vec<TI, 2>*>(src + 4 * p + 2);
          x[0] = in_cvt<T>(q0.v[0]);
          x[1] = in_cvt<T>(q0.v[1]);
          x[2] = in_cvt<T>(q1.v[0]);
          x[3] = in_cvt<T>(q1.v[1]);
        }
        v[si] = {x[0], x[2]};
        const T ry = __shfl_sync(full, x[1], mate), rx = __shfl_sync(full, x[3], mate);
        v[E - 1 - si] = neg ? cplx<T>{-rx, -ry} : cplx<T>{rx, ry};
      }
    }
    if (scaled) {
#pragma unroll
      for (int si = 0; si < E; ++si) v[si] = cscale(v[si], s);
    }
    fast::fft_stages<T, M, false, 0, 1, W>(v, lc, stw, t);
    if constexpr (TPL == 32) {
      // ---- post-processing in registers: pairs (k, M−k), Z_{M−k} from the partner lane ----
      // Lane t takes its slots j < E/2 (k = t + 32j) and writes the outputs of k and of
      // M − k, whose Z arrives by shuffle from slot E−1−j of lane (32 − t) mod 32; every
      // slot is read once. Lane 0's partners are its own slots E − j: the value it
      // shuffled to itself one iteration earlier (k = 0 pairs with itself), and after the
      // loop, the one of k = M/2.
      using LS = LaneSlots<M>;
      auto Y = [&](int i, T val) {
        if (live) dst[i] = st_cvt<TO, T>::f(val);
      };
      if (bc_iv(bc)) {
#pragma unroll
        for (int j = 0; j < E; ++j) {
          const int k = t + 32 * j;
          const cplx<T> c = cmul(xtw[M + k], v[LS::sout(j)]);
          Y(2 * k, c.x);
          Y(N - 1 - 2 * k, -c.y);
        }
      } else {
        const int pl = (32 - t) & 31;
        const bool rev = (bc == BC_DD);
        auto OUTQ = [&](int q, T val) { Y(rev ? (N - 1 - q) : q, val); };
        // outputs of k (and of M − k unless k = 0 or 2k = M) from Z_k and Z_{M−k}
        auto pair_out = [&](int k, cplx<T> Zk, cplx<T> Zmk, bool self) {
          cplx<T> Vk, Vmk;
          if (self) {  // k = M/2 is its own partner
            Vk = Vmk = cscale(conj_(Zk), (T)2 * h);
          } else {
            const cplx<T> Ek = cadd(Zk, conj_(Zmk));
            const cplx<T> Ok = mul_mi(csub(Zk, conj_(Zmk)));
            const cplx<T> B = cmul(ptw[k], Ok);
            Vk = split_add(Ek, B, h);
            Vmk = conj_(split_sub(Ek, B, h));
          }
          if (bc == BC_P) {
            if (k == 0) {
              Y(0, Vk.x);
              Y(N - 1, Vmk.x);
            } else {
              Y(2 * k - 1, Vk.x);
              Y(2 * k, -Vk.y);
              if (2 * k != M) {
                Y(2 * (M - k) - 1, Vmk.x);
                Y(2 * (M - k), -Vmk.y);
              }
            }
          } else if (k == 0) {
            OUTQ(0, Vk.x);
            OUTQ(M, (T)0.70710678118654752440 * Vmk.x);
          } else {
            const cplx<T> c1 = cmul(xtw[k], Vk);
            OUTQ(k, c1.x);
            OUTQ(N - k, -c1.y);
            if (2 * k != M) {
              const cplx<T> c2 = cmul(xtw[M - k], Vmk);
              OUTQ(M - k, c2.x);
              OUTQ(M + k, -c2.y);
            }
          }
        };
        cplx<T> prev = {(T)0, (T)0};
#pragma unroll
        for (int j = 0; j < E / 2; ++j) {
          const cplx<T> Zk = v[LS::sout(j)];
          const cplx<T> recv = {__shfl_sync(full, v[LS::sout(E - 1 - j)].x, pl),
                                __shfl_sync(full, v[LS::sout(E - 1 - j)].y, pl)};
          const cplx<T> Zmk = (t != 0) ? recv : (j == 0 ? Zk : prev);
          prev = recv;
          pair_out(t + 32 * j, Zk, Zmk, false);
        }
        if (t == 0) pair_out(M / 2, prev, prev, true);
      }
    } else {
      // ---- post-processing: pairs (k, M−k) through the exchange buffer, scalar stores ----
      __syncwarp();
  #pragma unroll
      for (int q = 0; q < E / RL; ++q)
  #pragma unroll
        for (int r = 0; r < RL; ++r) lc[cpad(t + q * TPL + r * (M / RL))] = v[q * RL + r];
      __syncwarp();
      auto Y = [&](int i, T val) {
        if (live) dst[i] = st_cvt<TO, T>::f(val);
      };
      if (bc_iv(bc)) {
  #pragma unroll
        for (int i = 0; i < E; ++i) {
          const int k = t + i * TPL;
          const cplx<T> c = cmul(xtw[M + k], lc[cpad(k)]);
          Y(2 * k, c.x);
          Y(N - 1 - 2 * k, -c.y);
        }
      } else {
        constexpr int NP = (M / 2) / TPL + 1;
  #pragma unroll
        for (int i = 0; i < NP; ++i) {
          const int k = t + i * TPL;
          if (k > M / 2) break;
          const cplx<T> Zk = lc[cpad(k)], Zmk = lc[cpad(k == 0 ? 0 : M - k)];
          cplx<T> Vk, Vmk;
          if (i == NP - 1) {  // k = M/2 is its own partner
            Vk = Vmk = cscale(conj_(Zk), (T)2 * h);
          } else {
            const cplx<T> Ek = cadd(Zk, conj_(Zmk));
            const cplx<T> Ok = mul_mi(csub(Zk, conj_(Zmk)));
            const cplx<T> B = cmul(ptw[k], Ok);
            Vk = split_add(Ek, B, h);
            Vmk = conj_(split_sub(Ek, B, h));
          }
          if (bc == BC_P) {
            if (k == 0) {
              Y(0, Vk.x);
              Y(N - 1, Vmk.x);
            } else {
              Y(2 * k - 1, Vk.x);
              Y(2 * k, -Vk.y);
              if (2 * k != M) {
                Y(2 * (M - k) - 1, Vmk.x);
                Y(2 * (M - k), -Vmk.y);
              }
            }
          } else {
            const bool rev = (bc == BC_DD);
            auto OUTQ = [&](int q, T val) { Y(rev ? (N - 1 - q) : q, val); };
            if (k == 0) {
              OUTQ(0, Vk.x);
              OUTQ(M, (T)0.70710678118654752440 * Vmk.x);
            } else {
              const cplx<T> c1 = cmul(xtw[k], Vk);
              OUTQ(k, c1.x);
              OUTQ(N - k, -c1.y);
              if (2 * k != M) {
                const cplx<T> c2 = cmul(xtw[M - k], Vmk);
                OUTQ(M - k, c2.x);
                OUTQ(M + k, -c2.y);
              }
            }
          }
        }
      }
      __syncwarp();  // buffer reads done before the next line overwrites it
    }
  } else {
    // The FP64 output modes read the line's base (FP32 Φ_0) or its accumulator (FP64
    // p) only when the outputs are written; ask L2 for them now, one 128-byte
    // segment per lane, so that those loads do not wait on HBM after the transform.
    if constexpr (sizeof(TO) == 8 && sizeof(T) == 4 && (OM == OM_BASE || OM == OM_ACC)) {
      if (live) {
        const char* pf = (OM == OM_BASE) ? reinterpret_cast<const char*>(a.base32 + base)
                                         : reinterpret_cast<const char*>(dst);
        constexpr int SEG = (OM == OM_BASE ? N * 4 : N * 8) / 128;  // 128-byte segments of the line
#pragma unroll
        for (int j = t; j < SEG; j += TPL) asm volatile("prefetch.global.L2 [%0];" ::"l"(pf + 128 * j));
      }
    }
    auto X = [&](int i) { return in_cvt<T>(src[i]); };
    if constexpr (TPL == 32) {
      // ---- backward pre-processing in registers: own V_k, V_{M−k} from the partner lane,
      // Z_k straight into its first-stage slot ----
      using LS = LaneSlots<M>;
      if (bc_iv(bc)) {
        // (x_{2k}, x_{n−1−2k})·e^{−iπk/n}; x_{n−1−2k} = x_{2k'+1} of k' = M−1−k (mirrored lane)
        cplx<T> z[E];
#pragma unroll
        for (int i = 0; i < E; ++i) {
          const int k = t + i * TPL;
          const vec<TI, 2> x = *reinterpret_cast<const vec<TI, 2>*>(src + 2 * k);
          z[i].x = in_cvt<T>(x.v[0]);
          z[E - 1 - i].y = __shfl_sync(full, in_cvt<T>(x.v[1]), mate);
        }
#pragma unroll
        for (int j = 0; j < E; ++j) v[LS::sin_(j)] = cmul(z[j], xtw[t + 32 * j]);
      } else {
        const bool rev = (bc == BC_DD);
        auto qx = [&](int q) { return rev ? (N - 1 - q) : q; };
        cplx<T> Vv[E];
#pragma unroll
        for (int j = 0; j < E; ++j) {
          const int k = t + 32 * j;
          if (bc == BC_P) {
            Vv[j] = (k == 0) ? cplx<T>{X(0), (T)0} : cplx<T>{X(2 * k - 1), -X(2 * k)};
          } else {
            const T x0 = X(qx(k)), x1 = (k == 0) ? (T)0 : X(qx(N - k));
            cplx<T> w = xtw[k];
            w.y = -w.y;
            Vv[j] = cmul(w, cplx<T>{x0, -x1});
          }
        }
        // V_M, the partner of k = 0 (lane 0)
        cplx<T> VM;
        if (bc == BC_P) {
          VM = {X(N - 1), (T)0};
        } else {
          const T xm = X(qx(M));
          cplx<T> w = xtw[M];
          w.y = -w.y;
          VM = cmul(w, cplx<T>{xm, -xm});
        }
        const int pl = (32 - t) & 31;
#pragma unroll
        for (int j = 0; j < E; ++j) {
          const int k = t + 32 * j;
          cplx<T> Vm = {__shfl_sync(full, Vv[E - 1 - j].x, pl), __shfl_sync(full, Vv[E - 1 - j].y, pl)};
          if (t == 0) Vm = (j == 0) ? VM : Vv[(E - j) % E];
          const cplx<T> Ek = cadd(Vv[j], conj_(Vm));
          cplx<T> wn = ptw[k];
          wn.y = -wn.y;
          const cplx<T> Ok = cmul(csub(Vv[j], conj_(Vm)), wn);
          v[LS::sin_(j)] = split_add(Ek, mul_i(Ok), h);
        }
      }
    } else {
      // ---- backward pre-processing: pairs (k, M−k) from the line into the buffer ----
      if (bc_iv(bc)) {
        // (x_{2k}, x_{n−1−2k})·e^{−iπk/n}; x_{n−1−2k} = x_{2k'+1} of k' = M−1−k
  #pragma unroll
        for (int i = 0; i < E; ++i) {
          const int k = t + i * TPL;
          const vec<TI, 2> x = *reinterpret_cast<const vec<TI, 2>*>(src + 2 * k);
          v[i].x = in_cvt<T>(x.v[0]);
          v[E - 1 - i].y = __shfl_sync(full, in_cvt<T>(x.v[1]), mate);
        }
  #pragma unroll
        for (int i = 0; i < E; ++i) {
          const int k = t + i * TPL;
          lc[cpad(k)] = cmul(v[i], xtw[k]);
        }
      } else {
        constexpr int NP = (M / 2) / TPL;  // pairs (k, M − k) of a thread; k = M/2, its own partner, is t = 0's
        const bool rev = (bc == BC_DD);
        T xv[NP][4], xs[2] = {(T)0, (T)0};
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          const int k = t + i * TPL;
          int q[4];
          bool use[4] = {true, true, true, true};
          if (bc == BC_P) {
            q[0] = k == 0 ? 0 : 2 * k - 1;
            q[1] = 2 * k;
            q[2] = k == 0 ? N - 1 : 2 * (M - k) - 1;
            q[3] = 2 * (M - k);
            use[1] = use[3] = k != 0;
          } else {
            const int qq[4] = {k, N - k, M - k, N - M + k};
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              q[u] = rev ? (N - 1 - qq[u]) : qq[u];
              use[u] = qq[u] < N;
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) xv[i][u] = use[u] ? X(q[u]) : (T)0;
        }
        if (t == 0) {
          xs[0] = X(bc == BC_P ? M - 1 : (rev ? N - 1 - M / 2 : M / 2));
          xs[1] = X(bc == BC_P ? M : (rev ? M / 2 - 1 : N - M / 2));
        }
        auto V = [&](int k, T x0, T x1) {
          if (bc == BC_P) return cplx<T>{x0, -x1};
          cplx<T> w = xtw[k];
          w.y = -w.y;
          return cmul(w, cplx<T>{x0, -x1});
        };
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          const int k = t + i * TPL;
          const cplx<T> Vk = V(k, xv[i][0], xv[i][1]), Vm = V(M - k, xv[i][2], xv[i][3]);
          const cplx<T> Ek = cadd(Vk, conj_(Vm));
          cplx<T> wn = ptw[k];
          wn.y = -wn.y;
          const cplx<T> Ok = cmul(csub(Vk, conj_(Vm)), wn);
          lc[cpad(k)] = split_add(Ek, mul_i(Ok), h);
          if (k != 0) lc[cpad(M - k)] = split_add(conj_(Ek), mul_i(conj_(Ok)), h);
        }
        if (t == 0) lc[cpad(M / 2)] = cscale(conj_(V(M / 2, xs[0], xs[1])), (T)2 * h);
      }
      __syncwarp();
  #pragma unroll
      for (int q = 0; q < E / R0; ++q)
  #pragma unroll
        for (int r = 0; r < R0; ++r) v[q * R0 + r] = lc[cpad(t + q * TPL + r * (M / R0))];
    }
    if (bc_iv(bc)) fast::fft_stages<T, M, false, 0, 1, W>(v, lc, stw, t);
    else fast::fft_stages<T, M, true, 0, 1, W>(v, lc, stw, t);
    __syncwarp();  // the last stage's buffer reads are done before the next line
    // ---- backward outputs straight from the last stage, as vectors ----
    // slot si = q·RL + r holds wavenumber k = t + q·TPL + r·(M/RL); k < M/2 iff r < RL/2
    // n consecutive outputs at i0; an FP64 output may also keep its FP32 value in out2
    // (the line's own input array: every input of the line is already in registers)
    auto put = [&](int i0, const T* val, auto n_tag) {
      constexpr int NV = decltype(n_tag)::value;
      constexpr bool F64OUT = sizeof(TO) == 8 && sizeof(T) == 4;
      vec<TO, NV> o;
      vec<T, NV> o2;
      if constexpr (OM == OM_ACC) o = *reinterpret_cast<const vec<TO, NV>*>(dst + i0);
      if constexpr (F64OUT && OM == OM_BASE) {
        const vec<float, NV> b32 = *reinterpret_cast<const vec<float, NV>*>(a.base32 + base + i0);
#pragma unroll
        for (int u = 0; u < NV; ++u) o.v[u] = widen_f32(b32.v[u]);
      }
#pragma unroll
      for (int u = 0; u < NV; ++u) {
        o2.v[u] = val[u];
        const TO x = st_cvt<TO, T>::f(o2.v[u]);
        if constexpr (OM == OM_ACC || (F64OUT && OM == OM_BASE)) o.v[u] = o.v[u] + x;
        else o.v[u] = x;
        if constexpr (sizeof(TO) == 8)
          if (live && (sizeof(T) == 4 || a.amax)) tmax = fmax(tmax, fabs(o2.v[u]));
      }
      if (live) {
        if constexpr (OM != OM_NONE) *reinterpret_cast<vec<TO, NV>*>(dst + i0) = o;
        if constexpr (F64OUT)
          if (a.out2) *reinterpret_cast<vec<T, NV>*>(a.out2 + base + i0) = o2;
      }
    };
    using two = std::integral_constant<int, 2>;
    using four = std::integral_constant<int, 4>;
    if (scaled) {
#pragma unroll
      for (int si = 0; si < E; ++si) v[si] = cscale(v[si], s);
    }
    if (bc == BC_P) {
#pragma unroll
      for (int si = 0; si < E; ++si) {
        const int k = t + (si / RL) * TPL + (si % RL) * (M / RL);
        const T val[2] = {v[si].x, v[si].y};
        put(2 * k, val, two{});
      }
    } else if (bc_iv(bc)) {
      // output 2k = Re(c_k), output n−1−2k = −Im(c_k) with c_k = e^{...}·z_k/n;
      // the pair (2k, 2k+1) takes −Im(c_{k'}) of k' = M−1−k from the mirrored slot
      // (DN, the reversed line: the two outputs of each k trade places)
      T re[E], im[E];
#pragma unroll
      for (int si = 0; si < E; ++si) {
        const int k = t + (si / RL) * TPL + (si % RL) * (M / RL);
        const cplx<T> c = cmul(xtw[M + k], v[si]);
        const T A = c.x, B = -c.y;
        re[si] = (bc == BC_DN) ? B : A;
        im[si] = (bc == BC_DN) ? A : B;
      }
#pragma unroll
      for (int si = 0; si < E; ++si) {
        const int k = t + (si / RL) * TPL + (si % RL) * (M / RL);
        const T val[2] = {re[si], __shfl_sync(full, im[E - 1 - si], mate)};
        put(2 * k, val, two{});
      }
    } else {
      // z_k → outputs (i0, i1) = (4k, 4k+2) for k < M/2 and the odd (2n−1−4k, 2n−3−4k)
      // for k ≥ M/2 (negated for DD): the 4-vector at 4k (k < M/2) is
      // (z_k.x, ±z_{k'}.y, z_k.y, ±z_{k'}.x), k' = M−1−k
      const bool neg = (bc == BC_DD);
#pragma unroll
      for (int si = 0; si < E; ++si) {
        const int j = E - 1 - si;  // every lane hands its mirrored slot to its mate
        const T hy = __shfl_sync(full, v[j].y, mate), hx = __shfl_sync(full, v[j].x, mate);
        if ((si % RL) >= RL / 2) continue;
        const int k = t + (si / RL) * TPL + (si % RL) * (M / RL);
        const T val[4] = {v[si].x, neg ? -hy : hy, v[si].y, neg ? -hx : hx};
        put(4 * k, val, four{});
      }
    }
  }
}

}  // namespace row

namespace col {

template <class T, int M, int CW>  // CW: x columns per CTA
struct CShape {
  static constexpr bool W = sizeof(T) == 8;  // FP64: the wide stages of fast::Shape
  static constexpr int TPL = W ? fast::Shape<M, true>::TPL : (M >= 128) ? 32 : 16;  // threads per column
  static constexpr int E = M / TPL;                 // complex points per thread
  static constexpr int NT = CW * TPL;               // threads per CTA
  // resident CTAs: FP64 keeps 168 registers a thread (three CTAs of 128), FP32 64
  static constexpr int CTAS = !W ? 1024 / NT : (NT <= 384 ? 384 / NT : 1);
  static constexpr int NST = W ? fast::Shape<M, true>::NST : (M == 128) ? 4 : 3;
  // radix of stage s, a divisor of E
  __host__ __device__ static constexpr int radix(int s) {
    if (M == 512) return s == 0 ? 16 : (s == 1 ? 8 : 4);
    if (W) return fast::Shape<M, true>::radix(s);
    return (M == 256) ? (s < 2 ? 8 : 4)
         : (M == 128) ? (s < 3 ? 4 : 2)
         : 4;
  }
};

// Stages STAGE… of the M-point FFT of this thread's column. On entry
// v[q·R + r] = x[b_q + r·M/R] with b_q = b + q·TPL; on return v holds the last
// stage's outputs, v[q·R + r] at position b_q + r·(M/R_last).
template <class T, int M, int CW, bool INV, int STAGE, int NS>
__device__ __forceinline__ void fft_col(cplx<T> (&v)[CShape<T, M, CW>::E], cplx<T>* buf, const cplx<T>* stw,
                                        int b, int c) {
  using S = CShape<T, M, CW>;
  constexpr int E = S::E, TPL = S::TPL;
  constexpr int R = S::radix(STAGE);
#pragma unroll
  for (int q = 0; q < E / R; ++q) {
    const int bq = b + q * TPL;
    if constexpr (STAGE > 0) {
      const int k = bq & (NS - 1);
#pragma unroll
      for (int r = 1; r < R; ++r) {
        cplx<T> w = stw[(r * k * (M / (NS * R))) & (M - 1)];
        if (INV) w.y = -w.y;
        v[q * R + r] = cmul(v[q * R + r], w);
      }
    }
    fast::dftR<T, R, INV>(&v[q * R]);
  }
  if constexpr (STAGE + 1 < S::NST) {
    constexpr int R2 = S::radix(STAGE + 1);
    __syncthreads();  // earlier readers of buf are done
#pragma unroll
    for (int q = 0; q < E / R; ++q) {
      const int bq = b + q * TPL;
      const int o = (bq / NS) * NS * R + (bq & (NS - 1));
#pragma unroll
      for (int r = 0; r < R; ++r) buf[(o + r * NS) * CW + c] = v[q * R + r];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < E / R2; ++q) {
      const int bq = b + q * TPL;
#pragma unroll
      for (int r = 0; r < R2; ++r) v[q * R2 + r] = buf[(bq + r * (M / R2)) * CW + c];
    }
    fft_col<T, M, CW, INV, STAGE + 1, NS * R>(v, buf, stw, b, c);
  }
}

template <class T, int M, int CW>
__host__ __device__ constexpr size_t col_smem(int bc) {
  return fast_table_bytes<T, M>(bc) + (size_t)M * CW * sizeof(cplx<T>);
}

// One tile of the y transform: CW consecutive x columns of one z plane (tile g
// of the n_z·n_x/CW tiles, x fastest); tables and the exchange buffer in shared
// memory. Starts with a block barrier (tables ready, earlier buffer reads done).
template <class T, int M, bool FWD, int CW>
__device__ __forceinline__ void col_tile(const FastArgs<T>& a, const cplx<T>* stw, const cplx<T>* ptw,
                                         const cplx<T>* xtw, cplx<T>* buf, int g) {
  using S = CShape<T, M, CW>;
  constexpr int N = 2 * M, E = S::E, TPL = S::TPL;
  constexpr int RL = S::radix(S::NST - 1);
  const int bc = a.bc;
  const int c = threadIdx.x % CW;
  // PAIR: the half-warps of warp w are b = w and 32 − w (0 and 16 for w = 0), so that the
  // thread holding wavenumber k = b + 32·j and the one holding M − k = (32 − b) + 32·(E−1−j)
  // are lanes apart by 16, or the same thread (b = 0: slot E − j; b = 16: slot E − 1 − j): the
  // pairs of Table 2 meet by shuffle instead of through the buffer (forward and backward,
  // µs: 512×256×256 78 → 74 and 84 → 81, 512³ 250 → 233 and 296 → 290, 1024³ 1881 → 1835
  // forward; backward M = 512 holds too many values for it: 2277 → 2322, so it keeps the buffer).
  constexpr bool PAIR = TPL == 32 && CW == 16 && (FWD || M < 512);
  const int wi = threadIdx.x / 32, hb = (threadIdx.x / CW) & 1;
  const int b = !PAIR ? (int)threadIdx.x / CW : (hb == 0 ? wi : (wi == 0 ? 16 : 32 - wi));
  const T* in = static_cast<const T*>(a.in);  // may equal out (in-place y passes)
  T* out = static_cast<T*>(a.out);
  const int nx = a.nx, ny = a.ny;
  const int tpz = nx / CW;
  const int zb = g / tpz, x0 = (g - zb * tpz) * CW;
  // DN is the ND problem on the reversed line: the forward transform reads its input
  // rows from row n−1 downwards and runs the ND code unchanged; the backward one swaps
  // the two outputs of each wavenumber
  const bool rv = FWD && (bc == BC_DN);
  const int sstr = rv ? -nx : nx;
  const T* src = in + (size_t)zb * ny * nx + x0 + c + (rv ? (size_t)(N - 1) * nx : 0);
  T* dst = out + (size_t)zb * ny * nx + x0 + c;
  // row offsets fit in 32 bits (n_y·n_x ≤ 2^20)
  auto X = [&](int q) { return src[q * sstr]; };
  auto Y = [&](int q, T val) { dst[q * nx] = val; };
  const bool scaled = a.plane_scale != nullptr;
  const T s = scaled ? a.plane_scale[zb] : (T)1;
  const T h = split_scale<T, M, FWD>(bc);
  cplx<T> v[E];
  __syncthreads();  // tables ready; the previous tile's buffer reads are done
  if (FWD) {
    // ---- pre-processing gathered from the rows into the first-stage operands ----
#pragma unroll
    for (int r = 0; r < E; ++r) {
      const int p = b + r * TPL;
      cplx<T> z;
      if (bc == BC_P) {
        z = {X(2 * p), X(2 * p + 1)};
      } else if (bc_iv(bc)) {  // (DN: rows addressed in reverse, see above)
        z = cmul(cplx<T>{X(2 * p), X(N - 1 - 2 * p)}, xtw[p]);
      } else {
        const int j0 = 2 * p, j1 = 2 * p + 1;
        T v0 = X(j0 < M ? 2 * j0 : 2 * N - 1 - 2 * j0);
        T v1 = X(j1 < M ? 2 * j1 : 2 * N - 1 - 2 * j1);
        if (bc == BC_DD) {
          if (j0 >= M) v0 = -v0;
          if (j1 >= M) v1 = -v1;
        }
        z = {v0, v1};
      }
      v[r] = z;
    }
    if (scaled) {
#pragma unroll
      for (int r = 0; r < E; ++r) v[r] = cscale(v[r], s);
    }
    fft_col<T, M, CW, false, 0, 1>(v, buf, stw, b, c);
    // ---- post-processing: pairs (k, M − k), rows out ----
    const bool rev = (bc == BC_DD);
    auto OUTQ = [&](int q, T val) { Y(rev ? (N - 1 - q) : q, val); };
    auto pair_out = [&](int k, cplx<T> Zk, cplx<T> Zmk, bool self) {
      cplx<T> Vk, Vmk;
      if (self) {  // k = M/2 is its own partner
        Vk = Vmk = cscale(conj_(Zk), (T)2 * h);
      } else {
        const cplx<T> Ek = cadd(Zk, conj_(Zmk));
        const cplx<T> Ok = mul_mi(csub(Zk, conj_(Zmk)));
        const cplx<T> B = cmul(ptw[k], Ok);
        Vk = split_add(Ek, B, h);
        Vmk = conj_(split_sub(Ek, B, h));
      }
      if (bc == BC_P) {
        if (k == 0) {
          Y(0, Vk.x);
          Y(N - 1, Vmk.x);
        } else {
          Y(2 * k - 1, Vk.x);
          Y(2 * k, -Vk.y);
          if (2 * k != M) {
            Y(2 * (M - k) - 1, Vmk.x);
            Y(2 * (M - k), -Vmk.y);
          }
        }
      } else {
        if (k == 0) {
          OUTQ(0, Vk.x);
          OUTQ(M, (T)0.70710678118654752440 * Vmk.x);
        } else {
          const cplx<T> c1 = cmul(xtw[k], Vk);
          OUTQ(k, c1.x);
          OUTQ(N - k, -c1.y);
          if (2 * k != M) {
            const cplx<T> c2 = cmul(xtw[M - k], Vmk);
            OUTQ(M - k, c2.x);
            OUTQ(M + k, -c2.y);
          }
        }
      }
    };
    if constexpr (PAIR) {
      // slot si holds j = si / RL + (si % RL)·(M/RL/32)
      auto so = [](int j) { return (j % (E / RL)) * RL + j / (E / RL); };
      if (bc_iv(bc)) {
#pragma unroll
        for (int j = 0; j < E; ++j) {
          const int k = b + 32 * j;
          const cplx<T> cc = cmul(xtw[M + k], v[so(j)]);
          Y(2 * k, cc.x);
          Y(N - 1 - 2 * k, -cc.y);
        }
      } else {
#pragma unroll
        for (int j = 0; j < E / 2; ++j) {
          const cplx<T> Zk = v[so(j)], up = v[so(E - 1 - j)];
          cplx<T> Zmk = {__shfl_xor_sync(0xffffffffu, up.x, 16), __shfl_xor_sync(0xffffffffu, up.y, 16)};
          if (wi == 0) Zmk = hb ? up : (j == 0 ? Zk : v[so((E - j) % E)]);
          pair_out(b + 32 * j, Zk, Zmk, false);
        }
        if (b == 0) pair_out(M / 2, v[so(E / 2)], v[so(E / 2)], true);
      }
    } else {
      // through the buffer
      __syncthreads();
#pragma unroll
      for (int q = 0; q < E / RL; ++q)
#pragma unroll
        for (int r = 0; r < RL; ++r) buf[(b + q * TPL + r * (M / RL)) * CW + c] = v[q * RL + r];
      __syncthreads();
      if (bc_iv(bc)) {
#pragma unroll
        for (int i = 0; i < E; ++i) {
          const int k = b + i * TPL;
          const cplx<T> cc = cmul(xtw[M + k], buf[k * CW + c]);
          Y(2 * k, cc.x);
          Y(N - 1 - 2 * k, -cc.y);
        }
      } else {
        constexpr int NP = (M / 2) / TPL + 1;
#pragma unroll
        for (int i = 0; i < NP; ++i) {
          const int k = b + i * TPL;
          if (k > M / 2) break;
          const cplx<T> Zk = buf[k * CW + c], Zmk = buf[(k == 0 ? 0 : M - k) * CW + c];
          pair_out(k, Zk, Zmk, i == NP - 1);
        }
      }
    }
  } else {
    // ---- backward pre-processing from the rows into the first stage's operands ----
    if (bc_iv(bc)) {
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int k = b + i * TPL;
        const cplx<T> z = cmul(cplx<T>{X(2 * k), X(N - 1 - 2 * k)}, xtw[k]);
        if constexpr (PAIR) v[i] = z;
        else buf[k * CW + c] = z;
      }
    } else {
      // all row loads of the pairs first (they are independent), then the arithmetic
      constexpr int NP = (M / 2) / TPL;  // pairs (k, M − k) of a thread; k = M/2, its own partner, is b = 0's
      const bool rev = (bc == BC_DD);
      T xv[NP][4], xs[2] = {(T)0, (T)0};
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const int k = b + i * TPL;
        int q[4];
        bool use[4] = {true, true, true, true};
        if (bc == BC_P) {
          q[0] = k == 0 ? 0 : 2 * k - 1;
          q[1] = 2 * k;
          q[2] = k == 0 ? N - 1 : 2 * (M - k) - 1;
          q[3] = 2 * (M - k);
          use[1] = use[3] = k != 0;
        } else {
          const int qq[4] = {k, N - k, M - k, N - M + k};
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            q[u] = rev ? (N - 1 - qq[u]) : qq[u];
            use[u] = qq[u] < N;
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) xv[i][u] = use[u] ? X(q[u]) : (T)0;
      }
      if (b == 0) {
        xs[0] = X(bc == BC_P ? M - 1 : (rev ? N - 1 - M / 2 : M / 2));
        xs[1] = X(bc == BC_P ? M : (rev ? M / 2 - 1 : N - M / 2));
      }
      auto V = [&](int k, T x0, T x1) {
        if (bc == BC_P) return cplx<T>{x0, -x1};
        cplx<T> w = xtw[k];
        w.y = -w.y;
        return cmul(w, cplx<T>{x0, -x1});
      };
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const int k = b + i * TPL;
        const cplx<T> Vk = V(k, xv[i][0], xv[i][1]), Vm = V(M - k, xv[i][2], xv[i][3]);
        const cplx<T> Ek = cadd(Vk, conj_(Vm));
        cplx<T> wn = ptw[k];
        wn.y = -wn.y;
        const cplx<T> Ok = cmul(csub(Vk, conj_(Vm)), wn);
        const cplx<T> zk = split_add(Ek, mul_i(Ok), h), zm = split_add(conj_(Ek), mul_i(conj_(Ok)), h);
        if constexpr (PAIR) {
          v[i] = zk;
          v[E - 1 - i] = zm;  // the partner's slot, exchanged below
        } else {
          buf[k * CW + c] = zk;
          if (k != 0) buf[(M - k) * CW + c] = zm;
        }
      }
      const cplx<T> zh = cscale(conj_(V(M / 2, xs[0], xs[1])), (T)2 * h);  // (b = 0)
      if constexpr (PAIR) {
        if (wi != 0) {
#pragma unroll
          for (int i = E / 2; i < E; ++i)
            v[i] = {__shfl_xor_sync(0xffffffffu, v[i].x, 16), __shfl_xor_sync(0xffffffffu, v[i].y, 16)};
        } else if (hb == 0) {  // own slots: M − k of slot i is slot E − i
#pragma unroll
          for (int i = E - 1; i > E / 2; --i) v[i] = v[i - 1];
          v[E / 2] = zh;
        }
      } else if (b == 0) {
        buf[(M / 2) * CW + c] = zh;
      }
    }
    if constexpr (!PAIR) {
      __syncthreads();
#pragma unroll
      for (int r = 0; r < E; ++r) v[r] = buf[(b + r * TPL) * CW + c];
    }
    if (bc_iv(bc)) fft_col<T, M, CW, false, 0, 1>(v, buf, stw, b, c);
    else fft_col<T, M, CW, true, 0, 1>(v, buf, stw, b, c);
    // ---- backward post-processing straight from the last stage to the rows ----
    if (scaled) {
#pragma unroll
      for (int r = 0; r < E; ++r) v[r] = cscale(v[r], s);
    }
#pragma unroll
    for (int q = 0; q < E / RL; ++q) {
#pragma unroll
      for (int r = 0; r < RL; ++r) {
        const int k = b + q * TPL + r * (M / RL);
        const cplx<T> zk = v[q * RL + r];
        if (bc_iv(bc)) {
          const cplx<T> cc = cmul(xtw[M + k], zk);
          const T A = cc.x, B = -cc.y;
          if (bc == BC_DN) {
            Y(2 * k, B);
            Y(N - 1 - 2 * k, A);
          } else {
            Y(2 * k, A);
            Y(N - 1 - 2 * k, B);
          }
        } else if (bc == BC_P) {
          Y(2 * k, zk.x);
          Y(2 * k + 1, zk.y);
        } else {
          const int j0 = 2 * k, j1 = 2 * k + 1;
          const int i0 = j0 < M ? 2 * j0 : 2 * N - 1 - 2 * j0;
          const int i1 = j1 < M ? 2 * j1 : 2 * N - 1 - 2 * j1;
          T v0 = zk.x, v1 = zk.y;
          if (bc == BC_DD) {
            if (i0 & 1) v0 = -v0;
            if (i1 & 1) v1 = -v1;
          }
          Y(i0, v0);
          Y(i1, v1);
        }
      }
    }
  }
}

}  // namespace col

}  // namespace ps
