// xform_fast.cuh — register-resident line transforms for n = 2M with M ∈ {64, 128, 256, 512}.
//
// Same mathematics as xform.cu (one M-point complex FFT per line of n reals
// with the Table 2 pre/post processing per BC), organised for throughput:
//   * TPL = M/E threads own one line, E complex points each (E = 16, 8, 4),
//     so a line lives in one warp (or a fraction of one) and stages synchronise
//     with __syncwarp only;
//   * Stockham stages of radix R | E; each thread does E/R butterflies per
//     stage with its operands in registers, exchanging through the line's own
//     shared-memory buffer between stages;
//   * all index arithmetic is compile-time (M is a template parameter);
//   * twiddles come from shared-memory tables loaded once per CTA; the grid is
//     persistent (CTAs stride over line groups);
//   * lines are staged through shared memory with 16-byte global accesses
//     (x: contiguous rows; y: a tile of LPC consecutive x columns, so every row
//     segment is LPC·sizeof(T) ≥ 64 bytes).
#pragma once
#include "internal.h"

namespace ps {
namespace fast {

// W: wide stages, for the FP64 lines of xform_row.cu. The FP64 pipe bounds them (504 G
// instructions/s), so they take the radices with the least arithmetic (a point of M = 128:
// 16·8 19.5 instructions, 4·4·4·2 22) and as few threads a line as those need. 256³ (DD, ND):
// x passes 600 and 620 → 510 and 540 µs, y passes 510 → 459 (27.5 instructions a point at
// the pipe's rate: 458).
template <int M, bool W = false>
struct Shape {
  static constexpr int E = W ? (M >= 128 ? 16 : 8) : (M >= 512) ? 16 : (M >= 256 ? 8 : 4);  // points per thread
  static constexpr int TPL = M / E;                                                           // threads per line
  // radix of stage s (all divide E); stages multiply to M
  static constexpr int NST = M == 512 ? 3 : W ? 2 : (M == 128 ? 4 : 3);
  __host__ __device__ static constexpr int radix(int s) {
    if (W) return (M == 256 || (M == 128 && s == 0)) ? 16 : 8;
    return (M == 512) ? 8 : (M == 256 ? (s < 2 ? 8 : 4) : (M == 128 ? (s < 3 ? 4 : 2) : 4));
  }
};

// Skewed index of the complex exchange buffer: one pad slot per 8 entries turns
// the stride-8 (64-byte) writes of a radix-8 stage into conflict-free ones.
__device__ __forceinline__ int cpad(int i) { return i + (i >> 3); }

template <class T, bool INV>
__device__ __forceinline__ void dft2(cplx<T>& a, cplx<T>& b) {
  cplx<T> t = a;
  a = cadd(t, b);
  b = csub(t, b);
}

template <class T, bool INV>
__device__ __forceinline__ void dft4(cplx<T>* v) {
  cplx<T> t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
  cplx<T> t2 = cadd(v[1], v[3]), t3 = csub(v[1], v[3]);
  t3 = INV ? mul_i(t3) : mul_mi(t3);
  v[0] = cadd(t0, t2);
  v[2] = csub(t0, t2);
  v[1] = cadd(t1, t3);
  v[3] = csub(t1, t3);
}

// dft4 of (v0, v1·h13, v2·h2, v3·h13): real factors ride in fused multiply-adds.
template <class T, bool INV>
__device__ __forceinline__ void dft4h(cplx<T>* v, T h2, T h13) {
  auto madd = [](T h, cplx<T> a, cplx<T> b) { return cplx<T>{fma(h, a.x, b.x), fma(h, a.y, b.y)}; };
  const cplx<T> t0 = madd(h2, v[2], v[0]), t1 = madd(-h2, v[2], v[0]);
  const cplx<T> t2 = cadd(v[1], v[3]);
  cplx<T> t3 = csub(v[1], v[3]);
  t3 = INV ? mul_i(t3) : mul_mi(t3);
  v[0] = madd(h13, t2, t0);
  v[2] = madd(-h13, t2, t0);
  v[1] = madd(h13, t3, t1);
  v[3] = madd(-h13, t3, t1);
}
// √2·W8·z and √2·W8³·z (forward e^{−2πi/8}, inverse conjugate): the factor 1/√2 is left to dft4h
template <class T, bool INV>
__device__ __forceinline__ cplx<T> rot1(cplx<T> z) {
  return INV ? cplx<T>{z.x - z.y, z.x + z.y} : cplx<T>{z.x + z.y, z.y - z.x};
}
template <class T, bool INV>
__device__ __forceinline__ cplx<T> rot3(cplx<T> z) {
  return INV ? cplx<T>{-(z.x + z.y), z.x - z.y} : cplx<T>{z.y - z.x, -(z.x + z.y)};
}

template <class T, bool INV>
__device__ __forceinline__ void dft8(cplx<T>* v) {
  // radix-2 over (r, r+4), twiddle by W8^r, then two radix-4 on evens/odds
  const T h = (T)0.70710678118654752440;
  cplx<T> a[4], b[4];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    a[r] = cadd(v[r], v[r + 4]);
    b[r] = csub(v[r], v[r + 4]);
  }
  b[1] = rot1<T, INV>(b[1]);
  b[2] = INV ? mul_i(b[2]) : mul_mi(b[2]);
  b[3] = rot3<T, INV>(b[3]);
  dft4<T, INV>(a);
  dft4h<T, INV>(b, (T)1, h);
  // outputs: X[2k] = A[k], X[2k+1] = B[k]
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    v[2 * k] = a[k];
    v[2 * k + 1] = b[k];
  }
}

// 16-point DFT in natural order, as 4 × 4: X[k1 + 4k2] =
// Σ_{n2} W4^{n2·k2} · W16^{n2·k1} · Σ_{n1} x[n2 + 4n1] · W4^{n1·k1}.
template <class T, bool INV>
__device__ __forceinline__ void dft16(cplx<T>* v) {
  const T c1 = (T)0.92387953251128675613, s1 = (T)0.38268343236508977173;  // cos, sin of π/8
  const T h = (T)0.70710678118654752440;
  cplx<T> a[4][4];
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < 4; ++n1) a[n2][n1] = v[n2 + 4 * n1];
    dft4<T, INV>(a[n2]);
  }
  // W16^m = (cos 2πm/16, −sin 2πm/16) for the forward transform, conjugate for the inverse
  auto tw = [&](cplx<T> z, T wr, T wi) {
    if (INV) wi = -wi;
    return cplx<T>{z.x * wr - z.y * wi, z.x * wi + z.y * wr};
  };
  a[1][1] = tw(a[1][1], c1, -s1);        // m = 1
  a[1][2] = rot1<T, INV>(a[1][2]);       // m = 2, without 1/√2
  a[1][3] = tw(a[1][3], s1, -c1);        // m = 3
  a[2][1] = rot1<T, INV>(a[2][1]);       // m = 2, without 1/√2
  a[2][2] = INV ? mul_i(a[2][2]) : mul_mi(a[2][2]);  // m = 4
  a[2][3] = rot3<T, INV>(a[2][3]);       // m = 6, without 1/√2
  a[3][1] = tw(a[3][1], s1, -c1);        // m = 3
  a[3][2] = rot3<T, INV>(a[3][2]);       // m = 6, without 1/√2
  a[3][3] = tw(a[3][3], -c1, s1);        // m = 9
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    cplx<T> b[4] = {a[0][k1], a[1][k1], a[2][k1], a[3][k1]};
    dft4h<T, INV>(b, (k1 & 1) ? h : (T)1, k1 == 2 ? h : (T)1);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) v[k1 + 4 * k2] = b[k2];
  }
}

template <class T, int R, bool INV>
__device__ __forceinline__ void dftR(cplx<T>* v) {
  if constexpr (R == 2) dft2<T, INV>(v[0], v[1]);
  if constexpr (R == 4) dft4<T, INV>(v);
  if constexpr (R == 8) dft8<T, INV>(v);
  if constexpr (R == 16) dft16<T, INV>(v);
}

// Stages STAGE… of the M-point FFT of one line. On entry v holds this stage's
// inputs in (butterfly q, element r) order: v[q*R + r] = x[b_q + r*M/R] with
// b_q = t + q*TPL. On return v holds the last stage's outputs, v[q*R + r] at
// position b_q + r*(M/R_last). buf is the line's M-complex shared buffer.
template <class T, int M, bool INV, int STAGE, int NS, bool W = false>
__device__ __forceinline__ void fft_stages(cplx<T> (&v)[Shape<M, W>::E], cplx<T>* buf,
                                           const cplx<T>* stw, int t) {
  using S = Shape<M, W>;
  constexpr int E = S::E, TPL = S::TPL;
  constexpr int R = S::radix(STAGE);
#pragma unroll
  for (int q = 0; q < E / R; ++q) {
    const int b = t + q * TPL;
    if constexpr (STAGE > 0) {
      const int k = b & (NS - 1);
#pragma unroll
      for (int r = 1; r < R; ++r) {
        cplx<T> w = stw[(r * k * (M / (NS * R))) & (M - 1)];
        if (INV) w.y = -w.y;
        v[q * R + r] = cmul(v[q * R + r], w);
      }
    }
    dftR<T, R, INV>(&v[q * R]);
  }
  if constexpr (STAGE + 1 < S::NST) {
    constexpr int R2 = S::radix(STAGE + 1);
    __syncwarp();
#pragma unroll
    for (int q = 0; q < E / R; ++q) {
      const int b = t + q * TPL;
      const int o = (b / NS) * NS * R + (b & (NS - 1));
#pragma unroll
      for (int r = 0; r < R; ++r) buf[cpad(o + r * NS)] = v[q * R + r];
    }
    __syncwarp();
#pragma unroll
    for (int q = 0; q < E / R2; ++q) {
      const int b = t + q * TPL;
#pragma unroll
      for (int r = 0; r < R2; ++r) v[q * R2 + r] = buf[cpad(b + r * (M / R2))];
    }
    fft_stages<T, M, INV, STAGE + 1, NS * R, W>(v, buf, stw, t);
  }
}

}  // namespace fast

// Bytes of the twiddle tables for a given BC (16-byte aligned): ω_M^t (M), the
// real-FFT split factors (M + 1) and, except for P, the BC factors (≤ 2M).
template <class T, int M>
__host__ __device__ constexpr size_t fast_table_bytes(int bc) {
  return ((size_t)(2 * M + 1 + (bc == 0 ? 0 : 2 * M + 1)) * sizeof(cplx<T>) + 15) / 16 * 16;
}

template <class T>
struct FastArgs {
  const void* in;
  void* out;
  int axis, nx, ny, nz, bc;
  int nlines;           // x: ny*nz rows; y: nx*nz columns
  const cplx<T>* tw;    // 8n-entry table, e^{−2πi t/(8n)}
  const T* plane_scale;
  int accumulate;
  const int* skip;
  unsigned long long* amax;  // FP64 output: atomicMax of |transform output| bit patterns, or null
  int lpc;              // lines per CTA
  float* out2;          // FP64 output (x lines): also store the FP32 transform output here, or null
  const float* base32;  // FP64 output (x lines): out = widen(base32) + v instead of (out +) v, or null
};

template <class T, class TI, class TO, int M, bool FWD>
cudaError_t launch_xform_fast(FastArgs<T> a, cudaStream_t st);

// x-axis lines read and written by their own warp (xform_row.cu): nx = 2M.
template <class T, class TI, class TO, int M, bool FWD>
cudaError_t launch_xform_row(FastArgs<T> a, cudaStream_t st);

// y-axis lines with the columns on lanes (xform_col.cu): ny = 2M, nx a multiple
// of 16, TI = TO = T, no accumulation and no FP64 max tracking.
template <class T, int M, bool FWD>
cudaError_t launch_xform_col(FastArgs<T> a, cudaStream_t st);

// Lines of n = 2M contiguous reals with M ∈ {1024, 2048, 4096}, one CTA per line
// (xform_long.cu): a.nlines lines, line ln in plane ln / a.ny; x-row output modes.
template <class T, class TI, class TO, int M, bool FWD>
cudaError_t launch_xform_long(FastArgs<T> a, cudaStream_t st);

// dst[z][c][r] = src[z][r][c] for every plane z < nz (rows × cols per plane).
template <class T>
cudaError_t launch_plane_transpose(const T* src, T* dst, int rows, int cols, int nz, const int* skip,
                                   cudaStream_t st);

}  // namespace ps
