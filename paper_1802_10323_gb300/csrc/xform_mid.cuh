// xform_mid.cuh — the generic line transform (xform_dev.cuh) with the line length at compile
// time, FP32, for the half lengths m = 2^a·3^b ≤ 486 that have no power-of-two kernel.
//
// Same slots, tables and steps as xform_group. With m known, the index arithmetic that took
// most of that kernel's issue slots (107–126 instructions a value) folds away, and the tile
// goes through registers where it can:
//   * one shared buffer: every thread reads all its butterflies of a stage (at most 24 complex
//     values) before any thread writes the next stage's inputs, so that a 16-line tile of a
//     line of 972 takes 66 KB and the shorter ones leave room for four or more CTAs per SM;
//   * y lines: the first stage's operands come straight from the rows, and the last stage's
//     results go straight to them where no pairing is needed (DCT-IV; every backward output);
//   * radices 12, 18 (prime-factor maps, no inner twiddles) so that two stages reach m = 324.
// What bounds it: load latency at 50 % of the resident warps (registers), then issue (50–90
// instructions a value, against 107–126 with run-time lengths). Figures beside the dispatch
// (xform.cu).
#pragma once
#include "xform_dev.cuh"

namespace ps {
namespace mid {

// 12 = 4 × 3: x[(3·n1 + 4·n2) mod 12] → X[(9·k1 + 4·k2) mod 12] (k ≡ k1 mod 4, k ≡ k2 mod 3)
template <class T>
__device__ __forceinline__ void dft12(cplx<T>* v) {
  cplx<T> a[3][4];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
#pragma unroll
    for (int r = 0; r < 4; ++r) a[q][r] = v[(3 * r + 4 * q) % 12];
    fast::dft4<T, false>(a[q]);
  }
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    cplx<T> b[3] = {a[0][k1], a[1][k1], a[2][k1]};
    dft3(b);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) v[(9 * k1 + 4 * k2) % 12] = b[k2];
  }
}
// 18 = 2 × 9: x[(9·n1 + 2·n2) mod 18] → X[k], k ≡ k1 mod 2, k ≡ k2 mod 9
template <class T>
__device__ __forceinline__ void dft18(cplx<T>* v) {
  cplx<T> a[2][9];
#pragma unroll
  for (int r = 0; r < 2; ++r) {
#pragma unroll
    for (int q = 0; q < 9; ++q) a[r][q] = v[(9 * r + 2 * q) % 18];
    dft9(a[r]);
  }
#pragma unroll
  for (int k2 = 0; k2 < 9; ++k2) {
    v[(10 * k2) % 18] = cadd(a[0][k2], a[1][k2]);
    v[(9 + 10 * k2) % 18] = csub(a[0][k2], a[1][k2]);
  }
}
template <class T, int R>
__device__ __forceinline__ void dft(cplx<T>* v) {
  if constexpr (R == 3) dft3(v);
  else if constexpr (R == 6) dft6(v);
  else if constexpr (R == 9) dft9(v);
  else if constexpr (R == 12) dft12(v);
  else if constexpr (R == 18) dft18(v);
  else fast::dftR<T, R, false>(v);
}

// Lines, threads and radices per half length. Threads: the butterflies of a stage in whole
// rounds (or nearly), at most 24 complex values a thread.
template <int M>
struct Mid;
#define PS_MID_SHAPE(M_, LG_, NT_, R0_, R1_, R2_)                                                   \
  template <>                                                                                        \
  struct Mid<M_> {                                                                                   \
    static constexpr int LG = LG_, NT = NT_, NST = (R2_ > 1) ? 3 : 2;                                \
    __host__ __device__ static constexpr int radix(int s) { return s == 0 ? R0_ : (s == 1 ? R1_ : R2_); } \
    static_assert((R0_) * (R1_) * (R2_) == M_, "radices");                                           \
  };
PS_MID_SHAPE(16, 5, 128, 4, 4, 1)
PS_MID_SHAPE(18, 5, 96, 6, 3, 1)
PS_MID_SHAPE(24, 5, 96, 8, 3, 1)
PS_MID_SHAPE(27, 5, 96, 9, 3, 1)
PS_MID_SHAPE(32, 5, 128, 8, 4, 1)
PS_MID_SHAPE(36, 5, 192, 6, 6, 1)
PS_MID_SHAPE(48, 4, 128, 8, 6, 1)
PS_MID_SHAPE(54, 4, 160, 9, 6, 1)
PS_MID_SHAPE(72, 4, 160, 9, 8, 1)
PS_MID_SHAPE(81, 4, 160, 9, 9, 1)
PS_MID_SHAPE(96, 4, 192, 12, 8, 1)
PS_MID_SHAPE(108, 4, 192, 12, 9, 1)
PS_MID_SHAPE(144, 4, 192, 12, 12, 1)
PS_MID_SHAPE(162, 4, 160, 18, 9, 1)
PS_MID_SHAPE(192, 4, 256, 16, 12, 1)
PS_MID_SHAPE(216, 4, 288, 18, 12, 1)
PS_MID_SHAPE(243, 4, 448, 9, 9, 3)
PS_MID_SHAPE(288, 4, 288, 18, 16, 1)
PS_MID_SHAPE(324, 4, 288, 18, 18, 1)
PS_MID_SHAPE(384, 4, 384, 8, 8, 6)
PS_MID_SHAPE(432, 4, 448, 9, 8, 6)
PS_MID_SHAPE(486, 4, 448, 9, 9, 6)

template <int M>
struct DimCt {
  static constexpr int L = 1 << Mid<M>::LG, LS = L + 1;
  __host__ __device__ static constexpr int n() { return 2 * M; }
  __host__ __device__ static constexpr int m() { return M; }
  __host__ __device__ static constexpr int lg() { return Mid<M>::LG; }
  __host__ __device__ static constexpr int ls() { return LS; }
  __device__ __forceinline__ int div_m(int i) const { return i / M; }
  __device__ __forceinline__ int div_h(int i) const { return i / M; }
};
template <int M>
__host__ __device__ constexpr size_t mid_smem() {
  return ((size_t)M * DimCt<M>::LS + M) * sizeof(cplx<float>);
}
// resident CTAs asked for: about 64 registers a thread (radix 18: 80)
template <int M>
__host__ __device__ constexpr int mid_ctas() {
  const int by_regs = 65536 / ((Mid<M>::radix(0) > 16 ? 80 : 64) * Mid<M>::NT), by_smem = (int)((227 * 1024) / (mid_smem<M>() + 1024));
  const int r = by_regs < by_smem ? by_regs : by_smem;
  return r < 1 ? 1 : (r > 8 ? 8 : r);
}

// Stages S… of the FFT. ld(p, l): input slot p of the first one; st(p, l, v): results of the
// last one; in between through buf. ld_buf / st_buf: whether they read and write buf (the
// barriers that this takes). Ends with a barrier if st_buf.
template <int M, int S, int NS, bool LD_BUF, bool ST_BUF, class Ld, class St>
__device__ __forceinline__ void stages(cplx<float>* buf, const cplx<float>* sw, Ld&& ld, St&& st) {
  using C = Mid<M>;
  using D = DimCt<M>;
  constexpr int R = C::radix(S), NT = C::NT, L = D::L, LS = D::LS, nb = M / R, NBF = nb * L;
  constexpr int NB = (NBF + NT - 1) / NT;
  constexpr bool LAST = S + 1 == C::NST;
  cplx<float> v[NB][R];
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int idx = threadIdx.x + q * NT;
    if (NB * NT == NBF || idx < NBF) {
      const int l = idx & (L - 1), j = idx >> D::lg();
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if constexpr (S == 0) v[q][r] = ld(j + r * nb, l);
        else v[q][r] = buf[(j + r * nb) * LS + l];
      }
    }
  }
  // every read of buf is done before it is written (a last stage that writes elsewhere needs none)
  if constexpr ((S > 0 || LD_BUF) && (!LAST || ST_BUF)) __syncthreads();
#pragma unroll
  for (int q = 0; q < NB; ++q) {
    const int idx = threadIdx.x + q * NT;
    if (NB * NT == NBF || idx < NBF) {
      const int l = idx & (L - 1), j = idx >> D::lg();
      const int k = j % NS, o = (j / NS) * NS * R + k;
      if constexpr (NS > 1) {
#pragma unroll
        for (int r = 1; r < R; ++r) v[q][r] = cmul(v[q][r], sw[r * k * (M / (NS * R))]);
      }
      dft<float, R>(v[q]);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if constexpr (LAST) st(o + r * NS, l, v[q][r]);
        else buf[(o + r * NS) * LS + l] = v[q][r];
      }
    }
  }
  if constexpr (!LAST || ST_BUF) __syncthreads();
  if constexpr (!LAST) stages<M, S + 1, NS * R, true, ST_BUF>(buf, sw, ld, st);
}

template <class TI, int M, int AXIS>
__device__ __forceinline__ void prefetch_tile(const XformArgs<float>& a, int g) {
  constexpr int n = 2 * M, L = DimCt<M>::L, NT = Mid<M>::NT;
  if constexpr (AXIS == 0) {
    const int live = min(L, a.nlines - g * L);
    const char* p = reinterpret_cast<const char*>(static_cast<const TI*>(a.in) + (size_t)g * L * n);
    const int bytes = live * n * (int)sizeof(TI);
    for (int o = threadIdx.x * 128; o < bytes; o += NT * 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + o));
  } else {
    const int gpz = (a.nx + L - 1) / L, zb = g / gpz, x0 = (g - zb * gpz) * L;
    const TI* p = static_cast<const TI*>(a.in) + (size_t)zb * n * a.nx + x0;
    for (int e = threadIdx.x; e < n; e += NT) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + e * a.nx));
  }
}

// One tile: L rows (AXIS 0) or L columns of a plane (AXIS 1).
template <class TI, class TO, int M, int AXIS, bool FWD>
__device__ __forceinline__ void tile(const XformArgs<float>& a, int grp, cplx<float>* buf, const cplx<float>* sw) {
  using T = float;
  using D = DimCt<M>;
  constexpr int n = 2 * M, L = D::L, LS = D::LS;
  const D dim{};
  const cplx<T>* t0 = a.tab.t0[FWD];
  const cplx<T>* t1 = a.tab.t1[FWD];
  const TI* in = static_cast<const TI*>(a.in);
  TO* out = static_cast<TO*>(a.out);
  const int nx = a.nx, ny = a.ny, bc = a.bc;
  const bool iv = bc_iv(bc);
  auto from_buf = [&](int p, int l) { return buf[p * LS + l]; };
  auto to_buf = [&](int p, int l, cplx<T> z) { buf[p * LS + l] = z; };
  if constexpr (AXIS == 0) {
    const size_t base = (size_t)grp * L * n;
    const int live = min(L, a.nlines - grp * L);
    auto scale_of = [&](int l) { return a.plane_scale[(grp * L + l) / ny]; };
    T* rb = reinterpret_cast<T*>(buf);
    x_load<D, T, TI, FWD>(dim, bc, in + base, live, rb, FWD && a.plane_scale, scale_of);
    __syncthreads();
    if (iv) {
      stages<M, 0, 1, true, true>(buf, sw, [&](int p, int l) { return cmul(buf[p * LS + l], ldg_c(t0 + p)); },
                                  [&](int p, int l, cplx<T> z) {
                                    const cplx<T> c = cmul(ldg_c(t1 + p), z);
                                    buf[p * LS + l] = {c.x, -c.y};
                                  });
    } else {
      if constexpr (!FWD) {
        pairs_bwd(dim, bc, buf, t0, t1, a.tab.inv2m, from_buf);
        __syncthreads();
      }
      stages<M, 0, 1, true, true>(buf, sw, from_buf, to_buf);
      if constexpr (FWD) {
        pairs_fwd(dim, bc, buf, t0, t1, [&](int k, int l, T v0, T v1) { buf[k * LS + l] = {v0, v1}; });
        __syncthreads();
      }
    }
    T tmax = 0.f;
    x_store<D, T, TO, FWD>(dim, a, out, base, live, rb, (!FWD && !iv) ? 1 : 0, false, !FWD && a.plane_scale, scale_of,
                           tmax);
    if constexpr (sizeof(TO) == 8) amax_out(a.amax, tmax);
  } else {
    const int gpz = (nx + L - 1) / L;
    const int zb = grp / gpz, x0 = (grp - zb * gpz) * L;
    const int live = min(L, nx - x0);
    const TI* src = in + (size_t)zb * ny * nx + x0;  // row offsets fit in 32 bits
    TO* dst = out + (size_t)zb * ny * nx + x0;
    const T sc = a.plane_scale ? a.plane_scale[zb] : 1.f;
    // columns beyond the plane's last take its values and are not stored
    auto at = [&](int e, int l) { return src[e * nx + min(l, live - 1)]; };
    auto store2 = [&](int e0, int e1, int l, T v0, T v1) {
      if (l < live) {
        dst[e0 * nx + l] = v0;
        dst[e1 * nx + l] = v1;
      }
    };
    by_kind(bc, [&](auto kind) {
      constexpr int KIND = decltype(kind)::value;
      const SlotMap<D, KIND> map{dim, bc};
      auto rows_in = [&](int p, int l) {  // the two values of slot p
        int e0, e1;
        if (FWD) map.phys(p, e0, e1);
        else map.spec(p, e0, e1);
        cplx<T> z = {at(e0, l), at(e1, l)};
        if constexpr (FWD) {
          z = cscale(z, sc);
          if (KIND == KIND_CT && bc == BC_DD) {  // Makhoul's order: odd elements from j ≥ m
            if (e0 & 1) z.x = -z.x;
            if (e1 & 1) z.y = -z.y;
          }
        }
        return z;
      };
      auto rows_out = [&](int k, int l, T v0, T v1) {
        int e0, e1;
        if (FWD) map.spec(k, e0, e1);
        else map.phys(k, e0, e1);
        if constexpr (!FWD) {
          v0 *= sc;
          v1 *= sc;
          if (KIND == KIND_CT && bc == BC_DD) {
            if (e0 & 1) v0 = -v0;
            if (e1 & 1) v1 = -v1;
          }
        }
        store2(e0, e1, l, v0, v1);
      };
      if constexpr (KIND == KIND_IV) {  // both ends straight from and to the rows
        stages<M, 0, 1, false, false>(buf, sw, [&](int p, int l) { return cmul(rows_in(p, l), ldg_c(t0 + p)); },
                                      [&](int p, int l, cplx<T> z) {
                                        const cplx<T> c = cmul(ldg_c(t1 + p), z);
                                        rows_out(p, l, c.x, -c.y);
                                      });
      } else if constexpr (FWD) {
        stages<M, 0, 1, false, true>(buf, sw, rows_in, to_buf);
        pairs_fwd(dim, bc, buf, t0, t1, rows_out);
      } else {
        pairs_bwd(dim, bc, buf, t0, t1, a.tab.inv2m, rows_in);
        __syncthreads();
        stages<M, 0, 1, true, false>(buf, sw, from_buf, [&](int p, int l, cplx<T> z) { rows_out(p, l, z.y, z.x); });
      }
    });
  }
}

template <class TI, class TO, int M, int AXIS, bool FWD>
__global__ void __launch_bounds__(Mid<M>::NT, mid_ctas<M>()) xform_mid_kernel(XformArgs<float> a, int ngroups) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<float>* sw = reinterpret_cast<cplx<float>*>(smem_raw);
  cplx<float>* buf = sw + M;
  for (int i = threadIdx.x; i < M; i += Mid<M>::NT) sw[i] = ldg_c(a.tab.w + i);
  pdl_wait();
  if (a.skip && *a.skip) return;
  for (int g = blockIdx.x; g < ngroups; g += gridDim.x) {
    // ask L2 for this CTA's next tile, whose loads then do not wait on HBM
    if (g + (int)gridDim.x < ngroups) prefetch_tile<TI, M, AXIS>(a, g + gridDim.x);
    __syncthreads();  // tables ready; the previous tile's reads of buf are done
    tile<TI, TO, M, AXIS, FWD>(a, g, buf, sw);
  }
}

template <class TI, class TO, int M, int AXIS, bool FWD>
cudaError_t launch_mid(const XformArgs<float>& a, int ngroups, cudaStream_t st) {
  auto k = xform_mid_kernel<TI, TO, M, AXIS, FWD>;
  constexpr size_t smem = mid_smem<M>();
  static int bps = 0;
  if (bps == 0) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    int b = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k, Mid<M>::NT, smem);
    if (e != cudaSuccess) return e;
    bps = b < 1 ? 1 : b;
  }
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = ngroups < sms * bps ? ngroups : sms * bps;
  return launch_k(k, grid, Mid<M>::NT, smem, st, a, ngroups);
}

}  // namespace mid

// One translation unit per group of lengths (xform_mid_*.cu) defines these.
template <class TI, class TO, int M, int AXIS, bool FWD>
cudaError_t launch_xform_mid(const XformArgs<float>& a, int ngroups, cudaStream_t st);

#define PS_MID_INST1(TI, TO, M, AXIS, FWD)                                                              \
  template <>                                                                                           \
  cudaError_t launch_xform_mid<TI, TO, M, AXIS, FWD>(const XformArgs<float>& a, int ng, cudaStream_t st) { \
    return mid::launch_mid<TI, TO, M, AXIS, FWD>(a, ng, st);                                            \
  }
#define PS_MID_INST(M)                       \
  PS_MID_INST1(float, float, M, 0, true)     \
  PS_MID_INST1(double, float, M, 0, true)    \
  PS_MID_INST1(float, float, M, 0, false)    \
  PS_MID_INST1(float, double, M, 0, false)   \
  PS_MID_INST1(float, float, M, 1, true)     \
  PS_MID_INST1(float, float, M, 1, false)

}  // namespace ps
