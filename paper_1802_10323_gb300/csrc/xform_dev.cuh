// xform_dev.cuh — device code of the generic line transforms (Table 2) along x or y.
//
// Every transform of length n (even) is reduced to one complex FFT of length
// m = n/2 done in shared memory (Stockham, radices 16, 9, 8, 6, 4, 3, 2), with
// BC-specific pre- and post-processing:
//   P   (DFT, half-complex layout): z_p = a_2p + i a_2p+1, then the standard
//        even/odd split X_k = E_k + e^{−2πik/n} O_k.
//   NN  (DCT-II / DCT-III): Makhoul's reordering v_j = a_2j, v_{n−1−j} = a_2j+1,
//        a real DFT of v, then X_q = 2 Re(e^{−iπq/2n} V_q).
//   DD  (DST-II / DST-III): DST-II(a)_q = DCT-II((−1)^p a_p)_{n−1−q}.
//   ND  (DCT-IV): u_r = (a_2r + i a_{n−1−2r}) e^{−iπr/n}, U = FFT_m(u),
//        X_2k = 2 Re(c_k), X_{n−1−2k} = −2 Im(c_k), c_k = e^{−iπ(4k+1)/4n} U_k;
//        DCT-IV is its own inverse up to 2n.
//   FD  (x/y face unknowns, DST-I of the interior, the wall entry copied): the odd
//        extension y of length 2n (y_0 = y_n = 0, y_t = a_t, y_{2n−t} = −a_t) is a
//        real sequence whose DFT is Y_k = −2i Σ_t a_t sin(πtk/n); it is done as an
//        FFT of m = n complex points z_j = y_2j + i y_2j+1 and the real-DFT split
//        Y_k = E_k + e^{−iπk/n} O_k, giving X_k = −Im(Y_k). DST-I is its own inverse
//        up to 2n, so the backward transform is the same with the factor 1/(2n).
// Backward transforms include Table 1's normalisation (1/n or 1/2n). Their inverse
// FFT is the forward one with the two parts of every complex value traded.
//
// One CTA transforms a tile of L lines (x: L consecutive rows of the
// [n_z][n_y][n_x] array; y: L consecutive x columns of one z plane, the last tile of
// a plane partial when L does not divide n_x). The line lengths are run-time values
// (any n/2 = 2^a·3^b); what keeps the index work small is the layout:
//   * shared memory holds the tile as complex slots [slot][line] with the lanes of a
//     half-warp (L = 16) on consecutive lines, so that every stage access is
//     conflict-free whatever the stride of the slots, and the butterfly index and
//     its twiddles are shared by those lanes (broadcast loads);
//   * the reals go straight to the slot and part where the FFT wants them (the
//     permutations of P, NN, DD and ND are such scatters), and the paired pre- and
//     post-processing works in place: slot k ends as the two outputs of wavenumber k;
//   * y lines are read and written as row segments of L values; x lines in pairs of
//     values with the lanes along the line (the slots' row pitch L + 1 keeps those
//     transposing accesses conflict-free);
//   * the factors ½, 2 and 1/m of the split and of the normalisation sit in the
//     plan's tables, and divisions by run-time lengths are multiplications by their
//     reciprocals.
// Bound by instruction issue (the index arithmetic of run-time lengths, 57–69 % issue
// active in FP32), in FP64 by the FP64 pipe. Measured on 384×288×201 against the kernel this
// one replaced (one row per line, radices 4, 2 and 3, twiddles at stride 16 from the plan's
// 8n-entry table): FP32 x pass 300 → 97 µs forward, 344 → 99 µs backward, y passes
// 247 → 113 and 230 → 105 µs; 192×96×65: 25–37 → 13–16 µs a pass.
#pragma once
#include "xform_units.cuh"

namespace ps {

template <class T>
__device__ __forceinline__ void dft3(cplx<T>* v) {
  const T s3 = (T)0.86602540378443864676;  // sin(π/3)
  const cplx<T> t = cadd(v[1], v[2]), d = csub(v[1], v[2]);
  const cplx<T> u = {v[0].x - (T)0.5 * t.x, v[0].y - (T)0.5 * t.y};
  v[0] = cadd(v[0], t);
  v[1] = {u.x + s3 * d.y, u.y - s3 * d.x};
  v[2] = {u.x - s3 * d.y, u.y + s3 * d.x};
}

// 6 = 2 × 3 by the prime-factor map: X[(3·k1 + 4·k2) mod 6] from x[(3·n1 + 2·n2) mod 6], no twiddles
template <class T>
__device__ __forceinline__ void dft6(cplx<T>* v) {
  cplx<T> a[3] = {v[0], v[2], v[4]}, b[3] = {v[3], v[5], v[1]};
  dft3(a);
  dft3(b);
  v[0] = cadd(a[0], b[0]);
  v[3] = csub(a[0], b[0]);
  v[4] = cadd(a[1], b[1]);
  v[1] = csub(a[1], b[1]);
  v[2] = cadd(a[2], b[2]);
  v[5] = csub(a[2], b[2]);
}

// 9 = 3 × 3: X[k1 + 3k2] = Σ_{n2} W3^{n2·k2} W9^{n2·k1} Σ_{n1} x[n2 + 3n1] W3^{n1·k1}
template <class T>
__device__ __forceinline__ void dft9(cplx<T>* v) {
  const cplx<T> w1 = {(T)0.76604444311897803520, (T)-0.64278760968653932632};   // e^{−2πi/9}
  const cplx<T> w2 = {(T)0.17364817766693034885, (T)-0.98480775301220805937};   // e^{−4πi/9}
  const cplx<T> w4 = {(T)-0.93969262078590838405, (T)-0.34202014332566873304};  // e^{−8πi/9}
  cplx<T> a[3][3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
#pragma unroll
    for (int r = 0; r < 3; ++r) a[q][r] = v[q + 3 * r];
    dft3(a[q]);
  }
  a[1][1] = cmul(a[1][1], w1);
  a[1][2] = cmul(a[1][2], w2);
  a[2][1] = cmul(a[2][1], w2);
  a[2][2] = cmul(a[2][2], w4);
#pragma unroll
  for (int k1 = 0; k1 < 3; ++k1) {
    cplx<T> b[3] = {a[0][k1], a[1][k1], a[2][k1]};
    dft3(b);
#pragma unroll
    for (int k2 = 0; k2 < 3; ++k2) v[k1 + 3 * k2] = b[k2];
  }
}

template <class T>
__device__ __forceinline__ cplx<T> ldg_c(const cplx<T>* p) {  // a table entry (constant for the kernel)
  if constexpr (sizeof(T) == 4) {
    const float2 t = __ldg(reinterpret_cast<const float2*>(p));
    return {t.x, t.y};
  } else {
    const double2 t = __ldg(reinterpret_cast<const double2*>(p));
    return {t.x, t.y};
  }
}

// ⌊i/d⌋ for 0 ≤ i < 2^16 from mg = ⌈2^32/d⌉ (d = 1: mg = 0)
__device__ __forceinline__ int div_mg(int i, unsigned mg) { return mg ? (int)__umulhi((unsigned)i, mg) : i; }

// One Stockham stage of radix R over the tile's lines. `pre`: a table to multiply the
// stage's inputs with (first stage of the DCT-IV family), or null.
template <class T, int R>
__device__ __forceinline__ void gen_stage(const cplx<T>* src, cplx<T>* dst, int lgL, int ls, int m,
                                          const FftStage& S, const cplx<T>* __restrict__ w,
                                          const cplx<T>* __restrict__ pre) {
  const int nb = S.nb, ns = S.ns, lm = (1 << lgL) - 1;
  for (int idx = threadIdx.x; idx < (nb << lgL); idx += blockDim.x) {
    const int l = idx & lm, j = idx >> lgL;
    const cplx<T>* s = src + j * ls + l;
    cplx<T> v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = s[r * nb * ls];
    if (pre) {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = cmul(v[r], ldg_c(pre + j + r * nb));
    }
    const int q = div_mg(j, S.mg), k = j - q * ns;
    if (ns > 1) {
      const cplx<T>* wk = w + k * S.tws;
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], ldg_c(wk + (r - 1) * k * S.tws));
    }
    if constexpr (R == 3) dft3(v);
    else if constexpr (R == 6) dft6(v);
    else if constexpr (R == 9) dft9(v);
    else fast::dftR<T, R, false>(v);
    cplx<T>* d = dst + (q * ns * R + k) * ls + l;
#pragma unroll
    for (int r = 0; r < R; ++r) d[r * ns * ls] = v[r];
  }
}

// A pair of consecutive values (e, e + 1), e even; al: the address is aligned to the pair
template <class V>
__device__ __forceinline__ void ld_pair(const V* p, bool al, V& a, V& b) {
  if (al) {
    const row::vec<V, 2> t = *reinterpret_cast<const row::vec<V, 2>*>(p);
    a = t.v[0];
    b = t.v[1];
  } else {
    a = p[0];
    b = p[1];
  }
}
template <class V>
__device__ __forceinline__ void st_pair(V* p, bool al, V a, V b) {
  if (al) {
    row::vec<V, 2> t;
    t.v[0] = a;
    t.v[1] = b;
    *reinterpret_cast<row::vec<V, 2>*>(p) = t;
  } else {
    p[0] = a;
    p[1] = b;
  }
}

// The sizes of a tile, at run time (this kernel) or compile time (xform_mid.cuh).
struct DimRt {
  int n_, m_, lg_, ls_;
  unsigned mg_m, mg_h;
  __device__ __forceinline__ int n() const { return n_; }
  __device__ __forceinline__ int m() const { return m_; }
  __device__ __forceinline__ int lg() const { return lg_; }   // log2 of the lines
  __device__ __forceinline__ int ls() const { return ls_; }   // row pitch of the slots
  __device__ __forceinline__ int div_m(int i) const { return div_mg(i, mg_m); }
  __device__ __forceinline__ int div_h(int i) const { return div_mg(i, mg_h); }  // by n/2
};

// The three kinds of boundary pair, as far as the slots go. by_kind(bc, f) calls f with the
// kind as a constant, so that loops over values are compiled per kind.
enum { KIND_P = 0, KIND_CT = 1 /* NN, DD */, KIND_IV = 2 /* ND, DN */ };
template <class F>
__device__ __forceinline__ void by_kind(int bc, F&& f) {
  if (bc == BC_P) f(std::integral_constant<int, KIND_P>{});
  else if (bc_iv(bc)) f(std::integral_constant<int, KIND_IV>{});
  else f(std::integral_constant<int, KIND_CT>{});
}

// Where the line elements sit in the slots. Physical side (the field's values): the
// elements (e0, e1) of slot p's two parts; spectral side: the coefficients (q0, q1) of slot
// k's; and the inverse maps for the pair (e, e + 1), e even: slot s and part c of each.
template <class D, int KIND>
struct SlotMap {
  D d;
  int bc;
  __device__ __forceinline__ int mk(int j) const {  // Makhoul (n = 2m)
    return j < d.m() ? 2 * j : 2 * d.n() - 1 - 2 * j;
  }
  __device__ __forceinline__ void phys(int p, int& e0, int& e1) const {
    if constexpr (KIND == KIND_P) {
      e0 = 2 * p;
      e1 = 2 * p + 1;
    } else if constexpr (KIND == KIND_IV) {  // DN, the reversed line: the two parts trade places
      const int lo = 2 * p, hi = d.n() - 1 - 2 * p;
      e0 = bc == BC_DN ? hi : lo;
      e1 = bc == BC_DN ? lo : hi;
    } else {
      e0 = mk(2 * p);
      e1 = mk(2 * p + 1);
    }
  }
  __device__ __forceinline__ void spec(int k, int& q0, int& q1) const {
    const int n = d.n(), m = d.m();
    if constexpr (KIND == KIND_P) {
      q0 = k == 0 ? 0 : 2 * k - 1;
      q1 = k == 0 ? n - 1 : 2 * k;
    } else if constexpr (KIND == KIND_IV) {
      q0 = 2 * k;
      q1 = n - 1 - 2 * k;
    } else {
      q0 = k;
      q1 = k == 0 ? m : n - k;
      if (bc == BC_DD) {
        q0 = n - 1 - q0;
        q1 = n - 1 - q1;
      }
    }
  }
  __device__ __forceinline__ void phys_of(int e, int& s0, int& c0, int& s1, int& c1) const {
    const int h = e >> 1, n = d.n(), m = d.m();
    if constexpr (KIND == KIND_P) {
      s0 = s1 = h;
      c0 = 0;
      c1 = 1;
    } else if constexpr (KIND == KIND_IV) {
      s0 = h;
      s1 = m - 1 - h;
      c0 = bc == BC_DN;
      c1 = bc != BC_DN;
    } else {
      const int j1 = n - 1 - h;
      s0 = h >> 1;
      c0 = h & 1;
      s1 = j1 >> 1;
      c1 = j1 & 1;
    }
  }
  __device__ __forceinline__ void spec_of(int e, int& s0, int& c0, int& s1, int& c1) const {
    const int n = d.n(), m = d.m(), h = e >> 1;
    if constexpr (KIND == KIND_P) {  // X_2h is part 1 of slot h, X_{2h+1} part 0 of slot h + 1; X_0, X_{n−1} in slot 0
      s0 = h;
      c0 = h > 0;
      s1 = h + 1 == m ? 0 : h + 1;
      c1 = h + 1 == m;
    } else if constexpr (KIND == KIND_IV) {
      s0 = h;
      c0 = 0;
      s1 = m - 1 - h;
      c1 = 1;
    } else {
      auto one = [&](int q, int& s, int& c) {
        c = q >= m;
        s = q == m ? 0 : (c ? n - q : q);
      };
      one(bc == BC_DD ? n - 1 - e : e, s0, c0);
      one(bc == BC_DD ? n - 2 - e : e + 1, s1, c1);
    }
  }
};

// ---- the steps shared with the compile-time kernels (xform_mid.cuh) ----------------------

// x lines into the slots (FWD: field values, else coefficients): pairs of consecutive
// values, the lanes along the line.
template <class D, class T, class TI, bool FWD, class Scale>
__device__ __forceinline__ void x_load(const D& d, int bc, const TI* in, int live, T* rA, bool scaled, Scale&& scale_of) {
  const int m = d.m(), ls = d.ls();
  const bool al = !((uintptr_t)in & (2 * sizeof(TI) - 1));
  const bool neg = FWD && bc == BC_DD;  // DST ordering: the odd elements change sign
  by_kind(bc, [&](auto kind) {
    constexpr int KIND = decltype(kind)::value;
    const SlotMap<D, KIND> map{d, bc};
#pragma unroll 4
    for (int idx = threadIdx.x; idx < live * m; idx += blockDim.x) {
      const int l = d.div_m(idx), e = 2 * (idx - l * m);
      TI u0, u1;
      ld_pair(in + 2 * idx, al, u0, u1);
      T v0 = ld_cvt<T, TI>::f(u0), v1 = ld_cvt<T, TI>::f(u1);
      if (scaled) {
        const T sc = scale_of(l);
        v0 *= sc;
        v1 *= sc;
      }
      if constexpr (FWD && KIND == KIND_P) {  // the pair is one slot
        reinterpret_cast<cplx<T>*>(rA)[(e >> 1) * ls + l] = {v0, v1};
      } else {
        int s0, c0, s1, c1;
        if (FWD) map.phys_of(e, s0, c0, s1, c1);
        else map.spec_of(e, s0, c0, s1, c1);
        rA[2 * (s0 * ls + l) + c0] = v0;
        rA[2 * (s1 * ls + l) + c1] = (FWD && KIND == KIND_CT && neg) ? -v1 : v1;
      }
    }
  });
}

// Backward P, NN, DD: the pairs (k, m−k), the parts traded for the inverse FFT:
// Z_k = (V_k + conj V_{m−k})/2m + pb_k·(V_k − conj V_{m−k}), pb_k = i·e^{+2πik/n}/2m; NN, DD:
// V_q = xb_q·(X_q − i X_{n−q}), xb_q = ½e^{+iπq/2n}. get(k, l): the two values of slot k.
template <class D, class T, class Get>
__device__ __forceinline__ void pairs_bwd(const D& d, int bc, cplx<T>* buf, const cplx<T>* t0, const cplx<T>* t1, T s,
                                          Get&& get) {
  const int m = d.m(), lg = d.lg(), ls = d.ls(), np = m / 2 + 1;
#pragma unroll 1
  for (int idx = threadIdx.x; idx < (np << lg); idx += blockDim.x) {
    const int l = idx & ((1 << lg) - 1), k = idx >> lg;
    const cplx<T> x = get(k, l), y = get(k == 0 ? 0 : m - k, l);
    cplx<T> V, W;
    if (bc == BC_P) {
      V = k == 0 ? cplx<T>{x.x, (T)0} : cplx<T>{x.x, -x.y};
      W = k == 0 ? cplx<T>{x.y, (T)0} : cplx<T>{y.x, -y.y};
    } else {
      V = cmul(ldg_c(t1 + k), k == 0 ? cplx<T>{x.x, (T)0} : cplx<T>{x.x, -x.y});
      W = cmul(ldg_c(t1 + m - k), k == 0 ? cplx<T>{x.y, -x.y} : cplx<T>{y.x, -y.y});
    }
    const cplx<T> Sm = cadd(V, conj_(W)), Dm = cmul(ldg_c(t0 + k), csub(V, conj_(W)));
    buf[k * ls + l] = {s * Sm.y + Dm.y, s * Sm.x + Dm.x};
    if (k != 0 && 2 * k != m) buf[(m - k) * ls + l] = {Dm.y - s * Sm.y, s * Sm.x - Dm.x};
  }
}

// Forward P, NN, DD: the real DFT of the packed sequence,
// V_k = (Z_k + conj Z_{m−k})/2 + pf_k·(Z_k − conj Z_{m−k}), pf_k = −(i/2)e^{−2πik/n}; NN, DD:
// X_q = Re(xf_q V_q), X_{n−q} = −Im, xf_q = 2e^{−iπq/2n}. put(k, l, v0, v1): slot k's outputs.
template <class D, class T, class Put>
__device__ __forceinline__ void pairs_fwd(const D& d, int bc, const cplx<T>* buf, const cplx<T>* t0,
                                          const cplx<T>* t1, Put&& put) {
  const int m = d.m(), lg = d.lg(), ls = d.ls(), np = m / 2 + 1;
#pragma unroll 1
  for (int idx = threadIdx.x; idx < (np << lg); idx += blockDim.x) {
    const int l = idx & ((1 << lg) - 1), k = idx >> lg;
    const cplx<T> Zk = buf[k * ls + l], Zm = buf[(k == 0 ? 0 : m - k) * ls + l];
    const cplx<T> Sm = cadd(Zk, conj_(Zm)), Dm = cmul(ldg_c(t0 + k), csub(Zk, conj_(Zm)));
    const cplx<T> V = {(T)0.5 * Sm.x + Dm.x, (T)0.5 * Sm.y + Dm.y};
    const cplx<T> W = {(T)0.5 * Sm.x - Dm.x, Dm.y - (T)0.5 * Sm.y};  // V_{m−k}
    if (bc == BC_P) {
      if (k == 0) put(0, l, V.x, W.x);
      else {
        put(k, l, V.x, -V.y);
        if (2 * k != m) put(m - k, l, W.x, -W.y);
      }
    } else if (k == 0) {
      put(0, l, (T)2 * V.x, (T)1.41421356237309504880 * W.x);
    } else {
      const cplx<T> c1 = cmul(ldg_c(t1 + k), V);
      put(k, l, c1.x, -c1.y);
      if (2 * k != m) {
        const cplx<T> c2 = cmul(ldg_c(t1 + m - k), W);
        put(m - k, l, c2.x, -c2.y);
      }
    }
  }
}

// The slots to x lines, with the output modes of XformArgs (compiled per mode). sw: the
// parts are traded; fd: the face-centred lines' slots, a value in part 0 of each.
template <class D, class T, class TO, bool FWD, class Args, class Scale>
__device__ __forceinline__ void x_store(const D& d, const Args& a, TO* out, size_t base, int live, const T* rS, int sw,
                                        bool fd, bool scaled, Scale&& scale_of, T& tmax) {
  const int n = d.n(), ls = d.ls(), bc = a.bc;
  const bool neg = !FWD && bc == BC_DD;
  const bool al = !((((uintptr_t)out) & (2 * sizeof(TO) - 1)) | (((uintptr_t)a.out2 | (uintptr_t)a.base32) & 7));
  TO* dst = out + base;
  const float* b32 = a.base32 ? a.base32 + base : nullptr;
  float* o2 = a.out2 ? a.out2 + base : nullptr;
  auto run = [&](auto kind, auto mode) {
    constexpr int KIND = decltype(kind)::value, OM = decltype(mode)::value;
    const SlotMap<D, KIND> map{d, bc};
#pragma unroll 4
    for (int idx = threadIdx.x; idx < live * (n >> 1); idx += blockDim.x) {
      const int l = d.div_h(idx), e = 2 * (idx - l * (n >> 1));
      int s0, c0, s1, c1;
      if (fd) {
        s0 = e;
        s1 = e + 1;
        c0 = c1 = 0;
      } else if (FWD) {
        map.spec_of(e, s0, c0, s1, c1);
      } else {
        map.phys_of(e, s0, c0, s1, c1);
      }
      T v0 = rS[2 * (s0 * ls + l) + (c0 ^ sw)], v1 = rS[2 * (s1 * ls + l) + (c1 ^ sw)];
      if constexpr (!FWD && KIND == KIND_CT) v1 = neg ? -v1 : v1;
      if (scaled) {
        const T sc = scale_of(l);
        v0 *= sc;
        v1 *= sc;
      }
      const int g = 2 * idx;
      if constexpr (sizeof(TO) == 8 && sizeof(T) == 4) {
        const double w0 = widen_f32(v0), w1 = widen_f32(v1);
        if constexpr (OM == row::OM_BASE) {
          float f0, f1;
          ld_pair(b32 + g, al, f0, f1);
          st_pair(dst + g, al, widen_f32(f0) + w0, widen_f32(f1) + w1);
        } else if constexpr (OM == row::OM_ACC) {
          double b0, b1;
          ld_pair(dst + g, al, b0, b1);
          st_pair(dst + g, al, b0 + w0, b1 + w1);
        } else if constexpr (OM == row::OM_STORE) {
          st_pair(dst + g, al, w0, w1);
        }
        tmax = fmaxf(tmax, fmaxf(fabsf(v0), fabsf(v1)));
        if (o2) st_pair(o2 + g, al, v0, v1);
      } else if constexpr (OM == row::OM_ACC) {
        TO b0, b1;
        ld_pair(dst + g, al, b0, b1);
        st_pair(dst + g, al, b0 + v0, b1 + v1);
      } else {
        st_pair(dst + g, al, v0, v1);
      }
    }
  };
  auto with_mode = [&](auto kind) {
    if constexpr (!FWD && sizeof(TO) == 8 && sizeof(T) == 4) {
      if (!out) return run(kind, std::integral_constant<int, row::OM_NONE>{});
      if (b32) return run(kind, std::integral_constant<int, row::OM_BASE>{});
    }
    if (a.accumulate) run(kind, std::integral_constant<int, row::OM_ACC>{});
    else run(kind, std::integral_constant<int, row::OM_STORE>{});
  };
  by_kind(bc, with_mode);
}

// max |value| of FP64 outputs (before widening: a 64-bit integer max would use the FP64 pipe)
template <class T>
__device__ __forceinline__ void amax_out(unsigned long long* amax, T tmax) {
  if constexpr (sizeof(T) == 4) {
    if (amax) {
      for (int o = 16; o > 0; o >>= 1) tmax = fmaxf(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
      const unsigned long long v = (unsigned long long)__double_as_longlong(st_cvt<double, T>::f(tmax));
      if ((threadIdx.x & 31) == 0 && v) atomicMax(amax, v);
    }
  }
}

// Transforms tile `grp`; every thread of the CTA takes part; smem_raw holds
// 2·(m + 1)·(L + 1) complex values (L = 1: 2·(m + 1)).
template <class T, class TI, class TO, bool FWD, int MAXR = 16>
__device__ void xform_group(const XformArgs<T>& a, int grp, unsigned char* smem_raw) {
  const LineTab<T>& tab = a.tab;
  const cplx<T>* t0 = tab.t0[FWD];
  const cplx<T>* t1 = tab.t1[FWD];
  const int n = a.n, m = a.m, lgL = a.lgL, L = 1 << lgL, lm = L - 1, ls = L > 1 ? L + 1 : 1;
  cplx<T>* bufA = reinterpret_cast<cplx<T>*>(smem_raw);
  cplx<T>* bufB = bufA + (m + 1) * ls;
  T* rA = reinterpret_cast<T*>(bufA);
  // no __restrict__: in and out may be the same array, and in the batched kernel
  // other CTAs rewrite it between tasks (the read-only cache path must not be used)
  const TI* in = static_cast<const TI*>(a.in);
  TO* out = static_cast<TO*>(a.out);
  const int nx = a.nx, ny = a.ny, bc = a.bc;
  const bool iv = bc_iv(bc), fd = bc == BC_FD;
  const DimRt dim{n, m, lgL, ls, tab.mg_m, tab.mg_h};
  const int tid = threadIdx.x, nt = blockDim.x;

  // ---- the tile: x: first element of row 0 of the group; y: column x0 of plane zb ----
  const int gpz = a.axis == 1 ? (nx + L - 1) >> lgL : 1;
  const int zb = a.axis == 1 ? grp / gpz : 0;
  const int x0 = a.axis == 1 ? (grp - zb * gpz) << lgL : 0;
  const size_t base = a.axis == 0 ? (size_t)grp * L * n : (size_t)zb * ny * nx + x0;
  const int live = a.axis == 0 ? min(L, a.nlines - grp * L) : min(L, nx - x0);
  auto scale_of = [&](int l) { return a.plane_scale[a.axis == 0 ? (grp * L + l) / ny : zb]; };
  const bool fscale = FWD && a.plane_scale, bscale = !FWD && a.plane_scale;

  // ---- 1. load into the slots of bufA ----
  if (fd) {
    // z_j = (y_2j, y_2j+1) of the odd extension, both directions (m = n); the wall
    // entry is kept in slot m, which no stage writes
    auto val = [&](int l, int t) -> T {
      if (t == 0 || t == n) return (T)0;
      const int e = t < n ? t : 2 * n - t;
      const T v = ld_cvt<T, TI>::f(a.axis == 0 ? in[base + (size_t)l * n + e] : in[base + (size_t)e * nx + l]);
      return t < n ? v : -v;
    };
    for (int idx = tid; idx < (m << lgL); idx += nt) {
      const int l = a.axis == 0 ? div_mg(idx, tab.mg_m) : (idx & lm);
      const int j = a.axis == 0 ? idx - l * m : idx >> lgL;
      if (l >= live) continue;
      const T sc = fscale ? scale_of(l) : (T)1;
      const cplx<T> z = {val(l, 2 * j), val(l, 2 * j + 1)};
      bufA[j * ls + l] = fscale ? cscale(z, sc) : z;
      if (j == 0) {
        const T w = ld_cvt<T, TI>::f(a.axis == 0 ? in[base + (size_t)l * n] : in[base + l]);
        bufA[m * ls + l] = cplx<T>{w * sc, (T)0};
      }
    }
  } else if (a.axis == 0) {
    x_load<DimRt, T, TI, FWD>(dim, bc, in + base, live, rA, fscale, scale_of);
  } else {
    const T sc = fscale ? a.plane_scale[zb] : (T)1;
    by_kind(bc, [&](auto kind) {
    const SlotMap<DimRt, decltype(kind)::value> map{dim, bc};
#pragma unroll 4
    for (int idx = tid; idx < (m << lgL); idx += nt) {
      const int l = idx & lm, p = idx >> lgL;
      if (l >= live) continue;
      int e0, e1;
      if (FWD) map.phys(p, e0, e1);
      else map.spec(p, e0, e1);
      T v0 = ld_cvt<T, TI>::f(in[base + (size_t)(e0 * nx) + l]), v1 = ld_cvt<T, TI>::f(in[base + (size_t)(e1 * nx) + l]);
      if (FWD) {
        if (bc == BC_DD) {
          if (e0 & 1) v0 = -v0;
          if (e1 & 1) v1 = -v1;
        }
        if (fscale) {
          v0 *= sc;
          v1 *= sc;
        }
      }
      bufA[p * ls + l] = cplx<T>{v0, v1};
    }
    });
  }
  __syncthreads();

  // ---- 2. backward P, NN, DD: the pairs (k, m−k), in place ----
  if (!FWD && !iv && !fd) {
    pairs_bwd(dim, bc, bufA, t0, t1, tab.inv2m, [&](int k, int l) { return bufA[k * ls + l]; });
    __syncthreads();
  }

  // ---- 3. the FFT ----
  cplx<T>* src = bufA;
  cplx<T>* dst = bufB;
  for (int st = 0; st < tab.nstages; ++st) {
    const FftStage& S = tab.stage[st];
    const cplx<T>* pre = (iv && st == 0) ? t0 : nullptr;
    switch (S.r) {
      case 16: if constexpr (MAXR >= 16) gen_stage<T, 16>(src, dst, lgL, ls, m, S, tab.w, pre); break;
      case 9: gen_stage<T, 9>(src, dst, lgL, ls, m, S, tab.w, pre); break;
      case 8: gen_stage<T, 8>(src, dst, lgL, ls, m, S, tab.w, pre); break;
      case 6: gen_stage<T, 6>(src, dst, lgL, ls, m, S, tab.w, pre); break;
      case 4: gen_stage<T, 4>(src, dst, lgL, ls, m, S, tab.w, pre); break;
      case 3: gen_stage<T, 3>(src, dst, lgL, ls, m, S, tab.w, pre); break;
      default: gen_stage<T, 2>(src, dst, lgL, ls, m, S, tab.w, pre); break;
    }
    __syncthreads();
    cplx<T>* t = src;
    src = dst;
    dst = t;
  }
  if (iv && tab.nstages == 0) {  // n = 2: the pre-factor of the one point
    for (int l = tid; l < L; l += nt) src[l] = cmul(src[l], ldg_c(t0));
    __syncthreads();
  }

  // ---- 4. post-processing in place (y, forward and DCT-IV: straight to the rows) ----
  T* rS = reinterpret_cast<T*>(src);
  T tmax = (T)0;
  auto emit = [&](size_t g, T v) {  // one output value
    const TO x = st_cvt<TO, T>::f(v);
    if constexpr (sizeof(TO) == 8) {
      if (out) {
        if constexpr (sizeof(T) == 4) {
          if (a.base32) out[g] = widen_f32(a.base32[g]) + x;
          else out[g] = a.accumulate ? out[g] + x : x;
        } else {
          out[g] = a.accumulate ? out[g] + x : x;
        }
      }
      if constexpr (sizeof(T) == 4) {
        tmax = fmaxf(tmax, fabsf(v));
        if (a.out2) a.out2[g] = v;
      }
    } else {
      out[g] = a.accumulate ? out[g] + x : x;
    }
  };
  const T yscale = (a.axis == 1 && bscale) ? a.plane_scale[zb] : (T)1;
  // the two values of slot k: kept in the slot (x), or written to their rows (y)
  auto put_as = [&](auto kind, int k, int l, T v0, T v1) {
    if (a.axis == 0) {
      src[k * ls + l] = cplx<T>{v0, v1};
    } else if (l < live) {
      const SlotMap<DimRt, decltype(kind)::value> map{dim, bc};
      int e0, e1;
      if (FWD) map.spec(k, e0, e1);
      else map.phys(k, e0, e1);
      emit(base + (size_t)(e0 * nx) + l, bscale ? v0 * yscale : v0);
      emit(base + (size_t)(e1 * nx) + l, bscale ? v1 * yscale : v1);
    }
  };
  if (fd) {  // X_k = −Im(Y_k), k = 1 … n−1 (× 1/2n backward), into part 0 of slot k
    const T sc = FWD ? (T)1 : tab.inv2m;
    for (int idx = tid; idx < ((m / 2 + 1) << lgL); idx += nt) {
      const int l = idx & lm, k = idx >> lgL;
      const cplx<T> Zk = src[k * ls + l], Zm = src[(k == 0 ? 0 : m - k) * ls + l];
      const cplx<T> Sm = cadd(Zk, conj_(Zm)), D = cmul(ldg_c(t0 + k), csub(Zk, conj_(Zm)));
      if (k == 0) {
        rS[2 * l] = bufA[m * ls + l].x;
      } else {
        rS[2 * (k * ls + l)] = -((T)0.5 * Sm.y + D.y) * sc;
        if (2 * k != m) rS[2 * ((m - k) * ls + l)] = ((T)0.5 * Sm.y - D.y) * sc;
      }
    }
    __syncthreads();
  } else if (iv) {  // c_k = t_k·U_k, t_k = 2e^{−iπ(4k+1)/4n} (backward: /2n); outputs Re, −Im
    for (int idx = tid; idx < (m << lgL); idx += nt) {
      const int l = idx & lm, k = idx >> lgL;
      const cplx<T> c = cmul(ldg_c(t1 + k), src[k * ls + l]);
      put_as(std::integral_constant<int, KIND_IV>{}, k, l, c.x, -c.y);
    }
    if (a.axis == 0) __syncthreads();
  } else if (FWD) {
    auto pairs = [&](auto kind) {
      pairs_fwd(dim, bc, src, t0, t1, [&](int k, int l, T v0, T v1) { put_as(kind, k, l, v0, v1); });
    };
    if (bc == BC_P) pairs(std::integral_constant<int, KIND_P>{});
    else pairs(std::integral_constant<int, KIND_CT>{});
    if (a.axis == 0) __syncthreads();
  }

  // ---- 5. store ----
  // backward P, NN, DD: the FFT's parts are still traded (part c of a slot is 1 − c)
  const int sw = (!FWD && !iv && !fd) ? 1 : 0;
  if (a.axis == 0) {
    x_store<DimRt, T, TO, FWD>(dim, a, out, base, live, rS, sw, fd, bscale, scale_of, tmax);
  } else if (fd) {
    for (int idx = tid; idx < (n << lgL); idx += nt) {
      const int l = idx & lm, e = idx >> lgL;
      if (l < live) emit(base + (size_t)(e * nx) + l, bscale ? rS[2 * (e * ls + l)] * yscale : rS[2 * (e * ls + l)]);
    }
  } else if (!FWD && !iv) {
    by_kind(bc, [&](auto kind) {
    const SlotMap<DimRt, decltype(kind)::value> map{dim, bc};
    for (int idx = tid; idx < (m << lgL); idx += nt) {
      const int l = idx & lm, p = idx >> lgL;
      if (l >= live) continue;
      const cplx<T> z = src[p * ls + l];
      int e0, e1;
      map.phys(p, e0, e1);
      const T v0 = (bc == BC_DD && (e0 & 1)) ? -z.y : z.y, v1 = (bc == BC_DD && (e1 & 1)) ? -z.x : z.x;
      emit(base + (size_t)(e0 * nx) + l, bscale ? v0 * yscale : v0);
      emit(base + (size_t)(e1 * nx) + l, bscale ? v1 * yscale : v1);
    }
    });
  }
  if constexpr (sizeof(TO) == 8) amax_out(a.amax, tmax);
}

}  // namespace ps
