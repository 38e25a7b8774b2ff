// tridiag.cu — the N_x·N_y tridiagonal systems of Eq. 5 along z.
//
// Column (q_x, q_y) solves a_k Φ̂_{k−1} + (b_k + λ_qx/Δx² + λ_qy/Δy²) Φ̂_k + c_k Φ̂_{k+1} = f̂_k.
// One thread per column; a warp covers 32 consecutive q_x, so every access to
// plane k is a coalesced row segment. Gauss elimination without pivoting
// (each column is weakly diagonally dominant with a strictly dominant row).
// FP64: the eliminated super-diagonal goes to a scratch array; the eliminated right-hand
// side overwrites the data in place and is replaced by Φ̂_k in the back substitution.
//
// Periodic z (§3: the cyclic system "reduced into two tridiagonal problems"): cyclic Gauss
// elimination with the last unknown kept aside (tridiag_dev.cuh), one forward and one
// backward sweep.
//
// Singular column (every axis P or NN): (q_x, q_y) = (0, 0) has λ = 0 and a
// singular z matrix. Its right-hand side loses its Δz^f-weighted mean, Φ̂_0 = 0
// is pinned (row 0 dropped), and the solution's weighted mean is removed. A warp
// of the same launch does this column.
#include <type_traits>

#include "tridiag_dev.cuh"

namespace ps {

// FP32 columns: the forward sweep keeps the elimination's state
// (G, V) only at the end of every chunk of ZK planes (1/8 of the data
// volume, in the scratch array); the backward sweep walks the chunks from the top,
// re-reads each chunk's right-hand side, recomputes its (C, V) from the
// checkpoint in registers (the same instructions on the same inputs, so
// bit-identical to the forward sweep) and back-substitutes. HBM traffic: read f̂
// twice (the second read of a chunk often hits L2), write Φ̂ once; loads of the
// next chunk are issued before the current chunk is processed. The coefficients
// (a_k, c_k), with a_0 = c_{n−1} = 0, sit in a shared table (one broadcast
// load per row) and whole chunks run without per-row bound tests.
// Periodic columns run the same two sweeps with the cyclic elimination of tridiag_dev.cuh
// (a third value F per checkpoint).
constexpr int ZB = 128;            // columns (threads) per CTA
constexpr int ZTAB_MAX = 4096;     // planes whose coefficient table sits in shared memory (32 KB)

// A column with a small |λ| (low wavenumbers) has κ ≈ ‖T_z‖/|λ| up to ~10^7 on the
// stretched channel grid. The elimination in excess form keeps λ's digits, but the FP32
// sums over the right-hand side still err by up to ~√n_z·ε_32 of Σ|f̂|/|λ|, smooth in z
// with a large amplitude: what an FP32 correction solve removes worst. The columns with
// the largest κ — a rectangle q_x < lowx, q_y < lowy fixed at plan creation (low_rect.h:
// κ > 10^5 in any case, down to 10^3 while two columns an SM are enough) — are solved here
// in double-float arithmetic, ~2^−46 relative per operation against ε_32 = 2^−24 (the
// singular column (0,0) with its weighted-mean pinning among them), by CTAs of the same
// launch as the FP32 columns, so they overlap them. Output rounded to FP32. (The line:
// FP32 solutions on 13 shapes are 1.1 to 5 times closer to 64 bits than they were with
// b + λ in FP32 and the line at 10^4; at 10^6 one of them is no better than it was and at
// 10^8 it is 5 times worse. At 10^4 with this elimination 1024^3 pays 0.4 ms a pass.)
//
// Double-float rather than FP64: on this part one FP64 warp instruction occupies its SM
// sub-partition's FP64 pipe for ~33 ns whatever the number of active lanes. And a warp per
// column (zpart_column) rather than a thread: the serial double-float chain of n_z rows
// bounded the whole z pass on small planes (512×256×256: 172 µs against 86 for the FP32
// columns; figures at the kernels below). The coefficients are split on the host.
__device__ __noinline__ void zlow_column(const ZArgs<float>& a, int t) {  // t: column of the rectangle
  const int nrect = a.lowx * a.lowy;
  if (t >= nrect) return;
  // (c'_k, d'_k) as float pairs in the FP64-sized scratch: [column][k] each
  float2* cs = reinterpret_cast<float2*>(a.scr64) + (size_t)t * a.nz;
  zcolumn_df(a, (t / a.lowx) * a.nx + t % a.lowx, cs, cs + (size_t)nrect * a.nz);
}

// 1/x by the hardware approximation (`rcp.approx.ftz.f32`, about 1 ulp): the pivots
// here are normal FP32 numbers far from the overflow range.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Loads and stores with an L2 eviction priority (a policy from createpolicy)
__device__ __forceinline__ float ld_pol(const float* p, uint64_t pol) {
  float v;
  asm volatile("ld.global.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ void st_pol(float* p, float v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.f32 [%0], %1, %2;" ::"l"(p), "f"(v), "l"(pol) : "memory");
}

// The two ends of a non-periodic column need no code of their own: row 0's extra excess (a
// Dirichlet end) enters as the state G above it with the table's a_0 = 1, and the last row's
// as the table's c_{n−1}, whose coupling meets Φ̂_n = 0. Periodic: G = V = 0 and F = 1 above
// row 0 make its a_0 the wrap coupling.
// ONE: columns of at most ZK rows, read once and without a checkpoint.
template <bool TAB, bool PER, bool ONE>
__device__ __forceinline__ void zsolve_ckpt(const ZArgs<float>& a, int nlowb) {
  int bulk = blockIdx.x;
  // The rectangle's columns run in CTAs of ZB/32 warps spread evenly over the launch (their
  // arithmetic then overlaps the other CTAs' memory traffic instead of filling the SMs first).
  if (nlowb > 0) {
    const int lo = (int)((long long)blockIdx.x * nlowb / gridDim.x);
    const int hi = (int)((long long)(blockIdx.x + 1) * nlowb / gridDim.x);
    if (hi > lo) {
      pdl_wait();
      if (a.skip && *a.skip) return;
      zlow_column(a, lo * (ZB / 32) + (threadIdx.x >> 5));
      return;
    }
    bulk -= lo;
  }
  extern __shared__ float2 ztab[];  // [nz] (a_k, c_k) when TAB
  const int nz = a.nz;
  auto coef_of = [&](int k) -> float2 {
    return make_float2(k > 0 || PER ? __ldg(a.za + k) : 1.f, k < nz - 1 || PER ? __ldg(a.zc + k) : a.ge1);
  };
  auto coef = [&](int k) -> float2 {
    if constexpr (TAB) return ztab[k];
    else return coef_of(k);
  };
  if constexpr (TAB) {
    for (int k = threadIdx.x; k < nz; k += ZB) ztab[k] = coef_of(k);
  }
  pdl_wait();
  if (a.skip && *a.skip) return;
  if constexpr (TAB) __syncthreads();
  const int ncol = a.nx * a.ny;
  // checkpoints: [nchunk][ncol] of (G, V), and of F when periodic (in the second scratch)
  float2* __restrict__ ck = reinterpret_cast<float2*>(a.scr_c);
  float* __restrict__ fk = PER ? a.scr_u : nullptr;
  const int col = bulk * ZB + threadIdx.x;
  const int colc = col < ncol ? col : ncol - 1;
  const int i = colc % a.nx, j = colc / a.nx;
  const bool act = col < ncol && !(a.singular && col == 0) && !(i < a.lowx && j < a.lowy);
  const float lam = -(a.lamx[i] + a.lamy[j]);
  const float g = lam + a.ga;  // every row's excess
  const float G0 = PER ? 0.f : a.ge0;
  const size_t st = (size_t)ncol;
  const int nr = PER ? nz - 1 : nz;  // rows eliminated (periodic: the last unknown is kept aside)
  const int nch = zckpt_chunks(nr), nfull = nr / ZK;
  float* __restrict__ d = a.data + colc;

  // A field beyond L2 (30 M values = 120 MB): the output, and of the input all but the top
  // planes that the backward sweep reads first, are marked to be evicted first. Without
  // that the output pushes the input out (1024^3: 2.60 ms a pass, with it 2.39; the input's
  // share is 0.02 of that).
  uint64_t pol_first, pol_norm;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol_first));
  asm("createpolicy.fractional.L2::evict_unchanged.b64 %0, 1.0;" : "=l"(pol_norm));
  const bool big = (size_t)ncol * nz > (size_t)30000000;
  const int ckeep = big ? nch - nch / 7 : 0;
  const uint64_t spol = big ? pol_first : pol_norm;

  // one chunk of the elimination (zsolve_column's): rows k0 … k0+ZK−1 (all present when FULL)
  float S = 0.f, Tc = 1.f, X = 0.f;
  auto eliminate = [&](int k0, const float* cur, float& G, float& V, float& F, float* ca, float* va, float* fa,
                       bool fwd, auto full_tag) {
    constexpr bool FULL = decltype(full_tag)::value;
#pragma unroll
    for (int u = 0; u < ZK; ++u) {
      const int k = k0 + u;
      if (FULL || k < nr) {
        const float2 q = coef(k);
        // (t and the diagonal c + t side by side: the chain of G is FMA, reciprocal, product)
        const float t = fmaf(q.x, G, g), cg = q.y + g;
        const float m = rcp_approx(PER ? fmaf(q.x, F, fmaf(q.x, G, cg)) : fmaf(q.x, G, cg));
        V = fmaf(q.x, V, -cur[u]) * m;
        G = t * m;
        if constexpr (PER) F = (q.x * F) * m;
        if (ca) {
          ca[u] = q.y * m;
          va[u] = V;
          if constexpr (PER) fa[u] = F;
        }
        if constexpr (PER) {
          if (fwd) {  // the forward sweep also composes Φ̂_0
            S = fmaf(Tc, V, S);
            X = fmaf(Tc, G, X);
            Tc = Tc * (q.y * m);
          }
        }
      }
    }
  };
  auto chunk = [&](int c, const float* cur, float& G, float& V, float& F, float* ca, float* va, float* fa, bool fwd) {
    if (c < nfull) eliminate(c * ZK, cur, G, V, F, ca, va, fa, fwd, std::true_type{});
    else eliminate(c * ZK, cur, G, V, F, ca, va, fa, fwd, std::false_type{});
  };
  auto load = [&](int c, float* buf, bool stream) {
    const float* src = d + (size_t)c * ZK * st;
    const uint64_t pol = stream ? pol_first : pol_norm;
    if (c < nfull) {
#pragma unroll
      for (int u = 0; u < ZK; ++u) buf[u] = ld_pol(src + (size_t)u * st, pol);
    } else {
#pragma unroll
      for (int u = 0; u < ZK; ++u) buf[u] = (c * ZK + u < nr) ? ld_pol(src + (size_t)u * st, pol) : 0.f;
    }
  };
  // L2 prefetch of the chunk after next (both sweeps), so that more of the column
  // is in flight than the registers of the next chunk allow; not for a field that L2 holds
  // (512×256×144: 49 µs a pass with it, 45 without)
  auto prefetch = [&](int c2) {
    if (big && c2 >= 0 && c2 < nfull) {
      const float* src = d + (size_t)c2 * ZK * st;
#pragma unroll
      for (int u = 0; u < ZK; ++u) asm volatile("prefetch.global.L2 [%0];" ::"l"(src + (size_t)u * st));
    }
  };
  float G = G0, V = 0.f, F = 1.f, x = 0.f, y = 0.f;
  float cur[ZK], ca[ZK], va[ZK], fa[PER ? ZK : 1];
  auto top = [&] {  // periodic: the last row gives the last unknown
    const float2 q = coef(nz - 1);
    const float dl = d[(size_t)(nz - 1) * st];
    y = fmaf(q.x, V, fmaf(q.y, S, -dl)) * rcp_approx(fmaf(q.y, X, fmaf(q.x, G, g)));
    if (act) d[(size_t)(nz - 1) * st] = y;
    x = y;
  };
  auto substitute = [&](int c) {
    float* dst = d + (size_t)c * ZK * st;
#pragma unroll
    for (int u = ZK - 1; u >= 0; --u) {
      if (c < nfull || c * ZK + u < nr) {
        x = fmaf(ca[u], x, va[u]);
        if constexpr (PER) x = fmaf(fa[u], y, x);
        if (act) st_pol(dst + (size_t)u * st, x, spol);
      }
    }
  };
  if constexpr (ONE) {
    load(0, cur, false);
    chunk(0, cur, G, V, F, ca, va, fa, true);
    if constexpr (PER) top();
    substitute(0);
  } else {
    float nxt[ZK];
    load(0, cur, 0 < ckeep);
    for (int c = 0; c < nch; ++c) {
      prefetch(c + 2);
      if (c + 1 < nch) load(c + 1, nxt, c + 1 < ckeep);
      chunk(c, cur, G, V, F, nullptr, nullptr, nullptr, true);
      ck[(size_t)c * ncol + colc] = make_float2(G, V);
      if constexpr (PER) fk[(size_t)c * ncol + colc] = F;
#pragma unroll
      for (int u = 0; u < ZK; ++u) cur[u] = nxt[u];
    }
    if constexpr (PER) top();
    // backward: chunks from the top; the chunk below in flight
    load(nch - 1, cur, big);
    for (int c = nch - 1; c >= 0; --c) {
      prefetch(c - 2);
      if (c > 0) load(c - 1, nxt, big);
      const float2 prev = (c > 0) ? ck[(size_t)(c - 1) * ncol + colc] : make_float2(G0, 0.f);
      G = prev.x;
      V = prev.y;
      if constexpr (PER) F = (c > 0) ? fk[(size_t)(c - 1) * ncol + colc] : 1.f;
      chunk(c, cur, G, V, F, ca, va, fa, false);
      substitute(c);
#pragma unroll
      for (int u = 0; u < ZK; ++u) cur[u] = nxt[u];
    }
  }
}

// Not bounded for residency: 93 registers and five CTAs per SM (periodic: 123 and four; one
// chunk: 72 and seven). Asked for five or six, the compiler spills and 1024^3 takes 2.50 or
// 2.62 ms. Measured (ms a pass, before → now): 1024^3 2.38 → 2.40 (12.7 B a point, HBM-bound),
// 512×256×256 0.172 → 0.086 and 128^3 0.071 → 0.012 (bound by the rectangle's serial chains
// before), 4096×4096×16 0.59 → 0.36 (one chunk: read once), 512^3 periodic 1.42 + 0.07 → 0.37
// (two tridiagonal sweeps per column, 48 B a point, and the singular column by one thread).
template <bool TAB, bool ONE>
__global__ void __launch_bounds__(ZB) zsolve_ckpt_kernel(ZArgs<float> a, int nlowb) {
  zsolve_ckpt<TAB, false, ONE>(a, nlowb);
}
template <bool TAB, bool ONE>
__global__ void __launch_bounds__(ZB) zsolve_ckpt_per_kernel(ZArgs<float> a, int nlowb) {
  zsolve_ckpt<TAB, true, ONE>(a, nlowb);
}

namespace {
template <bool TAB, bool PER, bool ONE>
cudaError_t launch_ckpt(const ZArgs<float>& a, int grid, int nlowb, size_t smem, cudaStream_t st) {
  auto k = PER ? zsolve_ckpt_per_kernel<TAB, ONE> : zsolve_ckpt_kernel<TAB, ONE>;
  return launch_k(k, grid, ZB, smem, st, a, nlowb);
}
}  // namespace

cudaError_t launch_zsolve_ckpt(ZArgs<float> a, cudaStream_t st) {
  const int ncol = a.nx * a.ny, wpc = ZB / 32;
  const int nlowb = (a.lowx * a.lowy + wpc - 1) / wpc;
  const int grid = nlowb + (ncol + ZB - 1) / ZB;
  const size_t smem = (size_t)a.nz * sizeof(float2);
  if ((a.periodic ? a.nz - 1 : a.nz) <= ZK)
    return a.periodic ? launch_ckpt<true, true, true>(a, grid, nlowb, smem, st)
                      : launch_ckpt<true, false, true>(a, grid, nlowb, smem, st);
  if (a.nz <= ZTAB_MAX)
    return a.periodic ? launch_ckpt<true, true, false>(a, grid, nlowb, smem, st)
                      : launch_ckpt<true, false, false>(a, grid, nlowb, smem, st);
  return a.periodic ? launch_ckpt<false, true, false>(a, grid, nlowb, 0, st)
                    : launch_ckpt<false, false, false>(a, grid, nlowb, 0, st);
}

// FP64: a thread per column, or on planes of few columns, where that leaves most of the chip
// idle behind serial chains, a warp per column. The singular column is always a warp's
// (block 0). Measured, a thread's chain takes 4 + 0.61·n_z µs, and warps 7 + N·(0.003 +
// 0.00009·n_z) µs for N columns; a warp each where that is less: n_z ≥ 12 at 1024 columns, 22 at
// 2048, 63 at 4096, never beyond 6700. Thread and warp, µs: 32×32×32 22 and 10, 64×64×64 43 and
// 43, 64×64×256 154 and 117, 128×64×64 41 and 67, 64×64×8 10 and 24. 256^3: 564 → 429 µs (11
// FP64 instructions a row instead of 20; the FP64 pipe binds, with 3.4 warps per sub-partition
// taking the time of four).
inline bool warp_columns(int ncol, int nz) { return (6800LL - ncol) * nz > 33LL * (1000 + ncol); }
__global__ void __launch_bounds__(128) zsolve64_kernel(ZArgs<double> a) {
  pdl_wait();
  int b = blockIdx.x;
  if (a.singular) {
    if (b == 0) {
      if (threadIdx.x < 32) zpart64(a, 0, true);
      return;
    }
    --b;
  }
  zsolve_column<double>(a, b * blockDim.x + threadIdx.x);
}

__global__ void __launch_bounds__(128) zpart64_kernel(ZArgs<double> a) {
  pdl_wait();
  const int col = blockIdx.x * 4 + (threadIdx.x >> 5);
  if (col < a.nx * a.ny) zpart64(a, col, a.singular && col == 0);
}

// FP32 plans without a rectangle (tiny planes, or a periodic z of fewer than 32 planes): the
// singular column in double-float by one warp
__global__ void __launch_bounds__(32) zsingular_kernel(ZArgs<float> a) {
  pdl_wait();
  if (a.skip && *a.skip) return;
  extern __shared__ __align__(16) float2 zsm[];
  zcolumn_df(a, 0, zsm, zsm + a.nz);
}

cudaError_t launch_zsolve64(ZArgs<double> a, cudaStream_t st) {
  const int ncol = a.nx * a.ny;
  if (warp_columns(ncol, a.nz) && (!a.periodic || a.nz >= 32))
    return launch_k(zpart64_kernel, (ncol + 3) / 4, 128, 0, st, a);
  return launch_k(zsolve64_kernel, (ncol + 127) / 128 + (a.singular ? 1 : 0), 128, 0, st, a);
}

cudaError_t launch_zsingular(ZArgs<float> a, cudaStream_t st) {
  const size_t smem = 2 * (size_t)a.nz * sizeof(float2);
  auto k = zsingular_kernel;
  // (for n_z = 8192, whatever this plan takes: another thread may set it before this launch)
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 2 * 8192 * (int)sizeof(float2));
  if (e != cudaSuccess) return e;
  return launch_k(k, 1, 32, smem, st, a);
}

}  // namespace ps
