// projection.cu — the velocity projection around the solve (Eqs. 2b–2c) and its adjoint.
//
// Staggered (MAC) grid of §2: the velocity component along an axis lives on the
// cell faces normal to that axis. Storage: each component has the cell array's
// shape [n_z][n_y][n_x]; entry i along its own axis is the face on the low side
// of cell i. On a periodic axis face 0 is the wrap face; on a Neumann-pressure
// axis (prescribed velocity, end of §2) face 0 is the wall (its value is
// carried through unchanged) and the high wall is implicit.
//
//   D u   (cell):  Σ_axes (u[i+1] − u[i]) / Δ_i, wall faces excluded
//   G φ   (face):  (φ[i] − φ[i−1]) / Δc_{i−1} on interior/periodic faces, 0 on walls
// with Δ_i the cell width and Δc the centre distance (Δz^f, Δz^c on the stretched
// z; the periodic wrap distance is (Δ_0 + Δ_{n−1})/2). D·G is the operator of
// Eq. 4. The projection (γΔt cancels): u = u* − G A⁻¹ D u*. Its vector–Jacobian
// product: ḡ* = ḡ − Dᵀ A⁻ᵀ Gᵀ ḡ, with
//   (Gᵀ g)[c] = Σ_axes g[i]/Δc_{i−1} − g[i+1]/Δc_i      (interior/periodic faces)
//   (Dᵀ s)[face i] = s[i−1]/Δ_{i−1} − s[i]/Δ_i         (interior/periodic faces; 0 on walls)
// Only P and NN axes are supported (the pressure BCs of periodic and wall axes).
#include "internal.h"

namespace ps {

// ProjArgs (internal.h): per[] = axis periodic; idx, idy = 1/Δx, 1/Δy; idzf[k] = 1/Δz^f_k;
// idzc[k] = 1/(centre distance between cells k−1 and k), idzc[0] = the periodic wrap.

// A row (j, k), or on few rows a part of one, per group of threadIdx.x, V consecutive cells a
// thread (16-byte accesses when n_x and the pointers allow, else V = 1): the ends of y and z are decided once per row, those
// of x for one cell of it, and no cell pays a division. The fused multiply-adds are written out:
// both widths then give the same bits. Bound by HBM in FP32 and by the FP64
// pipe in FP64 (6 instructions a cell and kernel, 627 G/s on this part). Measured on
// 512×256×256 against one cell per thread with the indices divided out, in µs: FP32 divergence
// 144 → 82, gradient 181 → 136, adjoints 186 → 81 and 244 → 135 (6.5 TB/s); FP64 391 → 380,
// 468 → 381, 401 → 372 and 577 → 445.
template <class T, int V>
struct alignas(sizeof(T) * V) CellVec {
  T v[V];
};
template <class T, int V>
__device__ __forceinline__ CellVec<T, V> ld_cells(const T* p) { return *reinterpret_cast<const CellVec<T, V>*>(p); }
template <class T, int V>
__device__ __forceinline__ void st_cells(T* p, const CellVec<T, V>& x) { *reinterpret_cast<CellVec<T, V>*>(p) = x; }

// One row and its neighbours: offsets to the rows above and below along y and z (wrapped),
// and whether they exist (a wall has none).
struct Row {
  int j, k;
  size_t base;                 // first cell
  long long yp, ym, zp, zm;    // offsets
  bool hyp, hym, hzp, hzm;
};
template <class T>
__device__ __forceinline__ bool row_of(const ProjArgs<T>& a, Row& r) {
  const int row = blockIdx.x * blockDim.y + threadIdx.y;
  if (row >= a.ny * a.nz) return false;
  r.k = row / a.ny;
  r.j = row - r.k * a.ny;
  const long long nx = a.nx, sxy = nx * a.ny;
  r.base = (size_t)row * nx;
  r.hyp = r.j + 1 < a.ny || a.per[1];
  r.hym = r.j > 0 || a.per[1];
  r.hzp = r.k + 1 < a.nz || a.per[2];
  r.hzm = r.k > 0 || a.per[2];
  r.yp = r.j + 1 < a.ny ? nx : (a.per[1] ? -(a.ny - 1) * nx : 0);
  r.ym = r.j > 0 ? -nx : (a.per[1] ? (a.ny - 1) * nx : 0);
  r.zp = r.k + 1 < a.nz ? sxy : (a.per[2] ? -(a.nz - 1) * sxy : 0);
  r.zm = r.k > 0 ? -sxy : (a.per[2] ? (a.nz - 1) * sxy : 0);
  return true;
}

template <class T, int V>
__global__ void __launch_bounds__(256) div_kernel(ProjArgs<T> a, const T* __restrict__ u, T* __restrict__ f) {
  pdl_wait();
  Row r;
  if (!row_of(a, r)) return;
  const size_t N = (size_t)a.nx * a.ny * a.nz;
  const T* __restrict__ ux = u + r.base;
  const T* __restrict__ uy = u + N + r.base;
  const T* __restrict__ uz = u + 2 * N + r.base;
  const T idz = a.idzf[r.k];
  for (int i = (blockIdx.y * blockDim.x + threadIdx.x) * V; i < a.nx; i += gridDim.y * blockDim.x * V) {
    const auto x = ld_cells<T, V>(ux + i), yl = ld_cells<T, V>(uy + i), zl = ld_cells<T, V>(uz + i);
    const auto yh = ld_cells<T, V>(uy + r.yp + i), zh = ld_cells<T, V>(uz + r.zp + i);
    const T xn = (i + V < a.nx) ? ux[i + V] : (a.per[0] ? ux[0] : (T)0);
    CellVec<T, V> o;
#pragma unroll
    for (int e = 0; e < V; ++e) {
      const T hx = e + 1 < V ? x.v[e + 1 < V ? e + 1 : 0] : xn;
      const T lx = (e > 0 || i > 0 || a.per[0]) ? x.v[e] : (T)0;
      const T hy = r.hyp ? yh.v[e] : (T)0, ly = r.hym ? yl.v[e] : (T)0;
      const T hz = r.hzp ? zh.v[e] : (T)0, lz = r.hzm ? zl.v[e] : (T)0;
      o.v[e] = fma(hz - lz, idz, fma(hy - ly, a.idy, (hx - lx) * a.idx));
    }
    st_cells<T, V>(f + r.base + i, o);
  }
}

// u = u* − G φ (all three components)
template <class T, int V>
__global__ void __launch_bounds__(256) grad_correct_kernel(ProjArgs<T> a, const T* us, const T* __restrict__ phi, T* u) {
  pdl_wait();
  Row r;
  if (!row_of(a, r)) return;
  const size_t N = (size_t)a.nx * a.ny * a.nz;
  const T* __restrict__ p = phi + r.base;
  const T idz = a.idzc[r.k];
  for (int i = (blockIdx.y * blockDim.x + threadIdx.x) * V; i < a.nx; i += gridDim.y * blockDim.x * V) {
    const auto pc = ld_cells<T, V>(p + i), py = ld_cells<T, V>(p + r.ym + i), pz = ld_cells<T, V>(p + r.zm + i);
    const bool hxm = i > 0 || a.per[0];
    const T px = i > 0 ? p[i - 1] : (a.per[0] ? p[a.nx - 1] : (T)0);
    const size_t g = r.base + i;
    auto x = ld_cells<T, V>(us + g), y = ld_cells<T, V>(us + N + g), z = ld_cells<T, V>(us + 2 * N + g);
#pragma unroll
    for (int e = 0; e < V; ++e) {
      if (e > 0 || hxm) x.v[e] = fma((e > 0 ? pc.v[e > 0 ? e - 1 : 0] : px) - pc.v[e], a.idx, x.v[e]);
      if (r.hym) y.v[e] = fma(py.v[e] - pc.v[e], a.idy, y.v[e]);
      if (r.hzm) z.v[e] = fma(pz.v[e] - pc.v[e], idz, z.v[e]);
    }
    st_cells<T, V>(u + g, x);
    st_cells<T, V>(u + N + g, y);
    st_cells<T, V>(u + 2 * N + g, z);
  }
}

// h = Gᵀ g (cells)
template <class T, int V>
__global__ void __launch_bounds__(256) grad_adjoint_kernel(ProjArgs<T> a, const T* __restrict__ gu, T* __restrict__ h) {
  pdl_wait();
  Row r;
  if (!row_of(a, r)) return;
  const size_t N = (size_t)a.nx * a.ny * a.nz;
  const T* __restrict__ gx = gu + r.base;
  const T* __restrict__ gy = gu + N + r.base;
  const T* __restrict__ gz = gu + 2 * N + r.base;
  const T dl = a.idzc[r.k], dh = a.idzc[r.k + 1 < a.nz ? r.k + 1 : 0];
  for (int i = (blockIdx.y * blockDim.x + threadIdx.x) * V; i < a.nx; i += gridDim.y * blockDim.x * V) {
    const auto x = ld_cells<T, V>(gx + i), yl = ld_cells<T, V>(gy + i), zl = ld_cells<T, V>(gz + i);
    const auto yh = ld_cells<T, V>(gy + r.yp + i), zh = ld_cells<T, V>(gz + r.zp + i);
    const bool hxp = i + V < a.nx || a.per[0];
    const T xn = (i + V < a.nx) ? gx[i + V] : (a.per[0] ? gx[0] : (T)0);
    CellVec<T, V> o;
#pragma unroll
    for (int e = 0; e < V; ++e) {
      T v = 0;
      // own low face (i) contributes +g/Δc, high face (i+1) contributes −g/Δc
      if (e > 0 || i > 0 || a.per[0]) v = x.v[e] * a.idx;
      if (e + 1 < V || hxp) v = fma(-(e + 1 < V ? x.v[e + 1 < V ? e + 1 : 0] : xn), a.idx, v);
      if (r.hym) v = fma(yl.v[e], a.idy, v);
      if (r.hyp) v = fma(-yh.v[e], a.idy, v);
      if (r.hzm) v = fma(zl.v[e], dl, v);
      if (r.hzp) v = fma(-zh.v[e], dh, v);
      o.v[e] = v;
    }
    st_cells<T, V>(h + r.base + i, o);
  }
}

// ḡ* = ḡ − Dᵀ s (faces)
template <class T, int V>
__global__ void __launch_bounds__(256) div_adjoint_correct_kernel(ProjArgs<T> a, const T* gu, const T* __restrict__ s_,
                                                                  T* out) {
  pdl_wait();
  Row r;
  if (!row_of(a, r)) return;
  const size_t N = (size_t)a.nx * a.ny * a.nz;
  const T* __restrict__ s = s_ + r.base;
  const T wm = a.idzf[r.k > 0 ? r.k - 1 : a.nz - 1], wc = a.idzf[r.k];
  for (int i = (blockIdx.y * blockDim.x + threadIdx.x) * V; i < a.nx; i += gridDim.y * blockDim.x * V) {
    // face i lies between cell i−1 (contributes s/Δ) and cell i (−s/Δ)
    const auto sc = ld_cells<T, V>(s + i), sy = ld_cells<T, V>(s + r.ym + i), sz = ld_cells<T, V>(s + r.zm + i);
    const bool hxm = i > 0 || a.per[0];
    const T sx = i > 0 ? s[i - 1] : (a.per[0] ? s[a.nx - 1] : (T)0);
    const size_t g = r.base + i;
    auto x = ld_cells<T, V>(gu + g), y = ld_cells<T, V>(gu + N + g), z = ld_cells<T, V>(gu + 2 * N + g);
#pragma unroll
    for (int e = 0; e < V; ++e) {
      if (e > 0 || hxm) x.v[e] = fma(sc.v[e] - (e > 0 ? sc.v[e > 0 ? e - 1 : 0] : sx), a.idx, x.v[e]);
      if (r.hym) y.v[e] = fma(sc.v[e] - sy.v[e], a.idy, y.v[e]);
      if (r.hzm) z.v[e] = z.v[e] - fma(sz.v[e], wm, -(sc.v[e] * wc));
    }
    st_cells<T, V>(out + g, x);
    st_cells<T, V>(out + N + g, y);
    st_cells<T, V>(out + 2 * N + g, z);
  }
}

namespace {
template <class T, int V>
cudaError_t launch_op(int op, const ProjArgs<T>& a, const T* a0, const T* a1, T* o, cudaStream_t st) {
  int tx = 1;  // threads of a row: a power of two, a warp at most
  while (tx < 32 && tx * V < a.nx) tx *= 2;
  const dim3 block(tx, 256 / tx);
  const unsigned rows = (unsigned)(((long long)a.ny * a.nz + block.y - 1) / block.y);
  // rows too few for eight CTAs an SM are cut along x, down to one vector a thread: a thread's
  // vectors are a chain of load latencies (FP64 divergence and gradient of 3072×4×2, µs: 98 in one
  // part, 13 in parts)
  const unsigned parts = (unsigned)((a.nx + tx * V - 1) / (tx * V)), want = 8 * kSMs / rows;
  const dim3 grid(rows, want < 1 ? 1 : (want < parts ? want : parts));
  switch (op) {
    case 0: return launch_k(div_kernel<T, V>, grid, block, 0, st, a, a0, o);
    case 1: return launch_k(grad_correct_kernel<T, V>, grid, block, 0, st, a, a0, a1, o);
    case 2: return launch_k(grad_adjoint_kernel<T, V>, grid, block, 0, st, a, a0, o);
    default: return launch_k(div_adjoint_correct_kernel<T, V>, grid, block, 0, st, a, a0, a1, o);
  }
}
}  // namespace

template <class T>
cudaError_t launch_projection(int op, const ProjArgs<T>& a, const void* x0, const void* x1, void* y,
                              cudaStream_t st) {
  constexpr int V = 16 / (int)sizeof(T);
  const T* a0 = static_cast<const T*>(x0);
  const T* a1 = static_cast<const T*>(x1);
  T* o = static_cast<T*>(y);
  const bool vec = a.nx % V == 0 && !(((uintptr_t)x0 | (uintptr_t)x1 | (uintptr_t)y) & 15);
  return vec ? launch_op<T, V>(op, a, a0, a1, o, st) : launch_op<T, 1>(op, a, a0, a1, o, st);
}

template cudaError_t launch_projection<float>(int, const ProjArgs<float>&, const void*, const void*, void*, cudaStream_t);
template cudaError_t launch_projection<double>(int, const ProjArgs<double>&, const void*, const void*, void*, cudaStream_t);

}  // namespace ps
