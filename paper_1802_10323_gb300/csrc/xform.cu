// xform.cu — launchers of the generic line transforms (device code in xform_dev.cuh).
#include "xform_dev.cuh"

namespace ps {

template <class T, class TI, class TO, bool FWD>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 4 : 2) xform_kernel(XformArgs<T> a) {
  pdl_wait();
  if (a.skip && *a.skip) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  xform_group<T, TI, TO, FWD>(a, blockIdx.x, smem_raw);
}

// ---- host-side launcher ------------------------------------------------------------------

namespace {
size_t tile_smem(int m, int lgL, size_t csize) {
  const size_t ls = lgL ? (size_t)(1 << lgL) + 1 : 1;
  return 2 * (size_t)(m + 1) * ls * csize;
}
}  // namespace

// Lines per tile: 16 (a 64-byte row segment of FP32 y lines, full half-warps) while four
// CTAs fit an SM (56 KB each); fewer on long lines, down to four (FP32: one 16-byte part of
// a sector) as long as a CTA's shared memory holds them; and fewer, down to four, while the
// tiles would leave SMs without work: on a 32^3 grid 16 lines make 64 tiles, four make 256.
template <class T, class TI, class TO, bool FWD>
cudaError_t launch_xform(XformArgs<T> a, cudaStream_t st) {
  constexpr size_t C = sizeof(cplx<T>);
  constexpr size_t kBest = 56 * 1024, kMost = 220 * 1024;
  auto tiles = [&](int lg) -> long long {
    const int L = 1 << lg;
    return a.axis == 0 ? (a.nlines + L - 1) / L : (long long)a.nz * ((a.nx + L - 1) / L);
  };
  int lg = 4;
  while (lg > 2 && tile_smem(a.m, lg, C) > kBest) --lg;
  while (lg > 0 && tile_smem(a.m, lg, C) > kMost) --lg;
  while (lg > 2 && tiles(lg) < 2 * 152) --lg;
  a.lgL = lg;
  const size_t smem = tile_smem(a.m, lg, C);
  // a thread per eight points of the tile, in whole warps
  int threads = (((a.m << lg) / 8 + 31) / 32) * 32;
  threads = threads < 64 ? 64 : (threads > 256 ? 256 : threads);
  auto k = xform_kernel<T, TI, TO, FWD>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_k(k, (unsigned)tiles(lg), threads, smem, st, a);
}

template cudaError_t launch_xform<double, double, double, true>(XformArgs<double>, cudaStream_t);
template cudaError_t launch_xform<double, double, double, false>(XformArgs<double>, cudaStream_t);
template cudaError_t launch_xform<float, float, float, true>(XformArgs<float>, cudaStream_t);
template cudaError_t launch_xform<float, float, float, false>(XformArgs<float>, cudaStream_t);
template cudaError_t launch_xform<float, double, float, true>(XformArgs<float>, cudaStream_t);
template cudaError_t launch_xform<float, float, double, false>(XformArgs<float>, cudaStream_t);

}  // namespace ps
