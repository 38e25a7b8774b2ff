// xform.cu — launchers of the generic line transforms (device code in xform_dev.cuh).
#include "xform_mid.cuh"

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

namespace {
// Half lengths with a compile-time kernel (xform_mid_*.cu).
template <class TI, class TO, int AXIS, bool FWD, int M>
cudaError_t mid_case(const XformArgs<float>& a, cudaStream_t st, bool* done) {
  const int L = mid::DimCt<M>::L;
  const long long tiles = AXIS == 0 ? (a.nlines + L - 1) / L : (long long)a.nz * ((a.nx + L - 1) / L);
  if (tiles < kSMs || (AXIS == 1 && tiles * L > 2LL * a.nz * a.nx)) return cudaSuccess;
  *done = true;
  return launch_xform_mid<TI, TO, M, AXIS, FWD>(a, (int)tiles, st);
}
// FP32 lines: the kernel with the length at compile time, where the grid gives every SM a
// tile of it and no more than half of a plane's tiles' columns are idle (else the run-time
// kernel, whose tiles shrink with the grid: 2 columns of 972, 4096 planes: 489 → 96 µs).
// 384×288×201 in µs, run-time → compile-time length: x 97 → 73 forward, 99 → 75 backward (into
// FP32 Φ_0), 160 → 136 (into p), y 113 → 54 and 105 → 56; 192×96×65 solve 45 → 32.
template <class TI, class TO, int AXIS, bool FWD>
cudaError_t launch_mid_if(const XformArgs<float>& a, cudaStream_t st, bool* done) {
  *done = false;
  if (a.bc == BC_FD) return cudaSuccess;
  switch (a.m) {
#define PS_MID_CASE(M) \
  case M: return mid_case<TI, TO, AXIS, FWD, M>(a, st, done);
    PS_MID_CASE(16) PS_MID_CASE(18) PS_MID_CASE(24) PS_MID_CASE(27) PS_MID_CASE(32) PS_MID_CASE(36) PS_MID_CASE(48)
    PS_MID_CASE(54) PS_MID_CASE(72) PS_MID_CASE(81) PS_MID_CASE(96) PS_MID_CASE(108) PS_MID_CASE(144)
    PS_MID_CASE(162) PS_MID_CASE(192) PS_MID_CASE(216) PS_MID_CASE(243) PS_MID_CASE(288) PS_MID_CASE(324)
    PS_MID_CASE(384) PS_MID_CASE(432) PS_MID_CASE(486)
#undef PS_MID_CASE
    default: return cudaSuccess;
  }
}
}  // namespace

// Lines per tile: 16 (a 64-byte row segment of FP32 y lines, full half-warps) while four
// CTAs fit an SM (56 KB each); fewer on long lines, down to four (FP32: one 16-byte part of
// a sector), and below that where only one such CTA would fit an SM (its 256 threads then
// wait out every load and FP64 chain alone: 4000 FP32 x lines of 4608, forward and backward,
// µs, with 4, 2 and 1 lines: 463, 329 and 254, of 7776 with 2 and 1: 946 and 454; 1400 FP64
// lines of 2592 with 4, 2 and 1: 541, 517 and 440); and fewer, down to four, while the tiles
// would leave SMs without work: on a 32^3 grid 16 lines make 64 tiles, four make 256. A tile
// of long lines (486 points or more) may go on to one line (24 FP64 x lines of 2592 with 4, 2
// and 1 lines: 185, 114 and 69 µs). More than 16 on the shortest lines, whose single butterfly
// a line (m = 16 and below) would leave half a warp idle, up to 512 points a tile (FP64 y lines
// of 6 and of 32, 1024 columns, 256 planes, forward, µs: 65 → 43 and 245 → 163). On planes of
// few columns no tile is twice as wide as the plane, and none of more than 512 points leaves
// more than a quarter of the columns' number idle (FP64, 6 columns of 1024, 1365 planes, forward
// and backward: 919 µs with tiles of four, 686 of two; 6 of 24: 40 with eight, 61 with two).
template <class T, class TI, class TO, bool FWD>
cudaError_t launch_xform(XformArgs<T> a, cudaStream_t st) {
  if constexpr (sizeof(T) == 4) {
    bool done = false;
    cudaError_t e = cudaSuccess;
    if (a.axis == 0) {
      e = launch_mid_if<TI, TO, 0, FWD>(a, st, &done);
    } else if constexpr (sizeof(TI) == 4 && sizeof(TO) == 4) {
      if (!a.accumulate) e = launch_mid_if<TI, TO, 1, FWD>(a, st, &done);
    }
    if (e != cudaSuccess || done) return e;
  }
  constexpr size_t C = sizeof(cplx<T>);
  constexpr size_t kBest = 56 * 1024, kTwo = 110 * 1024;  // four and two CTAs an SM
  auto tiles = [&](int lg) -> long long {
    const int L = 1 << lg;
    return a.axis == 0 ? (a.nlines + L - 1) / L : (long long)a.nz * ((a.nx + L - 1) / L);
  };
  int lg = 4;
  while (lg < 8 && (a.m << lg) < 512 && tiles(lg + 1) >= 4 * kSMs) ++lg;
  while (a.axis == 1 && lg > 1 &&
         ((1 << (lg - 1)) >= a.nx ||
          ((a.m << lg) > 512 && 4 * (tiles(lg) / a.nz * (1 << lg) - a.nx) > a.nx)))
    --lg;
  while (lg > 2 && tile_smem(a.m, lg, C) > kBest) --lg;
  while (lg > 0 && tile_smem(a.m, lg, C) > kTwo) --lg;
  while (lg > 0 && tiles(lg) < 2 * kSMs && (lg > 2 || (a.m << lg) >= 486)) --lg;
  a.lgL = lg;
  const size_t smem = tile_smem(a.m, lg, C);
  // a thread per eight points of the tile, in whole warps
  int threads = (((a.m << lg) / 8 + 31) / 32) * 32;
  threads = threads < 64 ? 64 : (threads > 256 ? 256 : threads);
  auto k = xform_kernel<T, TI, TO, FWD>;
  // the most a block may have, whatever this tile takes: another thread may set it before this launch
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
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
