// First FFT pass instantiations for one (precision, log2 N1), selected at
// build time by FS_REAL (float|double) and FS_L1 (6..12); the build compiles
// this file once per pair so that the units compile in parallel.
#include "passes.cuh"

#ifndef FS_REAL
#define FS_REAL float
#endif
#ifndef FS_L1
#define FS_L1 11
#endif

#define FS_CAT2(a, b, c) a##_##b##_##c
#define FS_CAT(a, b, c) FS_CAT2(a, b, c)

namespace fs {

namespace {
template <typename R, int L1, int SRC>
cudaError_t run(const ColsArgs<R>& a, dim3 grid, cudaStream_t s) {
  constexpr int C = cols_for<points_a<R>()>(L1);
  constexpr int NT = threads_for<R>(L1, C);
  constexpr size_t SM = cols_smem<R, L1, C>();
  auto kern = k_cols<R, L1, C, NT, SRC, 8>;
  // persistent grid: the blocks that fit on the device at once
  static DeviceOnce once;
  int resident = 0;
  const cudaError_t e = kernel_setup(once, kern, NT, SM, &resident);
  if (e != cudaSuccess) return e;
  if (resident < 1) resident = 1;
  const unsigned total = grid.x * grid.y;
  const unsigned cap = (unsigned)resident;
  return launch_after(starts_early<R>((int64_t)total * (C << L1)), kern, dim3(total < cap ? total : cap), NT, SM, s, a);
}
}  // namespace

cudaError_t FS_CAT(cols, FS_REAL, FS_L1)(const ColsArgs<FS_REAL>& a, int inplace, dim3 grid, cudaStream_t s) {
  return inplace ? run<FS_REAL, FS_L1, SRC_INPLACE>(a, grid, s) : run<FS_REAL, FS_L1, SRC_LOAD>(a, grid, s);
}
int FS_CAT(colsC, FS_REAL, FS_L1)() { return cols_for<points_a<FS_REAL>()>(FS_L1); }

}  // namespace fs
