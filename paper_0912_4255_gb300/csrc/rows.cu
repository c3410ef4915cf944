// Second FFT pass instantiations for one (precision, log2 N2), selected at
// build time by FS_REAL and FS_L2 (6..12).
#include "passes.cuh"

#ifndef FS_REAL
#define FS_REAL float
#endif
#ifndef FS_L2
#define FS_L2 11
#endif

#define FS_CAT2(a, b, c) a##_##b##_##c
#define FS_CAT(a, b, c) FS_CAT2(a, b, c)

namespace fs {

cudaError_t FS_CAT(rows, FS_REAL, FS_L2)(const RowsArgs<FS_REAL>& a, int inplace, dim3 grid, cudaStream_t s) {
  using R = FS_REAL;
  constexpr int L2 = FS_L2;
  constexpr int RR = rows_for<R>(L2);
  constexpr int NT = threads_for<R>(L2, RR);
  constexpr size_t SM = rows_smem<R, L2, RR>();
  auto kern = inplace ? (a.band ? k_rows<R, L2, RR, NT, true, true> : k_rows<R, L2, RR, NT, false, true>)
                      : (a.band ? k_rows<R, L2, RR, NT, true, false> : k_rows<R, L2, RR, NT, false, false>);
  // persistent grid: the blocks that fit on the device at once
  static DeviceOnce once[4];
  int resident = 0;
  const cudaError_t e = kernel_setup(once[(a.band ? 1 : 0) + (inplace ? 2 : 0)], kern, NT, SM, &resident);
  if (e != cudaSuccess) return e;
  if (resident < 1) resident = 1;
  const unsigned total = grid.x * grid.y;
  const dim3 blocks(total < (unsigned)resident ? total : (unsigned)resident);
  return launch_after(starts_early<R>((int64_t)total * (RR << L2)), kern, blocks, NT, SM, s, a);
}
int FS_CAT(rowsR, FS_REAL, FS_L2)() { return rows_for<FS_REAL>(FS_L2); }

}  // namespace fs
