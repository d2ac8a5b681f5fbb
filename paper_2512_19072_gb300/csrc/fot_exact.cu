// Exact passes: plan and sums of 2 rows per CTA in one kernel (fot_small.cuh).
#include "fot_small.cuh"

namespace fot {

template <int MODE, int MAXP>
void small_exact_launch(cudaStream_t s, const BandTable<MAXP>& t) {
  launch_small<MODE, kFormFp32, 2>(s, t);
}

template void small_exact_launch<0, 1>(cudaStream_t, const BandTable<1>&);
template void small_exact_launch<1, 1>(cudaStream_t, const BandTable<1>&);
template void small_exact_launch<0, 2>(cudaStream_t, const BandTable<2>&);
template void small_exact_launch<1, 2>(cudaStream_t, const BandTable<2>&);
template void small_exact_launch<0, kMaxBatch>(cudaStream_t, const BandTable<kMaxBatch>&);
template void small_exact_launch<1, kMaxBatch>(cudaStream_t, const BandTable<kMaxBatch>&);

template <int MAXP>
static cudaError_t configure(int bytes) {
  const cudaError_t e = cudaFuncSetAttribute(small_pass_kernel<0, kFormFp32, 2, MAXP>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(small_pass_kernel<1, kFormFp32, 2, MAXP>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}
cudaError_t small_exact_configure(int bytes) {
  cudaError_t e = configure<1>(bytes);
  if (e == cudaSuccess) e = configure<2>(bytes);
  if (e == cudaSuccess) e = configure<kMaxBatch>(bytes);
  return e;
}

}  // namespace fot
