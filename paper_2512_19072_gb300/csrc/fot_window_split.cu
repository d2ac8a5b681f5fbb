// The window kernels (fot_window.cuh) and one-kernel passes (fot_small.cuh) of one operand form, in
// a translation unit of its own so that the forms compile in parallel.
#include "fot_small.cuh"

namespace fot {

template <int MODE, int FORM, int MAXP>
void window_launch(cudaStream_t s, const BandTable<MAXP>& t) {
  launch_dependent(window_pass_kernel<MODE, FORM, MAXP>, dim3(t.items), kWinThreads, window_smem(t.pitch_max), s, t);
}

template void window_launch<0, kFormSplit, 1>(cudaStream_t, const BandTable<1>&);
template void window_launch<1, kFormSplit, 1>(cudaStream_t, const BandTable<1>&);
template void window_launch<0, kFormSplit, 2>(cudaStream_t, const BandTable<2>&);
template void window_launch<1, kFormSplit, 2>(cudaStream_t, const BandTable<2>&);
template void window_launch<0, kFormSplit, kMaxBatch>(cudaStream_t, const BandTable<kMaxBatch>&);
template void window_launch<1, kFormSplit, kMaxBatch>(cudaStream_t, const BandTable<kMaxBatch>&);

template <int MODE, int FORM, int MAXP>
void small_launch(cudaStream_t s, const BandTable<MAXP>& t) {
  launch_small<MODE, FORM, 8>(s, t);
}

template void small_launch<0, kFormSplit, 1>(cudaStream_t, const BandTable<1>&);
template void small_launch<1, kFormSplit, 1>(cudaStream_t, const BandTable<1>&);
template void small_launch<0, kFormSplit, 2>(cudaStream_t, const BandTable<2>&);
template void small_launch<1, kFormSplit, 2>(cudaStream_t, const BandTable<2>&);

}  // namespace fot
