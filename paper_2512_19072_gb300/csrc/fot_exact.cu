// The exact window kernels (fot_window.cuh).
#include "fot_window.cuh"

namespace fot {

template <int MODE, int MAXP>
void exact_launch(cudaStream_t s, const BandTable<MAXP>& t) {
  launch_dependent(exact_pass_kernel<MODE, MAXP>, dim3(t.items), kWinThreads, window_smem(t.pitch_max, 2), s, t);
}

template void exact_launch<0, 1>(cudaStream_t, const BandTable<1>&);
template void exact_launch<1, 1>(cudaStream_t, const BandTable<1>&);
template void exact_launch<0, 2>(cudaStream_t, const BandTable<2>&);
template void exact_launch<1, 2>(cudaStream_t, const BandTable<2>&);
template void exact_launch<0, kMaxBatch>(cudaStream_t, const BandTable<kMaxBatch>&);
template void exact_launch<1, kMaxBatch>(cudaStream_t, const BandTable<kMaxBatch>&);

}  // namespace fot
