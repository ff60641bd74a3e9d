// sweep_unpack.cu -- the unpack specializations of the body sweep (sweep_impl.cuh).
#include "sweep_impl.cuh"

namespace frk {

cudaError_t configure_sweep_unpack() { return configure_mode<kModeUnpack>(); }

cudaError_t launch_sweep_unpack(const SweepParams& p, int n_ctas, cudaStream_t s) {
  return launch_mode<kModeUnpack>(p, n_ctas, s);
}

cudaError_t launch_list_unpack(const ListParams& p, cudaStream_t s) { return launch_list<kModeUnpack>(p, s); }

}  // namespace frk
