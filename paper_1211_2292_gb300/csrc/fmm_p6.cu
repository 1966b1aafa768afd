// Fast multipole method kernels of expansion order 6.
#include "fmm_impl.cuh"

namespace nb {
namespace fmm {
template cudaError_t launch_fmm_order<6>(cudaStream_t, const FmmStreams &, const FmmParams &, bool,
                                         int &);
}  // namespace fmm
}  // namespace nb
