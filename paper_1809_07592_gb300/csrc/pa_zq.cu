// pa_zq.cu -- word-sized exact (number-theoretic) instances of the pass kernels and launchers.
#include "pa_launch.cuh"

namespace pa {
PA_INSTANTIATE_LAUNCHERS(Zq)
}  // namespace pa
