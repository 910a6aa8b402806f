// Persistent rollout instantiations, 4 particles per thread, up to 128 threads
// per filter.
#include "rollout_persistent.cuh"

namespace ut {
namespace persist {

cudaError_t launch_ppt4_wide(int nt, const EnvDev& d, int T, cudaStream_t s);  // rollout_persistent_c.cu

cudaError_t launch_ppt4(int nt, const EnvDev& d, int T, cudaStream_t s) {
  switch (nt) {
    case 32: return launch_shape<32, 4>(d, T, s);
    case 64: return launch_shape<64, 4>(d, T, s);
    case 128: return launch_shape<128, 4>(d, T, s);
    default: return launch_ppt4_wide(nt, d, T, s);
  }
}

}  // namespace persist
}  // namespace ut
