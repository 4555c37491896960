// The two-tile encoder kernels with selection and solver warps for 9 to 16
// atoms per signal.
#include "encode_core.cuh"

namespace dlsh {
namespace enc {

template int launch_split<true, 2, 128, 16>(const SplitArgs&, int, cudaStream_t);
template int launch_split<true, 2, 64, 16>(const SplitArgs&, int, cudaStream_t);

}  // namespace enc
}  // namespace dlsh
