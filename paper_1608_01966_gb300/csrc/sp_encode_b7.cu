// Encoder kernels of window sizes 7 and 9 (a translation unit per pair, so
// that they compile in parallel).
#include "sp_encode_kernel.cuh"

namespace sp {
namespace enc {
template cudaError_t launch_block<7>(const EncodeArgs&, bool, cudaStream_t);
template cudaError_t launch_block<9>(const EncodeArgs&, bool, cudaStream_t);
}  // namespace enc
}  // namespace sp
