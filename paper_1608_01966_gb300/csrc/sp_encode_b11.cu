// Encoder kernels of window sizes 11 and 13 (a translation unit per pair, so
// that they compile in parallel).
#include "sp_encode_kernel.cuh"

namespace sp {
namespace enc {
template cudaError_t launch_block<11>(const EncodeArgs&, bool, cudaStream_t);
template cudaError_t launch_block<13>(const EncodeArgs&, bool, cudaStream_t);
}  // namespace enc
}  // namespace sp
