// kern_mixed.cu -- engine kernels with FP32 forces and FP64 position/velocity accumulation.
#define DSDNA_KERN_MIXED 1   // the single force evaluation exists in mixed precision only
#include "kern_launch.cuh"
namespace dsdna {
template cudaError_t engine_occupancy<float>(int, int, int*, size_t*);
template cudaError_t engine_launch<float>(int, const KArgs<float>&, int, int, size_t, cudaStream_t);
template cudaError_t rebuild_launch<float>(const KArgs<float>&, int, cudaStream_t);
template cudaError_t rebuild_prepare<float>();
template cudaError_t resident_shape<float>(int64_t, int, bool, int, int*, int*, size_t*);
template cudaError_t resident_launch<float>(int, const KArgs<float>&, int, int, size_t, cudaStream_t);
}  // namespace dsdna
