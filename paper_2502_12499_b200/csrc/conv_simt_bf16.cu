#include "conv_simt_launch.cuh"
namespace ckpt {
namespace simt {
template int launch<__nv_bfloat16>(int, const ConvGeom&, const void*, const void*, void*, const float*, int, int, int, int, bool, bool, const Plan&, const SgdUpdate&, cudaStream_t, float*);
}
}  // namespace ckpt
