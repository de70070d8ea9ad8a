// Instances of the box step for the f32 storage format.
#include "lbm_box_impl.cuh"

namespace lbm {
namespace box {
template cudaError_t box_t<ST_F32>(const HostPhys &, const void *, void *, cudaStream_t, void *);
}  // namespace box
}  // namespace lbm
