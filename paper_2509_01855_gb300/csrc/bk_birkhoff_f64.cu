// FP64 instances of the Birkhoff transform templates (every FP64 transform kernel), compiled in
// their own translation unit so that the library builds in parallel. The definitions are those
// of bk_birkhoff.cu, included with its main-unit-only parts (globals, plans, entry points) left
// out.
#define BK_TRANSFORM_KERNEL_UNIT
#include "bk_birkhoff.cu"

namespace bk {

template bk_status set_smem_attrs<double>(const Plan* p);
template bool clusters_held<double>(int, size_t);
template bk_status re_attrs<double>();
template bk_status blue_spectrum<double>(Plan* p, cudaStream_t st);
template bk_status apply_batch_impl<double>(const Plan* const*, const void* const*, void* const*, const int*, int,
                                        const Plan* const*, const void* const*, void* const*, const int*, int, bool,
                                        cudaStream_t);
template bk_status apply_impl<double>(const Plan* p, const double* v, double* out, int nvec, bool trans, double s_scale,
                                     cudaStream_t st);

}  // namespace bk
