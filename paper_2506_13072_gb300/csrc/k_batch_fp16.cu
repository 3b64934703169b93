// k_batch_fp16.cu -- batched D2Q9 step kernels with __half storage.
#include "fvlb_batch_impl.cuh"

namespace fvlb {
template cudaError_t batch_step_impl<__half>(const BatchLaunch&);
template void batch_maps_impl<__half>(StageMaps*, int, const void*, const void*, const void*, long long);
template void batch_inst_fill_impl<__half>(void*, int, int, int, long long, double, double, double,
                                       double, int, const double*, double, const void*, long long,
                                       long long, long long, unsigned*);
}  // namespace fvlb
