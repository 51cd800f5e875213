// Per-element statistics and conditional means, FP64 form (kernels in bins_impl.cuh).
#include "bins_impl.cuh"

namespace pdfx {

template <>
void launch_stats_tiles<double>(const StatsArgs<double>& a, int num_sms, cudaStream_t s_small, cudaStream_t s_mid,
                               cudaStream_t s_large) {
  launch_stats_tiles_impl<double>(a, num_sms, s_small, s_mid, s_large);
}

template <>
void launch_stats_small<double>(const StatsArgs<double>& a, bool medium, cudaStream_t s) {
  launch_stats_small_impl<double>(a, medium, s);
}

}  // namespace pdfx
