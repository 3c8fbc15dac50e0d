// float64 instantiations of the fused filter kernels (kernels in filter_impl.cuh).
#include "filter_impl.cuh"

namespace mm {

void launch_filter_fft_f64(const FilterArgs& a, bool from_tod, cudaStream_t s) {
    if (a.split) {
        if (from_tod) launch_split_t<true>(a, s);
        else launch_split_t<false>(a, s);
    } else if (a.half) {
        if (from_tod) launch_half_t<double, true>(a, s);
        else launch_half_t<double, false>(a, s);
    } else {
        if (from_tod) launch_fft_t<double, true>(a, s);
        else launch_fft_t<double, false>(a, s);
    }
}
void launch_filter_direct_f64(const FilterArgs& a, bool from_tod, cudaStream_t s) {
    if (from_tod) launch_direct_t<double, true>(a, s);
    else launch_direct_t<double, false>(a, s);
}

}  // namespace mm
