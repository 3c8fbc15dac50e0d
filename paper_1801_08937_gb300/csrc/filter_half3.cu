// Instantiations of the three-pass whole-block float32 filter (filter_half3.cuh).
#include "filter_half3.cuh"

namespace mm {

bool half3_shape(int M, int* r0, int* r1) {
    switch (M) {
        case 9216: *r0 = 32; *r1 = 32; return true;
        case 4608: *r0 = 32; *r1 = 16; return true;
        case 2304: *r0 = 16; *r1 = 16; return true;
        default: return false;
    }
}

template <typename H, bool FROM_TOD, bool EVEN>
static void launch_h3(const FilterArgs& a, cudaStream_t s) {
    constexpr size_t sm = H::BUF;
    static std::atomic<size_t> configured{0};
    static std::atomic<int> resident{0};
    raise_smem_once(configured, sm, [](size_t v) {
        configure_smem(k_filter_half3<H, FROM_TOD, EVEN>, v, H::NT);
        int per_sm = 0, dev = 0, sms = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_filter_half3<H, FROM_TOD, EVEN>, H::NT, v);
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        resident.store(std::max(1, per_sm * sms));
    });
    FilterArgs f = a;
    f.ahead = resident.load();
    k_filter_half3<H, FROM_TOD, EVEN><<<a.n_work, H::NT, sm, s>>>(f);
    count_launches(1);
}
template <typename H>
static void launch_h3_any(const FilterArgs& a, bool from_tod, cudaStream_t s) {
    if (from_tod) launch_h3<H, true, false>(a, s);
    else if (a.even) launch_h3<H, false, true>(a, s);
    else launch_h3<H, false, false>(a, s);
}

void launch_filter_half3(const FilterArgs& a, bool from_tod, cudaStream_t s) {
    if (a.n_work <= 0) return;
    switch (a.L) {
        case 9216: return launch_h3_any<H3<32, 32>>(a, from_tod, s);
        case 4608: return launch_h3_any<H3<32, 16>>(a, from_tod, s);
        default: return launch_h3_any<H3<16, 16>>(a, from_tod, s);
    }
}

}  // namespace mm
