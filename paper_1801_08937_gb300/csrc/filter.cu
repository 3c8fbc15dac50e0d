// Set-up kernels of the filter (spectra, pointing weights) and the launch counter.
#include "filter_impl.cuh"

namespace mm {

static long long g_launches = 0;
long long launches_total() { return __atomic_load_n(&g_launches, __ATOMIC_RELAXED); }
void count_launches(int n) { __atomic_fetch_add(&g_launches, (long long)n, __ATOMIC_RELAXED); }
std::mutex& smem_config_mutex() {
    static std::mutex m;
    return m;
}

// ---------------- setup kernels ----------------
__global__ void k_fft_spectrum(const double* h, double* H, C2<double>* work, const C2<double>* tw,
                               const FftPasses fp) {
    const int L = fp.L;
    C2<double>* s = work + (int64_t)blockIdx.x * (L + (L >> 4));
    const double* hb = h + (int64_t)blockIdx.x * L;
    for (int i = threadIdx.x; i < L; i += blockDim.x) s[sidx(i)] = C2<double>{hb[i], 0.0};
    __syncthreads();
    fft_dif<double>(s, tw, fp);
    const double inv = 1.0 / (double)L;
    for (int i = threadIdx.x; i < L; i += blockDim.x) H[(int64_t)blockIdx.x * L + i] = s[sidx(i)].x * inv;
}

__global__ void k_weights64(const float* psi, double2* cs, int64_t n) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        double sn, c;
        sincos(2.0 * (double)psi[t], &sn, &c);
        cs[t] = make_double2(c, sn);
    }
}

// Double-float weights (cos 2psi, sin 2psi) from the float64 table.
__global__ void k_weights_df(const double2* cs, float4* out, int64_t n) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const double2 v = cs[t];
        const df c(v.x), s(v.y);
        out[t] = make_float4(c.hi, c.lo, s.hi, s.lo);
    }
}
__global__ void k_map_to_df(const V4<double>* src, V4<df>* dst, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const V4<double> v = src[i];
        dst[i] = V4<df>{df(v.x), df(v.y), df(v.z), df(0.0)};
    }
}

// Smallest and largest pixel of each block, and the range check of the
// pointing, in one pass over pix (DRAM-bound; slices of WIN_SLICE samples so a
// few long blocks still fill the device).
constexpr int WIN_SLICE = 16384;
__global__ void k_window_init(int2* win, int n) {
    const int b = blockIdx.x * blockDim.x + threadIdx.x;
    if (b < n) win[b] = make_int2(0x7fffffff, -1);
}
__global__ void __launch_bounds__(256) k_block_windows(const int32_t* __restrict__ pix, const int64_t* __restrict__ off,
                                                       int n_pix, int2* win, int* bad) {
    const int b = blockIdx.x;
    const int64_t o1 = off[b + 1];
    const int64_t t0 = off[b] + (int64_t)blockIdx.y * WIN_SLICE, t1 = t0 + WIN_SLICE < o1 ? t0 + WIN_SLICE : o1;
    if (t0 >= t1) return;
    int lo = 0x7fffffff, hi = -1;
    bool ok = true;
    auto take = [&](int p) {
        ok = ok && p >= -1 && p < n_pix;
        if (p >= 0) lo = min(lo, p);
        hi = max(hi, p);
    };
    int64_t t = t0 + threadIdx.x;
    for (; t + 3 * 256 < t1; t += 4 * 256) {
        int p[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) p[j] = __ldg(pix + t + j * 256);
#pragma unroll
        for (int j = 0; j < 4; ++j) take(p[j]);
    }
    for (; t < t1; t += 256) take(__ldg(pix + t));
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    if ((threadIdx.x & 31) == 0 && hi >= 0) {
        atomicMin(&win[b].x, lo);
        atomicMax(&win[b].y, hi);
    }
    if (!ok) *bad = 1;
}

// ---------------- launchers ----------------
void launch_block_windows(const int32_t* pix, const int64_t* block_off, int n_blocks, int64_t max_block, int n_pix,
                          int2* win, int* bad, cudaStream_t s) {
    k_window_init<<<(n_blocks + 255) / 256, 256, 0, s>>>(win, n_blocks);
    k_block_windows<<<dim3(n_blocks, (unsigned)((max_block + WIN_SLICE - 1) / WIN_SLICE)), 256, 0, s>>>(
        pix, block_off, n_pix, win, bad);
    count_launches(2);
}

size_t fft_smem_bytes(int L, bool f64) { return (size_t)(L + (L >> 4)) * (f64 ? 16 : 8); }
size_t direct_smem_bytes(int V, int lam, bool f64) {
    return (size_t)(((lam + 2) & ~1) + V + 2 * lam) * (f64 ? 8 : 4);
}


void launch_fft_spectrum(const double* h, double* H_out, double2* work, const double2* tw, int n_bands,
                         const FftPasses& fp, cudaStream_t s) {
    if (n_bands <= 0) return;
    k_fft_spectrum<<<n_bands, 256, 0, s>>>(h, H_out, reinterpret_cast<C2<double>*>(work),
                                           reinterpret_cast<const C2<double>*>(tw), fp);
    count_launches(1);
}

void launch_weights_df(const double2* cs, float4* out, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    const int64_t blocks = (n + 255) / 256;
    k_weights_df<<<(int)(blocks < 152 * 16 ? blocks : 152 * 16), 256, 0, s>>>(cs, out, n);
    count_launches(1);
}
void launch_map_to_df(const V4<double>* src, void* dst, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    const int64_t blocks = (n + 255) / 256;
    k_map_to_df<<<(int)(blocks < 152 * 8 ? blocks : 152 * 8), 256, 0, s>>>(src, reinterpret_cast<V4<df>*>(dst), n);
    count_launches(1);
}
void launch_weights64(const float* psi, double2* cs, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    const int64_t blocks = (n + 255) / 256;
    k_weights64<<<(int)(blocks < 152 * 16 ? blocks : 152 * 16), 256, 0, s>>>(psi, cs, n);
    count_launches(1);
}

}  // namespace mm
