// Set-up kernels of the filter (spectra, pointing weights) and the launch counter.
#include "filter_impl.cuh"
#include "sincos2.cuh"

namespace mm {

static long long g_launches = 0;
long long launches_total() { return __atomic_load_n(&g_launches, __ATOMIC_RELAXED); }
void count_launches(int n) { __atomic_fetch_add(&g_launches, (long long)n, __ATOMIC_RELAXED); }
std::mutex& smem_config_mutex() {
    static std::mutex m;
    return m;
}

// ---------------- trigonometric nodes ----------------
// cos and sin of 2 pi k / TRIG_N to about 100 bits by Taylor series in
// double-double arithmetic (Dekker; products through fma), for the first
// octant; the rest by symmetry.
namespace {
struct dd {
    double hi, lo;
};
dd dd_sum(double a, double b) {
    const double s = a + b, bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
dd dd_add(dd a, dd b) {
    const dd s = dd_sum(a.hi, b.hi);
    return dd_sum(s.hi, s.lo + a.lo + b.lo);
}
dd dd_mul(dd a, dd b) {
    const double p = a.hi * b.hi, e = std::fma(a.hi, b.hi, -p);
    return dd_sum(p, e + (a.hi * b.lo + a.lo * b.hi));
}
dd dd_div(dd a, double d) {
    const double q = a.hi / d;
    const double r = std::fma(-q, d, a.hi) + a.lo;
    return dd_sum(q, r / d);
}
}  // namespace

std::vector<double> trig_table() {
    const dd two_pi{6.283185307179586477, 2.4492935982947064e-16};
    constexpr int N = TRIG_N, O = N / 8;
    std::vector<dd> c(O + 1), s(O + 1);
    for (int k = 0; k <= O; ++k) {
        const dd x = dd_div(dd_mul(two_pi, dd{(double)k, 0.0}), (double)N), x2 = dd_mul(x, x);
        dd tc{1.0, 0.0}, ts = x;
        c[k] = tc;
        s[k] = ts;
        for (int i = 1; i <= 14; ++i) {
            tc = dd_div(dd_mul(tc, x2), -(2.0 * i - 1.0) * (2.0 * i));
            ts = dd_div(dd_mul(ts, x2), -(2.0 * i) * (2.0 * i + 1.0));
            c[k] = dd_add(c[k], tc);
            s[k] = dd_add(s[k], ts);
        }
    }
    std::vector<double> t(3 * (size_t)N);
    float* tail = reinterpret_cast<float*>(&t[2 * (size_t)N]);
    for (int k = 0; k < N; ++k) {
        const int quad = k / (N / 4), q = k % (N / 4);
        const dd cq = q <= O ? c[q] : s[N / 4 - q], sq = q <= O ? s[q] : c[N / 4 - q];
        dd cv = cq, sv = sq;
        if (quad == 1) {
            cv = {-sq.hi, -sq.lo};
            sv = cq;
        } else if (quad == 2) {
            cv = {-cq.hi, -cq.lo};
            sv = {-sq.hi, -sq.lo};
        } else if (quad == 3) {
            cv = sq;
            sv = {-cq.hi, -cq.lo};
        }
        t[2 * k] = cv.hi;
        t[2 * k + 1] = sv.hi;
        tail[2 * k] = (float)cv.lo;
        tail[2 * k + 1] = (float)sv.lo;
    }
    return t;
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

__global__ void k_weights64(const float* psi, const TrigTable trig, double2* cs, int64_t n) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        double sn, c;
        sincos_2psi(psi[t], trig, c, sn);
        cs[t] = make_double2(c, sn);
    }
}

// Double-float weights (cos 2psi, sin 2psi).
__global__ void k_weights_df(const float* psi, const double2* cs64, const TrigTable trig, float4* out, int64_t n) {
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        double sn, cs;
        if (cs64) {
            const double2 w = cs64[t];
            cs = w.x;
            sn = w.y;
        } else {
            sincos_2psi(psi[t], trig, cs, sn);
        }
        const float c = d2f_rn(cs), s = d2f_rn(sn);
        out[t] = make_float4(c, d2f_rn(cs - f2d_exact(c)), s, d2f_rn(sn - f2d_exact(s)));
    }
}
__global__ void k_map_to_df(const V4<double>* src, V4<df>* dst, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const V4<double> v = src[i];
        dst[i] = V4<df>{df(v.x), df(v.y), df(v.z), df(0.0)};
    }
}

__global__ void k_twiddles64(double2* tw, int N) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < N) {
        double sn, cs;
        sincospi(-2.0 * (double)e / (double)N, &sn, &cs);
        tw[e] = make_double2(cs, sn);
    }
}
__global__ void k_band_circle(const double* __restrict__ band, int lam, int N, double* h) {
    const int b = blockIdx.y;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
        const int d = min(i, N - i);
        h[(int64_t)b * N + i] = d <= lam ? band[(int64_t)b * (lam + 1) + d] : 0.0;
    }
}
// H_k = (c_0 + 2 sum_i c_i cos(2 pi k i / N)) / N, a warp per frequency and
// group of eight bands (they share the cosines): the band's transform in global
// memory takes 364 us on one SM for N = 18432 however few bands there are, the
// sums spread over the device.
constexpr int COS_B = 8;
__global__ void __launch_bounds__(256) k_band_cosines(const double* __restrict__ band, int lam, int n_bands, int N,
                                                      const double2* __restrict__ tw, double* H) {
    const int k = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, b0 = blockIdx.y * COS_B;
    if (k > N / 2) return;
    const double* c = band + (int64_t)b0 * (lam + 1);
    const int nb = min(COS_B, n_bands - b0);
    double s[COS_B] = {0, 0, 0, 0, 0, 0, 0, 0};
    const int step = (int)((int64_t)k * 32 % N);
    int e = (int)((int64_t)k * (lane + 1) % N);
#pragma unroll 2
    for (int i = lane + 1; i <= lam; i += 32) {
        const double w = tw[e].x;
#pragma unroll
        for (int b = 0; b < COS_B; ++b)
            if (b < nb) s[b] = fma(__ldg(c + (int64_t)b * (lam + 1) + i), w, s[b]);
        e += step;
        e -= e >= N ? N : 0;
    }
#pragma unroll
    for (int b = 0; b < COS_B; ++b) {
        if (b >= nb) break;
#pragma unroll
        for (int d = 16; d > 0; d >>= 1) s[b] += __shfl_down_sync(0xffffffffu, s[b], d);
        if (lane == 0) H[(int64_t)(b0 + b) * N + k] = (c[(int64_t)b * (lam + 1)] + 2.0 * s[b]) / (double)N;
    }
}
// Frequency at position p after the DIF passes (mixed-radix digit reversal:
// position sum_i d_i span_i / radix_i holds d_0 + radix_0 (d_1 + radix_1 ...)),
// and the position of a frequency.
__device__ __forceinline__ int dif_freq(const FftPasses& fp, int p) {
    int mult = 1, f = 0;
    for (int i = 0; i < fp.npass; ++i) {
        const int sr = fp.span[i] / fp.radix[i], d = p / sr;
        p -= d * sr;
        f += d * mult;
        mult *= fp.radix[i];
    }
    return f;
}
__device__ __forceinline__ int dif_pos(const FftPasses& fp, int f) {
    int p = 0;
    for (int i = 0; i < fp.npass; ++i) {
        p += f % fp.radix[i] * (fp.span[i] / fp.radix[i]);
        f /= fp.radix[i];
    }
    return p;
}
// Table values in the layouts of the kernels: KIND 0 float32, 1 float64, 2
// double-float (hi, lo).
template <int KIND> struct Tab;
template <> struct Tab<0> {
    static __device__ void put(void* t, int64_t i, double v) { reinterpret_cast<float*>(t)[i] = (float)v; }
};
template <> struct Tab<1> {
    static __device__ void put(void* t, int64_t i, double v) { reinterpret_cast<double*>(t)[i] = v; }
};
template <> struct Tab<2> {
    static __device__ void put(void* t, int64_t i, double v) {
        const float hi = (float)v;
        reinterpret_cast<float2*>(t)[i] = make_float2(hi, (float)(v - (double)hi));
    }
};
// tw[e] = exp(-2 pi i e / L); then the passes' own powers W_S^(j q), pass by pass, [q - 1][j], into twp (may be null)
template <int KIND>
__global__ void k_plan_twiddles(const FftPasses fp, void* tw, void* twp, int64_t n_twp) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    double sn, cs;
    if (i < fp.L) {
        sincospi(-2.0 * (double)i / (double)fp.L, &sn, &cs);
        Tab<KIND>::put(tw, 2 * i, cs);
        Tab<KIND>::put(tw, 2 * i + 1, sn);
    }
    if (twp && i < n_twp) {
        int64_t r = i;
        int p = 0;
        for (; p < fp.npass - 1; ++p) {
            const int64_t n = (int64_t)(fp.radix[p] - 1) * (fp.span[p] / fp.radix[p]);
            if (r < n) break;
            r -= n;
        }
        const int sr = fp.span[p] / fp.radix[p], q = (int)(r / sr) + 1, j = (int)(r % sr);
        sincospi(-2.0 * (double)((int64_t)j * q % fp.span[p]) / (double)fp.span[p], &sn, &cs);
        Tab<KIND>::put(twp, 2 * i, cs);
        Tab<KIND>::put(twp, 2 * i + 1, sn);
    }
}
// Spectrum of a two-segment plan: position p holds H at its frequency.
template <int KIND>
__global__ void k_plan_spectrum(const double* __restrict__ S, const FftPasses fp, int n_bands, void* H) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= fp.L) return;
    const int k = dif_freq(fp, p);
    for (int64_t b = blockIdx.y; b < n_bands; b += gridDim.y)
        Tab<KIND>::put(H, b * fp.L + p, S[b * fp.L + min(k, fp.L - k)]);
}
// Index tables of a half-length plan (one CTA).  Pairs (k, M - k), k = 0 ..
// M/2, in the order of the position of k: neighbouring threads then touch
// neighbouring points (the frequency order would stride by M / radix_0 and put a
// warp's accesses on one bank).  Items of the fused spectrum pass: the last
// pass of radix R works on butterflies c of R consecutive positions; butterfly
// c holds the frequencies kc + (M/R) q and its partner c' (frequency digits
// M/R - kc) their mirror images M - k, at output R - 1 - q (kc = 0 and kc =
// M/(2R) pair with themselves); one item per pair {c, c'}, kc = 0 .. M/(2R), in
// the order of c, bit 31 marking kc = 0.
__global__ void __launch_bounds__(1024) k_half_index(const FftPasses fp, uint32_t* pairs, int* pair_k, uint32_t* items,
                                                     int* item_k) {
    __shared__ int part[32];
    const int M = fp.L, R = fp.radix[fp.npass - 1], NB = M / R, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int which = 0; which < (items ? 2 : 1); ++which) {
        const int n = which ? NB : M;
        int base = 0;
        for (int c0 = 0; c0 < n; c0 += 1024) {
            const int c = c0 + threadIdx.x;
            const int k = c < n ? dif_freq(fp, which ? c * R : c) : n;
            const bool in = c < n && k <= n / 2;
            const unsigned m = __ballot_sync(0xffffffffu, in);
            if (lane == 0) part[warp] = __popc(m);
            __syncthreads();
            int at = base + __popc(m & ((1u << lane) - 1u)), all = 0;
            for (int w = 0; w < 32; ++w) {
                if (w < warp) at += part[w];
                all += part[w];
            }
            if (in) {
                if (which) {
                    items[at] = (uint32_t)c | (uint32_t)(dif_pos(fp, (NB - k) % NB) / R) << 16 | (k == 0 ? 0x80000000u : 0u);
                    item_k[at] = k;
                } else {
                    pairs[at] = (uint32_t)c | (uint32_t)dif_pos(fp, (M - k) % M) << 16;
                    pair_k[at] = k;
                }
            }
            base += all;
            __syncthreads();
        }
    }
}
// Coefficients (alpha_k, alpha_{M-k}, beta_k, 0) of the paired real-spectrum
// filter with 1/M folded in, from the spectra S [n_bands][2 M]: entry e of R
// consecutive ones per index takes k = idx[e / R] + (M / R) (e % R).
template <int KIND>
__global__ void k_half_coef(const double* __restrict__ S, int M, const int* __restrict__ idx, int n, int R, int n_bands,
                            void* C) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= n * R) return;
    const int k = idx[e / R] + M / R * (e % R), N = 2 * M;
    double sn, cs;
    sincospi(2.0 * (double)k / (double)N, &sn, &cs);
    for (int b = blockIdx.y; b < n_bands; b += gridDim.y) {
        const double h1 = 2.0 * S[(int64_t)b * N + k], h2 = 2.0 * S[(int64_t)b * N + M - k];
        const int64_t o = 4 * ((int64_t)b * n * R + e);
        Tab<KIND>::put(C, o, 0.5 * ((h1 + h2) + (h2 - h1) * sn));
        Tab<KIND>::put(C, o + 1, 0.5 * ((h1 + h2) - (h2 - h1) * sn));
        Tab<KIND>::put(C, o + 2, -0.5 * (h2 - h1) * cs);
        Tab<KIND>::put(C, o + 3, 0.0);
    }
}
__global__ void k_spectrum_order(const double* __restrict__ Hp, double* H, const FftPasses fp) {
    const int64_t b = (int64_t)blockIdx.y * fp.L;
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < fp.L; p += gridDim.x * blockDim.x)
        H[b + dif_freq(fp, p)] = Hp[b + p];
}
// Twiddles (rows of filter_half3.cuh's Pass1Twiddle; [9][r1]) and, per band,
// the coefficients of the paired spectrum step: item t pairs k = kc + r0 r1 q
// with M - k, kc in the order of h3_spectrum's items.
__global__ void k_half3_twiddles(int r0, int r1, float2* t1, float2* t2) {
    const int sr = 9 * r1, M = r0 * sr, ra = r0 / 4, n1 = (ra + 2) * sr, i = blockIdx.x * blockDim.x + threadIdx.x;
    double sn, cs;
    if (i < n1) {
        const int q = i / sr + 1, j = i % sr;
        sincospi(-2.0 * (double)(j * (q < ra ? q : (q - ra + 1) * ra) % M) / (double)M, &sn, &cs);
        t1[i] = make_float2((float)cs, (float)sn);
    } else if (i < n1 + sr) {
        const int j = (i - n1) / r1, q = (i - n1) % r1;
        sincospi(-2.0 * (double)(j * q % sr) / (double)sr, &sn, &cs);
        t2[i - n1] = make_float2((float)cs, (float)sn);
    }
}
__global__ void k_half3_coef(const double* __restrict__ H, int n_bands, int r0, int r1, float4* Hi) {
    const int nb = r0 * r1, ni = nb / 2 + 1, M = 9 * nb, N = 2 * M, i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= 9 * ni) return;
    const int q = i / ni, t = i % ni;
    int g = t / r1, r = t % r1;
    if (t == nb / 2) {
        g = 0;
        r = r1 / 2;
    } else if (g == 0) {
        if (r < r1 / 2) g = r0 / 2;
        else r -= r1 / 2;
    }
    const int k = g + r0 * r + nb * q;
    double sn, cs;
    sincospi(2.0 * (double)k / (double)N, &sn, &cs);
    for (int b = blockIdx.y; b < n_bands; b += gridDim.y) {
        const double h1 = 2.0 * H[(int64_t)b * N + k], h2 = 2.0 * H[(int64_t)b * N + M - k];   // H / M
        Hi[(int64_t)b * 9 * ni + i] = make_float4((float)(0.5 * ((h1 + h2) + (h2 - h1) * sn)),
                                                  (float)(0.5 * ((h1 + h2) - (h2 - h1) * sn)), (float)(-0.5 * (h2 - h1) * cs), 0.0f);
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
    int lo = 0x7fffffff, hi = -1;
    bool ok = true;
    auto take = [&](int p) {
        ok = ok && p >= -1 && p < n_pix;
        if (p >= 0) lo = min(lo, p);
        hi = max(hi, p);
    };
    for (int64_t t0 = off[b] + (int64_t)blockIdx.y * WIN_SLICE; t0 < o1; t0 += (int64_t)gridDim.y * WIN_SLICE) {
        const int64_t t1 = t0 + WIN_SLICE < o1 ? t0 + WIN_SLICE : o1;
        int64_t t = t0 + threadIdx.x;
        for (; t + 3 * 256 < t1; t += 4 * 256) {
            int p[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) p[j] = __ldg(pix + t + j * 256);
#pragma unroll
            for (int j = 0; j < 4; ++j) take(p[j]);
        }
        for (; t < t1; t += 256) take(__ldg(pix + t));
    }
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
    k_block_windows<<<dim3(n_blocks, (unsigned)std::min<int64_t>(65535, (max_block + WIN_SLICE - 1) / WIN_SLICE)), 256, 0, s>>>(
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

void launch_twiddles64(double2* tw, int N, cudaStream_t s) {
    k_twiddles64<<<(N + 255) / 256, 256, 0, s>>>(tw, N);
    count_launches(1);
}
void launch_band_circle(const double* band, int lam, int n_bands, int N, double* h, cudaStream_t s) {
    k_band_circle<<<dim3((N + 1023) / 1024, n_bands), 256, 0, s>>>(band, lam, N, h);
    count_launches(1);
}
void launch_band_cosines(const double* band, int lam, int n_bands, int N, const double2* tw, double* H, cudaStream_t s) {
    k_band_cosines<<<dim3((N / 2 + 8) / 8, (n_bands + COS_B - 1) / COS_B), 256, 0, s>>>(band, lam, n_bands, N, tw, H);
    count_launches(1);
}
void launch_spectrum_order(const double* Hp, double* H, int n_bands, const FftPasses& fp, cudaStream_t s) {
    k_spectrum_order<<<dim3((fp.L + 1023) / 1024, n_bands), 256, 0, s>>>(Hp, H, fp);
    count_launches(1);
}
template <int KIND>
static void plan_tables(const double* S, int n_bands, const FftPasses& fp, void* tw, void* H, cudaStream_t s) {
    k_plan_twiddles<KIND><<<(fp.L + 255) / 256, 256, 0, s>>>(fp, tw, nullptr, 0);
    k_plan_spectrum<KIND><<<dim3((fp.L + 255) / 256, std::min(n_bands, 64)), 256, 0, s>>>(S, fp, n_bands, H);
    count_launches(2);
}
void launch_plan_tables(const double* S, int n_bands, const FftPasses& fp, int kind, void* tw, void* H, cudaStream_t s) {
    if (kind == 0) plan_tables<0>(S, n_bands, fp, tw, H, s);
    else if (kind == 1) plan_tables<1>(S, n_bands, fp, tw, H, s);
    else plan_tables<2>(S, n_bands, fp, tw, H, s);
}
bool half_fused(const FftPasses& fp) {
    const int R = fp.radix[fp.npass - 1];
    return fp.span[fp.npass - 1] == R && (fp.L / R) % 2 == 0 && 16 % R == 0;
}
int64_t plan_powers(const FftPasses& fp) {
    int64_t n = 0;
    for (int i = 0; i < fp.npass; ++i) n += (int64_t)(fp.radix[i] - 1) * (fp.span[i] / fp.radix[i]);
    return n > 0 ? n : 1;
}
template <int KIND>
static void half_tables(const double* S, int n_bands, const FftPasses& fp, const HalfTables& t, cudaStream_t s) {
    const int M = fp.L, R = fp.radix[fp.npass - 1], np = M / 2 + 1, ni = M / R / 2 + 1;
    const bool fused = half_fused(fp);
    const int64_t n = std::max<int64_t>(M, plan_powers(fp));
    k_plan_twiddles<KIND><<<(unsigned)((n + 255) / 256), 256, 0, s>>>(fp, t.tw, t.twp, plan_powers(fp));
    k_half_index<<<1, 1024, 0, s>>>(fp, t.pairs, t.scratch, fused ? t.items : nullptr, t.scratch + np);
    const int gy = std::min(n_bands, 64);
    k_half_coef<KIND><<<dim3((np + 255) / 256, gy), 256, 0, s>>>(S, M, t.scratch, np, 1, n_bands, t.H);
    if (fused) k_half_coef<KIND><<<dim3((ni * R + 255) / 256, gy), 256, 0, s>>>(S, M, t.scratch + np, ni, R, n_bands, t.Hi);
    count_launches(fused ? 4 : 3);
}
void launch_half_tables(const double* S, int n_bands, const FftPasses& fp, int kind, const HalfTables& t, cudaStream_t s) {
    if (kind == 0) half_tables<0>(S, n_bands, fp, t, s);
    else if (kind == 1) half_tables<1>(S, n_bands, fp, t, s);
    else half_tables<2>(S, n_bands, fp, t, s);
}
void launch_half3_tables(const double* H, int n_bands, int r0, int r1, float2* t1, float2* t2, float4* Hi, cudaStream_t s) {
    const int n = (r0 / 4 + 3) * 9 * r1, ni = r0 * r1 / 2 + 1;
    k_half3_twiddles<<<(n + 255) / 256, 256, 0, s>>>(r0, r1, t1, t2);
    k_half3_coef<<<dim3((9 * ni + 255) / 256, n_bands < 64 ? n_bands : 64), 256, 0, s>>>(H, n_bands, r0, r1, Hi);
    count_launches(2);
}

void launch_weights_df(const float* psi, const double2* cs64, const TrigTable& trig, float4* out, int64_t n,
                       cudaStream_t s) {
    if (n <= 0) return;
    const int64_t blocks = (n + 255) / 256;
    k_weights_df<<<(int)(blocks < 152 * 16 ? blocks : 152 * 16), 256, 0, s>>>(psi, cs64, trig, out, n);
    count_launches(1);
}
void launch_map_to_df(const V4<double>* src, void* dst, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    const int64_t blocks = (n + 255) / 256;
    k_map_to_df<<<(int)(blocks < 152 * 8 ? blocks : 152 * 8), 256, 0, s>>>(src, reinterpret_cast<V4<df>*>(dst), n);
    count_launches(1);
}
void launch_weights64(const float* psi, const TrigTable& trig, double2* cs, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    const int64_t blocks = (n + 255) / 256;
    k_weights64<<<(int)(blocks < 152 * 16 ? blocks : 152 * 16), 256, 0, s>>>(psi, trig, cs, n);
    count_launches(1);
}

}  // namespace mm
