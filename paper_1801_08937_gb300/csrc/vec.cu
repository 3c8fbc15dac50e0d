// Map-space kernels: M_BD build and apply (Sect. 3.1, Eq. mbd), the fused
// PCG vector steps with float64 inner products (Sect. 3, Eq. pcg), the
// two-level preconditioner M_2l (Sect. 3.2, Eq. m2l) and the tall-skinny
// float64 products of the Arnoldi process (Appendix A).
//
// Every reduction is two-phase and deterministic: each CTA writes its
// partial sums, and the last CTA to finish (an atomic ticket, no waiting)
// adds them in CTA order and applies the scalar update.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "fconv.cuh"
#include "df64.cuh"
#include "sincos2.cuh"

namespace mm {

constexpr int VT = 256;

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += __shfl_down_sync(0xffffffffu, v, d);
    return v;
}

// Sum D per-thread values over the CTA; thread d < D writes partial[d].
template <int D>
__device__ __forceinline__ void block_partials(const double (&v)[D], double* out) {
    __shared__ double red[VT / 32][D > 0 ? D : 1];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int d = 0; d < D; ++d) {
        const double s = warp_sum(v[d]);
        if (lane == 0) red[warp][d] = s;
    }
    __syncthreads();
    if (threadIdx.x < D) {
        double s = 0.0;
        for (int w = 0; w < VT / 32; ++w) s += red[w][threadIdx.x];
        out[threadIdx.x] = s;
    }
}

// Last-CTA election for the reduction of slice `rhs` (grid.y); returns true
// in every thread of the CTA that finishes last.
__device__ __forceinline__ bool last_block(unsigned* counter, int rhs) {
    __shared__ bool is_last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned prev = atomicAdd(counter + rhs, 1u);
        is_last = (prev == gridDim.x - 1);
    }
    __syncthreads();
    if (is_last) __threadfence();
    return is_last;
}

// Sum of the CTA partials of value d for slice rhs, by the whole (last) CTA:
// strided per-thread sums, then warp and CTA trees -- a fixed order, so the
// result is deterministic.  Every thread of the CTA must call it; the sum is
// returned to all threads.
template <int D>
__device__ __forceinline__ double gather_partial(const double* partial, int nblk, int nrhs, int rhs, int d) {
    __shared__ double red[VT / 32];
    __shared__ double total;
    double s = 0.0;
    for (int b = threadIdx.x; b < nblk; b += VT) s += __ldcg(partial + ((int64_t)b * nrhs + rhs) * D + d);
    s = warp_sum(s);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) red[warp] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < VT / 32; ++w) t += red[w];
        total = t;
    }
    __syncthreads();
    return total;
}

// Warp w sums partials of the values c = w, w + 8, ... (k values per slice).
__device__ __forceinline__ double warp_gather(const double* partial, int nblk, int64_t stride, int64_t off) {
    const int lane = threadIdx.x & 31;
    double s = 0.0;
    for (int b = lane; b < nblk; b += 32) s += __ldcg(partial + (int64_t)b * stride + off);
    s = warp_sum(s);
    return __shfl_sync(0xffffffffu, s, 0);
}

__device__ __forceinline__ V4<double> ld4(const V4<double>* p) { return *p; }
__device__ __forceinline__ V4<double> ld4(const V4<float>* p) {
    const V4<float> v = *p;
    return {v.x, v.y, v.z, 0.0};
}
__device__ __forceinline__ double dot3(const V4<double>& a, const V4<double>& b) {
    return a.x * b.x + a.y * b.y + a.z * b.z;
}
__device__ __forceinline__ V4<double> bd_mul(const double* m, const V4<double>& v) {
    return {m[0] * v.x + m[1] * v.y + m[2] * v.z, m[1] * v.x + m[3] * v.y + m[4] * v.z,
            m[2] * v.x + m[4] * v.y + m[5] * v.z, 0.0};
}

#define PIX_LOOP(i) for (int i = blockIdx.x * VT + threadIdx.x; i < a.n_pix; i += gridDim.x * VT)

// ---------------- conversions ----------------
__global__ void k_map_in(const double* src, V4<double>* dst, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)VT + threadIdx.x; i < n; i += (int64_t)gridDim.x * VT)
        dst[i] = V4<double>{src[3 * i], src[3 * i + 1], src[3 * i + 2], 0.0};
}
__global__ void k_map_out(const V4<double>* src, double* dst, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)VT + threadIdx.x; i < n; i += (int64_t)gridDim.x * VT) {
        const V4<double> v = src[i];
        dst[3 * i] = v.x;
        dst[3 * i + 1] = v.y;
        dst[3 * i + 2] = v.z;
    }
}
__global__ void k_to_f32(const V4<double>* src, V4<float>* dst, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)VT + threadIdx.x; i < n; i += (int64_t)gridDim.x * VT) {
        const V4<double> v = src[i];
        dst[i] = V4<float>{(float)v.x, (float)v.y, (float)v.z, 0.0f};
    }
}
__global__ void k_from_f32(const V4<float>* src, V4<double>* dst, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)VT + threadIdx.x; i < n; i += (int64_t)gridDim.x * VT)
        dst[i] = ld4(src + i);
}
// mm_apply_A's input in one pass: the caller's (I, Q, U) to the operator's
// vectors (prec 0 float32, 1 float64, 2 double-float) and the accumulators to
// zero; and its output.  Four launches of conversions and clears around the
// filter became two (12 us -> 6 us of a product on a small map).
template <int PREC>
__global__ void k_apply_in(const double* __restrict__ src, void* dst, void* acc, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)VT + threadIdx.x; i < n; i += (int64_t)gridDim.x * VT) {
        const double x = src[3 * i], y = src[3 * i + 1], z = src[3 * i + 2];
        if constexpr (PREC == 0) {
            reinterpret_cast<V4<float>*>(dst)[i] = V4<float>{(float)x, (float)y, (float)z, 0.0f};
            reinterpret_cast<V4<float>*>(acc)[i] = V4<float>{0.0f, 0.0f, 0.0f, 0.0f};
        } else {
            if constexpr (PREC == 1) reinterpret_cast<V4<double>*>(dst)[i] = V4<double>{x, y, z, 0.0};
            else reinterpret_cast<V4<df>*>(dst)[i] = V4<df>{df(x), df(y), df(z), df(0.0)};
            reinterpret_cast<V4<double>*>(acc)[i] = V4<double>{0.0, 0.0, 0.0, 0.0};
        }
    }
}
__global__ void k_map_out_f32(const V4<float>* __restrict__ src, double* dst, int64_t n) {
    for (int64_t i = blockIdx.x * (int64_t)VT + threadIdx.x; i < n; i += (int64_t)gridDim.x * VT) {
        const V4<float> v = src[i];
        dst[3 * i] = v.x;
        dst[3 * i + 1] = v.y;
        dst[3 * i + 2] = v.z;
    }
}
static int grid_for(int64_t n) {
    const int64_t b = (n + VT - 1) / VT;
    return (int)(b < 152 * 8 ? (b > 0 ? b : 1) : 152 * 8);
}
void launch_apply_in(const double* src3, int prec, void* dst, void* acc, int64_t n, cudaStream_t s) {
    if (n <= 0) return;
    if (prec == 0) k_apply_in<0><<<grid_for(n), VT, 0, s>>>(src3, dst, acc, n);
    else if (prec == 1) k_apply_in<1><<<grid_for(n), VT, 0, s>>>(src3, dst, acc, n);
    else k_apply_in<2><<<grid_for(n), VT, 0, s>>>(src3, dst, acc, n);
    count_launches(1);
}
void launch_map_out_f32(const V4<float>* src4, double* dst3, int64_t n, cudaStream_t s) {
    if (n > 0) {
        k_map_out_f32<<<grid_for(n), VT, 0, s>>>(src4, dst3, n);
        count_launches(1);
    }
}
void launch_map_in(const double* src3, V4<double>* dst4, int64_t n, cudaStream_t s) {
    if (n > 0) {
        k_map_in<<<grid_for(n), VT, 0, s>>>(src3, dst4, n);
        count_launches(1);
    }
}
void launch_map_out(const V4<double>* src4, double* dst3, int64_t n, cudaStream_t s) {
    if (n > 0) {
        k_map_out<<<grid_for(n), VT, 0, s>>>(src4, dst3, n);
        count_launches(1);
    }
}
void launch_to_f32(const V4<double>* src, V4<float>* dst, int64_t n, cudaStream_t s) {
    if (n > 0) {
        k_to_f32<<<grid_for(n), VT, 0, s>>>(src, dst, n);
        count_launches(1);
    }
}
void launch_from_f32(const V4<float>* src, V4<double>* dst, int64_t n, cudaStream_t s) {
    if (n > 0) {
        k_from_f32<<<grid_for(n), VT, 0, s>>>(src, dst, n);
        count_launches(1);
    }
}
void launch_zero(void* p, size_t bytes, cudaStream_t s) {
    if (bytes) cudaMemsetAsync(p, 0, bytes, s);
}

// ---------------- M_BD ----------------
// Per sample: bucket j = number of right-hand-side lengths <= the sample's
// position in its detector timeline (lengths sorted ascending); the sample
// belongs to every right-hand side of sorted rank >= j.  Sums of
// c_0 w w^T (6 entries) and the hit count go to bucket j.
//
// A lane takes eight consecutive samples and sums its runs of equal pixels in
// registers; its first run joins the lane before it when that lane ends on the
// same pixel, so a run costs one set of atomics.  The weights come from the
// stored float64 ones, or from the table where a context keeps none.  Bound by
// the float64 pipe (17 operations a sample, 0.9 ms on 3.4e7 samples at its
// measured rate): 4433 -> 1191 us there against one sample per lane with the
// general sincos and seven five-step shuffled sums.
constexpr int BD_SLICE = 8192;   // samples per CTA and step: long blocks spread over the device
constexpr int BD_SLICES = 1024;  // CTAs per block at most (a grid holds 65535 rows): longer blocks are walked

struct BdSums {
    double c, s, cc, cs, ss;
    int n;
};
__device__ __forceinline__ void bd_flush(double* sums, int64_t key, double c0, const BdSums& v) {
    double* o = sums + key * 7;
    atomicAdd(o, c0 * (double)v.n);
    atomicAdd(o + 1, c0 * v.c);
    atomicAdd(o + 2, c0 * v.s);
    atomicAdd(o + 3, c0 * v.cc);
    atomicAdd(o + 4, c0 * v.cs);
    atomicAdd(o + 5, c0 * v.ss);
    atomicAdd(o + 6, (double)v.n);
}

// LENS: several lengths; a sample's key is its bucket's pixel (64 bits), else its pixel.
template <bool LENS>
__global__ void __launch_bounds__(VT) k_bd_accumulate(const int32_t* __restrict__ pix, const float* __restrict__ psi,
                                                      const double2* __restrict__ cs64, const TrigTable trig,
                                                      const int64_t* __restrict__ block_off,
                                                      const int32_t* __restrict__ block_band,
                                                      const double* __restrict__ band, int lam1, int64_t n_t,
                                                      const int64_t* __restrict__ sorted_len, int nrhs, double* sums,
                                                      int n_pix) {
    const int b = blockIdx.x;
    const int64_t o1 = block_off[b + 1];
    const int64_t det0 = block_off[b] / n_t * n_t;   // a block lies in one detector's timeline
    const double c0 = band[(int64_t)block_band[b] * lam1];
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    for (int64_t s0 = block_off[b] + (int64_t)blockIdx.y * BD_SLICE; s0 < o1; s0 += (int64_t)gridDim.y * BD_SLICE) {
        const int64_t s1 = s0 + BD_SLICE < o1 ? s0 + BD_SLICE : o1;
        for (int64_t w0 = s0 + (threadIdx.x >> 5) * 256; w0 < s1; w0 += VT * 8) {
            const int64_t t0 = w0 + 8 * lane;
            using Key = typename std::conditional<LENS, int64_t, int>::type;
            Key key[8];
            BdSums a{0, 0, 0, 0, 0, 0}, f{0, 0, 0, 0, 0, 0};
            bool multi = false;
            int j = 0;
            if (LENS && t0 < s1) {   // lengths up to the first sample's position
                const int64_t pos = t0 - det0;
                int hi = nrhs;
                while (j < hi) {
                    const int mid = (j + hi) >> 1;
                    if (sorted_len[mid] <= pos) j = mid + 1;
                    else hi = mid;
                }
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int64_t t = t0 + e;
                key[e] = -1;
                double cs = 0.0, sn = 0.0;
                if (t < s1) {
                    const int p = __ldg(pix + t);
                    if (LENS) {
                        while (j < nrhs && sorted_len[j] <= t - det0) ++j;
                        if (p >= 0 && j < nrhs) key[e] = (Key)j * n_pix + p;
                    } else {
                        key[e] = p;
                    }
                    if (key[e] >= 0) {
                        if (cs64) {
                            const double2 w = __ldg(cs64 + t);
                            cs = w.x;
                            sn = w.y;
                        } else {
                            sincos_2psi(__ldg(psi + t), trig, cs, sn);
                        }
                    }
                }
                if (e > 0 && key[e] != key[e - 1]) {
                    if (multi) {
                        if (key[e - 1] >= 0) bd_flush(sums, key[e - 1], c0, a);
                    } else {
                        f = a;
                        multi = true;
                    }
                    a = BdSums{0, 0, 0, 0, 0, 0};
                }
                a.c += cs;
                a.s += sn;
                a.cc = fma(cs, cs, a.cc);
                a.cs = fma(cs, sn, a.cs);
                a.ss = fma(sn, sn, a.ss);
                a.n += 1;
            }
            const Key klast = __shfl_up_sync(FULL, key[7], 1);
            const bool give = multi && lane > 0 && key[0] == klast;
            BdSums r;
            r.c = __shfl_down_sync(FULL, f.c, 1);
            r.s = __shfl_down_sync(FULL, f.s, 1);
            r.cc = __shfl_down_sync(FULL, f.cc, 1);
            r.cs = __shfl_down_sync(FULL, f.cs, 1);
            r.ss = __shfl_down_sync(FULL, f.ss, 1);
            r.n = __shfl_down_sync(FULL, f.n, 1);
            if (__shfl_down_sync(FULL, (int)give, 1) && lane < 31) {
                a.c += r.c;
                a.s += r.s;
                a.cc += r.cc;
                a.cs += r.cs;
                a.ss += r.ss;
                a.n += r.n;
            }
            if (multi && !give && key[0] >= 0) bd_flush(sums, key[0], c0, f);
            if (key[7] >= 0) bd_flush(sums, key[7], c0, a);
        }
    }
}

// Prefix over buckets: sorted rank r holds the sum of buckets 0..r.
__global__ void k_bd_prefix(double* sums, int n_pix, int nrhs) {
    for (int64_t i = blockIdx.x * (int64_t)VT + threadIdx.x; i < (int64_t)n_pix * 7; i += (int64_t)gridDim.x * VT) {
        double acc = 0.0;
        for (int j = 0; j < nrhs; ++j) {
            acc += sums[(int64_t)j * n_pix * 7 + i];
            sums[(int64_t)j * n_pix * 7 + i] = acc;
        }
    }
}

void launch_bd_accumulate(const int32_t* pix, const float* psi, const double2* cs64, const TrigTable& trig,
                          const int64_t* block_off, const int32_t* block_band, const double* band, int lam1, int n_blocks,
                          int64_t max_block, int64_t n_t, const int64_t* sorted_len, int nrhs, double* sums, int n_pix,
                          cudaStream_t s) {
    if (n_blocks <= 0) return;
    const dim3 g(n_blocks, (unsigned)std::min<int64_t>(BD_SLICES, (max_block + BD_SLICE - 1) / BD_SLICE));
    if (sorted_len)
        k_bd_accumulate<true><<<g, VT, 0, s>>>(pix, psi, cs64, trig, block_off, block_band, band, lam1, n_t, sorted_len,
                                               nrhs, sums, n_pix);
    else
        k_bd_accumulate<false><<<g, VT, 0, s>>>(pix, psi, cs64, trig, block_off, block_band, band, lam1, n_t, nullptr, 1,
                                                sums, n_pix);
    count_launches(1);
    if (nrhs > 1) {
        k_bd_prefix<<<grid_for((int64_t)n_pix * 7), VT, 0, s>>>(sums, n_pix, nrhs);
        count_launches(1);
    }
}

// Eigenvalues of a symmetric 3x3 matrix by cyclic Jacobi rotations.
__device__ void sym3_eig(double a[3][3], double& lmin, double& lmax) {
    for (int sweep = 0; sweep < 12; ++sweep) {
        const double off = fabs(a[0][1]) + fabs(a[0][2]) + fabs(a[1][2]);
        const double diag = fabs(a[0][0]) + fabs(a[1][1]) + fabs(a[2][2]);
        if (off <= 1e-300 || off <= 1e-17 * diag) break;
        for (int p = 0; p < 2; ++p)
            for (int q = p + 1; q < 3; ++q) {
                if (a[p][q] == 0.0) continue;
                const double theta = (a[q][q] - a[p][p]) / (2.0 * a[p][q]);
                const double t = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
                const double c = 1.0 / sqrt(t * t + 1.0), sn = t * c;
                for (int k = 0; k < 3; ++k) {
                    const double akp = a[k][p], akq = a[k][q];
                    a[k][p] = c * akp - sn * akq;
                    a[k][q] = sn * akp + c * akq;
                }
                for (int k = 0; k < 3; ++k) {
                    const double apk = a[p][k], aqk = a[q][k];
                    a[p][k] = c * apk - sn * aqk;
                    a[q][k] = sn * apk + c * aqk;
                }
            }
    }
    lmin = fmin(a[0][0], fmin(a[1][1], a[2][2]));
    lmax = fmax(a[0][0], fmax(a[1][1], a[2][2]));
}

// sums [nrhs][n_pix][7] -> bd [nrhs][n_pix][6] = inverse blocks (upper
// triangle by rows).  With set_good, the keep/drop decision is made here
// (hits >= 3 and rcond >= rcond_min); otherwise `good` is read and a kept
// pixel whose block is numerically singular for this right-hand side gets a
// zero block.
// stokes 1: only the (Q, U) block counts (pointing rows (0, cos, sin) of the
// differenced timeline): at least 2 hits and a conditioned 2x2 block; the I
// entries of the inverse are zero.  stokes 2: only I (rows (1, 0, 0) of the
// summed timeline): at least 1 hit, the 1x1 inverse, Q and U entries zero.
__global__ void k_bd_invert(const double* sums, double* bd, uint8_t* good, int* n_dropped, int n_pix, int nrhs,
                            double rcond_min, int set_good, int stokes) {
    const int64_t total = (int64_t)n_pix * nrhs;
    for (int64_t idx = blockIdx.x * (int64_t)VT + threadIdx.x; idx < total; idx += (int64_t)gridDim.x * VT) {
        const int p = (int)(idx % n_pix);
        const double* S = sums + idx * 7;
        const double s00 = S[0], s01 = S[1], s02 = S[2], s11 = S[3], s12 = S[4], s22 = S[5], hits = S[6];
        if (stokes == 2) {
            bool keep1;
            if (set_good) {
                keep1 = hits >= 1.0 && s00 > 0.0;
                good[p] = keep1 ? 1 : 0;
                if (!keep1) atomicAdd(n_dropped, 1);
            } else {
                keep1 = good[p] != 0 && s00 > 0.0;
            }
            double* o = bd + idx * 6;
            for (int e = 0; e < 6; ++e) o[e] = 0.0;
            if (keep1) o[0] = 1.0 / s00;
            continue;
        }
        if (stokes == 1) {
            const double tr = s11 + s22, det2 = s11 * s22 - s12 * s12;
            const double disc = sqrt(fmax(0.25 * (s11 - s22) * (s11 - s22) + s12 * s12, 0.0));
            const double lmax2 = 0.5 * tr + disc, lmin2 = 0.5 * tr - disc;
            const double rc2 = lmax2 > 0.0 ? lmin2 / lmax2 : 0.0;
            bool keep2;
            if (set_good) {
                keep2 = hits >= 2.0 && rc2 >= rcond_min;
                good[p] = keep2 ? 1 : 0;
                if (!keep2) atomicAdd(n_dropped, 1);
            } else {
                keep2 = good[p] != 0 && rc2 > 1e-12;
            }
            double* o = bd + idx * 6;
            for (int e = 0; e < 6; ++e) o[e] = 0.0;
            if (keep2) {
                o[3] = s22 / det2;
                o[4] = -s12 / det2;
                o[5] = s11 / det2;
            }
            continue;
        }
        double m[3][3] = {{s00, s01, s02}, {s01, s11, s12}, {s02, s12, s22}};
        double lmin, lmax;
        sym3_eig(m, lmin, lmax);
        const double rc = lmax > 0.0 ? lmin / lmax : 0.0;
        bool keep;
        if (set_good) {
            keep = hits >= 3.0 && rc >= rcond_min;
            good[p] = keep ? 1 : 0;
            if (!keep) atomicAdd(n_dropped, 1);
        } else {
            keep = good[p] != 0 && rc > 1e-12;
        }
        double* o = bd + idx * 6;
        if (!keep) {
            for (int e = 0; e < 6; ++e) o[e] = 0.0;
            continue;
        }
        // inverse of the symmetric block by cofactors
        const double c00 = s11 * s22 - s12 * s12;
        const double c01 = s02 * s12 - s01 * s22;
        const double c02 = s01 * s12 - s02 * s11;
        const double c11 = s00 * s22 - s02 * s02;
        const double c12 = s01 * s02 - s00 * s12;
        const double c22 = s00 * s11 - s01 * s01;
        const double det = s00 * c00 + s01 * c01 + s02 * c02;
        const double id = 1.0 / det;
        o[0] = c00 * id;
        o[1] = c01 * id;
        o[2] = c02 * id;
        o[3] = c11 * id;
        o[4] = c12 * id;
        o[5] = c22 * id;
    }
}
void launch_bd_invert(const double* sums, double* bd, uint8_t* good, int* n_dropped, int n_pix, int nrhs,
                      double rcond_min, int set_good, cudaStream_t s, int stokes) {
    k_bd_invert<<<grid_for((int64_t)n_pix * nrhs), VT, 0, s>>>(sums, bd, good, n_dropped, n_pix, nrhs, rcond_min,
                                                              set_good, stokes);
    count_launches(1);
}

// Nothing to flag when no pixel was dropped (the usual case on an observed patch): the pass over pix is skipped.
__global__ void k_flag_samples(int32_t* pix, const uint8_t* good, const int* dropped, int64_t n) {
    if (*dropped == 0) return;
    for (int64_t t = blockIdx.x * (int64_t)VT + threadIdx.x; t < n; t += (int64_t)gridDim.x * VT) {
        const int p = pix[t];
        if (p >= 0 && !good[p]) pix[t] = -1;
    }
}
void launch_flag_samples(int32_t* pix, const uint8_t* good, const int* dropped, int64_t n, cudaStream_t s) {
    if (n > 0) {
        k_flag_samples<<<grid_for(n), VT, 0, s>>>(pix, good, dropped, n);
        count_launches(1);
    }
}

__global__ void k_bd_apply(const double* bd, int per_rhs, const V4<double>* x, V4<double>* y, int n_pix) {
    const int rhs = blockIdx.y;
    for (int i = blockIdx.x * VT + threadIdx.x; i < n_pix; i += gridDim.x * VT) {
        const double* m = bd + ((int64_t)(per_rhs ? rhs : 0) * n_pix + i) * 6;
        y[(int64_t)rhs * n_pix + i] = bd_mul(m, x[(int64_t)rhs * n_pix + i]);
    }
}
void launch_bd_apply(const double* bd, int bd_per_rhs, const V4<double>* x, V4<double>* y, int n_pix, int nrhs,
                     cudaStream_t s) {
    dim3 g(grid_for(n_pix), nrhs);
    k_bd_apply<<<g, VT, 0, s>>>(bd, bd_per_rhs, x, y, n_pix);
    count_launches(1);
}

// ---------------- PCG ----------------
__device__ __forceinline__ const double* bd_of(const PcgArgs& a, int rhs, int i) {
    return a.bd + ((int64_t)(a.bd_per_rhs ? rhs : 0) * a.n_pix + i) * 6;
}

// x = 0, r = b, p = 0; ||b||.
__global__ void k_pcg_init(const PcgArgs a, const V4<double>* b) {
    const int rhs = blockIdx.y;
    const int64_t off = (int64_t)rhs * a.n_pix;
    double acc[1] = {0.0};
    const V4<double> zero{0, 0, 0, 0};
    PIX_LOOP(i) {
        const V4<double> bv = b[off + i];
        a.x[off + i] = zero;
        a.r[off + i] = bv;
        a.p[off + i] = zero;
        acc[0] += dot3(bv, bv);
    }
    double* part = a.partial + ((int64_t)blockIdx.x * a.nrhs + rhs) * 1;
    block_partials<1>(acc, part);
    if (last_block(a.counter, rhs)) {
        const double bb = gather_partial<1>(a.partial, gridDim.x, a.nrhs, rhs, 0);
        if (threadIdx.x == 0) {
            RhsState& st = a.st[rhs];
            st.bnorm = sqrt(bb);
            st.relres = 1.0;
            st.iters = 0;
            st.status = 0;
            st.alpha = st.beta = 0.0;
            st.active = (bb > 0.0 && st.max_iter > 0) ? 1 : 0;
            if (!(bb > 0.0)) st.relres = 0.0;
            a.hist[(int64_t)rhs * a.hist_stride] = st.relres;
            a.counter[rhs] = 0;
        }
    }
}

// z = M_BD r and r^T z; finalize_beta: beta = rz_new / rz (else rz = rz_new only).
__global__ void k_bd_dot(const PcgArgs a, int finalize_beta) {
    const int rhs = blockIdx.y;
    if (!a.st[rhs].active) return;
    const int64_t off = (int64_t)rhs * a.n_pix;
    double acc[1] = {0.0};
    PIX_LOOP(i) {
        const V4<double> rv = a.r[off + i];
        const V4<double> zv = bd_mul(bd_of(a, rhs, i), rv);
        a.z[off + i] = zv;
        acc[0] += dot3(rv, zv);
    }
    block_partials<1>(acc, a.partial + ((int64_t)blockIdx.x * a.nrhs + rhs));
    if (last_block(a.counter, rhs)) {
        const double rz = gather_partial<1>(a.partial, gridDim.x, a.nrhs, rhs, 0);
        if (threadIdx.x == 0) {
            RhsState& st = a.st[rhs];
            st.beta = finalize_beta ? rz / st.rz : 0.0;
            st.rz = rz;
            a.counter[rhs] = 0;
        }
    }
}

// p = z + beta p; src = p in the operator precision; qacc = 0.
__device__ __forceinline__ void pcg_direction(const PcgArgs& a, int64_t j, double beta) {
    const V4<double> zv = a.z[j];
    V4<double> pv = a.p[j];
    pv = V4<double>{zv.x + beta * pv.x, zv.y + beta * pv.y, zv.z + beta * pv.z, 0.0};
    a.p[j] = pv;
    if (a.src_f32 == 1) {
        reinterpret_cast<V4<float>*>(a.src)[j] = V4<float>{(float)pv.x, (float)pv.y, (float)pv.z, 0.0f};
        reinterpret_cast<V4<float>*>(a.qacc)[j] = V4<float>{0.f, 0.f, 0.f, 0.f};
    } else if (a.src_f32 == 2) {
        // double-float operator input, float64 accumulators
        reinterpret_cast<V4<df>*>(a.src)[j] = V4<df>{df(pv.x), df(pv.y), df(pv.z), df(0.0)};
        reinterpret_cast<V4<double>*>(a.qacc)[j] = V4<double>{0, 0, 0, 0};
    } else {
        reinterpret_cast<V4<double>*>(a.src)[j] = pv;
        reinterpret_cast<V4<double>*>(a.qacc)[j] = V4<double>{0, 0, 0, 0};
    }
}
__global__ void k_pcg_src(const PcgArgs a) {
    const int rhs = blockIdx.y;
    if (!a.st[rhs].active) return;
    const double beta = a.st[rhs].beta;
    const int64_t off = (int64_t)rhs * a.n_pix;
    PIX_LOOP(i) pcg_direction(a, off + i, beta);
}

__device__ __forceinline__ V4<double> load_q(const PcgArgs& a, int64_t j) {
    return a.q32 ? ld4(a.q32 + j) : a.q64[j];
}

// p^T q; alpha = rz / pq; a non-positive or non-finite pq is a breakdown.
__global__ void k_pcg_pq(const PcgArgs a) {
    const int rhs = blockIdx.y;
    if (!a.st[rhs].active) return;
    const int64_t off = (int64_t)rhs * a.n_pix;
    double acc[1] = {0.0};
    PIX_LOOP(i) acc[0] += dot3(a.p[off + i], load_q(a, off + i));
    block_partials<1>(acc, a.partial + ((int64_t)blockIdx.x * a.nrhs + rhs));
    if (last_block(a.counter, rhs)) {
        const double pq = gather_partial<1>(a.partial, gridDim.x, a.nrhs, rhs, 0);
        if (threadIdx.x == 0) {
            RhsState& st = a.st[rhs];
            st.pq = pq;
            if (!(pq > 0.0) || !isfinite(pq) || !isfinite(st.rz)) {
                st.status = 6;
                st.active = 0;
                st.alpha = 0.0;
            } else {
                st.alpha = st.rz / pq;
            }
            if (a.ahist) a.ahist[(int64_t)rhs * a.hist_stride + st.iters] = st.alpha;
            a.counter[rhs] = 0;
        }
    }
}

// x += alpha p, r -= alpha q, ||r||; with M_BD fused (two_level == 0) also
// z = M_BD r and r^T z, with M_2l (two_level == 1) t = Z^T r (k values)
// and u = E^-1 t.
template <int TWO_LEVEL>
__global__ void k_pcg_update(const PcgArgs a) {
    const int rhs = blockIdx.y;
    if (!a.st[rhs].active) return;
    const double alpha = a.st[rhs].alpha;
    const int64_t off = (int64_t)rhs * a.n_pix;
    double acc[2] = {0.0, 0.0};
    PIX_LOOP(i) {
        const V4<double> pv = a.p[off + i];
        const V4<double> qv = load_q(a, off + i);
        V4<double> xv = a.x[off + i], rv = a.r[off + i];
        xv.x += alpha * pv.x;
        xv.y += alpha * pv.y;
        xv.z += alpha * pv.z;
        rv.x -= alpha * qv.x;
        rv.y -= alpha * qv.y;
        rv.z -= alpha * qv.z;
        a.x[off + i] = xv;
        a.r[off + i] = rv;
        acc[0] += dot3(rv, rv);
        if (!TWO_LEVEL) {
            const V4<double> zv = bd_mul(bd_of(a, rhs, i), rv);
            a.z[off + i] = zv;
            acc[1] += dot3(rv, zv);
        }
    }
    block_partials<2>(acc, a.partial + ((int64_t)blockIdx.x * a.nrhs + rhs) * 2);
    if (last_block(a.counter, rhs)) {
        const double rr = gather_partial<2>(a.partial, gridDim.x, a.nrhs, rhs, 0);
        const double rz_new = TWO_LEVEL ? 0.0 : gather_partial<2>(a.partial, gridDim.x, a.nrhs, rhs, 1);
        if (threadIdx.x == 0) {
            RhsState& st = a.st[rhs];
            st.iters += 1;
            st.relres = sqrt(rr) / st.bnorm;
            a.hist[(int64_t)rhs * a.hist_stride + st.iters] = st.relres;
            if (!isfinite(st.relres)) {
                st.status = 6;
                st.active = 0;
            } else if (st.relres <= st.tol) {
                st.active = 0;
            } else if (st.iters >= st.max_iter) {
                st.status = 5;
                st.active = 0;
            }
            if (!TWO_LEVEL) {
                const double rz = rz_new;
                st.beta = rz / st.rz;
                st.rz = rz;
                if (a.bhist) a.bhist[(int64_t)rhs * a.hist_stride + st.iters - 1] = st.beta;
            }
            a.counter[rhs] = 0;
        }
    }
}

// The whole of a PCG iteration behind the product, with M_BD, for small maps:
// alpha from p^T q; x, r and z = M_BD r with ||r|| and r^T z; beta; the next
// search direction, the operator's input and cleared accumulators.  One cluster
// of eight CTAs per right-hand side sums over its CTAs through distributed
// shared memory (rank order), so the three launches and their last-CTA
// reductions (21 us an iteration at 1024 pixels) become one of 11 us.  Used up to
// STEP_MAX_PIX pixels, the largest size measured: whole iterations of 4096
// pixels, product included, 46 -> 35 us alone, 64 -> 44 for 8 maps, 245 -> 152
// for 64 (the product's share of that gain is not told apart).
constexpr int STEP_CL = 8;
constexpr int STEP_MAX_PIX = 4096;
// Scalars are formed by one warp each: a float64 division is some twenty
// instructions of 64 cycles, and every warp doing its own cost 4 us a step.
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The sum over the cluster's CTAs of *slot, in a fixed order, for a whole warp (behind a cluster barrier).
__device__ __forceinline__ double ranks_sum(const double* slot) {
    uint32_t ra;
    double x;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;"
                 : "=r"(ra)
                 : "r"((uint32_t)__cvta_generic_to_shared(slot)), "r"(threadIdx.x & (STEP_CL - 1)));
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(x) : "r"(ra) : "memory");
#pragma unroll
    for (int d = 1; d < STEP_CL; d <<= 1) x += __shfl_xor_sync(0xffffffffu, x, d);
    return x;
}
__global__ void __cluster_dims__(STEP_CL, 1, 1) __launch_bounds__(VT) k_pcg_step(const PcgArgs a) {
    __shared__ double red[2][VT / 32], slot[3], scal[3];   // scal: pq, relres, r^T z
    const int rhs = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const RhsState st0 = a.st[rhs];   // read before rank 0 updates it (behind the first cluster barrier)
    if (!st0.active) return;          // the whole cluster
    const int64_t off = (int64_t)rhs * a.n_pix;
    double acc = 0.0;
    PIX_LOOP(i) acc += dot3(a.p[off + i], load_q(a, off + i));
    acc = warp_sum(acc);
    if (lane == 0) red[0][warp] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
        double t = 0.0;
        for (int w = 0; w < VT / 32; ++w) t += red[0][w];
        slot[0] = t;
    }
    cluster_barrier();
    __shared__ double s_alpha, s_beta;
    __shared__ bool s_broken;
    if (warp == 0) {
        const double pq = ranks_sum(slot);
        if (lane == 0) {
            s_broken = !(pq > 0.0) || !isfinite(pq) || !isfinite(st0.rz);
            s_alpha = s_broken ? 0.0 : st0.rz / pq;
            scal[0] = pq;
        }
    }
    __syncthreads();
    const bool broken = s_broken;
    const double alpha = s_alpha;
    double rr = 0.0, rz = 0.0;
    if (!broken) {
        PIX_LOOP(i) {
            const V4<double> pv = a.p[off + i];
            const V4<double> qv = load_q(a, off + i);
            V4<double> xv = a.x[off + i], rv = a.r[off + i];
            xv.x += alpha * pv.x;
            xv.y += alpha * pv.y;
            xv.z += alpha * pv.z;
            rv.x -= alpha * qv.x;
            rv.y -= alpha * qv.y;
            rv.z -= alpha * qv.z;
            a.x[off + i] = xv;
            a.r[off + i] = rv;
            rr += dot3(rv, rv);
            const V4<double> zv = bd_mul(bd_of(a, rhs, i), rv);
            a.z[off + i] = zv;
            rz += dot3(rv, zv);
        }
    }
    rr = warp_sum(rr);
    rz = warp_sum(rz);
    if (lane == 0) {
        red[0][warp] = rr;
        red[1][warp] = rz;
    }
    __syncthreads();
    if (lane == 0 && warp < 2) {
        double t = 0.0;
        for (int w = 0; w < VT / 32; ++w) t += red[warp][w];
        slot[1 + warp] = t;
    }
    cluster_barrier();
    if (warp == 0) {
        const double t = ranks_sum(slot + 1);
        if (lane == 0) scal[1] = broken ? st0.relres : sqrt(t) / st0.bnorm;
    } else if (warp == 1) {
        const double t = ranks_sum(slot + 2);
        if (lane == 0) {
            scal[2] = t;
            s_beta = broken ? st0.beta : t / st0.rz;
        }
    }
    __syncthreads();
    RhsState st = st0;
    st.pq = scal[0];
    st.alpha = alpha;
    if (broken) {
        st.status = 6;
        st.active = 0;
    } else {
        st.iters += 1;
        st.relres = scal[1];
        st.beta = s_beta;
        st.rz = scal[2];
        if (!isfinite(st.relres)) {
            st.status = 6;
            st.active = 0;
        } else if (st.relres <= st.tol) {
            st.active = 0;
        } else if (st.iters >= st.max_iter) {
            st.status = 5;
            st.active = 0;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        a.st[rhs] = st;
        if (a.ahist) a.ahist[(int64_t)rhs * a.hist_stride + st0.iters] = alpha;
        if (!broken) {
            a.hist[(int64_t)rhs * a.hist_stride + st.iters] = st.relres;
            if (a.bhist) a.bhist[(int64_t)rhs * a.hist_stride + st.iters - 1] = st.beta;
        }
    }
    if (st.active) {
        PIX_LOOP(i) pcg_direction(a, off + i, st.beta);
    }
    cluster_barrier();   // no CTA leaves while another may still read its sums
}

// t = Z^T v for the k coarse vectors (one warp per coarse vector per pass),
// then u = E^-1 t in the last CTA.
template <bool F32>
__global__ void k_m2l_ztr(const PcgArgs a, const V4<double>* v) {
    const int rhs = blockIdx.y;
    if (a.st && !a.st[rhs].active) return;
    const int64_t off = (int64_t)rhs * a.n_pix;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = VT / 32;
    const int k = a.k;
    // this CTA's pixel range
    const int chunk = (a.n_pix + gridDim.x - 1) / gridDim.x;
    const int i0 = blockIdx.x * chunk, i1 = min(a.n_pix, i0 + chunk);
    // float32: the residual of the chunk is converted once and shared by the warps (each coarse vector's warp
    // converted it anew: 32 -> 14 us at 65536 pixels, k = 32)
    constexpr int STAGE = F32 ? 1024 : 1;
    __shared__ float vx[3][STAGE];
    const bool staged = F32 && chunk <= STAGE;
    if (staged) {
        for (int i = i0 + threadIdx.x; i < i1; i += VT) {
            const V4<double> x = v[off + i];
            vx[0][i - i0] = d2f_trunc(x.x);
            vx[1][i - i0] = d2f_trunc(x.y);
            vx[2][i - i0] = d2f_trunc(x.z);
        }
        __syncthreads();
    }
    for (int c = warp; c < k; c += nw) {
        double s = 0.0;
        if (staged) {
            const V4<float>* zc = a.Z32 + (int64_t)c * a.n_pix;
            float sf = 0.0f;
#pragma unroll 8
            for (int i = i0 + lane; i < i1; i += 32) {
                const V4<float> z = zc[i];
                sf = fmaf(z.x, vx[0][i - i0], fmaf(z.y, vx[1][i - i0], fmaf(z.z, vx[2][i - i0], sf)));
            }
            s = f2d_exact(sf);
        } else if (F32) {
            // float32 products summed per lane in float32 (a few dozen terms), the lanes in float64
            const V4<float>* zc = a.Z32 + (int64_t)c * a.n_pix;
            float sf = 0.0f;
#pragma unroll 4
            for (int i = i0 + lane; i < i1; i += 32) {
                const V4<float> z = zc[i];
                const V4<double> x = v[off + i];
                sf = fmaf(z.x, d2f_trunc(x.x), fmaf(z.y, d2f_trunc(x.y), fmaf(z.z, d2f_trunc(x.z), sf)));
            }
            s = f2d_exact(sf);
        } else {
            const V4<double>* zc = a.Z + (int64_t)c * a.n_pix;
#pragma unroll 4
            for (int i = i0 + lane; i < i1; i += 32) s += dot3(zc[i], v[off + i]);
        }
        s = warp_sum(s);
        if (lane == 0) a.partial[((int64_t)blockIdx.x * a.nrhs + rhs) * k + c] = s;
    }
    if (last_block(a.counter, rhs)) {
        __shared__ double t[MM_K_MAX];
        for (int c = warp; c < k; c += nw) {
            const double s = warp_gather(a.partial, gridDim.x, (int64_t)a.nrhs * k, (int64_t)rhs * k + c);
            if (lane == 0) t[c] = s;
        }
        __syncthreads();
        const double* Einv = a.Einv + (int64_t)rhs * a.einv_stride;
        for (int c = threadIdx.x; c < k; c += VT) {
            double s = 0.0;
            for (int j = 0; j < k; ++j) s += Einv[c * k + j] * t[j];
            a.u[(int64_t)rhs * k + c] = s;
        }
        if (threadIdx.x == 0) a.counter[rhs] = 0;
    }
}

// out = M_BD (v - AZ u) + Z u  (Sect. 3.2, Eq. m2l); with finalize_beta >= 0
// it also forms v^T out and updates rz/beta like k_bd_dot.
// G lanes per pixel, each 1/G of the coarse vectors, U of them in flight in float64.
template <int G, int U>
__global__ void k_m2l_apply(const PcgArgs a, const V4<double>* v, V4<double>* out, int finalize_beta) {
    const int rhs = blockIdx.y;
    if (a.st && !a.st[rhs].active) return;
    const int64_t off = (int64_t)rhs * a.n_pix;
    __shared__ double u[MM_K_MAX];
    __shared__ float uf[MM_K_MAX];
    for (int c = threadIdx.x; c < a.k; c += VT) {
        u[c] = a.u[(int64_t)rhs * a.k + c];
        uf[c] = d2f_trunc(u[c]);
    }
    __syncthreads();
    double acc[1] = {0.0};
    const V4<double>* AZ = a.AZ + (int64_t)rhs * a.az_stride;
    const int g = threadIdx.x % G;
    for (int base = blockIdx.x * (VT / G); base < a.n_pix; base += gridDim.x * (VT / G)) {
        const int i = base + threadIdx.x / G;
        const bool in = i < a.n_pix;
        double yx = 0.0, yy = 0.0, yz = 0.0, zx = 0.0, zy = 0.0, zz = 0.0;
        if (in) {
            if (a.Z32) {
                // the coarse sums AZ u and Z u in float32 (mixed precision), the rest in float64
                float fx = 0.0f, fy = 0.0f, fz = 0.0f, hx = 0.0f, hy = 0.0f, hz = 0.0f;
#pragma unroll(G == 1 ? 8 : 4)
                for (int c = g; c < a.k; c += G) {
                    const V4<float> azc = a.AZ32[(int64_t)c * a.n_pix + i];
                    const V4<float> zc = a.Z32[(int64_t)c * a.n_pix + i];
                    const float uc = uf[c];
                    fx = fmaf(azc.x, uc, fx);
                    fy = fmaf(azc.y, uc, fy);
                    fz = fmaf(azc.z, uc, fz);
                    hx = fmaf(zc.x, uc, hx);
                    hy = fmaf(zc.y, uc, hy);
                    hz = fmaf(zc.z, uc, hz);
                }
                yx = f2d_exact(fx);
                yy = f2d_exact(fy);
                yz = f2d_exact(fz);
                zx = f2d_exact(hx);
                zy = f2d_exact(hy);
                zz = f2d_exact(hz);
            } else {
#pragma unroll U
                for (int c = g; c < a.k; c += G) {
                    const V4<double> azc = AZ[(int64_t)c * a.n_pix + i];
                    const V4<double> zc = a.Z[(int64_t)c * a.n_pix + i];
                    const double uc = u[c];
                    yx = fma(azc.x, uc, yx);
                    yy = fma(azc.y, uc, yy);
                    yz = fma(azc.z, uc, yz);
                    zx = fma(zc.x, uc, zx);
                    zy = fma(zc.y, uc, zy);
                    zz = fma(zc.z, uc, zz);
                }
            }
        }
#pragma unroll
        for (int d = 1; d < G; d <<= 1) {
            yx += __shfl_xor_sync(0xffffffffu, yx, d);
            yy += __shfl_xor_sync(0xffffffffu, yy, d);
            yz += __shfl_xor_sync(0xffffffffu, yz, d);
            zx += __shfl_xor_sync(0xffffffffu, zx, d);
            zy += __shfl_xor_sync(0xffffffffu, zy, d);
            zz += __shfl_xor_sync(0xffffffffu, zz, d);
        }
        if (in && g == 0) {
            const V4<double> r = v[off + i];
            V4<double> o = bd_mul(bd_of(a, rhs, i), V4<double>{r.x - yx, r.y - yy, r.z - yz, 0.0});
            o.x += zx;
            o.y += zy;
            o.z += zz;
            out[off + i] = o;
            acc[0] += dot3(r, o);
        }
    }
    if (finalize_beta < 0) return;
    block_partials<1>(acc, a.partial + ((int64_t)blockIdx.x * a.nrhs + rhs));
    if (last_block(a.counter, rhs)) {
        const double rz = gather_partial<1>(a.partial, gridDim.x, a.nrhs, rhs, 0);
        if (threadIdx.x == 0) {
            RhsState& st = a.st[rhs];
            st.beta = finalize_beta ? rz / st.rz : 0.0;
            st.rz = rz;
            a.counter[rhs] = 0;
        }
    }
}

// Lanczos vectors of M_BD A from PCG with M_BD: v_j = z_j / sqrt(r_j^T z_j)
// (right-hand side 0), stored while j < harvest_m.
__global__ void k_harvest(const PcgArgs a) {
    const RhsState st = a.st[0];
    if (!st.active || st.iters >= a.harvest_m) return;
    const double sc = 1.0 / sqrt(st.rz);
    V4<double>* w = a.harvest + (int64_t)st.iters * a.n_pix;
    for (int i = blockIdx.x * VT + threadIdx.x; i < a.n_pix; i += gridDim.x * VT) {
        const V4<double> z = a.z[i];
        w[i] = V4<double>{z.x * sc, z.y * sc, z.z * sc, 0.0};
    }
}
void launch_harvest(const PcgArgs& a, cudaStream_t s) {
    k_harvest<<<a.grid_x, VT, 0, s>>>(a);
    count_launches(1);
}

void launch_pcg_init(const PcgArgs& a, const V4<double>* b, cudaStream_t s) {
    k_pcg_init<<<dim3(a.grid_x, a.nrhs), VT, 0, s>>>(a, b);
    count_launches(1);
}
void launch_pcg_src(const PcgArgs& a, cudaStream_t s) {
    k_pcg_src<<<dim3(a.grid_x, a.nrhs), VT, 0, s>>>(a);
    count_launches(1);
}
bool pcg_step_fits(const PcgArgs& a) { return a.n_pix <= STEP_MAX_PIX; }
void launch_pcg_step(const PcgArgs& a, cudaStream_t s) {
    k_pcg_step<<<dim3(STEP_CL, a.nrhs), VT, 0, s>>>(a);
    count_launches(1);
}
void launch_pcg_pq(const PcgArgs& a, cudaStream_t s) {
    k_pcg_pq<<<dim3(a.grid_x, a.nrhs), VT, 0, s>>>(a);
    count_launches(1);
}
void launch_pcg_update(const PcgArgs& a, int two_level, cudaStream_t s) {
    if (two_level) {
        k_pcg_update<1><<<dim3(a.grid_x, a.nrhs), VT, 0, s>>>(a);
        count_launches(1);
    }
    else {
        k_pcg_update<0><<<dim3(a.grid_x, a.nrhs), VT, 0, s>>>(a);
        count_launches(1);
    }
}
void launch_precond_bd_dot(const PcgArgs& a, int finalize_beta, cudaStream_t s) {
    k_bd_dot<<<dim3(a.grid_x, a.nrhs), VT, 0, s>>>(a, finalize_beta);
    count_launches(1);
}
// CTAs of k_m2l_ztr at most (the partials hold this many entries per value).
int m2l_ztr_grid(int n_pix) { return std::min(304, (n_pix + 63) / 64); }
// Chunks of whole warps (a ragged last row of 32 pixels costs the float64 pipe a full one), at least 64 and at
// most 256 pixels: one CTA per SM over all right-hand sides where that fits, else two.  Microseconds a call, one
// right-hand side, k = 32, float64, with 304 chunks whatever their length / with chunks of 256 / so (all with four
// lanes a pixel up to 16384 pixels and the loops unrolled below): 128 x 128 and 140 x 140 84 / 83 / 75, 180 x 180
// 94 / 83 / 78, 220 x 220 105 / 121 / 104.
static int m2l_grid(int n_pix, int nrhs) {
    auto chunk = [&](int ctas) { return std::max(64, ((n_pix + ctas - 1) / ctas + 31) / 32 * 32); };
    const int w = std::max(2, 304 / std::max(1, nrhs)), c1 = chunk(w / 2), c2 = chunk(w);
    const int c = std::min(256, c1 <= 256 ? c1 : c2);
    return std::min(304, (n_pix + c - 1) / c);
}
void launch_m2l_ztr(const PcgArgs& a, const V4<double>* v, cudaStream_t s) {
    const dim3 grid(m2l_grid(a.n_pix, a.nrhs), a.nrhs);
    if (a.Z32) k_m2l_ztr<true><<<grid, VT, 0, s>>>(a, v);
    else k_m2l_ztr<false><<<grid, VT, 0, s>>>(a, v);
    count_launches(1);
}
// Four lanes per pixel on small maps: the SMs' float64 pipes are filled and the loads of a pixel's vectors are in
// flight together.  From 16384 pixels on (over all right-hand sides) one lane per pixel spares the lanes' sums,
// which are float64 adds, and eight vectors in flight take their place for a single right-hand side.  k = 32, float64,
// us a call, four lanes / one: 100 x 100 72 / 78, 140 x 140 86 / 84, 180 x 180 101 / 93, 256 x 256 126 / 112.  One
// lane, four / eight in flight: 300 x 300 144 / 139; eight right-hand sides of 120 x 120, k = 64: 223 / 252.  Float32
// coarse sums (a.Z32) keep four lanes while all of them fit on the device at once.
void launch_m2l_apply(const PcgArgs& a, const V4<double>* v, V4<double>* out, int finalize_beta, cudaStream_t s) {
    const int rows = std::min(304, (a.n_pix + VT - 1) / VT);
    if ((int64_t)a.n_pix * a.nrhs < (a.Z32 ? 152 * 2048 / 4 : 16384))
        k_m2l_apply<4, 4><<<dim3(m2l_ztr_grid(a.n_pix), a.nrhs), VT, 0, s>>>(a, v, out, finalize_beta);
    else if (a.nrhs == 1)
        k_m2l_apply<1, 8><<<dim3(rows, a.nrhs), VT, 0, s>>>(a, v, out, finalize_beta);
    else
        k_m2l_apply<1, 4><<<dim3(rows, a.nrhs), VT, 0, s>>>(a, v, out, finalize_beta);
    count_launches(1);
}

// ---------------- tall-skinny float64 products ----------------
__global__ void k_multidot(const double* X, int64_t ldx, int m, const double* v, int64_t n, double* h,
                           double* partial, unsigned* counter) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = VT / 32;
    const int64_t chunk = (n + gridDim.x - 1) / gridDim.x;
    const int64_t i0 = blockIdx.x * chunk, i1 = min(n, i0 + chunk);
    for (int r = warp; r < m; r += nw) {
        const double* xr = X + (int64_t)r * ldx;
        double s = 0.0;
        for (int64_t i = i0 + lane; i < i1; i += 32) s += xr[i] * v[i];
        s = warp_sum(s);
        if (lane == 0) partial[(int64_t)blockIdx.x * m + r] = s;
    }
    if (last_block(counter, 0)) {
        for (int r = warp; r < m; r += nw) {
            const double s = warp_gather(partial, gridDim.x, m, r);
            if (lane == 0) h[r] = s;
        }
        if (threadIdx.x == 0) counter[0] = 0;
    }
}
void launch_multidot(const double* X, int64_t ldx, int m, const double* v, int64_t n, double* h, double* partial,
                     unsigned* counter, int grid_x, cudaStream_t s) {
    if (m <= 0) return;
    k_multidot<<<grid_x, VT, 0, s>>>(X, ldx, m, v, n, h, partial, counter);
    count_launches(1);
}

__global__ void k_sub_combo(const double* X, int64_t ldx, int m, const double* h, double* v, int64_t n) {
    extern __shared__ double hs[];
    for (int r = threadIdx.x; r < m; r += VT) hs[r] = h[r];
    __syncthreads();
    for (int64_t i = blockIdx.x * (int64_t)VT + threadIdx.x; i < n; i += (int64_t)gridDim.x * VT) {
        double acc = v[i];
        for (int r = 0; r < m; ++r) acc -= X[(int64_t)r * ldx + i] * hs[r];
        v[i] = acc;
    }
}
void launch_sub_combo(const double* X, int64_t ldx, int m, const double* h, double* v, int64_t n, cudaStream_t s) {
    if (m <= 0) return;
    k_sub_combo<<<grid_for(n), VT, m * sizeof(double), s>>>(X, ldx, m, h, v, n);
    count_launches(1);
}

// Y[c][i] = sum_r X[r][i] C[r*kc + c]: eight outputs per thread, a group of
// eight columns per grid row, so a small map still fills the device (85 -> 25 us
// for 32 columns of a 1024-pixel map).
__global__ void k_combo(const double* X, int64_t ldx, int m, const double* C, int kc, double* Y, int64_t ldy,
                        int64_t n) {
    const int c0 = 8 * blockIdx.y;
    for (int64_t i = blockIdx.x * (int64_t)VT + threadIdx.x; i < n; i += (int64_t)gridDim.x * VT) {
        double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll 4
        for (int r = 0; r < m; ++r) {
            const double xv = X[(int64_t)r * ldx + i];
#pragma unroll
            for (int c = 0; c < 8; ++c)
                if (c0 + c < kc) acc[c] += xv * C[(int64_t)r * kc + c0 + c];
        }
#pragma unroll
        for (int c = 0; c < 8; ++c)
            if (c0 + c < kc) Y[(int64_t)(c0 + c) * ldy + i] = acc[c];
    }
}
void launch_combo(const double* X, int64_t ldx, int m, const double* C, int kc, double* Y, int64_t ldy, int64_t n,
                  cudaStream_t s) {
    if (kc <= 0) return;
    k_combo<<<dim3(grid_for(n), (kc + 7) / 8), VT, 0, s>>>(X, ldx, m, C, kc, Y, ldy, n);
    count_launches(1);
}

// Gram matrices.  A CTA takes a 32 x 32 tile of products over a slice of
// pixels: both operands' slices pass through shared memory (the unused fourth
// entry of a pixel is left out), a thread keeps 2 x 2 sums.  Slices are chosen
// so that about two CTAs per SM run whatever the number of tiles, and the
// slices' sums are added in order by a second kernel, so the result does not
// depend on the schedule.  Bound by the float64 pipe (one product of 32 x 32 at
// 1024 pixels: 7 us at its measured rate); one multidot per column took 38 us
// each on four CTAs there, 1.2 ms a matrix.
constexpr int GT = 32;        // tile edge
constexpr int GP = 8;         // pixels staged at a time
__global__ void __launch_bounds__(256) k_gram(const V4<double>* __restrict__ X, int mx, const V4<double>* __restrict__ Y,
                                              int my, int64_t ld, int64_t n_pix, int64_t per, double* part) {
    __shared__ double xs[3 * GP][GT + 2], ys[3 * GP][GT + 2];
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    const int i0 = blockIdx.x * GT, j0 = blockIdx.y * GT;
    const int64_t p0 = blockIdx.z * per, p1 = p0 + per < n_pix ? p0 + per : n_pix;
    double acc[2][2] = {{0, 0}, {0, 0}};
    const int row = threadIdx.x >> 3, pp = threadIdx.x & 7;   // a thread stages pixel pp of row `row` of both tiles
    for (int64_t p = p0; p < p1; p += GP) {
        V4<double> x{0, 0, 0, 0}, y{0, 0, 0, 0};
        if (p + pp < p1) {
            if (i0 + row < mx) x = X[(int64_t)(i0 + row) * ld + p + pp];
            if (j0 + row < my) y = Y[(int64_t)(j0 + row) * ld + p + pp];
        }
        __syncthreads();
        xs[3 * pp][row] = x.x;
        xs[3 * pp + 1][row] = x.y;
        xs[3 * pp + 2][row] = x.z;
        ys[3 * pp][row] = y.x;
        ys[3 * pp + 1][row] = y.y;
        ys[3 * pp + 2][row] = y.z;
        __syncthreads();
#pragma unroll
        for (int e = 0; e < 3 * GP; ++e) {
            const double a0 = xs[e][tx], a1 = xs[e][tx + 16], b0 = ys[e][ty], b1 = ys[e][ty + 16];
            acc[0][0] = fma(a0, b0, acc[0][0]);
            acc[1][0] = fma(a1, b0, acc[1][0]);
            acc[0][1] = fma(a0, b1, acc[0][1]);
            acc[1][1] = fma(a1, b1, acc[1][1]);
        }
    }
    double* o = part + (int64_t)blockIdx.z * mx * my;
#pragma unroll
    for (int v = 0; v < 2; ++v)
#pragma unroll
        for (int u = 0; u < 2; ++u) {
            const int i = i0 + tx + 16 * u, j = j0 + ty + 16 * v;
            if (i < mx && j < my) o[(int64_t)j * mx + i] = acc[u][v];
        }
}
// Slices added in a fixed order: eight interleaved partial sums, then their sum.
__global__ void __launch_bounds__(VT) k_gram_sum(const double* part, int slices, int64_t n, double* G) {
    __shared__ double red[8][VT / 8];
    const int o = threadIdx.x % (VT / 8), g = threadIdx.x / (VT / 8);
    const int64_t i = (int64_t)blockIdx.x * (VT / 8) + o;
    double s = 0.0;
    if (i < n) {
#pragma unroll 4
        for (int z = g; z < slices; z += 8) s += part[z * n + i];
    }
    red[g][o] = s;
    __syncthreads();
    if (g == 0 && i < n) {
#pragma unroll
        for (int q = 1; q < 8; ++q) s += red[q][o];
        G[i] = s;
    }
}
static int gram_slices(int mx, int my, int64_t n_pix) {
    const int64_t tiles = (int64_t)((mx + GT - 1) / GT) * ((my + GT - 1) / GT);
    const int64_t want = (304 + tiles - 1) / tiles, most = (n_pix + GP - 1) / GP;
    return (int)std::max<int64_t>(1, std::min(want, most));
}
size_t gram_scratch_doubles(int mx, int my, int64_t n_pix) { return (size_t)gram_slices(mx, my, n_pix) * mx * my; }
void launch_gram(const V4<double>* X, int mx, const V4<double>* Y, int my, int64_t n_pix, double* G, double* scratch,
                 cudaStream_t s) {
    const int slices = gram_slices(mx, my, n_pix);
    const int64_t per = ((n_pix + slices - 1) / slices + GP - 1) / GP * GP;
    k_gram<<<dim3((mx + GT - 1) / GT, (my + GT - 1) / GT, slices), 256, 0, s>>>(X, mx, Y, my, n_pix, n_pix, per, scratch);
    k_gram_sum<<<(unsigned)(((int64_t)mx * my + VT / 8 - 1) / (VT / 8)), VT, 0, s>>>(scratch, slices, (int64_t)mx * my, G);
    count_launches(2);
}

__global__ void k_scale(double* v, int64_t n, double f) {
    for (int64_t i = blockIdx.x * (int64_t)VT + threadIdx.x; i < n; i += (int64_t)gridDim.x * VT) v[i] *= f;
}
void launch_scale_host(double* v, int64_t n, double f, cudaStream_t s) {
    if (n > 0) {
        k_scale<<<grid_for(n), VT, 0, s>>>(v, n, f);
        count_launches(1);
    }
}

}  // namespace mm

namespace mm {

// r_out = b - q (float64), and ||r_out||^2 per right-hand side into norms[rhs].
__global__ void k_residual(const V4<double>* b, const V4<double>* q, V4<double>* r_out, double* norms, int n_pix,
                           int nrhs, double* partial, unsigned* counter) {
    const int rhs = blockIdx.y;
    const int64_t off = (int64_t)rhs * n_pix;
    double acc[1] = {0.0};
    for (int i = blockIdx.x * VT + threadIdx.x; i < n_pix; i += gridDim.x * VT) {
        const V4<double> bv = b[off + i], qv = q[off + i];
        const V4<double> rv{bv.x - qv.x, bv.y - qv.y, bv.z - qv.z, 0.0};
        if (r_out) r_out[off + i] = rv;
        acc[0] += dot3(rv, rv);
    }
    block_partials<1>(acc, partial + ((int64_t)blockIdx.x * nrhs + rhs));
    if (last_block(counter, rhs)) {
        const double v = gather_partial<1>(partial, gridDim.x, nrhs, rhs, 0);
        if (threadIdx.x == 0) {
            norms[rhs] = v;
            counter[rhs] = 0;
        }
    }
}
void launch_residual(const V4<double>* b, const V4<double>* q, V4<double>* r_out, double* norms, int n_pix, int nrhs,
                     double* partial, unsigned* counter, int grid_x, cudaStream_t s) {
    k_residual<<<dim3(grid_x, nrhs), VT, 0, s>>>(b, q, r_out, norms, n_pix, nrhs, partial, counter);
    count_launches(1);
}

// y += x over n doubles, only for right-hand sides whose mask entry is set.
__global__ void k_axpy_masked(double* y, const double* x, int64_t n_per, const int32_t* mask) {
    const int rhs = blockIdx.y;
    if (mask && !mask[rhs]) return;
    const int64_t off = (int64_t)rhs * n_per;
    for (int64_t i = blockIdx.x * (int64_t)VT + threadIdx.x; i < n_per; i += (int64_t)gridDim.x * VT)
        y[off + i] += x[off + i];
}
void launch_axpy_masked(double* y, const double* x, int64_t n_per, int nrhs, const int32_t* mask, cudaStream_t s) {
    if (n_per <= 0 || nrhs <= 0) return;
    k_axpy_masked<<<dim3(grid_for(n_per), nrhs), VT, 0, s>>>(y, x, n_per, mask);
    count_launches(1);
}

}  // namespace mm
