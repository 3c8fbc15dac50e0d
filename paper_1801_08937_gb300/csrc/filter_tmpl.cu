// Template-filtered product A x = P^T F P x (and P^T F d, P^T F (d - P x)) for
// ground-based scans: F = F_B W^-1 F_G W^-1 F_B (Sect. 5.1) with the weighted
// template filter F_X = W - W X (X^T W X)^-1 X^T W of Sect. 2.1 (Eq.
// filtnoise), X = B the Legendre polynomials P_0..P_K of each azimuth sweep
// (subscan) and X = G the azimuth-bin indicators of each constant-elevation
// scan (Sect. 4), and W = w_b I on stationary block b (white noise, Sect.
// 4.1).  With W constant on a block both filters are w_b times orthogonal
// projections, so F = w_b (1 - Pi_B)(1 - Pi_G)(1 - Pi_B) on the block.
//
// One CTA per (block, right-hand side); the block's timeline lives in shared
// memory through
//   1. gather y = P x (rows (1, cos 2psi, sin 2psi); (0, cos, sin) for the
//      differenced timeline d^- and (1, 0, 0) for the summed timeline d^+ of
//      Sect. 5.1), or the timeline d, or d - P x;
//   2. y -= B (B^T B)^-1 B^T y per subscan: warps sum the moments
//      sum_i y_i P_j(u_i), u_i = 2 (i + 1/2)/m - 1, multiply by the
//      subscan's inverse Gram matrix (float64, precomputed on the host) and
//      subtract the fit (the order K is a compile-time parameter);
//   3. y -= bin means of y over the block's azimuth bins, all warps over the
//      whole block (runs of equal bins in a warp are summed before one
//      shared-memory atomic per run; folding this into the per-subscan
//      passes was slower);
//   4. step 2 again;
//   5. z = w_b y scattered into the map (P^T), runs of equal pixels summed in
//      the warp first.
// The arithmetic type is float32, float64, or double-float (float32 pairs,
// float64 atomics for the bin sums and the map); the double-float kernel gives
// float64-accurate products from the float32 units, which GB300 issues at 64
// times its float64 rate.
#include "filter_impl.cuh"

namespace mm {

// Most threads per block (tmpl_threads picks).
template <typename T> struct TmplThreads { static constexpr int value = sizeof(T) == 4 ? 512 : 1024; };

// Place of sample i in the block's shared timeline: permuted within groups of
// eight, so that lanes on eight consecutive samples each meet in a bank two at
// a time instead of eight.
__device__ __forceinline__ int ysw(int i) { return i ^ ((i >> 3) & 7); }

__device__ __forceinline__ int shfl_down_t(int v, int d) { return __shfl_down_sync(0xffffffffu, v, d); }
__device__ __forceinline__ float shfl_xor_t(float v, int d) { return __shfl_xor_sync(0xffffffffu, v, d); }
__device__ __forceinline__ double shfl_xor_t(double v, int d) { return __shfl_xor_sync(0xffffffffu, v, d); }
__device__ __forceinline__ df shfl_xor_t(df v, int d) {
    return df(__shfl_xor_sync(0xffffffffu, v.hi, d), __shfl_xor_sync(0xffffffffu, v.lo, d));
}

// 2 / m in the arithmetic type (double-float: from the float64 quotient).
template <typename T> __device__ __forceinline__ T two_over(int m) { return T(2) / T(m); }
template <> __device__ __forceinline__ df two_over<df>(int m) {
    // a float32 quotient and its exact remainder's (a float64 division costs some twenty warp instructions of
    // the float64 pipe, 64 cycles each, in every unit of the projections)
    const float fm = (float)m, q = __fdiv_rn(2.0f, fm);
    return df(q, __fmaf_rn(-q, fm, 2.0f) / fm);
}

// A value in the accumulator type of the bin sums and the map.
__device__ __forceinline__ float to_acc(float v) { return v; }
__device__ __forceinline__ double to_acc(double v) { return v; }
__device__ __forceinline__ double to_acc(df v) { return df_sum64(v); }

template <typename T>
__device__ __forceinline__ T warp_sum_all(T v) {
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) v += shfl_xor_t(v, d);
    return v;
}

// Legendre polynomials P_0..P_3 at u.
template <typename T>
__device__ __forceinline__ void legendre4(T u, T (&p)[4]) {
    p[0] = T(1);
    p[1] = u;
    p[2] = T(1.5) * u * u - T(0.5);
    p[3] = (T(2.5) * u * u - T(1.5)) * u;
}

// Coefficients c = G^-1 m of the subscan's Legendre fit from the moments m
// (every lane holds them after the warp sum).
template <typename T, int K>
__device__ __forceinline__ void fit_coef(const double* __restrict__ gi, const T (&mom)[4], T (&c)[4]) {
#pragma unroll
    for (int j = 0; j <= K; ++j) {
        T acc = T(0);
#pragma unroll
        for (int l = 0; l <= K; ++l) acc += from64<T>(__ldg(gi + j * 4 + l)) * mom[l];
        c[j] = acc;
    }
}

// a * f for an exact float32 factor
__device__ __forceinline__ float mulf(float a, float f) { return a * f; }
__device__ __forceinline__ double mulf(double a, float f) { return a * (double)f; }
__device__ __forceinline__ df mulf(df a, float f) {
    const float p = __fmul_rn(a.hi, f);
    return df(p, __fmaf_rn(a.lo, f, __fmaf_rn(a.hi, f, -p)));
}

// y -= B (B^T B)^-1 B^T y on every subscan of the block.  The subscans' samples
// are cut into parts so that all warps work (a block holds about ten sweeps
// for sixteen or thirty-two warps): unit (subscan, part) sums its moments, the parts' sums
// are added from shared memory in a fixed order, and each unit subtracts the
// fit on its own samples.  Up to first order the polynomials are taken in the
// odd integer t = 2 i + 1 - m = m u, exact in float32, so a sample costs two
// products with it and no evaluation of u (in double-float 38 operations a
// projection instead of 80); four samples in flight per lane hide the sums'
// latency.
constexpr int POLY_UNITS = 64;   // units of one round of the parts' shared sums
template <typename T, int K>
__device__ void project_poly(T* y, T (*part)[4], const TmplArgs& t, int blk, int64_t b0) {
    const int nw = blockDim.x >> 5;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sb0 = t.blk_sub[blk], sb1 = t.blk_sub[blk + 1];
    const int parts = sb1 - sb0 >= 2 * nw ? 1 : (sb1 - sb0 >= nw ? 2 : (sb1 - sb0 >= nw / 2 ? 4 : 6));
    const int per_round = POLY_UNITS / parts;
    for (int r0 = sb0; r0 < sb1; r0 += per_round) {
        const int ns = min(per_round, sb1 - r0), units = ns * parts;
        auto span = [&](int u, int& s, int& o, int& m, int& i0, int& i1) {
            s = r0 + u / parts;
            const int64_t s0 = t.sub_off[s];
            m = (int)(t.sub_off[s + 1] - s0);
            o = (int)(s0 - b0);
            const int len = ((m + parts - 1) / parts + 31) & ~31;
            i0 = min(m, u % parts * len);
            i1 = min(m, i0 + len);
        };
        for (int u = warp; u < units; u += nw) {
            int s, o, m, i0, i1;
            span(u, s, o, m, i0, i1);
            const T inv_m = two_over<T>(m) * T(0.5);
            T mom[2][4] = {{T(0), T(0), T(0), T(0)}, {T(0), T(0), T(0), T(0)}};
            int i = i0 + lane;
            auto add = [&](T (&acc)[4], int at) {
                const T v = y[ysw(o + at)];
                const float tf = (float)(2 * at + 1 - m);
                acc[0] += v;
                if constexpr (K == 1) acc[1] += mulf(v, tf);
                if constexpr (K > 1) {
                    T p[4];
                    legendre4<T>(mulf(inv_m, tf), p);
#pragma unroll
                    for (int j = 1; j <= K; ++j) acc[j] += v * p[j];
                }
            };
            for (; i + 32 < i1; i += 64) {
                add(mom[0], i);
                add(mom[1], i + 32);
            }
            if (i < i1) add(mom[0], i);
#pragma unroll
            for (int j = 0; j <= K; ++j) {
                const T sum = warp_sum_all(mom[0][j] + mom[1][j]);
                if (lane == 0) part[u][j] = sum;
            }
        }
        __syncthreads();
        for (int u = warp; u < units; u += nw) {
            int s, o, m, i0, i1;
            span(u, s, o, m, i0, i1);
            const T inv_m = two_over<T>(m) * T(0.5);
            T mom[4], c[4];
#pragma unroll
            for (int j = 0; j <= K; ++j) {
                mom[j] = part[u / parts * parts][j];
                for (int q = 1; q < parts; ++q) mom[j] += part[u / parts * parts + q][j];
            }
            if constexpr (K == 1) mom[1] = mom[1] * inv_m;
            fit_coef<T, K>(t.ginv + (int64_t)s * 16, mom, c);
            if constexpr (K == 1) c[1] = c[1] * inv_m;
#pragma unroll 4
            for (int i = i0 + lane; i < i1; i += 32) {
                const float tf = (float)(2 * i + 1 - m);
                T fit = c[0];
                if constexpr (K == 1) fit += mulf(c[1], tf);
                if constexpr (K > 1) {
                    T p[4];
                    legendre4<T>(mulf(inv_m, tf), p);
#pragma unroll
                    for (int j = 1; j <= K; ++j) fit += c[j] * p[j];
                }
                y[ysw(o + i)] -= fit;
            }
        }
        __syncthreads();
    }
}

// Map components a pointing row touches: stokes 0 (I, Q, U), 1 (Q, U: the
// differenced timeline), 2 (I: the summed timeline).
template <int ST> struct StokesCols { static constexpr int n = 3, c0 = 0; };
template <> struct StokesCols<1> { static constexpr int n = 2, c0 = 1; };
template <> struct StokesCols<2> { static constexpr int n = 1, c0 = 0; };

template <typename A> __device__ __forceinline__ A& vcomp(V4<A>* q, int c) {
    return c == 0 ? q->x : (c == 1 ? q->y : q->z);
}

// P^T of a warp's 256 consecutive samples, eight per lane, for NC map
// components starting at C0 (see scatter8_t); val(j, w) gives the NC
// contributions of sample j.
template <typename T, int NC, int C0, typename F>
__device__ __forceinline__ void tmpl_scatter8(const int (&p)[8], V4<typename AccT<T>::type>* q, F val) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    auto flush = [&](int px, const T (&s)[NC]) {
        V4<typename AccT<T>::type>* dst = q + px;
        if constexpr (NC == 3 && std::is_same<T, float>::value) {
            atomic_add3(dst, s[0], s[1], s[2]);
        } else {
#pragma unroll
            for (int c = 0; c < NC; ++c) atomicAdd(&vcomp(dst, C0 + c), to_acc(s[c]));
        }
    };
    T a[NC], b[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) a[c] = b[c] = T(0);
    bool multi = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (j > 0 && p[j] != p[j - 1]) {
            if (multi) {
                if (p[j - 1] >= 0) flush(p[j - 1], a);
            } else {
#pragma unroll
                for (int c = 0; c < NC; ++c) b[c] = a[c];
                multi = true;
            }
#pragma unroll
            for (int c = 0; c < NC; ++c) a[c] = T(0);
        }
        if (p[j] >= 0) {
            T w[NC];
            val(j, w);
#pragma unroll
            for (int c = 0; c < NC; ++c) a[c] += w[c];
        }
    }
    const int plast = __shfl_up_sync(FULL, p[7], 1);
    const bool give = multi && lane > 0 && p[0] == plast;
    T r[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) r[c] = shfl_down_t(b[c], 1);
    if (__shfl_down_sync(FULL, (int)give, 1) && lane < 31) {
#pragma unroll
        for (int c = 0; c < NC; ++c) a[c] += r[c];
    }
    if (multi && !give && p[0] >= 0) flush(p[0], b);
    if (p[7] >= 0) flush(p[7], a);
}

// Sums and counts over a warp's 256 consecutive samples by azimuth bin (g < 0:
// none): a bin lasts many samples, so a run covers several lanes.  Within a
// lane the first and the last run are kept apart (runs strictly inside go out
// directly); the last run takes in the following lanes' leading runs while
// they continue it, by doubling over lanes, and only the lane where a run
// starts adds it to the block's sums.
template <typename T, typename Acc>
__device__ __forceinline__ void bin_sums8(const int (&g)[8], const T (&v)[8], Acc* gsum, int* gcnt) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    auto flush = [&](int bin, T s, int n) {
        atomicAdd(gsum + bin, to_acc(s));
        atomicAdd(gcnt + bin, n);
    };
    T a = T(0), b = T(0);
    int na = 0, nb = 0;
    bool multi = false;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
        if (j > 0 && g[j] != g[j - 1]) {
            if (multi) {
                if (g[j - 1] >= 0) flush(g[j - 1], a, na);
            } else {
                b = a;
                nb = na;
                multi = true;
            }
            a = T(0);
            na = 0;
        }
        a += v[j];
        ++na;
    }
    // what the next lane hands over: its leading run, if it continues this lane's last one
    T x = shfl_down_t(multi ? b : a, 1);
    int nx = __shfl_down_sync(FULL, multi ? nb : na, 1);
    const int gnext = __shfl_down_sync(FULL, g[0], 1);
    const bool wnext = !__shfl_down_sync(FULL, (int)multi, 1);
    const bool cont = lane < 31 && gnext == g[7];
    if (!cont) {
        x = T(0);
        nx = 0;
    }
    bool chain = cont && wnext;   // the next lane is one run: what it takes in comes here too
#pragma unroll 1
    for (int d = 1; __any_sync(FULL, chain); d <<= 1) {
        const T o = shfl_down_t(x, d);
        const int no = __shfl_down_sync(FULL, nx, d);
        const bool co = __shfl_down_sync(FULL, (int)chain, d) != 0;
        if (chain) {
            x += o;
            nx += no;
        }
        chain = chain && co;
    }
    const int glast = __shfl_up_sync(FULL, g[7], 1);
    const bool head = lane == 0 || g[0] != glast;   // the lane's first run starts here
    if (multi && head && g[0] >= 0) flush(g[0], b, nb);
    if ((multi || head) && g[7] >= 0) flush(g[7], a + x, na + nx);
}

template <typename T, bool FROM_TOD, int K, int ST>
__global__ void __launch_bounds__(TmplThreads<T>::value) k_filter_tmpl(const FilterArgs a, const TmplArgs t) {
    const int TMPL_NT = blockDim.x;
    extern __shared__ __align__(16) unsigned char smraw[];
    const int blk = blockIdx.x, rhs = blockIdx.y;
    if (a.state && !a.state[rhs].active) return;
    const int64_t b0 = t.block_off[blk];
    const int nb = (int)(t.block_off[blk + 1] - b0);
    using Acc = typename AccT<T>::type;
    static_assert(sizeof(Acc) == sizeof(T), "bin means overwrite the bin sums in place");
    T* y = reinterpret_cast<T*>(smraw);
    Acc* gsum = reinterpret_cast<Acc*>(y + ((nb + 7) & ~7));
    int* gcnt = reinterpret_cast<int*>(gsum + t.n_bins);
    __shared__ T part[K >= 0 ? POLY_UNITS : 1][4];
    const T iw = ST == 1 ? T(0) : T(1);   // I column of P
    const T pw = ST == 2 ? T(0) : T(1);   // Q, U columns
    const V4<T>* xm = nullptr;
    if (!FROM_TOD) xm = reinterpret_cast<const V4<T>*>(a.src) + (int64_t)rhs * a.n_pix;
    else if (a.xmap) xm = reinterpret_cast<const V4<T>*>(a.xmap) + (int64_t)rhs * a.n_pix;
    // 1. gather (float32 and double-float: four consecutive samples per thread, vector pointing loads)
    if constexpr (!std::is_same<T, double>::value) {
        for (int u = threadIdx.x; 4 * u < nb; u += TMPL_NT) {
            const int i0 = 4 * u;
            const int64_t t0 = b0 + i0;
            int p[4];
            float ps[4];
            if constexpr (ST == 2) load4_pix(a, t0, true, nb - i0, p);   // intensity rows need no angle
            else load4(a, t0, true, nb - i0, p, ps);
            T v[4] = {T(0), T(0), T(0), T(0)};
            if (FROM_TOD) {
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (i0 + j < nb)
                        v[j] = a.tod_is_float ? T(__ldg(reinterpret_cast<const float*>(a.src) + rhs * a.n_samples + t0 + j))
                                              : from64<T>(__ldg(reinterpret_cast<const double*>(a.src) + rhs * a.n_samples + t0 + j));
            }
            if (xm) {
                V4<T> m[4];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (p[j] >= 0) m[j] = ldmap<T>(xm + p[j]);
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (p[j] >= 0) {
                        T px;
                        if constexpr (ST == 2) {
                            px = m[j].x;
                        } else {
                            T c, s;
                            weights_from(a, t0 + j, ps[j], c, s);
                            px = ST == 1 ? c * m[j].y + s * m[j].z : m[j].x + (c * m[j].y + s * m[j].z);
                        }
                        v[j] = FROM_TOD ? v[j] - px : px;
                    }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j)
                if (i0 + j < nb) y[ysw(i0 + j)] = v[j];
        }
    } else
    for (int i = threadIdx.x; i < nb; i += TMPL_NT) {
        const int64_t ts = b0 + i;
        T v = T(0);
        if (FROM_TOD)
            v = a.tod_is_float ? T(__ldg(reinterpret_cast<const float*>(a.src) + rhs * a.n_samples + ts))
                               : from64<T>(__ldg(reinterpret_cast<const double*>(a.src) + rhs * a.n_samples + ts));
        if (xm) {
            const int p = __ldg(a.pix + ts);
            if (p >= 0) {
                T c, s;
                weights(a, ts, c, s);
                const V4<T> m = ldmap<T>(xm + p);
                const T px = iw * m.x + pw * (c * m.y + s * m.z);
                v = FROM_TOD ? v - px : px;
            }
        }
        y[ysw(i)] = v;
    }
    for (int i = threadIdx.x; i < t.n_bins; i += TMPL_NT) {
        gsum[i] = Acc(0);
        gcnt[i] = 0;
    }
    __syncthreads();
    const bool ground = t.az && t.n_bins > 0;
    // 2. (1 - Pi_B) y (one warp per subscan)
    if constexpr (K >= 0) {
        project_poly<T, K>(y, part, t, blk, b0);
    }
    if (ground) {
        // 3. y - azimuth-bin means over the block (all warps, eight samples per lane)
        for (int base = (threadIdx.x >> 5) * 256; base < nb; base += TMPL_NT * 8) {
            const int i0 = base + 8 * (threadIdx.x & 31);
            int g[8];
            T v[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                g[j] = -1;
                v[j] = T(0);
                if (i0 + j < nb) {
                    g[j] = __ldg(t.az + b0 + i0 + j);
                    if (g[j] < 0 || g[j] >= t.n_bins) g[j] = -1;   // out-of-range bins belong to no column
                    v[j] = y[ysw(i0 + j)];
                }
            }
            bin_sums8<T>(g, v, gsum, gcnt);
        }
        __syncthreads();
        // bin means, in place of the sums (one division per bin, not per sample)
        T* gmean = reinterpret_cast<T*>(gsum);
        for (int i = threadIdx.x; i < t.n_bins; i += TMPL_NT) {
            const Acc sm = gsum[i];
            const int n = gcnt[i];
            gmean[i] = n > 0 ? from64<T>(sm / Acc(n)) : T(0);
        }
        __syncthreads();
        for (int i = threadIdx.x; i < nb; i += TMPL_NT) {
            const int g = __ldg(t.az + b0 + i);
            if (g >= 0 && g < t.n_bins) y[ysw(i)] -= gmean[g];
        }
        __syncthreads();
        // 4. (1 - Pi_B) again
        if constexpr (K >= 0) {
            project_poly<T, K>(y, part, t, blk, b0);
        }
    }
    // without a ground template F_B W^-1 F_B = w_b (1 - Pi_B)^2 = w_b (1 - Pi_B): one projection
    // 5. weight and scatter
    V4<Acc>* q = reinterpret_cast<V4<Acc>*>(a.dst) + (int64_t)rhs * a.n_pix;
    const T wb = T(t.w_block[blk]);
    constexpr int NC = StokesCols<ST>::n;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int base = warp * 256; base < nb; base += TMPL_NT * 8) {
        const int i0 = base + 8 * lane;
        const int64_t t0 = b0 + i0;
        int p[8];
        float ps[8] = {0, 0, 0, 0, 0, 0, 0, 0};
        {
            int (&pl)[4] = *reinterpret_cast<int (*)[4]>(p), (&ph)[4] = *reinterpret_cast<int (*)[4]>(p + 4);
            float (&fl)[4] = *reinterpret_cast<float (*)[4]>(ps), (&fh)[4] = *reinterpret_cast<float (*)[4]>(ps + 4);
            if constexpr (ST != 2 && std::is_same<T, float>::value) {   // only float32 rows compute their weights
                load4(a, t0, true, nb - i0, pl, fl);
                load4(a, t0 + 4, true, nb - i0 - 4, ph, fh);
            } else {
                load4_pix(a, t0, true, nb - i0, pl);
                load4_pix(a, t0 + 4, true, nb - i0 - 4, ph);
            }
        }
        const bool pairs = (t0 & 1) == 0 && i0 + 8 <= nb;
        T c2[2], s2[2];
        tmpl_scatter8<T, NC, StokesCols<ST>::c0>(p, q, [&](int j, T (&w)[NC]) {
            const T z = wb * y[ysw(i0 + j)];
            if constexpr (ST == 2) {
                w[0] = z;
            } else {
                T c, sn;
                if constexpr (std::is_same<T, float>::value) {
                    weights_from(a, t0 + j, ps[j], c, sn);
                } else if (pairs) {
                    weights2(a, t0 + (j & ~1), c2, s2);   // loaded once per pair
                    c = c2[j & 1];
                    sn = s2[j & 1];
                } else {
                    weights(a, t0 + j, c, sn);
                }
                if constexpr (ST == 0) w[0] = z;
                w[NC - 2] = z * c;
                w[NC - 1] = z * sn;
            }
        });
    }
}

size_t tmpl_smem_bytes(int64_t max_block, int n_bins, bool f64) {
    const size_t e = f64 ? 8 : 4;
    return (size_t)((max_block + 1) & ~1LL) * e + (size_t)n_bins * (e + 4);
}

// Threads of a CTA.  At 64 registers an SM holds 1024 threads of the 8-byte
// types, in as many CTAs as the blocks' timelines leave shared memory for:
// several small CTAs hide one another's barriers and serial parts.  Double-float,
// order 1 + ground, ms with 256 / 512 / 1024 threads: blocks of 16384 (one CTA
// fits) 1.199 / 0.887 / 0.825, of 12000 (two) 0.095 / 0.093 / 0.124, of 8192
// 0.155 / 0.160 / 0.223; order 3, blocks of 4096 0.094 / 0.114 / 0.156; 24 blocks
// of 7000, fewer than SMs, 0.054 / 0.049 / 0.050.  Native float64 is bound by the
// float64 pipe, which few warps keep busy: blocks of 16384 0.296 / 0.292 / 0.380,
// of 8192 0.339 / 0.398 / 0.529, 24 blocks of 7000 0.087 / 0.093 / 0.117.
template <typename T> static int tmpl_threads(size_t smem, int64_t ctas) {
    if (sizeof(T) == 4) return 512;
    const size_t fit = (228 * 1024) / (smem + 2048);
    if (std::is_same<T, double>::value) return fit >= 2 ? 256 : 512;
    return fit < 2 ? 1024 : (fit == 2 || ctas <= 152 ? 512 : 256);
}

template <typename T, bool FROM_TOD, int K, int ST>
static void launch_tmpl_ks(const FilterArgs& a, const TmplArgs& t, int nrhs, cudaStream_t s) {
    const size_t sm = tmpl_smem_bytes(t.max_block, t.n_bins, sizeof(T) == 8) + 64;   // whole groups of eight samples
    static std::atomic<size_t> configured{0};
    raise_smem_once(configured, sm, [](size_t v) {
        cudaFuncSetAttribute(k_filter_tmpl<T, FROM_TOD, K, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)v);
    });
    const int threads = tmpl_threads<T>(sm, t.n_blocks * (int64_t)nrhs);
    k_filter_tmpl<T, FROM_TOD, K, ST><<<dim3(t.n_blocks, nrhs), threads, sm, s>>>(a, t);
    count_launches(1);
}
template <typename T, bool FROM_TOD, int K>
static void launch_tmpl_k(const FilterArgs& a, const TmplArgs& t, int nrhs, cudaStream_t s) {
    switch (t.stokes) {
        case 1: return launch_tmpl_ks<T, FROM_TOD, K, 1>(a, t, nrhs, s);
        case 2: return launch_tmpl_ks<T, FROM_TOD, K, 2>(a, t, nrhs, s);
        default: return launch_tmpl_ks<T, FROM_TOD, K, 0>(a, t, nrhs, s);
    }
}

template <typename T, bool FROM_TOD>
static void launch_tmpl_t(const FilterArgs& a, const TmplArgs& t, int nrhs, cudaStream_t s) {
    switch (t.order) {
        case 0: return launch_tmpl_k<T, FROM_TOD, 0>(a, t, nrhs, s);
        case 1: return launch_tmpl_k<T, FROM_TOD, 1>(a, t, nrhs, s);
        case 2: return launch_tmpl_k<T, FROM_TOD, 2>(a, t, nrhs, s);
        case 3: return launch_tmpl_k<T, FROM_TOD, 3>(a, t, nrhs, s);
        default: return launch_tmpl_k<T, FROM_TOD, -1>(a, t, nrhs, s);
    }
}

void launch_filter_tmpl(const FilterArgs& a, const TmplArgs& t, int nrhs, int prec, bool from_tod, cudaStream_t s) {
    if (t.n_blocks <= 0 || nrhs <= 0) return;
    if (prec == 2) {
        if (from_tod) launch_tmpl_t<df, true>(a, t, nrhs, s);
        else launch_tmpl_t<df, false>(a, t, nrhs, s);
    } else if (prec == 1) {
        if (from_tod) launch_tmpl_t<double, true>(a, t, nrhs, s);
        else launch_tmpl_t<double, false>(a, t, nrhs, s);
    } else {
        if (from_tod) launch_tmpl_t<float, true>(a, t, nrhs, s);
        else launch_tmpl_t<float, false>(a, t, nrhs, s);
    }
}

}  // namespace mm
