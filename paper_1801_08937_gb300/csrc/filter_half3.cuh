// float32 A x and P^T W d with a whole block as one complex transform of
// M = R0 R1 9 points (half the block's padded length) in three passes.
//
// What bounds it: instruction issue and latency (two CTAs of nine warps per SM,
// 96 registers), not DRAM.  Against the four passes of radix 9, 16, 16, 4 at 64
// registers and 512 threads that it replaces, three passes keep up to 32 points
// of a transform in one thread's registers, so the block crosses shared memory
// five times instead of eight (shared-memory wavefronts 12.6 M -> 10.2 M, with
// the pointing's own now among them, warp instructions 69.4 M -> 54.0 M per
// 1.68e7 samples).  The gather was half the kernel's time while every row waited
// for its pointing and then for its map entries (30 K of 60 K cycles a block);
// the pointing now streams through shared memory by bulk copies ahead of its use
// and the block's pixel window is staged there (14 K cycles).  Measured on one
// GB300, 1.34e8 samples in blocks of 16384, lambda 2048 (M = 9216): 0.800 -> 0.634
// ms a product; blocks of 16384, lambda 512, 3.4e7 samples: 0.327 (overlap-save of
// 4096 points) -> 0.185 ms.
//
// Layout.  Point p = d0 (9 R1) + d1 9 + d2 sits at element d0 P + d1 9 + d2,
// P = 9 R1 + 9.  P and 9 are odd modulo 16, so every pass is free of bank
// conflicts: pass 1 walks d1, d2 over the lanes, pass 2 walks d0 (stride P; a
// warp then shares d2 and with it all its twiddles), pass 3 walks d1 (stride 9).
// Before the scatter the real samples are laid out again with one spare element
// in 16 (sidx), where eight consecutive samples a lane are free of conflicts.
//
// Spectrum step: the last pass (radix 9) of butterfly (d0, d1) holds the
// frequencies kc + R0 R1 q, kc = d0 + R0 d1, and the mirror images M - k sit in
// butterfly (R0 - d0, R1 - 1 - d1) at outputs 8 - q ((0, R1 - d1) for d0 = 0).
// A thread takes such a pair, so neither needs a table of pairs.
#pragma once
#include "filter_impl.cuh"

namespace mm {

template <int R0_, int R1_> struct H3 {
    static constexpr int R0 = R0_, R1 = R1_, R2 = 9;
    static constexpr int SR = R1 * R2;           // stride of pass 1
    static constexpr int M = R0 * SR;
    static constexpr int P = SR + 9;             // pitch of a row of SR points
    static constexpr int NB = R0 * R1;           // butterflies of the last pass
    static constexpr int NI = NB / 2 + 1;        // coefficient items (the last holds the second self-paired butterfly)
    static constexpr int RA = R0 / 4;            // pass-1 twiddles W^(j q): q = qa + RA qb
    static constexpr int NT = SR;
    static constexpr int PTS = (R0 * P > M + M / 16) ? R0 * P : M + M / 16;
    // gather: chunks of G rows of pointing, NS of them in flight, at the end of the buffer; the map entries of
    // the block's pixels (up to WIN) before them
    static constexpr int G = 4, NS = M > 2304 ? 3 : 2;
    static constexpr int CH = 2 * G * SR;                       // samples of a chunk
    static constexpr int CHB = 2 * (CH + 4) * 4;                // bytes of a chunk: pix and psi, one spare group each
    static constexpr int WIN0 = M > 4608 ? 0 : (M > 2304 ? 1536 : 512);
    static constexpr int BUF = PTS * 8 > NS * CHB + WIN0 * 16 ? PTS * 8 : NS * CHB + WIN0 * 16;   // bytes
    static constexpr int WIN = (BUF - NS * CHB) / 16;
    static constexpr int MINB = M > 4608 ? 2 : (M > 2304 ? 4 : 5);   // CTAs a SM holds (registers)
    static_assert((size_t)(CH + 8) * 4 <= POINTING_SPARE, "a chunk that starts inside the timeline stays inside the arrays");
};

// ---- bulk copies of the pointing to shared memory, completion on an mbarrier ----
__device__ __forceinline__ void h3_bar_init(uint32_t bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
// Chunk c of a block's pointing (base 16-byte aligned).  The arrays have spare
// room behind the last sample (POINTING_SPARE), so a chunk needs no clipping.
template <typename H>
__device__ __forceinline__ void h3_fetch(const int32_t* pix, const float* psi, int c, uint32_t dst, uint32_t bar) {
    constexpr uint32_t B = H::CHB / 2;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "n"(2 * B) : "memory");
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
                 "l"(pix + H::CH * c), "n"(B), "r"(bar)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cta.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst + B),
                 "l"(psi + H::CH * c), "n"(B), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ bool h3_bar_try(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return done != 0;
}
// false if the copy has not landed after `limit` nanoseconds
__device__ __forceinline__ bool h3_bar_wait(uint32_t bar, uint32_t parity, unsigned limit) {
    if (h3_bar_try(bar, parity)) return true;
    unsigned long long t0, t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
    for (;;) {
        if (h3_bar_try(bar, parity)) return true;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        if (t - t0 > limit) return false;
    }
}

// One pass over R elements in registers; DIT: twiddles first, then the DFT.
template <int R, bool DIT, typename W>
__device__ __forceinline__ void h3_butterfly(C2<float> (&a)[R], bool twiddle, W w) {
    if (DIT) {
        if (twiddle) {
#pragma unroll
            for (int q = 1; q < R; ++q) a[q] = cmul(a[q], w(q));
        }
        Dft<float, R>::run(a);
    } else {
        Dft<float, R>::run(a);
        if (twiddle) {
#pragma unroll
            for (int q = 1; q < R; ++q) a[q] = cmul(a[q], w(q));
        }
    }
}

// Twiddles of pass 1, W_M^(j q) = A[q mod RA] B[q / RA], from the rows of a table [RA + 2][SR].
template <typename H>
struct Pass1Twiddle {
    C2<float> A[H::RA], B[4];
    __device__ __forceinline__ Pass1Twiddle(const C2<float>* __restrict__ t, int j) {
#pragma unroll
        for (int q = 1; q < H::RA; ++q) A[q] = ldtw(t, (q - 1) * H::SR + j);
#pragma unroll
        for (int q = 1; q < 4; ++q) B[q] = ldtw(t, (H::RA - 2 + q) * H::SR + j);
    }
    __device__ __forceinline__ C2<float> operator()(int q) const {
        const int a = q % H::RA, b = q / H::RA;
        return b == 0 ? A[a] : (a == 0 ? B[b] : cmul(A[a], B[b]));
    }
};

template <typename H, bool DIT>
__device__ __forceinline__ void h3_pass2(C2<float>* s, const C2<float>* __restrict__ tw) {
#pragma unroll 1
    for (int bf = threadIdx.x; bf < H::R0 * 9; bf += H::NT) {
        const int g = bf % H::R0, j = bf / H::R0;
        C2<float>* b = s + g * H::P + j;
        C2<float> a[H::R1];
#pragma unroll
        for (int r = 0; r < H::R1; ++r) a[r] = b[9 * r];
        const C2<float>* w = tw + j * H::R1;
        h3_butterfly<H::R1, DIT>(a, j > 0, [&](int q) { return ldtw(w, q); });
#pragma unroll
        for (int r = 0; r < H::R1; ++r) b[9 * r] = a[r];
    }
}

__device__ __forceinline__ float4 h3_coef(const float4* __restrict__ c, int e) { return __ldg(c + e); }

template <typename H>
__device__ __forceinline__ void h3_spectrum(C2<float>* s, const float4* __restrict__ coef) {
    constexpr int R0 = H::R0, R1 = H::R1;
#pragma unroll 1
    for (int t = threadIdx.x; t < H::NB / 2; t += H::NT) {
        int g = t / R1, r = t % R1, g2 = R0 - g, r2 = R1 - 1 - r;
        if (g == 0) {
            if (r < R1 / 2) {            // d0 = R0 / 2 pairs within itself
                g = g2 = R0 / 2;
            } else {                     // d0 = 0: (0, r) with (0, R1 - r); (0, 0) and (0, R1 / 2) pair with themselves
                r -= R1 / 2;
                g2 = 0;
                r2 = r == 0 ? R1 / 2 : R1 - r;
            }
        }
        C2<float>*b0 = s + g * H::P + 9 * r, *b1 = s + g2 * H::P + 9 * r2;
        C2<float> x[9], y[9];
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            x[q] = b0[q];
            y[q] = b1[q];
        }
        Dft<float, 9>::run(x);
        Dft<float, 9>::run(y);
        C2<float> xo[9], yo[9];
        if (t != R1 / 2) {
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const float4 c = h3_coef(coef, q * H::NI + t);
                const C2<float> A = x[q], B = y[8 - q];
                xo[q] = C2<float>{c.x * A.x + c.z * B.y, -(c.x * A.y + c.z * B.x)};
                yo[8 - q] = C2<float>{c.y * B.x + c.z * A.y, -(c.y * B.y + c.z * A.x)};
            }
        } else {
#pragma unroll
            for (int q = 0; q < 9; ++q) {
                const float4 c = h3_coef(coef, q * H::NI + t), d = h3_coef(coef, q * H::NI + H::NB / 2);
                const C2<float> A = x[q], B = x[(9 - q) % 9], C = y[q], D = y[8 - q];
                xo[q] = C2<float>{c.x * A.x + c.z * B.y, -(c.x * A.y + c.z * B.x)};
                yo[q] = C2<float>{d.x * C.x + d.z * D.y, -(d.x * C.y + d.z * D.x)};
            }
        }
        Dft<float, 9>::run(xo);
        Dft<float, 9>::run(yo);
#pragma unroll
        for (int q = 0; q < 9; ++q) {
            b0[q] = xo[q];
            b1[q] = yo[q];
        }
    }
}

template <typename H, bool FROM_TOD, bool EVEN>
__global__ void __launch_bounds__(H::NT, H::MINB) k_filter_half3(const FilterArgs a) {
    extern __shared__ __align__(16) unsigned char smraw[];
    C2<float>* s = reinterpret_cast<C2<float>*>(smraw);
    const Seg S = a.segs[blockIdx.x];
    if (!seg_active<float>(a, S)) return;
    constexpr int R0 = H::R0, SR = H::SR;
    const int j = threadIdx.x;
    if (j == 0 && blockIdx.x + a.ahead < gridDim.x) {
        // the pointing of the block that follows on this SM, from DRAM to L2
        const Seg N = a.segs[blockIdx.x + a.ahead];
        const int64_t n0 = N.out0 & ~3ll;
        const uint32_t nb = (uint32_t)(N.out0 + N.n_out - n0) * 4u & ~15u;
        if (nb > 0) {
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.pix + n0), "r"(nb) : "memory");
            asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a.psi + n0), "r"(nb) : "memory");
        }
    }
    const C2<float>* t1 = reinterpret_cast<const C2<float>*>(a.twp);
    const C2<float>* t2 = reinterpret_cast<const C2<float>*>(a.tw);
    {
        C2<float> y[R0];
        if constexpr (FROM_TOD) {
            const int64_t o = (int64_t)S.rhs * a.n_samples + S.out0;
#pragma unroll
            for (int r = 0; r < R0; ++r) {
                const int i0 = 2 * (j + SR * r);
                float v[2];
#pragma unroll
                for (int e = 0; e < 2; ++e)
                    v[e] = i0 + e >= S.n_out ? 0.0f
                           : a.tod_is_float ? __ldg(reinterpret_cast<const float*>(a.src) + o + i0 + e)
                                            : (float)__ldg(reinterpret_cast<const double*>(a.src) + o + i0 + e);
                y[r] = C2<float>{v[0], v[1]};
            }
        } else {
            // The pointing streams through NS chunk buffers (in flight while earlier rows are pointed), and the
            // map entries of the block's pixel window are staged once: a row then waits for shared memory only.
            // A wider window (a block that wraps around the patch, a large patch) is read from L2.
            constexpr int G = H::G, NS = H::NS, NCH = R0 / G;
            const uint32_t sb = (uint32_t)__cvta_generic_to_shared(smraw), cb = sb + H::BUF - NS * H::CHB;
            const float4* map = reinterpret_cast<const float4*>(a.src) + (int64_t)S.rhs * a.n_pix;
            const int64_t base = S.out0 & ~3ll;
            const int d = (int)(S.out0 - base), nch = (S.n_out + H::CH - 1) / H::CH;
            __shared__ uint64_t full[NS];
            const uint32_t fb = (uint32_t)__cvta_generic_to_shared(full);
            if (j == 0) {
#pragma unroll
                for (int c = 0; c < NS; ++c) h3_bar_init(fb + 8 * c);
                asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
#pragma unroll
                for (int c = 0; c < NS; ++c)
                    if (c < nch) h3_fetch<H>(a.pix + base, a.psi + base, c, cb + c * H::CHB, fb + 8 * c);
            }
            const bool staged = S.nwin <= H::WIN;
            if (staged)
                for (int i = j; i < S.nwin; i += H::NT)
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sb + 16u * i), "l"(map + S.win0 + i) : "memory");
            asm volatile("cp.async.wait_all;" ::: "memory");
            bool ok = a.wait_ns != 0;   // a limit of zero gives up without a look
            int issued = min(NS, nch);   // thread 0: chunks asked for
            auto rows = [&](auto entry) {
#pragma unroll
                for (int c = 0; c < NCH; ++c) {
                    int32_t* lc = reinterpret_cast<int32_t*>(smraw + H::BUF - (NS - c % NS) * H::CHB) + d;
                    __syncthreads();   // everyone is done with chunk c - 1 (and has staged its map entries)
                    // (behind a wait that gave up the buffer's barrier still counts its last copy: no new one then)
                    if (c > 0 && c + NS - 1 < nch && j == 0 && ok) {
                        h3_fetch<H>(a.pix + base, a.psi + base, c + NS - 1, cb + ((c - 1) % NS) * H::CHB,
                                    fb + 8 * ((c - 1) % NS));
                        issued = c + NS;
                    }
                    if (c < nch) {
                        ok = ok && h3_bar_wait(fb + 8 * (c % NS), (c / NS) & 1, a.wait_ns);
                        if (S.n_out < (c + 1) * H::CH) {   // the end of the block: what follows is flagged
                            if (ok)   // (not while the copy may still land on it)
                                for (int k = S.n_out - c * H::CH + j; k < H::CH; k += H::NT) lc[k] = -1;
                            ok = __syncthreads_and(ok);
                        }
                    }
                    if (c < nch && ok) {
                        const int32_t* lp = lc + 2 * j;
                        const float* lf = reinterpret_cast<const float*>(lp + H::CH + 4);
#pragma unroll
                        for (int e = 0; e < G; ++e) {
                            int2 p;
                            float2 f;
                            if constexpr (EVEN) {
                                p = *reinterpret_cast<const int2*>(lp + 2 * SR * e);
                                f = *reinterpret_cast<const float2*>(lf + 2 * SR * e);
                            } else {
                                p = make_int2(lp[2 * SR * e], lp[2 * SR * e + 1]);
                                f = make_float2(lf[2 * SR * e], lf[2 * SR * e + 1]);
                            }
                            y[G * c + e] = C2<float>{pointed_value(p.x, f.x, entry(p.x)),
                                                     pointed_value(p.y, f.y, entry(p.y))};
                        }
                    } else {   // zero padding (or a copy that never came)
#pragma unroll
                        for (int e = 0; e < G; ++e) y[G * c + e] = C2<float>{0.0f, 0.0f};
                    }
                }
            };
            if (staged) rows([&](int p) { return reinterpret_cast<const float4*>(smraw)[max(p - S.win0, 0)]; });
            else rows([&](int p) { return __ldg(map + max(p, 0)); });
            if (!ok) {
                *reinterpret_cast<volatile int*>(a.fault) = 1;
                if (j == 0)   // let the copies in flight land before the buffer is reused
                    for (int c = max(0, issued - NS); c < issued; ++c) h3_bar_wait(fb + 8 * (c % NS), (c / NS) & 1, WAIT_NS);
            }
            __syncthreads();   // the buffer becomes the transform's
        }
        h3_butterfly<R0, false>(y, true, Pass1Twiddle<H>(t1, j));
#pragma unroll
        for (int q = 0; q < R0; ++q) s[q * H::P + j] = y[q];
    }
    __syncthreads();
    h3_pass2<H, false>(s, t2);
    __syncthreads();
    h3_spectrum<H>(s, reinterpret_cast<const float4*>(a.Hi) + (int64_t)S.band * 9 * H::NI);
    __syncthreads();
    h3_pass2<H, true>(s, t2);
    __syncthreads();
    {
        C2<float> y[R0];
#pragma unroll
        for (int q = 0; q < R0; ++q) y[q] = s[q * H::P + j];
        h3_butterfly<R0, true>(y, true, Pass1Twiddle<H>(t1, j));
        __syncthreads();   // every row is read: the samples take the scatter's layout
#pragma unroll
        for (int r = 0; r < R0; ++r)
            if (2 * (j + SR * r) < S.n_out) s[sidx(j + SR * r)] = y[r];
    }
    __syncthreads();
    half_scatter_f32<H::NT>(a, S, s, H::M);
}

}  // namespace mm
