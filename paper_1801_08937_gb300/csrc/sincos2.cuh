// Pointing weights cos 2psi, sin 2psi in float64 from a table.
//
// The float64 pipe of the GB300 runs about two operations per clock per SM, and
// the general sincos spends some fifty there.  Here the angle is reduced to a
// table node plus a remainder |r| <= pi / TRIG_N in two exact products and
//   cos(a + r) = C + (-S sin r - C (1 - cos r)),  sin(a + r) = S + (C sin r - S (1 - cos r)),
// sin r = r - r^3/6 + ..., 1 - cos r = r^2/2 - r^4/24 + ...  The nodes carry a
// float32 tail, so the error is half an ulp from the last sum plus 4e-17 (the
// cubic term, at most 7.6e-11, is formed in float32).  Twelve operations on
// the float64 pipe per sample.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "fconv.cuh"

namespace mm {

constexpr int TRIG_N = 4096;
// 2 pi / TRIG_N as a 33-bit head (its products with node numbers are exact) and a tail
constexpr double TRIG_STEP_HI = 0x1.921fb544p-10;
constexpr double TRIG_STEP_LO = 0x1.0b4611a626331p-44;

// nodes [TRIG_N] (cos, sin), then tails float2 [TRIG_N]
struct TrigTable {
    const double2* node;
    const float2* tail;
};

__device__ __forceinline__ void sincos_2psi(float psi, const TrigTable& t, double& c, double& s) {
    const float a = 2.0f * psi;
    if (!(fabsf(a) < 256.0f)) {   // far angles, infinities, NaN
        sincos(2.0 * (double)psi, &s, &c);
        return;
    }
    const float m = fmaf(a, (float)(TRIG_N / 6.283185307179586477), 12582912.0f);   // nearest node, in the low bits
    const int n = __float_as_int(m) - 0x4B400000;
    const double nd = __hiloint2double(0x43380000 + (n >> 31), n) - 6755399441055744.0;   // n as float64
    double r = fma(-nd, TRIG_STEP_HI, f2d_exact(a));
    r = fma(-nd, TRIG_STEP_LO, r);
    const double2 cs = __ldg(t.node + (n & (TRIG_N - 1)));
    const float2 lo = __ldg(t.tail + (n & (TRIG_N - 1)));
    const float rf = d2f_trunc(r), r2 = rf * rf;
    const double sr = r - f2d_exact(rf * r2 * fmaf(r2, -1.0f / 120.0f, 1.0f / 6.0f));
    const double q = fma(0.5 * r, r, -f2d_exact(r2 * r2 * (1.0f / 24.0f)));
    c = cs.x + fma(-cs.y, sr, fma(-cs.x, q, f2d_exact(lo.x)));
    s = cs.y + fma(cs.x, sr, fma(-cs.y, q, f2d_exact(lo.y)));
}

}  // namespace mm
