// Register arithmetic of the own FFT passes (kp_fft.cu, kp_fft2.cu): small DFTs, twiddles and the
// image band of an oversampled axis.
#pragma once

#include <cuda_runtime.h>

#include <cmath>
#include <vector>

namespace kp {

// An axis for the passes of run-time length (kp_fft2.cu).
constexpr int F2_MAXST = 8;       // radix stages at most
struct F2Axis {
    int N, nst;                   // at least two stages
    int r[F2_MAXST];              // radices in the order applied
    unsigned mg[F2_MAXST];        // 2^32 / m + 1 for the stage's m (bf / m by a high product)
    const float2* tw;             // e^{-2 pi i m / N}, then the first radix's table when it is summed directly
};
// Radices of N into ax (not tw); false if N is not handled.
bool fft_axis_factor(int N, F2Axis& ax);
// Points of the table that the directly summed first radix needs beside the N roots: w_R^(q t), q = 1 ..
// (R - 1) / 2 by rows, t = 0 .. (R - 1) / 2; 0 for a compiled radix.
__host__ __device__ inline int fft_axis_extra(const F2Axis& ax) {
    const int h = (ax.r[0] - 1) / 2;
    return ax.r[0] > 19 ? h * (h + 1) : 0;
}
// The axis's table (float64, rounded once) appended to h; ax.tw is to point at it on the device.
void fft_axis_table(const F2Axis& ax, std::vector<float2>& h);

struct FfConst {                 // float64 on the host, rounded once
    float s3, c51, s51, c52, s52;   // sqrt(3)/2, cos and sin of 2 pi/5 and of 4 pi/5
    float2 w16[10];                 // (cos, sin) of 2 pi j / 16, j = 0..9 (radix-16 and radix-8 twiddles)
};

inline FfConst ff_const() {
    FfConst k;
    k.s3 = (float)(std::sqrt(3.0) / 2.0);
    k.c51 = (float)std::cos(2.0 * M_PI / 5.0);
    k.s51 = (float)std::sin(2.0 * M_PI / 5.0);
    k.c52 = (float)std::cos(4.0 * M_PI / 5.0);
    k.s52 = (float)std::sin(4.0 * M_PI / 5.0);
    for (int j = 0; j < 10; ++j)
        k.w16[j] = make_float2((float)std::cos(2.0 * M_PI * j / 16.0), (float)std::sin(2.0 * M_PI * j / 16.0));
    return k;
}

// The image samples a first forward pass forms itself (coil multiply and apodisation, the
// NUFFT's pre-step fused into the FFT): x, the maps (null: unit maps) and 1/Phi per axis.
struct PreSrc {
    const float2* x;
    const void* maps;
    const float* apod;
};

__device__ __forceinline__ bool in_band(int i, int n, int g) { return i < n - n / 2 || i >= g - n / 2; }
// pixel index of grid index i (i in the band)
__device__ __forceinline__ int pix_index(int i, int n, int g) { return i < n - n / 2 ? i + n / 2 : i - g + n / 2; }
__device__ __forceinline__ int band_index(int bi, int n, int g) { return bi < n - n / 2 ? bi : bi + (g - n); }

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
// a * (-i s) for the forward sign (s = +1) or a * (+i) for the inverse (s = -1): (s a.y, -s a.x)
__device__ __forceinline__ float2 cmul_mi(float2 a, float s) { return make_float2(s * a.y, -s * a.x); }

// a e^{-s 2 pi i j / 16} for cs = (cos, sin)(2 pi j / 16)
__device__ __forceinline__ float2 cmul_w(float2 a, float2 cs, float s) {
    const float wy = -s * cs.y;
    return make_float2(a.x * cs.x - a.y * wy, a.x * wy + a.y * cs.x);
}

template <int R>
__device__ __forceinline__ void small_dft(float2* v, float s, const FfConst& k);

// 4-point DFT of (a, b, c, d) in place, outputs in natural order
__device__ __forceinline__ void dft4(float2& a, float2& b, float2& c, float2& d, float s) {
    const float2 t0 = cadd(a, c), t1 = csub(a, c), t2 = cadd(b, d), t3 = cmul_mi(csub(b, d), s);
    a = cadd(t0, t2);
    c = csub(t0, t2);
    b = cadd(t1, t3);
    d = csub(t1, t3);
}

// One R-point DFT of v[0..R-1] in place, sign s = +1 forward (omega = e^{-2 pi i / R}), -1 inverse.
// R = 16 and 8 run as 4 x 4 and 4 x 2 in registers: with q = 4 q1 + q2 (resp. 2 q1 + q2) and
// k = k1 + 4 k2, X[k] = sum_q2 w_R^(q2 k1) w^(q2 k2) [sum_q1 v[.] w_4^(q1 k1)].
template <int R>
__device__ __forceinline__ void small_dft(float2* v, float s, const FfConst& k) {
    static_assert(R == 2 || R == 3 || R == 4 || R == 5 || R == 8 || R == 16, "basic radix");
    if (R == 16) {
        float2 y[4][4];
#pragma unroll
        for (int q2 = 0; q2 < 4; ++q2) {
            float2 a = v[q2], b = v[4 + q2], c = v[8 + q2], d = v[12 + q2];
            dft4(a, b, c, d, s);
            y[q2][0] = a;
            y[q2][1] = b;
            y[q2][2] = c;
            y[q2][3] = d;
        }
#pragma unroll
        for (int q2 = 1; q2 < 4; ++q2)
#pragma unroll
            for (int k1 = 1; k1 < 4; ++k1) y[q2][k1] = cmul_w(y[q2][k1], k.w16[q2 * k1], s);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            float2 a = y[0][k1], b = y[1][k1], c = y[2][k1], d = y[3][k1];
            dft4(a, b, c, d, s);
            v[k1] = a;
            v[k1 + 4] = b;
            v[k1 + 8] = c;
            v[k1 + 12] = d;
        }
    } else if (R == 8) {
        float2 y0[4], y1[4];
        {
            float2 a = v[0], b = v[2], c = v[4], d = v[6];
            dft4(a, b, c, d, s);
            y0[0] = a; y0[1] = b; y0[2] = c; y0[3] = d;
        }
        {
            float2 a = v[1], b = v[3], c = v[5], d = v[7];
            dft4(a, b, c, d, s);
            y1[0] = a; y1[1] = b; y1[2] = c; y1[3] = d;
        }
#pragma unroll
        for (int k1 = 1; k1 < 4; ++k1) y1[k1] = cmul_w(y1[k1], k.w16[2 * k1], s);
#pragma unroll
        for (int k1 = 0; k1 < 4; ++k1) {
            v[k1] = cadd(y0[k1], y1[k1]);
            v[k1 + 4] = csub(y0[k1], y1[k1]);
        }
    } else if (R == 2) {
        const float2 a = v[0], b = v[1];
        v[0] = cadd(a, b);
        v[1] = csub(a, b);
    } else if (R == 4) {
        const float2 t0 = cadd(v[0], v[2]), t1 = csub(v[0], v[2]);
        const float2 t2 = cadd(v[1], v[3]), t3 = cmul_mi(csub(v[1], v[3]), s);
        v[0] = cadd(t0, t2);
        v[2] = csub(t0, t2);
        v[1] = cadd(t1, t3);
        v[3] = csub(t1, t3);
    } else if (R == 3) {
        // y1,2 = a0 - (a1 + a2)/2 -/+ i s sqrt(3)/2 (a1 - a2)
        const float2 sm = cadd(v[1], v[2]), d = cmul_mi(csub(v[1], v[2]), s * k.s3);
        const float2 m = make_float2(v[0].x - 0.5f * sm.x, v[0].y - 0.5f * sm.y);
        v[0] = cadd(v[0], sm);
        v[1] = cadd(m, d);
        v[2] = csub(m, d);
    } else {
        // R == 5: t1 = a1 + a4, t2 = a2 + a3, t3 = a1 - a4, t4 = a2 - a3;
        // y1,4 = a0 + c1 t1 + c2 t2 -/+ i (s1 t3 + s2 t4), y2,3 = a0 + c2 t1 + c1 t2 -/+ i (s2 t3 - s1 t4)
        const float2 a0 = v[0];
        const float2 t1 = cadd(v[1], v[4]), t2 = cadd(v[2], v[3]), t3 = csub(v[1], v[4]), t4 = csub(v[2], v[3]);
        const float2 p1 = make_float2(a0.x + k.c51 * t1.x + k.c52 * t2.x, a0.y + k.c51 * t1.y + k.c52 * t2.y);
        const float2 p2 = make_float2(a0.x + k.c52 * t1.x + k.c51 * t2.x, a0.y + k.c52 * t1.y + k.c51 * t2.y);
        const float2 q1 = cmul_mi(make_float2(k.s51 * t3.x + k.s52 * t4.x, k.s51 * t3.y + k.s52 * t4.y), s);
        const float2 q2 = cmul_mi(make_float2(k.s52 * t3.x - k.s51 * t4.x, k.s52 * t3.y - k.s51 * t4.y), s);
        v[0] = make_float2(a0.x + t1.x + t2.x, a0.y + t1.y + t2.y);
        v[1] = cadd(p1, q1);
        v[4] = csub(p1, q1);
        v[2] = cadd(p2, q2);
        v[3] = csub(p2, q2);
    }
}

// a * w for the twiddle w = tw[e] = e^{-2 pi i e / N}, conjugated for the inverse (s = -1)
__device__ __forceinline__ float2 twiddle(float2 x, float2 w, float s) {
    w.y *= s;
    return make_float2(x.x * w.x - x.y * w.y, x.x * w.y + x.y * w.x);
}

}  // namespace kp
