// Own 2D FFT of a plan's oversampled grids with the NUFFT's neighbouring steps fused in, used in
// place of cuFFT for 2D plans whose grid lengths have prime factors up to F2_MAXP (Sec. 6's
// oversampled FFT, unnormalised like cuFFT).
//
//   forward:  row pass     x -> coil multiply, apodise, pad, FFT along x; only the n0 image rows
//             column pass  FFT along y in place; reads only the image rows
//   adjoint:  column pass  inverse FFT along y of the spread grid into the work grid, writing
//                          only the image rows; the spread grid is left zero for the next spread
//             row pass     inverse FFT along x of one image row of every coil, crop, conj(s_c)
//                          combine, apodise, and the primal step of Sec. 4.1 / 4.2 or the norm of
//                          the power method
//
// A CTA takes LN lines (rows of one or several coils, or neighbouring columns), the line index
// fastest over its threads (in shared memory the lines lie side by side, so no bank conflicts; in
// global memory 8 lines x 4 points of a warp are whole 32-byte sectors).  Stockham stages: the
// first runs on the values loaded from global memory (all of a butterfly's loads in flight), the
// last stores to global memory, the ones between go through two shared-memory buffers.  The
// length is a run-time value: radices up to 10 are compiled butterflies, chosen for the fewest
// stages; one prime above 5 per axis goes first (above 19 summed directly, in pairs of outputs).
// Larger radices (two stages of 16 x 20 for 320 points) were no faster: fewer barriers, but long
// straight code run once by few threads.
//
// 3D grids whose lengths have no compiled pass in kp_fft.cu run the same stages (k_fftg_pass).
//
// These grids live in L2 and a pass is bound by its latency (launch, loads, one or two barriers,
// stores), not by bytes: what pays is fewer kernels, fewer dependent steps and every CTA resident
// in one wave (64 registers, four CTAs per SM).  One application of A^H P A
// (power iteration, against cuFFT with separate pre-step, combine and norm kernels): spiral 256^2 x
// 12 coils 84 against 97 us, radial 217 x 186 x 7 (272 x 234 grid) 60 against 72 us, radial 320^2 x 32
// 307 against 365 us.
#include "kp_fft_radix.cuh"
#include "kp_internal.cuh"

#include <algorithm>
#include <cstdlib>
#include <new>
#include <string>
#include <vector>

namespace kp {

constexpr int F2_MAXP = 127;      // largest prime factor summed directly
constexpr int F2_T = 256;         // threads per CTA at most
constexpr int F2_SMEM = 200 * 1024;

struct Fft2Plan {
    F2Axis ax[2];                 // y, x
    float2* d_tw = nullptr;
    FfConst k;
};

extern __shared__ __align__(16) float2 f2sm[];

// Factors (P, Q) of a radix done as a two-factor DFT in registers; P = 0 for the others.
constexpr int f2_split(int R) { return R == 6 || R == 10 ? 2 : R == 9 ? 3 : 0; }

// R-point DFT of v in place; w_R^e is tw[e nb], nb = N / R.
template <int R>
__device__ __forceinline__ void f2_dft(float2* v, float s, const FfConst& k, const float2* tw, int nb) {
    constexpr int P = f2_split(R);
    if constexpr (R == 7 || R == 11 || R == 13 || R == 17 || R == 19) {
        // odd prime, folded: with a_q = v_q + v_{R-q}, b_q = v_q - v_{R-q},
        // X_t, X_{R-t} = v_0 + sum_q a_q cos(2 pi q t / R) -/+ i s sum_q b_q sin(2 pi q t / R), summed
        // from the high frequencies (q = H) to the low ones and v_0 last: gridded k-space is largest there,
        // and each addition rounds at the size of what has been summed so far
        constexpr int H = (R - 1) / 2;
        float2 a[H], b[H], o[R];
        float2 x0 = make_float2(0.f, 0.f);
#pragma unroll
        for (int q = H - 1; q >= 0; --q) {
            a[q] = cadd(v[q + 1], v[R - 1 - q]);
            b[q] = csub(v[q + 1], v[R - 1 - q]);
            x0 = cadd(x0, a[q]);
        }
        o[0] = cadd(x0, v[0]);
#pragma unroll
        for (int t = 1; t <= H; ++t) {
            float2 e = make_float2(0.f, 0.f), d = e;
#pragma unroll
            for (int q = H; q >= 1; --q) {
                const float2 w = tw[(q * t % R) * nb];    // (cos, -sin)
                e.x = fmaf(a[q - 1].x, w.x, e.x);
                e.y = fmaf(a[q - 1].y, w.x, e.y);
                d.x = fmaf(b[q - 1].x, w.y, d.x);
                d.y = fmaf(b[q - 1].y, w.y, d.y);
            }
            // X_t = e + i s d, X_{R-t} = e - i s d
            e = cadd(e, v[0]);
            o[t] = make_float2(e.x - s * d.y, e.y + s * d.x);
            o[R - t] = make_float2(e.x + s * d.y, e.y - s * d.x);
        }
#pragma unroll
        for (int t = 0; t < R; ++t) v[t] = o[t];
    } else if constexpr (P == 0) {
        small_dft<R>(v, s, k);
    } else {
        constexpr int Q = R / P;
        float2 y[Q][P];
#pragma unroll
        for (int q2 = 0; q2 < Q; ++q2) {
#pragma unroll
            for (int q1 = 0; q1 < P; ++q1) y[q2][q1] = v[Q * q1 + q2];
            small_dft<P>(y[q2], s, k);
        }
#pragma unroll
        for (int q2 = 1; q2 < Q; ++q2)
#pragma unroll
            for (int k1 = 1; k1 < P; ++k1) y[q2][k1] = twiddle(y[q2][k1], tw[q2 * k1 * nb], s);
#pragma unroll
        for (int k1 = 0; k1 < P; ++k1) {
            float2 b[Q];
#pragma unroll
            for (int q2 = 0; q2 < Q; ++q2) b[q2] = y[q2][k1];
            small_dft<Q>(b, s, k);
#pragma unroll
            for (int k2 = 0; k2 < Q; ++k2) v[k1 + P * k2] = b[k2];
        }
    }
}

// Stockham stage of radix R after L points: butterfly (j, kk), j < m = N / (L R), kk < L, takes
// elements kk N / L + j + q m, multiplies input q by w^(q kk m) and puts output t of its R-point DFT
// at (kk + L t) m + j.  Element n of line l lies at n P + l.  A thread keeps one line l (the block
// size is a multiple of LN) and takes every (threads / LN)-th butterfly of it.

// First stage (L = 1): inputs from ld(n), outputs to the buffer at ib.
template <int R, int LN, int P, typename LD>
__device__ __forceinline__ void f2_first(LD ld, int ib, const float2* tw, int N, float s, const FfConst& k) {
    const int nb = N / R, l = threadIdx.x % LN;
    for (int j = threadIdx.x / LN; j < nb; j += blockDim.x / LN) {
        float2 v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = ld(j + q * nb);
        f2_dft<R>(v, s, k, tw, nb);
#pragma unroll
        for (int t = 0; t < R; ++t) f2sm[ib + (t * nb + j) * P + l] = v[t];
    }
}

// Stage between two buffers.
template <int R, int LN, int P>
__device__ __forceinline__ void f2_stage(int ia, int ib, const float2* tw, int N, int L, unsigned mg, float s,
                                         const FfConst& k) {
    const int nb = N / R, m = nb / L, NL = N / L, l = threadIdx.x % LN;
    for (int bf = threadIdx.x / LN; bf < nb; bf += blockDim.x / LN) {
        const int kk = m == 1 ? bf : (int)__umulhi((unsigned)bf, mg), j = bf - kk * m, e = kk * m;
        const float2* a = f2sm + ia + (kk * NL + j) * P + l;
        float2 v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = q > 0 ? twiddle(a[q * m * P], tw[q * e], s) : a[0];
        f2_dft<R>(v, s, k, tw, nb);
        float2* b = f2sm + ib + (e + j) * P + l;
#pragma unroll
        for (int t = 0; t < R; ++t) b[t * L * m * P] = v[t];
    }
}

// Last stage (m = 1): outputs to st(n, value).
template <int R, int LN, int P, typename ST>
__device__ __forceinline__ void f2_last(ST st, int ia, const float2* tw, int N, float s, const FfConst& k) {
    const int L = N / R, l = threadIdx.x % LN;
    for (int kk = threadIdx.x / LN; kk < L; kk += blockDim.x / LN) {
        const float2* a = f2sm + ia + kk * R * P + l;
        float2 v[R];
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = q > 0 ? twiddle(a[q * P], tw[q * kk], s) : a[0];
        f2_dft<R>(v, s, k, tw, L);
#pragma unroll
        for (int t = 0; t < R; ++t) st(kk + L * t, v[t]);
    }
}

// First stage for a prime radix without a compiled butterfly: the lines are copied to the buffer at
// ia, then each thread forms, for up to F2_TB values of t, the outputs t and R - t of a butterfly
// (folded as above) with the table w_R^(q t) that follows tw.  Bound by issue: per input pair and t one
// table load and four FMAs (one t per thread and table indices reduced mod R took 13 instead of 7).
// The sums run from q = H down to 1 in blocks of F2_QB, each added to the total, and the input of index
// 0 comes last: one running sum rounds H times at full size (relative error for R = 83: 1.2e-7 on white
// data and 1.6e-7 on data that decays like 1/k; this order 0.9e-7 and 0.6e-7).
constexpr int F2_TB = 4;
constexpr int F2_QB = 8;
template <int LN, int P, typename LD>
__device__ __forceinline__ void f2_first_prime(LD ld, int R, int ia, int ib, const float2* tw, int N, float s) {
    const int nb = N / R, H = (R - 1) / 2, l = threadIdx.x % LN, nq = (H + F2_TB) / F2_TB;
    for (int n = threadIdx.x / LN; n < N; n += blockDim.x / LN) f2sm[ia + n * P + l] = ld(n);
    __syncthreads();
    for (int o = threadIdx.x / LN; o < nq * nb; o += blockDim.x / LN) {
        const int t0 = o / nb, j = o - t0 * nb, st = nb * P;
        const float2 *a = f2sm + ia + j * P + l, *xq = a + H * st, *yq = a + (R - H) * st;
        const float2* w = tw + N + t0 + (H - 1) * (H + 1);
        float2 e[F2_TB], d[F2_TB];
        int to[F2_TB];                                       // t values past H repeat t = H
#pragma unroll
        for (int m = 0; m < F2_TB; ++m) {
            e[m] = d[m] = make_float2(0.f, 0.f);
            to[m] = min(t0 + m * nq, H) - t0;
        }
        for (int q = H; q > 0;) {
            const int q1 = max(q - F2_QB, 0);
            float2 be[F2_TB], bd[F2_TB];
#pragma unroll
            for (int m = 0; m < F2_TB; ++m) be[m] = bd[m] = make_float2(0.f, 0.f);
#pragma unroll 2
            for (; q > q1; --q, xq -= st, yq += st, w -= H + 1) {
                const float2 x = *xq, y = *yq, p = cadd(x, y), r = csub(x, y);
#pragma unroll
                for (int m = 0; m < F2_TB; ++m) {
                    const float2 c = w[to[m]];
                    be[m].x = fmaf(p.x, c.x, be[m].x);
                    be[m].y = fmaf(p.y, c.x, be[m].y);
                    bd[m].x = fmaf(r.x, c.y, bd[m].x);
                    bd[m].y = fmaf(r.y, c.y, bd[m].y);
                }
            }
#pragma unroll
            for (int m = 0; m < F2_TB; ++m) {
                e[m] = cadd(e[m], be[m]);
                d[m] = cadd(d[m], bd[m]);
            }
        }
#pragma unroll
        for (int m = 0; m < F2_TB; ++m) e[m] = cadd(e[m], a[0]);
#pragma unroll
        for (int m = 0; m < F2_TB; ++m) {
            const int t = t0 + m * nq;
            if (t > H) break;
            f2sm[ib + (t * nb + j) * P + l] = make_float2(e[m].x - s * d[m].y, e[m].y + s * d[m].x);
            if (t > 0) f2sm[ib + ((R - t) * nb + j) * P + l] = make_float2(e[m].x + s * d[m].y, e[m].y - s * d[m].x);
        }
    }
}

#define KP_F2_SMOOTH(X) X(2) X(3) X(4) X(5) X(6) X(8) X(9) X(10)
#define KP_F2_PRIMES(X) X(7) X(11) X(13) X(17) X(19)      // first stage only

// Every stage but the last, from ld into one of the buffers at 0 and ib; returns the one that holds
// the result.  tw: the CTA's copy of the roots of unity (complete after a barrier).
template <int LN, int P, typename LD>
__device__ __forceinline__ int f2_begin(const F2Axis& ax, LD ld, int ib, const float2* tw, float s, const FfConst& k) {
    const int N = ax.N;
    switch (ax.r[0]) {
#define KP_F2_CASE(r) case r: f2_first<r, LN, P>(ld, 0, tw, N, s, k); break;
        KP_F2_SMOOTH(KP_F2_CASE) KP_F2_PRIMES(KP_F2_CASE)
#undef KP_F2_CASE
        default: f2_first_prime<LN, P>(ld, ax.r[0], ib, 0, tw, N, s);
    }
    __syncthreads();
    int from = 0, to = ib, L = ax.r[0];
    for (int st = 1; st + 1 < ax.nst; ++st) {
        switch (ax.r[st]) {
#define KP_F2_CASE(r) case r: f2_stage<r, LN, P>(from, to, tw, N, L, ax.mg[st], s, k); break;
            KP_F2_SMOOTH(KP_F2_CASE)
#undef KP_F2_CASE
        }
        __syncthreads();
        L *= ax.r[st];
        const int t = from;
        from = to;
        to = t;
    }
    return from;
}

template <int LN, int P, typename ST>
__device__ __forceinline__ void f2_end(const F2Axis& ax, ST st, int from, const float2* tw, float s, const FfConst& k) {
    switch (ax.r[ax.nst - 1]) {
#define KP_F2_CASE(r) case r: f2_last<r, LN, P>(st, from, tw, ax.N, s, k); break;
        KP_F2_SMOOTH(KP_F2_CASE)
#undef KP_F2_CASE
    }
}

// Forward row pass: LN lines (image row, coil), coil fastest; coil c takes the image x + c xstride.
// PAIR: "coil" c is the pair (e, f) = pairs[c] of the preconditioner and its image s_e s_f^* (ones
// without maps).  iter (or null) is advanced and nrm (or null) shifted, nrm[0] = nrm[1], nrm[1] = 0, for
// the kernels that follow.
template <typename MT, int LN, bool PAIR>
__global__ void __launch_bounds__(F2_T, 4)
k_fft2_row_fwd(const float2* __restrict__ x, int64_t xstride, const int2* __restrict__ pairs, const MT* __restrict__ maps,
               const float* __restrict__ apod, Geom geo, F2Axis ax, FfConst k, float2* __restrict__ out,
               int* __restrict__ iter, double* __restrict__ nrm) {
    constexpr int P = LN;
    const int N = ax.N, n0 = geo.n[0], n1 = geo.n[1], g0 = geo.g[0];
    float2* tw = f2sm + 2 * N * P;
    const int nt = N + fft_axis_extra(ax);
    for (int i = threadIdx.x; i < nt; i += blockDim.x) tw[i] = ax.tw[i];
    pdl_begin();                                           // (the tables above are constant)
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        if (iter) *iter += 1;
        if (nrm) { nrm[0] = nrm[1]; nrm[1] = 0.0; }
    }
    const int line = blockIdx.x * LN + threadIdx.x % LN;
    const bool live = line < n0 * geo.C;
    const int iy = live ? line / geo.C : 0, c = live ? line - iy * geo.C : 0;
    const int ny = iy - n0 / 2;
    const float ay = PAIR ? 1.f : apod[iy];
    const float* ax1 = apod + n0;
    const float2* xr = x + (PAIR ? 0 : (size_t)c * xstride + (size_t)iy * n1);
    const int2 ef = PAIR && maps ? pairs[c] : make_int2(c, c);
    const MT* mr = maps ? maps + (size_t)ef.x * geo.N + (size_t)iy * n1 : nullptr;
    const MT* mf = PAIR && maps ? maps + (size_t)ef.y * geo.N + (size_t)iy * n1 : nullptr;
    __syncthreads();
    // loads without branches (points outside the band read the row's first pixel and drop it), so
    // that a butterfly's loads are all issued before the first is used
    const auto ld = [&](int n) {
        const bool in = live && in_band(n, n1, N) && KP_INB(3, pix_index(n, n1, N), n1);
        const int px = in ? pix_index(n, n1, N) : 0;
        if constexpr (PAIR) {
            const float2 e = maps ? ldc<MT>(mr, px) : make_float2(1.f, 0.f), f = maps ? ldc<MT>(mf, px) : make_float2(1.f, 0.f);
            return in ? cmulc(f, e) : make_float2(0.f, 0.f);
        }
        float2 v = xr[px];
        const float2 m = maps ? ldc<MT>(mr, px) : make_float2(1.f, 0.f);
        const float a = in ? ay * ax1[px] : 0.f;
        v.x *= a;
        v.y *= a;
        if (maps) v = cmul(m, v);
        return in ? v : make_float2(0.f, 0.f);
    };
    const int f = f2_begin<LN, P>(ax, ld, N * P, tw, 1.f, k);
    const int64_t base = (int64_t)c * geo.G + (int64_t)(ny < 0 ? ny + g0 : ny) * N;
    float2* o = out + base;
    f2_end<LN, P>(ax, [&](int n, float2 v) {
        if (live && KP_INB(2, base + n, (int64_t)geo.C * geo.G)) o[n] = v;
    }, f, tw, 1.f, k);
}

// Column pass over LN neighbouring columns of one coil.  Forward: reads the image rows, writes
// every row, in place.  Inverse: reads every row of `in` and clears it, writes the image rows of
// `out`.
template <bool INV, int LN>
__global__ void __launch_bounds__(F2_T, 4)
k_fft2_col(float2* in, float2* out, Geom geo, F2Axis ax, FfConst k) {
    constexpr int P = LN;
    const int N = ax.N, n0 = geo.n[0], g1 = geo.g[1];
    float2* tw = f2sm + 2 * N * P;
    const int nt = N + fft_axis_extra(ax);
    for (int i = threadIdx.x; i < nt; i += blockDim.x) tw[i] = ax.tw[i];
    const int xblocks = (g1 + LN - 1) / LN;
    const int xb = blockIdx.x % xblocks, c = blockIdx.x / xblocks;
    const int xx = xb * LN + threadIdx.x % LN;
    const bool live = xx < g1;
    const int64_t base = (int64_t)c * geo.G + xx, lim = (int64_t)geo.C * geo.G;
    pdl_begin();
    __syncthreads();
    float2* pi = in + base;                                // n g1 < G < 2^31
    float2* po = out + base;
    const int f = f2_begin<LN, P>(ax, [&](int n) {
        return live && (INV || in_band(n, n0, N)) && KP_INB(1, base + (int64_t)n * g1, lim) ? pi[n * g1]
                                                                                            : make_float2(0.f, 0.f);
    }, N * P, tw, INV ? -1.f : 1.f, k);
    f2_end<LN, P>(ax, [&](int n, float2 v) {
        if (!live || !KP_INB(2, base + (int64_t)n * g1, lim)) return;
        if (!INV || in_band(n, n0, N)) po[n * g1] = v;
        if (INV) pi[n * g1] = make_float2(0.f, 0.f);      // every load of this CTA's columns was done in the first stage
    }, f, tw, INV ? -1.f : 1.f, k);
}

struct F2Step {               // what the adjoint row pass does with A^H u at a pixel
    float2* x;                // F2_IMAGE: output; else the primal iterate
    float2* xbar;
    float2* z;                // F2_Z: output
    const float2* v;          // F2_TV: dual variable
    const float* sched;
    const int* iter;
    float lambda;
    double* nrm;              // F2_IMAGE: nrm[1] += ||x||^2 (or null)
};
enum { F2_IMAGE = 0, F2_L2 = 1, F2_Z = 2, F2_TV = 3 };

// Adjoint row pass.  A CTA takes one image row (RW rows when the coils of one do not fill its LN
// lines) and loops over its coils in groups of CS = min(C, LN); the group's crop is combined into
// the row's sums (coils in ascending order) before the next group loads.
template <typename MT, int LN>
__global__ void __launch_bounds__(F2_T, 4)
k_fft2_row_inv(const float2* __restrict__ in, const MT* __restrict__ maps, const float* __restrict__ apod, Geom geo,
               F2Axis ax, FfConst k, int mode, F2Step sp) {
    constexpr int P = LN + 1;                              // the combine reads a point's lines one after another
    const int N = ax.N, n0 = geo.n[0], n1 = geo.n[1], g0 = geo.g[0], C = geo.C;
    float2* tw = f2sm + 2 * N * P;
    float2* acc = tw + N + fft_axis_extra(ax);             // [RW][n1]
    const int CS = C < LN ? C : LN, RW = LN / CS;
    const int nt = N + fft_axis_extra(ax);
    for (int i = threadIdx.x; i < nt; i += blockDim.x) tw[i] = ax.tw[i];
    const int l = threadIdx.x % LN, r = l / CS, ci = l - r * CS;
    const int row0 = blockIdx.x * RW, nr = min(RW, n0 - row0), h1 = n1 / 2;
    const int ny = row0 + r - n0 / 2;
    pdl_begin();
    __syncthreads();
    for (int c0 = 0; c0 < C; c0 += CS) {
        const int cc = min(CS, C - c0);
        const bool live = r < nr && ci < cc;
        const int64_t base = (int64_t)(c0 + ci) * geo.G + (int64_t)(ny < 0 ? ny + g0 : ny) * N;
        const float2* pi = in + base;
        const int f = f2_begin<LN, P>(ax, [&](int n) {
            return live && KP_INB(1, base + n, (int64_t)C * geo.G) ? pi[n] : make_float2(0.f, 0.f);
        }, N * P, tw, -1.f, k);
        const int o = f ? 0 : N * P;
        f2_end<LN, P>(ax, [&](int n, float2 v) { f2sm[o + n * P + l] = v; }, f, tw, -1.f, k);
        __syncthreads();
        for (int q = 0; q < nr; ++q) {
            const int64_t j0 = (int64_t)(row0 + q) * n1;
            for (int px = threadIdx.x; px < n1; px += blockDim.x) {
                const float2* b = f2sm + o + (px < h1 ? px - h1 + N : px - h1) * P + q * CS;
                float2 m[LN];
#pragma unroll
                for (int e = 0; e < LN; ++e)
                    m[e] = maps && e < cc ? ldc<MT>(maps, (size_t)(c0 + e) * geo.N + j0 + px) : make_float2(1.f, 0.f);
                float2 s = c0 > 0 ? acc[q * n1 + px] : make_float2(0.f, 0.f);
#pragma unroll
                for (int e = 0; e < LN; ++e) {
                    if (e >= cc) break;
                    const float2 v = maps ? cmulc(m[e], b[e]) : b[e];
                    s.x += v.x;
                    s.y += v.y;
                }
                acc[q * n1 + px] = s;                      // owned by this thread in every group
            }
        }
        __syncthreads();                                   // the next group's first stage rewrites the buffers
    }
    float tau = 0.f, theta = 0.f;
    if (mode != F2_IMAGE) {
        const int it = *sp.iter;
        tau = sp.sched[3 * it + 1];
        theta = sp.sched[3 * it + 2];
    }
    double nn = 0.0;
    for (int q = 0; q < nr; ++q) {
        const float ay = geo.rsqrtN * apod[row0 + q];
        for (int px = threadIdx.x; px < n1; px += blockDim.x) {
            const int64_t j = (int64_t)(row0 + q) * n1 + px;
            if (!KP_INB(12, j, geo.N)) continue;
            const float a = ay * apod[n0 + px];
            const float2 s = acc[q * n1 + px];
            const float2 ah = make_float2(s.x * a, s.y * a);
            if (mode == F2_IMAGE) {
                sp.x[j] = ah;
                nn += (double)ah.x * ah.x + (double)ah.y * ah.y;
                continue;
            }
            const float2 xo = sp.x[j];
            float2 z = make_float2(xo.x - tau * ah.x, xo.y - tau * ah.y);
            if (mode == F2_Z) {
                sp.z[j] = z;
                continue;
            }
            if (mode == F2_L2) {
                const float sc = 1.f / (1.f + tau * sp.lambda);
                z.x *= sc;
                z.y *= sc;
            } else {                                       // G^H v = sum_a v_a[j - e_a] - v_a[j], periodic
                const int64_t jy = row0 + q > 0 ? j - n1 : j + (int64_t)(n0 - 1) * n1;
                const int64_t jx = px > 0 ? j - 1 : j + n1 - 1;
                const float2 v0 = sp.v[j], v1 = sp.v[geo.N + j], vy = sp.v[jy], vx = sp.v[geo.N + jx];
                z.x -= tau * ((vy.x - v0.x) + (vx.x - v1.x));
                z.y -= tau * ((vy.y - v0.y) + (vx.y - v1.y));
            }
            sp.xbar[j] = make_float2(z.x + theta * (z.x - xo.x), z.y + theta * (z.y - xo.y));
            sp.x[j] = z;
        }
    }
    if (mode == F2_IMAGE && sp.nrm) {
        __shared__ double ws[F2_T / 32];
        const int w = threadIdx.x >> 5;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) nn += __shfl_down_sync(0xffffffffu, nn, o);
        if ((threadIdx.x & 31) == 0) ws[w] = nn;
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int i = 1; i < (int)(blockDim.x >> 5); ++i) nn += ws[i];
            atomicAdd(sp.nrm + 1, nn);
        }
    }
}

// ---------------------------------------------------------------- 3D
// One pass along AXIS (0 = z, 1 = y, 2 = x) of every coil's 3D grid, for lengths without a compiled
// pass (kp_fft.cu, whose lines and pruning it follows: forward reads only the image band, inverse
// writes only it; x passes take only the rows of the band, y passes its planes).  In place for the y,
// z and inverse passes: a CTA's loads are all in the first stage, before a barrier.
template <int AXIS, bool INV, bool PRE, typename MT>
__global__ void __launch_bounds__(F2_T, 4) k_fftg_pass(const float2* in, float2* out, Geom geo, F2Axis ax, FfConst k, PreSrc pre) {
    constexpr int LN = 8, P = LN;
    const int N = ax.N, n0 = geo.n[0], n1 = geo.n[1], n2 = geo.n[2], g0 = geo.g[0], g1 = geo.g[1], g2 = geo.g[2];
    float2* tw = f2sm + 2 * N * P;
    const int nt = N + fft_axis_extra(ax);
    for (int i = threadIdx.x; i < nt; i += blockDim.x) tw[i] = ax.tw[i];
    const int l = threadIdx.x % LN, na = AXIS == 0 ? n0 : AXIS == 1 ? n1 : n2;
    const int64_t lim = (int64_t)geo.C * geo.G;
    int64_t base = 0, img = 0;                              // element 0 of this thread's line; its image row
    int stride = 1, c = 0;
    float ay = 1.f;
    bool live;
    if (AXIS == 2) {
        const int64_t line = (int64_t)blockIdx.x * LN + l;  // (image row, coil), coil fastest
        live = line < (int64_t)geo.C * n0 * n1;
        const int rem = live ? (int)(line / geo.C) : 0;
        c = live ? (int)(line % geo.C) : 0;
        const int z = band_index(rem / n1, n0, g0), y = band_index(rem % n1, n1, g1);
        base = (int64_t)c * geo.G + ((int64_t)z * g1 + y) * g2;
        if (PRE) {
            const int pz = pix_index(z, n0, g0), py = pix_index(y, n1, g1);
            img = ((int64_t)pz * n1 + py) * n2;
            ay = pre.apod[pz] * pre.apod[n0 + py];
        }
    } else {
        const int xblocks = (g2 + LN - 1) / LN, outer = AXIS == 1 ? n0 : g1;
        const int xb = blockIdx.x % xblocks, rest = blockIdx.x / xblocks, o = rest % outer;
        const int x = xb * LN + l;
        live = x < g2;
        base = (int64_t)(rest / outer) * geo.G + (AXIS == 1 ? (int64_t)band_index(o, n0, g0) * g1 * g2 : (int64_t)o * g2) + (live ? x : 0);
        stride = AXIS == 1 ? g2 : g1 * g2;                   // n stride < G < 2^31
    }
    const float2* pi = in + base;
    float2* po = out + base;
    const float* ax2 = PRE ? pre.apod + n0 + n1 : nullptr;
    const float2* xr = pre.x + img;
    const MT* mr = PRE && pre.maps ? (const MT*)pre.maps + (size_t)c * geo.N + img : nullptr;
    __syncthreads();
    const float s = INV ? -1.f : 1.f;
    const int f = f2_begin<LN, P>(ax, [&](int n) {
        const bool ok = live && (INV || in_band(n, na, N));
        if constexpr (PRE) {                                // no branches around the loads (see k_fft2_row_fwd)
            const int px = ok ? pix_index(n, n2, N) : 0;
            if (!KP_INB(3, px, n2)) return make_float2(0.f, 0.f);
            float2 v = xr[px];
            const float2 m = mr ? ldc<MT>(mr, px) : make_float2(1.f, 0.f);
            const float a = ok ? ay * ax2[px] : 0.f;
            v.x *= a;
            v.y *= a;
            if (mr) v = cmul(m, v);
            return ok ? v : make_float2(0.f, 0.f);
        } else {
            return ok && KP_INB(1, base + (int64_t)n * stride, lim) ? pi[n * stride] : make_float2(0.f, 0.f);
        }
    }, N * P, tw, s, k);
    f2_end<LN, P>(ax, [&](int n, float2 v) {
        if (live && (!INV || in_band(n, na, N)) && KP_INB(2, base + (int64_t)n * stride, lim)) po[n * stride] = v;
    }, f, tw, s, k);
}

// ---------------------------------------------------------------- host
static size_t fwd_smem(const F2Axis& ax, int ln) { return ((size_t)(2 * ln + 1) * ax.N + fft_axis_extra(ax)) * sizeof(float2); }
static size_t inv_smem(const F2Axis& ax, int ln, int acc) { return fwd_smem(ax, ln) + ((size_t)2 * ax.N + acc) * sizeof(float2); }

void fft_axis_table(const F2Axis& ax, std::vector<float2>& h) {
    const auto root = [](int m, int n) {
        const double a = -2.0 * M_PI * (double)m / (double)n;
        return make_float2((float)std::cos(a), (float)std::sin(a));
    };
    for (int m = 0; m < ax.N; ++m) h.push_back(root(m, ax.N));
    const int R = ax.r[0], H = (R - 1) / 2;
    if (fft_axis_extra(ax) > 0)
        for (int q = 1; q <= H; ++q)
            for (int t = 0; t <= H; ++t) h.push_back(root(q * t % R, R));
}

// Threads of a pass: its largest stage in as few equal rounds as F2_T threads allow.
static int pass_threads(const F2Axis& ax, int ln) {
    int items = 0;
    for (int i = 0; i < ax.nst; ++i) items = std::max(items, ax.N / (ax.r[i] > 19 ? 2 * F2_TB : ax.r[i]) * ln);
    const int rounds = (items + F2_T - 1) / F2_T;
    return ((items + rounds - 1) / rounds + 31) / 32 * 32;
}

// Radices of N: at most one prime above 5 (first), then the fewest radices (and the smallest sum)
// for the rest, at least two in all; false if N is not handled.
bool fft_axis_factor(int N, F2Axis& ax) {
    static const int rad[] = {10, 9, 8, 6, 5, 4, 3, 2};
    int rest = N;
    std::vector<int> r;
    for (int p : {2, 3, 5}) while (rest % p == 0) rest /= p;
    int smooth = N / rest;
    for (int p = 7; p <= F2_MAXP && rest > 1; p += 2)
        while (rest % p == 0) {
            r.push_back(p);
            rest /= p;
        }
    if (rest != 1) return false;
    std::sort(r.begin(), r.end(), [](int a, int b) { return a > b; });
    if (r.size() > 1) return false;
    // fewest stages (then the smallest sum) over the divisors of the smooth part
    std::vector<int> st(smooth + 1, 1 << 20), sum(smooth + 1, 0), by(smooth + 1, 0);
    st[1] = 0;
    for (int d = 2; d <= smooth; ++d) {
        if (smooth % d) continue;
        for (int q : rad)
            if (d % q == 0 && (st[d / q] + 1 < st[d] || (st[d / q] + 1 == st[d] && sum[d / q] + q < sum[d]))) {
                st[d] = st[d / q] + 1;
                sum[d] = sum[d / q] + q;
                by[d] = q;
            }
    }
    std::vector<int> small;
    for (int d = smooth; d > 1; d /= by[d]) small.push_back(by[d]);
    if (r.empty() && small.size() == 1)                    // one radix: split off its smallest factor
        for (int p : {2, 3, 5})
            if (small[0] % p == 0 && small[0] > p) { small = {small[0] / p, p}; break; }
    std::sort(small.begin(), small.end());
    r.insert(r.end(), small.begin(), small.end());
    if (r.size() < 2 || r.size() > F2_MAXST || (r[0] > 5 && small.empty())) return false;
    ax.N = N;
    ax.nst = (int)r.size();
    int L = 1;
    for (int i = 0; i < ax.nst; ++i) {
        ax.r[i] = r[i];
        const int m = N / r[i] / L;
        ax.mg[i] = m > 1 ? (unsigned)(((uint64_t)1 << 32) / m + 1) : 0;
        L *= r[i];
    }
    return true;
}

// Lines per CTA: 8, or 4 where 8 would leave SMs without a CTA (small images) or need more shared
// memory than a CTA has.
static int lines_for(int64_t blocks8, size_t smem8) { return blocks8 >= 152 && smem8 <= (size_t)F2_SMEM ? 8 : 4; }

// Passes for grids of g0 x g1 points (image rows up to n1 points); null when a length is not handled, or
// KPDHG_FFT=cufft.  *status tells an allocation failure from that.
Fft2Plan* fft2_make(int g0, int g1, int n1, kp_status* status) {
    *status = KP_OK;
    const char* env = std::getenv("KPDHG_FFT");
    if (env && std::string(env) == "cufft") return nullptr;
    Fft2Plan f{};
    if (!fft_axis_factor(g0, f.ax[0]) || !fft_axis_factor(g1, f.ax[1])) return nullptr;
    if (inv_smem(f.ax[1], 4, n1 * 4) > (size_t)F2_SMEM || fwd_smem(f.ax[0], 4) > (size_t)F2_SMEM) return nullptr;
    Fft2Plan* q = new (std::nothrow) Fft2Plan(f);
    *status = KP_ENOMEM;
    if (!q) { set_error("host allocation failed"); return nullptr; }
    std::vector<float2> h;
    fft_axis_table(f.ax[0], h);
    const size_t first = h.size();
    fft_axis_table(f.ax[1], h);
    if (cudaMalloc(&q->d_tw, h.size() * sizeof(float2)) != cudaSuccess ||
        cudaMemcpy(q->d_tw, h.data(), h.size() * sizeof(float2), cudaMemcpyHostToDevice) != cudaSuccess) {
        cudaGetLastError();
        fft2_free(q);
        set_error("device allocation failed");
        return nullptr;
    }
    *status = KP_OK;
    q->ax[0].tw = q->d_tw;
    q->ax[1].tw = q->d_tw + first;
    q->k = ff_const();
    return q;
}

void fft2_free(Fft2Plan* q) {
    if (!q) return;
    if (q->d_tw) cudaFree(q->d_tw);
    delete q;
}

kp_status fft2_create(kp_plan p) {
    const Geom& g = p->geo;
    if (g.D != 2) return KP_OK;
    kp_status st;
    p->fft2 = fft2_make(g.g[0], g.g[1], g.n[1], &st);
    if (!p->fft2) return st;
    // the spread grid is zero between adjoints (the inverse column pass clears what it reads)
    KP_TRY_CUDA(cudaMemset(p->d_grid2, 0, (size_t)g.C * g.G * sizeof(float2)));
    return KP_OK;
}

void fft2_destroy(kp_plan p) {
    fft2_free(p->fft2);
    p->fft2 = nullptr;
}

// Where a forward transform takes its images from (k_fft2_row_fwd).
struct F2Src {
    const float2* x;
    int64_t xstride;
    const int2* pairs;
    bool pair;
    const void* maps;
    const float* apod;
    int* iter;
    double* nrm;
};

template <typename MT, int LN, bool PAIR>
static kp_status launch_row_fwd(const Fft2Plan* f, const Geom& g, const F2Src& a, float2* out, cudaStream_t st) {
    static SmemLimit lim;
    const size_t sm = fwd_smem(f->ax[1], LN);
    KP_TRY_CUDA(lim.ensure(k_fft2_row_fwd<MT, LN, PAIR>, sm));
    const unsigned nb = (unsigned)(((int64_t)g.n[0] * g.C + LN - 1) / LN);
    KP_TRY_CUDA(launch_pdl(k_fft2_row_fwd<MT, LN, PAIR>, nb, pass_threads(f->ax[1], LN), sm, st, a.x, a.xstride, a.pairs,
                           (const MT*)a.maps, a.apod, g, f->ax[1], f->k, out, a.iter, a.nrm));
    return KP_OK;
}

template <typename MT>
static kp_status row_fwd_t(const Fft2Plan* f, const Geom& g, const F2Src& a, float2* out, cudaStream_t st) {
    const bool eight = lines_for(((int64_t)g.n[0] * g.C + 7) / 8, fwd_smem(f->ax[1], 8)) == 8;
    if (a.pair) return eight ? launch_row_fwd<MT, 8, true>(f, g, a, out, st) : launch_row_fwd<MT, 4, true>(f, g, a, out, st);
    return eight ? launch_row_fwd<MT, 8, false>(f, g, a, out, st) : launch_row_fwd<MT, 4, false>(f, g, a, out, st);
}

template <bool INV, int LN>
static kp_status launch_col(const Fft2Plan* f, const Geom& g, float2* in, float2* out, cudaStream_t st) {
    static SmemLimit lim;
    const size_t sm = fwd_smem(f->ax[0], LN);
    KP_TRY_CUDA(lim.ensure(k_fft2_col<INV, LN>, sm));
    const unsigned nb = (unsigned)((int64_t)g.C * ((g.g[1] + LN - 1) / LN));
    KP_TRY_CUDA(launch_pdl(k_fft2_col<INV, LN>, nb, pass_threads(f->ax[0], LN), sm, st, in, out, g, f->ax[0], f->k));
    return KP_OK;
}

template <bool INV>
static kp_status col_pass(const Fft2Plan* f, const Geom& g, float2* in, float2* out, cudaStream_t st) {
    if (lines_for((int64_t)g.C * ((g.g[1] + 7) / 8), fwd_smem(f->ax[0], 8)) == 8) return launch_col<INV, 8>(f, g, in, out, st);
    return launch_col<INV, 4>(f, g, in, out, st);
}

static kp_status forward_src(const Fft2Plan* f, const Geom& g, kp_cdtype mt, const F2Src& a, float2* out, int64_t& launches,
                             cudaStream_t st) {
    launches += 2;
    switch (a.maps ? mt : KP_C64) {
        case KP_C64: KP_TRY(row_fwd_t<float2>(f, g, a, out, st)); break;
        case KP_C32_BF16: KP_TRY(row_fwd_t<__nv_bfloat162>(f, g, a, out, st)); break;
        default: KP_TRY(row_fwd_t<__half2>(f, g, a, out, st)); break;
    }
    return col_pass<false>(f, g, out, out, st);
}

template <typename MT, int LN>
static kp_status launch_row_inv(kp_plan p, int mode, const F2Step& sp, cudaStream_t st) {
    static SmemLimit lim;
    const Geom& g = p->geo;
    const int rw = LN / std::min(g.C, LN);
    const size_t sm = inv_smem(p->fft2->ax[1], LN, rw * g.n[1]);
    KP_TRY_CUDA(lim.ensure(k_fft2_row_inv<MT, LN>, sm));
    const unsigned nb = (unsigned)((g.n[0] + rw - 1) / rw);
    KP_TRY_CUDA(launch_pdl(k_fft2_row_inv<MT, LN>, nb, pass_threads(p->fft2->ax[1], LN), sm, st, p->d_grid,
                           p->unit_maps ? nullptr : (const MT*)p->d_maps, p->d_apod, g, p->fft2->ax[1], p->fft2->k, mode, sp));
    return KP_OK;
}

template <typename MT>
static kp_status row_inv_t(kp_plan p, int mode, const F2Step& sp, cudaStream_t st) {
    const Geom& g = p->geo;
    const int rw = 8 / std::min(g.C, 8);
    // 4 lines for up to 4 coils: one image row each without idle lines (16 lines for 9 to 16 coils
    // measured the same as two groups of 8)
    if (g.C > 4 && lines_for((g.n[0] + rw - 1) / rw, inv_smem(p->fft2->ax[1], 8, rw * g.n[1])) == 8)
        return launch_row_inv<MT, 8>(p, mode, sp, st);
    return launch_row_inv<MT, 4>(p, mode, sp, st);
}

static kp_status row_inv(kp_plan p, int mode, const F2Step& sp, cudaStream_t st) {
    p->launches += 1;
    switch (p->unit_maps ? KP_C64 : p->maps_t) {
        case KP_C64: return row_inv_t<float2>(p, mode, sp, st);
        case KP_C32_BF16: return row_inv_t<__nv_bfloat162>(p, mode, sp, st);
        default: return row_inv_t<__half2>(p, mode, sp, st);
    }
}

kp_status fft2_forward_image(kp_plan p, const float2* x, int* iter, double* nrm, cudaStream_t st) {
    const F2Src a{x, 0, nullptr, false, p->unit_maps ? nullptr : p->d_maps, p->d_apod, iter, nrm};
    return forward_src(p->fft2, p->geo, p->maps_t, a, p->d_gridF, p->launches, st);
}

kp_status fft2_forward_batch(kp_plan p, const float2* x, int n, float2* out, cudaStream_t st) {
    Geom g = p->geo;
    g.C = n;
    const F2Src a{x, g.N, nullptr, false, nullptr, p->d_apod, nullptr, nullptr};
    return forward_src(p->fft2, g, KP_C64, a, out, p->launches, st);
}

kp_status fft2_forward_pairs(const Fft2Plan* f, const Geom& g, kp_cdtype mt, const void* maps, const int2* pairs, float2* out,
                             int64_t& launches, cudaStream_t st) {
    const F2Src a{nullptr, 0, pairs, true, maps, nullptr, nullptr, nullptr};
    return forward_src(f, g, mt, a, out, launches, st);
}

kp_status fft2_inverse_cols(kp_plan p, cudaStream_t st) {
    p->launches += 1;
    return col_pass<true>(p->fft2, p->geo, p->d_grid2, p->d_grid, st);
}

kp_status fft2_adjoint_image(kp_plan p, float2* x, double* nrm, cudaStream_t st) {
    F2Step sp{};
    sp.x = x;
    sp.nrm = nrm;
    return row_inv(p, F2_IMAGE, sp, st);
}

kp_status fft2_adjoint_primal(kp_plan p, int reg, float lambda, cudaStream_t st) {
    F2Step sp{};
    sp.x = p->d_x;
    sp.xbar = p->d_xbar;
    sp.z = p->d_z;
    sp.v = p->d_v;
    sp.sched = p->d_sched;
    sp.iter = p->d_iter;
    sp.lambda = lambda;
    return row_inv(p, reg == KP_REG_L2 ? F2_L2 : reg == KP_REG_TV ? F2_TV : F2_Z, sp, st);
}

bool fftg_fits(const F2Axis& ax) { return fwd_smem(ax, 8) <= (size_t)F2_SMEM; }

template <int AXIS, bool INV, bool PRE, typename MT>
kp_status fftg_pass(const F2Axis& ax, const FfConst& k, const Geom& g, const float2* in, float2* out, const PreSrc& pre, cudaStream_t st) {
    static SmemLimit lim;
    const size_t sm = fwd_smem(ax, 8);
    KP_TRY_CUDA(lim.ensure(k_fftg_pass<AXIS, INV, PRE, MT>, sm));
    const int64_t xblocks = (g.g[2] + 7) / 8;
    const int64_t nb = AXIS == 2 ? ((int64_t)g.C * g.n[0] * g.n[1] + 7) / 8 : (int64_t)g.C * (AXIS == 1 ? g.n[0] : g.g[1]) * xblocks;
    if (nb > INT32_MAX) { set_error("grid too large for the FFT passes"); return KP_EINVAL; }
    k_fftg_pass<AXIS, INV, PRE, MT><<<(unsigned)nb, pass_threads(ax, 8), sm, st>>>(in, out, g, ax, k, pre);
    KP_LAUNCH_CHECK();
    return KP_OK;
}
#define KP_FFTG(A, I, P, T) \
    template kp_status fftg_pass<A, I, P, T>(const F2Axis&, const FfConst&, const Geom&, const float2*, float2*, const PreSrc&, cudaStream_t);
KP_FFTG(2, false, true, float2)
KP_FFTG(2, false, true, __nv_bfloat162)
KP_FFTG(2, false, true, __half2)
KP_FFTG(2, false, false, float2)
KP_FFTG(1, false, false, float2)
KP_FFTG(0, false, false, float2)
KP_FFTG(0, true, false, float2)
KP_FFTG(1, true, false, float2)
KP_FFTG(2, true, false, float2)
#undef KP_FFTG

}  // namespace kp
