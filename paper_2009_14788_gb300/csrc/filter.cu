// Sinogram filtering for filtered backprojection (Section 3.1.3).
//
// The Fourier filter of Kak & Slaney (Chapter 3, Eq. 61) is the DFT of the band-limited ramp kernel
// h(0) = 1/4, h(m) = -1 / (pi^2 m^2) for odd m, 0 for even m != 0, zero-padded to P >= 2D - 1, times
// a window of the normalised frequency.  Applied to a zero-padded projection it is a circular
// convolution that, thanks to the padding, equals the linear convolution of the D bins with the
// kernel k = IDFT(filter) at offsets -(D-1) .. D-1.  The taps (pi / V) k are computed here once per
// geometry in FP64 (a radix-2 FFT for the windowed filters; Ram-Lak's taps are the closed form) and
// the kernel sums the linear convolution directly in FP32, with no FFT on the device.  Each tap is stored
// as an FP32 pair hi + lo: a high-pass filter cancels terms up to ~150 times the result, and one FP32
// rounding per tap (fixed, so it does not average out) would leave a systematic 1e-5-level error; the
// pair removes it.
#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

#include "dtype.cuh"
#include "f32x2.cuh"
#include "radon_internal.h"

namespace radon {

namespace {

constexpr int kFilterKinds = 5;
constexpr int kFilterThreads = 256;
constexpr int kFilterOut = 8;    // outputs per thread
constexpr int kLongOut = 4;      // consecutive outputs per thread of the kernel for long rows
// Taps nearer than this also add their lo part.  Every kernel here falls off like 1 / m^2: all farther taps
// together are at most 2.5e-3 (cosine; 1.6e-3 the others), so leaving their rounding (up to 2^-24 each) moves
// a result by at most 1.5e-10 of the largest input, a twenty-fifth of what one rounding of the sum at its
// largest moves it (2^-25 / 8).  With every lo part the errors against 64 bits are the same in three digits
// (91 .. 4000 bins, all windows, smooth and random rows), and 4000 bins take 655 instead of 309 us.
constexpr int kFilterNear = 64;

using cd = std::complex<double>;

// In-place radix-2 FFT of length a.size() (a power of two); inverse without the 1/P factor.
void fft(std::vector<cd>& a, bool inverse) {
    const size_t n = a.size();
    for (size_t i = 1, j = 0; i < n; ++i) {
        size_t bit = n >> 1;
        for (; j & bit; bit >>= 1) j ^= bit;
        j ^= bit;
        if (i < j) std::swap(a[i], a[j]);
    }
    for (size_t len = 2; len <= n; len <<= 1) {
        const double ang = 2.0 * M_PI / (double)len * (inverse ? 1.0 : -1.0);
        const cd wl(std::cos(ang), std::sin(ang));
        for (size_t i = 0; i < n; i += len) {
            cd w(1.0, 0.0);
            for (size_t k = 0; k < len / 2; ++k) {
                const cd u = a[i + k], v = a[i + k + len / 2] * w;
                a[i + k] = u + v;
                a[i + k + len / 2] = u - v;
                w *= wl;
            }
        }
    }
}

double ramp(long long m) {
    if (m == 0) return 0.25;
    if ((m & 1) == 0) return 0.0;
    return -1.0 / (M_PI * M_PI * (double)m * (double)m);
}

double window(int kind, double f) {
    switch (kind) {
        case RADON_FILTER_SHEPP_LOGAN: return f == 0.0 ? 1.0 : std::sin(M_PI * f) / (M_PI * f);
        case RADON_FILTER_COSINE: return std::cos(M_PI * f);
        case RADON_FILTER_HAMMING: return 0.54 + 0.46 * std::cos(2.0 * M_PI * f);
        case RADON_FILTER_HANN: return 0.5 + 0.5 * std::cos(2.0 * M_PI * f);
        default: return 1.0;
    }
}

// One row whose taps and bins do not fit one CTA's shared memory in the layout below (more than about
// 9600 bins): out[d] = sum_{d'} y[d'] taps[d - d' + D - 1], kLongOut outputs per thread; each tap is a
// (hi, lo) pair summed into two accumulators.
template <typename T>
__global__ void __launch_bounds__(kFilterThreads) filter_long_rows_kernel(const T* __restrict__ in, T* __restrict__ out,
                                                                     const float2* __restrict__ taps, int D) {
    extern __shared__ float fsm[];
    const int Dp = (D + kLongOut - 1) / kLongOut * kLongOut;   // bins padded to whole output groups
    float* y = fsm;                                           // [Dp], zero past D
    float2* t = reinterpret_cast<float2*>(fsm + Dp + (Dp & 1));   // taps at offset +kLongOut
    const long long row = blockIdx.x;
    const T* src = in + row * D;
    for (int d = threadIdx.x; d < Dp; d += blockDim.x) y[d] = d < D ? to_f32(src[d]) : 0.0f;
    const int nt = 2 * Dp + 2 * kLongOut;
    for (int j = threadIdx.x; j < nt; j += blockDim.x) {
        const int m = j - kLongOut;    // tap index relative to taps[0]
        t[j] = (m >= 0 && m < 2 * D - 1) ? taps[m] : make_float2(0.0f, 0.0f);
    }
    __syncthreads();
    T* dst = out + row * D;
    for (int d0 = threadIdx.x * kLongOut; d0 < D; d0 += blockDim.x * kLongOut) {
        float hi[kLongOut], lo[kLongOut];
#pragma unroll
        for (int o = 0; o < kLongOut; ++o) hi[o] = lo[o] = 0.0f;
        // tap of output d0 + o and input d' sits at t[d0 + o - d' + D - 1 + kLongOut]; the taps
        // of consecutive inputs slide by one, so a register window takes one new tap per input
        const float2* tb = t + d0 + D - 1 + kLongOut;
        float2 w[kLongOut];
#pragma unroll
        for (int o = 0; o < kLongOut; ++o) w[o] = tb[o];
        for (int q = 0; q < Dp; q += kLongOut) {
#pragma unroll
            for (int u = 0; u < kLongOut; ++u) {
                const float yv = y[q + u];
#pragma unroll
                for (int o = 0; o < kLongOut; ++o) {
                    hi[o] = fmaf(yv, w[o].x, hi[o]);
                    lo[o] = fmaf(yv, w[o].y, lo[o]);
                }
#pragma unroll
                for (int o = kLongOut - 1; o > 0; --o) w[o] = w[o - 1];
                w[0] = tb[-(q + u + 1)];
            }
        }
#pragma unroll
        for (int o = 0; o < kLongOut; ++o)
            if (d0 + o < D) dst[d0 + o] = from_f32<T>(hi[o] + lo[o]);
    }
}

// Shared-memory plan of a CTA (floats), the same on host and device.  The convolution runs as S sums over
// interleaved bins: with HALF (Ram-Lak, whose taps at even offsets but zero are exactly 0) the even
// outputs take the odd bins and the odd outputs the even ones, S = 2; otherwise S = 1.  Sum s has
// `A` outputs in groups of kFilterOut and `L4` bins (whole float4s, zero past the row).
struct FilterPlan {
    int L4;      // bins of one sum
    int A8;      // outputs of one sum, in whole groups
    int nt;      // reversed taps of one copy
    int c0;      // place of the tap of bin distance zero in the first copy
    int bl;      // reach of the near taps, in bins of the sum
    int ntl;     // reversed near (lo) taps of one copy
    int tap_floats, row_floats;
};

template <bool HALF>
__host__ __device__ inline FilterPlan filter_plan(int D) {
    FilterPlan f;
    const int A = HALF ? (D + 1) / 2 : D;
    f.L4 = (A + 3) / 4 * 4;
    f.A8 = (A + kFilterOut - 1) / kFilterOut * kFilterOut;
    f.c0 = f.A8 + 8;
    f.nt = f.A8 + f.L4 + 24;
    f.bl = HALF ? kFilterNear / 2 : kFilterNear;
    f.ntl = 2 * f.bl + 24;
    f.tap_floats = (HALF ? 2 : 1) * 2 * (f.nt + f.ntl);
    // an odd number of float4s: the rows that a warp reads at once lie in different banks
    f.row_floats = (((HALF ? 2 : 1) * f.L4 + D + 3) / 4 | 1) * 4;
    return f;
}

// out[d] = sum_d' y[d'] taps[d - d' + D - 1] for `rpc` rows per CTA, `tpr` threads per row, kFilterOut
// outputs of one sum per thread.  Bound by FP32 issue: products are paired over two neighbouring bins
// (fma.rn.f32x2: half the instructions), so an output's taps are needed as pairs at even and at odd
// offsets: the reversed taps lie in shared memory twice, the second copy shifted by one, and both
// windows slide in registers, one 16-byte load of each per four bins.  With Ram-Lak the zero taps are
// left out.  512 views of 725 bins, FP32: 73 us with one bin per scalar FMA, both tap parts and the
// zeros; 23 us so (29 us under the other windows; 500 views of 4000 bins 2078 -> 306 us).
template <typename T, bool HALF>
__global__ void __launch_bounds__(kFilterThreads) filter_rows_kernel(const T* __restrict__ in, T* __restrict__ out,
                                                                     const float2* __restrict__ taps, int D,
                                                                     long long rows, int rpc, int tpr) {
    extern __shared__ __align__(16) float fsm[];
    constexpr int S = HALF ? 2 : 1;
    const FilterPlan f = filter_plan<HALF>(D);
    const long long row0 = (long long)blockIdx.x * rpc;
    const int nrows = (int)min((long long)rpc, rows - row0);
    float* rowmem = fsm + f.tap_floats;
    // reversed taps of sum s: hi even copy [nt], hi odd copy, lo even copy [ntl], lo odd copy; entry x of
    // the even copies is the tap of bin distance (output - bin) = c0 - x (hi) or bl + 8 - x (lo), the odd
    // copies hold the same one place later
    for (int e = threadIdx.x; e < S * (f.nt + f.ntl); e += blockDim.x) {
        const int s = HALF ? e / (f.nt + f.ntl) : 0, x = e - s * (f.nt + f.ntl);
        const bool far = x < f.nt;
        float* dst = fsm + s * 2 * (f.nt + f.ntl) + (far ? x : 2 * f.nt + (x - f.nt));
        const int q = far ? f.c0 - x : f.bl + 8 - (x - f.nt);
#pragma unroll
        for (int odd = 0; odd < 2; ++odd) {
            const int m = HALF ? 2 * (q + odd) + 2 * s - 1 : q + odd;   // offset in bins of the row
            float v = 0.0f;
            if (m > -D && m < D) {
                const float2 t = __ldg(taps + m + D - 1);
                v = far ? t.x : (m > -kFilterNear && m < kFilterNear ? t.y : 0.0f);
            }
            dst[odd * (far ? f.nt : f.ntl)] = v;
        }
    }
    // rows: with HALF the odd bins first (the even outputs' sum), then the even bins
    bool odd_values = false;   // infinities or NaN
    // (an element's row by a multiplication: at most 64 rows of fewer than 2^16 bins leave its rounding no say)
    const int bins = S * f.L4;
    const float per_bins = 1.0f / (float)bins, per_D = 1.0f / (float)D;
    for (int e = threadIdx.x; e < nrows * bins; e += blockDim.x) {
        const int r = (int)(((float)e + 0.5f) * per_bins), d = e - r * bins;
        const float v = d < D ? to_f32(in[(row0 + r) * D + d]) : 0.0f;
        odd_values = odd_values || !(fabsf(v) < INFINITY);
        rowmem[r * f.row_floats + (HALF ? ((d & 1) ? d >> 1 : f.L4 + (d >> 1)) : d)] = v;
    }
    odd_values = __syncthreads_or(odd_values) != 0;
    const int r = (int)threadIdx.x / tpr, t0 = (int)threadIdx.x - r * tpr;
    if (r < nrows) {
        const float* y = rowmem + (size_t)r * f.row_floats;
        float* res = rowmem + (size_t)r * f.row_floats + S * f.L4;
        const int gps = f.A8 / kFilterOut;   // groups per sum
        for (int g = t0; g < S * gps; g += tpr) {
            const int s = HALF ? (g >= gps ? 1 : 0) : 0, a0 = (g - s * gps) * kFilterOut;
            const float* x = y + s * f.L4;
            const float* tp = fsm + s * 2 * (f.nt + f.ntl);
            f32x2 acc[kFilterOut];
#pragma unroll
            for (int o = 0; o < kFilterOut; ++o) acc[o] = 0ull;
            // bins [i0, i1) (multiples of 4) against the taps at e (outputs a0, a0 + 2, ...) and d (a0 + 1, ...)
            auto conv = [&](const float* xi, const float* e, const float* d, int n) {
                f32x2 e3 = *reinterpret_cast<const f32x2*>(e - 6), e2 = *reinterpret_cast<const f32x2*>(e - 4),
                      e1 = *reinterpret_cast<const f32x2*>(e - 2);
                f32x2 d3 = *reinterpret_cast<const f32x2*>(d - 6), d2 = *reinterpret_cast<const f32x2*>(d - 4),
                      d1 = *reinterpret_cast<const f32x2*>(d - 2);
#pragma unroll 2
                for (int i = 0; i < n; i += 4) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(xi + i);
                    const ulonglong2 ee = *reinterpret_cast<const ulonglong2*>(e + i);
                    const ulonglong2 dd = *reinterpret_cast<const ulonglong2*>(d + i);
                    acc[0] = f2_fma(v.x, ee.x, acc[0]);
                    acc[1] = f2_fma(v.x, dd.x, acc[1]);
                    acc[2] = f2_fma(v.x, e1, acc[2]);
                    acc[3] = f2_fma(v.x, d1, acc[3]);
                    acc[4] = f2_fma(v.x, e2, acc[4]);
                    acc[5] = f2_fma(v.x, d2, acc[5]);
                    acc[6] = f2_fma(v.x, e3, acc[6]);
                    acc[7] = f2_fma(v.x, d3, acc[7]);
                    acc[0] = f2_fma(v.y, ee.y, acc[0]);
                    acc[1] = f2_fma(v.y, dd.y, acc[1]);
                    acc[2] = f2_fma(v.y, ee.x, acc[2]);
                    acc[3] = f2_fma(v.y, dd.x, acc[3]);
                    acc[4] = f2_fma(v.y, e1, acc[4]);
                    acc[5] = f2_fma(v.y, d1, acc[5]);
                    acc[6] = f2_fma(v.y, e2, acc[6]);
                    acc[7] = f2_fma(v.y, d2, acc[7]);
                    e3 = e1;
                    e2 = ee.x;
                    e1 = ee.y;
                    d3 = d1;
                    d2 = dd.x;
                    d1 = dd.y;
                }
            };
            // the same from the last bins to the first
            auto conv_back = [&](const float* xi, const float* e, const float* d, int n) {
                ulonglong2 ee = *reinterpret_cast<const ulonglong2*>(e + n - 4), em = *reinterpret_cast<const ulonglong2*>(e + n - 8);
                ulonglong2 dd = *reinterpret_cast<const ulonglong2*>(d + n - 4), dm = *reinterpret_cast<const ulonglong2*>(d + n - 8);
#pragma unroll 3
                for (int i = n - 4; i >= 0; i -= 4) {
                    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(xi + i);
                    const ulonglong2 eb = *reinterpret_cast<const ulonglong2*>(e + i - 8);
                    const ulonglong2 db = *reinterpret_cast<const ulonglong2*>(d + i - 8);
                    acc[0] = f2_fma(v.y, ee.y, acc[0]);
                    acc[1] = f2_fma(v.y, dd.y, acc[1]);
                    acc[2] = f2_fma(v.y, ee.x, acc[2]);
                    acc[3] = f2_fma(v.y, dd.x, acc[3]);
                    acc[4] = f2_fma(v.y, em.y, acc[4]);
                    acc[5] = f2_fma(v.y, dm.y, acc[5]);
                    acc[6] = f2_fma(v.y, em.x, acc[6]);
                    acc[7] = f2_fma(v.y, dm.x, acc[7]);
                    acc[0] = f2_fma(v.x, ee.x, acc[0]);
                    acc[1] = f2_fma(v.x, dd.x, acc[1]);
                    acc[2] = f2_fma(v.x, em.y, acc[2]);
                    acc[3] = f2_fma(v.x, dm.y, acc[3]);
                    acc[4] = f2_fma(v.x, em.x, acc[4]);
                    acc[5] = f2_fma(v.x, dm.x, acc[5]);
                    acc[6] = f2_fma(v.x, eb.y, acc[6]);
                    acc[7] = f2_fma(v.x, db.y, acc[7]);
                    ee = em;
                    em = eb;
                    dd = dm;
                    dm = db;
                }
            };
            // the lo products, summed by themselves
            float lo[kFilterOut];
            const int i0 = max(a0 - f.bl, 0), i1 = min(a0 + kFilterOut + f.bl, f.L4);
            const float* tl = tp + 2 * f.nt + (i0 - a0 + f.bl + 8);
            if (i1 > i0) conv(x + i0, tl, tl + f.ntl, i1 - i0);
#pragma unroll
            for (int o = 0; o < kFilterOut; ++o) {
                float p, q;
                f2_unpack(acc[o], &p, &q);
                lo[o] = p + q;
                acc[o] = 0ull;
            }
            // A high-pass sum is as large as its centre taps make it and small again once they are in, so the
            // bins next to the outputs, [a0 - 4, a0 + 12), are added one by one in row order (the centre
            // tap in its place) between the farther ones of either side: as few additions round at
            // the large values as in a plain sum along the row (pairs throughout left 2.5 times its error).  The
            // farther ones are added from either end towards the outputs, the small terms first; starting the
            // right-hand ones with half of the sum so far in each half of a pair left that half to the end
            // where a window's taps differ at even and odd offsets (cosine: twice a plain sum's error).
            const float* hi = tp + (f.c0 - a0);
            if (a0 > 4) conv(x, hi, hi + f.nt, a0 - 4);
            float v[kFilterOut];
#pragma unroll
            for (int o = 0; o < kFilterOut; ++o) {
                float p, q;
                f2_unpack(acc[o], &p, &q);
                v[o] = p + q;
            }
            float t[24];   // taps of bin distance (bin - output) -12 .. 11
#pragma unroll
            for (int j = 0; j < 24; j += 4)
                *reinterpret_cast<float4*>(t + j) = *reinterpret_cast<const float4*>(tp + f.c0 - 12 + j);
            const float2 centre = __ldg(taps + D - 1);
            float own[kFilterOut];
#pragma unroll
            for (int o = 0; o < kFilterOut; ++o) {
                own[o] = HALF && a0 + o < f.L4 ? y[(1 - s) * f.L4 + a0 + o] : 0.0f;
                lo[o] = HALF ? fmaf(own[o], centre.y, lo[o]) : lo[o];
            }
#pragma unroll
            for (int j = -4; j < 12; j += 4) {
                const int i = a0 + j;
                float xi[4] = {0.0f, 0.0f, 0.0f, 0.0f};
                if (i >= 0 && i < f.L4) *reinterpret_cast<float4*>(xi) = *reinterpret_cast<const float4*>(x + i);
#pragma unroll
                for (int w = 0; w < 4; ++w)
#pragma unroll
                    for (int o = 0; o < kFilterOut; ++o) {
                        // with HALF an output's own bin, one of the other sum's, lies before bin a0 + o of the
                        // odd bins (s = 0) and after bin a0 + o of the even ones (s = 1)
                        if (HALF && j + w == o) v[o] = fmaf(s == 0 ? own[o] : 0.0f, centre.x, v[o]);
                        if (HALF && j + w == o + 1) v[o] = fmaf(s == 0 ? 0.0f : own[o], centre.x, v[o]);
                        v[o] = fmaf(xi[w], t[j + w - o + 12], v[o]);
                    }
            }
            if (HALF && odd_values) {
                // an infinity or NaN among the bins whose taps are left out still makes the output NaN
                float z = 0.0f;
                for (int i = 0; i < f.L4; ++i) z = fmaf(0.0f, y[(1 - s) * f.L4 + i], z);
#pragma unroll
                for (int o = 0; o < kFilterOut; ++o) lo[o] += z;
            }
            const int right = a0 + 12;
#pragma unroll
            for (int o = 0; o < kFilterOut; ++o) acc[o] = 0ull;
            if (right < f.L4) conv_back(x + right, hi + right, hi + f.nt + right, f.L4 - right);
#pragma unroll
            for (int o = 0; o < kFilterOut; ++o) {
                float p, q;
                f2_unpack(acc[o], &p, &q);
                const int a = a0 + o, dd = HALF ? 2 * a + s : a;
                if (dd < D) res[dd] = (v[o] + (p + q)) + lo[o];
            }
        }
    }
    __syncthreads();
    for (int e = threadIdx.x; e < nrows * D; e += blockDim.x) {
        const int q = (int)(((float)e + 0.5f) * per_D);
        out[row0 * D + e] = from_f32<T>(rowmem[q * f.row_floats + S * f.L4 + (e - q * D)]);
    }
}

// Shared memory of the kernel for long rows: the largest row served is the one whose bins and (hi, lo)
// taps one CTA holds.
size_t filter_long_smem(int D) {
    const int Dp = (D + kLongOut - 1) / kLongOut * kLongOut;
    return (size_t)(Dp + (Dp & 1)) * sizeof(float) + (size_t)(2 * Dp + 2 * kLongOut) * sizeof(float2);
}

template <typename T>
cudaError_t filter_launch_long(const void* in, void* out, const float2* taps, int D, long long rows, cudaStream_t s) {
    const size_t smem = filter_long_smem(D);
    cudaError_t e = cudaFuncSetAttribute(filter_long_rows_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    filter_long_rows_kernel<T><<<(unsigned)rows, kFilterThreads, smem, s>>>((const T*)in, (T*)out, taps, D);
    return cudaGetLastError();
}

template <typename T, bool HALF>
cudaError_t filter_launch(const void* in, void* out, const float2* taps, int D, long long rows, cudaStream_t s) {
    const FilterPlan f = filter_plan<HALF>(D);
    const int groups = (HALF ? 2 : 1) * f.A8 / kFilterOut;
    // Threads per row: one per group of outputs, in whole warps or a warp's half, quarter or eighth.
    int tpr = std::min(kFilterThreads, (groups + 31) / 32 * 32);
    while (tpr > 4 && tpr <= 32 && tpr / 2 >= groups) tpr /= 2;
    // Rows per CTA share its taps: two, or as many as 128 threads serve, while three CTAs' worth is left for
    // every SM and two CTAs fit it.
    int rpc = 1;
    if ((size_t)(f.tap_floats + f.row_floats) * sizeof(float) > 227 * 1024)
        return filter_launch_long<T>(in, out, taps, D, rows, s);
    while ((rpc + 1) * tpr <= (rpc == 1 ? kFilterThreads : 128) && rows >= (long long)(rpc + 1) * 152 * 3 &&
           (size_t)(f.tap_floats + (rpc + 1) * f.row_floats) * sizeof(float) <= 112 * 1024)
        ++rpc;
    // Laying out the taps is most of a short launch: few CTAs take more threads for it (us, 128 rows and 8192 rows
    // of 64 | 128 | 256 bins, Ram-Lak: a warp or more per row and no others 5.6, 18.3 | 8.0, 28.0 | 12.1,
    // 46.2; so 3.8, 8.6 | 4.6, 21.9 | 6.2, 46.2; one bin per scalar FMA 3.1, 11.0 | 5.2, 35.2 | 6.3, 122).
    const long long ctas = (rows + rpc - 1) / rpc;
    const int threads = std::max((rpc * tpr + 31) / 32 * 32, ctas <= 2 * 152 ? 256 : ctas <= 8 * 152 ? 128 : 32);
    const size_t smem = (size_t)(f.tap_floats + rpc * f.row_floats) * sizeof(float);
    cudaError_t e = cudaFuncSetAttribute(filter_rows_kernel<T, HALF>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)std::max<size_t>(smem, 48 * 1024));
    if (e != cudaSuccess) return e;
    filter_rows_kernel<T, HALF><<<(unsigned)ctas, threads, smem, s>>>(
        (const T*)in, (T*)out, taps, D, rows, rpc, tpr);
    return cudaGetLastError();
}

template <typename T>
cudaError_t filter_launch(const void* in, void* out, const float2* taps, int D, long long rows, radon_filter filter,
                          cudaStream_t s) {
    return filter == RADON_FILTER_RAM_LAK ? filter_launch<T, true>(in, out, taps, D, rows, s)
                                          : filter_launch<T, false>(in, out, taps, D, rows, s);
}

}  // namespace

radon_status upload_filter_taps(radon_geometry* g) {
    const int D = g->D;
    const long long n_taps = 2LL * D - 1;
    size_t P = 2;   // at least one positive and the Nyquist frequency (D = 1 still filters)
    while ((long long)P < n_taps) P <<= 1;
    std::vector<double> kpad(P);
    for (size_t m = 0; m < P; ++m) kpad[m] = ramp(m <= P / 2 ? (long long)m : (long long)m - (long long)P);
    std::vector<cd> H(P);
    for (size_t m = 0; m < P; ++m) H[m] = cd(kpad[m], 0.0);
    fft(H, false);
    std::vector<float2> taps((size_t)kFilterKinds * n_taps);
    const double scale = M_PI / (double)g->V;
    for (int kind = 0; kind < kFilterKinds; ++kind) {
        std::vector<double> k(P);
        if (kind == RADON_FILTER_RAM_LAK) {
            k = kpad;   // IDFT(DFT(kernel)) is the kernel itself
        } else {
            std::vector<cd> F(P);
            for (size_t m = 0; m < P; ++m) {
                const double f = (m < P / 2 ? (double)m : (double)m - (double)P) / (double)P;   // fftfreq
                F[m] = cd(H[m].real() * window(kind, f), 0.0);
            }
            fft(F, true);
            for (size_t m = 0; m < P; ++m) k[m] = F[m].real() / (double)P;
        }
        for (long long j = 0; j < n_taps; ++j) {
            const long long m = j - (D - 1);
            const double v = scale * k[(size_t)((m % (long long)P + (long long)P) % (long long)P)];
            const float vh = (float)v;
            taps[(size_t)kind * n_taps + j] = make_float2(vh, (float)(v - (double)vh));
        }
    }
    cudaError_t e = cudaMalloc(&g->d_filter_taps, taps.size() * sizeof(float2));
    if (e != cudaSuccess)
        return e == cudaErrorMemoryAllocation ? fail(RADON_ERR_OOM, "device allocation of filter taps failed")
                                              : cuda_fail(e, "cudaMalloc");
    e = cudaMemcpy(g->d_filter_taps, taps.data(), taps.size() * sizeof(float2), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy filter taps");
    return RADON_OK;
}

}  // namespace radon

using namespace radon;

extern "C" RADON_API radon_status radon_filter_sinogram(const radon_geometry* g, const void* sino, void* out,
                                                        radon_dtype dtype, int batch, radon_filter filter,
                                                        void* stream) {
    radon_status st = validate_call(g, sino, out, dtype, batch);
    if (st != RADON_OK) return st;
    if ((int)filter < 0 || (int)filter >= kFilterKinds) return fail(RADON_ERR_INVALID_ARG, "unknown filter");
    if (g->host_only) return fail(RADON_ERR_INVALID_ARG, "geometry was created host-only; it cannot launch");
    const size_t es = dtype == RADON_F32 ? 4 : 2;
    const long long rows = (long long)batch * g->V;
    const size_t bytes = (size_t)rows * g->D * es;
    const uintptr_t a = (uintptr_t)sino, b = (uintptr_t)out;
    if (batch > 0 && a < b + bytes && b < a + bytes) return fail(RADON_ERR_INVALID_ARG, "out overlaps sino");
    if (batch == 0) return RADON_OK;
    if (filter_long_smem(g->D) > 227 * 1024)
        return fail(RADON_ERR_UNSUPPORTED, "det_count too large for the filter kernel");
    if (rows > 0x7fffffffLL) return fail(RADON_ERR_UNSUPPORTED, "too many sinogram rows");
    st = check_device(g);
    if (st != RADON_OK) return st;
    const float2* taps = g->d_filter_taps + (size_t)filter * (2LL * g->D - 1);
    cudaStream_t s = (cudaStream_t)stream;
    cudaError_t e;
    switch (dtype) {
        case RADON_F16: e = filter_launch<__half>(sino, out, taps, g->D, rows, filter, s); break;
        case RADON_BF16: e = filter_launch<__nv_bfloat16>(sino, out, taps, g->D, rows, filter, s); break;
        default: e = filter_launch<float>(sino, out, taps, g->D, rows, filter, s); break;
    }
    if (e != cudaSuccess) return cuda_fail(e, "filter launch");
    count_launches(1);
    return RADON_OK;
}
