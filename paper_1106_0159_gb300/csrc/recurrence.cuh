// Pieces of the lambda recurrence shared by the FP64, double-float and tensor-core Legendre
// kernels (legendre.cu, legendre_df.cu, legendre_tc.cu): the exponent test of the rescaling
// scheme, the sectoral start value mu_m sin^m(theta) with its binary exponent carried apart
// (eq. pmm with the reading sin^m; rescaling as described in legendre.cu), and the two
// thresholds every kernel must agree on.  Included inside each file's anonymous namespace, so
// every translation unit keeps its own internal copy.
#pragma once

#include <climits>

#include "check.cuh"

constexpr int RESCALE_THR = 1023 + 256;  // biased exponent of y that triggers a rescale by 2^-512
constexpr double POLAR_SIN = 0.03;       // slot blocks starting below this sin(theta) use the Reinsch form

// Marks of the tensor-core synthesis (tc_scale_kernel).  Its terms are off by about 2^-57 of the product
// of two scales: the largest |c a_lm| of the column and the largest |y| of any slot.  reach[m][16] is that
// product's exponent (INT_MAX: the column holds what digits cannot carry), size[m][16] the exponent of the
// largest product c a_lm y_l of one l (tc_top_kernel).  On a grid with rings near the equator the two
// agree within 8 bits whatever the spectrum (lambda grows like sqrt(l) at the pole).  On a polar cap they
// need not: a single mode l = m = 100 is 2^-35 of its scales at theta = 0.9, and its sums kept 22 bits.  A
// column whose reach lies more than 2^MARK_BITS above the largest size of the whole map is left to the
// plain FP64 sums, so that the error stays near 2^(MARK_BITS - 57) of the map's largest terms; columns
// that are nothing beside others need no care.  Ordinary spectra, red, steep or smoothed, mark nothing
// on a cap either (theta <= 0.9 and <= 0.1, lmax 2048, 16 maps: 10.5 and 4.4 ms for each of them).
constexpr int MARK_BITS = 9;

// whether column g of m is marked; NC columns (1, or a spin pair) are judged together.  All threads of the
// block call it with the same arguments and get the same answer.
template <int NC>
__device__ bool synth_marked(const int *__restrict__ reach, const int *__restrict__ size, const int *mflag, int mmax, int m,
                             int g)
{
    __shared__ int s_top;
    int r = reach[m * 16 + g], p = size[m * 16 + g];
    for (int c = 1; c < NC; ++c) {
        r = max(r, reach[m * 16 + g + c]);
        p = max(p, size[m * 16 + g + c]);
    }
    if (r == INT_MAX) return true;
    if (r - p <= MARK_BITS) return false;
    __syncthreads();
    if (threadIdx.x == 0) s_top = 0;
    __syncthreads();
    int top = 0;
    for (int i = threadIdx.x; i <= mmax; i += blockDim.x)
        if (!mflag || mflag[i])
            for (int c = 0; c < NC; ++c) top = max(top, size[i * 16 + g + c]);
    atomicMax(&s_top, top);
    __syncthreads();
    return r - s_top > MARK_BITS;
}

// biased exponent field of v
__device__ __forceinline__ int dexp(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// v in [1, 2) times 2^e  <-  v (positive, normal)
__device__ __forceinline__ void normalise(double &v, int &e)
{
    int hi = __double2hiint(v);
    e += ((hi >> 20) & 0x7ff) - 1023;
    hi = (hi & 0x800fffff) | (1023 << 20);
    v = __hiloint2double(hi, __double2loint(v));
}

__device__ __forceinline__ double pow2i(int e)  // 2^e for -1022 <= e <= 1023
{
    return __hiloint2double((e + 1023) << 20, 0);
}

// lambda_mm = mu_m sin^m(theta) as y0 * 2^(512 k), k <= 0, y0 < 2 mu_m (binary powering of
// sin(theta) with the exponent kept in an int); 0 at the pole for m > 0
__device__ void sectoral_start(double s, double mu, int m, double &y0, int &k)
{
    if (m > 0 && !(s > 1e-300)) {
        y0 = 0.0;
        k = 0;
        return;
    }
    double r = 1.0;
    int er = 0;
    double b = s;
    int eb = 0;
    if (m > 0) normalise(b, eb);
    for (int mm = m; mm; mm >>= 1) {
        if (mm & 1) {
            r *= b;
            er += eb;
            normalise(r, er);
        }
        if (mm > 1) {
            b *= b;
            eb *= 2;
            normalise(b, eb);
        }
    }
    // r * 2^er, r in [1, 2), er <= 0;  k = ceil(er / 512)
    const int kk = (er >= 0) ? 0 : -((-er) >> 9);
    const int rem = er - 512 * kk;  // in (-512, 0]
    y0 = mu * r * pow2i(rem);
    k = kk;
}
