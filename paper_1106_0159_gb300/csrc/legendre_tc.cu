// Legendre synthesis on the tensor cores (eq. DeltaDef): the lambda recurrence
// stays in FP64, the sum over l runs as tcgen05 matrix products on digits.
//
// For one m, the sum Delta_m(r) = sum_l a_lm lambda_lm(r) over a block of 128
// ring slots and up to 16 maps is the matrix product of eq. (matrix_vec):
// [128 slots x l] . [l x 2 maps (re, im)], split by the parity of l - m into
// E (even) and O (odd) so that Delta_N = E + O, Delta_S = E - O.
//
// Both operands are cut into eight base-256 digits (tc_common.cuh), with one
// scale exponent per (m, slot) for y = lambda / c (the measured maximum of |y|
// over all l, once per plan) and one per (m, map column) for c_lm a_lm.  The products of digit pairs with i + j <= 7 are summed by
// tcgen05.mma, one accumulator block per class i + j, so every block adds
// numbers of one scale.  (The tensor core aligns a small addend to the
// accumulator and truncates it, so classes must not share one.)
//
// The sums are exact in FP32 for any operands, by carries (carry_classes below).  A class k >= 1 grows
// by at most k 2^14 per l term (|d_0| <= 64, |d_s| <= 128), so that 146 terms of one parity keep even
// class 7 below 2^24; digits need not look random (on the equator y_l = -y_(l-2), a zonal source there
// makes c_l a_l constant too, and class 5 reached 3.5 times 2^24 at lmax 4096: Delta_0 off by 2e-11).
// So every 9 chunks (144 terms) each class hands the multiple of 256 in its sum to the class above
// and keeps a remainder of at most 128.  Class 0 takes the carries: it stays within half a unit of the
// whole sum, below 2^12 per term while |y| < 2^Ey and |c a| < 2^Ea, which is 2^24 at 4096 terms; from lmax
// 8190 on E_a is one higher for every further 8190 (tc_scale_kernel).
//
// The epilogue adds the classes as integers and rounds once to FP64.  Eight digits
// and not seven: with one scale over all l, the y of a polar block (which
// grows like sqrt(l)) against a red spectrum (which falls like 1 / l) leave the
// low l, where the signal is, several bits below the scale; with seven digits
// (54 bits, classes up to 6) Delta_m was off by twice the plain FP64 sums' error
// (6.6e-14 against 3.1e-14 of its norm, lmax 2048).
//
// Per CTA (one m, 128 slots, 416 threads in three warp groups), per chunk of 32 l:
//   1. the recurrence warps run 32 steps (tc_common.cuh; Reinsch's form in a polar block), one
//      slot per thread, and write the values to a y stage in shared memory;
//   2. the split warps cut each value into digits, store them as the A tiles [parity][digit] of
//      the chunk's stage and copy in the a_lm digit tiles (prepared by tc_split_b_kernel);
//   3. one lane of the issuing warp issues the 2 x 20 MMAs (M = 128, N2 columns, K = 16) and
//      commits them to the stage's mbarrier.
// y values and tiles are double-buffered (16 maps), or a second CTA has the SM meanwhile (up to 8), so
// recurrence runs while a chunk is cut and multiplied.  The B operand stacks two a_lm digits along N: stack b/2 = [B_b | B_(b+1)],
// so one MMA A_a x stack adds class a + b to accumulator block a + b and class a + b + 1 to block
// a + b + 1 (20 MMAs per parity and chunk instead of 36).
//
// Spin 2 (polarisation).  With P+- = sum (E +- iB) lambda+- (spin.cu), Delta^Q = -(P+ + P-) / 2 and
// Delta^U = i (P+ - P-) / 2, and a mirror ring swaps lambda+ and lambda- up to (-1)^(l+m).  So a map's
// pair is two complex columns E + iB, E - iB, and two passes, one per sign of the recurrence, give
// P+- everywhere: the column of the pass's own sign on the northern rings (E + O), the other on the
// southern ones (E - O).  spin_combine_kernel then forms Q and U.  4 FP64 instructions per step and
// ring pair for up to 8 maps, where the FP64 kernels take 6 + 8 per map (lmax 1024, 1 map: whole synthesis
// 20.7 -> 5.19 ms; analysis of 2 maps 32.5 -> 7.64 ms).
//
// What bounds it: the FP64 recurrence, 64 FP64 instructions per warp and chunk = 4096 SM cycles, and the
// other roles' instructions that delay it (about 6.2K cycles a chunk at lmax 4096, 16 maps: 126 ms).
#include "sht_internal.h"

#include <algorithm>

namespace sht {
namespace {

#include "tc_common.cuh"

constexpr int TC_ATILE = TC_T * 16 * 2;      // bytes of one [128 x 16] fp16 tile
constexpr int TC_ESMALL = -900;              // E_a below which a column is cut from scaled values
constexpr size_t TC_SLAB_BYTES = size_t(2) << 30;  // a_lm digits held at a time (whole m)

// N columns (2 per map): 8, 16 or 32; NC CTAs per SM
template <int N, int NC = 1>
struct TcTile {
    static constexpr int N2 = 2 * N;                          // columns of one B stack
    static constexpr int B_TILE = N2 * 16 * 2;                // bytes of one [N2 x 16] stack
    static constexpr int NSTK = TC_S / 2;                     // stacks per parity
    // accumulator blocks per parity: classes 0 .. 7, and where there is room one that takes the second
    // halves of the class-7 stacks (incomplete, not read); else those MMAs take half a stack
    static constexpr int NCLS = N == 8 ? TC_S + 1 : TC_S;
    // Up to 8 maps two CTAs can share an SM (launch_slab), each with one stage of y values and tiles: while one waits for
    // its stage or for tensor memory the other's recurrence has the FP64 pipe, and where both run the
    // pipe is never short of a warp.  16 maps take all of tensor memory: one CTA, two stages.  Whole
    // synthesis, one CTA of two stages against two of one: 18.48 -> 17.02 ms (lmax 2048, 1 map), 1.34 ->
    // 1.25 ms (Gauss-Legendre, lmax 750, 5 maps), 6.33 -> 5.15 ms (spin 2, lmax 1024, 1 map).
    static constexpr int NST = NC == 1 ? 2 : 1;               // stages
    static constexpr int CP = NC == 1 ? 8 : 4;                // columns of one epilogue step
    static constexpr int G = NC == 1 ? 8 : 4;                 // recurrence steps of one group
    static constexpr int B_CHUNK = 2 * NSTK * B_TILE;         // a_lm digits of one chunk
    static constexpr int A_BYTES = 2 * TC_S * TC_ATILE;       // y digits of one chunk
    static constexpr int Y_BYTES = TC_CH * TC_T * 8;          // one stage of y values
    static constexpr int OFF_B = NST * A_BYTES;
    static constexpr int OFF_Y = OFF_B + NST * B_CHUNK;
    static constexpr int OFF_A = OFF_Y + NST * Y_BYTES;         // the recurrence warps' coefficients
    static constexpr int OFF_BAR = OFF_A + TC_ABUF;
    static constexpr int SMEM = OFF_BAR + 64;
    static constexpr int TMEM_COLS = N == 32 ? 512 : 256;     // 2 NCLS N, a power of two
    static_assert(2 * NCLS * N <= TMEM_COLS && NC * TMEM_COLS <= 512, "tensor memory");
    static_assert((NC + 1) * SMEM > 228 * 1024 && NC * (SMEM + 1024) <= 228 * 1024, "NC CTAs per SM, no more");
};

size_t chunk_bytes(int N) { return (size_t)N * 512; }
static_assert(TcTile<8>::B_CHUNK == 8 * 512 && TcTile<32>::B_CHUNK == 32 * 512, "chunk_bytes");

// ---------------------------------------------------------------- a_lm side

// coefficient (l, m) at index ix of column pair g: a_lm of map g, or (spin) E + iB (g even) / E - iB (g
// odd) of polarised map g / 2; imaginary parts at m = 0 are ignored
template <bool SPIN>
__device__ __forceinline__ double2 column_value(const TcArgs &A, int g, int m, int64_t ix)
{
    if (!SPIN) {
        const double2 a = A.alm[(int64_t)g * A.nalm + ix];
        return make_double2(a.x, m == 0 ? 0.0 : a.y);
    }
    double2 e = A.alm[(int64_t)(g & ~1) * A.nalm + ix], b = A.alm[(int64_t)(g | 1) * A.nalm + ix];
    if (m == 0) e.y = b.y = 0.0;
    return (g & 1) ? make_double2(e.x + b.y, e.y - b.x) : make_double2(e.x - b.y, e.y + b.x);
}
template <bool SPIN>
__device__ __forceinline__ double c_factor(const TcArgs &A, int64_t ix)
{
    return SPIN ? A.tab[ix].w : A.cfac[ix];
}

// E_a[m][n] with |c_lm a_lm| < 2^E_a 2^-(lmax / 8190) for all l (from exponent fields, no FP64 work), and
// per map the exponents that decide which columns the digits cannot carry (synth_marked): a value that
// is not finite or a maximum near the upper end of the FP64 range is one of them.  Subnormal values count
// as one of exponent field 1.
template <int N, bool SPIN>
__global__ void tc_scale_kernel(TcArgs A)
{
    __shared__ int s_max[N], s_size[N / 2], s_y;
    __shared__ int s_fix[N / 2];
    const int m = A.m0 + blockIdx.x;
    if (A.mflag && !A.mflag[m]) return;  // an m this plan does not compute: nothing reads its digits
    const int L = A.lmax;
    const int64_t base = (int64_t)m * (2 * L + 3 - m) / 2;
    if (threadIdx.x < N) s_max[threadIdx.x] = 0;
    if (threadIdx.x < N / 2) s_fix[threadIdx.x] = s_size[threadIdx.x] = 0;
    if (threadIdx.x == 0) s_y = 0;
    __syncthreads();
    int mx[N], sz[N / 2];
    unsigned bad = 0;  // maps with a non-finite value
#pragma unroll
    for (int g = 0; g < N / 2; ++g) sz[g] = 0;
#pragma unroll
    for (int n = 0; n < N; ++n) mx[n] = 0;
    for (int l = first_l<SPIN ? REC_SPIN : REC_Y>(m) + threadIdx.x; l <= L; l += blockDim.x) {
        const int64_t ix = base + (l - m);
        const int ec = dexp(c_factor<SPIN>(A, ix)), ey = A.Yl[ix];
#pragma unroll
        for (int g = 0; g < N / 2; ++g) {
            if (g < A.nmaps) {
                const double2 a = column_value<SPIN>(A, g, m, ix);
                const int er = dexp_nonzero(a.x), ei = dexp_nonzero(a.y);
                if (er == 0x7ff || ei == 0x7ff) bad |= 1u << g;
                if (er) mx[2 * g] = max(mx[2 * g], er + ec);
                if (ei) mx[2 * g + 1] = max(mx[2 * g + 1], ei + ec);
                if (ey && (er | ei)) sz[g] = max(sz[g], max(er, ei) + ec + ey);
            }
        }
    }
#pragma unroll
    for (int n = 0; n < N; ++n) {
        const int w = (int)__reduce_max_sync(0xffffffffu, (unsigned)mx[n]);
        if ((threadIdx.x & 31) == 0) atomicMax(&s_max[n], w);
    }
#pragma unroll
    for (int g = 0; g < N / 2; ++g) {
        const int w = (int)__reduce_max_sync(0xffffffffu, (unsigned)sz[g]);
        if ((threadIdx.x & 31) == 0 && w) atomicMax(&s_size[g], w);
    }
    for (int pass = 0; pass < (SPIN ? 2 : 1); ++pass)  // the largest |y| of any slot (spin: of both signs)
        for (int b = threadIdx.x; b < A.nblk; b += blockDim.x)
            atomicMax(&s_y, A.Ey[(int64_t)pass * 2 * (A.mmax + 1) * A.nblk + m * A.nblk + b] + 1022);
    bad = __reduce_or_sync(0xffffffffu, bad);
    if ((threadIdx.x & 31) == 0)
        for (int g = 0; g < N / 2; ++g)
            if (bad >> g & 1) s_fix[g] = 1;
    __syncthreads();
    if (threadIdx.x < N) {
        const int e = s_max[threadIdx.x];
        // L / 8190 more: |d_0| halves where a parity has over 4096 terms, so that class 0 stays below 2^24
        A.Ea[m * N + threadIdx.x] = e ? e - 2044 + L / 8190 : TC_EZERO;
        if (e > 1023 + TC_EHUGE) s_fix[threadIdx.x >> 1] = 1;
    }
    __syncthreads();
    if (threadIdx.x < N / 2 && (int)threadIdx.x < A.nmaps) {
        const int g = threadIdx.x, e = max(s_max[2 * g], s_max[2 * g + 1]);
        A.reach[m * 16 + g] = s_fix[g] ? INT_MAX : e ? e + s_y : 0;
        A.size[m * 16 + g] = s_size[g];
    }
}

// digits of c_lm a_lm for one (m, chunk) in the tile layout of the MMA B operand:
// [parity][stack][N2 x 16] fp16 with digit s in stack s / 2 at columns n + N (s & 1), core matrix
// (n2/8, k/8) at ((k/8) (N2/8) + n2/8) * 64 elements.  Thread (parity, k/8, n)
// cuts the 8 values k/8 .. k/8 + 7 of its column: each digit's 8 values are one core-matrix row,
// 16 contiguous bytes, stored as one vector.
//
// A column below 2^TC_ESMALL is cut from its values times 2^512, so that subnormal ones are cut exactly; in
// other columns their digits are 0, an error below 2^-99 of the scale.  Coefficients smoothed by a
// Gaussian beam run through the subnormal range where l sigma > 37.6, in every m of a band-limited set: left
// to the plain sums, columns with a subnormal value took 3132 ms for 158 (lmax 4096, 16 maps, FWHM 2
// degrees), and those with a maximum below 2^-923 alone 492.
template <int N, bool SPIN>
__global__ void tc_split_b_kernel(TcArgs A)
{
    const int64_t chunk = A.chunk0 + blockIdx.x;
    const int m = A.chunk_m[chunk];
    if (A.mflag && !A.mflag[m]) return;
    const int c = (int)(chunk - A.chunk_base[m]);
    const int L = A.lmax;
    const int64_t base = (int64_t)m * (2 * L + 3 - m) / 2;
    constexpr int N2 = TcTile<N>::N2;
    uint4 *out = A.bdig + (int64_t)blockIdx.x * (TcTile<N>::B_CHUNK / 16);
    const int t = threadIdx.x;  // 4 N threads
    const int n = t % N, kh = (t / N) & 1, eo = t / (2 * N);
    const int g = n >> 1;
    const int Ea = A.Ea[m * N + n];
    const bool small = Ea < TC_ESMALL;
    const int E = small ? Ea + 512 : Ea;
    uint32_t pk[4][TC_S];  // pairs of the 8 values, per digit
#pragma unroll
    for (int kk = 0; kk < 8; kk += 2) {
        uint2 f[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int l = first_l<SPIN ? REC_SPIN : REC_Y>(m) + TC_CH * c + 2 * (8 * kh + kk + h) + eo;
            double v = 0.0;
            if (l <= L && g < A.nmaps) {
                const int64_t ix = base + (l - m);
                const double2 a = column_value<SPIN>(A, g, m, ix);
                v = (n & 1) ? a.y : a.x;
                if (small) v *= 0x1p512;
                v *= c_factor<SPIN>(A, ix);
            }
            f[h] = digit_fields(v, E);
        }
        digit_pairs(f[0], f[1], pk[kk >> 1]);
    }
#pragma unroll
    for (int s = 0; s < TC_S; ++s) {
        const int n2 = n + N * (s & 1);
        const int off = (kh * (N2 / 8) + (n2 >> 3)) * 64 + (n2 & 7) * 8;  // elements; a multiple of 8
        out[((eo * TcTile<N>::NSTK + (s >> 1)) * (N2 * 16) + off) / 8] = make_uint4(pk[0][s], pk[1][s], pk[2][s], pk[3][s]);
    }
}

// ---------------------------------------------------------------- plan tables

// Per (m, slot block): E with |y| < 2^E over the kept values of the block's slots and all l (-1000
// when every value is dropped), how far each slot's own exponent lies below it, the first chunk of
// 32 l in which any slot keeps a value (every earlier chunk contributes exactly zero), and the
// recurrence state (y1, y2, k) of every slot at the start of that chunk, where the tensor-core kernels
// begin (at lmax 4096 on HEALPix about a quarter of the steps lie before it).  Same recurrence, operation
// for operation, as recurrence_warps, so that both see the same rescaling steps and the same values.

// lambda of the first l at one slot, y0 2^(512 k)
template <int KIND>
__device__ __forceinline__ void slot_start(const TcArgs &A, int m, int64_t base, int slot, double u, double &y0, int &k)
{
    if (KIND == REC_SPIN) {  // S_m sin^|m-2| times sin^p(theta/2) (+) or sigma cos^p(theta/2) (-): spin.cu
        sectoral_start(A.s[slot], A.start[m], m >= 2 ? m - 2 : 2 - m, y0, k);
        const double f = A.sig > 0 ? 0.5 * u : 1.0 - 0.5 * u;
        y0 *= m >= 2 ? f * f : m == 1 ? (A.sig > 0 ? f : -f) : 1.0;
    } else {
        sectoral_start(A.s[slot], A.alpha[base], m, y0, k);
    }
}

template <int KIND>
__device__ __forceinline__ void tables_body(const TcArgs &A, int m, int blk, int *s_max, int *s_first, RecCoef *s_c,
                                            double2 *ck_y, int *ck_k)
{
    const int tid = threadIdx.x;
    const int slot = blk * TC_T + tid;
    const bool active = slot < A.nslots;
    const int L = A.lmax;
    const int64_t base = (int64_t)m * (2 * L + 3 - m) / 2;
    const int lb = first_l<KIND>(m);
    const int nch = (L - lb + TC_CH) / TC_CH;
    const int64_t ci = (int64_t)(m * A.nblk + blk) * TC_T + tid;
    double u = 0.0, y1 = 0.0, y2 = 0.0;
    int k = 0;
    if (active) {
        u = A.u[slot];
        double y0;
        slot_start<KIND>(A, m, base, slot, u, y0, k);
        y2 = KIND == REC_REIN ? y0 : -y0;
    }
    double c1 = y1, c2 = y2;  // state at the start of the first live chunk
    int ckk = k, mx = 0;
    for (int c = 0; c < nch; ++c) {
        const int l0 = lb + TC_CH * c;
        __syncthreads();
        if (tid < TC_CH) s_c[tid] = load_coef<KIND>(A, base, m, l0 + tid);
        const bool dead = *s_first >= c;  // no value kept in the chunks before c
        __syncthreads();
        if (dead) {
            c1 = y1;
            c2 = y2;
            ckk = k;
        }
        bool live = false;
#pragma unroll 1
        for (int h = 0; h < 2; ++h) {
            const bool scaled = __any_sync(0xffffffffu, k < 0);
            const bool drop = scaled && k < 0;
            for (int j = 16 * h; j < 16 * h + 16; ++j) {
                const RecCoef C = s_c[j];
                double y;
                if (KIND == REC_REIN) {
                    y = rein_step(C.a, C.rh, C.b0, C.ci, u, y1, y2);
                } else {
                    y = fma(fma(-C.a, u, KIND == REC_SPIN ? C.rh : C.a), y1, -y2);
                    y2 = y1;
                    y1 = y;
                }
                if (l0 + j <= L && !drop) {
                    mx = max(mx, dexp(y));
                    live = true;
                }
            }
            if (drop && max(dexp(y1), dexp(y2)) > RESCALE_THR) {
                y1 *= 0x1p-512;
                y2 *= 0x1p-512;
                k += 1;
            }
        }
        if (active && live && dead) atomicMin(s_first, c);
    }
    atomicMax(s_max, active ? mx : 0);
    __syncthreads();
    ck_y[ci] = make_double2(c1, c2);
    ck_k[ci] = slot_state(ckk, min(*s_max - mx, 255));
}

template <bool SPIN>
__global__ void __launch_bounds__(TC_T) tc_tables_kernel(TcArgs A, int *Ey_out, int *first_out, double2 *ck_y, int *ck_k)
{
    __shared__ RecCoef s_c[TC_CH];
    __shared__ int s_max, s_first;
    const int m = blockIdx.x / A.nblk;
    const int blk = blockIdx.x - m * A.nblk;
    if (threadIdx.x == 0) {
        s_max = 0;
        s_first = (A.lmax - first_l<SPIN ? REC_SPIN : REC_Y>(m) + TC_CH) / TC_CH;
    }
    __syncthreads();
    if (SPIN)
        tables_body<REC_SPIN>(A, m, blk, &s_max, &s_first, s_c, ck_y, ck_k);
    else if (polar_block(A, m, blk))
        tables_body<REC_REIN>(A, m, blk, &s_max, &s_first, s_c, ck_y, ck_k);
    else
        tables_body<REC_Y>(A, m, blk, &s_max, &s_first, s_c, ck_y, ck_k);
    __syncthreads();
    if (threadIdx.x == 0) {
        Ey_out[m * A.nblk + blk] = s_max ? s_max - 1022 : -1000;
        first_out[m * A.nblk + blk] = s_first;
    }
}

// Exponent field of the largest kept |y_l| per (m, l) of up to 128 slots spread evenly over the grid, the
// most equatorward one among them; 0 where all are dropped (spin: of both signs of the recurrence).  One
// CTA per m, the y form or spin's recurrence: only exponents count.  2 bytes per coefficient.
template <bool SPIN>
__global__ void __launch_bounds__(TC_T) tc_top_kernel(TcArgs A, uint16_t *__restrict__ Yl)
{
    constexpr int KIND = SPIN ? REC_SPIN : REC_Y;
    __shared__ RecCoef s_c[TC_CH];
    __shared__ int s_m[TC_CH];
    const int m = blockIdx.x, tid = threadIdx.x;
    const bool active = tid < A.nslots;
    const int slot = A.nslots <= TC_T ? tid : A.nslots - 1 - (int)((int64_t)tid * (A.nslots - 1) / (TC_T - 1));
    const int L = A.lmax, lb = first_l<KIND>(m);
    const int64_t base = (int64_t)m * (2 * L + 3 - m) / 2;
    for (int l = m + tid; l < min(lb, L + 1); l += TC_T) Yl[base + l - m] = 0;
    for (int pass = 0; pass < (SPIN ? 2 : 1); ++pass) {
        A.sig = pass == 0 ? 1 : -1;
        double u = 0.0, y1 = 0.0, y2 = 0.0;
        int k = 0;
        if (active) {
            u = A.u[slot];
            double y0;
            slot_start<KIND>(A, m, base, slot, u, y0, k);
            y2 = -y0;
        }
        for (int l0 = lb; l0 <= L; l0 += TC_CH) {
            __syncthreads();
            if (tid < TC_CH) {
                s_c[tid] = load_coef<KIND>(A, base, m, l0 + tid);
                s_m[tid] = 0;
            }
            __syncthreads();
            for (int h = 0; h < 2; ++h) {
                const bool scaled = __any_sync(0xffffffffu, k < 0);
                const bool drop = scaled && k < 0;
                for (int j = 16 * h; j < 16 * h + 16; ++j) {
                    const RecCoef C = s_c[j];
                    const double y = fma(fma(-C.a, u, KIND == REC_SPIN ? C.rh : C.a), y1, -y2);
                    y2 = y1;
                    y1 = y;
                    const unsigned e = __reduce_max_sync(0xffffffffu, (unsigned)(drop || !active ? 0 : dexp(y)));
                    if ((tid & 31) == 0) atomicMax(&s_m[j], (int)e);
                }
                if (drop && max(dexp(y1), dexp(y2)) > RESCALE_THR) {
                    y1 *= 0x1p-512;
                    y2 *= 0x1p-512;
                    k += 1;
                }
            }
            __syncthreads();
            if (tid < TC_CH && l0 + tid <= L) {
                uint16_t *o = Yl + base + (l0 - m) + tid;
                *o = (uint16_t)(pass == 0 ? s_m[tid] : max((int)*o, s_m[tid]));
            }
        }
    }
}

// ---------------------------------------------------------------- the synthesis kernel

// Chunks between two carries: 9 x 16 terms of one parity, 144 x 7 x 2^14 + 128 < 2^24.
constexpr int TC_CARRY = 9;
static_assert(TC_CARRY * (TC_CH / 2) * (TC_S - 1) * (1 << 14) + 128 < (1 << 24), "class sums exact in FP32");

// two FP32 operations in one instruction (they delay the FP64 chain half as often)
__device__ __forceinline__ uint64_t f32x2(float x) { return 0x100000001ull * __float_as_uint(x); }
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b)
{
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c)
{
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}

// Carries between the accumulator blocks of one parity (8 blocks of N columns, the first at `acc`; this
// warp's 32 lanes), columns below ncols: from class 7 up, a sum S = 256 q + r with |r| <= 128 keeps r and q
// moves to the class above.  An accumulator holds S 2^-18, so q is rounded by an addition at ulp 2^-18;
// every step is exact.  No MMA may be in flight.  What it costs are its issue slots beside the recurrence:
// whole synthesis at lmax 4096, 16 maps 157.4 -> 158.6 ms, with plain FP32 operations 162.5, and with 4
// columns after every chunk instead of all of them after 9 no less (162.7).
template <int N>
__device__ __forceinline__ void carry_classes(uint32_t acc, int ncols)
{
#pragma unroll 1
    for (int c = 0; c < N && c < ncols; c += 4) {
        uint32_t v[TC_S][4];
#pragma unroll
        for (int k = 0; k < TC_S; ++k)
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                         : "=r"(v[k][0]), "=r"(v[k][1]), "=r"(v[k][2]), "=r"(v[k][3])
                         : "r"(acc + (uint32_t)(k * N + c)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int t = 0; t < 4; t += 2) {
            uint64_t up = 0;
#pragma unroll
            for (int k = TC_S - 1; k >= 0; --k) {
                uint64_t x = add2((uint64_t)v[k][t + 1] << 32 | v[k][t], up);
                if (k) {
                    up = add2(fma2(x, f32x2(0x1p-8f), f32x2(48.f)), f32x2(-48.f));  // |x| < 2^6: 48 + x / 256 has ulp 2^-18
                    x = fma2(up, f32x2(-256.f), x);
                }
                v[k][t] = (uint32_t)x;
                v[k][t + 1] = (uint32_t)(x >> 32);
            }
        }
#pragma unroll
        for (int k = 0; k < TC_S; ++k)
            asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(acc + (uint32_t)(k * N + c)),
                         "r"(v[k][0]), "r"(v[k][1]), "r"(v[k][2]), "r"(v[k][3])
                         : "memory");
    }
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// Warp groups per CTA (one m, 128 slots, 416 threads):
//   recurrence warps 0-3 (recurrence_warps): thread r runs the FP64 recurrence of slot r and
//     writes each chunk's 32 values to one of NST y stages in shared memory;
//   split warps 4-11: thread (par, r) cuts the 16 values of parity par of slot r into digits and
//     stores row r of the parity's A tiles (NST sets); all of them copy the chunk's a_lm
//     digit tiles and arrive on the stage's full mbarrier; at the end they read tensor memory,
//     warps 4-7 the even groups of CP columns and warps 8-11 the odd ones;
//   warp 12: waits on the full mbarrier, and one elected lane issues the chunk's MMAs
//     (warp-uniform descriptors) and commits them to the stage's done mbarrier.
// Stages: the y buffer is handed over with named barriers (FULL: recurrence arrives, split
// waits; EMPTY: split arrives, recurrence waits, only where a later chunk reuses the stage);
// the A/B tiles of a stage are rewritten after the done mbarrier of the MMAs that read them.
template <int N, int NC, bool SPIN>
__global__ void __launch_bounds__(TC_NT + 32, NC) tc_synth_kernel(TcArgs A)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    using W = TcTile<N, NC>;
    unsigned char *sA = smem;                               // [stage][parity][digit][128 x 16] fp16
    unsigned char *sB = smem + W::OFF_B;                    // [stage][parity][stack][N2 x 16] fp16
    double *ybuf = (double *)(smem + W::OFF_Y);             // [stage][32 l][128 slots]
    double *abuf = (double *)(smem + W::OFF_A);             // [recurrence warp][32 l]
    uint64_t *mbar = (uint64_t *)(smem + W::OFF_BAR);       // done[stage]: the stage's MMAs complete
    uint64_t *full = mbar + 2;                              // full[stage]: the stage's tiles written
    uint32_t *tslot = (uint32_t *)(mbar + 4);

    const int m = A.m0 + (int)(blockIdx.x / A.nblk);
    const int blk = (int)(blockIdx.x % A.nblk);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool rec = warp < 4, issuer = warp == TC_NT / 32;
    const int sp = tid - TC_T;                              // split-thread index 0..255
    const int r = rec ? tid : (sp & (TC_T - 1));            // slot within the block
    const int par = rec ? 0 : (sp >> 7);                    // split threads: parity of l - m they cut
    const int slot = blk * TC_T + r;
    const bool active = slot < A.nslots;
    const int L = A.lmax;
    const int64_t base = (int64_t)m * (2 * L + 3 - m) / 2;
    const int nch = (L - first_l<SPIN ? REC_SPIN : REC_Y>(m) + TC_CH) / TC_CH;
    const int cfirst = A.first[m * A.nblk + blk];           // chunks before it hold only dropped values
    const int nlive = nch - cfirst;

    if (nlive <= 0 || (A.mflag && !A.mflag[m])) {  // every value dropped, or an m this plan does not compute: zeros
        if (!rec && !issuer && par == 0 && active) {
            const int rn = A.slotN[slot], rs = A.slotS[slot];
            const int64_t mstride = A.mmax + 1;
            for (int g = 0; g < A.nmaps; ++g) {
                double2 *d = A.delta + (int64_t)g * A.nrings * mstride;
                const bool own = !SPIN || ((g & 1) == 0) == (A.sig > 0);  // spin: see the epilogue
                if (own && rn >= 0 && SHT_CHK(rn < A.nrings)) d[(int64_t)rn * mstride + m] = make_double2(0.0, 0.0);
                if ((!SPIN || !own) && rs >= 0 && SHT_CHK(rs < A.nrings))
                    d[(int64_t)rs * mstride + m] = make_double2(0.0, 0.0);
            }
        }
        return;
    }

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)),
                     "r"(W::TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&mbar[i], 1);              // commit
            mbar_init(&full[i], TC_NT - TC_T);   // split threads
        }
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tslot;

    bool ok = true;
    if (rec) {
        if (SPIN)
            recurrence_warps<REC_SPIN, false, TC_T, W::G, W::NST>(A, m, blk, r, active, base, nch, cfirst, ybuf, abuf);
        else if (polar_block(A, m, blk))
            recurrence_warps<REC_REIN, false, TC_T, W::G, W::NST>(A, m, blk, r, active, base, nch, cfirst, ybuf, abuf);
        else
            recurrence_warps<REC_Y, false, TC_T, W::G, W::NST>(A, m, blk, r, active, base, nch, cfirst, ybuf, abuf);
    } else if (issuer) {
        // ------------------------------------------------ MMA issue (one lane of the last warp)
        // per chunk: wait until the stage's tiles are written, issue its 2 x 20 MMAs (per parity eo,
        // A digit a against B stack b/2 for a + b <= 7) and commit them to the stage's done barrier
        const uint32_t idesc2 = umma_idesc<W::N2>(), idesc1 = umma_idesc<W::NCLS == TC_S ? N : W::N2>();
        const uint64_t dA0 = umma_desc(smem_u32(sA), 16 * 128, 128);
        const uint64_t dB0 = umma_desc(smem_u32(sB), (W::N2 / 8) * 128, 128);
        const uint32_t issue = elect_one();
        for (int q = 0; q < nlive; ++q) {
            const int st = q & (W::NST - 1);
            if (ok && !mbar_wait(&full[st], (uint32_t)((q >> (W::NST - 1)) & 1))) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint64_t aS = dA0 + (uint64_t)((st * W::A_BYTES) >> 4);  // address field: bytes / 16
            const uint64_t bS = dB0 + (uint64_t)((st * W::B_CHUNK) >> 4);
#pragma unroll
            for (int eo = 0; eo < 2; ++eo) {
#pragma unroll
                for (int a = 0; a < TC_S; ++a) {
#pragma unroll
                    for (int b = 0; b + a < TC_S; b += 2) {
                        // the a = 0 MMAs of the first live chunk write blocks 0-7 once each: they start the sums
                        const bool first = (q == 0) && (a == 0);
                        umma_f16_by(issue, tmem + (uint32_t)((eo * W::NCLS + a + b) * N),
                                    aS + (uint64_t)(((eo * TC_S + a) * TC_ATILE) >> 4),
                                    bS + (uint64_t)(((eo * W::NSTK + b / 2) * W::B_TILE) >> 4),
                                    a + b == TC_S - 1 ? idesc1 : idesc2, first ? 0u : 1u);
                    }
                }
            }
            umma_commit_by(issue, &mbar[st]);
        }
        if (lane == 0 && !ok) atomicOr(A.status, 1);
    } else {
        // ------------------------------------------------ split group
        const int64_t chunk0 = A.chunk_base[m] - A.chunk0;
        const int Ey = A.Ey[m * A.nblk + blk] - state_d(A.ck_k[(int64_t)(m * A.nblk + blk) * TC_T + r]);  // of this slot
        constexpr int NS = TC_NT - TC_T;                 // split threads
        constexpr int BTOT = W::B_CHUNK / 16;            // uint4 of one chunk's B tiles
        constexpr int BV = (BTOT + NS - 1) / NS;
        for (int q = 0; q < nlive; ++q) {
            const int st = q & (W::NST - 1);
            unsigned char *a_st = sA + st * W::A_BYTES;
            unsigned char *b_st = sB + st * W::B_CHUNK;
            uint4 breg[BV];
            const uint4 *bsrc = A.bdig + (chunk0 + cfirst + q) * BTOT;
#pragma unroll
            for (int i = 0; i < BV; ++i)
                if (i * NS + sp < BTOT) breg[i] = bsrc[i * NS + sp];
            bar_sync(BAR_FULL + st, TC_NT);  // y of chunk q is in its stage
            const double *yb = ybuf + (size_t)st * TC_CH * TC_T;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                uint32_t pk[4][TC_S];  // pairs of the 8 values, per digit
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const uint2 f0 = digit_fields(yb[(16 * h + 4 * p + par) * TC_T + r], Ey);
                    const uint2 f1 = digit_fields(yb[(16 * h + 4 * p + 2 + par) * TC_T + r], Ey);
                    digit_pairs(f0, f1, pk[p]);
                }
                if (h == 1 && q + W::NST < nlive) bar_arrive(BAR_EMPTY + st, TC_NT);  // y stage read
                // the MMAs of chunk q - NST read this stage's tiles: wait (bounded) before rewriting them
                // (after the first half is cut, which only reads the y stage)
                if (h == 0 && q >= W::NST && ok && !mbar_wait(&mbar[st], (uint32_t)(((q >> (W::NST - 1)) - 1) & 1))) ok = false;
                // k-group h of this parity's A tiles: core matrix (slot/8, h), row slot%8
                const int off = ((h * 16) + (r >> 3)) * 128 + (r & 7) * 16;
#pragma unroll
                for (int s = 0; s < TC_S; ++s)
                    *(uint4 *)(a_st + (par * TC_S + s) * TC_ATILE + off) =
                        make_uint4(pk[0][s], pk[1][s], pk[2][s], pk[3][s]);
            }
#pragma unroll
            for (int i = 0; i < BV; ++i)
                if (i * NS + sp < BTOT) ((uint4 *)b_st)[i * NS + sp] = breg[i];
            asm volatile("fence.proxy.async.shared::cta;");
            if (q && q % TC_CARRY == 0) {
                // carries of this parity, between the MMAs of chunk q - 1 (one stage: waited for above) and those
                // of chunk q, which start once every split thread has arrived
                if (W::NST == 2 && ok && !mbar_wait(&mbar[st ^ 1], (uint32_t)(((q - 1) >> 1) & 1))) ok = false;
                ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld and st are warp-wide
                asm volatile("tcgen05.fence::after_thread_sync;");
                if (ok) carry_classes<N>(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(par * W::NCLS * N), 2 * A.nmaps);
                asm volatile("tcgen05.fence::before_thread_sync;");
            }
            mbar_arrive(&full[st]);
        }
        // the last commits cover every MMA issued: wait (bounded) before TMEM is read
        if (ok && !mbar_wait(&mbar[(nlive - 1) & (W::NST - 1)], (uint32_t)(((nlive - 1) >> (W::NST - 1)) & 1))) ok = false;
        ok = bar_red_and(BAR_SPLIT, NS, ok);
        asm volatile("tcgen05.fence::after_thread_sync;");
        if (ok) {
            // accumulators: column (eo * NCLS + class) * N + n, lane = slot within the block.  Per column the
            // class sums are integers: classes 0-3 add up to hi, 4-7 to lo (units of class 3 and class 7),
            // Delta_N = E + O and Delta_S = E - O are formed on them and rounded once to FP64, all on the
            // integer pipe: the FP64 pipe of this SM has no other CTA's work to do meanwhile.
            constexpr int CP = W::CP;
            const int lw = warp & 3;  // this warp may read lanes 32 lw .. 32 lw + 31
            const int rn = active ? A.slotN[slot] : -1, rs = active ? A.slotS[slot] : -1;
            const int64_t mstride = A.mmax + 1;
#pragma unroll 1
            for (int cg = par; cg < N / CP; cg += 2) {  // CP columns: CP / 2 maps
                if (CP / 2 * cg >= A.nmaps) break;
                long long hi[2][CP], lo[2][CP];
#pragma unroll
                for (int eo = 0; eo < 2; ++eo) {
                    uint32_t v[TC_S][CP];
#pragma unroll
                    for (int cls = 0; cls < TC_S; ++cls) {
                        const uint32_t addr =
                            tmem + ((uint32_t)(lw * 32) << 16) + (uint32_t)((eo * W::NCLS + cls) * N + CP * cg);
                        if constexpr (CP == 8)
                            asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                                         : "=r"(v[cls][0]), "=r"(v[cls][1]), "=r"(v[cls][2]), "=r"(v[cls][3]),
                                           "=r"(v[cls][4]), "=r"(v[cls][5]), "=r"(v[cls][6]), "=r"(v[cls][7])
                                         : "r"(addr));
                        else
                            asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                                         : "=r"(v[cls][0]), "=r"(v[cls][1]), "=r"(v[cls][2]), "=r"(v[cls][3])
                                         : "r"(addr));
                    }
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
                    for (int t = 0; t < CP; ++t) {
                        long long h = class_sum(__uint_as_float(v[0][t]));
                        h = h * 256 + class_sum(__uint_as_float(v[1][t]));
                        h = h * 256 + class_sum(__uint_as_float(v[2][t]));
                        hi[eo][t] = h * 256 + class_sum(__uint_as_float(v[3][t]));
                        h = class_sum(__uint_as_float(v[4][t]));
                        h = h * 256 + class_sum(__uint_as_float(v[5][t]));
                        h = h * 256 + class_sum(__uint_as_float(v[6][t]));
                        lo[eo][t] = h * 256 + class_sum(__uint_as_float(v[7][t]));
                    }
                }
#pragma unroll
                for (int gg = 0; gg < CP / 2; ++gg) {
                    const int g = CP / 2 * cg + gg;  // map
                    if (g >= A.nmaps) break;
                    const bool own = !SPIN || ((g & 1) == 0) == (A.sig > 0);
                    double vn[2], vs[2];
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const int t = 2 * gg + c;
                        const int e = Ey + A.Ea[m * N + CP * cg + t] - 36;  // class 3: 2^(-6 - 6 - 24)
                        if (own) vn[c] = pair_to_double(hi[0][t] + hi[1][t], lo[0][t] + lo[1][t], e);
                        if (!SPIN || !own) vs[c] = pair_to_double(hi[0][t] - hi[1][t], lo[0][t] - lo[1][t], e);
                    }
                    // spin: l - m starts odd at m = 1, where (-1)^(l+m) and with it E - O change sign
                    if (SPIN && m == 1 && !own) {
                        vs[0] = -vs[0];
                        vs[1] = -vs[1];
                    }
                    double2 *d = A.delta + (int64_t)g * A.nrings * mstride;
                    if (own && rn >= 0 && SHT_CHK(rn < A.nrings && m <= A.mmax))
                        d[(int64_t)rn * mstride + m] = make_double2(vn[0], vn[1]);
                    if ((!SPIN || !own) && rs >= 0 && SHT_CHK(rs < A.nrings && m <= A.mmax))
                        d[(int64_t)rs * mstride + m] = make_double2(vs[0], vs[1]);
                }
            }
        } else if (sp == 0) {
            atomicOr(A.status, 1);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(W::TMEM_COLS));
}

// Q and U from P+ and P- (see above), in place: [nmaps][2] planes of n values
__global__ void spin_combine_kernel(double2 *__restrict__ delta, int64_t n, int nmaps)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n * nmaps; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = t / n, i = t - g * n;
        double2 *q = delta + 2 * g * n + i, *u = q + n;
        const double2 p = *q, w = *u;
        *q = make_double2(-0.5 * (p.x + w.x), -0.5 * (p.y + w.y));
        *u = make_double2(-0.5 * (p.y - w.y), 0.5 * (p.x - w.x));
    }
}

template <int N, int NC>
cudaError_t set_synth_smem(cudaFuncAttribute a)
{
    cudaError_t e = cudaFuncSetAttribute(tc_synth_kernel<N, NC, false>, a, TcTile<N, NC>::SMEM);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(tc_synth_kernel<N, NC, true>, a, TcTile<N, NC>::SMEM);
}

template <int N, bool SPIN>
cudaError_t launch_slab(const Plan &p, const TcArgs &A, int count_m, int64_t nchunks, cudaStream_t st)
{
    constexpr int NC2 = N == 32 ? 1 : 2;
    const unsigned ctas = (unsigned)(count_m * A.nblk);
    // Two CTAs per SM once there are enough of them.  With few, the time is that of the longest chain, a polar
    // block's Reinsch steps at low m, and a lone CTA with two stages runs it faster.  One map, one against two,
    // us: 386 CTAs (lmax 192) 73 / 92, 514 (256) 100 / 116, 963 (320) 174 / 149, 6152 (768) 1242 / 1085.  The
    // spin recurrence has no such blocks, whole synthesis: 193 CTAs 108 / 113, 386 158 / 133, 514 223 / 193.
    const bool two = NC2 == 2 && ctas >= (SPIN ? 2u : 5u) * 152u;
    tc_scale_kernel<N, SPIN><<<count_m, 256, 0, st>>>(A);
    tc_split_b_kernel<N, SPIN><<<(unsigned)nchunks, 4 * N, 0, st>>>(A);  // one thread per (parity, k half, column)
    if (!SPIN) {
        StageEvents ev(p, SHT_STAGE_TC_SYNTH_KERNEL, st);
        if (two)
            tc_synth_kernel<N, NC2, false><<<ctas, TC_NT + 32, TcTile<N, NC2>::SMEM, st>>>(A);
        else
            tc_synth_kernel<N, 1, false><<<ctas, TC_NT + 32, TcTile<N>::SMEM, st>>>(A);
        p.launches[SHT_STAGE_TC_SYNTH_KERNEL] += 1;
        ev.done();
    } else {  // both signs of the recurrence on the same columns
        const size_t tables = (size_t)(p.mmax + 1) * A.nblk;
        TcArgs B = A;
        for (int sig = 1; sig >= -1; sig -= 2) {
            B.sig = sig;
            if (two)
                tc_synth_kernel<N, NC2, true><<<ctas, TC_NT + 32, TcTile<N, NC2>::SMEM, st>>>(B);
            else
                tc_synth_kernel<N, 1, true><<<ctas, TC_NT + 32, TcTile<N>::SMEM, st>>>(B);
            B.Ey += 2 * tables;
            B.first += 2 * tables;
            B.ck_y += tables * TC_T;
            B.ck_k += tables * TC_T;
        }
    }
    return cudaGetLastError();
}

}  // namespace

int64_t tc_chunks_below(const Plan &p, int m)
{
    const int64_t L = p.lmax;
    // sum over m' < m of floor((L - m' + 32) / 32): with x = L - m', sum of floor(x / 32) + 1
    auto S = [](int64_t x) {  // sum over 0 <= t <= x of floor(t / 32), x >= -1
        const int64_t q = (x + 1) / 32, r = (x + 1) % 32;
        return 16 * q * (q - 1) + q * r;
    };
    return S(L) - S(L - m) + m;
}

namespace {

// columns of a group of n maps
int group_columns(int n) { return n > 8 ? 32 : n > 4 ? 16 : 8; }

// end of the slab of whole m that starts at m0 and whose digits fit `cap` bytes (at least one m)
int slab_end(const Plan &p, int m0, int N, size_t cap)
{
    int lo = m0 + 1, hi = p.mmax + 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) / 2;
        if ((size_t)(tc_chunks_below(p, mid) - tc_chunks_below(p, m0)) * chunk_bytes(N) <= cap)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

size_t exponent_bytes(const Plan &p) { return (size_t)(p.mmax + 1) * (32 + 2 * 16) * sizeof(int); }

}  // namespace

cudaError_t configure_tc_kernels()
{
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = set_synth_smem<32, 1>(a);
    if (e == cudaSuccess) e = set_synth_smem<16, 1>(a);
    if (e == cudaSuccess) e = set_synth_smem<16, 2>(a);
    if (e == cudaSuccess) e = set_synth_smem<8, 1>(a);
    if (e == cudaSuccess) e = set_synth_smem<8, 2>(a);
    if (e == cudaSuccess) e = configure_tc_anal_kernel();
    return e;
}

// Plan tables of the tensor-core kernels (synchronous, once per plan); spin: for both signs, + first.
static cudaError_t build_tables(const Plan &p, bool spin, int **ey_out, double2 **cky_out, int **ckk_out)
{
    TcArgs A{};
    A.u = p.d_u;
    A.s = p.d_s;
    A.alpha = p.d_alpha;
    A.cfac = p.d_cfac;
    A.rein = p.d_rein;
    A.tab = p.d_spin_tab;
    A.start = p.d_spin_start;
    A.mR = p.mR;
    A.nslots = p.nslots;
    A.nblk = (p.nslots + TC_T - 1) / TC_T;
    A.lmax = p.lmax;
    A.mmax = p.mmax;
    int *ey = nullptr;  // per sign [2][mmax + 1][nblk]: y exponents, then first live chunks; last uint16 [nalm]
    const size_t n = (size_t)(p.mmax + 1) * A.nblk, ns = spin ? 2 : 1;
    double2 *cky = nullptr;
    int *ckk = nullptr;
    cudaError_t e = sht::dev_malloc(&ey, sizeof(int) * 2 * n * ns + sizeof(uint16_t) * (size_t)p.nalm);
    if (e == cudaSuccess) e = sht::dev_malloc(&cky, sizeof(double2) * n * TC_T * ns);
    if (e == cudaSuccess) e = sht::dev_malloc(&ckk, sizeof(int) * n * TC_T * ns);
    for (size_t k = 0; k < ns && e == cudaSuccess; ++k) {
        A.sig = k == 0 ? 1 : -1;
        int *ek = ey + 2 * n * k;
        if (spin)
            tc_tables_kernel<true><<<(unsigned)n, TC_T>>>(A, ek, ek + n, cky + n * TC_T * k, ckk + n * TC_T * k);
        else
            tc_tables_kernel<false><<<(unsigned)n, TC_T>>>(A, ek, ek + n, cky, ckk);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) {
        uint16_t *yl = (uint16_t *)(ey + 2 * n * ns);
        if (spin)
            tc_top_kernel<true><<<(unsigned)(p.mmax + 1), TC_T>>>(A, yl);
        else
            tc_top_kernel<false><<<(unsigned)(p.mmax + 1), TC_T>>>(A, yl);
        e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
    if (e != cudaSuccess) {
        cudaFree(ey);
        cudaFree(cky);
        cudaFree(ckk);
        return e;
    }
    *ey_out = ey;
    *cky_out = cky;
    *ckk_out = ckk;
    return cudaSuccess;
}

cudaError_t build_tc_tables(Plan &p)
{
    return p.d_tc_Ey ? cudaSuccess : build_tables(p, false, &p.d_tc_Ey, &p.d_tc_ck_y, &p.d_tc_ck_k);
}

cudaError_t build_tc_spin_tables(Plan &p)
{
    return p.d_sp_Ey ? cudaSuccess : build_tables(p, true, &p.d_sp_Ey, &p.d_sp_ck_y, &p.d_sp_ck_k);
}

// FP64-mode plans whose Legendre steps run here instead of in the plain FP64 kernels of legendre.cu.
// The results do not depend on how maps are grouped into calls, so the rule looks at the plan only.
// Legendre synthesis / analysis of HEALPix plans (lmax = 2 Nside), plain kernels against these, us:
//     lmax 128: 1 map 35 / 61, 58 / 61    4 maps 62 / 173, 62 / 64      16 maps 247 / 677, 71 / 67
//     lmax 192: 1 map 77 / 132, 73 / 87   4 maps 151 / 403, 77 / 88     16 maps 601 / 1598, 95 / 97
//     lmax 1024: 1 map 3419 / 4599, 2322 / 3185                         16 maps 31672 / 55868, 3040 / 3861
// so that from lmax 192 on no number of maps loses.  Few rings, and mmax far below lmax (unpaired rings over
// both hemispheres):
//     16 rings, lmax 192: 1 map 48 / 87, 51 / 56      4 maps 98 / 249, 53 / 57
//     64 rings, lmax 512, mmax 4: 1 map 92 / 173, 78 / 83     4 maps 205 / 523, 80 / 85
//     130 rings, one block polar, lmax 192, mmax 2: 1 map 61 / 95, 82 / 86   4 maps 100 / 256, 85 / 86;
//         lmax 2048, mmax 4: 1 map 484 / 780, 511 / 526     4 maps 911 / 2353, 518 / 529
//     300 rings, lmax 4096, mmax 100: 1 map 1034 / 1859, 741 / 869    4 maps 2562 / 6331, 778 / 885
// There the one-map synthesis of a few m can lose 3 to 30 us (the chain of a polar block); every analysis
// and every call of more maps gains.
bool tc_fp64_plan(const Plan &p) { return p.lmax >= 192; }

// scratch of the synthesis: the a_lm digits of one m-slab, then the scale exponents and marks
size_t tc_workspace_bytes(const Plan &p, int nmaps)
{
    if (nmaps <= 0) return 0;
    const int N = group_columns(std::min(nmaps, p.tune[SHT_TUNE_TC_MAPS]));
    const size_t all = (size_t)p.tc_total_chunks * chunk_bytes(N);
    const size_t one = (size_t)((p.lmax + TC_CH) / TC_CH) * chunk_bytes(N);  // the largest single m
    return std::max(std::min(all, TC_SLAB_BYTES), one) + exponent_bytes(p) + 256;
}

// the least scratch the synthesis can run in (one m at a time); maps: per launch, 0 for the plan's knob
size_t tc_workspace_least(const Plan &p, int nmaps, int maps)
{
    const int N = group_columns(std::min(nmaps, maps ? maps : p.tune[SHT_TUNE_TC_MAPS]));
    return (size_t)((p.lmax + TC_CH) / TC_CH) * chunk_bytes(N) + exponent_bytes(p) + 256;
}

// Legendre synthesis on the tensor cores in `scratch_bytes` of scratch (tc_workspace_least or more):
// per group of up to 16 maps and per slab of whole m whose digits fit, the scale, split and synthesis
// kernels, and last the plain FP64 sums of the columns that were marked.  The slabs do not change
// the results.  spin: nmaps counts the column pairs (two per polarised map), delta ends as Q and U.
static cudaError_t synth_tc(const Plan &p, bool spin, const double2 *alm, double2 *delta, void *scratch,
                            size_t scratch_bytes, int nmaps, cudaStream_t st, int *nlaunch)
{
    *nlaunch = 0;
    TcArgs A{};
    A.slotN = p.d_slotN;
    A.slotS = p.d_slotS;
    A.u = p.d_u;
    A.s = p.d_s;
    A.alpha = p.d_alpha;
    A.cfac = p.d_cfac;
    A.rein = p.d_rein;
    A.tab = p.d_spin_tab;
    A.nblk = (p.nslots + TC_T - 1) / TC_T;
    A.Ey = spin ? p.d_sp_Ey : p.d_tc_Ey;
    A.first = A.Ey + (size_t)(p.mmax + 1) * A.nblk;
    A.Yl = (const uint16_t *)(A.Ey + (size_t)(spin ? 4 : 2) * (p.mmax + 1) * A.nblk);
    A.ck_y = spin ? p.d_sp_ck_y : p.d_tc_ck_y;
    A.ck_k = spin ? p.d_sp_ck_k : p.d_tc_ck_k;
    A.chunk_base = p.d_tc_chunk_base;
    A.chunk_m = p.d_tc_chunk_m;
    A.status = p.d_status;
    A.nslots = p.nslots;
    A.lmax = p.lmax;
    A.mmax = p.mmax;
    A.nrings = p.nrings;
    A.mR = p.mR;
    A.nalm = p.nalm;
    A.mflag = spin ? nullptr : p.d_mflag;
    A.reach = (int *)scratch;  // [mmax + 1][16], size the same, then Ea [mmax + 1][N], then the digits
    A.size = A.reach + (size_t)(p.mmax + 1) * 16;
    A.Ea = A.size + (size_t)(p.mmax + 1) * 16;
    const size_t head = (exponent_bytes(p) + 255) & ~(size_t)255;
    A.bdig = (uint4 *)((char *)scratch + head);
    const size_t cap = scratch_bytes - head;
    if (scratch_bytes < tc_workspace_least(p, nmaps)) return cudaErrorInvalidValue;
    const int64_t dstride = (int64_t)p.nrings * (p.mmax + 1);
    for (int g0 = 0; g0 < nmaps;) {
        const int nm = std::min(p.tune[SHT_TUNE_TC_MAPS], nmaps - g0);
        A.nmaps = nm;
        A.alm = alm + (int64_t)g0 * p.nalm;
        A.delta = delta + (int64_t)g0 * dstride;
        const int N = group_columns(nm);
        for (int m0 = 0; m0 <= p.mmax;) {
            const int m1 = slab_end(p, m0, N, cap);
            A.m0 = m0;
            A.chunk0 = tc_chunks_below(p, m0);
            const int64_t nch = tc_chunks_below(p, m1) - A.chunk0;
            cudaError_t e;
            if (spin)
                e = N == 32   ? launch_slab<32, true>(p, A, m1 - m0, nch, st)
                    : N == 16 ? launch_slab<16, true>(p, A, m1 - m0, nch, st)
                              : launch_slab<8, true>(p, A, m1 - m0, nch, st);
            else
                e = N == 32   ? launch_slab<32, false>(p, A, m1 - m0, nch, st)
                    : N == 16 ? launch_slab<16, false>(p, A, m1 - m0, nch, st)
                              : launch_slab<8, false>(p, A, m1 - m0, nch, st);
            *nlaunch += spin ? 4 : 3;
            if (e != cudaSuccess) return e;
            m0 = m1;
        }
        cudaError_t e;
        if (spin) {
            spin_combine_kernel<<<152 * 16, 256, 0, st>>>(A.delta, dstride, nm / 2);
            ++*nlaunch;
            e = cudaGetLastError();
            if (e == cudaSuccess) e = launch_spin_synth_fix(p, A.alm, A.delta, A.reach, A.size, nm / 2, st);
        } else {
            e = launch_legendre_synth_fix(p, A.alm, A.delta, A.reach, A.size, nm, st);
        }
        *nlaunch += 1;
        if (e != cudaSuccess) return e;
        g0 += nm;
    }
    return cudaSuccess;
}

cudaError_t launch_legendre_synth_tc(const Plan &p, const double2 *alm, double2 *delta, void *scratch,
                                     size_t scratch_bytes, int nmaps, cudaStream_t st, int *nlaunch)
{
    return synth_tc(p, false, alm, delta, scratch, scratch_bytes, nmaps, st, nlaunch);
}

// spin 2: alm [nmaps][2][nalm] (E, B) to delta [nmaps][2][nrings][mmax + 1] (Q, U), in
// tc_workspace_bytes(p, 2 nmaps) of scratch
cudaError_t launch_spin_synth_tc(const Plan &p, const double2 *alm, double2 *delta, void *scratch, size_t scratch_bytes,
                                 int nmaps, cudaStream_t st, int *nlaunch)
{
    return synth_tc(p, true, alm, delta, scratch, scratch_bytes, 2 * nmaps, st, nlaunch);
}

namespace {
SHT_CHECK_TAKE_DEF(take_check)
}  // namespace
cudaError_t take_check_word_tc(int *w) { return take_check(w); }

}  // namespace sht
