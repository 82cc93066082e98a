// Legendre analysis on the tensor cores (eq. almdef, Algorithm 5): the lambda
// recurrence stays in FP64, the sum over ring slots runs as tcgen05 matrix
// products on digits.
//
// a_lm = c_lm sum over ring slots of y_lm(slot) X_m(slot), X = Sigma = Delta_N + Delta_S for even
// l - m and X = D = Delta_N - Delta_S for odd.  For one m and a block of 128 slots this is the
// product [columns x slots] . [slots x l] (eq. matrix_vec transposed) with the map columns as the
// matrix rows: 64 rows (Sigma and D, re and im, of up to 16 maps), K = 16 slots per MMA, N = 32
// values of l (one 32-l chunk, its 16 even steps first).  Each row keeps the columns of its parity;
// the other half is computed and dropped.  One launch serves 16 maps with one pass of the FP64
// recurrence.
//
// Digits (tc_common.cuh): eight of y 2^d and eight of X 2^-d, with the plan's exponent per (m, block) and
// shift d per slot for y and an exponent per (m, block, row) measured in the CTA for X.  An MMA of 64 rows costs as much as one of
// 128, so each MMA stacks two digits on both sides: A = [X_a ; X_(a+1)] (rows 0-63, 64-127) and
// B = [Y_b | Y_(b+1)] (columns 0-31, 32-63), a and b even.  Its four quadrants collect
// the classes a + b, a + b + 1 (two) and a + b + 2 in the accumulator region of t = a + b (0, 2, 4, 6).
// The ten MMAs with a + b <= 6 cover every product of classes 0 to 7, and every quadrant holds one
// class: over 128 slots its sum stays below 2^24, exact in FP32.  The epilogue adds the classes as
// integers, rounds once to FP64 and writes the block's partial a_lm / c_lm, [block][index][map]; a
// block reduction adds the blocks in order and multiplies by c_lm.
//
// X is constant for the whole CTA and sits in tensor memory as the A operand (4 stacks x 8 K-steps x
// 8 columns = 256 columns).  Read from shared memory it cost 4 KB of the 6 KB that each MMA moved, and
// the 80 MMAs of a chunk held the shared-memory port for 3840 of the chunk's 4096 FP64-bound cycles;
// now an MMA reads the 2 KB of its y digits.  That leaves 256 columns for one set of accumulators,
// so the MMAs run region by region (t = 0, 2, 4, 6) over the chunk's 8 K-steps, and the epilogue
// reads one region while the next is computed: each region has its own full and free barrier.
//
// Spin 2 (polarisation).  With a+- = sum over rings of lambda+- (Dq +- i Du) (spin.cu), E = -(a+ + a-) / 2
// and B = i (a+ - a-) / 2.  A map's pair is two complex columns, and two passes, one per sign of the
// recurrence, each add to both: the northern ring of the pass's own sign, the same for every l, and
// the southern ring of the other sign times (-1)^(l+m).  The reduction of the second pass adds the
// first's result and forms E and B.
//
// What bounds it: the FP64 recurrence, 64 FP64 instructions per warp and chunk = 4096 SM cycles, and the
// other roles' instructions that delay it (about 7.5K cycles a chunk at lmax 4096, 16 maps: 151 ms).
#include "sht_internal.h"

#include <algorithm>
#include <vector>

namespace sht {
namespace {

#include "tc_common.cuh"

constexpr int TA_R = 64;                          // rows: [Sigma | D] x 16 maps x (re, im)
constexpr int TA_MAPS = 16;                       // maps per launch
constexpr int TA_REG = 4;                         // accumulator regions (t = 0, 2, 4, 6)
constexpr int TA_N = 2 * TC_CH;                   // MMA N: two y digits of one 32-l chunk
constexpr int TA_KS = TC_T / 16;                  // K-steps per chunk
constexpr int TA_YS = TC_T + 2;                   // y stage row stride (doubles): 16-byte reads of 8 rows
                                                  // by 8 lanes fall into different banks
constexpr int TA_SDIG = (TC_CH / 8) * 128;        // one digit of one 8-slot group in a y tile
constexpr int TA_SGRP = TC_S * TA_SDIG;           // one 8-slot group: [digit][l / 8] core matrices
constexpr int TA_TILE = (TC_T / 8) * TA_SGRP;     // y digits of one chunk: 64 KB
constexpr int TA_NEPI = 8 * 32;                   // epilogue threads (two warps per tensor-memory lane quarter)
constexpr int TA_XROW = TA_R + 1;                 // doubles per slot of the X staging area
constexpr int TA_OFF_Y = 2 * TA_TILE;
constexpr int TA_OFF_X = TA_OFF_Y + 2 * TC_CH * TA_YS * 8;  // exchange between the top and bottom halves
constexpr int TA_XCH = 32;                        // floats a lane hands over per chunk: 4 columns x 8 class sums
constexpr int TA_OFF_E = TA_OFF_X + TA_NEPI * TA_XCH * 4;
constexpr int TA_OFF_A = TA_OFF_E + TA_R * 4;     // the recurrence warps' coefficients
constexpr int TA_OFF_BAR = TA_OFF_A + TC_ABUF;
constexpr int TA_NBAR = 4 + 2 * TA_REG;           // full[2], done[2], rfull[4], rfree[4]
constexpr int TA_SMEM = TA_OFF_BAR + TA_NBAR * 8 + 16;
constexpr int TA_XCOL = 256;                      // tensor-memory columns: accumulators, then X
constexpr int TA_NT = TC_NT + TA_NEPI + 32;       // 4 recurrence + 8 split + 8 epilogue warps + 1 MMA-issuing warp
static_assert(TC_T * TA_XROW * 8 <= 2 * TA_TILE, "X is staged where the y tiles go later");
static_assert(TA_REG * TA_N <= TA_XCOL && TA_XCOL + 4 * TA_KS * 8 <= 512, "tensor memory");
static_assert(TA_SMEM > 114 * 1024 && TA_SMEM <= 227 * 1024, "one CTA per SM (it holds all tensor memory)");

// the MMA with the A operand in tensor memory
__device__ __forceinline__ void umma_f16_ts_by(uint32_t issue, uint32_t tmem_d, uint32_t tmem_a, uint64_t b,
                                               uint32_t idesc, uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(tmem_d),
        "r"(tmem_a), "l"(b), "r"(idesc), "r"(acc), "r"(issue));
}

// v 2^-d, d <= 255, integer pipe only; a value that would leave the normal range becomes the smallest
// subnormal, which marks a row that holds nothing larger; what is not finite stays
__device__ __forceinline__ double shift_down(double v, int d)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const int ex = (int)((hi >> 20) & 0x7ffu);
    if (ex > d && ex < 0x7ff) return __hiloint2double((int)(hi - ((uint32_t)d << 20)), (int)lo);
    if (ex == 0x7ff || ((hi << 1) | lo) == 0u) return v;
    return __hiloint2double(0, 1);
}

__device__ __forceinline__ void tmem_ld4(uint32_t addr, uint32_t v[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(addr));
}

__device__ __forceinline__ void tmem_st4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
                 : "memory");
}

// The sums of classes 0 .. 7 of one column as one integer in units of 2^-3 of class 5, rounded to FP64
__device__ __forceinline__ double classes_to_double(const float (&v)[8], int e)
{
    int S[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) S[c] = class_sum(v[c]);
    const long long H = (long long)S[0] * 65536 + (S[1] * 256 + S[2]);              // class 2
    const long long M = (long long)S[3] * 65536 + ((long long)S[4] * 256 + S[5]);  // class 5
    const long long Z = (long long)S[6] * 256 + S[7];                             // class 7
    return i64_to_double(H * (1ll << 27) + M * 8 + ((Z + 4096) >> 13), e);
}

// CTA: one m, 128 slots, 672 threads in four roles.
//   warps 0-3   recurrence (recurrence_warps, double-buffered y stage of 32 l, even steps first);
//   warps 4-19  first stage X = Sigma | D of the block in shared memory and cut it into tensor memory,
//               while the recurrence fills its two stages (whole analysis, with the recurrence waiting
//               for X cut by warps 4-11 alone against this: 23.59 -> 22.67 ms at lmax 2048, 1 map,
//               179.9 -> 173.0 at 4096, 4 maps, 200.6 -> 193.3 with 16); then
//   warps 4-11  split: cut each chunk's y values into one of two tile sets and arrive on its full barrier;
//   warps 12-19 epilogue, two per tensor-memory lane quarter (8 of the row's 16 columns each): wait for
//               each region, read it, release it, add the class sums of the top and bottom halves (lane
//               quarters 0, 1 and 2, 3) through shared memory and write the block's partial a_lm / c_lm;
//   warp 20     MMA issue: per chunk wait for the tile set, then per region until it is read out, issue
//               its MMAs and commit them to the region's full barrier, after the last one also to
//               the tile set's done barrier.
// Every barrier phase a warp waits for can run at most one phase ahead of that wait, so the
// parity tests are unambiguous; every mbarrier wait is bounded and the epilogue warps agree on
// their outcome (bar.red) so that their named barriers stay balanced.
// The code of the roles competes for the instruction caches, and each warp runs in order: with four
// epilogue warps of twice the code (everything unrolled) a chunk took them 9.7K cycles.
template <bool SPIN>
__global__ void __launch_bounds__(TA_NT, 1) tc_anal_kernel(TcArgs A)
{
    extern __shared__ __align__(1024) unsigned char smem[];
    unsigned char *sY = smem;                               // [set][8-slot group][digit][l / 8] core matrices
    double *xs = (double *)smem;                            // X staging, [slot][TA_XROW], before the first tile
    double *ybuf = (double *)(smem + TA_OFF_Y);             // [stage][32 rows][TA_YS]
    float4 *xch = (float4 *)(smem + TA_OFF_X);              // [8 quads][256 lanes] class sums handed over
    double *abuf = (double *)(smem + TA_OFF_A);             // [recurrence warp][32 l]
    int *sEx = (int *)(smem + TA_OFF_E);                    // [64] row exponents (biased, 0: all zero)
    uint64_t *full = (uint64_t *)(smem + TA_OFF_BAR);       // full[2]: a tile set written
    uint64_t *done = full + 2;                              // done[2]: the MMAs that read a tile set complete
    uint64_t *rfull = done + 2;                             // rfull[4]: a region complete
    uint64_t *rfree = rfull + TA_REG;                       // rfree[4]: a region read out
    uint32_t *tslot = (uint32_t *)(rfree + TA_REG);

    const int m = A.m0 + (int)(blockIdx.x / A.nblk);
    const int blk = (int)(blockIdx.x % A.nblk);

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const bool rec = warp < 4, splitw = warp >= 4 && warp < 12, epi = warp >= 12 && warp < 20;
    const bool issuer = warp == 20;
    const int sp = tid - TC_T;                              // split-thread index 0..255
    const int r = rec ? tid : (sp & (TC_T - 1));            // slot within the block
    const int slot = blk * TC_T + r;
    const bool active = slot < A.nslots;
    const int L = A.lmax;
    const int64_t base = (int64_t)m * (2 * L + 3 - m) / 2;
    const int lb = first_l<SPIN ? REC_SPIN : REC_Y>(m);
    const int nch = (L - lb + TC_CH) / TC_CH;
    const int cfirst = A.first[m * A.nblk + blk];           // chunks before it hold only dropped values:
    const int nlive = nch - cfirst;                         // the reduction leaves them out
    const int nm = A.nmaps;
    if (nlive <= 0 || (A.mflag && !A.mflag[m])) return;

    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tslot)), "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&full[i], 2 * TC_T);  // split threads
            mbar_init(&done[i], 1);         // commit
        }
        for (int i = 0; i < TA_REG; ++i) {
            mbar_init(&rfull[i], 1);        // commit
            mbar_init(&rfree[i], TA_NEPI);  // epilogue
        }
        asm volatile("fence.mbarrier_init.release.cluster;");
    }
    if (tid < TA_R) sEx[tid] = 0;
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = *tslot;

    if (splitw || epi) {
        // ------------------------------------------------ X into tensor memory, beside the first chunks of y
        {
            // rows 32 s + 2 g + c (s: Sigma, D; map g; c: re, im) of slot r: this thread's maps are
            // hh, hh + 4, ... (uniform per warp); the rows of absent maps are zero
            const int hh = sp >> 7;
            const int rn = active ? A.slotN[slot] : -1, rs = active ? A.slotS[slot] : -1;
            const int64_t mstride = A.mmax + 1, dstride = (int64_t)A.nrings * mstride;
            double *xr = xs + r * TA_XROW;
            const int sd = state_d(A.ck_k[(int64_t)(m * A.nblk + blk) * TC_T + r]);  // this slot's d
            const bool bn = rn >= 0 && SHT_CHK(rn < A.nrings), bs = rs >= 0 && SHT_CHK(rs < A.nrings);
            const double2 *dN = A.delta + (int64_t)(bn ? rn : 0) * mstride + m;
            const double2 *dS = A.delta + (int64_t)(bs ? rs : 0) * mstride + m;
            const double2 zero = make_double2(0.0, 0.0);
            if (SPIN) {
                // column pair 2 h + c of polarised map h (this thread: h = hh, hh + 4, ...): Dq +- i Du of the
                // northern ring for the pass's own sign c (0: +), of the southern ring for the other
#pragma unroll 1
                for (int h = hh; h < TA_MAPS / 2; h += 4) {
                    const bool have = 2 * h < nm;
#pragma unroll
                    for (int c = 0; c < 2; ++c) {
                        const bool own = (c == 0) == (A.sig > 0);
                        const double2 *d = (own ? dN : dS) + 2 * h * dstride;
                        const bool in = have && (own ? bn : bs);
                        const double2 q = in ? d[0] : zero, w = in ? d[dstride] : zero;
                        const double re = c == 0 ? q.x - w.y : q.x + w.y, im = c == 0 ? q.y + w.x : q.y - w.x;
                        const bool neg = !own && m == 1;  // (-1)^(l+m) of the even rows, l - max(m, 2) even
                        const double xre = shift_down(re, sd), xim = shift_down(im, sd);
                        double *x = xr + 2 * (2 * h + c);
                        x[0] = neg ? -xre : xre;
                        x[1] = neg ? -xim : xim;
                        x[32] = own || neg ? xre : -xre;
                        x[33] = own || neg ? xim : -xim;
                    }
                }
            } else {
                // rolled, one map ahead: unrolled over the 8 maps the loop was slower (its code is run once per
                // CTA: instruction fetch), 202.9 -> 200.5 ms for the whole analysis at lmax 4096, 16 maps
                double2 n = bn && hh < nm ? dN[hh * dstride] : zero, s = bs && hh < nm ? dS[hh * dstride] : zero;
#pragma unroll 1
                for (int g = hh; g < TA_MAPS; g += 4) {
                    const bool more = g + 4 < nm;
                    const double2 n1 = bn && more ? dN[(g + 4) * dstride] : zero, s1 = bs && more ? dS[(g + 4) * dstride] : zero;
                    double *x = xr + 2 * g;
                    if (g < nm) {
                        x[0] = shift_down(n.x + s.x, sd);
                        x[1] = shift_down(n.y + s.y, sd);
                        x[32] = shift_down(n.x - s.x, sd);
                        x[33] = shift_down(n.y - s.y, sd);
                    } else {
                        x[0] = x[1] = x[32] = x[33] = 0.0;
                    }
                    n = n1;
                    s = s1;
                }
            }
        }
        bar_sync(BAR_STAGED, 2 * TC_T + TA_NEPI);  // X staged
        {
            // lane quarter qd holds rows 32 (qd & 1) .. + 31: the even digits of each stack in quarters
            // 0, 1 and the odd ones in 2, 3.  Four warps each take 32 slots.
            const int qd = warp & 3, kh = (warp - 4) >> 2;
            const int row = 32 * (qd & 1) + lane;
            const double *xc = xs + (32 * kh) * TA_XROW + row;
            if (qd < 2) {  // row exponents and rows the digits cannot carry
                int mx = 0;
                bool odd = false;
#pragma unroll 4
                for (int k = 0; k < 32; ++k) {
                    const double v = xc[k * TA_XROW];
                    const int ex = dexp(v);
                    mx = max(mx, ex);
                    odd |= ex == 0 && (((uint32_t)__double2hiint(v) << 1) | (uint32_t)__double2loint(v)) != 0u;
                }
                if (odd) mx = max(mx, 1);  // subnormal values mark a row that holds nothing larger
                if (mx) atomicMax(&sEx[row], mx);
                if (mx > TC_EHUGE) A.fix[m * 16 + (lane >> 1)] = 1;
            }
            bar_sync(BAR_STAGED, 2 * TC_T + TA_NEPI);  // row exponents complete
            const int e = sEx[row];
            if (kh == 0 && qd < 2 && e && e < TC_ETINY) A.fix[m * 16 + (lane >> 1)] = 1;
            const int E = e ? e - 1022 : TC_EZERO;
            const uint32_t at = tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(TA_XCOL + 2 * kh * 8);
#pragma unroll 1
            for (int p0 = 0; p0 < 16; p0 += 4) {  // 4 slot pairs = 4 columns of K-step 2 kh + p0 / 8
                uint32_t w[4][4];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const uint2 f0 = digit_fields(xc[(2 * (p0 + p)) * TA_XROW], E);
                    const uint2 f1 = digit_fields(xc[(2 * (p0 + p) + 1) * TA_XROW], E);
                    uint32_t d[TC_S];
                    digit_pairs(f0, f1, d);
#pragma unroll
                    for (int i = 0; i < 4; ++i) w[i][p] = qd < 2 ? d[2 * i] : d[2 * i + 1];
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) tmem_st4(at + (uint32_t)(i * TA_KS * 8 + p0), w[i][0], w[i][1], w[i][2], w[i][3]);
            }
            asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
        }
        asm volatile("tcgen05.fence::before_thread_sync;");
    }

    bool ok = true;
    if (rec) {
        if (SPIN)
            recurrence_warps<REC_SPIN, true, TA_YS, 4>(A, m, blk, r, active, base, nch, cfirst, ybuf, abuf);
        else if (polar_block(A, m, blk))
            recurrence_warps<REC_REIN, true, TA_YS, 4>(A, m, blk, r, active, base, nch, cfirst, ybuf, abuf);
        else
            recurrence_warps<REC_Y, true, TA_YS, 4>(A, m, blk, r, active, base, nch, cfirst, ybuf, abuf);
    } else if (issuer) {
        // ------------------------------------------------ MMA issue (one lane of the last warp)
        const uint32_t idesc = umma_idesc<TA_N>();  // M = 128, N = 64
        const uint64_t dB0 = umma_desc(smem_u32(sY), TA_SGRP, 128);
        const uint32_t issue = elect_one();
        bar_sync(BAR_PREP, 2 * TC_T + TA_NEPI + 32);  // X is in tensor memory
        asm volatile("tcgen05.fence::after_thread_sync;");
        for (int q = 0; q < nlive && ok; ++q) {
            const int st = q & 1;
            if (!mbar_wait(&full[st], (uint32_t)((q >> 1) & 1))) ok = false;
            ok = __all_sync(0xffffffffu, ok);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;");
            const uint64_t bS = dB0 + (uint64_t)((st * TA_TILE) >> 4);  // address field: bytes / 16
#pragma unroll 1
            for (int t = 0; t < TA_REG; ++t) {   // region of classes 2 t .. 2 t + 2
                if (q >= 1 && !mbar_wait(&rfree[t], (uint32_t)((q - 1) & 1))) ok = false;
                ok = __all_sync(0xffffffffu, ok);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll 1
                for (int i = 0; i <= t; ++i) {   // [X_(2i) ; X_(2i+1)] against [Y_(2(t-i)) | Y_(2(t-i)+1)]
                    const uint32_t aT = tmem + (uint32_t)(TA_XCOL + i * TA_KS * 8);
                    const uint64_t bT = bS + (uint64_t)((2 * (t - i) * TA_SDIG) >> 4);
#pragma unroll
                    for (int kk = 0; kk < TA_KS; ++kk)
                        umma_f16_ts_by(issue, tmem + (uint32_t)(t * TA_N), aT + (uint32_t)(kk * 8),
                                       bT + (uint64_t)((kk * 2 * TA_SGRP) >> 4), idesc, (i == 0 && kk == 0) ? 0u : 1u);
                }
                umma_commit_by(issue, &rfull[t]);
            }
            if (ok) umma_commit_by(issue, &done[st]);
        }
        if (lane == 0 && !ok) atomicOr(A.status, 1);
    } else if (splitw) {
        // ------------------------------------------------ the y tiles
        const int Ey = A.Ey[m * A.nblk + blk];
        bar_sync(BAR_PREP, 2 * TC_T + TA_NEPI + 32);  // X in tensor memory, its staging area free
        // this thread cuts row n of the y stage (l - l0 = 2 (n % 16) + n / 16) for the 8-slot groups
        // sg and sg + 8: its 8 values of a digit are one 16-byte core-matrix row
        const int w8 = warp - 4;
        const int n = (lane & 7) + 8 * (w8 & 3), sg0 = (lane >> 3) + 4 * (w8 >> 2);
        // d of its 16 slots, a byte each
        uint32_t sd[4];
        {
            const int *ck = A.ck_k + (int64_t)(m * A.nblk + blk) * TC_T + 8 * sg0;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                sd[i] = 0;
#pragma unroll
                for (int j = 0; j < 4; ++j) sd[i] |= (uint32_t)state_d(ck[64 * (i >> 1) + 4 * (i & 1) + j]) << (8 * j);
            }
        }
        for (int q = 0; q < nlive; ++q) {
            const int st = q & 1;
            bar_sync(BAR_FULL + st, TC_NT);  // y of chunk q is in its stage
            const double *yb = ybuf + (size_t)st * TC_CH * TA_YS + n * TA_YS;
            unsigned char *yt = sY + st * TA_TILE + (n >> 3) * 128 + (n & 7) * 16;
#pragma unroll 1
            for (int i = 0; i < 2; ++i) {
                const int sg = sg0 + 8 * i;
                const uint32_t da = i ? sd[2] : sd[0], db = i ? sd[3] : sd[1];
                uint32_t pk[4][TC_S];
#pragma unroll
                for (int p = 0; p < 4; ++p) {
                    const double2 v = *reinterpret_cast<const double2 *>(yb + 8 * sg + 2 * p);
                    const uint32_t w = (p < 2 ? da : db) >> (16 * (p & 1));
                    digit_pairs(digit_fields(v.x, Ey - (int)(w & 255u)), digit_fields(v.y, Ey - (int)((w >> 8) & 255u)), pk[p]);
                }
                if (i == 1 && q + 2 < nlive) bar_arrive(BAR_EMPTY + st, TC_NT);  // y stage read
                // the MMAs of chunk q - 2 read this tile set: wait (bounded) before rewriting it
                if (i == 0 && q >= 2 && ok && !mbar_wait(&done[st], (uint32_t)(((q >> 1) - 1) & 1))) ok = false;
#pragma unroll
                for (int s = 0; s < TC_S; ++s)
                    *(uint4 *)(yt + sg * TA_SGRP + s * TA_SDIG) = make_uint4(pk[0][s], pk[1][s], pk[2][s], pk[3][s]);
            }
            asm volatile("fence.proxy.async.shared::cta;");
            mbar_arrive(&full[st]);
        }
        if (!ok && lane == 0) atomicOr(A.status, 1);
    } else if (epi) {
        // ------------------------------------------------ epilogue, two warps per lane quarter
        // lane quarter qd: row 32 (qd & 1) + lane, the top half (qd < 2) or the bottom half (qd >= 2)
        // of its sums; Sigma rows (qd even) keep the even l - m columns 0-15, D rows the odd 16-31.
        // In region t a top row holds class 2 t in the left columns and 2 t + 1 in the right ones, a
        // bottom row 2 t + 1 and 2 t + 2.  So with a[t], b[t] = left, right of region t in a top row and
        // right of region t - 1, left of region t in a bottom row, the sums of classes 2 t and 2 t + 1
        // are a[t] and b[t] added over the two (exact in FP32; class 8 is incomplete and left out).  Of
        // the 8 columns of this warp the top lane finishes 4 and the bottom lane of the same row the other
        // 4: each hands the other its sums of those, and the eight class sums of a column become one
        // integer in units of 2^-3 of class 5 (2^-55 of 2^(E_y + E_x)), rounded once to FP64.
        // Up to 8 (4) maps only lanes 0-15 (0-7) hold rows: they leave their own sums beside those handed
        // over, and all lanes take a share of the columns, W / 8 each (whole analysis, against every lane
        // finishing 4: 22.67 -> 22.02 ms at lmax 2048, 1 map, 173.0 -> 168.4 at 4096, 4 maps).
        const int qd = warp & 3, es = qd & 1, hc = (warp - 12) >> 2;
        const bool top = qd < 2;
        const int W = nm <= 4 ? 8 : nm <= 8 ? 16 : 32;
        const int rr = lane & (W - 1);          // this lane finishes columns of row 32 es + rr
        const int erow = 32 * es + rr;
        const int eg = rr >> 1, ec = rr & 1;
        const int t0 = 4 * hc + (top ? 0 : 8);  // this lane finishes columns t0 .. t0 + 3
        bar_sync(BAR_PREP, 2 * TC_T + TA_NEPI + 32);  // row exponents complete
        const int ex = sEx[erow];
        const int e = A.Ey[m * A.nblk + blk] + (ex ? ex - 1022 : 0) - 55;
        float4 *mine = xch + (tid - TC_NT), *other = xch + ((tid - TC_NT) ^ 64);
        const uint32_t row0 = tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(16 * es);
        // partial sum of column t0 + j: l = l1 + 2 j of the chunk
        const int l1 = lb + TC_CH * cfirst + es + 2 * t0;
        double *dst = (double *)(A.partial + (int64_t)blk * A.nalm_part * nm + (base - A.idx0 + (l1 - m)) * nm + eg) + ec;
        for (int q = 0; q < nlive; ++q) {
            float v[TA_REG][2][4];
            if (q >= 1) bar_sync(BAR_EPI, TA_NEPI);  // the other half has read the previous chunk's sums
#pragma unroll
            for (int t = 0; t < TA_REG; ++t) {
                if (ok && !mbar_wait(&rfull[t], (uint32_t)(q & 1))) ok = false;
                ok = __all_sync(0xffffffffu, ok);  // tcgen05.ld is warp-wide
                asm volatile("tcgen05.fence::after_thread_sync;");
                uint32_t l[4], r[4], ol[4], orr[4];
                if (ok) {
                    tmem_ld4(row0 + (uint32_t)(t * TA_N + t0), l);
                    tmem_ld4(row0 + (uint32_t)(t * TA_N + TC_CH + t0), r);
                    tmem_ld4(row0 + (uint32_t)(t * TA_N + (t0 ^ 8)), ol);
                    tmem_ld4(row0 + (uint32_t)(t * TA_N + TC_CH + (t0 ^ 8)), orr);
                    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                }
                asm volatile("tcgen05.fence::before_thread_sync;");
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&rfree[t])) : "memory");
                // own columns into v; the other half's into its hands: a[t] at quad 2 t, b[t] at 2 t + 1
                const float4 fl = make_float4(__uint_as_float(ol[0]), __uint_as_float(ol[1]), __uint_as_float(ol[2]),
                                              __uint_as_float(ol[3]));
                const float4 fr = make_float4(__uint_as_float(orr[0]), __uint_as_float(orr[1]), __uint_as_float(orr[2]),
                                              __uint_as_float(orr[3]));
                if (top) {
                    if (lane < W) {
                        mine[(2 * t) * TA_NEPI] = fl;
                        mine[(2 * t + 1) * TA_NEPI] = fr;
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        v[t][0][j] = __uint_as_float(l[j]);
                        v[t][1][j] = __uint_as_float(r[j]);
                    }
                } else {
                    if (lane < W) {
                        if (t == 0) mine[0] = make_float4(0.f, 0.f, 0.f, 0.f);
                        mine[(2 * t + 1) * TA_NEPI] = fl;
                        if (t + 1 < TA_REG) mine[(2 * t + 2) * TA_NEPI] = fr;
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        if (t == 0) v[0][0][j] = 0.f;
                        v[t][1][j] = __uint_as_float(l[j]);
                        if (t + 1 < TA_REG) v[t + 1][0][j] = __uint_as_float(r[j]);
                    }
                }
            }
            if (lane < W && W < 32) {
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const float *w = v[c >> 1][c & 1];
                    mine[c * TA_NEPI + W] = make_float4(w[0], w[1], w[2], w[3]);
                }
            }
            ok = bar_red_and(BAR_EPI + 1, TA_NEPI, ok);  // the sums are handed over; the warps agree
            if (ok && W < 32) {
                const float *po = (const float *)(other - lane + rr), *pm = (const float *)(mine - lane + W + rr);
#pragma unroll 1
                for (int j = lane / W * (W / 8), i = 0; i < W / 8; ++i, ++j) {
                    float f[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) f[c] = pm[4 * c * TA_NEPI + j] + po[4 * c * TA_NEPI + j];
                    const double d = classes_to_double(f, e);
                    const int l = l1 + TC_CH * q + 2 * j;
                    if (eg < nm && l <= L && SHT_CHK(base + (l - m) >= A.idx0 && base + (l - m) < A.idx0 + A.nalm_part))
                        dst[(int64_t)(4 * j) * nm] = d;
                }
            } else if (ok) {
#pragma unroll
                for (int t = 0; t < TA_REG; ++t)
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const float4 o = other[(2 * t + h) * TA_NEPI];
                        v[t][h][0] += o.x;
                        v[t][h][1] += o.y;
                        v[t][h][2] += o.z;
                        v[t][h][3] += o.w;
                    }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    float f[8];
#pragma unroll
                    for (int c = 0; c < 8; ++c) f[c] = v[c >> 1][c & 1][j];
                    const double d = classes_to_double(f, e);
                    const int l = l1 + TC_CH * q + 2 * j;
                    if (eg < nm && l <= L && SHT_CHK(base + (l - m) >= A.idx0 && base + (l - m) < A.idx0 + A.nalm_part))
                        dst[(int64_t)(4 * j) * nm] = d;
                }
            }
            dst += (int64_t)(2 * TC_CH) * nm;
        }
        if (!ok && lane == 0) atomicOr(A.status, 1);
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

// a_lm = c_lm sum over the slot blocks that are live at l, in block order; Im a_l0 = 0.  One CTA per
// 32-l chunk of one m: it reads the [32 l][nmaps] partial sums of each block as one contiguous
// piece and turns them through shared memory into the coefficient rows of each map.  Bound by
// DRAM: live blocks x 16 B read per coefficient and map, 16 B written.
// Spin: the first pass writes c_lm a+-, the second adds its own and turns the pair into E and B.
constexpr int TR_T = 256;
template <bool SPIN>
__global__ void __launch_bounds__(TR_T) tc_reduce_kernel(TcArgs A, double2 *__restrict__ alm)
{
    __shared__ double2 s_v[TC_CH * (TA_MAPS + 1)];
    __shared__ int s_blk[TR_T], s_n;
    const int64_t chunk = A.chunk0 + blockIdx.x;
    const int m = A.chunk_m[chunk];
    const int c = (int)(chunk - A.chunk_base[m]);
    const int lb = first_l<SPIN ? REC_SPIN : REC_Y>(m);
    const int l0 = lb + TC_CH * c, nl = max(0, min(TC_CH, A.lmax - l0 + 1)), nm = A.nmaps;
    const int64_t ix0 = (int64_t)m * (2 * A.lmax + 3 - m) / 2 + (l0 - m);
    if (SPIN && c == 0)  // no spin-2 function below l = 2
        for (int t = threadIdx.x; t < (min(lb, A.lmax + 1) - m) * nm; t += TR_T)
            alm[(int64_t)(t % nm) * A.nalm + ix0 - (lb - m) + t / nm] = make_double2(0.0, 0.0);
    const int tot = nl * nm;
    const int64_t bstride = A.nalm_part * nm;
    const double2 *src = A.partial + (ix0 - A.idx0) * nm;
    double2 v[2] = {make_double2(0.0, 0.0), make_double2(0.0, 0.0)};
    const int nblk = (A.mflag && !A.mflag[m]) ? 0 : A.nblk;  // an m this plan does not compute: zeros
    for (int b0 = 0; b0 < nblk; b0 += TR_T) {
        __syncthreads();
        if (threadIdx.x < 32) {  // the live blocks of this batch, in order
            int n = 0;
            for (int i = 0; i < TR_T; i += 32) {
                const int b = b0 + i + (int)threadIdx.x;
                const bool live = b < A.nblk && A.first[m * A.nblk + b] <= c;
                const unsigned mask = __ballot_sync(0xffffffffu, live);
                if (live) s_blk[n + __popc(mask & ((1u << threadIdx.x) - 1u))] = b;
                n += __popc(mask);
                if (b0 + i + 32 >= A.nblk) break;
            }
            if (threadIdx.x == 0) s_n = n;
        }
        __syncthreads();
        const int nb = s_n;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            const int t = threadIdx.x + i * TR_T;
            if (t < tot) {
#pragma unroll 8
                for (int b = 0; b < nb; ++b) {
                    const double2 p = src[s_blk[b] * bstride + t];
                    v[i].x += p.x;
                    v[i].y += p.y;
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
        const int t = threadIdx.x + i * TR_T;
        if (t < tot) s_v[(t / nm) * (TA_MAPS + 1) + t % nm] = v[i];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < tot; t += TR_T) {
        const int g = t / nl, l = t - g * nl;
        double2 *out = alm + (int64_t)g * A.nalm + ix0 + l;
        if (!SPIN) {
            const double cf = A.cfac[ix0 + l];
            const double2 s = s_v[l * (TA_MAPS + 1) + g];
            *out = make_double2(cf * s.x, m == 0 ? 0.0 : cf * s.y);
        } else if ((g & 1) == 0) {
            const double cf = A.tab[ix0 + l].w;
            const double2 s = s_v[l * (TA_MAPS + 1) + g], r = s_v[l * (TA_MAPS + 1) + g + 1];
            double2 p = make_double2(cf * s.x, cf * s.y), q = make_double2(cf * r.x, cf * r.y);
            if (A.sig < 0) {
                const double2 p0 = out[0], q0 = out[A.nalm];
                p = make_double2(p.x + p0.x, p.y + p0.y);
                q = make_double2(q.x + q0.x, q.y + q0.y);
                out[0] = make_double2(-0.5 * (p.x + q.x), m == 0 ? 0.0 : -0.5 * (p.y + q.y));
                out[A.nalm] = make_double2(-0.5 * (p.y - q.y), m == 0 ? 0.0 : 0.5 * (p.x - q.x));
            } else {
                out[0] = p;
                out[A.nalm] = q;
            }
        }
    }
}
static_assert(2 * TR_T >= TC_CH * TA_MAPS, "two values a thread");

// The analysis runs in m-slabs of about equal coefficient counts, each followed by its block
// reduction, so that the partial sums of one slab only are held at a time: at lmax 4096 all 32
// blocks x 16 maps x 16 B per coefficient would take 69 GB, a slab about 1/8 of that.  Boundaries:
// first m of each slab, then mmax + 1.
std::vector<int> anal_slabs(const Plan &p, int nm)
{
    const int nblk = (p.nslots + TC_T - 1) / TC_T;
    const int64_t full = (int64_t)nblk * nm * p.nalm * (int64_t)sizeof(double2);
    const int ns = full <= (int64_t(2) << 30) ? 1 : 8;
    const int64_t L = p.lmax;
    auto idx = [&](int64_t m) { return m * (2 * L + 3 - m) / 2; };
    std::vector<int> b{0};
    for (int k = 1; k < ns; ++k) {
        const int64_t want = p.nalm * k / ns;
        int m = b.back() + 1;
        while (m <= p.mmax && idx(m) < want) ++m;
        if (m <= p.mmax) b.push_back(m);
    }
    b.push_back(p.mmax + 1);
    return b;
}

int64_t slab_max_count(const Plan &p, const std::vector<int> &b)
{
    const int64_t L = p.lmax;
    auto idx = [&](int64_t m) { return m * (2 * L + 3 - m) / 2; };
    int64_t mx = 0;
    for (size_t k = 0; k + 1 < b.size(); ++k) mx = std::max(mx, (b[k + 1] > p.mmax ? p.nalm : idx(b[k + 1])) - idx(b[k]));
    return mx;
}

size_t fix_bytes(const Plan &p) { return ((size_t)(p.mmax + 1) * 16 * sizeof(int) + 255) & ~(size_t)255; }

}  // namespace

cudaError_t configure_tc_anal_kernel()
{
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t e = cudaFuncSetAttribute(tc_anal_kernel<false>, a, TA_SMEM);
    return e == cudaSuccess ? cudaFuncSetAttribute(tc_anal_kernel<true>, a, TA_SMEM) : e;
}

// marks of the columns left to the plain FP64 sums, then the partial a_lm / c_lm per 128-slot block
// for one group of up to 16 maps and one m-slab, [block][index][map]
size_t tc_anal_partial_bytes(const Plan &p, int nmaps)
{
    const int nblk = (p.nslots + TC_T - 1) / TC_T;
    size_t most = 0;
    for (int nm : {std::min(nmaps, TA_MAPS), nmaps % TA_MAPS})  // a full group and the last one
        if (nm > 0) most = std::max(most, (size_t)nblk * nm * (size_t)slab_max_count(p, anal_slabs(p, nm)) * sizeof(double2));
    return fix_bytes(p) + most;
}

// Legendre analysis on the tensor cores: per group of up to 16 maps and per m-slab the tensor-core
// kernel, the fixed-order block reduction of that slab into a_lm and the plain FP64 sums of the
// columns that were marked.  spin: nmaps counts the column pairs (two per polarised map).
static cudaError_t anal_tc(const Plan &p, bool spin, const double2 *delta, double2 *alm, void *partial, int nmaps,
                           cudaStream_t st, int *nlaunch)
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
    const size_t tables = (size_t)(p.mmax + 1) * A.nblk;
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
    A.fix = (int *)partial;
    A.partial = (double2 *)((char *)partial + fix_bytes(p));
    const int64_t dstride = (int64_t)p.nrings * (p.mmax + 1);
    const int64_t L = p.lmax;
    auto idx = [&](int64_t m) { return m * (2 * L + 3 - m) / 2; };
    for (int g0 = 0; g0 < nmaps; g0 += TA_MAPS) {
        const int nm = std::min(TA_MAPS, nmaps - g0);
        A.nmaps = nm;
        A.delta = const_cast<double2 *>(delta) + (int64_t)g0 * dstride;
        double2 *out = alm + (int64_t)g0 * p.nalm;
        cudaError_t e = cudaMemsetAsync(A.fix, 0, fix_bytes(p), st);
        if (e != cudaSuccess) return e;
        const std::vector<int> slabs = anal_slabs(p, nm);
        for (size_t k = 0; k + 1 < slabs.size(); ++k) {
            const int mlo = slabs[k], mhi = slabs[k + 1];
            A.m0 = mlo;
            A.idx0 = idx(mlo);
            A.nalm_part = (mhi > p.mmax ? p.nalm : idx(mhi)) - A.idx0;
            A.chunk0 = tc_chunks_below(p, mlo);
            const unsigned grid = (unsigned)((mhi - mlo) * A.nblk);
            const unsigned rgrid = (unsigned)(tc_chunks_below(p, mhi) - A.chunk0);
            for (int pass = 0; pass < (spin ? 2 : 1); ++pass) {
                A.sig = pass == 0 ? 1 : -1;
                A.Ey = (spin ? p.d_sp_Ey : p.d_tc_Ey) + 2 * tables * pass;
                A.first = A.Ey + tables;
                A.ck_y = (spin ? p.d_sp_ck_y : p.d_tc_ck_y) + tables * TC_T * pass;
                A.ck_k = (spin ? p.d_sp_ck_k : p.d_tc_ck_k) + tables * TC_T * pass;
                if (spin) {
                    tc_anal_kernel<true><<<grid, TA_NT, TA_SMEM, st>>>(A);
                    tc_reduce_kernel<true><<<rgrid, TR_T, 0, st>>>(A, out);
                } else {
                    StageEvents ev(p, SHT_STAGE_TC_ANAL_KERNEL, st);
                    tc_anal_kernel<false><<<grid, TA_NT, TA_SMEM, st>>>(A);
                    p.launches[SHT_STAGE_TC_ANAL_KERNEL] += 1;
                    ev.done();
                    tc_reduce_kernel<false><<<rgrid, TR_T, 0, st>>>(A, out);
                }
                *nlaunch += 2;
                e = cudaGetLastError();
                if (e != cudaSuccess) return e;
            }
            e = spin ? launch_spin_anal_fix(p, A.delta, out, A.partial, A.fix, nm / 2, mlo, mhi, A.idx0, A.nalm_part, st)
                     : launch_legendre_anal_fix(p, A.delta, out, A.partial, A.fix, nm, mlo, mhi, A.idx0, A.nalm_part, st);
            *nlaunch += 1;
            if (e != cudaSuccess) return e;
        }
    }
    return cudaSuccess;
}

cudaError_t launch_legendre_anal_tc(const Plan &p, const double2 *delta, double2 *alm, void *partial, int nmaps,
                                    cudaStream_t st, int *nlaunch)
{
    return anal_tc(p, false, delta, alm, partial, nmaps, st, nlaunch);
}

// spin 2: delta [nmaps][2][nrings][mmax + 1] (Q, U) to alm [nmaps][2][nalm] (E, B), in
// tc_anal_partial_bytes(p, 2 nmaps) of scratch
cudaError_t launch_spin_anal_tc(const Plan &p, const double2 *delta, double2 *alm, void *partial, int nmaps,
                                cudaStream_t st, int *nlaunch)
{
    return anal_tc(p, true, delta, alm, partial, 2 * nmaps, st, nlaunch);
}

namespace {
SHT_CHECK_TAKE_DEF(take_check)
}  // namespace
cudaError_t take_check_word_tc_anal(int *w) { return take_check(w); }

}  // namespace sht
