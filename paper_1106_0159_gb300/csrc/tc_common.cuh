// Pieces shared by the tensor-core Legendre kernels (legendre_tc.cu, legendre_tc_anal.cu): the digit
// split, the tcgen05 wrappers, the bounded waits and the recurrence warps.  Included inside each
// file's anonymous namespace, so every translation unit keeps its own internal copy.
//
// Digits.  A value v with |v| < 2^E is cut into S = 8 balanced base-256 digits,
//     v = 2^E sum_s d_s 2^(-6 - 8 s),  |d_0| <= 64, -128 <= d_s < 128 (s > 0),
// 62 bits below 2^E (truncated), so values down to 2^-9 of the scale keep their whole FP64
// significand.  Digits are held in fp16 as d_s 2^-9 (8 significant bits, exact); a product of two
// digits is d d' 2^-18 and tcgen05.mma (kind::f16) adds products in FP32.  A sum of products is
// exact while it stays below 2^24 in units of one digit product.  With products of digit pairs
// i + j <= 7 kept, a term y x is off by less than 2^-57 of max |y| max |x|.
//
// Why base 256 in fp16: the base-128 digits in bf16 that it replaced took a shift, a mask, a
// float add and half a byte permute per digit and kept 48 bits in seven digits.  A base-256 field is
// a byte: byte permutes put the same digit of two values into the two halves of a word, where the
// fields are subnormal halves (u 2^-24), and one HFMA2 turns both into d 2^-9.
#pragma once

#include "recurrence.cuh"

constexpr int TC_T = 128;                // slots per CTA = MMA M
constexpr int TC_S = 8;                  // digits per operand
constexpr int TC_B = 62;                 // bits kept below 2^E
constexpr int TC_CH = 32;                // l per chunk: 16 even + 16 odd l - m
constexpr long long WAIT_POLLS = 1ll << 26;
constexpr int TC_EZERO = 3000;           // scale exponent of an all-zero column or row: every digit 0
constexpr int TC_ETINY = 100, TC_EHUGE = 1990;  // a column whose maximum has a biased exponent above EHUGE
                                         // (analysis: or below ETINY) is left to the plain FP64 sums

// exponent field of v, 1 if v is a nonzero subnormal (0 for zero only)
__device__ __forceinline__ int dexp_nonzero(double v)
{
    const uint32_t hi = (uint32_t)__double2hiint(v) << 1, lo = (uint32_t)__double2loint(v);
    return max((int)(hi >> 21), (hi | lo) != 0u ? 1 : 0);
}

// v 2^(B - E) truncated to an integer F, plus 128 in every 8-bit field: byte s (from the top) of
// the result is d_s + 128.  Integer pipe only (a conversion would take an FP64 issue slot).
__device__ __forceinline__ uint2 digit_fields(double v, int E)
{
    const uint32_t hi = (uint32_t)__double2hiint(v), lo = (uint32_t)__double2loint(v);
    const int ex = (int)((hi >> 20) & 0x7ffu);
    const uint32_t mh = (__funnelshift_l(lo, hi, 10) & 0x3FFFFFFFu) | 0x40000000u;  // significand, top bit 62
    const unsigned long long M = ((unsigned long long)mh << 32) | (lo << 10);
    const int sh = min((1085 - TC_B) + E - ex, 63);      // >= 1 for |v| < 2^E; 63 leaves 0
    const unsigned long long F = M >> sh;
    const uint32_t s = (uint32_t)((int)hi >> 31);
    const unsigned long long Fs = ((unsigned long long)((uint32_t)(F >> 32) ^ s) << 32) | ((uint32_t)F ^ s);
    const unsigned long long G = Fs + (((unsigned long long)0x80808080u << 32) | (0x80808080u - s));
    return make_uint2((uint32_t)G, (uint32_t)(G >> 32));
}

// two fields (bytes 0 and 2 of x, subnormal halves u 2^-24) to the two digits (u - 128) 2^-9
__device__ __forceinline__ uint32_t fields_to_digits(uint32_t x)
{
    uint32_t r;
    asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(x), "r"(0x78007800u), "r"(0xB400B400u));
    return r;
}

// digits 4 h .. 4 h + 3 of two values from their field words: (digit of a, digit of b) as fp16 pairs
__device__ __forceinline__ void digit_quads(uint32_t a, uint32_t b, uint32_t out[4])
{
    const uint32_t t1 = __byte_perm(a, b, 0x7362), t0 = __byte_perm(a, b, 0x5140);
    out[0] = fields_to_digits(__byte_perm(t1, 0u, 0x4342));
    out[1] = fields_to_digits(__byte_perm(t1, 0u, 0x4140));
    out[2] = fields_to_digits(__byte_perm(t0, 0u, 0x4342));
    out[3] = fields_to_digits(__byte_perm(t0, 0u, 0x4140));
}
__device__ __forceinline__ void digit_pairs(uint2 a, uint2 b, uint32_t out[TC_S])
{
    digit_quads(a.y, b.y, out);
    digit_quads(a.x, b.x, out + 4);
}

// the digit-product sum of an accumulator value, an integer below 2^24
__device__ __forceinline__ int class_sum(float acc) { return __float2int_rn(acc * 262144.0f); }

// T 2^e rounded to nearest (ties away), integer pipe only and without branches, so that several of
// them overlap; a result below the normal range is 0, or with SUB a subnormal (the exponents used here
// cannot exceed the range)
template <bool SUB = false>
__device__ __forceinline__ double i64_to_double(long long T, int e)
{
    const long long s = T >> 63;
    unsigned long long a = (unsigned long long)((T ^ s) - s);
    const uint32_t ah = (uint32_t)(a >> 32), al = (uint32_t)a;
    const int lz = ah ? __clz((int)ah) : 32 + __clz((int)al);
    a <<= (lz & 63);                                       // leading one at bit 63
    const int ex = 1023 + 63 - lz + e;                     // biased exponent of the leading one
    if constexpr (SUB) {
        const int d = max(1 - ex, 0);                      // bits lost below the normal range
        a >>= 10 + min(d, 53);
        const unsigned long long mant = (a >> 1) + (a & 1ull);
        const unsigned long long r = (((unsigned long long)(uint32_t)(ex + d - 1) << 52) + mant) | ((unsigned long long)s << 63);
        return __longlong_as_double((long long)((T != 0 && d <= 53) ? r : 0ull));
    }
    const unsigned long long mant = (a >> 11) + ((a >> 10) & 1ull);  // may carry into 2^53
    const unsigned long long r = (((unsigned long long)(uint32_t)(ex - 1) << 52) + mant) | ((unsigned long long)s << 63);
    return __longlong_as_double((long long)((T != 0 && ex > 0) ? r : 0ull));
}

// (hi + lo 2^-32) 2^e, |hi| < 2^51, |lo| < 2^62: lo's carry into hi, then as many of its 32 bits as the
// 64-bit word has room for (at least 55 significant bits in all)
__device__ __forceinline__ double pair_to_double(long long hi, long long lo, int e)
{
    hi += lo >> 32;
    const long long r = lo & 0xFFFFFFFFll;
    const long long m = hi < 0 ? -hi : hi;
    const int sh = m < (1ll << 30) ? 32 : m < (1ll << 38) ? 24 : m < (1ll << 44) ? 18 : 11;
    return i64_to_double<true>(hi * (1ll << sh) + (r >> (32 - sh)), e - sh);
}

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// tcgen05 shared-memory matrix descriptor: K-major, no swizzle; lbo = byte stride between core
// matrices along K, sbo = along M/N; version 1.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = (uint64_t)((saddr & 0x3FFFF) >> 4);
    d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
    d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
    d |= (uint64_t)1 << 46;
    return d;
}

// kind::f16 instruction descriptor: F32 accumulate, F16 A and B, both K-major, M = 128
template <int N>
__device__ __forceinline__ uint32_t umma_idesc()
{
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

// 1 in one lane of the (converged) warp, 0 in the others
__device__ __forceinline__ uint32_t elect_one()
{
    uint32_t e;
    asm volatile("{\n .reg .pred p;\n .reg .b32 r;\n elect.sync r|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}"
                 : "=r"(e));
    return e;
}

// the MMA and the commit issued by the lane with issue != 0 while the whole warp runs the code, so
// that descriptors and addresses stay warp-uniform
__device__ __forceinline__ void umma_f16_by(uint32_t issue, uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                            uint32_t acc)
{
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 q, %5, 0;\n"
        " @q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(acc), "r"(issue));
}

__device__ __forceinline__ void umma_commit_by(uint32_t issue, uint64_t *mbar)
{
    asm volatile(
        "{\n .reg .pred q;\n setp.ne.b32 q, %1, 0;\n"
        " @q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}" ::"r"(smem_u32(mbar)),
        "r"(issue));
}

__device__ __forceinline__ void mbar_init(uint64_t *mbar, int count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t *mbar)
{
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(smem_u32(mbar)) : "memory");
}

// bounded wait for completion of the given phase parity; false on timeout
__device__ __forceinline__ bool mbar_wait(uint64_t *mbar, uint32_t parity)
{
    const uint32_t a = smem_u32(mbar);
    for (long long it = 0; it < WAIT_POLLS; ++it) {
        uint32_t done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
            : "=r"(done)
            : "r"(a), "r"(parity)
            : "memory");  // acquire: no shared-memory access moves above a successful wait
        if (done) return true;
        if (it > 64) __nanosleep(32);
    }
    return false;
}

// named barriers (id 0 is __syncthreads): count = threads taking part, a multiple of 32
__device__ __forceinline__ void bar_sync(int id, int count)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int count)
{
    asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(count) : "memory");
}
__device__ __forceinline__ bool bar_red_and(int id, int count, bool pred)
{
    uint32_t r;
    asm volatile(
        "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred q, %2, %3, p;\n selp.u32 %0, 1, 0, q;\n}"
        : "=r"(r)
        : "r"((uint32_t)pred), "r"(id), "r"(count)
        : "memory");
    return r != 0;
}

// FULL, EMPTY: one per stage; EPI: two
enum : int { BAR_FULL = 2, BAR_EMPTY = 4, BAR_SPLIT = 6, BAR_PREP = 7, BAR_STAGED = 8, BAR_EPI = 9 };

constexpr int TC_NT = 3 * TC_T;  // recurrence (128) and split (256) threads of a tensor-core CTA
constexpr int TC_ABUF = 4 * TC_CH * 8;  // bytes of the recurrence warps' coefficient buffers

struct TcArgs {
    const double2 *alm;      // synthesis: [nmaps][nalm], first map of this group
    double2 *delta;          // [nmaps][nrings][mmax+1] (synthesis: written; analysis: read)
    const int *slotN, *slotS;
    const double *u, *s;
    const double *alpha, *cfac;
    const double3 *rein;     // Reinsch coefficients for m <= mR (polar blocks)
    const double4 *tab;      // spin: (alpha, alpha (1 + g), alpha (1 - g), c) per (l, m)
    const double *start;     // spin: [mmax+1] start coefficients S_m
    int sig;                 // spin: this pass's sign, +1 or -1
    const int *mflag;        // [mmax+1] 1 for the m this plan computes (null: all)
    const int *Ey;           // [mmax+1][nblk] scale exponent of y per slot block: the largest of its slots'
    const int *first;        // [mmax+1][nblk] first chunk with a kept y value (nch: none)
    const double2 *ck_y;     // [mmax+1][nblk][128] recurrence state at chunk first
    const int *ck_k;         // [mmax+1][nblk][128] rescaling exponents k there, with the slot's scale (slot_state)
    int *Ea;                 // synthesis: [mmax+1][N] scale exponent of c a
    int *fix;                // analysis: [mmax+1][16] 1: the map's column of this m is left to the plain FP64 sums
    int *reach, *size;       // synthesis: [mmax+1][16] each, the same decided from them (synth_marked)
    const uint16_t *Yl;      // synthesis: [nalm] exponent field of the largest |y_l| of the grid (tc_top_kernel)
    const int64_t *chunk_base;  // [mmax+1] first chunk of each m
    const int *chunk_m;      // [total chunks] m of each chunk
    uint4 *bdig;             // synthesis: [chunks of the slab][B_CHUNK / 16]
    int64_t chunk0;          // first chunk of the slab
    double2 *partial;        // analysis: [nblk][index - idx0][nmaps] a_lm / c_lm per block
    int *status;             // device status word (bit 0: an mbarrier wait timed out)
    int nslots, nblk, lmax, mmax, nrings, mR, nmaps;
    int64_t nalm;
    int m0;                  // first m of this launch (an m-slab)
    int64_t idx0, nalm_part; // analysis: partial sums hold the indices idx0 .. idx0 + nalm_part - 1
};

// A block runs Reinsch's difference form (see legendre.cu) when its first slot is polar and m <= mR.
__device__ __forceinline__ bool polar_block(const TcArgs &A, int m, int blk)
{
    return m <= A.mR && A.s[blk * TC_T] < POLAR_SIN;
}

// The recurrence of a block: the y form, Reinsch's form (polar blocks), or one sign of the spin-2 pair
// (spin.cu: y_l = alpha_l (x + sig g) y_{l-1} - y_{l-2} from l = max(m, 2) on).
enum : int { REC_Y = 0, REC_REIN = 1, REC_SPIN = 2 };

// Scales.  y of slot r keeps its digits below 2^(E_y - d), where d = min(E_y - E_y(r), 255) and E_y(r) is the
// exponent of the slot's own largest value: the poleward slots of a block lie many powers of two below
// its equatorward ones at high m, and with one scale for all they lost as many bits.  In the
// synthesis a slot is a row of the product and keeps its own exponent; in the analysis the slots are
// summed, so X is divided by the 2^d that y is multiplied with.  With one exponent per block a pixel of
// 1e9 near the pole put errors of 2.7e-10 into the a_lm of m = 50 on HEALPix 256 (plain sums: 1.3e-13),
// although lambda is nothing there.  State word of a slot: k in the low half, d in the high one.
__device__ __forceinline__ int slot_state(int k, int d) { return (d << 16) | (k & 0xffff); }
__device__ __forceinline__ int state_k(int w) { return (int)(short)(w & 0xffff); }
__device__ __forceinline__ int state_d(int w) { return w >> 16; }

// first l of the recurrence: its chunks of 32 start here
template <int KIND>
__device__ __forceinline__ int first_l(int m)
{
    return KIND == REC_SPIN ? max(m, 2) : m;
}

// Recurrence coefficients of one l (the lane's own): (alpha, -, -, -), Reinsch (beta, rho, b0, 1 / c) or
// spin (alpha, alpha (1 + sig g), -, -); all zero above lmax.
struct RecCoef {
    double a, rh, b0, ci;
};
template <int KIND>
__device__ __forceinline__ RecCoef load_coef(const TcArgs &A, int64_t base, int m, int l)
{
    RecCoef c{0.0, 0.0, 0.0, 0.0};
    if (l <= A.lmax) {
        const int64_t ix = base + (l - m);
        if (KIND == REC_SPIN) {
            const double4 t = A.tab[ix];
            c.a = t.x;
            c.rh = A.sig > 0 ? t.y : t.z;
        } else if (KIND == REC_REIN) {
            const double3 t = A.rein[ix];
            c = RecCoef{t.x, t.y, t.z, 1.0 / A.cfac[ix]};
        } else {
            c.a = A.alpha[ix];
        }
    }
    return c;
}

// one Reinsch step: lambda_l and the difference D_l from those of l - 1; returns lambda_l / c_l
__device__ __forceinline__ double rein_step(double be, double rh, double b0, double ci, double u, double &lam, double &D)
{
    const double g = fma(-be, u, b0);
    D = fma(rh, D, fma(g, lam, D));
    lam += D;
    return lam * ci;
}

// The recurrence warps (threads 0-127, thread r = slot r of the block) of the tensor-core kernels:
// from the plan-time checkpoint at chunk cfirst (earlier chunks hold only dropped values) they run
// the recurrence and write each chunk's 32 values (0 where dropped) to one of NST (2 or 1) y stages, laid out
// [32 rows][YS doubles].  Row of step j: j, or with PAR the 16 even steps first.  Coefficients come
// from a register of lane j (warp shuffle), loaded one chunk ahead.  Stages are handed over with
// named barriers over all TC_NT threads: FULL (arrive here, the split warps wait) and EMPTY (the
// split warps arrive, wait here, only where a later chunk reuses the stage).
//
// This is the chain that bounds both kernels: 2 FP64 instructions per step, each holding one of the
// four quarter-SM FP64 pipes for 64 cycles a warp, so the warp must always have the next one ready.
// Chunks in which a lane of the warp may still be scaled (k < 0) or that run Reinsch's form take a
// plain loop with the tests; once every lane is at k = 0 it stays there, and the rest runs without
// tests in groups of G steps: the factors alpha x = alpha (1 - u) of the next group are computed
// between the dependent steps of this one, the coefficients of those factors are read from the warp's
// own small shared buffer a group earlier still (a read waits behind the split warps' traffic), and
// the values of the previous group are stored meanwhile (a store of this group's would wait for its
// last step).  Alone, a step takes 145 cycles (the pipe: 128); with the stores in their own group
// 152, with the tests and selects of dropped values 162.  G = 8, or 4 where registers are short.
template <bool PAR>
__device__ __forceinline__ int y_row(int j)
{
    return PAR ? (j & 1) * (TC_CH / 2) + (j >> 1) : j;
}

template <int KIND, bool PAR, int YS, int G, int NST = 2>
__device__ __forceinline__ void recurrence_warps(const TcArgs &A, int m, int blk, int r, bool active, int64_t base,
                                                 int nch, int cfirst, double *ybuf, double *abuf)
{
    constexpr bool REIN = KIND == REC_REIN, SPIN = KIND == REC_SPIN;
    const int lane = r & 31, lb = first_l<KIND>(m);
    double u = 0.0, y1 = 0.0, y2 = 0.0;
    int k = 0;
    if (active) {
        u = A.u[blk * TC_T + r];
        const int64_t ci = (int64_t)(m * A.nblk + blk) * TC_T + r;
        const double2 st = A.ck_y[ci];
        y1 = st.x;
        y2 = st.y;
        k = state_k(A.ck_k[ci]);
    }
    abuf += (r >> 5) * TC_CH;
    RecCoef cur = load_coef<KIND>(A, base, m, lb + TC_CH * cfirst + lane);
    int c = cfirst;
    for (; c < nch && (REIN || __any_sync(0xffffffffu, k < 0)); ++c) {
        const RecCoef nxt = load_coef<KIND>(A, base, m, lb + TC_CH * (c + 1) + lane);
        const int q = c - cfirst;
        double *yb = ybuf + (size_t)(q & (NST - 1)) * TC_CH * YS + r;
        if (q >= NST) bar_sync(BAR_EMPTY + (q & (NST - 1)), TC_NT);  // the split warps read chunk q - NST
        bool drop = false;
#pragma unroll 1
        for (int j0 = 0; j0 < TC_CH; j0 += 4) {
            if ((j0 & 15) == 0) drop = __any_sync(0xffffffffu, k < 0) && k < 0;
            double yv[4];
            if (REIN) {
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const double be = __shfl_sync(0xffffffffu, cur.a, j0 + j), rh = __shfl_sync(0xffffffffu, cur.rh, j0 + j);
                    const double b0 = __shfl_sync(0xffffffffu, cur.b0, j0 + j), ci = __shfl_sync(0xffffffffu, cur.ci, j0 + j);
                    yv[j] = rein_step(be, rh, b0, ci, u, y1, y2);
                }
            } else {
                double f[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const double a = __shfl_sync(0xffffffffu, cur.a, j0 + j);
                    f[j] = fma(-a, u, SPIN ? __shfl_sync(0xffffffffu, cur.rh, j0 + j) : a);
                }
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const double y = fma(f[j], y1, -y2);
                    y2 = y1;
                    y1 = y;
                    yv[j] = y;
                }
            }
            double *yr = yb + (PAR ? j0 >> 1 : j0) * YS;  // rows of steps j0 .. j0 + 3
#pragma unroll
            for (int j = 0; j < 4; ++j) yr[y_row<PAR>(j) * YS] = drop ? 0.0 : yv[j];
            if ((j0 & 15) == 12 && drop && max(dexp(y1), dexp(y2)) > RESCALE_THR) {
                y1 *= 0x1p-512;
                y2 *= 0x1p-512;
                k += 1;
            }
        }
        bar_arrive(BAR_FULL + (q & (NST - 1)), TC_NT);
        cur = nxt;
    }
    if (REIN || c >= nch) return;
    // factors of this group, coefficients of the next (spin: a second one), values of the previous
    double ax[G], al[G], al1[SPIN ? G : 1], pv[G];
    double2 *abuf2 = reinterpret_cast<double2 *>(abuf);  // spin: 16 steps of coefficient pairs
    if (SPIN) {
        if (lane < 16) abuf2[lane] = make_double2(cur.a, cur.rh);
    } else {
        abuf[lane] = cur.a;
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < G; ++j) {
        if (SPIN) {
            const double2 t = abuf2[j], w = abuf2[G + j];
            ax[j] = fma(-t.x, u, t.y);
            al[j] = w.x;
            al1[SPIN ? j : 0] = w.y;
        } else {
            const double a = abuf[j];
            ax[j] = fma(-a, u, a);
            al[j] = abuf[G + j];
        }
        pv[j] = 0.0;
    }
    double *pp = ybuf + r;  // where the previous group goes
    for (const int c0 = c; c < nch; ++c) {
        const RecCoef nxt = load_coef<KIND>(A, base, m, lb + TC_CH * (c + 1) + lane);
        const int q = c - cfirst;
        double *yb = ybuf + (size_t)(q & (NST - 1)) * TC_CH * YS + r;
#pragma unroll
        for (int j0 = 0; j0 < TC_CH; j0 += G) {
            // coefficients that are all read make room for the next ones: a chunk's 32, or (spin) 16 pairs
            if (SPIN && ((j0 + 2 * G) & 15) == 0) {
                const bool up = j0 + 2 * G < TC_CH;  // steps 16-31 of this chunk, else 0-15 of the next
                __syncwarp();
                if ((lane >= 16) == up) abuf2[lane & 15] = up ? make_double2(cur.a, cur.rh) : make_double2(nxt.a, nxt.rh);
                __syncwarp();
            } else if (!SPIN && j0 == TC_CH - 2 * G) {
                __syncwarp();
                abuf[lane] = nxt.a;
                __syncwarp();
            }
            double yv[G], axn[G], aln[G], al1n[SPIN ? G : 1];
            if (SPIN) {
#pragma unroll
                for (int j = 0; j < G; ++j) {
                    const double2 t = abuf2[((j0 + 2 * G) & 15) + j];
                    aln[j] = t.x;
                    al1n[SPIN ? j : 0] = t.y;
                }
            } else {
                const double2 *as = reinterpret_cast<const double2 *>(abuf + ((j0 + 2 * G) & 31));
#pragma unroll
                for (int j = 0; j < G / 2; ++j) {
                    const double2 t = as[j];
                    aln[2 * j] = t.x;
                    aln[2 * j + 1] = t.y;
                }
            }
            const bool store = j0 > 0 || c > c0;
#pragma unroll
            for (int j = 0; j < G; ++j) {
                const double y = fma(ax[j], y1, -y2);
                y2 = y1;
                y1 = y;
                yv[j] = y;
                axn[j] = fma(-al[j], u, SPIN ? al1[SPIN ? j : 0] : al[j]);
                if (store) pp[y_row<PAR>(((j0 - G) & 31) + j) * YS] = pv[j];  // steps j0 - G .. j0 - 1
            }
            if (j0 == 0) {
                if (c > c0) bar_arrive(BAR_FULL + ((q - 1) & (NST - 1)), TC_NT);
                if (q >= NST) bar_sync(BAR_EMPTY + (q & (NST - 1)), TC_NT);  // the split warps read chunk q - NST
                pp = yb;
            }
#pragma unroll
            for (int j = 0; j < G; ++j) {
                ax[j] = axn[j];
                al[j] = aln[j];
                if (SPIN) al1[SPIN ? j : 0] = al1n[SPIN ? j : 0];
                pv[j] = yv[j];
            }
        }
        cur = nxt;
    }
#pragma unroll
    for (int j = 0; j < G; ++j) pp[y_row<PAR>(TC_CH - G + j) * YS] = pv[j];
    bar_arrive(BAR_FULL + ((nch - 1 - cfirst) & (NST - 1)), TC_NT);
}
