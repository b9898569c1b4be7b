// gke_digits.cu -- FP64 correlator on the 5th-generation tensor cores by exact
// digit products (error-free splitting of a matrix product: Ozaki, Ogita,
// Oishi, Rump, Numer. Algorithms 59 (2012) 95-118).
//
// The FP64 pipe does 2 fused multiply-adds per clock and SM, the tensor cores
// 4096 in FP16: the 36 digit products that replace one FP64 product below
// still leave a factor of 50.
//
// Splitting.  All values of a row (wavenumber k, wall-normal point y) of one
// group of fields -- velocities; products; pressure -- share the exponent E
// of the largest of them over the batch's snapshots, |x| < 2^E.  Each value
// becomes the integer round(x 2^(61 - E)) and that its eight balanced base-256
// digits s_0 (|s_0| <= 33) .. s_7 (in [-128, 127]), exact in FP16.  61 bits
// below the row's largest value hold every bit of an FP64 value down to
// 2^-8 of that maximum; smaller values lose bits below 2^-61 of it, eight
// binary orders under the FP64 rounding of the sums they enter.
//
// Products.  With the digit products s_i t_j summed over the terms and
// snapshots of a contraction by order d = i + j (v_d, d <= 7; the orders
// above are below 2^-64 of the largest product),
//   sum a b = 2^(E_a + E_b - 34) [ (v_0 .. v_3) + 2^-32 (v_4 .. v_7) ],
//   (w_0 .. w_3) = 2^24 w_0 + 2^16 w_1 + 2^8 w_2 + w_3.
// A sum v_d runs over at most 4 terms x 16 snapshots x 2 real products, so
// |v_d| <= max(1, d) 4 2^19 < 2^24 (and < 2^22 for d <= 2, where s_0 enters every
// or all but one product): the FP32 accumulation in tensor memory is exact.  The eight sums are joined in a 64-bit integer and rounded to FP64
// once, all in integer arithmetic.  A sum over up to 16 snapshots therefore
// carries one rounding where the FMA chain carries 32 per term; further
// snapshots come in groups of 16, added in FP64.
//
// Mapping.  CTA = one SM, persistent over items (k, 128-row tile of y, tile of
// CW <= 32 columns y').  Per term and digit pair (i, j):
//   mma(A = ar_i, B = [br_j | bi_j], N = 2 CW) -> Re += ar br, Im += ar bi
//   mma(A = ai_i, B = [bi_j | -br_j], N = 2 CW) -> Re += ai bi, Im -= ai br
// (M = 128, K = 16 snapshots).  The B block holds the rows br, bi, -br, so
// both views are windows of it.  The orders run in two passes of four TMEM
// accumulators (d = 4..7, then 0..3): two sets fit in 512 columns, so the
// epilogue of one pass overlaps the MMAs of the next; the low half of a sum
// waits in registers as a 64-bit integer.  N = 64 keeps two sets in TMEM at
// the price of reading A from shared memory every 32 columns (96 clocks a
// digit pair against 64 of tensor work).
//   warp 0: bulk copies, the A digits of a term per stage of a ring, B blocks
//           into four slots by a schedule made on the host;
//   warp 1: MMAs;   the others: epilogue, a warp per TMEM lane quarter and 8 columns.
// Every wait is bounded (gke_split.cu has the same protocol).
//
// Measured, correlate stage (operands, contractions; FMA kernel -> here):
// 256 x 256 x 65, 16 snapshots 232.8 -> 33.9 ms, of which the operand kernel 6.5
// and the MMAs alone 23 (smem reads of A and B: 18.5 by count), which bound it
// with the epilogue (conversions and integer adds) close behind; 128 x 128 x 65,
// 32 snapshots 117.4 -> 18.2 ms.  Errors against 64-bit references equal the
// FMA kernel's or are below.
#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

#include "gke_digits.h"
#include "gke_kernels.h"
#include "gke_tc.cuh"

namespace gke {

constexpr int DG_S = 8;                    // digits
constexpr int DG_KS = 16;                  // snapshots per batch (one MMA K step)
constexpr int DG_MAXST = 8;                // A stages (one field: all digits, re and im), at most
constexpr int DG_NB = 4;                   // B slots
constexpr int dg_epi(int CW) { return CW / 2; }                    // epilogue warps: 8 columns x 32 rows each
constexpr int dg_threads(int CW) { return 64 + 32 * dg_epi(CW); }
constexpr int DG_SM_BAR = 512;             // barriers, then the B slots, then the A stages
constexpr int DG_SM = 232448;
constexpr int DG_MAXSTEP = 112, DG_MAXJOB = 16, DG_MAXF = 16, DG_MAXT = 4, DG_MAXG = 4;

enum { DF_NEG = 1, DF_LOAD = 2, DF_FREE = 4, DF_FIRST = 8, DF_LAST = 16, DF_HI = 32 };
// one term of one pass: conj(A field fa) B field fb; B in slot, loaded before
// (DF_LOAD) or released after it (DF_FREE)
struct DgStep { unsigned char fa, fb, slot, flags; };
// a contraction: exponent groups of its A and B fields, output index, power of two
struct DgJob { signed char ga, gb, out, pad; int e; };

struct DgBars {
    uint64_t full[DG_MAXST], empty[DG_MAXST], bfull[DG_NB], bempty[DG_NB], acc_full[2], acc_empty[2], drain;
    uint32_t tmem;
    int abort;
};
static_assert(sizeof(DgBars) <= DG_SM_BAR, "barrier area");

struct DgShape {
    int n, RT, MT, cov, NT, CW, nrow;      // rows per A tile, A tiles, rows they cover, column tiles, E rows
};

struct DgArgs {
    const __half* Aop; const __half* Bop; const int* E;
    DgShape s;
    int nfa, nfb, ngrp, tpk;               // fields of A, of B, exponent groups, tiles per wavenumber
    long long nitems;
    int nstep, njob;
    DgStep step[DG_MAXSTEP];
    DgJob job[DG_MAXJOB];
    int mul[4];                            // 2^5, 2^13, 2^21, 2^29 (mad_wide)
    int Kc, beta;
    zd* raw;
    int* err;
};

// A stages that fit beside the B slots
constexpr int dg_nst(int RT, int CW)
{
    const int n = (DG_SM - DG_SM_BAR - DG_NB * DG_S * 3 * CW * DG_KS * 2) / (DG_S * 2 * RT * DG_KS * 2);
    return n < DG_MAXST ? n : DG_MAXST;
}

static DgShape dg_shape(int n)
{
    DgShape s{};
    s.n = n;
    // rows of an A tile: the instantiated heights (short tiles copy less; an MMA
    // always takes 128 rows, reading past a short tile into lanes nobody reads)
    s.MT = 1;
    s.cov = n;
    s.RT = n <= 40 ? 40 : n <= 72 ? 72 : 128;
    if (n > 128) {
        const bool thin = n % 128 >= 1 && n % 128 <= 4;                           // thin remainder: k_dg_rows
        s.MT = thin ? n / 128 : (n + 127) / 128;
        s.cov = thin ? 128 * s.MT : n;
    }
    // column tiles of 24 or 32: an MMA takes 32 + CW / 2 clocks of shared-memory reads
    const int n24 = (n + 23) / 24, n32 = (n + 31) / 32;
    s.CW = n24 * 44 <= n32 * 48 ? 24 : 32;
    s.NT = s.CW == 24 ? n24 : n32;
    s.nrow = 128 * ((std::max(s.MT * s.RT, s.NT * s.CW) + 127) / 128);
    return s;
}
static size_t dg_a_halves(const DgShape& s) { return (size_t)s.MT * DG_S * 2 * s.RT * DG_KS; }      // per field and k
static size_t dg_b_halves(const DgShape& s) { return (size_t)s.NT * DG_S * 3 * s.CW * DG_KS; }

// ------------------------------------------------------------- digit operands
// field src of X (times 2^wexp), exponent group, A and B operand index (-1: not used)
struct DgField { short src; signed char wexp, grp; short ia, ib; };
struct DgPrep {
    DgShape s;
    int nf, nfa, nfb, ngrp, ns, s0, nsX, Nk, k0;
    DgField f[DG_MAXF];
    const zd* X;
    __half* Aop; __half* Bop; int* E;
};

// round(x 2^sh) for |x| 2^sh < 2^61, in integer arithmetic (a conversion would
// run on the FP64 pipe)
__device__ __forceinline__ unsigned long long dg_fixed(double x, int sh)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const int ef = (int)(b >> 52) & 0x7ff;
    unsigned long long m = b & 0xfffffffffffffull;
    if (ef) m |= 1ull << 52;
    const int s = max(ef, 1) - 1075 + sh;
    unsigned long long r;
    if (s >= 0) r = m << min(s, 63);
    else r = (s < -54) ? 0ull : (m + (1ull << (-s - 1))) >> (-s);
    return (b >> 63) ? 0ull - r : r;
}
// the biased digits of a fixed-point value: byte 7 - i holds digit i + 128
__device__ __forceinline__ unsigned long long dg_bytes(unsigned long long v)
{
    return (v + 0x0080808080808080ull) ^ 0x8000000000000000ull;
}
// digits of two values (byte c of a and b) as a pair of FP16 numbers: 1024 + byte, minus 1152
__device__ __forceinline__ uint32_t dg_pair(uint32_t a, uint32_t b, int c)
{
    const uint32_t p = (__byte_perm(a, b, c | (4 << 4) | ((c + 4) << 8) | (4 << 12)) & 0x00ff00ffu) | 0x64006400u;
    const __half2 h = __hsub2(*(const __half2*)&p, __half2half2(__ushort_as_half(0x6480)));
    return *(const uint32_t*)&h;
}

// CTA = one (wavenumber, exponent group, 128 rows): the rows' exponents, then
// the digit blocks of the group's fields.  Thread = one row x 8 snapshots, the
// 16 bytes of a core-matrix row; stores are contiguous over the rows.  Bound by
// memory: X is read twice (the second time from L2), 32 bytes of digits are
// written per A value.
__global__ void __launch_bounds__(256)
k_dg_prep(const __grid_constant__ DgPrep a)
{
    __shared__ int s_hi[128];
    const int nb = a.s.nrow / 128;
    int b = blockIdx.x;
    const int mb = b % nb; b /= nb;
    const int g = b % a.ngrp, k = b / a.ngrp;
    const int r = threadIdx.x & 127, kc = threadIdx.x >> 7;
    const int y = mb * 128 + r;
    if (threadIdx.x < 128) s_hi[threadIdx.x] = 0;
    __syncthreads();
    const int e0 = kc * 8, ne = y < a.s.n ? max(0, min(8, a.ns - e0)) : 0;
    int hi = 0;
    for (int f = 0; f < a.nf; ++f) {
        const DgField fd = a.f[f];
        if (fd.grp != g) continue;
        const zd* src = a.X + (((long long)fd.src * a.Nk + a.k0 + k) * a.nsX + a.s0 + e0) * a.s.n + y;
        for (int e = 0; e < ne; ++e) {
            const zd v = src[(long long)e * a.s.n];
            const int h = max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff);
            if (h >= 0x00100000) hi = max(hi, h + fd.wexp * 0x00100000);
        }
    }
    atomicMax(&s_hi[r], hi);
    __syncthreads();
    const int E = max(s_hi[r] >> 20, 1) - 1022;              // |x| < 2^E
    if (kc == 0) a.E[((long long)k * a.ngrp + g) * a.s.nrow + y] = E;
    const bool arow = mb < a.s.MT && r < a.s.RT && y < a.s.cov, astore = mb < a.s.MT && r < a.s.RT;
    const int c = y / a.s.CW, rc = y - c * a.s.CW;
    const bool bstore = c < a.s.NT;
    for (int f = 0; f < a.nf; ++f) {
        const DgField fd = a.f[f];
        if (fd.grp != g) continue;
        const zd* src = a.X + (((long long)fd.src * a.Nk + a.k0 + k) * a.nsX + a.s0 + e0) * a.s.n + y;
        unsigned long long dre[8], dim[8];
        #pragma unroll
        for (int e = 0; e < 8; ++e) {
            zd v = mk(0.0, 0.0);
            if (e < ne) v = src[(long long)e * a.s.n];
            dre[e] = dg_bytes(dg_fixed(v.x, 61 - E + fd.wexp));
            dim[e] = dg_bytes(dg_fixed(v.y, 61 - E + fd.wexp));
        }
        __half* da = fd.ia < 0 || !astore ? nullptr
                   : a.Aop + (((long long)k * a.nfa + fd.ia) * a.s.MT + mb) * (long long)(DG_S * 2 * a.s.RT * DG_KS)
                     + cm_index(r, e0, a.s.RT);
        __half* db = fd.ib < 0 || !bstore ? nullptr
                   : a.Bop + (((long long)k * a.nfb + fd.ib) * a.s.NT + c) * (long long)(DG_S * 3 * a.s.CW * DG_KS);
        const int b0 = cm_index(rc, e0, 3 * a.s.CW), bw = (a.s.CW >> 3) << 6;
        #pragma unroll
        for (int i = 0; i < DG_S; ++i) {
            uint4 re, im;
            uint32_t* pr = (uint32_t*)&re;
            uint32_t* pi = (uint32_t*)&im;
            #pragma unroll
            for (int h = 0; h < 4; ++h) {
                const int w = 32 * (i < 4), cc = (7 - i) & 3;
                pr[h] = dg_pair((uint32_t)(dre[2 * h] >> w), (uint32_t)(dre[2 * h + 1] >> w), cc);
                pi[h] = dg_pair((uint32_t)(dim[2 * h] >> w), (uint32_t)(dim[2 * h + 1] >> w), cc);
            }
            if (da) {
                const uint4 z = make_uint4(0, 0, 0, 0);
                *(uint4*)(da + (long long)(2 * i) * a.s.RT * DG_KS) = arow ? re : z;
                *(uint4*)(da + (long long)(2 * i + 1) * a.s.RT * DG_KS) = arow ? im : z;
            }
            if (db) {
                __half* d = db + (long long)i * 3 * a.s.CW * DG_KS + b0;
                *(uint4*)d = re;
                *(uint4*)(d + bw) = im;
                *(uint4*)(d + 2 * bw) = make_uint4(re.x ^ 0x80008000u, re.y ^ 0x80008000u, re.z ^ 0x80008000u,
                                                   re.w ^ 0x80008000u);
            }
        }
    }
}

// ------------------------------------------------------------- tensor-core kernel
// loads of one accumulator group: Re and Im, four orders, four columns (dg_ready waits for them)
__device__ __forceinline__ void dg_tmem(uint32_t t, int cw, uint32_t (&r)[2][4][4])
{
    #pragma unroll
    for (int d = 0; d < 4; ++d) {
        tmem_ld4(t + 64 * d, r[0][d]);
        tmem_ld4(t + 64 * d + cw, r[1][d]);
    }
}
// the wait names the registers, so that no use moves above it
__device__ __forceinline__ void dg_ready(uint32_t (&r)[2][4][4])
{
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0][0][0]), "+r"(r[0][0][1]), "+r"(r[0][0][2]), "+r"(r[0][0][3]),
                   "+r"(r[0][1][0]), "+r"(r[0][1][1]), "+r"(r[0][1][2]), "+r"(r[0][1][3]),
                   "+r"(r[0][2][0]), "+r"(r[0][2][1]), "+r"(r[0][2][2]), "+r"(r[0][2][3]),
                   "+r"(r[0][3][0]), "+r"(r[0][3][1]), "+r"(r[0][3][2]), "+r"(r[0][3][3]) :: "memory");
    asm volatile("" : "+r"(r[1][0][0]), "+r"(r[1][0][1]), "+r"(r[1][0][2]), "+r"(r[1][0][3]),
                   "+r"(r[1][1][0]), "+r"(r[1][1][1]), "+r"(r[1][1][2]), "+r"(r[1][1][3]),
                   "+r"(r[1][2][0]), "+r"(r[1][2][1]), "+r"(r[1][2][2]), "+r"(r[1][2][3]),
                   "+r"(r[1][3][0]), "+r"(r[1][3][1]), "+r"(r[1][3][2]), "+r"(r[1][3][3]) :: "memory");
}
// a b + c in 64 bits as one instruction (b a power of two in a register the
// compiler cannot see through; as a constant it becomes a shift and add chain)
__device__ __forceinline__ long long mad_wide(int a, int b, long long c)
{
    long long r;
    asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
    return r;
}
// A sum joined as the integer T = 2^21 (w_0 .. w_3) + 2^-11 (w_4 .. w_7) (w_6 and
// w_7 rounded; one unit is 2^-55 of the largest product),
// (w_0 .. w_3) = 2^24 w_0 + 2^16 w_1 + 2^8 w_2 + w_3, |T| < 2^62.  The epilogue is bound
// by the conversions (16 a clock and SM) and the integer adds (64): sums below
// 2^22 turn integer by an FP32 addition of 1.5 2^23, whose bits are DG_MAGIC + w;
// DG_BIAS takes the offsets of w_0, w_1, w_2 and of w_6 / 8 + w_7 / 2^11 out again.
constexpr float DG_MAGF = 12582912.f;                               // 1.5 2^23
constexpr unsigned long long DG_MAGIC = 0x4B400000ull;              // its bits
constexpr long long DG_BIAS = (long long)(0ull - DG_MAGIC - (DG_MAGIC << 29) - (DG_MAGIC << 37) - (DG_MAGIC << 45));
// orders 4..7 of column j (|w| <= 2^24)
__device__ __forceinline__ long long dg_low(const uint32_t (&r)[4][4], int j, int m13, int m5)
{
    const float g = fmaf(__uint_as_float(r[3][j]), 1.f / 2048.f, fmaf(__uint_as_float(r[2][j]), 1.f / 8.f, DG_MAGF));
    const long long v = mad_wide(__float2int_rz(__uint_as_float(r[1][j])), m5,
                                 mad_wide(__float2int_rz(__uint_as_float(r[0][j])), m13, DG_BIAS));
    return v + (long long)(unsigned long long)__float_as_uint(g);
}
// with the orders 0..3 (|w_0|, |w_1|, |w_2| < 2^22)
__device__ __forceinline__ long long dg_high(const uint32_t (&r)[4][4], int j, long long low, int m21, int m29)
{
    auto bits = [&](int d) { return __float_as_uint(__uint_as_float(r[d][j]) + DG_MAGF); };
    const long long v = mad_wide((int)bits(2), m29, mad_wide(__float2int_rz(__uint_as_float(r[3][j])), m21, low));
    const unsigned up = (unsigned)((unsigned long long)v >> 32) + (bits(0) << 13) + (bits(1) << 5);
    return (long long)(((unsigned long long)up << 32) | (unsigned)v);
}
// t 2^(e - 21) in general
__device__ __noinline__ double dg_value_edge(long long t, int e) { return scalbn((double)t, e - 21); }
// t 2^(e - 21), normalised and rounded to nearest in integer arithmetic (a
// conversion would hold the FP64 pipe of the whole SM for 16 clocks a warp).
// No branch, so that values interleave; edge is raised where the upper
// word is zero or the exponent may leave the normal range (dg_value_edge then).
__device__ __forceinline__ double dg_value(long long t, int e, bool& edge)
{
    unsigned h = (unsigned)((unsigned long long)t >> 32), l = (unsigned)t;
    const unsigned sg = (unsigned)((int)h >> 31);
    const unsigned long long m = ((unsigned long long)t ^ (((unsigned long long)sg << 32) | sg)) + (sg & 1u);
    h = (unsigned)(m >> 32);
    l = (unsigned)m;
    const int lz = __clz((int)h);
    edge |= (h == 0) ? l != 0 : (unsigned)(e + 900) > 1800u;
    const unsigned mh = __funnelshift_l(l, h, lz), ml = l << (lz & 31);
    unsigned rl = __funnelshift_r(ml, mh, 11), rh = (mh >> 11) + ((unsigned)(1022 + 42 - lz + e) << 20);
    const unsigned up = (ml >> 10) & 1u;
    rl += up;
    rh += rl < up;
    return h == 0 ? 0.0 : __hiloint2double((int)(rh | (sg & 0x80000000u)), (int)rl);
}
__device__ __forceinline__ void st_256(zd* p, zd a, zd b)
{
    asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(a.x), "d"(a.y), "d"(b.x), "d"(b.y) : "memory");
}

struct DgItem { int k, mt, c; };
__device__ __forceinline__ DgItem dg_item(const DgArgs& a, long long it)
{
    DgItem u;
    u.k = (int)(it / a.tpk);
    const int r = (int)(it - (long long)u.k * a.tpk);
    u.mt = r / a.s.NT;
    u.c = r - u.mt * a.s.NT;
    return u;
}

// the MMAs of one term in one pass, by one warp in step: the pairs unrolled
// with every operand a constant offset from the stage's, the descriptors'
// upper words fixed.  46 clocks an MMA at CW = 24 (smem: 44); with descriptors
// formed per pair 65, with loops over the pairs 94.
template <int RT, int CW, int DMIN>
__device__ __forceinline__ void dg_pairs(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t first)
{
    const uint32_t alo = (uint32_t)a, ahi = (uint32_t)(a >> 32), blo = (uint32_t)b, bhi = (uint32_t)(b >> 32);
    #pragma unroll
    for (int i = 0; i < DMIN + 4; ++i)
        #pragma unroll
        for (int j = (DMIN > i ? DMIN - i : 0); j <= DMIN + 3 - i; ++j) {
            const uint32_t dd = d + (uint32_t)(i + j - DMIN) * 64u;
            // offsets in 16 bytes: A digit 4 RT, its imaginary part 2 RT; B digit 6 CW, its rows bi CW
            mma_f16_u(dd, alo + i * RT * 4, ahi, blo + j * 6 * CW, bhi, idesc, i == 0 ? first : 1u);       // ar [br | bi]
            mma_f16_u(dd, alo + i * RT * 4 + RT * 2, ahi, blo + j * 6 * CW + CW, bhi, idesc, 1u);         // ai [bi | -br]
        }
}

template <int RT, int CW>
__global__ void __launch_bounds__(dg_threads(CW), 1)
k_dg_corr(const __grid_constant__ DgArgs a)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    DgBars* bars = (DgBars*)smem;
    volatile int* abort = &bars->abort;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    constexpr int NST = dg_nst(RT, CW);
    constexpr uint32_t BDIG = 3 * CW * DG_KS * 2;           // bytes of one B digit
    constexpr uint32_t BSLOT = DG_S * BDIG;
    constexpr uint32_t ADIG = 2 * RT * DG_KS * 2;           // bytes of one A digit (re, im)
    uint8_t* sb = smem + DG_SM_BAR;
    uint8_t* sa = sb + DG_NB * BSLOT;
    if (threadIdx.x == 0) {
        for (int i = 0; i < DG_MAXST; ++i) { mbar_init(&bars->full[i], 1); mbar_init(&bars->empty[i], 1); }
        for (int i = 0; i < DG_NB; ++i) { mbar_init(&bars->bfull[i], 1); mbar_init(&bars->bempty[i], 1); }
        for (int i = 0; i < 2; ++i) { mbar_init(&bars->acc_full[i], 1); mbar_init(&bars->acc_empty[i], dg_epi(CW)); }
        mbar_init(&bars->drain, 1);
        bars->abort = (*(volatile int*)a.err != 0) ? 1 : 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&bars->tmem)),
                     "r"(512) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = bars->tmem;
    auto fail = [&]() { *abort = 1; atomicExch(a.err, 1); };

    if (warp == 0) {
        if (lane == 0) {
            int st = 0, issued = 0;
            uint32_t ph = 0, bph = 0, bany = 0;              // ring phase; per slot: loads so far (parity), any
            for (long long it = blockIdx.x; it < a.nitems && !*abort; it += gridDim.x) {
                const DgItem u = dg_item(a, it);
                for (int q = 0; q < a.nstep; ++q) {
                    const DgStep s = a.step[q];
                    if (s.flags & DF_LOAD) {
                        if (!mbar_wait_ab(&bars->bempty[s.slot], ((bph >> s.slot) & 1u) ^ 1u, abort)) { fail(); goto producer_done; }
                        mbar_expect_tx(&bars->bfull[s.slot], BSLOT);
                        bulk_g2s(sb + s.slot * BSLOT,
                                 a.Bop + (((long long)u.k * a.nfb + s.fb) * a.s.NT + u.c) * (long long)(DG_S * 3 * CW * DG_KS),
                                 BSLOT, &bars->bfull[s.slot]);
                        bph ^= 1u << s.slot;
                        bany |= 1u << s.slot;
                    }
                    const __half* src = a.Aop + (((long long)u.k * a.nfa + s.fa) * a.s.MT + u.mt) *
                                                (long long)(DG_S * 2 * RT * DG_KS);
                    const uint32_t bytes = ((s.flags & DF_HI) ? 4 : DG_S) * ADIG;
                    if (!mbar_wait_ab(&bars->empty[st], ph ^ 1u, abort)) { fail(); goto producer_done; }
                    mbar_expect_tx(&bars->full[st], bytes);
                    bulk_g2s(sa + st * DG_S * ADIG, src, bytes, &bars->full[st]);
                    ++issued;
                    if (++st == NST) { st = 0; ph ^= 1u; }
                }
            }
        producer_done:
            // no copy may be in flight when the CTA exits: the last phase
            // issued on every stage and slot (bounded waits)
            for (int i = 0; i < NST && i < issued; ++i) {
                const int last = issued - 1 - i;
                mbar_wait(&bars->full[last % NST], (uint32_t)((last / NST) & 1));
            }
            for (int i = 0; i < DG_NB; ++i)
                if ((bany >> i) & 1u) mbar_wait(&bars->bfull[i], ((bph >> i) & 1u) ^ 1u);
        }
    } else if (warp == 1) {
        // every lane walks the items (uniform control flow); one issues
        int st = 0, acc = 0;
        uint32_t ph = 0, bph = 0, aph = 0;
        // D = F32, A = B = F16, K-major; N = 2 CW, M = 128
        constexpr uint32_t IDESC = (1u << 4) | ((uint32_t)(2 * CW >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
        constexpr uint32_t NEG_A = 1u << 13;
        const uint32_t alb = (uint32_t)(RT / 8) * 128u, blb = (uint32_t)(3 * CW / 8) * 128u;
        auto wait = [&](uint64_t* b, uint32_t parity) {
            return __all_sync(0xffffffffu, mbar_wait_ab(b, parity, abort));
        };
        bool ok = true;
        for (long long it = blockIdx.x; it < a.nitems && ok; it += gridDim.x) {
            for (int q = 0; q < a.nstep; ++q) {
                const DgStep s = a.step[q];
                if ((s.flags & DF_FIRST) && !wait(&bars->acc_empty[acc], aph ^ 1u)) { ok = false; break; }
                if (s.flags & DF_LOAD) {
                    if (!wait(&bars->bfull[s.slot], (bph >> s.slot) & 1u)) { ok = false; break; }
                    bph ^= 1u << s.slot;
                }
                if (!wait(&bars->full[st], ph)) { ok = false; break; }
                tc_fence_after();
                const uint32_t idesc = IDESC | ((s.flags & DF_NEG) ? NEG_A : 0u);
                const uint32_t d = tmem + (uint32_t)(acc * 256);
                const uint64_t bd = sdesc(sb + s.slot * BSLOT, blb, 128);
                const uint64_t ar = sdesc(sa + st * DG_S * ADIG, alb, 128);
                const uint32_t first = (s.flags & DF_FIRST) ? 0u : 1u;
                if (s.flags & DF_HI) dg_pairs<RT, CW, 0>(d, ar, bd, idesc, first);
                else dg_pairs<RT, CW, 4>(d, ar, bd, idesc, first);
                mma_commit_el(&bars->empty[st]);
                if (s.flags & DF_FREE) mma_commit_el(&bars->bempty[s.slot]);
                if (s.flags & DF_LAST) mma_commit_el(&bars->acc_full[acc]);
                if (++st == NST) { st = 0; ph ^= 1u; }
                if ((s.flags & DF_LAST) && ++acc == 2) { acc = 0; aph ^= 1u; }
            }
        }
        if (!ok && lane == 0) fail();
        // every MMA has completed before TMEM is released
        mma_commit_el(&bars->drain);
        mbar_wait(&bars->drain, 0);
        __syncwarp();
    } else {
        const int q = warp & 3, part = (warp - 2) >> 2;     // TMEM lane quarter, column part
        constexpr int HC = 8, NG = HC / 4;                  // columns and 4-column groups of this warp
        int acc = 0;
        uint32_t aph = 0;
        const int YB = (a.s.n + 7) / 8;
        const int m5 = a.mul[0], m13 = a.mul[1], m21 = a.mul[2], m29 = a.mul[3];
        const int r = q * 32 + lane;
        // exponents of an item: this row's, and lane j's column c0 + j, per
        // group; loaded an item ahead
        int ea[DG_MAXG], eb[DG_MAXG], na[DG_MAXG], nb[DG_MAXG];
        auto exponents = [&](long long it) {
            const DgItem u = dg_item(a, min(it, a.nitems - 1));
            #pragma unroll
            for (int g = 0; g < DG_MAXG; ++g) {
                const int* Eg = a.E + ((long long)u.k * a.ngrp + min(g, a.ngrp - 1)) * a.s.nrow;
                na[g] = Eg[min(u.mt * RT + r, a.s.nrow - 1)];
                nb[g] = Eg[u.c * CW + part * HC + (lane & (HC - 1))];
            }
        };
        exponents(blockIdx.x);
        for (long long it = blockIdx.x; it < a.nitems && !*abort; it += gridDim.x) {
            const DgItem u = dg_item(a, it);
            const int y = u.mt * RT + r, c0 = u.c * CW + part * HC;
            const bool live = q * 32 < RT && u.mt * RT + q * 32 < a.s.cov;    // uniform over the warp
            const bool row = r < RT && y < a.s.cov;
            #pragma unroll
            for (int g = 0; g < DG_MAXG; ++g) { ea[g] = na[g]; eb[g] = nb[g]; }
            exponents(it + gridDim.x);
            bool ok = true;
            for (int jb = 0; jb < a.njob; ++jb) {
                const DgJob job = a.job[jb];
                int ej = ea[0], ebj = eb[0];
                #pragma unroll
                for (int g = 1; g < DG_MAXG; ++g) {
                    if (job.ga == g) ej = ea[g];
                    if (job.gb == g) ebj = eb[g];
                }
                ej += job.e;
                long long lo[2][HC];
                uint32_t v[2][4][4];
                // orders 4..7
                if (!mbar_wait_ab(&bars->acc_full[acc], aph, abort)) { fail(); ok = false; break; }
                tc_fence_after();
                uint32_t t = tmem + (uint32_t)(acc * 256 + part * HC) + ((uint32_t)(q * 32) << 16);
                if (live) {
                    #pragma unroll
                    for (int g = 0; g < NG; ++g) {
                        dg_tmem(t + 4 * g, CW, v);
                        dg_ready(v);
                        #pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            lo[0][4 * g + j] = dg_low(v[0], j, m13, m5);
                            lo[1][4 * g + j] = dg_low(v[1], j, m13, m5);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->acc_empty[acc]);
                if (++acc == 2) { acc = 0; aph ^= 1u; }
                // orders 0..3, the FP64 values
                if (!mbar_wait_ab(&bars->acc_full[acc], aph, abort)) { fail(); ok = false; break; }
                tc_fence_after();
                t = tmem + (uint32_t)(acc * 256 + part * HC) + ((uint32_t)(q * 32) << 16);
                if (live) {
                    #pragma unroll
                    for (int g = 0; g < NG; ++g) {
                        dg_tmem(t + 4 * g, CW, v);
                        dg_ready(v);
                        const int yp = c0 + 4 * g;
                        zd o[4];
                        bool edge = false;
                        #pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int e = ej + __shfl_sync(0xffffffffu, ebj, 4 * g + j);
                            long long& t0 = lo[0][4 * g + j];
                            long long& t1 = lo[1][4 * g + j];
                            t0 = dg_high(v[0], j, t0, m21, m29);
                            t1 = dg_high(v[1], j, t1, m21, m29);
                            o[j] = mk(dg_value(t0, e, edge), dg_value(t1, e, edge));
                        }
                        if (__any_sync(0xffffffffu, edge && row)) {
                            #pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int e = ej + __shfl_sync(0xffffffffu, ebj, 4 * g + j);
                                o[j] = mk(dg_value_edge(lo[0][4 * g + j], e), dg_value_edge(lo[1][4 * g + j], e));
                            }
                        }
                        if (row && yp < 8 * YB) {
                            zd* dst = a.raw + raw_index(job.out, u.k, y, yp, a.Kc, YB);
                            if (a.beta) {
                                #pragma unroll
                                for (int j = 0; j < 4; ++j) o[j] = o[j] + dst[j];
                            }
                            st_256(dst, o[0], o[1]);
                            st_256(dst + 2, o[2], o[3]);
                        }
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->acc_empty[acc]);
                if (++acc == 2) { acc = 0; aph ^= 1u; }
            }
            if (!ok) break;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// Rows y in [cov, ny) of grids with a thin remainder past the last 128-row
// tile (the Chebyshev grids ny = 128 m + 1): a tile of their own would cost as
// much as a full one.  FP64 FMA chains, CTA = one wavenumber and row, thread = y'.
struct DgRowJob { int nt, out; int fa[DG_MAXT], fb[DG_MAXT]; };
struct DgRows { int njob; DgRowJob job[NJOB]; };
__global__ void __launch_bounds__(160)
k_dg_rows(const __grid_constant__ DgRows jobs, const zd* __restrict__ X, int ns, int ny, int Nk, int k0, int Kc,
          int cov, zd* __restrict__ raw)
{
    const int kl = blockIdx.x, k = k0 + kl, y = cov + blockIdx.y;
    for (int yp = threadIdx.x; yp < ny; yp += blockDim.x)
        for (int j = 0; j < jobs.njob; ++j) {
            const DgRowJob& jd = jobs.job[j];
            if (jd.out == J_D && yp < y) continue;
            zd acc = mk(0.0, 0.0);
            for (int t = 0; t < jd.nt; ++t) {
                const zd* A = X + ((long long)jd.fa[t] * Nk + k) * ns * ny + y;
                const zd* B = X + ((long long)jd.fb[t] * Nk + k) * ns * ny + yp;
                for (int s = 0; s < ns; ++s) {
                    const zd av = A[(long long)s * ny], bv = B[(long long)s * ny];
                    acc.x = fma(av.x, bv.x, acc.x);
                    acc.x = fma(av.y, bv.y, acc.x);
                    acc.y = fma(av.x, bv.y, acc.y);
                    acc.y = fma(-av.y, bv.x, acc.y);
                }
            }
            raw[raw_index(jd.out, kl, y, yp, Kc, (ny + 7) / 8)] = acc;
        }
}

// -------------------------------------------------------------------- host
// the contractions of gke_correlate_f64.cu
struct HostJob { int nt; int fa[DG_MAXT]; int fb[DG_MAXT]; };
static const HostJob kJobs[NJOB] = {
    /* E  */ {1, {F_U}, {F_V}},
    /* F  */ {1, {F_P}, {F_V}},
    /* GX */ {4, {F_Q, F_UU, F_UV, F_UW}, {F_U, F_U, F_V, F_W}},
    /* QV */ {1, {F_Q}, {F_V}},
    /* X2 */ {3, {F_UV, F_VV, F_VW}, {F_U, F_V, F_W}},
    /* GZ */ {4, {F_Q, F_UW, F_VW, F_WW}, {F_W, F_U, F_V, F_W}},
    /* D  */ {3, {F_U, F_V, F_W}, {F_U, F_V, F_W}},
};

// The steps of an item: every contraction's terms with orders 4..7, then again
// with orders 0..3; B fields stay in their slot until the slot whose field
// is needed last has to give way.
struct HostTerm { int fa, fb; bool neg; };
static void dg_schedule(DgArgs& a, const std::vector<std::vector<HostTerm>>& jobs)
{
    a.nstep = 0;
    for (const auto& j : jobs)
        for (int pass = 0; pass < 2; ++pass)
            for (size_t t = 0; t < j.size(); ++t) {
                DgStep s{};
                s.fa = (unsigned char)j[t].fa;
                s.fb = (unsigned char)j[t].fb;
                s.flags = (unsigned char)((j[t].neg ? DF_NEG : 0) | (pass ? DF_HI : 0) | (t == 0 ? DF_FIRST : 0) |
                                          (t + 1 == j.size() ? DF_LAST : 0));
                a.step[a.nstep++] = s;
            }
    int held[DG_NB], last[DG_NB];
    for (int i = 0; i < DG_NB; ++i) held[i] = last[i] = -1;
    for (int q = 0; q < a.nstep; ++q) {
        int slot = -1;
        for (int i = 0; i < DG_NB; ++i)
            if (held[i] == a.step[q].fb) slot = i;
        if (slot < 0) {
            int far = -1;
            for (int i = 0; i < DG_NB; ++i) {
                int next = a.nstep + (held[i] < 0 ? 1 : 0);
                for (int p = a.nstep - 1; p > q; --p)
                    if (a.step[p].fb == held[i]) next = p;
                if (next > far) { far = next; slot = i; }
            }
            if (held[slot] >= 0) a.step[last[slot]].flags |= DF_FREE;
            held[slot] = a.step[q].fb;
            a.step[q].flags |= DF_LOAD;
        }
        a.step[q].slot = (unsigned char)slot;
        last[slot] = q;
    }
    for (int i = 0; i < DG_NB; ++i)
        if (held[i] >= 0) a.step[last[i]].flags |= DF_FREE;
}

static int dg_sm_count()
{
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    return std::max(nsm, 1);
}

template <int RT, int CW> static void dg_launch(const DgArgs& a, cudaStream_t st)
{
    const unsigned grid = (unsigned)std::min<long long>(a.nitems, dg_sm_count());
    k_dg_corr<RT, CW><<<grid, dg_threads(CW), DG_SM, st>>>(a);
}
static void dg_run(const DgArgs& a, cudaStream_t st)
{
    if (a.s.RT == 40) a.s.CW == 24 ? dg_launch<40, 24>(a, st) : dg_launch<40, 32>(a, st);
    else if (a.s.RT == 72) a.s.CW == 24 ? dg_launch<72, 24>(a, st) : dg_launch<72, 32>(a, st);
    else a.s.CW == 24 ? dg_launch<128, 24>(a, st) : dg_launch<128, 32>(a, st);
}

cudaError_t digits_setup()
{
    const void* ks[] = {(const void*)k_dg_corr<40, 24>, (const void*)k_dg_corr<40, 32>, (const void*)k_dg_corr<72, 24>,
                        (const void*)k_dg_corr<72, 32>, (const void*)k_dg_corr<128, 24>, (const void*)k_dg_corr<128, 32>};
    for (const void* k : ks) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, DG_SM);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// channel: 11 A fields, 3 B fields, 3 exponent groups
constexpr int CH_NFA = 11, CH_NFB = 3, CH_NGRP = 3;
static size_t channel_bytes(const DgShape& s)
{
    return (CH_NFA * dg_a_halves(s) + CH_NFB * dg_b_halves(s)) * sizeof(__half) + (size_t)CH_NGRP * s.nrow * sizeof(int);
}
// digit operands are made and used in chunks of wavenumbers of this many bytes
static const size_t DG_CHUNK_BYTES = (size_t)512 << 20;

void digits_alloc(DigitWork& w, int n, int Kc)
{
    const size_t per = channel_bytes(dg_shape(n));
    w.bytes = per * std::max<size_t>(1, std::min<size_t>((size_t)Kc, DG_CHUNK_BYTES / per));
    if (cudaMalloc(&w.ws, w.bytes) != cudaSuccess) w.ws = nullptr;
    if (w.ws && (cudaMalloc((void**)&w.err, sizeof(int)) != cudaSuccess || cudaMemset(w.err, 0, sizeof(int)) != cudaSuccess))
        digits_free(w);
    cudaGetLastError();
}

// Against the FMA kernel (correlate stage, us, FMA -> digits): 544 wavenumbers
// x 4 snapshots: 507 -> 240 at ny = 17, 532 -> 407 at 33, 1954 -> 543 at 65,
// 7535 -> 1130 at 129; 4160 wavenumbers x 16 snapshots: 7423 -> 1659, 8085 -> 2799,
// 29421 -> 4326, 112586 -> 9462.  Only where the FMA kernel's CTAs, one
// 32 x 32 tile of at most one snapshot chunk each, all run at once are the two
// level (40 wavenumbers: 71 us, digits 66 at ny <= 17, 72 at 25): those keep it
// and need no workspace.
bool digits_pays(int n, int ns, long long Kc) { return !(Kc <= 64 && n <= 32 && ns <= 8); }

gke_status digits_correlate(DigitWork& w, const zd* Xop, int ns, int ny, int Nk, int k0, int Kc, zd* raw,
                            unsigned jobs, cudaStream_t st, std::string& err, int* launches)
{
    *launches = 0;
    const DgShape s = dg_shape(ny);
    const size_t per = channel_bytes(s);
    const int kmax = (int)std::min<size_t>((size_t)Kc, w.bytes / per);
    DgPrep p{};
    p.s = s;
    p.ngrp = CH_NGRP; p.nfa = CH_NFA; p.nfb = CH_NFB;
    for (int f = 0; f < NFIELD; ++f) {
        DgField& d = p.f[p.nf++];
        d.src = (short)f;
        d.grp = f <= F_W ? 0 : f == F_P ? 1 : 2;
        d.ia = (short)f;
        d.ib = (short)(f <= F_W ? f : -1);
    }
    p.X = Xop; p.nsX = ns; p.Nk = Nk;
    DgArgs a{};
    a.s = s;
    a.nfa = CH_NFA; a.nfb = CH_NFB; a.ngrp = CH_NGRP;
    a.tpk = s.MT * s.NT;
    a.Kc = Kc;
    for (int i = 0; i < 4; ++i) a.mul[i] = 1 << (5 + 8 * i);
    a.err = w.err;
    std::vector<std::vector<HostTerm>> terms;
    DgRows rows{};
    // long and short contractions alternate: the epilogue of a one-term job
    // takes longer than its MMAs, that of a four-term job less
    static const int order[NJOB] = {J_GX, J_E, J_GZ, J_F, J_X, J_QV, J_D};
    for (int j : order) {
        if (!((jobs >> j) & 1u)) continue;
        const HostJob& h = kJobs[j];
        std::vector<HostTerm> v;
        DgRowJob& rj = rows.job[rows.njob++];
        rj.nt = h.nt; rj.out = j;
        for (int t = 0; t < h.nt; ++t) {
            v.push_back({h.fa[t], h.fb[t], false});
            rj.fa[t] = h.fa[t]; rj.fb[t] = h.fb[t];
        }
        terms.push_back(v);
        DgJob& d = a.job[a.njob++];
        d.ga = (signed char)(h.fa[0] <= F_W ? 0 : h.fa[0] == F_P ? 1 : 2);
        d.gb = 0;
        d.out = (signed char)j;
        d.e = -34;
    }
    if (!a.njob) return GKE_OK;
    dg_schedule(a, terms);
    for (int kc0 = 0; kc0 < Kc; kc0 += kmax) {
        const int nk = std::min(kmax, Kc - kc0);
        p.Aop = (__half*)w.ws;
        p.Bop = p.Aop + (size_t)nk * CH_NFA * dg_a_halves(s);
        p.E = (int*)(p.Bop + (size_t)nk * CH_NFB * dg_b_halves(s));
        p.k0 = k0 + kc0;
        a.Aop = p.Aop; a.Bop = p.Bop; a.E = p.E;
        a.nitems = (long long)nk * a.tpk;
        a.raw = raw + (size_t)kc0 * 64;                       // raw_index: the wavenumber's stride is 64
        for (int s0 = 0; s0 < ns; s0 += DG_KS) {
            p.s0 = s0;
            p.ns = std::min(DG_KS, ns - s0);
            a.beta = s0 > 0;
            k_dg_prep<<<(unsigned)((long long)nk * CH_NGRP * (s.nrow / 128)), 256, 0, st>>>(p);
            dg_run(a, st);
            *launches += 2;
        }
    }
    if (s.cov < ny) {
        k_dg_rows<<<dim3((unsigned)Kc, (unsigned)(ny - s.cov)), 160, 0, st>>>(rows, Xop, ns, ny, Nk, k0, Kc, s.cov, raw);
        *launches += 1;
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) { err = std::string("digit correlator launch: ") + cudaGetErrorString(e); return GKE_ERR_CUDA; }
    return GKE_OK;
}

gke_status digits_check(DigitWork& w, cudaStream_t st, std::string& err)
{
    if (!w.err) return GKE_OK;
    int h = 0;
    if (cudaMemcpyAsync(&h, w.err, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess) {
        err = "digit correlator: cannot read the error flag";
        return GKE_ERR_CUDA;
    }
    if (h) { err = "digit correlator: a tensor-core pipeline wait timed out"; return GKE_ERR_CUDA; }
    return GKE_OK;
}

void digits_free(DigitWork& w)
{
    if (w.ws) cudaFree(w.ws);
    if (w.err) cudaFree(w.err);
    w.ws = nullptr;
    w.err = nullptr;
    w.bytes = 0;
}

}  // namespace gke
