// gke_digits.cuh -- FP64 sums of products on the 5th-generation tensor cores by
// exact digit products (error-free splitting of a matrix product: Ozaki, Ogita,
// Oishi, Rump, Numer. Algorithms 59 (2012) 95-118): operand kernel, contraction
// kernel, schedule of its steps.  gke_digits.cu (channel) and gke1h.cu (duct)
// give the fields, the contractions and what happens to the values.
//
// The FP64 pipe does 2 fused multiply-adds per clock and SM, the tensor cores
// 4096 in FP16: the 36 digit products that replace one FP64 product below
// still leave a factor of 50.
//
// Splitting.  The values of a row (wavenumber k, wall-normal point y) of the
// fields of one exponent group share the exponent E of the largest of them over
// the batch's snapshots, |x| < 2^E.  Each value becomes the integer
// round(x 2^(61 - E)) and that its eight balanced base-256 digits s_0
// (|s_0| <= 33) .. s_7 (in [-128, 127]), exact in FP16.
//
// Groups.  A field is held to 61 bits below its group's exponent, so a group
// holds only fields whose products are added (at most four; a field of a
// one-term contraction stands alone): v is not rounded at the size of u in
// <u v'>, however small it is.  A sum of several terms has the accuracy of its
// largest term only if that term is not itself far below the two groups'
// exponents.  Each row carries how many bits each field of the group lies below
// E (a nibble, 5 = more); where the nibbles of every term of a sum add up
// to more than dg_lmax bits, or a row holds an infinity or a NaN, the epilogue leaves a
// zero and a mark, and k_dg_far adds the value by FP64 FMAs from the fields: such
// values cost what the FMA kernels cost, and are right for any input.
//
// Products.  With the digit products s_i t_j summed over the terms and
// snapshots of a contraction by order d = i + j (v_d, d <= 7),
//   sum a b = 2^(E_a + E_b - 34) [ (v_0 .. v_3) + 2^-32 (v_4 .. v_7) ],
//   (w_0 .. w_3) = 2^24 w_0 + 2^16 w_1 + 2^8 w_2 + w_3.
// The orders above 7 are left out: a product loses up to 2^-57 of 2^(E_a + E_b)
// (seven digit products of order 8), 2^-60 typically.  A sum v_d runs over at most
// 4 terms x 16 snapshots x 2 real products, so
// |v_d| <= max(1, d) 4 2^19 < 2^24 (and < 2^22 for d <= 2, where s_0 enters every
// or all but one product): the FP32 accumulation in tensor memory is exact.  A
// batch of 16 / c snapshots or fewer takes its A digits times c = 2, 4, 8 or 16 (exact
// in FP16), so the same bounds hold and the joined sum's unit is c times finer.  The
// eight sums are joined in a 64-bit integer and rounded to FP64
// once, all in integer arithmetic.  A sum over up to 16 snapshots therefore
// carries one rounding where the FMA chain carries 32 per term; further
// snapshots come in groups of 16, added in FP64.
//
// Error against exact sums, over the 2-norms of the operands (rms; emulated with
// random operands; FMA chain): one term, 1 / 4 / 16 snapshots 4.7e-17 / 2.4e-17 /
// 1.4e-17 (5.8e-17 / 5.0e-17 / 4.8e-17); at dg_lmax bits 5.5e-17 / 3.2e-17 / 3.0e-17; three and four
// terms at their dg_lmax, 16 snapshots, 7.0e-17 and 1.4e-16 (1.25e-16 and 1.6e-16).
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
#pragma once
#include <cuda_fp16.h>

#include <algorithm>
#include <vector>

#include "gke_common.cuh"
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
constexpr int DG_MAXSTEP = 112, DG_MAXJOB = 20, DG_MAXF = 24, DG_MAXT = 4;

enum { DF_NEG = 1, DF_LOAD = 2, DF_FREE = 4, DF_FIRST = 8, DF_LAST = 16, DF_HI = 32 };
// one term of one pass: conj(A field fa) B field fb; B in slot, loaded before
// (DF_LOAD) or released after it (DF_FREE)
struct DgStep { unsigned char fa, fb, slot, flags; };
// a contraction: exponent groups of its A and B fields, output index and kind
// (DJ_ADD: add to what is there) and a second output (psi: with the factor half / 2);
// the value is 2^ex times the sum, 2^e times the joined digits' upper half.  Term t
// goes with nibble t of the B row's distances and nibble t of the A row's
// shifted by sa bits; first step of the schedule.
enum { DJ_ADD = 1 };
struct DgJob {
    signed char ga, gb, out, kind, out2, half;
    unsigned char sa, nt, step;
    short e, ex;
    unsigned short add, mask;
};
// bits that every term of a sum of nt terms may lie below its rows' exponents:
// up to there the digits' error stays under the FMA chain's (header)
__host__ __device__ constexpr int dg_lmax(int nt, int ns) { return nt == 1 ? (ns == 1 ? 3 : 2) : nt < 4 ? 3 : 4; }
constexpr int DG_FAR = 5;                                   // nibble of a field further below, or not finite

struct DgBars {
    uint64_t full[DG_MAXST], empty[DG_MAXST], bfull[DG_NB], bempty[DG_NB], acc_full[2], acc_empty[2], drain;
    uint32_t tmem;
    int abort;
};
static_assert(sizeof(DgBars) <= DG_SM_BAR, "barrier area");

struct DgShape {
    int n, RT, MT, cov, NT, CW, nrow;      // rows per A tile, A tiles, rows they cover, column tiles, E rows
};

// a field as the operands hold it: X_src times 2^wexp, or for src2 >= 0 the
// combination c X_src + c2 X_src2 (coefficient rows of n values), without c
// X_src + w2 X_src2; exponent group, A and B operand index (-1: not used)
struct DgField { short src, src2, ia, ib; signed char wexp, grp; float w2; const double* c; const double* c2; };
// the fields [src][k][s][y] of a batch of ns snapshots from s0 on
struct DgSrc {
    const zd* X;
    int n, s0, ns, nsX, Nk, k0, nf;
    DgField f[DG_MAXF];
};

struct DgArgs {
    const __half* Aop; const __half* Bop; const int* E;
    DgShape s;
    int nfa, nfb, ngrp, tpk;               // fields of A, of B, exponent groups, tiles per wavenumber
    int tri;                               // only tiles with a pair y <= y'
    long long nitems;
    int nstep, njob;
    DgStep step[DG_MAXSTEP];
    DgJob job[DG_MAXJOB];
    unsigned char af[DG_MAXF], bf[DG_MAXF];   // operand -> field of src
    DgSrc src;
    unsigned* far;                         // [item][contraction]: marks of a warp's 32 rows x 4 columns (dg_mark)
    int mul[4];                            // 2^5, 2^13, 2^21, 2^29 (mad_wide)
    int* err;
};

// A stages that fit beside the B slots
constexpr int dg_nst(int RT, int CW)
{
    const int n = (DG_SM - DG_SM_BAR - DG_NB * DG_S * 3 * CW * DG_KS * 2) / (DG_S * 2 * RT * DG_KS * 2);
    return n < DG_MAXST ? n : DG_MAXST;
}

// thin: a remainder of at most 4 rows past the last 128-row tile is left out (cov < n)
inline DgShape dg_shape(int n, bool thin_ok)
{
    DgShape s{};
    s.n = n;
    // rows of an A tile: the instantiated heights (short tiles copy less; an MMA
    // always takes 128 rows, reading past a short tile into lanes nobody reads)
    s.MT = 1;
    s.cov = n;
    s.RT = n <= 40 ? 40 : n <= 72 ? 72 : 128;
    if (n > 128) {
        const bool thin = thin_ok && n % 128 >= 1 && n % 128 <= 4;
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
inline size_t dg_a_halves(const DgShape& s) { return (size_t)s.MT * DG_S * 2 * s.RT * DG_KS; }      // per field and k
inline size_t dg_b_halves(const DgShape& s) { return (size_t)s.NT * DG_S * 3 * s.CW * DG_KS; }

// ------------------------------------------------------------- digit operands
struct DgPrep {
    DgShape s;
    int nfa, nfb, ngrp, cexp;              // cexp: the A digits carry the factor 2^cexp
    DgSrc src;
    __half* Aop; __half* Bop; int* E;
    unsigned* far; long long nfar;         // marks to clear
};
// without 2^wexp
__device__ __forceinline__ zd dg_load(const DgSrc& a, const DgField& fd, int k, int s, int y)
{
    const long long o = ((long long)(a.k0 + k) * a.nsX + a.s0 + s) * a.n + y, fs = (long long)a.Nk * a.nsX * a.n;
    const zd v = a.X[fd.src * fs + o];
    if (fd.src2 < 0) return v;
    const zd w = a.X[fd.src2 * fs + o];
    if (!fd.c) return mk(fma((double)fd.w2, w.x, v.x), fma((double)fd.w2, w.y, v.y));
    const double p = fd.c[y], q = fd.c2[y];
    return mk(p * v.x + q * w.x, p * v.y + q * w.y);
}

constexpr int DG_NAN = 8192;                                // exponent of a group's row with an infinity or a NaN

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

// CTA = one (wavenumber, exponent group, 128 rows): the rows' exponents with the
// fields' distances below them, then the digit blocks of the group's fields.
// Thread = one row x 8 snapshots, the 16 bytes of a core-matrix row; stores are contiguous over the rows.
// Bound by memory: X is read twice (the second time from L2), 32 bytes of digits are
// written per A value (256 x 256 x 65, 16 snapshots: 8.7 ms; with three CTAs an SM 9.2).
static __global__ void __launch_bounds__(256, 4)
k_dg_prep(const __grid_constant__ DgPrep a)
{
    __shared__ unsigned s_hi[DG_MAXT][128];
    const DgSrc& x = a.src;
    const int nb = a.s.nrow / 128;
    int b = blockIdx.x;
    const int mb = b % nb; b /= nb;
    const int g = b % a.ngrp, k = b / a.ngrp;
    const int r = threadIdx.x & 127, kc = threadIdx.x >> 7;
    const int y = mb * 128 + r;
    for (int i = threadIdx.x; i < DG_MAXT * 128; i += 256) (&s_hi[0][0])[i] = 0;
    for (long long i = blockIdx.x * 256ll + threadIdx.x; i < a.nfar; i += gridDim.x * 256ll) a.far[i] = 0;
    __syncthreads();
    const int e0 = kc * 8, ne = y < a.s.n ? max(0, min(8, x.ns - e0)) : 0;
    int nm = 0;                                             // fields of the group
    for (int f = 0; f < x.nf; ++f) {
        const DgField& fd = x.f[f];
        if (fd.grp != g) continue;
        unsigned hi = 0;
        for (int e = 0; e < ne; ++e) {
            const zd v = dg_load(x, fd, k, e0 + e, y);
            // (unsigned: an infinity or a NaN times 2^wexp stays above 0x7ff00000)
            const unsigned h = (unsigned)max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff);
            if (h >= 0x00100000u) hi = max(hi, h + fd.wexp * 0x00100000u);
        }
        atomicMax(&s_hi[nm++][r], hi);
    }
    __syncthreads();
    int E = -1021;
    for (int i = 0; i < nm; ++i) {
        const unsigned h = s_hi[i][r];
        E = max(E, h >= 0x7ff00000u ? DG_NAN : (int)(h >> 20) - 1022);                      // |x| < 2^E
    }
    if (kc == 0) {
        // (three fields: the fourth nibble repeats the first's, for a fourth term with the first field)
        unsigned far = 0;
        for (int i = 0; i < DG_MAXT; ++i) {
            const unsigned h = s_hi[i < nm ? i : 0][r];
            far |= (unsigned)(E == DG_NAN ? DG_FAR : min(E - max((int)(h >> 20) - 1022, -1021), DG_FAR)) << (4 * i);
        }
        a.E[((long long)k * a.ngrp + g) * a.s.nrow + y] = (int)((far << 16) | (unsigned)(E & 0xffff));
    }
    const __half2 cs = __half2half2(__int2half_rn(1 << a.cexp));
    const bool arow = mb < a.s.MT && r < a.s.RT && y < a.s.cov, astore = mb < a.s.MT && r < a.s.RT;
    const int c = y / a.s.CW, rc = y - c * a.s.CW;
    const bool bstore = c < a.s.NT;
    for (int f = 0; f < x.nf; ++f) {
        const DgField& fd = x.f[f];
        if (fd.grp != g) continue;
        unsigned long long dre[8], dim[8];
        #pragma unroll
        for (int e = 0; e < 8; ++e) {
            zd v = mk(0.0, 0.0);
            if (e < ne) v = dg_load(x, fd, k, e0 + e, y);
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
            if (db) {
                __half* d = db + (long long)i * 3 * a.s.CW * DG_KS + b0;
                *(uint4*)d = re;
                *(uint4*)(d + bw) = im;
                *(uint4*)(d + 2 * bw) = make_uint4(re.x ^ 0x80008000u, re.y ^ 0x80008000u, re.z ^ 0x80008000u,
                                                   re.w ^ 0x80008000u);
            }
            if (da) {
                if (a.cexp) {
                    #pragma unroll
                    for (int h = 0; h < 4; ++h) {
                        *(__half2*)&pr[h] = __hmul2(*(__half2*)&pr[h], cs);
                        *(__half2*)&pi[h] = __hmul2(*(__half2*)&pi[h], cs);
                    }
                }
                const uint4 z = make_uint4(0, 0, 0, 0);
                *(uint4*)(da + (long long)(2 * i) * a.s.RT * DG_KS) = arow ? re : z;
                *(uint4*)(da + (long long)(2 * i + 1) * a.s.RT * DG_KS) = arow ? im : z;
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
static __device__ __noinline__ double dg_value_edge(long long t, int e) { return scalbn((double)t, e - 21); }
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

// every term of a contraction too far below its rows' exponents: words wa, wb of the A and B row
// (no nibble overflows: 5 + 5 + 5)
__device__ __forceinline__ bool dg_far(const DgJob& job, int wa, int wb)
{
    return ((((unsigned)wa >> 16 >> job.sa) + ((unsigned)wb >> 16) + job.add) & job.mask) == job.mask;
}
// bit of the mark of a warp's four columns: TMEM lane quarter, 8-column part, 4-column group
__device__ __forceinline__ int dg_mark(int q, int part, int g) { return (part * 4 + q) * 2 + g; }

struct DgItem { int k, mt, c; };
__device__ __forceinline__ DgItem dg_item(const DgArgs& a, long long it)
{
    DgItem u;
    u.k = (int)(it / a.tpk);
    int r = (int)(it - (long long)u.k * a.tpk);
    if (a.tri) {
        // tiles with a column y' >= y: from the one that holds the row tile's first row
        u.mt = 0;
        for (int c0; r >= a.s.NT - (c0 = u.mt * a.s.RT / a.s.CW); ++u.mt) r -= a.s.NT - c0;
        u.c = u.mt * a.s.RT / a.s.CW + r;
        return u;
    }
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

// Out receives the values of a row and four columns: out(job, item, y, y', valid row, values)
template <int RT, int CW, typename Out>
__global__ void __launch_bounds__(dg_threads(CW), 1)
k_dg_corr(const __grid_constant__ DgArgs a, const __grid_constant__ Out out)
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
        const int m5 = a.mul[0], m13 = a.mul[1], m21 = a.mul[2], m29 = a.mul[3];
        const int r = q * 32 + lane;
        // exponents and distances of a contraction: this row's, and of lane j's column
        // c0 + j; loaded a contraction ahead
        int na, nb;
        auto fetch = [&](const DgItem& u, const DgJob& job) {
            const int* E = a.E + (long long)u.k * a.ngrp * a.s.nrow;
            na = E[job.ga * a.s.nrow + min(u.mt * RT + r, a.s.nrow - 1)];
            nb = E[job.gb * a.s.nrow + u.c * CW + part * HC + (lane & (HC - 1))];
        };
        DgItem u = dg_item(a, min((long long)blockIdx.x, a.nitems - 1));
        fetch(u, a.job[0]);
        for (long long it = blockIdx.x; it < a.nitems && !*abort; it += gridDim.x) {
            const DgItem next = dg_item(a, min(it + gridDim.x, a.nitems - 1));
            const int y = u.mt * RT + r, c0 = u.c * CW + part * HC;
            const bool live = q * 32 < RT && u.mt * RT + q * 32 < a.s.cov;    // uniform over the warp
            const bool row = r < RT && y < a.s.cov;
            bool ok = true;
            for (int jb = 0; jb < a.njob; ++jb) {
                const DgJob job = a.job[jb];
                const int wa = na, wb = nb;
                if (jb + 1 < a.njob) fetch(u, a.job[jb + 1]);
                else fetch(next, a.job[0]);
                const int ej = (int)(short)wa + job.e;
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
                        unsigned far = 0;
                        #pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            const int w = __shfl_sync(0xffffffffu, wb, 4 * g + j), e = ej + (int)(short)w;
                            far |= (unsigned)dg_far(job, wa, w) << j;
                            long long& t0 = lo[0][4 * g + j];
                            long long& t1 = lo[1][4 * g + j];
                            t0 = dg_high(v[0], j, t0, m21, m29);
                            t1 = dg_high(v[1], j, t1, m21, m29);
                            o[j] = mk(dg_value(t0, e, edge), dg_value(t1, e, edge));
                        }
                        if (__any_sync(0xffffffffu, edge && row)) {
                            #pragma unroll
                            for (int j = 0; j < 4; ++j) {
                                const int e = ej + (int)(short)__shfl_sync(0xffffffffu, wb, 4 * g + j);
                                o[j] = mk(dg_value_edge(lo[0][4 * g + j], e), dg_value_edge(lo[1][4 * g + j], e));
                            }
                        }
                        if (__any_sync(0xffffffffu, row && far)) {
                            #pragma unroll
                            for (int j = 0; j < 4; ++j)
                                if ((far >> j) & 1u) o[j] = mk(0.0, 0.0);
                            if (lane == 0) atomicOr(a.far + it * a.njob + jb, 1u << dg_mark(q, part, g));
                        }
                        if (row) out(job, u.k, y, yp, o);
                    }
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&bars->acc_empty[acc]);
                if (++acc == 2) { acc = 0; aph ^= 1u; }
            }
            if (!ok) break;
            u = next;
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 1) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
    }
}

// Adds the marked values by FP64 FMAs from the fields.  CTA = one item at a time, whose
// marks its warps share: a mark's contractions go to one warp in their order (one
// value may get several).  Lane = row; a mark's far values are taken in a chain per lane
// and column, as in the FMA kernels, where most rows have some, else row by row, the
// lanes shared out over its far columns and their products, and a tree.  Bound by latency with few
// marked items (one warp per item took 6.5 ms for the 171 items of the duct's m = 0,
// whose fluctuations are rounding noise; 16 warps, a column at a time, 1.9, so 1.4), else
// by the FP64 pipe.  Milliseconds at 128 x 128 x 65 / duct 256 x 33 x 33, 16 snapshots, where components
// differ in size: all equal 0.3 / 1.4; v (and w) falling one power faster to their walls 0.3 / 2.4;
// v and w 2^-10 of u 0.6 / 4.6; u 2^-4 of v and w 2.7 / 13.6; u 2^-10 of them 33 / 128 (the
// contractions by the FMA kernels: 59 / 334).
constexpr int DG_FARW = 16;                                 // warps of a CTA
template <typename Out>
__global__ void __launch_bounds__(32 * DG_FARW, 2)
k_dg_far(const __grid_constant__ DgArgs a, const __grid_constant__ Out out)
{
    const int lane = threadIdx.x & 31;
    static_assert(DG_MAXJOB <= 32, "a lane per contraction");
    const unsigned own = 0x00010001u << (threadIdx.x >> 5);
    static_assert(DG_FARW == 16, "marks of a warp");
    for (long long it = blockIdx.x; it < a.nitems; it += gridDim.x) {
        const unsigned mine = lane < a.njob ? a.far[it * a.njob + lane] & own : 0u;
        for (unsigned any = __ballot_sync(0xffffffffu, mine != 0); any; any &= any - 1) {
            const int src = __ffs(any) - 1;
            const DgItem u = dg_item(a, it);
            DgJob job = a.job[src];
            job.kind |= DJ_ADD;
            const int* E = a.E + (long long)u.k * a.ngrp * a.s.nrow;
            const int n = job.nt * a.src.ns;
            const double ce = __hiloint2double((1023 + job.ex) << 20, 0);
            for (unsigned m = __shfl_sync(0xffffffffu, mine, src); m; m &= m - 1) {
                const int b = __ffs(m) - 1, r = (b >> 1 & 3) * 32 + lane;
                const int y = u.mt * a.s.RT + r, y0 = u.c * a.s.CW + (b >> 3) * 8 + (b & 1) * 4;
                const bool row = r < a.s.RT && y < a.s.cov;
                const int wa = row ? E[job.ga * a.s.nrow + y] : 0;
                auto product = [&](int i, int ya, int yb, zd& acc) {
                    const int t = i / a.src.ns, s = i - t * a.src.ns;
                    const DgStep st = a.step[job.step + t];
                    const DgField &fa = a.src.f[a.af[st.fa]], &fb = a.src.f[a.bf[st.fb]];
                    const zd p = dg_load(a.src, fa, u.k, s, ya), v = dg_load(a.src, fb, u.k, s, yb);
                    const double c = __hiloint2double((1023 + fa.wexp + fb.wexp) << 20 | ((st.flags & DF_NEG) ? (int)0x80000000 : 0), 0);
                    acc.x = fma(c * p.x, v.x, acc.x);
                    acc.x = fma(c * p.y, v.y, acc.x);
                    acc.y = fma(c * p.x, v.y, acc.y);
                    acc.y = fma(-c * p.y, v.x, acc.y);
                };
                unsigned who[4], rows = 0;
                #pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int yp = y0 + j;
                    const bool far = row && yp < a.s.n && !(a.tri && yp < y) && dg_far(job, wa, E[job.gb * a.s.nrow + yp]);
                    who[j] = __ballot_sync(0xffffffffu, far);
                    rows |= who[j];
                }
                zd o[4] = {mk(0.0, 0.0), mk(0.0, 0.0), mk(0.0, 0.0), mk(0.0, 0.0)};
                if (__popc(rows) >= 24) {
                    #pragma unroll
                    for (int j = 0; j < 4; ++j)
                        if ((who[j] >> lane) & 1u)
                            for (int i = 0; i < n; ++i) product(i, y, y0 + j, o[j]);
                } else {
                    for (unsigned w = rows; w; w &= w - 1) {
                        const int l = __ffs(w) - 1, ya = __shfl_sync(0xffffffffu, y, l);
                        unsigned m = 0;                      // the row's far columns; g lanes side by side share them
                        #pragma unroll
                        for (int j = 0; j < 4; ++j) m |= ((who[j] >> l) & 1u) << j;
                        const int c = __popc(m), g = c > 2 ? 4 : c;
                        unsigned mine = m;
                        for (int i = lane & (g - 1); i > 0; --i) mine &= mine - 1;
                        zd p = mk(0.0, 0.0);
                        if (mine) {
                            const int yb = y0 + __ffs(mine) - 1;
                            for (int i = lane / g; i < n; i += 32 / g) product(i, ya, yb, p);
                        }
                        for (int h = 16; h >= g; h >>= 1) {
                            p.x += __shfl_xor_sync(0xffffffffu, p.x, h);
                            p.y += __shfl_xor_sync(0xffffffffu, p.y, h);
                        }
                        #pragma unroll
                        for (int j = 0; j < 4; ++j) {
                            if (!((m >> j) & 1u)) continue;
                            const int k = __popc(m & ((1u << j) - 1));
                            const zd v = mk(__shfl_sync(0xffffffffu, p.x, k), __shfl_sync(0xffffffffu, p.y, k));
                            if (lane == l) o[j] = v;
                        }
                    }
                }
                #pragma unroll
                for (int j = 0; j < 4; ++j) o[j] = mk(ce * o[j].x, ce * o[j].y);
                if (row) out(job, u.k, y, y0, o);
            }
        }
    }
}

// -------------------------------------------------------------------- host
// The steps of an item: every contraction's terms with orders 4..7, then again
// with orders 0..3; B fields stay in their slot until the slot whose field
// is needed last has to give way.
// False, and nothing scheduled, where a contraction has no term or more than DG_MAXT (more
// would break the exactness of the FP32 sums), or where there are more
// contractions or steps than the kernels' tables hold.
struct HostTerm { int fa, fb; bool neg; };
inline bool dg_schedule(DgArgs& a, const std::vector<std::vector<HostTerm>>& jobs)
{
    a.nstep = 0;
    size_t steps = 0;
    for (const auto& j : jobs) {
        if (j.empty() || j.size() > DG_MAXT) return false;
        steps += 2 * j.size();
    }
    if (jobs.size() > DG_MAXJOB || steps > DG_MAXSTEP) return false;
    for (size_t i = 0; i < jobs.size(); ++i) {
        const auto& j = jobs[i];
        DgJob& d = a.job[i];
        d.nt = (unsigned char)j.size();
        d.step = (unsigned char)a.nstep;
        const unsigned nibbles = (1u << (4 * d.nt)) - 1;
        d.mask = (unsigned short)(0x8888u & nibbles);
        for (int pass = 0; pass < 2; ++pass)
            for (size_t t = 0; t < j.size(); ++t) {
                DgStep s{};
                s.fa = (unsigned char)j[t].fa;
                s.fb = (unsigned char)j[t].fb;
                s.flags = (unsigned char)((j[t].neg ? DF_NEG : 0) | (pass ? DF_HI : 0) | (t == 0 ? DF_FIRST : 0) |
                                          (t + 1 == j.size() ? DF_LAST : 0));
                a.step[a.nstep++] = s;
            }
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
    return true;
}

inline int dg_sm_count()
{
    int dev = 0, nsm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    return std::max(nsm, 1);
}

template <int RT, int CW, typename Out> inline void dg_launch(const DgArgs& a, const Out& out, cudaStream_t st)
{
    const unsigned grid = (unsigned)std::min<long long>(a.nitems, dg_sm_count());
    k_dg_corr<RT, CW, Out><<<grid, dg_threads(CW), DG_SM, st>>>(a, out);
}
template <typename Out> inline void dg_run(const DgArgs& a, const Out& out, cudaStream_t st)
{
    if (a.s.RT == 40) a.s.CW == 24 ? dg_launch<40, 24>(a, out, st) : dg_launch<40, 32>(a, out, st);
    else if (a.s.RT == 72) a.s.CW == 24 ? dg_launch<72, 24>(a, out, st) : dg_launch<72, 32>(a, out, st);
    else a.s.CW == 24 ? dg_launch<128, 24>(a, out, st) : dg_launch<128, 32>(a, out, st);
}
// the operands of p, then the contractions (three kernels)
template <typename Out> inline void dg_pass(const DgPrep& p, const DgArgs& a, int nk, const Out& out, cudaStream_t st)
{
    k_dg_prep<<<(unsigned)((long long)nk * p.ngrp * (p.s.nrow / 128)), 256, 0, st>>>(p);
    dg_run(a, out, st);
    k_dg_far<Out><<<(unsigned)std::min<long long>(a.nitems, 4 * dg_sm_count()), 32 * DG_FARW, 0, st>>>(a, out);
}
template <typename Out> inline cudaError_t dg_attrs()
{
    const void* ks[] = {(const void*)k_dg_corr<40, 24, Out>, (const void*)k_dg_corr<40, 32, Out>,
                        (const void*)k_dg_corr<72, 24, Out>, (const void*)k_dg_corr<72, 32, Out>,
                        (const void*)k_dg_corr<128, 24, Out>, (const void*)k_dg_corr<128, 32, Out>};
    for (const void* k : ks) {
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, DG_SM);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}
// the next field: X_src times 2^wexp as A and B operand ia, ib (-1: none)
inline DgField& dg_field(DgPrep& p, DgArgs& a, int grp, int src, int ia, int ib, int wexp = 0)
{
    DgField f{};
    f.src = (short)src; f.src2 = -1; f.ia = (short)ia; f.ib = (short)ib;
    f.wexp = (signed char)wexp; f.grp = (signed char)grp;
    if (ia >= 0) a.af[ia] = (unsigned char)p.src.nf;
    if (ib >= 0) a.bf[ib] = (unsigned char)p.src.nf;
    return p.src.f[p.src.nf++] = f;
}
// tiles of one wavenumber
inline int dg_tiles(const DgShape& s, bool tri)
{
    int n = 0;
    for (int mt = 0; mt < s.MT; ++mt) n += s.NT - (tri ? mt * s.RT / s.CW : 0);
    return n;
}
// bytes of one wavenumber's operands, exponents and marks
inline size_t dg_bytes_per_k(const DgShape& s, int nfa, int nfb, int ngrp, int njob, bool tri)
{
    return (nfa * dg_a_halves(s) + nfb * dg_b_halves(s)) * sizeof(__half) + (size_t)ngrp * s.nrow * sizeof(int) +
           (size_t)dg_tiles(s, tri) * njob * sizeof(unsigned);
}
// places the operands of nk wavenumbers from k0 on in ws
inline void dg_place(DgPrep& p, DgArgs& a, void* ws, int k0, int nk)
{
    p.src.k0 = k0;
    p.Aop = (__half*)ws;
    p.Bop = p.Aop + (size_t)nk * p.nfa * dg_a_halves(p.s);
    p.E = (int*)(p.Bop + (size_t)nk * p.nfb * dg_b_halves(p.s));
    a.Aop = p.Aop; a.Bop = p.Bop; a.E = p.E;
    a.nitems = (long long)nk * a.tpk;
    p.far = a.far = (unsigned*)(p.E + (size_t)nk * p.ngrp * p.s.nrow);
    p.nfar = a.nitems * a.njob;
}
// the snapshots [s0, s0 + ns), ns <= 16: with them the digits' factor c and what depends on it
inline void dg_batch(DgPrep& p, DgArgs& a, int s0, int ns)
{
    p.cexp = 0;
    while ((ns << (p.cexp + 1)) <= DG_KS) ++p.cexp;
    p.src.s0 = s0;
    p.src.ns = ns;
    a.src = p.src;
    for (int i = 0; i < a.njob; ++i) {
        DgJob& d = a.job[i];
        d.e = (short)(d.ex - 34 - p.cexp);
        d.add = (unsigned short)((d.mask >> 3) * (7 - dg_lmax(d.nt, ns)));
    }
}
// tiles per wavenumber, shape and constants; X: fields of Nk wavenumbers and ns snapshots
inline void dg_init(DgPrep& p, DgArgs& a, const DgShape& s, int nfa, int nfb, int ngrp, bool tri, const zd* X, int Nk,
                    int ns, int* err)
{
    p.s = a.s = s;
    p.src.X = X; p.src.n = s.n; p.src.Nk = Nk; p.src.nsX = ns;
    p.nfa = a.nfa = nfa; p.nfb = a.nfb = nfb; p.ngrp = a.ngrp = ngrp;
    a.tri = tri;
    a.tpk = dg_tiles(s, tri);
    for (int i = 0; i < 4; ++i) a.mul[i] = 1 << (5 + 8 * i);
    a.err = err;
}

}  // namespace gke
