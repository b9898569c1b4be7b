// gke_digits.cu -- the channel's FP64 contractions by exact digit products
// (gke_digits.cuh has the method).
//
// Measured, correlate stage (operands, contractions; FMA kernel -> here):
// 256 x 256 x 65, 16 snapshots 232.8 -> 39.5 ms, of which the operand kernel 8.7
// and the MMAs alone 23 (smem reads of A and B: 18.5 by count), which bound it
// with the epilogue (conversions and integer adds) close behind; 128 x 128 x 65,
// 32 snapshots 117.4 -> 21.5 ms.  (One exponent per row for u, v, w and one for all
// products took 34.7 and 18.6 ms, but held v and w at the size of u.)
#include "gke_digits.h"
#include "gke_digits.cuh"
#include "gke_kernels.h"

namespace gke {

// raw[job][y / 8][y' / 8][k][8][8] (raw_index); beta, or a job's DJ_ADD, adds to what is there
struct RawOut {
    zd* raw;
    int n, Kc, beta;
    __device__ __forceinline__ void operator()(const DgJob& job, int k, int y, int yp, zd (&o)[4]) const
    {
        const int YB = (n + 7) / 8;
        if (yp >= 8 * YB) return;
        zd* dst = raw + raw_index(job.out, k, y, yp, Kc, YB);
        if (beta || (job.kind & DJ_ADD)) {
            #pragma unroll
            for (int j = 0; j < 4; ++j) o[j] = o[j] + dst[j];
        }
        st_256(dst, o[0], o[1]);
        st_256(dst + 2, o[2], o[3]);
    }
};

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

// The operands.  Fields that are added share a group: u, v, w; q with the products
// of u; the products of v and of w, which fall faster towards a wall than q.  u, v and w
// also stand alone, for the contractions of one term, so that those are exact to the
// size of the smaller field (q of <q v'> and <q w'> is nearly always of its group's size).
// GZ is q w and the products of w apart: with a w far below u no term of a joint sum
// would reach the shared exponents.
enum { CG_V = 0, CG_U1, CG_P1, CG_V1, CG_W1, CG_PX, CG_PY, CG_PZ, CH_NGRP };
constexpr int CH_NFA = 15, CH_NFB = 5;
static void channel_fields(DgPrep& p, DgArgs& a)
{
    for (int i = 0; i < 3; ++i) dg_field(p, a, CG_V, F_U + i, i, i);
    dg_field(p, a, CG_U1, F_U, 3, -1);
    dg_field(p, a, CG_P1, F_P, 4, -1);
    dg_field(p, a, CG_V1, F_V, -1, 3);
    dg_field(p, a, CG_W1, F_W, -1, 4);
    static const int px[] = {F_UU, F_UV, F_UW, F_Q}, py[] = {F_UV, F_VV, F_VW}, pz[] = {F_UW, F_VW, F_WW};
    for (int i = 0; i < 4; ++i) dg_field(p, a, CG_PX, px[i], 5 + i, -1);
    for (int i = 0; i < 3; ++i) dg_field(p, a, CG_PY, py[i], 9 + i, -1);
    for (int i = 0; i < 3; ++i) dg_field(p, a, CG_PZ, pz[i], 12 + i, -1);
}
// contractions (operand indices); the second of GZ is added to the first.  Long and
// short alternate: the epilogue of a one-term contraction takes longer than its
// MMAs, that of a four-term one less.
struct DigitJob { int out, kind, ga, gb, sa, nt, fa[DG_MAXT], fb[DG_MAXT]; };
static const DigitJob kDigitJobs[] = {
    {J_GX, 0, CG_PX, CG_V, 0, 4, {5, 6, 7, 8}, {0, 1, 2, 0}},
    {J_GZ, 0, CG_PX, CG_W1, 12, 1, {8}, {4}},
    {J_D, 0, CG_V, CG_V, 0, 3, {0, 1, 2}, {0, 1, 2}},
    {J_E, 0, CG_U1, CG_V1, 0, 1, {3}, {3}},
    {J_GZ, DJ_ADD, CG_PZ, CG_V, 0, 3, {12, 13, 14}, {0, 1, 2}},
    {J_F, 0, CG_P1, CG_V1, 0, 1, {4}, {3}},
    {J_X, 0, CG_PY, CG_V, 0, 3, {9, 10, 11}, {0, 1, 2}},
    {J_QV, 0, CG_PX, CG_V1, 12, 1, {8}, {3}},
};

size_t digits_per_k(int n)
{
    return dg_bytes_per_k(dg_shape(n, true), CH_NFA, CH_NFB, CH_NGRP, (int)(sizeof(kDigitJobs) / sizeof(kDigitJobs[0])), false);
}

void digits_alloc(DigitWork& w, size_t per, int Kc, cudaStream_t st, size_t limit)
{
    w.ws = nullptr;
    for (size_t nk = std::max<size_t>(1, std::min<size_t>((size_t)Kc, limit / per)); nk && !w.ws; nk /= 2) {
        w.bytes = per * nk;
        if (cudaMalloc(&w.ws, w.bytes) != cudaSuccess) w.ws = nullptr;
    }
    if (w.ws && (cudaMalloc((void**)&w.err, sizeof(int)) != cudaSuccess || cudaMemsetAsync(w.err, 0, sizeof(int), st) != cudaSuccess))
        digits_free(w);
    cudaGetLastError();
}

cudaError_t digits_setup(DigitWork& w, int n, int Kc, cudaStream_t st)
{
    const cudaError_t e = dg_attrs<RawOut>();
    if (e == cudaSuccess) digits_alloc(w, digits_per_k(n), Kc, st);
    return e;
}

// Against the FMA kernel (correlate stage, us, FMA -> digits): 544 wavenumbers
// x 4 snapshots: 506 -> 307 at ny = 17, 532 -> 502 at 33, 1946 -> 648 at 65,
// 7529 -> 1429 at 129; 4224 wavenumbers x 16 snapshots: 7548 -> 2185, 8218 -> 3644,
// 29927 -> 5266, 114521 -> 12038; 144 x 4: 158 -> 108, 152 -> 163, 635 -> 217, 2224 -> 432.  Only
// where the FMA kernel's CTAs, one 32 x 32 tile (and its strips) of at most one
// snapshot chunk each, all run at once is it ahead (40 wavenumbers, up to 8 snapshots:
// 70 to 80 us, digits 72 to 108 at ny <= 33; 267 against 109 at 65): those keep it and
// need no workspace.
bool digits_pays(int n, int ns, long long Kc) { return !(Kc <= 64 && n <= 33 && ns <= 8); }

gke_status digits_correlate(DigitWork& w, const zd* Xop, int ns, int ny, int Nk, int k0, int Kc, zd* raw,
                            unsigned jobs, cudaStream_t st, std::string& err, int* launches)
{
    *launches = 0;
    DgPrep p{};
    DgArgs a{};
    const DgShape s = dg_shape(ny, true);
    dg_init(p, a, s, CH_NFA, CH_NFB, CH_NGRP, false, Xop, Nk, ns, w.err);
    channel_fields(p, a);
    const int kmax = (int)std::min<size_t>((size_t)Kc, w.bytes / digits_per_k(ny));
    std::vector<std::vector<HostTerm>> terms;
    for (const DigitJob& h : kDigitJobs) {
        if (!((jobs >> h.out) & 1u)) continue;
        std::vector<HostTerm> v;
        for (int t = 0; t < h.nt; ++t) v.push_back({h.fa[t], h.fb[t], false});
        terms.push_back(v);
        DgJob& d = a.job[a.njob++];
        d.ga = (signed char)h.ga; d.gb = (signed char)h.gb; d.sa = (unsigned char)h.sa;
        d.out = (signed char)h.out; d.kind = (signed char)h.kind; d.out2 = -1;
    }
    DgRows rows{};
    for (int j = 0; j < NJOB; ++j) {
        if (!((jobs >> j) & 1u)) continue;
        const HostJob& h = kJobs[j];
        DgRowJob& rj = rows.job[rows.njob++];
        rj.nt = h.nt; rj.out = j;
        for (int t = 0; t < h.nt; ++t) { rj.fa[t] = h.fa[t]; rj.fb[t] = h.fb[t]; }
    }
    if (!a.njob) return GKE_OK;
    if (!dg_schedule(a, terms)) { err = "digit correlator: contractions beyond the kernel's tables"; return GKE_ERR_UNSUPPORTED; }
    for (int kc0 = 0; kc0 < Kc; kc0 += kmax) {
        const int nk = std::min(kmax, Kc - kc0);
        dg_place(p, a, w.ws, k0 + kc0, nk);
        for (int s0 = 0; s0 < ns; s0 += DG_KS) {
            dg_batch(p, a, s0, std::min(DG_KS, ns - s0));
            // raw_index: the wavenumber's stride is 64
            dg_pass(p, a, nk, RawOut{raw + (size_t)kc0 * 64, ny, Kc, s0 > 0}, st);
            *launches += 3;
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
