// gke_step1.cu -- Step 1 for velocity-vorticity databases (Sec. 3.2, Step 1).
//
// DNS solvers in velocity-vorticity form store the wall-normal velocity v and
// vorticity eta = du/dz - dw/dx as Fourier coefficients in x, z, plus the plane
// averages of u and w.  Step 1 recovers u, w and the pressure p per snapshot,
// all in FP64, as the fields [4][ny][nz][nxh] the GKE path consumes:
//   k_s1_velocity     u = (i kx dv/dy - i kz eta) / k^2, w = (i kz dv/dy + i kx eta) / k^2
//                     (continuity and the definition of eta solved for u, w);
//   k_s1_col          inverse / forward DFT along z of column groups (fft_block),
//   k_s1_col_r        for the register lengths in fixed point (gke_fixed.cuh);
//   k_s1_row_products per (y, z) row: inverse real DFT along x of u, v, w
//                     (u + i v and w as complex sequences), the six products
//                     u_i u_j, forward DFT of them packed in pairs;
//                     k_s1_row_products_r for the register lengths;
//   k_s1_factor       LU (partial pivoting) of the banded Poisson operator
//                     d2/dy2 - k^2 with its Neumann wall rows, once per plan;
//   k_s1_source       the source -d_i d_j (u_i u_j) and the wall values
//                     dp/dy = nu d2v/dy2 (y-momentum at no-slip walls);
//   k_s1_solve        the banded solve, per wavenumber and part.
// Conventions: odd x / z derivatives use the signed wavenumber with 0 on the
// Nyquist lines, second derivatives the true square; d/dy and d2/dy2 are the
// 5-point weights on the nodes l0 .. l0 + 4 of each row; the singular (0, 0)
// Poisson problem has its first row replaced by p(y_0) = 0.
#include <type_traits>

#include "gke_common.cuh"
#include "gke_fixed.cuh"
#include "gke_kernels.h"

namespace gke {

// band of the Poisson rows: interior rows reach 2 below and 2 above the
// diagonal, the one-sided wall rows 4; partial pivoting adds S1_KL columns
// of fill above, so a row is stored from col r - KL to r + KU + KL
constexpr int S1_KL = 4, S1_KU = 4, S1_W = 2 * S1_KL + S1_KU + 1;
constexpr double TWO_PI = 6.283185307179586476925286766559;

__device__ __forceinline__ double kodd(int m, int n, double L) { return TWO_PI * signed_bin(m, n) / L; }
__device__ __forceinline__ double ktrue2(int m, int n, double L)
{
    const int s = (2 * m > n) ? m - n : m;           // the true bin on the Nyquist line
    const double k = TWO_PI * s / L;
    return k * k;
}

// The five nodes of a row's stencil in registers while a thread walks down y:
// seek(l) moves the window to the rows l .. l + 4 (l never decreases), get(r)
// being the value of row r.
struct Window {
    zd w[5];
    int base;
    template <typename G> __device__ __forceinline__ void open(int l, G get)
    {
        base = l;
        #pragma unroll
        for (int i = 0; i < 5; ++i) w[i] = get(l + i);
    }
    template <typename G> __device__ __forceinline__ void seek(int l, G get)
    {
        for (; base < l; ++base) {
            #pragma unroll
            for (int i = 0; i < 4; ++i) w[i] = w[i + 1];
            w[4] = get(base + 5);
        }
    }
    __device__ __forceinline__ zd apply(const double* __restrict__ c) const
    {
        zd s = mk(0.0, 0.0);
        #pragma unroll
        for (int i = 0; i < 5; ++i) s = mk(s.x + c[i] * w[i].x, s.y + c[i] * w[i].y);
        return s;
    }
};
constexpr int S1_ROWS = 16;                          // rows a thread walks down

// u, w of one snapshot; v copied; (0, 0) modes from the plane averages.  Thread
// = one wavenumber, S1_ROWS rows: the FP64 pipe bounds it, so the wavenumber's
// divisions are done once per thread (256 x 256 x 129: 575 -> 169 us with a thread per
// coefficient before).
__global__ void k_s1_velocity(const zd* __restrict__ v, const zd* __restrict__ eta, const double* __restrict__ mean_uw,
                              int ny, int nz, int nx, double Lx, double Lz, const double* __restrict__ w1,
                              const int* __restrict__ l0, zd* __restrict__ out)
{
    const int nxh = nx / 2 + 1;
    const long long Nk = (long long)nz * nxh, fs = (long long)ny * Nk;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Nk) return;
    const int kz_i = (int)(k / nxh), kx_i = (int)(k - (long long)kz_i * nxh);
    const double kx = kodd(kx_i, nx, Lx), kz = kodd(kz_i, nz, Lz), k2 = kx * kx + kz * kz;
    const double cx = k2 > 0.0 ? kx / k2 : 0.0, cz = k2 > 0.0 ? kz / k2 : 0.0;
    const int j0 = blockIdx.y * S1_ROWS, j1 = min(j0 + S1_ROWS, ny);
    auto get = [&](int r) { return v[(long long)r * Nk + k]; };
    Window win;
    win.open(l0[j0], get);
    for (int j = j0; j < j1; ++j) {
        const long long i = (long long)j * Nk + k;
        win.seek(l0[j], get);
        const zd dv = win.apply(w1 + 5 * j), e = eta[i];
        // i kx dv - i kz e, i kz dv + i kx e, over k^2
        zd u = mk(cz * e.y - cx * dv.y, cx * dv.x - cz * e.x), w = mk(-cz * dv.y - cx * e.y, cz * dv.x + cx * e.x);
        if (k == 0) {
            u = mk(mean_uw[j], 0.0);
            w = mk(mean_uw[ny + j], 0.0);
        } else if (!(k2 > 0.0)) u = w = mk(0.0, 0.0);
        out[i] = u;
        out[fs + i] = get(j);
        out[2 * fs + i] = w;
    }
}

// DFT along z of nf fields [f][ny][nz][nxh]: CTA = (field, y, NC columns kx);
// INV: unnormalised inverse; forward: scaled by 1 / nz
template <bool INV>
__global__ void k_s1_col(const zd* __restrict__ in, int ny, int nz, int nxh, int NC, const zd* __restrict__ tw,
                         zd* __restrict__ out)
{
    extern __shared__ __align__(16) unsigned char sh_s1c[];
    zd* stw = (zd*)sh_s1c;
    zd* xa = stw + nz;
    zd* xb = xa + (size_t)NC * nz;
    const int f = blockIdx.z, j = blockIdx.y, kx0 = blockIdx.x * NC;
    const long long plane = ((long long)f * ny + j) * nz * nxh;
    load_twiddles(stw, tw, nz);
    for (int e = threadIdx.x; e < NC * nz; e += blockDim.x) {
        const int c = e % NC, kz = e / NC;
        xa[(size_t)c * nz + kz] = (kx0 + c < nxh) ? in[plane + (long long)kz * nxh + kx0 + c] : mk(0.0, 0.0);
    }
    const zd* r = fft_block<double, INV>(xa, xb, nz, NC, nz, stw);
    const double sc = INV ? 1.0 : 1.0 / nz;
    for (int e = threadIdx.x; e < NC * nz; e += blockDim.x) {
        const int c = e % NC, z = e / NC;
        if (kx0 + c < nxh) {
            const zd a = r[(size_t)c * nz + z];
            out[plane + (long long)z * nxh + kx0 + c] = mk(sc * a.x, sc * a.y);
        }
    }
}

// One (y, z) row: A[3][ny][nz][nxh] (x half spectra of u, v, w at fixed z)
// -> the x half spectra of uu, uv, uw, vv, vw, ww, scaled by 1 / nx, into
// B[6][ny][nz][nxh].
__global__ void k_s1_row_products(const zd* __restrict__ A, int ny, int nz, int nx, const zd* __restrict__ tw,
                                  zd* __restrict__ B)
{
    extern __shared__ __align__(16) unsigned char sh_s1r[];
    const int nxh = nx / 2 + 1;
    zd* stw = (zd*)sh_s1r;
    zd* xa = stw + nx;                 // 3 sequences of nx
    zd* xb = xa + 3 * (size_t)nx;      // 3 sequences of nx
    const int z = blockIdx.x, j = blockIdx.y;
    const long long fs = (long long)ny * nz * nxh, row = ((long long)j * nz + z) * nxh;
    load_twiddles(stw, tw, nx);
    // Hermitian extension of a half spectrum; the kx = 0 and nx/2 bins keep
    // their real parts (a real sequence's DFT is real there)
    auto H = [&](int f, int m) -> zd {
        if (m == 0 || 2 * m == nx) return mk(A[f * fs + row + m].x, 0.0);
        if (2 * m < nx) return A[f * fs + row + m];
        const zd a = A[f * fs + row + (nx - m)];
        return mk(a.x, -a.y);
    };
    for (int m = threadIdx.x; m < nx; m += blockDim.x) {
        const zd u = H(0, m), v = H(1, m), w = H(2, m);
        xa[m] = mk(u.x - v.y, u.y + v.x);             // U + i V
        xa[nx + m] = w;
    }
    zd* r = fft_block<double, true>(xa, xb, nx, 2, nx, stw);    // u + i v, w (+ 0 i)
    zd* o = (r == xa) ? xb : xa;
    for (int m = threadIdx.x; m < nx; m += blockDim.x) {
        const double u = r[m].x, v = r[m].y, w = r[nx + m].x;
        o[m] = mk(u * u, v * v);                        // uu + i vv
        o[nx + m] = mk(w * w, u * v);                   // ww + i uv
        o[2 * nx + m] = mk(u * w, v * w);               // uw + i vw
    }
    zd* q = fft_block<double, false>(o, r, nx, 3, nx, stw);
    // unpack a + i b: a^(m) = (Z(m) + conj Z(-m)) / 2, b^(m) = (Z(m) - conj Z(-m)) / (2 i)
    const double sc = 0.5 / nx;
    // output product index of (sequence, part): uu 0, uv 1, uw 2, vv 3, vw 4, ww 5
    const int dst[3][2] = {{0, 3}, {5, 1}, {2, 4}};
    for (int e = threadIdx.x; e < 3 * nxh; e += blockDim.x) {
        const int s = e / nxh, m = e - s * nxh;
        const zd Z = q[(size_t)s * nx + m], Zc = q[(size_t)s * nx + (nx - m) % nx];
        B[dst[s][0] * fs + row + m] = mk(sc * (Z.x + Zc.x), sc * (Z.y - Zc.y));
        B[dst[s][1] * fs + row + m] = mk(sc * (Z.y + Zc.y), sc * (Zc.x - Z.x));
    }
}

// The same by register transforms in fixed point (nz = N1 N2): CTA = CW
// columns x N2 lanes (256 threads); the forward scale is in the exponent.  k_s1_col's
// transforms are bound by the FP64 pipe (256 x 256 x 129: three inverse fields
// 676 -> 170 us, six forward ones 1408 -> 333 us).
template <int N1, int N2, bool INV>
__global__ void __launch_bounds__(256, 2)
k_s1_col_r(const zd* __restrict__ in, int ny, int nxh, const zd* __restrict__ tw, zd* __restrict__ out)
{
    constexpr int N = N1 * N2, CW = 256 / N2;
    extern __shared__ __align__(16) unsigned char sh_s1cr[];
    zd* stw = (zd*)sh_s1cr;
    zd* xs = stw + N;
    __shared__ int smx[256];
    const int c = threadIdx.x % CW, lane = threadIdx.x / CW;
    // columns (y, kx) of a field, consecutive kx first
    const long long q = (long long)blockIdx.x * CW + c;
    const int j = (int)(q / nxh), kx = (int)(q - (long long)j * nxh);
    const bool live = j < ny;
    const long long base = ((long long)blockIdx.y * ny + j) * N * nxh + kx;
    load_twiddles2l<double>(stw, tw, N);
    zd v[N1];
    #pragma unroll
    for (int m = 0; m < N1; ++m) v[m] = live ? in[base + (long long)(lane + N2 * m) * nxh] : mk(0.0, 0.0);
    __syncthreads();
    constexpr int lg = N == 32 ? 5 : N == 64 ? 6 : N == 128 ? 7 : 8;
    static_assert(N == 1 << lg, "register lengths");
    fft2l_cols<double, N1, N2, INV>(v, c, CW, lane, xs + c, N2 * CW + 1, CW, stw, smx, INV ? 0 : -lg);
    if (live) {
        #pragma unroll
        for (int m = 0; m < N1; ++m) out[base + (long long)(lane + N2 * m) * nxh] = v[m];
    }
}

// k_s1_row_products by register transforms (nx = N1 N2): a row on N2 lanes of
// a warp, u, v, w of the row in shared memory between the transforms
// (256 x 256 x 129: 2537 -> 679 us).
template <int N1, int N2>
__global__ void __launch_bounds__(64)
k_s1_row_products_r(const zd* __restrict__ A, int ny, int nz, const zd* __restrict__ tw, zd* __restrict__ B)
{
    constexpr int N = N1 * N2, nxh = N / 2 + 1, RZ = 64 / N2;
    extern __shared__ __align__(16) unsigned char sh_s1rr[];
    zd* stw = (zd*)sh_s1rr;
    zd* xs = stw + N;
    const int lane = threadIdx.x % N2, r = threadIdx.x / N2;
    const int z = blockIdx.x * RZ + r, j = blockIdx.y;
    const bool live = z < nz;
    const long long fs = (long long)ny * nz * nxh, row = ((long long)j * nz + (live ? z : 0)) * nxh;
    zd* xr = xs + r * N1 * (N2 + 1);
    double* ph = (double*)(xs + RZ * N1 * (N2 + 1)) + r * 3 * N + lane;
    load_twiddles2l<double>(stw, tw, N);
    __syncthreads();
    // Hermitian extension of a half spectrum; the kx = 0 and nx/2 bins keep
    // their real parts (a real sequence's DFT is real there)
    auto H = [&](int f, int m) -> zd {
        zd a = A[f * fs + row + (m < nxh ? m : N - m)];
        if (m >= nxh) a.y = -a.y;
        if (m == 0 || 2 * m == N) a.y = 0.0;
        return a;
    };
    #pragma unroll 1
    for (int q = 0; q < 2; ++q) {
        zd v[N1];
        #pragma unroll
        for (int m = 0; m < N1; ++m) {
            const int k = lane + N2 * m;
            if (q) v[m] = H(2, k);
            else {
                const zd a = H(0, k), b = H(1, k);
                v[m] = mk(a.x - b.y, a.y + b.x);              // U + i V
            }
        }
        __syncwarp();
        fft2l_rows<double, N1, N2, true>(v, lane, xr, N2 + 1, 1, stw);
        #pragma unroll
        for (int m = 0; m < N1; ++m) {
            ph[2 * q * N + N2 * m] = v[m].x;
            if (!q) ph[N + N2 * m] = v[m].y;
        }
    }
    // products of (sequence, part): uu + i vv, ww + i uv, uw + i vw; B's order uu 0, uv 1, uw 2, vv 3, vw 4, ww 5
    #pragma unroll 1
    for (int s = 0; s < 3; ++s) {
        zd f[N1];
        #pragma unroll
        for (int m = 0; m < N1; ++m) {
            const double u = ph[N2 * m], v = ph[N + N2 * m], w = ph[2 * N + N2 * m];
            f[m] = s == 0 ? mk(u * u, v * v) : s == 1 ? mk(w * w, u * v) : mk(u * w, v * w);
        }
        __syncwarp();
        zd* ba = B + (s == 0 ? 0 : s == 1 ? 5 : 2) * fs + row;
        zd* bb = B + (s == 0 ? 3 : s == 1 ? 1 : 4) * fs + row;
        fft2l_split<double, N1, N2>(f, lane, xr, stw, [&](int k, zd a, zd b) {
            if (live) { ba[k] = a; bb[k] = b; }
        });
    }
}

// band storage of wavenumber k: row r, column c (|c - r| within the window)
__device__ __forceinline__ double& band(double* ab, long long Nk, long long k, int r, int c)
{
    return ab[((long long)r * S1_W + (c - r + S1_KL)) * Nk + k];
}

// LU with partial pivoting of the Poisson operator of every wavenumber
__global__ void k_s1_factor(int ny, int nz, int nx, double Lx, double Lz, const double* __restrict__ w1,
                            const double* __restrict__ w2, const int* __restrict__ l0, double* __restrict__ ab,
                            unsigned char* __restrict__ piv)
{
    const int nxh = nx / 2 + 1;
    const long long Nk = (long long)nz * nxh;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Nk) return;
    const int kz_i = (int)(k / nxh), kx_i = (int)(k - (long long)kz_i * nxh);
    const double k2 = ktrue2(kx_i, nx, Lx) + ktrue2(kz_i, nz, Lz);
    for (int r = 0; r < ny; ++r)
        for (int c = 0; c < S1_W; ++c) ab[((long long)r * S1_W + c) * Nk + k] = 0.0;
    for (int r = 0; r < ny; ++r) {
        const bool wall = (r == 0 || r == ny - 1);
        for (int l = 0; l < 5; ++l) band(ab, Nk, k, r, l0[r] + l) = wall ? w1[5 * r + l] : w2[5 * r + l];
        if (!wall) band(ab, Nk, k, r, r) -= k2;
    }
    if (k2 == 0.0) {                                  // p(y_0) = 0
        for (int l = 0; l < 5; ++l) band(ab, Nk, k, 0, l) = 0.0;
        band(ab, Nk, k, 0, 0) = 1.0;
    }
    for (int j = 0; j < ny; ++j) {
        const int rmax = min(j + S1_KL, ny - 1), cmax = min(j + S1_KL + S1_KU, ny - 1);
        int p = j;
        double best = fabs(band(ab, Nk, k, j, j));
        for (int r = j + 1; r <= rmax; ++r) {
            const double a = fabs(band(ab, Nk, k, r, j));
            if (a > best) { best = a; p = r; }
        }
        piv[(long long)j * Nk + k] = (unsigned char)(p - j);
        if (p != j)
            for (int c = j; c <= cmax; ++c) {
                const double t = band(ab, Nk, k, j, c);
                band(ab, Nk, k, j, c) = band(ab, Nk, k, p, c);
                band(ab, Nk, k, p, c) = t;
            }
        const double d = band(ab, Nk, k, j, j);
        for (int r = j + 1; r <= rmax; ++r) {
            const double m = band(ab, Nk, k, r, j) / d;
            band(ab, Nk, k, r, j) = m;
            if (m != 0.0)
                for (int c = j + 1; c <= cmax; ++c) band(ab, Nk, k, r, c) -= m * band(ab, Nk, k, j, c);
        }
    }
}

// Source and wall values of one snapshot: P[6][ny][Nk] (product spectra uu,
// uv, uw, vv, vw, ww), v = the snapshot's v spectra, into b[ny][Nk].  Thread =
// one wavenumber, S1_ROWS rows.  Bound by the FP64 pipe: kx uv + kz vw is formed
// once per row and differentiated, and with the wavenumbers' rows spread over
// the chip (and apart from the solve) no thread waits for its own serial loads
// (256 x 256 x 129: source and solve in one thread per wavenumber 1284 us, now
// 324 + 413 us).
__global__ void k_s1_source(const zd* __restrict__ P, const zd* __restrict__ v, int ny, int nz, int nx, double Lx,
                            double Lz, double nu, const double* __restrict__ w1, const double* __restrict__ w2,
                            const int* __restrict__ l0, zd* __restrict__ b)
{
    const int nxh = nx / 2 + 1;
    const long long Nk = (long long)nz * nxh, fs = (long long)ny * Nk;
    const long long k = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (k >= Nk) return;
    const int kz_i = (int)(k / nxh), kx_i = (int)(k - (long long)kz_i * nxh);
    const double kx = kodd(kx_i, nx, Lx), kz = kodd(kz_i, nz, Lz);
    const double kx2 = ktrue2(kx_i, nx, Lx), kz2 = ktrue2(kz_i, nz, Lz), k2 = kx2 + kz2, kxz = 2.0 * kx * kz;
    const int j0 = blockIdx.y * S1_ROWS, j1 = min(j0 + S1_ROWS, ny);
    const zd *Puu = P + k, *Puv = Puu + fs, *Puw = Puv + fs, *Pvv = Puw + fs, *Pvw = Pvv + fs, *Pww = Pvw + fs;
    auto getv = [&](int r) { return Pvv[(long long)r * Nk]; };
    auto getc = [&](int r) {
        const zd c = Puv[(long long)r * Nk], d = Pvw[(long long)r * Nk];
        return mk(kx * c.x + kz * d.x, kx * c.y + kz * d.y);
    };
    Window wv, wc;
    wv.open(l0[j0], getv);
    wc.open(l0[j0], getc);
    for (int r = j0; r < j1; ++r) {
        const long long i = (long long)r * Nk;
        wv.seek(l0[r], getv);
        wc.seek(l0[r], getc);
        zd o;
        if (r == 0 || r == ny - 1) {
            zd d2v = mk(0.0, 0.0);
            for (int l = 0; l < 5; ++l) {
                const zd a = v[(long long)(l0[r] + l) * Nk + k];
                d2v = mk(d2v.x + w2[5 * r + l] * a.x, d2v.y + w2[5 * r + l] * a.y);
            }
            o = (r == 0 && k2 == 0.0) ? mk(0.0, 0.0) : mk(nu * d2v.x, nu * d2v.y);
        } else {
            // d_i d_j (u_i u_j) = -kx^2 uu - kz^2 ww + (vv)'' - 2 kx kz uw + 2 i kx (uv)' + 2 i kz (vw)'
            const zd uu = Puu[i], ww = Pww[i], uw = Puw[i], vv2 = wv.apply(w2 + 5 * r), c1 = wc.apply(w1 + 5 * r);
            o = mk(kx2 * uu.x + kz2 * ww.x - vv2.x + kxz * uw.x + 2.0 * c1.y,
                   kx2 * uu.y + kz2 * ww.y - vv2.y + kxz * uw.y - 2.0 * c1.x);
        }
        b[i + k] = o;
    }
}

// The banded solve: thread = the real or the imaginary part of one wavenumber
// (b, p as doubles; two neighbours read the same factors).  The rows in reach are a
// window of registers, and the next row's factors are read a step ahead.
__global__ void __launch_bounds__(64)
k_s1_solve(const double* __restrict__ b, int ny, long long Nk, const double* __restrict__ ab,
           const unsigned char* __restrict__ piv, double* __restrict__ p)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x, k = i >> 1, S = 2 * Nk;
    if (k >= Nk) return;
    // forward substitution with the row exchanges; x[q] = row j + q
    double x[S1_KL + 1], m[S1_KL];
    auto mult = [&](int j, int q) {                   // multiplier of row j + q, 1 <= q <= KL
        return j + q < ny ? ab[((long long)(j + q) * S1_W + (S1_KL - q)) * Nk + k] : 0.0;
    };
    #pragma unroll
    for (int q = 0; q <= S1_KL; ++q) x[q] = q < ny ? b[q * S + i] : 0.0;
    #pragma unroll
    for (int q = 0; q < S1_KL; ++q) m[q] = mult(0, q + 1);
    int pv = piv[k];
    for (int j = 0; j < ny; ++j) {
        double mn[S1_KL];
        #pragma unroll
        for (int q = 0; q < S1_KL; ++q) mn[q] = mult(j + 1, q + 1);
        const int pn = j + 1 < ny ? piv[(long long)(j + 1) * Nk + k] : 0;
        const double xn = j + S1_KL + 1 < ny ? b[(long long)(j + S1_KL + 1) * S + i] : 0.0;
        double top = x[0];
        #pragma unroll
        for (int q = 1; q <= S1_KL; ++q)
            if (pv == q) { top = x[q]; x[q] = x[0]; }
        p[(long long)j * S + i] = top;
        #pragma unroll
        for (int q = 0; q < S1_KL; ++q) { x[q] = x[q + 1] - m[q] * top; m[q] = mn[q]; }
        x[S1_KL] = xn;
        pv = pn;
    }
    // back substitution; y[q] = row j + 1 + q
    constexpr int KW = S1_KU + S1_KL;
    double y[KW], a[KW], d, s;
    auto fact = [&](int j, int q) {                   // coefficient of row j on row j + q
        return j >= 0 && j + q < ny ? ab[((long long)j * S1_W + (S1_KL + q)) * Nk + k] : 0.0;
    };
    #pragma unroll
    for (int q = 0; q < KW; ++q) { y[q] = 0.0; a[q] = fact(ny - 1, q + 1); }
    d = fact(ny - 1, 0);
    s = p[(long long)(ny - 1) * S + i];
    for (int j = ny - 1; j >= 0; --j) {
        double an[KW];
        #pragma unroll
        for (int q = 0; q < KW; ++q) an[q] = fact(j - 1, q + 1);
        const double dn = fact(j - 1, 0), sn = j > 0 ? p[(long long)(j - 1) * S + i] : 0.0;
        #pragma unroll
        for (int q = 0; q < KW; ++q) s -= a[q] * y[q];
        const double xj = s / d;
        p[(long long)j * S + i] = xj;
        #pragma unroll
        for (int q = KW - 1; q > 0; --q) y[q] = y[q - 1];
        y[0] = xj;
        #pragma unroll
        for (int q = 0; q < KW; ++q) a[q] = an[q];
        d = dn;
        s = sn;
    }
}

// ------------------------------------------------------------ launchers
size_t s1_band_doubles(int ny, long long Nk) { return (size_t)ny * S1_W * (size_t)Nk; }

static int col_nc(int nz) { return nz <= 256 ? 8 : 4; }
static size_t col_smem(int nz) { return (size_t)(1 + 2 * col_nc(nz)) * nz * sizeof(zd); }
static size_t row_smem(int nx) { return (size_t)7 * nx * sizeof(zd); }

// register transforms, but those of 32 points only where enough rows hide their
// longer chain of integer instructions (a call of 2 snapshots, us, shared memory against
// registers: 32 x 32 x 9 187 / 199, x 17 270 / 274, x 25 315 / 302, x 33 354 / 336, x 129 846 / 679; 32 x 8 x 65
// 435 / 443, x 129 696 / 687)
static bool s1_reg(int n, int other, int ny) { return reg_len(n) && (n > 32 || (long long)other * ny >= 1024); }
static size_t col_r_smem(int n1, int n2) { return (size_t)(n1 * n2 + n1 * (256 + 1)) * sizeof(zd); }
static size_t row_r_smem(int n1, int n2)
{
    const int rz = 64 / n2;
    return (size_t)(n1 * n2 + rz * n1 * (n2 + 1)) * sizeof(zd) + (size_t)rz * 3 * n1 * n2 * sizeof(double);
}

cudaError_t s1_set_attrs(int nx, int nz)
{
    cudaError_t e = cudaSuccess;
    auto attr = [&](const void* k, size_t sh) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sh);
    };
    attr((const void*)k_s1_col<true>, col_smem(nz));
    attr((const void*)k_s1_col<false>, col_smem(nz));
    attr((const void*)k_s1_row_products, row_smem(nx));
    if (reg_len(nz))
        with_reg_len(nz, [&](auto L) {
            typedef decltype(L) R;
            attr((const void*)k_s1_col_r<R::N1, R::N2, true>, col_r_smem(R::N1, R::N2));
            attr((const void*)k_s1_col_r<R::N1, R::N2, false>, col_r_smem(R::N1, R::N2));
        });
    if (reg_len(nx))
        with_reg_len(nx, [&](auto L) {
            typedef decltype(L) R;
            attr((const void*)k_s1_row_products_r<R::N1, R::N2>, row_r_smem(R::N1, R::N2));
        });
    return e;
}

int s1_factor_launch(int ny, int nz, int nx, double Lx, double Lz, const double* w1, const double* w2, const int* l0,
                     double* ab, unsigned char* piv, cudaStream_t st)
{
    const long long Nk = (long long)nz * (nx / 2 + 1);
    k_s1_factor<<<(unsigned)((Nk + 127) / 128), 128, 0, st>>>(ny, nz, nx, Lx, Lz, w1, w2, l0, ab, piv);
    return 1;
}

int s1_snapshot_launch(const zd* v_eta, const double* mean_uw, int ny, int nz, int nx, double Lx, double Lz,
                       double nu, const double* w1, const double* w2, const int* l0, const zd* tw_x, const zd* tw_z,
                       const double* ab, const unsigned char* piv, zd* bufA, zd* bufB, zd* out, cudaStream_t st)
{
    const int nxh = nx / 2 + 1;
    const long long Nk = (long long)nz * nxh, fs = (long long)ny * Nk;
    const dim3 gk((unsigned)((Nk + 127) / 128), (unsigned)((ny + S1_ROWS - 1) / S1_ROWS));
    k_s1_velocity<<<gk, 128, 0, st>>>(v_eta, v_eta + fs, mean_uw, ny, nz, nx, Lx, Lz, w1, l0, out);
    const int nc = col_nc(nz);
    const bool reg_z = s1_reg(nz, 2 * nxh, ny), reg_x = s1_reg(nx, nz, ny);
    auto col = [&](auto inv, const zd* in, int nf, zd* o) {
        constexpr bool INV = decltype(inv)::value;
        if (!reg_z) {
            const dim3 g((unsigned)((nxh + nc - 1) / nc), (unsigned)ny, (unsigned)nf);
            k_s1_col<INV><<<g, 256, col_smem(nz), st>>>(in, ny, nz, nxh, nc, tw_z, o);
            return;
        }
        with_reg_len(nz, [&](auto L) {
            typedef decltype(L) R;
            constexpr int cw = 256 / R::N2;
            const dim3 g((unsigned)(((long long)ny * nxh + cw - 1) / cw), (unsigned)nf);
            k_s1_col_r<R::N1, R::N2, INV><<<g, 256, col_r_smem(R::N1, R::N2), st>>>(in, ny, nxh, tw_z, o);
        });
    };
    col(std::true_type(), out, 3, bufA);
    if (reg_x)
        with_reg_len(nx, [&](auto L) {
            typedef decltype(L) R;
            constexpr int rz = 64 / R::N2;
            const dim3 g((unsigned)((nz + rz - 1) / rz), (unsigned)ny);
            k_s1_row_products_r<R::N1, R::N2><<<g, 64, row_r_smem(R::N1, R::N2), st>>>(bufA, ny, nz, tw_x, bufB);
        });
    else
        k_s1_row_products<<<dim3((unsigned)nz, (unsigned)ny), 256, row_smem(nx), st>>>(bufA, ny, nz, nx, tw_x, bufB);
    col(std::false_type(), bufB, 6, bufA);
    k_s1_source<<<gk, 128, 0, st>>>(bufA, out + fs, ny, nz, nx, Lx, Lz, nu, w1, w2, l0, bufB);
    k_s1_solve<<<(unsigned)((2 * Nk + 63) / 64), 64, 0, st>>>((const double*)bufB, ny, Nk, ab, piv, (double*)(out + 3 * fs));
    return 6;
}

}  // namespace gke
