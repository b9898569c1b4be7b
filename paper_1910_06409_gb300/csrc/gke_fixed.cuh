// gke_fixed.cuh -- the FP64 register transforms in 64-bit fixed point.
//
// The FP64 pipe does 2 operations a clock and SM, the integer units 64: a
// 64-bit addition costs 2 instructions against 16 clocks, a multiplication by a
// constant about 7.  So a sequence of a two-level transform (fft2l) is turned
// into integers on its own exponent E, transformed, and turned back into FP64,
// all in integer instructions.
//
// E comes from the sequence's 1-norm, sum (|re| + |im|) < 2^E: no partial sum of a
// transform exceeds it, so the integers take 61 bits below 2^E and nothing
// overflows (x +- y of a complex value: 2^61.5).  Rounding: half a unit 2^(E - 61) per
// input, half a unit per constant product, and S = 2 bits in the twiddle product;
// at N = 256 about 7 units in an output, 2^-58 of 2^E.  2^E is at most twice the 1-norm and
// that sqrt(2 N) = 22.6 times the 2-norm, so at worst 2^-52.7 of the 2-norm; an
// FP64 transform's error is about 2^-52.3 of it.
//
// Measured (FP64 transforms -> here): 256 x 256 x 65, 16 snapshots: inverse transforms
// of the terms 56.9 -> 19.7 ms, products stage 46.7 -> 21.1 ms; duct 256 x 33 x 33:
// 30.0 -> 9.9 ms; 128 x 128 x 65, 32 snapshots (from shared-memory stages of FP64):
// products 28.7 -> 11.1 ms, terms 15.3 -> 4.9 ms.  Errors of the terms against 64-bit references do not grow (duct
// A 1.7e-16 -> 1.1e-16).  (Exponents from the largest component and 56 bits were as
// fast, but raised them by up to a half.)
#pragma once
#include "gke_common.cuh"

namespace gke {

typedef cplx<long long> zx;

constexpr int FX_S = 2;                                   // bits dropped by the twiddle product
constexpr int FX_IB = 61;                                 // bits of the integers below the 1-norm's power of two
// (twiddle table: cos, sin times 2^(64 - FX_S) = 2^62)

__device__ __forceinline__ int fx_lo(long long a) { return (int)a; }
// upper word for a signed lower word: a = hi 2^32 + lo
__device__ __forceinline__ int fx_hi(long long a) { return (int)(a >> 32) + (int)((unsigned)(int)a >> 31); }

// round(a c) for |a| < 2^62, |c| < 1 given as c 2^63 = ch 2^32 + cl (signed words)
__device__ __forceinline__ long long fx_mulc(long long a, int ch, int cl)
{
    const int l = fx_lo(a), h = fx_hi(a);
    const long long t = (long long)h * cl + ((long long)l * ch + (1ll << 30));
    return (long long)(2 * h) * ch + (t >> 31);
}

// round(a w / 4): the twiddle product of fft2l, w from the table (2^62)
__device__ __forceinline__ zx operator*(zx a, zx w)
{
    const int al = fx_lo(a.x), ah = fx_hi(a.x), bl = fx_lo(a.y), bh = fx_hi(a.y);
    const int cl = fx_lo(w.x), ch = fx_hi(w.x), dl = fx_lo(w.y), dh = fx_hi(w.y);
    const long long n = -w.y;
    const int nl = fx_lo(n), nh = fx_hi(n);
    const long long half = 1ll << 31;
    const long long tr = (long long)ah * cl + ((long long)al * ch + ((long long)bh * nl + ((long long)bl * nh + half)));
    const long long ti = (long long)ah * dl + ((long long)al * dh + ((long long)bh * cl + ((long long)bl * ch + half)));
    zx r;
    r.x = (long long)ah * ch + ((long long)bh * nh + (tr >> 32));
    r.y = (long long)ah * dh + ((long long)bh * ch + (ti >> 32));
    return r;
}
__device__ __forceinline__ long long fx_mid(long long a) { return (a + (1 << (FX_S - 1))) >> FX_S; }

// W_32^m for the register DFTs: constants times 2^63, rounded to integers, as signed word
// pairs (an FP64 constant is up to 8.5e-17 of itself off, sqrt(1/2) 6.8e-17 too large, and every
// value of a stage would carry that)
struct FxC { int h, l; };
__host__ __device__ constexpr FxC fxc(long long v)
{
    return FxC{(int)((v - (long long)(int)(v & 0xffffffffll)) >> 32), (int)(v & 0xffffffffll)};
}
template <bool INV> __device__ __forceinline__ zx fx_twiddle(zx w, int m)
{
    constexpr FxC q = fxc(6521908912666391106ll);
    if (m == 0) return w;
    if (m == 8) return INV ? mk(-w.y, w.x) : mk(w.y, -w.x);
    if (m == 4 || m == 12) {
        const long long s = fx_mulc(w.x + w.y, q.h, q.l), d = fx_mulc(w.x - w.y, q.h, q.l);
        if (m == 4) return INV ? mk(d, s) : mk(s, -d);
        return INV ? mk(-s, d) : mk(-d, -s);
    }
    // cos, sin of 2 pi m / 32 in the first octant, then by symmetry
    constexpr FxC c1 = fxc(9046147529429926059ll), s1 = fxc(1799390620744551094ll), c2 = fxc(8521284645587064995ll),
                  s2 = fxc(3529631669043774883ll), c3 = fxc(7668953571605777421ll), s3 = fxc(5124230951741890994ll);
    const int k = m < 8 ? m : 16 - m;                       // cos of m in 9..15 is minus that of 16 - m
    const FxC c = k == 1 ? c1 : k == 2 ? c2 : k == 3 ? c3 : k == 5 ? s3 : k == 6 ? s2 : s1;
    const FxC s = k == 1 ? s1 : k == 2 ? s2 : k == 3 ? s3 : k == 5 ? c3 : k == 6 ? c2 : c1;
    long long cx = fx_mulc(w.x, c.h, c.l), cy = fx_mulc(w.y, c.h, c.l);
    const long long sx = fx_mulc(w.x, s.h, s.l), sy = fx_mulc(w.y, s.h, s.l);
    if (m > 8) { cx = -cx; cy = -cy; }
    // w (c - i s), conjugate if INV
    return INV ? mk(cx - sy, cy + sx) : mk(cx + sy, cy - sx);
}
template <> __device__ __forceinline__ zx twiddle_mul<long long, false>(zx w, int m) { return fx_twiddle<false>(w, m); }
template <> __device__ __forceinline__ zx twiddle_mul<long long, true>(zx w, int m) { return fx_twiddle<true>(w, m); }

// ------------------------------------------------------------ conversions
// x 2^(FX_IB - E) rounded, s = E + 1085 - FX_IB (the exponent field of |x| < 2^E is at
// most E + 1022, so every shift is at least 2)
__device__ __forceinline__ long long fx_from(double x, int s)
{
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const unsigned mh = ((unsigned)hi & 0xfffffu) | 0x100000u;
    const unsigned long long m = ((unsigned long long)__funnelshift_l((unsigned)lo, mh, 10) << 32) | ((unsigned)lo << 10);
    const int r = s - 1 - ((hi >> 20) & 0x7ff);                          // >= 1
    const long long v = (long long)(((m >> min(r, 63)) + 1) >> 1);
    const long long sg = (long long)(hi >> 31);
    return (v ^ sg) - sg;
}
// v 2^e, exponents known to stay in the normal range.  Ties go to even: a transform's results have
// only a few bits to drop, so ties are frequent, and away from zero they would raise the
// energy (by 2.5e-17 to 4e-17 in the two transforms of 32 or 128 points a side).
__device__ __forceinline__ double fx_to(long long v, int e)
{
    const unsigned sg = (unsigned)((int)(v >> 32) >> 31);
    const unsigned long long m = ((unsigned long long)v ^ (((unsigned long long)sg << 32) | sg)) + (sg & 1u);
    unsigned h = (unsigned)(m >> 32), l = (unsigned)m;
    const bool z = h == 0;
    if (z) { h = l; l = 0; }
    const int lz = __clz((int)h);
    const unsigned mh = __funnelshift_l(l, h, lz), ml = l << (lz & 31);
    unsigned rl = __funnelshift_r(ml, mh, 11), rh = (mh >> 11) + ((unsigned)(1022 + 63 + e - (z ? 32 : 0) - lz) << 20);
    const unsigned up = ((ml & 0x7ffu) + 0x3ffu + (rl & 1u)) >> 11;
    rl += up;
    rh += rl < up;
    return h == 0 ? 0.0 : __hiloint2double((int)(rh | (sg & 0x80000000u)), (int)rl);
}

constexpr int FX_NAN = 8192;                              // exponent of a sequence with an infinity or a NaN
__device__ __forceinline__ bool fx_safe(int E) { return E > -900 && E < 900; }
// v 2^e of a sequence of any exponent E
__device__ __noinline__ static double fx_to_edge(long long v, int e, int E)
{
    return E == FX_NAN ? __longlong_as_double(0x7ff8000000000000ll) : scalbn((double)v, e);
}
__device__ __noinline__ static double fx_scale_edge(double x, int e) { return scalbn(x, e); }
// Two-level transform of a sequence in fixed point: fft2l's arguments; E: the
// sequence's exponent.  put(m, w, false) takes output m of this thread, the
// value w 2^(E - FX_IB + FX_S), |w| < 2^59.5; exponents near the ends of the FP64
// range take the conversions of the math library and put(m, w, true) as well.
template <int N1, int N2, bool INV, bool WARP, typename F>
__device__ __forceinline__ void fft2l_raw(const zd* v, int E, int lane, zx* xs, int s1, int s2, const zx* stw, F put)
{
    static_assert(N1 % N2 == 0, "N1 must be a multiple of N2");
    constexpr int R = N1 / N2;
    zx w[N1];
    if (fx_safe(E)) {
        const int s = E + 1085 - FX_IB;
        #pragma unroll
        for (int j = 0; j < N1; ++j) w[j] = mk(fx_from(v[j].x, s), fx_from(v[j].y, s));
    } else {
        #pragma unroll
        for (int j = 0; j < N1; ++j)
            w[j] = mk((long long)rint(fx_scale_edge(v[j].x, FX_IB - E)), (long long)rint(fx_scale_edge(v[j].y, FX_IB - E)));
    }
    dft_reg<long long, N1, INV>(w);
    w[0] = mk(fx_mid(w[0].x), fx_mid(w[0].y));
    #pragma unroll
    for (int k1 = 1; k1 < N1; ++k1) {
        zx t = stw[lane * k1];
        if (INV) t.y = -t.y;
        w[k1] = w[k1] * t;
    }
    #pragma unroll
    for (int k1 = 0; k1 < N1; ++k1) xs[k1 * s1 + lane * s2] = w[k1];
    sync_lanes<WARP>();
    #pragma unroll
    for (int jj = 0; jj < R; ++jj) {
        const int k1 = lane + N2 * jj;
        zx b[N2];
        #pragma unroll
        for (int n2 = 0; n2 < N2; ++n2) b[n2] = xs[k1 * s1 + n2 * s2];
        dft_reg<long long, N2, INV>(b);
        #pragma unroll
        for (int k2 = 0; k2 < N2; ++k2) put(jj + R * k2, b[k2], false);
        if (!fx_safe(E)) {
            #pragma unroll
            for (int k2 = 0; k2 < N2; ++k2) put(jj + R * k2, b[k2], true);
        }
    }
}
// the same back to FP64, times 2^sh
template <int N1, int N2, bool INV, bool WARP>
__device__ __forceinline__ void fft2l_fixed(zd* v, int E, int sh, int lane, zx* xs, int s1, int s2, const zx* stw)
{
    const int e = E - FX_IB + FX_S + sh;
    fft2l_raw<N1, N2, INV, WARP>(v, E, lane, xs, s1, s2, stw, [&](int m, zx w, bool edge) {
        v[m] = edge ? mk(fx_to_edge(w.x, e, E), fx_to_edge(w.y, e, E)) : mk(fx_to(w.x, e), fx_to(w.y, e));
    });
}

// lengths with a register transform
inline bool fx_len(int n) { return n == 32 || n == 64 || n == 128 || n == 256 || n == 512; }
// cos, sin of 2 pi m / 512 times 2^62, rounded, m = 0 .. 64
static const long long fx_octant[65][2] = {
    {4611686018427387904ll, 0ll}, {4611338766951757487ll, 56592481536850979ll},
    {4610297064819661174ll, 113176440454146016ll}, {4608561068907608378ll, 169743355415804323ll},
    {4606131040650197959ll, 226284707652502141ll}, {4603007346000747137ll, 282791982244568062ll},
    {4599190455376180266ll, 339256669404298611ll}, {4594680943586185780ll, 395670265757500976ll},
    {4589479489746651964ll, 452024275624069880ll}, {4583586877177394601ll, 508310212297405757ll},
    {4577003993284191887ll, 564519599322481549ll}, {4569731829425144391ll, 620643971772365654ll},
    {4561771480761380163ll, 676674877523008785ll}, {4553124146092127503ll, 732603878526102765ll},
    {4543791127674180203ll, 788422552079819562ll}, {4533773831025782466ll, 844122492097239204ll},
    {4523073764714963030ll, 899695310372275547ll}, {4511692540132350364ll, 955132637842909263ll},
    {4499631871248503178ll, 1010426125851537790ll}, {4486893574355792752ll, 1065567447402252463ll},
    {4473479567794875989ll, 1120548298414853464ll}, {4459391871665800370ll, 1175360398975413759ll},
    {4444632607523784314ll, 1229995494583203681ll}, {4429203998059718770ll, 1284445357393788370ll},
    {4413108366765438139ll, 1338701787458110889ll}, {4396348137583810956ll, 1392756613957374385ll},
    {4378925834543703005ll, 1446601696433537347ll}, {4360844081379867860ll, 1500228926015236645ll},
    {4342105601137822079ll, 1553630226638953726ll}, {4322713215763764567ll, 1606797556265240081ll},
    {4302669845679601858ll, 1659722908089818799ll}, {4281978509343143317ll, 1712398311749379842ll},
    {4260642322793532497ll, 1764815834521887442ll}, {4238664499181983110ll, 1816967582521218861ll},
    {4216048348287890265ll, 1868845701885954606ll}, {4192797276020389871ll, 1920442379962141067ll},
    {4168914783905441250ll, 1971749846479847467ll}, {4144404468558510201ll, 2022760374723339936ll},
    {4119270021142931949ll, 2073466282694696471ll}, {4093515226814035515ll, 2123859934270687573ll},
    {4067143964149113252ll, 2173933740352748318ll}, {4040160204563321371ll, 2223680160009868681ll},
    {4012568011711599423ll, 2273091701614230011ll}, {3984371540876698815ll, 2322160923969416627ll},
    {3955575038343412514ll, 2370880437431032621ll}, {3926182840759100170ll, 2419242905019555129ll},
    {3896199374480604983ll, 2467241043525256456ll}, {3865629154907660636ll, 2514867624605028673ll},
    {3834476785802888710ll, 2562115475870945497ll}, {3802746958598488966ll, 2608977481970397539ll},
    {3770444451689726907ll, 2655446585657638225ll}, {3737574129715325036ll, 2701515788856579055ll},
    {3704140942824866152ll, 2747178153714674114ll}, {3670149925933319029ll, 2792426803647735152ll},
    {3635606197962798751ll, 2837254924375519865ll}, {3600514961071675858ll, 2881655764947937435ll},
    {3564881499871150442ll, 2925622638761716784ll}, {3528711180629409129ll, 2969148924567384428ll},
    {3492009450463484836ll, 3012228067466400296ll}, {3454781836518940978ll, 3054853579898301336ll},
    {3417033945137503676ll, 3097019042617704261ll}, {3378771461012767319ll, 3138718105661020291ll},
    {3340000146334100615ll, 3179944489302736311ll}, {3300725839918882066ll, 3220691985001118434ll},
    {3260954456333195553ll, 3260954456333195553ll}};
// host: the fixed-point twiddles e^{-2 pi i m / n} of a register length n behind the n FP64
// ones (tab[2 n]), from the first octant by symmetry
inline void fx_table(int n, zd* tab)
{
    if (!fx_len(n)) return;
    zx* f = (zx*)(tab + n);
    for (int m = 0; m < n; ++m) {
        const int k = m * (512 / n), q = k >> 7, r = k & 127;             // quarter turns, remainder
        const long long c = r <= 64 ? fx_octant[r][0] : fx_octant[128 - r][1];
        const long long s = r <= 64 ? fx_octant[r][1] : fx_octant[128 - r][0];
        f[m].x = q == 0 ? c : q == 1 ? -s : q == 2 ? -c : s;
        f[m].y = -(q == 0 ? s : q == 1 ? c : q == 2 ? -s : -c);
    }
}

// |x| in FP32, from its upper word, times 2^(896 - bias); the usual bias is 896, the
// difference of the FP64 and FP32 exponent offsets
__device__ __forceinline__ float fx_mag(double x, int bias)
{
    return __int_as_float(min(max((__double2hiint(x) & 0x7fffffff) - (bias << 20), 0), 0x0fe00000) << 3);
}
// 1-norm of this thread's values, scaled so
template <int N1> __device__ __forceinline__ float fx_norm(const zd* v, int bias)
{
    float s = 0.f;
    #pragma unroll
    for (int j = 0; j < N1; ++j) s += fx_mag(v[j].x, bias) + fx_mag(v[j].y, bias);
    return s;
}
// largest upper word of |re|, |im|
template <int N1> __device__ __forceinline__ int fx_max(const zd* v)
{
    int m = 0;
    #pragma unroll
    for (int j = 0; j < N1; ++j)
        m = max(m, max(__double2hiint(v[j].x) & 0x7fffffff, __double2hiint(v[j].y) & 0x7fffffff));
    return m;
}
// whether s leaves FP32's range although the values are not all zero
template <int N1> __device__ __forceinline__ bool fx_far(float s, const zd* v)
{
    return !(s > 1e-30f && s < 1e30f) && fx_max<N1>(v) != 0;
}
// the exponent E of a sequence whose norms sum to s (under bias); 0 for zeros
__device__ __forceinline__ int fx_exponent(float s, int bias)
{
    return s > 0.f ? ((__float_as_int(s * 1.001f) >> 23) & 0xff) - 126 + bias - 896 : 0;
}

template <int N2, typename T, typename F> __device__ __forceinline__ T fx_reduce(T x, F f)
{
    #pragma unroll
    for (int o = N2 / 2; o > 0; o >>= 1) x = f(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
}
// the exponent of a sequence held by N2 consecutive threads of a warp
template <int N1, int N2> __device__ __forceinline__ int fx_rows_exponent(const zd* v)
{
    auto add = [](float a, float b) { return a + b; };
    float s = fx_reduce<N2>(fx_norm<N1>(v, 896), add);
    int bias = 896;
    if (__any_sync(0xffffffffu, fx_far<N1>(s, v))) {
        bias = (fx_reduce<N2>(fx_max<N1>(v), [](int a, int b) { return max(a, b); }) >> 20) - 127;
        s = fx_reduce<N2>(fx_norm<N1>(v, bias), add);
        if (bias == 0x7ff - 127) return FX_NAN;
    }
    return fx_exponent(s, bias);
}

// Two sequences a, b in one transform (a + i b of real, or A + i B of Hermitian
// sequences): the sum of both would round each at the size of the larger.  Each has its
// own exponent (from its 1-norm), the smaller is scaled up to the larger's by a power of
// two and the result's half scaled back: both come out as if transformed alone.
constexpr int FX_ZERO = -9000;                            // exponent of a sequence of zeros
// the exponent of get(0) .. get(N1 - 1) of N2 consecutive threads of a warp
template <int N1, int N2, typename G> __device__ __forceinline__ int fx_part_exponent(G get)
{
    auto add = [](float a, float b) { return a + b; };
    float s = 0.f;
    int m = 0;
    #pragma unroll
    for (int j = 0; j < N1; ++j) {
        const zd v = get(j);
        s += fx_mag(v.x, 896) + fx_mag(v.y, 896);
        m = max(m, max(__double2hiint(v.x) & 0x7fffffff, __double2hiint(v.y) & 0x7fffffff));
    }
    const bool far = !(s > 1e-30f && s < 1e30f) && m != 0;
    s = fx_reduce<N2>(s, add);
    int bias = 896;
    if (__any_sync(0xffffffffu, far)) {
        m = fx_reduce<N2>(m, [](int a, int b) { return max(a, b); });
        bias = (m >> 20) - 127;
        s = 0.f;
        #pragma unroll
        for (int j = 0; j < N1; ++j) {
            const zd v = get(j);
            s += fx_mag(v.x, bias) + fx_mag(v.y, bias);
        }
        s = m == 0 ? 0.f : fx_reduce<N2>(s, add);
        if (bias == 0x7ff - 127) return FX_NAN;
    }
    return s > 0.f ? fx_exponent(s, bias) : FX_ZERO;
}
// exponent of the sum, powers of two that a and b are scaled up by; a part with an
// infinity or a NaN is left out of the transform (its results are NaN)
struct FxPair {
    int E, up[2];
    bool nan[2], safe;
    __device__ __forceinline__ FxPair(int ea, int eb)
    {
        nan[0] = ea == FX_NAN; nan[1] = eb == FX_NAN;
        if (nan[0]) ea = FX_ZERO;
        if (nan[1]) eb = FX_ZERO;
        const int top = max(ea, eb);
        up[0] = ea == FX_ZERO ? 0 : top - ea;
        up[1] = eb == FX_ZERO ? 0 : top - eb;
        E = top == FX_ZERO ? 0 : top + (ea != FX_ZERO && eb != FX_ZERO);
        safe = fx_safe(E) && fx_safe(E - up[0]) && fx_safe(E - up[1]);
    }
    // a value of part h, scaled up
    __device__ __forceinline__ double in(int h, double x) const
    {
        const int hi = __double2hiint(x);
        if (nan[h]) return 0.0;
        if (up[h] == 0) return x;
        if ((hi & 0x7ff00000) == 0) return x == 0.0 ? x : fx_scale_edge(x, up[h]);
        return __hiloint2double(hi + (up[h] << 20), __double2loint(x));
    }
    // an output w 2^e of part h, scaled back
    __device__ __forceinline__ double out(int h, long long w, int e) const
    {
        if (nan[h]) return __longlong_as_double(0x7ff8000000000000ll);
        return safe ? fx_to(w, e - up[h]) : fx_to_edge(w, e - up[h], 0);
    }
};

// fft2l with the lanes of a sequence side by side (N2 consecutive threads of a
// warp, xs their own: synchronises the warp only) or spread over the block
// (thread = seq + nseq * lane; smx: a shared array of one int per thread).
// Norms outside FP32's range are taken again about the largest exponent.
// FP32 sequences run fft2l as it is.
template <typename T, int N1, int N2, bool INV>
__device__ __forceinline__ void fft2l_rows(cplx<T>* v, int lane, cplx<T>* xs, int s1, int s2, const cplx<T>* stw)
{
    if constexpr (sizeof(T) == 4) fft2l<T, N1, N2, INV, true>(v, lane, xs, s1, s2, stw);
    else fft2l_fixed<N1, N2, INV, true>(v, fx_rows_exponent<N1, N2>(v), 0, lane, (zx*)xs, s1, s2, (const zx*)stw);
}
// (results times 2^sh)
template <typename T, int N1, int N2, bool INV>
__device__ __forceinline__ void fft2l_cols(cplx<T>* v, int seq, int nseq, int lane, cplx<T>* xs, int s1, int s2,
                                           const cplx<T>* stw, int* smx, int sh = 0)
{
    if constexpr (sizeof(T) == 4) {
        fft2l<T, N1, N2, INV>(v, lane, xs, s1, s2, stw);
        if (sh != 0) {
            const T c = __int_as_float((127 + sh) << 23);
            #pragma unroll
            for (int m = 0; m < N1; ++m) v[m] = c * v[m];
        }
    } else {
        const float n = fx_norm<N1>(v, 896);
        auto sum = [&]() {
            float s = 0.f;
            #pragma unroll
            for (int o = 0; o < N2; ++o) s += __int_as_float(smx[o * nseq + seq]);
            return s;
        };
        smx[lane * nseq + seq] = __float_as_int(n);
        const bool far = __syncthreads_or(fx_far<N1>(n, v)) != 0;
        float s = sum();
        int bias = 896;
        if (far) {
            __syncthreads();
            smx[lane * nseq + seq] = fx_max<N1>(v);
            __syncthreads();
            int m = 0;
            for (int o = 0; o < N2; ++o) m = max(m, smx[o * nseq + seq]);
            bias = (m >> 20) - 127;
            __syncthreads();
            smx[lane * nseq + seq] = __float_as_int(fx_norm<N1>(v, bias));
            __syncthreads();
            s = sum();
        }
        const int E = bias == 0x7ff - 127 ? FX_NAN : fx_exponent(s, bias);
        fft2l_fixed<N1, N2, INV, false>(v, E, sh, lane, (zx*)xs, s1, s2, (const zx*)stw);
    }
}
// Forward transform of a + i b (a, b real) and its Hermitian split
// a^(m) = (Z(m) + conj Z(-m)) / (2 N), b^(m) = (Z(m) - conj Z(-m)) / (2 i N),
// N = N1 N2, handed to put(m, a^, b^), m = 0 .. N / 2, by the N2 lanes of the
// sequence; xr: their shared buffer.  FP64: the sums are integers' and 1 / (2 N)
// is in the exponent (in FP64 they took half of the row kernels' FP64 operations:
// products stage of 256 x 256 x 65, 16 snapshots, 23.0 -> 21.0 ms).  PARTS: a and b rounded
// at their own sizes (FxPair).
template <typename T, int N1, int N2, bool PARTS = false, typename F>
__device__ __forceinline__ void fft2l_split(cplx<T>* f, int lane, cplx<T>* xr, const cplx<T>* stw, F put)
{
    constexpr int N = N1 * N2;
    if constexpr (sizeof(T) == 4) {
        fft2l<T, N1, N2, false, true>(f, lane, xr, N2 + 1, 1, stw);
        __syncwarp();
        #pragma unroll
        for (int m = 0; m < N1; ++m) xr[lane + N2 * m] = f[m];
        __syncwarp();
        const T h = (T)0.5 / (T)N;
        for (int k = lane; k <= N / 2; k += N2) {
            const cplx<T> Z = xr[k], Zc = conj(xr[(N - k) & (N - 1)]);
            const cplx<T> D = Z - Zc;
            put(k, h * (Z + Zc), mk(h * D.y, -h * D.x));
        }
    } else {
        auto part = [&](int h) {
            return fx_part_exponent<N1, N2>([&](int j) { return mk(h ? f[j].y : f[j].x, 0.0); });
        };
        const FxPair pr = PARTS ? FxPair(part(0), part(1)) : FxPair(FX_ZERO, FX_ZERO);
        if (PARTS) {
            #pragma unroll
            for (int m = 0; m < N1; ++m) f[m] = mk(pr.in(0, f[m].x), pr.in(1, f[m].y));
        }
        const int E = PARTS ? pr.E : fx_rows_exponent<N1, N2>(f);
        zx* x = (zx*)xr;
        zx w[N1];
        fft2l_raw<N1, N2, false, true>(f, E, lane, x, N2 + 1, 1, (const zx*)stw, [&](int m, zx a, bool) { w[m] = a; });
        __syncwarp();
        #pragma unroll
        for (int m = 0; m < N1; ++m) x[lane + N2 * m] = w[m];
        __syncwarp();
        constexpr int lg = N == 32 ? 5 : N == 64 ? 6 : N == 128 ? 7 : N == 256 ? 8 : 9;
        static_assert(N == 1 << lg, "lengths with a register transform");
        const int e = E - FX_IB + FX_S - lg - 1;
        for (int k = lane; k <= N / 2; k += N2) {
            const zx Z = x[k], Y = x[(N - k) & (N - 1)];
            const long long ax = Z.x + Y.x, ay = Z.y - Y.y, bx = Z.y + Y.y, by = Y.x - Z.x;
            if (PARTS) put(k, mk(pr.out(0, ax, e), pr.out(0, ay, e)), mk(pr.out(1, bx, e), pr.out(1, by, e)));
            else if (fx_safe(E)) put(k, mk(fx_to(ax, e), fx_to(ay, e)), mk(fx_to(bx, e), fx_to(by, e)));
            else put(k, mk(fx_to_edge(ax, e, E), fx_to_edge(ay, e, E)), mk(fx_to_edge(bx, e, E), fx_to_edge(by, e, E)));
        }
    }
}
// ints of the smx array (none for FP32)
template <typename T> __host__ __device__ constexpr int fx_smx(int threads) { return sizeof(T) == 4 ? 1 : threads; }

// stages fft2l's twiddles: FP32 the table itself, FP64 its fixed-point copy,
// which follows the N FP64 entries (fx_table)
template <typename T>
__device__ __forceinline__ void load_twiddles2l(cplx<T>* sh_tw, const cplx<T>* __restrict__ tw, int N)
{
    load_twiddles(sh_tw, tw + (sizeof(T) == 4 ? 0 : N), N);
}

}  // namespace gke
