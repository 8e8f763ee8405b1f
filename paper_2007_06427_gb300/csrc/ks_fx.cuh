// ks_fx.cuh - the double transforms, in 64-bit fixed point on the integer pipes.
//
// Included by ks_items.cuh (which declares cpx, tw_swz, part_sync and the KS_* macros).
//
// On GB300 a double-precision warp instruction holds its sub-partition's FP64 pipe for 64 clocks,
// while a 32 x 32 + 64-bit multiply-add (IMAD.WIDE) takes 2 and a 32-bit addition 1.  A radix-4
// butterfly is 24 FP64 instructions (1536 clocks per warp) or, on 64-bit integers, 36 wide
// multiply-adds and about a hundred short instructions (under 300).  So a double transform
// converts its input once to integers with one common scale, runs its passes on them and
// converts the result back.
//
// The scale.  Every intermediate value of a transform is a sum of a subset of its inputs with
// factors of modulus 1, so nothing in it exceeds S, the sum of the inputs' moduli (taken as
// max + min / 2 of the components, rounded up).  The inputs are scaled by the power of two that
// puts 9/8 S just below 2^63: no pass can overflow and no pass needs a scaling of its own.  The
// quantum, of the input and of the rounding of each twiddle product, is at most 9/4 2^-63 S,
// against rounding relative to each intermediate value in 53-bit arithmetic.  Measured over
// flat, decaying and single-mode random inputs of several amplitudes (9/8 S lies anywhere between
// two powers of two) against long double, the 2-norm error over that of the double radix-4
// transform lies between 0.27 and 0.83: flat inputs of 64 to 256 points 0.30 to 0.48 (the rounding
// of the results to double is most of it), of 512 0.49 to 0.83, of 1024 0.41 to 0.75.
//
// A transform that holds an infinity or a NaN returns NaN in every element (each output depends on
// each input); inputs below 2^-913 count as zero.
#pragma once

#include <vector>

namespace ks {

// A twiddle c + i s, negated: -c = rh 2^-31 + rl 2^-63 to the nearest multiple of 2^-63, -s
// alike (negated because the tables hold 1 and i but not -1 and -i, and -2^31 fits a signed word
// where 2^31 does not).  Sixteen bytes, as a complex double.
struct alignas(16) fxw {
    int rh, rl, ih, il;
};
// A complex value of a transform.
struct alignas(16) fxc {
    long long x, y;
};

// The tables are built on the host, in long double (the words hold ten bits more than a double).
inline void fx_word(long double c, int& h, int& l) {
    const long double H = -c * 2147483648.0L;  // 2^31
    const long double hr = floorl(H + 0.5L);
    const long double lr = floorl((H - hr) * 4294967296.0L + 0.5L);  // within +-2^31: |H - hr| <= 1/2
    h = hr >= 2147483647.0L ? 2147483647 : (int)hr;
    l = lr >= 2147483647.0L ? 2147483647 : (lr <= -2147483647.0L ? -2147483647 : (int)lr);
}
inline fxw fx_words(long double c, long double s) {
    fxw w;
    fx_word(c, w.rh, w.rl);
    fx_word(s, w.ih, w.il);
    return w;
}
// The twiddles in the order the passes read them, w_m^t = exp(2 pi i t / m): for each power of
// four s = 4, 16, 64, 256 the radix-2 pass that ends a transform of length 2 s (w_{2s}^j, j < s),
// then the radix-4 pass of span s (w_{4s}^{q jm}, q = 1, 2, 3, for jm = 0 .. s - 1: three
// neighbours per butterfly, so the lanes of a 128-byte wavefront read stride 48 bytes, free of
// bank conflicts, at one address computation).  A transform of length n reads a prefix.
constexpr int FX_TABLE = 4 * 340;
KS_HDX constexpr int fx_r2_at(int s) { return 4 * ((s - 1) / 3) - 4; }  // 0, 16, 80, 336
KS_HDX constexpr int fx_r4_at(int s) { return fx_r2_at(s) + s; }        // 4, 32, 144, 592
KS_HDX int fx_table_len(int n) {  // entries read by lengths up to n
    int s = 4;
    while (4 * s < n) s *= 4;
    return 2 * s >= n ? fx_r4_at(s) : fx_r4_at(s) + 3 * s;
}
KS_HDX void fx_table_entry(int i, int& t, int& m) {  // entry i is exp(2 pi i t / m)
    int s = 4;
    while (i >= fx_r4_at(s) + 3 * s) s *= 4;
    if (i < fx_r4_at(s)) {
        t = i - fx_r2_at(s);
        m = 2 * s;
    } else {
        const int k = i - fx_r4_at(s);
        t = (k / 3) * (k % 3 + 1);
        m = 4 * s;
    }
}

// The table (host), built once per process: long double functions are software on some machines (1.0 ms for
// the 1360 entries of each handle on Arm), so 129 angles of the first octant serve all of them.
inline const std::vector<fxw>& fx_table() {
    static const std::vector<fxw> table = [] {
        constexpr int N = 1024, Q = N / 4;
        std::vector<long double> c(Q + 1), s(Q + 1);
        for (int t = 0; t <= Q / 2; ++t) {
            const long double a = 6.283185307179586476925286766559006L * t / N;
            c[t] = s[Q - t] = t ? cosl(a) : 1;
            s[t] = c[Q - t] = t ? sinl(a) : 0;
        }
        std::vector<fxw> w(FX_TABLE);
        for (int i = 0; i < FX_TABLE; ++i) {
            int t, m;
            fx_table_entry(i, t, m);
            t *= N / m;
            const long double x = c[t % Q], y = s[t % Q];
            switch (t / Q) {
            case 0: w[i] = fx_words(x, y); break;
            case 1: w[i] = fx_words(-y, x); break;
            case 2: w[i] = fx_words(-x, -y); break;
            default: w[i] = fx_words(y, -x); break;
            }
        }
        return w;
    }();
    return table;
}

// Entry i of the table at tw (the host build of the items has its own).
KS_HD fxw fx_tw(const cpx<double>* tw, int i) {
#ifdef KS_HOST_EMULATION
    return fx_table()[i];
#else
    return reinterpret_cast<const fxw*>(tw)[i];
#endif
}

// Products of 32-bit words.  As an instruction with a 64-bit result, of which the high half is
// used at times: left to the compiler those become the high-product instruction, which takes
// twice as long.
KS_HD long long fx_wide(int a, int b) {
#ifdef KS_HOST_EMULATION
    return (long long)a * b;
#else
    long long r;
    asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
#endif
}
KS_HD int fx_top(long long v) { return (int)((unsigned long long)v >> 32); }

// v times the twiddle of w: each component of v splits as h 2^32 + l with l signed, and with
// words wh, wl
//   v w = 2 (h wh + (l wh + h wl) 2^-32) + l wl 2^-63,
// of which the last product (below a half) is left out.  The pairs of middle products of a
// component stay below sqrt(2) 2^62 for a twiddle of modulus 1 and |v| < 2^63.  FINE = false: the
// middle products enter by their high words, an error of 1.2 units rms; twelve products and 32-bit
// sums, 58 clocks a warp (124 with the middle products in one 64-bit sum).  FINE = true: their sums
// are rounded to the unit, at 1024 points, where the coarse products would take the error of flat
// inputs above that of the double transform (up to 1.6 times; 0.41 to 0.75 so).
template <bool FINE>
KS_HD fxc fx_mul(fxc v, fxw w) {
    const int al = (int)v.x, ah = fx_top(v.x) + (int)((unsigned)al >> 31);
    const int bl = (int)v.y, bh = fx_top(v.y) + (int)((unsigned)bl >> 31);
    if constexpr (FINE) {
        const long long r1 = fx_wide(al, w.rh) - fx_wide(bl, w.ih), r2 = fx_wide(ah, w.rl) - fx_wide(bh, w.il);
        const long long i1 = fx_wide(al, w.ih) + fx_wide(bl, w.rh), i2 = fx_wide(ah, w.il) + fx_wide(bh, w.rl);
        // the low words of the sums as 30 bits each, so that they and the half fit 32; bit 29 is the unit
        const unsigned fr = ((unsigned)r1 >> 2) + ((unsigned)r2 >> 2) + (1u << 28);
        const unsigned fi = ((unsigned)i1 >> 2) + ((unsigned)i2 >> 2) + (1u << 28);
        const long long x = fx_wide(ah, w.rh) - fx_wide(bh, w.ih) + fx_top(r1) + fx_top(r2);
        const long long y = fx_wide(ah, w.ih) + fx_wide(bh, w.rh) + fx_top(i1) + fx_top(i2);
        return fxc{-(x + x + (fr >> 29)), -(y + y + (fi >> 29))};
    }
    const int r1 = fx_top(fx_wide(al, w.rh)) - fx_top(fx_wide(bl, w.ih));
    const int r2 = fx_top(fx_wide(ah, w.rl)) - fx_top(fx_wide(bh, w.il));
    const int i1 = fx_top(fx_wide(al, w.ih)) + fx_top(fx_wide(bl, w.rh)) + 2;  // four floors
    const int i2 = fx_top(fx_wide(ah, w.il)) + fx_top(fx_wide(bh, w.rl));
    const long long x = fx_wide(bh, w.ih) - fx_wide(ah, w.rh) - r1 - r2;
    const long long y = -fx_wide(ah, w.ih) - fx_wide(bh, w.rh) - i1 - i2;
    return fxc{x + x, y + y};
}
KS_HD fxc operator+(fxc a, fxc b) { return fxc{a.x + b.x, a.y + b.y}; }
KS_HD fxc operator-(fxc a, fxc b) { return fxc{a.x - b.x, a.y - b.y}; }

// ---- conversion ------------------------------------------------------------------------------
KS_HD unsigned fx_hi(double v) {
#ifdef KS_HOST_EMULATION
    unsigned long long b;
    __builtin_memcpy(&b, &v, 8);
    return (unsigned)(b >> 32);
#else
    return (unsigned)__double2hiint(v);
#endif
}
KS_HD unsigned fx_lo(double v) {
#ifdef KS_HOST_EMULATION
    unsigned long long b;
    __builtin_memcpy(&b, &v, 8);
    return (unsigned)b;
#else
    return (unsigned)__double2loint(v);
#endif
}
KS_HD unsigned long long fx_shr(unsigned long long v, unsigned r) {  // 0 for r >= 64
#ifdef KS_HOST_EMULATION
    return r < 64 ? v >> r : 0;
#else
    unsigned long long o;
    asm("shr.u64 %0, %1, %2;" : "=l"(o) : "l"(v), "r"(r));  // the shift saturates
    return o;
#endif
}
// The scale of a transform as the reference exponent E: a double of biased exponent e enters as
// its 64-bit left-aligned significand shifted right by E - e.  FX_ZERO: every input shifts out.
// FX_NAN: an input is not finite (or the sum may overflow).
constexpr int FX_ZERO = 5000, FX_NAN = 1 << 30;

// flip: 0, or 0x80000000 to negate.
KS_HD long long fx_in(double v, int E, unsigned flip) {
    const unsigned hi = fx_hi(v), lo = fx_lo(v);
    const unsigned e = (hi + hi) >> 21;
    const unsigned long long m =
        ((unsigned long long)(0x80000000u | (hi << 11) | (lo >> 21)) << 32) | (unsigned)(lo << 11);
    const unsigned long long a = fx_shr(m, (unsigned)E - e);  // E - e >= 1
    return (int)(hi ^ flip) < 0 ? -(long long)a : (long long)a;
}
// The double of v at scale E: the conversion instruction, then the scale added to the exponent
// field.  It takes 64 clocks a warp on the FP64 pipe, which the passes leave idle, and one issue
// slot; the normalisation below takes about 55 on the integer pipes.  A result takes one of each:
// the last pass of 64 points, eight values a lane, took 433 clocks a warp with eight instructions
// (two warps a sub-partition), 389 with eight normalisations and 373 with four of each.
// del is fx_del(E), plus 2^31 to negate.
KS_HD unsigned fx_del(int E) { return (unsigned)(E - 1086) << 20; }
KS_HD double fx_out(long long v, unsigned del) {
    const double d = (double)v;
    const unsigned hi = v != 0 ? fx_hi(d) + del : 0;
#ifdef KS_HOST_EMULATION
    const unsigned long long b = ((unsigned long long)hi << 32) | fx_lo(d);
    double r;
    __builtin_memcpy(&r, &b, 8);
    return r;
#else
    return __hiloint2double((int)hi, (int)fx_lo(d));
#endif
}

// |v| as a float: sign dropped, exponent rebiased, mantissa cut to 20 bits; 0 below 2^-127, an
// infinity from 2^128 on.  (Integer steps: the conversion instruction runs on the FP64 pipe.)
KS_HD float fx_abs(double v) {
    int t = (int)(fx_hi(v) & 0x7fffffffu) - (896 << 20);
    t = t > 0 ? t : 0;
    t = t < 0x0ff00000 ? t : 0x0ff00000;
    const unsigned b = (unsigned)t << 3;
#ifdef KS_HOST_EMULATION
    float r;
    __builtin_memcpy(&r, &b, 4);
    return r;
#else
    return __uint_as_float(b);
#endif
}
KS_HD float fx_abs(cpx<double> v) {  // |v| <= max + min / 2
    const float a = fx_abs(v.x), b = fx_abs(v.y);
    return fmaf(0.5f, a < b ? a : b, a < b ? b : a);
}
// The scale from the sum S of the moduli: 9/8 S < 2^(E - 1023).
KS_HD bool fx_sum_ok(float S) { return S >= 7.9e-31f && S <= 1.2e30f; }  // 2^-100 .. 2^100
KS_HD int fx_ref(float S) {
    const float g = S * 1.125f;
#ifdef KS_HOST_EMULATION
    unsigned b;
    __builtin_memcpy(&b, &g, 4);
#else
    const unsigned b = __float_as_uint(g);
#endif
    return (int)(b >> 23) + 897;
}

// Outside that range: the largest exponent first, then the sum relative to it, in units of 2^-19
// of it and rounded up.
KS_HD unsigned fx_maxhi(cpx<double> v) {
    const unsigned a = fx_hi(v.x) & 0x7fffffffu, b = fx_hi(v.y) & 0x7fffffffu;
    return a > b ? a : b;
}
KS_HD unsigned fx_mag(double v, unsigned e0) {
    const unsigned hi = fx_hi(v) & 0x7fffffffu, d = e0 - (hi >> 20);
    return (d > 30 ? 0u : ((hi & 0xfffffu) | 0x100000u) >> (1 + d)) + 1u;
}
KS_HD unsigned fx_mag(cpx<double> v, unsigned e0) { return fx_mag(v.x, e0) + fx_mag(v.y, e0); }
KS_HD int fx_ref(unsigned maxhi, unsigned sum) {
    const int e0 = (int)(maxhi >> 20);
    sum += sum >> 3;
    int bits = 0;
    while (bits < 32 && (sum >> bits)) ++bits;
    const int E = bits - 19 + e0;
    if (e0 == 0x7ff || E > 2046) return FX_NAN;
    return e0 < 110 ? FX_ZERO : E;  // the smallest result keeps a positive exponent, scaled down too
}

#ifndef KS_HOST_EMULATION
// Sum / maximum over the g lanes (a power of two, aligned) that share a transform; every lane of
// the warp calls.  An xor tree: all lanes of a group get the same bits.
template <typename T, typename Op>
__device__ __forceinline__ T fx_reduce(T v, int g, Op op) {
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
        if (o < g) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}
// Scale of the transform whose inputs the g lanes hold, N = 2 or 4 each (called by whole warps).
// The order of the float sum, ((0, 1), (2, 3)) and then the xor tree, is the same for two lanes of
// two inputs, for a lane of four and in fx_scales.
template <int N>
__device__ __forceinline__ int fx_group_scale(const cpx<double> (&v)[N], int g) {
    float S = fx_abs(v[0]) + fx_abs(v[1]);
    if constexpr (N == 4) S += fx_abs(v[2]) + fx_abs(v[3]);
    S = fx_reduce(S, g, [](float a, float b) { return a + b; });
    int E = fx_ref(S);
    if (__any_sync(0xffffffffu, !fx_sum_ok(S))) {
        unsigned mx = 0, sum = 0;
        for (int q = 0; q < N; ++q) mx = max(mx, fx_maxhi(v[q]));
        mx = fx_reduce(mx, g, [](unsigned a, unsigned b) { return max(a, b); });
        for (int q = 0; q < N; ++q) sum += fx_mag(v[q], mx >> 20);
        sum = fx_reduce(sum, g, [](unsigned a, unsigned b) { return a + b; });
        if (!fx_sum_ok(S)) E = fx_ref(mx, sum);
    }
    return E;
}
#endif

// Scales of the cnt transforms at a: one warp per transform (NT threads).
KS_HD void fx_scales(const cpx<double>* a, int lg, int cnt, int* sc, int NT) {
    const int n = 1 << lg;
#ifdef KS_HOST_EMULATION
    (void)NT;
    for (int f = 0; f < cnt; ++f) {
        const cpx<double>* s = a + (size_t)f * n;
        float S = 0.f;
        for (int i = 0; i < n; ++i) S += fx_abs(s[i]);
        unsigned mx = 0, sum = 0;
        for (int i = 0; i < n; ++i) mx = fx_maxhi(s[i]) > mx ? fx_maxhi(s[i]) : mx;
        for (int i = 0; i < n; ++i) sum += fx_mag(s[i], mx >> 20);
        sc[f] = fx_sum_ok(S) ? fx_ref(S) : fx_ref(mx, sum);
    }
#else
    for (int f = threadIdx.x >> 5; f < cnt; f += NT >> 5) {
        const cpx<double>* s = a + ((unsigned)f << lg) + (threadIdx.x & 31);
        float S = 0.f;
        for (int i = 0; i < n; i += 128)
            S += (fx_abs(s[i]) + fx_abs(s[i + 32])) + (fx_abs(s[i + 64]) + fx_abs(s[i + 96]));
        S = fx_reduce(S, 32, [](float x, float y) { return x + y; });
        int E = fx_ref(S);
        if (!fx_sum_ok(S)) {
            unsigned mx = 0, sum = 0;
            for (int i = 0; i < n; i += 32) mx = max(mx, fx_maxhi(s[i]));
            mx = __reduce_max_sync(0xffffffffu, mx);
            for (int i = 0; i < n; i += 32) sum += fx_mag(s[i], mx >> 20);
            E = fx_ref(mx, __reduce_add_sync(0xffffffffu, sum));
        }
        if ((threadIdx.x & 31) == 0) sc[f] = E;
    }
#endif
}

// The same on the integer pipes.
KS_HD double fx_out_int(long long v, unsigned del) {
    const long long s = v >> 63;
    const unsigned long long m = (unsigned long long)((v ^ s) - s);
#ifdef KS_HOST_EMULATION
    const int lz = m ? __builtin_clzll(m) : 64;
#else
    const int lz = __clzll((long long)m);
#endif
    const unsigned long long M = m << (lz & 63) >> 1;  // |v| < 2^63: exact, leading bit at 62
    // to nearest, ties to even, as the instruction: leading bit at 52, or 53 after rounding
    const unsigned long long q = (M + 0x1ff + ((M >> 10) & 1)) >> 10;
    const unsigned hi = (unsigned)(q >> 32) + ((unsigned)(1085 - lz) << 20) + (((unsigned)(s >> 32)) & 0x80000000u) + del;
    const unsigned h = m != 0 ? hi : 0;
#ifdef KS_HOST_EMULATION
    const unsigned long long b = ((unsigned long long)h << 32) | (unsigned)q;
    double r;
    __builtin_memcpy(&r, &b, 8);
    return r;
#else
    return __hiloint2double((int)h, (int)(unsigned)q);
#endif
}

// The scale of results that come out multiplied by 2^-down.
KS_HD int fx_down(int E, int down) { return E >= FX_ZERO ? E : E - down; }

// One result at scale E; flip: 2^31 for the conjugate.
KS_HD cpx<double> fx_result(fxc v, int E, unsigned flip) {
    if (E >= FX_ZERO) {  // nothing of the input got in: zeros, or NaN
        const double z = E == FX_ZERO ? 0.0 : NAN;
        return mk<double>(z, z);
    }
    const unsigned del = fx_del(E);
    return mk<double>(fx_out(v.x, del), fx_out_int(v.y, del + flip));
}

// Where element i of a pass's output sits in its transform's buffer.  The first pass writes four
// neighbours 4j .. 4j + 3 per butterfly and the second two runs of four per eight lanes: in natural
// order four or two lanes of a 128-byte wavefront share their banks, so those outputs are
// permuted within aligned groups of four (pass 1) or eight (pass 2) and the next pass reads them
// through the same map.  Later passes write runs of sixteen, in natural order, as does the last.
template <int LAY>
KS_HD int fx_pos(int i) {
    return LAY == 1 ? i ^ ((i >> 3) & 3) : LAY == 2 ? i ^ (((i >> 4) & 1) << 2) : i;
}

// The radix-4 pass of one span (4 .. 256) on the transforms at a.  LAST: the result is converted
// to double.
template <int SPAN, bool LAST, bool FINE = false>
KS_HD void fx_pass4(const fxc* a, fxc* b, int lg, int total, unsigned flip, const cpx<double>* tw,
                    const int* sc, int NT, int down) {
    constexpr int LI = SPAN == 4 ? 1 : SPAN == 16 ? 2 : 0, LO = (LAST || SPAN != 4) ? 0 : 2;
    const int nb = 1 << (lg - 2);
    for (int i = KS_TID; i < total; i += NT) {
        const int f = i >> (lg - 2), j = i & (nb - 1);
        const fxc* s = a + ((unsigned)f << lg);
        fxc* d = b + ((unsigned)f << lg);
        const int jm = j & (SPAN - 1), od = ((j - jm) << 2) + jm, t = fx_r4_at(SPAN) + 3 * jm;
        const fxc v0 = s[fx_pos<LI>(j)];
        const fxc a1 = fx_mul<FINE>(s[fx_pos<LI>(j + nb)], fx_tw(tw, t));
        const fxc a2 = fx_mul<FINE>(s[fx_pos<LI>(j + 2 * nb)], fx_tw(tw, t + 1));
        const fxc a3 = fx_mul<FINE>(s[fx_pos<LI>(j + 3 * nb)], fx_tw(tw, t + 2));
        const fxc t0 = v0 + a2, t1 = v0 - a2, t2 = a1 + a3, t3 = a1 - a3;
        const fxc o0 = t0 + t2, o2 = t0 - t2;
        const fxc o1{t1.x - t3.y, t1.y + t3.x}, o3{t1.x + t3.y, t1.y - t3.x};
        if constexpr (LAST) {
            cpx<double>* e = reinterpret_cast<cpx<double>*>(d) + od;
            const int E = fx_down(sc[f], down);
            e[0] = fx_result(o0, E, flip);
            e[SPAN] = fx_result(o1, E, flip);
            e[2 * SPAN] = fx_result(o2, E, flip);
            e[3 * SPAN] = fx_result(o3, E, flip);
        } else {
            d[fx_pos<LO>(od)] = o0;
            d[fx_pos<LO>(od + SPAN)] = o1;
            d[fx_pos<LO>(od + 2 * SPAN)] = o2;
            d[fx_pos<LO>(od + 3 * SPAN)] = o3;
        }
    }
}

// The radix-2 pass that ends a transform of length 2 SPAN (SPAN = 4, 16, 64 or 256).
template <int SPAN>
KS_HD void fx_pass2(const fxc* a, fxc* b, int cnt, unsigned flip, const cpx<double>* tw,
                    const int* sc, int NT, int down) {
    constexpr int LI = SPAN == 4 ? 1 : SPAN == 16 ? 2 : 0, n = 2 * SPAN;
    for (int i = KS_TID; i < cnt * SPAN; i += NT) {
        const int f = i / SPAN, j = i & (SPAN - 1);
        const fxc* s = a + f * n;
        const int E = fx_down(sc[f], down);
        const fxc v0 = s[fx_pos<LI>(j)];
        const fxc v1 = fx_mul<false>(s[fx_pos<LI>(j + SPAN)], fx_tw(tw, fx_r2_at(SPAN) + j));
        const fxc x = v0 + v1, y = v0 - v1;
        cpx<double>* d = reinterpret_cast<cpx<double>*>(b + f * n) + j;
        d[0] = fx_result(x, E, flip);
        d[SPAN] = fx_result(y, E, flip);
    }
}

#ifndef KS_HOST_EMULATION
// ---- two threads per butterfly ------------------------------------------------------------------
// Where a call has fewer butterflies than half its threads (single loops, whose blocks hold one or
// two columns or row pairs), two neighbouring lanes share a butterfly: lane c = 0 computes the real
// parts, c = 1 the imaginary ones, from the same inputs.  The integers are the same, in half the
// instructions a lane: two 64-point transforms take 2640 clocks a block, 3070 with one thread a butterfly
// (32 points: 1970 against 2310).

// component c of fx_mul<false>: a, b the value's components, w the halves (hi, lo) of the twiddle
// that multiply them (c = 0: re, im; c = 1: im, re)
__device__ __forceinline__ long long fx_mul_part(long long a, long long b, int2 wa, int2 wb, int c) {
    const int al = (int)a, ah = fx_top(a) + (int)((unsigned)al >> 31);
    const int bl = (int)b, bh = fx_top(b) + (int)((unsigned)bl >> 31);
    const int a1 = fx_top(fx_wide(al, wa.x)), a2 = fx_top(fx_wide(ah, wa.y));
    const int b1 = fx_top(fx_wide(bl, wb.x)) + 2 * c, b2 = fx_top(fx_wide(bh, wb.y));
    const long long A = fx_wide(ah, wa.x) + a1 + a2, B = fx_wide(bh, wb.x) + b1 + b2;
    const long long x = (c ? -B : B) - A;
    return x + x;
}
__device__ __forceinline__ long long fx_shfl1(long long v) {
    const int lo = __shfl_xor_sync(0xffffffffu, (int)v, 1), hi = __shfl_xor_sync(0xffffffffu, fx_top(v), 1);
    return (long long)(((unsigned long long)(unsigned)hi << 32) | (unsigned)lo);
}
__device__ __forceinline__ double fx_result_part(long long v, int E, unsigned flip) {
    if (E >= FX_ZERO) return E == FX_ZERO ? 0.0 : NAN;
    return fx_out(v, fx_del(E) + flip);
}

template <int SPAN, bool LAST>
__device__ __forceinline__ void fx_split4(const fxc* a, fxc* b, int lg, int total, unsigned flip,
                                          const cpx<double>* tw, const int* sc, int NT, int down) {
    constexpr int LI = SPAN == 4 ? 1 : SPAN == 16 ? 2 : 0, LO = (LAST || SPAN != 4) ? 0 : 2;
    const int nb = 1 << (lg - 2), c = threadIdx.x & 1;
    for (int i0 = threadIdx.x; (i0 & ~31) < 2 * total; i0 += NT) {  // by whole warps
        const int i = min(i0 >> 1, total - 1);
        const int f = i >> (lg - 2), j = i & (nb - 1);
        const fxc* s = a + ((unsigned)f << lg);
        const int jm = j & (SPAN - 1), od = ((j - jm) << 2) + jm;
        const int2* w = reinterpret_cast<const int2*>(tw) + 2 * (fx_r4_at(SPAN) + 3 * jm);
        const long long v0 = reinterpret_cast<const long long*>(s + fx_pos<LI>(j))[c];
        const fxc v1 = s[fx_pos<LI>(j + nb)], v2 = s[fx_pos<LI>(j + 2 * nb)], v3 = s[fx_pos<LI>(j + 3 * nb)];
        const long long a1 = fx_mul_part(v1.x, v1.y, w[c], w[c ^ 1], c);
        const long long a2 = fx_mul_part(v2.x, v2.y, w[2 + c], w[2 + (c ^ 1)], c);
        const long long a3 = fx_mul_part(v3.x, v3.y, w[4 + c], w[4 + (c ^ 1)], c);
        const long long t0 = v0 + a2, t1 = v0 - a2, t2 = a1 + a3;
        const long long u3 = fx_shfl1(a1 - a3), t3 = c ? u3 : -u3;  // i t3
        const long long o[4] = {t0 + t2, t1 + t3, t0 - t2, t1 - t3};
        if (i0 >= 2 * total) continue;
        if constexpr (LAST) {
            double* e = reinterpret_cast<double*>(b + ((unsigned)f << lg) + od) + c;
            const int E = fx_down(sc[f], down);
            const unsigned fl = c ? flip : 0u;
#pragma unroll
            for (int q = 0; q < 4; ++q) e[2 * q * SPAN] = fx_result_part(o[q], E, fl);
        } else {
            long long* d = reinterpret_cast<long long*>(b + ((unsigned)f << lg)) + c;
#pragma unroll
            for (int q = 0; q < 4; ++q) d[2 * fx_pos<LO>(od + q * SPAN)] = o[q];
        }
    }
}

template <int SPAN>
__device__ __forceinline__ void fx_split2(const fxc* a, fxc* b, int cnt, unsigned flip, const cpx<double>* tw,
                                          const int* sc, int NT, int down) {
    constexpr int LI = SPAN == 4 ? 1 : SPAN == 16 ? 2 : 0, n = 2 * SPAN;
    const int c = threadIdx.x & 1;
    for (int i = threadIdx.x; i < cnt * 2 * SPAN; i += NT) {
        const int f = i / (2 * SPAN), j = (i >> 1) & (SPAN - 1);
        const fxc* s = a + f * n;
        const int2* w = reinterpret_cast<const int2*>(tw) + 2 * (fx_r2_at(SPAN) + j);
        const long long v0 = reinterpret_cast<const long long*>(s + fx_pos<LI>(j))[c];
        const fxc v1 = s[fx_pos<LI>(j + SPAN)];
        const long long p = fx_mul_part(v1.x, v1.y, w[c], w[c ^ 1], c);
        double* d = reinterpret_cast<double*>(b + f * n + j) + c;
        const int E = fx_down(sc[f], down);
        const unsigned fl = c ? flip : 0u;
        d[0] = fx_result_part(v0 + p, E, fl);
        d[2 * SPAN] = fx_result_part(v0 - p, E, fl);
    }
}

// The first pass (n <= 64: 2 n / 4 lanes hold a transform).
__device__ __forceinline__ void fx_split_first(const cpx<double>* a, fxc* b, int lg, int total, unsigned flip,
                                               int* sc, int NT) {
    const int nb = 1 << (lg - 2), c = threadIdx.x & 1;
    for (int i0 = threadIdx.x; (i0 & ~31) < 2 * total; i0 += NT) {
        const int i = min(i0 >> 1, total - 1);
        const int f = i >> (lg - 2), j = i & (nb - 1);
        const cpx<double>* s = a + ((unsigned)f << lg) + j;
        const cpx<double> m[2] = {s[2 * c * nb], s[(2 * c + 1) * nb]};
        const int E = fx_group_scale(m, 2 * nb);
        long long x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
            x[q] = fx_in(reinterpret_cast<const double*>(s + q * nb)[c], E, c ? flip : 0u);
        const long long t0 = x[0] + x[2], t1 = x[0] - x[2], t2 = x[1] + x[3];
        const long long u3 = fx_shfl1(x[1] - x[3]), t3 = c ? u3 : -u3;
        if (i0 >= 2 * total) continue;
        if (j == 0 && c == 0) sc[f] = E;
        const int o = fx_pos<1>(j << 2);
        long long* d = reinterpret_cast<long long*>(b + ((unsigned)f << lg)) + c;
        d[2 * o] = t0 + t2;
        d[2 * (o ^ 1)] = t1 + t3;
        d[2 * (o ^ 2)] = t0 - t2;
        d[2 * (o ^ 3)] = t1 - t3;
    }
}
#endif

// cnt transforms of length n = 2^lg (n >= 8), stored contiguously in a, b scratch of the same
// size: the conventions of fft_batch.  Radix-4 passes, a radix-2 pass last when lg is odd; the
// first pass converts its input to integers, the last one converts back.  The passes have the
// sign +1; for -1 the input and the output are conjugated.  sc: cnt ints of shared memory for the
// scales.  Lengths up to 128 form the scale in the first pass, among the n / 4 lanes that hold
// the transform; longer ones in a pass of their own before it (a transform per warp).  The
// arithmetic does not depend on the thread count.  True when the result is in b.
// down: the results come out multiplied by 2^-down (a normalisation that costs nothing here).
// SPLIT: lengths up to 64 take two threads a butterfly when there are threads for it (128 points: 3490
// clocks for two transforms against 3370 with one thread, 256: 4630 against 4360, so not there).
template <bool SPLIT>
KS_HD bool fx_run(cpx<double>* a, cpx<double>* b, int lg, int cnt, int dir,
                  const cpx<double>* tw, int* sc, int nthr, int down) {
#ifdef KS_HOST_EMULATION
    const int NT = KS_NT;
    const bool pre = true;
#else
    const int NT = nthr > 0 ? nthr : KS_NT;
    const bool pre = lg > 7;
#endif
    const int n = 1 << lg, nb = n >> 2, total = cnt << (lg - 2);
    const unsigned flip = dir < 0 ? 0x80000000u : 0u;
    auto sync = [&]() {
        if (nthr > 0) part_sync(nthr);
        else KS_SYNC();
    };
    if (pre) {
        fx_scales(a, lg, cnt, sc, NT);
        sync();
    }
    fxc* fa = reinterpret_cast<fxc*>(a);
    fxc* fb = reinterpret_cast<fxc*>(b);
#ifndef KS_HOST_EMULATION
    const bool split = SPLIT && 2 * total <= NT && lg <= 6;
    if (split) {
        fx_split_first(a, fb, lg, total, flip, sc, NT);
    } else
#endif
    // span 1: no twiddles.  By whole warps: lanes past the end hold the last butterfly and store
    // nothing (the lanes of a transform are all in or all out).
    for (int i0 = KS_TID; (i0 & ~31) < total; i0 += NT) {
        const int i = i0 < total ? i0 : total - 1;
        const int f = i >> (lg - 2), j = i & (nb - 1);
        const cpx<double>* s = a + ((unsigned)f << lg);
        fxc* d = fb + ((unsigned)f << lg);
        const cpx<double> v[4] = {s[j], s[j + nb], s[j + 2 * nb], s[j + 3 * nb]};
        int E;
#ifndef KS_HOST_EMULATION
        if (!pre) {
            E = fx_group_scale(v, nb);
            if (j == 0) sc[f] = E;
        } else
#endif
            E = sc[f];
        if (i0 >= total) continue;
        fxc x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = fxc{fx_in(v[q].x, E, 0), fx_in(v[q].y, E, flip)};
        const fxc t0 = x[0] + x[2], t1 = x[0] - x[2], t2 = x[1] + x[3], t3 = x[1] - x[3];
        const int o = fx_pos<1>(j << 2);
        d[o] = t0 + t2;
        d[o ^ 1] = fxc{t1.x - t3.y, t1.y + t3.x};
        d[o ^ 2] = t0 - t2;
        d[o ^ 3] = fxc{t1.x + t3.y, t1.y - t3.x};
    }
    sync();
    // the data is in b now; the passes alternate
#ifndef KS_HOST_EMULATION
    if constexpr (SPLIT) {
        if (split) {
            if (lg == 3) {
                fx_split2<4>(fb, fa, cnt, flip, tw, sc, NT, down);
                sync();
                return false;
            }
            if (lg == 4) {
                fx_split4<4, true>(fb, fa, lg, total, flip, tw, sc, NT, down);
                sync();
                return false;
            }
            fx_split4<4, false>(fb, fa, lg, total, flip, tw, sc, NT, down);
            sync();
            if (lg == 5) fx_split2<16>(fa, fb, cnt, flip, tw, sc, NT, down);
            else fx_split4<16, true>(fa, fb, lg, total, flip, tw, sc, NT, down);
            sync();
            return true;
        }
    }
#endif
    switch (lg) {
    case 10:
        fx_pass4<4, false, true>(fb, fa, lg, total, flip, tw, sc, NT, down);
        sync();
        fx_pass4<16, false, true>(fa, fb, lg, total, flip, tw, sc, NT, down);
        sync();
        fx_pass4<64, false, true>(fb, fa, lg, total, flip, tw, sc, NT, down);
        sync();
        fx_pass4<256, true, true>(fa, fb, lg, total, flip, tw, sc, NT, down);
        sync();
        return true;
    case 3:
        fx_pass2<4>(fb, fa, cnt, flip, tw, sc, NT, down);
        sync();
        return false;
    case 4:
        fx_pass4<4, true>(fb, fa, lg, total, flip, tw, sc, NT, down);
        sync();
        return false;
    }
    fx_pass4<4, false>(fb, fa, lg, total, flip, tw, sc, NT, down);
    sync();
    switch (lg) {
    case 5:
        fx_pass2<16>(fa, fb, cnt, flip, tw, sc, NT, down);
        sync();
        return true;
    case 6:
        fx_pass4<16, true>(fa, fb, lg, total, flip, tw, sc, NT, down);
        sync();
        return true;
    }
    fx_pass4<16, false>(fa, fb, lg, total, flip, tw, sc, NT, down);
    sync();
    switch (lg) {
    case 7:
        fx_pass2<64>(fb, fa, cnt, flip, tw, sc, NT, down);
        sync();
        return false;
    case 8:
        fx_pass4<64, true>(fb, fa, lg, total, flip, tw, sc, NT, down);
        sync();
        return false;
    }
    fx_pass4<64, false>(fb, fa, lg, total, flip, tw, sc, NT, down);
    sync();
    fx_pass2<256>(fa, fb, cnt, flip, tw, sc, NT, down);
    sync();
    return true;
}

#ifndef KS_HOST_EMULATION
// One copy of the code, called by every transform of the cluster kernel: the eight transforms of a
// step then share their instructions.  The buffers are passed as offsets into the block's dynamic shared memory, so the
// accesses stay in the shared space.
static __device__ __noinline__ bool fx_call(int ao, int bo, int lg, int cnt, int dir, int two, int sco,
                                          int nthr, int down) {
    extern __shared__ __align__(16) unsigned char smem[];
    return fx_run<true>(reinterpret_cast<cpx<double>*>(smem + ao), reinterpret_cast<cpx<double>*>(smem + bo),
                  lg, cnt, dir, reinterpret_cast<const cpx<double>*>(smem + two),
                  reinterpret_cast<int*>(smem + sco), nthr, down);
}
__device__ __forceinline__ int fx_off(const void* p) {
    extern __shared__ __align__(16) unsigned char smem[];
    return (int)((unsigned)__cvta_generic_to_shared(p) - (unsigned)__cvta_generic_to_shared(smem));
}
#endif

// the transform under the conventions of fft_batch; on the device every buffer, the table (its
// prefix, see FX_TABLE) included, is in shared memory.  fft_fx_call: through the shared copy.
KS_HD cpx<double>* fft_fx(cpx<double>* a, cpx<double>* b, int lg, int cnt, int dir,
                          const cpx<double>* tw, int* sc, int nthr = 0, int down = 0) {
    return fx_run<false>(a, b, lg, cnt, dir, tw, sc, nthr, down) ? b : a;
}
#ifndef KS_HOST_EMULATION
__device__ __forceinline__ cpx<double>* fft_fx_call(cpx<double>* a, cpx<double>* b, int lg, int cnt,
                                                    int dir, const cpx<double>* tw, int* sc, int nthr = 0,
                                                    int down = 0) {
    return fx_call(fx_off(a), fx_off(b), lg, cnt, dir, fx_off(tw), fx_off(sc), nthr, down) ? b : a;
}
#endif

}  // namespace ks
