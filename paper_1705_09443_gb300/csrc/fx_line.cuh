// Line FFTs of the LS operator in 64-bit fixed point.
//
// This GPU issues 2 FP64 multiply-adds per clock and SM but 14 to 22 32 x 32 ->
// 64-bit integer ones and 122 32-bit additions (probe, 32 warps per SM): an FFT in
// 64-bit integers takes a fraction of the FP64 pipe's time, which bounded the
// operator (n = 512, 64 right-hand sides: 13.4 -> 3.24 ms; 3D n = 64: 365 ->
// 136 us).  A line is held as integers with one exponent, v * 2^E, scaled so
// that its largest entry uses the bits that a pass's growth leaves free:
//  - additions are exact,
//  - the product with a twiddle factor (2^62 exp(-2 pi i k / L)) keeps the high
//    64 bits, rounded, so every factor between two passes also scales by 1/4,
//  - between two passes the line is shifted so that its largest entry has
//    60 or 61 - lg(radix) bits (the largest entry is an OR over the line,
//    formed on the way through shared memory), whatever the line grew by,
//  - every rounding is to nearest, ties to even.  An entry is an integer, so
//    ties are common (a quarter of the entries where a factor is 1); rounded
//    up, or the fraction of a product dropped, the mean error of an entry is
//    not zero and adds up at index 0 of the inverse transform (n = 200, noise:
//    first row 1.3e-15 of the field against 1.5e-16 in the others; now 1.0e-16
//    in all).  It costs 8 to 10 % of the operator (n = 512: 2.98 -> 3.24 ms).
// The error of the convolution relative to the 2-norm of its result is, on wave
// fields against 80-bit arithmetic, 1.5e-16 (L = 512), 1.8e-16 (1024) and
// 1.9e-16 (2048); that of FP64 transforms 2.3e-16, 3.1e-16 and 2.8e-16.  An
// entry's own error is a fraction of its line's largest entry, where FP64's is
// one of the entry: it was compared row by row and for fields whose transform
// is concentrated (constant, alternating in sign, rows from 1 to 1e-12), and
// is below FP64's in all of them (tests/fixed_fft_host.cu).
// Non-finite input marks its line (exponent kFxBad) and through it every
// line that reads it, so the result is NaN as in floating point.
#pragma once
#include <cmath>
#include <type_traits>

#include "lss_common.cuh"

constexpr int kFxBad = 1 << 24;    // line exponent of a line with non-finite entries
constexpr int kFxMinLg = 6, kFxMaxLg = 11;   // line lengths 64 .. 2048
constexpr int kFxBase = 8;        // the plan whose storage order the kernel transform is kept in

struct fx2 { long long x, y; };

#define FX_HD __host__ __device__ __forceinline__

FX_HD fx2 operator+(fx2 a, fx2 b) { return {a.x + b.x, a.y + b.y}; }
FX_HD fx2 operator-(fx2 a, fx2 b) { return {a.x - b.x, a.y - b.y}; }
FX_HD fx2 fx_mul_mi(fx2 a) { return {a.y, -a.x}; }   // -i a
FX_HD fx2 fx_swap(fx2 a) { return {a.y, a.x}; }

// v = hi 2^32 + lo with both digits signed
struct fx_digits { int hi, lo; };
FX_HD fx_digits fx_split(long long v) {
    return {(int)((v + 0x80000000ll) >> 32), (int)v};
}
// a b + c modulo 2^64
FX_HD long long fx_mad(int a, int b, long long c) {
    return (long long)((unsigned long long)((long long)a * b) + (unsigned long long)c);
}

// Twiddle factor as signed digits: re = ch 2^32 + cl, im = sh 2^32 + sl, scaled by 2^62.
struct __align__(16) fx_tw { int ch, cl, sh, sl; };

// (h 2^32 + m) / 2^32 rounded, where m is kept as m + 2^63 + 2^31 and h as
// h - 2^31: the middle sum is then unsigned and its high word needs no sign.
// Its low word is zero on a tie (factors 1, i, -1, -i), which goes to even.
constexpr long long kFxMid = (long long)0x8000000080000000ull, kFxTop = -0x80000000ll;
FX_HD long long fx_join(long long h, long long m) {
    const unsigned long long r = (unsigned long long)h + ((unsigned long long)m >> 32);
    return (long long)(r & ~(unsigned long long)((unsigned)m == 0));
}

// w x / 2^64, rounded; the product of the two low digits (below one unit) is
// left out.  |x| <= 2^62 keeps every sum below 2^63.
FX_HD fx2 fx_cmul(fx2 v, fx_tw w) {
    const fx_digits r = fx_split(v.x), i = fx_split(v.y);
    long long a = fx_mad(r.hi, w.cl, kFxMid);
    a = fx_mad(r.lo, w.ch, a);
    a = fx_mad(i.hi, -w.sl, a);
    a = fx_mad(i.lo, -w.sh, a);
    long long b = fx_mad(r.hi, w.sl, kFxMid);
    b = fx_mad(r.lo, w.sh, b);
    b = fx_mad(i.hi, w.cl, b);
    b = fx_mad(i.lo, w.ch, b);
    return {fx_join(fx_mad(r.hi, w.ch, fx_mad(i.hi, -w.sh, kFxTop)), a),
            fx_join(fx_mad(r.hi, w.sh, fx_mad(i.hi, w.ch, kFxTop)), b)};
}
// The same with three real products instead of four: with t = re + im,
// (c t - (c + s) im, c t + (s - c) re).  The sums c + s reach 2^62.5, so
// |x| <= 2^61 here.
struct __align__(16) fx_tw3 { int ch, cl, ph, pl, qh, ql, z0, z1; };   // c, -(c + s), s - c
FX_HD fx2 fx_cmul(fx2 v, const fx_tw3& w) {
    const fx_digits r = fx_split(v.x), i = fx_split(v.y), t = fx_split(v.x + v.y);
    long long m = fx_mad(t.hi, w.cl, kFxMid);
    m = fx_mad(t.lo, w.ch, m);
    const long long h = fx_mad(t.hi, w.ch, kFxTop);
    const long long a = fx_mad(i.lo, w.ph, fx_mad(i.hi, w.pl, m));
    const long long b = fx_mad(r.lo, w.qh, fx_mad(r.hi, w.ql, m));
    return {fx_join(fx_mad(i.hi, w.ph, h), a), fx_join(fx_mad(r.hi, w.qh, h), b)};
}
// v sqrt(1/2)
FX_HD long long fx_rsqrt2(long long v) {
    constexpr int h = 759250125, l = -25716447;   // 2^62 sqrt(1/2) = h 2^32 + l
    const fx_digits d = fx_split(v);
    long long a = fx_mad(d.hi, l, 0x20000000ll);
    a = fx_mad(d.lo, h, a);
    return (((long long)d.hi * h) << 2) + (a >> 30);
}
FX_HD fx2 fx_mul_w8(fx2 a) { return {fx_rsqrt2(a.x + a.y), fx_rsqrt2(a.y - a.x)}; }        // a exp(-i pi/4)
FX_HD fx2 fx_mul_w8_3(fx2 a) { return {fx_rsqrt2(a.y - a.x), fx_rsqrt2(-a.x - a.y)}; }     // a exp(-3 i pi/4)
FX_HD long long fx_quarter(long long v) { return (v + 1 + ((v >> 2) & 1)) >> 2; }
FX_HD fx2 fx_quarter(fx2 a) { return {fx_quarter(a.x), fx_quarter(a.y)}; }

FX_HD void fx_dft4(fx2& a, fx2& b, fx2& c, fx2& d) {
    const fx2 s = a + c, t = a - c, u = b + d, w = fx_mul_mi(b - d);
    a = s + u;
    b = t + w;
    c = s - u;
    d = t - w;
}
// c = d = 0 on entry
FX_HD void fx_dft4_half(fx2& a, fx2& b, fx2& c, fx2& d) {
    const fx2 p = a, q = b, w = fx_mul_mi(b);
    a = p + q;
    b = p + w;
    c = p - q;
    d = p - w;
}

// DFT of v[0..R) in place, natural order.  HALF: the upper half is zero on entry.
template <int R, bool HALF>
FX_HD void fx_dft(fx2* v) {
    if constexpr (R == 2) {
        const fx2 a = v[0], b = HALF ? fx2{0, 0} : v[1];
        v[0] = a + b;
        v[1] = a - b;
    } else if constexpr (R == 4) {
        if (HALF) fx_dft4_half(v[0], v[1], v[2], v[3]);
        else fx_dft4(v[0], v[1], v[2], v[3]);
    } else {
        static_assert(R == 8, "radix 2, 4 or 8");
        fx2 e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
        if (HALF) { fx_dft4_half(e0, e1, e2, e3); fx_dft4_half(o0, o1, o2, o3); }
        else { fx_dft4(e0, e1, e2, e3); fx_dft4(o0, o1, o2, o3); }
        o1 = fx_mul_w8(o1);
        o2 = fx_mul_mi(o2);
        o3 = fx_mul_w8_3(o3);
        v[0] = e0 + o0; v[4] = e0 - o0;
        v[1] = e1 + o1; v[5] = e1 - o1;
        v[2] = e2 + o2; v[6] = e2 - o2;
        v[3] = e3 + o3; v[7] = e3 - o3;
    }
}

// The passes of a line of length 2^LG with E entries per thread, radix
// 2^lg(p) <= E, decimation in frequency: after pass p the line is split into
// blocks of M(p) = L / (r_1 .. r_p) entries.  E = 8 (64 registers, 32 warps per
// SM): 16 entries per thread save an exchange but leave half the warps and
// overflow the instruction cache (n = 512, 64 right-hand sides: 3.36 ms per
// operator against 2.95; 80 registers with 24 warps 3.10).  E = 4 where a pass
// has too few entries to give the SMs warps (lss_fx_entries).  At L = 1024 two
// lines per CTA (2.94 ms) beat four (3.07 ms: 512-thread barriers).
template <int LG, int E>
struct FxPlan {
    static constexpr int L = 1 << LG;
    static constexpr int T = L / E;                                      // threads per line
    // lines per CTA, interleaved in shared memory (C x 16 bytes contiguous)
    static constexpr int C = LG <= 9 ? 4 : 2;
    static constexpr int TPB = C * T;
    static constexpr int lg(int p) {
        constexpr int t8[6][5] = {{3, 3}, {3, 2, 2}, {3, 3, 2}, {3, 3, 3}, {3, 3, 2, 2}, {3, 3, 3, 2}};
        constexpr int t4[6][5] = {{2, 2, 2}, {2, 2, 2, 1}, {2, 2, 2, 2}, {2, 2, 2, 2, 1}, {2, 2, 2, 2, 2}, {}};
        return E == 8 ? t8[LG - 6][p] : t4[LG - 6][p];
    }
    static constexpr int np() {
        int k = 0;
        while (k < 5 && lg(k)) ++k;
        return k;
    }
    static constexpr int NP = np();
    static constexpr int lgB(int p) {   // block length before pass p
        int b = LG;
        for (int q = 0; q < p; ++q) b -= lg(q);
        return b;
    }
    static constexpr int lgM(int p) { return lgB(p) - lg(p); }
    // three products where the lost bit is free: not at L = 2048, nor below 256,
    // whose lines the 3D operator passes through five times
    static constexpr bool kThree = LG >= 8 && LG <= 10;
    using Tw = std::conditional_t<kThree, fx_tw3, fx_tw>;
    static constexpr int kMax = kThree ? 60 : 61;
    // bits of an entry at the start of pass p: the pass multiplies the modulus
    // by at most 2^lg(p) sqrt(2), and 2^61 (2^62) is the limit of the products
    static constexpr int bits(int p) { return kMax - lg(p); }
    static constexpr int bits_half() { return kMax + 1 - lg(0); }   // first pass of a line whose upper half is zero
};

// Host: the digits of 2^62 v (|v| < 2); both digits have negatives.
inline fx_digits fx_host_digits(long double v) {
    fx_digits d = fx_split(llrintl(ldexpl(v, 62)));
    if (d.lo == (int)0x80000000) d.lo += 1;
    return d;
}
inline void fx_host_tw(long double c, long double s, fx_tw& w) {
    const fx_digits a = fx_host_digits(c), b = fx_host_digits(s);
    w = {a.hi, a.lo, b.hi, b.lo};
}
inline void fx_host_tw(long double c, long double s, fx_tw3& w) {
    const fx_digits a = fx_host_digits(c), p = fx_host_digits(-(c + s)), q = fx_host_digits(s - c);
    w = {a.hi, a.lo, p.hi, p.lo, q.hi, q.lo, 0, 0};
}
// Host: c[k] + i s[k] = exp(-2 pi i k / L), 8 | L, from the first octant.  Every
// context makes this table; the functions take 0.2 microseconds each
// in 128-bit long double (n = 256, all of them evaluated: 0.4 ms of 3.3 ms
// of set-up).
inline void fx_host_roots(int L, long double* c, long double* s) {
    const long double u = 2.0L * 3.14159265358979323846264338327950288L / (long double)L;
    for (int k = 0; k <= L / 8; ++k) {
        c[k] = cosl(u * k);
        s[k] = -sinl(u * k);
    }
    for (int k = L / 8 + 1; k <= L / 4; ++k) {   // mirrored at pi / 4
        c[k] = -s[L / 4 - k];
        s[k] = -c[L / 4 - k];
    }
    for (int k = L / 4 + 1; k < L; ++k) {        // a quarter turn on
        c[k] = s[k - L / 4];
        s[k] = -c[k - L / 4];
    }
}

// Position in the line of entry e (butterfly e / r, input e % r) of thread t in pass P.
template <int LG, int E, int P>
FX_HD int fx_pos(int t, int e) {
    using PL = FxPlan<LG, E>;
    constexpr int r = 1 << PL::lg(P), lgM = PL::lgM(P), lgB = PL::lgB(P);
    const int q = t + PL::T * (e / r), k = e % r;
    return ((q >> lgM) << lgB) + (k << lgM) + (q & ((1 << lgM) - 1));
}
// Where a transformed line stores the same entry of the last pass (order that
// lets neighbouring threads write neighbouring entries).
template <int LG, int E>
FX_HD int fx_spos(int t, int e) {
    using PL = FxPlan<LG, E>;
    constexpr int lgr = PL::lg(PL::NP - 1), r = 1 << lgr;
    return ((e % r) << (LG - lgr)) + t + PL::T * (e / r);
}
// Frequency stored at position s of a transformed line.
template <int LG, int E>
FX_HD int fx_freq(int s) {
    using PL = FxPlan<LG, E>;
    constexpr int lgl = PL::lg(PL::NP - 1);
    int q = s & ((1 << (LG - lgl)) - 1);   // block of the last pass: k_1 r_2 .. + k_2 r_3 .. + ..
    int f = (s >> (LG - lgl)) << (LG - lgl), lo = 0, left = LG - lgl;
    for (int p = 0; p + 1 < PL::NP; ++p) {
        left -= PL::lg(p);
        f += (q >> left) << lo;
        q &= (1 << left) - 1;
        lo += PL::lg(p);
    }
    return f;
}
// Position at which a line stores frequency f (the inverse of fx_freq).
template <int LG, int E>
FX_HD int fx_store(int f) {
    using PL = FxPlan<LG, E>;
    constexpr int lgl = PL::lg(PL::NP - 1);
    int q = 0;
    for (int p = 0; p + 1 < PL::NP; ++p) {
        q = (q << PL::lg(p)) | (f & ((1 << PL::lg(p)) - 1));
        f >>= PL::lg(p);
    }
    return (f << (LG - lgl)) + q;
}
// Shared-memory index (entries) of position pos of line c of the CTA.  The
// lines are interleaved; the position's low bits are mixed with the bits that
// neighbouring threads of the last pass differ in, so that the eight threads
// of a 128-byte access always fall on different banks.
template <int LG, int E>
FX_HD int fx_sidx(int pos, int c) {
    using PL = FxPlan<LG, E>;
    constexpr int lgr = PL::lg(PL::NP - 1), mix = 8 / PL::C - 1;
    return (pos ^ ((pos >> lgr) & mix)) * PL::C + c;
}

// Pass P of the forward transform on a thread's entries: butterflies, then the
// twiddle factors (not after the last pass).  FIRST_HALF: the line's upper half is zero.
template <int LG, int E, int P>
FX_HD void fx_fwd_pass(fx2* v, int t, const typename FxPlan<LG, E>::Tw* __restrict__ tw) {
    using PL = FxPlan<LG, E>;
    constexpr int r = 1 << PL::lg(P), lgM = PL::lgM(P), sc = LG - PL::lgB(P);
#pragma unroll
    for (int i = 0; i < E / r; ++i) {
        fx_dft<r, P == 0>(v + i * r);
        if constexpr (P + 1 < PL::NP) {
            const int m = (t + PL::T * i) & ((1 << lgM) - 1);
            v[i * r] = fx_quarter(v[i * r]);
#pragma unroll
            for (int k = 1; k < r; ++k) v[i * r + k] = fx_cmul(v[i * r + k], tw[(m * k) << sc]);
        }
    }
}
// Pass P of the inverse transform (passes run from the last to the first) on
// entries with real and imaginary parts exchanged, which turns the forward
// factors and butterflies into the inverse ones.
template <int LG, int E, int P>
FX_HD void fx_inv_pass(fx2* v, int t, const typename FxPlan<LG, E>::Tw* __restrict__ tw) {
    using PL = FxPlan<LG, E>;
    constexpr int r = 1 << PL::lg(P), lgM = PL::lgM(P), sc = LG - PL::lgB(P);
#pragma unroll
    for (int i = 0; i < E / r; ++i) {
        if constexpr (P + 1 < PL::NP) {
            const int m = (t + PL::T * i) & ((1 << lgM) - 1);
            v[i * r] = fx_quarter(v[i * r]);
#pragma unroll
            for (int k = 1; k < r; ++k) v[i * r + k] = fx_cmul(v[i * r + k], tw[(m * k) << sc]);
        }
        fx_dft<r, false>(v + i * r);
    }
}

// v 2^s, rounded (ties to even)
FX_HD long long fx_shift(long long v, int s) {
    if (s >= 0) return (long long)((unsigned long long)v << (s & 63));
    const int b = -s > 62 ? 62 : -s;
    return (v + ((1ll << (b - 1)) - 1) + ((v >> b) & 1)) >> b;
}
// The shift of a whole line (0 <= s < 32 but for the rare line that grew)
template <int E>
FX_HD void fx_shift_line(fx2* v, int s) {
    if (s < 0) {
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = {fx_shift(v[e].x, s), fx_shift(v[e].y, s)};
    } else {
        s = s < 31 ? s : 31;
#pragma unroll
        for (int e = 0; e < E; ++e)
            v[e] = {(long long)((unsigned long long)v[e].x << s), (long long)((unsigned long long)v[e].y << s)};
    }
}
// Bits that the larger part of v uses (not below 32).
FX_HD int fx_clz32(unsigned u) {
#ifdef __CUDA_ARCH__
    return __clz((int)u);
#else
    return u ? __builtin_clz(u) : 32;
#endif
}
FX_HD unsigned fx_fold(fx2 v) {
    const int a = (int)(v.x >> 32), b = (int)(v.y >> 32);
    return (unsigned)((a ^ (a >> 31)) | (b ^ (b >> 31)));
}
FX_HD int fx_bits(unsigned fold) { return 64 - fx_clz32(fold); }

// d as mantissa and exponent: d = v 2^e, |v| < 2^53; e = kFxBad when d is not finite.
FX_HD long long fx_from_double(double d, int& e) {
#ifdef __CUDA_ARCH__
    const long long b = __double_as_longlong(d);
#else
    long long b;
    __builtin_memcpy(&b, &d, 8);
#endif
    const int x = (int)((b >> 52) & 0x7ff);
    long long v = b & 0xfffffffffffffll;
    if (x) v |= 1ll << 52;
    e = x == 0x7ff ? kFxBad : (x ? x : 1) - 1075;
    return b < 0 ? -v : v;
}

// Kernel-transform entries: digits below 2^61 with one exponent per line, 2^x
// per unit (field: the exponent field of the line's largest part).
FX_HD int fx_kernel_exp(unsigned field) { return (field > 64 ? (int)field : 64) - 1022 - 61; }
FX_HD fx_tw fx_kernel_digits(long long re, long long im) {
    fx_digits a = fx_split(re), b = fx_split(im);
    if (a.lo == (int)0x80000000) a.lo += 1;   // its negative has to be a digit too
    if (b.lo == (int)0x80000000) b.lo += 1;
    return {a.hi, a.lo, b.hi, b.lo};
}

// Product with a kernel-transform entry: w = (v k) >> 64 with 16 more bits in
// the upper half of frac, shifted right by PS.  The bits below those are folded
// into the last of the 16 (rounding to odd, so that fx_lift's rounding is that
// of the product; the lower half is not to be used).  The products of the low digits count here: an entry that the
// kernel makes small is shifted up afterwards, by many bits where the line's
// energy lies far from its resonance (n = 512, a field of alternating sign:
// error 1.3e-16 against 5.4e-15 without them, 6.2e-16 in FP64).
template <int PS>
FX_HD void fx_kmul(fx2 v, fx_tw k, fx2& w, unsigned& fx, unsigned& fy) {
    const fx_digits r = fx_split(v.x), i = fx_split(v.y);
    long long a = fx_mad(r.lo, k.cl, fx_mad(i.lo, -k.sl, 0)) >> 32;
    a = fx_mad(r.hi, k.cl, a);
    a = fx_mad(r.lo, k.ch, a);
    a = fx_mad(i.hi, -k.sl, a);
    a = fx_mad(i.lo, -k.sh, a);
    long long b = fx_mad(r.lo, k.sl, fx_mad(i.lo, k.cl, 0)) >> 32;
    b = fx_mad(r.hi, k.sl, b);
    b = fx_mad(r.lo, k.sh, b);
    b = fx_mad(i.hi, k.cl, b);
    b = fx_mad(i.lo, k.ch, b);
    const long long x = fx_mad(r.hi, k.ch, fx_mad(i.hi, -k.sh, a >> 32));
    const long long y = fx_mad(r.hi, k.sh, fx_mad(i.hi, k.ch, b >> 32));
    fx = (unsigned)((((unsigned long long)(unsigned)x << 32) | (unsigned)a) >> PS);
    fy = (unsigned)((((unsigned long long)(unsigned)y << 32) | (unsigned)b) >> PS);
    fx |= (unsigned)((fx & 0xffffu) != 0) << 16;
    fy |= (unsigned)((fy & 0xffffu) != 0) << 16;
    w = {x >> PS, y >> PS};
}
// (w : frac) 2^s rounded to units, ties to even; 0 <= s < 32, frac a multiple of 2^16
FX_HD long long fx_lift(long long w, unsigned frac, int s) {
    const unsigned long long f = (unsigned long long)frac << s;
    const long long v = (long long)(((unsigned long long)w << s) + (f >> 32));
    return v + ((unsigned)f + (unsigned)(v & 1) > 0x80000000u);
}
