// Host harness of the fixed-point line transforms (fx_line.cuh): convolutions
// of lines with a kernel line, as the operator's column pass forms them, in
// the shipped integer arithmetic, in double and in long double.
//   fixed_fft_host LG E LINES  <stdin: LINES x n and L complex doubles>
// writes, per line, the n fixed-point and the n double results minus the long
// double one, and that one (complex doubles).
#include <algorithm>
#include <cmath>
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "fx_line.cuh"

namespace {

using cd = std::complex<double>;
template <typename R> using cxv = std::vector<std::complex<R>>;

template <int LG, int E>
struct Host {
    using PL = FxPlan<LG, E>;
    static constexpr int L = PL::L, T = PL::T, NP = PL::NP, r0 = 1 << PL::lg(0);
    std::vector<typename PL::Tw> tw = std::vector<typename PL::Tw>(L);
    std::vector<fx2> v = std::vector<fx2>(L), sm = std::vector<fx2>(L);   // entry e of thread t at t E + e
    int ex = 0;

    Host() {
        for (int k = 0; k < L; ++k) {
            const long double a = -2.0L * acosl(-1.0L) * k / L;
            fx_host_tw(cosl(a), sinl(a), tw[k]);
        }
    }
    unsigned fold() const {
        unsigned f = 0;
        for (const fx2& q : v) f |= fx_fold(q);
        return f;
    }
    template <int A, int B> void exchange() {
        const int s = std::min(PL::bits(B) - fx_bits(fold()), 31);
        for (int t = 0; t < T; ++t)
            for (int e = 0; e < E; ++e) sm[fx_pos<LG, E, A>(t, e)] = v[t * E + e];
        for (int t = 0; t < T; ++t) {
            for (int e = 0; e < E; ++e) v[t * E + e] = sm[fx_pos<LG, E, B>(t, e)];
            fx_shift_line<E>(&v[t * E], s);
        }
        ex -= s;
    }
    template <int P> void forward() {
        if constexpr (P > 0) exchange<P - 1, P>();
        for (int t = 0; t < T; ++t) fx_fwd_pass<LG, E, P>(&v[t * E], t, tw.data());
        if constexpr (P + 1 < NP) { ex += 2; forward<P + 1>(); }
    }
    template <int P> void inverse() {
        if constexpr (P + 1 < NP) { exchange<P + 1, P>(); ex += 2; }
        for (int t = 0; t < T; ++t) fx_inv_pass<LG, E, P>(&v[t * E], t, tw.data());
        if constexpr (P > 0) inverse<P - 1>();
    }
    void conv(const cd* x, const cd* k, int n, cd* y) {
        std::vector<int> e1(2 * L, 0);
        int top = -100000;
        for (int t = 0; t < T; ++t)
            for (int e = 0; e < E; ++e) {
                const int j = fx_pos<LG, E, 0>(t, e), q = t * E + e;
                v[q] = {0, 0};
                if (e % r0 >= r0 / 2 || j >= n) continue;
                v[q] = {fx_from_double(x[j].real(), e1[2 * q]), fx_from_double(x[j].imag(), e1[2 * q + 1])};
                if (x[j].real() != 0) top = std::max(top, e1[2 * q] + 53);
                if (x[j].imag() != 0) top = std::max(top, e1[2 * q + 1] + 53);
            }
        ex = top - PL::bits_half();
        for (int q = 0; q < L; ++q) v[q] = {fx_shift(v[q].x, e1[2 * q] - ex), fx_shift(v[q].y, e1[2 * q + 1] - ex)};
        forward<0>();
        constexpr int PS = PL::lg(NP - 1) - 1;
        unsigned field = 0;
        for (int j = 0; j < 2 * L; ++j) {
            unsigned long long b;
            memcpy(&b, (const double*)k + j, 8);
            field = std::max(field, (unsigned)(b >> 52) & 0x7ffu);
        }
        const int kx = fx_kernel_exp(field);
        std::vector<unsigned> fr(2 * L);
        for (int t = 0; t < T; ++t)
            for (int e = 0; e < E; ++e) {
                const int q = t * E + e;
                const cd w = k[fx_freq<LG, E>(fx_spos<LG, E>(t, e))];
                fx_kmul<PS>(v[q], fx_kernel_digits(llrint(scalbn(w.real(), -kx)), llrint(scalbn(w.imag(), -kx))), v[q],
                            fr[2 * q], fr[2 * q + 1]);
            }
        const int s = std::min(PL::bits(NP - 1) - fx_bits(fold()), 31);
        for (int q = 0; q < L; ++q)
            v[q] = {fx_lift(v[q].x, fr[2 * q] & 0xffff0000u, s), fx_lift(v[q].y, fr[2 * q + 1] & 0xffff0000u, s)};
        ex += kx + 64 + PS - s;
        for (fx2& q : v) q = fx_swap(q);
        inverse<NP - 1>();
        for (fx2& q : v) q = fx_swap(q);
        for (int t = 0; t < T; ++t)
            for (int e = 0; e < E; ++e) {
                const int j = fx_pos<LG, E, 0>(t, e);
                if (e % r0 < r0 / 2 && j < n) y[j] = cd(scalbn((double)v[t * E + e].x, ex), scalbn((double)v[t * E + e].y, ex));
            }
    }
};

template <typename R>
void fft(cxv<R>& a, bool back) {   // radix 2, decimation in time
    const int L = (int)a.size();
    for (int i = 1, j = 0; i < L; ++i) {
        int b = L >> 1;
        for (; j & b; b >>= 1) j ^= b;
        j ^= b;
        if (i < j) std::swap(a[i], a[j]);
    }
    for (int h = 1; h < L; h *= 2)
        for (int q = 0; q < h; ++q) {
            const long double t = (back ? 1 : -1) * acosl(-1.0L) * q / h;
            const R c = (R)cosl(t), s = (R)sinl(t);
            for (int i = q; i < L; i += 2 * h) {
                const std::complex<R> u = a[i], z = a[i + h];
                const std::complex<R> p(z.real() * c - z.imag() * s, z.real() * s + z.imag() * c);
                a[i] = u + p;
                a[i + h] = u - p;
            }
        }
}
template <typename R>
cxv<R> conv(const cd* x, const cd* k, int n, int L) {
    cxv<R> a(L);
    for (int j = 0; j < n; ++j) a[j] = std::complex<R>(x[j].real(), x[j].imag());
    fft(a, false);
    for (int j = 0; j < L; ++j) {
        const R kr = k[j].real(), ki = k[j].imag(), ar = a[j].real(), ai = a[j].imag();
        a[j] = std::complex<R>(ar * kr - ai * ki, ar * ki + ai * kr);
    }
    fft(a, true);
    return a;
}

template <int LG, int E>
int run(int lines) {
    constexpr int L = 1 << LG, n = L / 2;
    std::vector<cd> x((size_t)lines * n), k(L), y(n), out((size_t)3 * lines * n);
    if (fread(x.data(), sizeof(cd), x.size(), stdin) != x.size() || fread(k.data(), sizeof(cd), L, stdin) != (size_t)L) return 2;
    Host<LG, E> H;
    for (int l = 0; l < lines; ++l) {
        const cxv<long double> r = conv<long double>(&x[(size_t)l * n], k.data(), n, L);
        const cxv<double> d = conv<double>(&x[(size_t)l * n], k.data(), n, L);
        H.conv(&x[(size_t)l * n], k.data(), n, y.data());
        for (int j = 0; j < n; ++j) {
            cd* o = &out[(size_t)3 * l * n + j];
            o[0] = cd((double)(y[j].real() - r[j].real()), (double)(y[j].imag() - r[j].imag()));
            o[n] = cd((double)(d[j].real() - r[j].real()), (double)(d[j].imag() - r[j].imag()));
            o[2 * n] = cd((double)r[j].real(), (double)r[j].imag());
        }
    }
    return fwrite(out.data(), sizeof(cd), out.size(), stdout) == out.size() ? 0 : 2;
}

}  // namespace

int main(int argc, char** argv) {
    if (argc != 4) return 1;
    const int lg = atoi(argv[1]), E = atoi(argv[2]), lines = atoi(argv[3]);
    switch (10 * lg + E) {
        case 64: return run<6, 4>(lines);
        case 78: return run<7, 8>(lines);
        case 88: return run<8, 8>(lines);
        case 98: return run<9, 8>(lines);
        case 104: return run<10, 4>(lines);
        case 108: return run<10, 8>(lines);
        case 118: return run<11, 8>(lines);
        default: return 1;
    }
}
