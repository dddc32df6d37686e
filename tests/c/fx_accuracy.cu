// fx_accuracy.cu -- the fixed-point transforms (gsm_fx.cuh) on the host: one zero-padded line
// forward, times the multiplier 1/k^2 (2 at k = 0), inverse.  Prints, per line, the maximum error
// over the maximum of the result in fixed point and of a plain FFT in doubles, both against long
// double (tests/test_fixed_point_host.py).
#include <stdio.h>

#include <algorithm>
#include <complex>
#include <random>
#include <vector>

#include "gsm_fx.cuh"

using namespace gsm;
typedef long double ld;

static const ld kPi = 3.14159265358979323846264338327950288L;

struct In : FxDoubles {
    const double *re, *im;
    raw load(int b, int off) const { return {re[b + off], im[b + off]}; }
};
struct NoOut {
    static constexpr bool kSmem = false;
    void operator()(int, int, cx<long long>) const {}
};
struct Out {
    static constexpr bool kSmem = false;
    std::complex<double> *u;
    int n;
    const FxLine *ln;
    void operator()(int b, int off, cx<long long> v) const
    {
        if (b + off < n) u[b + off] = {fx_out_double(v.re, ln->E), fx_out_double(v.im, ln->E)};
    }
};
struct Mult {
    const int2 *row;
    int M;
    template <int R>
    int2 at(int b, int t, int nb) const
    {
        const int k = b + t * nb;
        return row[std::min(k, M - k)];
    }
};

template <class SC>
std::vector<int4> stage_table()
{
    std::vector<int4> t(SC::M);
    const auto l = SC::list();
    int Ns = l.r[0];
    for (int st = 1; st < l.n; Ns *= l.r[st++])
        for (int q = 1; q < l.r[st]; ++q)
            for (int j = 0; j < Ns; ++j) {
                const long D = (long)l.r[st] * Ns, k = (long)j * q;
                const ld a = 2 * kPi * k / D;
                ld c = cosl(a), s = sinl(a);
                if (4 * k % D == 0) c = roundl(c), s = roundl(s);
                const int2 x = fx_factor((double)c, (double)(c - (double)c)), y = fx_factor((double)s, (double)(s - (double)s));
                t[Ns - l.r[0] + (q - 1) * Ns + j] = make_int4(x.x, x.y, y.x, y.y);
            }
    return t;
}

template <int n>
std::vector<std::complex<double>> fixed(const std::vector<double> &re, const std::vector<double> &im,
                                        const std::vector<double> &mult)
{
    constexpr int M = 2 * n;
    using F = FixedSched<M>;
    using I = FixedSched<M, true>;
    const std::vector<int4> tw = stage_table<F>(), twi = stage_table<I>();
    int e;
    frexp(*std::max_element(mult.begin(), mult.end()), &e);
    std::vector<int2> row(n + 1);
    for (int k = 0; k <= n; ++k) row[k] = fx_mult_factor(ldexp(mult[k], -e));
    std::vector<fxc> s(M + M / 8 + 1);
    std::vector<std::complex<double>> u(n);
    int red[kFxRedWords];
    const Group g{0, 1, -1};
    FxLine ln{0, F::pad, M > kFxLongM, red, 1};
    In in;
    in.re = re.data();
    in.im = im.data();
    fx_begin<true, M, true, true>(s.data(), F(), g, ln, in, NoOut());
    fx_rest_of<true, M, false, true>(s.data(), F(), tw.data(), g, ln, NoOut());
    fx_mid_of<M>(s.data(), F(), I(), tw.data(), g, ln, Mult{row.data(), M}, e);
    fx_rest_of<false, M, true, false>(s.data(), I(), twi.data(), g, ln, Out{u.data(), n, &ln});
    return u;
}

template <class T>
void fft(std::vector<std::complex<T>> &x, int sign)   // recursive, smallest factor first
{
    const int n = (int)x.size();
    if (n == 1) return;
    int r = 2;
    while (n % r) ++r;
    const int m = n / r;
    std::vector<std::vector<std::complex<T>>> y(r, std::vector<std::complex<T>>(m));
    for (int i = 0; i < n; ++i) y[i % r][i / r] = x[i];
    for (auto &v : y) fft(v, sign);
    for (int k = 0; k < n; ++k) {
        x[k] = y[0][k % m];
        for (int t = 1; t < r; ++t) {
            const ld a = sign * 2 * kPi * ((long)k * t % n) / n;
            const T c = (T)cosl(a), s = (T)sinl(a);
            const std::complex<T> v = y[t][k % m];
            x[k] += std::complex<T>(v.real() * c - v.imag() * s, v.real() * s + v.imag() * c);
        }
    }
}
template <class T>
std::vector<std::complex<T>> floating(const std::vector<double> &re, const std::vector<double> &im,
                                      const std::vector<double> &mult)
{
    const int n = (int)re.size();
    std::vector<std::complex<T>> x(2 * n);
    for (int i = 0; i < n; ++i) x[i] = std::complex<T>(re[i], im[i]);
    fft(x, -1);
    for (int k = 0; k < 2 * n; ++k) x[k] *= (T)mult[std::min(k, 2 * n - k)];
    fft(x, 1);
    return x;
}

template <int n>
void run()
{
    std::vector<double> mult(n + 1, 2.0);
    for (int k = 1; k <= n; ++k) mult[k] = 1.0 / ((double)k * k);
    for (int c = 0; c < 6; ++c) {
        std::mt19937 r(n + c);
        std::normal_distribution<double> normal;
        std::vector<double> re(n), im(n);
        for (int i = 0; i < n; ++i) {
            const double t = (i - 0.45 * n) / (0.06 * n), g = exp(-t * t);
            switch (c) {
            case 0: re[i] = g; im[i] = 0.3 * g; break;                             // smooth
            case 1: re[i] = i == n / 3; break;                                     // a single point
            case 2: re[i] = normal(r); im[i] = normal(r); break;                   // white noise
            case 3: re[i] = g * cos(0.9 * M_PI * i); break;                        // a wave near Nyquist
            case 4: re[i] = i == n / 3 ? 1.0 : 1e-9 * fabs(normal(r)); break;      // a point over a floor
            default: re[i] = (i & 1 ? -1 : 1) * (1.0 + 1e-3 * normal(r)); break;   // alternating
            }
        }
        const auto u = fixed<n>(re, im, mult);
        const auto d = floating<double>(re, im, mult);
        const auto x = floating<ld>(re, im, mult);
        double mx = 0, ef = 0, ed = 0;
        for (int i = 0; i < n; ++i) {
            mx = std::max(mx, (double)std::abs(x[i]));
            ef = std::max(ef, (double)std::abs(x[i] - std::complex<ld>(u[i].real(), u[i].imag())));
            ed = std::max(ed, (double)std::abs(x[i] - std::complex<ld>(d[i].real(), d[i].imag())));
        }
        printf("%d %d %.3e %.3e\n", n, c, ef / mx, ed / mx);
    }
}

int main()
{
    run<50>();
    run<216>();
    run<250>();
    run<256>();
    run<1024>();
    run<2048>();
    return 0;
}
