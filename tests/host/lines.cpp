// Single lines of the FP64 transforms' engines, thread by thread on the CPU: the fixed-point engine
// (csrc/fx.cuh, fft4.cuh, fxg.cuh) and the same plan in FP64 against long double.
//   lines accuracy   per length, field and direction: rms relative errors of both engines
//   lines range      per plan: range errors (sums or factors that leave their words) over lines at
//                    the full scale, aligned with each frequency in turn
//   lines zeros      per plan and direction: outputs that cancel exactly but come out nonzero
//   lines convert    conversions to FP64 that are not the nearest value (either one at a tie)
#include "fft4.cuh"
#include "fxg.cuh"

#include <complex>
#include <cstdio>
#include <random>
#include <string>
#include <vector>

using namespace lsm;
typedef std::complex<long double> cl;
typedef std::vector<double2> Line;

struct Tables {
    std::vector<int4> fx[4];   // entries times 2^-2, 2^-3 at [2], [3]
    Line d;
    std::vector<cl> exact;
    explicit Tables(int L) {
        const long double pi = 3.141592653589793238462643383279502884L;
        for (int k = 0; k < L; ++k) {
            const long double a = -2 * pi * k / L, c = cosl(a), s = sinl(a);
            exact.push_back({c, s});
            d.push_back({(double)c, (double)s});
            for (int K = 2; K < 4; ++K) {
                int4 w;
                fx_table_words(ldexpl(c, -K), &w.x, &w.y);
                fx_table_words(ldexpl(s, -K), &w.z, &w.w);
                fx[K].push_back(w);
            }
        }
    }
};

template <int A, int B, int S, int NZ, int NO, class C, class Tw, class St>
static void two_step(const C* in, const Tw* tw, St st) {
    constexpr int L = A * B;
    static C mid[L];
    for (int t = 0; t < B; ++t) {
        C v[A];
        for (int k = 0; k < A; ++k) v[k] = k < NZ ? in[t + B * k] : czero<C>();
        dft_reg_p<A, S, NZ, A>(v);
        tw_row<S, L, A>(v, tw, t);
        for (int k = 0; k < A; ++k) mid[t * A + k] = v[k];
    }
    for (int k1 = 0; k1 < A; ++k1) {
        C w[B];
        for (int t = 0; t < B; ++t) w[t] = mid[t * A + k1];
        dft_reg_p<B, S, B, NO>(w);
        for (int k = 0; k < NO; ++k) st(k1 + A * k, w[k]);
    }
}

// One length: forward lines of n nodes at offset 1 (the first half of the line and one more element
// may hold them), inverse lines of which the first n + 2 outputs are wanted.
struct Plan {
    int L;
    virtual void fixed(int S, const Line& in, int nin, Line& out, const Tables& T) const = 0;
    virtual void fp64(int S, const Line& in, Line& out, const Tables& T) const = 0;
    virtual int scale_bits(int S, int nin) const = 0;                          // of the integers `raw` takes
    virtual void raw(int S, const fxc* in, int nin, const Tables& T) const = 0;
    virtual ~Plan() {}
};

template <int A, int B> struct TwoStep : Plan {
    TwoStep() { L = A * B; }
    static int bits(int S, int nin) { return fx_bits(A * B, nin, S < 0 ? A / 2 + 1 : A, B); }
    int scale_bits(int S, int nin) const override { return bits(S, nin) + fx_prescale(A * B); }
    template <class C, class Tw, class St> static void any(int S, const C* in, const Tw* tw, St st) {
        if (S < 0) two_step<A, B, -1, A / 2 + 1, B>(in, tw, st);
        else two_step<A, B, 1, A, B / 2 + 1>(in, tw, st);
    }
    void fixed(int S, const Line& in, int nin, Line& out, const Tables& T) const override {
        unsigned mag = 0;
        for (const double2& v : in) mag = max(mag, max(fx_mag(v.x), fx_mag(v.y)));
        const FxScale sc(mag);
        std::vector<fxc> q;
        for (const double2& v : in) q.push_back(fx_from(v, sc, scale_bits(S, nin)));
        const FxUnit un(sc.unit(bits(S, nin)), sc.bad, mag == 0);
        any(S, q.data(), T.fx[fx_twiddle_k(A * B)].data(), [&](int k, fxc r) { out[k] = un.odd ? fx_to_odd(r, un) : fx_to(r, un); });
    }
    void fp64(int S, const Line& in, Line& out, const Tables& T) const override {
        any(S, in.data(), T.d.data(), [&](int k, double2 r) { out[k] = r; });
    }
    void raw(int S, const fxc* in, int, const Tables& T) const override {
        any(S, in, T.fx[fx_twiddle_k(A * B)].data(), [](int, fxc) {});
    }
};

// the runtime engine, one thread for a tile of one line
struct Runtime : Plan {
    FxPlan p;
    explicit Runtime(int len) {
        L = len;
        factor_plan(len, p);
    }
    int scale_bits(int, int) const override { return p.fxbits; }
    template <int S, bool DYN> fxc* run(std::vector<fxc>& a, std::vector<fxc>& b, const Tables& T, int& esum) const {
        unsigned hi[3] = {0, 0, 0};
        return fxg_fft<S, 1, DYN, 1>(a.data(), b.data(), p, FxTables{T.fx[2].data(), T.fx[3].data()}, 0, 0, 1, hi, 0, esum);
    }
    fxc* any(int S, std::vector<fxc>& a, std::vector<fxc>& b, const Tables& T, int& esum) const {
        if (S < 0) return p.fxdyn ? run<-1, true>(a, b, T, esum) : run<-1, false>(a, b, T, esum);
        return p.fxdyn ? run<1, true>(a, b, T, esum) : run<1, false>(a, b, T, esum);
    }
    void fixed(int S, const Line& in, int, Line& out, const Tables& T) const override {
        unsigned mag = 0;
        for (const double2& v : in) mag = max(mag, max(fx_mag(v.x), fx_mag(v.y)));
        const FxScale sc(mag);
        std::vector<fxc> q, b(L);
        for (const double2& v : in) q.push_back(fx_from(v, sc, p.fxbits));
        int esum;
        const fxc* r = any(S, q, b, T, esum);
        const FxUnit un(sc.unit(p.fxbits) + esum, sc.bad, mag == 0);
        for (int k = 0; k < L; ++k) out[k] = un.odd ? fx_to_odd(r[k], un) : fx_to(r[k], un);
    }
    void fp64(int S, const Line& in, Line& out, const Tables& T) const override {
        Line a = in, b(L);
        const double2* r = S < 0 ? fft_smem<-1>(a.data(), b.data(), p, 1, 1, T.d.data(), 0, 1)
                                 : fft_smem<1>(a.data(), b.data(), p, 1, 1, T.d.data(), 0, 1);
        for (int k = 0; k < L; ++k) out[k] = r[k];
    }
    void raw(int S, const fxc* in, int, const Tables& T) const override {
        std::vector<fxc> a(in, in + L), b(L);
        int esum;
        any(S, a, b, T, esum);
    }
};

static void dft(int S, const Line& in, std::vector<cl>& out, const Tables& T) {
    const int L = (int)in.size();
    out.assign(L, 0);
    for (int k = 0; k < L; ++k)
        for (int n = 0; n < L; ++n) {
            const cl w = T.exact[(long long)k * n % L];
            out[k] += cl(in[n].x, in[n].y) * (S > 0 ? std::conj(w) : w);
        }
}
static double rel2(const Line& a, const std::vector<cl>& r, int n0, int n1) {
    long double e = 0, m = 0;
    for (int k = n0; k < n1; ++k) {
        e += std::norm(cl(a[k].x, a[k].y) - r[k]);
        m += std::norm(r[k]);
    }
    return (double)(e / m);
}

static std::mt19937_64 rng(5);
static double uniform() { return (double)(rng() >> 11) / 9007199254740992.0; }
static double normal() { return std::sqrt(-2 * std::log(uniform() + 1e-300)) * std::cos(2 * M_PI * uniform()); }

static const char* FIELDS[] = {"smooth", "white", "point", "difference", "plane", "decaying"};
static Line field(int kind, int n, double nodes_per_wave) {
    Line f(n, double2{0, 0});
    const double k0 = 2 * M_PI / nodes_per_wave;
    if (kind == 0) {
        for (int m = -3; m < 3; ++m) {
            const double a = normal(), b = normal(), k = k0 * (m + 0.3 * normal()) / 2.5;
            for (int i = 0; i < n; ++i) {
                f[i].x += a * std::cos(k * i) - b * std::sin(k * i);
                f[i].y += a * std::sin(k * i) + b * std::cos(k * i);
            }
        }
    } else if (kind == 1) {
        for (double2& v : f) v = double2{normal(), normal()};
    } else if (kind == 2) {
        f[n / 3] = double2{0.7, -0.4};
    } else if (kind == 3) {
        f[n / 3] = double2{1.0, 0.2};
        f[n / 3 + 2] = double2{-1.0, -0.2};
    } else if (kind == 4) {
        for (int i = 0; i < n; ++i) f[i] = double2{std::cos(k0 * i + 0.3), std::sin(k0 * i + 0.3)};
    } else {   // by eight decades along the line
        for (int i = 0; i < n; ++i) f[i] = double2{normal() * std::pow(10.0, -8.0 * i / n), normal() * std::pow(10.0, -8.0 * i / n)};
    }
    return f;
}

// Forward lines of each field, and inverse lines of their spectra times the spectrum of a scalar Green
// table exp(i kz |m|) / kz at transverse wavenumbers below, near and above the wave's
static void accuracy(const Plan& p) {
    const int L = p.L, n = L / 2;
    const Tables T(L);
    for (int kind = 0; kind < 6; ++kind) {
        double e[2][2] = {{0, 0}, {0, 0}};
        for (double npw : {10.0, 25.0})
            for (int rep = 0; rep < 3; ++rep) {
                const Line f = field(kind, n, npw);
                Line in(L, double2{0, 0}), out(L);
                for (int i = 0; i < n; ++i) in[i + 1] = f[i];
                std::vector<cl> F, G, want;
                dft(-1, in, F, T);
                p.fixed(-1, in, n, out, T);
                e[0][0] += rel2(out, F, 0, L) / 6;
                p.fp64(-1, in, out, T);
                e[0][1] += rel2(out, F, 0, L) / 6;
                const double k0 = 2 * M_PI / npw;
                for (double s : {0.0, 0.5, 0.95, 1.3}) {
                    const cl kz = std::sqrt(cl(k0 * k0 * (1 - s * s), 1e-4 * k0 * k0));
                    Line g(L, double2{0, 0});
                    for (int m = 1 - n; m < n; ++m) {
                        const cl v = std::exp(cl(0, 1) * kz * cl(std::abs(m))) / kz;
                        g[(m + L) % L] = double2{(double)v.real(), (double)v.imag()};
                    }
                    dft(-1, g, G, T);
                    for (int k = 0; k < L; ++k) {
                        const cl v = G[k] * F[k];
                        g[k] = double2{(double)v.real(), (double)v.imag()};
                    }
                    dft(1, g, want, T);
                    p.fixed(1, g, L, out, T);
                    e[1][0] += rel2(out, want, 1, n + 1) / 24;
                    p.fp64(1, g, out, T);
                    e[1][1] += rel2(out, want, 1, n + 1) / 24;
                }
            }
        for (int d = 0; d < 2; ++d)
            std::printf("%d %s %s %.4e %.4e\n", L, d ? "inverse" : "forward", FIELDS[kind], std::sqrt(e[d][0]), std::sqrt(e[d][1]));
    }
}

static void range(const Plan& p) {
    const int L = p.L, n = L / 2;
    const Tables T(L);
    for (int c = 0; c < 4; ++c) {
        const int S = c < 3 ? -1 : 1, nin = c == 0 ? n + 2 : (c < 3 ? n : L), off = c == 2 ? 1 : 0;
        const long long top = 1LL << p.scale_bits(S, nin);   // components lie in [-top, top)
        const long before = fx_range_errors;
        std::vector<fxc> in(L);
        for (int m = 0; m < L; ++m)
            for (int phase = 0; phase < 4; ++phase)
                for (int signs = 0; signs < 2; ++signs) {
                    for (fxc& v : in) v = czero<fxc>();
                    for (int i = 0; i < nin; ++i) {
                        const double a = -S * 2 * M_PI * ((long long)m * (i + off) % L) / L + M_PI / 8 * phase + 0.01;
                        const double x = std::cos(a), y = std::sin(a);
                        in[i + off] = signs ? fxc{fx_r(x > 0 ? top - 1 : -top), fx_r(y > 0 ? top - 1 : -top)}
                                            : fxc{fx_r((long long)(x * (double)(top - 1))), fx_r((long long)(y * (double)(top - 1)))};
                    }
                    p.raw(S, in.data(), nin, T);
                }
        std::printf("%d %d %d %d %ld\n", L, S, nin, off, fx_range_errors - before);
    }
}

// Two equal elements half a line apart: every odd output is x - x
static void zeros(const Plan& p) {
    const int L = p.L;
    const Tables T(L);
    for (int S = -1; S <= 1; S += 2) {
        Line in(L, double2{0, 0}), out(L, double2{0, 0});
        in[0] = in[L / 2] = double2{0.3, -1.7};
        p.fixed(S, in, S < 0 ? L / 2 + 1 : L, out, T);
        int bad = 0;
        for (int k = 1; k <= L / 2; k += 2) bad += out[k].x != 0.0 || out[k].y != 0.0;
        std::printf("%d %d %d\n", L, S, bad);
    }
}

static void convert() {
    long bad = 0, subnormal = 0;
    for (int i = 0; i < 400000; ++i) {
        const long long v = (long long)((unsigned long long)((long long)(rng() >> 1) >> (i % 63)) << (i / 63 % 3));
        const int E = -1140 + (int)(rng() % 2110);
        if (v < 0) continue;
        const long double exact = ldexpl((long double)(i & 1 ? -v : v), E);
        const FxUnit un(E, false, false);
        const double got = un.odd ? fx_to_odd(fx_r(i & 1 ? -v : v), un) : fx_to(fx_r(i & 1 ? -v : v), un);
        const double near = (double)exact;
        subnormal += near != 0.0 && std::fabs(near) < 2.2250738585072014e-308;
        if (std::isinf(near) ? got != near : fabsl(got - exact) != fabsl(near - exact)) ++bad;
    }
    std::printf("%ld %ld\n", bad, subnormal);
}

int main(int argc, char** argv) {
    const std::string what = argc > 1 ? argv[1] : "";
    if (what == "convert") {
        convert();
        return 0;
    }
    auto go = [&](const Plan& p) {
        if (what == "accuracy") accuracy(p);
        else if (what == "range") range(p);
        else zeros(p);
    };
    go(TwoStep<4, 4>());
    go(TwoStep<4, 8>());
    go(TwoStep<8, 8>());
    go(TwoStep<8, 16>());
    go(TwoStep<16, 16>());
    go(TwoStep<16, 32>());
    // the runtime engine: short plans, every radix last, the longest static plans, dynamic plans of
    // every first and last radix
    for (int L : {12, 18, 30, 48, 64, 90, 100, 120, 128, 192, 200, 256, 144, 150, 162, 180, 240, 250, 270, 288, 300, 320, 360, 384, 400,
                  432, 450, 480, 486, 500, 512})
        go(Runtime(L));
    return 0;
}
