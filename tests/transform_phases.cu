// Host run of the transform phases that the matvec and D-hat kernels are made
// of (the same source, compiled for the host): every two-radix plan against
// sums of roots of unity in long double, and the slab plans of every lattice.
//
// Prints one line per finding and exits non-zero when there is one.
#include <complex>
#include <cstdio>
#include <cstdlib>
#include <random>
#include <vector>

#include "dhat.cuh"
#include "slab.cuh"
#include "xline.cuh"

using namespace eels;
using Z = std::complex<long double>;
static int g_bad = 0;
static std::mt19937 g_rng(7);

static Z unit(int num, int L) {                    // exp(-2 pi i num / L)
    const long double a = -2.0L * 3.14159265358979323846264338327950288L * (num % L) / L;
    return {cosl(a), sinl(a)};
}
static Z rnd() {
    std::normal_distribution<double> d;
    const double re = (float)d(g_rng), im = (float)d(g_rng);   // exact in FP32
    return {re, im};
}
template <typename C> static C to_c(Z z) { return mk<C>((double)z.real(), (double)z.imag()); }
template <typename C> static Z to_z(C c) { return {(long double)c.x, (long double)c.y}; }
static std::vector<Z> dft(const std::vector<Z>& x, int L, bool inv) {
    std::vector<Z> w(L), y(L);
    for (int t = 0; t < L; ++t) w[t] = inv ? std::conj(unit(t, L)) : unit(t, L);
    for (int k = 0; k < L; ++k)
        for (int n = 0; n < (int)x.size(); ++n) y[k] += x[n] * w[k * n % L];
    return y;
}
// Relative 2-norm error of `steps` transforms of length L each: a radix step
// rounds every element a few times (butterfly levels, one twiddle), so 4 eps per
// level of log2 L bounds what the steps add.
struct Err {
    long double d = 0, n = 0;
    void add(Z got, Z want) { d += std::norm(got - want); n += std::norm(want); }
    void check(const char* what, int L, int n_in, double eps, int steps) const {
        const double e = (double)sqrtl(d / n), lim = 4.0 * eps * steps * (log2((double)L) + 1.0);
        if (!(e <= lim)) { printf("%s: L=%d n=%d: error %.2e above %.2e\n", what, L, n_in, e, lim); ++g_bad; }
    }
};
template <typename C> static std::vector<C> twiddles(const Plan2& p) {
    std::vector<C> w(p.L);
    for (int t = 0; t < p.L; ++t) w[t] = to_c<C>(unit((t / p.Re) * (t % p.Re), p.L));
    return w;
}

// Columns: forward y1, ymid and inverse ymid, y2i on ncol columns of n inputs.
template <typename Rl> static void slab_columns(int L, int n, int ncol, int nthr) {
    using C = cx<Rl>;
    const Plan2 p = make_plan2(L);
    const std::vector<C> tw = twiddles<C>(p);
    SlabCtx<Rl> s{};
    s.twy = tw.data();
    s.sls = ncol | 1;
    s.ncol = ncol;
    std::vector<C> S((size_t)L * s.sls, mk<C>(1e3, 1e3));
    s.S = S.data();
    std::vector<std::vector<Z>> x(ncol, std::vector<Z>(n));
    for (auto& c : x) for (Z& v : c) v = rnd();
    const FastDiv dcol = fast_div(ncol);
    const RtPlan rt{p};
    auto in = [&](int c, int y) { return to_c<C>(x[c][y]); };
    for (int t = 0; t < nthr; ++t) {
#define Y1(R) case R: slab_y1<R, Rl>(s, rt, dcol, n, t, nthr, in); break;
        EELS_SWITCH_RE(p.Re, Y1)
    }
    for (int t = 0; t < nthr; ++t) {
#define YM(R) case R: slab_ymid<R, false, Rl>(s, rt, dcol, t, nthr); break;
        EELS_SWITCH_RO(p.Ro, YM)
    }
    Err f, b;
    std::vector<std::vector<Z>> X(ncol);
    for (int c = 0; c < ncol; ++c) {
        X[c] = dft(x[c], L, false);
        for (int k = 0; k < L; ++k) f.add(to_z(S[(size_t)k * s.sls + c]), X[c][k]);
    }
    const double eps = sizeof(Rl) == 4 ? 5.97e-8 : 1.12e-16;
    f.check("columns forward", L, n, eps, 1);
    for (int t = 0; t < nthr; ++t) {
#define YI(R) case R: slab_ymid<R, true, Rl>(s, rt, dcol, t, nthr); break;
        EELS_SWITCH_RO(p.Ro, YI)
    }
    std::vector<int> seen((size_t)ncol * n, 0);
    auto out = [&](int c, int y, C v) { b.add(to_z(v), x[c][y] * (long double)L); ++seen[(size_t)c * n + y]; };
    for (int t = 0; t < nthr; ++t) {
#define Y2(R) case R: slab_y2i<R, Rl>(s, rt, dcol, n, t, nthr, out); break;
        EELS_SWITCH_RE(p.Re, Y2)
    }
    b.check("columns back", L, n, eps, 2);
    for (int v : seen) if (v != 1) { printf("columns back: L=%d n=%d: an output %d times\n", L, n, v); ++g_bad; break; }
}

// Rows: z1, z2 and z1i, z2i on g rows through the exchange tile.
template <typename Rl> static void slab_rows(int L, int n, int g) {
    using C = cx<Rl>;
    const Plan2 p = make_plan2(L);
    const std::vector<C> tw = twiddles<C>(p);
    std::vector<C> x((size_t)g * n), X((size_t)g * L), y((size_t)g * n), T((size_t)g * p.Ro * (p.Re + 1));
    for (C& v : x) v = to_c<C>(rnd());
    const RtPlan rt{p};
    auto in = [&](int q, int j, int dz) -> const C* { return &x[(size_t)q * n + j + dz]; };
    auto mid = [&](int q, int k) -> C* { return X.data() + (size_t)q * L + k; };
    auto out = [&](int q, int j, int dz) -> C* { return &y[(size_t)q * n + j + dz]; };
    for (int l = 0; l < 32; ++l) {
#define Z1(R) case R: slab_z1<R, C>(rt, n, g, T.data(), l, in); break;
        EELS_SWITCH_RE(p.Re, Z1)
    }
    for (int l = 0; l < 32; ++l) {
#define Z2(R) case R: slab_z2<R, C>(rt, g, T.data(), tw.data(), l, mid); break;
        EELS_SWITCH_RO(p.Ro, Z2)
    }
    const double eps = sizeof(Rl) == 4 ? 5.97e-8 : 1.12e-16;
    Err f, b;
    for (int q = 0; q < g; ++q) {
        std::vector<Z> xi(n);
        for (int i = 0; i < n; ++i) xi[i] = to_z(x[(size_t)q * n + i]);
        const std::vector<Z> w = dft(xi, L, false);
        for (int k = 0; k < L; ++k) f.add(to_z(X[(size_t)q * L + k]), w[k]);
    }
    f.check("rows forward", L, n, eps, 1);
    for (int l = 0; l < 32; ++l) {
#define Z1I(R) case R: slab_z1i<R, C>(rt, g, T.data(), tw.data(), l, mid); break;
        EELS_SWITCH_RO(p.Ro, Z1I)
    }
    for (int l = 0; l < 32; ++l) {
#define Z2I(R) case R: slab_z2i<R, C>(rt, n, g, T.data(), l, out); break;
        EELS_SWITCH_RE(p.Re, Z2I)
    }
    for (size_t i = 0; i < x.size(); ++i) b.add(to_z(y[i]), to_z(x[i]) * (long double)L);
    b.check("rows back", L, n, eps, 2);
}

// The x pass: transform, symmetric product per frequency, transform back.
template <typename Rl, int RE, int RO> static void x_lines(int n, int nw, int nthr, bool split) {
    using C = cx<Rl>;
    constexpr int L = RE * RO, lgw = 2, W = 1 << lgw;
    const std::vector<C> tw = twiddles<C>(make_plan2(L));
    std::vector<C> A((size_t)L * 3 * W), x((size_t)3 * W * n), y(x.size()), D((size_t)6 * L * W);
    for (C& v : x) v = to_c<C>(rnd());
    for (C& v : D) v = to_c<C>(rnd());
    auto at = [&](int c, int w, int i) { return ((size_t)c * W + w) * n + i; };
    for (int t = 0; t < nthr; ++t)
        xline_1<RE, RO>(A.data(), lgw, n, t, nthr, [&](int c, int w, int i) {
            return w < nw ? x[at(c, w, i)] : mk<C>(0.0, 0.0);
        });
    if (split) {
        for (int w = 0; w < nw; ++w)
            for (int j = 0; j < RE; ++j) {
                C v[3][RO], u[3][RO];
                auto row = [&](int c) { return A.data() + j * 3 * W + c * W + w; };
                for (int c = 0; c < 3; ++c) xline_mid_in<RE, RO>(row(c), 3 * W, tw.data() + j, v[c]);
                for (int c = 0; c < 3; ++c)
                    for (int r = 0; r < RO; ++r) {
                        auto g = [&](int i) { return D[((size_t)i * L + j + r * RE) * W + w]; };
                        u[c][r] = g(sym_own(c)) * v[c][r] + g(sym_next(c)) * v[(c + 1) % 3][r] +
                                  g(sym_prev(c)) * v[(c + 2) % 3][r];
                    }
                for (int c = 0; c < 3; ++c) xline_mid_out<RE, RO>(row(c), 3 * W, tw.data() + j, u[c]);
            }
    } else {
        for (int t = 0; t < nthr; ++t)
            xline_mid<RE, RO>(A.data(), lgw, nw, tw.data(), t, nthr, [&](int w, int k, C (&g)[6]) {
                for (int c = 0; c < 6; ++c) g[c] = D[((size_t)c * L + k) * W + w];
            });
    }
    for (int t = 0; t < nthr; ++t)
        xline_2<RE, RO>(A.data(), lgw, n, t, nthr, [&](int c, int w, int i, C v) { if (w < nw) y[at(c, w, i)] = v; });
    const int sym[3][3] = {{0, 1, 2}, {1, 3, 4}, {2, 4, 5}};
    Err e;
    for (int w = 0; w < nw; ++w) {
        std::vector<Z> X[3];
        for (int c = 0; c < 3; ++c) {
            std::vector<Z> xi(n);
            for (int i = 0; i < n; ++i) xi[i] = to_z(x[at(c, w, i)]);
            X[c] = dft(xi, L, false);
        }
        for (int c = 0; c < 3; ++c) {
            std::vector<Z> P(L);
            for (int k = 0; k < L; ++k)
                for (int d = 0; d < 3; ++d) P[k] += to_z(D[((size_t)sym[c][d] * L + k) * W + w]) * X[d][k];
            const std::vector<Z> r = dft(P, L, true);
            for (int i = 0; i < n; ++i) e.add(to_z(y[at(c, w, i)]), r[i]);
        }
    }
    // the outputs wanted are a part of the inverse transform whose whole carries the rounding: sqrt(L / n) more
    const double eps = sizeof(Rl) == 4 ? 5.97e-8 : 1.12e-16;
    e.check("x lines", L, n, eps * std::sqrt((double)L / n), 3);
}

// One axis of the D-hat build: an even or odd sequence from its octant.
template <int RE, int RO> static void dhat_line(int n, bool odd, int nthr) {
    constexpr int L = RE * RO, W = 3, ES = 4;
    const std::vector<double2> tw = twiddles<double2>(make_plan2(L));   // the rows j <= RO/2 are read
    constexpr int rows = DhatLine<RE, RO>::ROWS;
    std::vector<double2> A((size_t)rows * ES), F_((size_t)(L / 2 + 1) * W);
    std::vector<int> seen(F_.size(), 0);
    std::vector<std::vector<Z>> g(W, std::vector<Z>(n));
    for (auto& l : g) for (Z& v : l) v = rnd();
    if (odd) for (auto& l : g) l[0] = 0;
    for (int t = 0; t < nthr; ++t)
        dhat_1<RE, RO>(A.data(), ES, W, n, odd, t, nthr, [&](int w, int i) { return to_c<double2>(g[w][i]); });
    for (int t = 0; t < nthr; ++t)
        dhat_2<RE, RO>(A.data(), ES, W, odd, tw.data(), t, nthr, [&](int w, int k, double2 v) {
            F_[(size_t)k * W + w] = v;
            ++seen[(size_t)k * W + w];
        });
    for (int v : seen) if (v != 1) { printf("D-hat: L=%d: an output %d times\n", L, v); ++g_bad; break; }
    Err e;
    for (int w = 0; w < W; ++w) {
        std::vector<Z> full(L);
        for (int i = 0; i < n; ++i) {
            full[i] += g[w][i];
            if (i) full[L - i] += odd ? -g[w][i] : g[w][i];
        }
        const std::vector<Z> F = dft(full, L, false);
        for (int k = 0; k <= L / 2; ++k) e.add(to_z(F_[(size_t)k * W + w]), F[k]);
    }
    // an odd line of one entry vanishes
    if (e.n > 0) e.check(odd ? "D-hat odd" : "D-hat even", L, n, 1.12e-16, 2);
}

template <int RE, int RO> static void one_length() {
    constexpr int L = RE * RO;
    // the lattice extents that are padded to L, and a short one
    for (int n : {(L + 1) / 2, L / 2 - 1, 1}) {
        if (n < 1 || 2 * n - 1 > L) continue;
        slab_columns<float>(L, n, 5, 64); slab_columns<double>(L, n, 1, 96);
        slab_rows<float>(L, n, 3); slab_rows<double>(L, n, 1);
        x_lines<float, RE, RO>(n, 4, 64, false); x_lines<double, RE, RO>(n, 3, 96, false); x_lines<double, RE, RO>(n, 3, 64, true);
        if (2 * n <= L) { dhat_line<RE, RO>(n, false, 64); dhat_line<RE, RO>(n, true, 64); }
    }
}

static void slab_plans() {
    std::vector<int> lens;
#define LEN(RE, RO) lens.push_back(RE * RO);
    EELS_PLANS(LEN)
    for (int My : lens)
        for (int Mz : lens)
            for (int less : {0, 1}) {
                LatticeDev L{};
                L.My = My; L.Mz = Mz;
                L.Ny = My / 2 > 1 ? My / 2 - less : 1;
                L.Nz = Mz / 2 > 1 ? Mz / 2 - less : 1;
                L.qy = make_plan2(My); L.qz = make_plan2(Mz);
                for (size_t el : {sizeof(float2), sizeof(double2)}) {
                    const SlabPlan p = make_slab_plan(L, el);
                    const bool ok = p.nthr >= 64 && p.nthr % 32 == 0 && p.nthr <= (el == 8 ? 768 : 512) && p.G >= 1 &&
                                    p.CL >= 1 && p.CL <= 8 && p.CL * p.cpc >= L.Nz && p.CL * p.rpc >= My &&
                                    p.sls >= p.cpc && slab_smem(L, p, el) <= 224 * 1024;
                    if (!ok) { printf("slab plan: My=%d Mz=%d el=%zu\n", My, Mz, el); ++g_bad; }
                }
            }
}

static void divisions() {
    for (int d = 1; d <= 256; ++d) {
        const FastDiv f = fast_div(d);
        for (unsigned n = 0; n < 65536; ++n)
            if (f.div(n) != n / d) { printf("division: %u / %d\n", n, d); ++g_bad; break; }
    }
}

int main() {
    divisions();
    slab_plans();
#define ONE(RE, RO) one_length<RE, RO>();
    EELS_PLANS(ONE)
    printf("%d findings\n", g_bad);
    return g_bad ? 1 : 0;
}
