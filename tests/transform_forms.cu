// Host run of the forms of the slab phases that transform_phases.cu leaves out,
// against the ones it compares with sums of roots of unity: the compiled-in plans,
// and rows shared by a whole block.  The arithmetic is the same statement for
// statement, and the host rounds every operation by itself, so the bits have to be
// the same.  Also how full the FP64 slab plans keep the lanes of their z transforms.
//
// Prints one line per finding and exits non-zero when there is one.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "slab.cuh"

using namespace eels;
static int g_bad = 0;
static std::mt19937 g_rng(11);

template <typename C> static C rnd() {
    std::normal_distribution<double> d;
    const double re = d(g_rng), im = d(g_rng);
    return mk<C>(re, im);
}
template <typename C> static std::vector<C> twiddles(int RE, int RO) {
    std::vector<C> w(RE * RO);
    for (int t = 0; t < RE * RO; ++t) {
        const double a = -2.0 * 3.14159265358979323846 * ((t / RE) * (t % RE)) / (RE * RO);
        w[t] = mk<C>(cos(a), sin(a));
    }
    return w;
}
template <typename C> static void same(const char* what, int L, const std::vector<C>& a, const std::vector<C>& b) {
    if (a.size() == b.size() && std::memcmp(a.data(), b.data(), a.size() * sizeof(C)) == 0) return;
    printf("%s: L=%d differs\n", what, L);
    ++g_bad;
}

// All four phases of ncol columns; the results of both directions.
template <typename Rl, int RE, int RO, class P> static std::vector<cx<Rl>> columns(P p, const std::vector<cx<Rl>>& x, int n, int ncol, int nthr) {
    using C = cx<Rl>;
    constexpr int L = RE * RO;
    const std::vector<C> tw = twiddles<C>(RE, RO);
    SlabCtx<Rl> s{};
    s.twy = tw.data();
    s.sls = ncol | 1;
    s.ncol = ncol;
    std::vector<C> S((size_t)L * s.sls, mk<C>(0.0, 0.0)), y((size_t)ncol * n, mk<C>(0.0, 0.0));
    s.S = S.data();
    const FastDiv dcol = fast_div(ncol);
    auto in = [&](int c, int i) { return x[(size_t)c * n + i]; };
    auto out = [&](int c, int i, C v) { y[(size_t)c * n + i] = v; };
    for (int t = 0; t < nthr; ++t) slab_y1<RE, Rl>(s, p, dcol, n, t, nthr, in);
    for (int t = 0; t < nthr; ++t) slab_ymid<RO, false, Rl>(s, p, dcol, t, nthr);
    std::vector<C> r = S;
    for (int t = 0; t < nthr; ++t) slab_ymid<RO, true, Rl>(s, p, dcol, t, nthr);
    for (int t = 0; t < nthr; ++t) slab_y2i<RE, Rl>(s, p, dcol, n, t, nthr, out);
    r.insert(r.end(), y.begin(), y.end());
    return r;
}
// All four phases of g rows, shared by nl lanes.
template <typename Rl, int RE, int RO, class P> static std::vector<cx<Rl>> rows(P p, const std::vector<cx<Rl>>& x, int n, int g, int nl) {
    using C = cx<Rl>;
    constexpr int L = RE * RO;
    const std::vector<C> tw = twiddles<C>(RE, RO);
    std::vector<C> X((size_t)g * L), y((size_t)g * n), T((size_t)g * RO * (RE + 1));
    auto in = [&](int q, int j, int dz) -> const C* { return &x[(size_t)q * n + j + dz]; };
    auto mid = [&](int q, int k) -> C* { return X.data() + (size_t)q * L + k; };
    auto out = [&](int q, int j, int dz) -> C* { return &y[(size_t)q * n + j + dz]; };
    for (int l = 0; l < nl; ++l) slab_z1<RE, C>(p, n, g, T.data(), l, in, nl);
    for (int l = 0; l < nl; ++l) slab_z2<RO, C>(p, g, T.data(), tw.data(), l, mid, nl);
    std::vector<C> r = X;
    for (int l = 0; l < nl; ++l) slab_z1i<RO, C>(p, g, T.data(), tw.data(), l, mid, nl);
    for (int l = 0; l < nl; ++l) slab_z2i<RE, C>(p, n, g, T.data(), l, out, nl);
    r.insert(r.end(), y.begin(), y.end());
    return r;
}
template <typename Rl, int RE, int RO> static void one_length() {
    using C = cx<Rl>;
    constexpr int L = RE * RO;
    const Plan2 p = make_plan2(L);
    if (p.Re != RE || p.Ro != RO) { printf("plan of L=%d\n", L); ++g_bad; return; }
    for (int n : {L / 2, 1}) {
        std::vector<C> x((size_t)24 * n);
        for (C& v : x) v = rnd<C>();
        same("columns", L, columns<Rl, RE, RO>(RtPlan{p}, x, n, 5, 64), columns<Rl, RE, RO>(CtPlan<RE, RO>{}, x, n, 5, 96));
        const std::vector<C> r = rows<Rl, RE, RO>(RtPlan{p}, x, n, 24, 32);
        same("rows", L, r, rows<Rl, RE, RO>(CtPlan<RE, RO>{}, x, n, 24, 32));
        same("rows of a block", L, r, rows<Rl, RE, RO>(RtPlan{p}, x, n, 24, 256));
        same("rows of a block", L, r, rows<Rl, RE, RO>(CtPlan<RE, RO>{}, x, n, 24, 192));
    }
}

// Of the lanes of the FP64 z instructions that a slab issues, at least 60 % have a
// butterfly (lines of 32 points and more; a line's radices leave 20 % idle at the
// worst of full turns).
static void lanes() {
    std::vector<int> lens;
#define LEN(RE, RO) lens.push_back(RE * RO);
    EELS_PLANS(LEN)
    auto up = [](int a, int b) { return (a + b - 1) / b; };
    for (int My : lens)
        for (int Mz : lens)
            for (int Nx : {1, 12, 64}) {
                if (My < 32 || Mz < 32) continue;
                LatticeDev L{};
                L.Nx = Nx; L.My = My; L.Mz = Mz; L.Ny = My / 2; L.Nz = Mz / 2;
                L.qy = make_plan2(My); L.qz = make_plan2(Mz);
                const SlabPlan p = make_slab_plan(L, sizeof(double2));
                const int Re = L.qz.Re, Ro = L.qz.Ro, turn = p.wide ? p.G * p.nthr / 32 : p.G;
                double used = 0, issued = 0;
                for (int row = 0; row < p.rpc; row += turn) {
                    const int g = std::min(turn, p.rpc - row);
                    used += 2.0 * g * Re * Ro;
                    issued += 32.0 * (up(g * Ro, 32) * Re + up(g * Re, 32) * Ro);
                }
                if (used < 0.6 * issued || slab_smem(L, p, sizeof(double2)) > 224 * 1024) {
                    printf("Nx=%d My=%d Mz=%d: %.0f %% of the lanes of the z transforms\n", Nx, My, Mz,
                           100 * used / issued);
                    ++g_bad;
                }
            }
}

int main() {
    lanes();
#define ONE(RE, RO) one_length<float, RE, RO>(); one_length<double, RE, RO>();
    EELS_PLANS(ONE)
    printf("%d findings\n", g_bad);
    return g_bad ? 1 : 0;
}
