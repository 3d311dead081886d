// Length-R DFTs in registers, R <= 25, and the two-radix plan of a line.
//
// A line of L = Re * Ro points (Re even) is transformed in two register
// steps with one exchange between them:
//   forward   step 1: for j < Ro, a length-Re DFT over the inputs j + r Ro
//             (r < Re), its output r kept at place r of set j;
//             step 2: for j < Re, a length-Ro DFT over the places j of the
//             sets r < Ro, input r times w^(r j), w = exp(-2 pi i / L): its
//             output r is element j + r Re of the transform;
//   inverse   step 1: for j < Re, a length-Ro DFT over the elements j + r Re,
//             output r times conj(w^(r j)), kept at place j of set r;
//             step 2: for j < Ro, a length-Re DFT over set j: its output r is
//             element j + r Ro (unnormalised).
// Step 2 forward and step 1 inverse read and write the same places, so they
// run in place.  A lattice of N cells is padded to L >= 2N, L even: only the
// first half of a line holds inputs, and only the first half of an inverse
// transform is wanted.  Step 1 forward therefore takes inputs r < Re/2 only
// (dft_hin) and step 2 inverse forms outputs r < Re/2 only (dft_hout).
//
// Composite lengths use the prime-factor map (Good 1958, Thomas 1963) where
// the factors are coprime (no twiddles), else one Cooley-Tukey step.
#pragma once
#include "common.cuh"

namespace eels {

#define HD __host__ __device__ __forceinline__

// sqrt(1/2), cos/sin(2 pi/3), and the R = 5, 7 roots of unity (values of
// elementary closed forms, e.g. cos(2 pi/5) = (sqrt 5 - 1)/4).
#define K_SQRT_HALF 0.70710678118654752440
#define K_C3 (-0.5)
#define K_S3 0.86602540378443864676
#define K_C5_1 0.30901699437494742410
#define K_S5_1 0.95105651629515357212
#define K_C5_2 (-0.80901699437494742410)
#define K_S5_2 0.58778525229247312917
#define K_C7_1 0.62348980185873353053
#define K_S7_1 0.78183148246802980871
#define K_C7_2 (-0.22252093395631440429)
#define K_S7_2 0.97492791218182360702
#define K_C7_3 (-0.90096886790241912624)
#define K_S7_3 0.43388373911755812048

// cos and sin of 2 pi k / N for the lengths whose twiddles are compiled in
// (k < N; after unrolling k is a constant and so is the result).
template <int N> HD double cos_2pi(int k);
template <> HD double cos_2pi<2>(int k) { return k ? -1.0 : 1.0; }
template <> HD double cos_2pi<4>(int k) { const double c[4] = {1, 0, -1, 0}; return c[k]; }
template <> HD double cos_2pi<6>(int k) { const double c[6] = {1, 0.5, -0.5, -1, -0.5, 0.5}; return c[k]; }
template <> HD double cos_2pi<8>(int k) {
    const double h = K_SQRT_HALF, c[8] = {1, h, 0, -h, -1, -h, 0, h};
    return c[k];
}
template <> HD double cos_2pi<9>(int k) {
    const double a = 0.766044443118978035202, b = 0.173648177666930348852, d = -0.939692620785908384054,
                 c[9] = {1, a, b, -0.5, d, d, -0.5, b, a};
    return c[k];
}
template <> HD double cos_2pi<10>(int k) {
    const double a = -K_C5_2, b = K_C5_1, c[10] = {1, a, b, -b, -a, -1, -a, -b, b, a};
    return c[k];
}
template <> HD double cos_2pi<12>(int k) {
    const double a = K_S3, c[12] = {1, a, 0.5, 0, -0.5, -a, -1, -a, -0.5, 0, 0.5, a};
    return c[k];
}
template <> HD double cos_2pi<14>(int k) {
    const double a = -K_C7_3, b = K_C7_1, d = -K_C7_2, c[14] = {1, a, b, d, -d, -b, -a, -1, -a, -b, -d, d, b, a};
    return c[k];
}
template <> HD double cos_2pi<16>(int k) {
    const double a = 0.923879532511286756128, h = K_SQRT_HALF, b = 0.382683432365089771728,
                 c[16] = {1, a, h, b, 0, -b, -h, -a, -1, -a, -h, -b, 0, b, h, a};
    return c[k];
}
template <> HD double cos_2pi<18>(int k) {
    const double a = 0.939692620785908384054, b = 0.766044443118978035202, d = 0.173648177666930348852,
                 c[18] = {1, a, b, 0.5, d, -d, -0.5, -b, -a, -1, -a, -b, -0.5, -d, d, 0.5, b, a};
    return c[k];
}
template <> HD double cos_2pi<20>(int k) {
    const double a = K_S5_1, b = -K_C5_2, d = K_S5_2, e = K_C5_1,
                 c[20] = {1, a, b, d, e, 0, -e, -d, -b, -a, -1, -a, -b, -d, -e, 0, e, d, b, a};
    return c[k];
}
template <> HD double cos_2pi<25>(int k) {
    const double c[25] = {1, 0.968583161128631119490, 0.876306680043863587308, 0.728968627421411523147,
                          0.535826794978996618271, K_C5_1, 0.0627905195293133760762, -0.187381314585724630543,
                          -0.425779291565072648863, -0.637423989748689710177, K_C5_2, -0.929776485888251403660,
                          -0.992114701314477831049, -0.992114701314477831049, -0.929776485888251403660, K_C5_2,
                          -0.637423989748689710177, -0.425779291565072648863, -0.187381314585724630543,
                          0.0627905195293133760762, K_C5_1, 0.535826794978996618271, 0.728968627421411523147,
                          0.876306680043863587308, 0.968583161128631119490};
    return c[k];
}
template <int N> HD double sin_2pi(int k);
// sin(2 pi k / N) = cos(2 pi (k - N/4) / N) where 4 divides N
template <> HD double sin_2pi<2>(int) { return 0.0; }
template <> HD double sin_2pi<4>(int k) { return cos_2pi<4>((k + 3) % 4); }
template <> HD double sin_2pi<6>(int k) { const double s = K_S3, c[6] = {0, s, s, 0, -s, -s}; return c[k]; }
template <> HD double sin_2pi<8>(int k) { return cos_2pi<8>((k + 6) % 8); }
template <> HD double sin_2pi<9>(int k) {
    const double a = 0.642787609686539326323, b = 0.984807753012208059367, d = 0.342020143325668733044, s = K_S3,
                 c[9] = {0, a, b, s, d, -d, -s, -b, -a};
    return c[k];
}
template <> HD double sin_2pi<10>(int k) {
    const double a = K_S5_2, b = K_S5_1, c[10] = {0, a, b, b, a, 0, -a, -b, -b, -a};
    return c[k];
}
template <> HD double sin_2pi<12>(int k) { return cos_2pi<12>((k + 9) % 12); }
template <> HD double sin_2pi<14>(int k) {
    const double a = K_S7_3, b = K_S7_1, d = K_S7_2, c[14] = {0, a, b, d, d, b, a, 0, -a, -b, -d, -d, -b, -a};
    return c[k];
}
template <> HD double sin_2pi<16>(int k) { return cos_2pi<16>((k + 12) % 16); }
template <> HD double sin_2pi<18>(int k) {
    const double a = 0.342020143325668733044, b = 0.642787609686539326323, s = K_S3, d = 0.984807753012208059367,
                 c[18] = {0, a, b, s, d, d, s, b, a, 0, -a, -b, -s, -d, -d, -s, -b, -a};
    return c[k];
}
template <> HD double sin_2pi<20>(int k) { return cos_2pi<20>((k + 15) % 20); }

// x times exp(-+2 pi i k / N), k a constant after unrolling (the trivial
// angles cost no multiplication).
template <bool INV, typename C> HD C rot_mi(C a) { return INV ? mul_i(a) : mul_mi(a); }   // * exp(-+ i pi/2)
template <int N, bool INV, typename C> HD C rot_w(C x, int k) {
    using Rl = decltype(x.x);
    k %= N;
    if (k == 0) return x;
    if (4 * k == N) return rot_mi<INV>(x);
    if (2 * k == N) return -x;
    if (4 * k == 3 * N) return -rot_mi<INV>(x);
    const Rl c = (Rl)cos_2pi<N>(k), s = (Rl)(INV ? sin_2pi<N>(k) : -sin_2pi<N>(k));
    C r;
    r.x = x.x * c - x.y * s;
    r.y = x.x * s + x.y * c;
    return r;
}

// Length-R DFT in registers.  INV=false: X_p = sum_q v_q exp(-2 pi i p q / R).
template <int R, bool INV, typename C> struct Dft;

template <bool INV, typename C> struct Dft<1, INV, C> {
    HD static void run(C*) {}
};
template <bool INV, typename C> struct Dft<2, INV, C> {
    HD static void run(C* v) { C a = v[0], b = v[1]; v[0] = a + b; v[1] = a - b; }
};
template <bool INV, typename C> struct Dft<3, INV, C> {
    HD static void run(C* v) {
        using Rl = decltype(v[0].x);
        const Rl c = (Rl)K_C3, s = (Rl)(INV ? -K_S3 : K_S3);
        C a = v[1] + v[2], b = v[1] - v[2];
        const C m = fma_s(c, a, v[0]), jb = mul_mi(b);   // +- s (-i b)
        v[0] = v[0] + a;
        v[1] = fma_s(s, jb, m);
        v[2] = fma_s(-s, jb, m);
    }
};
template <bool INV, typename C> struct Dft<4, INV, C> {
    HD static void run(C* v) {
        C s0 = v[0] + v[2], d0 = v[0] - v[2];
        C s1 = v[1] + v[3], d1 = rot_mi<INV>(v[1] - v[3]);
        v[0] = s0 + s1; v[2] = s0 - s1;
        v[1] = d0 + d1; v[3] = d0 - d1;
    }
};
template <bool INV, typename C> struct Dft<8, INV, C> {
    HD static void run(C* v) {
        using Rl = decltype(v[0].x);
        const Rl h = (Rl)K_SQRT_HALF;
        C e[4] = {v[0], v[2], v[4], v[6]};
        C o[4] = {v[1], v[3], v[5], v[7]};
        Dft<4, INV, C>::run(e);
        Dft<4, INV, C>::run(o);
        // twiddles exp(-+ 2 pi i p / 8), p = 1, 2, 3: h (1 -+ i), -+i, -h (1 +- i)
        C w1, w3;
        if (!INV) {
            w1.x = o[1].x + o[1].y; w1.y = o[1].y - o[1].x;
            w3.x = o[3].y - o[3].x; w3.y = -o[3].x - o[3].y;
        } else {
            w1.x = o[1].x - o[1].y; w1.y = o[1].y + o[1].x;
            w3.x = -o[3].x - o[3].y; w3.y = o[3].x - o[3].y;
        }
        const C t2 = rot_mi<INV>(o[2]);
        v[0] = e[0] + o[0]; v[4] = e[0] - o[0];
        v[1] = fma_s(h, w1, e[1]); v[5] = fma_s(-h, w1, e[1]);
        v[2] = e[2] + t2;   v[6] = e[2] - t2;
        v[3] = fma_s(h, w3, e[3]); v[7] = fma_s(-h, w3, e[3]);
    }
};

// Odd lengths 5 and 7 from symmetric pairs:
// X_p = v0 + sum_{q=1}^{(R-1)/2} [ (v_q + v_{R-q}) cos(2 pi p q/R) -+ i (v_q - v_{R-q}) sin(2 pi p q/R) ]
template <int R, bool INV, typename C> struct DftOdd {
    HD static void run(C* v, const double* cs, const double* sn) {
        using Rl = decltype(v[0].x);
        constexpr int H = (R - 1) / 2;
        C sp[H], sm[H];
#pragma unroll
        for (int q = 1; q <= H; ++q) { sp[q - 1] = v[q] + v[R - q]; sm[q - 1] = v[q] - v[R - q]; }
        const C v0 = v[0];
        C x0 = v0;
#pragma unroll
        for (int q = 0; q < H; ++q) x0 = x0 + sp[q];
        v[0] = x0;
#pragma unroll
        for (int p = 1; p <= H; ++p) {
            C re = fma_s((Rl)cs[p], sp[0], v0), im = (Rl)sn[p] * sm[0];
#pragma unroll
            for (int q = 2; q <= H; ++q) {
                re = fma_s((Rl)cs[(p * q) % R], sp[q - 1], re);
                im = fma_s((Rl)sn[(p * q) % R], sm[q - 1], im);
            }
            const C jim = INV ? mul_i(im) : mul_mi(im);   // forward: -i im; inverse: +i im
            v[p] = re + jim;
            v[R - p] = re - jim;
        }
    }
};
template <bool INV, typename C> struct Dft<5, INV, C> {
    HD static void run(C* v) {
        const double cs[5] = {1.0, K_C5_1, K_C5_2, K_C5_2, K_C5_1};
        const double sn[5] = {0.0, K_S5_1, K_S5_2, -K_S5_2, -K_S5_1};
        DftOdd<5, INV, C>::run(v, cs, sn);
    }
};
template <bool INV, typename C> struct Dft<7, INV, C> {
    HD static void run(C* v) {
        const double cs[7] = {1.0, K_C7_1, K_C7_2, K_C7_3, K_C7_3, K_C7_2, K_C7_1};
        const double sn[7] = {0.0, K_S7_1, K_S7_2, K_S7_3, -K_S7_3, -K_S7_2, -K_S7_1};
        DftOdd<7, INV, C>::run(v, cs, sn);
    }
};

// a with a b = 1 mod m (m small)
__host__ __device__ constexpr int inv_mod(int b, int m) {
    for (int a = 0; a < m; ++a)
        if ((a * b) % m == 1 % m) return a;
    return 0;
}

// R = A B, coprime: input n = B n1 + A n2, output k = B (B^-1 mod A) k1 + A (A^-1 mod B) k2 (mod R).
template <int A, int B, bool INV, typename C> struct DftPfa {
    HD static void run(C* v) {
        constexpr int R = A * B, EA = B * inv_mod(B, A), EB = A * inv_mod(A, B);
        C t[A][B];
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) {
#pragma unroll
            for (int n2 = 0; n2 < B; ++n2) t[n1][n2] = v[(B * n1 + A * n2) % R];
            Dft<B, INV, C>::run(t[n1]);
        }
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) {
            C u[A];
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) u[n1] = t[n1][k2];
            Dft<A, INV, C>::run(u);
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1) v[(EA * k1 + EB * k2) % R] = u[k1];
        }
    }
};
// R = A B by one Cooley-Tukey step: n = n1 + A n2, k = k2 + B k1.
template <int A, int B, bool INV, typename C> struct DftCt {
    HD static void run(C* v) {
        constexpr int R = A * B;
        C t[A][B];
#pragma unroll
        for (int n1 = 0; n1 < A; ++n1) {
#pragma unroll
            for (int n2 = 0; n2 < B; ++n2) t[n1][n2] = v[n1 + A * n2];
            Dft<B, INV, C>::run(t[n1]);
        }
#pragma unroll
        for (int k2 = 0; k2 < B; ++k2) {
            C u[A];
#pragma unroll
            for (int n1 = 0; n1 < A; ++n1) u[n1] = rot_w<R, INV>(t[n1][k2], n1 * k2);
            Dft<A, INV, C>::run(u);
#pragma unroll
            for (int k1 = 0; k1 < A; ++k1) v[k2 + B * k1] = u[k1];
        }
    }
};
template <bool INV, typename C> struct Dft<6, INV, C> : DftPfa<2, 3, INV, C> {};
template <bool INV, typename C> struct Dft<9, INV, C> : DftCt<3, 3, INV, C> {};
template <bool INV, typename C> struct Dft<10, INV, C> : DftPfa<2, 5, INV, C> {};
template <bool INV, typename C> struct Dft<12, INV, C> : DftPfa<3, 4, INV, C> {};
template <bool INV, typename C> struct Dft<14, INV, C> : DftPfa<2, 7, INV, C> {};
template <bool INV, typename C> struct Dft<15, INV, C> : DftPfa<3, 5, INV, C> {};
template <bool INV, typename C> struct Dft<16, INV, C> : DftCt<4, 4, INV, C> {};
template <bool INV, typename C> struct Dft<18, INV, C> : DftPfa<2, 9, INV, C> {};
template <bool INV, typename C> struct Dft<20, INV, C> : DftPfa<4, 5, INV, C> {};
template <> HD double sin_2pi<25>(int k) {
    const double c[13] = {0, 0.248689887164854788243, 0.481753674101715274987, 0.684547105928688673732,
                          0.844327925502015078549, K_S5_1, 0.998026728428271561952, 0.982287250728688681085,
                          0.904827052466019527713, 0.770513242775789230803, K_S5_2, 0.368124552684677959157,
                          0.125333233564304245373};
    return k < 13 ? c[k] : -c[25 - k];
}
// Length 25 occurs in one plan only (250 points): a call on a local array, so
// that its 50 registers do not set the register count of every kernel.
template <bool INV, typename C> struct Dft<25, INV, C> {
    __host__ __device__ __noinline__ static void run(C* v) { DftCt<5, 5, INV, C>::run(v); }
};

// Length-R DFT (R even) of inputs v[0..R/2); v[R/2..R) are zero and not read:
// X_{2k} = DFT_{R/2}(v), X_{2k+1} = DFT_{R/2}(v_q w^q).
template <int R, bool INV, typename C> HD void dft_hin(C (&v)[R]) {
    constexpr int H = R / 2;
    C e[H], o[H];
#pragma unroll
    for (int q = 0; q < H; ++q) { e[q] = v[q]; o[q] = rot_w<R, INV>(v[q], q); }
    Dft<H, INV, C>::run(e);
    Dft<H, INV, C>::run(o);
#pragma unroll
    for (int q = 0; q < H; ++q) { v[2 * q] = e[q]; v[2 * q + 1] = o[q]; }
}
// The first R/2 outputs (R even): X_k = E_k + w^k O_k with E, O the DFTs of
// the even and odd inputs.
template <int R, bool INV, typename C> HD void dft_hout(C (&v)[R]) {
    constexpr int H = R / 2;
    C e[H], o[H];
#pragma unroll
    for (int q = 0; q < H; ++q) { e[q] = v[2 * q]; o[q] = v[2 * q + 1]; }
    Dft<H, INV, C>::run(e);
    Dft<H, INV, C>::run(o);
#pragma unroll
    for (int q = 0; q < H; ++q) v[q] = e[q] + rot_w<R, INV>(o[q], q);
}

// Division of n < 65536 by a run-time d: n / d = umulhi(n, ceil(2^32 / d)).
struct FastDiv {
    unsigned d, m;
    HD unsigned div(unsigned n) const {
#ifdef __CUDA_ARCH__
        return d == 1 ? n : __umulhi(n, m);
#else
        return d == 1 ? n : (unsigned)(((unsigned long long)n * m) >> 32);
#endif
    }
};
HD FastDiv fast_div(int d) { return FastDiv{(unsigned)d, d <= 1 ? 0u : 0xffffffffu / (unsigned)d + 1u}; }

// Plan of one axis: L = Re * Ro, Re even.
struct Plan2 {
    int L, Re, Ro;
    FastDiv dRe, dRo;
};

// The plan (Re, Ro) of every padded length (the even 7-smooth numbers up to
// 256): the pair of the radices below with the smallest max(2 Re, 3 Ro), because
// a thread of the x pass holds three lines in its middle step.  Ro = 2 is not
// among them: it would serve L = 4 and 8 alone, (2, 2) and (4, 2), whose passes
// take no longer than their launches.
#define EELS_PLANS(X) \
    X(2, 1) X(4, 1) X(2, 3) X(2, 4) X(2, 5) X(4, 3) X(2, 7) X(4, 4) X(6, 3) X(4, 5) X(6, 4) X(4, 7) X(6, 5) \
    X(8, 4) X(6, 6) X(8, 5) X(6, 7) X(8, 6) X(10, 5) X(6, 9) X(8, 7) X(10, 6) X(8, 8) X(10, 7) X(12, 6) \
    X(10, 8) X(12, 7) X(10, 9) X(12, 8) X(14, 7) X(10, 10) X(12, 9) X(14, 8) X(12, 10) X(14, 9) X(16, 8) \
    X(14, 10) X(16, 9) X(10, 15) X(16, 10) X(18, 9) X(14, 12) X(18, 10) X(16, 12) X(14, 14) X(20, 10) \
    X(14, 15) X(18, 12) X(16, 14) X(20, 12) X(10, 25) X(18, 14) X(16, 16)

// The radices that occur in them: Re runs step 1 forward and step 2 inverse,
// Ro the middle.
#define EELS_RE_LIST(X) X(2) X(4) X(6) X(8) X(10) X(12) X(14) X(16) X(18) X(20)
#define EELS_RO_LIST(X) X(1) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(12) X(14) X(15) X(16) X(25)

}  // namespace eels
