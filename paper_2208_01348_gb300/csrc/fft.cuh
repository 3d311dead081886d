// Shared-memory mixed-radix FFT core (radices 2, 3, 4, 5, 7, 8).
//
// Stockham auto-sort formulation (decimation in time, out of place between
// two shared-memory buffers): at a stage of radix R, with Ns the length of
// the sub-transforms already done, butterfly j (0 <= j < L/R) reads the R
// inputs a[j + r L/R], multiplies input r by w^(r k), k = j mod Ns,
// w = exp(-+2 pi i / (Ns R)), takes a length-R DFT and writes output r to
// b[(j / Ns) Ns R + k + r Ns].  After all stages the result is in natural
// order.  Forward uses exp(-2 pi i n k / L); the inverse is unnormalised.
//
// A batch of NL lines is transformed together: element i of line l lives at
// buf[l * lstride + i * estride], so the same routine serves lines stored
// contiguously (estride = 1) and lines interleaved across a tile
// (lstride = 1).  Twiddles come from a table tw[t] = exp(-2 pi i t / L).
#pragma once
#include "dft.cuh"

namespace eels {

#define FFT_MAX_STAGES 12
#define FFT_MAX_LEN 512

// One Stockham stage: radix R after sub-transforms of length Ns; nb = L/R
// butterflies per line; ts = L/(Ns R) is the twiddle-table stride.  The
// shifts are log2 of Ns and nb when those are powers of two (else -1), so
// the index arithmetic of the common power-of-two lengths avoids divisions.
struct FftStage {
    int R, Ns, ns_shift, nb, nb_shift, ts;
};

struct FftPlan {
    int L;
    int nst;
    FftStage st[FFT_MAX_STAGES];
};

// One Stockham stage of radix R over NL lines.  LINE_FAST: adjacent
// threads take adjacent lines (good when lstride == 1).
template <int R, bool INV, bool LINE_FAST, int NL, typename C>
__device__ __forceinline__ void fft_stage(const C* __restrict__ a, C* __restrict__ b, int lstride, int estride,
                                          const FftStage sd, const C* __restrict__ tw) {
    const int nb = sd.nb, Ns = sd.Ns;
    const int total = NL * nb;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        int line, j;
        if (LINE_FAST) {
            line = t % NL;
            j = t / NL;
        } else if (sd.nb_shift >= 0) {
            j = t & (nb - 1);
            line = t >> sd.nb_shift;
        } else {
            j = t % nb;
            line = t / nb;
        }
        int k, jq;
        if (sd.ns_shift >= 0) {
            k = j & (Ns - 1);
            jq = j >> sd.ns_shift;
        } else {
            k = j % Ns;
            jq = j / Ns;
        }
        const C* src = a + line * lstride;
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = src[(j + r * nb) * estride];
        if (Ns > 1) {
            const int step = k * sd.ts;
#pragma unroll
            for (int r = 1; r < R; ++r) {
                C w = tw[r * step];
                if (INV) w.y = -w.y;
                v[r] = v[r] * w;
            }
        }
        Dft<R, INV, C>::run(v);
        C* dst = b + line * lstride;
        const int base = jq * Ns * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) dst[(base + r * Ns) * estride] = v[r];
    }
}

// Stage with arbitrary element access: inputs come from in(line, i), outputs
// go to out(line, i, value).  Used for the first and last stages, which read
// and write global memory (or another shared buffer) directly.
template <int R, bool INV, bool LINE_FAST, int NL, typename C, class In, class Out>
__device__ __forceinline__ void fft_stage_f(const FftStage sd, const C* __restrict__ tw, In in, Out out) {
    const int nb = sd.nb, Ns = sd.Ns;
    const int total = NL * nb;
    for (int t = threadIdx.x; t < total; t += blockDim.x) {
        int line, j;
        if (LINE_FAST) {
            line = t % NL;
            j = t / NL;
        } else if (sd.nb_shift >= 0) {
            j = t & (nb - 1);
            line = t >> sd.nb_shift;
        } else {
            j = t % nb;
            line = t / nb;
        }
        int k, jq;
        if (sd.ns_shift >= 0) {
            k = j & (Ns - 1);
            jq = j >> sd.ns_shift;
        } else {
            k = j % Ns;
            jq = j / Ns;
        }
        C v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = in(line, j + r * nb);
        if (Ns > 1) {
            const int step = k * sd.ts;
#pragma unroll
            for (int r = 1; r < R; ++r) {
                C w = tw[r * step];
                if (INV) w.y = -w.y;
                v[r] = v[r] * w;
            }
        }
        Dft<R, INV, C>::run(v);
        const int base = jq * Ns * R + k;
#pragma unroll
        for (int r = 0; r < R; ++r) out(line, base + r * Ns, v[r]);
    }
}

template <bool INV, bool LINE_FAST, int NL, typename C, class In, class Out>
__device__ __forceinline__ void fft_stage_any(const FftStage sd, const C* tw, In in, Out out) {
    switch (sd.R) {
        case 2: fft_stage_f<2, INV, LINE_FAST, NL>(sd, tw, in, out); break;
        case 3: fft_stage_f<3, INV, LINE_FAST, NL>(sd, tw, in, out); break;
        case 4: fft_stage_f<4, INV, LINE_FAST, NL>(sd, tw, in, out); break;
        case 5: fft_stage_f<5, INV, LINE_FAST, NL>(sd, tw, in, out); break;
        case 7: fft_stage_f<7, INV, LINE_FAST, NL>(sd, tw, in, out); break;
        default: fft_stage_f<8, INV, LINE_FAST, NL>(sd, tw, in, out); break;
    }
}

// Full transform of NL lines whose inputs are read through ld(line, i) by
// the first stage and whose outputs are handed to st(line, i, value) by the
// last stage; the stages in between ping-pong between the shared buffers A
// and B (element i of line l at l * lstride + i * estride; with PAD8 one
// padding slot follows every 8 elements, i -> i + i/8, which together with a
// line stride of 8 mod 16 makes the radix-8 stride-8 scatter of the first
// stage free of bank conflicts).  The block is synchronised between stages
// and after the last one.
template <bool INV, bool LINE_FAST, int NL, bool PAD8 = false, typename C, class Ld, class St>
__device__ void fft_lines_io(C* A, C* B, int lstride, int estride, const FftPlan& p, const C* tw, Ld ld, St st) {
    auto sm_in = [&](const C* buf) {
        return [=](int l, int i) { return buf[l * lstride + (PAD8 ? i + (i >> 3) : i) * estride]; };
    };
    auto sm_out = [&](C* buf) {
        return [=](int l, int i, C v) { buf[l * lstride + (PAD8 ? i + (i >> 3) : i) * estride] = v; };
    };
    if (p.nst == 1) {
        fft_stage_any<INV, LINE_FAST, NL>(p.st[0], tw, ld, st);
        __syncthreads();
        return;
    }
    fft_stage_any<INV, LINE_FAST, NL>(p.st[0], tw, ld, sm_out(A));
    __syncthreads();
    C* a = A;
    C* b = B;
    for (int s = 1; s + 1 < p.nst; ++s) {
        fft_stage_any<INV, LINE_FAST, NL>(p.st[s], tw, sm_in(a), sm_out(b));
        __syncthreads();
        C* t = a;
        a = b;
        b = t;
    }
    fft_stage_any<INV, LINE_FAST, NL>(p.st[p.nst - 1], tw, sm_in(a), st);
    __syncthreads();
}

// Full transform of NL lines; returns the buffer that holds the result (a
// or b).  Synchronises the block after every stage (callers sync before).
template <bool INV, bool LINE_FAST, int NL, typename C>
__device__ C* fft_lines(C* a, C* b, int lstride, int estride, const FftPlan& p, const C* tw) {
    for (int st = 0; st < p.nst; ++st) {
        const FftStage sd = p.st[st];
        switch (sd.R) {
            case 2: fft_stage<2, INV, LINE_FAST, NL>(a, b, lstride, estride, sd, tw); break;
            case 3: fft_stage<3, INV, LINE_FAST, NL>(a, b, lstride, estride, sd, tw); break;
            case 4: fft_stage<4, INV, LINE_FAST, NL>(a, b, lstride, estride, sd, tw); break;
            case 5: fft_stage<5, INV, LINE_FAST, NL>(a, b, lstride, estride, sd, tw); break;
            case 7: fft_stage<7, INV, LINE_FAST, NL>(a, b, lstride, estride, sd, tw); break;
            default: fft_stage<8, INV, LINE_FAST, NL>(a, b, lstride, estride, sd, tw); break;
        }
        __syncthreads();
        C* t = a;
        a = b;
        b = t;
    }
    return a;
}

}  // namespace eels
