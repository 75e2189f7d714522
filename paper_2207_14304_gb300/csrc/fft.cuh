// FFTs of square power-of-two tiles (T = 256, 512, 1024): Stockham auto-sort
// passes of radix 8 (then 4 or 2 to finish) with a twiddle table of
// e^{-2 pi i m / T} built in double precision on the host.  Forward transforms
// are unnormalised, inverse transforms are unscaled (the caller divides by T^2),
// as in numpy.  The real type is float (image data) or double (PSF transforms).
// The first half states the butterflies and a pass over a sequence in memory (the form
// of whole transforms on the CPU); the second half is the register form the kernels
// run, whose steps and lane maps are host-callable too.
#pragma once

#include <cuda_runtime.h>

// the butterflies and the pass are host-callable too, so that a CPU driver can
// run the same code thread by thread
#define FFT_HD __host__ __device__ __forceinline__

namespace fft {

template <typename R> struct Cx;
template <> struct Cx<float> { using T = float2; };
template <> struct Cx<double> { using T = double2; };

template <typename C> FFT_HD C cadd(C a, C b) { return {a.x + b.x, a.y + b.y}; }
template <typename C> FFT_HD C csub(C a, C b) { return {a.x - b.x, a.y - b.y}; }
template <typename C> FFT_HD C cmul(C a, C b) {
    return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <typename C> FFT_HD C cconj(C a) { return {a.x, -a.y}; }
// a * (s i), s = -1 (forward) or +1 (inverse)
template <int S, typename C> FFT_HD C cmul_i(C a) {
    return S < 0 ? C{a.y, -a.x} : C{-a.y, a.x};
}

template <int S, typename C> FFT_HD void dft2(C* v) {
    const C a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
}

template <int S, typename C> FFT_HD void dft4(C& a0, C& a1, C& a2, C& a3) {
    const C t0 = cadd(a0, a2), t1 = csub(a0, a2), t2 = cadd(a1, a3), t3 = cmul_i<S>(csub(a1, a3));
    a0 = cadd(t0, t2);
    a1 = cadd(t1, t3);
    a2 = csub(t0, t2);
    a3 = csub(t1, t3);
}

template <int S, typename C> FFT_HD void dft8(C* v) {
    using R = decltype(v[0].x);
    C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    C o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<S>(e0, e1, e2, e3);
    dft4<S>(o0, o1, o2, o3);
    const R r = (R)0.70710678118654752440;
    o1 = cmul(o1, C{r, (R)S * r});           // e^{S i pi / 4}
    o2 = cmul_i<S>(o2);                       // e^{S i pi / 2}
    o3 = cmul(o3, C{-r, (R)S * r});          // e^{S 3 i pi / 4}
    v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
    v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
    v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
}

// dft8 of values whose elements 2 .. 5 are zero, with the same roundings.
template <int S, typename C> FFT_HD void dft8_few(C* v) {
    using R = decltype(v[0].x);
    const C a = v[0], b = v[1], c = v[6], d = v[7], ci = cmul_i<S>(c), di = cmul_i<S>(d);
    const C e0 = cadd(a, c), e1 = csub(a, ci), e2 = csub(a, c), e3 = cadd(a, ci);
    const C o0 = cadd(b, d);
    C o1 = csub(b, di), o2 = csub(b, d), o3 = cadd(b, di);
    const R r = (R)0.70710678118654752440;
    o1 = cmul(o1, C{r, (R)S * r});
    o2 = cmul_i<S>(o2);
    o3 = cmul(o3, C{-r, (R)S * r});
    v[0] = cadd(e0, o0); v[4] = csub(e0, o0);
    v[1] = cadd(e1, o1); v[5] = csub(e1, o1);
    v[2] = cadd(e2, o2); v[6] = csub(e2, o2);
    v[3] = cadd(e3, o3); v[7] = csub(e3, o3);
}

// One Stockham pass of radix RAD over a sequence of length T held in a
// (stride 1), writing b: butterfly j (0 <= j < T / RAD) reads a[j + r T/RAD],
// multiplies by e^{S 2 pi i r k / (Ns RAD)} (k = j mod Ns) and writes the
// RAD-point DFT to b[(j / Ns) Ns RAD + k + r Ns].  tw[m] = e^{-2 pi i m / T}.
template <int T, int RAD, int S, typename C>
FFT_HD void stockham_pass(const C* a, C* b, const C* tw, int Ns, int lane, int nlanes) {
    for (int j = lane; j < T / RAD; j += nlanes) {
        C v[RAD];
        const int k = j & (Ns - 1);
        const int step = T / (Ns * RAD);
#pragma unroll
        for (int r = 0; r < RAD; r++) {
            v[r] = a[j + r * (T / RAD)];
            if (r) {
                const C w = tw[(r * k * step) & (T - 1)];
                v[r] = cmul(v[r], S < 0 ? w : cconj(w));
            }
        }
        if (RAD == 8) dft8<S>(v);
        else if (RAD == 4) dft4<S>(v[0], v[1], v[2], v[3]);
        else dft2<S>(v);
        const int d = (j / Ns) * Ns * RAD + k;
#pragma unroll
        for (int r = 0; r < RAD; r++) b[d + r * Ns] = v[r];
    }
}

// Sequences per CTA and threads per sequence for a T-point transform.
template <int T, typename R> struct Shape {
    static constexpr int SEQ = (sizeof(R) == 4 ? 16 : 8) / (T > 512 ? 2 : 1);
    static constexpr int LANES = T / 8;                  // one radix-8 butterfly per thread
    static constexpr int THREADS = SEQ * LANES;
    static constexpr int PAD = T + 1;                    // padded shared row (transposed loads)
    static constexpr size_t SMEM = (2 * (size_t)SEQ * PAD + T) * sizeof(typename Cx<R>::T);
};

// ---------------------------------------------------------------------------
// The transforms the kernels run: one T-point sequence on T / 8 lanes, eight
// values per lane in registers, lane l holding elements l + m T/8 (m = 0..7)
// before and after, so a transform can start from and end in global memory with
// consecutive lanes on consecutive elements, and a forward transform, a
// pointwise product and an inverse one chain without leaving the registers.
// Radices 8, 8, 4 (T = 256), 8, 8, 8 (512) and 8, 8, 4, 4 (1024); between two
// passes the values cross through shared memory once (position p at p + p / 8:
// the strided writes of a pass then fall on different banks), alternating
// between two buffers so that a crossing needs one barrier.  The version that
// kept the sequence in shared memory through all passes (one load, three
// read-modify-write passes, one store) ran at 1.7 TB/s on 216 tiles of 512^2.
template <int T> struct Reg {
    static constexpr int LANES = T / 8;
    static constexpr int CB = T == 256 ? 8 : 4;           // sequences per CTA and columns per block of the layout
    static constexpr int THREADS = LANES * CB;
    static constexpr int PT = T + T / 8;                  // padded shared sequence
    static constexpr int NTW = T == 256 ? 13 : T == 512 ? 14 : 16;   // twiddles a lane uses
};

// Where position p of a sequence lies in its padded shared row.
FFT_HD int pad(int p) { return p + (p >> 3); }

// Index into the twiddle table of slot i of a lane: pass 2 (radix 8, Ns = 8) in
// slots 0..6, then pass 3 (and 4), per butterfly.
template <int T> FFT_HD int tw_index(int i, int lane) {
    if (i < 7) return ((i + 1) * (lane & 7) * (T / 64)) & (T - 1);
    i -= 7;
    if (T == 512) return ((i + 1) * lane) & (T - 1);                           // radix 8, Ns = 64
    if (T == 256) return ((i % 3 + 1) * (lane + (i / 3) * (T / 8))) & (T - 1); // radix 4, Ns = 64
    if (i < 3) return ((i + 1) * (lane & 63) * (T / 256)) & (T - 1);           // radix 4, Ns = 64
    i -= 3;
    return ((i % 3 + 1) * (lane + (i / 3) * (T / 8))) & (T - 1);               // radix 4, Ns = 256
}

// Twiddles of a lane, held in registers (FP32) or read from the table as they
// are needed (FP64, where the arithmetic hides the reads).
template <int T> struct TwReg {
    float2 w[Reg<T>::NTW];
    __device__ __forceinline__ TwReg(const float2* tab, int lane) {
#pragma unroll
        for (int i = 0; i < Reg<T>::NTW; i++) w[i] = __ldg(tab + tw_index<T>(i, lane));
    }
    FFT_HD float2 get(int i) const { return w[i]; }
};
template <int T> struct TwTab {
    const double2* tab;
    int lane;
    FFT_HD double2 get(int i) const {
#ifdef __CUDA_ARCH__
        return __ldg(tab + tw_index<T>(i, lane));
#else
        return tab[tw_index<T>(i, lane)];
#endif
    }
};

// Where value i of a lane goes in the padded row between pass STEP and the next (passes are
// counted from 0; the first two are of radix 8, then 8 or 4): butterfly j's output r to
// (j / Ns) Ns RAD + j mod Ns + r Ns.
template <int T, int STEP> FFT_HD int cross_to(int lane, int i) {
    constexpr int RAD = STEP < 2 ? 8 : 4, Ns = STEP == 0 ? 1 : (STEP == 1 ? 8 : 64), NB = 8 / RAD;
    const int j = lane + i % NB * (T / 8);
    return pad((j / Ns) * Ns * RAD + (j & (Ns - 1)) + i / NB * Ns);
}

// Lane values of pass STEP to the next pass's; ST the element stride of the sequence in
// shared memory.  FEW: only values 0, 1, 6 and 7 are used next.
template <int T, int STEP, int ST, bool FEW = false, typename C>
__device__ __forceinline__ void cross(C (&v)[8], C*& s0, C*& s1, int lane) {
#pragma unroll
    for (int i = 0; i < 8; i++) s0[cross_to<T, STEP>(lane, i) * ST] = v[i];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 8; m++) {
        if (FEW && m >= 2 && m < 6) continue;
        v[m] = s0[pad(lane + m * (T / 8)) * ST];
    }
    C* t = s0;
    s0 = s1;
    s1 = t;
}

template <int S, typename C> FFT_HD C tmul(C v, C w) { return cmul(v, S < 0 ? w : cconj(w)); }

// One radix-4 pass: butterflies b = 0, 1 on v[b], v[b + 2], v[b + 4], v[b + 6],
// twiddle slots i0 + (PER ? 3 b : 0) + r - 1.
template <int S, bool PER, typename C, typename TW>
FFT_HD void radix4(C (&v)[8], const TW& tw, int i0) {
#pragma unroll
    for (int b = 0; b < 2; b++) {
#pragma unroll
        for (int r = 1; r < 4; r++) v[b + 2 * r] = tmul<S>(v[b + 2 * r], tw.get(i0 + (PER ? 3 * b : 0) + r - 1));
        dft4<S>(v[b], v[b + 2], v[b + 4], v[b + 6]);
    }
}

// The butterflies of pass STEP > 0 on a lane's values.  FEW (pass 1): values 2 .. 5 are zero.
template <int T, int S, int STEP, bool FEW = false, typename C, typename TW>
FFT_HD void pass(C (&v)[8], const TW& tw) {
    if constexpr (STEP == 1) {
#pragma unroll
        for (int r = 1; r < 8; r++)
            if (!FEW || r < 2 || r > 5) v[r] = tmul<S>(v[r], tw.get(r - 1));
        if (FEW) dft8_few<S>(v);
        else dft8<S>(v);
    } else if constexpr (T == 512) {
#pragma unroll
        for (int r = 1; r < 8; r++) v[r] = tmul<S>(v[r], tw.get(6 + r));
        dft8<S>(v);
    } else if constexpr (T == 256) {
        radix4<S, true>(v, tw, 7);
    } else {
        radix4<S, STEP == 3>(v, tw, STEP == 3 ? 10 : 7);
    }
}

// Every pass after the first (whose butterflies the caller has done: the PSF
// transforms skip its zeros).  Every thread of the CTA calls it.  FEW: only the
// lanes below T/32 and from T/8 - T/32 on hold values after the first pass, which the
// second pass meets as its elements 0, 1, 6 and 7.
template <int T, int S, int ST, bool FEW = false, typename C, typename TW>
__device__ __forceinline__ void fft_tail(C (&v)[8], const TW& tw, C*& s0, C*& s1, int lane) {
    cross<T, 0, ST, FEW>(v, s0, s1, lane);
    pass<T, S, 1, FEW>(v, tw);
    cross<T, 1, ST>(v, s0, s1, lane);
    pass<T, S, 2>(v, tw);
    if constexpr (T == 1024) {
        cross<T, 2, ST>(v, s0, s1, lane);
        pass<T, S, 3>(v, tw);
    }
}

// Two sequences of a lane side by side: one barrier serves both crossings, and each one's
// arithmetic hides the other's latency.
template <int T, int STEP, int ST, typename C>
__device__ __forceinline__ void cross2(C (&v)[8], C (&w)[8], C*& v0, C*& v1, C*& w0, C*& w1, int lane) {
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const int to = cross_to<T, STEP>(lane, i) * ST;
        v0[to] = v[i];
        w0[to] = w[i];
    }
    __syncthreads();
#pragma unroll
    for (int m = 0; m < 8; m++) {
        const int from = pad(lane + m * (T / 8)) * ST;
        v[m] = v0[from];
        w[m] = w0[from];
    }
    C* t = v0;
    v0 = v1;
    v1 = t;
    t = w0;
    w0 = w1;
    w1 = t;
}
template <int T, int S, int ST, typename C, typename TW>
__device__ __forceinline__ void fft_reg2(C (&v)[8], C (&w)[8], const TW& tw, C*& v0, C*& v1, C*& w0, C*& w1, int lane) {
    dft8<S>(v);
    dft8<S>(w);
    cross2<T, 0, ST>(v, w, v0, v1, w0, w1, lane);
    pass<T, S, 1>(v, tw);
    pass<T, S, 1>(w, tw);
    cross2<T, 1, ST>(v, w, v0, v1, w0, w1, lane);
    pass<T, S, 2>(v, tw);
    pass<T, S, 2>(w, tw);
    if constexpr (T == 1024) {
        cross2<T, 2, ST>(v, w, v0, v1, w0, w1, lane);
        pass<T, S, 3>(v, tw);
        pass<T, S, 3>(w, tw);
    }
}

template <int T, int S, int ST, typename C, typename TW>
__device__ __forceinline__ void fft_reg(C (&v)[8], const TW& tw, C*& s0, C*& s1, int lane) {
    dft8<S>(v);
    fft_tail<T, S, ST>(v, tw, s0, s1, lane);
}

}  // namespace fft
