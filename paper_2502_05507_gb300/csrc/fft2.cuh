// Register-resident FFT building blocks for the convolution passes.
//
// A transform of length L = R1 * R2 (R2 = R1 or 2 R1) is done by R1 threads
// per line with the four-step factorisation n = n1 + R1 n2, k = k2 + R2 k1:
//   X[k2 + R2 k1] = sum_n1 W_R1^{n1 k1} W_L^{n1 k2} sum_n2 x[n1 + R1 n2] W_R2^{n2 k2}.
// "n-layout": thread t holds x[t + R1 m], m < R2 (global loads/stores of a
// strided line are coalesced across the columns a warp covers).
// "k-layout": thread t holds X[k2 + R2 k1] for k2 = t + q R1 (q < R2/R1),
// k1 < R1, in v[q R1 + k1].
// Forward: R2-point DFT in registers, twiddle, one exchange through shared
// memory, R1-point DFTs in registers. The inverse runs the same steps
// backwards from the k-layout to the n-layout. Every register DFT has
// compile-time indices and constant twiddles, so nothing is spilled to
// local memory; one shared-memory round trip per transform.
#pragma once

#include <type_traits>

#include "common.cuh"

namespace bae {

// cos and sin of 2 pi m / 32 from the first-octant values by symmetry
struct Root32 {
    double c, s;
};
__host__ __device__ constexpr Root32 root32(int m) {
    // cos(pi j / 16), j = 0..8
    constexpr double C[9] = {1.0,
                             0.98078528040323044913,
                             0.92387953251128675613,
                             0.83146961230254523708,
                             0.70710678118654752440,
                             0.55557023301960222474,
                             0.38268343236508977173,
                             0.19509032201612826785,
                             0.0};
    m = ((m % 32) + 32) % 32;
    const int q = m / 8, r = m % 8;  // angle = q pi/2 + r pi/16
    const double cr = C[r], sr = C[8 - r];
    if (q == 0) return {cr, sr};
    if (q == 1) return {-sr, cr};
    if (q == 2) return {-cr, -sr};
    return {sr, -cr};
}

// cos and sin of 2 pi m / 24, the same for the lengths with a factor of three
__host__ __device__ constexpr Root32 root24(int m) {
    // cos(pi j / 12), j = 0..6
    constexpr double C[7] = {1.0, 0.96592582628906828675, 0.86602540378443864676, 0.70710678118654752440,
                             0.5, 0.25881904510252076235, 0.0};
    m = ((m % 24) + 24) % 24;
    const int q = m / 6, r = m % 6;
    const double cr = C[r], sr = C[6 - r];
    if (q == 0) return {cr, sr};
    if (q == 1) return {-sr, cr};
    if (q == 2) return {-cr, -sr};
    return {sr, -cr};
}
// cos and sin of 2 pi M / R, R dividing 32 or 24
template <int R>
__host__ __device__ constexpr Root32 root_of(int M) {
    if constexpr (32 % R == 0) return root32(M * (32 / R));
    else return root24(M * (24 / R));
}

// x (c + i s)
template <typename C, typename T>
__device__ __forceinline__ C crot(C x, T c, T s) {
    return cmake<C>(x.x * c - x.y * s, x.x * s + x.y * c);
}

// x * exp(-/+ 2 pi i M / R) with compile-time M, R dividing 32 or 24
template <int R, int M, bool INV, typename C>
__device__ __forceinline__ C wmul(C x) {
    using T = decltype(x.x);
    constexpr int m = ((M % R) + R) % R;
    if constexpr (m == 0) return x;
    if constexpr (2 * m == R) return cmake<C>(-x.x, -x.y);
    if constexpr (4 * m == R) {       // forward: -i, inverse: +i
        if constexpr (INV) return cmake<C>(-x.y, x.x);
        else return cmake<C>(x.y, -x.x);
    }
    if constexpr (4 * m == 3 * R) {   // forward: +i, inverse: -i
        if constexpr (INV) return cmake<C>(x.y, -x.x);
        else return cmake<C>(-x.y, x.x);
    }
    constexpr Root32 w = root_of<R>(m);
    const T c = (T)w.c;
    const T s = INV ? (T)w.s : (T)-w.s;
    return crot(x, c, s);
}

template <bool INV, typename C>
__device__ __forceinline__ void rdft2(C& a, C& b) {
    const C t = a;
    a = cadd(t, b);
    b = csub(t, b);
}

template <bool INV, typename C>
__device__ __forceinline__ void rdft4(C& x0, C& x1, C& x2, C& x3) {
    const C t0 = cadd(x0, x2), t1 = csub(x0, x2), t2 = cadd(x1, x3);
    const C t3 = wmul<4, 1, INV>(csub(x1, x3));
    x0 = cadd(t0, t2);
    x2 = csub(t0, t2);
    x1 = cadd(t1, t3);
    x3 = csub(t1, t3);
}

__device__ __forceinline__ float fma_t(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_t(double a, double b, double c) { return __fma_rn(a, b, c); }

// The radix-2 butterfly lo = e + W o, hi = e - W o with W = W_R^{+-K} a
// compile-time root. For float32 and float64 a general rotation is folded
// into the butterfly with fused multiply-adds (the factorisation of Linzer
// and Feig, "Implementation of efficient FFT algorithms on fused
// multiply-add architectures", IEEE Trans. Signal Process. 41, 1993):
// W o = f (o + i r o) with f the larger of |cos|, |sin| (so |r| <= 1), then
// e +- f u: six fused operations instead of a four-operation rotation and
// four additions. Rotations by multiples of pi/2 and the double-float type
// keep the plain form.
template <int R, int K, bool INV, typename C>
__device__ __forceinline__ void bfly(const C& e, const C& o, C& lo, C& hi) {
    using T = decltype(o.x);
    if constexpr (!(std::is_same<T, float>::value || std::is_same<T, double>::value) || (4 * K) % R == 0) {
        const C w = wmul<R, K, INV>(o);
        lo = cadd(e, w);
        hi = csub(e, w);
    } else {
        constexpr Root32 w = root_of<R>(K);
        constexpr double c = w.c, sn = INV ? w.s : -w.s;   // W = c + i sn
        T ux, uy, f;
        if constexpr (c * c >= sn * sn) {   // W = c (1 + i sn/c)
            constexpr double r = sn / c;
            ux = fma_t((T)-r, o.y, o.x);
            uy = fma_t((T)r, o.x, o.y);
            f = (T)c;
        } else {                            // W = sn (c/sn + i)
            constexpr double r = c / sn;
            ux = fma_t((T)r, o.x, -o.y);
            uy = fma_t((T)r, o.y, o.x);
            f = (T)sn;
        }
        lo = cmake<C>(fma_t(f, ux, e.x), fma_t(f, uy, e.y));
        hi = cmake<C>(fma_t(-f, ux, e.x), fma_t(-f, uy, e.y));
    }
}

// the butterflies k = K .. R/2 - 1 of a radix-2 step: v[k], v[k + R/2]
template <int R, bool INV, typename C, int K>
struct Bflies {
    __device__ __forceinline__ static void run(const C* e, const C* o, C* v) {
        bfly<R, K, INV>(e[K], o[K], v[K], v[K + R / 2]);
        if constexpr (K + 1 < R / 2) Bflies<R, INV, C, K + 1>::run(e, o, v);
    }
};

// x / 2
template <typename C>
__device__ __forceinline__ C chalf(C x) {
    using T = decltype(x.x);
    return cmake<C>(x.x * (T)0.5, x.y * (T)0.5);
}

// x with its parts in order: its sums' low parts below half a unit of the high ones
// (double-float; dsf.cuh), nothing for the other types
template <typename C>
__device__ __forceinline__ C cnorm(C x) { return x; }
template <int R, typename C>
__device__ __forceinline__ void cnorm_all(C* v) {
#pragma unroll
    for (int i = 0; i < R; ++i) v[i] = cnorm(v[i]);
}

// Three points: y0 = x0 + x1 + x2, y1, y2 = x0 - (x1 + x2) / 2 -/+ i (sqrt 3 /
// 2) (x1 - x2) (forward). NZ: how many of the inputs are nonzero.
template <bool INV, int NZ, typename C>
__device__ __forceinline__ void rdft3(C* v) {
    using T = decltype(v[0].x);
    if constexpr (NZ == 1) {
        v[1] = v[2] = v[0];
        return;
    }
    const C t = NZ == 2 ? v[1] : cadd(v[1], v[2]);
    const C d = cscale(NZ == 2 ? v[1] : csub(v[1], v[2]), (T)0.86602540378443864676);
    const C m = csub(v[0], chalf(t));
    const C e = INV ? cmake<C>(-d.y, d.x) : cmake<C>(d.y, -d.x);   // +i d, -i d
    v[0] = cnorm(cadd(v[0], t));
    v[1] = cnorm(cadd(m, e));
    v[2] = cnorm(csub(m, e));
}

// In-register DFT of v[0..R) in natural order, R = 2^p <= 32 or 3 2^p <= 24.
template <int R, bool INV, typename C>
__device__ __forceinline__ void rdft(C* v);

template <int R, bool INV, typename C>
__device__ __forceinline__ void rdft(C* v) {
    if constexpr (R == 2) {
        rdft2<INV>(v[0], v[1]);
    } else if constexpr (R == 3) {
        rdft3<INV, 3>(v);
    } else if constexpr (R == 4) {
        rdft4<INV>(v[0], v[1], v[2], v[3]);
    } else {
        // radix-2 decimation in time: even and odd halves, then butterflies
        C e[R / 2], o[R / 2];
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
            e[i] = v[2 * i];
            o[i] = v[2 * i + 1];
        }
        rdft<R / 2, INV>(e);
        rdft<R / 2, INV>(o);
        Bflies<R, INV, C, 0>::run(e, o, v);
    }
}

// rdft of v[0..R) whose upper half v[R/2..R) is zero (the zero-padded
// inputs of the forward transforms): the butterflies with a zero operand
// are dropped (same values as rdft up to the sign of zeros)
template <int R, bool INV, typename C>
__device__ __forceinline__ void rdft_zhi(C* v) {
    if constexpr (R == 2) {
        v[1] = v[0];
    } else if constexpr (R == 4) {
        const C x0 = v[0], x1 = v[1];
        const C t3 = wmul<4, 1, INV>(x1);
        v[0] = cadd(x0, x1);
        v[2] = csub(x0, x1);
        v[1] = cadd(x0, t3);
        v[3] = csub(x0, t3);
    } else if constexpr (R == 6) {   // v[0..3) nonzero
        C e[3] = {v[0], v[2], v[2]}, o[3] = {v[1], v[1], v[1]};
        rdft3<INV, 2>(e);
        Bflies<R, INV, C, 0>::run(e, o, v);
    } else {
        C e[R / 2], o[R / 2];   // both halves have a zero upper half again
#pragma unroll
        for (int i = 0; i < R / 2; ++i) {
            e[i] = v[2 * i];
            o[i] = v[2 * i + 1];
        }
        rdft_zhi<R / 2, INV>(e);
        rdft_zhi<R / 2, INV>(o);
        Bflies<R, INV, C, 0>::run(e, o, v);
    }
}

// the same with v[R/4..R) zero, R = 8
template <int R, bool INV, typename C>
__device__ __forceinline__ void rdft_zquarter(C* v) {
    static_assert(R == 8, "two values");
    const C e[4] = {v[0], v[0], v[0], v[0]}, o[4] = {v[1], v[1], v[1], v[1]};
    Bflies<R, INV, C, 0>::run(e, o, v);
}

// The barrier around an exchange: the CTA's, or (WARP) the warp's where all
// threads of a line are in one warp.
template <bool WARP>
__device__ __forceinline__ void xch_sync() {
    if constexpr (WARP) __syncwarp();
    else __syncthreads();
}

template <int L> struct Factors;
template <> struct Factors<16> { static constexpr int R1 = 4, R2 = 4; };
template <> struct Factors<32> { static constexpr int R1 = 4, R2 = 8; };
template <> struct Factors<64> { static constexpr int R1 = 8, R2 = 8; };
template <> struct Factors<128> { static constexpr int R1 = 8, R2 = 16; };
template <> struct Factors<256> { static constexpr int R1 = 16, R2 = 16; };
template <> struct Factors<512> { static constexpr int R1 = 16, R2 = 32; };

// Exchange buffer for one transform: R2 x R1 complex at
// xch[base + k2 * sk + n1 * sn]; the caller picks the strides so that the
// lanes of a warp touch distinct banks (columns interleaved: sk = R1 W,
// sn = W, base = column; lines: sk = R1 + 1, sn = 1, base = line offset).

// n-layout -> k-layout (forward, or inverse when INV: then from the
// n-layout of X to the k-layout of the inverse transform, same steps with
// conjugate twiddles). tw: exp(-2 pi i m / L), m < L, followed by the table
// exp(-2 pi i n1 k2 / L) at [k2 R1 + n1], which the threads of a line in one
// warp (WARP) read at consecutive places and compile-time offsets (the column
// passes, whose lanes share n1, ran slower with it: 38 against 28 us for the
// float32 i pass at N = 128). ZHI: the input rows
// n >= L/2 are zero (v[m] = 0 for m >= R2 / 2).
template <int L, bool INV, bool ZHI = false, bool WARP = false, typename C>
__device__ __forceinline__ void fft_n2k(C* v, C* xch, int base, int sk, int sn, int t, const C* __restrict__ tw) {
    constexpr int R1 = Factors<L>::R1, R2 = Factors<L>::R2, Q = R2 / R1;
    if constexpr (ZHI) rdft_zhi<R2, INV>(v);          // v[k2] = Y[t][k2]
    else rdft<R2, INV>(v);
#pragma unroll
    for (int k2 = 1; k2 < R2; ++k2) {
        const C w = ldg_c(WARP ? tw + L + k2 * R1 + t : tw + t * k2);
        v[k2] = INV ? cmulc(v[k2], w) : cmul(v[k2], w);
    }
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) xch[base + k2 * sk + t * sn] = v[k2];
    xch_sync<WARP>();
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) v[q * R1 + n1] = xch[base + (t + q * R1) * sk + n1 * sn];
    xch_sync<WARP>();
#pragma unroll
    for (int q = 0; q < Q; ++q) rdft<R1, INV>(v + q * R1);   // v[q R1 + k1] = X[k2 + R2 k1]
}

// k-layout -> n-layout (inverse when INV, the mirror of fft_n2k).
template <int L, bool INV, bool WARP = false, typename C>
__device__ __forceinline__ void fft_k2n(C* v, C* xch, int base, int sk, int sn, int t, const C* __restrict__ tw) {
    constexpr int R1 = Factors<L>::R1, R2 = Factors<L>::R2, Q = R2 / R1;
#pragma unroll
    for (int q = 0; q < Q; ++q) rdft<R1, INV>(v + q * R1);   // v[q R1 + n1] = Z[k2][n1]
#pragma unroll
    for (int q = 0; q < Q; ++q)
#pragma unroll
        for (int n1 = 0; n1 < R1; ++n1) {
            const int k2 = t + q * R1;
            if (n1 > 0 && k2 > 0) {
                // (R1 = R2: the table is symmetric, and a warp reads it in order)
                const C w = ldg_c(WARP ? tw + L + (R1 == R2 ? n1 * R1 + k2 : k2 * R1 + n1) : tw + n1 * k2);
                v[q * R1 + n1] = INV ? cmulc(v[q * R1 + n1], w) : cmul(v[q * R1 + n1], w);
            }
            xch[base + k2 * sk + n1 * sn] = v[q * R1 + n1];
        }
    xch_sync<WARP>();
#pragma unroll
    for (int k2 = 0; k2 < R2; ++k2) v[k2] = xch[base + k2 * sk + t * sn];
    xch_sync<WARP>();
    rdft<R2, INV>(v);                                   // v[n2] = x[t + R1 n2]
}


// ------------------------------------------------------------ transform plans
// A plan fixes how one line of length L is spread over the threads that
// transform it: TH threads per line, S values per thread. In both plans the
// n-layout is "thread t holds x[t + TH m] in slot m" (m < S), so a forward
// transform's zero upper half is exactly the slots m >= S / 2; the k-layout
// (after a forward transform, before an inverse one) is given by kidx(t, s).
// The exchange area of a line holds XLEN positions; position p of the line
// whose area starts at xch + base sits at xch[base + p * es], es = 1 for a
// private area per line (line passes; XS positions apart) or es = the number
// of lines interleaved element by element (column passes).

// Two levels (fft_n2k / fft_k2n above): TH = R1, S = R2.
template <int L>
struct Plan2 {
    static constexpr int R1 = Factors<L>::R1, R2 = Factors<L>::R2;
    static constexpr int TH = R1, S = R2;
    static constexpr int XS = R2 * (R1 + 1) + 1;   // private area stride (odd)
    static constexpr int XLEN = L;
    // slot s = q R1 + k1 holds X[t + q R1 + R2 k1]
    __host__ __device__ static constexpr int kidx(int t, int s) { return t + (s / R1) * R1 + R2 * (s % R1); }
    template <bool ZHI, bool WARP = false, typename C>
    __device__ __forceinline__ static void fwd(C* v, C* xch, int base, int es, int t, const C* __restrict__ tw) {
        fft_n2k<L, false, ZHI, WARP>(v, xch, base, es == 1 ? R1 + 1 : R1 * es, es, t, tw);
    }
    template <bool WARP = false, typename C>
    __device__ __forceinline__ static void inv(C* v, C* xch, int base, int es, int t, const C* __restrict__ tw) {
        fft_k2n<L, true, WARP>(v, xch, base, es == 1 ? R1 + 1 : R1 * es, es, t, tw);
    }
};

// Three levels for L = 512 = 8 x 8 x 8: 64 threads per line, 8 values each
// (the two-level 16 x 32 split holds 32 values per thread, which for
// 16-byte elements means ~200-255 registers and few warps per SM). With
// n = t + 64 m, t = t1 + 8 t2, and k = k3 + 8 k2 + 64 k1:
//   X[k] = sum_t1 W8^{t1 k1} W64^{t1 k2} sum_t2 W8^{t2 k2}
//          [ W512^{t k3} sum_m W8^{m k3} x[t + 64 m] ]
// stage A: thread t, DFT over m (slots k3), twiddle W512^{t k3};
// exchange; stage B: thread t1 + 8 k3, DFT over t2 (slots k2), twiddle
// W64^{t1 k2}; exchange; stage C: thread k3 + 8 k2, DFT over t1: slot k1
// holds X[t + 64 k1]. The inverse runs the stages backwards with conjugate
// twiddles. Positions are padded by one per 64 so that 16-byte accesses of
// the line passes do not collide in shared-memory banks.
struct Plan3_512 {
    static constexpr int TH = 64, S = 8;
    static constexpr int XLEN = 512 + 8;
    static constexpr int XS = XLEN + 1;
    __host__ __device__ static constexpr int kidx(int t, int s) { return t + 64 * s; }
    __device__ __forceinline__ static int pos(int p) { return p + (p >> 6); }

    // (the threads of a line are two warps: the barriers are the CTA's)
    // Z: 1 the upper half of the input is zero, 2 its upper three quarters
    template <int Z, bool = false, typename C>
    __device__ __forceinline__ static void fwd(C* v, C* xch, int base, int es, int t, const C* __restrict__ tw) {
        if constexpr (Z == 2) rdft_zquarter<8, false>(v);   // v[k3]
        else if constexpr (Z == 1) rdft_zhi<8, false>(v);
        else rdft<8, false>(v);
#pragma unroll
        for (int k3 = 1; k3 < 8; ++k3) v[k3] = cmul(v[k3], ldg_c(tw + t * k3));
#pragma unroll
        for (int k3 = 0; k3 < 8; ++k3) xch[base + pos(k3 * 64 + t) * es] = v[k3];
        __syncthreads();
        const int t1 = t & 7, k3 = t >> 3;
#pragma unroll
        for (int t2 = 0; t2 < 8; ++t2) v[t2] = xch[base + pos(k3 * 64 + t1 + 8 * t2) * es];
        __syncthreads();
        rdft<8, false>(v);                               // v[k2]
#pragma unroll
        for (int k2 = 1; k2 < 8; ++k2) v[k2] = cmul(v[k2], ldg_c(tw + 8 * t1 * k2));
#pragma unroll
        for (int k2 = 0; k2 < 8; ++k2) xch[base + pos((k3 * 8 + k2) * 8 + t1) * es] = v[k2];
        __syncthreads();
        const int c3 = t & 7, c2 = t >> 3;
#pragma unroll
        for (int u1 = 0; u1 < 8; ++u1) v[u1] = xch[base + pos((c3 * 8 + c2) * 8 + u1) * es];
        __syncthreads();
        rdft<8, false>(v);                               // v[k1] = X[t + 64 k1]
    }

    template <bool = false, typename C>
    __device__ __forceinline__ static void inv(C* v, C* xch, int base, int es, int t, const C* __restrict__ tw) {
        const int c3 = t & 7, c2 = t >> 3;               // this thread's (k3, k2)
        rdft<8, true>(v);                                // v[t1]
#pragma unroll
        for (int u1 = 0; u1 < 8; ++u1) xch[base + pos((c3 * 8 + c2) * 8 + u1) * es] = v[u1];
        __syncthreads();
        const int t1 = t & 7, k3 = t >> 3;
#pragma unroll
        for (int k2 = 0; k2 < 8; ++k2) v[k2] = xch[base + pos((k3 * 8 + k2) * 8 + t1) * es];
        __syncthreads();
#pragma unroll
        for (int k2 = 1; k2 < 8; ++k2) v[k2] = cmulc(v[k2], ldg_c(tw + 8 * t1 * k2));
        rdft<8, true>(v);                                // v[t2]
#pragma unroll
        for (int t2 = 0; t2 < 8; ++t2) xch[base + pos(k3 * 64 + t1 + 8 * t2) * es] = v[t2];
        __syncthreads();
#pragma unroll
        for (int j3 = 0; j3 < 8; ++j3) v[j3] = xch[base + pos(j3 * 64 + t) * es];
        __syncthreads();
#pragma unroll
        for (int j3 = 1; j3 < 8; ++j3) v[j3] = cmulc(v[j3], ldg_c(tw + t * j3));
        rdft<8, true>(v);                                // v[m] = x[t + 64 m]
    }
};

// Three levels for L = 256 = 8 x 8 x 4: 32 threads per line (one warp), 8
// values each (the two-level 16 x 16 split holds 16 values per thread:
// 170-210 registers for 16-byte elements, one 256-thread CTA per SM). With
// n = t + 32 m, t = t1 + 4 t2 (t1 < 4, t2 < 8), k = k3 + 8 k2 + 64 k1:
//   X[k] = sum_t1 W4^{t1 k1} W32^{t1 k2} sum_t2 W8^{t2 k2}
//          [ W256^{t k3} sum_m W8^{m k3} x[t + 32 m] ]
// stage A: thread t, DFT over m (slots k3), twiddle W256^{t k3}; exchange;
// stage B: thread t1 + 4 k3, DFT over t2 (slots k2), twiddle W32^{t1 k2};
// exchange; stage C: thread u takes the two pairs (k3, k2) = (u % 8,
// u / 8 + 4 h), h < 2, each a 4-point DFT over t1. Slot s = h + 2 k1 then
// holds X[u + 32 s]. The inverse runs the stages backwards with conjugate
// twiddles. Positions are swizzled, p -> p ^ rev3((p >> 5) & 7) (rev3
// reverses three bits), so that the 16-byte accesses of a line (one warp)
// hit eight distinct bank groups in every stage: rows of 32 positions
// apart land on distinct groups, and the two 4-aligned blocks read in stage
// B land in different halves.
struct Plan3_256 {
    static constexpr int TH = 32, S = 8;
    static constexpr int XLEN = 256;
    static constexpr int XS = XLEN + 1;
    __host__ __device__ static constexpr int kidx(int t, int s) { return t + 32 * s; }
    __device__ __forceinline__ static int pos(int p) {
        const int r = (p >> 5) & 7;
        return p ^ (((r & 1) << 2) | (r & 2) | ((r >> 2) & 1));
    }

    template <bool ZHI, bool WARP = false, typename C>
    __device__ __forceinline__ static void fwd(C* v, C* xch, int base, int es, int t, const C* __restrict__ tw) {
        if constexpr (ZHI) rdft_zhi<8, false>(v);       // v[k3]
        else rdft<8, false>(v);
#pragma unroll
        for (int k3 = 1; k3 < 8; ++k3) v[k3] = cmul(v[k3], ldg_c(tw + t * k3));
#pragma unroll
        for (int k3 = 0; k3 < 8; ++k3) xch[base + pos(k3 * 32 + t) * es] = v[k3];
        xch_sync<WARP>();
        const int t1 = t & 3, k3 = t >> 2;
#pragma unroll
        for (int t2 = 0; t2 < 8; ++t2) v[t2] = xch[base + pos(k3 * 32 + t1 + 4 * t2) * es];
        xch_sync<WARP>();
        rdft<8, false>(v);                               // v[k2]
#pragma unroll
        for (int k2 = 1; k2 < 8; ++k2) v[k2] = cmul(v[k2], ldg_c(tw + 8 * t1 * k2));
#pragma unroll
        for (int k2 = 0; k2 < 8; ++k2) xch[base + pos((k3 * 8 + k2) * 4 + t1) * es] = v[k2];
        xch_sync<WARP>();
        const int c3 = t & 7, c2 = t >> 3;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            C w[4];
#pragma unroll
            for (int u1 = 0; u1 < 4; ++u1) w[u1] = xch[base + pos((c3 * 8 + c2 + 4 * h) * 4 + u1) * es];
            rdft<4, false>(w);                           // w[k1]
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) v[h + 2 * k1] = w[k1];   // X[t + 32 (h + 2 k1)]
        }
        xch_sync<WARP>();
    }

    template <bool WARP = false, typename C>
    __device__ __forceinline__ static void inv(C* v, C* xch, int base, int es, int t, const C* __restrict__ tw) {
        const int c3 = t & 7, c2 = t >> 3;               // this thread's pairs (k3, k2 + 4 h)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            C w[4];
#pragma unroll
            for (int k1 = 0; k1 < 4; ++k1) w[k1] = v[h + 2 * k1];
            rdft<4, true>(w);                            // w[t1]
#pragma unroll
            for (int u1 = 0; u1 < 4; ++u1) xch[base + pos((c3 * 8 + c2 + 4 * h) * 4 + u1) * es] = w[u1];
        }
        xch_sync<WARP>();
        const int t1 = t & 3, k3 = t >> 2;
#pragma unroll
        for (int k2 = 0; k2 < 8; ++k2) v[k2] = xch[base + pos((k3 * 8 + k2) * 4 + t1) * es];
        xch_sync<WARP>();
#pragma unroll
        for (int k2 = 1; k2 < 8; ++k2) v[k2] = cmulc(v[k2], ldg_c(tw + 8 * t1 * k2));
        rdft<8, true>(v);                                // v[t2]
#pragma unroll
        for (int t2 = 0; t2 < 8; ++t2) xch[base + pos(k3 * 32 + t1 + 4 * t2) * es] = v[t2];
        xch_sync<WARP>();
#pragma unroll
        for (int j3 = 0; j3 < 8; ++j3) v[j3] = xch[base + pos(j3 * 32 + t) * es];
        xch_sync<WARP>();
#pragma unroll
        for (int j3 = 1; j3 < 8; ++j3) v[j3] = cmulc(v[j3], ldg_c(tw + t * j3));
        rdft<8, true>(v);                                // v[m] = x[t + 32 m]
    }
};

// Three levels for the lengths 3 2^p: L = RA x RB x RC, TH = RB RC threads per
// line (a power of two, within a warp), RA = 12 or 24 values each (12 x 8 x 4 for
// 16-byte elements at L = 384: with 24 values they take 255 registers). With n = t +
// TH m, t = t1 + RC t2, k = k3 + RA k2 + RA RB k1:
//   X[k] = sum_t1 W_RC^{t1 k1} W_TH^{t1 k2} sum_t2 W_RB^{t2 k2}
//          [ W_L^{t k3} sum_m W_RA^{m k3} x[t + TH m] ]
// stage A: thread t, DFT over m; exchange; stage B: RA / RB transforms (k3, t1)
// per thread over t2, in place in the exchange area; stage C: RA / RC
// transforms (k3, k2) per thread over t1. Rows of TH values are PITCH = TH + RC
// + 1 apart, so that the 16 lanes of a half warp read distinct 8-byte banks in
// stage C (rows k3 = lane mod RA: 21 k3 mod 16 for TH = 16) and nearly so in B.
//
// In double-float the results of every stage are put in order (cnorm): the stages
// of 12 points are five sums deep where those of 8 are three, and the window's
// rounding noise falls on 0.42 of the whole grid's volume. Without it the operator's
// error was 1.1 to 1.4 times the whole grid's (5.7e-15 against 4.2e-15 for an
// ellipsoid at N = 128), with it 0.8 to 1.1 times (4.5e-15); the windowed operators
// take 3 to 7% longer.
template <int RA, int RB, int RC>
struct PlanQ {
    static constexpr int TH = RB * RC, S = RA, L = RA * TH;
    static constexpr int PITCH = TH + RC + 1, XLEN = RA * PITCH, XS = XLEN | 1;
    static constexpr int QB = (RA + RB - 1) / RB;   // stage B transforms per thread (the last round may be partial)
    static_assert(RA % RC == 0 && TH <= 32, "a line in a warp, whole stage C transforms per thread");
    // slot s = q RC + k1 of thread t holds X[t + TH q + RA RB k1]
    __host__ __device__ static constexpr int kidx(int t, int s) { return t + TH * (s / RC) + RA * RB * (s % RC); }

    template <bool ZHI, bool WARP = false, typename C>
    __device__ __forceinline__ static void fwd(C* v, C* xch, int base, int es, int t, const C* __restrict__ tw) {
        if constexpr (ZHI) rdft_zhi<RA, false>(v);
        else rdft<RA, false>(v);
        cnorm_all<RA>(v);
#pragma unroll
        for (int k3 = 1; k3 < RA; ++k3) v[k3] = cmul(v[k3], ldg_c(WARP && TH <= 16 ? tw + L + k3 * TH + t : tw + t * k3));
#pragma unroll
        for (int k3 = 0; k3 < RA; ++k3) xch[base + (k3 * PITCH + t) * es] = v[k3];
        xch_sync<WARP>();
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int i = t + TH * q, k3 = i / RC, t1 = i % RC;
            if (RA % RB != 0 && k3 >= RA) continue;
            C* x = xch + base + (k3 * PITCH + t1) * es;
            C w[RB];
#pragma unroll
            for (int t2 = 0; t2 < RB; ++t2) w[t2] = x[t2 * RC * es];
            rdft<RB, false>(w);
            cnorm_all<RB>(w);
            x[0] = w[0];
#pragma unroll
            for (int k2 = 1; k2 < RB; ++k2) x[k2 * RC * es] = cmul(w[k2], ldg_c(tw + RA * t1 * k2));
        }
        xch_sync<WARP>();
#pragma unroll
        for (int q = 0; q < RA / RC; ++q) {
            const int i = t + TH * q, k3 = i % RA, k2 = i / RA;
            const C* x = xch + base + (k3 * PITCH + k2 * RC) * es;
#pragma unroll
            for (int t1 = 0; t1 < RC; ++t1) v[q * RC + t1] = x[t1 * es];
            rdft<RC, false>(v + q * RC);
            cnorm_all<RC>(v + q * RC);
        }
        xch_sync<WARP>();
    }

    template <bool WARP = false, typename C>
    __device__ __forceinline__ static void inv(C* v, C* xch, int base, int es, int t, const C* __restrict__ tw) {
#pragma unroll
        for (int q = 0; q < RA / RC; ++q) {
            const int i = t + TH * q, k3 = i % RA, k2 = i / RA;
            C* x = xch + base + (k3 * PITCH + k2 * RC) * es;
            rdft<RC, true>(v + q * RC);
            cnorm_all<RC>(v + q * RC);
#pragma unroll
            for (int t1 = 0; t1 < RC; ++t1) x[t1 * es] = v[q * RC + t1];
        }
        xch_sync<WARP>();
#pragma unroll
        for (int q = 0; q < QB; ++q) {
            const int i = t + TH * q, k3 = i / RC, t1 = i % RC;
            if (RA % RB != 0 && k3 >= RA) continue;
            C* x = xch + base + (k3 * PITCH + t1) * es;
            C w[RB];
            w[0] = x[0];
#pragma unroll
            for (int k2 = 1; k2 < RB; ++k2) w[k2] = cmulc(x[k2 * RC * es], ldg_c(tw + RA * t1 * k2));
            rdft<RB, true>(w);
            cnorm_all<RB>(w);
#pragma unroll
            for (int t2 = 0; t2 < RB; ++t2) x[t2 * RC * es] = w[t2];
        }
        xch_sync<WARP>();
        v[0] = xch[base + t * es];
#pragma unroll
        for (int k3 = 1; k3 < RA; ++k3)
            v[k3] = cmulc(xch[base + (k3 * PITCH + t) * es], ldg_c(WARP && TH <= 16 ? tw + L + k3 * TH + t : tw + t * k3));
        xch_sync<WARP>();
        rdft<RA, true>(v);   // v[m] = x[t + TH m]
        cnorm_all<RA>(v);
    }
};

// PlanQ<RA, 4, 4> for lines with private areas (line passes only: the exchange
// has unit stride). Rows of 16 values, the value of column x in row k3 at
// 16 k3 + (x ^ 5 (k3 mod 4)), and stage C's transforms dealt to the threads as k2 =
// t mod 4, k3 = t / 4 + 4 q: every access of a half warp (one line) then touches
// 16 distinct 8-byte banks in all three stages, where the padded rows of PlanQ
// take two passes in stages B and C, and a line takes L values instead of 21 RA
// (the float32 even-odd kernels at L = 192, 64 right-hand sides: 80.7 + 258 + 66.3
// to 68.9 + 230 + 58.0 us).
template <int RA>
struct PlanL {
    static constexpr int TH = 16, S = RA, L = 16 * RA, XLEN = L, XS = L + 1;
    static_assert(RA % 4 == 0, "four-point transforms");
    // slot s = 4 q + k1 of thread t holds X[t / 4 + 4 q + RA (t mod 4) + 4 RA k1]
    __host__ __device__ static constexpr int kidx(int t, int s) { return t / 4 + 4 * (s / 4) + RA * (t % 4) + 4 * RA * (s % 4); }
    __device__ __forceinline__ static int pos(int k3, int x) { return 16 * k3 + (x ^ (5 * (k3 & 3))); }

    template <bool ZHI, bool WARP, typename C>
    __device__ __forceinline__ static void fwd(C* v, C* xch, int base, int, int t, const C* __restrict__ tw) {
        C* x = xch + base;
        if constexpr (ZHI) rdft_zhi<RA, false>(v);
        else rdft<RA, false>(v);
        cnorm_all<RA>(v);
#pragma unroll
        for (int k3 = 1; k3 < RA; ++k3) v[k3] = cmul(v[k3], ldg_c(tw + L + k3 * 16 + t));
#pragma unroll
        for (int k3 = 0; k3 < RA; ++k3) x[pos(k3, t)] = v[k3];
        xch_sync<WARP>();
        const int t1 = t & 3, th = t >> 2;
#pragma unroll
        for (int q = 0; q < RA / 4; ++q) {   // row k3 = th + 4 q, so k3 mod 4 = th
            C* r = x + 16 * (th + 4 * q);
            C w[4];
#pragma unroll
            for (int t2 = 0; t2 < 4; ++t2) w[t2] = r[(t1 + 4 * t2) ^ (5 * th)];
            rdft4<false>(w[0], w[1], w[2], w[3]);
            cnorm_all<4>(w);
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2)
                r[(t1 + 4 * k2) ^ (5 * th)] = k2 == 0 ? w[0] : cmul(w[k2], ldg_c(tw + RA * t1 * k2));
        }
        xch_sync<WARP>();
#pragma unroll
        for (int q = 0; q < RA / 4; ++q) {
            const C* r = x + 16 * (th + 4 * q);
#pragma unroll
            for (int u1 = 0; u1 < 4; ++u1) v[4 * q + u1] = r[(u1 + 4 * t1) ^ (5 * th)];   // k2 = t mod 4
            rdft4<false>(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            cnorm_all<4>(v + 4 * q);
        }
        xch_sync<WARP>();
    }

    template <bool WARP, typename C>
    __device__ __forceinline__ static void inv(C* v, C* xch, int base, int, int t, const C* __restrict__ tw) {
        C* x = xch + base;
        const int t1 = t & 3, th = t >> 2;
#pragma unroll
        for (int q = 0; q < RA / 4; ++q) {
            C* r = x + 16 * (th + 4 * q);
            rdft4<true>(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
            cnorm_all<4>(v + 4 * q);
#pragma unroll
            for (int u1 = 0; u1 < 4; ++u1) r[(u1 + 4 * t1) ^ (5 * th)] = v[4 * q + u1];
        }
        xch_sync<WARP>();
#pragma unroll
        for (int q = 0; q < RA / 4; ++q) {
            C* r = x + 16 * (th + 4 * q);
            C w[4];
            w[0] = r[t1 ^ (5 * th)];
#pragma unroll
            for (int k2 = 1; k2 < 4; ++k2) w[k2] = cmulc(r[(t1 + 4 * k2) ^ (5 * th)], ldg_c(tw + RA * t1 * k2));
            rdft4<true>(w[0], w[1], w[2], w[3]);
            cnorm_all<4>(w);
#pragma unroll
            for (int t2 = 0; t2 < 4; ++t2) r[(t1 + 4 * t2) ^ (5 * th)] = w[t2];
        }
        xch_sync<WARP>();
        v[0] = x[pos(0, t)];
#pragma unroll
        for (int k3 = 1; k3 < RA; ++k3) v[k3] = cmulc(x[pos(k3, t)], ldg_c(tw + L + k3 * 16 + t));
        xch_sync<WARP>();
        rdft<RA, true>(v);   // v[m] = x[t + 16 m]
        cnorm_all<RA>(v);
    }
};

}  // namespace bae
