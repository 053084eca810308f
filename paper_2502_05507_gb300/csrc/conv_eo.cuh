// The even-odd schedule of the potential apply: three kernels instead of
// five, for a plane range whose rows fit in shared memory.
//
// The i pass of a pruned apply is a symmetric Toeplitz product over the n
// planes [p0, p1) (conv_direct.cuh), which the sums and differences of the
// mirrored planes i and n-1-i decouple into two products of half the size.
// The transforms along k and j act on each plane alike, so the sums and
// differences are taken where the sources enter, and undone where the
// potential leaves; between the two, the even and the odd half of the data
// are independent problems with m = n / 2 rows each (n rounded up to even):
//   k_eo_fwd : two real lines per complex transform, E + i O with E = x(i, j)
//              + x(i', j), O = x(i, j) - x(i', j), i' the mirrored plane;
//              spectra to A[kk][half][row][j] (transposed, so that the next
//              kernel reads its rows contiguously)
//   k_eo_mid : one CTA per (kk, half, right-hand side) holds the m rows of 2N
//              values in shared memory: transforms them along j, applies the
//              m x m product at every jj, transforms back and writes the rows
//              to the same place
//   k_eo_inv : the inverse of the first: two real lines out, v(i, j) = (E + O)
//              / 2 and v(i', j) = (E - O) / 2
// The 2N-wide rows (B of the five passes) never reach global memory: per
// plane and line 4 complex values of A move instead of 2 of A and 8 of B.
// (Plane counts below up to the figures of L = 512 are those of
// bae_problem_conv_planes, two more than are transformed on a window.)
// Measured at N = 128, 32 planes, 64 right-hand sides (five passes with the
// direct i pass / these): float32 789 / 468 us per apply (the middle pass 317:
// 70% of the issue slots, a fifth of HBM), double-float 3.21 / 2.77 ms (the
// float32 pipes). On the window of 96 nodes that torus fits: float32 357 us (the
// middle pass 230), double-float 1.87 ms (the middle pass 1.34).
// Rows of A hold the lines [q0, q1) only, and column 0 packs the real kk = 0
// and kk = N spectra as in the five passes (conv_geo.cuh).
#pragma once

#include "conv_direct.cuh"

namespace bae {

// Plans of the even-odd kernels: all threads of a line in one warp, but for
// the k passes of the 16-byte elements at L = 512.
template <typename T, int L> struct EoPlan { using type = Plan2<L>; };
template <> struct EoPlan<double, 256> { using type = Plan3_256; };
template <> struct EoPlan<dsf, 256> { using type = Plan3_256; };
template <typename T> struct EoPlan<T, 96> : PlanWin<T, 96> {};
template <typename T> struct EoPlan<T, 192> { using type = PlanL<12>; };
template <typename T> struct EoPlan<T, 384> : PlanWin<T, 384> {};
template <> struct EoPlan<float, 384> { using type = PlanL<24>; };
template <> struct EoPlan<double, 512> { using type = Plan3_512; };
template <> struct EoPlan<dsf, 512> { using type = Plan3_512; };

// k passes: P line pairs per CTA (8 pairs: 64- or 128-byte runs of j in the
// transposed rows)
template <typename T, int L> struct EoGeo {
    using C = cplx_t<T>;
    using PL = typename EoPlan<T, L>::type;
    static constexpr int TH = PL::TH, S = PL::S;
    // lines of the k passes XS values apart: 2 mod 16 (8-byte values) or odd, so
    // that the transposed accesses (lanes: 8 lines of 2 or 1 frequencies) touch
    // distinct banks
    static constexpr int XS = sizeof(C) == 8 ? (PL::XS + 12) / 16 * 16 + 2 : PL::XS;
    static constexpr int P = 8, KT = P * TH;
    static constexpr int RS = L + (sizeof(T) == 4 && TH < 32 ? TH : 0);
    static constexpr size_t SMEM_KF = (size_t)P * XS * sizeof(C) + (size_t)P * RS * sizeof(T);
    static constexpr size_t SMEM_KI = (size_t)P * XS * sizeof(C);
};

// Middle pass. SP: one CTA takes every second frequency along j (the even or
// the odd ones) by a transform of length N: half the shared memory per row
// and twice the CTAs, but both read the rows and each writes a part of the
// result, which the inverse k pass adds. RL: values per row, FR: frequencies
// below the middle one (the lanes).
template <typename T, int L, bool SP> struct EoMid {
    static constexpr int N = L / 2, RL = SP ? N : L, FR = RL / 2, NT = (FR + 31) / 32;
    using PL = typename EoPlan<T, RL>::type;
    static constexpr int TI = DirTile<T>::TI;
    // warps at most: small shapes run several CTAs of 8 warps per SM, large
    // ones one of 16. Float32 with 16 values per thread has an instantiation
    // of its own for the small shapes (three CTAs per SM: 80 registers), the
    // others one for both (128 registers: two small CTAs)
    static constexpr int max_warps(bool big) { return big ? 16 : 8; }
    static constexpr bool THREE = sizeof(T) == 4 && PL::S <= 16;
};

// Shape of the middle pass for n planes: rows m per half (mr: filled up to
// whole warps of the transforms), row blocks mb, warps w, tiles of 32
// frequencies per step tps, entries of gt tiles in shared memory at a time;
// w == 0: does not fit.
struct EoShape {
    int n = 0, m = 0, mr = 0, mb = 0, w = 0, tps = 0, gt = 0;
    bool big = false;
    size_t smem = 0;
};

template <typename T, int L, bool SP>
EoShape eo_shape(int planes) {
    using M = EoMid<T, L, SP>;
    using PL = typename M::PL;
    constexpr size_t SMEM_MAX = 227 * 1024, SMEM_TWO = 113 * 1024;
    EoShape s;
    s.n = planes + (planes & 1);
    s.m = s.n / 2;
    s.mb = (s.m + M::TI - 1) / M::TI;
    s.mr = (s.m + 32 / PL::TH - 1) / (32 / PL::TH) * (32 / PL::TH);
    const size_t rows = ((size_t)s.mr * PL::XS * sizeof(cplx_t<T>) + 15) / 16 * 16;
    // the entries and results of frequency 0, and the rows of entries that the blocks at
    // the edges address beyond the ends (and do not use)
    const size_t extra = (size_t)(s.n + 3 * M::TI * 32) * sizeof(T) + (size_t)s.m * sizeof(cplx_t<T>);
    for (s.gt = M::NT; s.gt >= 1; s.gt = s.gt > 1 ? (s.gt + 1) / 2 : 0) {
        s.smem = rows + (size_t)s.n * s.gt * 32 * sizeof(T) + extra;
        if (s.smem <= SMEM_MAX) break;
    }
    if (s.gt < 1) return s;
    s.big = s.smem > SMEM_TWO || s.mb > M::max_warps(false);
    const int maxw = M::max_warps(s.big);
    if (s.mb > maxw) return s;
    s.tps = std::max(1, std::min(s.gt, maxw / s.mb));
    const int wf = s.mr * PL::TH / 32;   // warps that transform every row at once
    s.w = std::min(maxw, std::max(s.mb * s.tps, wf));
    return s;
}

namespace {

template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(d), "l"(src), "n"(BYTES) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// ------------------------------------------------------------ k pass (R2C)
// Tile (row r, block of P lines j) of right-hand side b.
template <typename T, int L>
__global__ void __launch_bounds__(EoGeo<T, L>::KT) k_eo_fwd(ConvArgs<T> a, int n, int njb) {
    wait_prior_grid();
    using C = cplx_t<T>;
    using G = EoGeo<T, L>;
    using PL = typename G::PL;
    constexpr int N = L / 2, TH = G::TH, S = G::S, P = G::P;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* xch = reinterpret_cast<C*>(smem_raw);              // P * XS
    T* rho = reinterpret_cast<T*>(xch + P * G::XS);       // P * RS: line i, line i'

    const int b = blockIdx.y;
    if (a.active && !a.active[b]) return;
    const int r = blockIdx.x / njb, jb = blockIdx.x - r * njb;
    const int q0 = a.line_lo(), nj = a.line_hi() - q0, m = n / 2;
    const int j0 = jb * P, cnt = min(P, nj - j0);         // the CTA's lines q0 + j0 + [0, cnt)
    const int pi = a.plane_lo() + r, pj = a.plane_lo() + n - 1 - r;
    const bool two = pj < a.plane_hi();                   // the mirrored plane exists
    const int t = threadIdx.x % TH, p = threadIdx.x / TH;
    const bool on = p < cnt;
    const int NG = a.N;   // the grid's pitch; first lines of the grid:
    const long long la = (long long)(pi + a.w0) * NG + q0 + j0 + a.w1, lb = (long long)(pj + a.w0) * NG + q0 + j0 + a.w1;
    const T zero = dir_zero(T());

    C v[S];
    if (a.mode == SRC_DENSITY) {
        T* ro = rho + p * G::RS;
        for (int k = t; k < 2 * N; k += TH) {
            const bool first = k < N;
            ro[k] = (on && (first || two))
                        ? volume_or_zero(a, b, ((first ? la : lb) + p) * NG + a.w2 + (first ? k : k - N)) : zero;
        }
        __syncthreads();
        const double* q = a.q + (long long)b * a.q_stride + (a.q_row ? (long long)a.q_row[b] * a.q_row_stride : 0);
        const float* q32 = a.q32 ? a.q32 + (long long)b * a.q32_stride : nullptr;
        const int a0 = a.rec.line_off[la], na = a.rec.line_off[la + cnt] - a0;
        const int b0 = two ? a.rec.line_off[lb] : 0, nb = two ? a.rec.line_off[lb + cnt] - b0 : 0;
        for (int e = threadIdx.x; e < na + nb; e += blockDim.x) {
            const bool first = e < na;
            const int s = first ? a0 + e : b0 + e - na;
            const int x = a.rec.src_lin[s] - (int)((first ? la : lb) * NG);   // (line, k) within the CTA's lines
            rho[(x / NG) * G::RS + (first ? 0 : N) + x % NG - a.w2] = source_value<T>(a.rec, s, q, q32);
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int x = t + TH * s;
            v[s] = s < S / 2 ? cmake<C>(ro[x] + ro[N + x], ro[x] - ro[N + x]) : cmake<C>(zero, zero);
        }
    } else {
        const double* f = a.f + (long long)b * NG * NG * NG;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            T va = zero, vb = zero;
            if (s < S / 2 && on) {
                const long long xa = (la + p) * NG + a.w2 + t + TH * s, xb = (lb + p) * NG + a.w2 + t + TH * s;
                if (a.flags[xa] & 1) va = (T)(a.scale * f[swap_axes(xa, a.f_swap, NG)]);
                if (two && (a.flags[xb] & 1)) vb = (T)(a.scale * f[swap_axes(xb, a.f_swap, NG)]);
            }
            v[s] = cmake<C>(va + vb, va - vb);
        }
    }
    PL::template fwd<true, true>(v, xch, p * G::XS, 1, t, a.tw);
    C* z = xch + p * G::XS;
#pragma unroll
    for (int s = 0; s < S; ++s) z[PL::kidx(t, s)] = v[s];
    __syncthreads();
    // transposed store: the lines of the CTA are consecutive in a row of A
    C* A = a.A + (long long)b * N * N * (N + 1);
    for (int e = threadIdx.x; e < P * N; e += G::KT) {
        const int pp = e % P, k = e / P;
        if (pp >= cnt) continue;
        C xe, xo;
        split_lines(xch + pp * G::XS, k, L, xe, xo);
        C* o = A + ((long long)k * 2 * m + r) * nj + j0 + pp;
        o[0] = xe;
        o[(long long)m * nj] = xo;
    }
}

// ------------------------------------------------------------ k pass (C2R)
template <typename T, int L, bool SP>
__global__ void __launch_bounds__(EoGeo<T, L>::KT) k_eo_inv(ConvArgs<T> a, int n, int njb) {
    wait_prior_grid();
    using C = cplx_t<T>;
    using G = EoGeo<T, L>;
    using PL = typename G::PL;
    constexpr int N = L / 2, TH = G::TH, S = G::S, P = G::P;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    C* xch = reinterpret_cast<C*>(smem_raw);              // P * XS

    const int b = blockIdx.y;
    if (a.active && !a.active[b]) return;
    const int r = blockIdx.x / njb, jb = blockIdx.x - r * njb;
    const int q0 = a.line_lo(), nj = a.line_hi() - q0, m = n / 2;
    const int j0 = jb * P, cnt = min(P, nj - j0);
    const int pi = a.plane_lo() + r, pj = a.plane_lo() + n - 1 - r;
    const bool two = pj < a.plane_hi();
    const int t = threadIdx.x % TH, p = threadIdx.x / TH;

    // z[k] = E[k] + i O[k] of every line, the upper half by symmetry
    // (SP: the sum of the parts of the even and of the odd frequencies)
    const C* A = SP ? a.B + (long long)b * N * 2 * N * (N + 1) : a.A + (long long)b * N * N * (N + 1);
    const long long part = (long long)2 * N * m * nj;
#pragma unroll 4
    for (int e = threadIdx.x; e < P * N; e += G::KT) {
        const int pp = e % P, k = e / P;
        if (pp >= cnt) continue;
        const C* in = A + ((long long)k * 2 * m + r) * nj + j0 + pp;
        C xe = in[0], xo = in[(long long)m * nj];
        if (SP) {
            xe = cadd(xe, in[part]);
            xo = cadd(xo, in[part + (long long)m * nj]);
        }
        C* z = xch + pp * G::XS;
        if (k == 0) {
            z[0] = cmake<C>(xe.x, xo.x);
            z[N] = cmake<C>(xe.y, xo.y);
        } else {
            z[k] = cmake<C>(xe.x - xo.y, xe.y + xo.x);
            z[L - k] = cmake<C>(xe.x + xo.y, xo.x - xe.y);
        }
    }
    __syncthreads();
    C v[S];
    const C* z = xch + p * G::XS;
#pragma unroll
    for (int s = 0; s < S; ++s) v[s] = z[PL::kidx(t, s)];
    xch_sync<TH <= 32>();
    PL::template inv<true>(v, xch, p * G::XS, 1, t, a.tw);
    if (p < cnt) {
        const int NG = a.N;
        typename OutOf<T>::type* out = a.v + (long long)b * NG * NG * NG + a.w2;
        const long long la = (long long)(pi + a.w0) * NG + q0 + j0 + a.w1 + p;
        const long long lb = (long long)(pj + a.w0) * NG + q0 + j0 + a.w1 + p;
#pragma unroll
        for (int s = 0; s < S / 2; ++s) {
            const int x = t + TH * s;
            out[la * NG + x] = to_out(dir_half(v[s].x + v[s].y));
            if (two) out[lb * NG + x] = to_out(dir_half(v[s].x - v[s].y));
        }
    }
}

// ------------------------------------------------- middle pass (j, i, j^-1)
// entry g(|i-j|) +- g(n-1-i-j): one fused multiply-add with the sign, or the
// sum with a value flipped when it was loaded (double-float)
template <typename T>
__device__ __forceinline__ T eo_sign(T, bool odd) { return odd ? (T)-1 : (T)1; }
__device__ __forceinline__ dsf eo_sign(dsf, bool) { return dsf(0.f, 0.f); }
template <typename T>
__device__ __forceinline__ T eo_flip(T h, bool) { return h; }
__device__ __forceinline__ dsf eo_flip(dsf h, bool odd) { return odd ? -h : h; }
__device__ __forceinline__ float eo_entry(float t, float h, float sgn) { return __fmaf_rn(sgn, h, t); }
__device__ __forceinline__ double eo_entry(double t, double h, double sgn) { return __fma_rn(sgn, h, t); }
__device__ __forceinline__ dsf eo_entry(dsf t, dsf h, dsf) { return add_nr(t, h); }

// acc = rows [TI ib, TI ib + TI) of the m x m product of one half, for the
// four real vectors of the values at pa[j * pitch] and pb[j * pitch], j < m:
// entries g(|i-j|) +- g(n-1-i-j), g(d) at gs[d * 32]. Blocks off the diagonal
// address g(|i-j|) forwards or backwards from one base, so every shared-memory
// load has a compile-time offset. Rows i >= m and the windows' ends beyond
// [0, n) read whatever lies there; their products are not stored.
template <typename T, typename C>
__device__ __forceinline__ void eo_product(T (&acc)[DirTile<T>::TI][4], const T* gs, bool odd, int n, int m, int ib,
                                           const C* pa, const C* pb, int pitch) {
    constexpr int TI = DirTile<T>::TI, TJ = DirTile<T>::TJ, NW = TI + TJ - 1;
#pragma unroll
    for (int i = 0; i < TI; ++i)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[i][v] = dir_zero(T());
    const T sgn = eo_sign(T(), odd);
    auto block = [&](int jb, int cnt, auto whole) {
        T tw[NW], hw[NW];
        const int d = TI * (ib - jb);   // i - j = d + w - (TJ - 1)
        if (d > 0) {
            const T* g = gs + (d - (TJ - 1)) * 32;
#pragma unroll
            for (int w = 0; w < NW; ++w) tw[w] = g[w * 32];
        } else if (d < 0) {
            const T* g = gs + (-d + (TJ - 1)) * 32;
#pragma unroll
            for (int w = 0; w < NW; ++w) tw[w] = g[-w * 32];
        } else {
#pragma unroll
            for (int w = 0; w < TJ; ++w) tw[TJ - 1 + w] = tw[TJ - 1 - w] = gs[w * 32];
        }
        const T* h = gs + (n - 1 - TI * (ib + jb)) * 32;
#pragma unroll
        for (int w = 0; w < NW; ++w) hw[w] = eo_flip(h[-w * 32], odd);
#pragma unroll
        for (int j = 0; j < TJ; ++j) {
            if (decltype(whole)::value || j < cnt) {
                const C xa = pa[(TJ * jb + j) * pitch], xb = pb[(TJ * jb + j) * pitch];
#pragma unroll
                for (int i = 0; i < TI; ++i) {
                    const T p = eo_entry(tw[i - j + TJ - 1], hw[i + j], sgn);
                    dir_fma(acc[i][0], p, xa.x);
                    dir_fma(acc[i][1], p, xa.y);
                    dir_fma(acc[i][2], p, xb.x);
                    dir_fma(acc[i][3], p, xb.y);
                }
            }
        }
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[i][v] = dir_norm(acc[i][v]);
    };
    const int full = m / TJ;
    for (int jb = 0; jb < full; ++jb) block(jb, TJ, std::true_type{});
    if (full * TJ < m) block(full, m - full * TJ, std::false_type{});
}

__device__ __forceinline__ float dir_shfl(float a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ double dir_shfl(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ dsf dir_shfl(dsf a, int o) { return dsf(dir_shfl(a.hi, o), dir_shfl(a.lo, o)); }

// frequency 0, its own mirror image: a warp per row, lanes over the products,
// results to y[m]; entries g(d) at g0[d]
template <typename T, typename C>
__device__ __forceinline__ void eo_single(const C* col, int pitch, const T* g0, bool odd, int n, int m, C* y) {
    const int lane = threadIdx.x & 31, nwarp = blockDim.x >> 5;
    for (int i = threadIdx.x >> 5; i < m; i += nwarp) {
        T yr = dir_zero(T()), yi = dir_zero(T());
        for (int j = lane; j < m; j += 32) {
            const C x = col[j * pitch];
            const T t = g0[abs(i - j)], h = g0[n - 1 - i - j];
            const T p = t + (odd ? -h : h);
            dir_fma(yr, p, x.x);
            dir_fma(yi, p, x.y);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            yr = yr + dir_shfl(yr, o);
            yi = yi + dir_shfl(yi, o);
        }
        if (lane == 0) y[i] = cmake<C>(yr, yi);
    }
}

// One half (even or odd) of column kk <= N (kk = 0 and N: the real and the
// imaginary part of column 0 as real rows) of right-hand side b; SP: the
// frequencies of parity par along j.
// Grid x: (column kk, half, parity), y: right-hand side.
template <typename T, int L, bool SP, int MAXW, int MINB>
__global__ void __launch_bounds__(MAXW * 32, MINB) k_eo_mid(ConvArgs<T> a, EoShape sh) {
    using C = cplx_t<T>;
    using M = EoMid<T, L, SP>;
    using PL = typename M::PL;
    constexpr int N = L / 2, N1 = N + 1, RL = M::RL, FR = M::FR, NT = M::NT;
    constexpr int TH = PL::TH, S = PL::S, XS = PL::XS, TI = M::TI;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int n = sh.n, m = sh.m, n0 = a.plane_hi() - a.plane_lo();
    C* rows = reinterpret_cast<C*>(smem_raw);                     // [mr][XS]
    // [gt][n][32], on a 16-byte boundary, room for 2 TI rows before and TI behind
    T* gs = reinterpret_cast<T*>(smem_raw + ((size_t)sh.mr * XS * sizeof(C) + 15) / 16 * 16) + 2 * TI * 32;
    C* y0 = reinterpret_cast<C*>(gs + ((size_t)sh.gt * n + TI) * 32);   // [m]
    T* g0 = reinterpret_cast<T*>(y0 + m);                               // [n]
    const int b = blockIdx.y;
    const int par = SP ? blockIdx.x & 1 : 0, kh = SP ? blockIdx.x >> 1 : blockIdx.x, kk = kh >> 1;
    const bool odd = kh & 1;
    const int tid = threadIdx.x, nth = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nth >> 5;
    // value c of a row is frequency c (SP: 2 c + par); lane f of the tiles
    // holds c = f + c1 and its mirror image
    const int c1 = SP && par ? 0 : 1, jstep = SP ? 2 : 1;
    // g is symmetric in the two frequencies: row kk holds those along j in
    // order, c = 1 on a 16-byte boundary (mix_index)
    const long long dstride = mix_index(N, 1, 0, 0) - mix_index(N, 0, 0, 0);
    const T* gk = a.gmix + mix_index(N, 0, kk, 0);
    auto load_entries = [&](int first, int count) {
        if constexpr (!SP && FR % 32 == 0) {
            constexpr int V = 16 / sizeof(T), LV = 32 / V;   // values per piece, pieces per 32
            for (int d = tid / LV; d < n; d += nth / LV) {
                const T* src = gk + min(d, n0 - 1) * dstride + 1 + first * 32 + tid % LV * V;
                T* dst = gs + d * 32 + tid % LV * V;
                for (int tile = 0; tile < count; ++tile) cp_async<16>(dst + (size_t)tile * n * 32, src + tile * 32);
            }
        } else {
            for (int d = warp; d < n; d += nwarp) {
                const T* src = gk + min(d, n0 - 1) * dstride + jstep * (first * 32 + lane + c1) + (SP ? par : 0);
                T* dst = gs + d * 32 + lane;
                for (int tile = 0; tile < count; ++tile)
                    if (FR % 32 == 0 || (first + tile) * 32 + lane < FR)
                        cp_async<sizeof(T)>(dst + (size_t)tile * n * 32, src + jstep * tile * 32);
            }
        }
    };
    // the entries do not depend on the kernel before
    load_entries(0, min(sh.gt, NT));
    for (int d = tid; d < n; d += nth) cp_async<sizeof(T)>(g0 + d, gk + min(d, n0 - 1) * dstride);
    wait_prior_grid();
    if (a.active && !a.active[b]) {   // whole CTA
        cp_async_wait();
        return;
    }
    const int q0 = a.line_lo(), nj = a.line_hi() - q0;
    const long long rowbase = (long long)(2 * (kk == N ? 0 : kk) + (odd ? 1 : 0)) * m * nj;
    const C* A = a.A + (long long)b * N * N * N1 + rowbase;
    C* out = SP ? a.B + (long long)b * N * 2 * N * N1 + (long long)par * 2 * N * m * nj + rowbase : const_cast<C*>(A);
    const bool realrow = kk == 0 || kk == N;
    const C zero = cmake<C>(dir_zero(T()), dir_zero(T()));
    const int t = tid % TH, slot = tid / TH, nslot = nth / TH;

    // ---- along j, rows in place (rows m..mr fill up the last warp)
    for (int r = slot; r < sh.mr; r += nslot) {
        C v[S];
        const int jr = r < m ? nj : 0;   // a missing row has no values
        const C* in = A + (long long)r * nj - q0;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            v[s] = zero;
            if ((SP || s < S / 2) && (unsigned)(t + TH * s - q0) < (unsigned)jr) {
                if (!realrow) v[s] = in[t + TH * s];
                else v[s].x = reinterpret_cast<const T*>(in + t + TH * s)[kk == N];   // the other part is another CTA's
            }
        }
        if (SP && par) {
#pragma unroll
            for (int s = 0; s < S; ++s) v[s] = cmul(v[s], ldg_c(a.tw + t + TH * s));
        }
        C* row = rows + (size_t)r * XS;
        PL::template fwd<!SP, true>(v, row, 0, 1, t, a.tw + (SP ? 2 * L : 0));
#pragma unroll
        for (int s = 0; s < S; ++s) row[PL::kidx(t, s)] = v[s];
    }
    cp_async_wait();
    __syncthreads();

    // ---- along i: a step's warps hold one row block of one tile each and
    // write after all have read
    if (c1) eo_single(rows, XS, g0, odd, n, m, y0);
    const int tl = warp / sh.mb, ib = warp - tl * sh.mb;
    for (int first = 0; first < NT; first += sh.gt) {
        const int last = min(first + sh.gt, NT);
        if (first > 0) {
            __syncthreads();   // the entries before are read
            load_entries(first, last - first);
            cp_async_wait();
            __syncthreads();
        }
        for (int t0 = first; t0 < last; t0 += sh.tps) {
            const bool act = tl < sh.tps && t0 + tl < last;
            const int f = (t0 + tl) * 32 + lane;
            const int c = min(f, FR - 1) + c1;   // its mirror image: RL - c, or RL - 1 - c for the odd frequencies
            C* pa = rows + c;
            C* pb = rows + RL - 1 + c1 - c;
            T acc[TI][4];
            if (act) eo_product(acc, gs + (size_t)(t0 - first + tl) * n * 32 + lane, odd, n, m, ib, pa, pb, XS);
            __syncthreads();
            if (c1 && t0 == 0)
                for (int r = tid; r < m; r += nth) rows[(size_t)r * XS] = y0[r];
            if (act && f < FR) {
#pragma unroll
                for (int i = 0; i < TI; ++i) {
                    const int r = TI * ib + i;
                    if (r < m) {   // the middle frequency is its own image: the same value twice
                        pa[r * XS] = cmake<C>(acc[i][0], acc[i][1]);
                        pb[r * XS] = cmake<C>(acc[i][2], acc[i][3]);
                    }
                }
            }
        }
    }
    __syncthreads();

    // ---- back along j
    for (int r = slot; r < sh.mr; r += nslot) {
        C* row = rows + (size_t)r * XS;
        C v[S];
#pragma unroll
        for (int s = 0; s < S; ++s) v[s] = row[PL::kidx(t, s)];
        __syncwarp();
        PL::template inv<true>(v, row, 0, 1, t, a.tw + (SP ? 2 * L : 0));
        const int jr = r < m ? nj : 0;
        C* o = out + (long long)r * nj - q0;
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int x = t + TH * s;
            if ((SP || s < S / 2) && (unsigned)(x - q0) < (unsigned)jr) {
                C y = v[s];
                if (SP && par) y = cmulc(y, ldg_c(a.tw + x));
                if (!realrow) o[x] = y;
                else reinterpret_cast<T*>(o + x)[kk == N] = y.x;
            }
        }
    }
}

template <typename T, int L, bool SP>
void eo_launch(const ConvArgs<T>& a, const EoShape& sh, cudaStream_t st) {
    using G = EoGeo<T, L>;
    constexpr int N = L / 2;
    const int njb = ceil_div(a.line_hi() - a.line_lo(), G::P);
    const dim3 gk(sh.m * njb, a.nbatch), gm(2 * (N + 1) * (SP ? 2 : 1), a.nbatch);
    BAE_LAUNCH(kname<T>("conv_eo_fwd.f32", "conv_eo_fwd.f64", "conv_eo_fwd.df64"), st,
               launch_pdl(k_eo_fwd<T, L>, gk, G::KT, G::SMEM_KF, st, a, sh.n, njb));
    auto mid = k_eo_mid<T, L, SP, 16, 1>;
    if constexpr (EoMid<T, L, SP>::THREE)
        if (!sh.big) mid = k_eo_mid<T, L, SP, 8, 3>;
    BAE_LAUNCH(kname<T>("conv_eo_mid.f32", "conv_eo_mid.f64", "conv_eo_mid.df64"), st,
               launch_pdl(mid, gm, sh.w * 32, sh.smem, st, a, sh));
    BAE_LAUNCH(kname<T>("conv_eo_inv.f32", "conv_eo_inv.f64", "conv_eo_inv.df64"), st,
               launch_pdl(k_eo_inv<T, L, SP>, gk, G::KT, G::SMEM_KI, st, a, sh.n, njb));
}

}  // namespace

// Sets the kernel attributes (once per process).
template <typename T, int L>
void eo_configure() {
    using G = EoGeo<T, L>;
    static const bool configured = []() {
        auto set = [](auto k, size_t smem) {
            BAE_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        };
        if constexpr (!EoUse<T, L>::none) set(k_eo_fwd<T, L>, G::SMEM_KF);
        auto set_form = [&](auto split) {
            constexpr bool SP = decltype(split)::value;
            set(k_eo_inv<T, L, SP>, G::SMEM_KI);
            set(k_eo_mid<T, L, SP, 16, 1>, 227 * 1024);
            if constexpr (EoMid<T, L, SP>::THREE) set(k_eo_mid<T, L, SP, 8, 3>, 113 * 1024);
        };
        if constexpr (EoUse<T, L>::whole) set_form(std::false_type{});
        if constexpr (EoUse<T, L>::split) set_form(std::true_type{});
        return true;
    }();
    (void)configured;
}

// Planes up to which the schedule is taken where it fits: its products grow
// with n^2, the FFT i pass of the other schedules does not. The lines lie
// where the two meet (mixed solves of spheres, all convolution kernels of one
// float32 apply in microseconds, the five passes or plane kernels / these):
//   float32 N = 128, one right-hand side: 44 planes 61.6 / 36.2, 64 65.1 /
//     40.7, 96 70.3 / 56.6, 108 74.7 / 69.1; 32: 44 planes 824 / 327, 96
//     1234 / 1075, 108 1344 / 1392
//   float32 N = 256, one: 82 planes 318 / 151, 108 351 / 212, 134 395 / 352;
//     four: 82 1148 / 546, 134 1451 / 1283
//   double-float N = 128, boundary operator, one: 50 planes 190 / 112, 66
//     222 / 164, 82 234 / 290
//   float64 N = 128, boundary operator, one: 26 planes 892 / 223, 64 1032 /
//     623, 82 1117 / 996, 102 1231 / 1398
// and at N <= 64 it is the faster one for every plane count (float32 N = 64:
// 16 planes 60.9 / 54.9, 60 planes 63.8 / 63.5 with the call around it).
// On windows, against the five passes on the same window:
//   float32 96 nodes, one: 44 planes 48.6 / 34.7, 82 57.2 / 49.5, 96 59.6 / 57.5;
//     32: 44 planes 491 / 249, 96 859 / 854
//   float32 192 nodes, one: 82 planes 122 / 106, 108 187 / 159, 134 208 / 248
//   double-float 192 nodes, operator, one: 82 planes 748 / 573, 96 772 / 690 (both
//     sides 4 to 7% less than now: their sums were not put in order); 96 nodes up to
//     64 planes (beyond, nine row blocks leave warps idle)
//   float64 96 and 192 nodes: never (EoUse; the even-odd schedule / the passes
//     with the direct i pass: 96 nodes 44 planes 299 / 266, 192 nodes 82 planes
//     2073 / 1945; the FP64 pipe bounds both).
// At L = 512 (the whole grid at N = 256) every type takes it as far as its rows fit,
// against the five passes with the direct i pass (bodies of 210 x 120 nodes, operator,
// one; the 8-byte types fit to 96 planes):
//   float32 44 planes 116 / 100, 92 277 / 206, 124 384 / 341
//   double-float 16 planes 116 / 110, 44 390 / 361, 60 518 / 520, 92 1031 / 978
//   float64 16 planes 413 / 387, 44 1498 / 1427, 92 4330 / 4064
template <typename T, int L>
constexpr int eo_limit() {
    if constexpr (L == 512) return 144;
    else if constexpr (L == 192 && std::is_same<T, dsf>::value) return 64;
    else if constexpr (L == 384) return sizeof(T) == 4 ? 116 : 96;
    else if constexpr (L >= 192) return sizeof(T) == 4 ? 104 : (std::is_same<T, dsf>::value ? 72 : 86);
    else return L / 2;
}

// The form an apply takes, by the element type, L and the plane range only
// (so that a batch and a single right-hand side give the same bits): 0 none,
// 1 whole rows, 2 split frequencies. Whole rows where they fit (float32 N =
// 128, 96 planes, 32 right-hand sides: 1075 against 1446 us split, which
// reads A twice and adds two parts); at L = 512 only where two CTAs fit an SM
// (82 planes: 173 us whole, one CTA per SM, against 151 us split).
template <typename T, int L>
int eo_form(const ConvArgs<T>& a, EoShape& sh) {
    if (a.box || !a.gmix) return 0;
    const int planes = a.plane_hi() - a.plane_lo();
    if (planes > eo_limit<T, L>()) return 0;
    if constexpr (EoUse<T, L>::whole) {
        sh = eo_shape<T, L, false>(planes);
        if (sh.w > 0 && !(L >= 384 && sh.big)) return 1;
    }
    if constexpr (EoUse<T, L>::split) {
        sh = eo_shape<T, L, true>(planes);
        if (sh.w > 0) return 2;
    }
    return 0;
}

template <typename T, int L>
bool eo_runs(const ConvArgs<T>& a) {
    EoShape sh;
    return eo_form<T, L>(a, sh) != 0;
}

template <typename T, int L>
bool eo_apply(const ConvArgs<T>& a, cudaStream_t st) {
    EoShape sh;
    const int form = eo_form<T, L>(a, sh);
    if (form == 0) return false;
    eo_configure<T, L>();
    if constexpr (EoUse<T, L>::whole)
        if (form == 1) eo_launch<T, L, false>(a, sh, st);
    if constexpr (EoUse<T, L>::split)
        if (form == 2) eo_launch<T, L, true>(a, sh, st);
    return true;
}

}  // namespace bae
