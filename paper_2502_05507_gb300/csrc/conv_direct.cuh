// The i pass as a direct sum (the alternative to the FFT i pass of
// conv_impl.cuh).
//
// After the k and j transforms the convolution with G_s is diagonal in
// (jj, kk) and a real, even convolution along i:
//   y(i) = sum_i' g(|i - i'|; jj, kk) x(i'),   i, i' in the planes [p0, p1),
// with g(d; jj, kk) = 1/(2N)^2 sum over the other two offsets of G_s(d, ., .)
// times the two cosines (the LGF spectrum before its transform along the
// first axis, the mixed form of the spectrum). The FFT i pass transforms 2N values per pencil
// whatever the number n of planes; the sum costs n^2 products, needs no
// padding, no twiddles and no exchange, and for the plane counts that the
// pruned applies have it is the cheaper form (see direct_i_limit). Measured
// at N = 128 with 32 planes, the FFT over the few nonzero rows before / the
// sum: 64 right-hand sides float32 921 / 332 us, double-float 7150 / 1525 us
// per launch (bound by the float32 pipes; the float32 sum moves its 1.1 GB at
// 3.2 TB/s); one right-hand side float64 723 / 104 us (the FP64 pipe).
//
// g is symmetric and Toeplitz, hence centrosymmetric: with n even and
// m = n / 2, the sums e(j) = x(j) + x(n-1-j) and differences o(j) = x(j) -
// x(n-1-j) decouple,
//   y(i) +- y(n-1-i) = sum_{j<m} (g(|i-j|) +- g(n-1-i-j)) {e, o}(j),
// two m x m products per real vector instead of one n x n. The entries
// g +- g are formed in registers and used for four real vectors: the real
// and imaginary parts of the pencils jj and 2N - jj, which have the same g.
//
// Column 0 holds the kk = 0 and kk = N spectra packed (conv_geo.cuh): its
// slots jj < N have g(.; jj, 0), its slots jj > N have g(.; 2N - jj, N), and
// at jj = 0 and N the real part has the former and the imaginary part the
// latter. Its real and imaginary parts are separate vectors of extra CTAs.
#pragma once

#include "conv_geo.cuh"

namespace bae {

namespace {

// output rows (of the m e/o rows) per warp pass and input rows per step: the
// accumulators of TI rows (e and o, four real vectors) and the two windows
// of TI + TJ - 1 entries stay in registers (float32 ~115; 8-byte types at 4
// rows ~130)
template <typename T> struct DirTile {
    static constexpr int TI = sizeof(T) == 4 ? 8 : 4, TJ = TI;
    static constexpr int MAXW = 16;   // warps per CTA at most
};

// acc += p x; for double-float the product's error, its cross terms and the
// sum's error go to the low part (12 float operations). The low part's own
// rounding grows with it, so dir_norm puts the sum in order after every block
// of TJ terms.
__device__ __forceinline__ void dir_fma(float& acc, float p, float x) { acc = __fmaf_rn(p, x, acc); }
__device__ __forceinline__ void dir_fma(double& acc, double p, double x) { acc = __fma_rn(p, x, acc); }
__device__ __forceinline__ void dir_fma(dsf& acc, dsf p, dsf x) {
    const float h = __fmul_rn(p.hi, x.hi);
    float e = __fmaf_rn(p.hi, x.hi, -h);
    e = __fmaf_rn(p.hi, x.lo, e);
    e = __fmaf_rn(p.lo, x.hi, e);
    const dsf s = two_sum(acc.hi, h);
    acc = dsf(s.hi, __fadd_rn(acc.lo, __fadd_rn(s.lo, e)));
}
__device__ __forceinline__ float dir_norm(float a) { return a; }
__device__ __forceinline__ double dir_norm(double a) { return a; }
__device__ __forceinline__ dsf dir_norm(dsf a) { return fast_two_sum(a.hi, a.lo); }
__device__ __forceinline__ float dir_half(float a) { return 0.5f * a; }
__device__ __forceinline__ double dir_half(double a) { return 0.5 * a; }
__device__ __forceinline__ dsf dir_half(dsf a) { return dsf(0.5f * a.hi, 0.5f * a.lo); }
__device__ __forceinline__ float dir_zero(float) { return 0.f; }
__device__ __forceinline__ double dir_zero(double) { return 0.0; }
__device__ __forceinline__ dsf dir_zero(dsf) { return dsf(0.f, 0.f); }

// NV real vectors of one lane, in units of at most 16 bytes: unit u of lane
// l of a row sits at [row][u][l], so that the lanes of a warp read
// consecutive 16-byte (8-, 4-byte) words
template <typename T, int NV> struct DirRow {
    static constexpr int UV = (int)(16 / sizeof(T)) < NV ? (int)(16 / sizeof(T)) : NV;   // vectors per unit
    static constexpr int NU = NV / UV;
    struct __align__(sizeof(T) * UV) Unit { T v[UV]; };
    __device__ __forceinline__ static void put(Unit* row, int lane, const T* x) {
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            Unit w;
#pragma unroll
            for (int k = 0; k < UV; ++k) w.v[k] = x[u * UV + k];
            row[u * 32 + lane] = w;
        }
    }
    __device__ __forceinline__ static void get(const Unit* row, int lane, T* x) {
#pragma unroll
        for (int u = 0; u < NU; ++u) {
            const Unit w = row[u * 32 + lane];
#pragma unroll
            for (int k = 0; k < UV; ++k) x[u * UV + k] = w.v[k];
        }
    }
};

// The m x m products of one group of 32 lanes: rows `xs` ([mp][e, o][units],
// mp = m rounded up to whole blocks, zero beyond m) and entries `gs`
// ([n][32]) in shared memory; store(i, v) gets y(i), y(n-1-i) of vector v.
template <typename T, int NV, typename Store>
__device__ __forceinline__ void direct_rows_product(const typename DirRow<T, NV>::Unit* xs, const T* gs, int n, int mb,
                                                    int lane, int warp, int nwarp, Store store) {
    using R = DirRow<T, NV>;
    constexpr int TI = DirTile<T>::TI, TJ = DirTile<T>::TJ, NW = TI + TJ - 1;
    for (int ib = warp; ib < mb; ib += nwarp) {
        T ae[TI][NV], ao[TI][NV];
#pragma unroll
        for (int i = 0; i < TI; ++i)
#pragma unroll
            for (int v = 0; v < NV; ++v) ae[i][v] = ao[i][v] = dir_zero(T());
        for (int jb = 0; jb < mb; ++jb) {
            // g(|i - j|) for i - j = TI ib - TJ jb - (TJ - 1) + w and
            // g(n-1-i-j) for i + j = TI ib + TJ jb + w (rows beyond m
            // multiply zeros or are not stored: any entry in range does)
            T tw[NW], hw[NW];
#pragma unroll
            for (int w = 0; w < NW; ++w) {
                tw[w] = gs[min(abs(TI * ib - TJ * jb - (TJ - 1) + w), n - 1) * 32 + lane];
                hw[w] = gs[min(abs(n - 1 - (TI * ib + TJ * jb + w)), n - 1) * 32 + lane];
            }
#pragma unroll
            for (int j = 0; j < TJ; ++j) {
                T xe[NV], xo[NV];
                const typename R::Unit* row = xs + (long long)(TJ * jb + j) * 2 * R::NU * 32;
                R::get(row, lane, xe);
                R::get(row + R::NU * 32, lane, xo);
#pragma unroll
                for (int i = 0; i < TI; ++i) {
                    const T t = tw[i - j + TJ - 1], h = hw[i + j];
                    const T p = t + h, q = t - h;
#pragma unroll
                    for (int v = 0; v < NV; ++v) {
                        dir_fma(ae[i][v], p, xe[v]);
                        dir_fma(ao[i][v], q, xo[v]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < TI; ++i)
#pragma unroll
                for (int v = 0; v < NV; ++v) {
                    ae[i][v] = dir_norm(ae[i][v]);
                    ao[i][v] = dir_norm(ao[i][v]);
                }
        }
#pragma unroll
        for (int i = 0; i < TI; ++i) {
            T lo[NV], hi[NV];
#pragma unroll
            for (int v = 0; v < NV; ++v) {
                lo[v] = dir_half(ae[i][v] + ao[i][v]);
                hi[v] = dir_half(ae[i][v] - ao[i][v]);
            }
            store(TI * ib + i, lo, hi);
        }
    }
}

// One CTA per 32 pencil pairs (jj, 2N - jj) of one right-hand side (grid x <
// nreg; pair-pencil pp = pair * N + kk, pair 0..N, kk = 0 left out), then the
// CTAs of column 0 (32 of its 4N real vectors each); grid y: right-hand side.
// In place in B.
template <typename T>
__global__ void __launch_bounds__(DirTile<T>::MAXW * 32) k_direct_i(ConvArgs<T> a, int nreg) {
    using C = cplx_t<T>;
    constexpr int TI = DirTile<T>::TI;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const int N = a.nt, N1 = N + 1;
    const int p0 = a.plane_lo(), n0 = a.plane_hi() - p0;
    const int n = n0 + (n0 & 1), m = n / 2, mb = (m + TI - 1) / TI, mp = mb * TI;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int b = blockIdx.y;
    T* gs = reinterpret_cast<T*>(smem_raw);                         // [n][32]
    unsigned char* xraw = smem_raw + (size_t)n * 32 * sizeof(T);    // n even: a multiple of 256 bytes
    const long long dstride = mix_index(N, 1, 0, 0) - mix_index(N, 0, 0, 0);   // entries g(d) and g(d + 1) apart
    const long long istride = (long long)(2 * N) * N1;              // planes of B apart
    C* Bb = a.B + (long long)b * N * istride + (long long)p0 * istride;

    if ((int)blockIdx.x < nreg) {
        using R = DirRow<T, 4>;
        typename R::Unit* xs = reinterpret_cast<typename R::Unit*>(xraw);
        const int pp = blockIdx.x * 32 + lane;
        const int pair = pp / N, kk = pp - pair * N;
        const bool on = pair <= N && kk != 0;
        const bool two = on && pair != 0 && pair != N;   // 2N - jj is another pencil
        // the entries first: they do not depend on the kernel before
        const T* g = a.gmix + (on ? mix_index(N, 0, pair, kk) : 0);
        for (int d = warp; d < n; d += nwarp) gs[d * 32 + lane] = g[min(d, n0 - 1) * dstride];
        wait_prior_grid();
        if (a.active && !a.active[b]) return;   // whole CTA
        C* pa = Bb + (on ? (long long)pair * N1 + kk : 0);
        C* pb = Bb + (two ? (long long)(2 * N - pair) * N1 + kk : 0);
        const C zero = cmake<C>(dir_zero(T()), dir_zero(T()));
#pragma unroll 4
        for (int r = warp; r < mp; r += nwarp) {
            const int rh = n - 1 - r;
            const bool l0 = r < m, l1 = l0 && rh < n0;
            const C a0 = (on && l0) ? pa[r * istride] : zero, a1 = (on && l1) ? pa[rh * istride] : zero;
            const C b0 = (two && l0) ? pb[r * istride] : zero, b1 = (two && l1) ? pb[rh * istride] : zero;
            const T e[4] = {a0.x + a1.x, a0.y + a1.y, b0.x + b1.x, b0.y + b1.y};
            const T o[4] = {a0.x - a1.x, a0.y - a1.y, b0.x - b1.x, b0.y - b1.y};
            typename R::Unit* row = xs + (long long)r * 2 * R::NU * 32;
            R::put(row, lane, e);
            R::put(row + R::NU * 32, lane, o);
        }
        __syncthreads();
        direct_rows_product<T, 4>(xs, gs, n, mb, lane, warp, nwarp, [&](int i, const T* lo, const T* hi) {
            if (i >= m) return;
            const int ih = n - 1 - i;
            if (on) {
                pa[i * istride] = cmake<C>(lo[0], lo[1]);
                if (ih < n0) pa[ih * istride] = cmake<C>(hi[0], hi[1]);
            }
            if (two) {
                pb[i * istride] = cmake<C>(lo[2], lo[3]);
                if (ih < n0) pb[ih * istride] = cmake<C>(hi[2], hi[3]);
            }
        });
    } else {
        using R = DirRow<T, 1>;
        typename R::Unit* xs = reinterpret_cast<typename R::Unit*>(xraw);
        const int c = (blockIdx.x - nreg) * 32 + lane;   // slot of column 0, real or imaginary part
        const bool on = c < 4 * N;
        const int slot = on ? c >> 1 : 0, comp = c & 1;
        const int jj = slot <= N ? slot : 2 * N - slot;
        const int kn = (slot > N || ((slot == 0 || slot == N) && comp)) ? N : 0;
        const T* g = a.gmix + mix_index(N, 0, jj, kn);
        for (int d = warp; d < n; d += nwarp) gs[d * 32 + lane] = g[min(d, n0 - 1) * dstride];
        wait_prior_grid();
        if (a.active && !a.active[b]) return;   // whole CTA
        T* px = reinterpret_cast<T*>(Bb + (long long)slot * N1) + comp;
#pragma unroll 4
        for (int r = warp; r < mp; r += nwarp) {
            const int rh = n - 1 - r;
            const bool l0 = on && r < m, l1 = l0 && rh < n0;
            const T x0 = l0 ? px[2 * r * istride] : dir_zero(T()), x1 = l1 ? px[2 * rh * istride] : dir_zero(T());
            const T e = x0 + x1, o = x0 - x1;
            typename R::Unit* row = xs + (long long)r * 2 * 32;
            R::put(row, lane, &e);
            R::put(row + 32, lane, &o);
        }
        __syncthreads();
        direct_rows_product<T, 1>(xs, gs, n, mb, lane, warp, nwarp, [&](int i, const T* lo, const T* hi) {
            if (i >= m || !on) return;
            const int ih = n - 1 - i;
            px[2 * i * istride] = lo[0];
            if (ih < n0) px[2 * ih * istride] = hi[0];
        });
    }
}

}  // namespace

// Sets the kernel attribute (once per process; before any capture).
template <typename T>
void direct_configure() {
    static const bool configured = []() {
        BAE_CUDA(cudaFuncSetAttribute(k_direct_i<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
        return true;
    }();
    (void)configured;
}

template <typename T>
void launch_direct_i(const ConvArgs<T>& a, cudaStream_t st) {
    constexpr int TI = DirTile<T>::TI, MAXW = DirTile<T>::MAXW;
    const int N = a.nt, n0 = a.plane_hi() - a.plane_lo();
    const int n = n0 + (n0 & 1), mb = (n / 2 + TI - 1) / TI;
    const int nreg = ceil_div((long long)N * (N + 1), 32), ncol = ceil_div(4 * N, 32);
    const size_t smem = (size_t)n * 32 * sizeof(T) + (size_t)mb * TI * 2 * 4 * 32 * sizeof(T);
    direct_configure<T>();
    const dim3 grid(nreg + ncol, a.nbatch);
    const int threads = 32 * (mb < MAXW ? mb : MAXW);
    BAE_LAUNCH(kname<T>("conv_i.f32", "conv_i.f64", "conv_i.df64"), st,
               launch_pdl(k_direct_i<T>, grid, threads, smem, st, a, nreg));
}

}  // namespace bae
