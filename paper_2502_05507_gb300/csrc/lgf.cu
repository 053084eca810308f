// Lattice Green's function of (6+s) - (sum of the six neighbours), s = sigma h^2
// (Section 2.2, eq. [lgf] with h = 1), by Watson's Bessel integral
// (eq. [lgf_bessel], with exp(-(6+s)t) for sigma > 0):
//
//   G_s(n) = int_0^inf exp(-s t) Ie_a(2t) Ie_b(2t) Ie_c(2t) dt,  Ie_n(x) = e^{-x} I_n(x).
//
// The paper splits the integral at T* into a quadrature part and a tail
// evaluated from the large-argument expansion of I_n (mu = 4n^2). Here:
//  * [0, e^-Q] in t: 20-point Gauss-Legendre, Q = ceil(ln s) for s > 1 else 0;
//    [e^-Q, e^P] in u = ln t: unit panels of 16-point Gauss-Legendre (the
//    integrand is analytic in u), P chosen per offset from max(n).
//  * Ie_n(2 t_j), n < N, for every node t_j: the large-argument series for x =
//    2 t_j >= max(N^2 / 2, 40), else Miller's backward recurrence I_{k-1} =
//    (2k/x) I_k + I_{k+1}, started at sqrt(N^2 + 80x) + 20 and normalised by
//    Ie_0 + 2 sum_k Ie_k = 1.
//  * Tail from T = e^P, T >= 100 max(n)^2: the product of the three
//    large-argument series (6 terms each) integrated term by term against
//    exp(-s t) t^{-3/2-k}: closed form for s = 0, erfc and upward recurrence
//    for 0 < s T <= 1. For s T* > 1 the panels are instead extended to
//    t = 45 / s, where exp(-s t) makes the rest negligible.
// The spectrum of the evenly embedded table is a separable cosine transform
// evaluated in three passes that use its symmetries (k_cos_fold).
#include <cmath>
#include <vector>

#include "conv.cuh"
#include "lgf.cuh"

namespace bae {

namespace {

constexpr int NODES0 = 20;    // Gauss-Legendre points on [0, 1]
constexpr int NODESP = 16;    // points per unit panel in ln t
constexpr int TAIL_K = 7;     // tail series terms (k = 0..6)

// Gauss-Legendre nodes and weights on [-1, 1] by Newton's method on P_n.
void gauss_legendre(int n, std::vector<double>& x, std::vector<double>& w) {
    x.assign(n, 0.0);
    w.assign(n, 0.0);
    for (int i = 0; i < n; ++i) {
        double z = std::cos(M_PI * (i + 0.75) / (n + 0.5));
        double dp = 1.0;
        for (int it = 0; it < 100; ++it) {
            double p0 = 1.0, p1 = z;
            for (int k = 2; k <= n; ++k) {
                double pk = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = pk;
            }
            dp = n * (z * p1 - p0) / (z * z - 1.0);
            double dz = p1 / dp;
            z -= dz;
            if (std::fabs(dz) < 1e-16) break;
        }
        {   // final derivative at the converged node
            double p0 = 1.0, p1 = z;
            for (int k = 2; k <= n; ++k) {
                double pk = ((2.0 * k - 1.0) * z * p1 - (k - 1.0) * p0) / k;
                p0 = p1;
                p1 = pk;
            }
            dp = n * (z * p1 - p0) / (z * z - 1.0);
        }
        x[i] = z;
        w[i] = 2.0 / ((1.0 - z * z) * dp * dp);
    }
}

struct Plan {
    int N = 0;
    double s = 0.0;
    int n_nodes = 0;
    int q0 = 0;                             // panels below t = 1
    std::vector<double> t, wexp;            // nodes and weights * exp(-s t)
    std::vector<int> panels;                // P per max index a
    std::vector<int> tail_mode;             // 0 none, 1 s = 0, 2 erfc recurrence
};

Plan make_plan(int N, double s) {
    Plan p;
    p.N = N;
    p.s = s;
    p.panels.resize(N);
    p.tail_mode.resize(N);
    int pmax = 1;
    for (int a = 0; a < N; ++a) {
        int P = 7;
        if (a > 0) P = std::max(7, (int)std::ceil(std::log(100.0 * a * a)));
        int mode = (s == 0.0) ? 1 : 2;
        if (s > 0.0 && s * std::exp((double)P) > 1.0) {
            P = std::max(1, (int)std::ceil(std::log(45.0 / s)));
            mode = 0;
        }
        p.panels[a] = P;
        p.tail_mode[a] = mode;
        pmax = std::max(pmax, P);
    }
    p.q0 = s > 1.0 ? (int)std::ceil(std::log(s)) : 0;
    const double t0 = std::exp(-(double)p.q0);
    std::vector<double> x20, w20, x16, w16;
    gauss_legendre(NODES0, x20, w20);
    gauss_legendre(NODESP, x16, w16);
    for (int i = 0; i < NODES0; ++i) {
        p.t.push_back(0.5 * t0 * (x20[i] + 1.0));
        p.wexp.push_back(0.5 * t0 * w20[i]);
    }
    for (int q = 1 - p.q0; q <= pmax; ++q)
        for (int i = 0; i < NODESP; ++i) {
            const double u = q - 0.5 + 0.5 * x16[i];
            const double tt = std::exp(u);
            p.t.push_back(tt);
            p.wexp.push_back(0.5 * w16[i] * tt);
        }
    p.n_nodes = (int)p.t.size();
    for (int j = 0; j < p.n_nodes; ++j) p.wexp[j] *= std::exp(-s * p.t[j]);
    return p;
}

// Ie_n(2 t_j), n < N, one CTA per node. From x = 2 t_j = x_asym = max(N^2 / 2,
// 40) on the large-argument series (terms below (n^2 / 2x)^k / k! until they
// are far under round-off), a thread per n; below, thread 0 runs Miller's
// recurrence. The recurrence is a chain of ~sqrt(80 x) dependent float64
// operations (64 cycles each): up to the largest node, x ~ 6e6 at N = 128, it
// took 357 us; up to x_asym it is 6.4 N steps. What is left is the float64
// operations per step (one thread, 64 cycles each): the product, the fused
// multiply-add and the sum, the overflow test on the exponent bits.
__global__ void k_bessel_rows(const double* __restrict__ t, int N, double x_asym, double* __restrict__ rows) {
    extern __shared__ double s_row[];
    const int j = blockIdx.x;
    const double x = 2.0 * t[j];
    if (x >= x_asym) {
        const double scale = rsqrt(2.0 * M_PI * x), q = -1.0 / (8.0 * x);
        for (int n = threadIdx.x; n < N; n += blockDim.x) {
            const double mu = 4.0 * (double)n * (double)n;
            double term = 1.0, sum = 1.0;
#pragma unroll
            for (int k = 1; k <= 32; ++k) {
                term *= (mu - (double)((2 * k - 1) * (2 * k - 1))) * (q * (1.0 / k));
                sum += term;
            }
            rows[(long long)j * N + n] = sum * scale;
        }
        return;
    }
    if (threadIdx.x == 0) {
        const long long M = (long long)ceil(sqrt((double)N * N + 80.0 * x)) + 20;
        const double twox = 2.0 / x;
        double y1 = 0.0, y0 = 1e-280, S = 0.0;   // S: half the sum over k >= 1
        const int big = __double2hiint(1e250);
        for (int n = 0; n < N; ++n) s_row[n] = 0.0;
        for (int k = (int)M; k >= 1; --k) {
            if (k < N) s_row[k] = y0;
            S += y0;
            const double ym = (double)k * twox * y0 + y1;
            y1 = y0;
            y0 = ym;
            if (__double2hiint(ym) > big) {
                y1 *= 1e-250;
                y0 *= 1e-250;
                S *= 1e-250;
                const int top = k < N ? k : N;
                for (int n = top; n < N; ++n) s_row[n] *= 1e-250;
            }
        }
        s_row[0] = y0;
        const double inv = 1.0 / (2.0 * S + y0);
        for (int n = 0; n < N; ++n) s_row[n] *= inv;
    }
    __syncthreads();
    for (int n = threadIdx.x; n < N; n += blockDim.x) rows[(long long)j * N + n] = s_row[n];
}

__device__ __forceinline__ long long tet(long long a) { return a * (a + 1) * (a + 2) / 6; }
__device__ __forceinline__ long long tri2(long long b) { return b * (b + 1) / 2; }

// Coefficients alpha_j(n) of Ie_n(2t) ~ (4 pi t)^{-1/2} sum_j alpha_j t^{-j}:
// alpha_j = (-1)^j a_j(mu) / 2^j, a_j = prod_{i<=j} (mu - (2i-1)^2) / (j! 8^j).
__device__ void tail_alpha(int n, double* al) {
    const double mu = 4.0 * (double)n * (double)n;
    double c = 1.0;
    al[0] = 1.0;
    for (int j = 1; j < TAIL_K; ++j) {
        c *= (mu - (double)((2 * j - 1) * (2 * j - 1))) / (8.0 * j);
        al[j] = ((j & 1) ? -c : c) / (double)(1LL << j);
    }
}

// G(a, b, c) for one a, TC consecutive c and every b >= c per CTA (a thread
// per b): the sum over the nodes is a product of the rows r_a r_b (one product
// per node and b) and r_c, one fused multiply-add per entry and node instead
// of three float64 operations (N = 128: 278 us, 409 us with a thread per
// entry), and the tail integrals E_k are formed once per a.
constexpr int TC = 8;      // entries per thread
constexpr int TNODES = 256;   // nodes in shared memory at a time
__global__ void __launch_bounds__(256) k_lgf_table(const double* __restrict__ rows, const double* __restrict__ wexp,
                                                   const int* __restrict__ panels, const int* __restrict__ tail_mode,
                                                   int N, double s, int q0, double* __restrict__ out) {
    __shared__ double wa[TNODES], rc[TNODES][TC], Ek[TAIL_K], ac[TC][TAIL_K];   // w_j r_a(j), r_c(j), E_k, alpha(c)
    const int a = N - 1 - (int)blockIdx.x, c0 = (int)blockIdx.y * TC;
    if (c0 > a) return;
    const int P = panels[a], mode = tail_mode[a];
    const int nn = NODES0 + NODESP * (P + q0);
    const int b = c0 + (int)threadIdx.x;   // a < N <= 256: one b per thread
    const bool on = b <= a;
    if (mode != 0 && threadIdx.x < TC) tail_alpha(c0 + threadIdx.x, ac[threadIdx.x]);
    if (mode != 0 && threadIdx.x == 32) {
        const double T = exp((double)P), rT = 1.0 / sqrt(T);
        const double eT = (mode == 2) ? exp(-s * T) : 1.0;
        double E = 0.0, Tpow = rT;   // Tpow = T^{-1/2-k}
        for (int k = 0; k < TAIL_K; ++k) {
            if (mode == 1) {
                E = Tpow / (k + 0.5);
            } else if (k == 0) {
                E = 2.0 * rT * eT - 2.0 * sqrt(M_PI * s) * erfc(sqrt(s * T));
            } else {
                E = (Tpow * eT - s * E) / (k + 0.5);
            }
            Ek[k] = E;
            Tpow /= T;
        }
    }
    double acc[TC];
#pragma unroll
    for (int q = 0; q < TC; ++q) acc[q] = 0.0;
    for (int j0 = 0; j0 < nn; j0 += TNODES) {
        const int cnt = min(TNODES, nn - j0);
        __syncthreads();   // the nodes before are read
        for (int j = threadIdx.x; j < cnt; j += blockDim.x) {
            const double* r = rows + (long long)(j0 + j) * N;
            wa[j] = wexp[j0 + j] * r[a];
#pragma unroll
            for (int q = 0; q < TC; ++q) rc[j][q] = c0 + q < N ? r[c0 + q] : 0.0;
        }
        __syncthreads();
        if (on) {
            const double* rb = rows + (long long)j0 * N + b;
            for (int j = 0; j < cnt; ++j) {
                const double p = wa[j] * rb[(long long)j * N];
#pragma unroll
                for (int q = 0; q < TC; ++q) acc[q] += p * rc[j][q];
            }
        }
    }
    if (!on) return;
    double ab[TAIL_K];   // the series of Ie_a Ie_b
    if (mode != 0) {
        double al[TAIL_K], bl[TAIL_K];
        tail_alpha(a, al);
        tail_alpha(b, bl);
        for (int k = 0; k < TAIL_K; ++k) {
            double v = 0.0;
            for (int i = 0; i <= k; ++i) v += al[i] * bl[k - i];
            ab[k] = v;
        }
    }
#pragma unroll
    for (int q = 0; q < TC; ++q) {
        const int c = c0 + q;
        if (c > b) break;
        double v = acc[q];
        if (mode != 0) {
            double tail = 0.0;
            for (int k = 0; k < TAIL_K; ++k) {
                double beta = 0.0;
                for (int i = 0; i <= k; ++i) beta += ab[i] * ac[q][k - i];
                tail += beta * Ek[k];
            }
            v += tail * (1.0 / (8.0 * M_PI * sqrt(M_PI)));  // (4 pi)^{-3/2}
        }
        out[tet(a) + tri2(b) + c] = v;
    }
}

// The spectrum of the evenly embedded table: a cosine transform along each
// axis, out(k) = sum_n w(n) cos(pi k n / N) x(n), k <= N, n < N, w(0) = 1, w(n)
// = 2. Bound by the FP64 pipe (64 cycles per warp instruction), so what counts
// is the number of products:
//  - the table is symmetric in the three indices, hence so are the frequency
//    pairs after two passes and the triples after three: pass 1 transforms the
//    lines j <= k, pass 2 forms the outputs mu <= kappa, pass 3 nu <= mu <=
//    kappa (a half, a half and a sixth of the outputs);
//  - cos(pi k (N - n) / N) = (-1)^k cos(pi k n / N): sums and differences of
//    mirrored inputs serve the even and the odd k, and once more for the even
//    ones, so an output takes N / 2 or N / 4 products.
// N = 128: the three passes take 511 us, 1590 us with full lines before.
// Element e of line (o, lane l), o the index the CTA shares:
//   PASS 1: G(e, o, l), l >= o   -> P1[k][o][l]     (axis 0 of the cube)
//   PASS 2: P1[o][e, l sorted]   -> P2[o][k][l]     k <= o
//   PASS 3: P2[o][l][e], l <= o  -> T3[o][k][l]     k <= l
// with P1[N+1][N][N], P2[N+1][N+1][N], T3[N+1][N+1][N+1].
template <int PASS>
__global__ void __launch_bounds__(256) k_cos_fold(const double* __restrict__ in, double* __restrict__ out, int N) {
    extern __shared__ double s_fold[];
    constexpr int LS = 33;                       // lanes, padded
    const int N1 = N + 1, L = 2 * N, H = N / 2, Q = N / 4;
    double* ct = s_fold;                         // [2N] cos(pi m / N)
    double* V = ct + L;                          // [H][LS] x(n) - x(N-n)
    double* VV = V + H * LS;                     // [Q][LS]
    double* UU = VV + Q * LS;                    // [Q+1][LS]
    const int nl = PASS == 3 ? N1 : N;           // lanes in all
    const int nblk = (nl + 31) / 32;
    const int o = blockIdx.x / nblk, l0 = (blockIdx.x % nblk) * 32;
    if ((PASS == 1 && l0 + 31 < o) || (PASS == 3 && l0 > o)) return;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    const int l = l0 + lane;
    const bool on = l < nl && (PASS != 1 || l >= o) && (PASS != 3 || l <= o);
    for (int m = threadIdx.x; m < L; m += blockDim.x) ct[m] = cospi((double)m / (double)N);
    auto x = [&](int e) -> double {   // w(e) x(e), e < N
        if (!on) return 0.0;
        double v;
        if (PASS == 1) {
            const int p = max(e, l), q = min(e, o), r = e + o + l - p - q;   // o <= l
            v = in[tet(p) + tri2(r) + q];
        } else if (PASS == 2) {
            v = in[((long long)o * N + min(e, l)) * N + max(e, l)];
        } else {
            v = in[((long long)o * N1 + l) * N + e];
        }
        return e == 0 ? v : 2.0 * v;
    };
    for (int n = warp; n <= Q; n += nwarp) {
        const int h = H - n;
        const double x1 = x(n), x2 = n ? x(N - n) : 0.0;
        const double u1 = x1 + x2;
        V[n * LS + lane] = x1 - x2;
        if (n == Q) {
            UU[n * LS + lane] = u1;
        } else {
            const double x3 = x(h), x4 = n ? x(N - h) : 0.0;   // n = 0: h = N - h
            const double u2 = x3 + x4;
            if (n) V[h * LS + lane] = x3 - x4;
            UU[n * LS + lane] = u1 + u2;
            VV[n * LS + lane] = u1 - u2;
        }
    }
    __syncthreads();
    const int kmax = PASS == 1 ? N : (PASS == 2 ? o : min(o, l0 + 31));
    auto sum = [&](const double* v, int terms, int k) -> double {
        double acc = 0.0;
        int m = 0;
        for (int n = 0; n < terms; ++n) {
            acc += ct[m] * v[n * LS + lane];
            m += k;
            if (m >= L) m -= L;
        }
        return acc;
    };
    for (int g = 4 * warp; g <= kmax; g += 4 * nwarp)
        for (int k = g; k < g + 4 && k <= kmax; ++k) {
            const double v = k & 1 ? sum(V, H, k) : (k & 2 ? sum(VV, Q, k) : sum(UU, Q + 1, k));
            if (!on) continue;
            if (PASS == 1) out[((long long)k * N + o) * N + l] = v;
            else if (PASS == 2) out[((long long)o * N1 + k) * N + l] = v;
            else out[((long long)o * N1 + k) * N1 + l] = v;
        }
}

// The spectrum of the (2N)-periodic Green's function in closed form, i.e.
// the 2N-point trapezoid rule of the Fourier integral eq. [lgf] read in
// frequency space (Section 2.2, sigma > 0): scale / (6 + s - 2 sum_i
// cos(pi k_i / N)) on the octant 0 <= k_i <= N.
__global__ void k_periodic_spectrum(int N, double s, double scale, double* g64, float* g32) {
    const long long N1 = N + 1, n3 = N1 * N1 * N1;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n3; x += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(x / (N1 * N1)), j = (int)((x / N1) % N1), k = (int)(x % N1);
        const double c = cospi((double)i / N) + cospi((double)j / N) + cospi((double)k / N);
        const double v = scale / (6.0 + s - 2.0 * c);
        g64[x] = v;
        if (g32) g32[x] = (float)v;
    }
}

// ghat(i, j, k) = scale * T3[a][c][b], a >= b >= c the sorted indices
__global__ void k_spectrum_out(const double* __restrict__ t3, int N, double scale, double* g64, float* g32) {
    const long long N1 = N + 1, n = N1 * N1 * N1;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n; x += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(x / (N1 * N1)), j = (int)((x / N1) % N1), k = (int)(x % N1);
        const int a = max(i, max(j, k)), c = min(i, min(j, k)), b = i + j + k - a - c;
        const double v = t3[((long long)a * N1 + c) * N1 + b] * scale;
        g64[x] = v;
        if (g32) g32[x] = (float)v;
    }
}

__global__ void k_twiddles(int L, double2* tw64, float2* tw32) {
    for (int m = blockIdx.x * blockDim.x + threadIdx.x; m < L; m += gridDim.x * blockDim.x) {
        double sn, cs;
        sincospi(2.0 * (double)m / (double)L, &sn, &cs);
        tw64[m] = make_double2(cs, -sn);
        tw32[m] = make_float2((float)cs, (float)-sn);
    }
}

// threads per line of the plans that read the products table of a transform
// of length L (Factors<L>::R1; PlanQ with at most 16 threads)
__host__ __device__ inline int level_one(int L) { return L <= 48 ? 4 : (L <= 128 ? 8 : 16); }

// out[k2 R1 + n1] = exp(-2 pi i n1 k2 / L), n1 < R1, k2 < L / R1
__global__ void k_twiddle_products(int L, int R1, double2* tw64, float2* tw32) {
    for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < L; x += gridDim.x * blockDim.x) {
        double sn, cs;
        sincospi(2.0 * (double)((x % R1) * (x / R1)) / (double)L, &sn, &cs);
        tw64[x] = make_double2(cs, -sn);
        tw32[x] = make_float2((float)cs, (float)-sn);
    }
}

template <typename T>
struct DevBuf {
    T* p = nullptr;
    cudaStream_t st;
    DevBuf(size_t n, cudaStream_t s) : st(s) { p = dev_alloc_n<T>((long long)n, s); }
    ~DevBuf() { dev_free(p, st); }
    DevBuf(const DevBuf&) = delete;
    DevBuf& operator=(const DevBuf&) = delete;
};

void table_into(int N, double s, double* out, cudaStream_t st) {
    Plan plan = make_plan(N, s);
    DevBuf<double> d_t(plan.n_nodes, st), d_w(plan.n_nodes, st), d_rows((size_t)plan.n_nodes * N, st);
    DevBuf<int> d_p(N, st), d_m(N, st);
    BAE_CUDA(cudaMemcpyAsync(d_t.p, plan.t.data(), plan.n_nodes * sizeof(double), cudaMemcpyHostToDevice, st));
    BAE_CUDA(cudaMemcpyAsync(d_w.p, plan.wexp.data(), plan.n_nodes * sizeof(double), cudaMemcpyHostToDevice, st));
    BAE_CUDA(cudaMemcpyAsync(d_p.p, plan.panels.data(), N * sizeof(int), cudaMemcpyHostToDevice, st));
    BAE_CUDA(cudaMemcpyAsync(d_m.p, plan.tail_mode.data(), N * sizeof(int), cudaMemcpyHostToDevice, st));
    const double x_asym = std::max(0.5 * N * N, 40.0);
    BAE_LAUNCH("k_bessel_rows", st,
               k_bessel_rows<<<plan.n_nodes, 128, N * sizeof(double), st>>>(d_t.p, N, x_asym, d_rows.p));
    BAE_LAUNCH("k_lgf_table", st,
               k_lgf_table<<<dim3(N, ceil_div(N, TC)), 256, 0, st>>>(d_rows.p, d_w.p, d_p.p, d_m.p, N, s, plan.q0, out));
    BAE_CUDA(cudaStreamSynchronize(st));  // host vectors and scratch die here
}

}  // namespace

void lgf_table(int N, double s, double* out, cudaStream_t st) {
    BAE_REQUIRE(N >= 2 && N <= 256, BAE_ERR_INVALID_ARG, "lgf_table: N must be in [2, 256]");
    BAE_REQUIRE(std::isfinite(s) && s >= 0.0, BAE_ERR_INVALID_ARG, "lgf_table: s must be finite and >= 0");
    table_into(N, s, out, st);
}

// The spectrum of the finite-box Green's function of eq. [aux]: with the
// source extended oddly about the layers 0 and N in every axis, the box
// solve is the convolution with the (2N)-periodic Green's function, whose
// spectrum is scale / (6 + s - 2 sum cos(pi k_d / N)). Its only pole (s = 0,
// k = 0) multiplies a zero of the odd data and is set to 0.
__global__ void k_box_spectrum(int N, double s, double scale, double* g64, float* g32) {
    const long long N1 = N + 1, n3 = N1 * N1 * N1;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n3; x += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(x / (N1 * N1)), j = (int)((x / N1) % N1), k = (int)(x % N1);
        const double c = cospi((double)i / N) + cospi((double)j / N) + cospi((double)k / N);
        const double d = 6.0 + s - 2.0 * c;
        const double v = d != 0.0 ? scale / d : 0.0;
        g64[x] = v;
        if (g32) g32[x] = (float)v;
    }
}

void box_spectrum(int N, double s, double scale, double* g64, float* g32, cudaStream_t st) {
    BAE_REQUIRE(is_pow2(N) && N >= 8 && N <= 256, BAE_ERR_INVALID_ARG,
                "box_spectrum: N must be a power of two in [8, 256]");
    BAE_REQUIRE(std::isfinite(s) && s >= 0.0, BAE_ERR_INVALID_ARG, "box_spectrum: s must be finite and >= 0");
    const long long N1 = N + 1, n3 = N1 * N1 * N1;
    BAE_LAUNCH("k_box_spectrum", st,
               k_box_spectrum<<<(int)std::min<long long>((n3 + 255) / 256, 152LL * 16), 256, 0, st>>>(N, s, scale,
                                                                                                        g64, g32));
}

bool periodic_spectrum_applies(int N, double s) {
    if (!(s > 0.0)) return false;
    const double mu = std::acosh(1.0 + 0.5 * s);   // G_s ~ exp(-mu |n|) along an axis
    return std::pow(2.0 * N, 3) * std::exp(-mu * N) < 1e-14;
}

// The mixed spectrum of the direct i pass (layout: mix_index) from the table
// transformed along two axes, P2[max(j, k)][min(j, k)][d]: 32 x 32 tiles (k,
// d) per j, transposed through shared memory so that both sides are contiguous
__global__ void __launch_bounds__(256) k_mixed_out(const double* __restrict__ p2, int N, double scale, double* m64,
                                                   float* m32) {
    __shared__ double tile[32][33];
    const int N1 = N + 1, j = blockIdx.z, k0 = blockIdx.y * 32, d0 = blockIdx.x * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int r = ty; r < 32; r += 8) {
        const int k = k0 + r, d = d0 + tx;
        if (k < N1 && d < N) tile[r][tx] = p2[((long long)max(j, k) * N1 + min(j, k)) * N + d] * scale;
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
        const int d = d0 + r, k = k0 + tx;
        if (k < N1 && d < N) {
            const long long y = mix_index(N, d, j, k);
            const double v = tile[tx][r];
            m64[y] = v;
            if (m32) m32[y] = (float)v;
        }
    }
}

// The mixed spectrum of the (2N)-periodic Green's function in closed form:
// with c = 6 + s - 2 cos(pi jj / N) - 2 cos(pi kk / N) = lam + 1/lam, lam < 1,
// the inverse transform of 1 / (c - 2 cos(pi p / N)) along p is
// (lam^d + lam^(2N-d)) / ((1/lam - lam) (1 - lam^2N)). c - 2 is summed from
// its small terms, so nothing cancels.
__global__ void k_periodic_mixed(int N, double s, double scale, double* m64, float* m32) {
    const long long N1 = N + 1, n = N * N1 * N1;
    for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n; x += (long long)gridDim.x * blockDim.x) {
        const int d = (int)(x / (N1 * N1)), j = (int)((x / N1) % N1), k = (int)(x % N1);
        const double sj = sinpi(0.5 * j / N), sk = sinpi(0.5 * k / N);
        const double c2 = s + 4.0 * (sj * sj + sk * sk);      // c - 2
        const double r = sqrt(c2 * (c2 + 4.0));               // 1/lam - lam
        const double lam = 2.0 / (c2 + 2.0 + r);
        const double v = scale * (pow(lam, (double)d) + pow(lam, (double)(2 * N - d))) / (r * (1.0 - pow(lam, 2.0 * N)));
        const long long y = mix_index(N, d, j, k);
        m64[y] = v;
        if (m32) m32[y] = (float)v;
    }
}

void lgf_spectrum(int N, double s, double scale, double* g64, float* g32, cudaStream_t st, double mix_scale,
                  double* mix64, float* mix32) {
    BAE_REQUIRE(N % 8 == 0 && N >= 8 && N <= 256, BAE_ERR_INVALID_ARG,
                "lgf_spectrum: N must be a multiple of eight in [8, 256]");
    BAE_REQUIRE(std::isfinite(s) && s >= 0.0, BAE_ERR_INVALID_ARG, "lgf_spectrum: s must be finite and >= 0");
    const long long N1 = N + 1;
    const long long n3 = N1 * N1 * N1;
    if (periodic_spectrum_applies(N, s)) {
        // the images of the (2N)-periodic Green's function are below
        // round-off: no table, no cosine transform
        if (g64)
            BAE_LAUNCH("k_periodic_spectrum", st,
                   k_periodic_spectrum<<<(int)std::min<long long>((n3 + 255) / 256, 152LL * 16), 256, 0, st>>>(
                       N, s, scale, g64, g32));
        if (mix64)
            BAE_LAUNCH("k_periodic_mixed", st,
                       k_periodic_mixed<<<(int)std::min<long long>((n3 + 255) / 256, 152LL * 16), 256, 0, st>>>(
                           N, s, mix_scale, mix64, mix32));
        BAE_CUDA(cudaStreamSynchronize(st));
        return;
    }
    const long long ntri = (long long)N * (N + 1) * (N + 2) / 6;
    DevBuf<double> tab(ntri, st), c0(n3, st), c1(n3, st);
    table_into(N, s, tab.p, st);
    const size_t smem = (2 * (size_t)N + 33 * ((size_t)N + 1)) * sizeof(double);
    for (auto k : {k_cos_fold<1>, k_cos_fold<2>, k_cos_fold<3>})
        BAE_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const int nb = ceil_div(N, 32), nb1 = ceil_div(N1, 32);
    BAE_LAUNCH("k_cos_fold", st, k_cos_fold<1><<<N * nb, 256, smem, st>>>(tab.p, c0.p, N));
    BAE_LAUNCH("k_cos_fold", st, k_cos_fold<2><<<(unsigned)(N1 * nb), 256, smem, st>>>(c0.p, c1.p, N));
    if (mix64)
        BAE_LAUNCH("k_mixed_out", st,
                   k_mixed_out<<<dim3(nb, nb1, (unsigned)N1), 256, 0, st>>>(c1.p, N, mix_scale, mix64, mix32));
    if (g64) {
        BAE_LAUNCH("k_cos_fold", st, k_cos_fold<3><<<(unsigned)(N1 * nb1), 256, smem, st>>>(c1.p, c0.p, N));
        BAE_LAUNCH("k_spectrum_out", st, k_spectrum_out<<<(int)std::min<long long>((n3 + 255) / 256, 152LL * 16), 256, 0, st>>>(c0.p, N, scale, g64, g32));
    }
    BAE_CUDA(cudaStreamSynchronize(st));
}

void make_twiddles(int L, double2* tw64, float2* tw32, cudaStream_t st) {
    for (int len = L, off = 0; len >= L / 2; off += 2 * len, len /= 2) {
        BAE_LAUNCH("k_twiddles", st, k_twiddles<<<ceil_div(len, 256), 256, 0, st>>>(len, tw64 + off, tw32 + off));
        BAE_LAUNCH("k_twiddle_products", st,
                   k_twiddle_products<<<ceil_div(len, 256), 256, 0, st>>>(len, level_one(len), tw64 + off + len,
                                                                          tw32 + off + len));
    }
}

}  // namespace bae
