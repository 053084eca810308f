// Classification of the grid from level-set samples (Section 2.1), the
// Dirichlet closure (eq. [bc], hat functions on the grid edge to the M+
// neighbour whose phi-linear zero crossing is nearest), and the source
// stencil of the layer potentials (Section 3.2) in a form the convolution's
// first pass reads line by line.
//
// Every list is produced in lexicographic (i,j,k) order by a deterministic
// exclusive scan, so the results are bit-identical from run to run.
#include <algorithm>
#include <cstdlib>
#include <vector>

#include "classify.cuh"

namespace bae {

namespace {

constexpr int SCAN_E = 16;   // entries per thread of the line-count scans

__constant__ int c_dir[6][3] = {{1, 0, 0}, {-1, 0, 0}, {0, 1, 0}, {0, -1, 0}, {0, 0, 1}, {0, 0, -1}};

// ---------------------------------------------------------------- scans
// exclusive scan over the CTA (blockDim.x a multiple of 32, at most 1024);
// the CTA total is left in s_warp[32]
__device__ int block_exclusive_scan(int v, int* s_warp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        int w = (lane < (int)(blockDim.x >> 5)) ? s_warp[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, w, o);
            if (lane >= o) w += y;
        }
        s_warp[lane] = w;   // inclusive warp totals
    }
    __syncthreads();
    const int before = warp > 0 ? s_warp[warp - 1] : 0;
    const int total = s_warp[(blockDim.x >> 5) - 1];
    __syncthreads();
    s_warp[32] = total;
    return before + x - v;  // exclusive
}

// ------------------------------------------------------------ point sets
// A warp per grid line (i, j), its lanes over k; N^2 lines are a multiple of
// the eight warps of a CTA (N a power of two, at least 8).

// slots of the small device record the host reads once
// (I_NGM .. I_GP: the totals of the scans, in the order of their arrays)
enum { I_ERR = 0, I_FIRST, I_LAST, I_NGM, I_NSRC, I_NTERM, I_GP, I_MP, I_FIRSTY, I_LASTY, I_FIRSTZ, I_LASTZ,
       I_COUNT };

__device__ __forceinline__ bool in_grid(int i, int j, int k, int N) {
    return (unsigned)i < (unsigned)N && (unsigned)j < (unsigned)N && (unsigned)k < (unsigned)N;
}

// phi < 0 and phi not finite, by integer operations: a float64 comparison
// holds GB300's FP64 pipe for 64 cycles per warp
__device__ __forceinline__ bool negative(double p) {
    const int hi = __double2hiint(p);
    return hi < 0 && (((hi & 0x7fffffff) | __double2loint(p)) != 0);
}
__device__ __forceinline__ bool not_finite(double p) { return (__double2hiint(p) & 0x7ff00000) == 0x7ff00000; }

// The node classes are formed as bit words: word w of a line holds the nodes
// 32 w .. 32 w + 31 (N < 32: one word of N bits). As one CTA per line with six
// byte loads per node the two passes took 40 + 47 us at N = 128, almost all of
// it instruction issue; three passes over words take a seventh of that.
__device__ __forceinline__ int words(int N) { return (N + 31) >> 5; }

// the word of the same k's in a neighbouring line (di, dj), 0 outside the box
__device__ __forceinline__ unsigned line_word(const unsigned* __restrict__ m, int i, int j, int w, int N) {
    return (unsigned)i < (unsigned)N && (unsigned)j < (unsigned)N ? m[(i * N + j) * words(N) + w] : 0u;
}

// bit k of q[d] = bit of the neighbour of node k in direction d (order of
// c_dir; 0 outside the box): the four neighbouring lines' words, and the
// word itself moved by one node with the adjoining words' end bits
__device__ __forceinline__ void neighbour_words(const unsigned* __restrict__ m, int i, int j, int w, int N,
                                                unsigned q[6]) {
    const unsigned* row = m + (i * N + j) * words(N);
    const unsigned me = row[w];
    q[0] = line_word(m, i + 1, j, w, N);
    q[1] = line_word(m, i - 1, j, w, N);
    q[2] = line_word(m, i, j + 1, w, N);
    q[3] = line_word(m, i, j - 1, w, N);
    q[4] = (me >> 1) | (w + 1 < words(N) ? row[w + 1] << 31 : 0u);
    q[5] = (me << 1) | (w > 0 ? row[w - 1] >> 31 : 0u);
}

// M+ (phi < 0) as words; a phi that is not finite ends the problem, whatever its
// bit. A warp takes four words, their loads in flight together.
__global__ void __launch_bounds__(256) k_inside(const double* __restrict__ phi, int N, unsigned* __restrict__ in,
                                               int* __restrict__ info) {
    constexpr int U = 4;
    const int nw = words(N), lane = threadIdx.x & 31, total = N * N * nw;
    const int w0 = U * (blockIdx.x * 8 + (threadIdx.x >> 5));
    double p[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
        const int word = w0 + u, line = word / nw, k = 32 * (word - line * nw) + lane;
        p[u] = word < total && k < N ? phi[(long long)line * N + k] : 1.0;
    }
    unsigned mine = 0;
    bool bad = false;
#pragma unroll
    for (int u = 0; u < U; ++u) {
        bad |= not_finite(p[u]);
        const unsigned b = __ballot_sync(0xffffffffu, negative(p[u]));
        if (lane == u) mine = b;
    }
    if (bad) atomicOr(info + I_ERR, 1);
    if (lane < U && w0 + lane < total) in[w0 + lane] = mine;
}

// gamma- = outside M+ with an M+ neighbour, and gamma+ = M+ with an exterior
// neighbour (nodes outside the box count as exterior); a thread per word
__global__ void __launch_bounds__(256) k_gamma_words(const unsigned* __restrict__ in, int N, unsigned* __restrict__ gm,
                                                    unsigned* __restrict__ gp) {
    const int nw = words(N), word = blockIdx.x * 256 + threadIdx.x;
    if (word >= N * N * nw) return;
    const int line = word / nw, w = word - line * nw, i = line / N, j = line - i * N;
    const unsigned valid = N < 32 ? (1u << N) - 1u : 0xffffffffu, me = in[word];
    unsigned q[6];
    neighbour_words(in, i, j, w, N, q);
    gm[word] = valid & ~me & (q[0] | q[1] | q[2] | q[3] | q[4] | q[5]);
    gp[word] = me & ~(q[0] & q[1] & q[2] & q[3] & q[4] & q[5]);
}

// per line: M+ nodes (at most 256), N - the first and 1 + the last k of its
// sources (0, 0: none), nine bits each
__device__ __forceinline__ int line_box(int mp, int first, int last) { return mp | (first << 9) | (last << 18); }

// Node flags: M+ (bit0), gamma- (bit1), gamma+ (bit2), D-node = outside N+ =
// M+ and gamma-, next to a gamma- node (bit3), and for gamma- nodes |D_n| =
// the neighbours outside N+ (bits 4-6). A warp per line; lane = node of the
// word. Per line, by population counts that every lane forms: the gamma-
// nodes, the sources (flags & src_mask) and their stencil terms (a D-node: one
// per gamma- neighbour; a gamma- node: 1, or with `direct` 1 + its neighbours
// in gamma = gamma- u gamma+), the gamma+ nodes, and in one int the M+ nodes
// and the k range of the sources (line_box); k_scan_lines forms totals and
// ranges from them.
__global__ void __launch_bounds__(256) k_flags_lines(const unsigned* __restrict__ in, const unsigned* __restrict__ gmw,
                                                    const unsigned* __restrict__ gpw, int N, int src_mask,
                                                    bool direct, uint8_t* __restrict__ flags,
                                                    int* __restrict__ cnt_gm, int* __restrict__ cnt_src,
                                                    int* __restrict__ cnt_term, int* __restrict__ cnt_gp,
                                                    int* __restrict__ cnt_box, int* __restrict__ info) {
    const int nw = words(N), lane = threadIdx.x & 31;
    const int line = blockIdx.x * 8 + (threadIdx.x >> 5), i = line / N, j = line - i * N;
    int c_gm = 0, c_src = 0, c_term = 0, c_gp = 0, c_in = 0, klo = N, khi = -1;
    unsigned touch = 0;   // gamma- and M+ nodes on a face of the box
    for (int w = 0; w < nw; ++w) {
        const unsigned I = in[line * nw + w], G = gmw[line * nw + w], P = gpw[line * nw + w];
        unsigned g[6], a[6];
        neighbour_words(gmw, i, j, w, N, g);
        if (!(I | G | g[0] | g[1] | g[2] | g[3] | g[4] | g[5])) {   // the most words: no M+, gamma- or D-node
            if (32 * w + lane < N) flags[(long long)line * N + 32 * w + lane] = 0;
            continue;
        }
        neighbour_words(in, i, j, w, N, a);
        const unsigned D = ~I & ~G & (g[0] | g[1] | g[2] | g[3] | g[4] | g[5]) & (N < 32 ? (1u << N) - 1u : 0xffffffffu);
        const unsigned S = (src_mask & 2 ? G : 0u) | (src_mask & 8 ? D : 0u);
        int n_out = 6;
#pragma unroll
        for (int d = 0; d < 6; ++d) {
            c_term += __popc(S & D & g[d]);
            n_out -= ((a[d] | g[d]) >> lane) & 1;
        }
        if (direct && G) {
            unsigned p[6];
            neighbour_words(gpw, i, j, w, N, p);
#pragma unroll
            for (int d = 0; d < 6; ++d) c_term += __popc(G & (g[d] | p[d]));
        }
        c_term += __popc(S & G);
        c_gm += __popc(G);
        c_src += __popc(S);
        c_gp += __popc(P);
        c_in += __popc(I);
        if (S) {
            klo = min(klo, 32 * w + __ffs(S) - 1);
            khi = 32 * w + 31 - __clz(S);
        }
        if (i == 0 || j == 0 || i == N - 1 || j == N - 1) touch |= I | G;
        if (w == 0) touch |= (I | G) & 1u;
        if (w == nw - 1) touch |= (I | G) & (1u << ((N - 1) & 31));
        const int f = ((I >> lane) & 1) | (((G >> lane) & 1) << 1) | (((P >> lane) & 1) << 2) | (((D >> lane) & 1) << 3) |
                      ((G >> lane) & 1 ? n_out << 4 : 0);
        if (32 * w + lane < N) flags[(long long)line * N + 32 * w + lane] = (uint8_t)f;
    }
    if (lane == 0) {
        if (touch) atomicOr(info + I_ERR, 2);
        cnt_gm[line] = c_gm;
        cnt_src[line] = c_src;
        cnt_term[line] = c_term;
        cnt_gp[line] = c_gp;
        cnt_box[line] = line_box(c_in, N - klo, khi + 1);
    }
}

// In-place exclusive scans of the per-line counts (nl + 1 entries, the last
// one becomes the total; nl = N^2 a multiple of SCAN_E), one CTA each; totals to
// info, and from the source counts (c1) the range of their i and j. CTA 4: the
// M+ total and the k range of the sources from the lines' boxes (not scanned).
__device__ __forceinline__ int block_max(int v, int* s_warp) {
    v = __reduce_max_sync(0xffffffffu, v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) s_warp[threadIdx.x >> 5] = v;
    __syncthreads();
    return __reduce_max_sync(0xffffffffu, s_warp[threadIdx.x & 31]);   // 32 warps
}
__global__ void __launch_bounds__(1024) k_scan_lines(int* c0, int* c1, int* c2, int* c3, const int* box, int N,
                                                     int* info) {
    const int nl = N * N, lg = 31 - __clz(N);
    __shared__ int s_warp[33];
    __shared__ int s_carry;
    if (blockIdx.x == 4) {
        int mp = 0, first = 0, last = 0;
        auto take = [&](int v) {
            mp += v & 511;
            first = max(first, (v >> 9) & 511);
            last = max(last, v >> 18);
        };
#pragma unroll 4
        for (int l = threadIdx.x; l < nl / 4; l += blockDim.x) {
            const int4 q = reinterpret_cast<const int4*>(box)[l];
            take(q.x);
            take(q.y);
            take(q.z);
            take(q.w);
        }
        block_exclusive_scan(mp, s_warp);
        const int total = s_warp[32];
        first = block_max(first, s_warp);
        last = block_max(last, s_warp);
        if (threadIdx.x == 0) {
            info[I_MP] = total;
            info[I_FIRSTZ] = first;
            info[I_LASTZ] = last;
        }
        return;
    }
    int* arr = blockIdx.x == 0 ? c0 : (blockIdx.x == 1 ? c1 : (blockIdx.x == 2 ? c2 : c3));
    int r[4] = {0, 0, 0, 0};   // N - first and 1 + last i, then j, of the lines with a count
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int base = 0; base < nl; base += blockDim.x * SCAN_E) {
        int v[SCAN_E], tot = 0;
        const int b0 = base + threadIdx.x * SCAN_E;
        const bool in = b0 < nl;   // all of the thread's entries or none
#pragma unroll
        for (int e = 0; e < SCAN_E; e += 4) {
            const int4 q = in ? *reinterpret_cast<const int4*>(arr + b0 + e) : make_int4(0, 0, 0, 0);
            v[e] = q.x;
            v[e + 1] = q.y;
            v[e + 2] = q.z;
            v[e + 3] = q.w;
            tot += q.x + q.y + q.z + q.w;
        }
        // eight entries lie on one line of i (N a power of two, at least 8)
#pragma unroll
        for (int e = 0; e < SCAN_E; e += 8) {
            unsigned m = 0;
#pragma unroll
            for (int x = 0; x < 8; ++x) m |= v[e + x] ? 1u << x : 0u;
            if (m) {
                const int i = (b0 + e) >> lg, j = (b0 + e) & (N - 1);
                r[0] = max(r[0], N - i);
                r[1] = max(r[1], i + 1);
                r[2] = max(r[2], N - (j + __ffs(m) - 1));
                r[3] = max(r[3], j + 32 - __clz(m));
            }
        }
        const int ex = block_exclusive_scan(tot, s_warp);
        int run = ex + s_carry;
#pragma unroll
        for (int e = 0; e < SCAN_E; e += 4) {
            const int4 q = make_int4(run, run + v[e], run + v[e] + v[e + 1], run + v[e] + v[e + 1] + v[e + 2]);
            if (in) *reinterpret_cast<int4*>(arr + b0 + e) = q;
            run = q.w + v[e + 3];
        }
        __syncthreads();
        if (threadIdx.x == 0) s_carry += s_warp[32];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        arr[nl] = s_carry;
        info[I_NGM + blockIdx.x] = s_carry;
    }
    if (blockIdx.x == 1) {
        const int slot[4] = {I_FIRST, I_LAST, I_FIRSTY, I_LASTY};
#pragma unroll
        for (int x = 0; x < 4; ++x) {
            const int v = block_max(r[x], s_warp);
            if (threadIdx.x == 0) info[slot[x]] = v;
        }
    }
}

// inclusive sum over the lanes of a warp
__device__ __forceinline__ int warp_inclusive_scan(int x) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    return x;
}

// The lists in lexicographic order: a warp per line, which ranks its nodes by
// ballots (and the terms by a shuffle scan) from the line's offsets; a line
// without sources and gamma+ nodes ends at once.
// node_of[x] = index of gamma- node x, n_gm + index of gamma+ node x (set
// only there: the unknown numbers of the direct formulation); term_off[s] =
// first term of source s.
__global__ void __launch_bounds__(256) k_scatter_lines(const uint8_t* __restrict__ flags, int N, int src_mask,
                                                      bool direct, const int* __restrict__ off_gm,
                                                      const int* __restrict__ off_src,
                                                      const int* __restrict__ off_term,
                                                      const int* __restrict__ off_gp, const int* __restrict__ info,
                                                      int* __restrict__ gm, int* __restrict__ gp,
                                                      int* __restrict__ node_of, int* __restrict__ src_lin,
                                                      int* __restrict__ term_off) {
    const int lane = threadIdx.x & 31;
    const int line = blockIdx.x * 8 + (threadIdx.x >> 5), i = line / N, j = line - i * N;
    if (line == N * N - 1 && lane == 0) term_off[info[I_NSRC]] = info[I_NTERM];
    int pg = off_gm[line], ps = off_src[line], pt = off_term[line], pp = off_gp[line];
    const int ngm = info[I_NGM];
    if (ps == off_src[line + 1] && pp == off_gp[line + 1]) return;   // nothing on this line: the whole warp
    const int base = line * N;
    const unsigned below = (1u << lane) - 1u;
    for (int k0 = 0; k0 < N; k0 += 32) {
        const int k = k0 + lane;
        const int f = k < N ? flags[base + k] : 0;
        const bool g = f & 2, p = f & 4, s = (f & src_mask) != 0;
        const unsigned mg = __ballot_sync(0xffffffffu, g), mp = __ballot_sync(0xffffffffu, p);
        const unsigned ms = __ballot_sync(0xffffffffu, s);
        if (!(ms | mp)) continue;
        int nt = 0;
        if (s) {
            const int want = g ? 6 : 2;   // gamma- and gamma+ neighbours, or gamma- neighbours
            nt = g ? 1 : 0;
            if (!g || direct)
                for (int d = 0; d < 6; ++d) {
                    const int ii = i + c_dir[d][0], jj = j + c_dir[d][1], kk = k + c_dir[d][2];
                    if (in_grid(ii, jj, kk, N) && (flags[(ii * N + jj) * N + kk] & want)) ++nt;
                }
        }
        const int et = warp_inclusive_scan(nt);
        if (p) {
            const int x = pp + __popc(mp & below);
            gp[x] = base + k;
            node_of[base + k] = ngm + x;
        }
        if (g) {
            const int x = pg + __popc(mg & below);
            gm[x] = base + k;
            node_of[base + k] = x;
        }
        if (s) {
            const int x = ps + __popc(ms & below);
            src_lin[x] = base + k;
            term_off[x] = pt + et - nt;
        }
        pp += __popc(mp);
        pg += __popc(mg);
        ps += __popc(ms);
        pt += __shfl_sync(0xffffffffu, et, 31);
    }
}

// Closure per gamma- node: partner p with the largest t = phi(p)/(phi(p)-phi(m)),
// first in the order +x,-x,+y,-y,+z,-z on ties; x* = x_p + t (x_m - x_p).
// Separate round-to-nearest operations (no contraction) so that the values
// are reproducible by any IEEE float64 implementation of the same formula.
__global__ void k_closure(const double* __restrict__ phi, const uint8_t* __restrict__ flags, const int* __restrict__ gm,
                          int n, int N, double h, double o0, double o1, double o2,
                          int* __restrict__ partner, double* __restrict__ tw, double* __restrict__ xstar) {
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) {
        const int m = gm[r];
        const int i = m / (N * N), j = (m / N) % N, k = m % N;
        const double pm = phi[m];
        double best = -1.0;
        int bp = m, bd = 0;
        for (int d = 0; d < 6; ++d) {
            const int ii = i + c_dir[d][0], jj = j + c_dir[d][1], kk = k + c_dir[d][2];
            const int p = (ii * N + jj) * N + kk;   // in the grid: gamma- is off the faces
            if (flags[p] & 1) {
                const double pp = phi[p];
                const double t = __ddiv_rn(pp, __dsub_rn(pp, pm));
                if (t > best) { best = t; bp = p; bd = d; }
            }
        }
        partner[r] = bp;
        tw[r] = best;
        const int ip[3] = {i + c_dir[bd][0], j + c_dir[bd][1], k + c_dir[bd][2]};
        const int im[3] = {i, j, k};
        const double org[3] = {o0, o1, o2};
        for (int c = 0; c < 3; ++c) {
            const double xp = __dadd_rn(org[c], __dmul_rn((double)ip[c], h));
            const double xm = __dadd_rn(org[c], __dmul_rn((double)im[c], h));
            xstar[3 * (long long)r + c] = __dadd_rn(xp, __dmul_rn(best, __dsub_rn(xm, xp)));
        }
    }
}

// unknown number of each gamma- node's closure partner (a gamma+ node)
__global__ void k_partner_unknown(const int* __restrict__ partner, int n, const int* __restrict__ node_of,
                                  int* __restrict__ pu) {
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < n; r += gridDim.x * blockDim.x) pu[r] = node_of[partner[r]];
}

// ------------------------------------------------------------ source recipe
// rho(x) = coef(x) q(x) on gamma- (coef = |D_x| for the double layer, or 1
// when D_x is empty or for the single layer); rho(k) = -sum q(n) over the
// gamma- neighbours n of a D-node k (k is in D_n for each of them).
//
// Direct formulation (eq. [dp]): rho = chi_{M-} (6 + s - neighbour sum) u
// on gamma: at a gamma- node n, (6 + s) u(n) minus u at its neighbours in
// gamma (gamma- and gamma+); at a D-node, minus u at its gamma- neighbours
// (a node outside N+ has no gamma+ neighbour). gidx holds the unknown
// number of every gamma node.
__global__ void k_term_fill(const int* __restrict__ src, int ns, const uint8_t* __restrict__ flags, int N,
                            const int* __restrict__ gidx, const int* __restrict__ off, int layer, double s6,
                            int* __restrict__ tidx, double* __restrict__ tcoef) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < ns; s += gridDim.x * blockDim.x) {
        const int x = src[s];
        int e = off[s];
        const uint8_t f = flags[x];
        if ((f & 2) && layer == BAE_LAYER_DIRECT) {
            tidx[e] = gidx[x];
            tcoef[e] = s6;
            ++e;
            const int i = x / (N * N), j = (x / N) % N, k = x % N;
            for (int d = 0; d < 6; ++d) {
                const int y = ((i + c_dir[d][0]) * N + j + c_dir[d][1]) * N + k + c_dir[d][2];   // in the grid
                if (flags[y] & 6) {
                    tidx[e] = gidx[y];
                    tcoef[e] = -1.0;
                    ++e;
                }
            }
            continue;
        }
        if (f & 2) {
            const int c = f >> 4;
            tidx[e] = gidx[x];
            tcoef[e] = (layer == BAE_LAYER_DOUBLE && c > 0) ? (double)c : 1.0;
            continue;
        }
        const int i = x / (N * N), j = (x / N) % N, k = x % N;
        for (int d = 0; d < 6; ++d) {
            const int ii = i + c_dir[d][0], jj = j + c_dir[d][1], kk = k + c_dir[d][2];
            if (!in_grid(ii, jj, kk, N)) continue;
            const int y = (ii * N + jj) * N + kk;
            if (flags[y] & 2) {
                tidx[e] = gidx[y];
                tcoef[e] = -1.0;
                ++e;
            }
        }
    }
}

struct Scratch {
    cudaStream_t st;
    std::vector<void*> ptrs;
    explicit Scratch(cudaStream_t s) : st(s) {}
    ~Scratch() { for (void* p : ptrs) dev_free(p, st); }
    template <typename T> T* get(long long n) { T* p = dev_alloc_n<T>(n, st); ptrs.push_back(p); return p; }
};

// out[i] = nearest float32 of in[i]
__global__ void k_to_float(const double* __restrict__ in, long long n, float* __restrict__ out) {
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
        out[i] = (float)in[i];
}

int grid_for(long long n) { return (int)std::min<long long>((n + 255) / 256, 152LL * 32); }

// ------------------------------------------------- swapped convolution view
// out[swap_axes(x)] = in[x] over the N^3 grid. sw = 1 maps k-lines onto
// k-lines (a copy, grid-stride); sw = 2 transposes the (i, k) plane of
// every j through a 32 x 32 shared-memory tile (grid: k tiles, i tiles, j;
// 256 threads), so that reads and writes are both coalesced.
template <typename T>
__global__ void k_swap_grid(const T* __restrict__ in, T* __restrict__ out, int N, int sw) {
    if (sw == 1) {
        const long long n3 = (long long)N * N * N;
        for (long long x = blockIdx.x * (long long)blockDim.x + threadIdx.x; x < n3; x += (long long)gridDim.x * blockDim.x)
            out[swap_axes(x, 1, N)] = in[x];
        return;
    }
    __shared__ T tile[32][33];
    const int j = blockIdx.z, i0 = blockIdx.y * 32, k0 = blockIdx.x * 32;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int r = ty; r < 32; r += 8) {
        const int i = i0 + r, k = k0 + tx;
        if (i < N && k < N) tile[r][tx] = in[((long long)i * N + j) * N + k];
    }
    __syncthreads();
    for (int r = ty; r < 32; r += 8) {
        const int k = k0 + r, i = i0 + tx;
        if (i < N && k < N) out[((long long)k * N + j) * N + i] = tile[tx][r];
    }
}

// smap[src_lin[s]] = s (smap preset to -1)
__global__ void k_src_map(const int* __restrict__ src_lin, int ns, int* __restrict__ smap) {
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < ns; s += gridDim.x * blockDim.x) smap[src_lin[s]] = s;
}

// Per line of the swapped grid: the number of its sources (swapped flags &
// src_mask: the nodes the plain recipe lists) and of their terms. A warp per
// line.
__global__ void __launch_bounds__(256) k_view_count(const uint8_t* __restrict__ vflags, int N, int sw, int src_mask,
                                                   const int* __restrict__ smap, const int* __restrict__ term_off,
                                                   int* __restrict__ cnt_src, int* __restrict__ cnt_term) {
    const int line = blockIdx.x * 8 + (threadIdx.x >> 5);
    const long long base = (long long)line * N;
    int c0 = 0, c1 = 0;
    for (int k = threadIdx.x & 31; k < N; k += 32) {
        const int s = (vflags[base + k] & src_mask) ? smap[swap_axes(base + k, sw, N)] : -1;
        if (s >= 0) {   // every source node of the swapped flags is in the plain recipe
            c0 += 1;
            c1 += term_off[s + 1] - term_off[s];
        }
    }
    c0 = __reduce_add_sync(0xffffffffu, c0);
    c1 = __reduce_add_sync(0xffffffffu, c1);
    if ((threadIdx.x & 31) == 0) {
        cnt_src[line] = c0;
        cnt_term[line] = c1;
    }
}

// The swapped recipe in lexicographic order of the swapped grid: a warp per
// line ranks its sources from the line's offsets; vorig[pos] = the source's
// number in the plain recipe.
__global__ void __launch_bounds__(256) k_view_scatter(const uint8_t* __restrict__ vflags, int N, int sw, int src_mask,
                                                     const int* __restrict__ smap, const int* __restrict__ term_off,
                                                     const int* __restrict__ off_src,
                                                     const int* __restrict__ off_term, int n_src, int n_terms,
                                                     int* __restrict__ vsrc_lin, int* __restrict__ vterm_off,
                                                     int* __restrict__ vorig) {
    const int lane = threadIdx.x & 31;
    const int line = blockIdx.x * 8 + (threadIdx.x >> 5);
    if (line == N * N - 1 && lane == 0) vterm_off[n_src] = n_terms;
    int ps = off_src[line], pt = off_term[line];
    if (ps == off_src[line + 1]) return;   // no source on this line: the whole warp
    const long long base = (long long)line * N;
    for (int k0 = 0; k0 < N; k0 += 32) {
        const int k = k0 + lane;
        int nt = 0, s = -1;
        if (k < N && (vflags[base + k] & src_mask)) s = smap[swap_axes(base + k, sw, N)];
        const unsigned ms = __ballot_sync(0xffffffffu, s >= 0);   // the same nodes as k_view_count counts
        if (!ms) continue;
        if (s >= 0) nt = term_off[s + 1] - term_off[s];
        const int et = warp_inclusive_scan(nt);
        if (s >= 0) {
            const int pos = ps + __popc(ms & ((1u << lane) - 1u));
            vsrc_lin[pos] = (int)(base + k);
            vterm_off[pos] = pt + et - nt;
            vorig[pos] = s;
        }
        ps += __popc(ms);
        pt += __shfl_sync(0xffffffffu, et, 31);
    }
}

// the terms of swapped source pos: those of plain source vorig[pos]
__global__ void k_view_terms(const int* __restrict__ vorig, const int* __restrict__ vterm_off, int ns,
                             const int* __restrict__ term_off, const int* __restrict__ term_idx,
                             const double* __restrict__ term_coef, const float* __restrict__ term_coef32,
                             int* __restrict__ vidx, double* __restrict__ vcoef, float* __restrict__ vcoef32) {
    for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < ns; p += gridDim.x * blockDim.x) {
        const int s = vorig[p];
        if (s < 0 || s >= ns) continue;   // preset -1: a position no scatter wrote
        const int o = term_off[s], n = term_off[s + 1] - o, d = vterm_off[p];
        for (int e = 0; e < n; ++e) {
            vidx[d + e] = term_idx[o + e];
            vcoef[d + e] = term_coef[o + e];
            vcoef32[d + e] = term_coef32[o + e];
        }
    }
}

// out[r] = swap_axes(in[r])
__global__ void k_swap_index(const int* __restrict__ in, long long n, int N, int sw, int* __restrict__ out) {
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < n; r += (long long)gridDim.x * blockDim.x)
        out[r] = (int)swap_axes(in[r], sw, N);
}

// Builds the swapped view (Geometry::cv_*) of a built geometry.
void build_view(Geometry& g, int sw, int src_mask, Scratch& sc, cudaStream_t st) {
    const int N = g.N;
    const long long n3 = (long long)N * N * N, nl = (long long)N * N;
    g.cv_swap = sw;
    g.cv_lo = g.ext_lo[sw];
    g.cv_hi = g.ext_hi[sw];
    g.cv_flags = dev_alloc_n<uint8_t>(n3, st);
    if (sw == 1)
        BAE_LAUNCH("k_swap_grid", st, k_swap_grid<uint8_t><<<grid_for(n3), 256, 0, st>>>(g.flags, g.cv_flags, N, sw));
    else
        BAE_LAUNCH("k_swap_grid", st,
                   k_swap_grid<uint8_t><<<dim3(ceil_div(N, 32), ceil_div(N, 32), N), 256, 0, st>>>(g.flags, g.cv_flags,
                                                                                                   N, sw));
    int* smap = sc.get<int>(n3);
    BAE_CUDA(cudaMemsetAsync(smap, 0xff, n3 * sizeof(int), st));
    BAE_LAUNCH("k_src_map", st, k_src_map<<<grid_for(g.n_src), 256, 0, st>>>(g.src_lin, (int)g.n_src, smap));
    g.cv_line_off = dev_alloc_n<int>(nl + 1, st);   // per-line source counts, then their scan
    int* off_src = g.cv_line_off;
    int* off_term = sc.get<int>(nl + 1);
    int* info = sc.get<int>(I_COUNT);
    BAE_LAUNCH("k_view_count", st,
               k_view_count<<<(unsigned)(nl / 8), 256, 0, st>>>(g.cv_flags, N, sw, src_mask, smap, g.term_off, off_src,
                                                             off_term));
    // CTAs 0 and 1 scan the two counts (the other arrays are not read)
    BAE_LAUNCH("k_scan_lines", st, k_scan_lines<<<2, 1024, 0, st>>>(off_src, off_term, off_src, off_term, nullptr, N, info));
    g.cv_src_lin = dev_alloc_n<int>(g.n_src, st);
    g.cv_term_off = dev_alloc_n<int>(g.n_src + 1, st);
    int* vorig = sc.get<int>(std::max(1LL, g.n_src));
    BAE_CUDA(cudaMemsetAsync(vorig, 0xff, std::max(1LL, g.n_src) * sizeof(int), st));
    BAE_LAUNCH("k_view_scatter", st,
               k_view_scatter<<<(unsigned)(nl / 8), 256, 0, st>>>(g.cv_flags, N, sw, src_mask, smap, g.term_off, off_src,
                                                               off_term, (int)g.n_src, (int)g.n_terms, g.cv_src_lin,
                                                               g.cv_term_off, vorig));
    g.cv_term_idx = dev_alloc_n<int>(g.n_terms, st);
    g.cv_term_coef = dev_alloc_n<double>(g.n_terms, st);
    g.cv_term_coef32 = dev_alloc_n<float>(g.n_terms, st);
    BAE_LAUNCH("k_view_terms", st,
               k_view_terms<<<grid_for(g.n_src), 256, 0, st>>>(vorig, g.cv_term_off, (int)g.n_src, g.term_off,
                                                               g.term_idx, g.term_coef, g.term_coef32, g.cv_term_idx,
                                                               g.cv_term_coef, g.cv_term_coef32));
    g.cv_gm = dev_alloc_n<int>(g.n_gm, st);
    g.cv_partner = dev_alloc_n<int>(g.n_gm, st);
    BAE_LAUNCH("k_swap_index", st, k_swap_index<<<grid_for(g.n_gm), 256, 0, st>>>(g.gm, g.n_gm, N, sw, g.cv_gm));
    BAE_LAUNCH("k_swap_index", st,
               k_swap_index<<<grid_for(g.n_gm), 256, 0, st>>>(g.partner, g.n_gm, N, sw, g.cv_partner));
}

}  // namespace

void Geometry::release() {
    void* ps[] = {flags,    gm,          gp,         node_of,     partner,      partner_u,   t,
                  xstar,    line_off,    src_lin,    term_off,    term_idx,     term_coef,   term_coef32,
                  cv_flags, cv_gm,       cv_partner, cv_line_off, cv_src_lin,   cv_term_off, cv_term_idx,
                  cv_term_coef, cv_term_coef32};
    for (void* p : ps) if (p) dev_free(p, stream);
    flags = nullptr; gm = gp = node_of = partner = partner_u = nullptr; t = xstar = nullptr;
    line_off = src_lin = term_off = term_idx = nullptr; term_coef = nullptr; term_coef32 = nullptr;
    cv_flags = nullptr; cv_gm = cv_partner = cv_line_off = cv_src_lin = cv_term_off = cv_term_idx = nullptr;
    cv_term_coef = nullptr; cv_term_coef32 = nullptr;
    cv_swap = 0;
}

void build_geometry(const double* phi, int N, double h, const double origin[3], int layer, double s, Geometry& g,
                    cudaStream_t st) {
    const long long n3 = (long long)N * N * N;
    Scratch sc(st);
    g.stream = st;
    g.N = N;
    g.h = h;
    for (int c = 0; c < 3; ++c) g.origin[c] = origin[c];
    g.layer = layer;

    const long long nl = (long long)N * N;
    int* info = sc.get<int>(I_COUNT);
    BAE_CUDA(cudaMemsetAsync(info, 0, I_COUNT * sizeof(int), st));
    const int n_words = (int)nl * ceil_div(N, 32);
    unsigned* w_in = sc.get<unsigned>(n_words);
    unsigned* w_gm = sc.get<unsigned>(n_words);
    unsigned* w_gp = sc.get<unsigned>(n_words);
    BAE_LAUNCH("k_inside", st, k_inside<<<ceil_div(n_words, 32), 256, 0, st>>>(phi, N, w_in, info));
    BAE_LAUNCH("k_gamma_words", st, k_gamma_words<<<ceil_div(n_words, 256), 256, 0, st>>>(w_in, N, w_gm, w_gp));
    const bool direct = layer == BAE_LAYER_DIRECT;
    // gamma- and D-nodes (double layer, direct formulation), or gamma- only
    const int src_mask = layer == BAE_LAYER_SINGLE ? 2 : (2 | 8);
    g.flags = dev_alloc_n<uint8_t>(n3, st);
    g.line_off = dev_alloc_n<int>(nl + 1, st);   // per-line source counts, then their scan
    int* off_gm = sc.get<int>(nl + 1);
    int* off_term = sc.get<int>(nl + 1);
    int* off_gp = sc.get<int>(nl + 1);
    int* box = sc.get<int>(nl);
    BAE_LAUNCH("k_flags_lines", st,
               k_flags_lines<<<(unsigned)(nl / 8), 256, 0, st>>>(w_in, w_gm, w_gp, N, src_mask, direct, g.flags, off_gm,
                                                                 g.line_off, off_term, off_gp, box, info));
    BAE_LAUNCH("k_scan_lines", st, k_scan_lines<<<5, 1024, 0, st>>>(off_gm, g.line_off, off_term, off_gp, box, N, info));
    int rec[I_COUNT];
    BAE_CUDA(cudaMemcpyAsync(rec, info, sizeof(rec), cudaMemcpyDeviceToHost, st));
    BAE_CUDA(cudaStreamSynchronize(st));
    if (rec[I_ERR] & 1) throw Error(BAE_ERR_INVALID_ARG, "phi contains non-finite values");
    if (rec[I_ERR] & 2) throw Error(BAE_ERR_GEOMETRY, "M+ or gamma- reaches the faces of the grid box");
    g.n_gm = rec[I_NGM];
    g.n_src = rec[I_NSRC];
    g.n_terms = rec[I_NTERM];
    g.n_gp = rec[I_GP];
    g.n_mp = rec[I_MP];
    if (g.n_gm == 0) throw Error(BAE_ERR_GEOMETRY, "gamma- is empty (no interior node)");

    g.n_unk = direct ? g.n_gm + g.n_gp : g.n_gm;
    g.gm = dev_alloc_n<int>(g.n_gm, st);
    g.gp = dev_alloc_n<int>(std::max(1LL, g.n_gp), st);
    g.node_of = dev_alloc_n<int>(n3, st);
    g.src_lin = dev_alloc_n<int>(g.n_src, st);
    g.term_off = dev_alloc_n<int>(g.n_src + 1, st);
    BAE_LAUNCH("k_scatter_lines", st,
               k_scatter_lines<<<(unsigned)(nl / 8), 256, 0, st>>>(g.flags, N, src_mask, direct, off_gm, g.line_off,
                                                                off_term, off_gp, info, g.gm, g.gp, g.node_of,
                                                                g.src_lin, g.term_off));
    // closure
    g.partner = dev_alloc_n<int>(g.n_gm, st);
    g.t = dev_alloc_n<double>(g.n_gm, st);
    g.xstar = dev_alloc_n<double>(3 * g.n_gm, st);
    BAE_LAUNCH("k_closure", st, k_closure<<<grid_for(g.n_gm), 256, 0, st>>>(phi, g.flags, g.gm, (int)g.n_gm, N, h, origin[0], origin[1], origin[2],
                                                g.partner, g.t, g.xstar));
    if (direct) {
        g.partner_u = dev_alloc_n<int>(g.n_gm, st);
        BAE_LAUNCH("k_partner_unknown", st,
                   k_partner_unknown<<<grid_for(g.n_gm), 256, 0, st>>>(g.partner, (int)g.n_gm, g.node_of, g.partner_u));
    }
    // source recipe
    g.term_idx = dev_alloc_n<int>(g.n_terms, st);
    g.term_coef = dev_alloc_n<double>(g.n_terms, st);
    BAE_LAUNCH("k_term_fill", st, k_term_fill<<<grid_for(g.n_src), 256, 0, st>>>(g.src_lin, (int)g.n_src, g.flags, N, g.node_of, g.term_off, layer,
                                                   6.0 + s, g.term_idx, g.term_coef));
    g.term_coef32 = dev_alloc_n<float>(g.n_terms, st);
    BAE_LAUNCH("k_to_float", st, k_to_float<<<grid_for(g.n_terms), 256, 0, st>>>(g.term_coef, g.n_terms, g.term_coef32));
    // planes holding every source (gamma- and D-nodes, or M+ for the
    // volume term, whose planes lie between) and every gathered node
    // (gamma- and the partners, one step from gamma-), along each axis
    const int slot[3][2] = {{I_FIRST, I_LAST}, {I_FIRSTY, I_LASTY}, {I_FIRSTZ, I_LASTZ}};
    for (int ax = 0; ax < 3; ++ax) {
        const long long first = N - rec[slot[ax][0]], last = rec[slot[ax][1]] - 1;
        g.src_lo[ax] = (int)first;
        g.src_hi[ax] = (int)last + 1;
        g.ext_lo[ax] = (int)std::max(0LL, first - 1);
        g.ext_hi[ax] = (int)std::min((long long)N, last + 2);
    }
    g.plane_lo = g.ext_lo[0];
    g.plane_hi = g.ext_hi[0];
    // the axis of fewest planes (by more than a tenth) for the pruned
    // applies, which transform only the planes of their first axis
    const char* env = std::getenv("BAE_CONV_AXIS");
    const bool keep_x = env && (env[0] == 'x' || env[0] == 'X');
    int sw = 0;
    if (!direct && !keep_x)
        for (int ax = 1; ax < 3; ++ax)
            if (10 * (g.ext_hi[ax] - g.ext_lo[ax]) < 9 * (g.ext_hi[sw] - g.ext_lo[sw])) sw = ax;
    g.view_axis = sw;
}

void build_geometry_view(Geometry& g, cudaStream_t st) {
    if (g.view_axis == 0) return;
    Scratch sc(st);
    build_view(g, g.view_axis, g.layer == BAE_LAYER_SINGLE ? 2 : (2 | 8), sc, st);
}

}  // namespace bae
