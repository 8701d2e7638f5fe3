// Amplitudes of explicit outputs from two half expansions.
//
// Split the photons at k1 = ceil(n / 2).  With C_P the coefficients of the
// state expansion (slos.cu) of photons 0..k1-1 and D_Q those of the other
// k2 = n - k1, prod_j (sum_r U[r][c_j] a_r^dagger) is the product of two
// polynomials in the a_r^dagger, so
//     a(S) = norm_t sqrt(prod S!) sum_{P + Q = S, |P| = k1} C_P D_Q,
// at most C(n, k1) complex multiply-adds per output where Glynn's sum takes
// 2^{n-1} (n - 1) complex products (n = 10: 252 against 4608).  The tables
// hold every P of S_{m,k1} and every Q of S_{m,k2} and cost as much as a few
// dozen outputs.
//
// A sub-multiset P of S is a set of k1 positions of S's sorted mode list, as a
// bit mask; of the masks that name the same P only the one that takes the
// first copies of each mode counts.  With w_l = m - l the rank of a sorted list
// l_0 <= ... <= l_{L-1} in S_{m,L} is
//     C(m+L-1, L) - 1 - sum_a MC(w_{l_a} - 1, L - a),
// (the telescoped form of the sum in expansion.cuh), one table entry per
// position, so both ranks of a mask take one pass over the n positions.
//
// Kernels:
//   split_kernel        tables in global memory (built by the expansion's
//                       level launches), LANES lanes per output, each a
//                       contiguous range of masks, added by a fixed shuffle
//                       tree;
//   split_multi_kernel  the same outputs for many unitaries: a block builds
//                       both tables of its unitaries in shared memory and a
//                       thread takes an output.  The ranks do not depend on
//                       the unitary, so a thread forms them once for the
//                       block's kMulti unitaries.  Its callers take logarithms
//                       of probabilities that can be zero but for rounding; an
//                       amplitude below 2^-30 of the product of its rows'
//                       norms, where rounding decides, is formed by Glynn's
//                       sum in the tile kernel's FP64 order (glynn_row_sums).

#include <algorithm>
#include <cmath>

#include "expansion.cuh"

namespace pcv {
namespace {

constexpr int kThreads = 256;
constexpr int kMaxN = 16;                // photons of the split form
constexpr int kMulti = 2;                // unitaries per block of split_multi_kernel

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

int64_t mset_h(int w, int k)
{
    if (k == 0) return 1;
    if (w <= 0) return 0;
    unsigned __int128 c = 1;
    for (int i = 1; i <= k; ++i) {
        c = c * (unsigned __int128)(w - 1 + i) / (unsigned __int128)i;
        if (c > (unsigned __int128)INT64_MAX) return -1;
    }
    return (int64_t)c;
}

int64_t binom_h(int a, int b)
{
    int64_t c = 1;
    for (int i = 1; i <= b; ++i) c = c * (a + 1 - i) / i;
    return c;
}

// FP64 instructions of the two half expansions (4 per state and occupied
// mode), or -1 where a level's ranks pass 32 bits.
double half_cost(int m, int n)
{
    const int k1 = (n + 1) / 2, k2 = n - k1;
    double c = 0.0;
    for (int k = 1; k <= k1; ++k) {
        const int64_t N = mset_h(m, k);
        if (N < 0 || N > (int64_t)UINT32_MAX) return -1.0;
        c += (k <= k2 ? 2.0 : 1.0) * 4.0 * m * (double)mset_h(m, k - 1);
    }
    return c;
}

struct SplitOut {
    int m, n, k1, k2;
    int64_t masks;                       // C(n, k1)
    const uint8_t* outputs;              // [n_out][m]
    int64_t n_out;
    double norm_t;
    double2* amp;                        // or null
    double* prob;                        // or null
};

// MC(w, j) for w <= m, j <= k1 as 32-bit counts: t[w * (k1 + 1) + j] =
// C(w + j - 1, j).
__device__ void count_table(uint32_t* t, int m, int k1)
{
    for (int w = threadIdx.x; w <= m; w += blockDim.x) {
        uint64_t c = 1;
        t[w * (k1 + 1)] = 1;
        for (int j = 1; j <= k1; ++j) {
            c = c * (uint64_t)(w + j - 1) / (uint64_t)j;
            t[w * (k1 + 1) + j] = (uint32_t)c;
        }
    }
}

// The b-th mask of k bits in increasing order.
__device__ uint32_t nth_mask(int64_t b, int k)
{
    uint32_t mask = 0;
    for (int j = k; j >= 1; --j) {
        int t = j - 1;
        int64_t c = 0;                   // C(t, j)
        for (;;) {
            const int64_t nx = c == 0 ? 1 : c * (t + 1) / (t + 1 - j);
            if (nx > b) break;
            c = nx;
            ++t;
        }
        mask |= 1u << t;
        b -= c;
    }
    return mask;
}

// The next larger mask with as many bits.
__device__ __forceinline__ uint32_t next_mask(uint32_t x)
{
    const uint32_t c = x & (0u - x), r = x + c;
    return r | (((x ^ r) >> 2) >> (__ffs(x) - 1));
}

// Ranks of the positions in `mask` (P) and of the others (Q); row[p] is the
// count table's row of position p's mode.
template <int NMAX>
__device__ __forceinline__ void split_ranks(const uint32_t* t, const int* row, int n, int k1, int k2, uint32_t mask,
                                            uint32_t& rp, uint32_t& rq)
{
    int a = k1, c = k2;
#pragma unroll
    for (int p = 0; p < NMAX; ++p) {
        if (p >= n) break;
        const bool in = (mask >> p) & 1u;
        const uint32_t v = t[row[p] + (in ? a : c)];
        if (in) {
            rp -= v;
            --a;
        } else {
            rq -= v;
            --c;
        }
    }
}

// Output o as count-table rows of its sorted list; same: bit p set where
// position p repeats the mode of p - 1; f = prod S!.  False when its photon
// number is not n.
template <int NMAX>
__device__ __forceinline__ bool decode_rows(const SplitOut& a, int64_t o, int* row, uint32_t& same, double& f)
{
    const int m = a.m, n = a.n;
    const uint8_t* occ = a.outputs + o * m;
    int r = 0, left = occ[0], run = 0, cnt = 0;
    same = 0;
    f = 1.0;
#pragma unroll
    for (int p = 0; p < NMAX; ++p) {
        if (p >= n) break;
        while (left == 0 && r + 1 < m) {
            ++r;
            left = occ[r];
            run = 0;
        }
        row[p] = (m - r - 1) * (a.k1 + 1);
        if (left > 0) {
            --left;
            ++cnt;
            if (run > 0) same |= 1u << p;
            f *= ++run;
        }
    }
    for (cnt += left, ++r; r < m; ++r) cnt += occ[r];
    return cnt == n;
}

struct SplitArgs {
    SplitOut o;
    uint32_t n1, n2;                     // |S_{m,k1}| - 1, |S_{m,k2}| - 1
    const double2* F;                    // [S_{m,k1}]
    const double2* G;                    // [S_{m,k2}]
};

template <int NMAX, int LANES>
__global__ void __launch_bounds__(kThreads) split_kernel(const __grid_constant__ SplitArgs a)
{
    extern __shared__ uint32_t s_t[];
    const int m = a.o.m, n = a.o.n, k1 = a.o.k1, k2 = a.o.k2;
    count_table(s_t, m, k1);
    __syncthreads();
    const int lane = threadIdx.x % LANES;
    const int64_t o = ((int64_t)blockIdx.x * kThreads + threadIdx.x) / LANES;
    const bool live = o < a.o.n_out;
    int row[NMAX];
    uint32_t same = 0;
    double f = 1.0;
    const bool ok = live && decode_rows<NMAX>(a.o, o, row, same, f);
    double2 acc = make_double2(0.0, 0.0);
    if (ok) {
        const int64_t per = (a.o.masks + LANES - 1) / LANES;
        const int64_t q0 = lane * per, q1 = min(a.o.masks, q0 + per);
        if (q0 < q1) {
            uint32_t mask = nth_mask(q0, k1);
            for (int64_t q = q0; q < q1; ++q) {
                if (((mask & same) & ~(mask << 1)) == 0) {
                    uint32_t rp = a.n1, rq = a.n2;
                    split_ranks<NMAX>(s_t, row, n, k1, k2, mask, rp, rq);
                    cmac(acc, __ldg(a.F + rp), __ldg(a.G + rq));
                }
                mask = next_mask(mask);
            }
        }
    }
    for (int off = LANES / 2; off > 0; off >>= 1) {
        acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
        acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
    }
    if (live && lane == 0) {
        double2 v = make_double2(0.0, 0.0);
        if (ok) {
            const double sc = sqrt(f) * a.o.norm_t;
            v = make_double2(acc.x * sc, acc.y * sc);
        }
        if (a.o.amp) a.o.amp[o] = v;
        if (a.o.prob) a.o.prob[o] = fma(v.x, v.x, v.y * v.y);
    }
}

struct SplitMultiArgs {
    SplitOut o;
    const double2* U;                    // [B][m][m]
    int B;
    int cols[kMaxN];
    int64_t per_block;                   // outputs per block
    int n1, n2, ns;                      // |S_{m,k1}|, |S_{m,k2}|, |S_{m,k1-1}| (scratch)
};

// Glynn's sum of one output in Gray order, rows ascending, FP64 throughout.
template <int NMAX>
__device__ __forceinline__ double2 glynn_row_sums(const double2* U, const SplitMultiArgs& a, const int* row)
{
    const int m = a.o.m, n = a.o.n, w1 = a.o.k1 + 1;
    double2 y[NMAX];
    for (int i = 0; i < n; ++i) {
        const double2* Ur = U + (size_t)(m - 1 - row[i] / w1) * m;
        y[i] = Ur[a.cols[0]];
        for (int j = 1; j < n; ++j) caxpy(y[i], 1.0, Ur[a.cols[j]]);
    }
    double2 acc = make_double2(0.0, 0.0);
    const uint32_t steps = 1u << (n - 1);
    for (uint32_t k = 0; k < steps; ++k) {
        double2 p = y[0];
        for (int i = 1; i < n; ++i) p = cmul(p, y[i]);
        caxpy(acc, (k & 1) ? -1.0 : 1.0, p);
        if (k + 1 == steps) break;
        const int b = __ffs(k + 1) - 1;
        const double sd = (((k + 1) >> (b + 1)) & 1) ? 2.0 : -2.0;
        for (int i = 0; i < n; ++i) caxpy(y[i], sd, U[(size_t)(m - 1 - row[i] / w1) * m + a.cols[b + 1]]);
    }
    return acc;
}

template <int NMAX>
__global__ void __launch_bounds__(kThreads, 2) split_multi_kernel(const __grid_constant__ SplitMultiArgs a)
{
    extern __shared__ double2 s_tab[];   // per unitary F, G; one scratch level; one column; the counts
    __shared__ int s_lost;
    __shared__ uint16_t s_list[kThreads * kMulti];
    const int m = a.o.m, n = a.o.n, k1 = a.o.k1, k2 = a.o.k2, w1 = k1 + 1;
    double2* s_scratch = s_tab + kMulti * (a.n1 + a.n2);
    double2* s_u = s_scratch + a.ns;
    uint32_t* s_t = (uint32_t*)(s_u + m);
    int* s_e = (int*)(s_t + (m + 1) * w1);   // per unitary and mode: exponent of the row's squared norm, stride w1
    const int b0 = blockIdx.y * kMulti;
    count_table(s_t, m, k1);
    for (int q = threadIdx.x; q < kMulti * m; q += kThreads) {
        const double2* Ur = a.U + ((size_t)min(b0 + q / m, a.B - 1) * m + q % m) * m;
        double f = 0.0;
        for (int j = 0; j < n; ++j) {
            const double2 u = Ur[a.cols[j]];
            f = fma(u.x, u.x, fma(u.y, u.y, f));
        }
        s_e[q / m * m * w1 + (m - 1 - q % m) * w1] = f > 0.0 && isfinite(f) ? ilogb(f) : 0;   // at the mode's table row
    }
    // both tables of each unitary, level by level; the last level lands in
    // place, the one before in the scratch, and so on back
    for (int j = 0; j < kMulti; ++j) {
        const int b = min(b0 + j, a.B - 1);
        const double2* U = a.U + (size_t)b * m * m;
        for (int side = 0; side < 2; ++side) {
            const int K = side ? k2 : k1;
            uint32_t prev_n = 1;
            double2* fin = s_tab + j * (a.n1 + a.n2) + (side ? a.n1 : 0);
            for (int k = 1; k <= K; ++k) {
                double2* cur = ((K - k) & 1) ? s_scratch : fin;
                const double2* prev = ((K - k) & 1) ? fin : s_scratch;
                __syncthreads();
                const int col = a.cols[(side ? k1 : 0) + k - 1];
                for (int r = threadIdx.x; r < m; r += kThreads) s_u[r] = U[(size_t)r * m + col];
                __syncthreads();
                uint32_t N = 1;          // |S_{m,k}|
                for (int q = 1; q <= k; ++q) N = (uint32_t)((uint64_t)N * (m + q - 1) / q);
                for (uint32_t i = threadIdx.x; i < N; i += kThreads) {
                    constexpr int KM = (NMAX + 1) / 2;
                    int row[KM];                     // the list as count-table rows
                    uint32_t idx = i, pre = 0, suf = 0;
                    int v = 0;
#pragma unroll
                    for (int p = 0; p < KM; ++p) {
                        if (p >= k) break;
                        v = next_mode<uint32_t>(s_t, w1, m, v, k - 1 - p, idx);
                        row[p] = (m - v - 1) * w1;
                    }
                    // predecessor ranks as in slos.cu
                    pre = prev_n - 1;
#pragma unroll
                    for (int q = 1; q < KM; ++q)
                        if (q < k) suf += s_t[row[q] + k - q];
                    double2 acc = make_double2(0.0, 0.0);
#pragma unroll
                    for (int p = 0; p < KM; ++p) {
                        if (p >= k) break;
                        const int nxt = p + 1 < k ? row[p + 1 < KM ? p + 1 : p] : -1;
                        if (nxt != row[p]) {
                            const double2 u = s_u[m - 1 - row[p] / w1];
                            if (k == 1) acc = u;
                            else cmac(acc, u, prev[pre - suf]);
                        }
                        if (p + 1 < k) {
                            pre -= s_t[row[p] + k - 1 - p];
                            suf -= s_t[nxt + k - 1 - p];
                        }
                    }
                    cur[i] = acc;
                }
                prev_n = N;
            }
        }
    }
    __syncthreads();
    const int64_t o0 = (int64_t)blockIdx.x * a.per_block;
    const int64_t o1 = min(a.o.n_out, o0 + a.per_block);
    for (int64_t base = o0; base < o1; base += kThreads) {
        if (threadIdx.x == 0) s_lost = 0;
        __syncthreads();
        const int64_t o = base + threadIdx.x;
        if (o < o1) {
            int row[NMAX];
            uint32_t same;
            double f;
            const bool ok = decode_rows<NMAX>(a.o, o, row, same, f);
            double2 acc[kMulti];
#pragma unroll
            for (int j = 0; j < kMulti; ++j) acc[j] = make_double2(0.0, 0.0);
            if (ok) {
                uint32_t mask = (1u << k1) - 1;
                for (int64_t q = 0; q < a.o.masks; ++q) {
                    if (((mask & same) & ~(mask << 1)) == 0) {
                        uint32_t rp = a.n1 - 1, rq = a.n2 - 1;
                        split_ranks<NMAX>(s_t, row, n, k1, k2, mask, rp, rq);
#pragma unroll
                        for (int j = 0; j < kMulti; ++j) {
                            const double2* F = s_tab + j * (a.n1 + a.n2);
                            cmac(acc[j], F[rp], F[a.n1 + rq]);
                        }
                    }
                    mask = next_mask(mask);
                }
            }
            const double sc = sqrt(f) * a.o.norm_t;
#pragma unroll
            for (int j = 0; j < kMulti; ++j) {
                if (b0 + j >= a.B) break;
                const double2 v = ok ? make_double2(acc[j].x * sc, acc[j].y * sc) : make_double2(0.0, 0.0);
                const int64_t at = (int64_t)(b0 + j) * a.o.n_out + o;
                if (a.o.amp) a.o.amp[at] = v;
                if (a.o.prob) a.o.prob[at] = fma(v.x, v.x, v.y * v.y);
                if (!ok) continue;
                const double w = fma(acc[j].x, acc[j].x, acc[j].y * acc[j].y) * f;      // |Perm|^2 / prod S!
                int e = -60;
#pragma unroll
                for (int p = 0; p < NMAX; ++p)
                    if (p < n) e += s_e[j * m * w1 + row[p]];
                if (w < scalbn(1.0, e)) s_list[atomicAdd(&s_lost, 1)] = (uint16_t)(threadIdx.x * kMulti + j);
            }
        }
        __syncthreads();
        // the outputs lost in rounding, a thread each (their order does not matter)
        for (int q = threadIdx.x; q < s_lost; q += kThreads) {
            const int j = s_list[q] % kMulti;
            const int64_t lo = base + s_list[q] / kMulti;
            int row[NMAX];
            uint32_t same;
            double f;
            decode_rows<NMAX>(a.o, lo, row, same, f);
            const double gs = ldexp(1.0 / sqrt(f) * a.o.norm_t, -(n - 1));
            const double2 g = glynn_row_sums<NMAX>(a.U + (size_t)(b0 + j) * m * m, a, row);
            const double2 v = make_double2(g.x * gs, g.y * gs);
            const int64_t at = (int64_t)(b0 + j) * a.o.n_out + lo;
            if (a.o.amp) a.o.amp[at] = v;
            if (a.o.prob) a.o.prob[at] = fma(v.x, v.x, v.y * v.y);
        }
        __syncthreads();
    }
}

template <int NMAX, int LANES>
cudaError_t go_split(const SplitArgs& a, cudaStream_t s)
{
    const size_t smem = (size_t)(a.o.m + 1) * (a.o.k1 + 1) * sizeof(uint32_t);
    if (smem > 48 * 1024) return cudaErrorInvalidConfiguration;
    const int64_t blocks = (a.o.n_out * LANES + kThreads - 1) / kThreads;
    split_kernel<NMAX, LANES><<<(unsigned)blocks, kThreads, smem, s>>>(a);
    note_launches(1);
    return cudaGetLastError();
}

template <int NMAX>
cudaError_t go_multi(const SplitMultiArgs& a, size_t smem, cudaStream_t s)
{
    const cudaError_t e = allow_dynamic_smem((const void*)split_multi_kernel<NMAX>, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((a.o.n_out + a.per_block - 1) / a.per_block), (unsigned)((a.B + kMulti - 1) / kMulti));
    split_multi_kernel<NMAX><<<grid, kThreads, smem, s>>>(a);
    note_launches(1);
    return cudaGetLastError();
}

size_t multi_smem(int m, int n)
{
    const int k1 = (n + 1) / 2;
    const int64_t n1 = mset_h(m, k1), n2 = mset_h(m, n - k1), ns = mset_h(m, k1 - 1);
    if (n1 < 0 || n1 > (1 << 20)) return SIZE_MAX;
    return (size_t)(kMulti * (n1 + n2) + ns + m) * sizeof(double2) + (size_t)(m + 1) * (k1 + 1) * sizeof(uint32_t) +
           (size_t)kMulti * m * (k1 + 1) * sizeof(int);
}

SplitOut split_out(const pcv_batch_desc& d, double norm_t)
{
    SplitOut o;
    o.m = d.m;
    o.n = d.n;
    o.k1 = (d.n + 1) / 2;
    o.k2 = d.n - o.k1;
    o.masks = binom_h(d.n, o.k1);
    o.outputs = d.outputs;
    o.n_out = d.n_out;
    o.norm_t = norm_t;
    o.amp = (double2*)d.amp;
    o.prob = d.prob;
    return o;
}

}  // namespace

// FP64 instructions of `n_out` outputs by split_kernel, its tables included
// (-1 where it does not apply: 2 <= n <= 16, 32-bit ranks).
double split_cost(int m, int n, int64_t n_out)
{
    if (n < 2 || n > kMaxN || (size_t)(m + 1) * (n / 2 + 2) * sizeof(uint32_t) > 48 * 1024) return -1.0;
    const double h = half_cost(m, n);
    return h < 0.0 ? -1.0 : h + 4.0 * (double)binom_h(n, n / 2) * (double)n_out;
}

// The count table, and two buffers for the levels of both halves.
int64_t split_workspace(int m, int n)
{
    const int k1 = (n + 1) / 2;
    return (int64_t)(al256((size_t)(m + 1) * (k1 + 1) * sizeof(int64_t)) +
                     2 * al256((size_t)2 * mset_h(m, k1) * sizeof(double2)));
}

cudaError_t launch_split(const Plan& p, const pcv_batch_desc& d, void* ws, cudaStream_t s)
{
    SplitArgs a;
    a.o = split_out(d, p.norm_t);
    const int m = d.m, k1 = a.o.k1, k2 = a.o.k2;
    const int64_t n1 = mset_h(m, k1);
    char* w = (char*)ws;
    int64_t* mc = (int64_t*)w;           w += al256((size_t)(m + 1) * (k1 + 1) * sizeof(int64_t));
    double2* buf[2];
    buf[0] = (double2*)w;                w += al256((size_t)2 * n1 * sizeof(double2));
    buf[1] = (double2*)w;
    cudaError_t e = build_multiset_table(mc, m, k1, s);
    if (e != cudaSuccess) return e;
    ExpandArgs x;
    expand_defaults(&x);
    x.source = kExpandSides;
    x.U = (const double2*)d.U;
    x.m = m;
    x.mc = mc;
    x.kmax = k1;
    x.prev_stride = x.cur_stride = n1;
    for (int k = 1; k <= k1; ++k) {
        x.k = k;
        x.B = k <= k2 ? 2 : 1;
        x.col[0] = p.cols[k - 1];
        x.col[1] = k <= k2 ? p.cols[k1 + k - 1] : 0;
        x.count = x.hi = mset_h(m, k);
        x.prev_count = mset_h(m, k - 1);
        x.prev = buf[(k - 1) & 1];
        x.cur = buf[k & 1];
        if ((e = launch_expand(x, s)) != cudaSuccess) return e;
    }
    a.n1 = (uint32_t)(n1 - 1);
    a.n2 = (uint32_t)(mset_h(m, k2) - 1);
    a.F = buf[k1 & 1];
    a.G = buf[k2 & 1] + n1;
    // a warp per output while that leaves the SMs room, then fewer lanes
    const bool many = d.n_out >= 152 * 256;
    if (d.n <= 4) return go_split<4, 1>(a, s);
    if (d.n <= 8) return many ? go_split<8, 4>(a, s) : go_split<8, 16>(a, s);
    if (d.n <= 10) return many ? go_split<10, 8>(a, s) : go_split<10, 32>(a, s);
    return many && d.n <= 12 ? go_split<16, 8>(a, s) : go_split<16, 32>(a, s);
}

// Whether split_multi_kernel takes these sizes: both tables of kMulti
// unitaries fit in shared memory (with two blocks per SM) and it needs fewer
// FP64 instructions than the tile kernel's 2^{n-1} (4n - 2) per output.
bool split_multi_applies(int m, int n, int64_t n_out)
{
    if (n < 2 || n > 10 || multi_smem(m, n) > 110 * 1024) return false;
    const double per = 4.0 * (double)binom_h(n, n / 2);
    return half_cost(m, n) + per * (double)n_out < std::ldexp(4.0 * n - 2.0, n - 1) * (double)n_out;
}

cudaError_t launch_split_multi(const Plan& p, const pcv_batch_desc& d, int B, cudaStream_t s)
{
    SplitMultiArgs a;
    a.o = split_out(d, p.norm_t);
    a.U = (const double2*)d.U;
    a.B = B;
    for (int j = 0; j < kMaxN; ++j) a.cols[j] = p.cols[j];
    a.n1 = (int)mset_h(d.m, a.o.k1);
    a.n2 = (int)mset_h(d.m, a.o.k2);
    a.ns = (int)mset_h(d.m, a.o.k1 - 1);
    // one block per pair of unitaries unless that leaves SMs idle; the tables
    // are built once per block, so a block keeps at least 128 outputs
    const int64_t pairs = (B + kMulti - 1) / kMulti;
    const int64_t want = std::max<int64_t>(1, (152 * 2 + pairs - 1) / pairs);
    a.per_block = std::max<int64_t>(128, (d.n_out + want - 1) / want);
    const size_t smem = multi_smem(d.m, d.n);
    if (d.n <= 4) return go_multi<4>(a, smem, s);
    if (d.n <= 6) return go_multi<6>(a, smem, s);
    return go_multi<10>(a, smem, s);
}

}  // namespace pcv
