// Output distributions of partially distinguishable photons.
//
// Photons of one class are identical. Photons of different classes have
// orthogonal internal states, and the detectors count photons per mode only.
// Each class then evolves on its own, and the distribution of the total
// occupation is the multiset convolution of the classes' distributions:
//     P(S) = sum_{S_1 + S_2 = S} P_1(S_1) P_2(S_2),
// where each P_g is Eq. eqperm for that class's photons alone. A single
// photon entering in mode c lands in mode r with probability |U[r][c]|^2, so
// convolving with it is a gather over the occupied modes of S:
//     C(S) = sum_{r : s_r >= 1} A(S - e_r) |U[r][c]|^2.
// The source model mixes such terms with weights: the photon is absent,
// pure (in the one class of pure photons) or noisy (a class of its own).
// The host loop in pcv_api.cu sequences the launches; the kernels here
// compute one convolution step.
//
// The whole source model (launch_source) takes all 2^n pure sets together.
// The mixture is sum_P gamma^{|P|} (prod_{j not in P} T_j) p_P, p_P the
// distribution of the pure set P and T_j = alpha + beta (photon j's step).
// One photon is eliminated at a time, the last first,
//     X_{j-1}(P) = T_j X_j(P) + X_j(P u {j}),   P a subset of the photons < j,
// so a stage is one launch over every remaining set, and the 2^n - 1 steps
// T_j replace the sum over sets of n - |P| steps.  The p_P come from the
// state expansion (slos.cu) with the sets of one size as its batch: each set
// adds its last photon to the entry of the others.  2 n + 2 launches in all,
// where one set at a time took 64 distributions and 192 steps at n = 6
// (bound by about 1900 launches).
//
// Layout: a distribution over S_{m,k} is a dense float64 vector in canonical
// order. Ranks use the CUM table built by build_cum_table (O(k) per rank),
// and unranking uses the multiset-count table MC.

#include <algorithm>
#include <cmath>

#include "expansion.cuh"

namespace pcv {
namespace {

struct RankTables {
    const int64_t* mc;     // MC[a*W + k] = C(a+k-1, k)
    const int64_t* cum;    // CUM[a*W + k] = sum_{v<a} MC[(m-v)*W + k]
    int m, W;              // W = kmax + 1
};

template <int KMAX>
__device__ __forceinline__ void unrank_modes(const RankTables& t, int k, int64_t idx, int* modes)
{
    int v = 0;
    for (int p = 0; p < k; ++p) {
        const int rest = k - p - 1;
        for (;;) {
            const int64_t c = t.mc[(t.m - v) * t.W + rest];
            if (idx < c) break;
            idx -= c;
            ++v;
        }
        modes[p] = v;
    }
}

// Rank in S_{m,len} of the sorted list holding cnt[j] copies of mode dm[j].
__device__ __forceinline__ int64_t rank_counts(const RankTables& t, const int* dm, const int* cnt, int d, int len)
{
    int64_t r = 0;
    int prev = 0, pos = 0;
    for (int j = 0; j < d; ++j) {
        for (int q = 0; q < cnt[j]; ++q) {
            const int rest = len - pos - 1;
            r += t.cum[dm[j] * t.W + rest] - t.cum[prev * t.W + rest];
            prev = dm[j];
            ++pos;
        }
    }
    return r;
}

// out(S) = alpha in_same(S) + beta sum_{r: s_r >= 1} in_prev(S - e_r) |U[r][c]|^2,
// S in S_{m,k}; in_same (S_{m,k}) and in_prev (S_{m,k-1}) may be null.
struct PhotonStep {
    RankTables t;
    int k, c;
    const double2* U;
    const double* in_same;
    const double* in_prev;
    double alpha, beta;
    double* out;
    int64_t count;
};

template <int KMAX>
__global__ void __launch_bounds__(256) photon_step_kernel(const PhotonStep a)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= a.count) return;
    double acc = a.in_same ? a.alpha * a.in_same[i] : 0.0;
    if (a.in_prev && a.k >= 1) {
        int modes[KMAX];
        unrank_modes<KMAX>(a.t, a.k, i, modes);
        const int m = a.t.m, W = a.t.W, k = a.k;
        double g = 0.0;
        for (int p = 0; p < k; ++p) {
            if (p + 1 < k && modes[p + 1] == modes[p]) continue;     // last copy of each occupied mode
            // rank of the list without position p, in S_{m,k-1}
            int64_t rk = 0;
            int prev = 0, pos = 0;
            for (int q = 0; q < k; ++q) {
                if (q == p) continue;
                const int rest = (k - 1) - pos - 1;
                rk += a.t.cum[modes[q] * W + rest] - a.t.cum[prev * W + rest];
                prev = modes[q];
                ++pos;
            }
            const double2 u = a.U[(size_t)modes[p] * m + a.c];
            g = fma(fma(u.x, u.x, u.y * u.y), a.in_prev[rk], g);
        }
        acc = fma(a.beta, g, acc);
    }
    a.out[i] = acc;
}

// C(S) = sum over S_1 <= S with |S_1| = a of A(S_1) B(S - S_1), S in S_{m,a+b}.
// The sub-multisets are the bounded compositions k_j in [0, mu_j] with
// sum k_j = a over the distinct modes of S, visited in lexicographic order:
// the successor raises the last k_j that still has room while something
// remains to its right, then refills the right part as low as it can go.
struct ClassConv {
    RankTables t;
    int a, b;
    const double* A;       // S_{m,a}
    const double* B;       // S_{m,b}
    double* C;             // S_{m,a+b}
    int64_t count;
};

template <int KMAX>
__global__ void __launch_bounds__(256) class_conv_kernel(const ClassConv g)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= g.count) return;
    const int n = g.a + g.b;
    int modes[KMAX];
    unrank_modes<KMAX>(g.t, n, i, modes);
    int dm[KMAX], mu[KMAX], cap[KMAX + 1], k[KMAX], rest[KMAX];
    int d = 0;
    for (int p = 0; p < n; ++p) {
        if (p == 0 || modes[p] != modes[p - 1]) {
            dm[d] = modes[p];
            mu[d] = 0;
            ++d;
        }
        mu[d - 1] += 1;
    }
    cap[d] = 0;
    for (int j = d - 1; j >= 0; --j) cap[j] = cap[j + 1] + mu[j];
    int rem = g.a;
    for (int j = 0; j < d; ++j) {
        k[j] = max(0, rem - cap[j + 1]);
        rem -= k[j];
    }
    double acc = 0.0;
    for (;;) {
        for (int j = 0; j < d; ++j) rest[j] = mu[j] - k[j];
        const int64_t r1 = rank_counts(g.t, dm, k, d, g.a);
        const int64_t r2 = rank_counts(g.t, dm, rest, d, g.b);
        acc = fma(g.A[r1], g.B[r2], acc);
        int j = d - 2, suf = k[d - 1];
        while (j >= 0 && !(k[j] < mu[j] && suf >= 1)) {
            suf += k[j];
            --j;
        }
        if (j < 0) break;
        k[j] += 1;
        rem = suf - 1;
        for (int q = j + 1; q < d; ++q) {
            k[q] = max(0, rem - cap[q + 1]);
            rem -= k[q];
        }
    }
    g.C[i] = acc;
}

// acc[i] += w x[i]
__global__ void scale_add_kernel(double* __restrict__ acc, const double* __restrict__ x, double w, int64_t count)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) acc[i] = fma(w, x[i], acc[i]);
}

__global__ void set_one_kernel(double* p) { *p = 1.0; }

// One elimination stage: photon `photon` (the last of the j remaining ones)
// leaves.  Sets of c photons are numbered in colex order, so a set keeps its
// number as the photons above it leave, and P u {photon} has number
// C(j-1, c+1) + that of P.  A set of size c holds the blocks S_{m,c} ..
// S_{m,c+n-j}, each set's blocks concatenated, sets of one size together.
struct SourceStage {
    const int64_t* mc;             // row length n + 1
    int m, n, j;
    int col;                       // input mode of the photon that leaves
    const double2* U;
    double alpha, beta;
    const double* in;
    double* out;
    int64_t N[18];                 // |S_{m,k}|
    int64_t in_base[18], out_base[18];   // first value of the sets of size c
    int64_t in_len[18], out_len[18];     // values per set of size c
    int64_t up[18];                      // C(j-1, c+1)
    int64_t nsets[18];                   // C(j-1, c): sets of size c after the stage
    int npairs;                          // (c, block) pairs
    int pc[90], pk[90];
    int64_t pend[90];                    // blocks of 256 threads up to and including this pair
};

template <int KMAX>
__global__ void __launch_bounds__(256) source_stage_kernel(const __grid_constant__ SourceStage a)
{
    extern __shared__ double s_w[];            // |U[r][col]|^2, then the count table
    const int m = a.m, w1 = a.n + 1;
    int64_t* s_mc = (int64_t*)(s_w + m);
    for (int r = threadIdx.x; r < m; r += blockDim.x) {
        const double2 u = a.U[(size_t)r * m + a.col];
        s_w[r] = fma(u.x, u.x, u.y * u.y);
    }
    for (int q = threadIdx.x; q < (m + 1) * w1; q += blockDim.x) s_mc[q] = a.mc[q];
    __syncthreads();
    int pr = 0;
    while ((int64_t)blockIdx.x >= a.pend[pr]) ++pr;
    const int c = a.pc[pr], k = a.pk[pr];
    const int64_t e = ((int64_t)blockIdx.x - (pr ? a.pend[pr - 1] : 0)) * blockDim.x + threadIdx.x;
    const int64_t Nk = a.N[k];
    const int64_t b = e / Nk, i = e % Nk;      // set, state
    if (b >= a.nsets[c]) return;
    const double* x = a.in + a.in_base[c] + b * a.in_len[c];
    const int top = c + a.n - a.j;             // last block of a set of size c before the stage
    int64_t o = 0;                             // first value of block k in a set of size c
    for (int q = c; q < k; ++q) o += a.N[q];
    double acc = k <= top ? a.alpha * x[o + i] : 0.0;
    if (k > c) {
        const double* y = x + (o - a.N[k - 1]);
        int l[KMAX];
        int64_t idx = i;
        int v = 0;
#pragma unroll
        for (int p = 0; p < KMAX; ++p) {
            if (p >= k) break;
            v = next_mode<int64_t>(s_mc, w1, m, v, k - 1 - p, idx);
            l[p] = v;
        }
        auto t = [&](int mode, int q) { return s_mc[(m - mode - 1) * w1 + q]; };
        int64_t pre = a.N[k - 1] - 1, suf = 0;     // rank without position p, as in slos.cu
#pragma unroll
        for (int q = 1; q < KMAX; ++q)
            if (q < k) suf += t(l[q], k - q);
        double st = 0.0;
#pragma unroll
        for (int p = 0; p < KMAX; ++p) {
            if (p >= k) break;
            const int nxt = p + 1 < k ? l[p + 1 < KMAX ? p + 1 : p] : -1;
            if (nxt != l[p]) st = fma(s_w[l[p]], y[pre - suf], st);
            if (p + 1 < k) {
                pre -= t(l[p], k - 1 - p);
                suf -= t(nxt, k - 1 - p);
            }
        }
        acc = fma(a.beta, st, acc);
        // the set with the photon: its blocks start at k = c + 1
        acc += a.in[a.in_base[c + 1] + (a.up[c] + b) * a.in_len[c + 1] + (o - a.N[c]) + i];
    }
    a.out[a.out_base[c] + b * a.out_len[c] + o + i] = acc;
}

unsigned blocks_for(int64_t count) { return (unsigned)((count + 255) / 256); }

int64_t choose(int a, int b)
{
    if (b < 0 || b > a) return 0;
    int64_t c = 1;
    for (int i = 1; i <= b; ++i) c = c * (a + 1 - i) / i;
    return c;
}

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// Values of stage j (j photons remaining): per set size c the first value
// and the values per set; returns their sum.
int64_t stage_layout(const int64_t* N, int n, int j, int64_t* base, int64_t* len)
{
    int64_t t = 0;
    for (int c = 0; c <= j; ++c) {
        len[c] = 0;
        for (int k = c; k <= c + n - j; ++k) len[c] += N[k];
        base[c] = t;
        t += choose(j, c) * len[c];
    }
    return t;
}

}  // namespace

// Workspace of launch_source: the count table, two level buffers (all sets
// of one size), two stages.
SourcePlan source_plan(int m, int n, const int64_t* N)
{
    SourcePlan p{};
    p.total = -1;
    if (n < 1 || n > 16) return p;
    int64_t amp = 1, st[2] = {0, 0};
    int64_t base[18], len[18];
    for (int k = 0; k <= n; ++k) {
        p.N[k] = N[k];
        if (N[k] < 0 || N[k] > (int64_t)UINT32_MAX) return p;
        if (k < n) amp = std::max(amp, choose(n, k) * N[k]);
    }
    for (int j = n; j >= 1; --j) st[j & 1] = std::max(st[j & 1], stage_layout(N, n, j, base, len));
    p.table = al256((size_t)(m + 1) * (n + 1) * sizeof(int64_t));
    p.amp = al256((size_t)amp * sizeof(double2));
    p.st[0] = al256((size_t)std::max<int64_t>(st[0], 1) * sizeof(double));
    p.st[1] = al256((size_t)std::max<int64_t>(st[1], 1) * sizeof(double));
    p.total = (int64_t)(p.table + 2 * p.amp + p.st[0] + p.st[1]);
    return p;
}

// alpha, beta, gamma: a photon is absent, noisy, pure.  modes: the photons'
// input modes, non-decreasing.
cudaError_t launch_source(const SourcePlan& p, int m, int n, const int* modes, const double2* U, double alpha,
                          double beta, double gamma, double* prob, void* ws, cudaStream_t s)
{
    char* w = (char*)ws;
    int64_t* mc = (int64_t*)w;            w += p.table;
    double2* amp[2];
    amp[0] = (double2*)w;                 w += p.amp;
    amp[1] = (double2*)w;                 w += p.amp;
    double* st[2];
    st[0] = (double*)w;                   w += p.st[0];
    st[1] = (double*)w;
    cudaError_t e = build_multiset_table(mc, m, n, s);
    if (e != cudaSuccess) return e;
    SourceStage g;
    stage_layout(p.N, n, n, g.in_base, g.in_len);
    if ((e = launch_set_one(st[n & 1], s)) != cudaSuccess) return e;        // the empty set
    ExpandArgs a;
    expand_defaults(&a);
    a.source = kExpandSubsets;
    a.U = U;
    a.m = m;
    a.mc = mc;
    a.kmax = n;
    for (int j = 0; j < n; ++j) a.col[j] = modes[j];
    double wk = 1.0;
    for (int k = 1; k <= n; ++k) {
        wk *= gamma;
        a.k = k;
        a.B = (int)choose(n, k);
        a.count = a.hi = p.N[k];
        a.prev_count = p.N[k - 1];
        a.prev = amp[(k - 1) & 1];
        a.prev_stride = p.N[k - 1];
        a.cur = k < n ? amp[k & 1] : nullptr;
        a.cur_stride = p.N[k];
        a.weighted = st[n & 1] + g.in_base[k];
        a.weight = wk;
        if ((e = launch_expand(a, s)) != cudaSuccess) return e;
    }
    g.mc = mc;
    g.m = m;
    g.n = n;
    g.U = U;
    g.alpha = alpha;
    g.beta = beta;
    for (int k = 0; k <= n; ++k) g.N[k] = p.N[k];
    const size_t smem = (size_t)m * sizeof(double) + (size_t)(m + 1) * (n + 1) * sizeof(int64_t);
    for (int j = n; j >= 1; --j) {
        g.j = j;
        g.col = modes[j - 1];
        g.in = st[j & 1];
        g.out = j > 1 ? st[(j - 1) & 1] : prob;
        stage_layout(p.N, n, j, g.in_base, g.in_len);
        stage_layout(p.N, n, j - 1, g.out_base, g.out_len);
        g.npairs = 0;
        int64_t blocks = 0;
        for (int c = 0; c < j; ++c) {
            g.up[c] = choose(j - 1, c + 1);
            g.nsets[c] = choose(j - 1, c);
            for (int k = c; k <= c + n - j + 1; ++k) {
                blocks += blocks_for(g.nsets[c] * p.N[k]);
                g.pc[g.npairs] = c;
                g.pk[g.npairs] = k;
                g.pend[g.npairs++] = blocks;
            }
        }
        if (blocks > INT32_MAX) return cudaErrorInvalidConfiguration;
        auto go = [&](auto kernel) {
            const cudaError_t r = allow_dynamic_smem((const void*)kernel, smem);
            if (r != cudaSuccess) return r;
            kernel<<<(unsigned)blocks, 256, smem, s>>>(g);
            note_launches(1);
            return cudaGetLastError();
        };
        e = n <= 8 ? go(source_stage_kernel<8>) : go(source_stage_kernel<16>);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_photon_step(const int64_t* mc, const int64_t* cum, int m, int kmax, int k, const double2* U, int c,
                               const double* in_same, const double* in_prev, double alpha, double beta, double* out,
                               int64_t count, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    PhotonStep a;
    a.t = RankTables{mc, cum, m, kmax + 1};
    a.k = k;
    a.c = c;
    a.U = U;
    a.in_same = in_same;
    a.in_prev = in_prev;
    a.alpha = alpha;
    a.beta = beta;
    a.out = out;
    a.count = count;
    if (k <= 16) photon_step_kernel<16><<<blocks_for(count), 256, 0, s>>>(a);
    else photon_step_kernel<PCV_MAX_PHOTONS><<<blocks_for(count), 256, 0, s>>>(a);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_class_conv(const int64_t* mc, const int64_t* cum, int m, int kmax, int a, int b, const double* A,
                              const double* B, double* C, int64_t count, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    ClassConv g;
    g.t = RankTables{mc, cum, m, kmax + 1};
    g.a = a;
    g.b = b;
    g.A = A;
    g.B = B;
    g.C = C;
    g.count = count;
    if (a + b <= 16) class_conv_kernel<16><<<blocks_for(count), 256, 0, s>>>(g);
    else class_conv_kernel<PCV_MAX_PHOTONS><<<blocks_for(count), 256, 0, s>>>(g);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_scale_add(double* acc, const double* x, double w, int64_t count, cudaStream_t s)
{
    if (count == 0) return cudaSuccess;
    scale_add_kernel<<<blocks_for(count), 256, 0, s>>>(acc, x, w, count);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_set_one(double* p, cudaStream_t s)
{
    set_one_kernel<<<1, 1, 0, s>>>(p);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace pcv
