// Full output distribution by photon-by-photon state expansion, the approach
// of the paper's SLOS back-end (Sec. 3.2.3: the full computation path unfolded
// in memory, O(n C(m+n-1, n)) time and memory), written for the GPU.
//
// The output state is prod_j (sum_r U[r][c_j] a_r^dagger) |0> / sqrt(prod t!)
// (Eq. eqperm's amplitudes are its coefficients).  With
// |psi_k> = prod_{j<=k} (sum_r U[r][c_j] a_r^dagger) |0> = sum_{s in S_{m,k}} B_k(s) |s>
// and a_r^dagger |s - e_r> = sqrt(s_r) |s>,
//     B_k(s) = sum_{r : s_r >= 1} U[r][c_k] sqrt(s_r) B_{k-1}(s - e_r),
// B_0 = 1, and a(S) = B_n(S) / sqrt(prod t!).  The kernels carry
// C_k(s) = B_k(s) / sqrt(prod_r s_r!) instead: since (s - e_r)! differs from
// s! by the factor s_r, the square roots cancel and
//     C_k(s) = sum_{r : s_r >= 1} U[r][c_k] C_{k-1}(s - e_r),
// a plain gather with one complex multiply-add per distinct occupied mode
// and no square root; the last level applies
// a(S) = C_n(S) sqrt(prod s!) / sqrt(prod t!).  One thread per state s of
// S_{m,k} (canonical order); the last level is the distribution in
// canonical order.
//
// What bounds it: the FP64 pipe (4 DFMA per state and occupied mode) on large
// levels, the launches on small ones.  Everything else is chosen to stay
// under the FP64 time: ranks are 32-bit and come from a table of counts in
// shared memory, the mode list and the ranks stay in registers (KMAX is a
// template bound), and with a batch a thread unranks its state once for
// kGroup batch entries.

#include <cmath>

#include "expansion.cuh"

namespace pcv {
namespace {

constexpr int kThreads = 256;
constexpr int kGroup = 4;                     // batch entries per thread where the batch is large enough
constexpr int64_t kGroupMinThreads = 152 * 1024;

// The bits of the b-th k-subset in colex order (increasing masks).
__device__ uint32_t colex_mask(int b, int k)
{
    uint32_t mask = 0;
    for (int j = k; j >= 1; --j) {
        int t = j - 1, c = 0;                 // largest t with C(t, j) <= b
        for (;;) {
            int n = 1;                        // C(t + 1, j)
            for (int i = 1; i <= j; ++i) n = n * (t + 2 - i) / i;
            if (n > b) break;
            c = n;
            ++t;
        }
        mask |= 1u << t;
        b -= c;
    }
    return mask;
}

template <int KMAX, int GROUP, typename I>
__global__ void __launch_bounds__(kThreads) expand_kernel(const __grid_constant__ ExpandArgs a)
{
    extern __shared__ double2 s_u[];           // [GROUP][m] columns, then the count table
    const int m = a.m, k = a.k, w1 = k + 1;
    I* s_mc = (I*)(s_u + GROUP * m);
    __shared__ int64_t s_parent[GROUP];
    __shared__ double s_norm[GROUP];
    __shared__ int s_col[GROUP];
    const int b0 = blockIdx.y * GROUP;
    if (threadIdx.x < GROUP) {
        const int b = min(b0 + (int)threadIdx.x, a.B - 1);
        int64_t parent = b;
        double norm = a.norm_t;
        int col = a.source == kExpandSides ? a.col[b] : a.col[0];
        if (a.source == kExpandSubsets) {
            const uint32_t mask = colex_mask(b, k);
            const int top = 31 - __clz(mask);
            int64_t c = 1;                     // C(top, k): colex rank without the largest photon
            for (int i = 1; i <= k; ++i) c = c * (top + 1 - i) / i;
            parent = b - (top >= k ? c : 0);
            double f = 1.0;                    // prod t! of the subset's input
            int run = 0, last = -1;
            for (int j = 0; j <= top; ++j)
                if ((mask >> j) & 1u) {
                    run = a.col[j] == last ? run + 1 : 1;
                    last = a.col[j];
                    f *= run;
                }
            norm = 1.0 / f;                    // squared norm: `weighted` holds probabilities
            col = a.col[top];
        }
        s_col[threadIdx.x] = col;
        s_parent[threadIdx.x] = parent;
        s_norm[threadIdx.x] = norm;
    }
    for (int q = threadIdx.x; q < (m + 1) * w1; q += kThreads)
        s_mc[q] = (I)a.mc[(q / w1) * (a.kmax + 1) + q % w1];
    __syncthreads();
    for (int q = threadIdx.x; q < GROUP * m; q += kThreads) {
        const int j = q / m, r = q % m;
        const size_t ub = a.source == kExpandBatch ? (size_t)min(b0 + j, a.B - 1) * m * m : 0;
        s_u[q] = a.U[ub + (size_t)r * m + s_col[j]];
    }
    __syncthreads();

    const int64_t i = a.lo + (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i >= a.hi) return;
    int l[KMAX];                               // sorted mode list of state i
    {
        I idx = (I)i;
        int v = 0;
#pragma unroll
        for (int p = 0; p < KMAX; ++p) {
            if (p >= k) break;
            v = next_mode<I>(s_mc, w1, m, v, k - 1 - p, idx);
            l[p] = v;
        }
    }
    auto t = [&](int mode, int j) { return s_mc[(m - mode - 1) * w1 + j]; };
    // |S_{m,k-1}| - 1 minus the terms of the list without position p: `pre`
    // those before it, `suf` those after it (moved up by one)
    I pre = (I)(a.prev_count - 1), suf = 0;
#pragma unroll
    for (int q = 1; q < KMAX; ++q)
        if (q < k) suf += t(l[q], k - q);
    double2 acc[GROUP];
#pragma unroll
    for (int j = 0; j < GROUP; ++j) acc[j] = make_double2(0.0, 0.0);
    double sfac = 1.0;                         // sqrt(prod s!)
    int mult = 0;
#pragma unroll
    for (int p = 0; p < KMAX; ++p) {
        if (p >= k) break;
        const int r = l[p];
        mult = (p > 0 && l[p > 0 ? p - 1 : 0] == r) ? mult + 1 : 1;
        const int nxt = p + 1 < k ? l[p + 1 < KMAX ? p + 1 : p] : -1;
        if (nxt != r) {                        // one term per occupied mode, at its last copy
            const I rk = pre - suf;
#pragma unroll
            for (int j = 0; j < GROUP; ++j) {
                const double2 u = s_u[j * m + r];
                if (k == 1) acc[j] = u;
                else cmac(acc[j], u, a.prev[s_parent[j] * a.prev_stride + rk]);
            }
            if (mult > 1) sfac *= a.sqrtfact[mult];
        }
        if (p + 1 < k) {
            pre -= t(r, k - 1 - p);
            suf -= t(nxt, k - 1 - p);
        }
    }
#pragma unroll
    for (int j = 0; j < GROUP; ++j) {
        const int b = b0 + j;
        if (b >= a.B) break;
        if (a.cur) a.cur[(size_t)b * a.cur_stride + i] = acc[j];
        if (a.weighted) {
            const double f = a.weight * s_norm[j] * sfac * sfac;
            a.weighted[(size_t)b * a.count + i] = f * fma(acc[j].x, acc[j].x, acc[j].y * acc[j].y);
        }
        if (a.amp || a.prob) {
            const double sc = sfac * a.norm_t;
            const double2 v = make_double2(acc[j].x * sc, acc[j].y * sc);
            const size_t o = (size_t)b * a.out_stride + (i - a.lo);
            if (a.amp) a.amp[o] = v;
            if (a.prob) a.prob[o] = fma(v.x, v.x, v.y * v.y);
        }
    }
}

template <int KMAX, int GROUP, typename I>
cudaError_t launch_one(const ExpandArgs& a, cudaStream_t s)
{
    const size_t smem = (size_t)GROUP * a.m * sizeof(double2) + (size_t)(a.m + 1) * (a.k + 1) * sizeof(I);
    if (smem > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(expand_kernel<KMAX, GROUP, I>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e != cudaSuccess) return e;
    }
    const dim3 grid((unsigned)((a.hi - a.lo + kThreads - 1) / kThreads), (unsigned)((a.B + GROUP - 1) / GROUP));
    expand_kernel<KMAX, GROUP, I><<<grid, kThreads, smem, s>>>(a);
    note_launches(1);
    return cudaGetLastError();
}

template <int GROUP>
cudaError_t launch_group(const ExpandArgs& a, cudaStream_t s)
{
    if (a.k <= 4) return launch_one<4, GROUP, uint32_t>(a, s);
    if (a.k <= 8) return launch_one<8, GROUP, uint32_t>(a, s);
    return launch_one<16, GROUP, uint32_t>(a, s);
}

int64_t mset_s(int w, int k)
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

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

// CUM[a][k] = sum_{v < a} MC(m - v, k): the rank contribution of all lists
// whose current position is below a.
__global__ void cum_table_kernel(const int64_t* __restrict__ mc, int m, int kmax, int64_t* __restrict__ cum)
{
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    if (k > kmax) return;
    int64_t acc = 0;
    for (int a = 0; a <= m; ++a) {
        cum[a * (kmax + 1) + k] = acc;
        if (a < m) acc += mc[(m - a) * (kmax + 1) + k];
    }
}

}  // namespace

void expand_defaults(ExpandArgs* a)
{
    *a = ExpandArgs{};
    a->B = 1;
    a->norm_t = 1.0;
    a->weight = 1.0;
    double f = 1.0;
    a->sqrtfact[0] = 1.0;
    for (int j = 1; j <= PCV_MAX_PHOTONS; ++j) {
        f *= j;
        a->sqrtfact[j] = std::sqrt(f);
    }
}

// 32-bit ranks and the list in registers up to 16 photons; beyond either the
// 64-bit form with the list in local memory.  Four batch entries share a
// thread's unranking once that still leaves every SM 1024 threads (measured
// on the mesh forward, 64 entries of m=12 n=6).
cudaError_t launch_expand(const ExpandArgs& a, cudaStream_t s)
{
    if (a.hi <= a.lo || a.B < 1) return cudaSuccess;
    if (a.k > 16 || a.count > (int64_t)UINT32_MAX) return launch_one<PCV_MAX_PHOTONS, 1, int64_t>(a, s);
    if (a.B >= kGroup && (a.hi - a.lo) * (a.B / kGroup) >= kGroupMinThreads) return launch_group<kGroup>(a, s);
    return launch_group<1>(a, s);
}

cudaError_t build_cum_table(const int64_t* mc, int m, int kmax, int64_t* cum, cudaStream_t s)
{
    cum_table_kernel<<<(kmax + 32) / 32, 32, 0, s>>>(mc, m, kmax, cum);
    note_launches(1);
    return cudaGetLastError();
}

// Workspace: the count table, then two level buffers of the largest
// intermediate level per batch entry.
int64_t slos_workspace(int B, int m, int n)
{
    int64_t half = 1;
    for (int k = 0; k < n; ++k) {
        const int64_t c = mset_s(m, k);
        if (c < 0) return -1;
        half = c > half ? c : half;
    }
    if (half > INT64_MAX / ((int64_t)B * 64)) return -1;
    return (int64_t)(2 * al256((size_t)(m + 1) * (n + 1) * sizeof(int64_t)) +
                     2 * al256((size_t)B * half * sizeof(double2)));
}

cudaError_t launch_slos(const Plan& p, int B, const double2* U, int64_t lo, int64_t hi, double* prob, double2* amp,
                        void* ws, cudaStream_t s)
{
    const int m = p.m, n = p.n;
    int64_t half = 1;
    for (int k = 0; k < n; ++k) {
        const int64_t c = mset_s(m, k);
        half = c > half ? c : half;
    }
    char* w = (char*)ws;
    int64_t* mc = (int64_t*)w;          w += 2 * al256((size_t)(m + 1) * (n + 1) * sizeof(int64_t));
    double2* buf[2];
    buf[0] = (double2*)w;               w += al256((size_t)B * half * sizeof(double2));
    buf[1] = (double2*)w;
    if (!amp && !prob) return cudaErrorInvalidValue;
    cudaError_t e = build_multiset_table(mc, m, n, s);
    if (e != cudaSuccess) return e;
    ExpandArgs a;
    expand_defaults(&a);
    a.source = kExpandBatch;
    a.U = U;
    a.m = m;
    a.mc = mc;
    a.kmax = n;
    a.B = B;
    a.norm_t = p.norm_t;
    a.prev_stride = a.cur_stride = half;
    for (int k = 1; k <= n; ++k) {
        const bool last = k == n;
        a.k = k;
        a.col[0] = p.cols[k - 1];
        a.count = mset_s(m, k);
        a.lo = last ? lo : 0;
        a.hi = last ? hi : a.count;
        a.prev_count = mset_s(m, k - 1);
        a.prev = buf[(k - 1) & 1];
        a.cur = last ? nullptr : buf[k & 1];
        a.amp = last ? amp : nullptr;
        a.prob = last ? prob : nullptr;
        a.out_stride = hi - lo;
        if ((e = launch_expand(a, s)) != cudaSuccess) return e;
    }
    return cudaSuccess;
}

}  // namespace pcv
