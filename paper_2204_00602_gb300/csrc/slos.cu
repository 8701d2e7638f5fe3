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

#include <algorithm>
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
    if (k == 1) level_below_done();
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
    if (k > 1) level_below_done();

    const int64_t i = a.lo + (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i >= a.hi) return;
    double2 acc[GROUP];
#pragma unroll
    for (int j = 0; j < GROUP; ++j) acc[j] = make_double2(0.0, 0.0);
    const double sfac = expand_state<KMAX, I>(s_mc, w1, m, k, (I)i, (I)a.prev_count, a.sqrtfact, [&](int r, I rk, int) {
#pragma unroll
        for (int j = 0; j < GROUP; ++j) {
            const double2 u = s_u[j * m + r];
            if (k == 1) acc[j] = u;
            else cmac(acc[j], u, a.prev[s_parent[j] * a.prev_stride + rk]);
        }
    });
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
    const cudaError_t e = allow_dynamic_smem((const void*)expand_kernel<KMAX, GROUP, I>, smem);
    if (e != cudaSuccess) return e;
    const dim3 grid((unsigned)((a.hi - a.lo + kThreads - 1) / kThreads), (unsigned)((a.B + GROUP - 1) / GROUP));
    return launch_level_kernel(expand_kernel<KMAX, GROUP, I>, grid, kThreads, smem, s, a);
}

template <int GROUP>
cudaError_t launch_group(const ExpandArgs& a, cudaStream_t s)
{
    if (a.k <= 4) return launch_one<4, GROUP, uint32_t>(a, s);
    if (a.k <= 8) return launch_one<8, GROUP, uint32_t>(a, s);
    return launch_one<16, GROUP, uint32_t>(a, s);
}

// Small problems: every level of a batch entry in one block, the levels below
// the last in shared memory, one launch in all (the count table and the call's
// status word included).  Level by level the launches bound such a call: m=6
// n=3 took 65 us with the ten launches of the tensor-core plan, 31 with one
// (most of it the host's call).
struct SmallArgs {
    const double2* U;          // [B][m][m]
    int m, n;
    int col[16];
    uint32_t count[17];        // states of level k
    uint32_t even;             // entries of the even levels' buffer
    int64_t lo, hi;            // outputs, at [b][o - lo]
    double2* amp;
    double* prob;
    int64_t out_stride;
    double norm_t;
    int64_t* status;           // two words zeroed, or null
    double sqrtfact[17];
};

template <int KMAX>
__global__ void __launch_bounds__(kThreads) expand_small_kernel(const __grid_constant__ SmallArgs a)
{
    extern __shared__ double2 s_lev[];         // even levels, odd levels, U's columns [n][m], the counts
    const int m = a.m, n = a.n, w1 = n + 1, b = blockIdx.x;
    uint32_t odd = 1;
    for (int k = 1; k < n; k += 2) odd = max(odd, a.count[k]);
    double2* s_u = s_lev + a.even + odd;
    uint32_t* s_mc = (uint32_t*)(s_u + n * m);
    if (a.status && b == 0 && threadIdx.x < 2) a.status[threadIdx.x] = 0;
    for (int q = threadIdx.x; q < n * m; q += kThreads)
        s_u[q] = a.U[((size_t)b * m + q % m) * m + a.col[q / m]];
    for (int w = threadIdx.x; w <= m; w += kThreads) {
        uint64_t c = 1;
        s_mc[w * w1] = 1;
        for (int j = 1; j <= n; ++j) {
            c = c * (uint64_t)(w + j - 1) / (uint64_t)j;
            s_mc[w * w1 + j] = (uint32_t)c;
        }
    }
    __syncthreads();
    for (int k = 1; k <= n; ++k) {
        const bool last = k == n;
        const double2* prev = s_lev + (k & 1 ? 0 : a.even);
        double2* cur = s_lev + (k & 1 ? a.even : 0);
        const double2* u = s_u + (k - 1) * m;
        const int64_t hi = last ? a.hi : (int64_t)a.count[k];
        for (int64_t i = (last ? a.lo : 0) + threadIdx.x; i < hi; i += kThreads) {
            double2 acc = make_double2(0.0, 0.0);
            const double sf = expand_state<KMAX, uint32_t>(s_mc, w1, m, k, (uint32_t)i, a.count[k - 1], a.sqrtfact,
                                                           [&](int r, uint32_t rk, int) {
                                                               if (k == 1) acc = u[r];
                                                               else cmac(acc, u[r], prev[rk]);
                                                           });
            if (!last) {
                cur[i] = acc;
                continue;
            }
            const double sc = sf * a.norm_t;
            const double2 v = make_double2(acc.x * sc, acc.y * sc);
            const size_t o = (size_t)b * a.out_stride + (i - a.lo);
            if (a.amp) a.amp[o] = v;
            if (a.prob) a.prob[o] = fma(v.x, v.x, v.y * v.y);
        }
        __syncthreads();
    }
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

namespace {

// Shared memory of expand_small_kernel, or 0 where the launches per level are
// the better form: one SM would need more time for the multiply-adds (2 cycles
// each) than n launches take (about 4,800 cycles each).
size_t small_smem(int m, int n, SmallArgs* a)
{
    if (n < 1 || n > 16 || m > 256) return 0;
    double terms = 0.0;
    int64_t even = 1, odd = 1;
    for (int k = 0; k <= n; ++k) {
        const int64_t c = mset_s(m, k);
        if (c < 0 || c > 100000) return 0;
        a->count[k] = (uint32_t)c;
        if (k < n) {
            terms += (double)m * (double)c;
            (k & 1 ? odd : even) = std::max(k & 1 ? odd : even, c);
        }
    }
    a->even = (uint32_t)even;
    if (2.0 * terms > 4800.0 * n) return 0;
    const size_t b = (size_t)(even + odd + (int64_t)n * m) * sizeof(double2) + (size_t)(m + 1) * (n + 1) * sizeof(uint32_t);
    return b <= 100 * 1024 ? b : 0;
}

}  // namespace

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

cudaError_t launch_slos(const Plan& p, int B, const double2* U, int64_t lo, int64_t hi, bool fixed, double* prob,
                        double2* amp, void* ws, void* status, cudaStream_t s)
{
    const int m = p.m, n = p.n;
    if (!amp && !prob) return cudaErrorInvalidValue;
    SmallArgs sm;
    if (const size_t smem = small_smem(m, n, &sm)) {
        ExpandArgs d;
        expand_defaults(&d);
        sm.U = U;
        sm.m = m;
        sm.n = n;
        for (int j = 0; j < n; ++j) sm.col[j] = p.cols[j];
        sm.lo = lo;
        sm.hi = hi;
        sm.amp = amp;
        sm.prob = prob;
        sm.out_stride = hi - lo;
        sm.norm_t = p.norm_t;
        sm.status = (int64_t*)status;
        for (int j = 0; j <= 16; ++j) sm.sqrtfact[j] = d.sqrtfact[j];
        auto go = [&](auto kernel) {
            const cudaError_t e = allow_dynamic_smem((const void*)kernel, smem);
            if (e != cudaSuccess) return e;
            kernel<<<B, kThreads, smem, s>>>(sm);
            note_launches(1);
            return cudaGetLastError();
        };
        return n <= 4 ? go(expand_small_kernel<4>) : n <= 8 ? go(expand_small_kernel<8>) : go(expand_small_kernel<16>);
    }
    int64_t half = 1, states = 0;
    int64_t count[PCV_MAX_PHOTONS + 1];
    for (int k = 0; k <= n; ++k) {
        count[k] = mset_s(m, k);
        if (k < n) half = std::max(half, count[k]);
        states += count[k] < kFixedMinStates ? count[k] : kFixedMinStates;
    }
    fixed = fixed && B == 1 && hi > lo && expand_fixed_applies(m, n, std::max(half, count[n]), states);
    if (status && !fixed) {
        const cudaError_t e = cudaMemsetAsync(status, 0, 16, s);
        if (e != cudaSuccess) return e;
    }
    char* w = (char*)ws;
    int64_t* mc = (int64_t*)w;          w += al256((size_t)(m + 1) * (n + 1) * sizeof(int64_t));
    void* header = w;                   w += al256((size_t)(m + 1) * (n + 1) * sizeof(int64_t));
    double2* buf[2];
    buf[0] = (double2*)w;               w += al256((size_t)B * half * sizeof(double2));
    buf[1] = (double2*)w;
    cudaError_t e = build_multiset_table(mc, m, n, s);
    if (e != cudaSuccess) return e;
    if (fixed) return launch_expand_fixed(p, U, count, lo, hi, prob, amp, mc, header, buf, (int64_t*)status, s);
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
        a.count = count[k];
        a.lo = last ? lo : 0;
        a.hi = last ? hi : a.count;
        a.prev_count = count[k - 1];
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
