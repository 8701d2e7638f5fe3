// Adjoint of the full distribution by the state expansion (slos.cu run
// backwards): dL/dU from dL/da over every output of S_{m,n}, for B unitaries.
//
// Forward, with photon k entering mode c_k:
//     C_k(s) = sum_{r : s_r >= 1} U[r][c_k] C_{k-1}(s - e_r),
//     a(S) = C_n(S) sqrt(prod S!) norm_t.
// With the dL/dRe + i dL/dIm convention (a is holomorphic in U) the reverse
// sweep carries D_k(s) = dL/dC_k(s):
//     D_n(S) = gbar(S) sqrt(prod S!) norm_t,
//     D_{k-1}(s) = sum_r conj(U[r][c_k]) D_k(s + e_r),
//     dL/dU[r][c_k] += sum_s D_k(s + e_r) conj(C_{k-1}(s)),
// both over the states s of S_{m,k-1}: 8 DFMA per state and mode, against
// 2^{n-1} (8n + 2n^2 ...) per output for minors as Glynn sums (adjoint.cu,
// which stays for explicit outputs and for workspaces too small for the
// levels).
//
// Kernels:
//   succ_kernel        the rank of s + e_r in S_{m,k} for every state s of the
//                      levels 0..n-1 and every mode r, once per call: shared
//                      by all batch entries and by the whole reverse sweep;
//   seed_kernel        D_n;
//   grad_level_kernel  one level: a block takes 32 T states, its warps the
//                      modes r = warp, warp + 8, ...; a lane holds T states,
//                      so a mode's products are summed in registers over T
//                      states before one warp reduction, and the eight warps'
//                      shares of D_{k-1} are added in warp order;
//   grad_final_kernel  dL/dU[r][c]: the blocks' partial sums of every level
//                      whose photon enters c, in one fixed order.
// No atomics: a call gives the same bits every time.

#include <algorithm>

#include "expansion.cuh"

namespace pcv {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

size_t al256(size_t x) { return (x + 255) & ~(size_t)255; }

int64_t mset_g(int w, int k)
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

struct SuccArgs {
    const int64_t* mc;               // MC, row length n + 1
    int m, n;
    int64_t off[PCV_MAX_PHOTONS + 2];   // states of the levels before L, L <= n + 1
    uint32_t* succ;                  // level L at m * off[L]: [r][states of L]
};

__global__ void __launch_bounds__(kThreads) succ_kernel(const __grid_constant__ SuccArgs a)
{
    const int64_t t = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (t >= a.off[a.n]) return;
    int L = 0;
    while (t >= a.off[L + 1]) ++L;
    const int64_t i = t - a.off[L], cnt = a.off[L + 1] - a.off[L];
    const int m = a.m, w1 = a.n + 1, k = L + 1;
    int l[PCV_MAX_PHOTONS];
    {
        int64_t idx = i;
        int v = 0;
        for (int p = 0; p < L; ++p) {
            v = next_mode<int64_t>(a.mc, w1, m, v, L - 1 - p, idx);
            l[p] = v;
        }
    }
    auto tt = [&](int mode, int j) { return a.mc[(m - mode - 1) * w1 + j]; };
    // inserting r at position p: the positions before p keep their terms of
    // S_{m,k} (pre), the others move up by one (suf)
    int64_t pre = a.off[L + 2] - a.off[L + 1] - 1, suf = 0;
    for (int q = 0; q < L; ++q) suf += tt(l[q], k - q - 1);
    uint32_t* out = a.succ + (int64_t)m * a.off[L] + i;
    int p = 0;
    for (int r = 0; r < m; ++r) {
        while (p < L && l[p] <= r) {
            pre -= tt(l[p], k - p);
            suf -= tt(l[p], k - p - 1);
            ++p;
        }
        out[(int64_t)r * cnt] = (uint32_t)(pre - suf - tt(r, k - p));
    }
}

struct SeedArgs {
    const int64_t* mc;
    int m, n, B;
    double norm_t;
    double sqrtfact[PCV_MAX_PHOTONS + 1];
    int64_t count;
    const double2* gbar;             // [B][count]
    double2* D;                      // [B][count]
};

__global__ void __launch_bounds__(kThreads) seed_kernel(const __grid_constant__ SeedArgs a)
{
    const int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x;
    if (i >= a.count) return;
    const int w1 = a.n + 1;
    int64_t idx = i;
    int v = 0, run = 0;
    double f = a.norm_t;
    for (int p = 0; p < a.n; ++p) {
        const int u = next_mode<int64_t>(a.mc, w1, a.m, v, a.n - 1 - p, idx);
        if (p > 0 && u != v) {
            f *= a.sqrtfact[run];
            run = 0;
        }
        v = u;
        ++run;
    }
    f *= a.sqrtfact[run];
    for (int b = blockIdx.y; b < a.B; b += gridDim.y) {
        const double2 g = a.gbar[(size_t)b * a.count + i];
        a.D[(size_t)b * a.count + i] = make_double2(f * g.x, f * g.y);
    }
}

struct GradLevelArgs {
    const double2* U;                // [B][m][m]
    int m, col;
    int64_t cnt, up;                 // states of level k - 1 and of level k
    const uint32_t* succ;            // [m][cnt]
    const double2* C;                // [B][cnt], or null (level 0: 1)
    const double2* D;                // [B][up]
    double2* Dout;                   // [B][cnt], or null (level 0)
    double2* part;                   // [B][part_stride]: this level at tile * m + r
    int64_t part_stride;
};

template <int T>
__global__ void __launch_bounds__(kThreads) grad_level_kernel(const __grid_constant__ GradLevelArgs a)
{
    __shared__ double2 s_d[kWarps][32 * T];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int b = blockIdx.y, m = a.m;
    const int64_t s0 = (int64_t)blockIdx.x * (32 * T) + lane;
    const double2* D = a.D + (size_t)b * a.up;
    const double2* U = a.U + (size_t)b * m * m + a.col;
    double2 c[T], d[T];
    bool live[T];
#pragma unroll
    for (int t = 0; t < T; ++t) {
        live[t] = s0 + 32 * t < a.cnt;
        d[t] = make_double2(0.0, 0.0);
        c[t] = make_double2(0.0, 0.0);
        if (live[t]) c[t] = a.C ? a.C[(size_t)b * a.cnt + s0 + 32 * t] : make_double2(1.0, 0.0);
    }
    double2* part = a.part + (size_t)b * a.part_stride + (int64_t)blockIdx.x * m;
    for (int r = warp; r < m; r += kWarps) {
        const double2 u = __ldg(U + (size_t)r * m);
        const uint32_t* sr = a.succ + (int64_t)r * a.cnt;
        double2 v[T];
#pragma unroll
        for (int t = 0; t < T; ++t) v[t] = live[t] ? D[sr[s0 + 32 * t]] : make_double2(0.0, 0.0);
        double2 g = make_double2(0.0, 0.0);
#pragma unroll
        for (int t = 0; t < T; ++t) {
            cmac(d[t], make_double2(u.x, -u.y), v[t]);
            cmac(g, v[t], make_double2(c[t].x, -c[t].y));
        }
        for (int off = 16; off > 0; off >>= 1) {
            g.x += __shfl_xor_sync(0xffffffffu, g.x, off);
            g.y += __shfl_xor_sync(0xffffffffu, g.y, off);
        }
        if (lane == 0) part[r] = g;
    }
    if (!a.Dout) return;
#pragma unroll
    for (int t = 0; t < T; ++t) s_d[warp][lane + 32 * t] = d[t];
    __syncthreads();
    for (int q = threadIdx.x; q < 32 * T; q += kThreads) {
        const int64_t st = (int64_t)blockIdx.x * (32 * T) + q;
        if (st >= a.cnt) break;
        double2 v = s_d[0][q];
        for (int w = 1; w < kWarps; ++w) v = cadd(v, s_d[w][q]);
        a.Dout[(size_t)b * a.cnt + st] = v;
    }
}

struct FinalArgs {
    int m, n;
    int col[PCV_MAX_PHOTONS];
    int64_t base[PCV_MAX_PHOTONS];   // photon k's partial sums: [tiles[k]][m] at base[k]
    int tiles[PCV_MAX_PHOTONS];
    const double2* part;
    int64_t part_stride;
    double2* gradU;                  // [B][m][m]
};

// A warp per (batch entry, r, c): lanes stride the tiles, photon by photon,
// then one warp reduction.  Columns without a photon get zero.
__global__ void __launch_bounds__(kThreads) grad_final_kernel(const __grid_constant__ FinalArgs a)
{
    const int lane = threadIdx.x & 31;
    const int64_t e = (int64_t)blockIdx.x * kWarps + (threadIdx.x >> 5);
    if (e >= (int64_t)a.m * a.m) return;
    const int r = (int)(e / a.m), c = (int)(e % a.m);
    const double2* part = a.part + (size_t)blockIdx.y * a.part_stride;
    double2 v = make_double2(0.0, 0.0);
    bool any = false;
    for (int k = 0; k < a.n; ++k) {
        if (a.col[k] != c) continue;
        any = true;
        for (int t = lane; t < a.tiles[k]; t += 32) v = cadd(v, part[a.base[k] + (int64_t)t * a.m + r]);
    }
    if (any)
        for (int off = 16; off > 0; off >>= 1) {
            v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
            v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
        }
    if (lane == 0) a.gradU[(size_t)blockIdx.y * a.m * a.m + e] = v;
}

// Four states per lane once that fills the GPU, else one.
int level_t(int64_t cnt, int B) { return cnt * B >= 152 * 8 * 128 ? 4 : 1; }

}  // namespace

// The workspace's parts: the count table, the successor ranks, levels 1..n-1
// of C, two buffers for D, the partial sums.
ExpandGradPlan expand_grad_plan(int m, int n, int B)
{
    ExpandGradPlan p{};
    p.total = -1;
    if (n < 1) return p;
    int64_t states = 0, parts = 0;
    for (int L = 0; L <= n; ++L) {
        const int64_t c = mset_g(m, L);
        if (c < 0 || c > (int64_t)UINT32_MAX) return p;
        p.cnt[L] = c;
        if (L == n) break;
        p.off[L] = states;
        states += c;
        p.tiles[L] = (c + 32 * level_t(c, B) - 1) / (32 * level_t(c, B));
        p.base[L] = parts;
        parts += p.tiles[L] * m;
    }
    p.off[n] = states;
    p.parts = parts;
    const unsigned __int128 bytes = (unsigned __int128)B * ((unsigned __int128)(states + parts) + p.cnt[n] + p.cnt[n - 1]) * 16 +
                                    (unsigned __int128)states * m * 4;
    if (bytes > ((unsigned __int128)1 << 50)) return p;
    p.table = al256((size_t)(m + 1) * (n + 1) * sizeof(int64_t));
    p.succ = al256((size_t)states * m * sizeof(uint32_t));
    p.levels = al256((size_t)B * states * sizeof(double2));
    p.d0 = al256((size_t)B * p.cnt[n] * sizeof(double2));
    p.d1 = al256((size_t)B * p.cnt[n - 1] * sizeof(double2));
    p.part = al256((size_t)B * parts * sizeof(double2));
    p.total = (int64_t)(p.table + p.succ + p.levels + p.d0 + p.d1 + p.part);
    return p;
}

cudaError_t launch_expand_grad(const Plan& pl, const double2* U, int B, const double2* gbar, double2* gradU, void* ws,
                               const ExpandGradPlan& p, cudaStream_t s)
{
    const int m = pl.m, n = pl.n;
    char* w = (char*)ws;
    int64_t* mc = (int64_t*)w;            w += p.table;
    uint32_t* succ = (uint32_t*)w;        w += p.succ;
    double2* levels = (double2*)w;        w += p.levels;
    double2* D[2];
    D[0] = (double2*)w;                   w += p.d0;
    D[1] = (double2*)w;                   w += p.d1;
    double2* part = (double2*)w;
    cudaError_t e = build_multiset_table(mc, m, n, s);
    if (e != cudaSuccess) return e;

    SuccArgs su;
    su.mc = mc;
    su.m = m;
    su.n = n;
    for (int L = 0; L <= n; ++L) su.off[L] = p.off[L];
    su.off[n + 1] = p.off[n] + p.cnt[n];
    su.succ = succ;
    succ_kernel<<<(unsigned)((p.off[n] + kThreads - 1) / kThreads), kThreads, 0, s>>>(su);
    note_launches(1);

    // forward levels 1 .. n-1, each kept: level L at B * off[L]
    ExpandArgs a;
    expand_defaults(&a);
    a.source = kExpandBatch;
    a.U = U;
    a.m = m;
    a.mc = mc;
    a.kmax = n;
    a.B = B;
    for (int k = 1; k < n; ++k) {
        a.k = k;
        a.col[0] = pl.cols[k - 1];
        a.count = a.hi = p.cnt[k];
        a.prev_count = p.cnt[k - 1];
        a.prev = levels + (size_t)B * p.off[k - 1];
        a.prev_stride = p.cnt[k - 1];
        a.cur = levels + (size_t)B * p.off[k];
        a.cur_stride = p.cnt[k];
        if ((e = launch_expand(a, s)) != cudaSuccess) return e;
    }

    SeedArgs sd;
    sd.mc = mc;
    sd.m = m;
    sd.n = n;
    sd.B = B;
    sd.norm_t = pl.norm_t;
    for (int j = 0; j <= PCV_MAX_PHOTONS; ++j) sd.sqrtfact[j] = a.sqrtfact[j];
    sd.count = p.cnt[n];
    sd.gbar = gbar;
    sd.D = D[0];
    seed_kernel<<<dim3((unsigned)((p.cnt[n] + kThreads - 1) / kThreads), (unsigned)std::min(B, 8)), kThreads, 0, s>>>(sd);
    note_launches(1);

    FinalArgs f;
    f.m = m;
    f.n = n;
    int cur = 0;
    for (int k = n; k >= 1; --k) {
        GradLevelArgs g;
        g.U = U;
        g.m = m;
        g.col = pl.cols[k - 1];
        g.cnt = p.cnt[k - 1];
        g.up = p.cnt[k];
        g.succ = succ + (size_t)m * p.off[k - 1];
        g.C = k > 1 ? levels + (size_t)B * p.off[k - 1] : nullptr;
        g.D = D[cur];
        g.Dout = k > 1 ? D[cur ^ 1] : nullptr;
        g.part = part + p.base[k - 1];
        g.part_stride = p.parts;
        const dim3 grid((unsigned)p.tiles[k - 1], (unsigned)B);
        if (level_t(g.cnt, B) == 4) grad_level_kernel<4><<<grid, kThreads, 0, s>>>(g);
        else grad_level_kernel<1><<<grid, kThreads, 0, s>>>(g);
        note_launches(1);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
        f.col[k - 1] = pl.cols[k - 1];
        f.base[k - 1] = p.base[k - 1];
        f.tiles[k - 1] = (int)p.tiles[k - 1];
        cur ^= 1;
    }
    f.part = part;
    f.part_stride = p.parts;
    f.gradU = gradU;
    grad_final_kernel<<<dim3((unsigned)((m * m + kWarps - 1) / kWarps), (unsigned)B), kThreads, 0, s>>>(f);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace pcv
