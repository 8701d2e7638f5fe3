// Photon-by-photon state expansion: index arithmetic and launch interface
// shared by the full distribution (slos.cu), its adjoint (expansion_grad.cu),
// the source model (distinguish.cu) and the split amplitudes (split.cu).
//
// Ranks.  With MC(w, j) = C(w + j - 1, j), the multisets of size j over w
// modes, and t(l, j) = MC(m - l - 1, j), those over the modes above l, the
// canonical index of a sorted mode list l_0 <= ... <= l_{L-1} of S_{m,L} is
//     rank = |S_{m,L}| - 1 - sum_q t(l_q, L - q):
// the q-th sum of the lists before it, MC(m - l_{q-1}, L - q) - MC(m - l_q,
// L - q), telescopes through MC(w, j) = MC(w - 1, j) + MC(w, j - 1).  So each
// position contributes one entry of the table of counts, and taking a photon
// out, or putting one in, moves the later positions' entries by one column.
#pragma once

#include "pcv_common.cuh"

namespace pcv {

// Where a batch entry of a level launch takes its photon and its parent from.
enum ExpandSource {
    kExpandBatch = 0,    // entry b: unitary b, the same photon (column col[0]) for all
    kExpandSides = 1,    // entry b: column col[b] of one unitary
    kExpandSubsets = 2,  // entry b: the b-th k-subset of the photons (colex order); its
                         // largest photon is added to the entry of the other k - 1
};

struct ExpandArgs {
    int source;
    const double2* U;          // [B][m][m] (kExpandBatch) or [m][m]
    int m, k;                  // modes, level built (k >= 1)
    int col[PCV_MAX_PHOTONS];  // columns (kExpandSubsets: of every photon)
    const int64_t* mc;         // multiset counts MC[a][j], row length kmax + 1
    int kmax;
    int B;                     // batch entries
    int64_t count;             // states of level k
    int64_t prev_count;        // states of level k - 1
    int64_t lo, hi;            // states written (the whole level unless it is the last one)
    const double2* prev;       // [entries of level k-1][prev_stride]; not read at k = 1
    int64_t prev_stride;
    double2* cur;              // [B][cur_stride] (or null: the last level)
    int64_t cur_stride;
    double2* amp;              // last level: at [b][i - lo], stride out_stride, scaled
    double* prob;
    int64_t out_stride;
    double norm_t;             // 1 / sqrt(prod t!)
    double* weighted;          // kExpandSubsets: weight * |a|^2 at [b][i], stride count, or null
    double weight;
    double sqrtfact[PCV_MAX_PHOTONS + 1];   // sqrt(j!)
};

// Fills the fields that depend on no particular level (sqrtfact included).
void expand_defaults(ExpandArgs* a);
cudaError_t launch_expand(const ExpandArgs& a, cudaStream_t s);

// The same levels of one unitary in fixed point (expansion_fixed.cu); count[k]:
// the states of level k, buf: two levels, header: 256 bytes.
constexpr int64_t kFixedMinStates = 500000;
bool expand_fixed_applies(int m, int n, int64_t largest, int64_t states);
cudaError_t launch_expand_fixed(const Plan& p, const double2* U, const int64_t* count, int64_t lo, int64_t hi,
                                double* prob, double2* amp, const int64_t* mc, void* header, double2* const* buf,
                                int64_t* status, cudaStream_t s);

#ifdef __CUDACC__
// Levels follow one another on the stream with programmatic launch: a level's
// blocks come up and fetch their tables while the level below still runs, and
// wait for it before they read or write a state.  Level 1 waits first: the
// kernel before it writes the count table, and nothing says who wrote U.  Every
// level waits before it lets the next one come up, so whatever was written two
// launches ago is complete when a level starts.  On the device (plain launches
// before): m=13 n=7 51 to 35 us, m=16 n=8 88 to 65, m=12 n=12 203 to 168, the
// source model at m=12 n=6 108 to 85, 4,096 outputs at m=20 n=10 67 to 61.
template <typename... P, typename A>
cudaError_t launch_level_kernel(void (*kernel)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s, const A& a)
{
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &attr;
    c.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&c, kernel, a);
    if (e == cudaSuccess) note_launches(1);
    return e;
}

__device__ __forceinline__ void level_below_done()
{
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
}

// Sorted mode list of index i of S_{m,k}, from the shared or global table t
// (row length w1): t[a * w1 + j] = MC(a, j).
template <typename I>
__device__ __forceinline__ int next_mode(const I* t, int w1, int m, int v, int rest, I& idx)
{
    for (;;) {
        const I c = t[(m - v) * w1 + rest];
        if (idx < c) return v;
        idx -= c;
        ++v;
    }
}

// State i of S_{m,k} (count table mc, row length w1): term(r, rank, photons) for
// every occupied mode r, rank that of the state without one photon of r among
// the prev_n states of S_{m,k-1}.  Returns sqrt(prod s!) (1 without the table).
template <int KMAX, typename I, typename F>
__device__ __forceinline__ double expand_state(const I* mc, int w1, int m, int k, I i, I prev_n, const double* sqrtfact,
                                               F&& term)
{
    int l[KMAX];                               // sorted mode list
    {
        int v = 0;
#pragma unroll
        for (int p = 0; p < KMAX; ++p) {
            if (p >= k) break;
            // below the last position every mode counts for one state
            v = p + 1 < k ? next_mode<I>(mc, w1, m, v, k - 1 - p, i) : v + (int)i;
            l[p] = v;
        }
    }
    auto t = [&](int mode, int j) { return mc[(m - mode - 1) * w1 + j]; };
    // prev_n - 1 minus the terms of the list without position p: `pre` those
    // before it, `suf` those after it (moved up by one)
    I pre = prev_n - 1, suf = 0;
#pragma unroll
    for (int q = 1; q < KMAX; ++q)
        if (q < k) suf += t(l[q], k - q);
    double sfac = 1.0;
    int mult = 0;
#pragma unroll
    for (int p = 0; p < KMAX; ++p) {
        if (p >= k) break;
        const int r = l[p];
        mult = (p > 0 && l[p > 0 ? p - 1 : 0] == r) ? mult + 1 : 1;
        const int nxt = p + 1 < k ? l[p + 1 < KMAX ? p + 1 : p] : -1;
        if (nxt != r) {                        // one term per occupied mode, at its last copy
            term(r, (I)(pre - suf), mult);
            if (mult > 1 && sqrtfact) sfac *= sqrtfact[mult];
        }
        if (p + 1 < k) {
            pre -= t(r, k - 1 - p);
            suf -= t(nxt, k - 1 - p);
        }
    }
    return sfac;
}
#endif

}  // namespace pcv
